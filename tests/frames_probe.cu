// Host-only probe of the diagonal-frame planner (qng_frames_plan.cu), built and run by
// tests/test_frames_host.py: reads a circuit with its Hamiltonian and angles, builds the program and
// executes it in float64 on the host, step by step as the kernels do (exchanges, permutations,
// Hadamards on a thread's own bits, runs), and prints
//   E <energy>, grad <P values>, L <re im> for i < j, sigma <P values>, ctrl <P values>
// Structural invariants are checked on the way ("bad <what>", exit 1). Both forms of a program, for float32 and
// for fixed-point vectors, are executed and have to agree; halvings are where the kernels have them.
// The same for the streaming program (tiles of 2^tb amplitudes, `low` contiguous low bits) when tb > 0.
// Input (stdin): n P G T kb cl tb low, G lines "kind q0 q1 param xmask zmask", T lines "coeff x z", P angles.
#include <cmath>
#include <complex>
#include <cstdio>
#include <cstdlib>
#include <vector>

#include "qng_frames.h"

using namespace qng;
using namespace qng::frames;
typedef std::complex<double> cd;

static void bad(const char *what, long a, long b) {
    std::printf("bad %s %ld %ld\n", what, a, b);
    std::exit(1);
}

// Halvings. Fixed-point vectors have room for 2^4.5 of their norm, float32 ones are left to grow to 2^(kTableHalf / 2).
static void scale(std::vector<cd> &v, int shift, bool fixed) {
    double nrm = 0, f = std::ldexp(1.0, -shift);
    for (const cd &x : v) nrm += std::norm(x);
    if (std::sqrt(nrm) > std::ldexp(1.0001, fixed ? 5 : kTableHalf / 2)) bad("growth", (long)std::log2(nrm), shift);
    if (shift < 0 || shift > 32) bad("shift", shift, 0);
    for (cd &x : v) x *= f;
}

static cd member_factor(const std::vector<Member> &mem, const Run &rn, const std::vector<double> &th, uint32_t m) {
    cd f = std::pow(0.5, 0.5 * rn.khalf);
    for (int k = 0; k < rn.mem_count; ++k) {
        const Member &e = mem[rn.mem_begin + k];
        const int par = __builtin_popcount(m & e.z) & 1;
        const double lam = par ? -e.sgn : e.sgn;
        if (e.kind == 2) { if (par) f *= cd(0, -1); continue; }
        if ((m & e.ctrl) != e.cval) continue;
        f *= e.kind == 1 ? cd(lam) : cd(std::cos(th[e.param] / 2), -lam * std::sin(th[e.param] / 2));
    }
    return f;
}

// Prints the first form's results and holds the second's against them.
static void print_all(double E, const std::vector<double> &grad, const std::vector<double> &sig, const std::vector<double> &ctrl,
                      const std::vector<cd> &Lm, int P, int R) {
    static std::vector<double> first;
    std::vector<double> all{E};
    for (const auto *x : {&grad, &sig, &ctrl}) all.insert(all.end(), x->begin(), x->end());
    for (int j = 0; j < P; ++j) for (int i = 0; i < j; ++i) { all.push_back(Lm[(size_t)i * P + j].real()); all.push_back(Lm[(size_t)i * P + j].imag()); }
    if (!first.empty()) {
        for (size_t k = 0; k < all.size(); ++k)
            if (!(std::fabs(all[k] - first[k]) <= 1e-11 * (1 + std::fabs(first[k])))) bad("forms differ", (long)k, P);
        return;
    }
    first = all;
    std::printf("E %.17g\nruns %d\n", E, R);
    auto vec = [&](const char *nm, const std::vector<double> &x) {
        std::printf("%s", nm);
        for (double t : x) std::printf(" %.17g", t);
        std::printf("\n");
    };
    vec("grad", grad);
    vec("sigma", sig);
    vec("ctrl", ctrl);
    std::printf("L");
    for (int j = 0; j < P; ++j) for (int i = 0; i < j; ++i) std::printf(" %.17g %.17g", Lm[(size_t)i * P + j].real(), Lm[(size_t)i * P + j].imag());
    std::printf("\n");
}

static int stream(const std::vector<qng_gate> &gates, const std::vector<qng_pauli> &terms, const std::vector<double> &th, int n,
                  int P, int kb, int tb, int lowbits, bool fixed) {
    StreamProgram pr;
    build_stream(gates, terms, n, kb, tb, lowbits, fixed, pr);
    for (const Run &r : pr.runs) if (r.khalf > kTableHalf) bad("factor", r.khalf, 0);
    const uint32_t N = 1u << n;
    const int R = (int)pr.runs.size(), w = tb - lowbits;
    int low = -1;
    auto local = [&](const SPass &ps, uint32_t m) { return (m & ((1u << lowbits) - 1)) | (((m >> ps.s) & ((1u << w) - 1)) << lowbits); };
    auto global = [&](const SPass &ps, uint32_t l) { return (l & ((1u << lowbits) - 1)) | ((l >> lowbits) << ps.s); };
    auto move = [&](std::vector<cd> &v, const SPass &ps, const UOp &u) {
        if (u.low >= 0) {
            low = u.low;
            if (u.perm >= 0) {
                std::vector<cd> x(N);
                for (uint32_t m = 0; m < N; ++m) {
                    const uint32_t l = local(ps, m), out = m & ~global(ps, (1u << tb) - 1);
                    uint32_t s = 0;
                    for (int b = 0; b < tb; ++b) if ((l >> b) & 1) s ^= pr.perms[u.perm].limg[b];
                    for (int b = 0; b < n; ++b) if ((out >> b) & 1) s ^= pr.perms[u.perm].oimg[b];
                    if (s >> tb) bad("perm", m, s);
                    x[m] = v[out | global(ps, s)];
                }
                v.swap(x);
            }
        }
        if (low < 0 || low + kb > tb || ps.s + w > n || (ps.s > lowbits && ps.s < tb && ps.s + w != n)) bad("arrangement", low, ps.s);
        for (int b = 0; b < kb; ++b)
            if ((u.hm >> b) & 1) {
                const uint32_t bit = global(ps, 1u << (low + b));
                for (uint32_t m = 0; m < N; ++m)
                    if (!(m & bit)) {
                        const cd x = v[m], y = v[m | bit];
                        v[m] = x + y;
                        v[m | bit] = x - y;
                    }
            }
        scale(v, u.shift, fixed);
    };
    std::vector<std::vector<cd>> psi(R);
    std::vector<cd> v(N, 0.0);
    v[0] = 1;
    int last = -1;
    for (const SPass &ps : pr.fwd) {
        low = ps.load_low;
        if (low == 0 && tb > kb) bad("load", low, 0);
        for (int o = 0; o < ps.nops; ++o) {
            const UOp &u = pr.ops[ps.op_begin + o];
            move(v, ps, u);
            if (u.run < 0) continue;
            if (u.run != last + 1) bad("run order", u.run, last);
            last = u.run;
            scale(v, u.rshift, fixed);
            double nrm = 0;
            for (uint32_t m = 0; m < N; ++m) nrm += std::norm(v[m] *= member_factor(pr.members, pr.runs[u.run], th, m));
            if (std::fabs(nrm - 1) > 1e-9) bad("norm", u.run, (long)(nrm * 1e6));
            psi[u.run] = v;
        }
        scale(v, ps.shift, fixed);
    }
    if (last != R - 1) bad("forward end", last, R);
    std::vector<cd> eta(N, 0.0);
    double E = 0;
    for (const DevTerm &t : pr.terms)
        for (uint32_t m = 0; m < N; ++m) {
            const uint32_t s = m ^ (uint32_t)t.x;
            eta[m] += t.coeff * std::pow(cd(0, 1), (t.ny + 2 * (__builtin_popcount(s & (uint32_t)t.z) & 1)) & 3) * v[s];
        }
    for (uint32_t m = 0; m < N; ++m) E += std::real(std::conj(v[m]) * eta[m]);
    std::vector<cd> Lm((size_t)P * P, 0.0), p(N);
    std::vector<double> sig(P, 0.0), ctrl(P, 1.0), grad(P, 0.0);
    auto ip_of = [&](const SPass &ps, const SIp &ip) {  // the kernel's split: the thread's own bit, or an index bit
        const int th = ip.src >= 8 ? ip.src - 8 : -1;
        const uint32_t own = ip.src == 0 ? 0u : global(ps, 1u << (th < 0 ? low + ip.src - 1 : (th < low ? th : th + kb)));
        if ((own | ip.z) != ip.zall || (own && ip.z)) bad("parameter bits", ip.zall, own);
        cd s = 0;
        for (uint32_t m = 0; m < N; ++m) s += ((m & (own | ip.z)) != 0) != (ip.sgn < 0) ? -p[m] : p[m];
        return s;
    };
    auto walk = [&](std::vector<cd> b, int col, int run) {
        const size_t p0 = run == R ? 0 : pr.entry[run].pass;
        for (size_t k = p0; k < pr.bwd.size(); ++k) {
            const SPass &ps = pr.bwd[k];
            low = ps.load_low;
            const bool st = run < R && k == p0;
            for (int o = st ? pr.entry[run].op : 0; o < ps.nops; ++o) {
                const UOp &u = pr.ops[ps.op_begin + o];
                const bool own = st && o == pr.entry[run].op;
                if (own) low = pr.entry[run].low;
                else move(b, ps, u);
                if (own && u.run != run) bad("entry", run, u.run);
                if (u.run < 0) continue;
                if (low == 0 && tb > kb) bad("run in block 0", u.run, 0);
                if (!own) scale(b, u.rshift, fixed);
                const Run &rn = pr.runs[u.run];
                for (uint32_t m = 0; m < N; ++m) p[m] = std::conj(psi[u.run][m]) * b[m];
                for (int q = 0; q < rn.ip_count; ++q) {
                    const cd x = ip_of(ps, pr.ips[rn.ip_begin + q]);
                    const int i = rn.ip_first + q;
                    if (run == R) grad[i] = -std::imag(x);
                    else if (i < col) Lm[(size_t)i * P + col] = 0.25 * x;
                }
                if (own) { cd s = 0; for (const cd &x : p) s += x; sig[col] = std::real(s); }
                for (uint32_t m = 0; m < N; ++m) b[m] *= std::conj(member_factor(pr.members, rn, th, m));
            }
            scale(b, ps.shift, fixed);
        }
    };
    for (int r = 0; r < R; ++r)
        for (int c = 0; c < pr.runs[r].ip_count; ++c) {
            const SIp &ip = pr.ips[pr.runs[r].ip_begin + c];
            std::vector<cd> b(N);
            for (uint32_t m = 0; m < N; ++m) b[m] = ((m & ip.zall) != 0) != (ip.sgn < 0) ? -psi[r][m] : psi[r][m];
            walk(b, pr.runs[r].ip_first + c, r);
        }
    walk(eta, P, R);
    std::printf("passes %d %d\n", (int)pr.fwd.size(), (int)pr.bwd.size());
    print_all(E, grad, sig, ctrl, Lm, P, R);
    return 0;
}

static int onchip(const std::vector<qng_gate> &gates, const std::vector<uint64_t> &masks, const std::vector<qng_pauli> &terms,
                  const std::vector<double> &th, int n, int P, int kb, int cl, bool fixed) {
    Program pr;
    build_program(gates, masks, terms, n, kb, cl, fixed, pr);
    for (const Run &r : pr.runs) if (r.khalf > kTableHalf) bad("factor", r.khalf, 0);
    const uint32_t N = 1u << pr.nE;
    const int R = (int)pr.runs.size();
    auto factor = [&](int r, uint32_t m) {
        cd f = std::pow(0.5, 0.5 * pr.runs[r].khalf);
        for (int k = 0; k < pr.runs[r].mem_count; ++k) {
            const Member &e = pr.members[pr.runs[r].mem_begin + k];
            const int par = __builtin_popcount(m & e.z) & 1;
            const double lam = par ? -e.sgn : e.sgn;
            if (e.kind == 2) { if (par) f *= cd(0, -1); continue; }
            if ((m & e.ctrl) != e.cval) continue;
            f *= e.kind == 1 ? cd(lam) : cd(std::cos(th[e.param] / 2), -lam * std::sin(th[e.param] / 2));
        }
        return f;
    };
    int low = pr.start0;
    auto move = [&](std::vector<cd> &v, const UOp &u) {
        if (u.low >= 0) {
            low = u.low;
            if (u.perm >= 0) {
                std::vector<cd> w(N);
                for (uint32_t m = 0; m < N; ++m) {
                    uint32_t s = 0;
                    for (int b = 0; b < 16; ++b) if ((m >> b) & 1) s ^= pr.perms[u.perm].img[b];
                    if (s >= N) bad("perm", m, s);
                    w[m] = v[s];
                }
                v.swap(w);
            }
        }
        if (low + kb > pr.nE || (low + kb > pr.nE - cl && low != pr.nE - kb)) bad("arrangement", low, cl);
        for (int b = 0; b < kb; ++b)
            if ((u.hm >> b) & 1)
                for (uint32_t m = 0; m < N; ++m)
                    if (!((m >> (low + b)) & 1)) {
                        const cd x = v[m], y = v[m | (1u << (low + b))];
                        v[m] = x + y;
                        v[m | (1u << (low + b))] = x - y;
                    }
        scale(v, u.shift, fixed);
    };
    std::vector<std::vector<cd>> psi(R);
    std::vector<cd> v(N, 0.0);
    v[0] = 1;
    int last = -1;
    for (const UOp &u : pr.fwd) {
        move(v, u);
        if (u.run < 0) continue;
        if (u.run != last + 1) bad("run order", u.run, last);
        last = u.run;
        if (low != pr.runs[u.run].low) bad("run arrangement", low, pr.runs[u.run].low);
        double nrm = 0;
        for (uint32_t m = 0; m < N; ++m) nrm += std::norm(v[m] *= factor(u.run, m));
        if (std::fabs(nrm - 1) > 1e-9) bad("norm", u.run, (long)(nrm * 1e6));
        psi[u.run] = v;
    }
    if (last != R - 1 || low != pr.end_low) bad("forward end", last, low);
    std::vector<cd> eta(N, 0.0);
    double E = 0;
    for (const DevTerm &t : pr.terms)
        for (uint32_t m = 0; m < N; ++m) {
            const uint32_t s = m ^ (uint32_t)t.x;
            cd f = std::pow(cd(0, 1), (t.ny + 2 * (__builtin_popcount(s & (uint32_t)t.z) & 1)) & 3);
            eta[m] += t.coeff * f * v[s];
        }
    for (uint32_t m = 0; m < N; ++m) E += std::real(std::conj(v[m]) * eta[m]);
    // a parameter's inner product read off p as the column kernel does: thread index and own bits
    auto ip_of = [&](const Ip &ip, int L, const std::vector<cd> &p) {
        cd s = 0;
        for (uint32_t m = 0; m < N; ++m) {
            const uint32_t t = (m & ((1u << L) - 1)) | ((m >> (L + kb)) << L), k = (m >> L) & ((1u << kb) - 1);
            if ((t & ip.ctrl) != ip.cval || !((ip.incl16 >> k) & 1)) continue;
            const int neg = (__builtin_popcount(t & ip.z) & 1) ^ ((ip.sign16 >> k) & 1) ^ (ip.sgn < 0);
            s += neg ? -p[m] : p[m];
        }
        return s;
    };
    std::vector<cd> Lm((size_t)P * P, 0.0), p(N);
    std::vector<double> sig(P, 0.0), ctrl(P, 0.0), grad(P, 0.0);
    std::vector<int> seen(P, 0);
    for (int r0 = 0; r0 < R; ++r0)
        for (int c = 0; c < pr.runs[r0].ip_count; ++c) {
            const Ip &me = pr.ips[pr.runs[r0].ip_begin + c];
            const int j = pr.runs[r0].ip_first + c;
            if (pr.members[pr.runs[r0].mem_begin].kind == 0 && pr.members[pr.runs[r0].mem_begin].param != pr.runs[r0].ip_first)
                bad("parameter order", j, r0);
            ++seen[j];
            const int L0 = pr.runs[r0].low;
            std::vector<cd> b(N);
            for (uint32_t m = 0; m < N; ++m) {
                const uint32_t t = (m & ((1u << L0) - 1)) | ((m >> (L0 + kb)) << L0), k = (m >> L0) & ((1u << kb) - 1);
                const bool on = (t & me.ctrl) == me.cval && ((me.incl16 >> k) & 1);
                const int neg = (__builtin_popcount(t & me.z) & 1) ^ ((me.sign16 >> k) & 1) ^ (me.sgn < 0);
                b[m] = on ? (neg ? -psi[r0][m] : psi[r0][m]) : cd(0);
            }
            bool first = true;
            low = L0;
            for (size_t o = pr.bwd_entry[r0]; o < pr.bwd.size(); ++o) {
                const UOp &u = pr.bwd[o];
                if (!first) move(b, u);
                first = false;
                if (u.run < 0) continue;
                const Run &rn = pr.runs[u.run];
                if (low != rn.low) bad("walk arrangement", low, rn.low);
                for (uint32_t m = 0; m < N; ++m) p[m] = std::conj(psi[u.run][m]) * b[m];
                for (int q = 0; q < rn.ip_count; ++q) {
                    const Ip &ip = pr.ips[rn.ip_begin + q];
                    const int i = rn.ip_first + q;
                    if (i < j) Lm[(size_t)i * P + j] = 0.25 * ip_of(ip, rn.low, p);
                    if (i == j) ctrl[j] = std::real(ip_of(ip, rn.low, p));
                }
                if (u.run == r0) { cd s = 0; for (const cd &x : p) s += x; sig[j] = std::real(s); }
                for (uint32_t m = 0; m < N; ++m) b[m] *= std::conj(factor(u.run, m));
            }
        }
    for (int j = 0; j < P; ++j) if (seen[j] != 1) bad("parameter", j, seen[j]);
    low = pr.end_low;
    for (const UOp &u : pr.bwd) {
        move(eta, u);
        if (u.run < 0) continue;
        const Run &rn = pr.runs[u.run];
        for (uint32_t m = 0; m < N; ++m) p[m] = std::conj(psi[u.run][m]) * eta[m];
        for (int q = 0; q < rn.ip_count; ++q) {
            const Ip &ip = pr.ips[rn.ip_begin + q];
            grad[rn.ip_first + q] = -std::imag(ip_of(ip, rn.low, p));
        }
        for (uint32_t m = 0; m < N; ++m) eta[m] *= std::conj(factor(u.run, m));
    }
    print_all(E, grad, sig, ctrl, Lm, P, R);
    return 0;
}

int main() {
    int n, P, G, T, kb, cl, tb, lowbits;
    if (std::scanf("%d %d %d %d %d %d %d %d", &n, &P, &G, &T, &kb, &cl, &tb, &lowbits) != 8) return 2;
    std::vector<qng_gate> gates(G);
    std::vector<uint64_t> masks(2 * G);
    for (int g = 0; g < G; ++g) {
        unsigned long long x, z;
        if (std::scanf("%d %d %d %d %llu %llu", &gates[g].kind, &gates[g].q0, &gates[g].q1, &gates[g].param, &x, &z) != 6) return 2;
        masks[2 * g] = x;
        masks[2 * g + 1] = z;
    }
    std::vector<qng_pauli> terms(T);
    for (qng_pauli &t : terms) {
        unsigned long long x, z;
        if (std::scanf("%lf %llu %llu", &t.coeff, &x, &z) != 3) return 2;
        t.xmask = x;
        t.zmask = z;
    }
    std::vector<double> th(P);
    for (double &t : th) if (std::scanf("%lf", &t) != 1) return 2;
    for (const bool fixed : {false, true}) {
        const int rc = tb > 0 ? stream(gates, terms, th, n, P, kb, tb, lowbits, fixed) : onchip(gates, masks, terms, th, n, P, kb, cl, fixed);
        if (rc) return rc;
    }
    std::printf("ok\n");
    return 0;
}
