// Host-only probe of the diagonal-frame planner (qng_frames_plan.cu), built and run by
// tests/test_frames_host.py: reads a circuit with its Hamiltonian and angles, builds the program and
// executes it in float64 on the host, step by step as the kernels do (exchanges, permutations,
// Hadamards on a thread's own bits, runs), and prints
//   E <energy>, grad <P values>, L <re im> for i < j, sigma <P values>, ctrl <P values>
// Structural invariants are checked on the way ("bad <what>", exit 1).
// Input (stdin): n P G T kb cl, G lines "kind q0 q1 param xmask zmask", T lines "coeff x z", P angles.
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

int main() {
    int n, P, G, T, kb, cl;
    if (std::scanf("%d %d %d %d %d %d", &n, &P, &G, &T, &kb, &cl) != 6) return 2;
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
    Program pr;
    build_program(gates, masks, terms, n, kb, cl, pr);
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
    std::printf("E %.17g\n", E);
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
    std::printf("runs %d\n", R);
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
    std::printf("\nok\n");
    return 0;
}
