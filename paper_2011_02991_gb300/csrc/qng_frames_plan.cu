// Host planner of the diagonal-frame path: one circuit -> runs of diagonal gates, the transitions
// between them, and the steps a CTA takes through them (qng_frames.h).
//
// The frame of qubit q is a one-qubit Clifford C_q with psi = (C_1 x C_2 x ...) v for the stored vector
// v. It is kept as the signed Paulis C_q^dag X C_q and C_q^dag Z C_q: a gate's generator on qubit q
// acts on v through these images.
#include <algorithm>
#include <cstdlib>

#include "qng_frames.h"

namespace qng {
namespace frames {

namespace {

enum { PX = 1, PY = 2, PZ = 3 };  // Pauli labels
struct SP { int p, s; };          // signed Pauli

struct Frame {
    SP x{PX, 1}, z{PZ, 1};
    SP y() const {  // Y = i X Z: the product of the images, i P Q = (+-) R for P != Q
        // i X Z = Y, i Z Y = X, i Y X = Z; the other order gives a minus sign
        const int a = x.p, b = z.p;
        const int r = 6 - a - b;  // the third label
        const bool pos = (a == PX && b == PZ) || (a == PZ && b == PY) || (a == PY && b == PX);
        return SP{r, x.s * z.s * (pos ? 1 : -1)};
    }
    SP image(int axis) const { return axis == kAxisX ? x : (axis == kAxisY ? y() : z); }
};

SP conj_h(SP a) { return a.p == PY ? SP{PY, -a.s} : SP{a.p == PX ? PZ : PX, a.s}; }             // H P H
SP conj_sdg(SP a) { return a.p == PX ? SP{PY, -a.s} : (a.p == PY ? SP{PX, a.s} : a); }          // S^dag P S

// Linear map of index bits, as the images of the basis vectors.
struct Lin {
    uint32_t img[kMaxQubits];
    Lin() { for (int b = 0; b < kMaxQubits; ++b) img[b] = 1u << b; }
    // mask z' with parity(m & z') = parity(A m & z)
    uint32_t pull(uint32_t z) const {
        uint32_t r = 0;
        for (int b = 0; b < kMaxQubits; ++b) r |= (uint32_t)(__builtin_popcount(img[b] & z) & 1) << b;
        return r;
    }
    Lin inverse() const {
        uint32_t a[kMaxQubits];
        Lin inv;
        for (int b = 0; b < kMaxQubits; ++b) a[b] = img[b];
        // column operations: reduce a to the identity, the same operations on inv
        for (int b = 0; b < kMaxQubits; ++b) {
            int p = b;
            while (!((a[p] >> b) & 1)) ++p;
            std::swap(a[p], a[b]);
            std::swap(inv.img[p], inv.img[b]);
            for (int k = 0; k < kMaxQubits; ++k)
                if (k != b && ((a[k] >> b) & 1)) { a[k] ^= a[b]; inv.img[k] ^= inv.img[b]; }
        }
        return inv;
    }
};

struct Stage {
    bool perm = false;
    uint32_t h = 0;  // Hadamards (perm = false)
    Lin map;         // new index of old index m is map(m) (perm = true)
    std::vector<std::pair<int, int>> cnots;  // the gates of the map, (control, target)
};

struct Builder {
    std::vector<Frame> fr;
    std::vector<std::vector<Member>> run_members;  // closed runs and, last, the open one
    std::vector<std::vector<Stage>> tau;           // tau[r]: the transition before run r

    explicit Builder(int n) : fr(n), run_members(1), tau(1) {}

    std::vector<Member> &open() { return run_members.back(); }
    std::vector<Stage> &otau() { return tau.back(); }
    void close() {
        run_members.emplace_back();
        tau.emplace_back();
    }
    bool open_touches(uint32_t mask) {
        for (const Member &m : open()) if ((m.z | m.ctrl) & mask) return true;
        return false;
    }
    // S^dag on qubit q of the vector as it is at the end of the open transition: into the run before
    // it, as a parity of that run's index. False if a Hadamard in between does not commute with it.
    bool sdg_before_open(int q) {
        uint32_t z = 1u << q;
        for (int s = (int)otau().size() - 1; s >= 0; --s) {
            const Stage &st = otau()[s];
            if (st.perm) z = st.map.pull(z);
            else if (st.h & z) return false;
        }
        if (run_members.size() == 1) return true;  // |0...0>: parity 0
        run_members[run_members.size() - 2].push_back(Member{2, -1, z, 0, 0, 1});
        return true;
    }
    // Make the images of (qubit, axis) requirements Z-type.
    void diagonalise(const std::vector<std::pair<int, int>> &req) {
        uint32_t need = 0;
        for (auto &r : req) if (fr[r.first].image(r.second).p != PZ) need |= 1u << r.first;
        if (!need) return;
        if (open_touches(need)) close();
        for (auto &r : req) {
            const int q = r.first;
            if (!((need >> q) & 1)) continue;
            if (fr[q].image(r.second).p == PY) {
                if (!sdg_before_open(q)) {
                    // the S^dag has to come between two Hadamards of this transition: a run of its own
                    close();
                    run_members[run_members.size() - 2].push_back(Member{2, -1, 1u << q, 0, 0, 1});
                }
                fr[q].x = conj_sdg(fr[q].x);
                fr[q].z = conj_sdg(fr[q].z);
            }
            if (otau().empty() || otau().back().perm) otau().emplace_back();
            otau().back().h ^= 1u << q;
            fr[q].x = conj_h(fr[q].x);
            fr[q].z = conj_h(fr[q].z);
        }
    }
    void rotation(int param, const std::vector<std::pair<int, int>> &req, int control) {
        std::vector<std::pair<int, int>> all(req);
        if (control >= 0) all.push_back({control, kAxisZ});
        diagonalise(all);
        Member m{0, param, 0, 0, 0, 1};
        for (auto &r : req) {
            m.z |= 1u << r.first;
            m.sgn *= fr[r.first].image(r.second).s;
        }
        if (control >= 0) {  // acts where the control is 1: the Z image's eigenvalue -1
            m.ctrl = 1u << control;
            m.cval = fr[control].z.s > 0 ? m.ctrl : 0;
        }
        open().push_back(m);
    }
    // controlled Pauli (axis on the target) as a diagonal sign
    void controlled_sign(int c, int t, int axis) {
        Member m{1, -1, 1u << t, 1u << c, 0, fr[t].image(axis).s};
        m.cval = fr[c].z.s > 0 ? m.ctrl : 0;
        open().push_back(m);
    }
    // CNOT c -> t; touched: the qubits that it and the CNOTs after it in its stretch join it with
    void cnot(int c, int t, uint32_t touched) {
        if (fr[c].z.p == PZ && fr[t].x.p == PZ) { controlled_sign(c, t, kAxisX); return; }
        // Frames whose Z and X images are Z and X: for all of the CNOTs to come at once, so that a ladder is one
        // index permutation behind one transition and at most one run of S^dag (a CNOT at a time, a ladder on n
        // qubits cut n - 1 runs without a parameter: 12 qubits, 16 x [Ry, CNOT ladder], 192 runs for 32 now)
        std::vector<std::pair<int, int>> req;
        for (int q = 0; q < (int)fr.size(); ++q) if ((touched >> q) & 1) req.push_back({q, kAxisZ});
        diagonalise(req);
        for (auto &r : req) {
            const int q = r.first;
            if (fr[q].x.p != PY) continue;
            // an S^dag turns the X image back to X: into the run before where nothing of the open one asks for it
            if (!open().empty() || !sdg_before_open(q)) open().push_back(Member{2, -1, 1u << q, 0, 0, 1});
            fr[q].x = conj_sdg(fr[q].x);
            fr[q].z = conj_sdg(fr[q].z);
        }
        if (!open().empty()) close();
        if (otau().empty() || !otau().back().perm) { otau().emplace_back(); otau().back().perm = true; }
        Lin &A = otau().back().map;
        for (int b = 0; b < kMaxQubits; ++b) A.img[b] ^= ((A.img[b] >> c) & 1u) << t;
        otau().back().cnots.push_back({c, t});
        // the frames of c and t are Paulis X^a Z^b: X_c -> X_c X_t, Z_t -> Z_c Z_t
        fr[t].z.s *= fr[c].z.s;
        fr[c].x.s *= fr[t].x.s;
    }
};

std::vector<std::pair<int, int>> string_req(uint64_t x, uint64_t z, int n) {
    std::vector<std::pair<int, int>> r;
    for (int q = 0; q < n; ++q) {
        const int hx = (int)((x >> q) & 1), hz = (int)((z >> q) & 1);
        if (hx || hz) r.push_back({q, hx ? (hz ? kAxisY : kAxisX) : kAxisZ});
    }
    return r;
}

// The circuit's gates, in order, into runs and transitions.
void walk_gates(const std::vector<qng_gate> &gates, const std::vector<uint64_t> &masks, int n, Builder &B) {
    size_t stretch = 0, stretch_end = 0;
    std::vector<uint32_t> touched;
    for (size_t gi = 0; gi < gates.size(); ++gi) {
        const qng_gate &g = gates[gi];
        Frame *f = (g.q0 >= 0 && g.q0 < n) ? &B.fr[g.q0] : nullptr;
        switch (g.kind) {
        case QNG_GATE_RX: B.rotation(g.param, {{g.q0, kAxisX}}, -1); break;
        case QNG_GATE_RY: B.rotation(g.param, {{g.q0, kAxisY}}, -1); break;
        case QNG_GATE_RZ: B.rotation(g.param, {{g.q0, kAxisZ}}, -1); break;
        case QNG_GATE_CRX: B.rotation(g.param, {{g.q1, kAxisX}}, g.q0); break;
        case QNG_GATE_CRY: B.rotation(g.param, {{g.q1, kAxisY}}, g.q0); break;
        case QNG_GATE_CRZ: B.rotation(g.param, {{g.q1, kAxisZ}}, g.q0); break;
        case QNG_GATE_RP: B.rotation(g.param, string_req(masks[2 * gi], masks[2 * gi + 1], n), -1); break;
        case QNG_GATE_CRP: B.rotation(g.param, string_req(masks[2 * gi], masks[2 * gi + 1], n), g.q0); break;
        case QNG_GATE_X: f->z.s = -f->z.s; break;
        case QNG_GATE_Y: f->x.s = -f->x.s; f->z.s = -f->z.s; break;
        case QNG_GATE_Z: f->x.s = -f->x.s; break;
        case QNG_GATE_H: std::swap(f->x, f->z); break;
        case QNG_GATE_CZ:
            B.diagonalise({{g.q0, kAxisZ}, {g.q1, kAxisZ}});
            B.controlled_sign(g.q0, g.q1, kAxisZ);
            break;
        case QNG_GATE_CNOT:
            if (gi >= stretch_end) {  // per CNOT, the qubits that it and those after it in the stretch join it with
                uint32_t joined[kMaxQubits];
                for (int q = 0; q < n; ++q) joined[q] = 1u << q;
                stretch = stretch_end = gi;
                while (stretch_end < gates.size() && gates[stretch_end].kind == QNG_GATE_CNOT) ++stretch_end;
                touched.resize(stretch_end - gi);
                for (size_t k = stretch_end; k-- > gi;) {
                    const uint32_t m = joined[gates[k].q0] | joined[gates[k].q1];
                    for (int q = 0; q < n; ++q) if ((m >> q) & 1) joined[q] = m;
                    touched[k - gi] = m;
                }
            }
            B.cnot(g.q0, g.q1, touched[gi - stretch]);
            break;
        default: break;
        }
    }
}

// The Hamiltonian in the final frame, terms grouped by X mask.
std::vector<DevTerm> final_terms(const std::vector<qng_pauli> &terms, int n, const Builder &B) {
    std::vector<DevTerm> out;
    for (const qng_pauli &t : terms) {
        DevTerm d = {};
        d.coeff = t.coeff;
        for (int q = 0; q < n; ++q) {
            const int hx = (int)((t.xmask >> q) & 1), hz = (int)((t.zmask >> q) & 1);
            if (!hx && !hz) continue;
            const SP im = B.fr[q].image(hx ? (hz ? kAxisY : kAxisX) : kAxisZ);
            if (im.s < 0) d.coeff = -d.coeff;
            if (im.p != PZ) d.x |= 1ull << q;
            if (im.p != PX) d.z |= 1ull << q;
        }
        d.ny = __builtin_popcountll(d.x & d.z) & 3;
        out.push_back(d);
    }
    std::stable_sort(out.begin(), out.end(), [](const DevTerm &a, const DevTerm &b) { return a.x < b.x; });
    return out;
}

}  // namespace

void build_program(const std::vector<qng_gate> &gates, const std::vector<uint64_t> &masks,
                   const std::vector<qng_pauli> &terms, int n, int kb, int cl, bool fixed, Program &out) {
    out = Program();
    out.n = n;
    out.kb = kb;
    const int nE = out.nE = std::max(n, kb);
    Builder B(n);
    walk_gates(gates, masks, n, B);
    // Without members left, a last transition that holds Hadamards still needs a run to carry their
    // normalisation; one of permutations alone, or an empty one, does not.
    bool last_h = false;
    for (const Stage &s : B.otau()) last_h = last_h || (!s.perm && s.h);
    std::vector<Stage> tail;
    if (B.open().empty() && !last_h) {
        tail = B.otau();
        B.run_members.pop_back();
        B.tau.pop_back();
    }
    const int R = (int)B.run_members.size();

    // arrangements: kb consecutive index bits; blocks within a CTA's own bits, the last one flush with
    // their top, and one at the very top for the distributed bits (local or not, nl >= kb)
    const int nl = nE - cl;
    std::vector<int> lows;
    for (int lo = 0; lo + kb <= nl; lo += kb) lows.push_back(lo);
    if (nl % kb) lows.push_back(nl - kb);
    if (cl > 0) lows.push_back(nE - kb);
    auto block_of = [&](int q) {
        for (int lo : lows) if (q >= lo && q < lo + kb) return lo;
        return lows.back();
    };

    // elementary steps in circuit order
    struct Step { int kind, low0, low1, perm; uint32_t h; int run; };
    std::vector<Step> el;
    std::vector<Lin> maps;
    int cur = -1;  // arrangement (decided by the first step that needs one)
    auto blocks_in = [&](uint32_t h) {
        std::vector<int> b;
        for (int q = 0; q < nE; ++q) if ((h >> q) & 1) { int lo = block_of(q); if (std::find(b.begin(), b.end(), lo) == b.end()) b.push_back(lo); }
        std::sort(b.begin(), b.end());
        return b;
    };
    auto first_need = [&](const std::vector<Stage> &t, size_t s, int dflt) {
        for (; s < t.size(); ++s)
            if (!t[s].perm && t[s].h) {
                auto b = blocks_in(t[s].h);
                return (std::find(b.begin(), b.end(), dflt) != b.end()) ? dflt : b.front();
            }
        return dflt;
    };
    auto emit_tau = [&](const std::vector<Stage> &t) {
        for (size_t s = 0; s < t.size(); ++s) {
            if (t[s].perm) {
                maps.push_back(t[s].map);
                const int to = first_need(t, s + 1, cur);
                el.push_back(Step{0, cur, to, (int)maps.size() - 1, 0, -1});
                cur = to;
            } else if (t[s].h) {
                std::vector<int> b = blocks_in(t[s].h);
                // the current arrangement first, then away from it in order
                if (cur != b.front() && (cur == b.back() || std::abs(cur - b.back()) < std::abs(cur - b.front())))
                    std::reverse(b.begin(), b.end());
                auto it = std::find(b.begin(), b.end(), cur);
                if (it != b.end()) std::rotate(b.begin(), it, it + 1);
                for (int lo : b) {
                    if (lo != cur) { el.push_back(Step{0, cur, lo, -1, 0, -1}); cur = lo; }
                    uint32_t h = 0;
                    for (int q = 0; q < nE; ++q) if (((t[s].h >> q) & 1) && block_of(q) == lo) h |= 1u << (q - lo);
                    el.push_back(Step{1, lo, lo, -1, h, -1});
                }
            }
        }
    };
    std::vector<int> had(R + 1, 0);  // Hadamards of the transition before run r (none after the last)
    for (int r = 0; r < R; ++r)
        for (const Stage &s : B.tau[r]) if (!s.perm) had[r] += __builtin_popcount(s.h);
    const int dflt = cl > 0 ? lows.front() : lows.back();
    cur = R > 0 ? first_need(B.tau[0], 0, dflt) : first_need(tail, 0, dflt);
    out.start0 = cur;
    for (int r = 0; r < R; ++r) {
        emit_tau(B.tau[r]);
        el.push_back(Step{2, cur, cur, -1, 0, r});
        Run run = {};
        run.low = cur;
        run.mem_begin = (int)out.members.size();
        run.mem_count = (int)B.run_members[r].size();
        run.ip_begin = (int)out.ips.size();
        run.ip_first = -1;
        run.simple = 1;
        run.khalf = table_half(had[r], fixed);
        const int L = cur;
        auto thr = [&](uint32_t m) { return (m & ((1u << L) - 1u)) | ((m >> (L + kb)) << L); };
        auto reg = [&](uint32_t m) { return (m >> L) & ((1u << kb) - 1u); };
        for (const Member &m : B.run_members[r]) {
            out.members.push_back(m);
            if (m.kind != 0) continue;
            if (run.ip_first < 0) run.ip_first = m.param;
            Ip ip = {};
            ip.z = (uint16_t)thr(m.z);
            ip.ctrl = (uint16_t)thr(m.ctrl);
            ip.cval = (uint16_t)thr(m.cval);
            ip.sgn = (int16_t)m.sgn;
            ip.zreg = (uint16_t)reg(m.z);
            ip.all16 = (uint16_t)((1u << (1 << kb)) - 1u);
            for (uint32_t k = 0; k < (1u << kb); ++k) {
                if ((k & reg(m.ctrl)) == reg(m.cval)) ip.incl16 |= (uint16_t)(1u << k);
                if (__builtin_popcount(k & reg(m.z)) & 1) ip.sign16 |= (uint16_t)(1u << k);
            }
            if (m.ctrl || (ip.zreg & (ip.zreg - 1))) run.simple = 0;
            out.ips.push_back(ip);
        }
        run.ip_count = (int)out.ips.size() - run.ip_begin;
        if (run.ip_first < 0) run.ip_first = 0;
        out.runs.push_back(run);
    }
    emit_tau(tail);
    out.end_low = cur;

    // fuse into steps: exchange, then Hadamards, then a run. Halvings keep the vector within sqrt 2 of unit
    // norm: floor(k / 2) after k Hadamards of a transition, unless its run's factor takes all of them.
    auto fuse = [&](const std::vector<Step> &v, bool back, std::vector<UOp> &ops) {
        int k = 0, tr = back ? R : 0;  // the transition that the next steps belong to
        UOp u{-1, 0, 0, 0, -1, -1};
        int stage = 0;  // 0 nothing yet, 1 exchange, 2 Hadamards
        auto flush = [&]() { ops.push_back(u); u = UOp{-1, 0, 0, 0, -1, -1}; stage = 0; };
        for (const Step &s : v) {
            if (s.kind == 0) {
                if (stage > 0) flush();
                u.low = (int16_t)(back ? s.low0 : s.low1);
                if (s.perm >= 0) {
                    // gather: forward new[m] = old[A^-1 m], adjoint new[m] = old[A m]
                    const Lin A = back ? maps[s.perm] : maps[s.perm].inverse();
                    Perm p;
                    std::copy(A.img, A.img + 16, p.img);
                    u.perm = (int32_t)out.perms.size();
                    out.perms.push_back(p);
                }
                stage = 1;
            } else if (s.kind == 1) {
                if (stage > 1) flush();
                u.hm = (int16_t)s.h;
                const int k1 = k + __builtin_popcount(s.h);
                u.shift = (int16_t)(table_half(had[tr], fixed) == had[tr] ? 0 : k1 / 2 - k / 2);
                k = k1;
                stage = 2;
            } else {
                u.run = s.run;
                if (back) out.bwd_entry[s.run] = (int32_t)ops.size();
                flush();
                k = 0;
                tr = back ? s.run : s.run + 1;
            }
        }
        if (stage > 0) flush();
    };
    out.bwd_entry.assign(R, -1);
    fuse(el, false, out.fwd);
    std::vector<Step> rel(el.rbegin(), el.rend());
    // the walk ends at run 0 (what precedes it is never needed)
    std::vector<Step> cut;
    for (const Step &s : rel) {
        cut.push_back(s);
        if (s.kind == 2 && s.run == 0) break;
    }
    if (R > 0) fuse(cut, true, out.bwd);

    out.terms = final_terms(terms, n, B);
}

// ------------------------------------------------------------------------------------------
// Streaming: vectors in global memory, passes over tiles of 2^tb amplitudes.
namespace {

struct Atom { int kind, q, c, run; };  // 0 Hadamard on q; 1 CNOT c -> q; 2 run

struct Window { int low, s, w; };
bool holds(const Window &W, int q) { return q < W.low || (q >= W.s && q < W.s + W.w); }

// The atoms of the list (those not done) that a pass over window W can execute: in order, each one
// whose pair qubit the window holds and that no skipped atom shares a qubit with.
std::vector<int> executable(const std::vector<Atom> &at, const std::vector<uint8_t> &done, size_t from, const Window &W, int n) {
    std::vector<int> ex;
    uint32_t blocked = 0;
    for (size_t k = from; k < at.size() && blocked != (1u << n) - 1u; ++k) {
        if (done[k]) continue;
        const Atom &a = at[k];
        if (a.kind == 2) {
            if (blocked) break;
            ex.push_back((int)k);
            continue;
        }
        const uint32_t m = (1u << a.q) | (a.kind == 1 ? 1u << a.c : 0u);
        if (!(m & blocked) && holds(W, a.q)) ex.push_back((int)k);
        else blocked |= m;
    }
    return ex;
}

void pack_passes(const std::vector<Atom> &at, bool back, bool fixed, const std::vector<int> &had, StreamProgram &P,
                 std::vector<SPass> &out) {
    const int n = P.n, kb = P.kb, tb = P.tb;
    std::vector<Window> wins;
    wins.push_back(Window{P.low, P.low, tb - P.low});  // the lowest tb bits
    for (int s = tb; s < n; s += tb - P.low) wins.push_back(Window{P.low, std::min(s, n - (tb - P.low)), tb - P.low});
    std::vector<int> lows;
    for (int lo = 0; lo + kb <= tb; lo += kb) lows.push_back(lo);
    if (tb % kb) lows.push_back(tb - kb);
    auto block_of = [&](int b) {
        for (int lo : lows) if (b >= lo && b < lo + kb) return lo;
        return lows.back();
    };
    std::vector<uint8_t> done(at.size(), 0);
    size_t from = 0;
    // Hadamards since the last run, and halvings (fixed point: once three are due, at a run and at the end of a
    // pass): floor(k / 2) in all, the odd sqrt 1/2 is in the run's factor. Between them the vector grows to
    // 2^4.5 of its norm at most (two halvings due, an odd Hadamard, a block of four more). float32 halves after
    // each step of the transitions whose factor does not take it all
    int k = 0, halved = 0, tr = back ? (int)P.runs.size() : 0;
    auto due = [&]() { return table_half(had[tr], fixed) == had[tr] ? 0 : k / 2 - halved; };
    while (from < at.size()) {
        std::vector<int> best;
        Window W = wins[0];
        for (const Window &w : wins) {
            std::vector<int> ex = executable(at, done, from, w, n);
            if (ex.size() > best.size()) { best = ex; W = w; }
        }
        SPass ps = {};
        ps.run0 = -1;
        ps.s = W.s;
        ps.op_begin = (int32_t)P.ops.size();
        auto local = [&](int q) { return q < W.low ? q : q - W.s + W.low; };
        int cur = -1;
        UOp u{-1, 0, 0, 0, -1, -1};
        int stage = 0;
        auto flush = [&]() { if (stage) { P.ops.push_back(u); u = UOp{-1, 0, 0, 0, -1, -1}; stage = 0; } };
        auto goto_low = [&](int lo, int perm) {
            if (cur < 0 && perm < 0) { cur = lo; ps.load_low = lo; return; }
            if (cur < 0) { cur = lows.back(); ps.load_low = cur; }
            if (cur == lo && perm < 0) return;
            flush();
            u.low = (int16_t)lo;
            u.perm = perm;
            stage = 1;
            cur = lo;
        };
        for (size_t i = 0; i < best.size();) {
            const Atom &a = at[best[i]];
            if (a.kind == 0) {
                // over local bits; two on one qubit (with nothing on it between them) are two steps, as either
                // counts for the norm
                uint32_t h = 0;
                while (i < best.size() && at[best[i]].kind == 0 && !((h >> local(at[best[i]].q)) & 1)) h |= 1u << local(at[best[i++]].q);
                std::vector<int> bl;
                for (int b = 0; b < tb; ++b) if ((h >> b) & 1) { const int lo = block_of(b); if (!std::count(bl.begin(), bl.end(), lo)) bl.push_back(lo); }
                // the current block first, block 0 next, the others last: runs, loads and stores want their
                // low bits on the threads
                std::vector<int> ord;
                if (cur < 0) { if (*std::max_element(bl.begin(), bl.end()) > 0) ord.push_back(*std::max_element(bl.begin(), bl.end())); }
                else if (std::count(bl.begin(), bl.end(), cur)) ord.push_back(cur);
                if (std::count(bl.begin(), bl.end(), 0) && !std::count(ord.begin(), ord.end(), 0)) ord.push_back(0);
                for (int lo : bl) if (!std::count(ord.begin(), ord.end(), lo)) ord.push_back(lo);
                for (int lo : ord) {
                    if (cur < 0 && lo == 0) goto_low(lows.back(), -1);
                    goto_low(lo, -1);
                    uint32_t m = 0;
                    for (int b = 0; b < tb; ++b) if (((h >> b) & 1) && block_of(b) == lo) m |= 1u << (b - lo);
                    if (stage > 1) flush();
                    u.hm = (int16_t)m;
                    k += __builtin_popcount(m);
                    if (due() >= (fixed ? 3 : 1)) {
                        u.shift = (int16_t)due();
                        halved = k / 2;
                    }
                    stage = 2;
                }
            } else if (a.kind == 1) {
                Lin A;  // new index of old index m is A(m): the pass's CNOTs in the order they run
                while (i < best.size() && at[best[i]].kind == 1) {
                    const Atom &c = at[best[i++]];
                    for (int b = 0; b < kMaxQubits; ++b) A.img[b] ^= ((A.img[b] >> c.c) & 1u) << c.q;
                }
                const Lin inv = A.inverse();  // gather: new[m] = old[A^-1 m]
                SPerm p = {};
                for (int b = 0; b < n; ++b) {
                    uint32_t l = 0;
                    for (int q = 0; q < n; ++q) if (((inv.img[b] >> q) & 1) && holds(W, q)) l |= 1u << local(q);
                    if (holds(W, b)) p.limg[local(b)] = l;
                    else p.oimg[b] = l;
                }
                P.perms.push_back(p);
                goto_low(cur > 0 ? cur : lows.back(), (int)P.perms.size() - 1);
            } else {
                if (cur <= 0 && lows.back() > 0) goto_low(lows.back(), -1);
                else if (cur < 0) goto_low(lows.back(), -1);
                u.run = a.run;
                if (ps.run0 < 0) ps.run0 = a.run;
                stage = 3;
                if (back) {
                    P.entry[a.run] = SEntry{(int32_t)out.size(), (int32_t)P.ops.size() - ps.op_begin, cur, 0};
                    // parameters of the run: which of the thread's bits, if any, each one's qubit is here
                    Run &rn = P.runs[a.run];
                    rn.low = cur;
                    for (int x = 0; x < rn.ip_count; ++x) {
                        SIp &ip = P.ips[rn.ip_begin + x];
                        const int q = __builtin_ctz(ip.zall), lb = holds(W, q) ? local(q) : -1;
                        const int th = lb < cur ? lb : lb - kb;  // its bit of the thread index
                        ip.src = 0;
                        if (lb >= cur && lb < cur + kb) ip.src = (int16_t)(1 + lb - cur);
                        else if (lb >= 0 && th < 5 && th < tb - kb) ip.src = (int16_t)(8 + th);
                        ip.z = ip.src ? 0u : ip.zall;
                    }
                }
                u.rshift = (int16_t)due();
                flush();
                k = halved = 0;
                tr = back ? a.run : a.run + 1;
                ++i;
            }
        }
        if (cur <= 0 && lows.back() > 0) goto_low(lows.back(), -1);
        flush();
        ps.shift = due();
        halved = k / 2;
        ps.nops = (int32_t)P.ops.size() - ps.op_begin;
        out.push_back(ps);
        for (int x : best) done[x] = 1;
        while (from < at.size() && done[from]) ++from;
    }
}

}  // namespace

void build_stream(const std::vector<qng_gate> &gates, const std::vector<qng_pauli> &terms, int n, int kb, int tb, int low,
                  bool fixed, StreamProgram &out) {
    out = StreamProgram();
    out.n = n;
    out.kb = kb;
    out.tb = tb;
    out.low = low;
    // halves of the factor tables: the second window's first bit, so that (but for narrow windows) the thread's
    // bits at a run lie in one half
    out.hl = std::min(tb, n - 1);
    if (n > tb && n - (tb - low) < tb) out.hl = n - (tb - low);
    Builder B(n);
    walk_gates(gates, {}, n, B);
    bool last_h = false;
    for (const Stage &s : B.otau()) last_h = last_h || (!s.perm && s.h);
    std::vector<Stage> tail;
    if (B.open().empty() && !last_h) {
        tail = B.otau();
        B.run_members.pop_back();
        B.tau.pop_back();
    }
    const int R = (int)B.run_members.size();
    std::vector<int> had(R + 1, 0);
    std::vector<Atom> fwd;
    auto add_tau = [&](const std::vector<Stage> &t) {
        for (const Stage &s : t) {
            if (s.perm) for (auto &c : s.cnots) fwd.push_back(Atom{1, c.second, c.first, -1});
            else for (int q = 0; q < n; ++q) if ((s.h >> q) & 1) fwd.push_back(Atom{0, q, -1, -1});
        }
    };
    for (int r = 0; r < R; ++r) {
        add_tau(B.tau[r]);
        fwd.push_back(Atom{2, -1, -1, r});
        Run run = {};
        run.mem_begin = (int)out.members.size();
        run.mem_count = (int)B.run_members[r].size();
        run.ip_begin = (int)out.ips.size();
        run.ip_first = -1;
        for (const Stage &s : B.tau[r]) if (!s.perm) had[r] += __builtin_popcount(s.h);
        run.khalf = table_half(had[r], fixed);
        for (const Member &m : B.run_members[r]) {
            out.members.push_back(m);
            if (m.kind != 0) continue;
            if (run.ip_first < 0) run.ip_first = m.param;
            out.ips.push_back(SIp{m.z, m.z, (int16_t)m.sgn, 0});
        }
        run.ip_count = (int)out.ips.size() - run.ip_begin;
        if (run.ip_first < 0) run.ip_first = 0;
        out.runs.push_back(run);
    }
    add_tau(tail);
    std::vector<Atom> bwd;
    for (auto it = fwd.rbegin(); it != fwd.rend(); ++it) {
        bwd.push_back(*it);
        if (it->kind == 2 && it->run == 0) break;
    }
    out.entry.assign(R, SEntry{0, 0, 0, 0});
    pack_passes(fwd, false, fixed, had, out, out.fwd);
    if (out.fwd.empty()) out.fwd.push_back(SPass{low, tb - kb, 0, 0, -1, 0});  // no gate that moves |0...0>
    if (R > 0) pack_passes(bwd, true, fixed, had, out, out.bwd);
    out.terms = final_terms(terms, n, B);
}

}  // namespace frames
}  // namespace qng
