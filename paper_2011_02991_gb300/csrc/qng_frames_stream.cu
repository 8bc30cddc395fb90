// sm_103a kernels of the diagonal-frame path for one instance whose vectors lie in global memory
// (qng_frames.h, StreamProgram).
//
//   k_half    per run, the factor tables of the low and the high half of the index bits
//   k_stream  one pass over a vector (forward sweep) or over several columns (walk): each CTA loads a
//             tile of 2^tb amplitudes into registers, exchanges through shared memory, stores it back
//   k_sheff   H psi, <E> and |H psi|
//   k_sfinish integer sums to float64
//
// A walk takes one pass per run while two windows cover the index bits (complex64 to 24 qubits,
// complex128 to 22): the run sits between the Hadamards of the transition before and after it, all
// in one window, and the windows alternate. Per amplitude and pass a column moves one load and one store
// and reads its run's checkpoint, which the columns of a launch share through L2.
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <cstdint>
#include <type_traits>

#include "qng_frames.cuh"

namespace qng {
namespace frames {

// complex128 vectors are multiples of 2^-58 here: eight Hadamards then need no halving in between (they grow
// the vector by 2^4), and as every rounding is unbiased (see hash) a unit of 2^-58 on each component moves an
// inner product with a unit vector by no more.
constexpr int kUnit = 58;
// Inner products are sums of 2^-62: unit vectors, so no partial sum of products exceeds 1 in magnitude. What lies
// below the unit is kept as well and a warp's sum rounded once; what that leaves is a unit times 2^((n - 9)/2).
// 22 qubits, two-norm errors of gradient and g: 2.8e-15 and 4.4e-15 with every product rounded,
// 2.0e-15 and 4.2e-15 so (float64 on the gate-by-gate passes: 2.1e-15 and 4.4e-15); 17.58 and 17.83 ms. 26 qubits,
// gradient entries against the oracle: 7.0e-14, 1.3e-14 so (float64: 1.2e-14).
constexpr int kSumUnit = 62;
constexpr int kHalfThreads = 128;
constexpr int kRows = 32;  // parameters of a run kept in shared memory

// CTAs of NT threads with 2^KB amplitudes each per SM, that the registers are held to. complex64 vectors of 21
// qubits and more: 32 amplitudes a thread and 16 warps (24 qubits: 67 ms against 78 ms with 16 amplitudes
// and 32 warps, which exchange more often); smaller ones 16 amplitudes and 32 warps. complex128: 16 amplitudes,
// 16 warps.
template <class T> constexpr int ctas_per_sm(int kb, int nt) {
    return (sizeof(typename T::A) == 16 || kb == 5 ? 512 : 1024) / nt;
}

// ------------------------------------------------------------------------------------------
// One entry of a half table per thread. Members on one half's bits multiply its factor; a CZ across the
// halves is bilinear in its two bits: its linear parts go to the halves, the product to the mask. An
// S^dag of a parity p = p_lo xor p_hi is (-i)^p_lo (-i)^p_hi (-1)^(p_lo p_hi).
__global__ void __launch_bounds__(kHalfThreads) k_half(SWork w, int fix) {
    __shared__ int4 cs[kHalfThreads];
    __shared__ Member mem[kHalfThreads];
    grid_ready();
    const int r = blockIdx.x;
    const Run &rn = w.run[r];
    const uint32_t nlo = 1u << w.hl, nhi = 1u << (w.n - w.hl);
    const uint32_t e = blockIdx.y * kHalfThreads + threadIdx.x;
    const bool lo = e < nlo;
    const bool on = e < nlo + nhi;
    const uint32_t own = lo ? nlo - 1u : ~(nlo - 1u);       // this half's bits
    const uint32_t m = lo ? e : (e - nlo) << w.hl;          // index with the other half 0
    const int mem_count = rn.mem_count, mem_begin = rn.mem_begin;
    const int half = rn.khalf;
    longlong2 f = {1ll << 61, 0};
    if (lo) f.x = root_half(half);
    uint32_t mask = 0;
    for (int e0 = 0; e0 < mem_count; e0 += kHalfThreads) {
        __syncthreads();
        if (e0 + (int)threadIdx.x < mem_count) {
            const Member x = w.member[mem_begin + e0 + threadIdx.x];
            mem[threadIdx.x] = x;
            if (x.kind == 0) {
                const double th = w.theta[x.param];
                double s, c;
                if (!isfinite(th)) { *w.bad = 1; atomicCAS(w.status, 0, (int)QNG_ERR_ARG); }
                sincos(0.5 * th, &s, &c);
                if (blockIdx.y == 0) w.pctrl[x.param] = 1.0;
                cs[threadIdx.x] = rotation_pair(c, x.sgn > 0 ? -s : s);
            }
        }
        __syncthreads();
        const int ne = min(mem_count - e0, kHalfThreads);
        for (int q = 0; q < ne; ++q) {
            const Member &x = mem[q];
            const uint32_t z = x.z & own;
            const int par = __popc(m & z) & 1;
            if (x.kind == 0) {  // one qubit
                if (z) f = par ? mul<1>(f, cs[q]) : mul<0>(f, cs[q]);
            } else if (x.kind == 2) {
                if (par) f = longlong2{f.y, -f.x};
                if (!lo && par) mask ^= x.z & (nlo - 1u);
            } else {
                // (-1)^((c + nvc)(s + t)): c t + s c + nvc t + nvc s over the control bit c and target bit t
                const int nvc = x.cval ? 0 : 1, s = x.sgn < 0;
                const bool hc = x.ctrl & own, ht = z != 0;
                const int c = (m & x.ctrl) != 0;
                int neg = 0;
                if (hc && ht) neg = (c ^ nvc) & (s ^ par);
                else if (hc) neg = s & c;
                else if (ht) neg = nvc & par;
                if (hc != ht && lo) neg ^= nvc & s;
                if (!lo && hc != ht) {
                    if (hc && c) mask ^= x.z;
                    if (ht && par) mask ^= x.ctrl;
                }
                if (neg) f = longlong2{-f.x, -f.y};
            }
        }
    }
    if (!on) return;
    if (fix) {
        int4 *d = reinterpret_cast<int4 *>(lo ? w.lo : w.hi) + (size_t)r * (lo ? nlo : nhi) + (lo ? e : e - nlo);
        store_factor(d, f);
    } else {
        float2 *d = reinterpret_cast<float2 *>(lo ? w.lo : w.hi) + (size_t)r * (lo ? nlo : nhi) + (lo ? e : e - nlo);
        store_factor(d, f);
    }
    if (!lo) w.mask[(size_t)r * nhi + (e - nlo)] = mask;
}

// ------------------------------------------------------------------------------------------
// Tile-local exchange: as the on-chip kernels', over tb local bits in one CTA.
template <class T> __device__ __forceinline__ uint32_t sslot(uint32_t l) {
    return (l ^ ((l >> 4) & T::kSwz) ^ ((l >> 8) & T::kSwz)) * (uint32_t)sizeof(typename T::A);
}
// element g of an array of at most 4 GiB
template <typename E> __device__ __forceinline__ E &at(E *p, uint32_t g) {
    return *reinterpret_cast<E *>(reinterpret_cast<char *>(const_cast<typename std::remove_const<E>::type *>(p)) +
                                  (size_t)(g * (uint32_t)sizeof(E)));
}
template <int KB> __device__ __forceinline__ uint32_t tbase(uint32_t t, int low) {
    return ((t >> low) << (low + KB)) | (t & ((1u << low) - 1u));
}

template <class T, int KB, typename F>
__device__ __forceinline__ void slots_of(unsigned char *smem, uint32_t b0, const uint32_t (&st)[KB], F &&f) {
    uint32_t s = sslot<T>(b0), d[KB];
#pragma unroll
    for (int j = 0; j < KB; ++j) d[j] = sslot<T>(st[j]);
#pragma unroll
    for (int i = 0; i < (1 << KB); ++i) {
        f(i ^ (i >> 1), reinterpret_cast<typename T::A *>(smem + s));
        if (i + 1 < (1 << KB)) s ^= d[(i & 1) == 0 ? 0 : ((i & 2) == 0 ? 1 : ((i & 4) == 0 ? 2 : ((i & 8) == 0 ? 3 : KB - 1)))];
    }
}

// Rounding offsets of complex128 products: pseudo-random over the amplitudes (a hash of thread and tile,
// xor a constant per amplitude), uniform below one unit. Rounding to nearest would not do at these
// sizes: shallow circuits leave the state with few distinct values, each of which is rounded alike on
// all of its amplitudes, and the errors of 2^22 products add up instead of cancelling.
// x 2^-s, rounded by the dither's bits; s uniform over the launch
__device__ __forceinline__ void scale_down(longlong2 &x, int s, uint32_t dither) {
    if (s) {
        x.x = (x.x + (ll)(dither >> (32 - s))) >> s;
        x.y = (x.y + (ll)((dither * 5u) >> (32 - s))) >> s;
    }
}
__device__ __forceinline__ void scale_down(float2 &, int, uint32_t) {}

// -i eta, rounded by the dither
__device__ __forceinline__ longlong2 seed_dithered(double2 e, const SeedScale &up, uint32_t d) {
    return longlong2{__double2ll_rd(up(e.y) + (double)d * 0x1p-32), __double2ll_rd(-up(e.x) + (double)(d * 5u) * 0x1p-32)};
}
__device__ __forceinline__ float2 seed_dithered(float2 e, const SeedScale &, uint32_t) { return float2{e.y, -e.x}; }

// MIM: both parts of the metric's inner products. FWD: the forward sweep (one vector, checkpoints out).
template <class T, int MIM, int FWD, int KB, int NT>
__global__ void __launch_bounds__(NT, ctas_per_sm<T>(KB, NT)) k_stream(SWork w, SPass ps, int pass, int col0, int ncol, int flag) {
    constexpr int NA = 1 << KB;
    using A = typename T::A;
    using S = typename T::S;
    using Acc = typename T::Acc;
    extern __shared__ __align__(1024) unsigned char smem[];
    using Red = typename T::Red;
    __shared__ Red red[16][NT / 32][MIM ? 2 : 1];
    // the pass's steps and the parameters of its (first) run: read once, or each would wait on L2
    constexpr int kOpsMax = 48;
    __shared__ UOp ops_sh[kOpsMax];
    __shared__ SIp ips_sh[kRows];
    for (int x = threadIdx.x; x < min(ps.nops, kOpsMax); x += NT) ops_sh[x] = w.uop[ps.op_begin + x];
    if (!FWD && ps.run0 >= 0) {
        const Run &rn = w.run[ps.run0];
        for (int x = threadIdx.x; x < min(rn.ip_count, kRows); x += NT) ips_sh[x] = w.ip[rn.ip_begin + x];
    }
    grid_ready();
    const int slot = FWD ? col0 : (int)(blockIdx.x % (unsigned)ncol);
    const uint32_t tile = FWD ? blockIdx.x : blockIdx.x / (unsigned)ncol;
    const int wn = w.tb - w.low;  // window bits
    const uint32_t lowmask = (1u << w.low) - 1u;
    // global index of local index l: tile | spread(l), both linear
    const uint32_t gtile = ((tile & ((1u << (ps.s - w.low)) - 1u)) << w.low) | ((tile >> (ps.s - w.low)) << (ps.s + wn));
    auto spread = [&](uint32_t l) { return (l & lowmask) | ((l >> w.low) << ps.s); };
    const uint32_t t = threadIdx.x;
    const SCol me = FWD ? SCol{0, 0} : w.col[col0 + slot];
    const bool grad = !FWD && me.run == w.R;
    A *buf = reinterpret_cast<A *>(w.b) + ((size_t)slot << w.n);
    int low = ps.load_low, o = 0;
    A b[NA];
    // index of the thread's amplitude k: g0 + (k << gsh) (loads, stores and runs never use block 0, whose bits
    // may straddle the window's edge)
    uint32_t g0 = 0;
    int gsh = 0;
    auto set_g = [&]() {
        g0 = gtile | spread(tbase<KB>(t, low));
        gsh = low - w.low + ps.s;
    };
    auto gidx = [&](int k) { return g0 + ((uint32_t)k << gsh); };
    const uint32_t h0 = sizeof(A) == 16 ? hash(tile * NT + t) : 0u;
    auto dith = [&](int k) { return sizeof(A) == 16 ? (h0 ^ salt(k)) | 64u : 0u; };
    bool start = false;
    if (FWD) {
        set_g();
        if (flag & 1) {  // the first pass starts from |0...0>
#pragma unroll
            for (int k = 0; k < NA; ++k) b[k] = A{0, 0};
            if (g0 == 0) {
                if constexpr (sizeof(A) == 16) b[0].x = 1ll << kUnit;
                else b[0].x = 1.0f;
            }
        } else {
#pragma unroll
            for (int k = 0; k < NA; ++k) b[k] = at(buf, gidx(k));
        }
    } else {
        const SEntry en = grad ? SEntry{0, 0, ps.load_low, 0} : w.entry[me.run];
        start = !grad && en.pass == pass;
        if (start) {  // column j of run r starts as K_j Psi_r
            o = en.op;
            low = en.low;
            set_g();
            const Run &rn = w.run[me.run];
            const SIp &ip = w.ip[rn.ip_begin + me.col - rn.ip_first];
            const S *a = reinterpret_cast<const S *>(w.a) + ((size_t)me.run << w.n);
            const uint32_t z = ip.zall;
            const bool neg = ip.sgn < 0;
#pragma unroll
            for (int k = 0; k < NA; ++k) {
                const uint32_t g = gidx(k);
                A x = unpack(at(a, g));
                if (((g & z) != 0) != neg) { x.x = -x.x; x.y = -x.y; }
                b[k] = x;
            }
        } else {
            set_g();
            if (grad && pass == 0) {
                const typename T::Eta *eta = reinterpret_cast<const typename T::Eta *>(buf);
                const SeedScale up(sizeof(A) == 16 ? kUnit - *w.etaexp : 0);
#pragma unroll
                for (int k = 0; k < NA; ++k) b[k] = seed_dithered(at(eta, gidx(k)), up, dith(k + 320));
            } else {
#pragma unroll
                for (int k = 0; k < NA; ++k) b[k] = at(buf, gidx(k));
            }
        }
    }
    const uint32_t nlo = 1u << w.hl, nhi = 1u << (w.n - w.hl);
    __syncthreads();
    for (; o < ps.nops; ++o) {
        const UOp u = o < kOpsMax ? ops_sh[o] : w.uop[ps.op_begin + o];
        if (!start) {
            if (u.low >= 0) {
                uint32_t st[KB];
#pragma unroll
                for (int j = 0; j < KB; ++j) st[j] = 1u << (low + j);
                slots_of<T, KB>(smem, tbase<KB>(t, low), st, [&](int k, A *s) { *s = b[k]; });
                __syncthreads();
                low = u.low;
                uint32_t b0 = tbase<KB>(t, low);
                if (u.perm >= 0) {
                    const SPerm &pm = w.perm[u.perm];
                    const int q0 = (int)(t & 31u);
                    uint32_t x = __reduce_xor_sync(0xffffffffu, ((gtile >> q0) & 1u) ? pm.oimg[q0] : 0u);
                    for (int q = 0; q < w.tb; ++q) x ^= ((b0 >> q) & 1u) ? pm.limg[q] : 0u;
                    b0 = x;
#pragma unroll
                    for (int j = 0; j < KB; ++j) st[j] = pm.limg[low + j];
                } else {
#pragma unroll
                    for (int j = 0; j < KB; ++j) st[j] = 1u << (low + j);
                }
                slots_of<T, KB>(smem, b0, st, [&](int k, A *s) { b[k] = *s; });
                if (u.perm >= 0) __syncthreads();  // others still read what this thread writes next
            }
            if (u.hm) hadamards<T, KB>(b, u.hm, 0);
            if (u.shift) {
#pragma unroll
                for (int k = 0; k < NA; ++k) {
                    if constexpr (sizeof(A) == 16) scale_down(b[k], u.shift, dith(k + 384));
                    else halve(b[k], u.shift);
                }
            }
        }
        if (u.run >= 0) {
            set_g();
            const int r = u.run;
            const S *tlo = reinterpret_cast<const S *>(w.lo) + (size_t)r * nlo;
            const S *thi = reinterpret_cast<const S *>(w.hi) + (size_t)r * nhi;
            const uint32_t *tm = w.mask + (size_t)r * nhi;
            S *a = reinterpret_cast<S *>(w.a) + ((size_t)r << w.n);
            if (FWD) {
#pragma unroll
                for (int k = 0; k < NA; ++k) {
                    const uint32_t g = gidx(k), l = g & (nlo - 1u), h = g >> w.hl;
                    A x = b[k];
                    if (sizeof(A) == 16) scale_down(x, u.rshift, dith(k + 192));
                    x = mul<0>(mul<0>(x, tlo[l], dith(k)), thi[h], dith(k + 64));
                    if (__popc(l & tm[h]) & 1) { x.x = -x.x; x.y = -x.y; }
                    b[k] = x;
                    at(a, g) = pack(x);
                }
            } else {
                const bool mult = r > 0;
                const int shift = start ? 0 : u.rshift;  // a column that starts here has no Hadamards behind it
                constexpr int UP = 60 - kUnit + (kSumUnit - 60) / 2;  // a product's unit is 2^-60 at 60 - kUnit
                using Part = typename T::Part;
                Part pr[1 + KB] = {}, pi[1 + KB] = {};  // all products; signed by each of the thread's bits
                // A loop over the thread's slots instead of unrolled registers: the vector is out of the
                // registers meanwhile, which hold U checkpoint and factor reads in flight. The thread's bits lie
                // in one half of the index (else, in narrow windows: `both`): the other half's factor is the same
                // for all of its amplitudes, and the sign, bilinear in the halves, is linear in k: par0 ^ bit k
                // of sgnw.
                constexpr int U = KB == 5 ? 8 : 4, LU = KB == 5 ? 3 : 2;
                constexpr uint32_t kWalsh[5] = {0xaaaaaaaau, 0xccccccccu, 0xf0f0f0f0u, 0xff00ff00u, 0xffff0000u};
                const bool hi_var = gsh + KB > w.hl, both = hi_var && gsh < w.hl;
                const uint32_t l0 = g0 & (nlo - 1u), hh = g0 >> w.hl;
                const S *vt = hi_var ? thi : tlo;
                const uint32_t v0 = hi_var ? hh : l0;
                const int vsh = hi_var ? gsh - w.hl : gsh;
                const S ov0 = hi_var ? tlo[l0] : thi[hh];
                const uint32_t m0 = tm[hh];
                uint32_t sgnw = 0;
                if (!both) {
#pragma unroll
                    for (int j = 0; j < KB; ++j) {
                        const bool odd = hi_var ? __popc(l0 & tm[1u << (vsh + j)]) & 1 : (m0 >> (vsh + j)) & 1;
                        if (odd) sgnw ^= kWalsh[j];
                    }
                    if (__popc(l0 & m0) & 1) sgnw = ~sgnw;
                }
                uint32_t st[KB];
#pragma unroll
                for (int j = 0; j < KB; ++j) st[j] = 1u << (low + j);
                const uint32_t tb0 = tbase<KB>(t, low);
                slots_of<T, KB>(smem, tb0, st, [&](int k, A *s) { *s = b[k]; });
                uint32_t sin[U];  // slot offsets within a step of the loop
#pragma unroll
                for (int k = 0; k < U; ++k) sin[k] = sslot<T>((uint32_t)k << low);
                const uint32_t s0 = sslot<T>(tb0);
#pragma unroll 1
                for (int k0 = 0; k0 < NA; k0 += U) {
                    Part pu = {}, qu = {};
                    S av[U], vv[U];
                    const uint32_t ga = g0 + ((uint32_t)k0 << gsh), gv = both ? 0u : v0 + ((uint32_t)k0 << vsh);
                    const uint32_t sb = s0 ^ sslot<T>((uint32_t)k0 << low), sw = sgnw >> k0;
#pragma unroll
                    for (int k = 0; k < U; ++k) {
                        av[k] = at(a, ga + ((uint32_t)k << gsh));
                        if (mult) vv[k] = both ? tlo[(ga + ((uint32_t)k << gsh)) & (nlo - 1u)] : at(vt, gv + ((uint32_t)k << vsh));
                    }
#pragma unroll
                    for (int k = 0; k < U; ++k) {
                        A *sp = reinterpret_cast<A *>(smem + (sb ^ sin[k]));
                        A x = *sp;
                        const uint32_t dk = sizeof(A) == 16 ? (h0 ^ (0x9e3779b9u * (uint32_t)(k0 + k + 1))) | 64u : 0u;
                        if (sizeof(A) == 16) scale_down(x, shift, dk * 11u);
                        const Part p = prod_part<0, UP>(av[k], x);
                        add(pu, p, false);
#pragma unroll
                        for (int j = 0; j < LU; ++j) add(pr[1 + j], p, (k >> j) & 1);
                        if (MIM) {
                            const Part q = prod_part<1, UP>(av[k], x);
                            add(qu, q, false);
#pragma unroll
                            for (int j = 0; j < LU; ++j) add(pi[1 + j], q, (k >> j) & 1);
                        }
                        if (mult) {
                            S ov = ov0;
                            bool neg = (sw >> k) & 1;
                            if (both) {
                                const uint32_t g = ga + ((uint32_t)k << gsh), gh = g >> w.hl;
                                ov = thi[gh];
                                neg = __popc(g & (nlo - 1u) & tm[gh]) & 1;
                            }
                            x = mul<1>(mul<1>(x, vv[k], dk * 3u), ov, dk * 7u);
                            if (neg) { x.x = -x.x; x.y = -x.y; }
                            *sp = x;
                        }
                    }
                    add(pr[0], pu, false);
                    if (MIM) add(pi[0], qu, false);
#pragma unroll
                    for (int j = LU; j < KB; ++j) {
                        add(pr[1 + j], pu, (k0 >> j) & 1);
                        if (MIM) add(pi[1 + j], qu, (k0 >> j) & 1);
                    }
                }
                slots_of<T, KB>(smem, tb0, st, [&](int k, A *s) { b[k] = *s; });
                // The run's rows, its parameters and (in the column's own run) <sigma_j>: each is one of the
                // warp's 16 sums, of the products as they are (0), signed by one of the thread's bits (1 + j)
                // or by a lane bit (8 + j), with a sign per warp for a bit that distinguishes warps or tiles.
                const Run &rn = w.run[r];
                const int ipc = rn.ip_count, ipf = rn.ip_first, nrow = ipc + (start ? 1 : 0);
                const int lane = t & 31, wid = t >> 5;
                {
                    // A warp's sums are rounded once each (512 products, whose parts below the unit add up to less
                    // than 2^31): 2^(n - 9) roundings in all instead of 2^n
                    Part ar[8], ai[8];
#pragma unroll
                    for (int half = 0; half < 2; ++half) {
#pragma unroll
                        for (int g = 0; g < 8; ++g) {
                            if (half == 0) {
                                ar[g] = g <= KB ? pr[g <= KB ? g : 0] : Part{};
                                ai[g] = g <= KB ? pi[g <= KB ? g : 0] : Part{};
                            } else {
                                const bool neg = g < 5 && ((lane >> g) & 1);
                                ar[g] = g < 5 ? (neg ? -pr[0] : pr[0]) : Part{};
                                ai[g] = g < 5 ? (neg ? -pi[0] : pi[0]) : Part{};
                            }
                        }
                        const auto xr = warp8(ar, lane);
                        auto xi = across(Part{});
                        if (MIM) xi = warp8(ai, lane);
                        if ((lane & 3) == 0) {
                            const int row = half * 8 + (lane >> 2);
                            red[row][wid][0] = rounded<UP, 1>(xr, h0 ^ salt(160 + half));
                            if (MIM) red[row][wid][1] = rounded<UP, 1>(xi, h0 ^ salt(162 + half));
                        }
                    }
                }
                __syncthreads();
                for (int x = t; x < nrow * (MIM ? 2 : 1); x += NT) {
                    const int q = MIM ? x >> 1 : x, part = MIM ? x & 1 : 0, row = ipf + q;
                    SIp ip = {0, 0, 1, 0};
                    if (q < ipc) ip = r == ps.run0 && q < kRows ? ips_sh[q] : w.ip[rn.ip_begin + q];
                    Red d = 0;
                    for (int k = 0; k < NT / 32; ++k) {
                        const uint32_t g = gtile | spread(tbase<KB>(k * 32, low));
                        const Red y = red[ip.src][k][part];
                        d += ((g & ip.z) != 0) != (ip.sgn < 0) ? -y : y;
                    }
                    ll v;
                    if constexpr (sizeof(A) == 16) v = d;
                    else v = __double2ll_rn(scalbn(d, kSumUnit - (grad ? *w.etaexp : 0)));
                    ll *dst = nullptr;
                    if (q == ipc) dst = part ? nullptr : w.sacc + me.col;
                    else if (grad) dst = w.gacc + row;
                    else if (row < me.col) dst = w.acc + (size_t)part * w.P * w.P + (size_t)row * w.P + me.col;
                    if (dst) atomicAdd(reinterpret_cast<unsigned long long *>(dst), (unsigned long long)v);
                }
                __syncthreads();
            }
        }
        start = false;
    }
    if (FWD || (flag & 1)) {  // flag of the walk: a later pass follows
        set_g();
#pragma unroll
        for (int k = 0; k < NA; ++k) {
            scale_down(b[k], ps.shift, dith(k + 256));
            at(buf, gidx(k)) = b[k];
        }
    }
}

// ------------------------------------------------------------------------------------------
// eta = H psi in the final frame: one gather per distinct X mask; the coefficients of a mask's terms
// combine to one factor per amplitude first (for TFIM the n - 1 ZZ terms are one real factor of psi[m]).
// complex64 sums in float32, the precision it is stored in. complex128 in fixed point: coefficients as
// multiples of 2^(eexp - 62), sums as multiples of 2^(eexp - 61); the float64 pipe would take four times as
// long (22 qubits, 43 terms: 3.4 ms). <E> and |eta|^2 in float64 and then fixed point (as the on-chip
// kernel), complex64 in two float32 over a thread's four amplitudes first. The next mask's
// loads go out before a mask's products (20 qubits, 41 masks, complex64: 56 to 45 us, 344 MB of gathers from L2;
// and float64 conversions and warp sums taken to once per thread and CTA).
template <class T> struct Coef;
template <> struct Coef<Fix> {
    using C = ll;
    using S = double;   // a thread's share of |eta|^2
    using S4 = double;  // of <E>, over four amplitudes
    static __device__ __forceinline__ C of(double c, int eexp) { return __double2ll_rn(scalbn(c, 62 - eexp)); }
    static __device__ __forceinline__ ll mul(ll c, ll x) {
        const int ch = hi_of(c), cl = lo_of(c), xh = hi_of(x), xl = lo_of(x);
        // 2^-62 times 2^-kUnit to 2^-61: the sum's unit
        constexpr int S = kUnit + 1 - 32;
        const ll m = wide(ch, xl) + wide(cl, xh) + (wide(cl, xl) >> 32);
        return (wide(ch, xh) << (32 - S)) + ((m + (1ll << (S - 1))) >> S);
    }
    static __device__ __forceinline__ double value(ll h, int eexp) { return scalbn((double)h, eexp - 61); }
    // h / 2^eexp: at most 1, so that its square stays in range
    static __device__ __forceinline__ double scaled(ll h, float) { return (double)h * 0x1p-61; }
};
template <> struct Coef<Flt> {
    using C = float;
    using S = float;
    using S4 = Two;
    static __device__ __forceinline__ C of(double c, int) { return (float)c; }
    static __device__ __forceinline__ float mul(float c, float x) { return c * x; }
    static __device__ __forceinline__ float value(float h, int) { return h; }
    static __device__ __forceinline__ float scaled(float h, float fs) { return h * fs; }
};

__device__ __forceinline__ double2 amp_at(longlong2 x) {
    return double2{scalbn((double)x.x, -kUnit), scalbn((double)x.y, -kUnit)};
}
__device__ __forceinline__ float2 amp_at(float2 x) { return x; }

template <class T> __global__ void __launch_bounds__(256) k_sheff(SWork w, int in, int out) {
    using A = typename T::A;
    using E = typename T::Eta;
    using K = Coef<T>;
    using C = typename K::C;
    constexpr int kTerms = 128, NA = 4;  // terms staged at a time; amplitudes per thread
    __shared__ C coef[kTerms];
    __shared__ uint32_t tx[kTerms], tz[kTerms];
    __shared__ int tny[kTerms];
    using S = typename K::S;
    __shared__ double red[256][2];
    grid_ready();
    const A *v = reinterpret_cast<const A *>(w.b) + ((size_t)in << w.n);
    E *eta = reinterpret_cast<E *>(reinterpret_cast<A *>(w.b) + ((size_t)out << w.n));
    const uint64_t N = 1ull << w.n;
    const int sc = max(-120, min(120, -w.eexp));  // complex64: eta / 2^eexp, within float32's range
    const float fs = scalbnf(1.0f, sc);
    double e = 0.0, n2 = 0.0;
    for (uint64_t m0 = (uint64_t)blockIdx.x * (256 * NA); m0 < N; m0 += (uint64_t)gridDim.x * (256 * NA)) {
        const uint32_t m = (uint32_t)m0 + threadIdx.x;  // and m + 256, ..
        A h[NA];
        C cr[NA], ci[NA];
#pragma unroll
        for (int k = 0; k < NA; ++k) { h[k] = A{0, 0}; cr[k] = ci[k] = 0; }
        int kinds = 0;  // parts of the factor that the mask's terms have: 1 real, 2 imaginary
        A y[NA];        // psi at the mask's sources
        auto load = [&](uint32_t x) {
#pragma unroll
            for (int k = 0; k < NA; ++k) y[k] = v[(m + 256 * k) ^ x];
        };
        auto add = [&](const A *y) {
#pragma unroll
            for (int k = 0; k < NA; ++k) {
                if (kinds & 1) { h[k].x += K::mul(cr[k], y[k].x); h[k].y += K::mul(cr[k], y[k].y); }
                if (kinds & 2) { h[k].x -= K::mul(ci[k], y[k].y); h[k].y += K::mul(ci[k], y[k].x); }
                cr[k] = ci[k] = 0;
            }
            kinds = 0;
        };
        for (int t0 = 0; t0 < w.nterms; t0 += kTerms) {
            const int nt = min(kTerms, w.nterms - t0);
            if (w.nterms > kTerms || m0 == (uint64_t)blockIdx.x * (256 * NA)) {
                __syncthreads();
                for (int t = threadIdx.x; t < nt; t += 256) {
                    const DevTerm tm = w.term[t0 + t];
                    coef[t] = K::of((tm.ny & 2) ? -tm.coeff : tm.coeff, w.eexp);
                    tx[t] = (uint32_t)tm.x;
                    tz[t] = (uint32_t)tm.z;
                    tny[t] = tm.ny & 1;
                }
                __syncthreads();
            }
            load(tx[0]);
            for (int t = 0; t < nt; ++t) {
                const uint32_t x = tx[t];
                const C c = coef[t];
                const uint32_t z = tz[t];
                if (tny[t]) {
                    kinds |= 2;
#pragma unroll
                    for (int k = 0; k < NA; ++k) ci[k] += (__popc(((m + 256 * k) ^ x) & z) & 1) ? -c : c;
                } else {
                    kinds |= 1;
#pragma unroll
                    for (int k = 0; k < NA; ++k) cr[k] += (__popc(((m + 256 * k) ^ x) & z) & 1) ? -c : c;
                }
                const bool last = t + 1 == nt;
                if (last || tx[t + 1] != x) {  // the mask's last term: the next mask's loads go out first
                    A u[NA];
#pragma unroll
                    for (int k = 0; k < NA; ++k) u[k] = y[k];
                    if (!last) load(tx[t + 1]);
                    add(u);
                }
            }
        }
        typename K::S4 e4 = {};  // a thread's four amplitudes
        S n4 = 0;                // (an upper bound is all that is made of it)
#pragma unroll
        for (int k = 0; k < NA; ++k) {
            const auto y = amp_at(v[m + 256 * k]);
            E o;
            const S hr = K::value(h[k].x, w.eexp), hi = K::value(h[k].y, w.eexp);
            o.x = hr;
            o.y = hi;
            eta[m + 256 * k] = o;
            if constexpr (sizeof(S) == 4) e4 = (e4 + exact_product(y.x, hr)) + exact_product(y.y, hi);
            else e4 += y.x * hr + y.y * hi;
            const S ar = K::scaled(h[k].x, fs), ai = K::scaled(h[k].y, fs);
            n4 += ar * ar + ai * ai;
        }
        e += (double)e4;
        n2 += n4;
    }
    red[threadIdx.x][0] = e;
    red[threadIdx.x][1] = n2;
    __syncthreads();
    if (threadIdx.x >= 32) return;
    double s = 0.0, s2 = 0.0;
    for (int k = 0; k < 8; ++k) { s += red[32 * k + threadIdx.x][0]; s2 += red[32 * k + threadIdx.x][1]; }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        s += __shfl_xor_sync(0xffffffffu, s, o);
        s2 += __shfl_xor_sync(0xffffffffu, s2, o);
    }
    if (threadIdx.x == 0) {
        if (sizeof(S) == 4) s2 = scalbn(s2, -2 * (sc + w.eexp));  // of (eta / 2^eexp)^2
        atomicAdd(w.eacc, (unsigned long long)__double2ll_rn(scalbn(s, 60 - w.eexp)));
        atomicAdd(w.eacc + 1, (unsigned long long)__double2ll_ru(s2 * 0x1p60) + 1ull);
        __threadfence();
        if (atomicAdd(w.eacc + 2, 1ull) == (unsigned long long)(gridDim.x - 1)) {
            const double en = scalbn((double)(ll)atomicExch(w.eacc, 0ull), w.eexp - 60);
            const double nrm = sqrt((double)atomicExch(w.eacc + 1, 0ull)) * 0x1p-30 * (1.0 + (sizeof(S) == 4 ? 0x1p-20 : 0x1p-40));
            atomicExch(w.eacc + 2, 0ull);
            *w.etaexp = w.eexp + ilogb(nrm) + 1;
            *w.energy = *w.bad ? __longlong_as_double(0x7ff8000000000000ll) : en;
        }
    }
}

__global__ void k_sfinish(SWork w, int what) {
    grid_ready();
    const size_t PP = (size_t)w.P * w.P, x = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    constexpr double unit = 1.0 / (double)(1ll << kSumUnit);
    const double nan = __longlong_as_double(0x7ff8000000000000ll);
    const bool bad = *w.bad != 0;
    if ((what & 1) && x < PP) {
        w.L[x] = bad ? nan : 0.25 * unit * (double)w.acc[x];
        if (what & 4) w.Lim[x] = bad ? nan : 0.25 * unit * (double)w.acc[PP + x];
    }
    if (x < (size_t)w.P) {
        if (what & 1) w.sigma[x] = bad ? nan : unit * (double)w.sacc[x];
        if (what & 2) w.gradraw[x] = bad ? nan : -scalbn((double)w.gacc[x], *w.etaexp - kSumUnit);
    }
}

// ------------------------------------------------------------------------------------------
static size_t tile_bytes(int precision, int tb) { return (size_t)(precision == QNG_C128 ? 16 : 8) << tb; }

template <class T, int KB, int NT> static cudaError_t prepare_nt(size_t sm) {
    cudaError_t e = raise_smem_limit(reinterpret_cast<const void *>(k_stream<T, 0, 0, KB, NT>), sm);
    if (e == cudaSuccess) e = raise_smem_limit(reinterpret_cast<const void *>(k_stream<T, 1, 0, KB, NT>), sm);
    if (e == cudaSuccess) e = raise_smem_limit(reinterpret_cast<const void *>(k_stream<T, 0, 1, KB, NT>), sm);
    return e;
}

// the kernel of a precision and tile of 2^tb amplitudes
#define QNG_STREAM(F, tb)                                                                                     \
    (precision == QNG_C128 ? (tb == 11 ? F(Fix, 4, 128) : F(Fix, 4, 256))                                     \
                           : (tb == 11 ? F(Flt, 4, 128) : tb == 12 ? F(Flt, 4, 256) : F(Flt, 5, 256)))

cudaError_t prepare_stream(int precision, int tb) {
    const size_t sm = tile_bytes(precision, tb);
#define QNG_F(T, KB, NT) prepare_nt<T, KB, NT>(sm)
    return QNG_STREAM(QNG_F, tb);
#undef QNG_F
}

cudaError_t launch_stream_tables(const SWork &w, int precision, cudaStream_t st) {
    cudaError_t e = cudaMemsetAsync(w.bad, 0, sizeof(int32_t), st);
    if (e != cudaSuccess || w.R == 0) return e;
    const unsigned n = (1u << w.hl) + (1u << (w.n - w.hl));
    return launch_next(false, k_half, dim3(w.R, (n + kHalfThreads - 1) / kHalfThreads), kHalfThreads, 0, 1, st, w,
                       (int)(precision == QNG_C128));
}

cudaError_t launch_stream_forward(const SWork &w, const SPass &p, int first, int slot, int precision, cudaStream_t st) {
    const unsigned tiles = 1u << (w.n - w.tb);
    const size_t sm = tile_bytes(precision, w.tb);
#define QNG_F(T, KB, NT) launch_next(w.chain, k_stream<T, 0, 1, KB, NT>, tiles, NT, sm, 1, st, w, p, 0, slot, 1, (int)first)
    return QNG_STREAM(QNG_F, w.tb);
#undef QNG_F
}

cudaError_t launch_stream_walk(const SWork &w, const SPass &p, int pass, int col0, int ncol, int store, int precision,
                               int metric_im, cudaStream_t st) {
    const unsigned grid = (1u << (w.n - w.tb)) * (unsigned)ncol;
    const size_t sm = tile_bytes(precision, w.tb);
#define QNG_F(T, KB, NT)                                                                                            \
    launch_next(w.chain, metric_im ? k_stream<T, 1, 0, KB, NT> : k_stream<T, 0, 0, KB, NT>, grid, NT, sm, 1, st, w, p, pass, \
                col0, ncol, (int)store)
    return QNG_STREAM(QNG_F, w.tb);
#undef QNG_F
}

cudaError_t launch_stream_hpsi(const SWork &w, int in, int out, int precision, cudaStream_t st) {
    return launch_next(w.chain, precision == QNG_C128 ? k_sheff<Fix> : k_sheff<Flt>, w.hblocks, 256, 0, 1, st, w, in, out);
}

cudaError_t launch_stream_finish(const SWork &w, int what, cudaStream_t st) {
    if (w.P == 0) return cudaSuccess;
    const size_t n = (what & 1) ? (size_t)w.P * w.P : (size_t)w.P;
    return launch_next(w.chain, k_sfinish, (unsigned)((n + 255) / 256), 256, 0, 1, st, w, what);
}

}  // namespace frames
}  // namespace qng
