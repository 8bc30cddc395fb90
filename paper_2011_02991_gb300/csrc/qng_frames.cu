// sm_103a kernels of the diagonal-frame path (qng_frames.h): on-chip instances, n <= 16.
//
//   k_tables   per run, the complex factor that its gates put on every amplitude
//   k_fwd      one cluster per instance: psi through every run, a checkpoint after each
//   k_heff     H psi in the final frame, <E>, and the seed eta of the gradient column
//   k_cols     one CTA (or cluster) per group of columns: the walk down the runs
//
// A vector lives in registers, 16 amplitudes per thread over four index bits ("arrangement"); changing
// the four bits goes through shared memory. Hadamards on a thread's own bits are additions.
//
// complex128. The float64 pipe of this part does 2 lanes a clock and SM (DADD, DFMA and int64
// conversions alike; measured 1.98), the integer pipes 60 64-bit additions and 16 to 19 products
// 32 x 32 -> 64 (IMAD.WIDE). The vector is therefore kept in 64-bit fixed point, 2^60 = 1: states have
// unit norm, so no component ever exceeds sqrt 2 between transitions (4 sqrt 2 inside one), additions
// are exact and a product rounds at 2^-60, where float64 would round at 2^-53 of the component.
// Products come from 32-bit halves in signed (balanced) form, x = hi 2^32 + lo: hi hi and the two
// cross terms, six IMAD.WIDE for a sum of two products; lo lo (below 2^-62) is left out of the factors'
// products and taken into the inner products'. Those sum 2^-62 units exactly in 64-bit integers, whatever
// the order.
// complex64 runs the same steps on float32 amplitudes; its inner products leave the thread as two float32 words.
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <cstdint>

#include "qng_frames.cuh"

namespace cg = cooperative_groups;

namespace qng {
namespace frames {

// Where a thread's amplitudes are: thread t of the vector's 2^(nE-KB), arrangement low.
template <int KB> struct Place {
    uint32_t t;      // thread index within the vector, over all of its CTAs
    int nl, cl;      // index bits held by one CTA; log2 CTAs
    __device__ __forceinline__ uint32_t base(int low) const {
        return ((t >> low) << (low + KB)) | (t & ((1u << low) - 1u));
    }
    __device__ __forceinline__ bool remote(int low) const { return low + KB > nl; }
};

// Shared-memory offset (bytes) of index m within the vector's buffer: 16 consecutive threads (8 for
// 16-byte amplitudes) hit distinct banks in every arrangement. The map is linear over the bits of m, and
// a buffer starts at a multiple of its size, so a thread's offsets follow from one by XOR.
template <class T> __device__ __forceinline__ uint32_t slot(uint32_t m) {
    return (m ^ ((m >> 4) & T::kSwz)) * (uint32_t)sizeof(typename T::A);
}

__device__ __forceinline__ void vsync(bool cluster, int tpc) {
    if (cluster) cg::this_cluster().sync();
    else if (tpc <= 32) __syncwarp();
    else __syncthreads();
}

// Visit the thread's slots in arrangement low (through perm's index map when given): f(k, address),
// in Gray-code order of k. smem + boff is the vector's buffer.
template <class T, int KB, typename F>
__device__ __forceinline__ void each_slot(unsigned char *smem, uint32_t boff, const Place<KB> &p, int low, const Perm *perm,
                                          F &&f) {
    using A = typename T::A;
    uint32_t b0 = p.base(low), st[KB];
    bool rem = p.remote(low);
    if (perm) {
        uint32_t s = 0;
#pragma unroll
        for (int b = 0; b < 16; ++b) s ^= ((b0 >> b) & 1u) ? perm->img[b] : 0u;
        b0 = s;
#pragma unroll
        for (int j = 0; j < KB; ++j) st[j] = perm->img[low + j];
        rem = p.cl > 0;
    } else {
#pragma unroll
        for (int j = 0; j < KB; ++j) st[j] = 1u << (low + j);
    }
    if (!rem) {
        const uint32_t lm = ((uint32_t)sizeof(A) << p.nl) - 1u;
        uint32_t s = boff + (slot<T>(b0) & lm);
#pragma unroll
        for (int j = 0; j < KB; ++j) st[j] = slot<T>(st[j]) & lm;
#pragma unroll
        for (int i = 0; i < (1 << KB); ++i) {
            f(i ^ (i >> 1), reinterpret_cast<A *>(smem + s));
            // Gray code: step i to i + 1 flips bit ctz(i + 1)
            if (i + 1 < (1 << KB)) s ^= st[(i & 1) == 0 ? 0 : ((i & 2) == 0 ? 1 : ((i & 4) == 0 ? 2 : KB - 1))];
        }
    } else {
        cg::cluster_group cl = cg::this_cluster();
        const uint32_t lm = (1u << p.nl) - 1u;
#pragma unroll
        for (int k = 0; k < (1 << KB); ++k) {
            uint32_t m = b0;
#pragma unroll
            for (int j = 0; j < KB; ++j) if ((k >> j) & 1) m ^= st[j];
            f(k, reinterpret_cast<A *>(cl.map_shared_rank(smem + boff + (slot<T>(m & lm)), m >> p.nl)));
        }
    }
}

// Exchange the vector from arrangement low (updated) to u.low. The thread writes the slots that it
// alone read last, so one barrier is enough; after a permuted read a second one keeps later writes
// off slots that are still being read. Threads without amplitudes (on = false) share the barriers.
template <class T, int KB>
__device__ __forceinline__ void exchange(typename T::A (&b)[1 << KB], unsigned char *smem, uint32_t boff,
                                         const Place<KB> &p, int tpc, int &low,
                                         const UOp &u, const Perm *perms, bool on = true) {
    const Perm *perm = u.perm >= 0 ? perms + u.perm : nullptr;
    const bool cl = p.cl > 0 && (perm || p.remote(low) || p.remote(u.low));
    if (on) each_slot<T, KB>(smem, boff, p, low, nullptr, [&](int k, typename T::A *s) { *s = b[k]; });
    vsync(cl, tpc);
    if (on) each_slot<T, KB>(smem, boff, p, u.low, perm, [&](int k, typename T::A *s) { b[k] = *s; });
    if (perm) vsync(cl, tpc);
    low = u.low;
}

// ------------------------------------------------------------------------------------------
// Factor tables: entry k * 2^(nE-kb) + t of run r is the factor of amplitude (t, k) in the run's
// arrangement, times 2^(-khalf/2) of the transition before it (table_half). The products are taken in fixed point for both
// precisions (2^61 = 1, cos and sin of float64): members that do not touch the thread's own two index
// bits multiply one common factor, the others each of the four.
template <class T> __global__ void __launch_bounds__(kTabThreads) k_tables(FWork w, int kb) {
    __shared__ int4 cs[kTabThreads];    // cos, sin of a member, 2^62 = 1
    __shared__ Member mem[kTabThreads];
    __shared__ int any_bad;
    grid_ready();
    const TabItem it = w.tab[blockIdx.x];
    const Inst &in = w.inst[it.inst];
    const Run &rn = w.run[in.run_off + it.run];
    const int low = rn.low, mem_count = rn.mem_count, mem_begin = rn.mem_begin;
    const uint32_t TC = 1u << (in.nE - kb), N4 = (1u << in.nE) / kTabAmps;
    const uint32_t u = it.first / kTabAmps + threadIdx.x;
    const bool on = u < N4;
    // four entries k = kq..kq + 3 of thread t: the arrangement's two lowest bits
    const uint32_t t = u & (TC - 1u), kq = (u / TC) * kTabAmps;
    const uint32_t base = ((t >> low) << (low + kb)) | (t & ((1u << low) - 1u)) | (kq << low);
    const uint32_t own = (uint32_t)(kTabAmps - 1) << low;
    const int half = rn.khalf;
    longlong2 com = {root_half(half), 0};
    longlong2 f[kTabAmps];
    bool any_own = false;  // uniform over the block
    if (threadIdx.x == 0) any_bad = 0;
    const double *theta = w.theta + in.param_off;
    for (int pass = 0; pass < 2; ++pass) {  // common members, then those on the thread's own bits
        if (pass == 1) {
#pragma unroll
            for (int k = 0; k < kTabAmps; ++k) f[k] = com;
            if (!any_own) break;
        }
        for (int e0 = 0; e0 < mem_count; e0 += kTabThreads) {
            const bool reload = pass == 0 || mem_count > kTabThreads;
            if (reload) {
                __syncthreads();
                if (e0 + (int)threadIdx.x < mem_count) {
                    const Member e = w.member[mem_begin + e0 + threadIdx.x];
                    mem[threadIdx.x] = e;
                    if (e.kind == 0) {
                        const double th = theta[e.param];
                        double s, c;
                        if (!isfinite(th)) { any_bad = 1; atomicCAS(w.status, 0, (int)QNG_ERR_ARG); }
                        sincos(0.5 * th, &s, &c);
                        if (it.first == 0) w.pctrl[in.param_off + e.param] = 1.0;  // controlled ones: their column
                        cs[threadIdx.x] = rotation_pair(c, e.sgn > 0 ? -s : s);  // c - i lam s
                    }
                }
                __syncthreads();
            }
            const int ne = min(mem_count - e0, kTabThreads);
            for (int q = 0; q < ne; ++q) {
                const Member &e = mem[q];
                const bool mine = ((e.z | e.ctrl) & own) != 0;
                if (mine) any_own = true;
                if (mine != (pass == 1)) continue;
                if (pass == 0) {
                    if ((base & e.ctrl) != e.cval) continue;
                    const bool par = __popc(base & e.z) & 1;
                    if (e.kind == 0) com = par ? mul<1>(com, cs[q]) : mul<0>(com, cs[q]);
                    else if (e.kind == 1) { if (par ^ (e.sgn < 0)) com = longlong2{-com.x, -com.y}; }
                    else if (par) com = longlong2{com.y, -com.x};  // times -i
                } else {
#pragma unroll
                    for (int k = 0; k < kTabAmps; ++k) {
                        const uint32_t m = base | ((uint32_t)k << low);
                        if ((m & e.ctrl) != e.cval) continue;
                        const bool par = __popc(m & e.z) & 1;
                        if (e.kind == 0) f[k] = par ? mul<1>(f[k], cs[q]) : mul<0>(f[k], cs[q]);
                        else if (e.kind == 1) { if (par ^ (e.sgn < 0)) f[k] = longlong2{-f[k].x, -f[k].y}; }
                        else if (par) f[k] = longlong2{f[k].y, -f[k].x};
                    }
                }
            }
        }
    }
    __syncthreads();
    if (it.first == 0 && threadIdx.x == 0) w.bad_run[in.run_off + it.run] = any_bad;
    if (!on) return;
    typename T::S *d = reinterpret_cast<typename T::S *>(w.d) + in.d_off + ((int64_t)it.run << in.nE);
#pragma unroll
    for (int k = 0; k < kTabAmps; ++k) store_factor(d + (kq + k) * TC + t, f[k]);
}

// ------------------------------------------------------------------------------------------
// Forward sweep: one cluster per instance, 2^(nE-KB-cl) active threads per CTA.
template <class T, int KB> __global__ void __launch_bounds__(512) k_fwd(FWork w, int first, int cl) {
    constexpr int NA = 1 << KB;
    using A = typename T::A;
    using S = typename T::S;
    extern __shared__ __align__(1024) unsigned char smem[];
    const int inst = w.order[first + (blockIdx.x >> cl)];
    const Inst &in = w.inst[inst];
    const int rank = cl ? (int)cg::this_cluster().block_rank() : 0;
    const uint32_t TC = 1u << (in.nE - KB), tpc = TC >> cl;
    if (cl) cg::this_cluster().sync();  // every CTA runs before its shared memory is touched
    const bool on = threadIdx.x < tpc;
    const Place<KB> p{on ? rank * tpc + threadIdx.x : 0u, in.nE - cl, cl};
    A b[NA];
#pragma unroll
    for (int k = 0; k < (1 << KB); ++k) b[k] = A{0, 0};
    if (on && p.t == 0) {
        if constexpr (sizeof(A) == 16) b[0].x = 1ll << 60;
        else b[0].x = 1.0f;
    }
    int low = in.start0;
    const int tp = (int)blockDim.x;  // inactive threads share the barriers
    const int nE = in.nE, nops = in.fwd_cnt;
    UOp *ops = reinterpret_cast<UOp *>(smem + ((size_t)blockDim.x << KB) * sizeof(A));
    for (int x = threadIdx.x; x < nops; x += blockDim.x) ops[x] = w.uop[in.fwd_off + x];
    grid_ready();
    if (rank == 0 && threadIdx.x == 0) {
        int bad = 0;
        for (int r = 0; r < in.R; ++r) bad |= w.bad_run[in.run_off + r];
        w.bad[inst] = bad;
    }
    const S *dall = reinterpret_cast<const S *>(w.d) + in.d_off;
    S *aall = reinterpret_cast<S *>(w.a) + in.a_off;
    __syncthreads();
    for (int o = 0; o < nops; ++o) {
        const UOp u = ops[o];
        const S *d = dall + ((int64_t)max(u.run, 0) << nE) + p.t;
        if (u.low >= 0) exchange<T, KB>(b, smem, 0u, p, tp, low, u, w.perm, on);
        if (u.hm) hadamards<T, KB>(b, u.hm, u.shift);
        if (u.run >= 0 && on) {
            S *a = aall + ((int64_t)u.run << nE) + p.t;
#pragma unroll
            for (int k0 = 0; k0 < NA; k0 += 4) {
                S dv[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) dv[k] = d[(k0 + k) * TC];
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    b[k0 + k] = mul<0>(b[k0 + k], dv[k]);
                    a[(k0 + k) * TC] = pack(b[k0 + k]);
                }
            }
        }
    }
    if (on) {  // the final vector, natural order
        A *v = reinterpret_cast<A *>(w.v) + in.v_off;
        const uint32_t mb = p.base(low);
#pragma unroll
        for (int k = 0; k < (1 << KB); ++k) v[mb | (k << low)] = b[k];
    }
    if (cl) cg::this_cluster().sync();
}

// ------------------------------------------------------------------------------------------
// eta = H psi in the final frame, float64 sums, kHSplit threads per amplitude (each a share of the
// terms); <E> = <psi|eta> and |eta|^2 summed over the instance's CTAs in fixed point (units of
// 2^(eexp - 60) and 2^(2 eexp - 60): integer sums do not depend on the order). The CTA that finishes
// last turns <E> into float64 and |eta| into the power of two that bounds it, the unit that the
// gradient column's fixed-point walk starts with.
template <class T> __global__ void __launch_bounds__(kHThreads) k_heff(FWork w, int first) {
    using A = typename T::A;
    using E = typename T::Eta;
    constexpr int kTerms = 64;
    __shared__ DevTerm terms[kTerms];
    __shared__ double red[kHThreads / 32][2];
    grid_ready();
    const HItem it = w.hitem[first + blockIdx.x];
    const Inst &in = w.inst[it.inst];
    // 8 consecutive amplitudes and 4 shares of the terms per warp
    const int lane = threadIdx.x & 31, share = lane >> 3;
    const uint32_t N = 1u << in.nE;
    const uint32_t m = it.chunk * (kHThreads / kHSplit) + (threadIdx.x >> 5) * 8 + (lane & 7);
    const int nterms = in.nterms;
    const A *v = reinterpret_cast<const A *>(w.v) + in.v_off;
    double hr = 0.0, hi = 0.0;
    for (int t0 = 0; t0 < nterms; t0 += kTerms) {
        __syncthreads();
        for (int t = threadIdx.x; t < min(kTerms, nterms - t0); t += kHThreads) terms[t] = w.term[in.term_off + t0 + t];
        __syncthreads();
        if (m >= N) continue;
#pragma unroll 4
        for (int t = share; t < min(kTerms, nterms - t0); t += kHSplit) {
            const DevTerm &tm = terms[t];
            const uint32_t src = m ^ (uint32_t)tm.x;
            const double2 x = amp_of(v[src]);
            const int ph = (tm.ny + 2 * (__popc(src & (uint32_t)tm.z) & 1)) & 3;  // i^ph coeff x
            const double cr = (ph == 2 || ph == 1) ? -tm.coeff : tm.coeff, ci = (ph & 2) ? -tm.coeff : tm.coeff;
            hr = fma(cr, (ph & 1) ? x.y : x.x, hr);
            hi = fma(ci, (ph & 1) ? x.x : x.y, hi);
        }
    }
#pragma unroll
    for (int o = 8; o < 32; o <<= 1) {
        hr += __shfl_xor_sync(0xffffffffu, hr, o);
        hi += __shfl_xor_sync(0xffffffffu, hi, o);
    }
    double e = 0.0, n2 = 0.0;
    if (m < N && share == 0) {
        const double2 x = amp_of(v[m]);
        e = fma(x.x, hr, x.y * hi);
        // |eta| / 2^eexp <= 1 before it is squared (coefficients beyond 1e154 or below 1e-154 would leave float64's
        // range squared); two factors, as 2^-eexp alone can leave it too
        const double f0 = scalbn(1.0, -(in.eexp / 2)), f1 = scalbn(1.0, in.eexp / 2 - in.eexp);
        const double sr = hr * f0 * f1, si = hi * f0 * f1;
        n2 = fma(sr, sr, si * si);
        E *eta = reinterpret_cast<E *>(w.eta) + in.v_off;
        E h;
        h.x = hr;
        h.y = hi;
        eta[m] = h;
    }
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) {
        e += __shfl_xor_sync(0xffffffffu, e, o);
        n2 += __shfl_xor_sync(0xffffffffu, n2, o);
    }
    if (lane == 0) { red[threadIdx.x >> 5][0] = e; red[threadIdx.x >> 5][1] = n2; }
    __syncthreads();
    if (threadIdx.x == 0) {
        double s = 0.0, s2 = 0.0;
        for (int k = 0; k < kHThreads / 32; ++k) { s += red[k][0]; s2 += red[k][1]; }
        unsigned long long *acc = w.eacc + 3 * it.inst;
        atomicAdd(acc, (unsigned long long)__double2ll_rn(scalbn(s, 60 - in.eexp)));
        // rounded up, so that the sum never falls below the true one
        atomicAdd(acc + 1, (unsigned long long)__double2ll_ru(s2 * 0x1p60) + 1ull);
        __threadfence();
        if (atomicAdd(acc + 2, 1ull) == (unsigned long long)(in.hchunks - 1)) {
            const double en = scalbn((double)(ll)atomicExch(acc, 0ull), in.eexp - 60);
            const double nrm = sqrt((double)atomicExch(acc + 1, 0ull)) * 0x1p-30 * (1.0 + 0x1p-40);  // |eta| / 2^eexp
            atomicExch(acc + 2, 0ull);
            w.etaexp[it.inst] = in.eexp + ilogb(nrm) + 1;
            w.energy[it.inst] = w.bad[it.inst] ? __longlong_as_double(0x7ff8000000000000ll) : en;
        }
    }
}

// ------------------------------------------------------------------------------------------
// Column walk. MIM = 1: metric columns take Im L_ij as well.
// Inner products are sums of 2^-62 (vectors: 2^-60); each product is rounded by pseudo-random bits, as rounding to
// nearest is the same for the equal amplitudes of a structured state and adds up over them.
constexpr int kSumUp = 1;

// One run of the walk: products with the checkpoint, f(k, re, im), then (mult) the run's adjoint factors.
template <class T, int KB, int MIM, typename F>
__device__ __forceinline__ void run_step(typename T::A (&b)[1 << KB], const typename T::S *a, const typename T::S *d,
                                         uint32_t TC, bool mult, uint32_t h0, F &&f) {
    constexpr int B = 4;  // loads in flight
#pragma unroll
    for (int k0 = 0; k0 < (1 << KB); k0 += B) {
        typename T::S av[B], dv[B];
#pragma unroll
        for (int k = 0; k < B; ++k) {
            av[k] = a[(k0 + k) * TC];
            if (mult) dv[k] = d[(k0 + k) * TC];
        }
#pragma unroll
        for (int k = 0; k < B; ++k) {
            const typename T::Acc p = prod<0, kSumUp>(av[k], b[k0 + k], h0 ^ salt(k0 + k));
            const typename T::Acc q = MIM ? prod<1, kSumUp>(av[k], b[k0 + k], h0 ^ salt(64 + k0 + k)) : typename T::Acc(0);
            f(k0 + k, p, q);
            if (mult) b[k0 + k] = mul<1>(b[k0 + k], dv[k]);
        }
    }
}

// A thread's products summed with a parameter's signs, over those that its control includes.
template <class Acc, int NA> __device__ __forceinline__ Acc signed_sum(const Acc (&p)[NA], uint32_t incl, uint32_t sign) {
    Acc v = 0;
#pragma unroll
    for (int k = 0; k < NA; ++k) {
        const Acc x = (incl >> k) & 1 ? p[k] : Acc(0);
        v += (sign >> k) & 1 ? -x : x;
    }
    return v;
}

// GEN = 1: instances with controlled and string rotations, whose parameters take the thread's products with signs
// and controls of their own. A run that holds one keeps its products in registers and sums them once per parameter (runs
// of such circuits have one or two).
template <class T, int KB, int MIM, int GEN>
__global__ void __launch_bounds__(512, 1) k_cols(FWork w, int first, int cl, int max_P) {
    constexpr int NA = 1 << KB;
    using A = typename T::A;
    using S = typename T::S;
    using Acc = typename T::Acc;
    using Red = typename T::Red;
    extern __shared__ __align__(1024) unsigned char smem[];
    const Item it = w.item[first + (blockIdx.x >> cl)];
    const Inst &in = w.inst[it.inst];
    const int nE = in.nE, P = in.P;
    const int rank = cl ? (int)cg::this_cluster().block_rank() : 0;
    const uint32_t TC = 1u << (nE - KB);
    const int ltpc = nE - KB - cl, tpc = 1 << ltpc;  // threads of a column in this CTA
    const int sl = threadIdx.x >> ltpc, tin = threadIdx.x & (tpc - 1);
    const uint32_t boff = ((uint32_t)sl << (nE - cl)) * (uint32_t)sizeof(A);
    // per-warp partial sums [slot][row][warp], rows 0..P-1 the parameters, row P <sigma_j>
    Red *red = reinterpret_cast<Red *>(reinterpret_cast<A *>(smem) + (size_t)blockDim.x * NA);
    const int nw = tpc >= 32 ? tpc / 32 : 1;
    const bool direct = nw == 1 && cl == 0;  // the column is one warp's: no sums over warps
    const size_t rows = (size_t)(max_P + 1) * (blockDim.x / 32);
    if (cl) cg::this_cluster().sync();
    const Place<KB> p{rank * (uint32_t)tpc + tin, nE - cl, cl};
    const bool grad = it.ncol == 0;
    const bool live = grad ? sl == 0 : sl < it.ncol;
    const int col = grad ? P : (live ? w.cols[it.list + sl] : -1);
    const double unit = sizeof(A) == 16 ? 0x1p-62 : 1.0;
    const uint32_t h0 = sizeof(A) == 16 ? hash(p.t) : 0u;

    // the walk's tables in shared memory: steps, runs and parameters (a table read per run would wait on
    // L2 each time)
    Ip *ips = reinterpret_cast<Ip *>(red + (MIM ? 2 : 1) * rows);
    Run *runs = reinterpret_cast<Run *>(ips + it.nip);
    UOp *ops = reinterpret_cast<UOp *>(runs + (it.nruns));
    const int nops = in.bwd_cnt - it.entry;
    for (int x = threadIdx.x; x < it.nip; x += blockDim.x) ips[x] = w.ip[in.ip_off + x];
    for (int x = threadIdx.x; x < it.nruns; x += blockDim.x) runs[x] = w.run[in.run_off + x];
    for (int x = threadIdx.x; x < nops; x += blockDim.x) ops[x] = w.uop[in.bwd_off + it.entry + x];
    grid_ready();
    const bool bad = w.bad[it.inst] != 0;
    __syncthreads();

    // a finished sum of the column c's row: a parameter below c, c itself (its control probability), or P
    auto put = [&](int c, int row, double re, double im) {
        if (bad) re = im = __longlong_as_double(0x7ff8000000000000ll);
        if (grad) {
            w.gradraw[in.param_off + row] = sizeof(A) == 16 ? -scalbn(re, w.etaexp[it.inst] - 62) : -re;
        } else if (row == P) {
            w.sigma[in.param_off + c] = re * unit;
        } else if (row < c) {
            w.L[in.metric_off + (int64_t)row * P + c] = 0.25 * unit * re;
            if (MIM) w.Lim[in.metric_off + (int64_t)row * P + c] = 0.25 * unit * im;
        } else if (row == c) {
            const Ip &me = ips[c];
            if (me.ctrl != 0 || me.incl16 != me.all16) w.pctrl[in.param_off + c] = re * unit;
        }
    };

    A b[NA];
    int low;
    if (grad) {  // Im <a|K b> = Re <a|K (-i b)>: the gradient column walks -i eta
        low = in.end_low;
        const typename T::Eta *eta = reinterpret_cast<const typename T::Eta *>(w.eta) + in.v_off;
        const uint32_t mb = p.base(low);
        const SeedScale up(sizeof(A) == 16 ? 60 - w.etaexp[it.inst] : 0);
#pragma unroll
        for (int k = 0; k < NA; ++k) b[k] = seed(eta[mb | (k << low)], up);
    } else {  // column j of run r starts as K_j Psi_r
        low = runs[it.run].low;
        const S *a = reinterpret_cast<const S *>(w.a) + in.a_off + ((int64_t)it.run << nE) + p.t;
        const Ip &me = ips[live ? col : 0];
        const bool on = live && (p.t & me.ctrl) == me.cval;
        const uint32_t incl = on ? me.incl16 : 0u;
        const uint32_t sign = me.sign16 ^ (((__popc(p.t & me.z) & 1) ^ (me.sgn < 0)) ? 0xffffu : 0u);
#pragma unroll
        for (int k = 0; k < (1 << KB); ++k) {
            A x = unpack(a[k * TC]);
            if ((sign >> k) & 1) { x.x = -x.x; x.y = -x.y; }
            b[k] = ((incl >> k) & 1) ? x : A{0, 0};
        }
    }
    bool start = !grad;
    for (int o = 0; o < nops; ++o) {
        const UOp u = ops[o];
        if (!start) {
            if (u.low >= 0) exchange<T, KB>(b, smem, boff, p, tpc, low, u, w.perm);
            if (u.hm) hadamards<T, KB>(b, u.hm, u.shift);
        }
        if (u.run >= 0) {
            const Run &rn = runs[u.run];
            const int64_t off = ((int64_t)u.run << nE) + p.t;
            const S *a = reinterpret_cast<const S *>(w.a) + in.a_off + off, *d = reinterpret_cast<const S *>(w.d) + in.d_off + off;
            const int ipc = rn.ip_count, ipf = rn.ip_first;
            const int nrow = ipc + (start ? 1 : 0);  // the column's own run: <sigma_j> as one more row
            if (GEN && !rn.simple) {
                Acc pr[NA], pi[NA];
                run_step<T, KB, MIM>(b, a, d, TC, u.run > 0, h0, [&](int k, Acc p, Acc q) { pr[k] = p; pi[k] = q; });
#pragma unroll 1
                for (int q = 0; q < nrow; ++q) {
                    uint32_t incl = 0xffffu, sign = 0;
                    if (q < ipc) {
                        const Ip &ip = ips[ipf + q];
                        incl = (p.t & ip.ctrl) == ip.cval ? ip.incl16 : 0u;
                        sign = ip.sign16 ^ (((__popc(p.t & ip.z) & 1) ^ (ip.sgn < 0)) ? 0xffffu : 0u);
                    }
                    auto xr = across(signed_sum<Acc, NA>(pr, incl, sign)), xi = across(Acc(0));
                    if (MIM) xi = across(signed_sum<Acc, NA>(pi, incl, sign));
                    for (int s = min(tpc, 32) >> 1; s > 0; s >>= 1) {
                        xr = xr + shfl(xr, s);
                        if (MIM) xi = xi + shfl(xi, s);
                    }
                    if (!live || (tin & 31) != 0) continue;
                    const int row = q < ipc ? ipf + q : P;
                    if (direct || tpc < 32) {
                        put(col, row, (double)xr, (double)xi);
                    } else {
                        const size_t at = ((size_t)sl * (max_P + 1) + row) * nw + (tin >> 5);
                        red[at] = (Red)xr;
                        if (MIM) red[rows + at] = (Red)xi;
                    }
                }
                start = false;
                continue;
            }
            Sums<T, KB> sr, si;
            sr.all = si.all = 0;
#pragma unroll
            for (int j = 0; j < KB; ++j) sr.bit[j] = si.bit[j] = 0;
            run_step<T, KB, MIM>(b, a, d, TC, u.run > 0, h0, [&](int k, Acc p, Acc q) {
                sr.all += p;
                if (MIM) si.all += q;
#pragma unroll
                for (int j = 0; j < KB; ++j) {
                    sr.bit[j] += (k >> j) & 1 ? -p : p;
                    if (MIM) si.bit[j] += (k >> j) & 1 ? -q : q;
                }
            });
            for (int q0 = 0; q0 < nrow; q0 += 8) {
                Acc ar[8], ai[8];
#pragma unroll
                for (int g = 0; g < 8; ++g) {
                    const int q = q0 + g;
                    Acc vr = 0, vi = 0;
                    if (q < ipc) {
                        const Ip &ip = ips[ipf + q];
                        const uint32_t sgn = (__popc(p.t & ip.z) & 1) ^ (ip.sgn < 0);
                        vr = pick<T, KB>(sr, ip.zreg);
                        if (MIM) vi = pick<T, KB>(si, ip.zreg);
                        if (sgn) { vr = -vr; vi = -vi; }
                    } else if (q < nrow) {
                        vr = sr.all;
                    }
                    ar[g] = vr;
                    if (MIM) ai[g] = vi;
                }
                if (tpc >= 32) {
                    const int lane = threadIdx.x & 31, q = q0 + ((lane >> 2) & 7);
                    const auto xr = warp8(ar, lane);
                    auto xi = across(Acc(0));
                    if (MIM) xi = warp8(ai, lane);
                    if (live && (lane & 3) == 0 && q < nrow) {
                        const int row = q < ipc ? ipf + q : P;
                        if (direct) {
                            put(col, row, (double)xr, (double)xi);
                        } else {
                            const size_t at = ((size_t)sl * (max_P + 1) + row) * nw + (tin >> 5);
                            red[at] = (Red)xr;
                            if (MIM) red[rows + at] = (Red)xi;
                        }
                    }
                } else {
#pragma unroll
                    for (int g = 0; g < 8; ++g) {
                        if (q0 + g >= nrow) break;
                        auto xr = across(ar[g]), xi = across(MIM ? ai[g] : Acc(0));
                        for (int s = tpc >> 1; s > 0; s >>= 1) {
                            xr = xr + shfl(xr, s);
                            if (MIM) xi = xi + shfl(xi, s);
                        }
                        if (live && tin == 0) put(col, q0 + g < ipc ? ipf + q0 + g : P, (double)xr, (double)xi);
                    }
                }
            }
        }
        start = false;
    }
    if (direct) return;
    __syncthreads();
    if (cl) cg::this_cluster().sync();
    if (rank == 0) {
        const int slots = blockDim.x >> ltpc;
        for (int x = threadIdx.x; x < slots * (P + 1); x += blockDim.x) {
            const int s2 = x / (P + 1), row = x % (P + 1);
            if (grad ? (s2 > 0 || row == P) : s2 >= it.ncol) continue;
            const int c = grad ? P : w.cols[it.list + s2];
            if (!grad && row > c && row != P) continue;
            Red tr = 0, ti = 0;
            for (int r = 0; r < (1 << cl); ++r) {
                const Red *rr = cl ? cg::this_cluster().map_shared_rank(red, r) : red;
                for (int k = 0; k < nw; ++k) {
                    const size_t at = ((size_t)s2 * (max_P + 1) + row) * nw + k;
                    tr += rr[at];
                    if (MIM) ti += rr[rows + at];
                }
            }
            put(c, row, (double)tr, (double)ti);
        }
    }
    if (cl) cg::this_cluster().sync();
}

// ------------------------------------------------------------------------------------------
#define QNG_FRAMES(F)                                                                       \
    (precision == QNG_C128 ? (kb == 3 ? F(Fix, 3) : F(Fix, 4)) : (kb == 3 ? F(Flt, 3) : F(Flt, 4)))

// takes_general: complex128 with 16 amplitudes a thread has no registers for a run's products (1.3 KB of spills)
template <class T, int KB> constexpr int kGeneral = sizeof(typename T::A) == 16 && KB == 4 ? 0 : 1;

template <class T, int KB> static cudaError_t prepare_t(size_t smem_fwd, size_t smem_col, size_t smem_col_im) {
    cudaError_t e = raise_smem_limit(reinterpret_cast<const void *>(k_fwd<T, KB>), smem_fwd);
    if (e == cudaSuccess) e = raise_smem_limit(reinterpret_cast<const void *>(k_cols<T, KB, 0, 0>), smem_col);
    if (e == cudaSuccess) e = raise_smem_limit(reinterpret_cast<const void *>(k_cols<T, KB, 1, 0>), smem_col_im);
    constexpr int G = kGeneral<T, KB>;
    if (e == cudaSuccess) e = raise_smem_limit(reinterpret_cast<const void *>(k_cols<T, KB, 0, G>), smem_col);
    if (e == cudaSuccess) e = raise_smem_limit(reinterpret_cast<const void *>(k_cols<T, KB, 1, G>), smem_col_im);
    return e;
}

cudaError_t prepare(int precision, int kb, size_t smem_fwd, size_t smem_col, size_t smem_col_im) {
#define QNG_F(T, KB) prepare_t<T, KB>(smem_fwd, smem_col, smem_col_im)
    return QNG_FRAMES(QNG_F);
#undef QNG_F
}

cudaError_t launch_tables(const FWork &w, int ntab, int kb, int precision, cudaStream_t st) {
    if (ntab == 0) return cudaSuccess;
    return launch_next(false, precision == QNG_C128 ? k_tables<Fix> : k_tables<Flt>, ntab, kTabThreads, 0, 1, st, w, kb);
}

cudaError_t launch_forward(const FWork &w, const Class &c, int precision, cudaStream_t st) {
    if (c.num_inst == 0) return cudaSuccess;
    const int kb = c.kb;
#define QNG_F(T, KB) launch_next(w.chain, k_fwd<T, KB>, c.num_inst << c.cl, c.fwd_threads, c.smem_fwd, 1u << c.cl, st, w, c.first_inst, c.cl)
    return QNG_FRAMES(QNG_F);
#undef QNG_F
}

cudaError_t launch_hpsi(const FWork &w, int first, int num, int precision, cudaStream_t st) {
    if (num == 0) return cudaSuccess;
    return launch_next(w.chain, precision == QNG_C128 ? k_heff<Fix> : k_heff<Flt>, num, kHThreads, 0, 1, st, w, first);
}

cudaError_t launch_columns(const FWork &w, const Class &c, int precision, int first, int num, int metric_im,
                           cudaStream_t st) {
    if (num == 0) return cudaSuccess;
    const int kb = c.kb;
#define QNG_F(T, KB)                                                                                             \
    launch_next(w.chain, c.general ? (metric_im ? k_cols<T, KB, 1, kGeneral<T, KB>> : k_cols<T, KB, 0, kGeneral<T, KB>>) \
                                   : (metric_im ? k_cols<T, KB, 1, 0> : k_cols<T, KB, 0, 0>), num << c.cl, c.threads, \
                metric_im ? c.smem_col_im : c.smem_col, 1u << c.cl, st, w, first, c.cl, c.max_P)
    return QNG_FRAMES(QNG_F);
#undef QNG_F
}

}  // namespace frames
}  // namespace qng
