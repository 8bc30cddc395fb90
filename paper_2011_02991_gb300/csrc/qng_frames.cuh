// Arithmetic of the diagonal-frame kernels, shared by the on-chip (qng_frames.cu) and streaming
// (qng_frames_stream.cu) ones: the two amplitude types, their products and sums.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

#include "qng_frames.h"

namespace qng {
namespace frames {

typedef long long ll;

struct Part;
struct Fix {  // complex128: fixed point
    using A = longlong2;  // amplitude, 2^60 = 1
    using S = int4;       // stored: (re hi, re lo, im hi, im lo), value = hi 2^32 + lo, lo signed
    using Acc = ll;       // inner products
    using Part = frames::Part;
    using Red = ll;
    using Eta = double2;  // H psi
    static constexpr uint32_t kSwz = 7;  // eight 16-byte banks
};
struct Flt {  // complex64
    using A = float2;
    using S = float2;
    using Acc = float;
    using Part = float;
    using Red = double;
    using Eta = float2;
    static constexpr uint32_t kSwz = 15;  // sixteen 8-byte banks
};

__device__ __forceinline__ int hi_of(ll x) { return (int)((x + 0x80000000ll) >> 32); }
__device__ __forceinline__ int lo_of(ll x) { return (int)x; }
__device__ __forceinline__ ll join(int hi, int lo) { return ((ll)hi << 32) + lo; }
__device__ __forceinline__ ll wide(int a, int b) { return (ll)a * (ll)b; }

__device__ __forceinline__ int4 pack(longlong2 x) { return int4{hi_of(x.x), lo_of(x.x), hi_of(x.y), lo_of(x.y)}; }
__device__ __forceinline__ float2 pack(float2 x) { return x; }
__device__ __forceinline__ longlong2 unpack(int4 s) { return longlong2{join(s.x, s.y), join(s.z, s.w)}; }
__device__ __forceinline__ float2 unpack(float2 s) { return s; }

// c 2^-30 to nearest, halves away from zero: x d and (-x) d are negatives of each other, so states that
// are symmetric stay exactly so (ties are common where x is a power of two)
__device__ __forceinline__ ll round30(ll c) { return (c + ((1ll << 29) + (c >> 63))) >> 30; }

// x d (CONJ = 0) or x conj(d); d is stored with 2^62 = 1
template <int CONJ> __device__ __forceinline__ longlong2 mul(longlong2 x, int4 d, uint32_t dither = 0) {
    const int rh = hi_of(x.x), rl = lo_of(x.x), ih = hi_of(x.y), il = lo_of(x.y);
    // y_r = x_r c + x_i m, y_i = x_i c + x_r p with (m, p) = (-s, s), conjugate (s, -s)
    const int mh = CONJ ? d.z : -d.z, ml = CONJ ? d.w : -d.w, ph = -mh, pl = -ml;
    const ll h0 = wide(rh, d.x) + wide(ih, mh), h1 = wide(ih, d.x) + wide(rh, ph);
    const ll c0 = wide(rh, d.y) + wide(rl, d.x) + wide(ih, ml) + wide(il, mh);
    const ll c1 = wide(ih, d.y) + wide(il, d.x) + wide(rh, pl) + wide(rl, ph);
    if (dither) {
        const ll l0 = wide(rl, d.y) + wide(il, ml), l1 = wide(il, d.y) + wide(rl, pl);
        return longlong2{(h0 << 2) + ((c0 + (l0 >> 32) + (ll)(dither >> 2)) >> 30),
                         (h1 << 2) + ((c1 + (l1 >> 32) + (ll)((dither * 5u) >> 2)) >> 30)};
    }
    return longlong2{(h0 << 2) + round30(c0), (h1 << 2) + round30(c1)};
}
template <int CONJ> __device__ __forceinline__ float2 mul(float2 x, float2 d, uint32_t = 0) {
    const float s = CONJ ? -d.y : d.y;
    return float2{fmaf(x.x, d.x, -x.y * s), fmaf(x.x, s, x.y * d.x)};
}

// A sum over threads of float32 partial sums, as the float32 nearest to it and what is left: 48 bits on the float32
// pipe, which takes 64 times what the float64 pipe does.
struct Two {
    float s, e;
    __device__ __forceinline__ explicit operator double() const { return (double)s + (double)e; }
};
__device__ __forceinline__ Two exact_sum(float a, float b) {  // s + e = a + b
    const float s = a + b, t = s - a;
    return Two{s, (a - (s - t)) + (b - t)};
}
__device__ __forceinline__ Two exact_product(float a, float b) {
    const float p = a * b;
    return Two{p, fmaf(a, b, -p)};
}
__device__ __forceinline__ Two operator+(Two a, Two b) {
    const Two r = exact_sum(a.s, b.s);
    return Two{r.s, r.e + (a.e + b.e)};
}

// Re (IM = 0) or Im (IM = 1) of conj(a) b for fixed-point vectors of unit 2^-u, as a multiple v of
// 2^-(2u - 60 + 2 UP) (2^-62 for both paths) and what is left below it (f, kFracBits bits, never negative). Inner
// products are between vectors of norm 1 at most, so sums stay within 1 in magnitude. lo lo counts: at 2^12 amplitudes
// and more a product is 2^-12 and less.
struct Part {
    ll v;
    int f;
};
template <int UP> constexpr int kFracBits = 28 - 2 * UP;
template <int IM, int UP> __device__ __forceinline__ Part prod_part(int4 a, longlong2 b) {
    const int rh = hi_of(b.x), rl = lo_of(b.x), ih = hi_of(b.y), il = lo_of(b.y);
    constexpr int F = kFracBits<UP>;
    const ll half = 1ll << 31;
    ll h, c;
    if constexpr (IM == 0) {
        h = wide(a.x, rh) + wide(a.z, ih);
        const ll l = wide(a.y, rl) + wide(a.w, il) + half;
        c = wide(a.x, rl) + wide(a.y, rh) + wide(a.z, il) + wide(a.w, ih) + (l >> 32);
    } else {
        h = wide(a.x, ih) - wide(a.z, rh);
        const ll l = wide(a.y, il) - wide(a.w, rl) + half;
        c = wide(a.x, il) + wide(a.y, ih) - wide(a.z, rl) - wide(a.w, rh) + (l >> 32);
    }
    return Part{(h << (32 - F)) + (c >> F), (int)((unsigned)c & ((1u << F) - 1u))};
}
template <int IM, int UP> __device__ __forceinline__ float prod_part(float2 a, float2 b) {
    return IM ? fmaf(a.x, b.y, -a.y * b.x) : fmaf(a.x, b.x, a.y * b.y);
}
__device__ __forceinline__ void add(Part &s, Part p, bool neg) {
    s.v += neg ? -p.v : p.v;
    s.f += neg ? -p.f : p.f;
}
__device__ __forceinline__ void add(float &s, float p, bool neg) { s += neg ? -p : p; }
__device__ __forceinline__ Part operator-(Part p) { return Part{-p.v, -p.f}; }
__device__ __forceinline__ Part operator+(Part a, Part b) { return Part{a.v + b.v, a.f + b.f}; }
// A sum rounded by rnd, uniform below one unit; DROP: low bits of f left out, so that adding to it stays in range.
template <int UP, int DROP = 0> __device__ __forceinline__ ll rounded(Part s, uint32_t rnd) {
    constexpr int F = kFracBits<UP> - DROP;
    return s.v + (((s.f >> DROP) + (int)(rnd >> (32 - F))) >> F);
}
template <int UP, int DROP = 0> __device__ __forceinline__ double rounded(Two s, uint32_t) { return (double)s; }
// One product, rounded by rnd.
template <int IM, int UP> __device__ __forceinline__ ll prod(int4 a, longlong2 b, uint32_t rnd) {
    return rounded<UP>(prod_part<IM, UP>(a, b), rnd);
}
template <int IM, int UP> __device__ __forceinline__ float prod(float2 a, float2 b, uint32_t) { return prod_part<IM, UP>(a, b); }

// Pseudo-random bits over the amplitudes: a thread's (hash of its index), xor a constant per amplitude. The hash is
// the 32-bit mixer that Chris Wellons published as lowbias32 (public domain).
__device__ __forceinline__ uint32_t hash(uint32_t x) {
    x = (x ^ (x >> 16)) * 0x7feb352du;
    x = (x ^ (x >> 15)) * 0x846ca68bu;
    return x ^ (x >> 16);
}
__host__ __device__ constexpr uint32_t salt(int k) { return 0x9e3779b9u * (uint32_t)(2 * k + 1); }

__device__ __forceinline__ longlong2 operator+(longlong2 a, longlong2 b) { return longlong2{a.x + b.x, a.y + b.y}; }
__device__ __forceinline__ longlong2 operator-(longlong2 a, longlong2 b) { return longlong2{a.x - b.x, a.y - b.y}; }
// both components of a complex64 amplitude in one instruction
__device__ __forceinline__ float2 operator+(float2 a, float2 b) {
    float2 r;
    asm("{.reg .b64 x, y;\n mov.b64 x, {%2, %3};\n mov.b64 y, {%4, %5};\n add.rn.f32x2 x, x, y;\n mov.b64 {%0, %1}, x;}"
        : "=f"(r.x), "=f"(r.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return r;
}
__device__ __forceinline__ float2 operator-(float2 a, float2 b) {  // fma(b, -1, a) rounds once, as a - b does
    float2 r;
    asm("{.reg .b64 x, y, m;\n mov.b64 x, {%2, %3};\n mov.b64 y, {%4, %5};\n mov.b64 m, 0xbf800000bf800000;\n"
        " fma.rn.f32x2 x, y, m, x;\n mov.b64 {%0, %1}, x;}"
        : "=f"(r.x), "=f"(r.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return r;
}

// x 2^-s to nearest, ties to even. Rounding down instead would put the same -1/2 unit on every component:
// a constant vector, and states can overlap with that one (22 qubits: g off by 6e-13 instead of 1e-15).
__device__ __forceinline__ void halve(longlong2 &x, int s) {
    const ll h = (1ll << (s - 1)) - 1;
    x.x = (x.x + (h + (((int)x.x >> s) & 1))) >> s;
    x.y = (x.y + (h + (((int)x.y >> s) & 1))) >> s;
}

__device__ __forceinline__ void halve(float2 &x, int s) {
    const float h = __int_as_float((127 - s) << 23);
    x.x *= h;
    x.y *= h;
}

__device__ __forceinline__ ll shfl(ll v, int o) { return __shfl_xor_sync(0xffffffffu, v, o); }
__device__ __forceinline__ float shfl(float v, int o) { return __shfl_xor_sync(0xffffffffu, v, o); }

__device__ __forceinline__ Two shfl(Two v, int o) { return Two{shfl(v.s, o), shfl(v.e, o)}; }
__device__ __forceinline__ Part shfl(Part p, int o) { return Part{shfl(p.v, o), __shfl_xor_sync(0xffffffffu, p.f, o)}; }

// the type that sums over threads are carried in
__device__ __forceinline__ ll across(ll v) { return v; }
__device__ __forceinline__ Part across(Part p) { return p; }
__device__ __forceinline__ Two across(float v) { return Two{v, 0.0f}; }
__device__ __forceinline__ ll pair_sum(ll a, ll b) { return a + b; }
__device__ __forceinline__ Part pair_sum(Part a, Part b) { return a + b; }
__device__ __forceinline__ Two pair_sum(float a, float b) { return exact_sum(a, b); }

// Warp sums of 8 values: the lane returns the sum of a[(lane >> 2) & 7].
template <typename T> __device__ __forceinline__ auto warp8(const T (&a)[8], int lane) {
    const bool b4 = lane & 16, b3 = lane & 8, b2 = lane & 4;
    decltype(across(a[0])) t[4], u[2];
#pragma unroll
    for (int k = 0; k < 4; ++k) t[k] = pair_sum(b4 ? a[4 + k] : a[k], shfl(b4 ? a[k] : a[4 + k], 16));
#pragma unroll
    for (int k = 0; k < 2; ++k) u[k] = (b3 ? t[2 + k] : t[k]) + shfl(b3 ? t[k] : t[2 + k], 8);
    auto v = (b2 ? u[1] : u[0]) + shfl(b2 ? u[0] : u[1], 4);
    v = v + shfl(v, 2);
    return v + shfl(v, 1);
}

// Hadamards (unnormalised) on the thread's bits hm, then `shift` halvings.
template <class T, int KB> __device__ __forceinline__ void hadamards(typename T::A (&b)[1 << KB], int hm, int shift) {
#pragma unroll
    for (int j = 0; j < KB; ++j)
        if ((hm >> j) & 1) {
#pragma unroll
            for (int k = 0; k < (1 << KB); ++k)
                if (!((k >> j) & 1)) {
                    const typename T::A x = b[k], y = b[k | (1 << j)];
                    b[k] = x + y;
                    b[k | (1 << j)] = x - y;
                }
        }
    if (shift) {
#pragma unroll
        for (int k = 0; k < (1 << KB); ++k) halve(b[k], shift);
    }
}

// 2^(-half / 2), 2^61 = 1: sqrt(1/2) to all of its bits. The float64 one is 1.4e-16 of its square short, and as
// every transition with an odd number of Hadamards multiplies by it, the norm drifted by that much each time (11 qubits,
// 21 such transitions: <E> 2.5e-15 off, 0.6e-15 now).
__host__ __device__ __forceinline__ ll root_half(int half) {
    const ll r = (half & 1) ? 1630477228166597777ll : 1ll << 61;
    const int s = half >> 1;
    return s ? (r + (1ll << (s - 1))) >> s : r;
}

// (c, s) of a rotation, 2^62 = 1, brought to c^2 + s^2 = 1: float64 rounds each of them at 2^-54, which leaves the
// norm of every rotation off by about 1e-16, and a circuit's by the sum of that.
__host__ __device__ __forceinline__ longlong2 unit_pair(ll c, ll s) {
#ifdef __CUDA_ARCH__
    const unsigned long long ch = __umul64hi(c < 0 ? -c : c, c < 0 ? -c : c), sh = __umul64hi(s < 0 ? -s : s, s < 0 ? -s : s);
#else
    const unsigned long long ch = (unsigned long long)(((__int128)c * c) >> 64), sh = (unsigned long long)(((__int128)s * s) >> 64);
#endif
    const unsigned long long cl = (unsigned long long)c * (unsigned long long)c, sl = (unsigned long long)s * (unsigned long long)s;
    const unsigned long long lo = cl + sl, hi = ch + sh + (lo < cl);  // c^2 + s^2, 2^124 = 1
    // e = 1 - c^2 - s^2, 2^62 = 1; c (1 + e / 2)
    const ll e = (ll)((((1ull << 60) - hi - (lo != 0)) << 2) | ((0ull - lo) >> 62));
    return longlong2{c + (((c >> 20) * e + (1ll << 42)) >> 43), s + (((s >> 20) * e + (1ll << 42)) >> 43)};
}

// (cos, lam sin) of theta / 2 as the factor tables multiply by it, 2^62 = 1; sin's low half is negated there: off -2^31
__device__ __forceinline__ int4 rotation_pair(double c, double s) {
    longlong2 p = unit_pair(__double2ll_rn(c * 0x1p62), __double2ll_rn(s * 0x1p62));
    if ((int)p.y == INT32_MIN) ++p.y;
    return pack(p);
}

__device__ __forceinline__ void store_factor(int4 *d, longlong2 f) {
    ll y = f.y << 1;
    // the low half of the sine is negated by the product: keep it off -2^31
    if ((int)y == INT32_MIN) ++y;
    *d = pack(longlong2{f.x << 1, y});
}
__device__ __forceinline__ void store_factor(float2 *d, longlong2 f) {
    *d = float2{(float)f.x * 0x1p-61f, (float)f.y * 0x1p-61f};
}

__device__ __forceinline__ double2 amp_of(longlong2 x) { return double2{(double)x.x * 0x1p-60, (double)x.y * 0x1p-60}; }
__device__ __forceinline__ double2 amp_of(float2 x) { return double2{(double)x.x, (double)x.y}; }

// A factor 2^k. Only for Hamiltonians below 1e-280 or so does it take more than one float64 (the same in every thread).
struct SeedScale {
    double f, g;
    __device__ __forceinline__ explicit SeedScale(int k) : f(scalbn(1.0, min(k, 1000))), g(k > 1000 ? scalbn(1.0, k - 1000) : 0.0) {}
    __device__ __forceinline__ double operator()(double x) const { return g != 0.0 ? x * f * g : x * f; }
};
__device__ __forceinline__ longlong2 seed(double2 e, const SeedScale &up) {  // -i eta
    return longlong2{__double2ll_rn(up(e.y)), __double2ll_rn(-up(e.x))};
}
__device__ __forceinline__ float2 seed(float2 e, const SeedScale &) { return float2{e.y, -e.x}; }

template <class T, int KB> struct Sums {  // of the thread's products: all, and signed by each of its bits
    typename T::Acc all, bit[KB];
};

template <class T, int KB> __device__ __forceinline__ typename T::Acc pick(const Sums<T, KB> &s, int z) {
    typename T::Acc v = s.all;
#pragma unroll
    for (int j = 0; j < KB; ++j) if (z == (1 << j)) v = s.bit[j];
    return v;
}

}  // namespace frames
}  // namespace qng
