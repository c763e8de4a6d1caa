// Shared device helpers of the TILD step: complex arithmetic, the
// Philox4x32-10 generator, Deserno-Holm assignment weights and the implicit
// chain topology.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

namespace tild {

// Programmatic dependent launch: a kernel launched with that attribute may start
// while its predecessor runs. dependency_wait() returns when the predecessor
// has finished and its writes are visible; nothing that another kernel writes
// is touched before it. It also lets the successor start (its blocks then wait
// in turn), so at most one kernel waits behind the running one, and what
// earlier kernels wrote is complete when a kernel starts. What the predecessor
// itself writes must not be read through the read-only cache (it changes while
// the kernel is resident): those reads are __ldcg, __ldca or __ldcs. Without
// the attribute both instructions do nothing.
__device__ __forceinline__ void dependency_wait() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// ---------------------------------------------------------------- types

template <typename T> struct cplx_of;
template <> struct cplx_of<float> { using type = float2; };
template <> struct cplx_of<double> { using type = double2; };
template <typename T> using cplx_t = typename cplx_of<T>::type;

template <class V> __device__ __forceinline__ V c_add(V a, V b) { return {a.x + b.x, a.y + b.y}; }
template <class V> __device__ __forceinline__ V c_sub(V a, V b) { return {a.x - b.x, a.y - b.y}; }
// Products rounded by themselves and fused multiply-adds, written out where a
// sum has two products: left to the compiler, which of them is fused may differ
// between two instantiations of the same code, and the launch shapes, the
// batched and the single kernels have to give the same bits.
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float fma_rn(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double fma_rn(double a, double b, double c) { return __fma_rn(a, b, c); }
template <class V> __device__ __forceinline__ V c_mul(V a, V b) {
    return {fma_rn(a.x, b.x, -mul_rn(a.y, b.y)), fma_rn(a.y, b.x, mul_rn(a.x, b.y))};
}
template <class V> __device__ __forceinline__ V c_conj(V a) { return {a.x, -a.y}; }
// multiply by -i (forward-transform quarter turn) or +i
template <class V> __device__ __forceinline__ V c_mul_negi(V a) { return {a.y, -a.x}; }
template <class V> __device__ __forceinline__ V c_mul_posi(V a) { return {-a.y, a.x}; }

// Deterministic density accumulation: every bead weight w in [0, 1] is
// rounded once to an integer, round(w * 2^F), and all sums are integer sums,
// which are associative: the grids are bit-identical for any order of
// contributions, blocks or re-binning.
//   FP32 path: F = 22. A tile's shared-memory patch holds 32-bit sums; a tile
//     of at most 1023 beads cannot overflow (1023 * 2^22 < 2^32), larger tiles
//     spread straight into the 64-bit grid. Quantisation <= 2^-23 per
//     contribution, comparable to the FP32 rounding of the weights.
//   FP64 path: F = 44, 64-bit patch sums; quantisation <= 2^-45.
// The global grid is 64-bit in both cases.
template <typename T> struct FixedPoint;
// FP32: one 32-bit shared word per patch point and species.
template <> struct FixedPoint<float> {
    using patch_t = unsigned int;
    static constexpr double scale = 4194304.0;  // 2^22
    static constexpr int max_tile_beads = 1023;
    // round(w 2^22) of a weight w = wx wyz in [0, 1], from wx and scaled(wyz); w
    // is the float product, so that the integers are those of every kernel that
    // forms the weight first. Adding 1.5 2^23 rounds to nearest and leaves the
    // integer in the low bits: the conversion instruction runs at a quarter of the rate.
    static __device__ __forceinline__ float scaled(float wyz) { return wyz * 4194304.0f; }
    static __device__ __forceinline__ unsigned int to_patch(float wx, float wyz_s) {
        return __float_as_uint(__fadd_rn(__fmul_rn(wx, wyz_s), 12582912.0f)) - 0x4B400000u;
    }
    static __device__ __forceinline__ unsigned long long to_grid(float wx, float wyz_s) { return to_patch(wx, wyz_s); }
};
// FP64: one 64-bit shared word per point and species.
template <> struct FixedPoint<double> {
    using patch_t = unsigned long long;
    static constexpr double scale = 17592186044416.0;  // 2^44
    static constexpr int max_tile_beads = 0x7fffffff;
    static __device__ __forceinline__ double scaled(double wyz) { return wyz * scale; }
    static __device__ __forceinline__ unsigned long long to_patch(double wx, double wyz_s) {
        return (unsigned long long)__double2ll_rn(wx * wyz_s);
    }
    static __device__ __forceinline__ unsigned long long to_grid(double wx, double wyz_s) { return to_patch(wx, wyz_s); }
};
// Fixed point -> density (scale = 2^-F / dV); no FP64 in the FP32 path.
// (FP32: the 64-bit conversion instruction is slow; the leading 32 bits of |v|
// with a sticky bit for the rest round to the same float)
__device__ __forceinline__ float ll_to_float(long long v) {
    const unsigned long long a = v < 0 ? 0ull - (unsigned long long)v : (unsigned long long)v;
    const unsigned hi = (unsigned)(a >> 32), lo = (unsigned)a;
    const int s = __clz(hi);  // 32: |v| < 2^32
    const unsigned top = s == 32 ? lo : __funnelshift_l(lo, hi, s) | ((lo << s) != 0u ? 1u : 0u);
    const float f = __uint2float_rn(top);
    const float r = s == 32 ? f : f * __int_as_float((127 + 32 - s) << 23);
    return v < 0 ? -r : r;
}
__device__ __forceinline__ float from_fixed(long long v, float scale) { return mul_rn(ll_to_float(v), scale); }
__device__ __forceinline__ double from_fixed(long long v, double scale) { return mul_rn((double)v, scale); }
// The same for densities (v >= 0). A sum below 2^32 (a thousand beads on one
// point) is converted from 32 bits: the 64-bit conversion runs at a small
// fraction of that rate, and both round the same value to nearest.
__device__ __forceinline__ float density_from_fixed(long long v, float scale) {
    const float f = (v >> 32) == 0 ? __uint2float_rn((unsigned)v) : __ll2float_rn(v);
    return mul_rn(f, scale);
}
__device__ __forceinline__ double density_from_fixed(long long v, double scale) { return from_fixed(v, scale); }

// Sums of observables (energies, forces): at least the precision of FP64 sums.
// FP64 contexts sum in FP64. The FP64 unit of this part does two operations per
// clock and SM, and FP64 sums of float terms took longer than the passes that
// feed them; FP32 contexts therefore sum triples of floats. A sum (hi, mid)
// keeps the rounding errors of hi exactly in mid, and those of mid in lo
// (Knuth's two-sum), and a product its own (by a fused multiply-add; Dekker
// 1971): what is lost is below 2^-70 of the sum per term. Per block the
// triples become doubles. The exponent range remains that of floats, so terms
// are scaled to be near 1, and a sum that left the range (wide_in_range) is
// taken again in FP64 by bead_sums64 and spectral_sums64. Forces, energies and
// density of 1.6M beads on 128^3: 437 us with FP64 sums, 246 with these (220
// with pairs of floats, which hold 48 bits at best and fewer where the terms
// are uneven).
template <typename T> struct Wide;
template <> struct Wide<double> {
    using stored = double;
    double v = 0.0;
    static __device__ __forceinline__ Wide prod(double a, double b) { return {a * b}; }
    static __device__ __forceinline__ Wide sum(double a, double b) { return {a + b}; }
    __device__ __forceinline__ void add(double x) { v += x; }
    __device__ __forceinline__ void add_prod(double a, double b) { v = fma(a, b, v); }
    __device__ __forceinline__ void add(const Wide& o) { v += o.v; }
    __device__ __forceinline__ Wide times(double s) const { return {v * s}; }
    __device__ __forceinline__ Wide square() const { return {v * v}; }
    __device__ __forceinline__ Wide shfl_down(int o) const { return {__shfl_down_sync(0xffffffffu, v, o)}; }
    __device__ __forceinline__ stored store() const { return v; }
    static __device__ __forceinline__ Wide load(stored s) { return {s}; }
    __device__ __forceinline__ double value() const { return v; }
};
// s + e = a + b, s the rounded sum
__device__ __forceinline__ float two_sum(float a, float b, float& e) {
    const float s = __fadd_rn(a, b), t = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, t)), __fsub_rn(b, t));
    return s;
}
template <> struct Wide<float> {
    using stored = float3;
    float hi = 0.f, mid = 0.f, lo = 0.f;
    static __device__ __forceinline__ Wide prod(float a, float b) {
        const float p = __fmul_rn(a, b);
        return {p, __fmaf_rn(a, b, -p), 0.f};
    }
    static __device__ __forceinline__ Wide sum(float a, float b) {
        Wide r;
        r.hi = two_sum(a, b, r.mid);
        return r;
    }
    __device__ __forceinline__ void add_mid(float x) {
        float e;
        mid = two_sum(mid, x, e);
        lo = __fadd_rn(lo, e);
    }
    __device__ __forceinline__ void add(float x) {
        float e;
        hi = two_sum(hi, x, e);
        add_mid(e);
    }
    __device__ __forceinline__ void add_prod(float a, float b) {
        const float p = __fmul_rn(a, b);
        add(p);
        add_mid(__fmaf_rn(a, b, -p));
    }
    __device__ __forceinline__ void add(const Wide& o) {
        add(o.hi);
        add_mid(o.mid);
        lo = __fadd_rn(lo, o.lo);
    }
    __device__ __forceinline__ Wide times(float s) const {
        Wide r = prod(hi, s);
        const float q = __fmul_rn(mid, s);
        r.lo = __fmaf_rn(lo, s, __fmaf_rn(mid, s, -q));
        r.add_mid(q);
        return r;
    }
    __device__ __forceinline__ Wide square() const {
        Wide r = prod(hi, hi);
        const float h2 = __fadd_rn(hi, hi), q = __fmul_rn(h2, mid);
        r.lo = __fmaf_rn(h2, lo, __fmaf_rn(mid, mid, __fmaf_rn(h2, mid, -q)));
        r.add_mid(q);
        return r;
    }
    __device__ __forceinline__ Wide shfl_down(int o) const {
        return {__shfl_down_sync(0xffffffffu, hi, o), __shfl_down_sync(0xffffffffu, mid, o), __shfl_down_sync(0xffffffffu, lo, o)};
    }
    __device__ __forceinline__ stored store() const { return make_float3(hi, mid, lo); }
    static __device__ __forceinline__ Wide load(stored s) { return {s.x, s.y, s.z}; }
    // an infinite sum stays infinite: its rounding errors (inf - inf) say nothing
    __device__ __forceinline__ double value() const { return isfinite(hi) ? (double)hi + ((double)mid + (double)lo) : (double)hi; }
};
// Whether the value of an FP32 context's Wide sum can be taken as it is: finite,
// and so large that products below the range of floats (2^-149 each) are no
// part of it. zero_ok: whether a zero is known to be no such loss.
template <typename T> inline bool wide_in_range(double v, bool zero_ok) {
    return sizeof(T) == 8 || (v - v == 0.0 && (v == 0.0 ? zero_ok : v > 0x1p-60 || v < -0x1p-60));
}

// Sums of the K values over a block (whole warps, up to 32), in a fixed order;
// out(k, sum) is called by one thread for each k.
template <int K, typename T, class Out> __device__ __forceinline__ void block_sum(Wide<T> (&acc)[K], Out out) {
    __shared__ typename Wide<T>::stored red[K][32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, warps = blockDim.x >> 5;
#pragma unroll
    for (int k = 0; k < K; ++k) {
        for (int o = 16; o > 0; o >>= 1) acc[k].add(acc[k].shfl_down(o));
        if (lane == 0) red[k][wid] = acc[k].store();
    }
    __syncthreads();
    for (int k = wid; k < K; k += warps) {
        Wide<T> s;
        if (lane < warps) s = Wide<T>::load(red[k][lane]);
        for (int o = 16; o > 0; o >>= 1) s.add(s.shfl_down(o));
        if (lane == 0) out(k, s.value());
    }
}

// out[k] = sum of component k = blockIdx.x of the K-component block sums.
static __global__ void __launch_bounds__(1024) sum_partials(const double* __restrict__ partials, int n_blocks, int K,
                                                            double* __restrict__ out) {
    Wide<double> acc[1];
    const int k = blockIdx.x;
#pragma unroll 4
    for (int b = threadIdx.x; b < n_blocks; b += blockDim.x) acc[0].add(partials[(size_t)b * K + k]);
    block_sum<1, double>(acc, [&](int, double s) { out[k] = s; });
}

// Tiles of the bead kernel: beads are binned by 8x8x8 grid cells.
constexpr int kTile = 8;
constexpr int kTileCells = kTile * kTile * kTile;

// ---------------------------------------------------------------- Philox

// Philox4x32-10 (Salmon, Moraes, Dror & Shaw, SC'11): multipliers
// 0xD2511F53 / 0xCD9E8D57, Weyl key increments 0x9E3779B9 / 0xBB67AE85.
struct u32x4 {
    uint32_t x, y, z, w;
};

__device__ __forceinline__ u32x4 philox4x32_10(u32x4 c, uint32_t k0, uint32_t k1) {
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        const uint32_t lo0 = 0xD2511F53u * c.x;
        const uint32_t hi0 = __umulhi(0xD2511F53u, c.x);
        const uint32_t lo1 = 0xCD9E8D57u * c.z;
        const uint32_t hi1 = __umulhi(0xCD9E8D57u, c.z);
        c = {hi1 ^ c.y ^ k0, lo1, hi0 ^ c.w ^ k1, lo0};
        k0 += 0x9E3779B9u;
        k1 += 0xBB67AE85u;
    }
    return c;
}

// Three standard normals for (bead id, step) from one Philox block:
// u_j = (x_j + 1/2) 2^-32, Box-Muller on (u0, u1) gives two normals and
// sqrt(-2 ln u2) cos(2 pi u3) the third.
template <typename T> struct normal3 {
    T a, b, c;
};

__device__ __forceinline__ normal3<float> gaussian3(uint32_t id, uint64_t step, uint64_t seed, float) {
    const u32x4 r = philox4x32_10({id, (uint32_t)step, (uint32_t)(step >> 32), 0u}, (uint32_t)seed,
                                  (uint32_t)(seed >> 32));
    const float s = 2.3283064365386963e-10f;  // 2^-32
    const float u0 = fmaf((float)r.x, s, 0.5f * s);
    const float u1 = fmaf((float)r.y, s, 0.5f * s);
    const float u2 = fmaf((float)r.z, s, 0.5f * s);
    const float u3 = fmaf((float)r.w, s, 0.5f * s);
    // CUDA's fast log and sine/cosine intrinsics (absolute errors near
    // 1e-6); the angle 2 pi u - pi lies in their accurate range [-pi, pi],
    // and sin, cos of 2 pi u are minus those of 2 pi u - pi
    const float m1 = sqrtf(fmaxf(-2.0f * __logf(u0), 0.0f));
    const float m2 = sqrtf(fmaxf(-2.0f * __logf(u2), 0.0f));
    float s1, c1, s3, c3;
    __sincosf(fmaf(6.28318530717958648f, u1, -3.14159265358979324f), &s1, &c1);
    __sincosf(fmaf(6.28318530717958648f, u3, -3.14159265358979324f), &s3, &c3);
    return {-m1 * c1, -m1 * s1, -m2 * c3};
}

__device__ __forceinline__ normal3<double> gaussian3(uint32_t id, uint64_t step, uint64_t seed, double) {
    const u32x4 r = philox4x32_10({id, (uint32_t)step, (uint32_t)(step >> 32), 0u}, (uint32_t)seed,
                                  (uint32_t)(seed >> 32));
    const double s = 2.3283064365386962890625e-10;  // 2^-32
    const double u0 = ((double)r.x + 0.5) * s;
    const double u1 = ((double)r.y + 0.5) * s;
    const double u2 = ((double)r.z + 0.5) * s;
    const double u3 = ((double)r.w + 0.5) * s;
    const double m1 = sqrt(-2.0 * log(u0));
    const double m2 = sqrt(-2.0 * log(u2));
    double s1, c1, s3, c3;
    sincospi(2.0 * u1, &s1, &c1);
    sincospi(2.0 * u3, &s3, &c3);
    return {m1 * c1, m1 * s1, m2 * c3};
}

// Periodic grid index for j in [-n, 2n) (any n; stencils and patches never
// reach further than one period).
__host__ __device__ __forceinline__ int pwrap(int j, int n) { return j < 0 ? j + n : (j >= n ? j - n : j); }

// ------------------------------------------------- assignment weights

// floor(s) as a value and as an integer. FP32 (|s| < 2^22; grid coordinates are
// at most a few hundred): the sum with 1.5 2^23 rounded down holds the integer
// in its low bits, without the slow conversion and rounding instructions.
__device__ __forceinline__ float floor_int(float s, int& j) {
    const float r = __fadd_rd(s, 12582912.0f);
    j = __float_as_int(r) - 0x4B400000;
    return __fsub_rn(r, 12582912.0f);
}
__device__ __forceinline__ double floor_int(double s, int& j) {
    const double f = floor(s);
    j = (int)f;
    return f;
}
// round to nearest (even) of a x b, |a b| < 2^22 in FP32
__device__ __forceinline__ float round_prod(float a, float b) { return __fsub_rn(__fmaf_rn(a, b, 12582912.0f), 12582912.0f); }
__device__ __forceinline__ double round_prod(double a, double b) { return rint(a * b); }

// Charge-assignment weights of order P (P points per dimension), the
// closed-form polynomials of Deserno & Holm (J. Chem. Phys. 109, 7678,
// 1998, appendix) cited by the paper for its spline weights. s is the
// position in grid units; j0 receives the first grid point (not wrapped).
// Even P: t = s - floor(s) in [0, 1), points floor(s)-P/2+1 .. floor(s)+P/2.
// Odd P:  t = s - floor(s + 1/2) in [-1/2, 1/2), points centred on the
//         nearest grid point.
template <int P, typename T> __device__ __forceinline__ void dh_weights(T s, int& j0, T (&w)[P]) {
    if constexpr (P == 2) {
        const T t = s - floor_int(s, j0);
        w[0] = T(1) - t;
        w[1] = t;
    } else if constexpr (P == 3) {
        const T t = s - floor_int(s + T(0.5), j0);
        --j0;
        w[0] = T(0.5) * (T(0.5) - t) * (T(0.5) - t);
        w[1] = T(0.75) - t * t;
        w[2] = T(0.5) * (T(0.5) + t) * (T(0.5) + t);
    } else if constexpr (P == 4) {
        const T t = s - floor_int(s, j0);
        const T t2 = t * t, t3 = t2 * t, u = T(1) - t;
        --j0;
        w[0] = u * u * u * T(1.0 / 6.0);
        w[1] = (T(4) - T(6) * t2 + T(3) * t3) * T(1.0 / 6.0);
        w[2] = (T(1) + T(3) * t + T(3) * t2 - T(3) * t3) * T(1.0 / 6.0);
        w[3] = t3 * T(1.0 / 6.0);
    } else {
        static_assert(P == 5, "orders 1..4 (P = 2..5)");
        const T t = s - floor_int(s + T(0.5), j0);
        const T t2 = t * t, t3 = t2 * t, t4 = t2 * t2;
        const T a = T(1) - T(2) * t, b = T(1) + T(2) * t;
        j0 -= 2;
        w[0] = a * a * a * a * T(1.0 / 384.0);
        w[1] = (T(19) - T(44) * t + T(24) * t2 + T(16) * t3 - T(16) * t4) * T(1.0 / 96.0);
        w[2] = (T(115) - T(120) * t2 + T(48) * t4) * T(1.0 / 192.0);
        w[3] = (T(19) + T(44) * t + T(24) * t2 - T(16) * t3 - T(16) * t4) * T(1.0 / 96.0);
        w[4] = b * b * b * b * T(1.0 / 384.0);
    }
}

// d/ds of the weights of dh_weights (same points).
template <int P, typename T> __device__ __forceinline__ void dh_weight_derivs(T s, T (&dw)[P]) {
    if constexpr (P == 2) {
        dw[0] = T(-1);
        dw[1] = T(1);
    } else if constexpr (P == 3) {
        const T t = s - floor(s + T(0.5));
        dw[0] = t - T(0.5);
        dw[1] = T(-2) * t;
        dw[2] = T(0.5) + t;
    } else if constexpr (P == 4) {
        const T t = s - floor(s);
        const T u = T(1) - t;
        dw[0] = T(-0.5) * u * u;
        dw[1] = T(-2) * t + T(1.5) * t * t;
        dw[2] = T(0.5) + t - T(1.5) * t * t;
        dw[3] = T(0.5) * t * t;
    } else {
        const T t = s - floor(s + T(0.5));
        const T t2 = t * t, t3 = t2 * t;
        const T a = T(1) - T(2) * t, b = T(1) + T(2) * t;
        dw[0] = -a * a * a * T(1.0 / 48.0);
        dw[1] = (T(-44) + T(48) * t + T(48) * t2 - T(64) * t3) * T(1.0 / 96.0);
        dw[2] = T(-1.25) * t + t3;
        dw[3] = (T(44) + T(48) * t - T(48) * t2 - T(64) * t3) * T(1.0 / 96.0);
        dw[4] = b * b * b * T(1.0 / 48.0);
    }
}

// Stencil extent relative to the cell floor(s): points floor(s)+lo ..
// floor(s)+hi can receive weight.
template <int P> struct stencil_extent {
    static constexpr int lo = (P % 2 == 0) ? -(P / 2 - 1) : -((P - 1) / 2);
    static constexpr int hi = (P % 2 == 0) ? (P / 2) : ((P - 1) / 2 + 1);
};

// ------------------------------------------------------ chain topology

constexpr int kMaxTypes = 8;

// Linear chains numbered type by type (see tild.h). Passed by value to the
// kernels that need species or bonded neighbours of a bead id.
struct Topology {
    int n_types;
    int start[kMaxTypes + 1];  // first bead id of each type (n_beads < 2^31)
    int N[kMaxTypes];
    int n_a[kMaxTypes];
};

struct BeadInfo {
    int species;
    int prev;  // id of the bonded predecessor or -1
    int next;  // id of the bonded successor or -1
};

__host__ __device__ __forceinline__ BeadInfo bead_info(const Topology& t, int id) {
    int k = 0;
    while (k + 1 < t.n_types && id >= t.start[k + 1]) ++k;
    const int s = (id - t.start[k]) % t.N[k];
    BeadInfo b;
    b.species = s < t.n_a[k] ? 0 : 1;
    b.prev = s > 0 ? id - 1 : -1;
    b.next = s < t.N[k] - 1 ? id + 1 : -1;
    return b;
}

// Error flags raised by kernels (read by the host on demand).
constexpr unsigned kErrNonFinite = 1u;
constexpr unsigned kErrBounds = 2u;  // a bounds check of the debug build failed

// Debug build (compiled with -DTILD_DEBUG=1, `_build.build(debug=True)`):
// the bead kernels, tiled and per bead, and the adjoint kernels check bead ids,
// slots, species and grid indices before they use them; a failed check records
// kErrBounds in the context's error word and the access is skipped (no trap),
// and the next synchronising call returns TILD_EDEVICE. In the normal build
// every check is the constant true.
#ifndef TILD_DEBUG
#define TILD_DEBUG 0
#endif
__device__ __forceinline__ bool debug_check(bool ok, unsigned int* err) {
#if TILD_DEBUG
    if (!ok) atomicOr(err, kErrBounds);
    return ok;
#else
    (void)err;
    return true;
#endif
}

}  // namespace tild
