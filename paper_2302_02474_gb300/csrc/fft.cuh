// Hand-written FFT building blocks for lengths 8..256 that split as
// N = N1 * N2 with N1 in {4, 8, 16} and N2 in {1, 3, 4, 5, 8, 16}
// (powers of two, 24, 40, 48, 80).
//
// A length-N transform is split N = N1 * N2 (four-step / Cooley-Tukey):
//   input index  j = j2 + N2 * j1,  output index k = k1 + N1 * k2,
//   X[k1 + N1 k2] = sum_j2 W_N^{j2 k1} W_N2^{j2 k2} sum_j1 x[j2 + N2 j1] W_N1^{j1 k1}.
// Stage A does the N1-point DFTs over j1 in registers and applies the
// twiddle W_N^{j2 k1}; stage B does the N2-point DFTs over j2 in registers
// and writes the result in natural order. Lines live in shared memory; the
// thread-to-data mapping puts consecutive threads on consecutive lines so
// that every shared-memory access of a warp touches consecutive lines at
// the same offset (conflict-free when the line stride is odd in 8-byte
// words, or 1).
//
// Sign convention: forward (DIR = -1) uses exp(-2 pi i jk/N), inverse
// (DIR = +1) exp(+2 pi i jk/N); neither is normalised.
#pragma once

#include "common.cuh"

namespace tild {

// ------------------------------------------------------------- radices

template <int N> struct fft_split;
template <> struct fft_split<8> { static constexpr int N1 = 8, N2 = 1; };
template <> struct fft_split<16> { static constexpr int N1 = 4, N2 = 4; };
template <> struct fft_split<32> { static constexpr int N1 = 8, N2 = 4; };
template <> struct fft_split<64> { static constexpr int N1 = 8, N2 = 8; };
template <> struct fft_split<128> { static constexpr int N1 = 16, N2 = 8; };
template <> struct fft_split<256> { static constexpr int N1 = 16, N2 = 16; };
template <> struct fft_split<24> { static constexpr int N1 = 8, N2 = 3; };
template <> struct fft_split<40> { static constexpr int N1 = 8, N2 = 5; };
template <> struct fft_split<48> { static constexpr int N1 = 16, N2 = 3; };
template <> struct fft_split<80> { static constexpr int N1 = 16, N2 = 5; };

// Multiply v by W_16^m = exp(DIR * 2 pi i m / 16), a factor of the R-point
// radix (R = 8, 16); m is a compile-time constant after unrolling, so the
// branches fold away. Which product of a sum is rounded by itself is part of
// the transform's definition here: sums that nearly cancel, as the parameter
// derivatives of a force product do, show the last bits of a spectrum, and a
// spectrum is the same bits whatever kernel computes it.
template <int DIR, int R, class V> __device__ __forceinline__ V w16_mul(int m, V v) {
    using T = decltype(v.x);
    const T c1 = T(0.92387953251128675613), s1 = T(0.38268343236508977173);  // cos, sin(pi/8)
    const T h = T(0.70710678118654752440);                                    // cos(pi/4)
    m &= 15;
    // value of exp(-2 pi i m / 16) = (cr, ci); inverse uses the conjugate
    T cr, ci;
    switch (m) {
        case 0: return v;
        case 4: return DIR < 0 ? c_mul_negi(v) : c_mul_posi(v);
        case 8: return {-v.x, -v.y};
        case 12: return DIR < 0 ? c_mul_posi(v) : c_mul_negi(v);
        case 1: cr = c1; ci = -s1; break;
        case 2: cr = h; ci = -h; break;
        case 3: cr = s1; ci = -c1; break;
        case 5: cr = -s1; ci = -c1; break;
        case 6: cr = -h; ci = -h; break;
        case 7: cr = -c1; ci = -s1; break;
        case 9: cr = -c1; ci = s1; break;
        case 10: cr = -h; ci = h; break;
        case 11: cr = -s1; ci = c1; break;
        case 13: cr = s1; ci = c1; break;
        case 14: cr = h; ci = h; break;
        default: cr = c1; ci = s1; break;  // 15
    }
    if (DIR > 0) ci = -ci;
    if (m % 4 != 2) return c_mul(v, V{cr, ci});
    // odd multiples of pi/4
    const bool x_first = DIR < 0 ? R == 16 || m == 2 : R == 8 || m == 6, y_first = R == 16 ? m == 6 : m == 2;
    return {x_first ? fma_rn(v.x, cr, -mul_rn(v.y, ci)) : fma_rn(-v.y, ci, mul_rn(v.x, cr)),
            y_first ? fma_rn(v.x, ci, mul_rn(v.y, cr)) : fma_rn(v.y, cr, mul_rn(v.x, ci))};
}

// In-register DFT of R points (R = 1, 2, 4, 8, 16 by radix-2 decimation in
// time; 3 and 5 directly), natural order in and out.
template <int R, int DIR, class V> struct reg_dft {
    static __device__ __forceinline__ void run(V (&v)[R]) {
        V e[R / 2], o[R / 2];
#pragma unroll
        for (int i = 0; i < R / 2; ++i) {
            e[i] = v[2 * i];
            o[i] = v[2 * i + 1];
        }
        reg_dft<R / 2, DIR, V>::run(e);
        reg_dft<R / 2, DIR, V>::run(o);
#pragma unroll
        for (int k = 0; k < R / 2; ++k) {
            const V t = w16_mul<DIR, R>(k * (16 / R), o[k]);
            v[k] = c_add(e[k], t);
            v[k + R / 2] = c_sub(e[k], t);
        }
    }
};
template <int DIR, class V> struct reg_dft<1, DIR, V> {
    static __device__ __forceinline__ void run(V (&)[1]) {}
};

// 3 points: X1,2 = x0 + cos(2pi/3)(x1 + x2) +/- i DIR' sin(2pi/3)(x1 - x2),
// with the sign of the exponent DIR.
template <int DIR, class V> struct reg_dft<3, DIR, V> {
    static __device__ __forceinline__ void run(V (&v)[3]) {
        using T = decltype(v[0].x);
        const T c = T(-0.5), s = T(DIR) * T(0.86602540378443864676);  // DIR sin(2 pi / 3)
        const V t1 = c_add(v[1], v[2]), t3 = c_sub(v[1], v[2]);
        const V m = {fma_rn(c, t1.x, v[0].x), fma_rn(c, t1.y, v[0].y)};
        v[0] = c_add(v[0], t1);
        v[1] = {fma_rn(-s, t3.y, m.x), fma_rn(s, t3.x, m.y)};  // m +- i s (x1 - x2)
        v[2] = {fma_rn(s, t3.y, m.x), fma_rn(-s, t3.x, m.y)};
    }
};

// 5 points with t1 = x1 + x4, t2 = x2 + x3, t3 = x1 - x4, t4 = x2 - x3:
// X1,4 = x0 + c1 t1 + c2 t2 +/- i (s1 t3 + s2 t4), X2,3 = x0 + c2 t1 + c1 t2
// +/- i (s2 t3 - s1 t4), c_k = cos(2 pi k / 5), s_k = DIR sin(2 pi k / 5).
template <int DIR, class V> struct reg_dft<5, DIR, V> {
    static __device__ __forceinline__ void run(V (&v)[5]) {
        using T = decltype(v[0].x);
        const T c1 = T(0.30901699437494742410), c2 = T(-0.80901699437494742410);
        const T s1 = T(DIR) * T(0.95105651629515357212), s2 = T(DIR) * T(0.58778525229247312917);
        const V t1 = c_add(v[1], v[4]), t2 = c_add(v[2], v[3]);
        const V t3 = c_sub(v[1], v[4]), t4 = c_sub(v[2], v[3]);
        const V a = {fma_rn(c2, t2.x, fma_rn(c1, t1.x, v[0].x)), fma_rn(c2, t2.y, fma_rn(c1, t1.y, v[0].y))};
        const V b = {fma_rn(c1, t2.x, fma_rn(c2, t1.x, v[0].x)), fma_rn(c1, t2.y, fma_rn(c2, t1.y, v[0].y))};
        const V p = {fma_rn(s1, t3.x, mul_rn(s2, t4.x)), fma_rn(s1, t3.y, mul_rn(s2, t4.y))};
        const V q = {fma_rn(s2, t3.x, -mul_rn(s1, t4.x)), fma_rn(s2, t3.y, -mul_rn(s1, t4.y))};
        const V ip = {-p.y, p.x}, iq = {-q.y, q.x};
        v[0] = {v[0].x + t1.x + t2.x, v[0].y + t1.y + t2.y};
        v[1] = c_add(a, ip);
        v[4] = c_sub(a, ip);
        v[2] = c_add(b, iq);
        v[3] = c_sub(b, iq);
    }
};

// Twiddle table W_N^m = exp(-2 pi i m / N), m in [0, N), computed on the
// host in FP64 and rounded to T; copied to shared memory by each CTA.
template <int DIR, class V> __device__ __forceinline__ V twiddle(const V* tw, int m) {
    const V w = tw[m];
    return DIR < 0 ? w : c_conj(w);
}

// ----------------------------------------------------- line transforms

// FFT of NLINES lines of length N held in shared memory. Element e of
// line l lives at buf[addr(l) + e * es]. All NTHR threads of the CTA call
// this; it ends with __syncthreads(). Stage B keeps all of its work units
// in registers (UPT per thread), so one round covers every line.
// Stage A of smem_fft_lines alone (ends with __syncthreads()): unit
// (line, j2) transforms x[j2 + N2 j1] over j1 and applies W_N^{j2 k1}.
template <int N, int DIR, int NLINES, int NTHR, class V, class Addr>
__device__ __forceinline__ void smem_fft_stage_a(V* buf, Addr addr, int es, const V* tw) {
    constexpr int N1 = fft_split<N>::N1;
    constexpr int N2 = fft_split<N>::N2;
    // Stage A: unit (line, j2); reads and writes only its own positions.
    for (int u = threadIdx.x; u < NLINES * N2; u += NTHR) {
        const int l = u % NLINES;
        const int j2 = u / NLINES;
        V* p = buf + addr(l) + j2 * es;
        V v[N1];
#pragma unroll
        for (int j1 = 0; j1 < N1; ++j1) v[j1] = p[j1 * N2 * es];
        reg_dft<N1, DIR, V>::run(v);
        if (N2 > 1) {
#pragma unroll
            for (int k1 = 1; k1 < N1; ++k1) v[k1] = c_mul(v[k1], twiddle<DIR>(tw, j2 * k1));
        }
#pragma unroll
        for (int k1 = 0; k1 < N1; ++k1) p[k1 * N2 * es] = v[k1];
    }
    __syncthreads();
}

template <int N, int DIR, int NLINES, int NTHR, class V, class Addr>
__device__ __forceinline__ void smem_fft_lines(V* buf, Addr addr, int es, const V* tw) {
    constexpr int N1 = fft_split<N>::N1;
    constexpr int N2 = fft_split<N>::N2;
    constexpr int nthr = NTHR;
    constexpr int UPT = (NLINES * N1 + NTHR - 1) / NTHR;
    const int tid = threadIdx.x;

    smem_fft_stage_a<N, DIR, NLINES, NTHR>(buf, addr, es, tw);
    if (N2 == 1) return;

    // Stage B: unit (line, k1) reads the N2 positions j2 + N2 k1 and writes
    // X[k1 + N1 k2]; positions overlap other units, so every unit of a
    // round is loaded before any is stored.
    {
        constexpr int l0 = 0;
        constexpr int nl = NLINES;
        V v[UPT][N2];
#pragma unroll
        for (int r = 0; r < UPT; ++r) {
            const int u = tid + r * nthr;
            if (u < nl * N1) {
                const int l = l0 + u % nl;
                const int k1 = u / nl;
                const V* p = buf + addr(l) + k1 * N2 * es;
#pragma unroll
                for (int j2 = 0; j2 < N2; ++j2) v[r][j2] = p[j2 * es];
            }
        }
        __syncthreads();
#pragma unroll
        for (int r = 0; r < UPT; ++r) {
            const int u = tid + r * nthr;
            if (u < nl * N1) {
                const int l = l0 + u % nl;
                const int k1 = u / nl;
                reg_dft<N2, DIR, V>::run(v[r]);
                V* p = buf + addr(l) + k1 * es;
#pragma unroll
                for (int k2 = 0; k2 < N2; ++k2) p[k2 * N1 * es] = v[r][k2];
            }
        }
        __syncthreads();
    }
}

// ------------------------------------------------- register-first stages
//
// The passes of the step run each stage of a line transform as one visit of
// shared memory: the first stage takes its inputs straight from global
// memory (or from the registers of the stage before), and the last one hands
// its outputs straight to global memory. Every stage works in place: unit
// (line, j2) of stage A owns the slots k1 N2 + j2 and unit (line, k1) of stage
// B the slots k1 N2 + j2, so a stage reads and writes its own slots only and
// needs no barrier in between, its units can run one after the other (small
// code, few registers), and one barrier separates two stages. The price is
// that the transform is left in the order slot k1 N2 + k2 <-> X[k1 + N1 k2],
// which the consumer of the lines undoes in its addressing.
//
// Rows of a plane keep slot i at i XOR swz(i) (the low bits of an even N2, with
// bits of k1), so that lanes over k1 at one j2 and lanes over consecutive slots
// both fall into distinct banks (16 lanes of 8-byte words); padding a row after
// every N2 slots made every access along columns a two-way conflict. Rows are
// N2 modulo 16 words apart, for lanes over (j2, row). Odd N2 need neither.
template <int N> struct LineSlots {
    static constexpr int N1 = fft_split<N>::N1, N2 = fft_split<N>::N2;
    static constexpr int make_pitch() {
        int p = N;
        while (p % 16 != N2 % 16) ++p;
        return p;
    }
    static constexpr int pitch = make_pitch();
    static __device__ __forceinline__ int swz(int i) {
        if constexpr (N2 == 16)
            return (i >> 4) & 15;
        else if constexpr (N2 == 8)
            return (N1 == 16 ? i >> 4 : i >> 3) & 7;
        else if constexpr (N2 == 4)
            return (i >> 4) & 3;
        else
            return 0;
    }
    // position of slot i in a row
    static __device__ __forceinline__ int at(int i) { return i ^ swz(i); }
    // the slot that holds X[k] after stage B, and its inverse
    static __device__ __forceinline__ int slot_of(int k) { return (k % N1) * N2 + k / N1; }
    static __device__ __forceinline__ int index_of(int slot) { return slot / N2 + N1 * (slot % N2); }
    // slot_of(j + N2 m), j < N2; where N2 divides N1 the parts of j and m separate,
    // so that unrolled accesses over either share one address
    static __device__ __forceinline__ int slot_of_part(int j, int m) {
        if constexpr (N1 % N2 == 0)
            return j * N2 + (m % (N1 / N2)) * N2 * N2 + m / (N1 / N2);
        else
            return slot_of(j + N2 * m);
    }
};

// v * s with each product rounded by itself: the same bits in every pass that
// scales a field.
template <class V, typename T> __device__ __forceinline__ V c_scale_rn(V v, T s) { return {mul_rn(v.x, s), mul_rn(v.y, s)}; }

// Stage A of one unit in registers: the N1-point DFT over j1 and the twiddle
// W_N^{j2 k1}.
template <int N, int DIR, class V>
__device__ __forceinline__ void stage_a_regs(V (&v)[fft_split<N>::N1], int j2, const V* tw) {
    constexpr int N1 = fft_split<N>::N1;
    reg_dft<N1, DIR, V>::run(v);
    if (fft_split<N>::N2 > 1) {
#pragma unroll
        for (int k1 = 1; k1 < N1; ++k1) v[k1] = c_mul(v[k1], twiddle<DIR>(tw, j2 * k1));
    }
}

// Grid sizes whose xy-plane of values of `bytes` fits the shared memory of one
// CTA (FP32 up to 128, FP64 up to 80).
__host__ __device__ constexpr bool plane_fits(int n, int bytes) { return n * (n + 1) * bytes <= 200 * 1024; }

}  // namespace tild
