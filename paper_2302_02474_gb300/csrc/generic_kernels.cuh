// Grid and bead kernels for any grid size and for two-dimensional boxes
// (Sec. "TILD Branch": periodic boxes in two or three dimensions; Listing
// infile runs D = 2 on a 65 x 65 grid). The same method as the tiled path,
// organised for any size:
//   - beads: one thread per bead (no tiles or shared patches); the density
//     is accumulated with 64-bit fixed-point global atomics, so it is as
//     bit-reproducible as the tiled path's;
//   - FFT: each line is transformed in two factors n = n1 n2 (Cooley-Tukey)
//     with direct DFTs of lengths n1 and n2 and one twiddle table of length n,
//     so odd sizes (65 = 5 x 13, 45, 75, primes) need no special radix;
//   - step passes ("Line passes" below): the x pass reads the densities, the
//     pass of the last axis transforms, multiplies and transforms back, and
//     the x and y dimensions stay in the order their transform leaves them in;
//   - whole-axis passes with a separate spectral multiply (one thread per
//     wavevector): the spectrum read-out, and lines too long for the fused
//     last pass.
// Grids are [..][nz][n][n] with nz = n (D = 3) or 1 (D = 2); spectra are
// complex, species pairs packed as in the tiled path (rho_2p + i rho_2p+1).
#pragma once

#include "bead_kernels.cuh"
#include "grid_kernels.cuh"

namespace tild {

// ---------------------------------------------------------------- FFT

// Twiddle W_n^m for any m >= 0 (the table holds exp(-2 pi i m/n), m < n).
template <int DIR, class V> __device__ __forceinline__ V gtw(const V* tw, int m) {
    const V w = tw[m];
    return DIR < 0 ? w : c_conj(w);
}

// Transform the lines of one tile along `axis` (0 = x, 1 = y, 2 = z) of
// `fields` complex arrays [F][nz][n][n]. A CTA takes C lines that are
// adjacent in x (axis y or z) or adjacent rows (axis x) and keeps them in
// shared memory as buf[line][j] (pitch n + 1), with a second buffer for the
// intermediate of the two-factor transform:
//   t[j2 + n2 k1] = W_n^{j2 k1} sum_j1 x[j2 + n2 j1] W_n^{n2 j1 k1},
//   X[k1 + n1 k2] = sum_j2 t[j2 + n2 k1] W_n^{n1 j2 k2}.
// grid.x = tiles of lines per field, grid.y = field.
template <typename T, int DIR>
__global__ void __launch_bounds__(256) generic_axis_fft(cplx_t<T>* __restrict__ data, int n, int nz, int axis, int C,
                                                        int n1, int n2, const cplx_t<T>* __restrict__ tw_g) {
    using V = cplx_t<T>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    V* tw = reinterpret_cast<V*>(smem_raw);
    const int pitch = n + 1;
    V* buf = tw + n;
    V* tmp = buf + (size_t)C * pitch;
    for (int i = threadIdx.x; i < n; i += blockDim.x) tw[i] = tw_g[i];
    const size_t M = (size_t)nz * n * n;
    V* f = data + (size_t)blockIdx.y * M;
    // line l of this tile: start offset and element stride
    const size_t stride = axis == 0 ? 1 : axis == 1 ? (size_t)n : (size_t)n * n;
    const int lines_per_field = (int)(M / n);
    const int l0 = blockIdx.x * C;
    auto line_start = [&](int l) -> size_t {
        // lines are numbered so that consecutive numbers are adjacent in x
        // (axes y, z) or consecutive rows (axis x)
        if (axis == 0) return (size_t)l * n;
        if (axis == 1) {
            const int x = l % n, z = l / n;
            return (size_t)z * n * n + x;
        }
        return (size_t)l;  // axis 2: l = y n + x
    };
    const int nl = min(C, lines_per_field - l0);
    for (int i = threadIdx.x; i < nl * n; i += blockDim.x) {
        // consecutive threads: consecutive lines (axes y, z) or consecutive elements (axis x)
        int l, j;
        if (axis == 0) {
            l = i / n;
            j = i % n;
        } else {
            l = i % nl;
            j = i / nl;
        }
        buf[l * pitch + j] = f[line_start(l0 + l) + (size_t)j * stride];
    }
    __syncthreads();
    // stage A
    for (int u = threadIdx.x; u < nl * n; u += blockDim.x) {
        const int l = u % nl, r = u / nl;
        const int k1 = r % n1, j2 = r / n1;
        const V* x = buf + l * pitch;
        V acc = {T(0), T(0)};
        int m = 0;
        const int step = (n2 * k1) % n;
        for (int j1 = 0; j1 < n1; ++j1) {
            acc = c_add(acc, c_mul(x[j2 + n2 * j1], gtw<DIR>(tw, m)));
            m += step;
            if (m >= n) m -= n;
        }
        tmp[l * pitch + j2 + n2 * k1] = c_mul(acc, gtw<DIR>(tw, (j2 * k1) % n));
    }
    __syncthreads();
    // stage B
    for (int u = threadIdx.x; u < nl * n; u += blockDim.x) {
        const int l = u % nl, r = u / nl;
        const int k1 = r % n1, k2 = r / n1;
        const V* t = tmp + l * pitch;
        V acc = {T(0), T(0)};
        int m = 0;
        const int step = (n1 * k2) % n;
        for (int j2 = 0; j2 < n2; ++j2) {
            acc = c_add(acc, c_mul(t[j2 + n2 * k1], gtw<DIR>(tw, m)));
            m += step;
            if (m >= n) m -= n;
        }
        buf[l * pitch + k1 + n1 * k2] = acc;
    }
    __syncthreads();
    for (int i = threadIdx.x; i < nl * n; i += blockDim.x) {
        int l, j;
        if (axis == 0) {
            l = i / n;
            j = i % n;
        } else {
            l = i % nl;
            j = i / nl;
        }
        f[line_start(l0 + l) + (size_t)j * stride] = buf[l * pitch + j];
    }
}

// Fixed-point densities [2 NP][M] -> complex pairs Z_p = rho_2p + i rho_2p+1
// ([NP][M]); zero the fixed-point grid when asked. A step's first kernel
// advances the noise counter.
template <typename T>
__global__ void generic_load_density(size_t M, int np, unsigned long long* __restrict__ rho_fx, cplx_t<T>* __restrict__ Z,
                                     T scale, int zero_after, unsigned long long* step_ctr) {
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (step_ctr && i == 0) *step_ctr += 1ull;
    if (i >= (size_t)np * M) return;
    const size_t p = i / M, g = i % M;
    unsigned long long* a = rho_fx + 2 * p * M + g;
    unsigned long long* b = a + M;
    const long long va = (long long)*a, vb = (long long)*b;
    if (zero_after) {
        *a = 0ull;
        *b = 0ull;
    }
    Z[i] = cplx_t<T>{from_fixed(va, scale), from_fixed(vb, scale)};
}

// Spectral multiply over the whole spectrum, one thread per wavevector k:
// species spectra from the packed pairs (Hermitian separation with Z(-k)),
// w~_K = u_hat(k) sum_K' eps_KK' rho~_K', and per pair
//   out[p][d] = i k~_d Q_p (d < D; k~ with the Nyquist index zeroed),
//   Q_p = w~_2p + i w~_2p+1.
// Energy partials per block as in the z pass: [0] sum u_hat Re[conj(rho~_0)
// rho~_1] (one pair) or the chi-weighted sum over species pairs (two
// pairs), [1] sum_{k != 0} u_hat |sum_K rho~_K|^2 (rho~ times e_rho), the
// others 0. u_hat = e1[kx] e1[ky] (e1[kz]).
template <typename T, int NP>
__global__ void __launch_bounds__(256) generic_spectral(const cplx_t<T>* __restrict__ Z, cplx_t<T>* __restrict__ out,
                                                        int n, int nz, SpectralParams<T> sp,
                                                        double* __restrict__ partials) {
    using V = cplx_t<T>;
    const size_t M = (size_t)nz * n * n;
    const size_t g = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    Wide<T> acc[5];
    if (g < M) {
        const int x = (int)(g % n), y = (int)((g / n) % n), z = (int)(g / ((size_t)n * n));
        const int mx = x == 0 ? 0 : n - x, my = y == 0 ? 0 : n - y, mz = z == 0 ? 0 : nz - z;
        const size_t gm = ((size_t)mz * n + my) * n + mx;
        auto freq = [&](int i, int len) { return (T)(2 * i < len ? i : i - len); };  // 2 i == len: -len/2
        auto kgrad = [&](int i, int len) { return (len % 2 == 0 && 2 * i == len) ? T(0) : sp.two_pi_over_L * freq(i, len); };
        const T kd[3] = {kgrad(x, n), kgrad(y, n), nz > 1 ? kgrad(z, nz) : T(0)};
        const T uh = sp.kernel1d[x] * sp.kernel1d[y] * (nz > 1 ? sp.kernel1d[z] : T(1));
        V A[2 * NP];
#pragma unroll
        for (int p = 0; p < NP; ++p) {
            const V Zk = Z[p * M + g], Zm = Z[p * M + gm];
            A[2 * p] = {T(0.5) * (Zk.x + Zm.x), T(0.5) * (Zk.y - Zm.y)};
            A[2 * p + 1] = {T(0.5) * (Zk.y + Zm.y), -T(0.5) * (Zk.x - Zm.x)};
        }
        if (partials) {
            if constexpr (NP == 1)
                add_energies<T, 1>(acc, A[0], A[1], uh, sp.e_rho, T(1), g == 0, T(0));
            else
                add_energies4<T, NP>(acc, A, sp, uh, g == 0);
        }
#pragma unroll
        for (int p = 0; p < NP; ++p) {
            V w[2];
#pragma unroll
            for (int s = 0; s < 2; ++s) {
                const int K = 2 * p + s;
                T wr = 0, wi = 0;
                if (NP == 1) {
                    const T e0 = s == 0 ? sp.eAA : sp.eAB, e1v = s == 0 ? sp.eAB : sp.eBB;
                    wr = e0 * A[0].x + e1v * A[1].x;
                    wi = e0 * A[0].y + e1v * A[1].y;
                } else {
#pragma unroll
                    for (int K2 = 0; K2 < 2 * NP; ++K2) {
                        wr += sp.eps4[K][K2] * A[K2].x;
                        wi += sp.eps4[K][K2] * A[K2].y;
                    }
                }
                w[s] = {uh * wr, uh * wi};
            }
            const V iQ = {-(w[0].y + w[1].x), w[0].x - w[1].y};
            V* o = out + (size_t)4 * p * M;
            o[g] = {kd[0] * iQ.x, kd[0] * iQ.y};
            o[M + g] = {kd[1] * iQ.x, kd[1] * iQ.y};
            if (nz > 1) o[2 * M + g] = {kd[2] * iQ.x, kd[2] * iQ.y};
        }
    }
    if (partials) {
        block_sum<5, T>(acc, [&](int k, double v) { partials[5 * (size_t)blockIdx.x + k] = v; });
    }
}

// ------------------------------------------------------- line passes
//
// Bound by latency at the sizes in use (65^2: 4,225 points; 45^3: 91,125): what
// counts is the number of dependent launches, CTAs on every SM, and short
// serial chains. A thread transforms n1 or n2 points in registers (up to 16;
// symmetric sums halve the products of an odd length twice), CTAs hold as few
// lines as still give the chip about two CTAs per SM, and the index arithmetic
// has no division per element. Stages work in place as those of the tiled
// grids do (see fft.cuh): the forward transform leaves X[k1 + n1 k2] in slot
// k1 n2 + k2 and the inverse starts from there with the factors swapped (n2
// points over k2, twiddle, n1 points over k1, natural order out), so nothing
// reorders the spectrum. Only the last pass needs wavenumbers of slots.
// Step of 5,000 beads on 65^2: 72 -> 19 us in 4 launches (was 7); of 55,000
// beads of three species on 45^3: 163 -> 57 us in 6 launches (was 12).

// cos(2 pi m / R) and sin(2 pi m / R) at compile time (Taylor series on [0, pi/4]).
struct TrigSeries {
    static constexpr double pi = 3.14159265358979323846;
    static constexpr double cos0(double x) {
        double t = 1.0, s = 1.0;
        for (int i = 1; i < 14; ++i) {
            t *= -x * x / ((2 * i - 1) * (2 * i));
            s += t;
        }
        return s;
    }
    static constexpr double sin0(double x) {
        double t = x, s = x;
        for (int i = 1; i < 14; ++i) {
            t *= -x * x / ((2 * i) * (2 * i + 1));
            s += t;
        }
        return s;
    }
    // m in [0, R)
    static constexpr double cosine(int m, int R) {
        if (2 * m > R) m = R - m;
        if (4 * m > R) return -cosine_half(R - 2 * m, 2 * R);
        return cosine_half(2 * m, 2 * R);
    }
    static constexpr double sine(int m, int R) {
        if (2 * m > R) return -sine(R - m, R);
        if (4 * m > R) return sine_quarter(R - 2 * m, 2 * R);
        return sine_quarter(2 * m, 2 * R);
    }
    // angle 2 pi m / R in [0, pi/2]
    static constexpr double cosine_half(int m, int R) {
        return 8 * m > R ? sin0(2 * pi * (R - 4 * m) / (4.0 * R)) : cos0(2 * pi * m / R);
    }
    static constexpr double sine_quarter(int m, int R) {
        return 8 * m > R ? cos0(2 * pi * (R - 4 * m) / (4.0 * R)) : sin0(2 * pi * m / R);
    }
};
template <int R> struct Trig {
    double c[R] = {}, s[R] = {};
    constexpr Trig() {
        for (int m = 0; m < R; ++m) {
            c[m] = TrigSeries::cosine(m, R);
            s[m] = TrigSeries::sine(m, R);
        }
    }
};

// DFT of R points in registers, natural order: the radices of the tiled grids,
// else direct with x_j +- x_{R-j} (a real and an imaginary sum of (R - 1)/2
// products give X_k and X_{R-k}).
template <int R, int DIR, class V> __device__ __forceinline__ void any_dft(V (&v)[R]) {
    using T = decltype(v[0].x);
    if constexpr (R == 2 || R == 3 || R == 4 || R == 5 || R == 8 || R == 16) {
        reg_dft<R, DIR, V>::run(v);
    } else {
        constexpr Trig<R> t{};
        constexpr int H = (R - 1) / 2;
        V s[H], d[H];
#pragma unroll
        for (int j = 0; j < H; ++j) {
            s[j] = c_add(v[j + 1], v[R - 1 - j]);
            d[j] = c_sub(v[j + 1], v[R - 1 - j]);
        }
        const V x0 = v[0], xm = v[R / 2];
#pragma unroll
        for (int k = 0; k <= H; ++k) {
            V a = x0, b = {T(0), T(0)};
            if (R % 2 == 0) a = (k & 1) ? c_sub(a, xm) : c_add(a, xm);
#pragma unroll
            for (int j = 0; j < H; ++j) {
                const T c = (T)t.c[((j + 1) * k) % R], sn = (T)(DIR * t.s[((j + 1) * k) % R]);
                a = {fma_rn(c, s[j].x, a.x), fma_rn(c, s[j].y, a.y)};
                b = {fma_rn(sn, d[j].x, b.x), fma_rn(sn, d[j].y, b.y)};
            }
            v[k] = {a.x - b.y, a.y + b.x};  // a + i b
            if (k > 0) v[R - k] = {a.x + b.y, a.y - b.x};
        }
        if (R % 2 == 0) {
            V a = (R / 2) & 1 ? c_sub(x0, xm) : c_add(x0, xm);
#pragma unroll
            for (int j = 0; j < H; ++j) a = (j & 1) ? c_add(a, s[j]) : c_sub(a, s[j]);  // (-1)^(j + 1)
            v[R / 2] = a;
        }
    }
}

// Lines in shared memory: element e of line l at e ES + l LS; 2^lg lines.
struct LineBuf {
    int n, n1, n2, ES, LS, lg;
};

// One stage over all lines: `other` units per line, unit o on the R elements
// o bs + k es, times W_n^{o k} at the end when `tw_on`. Up to 16 points stay in
// registers and in place; longer (prime) factors go through `alt`, one thread
// per pair of outputs (k, R - k), and buf and alt change places.
template <int R, int DIR, class V>
__device__ __forceinline__ void line_stage_small(V* buf, const LineBuf& L, int other, int bs, int es, bool tw_on, const V* tw) {
    const int st = es * L.ES;
    for (int u = threadIdx.x; u < (other << L.lg); u += blockDim.x) {
        const int l = u & ((1 << L.lg) - 1), o = u >> L.lg;
        V* p = buf + l * L.LS + o * bs * L.ES;
        V v[R];
#pragma unroll
        for (int k = 0; k < R; ++k) v[k] = p[k * st];
        any_dft<R, DIR>(v);
        if (tw_on) {
#pragma unroll
            for (int k = 1; k < R; ++k) v[k] = c_mul(v[k], gtw<DIR>(tw, o * k));
        }
#pragma unroll
        for (int k = 0; k < R; ++k) p[k * st] = v[k];
    }
}
template <int DIR, class V>
__device__ __noinline__ void line_stage_big(const V* buf, V* alt, const LineBuf& L, int R, int other, int bs, int es, bool tw_on,
                                            const V* tw) {
    using T = decltype(buf->x);
    const int st = es * L.ES, pairs = R / 2 + 1, wstep = L.n / R;
    for (int u = threadIdx.x; u < ((other * pairs) << L.lg); u += blockDim.x) {
        const int l = u & ((1 << L.lg) - 1), r = u >> L.lg;
        const int o = r % other, k = r / other;
        const int base = l * L.LS + o * bs * L.ES;
        const V* p = buf + base;
        V a = p[0], b = {T(0), T(0)};
        int m = 0;
        for (int j = 1; 2 * j <= R; ++j) {
            m += k;
            if (m >= R) m -= R;
            const V w = tw[m * wstep];  // (cos, -sin)
            const V x = p[j * st];
            if (2 * j == R) {  // R even: (-1)^k x_{R/2}
                a = {fma_rn(w.x, x.x, a.x), fma_rn(w.x, x.y, a.y)};
            } else {
                const V y = p[(R - j) * st];
                const V s = c_add(x, y), d = c_sub(x, y);
                const T sn = DIR < 0 ? w.y : -w.y;
                a = {fma_rn(w.x, s.x, a.x), fma_rn(w.x, s.y, a.y)};
                b = {fma_rn(sn, d.x, b.x), fma_rn(sn, d.y, b.y)};
            }
        }
        V x1 = {a.x - b.y, a.y + b.x}, x2 = {a.x + b.y, a.y - b.x};
        V* q = alt + base;
        q[k * st] = tw_on ? c_mul(x1, gtw<DIR>(tw, o * k)) : x1;
        if (k > 0 && 2 * k != R) q[(R - k) * st] = tw_on ? c_mul(x2, gtw<DIR>(tw, o * (R - k))) : x2;
    }
}
template <int DIR, class V>
__device__ __forceinline__ void line_stage(V*& buf, V*& alt, const LineBuf& L, int R, int other, int bs, int es, bool tw_on,
                                           const V* tw) {
    switch (R) {
#define TILD_STAGE(r) \
    case r: line_stage_small<r, DIR>(buf, L, other, bs, es, tw_on, tw); break;
        case 1: break;
        TILD_STAGE(2) TILD_STAGE(3) TILD_STAGE(4) TILD_STAGE(5) TILD_STAGE(6) TILD_STAGE(7) TILD_STAGE(8) TILD_STAGE(9)
        TILD_STAGE(10) TILD_STAGE(11) TILD_STAGE(12) TILD_STAGE(13) TILD_STAGE(14) TILD_STAGE(15) TILD_STAGE(16)
#undef TILD_STAGE
        default: {
            line_stage_big<DIR>(buf, alt, L, R, other, bs, es, tw_on, tw);
            V* t = buf;
            buf = alt;
            alt = t;
        }
    }
    __syncthreads();
}
// natural order in, slot order out / slot order in, natural order out
template <class V> __device__ __forceinline__ void lines_forward(V*& buf, V*& alt, const LineBuf& L, const V* tw) {
    line_stage<-1>(buf, alt, L, L.n1, L.n2, 1, L.n2, true, tw);
    line_stage<-1>(buf, alt, L, L.n2, L.n1, L.n2, 1, false, tw);
}
template <class V> __device__ __forceinline__ void lines_inverse(V*& buf, V*& alt, const LineBuf& L, const V* tw) {
    line_stage<+1>(buf, alt, L, L.n2, L.n1, L.n2, 1, true, tw);
    line_stage<+1>(buf, alt, L, L.n1, L.n2, 1, L.n2, false, tw);
}

// What the line passes share. H: [NP][3][M] (field 0: G, field 2: G of the last
// axis times its wavenumber, between them the y pass's third field).
template <typename T> struct LineArgs {
    int n, nz, n1, n2, lg;   // grid, factors, log2 of the lines per CTA
    int half;                // complex values of one line buffer (0: no second buffer)
    const cplx_t<T>* tw;
    T two_pi_over_L;
};
template <typename T> __device__ __forceinline__ T any_grad_k(int i, int n, T two_pi_over_L) {
    return (n % 2 == 0 && 2 * i == n) ? T(0) : two_pi_over_L * (T)(2 * i < n ? i : i - n);
}
// wavenumber index of a slot, and the slot of an index
__device__ __forceinline__ int slot_index(int s, int n1, int n2) { return s / n2 + n1 * (s % n2); }
__device__ __forceinline__ int index_slot(int k, int n1, int n2) { return (k % n1) * n2 + k / n1; }

// Shared memory of a line pass: twiddles [n], wavenumbers by slot [n] (in the
// space of n complex values), then the line buffers.
template <typename T> struct LineShared {
    cplx_t<T>*tw, *buf, *alt;
    T* ks;
    __device__ __forceinline__ LineShared(unsigned char* raw, const LineArgs<T>& g) {
        tw = reinterpret_cast<cplx_t<T>*>(raw);
        ks = reinterpret_cast<T*>(tw + g.n);
        buf = tw + 2 * g.n;
        alt = buf + g.half;
    }
    __device__ __forceinline__ void fill(const LineArgs<T>& g) const {
        for (int i = threadIdx.x; i < g.n; i += 128) {
            tw[i] = g.tw[i];
            ks[i] = any_grad_k(slot_index(i, g.n1, g.n2), g.n, g.two_pi_over_L);
        }
    }
};

// f(l, e) in batches of four loads for the elements e of the CTA's rows l: a
// warp or more per row; load(l, e) -> R, then store(l, e, R).
template <class R, class Load, class Store>
__device__ __forceinline__ void for_rows(int lg, int rows, int n, Load load, Store store) {
    const int ts = lg >= 2 ? 5 : 7 - lg, tpr = 1 << ts, rpp = 128 >> ts;
    const int e0 = threadIdx.x & (tpr - 1);
    int l = threadIdx.x >> ts, e = e0;
    while (l < rows) {
        R v[4];
        int la[4], ea[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            la[k] = l;
            ea[k] = e;
            if (l < rows && e < n) v[k] = load(l, e);
            e += tpr;
            if (e >= n) {
                e = e0;
                l += rpp;
            }
        }
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (la[k] < rows && ea[k] < n) store(la[k], ea[k], v[k]);
    }
}

// x pass forward: rows of the fixed-point densities (zeroed when asked, once
// every row of the CTA is loaded: zeroing between the loads would serialise
// them) -> Z. grid = (row tiles, NP).
template <typename T>
__global__ void __launch_bounds__(128) line_x_forward(LineArgs<T> g, unsigned long long* __restrict__ rho_fx,
                                                      cplx_t<T>* __restrict__ Z, T scale, int zero_after,
                                                      unsigned long long* step_ctr) {
    using V = cplx_t<T>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    LineShared<T> sh(smem_raw, g);
    const int pitch = g.n | 1;
    const size_t M = (size_t)g.nz * g.n * g.n;
    const int r0 = blockIdx.x << g.lg, rows = min(1 << g.lg, g.nz * g.n - r0);
    unsigned long long* a = rho_fx + 2 * blockIdx.y * M + (size_t)r0 * g.n;
    Z += blockIdx.y * M + (size_t)r0 * g.n;
    sh.fill(g);
    dependency_wait();
    if (step_ctr && blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) *step_ctr += 1ull;
    for_rows<longlong2>(
        g.lg, rows, g.n,
        [&](int l, int e) { return make_longlong2((long long)a[l * g.n + e], (long long)a[M + l * g.n + e]); },
        [&](int l, int e, longlong2 v) {
            sh.buf[l * pitch + e] = V{density_from_fixed(v.x, scale), density_from_fixed(v.y, scale)};
        });
    __syncthreads();
    if (zero_after)
        for (int i = threadIdx.x; i < rows * g.n; i += 128) {
            a[i] = 0ull;
            a[M + i] = 0ull;
        }
    lines_forward(sh.buf, sh.alt, LineBuf{g.n, g.n1, g.n2, 1, pitch, g.lg}, sh.tw);
    for_rows<V>(
        g.lg, rows, g.n, [&](int l, int e) { return sh.buf[l * pitch + e]; },
        [&](int l, int e, V v) { Z[l * g.n + e] = v; });
}

// x pass inverse: field d of pair q (grid.y = q D + d) -> grad field d. d = 0:
// G times k_x; in 2D field 1 lies in H's field 2 (the last axis).
template <typename T>
__global__ void __launch_bounds__(128) line_x_inverse(LineArgs<T> g, const cplx_t<T>* __restrict__ H, cplx_t<T>* __restrict__ grad,
                                                      int D) {
    using V = cplx_t<T>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    LineShared<T> sh(smem_raw, g);
    const int pitch = g.n | 1;
    const size_t M = (size_t)g.nz * g.n * g.n;
    const int r0 = blockIdx.x << g.lg, rows = min(1 << g.lg, g.nz * g.n - r0);
    const int q = blockIdx.y / D, d = blockIdx.y - q * D;
    const V* src = H + (3 * q + (D == 2 && d == 1 ? 2 : d)) * M + (size_t)r0 * g.n;
    grad += (4 * q + d) * M + (size_t)r0 * g.n;
    sh.fill(g);
    dependency_wait();
    for_rows<V>(
        g.lg, rows, g.n, [&](int l, int e) { return __ldca(src + l * g.n + e); }, [&](int l, int e, V v) { sh.buf[l * pitch + e] = v; });
    __syncthreads();
    if (d == 0) {
        for_rows<V>(
            g.lg, rows, g.n, [&](int l, int e) { return sh.buf[l * pitch + e]; },
            [&](int l, int e, V v) { sh.buf[l * pitch + e] = c_scale_rn(v, sh.ks[e]); });
        __syncthreads();
    }
    lines_inverse(sh.buf, sh.alt, LineBuf{g.n, g.n1, g.n2, 1, pitch, g.lg}, sh.tw);
    for_rows<V>(
        g.lg, rows, g.n, [&](int l, int e) { return sh.buf[l * pitch + e]; },
        [&](int l, int e, V v) { grad[l * g.n + e] = v; });
}

// y pass (3D): CTA = (tile of column slots, z plane, part). Forward: Z in place
// (grid.z = pair). Inverse on H (grid.z = 2 pair + part): part 0 reads G and
// writes field 0 (G) and field 1 (k_y G), part 1 transforms field 2.
template <typename T, int DIR>
__global__ void __launch_bounds__(128) line_y(LineArgs<T> g, cplx_t<T>* __restrict__ data) {
    using V = cplx_t<T>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    LineShared<T> sh(smem_raw, g);
    const int n = g.n;
    const size_t M = (size_t)g.nz * n * n;
    const int part = DIR < 0 ? 0 : (int)(blockIdx.z & 1);
    data += DIR < 0 ? blockIdx.z * M : 3 * (blockIdx.z >> 1) * M;
    const bool two = DIR > 0 && part == 0;
    // lg counts the lines of the buffer: half of them columns when two fields come out
    const int clg = two ? g.lg - 1 : g.lg, C = 1 << clg, LN = 1 << g.lg;
    const int x0 = blockIdx.x * C;
    if (x0 >= n) return;
    V* base = data + (DIR > 0 && part == 1 ? 2 * M : 0) + (size_t)blockIdx.y * n * n + x0;
    sh.fill(g);
    dependency_wait();
    for (int i0 = threadIdx.x; i0 < n * C; i0 += 4 * 128) {
        V v[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int i = i0 + k * 128, c = i & (C - 1), e = i >> clg;
            if (e < n && x0 + c < n) v[k] = base[e * n + c];
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int i = i0 + k * 128, c = i & (C - 1), e = i >> clg;
            if (e < n && x0 + c < n) sh.buf[e * LN + c] = v[k];
        }
    }
    __syncthreads();
    if (two) {
        for (int i = threadIdx.x; i < n * C; i += 128) {
            const int c = i & (C - 1), e = i >> clg;
            sh.buf[e * LN + C + c] = c_scale_rn(sh.buf[e * LN + c], sh.ks[e]);
        }
        __syncthreads();
    }
    const LineBuf L{n, g.n1, g.n2, LN, 1, g.lg};
    if (DIR < 0)
        lines_forward(sh.buf, sh.alt, L, sh.tw);
    else
        lines_inverse(sh.buf, sh.alt, L, sh.tw);
    for (int i = threadIdx.x; i < n * C; i += 128) {
        const int c = i & (C - 1), e = i >> clg;
        if (x0 + c >= n) continue;
        base[e * n + c] = sh.buf[e * LN + c];
        if (two) base[M + e * n + c] = sh.buf[e * LN + C + c];
    }
}

// Last axis (z in 3D, y in 2D): forward transform, spectral multiply, inverse
// transform. CTA = (tile of CP column slots, row pair {ky, -ky}); it holds
// every column's line A = (ky, kx) and mirror line B = (-ky, -kx) of every
// species pair. Rows that are their own mirror (ky = 0, n/2; 2D) store A only.
// Lines [field][pair q][A, B][CP]: field 0 becomes G = i Q, field 1
// i k_last Q, Q_p = w~_2p + i w~_2p+1 (as in the z pass of the tiled grids).
template <typename T, int NP, int D>
__global__ void __launch_bounds__(128) line_last(LineArgs<T> g, const cplx_t<T>* __restrict__ Z, cplx_t<T>* __restrict__ H,
                                                 SpectralParams<T> sp, double* __restrict__ partials) {
    using V = cplx_t<T>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    LineShared<T> sh(smem_raw, g);
    const int n = g.n, n1 = g.n1, n2 = g.n2;
    const int LN = 1 << g.lg, flg = g.lg - 1, F = LN / 2;  // lines, and those of one field
    const int cpl = g.lg - (NP == 2 ? 3 : 2), CP = 1 << cpl;  // 4 NP lines per column
    const size_t M = (size_t)g.nz * n * n;
    const int stride = D == 3 ? n * n : n;
    const int ky = D == 3 ? (int)blockIdx.y : 0, my = ky == 0 ? 0 : n - ky;
    const bool self = ky == my;
    const int x0 = blockIdx.x * CP;
    __shared__ int s_off[64];  // first element of field 0's line l (-1: none)
    if (threadIdx.x < F) {
        const int c = threadIdx.x & (CP - 1), h = threadIdx.x >> cpl;  // h = 2 q + (A: 0, B: 1)
        int x = x0 + c;
        if (h & 1) {  // the slot of -kx
            const int k = slot_index(x, n1, n2);
            x = index_slot(k == 0 ? 0 : n - k, n1, n2);
        }
        const int row = D == 3 ? index_slot((h & 1) ? my : ky, n1, n2) * n : 0;
        s_off[threadIdx.x] = x0 + c < n ? row + x : -1;
    }
    sh.fill(g);
    dependency_wait();
    __syncthreads();
    // lanes over columns, then A/B, pairs and elements
    for (int i0 = threadIdx.x; i0 < n << flg; i0 += 4 * 128) {
        V v[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int i = i0 + k * 128, l = i & (F - 1), e = i >> flg;
            if (e < n && s_off[l] >= 0) v[k] = __ldca(Z + ((l >> cpl) >> 1) * M + (size_t)e * stride + s_off[l]);
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int i = i0 + k * 128, l = i & (F - 1), e = i >> flg;
            if (e < n) sh.buf[e * LN + l] = s_off[l] >= 0 ? v[k] : V{T(0), T(0)};
        }
    }
    __syncthreads();
    // the forward transform of field 0's lines alone: half of the buffer
    lines_forward(sh.buf, sh.alt, LineBuf{n, n1, n2, LN, 1, flg}, sh.tw);
    V* buf = sh.buf;
    Wide<T> acc[5];
    // multiply: unit (column, slot k1 n2 + k2 of A); -k lies in another slot of B
    for (int u = threadIdx.x; u < n << cpl; u += 128) {
        const int c = u & (CP - 1), sl = u >> cpl;
        if (x0 + c >= n) continue;
        const int kx = slot_index(x0 + c, n1, n2);
        const T exy = sp.kernel1d[kx] * (D == 3 ? sp.kernel1d[ky] : T(1));
        {
            const int k1 = sl / n2, k2 = sl - k1 * n2;
            const int kl = k1 + n1 * k2;
            const int sm = k1 == 0 ? (k2 == 0 ? 0 : n2 - k2) : (n1 - k1) * n2 + n2 - 1 - k2;
            const int eA = sl * LN + c, eB = sm * LN + c;
            const T uh = exy * sp.kernel1d[kl];
            V zA[NP], zB[NP];
#pragma unroll
            for (int q = 0; q < NP; ++q) {
                zA[q] = buf[eA + (2 * q) * CP];
                zB[q] = buf[eB + (2 * q + 1) * CP];
            }
#pragma unroll
            for (int s = 0; s < 2; ++s) {
                V A[2 * NP];
#pragma unroll
                for (int q = 0; q < NP; ++q) {
                    const V Zk = s == 0 ? zA[q] : zB[q], Zm = s == 0 ? zB[q] : zA[q];
                    A[2 * q] = {T(0.5) * (Zk.x + Zm.x), T(0.5) * (Zk.y - Zm.y)};
                    A[2 * q + 1] = {T(0.5) * (Zk.y + Zm.y), -T(0.5) * (Zk.x - Zm.x)};
                }
                if (partials && s == 0) {  // k and -k contribute the same
                    const bool zero = kx == 0 && ky == 0 && kl == 0;
                    const T weight = self ? T(1) : T(2);
                    if constexpr (NP == 1)
                        add_energies<T, 1>(acc, A[0], A[1], uh, sp.e_rho, weight, zero, T(0));
                    else
                        add_energies4<T, NP>(acc, A, sp, uh * weight, zero);
                }
                const T kg = sh.ks[s == 0 ? sl : sm];
                V w[2 * NP];
#pragma unroll
                for (int K = 0; K < 2 * NP; ++K) {
                    T wr = 0, wi = 0;
#pragma unroll
                    for (int K2 = 0; K2 < 2 * NP; ++K2) {
                        const T eps = NP == 1 ? (K == K2 ? (K == 0 ? sp.eAA : sp.eBB) : sp.eAB) : sp.eps4[K][K2];
                        wr = fma_rn(eps, A[K2].x, wr);
                        wi = fma_rn(eps, A[K2].y, wi);
                    }
                    w[K] = {uh * wr, uh * wi};
                }
#pragma unroll
                for (int q = 0; q < NP; ++q) {
                    const V iQ = {-(w[2 * q].y + w[2 * q + 1].x), w[2 * q].x - w[2 * q + 1].y};
                    const int at = (s == 0 ? eA + (2 * q) * CP : eB + (2 * q + 1) * CP);
                    buf[at] = iQ;
                    buf[at + F] = c_scale_rn(iQ, kg);
                }
            }
        }
    }
    __syncthreads();
    lines_inverse(sh.buf, sh.alt, LineBuf{n, n1, n2, LN, 1, g.lg}, sh.tw);
    for (int i = threadIdx.x; i < n << g.lg; i += 128) {
        const int l = i & (LN - 1), e = i >> g.lg, lf = l & (F - 1);
        const int h = lf >> cpl, f = l >= F ? 2 : 0;
        if (s_off[lf] < 0 || (self && (h & 1))) continue;
        H[(3 * (h >> 1) + f) * M + (size_t)e * stride + s_off[lf]] = sh.buf[e * LN + l];
    }
    if (partials) {
        const size_t b = (size_t)blockIdx.y * gridDim.x + blockIdx.x;
        block_sum<5, T>(acc, [&](int k, double v) { partials[5 * b + k] = v; });
    }
}

// ---------------------------------------------------------------- beads

// One thread per bead slot: the bead modes of the tiled kernel (spread,
// force and observables, set velocity, step) with D = 2 or 3 and any n.
// grad: [NS/2][4][M] (d_x, d_y, d_z, potentials) per species pair.
template <int P, int MODE, typename T, int D>
__global__ void __launch_bounds__(256) generic_bead_kernel(BeadParams<T> p, BeadBuffers<T> bf, int nz) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const bool active = i < p.n_beads;
    const bool sums = MODE == kModeForce && bf.partials;
    Wide<T> acc[5];
    dependency_wait();
    if (active) {
        const int n = p.n;
        const size_t M = (size_t)nz * n * n;
        T x = bf.px[i], y = bf.py[i], z = D == 3 ? bf.pz[i] : T(0);
        const int tag = bf.id[i];
        const int bid = slot_bead_id(tag), species = slot_species(tag);
        Stencil<P, T> st;
        st.set(x, y, z, p.inv_dx);
        constexpr int PZ = D == 3 ? P : 1;
        if (MODE != kModeSpread && bead_ok(p, bf, st, bid, species)) {
            // field force: -sum_g W(r - g) grad w_K(g)
            const cplx_t<T>* gp = bf.grad + (size_t)(species >> 1) * 4 * M;
            const int comp = species & 1;
            T gx = 0, gy = 0, gz = 0;
#pragma unroll
            for (int c = 0; c < PZ; ++c) {
                const size_t oz = D == 3 ? (size_t)pwrap(st.jz + c, n) * n * n : 0;
                const T wz = D == 3 ? st.wz[c] : T(1);
#pragma unroll
                for (int b = 0; b < P; ++b) {
                    const size_t oy = oz + (size_t)pwrap(st.jy + b, n) * n;
                    const T wyz = st.wy[b] * wz;
#pragma unroll
                    for (int a = 0; a < P; ++a) {
                        const size_t g = oy + pwrap(st.jx + a, n);
                        const T w = st.wx[a] * wyz;
                        const cplx_t<T> vx = __ldca(gp + g), vy = __ldca(gp + M + g);
                        gx += w * (comp ? vx.y : vx.x);
                        gy += w * (comp ? vy.y : vy.x);
                        if (D == 3) {
                            const cplx_t<T> vz = __ldca(gp + 2 * M + g);
                            gz += w * (comp ? vz.y : vz.x);
                        }
                    }
                }
            }
            T fx = -gx, fy = -gy, fz = -gz;
            const int2 nb = bf.nbr[i];
            auto bond = [&](int s) {
                if (!slot_ok(p, bf, s)) return;
                const T dx = min_image(x - bf.px[s], p.L, p.inv_L);
                const T dy = min_image(y - bf.py[s], p.L, p.inv_L);
                const T dz = D == 3 ? min_image(z - bf.pz[s], p.L, p.inv_L) : T(0);
                fx -= p.k_bond * dx;
                fy -= p.k_bond * dy;
                fz -= p.k_bond * dz;
                if (MODE == kModeForce && sums) add_squares(acc[0], dx, dy, dz, p.e_len);
            };
            if (nb.x >= 0) bond(nb.x);
            if (nb.y >= 0) bond(nb.y);
            for_each_extra_bond(nb, bf.ext, bond);
            if (not_finite(fx, fy, fz)) atomicOr(bf.err, kErrNonFinite);
            T ux = 0, uy = 0, uz = 0;
            if (MODE != kModeSetVel) {
                ux = bf.ux[i];
                uy = bf.uy[i];
                uz = D == 3 ? bf.uz[i] : T(0);
            }
            if (MODE == kModeForce) {
                normal3<T> g = {T(0), T(0), T(0)};
                if (p.vg != T(0)) g = gaussian3((uint32_t)bid, *bf.step, p.seed, T(0));
                const T vx = velocity_of(p, ux, fx, g.a);
                const T vy = velocity_of(p, uy, fy, g.b);
                const T vz = D == 3 ? velocity_of(p, uz, fz, g.c) : T(0);
                if (sums) {
                    add_squares(acc[1], vx, vy, vz, p.e_vel);
                    acc[2].add(fx);
                    acc[3].add(fy);
                    acc[4].add(fz);
                }
                if (bf.f_out) {
                    bf.f_out[3 * (size_t)bid + 0] = fx;
                    bf.f_out[3 * (size_t)bid + 1] = fy;
                    bf.f_out[3 * (size_t)bid + 2] = fz;
                }
                if (bf.v_out) {
                    bf.v_out[3 * (size_t)bid + 0] = vx;
                    bf.v_out[3 * (size_t)bid + 1] = vy;
                    bf.v_out[3 * (size_t)bid + 2] = vz;
                }
            } else if (MODE == kModeSetVel) {
                T vx, vy, vz;
                if (bf.v_in) {
                    vx = bf.v_in[3 * (size_t)bid + 0];
                    vy = bf.v_in[3 * (size_t)bid + 1];
                    vz = bf.v_in[3 * (size_t)bid + 2];
                } else {
                    const normal3<T> g = gaussian3((uint32_t)bid, ~0ull, p.seed, T(0));
                    vx = p.sigma_v * g.a;
                    vy = p.sigma_v * g.b;
                    vz = p.sigma_v * g.c;
                }
                normal3<T> g = {T(0), T(0), T(0)};
                if (p.wg != T(0)) g = gaussian3((uint32_t)bid, *bf.step, p.seed, T(0));
                bf.ux[i] = carried_of(p, vx, fx, g.a);
                bf.uy[i] = carried_of(p, vy, fy, g.b);
                bf.uz[i] = D == 3 ? carried_of(p, vz, fz, g.c) : T(0);
            } else {  // step
                const normal3<T> g = gaussian3((uint32_t)bid, *bf.step - (uint64_t)p.noise_lag, p.seed, T(0));
                step_update(p, x, ux, fx, g.a);
                step_update(p, y, uy, fy, g.b);
                if (D == 3) step_update(p, z, uz, fz, g.c);
                bf.qx[i] = x;
                bf.qy[i] = y;
                bf.qz[i] = z;
                bf.ux[i] = ux;
                bf.uy[i] = uy;
                bf.uz[i] = uz;
                st.set(x, y, z, p.inv_dx);
            }
        }
        if ((MODE == kModeSpread || MODE == kModeStep) && bead_ok(p, bf, st, bid, species)) {
            using FP = FixedPoint<T>;
            unsigned long long* rk = bf.rho_fx + (size_t)species * M;
#pragma unroll
            for (int c = 0; c < PZ; ++c) {
                const size_t oz = D == 3 ? (size_t)pwrap(st.jz + c, n) * n * n : 0;
                const T wz = D == 3 ? st.wz[c] : T(1);
#pragma unroll
                for (int b = 0; b < P; ++b) {
                    const size_t oy = oz + (size_t)pwrap(st.jy + b, n) * n;
                    const T wyz = FP::scaled(st.wy[b] * wz);
#pragma unroll
                    for (int a = 0; a < P; ++a) atomicAdd(rk + oy + pwrap(st.jx + a, n), FP::to_grid(st.wx[a], wyz));
                }
            }
        }
    }
    if (MODE == kModeForce && sums) {
        block_sum<5, T>(acc, [&](int k, double v) { bf.partials[5 * (size_t)blockIdx.x + k] = v; });
    }
}

}  // namespace tild
