// Grid stages of the TILD step (Eq. PMM evaluated by FFT):
//   forward:  int64 fixed-point densities -> Z = DFT_xy(rho_A + i rho_B)
//   z pass:   DFT_z, spectral multiply with the smeared chi/kappa kernel and
//             i k (one CTA per pencil tile), inverse DFT_z -> H_d
//   inverse:  H_d -> IDFT_xy -> (d w_A/dr_d, d w_B/dr_d) on the grid
//
// Two real species are carried as one complex field Z = rho_A + i rho_B.
// Their spectra are separated in the z pass with Hermitian symmetry:
//   rho~_A(k) = (Z(k) + conj Z(-k)) / 2,  rho~_B(k) = (Z(k) - conj Z(-k)) / (2i),
// and the three gradient spectra are packed back as
//   H_d(k) = i k~_d (w~_A(k) + i w~_B(k)),
// whose inverse transform is real part d w_A/dr_d, imaginary part
// d w_B/dr_d (both gradient fields are real).
//
// With more than two species (up to four) the species go in pairs: pair p
// carries species 2p and 2p+1 exactly as A and B above, and every array
// below gains a leading pair index; only the z pass sees all pairs at once
// (the spectral multiply couples every species).
//
// Memory layouts (n^3 points, index g = (z n + y) n + x; NP pairs):
//   rho_fx  int64 [2 NP][M]           fixed-point densities (2^22 or 2^44 per bead weight)
//   Zxy     complex [NP][z][ky][pos(kx)]  after the forward x and y transforms
//   H       complex [NP][3][z][ky][pos(kx)] after the z pass (z back in real space)
// (pos(kx): mirror-paired column order, see kx_of_pos)
//   grad    complex [NP][4][z][y][x]  (d w_2p, d w_2p+1) per point and direction,
//                                     then the potentials i (w_2p + i w_2p+1)
#pragma once

#include "fft.cuh"

namespace tild {

template <typename T> struct SpectralParams {
    T two_pi_over_L;   // 2 pi / L
    T eAA, eAB, eBB;   // eps matrix / M (the 1/M of the inverse DFT folded in)
    T eps4[4][4];      // more than two species: eps_KK' / M
    T chi4[4][4];      // more than two species: chi_KK' (the energy sum of the z pass weights by it)
    T e_rho;           // a power of two near dV: the energy sums take rho~ times e_rho (1 in FP64)
    const T* kernel1d; // exp(-a^2 k_m^2) per 1-D frequency index m (FP64 on the host)
    // smeared-charge electrostatics: w_K += q_K c(k) (q_A rho~_A + q_B rho~_B) with
    // c(k) = el_scale exp(-a_e^2 |k|^2) / |k|^2 (0 at k = 0); el_scale = 4 pi l_B / M
    // (0: no charges); kernel1d_el = exp(-a_e^2 k_m^2)
    T el_scale, qA, qB;
    const T* kernel1d_el;
};

template <int N> __host__ __device__ __forceinline__ int kx_of_pos(int p);
template <int N> __host__ __device__ __forceinline__ int pos_of_kx(int kx);
template <int C, int STRIDE> struct TileAddr;

// Wavenumber 2 pi m / L of FFT index i (m = i or i - n; the Nyquist index
// n/2 counts as -n/2).
template <typename T, int N> __device__ __forceinline__ T raw_k(int i, T two_pi_over_L) {
    return two_pi_over_L * (T)(i < N / 2 ? i : i - N);
}

// Wavenumber used for spectral differentiation at FFT index i: 2 pi m / L
// with m = i (i < n/2) or i - n, and 0 at the Nyquist index n/2.
template <typename T, int N> __device__ __forceinline__ T grad_k(int i, T two_pi_over_L) {
    return i == N / 2 ? T(0) : two_pi_over_L * (T)(i < N / 2 ? i : i - N);
}

// 1/x: the correctly rounded reciprocal intrinsic in FP32 (no division
// slow path), a plain division in FP64.
__device__ __forceinline__ float recip(float x) { return __frcp_rn(x); }
__device__ __forceinline__ double recip(double x) { return 1.0 / x; }

// Host side of LineSlots<n>::pitch: complex values of shared memory per row of
// the xy passes (0: no hand-written transform of that length).
inline int row_pitch(int n) {
    switch (n) {
        case 8: return LineSlots<8>::pitch;
        case 16: return LineSlots<16>::pitch;
        case 24: return LineSlots<24>::pitch;
        case 32: return LineSlots<32>::pitch;
        case 40: return LineSlots<40>::pitch;
        case 48: return LineSlots<48>::pitch;
        case 64: return LineSlots<64>::pitch;
        case 80: return LineSlots<80>::pitch;
        case 128: return LineSlots<128>::pitch;
        case 256: return LineSlots<256>::pitch;
    }
    return 0;
}

template <class V> __device__ __forceinline__ void load_twiddles(V* s_tw, const V* g_tw, int n) {
    for (int i = threadIdx.x; i < n; i += blockDim.x) s_tw[i] = g_tw[i];
}

// Copy COUNT elements from global to shared memory with up to 16
// independent loads in flight per thread: dst(i, value) stores element i.
// Accesses are guarded by i < COUNT unless every thread's batches are full
// (COUNT a multiple of NTHR and PER a multiple of the batch); otherwise the
// last batch of a thread may be partial.
template <int COUNT, int NTHR, class V, class Src, class Dst>
__device__ __forceinline__ void batched_load(Src src, Dst dst) {
    constexpr int PER = (COUNT + NTHR - 1) / NTHR;
    constexpr int B = PER < 16 ? PER : 16;
    constexpr bool kFull = COUNT % NTHR == 0 && PER % B == 0;
#pragma unroll 1
    for (int k0 = 0; k0 < PER; k0 += B) {
        V v[B];
#pragma unroll
        for (int k = 0; k < B; ++k) {
            const int i = threadIdx.x + (k0 + k) * NTHR;
            if (kFull || i < COUNT) v[k] = src(i);
        }
#pragma unroll
        for (int k = 0; k < B; ++k) {
            const int i = threadIdx.x + (k0 + k) * NTHR;
            if (kFull || i < COUNT) dst(i, v[k]);
        }
    }
}

// The N1 inputs of stage-A unit j2 of one row of fixed-point densities
// (ga, gb: the row of either species): rho_A + i rho_B at x = j2 + N2 j1. Up to
// eight loads of each species are in flight (the raw 64-bit values of more
// would not leave registers for the transform). Lanes take consecutive j2,
// so a warp reads whole sectors.
template <int N, class V, typename T>
__device__ __forceinline__ void load_fixed_unit(const long long* __restrict__ ga, const long long* __restrict__ gb, int j2,
                                                T scale, V (&v)[fft_split<N>::N1]) {
    constexpr int N1 = fft_split<N>::N1, N2 = fft_split<N>::N2;
    constexpr int B = N1 < 8 ? N1 : 8;
#pragma unroll
    for (int h = 0; h < N1; h += B) {
        long long a[B], b[B];
#pragma unroll
        for (int k = 0; k < B; ++k) {
            a[k] = __ldcs(ga + j2 + N2 * (h + k));
            b[k] = __ldcs(gb + j2 + N2 * (h + k));
        }
#pragma unroll
        for (int k = 0; k < B; ++k) v[h + k] = V{density_from_fixed(a[k], scale), density_from_fixed(b[k], scale)};
    }
}

// Zero `count` values (16-byte stores; count even, base 16-byte aligned).
template <int NTHR> __device__ __forceinline__ void zero_fixed(unsigned long long* g, int count) {
    longlong2* p = reinterpret_cast<longlong2*>(g);
    for (int i = threadIdx.x; i < count / 2; i += NTHR) p[i] = make_longlong2(0, 0);
}

// --------------------------------------------------------------------------
// Transforms of one whole xy-plane held in shared memory, [row][LineSlots],
// four stages with three barriers: x stage A from the loader, x stage B, y
// stage A, y stage B to global memory (forward), and the mirror image
// (inverse). Bound by shared memory and latency (one CTA per SM at 128^3):
// a stage visits shared memory once, in place, where a separate load, two
// stages with their own barriers, a scaling pass and a store pass per
// direction visited it ten to twelve times (inverse at 128^3, 512 threads:
// 38.1 -> 31.7 us, 34.8 of it before rows were swizzled).
// --------------------------------------------------------------------------
// Column position of lane-ordered index i: a warp's 32 positions, those of its
// first half-warp kx = k, k + 1, ..., those of the second the mirror columns
// n - k, ...: consecutive columns in each phase of a shared-memory access
// (position order alternates between the two), the same 256 bytes of global memory.
template <int N> __device__ __forceinline__ int lane_pos(int i) {
    return N % 32 == 0 ? (i & ~31) + ((i & 15) << 1) + ((i >> 4) & 1) : i;
}

// load(y, j2, v): inputs x = j2 + N2 j1 of row y; after_load(): runs once all
// rows have been loaded; dst: [ky][pos(kx)].
template <typename T, int N, int NT, class Load, class After>
__device__ __forceinline__ void plane_forward_xy(cplx_t<T>* plane, cplx_t<T>* tw, const cplx_t<T>* __restrict__ tw_g, Load load,
                                                 After after_load, cplx_t<T>* __restrict__ dst) {
    using V = cplx_t<T>;
    using LS = LineSlots<N>;
    constexpr int N1 = LS::N1, N2 = LS::N2, PITCH = LS::pitch;
    {
        // x stage A: unit (row, j2), lanes over j2
        int u = threadIdx.x;
        V v[N1];
        load_twiddles(tw, tw_g, N);
        dependency_wait();
        if (u < N * N2) load(u / N2, u % N2, v);
        __syncthreads();
#pragma unroll 1
        while (u < N * N2) {
            const int r = u / N2, j2 = u % N2;
            stage_a_regs<N, -1>(v, j2, tw);
            V* p = plane + r * PITCH;
#pragma unroll
            for (int k1 = 0; k1 < N1; ++k1) p[LS::at(k1 * N2 + j2)] = v[k1];
            u += NT;
            if (u < N * N2) load(u / N2, u % N2, v);
        }
    }
    __syncthreads();
    after_load();
    // x stage B: unit (row, k1), lanes over k1
#pragma unroll 1
    for (int u = threadIdx.x; u < N * N1; u += NT) {
        V* p = plane + (u / N1) * PITCH;
        const int s0 = (u % N1) * N2;
        V v[N2];
#pragma unroll
        for (int j = 0; j < N2; ++j) v[j] = p[LS::at(s0 + j)];
        reg_dft<N2, -1, V>::run(v);
#pragma unroll
        for (int j = 0; j < N2; ++j) p[LS::at(s0 + j)] = v[j];
    }
    __syncthreads();
    // y stage A: unit (column slot, j2), lanes over columns
#pragma unroll 1
    for (int u = threadIdx.x; u < N * N2; u += NT) {
        const int j2 = u / N;
        V* p = plane + j2 * PITCH + LS::at(u % N);
        V v[N1];
#pragma unroll
        for (int k = 0; k < N1; ++k) v[k] = p[k * N2 * PITCH];
        stage_a_regs<N, -1>(v, j2, tw);
#pragma unroll
        for (int k = 0; k < N1; ++k) p[k * N2 * PITCH] = v[k];
    }
    __syncthreads();
    // y stage B: unit (column position, k1), lanes over positions, to global memory
#pragma unroll 1
    for (int u = threadIdx.x; u < N * N1; u += NT) {
        const int q = lane_pos<N>(u % N), k1 = u / N;
        const V* p = plane + k1 * N2 * PITCH + LS::at(LS::slot_of(kx_of_pos<N>(q)));
        V v[N2];
#pragma unroll
        for (int j = 0; j < N2; ++j) v[j] = p[j * PITCH];
        reg_dft<N2, -1, V>::run(v);
#pragma unroll
        for (int k2 = 0; k2 < N2; ++k2) dst[(k1 + N1 * k2) * N + q] = v[k2];
    }
}

// load(ky, pos): the input at row ky, column position pos; scale(kx): the
// factor of the columns between the two transforms (x_scale: apply it);
// dst: [y][x].
template <typename T, int N, int NT, class Load>
__device__ __forceinline__ void plane_inverse_yx(cplx_t<T>* plane, cplx_t<T>* tw, const cplx_t<T>* __restrict__ tw_g, Load load,
                                                 bool x_scale, T two_pi_over_L, cplx_t<T>* __restrict__ dst) {
    using V = cplx_t<T>;
    using LS = LineSlots<N>;
    constexpr int N1 = LS::N1, N2 = LS::N2, PITCH = LS::pitch;
    {
        // y stage A: unit (column position, j2), lanes over positions
        int u = threadIdx.x;
        V v[N1];
        auto fetch = [&]() {
#pragma unroll
            for (int k = 0; k < N1; ++k) v[k] = load(u / N + N2 * k, lane_pos<N>(u % N));
        };
        load_twiddles(tw, tw_g, N);
        dependency_wait();
        if (u < N * N2) fetch();
        __syncthreads();
#pragma unroll 1
        while (u < N * N2) {
            const int j2 = u / N;
            stage_a_regs<N, +1>(v, j2, tw);
            // columns in slot order of their natural index kx
            V* p = plane + j2 * PITCH + LS::at(kx_of_pos<N>(lane_pos<N>(u % N)));
#pragma unroll
            for (int k1 = 0; k1 < N1; ++k1) p[k1 * N2 * PITCH] = v[k1];
            u += NT;
            if (u < N * N2) fetch();
        }
    }
    __syncthreads();
    // y stage B: unit (column, k1), lanes over columns
#pragma unroll 1
    for (int u = threadIdx.x; u < N * N1; u += NT) {
        const int kx = u % N;
        V* p = plane + (u / N) * N2 * PITCH + LS::at(kx);
        V v[N2];
#pragma unroll
        for (int j = 0; j < N2; ++j) v[j] = p[j * PITCH];
        reg_dft<N2, +1, V>::run(v);
        if (x_scale) {
            const T s = grad_k<T, N>(kx, two_pi_over_L);
#pragma unroll
            for (int j = 0; j < N2; ++j) v[j] = c_scale_rn(v[j], s);
        }
#pragma unroll
        for (int j = 0; j < N2; ++j) p[j * PITCH] = v[j];
    }
    __syncthreads();
    // x stage A: unit (row, j2), lanes over j2; row r holds y = index_of(r)
#pragma unroll 1
    for (int u = threadIdx.x; u < N * N2; u += NT) {
        const int j2 = u % N2;
        V* p = plane + (u / N2) * PITCH;
        V v[N1];
#pragma unroll
        for (int k = 0; k < N1; ++k) v[k] = p[LS::at(k * N2 + j2)];
        stage_a_regs<N, +1>(v, j2, tw);
#pragma unroll
        for (int k = 0; k < N1; ++k) p[LS::at(k * N2 + j2)] = v[k];
    }
    __syncthreads();
    // x stage B: unit (row, k1), lanes over k1, to global memory
#pragma unroll 1
    for (int u = threadIdx.x; u < N * N1; u += NT) {
        const int r = u / N1, k1 = u % N1;
        const V* p = plane + r * PITCH;
        V v[N2];
#pragma unroll
        for (int j = 0; j < N2; ++j) v[j] = p[LS::at(k1 * N2 + j)];
        reg_dft<N2, +1, V>::run(v);
        V* o = dst + LS::index_of(r) * N + k1;
#pragma unroll
        for (int k2 = 0; k2 < N2; ++k2) o[N1 * k2] = v[k2];
    }
}

// --------------------------------------------------------------------------
// Forward xy pass on whole z-planes (plane fits in shared memory).
// grid = n (one CTA per z-plane), block = NT (512, or 128/256 for small
// planes, where several CTAs then share an SM).
// --------------------------------------------------------------------------
template <typename T> struct ForwardArgs {
    unsigned long long* rho_fx;
    cplx_t<T>* Zxy;
    const cplx_t<T>* tw;
    T scale;
    int zero_after;
    unsigned long long* step_ctr;
};

template <typename T, int N, int NT = 512>
__device__ __forceinline__ void xy_forward_plane_body(const ForwardArgs<T>& args, int bx) {
    using V = cplx_t<T>;
    unsigned long long* __restrict__ rho_fx = args.rho_fx;
    cplx_t<T>* __restrict__ Zxy = args.Zxy;
    const cplx_t<T>* __restrict__ tw_g = args.tw;
    const T scale = args.scale;
    const int zero_after = args.zero_after;
    unsigned long long* step_ctr = args.step_ctr;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    V* tw = reinterpret_cast<V*>(smem_raw);
    V* plane = tw + N;
    const size_t M = (size_t)N * N * N;
    const size_t base = (size_t)bx * N * N;
    const long long* ra = reinterpret_cast<const long long*>(rho_fx + base);
    const long long* rb = ra + M;
    plane_forward_xy<T, N, NT>(
        plane, tw, tw_g,
        [&](int y, int j2, V (&v)[fft_split<N>::N1]) { load_fixed_unit<N>(ra + y * N, rb + y * N, j2, scale, v); },
        [&]() {
            // a step's first kernel advances the noise counter to n+1
            if (step_ctr && bx == 0 && threadIdx.x == 0) *step_ctr += 1ull;
            if (zero_after) {  // every density of the plane has been read
                zero_fixed<NT>(rho_fx + base, N * N);
                zero_fixed<NT>(rho_fx + M + base, N * N);
            }
        },
        Zxy + base);
}

// grid = (n, NP): species pair blockIdx.y
template <typename T, int N, int NT = 512>
__global__ void __launch_bounds__(NT) xy_forward_plane(unsigned long long* __restrict__ rho_fx,
                                                         cplx_t<T>* __restrict__ Zxy,
                                                         const cplx_t<T>* __restrict__ tw_g, T scale,
                                                         int zero_after, unsigned long long* step_ctr) {
    const size_t M = (size_t)N * N * N;
    const int pr = blockIdx.y;
    xy_forward_plane_body<T, N, NT>(
        ForwardArgs<T>{rho_fx + 2 * pr * M, Zxy + pr * M, tw_g, scale, zero_after, pr == 0 ? step_ctr : nullptr},
        blockIdx.x);
}

// Batched form: replica blockIdx.y of a table of replicas with the same grid.
template <typename T, int N, int NT = 512>
__global__ void __launch_bounds__(NT) xy_forward_plane_batched(const ForwardArgs<T>* __restrict__ args) {
    xy_forward_plane_body<T, N, NT>(args[blockIdx.y], blockIdx.x);
}

// --------------------------------------------------------------------------
// Inverse xy pass on whole z-planes: grid = (n, 3), block = NT.
// --------------------------------------------------------------------------
template <typename T> struct InverseArgs {
    const cplx_t<T>* H;
    cplx_t<T>* grad;
    const cplx_t<T>* tw;
    T two_pi_over_L;
    int d0;  // first direction (blockIdx.y + d0); 3 alone: the potentials only
};

template <typename T, int N, int NT = 512>
__device__ __forceinline__ void xy_inverse_plane_body(const InverseArgs<T>& args, int bx, int by) {
    using V = cplx_t<T>;
    const cplx_t<T>* __restrict__ H = args.H;
    cplx_t<T>* __restrict__ grad = args.grad;
    const cplx_t<T>* __restrict__ tw_g = args.tw;
    const T two_pi_over_L = args.two_pi_over_L;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    V* tw = reinterpret_cast<V*>(smem_raw);
    V* plane = tw + N;

    // direction d: x from i k_x G, y from i k_y G, z from G_z (field 2);
    // d = 3 (optional): the potentials themselves, i (w_A + i w_B), from G
    const int d = by + args.d0;
    const size_t M = (size_t)N * N * N;
    const V* src = H + (d == 2 ? 2 * M : 0) + (size_t)bx * N * N;
    plane_inverse_yx<T, N, NT>(
        plane, tw, tw_g,
        [&](int ky, int q) {
            const V v = __ldcg(src + ky * N + q);
            return d == 1 ? c_scale_rn(v, grad_k<T, N>(ky, two_pi_over_L)) : v;
        },
        d == 0, two_pi_over_L, grad + (size_t)d * M + (size_t)bx * N * N);
}

// grid = (n, directions, NP): species pair blockIdx.z
template <typename T, int N, int NT = 512>
__global__ void __launch_bounds__(NT) xy_inverse_plane(const cplx_t<T>* __restrict__ H,
                                                         cplx_t<T>* __restrict__ grad,
                                                         const cplx_t<T>* __restrict__ tw_g, T two_pi_over_L, int d0) {
    const size_t M = (size_t)N * N * N;
    const int pr = blockIdx.z;
    xy_inverse_plane_body<T, N, NT>(InverseArgs<T>{H + 3 * pr * M, grad + 4 * pr * M, tw_g, two_pi_over_L, d0},
                                    blockIdx.x, blockIdx.y);
}

// Batched form: replica blockIdx.z.
template <typename T, int N, int NT = 512>
__global__ void __launch_bounds__(NT) xy_inverse_plane_batched(const InverseArgs<T>* __restrict__ args) {
    xy_inverse_plane_body<T, N, NT>(args[blockIdx.z], blockIdx.x, blockIdx.y);
}

// --------------------------------------------------------------------------
// Split passes for planes that do not fit in shared memory.
// Row pass along x: CTA handles R consecutive rows (row r = z n + y).
// --------------------------------------------------------------------------
template <typename T, int N, int R>
__global__ void __launch_bounds__(256) x_forward_rows(unsigned long long* __restrict__ rho_fx,
                                                       cplx_t<T>* __restrict__ Zxy,
                                                       const cplx_t<T>* __restrict__ tw_g, T scale,
                                                       int zero_after, unsigned long long* step_ctr) {
    using V = cplx_t<T>;
    using LS = LineSlots<N>;
    constexpr int N1 = LS::N1, N2 = LS::N2, PITCH = LS::pitch;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    V* tw = reinterpret_cast<V*>(smem_raw);
    V* rows = tw + N;
    const size_t M = (size_t)N * N * N;
    const size_t base = (size_t)blockIdx.x * R * N;
    const int pr = blockIdx.y;  // species pair
    rho_fx += 2 * pr * M;
    Zxy += pr * M;
    const long long* ra = reinterpret_cast<const long long*>(rho_fx + base);
    const long long* rb = ra + M;
    {
        int u = threadIdx.x;  // stage A: unit (row, j2), lanes over j2
        V v[N1];
        auto fetch = [&]() { load_fixed_unit<N>(ra + (u / N2) * N, rb + (u / N2) * N, u % N2, scale, v); };
        load_twiddles(tw, tw_g, N);
        dependency_wait();
        if (step_ctr && blockIdx.x == 0 && pr == 0 && threadIdx.x == 0) *step_ctr += 1ull;
        if (u < R * N2) fetch();
        __syncthreads();
#pragma unroll 1
        while (u < R * N2) {
            const int j2 = u % N2;
            stage_a_regs<N, -1>(v, j2, tw);
            V* p = rows + (u / N2) * PITCH;
#pragma unroll
            for (int k1 = 0; k1 < N1; ++k1) p[LS::at(k1 * N2 + j2)] = v[k1];
            u += 256;
            if (u < R * N2) fetch();
        }
    }
    __syncthreads();
    if (zero_after) {
        zero_fixed<256>(rho_fx + base, R * N);
        zero_fixed<256>(rho_fx + M + base, R * N);
    }
    // stage B in place; the store below takes the columns in position order
#pragma unroll 1
    for (int u = threadIdx.x; u < R * N1; u += 256) {
        V* p = rows + (u / N1) * PITCH;
        const int s0 = (u % N1) * N2;
        V v[N2];
#pragma unroll
        for (int j = 0; j < N2; ++j) v[j] = p[LS::at(s0 + j)];
        reg_dft<N2, -1, V>::run(v);
#pragma unroll
        for (int j = 0; j < N2; ++j) p[LS::at(s0 + j)] = v[j];
    }
    __syncthreads();
    for (int i = threadIdx.x; i < R * N; i += 256)
        Zxy[base + i] = rows[(i / N) * PITCH + LS::at(LS::slot_of(kx_of_pos<N>(i % N)))];
}

template <typename T, int N, int R>
__global__ void __launch_bounds__(256) x_inverse_rows(const cplx_t<T>* __restrict__ H, cplx_t<T>* __restrict__ grad,
                                                       const cplx_t<T>* __restrict__ tw_g, T two_pi_over_L, int d0) {
    using V = cplx_t<T>;
    using LS = LineSlots<N>;
    constexpr int N1 = LS::N1, N2 = LS::N2, PITCH = LS::pitch;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    V* tw = reinterpret_cast<V*>(smem_raw);
    V* rows = tw + N;
    const size_t M = (size_t)N * N * N;
    const int d = (int)blockIdx.y + d0;
    H += 3 * (size_t)blockIdx.z * M;  // species pair blockIdx.z
    grad += 4 * (size_t)blockIdx.z * M;
    const size_t base = (size_t)d * M + (size_t)blockIdx.x * R * N;
    // field 3 (optional, the potentials) is the plain transform of field 0
    const V* src = H + (size_t)(d == 3 ? 0 : d) * M + (size_t)blockIdx.x * R * N;
    const bool kx_mult = d == 0;  // d_x: multiply by k_x before the x transform
    {
        // stage A: unit (row, j2), lanes over j2. Column kx lies at position
        // 2 kx or 2 (n - kx) + 1, so lanes read every other value; the values
        // between them are the mirror columns, which the same CTA reads with
        // another j1 (from L1)
        int u = threadIdx.x;
        V v[N1];
        auto fetch = [&]() {
            const V* row = src + (u / N2) * N;
#pragma unroll
            for (int k = 0; k < N1; ++k) {
                const int kx = u % N2 + N2 * k;
                const V t = __ldca(row + pos_of_kx<N>(kx));
                v[k] = kx_mult ? c_scale_rn(t, grad_k<T, N>(kx, two_pi_over_L)) : t;
            }
        };
        load_twiddles(tw, tw_g, N);
        dependency_wait();
        if (u < R * N2) fetch();
        __syncthreads();
#pragma unroll 1
        while (u < R * N2) {
            const int j2 = u % N2;
            stage_a_regs<N, +1>(v, j2, tw);
            V* p = rows + (u / N2) * PITCH;
#pragma unroll
            for (int k1 = 0; k1 < N1; ++k1) p[LS::at(k1 * N2 + j2)] = v[k1];
            u += 256;
            if (u < R * N2) fetch();
        }
    }
    __syncthreads();
    // stage B: unit (row, k1), lanes over k1, to global memory
#pragma unroll 1
    for (int u = threadIdx.x; u < R * N1; u += 256) {
        const int r = u / N1, k1 = u % N1;
        const V* p = rows + r * PITCH;
        V v[N2];
#pragma unroll
        for (int j = 0; j < N2; ++j) v[j] = p[LS::at(k1 * N2 + j)];
        reg_dft<N2, +1, V>::run(v);
        V* o = grad + base + r * N + k1;
#pragma unroll
        for (int k2 = 0; k2 < N2; ++k2) o[N1 * k2] = v[k2];
    }
}

// Column pass along y: CTA (x tile, z plane, part) handles C columns.
// Forward (DIR = -1): Zxy in place; blockIdx.z = species pair.
// Inverse (DIR = +1) on H: part 0 loads a tile of G (field 0) and writes
// the transforms of G (field 0) and of i k_y G (field 1) from the same
// load; part 1 transforms G_z (field 2) in place; blockIdx.z = 2 pair +
// part. With only_g, one part transforms G alone (blockIdx.z = pair).
// Stage A reads global memory and stage B writes it: one visit of shared
// memory (the tile) in between. A CTA reads all of its columns before the
// barrier and writes them after it, so the pass works in place. At 256^3 the
// inverse row and column passes move 1.48 GB in 258 us (303 us with the
// lines loaded to and stored from shared memory), 84% of the copy rate.
template <typename T, int N, int C, int DIR>
__global__ void __launch_bounds__(256) y_columns(cplx_t<T>* __restrict__ data, const cplx_t<T>* __restrict__ tw_g,
                                                 T two_pi_over_L, int only_g) {
    using V = cplx_t<T>;
    constexpr int N1 = fft_split<N>::N1, N2 = fft_split<N>::N2;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    V* tw = reinterpret_cast<V*>(smem_raw);
    V* tile = tw + N;  // [2][slot][c]
    constexpr int TS = N * C;
    const size_t M = (size_t)N * N * N;
    const int part = (DIR < 0 || only_g) ? 0 : (int)(blockIdx.z & 1);
    const int pr = (DIR < 0 || only_g) ? (int)blockIdx.z : (int)(blockIdx.z >> 1);
    data += (DIR < 0 ? 1 : 3) * (size_t)pr * M;
    const bool two = DIR > 0 && part == 0 && !only_g;  // only_g: G alone (one part)
    const size_t off = (size_t)blockIdx.y * N * N + (size_t)blockIdx.x * C;
    const size_t src = (DIR > 0 && part == 1 ? 2 * M : 0) + off;
    {
        int u = threadIdx.x;  // stage A: unit (column, j2), lanes over columns
        V v[N1];
        auto fetch = [&]() {
#pragma unroll
            for (int k = 0; k < N1; ++k) v[k] = data[src + (size_t)(u / C + N2 * k) * N + u % C];
        };
        load_twiddles(tw, tw_g, N);
        dependency_wait();
        if (u < C * N2) fetch();
        __syncthreads();
#pragma unroll 1
        while (u < C * N2) {
            const int j2 = u / C;
            V* p = tile + j2 * C + u % C;
            if (two) {
                V w[N1];
#pragma unroll
                for (int k = 0; k < N1; ++k) w[k] = c_scale_rn(v[k], grad_k<T, N>(j2 + N2 * k, two_pi_over_L));
                stage_a_regs<N, DIR>(w, j2, tw);
#pragma unroll
                for (int k1 = 0; k1 < N1; ++k1) p[TS + k1 * N2 * C] = w[k1];
            }
            stage_a_regs<N, DIR>(v, j2, tw);
#pragma unroll
            for (int k1 = 0; k1 < N1; ++k1) p[k1 * N2 * C] = v[k1];
            u += 256;
            if (u < C * N2) fetch();
        }
    }
    __syncthreads();
    // stage B: unit (column, k1, field), lanes over columns
#pragma unroll 1
    for (int u = threadIdx.x; u < (two ? 2 : 1) * C * N1; u += 256) {
        const int c = u % C, k1 = (u / C) % N1, f = u / (C * N1);
        const V* p = tile + f * TS + k1 * N2 * C + c;
        V v[N2];
#pragma unroll
        for (int j = 0; j < N2; ++j) v[j] = p[j * C];
        reg_dft<N2, DIR, V>::run(v);
        V* o = data + src + f * M + (size_t)k1 * N + c;
#pragma unroll
        for (int k2 = 0; k2 < N2; ++k2) o[(size_t)(N1 * k2) * N] = v[k2];
    }
}

// --------------------------------------------------------------------------
// Column order of the xy-transformed arrays (Zxy and H): mirror pairs
// (kx, -kx) are adjacent so that a tile of an even number of positions is
// closed under kx -> -kx. Position 0 holds kx = 0, position 1 kx = n/2, and
// positions 2k, 2k+1 hold kx = k and n - k (k = 1 .. n/2 - 1).
// --------------------------------------------------------------------------
template <int N> __host__ __device__ __forceinline__ int kx_of_pos(int p) {
    return p == 0 ? 0 : p == 1 ? N / 2 : (p & 1) ? N - (p >> 1) : (p >> 1);
}
__host__ __device__ __forceinline__ int mirror_pos(int p) { return p < 2 ? p : (p ^ 1); }
template <int N> __host__ __device__ __forceinline__ int pos_of_kx(int kx) {
    return kx == 0 ? 0 : kx == N / 2 ? 1 : kx < N / 2 ? 2 * kx : 2 * (N - kx) + 1;
}

template <int C, int STRIDE> struct TileAddr {  // buffer b of a tile set starts at b * STRIDE
    __device__ __forceinline__ int operator()(int l) const { return (l / C) * STRIDE + l % C; }
};

// Square of the integer frequency of FFT index i (exact in floats).
template <typename T, int N> __device__ __forceinline__ T freq_sq(int i) {
    const T m = (T)(i < N / 2 ? i : i - N);
    return m * m;
}

// Energy sums of one wavevector with species spectra A, B (times e_rho), each
// times `weight`: [0] u_hat Re[conj(A) B], [1] u_hat |A + B|^2 (k != 0), and
// (WANT_E = 2) [2], [3] the same times m2 = |k L / 2 pi|^2
// (d u_hat / d a = -2 a |k|^2 u_hat).
template <typename T, int WANT_E, class V>
__device__ __forceinline__ void add_energies(Wide<T> (&acc)[5], V A, V B, T uh, T e_rho, T weight, bool zero, T m2) {
    const T ar = A.x * e_rho, ai = A.y * e_rho, br = B.x * e_rho, bi = B.y * e_rho;
    Wide<T> f = Wide<T>::prod(ar, br);
    f.add_prod(ai, bi);
    f = f.times(uh * weight);
    acc[0].add(f);
    if (WANT_E > 1) acc[2].add(f.times(m2));
    Wide<T> q = Wide<T>::sum(ar, br).square();
    q.add(Wide<T>::sum(ai, bi).square());
    q = q.times(zero ? T(0) : uh * weight);
    acc[1].add(q);
    if (WANT_E > 1) acc[3].add(q.times(m2));
}

// --------------------------------------------------------------------------
// z pass: forward DFT along z, spectral multiply + gradient, inverse DFT
// along z. CTA (tile of C column positions, ky pair {ky, -ky}); the tile
// holds every column's mirror, so each CTA has Z(k) and Z(-k) for all of its
// elements and transforms each input line once.
//   R = 1 row when ky = -ky (ky = 0 or n/2), else 2 rows.
// Outputs (linearity: k_x and k_y are constant along a z line):
//   G   = IDFT_z[ i Q ]       (field 0; d_x and d_y follow in the xy pass)
//   G_z = IDFT_z[ i k_z Q ]   (field 2)
// with Q = w~_A + i w~_B. Buffers [2R][N][C]: G of row r in buffer r
// (overwriting the input), G_z in buffer R + r.
// --------------------------------------------------------------------------
//
// Bound by L2 and HBM traffic and by the tail of its 1.1 to 1.7 waves. Each
// value visits shared memory twice and the CTA meets at three barriers, where
// load, transform, multiply and inverse as separate passes visited it five
// times: 24.1 -> 16.9 us at 128^3, 190 -> 114 us at 256^3, 16 column tiles
// (256^3: 8), isolated launches.
//   1. stage A of the forward transform from global memory;
//   2. stage B in registers; the spectral multiply where it left X[k]; and,
//      where the two factors are equal (16, 64, 256), the first stage of the
//      inverse transform on the products without leaving registers: its inputs
//      are the N2 outputs of one stage-B unit;
//   3. the inverse's second stage, to global memory.
// Where the factors differ the inverse's first stage takes N1 points that lie
// in N2 units: the products G go to the slots that their unit read, and a visit
// of shared memory more makes the first stages of G and G_z (128^3: 0.4 us of a
// step). Taking the factors in the other order fuses everywhere, but rounds
// otherwise: that form serves FP64, the potentials and charges, whose results
// are not the sums that nearly cancel.
// The unit (row, column c, k1) of step 2 needs Z(-k) as well, the outputs of
// the mirror unit (mirror row, mirror column, (N1 - k1) mod N1). PAIRED: a
// thread takes both units and writes both; otherwise each unit has its own
// thread, which transforms the mirror unit's inputs a second time (half the
// registers and twice the threads, for tiles that leave threads idle).
template <typename T, int N, int C, bool OTHER = false> struct ZTile {
    static constexpr int N1 = fft_split<N>::N1, N2 = fft_split<N>::N2;
    static constexpr bool paired = 2 * C * N1 > 256, fused = sizeof(T) == 8 || OTHER || N1 == N2 || N2 == 1;
    static_assert(256 % C == 0 && C * N1 <= 256, "every unit of a row has a thread");
};

// fetch(r, z, c): the input of row r; out(b, c, z, v): output element z of
// column c of buffer b (buffers: G of row r in r, G_z in R + r).
template <typename T, int N, int C, bool G_ONLY, bool EL, int WANT_E, class Fetch, class Out>
__device__ __forceinline__ void z_tile(cplx_t<T>* buf, cplx_t<T>* tw, const cplx_t<T>* __restrict__ tw_g, T* e1, T* e2,
                                       const SpectralParams<T>& sp, int p0, const int (&ky)[2], int R, Wide<T> (&acc)[5],
                                       Fetch fetch, Out out) {
    using V = cplx_t<T>;
    constexpr int TS = N * C, N1 = ZTile<T, N, C>::N1, N2 = ZTile<T, N, C>::N2;
    constexpr bool FUSED = ZTile<T, N, C, G_ONLY || EL>::fused;
    {
        int u = threadIdx.x;  // unit (row, j2, column), lanes over columns
        V v[N1];
        auto load = [&]() {
#pragma unroll
            for (int k = 0; k < N1; ++k) v[k] = fetch(u / (C * N2), (u / C) % N2 + N2 * k, u % C);
        };
        const int units = R * C * N2;
        load_twiddles(tw, tw_g, N);
        for (int i = threadIdx.x; i < N; i += 256) {
            e1[i] = sp.kernel1d[i];
            if (EL) e2[i] = sp.kernel1d_el[i];
        }
        dependency_wait();
        if (u < units) load();
        __syncthreads();
#pragma unroll 1
        while (u < units) {
            const int j2 = (u / C) % N2;
            stage_a_regs<N, -1>(v, j2, tw);
            V* p = buf + (u / (C * N2)) * TS + j2 * C + u % C;
#pragma unroll
            for (int k1 = 0; k1 < N1; ++k1) p[k1 * N2 * C] = v[k1];
            u += 256;
            if (u < units) load();
        }
    }
    __syncthreads();
    {
        constexpr bool PAIRED = ZTile<T, N, C>::paired;
        const int q = threadIdx.x;
        const bool active = q < (PAIRED ? 1 : R) * C * N1;
        int c = q % C, k1 = (q / C) % N1, r = PAIRED ? 0 : q / (C * N1);
        int cB = mirror_pos(p0 + c) - p0, k1B = (N1 - k1) % N1, rB = R == 2 ? 1 - r : 0;
        V va[N2], vb[N2];
        if (active) {
            const V* pa = buf + r * TS + k1 * N2 * C + c;
            const V* pb = buf + rB * TS + k1B * N2 * C + cB;
#pragma unroll
            for (int j = 0; j < N2; ++j) {
                va[j] = pa[j * C];
                vb[j] = pb[j * C];
            }
        }
        if (!PAIRED || R == 1) __syncthreads();  // a unit's inputs are read by its mirror's thread too
        if (active) {
            reg_dft<N2, -1, V>::run(va);
            reg_dft<N2, -1, V>::run(vb);
            // unit (r, c, k1): X[k1 + N1 k2] = va[k2]; the mirror of output k2 is
            // vb[(N2 - k2) mod N2] when k1 = 0, else vb[N2 - 1 - k2]. Both
            // densities are real, so the mirror wavevector's products are the
            // conjugates of this one's (u_hat and the Coulomb factor are even):
            // one multiply serves both outputs, which replace va and vb.
            const int kx = kx_of_pos<N>(p0 + c), kyr = ky[r];
            const T exy = e1[kx] * e1[kyr];
            const T exy2 = EL ? e2[kx] * e2[kyr] : T(0);
            const T qx = raw_k<T, N>(kx, sp.two_pi_over_L), qy = raw_k<T, N>(kyr, sp.two_pi_over_L);
            const T kxy2 = fma_rn(qx, qx, mul_rn(qy, qy));  // the Nyquist index counts as -n/2
            const T mxy = freq_sq<T, N>(kx) + freq_sq<T, N>(kyr);
            const T weight = PAIRED && R == 2 ? T(2) : T(1);  // k and -k contribute the same
            const bool zero = kx == 0 && kyr == 0;
            V ga[FUSED ? N2 : 1], gb[FUSED && PAIRED ? N2 : 1];
#pragma unroll
            for (int k2 = 0; k2 < N2; ++k2) {
                const V Z = va[k2], Zm = k1 == 0 ? vb[(N2 - k2) % N2] : vb[N2 - 1 - k2];
                const int kz = k1 + N1 * k2;
                const T uh = exy * e1[kz];
                // rho~_A = (Z + conj Zm)/2, rho~_B = -i (Z - conj Zm)/2
                const V A = {T(0.5) * (Z.x + Zm.x), T(0.5) * (Z.y - Zm.y)};
                const V B = {T(0.5) * (Z.y + Zm.y), -T(0.5) * (Z.x - Zm.x)};
                const V tA = {fma_rn(sp.eAA, A.x, mul_rn(sp.eAB, B.x)), fma_rn(sp.eAA, A.y, mul_rn(sp.eAB, B.y))};
                const V tB = {fma_rn(sp.eAB, A.x, mul_rn(sp.eBB, B.x)), fma_rn(sp.eAB, A.y, mul_rn(sp.eBB, B.y))};
                if (WANT_E)
                    add_energies<T, WANT_E>(acc, A, B, uh, sp.e_rho, weight, zero && kz == 0, mxy + freq_sq<T, N>(kz));
                // G = i (w~_A + i w~_B), k_x and k_y follow in the xy pass, and the same of -k
                V G, Gm;
                if constexpr (!EL) {
                    G = {-fma_rn(uh, tA.y, mul_rn(uh, tB.x)), fma_rn(uh, tA.x, -mul_rn(uh, tB.y))};
                    Gm = {fma_rn(uh, tA.y, -mul_rn(uh, tB.x)), fma_rn(uh, tA.x, mul_rn(uh, tB.y))};
                } else {
                    V wA = {mul_rn(uh, tA.x), mul_rn(uh, tA.y)}, wB = {mul_rn(uh, tB.x), mul_rn(uh, tB.y)};
                    // w_K += q_K c(k) rho~_q with rho~_q = q_A rho~_A + q_B rho~_B
                    const T qzv = raw_k<T, N>(kz, sp.two_pi_over_L);
                    const T k2sq = fma_rn(qzv, qzv, kxy2);
                    const T gq = k2sq > T(0) ? exy2 * e2[kz] * recip(k2sq) : T(0);
                    const V rq = {fma_rn(sp.qA, A.x, mul_rn(sp.qB, B.x)), fma_rn(sp.qA, A.y, mul_rn(sp.qB, B.y))};
                    const T cA = mul_rn(sp.el_scale * gq, sp.qA), cB2 = mul_rn(sp.el_scale * gq, sp.qB);
                    wA.x = fma_rn(cA, rq.x, wA.x);
                    wA.y = fma_rn(cA, rq.y, wA.y);
                    wB.x = fma_rn(cB2, rq.x, wB.x);
                    wB.y = fma_rn(cB2, rq.y, wB.y);
                    if (WANT_E) {
                        Wide<T> f = Wide<T>::prod(rq.x * sp.e_rho, rq.x * sp.e_rho);
                        f.add_prod(rq.y * sp.e_rho, rq.y * sp.e_rho);
                        acc[4].add(f.times(weight * gq));
                    }
                    G = {-(wA.y + wB.x), wA.x - wB.y};
                    Gm = {wA.y - wB.x, wA.x + wB.y};
                }
                if constexpr (FUSED) {
                    ga[k2] = G;
                    if constexpr (PAIRED) gb[k2] = Gm;
                } else {  // to the slots that the units' inputs came from
                    buf[r * TS + (k1 * N2 + k2) * C + c] = G;
                    if constexpr (PAIRED) {
                        const int mk = k1 == 0 ? (N2 - k2) % N2 : N2 - 1 - k2;
                        if (R == 2) buf[rB * TS + (k1B * N2 + mk) * C + cB] = Gm;
                    }
                }
            }
            // the inverse transform's first stage of G and G_z of one unit
            auto emit = [&](V (&g)[N2], int row, int col, int kk) {
                V* o = buf + row * TS + kk * N2 * C + col;
                if constexpr (!G_ONLY) {
                    V gz[N2];
#pragma unroll
                    for (int k2 = 0; k2 < N2; ++k2) gz[k2] = c_scale_rn(g[k2], grad_k<T, N>(kk + N1 * k2, sp.two_pi_over_L));
                    reg_dft<N2, +1, V>::run(gz);
#pragma unroll
                    for (int m = 0; m < N2; ++m) o[R * TS + m * C] = m == 0 ? gz[0] : c_mul(gz[m], twiddle<+1>(tw, kk * m));
                }
                reg_dft<N2, +1, V>::run(g);
#pragma unroll
                for (int m = 0; m < N2; ++m) o[m * C] = m == 0 ? g[0] : c_mul(g[m], twiddle<+1>(tw, kk * m));
            };
            if constexpr (FUSED && PAIRED) {
                int sides = R;
#pragma unroll 1
                while (true) {
                    emit(ga, r, c, k1);
                    if (--sides == 0) break;
                    // the mirror unit, in the order of its own outputs
#pragma unroll
                    for (int k2 = 0; k2 < N2; ++k2) ga[k2] = k1 == 0 ? gb[(N2 - k2) % N2] : gb[N2 - 1 - k2];
                    r = rB;
                    c = cB;
                    k1 = k1B;
                }
            } else if constexpr (FUSED) {
                emit(ga, r, c, k1);
            }
        }
    }
    __syncthreads();
    if constexpr (!FUSED) {
        // the inverse's first stage, in place: unit (row, j2, column) on X[j2 + N2 j1]
#pragma unroll 1
        for (int u = threadIdx.x; u < R * C * N2; u += 256) {
            const int j2 = (u / C) % N2;
            V* p = buf + (u / (C * N2)) * TS + u % C;
            V v[N1];
            auto load = [&]() {
#pragma unroll
                for (int k = 0; k < N1; ++k) v[k] = p[LineSlots<N>::slot_of_part(j2, k) * C];
            };
            load();
            if constexpr (!G_ONLY) {
#pragma unroll
                for (int k = 0; k < N1; ++k) v[k] = c_scale_rn(v[k], grad_k<T, N>(j2 + N2 * k, sp.two_pi_over_L));
                stage_a_regs<N, +1>(v, j2, tw);
#pragma unroll
                for (int k = 0; k < N1; ++k) p[R * TS + LineSlots<N>::slot_of_part(j2, k) * C] = v[k];
                load();  // (a second copy in registers spills)
            }
            stage_a_regs<N, +1>(v, j2, tw);
#pragma unroll
            for (int k = 0; k < N1; ++k) p[LineSlots<N>::slot_of_part(j2, k) * C] = v[k];
        }
        __syncthreads();
    }
    // the second stage: NB points over the NA units
    constexpr int NB = FUSED ? N1 : N2, NA = N / NB;
    const int units = (G_ONLY ? 1 : 2) * R * C * NA;
#pragma unroll 1
    for (int u = threadIdx.x; u < units; u += 256) {
        const int c = u % C, m = (u / C) % NA, b = u / (C * NA);
        const V* p = buf + b * TS + c;
        V v[NB];
#pragma unroll
        for (int k = 0; k < NB; ++k) v[k] = p[(FUSED ? k * NA + m : LineSlots<N>::slot_of_part(k, m)) * C];
        reg_dft<NB, +1, V>::run(v);
#pragma unroll
        for (int k = 0; k < NB; ++k) out(b, c, m + NA * k, v[k]);
    }
}

template <typename T> struct ZArgs {
    const cplx_t<T>* Zxy;
    cplx_t<T>* H;
    const cplx_t<T>* tw;
    SpectralParams<T> sp;
    double* energy_partials;
};

template <typename T, int N, int C, bool G_ONLY = false, bool EL = false, int WANT_E = 0>
__device__ __forceinline__ void z_spectral_body(const ZArgs<T>& args, int bx, int by, int gdx) {
    using V = cplx_t<T>;
    const cplx_t<T>* __restrict__ Zxy = args.Zxy;
    cplx_t<T>* __restrict__ H = args.H;
    const SpectralParams<T> sp = args.sp;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    V* tw = reinterpret_cast<V*>(smem_raw);
    V* buf = tw + N;
    __shared__ T e1[N];  // separable Gaussian kernel: u_hat = e1[kx] e1[ky] e1[kz]
    __shared__ T e2[EL ? N : 1];  // charge smearing exp(-a_e^2 k_m^2), when charges are on

    const int p0 = bx * C;
    const int ky[2] = {by, by == 0 ? 0 : N - by};
    const int R = (ky[0] == ky[1]) ? 1 : 2;
    const size_t NN = (size_t)N * N, M = NN * N;
    Wide<T> acc[5];
    z_tile<T, N, C, G_ONLY, EL, WANT_E>(
        buf, tw, args.tw, e1, e2, sp, p0, ky, R, acc,
        [&](int r, int z, int c) { return __ldcg(Zxy + z * NN + (size_t)ky[r] * N + p0 + c); },
        [&](int b, int c, int z, V v) {
            // G of row r to field 0, G_z to field 2, at (z, ky[r], p0 + c)
            const int f = b < R ? 0 : 2, r = b < R ? b : b - R;
            H[f * M + z * NN + (size_t)ky[r] * N + p0 + c] = v;
        });
    if constexpr (WANT_E != 0) {
        const size_t b = (size_t)by * gdx + bx;
        block_sum<5, T>(acc, [&](int k, double v) { args.energy_partials[5 * b + k] = v; });
    }
}

// The forward z transform alone: the spectrum in natural kx order.
template <typename T, int N, int C>
__global__ void __launch_bounds__(256) z_spectrum(const cplx_t<T>* __restrict__ Zxy, const cplx_t<T>* __restrict__ tw_g,
                                                  cplx_t<T>* __restrict__ spectrum) {
    using V = cplx_t<T>;
    constexpr int N1 = ZTile<T, N, C>::N1, N2 = ZTile<T, N, C>::N2;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    V* tw = reinterpret_cast<V*>(smem_raw);
    V* buf = tw + N;
    load_twiddles(tw, tw_g, N);
    dependency_wait();
    __syncthreads();
    const int p0 = blockIdx.x * C, ky = blockIdx.y;
    const size_t NN = (size_t)N * N;
    for (int u = threadIdx.x; u < C * N2; u += 256) {
        const int c = u % C, j2 = u / C;
        V v[N1];
#pragma unroll
        for (int k = 0; k < N1; ++k) v[k] = Zxy[(j2 + N2 * k) * NN + (size_t)ky * N + p0 + c];
        stage_a_regs<N, -1>(v, j2, tw);
#pragma unroll
        for (int k1 = 0; k1 < N1; ++k1) buf[(k1 * N2 + j2) * C + c] = v[k1];
    }
    __syncthreads();
    for (int u = threadIdx.x; u < C * N1; u += 256) {
        const int c = u % C, k1 = u / C;
        V v[N2];
#pragma unroll
        for (int j = 0; j < N2; ++j) v[j] = buf[(k1 * N2 + j) * C + c];
        reg_dft<N2, -1, V>::run(v);
#pragma unroll
        for (int k2 = 0; k2 < N2; ++k2) spectrum[(k1 + N1 * k2) * NN + (size_t)ky * N + kx_of_pos<N>(p0 + c)] = v[k2];
    }
}

// G_ONLY: write G alone (the potentials' path of the analytic force).
// EL: add the smeared-charge Coulomb term (charges on).
// WANT_E: the energy sums as well (2: and their |k|^2-weighted versions), an
// instantiation of its own, so that the step's kernel carries none of their
// code or registers.
// (Resident CTAs: 16 columns of 128 whose inverse is not fused spill at three
// CTAs' 80 registers, 18.2 us in the step against 17.4 with two.)
template <typename T, int N, int C, bool OTHER = false> __host__ __device__ constexpr int z_ctas() {
    return sizeof(T) == 8 ? 1 : N == 256 ? (C <= 8 ? 2 : 1) : C <= 8 ? 4 : N == 128 && !OTHER ? 2 : 3;
}
template <typename T, int N, int C, bool G_ONLY = false, bool EL = false, int WANT_E = 0>
__global__ void __launch_bounds__(256, z_ctas<T, N, C, G_ONLY || EL>()) z_spectral(const cplx_t<T>* __restrict__ Zxy, cplx_t<T>* __restrict__ H,
                                                  const cplx_t<T>* __restrict__ tw_g, SpectralParams<T> sp,
                                                  double* __restrict__ energy_partials) {
    z_spectral_body<T, N, C, G_ONLY, EL, WANT_E>(ZArgs<T>{Zxy, H, tw_g, sp, energy_partials}, blockIdx.x, blockIdx.y,
                                                 gridDim.x);
}

// Batched form: replica blockIdx.z.
template <typename T, int N, int C, bool EL = false>
__global__ void __launch_bounds__(256, sizeof(T) == 4 ? 3 : 1) z_spectral_batched(const ZArgs<T>* __restrict__ args) {
    z_spectral_body<T, N, C, false, EL>(args[blockIdx.z], blockIdx.x, blockIdx.y, gridDim.x);
}

// --------------------------------------------------------------------------
// z pass with two species pairs (three or four species): as z_spectral, on
// both pairs' columns at once. Buffers [2 NP R][N][C]: the input (then G) of
// pair p, row r in buffer p R + r; G_z in buffer NP R + p R + r. The
// species spectra of pair p are rho~_2p = (Z_p(k) + conj Z_p(-k))/2 and
// rho~_2p+1 = -i (Z_p(k) - conj Z_p(-k))/2; w~_K = u_hat sum_K' eps_KK'
// rho~_K'; Q_p = w~_2p + i w~_2p+1. Energy partials: [0] sum_k u_hat
// sum_{K<K'} chi_KK' Re[conj(rho~_K) rho~_K'], [1] sum_{k != 0} u_hat
// |sum_K rho~_K|^2, the others 0 (rho~ times e_rho).
// --------------------------------------------------------------------------
template <typename T, int NP, class V>
__device__ __forceinline__ void add_energies4(Wide<T> (&acc)[5], const V (&A)[2 * NP], const SpectralParams<T>& sp, T uh, bool zero) {
    V S[2 * NP];
#pragma unroll
    for (int K = 0; K < 2 * NP; ++K) S[K] = {A[K].x * sp.e_rho, A[K].y * sp.e_rho};
    Wide<T> fchi, tr, ti;
#pragma unroll
    for (int K = 0; K < 2 * NP; ++K) {
#pragma unroll
        for (int K2 = K + 1; K2 < 2 * NP; ++K2) {
            Wide<T> f = Wide<T>::prod(S[K].x, S[K2].x);
            f.add_prod(S[K].y, S[K2].y);
            fchi.add(f.times(sp.chi4[K][K2]));
        }
        tr.add(S[K].x);
        ti.add(S[K].y);
    }
    acc[0].add(fchi.times(uh));
    if (!zero) {
        Wide<T> q = tr.square();
        q.add(ti.square());
        acc[1].add(q.times(uh));
    }
}

template <typename T, int N, int C, int R, bool G_ONLY>
__device__ __forceinline__ void z_tile_pairs(cplx_t<T>* buf, const cplx_t<T>* tw, const T* e1, const SpectralParams<T>& sp,
                                             int p0, const int (&ky)[2], bool want_e, Wide<T> (&acc)[5]) {
    using V = cplx_t<T>;
    constexpr int TS = N * C;
    constexpr int NP = 2;
    smem_fft_lines<N, -1, NP * R * C, 256>(buf, TileAddr<C, TS>{}, C, tw);
    static_assert(256 % C == 0, "a thread keeps one column");
    constexpr int rB = R - 1;
    const int c = threadIdx.x % C;
    const int cB = mirror_pos(p0 + c) - p0;
    const int kxA = kx_of_pos<N>(p0 + c), kxB = kx_of_pos<N>(p0 + cB);
    const T exyA = e1[kxA] * e1[ky[0]], exyB = e1[kxB] * e1[ky[rB]];
    const bool zeroA = (kxA == 0 && ky[0] == 0), zeroB = (kxB == 0 && ky[rB] == 0);
    for (int kz = threadIdx.x / C; kz < N; kz += 256 / C) {
        const int kzB = kz == 0 ? 0 : N - kz;
        if (R == 1 && kzB * C + cB < kz * C + c) continue;  // the mirror element owns this pair
        const bool same = (R == 1) && (kzB == kz) && (cB == c);
        V ZA[NP], ZB[NP];
#pragma unroll
        for (int q = 0; q < NP; ++q) {
            ZA[q] = buf[(q * R) * TS + kz * C + c];
            ZB[q] = buf[(q * R + rB) * TS + kzB * C + cB];
        }
        V out[2][NP][2];
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            if (s == 1 && same) break;
            const int kzi = s == 0 ? kz : kzB;
            const T kzv = grad_k<T, N>(kzi, sp.two_pi_over_L);
            const T uh = (s == 0 ? exyA : exyB) * e1[kzi];
            V A[2 * NP];
#pragma unroll
            for (int q = 0; q < NP; ++q) {
                const V Z = s == 0 ? ZA[q] : ZB[q];
                const V Zm = s == 0 ? ZB[q] : ZA[q];
                A[2 * q] = {T(0.5) * (Z.x + Zm.x), T(0.5) * (Z.y - Zm.y)};
                A[2 * q + 1] = {T(0.5) * (Z.y + Zm.y), -T(0.5) * (Z.x - Zm.x)};
            }
            if (want_e) {
                add_energies4<T, NP>(acc, A, sp, uh, (s == 0 ? zeroA : zeroB) && kzi == 0);
            }
            V w[2 * NP];
#pragma unroll
            for (int K = 0; K < 2 * NP; ++K) {
                T wr = 0, wi = 0;
#pragma unroll
                for (int K2 = 0; K2 < 2 * NP; ++K2) {
                    wr += sp.eps4[K][K2] * A[K2].x;
                    wi += sp.eps4[K][K2] * A[K2].y;
                }
                w[K] = {uh * wr, uh * wi};
            }
#pragma unroll
            for (int q = 0; q < NP; ++q) {
                const V iQ = {-(w[2 * q].y + w[2 * q + 1].x), w[2 * q].x - w[2 * q + 1].y};  // i (w~_2q + i w~_2q+1)
                out[s][q][0] = iQ;
                out[s][q][1] = {kzv * iQ.x, kzv * iQ.y};
            }
        }
#pragma unroll
        for (int d = 0; d < 2; ++d) {
            if (d == 1 && G_ONLY) break;
#pragma unroll
            for (int q = 0; q < NP; ++q) {
                buf[(d * NP * R + q * R) * TS + kz * C + c] = out[0][q][d];
                if (!same) buf[(d * NP * R + q * R + rB) * TS + kzB * C + cB] = out[1][q][d];
            }
        }
    }
    __syncthreads();
    smem_fft_lines<N, +1, (G_ONLY ? 1 : 2) * NP * R * C, 256>(buf, TileAddr<C, TS>{}, C, tw);
}

template <typename T, int N, int C, bool G_ONLY = false>
__global__ void __launch_bounds__(256, sizeof(T) == 4 ? 3 : 1) z_spectral_pairs(const cplx_t<T>* __restrict__ Zxy,
                                                                                cplx_t<T>* __restrict__ H,
                                                                                const cplx_t<T>* __restrict__ tw_g,
                                                                                SpectralParams<T> sp,
                                                                                double* __restrict__ energy_partials) {
    using V = cplx_t<T>;
    constexpr int NP = 2;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    V* tw = reinterpret_cast<V*>(smem_raw);
    V* buf = tw + N;
    constexpr int TS = N * C;
    __shared__ T e1[N];
    load_twiddles(tw, tw_g, N);
    for (int i = threadIdx.x; i < N; i += blockDim.x) e1[i] = sp.kernel1d[i];
    dependency_wait();
    const int bx = blockIdx.x, by = blockIdx.y;
    const int p0 = bx * C;
    const int ky[2] = {by, by == 0 ? 0 : N - by};
    const int R = (ky[0] == ky[1]) ? 1 : 2;
    const size_t NN = (size_t)N * N, M = NN * N;
    // buffer b = q R + r (pair q, row r)
    auto zsrc = [&](int i) {
        const int b = i / TS, rem = i % TS;
        const int q = b / R, r = b % R;
        const int z = rem / C, c = rem % C;
        return __ldcg(Zxy + q * M + z * NN + (size_t)ky[r] * N + p0 + c);
    };
    auto zdst = [&](int i, V v) { buf[i] = v; };
    if (R == 1)
        batched_load<NP * TS, 256, V>(zsrc, zdst);
    else
        batched_load<NP * 2 * TS, 256, V>(zsrc, zdst);
    __syncthreads();
    Wide<T> acc[5];
    const bool want_e = energy_partials != nullptr;
    if (R == 1)
        z_tile_pairs<T, N, C, 1, G_ONLY>(buf, tw, e1, sp, p0, ky, want_e, acc);
    else
        z_tile_pairs<T, N, C, 2, G_ONLY>(buf, tw, e1, sp, p0, ky, want_e, acc);
    if (want_e) {
        const size_t b = (size_t)by * gridDim.x + bx;
        block_sum<5, T>(acc, [&](int k, double v) { energy_partials[5 * b + k] = v; });
    }
    // buffer b = (d NP + q) R + r: field 0 (G) or 2 (G_z) of pair q, row r
    const int nbuf = (G_ONLY ? 1 : 2) * NP * R * TS;
    for (int i = threadIdx.x; i < nbuf; i += blockDim.x) {
        const int b = i / TS, rem = i % TS;
        const int d = b / (NP * R), q = (b / R) % NP, r = b % R;
        const int z = rem / C, c = rem % C;
        H[(3 * q + 2 * d) * M + z * NN + (size_t)ky[r] * N + p0 + c] = buf[i];
    }
}

// The z pass's energy sums in FP64, not scaled, from the spectra Z in natural
// order ([NP][nz][n][n]; any n, one layer in two dimensions): [0 .. 4] of
// add_energies (one pair; the Coulomb sum with el) or add_energies4. Takes the
// place of an FP32 context's Wide sums that left the range of floats.
template <typename T, int NP>
__global__ void __launch_bounds__(256) spectral_sums64(const cplx_t<T>* __restrict__ Z, int n, int nz, SpectralParams<T> sp, int el,
                                                       double* __restrict__ partials) {
    using V = cplx_t<T>;
    const size_t M = (size_t)nz * n * n, g = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    Wide<double> acc[5];
    if (g < M) {
        const int i[3] = {(int)(g % n), (int)((g / n) % n), (int)(g / ((size_t)n * n))}, len[3] = {n, n, nz};
        size_t gm = 0;
        T uh = T(1), uc = T(1), q[3] = {T(0), T(0), T(0)};
        double m2 = 0.0;
        for (int d = 2; d >= 0; --d) gm = gm * len[d] + (i[d] == 0 ? 0 : len[d] - i[d]);
        for (int d = 0; d < (nz > 1 ? 3 : 2); ++d) {
            const T m = (T)(2 * i[d] < len[d] ? i[d] : i[d] - len[d]);
            uh *= sp.kernel1d[i[d]];
            if (el) uc *= sp.kernel1d_el[i[d]];
            q[d] = sp.two_pi_over_L * m;
            m2 += (double)m * m;
        }
        V A[2 * NP];
        double tr = 0.0, ti = 0.0, chi = 0.0;
        for (int q = 0; q < NP; ++q) {
            const V Zk = Z[q * M + g], Zm = Z[q * M + gm];
            A[2 * q] = {T(0.5) * (Zk.x + Zm.x), T(0.5) * (Zk.y - Zm.y)};
            A[2 * q + 1] = {T(0.5) * (Zk.y + Zm.y), -T(0.5) * (Zk.x - Zm.x)};
        }
        for (int K = 0; K < 2 * NP; ++K) {
            tr += A[K].x;
            ti += A[K].y;
            for (int K2 = K + 1; K2 < 2 * NP; ++K2)
                chi += (NP == 1 ? 1.0 : (double)sp.chi4[K][K2]) * ((double)A[K].x * A[K2].x + (double)A[K].y * A[K2].y);
        }
        const double fchi = uh * chi, fkap = g == 0 ? 0.0 : uh * (tr * tr + ti * ti);
        acc[0].add(fchi);
        acc[1].add(fkap);
        acc[2].add(m2 * fchi);
        acc[3].add(m2 * fkap);
        const T k2 = fma_rn(q[2], q[2], fma_rn(q[0], q[0], mul_rn(q[1], q[1])));
        if (el && k2 > T(0)) {
            const double rx = fma_rn(sp.qA, A[0].x, mul_rn(sp.qB, A[1].x)), ry = fma_rn(sp.qA, A[0].y, mul_rn(sp.qB, A[1].y));
            acc[4].add((double)(uc * recip(k2)) * (rx * rx + ry * ry));
        }
    }
    block_sum<5, double>(acc, [&](int k, double s) { partials[5 * (size_t)blockIdx.x + k] = s; });
}

}  // namespace tild
