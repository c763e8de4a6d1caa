// Host engine of the TILD step: owns device buffers, launches the kernels
// of one step in stream order and replays whole re-binning cycles as CUDA
// graphs. Instantiated once per precision (engine_f32.cu, engine_f64.cu).
#pragma once

#include <algorithm>
#include <unordered_map>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <string>
#include <vector>

#include <nvtx3/nvToolsExt.h>

#include "bead_kernels.cuh"
#include "vjp_kernels.cuh"
#include "engine_api.h"
#include "grid_kernels.cuh"
#include "generic_kernels.cuh"

namespace tild {

#define TILD_CUDA(call)                                                                        \
    do {                                                                                       \
        cudaError_t e_ = (call);                                                               \
        if (e_ != cudaSuccess) {                                                               \
            err = std::string(#call) + ": " + cudaGetErrorString(e_);                          \
            return e_ == cudaErrorMemoryAllocation ? TILD_ENOMEM : TILD_EDEVICE;               \
        }                                                                                      \
    } while (0)

constexpr uint64_t kStateMagic = 0x54494c4453544154ull;  // "TILDSTAT"

template <typename T> class BatchEngine;

template <typename T> class Engine final : public EngineBase {
    using V = cplx_t<T>;
    friend class BatchEngine<T>;

   public:
    ~Engine() override { release(); }

    tild_status init(HostConfig* cfg) override {
        cfg_ = cfg;
        n_ = cfg->n;
        generic_ = cfg->generic;
        nz_ = cfg->dim == 2 ? 1 : n_;
        M_ = (size_t)nz_ * n_ * n_;
        tiles_ = (n_ + kTile - 1) / kTile;
        P_ = cfg->pmeorder + 1;
        plane_fits_ = plane_fits(n_, sizeof(V));
        // default launch shape of the planes (tild_set_launch_shapes, tild_autotune
        // choose others): 512 threads; 1,024 at 128^3 FP32, whose one CTA per SM
        // leaves its latency to them; at 64^3 FP64 the row and column passes, which
        // spread over every SM's FP64 unit where 64 planes reach 64 of 152. Step at
        // 0.4 beads per point, us, as rows and columns / 512 / 1,024 threads:
        //   FP64  24^3 53/48  32^3 58/55  40^3 77/83  48^3 160/127  64^3 222/260  80^3 563/514
        //   FP32  48^3 23/20  64^3 27/26  80^3 47/42/44  128^3 131/126/122
        // (40^3 FP64 would gain too and keeps its planes.)
        plane_nt_ = sizeof(T) == 4 && n_ == 128 ? 1024 : sizeof(T) == 8 && n_ == 64 ? 0 : 512;
        C_ = std::min(n_, (int)(128 / sizeof(V)));  // y-column tiles of the split passes
        CZ_ = zpass_cols(n_);                          // column tiles of the z pass
        TILD_CUDA(cudaGetDevice(&device_));
        TILD_CUDA(cudaStreamCreateWithFlags(&own_stream_, cudaStreamNonBlocking));
        stream_ = own_stream_;
        tild_status gst = alloc_grids(1);
        if (gst) return gst;
        TILD_CUDA(dev_malloc((void**)&tw_, n_ * sizeof(V)));
        TILD_CUDA(dev_malloc((void**)&kernel1d_, 2 * n_ * sizeof(T)));  // exp(-a^2 k_m^2), then exp(-a_e^2 k_m^2)
        TILD_CUDA(dev_malloc((void**)&counters_, kWords * sizeof(unsigned long long)));
        TILD_CUDA(cudaMemset(counters_, 0, kWords * sizeof(unsigned long long)));
        // tiles of 8^3 cells (one layer of tiles on a 2D grid)
        n_tiles_ = tiles_ * tiles_ * ((nz_ + kTile - 1) / kTile);
        n_fine_ = (size_t)kFineBins * n_tiles_ + 1;  // re-binning bins (tile, edge class, bank group)
        TILD_CUDA(dev_malloc((void**)&counts_, n_fine_ * sizeof(int)));
        TILD_CUDA(cudaMemset(counts_, 0, n_fine_ * sizeof(int)));  // and every re-binning leaves it zero
        TILD_CUDA(dev_malloc((void**)&tile_start_, (n_tiles_ + 1) * sizeof(int)));
        TILD_CUDA(dev_malloc((void**)&fine_start_, n_fine_ * sizeof(int)));
        scan_blocks_ = (int)((n_fine_ + 1023) / 1024);
        TILD_CUDA(dev_malloc((void**)&block_sums_, scan_blocks_ * sizeof(int)));
        n_z_blocks_ = generic_ ? (size_t)blocks(M_) : (size_t)(n_ / CZ_) * (n_ / 2 + 1);  // two species pairs: twice as many (zpass_cols2)
        n_partials_ = std::max(10 * n_z_blocks_, 5 * (size_t)tiles_ * tiles_ * tiles_);  // 8 bytes each
        n_partials_ = std::max(n_partials_, 3 * (size_t)(n_ / vjp_cols(n_)) * (n_ / 2 + 1));
        TILD_CUDA(dev_malloc((void**)&partials_, n_partials_ * sizeof(double)));
        partials_bytes_ = n_partials_ * sizeof(double);
        // twiddles W_n^m = exp(-2 pi i m / n) in FP64, rounded to T
        std::vector<V> tw(n_);
        for (int m = 0; m < n_; ++m) {
            const double ang = -2.0 * 3.14159265358979323846 * (double)m / (double)n_;
            tw[m] = V{(T)std::cos(ang), (T)std::sin(ang)};
        }
        TILD_CUDA(cudaMemcpy(tw_, tw.data(), n_ * sizeof(V), cudaMemcpyHostToDevice));
        if (generic_) {
            TILD_CUDA(cudaFuncSetAttribute(generic_axis_fft<T, -1>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)gaxis_smem()));
            TILD_CUDA(cudaFuncSetAttribute(generic_axis_fft<T, +1>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)gaxis_smem()));
            // the two factors of the line length: the most balanced split n = n1 n2
            gn1_ = 1;
            for (int f = 1; f * f <= n_; ++f)
                if (n_ % f == 0) gn1_ = f;
            gn2_ = n_ / gn1_;
            TILD_CUDA(cudaFuncSetAttribute(line_x_forward<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, kLineSmem));
            TILD_CUDA(cudaFuncSetAttribute(line_x_inverse<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, kLineSmem));
            TILD_CUDA(cudaFuncSetAttribute(line_y<T, -1>, cudaFuncAttributeMaxDynamicSharedMemorySize, kLineSmem));
            TILD_CUDA(cudaFuncSetAttribute(line_y<T, +1>, cudaFuncAttributeMaxDynamicSharedMemorySize, kLineSmem));
            TILD_CUDA(cudaFuncSetAttribute(line_last<T, 1, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize, kLineSmem));
            TILD_CUDA(cudaFuncSetAttribute(line_last<T, 2, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize, kLineSmem));
            TILD_CUDA(cudaFuncSetAttribute(line_last<T, 1, 3>, cudaFuncAttributeMaxDynamicSharedMemorySize, kLineSmem));
            TILD_CUDA(cudaFuncSetAttribute(line_last<T, 2, 3>, cudaFuncAttributeMaxDynamicSharedMemorySize, kLineSmem));
            return TILD_OK;
        }
        return set_kernel_attributes();
    }

    tild_status set_chains() override {
        invalidate_graph();
        free_beads();
        if (NP_ != 1) {
            tild_status gst = alloc_grids(1);  // the chains give two species
            if (gst) return gst;
        }
        const size_t N = (size_t)cfg_->n_beads;
        for (int k = 0; k < 2; ++k) {
            TILD_CUDA(dev_malloc((void**)&pos_[k], 3 * N * sizeof(T)));
            TILD_CUDA(dev_malloc((void**)&u_[k], 3 * N * sizeof(T)));
            TILD_CUDA(dev_malloc((void**)&id_[k], N * sizeof(int)));
            TILD_CUDA(cudaMemset(u_[k], 0, 3 * N * sizeof(T)));
        }
        TILD_CUDA(dev_malloc((void**)&nbr_, N * sizeof(int2)));
        TILD_CUDA(dev_malloc((void**)&slot_of_id_, N * sizeof(int)));
        TILD_CUDA(dev_malloc((void**)&keys_, N * sizeof(int)));
        TILD_CUDA(dev_malloc((void**)&ranks_, N * sizeof(int)));
        have_pos_ = have_vel_ = false;
        return upload_topology();
    }

    // Species count, per-bead species and bond list from the HostConfig:
    // grids for the species pairs, the device topology arrays, and (with
    // positions) a re-binning and a fresh density.
    tild_status set_topology() override {
        invalidate_graph();
        tild_status st;
        const int np = cfg_->n_species > 2 ? 2 : 1;  // pairs of species on the grids
        if (np != NP_ && (st = alloc_grids(np))) return st;
        if ((st = upload_topology())) return st;
        if (have_pos_) {
            if ((st = enqueue_sort()) || (st = respread())) return st;
            TILD_CUDA(cudaStreamSynchronize(stream_));
        }
        return TILD_OK;
    }

    tild_status io_scratch(size_t bytes, void** ptr) override {
        tild_status st;
        if ((st = device_buffer(&io_, io_bytes_, bytes))) return st;
        *ptr = io_;
        return TILD_OK;
    }

    tild_status transpose3(const void* in, void* out, size_t n, int dtype, bool to_aos) override {
        if (dtype == TILD_DTYPE_F32)
            transpose_vec3<float><<<blocks(3 * n), 256, 0, stream_>>>(n, (const float*)in, (float*)out, to_aos);
        else
            transpose_vec3<double><<<blocks(3 * n), 256, 0, stream_>>>(n, (const double*)in, (double*)out, to_aos);
        TILD_CUDA(cudaGetLastError());
        TILD_CUDA(cudaStreamSynchronize(stream_));
        return TILD_OK;
    }

    tild_status set_stream(cudaStream_t s) override {
        invalidate_graph();
        stream_ = s ? s : own_stream_;
        return TILD_OK;
    }
    cudaStream_t stream() const override { return stream_; }

    tild_status set_positions(const void* xyz, int dtype, int where) override {
        const int N = cfg_->n_beads;
        const void* src = xyz;
        tild_status st = stage_in(&src, xyz, (size_t)3 * N, dtype, where);
        if (st) return st;
        cur_pos_ = cur_u_ = cur_id_ = 0;
        const T L = (T)cfg_->L;
        if (dtype == TILD_DTYPE_F32)
            load_positions<T, float><<<blocks(N), 256, 0, stream_>>>(N, (const float*)src, L, (T)(1.0 / cfg_->L), pos_[0], id_[0], err_ptr());
        else
            load_positions<T, double><<<blocks(N), 256, 0, stream_>>>(N, (const double*)src, L, (T)(1.0 / cfg_->L), pos_[0], id_[0], err_ptr());
        TILD_CUDA(cudaGetLastError());
        if ((st = zero_z())) return st;
        if ((st = enqueue_sort())) return st;
        if ((st = respread())) return st;
        if ((st = finish())) return st;
        have_pos_ = true;
        have_vel_ = false;
        return TILD_OK;
    }

    tild_status set_velocities(const void* v, int dtype, int where) override {
        const int N = cfg_->n_beads;
        tild_status st;
        const T* vin = nullptr;
        if (v) {
            // bring to device in precision T (AoS by id)
            const void* src = v;
            if ((st = stage_in(&src, v, (size_t)3 * N, dtype, where))) return st;
            if ((st = ensure_aux((size_t)3 * N * sizeof(T)))) return st;
            if (dtype == TILD_DTYPE_F32)
                convert_copy<float, T><<<blocks(3 * (size_t)N), 256, 0, stream_>>>((size_t)3 * N, (const float*)src, (T*)aux_);
            else
                convert_copy<double, T><<<blocks(3 * (size_t)N), 256, 0, stream_>>>((size_t)3 * N, (const double*)src, (T*)aux_);
            TILD_CUDA(cudaGetLastError());
            vin = (const T*)aux_;
        }
        if ((st = enqueue_fields(0, nullptr, nullptr))) return st;
        BeadBuffers<T> bf = bead_buffers();
        bf.v_in = vin;
        if ((st = launch_bead(kModeSetVel, bf))) return st;
        TILD_CUDA(cudaMemsetAsync(counters_, 0, 4 * sizeof(unsigned long long), stream_));
        TILD_CUDA(cudaStreamSynchronize(stream_));
        host_step_ = 0;
        steps_since_sort_ = 0;
        have_vel_ = true;
        return TILD_OK;
    }

    tild_status step(int64_t n) override {
        tild_status st;
        const int K = cfg_->sort_every;
        while (n > 0) {
            if (steps_since_sort_ >= K && n >= 2 * (int64_t)K) {
                // a full cycle (sort, K steps, sort, K steps) as one graph
                if ((st = run_cycle_graph())) return st;
                n -= 2 * (int64_t)K;
                host_step_ += 2 * (int64_t)K;
                continue;
            }
            if (steps_since_sort_ >= K) {
                if ((st = enqueue_sort())) return st;
            }
            if ((st = enqueue_step())) return st;
            --n;
            ++host_step_;
        }
        return TILD_OK;
    }

    tild_status synchronize() override {
        return finish();
    }

    tild_status compute(unsigned what, tild_energy* e, void* f, int dtype, int where) override {
        tild_status st;
        const bool want_e = (what & TILD_COMPUTE_ENERGY) != 0;
        if ((st = ensure_partials())) return st;
        if ((st = enqueue_fields(want_e ? 1 : 0, partials_, nullptr))) return st;
        if (want_e && (st = reduce_partials(z_blocks(), 5, sums()))) return st;
        BeadBuffers<T> bf = bead_buffers();
        if (e) bf.partials = partials_;
        const size_t n3 = (size_t)3 * cfg_->n_beads;
        const bool direct = f && device_native(dtype, where);  // the kernel writes the caller's array
        if (f) {
            if (!direct && (st = ensure_aux(n3 * sizeof(T)))) return st;
            bf.f_out = direct ? (T*)f : (T*)aux_;
        }
        if ((st = launch_bead(kModeForce, bf))) return st;
        if (e && (st = reduce_partials(bead_blocks(), 5, sums() + 5))) return st;
        if (f && !direct && (st = stage_out_vec((T*)aux_, n3, f, dtype, where))) return st;
        if ((st = finish())) return st;
        const BeadParams<T> p = bead_params();
        double h[10], el = p.e_len, ev = p.e_vel, er = spectral_params().e_rho;
        std::copy(host_sums(), host_sums() + 10, h);
        if (e) {
            const bool bead_ok = wide_in_range<T>(h[5], !has_bonds()) && wide_in_range<T>(h[6], p.vu == T(0) && p.vf == T(0) && p.vg == T(0)) &&
                                 std::isfinite(h[7] + h[8] + h[9]);
            const bool k_ok = !want_e || (wide_in_range<T>(h[0], true) && wide_in_range<T>(h[1], true) && wide_in_range<T>(h[4], true));
            if (sizeof(T) == 4 && !(bead_ok && k_ok)) {
                if ((st = sums_fp64(want_e, true, h))) return st;
                el = ev = er = 1.0;
            }
        }
        if (e) {
            e->e_bond = 0.75 / (cfg_->b * cfg_->b) * h[5] / (el * el);  // every bond from both ends
            e->kinetic = 0.5 * cfg_->mass * h[6] / (ev * ev);
            for (int d = 0; d < 3; ++d) e->net_force[d] = h[7 + d];
            e->e_chi = e->e_kappa = e->e_elec = 0.0;
        }
        if (want_e && e) {
            const double V = volume();
            const double dV = V / (double)M_;
            const double rho0 = cfg_->n_beads / V;
            // one pair: the z pass sums Re[conj(rho_A) rho_B]; two pairs: chi-weighted sums
            e->e_chi = (NP_ == 1 ? cfg_->chi : 1.0) / rho0 * dV * dV / V * (h[0] / (er * er));
            e->e_kappa = cfg_->kappa / (2.0 * rho0) * dV * dV / V * (h[1] / (er * er));
            e->e_elec = e_elec_from(h[4] / (er * er));
        }
        return TILD_OK;
    }

    tild_status energy_gradient(tild_energy_grad* g, void* dUdr, int dtype, int where) override {
        tild_status st;
        if (generic_) {
            err = "energy_gradient: implemented for the 3D grid sizes of the tiled kernels";
            return TILD_EUNSUPPORTED;
        }
        if (NP_ != 1) {
            err = "energy_gradient: implemented for one or two species";
            return TILD_EUNSUPPORTED;
        }
        const size_t N = cfg_->n_beads;
        if ((st = device_buffer(&partials_, partials_bytes_, std::max(partials_bytes_, (size_t)blocks(N) * sizeof(double))))) return st;
        if ((st = enqueue_fields(2, partials_, nullptr, kInvPot))) return st;
        if ((st = reduce_partials(n_z_blocks_, 5, sums()))) return st;
        BeadBuffers<T> bf = bead_buffers();
        bf.partials = partials_;
        const bool direct = dUdr && device_native(dtype, where);
        if (dUdr && !direct && (st = ensure_aux(3 * N * sizeof(T)))) return st;
        T* out = !dUdr ? nullptr : direct ? (T*)dUdr : (T*)aux_;
        const BeadParams<T> p = bead_params();
        const V* pot = grad_ + 3 * M_;
        if ((st = dispatch_p([&](auto pp) -> tild_status {
                 adjoint_kernel<decltype(pp)::value, T><<<blocks(N), 256, 0, stream_>>>(p, bf, pot, out);
                 return TILD_OK;
             })))
            return st;
        TILD_CUDA(cudaGetLastError());
        if ((st = reduce_partials(blocks(N), 1, sums() + 5))) return st;
        if (dUdr && !direct && (st = stage_out_vec((T*)aux_, 3 * N, dUdr, dtype, where))) return st;
        if ((st = finish())) return st;
        const double kk = 2.0 * 3.14159265358979323846 / cfg_->L;
        double s[6], el = p.e_len, er = spectral_params().e_rho;
        std::copy(host_sums(), host_sums() + 6, s);
        bool ok = wide_in_range<T>(s[5], !has_bonds());
        for (int k = 0; k < 5; ++k) ok = ok && wide_in_range<T>(s[k], true);
        if (sizeof(T) == 4 && !ok) {
            if ((st = sums_fp64(true, false, s))) return st;
            el = er = 1.0;
        }
        for (int k = 0; k < 5; ++k) s[k] /= er * er;
        s[2] *= kk * kk;  // summed with integer frequencies
        s[3] *= kk * kk;
        const double eb = 0.75 / (cfg_->b * cfg_->b) * s[5] / (el * el);
        const double V = cfg_->L * cfg_->L * cfg_->L;
        const double dV = V / (double)M_;
        const double rho0 = cfg_->n_beads / V;
        const double f = dV * dV / V;
        // E_chi = chi/rho0 f S0, E_kappa = kappa/(2 rho0) f S1; d u_hat/d a = -2 a |k|^2 u_hat
        g->e_bond = eb;
        g->e_chi = cfg_->chi / rho0 * f * s[0];
        g->e_kappa = cfg_->kappa / (2.0 * rho0) * f * s[1];
        g->e_elec = e_elec_from(s[4]);
        g->energy = g->e_bond + g->e_chi + g->e_kappa + g->e_elec;
        g->dU_dchi = f * s[0] / rho0;
        g->dU_dkappa = f * s[1] / (2.0 * rho0);
        g->dU_da = -2.0 * cfg_->a * (cfg_->chi / rho0 * f * s[2] + cfg_->kappa / (2.0 * rho0) * f * s[3]);
        return TILD_OK;
    }

    tild_status vjp_supported() {
        if (generic_) {
            err = "force_vjp: implemented for the 3D grid sizes of the tiled kernels";
            return TILD_EUNSUPPORTED;
        }
        if (NP_ != 1) {
            err = "force_vjp: implemented for one or two species";
            return TILD_EUNSUPPORTED;
        }
        if (analytic()) {
            err = "force_vjp: implemented for the ik force";
            return TILD_EUNSUPPORTED;
        }
        if (!plane_fits_) {
            err = "force_vjp: the grid must fit the single-plane xy passes (FP32 up to 128^3, FP64 up to 64^3)";
            return TILD_EUNSUPPORTED;
        }
        return TILD_OK;
    }
    size_t vjp_blocks() const { return (size_t)(n_ / vjp_cols(n_)) * (n_ / 2 + 1); }
    // fixed-point bits of the adjoint spread: S = min(S_max, 62 - ceil(log2 n_beads))
    int vjp_fixed_bits() const {
        int lg = 0;
        while ((1ull << lg) < (unsigned long long)cfg_->n_beads) ++lg;
        return std::min(AdjointFixed<T>::s_max, 62 - lg);
    }
    // the fixed-point spread [3][M] int64 pairs and the max|lam| bits, zero
    // between calls (the xy pass and the z pass of a VJP leave them so)
    size_t vjp_fx_need() const { return 6 * M_ * sizeof(unsigned long long) + 16; }
    tild_status vjp_prepare() {
        tild_status st;
        if ((st = vjp_supported())) return st;
        if (vjp_fx_bytes_ >= vjp_fx_need()) return TILD_OK;
        if ((st = device_buffer(&vjp_fx_, vjp_fx_bytes_, vjp_fx_need()))) return st;
        TILD_CUDA(cudaMemsetAsync(vjp_fx_, 0, vjp_fx_need(), stream_));
        return TILD_OK;
    }

    // J^T lam at the positions of bf into out_d (T, by id), and the parameter
    // sums added to theta_acc (device, 3 doubles); stream-ordered, no host
    // synchronisation (see vjp_kernels.cuh). fields, zxy: D w and the
    // xy-transformed density of those positions, as a step starting from them
    // leaves them (null: computed here, for the context's own positions).
    tild_status vjp_core(const T* lam_d, T* out_d, double* theta_acc, const BeadBuffers<T>& bf, const V* fields = nullptr,
                         const V* zxy = nullptr) {
        const size_t N = cfg_->n_beads;
        tild_status st;
        if (!fields) {
            if ((st = enqueue_fields(0, nullptr, nullptr, kInvGrad))) return st;  // D w at r; Zxy = xy(rho)
            fields = grad_;
            zxy = Zxy_;
        }
        using Bits = typename AdjointFixed<T>::bits_t;
        unsigned long long* fx = (unsigned long long*)vjp_fx_;
        Bits* bits = (Bits*)(fx + 6 * M_);
        const int S = vjp_fixed_bits();
        launch(lam_absmax<T>, (int)std::min<size_t>(blocks(3 * N), 2 * 152), 256, 0, 3 * N, lam_d, bits);
        const BeadParams<T> p = bead_params();
        if ((st = dispatch_p([&](auto pp) -> tild_status {
                 constexpr int P = decltype(pp)::value;
                 if constexpr (sizeof(T) == 4)
                     launch(vjp_spread_tiled<P>, n_tiles_, 256, vjp_spread_smem<P>(), p, bf, lam_d, fx, bits, S);
                 else
                     vjp_spread<P, T><<<blocks(N), 256, 0, stream_>>>(p, bf, lam_d, fx, bits, S);
                 return TILD_OK;
             })))
            return st;
        const SpectralParams<T> sp = spectral_params();
        const int el = c_el_on() ? 1 : 0;
        if ((st = dispatch_n([&](auto nn) -> tild_status {
                 constexpr int NN = decltype(nn)::value;
                 if constexpr (plane_fits(NN, sizeof(V))) {
                     constexpr int CV = vjp_cols(NN);
                     launch(xy_forward_cplx<T, NN>, dim3(NN, 3), 512, plane_smem(), (longlong2*)fx, bits, S, H_, tw_);
                     launch(z_vjp<T, NN, CV>, dim3(NN / CV, NN / 2 + 1), 256, vjp_smem(), H_, zxy, tw_, sp, partials_, el, bits);
                 }
                 return TILD_OK;
             })))
            return st;
        TILD_CUDA(cudaGetLastError());
        launch(accumulate_partials, 1, 256, 0, partials_, (int)vjp_blocks(), theta_acc);
        if ((st = enqueue_inverse(kInvPot))) return st;  // psi into the potential slot
        const double dV = cfg_->L * cfg_->L * cfg_->L / (double)M_;
        const V* psi = grad_ + 3 * M_;
        if ((st = dispatch_p([&](auto pp) -> tild_status {
                 constexpr int P = decltype(pp)::value;
                 if constexpr (sizeof(T) == 4)
                     launch(vjp_beads_tiled<P>, n_tiles_, 256, vjp_beads_smem<P>(), p, bf, fields, psi, lam_d, (T)(1.0 / dV), out_d);
                 else
                     vjp_beads<P, T><<<blocks(N), 256, 0, stream_>>>(p, bf, fields, psi, lam_d, (T)(1.0 / dV), out_d);
                 return TILD_OK;
             })))
            return st;
        TILD_CUDA(cudaGetLastError());
        return TILD_OK;
    }
    // d(lam . F)/d(chi, kappa, a) from the accumulated sums
    void theta_from_sums(const double* s, double* dtheta) const {
        const double rho0 = cfg_->n_beads / (cfg_->L * cfg_->L * cfg_->L);
        dtheta[0] = s[0] / (rho0 * (double)M_);
        dtheta[1] = s[1] / (rho0 * (double)M_);
        dtheta[2] = -2.0 * cfg_->a * s[2];
    }
    // a device scratch of `bytes` that lives as long as the context
    template <class P> tild_status device_buffer(P** ptr, size_t& have, size_t bytes) {
        if (have >= bytes) return TILD_OK;
        TILD_CUDA(cudaStreamSynchronize(stream_));
        dev_free(*ptr);
        *ptr = nullptr;
        have = 0;
        TILD_CUDA(dev_malloc((void**)ptr, bytes));
        have = bytes;
        return TILD_OK;
    }

    // J^T lam of the ik force at the current positions; dtheta (optional):
    // d(lam . F)/d(chi, kappa, a).
    tild_status force_vjp(const void* lam, void* out, int dtype, int where, double* dtheta) override {
        tild_status st;
        if ((st = vjp_prepare())) return st;
        const size_t N = cfg_->n_beads, bytes = 3 * N * sizeof(T);
        const bool direct = device_native(dtype, where);  // the kernels read and write the caller's arrays
        const bool overlap = (const char*)lam < (const char*)out + bytes && (const char*)out < (const char*)lam + bytes;
        T* out_d = (T*)out;
        const T* lam_d = (const T*)lam;
        if (!direct || overlap) {
            const void* src = lam;
            if ((st = stage_in(&src, lam, 3 * N, dtype, where))) return st;
            if ((st = ensure_aux(2 * bytes))) return st;
            T* copy = (T*)aux_;
            if (dtype == TILD_DTYPE_F32)
                convert_copy<float, T><<<blocks(3 * N), 256, 0, stream_>>>(3 * N, (const float*)src, copy);
            else
                convert_copy<double, T><<<blocks(3 * N), 256, 0, stream_>>>(3 * N, (const double*)src, copy);
            TILD_CUDA(cudaGetLastError());
            lam_d = copy;
            if (!direct) out_d = copy + 3 * N;
        }
        TILD_CUDA(cudaMemsetAsync(sums(), 0, 3 * sizeof(double), stream_));
        if ((st = vjp_core(lam_d, out_d, sums(), bead_buffers()))) return st;
        if (!direct && (st = stage_out_vec(out_d, 3 * N, out, dtype, where))) return st;
        if ((st = finish())) return st;
        if (dtheta) theta_from_sums(host_sums(), dtheta);
        return TILD_OK;
    }

    // d/dr_i of sum_{K,g} psi_K(g) rho_K(g) for a grid adjoint psi [S][M]
    // (dtype/where), by bead id ([N][3], dtype/where).
    tild_status density_vjp(const void* psi, void* out, int dtype, int where) override {
        if (cfg_->dim != 3) {
            err = "density_vjp: three-dimensional boxes";
            return TILD_EUNSUPPORTED;
        }
        tild_status st;
        const size_t N = cfg_->n_beads, G = (size_t)cfg_->n_species * M_;
        const bool direct = device_native(dtype, where);
        const bool overlap = (const char*)psi < (const char*)out + 3 * N * sizeof(T) &&
                             (const char*)out < (const char*)psi + G * sizeof(T);
        const T* psi_d = (const T*)psi;
        T* out_d = (T*)out;
        if (!direct || overlap) {
            const void* src = psi;
            if ((st = stage_in(&src, psi, G, dtype, where))) return st;
            if ((st = ensure_aux((G + 3 * N) * sizeof(T)))) return st;
            T* copy = (T*)aux_;
            if (dtype == TILD_DTYPE_F32)
                convert_copy<float, T><<<blocks(G), 256, 0, stream_>>>(G, (const float*)src, copy);
            else
                convert_copy<double, T><<<blocks(G), 256, 0, stream_>>>(G, (const double*)src, copy);
            TILD_CUDA(cudaGetLastError());
            psi_d = copy;
            if (!direct) out_d = copy + G;
        }
        const BeadParams<T> p = bead_params();
        const BeadBuffers<T> bf = bead_buffers();
        const T inv_dV = (T)((double)M_ / volume());
        if ((st = dispatch_p([&](auto pp) -> tild_status {
                 density_vjp_kernel<decltype(pp)::value, T><<<blocks(N), 256, 0, stream_>>>(p, bf, psi_d, inv_dV, out_d);
                 return TILD_OK;
             })))
            return st;
        TILD_CUDA(cudaGetLastError());
        if (!direct && (st = stage_out_vec(out_d, 3 * N, out, dtype, where))) return st;
        return finish();
    }

    // positions and carried velocities by id ([2][N][3] T) <-> the context
    void store_state(T* dst) {
        const int N = cfg_->n_beads;
        store_by_id<T, T><<<blocks(N), 256, 0, stream_>>>(N, pos_[cur_pos_], id_[cur_id_], dst);
        store_by_id<T, T><<<blocks(N), 256, 0, stream_>>>(N, u_[cur_u_], id_[cur_id_], dst + 3 * (size_t)N);
    }
    tild_status restore_state(const T* src, int64_t step) {
        const int N = cfg_->n_beads;
        invalidate_graph();
        cur_pos_ = cur_u_ = cur_id_ = 0;
        load_positions<T, T><<<blocks(N), 256, 0, stream_>>>(N, src, (T)cfg_->L, (T)(1.0 / cfg_->L), pos_[0], id_[0], err_ptr());
        if (zero_z()) return TILD_EDEVICE;
        load_by_id<T, T><<<blocks(N), 256, 0, stream_>>>(N, src + 3 * (size_t)N, id_[0], u_[0]);
        TILD_CUDA(cudaGetLastError());
        tild_status st;
        if ((st = enqueue_sort()) || (st = respread())) return st;
        set_counter<<<1, 1, 0, stream_>>>(counters_, (unsigned long long)step);
        TILD_CUDA(cudaGetLastError());
        host_step_ = step;
        steps_since_sort_ = 0;
        return TILD_OK;
    }

    // A binned snapshot of the current positions, what the force VJP reads:
    // positions in slot order, slot tags, neighbour slots (with beads of more
    // than two bonds, their lists as well) and tile starts. The VJP reads it in
    // place. The fields a step computed from those positions (D w, grad_
    // fields 0..2, and the xy-transformed density Zxy) follow it.
    static size_t snap_part(size_t b) { return (b + 255) / 256 * 256; }
    static constexpr int kSnapParts = 5;
    void snapshot_parts(const void* (&ptr)[kSnapParts], size_t (&bytes)[kSnapParts]) const {
        const size_t N = cfg_->n_beads;
        const void* p[kSnapParts] = {pos_[cur_pos_], id_[cur_id_], nbr_, tile_start_, ext_slots_};
        const size_t b[kSnapParts] = {3 * N * sizeof(T), N * sizeof(int), N * sizeof(int2), (n_tiles_ + 1) * sizeof(int),
                                      n_ext_ * sizeof(int)};
        for (int k = 0; k < kSnapParts; ++k) {
            ptr[k] = p[k];
            bytes[k] = b[k];
        }
    }
    size_t snapshot_bytes() const {
        const void* p[kSnapParts];
        size_t b[kSnapParts], total = 0;
        snapshot_parts(p, b);
        for (int k = 0; k < kSnapParts; ++k) total += snap_part(b[k]);
        return total;
    }
    size_t field_snapshot_bytes() const { return snap_part(3 * M_ * sizeof(V)) + snap_part(M_ * sizeof(V)); }
    // the bead state into s and the fields into f (either may be null), one launch
    tild_status snapshot(unsigned char* s, unsigned char* f) {
        CopyList c = {};
        int n = 0;
        size_t most = 0;
        cudaError_t ce = cudaSuccess;
        auto add = [&](const void* src, void* dst, size_t bytes) {
            if (bytes == 0) return;
            if (((uintptr_t)src | (uintptr_t)dst) & 15) {  // a caller's allocator may align to less
                ce = cudaMemcpyAsync(dst, src, bytes, cudaMemcpyDeviceToDevice, stream_);
                return;
            }
            c.src[n] = src;
            c.dst[n] = dst;
            c.bytes[n++] = bytes;
            most = std::max(most, bytes);
        };
        if (s) {
            const void* p[kSnapParts];
            size_t b[kSnapParts];
            snapshot_parts(p, b);
            for (int k = 0; k < kSnapParts; ++k) {
                add(p[k], s, b[k]);
                s += snap_part(b[k]);
            }
        }
        if (f) {
            add(grad_, f, 3 * M_ * sizeof(V));
            add(Zxy_, f + snap_part(3 * M_ * sizeof(V)), M_ * sizeof(V));
        }
        TILD_CUDA(ce);
        const unsigned grid = (unsigned)std::min<size_t>(304, (most / 16 + 1023) / 1024 + 1);
        if (n) launch(copy_list, dim3(grid, n), 256, 0, c);
        TILD_CUDA(cudaGetLastError());
        return TILD_OK;
    }
    // the context's bead buffers with the snapshot's positions and topology
    BeadBuffers<T> snapshot_buffers(const unsigned char* s) const {
        const void* p[kSnapParts];
        size_t b[kSnapParts];
        snapshot_parts(p, b);
        const unsigned char* at[kSnapParts];
        for (int k = 0; k < kSnapParts; ++k) {
            at[k] = s;
            s += snap_part(b[k]);
        }
        BeadBuffers<T> bf = bead_buffers();
        bf.px = (const T*)at[0];
        bf.py = bf.px + cfg_->n_beads;
        bf.pz = bf.py + cfg_->n_beads;
        bf.id = (const int*)at[1];
        bf.nbr = (const int2*)at[2];
        bf.tile_start = (const int*)at[3];
        bf.ext = n_ext_ ? (const int*)at[4] : nullptr;
        return bf;
    }

    // Reverse-mode derivatives of L(r^K, v^K) through K steps of the context's
    // scheme with the noise held fixed, checkpoints every C steps; the
    // recursion is that of the scheme's update form (scheme_coeffs; the
    // kernels adjoint_init and adjoint_step). Leaves the context at step K.
    tild_status trajectory_vjp(int64_t K, int C, const void* rbar, const void* vbar, int dtype, int where, void* r0,
                               void* v0, double* dtheta) override {
        tild_status st;
        if ((st = vjp_prepare())) return st;
        const size_t N = cfg_->n_beads, n3 = 3 * N, sb = 6 * N;  // one state: sb values of T
        if (C > K) C = K > 0 ? (int)K : 1;  // no snapshot beyond the trajectory
        const int64_t n_ckpt = K / C + 1;
        const size_t bsnap = snapshot_bytes(), snap = bsnap + field_snapshot_bytes();
        const size_t head = snap_part(sizeof(T) * (sb * ((size_t)n_ckpt + 1) + 2 * n3));
        const size_t need = head + snap * (size_t)C + sizeof(double) * 3 * n3;
        if ((st = device_buffer(&traj_, traj_bytes_, need))) return st;
        T* ckpt = (T*)traj_;                        // [n_ckpt][sb] by id
        T* fin = ckpt + sb * n_ckpt;                // [sb]
        T* lam = fin + sb;                          // [n3]
        T* jt = lam + n3;                           // [n3]
        unsigned char* seg = (unsigned char*)traj_ + head;  // [C] binned snapshots + fields (256-byte aligned)
        double* rb = (double*)(seg + snap * (size_t)C);
        double* ub = rb + n3;  // dL/dv^K on entry, then the adjoint of u
        double* vout = ub + n3;
        double* acc = sums();
        const SchemeCoeffs q = scheme_coeffs(*cfg_);
        const int64_t step0 = host_step_;
        // forward with checkpoints
        store_state(ckpt);
        for (int64_t s = 0; s < K; ++s) {
            if ((st = step(1))) return st;
            if ((s + 1) % C == 0) store_state(ckpt + sb * ((s + 1) / C));
        }
        store_state(fin);
        // adjoint vectors
        const void* src = rbar;
        if ((st = stage_in(&src, rbar, n3, dtype, where))) return st;
        if (dtype == TILD_DTYPE_F32)
            convert_copy<float, double><<<blocks(n3), 256, 0, stream_>>>(n3, (const float*)src, rb);
        else
            convert_copy<double, double><<<blocks(n3), 256, 0, stream_>>>(n3, (const double*)src, rb);
        if (vbar) {
            src = vbar;
            if ((st = stage_in(&src, vbar, n3, dtype, where))) return st;
            if (dtype == TILD_DTYPE_F32)
                convert_copy<float, double><<<blocks(n3), 256, 0, stream_>>>(n3, (const float*)src, ub);
            else
                convert_copy<double, double><<<blocks(n3), 256, 0, stream_>>>(n3, (const double*)src, ub);
        } else {
            TILD_CUDA(cudaMemsetAsync(ub, 0, n3 * sizeof(double), stream_));
        }
        TILD_CUDA(cudaMemsetAsync(acc, 0, 3 * sizeof(double), stream_));
        adjoint_init<T><<<blocks(n3), 256, 0, stream_>>>(n3, ub, lam, q.vu, q.vf, q.wf, K == 0 ? 1 : 0);
        TILD_CUDA(cudaGetLastError());
        for (int64_t s0 = ((K - 1) / C) * C; K > 0 && s0 >= 0; s0 -= C) {
            const int64_t s1 = std::min<int64_t>(s0 + C, K);
            if ((st = restore_state(ckpt + sb * (s0 / C), step0 + s0))) return st;
            for (int64_t j = s0; j < s1; ++j) {
                if ((st = step(1))) return st;
                // step j started from r^j: its fields belong to state j (snapshot j - 1 - s0);
                // the last state of the segment stays in the context
                unsigned char* fields = j > s0 ? seg + snap * (size_t)(j - 1 - s0) + bsnap : nullptr;
                unsigned char* beads = j + 1 < s1 ? seg + snap * (size_t)(j - s0) : nullptr;
                if ((fields || beads) && (st = snapshot(beads, fields))) return st;
            }
            for (int64_t j = s1 - 1; j >= s0; --j) {
                // the VJP at r^{j+1}: the context's own state (with a field pass
                // of its own) or the snapshot, read in place
                const unsigned char* at = seg + snap * (size_t)(j - s0);
                const V* fields = (const V*)(at + bsnap);
                if (j + 1 == s1)
                    st = vjp_core(lam, jt, acc, bead_buffers());
                else
                    st = vjp_core(lam, jt, acc, snapshot_buffers(at), fields,
                                  (const V*)(at + bsnap + snap_part(3 * M_ * sizeof(V))));
                if (st) return st;
                launch(adjoint_step<T>, blocks(n3), 256, 0, n3, jt, rb, ub, lam, q.sd, q.sh, q.su, q.sf, q.wf,
                                                                  j == 0 ? 1 : 0);
                TILD_CUDA(cudaGetLastError());
            }
        }
        // the force at r^0; dL/dv^0 = wu ub
        if ((st = restore_state(ckpt, step0)) || (st = vjp_core(lam, jt, acc, bead_buffers()))) return st;
        add_into<T><<<blocks(n3), 256, 0, stream_>>>(n3, rb, jt, rb);
        scale_copy<double><<<blocks(n3), 256, 0, stream_>>>(n3, ub, q.wu, vout);
        TILD_CUDA(cudaGetLastError());
        if ((st = restore_state(fin, step0 + K))) return st;
        if ((st = stage_out_double(rb, n3, r0, dtype, where)) || (st = stage_out_double(vout, n3, v0, dtype, where)))
            return st;
        if ((st = finish())) return st;
        if (dtheta) theta_from_sums(host_sums(), dtheta);
        return TILD_OK;
    }

    // Device FP64 array -> caller buffer (dtype, host or device).
    tild_status stage_out_double(const double* src, size_t count, void* out, int dtype, int where) {
        tild_status st;
        void* dst = out;
        if (where == TILD_HOST) {
            if ((st = ensure_stage(count * dtype_size(dtype)))) return st;
            dst = stage_;
        }
        if (dtype == TILD_DTYPE_F32)
            convert_copy<double, float><<<blocks(count), 256, 0, stream_>>>(count, src, (float*)dst);
        else
            convert_copy<double, double><<<blocks(count), 256, 0, stream_>>>(count, src, (double*)dst);
        TILD_CUDA(cudaGetLastError());
        if (where == TILD_HOST) {
            TILD_CUDA(cudaMemcpyAsync(out, stage_, count * dtype_size(dtype), cudaMemcpyDeviceToHost, stream_));
            TILD_CUDA(cudaStreamSynchronize(stream_));
        }
        return TILD_OK;
    }

    tild_status get_positions(void* out, int dtype, int where) override {
        return out_by_id(pos_[cur_pos_], out, dtype, where);
    }

    tild_status get_velocities(void* out, int dtype, int where) override {
        tild_status st;
        if ((st = enqueue_fields(0, nullptr, nullptr))) return st;
        const size_t n3 = (size_t)3 * cfg_->n_beads;
        const bool direct = device_native(dtype, where);
        if (!direct && (st = ensure_aux(n3 * sizeof(T)))) return st;
        BeadBuffers<T> bf = bead_buffers();
        bf.v_out = direct ? (T*)out : (T*)aux_;
        if ((st = launch_bead(kModeForce, bf))) return st;
        if (!direct && (st = stage_out_vec((T*)aux_, n3, out, dtype, where))) return st;
        return finish();
    }

    tild_status get_density(void* out, int dtype, int where) override {
        const double scale = 1.0 / FixedPoint<T>::scale / (volume() / (double)M_);
        const size_t count = (size_t)cfg_->n_species * M_;
        tild_status st;
        void* dst = out;
        if (where == TILD_HOST) {
            if ((st = ensure_aux(count * 8))) return st;
            dst = aux_;
        }
        const float2 pair = make_float2((float)scale, (float)(scale - (double)(float)scale));
        const unsigned grid = (unsigned)((count + 1023) / 1024);
        if (dtype == TILD_DTYPE_F32)
            density_out<float><<<grid, 256, 0, stream_>>>(count, rho_fx_, scale, pair, (float*)dst);
        else
            density_out<double><<<grid, 256, 0, stream_>>>(count, rho_fx_, scale, scale, (double*)dst);
        TILD_CUDA(cudaGetLastError());
        if (where == TILD_HOST)
            TILD_CUDA(cudaMemcpyAsync(out, dst, count * dtype_size(dtype), cudaMemcpyDeviceToHost, stream_));
        TILD_CUDA(cudaStreamSynchronize(stream_));
        return TILD_OK;
    }

    tild_status get_spectrum(void* out, int dtype, int where) override {
        tild_status st;
        if ((st = device_buffer(&spec_, spec_bytes_, NP_ * M_ * sizeof(V)))) return st;
        if ((st = enqueue_fields(0, nullptr, spec_))) return st;
        if ((st = stage_out_vec((T*)spec_, 2 * NP_ * M_, out, dtype, where))) return st;
        TILD_CUDA(cudaStreamSynchronize(stream_));
        return TILD_OK;
    }

    tild_status get_field_gradient(void* out, int dtype, int where) override {
        tild_status st;
        if ((st = enqueue_fields(0, nullptr, nullptr, kInvGrad))) return st;
        const int D = cfg_->dim;
        for (int q = 0; q < NP_; ++q) {
            char* o = (char*)out + (size_t)q * 2 * D * M_ * dtype_size(dtype);
            if ((st = stage_out_vec((T*)(grad_ + 4 * q * M_), 2 * D * M_, o, dtype, where))) return st;
            if (where == TILD_HOST) TILD_CUDA(cudaStreamSynchronize(stream_));  // the staging buffer is reused
        }
        TILD_CUDA(cudaStreamSynchronize(stream_));
        return TILD_OK;
    }

    int64_t host_step() const override { return host_step_; }
    // blocks of the z pass (energy partials): twice as many column tiles with two species pairs
    size_t z_blocks() const {
        if (use_lines()) return (size_t)line_last_grid().x * line_last_grid().y;
        return generic_ ? n_z_blocks_ : NP_ == 2 ? (size_t)(n_ / zpass_cols2(n_)) * (n_ / 2 + 1) : n_z_blocks_;
    }

    // blob: magic, n_beads, sizeof(T), step, seed | pos[N][3] | u[N][3] (by id, T)
    size_t state_bytes() const override { return 5 * sizeof(uint64_t) + 6 * (size_t)cfg_->n_beads * sizeof(T); }

    // blob: 5 uint64 (magic, beads, sizeof(T), step, seed), then positions
    // and carried velocities by bead id ([2][N][3] T); in host or device memory
    tild_status get_state(void* blob, int where) override {
        const size_t N = cfg_->n_beads;
        uint64_t h[5] = {kStateMagic, N, sizeof(T), (uint64_t)host_step_, cfg_->seed};
        tild_status st;
        T* d;
        if (where == TILD_DEVICE) {
            TILD_CUDA(cudaMemcpyAsync(blob, h, sizeof(h), cudaMemcpyHostToDevice, stream_));
            d = (T*)((char*)blob + sizeof(h));
        } else {
            std::memcpy(blob, h, sizeof(h));
            if ((st = ensure_aux(6 * N * sizeof(T)))) return st;
            d = (T*)aux_;
        }
        store_by_id<T, T><<<blocks(N), 256, 0, stream_>>>((int)N, pos_[cur_pos_], id_[cur_id_], d);
        store_by_id<T, T><<<blocks(N), 256, 0, stream_>>>((int)N, u_[cur_u_], id_[cur_id_], d + 3 * N);
        TILD_CUDA(cudaGetLastError());
        if (where != TILD_DEVICE)
            TILD_CUDA(cudaMemcpyAsync((char*)blob + sizeof(h), d, 6 * N * sizeof(T), cudaMemcpyDeviceToHost, stream_));
        TILD_CUDA(cudaStreamSynchronize(stream_));
        return TILD_OK;
    }

    tild_status set_state(const void* blob, int where) override {
        const size_t N = cfg_->n_beads;
        uint64_t h[5];
        if (where == TILD_DEVICE) {
            TILD_CUDA(cudaMemcpyAsync(h, blob, sizeof(h), cudaMemcpyDeviceToHost, stream_));
            TILD_CUDA(cudaStreamSynchronize(stream_));
        } else {
            std::memcpy(h, blob, sizeof(h));
        }
        if (h[0] != kStateMagic || h[1] != N || h[2] != sizeof(T) || h[4] != cfg_->seed) {
            err = "state blob does not match this context (beads, precision or seed)";
            return TILD_EINVAL;
        }
        invalidate_graph();
        tild_status st;
        const T* d;
        if (where == TILD_DEVICE) {
            d = (const T*)((const char*)blob + sizeof(h));
        } else {
            if ((st = ensure_aux(6 * N * sizeof(T)))) return st;
            TILD_CUDA(cudaMemcpyAsync(aux_, (const char*)blob + sizeof(h), 6 * N * sizeof(T), cudaMemcpyHostToDevice,
                                      stream_));
            d = (const T*)aux_;
        }
        cur_pos_ = cur_u_ = cur_id_ = 0;
        load_positions<T, T><<<blocks(N), 256, 0, stream_>>>((int)N, d, (T)cfg_->L, (T)(1.0 / cfg_->L), pos_[0], id_[0], err_ptr());
        if ((st = zero_z())) return st;
        load_by_id<T, T><<<blocks(N), 256, 0, stream_>>>((int)N, d + 3 * N, id_[0], u_[0]);
        TILD_CUDA(cudaGetLastError());
        if ((st = enqueue_sort())) return st;
        if ((st = respread())) return st;
        host_step_ = (int64_t)h[3];
        const unsigned long long dstep = h[3];
        TILD_CUDA(cudaMemcpyAsync(counters_, &dstep, sizeof(dstep), cudaMemcpyHostToDevice, stream_));
        TILD_CUDA(cudaStreamSynchronize(stream_));
        steps_since_sort_ = 0;
        have_pos_ = have_vel_ = true;
        return TILD_OK;
    }

    tild_status profile(int nsteps, double* ms) override {
        tild_status st;
        cudaEvent_t ev[6];
        for (auto& e : ev) TILD_CUDA(cudaEventCreate(&e));
        double acc[5] = {0, 0, 0, 0, 0};
        const int K = cfg_->sort_every;
        for (int s = 0; s < nsteps; ++s) {
            TILD_CUDA(cudaEventRecord(ev[0], stream_));
            if (steps_since_sort_ >= K) {
                if ((st = enqueue_sort())) return st;
            }
            TILD_CUDA(cudaEventRecord(ev[1], stream_));
            if ((st = enqueue_forward(true))) return st;
            TILD_CUDA(cudaEventRecord(ev[2], stream_));
            if ((st = enqueue_zpass(nullptr, nullptr, analytic()))) return st;
            TILD_CUDA(cudaEventRecord(ev[3], stream_));
            if ((st = enqueue_inverse(force_fields()))) return st;
            TILD_CUDA(cudaEventRecord(ev[4], stream_));
            BeadBuffers<T> bf = bead_buffers();
            bf.qx = pos_[1 - cur_pos_];
            bf.qy = bf.qx + cfg_->n_beads;
            bf.qz = bf.qy + cfg_->n_beads;
            if ((st = launch_bead(kModeStep, bf))) return st;
            TILD_CUDA(cudaEventRecord(ev[5], stream_));
            cur_pos_ = 1 - cur_pos_;
            ++steps_since_sort_;
            ++host_step_;
            TILD_CUDA(cudaEventSynchronize(ev[5]));
            float t;
            TILD_CUDA(cudaEventElapsedTime(&t, ev[1], ev[2])); acc[0] += t;
            TILD_CUDA(cudaEventElapsedTime(&t, ev[2], ev[3])); acc[1] += t;
            TILD_CUDA(cudaEventElapsedTime(&t, ev[3], ev[4])); acc[2] += t;
            TILD_CUDA(cudaEventElapsedTime(&t, ev[4], ev[5])); acc[3] += t;
            TILD_CUDA(cudaEventElapsedTime(&t, ev[0], ev[1])); acc[4] += t;
        }
        for (auto& e : ev) cudaEventDestroy(e);
        for (int k = 0; k < 5; ++k) ms[k] = nsteps > 0 ? acc[k] / nsteps : 0.0;
        return check_err();
    }

    int64_t sort_launches() const { return n_fine_ <= kScanOne ? 4 : 7; }  // of one re-binning
    int64_t launches(int64_t n) const override {
        const int D = cfg_->dim;
        const int64_t per_step = generic_ ? (use_lines() ? 2 * D : (1 + D) + 1 + (int64_t)NP_ * D + 1) : (use_planes() ? 2 : 4) + 2;
        const int64_t per_sort = sort_launches();
        const int K = cfg_->sort_every;
        int64_t since = steps_since_sort_, sorts = 0;
        for (int64_t s = 0; s < n; ++s) {
            if (since >= K) {
                ++sorts;
                since = 0;
            }
            ++since;
        }
        return n * per_step + sorts * per_sort;
    }

    bool has_positions() const override { return have_pos_; }
    bool has_velocities() const override { return have_vel_; }

    tild_status save_velocities() override {
        const size_t N = cfg_->n_beads;
        if (!vsave_) TILD_CUDA(dev_malloc((void**)&vsave_, 3 * N * sizeof(T)));
        tild_status st;
        if ((st = enqueue_fields(0, nullptr, nullptr))) return st;
        BeadBuffers<T> bf = bead_buffers();
        bf.v_out = vsave_;
        if ((st = launch_bead(kModeForce, bf))) return st;
        TILD_CUDA(cudaStreamSynchronize(stream_));
        return TILD_OK;
    }

    tild_status restore_velocities() override {
        invalidate_graph();
        tild_status st;
        if ((st = enqueue_fields(0, nullptr, nullptr))) return st;
        BeadBuffers<T> bf = bead_buffers();
        bf.v_in = vsave_;
        if ((st = launch_bead(kModeSetVel, bf))) return st;
        TILD_CUDA(cudaStreamSynchronize(stream_));
        return TILD_OK;
    }

    void params_changed() override { invalidate_graph(); }

    // Launch shapes: plane threads (128, 256 or 512 where the grid allows)
    // and the z pass's column tile (the default or the alternative).
    void launch_shapes(int* plane_threads, int* z_cols, int* z_default, int* z_alt) const override {
        *plane_threads = plane_nt_;
        const int cdef = dispatch_cols(false), calt = dispatch_cols(true);
        *z_cols = zalt_ ? calt : cdef;
        if (z_default) *z_default = cdef;
        if (z_alt) *z_alt = calt;
    }
    tild_status set_launch_shapes(int plane_threads, int z_cols) override {
        if (generic_) {
            err = "launch shapes: the any-size kernels have none";
            return TILD_EUNSUPPORTED;
        }
        bool ok = false;
        dispatch_n([&](auto nn) {
            constexpr int NN = decltype(nn)::value;
            ok = plane_threads == 512 || (plane_fits_ && ((plane_threads == 256 && plane_nt_ok(NN, 256)) ||
                                                         (plane_threads == 128 && plane_nt_ok(NN, 128)) ||
                                                         (plane_threads == 1024 && plane_nt_ok(NN, 1024)) ||
                                                         (plane_threads == 0 && split_ok(NN))));
            return TILD_OK;
        });
        const int cdef = dispatch_cols(false), calt = dispatch_cols(true);
        if (!ok || (z_cols != cdef && z_cols != calt)) {
            err = "launch shapes: plane threads must be 512 (or 128/256/1024 where the grid allows, or 0 for the row "
                  "and column passes) and the z columns the default or the alternative tile";
            return TILD_EINVAL;
        }
        invalidate_graph();
        plane_nt_ = plane_threads;
        zalt_ = z_cols != cdef;
        return TILD_OK;
    }
    int dispatch_cols(bool alt) const {
        int c = 0;
        const_cast<Engine*>(this)->dispatch_n([&](auto nn) {
            c = alt ? zpass_cols_alt(decltype(nn)::value) : zpass_cols(decltype(nn)::value);
            return TILD_OK;
        });
        return c;
    }

   private:
    T* vsave_ = nullptr;
    HostConfig* cfg_ = nullptr;
    // species pairs of the grids (1: up to two species, 2: three or four) and
    // species slots of the bead kernels (2 NP)
    int NP_ = 1, NS_ = 2;
    // launch shapes of the step (tild_set_launch_shapes, tild_autotune):
    // threads of the xy plane CTAs and the z pass's column tile
    int plane_nt_ = 512;
    bool zalt_ = false;
    // any-size / 2D kernels: grid planes along z, the two factors of n
    bool generic_ = false;
    int nz_ = 0, gn1_ = 1, gn2_ = 1;
    size_t partials_bytes_ = 0;
    // explicit topology (by bead id): species, first two neighbours, and the
    // extra neighbour lists of beads with more than two bonds (ids and slots)
    unsigned char* sp_of_id_ = nullptr;
    int2* adj_ = nullptr;
    int* ext_ids_ = nullptr;
    int* ext_slots_ = nullptr;
    size_t n_ext_ = 0;
    void* io_ = nullptr;  // per-bead vectors in the other layout
    size_t io_bytes_ = 0;
    size_t spec_bytes_ = 0;
    std::unordered_map<void*, size_t> live_;  // blocks from the caller's allocator
    int device_ = 0;
    int n_ = 0, tiles_ = 0, P_ = 2, C_ = 16, CZ_ = 8;
    size_t M_ = 0;
    bool plane_fits_ = true;
    cudaStream_t own_stream_ = nullptr, stream_ = nullptr;
    // grids
    unsigned long long* rho_fx_ = nullptr;
    V* Zxy_ = nullptr;
    V* H_ = nullptr;
    V* grad_ = nullptr;
    V* tw_ = nullptr;
    T* kernel1d_ = nullptr;
    double kernel_a_ = -1.0, kernel_ae_ = -1.0;
    V* spec_ = nullptr;
    // [0] noise step counter, [1] error flags, [4 ..] sums of one call (FP64);
    // words_: their host copy, one transfer per synchronising call (pageable: a
    // pinned one cost a context 350 us of its 570 to create and free, and saved
    // nothing: an empty synchronising call takes 13.5 us either way)
    static constexpr int kWords = 16;
    unsigned long long* counters_ = nullptr;
    unsigned long long words_[kWords] = {};
    double* partials_ = nullptr;
    size_t n_partials_ = 0, n_z_blocks_ = 0;
    // beads
    T* pos_[2] = {nullptr, nullptr};
    T* u_[2] = {nullptr, nullptr};
    int* id_[2] = {nullptr, nullptr};
    int2* nbr_ = nullptr;
    int* slot_of_id_ = nullptr;
    int* keys_ = nullptr;   // re-binning: fine bin of each bead
    int* ranks_ = nullptr;  // and its rank in the bin
    int* counts_ = nullptr;  // [n_fine_] bead counts of the fine bins
    size_t n_fine_ = 0;
    // Bins up to which one block scans them, in rounds of 4,096 (24^3: one launch
    // of 3 us for four of 14 us in all; at 128^3, 65,537 bins, the 17 rounds take
    // 36 us and the three scan kernels stay)
    static constexpr size_t kScanOne = 16384;
    int* tile_start_ = nullptr;
    int n_tiles_ = 0;
    int* fine_start_ = nullptr;  // [n_fine_] exclusive scan of counts_
    int* block_sums_ = nullptr;
    int scan_blocks_ = 0;
    int cur_pos_ = 0, cur_u_ = 0, cur_id_ = 0;
    int steps_since_sort_ = 0;
    int64_t host_step_ = 0;
    bool have_pos_ = false, have_vel_ = false;
    // staging
    void* aux_ = nullptr;
    size_t aux_bytes_ = 0;
    void* traj_ = nullptr;     // trajectory derivatives: checkpoints and adjoint vectors
    size_t traj_bytes_ = 0;
    void* vjp_fx_ = nullptr;   // force VJP: fixed-point spread of lam
    size_t vjp_fx_bytes_ = 0;
    void* stage_ = nullptr;
    size_t stage_bytes_ = 0;
    // graph cache
    cudaGraphExec_t graph_ = nullptr;
    int graph_key_ = -1;

    unsigned int* err_ptr() const { return reinterpret_cast<unsigned int*>(counters_ + 1) + 1; }

    static unsigned blocks(size_t count) { return (unsigned)((count + 255) / 256); }
    static size_t dtype_size(int dtype) { return dtype == TILD_DTYPE_F32 ? 4 : 8; }

    // the planes (and the rows) of the xy passes, with twiddles
    size_t plane_smem() const { return ((size_t)n_ + (size_t)n_ * row_pitch(n_)) * sizeof(V); }
    // two dimensions: z stays 0
    tild_status zero_z() {
        if (cfg_->dim == 2)
            TILD_CUDA(cudaMemsetAsync(pos_[0] + 2 * (size_t)cfg_->n_beads, 0, (size_t)cfg_->n_beads * sizeof(T), stream_));
        return TILD_OK;
    }
    double volume() const { return cfg_->dim == 2 ? cfg_->L * cfg_->L : cfg_->L * cfg_->L * cfg_->L; }
    // lines per CTA of the any-size axis transform: about 96 KB of shared memory
    int gaxis_lines() const {
        const long c = ((long)(96 * 1024 / sizeof(V)) - n_) / (2L * (n_ + 1));
        return (int)std::max(1L, std::min(32L, c));
    }
    size_t gaxis_smem() const { return ((size_t)n_ + 2 * (size_t)gaxis_lines() * (n_ + 1)) * sizeof(V); }
    // blocks of the bead kernel (its partial sums)
    size_t bead_blocks() const {
        return per_bead() ? ((size_t)cfg_->n_beads + bead_threads() - 1) / bead_threads() : (size_t)n_tiles_;
    }
    tild_status ensure_partials() {
        const size_t need = 5 * std::max(bead_blocks(), z_blocks()) * sizeof(double);
        return device_buffer(&partials_, partials_bytes_, need);
    }
    // Line passes of the any-size grids: lines per CTA (2^lg) so that the launch
    // has about two CTAs per SM, not below `lo` (short rows of memory); shared
    // memory within kLineSmem.
    static constexpr int kLineSmem = 200 * 1024;
    bool line_big() const { return std::max(gn1_, gn2_) > 16; }
    size_t line_smem(int half) const { return ((size_t)2 * n_ + (size_t)half * (line_big() ? 2 : 1)) * sizeof(V); }
    // lines: of the launch at 2^lg per CTA; f(lg) = CTAs
    template <class F> int line_lg(int hi, int lo, int per_line, F&& ctas) const {
        int lg = hi;
        while (lg > lo && (ctas(lg) < 304 || line_smem(per_line << lg) > (size_t)kLineSmem / 2)) --lg;
        return lg;
    }
    LineArgs<T> line_args(int lg, int per_line) const {
        return LineArgs<T>{n_, nz_, gn1_, gn2_, lg, line_big() ? per_line << lg : 0, tw_, two_pi_L()};
    }
    static int div_up(int a, int b) { return (a + b - 1) / b; }
    int line_rows_lg(int fields) const {
        return line_lg(4, 0, n_ | 1, [&](int lg) { return div_up(nz_ * n_, 1 << lg) * fields; });
    }
    int line_last_lg() const {  // 4 NP lines per column
        const int c = NP_ == 2 ? 3 : 2;
        return line_lg(c + 3, c, n_, [&](int lg) { return div_up(n_, 1 << (lg - c)) * (cfg_->dim == 3 ? n_ / 2 + 1 : 1); });
    }
    dim3 line_last_grid() const {
        const int lg = line_last_lg() - (NP_ == 2 ? 3 : 2);
        return dim3(div_up(n_, 1 << lg), cfg_->dim == 3 ? n_ / 2 + 1 : 1);
    }
    // Whether the line passes serve the grid. The lines of one column have to fit
    // the last pass (2D grids of a few thousand points per edge do not). Long 2D
    // lines in FP32 leave it few CTAs per SM, each with a direct DFT of a large
    // factor: above 600 points per edge it pays where it runs in two waves at
    // most, the second at least half full. Step, us, whole-axis passes / lines,
    // one pair: 509 1262/606, 600 266/124, 641 1638/1983, 719 6654/1488, 800
    // 382/305, 900 354/303, 1000 523/582, 1021 3973/4965, 1500 1090/1667, 2000
    // 1860/3423; two pairs: 600 389/233, 641 2444/3008, 800 648/751, 1000 941/1218.
    // FP64 gains at every size that fits (1200 7568/6149, 1021 75.9/51.5 ms).
    bool use_lines() const {
        if (!generic_ || line_smem((NP_ == 2 ? 8 : 4) * n_) > (size_t)kLineSmem) return false;
        if (sizeof(T) == 8 || cfg_->dim == 3 || n_ <= 600) return true;
        const size_t per_cta = line_smem(n_ << line_last_lg()) + 1024;
        const unsigned resident = 152u * (unsigned)(228 * 1024 / per_cta), ctas = line_last_grid().x;
        return ctas <= resident || (ctas <= 2 * resident && 2 * (ctas - resident) >= resident);
    }
    tild_status line_forward(bool zero_after) {
        const int lg = line_rows_lg(NP_);
        launch(line_x_forward<T>, dim3(div_up(nz_ * n_, 1 << lg), NP_), 128, line_smem((n_ | 1) << lg), 
            line_args(lg, n_ | 1), rho_fx_, Zxy_, density_scale(), zero_after ? 1 : 0, zero_after ? counters_ : nullptr);
        if (cfg_->dim == 3) {
            const int ly = line_lg(4, 2, n_, [&](int l) { return div_up(n_, 1 << l) * nz_ * NP_; });
            launch(line_y<T, -1>, dim3(div_up(n_, 1 << ly), nz_, NP_), 128, line_smem(n_ << ly), line_args(ly, n_), Zxy_);
        }
        TILD_CUDA(cudaGetLastError());
        return TILD_OK;
    }
    tild_status line_spectral(double* partials) {
        const int lg = line_last_lg();
        const SpectralParams<T> sp = spectral_params();
        const LineArgs<T> a = line_args(lg, n_);
        const size_t sm = line_smem(n_ << lg);
        if (cfg_->dim == 3) {
            if (NP_ == 2) launch(line_last<T, 2, 3>, line_last_grid(), 128, sm, a, Zxy_, H_, sp, partials);
            else launch(line_last<T, 1, 3>, line_last_grid(), 128, sm, a, Zxy_, H_, sp, partials);
        } else {
            if (NP_ == 2) launch(line_last<T, 2, 2>, line_last_grid(), 128, sm, a, Zxy_, H_, sp, partials);
            else launch(line_last<T, 1, 2>, line_last_grid(), 128, sm, a, Zxy_, H_, sp, partials);
        }
        TILD_CUDA(cudaGetLastError());
        return TILD_OK;
    }
    tild_status line_inverse() {
        const int D = cfg_->dim;
        if (D == 3) {
            const int ly = line_lg(5, 3, n_, [&](int l) { return div_up(n_, 1 << (l - 1)) * nz_ * NP_; });
            launch(line_y<T, +1>, dim3(div_up(n_, 1 << (ly - 1)), nz_, 2 * NP_), 128, line_smem(n_ << ly), line_args(ly, n_), H_);
        }
        const int lg = line_rows_lg(D * NP_);
        launch(line_x_inverse<T>, dim3(div_up(nz_ * n_, 1 << lg), D * NP_), 128, line_smem((n_ | 1) << lg), 
            line_args(lg, n_ | 1), H_, grad_, D);
        TILD_CUDA(cudaGetLastError());
        return TILD_OK;
    }
    // the any-size transforms of `count` contiguous fields at f along every axis
    tild_status generic_fft(V* f, int count, int dir) {
        const int C = gaxis_lines();
        const unsigned tiles = (unsigned)((M_ / n_ + C - 1) / C);
        for (int axis = 0; axis < cfg_->dim; ++axis) {
            if (dir < 0)
                generic_axis_fft<T, -1><<<dim3(tiles, count), 256, gaxis_smem(), stream_>>>(f, n_, nz_, axis, C, gn1_, gn2_, tw_);
            else
                generic_axis_fft<T, +1><<<dim3(tiles, count), 256, gaxis_smem(), stream_>>>(f, n_, nz_, axis, C, gn1_, gn2_, tw_);
        }
        TILD_CUDA(cudaGetLastError());
        return TILD_OK;
    }
    size_t rows_smem() const { return ((size_t)n_ + (size_t)16 * row_pitch(n_)) * sizeof(V); }
    size_t ycol_smem() const { return ((size_t)n_ + 2 * (size_t)n_ * C_) * sizeof(V); }
    size_t zpass_smem() const { return ((size_t)n_ + 4 * (size_t)n_ * CZ_) * sizeof(V); }
    bool analytic() const { return cfg_->force_method == TILD_FORCE_ANALYTIC; }
    bool c_el_on() const { return cfg_->bjerrum > 0 && (cfg_->q_a != 0 || cfg_->q_b != 0); }
    // E_el = (4 pi l_B) dV^2 / (2 V) sum_k exp(-a_e^2 k^2)/k^2 |q_A rho^_A + q_B rho^_B|^2
    double e_elec_from(double s4) const {
        const double V = cfg_->L * cfg_->L * cfg_->L, dV = V / (double)M_;
        return c_el_on() ? 4.0 * 3.14159265358979323846 * cfg_->bjerrum * dV * dV / (2.0 * V) * s4 : 0.0;
    }
    size_t bead_smem() const { return bead_smem(analytic(), NS_); }
    // width and first stencil offset of the bead kernels' shared patch
    void patch_geometry(int* w, int* lo) const {
        switch (P_) {
            case 2: *w = Patch<2>::W; *lo = Patch<2>::lo; break;
            case 3: *w = Patch<3>::W; *lo = Patch<3>::lo; break;
            case 4: *w = Patch<4>::W; *lo = Patch<4>::lo; break;
            default: *w = Patch<5>::W; *lo = Patch<5>::lo; break;
        }
    }
    template <int P> static size_t bead_smem_p(bool an, int ns) {
        if (ns == 4) return an ? bead_smem_bytes<P, T, true, 4>() : bead_smem_bytes<P, T, false, 4>();
        return an ? bead_smem_bytes<P, T, true>() : bead_smem_bytes<P, T>();
    }
    size_t bead_smem(bool an, int ns) const {
        switch (P_) {
            case 2: return bead_smem_p<2>(an, ns);
            case 3: return bead_smem_p<3>(an, ns);
            case 4: return bead_smem_p<4>(an, ns);
            default: return bead_smem_p<5>(an, ns);
        }
    }

    // Device memory through the caller's allocator when one was given.
    cudaError_t dev_malloc(void** p, size_t bytes) {
        const tild_allocator& a = cfg_->allocator;
        if (!a.alloc) return cudaMalloc(p, bytes);
        *p = bytes ? a.alloc(bytes, a.user) : nullptr;
        if (bytes && !*p) return cudaErrorMemoryAllocation;
        if (*p) live_[*p] = bytes;
        return cudaSuccess;
    }
    void dev_free(void* p) {
        if (!p) return;
        const tild_allocator& a = cfg_->allocator;
        if (!a.alloc) {
            cudaFree(p);
            return;
        }
        auto it = live_.find(p);
        const size_t bytes = it == live_.end() ? 0 : it->second;
        if (it != live_.end()) live_.erase(it);
        if (a.free) a.free(p, bytes, a.user);
    }

    // Density, spectrum and field grids for np species pairs.
    tild_status alloc_grids(int np) {
        if (stream_) TILD_CUDA(cudaStreamSynchronize(stream_));
        void* old[] = {rho_fx_, Zxy_, H_, grad_};
        for (void* q : old) dev_free(q);
        rho_fx_ = nullptr;
        Zxy_ = H_ = grad_ = nullptr;
        NP_ = np;
        NS_ = 2 * np;
        TILD_CUDA(dev_malloc((void**)&rho_fx_, 2 * np * M_ * sizeof(unsigned long long)));
        TILD_CUDA(dev_malloc((void**)&Zxy_, np * M_ * sizeof(V)));
        TILD_CUDA(dev_malloc((void**)&H_, 3 * np * M_ * sizeof(V)));
        TILD_CUDA(dev_malloc((void**)&grad_, 4 * np * M_ * sizeof(V)));  // per pair: 3 gradients + (optional) potentials
        TILD_CUDA(cudaMemset(rho_fx_, 0, 2 * np * M_ * sizeof(unsigned long long)));
        return TILD_OK;
    }

    // Device copies of the explicit species and bonds (none: the chains'
    // pattern and linear bonds).
    tild_status upload_topology() {
        TILD_CUDA(cudaStreamSynchronize(stream_));
        dev_free(sp_of_id_);
        dev_free(adj_);
        dev_free(ext_ids_);
        dev_free(ext_slots_);
        sp_of_id_ = nullptr;
        adj_ = nullptr;
        ext_ids_ = ext_slots_ = nullptr;
        n_ext_ = 0;
        const size_t N = cfg_->n_beads;
        if (N == 0) return TILD_OK;
        if (!cfg_->species_of_bead.empty()) {
            TILD_CUDA(dev_malloc((void**)&sp_of_id_, N));
            TILD_CUDA(cudaMemcpy(sp_of_id_, cfg_->species_of_bead.data(), N, cudaMemcpyHostToDevice));
        }
        if (cfg_->explicit_bonds) {
            // adjacency by id, neighbours in increasing id order
            std::vector<std::vector<int>> nb(N);
            const std::vector<int>& bp = cfg_->bond_pairs;
            for (size_t k = 0; k + 1 < bp.size(); k += 2) {
                nb[bp[k]].push_back(bp[k + 1]);
                nb[bp[k + 1]].push_back(bp[k]);
            }
            std::vector<int2> adj(N, make_int2(-1, -1));
            std::vector<int> ext;
            for (size_t b = 0; b < N; ++b) {
                std::vector<int>& v = nb[b];
                std::sort(v.begin(), v.end());
                if (v.size() >= 1) adj[b].x = v[0];
                if (v.size() == 2) adj[b].y = v[1];
                if (v.size() > 2) {
                    adj[b].y = -2 - (int)ext.size();
                    ext.push_back((int)v.size() - 1);
                    ext.insert(ext.end(), v.begin() + 1, v.end());
                }
            }
            TILD_CUDA(dev_malloc((void**)&adj_, N * sizeof(int2)));
            TILD_CUDA(cudaMemcpy(adj_, adj.data(), N * sizeof(int2), cudaMemcpyHostToDevice));
            if (!ext.empty()) {
                n_ext_ = ext.size();
                TILD_CUDA(dev_malloc((void**)&ext_ids_, n_ext_ * sizeof(int)));
                TILD_CUDA(dev_malloc((void**)&ext_slots_, n_ext_ * sizeof(int)));
                TILD_CUDA(cudaMemcpy(ext_ids_, ext.data(), n_ext_ * sizeof(int), cudaMemcpyHostToDevice));
            }
        }
        return TILD_OK;
    }

    void free_beads() {
        for (int k = 0; k < 2; ++k) {
            dev_free(pos_[k]);
            dev_free(u_[k]);
            dev_free(id_[k]);
            pos_[k] = u_[k] = nullptr;
            id_[k] = nullptr;
        }
        dev_free(nbr_);
        dev_free(slot_of_id_);
        dev_free(keys_);
        dev_free(ranks_);
        dev_free(vsave_);
        vsave_ = nullptr;
        nbr_ = nullptr;
        slot_of_id_ = keys_ = ranks_ = nullptr;
    }

    void release() {
        invalidate_graph();
        if (stream_) cudaStreamSynchronize(stream_);  // no kernel may still use a block handed back
        free_beads();
        void* ptrs[] = {rho_fx_, Zxy_, H_, grad_, tw_, kernel1d_, spec_, counters_, partials_, counts_,
                        tile_start_, fine_start_, block_sums_, aux_, stage_, traj_, vjp_fx_,
                        sp_of_id_, adj_, ext_ids_, ext_slots_, io_};
        for (void* p : ptrs) dev_free(p);
        rho_fx_ = nullptr;
        if (own_stream_) cudaStreamDestroy(own_stream_);
        own_stream_ = nullptr;
    }

    void invalidate_graph() {
        if (graph_) cudaGraphExecDestroy(graph_);
        graph_ = nullptr;
        graph_key_ = -1;
    }

    double* sums() const { return reinterpret_cast<double*>(counters_ + 4); }
    const double* host_sums() const { return reinterpret_cast<const double*>(words_ + 4); }
    // sums()[k] of the K-component block sums in partials_
    tild_status reduce_partials(size_t n_blocks, int K, double* out) {
        sum_partials<<<K, (unsigned)std::min<size_t>(1024, (n_blocks + 31) / 32 * 32), 0, stream_>>>(partials_, (int)n_blocks, K, out);
        TILD_CUDA(cudaGetLastError());
        return TILD_OK;
    }
    bool has_bonds() const {
        if (cfg_->explicit_bonds) return !cfg_->bond_pairs.empty();
        for (int k = 0; k < cfg_->topo.n_types; ++k)
            if (cfg_->topo.N[k] > 1) return true;
        return false;
    }
    // The sums of an observable again in FP64 (an FP32 context's that left the
    // range of floats), not scaled: s[0 .. 4] the spectral ones, s[5] of the
    // bonds and, with velocities and forces, s[6 .. 9].
    tild_status sums_fp64(bool spectral, bool forces, double* s) {
        const size_t N = cfg_->n_beads;
        tild_status st;
        if ((st = device_buffer(&partials_, partials_bytes_, 5 * (size_t)blocks(std::max(N, M_)) * sizeof(double)))) return st;
        T *v = nullptr, *f = nullptr;
        if (forces) {  // (the fields at the beads are those of the call)
            if ((st = ensure_aux(6 * N * sizeof(T)))) return st;
            BeadBuffers<T> bf = bead_buffers();
            bf.f_out = f = (T*)aux_;
            bf.v_out = v = f + 3 * N;
            if ((st = launch_bead(kModeForce, bf))) return st;
        }
        bead_sums64<T><<<blocks(N), 256, 0, stream_>>>(bead_params(), bead_buffers(), v, f, partials_);
        TILD_CUDA(cudaGetLastError());
        if ((st = reduce_partials(blocks(N), 5, sums() + 5))) return st;
        if (spectral) {
            if ((st = device_buffer(&spec_, spec_bytes_, NP_ * M_ * sizeof(V)))) return st;
            if ((st = enqueue_forward(false, true)) || (st = enqueue_zpass(nullptr, spec_))) return st;
            const SpectralParams<T> sp = spectral_params();
            const int el = c_el_on() ? 1 : 0;
            if (NP_ == 2)
                spectral_sums64<T, 2><<<blocks(M_), 256, 0, stream_>>>(spec_, n_, nz_, sp, el, partials_);
            else
                spectral_sums64<T, 1><<<blocks(M_), 256, 0, stream_>>>(spec_, n_, nz_, sp, el, partials_);
            TILD_CUDA(cudaGetLastError());
            if ((st = reduce_partials(blocks(M_), 5, sums()))) return st;
        }
        if ((st = finish())) return st;
        std::copy(host_sums() + (spectral ? 0 : 5), host_sums() + (forces ? 10 : 6), s + (spectral ? 0 : 5));
        return TILD_OK;
    }
    // whether the caller's array can be a kernel's own input or output
    static bool device_native(int dtype, int where) {
        return where == TILD_DEVICE && dtype == (sizeof(T) == 4 ? TILD_DTYPE_F32 : TILD_DTYPE_F64);
    }

    // Wait for the context's stream, with the error flags and the call's sums
    // read back behind its work.
    tild_status finish() {
        TILD_CUDA(cudaMemcpyAsync(words_, counters_, kWords * sizeof(unsigned long long), cudaMemcpyDeviceToHost, stream_));
        TILD_CUDA(cudaStreamSynchronize(stream_));
        return check_flags(reinterpret_cast<const unsigned int*>(words_)[3]);
    }
    tild_status check_err() {
        unsigned int h = 0;
        TILD_CUDA(cudaMemcpy(&h, err_ptr(), sizeof(h), cudaMemcpyDeviceToHost));
        return check_flags(h);
    }
    tild_status check_flags(unsigned int h) {
        if (h & kErrBounds) {
            TILD_CUDA(cudaMemset(err_ptr(), 0, sizeof(unsigned int)));
            err = "a bounds check of the debug build failed on the device (the access was skipped)";
            return TILD_EDEVICE;
        }
        if (h & kErrNonFinite) {
            TILD_CUDA(cudaMemset(err_ptr(), 0, sizeof(unsigned int)));
            err = "non-finite position or force detected on the device";
            return TILD_ENAN;
        }
        return TILD_OK;
    }

    tild_status ensure_aux(size_t bytes) {
        if (aux_bytes_ >= bytes) return TILD_OK;
        TILD_CUDA(cudaStreamSynchronize(stream_));
        dev_free(aux_);
        aux_ = nullptr;
        aux_bytes_ = 0;
        TILD_CUDA(dev_malloc(&aux_, bytes));
        aux_bytes_ = bytes;
        return TILD_OK;
    }

    tild_status ensure_stage(size_t bytes) {
        if (stage_bytes_ >= bytes) return TILD_OK;
        TILD_CUDA(cudaStreamSynchronize(stream_));
        dev_free(stage_);
        stage_ = nullptr;
        stage_bytes_ = 0;
        TILD_CUDA(dev_malloc(&stage_, bytes));
        stage_bytes_ = bytes;
        return TILD_OK;
    }

    // Host input -> device staging buffer (same dtype); device input as is.
    tild_status stage_in(const void** dev, const void* src, size_t count, int dtype, int where) {
        if (where == TILD_DEVICE) {
            *dev = src;
            return TILD_OK;
        }
        tild_status st;
        if ((st = ensure_stage(count * dtype_size(dtype)))) return st;
        TILD_CUDA(cudaMemcpyAsync(stage_, src, count * dtype_size(dtype), cudaMemcpyHostToDevice, stream_));
        *dev = stage_;
        return TILD_OK;
    }

    // Device array of T -> caller buffer (dtype, host or device).
    tild_status stage_out_vec(const T* src, size_t count, void* out, int dtype, int where) {
        tild_status st;
        void* dst = out;
        if (where == TILD_HOST) {
            if ((st = ensure_stage(count * dtype_size(dtype)))) return st;
            dst = stage_;
        }
        if (dtype == TILD_DTYPE_F32)
            convert_copy<T, float><<<blocks(count), 256, 0, stream_>>>(count, src, (float*)dst);
        else
            convert_copy<T, double><<<blocks(count), 256, 0, stream_>>>(count, src, (double*)dst);
        TILD_CUDA(cudaGetLastError());
        if (where == TILD_HOST)
            TILD_CUDA(cudaMemcpyAsync(out, dst, count * dtype_size(dtype), cudaMemcpyDeviceToHost, stream_));
        return TILD_OK;
    }

    tild_status out_by_id(const T* src, void* out, int dtype, int where) {
        const int N = cfg_->n_beads;
        tild_status st;
        void* dst = out;
        if (where == TILD_HOST) {
            if ((st = ensure_stage((size_t)3 * N * dtype_size(dtype)))) return st;
            dst = stage_;
        }
        if (dtype == TILD_DTYPE_F32)
            store_by_id<T, float><<<blocks(N), 256, 0, stream_>>>(N, src, id_[cur_id_], (float*)dst);
        else
            store_by_id<T, double><<<blocks(N), 256, 0, stream_>>>(N, src, id_[cur_id_], (double*)dst);
        TILD_CUDA(cudaGetLastError());
        if (where == TILD_HOST)
            TILD_CUDA(cudaMemcpyAsync(out, dst, (size_t)3 * N * dtype_size(dtype), cudaMemcpyDeviceToHost, stream_));
        TILD_CUDA(cudaStreamSynchronize(stream_));
        return TILD_OK;
    }

    // ---------------------------------------------------------- kernels

    // Launch of a step's kernel, overlapping its start with the end of the
    // kernel before it where overlap() says so. The overlap hides the launch
    // latency, but the blocks that start early are placed among those still
    // running, unevenly, which costs more than it saves where a kernel fills
    // the chip or the FP64 unit. FP32 only; us per step without / with, as
    // graph replay and as single launches:
    //   24^3, 4,060 beads      15.5 / 13.0    24.2 / 14.4
    //   48^3, 22,000           20.1 / 19.1    30.4 / 20.7
    //   64^3, 200,000          30.1 / 34.8    39.4 / 36.4
    //   80^3, 400,000          47.3 / 50.2    56.6 / 51.8
    //   128^3, 1.6M           153.3 / 162.2  162.4 / 163.1
    //   65^2, 5,000            18.6 / 16.2    29.4 / 18.6
    //   45^3, 54,000           34.5 / 37.0    50.2 / 40.2
    //   FP64 32^3, 20,000      58.1 / 75.9    67.7 / 77.6
    bool overlap() const {
        if (sizeof(T) == 8 || M_ > 80 * 80 * 80) return false;
        if (M_ <= (generic_ ? 32 * 32 * 32 : 48 * 48 * 48)) return true;
        cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
        return cudaStreamIsCapturing(stream_, &cap) == cudaSuccess && cap == cudaStreamCaptureStatusNone;
    }
    template <class... KA, class... A>
    void launch(void (*k)(KA...), dim3 grid, unsigned threads, size_t smem, A&&... a) {
        launch_on(stream_, overlap(), k, grid, threads, smem, std::forward<A>(a)...);
    }
    template <class... KA, class... A>
    static void launch_on(cudaStream_t stream_, bool overlap, void (*k)(KA...), dim3 grid, unsigned threads, size_t smem, A&&... a) {
        cudaLaunchConfig_t c = {};
        c.gridDim = grid;
        c.blockDim = dim3(threads);
        c.dynamicSmemBytes = smem;
        c.stream = stream_;
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        at[0].val.programmaticStreamSerializationAllowed = 1;
        c.attrs = at;
        c.numAttrs = overlap ? 1 : 0;
        cudaLaunchKernelEx(&c, k, static_cast<KA>(a)...);  // (errors: cudaGetLastError at the call site)
    }

    template <int NN> tild_status attrs_n() {
        if (plane_fits_) {
            if constexpr (plane_fits(NN, sizeof(V))) {
                TILD_CUDA(cudaFuncSetAttribute(xy_forward_plane<T, NN>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)plane_smem()));
                TILD_CUDA(cudaFuncSetAttribute(xy_inverse_plane<T, NN>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)plane_smem()));
                if constexpr (plane_nt_ok(NN, 256)) {
                    TILD_CUDA(cudaFuncSetAttribute(xy_forward_plane<T, NN, 256>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)plane_smem()));
                    TILD_CUDA(cudaFuncSetAttribute(xy_inverse_plane<T, NN, 256>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)plane_smem()));
                }
                if constexpr (plane_nt_ok(NN, 128)) {
                    TILD_CUDA(cudaFuncSetAttribute(xy_forward_plane<T, NN, 128>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)plane_smem()));
                    TILD_CUDA(cudaFuncSetAttribute(xy_inverse_plane<T, NN, 128>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)plane_smem()));
                }
                if constexpr (plane_nt_ok(NN, 1024)) {
                    TILD_CUDA(cudaFuncSetAttribute(xy_forward_plane<T, NN, 1024>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)plane_smem()));
                    TILD_CUDA(cudaFuncSetAttribute(xy_inverse_plane<T, NN, 1024>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)plane_smem()));
                }
                TILD_CUDA(cudaFuncSetAttribute(xy_forward_cplx<T, NN>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)plane_smem()));
                TILD_CUDA(cudaFuncSetAttribute(z_vjp<T, NN, vjp_cols(NN)>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)vjp_smem()));
            }
        }
        if (!plane_fits_ || split_ok(NN)) {
            TILD_CUDA(cudaFuncSetAttribute(x_forward_rows<T, NN, 16>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)rows_smem()));
            TILD_CUDA(cudaFuncSetAttribute(x_inverse_rows<T, NN, 16>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)rows_smem()));
            TILD_CUDA(cudaFuncSetAttribute(y_columns<T, NN, 128 / sizeof(V), -1>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ycol_smem()));
            TILD_CUDA(cudaFuncSetAttribute(y_columns<T, NN, 128 / sizeof(V), +1>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ycol_smem()));
        }
        constexpr int CC = zpass_cols(NN);
        constexpr int C2 = zpass_cols2(NN);
        TILD_CUDA(cudaFuncSetAttribute(z_spectral_pairs<T, NN, C2>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)zpass2_smem()));
        TILD_CUDA(cudaFuncSetAttribute(z_spectral_pairs<T, NN, C2, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)zpass2_smem()));
        TILD_CUDA(cudaFuncSetAttribute(z_spectrum<T, NN, CC>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)zpass_smem()));
        tild_status st = with_z<NN>([&](auto cc, auto g, auto el, auto e) -> tild_status {
            TILD_CUDA(cudaFuncSetAttribute(z_spectral<T, NN, decltype(cc)::value, decltype(g)::value != 0, decltype(el)::value != 0, decltype(e)::value>,
                                           cudaFuncAttributeMaxDynamicSharedMemorySize, (int)zpass_smem_cols(decltype(cc)::value)));
            return TILD_OK;
        }, true);
        if (st) return st;
        return TILD_OK;
    }

    template <int P> tild_status attrs_p() {
        if constexpr (sizeof(T) == 4) {
            TILD_CUDA(cudaFuncSetAttribute(vjp_spread_tiled<P>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)vjp_spread_smem<P>()));
            TILD_CUDA(cudaFuncSetAttribute(vjp_beads_tiled<P>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)vjp_beads_smem<P>()));
        }
        const int s4 = (int)bead_smem(false, 4), sa4 = (int)bead_smem(true, 4);
        TILD_CUDA(cudaFuncSetAttribute(bead_kernel<P, kModeSpread, T, false, 4>, cudaFuncAttributeMaxDynamicSharedMemorySize, s4));
        if constexpr (sizeof(T) == 4) {  // (FP64: per_bead)
            TILD_CUDA(cudaFuncSetAttribute(bead_kernel<P, kModeForce, T, false, 4>, cudaFuncAttributeMaxDynamicSharedMemorySize, s4));
            TILD_CUDA(cudaFuncSetAttribute(bead_kernel<P, kModeSetVel, T, false, 4>, cudaFuncAttributeMaxDynamicSharedMemorySize, s4));
            TILD_CUDA(cudaFuncSetAttribute(bead_kernel<P, kModeStep, T, false, 4>, cudaFuncAttributeMaxDynamicSharedMemorySize, s4));
        }
        TILD_CUDA(cudaFuncSetAttribute(bead_kernel<P, kModeForce, T, true, 4>, cudaFuncAttributeMaxDynamicSharedMemorySize, sa4));
        TILD_CUDA(cudaFuncSetAttribute(bead_kernel<P, kModeSetVel, T, true, 4>, cudaFuncAttributeMaxDynamicSharedMemorySize, sa4));
        TILD_CUDA(cudaFuncSetAttribute(bead_kernel<P, kModeStep, T, true, 4>, cudaFuncAttributeMaxDynamicSharedMemorySize, sa4));
        const int s = (int)bead_smem(false, 2);
        TILD_CUDA(cudaFuncSetAttribute(bead_kernel<P, kModeSpread, T>, cudaFuncAttributeMaxDynamicSharedMemorySize, s));
        if constexpr (sizeof(T) == 4) {  // (FP64: per_bead)
            TILD_CUDA(cudaFuncSetAttribute(bead_kernel<P, kModeForce, T>, cudaFuncAttributeMaxDynamicSharedMemorySize, s));
            TILD_CUDA(cudaFuncSetAttribute(bead_kernel<P, kModeSetVel, T>, cudaFuncAttributeMaxDynamicSharedMemorySize, s));
            TILD_CUDA(cudaFuncSetAttribute(bead_kernel<P, kModeStep, T>, cudaFuncAttributeMaxDynamicSharedMemorySize, s));
        }
        const int sa = (int)bead_smem(true, 2);
        TILD_CUDA(cudaFuncSetAttribute(bead_kernel<P, kModeForce, T, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, sa));
        TILD_CUDA(cudaFuncSetAttribute(bead_kernel<P, kModeSetVel, T, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, sa));
        TILD_CUDA(cudaFuncSetAttribute(bead_kernel<P, kModeStep, T, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, sa));
        return TILD_OK;
    }

    tild_status set_kernel_attributes() {
        tild_status st = dispatch_n([&](auto nn) { return this->template attrs_n<decltype(nn)::value>(); });
        if (st) return st;
        return dispatch_p([&](auto pp) { return this->template attrs_p<decltype(pp)::value>(); });
    }

    template <int V_> struct ic { static constexpr int value = V_; };


    template <class F> tild_status dispatch_n(F&& f) {
        switch (n_) {
            case 8: return f(ic<8>{});
            case 16: return f(ic<16>{});
            case 32: return f(ic<32>{});
            case 64: return f(ic<64>{});
            case 128: return f(ic<128>{});
            case 24: return f(ic<24>{});
            case 40: return f(ic<40>{});
            case 48: return f(ic<48>{});
            case 80: return f(ic<80>{});
            case 256: return dispatch_256(f);
        }
        err = "unsupported grid size";
        return TILD_EUNSUPPORTED;
    }
    template <class F> tild_status dispatch_256(F&& f) {
        if constexpr (sizeof(T) == 4) return f(ic<256>{});
        err = "FP64 grids are limited to 128^3";
        return TILD_EUNSUPPORTED;
    }
    template <class F> tild_status dispatch_p(F&& f) {
        switch (P_) {
            case 2: return f(ic<2>{});
            case 3: return f(ic<3>{});
            case 4: return f(ic<4>{});
            case 5: return f(ic<5>{});
        }
        err = "unsupported pmeorder";
        return TILD_EUNSUPPORTED;
    }

    T density_scale() const {
        const double dV = volume() / (double)M_;
        return (T)(1.0 / FixedPoint<T>::scale / dV);
    }

    template <int NN> tild_status forward_n(bool zero_after) {
        if (use_planes()) {
            if constexpr (plane_fits(NN, sizeof(V))) {
                with_nt<NN>([&](auto nt) {
                    constexpr int NT = decltype(nt)::value;
                    launch(xy_forward_plane<T, NN, NT>, dim3(NN, NP_), NT, plane_smem(), 
                        rho_fx_, Zxy_, tw_, density_scale(), zero_after ? 1 : 0, zero_after ? counters_ : nullptr);
                });
            }
        } else {
            constexpr int CC = 128 / sizeof(V);
            if constexpr (NN >= 16 && NN >= CC) {
                launch(x_forward_rows<T, NN, 16>, dim3((unsigned)((size_t)NN * NN / 16), NP_), 256, rows_smem(), 
                    rho_fx_, Zxy_, tw_, density_scale(), zero_after ? 1 : 0, zero_after ? counters_ : nullptr);
                launch(y_columns<T, NN, CC, -1>, dim3(NN / CC, NN, NP_), 256, ycol_smem(), Zxy_, tw_, two_pi_L(), 0);
            }
        }
        TILD_CUDA(cudaGetLastError());
        return TILD_OK;
    }
    // whole: any-size grids by whole-axis passes (natural order; the spectrum read-out)
    tild_status enqueue_forward(bool zero_after, bool whole = false) {
        if (use_lines() && !whole) return line_forward(zero_after);
        if (generic_) {
            generic_load_density<T><<<blocks((size_t)NP_ * M_), 256, 0, stream_>>>(
                M_, NP_, rho_fx_, Zxy_, density_scale(), zero_after ? 1 : 0, zero_after ? counters_ : nullptr);
            TILD_CUDA(cudaGetLastError());
            return generic_fft(Zxy_, NP_, -1);
        }
        return dispatch_n([&](auto nn) { return this->template forward_n<decltype(nn)::value>(zero_after); });
    }

    // z-pass column tile: 128 bytes of complex values, or the largest power of
    // two dividing n when that is smaller
    // force-VJP z pass column tile: the z pass's up to 64^3 (shared memory
    // 8 n C elements), half of it above, at least 2
    static constexpr int vjp_cols(int n) {
        return n <= 64 ? zpass_cols(n) : (zpass_cols(n) / 2 < 2 ? 2 : zpass_cols(n) / 2);
    }
    size_t vjp_smem() const { return ((size_t)n_ + 8 * (size_t)n_ * vjp_cols(n_)) * sizeof(V); }

    // At 256^3 half of that: 16 columns take 133 KB (one CTA per SM) and 177
    // registers, 8 columns 67 KB and two CTAs per SM (z pass 148 against 114 us).
    static constexpr int zpass_cols(int n) {
        if (n == 256) return (int)(64 / sizeof(V));
        int c = (int)(128 / sizeof(V));
        while (c > 1 && (n % c) != 0) c /= 2;
        return c < n ? c : n;
    }
    // two species pairs: half the columns (twice the buffers), at least 2
    static constexpr int zpass_cols2(int n) { return zpass_cols(n) / 2 < 2 ? 2 : zpass_cols(n) / 2; }
    // the alternative column tile of the z pass (launch shapes): half the
    // default, at least 2
    static constexpr int zpass_cols_alt(int n) { return zpass_cols2(n); }
    size_t zpass_smem_cols(int c) const { return ((size_t)n_ + 4 * (size_t)n_ * c) * sizeof(V); }
    // plane kernels with NT threads: 512, or for small planes (several per SM) 256
    // or 128 with at most 32 complex values of a line transform's stage per thread.
    // 1024 threads where every thread has a stage-B unit (n N1 >= 1024).
    static constexpr bool plane_nt_ok(int n, int nt) {
        if (nt == 512) return true;
        const int n1 = n == 8 ? 8 : n == 16 ? 4 : (n == 48 || n == 80 || n == 128 || n == 256) ? 16 : 8;
        const int n2 = n / n1;
        if (nt == 1024) return sizeof(V) == 8 && n * n1 >= 1024 && n <= 128;
        if (n > 80 || (nt != 128 && nt != 256)) return false;
        return (n * n1 + nt - 1) / nt * n2 <= 32;
    }
    // The row and column passes (x rows, then y columns, through global
    // memory) serve grids whose planes do not fit shared memory, and are the
    // launch shape plane_threads = 0 for those that do.
    static constexpr bool split_ok(int n) {
        return n >= 16 && n % (int)(128 / sizeof(V)) == 0;  // whole column tiles (and rows in blocks of 16)
    }
    bool use_planes() const { return plane_fits_ && plane_nt_ != 0; }
    // runtime forms for the batch's groups
    static bool plane_nt_allowed(int n, int nt) { return plane_nt_ok(n, nt) && plane_fits(n, sizeof(V)); }
    static int zpass_cols_n(int n) { return zpass_cols(n); }
    static int zpass_cols_alt_n(int n) { return zpass_cols_alt(n); }
    template <int NN, class F> void with_nt(F&& f) {
        if constexpr (plane_nt_ok(NN, 1024))
            if (plane_nt_ == 1024) return f(ic<1024>{});
        if constexpr (plane_nt_ok(NN, 128))
            if (plane_nt_ == 128) return f(ic<128>{});
        if constexpr (plane_nt_ok(NN, 256))
            if (plane_nt_ == 256) return f(ic<256>{});
        return f(ic<512>{});
    }
    size_t zpass2_smem() const { return ((size_t)n_ + 8 * (size_t)n_ * zpass_cols2(n_)) * sizeof(V); }

    T two_pi_L() const { return (T)(2.0 * 3.14159265358979323846 / cfg_->L); }

    // a power of two near x for the scaled sums of Wide<T> (1 in FP64)
    static T power_of_two(double x) {
        if (sizeof(T) == 8 || !(x > 0) || !std::isfinite(x)) return T(1);
        return (T)std::ldexp(1.0, std::max(-100, std::min(100, std::ilogb(x))));
    }

    SpectralParams<T> spectral_params() const {
        const double V = volume();
        const double rho0 = cfg_->n_beads / V;
        SpectralParams<T> sp;
        sp.two_pi_over_L = (T)(2.0 * 3.14159265358979323846 / cfg_->L);
        sp.eAA = (T)(cfg_->kappa / rho0 / (double)M_);
        sp.eBB = sp.eAA;
        sp.eAB = (T)((cfg_->chi + cfg_->kappa) / rho0 / (double)M_);
        for (int K = 0; K < 4; ++K)
            for (int K2 = 0; K2 < 4; ++K2) {
                const double chi = K == K2 ? 0.0 : cfg_->chi_mat[K][K2];
                sp.eps4[K][K2] = (T)((chi + cfg_->kappa) / rho0 / (double)M_);
                sp.chi4[K][K2] = (T)chi;
            }
        sp.e_rho = power_of_two(V / (double)M_);
        sp.kernel1d = kernel1d_;
        const bool charged = c_el_on();
        sp.el_scale = charged ? (T)(4.0 * 3.14159265358979323846 * cfg_->bjerrum / (double)M_) : T(0);
        sp.qA = (T)cfg_->q_a;
        sp.qB = (T)cfg_->q_b;
        sp.kernel1d_el = kernel1d_ + n_;
        return sp;
    }

    template <int NN> tild_status zpass_n(double* partials, V* spec_out, bool g_only, int want_e) {
        constexpr int CC = zpass_cols(NN);
        const SpectralParams<T> sp = spectral_params();
        const bool el = c_el_on();
        if (spec_out) {
            // the spectra alone: each pair's forward z transform (no coupling)
            for (int q = 0; q < NP_; ++q)
                z_spectrum<T, NN, CC><<<dim3(NN / CC, NN), 256, zpass_smem(), stream_>>>(Zxy_ + q * M_, tw_, spec_out + q * M_);
            TILD_CUDA(cudaGetLastError());
            return TILD_OK;
        }
        if (NP_ == 2) {
            constexpr int C2 = zpass_cols2(NN);
            const dim3 grid2(NN / C2, NN / 2 + 1);
            if (g_only)
                launch(z_spectral_pairs<T, NN, C2, true>, grid2, 256, zpass2_smem(), Zxy_, H_, tw_, sp, partials);
            else
                launch(z_spectral_pairs<T, NN, C2>, grid2, 256, zpass2_smem(), Zxy_, H_, tw_, sp, partials);
            TILD_CUDA(cudaGetLastError());
            return TILD_OK;
        }
        return with_z<NN>([&](auto cc, auto g, auto e_l, auto e) -> tild_status {
            constexpr int CZ = decltype(cc)::value;
            launch(z_spectral<T, NN, CZ, decltype(g)::value != 0, decltype(e_l)::value != 0, decltype(e)::value>, dim3(NN / CZ, NN / 2 + 1), 256, zpass_smem_cols(CZ), Zxy_, H_, tw_, sp, partials);
            TILD_CUDA(cudaGetLastError());
            return TILD_OK;
        }, false, g_only, el, want_e);
    }
    // f(columns, G alone, charges, energies) for the z pass to launch, or for
    // every instantiation when `all`. The alternative column tile serves the
    // plain step only (launch shapes).
    template <int NN, class F>
    tild_status with_z(F&& f, bool all, bool g_only = false, bool el = false, int want_e = 0) {
        constexpr int CC = zpass_cols(NN), CA = zpass_cols_alt(NN);
        tild_status st = TILD_OK;
        bool found = false;
        auto pick = [&](auto cc, auto g, auto e_l, auto e) {
            const bool alt = decltype(cc)::value != CC;
            const bool plain = !g_only && !el && want_e == 0;
            const bool take = g_only == (decltype(g)::value != 0) && el == (decltype(e_l)::value != 0) &&
                              want_e == decltype(e)::value && alt == (CA != CC && zalt_ && plain);
            if (!st && (all || take)) st = f(cc, g, e_l, e);
            found = found || take;
        };
        if constexpr (CA != CC) pick(ic<CA>{}, ic<0>{}, ic<0>{}, ic<0>{});
        pick(ic<CC>{}, ic<0>{}, ic<0>{}, ic<0>{});
        pick(ic<CC>{}, ic<1>{}, ic<0>{}, ic<0>{});
        pick(ic<CC>{}, ic<0>{}, ic<1>{}, ic<0>{});
        pick(ic<CC>{}, ic<1>{}, ic<1>{}, ic<0>{});
        pick(ic<CC>{}, ic<0>{}, ic<0>{}, ic<1>{});
        pick(ic<CC>{}, ic<1>{}, ic<0>{}, ic<1>{});
        pick(ic<CC>{}, ic<0>{}, ic<1>{}, ic<1>{});
        pick(ic<CC>{}, ic<1>{}, ic<1>{}, ic<1>{});
        pick(ic<CC>{}, ic<1>{}, ic<0>{}, ic<2>{});
        pick(ic<CC>{}, ic<1>{}, ic<1>{}, ic<2>{});
        if (!st && !all && !found) {
            err = "no z pass for these options";
            return TILD_EUNSUPPORTED;
        }
        return st;
    }
    // separable Gaussian tables exp(-s^2 k_m^2), k_m = 2 pi m / L, m in FFT
    // index order: the pair kernel's (s = a) and, with charges, the charge
    // smearing's (s = a_e); rebuilt when the parameter changes
    tild_status refresh_tables() {
        auto refresh = [&](double s, double& cached, T* dst) -> tild_status {
            if (cached == s) return TILD_OK;
            std::vector<T> e(n_);
            for (int i = 0; i < n_; ++i) {
                const double m = 2 * i < n_ ? i : i - n_;  // odd n: frequencies -(n-1)/2 .. (n-1)/2
                const double k = 2.0 * 3.14159265358979323846 * m / cfg_->L;
                e[i] = (T)std::exp(-s * s * k * k);
            }
            TILD_CUDA(cudaStreamSynchronize(stream_));  // no z pass may still read the old table
            TILD_CUDA(cudaMemcpy(dst, e.data(), n_ * sizeof(T), cudaMemcpyHostToDevice));
            cached = s;
            return TILD_OK;
        };
        tild_status st;
        if ((st = refresh(cfg_->a, kernel_a_, kernel1d_))) return st;
        if (c_el_on() && (st = refresh(cfg_->charge_smear, kernel_ae_, kernel1d_ + n_))) return st;
        return TILD_OK;
    }
    tild_status enqueue_zpass(double* partials, V* spec_out, bool g_only = false, int want_e = 1) {
        tild_status st;
        if ((st = refresh_tables())) return st;
        if (generic_) {
            if (spec_out) {  // the spectrum is complete after the forward transforms
                TILD_CUDA(cudaMemcpyAsync(spec_out, Zxy_, NP_ * M_ * sizeof(V), cudaMemcpyDeviceToDevice, stream_));
                return TILD_OK;
            }
            if (use_lines()) return line_spectral(partials);
            const SpectralParams<T> sp = spectral_params();
            if (NP_ == 2)
                generic_spectral<T, 2><<<blocks(M_), 256, 0, stream_>>>(Zxy_, grad_, n_, nz_, sp, partials);
            else
                generic_spectral<T, 1><<<blocks(M_), 256, 0, stream_>>>(Zxy_, grad_, n_, nz_, sp, partials);
            TILD_CUDA(cudaGetLastError());
            return TILD_OK;
        }
        return dispatch_n([&](auto nn) { return this->template zpass_n<decltype(nn)::value>(partials, spec_out, g_only, partials ? want_e : 0); });
    }

    // what the inverse xy pass produces
    static constexpr int kInvGrad = 0, kInvPot = 1;
    template <int NN> tild_status inverse_n(int what) {
        const unsigned nd = what == kInvGrad ? 3 : 1;
        const int d0 = what == kInvPot ? 3 : 0;
        if (use_planes()) {
            if constexpr (plane_fits(NN, sizeof(V))) {
                with_nt<NN>([&](auto nt) {
                    constexpr int NT = decltype(nt)::value;
                    launch(xy_inverse_plane<T, NN, NT>, dim3(NN, nd, NP_), NT, plane_smem(), H_, grad_, tw_, two_pi_L(), d0);
                });
            }
        } else {
            constexpr int CC = 128 / sizeof(V);
            if constexpr (NN >= 16 && NN >= CC) {
                launch(y_columns<T, NN, CC, +1>, dim3(NN / CC, NN, (what == kInvPot ? 1 : 2) * NP_), 256, ycol_smem(), 
                    H_, tw_, two_pi_L(), what == kInvPot ? 1 : 0);
                launch(x_inverse_rows<T, NN, 16>, dim3((unsigned)((size_t)NN * NN / 16), nd, NP_), 256, rows_smem(), 
                    H_, grad_, tw_, two_pi_L(), d0);
            }
        }
        TILD_CUDA(cudaGetLastError());
        return TILD_OK;
    }
    tild_status enqueue_inverse(int what) {
        if (generic_) {  // (the gradients: nothing on these grids takes the potentials)
            if (use_lines()) return line_inverse();
            tild_status st;
            for (int q = 0; q < NP_; ++q)
                if ((st = generic_fft(grad_ + 4 * q * M_, cfg_->dim, +1))) return st;
            return TILD_OK;
        }
        return dispatch_n([&](auto nn) { return this->template inverse_n<decltype(nn)::value>(what); });
    }
    // the fields the bead kernel's force needs: ik gradients or the potentials
    int force_fields() const { return analytic() ? kInvPot : kInvGrad; }

    // energy: 0, 1 (energy sums of the z pass into partials) or 2 (and their
    // |k|^2-weighted versions; potentials only)
    tild_status enqueue_fields(int energy, double* partials, V* spec_out, int what = -1) {
        if (what < 0) what = force_fields();
        tild_status st;
        if (!have_pos_) {
            err = "positions have not been set";
            return TILD_ESTATE;
        }
        if ((st = enqueue_forward(false, spec_out != nullptr))) return st;
        if (generic_ && spec_out) return enqueue_zpass(nullptr, spec_out);
        if ((st = enqueue_zpass(energy ? partials : nullptr, spec_out, what == kInvPot, energy))) return st;
        return enqueue_inverse(what);
    }

    // Constants of the integrator update (see BeadParams), from FP64.
    // The update of every scheme in one form (state: positions r and carried
    // velocity u; F = F(r); xi the step's normals):
    //   h = su u + sf F + sg xi,  r' = r + sd h + se xi,  u' = sh h + sk xi,
    // the velocity of a state v = vu u + vf F + vg xi, and u from (r, v):
    // u = wu v + wf F + wg xi.
    struct SchemeCoeffs {
        double su, sf, sg, sd, se, sh, sk, vu, vf, vg, wu, wf, wg;
        int lag;
    };
    static SchemeCoeffs scheme_coeffs(const HostConfig& c) {
        const double dt = c.dt, m = c.mass, al = c.friction, kT = c.kT;
        const double hdm = dt / (2.0 * m);
        SchemeCoeffs k{1, 2 * hdm, 0, dt, 0, 1, 0, 1, hdm, 0, 1, -hdm, 0, 0};
        if (c.scheme == kSchemeGJF) {
            // GJF: a = (1 - alpha dt/2m)/(1 + alpha dt/2m), b = 1/(1 + alpha dt/2m), beta = sigma xi
            const double den = 1.0 + al * hdm, ga = (1.0 - al * hdm) / den, gb = 1.0 / den;
            const double sb = std::sqrt(2.0 * al * kT * dt);
            k.sd = gb * dt;
            k.se = gb * dt * sb / (2.0 * m);
            k.sh = ga;
            k.sk = gb * sb / m;
        } else if (c.scheme == kSchemeEM) {
            // r' = r + (dt/alpha) F + sqrt(2 kT dt/alpha) xi; no velocity
            k.su = 0;
            k.sf = al > 0 ? dt / al : 0;
            k.sg = al > 0 ? std::sqrt(2.0 * kT * dt / al) : 0;
            k.sd = 1;
            k.sh = 0;
            k.vu = k.vf = k.wu = k.wf = 0;
        } else {
            // VV: F = F_c - alpha u + s xi^n (s = sqrt(2 alpha kT/dt)), h = u + (dt/m) F
            const double sv = std::sqrt(2.0 * al * kT / dt), inv = 1.0 / (1.0 - al * hdm);
            k.su = 1.0 - 2.0 * hdm * al;
            k.sg = 2.0 * hdm * sv;
            k.lag = 1;
            k.vu = 1.0 - hdm * al;
            k.vg = hdm * sv;
            k.wu = inv;
            k.wf = -inv * hdm;
            k.wg = -inv * hdm * sv;
        }
        return k;
    }
    static void integrator_constants(const HostConfig& c, BeadParams<T>& p) {
        const SchemeCoeffs k = scheme_coeffs(c);
        p.su = (T)k.su; p.sf = (T)k.sf; p.sg = (T)k.sg; p.sd = (T)k.sd; p.se = (T)k.se; p.sh = (T)k.sh; p.sk = (T)k.sk;
        p.vu = (T)k.vu; p.vf = (T)k.vf; p.vg = (T)k.vg; p.wu = (T)k.wu; p.wf = (T)k.wf; p.wg = (T)k.wg;
        p.noise_lag = k.lag;
    }

    BeadParams<T> bead_params() const {
        BeadParams<T> p;
        const HostConfig& c = *cfg_;
        p.n_beads = c.n_beads;
        p.n = n_;
        p.tiles = tiles_;
        p.L = (T)c.L;
        p.inv_L = (T)(1.0 / c.L);
        p.inv_dx = (T)((double)n_ / c.L);
        p.k_bond = (T)(3.0 / (c.b * c.b));
        integrator_constants(c, p);
        p.sigma_v = (T)std::sqrt(c.kT / c.mass);
        p.species = NS_;
        p.e_len = power_of_two(1.0 / c.L);
        p.e_vel = power_of_two(c.kT > 0 ? std::sqrt(c.mass / c.kT) : 1.0);
        p.seed = c.seed;
        p.topo = c.topo;
        return p;
    }

    BeadBuffers<T> bead_buffers() const {
        BeadBuffers<T> b;
        const size_t N = cfg_->n_beads;
        b.px = pos_[cur_pos_];
        b.py = b.px + N;
        b.pz = b.py + N;
        b.qx = b.qy = b.qz = nullptr;
        b.ux = u_[cur_u_];
        b.uy = b.ux + N;
        b.uz = b.uy + N;
        b.id = id_[cur_id_];
        b.nbr = nbr_;
        b.ext = ext_slots_;
        b.tile_start = tile_start_;
        b.grad = grad_;
        b.rho_fx = rho_fx_;
        b.step = counters_;
        b.err = err_ptr();
        b.f_out = nullptr;
        b.v_out = nullptr;
        b.v_in = nullptr;
        b.partials = nullptr;
        return b;
    }

    template <int P, int NS> tild_status bead_pn(int mode, const BeadBuffers<T>& bf) {
        const unsigned grid = (unsigned)tiles_ * tiles_ * tiles_;
        const BeadParams<T> p = bead_params();
        if (analytic() && mode != kModeSpread) {
            const size_t sm = bead_smem(true, NS);
            switch (mode) {
                case kModeForce: launch(bead_kernel<P, kModeForce, T, true, NS>, grid, 256, sm, p, bf); break;
                case kModeSetVel: launch(bead_kernel<P, kModeSetVel, T, true, NS>, grid, 256, sm, p, bf); break;
                default: launch(bead_kernel<P, kModeStep, T, true, NS>, grid, 256, sm, p, bf); break;
            }
        } else {
            const size_t sm = bead_smem(false, NS);
            if constexpr (sizeof(T) == 8) {  // the analytic force's spread; everything else is per_bead
                launch(bead_kernel<P, kModeSpread, T, false, NS>, grid, 256, sm, p, bf);
            } else {
                switch (mode) {
                    case kModeSpread: launch(bead_kernel<P, kModeSpread, T, false, NS>, grid, 256, sm, p, bf); break;
                    case kModeForce: launch(bead_kernel<P, kModeForce, T, false, NS>, grid, 256, sm, p, bf); break;
                    case kModeSetVel: launch(bead_kernel<P, kModeSetVel, T, false, NS>, grid, 256, sm, p, bf); break;
                    default: launch(bead_kernel<P, kModeStep, T, false, NS>, grid, 256, sm, p, bf); break;
                }
            }
        }
        TILD_CUDA(cudaGetLastError());
        return TILD_OK;
    }
    // Whether beads go through the per-bead kernel (one thread per bead, fields
    // and density in global memory) instead of the tiled one. Measured on melts
    // of 20-bead chains (us of the bead kernel in the step, tiled / per bead):
    //   FP64: bound by the FP64 unit (two operations per clock and SM), which
    //   the tiles of a small grid leave idle on most SMs; order 1, 32^3, 20,000
    //   beads 44.9 / 22.5, 64^3, 200,000 168 / 131; order 3 118 / 55, 419 / 326.
    //   FP32, order 1: up to about 48,000 beads latency decides, and a tile's
    //   patch adds barriers and a flush to the chain; beyond that the global
    //   atomics do (64^3, 200,000: 30.6 / 37.4), and at higher orders at every
    //   size (order 3, 24^3: 20.2 / 22.5). Step, tiled / per bead:
    //     8^3    2,000 beads 25.2 / 9.6   48,000 484 / 27.2
    //     16^3   2,000 10.7 / 10.4        48,000 75.9 / 14.7
    //     24^3   4,000 11.4 / 12.0        14,000 14.9 / 11.9   48,000 29.1 / 14.4
    //     32^3   20,000 13.9 / 13.3       48,000 18.3 / 16.6
    //     40^3   20,000 14.8 / 15.0       32,000 15.9 / 16.0   48,000 16.9 / 19.2
    //     48^3   22,000 18.7 / 18.7       30,000 19.3 / 20.1   48,000 20.3 / 25.9
    //     64^3   48,000 23.5 / 22.5       80^3 37.3 / 31.9     128^3 98.4 / 75.9
    //   At 40^3 and 48^3 the tiles are many and the launches overlap (above
    //   48^3 a graph's do not), so the per-bead form ends at 22,000 beads there.
    bool per_bead() const {
        if (generic_) return true;
        if (analytic()) return false;
        const bool few_tiles = M_ <= 32 * 32 * 32, graph_overlaps = M_ <= 48 * 48 * 48;
        return sizeof(T) == 8 || (P_ == 2 && cfg_->n_beads <= (few_tiles || !graph_overlaps ? 48000 : 22000));
    }
    // Threads per block: small blocks spread few beads over all SMs (FP64,
    // 32^3: 22.5 us with 32 threads, 28.7 with 128).
    int bead_threads() const { return !per_bead() ? 256 : sizeof(T) == 8 ? 32 : cfg_->n_beads <= 100000 ? 64 : 256; }
    template <int P, int D> tild_status bead_generic(int mode, const BeadBuffers<T>& bf) {
        const BeadParams<T> p = bead_params();
        const unsigned bt = (unsigned)bead_threads(), g = (unsigned)bead_blocks();
        switch (mode) {
            case kModeSpread: launch(generic_bead_kernel<P, kModeSpread, T, D>, g, bt, 0, p, bf, nz_); break;
            case kModeForce: launch(generic_bead_kernel<P, kModeForce, T, D>, g, bt, 0, p, bf, nz_); break;
            case kModeSetVel: launch(generic_bead_kernel<P, kModeSetVel, T, D>, g, bt, 0, p, bf, nz_); break;
            default: launch(generic_bead_kernel<P, kModeStep, T, D>, g, bt, 0, p, bf, nz_); break;
        }
        TILD_CUDA(cudaGetLastError());
        return TILD_OK;
    }
    template <int P> tild_status bead_p(int mode, const BeadBuffers<T>& bf) {
        if (per_bead()) return cfg_->dim == 2 ? bead_generic<P, 2>(mode, bf) : bead_generic<P, 3>(mode, bf);
        return NS_ == 4 ? bead_pn<P, 4>(mode, bf) : bead_pn<P, 2>(mode, bf);
    }
    tild_status launch_bead(int mode, const BeadBuffers<T>& bf) {
        return dispatch_p([&](auto pp) { return this->template bead_p<decltype(pp)::value>(mode, bf); });
    }

    tild_status respread() {
        TILD_CUDA(cudaMemsetAsync(rho_fx_, 0, 2 * NP_ * M_ * sizeof(unsigned long long), stream_));
        return launch_bead(kModeSpread, bead_buffers());
    }

    // NVTX range on the host thread for profilers (no cost without one attached)
    struct Range {
        explicit Range(const char* name) { nvtxRangePushA(name); }
        ~Range() { nvtxRangePop(); }
    };

    tild_status enqueue_step() {
        Range range("tild step: forward, z pass, inverse, beads");
        tild_status st;
        if ((st = enqueue_forward(true))) return st;
        if ((st = enqueue_zpass(nullptr, nullptr, analytic()))) return st;
        if ((st = enqueue_inverse(force_fields()))) return st;
        BeadBuffers<T> bf = bead_buffers();
        bf.qx = pos_[1 - cur_pos_];
        bf.qy = bf.qx + cfg_->n_beads;
        bf.qz = bf.qy + cfg_->n_beads;
        if ((st = launch_bead(kModeStep, bf))) return st;
        cur_pos_ = 1 - cur_pos_;
        ++steps_since_sort_;
        return TILD_OK;
    }

    tild_status enqueue_sort(cudaStream_t on = nullptr) {
        Range range("tild re-binning");
        cudaStream_t st = on ? on : stream_;  // the batch re-bins on its own streams
        const bool ov = !on && overlap();
        const int N = cfg_->n_beads;
        const size_t N3 = N;
        const T* p = pos_[cur_pos_];
        int pw = 0, plo = 0;
        patch_geometry(&pw, &plo);
        launch_on(st, ov, bin_count_fine<T>, blocks(N), 256, 0, N, p, p + N3, p + 2 * N3, (T)((double)n_ / cfg_->L), n_, nz_,
                  tiles_, pw, plo, cfg_->topo, sp_of_id_, id_[cur_id_], keys_, ranks_, counts_);
        if (n_fine_ <= kScanOne) {
            launch_on(st, ov, scan_one, 1, 1024, 0, counts_, fine_start_, (int)n_fine_, n_tiles_, tile_start_);
        } else {
            scan_blocks<<<scan_blocks_, 1024, 0, st>>>(counts_, fine_start_, block_sums_, (int)n_fine_);
            scan_top<<<1, 1024, 0, st>>>(block_sums_, scan_blocks_);
            scan_add<<<scan_blocks_, 1024, 0, st>>>(fine_start_, block_sums_, (int)n_fine_);
            bin_tile_start<<<blocks((size_t)n_tiles_ + 1), 256, 0, st>>>(fine_start_, n_tiles_, tile_start_);
        }
        launch_on(st, ov, bin_scatter_fine<T>, blocks(N), 256, 0, N, cfg_->topo, sp_of_id_, keys_, ranks_, counts_, fine_start_,
                  pos_[cur_pos_], pos_[1 - cur_pos_], u_[cur_u_], u_[1 - cur_u_], id_[cur_id_], id_[1 - cur_id_], slot_of_id_);
        if (adj_)
            launch_on(st, ov, bin_neighbours_explicit, blocks(N), 256, 0, N, id_[1 - cur_id_], slot_of_id_, adj_, ext_ids_,
                      ext_slots_, nbr_, counts_, (int)n_fine_);
        else
            launch_on(st, ov, bin_neighbours, blocks(N), 256, 0, N, cfg_->topo, id_[1 - cur_id_], slot_of_id_, nbr_, counts_,
                      (int)n_fine_);
        TILD_CUDA(cudaGetLastError());
        cur_pos_ = 1 - cur_pos_;
        cur_u_ = 1 - cur_u_;
        cur_id_ = 1 - cur_id_;
        steps_since_sort_ = 0;
        return TILD_OK;
    }

    tild_status run_cycle_graph() {
        Range range("tild re-binning cycles (graph)");
        const int key = cur_pos_ | (cur_u_ << 1) | (cur_id_ << 2);
        tild_status st;
        if (!graph_ || graph_key_ != key) {
            invalidate_graph();
            const int sp = cur_pos_, su = cur_u_, si = cur_id_, ss = steps_since_sort_;
            cudaGraph_t g;
            TILD_CUDA(cudaStreamBeginCapture(stream_, cudaStreamCaptureModeThreadLocal));
            for (int half = 0; half < 2; ++half) {
                st = enqueue_sort();
                for (int s = 0; !st && s < cfg_->sort_every; ++s) st = enqueue_step();
                if (st) break;
            }
            cudaError_t e = cudaStreamEndCapture(stream_, &g);
            if (st) return st;
            TILD_CUDA(e);
            e = cudaGraphInstantiate(&graph_, g, 0);
            cudaGraphDestroy(g);
            TILD_CUDA(e);
            graph_key_ = key;
            // capture only recorded the launches; restore the host-side state
            cur_pos_ = sp;
            cur_u_ = su;
            cur_id_ = si;
            steps_since_sort_ = ss;
        }
        TILD_CUDA(cudaGraphLaunch(graph_, stream_));
        // two sorts and 2K steps flip every double buffer an even number of
        // times, so the parities are those the graph was captured with
        steps_since_sort_ = cfg_->sort_every;
        return TILD_OK;
    }
};

}  // namespace tild
