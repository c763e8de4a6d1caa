"""The debug build's checks of the per-bead and adjoint kernels: an index
outside a context's arrays raises kErrBounds and is not used.

Every array is allocated several times as large as the kernels are told, and
the planted indices (a neighbour slot, a bead id, a species, a position more
than a period away) stay within that allocation, so no access leaves it,
checked or not. What an unchecked access would change or read holds a marker.
"""
import os
import shutil
import subprocess

import pytest

from paper_2302_02474_gb300 import _build

SRC = r'''
#include <cstdio>
#include <vector>
#include "generic_kernels.cuh"
#include "vjp_kernels.cuh"
using namespace tild;
constexpr int N = 8, n = 8, M = n * n * n, PAD = 8;
template <typename T> T* dev(const std::vector<T>& h) {
    T* d;
    cudaMalloc(&d, h.size() * sizeof(T));
    cudaMemcpy(d, h.data(), h.size() * sizeof(T), cudaMemcpyHostToDevice);
    return d;
}
enum { kGood, kSlot, kId, kSpecies, kFar };
template <typename T> void run(const char* type, int fault) {
    std::vector<T> pos(PAD * N, T(1.3)), vec(PAD * 3 * N, T(1));
    std::vector<int> id(PAD * N);
    for (int i = 0; i < PAD * N; ++i) id[i] = i < N ? i : 0;
    std::vector<int2> nbr(N, make_int2(-1, -1));
    if (fault == kSlot) nbr[3] = make_int2(N, -1);
    if (fault == kId) id[3] = N + 1;
    if (fault == kSpecies) id[3] |= 3 << kSpeciesShift;
    if (fault == kFar) pos[3] = T(2.6 * 8.0);
    BeadParams<T> p = {};
    p.n_beads = N;
    p.n = n;
    p.tiles = 1;
    p.species = 2;
    p.L = T(8);
    p.inv_L = T(0.125);
    p.inv_dx = T(1);
    p.su = p.sd = p.sh = p.vu = p.wu = p.e_len = p.e_vel = T(1);
    BeadBuffers<T> b = {};
    b.px = dev(pos);
    b.py = b.pz = dev(std::vector<T>(PAD * N, T(1.3)));
    b.qx = dev(pos);
    b.qy = dev(pos);
    b.qz = dev(pos);
    b.ux = dev(pos);
    b.uy = dev(pos);
    b.uz = dev(pos);
    b.id = dev(id);
    b.nbr = dev(nbr);
    b.tile_start = dev(std::vector<int>{0, N});
    std::vector<cplx_t<T>> zero(8 * PAD * M, cplx_t<T>{T(0), T(0)});
    b.grad = dev(zero);
    b.rho_fx = dev(std::vector<unsigned long long>(8 * PAD * M, 0ull));
    b.step = dev(std::vector<unsigned long long>{1});
    b.err = dev(std::vector<unsigned>{0});
    b.f_out = dev(vec);
    b.v_out = dev(vec);
    b.partials = dev(std::vector<double>(1024, 0.0));
    unsigned long long* fx = dev(std::vector<unsigned long long>(6 * PAD * M, 0ull));
    const T *lam = dev(vec), *grid = dev(std::vector<T>(8 * PAD * M, T(0)));
    T* out = dev(vec);
    auto* bits = dev(std::vector<typename AdjointFixed<T>::bits_t>{AdjointFixed<T>::abs_bits_host()});
    auto say = [&](const char* kernel) {
        unsigned e = 0;
        cudaMemcpy(&e, b.err, sizeof(e), cudaMemcpyDeviceToHost);
        cudaMemset(b.err, 0, sizeof(e));
        printf("%s %s %d %u %d\n", kernel, type, fault, e, (int)cudaGetLastError());
    };
    generic_bead_kernel<2, kModeSpread, T, 3><<<1, 32>>>(p, b, n);
    say("spread");
    generic_bead_kernel<2, kModeForce, T, 3><<<1, 32>>>(p, b, n);
    say("force");
    generic_bead_kernel<2, kModeSetVel, T, 3><<<1, 32>>>(p, b, n);
    say("set_velocity");
    generic_bead_kernel<2, kModeStep, T, 3><<<1, 32>>>(p, b, n);
    say("step");
    adjoint_kernel<2, T><<<1, 256>>>(p, b, b.grad, out);
    say("adjoint");
    bead_sums64<T><<<1, 256>>>(p, b, lam, lam, b.partials);
    say("sums64");
    density_vjp_kernel<2, T><<<1, 256>>>(p, b, grid, T(1), out);
    say("density_vjp");
    vjp_spread<2, T><<<1, 256>>>(p, b, lam, fx, bits, 40);
    say("vjp_spread");
    vjp_beads<2, T><<<1, 256>>>(p, b, b.grad, b.grad, lam, T(1), out);
    say("vjp_beads");
    if constexpr (sizeof(T) == 4) {
        vjp_spread_tiled<2><<<1, 256, vjp_spread_smem<2>()>>>(p, b, lam, fx, bits, 40);
        say("vjp_spread_tiled");
        vjp_beads_tiled<2><<<1, 256, vjp_beads_smem<2>()>>>(p, b, b.grad, b.grad, lam, T(1), out);
        say("vjp_beads_tiled");
    }
}
int main() {
    cudaFuncSetAttribute(vjp_spread_tiled<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)vjp_spread_smem<2>());
    cudaFuncSetAttribute(vjp_beads_tiled<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)vjp_beads_smem<2>());
    for (int fault = kGood; fault <= kFar; ++fault) {
        run<float>("float", fault);
        run<double>("double", fault);
    }
    return 0;
}
'''
# what each kernel indexes with: neighbour slot, bead id, species, stencil
USES = {
    "spread": "-isf", "force": "sisf", "set_velocity": "sisf", "step": "sisf", "adjoint": "sisf", "sums64": "s---",
    "density_vjp": "-isf", "vjp_spread": "-isf", "vjp_beads": "sisf", "vjp_spread_tiled": "-isf", "vjp_beads_tiled": "sisf",
}
K_ERR_BOUNDS = 2


def _compile(tmp_path):
    src, exe = tmp_path / "checks.cu", tmp_path / "checks"
    # 1.0's bit pattern, for max|lam|
    src.write_text(SRC.replace("AdjointFixed<T>::abs_bits_host()", "sizeof(T) == 4 ? 0x3f800000ull : 0x3ff0000000000000ull"))
    cmd = [_build._nvcc(), *_build.ARCH, "-O1", "-std=c++17", "-DTILD_DEBUG=1", "-I", _build.INCLUDE, "-I", _build.CSRC, str(src), "-o", str(exe)]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
    return exe


def test_checked_kernels_compile(tmp_path):
    if not (shutil.which("nvcc") or os.path.exists("/usr/local/cuda/bin/nvcc")):
        pytest.skip("no nvcc")
    _compile(tmp_path)


@pytest.mark.gpu
def test_an_index_out_of_range_raises_the_flag(tmp_path):
    r = subprocess.run([str(_compile(tmp_path))], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stderr
    rows = [line.split() for line in r.stdout.splitlines()]
    assert len(rows) == 5 * (11 + 9)
    for kernel, kind, fault, err, status in rows:
        flagged = int(fault) > 0 and USES[kernel][int(fault) - 1] != "-"
        assert int(status) == 0
        assert int(err) & K_ERR_BOUNDS == (K_ERR_BOUNDS if flagged else 0), (kernel, kind, fault)
