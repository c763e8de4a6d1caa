"""Roundings that are part of the definition of an FP32 context's results.

Density: every weight is round(fl(w_x fl(w_y w_z)) 2^22), by whichever bead
kernel it is spread. Parameter derivatives of a force product: sums over
wavevectors that nearly cancel, so their last digits show the roundings of the
weights and of every stage of the transforms; tests/golden/force_vjp_theta.txt
holds them, with their errors against the FP64 oracle, as bits. Steps: checksums
and derivatives in tests/golden/trajectory_bits.txt, of noiseless trajectories on
every split of the transform lengths. Comparisons
are exact.
"""
import os

import numpy as np
import pytest

from paper_2302_02474_gb300 import inputs as I

pytestmark = pytest.mark.gpu
GOLDEN = os.path.join(os.path.dirname(os.path.abspath(__file__)), "golden", "force_vjp_theta.txt")


@pytest.fixture(scope="module")
def B():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2302_02474_gb300 import _build, binding

    _build.build()
    return binding


# tiled grids by the per-bead and by the tiled kernel, an any-size grid
@pytest.mark.parametrize("n,n_chains", [(16, 200), (24, 6000), (30, 700)])
def test_density_is_the_sum_of_rounded_weights(B, n, n_chains):
    spec = I.small_system(n_chains=n_chains, N=10, n_a=4, L=0.5 * n, n=n, precision="fp32")
    t = B.Tild.from_spec(spec)
    pos = I.initial_positions(spec).astype(np.float32)
    t.set_positions(pos)
    s = pos * np.float32(2.0)  # grid units, exact
    cell = np.floor(s)
    frac = s - cell
    w = np.stack([np.float32(1) - frac, frac])  # [point, bead, axis]
    want = np.zeros((2, n, n, n), dtype=np.int64)
    sp = I.species_of_beads(spec.moltypes)
    j = cell.astype(np.int64)
    for c in range(2):
        for b in range(2):
            wyz = w[b, :, 1] * w[c, :, 2]
            for a in range(2):
                k = np.rint((w[a, :, 0] * wyz).astype(np.float64) * 2.0**22).astype(np.int64)
                np.add.at(want, (sp, (j[:, 2] + c) % n, (j[:, 1] + b) % n, (j[:, 0] + a) % n), k)
    got = t.density(dtype=np.float64) * (spec.L / n) ** 3 * 2.0**22
    assert np.array_equal(np.rint(got).astype(np.int64), want)


def _golden():
    rows = []
    with open(GOLDEN) as f:
        for line in f:
            if line.strip() and not line.startswith("#"):
                p = line.split()
                rows.append((int(p[0]), int(p[1]), int(p[2]), [float.fromhex(x) for x in p[3:6]]))
    return rows


def theta(B, n, order, n_chains):
    spec = I.small_system(n_chains=n_chains, N=10, n_a=4, L=0.5 * n, n=n, pmeorder=order, precision="fp32")
    t = B.Tild.from_spec(spec)
    t.set_positions(I.initial_positions(spec).astype(np.float32))
    lam = np.random.default_rng(17 * n + order).normal(size=(spec.n_beads, 3)).astype(np.float32)
    th = t.force_vjp(lam)[1]
    return [th[k] for k in ("chi", "kappa", "a")]


@pytest.mark.parametrize("n,order,n_chains,want", _golden())
def test_parameter_derivatives_of_a_force_product(B, n, order, n_chains, want):
    assert theta(B, n, order, n_chains) == want


def _trajectory_golden():
    with open(os.path.join(os.path.dirname(GOLDEN), "trajectory_bits.txt")) as f:
        return [line.split() for line in f if line.strip() and not line.startswith("#")]


def trajectory(B, n, order, n_chains, scheme):
    """Checksums of positions and velocities after 9 steps, and the bits of the
    parameter derivatives through 4 steps."""
    import zlib

    from paper_2302_02474_gb300.trajectory import trajectory_vjp

    spec = I.small_system(n_chains=n_chains, N=10, n_a=4, L=0.5 * n, n=n, pmeorder=order, precision="fp32")
    t = B.Tild.from_spec(spec)
    t.set_integrator(0.005, 1.0, 0.0, 1.0)  # no noise: sums and products alone
    t.set_scheme(scheme)
    t.set_positions(I.initial_positions(spec).astype(np.float32))
    rng = np.random.default_rng(n + order)
    t.set_velocities(rng.normal(size=(spec.n_beads, 3)).astype(np.float32))
    lam = rng.normal(size=(spec.n_beads, 3)).astype(np.float32)
    g = trajectory_vjp(t, 4, lam, lam, 4)
    t.step(5)
    sums = ["%08x" % zlib.crc32(np.ascontiguousarray(x).tobytes()) for x in (t.positions(dtype=np.float32), t.velocities(dtype=np.float32))]
    return sums + [float(g[k]).hex() for k in ("chi", "kappa", "a")]


@pytest.mark.parametrize("row", _trajectory_golden(), ids=lambda r: "-".join(r[:4]))
def test_steps_and_derivatives_through_them(B, row):
    assert trajectory(B, int(row[0]), int(row[1]), int(row[2]), row[3]) == row[4:]
