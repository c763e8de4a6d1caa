"""Edges of the tiled adjoint kernels (FP32 contexts): tiles above the bead
limit of their 32-bit sums, beads that left their tile's patch since the last
re-binning, every assignment order, and a trajectory window whose segments are
one and several steps long.

Tolerances: those of the force VJP's parity test in FP32 (1e-4). Repeated
calls and calls with out = lam agree bitwise.
"""
import numpy as np
import pytest

from oracle import tild_oracle as O
from paper_2302_02474_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2302_02474_gb300 import _build, binding

    _build.build()
    return binding


def _rel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


@pytest.mark.parametrize("order", [1, 2, 3, 4])
@pytest.mark.parametrize("n_chains,n,steps", [(60, 16, 0), (60, 24, 30), (900, 8, 0)])  # the last: 9,000 beads in one tile
def test_force_vjp_matches_oracle(B, order, n_chains, n, steps):
    import torch

    spec = I.small_system(n_chains=n_chains, N=10, n_a=4, L=0.5 * n, n=n, pmeorder=order, precision="fp32")
    pos = I.initial_positions(spec).astype(np.float32).astype(np.float64)
    t = B.Tild.from_spec(spec, sort_every=1000)
    t.set_positions(pos)
    if steps:  # far from the last re-binning
        t.init_velocities()
        t.step(steps)
        pos = t.positions()
    lam = np.random.default_rng(3).normal(size=pos.shape).astype(np.float32)
    m = O.model_from_spec(spec, I.species_of_beads(spec.moltypes), I.bond_pairs(spec.moltypes))
    ref = O.force_vjp(m, pos, lam.astype(np.float64))
    j, th = t.force_vjp(lam)
    assert _rel(j, ref["r"]) < 1e-4
    for k in ("chi", "kappa", "a"):
        assert th[k] == pytest.approx(ref[k], rel=1e-4, abs=1e-7 * abs(ref["a"])), k
    d = torch.from_numpy(lam).cuda()
    out = torch.empty_like(d)
    torch.cuda.synchronize()
    t.force_vjp(d, out=out)
    assert np.array_equal(out.cpu().numpy(), j)
    t.force_vjp(d, out=d)
    assert np.array_equal(d.cpu().numpy(), j)


@pytest.mark.parametrize("every", [1, 3, 8])
def test_trajectory_segments_agree(B, every):
    """Checkpoint distances give the same derivatives: every VJP reads either
    the context's state or its snapshot of the same state. Only beads that a
    different re-binning sends to the other gather differ, by rounding (1e-6)."""
    from paper_2302_02474_gb300.trajectory import trajectory_vjp

    spec = I.small_system(n_chains=50, N=10, n_a=4, L=8.0, n=16, pmeorder=2, precision="fp32")
    rng = np.random.default_rng(5)
    rb, vb = rng.normal(size=(spec.n_beads, 3)), rng.normal(size=(spec.n_beads, 3))
    got = []
    for c in (every, 20):
        t = B.Tild.from_spec(spec, sort_every=4)
        t.set_positions(I.initial_positions(spec))
        t.init_velocities()
        got.append(trajectory_vjp(t, 8, rb, vb, c))
    for k in ("r0", "v0"):
        assert _rel(got[0][k], got[1][k]) < 1e-6
