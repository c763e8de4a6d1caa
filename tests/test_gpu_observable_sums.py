"""Sums of observables in FP32 contexts (pairs of floats) and the density
read-out: independence of the unit system, and agreement with FP64.

Tolerances: scaling every length by s leaves the energies (in kT) unchanged;
the FP32 positions of the two systems round differently, 6e-8 of a coordinate
of up to 20 bond lengths, so bonds and fields agree to about 20 x 6e-8 x 2 and
5e-6 bounds the energies. A density is the exact integer sum times the scale,
rounded once: the FP32 read-out is within one unit in the last place of the
FP64 read-out.
"""
import numpy as np
import pytest

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


@pytest.mark.parametrize("n", [16, 21])  # tiled and any-size kernels
@pytest.mark.parametrize("scale", [1e-9])
def test_energies_do_not_depend_on_the_length_unit(B, n, scale):
    spec = I.small_system(n_chains=300, N=10, n_a=4, L=8.0, n=n, precision="fp32")
    pos = I.initial_positions(spec)
    out = []
    for s in (1.0, scale):
        t = B.Tild(spec.L * s, n, 1, "fp32", 3)
        t.set_chains([(m.n_chains, m.N, m.n_a) for m in spec.moltypes], spec.b * s)
        t.set_interactions(spec.chi, spec.kappa, spec.a * s)
        t.set_positions(pos * s)
        _, e = t.compute(forces=False)
        out.append(e)
        if n == 16:
            g, _ = t.energy_gradient(with_positions=False)
            for k, ref in (("e_bond", e["bond"]), ("e_chi", e["chi"]), ("e_kappa", e["kappa"])):
                assert abs(g[k] - ref) <= 1e-12 * abs(ref), k
            out[-1]["da"] = g["dU_da"] * s
    for k in ("bond", "chi", "kappa") + (("da",) if n == 16 else ()):
        assert abs(out[1][k] - out[0][k]) <= 5e-6 * abs(out[0][k]), k


@pytest.mark.parametrize("n_chains,n", [(7, 8), (3000, 16), (40000, 8)])  # the last: sums beyond 2^31
def test_density_float_readout(B, n_chains, n):
    spec = I.small_system(n_chains=n_chains, N=10, n_a=4, L=0.5 * n, n=n, precision="fp32")
    t = B.Tild.from_spec(spec)
    t.set_positions(np.full((spec.n_beads, 3), 0.3) if n_chains == 40000 else I.initial_positions(spec))
    d64, d32 = t.density(dtype=np.float64), t.density(dtype=np.float32)
    assert d64.max() > 0
    assert np.all(np.abs(d32 - d64) <= np.spacing(np.abs(d64).astype(np.float32)))


@pytest.mark.parametrize("n", [16, 21])  # tiled and any-size kernels
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_an_infinite_velocity_gives_an_infinite_kinetic_energy(B, n, precision):
    spec = I.small_system(n_chains=300, N=10, n_a=4, L=8.0, n=n, precision=precision)
    t = B.Tild(spec.L, n, 1, precision, 3)
    t.set_chains([(m.n_chains, m.N, m.n_a) for m in spec.moltypes], spec.b)
    t.set_interactions(spec.chi, spec.kappa, spec.a)
    t.set_integrator(0.005, 1.0, 1.0)
    t.set_positions(I.initial_positions(spec))
    v = np.zeros((3000, 3))
    v[7, 1] = -np.inf
    t.set_velocities(v)
    _, e = t.compute(forces=False)
    assert e["kinetic"] == np.inf
    assert np.isfinite(e["bond"]) and np.isfinite(e["chi"]) and np.isfinite(e["kappa"])
