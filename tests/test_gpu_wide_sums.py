"""Sums of observables in FP32 contexts have the precision and the range of
FP64 sums: against math.fsum of the terms, which the test forms in 64 bits from
the float velocities, positions and spectra that the context reports.

Tolerance: the terms enter exactly; a block's sum is rounded to 53 bits, at
most 32 blocks are added in a tree of five levels, and the formula around the
sum has four products: ten roundings of 2^-53, 1.2e-15.
"""
import math

import numpy as np
import pytest

from paper_2302_02474_gb300 import inputs as I

pytestmark = pytest.mark.gpu
TOL = 1.2e-15


@pytest.fixture(scope="module")
def B():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2302_02474_gb300 import _build, binding

    _build.build()
    return binding


def _context(B, n, order, n_chains, N, kT=1.0, chi=0.0, kappa=0.0, a=0.5, species=2):
    t = B.Tild(8.0, n, order, "fp32", 3)
    t.set_chains([(n_chains, N, N // 2)], 1.0)
    t.set_interactions(chi, kappa, a)
    if species > 2:
        t.set_species(species, np.arange(n_chains * N) % species)
        t.set_chi_matrix([[0.0 if i == j else 0.3 + 0.1 * (i + j) for j in range(species)] for i in range(species)])
    t.set_integrator(0.005, 1.0, kT, 1.0)
    return t


# tiled (16, order 3), per bead (16, order 1) and any-size (15) kernels
@pytest.mark.parametrize("n,order,beads", [(16, 3, 20000), (16, 1, 2000), (15, 1, 2000)])
@pytest.mark.parametrize("size,kT", [(1.0, 1.0), (1e25, 1.0), (1e-30, 0.0), (1e-30, 1.0)])
def test_kinetic_energy(B, n, order, beads, size, kT):
    rng = np.random.default_rng(n)
    t = _context(B, n, order, beads, 1, kT)  # free beads: the velocities are what was set
    t.set_positions(rng.random((beads, 3)) * 8.0)
    v = rng.normal(size=(beads, 3)).astype(np.float32)
    v[beads // 3, 1] = 4096.0  # its square is the larger part of the sum
    t.set_velocities(v * np.float32(size))
    _, e = t.compute(forces=False)
    got = t.velocities(dtype=np.float64)
    want = math.fsum(x * x for x in got.ravel().tolist()) * 0.5
    assert want > 0 and abs(e["kinetic"] - want) <= TOL * want


@pytest.mark.parametrize("n,order,beads", [(16, 3, 20000), (16, 1, 2000), (15, 1, 2000)])
@pytest.mark.parametrize("size", [1.0, 1e-18])
def test_bond_energy(B, n, order, beads, size):
    rng = np.random.default_rng(n)
    t = _context(B, n, order, beads // 2, 2)
    pos = np.float32(0.25) + (rng.random((beads // 2, 2, 3)) * 3.5 * size).astype(np.float32)
    if size < 1:  # every bead at the origin but for that
        pos = (rng.random((beads // 2, 2, 3)) * size).astype(np.float32)
    t.set_positions(pos.reshape(-1, 3))
    _, e = t.compute(forces=False)
    d = (pos[:, 0] - pos[:, 1]).astype(np.float64)  # float differences
    want = 1.5 * math.fsum(x * x for x in d.ravel().tolist())
    assert want > 0 and abs(e["bond"] - want) <= TOL * want
    if n == 16:
        g, _ = t.energy_gradient(with_positions=False)
        assert abs(g["e_bond"] - want) <= TOL * want


@pytest.mark.parametrize("species", [2, 4])
@pytest.mark.parametrize("a", [0.5, 9.0])  # 9: every smeared mode but k = 0 below e^-50
def test_field_energies(B, species, a):
    n, beads, L = 16, 4000, 8.0
    t = _context(B, n, 1, beads // 4, 4, chi=0.8, kappa=20.0, a=a, species=species)
    t.set_positions((np.random.default_rng(1).random((beads, 3)) * L).astype(np.float32))
    _, e = t.compute(forces=False)
    Z = np.atleast_1d(t.spectrum(dtype=np.float32)).reshape(-1, n, n, n).astype(np.complex64)
    m = np.fft.fftfreq(n, 1.0 / n)
    e1 = np.exp(-(a * 2 * math.pi * m / L) ** 2).astype(np.float32)
    uh = ((e1[None, None, :] * e1[None, :, None]) * e1[:, None, None]).astype(np.float64)
    idx = (-np.arange(n)) % n
    A = []
    for z in Z:
        zm = z[np.ix_(idx, idx, idx)]
        h = np.float32(0.5)
        A += [(h * (z.real + zm.real), h * (z.imag - zm.imag)), (h * (z.imag + zm.imag), -h * (z.real - zm.real))]
    A = [(x.astype(np.float64), y.astype(np.float64)) for x, y in A]
    V, rho0 = L**3, beads / L**3
    dV = V / n**3
    tx, ty = sum(x for x, _ in A), sum(y for _, y in A)
    kap = uh * (tx * tx + ty * ty)
    kap[0, 0, 0] = 0.0
    want = {"kappa": 20.0 / (2 * rho0) * dV * dV / V * math.fsum(kap.ravel().tolist())}
    pairs = [(i, j) for i in range(len(A)) for j in range(i + 1, len(A))]
    w = lambda i, j: 1.0 if species == 2 else float(np.float32(0.3 + 0.1 * (i + j)))  # noqa: E731
    chi = sum(w(i, j) * uh * (A[i][0] * A[j][0] + A[i][1] * A[j][1]) for i, j in pairs)
    want["chi"] = (0.8 if species == 2 else 1.0) / rho0 * dV * dV / V * math.fsum(chi.ravel().tolist())
    for k in want:
        # the test's own terms have up to four roundings each, of alternating sign over 4,096 modes
        assert want[k] != 0 and abs(e[k] - want[k]) <= 4 * TOL * abs(want[k]), k


# A velocity outside the range of floats sends every sum of the call to FP64; the
# energies are those of the ordinary sums, whose spectra are the same bits on
# tiled grids (TOL, twice) and differ by FP32 transforms of other factors elsewhere.
@pytest.mark.parametrize("n,dim,species,charged", [(16, 3, 2, False), (24, 3, 2, True), (16, 3, 4, False), (15, 3, 2, False), (21, 2, 3, False)])
def test_sums_again_in_fp64(B, n, dim, species, charged):
    chains, N, L = 250, 8, 8.0
    t = B.Tild(L, n, 1, "fp32", 3, dim=dim)
    t.set_chains([(chains, N, N // 2)], 1.0)
    t.set_interactions(0.8, 20.0, 0.5)
    if species > 2:
        t.set_species(species, np.arange(chains * N) % species)
        t.set_chi_matrix([[0.0 if i == j else 0.3 + 0.1 * (i + j) for j in range(species)] for i in range(species)])
    if charged:
        t.set_electrostatics(1.0, -1.0, 1.0, 0.5)
    t.set_integrator(0.005, 1.0, 1.0, 1.0)
    rng = np.random.default_rng(n)
    pos, v = rng.random((chains * N, 3)) * L, rng.normal(size=(chains * N, 3))
    if dim == 2:
        pos[:, 2] = v[:, 2] = 0.0
    t.set_positions(pos)
    t.set_velocities(v)
    _, e = t.compute(forces=False)
    t.set_velocities(v * 1e25)
    f, w = t.compute()
    for k in ("bond", "chi", "kappa", "elec"):
        assert abs(w[k] - e[k]) <= (2 * TOL if n % 8 == 0 else 2e-6) * abs(e[k]), k
    assert (e["elec"] != 0) == charged
    np.testing.assert_allclose(w["net_force"], f.astype(np.float64).sum(0), rtol=0, atol=1e-12 * np.abs(f).sum())


def test_energy_gradient_again_in_fp64(B):
    """Bonds of 1e-18: the gradient's sums in FP64 against an FP64 context's (2e-5, FP32 transforms)."""
    rng = np.random.default_rng(3)
    pos = (np.repeat(rng.random((500, 1, 3)) * 8.0, 4, axis=1)).astype(np.float32)
    pos[:3] = rng.random((3, 4, 3)) * 1e-18  # the only bonds that are not zero
    out = []
    for prec in ("fp32", "fp64"):
        t = B.Tild(8.0, 16, 2, prec, 3)
        t.set_chains([(500, 4, 2)], 1.0)
        t.set_interactions(0.8, 20.0, 0.5)
        t.set_positions(pos.reshape(-1, 3).astype(np.float64))
        out.append(t.energy_gradient(with_positions=False)[0])
    for k, ref in out[1].items():
        assert abs(out[0][k] - ref) <= 2e-5 * abs(ref), k
    assert 0 < out[0]["e_bond"] < 1e-30
