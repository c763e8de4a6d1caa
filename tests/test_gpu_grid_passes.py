"""The transforms of the tiled grids at every length and launch shape: the
spectrum and the field gradients against numpy's FP64 transforms of the same
density.

Tolerance: a transform of M points in precision eps has a relative L2 error
of at most about eps log2 M; the spectrum takes one, a gradient two and the
multiply, so 3 eps log2(M) bounds both (norm-wise).
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


CASES = [(n, "fp32") for n in (8, 16, 24, 32, 40, 48, 64, 80, 128, 256)] + [(n, "fp64") for n in (8, 24, 32, 48, 64, 80, 128)]


@pytest.mark.parametrize("n,prec", CASES)
def test_spectrum_and_gradients_match_numpy(B, n, prec):
    spec = I.small_system(n_chains=150, N=8, n_a=3, L=0.55 * n, n=n, precision=prec)
    t = B.Tild.from_spec(spec)
    t.set_positions(I.initial_positions(spec))
    rho = t.density(dtype=np.float64)
    z = np.fft.fftn(rho, axes=(1, 2, 3))
    f = np.fft.fftfreq(n, 1.0 / n) * 2 * np.pi / spec.L
    g = f.copy()
    g[n // 2] = 0.0
    k2 = f[:, None, None] ** 2 + f[None, :, None] ** 2 + f[None, None, :] ** 2
    rho0 = spec.n_beads / spec.L**3
    u = np.exp(-k2 * spec.a**2) / rho0
    w = [u * (spec.kappa * z[0] + (spec.chi + spec.kappa) * z[1]), u * ((spec.chi + spec.kappa) * z[0] + spec.kappa * z[1])]
    want = np.empty((3, n, n, n, 2))
    for d, k in enumerate((g[None, None, :], g[None, :, None], g[:, None, None])):
        for s in range(2):
            want[d, ..., s] = np.fft.ifftn(1j * k * w[s]).real
    eps = np.finfo(np.float32 if prec == "fp32" else np.float64).eps
    tol = 3 * eps * np.log2(n**3)
    zc = z[0] + 1j * z[1]
    shapes = [(512, t.launch_shapes()[1])]
    for s in [(1024, shapes[0][1]), (256, shapes[0][1]), (128, shapes[0][1]), (0, shapes[0][1])]:
        try:
            t.set_launch_shapes(*s)
            shapes.append(s)
        except B.TildError:
            pass
    for s in shapes:
        t.set_launch_shapes(*s)
        got = t.spectrum(dtype=np.float64)
        assert np.linalg.norm(got - zc) <= tol * np.linalg.norm(zc), s
        got = t.field_gradient(dtype=np.float64)
        assert np.linalg.norm(got - want) <= tol * np.linalg.norm(want), s


ANY = [(3, n) for n in (4, 7, 17, 20, 26, 34, 45, 55)] + [(2, n) for n in (4, 13, 32, 65, 127, 300, 1500)]


@pytest.mark.parametrize("species", [2, 3])
@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("dim,n", ANY)
def test_any_size_gradients_match_numpy(B, dim, n, prec, species):
    """Factors in registers and through the second line buffer (primes), both
    last axes, one and two species pairs, and lines too long for the fused
    last pass. A factor of R points is a direct sum of R terms, so a line of
    n1 n2 points has a relative error of at most about eps (n1 + n2); the
    gradients take dim axes twice."""
    mt = (I.MolType(120, 6, 3),)
    L = 0.55 * n
    draw = I.random_walk_positions_2d if dim == 2 else I.random_walk_positions
    t = B.Tild(L, n, 1, prec, 5, dim=dim)
    t.set_chains([(m.n_chains, m.N, m.n_a) for m in mt], 1.0)
    chi = np.array([[0.0, 1.1, 0.6], [1.1, 0.0, 0.4], [0.6, 0.4, 0.0]])[:species, :species]
    if species == 3:
        t.set_species(3, np.arange(720) % 3)
    t.set_interactions(1.1, 6.0, 0.5)
    if species == 3:
        t.set_chi_matrix(chi)
    t.set_positions(draw(mt, L, 1.0, 7))
    rho = t.density(dtype=np.float64)
    axes = (1, 2, 3) if dim == 3 else (2, 3)
    f = np.fft.fftfreq(n, 1.0 / n) * 2 * np.pi / L
    g = f.copy()
    if n % 2 == 0:
        g[n // 2] = 0.0
    kz = f if dim == 3 else np.zeros(1)
    k2 = kz[:, None, None] ** 2 + f[None, :, None] ** 2 + f[None, None, :] ** 2
    u = np.exp(-k2 * 0.5**2) / (720 / L**dim)
    z = np.fft.fftn(rho, axes=axes)
    w = [u * sum((chi[i, j] + 6.0) * z[j] for j in range(species)) for i in range(species)]
    got = t.field_gradient(dtype=np.float64)
    got = got[None] if species == 2 else got  # [pair, D, z, y, x, 2]
    n1 = max(d for d in range(1, int(n**0.5) + 1) if n % d == 0)
    tol = 2 * dim * np.finfo(np.float32 if prec == "fp32" else np.float64).eps * (n1 + n // n1)
    ks = (g[None, None, :], g[None, :, None], g[:, None, None])[:dim]
    for d in range(dim):
        for s in range(species):
            want = np.fft.ifftn(1j * ks[d] * w[s], axes=tuple(a - 1 for a in axes)).real
            err = np.linalg.norm(got[s // 2, d, ..., s % 2] - want)
            assert err <= tol * np.linalg.norm(want), (d, s)
