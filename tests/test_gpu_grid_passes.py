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
