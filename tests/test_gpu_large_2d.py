"""Large 2D grids on either side of the rule that chooses line passes or
whole-axis passes: FP32 forces against an FP64 context's at the same float
positions, within the parity tests' 1e-5."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,species", [(600, 2), (601, 2), (641, 2), (719, 2), (1021, 2), (600, 4), (719, 4)])
def test_forces_match_fp64(n, species):
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2302_02474_gb300 import _build, binding as B

    _build.build()
    L, beads = 0.5 * n, 4000
    pos = (np.random.default_rng(n).random((beads, 3)) * L * np.array([1.0, 1.0, 0.0])).astype(np.float32).astype(np.float64)
    f = []
    for prec in ("fp32", "fp64"):
        t = B.Tild(L, n, 1, prec, 3, dim=2)
        t.set_chains([(beads // 4, 4, 2)], 1.0)
        t.set_interactions(0.8, 20.0, 0.5)
        if species > 2:
            t.set_species(species, np.arange(beads) % species)
            t.set_chi_matrix([[0.0 if i == j else 0.5 for j in range(species)] for i in range(species)])
        t.set_positions(pos)
        f.append(t.compute(energy=False)[0])
    assert np.linalg.norm(f[0] - f[1]) <= 1e-5 * np.linalg.norm(f[1])
