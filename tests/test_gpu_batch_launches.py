"""Launches that a batch announces: those of its steps, and per re-binning
those of every replica as the replica itself counts them (four on small grids,
seven above 16,384 bins, as at 128^3)."""
import pytest

from paper_2302_02474_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("grids", [(24, 24), (24, 128), (128, 128)])
def test_batch_counts_every_replicas_rebinning(grids):
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2302_02474_gb300 import _build, binding as B

    _build.build()
    ts = []
    for n in grids:
        spec = I.small_system(n_chains=50, N=10, n_a=4, L=0.5 * n, n=n, precision="fp32")
        t = B.Tild.from_spec(spec, sort_every=5)
        t.set_positions(I.initial_positions(spec))
        t.init_velocities()
        ts.append(t)
    with B.TildBatch(ts) as bt:
        if bt.persistent:
            bt.set_persistent(False)
        for steps in (5, 10, 23):
            rebinning = sum(t.launches(steps) - 4 * steps for t in ts)  # an own step takes four
            assert bt.launches(steps) == 4 * steps * len(set(grids)) + rebinning
