"""Infinite and NaN samples: they reach the outputs whose rows hold an entry
for them and no others, in the tile products as in the row products, wherever
the record falls in a tile's list and whatever the dense width."""
import numpy as np
import pytest

from tests.gpu_helpers import geom_pair

pytestmark = pytest.mark.gpu


# mz up to 64: A1^T split over the passes; 100: one chunk, 132: two chunks of
# columns.  n_phi 16 and 160: A2 and A2^T below and above 128 columns.
@pytest.mark.parametrize("mz", [16, 64, 100, 132])
@pytest.mark.parametrize("n_phi", [16, 160])
@pytest.mark.parametrize("form", [dict(), dict(a1_full=True), dict(weight_dtype="bf16")])
def test_reaches_the_same_outputs_as_row_by_row(orc, mz, n_phi, form):
    import torch
    from paper_2402_15641_gb300 import srt as S
    g, _ = geom_pair(orc, ms=12, mz=mz, dxy=0.4, dz=0.4, radius=6.0, n_phi=n_phi, n_zs=mz, n_ell=23, **form)
    a, b = S.Plan(g), S.Plan(g.with_(rowwise=True))
    gen = np.random.default_rng(3)
    reached = 0
    for bad in (float("nan"), float("inf"), -float("inf")):
        for _ in range(4):
            f = torch.rand(g.f_shape, device="cuda")
            p = torch.randn(g.p_shape, device="cuda")
            f[tuple(int(gen.integers(0, n)) for n in g.f_shape)] = bad
            p[tuple(int(gen.integers(0, n)) for n in g.p_shape)] = bad
            for x, y in ((a.forward(f), b.forward(f)), (a.adjoint(p), b.adjoint(p))):
                reached += int((~torch.isfinite(y)).sum())
                assert torch.equal(torch.isfinite(x), torch.isfinite(y))
    assert reached > 0
