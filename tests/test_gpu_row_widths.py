"""The row products over the width classes of their dispatch: vectors of 4, 2
and 1 columns, 4 to 32 lanes to a row, two to four chunks, rows split over
blocks, few rows (four gathers in flight) and many (two, or one).

Against the FP64 oracle on seeded samples, with the bound of FP32 sums of a
row's entries (at most a few hundred), 1e-5 relative, as in the parity tests;
and bitwise between batch sizes: every variant sums a row in the same order, so
an item's result does not depend on the variant that its batch selects."""
import numpy as np
import pytest

from tests.gpu_helpers import geom_pair, rel_l2, to_dev, to_np

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def srt():
    import torch
    from paper_2402_15641_gb300 import build, srt as S
    assert torch.cuda.is_available()
    build.build()
    return S


def _sample_check(srt, orc, sz, opts, batch, n_shells, n_vox):
    g, o = geom_pair(orc, **opts, **sz)
    plan = srt.Plan(g)
    rng = np.random.default_rng(61)
    f = rng.uniform(0, 1, (batch, *g.f_shape)).astype(np.float32)
    y = rng.standard_normal((batch, *g.p_shape)).astype(np.float32)
    p = to_np(plan.forward(to_dev(f)))
    a = to_np(plan.adjoint(to_dev(y)))
    sh = np.stack([rng.integers(0, n, n_shells) for n in g.p_shape], axis=1)
    vx = np.stack([rng.integers(0, n, n_vox) for n in g.f_shape], axis=1)
    for b in range(batch):
        want = orc.forward_shells(o, f[b].astype(np.float64), sh)
        assert rel_l2(p[b][sh[:, 0], sh[:, 1], sh[:, 2]], want) <= 1e-5
        want = orc.adjoint_voxels(o, y[b].astype(np.float64), vx)
        assert rel_l2(a[b][vx[:, 0], vx[:, 1], vx[:, 2]], want) <= 1e-5


@pytest.mark.parametrize("mz", [1, 2, 3, 6, 9, 16, 17, 33, 36, 52, 64, 65, 70, 100, 132, 194, 260, 264])
@pytest.mark.parametrize("form", [dict(), dict(rowwise=True), dict(csr_only=True, rowwise=True, a1_full=True)])
def test_few_rows(srt, orc, mz, form):
    """Slab counts that are and are not whole vectors, below and above one
    part of 64 vectors; 12 sensor columns (quarter turns) of batch 2."""
    sz = dict(ms=7, mz=mz, dxy=0.4, dz=0.4 / max(1, mz // 16), radius=6.0, n_phi=12, n_zs=3, n_ell=17)
    _sample_check(srt, orc, sz, form, 2, 120, 40)


@pytest.mark.parametrize("mz,n_phi,n_ell,form", [(132, 64, 400, dict()), (66, 90, 480, dict()),
                                                 (101, 64, 400, dict(a1_full=True)),
                                                 (264, 64, 400, dict(a1_full=True)),
                                                 (20, 256, 400, dict(rowwise=True)),
                                                 (8, 512, 200, dict(rowwise=True))])
def test_many_rows(srt, orc, mz, n_phi, n_ell, form):
    """Enough rows to fill the GPU, so that the loop keeps two gathers in
    flight."""
    sz = dict(ms=8, mz=mz, dxy=0.4, dz=0.05, radius=6.0, n_phi=n_phi, n_zs=2, n_ell=n_ell)
    _sample_check(srt, orc, sz, form, 1, 150, 30)


@pytest.mark.parametrize("mz", [4, 16, 20, 32, 36, 64, 68])
@pytest.mark.parametrize("form", [dict(), dict(a1_rotation=True), dict(weight_dtype="bf16")])
def test_adjoint_group_passes(srt, orc, mz, form):
    """A1^T with the symmetry passes shared by a warp's groups of lanes (at
    most 64 slabs: 4, 8 and 16 lanes to a group; quarter turns keep 8) and
    with a warp to a pass (68), batch 3, an odd number of tiles."""
    sz = dict(ms=10, mz=mz, dxy=0.4, dz=0.4, radius=6.0, n_phi=16, n_zs=3, n_ell=21)
    bf16 = form.get("weight_dtype") == "bf16"
    g, o = geom_pair(orc, **form, **sz)
    plan = srt.Plan(g)
    assert plan.info["a1_rot"] == (1 if form.get("a1_rotation") else 2)
    y = np.random.default_rng(63).standard_normal((3, *g.p_shape)).astype(np.float32)
    a = to_np(plan.adjoint(to_dev(y)))
    for b in range(3):
        want = orc.adjoint(o, y[b].astype(np.float64))
        assert rel_l2(a[b], want) <= (5e-3 if bf16 else 1e-5)


@pytest.mark.parametrize("ms,mz,n_phi,batch", [(128, 132, 72, 8), (130, 260, 16, 8), (134, 160, 16, 8),
                                                (72, 136, 16, 8)])
@pytest.mark.parametrize("form", [dict(), dict(a1_full=True), dict(weight_dtype="bf16")])
def test_a1t_of_large_batches(srt, orc, ms, mz, n_phi, batch, form):
    """A1^T of more than 128 slabs runs in blocks of 4 x 2 tiles where a batch
    fills many of them (4096, or 1024 with at most 64 columns), one of these
    volumes in 2 x 2: bitwise the same for every item, with tile counts that are
    and are not whole blocks and super-tiles."""
    import torch
    g, _ = geom_pair(orc, ms=ms, mz=mz, dxy=0.4, dz=0.3, radius=0.4 * ms, n_phi=n_phi, n_zs=5, n_ell=24, **form)
    plan = srt.Plan(g)
    y = torch.randn((batch, *g.p_shape), generator=torch.Generator(device="cuda").manual_seed(17), device="cuda")
    a = plan.adjoint(y)
    for b in range(batch):
        assert torch.equal(a[b], plan.adjoint(y[b].contiguous()))


def _batches_equal_single_items(plan, fn, shape, batches, seed):
    import torch
    x = torch.randn((max(batches), *shape), generator=torch.Generator(device="cuda").manual_seed(seed), device="cuda")
    one = [fn(x[b].contiguous()).clone() for b in range(max(batches))]
    for n in batches:
        if n > 1:
            y = fn(x[:n].contiguous())
            assert all(torch.equal(y[b], one[b]) for b in range(n)), n
    return one


@pytest.mark.parametrize("mz", [8, 32, 33, 34, 64, 66, 100, 101, 128, 132, 160, 192, 200, 202, 256, 264])
@pytest.mark.parametrize("ms", [127, 128])
@pytest.mark.parametrize("form", [dict(), dict(a1_full=True), dict(weight_dtype="bf16")])
def test_pixel_rows_bitwise_over_batches(srt, orc, mz, ms, form):
    """A1^T row by row at 128 x 128 pixels: one volume counts as few rows, five
    as many (two from 132 slabs on), so the same sums run with four, two and
    one gathers in flight, in half warps and whole ones, over super-tiles
    (128) and bands (127)."""
    g, _ = geom_pair(orc, ms=ms, mz=mz, dxy=0.2, dz=0.2, radius=20.0, n_phi=8, n_zs=3, n_ell=14, rowwise=True,
                     **form)
    plan = srt.Plan(g)
    _batches_equal_single_items(plan, plan.adjoint, g.p_shape, (1, 2, 5), 7)


@pytest.mark.parametrize("mz", [8, 16, 18, 21, 32, 33, 36, 48, 62, 64, 66, 80, 96, 100, 101, 128, 130, 132, 160,
                                192, 200, 201, 256, 258, 264, 300])
@pytest.mark.parametrize("form", [dict(), dict(a1_full=True), dict(weight_dtype="bf16")])
def test_a1_rows_bitwise_over_batches(srt, orc, mz, form):
    """A1 with 19264 rows an item, more than half a warp each fills the GPU with:
    one item counts as few rows, two as many where a row has more than 32
    vectors, five as many at every width."""
    g, _ = geom_pair(orc, ms=10, mz=mz, dxy=0.4, dz=0.1, radius=6.0, n_phi=64, n_zs=2, n_ell=301, **form)
    plan = srt.Plan(g)
    _batches_equal_single_items(plan, plan.forward, g.f_shape, (1, 2, 5), 9)


@pytest.mark.parametrize("n_phi", [3, 5, 8, 12, 16, 20, 24, 30, 33, 40, 48, 57, 64, 66, 72, 90, 101, 130])
@pytest.mark.parametrize("form", [dict(rowwise=True), dict(csr_only=True, rowwise=True),
                                  dict(rowwise=True, weight_dtype="bf16")])
def test_shell_rows_bitwise_over_batches(srt, orc, n_phi, form):
    """A2 and A2^T row by row, from the taps and as CSR, with 20480 rows: the
    dense width is the batch's columns, so one, two, three and eight items run in
    different width classes."""
    g, _ = geom_pair(orc, ms=6, mz=64, dxy=0.4, dz=0.1, radius=6.0, n_phi=n_phi, n_zs=64, n_ell=320, **form)
    plan = srt.Plan(g)
    _batches_equal_single_items(plan, plan.forward, g.f_shape, (1, 2, 3, 8), 11)
    _batches_equal_single_items(plan, plan.adjoint, g.p_shape, (1, 2, 3, 8), 12)


@pytest.mark.parametrize("n_ell,batch", [(38, 1), (39, 1), (304, 1), (305, 1), (304, 2), (38, 8)])
def test_edges_of_the_row_rules(srt, orc, n_ell, batch):
    """Just below and above the row counts at which the variants change (9728:
    four lanes a row; 77824 rows of four to a warp, 19456 of one: two gathers)."""
    for mz, n_phi in ((8, 256), (64, 256), (136, 64)):
        sz = dict(ms=8, mz=mz, dxy=0.4, dz=0.05, radius=6.0, n_phi=n_phi, n_zs=2, n_ell=n_ell)
        _sample_check(srt, orc, sz, dict(), batch, 60, 10)
