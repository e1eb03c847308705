"""Small calls back to back on one stream, their inputs and buffers changing
from call to call: each kernel of a call may be resident while the one before
still writes its operand.  Reference: the same plan with stage timing, where an
event between the stages keeps every kernel behind the one before; results
must agree bitwise."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ms,mz,n_phi,n_zs,n_ell,batch", [
    (16, 16, 32, 16, 48, 1),      # whole vectors, tiles, A1^T split over the passes
    (32, 32, 64, 32, 96, 2),
    (15, 13, 18, 11, 37, 1),      # nothing a multiple of 4: scalar reshapes, A2 entry by entry
    (64, 64, 128, 64, 256, 1),
])
def test_repeated_calls_match_ordered_ones(ms, mz, n_phi, n_zs, n_ell, batch):
    import torch
    from paper_2402_15641_gb300 import srt as S
    dz = 0.5
    g = S.Geometry(ms, mz, 0.5, dz, 0.9 * ms, n_phi, 0.0, n_zs, -0.5 * n_zs * dz, 0.5 * n_zs * dz, n_ell,
                   0.9 * ms - 0.36 * ms, 0.9 * ms + 0.36 * ms)
    plan = S.Plan(g)
    gen = torch.Generator(device="cuda").manual_seed(5)
    lead = () if batch == 1 else (batch,)
    fs = [torch.rand(*lead, *g.f_shape, generator=gen, device="cuda") for _ in range(8)]
    ps = [torch.randn(*lead, *g.p_shape, generator=gen, device="cuda") for _ in range(8)]
    plan.set_timing(True)
    want = []
    for f, p in zip(fs, ps):
        want.append((plan.forward(f).clone(), plan.adjoint(p).clone()))
        torch.cuda.synchronize()
    plan.set_timing(False)
    bad = torch.zeros((), dtype=torch.int64, device="cuda")
    x = torch.empty_like(fs[0])   # one buffer for all calls, written just before each
    y = torch.empty_like(ps[0])
    for i in range(400):
        k = (5 * i + 3) % 8
        x.copy_(fs[k])
        q = plan.forward(x)
        y.copy_(ps[k])
        a = plan.adjoint(y)
        bad += (q != want[k][0]).sum() + (a != want[k][1]).sum()
    assert int(bad) == 0
    plan.close()
