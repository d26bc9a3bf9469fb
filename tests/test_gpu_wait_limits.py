"""Waits that run out in the middle of a double-precision pass: whatever the limit, a step
either ends within it or is reported, the grid recovers, and nothing is left behind that
disturbs the next step."""
import pytest
import torch

from gpu_common import T, absorber_workload, cuda, host, pair, rel_l2, setup_both

pytestmark = pytest.mark.gpu


# two CTAs an SM; copies in turn and streamed matrices; several accumulator groups
@pytest.mark.parametrize("n", [(17, 8, 8, 16, 16), (65, 3, 4, 6, 10), (3, 32, 32, 4, 8)], ids=str)
@pytest.mark.parametrize("limit", [-1, 1, 2, 4, 16, 64, 256])
def test_step_ends_or_is_reported(n, limit):
    ts = T()
    og, gg = pair(0.2, 1.0, *n, G=2)
    kap, eta, ks, F0, g1, g2 = absorber_workload(og)
    op = setup_both(og, gg, kap, eta, ks, g1, g2)
    dt = 0.05 / (n[0] ** 2 + 4 * n[1] * n[2] + n[3] * n[4] * n[1])
    want = cuda(F0)
    gg.step(want, dt, 1)
    ts.ts_sync_status(gg.handle)
    ts.ts_set_wait_limit(gg.handle, limit)
    F = cuda(F0)
    gg.step(F, dt, 1)
    try:
        ts.ts_sync_status(gg.handle)
        assert limit > 0 and torch.equal(F, want)
    except ts.TSError as e:
        assert e.status == ts.TS_ERR_TIMEOUT
    ts.ts_set_wait_limit(gg.handle, 0)
    F = cuda(F0)
    gg.step(F, dt, 1)
    ts.ts_sync_status(gg.handle)
    assert torch.equal(F, want)
    assert rel_l2(host(F), op.run(F0, dt, 1)) < 1e-12
