"""Chunks that fall on ever other phases of the residual check: the same states as the
persistent schedule, and ddflb_batch_step stays asynchronous however many there are."""
import time

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _batch(schedule, check, chunk):
    from paper_1908_06742_gb300 import ddflb as D
    cfgs = [D.Config(nx=n, ny=n, bc="cavity", u_lid=0.05, check_every=check) for n in (40, 64, 90)]
    b = D.Batch(cfgs).set_schedule(schedule).set_run(tol=0.0, steps_per_launch=chunk)
    for i, c in enumerate(cfgs):
        one = np.ones((c.ny, c.nx), np.float32)
        b.init(i, one, 0 * one, 0 * one, 0.5 * one)
    return b


@pytest.mark.parametrize("check,chunk,calls", [(37, 50, 90), (7, 10, 40), (10, 3, 40), (20, 40, 5)])
def test_many_phases(check, chunk, calls):
    import torch
    a, b = _batch(0, check, chunk), _batch(1, check, chunk)
    for x in (a, b):
        for _ in range(calls):
            x.step(chunk)
    sa, sb = a.stats(), b.stats()
    for i in range(3):
        for k, v in a.fields(i).items():
            # (bits: the vorticity is NaN where the scalar vanishes, in two corners)
            assert torch.equal(v.view(torch.int32), b.fields(i)[k].view(torch.int32)), (i, k)
    assert np.array_equal(sa["state_time"], sb["state_time"])
    # (the tiles' sums are added in the order of each schedule's own reduction)
    assert np.allclose(sa["residual"], sb["residual"], rtol=1e-10, atol=0.0)


def test_step_stays_asynchronous():
    import torch
    b = _batch(1, 37, 50)
    for _ in range(30):  # more phases than graphs are kept
        b.step(50)
    torch.cuda.synchronize()
    torch.cuda._sleep(1_000_000_000)  # half a second of the device's time
    t0 = time.perf_counter()
    for _ in range(3):
        b.step(50)
    queued = time.perf_counter() - t0
    torch.cuda.synchronize()
    total = time.perf_counter() - t0
    assert total > 0.3 and queued < 0.5 * total
