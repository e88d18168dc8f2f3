"""Both sides of the rule by which schedule 1 takes one or two steps per launch: a few
large lattices beside the small ragged ones take the batch to two steps.  Against
single lattices stepped one node per thread, bit for bit."""
import pytest

from tests.test_gpu_batch_two_step import _cfgs, _fields, _same, _want

pytestmark = pytest.mark.gpu


def _run(storage, check, chunk, extra):
    import torch
    from paper_1908_06742_gb300 import ddflb as D
    cfgs = _cfgs(D, storage, check)
    for k, (nx, ny) in enumerate(extra):
        cfgs.append(D.Config(nx=nx, ny=ny, bc=("periodic", "cavity", "channel")[k % 3],
                             storage=storage, nu=0.03, diffusivity=0.03, u_lid=0.05, phi_lid=1.1,
                             phi_wall=0.4, check_every=check))
    b = D.Batch(cfgs).set_run(tol=0.0, steps_per_launch=chunk).set_schedule(1)
    fs = [_fields(torch, c.nx, c.ny, i) for i, c in enumerate(cfgs)]
    for i, f in enumerate(fs):
        b.set_instance_run(i, -1.0, 2 * check if check and i % 3 == 1 else 0)
        b.init(i, *f)
    b.step(2 * chunk + 3)
    b.init(4, *fs[4])          # an instance that joins at an odd time
    b.set_schedule(0).step(4)
    b.set_schedule(1).step(chunk + 2)
    st = b.stats()
    for i, c in enumerate(cfgs):
        steps = int(st["state_time"][i] - st["init_time"][i])
        assert _same(torch, b.fields(i), _want(D, c, fs[i], steps)), (i, c.nx, c.ny, c.bc)


@pytest.mark.parametrize("storage,check,chunk", [("fp32", 7, 5), ("fp32", 0, 6), ("fp16", 4, 9),
                                                 ("bf16", 1, 3), ("fp32", 1000, 11)])
@pytest.mark.parametrize("extra", [[], [(1000, 901), (1021, 1300), (1300, 997)]])
def test_either_side_of_the_rule(storage, check, chunk, extra):
    _run(storage, check, chunk, extra)
