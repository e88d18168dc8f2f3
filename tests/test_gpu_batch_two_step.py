"""Two-step launches of a batch (schedule 1) against single lattices stepped one
node per thread: bit-identical, for sizes at the edges of the 64-column strips,
mixed boundary kinds, odd chunks around the residual checks, instances that
join late or freeze, and changes of schedule on the way."""
import pytest

pytestmark = pytest.mark.gpu

SIZES = [(33, 9), (62, 17), (64, 64), (65, 20), (66, 33), (100, 31), (124, 40), (125, 8), (192, 50)]


def _cfgs(D, storage, check):
    bcs = ("cavity", "periodic", "channel")
    return [D.Config(nx=nx, ny=ny, bc=bcs[i % 3], storage=storage, nu=0.02 + 0.002 * i,
                     diffusivity=0.03, u_lid=0.05 + 0.003 * i, phi_lid=1.1, phi_wall=0.4,
                     check_every=check, scalar_model="srt" if i % 4 == 3 else "mrt")
            for i, (nx, ny) in enumerate(SIZES)]


def _fields(torch, nx, ny, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    r = lambda: torch.randn(ny, nx, generator=g, device="cuda")
    return 1 + 0.01 * r(), 0.02 * r(), 0.02 * r(), 1 + 0.1 * r()


def _want(D, cfg, f, steps):
    lat = D.Lattice(cfg).set_path(1).init(*f).step(steps)
    return lat.fields()


def _same(torch, a, b):
    return all(torch.equal(torch.nan_to_num(a[k], nan=7.0), torch.nan_to_num(b[k], nan=7.0))
               for k in a)


@pytest.mark.parametrize("storage,check,chunk", [("fp32", 7, 5), ("fp32", 0, 6), ("fp16", 4, 9),
                                                 ("bf16", 1, 3), ("fp32", 1000, 11)])
def test_batch_matches_single_lattices(storage, check, chunk):
    import torch
    from paper_1908_06742_gb300 import ddflb as D
    cfgs = _cfgs(D, storage, check)
    b = D.Batch(cfgs).set_run(tol=0.0, steps_per_launch=chunk).set_schedule(1)
    fs = [_fields(torch, c.nx, c.ny, i) for i, c in enumerate(cfgs)]
    for i, f in enumerate(fs):
        b.init(i, *f)
    b.step(2 * chunk + 3)
    b.init(4, *fs[4])          # an instance that joins at an odd time
    b.set_schedule(0).step(4)
    b.set_schedule(1).step(chunk + 2)
    n = 3 * chunk + 9
    for i, c in enumerate(cfgs):
        steps = n - (2 * chunk + 3) if i == 4 else n
        assert _same(torch, b.fields(i), _want(D, c, fs[i], steps)), (i, c.nx, c.ny, c.bc)


def test_frozen_instances_keep_their_state():
    """Instances that reach their step limit freeze one step past the check, and
    their state stays what it was while the others go on."""
    import torch
    from paper_1908_06742_gb300 import ddflb as D
    cfgs = _cfgs(D, "fp32", 6)
    b = D.Batch(cfgs).set_run(tol=0.0, steps_per_launch=10).set_schedule(1)
    fs = [_fields(torch, c.nx, c.ny, 50 + i) for i, c in enumerate(cfgs)]
    for i, f in enumerate(fs):
        b.set_instance_run(i, -1.0, 12 if i % 2 else 0)
        b.init(i, *f)
    b.step(37)
    st = b.stats()
    for i, c in enumerate(cfgs):
        assert bool(st["flags"][i]) == bool(i % 2)
        t = int(st["state_time"][i])
        assert t == (13 if i % 2 else 37)
        assert _same(torch, b.fields(i), _want(D, c, fs[i], t)), i
