"""Steps that a caller captures into a CUDA graph of its own advance the state
at every replay: an even number of steps ends in the buffer it started from."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _fields(nx, ny):
    y, x = np.meshgrid(np.arange(ny) / ny, np.arange(nx) / nx, indexing="ij")
    u = 0.01 * np.sin(2 * np.pi * x) * np.cos(2 * np.pi * y)
    v = -0.01 * np.cos(2 * np.pi * x) * np.sin(2 * np.pi * y)
    phi = 1 + 0.1 * np.sin(2 * np.pi * x) * np.sin(2 * np.pi * y)
    return [a.astype(np.float32) for a in (np.ones_like(u), u, v, phi)]


def _replay(stream, step, times):
    import torch
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph, stream=stream):
        step()
    with torch.cuda.stream(stream):
        for _ in range(times):
            graph.replay()
    torch.cuda.synchronize()


@pytest.mark.parametrize("bc", ["periodic", "cavity"])
@pytest.mark.parametrize("nx,ny,n", [(64, 64, 4), (64, 64, 12), (64, 64, 68), (160, 96, 2),
                                     (400, 300, 2), (1504, 1408, 2), (1504, 1408, 6),
                                     (1504, 1408, 66)])
def test_lattice_steps_in_a_callers_graph(nx, ny, n, bc):
    import torch
    from paper_1908_06742_gb300 import ddflb as D
    s = torch.cuda.Stream()
    cfg = D.Config(nx=nx, ny=ny, bc=bc, u_lid=0.05 if bc == "cavity" else 0.0)
    lats = [D.Lattice(cfg, stream=s) for _ in range(2)]
    for lat in lats:
        lat.init(*_fields(nx, ny))
    lats[0].set_path(1)
    lats[0].step(3 * n)
    _replay(s, lambda: lats[1].step(n), 3)
    f, g = [torch.cat([p.reshape(-1) for p in lat.populations()]) for lat in lats]
    torch.cuda.synchronize()
    assert torch.equal(f, g)


@pytest.mark.parametrize("schedule", [0, 1])
@pytest.mark.parametrize("check,n,chunk", [(0, 6, 500), (4, 8, 500), (4, 8, 8), (5, 10, 10),
                                           (5, 10, 5), (3, 4, 2)])
def test_batch_steps_in_a_callers_graph(check, n, chunk, schedule):
    import torch
    from paper_1908_06742_gb300 import ddflb as D
    s = torch.cuda.Stream()
    cfgs = [D.Config(nx=k, ny=k + 6, bc="cavity", u_lid=0.05, check_every=check)
            for k in (40, 64, 70)]
    got = []
    for captured in (False, True):
        b = D.Batch(cfgs, stream=s).set_schedule(schedule)
        b.set_run(tol=0.0, steps_per_launch=chunk)
        for i, c in enumerate(cfgs):
            b.init(i, *_fields(c.nx, c.ny))
        b.step(n)  # (the step from time 0 takes no check: captured steps start after it)
        if captured:
            _replay(s, lambda: b.step(n), 3)
        else:
            b.step(3 * n)
        fields = [torch.stack(list(b.fields(i).values())) for i in range(3)]
        torch.cuda.synchronize()
        got.append((fields, b.stats()["residual"]))
    for f, g in zip(got[0][0], got[1][0]):
        assert torch.equal(f, g)
    assert np.array_equal(got[0][1], got[1][1], equal_nan=True)
