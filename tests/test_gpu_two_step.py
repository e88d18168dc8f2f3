"""The two-steps-per-launch kernel of large lattices (k_march2) against the
one-node-per-thread kernel: the same arithmetic, so bit-identical.  Thin
lattices above its size limit reach the edges of its 60-column strips and of
its row chunks."""
import pytest

pytestmark = pytest.mark.gpu

NODES = 1 << 21  # the smallest lattice that takes two steps per launch


def _fields(torch, nx, ny, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    r = lambda: torch.randn(ny, nx, generator=g, device="cuda")
    return 1 + 0.01 * r(), 0.02 * r(), 0.02 * r(), 1 + 0.1 * r()


def _run(D, cfg, fields, path, steps):
    lat = D.Lattice(cfg).set_path(path).init(*fields)
    for n in steps:
        lat.step(n)
    return (*lat.populations(), lat.fields(names=("omega",))["omega"])


def _same(torch, a, b):
    return all(torch.equal(torch.nan_to_num(x, nan=7.0), torch.nan_to_num(y, nan=7.0))
               for x, y in zip(a, b))


SHAPES = [(40, 52500), (59, None), (60, None), (61, None), (62, None), (119, None), (121, None),
          (122, None), (190, None), (1 << 20, 2), (700001, 3), (300003, 7), (1025, 2049)]


@pytest.mark.parametrize("storage", ["fp32", "fp16", "bf16"])
@pytest.mark.parametrize("bc", ["periodic", "cavity", "channel"])
@pytest.mark.parametrize("nx,ny", SHAPES)
def test_two_steps_match_single_steps(bc, storage, nx, ny):
    import torch
    from paper_1908_06742_gb300 import ddflb as D
    ny = ny or -(-NODES // nx)
    cfg = D.Config(nx=nx, ny=ny, bc=bc, storage=storage, nu=0.02, diffusivity=0.03, u_lid=0.08,
                   phi_lid=1.2, phi_wall=0.4)
    f = _fields(torch, nx, ny, nx + ny)
    # two launches of two steps, one single step, then 64 steps as a graph
    assert _same(torch, _run(D, cfg, f, 0, (5,)), _run(D, cfg, f, 1, (5,)))
    if nx in (61, 121, 1025):
        assert _same(torch, _run(D, cfg, f, 0, (67,)), _run(D, cfg, f, 1, (67,)))


@pytest.mark.parametrize("storage", ["fp32", "fp16"])
def test_checks_and_srt(storage):
    """Launches of two steps stop at the residual checks (every 3 steps), and
    the SRT collision runs through the same kernel."""
    import torch
    from paper_1908_06742_gb300 import ddflb as D
    cfg = D.Config(nx=1537, ny=1400, storage=storage, scalar_model="srt", check_every=3)
    f = _fields(torch, 1537, 1400, 9)
    got = []
    for path in (0, 1):
        lat = D.Lattice(cfg).set_path(path).init(*f)
        lat.step(2).step(6)
        st = lat.stats()
        got.append((st["residual"], st["mass"], st["scalar"], st["step"], *lat.populations()))
    assert got[0][:4] == got[1][:4]
    assert _same(torch, got[0][4:], got[1][4:])
