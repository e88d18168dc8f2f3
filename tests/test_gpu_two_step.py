"""The two-steps-per-launch kernel of large lattices (k_march2) against the
one-node-per-thread kernel: the same arithmetic, so bit-identical.  Thin
lattices above its size limit reach the edges of its 60-column strips and of
its row chunks."""
import pytest

pytestmark = pytest.mark.gpu

# lattices large enough to take two steps per launch, by storage
NODES = {"fp32": 1 << 21, "fp16": 10_100_000, "bf16": 10_100_000}


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


WIDTHS = {"fp32": (40, 59, 60, 61, 62, 119, 121, 122, 190), "fp16": (179, 180, 181, 182, 242),
          "bf16": (239, 240, 241, 245)}
HEIGHTS = (2, 3, 7, 2049)


@pytest.mark.parametrize("bc", ["periodic", "cavity", "channel"])
@pytest.mark.parametrize("storage,nx,ny", [(s, w, -(-NODES[s] // w)) for s in WIDTHS
                                           for w in WIDTHS[s]]
                         + [(s, NODES[s] // h + 1, h) for s in WIDTHS for h in HEIGHTS])
def test_two_steps_match_single_steps(bc, storage, nx, ny):
    import torch
    from paper_1908_06742_gb300 import ddflb as D
    cfg = D.Config(nx=nx, ny=ny, bc=bc, storage=storage, nu=0.02, diffusivity=0.03, u_lid=0.08,
                   phi_lid=1.2, phi_wall=0.4)
    f = _fields(torch, nx, ny, nx + ny)
    # two launches of two steps, one single step; at a few sizes also a graph of 64
    for steps in ((5,), (67,)) if nx in (61, 121, 181, 241) else ((5,),):
        assert _same(torch, _run(D, cfg, f, 0, steps), _run(D, cfg, f, 1, steps))


@pytest.mark.parametrize("storage", ["fp32", "fp16"])
def test_checks_and_srt(storage):
    """Launches of two steps stop at the residual checks (every 3 steps), and
    the SRT collision runs through the same kernel."""
    import torch
    from paper_1908_06742_gb300 import ddflb as D
    cfg = D.Config(nx=1537, ny=NODES[storage] // 1537 + 1, storage=storage, scalar_model="srt", check_every=3)
    f = _fields(torch, cfg.nx, cfg.ny, 9)
    got = []
    for path in (0, 1):
        lat = D.Lattice(cfg).set_path(path).init(*f)
        lat.step(2).step(6)
        st = lat.stats()
        got.append((st["residual"], st["mass"], st["scalar"], st["step"], *lat.populations()))
    assert got[0][:4] == got[1][:4]
    assert _same(torch, got[0][4:], got[1][4:])
