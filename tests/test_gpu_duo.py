"""The single-step kernel with two nodes per thread and packed arithmetic
(k_step_duo) against the one-node-per-thread kernel: the same arithmetic, so
bit-identical; even and odd widths, rows and columns at the lattice's edges."""
import pytest

pytestmark = pytest.mark.gpu


def _fields(torch, nx, ny, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    r = lambda: torch.randn(ny, nx, generator=g, device="cuda")
    return 1 + 0.01 * r(), 0.02 * r(), 0.02 * r(), 1 + 0.1 * r()


def _run(D, cfg, fields, path, steps):
    lat = D.Lattice(cfg).set_path(path).init(*fields)
    for n in steps:
        lat.step(n)
    return (*lat.populations(), lat.fields(names=("omega",))["omega"])


# 4 is the narrowest that has enough rows; 1100 x 1200 alternates its direction
SHAPES = [(450, 450), (447, 449), (4, 60000), (5, 50001), (100001, 2), (66670, 3), (512, 401),
          (257, 800), (1023, 767), (1100, 1200)]


@pytest.mark.parametrize("storage", ["fp32", "fp16", "bf16"])
@pytest.mark.parametrize("bc", ["periodic", "cavity", "channel"])
@pytest.mark.parametrize("nx,ny", SHAPES)
def test_pairs_match_single_nodes(bc, storage, nx, ny):
    import torch
    from paper_1908_06742_gb300 import ddflb as D
    cfg = D.Config(nx=nx, ny=ny, bc=bc, storage=storage, nu=0.02, diffusivity=0.03, u_lid=0.08,
                   phi_lid=1.2, phi_wall=0.4, scalar_model="srt" if nx % 2 else "mrt")
    f = _fields(torch, nx, ny, nx + ny)
    for steps in ((3,), (66,)):
        a, b = _run(D, cfg, f, 0, steps), _run(D, cfg, f, 1, steps)
        assert all(torch.equal(torch.nan_to_num(x, nan=7.0), torch.nan_to_num(y, nan=7.0))
                   for x, y in zip(a, b))
