"""The four-steps-per-launch kernel of small lattices (k_tile) against the
one-node-per-thread kernel: the same arithmetic, so bit-identical.  Sizes at the
edges of its tiles (8 x 4 to 32 x 14) and of the range it is used for."""
import pytest

pytestmark = pytest.mark.gpu


def _fields(torch, nx, ny, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    r = lambda: torch.randn(ny, nx, generator=g, device="cuda")
    return 1 + 0.01 * r(), 0.02 * r(), 0.02 * r(), 1 + 0.1 * r()


def _run(D, cfg, fields, path, steps, field=None):
    lat = D.Lattice(cfg).set_path(path).init(*fields)
    if field is not None:
        lat.set_force_field(field)
    for n in steps:
        lat.step(n)
    return (*lat.populations(), lat.fields(names=("omega",))["omega"])


def _same(torch, a, b):
    return all(torch.equal(torch.nan_to_num(x, nan=7.0), torch.nan_to_num(y, nan=7.0))
               for x, y in zip(a, b))


SHAPES = [(4, 4), (5, 4), (4, 7), (8, 4), (9, 5), (31, 33), (64, 64), (65, 63), (97, 96), (128, 129),
          (130, 100), (200, 180), (255, 256), (300, 210), (3000, 4), (4, 600)]


@pytest.mark.parametrize("storage", ["fp32", "fp16", "bf16"])
@pytest.mark.parametrize("bc", ["periodic", "cavity", "channel"])
@pytest.mark.parametrize("nx,ny", SHAPES)
def test_four_steps_match_single_steps(bc, storage, nx, ny):
    import torch
    from paper_1908_06742_gb300 import ddflb as D
    cfg = D.Config(nx=nx, ny=ny, bc=bc, storage=storage, nu=0.02, diffusivity=0.03, u_lid=0.08,
                   phi_lid=1.2, phi_wall=0.4)
    f = _fields(torch, nx, ny, nx + ny)
    # two launches, two single steps; then a graph of 64 steps and the rest
    for steps in ((10,), (75, 3)):
        assert _same(torch, _run(D, cfg, f, 0, steps), _run(D, cfg, f, 1, steps))


@pytest.mark.parametrize("bc", ["periodic", "cavity", "channel"])
@pytest.mark.parametrize("model", ["mrt", "srt"])
def test_with_force_field_and_checks(bc, model):
    import torch
    from paper_1908_06742_gb300 import ddflb as D
    nx, ny = 90, 101
    cfg = D.Config(nx=nx, ny=ny, bc=bc, scalar_model=model, fx=2e-5, fy=-1e-5, u_lid=0.05,
                   check_every=6)
    f = _fields(torch, nx, ny, 3)
    g = torch.Generator(device="cuda").manual_seed(4)
    field = 1e-5 * torch.randn(2, ny, nx, generator=g, device="cuda")
    assert _same(torch, _run(D, cfg, f, 0, (5, 20), field), _run(D, cfg, f, 1, (5, 20), field))
