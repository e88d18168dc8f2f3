"""Four time steps per launch (k_tile) with the central-moment scalar models
against the one-step kernel: bit-identical."""
import pytest

pytestmark = pytest.mark.gpu


# the smallest lattice, one edge beyond a tile, the largest of each tile shape
@pytest.mark.parametrize("storage", ["fp32", "fp16", "bf16"])
@pytest.mark.parametrize("bc", ["periodic", "cavity", "channel"])
@pytest.mark.parametrize("nx,ny", [(4, 4), (9, 5), (31, 33), (64, 64), (97, 96), (130, 100),
                                   (200, 180), (255, 256)])
def test_four_steps_match_single_steps(bc, storage, nx, ny):
    import torch
    from paper_1908_06742_gb300 import ddflb as D
    g = torch.Generator(device="cuda").manual_seed(nx + ny)
    r = lambda *s: torch.randn(*s, generator=g, device="cuda")
    f = 1 + 0.01 * r(ny, nx), 0.02 * r(ny, nx), 0.02 * r(ny, nx), 1 + 0.1 * r(ny, nx)
    field = 1e-5 * r(2, ny, nx)
    for model in ("cascaded", "central"):
        for force in (False, True):
            cfg = D.Config(nx=nx, ny=ny, bc=bc, storage=storage, nu=0.02, diffusivity=0.03,
                           u_lid=0.08, phi_lid=1.2, phi_wall=0.4, scalar_model=model)
            out = []
            for path in (0, 1):
                lat = D.Lattice(cfg).set_path(path)
                if force:
                    lat.set_force_field(field)
                lat.init(*f).step(75)
                out.append((*lat.populations(), lat.fields(names=("omega",))["omega"]))
            for x, y in zip(*out):
                assert torch.equal(torch.nan_to_num(x, nan=7.0), torch.nan_to_num(y, nan=7.0)), \
                    (model, force)
