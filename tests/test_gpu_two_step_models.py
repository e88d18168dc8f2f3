"""Two time steps per launch (k_march2) with a uniform force and with the
central-moment scalar models (FP32) against the one-step kernel: bit-identical."""
import pytest

pytestmark = pytest.mark.gpu


# just above the smallest such lattices; odd widths, short and narrow ones
@pytest.mark.parametrize("bc", ["periodic", "cavity", "channel"])
@pytest.mark.parametrize("nx,ny", [(3201, 3202), (3600, 2801), (70001, 145), (161, 64001)])
def test_two_steps_match_single_steps(bc, nx, ny):
    import torch
    from paper_1908_06742_gb300 import ddflb as D
    g = torch.Generator(device="cuda").manual_seed(nx + ny)
    r = lambda *s: torch.randn(*s, generator=g, device="cuda")
    f = 1 + 0.01 * r(ny, nx), 0.02 * r(ny, nx), 0.02 * r(ny, nx), 1 + 0.1 * r(ny, nx)
    for model, fx in (("mrt", 2e-5), ("cascaded", 0.0), ("cascaded", 2e-5), ("central", 0.0),
                      ("central", 2e-5)):
        cfg = D.Config(nx=nx, ny=ny, bc=bc, nu=0.02, diffusivity=0.03, u_lid=0.08, phi_lid=1.2,
                       phi_wall=0.4, scalar_model=model, fx=fx, fy=-fx / 2)
        out = []
        for path in (0, 1):
            lat = D.Lattice(cfg).set_path(path).init(*f)
            lat.step(11)
            out.append((*lat.populations(), lat.fields(names=("omega",))["omega"]))
        for x, y in zip(*out):
            assert torch.equal(torch.nan_to_num(x, nan=7.0), torch.nan_to_num(y, nan=7.0)), \
                (model, fx)


def test_a_force_field_set_and_taken_away():
    import torch
    from paper_1908_06742_gb300 import ddflb as D
    nx, ny = 1751, 1752
    g = torch.Generator(device="cuda").manual_seed(5)
    r = lambda *s: torch.randn(*s, generator=g, device="cuda")
    f = 1 + 0.01 * r(ny, nx), 0.02 * r(ny, nx), 0.02 * r(ny, nx), 1 + 0.1 * r(ny, nx)
    field = 1e-5 * r(2, ny, nx)
    out = []
    for path in (0, 1):
        lat = D.Lattice(D.Config(nx=nx, ny=ny, bc="channel", nu=0.02, diffusivity=0.03,
                                 phi_lid=1.2, fx=2e-5)).set_path(path).init(*f)
        for field_now in (None, field, None):
            lat.set_force_field(field_now)
            lat.step(7)
        out.append(lat.populations())
    assert all(torch.equal(x, y) for x, y in zip(*out))
