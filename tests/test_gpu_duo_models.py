"""The two-nodes-per-thread kernel with a body force and with the central-moment
scalar models against the one-node-per-thread kernel: the same operations in the
same order, so bit-identical."""
import pytest

pytestmark = pytest.mark.gpu

MODELS = [("mrt", "const"), ("srt", "field"), ("mrt", "wave"), ("cascaded", None),
          ("cascaded", "const"), ("cascaded", "field"), ("central", None), ("central", "const"),
          ("central", "wave")]


def _inputs(torch, nx, ny, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    r = lambda *s: torch.randn(*s, generator=g, device="cuda")
    return (1 + 0.01 * r(ny, nx), 0.02 * r(ny, nx), 0.02 * r(ny, nx), 1 + 0.1 * r(ny, nx)), \
        1e-5 * r(2, ny, nx)


def _run(D, cfg, fields, field, path, steps):
    lat = D.Lattice(cfg).set_path(path)
    if field is not None:
        lat.set_force_field(field)
    lat.init(*fields)
    lat.step(steps)
    return (*lat.populations(), lat.fields(names=("omega",))["omega"])


# odd and even widths, blocks of 32, 64 and 128 pairs and one pair more, few columns
@pytest.mark.parametrize("storage", ["fp32", "fp16", "bf16"])
@pytest.mark.parametrize("bc", ["periodic", "cavity", "channel"])
@pytest.mark.parametrize("nx,ny", [(3, 40001), (64, 1800), (129, 900), (257, 450), (258, 440),
                                   (350, 350), (701, 613), (1100, 1200)])
def test_models_match_single_nodes(bc, storage, nx, ny):
    import torch
    from paper_1908_06742_gb300 import ddflb as D
    f, ff = _inputs(torch, nx, ny, nx + ny)
    for model, force in MODELS:
        if bc == "cavity" and force is not None and nx > 300:
            continue
        cfg = D.Config(nx=nx, ny=ny, bc=bc, storage=storage, nu=0.02, diffusivity=0.03, u_lid=0.08,
                       phi_lid=1.2, phi_wall=0.4, scalar_model=model,
                       fx=2e-5 if force else 0.0, fy=-1e-5 if force else 0.0,
                       force_omega=0.1 if force == "wave" else 0.0)
        field = ff if force == "field" else None
        a, b = (_run(D, cfg, f, field, path, 21) for path in (0, 1))
        for x, y in zip(a, b):
            assert torch.equal(torch.nan_to_num(x, nan=7.0), torch.nan_to_num(y, nan=7.0)), \
                (model, force)
