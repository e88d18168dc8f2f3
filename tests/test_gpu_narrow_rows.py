"""Lattices on either side of the rules on the width of a row: the automatic path
against one node per thread, bit for bit."""
import pytest

pytestmark = pytest.mark.gpu

SHAPES = [(3, 151), (31, 4000), (32, 3600), (33, 3500), (64, 1800), (65, 1800), (96, 1200),
          (97, 1200), (64, 25000), (64, 60000), (128, 12500), (200, 8000), (180, 8888),
          (300, 27000), (256, 46875), (2000, 1500), (1999, 1501), (8192, 367), (8188, 367)]


@pytest.mark.parametrize("nx,ny", SHAPES)
@pytest.mark.parametrize("bc", ["periodic", "cavity", "channel"])
@pytest.mark.parametrize("storage,model,fx", [("fp32", "mrt", 0.0), ("bf16", "mrt", 0.0),
                                              ("fp32", "cascaded", 0.0), ("fp16", "mrt", 1e-6)])
def test_automatic_path(nx, ny, bc, storage, model, fx):
    import torch
    from paper_1908_06742_gb300 import ddflb as D
    if bc == "cavity" and fx:
        fx, model = 0.0, "central"
    cfg = D.Config(nx=nx, ny=ny, bc=bc, storage=storage, scalar_model=model, fx=fx,
                   u_lid=0.05 if bc == "cavity" else 0.0)
    g = torch.Generator(device="cuda").manual_seed(nx + ny)
    r = lambda: torch.randn(ny, nx, generator=g, device="cuda")
    f = (1 + 0.01 * r(), 0.02 * r(), 0.02 * r(), 1 + 0.1 * r())
    out = []
    for path in (1, 0):
        lat = D.Lattice(cfg).set_path(path).init(*f).step(9)
        out.append(lat.populations())
    for a, b in zip(*out):
        assert torch.equal(a, b)
