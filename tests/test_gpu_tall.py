"""Lattices of more than 65535 rows (the largest launch grid in y) on the
automatic path, against one node per thread with blocks of 8 rows."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,bc,storage,fx", [
    (8, 70000, "periodic", "fp32", 0.0), (9, 65536, "channel", "fp32", 1e-6),
    (24, 70001, "periodic", "fp32", 0.0), (6, 65537, "cavity", "fp16", 0.0),
    (7, 131072, "periodic", "bf16", 0.0), (16, 65600, "periodic", "fp16", 0.0)])
def test_tall_lattice_on_the_automatic_path(nx, ny, bc, storage, fx):
    import torch
    from paper_1908_06742_gb300 import ddflb as D
    cfg = D.Config(nx=nx, ny=ny, bc=bc, storage=storage, fx=fx,
                   u_lid=0.05 if bc == "cavity" else 0.0)
    y = np.arange(ny, dtype=np.float64)[:, None] + 0.25 * np.arange(nx)[None, :]
    f = [np.ones((ny, nx)), 0.01 * np.sin(0.02 * y), 0.01 * np.cos(0.03 * y),
         1 + 0.1 * np.sin(0.05 * y)]
    out = []
    for path in (1, 0):
        lat = D.Lattice(cfg)
        D._check(lat.lib.ddflb_set_block(lat._h, 32, 8))
        lat.set_path(path)
        lat.init(*[a.astype(np.float32) for a in f])
        lat.step(3).step(4)  # (odd counts, so single steps remain beside two-step launches)
        out.append(torch.cat([p.reshape(-1) for p in lat.populations()]))
    torch.cuda.synchronize()
    assert torch.equal(out[0], out[1])
