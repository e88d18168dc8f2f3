"""The kernel that the automatic path takes, on either side of its rules."""
import pytest

pytestmark = pytest.mark.gpu

RULES = [
    ((256, 256, "cavity", "fp32"), ("k_tile", 4)), ((257, 257, "cavity", "fp32"), ("k_step", 1)),
    ((3, 151, "channel", "fp16"), ("k_step", 1)), ((20, 20000, "periodic", "fp32"), ("k_step", 1)),
    ((33, 4000, "periodic", "fp32"), ("k_step_duo", 1)),
    ((66, 6060, "periodic", "fp32"), ("k_step", 1)), ((97, 4000, "periodic", "fp32"), ("k_step_duo", 1)),
    ((8, 60000, "periodic", "bf16"), ("k_step", 1)), ((40, 65535, "periodic", "fp32"), ("k_step_duo", 1)),
    ((40, 65536, "periodic", "fp32"), ("k_step", 1)), ((42, 65536, "periodic", "fp16"), ("k_step_pair", 1)),
    ((1024, 1024, "periodic", "fp32"), ("k_step_duo", 1)),
    ((1024, 1024, "periodic", "fp16"), ("k_step_quad", 1)),
    ((1200, 1200, "periodic", "fp32"), ("k_march2", 2)),
    ((64, 25000, "periodic", "fp32"), ("k_step_duo", 1)),
    ((128, 31250, "cavity", "fp32"), ("k_step_duo", 1)),
    ((180, 22222, "channel", "fp32"), ("k_march2", 2)),
    ((2000, 2000, "channel", "fp16"), ("k_step_quad", 1)),
    ((2001, 2000, "channel", "fp16"), ("k_step_duo", 1)),
    ((1600, 1600, "channel", "fp16"), ("k_step_duo", 1)),
    ((2048, 2048, "cavity", "bf16"), ("k_step_duo", 1)),
    ((16000, 250, "cavity", "bf16"), ("k_step_quad", 1)),
    ((2500, 2500, "channel", "bf16"), ("k_step_quad", 1)),
    ((3000, 3000, "channel", "bf16"), ("k_march2", 2)),
    ((256, 46875, "channel", "bf16"), ("k_step_quad", 1))]


@pytest.mark.parametrize("shape,want", RULES)
def test_automatic_path(shape, want):
    from paper_1908_06742_gb300 import ddflb as D
    nx, ny, bc, storage = shape
    lat = D.Lattice(D.Config(nx=nx, ny=ny, bc=bc, storage=storage,
                             u_lid=0.05 if bc == "cavity" else 0.0))
    assert lat.step_kernel() == want
    assert lat.set_path(1).step_kernel() == ("k_step", 1)
    assert lat.set_path(0).step_kernel() == want


@pytest.mark.parametrize("n,size,want", [(4, 64, 1), (256, 64, 2), (16, 256, 1), (32, 256, 2)])
def test_batch(n, size, want):
    from paper_1908_06742_gb300 import ddflb as D
    b = D.Batch([D.Config(nx=size, ny=size, bc="cavity", u_lid=0.05) for _ in range(n)])
    b.set_run(steps_per_launch=77)
    assert b.steps_per_launch() == 77
    assert b.set_schedule(1).steps_per_launch() == want
