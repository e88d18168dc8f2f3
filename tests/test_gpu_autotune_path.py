"""The autotuner times the automatic path too; whatever it keeps gives the same state."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,storage,model,fx", [
    (64, 64, "fp32", "mrt", 0.0), (50, 70, "bf16", "cascaded", 1e-5), (501, 400, "fp16", "mrt", 0.0),
    (640, 480, "fp32", "central", 1e-5), (1300, 1200, "fp32", "mrt", 0.0)])
def test_tuned_matches_one_node(nx, ny, storage, model, fx):
    import torch
    from paper_1908_06742_gb300 import ddflb as D
    g = torch.Generator(device="cuda").manual_seed(nx)
    r = lambda: torch.randn(ny, nx, generator=g, device="cuda")
    f = 1 + 0.01 * r(), 0.02 * r(), 0.02 * r(), 1 + 0.1 * r()
    cfg = D.Config(nx=nx, ny=ny, bc="channel", storage=storage, nu=0.02, diffusivity=0.03,
                   scalar_model=model, fx=fx)
    tuned = D.Lattice(cfg)
    rec = tuned.autotune(trial_steps=9, cache=False)
    assert rec["choice"][2] in (0, 1, 2, 3) and rec["ms_per_step"] > 0
    tuned.init(*f).step(13)
    plain = D.Lattice(cfg).set_path(1).init(*f)
    plain.step(13)
    assert all(torch.equal(a, b) for a, b in zip(tuned.populations(), plain.populations()))
