"""An autotuner trial that fails to launch leaves the path and the block as they were."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_failed_trial_keeps_path_and_block():
    import torch
    from paper_1908_06742_gb300 import ddflb as D
    # a trial with blocks of one row has more than 65535 of them: refused at launch
    nx, ny = 32, 70000
    y = np.arange(ny, dtype=np.float64)[:, None] + np.zeros((1, nx))
    f = [np.ones((ny, nx)), 0.01 * np.sin(0.02 * y), 0.01 * np.cos(0.03 * y), 1 + 0 * y]
    f = [a.astype(np.float32) for a in f]
    out = []
    for tuned in (False, True):
        lat = D.Lattice(D.Config(nx=nx, ny=ny))
        D._check(lat.lib.ddflb_set_block(lat._h, 32, 8))
        lat.set_path(1)
        if tuned:
            with pytest.raises(D.DdflbError):
                lat.autotune(trial_steps=2, cache=False)
        lat.init(*f).step(4)
        out.append(torch.cat([p.reshape(-1) for p in lat.populations()]))
        torch.cuda.synchronize()
    assert torch.equal(*out)
