"""A bulk copy of a two-step launch that does not arrive in time: the kernel sets a
status word, here set from the host.  The steps then leave the state alone and the
calls that synchronise report it, until the state is initialised again."""
import struct

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _fields(nx, ny):
    y, x = np.meshgrid(np.arange(ny) / ny, np.arange(nx) / nx, indexing="ij")
    f = [np.ones((ny, nx)), 0.01 * np.sin(2 * np.pi * x), 0.01 * np.cos(2 * np.pi * y),
         1 + 0.1 * np.sin(2 * np.pi * (x + y))]
    return [a.astype(np.float32) for a in f]


@pytest.mark.parametrize("nx,ny,storage", [(64, 64, "fp32"), (400, 301, "fp16"),
                                           (1500, 1400, "fp32"), (1024, 1024, "bf16")])
def test_lattice(nx, ny, storage):
    import torch
    from paper_1908_06742_gb300 import ddflb as D
    lat = D.Lattice(D.Config(nx=nx, ny=ny, storage=storage, host_io=False))
    lat.init(*_fields(nx, ny)).step(4)
    before = [p.clone() for p in lat.populations()]
    # the status block (5 doubles, then the stop bits) ends the workspace
    lat.workspace[-256:].view(torch.int32)[10] = 2
    lat.step(8)
    for a, b in zip(before, lat.populations()):
        assert torch.equal(a, b)
    for call in (lat.stats, lat.sums):
        with pytest.raises(D.DdflbError, match="bulk copy"):
            call()
    lat.init(*_fields(nx, ny)).step(4)
    assert lat.stats()["step"] == 4
    for a, b in zip(before, lat.populations()):
        assert torch.equal(a, b)


def test_host_fields_report_it():
    import torch
    from paper_1908_06742_gb300 import ddflb as D
    lat = D.Lattice(D.Config(nx=64, ny=64, host_io=True))
    lat.init(*_fields(64, 64)).step(2)
    out = [torch.empty(64, 64).pin_memory() for _ in range(8)]
    host = lambda: lat.lib.ddflb_fields_host(lat._h, *[t.data_ptr() for t in out])
    assert host() == D.OK
    io = (10 + 8) * 64 * 64 * 4  # staging areas after the status block
    lat.workspace[-256 - io:-io].view(torch.int32)[10] = 2
    assert host() == D.ETIMEOUT


@pytest.mark.parametrize("schedule", [0, 1])
def test_batch_instance(schedule):
    import torch
    from paper_1908_06742_gb300 import ddflb as D
    cfgs = [D.Config(nx=n, ny=n + 2, bc="cavity", u_lid=0.05, check_every=10) for n in (66, 70)]
    make = lambda: D.Batch(cfgs).set_schedule(schedule).set_run(tol=1e-30, steps_per_launch=9)
    b, ref = make(), make()
    for x in (b, ref):
        for i, c in enumerate(cfgs):
            x.init(i, *_fields(c.nx, c.ny))
            x.set_instance_run(i, tol=0.123456789 if i == 0 else -1.0)
        x.step(8)
    # instance 0's status: its flags stand 8 bytes before its tolerance
    raw = bytes(b.workspace.cpu().numpy())
    at = raw.index(struct.pack("<d", 0.123456789)) - 8
    assert raw[at:at + 4] == b"\0\0\0\0"
    b.workspace[at:at + 4].view(torch.int32)[0] = D.INST_LOST
    for x in (b, ref):
        x.step(30)
    st = b.stats()
    assert st["status"] == D.ETIMEOUT and "bulk copy" in b.lib.ddflb_last_error().decode()
    assert st["flags"][0] == D.INST_LOST and st["flags"][1] == 0
    with pytest.raises(D.DdflbError, match="bulk copy"):
        b.fields(0)
    for k, v in ref.fields(1).items():
        assert torch.equal(v, b.fields(1)[k])
    b.init(0, *_fields(cfgs[0].nx, cfgs[0].ny)).step(3)
    assert b.stats()["status"] == D.OK
    b.fields(0)
