"""What a user of the framework has it do, as cases that can be timed and checked.

Three kinds of work:

* ``lattice``: one double-distribution lattice, from its initial fields through
  a number of fused time steps to its local fields (u, phi, S, omega): init,
  step, fields, as in the README's example.
* ``batch``: many lid-driven cavities of uneven sizes advanced together.
* the warm-start network: ``unet_train`` (forward, loss and all gradients of
  one minibatch), ``unet_predict`` (whole-batch inference) and ``conv3x3``
  (one convolution layer through the library's entry point).

``exact`` restates the method (Hajabdollahi & Premnath, arXiv 1908.06742,
Secs. 2-5, Apps. C and D) and the network in plain FP64 torch.
"""
from __future__ import annotations

import math

import torch

from paper_1908_06742_gb300 import ddflb as D
from paper_1908_06742_gb300 import surrogate as S

DEV = "cuda"
C3 = 1.0 / 3.0
SIZES = (64, 96, 128, 192, 256, 384, 512)   # cavity sizes of the batched workload
NAMES = ("rho", "ux", "uy", "phi", "sxx", "sxy", "syy", "omega")


def _lat(name, bc, nx, ny, storage, steps, model="mrt", force=False, check=0):
    c = dict(kind="lattice", bc=bc, nx=nx, ny=ny, storage=storage, steps=steps, model=model,
             force=force, check=check)
    return dict(name=name, **c) if name else c


def listed():
    return [
        # the smallest run: the 64^2 Taylor-Green validation flow, 1000 steps (launch-bound)
        _lat("taylor_green_64_fp32", "periodic", 64, 64, "fp32", 1000),
        # a steady-state cavity run, residual check and field output every 1000 steps
        _lat("cavity_256_fp32", "cavity", 256, 256, "fp32", 1000, check=1000),
        # pressure-driven channel, cascaded scalar collision, odd non-square size
        _lat("channel_1021x509_fp32", "channel", 1021, 509, "fp32", 200, model="cascaded", force=True),
        # the throughput sweep's smallest size (about as large as L2)
        _lat("taylor_green_1024_fp32", "periodic", 1024, 1024, "fp32", 200),
        # 16-bit storage at a ragged size, where no wide access lines up
        _lat("periodic_1023x767_fp16", "periodic", 1023, 767, "fp16", 200),
        # 16-bit storage with walls on all sides
        _lat("cavity_2048_bf16", "cavity", 2048, 2048, "bf16", 200),
        # the throughput sweep proper: populations far larger than L2
        _lat("taylor_green_8192_fp32", "periodic", 8192, 8192, "fp32", 200),
        # its largest size, in 16-bit storage
        _lat("taylor_green_16384_fp16", "periodic", 16384, 16384, "fp16", 100),
        # training data and parameter studies: 512 uneven cavities, one default chunk of steps
        dict(name="cavities_batch_512", kind="batch", n=512, storage="fp32", steps=500),
        # one minibatch of the warm-start network's training (forward, loss, gradients)
        dict(name="unet_train_128", kind="unet_train", size=128, batch=16, width=32),
        # prediction for a whole batch at the production grid size
        dict(name="unet_predict_256", kind="unet_predict", size=256, batch=16, width=32),
        # a single convolution layer of the network (level 1, 64 -> 64 channels)
        dict(name="conv3x3_128_64to64", kind="conv3x3", size=128, batch=16, cin=64, cout=64),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["lattice"] * 7 + ["batch"] * 2 + ["unet_train", "unet_predict", "conv3x3"])
    if kind == "lattice":
        nx = _log(rng, 64, 8192)
        ny = min(8192, max(48, int(nx * math.exp(rng.uniform(math.log(0.5), math.log(2.0))))))
        if rng.random() < 0.5:  # half of the sizes are multiples of 4, the others anything
            nx = (nx + 3) // 4 * 4
        # 1000 steps of small lattices, down to 50 of the largest
        steps = max(50, min(1000, int(6.0e9 / (nx * ny))))
        bc = rng.choice(["periodic", "cavity", "channel"])
        storage = rng.choice(["fp32", "fp32", "fp16", "bf16"])
        model = rng.choice(["mrt", "mrt", "mrt", "srt", "cascaded", "central"])
        force = bc != "cavity" and rng.random() < 0.4
        return _lat(None, bc, nx, ny, storage, steps, model, force,
                    check=rng.choice([0, 0, max(1, steps // rng.randint(1, 3))]))
    if kind == "batch":
        return dict(kind="batch", n=_log(rng, 4, 300), storage=rng.choice(["fp32", "fp32", "bf16"]),
                    steps=rng.choice([200, 300, 500]))
    if kind == "conv3x3":
        return dict(kind="conv3x3", size=rng.choice([32, 64, 128, 256]), batch=rng.choice([4, 8, 16]),
                    cin=rng.choice([64, 128, 256]), cout=rng.choice([32, 64, 96, 128]))
    return dict(kind=kind, size=rng.choice([64, 96, 128, 192]), batch=rng.choice([4, 8, 12, 16]),
                width=rng.choice([16, 32]))


# ------------------------------------------------------------------ inputs
def _gen(seed):
    return torch.Generator().manual_seed(1000003 * int(seed) + 17)


def _u(g, lo, hi):
    return lo + (hi - lo) * float(torch.rand((), generator=g, dtype=torch.float64))


def _omega(nu):
    return 1.0 / (3.0 * nu + 0.5)


def _lattice_params(case, seed):
    """Rates, walls and force of a lattice case, drawn from the seed."""
    g = _gen(seed)
    p = dict(b1=1.0, b2=0.9, rho0=1.0, phi0=1.0, u_lid=0.0, phi_lid=1.0, phi_wall=0.0, fx=0.0)
    if case["bc"] == "cavity":
        # Re log-uniform in [100, 3200], Pe = Re
        p["u_lid"] = _u(g, 0.05, 0.1)
        re = math.exp(_u(g, math.log(100.0), math.log(3200.0)))
        nu = max(p["u_lid"] * case["nx"] / re, 0.004)
        dif = nu
    else:
        nu, dif = _u(g, 0.008, 0.03), _u(g, 0.008, 0.03)
    if case["force"]:
        p["fx"] = _u(g, 1e-6, 5e-6)
    w, wp = _omega(nu), _omega(dif)
    p["wf"] = (0.0, 0.0, 0.0, 1.2, w, w, 1.2, 1.2, 1.2)
    p["wg"] = (0.0, wp, wp, 1.2, 1.2, 1.2, 1.2, 1.2, 1.2)
    p["u0"], p["amp"] = _u(g, 0.008, 0.02), _u(g, 0.05, 0.15)
    p["sx"], p["sy"] = _u(g, 0.0, 1.0), _u(g, 0.0, 1.0)
    p["start"] = _u(g, 0.3, 0.7)  # initial scalar of a walled lattice
    return p


def _lattice_fields(case, p):
    """FP32 initial fields on the device: rho, ux, uy, phi, and the gradients."""
    nx, ny = case["nx"], case["ny"]
    f64 = dict(dtype=torch.float64, device=DEV)
    if case["bc"] != "periodic":
        # fluid at rest with a uniform scalar
        one = torch.ones(ny, nx, dtype=torch.float32, device=DEV)
        zero = torch.zeros_like(one)
        uy, phi = zero.clone(), one * p["start"]
        if case["bc"] == "channel":  # a wave along the channel, zero on its walls
            x = (torch.arange(nx, **f64) * (2 * math.pi / nx) + 2 * math.pi * p["sx"]).sin()[None, :]
            y = ((torch.arange(ny, **f64) + 0.5) * (math.pi / ny)).sin()[:, None]
            uy, phi = (p["u0"] * x * y).float(), (p["start"] * (1 + p["amp"] * x * y)).float()
        return one, zero, uy, phi, None
    # decaying Taylor-Green vortex at a phase of its own, with exact gradients
    kx, ky, u0, amp = 2 * math.pi / nx, 2 * math.pi / ny, p["u0"], p["amp"]
    x = (torch.arange(nx, **f64) * kx + 2 * math.pi * p["sx"])[None, :]
    y = (torch.arange(ny, **f64) * ky + 2 * math.pi * p["sy"])[:, None]
    cx, sx, cy, sy = x.cos(), x.sin(), y.cos(), y.sin()
    rho = 1.0 - 0.75 * u0 * u0 * ((2 * x).cos() + (2 * y).cos())
    out = [rho.float(), (-u0 * cx * sy).float(), (u0 * sx * cy).float(), (1.0 + amp * sx * sy).float()]
    grads = torch.empty(6, ny, nx, dtype=torch.float32, device=DEV)
    for k, v in enumerate(((u0 * kx * sx, sy), (-u0 * ky * cx, cy), (u0 * kx * cx, cy),
                           (-u0 * ky * sx, sy), (amp * kx * cx, sy), (amp * ky * sx, cy))):
        grads[k] = (v[0] * v[1]).float()
    return (*out, grads)


def _batch_params(case, seed):
    """Sizes uniform over SIZES, Re log-uniform in [100, 3200], Pe = Re."""
    g = _gen(seed)
    # the sizes are the case's own (another seed is other flows on the same grids)
    sizes = torch.randint(0, len(SIZES), (case["n"],), generator=_gen(7), dtype=torch.int64).tolist()
    out = []
    for k in sizes:
        n, u = SIZES[k], _u(g, 0.05, 0.1)
        re = math.exp(_u(g, math.log(100.0), math.log(3200.0)))
        w = _omega(u * n / re)
        out.append(dict(n=n, u_lid=u, start=_u(g, 0.3, 0.7), b1=1.0, b2=0.9, rho0=1.0, phi0=1.0,
                        phi_lid=1.0, phi_wall=0.0, fx=0.0,
                        wf=(0.0, 0.0, 0.0, 1.2, w, w, 1.2, 1.2, 1.2),
                        wg=(0.0, w, w, 1.2, 1.2, 1.2, 1.2, 1.2, 1.2)))
    return out


def _config(p, **kw):
    return D.Config(omega_f=p["wf"], omega_g=p["wg"], beta1=p["b1"], beta2=p["b2"], rho0=p["rho0"],
                    phi0=p["phi0"], u_lid=p["u_lid"], phi_lid=p["phi_lid"], phi_wall=p["phi_wall"],
                    fx=p["fx"], **kw)


def _net_specs(c, cin=16, cout=8):
    return [("e1a", cin, c), ("e1b", c, c), ("e2a", c, 2 * c), ("e2b", 2 * c, 2 * c),
            ("e3a", 2 * c, 4 * c), ("e3b", 4 * c, 4 * c), ("b1", 4 * c, 4 * c), ("b2", 4 * c, 4 * c),
            ("d3a", 8 * c, 4 * c), ("d3b", 4 * c, 2 * c), ("d2a", 4 * c, 2 * c), ("d2b", 2 * c, c),
            ("d1a", 2 * c, c), ("d1b", c, c), ("head", c, cout)]


def _net_weights(case, seed):
    """FP32 master weights of a network a program would load: He-scaled normals."""
    g = torch.Generator(device=DEV).manual_seed(1000003 * int(seed) + 29)
    out = {}
    for name, ci, co in _net_specs(case["width"]):
        k = ci if name == "head" else 9 * ci
        std = math.sqrt((1.0 if name == "head" else 2.0) / k)
        out[name] = (torch.randn(co, k, generator=g, device=DEV) * std,
                     torch.randn(co, generator=g, device=DEV) * 0.01)
    return out


def _net_batch(case, seed):
    """Input planes (parameters and coordinates) and smooth steady-like targets."""
    g = torch.Generator(device=DEV).manual_seed(1000003 * int(seed) + 31)
    B, n = case["batch"], case["size"]
    x = torch.zeros(B, n, n, 16, device=DEV)
    x[..., :3] = (torch.rand(B, 1, 1, 3, generator=g, device=DEV) * 2 - 1)
    s = (torch.arange(n, device=DEV) + 0.5) / n * 2 - 1
    x[..., 3], x[..., 4] = s[None, None, :], s[None, :, None]
    t = torch.zeros(B, n, n, 8, device=DEV)
    a = torch.randn(B, 5, generator=g, device=DEV)
    for ch in range(5):
        t[..., ch] = a[:, ch, None, None] * (torch.cos((1 + ch % 3) * math.pi * s)[None, None, :]
                                              * torch.sin((1 + ch // 2) * math.pi * s)[None, :, None])
    return x.to(torch.bfloat16), t


def _conv_inputs(case, seed):
    g = torch.Generator(device=DEV).manual_seed(1000003 * int(seed) + 37)
    B, n, ci, co = case["batch"], case["size"], case["cin"], case["cout"]
    x = torch.randn(B, n, n, ci, generator=g, device=DEV).to(torch.bfloat16)
    w = (torch.randn(co, 9 * ci, generator=g, device=DEV) * math.sqrt(2.0 / (9 * ci))).to(torch.bfloat16)
    return x, w, torch.randn(co, generator=g, device=DEV) * 0.01


def prepare(case, seed):
    kind = case["kind"]
    if kind == "lattice":
        p = _lattice_params(case, seed)
        cfg = _config(p, nx=case["nx"], ny=case["ny"], bc=case["bc"], storage=case["storage"],
                      scalar_model=case["model"], check_every=case["check"])
        return dict(case=case, lat=D.Lattice(cfg), fields=_lattice_fields(case, p))
    if kind == "batch":
        ps = _batch_params(case, seed)
        b = D.Batch([_config(p, nx=p["n"], ny=p["n"], bc="cavity", storage=case["storage"],
                             check_every=1000) for p in ps])
        b.set_run(tol=0.0, steps_per_launch=case["steps"])
        b.autotune(trial_steps=4, cache=False)
        rest = {}
        for n in set(p["n"] for p in ps):
            one = torch.ones(n, n, device=DEV)
            rest[n] = (one, torch.zeros_like(one))
        fields = [(*rest[p["n"]], rest[p["n"]][1], rest[p["n"]][0] * p["start"]) for p in ps]
        return dict(case=case, batch=b, fields=fields)
    if kind == "conv3x3":
        x, w, b = _conv_inputs(case, seed)
        y = torch.empty(*x.shape[:3], case["cout"], dtype=torch.bfloat16, device=DEV)
        return dict(case=case, x=x, w=w, b=b, y=y, lib=D.load())
    net = S.UNet(c=case["width"], batch=case["batch"], H=case["size"], W=case["size"], device=DEV)
    for name, (w, b) in _net_weights(case, seed).items():
        net.p[name]["w"].copy_(w)
        net.p[name]["wb"].copy_(w)
        net.p[name]["b"].copy_(b)
    x, t = _net_batch(case, seed)
    return dict(case=case, net=net, x=x, t=t)


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "lattice":
        lat = state["lat"]
        lat.init(*state["fields"])
        lat.step(case["steps"])
        return lat.fields()
    if kind == "batch":
        b = state["batch"]
        for i, f in enumerate(state["fields"]):
            b.init(i, *f)
        b.step(case["steps"])
        got = [b.fields(i, names=("ux", "uy", "phi", "omega")) for i in range(case["n"])]
        return {k: torch.cat([f[k].reshape(-1) for f in got]) for k in ("ux", "uy", "phi", "omega")}
    if kind == "conv3x3":
        x, y, n, lib = state["x"], state["y"], case["size"], state["lib"]
        st = lib.ddflb_nn_conv3x3(x.data_ptr(), case["batch"], n, n, case["cin"], case["cin"],
                                  state["w"].data_ptr(), case["cout"], None, 0, y.data_ptr(),
                                  case["cout"], state["b"].data_ptr(), 1, 0,
                                  torch.cuda.current_stream().cuda_stream)
        if st != D.OK:
            raise RuntimeError(lib.ddflb_last_error().decode())
        return y
    net = state["net"]
    if kind == "unet_predict":
        return S.predict(net, state["x"])
    out = net.forward(state["x"])
    loss = net.backward(state["t"])
    got = {"out": out, "loss": loss.float()}
    for name in net.p:
        got[name + ".w"], got[name + ".b"] = net.p[name]["gw"], net.p[name]["gb"]
    return got


# What the path cannot do without.  A lattice pass reads the initial fields and
# writes the result fields once; in between it does, per node and step, about
# 250 floating-point operations (two moment transforms, two collisions and the
# back transforms).  The network reads its inputs and weights and writes its
# results once; its operations are those of its convolutions.
FLOPS_PER_NODE_STEP = 250


def _net_macs(case):
    lv = dict(e1a=0, e1b=0, e2a=1, e2b=1, e3a=2, e3b=2, b1=3, b2=3, d3a=2, d3b=2, d2a=1, d2b=1,
              d1a=0, d1b=0, head=0)
    px = case["batch"] * case["size"] ** 2
    return sum(px // 4 ** lv[n] * ci * co * (1 if n == "head" else 9)
               for n, ci, co in _net_specs(case["width"]))


def work(case):
    kind = case["kind"]
    if kind == "lattice":
        cells = case["nx"] * case["ny"]
        planes_in = 10 if case["bc"] == "periodic" else 4
        return {"bytes": 4 * cells * (planes_in + 8),
                "flops": FLOPS_PER_NODE_STEP * cells * case["steps"]}
    if kind == "batch":
        cells = sum(p["n"] ** 2 for p in _batch_params(case, 0))
        return {"bytes": 4 * cells * (4 + 4), "flops": FLOPS_PER_NODE_STEP * cells * case["steps"]}
    if kind == "conv3x3":
        px = case["batch"] * case["size"] ** 2
        return {"bytes": 2 * px * (case["cin"] + case["cout"]) + 18 * case["cin"] * case["cout"],
                "flops": 18 * px * case["cin"] * case["cout"]}
    px, weights = case["batch"] * case["size"] ** 2, sum(
        ci * co * (1 if n == "head" else 9) for n, ci, co in _net_specs(case["width"]))
    if kind == "unet_predict":
        return {"bytes": px * (32 + 32) + 2 * weights, "flops": 2 * _net_macs(case)}
    return {"bytes": px * (32 + 32 + 32) + 6 * weights, "flops": 6 * _net_macs(case)}


# ------------------------------------------------------------------ FP64 restatement
EX = (0, 1, 0, -1, 0, 1, -1, -1, 1)
EY = (0, 0, 1, 0, -1, 1, 1, -1, -1)
OPP = (0, 3, 4, 1, 2, 7, 8, 5, 6)
W9 = (4 / 9, 1 / 9, 1 / 9, 1 / 9, 1 / 9, 1 / 36, 1 / 36, 1 / 36, 1 / 36)


def _basis():
    x = torch.tensor(EX, dtype=torch.float64, device=DEV)
    y = torch.tensor(EY, dtype=torch.float64, device=DEV)
    return torch.stack([torch.ones_like(x), x, y, x * x + y * y, x * x - y * y, x * y, x * x * y,
                        x * y * y, x * x * y * y])


class _Flow:
    """G lattices of one size and boundary kind, [G, 9, ny, nx] populations."""

    def __init__(self, ps, bc, model):
        col = lambda k: torch.tensor([p[k] for p in ps], dtype=torch.float64, device=DEV).view(-1, 1, 1)
        rates = lambda k: torch.tensor([p[k] for p in ps], dtype=torch.float64, device=DEV).view(-1, 9, 1, 1)
        self.bc, self.cm = bc, model in ("cascaded", "central")
        self.wf, self.wg = rates("wf"), rates("wg")
        if model == "srt":  # one rate for every non-conserved scalar moment
            self.wg = self.wg.clone()
            self.wg[:, 1:] = self.wg[:, 1:2]
        self.b1, self.b2, self.fx = col("b1"), col("b2"), col("fx")
        self.u_lid, self.phi_lid, self.phi_wall, self.rho0 = (col("u_lid"), col("phi_lid"),
                                                              col("phi_wall"), col("rho0"))
        self.forced = any(p["fx"] != 0.0 for p in ps)
        self.M = _basis()
        self.Mi = torch.linalg.inv(self.M)

    def _to(self, A, f):
        return torch.einsum("ij,gjyx->giyx", A, f)

    def _eq(self, a, ux, uy, third, fourth):
        xx, yy = ux * ux, uy * uy
        return torch.stack([a, a * ux, a * uy, a * (2 * C3 + xx + yy), a * (xx - yy), a * ux * uy,
                            a * uy * (third[0] * C3 + xx), a * ux * (third[1] * C3 + yy),
                            a * (C3 * C3 + C3 * (xx + yy) + xx * yy + fourth)], 1)

    def eq_f(self, rho, ux, uy):
        return self._eq(rho, ux, uy, (1.0, 1.0), 0.0)

    def eq_g(self, phi, ux, uy):
        # the central-moment models' equilibrium is larger in the fourth order
        more = 2 * C3 * ((self.b2 - 1) * ux * ux + (self.b1 - 1) * uy * uy) if self.cm else 0.0
        return self._eq(phi, ux, uy, (self.b1, self.b2), more)

    def source(self, ux, uy):
        F, z = self.fx.expand_as(ux), torch.zeros_like(ux)
        return torch.stack([z, F, z, 2 * F * ux, 2 * F * ux, F * uy, 2 * F * ux * uy, F * uy * uy,
                            2 * F * ux * uy * uy], 1)

    def init(self, rho, ux, uy, phi, grads):
        mf, mg = self.eq_f(rho, ux, uy), self.eq_g(phi, ux, uy)
        if grads is not None:  # Chapman-Enskog non-equilibrium parts
            dxux, dyux, dxuy, dyuy, dxp, dyp = grads
            w, v = self.wf[:, :, 0], self.wg[:, :, 0]
            wf, wg = (lambda k: w[:, k:k + 1]), (lambda k: v[:, k:k + 1])
            mf[:, 3] += -2 * C3 * rho / wf(3) * (dxux + dyuy)
            mf[:, 4] += -2 * C3 * rho / wf(4) * (dxux - dyuy)
            mf[:, 5] += -C3 * rho / wf(5) * (dxuy + dyux)
            N = phi * (self.b1 * dxuy + self.b2 * dyux)
            ex, ey = -C3 / wg(1) * dxp, -C3 / wg(2) * dyp
            if not self.cm:
                mg[:, 1] += ex
                mg[:, 2] += ey
                mg[:, 5] += -C3 / wg(5) * (N + self.b1 * uy * dxp + self.b2 * ux * dyp)
            else:
                exy = -C3 / wg(5) * (N + (self.b1 - 1) * uy * dxp + (self.b2 - 1) * ux * dyp)
                z = torch.zeros_like(ex)
                mg += self._raw((ex, ey, z, z, exy, z, z, z), ux, uy)
        if self.forced:
            mf -= 0.5 * self.source(ux, uy)
        self.f, self.g = self._to(self.Mi, mf), self._to(self.Mi, mg)

    def macro(self):
        mf, mg = self._to(self.M, self.f), self._to(self.M, self.g)
        rho, phi = mf[:, 0], mg[:, 0]
        ux, uy = (mf[:, 1] + 0.5 * self.fx) / rho, mf[:, 2] / rho
        return mf, mg, rho, ux, uy, phi

    @staticmethod
    def _central(n, ux, uy):
        """Central moments (x, y, xx, yy, xy, xxy, xyy, xxyy) of raw ones with zero sum."""
        x, y, xy, xxy, xyy, q = n[:, 1], n[:, 2], n[:, 5], n[:, 6], n[:, 7], n[:, 8]
        xx, yy = 0.5 * (n[:, 3] + n[:, 4]), 0.5 * (n[:, 3] - n[:, 4])
        return (x, y, xx - 2 * ux * x, yy - 2 * uy * y, xy - uy * x - ux * y,
                xxy - 2 * ux * xy + ux * ux * y - uy * xx + 2 * ux * uy * x,
                xyy - 2 * uy * xy + uy * uy * x - ux * yy + 2 * ux * uy * y,
                q - 2 * ux * xyy - 2 * uy * xxy + ux * ux * yy + uy * uy * xx + 4 * ux * uy * xy
                - 2 * ux * ux * uy * y - 2 * ux * uy * uy * x)

    @staticmethod
    def _raw(c, ux, uy):
        """The raw moments of central ones (the shift by -u undone)."""
        x, y, xx, yy, xy, xxy, xyy, q = c
        rxx, ryy = xx + 2 * ux * x, yy + 2 * uy * y
        return torch.stack([torch.zeros_like(x), x, y, rxx + ryy, rxx - ryy, xy + uy * x + ux * y,
                            xxy + 2 * ux * xy + ux * ux * y + uy * xx + 2 * ux * uy * x,
                            xyy + 2 * uy * xy + uy * uy * x + ux * yy + 2 * ux * uy * y,
                            q + 2 * ux * xyy + 2 * uy * xxy + ux * ux * yy + uy * uy * xx
                            + 4 * ux * uy * xy + 2 * ux * ux * uy * y + 2 * ux * uy * uy * x], 1)

    def _stream(self, p, kind):
        out = torch.empty_like(p)
        for a in range(9):
            out[:, a] = torch.roll(p[:, a], (EY[a], EX[a]), (1, 2))
            if self.bc == "periodic":
                continue
            links = []  # (rows, columns, lid) of the nodes whose source lies beyond a wall
            if self.bc == "cavity" and EX[a]:
                links.append((slice(None), 0 if EX[a] == 1 else -1, False))
            if EY[a]:
                links.append((0 if EY[a] == 1 else -1, slice(None), EY[a] == -1))
            for ys, xs, lid in links:
                own = p[:, OPP[a]][:, ys, xs]
                if kind == "f":
                    more = 2 * W9[a] * EX[a] * 3.0 * (self.rho0 * self.u_lid)[:, 0] if lid else 0.0
                    out[:, a][:, ys, xs] = own + more
                else:
                    wall = (self.phi_lid if lid else self.phi_wall)[:, 0]
                    out[:, a][:, ys, xs] = 2 * W9[a] * wall - own
        return out

    def step(self):
        mf, mg, rho, ux, uy, phi = self.macro()
        df = -self.wf * (mf - self.eq_f(rho, ux, uy))
        if self.forced:
            df += (1 - 0.5 * self.wf) * self.source(ux, uy)
        ng = mg - self.eq_g(phi, ux, uy)
        if self.cm:
            c = self._central(ng, ux, uy)
            w = self.wg[:, :, 0].unsqueeze(-1).unbind(1)
            s, d = -w[3] * (c[2] + c[3]), -w[4] * (c[2] - c[3])
            dg = self._raw((-w[1] * c[0], -w[2] * c[1], 0.5 * (s + d), 0.5 * (s - d), -w[5] * c[4],
                            -w[6] * c[5], -w[7] * c[6], -w[8] * c[7]), ux, uy)
        else:
            dg = -self.wg * ng
        self.f = self._stream(self.f + self._to(self.Mi, df), "f")
        self.g = self._stream(self.g + self._to(self.Mi, dg), "g")

    def fields(self):
        mf, mg, rho, ux, uy, phi = self.macro()
        nf, ng = mf - self.eq_f(rho, ux, uy), mg - self.eq_g(phi, ux, uy)
        if self.forced:
            nf = nf + 0.5 * self.source(ux, uy)
        w, v = self.wf[:, :, 0].unsqueeze(-1).unbind(1), self.wg[:, :, 0].unsqueeze(-1).unbind(1)
        dxp, dyp = -3 * v[1] * ng[:, 1], -3 * v[2] * ng[:, 2]
        N = -3 * w[5] * nf[:, 5] / rho
        n5, c1, c2 = ng[:, 5], self.b1, self.b2
        if self.cm:
            n5, c1, c2 = n5 - uy * ng[:, 1] - ux * ng[:, 2], c1 - 1, c2 - 1
        Np = (-3 * v[5] * n5 - (c1 * uy * dxp + c2 * ux * dyp)) / phi
        om = (2 * Np - (self.b1 + self.b2) * N) / (self.b1 - self.b2)
        om = torch.where(phi.abs() >= 1e-3, om, torch.full_like(om, math.nan))
        k = -0.75 / rho
        return dict(rho=rho, ux=ux, uy=uy, phi=phi, sxx=k * (w[3] * nf[:, 3] + w[4] * nf[:, 4]),
                    sxy=0.5 * N, syy=k * (w[3] * nf[:, 3] - w[4] * nf[:, 4]), omega=om)


def _exact_lattice(case, seed):
    if case["nx"] * case["ny"] * case["steps"] > 9e8 or case["nx"] * case["ny"] > 5e6:
        return None
    p = _lattice_params(case, seed)
    *f, grads = _lattice_fields(case, p)
    fl = _Flow([p], case["bc"], case["model"])
    fl.init(*[v.double()[None] for v in f], None if grads is None else grads.double().unsqueeze(1))
    for _ in range(case["steps"]):
        fl.step()
    # with 16-bit storage the rounding of the populations is as large as the
    # non-equilibrium signal, so S and omega have no value to be held to
    keep = NAMES if case["storage"] == "fp32" else NAMES[:4]
    return {k: v[0] if k in keep else None for k, v in fl.fields().items()}


def _exact_batch(case, seed):
    ps = _batch_params(case, seed)
    if sum(p["n"] ** 2 for p in ps) * case["steps"] > 3e9:
        return None
    got = [None] * len(ps)
    for n in sorted(set(p["n"] for p in ps)):
        idx = [i for i, p in enumerate(ps) if p["n"] == n]
        fl = _Flow([ps[i] for i in idx], "cavity", "mrt")
        one = torch.ones(len(idx), n, n, dtype=torch.float64, device=DEV)
        start = torch.tensor([ps[i]["start"] for i in idx], dtype=torch.float32).double().to(DEV)
        fl.init(one, 0 * one, 0 * one, one * start.view(-1, 1, 1), None)
        for _ in range(case["steps"]):
            fl.step()
        f = fl.fields()
        for j, i in enumerate(idx):
            got[i] = {k: f[k][j].reshape(-1) for k in ("ux", "uy", "phi", "omega")}
    out = {k: torch.cat([g[k] for g in got]) for k in ("ux", "uy", "phi", "omega")}
    if case["storage"] != "fp32":  # as for one lattice
        out["omega"] = None
    return out


def _conv64(x, w, b=None):
    """3x3 convolution, NHWC, weights [co][3][3][ci], as nine shifted products."""
    B, H, W, ci = x.shape
    co = w.shape[0]
    w = w.reshape(co, 3, 3, ci)
    xp = torch.nn.functional.pad(x, (0, 0, 1, 1, 1, 1))
    y = 0
    for dy in range(3):
        for dx in range(3):
            y = y + xp[:, dy:dy + H, dx:dx + W, :] @ w[:, dy, dx, :].t()
    return y if b is None else y + b


def _leaky(z):
    return torch.where(z > 0, z, 0.02 * z)


def _net64(x, P):
    cv = lambda n, v: _leaky(_conv64(v, *P[n]))
    pool = lambda v: v.reshape(v.shape[0], v.shape[1] // 2, 2, v.shape[2] // 2, 2, -1).mean((2, 4))
    up = lambda v: v.repeat_interleave(2, 1).repeat_interleave(2, 2)
    e1 = cv("e1b", cv("e1a", x))
    e2 = cv("e2b", cv("e2a", pool(e1)))
    e3 = cv("e3b", cv("e3a", pool(e2)))
    b = cv("b2", cv("b1", pool(e3)))
    d3 = cv("d3b", cv("d3a", torch.cat([up(b), e3], -1)))
    d2 = cv("d2b", cv("d2a", torch.cat([up(d3), e2], -1)))
    d1 = cv("d1b", cv("d1a", torch.cat([up(d2), e1], -1)))
    return d1 @ P["head"][0].t() + P["head"][1]


def exact(case, seed):
    kind = case["kind"]
    if kind == "lattice":
        return _exact_lattice(case, seed)
    if kind == "batch":
        return _exact_batch(case, seed)
    if kind == "conv3x3":
        x, w, b = _conv_inputs(case, seed)
        return _leaky(_conv64(x.double(), w.double(), b.double()))
    # the weights as the network holds them: BF16 for the products, FP32 biases
    P = {n: (w.to(torch.bfloat16).double(), b.double()) for n, (w, b) in _net_weights(case, seed).items()}
    x, t = _net_batch(case, seed)
    if kind == "unet_predict":
        with torch.no_grad():
            return torch.cat([_net64(x[i:i + 2].double(), P) for i in range(0, case["batch"], 2)])
    for w, b in P.values():
        w.requires_grad_(True)
        b.requires_grad_(True)
    count, outs, loss = t.numel(), [], 0.0
    for i in range(0, case["batch"], 2):  # a few samples at a time: the gradients add up
        y = _net64(x[i:i + 2].double(), P)
        part = ((y - t[i:i + 2].double()) ** 2).sum() / count
        part.backward()
        outs.append(y.detach())
        loss = loss + part.detach()
    got = {"out": torch.cat(outs), "loss": loss.reshape(1)}
    for n, (w, b) in P.items():
        got[n + ".w"], got[n + ".b"] = w.grad, b.grad
    return got
