"""The work this framework is measured on: what its users have it do,
through the public classes (``lbm.Solver``, ``mlp.Mlp``), from the smallest
calls to the largest that fit a short measurement.

Kinds of case:

* ``job``   -- one lattice, whole call: create from host arrays, advance,
  read the observables, the densities and the solid mask, release.
* ``step``  -- lattices already on the GPU, in the middle of their life (A
  fills part of the section, deposits between 0 and the threshold, so nodes
  keep turning solid): advance, read the observables and the masks, and the
  densities of a single lattice.
* ``sweepjob`` -- a batch of uneven capillaries, whole call: create, advance
  with the observables read at intervals, read every mask, release.
* ``forward`` / ``grad`` / ``fit`` -- the surrogate network: inference, loss
  and gradient, a run of optimizer steps.

Observables of several lattices are kept in 32 bits, as the surrogate's
training targets keep them; those of one lattice are the plain numbers that
``Solver.observables`` returns.
"""
import math

import numpy as np
import torch

from paper_1309_6726_gb300 import inputs as I
from paper_1309_6726_gb300 import lbm, mlp

#: observables that are numbers of a lattice's state
OBS = ("front", "wetted_lower", "wetted_upper", "r_min", "r_h", "r_ave",
       "delta_e", "precip_mass", "mass_a", "mass_b", "mass_c", "ledger_a",
       "ledger_b", "ledger_c", "ledger_m")


def listed():
    return [
        # a smoke-sized capillary, odd sizes, 16-bit storage: creation, launches
        # and read-back are all there is
        dict(name="job tiny fp16", kind="job", geom="capillary", nx=131, ny=13,
             x_res=32, x_out=16, steps=200, precision="fp16"),
        # the small single capillary at its stated 2000 steps (a state that
        # fits the chip: the latency of a step counts)
        dict(name="job small fp32", kind="job", geom="capillary", nx=256, ny=32,
             x_res=64, x_out=32, steps=2000, precision="fp32"),
        # the paper-scale capillary, observables every 500 steps
        dict(name="step paper fp32", kind="step", geom="capillary", nx=4096,
             ny=128, x_res=256, x_out=128, count=1, steps=500,
             precision="fp32"),
        # the paper-scale study: three reaction rates in one handle, 16 bits
        dict(name="step paper x3 fp16", kind="step", geom="capillary", nx=4096,
             ny=128, x_res=256, x_out=128, count=3, steps=500,
             precision="fp16"),
        # a disc preform: solid everywhere, periodic in y, larger than L2
        dict(name="step preform fp32", kind="step", geom="preform", nx=1024,
             ny=1024, x_res=128, x_out=128, count=1, steps=200,
             precision="fp32"),
        # the batched sweep between two readings (production), full precision
        # and 16-bit storage
        dict(name="step sweep fp32", kind="step", geom="sweep", count=40,
             steps=100, precision="fp32"),
        dict(name="step sweep fp16", kind="step", geom="sweep", count=40,
             steps=100, precision="fp16"),
        # a whole sweep job from host arrays, BF16 storage, observables every
        # 10 of 50 steps
        dict(name="sweep job bf16", kind="sweepjob", count=32, steps=50,
             every=10, precision="bf16"),
        # the surrogate's inference at its stated batch
        dict(name="forward 8192", kind="forward", n_in=5, hidden=256, layers=3,
             n_out=65, batch=8192),
        # answering 256 held-out runs
        dict(name="forward 256", kind="forward", n_in=5, hidden=256, layers=3,
             n_out=65, batch=256),
        # loss and gradient of a ragged batch
        dict(name="grad 1000", kind="grad", n_in=4, hidden=256, layers=3,
             n_out=65, batch=1000),
        # sixteen optimizer steps on minibatches of 1024, then the weights
        dict(name="fit 16 x 1024", kind="fit", n_in=5, hidden=256, layers=3,
             n_out=65, batch=1024, steps=16),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["job", "job", "step", "step", "step", "sweepjob",
                       "forward", "grad", "fit"])
    prec = rng.choice(["fp32", "fp16", "bf16"])
    if kind == "job":
        nx, ny = _log(rng, 70, 1100), _log(rng, 7, 90)
        x_res, x_out = nx // 4, nx // 8
        # the front stays within what half the reservoir feeds (its speed is
        # about 0.13 height / length)
        far = 0.5 * x_res * (nx - x_res - x_out) / (0.13 * (ny - 2))
        return dict(kind=kind, geom="capillary", nx=nx, ny=ny, x_res=x_res,
                    x_out=x_out,
                    steps=max(20, min(_log(rng, 50, 2000), int(far),
                                      int(3e7 / (nx * ny)))),
                    precision=prec)
    if kind == "step":
        geom = rng.choice(["capillary", "preform", "sweep"])
        if geom == "capillary":
            return dict(kind=kind, geom=geom, nx=rng.randint(2800, 4600),
                        ny=rng.randint(64, 160), x_res=256, x_out=128,
                        count=rng.randint(1, 3), steps=rng.randint(200, 500),
                        precision=prec)
        if geom == "preform":
            n = rng.randint(700, 1100)
            return dict(kind=kind, geom=geom, nx=n, ny=n, x_res=128, x_out=128,
                        count=1, steps=rng.randint(100, 200), precision=prec)
        return dict(kind=kind, geom=geom, count=rng.randint(12, 40),
                    steps=rng.randint(40, 100), precision=prec)
    if kind == "sweepjob":
        return dict(kind=kind, count=rng.randint(4, 32),
                    steps=rng.randint(20, 50), every=rng.randint(7, 20),
                    precision=prec)
    net = dict(kind=kind, n_in=rng.randint(3, 8),
               hidden=16 * _log(rng, 2, 24), layers=rng.randint(1, 4),
               n_out=rng.randint(2, 96))
    if kind == "forward":
        return dict(net, batch=_log(rng, 1, 8192))
    if kind == "grad":
        return dict(net, batch=_log(rng, 32, 4096))
    return dict(net, batch=_log(rng, 64, 2048), steps=rng.randint(4, 16))


# ---- inputs ------------------------------------------------------------------

def _lattices(case, seed):
    """[(geometry, parameters)] of a solver case.  Reaction rate, contact
    angle and viscosity ratio as in the batched sweep (the ratio from 0.8
    up: below about 0.7 the model itself turns non-finite in a long run)."""
    rng = np.random.default_rng([seed, 77])
    sizes = np.random.default_rng(1236)  # a sweep's widths and lengths
    geom = case.get("geom", "sweep")
    out = []
    for _ in range(case.get("count", 1)):
        p = I.ModelParams(
            tau_a=float(rng.uniform(0.8, 1.5)), tau_b=1.0,
            g_ads=I.g_ads_for_angle(float(rng.uniform(20, 60))),
            k_r=float(10 ** rng.uniform(-5, -2)), inlet=1)
        if geom == "sweep":
            w, ln = int(sizes.integers(16, 129)), int(sizes.integers(1024, 4097))
            x_res = 64 if case["kind"] == "sweepjob" else 256
            g = I.capillary(ln + x_res + 32, w + 2, x_res, 32)
        elif geom == "preform":
            g = I.preform(n=case["nx"], seed=int(rng.integers(1 << 30)),
                          x_res=case["x_res"], x_out=case["x_out"],
                          solid_fraction=0.45)
        else:
            g = I.capillary(case["nx"], case["ny"], case["x_res"],
                            case["x_out"])
        if case["kind"] != "sweepjob":
            # A has filled part of the section; its solute thins out along it
            nx = g.solid.shape[1]
            xf = g.cap_x0 + float(rng.uniform(0.1, 0.4)) * (g.cap_x1 - g.cap_x0)
            x = np.arange(nx)[None, :] + 0 * g.solid
            fluid = g.solid == 0
            a = (x < xf) & fluid
            g.rho_a = np.where(a, I.RHO_MAJOR, I.RHO_MINOR * fluid).astype(np.float32)
            g.rho_b = np.where(a, I.RHO_MINOR, I.RHO_MAJOR * fluid).astype(np.float32)
            g.conc = (np.clip(1.0 - x / xf, 0, 1) * a).astype(np.float32)
        out.append((g, p))
    return out


def _deposit(solid, seed, k):
    """Deposits of a lattice in mid-life: 0 to the threshold on the nodes
    that touch the solid."""
    s = solid.astype(bool)
    near = (np.roll(s, 1, 0) | np.roll(s, -1, 0) | np.roll(s, 1, 1)
            | np.roll(s, -1, 1)) & ~s
    m = np.zeros(s.shape)
    m[near] = np.random.default_rng([seed, 78, k]).uniform(0, 0.9999, int(near.sum()))
    return m


def _net_inputs(case, seed, device):
    """Packed weights (Glorot uniform, as the surrogate's), inputs in
    [-1, 1] and smooth targets, a few of them unknown (NaN)."""
    rng = np.random.default_rng([seed, 79])
    shapes = mlp.layer_shapes(case["n_in"], case["hidden"], case["layers"],
                              case["n_out"])
    ws = [rng.uniform(-1, 1, s) * math.sqrt(6.0 / (s[0] + s[1])) for s in shapes]
    bs = [rng.uniform(-0.05, 0.05, s[0]) for s in shapes]
    g = torch.Generator(device=device).manual_seed(int(seed) * 9 + 1)
    n = case["batch"] * case.get("steps", 1)
    x = torch.rand((n, case["n_in"]), generator=g, device=device) * 2 - 1
    f = torch.arange(1, case["n_out"] + 1, device=device) * 0.1
    t = torch.sin(x.sum(1, keepdim=True) * f) + 0.3 * x[:, :1]
    t[::11, 0] = float("nan")
    return mlp.pack(ws, bs), x, t


#: learning rate of the optimizer steps: the end of the surrogate's schedule
LR = 1e-5


def prepare(case, seed):
    if case["kind"] in ("forward", "grad", "fit"):
        dev = torch.device("cuda", torch.cuda.current_device())
        theta, x, t = _net_inputs(case, seed, dev)
        net = mlp.Mlp(case["n_in"], case["hidden"], case["layers"],
                      case["n_out"], case["batch"])
        net.set_params(theta)
        b = case["batch"]
        return dict(case=case, net=net, x=x, t=t,
                    parts=[(x[i:i + b], t[i:i + b])
                           for i in range(0, x.shape[0], b)])
    pairs = _lattices(case, seed)
    geoms, params = [g for g, _ in pairs], [p for _, p in pairs]
    st = dict(case=case, geoms=geoms, params=params)
    if case["kind"] != "job":
        # masks come back into pinned memory, as a sweep program keeps it
        n = sum(g.solid.size for g in geoms)
        st["masks"] = torch.empty(n, dtype=torch.uint8, pin_memory=True).numpy()
    if case["kind"] == "step":
        s = lbm.Solver(geoms, params, case["precision"])
        for k, g in enumerate(geoms):
            s.set_deposit(_deposit(g.solid, seed, k), k)
        st["solver"] = s
        st["geoms"] = None
    return st


# ---- one pass ----------------------------------------------------------------

def _table(arr):
    return {k: arr[k].astype(np.float32) for k in OBS}


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "job":
        with lbm.Solver(st["geoms"][0], st["params"][0], case["precision"]) as s:
            s.step(case["steps"])
            o = s.observables(allow_nan=True)[0]
            return {"obs": {k: o[k] for k in OBS}, "density": [s.densities()],
                    "solid": s.solid_mask()}
    if kind == "step":
        s = st["solver"]
        s.step(case["steps"])
        obs = _table(s.observables_array(allow_nan=True))
        s.solid_masks(out=st["masks"])
        # a batch's program goes on with the observables and the masks, one
        # lattice's also with its fields
        return {"obs": obs, "density": [s.densities()] if s.count == 1 else [],
                "solid": st["masks"]}
    if kind == "sweepjob":
        rows, done = [], 0
        with lbm.Solver(st["geoms"], st["params"], case["precision"]) as s:
            while done < case["steps"]:
                n = min(case["every"], case["steps"] - done)
                s.step(n)
                done += n
                rows.append(s.observables_array(allow_nan=True))
            s.solid_masks(out=st["masks"])
        return {"obs": _table(np.stack(rows)), "solid": st["masks"]}
    net = st["net"]
    if kind == "forward":
        return net.forward(st["x"])
    if kind == "grad":
        g, loss = net.grad(st["x"], st["t"])
        return {"grad": g, "loss": loss}
    for x, t in st["parts"]:
        net.train_step(x, t, LR)
    return net.params()


# ---- what a pass cannot do without ---------------------------------------------

def work(case):
    """Solver: each of the 22 populations of a fluid node read and written
    once per step at the storage precision, and its mask byte read (the
    state is larger than what a step can keep on chip, but for the small
    jobs); about 520 flops per node and step.  Network: the products'
    operands and results once, two flops per multiply-add."""
    kind = case["kind"]
    if kind in ("forward", "grad", "fit"):
        dims = [case["n_in"]] + [case["hidden"]] * case["layers"] + [case["n_out"]]
        macs = sum(a * b for a, b in zip(dims, dims[1:]))
        b = case["batch"]
        if kind == "forward":
            return {"bytes": 2.0 * macs + 4.0 * b * (dims[0] + dims[-1]),
                    "flops": 2.0 * macs * b}
        # forward, the gradients of the weights, those of the activations
        fl = 2.0 * b * (3 * macs - dims[0] * dims[1])
        io = 4.0 * b * (dims[0] + dims[-1])
        if kind == "grad":
            return {"bytes": 2.0 * macs + io + 4.0 * macs, "flops": fl}
        n = case["steps"]  # weights and two moments, read and written
        return {"bytes": n * (24.0 * macs + io), "flops": n * fl}
    if kind == "sweepjob" or case["geom"] == "sweep":
        nodes = case["count"] * (2560 + 200) * 74.0  # of the drawn sizes' mean
    else:
        nodes = float(case.get("count", 1) * case["nx"] * case["ny"])
        if case["geom"] == "preform":
            nodes -= 0.45 * (case["nx"] - case["x_res"] - case["x_out"]) * case["ny"]
    per = 177.0 if case["precision"] == "fp32" else 89.0
    reads = 1 if kind != "sweepjob" else -(-case["steps"] // case["every"])
    back = 13.0 * nodes if case.get("count", 1) == 1 and kind != "sweepjob" else nodes
    made = 13.0 * nodes if kind != "step" else 0.0
    return {"bytes": per * nodes * case["steps"] + 9.0 * nodes * reads + back + made,
            "flops": 520.0 * nodes * case["steps"]}


# ---- the same in 64 bits ---------------------------------------------------------

_EX = [0, 1, 0, -1, 0, 1, -1, -1, 1]
_EY = [0, 0, 1, 0, -1, 1, 1, -1, -1]
_W = [4 / 9] + [1 / 9] * 4 + [1 / 36] * 4
_OPP = [0, 3, 4, 1, 2, 7, 8, 5, 6]


class _Lattice64:
    """The method on one lattice in float64 torch, one operation after the
    other: moments, Martys-Chen forces, Shan-Chen shift, BGK of A and B, of
    the solute, surface reaction, streaming with half-way bounce-back,
    growth."""

    def __init__(self, g, p, deposit, dev):
        def t(a):
            return torch.from_numpy(np.ascontiguousarray(a)).to(dev).double()
        self.p, self.dev = p, dev
        self.x0, self.x1 = g.cap_x0, g.cap_x1
        self.solid = torch.from_numpy(g.solid != 0).to(dev)
        self.solid0 = self.solid.clone()
        fl = (~self.solid).double()
        self.w = torch.tensor(_W, dtype=torch.float64, device=dev).view(1, 9, 1, 1)
        self.ex = torch.tensor(_EX, dtype=torch.float64, device=dev).view(1, 9, 1, 1)
        self.ey = torch.tensor(_EY, dtype=torch.float64, device=dev).view(1, 9, 1, 1)
        rho = torch.stack([t(g.rho_a), t(g.rho_b)]) * fl
        self.f = self.w * rho[:, None]
        self.g = (0.25 * t(g.conc) * fl)[None].repeat(4, 1, 1)
        self.m = t(deposit)
        self.led = torch.zeros(4, dtype=torch.float64, device=dev)
        self._around()

    def _around(self):
        """What depends on the solid set alone."""
        s = self.solid.double()
        nb = [torch.roll(s, (-_EY[i], -_EX[i]), (0, 1)) for i in range(9)]
        self.ax = sum(_W[i] * _EX[i] * nb[i] for i in range(1, 9))
        self.ay = sum(_W[i] * _EY[i] * nb[i] for i in range(1, 9))
        self.ns = nb[1] + nb[2] + nb[3] + nb[4]
        self.fl = 1.0 - s
        # source node x - e_i solid: the value bounces back
        self.back = torch.stack([torch.roll(self.solid, (_EY[i], _EX[i]), (0, 1))
                                 for i in range(9)])

    def step(self):
        p, f, w, ex, ey = self.p, self.f, self.w, self.ex, self.ey
        rho = f.sum(1)                                     # [2, ny, nx]
        jx, jy = (f * ex).sum(1), (f * ey).sum(1)
        sx = sy = 0.0
        other = rho.flip(0)
        for i in range(1, 9):
            nb = torch.roll(other, (-_EY[i], -_EX[i]), (1, 2))
            if _EX[i]:
                sx = sx + _W[i] * _EX[i] * nb
            if _EY[i]:
                sy = sy + _W[i] * _EY[i] * nb
        sign = torch.tensor([1.0, -1.0], dtype=torch.float64, device=self.dev).view(2, 1, 1)
        fx = rho * (sign * p.g_ads * self.ax - p.g_coh * sx + p.body_force_x)
        fy = rho * (sign * p.g_ads * self.ay - p.g_coh * sy)
        tau = torch.tensor([p.tau_a, p.tau_b], dtype=torch.float64, device=self.dev).view(2, 1, 1)
        den = (rho / tau).sum(0).clamp_min(1e-300)
        live = rho > 1e-12
        inv = torch.where(live, tau / torch.where(live, rho, 1.0), 0.0)
        ux = (jx / tau).sum(0) / den + inv * fx
        uy = (jy / tau).sum(0) / den + inv * fy
        eu = ex * ux[:, None] + ey * uy[:, None]
        uu = (ux * ux + uy * uy)[:, None]
        feq = w * rho[:, None] * (1 + 3 * eu + 4.5 * eu * eu - 1.5 * uu)
        f = f + (feq - f) / tau[:, None]
        rt = rho.sum(0).clamp_min(1e-300)
        bx, by = (jx + 0.5 * fx).sum(0) / rt, (jy + 0.5 * fy).sum(0) / rt
        g = self.g
        c = g.sum(0)
        geq = torch.stack([0.25 * c + 0.5 * c * bx, 0.25 * c + 0.5 * c * by,
                           0.25 * c - 0.5 * c * bx, 0.25 * c - 0.5 * c * by])
        new = g + (geq - g) / p.tau_d
        if p.inlet:
            q, ci = 0.25 * p.c_in, 0.5 * p.c_in
            new[:, :, 0] = torch.stack([q + ci * bx[:, 0], q + ci * by[:, 0],
                                        q - ci * bx[:, 0], q - ci * by[:, 0]])
        g = new
        lost = (p.k_r * self.ns).clamp_max(1.0) * (rho[0] > rho[1]) * self.fl
        dm = g.sum(0) * lost
        g = g - g * lost
        # streaming: pull from x - e_i, or the node's own opposite
        out = torch.empty_like(f)
        for i in range(9):
            out[:, i] = torch.where(self.back[i], f[:, _OPP[i]],
                                    torch.roll(f[:, i], (_EY[i], _EX[i]), (1, 2)))
        gs = torch.empty_like(g)
        for k in range(4):
            i = k + 1
            gs[k] = torch.where(self.back[i], g[_OPP[i] - 1],
                                torch.roll(g[k], (_EY[i], _EX[i]), (0, 1)))
        self.m = self.m + dm
        flip = (self.m >= p.m_threshold) & ~self.solid
        if bool(flip.any()):
            fd = flip.double()
            self.led += torch.stack([(out[0].sum(0) * fd).sum(), (out[1].sum(0) * fd).sum(),
                                     (gs.sum(0) * fd).sum(), (self.m * fd).sum()])
            self.m = self.m * (1 - fd)
            self.solid = self.solid | flip
            self._around()
        self.f, self.g = out * self.fl, gs * self.fl

    def density(self):
        return torch.stack([self.f[0].sum(0), self.f[1].sum(0), self.g.sum(0)])

    def obs(self):
        """Front, wall profiles and masses (OBS order)."""
        ra, rb, c = self.density().cpu().numpy()
        s, s0 = self.solid.cpu().numpy(), self.solid0.cpu().numpy()
        ny, nx = s.shape
        x0, x1 = self.x0, self.x1
        phi = ra - rb
        z = []
        for y in sorted({(ny - 1) // 2, ny // 2}):
            a = max(x0 - 1, 0)
            hit = [x for x in range(a, nx - 1)
                   if not s[y, x] and not s[y, x + 1] and phi[y, x] > 0 >= phi[y, x + 1]]
            z.append(hit[0] + phi[y, hit[0]] / (phi[y, hit[0]] - phi[y, hit[0] + 1])
                     - (x0 - 0.5) if hit else math.nan)

        def walls(m):
            fl = ~m[:, x0:x1]
            some = fl.any(0)
            return (np.where(some, fl.argmax(0), ny),
                    np.where(some, fl[::-1].argmax(0), ny), fl.sum(0))
        b, t, h = walls(s)
        b0, t0, _ = walls(s0)
        open_ = h > 0
        cols = np.arange(x0, x1)
        lo = (phi[np.minimum(b, ny - 1), cols] > 0) & open_
        up = (phi[np.maximum(ny - 1 - t, 0), cols] > 0) & open_
        grown = np.where(open_, np.maximum(b - b0, t - t0), (ny - b0 - t0) / 2.0)
        area = np.maximum(0.0, (ny - 1) / 2.0 - (b - 0.5)).sum()
        per = len(b) + np.abs(np.diff(b)).sum()
        led = self.led.tolist()
        m = float((self.m * (~self.solid)).sum())
        return [float(np.mean(z)), lo.sum(), up.sum(), h.min() / 2.0, area / per,
                h.mean() / 2.0, grown.max(), m + led[3], ra.sum(), rb.sum(),
                c.sum()] + led


def exact(case, seed):
    dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
    if case["kind"] in ("forward", "grad", "fit"):
        return _exact_net(case, seed, dev)
    pairs = _lattices(case, seed)
    lats = []
    for k, (g, p) in enumerate(pairs):
        dep = (_deposit(g.solid, seed, k) if case["kind"] == "step"
               else np.zeros(g.solid.shape))
        lats.append(_Lattice64(g, p, dep, dev))
    every = case.get("every", case["steps"])
    rows, done = [], 0
    while done < case["steps"]:
        n = min(every, case["steps"] - done)
        for lat in lats:
            for _ in range(n):
                lat.step()
        done += n
        rows.append([lat.obs() for lat in lats])
    tab = np.asarray(rows, np.float64)  # [reading, lattice, observable]
    if case["kind"] == "job":
        return {"obs": {k: float(tab[0, 0, j]) for j, k in enumerate(OBS)},
                "density": [lats[0].density().cpu().numpy()], "solid": None}
    if case["kind"] == "step":
        return {"obs": {k: tab[0, :, j] for j, k in enumerate(OBS)},
                "density": [lat.density().cpu().numpy() for lat in lats
                            if len(lats) == 1], "solid": None}
    return {"obs": {k: tab[:, :, j] for j, k in enumerate(OBS)}, "solid": None}


def _exact_net(case, seed, dev):
    theta, x, t = _net_inputs(case, seed, dev)
    th = torch.from_numpy(theta).to(dev).double()
    sizes = []
    for r, c in mlp.layer_shapes(case["n_in"], case["hidden"], case["layers"],
                                 case["n_out"]):
        sizes += [(r, c), (r,)]

    def forward(v, xb):
        o, h = 0, xb
        for j in range(0, len(sizes), 2):
            (r, c), n = sizes[j], sizes[j][0] * sizes[j][1]
            h = h @ v[o:o + n].view(r, c).T + v[o + n:o + n + r]
            o += n + r
            if j + 2 < len(sizes):
                h = torch.tanh(h)
        return h

    def grad(v, xb, tb):
        v = v.detach().requires_grad_(True)
        y = forward(v, xb)
        d = torch.where(torch.isnan(tb), torch.zeros_like(y), y - torch.nan_to_num(tb))
        loss = (d * d).sum() / y.numel()
        loss.backward()
        return v.grad, float(loss.detach())

    x, t = x.double(), t.double()
    if case["kind"] == "forward":
        return forward(th, x)
    if case["kind"] == "grad":
        g, loss = grad(th, x, t)
        return {"grad": g, "loss": loss}
    m1, m2, b = torch.zeros_like(th), torch.zeros_like(th), case["batch"]
    for k in range(case["steps"]):
        g, _ = grad(th, x[k * b:(k + 1) * b], t[k * b:(k + 1) * b])
        m1, m2 = 0.9 * m1 + 0.1 * g, 0.999 * m2 + 0.001 * g * g
        th = th - LR * (m1 / (1 - 0.9 ** (k + 1))) / (
            (m2 / (1 - 0.999 ** (k + 1))).sqrt() + 1e-8)
    return th.cpu().numpy()
