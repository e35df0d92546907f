"""Workloads of the active flux solver as a user's program runs them, for timing and for
comparing results: `listed()` and `draw(rng)` describe cases, `prepare` makes what the
program holds beforehand (a context with its state, a batch, a network), `run` is one pass
through the public entry points, `work` what a pass cannot do without, and `exact` the same
pass in 64 bits in plain torch and numpy.

Kinds of case:
  run    march over a given time (Solver.run) and read the state back: the paper's examples
         at their printed sizes, where launches and latency count
  step   one CFL time step (Solver.step) of a mesh that stays on the device
  batch  one CFL time step of many meshes of uneven sizes (af_batch_step)
  train  training data from a state (af_mlp_features) and Adam steps of the learned
         indicator (af_mlp_train)
"""
import math

import numpy as np
import torch

import af_inputs as ai
from paper_2510_11527_gb300 import Solver, capi

# ---------------------------------------------------------------------------------------
# cases


def listed():
    return [
        # Example 6.5 as printed: 200 cells, Dirichlet ends, 70,772 steps to its final time
        # -- a run of it is nothing but small launches
        dict(name="run_1d_evje_karlsen_200", kind="run", problem="evje_karlsen", nx=200, precision="fp64", rk=3,
             blend="off", steps=64),
        # Example 6.4 as printed: 100 x 100 cells, 3054 steps to its final time
        dict(name="run_2d_two_hills_100", kind="run", problem="two_hills", nx=100, ny=100, precision="fp64", rk=3,
             blend="off", steps=32),
        # the benchmark's headline: degenerate Burgers, plain FP64
        dict(name="step_fp64_burgers_1024", kind="step", problem="degenerate_burgers2d", nx=1024, ny=1024,
             precision="fp64", rk=3, blend="off"),
        # the same problem in the FP32-mixed form at the benchmark's second size
        dict(name="step_fp32_burgers_2048", kind="step", problem="degenerate_burgers2d", nx=2048, ny=2048,
             precision="fp32_mixed", rk=3, blend="off"),
        # porous medium at the benchmark's full size, five-stage scheme
        dict(name="step_fp32_pme_4096_rk54", kind="step", problem="pme2d", nx=4096, ny=4096,
             precision="fp32_mixed", rk=54, blend="off"),
        # Buckley-Leverett with gravity and the smoothness blend at the benchmark's full size
        dict(name="step_fp32_bl_blend_4096", kind="step", problem="buckley_leverett2d", nx=4096, ny=4096,
             precision="fp32_mixed", rk=3, blend="plain"),
        # the same with the learned indicator, an uneven mesh
        dict(name="step_fp32_bl_learned_2001x1500", kind="step", problem="buckley_leverett2d", nx=2001, ny=1500,
             precision="fp32_mixed", rk=3, blend="learned"),
        # Example 6.9's problem (outflow ends) on a fine mesh
        dict(name="step_fp32_outflow_1536", kind="step", problem="strongly_degenerate2d", nx=1536, ny=1536,
             precision="fp32_mixed", rk=3, blend="off"),
        # 16 instances of the benchmark's batch (64 to 1024 cells a side)
        dict(name="batch_fp32_16", kind="batch", count=16, nmin=64, nmax=1024, precision="fp32_mixed", rk=3,
             blend="off"),
        # 3D porous medium: Table 4's 3D size and scheme in FP64, the benchmark's size in FP32-mixed
        dict(name="step_3d_fp64_pme_80_rk54", kind="step", problem="pme3d", nx=80, ny=80, nz=80, precision="fp64",
             rk=54, blend="off"),
        dict(name="step_3d_fp32_pme_128", kind="step", problem="pme3d", nx=128, ny=128, nz=128,
             precision="fp32_mixed", rk=3, blend="off"),
        # the learned indicator's training at the benchmark's minibatch
        dict(name="train_512_batch_4096", kind="train", problem="buckley_leverett2d", nx=512, ny=512,
             precision="fp32_mixed", batch=4096, steps=24),
    ]


def draw(rng):
    def size(lo, hi):
        return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))

    what = rng.choice(["run1d", "run2d", "step64", "step32", "step32", "outflow", "batch", "3d64", "3d32", "train"])
    prec = rng.choice(["fp64", "fp32_mixed"])
    if what == "run1d":
        p = rng.choice(["evje_karlsen", "strongly_degenerate1d", "buckley_leverett1d_ibvp"])
        return dict(kind="run", problem=p, nx=size(50, 4000), precision=prec, rk=rng.choice([3, 54]),
                    blend="plain" if p == "strongly_degenerate1d" else "off", steps=rng.randint(16, 64))
    if what == "run2d":
        p = rng.choice(["two_hills", "buckley_leverett2d_outflow", "strongly_degenerate2d"])
        return dict(kind="run", problem=p, nx=size(40, 250), ny=size(40, 250), precision=prec, rk=rng.choice([3, 54]),
                    blend="off", steps=rng.randint(8, 32))
    if what == "step64":
        p = rng.choice(["degenerate_burgers2d", "pme2d", "buckley_leverett2d"])
        return dict(kind="step", problem=p, nx=size(100, 1024), ny=size(100, 1024), precision="fp64", rk=3,
                    blend="plain" if p == "buckley_leverett2d" else "off")
    if what == "step32":
        p = rng.choice(["degenerate_burgers2d", "pme2d", "buckley_leverett2d"])
        return dict(kind="step", problem=p, nx=size(200, 4096), ny=size(200, 4096), precision="fp32_mixed",
                    rk=rng.choice([3, 54]) if p != "buckley_leverett2d" else 3,
                    blend=rng.choice(["plain", "learned", "off"]) if p == "buckley_leverett2d" else rng.choice(["plain", "off", "off"]) if p == "degenerate_burgers2d" else "off")
    if what == "outflow":
        p = rng.choice(["strongly_degenerate2d", "buckley_leverett2d_outflow"])
        hi = 2048 if prec == "fp32_mixed" else 800
        return dict(kind="step", problem=p, nx=size(100, hi), ny=size(100, hi), precision=prec, rk=3,
                    blend="plain" if p == "strongly_degenerate2d" and rng.random() < 0.3 else "off")
    if what == "batch":
        return dict(kind="batch", count=rng.randint(4, 16), nmin=64, nmax=rng.choice([256, 512, 1024]),
                    precision="fp32_mixed" if rng.random() < 0.7 else "fp64", rk=3, blend=rng.choice(["off", "off", "plain"]))
    if what in ("3d64", "3d32"):
        hi = 80 if what == "3d64" else 128
        p = rng.choice(["pme3d", "pme3d", "burgers3d"])
        return dict(kind="step", problem=p, nx=size(20, hi), ny=size(20, hi), nz=size(20, hi),
                    precision="fp64" if what == "3d64" else "fp32_mixed", rk=rng.choice([3, 54]), blend="off")
    return dict(kind="train", problem="buckley_leverett2d", nx=size(100, 1024), ny=size(100, 1024), precision=prec,
                batch=rng.choice([1024, 2048, 4096, 5000]), steps=rng.randint(8, 24))


# ---------------------------------------------------------------------------------------
# problems and inputs

# floating-point operations of one limited forward-Euler evaluation, per cell (adds,
# multiplies and divisions of the method written out in 64 bits)
FLOPS = {"evje_karlsen": 137, "strongly_degenerate1d": 226, "buckley_leverett1d_ibvp": 254, "two_hills": 519,
         "buckley_leverett2d_outflow": 1200, "strongly_degenerate2d": 571, "degenerate_burgers2d": 571, "pme2d": 519,
         "buckley_leverett2d": 1686, "batch": 571, "pme3d": 792, "burgers3d": 1896}
MLP_FLOPS = 2 * (21 * 32 + 32 * 32 + 32)   # one forward evaluation of the network


def _spec(case):
    n, ny, nz = case["nx"], case.get("ny", 1), case.get("nz", 1)
    p = case["problem"]
    if p == "evje_karlsen":
        s = ai.evje_karlsen(n)
    elif p == "strongly_degenerate1d":
        s = ai.strongly_degenerate_1d(n)
    elif p == "buckley_leverett1d_ibvp":
        s = ai.buckley_leverett_1d(n, gravity=True)
    elif p == "two_hills":
        s = ai.two_hills(n)
    elif p == "buckley_leverett2d_outflow":
        s = ai.buckley_leverett_2d_outflow(n)
    elif p == "strongly_degenerate2d":
        s = ai.strongly_degenerate_2d(n)
    elif p == "degenerate_burgers2d":
        s = ai.config2(n)
    elif p == "pme2d":
        s = ai.config3(n)
    elif p == "buckley_leverett2d":
        s = ai.config5(n)
    elif p == "pme3d":
        s = ai.pme_3d(n)
    elif p == "burgers3d":
        s = ai.Spec(dim=3, nx=n, flux=("burgers", (0.5,)), diff=("const", (0.01,)), umin=0.0, umax=1.0,
                    limiter=True, name="burgers3d")
    else:
        raise KeyError(p)
    s = s.with_size(n, ny if s.dim >= 2 else 1, nz if s.dim == 3 else 1)
    b = case.get("blend", "off")
    s.blend = "external" if b == "learned" else b
    s.rk = case.get("rk", 3)
    return s


def _device():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _initial(spec, seed):
    """The problem's initial data, moved and scaled a little by the seed, on the GPU."""
    rng = np.random.default_rng(seed)
    dx, dy, dz = (float(v) for v in rng.uniform(-0.1, 0.1, 3))
    sc = float(rng.uniform(0.9, 1.1))
    dev = _device()
    if spec.name == "evje_karlsen":
        return ai.state_1d(lambda x: ai.evje_karlsen_fn(x + 0.5 * dx), spec, device=dev)
    if spec.name == "strongly_degenerate1d":
        return ai.state_1d(lambda x: ai.strongly_degenerate_fn(sc * x + dx), spec, device=dev)
    if spec.name == "buckley_leverett1d_ibvp":
        return ai.state_1d(lambda x: ai.bl1d_ibvp_fn(x * sc), spec, device=dev)
    if spec.name == "pme3d":
        return _state_3d(lambda x, y, z: ai.barenblatt_3d(sc * x + dx, sc * y + dy, sc * z + dz, 1.0), spec, dev)
    if spec.name == "burgers3d":
        def wave(x, y, z):
            return 0.5 + 0.45 * torch.sin(2 * math.pi * (x + dx)) * torch.cos(2 * math.pi * (y - z + dy))
        return _state_3d(wave, spec, dev)
    f = {"two_hills": ai.two_hills_fn, "degenerate_burgers2d": ai.discs_fn,
         "pme2d": lambda x, y: ai.barenblatt(x, y, 1.0), "buckley_leverett2d": ai.bl_disc_fn,
         "buckley_leverett2d_outflow": lambda x, y: ai.bl_disc_fn(x, y, math.sqrt(0.5)),
         "strongly_degenerate2d": ai.strongly_degenerate_2d_fn}[spec.name]
    st = ai.state_2d(lambda x, y: f(sc * x + dx, sc * y + dy), spec, device=dev, sub=2, order=3)
    return [a.clamp(spec.umin, spec.umax) for a in st]


def _state_3d(f, spec, dev):
    """Cell averages by a two-point Gauss rule on each half-cell, point values exact."""
    g = 0.25 / math.sqrt(3.0)
    offs = (0.25 - g, 0.25 + g, 0.75 - g, 0.75 + g)
    i, j, k = (torch.arange(n, dtype=torch.float64, device=dev) for n in (spec.nx, spec.ny, spec.nz))

    def at(ox, oy, oz):
        return f((spec.x0 + (i + ox) * spec.dx)[None, None, :], (spec.y0 + (j + oy) * spec.dy)[None, :, None],
                 (spec.z0 + (k + oz) * spec.dz)[:, None, None]).expand(spec.nz, spec.ny, spec.nx)

    ub = sum(at(a, b, c) for a in offs for b in offs for c in offs) / 64.0
    pts = [at(0.5 + 0.5 * (s & 1), 0.5 + 0.5 * ((s >> 1) & 1), 0.5 + 0.5 * ((s >> 2) & 1)) for s in range(1, 8)]
    return [a.clamp(spec.umin, spec.umax).contiguous() for a in [ub] + pts]


def _batch_specs(case, seed=0):
    """The benchmark batch's meshes and coefficients, the initial data from the seed."""
    mesh = ai.batch_instances(count=case["count"], nmin=case["nmin"], nmax=case["nmax"])
    data = ai.batch_instances(count=case["count"], seed=seed, nmin=case["nmin"], nmax=case["nmax"])
    return [(s, m) for (s, _), (_, m) in zip(mesh, data)]


def _params(seed):
    return ai.mlp_init_params(1000 + seed)


# ---------------------------------------------------------------------------------------
# prepare and run


class _Owner:
    """Contexts and networks, given back when nothing refers to them any more."""

    def __init__(self):
        self.closers = []

    def __del__(self):
        for f in reversed(self.closers):
            f()


class _View:
    """Device memory of a context or batch, which lives as long as a view of it."""

    def __init__(self, ptr, shape, typestr, owner):
        self.__cuda_array_interface__ = {"shape": shape, "typestr": typestr, "data": (ptr, False), "version": 3}
        self.owner = owner


class _Hold:
    """What a program keeps between passes."""

    def __init__(self, **kw):
        self.__dict__.update(kw)


def _views(ptrs, sizes, shape, owner):
    return [torch.as_tensor(_View(p, shape, "<f%d" % sizes[min(k, 1)], owner), device="cuda")
            for k, p in enumerate(ptrs)]


def prepare(case, seed):
    if case["kind"] == "batch":
        inst = _batch_specs(case, seed)
        g, f, d, bd = [], [], [], []
        for s, _ in inst:
            g.append(capi.af_grid(2, s.nx, s.ny, s.x0, s.x1, s.y0, s.y1))
            fl, df = capi.af_flux(), capi.af_diff()
            fl.kind, df.kind = capi.FLUX["burgers"], capi.DIFF["pwl"]
            fl.p[0] = s.flux[1][0]
            for k, v in enumerate(s.diff[1]):
                df.p[k] = v
            f.append(fl)
            d.append(df)
            bd.append(capi.af_bounds_t(s.umin, s.umax, 0))
        o = capi.af_opts(capi.PREC[case["precision"]], case["rk"], 0.0, 0.0, 1, capi.BLEND[case["blend"]], 1.0)
        b = capi.af_batch_create(g, f, d, bd, o)
        owner, outs = _Owner(), []
        owner.closers.append(lambda: capi.af_batch_destroy(b))
        for k, (s, m) in enumerate(inst):
            st = ai.batch_state(s, m, device=_device())
            capi.af_batch_set_state(b, k, s.cells, *[a.cpu().numpy() for a in st])
        # the state stays in the same buffers, so their views are made once
        for k, (s, m) in enumerate(inst):
            outs.append(_views(*capi.af_batch_device_ptrs(b, k), (s.ny, s.nx), owner))
        return _Hold(kind="batch", b=b, owner=owner, outs=outs)
    spec = _spec(case)
    s = Solver(spec, precision=case["precision"], rk=spec.rk)
    owner = _Owner()
    owner.closers.append(s.close)
    s.set_state([a.cpu().numpy() for a in _initial(spec, seed)])
    hold = _Hold(kind=case["kind"], s=s, owner=owner)
    if case["kind"] == "run":
        # a stretch of time that this many steps cover
        hold.dT = (case["steps"] - 0.5) * s.dt_cfl()
        hold.T = 0.0
    elif case["kind"] == "step":
        if case["blend"] == "learned":
            net = capi.af_mlp_create()
            owner.closers.insert(0, lambda: capi.af_mlp_destroy(net))
            capi.af_mlp_set_params(net, _params(seed))
            capi.af_set_mlp(s.ctx, net)
        shape = (spec.nz, spec.ny, spec.nx) if spec.dim == 3 else (spec.ny, spec.nx)
        if spec.bc != "periodic":
            shape = (spec.ny + 1, spec.nx + 1)
        hold.outs = _views(*(capi.af_device_ptrs_arrays(s.ctx, 8) if spec.dim == 3 else capi.af_device_ptrs(s.ctx)),
                           shape, owner)
    else:
        net = capi.af_mlp_create()
        owner.closers.append(lambda: capi.af_mlp_destroy(net))
        hold.net, hold.params, hold.case, hold.seed = net, _params(seed), case, seed
        hold.feat = torch.empty((spec.cells, 21), dtype=torch.float32, device="cuda")
        hold.label = torch.empty(spec.cells, dtype=torch.float32, device="cuda")
    return hold


def run(h):
    if h.kind == "run":
        h.T += h.dT
        n = h.s.run(h.T)
        return {"state": h.s.get_state(), "steps": n}
    if h.kind == "step":
        h.s.step()
        return h.outs
    if h.kind == "batch":
        capi.af_batch_step(h.b, 1)
        return h.outs
    c = h.case
    capi.af_mlp_features(h.s.ctx, h.feat.data_ptr(), h.label.data_ptr())
    capi.af_mlp_set_params(h.net, h.params)
    loss = capi.af_mlp_train(h.net, h.feat.data_ptr(), h.label.data_ptr(), h.label.numel(), c["batch"], c["steps"],
                             3e-3, h.seed + 1)
    return {"params": capi.af_mlp_get_params(h.net), "loss": loss, "feat": h.feat, "label": h.label}


def _evaluations(rk):
    return 3 if rk == 3 else 6   # the fourth stage of SSP-RK(5,4) has two outputs


def work(case):
    if case["kind"] == "batch":
        cells = sum(s.cells for s, _ in _batch_specs(case))
        return {"bytes": 2 * cells * (32 if case["precision"] == "fp64" else 20), "flops": cells * 571 * 3}
    cells = case["nx"] * case.get("ny", 1) * case.get("nz", 1)
    dim = 3 if "nz" in case else 2 if "ny" in case else 1
    point = 8 if case["precision"] == "fp64" else 4
    state = cells * (8 + point * (2 ** dim - 1))
    if case["kind"] == "train":
        return {"bytes": state + cells * 88 + 4 * 1793 * 2,
                "flops": cells * 100.0 + 3.0 * MLP_FLOPS * case["batch"] * case["steps"]}
    per = FLOPS[case["problem"]] + (MLP_FLOPS if case["blend"] == "learned" else 0)
    return {"bytes": 2 * state, "flops": float(cells) * per * _evaluations(case["rk"]) * case.get("steps", 1)}


# ---------------------------------------------------------------------------------------
# the same in 64 bits: the method written on the kinds of the half-spaced grid. A state is
# a list of 2^d arrays by kind s = s_x + 2 s_y + 4 s_z (0: cell averages); the location at
# fine offset f from a cell's centre is kind f mod 2 of the cell shifted by floor(f / 2).


def _crit(direction, g):
    """Interior extrema c of f' for the Buckley-Leverett flux, and |f'(c)|."""
    fp = lambda u: _bl(u, g, direction)[1]
    x = np.linspace(-1.0, 2.0, 60001)
    y = fp(x)
    out = []
    for k in range(1, 60000):
        sign = 1.0 if y[k] >= y[k - 1] and y[k] > y[k + 1] else -1.0 if y[k] <= y[k - 1] and y[k] < y[k + 1] else 0.0
        if not sign:
            continue
        lo, hi = x[k - 1], x[k + 1]
        for _ in range(120):
            a, b = lo + (hi - lo) / 3.0, hi - (hi - lo) / 3.0
            if sign * fp(a) < sign * fp(b):
                lo = a
            else:
                hi = b
        out.append((0.5 * (lo + hi), abs(fp(0.5 * (lo + hi)))))
    return out


def _bl(u, g, direction):
    v = 1.0 - u
    D = u * u + v * v
    f, d = u * u / D, 2.0 * u * v / (D * D)
    if direction == 0:
        return f, d
    w = 1.0 - g * v * v
    return f * w, d * w + 2.0 * g * v * f


class _Method:
    def __init__(self, spec):
        self.s, self.d = spec, spec.dim
        self.h = [spec.dx, spec.dy, spec.dz][:spec.dim]
        self.fk, self.fp = spec.flux
        self.dk, self.dp = spec.diff
        self.crit = {}
        if self.fk == "bl":
            for l in range(self.d):
                self.crit[l] = _crit(1 if self.d == 1 else l, self.fp[0])
        diffuses = self.dk == "pme" or (self.dk != "none" and any(self.dp[k] != 0.0 for k in ((0, 2) if self.dk == "pwl" else (0,) if self.dk in ("const", "ramp") else (0, 1, 2))))
        self.parts = 3 if diffuses else 1
        u = np.linspace(spec.umin, spec.umax, 200001)
        self.kmax = float(max(self._kappa(u)))
        if self.dk in ("cubic", "cubic01"):
            uv = -self.dp[1] / (3.0 * self.dp[2])
            if spec.umin < uv < spec.umax:
                self.kmax = max(self.kmax, float(self._kappa(np.array([uv]))[0]))

    def _kappa(self, u):
        p = self.dp
        if self.dk == "const":
            return np.full_like(u, p[0])
        if self.dk == "pwl":
            return np.where(u < p[1], p[0], 0.0) + np.where(u > p[3], p[2], 0.0)
        if self.dk == "pme":
            return p[0] * u ** (p[0] - 1)
        if self.dk in ("cubic", "cubic01"):
            return p[0] + 2 * p[1] * u + 3 * p[2] * u * u
        if self.dk == "ramp":
            return np.clip((u - p[1]) / p[2], 0.0, 1.0) * p[0]
        return np.zeros_like(u)

    def a(self, u):
        p = self.dp
        if self.dk == "const":
            return p[0] * u
        if self.dk == "pwl":
            return p[0] * (u - p[1]).clamp(max=0.0) + p[2] * (u - p[3]).clamp(min=0.0)
        if self.dk == "pme":
            return u ** p[0]
        if self.dk == "cubic01":
            u = u.clamp(0.0, 1.0)
        if self.dk in ("cubic", "cubic01"):
            return ((p[2] * u + p[1]) * u + p[0]) * u
        if self.dk == "ramp":
            r = u - p[1]
            return torch.where(r <= 0, torch.zeros_like(u), torch.where(r < p[2], p[0] * r * r / (2 * p[2]), p[0] * (r - 0.5 * p[2])))
        return torch.zeros_like(u)

    def f(self, l, u):
        """f_l(u), |f_l'(u)|"""
        if self.fk == "linear":
            return self.fp[l] * u, torch.full_like(u, abs(self.fp[l]))
        if self.fk == "burgers":
            return self.fp[0] * u * u, (2 * self.fp[0] * u).abs()
        if self.fk == "bl":
            f, d = _bl(u, self.fp[0], 1 if self.d == 1 else l)
            return f, d.abs()
        return torch.zeros_like(u), torch.zeros_like(u)

    def speed(self, l, a, b):
        """max |f_l'| between a and b"""
        best = torch.maximum(self.f(l, a)[1], self.f(l, b)[1])
        lo, hi = torch.minimum(a, b), torch.maximum(a, b)
        for c, v in self.crit.get(l, []):
            best = torch.where((lo < c) & (c < hi), best.clamp(min=v), best)
        return best

    def llf(self, l, a, b):
        return 0.5 * (self.f(l, a)[0] + self.f(l, b)[0]) - 0.5 * self.speed(l, a, b) * (b - a)

    def sh(self, x, l, k):
        return torch.roll(x, -k, dims=x.dim() - 1 - l) if k else x

    def at(self, table, f):
        kind, x = sum((f[l] & 1) << l for l in range(self.d)), None
        x = table[kind]
        for l in range(self.d):
            x = self.sh(x, l, f[l] >> 1)
        return x

    def offs(self, skip=None):
        """Simpson offsets and weights over the axes (skip: weight 1, offset 0 along it)"""
        out = [((), 1.0)]
        for l in range(self.d):
            out = [(o + (m,), w * ww) for o, w in out for m, ww in ([(0, 1.0)] if l == skip else [(-1, 1.0), (0, 4.0), (1, 1.0)])]
        return out

    def theta(self, lo, hi):
        u0, u1 = self.s.umin, self.s.umax
        den = torch.where(lo == hi, torch.ones_like(lo), lo - hi)
        t = torch.ones_like(lo)
        t = torch.where(hi < u0, ((lo - u0) / den).clamp(0.0, 1.0), t)
        t = torch.where(hi > u1, ((lo - u1) / den).clamp(0.0, 1.0), t)
        return torch.where(lo == hi, torch.ones_like(lo), t)

    def evaluate(self, st, tau, ext=None):
        """One limited forward-Euler evaluation on a periodic mesh."""
        d, s = self.d, self.s
        ub, nk = st[0], 1 << self.d
        z = list(st)
        acc = sum(w * self.at(z, o) for o, w in self.offs() if any(o))
        z[0] = (6.0 ** d * ub - acc) / 4.0 ** d
        av = [self.a(v) for v in z]
        au = self.a(ub)
        out = torch.zeros_like(ub)
        res = [None] * nk
        for l in range(d):
            h = self.h[l]
            mu, nu = tau / h, tau / (h * h)
            fd = [self.f(l, v) for v in z]
            fv, dv = [p[0] for p in fd], [p[1] for p in fd]
            e = lambda o, k: o[:l] + (o[l] + k,) + o[l + 1:]
            FH, AH = torch.zeros_like(ub), torch.zeros_like(ub)
            for o, w in self.offs(skip=l):
                FH = FH + w * self.at(fv, e(o, 1))
                AH = AH + w * (8.0 * self.at(av, o) - self.at(av, e(o, -1)) - self.at(av, e(o, 1))) / 6.0
            FH, AH = FH / 6.0 ** (d - 1), AH / 6.0 ** (d - 1)
            up, fu = self.sh(ub, l, 1), self.f(l, ub)[0]
            FL = self.llf(l, ub, up)
            aup, aum, FLm = self.sh(au, l, 1), self.sh(au, l, -1), self.sh(FL, l, -1)
            ulp = ub - 2 * d * mu * (FL - fu) + 2 * d * nu * (aup - au)
            ulm = ub - 2 * d * mu * (fu - FLm) - 2 * d * nu * (au - aum)
            tc = td = None
            if s.blend != "off":
                if ext is None:
                    um = self.sh(ub, l, -1)
                    r = (um - 2 * ub + up).abs() / (um.abs() + 2 * ub.abs() + up.abs() + 1e-13)
                    r = (self.sh(r, l, -1) + 4 * r + self.sh(r, l, 1)) / 6.0
                else:
                    r = ext
                tc, td = torch.exp(-s.gamma * 0.5 * (r + self.sh(r, l, 1))), torch.exp(-s.gamma * r)
                FH, AH = tc * FH + (1 - tc) * FL, td * AH + (1 - td) * au
            for k in range(1, nk):
                o = tuple((k >> t) & 1 for t in range(d))
                q = [e(o, t) for t in (-2, -1, 0, 1, 2)]
                Z, F, A = [self.at(z, t) for t in q], [self.at(fv, t) for t in q], [self.at(av, t) for t in q]
                al = self.at(dv, q[0])
                for t in q[1:]:
                    al = torch.maximum(al, self.at(dv, t))
                r = (16 * (A[1] + A[3]) - (A[0] + A[4]) - 30 * A[2]) / (3 * h * h) - (
                    (F[0] - F[4]) + 8 * (F[3] - F[1]) + al * ((Z[0] + Z[4]) - 4 * (Z[1] + Z[3]) + 6 * Z[2])) / (6 * h)
                if tc is not None:
                    w = tc if o[l] else td
                    for t in range(d):
                        if t != l and o[t]:
                            w = torch.minimum(w, self.sh(w, t, 1))
                    low = [ub] + list(st[1:])
                    zm, z0, zp = (self.at(low, e(o, t)) for t in (-1, 0, 1))
                    rl = (self.a(zp) - 2 * self.a(z0) + self.a(zm)) * 4 / (h * h) - (self.llf(l, z0, zp) - self.llf(l, zm, z0)) * 2 / h
                    r = w * r + (1 - w) * rl
                res[k] = r if res[k] is None else res[k] + r
            if s.limiter:
                kc, kd = 2 * d * self.parts * mu, 6 * d * nu
                dF, dA = FH - FL, kd * (AH - au)
                ulmp, ulpm = self.sh(ulm, l, 1), self.sh(ulp, l, -1)
                t = torch.minimum(self.theta(ulp, ulp - kc * dF), self.theta(ulmp, ulmp + kc * dF))
                FH = torch.where(t == 1, FH, FL + t * dF)
                t = torch.minimum(torch.minimum(self.theta(ulpm, ulpm + dA), self.theta(ulp, ulp - dA)),
                                  torch.minimum(self.theta(ulm, ulm - dA), self.theta(ulmp, ulmp + dA)))
                AH = torch.where(t == 1, AH, au + t * (AH - au))
            out = out - mu * (FH - self.sh(FH, l, -1)) + nu * (self.sh(AH, l, 1) - 2 * AH + self.sh(AH, l, -1))
        new = [ub + out]
        for k in range(1, nk):
            v = st[k] + tau * res[k]
            new.append(v.clamp(s.umin, s.umax) if s.limiter else v)
        return new

    def fe(self, st, tau, net=None):
        s, G = self.s, 5
        if s.bc == "periodic":
            return self.evaluate(st, tau, None if net is None else _network(net, _patches(st)))
        dev = st[0].device

        def cells(n):
            i = torch.arange(-G, n + G, device=dev) % (2 * n)
            return torch.where(i < n, i, 2 * n - 1 - i)

        def faces(n):   # stored index k holds the point at x0 + k h
            i = torch.arange(-G + 1, n + G + 1, device=dev) % (2 * n)
            return torch.where(i <= n, i, 2 * n - i)

        if s.bc == "dirichlet":
            gl, gr = (torch.full((G,), v, dtype=torch.float64, device=dev) for v in s.bc_values)
            new = self.evaluate([torch.cat([gl, st[0], gr]), torch.cat([gl[1:], st[1], gr])], tau)
            P = new[1][G - 1:G + s.nx].clone()
            P[0], P[-1] = s.bc_values
            return [new[0][G:G + s.nx], P]
        if self.d == 1:
            new = self.evaluate([st[0][cells(s.nx)], st[1][faces(s.nx)]], tau)
            return [new[0][G:G + s.nx], new[1][G - 1:G + s.nx]]
        cx, cy, fx, fy = cells(s.nx), cells(s.ny), faces(s.nx), faces(s.ny)
        new = self.evaluate([st[0][cy][:, cx], st[1][cy][:, fx], st[2][fy][:, cx], st[3][fy][:, fx]], tau)
        c, p = (lambda n: slice(G, G + n)), (lambda n: slice(G - 1, G + n))
        return [new[0][c(s.ny), c(s.nx)], new[1][c(s.ny), p(s.nx)], new[2][p(s.ny), c(s.nx)], new[3][p(s.ny), p(s.nx)]]

    def dt(self, ub):
        s, rate = self.s, 0.0
        for l in range(self.d):
            al = float(self.f(l, ub)[1].max())
            if s.bc == "dirichlet":
                g = torch.tensor(s.bc_values, dtype=torch.float64)
                al = max(al, float(self.f(l, g)[1].max()))
                ub = torch.cat([g[:1].to(ub), ub, g[1:].to(ub)])
            n = ub.shape[ub.dim() - 1 - l]
            a, b = ub, self.sh(ub, l, 1)
            if s.bc != "periodic":
                a, b = (x.narrow(x.dim() - 1 - l, 0, n - 1) for x in (a, b))
            if self.crit.get(l):
                al = max(al, float(self.speed(l, a, b).max()))
            rate = max(rate, al / self.h[l] + self.kmax / self.h[l] ** 2)
        cd = {1: (0.157, 0.333), 2: (0.0616, 0.1307), 3: (2.5127 / 63.335, 5.330 / 63.335)}[self.d][0 if s.rk == 3 else 1] * 0.9
        return 1.0 / max(rate / (0.33 / self.d), self.kmax / (min(self.h) ** 2 * cd))

    def step(self, u, dt, net=None):
        fe = lambda v, tau: self.fe(v, tau, net)
        mix = lambda *t: [sum(c * v[k] for c, v in t) for k in range(len(u))]
        if self.s.rk == 3:
            u1 = fe(u, dt)
            u2 = mix((0.75, u), (0.25, fe(u1, dt)))
            return mix((1.0 / 3.0, u), (2.0 / 3.0, fe(u2, dt)))
        # Spiteri and Ruuth's SSP-RK(5,4)
        u1 = fe(u, 0.391752226571890 * dt)
        r = lambda a, b: b / a * dt
        u2 = mix((0.444370493651235, u), (0.555629506348765, fe(u1, r(0.555629506348765, 0.368410593050371))))
        u3 = mix((0.620101851488403, u), (0.379898148511597, fe(u2, r(0.379898148511597, 0.251891774271694))))
        u4 = mix((0.178079954393132, u), (0.821920045606868, fe(u3, r(0.821920045606868, 0.544974750228521))))
        return mix((0.517231671970585, u2), (0.096059710526147, fe(u3, r(0.096059710526147, 0.063692468666290))),
                   (0.386708617503269, fe(u4, r(0.386708617503269, 0.226007483236906))))


def _bf16(x):
    return x.to(torch.float32).to(torch.bfloat16).to(torch.float64)


def _patches(st):
    """Normalised patch of every cell from the arrays by kind (ub, X, Y, V)."""
    ub, X, Y, V = st
    at = lambda x, i, j: torch.roll(x, (-j, -i), dims=(0, 1))
    p = [at(ub, i, j) for j in (-1, 0, 1) for i in (-1, 0, 1)] + [at(ub, -2, 0), at(ub, 2, 0), at(ub, 0, -2), at(ub, 0, 2)]
    p += [at(V, -1, -1), at(V, 0, -1), at(V, -1, 0), V, at(X, -1, 0), X, at(Y, 0, -1), Y]
    scale = p[0].abs()
    for v in p[1:]:
        scale = torch.maximum(scale, v.abs())
    return torch.stack([(v - ub) / (scale + 1e-13) for v in p], dim=-1)


def _layers(p):
    W1, b1, W2, b2, w3, b3 = torch.split(p, [672, 32, 1024, 32, 32, 1])
    return W1.view(32, 21), b1, W2.view(32, 32), b2, w3, b3


def _network(params, x):
    """The network with its rounding points: inputs, weights and activations of the two
    hidden layers in bfloat16."""
    W1, b1, W2, b2, w3, b3 = _layers(params)
    h1 = _bf16((_bf16(x) @ _bf16(W1).T + b1).clamp(min=0.0))
    h2 = (h1 @ _bf16(W2).T + b2).clamp(min=0.0)
    return torch.nn.functional.softplus(h2 @ w3 + b3, threshold=50.0)


def _by_kind(spec, st):
    return [st[0], st[2], st[3], st[1]] if spec.dim == 2 else st


def _as_stored(spec, st):
    return [st[0], st[3], st[1], st[2]] if spec.dim == 2 else st


def _padded(spec, st):
    """The device layout of a rectangle with ends: (ny + 1) x (nx + 1) entries per array."""
    out = []
    for x in st:
        y = torch.zeros((spec.ny + 1, spec.nx + 1), dtype=x.dtype, device=x.device)
        y[spec.ny + 1 - x.shape[0]:, spec.nx + 1 - x.shape[1]:] = x
        out.append(y)
    return out


def _splitmix64(z):
    with np.errstate(over="ignore"):
        z = z + np.uint64(0x9E3779B97F4A7C15)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        return z ^ (z >> np.uint64(31))


def _train(case, seed, feat, label):
    """Adam on minibatches drawn with splitmix64; the gradient of the mean squared error
    with the network's rounding points."""
    p = torch.tensor(_params(seed), dtype=torch.float64, device=feat.device)
    m, v, loss = torch.zeros_like(p), torch.zeros_like(p), 0.0
    n, batch = feat.shape[0], case["batch"]
    for t in range(case["steps"]):
        k = np.arange(batch, dtype=np.uint64) ^ np.uint64(seed + 1) ^ (np.uint64(t) << np.uint64(32))
        idx = torch.from_numpy((_splitmix64(k) % np.uint64(n)).astype(np.int64)).to(feat.device)
        x, y = _bf16(feat[idx]), label[idx]
        W1, b1, W2, b2, w3, b3 = _layers(p)
        z1 = x @ _bf16(W1).T + b1
        h1 = _bf16(z1.clamp(min=0.0))
        z2 = h1 @ _bf16(W2).T + b2
        h2 = z2.clamp(min=0.0)
        z3 = h2 @ w3 + b3
        r = torch.nn.functional.softplus(z3, threshold=50.0) - y
        loss = float((r * r).mean())
        d3 = 2.0 / batch * r * torch.sigmoid(z3)
        d2 = (d3[:, None] * w3) * (z2 > 0)
        d1 = (d2 @ _bf16(W2)) * (z1 > 0)
        g = torch.cat([(d1.T @ x).reshape(-1), d1.sum(0), (d2.T @ h1).reshape(-1), d2.sum(0), h2.T @ d3, d3.sum().reshape(1)])
        m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
        p = p - 3e-3 * (m / (1 - 0.9 ** (t + 1))) / (torch.sqrt(v / (1 - 0.999 ** (t + 1))) + 1e-8)
    return p, loss


def exact(case, seed):
    if case["kind"] == "batch":
        out = []
        for s, m in _batch_specs(case, seed):
            s.rk, s.blend = case["rk"], case["blend"]
            M, st = _Method(s), _by_kind(s, ai.batch_state(s, m, device=_device()))
            out.append(_as_stored(s, M.step(st, M.dt(st[0]))))
        return out
    spec = _spec(case)
    st = _by_kind(spec, _initial(spec, seed))
    if case["kind"] == "train":
        if case["precision"] != "fp64":
            st = [st[0]] + [a.to(torch.float32).double() for a in st[1:]]
        feat = _patches(st).reshape(-1, 21)
        ind = []
        for dim in (1, 0):
            u = st[0]
            um, up = torch.roll(u, 1, dims=dim), torch.roll(u, -1, dims=dim)
            r = (um - 2 * u + up).abs() / (um.abs() + 2 * u.abs() + up.abs() + 1e-13)
            ind.append((torch.roll(r, 1, dims=dim) + 4 * r + torch.roll(r, -1, dims=dim)) / 6.0)
        label = torch.maximum(*ind).reshape(-1)
        params, loss = _train(case, seed, feat, label)
        return {"params": params, "loss": loss, "feat": feat, "label": label}
    M = _Method(spec)
    dt = M.dt(st[0])
    if case["kind"] == "run":
        t, T, n = 0.0, (case["steps"] - 0.5) * dt, 0
        while t < T * (1.0 - 1e-14):
            tau = min(M.dt(st[0]), T - t)
            st, t, n = M.step(st, tau), t + tau, n + 1
        return {"state": _as_stored(spec, st), "steps": n}
    net = torch.tensor(_params(seed), dtype=torch.float64, device=st[0].device) if case["blend"] == "learned" else None
    st = _as_stored(spec, M.step(st, dt, net))
    return _padded(spec, st) if spec.dim == 2 and spec.bc != "periodic" else st
