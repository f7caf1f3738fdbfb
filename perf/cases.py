"""The work that this framework is measured on: what its users have it do, through its public entry points.

Kinds of cases, with the part of the framework that each calls:

- "step": a solver (`vlbm.Solver`) advanced some RK3 steps, then its moments read (a simulation that looks at its
  fields every so often; one step and a look for a coupled program);
- "ensemble": many runs of uneven grids advanced together (`vlbm.Batch`), then every run's moments;
- "rollout": a coarse solver with the learned correction after every step (`LearnedCorrection.rollout`);
- "train": optimiser steps of the correction network on samples (`LearnedCorrection.train_step`), then its weights;
- "gradients": loss and gradient of one sample (`LearnedCorrection.gradients`) and its prediction;
- "diagnostics": conserved sums of a population array that the caller owns on the device
  (`vlbm_diagnostics_noalloc`);
- "checkpoint": populations set, one step, diagnostics, populations read (restart, coarse-graining of fine runs).

The FP32 solver's numbers are handed on in FP32 (its moments come as FP64 host arrays that hold FP32-accurate values).
"""
import math

import numpy as np
import torch

from paper_2504_15574_gb300 import inputs, learned, vlbm

VMAX = {"d2q16": math.sqrt(3.0 + math.sqrt(6.0)), "d2q9": math.sqrt(3.0)}
#: cell-steps of the largest listed case; drawn ones stay below
MOST_CELL_STEPS = 1024 * 2048 * 64


def _step(name, nt, np_, steps, tau, precision="fp32", scheme="weno5", komissarov=False, vset="d2q16", polar=False,
          field="vortices", read="moments"):
    return {"name": name, "kind": "step", "nt": nt, "np": np_, "steps": steps, "tau": tau, "precision": precision,
            "scheme": scheme, "komissarov": komissarov, "vset": vset, "polar": polar, "field": field, "read": read}


def listed():
    return [
        # the FP64 shear-decay configuration (32 x 64, tau = 0.02), a piece of its 500 steps: the default precision
        _step("fp64_32x64", 32, 64, 20, 0.02, precision="fp64", field="waves"),
        # the FP64 sound / shear configuration (256 x 512)
        _step("fp64_256x512", 256, 512, 2, 0.02, precision="fp64", field="waves"),
        # the smallest call: one FP32 step of a small ragged grid and a look at everything (a coupled program)
        _step("fp32_40x100_one", 40, 100, 1, 0.02, read="populations"),
        # a coarse FP32 run between two looks, the learned-coarse grid (128 x 256)
        _step("fp32_128x256", 128, 256, 200, 2e-3),
        # a 1-degree grid with an odd row count, the polar filter on (dt follows the theta spacing)
        _step("fp32_181x384_polar", 181, 384, 100, 5e-3, polar=True),
        # the throughput workload (1024 x 2048 shock, WENO-5, polar filter, T = 1.5 in the cap)
        _step("fp32_shock_1024x2048", 1024, 2048, 64, 1e-3, polar=True, field="shock"),
        # the upwind scheme with the Komissarov flux, as the schemes are compared
        _step("fp32_u3k_512x1024", 512, 1024, 100, 2e-3, scheme="u3", komissarov=True, polar=True),
        # the nine-velocity set on the sound / shear grid
        _step("fp32_d2q9_256x512", 256, 512, 100, 5e-3, vset="d2q9"),
        # the mixed-grid vortex ensemble (64x128 to 512x1024 in equal counts), fewer runs of each class
        {"name": "ensemble_16_runs", "kind": "ensemble", "runs": 4, "smallest": 64, "classes": 4, "steps": 20,
         "tau": 2e-3, "polar": False, "scheme": "weno5", "vset": "d2q16"},
        # the learned correction's rollout on its grid
        {"name": "rollout_128x256", "kind": "rollout", "nt": 128, "np": 256, "steps": 100, "tau": 2e-3,
         "form": "direct"},
        # its training: one optimiser step per sample
        {"name": "train_128x256", "kind": "train", "nt": 128, "np": 256, "steps": 4, "form": "direct"},
        # the conserved sums of a device array, in a program with its own memory pool
        {"name": "diagnostics_512x1024", "kind": "diagnostics", "nt": 512, "np": 1024},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _columns(rng, nt, polar):
    """An even column count near 1 to 2 times the rows. With the polar filter a multiple of the widest ring block that
    its rule asks for (at least n_phi / 4 pi, a power of two): with fewer factors of two the long time step is unstable."""
    np_ = 2 * _log(rng, nt // 2, nt)
    unit = 2
    while polar and unit * 4.0 * math.pi < 1.1 * np_:
        unit *= 2
    return max(unit, (np_ + unit // 2) // unit * unit)


def draw(rng):
    kind = rng.choice(["fp64", "fp32", "fp32", "fp32", "ensemble", "rollout", "train", "gradients", "diagnostics",
                       "checkpoint"])
    if kind == "fp64":
        nt = _log(rng, 12, 400)
        polar = rng.random() < 0.3
        np_ = _columns(rng, nt, polar)
        c = _step("", nt, np_, 1, rng.choice([5e-3, 0.02]), precision="fp64", polar=polar,
                  vset="d2q9" if rng.random() < 0.25 else "d2q16", field=rng.choice(["waves", "vortices"]))
        if rng.random() < 0.25:
            c.update(scheme="u3", komissarov=True)
        c["steps"] = max(1, min(20, int(256 * 512 * 2 / (nt * np_))))
    elif kind == "fp32":
        nt = _log(rng, 24, 1024)
        polar = rng.random() < 0.5
        np_ = _columns(rng, nt, polar)
        c = _step("", nt, np_, 1, rng.choice([1e-3, 2e-3, 5e-3, 0.02]), polar=polar,
                  field=rng.choice(["vortices", "shock"]))
        o = rng.random()
        if o < 0.3:
            c.update(scheme="u3", komissarov=rng.random() < 0.5)
        elif o < 0.4:
            c.update(komissarov=True)
        if rng.random() < 0.25:
            c.update(vset="d2q9")
        c["steps"] = max(1, min(200, rng.choice([1, 30, 100, 200]), int(MOST_CELL_STEPS / (2 * nt * np_))))
    elif kind == "ensemble":
        c = {"kind": "ensemble", "runs": rng.randint(1, 6), "smallest": rng.choice([32, 48, 64, 96]),
             "classes": rng.randint(2, 3), "steps": rng.choice([5, 20, 40]), "tau": 2e-3, "polar": rng.random() < 0.5,
             "scheme": rng.choice(["weno5", "weno5", "u3"]), "vset": rng.choice(["d2q16", "d2q16", "d2q9"])}
    elif kind == "rollout":
        nt = _log(rng, 32, 200)
        c = {"kind": "rollout", "nt": nt, "np": 2 * nt, "steps": rng.choice([10, 50, 100]), "tau": 2e-3,
             "form": rng.choice(["direct", "direct", "stream", "vorticity"])}
    elif kind in ("train", "gradients"):
        nt = _log(rng, 16, 200)
        c = {"kind": kind, "nt": nt, "np": 2 * nt + 2 * rng.randint(0, 3),
             "form": rng.choice(["direct", "direct", "stream", "vorticity"])}
        if kind == "train":
            c["steps"] = rng.randint(1, 4)
    elif kind == "diagnostics":
        nt = _log(rng, 16, 800)
        c = {"kind": "diagnostics", "nt": nt, "np": max(2, _log(rng, nt, 2 * nt))}
    else:
        nt = _log(rng, 24, 256)
        c = {"kind": "checkpoint", "nt": nt, "np": _columns(rng, nt, False), "tau": 5e-3,
             "precision": rng.choice(["fp32", "fp32", "fp64"])}
    c.pop("name", None)
    return c


# ---- inputs --------------------------------------------------------------------------------------------------------

def _field(nt, np_, field, seed):
    """(rho, u^theta, u^phi, T or None) host arrays of one start."""
    if field == "shock":
        # a hot dense cap of radius 0.2 about a random centre, smoothly off the grid's axis
        rng = np.random.default_rng(seed)
        z, ph0 = rng.uniform(-0.9, 0.9), rng.uniform(0.0, 2.0 * math.pi)
        th, ph = inputs.cell_centres(nt, np_)
        cosd = np.cos(th)[:, None] * z + np.sin(th)[:, None] * math.sqrt(1 - z * z) * np.cos(ph[None, :] - ph0)
        inside = cosd > math.cos(0.2)
        zero = np.zeros((nt, np_))
        # a gentle swirl everywhere, so that no part of the sphere is exactly at rest
        return (np.where(inside, 4.0, 1.0), zero, 0.05 * np.sin(th)[:, None] + zero,
                np.where(inside, 1.5, 1.0))
    rho, ut, up, _ = inputs.gaussian_vortices(nt, np_, run=seed)
    rho = rho + 1e-3 * inputs.legendre_field(nt, np_, 2 + seed % 3)
    if field == "waves":
        _, vt, vp, _ = inputs.shear_legendre(nt, np_, 3)
        a = 0.1 + 0.01 * (seed % 7)
        return rho, a * ut + vt, a * up + vp, None
    return rho, ut, up, None


def _dt(c, nt=None, np_=None):
    vs = vlbm.VLBM_D2Q9 if c.get("vset") == "d2q9" else vlbm.VLBM_D2Q16
    return vlbm.vlbm_max_stable_dt(nt or c["nt"], np_ or c["np"], c["tau"], polar_filter=c.get("polar", False),
                                   velocity_set=vs)


def _solver(c):
    return vlbm.Solver(c["nt"], c["np"], c["tau"], _dt(c), precision=c.get("precision", "fp32"),
                       polar_filter=c.get("polar", False), scheme=c.get("scheme", "weno5"),
                       komissarov=c.get("komissarov", False), velocity_set=c.get("vset", "d2q16"))


def _grids(c):
    return [(c["smallest"] << k, c["smallest"] << (k + 1)) for k in range(c["classes"]) for _ in range(c["runs"])]


def _samples(c, seed, count):
    """Moments of a coarse run and small smooth targets, [N, 4, H, W] and [N, 3, H, W]."""
    H, W = c["nt"], c["np"]
    th, ph = inputs.cell_centres(H, W)
    X, Y = [], []
    for k in range(count):
        rho, ut, up, _ = _field(H, W, "vortices", seed + 101 * k)
        # waves of about ten cells, the short scales that a coarse run carries (and its error comes from)
        short = np.sin(th)[:, None] ** 2 * np.cos(0.6 * np.arange(H) + k)[:, None] * np.cos(round(0.1 * W) * ph)[None, :]
        rho, ut, up = rho + 1e-4 * short, ut + 1e-3 * short, up - 1e-3 * np.roll(short, 2, 1)
        T = 1.0 + 0.1 * (rho - 1.0) + 0.1 * (ut * ut + up * up)
        X.append(np.stack([rho, ut, up, T]))
        m = 1 + (seed + k) % 4
        wave = np.sin(th)[:, None] ** m * np.cos(m * ph[None, :] + 0.7 * k)
        Y.append(np.stack([1e-8 * wave, 1e-6 * (wave + 20.0 * ut * wave), 1e-6 * (wave - 20.0 * up * wave)]))
    return np.array(X), np.array(Y)


def _scales(c, X, Y):
    setup = learned.Setup(coarse=(c["nt"], c["np"]), polar_filter=False)
    ins, outs = learned.scales(X, Y)
    if c["form"] == "stream":
        outs = [learned.stream_scale(setup, outs), outs[1], outs[2]]
    elif c["form"] == "vorticity":
        outs = [learned.vorticity_scale(setup, outs), outs[1], outs[2]]
    return ins, outs


def _net(c, seed):
    X, Y = _samples(c, seed, c["steps"] if c["kind"] == "train" else 1)
    # a rollout corrects the drift of one short step, about 1e-8 of a velocity
    ins, outs = _scales(c, X, 0.01 * Y if c["kind"] == "rollout" else Y)
    net = vlbm.LearnedCorrection(c["nt"], c["np"], seed=1 + seed % 1000, in_scale=ins, out_scale=outs, form=c["form"])
    return net, X, Y, ins, outs


def _populations(nt, np_, seed):
    """A D2Q16 population array [16][nt][np] near equilibrium (FP64, host)."""
    rho, ut, up, _ = _field(nt, np_, "vortices", seed)
    v, w, _, _ = _velocities("d2q16")
    f = np.empty((16, nt, np_))
    for k in range(16):
        xi = v[k // 4] * ut + v[k % 4] * up
        f[k] = w[k // 4] * w[k % 4] * rho * (1.0 + xi + 0.5 * (xi * xi - ut * ut - up * up)) + 1e-6 * math.cos(k) * ut
    return f


def prepare(case, seed):
    c = dict(case)
    kind = c["kind"]
    if kind == "step":
        s = _solver(c)
        s.init_moments(*_field(c["nt"], c["np"], c["field"], seed))
        return {"case": c, "solver": s}
    if kind == "ensemble":
        grids = _grids(c)
        b = vlbm.Batch(grids, c["tau"], [_dt(c, *g) for g in grids], polar_filter=c["polar"], scheme=c["scheme"],
                       komissarov=False, velocity_set=c["vset"], guard=False)
        for r, g in enumerate(grids):
            b.init_moments(r, *_field(*g, "vortices", seed + 31 * r)[:3])
        # one CTA per tile, the schedule that the autotuner takes for mixes like this one
        b.set_schedule(8, -1)
        return {"case": c, "batch": b}
    if kind == "rollout":
        net = _net(c, seed)[0]
        s = vlbm.Solver(c["nt"], c["np"], c["tau"], _dt(c), precision="fp32", guard=False)
        s.init_moments(*_field(c["nt"], c["np"], "vortices", seed))
        return {"case": c, "solver": s, "net": net}
    if kind in ("train", "gradients"):
        net, X, Y, _, _ = _net(c, seed)
        return {"case": c, "net": net, "X": X, "Y": Y}
    f = _populations(c["nt"], c["np"], seed)
    if kind == "diagnostics":
        return {"case": c, "f": torch.from_numpy(f).cuda(), "out": torch.zeros(6, dtype=torch.float64, device="cuda")}
    s = _solver(c)
    s.set_populations(f)
    return {"case": c, "solver": s, "f": f}


# ---- the passes ----------------------------------------------------------------------------------------------------

def _fp32(arrays):
    return [torch.from_numpy(a).float() for a in arrays]


def run(state):
    c = state["case"]
    kind = c["kind"]
    if kind == "step":
        s = state["solver"]
        s.step(c["steps"])
        out = [s.get_populations()] if c["read"] == "populations" else s.moments()
        return list(out) if c["precision"] == "fp64" else _fp32(out)
    if kind == "ensemble":
        b = state["batch"]
        b.step(c["steps"])
        return [_fp32(b.moments(r)) for r in range(len(b))]
    if kind == "rollout":
        s = state["solver"]
        state["net"].rollout(s, c["steps"])
        return _fp32(s.moments(with_T=True))
    if kind == "train":
        net = state["net"]
        losses = [net.train_step(x, y, 1e-3) for x, y in zip(state["X"], state["Y"])]
        return [np.asarray(losses, dtype=np.float32), net.get_weights()]
    if kind == "gradients":
        net, x, y = state["net"], state["X"][0], state["Y"][0]
        loss, g = net.gradients(x, y)
        return [np.float32(loss), g, torch.from_numpy(net.predict(x) / net.out_scale[1]).float()]
    if kind == "diagnostics":
        f, out = state["f"], state["out"]
        vlbm.vlbm_diagnostics_noalloc(f.data_ptr(), c["nt"], c["np"], 1.0, out.data_ptr(),
                                      torch.cuda.current_stream().cuda_stream)
        return [out[0], out[1:4], out[4:5], out[5]]
    s = state["solver"]
    s.set_populations(state["f"])
    s.step(1)
    d = s.diagnostics()
    sums = np.array([d["mass"], d["energy"]])
    f = s.get_populations()
    return [sums, f] if c["precision"] == "fp64" else _fp32([sums, f])


# ---- what a pass cannot do without ---------------------------------------------------------------------------------

def _stage_work(cells, vset, steps, scheme, elem):
    q = 9 if vset == "d2q9" else 16
    # per population and stage: two interface values (WENO-5 about 50 operations, an upwind stencil 5), their
    # differences, the force's two short dot products, the equilibrium, the stage combination
    flops = q * (2 * (50 if scheme == "weno5" else 5) + 4 * (2 * int(math.sqrt(q))) + 24)
    # per step: three stages read their input and write their output, the last two read the step's start too
    return {"bytes": 8.0 * q * elem * cells * steps, "flops": 3.0 * flops * cells * steps}


def _net_macs(cells):
    return cells * 9 * (16 * 32 + 2 * 32 * 32 + 32 * 3)


def work(case):
    c = case
    kind = c["kind"]
    if kind in ("step", "checkpoint"):
        cells = c["nt"] * c["np"]
        elem = 8 if c.get("precision") == "fp64" else 4
        w = _stage_work(cells, c.get("vset", "d2q16"), c.get("steps", 1), c.get("scheme", "weno5"), elem)
        if kind == "checkpoint":
            w["bytes"] += 2.0 * 16 * 8 * cells
        elif c["read"] == "populations":
            w["bytes"] += 16.0 * 8 * cells
        else:
            w["bytes"] += 3.0 * 8 * cells
        return w
    if kind == "ensemble":
        cells = sum(a * b for a, b in _grids(c))
        w = _stage_work(cells, c["vset"], c["steps"], c["scheme"], 4)
        w["bytes"] += 3.0 * 8 * cells
        return w
    cells = c["nt"] * c["np"]
    if kind == "rollout":
        w = _stage_work(cells, "d2q16", c["steps"], "weno5", 4)
        w["bytes"] += c["steps"] * 2.0 * 64 * cells + 4.0 * 8 * cells
        w["flops"] += c["steps"] * 2.0 * _net_macs(cells)
        return w
    if kind in ("train", "gradients"):
        n = c.get("steps", 1)
        return {"bytes": n * 7.0 * 8 * cells, "flops": n * 6.0 * _net_macs(cells)}
    return {"bytes": 16.0 * 8 * cells, "flops": 16.0 * 8 * cells}


# ---- the same in 64 bits, without the framework -------------------------------------------------------------------

def _device():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _velocities(vset):
    """v, w, K, Kt of the Gauss-Hermite set: roots of He_Q, weights Q! / He_{Q+1}^2, derivative kernels."""
    q = 3 if vset == "d2q9" else 4
    if q == 3:
        v = np.array([-math.sqrt(3.0), 0.0, math.sqrt(3.0)])
    else:
        a, b = math.sqrt(3.0 + math.sqrt(6.0)), math.sqrt(3.0 - math.sqrt(6.0))
        v = np.array([-a, -b, b, a])
    he = [np.ones_like(v), v]
    for n in range(1, q + 1):
        he.append(v * he[n] - n * he[n - 1])
    w = math.factorial(q) / he[q + 1] ** 2
    K, Kt = np.zeros((q, q)), np.zeros((q, q))
    for n in range(q):
        K -= np.outer(w * he[n + 1], he[n]) / math.factorial(n)
        Kt -= np.outer(w * he[n + 1], he[n + 1] + (n * he[n - 1] if n else 0.0)) / math.factorial(n)
    return v, w, K, Kt


class _Sphere:
    """The scheme on dense FP64 tensors: f [Q^2][nt][np]."""

    def __init__(self, nt, np_, tau, dt, scheme="weno5", komissarov=False, vset="d2q16", polar=False, eps=1e-6):
        self.nt, self.np, self.tau, self.dt, self.eps = nt, np_, tau, dt, eps
        self.scheme, self.kom = scheme, komissarov
        v, w, K, Kt = _velocities(vset)
        self.q = len(v)
        q = self.q
        dev = self.dev = _device()
        t = lambda a: torch.tensor(np.asarray(a), dtype=torch.float64, device=dev)  # noqa: E731
        self.va, self.vb = t(np.repeat(v, q)), t(np.tile(v, q))
        self.w = t(np.outer(w, w).reshape(-1)).view(-1, 1, 1)
        self.K, self.Kt = t(K), t(Kt)
        self.dth, self.dph = math.pi / nt, 2.0 * math.pi / np_
        th = (np.arange(nt) + 0.5) * self.dth
        half = np.arange(nt) >= (nt + 1) // 2
        mirror = (np.arange(nt)[::-1] + 0.5) * self.dth
        s = np.where(half, np.sin(mirror), np.sin(th))
        co = np.where(half, -np.cos(mirror), np.cos(th))
        if nt % 2:
            co[nt // 2] = 0.0
        self.s, self.cot = t(s).view(1, -1, 1), t(co / s).view(1, -1, 1)
        self.s_ext = t(np.concatenate([-s[:3][::-1], s, -s[-3:][::-1]])).view(1, -1, 1)
        fi = np.arange(nt + 1) * self.dth
        sf, cf = np.sin(fi), np.cos(fi)
        sf[0] = sf[-1] = 0.0
        self.sf, self.dcos = t(sf).view(1, -1, 1), t(cf[:-1] - cf[1:]).view(1, -1, 1)
        self.rows = []
        if polar and np_ >= 2:
            for i in range(nt):
                b, want = 1, self.dth / (4.0 * s[i] * self.dph)
                while b < want and b < np_:
                    b *= 2
                while np_ % b:
                    b //= 2
                if b > 1:
                    self.rows.append((i, b))

    def _value(self, a, b, c, d, e):
        if self.scheme == "u1":
            return c
        if self.scheme == "u2":
            return 1.5 * c - 0.5 * b
        if self.scheme == "u3":
            return (2.0 * d + 5.0 * c - b) / 6.0
        s1 = 13.0 / 12.0 * (a - 2 * b + c) ** 2 + 0.25 * (a - 4 * b + 3 * c) ** 2
        s2 = 13.0 / 12.0 * (b - 2 * c + d) ** 2 + 0.25 * (b - d) ** 2
        s3 = 13.0 / 12.0 * (c - 2 * d + e) ** 2 + 0.25 * (3 * c - 4 * d + e) ** 2
        w1, w2, w3 = 0.1 / (s1 + self.eps) ** 2, 0.6 / (s2 + self.eps) ** 2, 0.3 / (s3 + self.eps) ** 2
        num = w1 * (2 * a - 7 * b + 11 * c) + w2 * (-b + 5 * c + 2 * d) + w3 * (2 * c + 5 * d - e)
        return num / (6.0 * (w1 + w2 + w3))

    def tendency(self, f):
        nt, np_, q = self.nt, self.np, self.q
        n = f.sum(0)
        ut, up = torch.einsum("k,kij->ij", self.va, f) / n, torch.einsum("k,kij->ij", self.vb, f) / n
        xi = self.va.view(-1, 1, 1) * ut + self.vb.view(-1, 1, 1) * up
        u2 = ut * ut + up * up
        poly = 1.0 + xi + 0.5 * (xi * xi - u2)
        if q == 4:
            poly = poly + xi * (xi * xi - 3.0 * u2) / 6.0
        L = (self.w * n * poly - f) / self.tau
        g = f.view(q, q, nt, np_)
        kg = torch.einsum("am,mbij->abij", self.K, g).reshape(-1, nt, np_)
        ktg = torch.einsum("bm,amij->abij", self.Kt, g).reshape(-1, nt, np_)
        L -= self.cot * (self.vb.view(-1, 1, 1) ** 2 * kg - self.va.view(-1, 1, 1) * ktg)
        del kg, ktg, xi, poly
        # the pole condition: a row beyond a pole is the mirrored row of the reversed population, half way round
        back = torch.roll(torch.flip(f, (0,)), -(np_ // 2), 2)
        e = torch.cat([torch.flip(back[:, :3], (1,)), f, torch.flip(back[:, -3:], (1,))], 1)
        if not self.kom:
            e = e * self.s_ext
        for sign in (1, -1):
            k = torch.nonzero(self.va * sign > 0).flatten()
            if len(k):
                x = e[k]
                cut = [x[:, m:m + nt + 1] for m in range(6)]
                r = self._value(*(cut[:5] if sign > 0 else cut[:0:-1])) * self.va[k].view(-1, 1, 1)
                if self.kom:
                    L[k] -= ((r * self.sf)[:, 1:] - (r * self.sf)[:, :-1]) / self.dcos
                else:
                    L[k] -= (r[:, 1:] - r[:, :-1]) / (self.s * self.dth)
            k = torch.nonzero(self.vb * sign > 0).flatten()
            if len(k):
                x = f[k]
                # the interface between columns j - 1 and j
                cut = [torch.roll(x, 3 - m, 2) for m in range(6)]
                r = self._value(*(cut[:5] if sign > 0 else cut[:0:-1])) * self.vb[k].view(-1, 1, 1)
                L[k] -= (torch.roll(r, -1, 2) - r) / (self.s * self.dph)
        return L

    def smooth(self, f):
        for i, b in self.rows:
            m = f[:, i].reshape(f.shape[0], self.np // b, b).mean(2, keepdim=True)
            f[:, i] = m.expand(-1, -1, b).reshape(f.shape[0], self.np)
        return f

    def step(self, f):
        f1 = self.smooth(f + self.dt * self.tendency(f))
        f2 = self.smooth(0.75 * f + 0.25 * f1 + 0.25 * self.dt * self.tendency(f1))
        return self.smooth(f / 3.0 + 2.0 / 3.0 * f2 + 2.0 / 3.0 * self.dt * self.tendency(f2))

    def start(self, rho, ut, up, T=None):
        t = lambda a: torch.from_numpy(np.array(a)).to(self.dev)  # noqa: E731
        rho, ut, up = t(rho), t(ut), t(up)
        dT = t(T) - 1.0 if T is not None else torch.zeros_like(rho)
        va, vb = self.va.view(-1, 1, 1), self.vb.view(-1, 1, 1)
        xi, u2, v2 = va * ut + vb * up, ut * ut + up * up, va * va + vb * vb
        poly = 1.0 + xi + 0.5 * (xi * xi - u2 + dT * (v2 - 2.0))
        if self.q == 4:
            poly = poly + (xi * (xi * xi - 3.0 * u2) + 3.0 * dT * xi * (v2 - 4.0)) / 6.0
        return self.w * rho * poly

    def equilibrium(self, rho, ut, up):
        xi = self.va.view(-1, 1, 1) * ut + self.vb.view(-1, 1, 1) * up
        u2 = ut * ut + up * up
        return self.w * rho * (1.0 + xi + 0.5 * (xi * xi - u2) + xi * (xi * xi - 3.0 * u2) / 6.0)

    def moments(self, f):
        n = f.sum(0)
        ut, up = torch.einsum("k,kij->ij", self.va, f) / n, torch.einsum("k,kij->ij", self.vb, f) / n
        va, vb = self.va.view(-1, 1, 1), self.vb.view(-1, 1, 1)
        T = (f * ((va - ut) ** 2 + (vb - up) ** 2)).sum(0) / (2.0 * n)
        return n, ut, up, T

    def sums(self, f):
        """Mass, Cartesian momentum and energy."""
        area = self.s[0] * self.dth * self.dph
        n, ut, up, _ = self.moments(f)
        th = torch.atan2(self.s[0], self.cot[0] * self.s[0])
        ph = (torch.arange(self.np, device=self.dev, dtype=torch.float64).view(1, -1) + 0.5) * self.dph
        p = [(n * (ut * torch.cos(th) * torch.cos(ph) - up * torch.sin(ph)) * area).sum(),
             (n * (ut * torch.cos(th) * torch.sin(ph) + up * torch.cos(ph)) * area).sum(),
             (-n * ut * torch.sin(th) * area).sum()]
        v2 = (self.va ** 2 + self.vb ** 2).view(-1, 1, 1)
        return (n * area).sum(), torch.stack(p), 0.5 * (f * v2 * area).sum()


def _bf16(x):
    """x rounded to bfloat16, its derivative passed on."""
    return x + (x.detach().float().bfloat16().double() - x.detach())


class _Net:
    """The correction network in FP64 arithmetic on what its format stores: features, weights, hidden activations and
    the gradients at the layers' sums are bfloat16 values."""
    SHAPES = ((16, 32), (32, 32), (32, 32), (32, 3))
    D4, D6 = (1.0, -4.0, 6.0, -4.0, 1.0), (1.0, -6.0, 15.0, -20.0, 15.0, -6.0, 1.0)

    def __init__(self, H, W, weights, ins, outs, form):
        dev = self.dev = _device()
        self.H, self.W, self.form = H, W, form
        self.p = torch.tensor(weights, dtype=torch.float64, device=dev)
        self.ins = torch.tensor(ins, dtype=torch.float64, device=dev)
        # scales are held in 32 bits
        self.outs = torch.tensor(np.asarray(outs, dtype=np.float32).astype(np.float64), device=dev)
        th = (torch.arange(H, dtype=torch.float64, device=dev) + 0.5) * math.pi / H
        self.sin, self.cos = torch.sin(th).view(-1, 1), torch.cos(th).view(-1, 1)
        self.dth, self.dph = math.pi / H, 2.0 * math.pi / W
        self.inv = None

    def _rows(self, a, h, odd):
        """h rows beyond each pole: mirrored, half way round, odd channels negated."""
        o = torch.roll(a, -(self.W // 2), -1) * (-1.0 if odd else 1.0)
        return torch.cat([torch.flip(o[..., :h, :], (-2,)), a, torch.flip(o[..., -h:, :], (-2,))], -2)

    def _difference(self, a, odd, st, axis):
        h = len(st) // 2
        if axis:
            return sum(w * torch.roll(a, h - m, -1) for m, w in enumerate(st))
        e = self._rows(a, h, odd)
        return sum(w * e[m:m + self.H] for m, w in enumerate(st))

    def features(self, rho, ut, up, T):
        d = [(rho, False, self.D6), (ut, True, self.D6), (up, True, self.D6), (ut, True, self.D4), (up, True, self.D4)]
        raw = [rho - 1.0, ut, up, T - 1.0] + [self._difference(a, o, st, ax) for a, o, st in d for ax in (0, 1)]
        x = [torch.clamp(r / s, -8.0, 8.0) for r, s in zip(raw, self.ins)]
        one = torch.ones_like(rho)
        return torch.stack(x[:4] + [self.cos * one, self.sin * one] + x[4:])

    def forward(self, x, p=None):
        p, o = self.p if p is None else p, 0
        x = _bf16(x)
        odd = torch.ones(16, dtype=torch.float64, device=self.dev)
        odd[[1, 2, 5] + list(range(8, 16))] = -1.0
        for layer, (ci, co) in enumerate(self.SHAPES):
            w = _bf16(p[o:o + co * ci * 9]).view(co, ci, 3, 3)
            b = p[o + co * ci * 9:o + co * ci * 9 + co]
            o += co * ci * 9 + co
            back = torch.roll(x, -(self.W // 2), -1)
            if layer == 0:
                back = back * odd.view(-1, 1, 1)
            e = torch.cat([back[:, :1], x, back[:, -1:]], 1)
            e = torch.cat([e[..., -1:], e, e[..., :1]], -1)
            y = b.view(-1, 1, 1)
            for t in range(9):
                y = y + torch.einsum("oc,cij->oij", w[:, :, t // 3, t % 3], e[:, t // 3:t // 3 + self.H, t % 3:t % 3 + self.W])
            if y.requires_grad:
                y.register_hook(lambda g: g.float().bfloat16().double())
            x = _bf16(torch.relu(y)) if layer < 3 else y
        return x

    def _curl(self, psi):
        e = self._rows(psi, 1, False)
        return torch.stack([(torch.roll(psi, -1, 1) - torch.roll(psi, 1, 1)) / (2.0 * self.dph * self.sin),
                            -(e[2:] - e[:-2]) / (2.0 * self.dth)])

    def _poisson(self, w):
        H, W = self.H, self.W
        w = w - (w * self.sin).sum() / (self.sin.sum() * W)
        if self.inv is None:
            s = self.sin.flatten()
            sf = torch.sin(torch.arange(H + 1, dtype=torch.float64, device=self.dev) * self.dth)
            sf[0] = sf[-1] = 0.0
            lo, hi = sf[:-1] / (s * self.dth ** 2), sf[1:] / (s * self.dth ** 2)
            A = torch.diag(-(lo + hi)) + torch.diag(hi[:-1], 1) + torch.diag(lo[1:], -1)
            m = torch.arange(W // 2 + 1, dtype=torch.float64, device=self.dev)
            lam = (2.0 * torch.sin(0.5 * m * self.dph) / self.dph) ** 2
            A = A.unsqueeze(0) - torch.diag_embed(lam.view(-1, 1) / (s * s))
            A[0] += torch.outer(torch.ones_like(s), s)   # the constant of the axisymmetric mode
            self.inv = torch.linalg.inv(A)
        X = torch.fft.rfft(w, dim=1)
        re, im = torch.einsum("mij,jm->im", self.inv, X.real), torch.einsum("mij,jm->im", self.inv, X.imag)
        return torch.fft.irfft(torch.complex(re, im), n=W, dim=1)

    def correction(self, y):
        if self.form == "direct":
            return y * self.outs.view(-1, 1, 1)
        psi = y[0] * self.outs[0]
        if self.form == "vorticity":
            psi = self._poisson(psi)
        return torch.cat([torch.zeros_like(psi).unsqueeze(0), self._curl(psi)])

    def loss(self, x, target, p):
        w = self.sin / (self.sin.sum() * self.W)
        d = self.correction(self.forward(self.features(*x), p)) - target
        r = d / self.outs.view(-1, 1, 1)
        return (w * r ** 2).sum() / 3.0 if self.form == "direct" else 0.5 * (w * r[1:] ** 2).sum()

    def gradient(self, x, target):
        p = self.p.clone().requires_grad_(True)
        loss = self.loss(x, target, p)
        loss.backward()
        return loss.detach(), p.grad

    def train(self, X, Y, lr=1e-3, b1=0.9, b2=0.999, eps=1e-8):
        m, v = torch.zeros_like(self.p), torch.zeros_like(self.p)
        losses = []
        for t, (x, y) in enumerate(zip(X, Y), 1):
            loss, g = self.gradient(x, y)
            losses.append(loss)
            m, v = b1 * m + (1 - b1) * g, b2 * v + (1 - b2) * g * g
            self.p = self.p - lr * (m / (1 - b1 ** t)) / (torch.sqrt(v / (1 - b2 ** t)) + eps)
        return torch.stack(losses), self.p


def exact(case, seed):
    c = dict(case)
    kind = c["kind"]
    if kind == "step":
        sp = _Sphere(c["nt"], c["np"], c["tau"], _dt(c), c["scheme"], c["komissarov"], c["vset"], c["polar"])
        f = sp.start(*_field(c["nt"], c["np"], c["field"], seed))
        for _ in range(c["steps"]):
            f = sp.step(f)
        return [f] if c["read"] == "populations" else list(sp.moments(f)[:3])
    if kind == "ensemble":
        out = []
        for r, g in enumerate(_grids(c)):
            sp = _Sphere(*g, c["tau"], _dt(c, *g), c["scheme"], False, c["vset"], c["polar"])
            f = sp.start(*_field(*g, "vortices", seed + 31 * r))
            for _ in range(c["steps"]):
                f = sp.step(f)
            out.append(list(sp.moments(f)[:3]))
        return out
    if kind in ("diagnostics", "checkpoint"):
        sp = _Sphere(c["nt"], c["np"], c.get("tau", 1.0), _dt(c) if "tau" in c else 1.0)
        f = torch.from_numpy(_populations(c["nt"], c["np"], seed)).to(sp.dev)
        if kind == "checkpoint":
            f = sp.step(f)
            mass, _, energy = sp.sums(f)
            return [torch.stack([mass, energy]), f]
        mass, p, energy = sp.sums(f)
        return [mass, p, energy.view(1), None]
    net, X, Y, ins, outs = _net(c, seed)
    ref = _Net(c["nt"], c["np"], net.get_weights(), ins, outs, c["form"])
    net.close()
    t = lambda a: torch.from_numpy(a).to(ref.dev)  # noqa: E731
    if kind == "train":
        losses, p = ref.train([t(x) for x in X], [t(y) for y in Y])
        return [losses, p]
    if kind == "gradients":
        loss, g = ref.gradient(t(X[0]), t(Y[0]))
        y = ref.correction(ref.forward(ref.features(*t(X[0]))))
        return [loss, g, y / outs[1]]
    sp = _Sphere(c["nt"], c["np"], c["tau"], _dt(c))
    f = sp.start(*_field(c["nt"], c["np"], "vortices", seed))
    w = sp.s[0] / (sp.s.sum() * c["np"])
    for _ in range(c["steps"]):
        f = sp.step(f)
        rho, ut, up, T = sp.moments(f)
        d = ref.correction(ref.forward(ref.features(rho, ut, up, T)))
        drho = d[0] - (d[0] * w).sum()
        f = f + sp.equilibrium(rho + drho, ut + d[1], up + d[2]) - sp.equilibrium(rho, ut, up)
    return list(sp.moments(f))
