"""Workloads of the fine-burst engine, timed through its public binding.

Every case is a call that a user of the engine makes: one force evaluation,
one fine burst (plain, ramped, with mean positions), one coarse step, one
burst of a batch.  Shapes and lengths come from the benchmark's workloads
(10- to 49-cell cubes, replica ensembles, uneven batches), from the parity
tests (the small and ragged blocks) or are generic.

A pass continues the trajectory of the pass before it, as a run does; the
grip displacement changes sign from pass to pass, so that a specimen is
loaded and unloaded and stays intact however often it is run.

The mixed form forms its pair terms in FP32; its results are handed on as
float32.  The FP64 form's stay float64.
"""
import math

import numpy as np
import torch

import paper_2603_07321_gb300 as P

A0 = 4.05                    # lattice parameter, A
MASS = 26.9815385            # amu
KB = 1.380649e-23 / 1.602176634e-19                               # eV / K
MV2 = 1.66053906660e-27 * 1e-20 / 1e-30 / 1.602176634e-19          # amu A^2/fs^2 -> eV
GPA = 1.602176634e-19 / 1e-30 / 1e9                               # eV/A^3 -> GPa
EPS, PN, PM, RC = 3.3147e-2, 7, 6, 2.0 * A0
BASIS = ((0.0, 0.0, 0.0), (0.5, 0.5, 0.0), (0.5, 0.0, 0.5), (0.0, 0.5, 0.5))

# FP64 pair terms run at ~1/25 of the mixed form's rate per atom and step
FP64_COST = 25.0
MOST_ATOM_STEPS = 470596 * 200


def _one(kind, shape, prec, steps, T0=300.0, d_eps=1e-3, axis=2, **kw):
    return dict(kind=kind, nx=shape[0], ny=shape[1], nz=shape[2], prec=prec, steps=steps, T0=T0,
                d_eps=d_eps, axis=axis, **kw)


def listed():
    return [
        # one force and energy evaluation of a few hundred atoms in FP64: the
        # smallest call, what a user checks a configuration with
        dict(name="forces_fp64_5x4x6", **_one("forces", (5, 4, 6), "fp64", 1)),
        # the same on a ragged block of ordinary size, mixed precision
        dict(name="forces_mixed_25x17x31", **_one("forces", (25, 17, 31), "mixed", 1)),
        # a short burst of a small odd block: per-step latency
        dict(name="burst_mixed_6x5x7", **_one("burst", (6, 5, 7), "mixed", 100)),
        # the plain form: 4,000-atom cube in FP64, one tension step, one burst
        dict(name="burst_fp64_n10", **_one("burst", (10, 10, 10), "fp64", 400)),
        # the same cube in mixed precision: the smallest served specimen
        dict(name="burst_mixed_n10", **_one("burst", (10, 10, 10), "mixed", 400)),
        # the 8 nm cube of the paper, FP64 reference run
        dict(name="burst_fp64_n20", **_one("burst", (20, 20, 20), "fp64", 60)),
        # the 8 nm cube, mixed precision, cold and in compression
        dict(name="burst_mixed_n20", **_one("burst", (20, 20, 20), "mixed", 300, T0=100.0,
                                            d_eps=-1e-3)),
        # the 20 nm cube: the largest single specimen
        dict(name="burst_mixed_n49", **_one("burst", (49, 49, 49), "mixed", 200)),
        # continuous loading along x of an odd plate, with every atom's mean
        # position (verification runs)
        dict(name="ramp_mixed_30x23x9", **_one("ramp", (30, 23, 9), "mixed", 150, axis=0)),
        # one coarse step (three bursts and the slow-variable update): what
        # the server runs per specimen and tick
        dict(name="coarse_mixed_n15", **_one("coarse", (15, 15, 15), "mixed", 120)),
        # replica ensemble, one launch set per fine step
        dict(name="batch_mixed_12xn20", kind="batch", sizes=",".join(["20"] * 12), prec="mixed",
             steps=100, T0=300.0, d_eps=1e-3, axis=2),
        # uneven batch: what the server holds on the device at once
        dict(name="batch_mixed_uneven", kind="batch", sizes="10,13,15,20,25,30,40", prec="mixed",
             steps=80, T0=300.0, d_eps=1e-3, axis=2),
    ]


def draw(rng):
    kind = rng.choice(["forces", "burst", "burst", "burst", "ramp", "coarse", "batch"])
    prec = rng.choice(["fp64", "mixed", "mixed"])
    T0 = rng.choice([10.0, 100.0, 300.0])
    d_eps = rng.choice([-1.0, 1.0]) * 10.0 ** rng.uniform(-4.0, -3.0)
    side = lambda lo, hi: int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))  # noqa: E731
    top = 49 if prec == "mixed" else 24
    if kind == "batch":
        count = side(2, 12)
        sizes = [side(5, 30 if prec == "mixed" else 12) for _ in range(count)]
        atoms = sum(4 * n ** 3 for n in sizes)
    else:
        n = side(4, top)
        shape = [max(3, min(top, int(round(n * rng.uniform(0.6, 1.4))))) for _ in range(3)]
        atoms = 4 * shape[0] * shape[1] * shape[2]
    steps = side(40, 400)
    if kind == "coarse":
        steps = max(20, steps // 3)
    cost = atoms * (FP64_COST if prec == "fp64" else 1.0) * (3 if kind == "coarse" else 1)
    steps = max(4, min(steps, int(0.6 * MOST_ATOM_STEPS / cost)))
    if kind == "forces":
        steps = 1
    if kind == "batch":
        return dict(kind=kind, sizes=",".join(str(n) for n in sizes), prec=prec, steps=steps, T0=T0,
                    d_eps=d_eps, axis=2)
    return _one(kind, shape, prec, steps, T0=T0, d_eps=d_eps, axis=rng.choice([0, 1, 2, 2]))


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _shapes(case):
    if case["kind"] == "batch":
        return [(int(n),) * 3 for n in case["sizes"].split(",")]
    return [(case["nx"], case["ny"], case["nz"])]


def _sites(shape):
    k, j, i = np.meshgrid(np.arange(shape[2]), np.arange(shape[1]), np.arange(shape[0]),
                          indexing="ij")
    cells = np.stack([i.ravel(), j.ravel(), k.ravel()], axis=1).astype(np.float64)
    return (A0 * (cells[:, None, :] + np.array(BASIS)[None])).reshape(-1, 3)


def _state(shape, axis, T0, seed):
    """A thermal snapshot: sites displaced by the rms thermal amplitude at T0
    (0.1 A at 300 K), Maxwell-Boltzmann velocities, grips at rest.  Positions
    on a 2^-24 A grid and velocities in float32, which both forms hold
    exactly."""
    rng = np.random.default_rng(seed)
    site = _sites(shape)
    x = site[:, axis]
    flag = np.where(x <= A0 + 1e-6, 1, np.where(x >= x.max() - A0 - 1e-6, 2, 0))
    pos = site + rng.normal(0.0, 0.1 * math.sqrt(T0 / 300.0), size=site.shape)
    pos = np.round(pos * 2.0 ** 24) / 2.0 ** 24
    vel = rng.normal(0.0, math.sqrt(KB * T0 / (MASS * MV2)), size=site.shape)
    vel = vel.astype(np.float32).astype(np.float64)
    vel[flag != 0] = 0.0
    return pos, vel, flag


def _inputs(case, seed):
    return [_state(sh, case["axis"], case["T0"], [seed, i]) for i, sh in enumerate(_shapes(case))]


def _recorded_means(n):
    """Slow variables of an earlier coarse step (K, U in eV, T in GPa)."""
    return np.array([[0.018 * n, -3.10 * n, 0.10], [0.018 * n, -3.10 * n, 0.11],
                     [0.018 * n, -3.10 * n, 0.12]])


def prepare(case, seed):
    prec = P.PREC_FP64 if case["prec"] == "fp64" else P.PREC_MIXED
    ctxs = []
    for shape, (pos, vel, _) in zip(_shapes(case), _inputs(case, seed)):
        # a coarse step of h = 1 s moves the grip by strain_rate * h
        c = P.Ctx(shape, T0=case["T0"], seed=seed, precision=prec, load_axis=case["axis"],
                  burst_steps=case["steps"], strain_rate=0.1 * case["d_eps"],
                  mean_positions=1 if case["kind"] == "ramp" else 0)
        c.set_state(pos, vel)
        if case["kind"] == "coarse":
            c.coarse_update(_recorded_means(c.n))
        ctxs.append(c)
    s = {"case": case, "ctx": ctxs, "sign": 1.0}
    if case["kind"] == "batch":
        s["batch"] = P.Batch(ctxs)
    return s


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def run(state):
    case, ctx = state["case"], state["ctx"][0]
    steps, kind = case["steps"], case["kind"]
    d = case["d_eps"] * state["sign"]
    state["sign"] = -state["sign"]
    as_type = (lambda a: a) if case["prec"] == "fp64" else (lambda a: np.asarray(a, np.float32))
    if kind == "forces":
        f, pe, obs = ctx.forces()
        return {"f": as_type(f), "pe": as_type(pe), "obs": as_type(obs)}
    if kind == "batch":
        b = state["batch"]
        # half of the replicas in tension, half in compression
        b.apply_strain([d if i % 2 == 0 else -d for i in range(len(state["ctx"]))])
        avg = b.fine_burst(steps)
        means, members = np.array([list(a.mean) for a in avg]), state["ctx"]
    elif kind == "coarse":
        r = ctx.coarse_step()
        members = [ctx]
        means = np.array([list(r.burst[b].mean) for b in range(3)]
                         + [list(r.v), list(r.v_pred), list(r.v_d)])
    else:
        if kind == "ramp":
            avg = ctx.ramp_burst(steps, d / steps)
        else:
            ctx.apply_strain(d)
            avg = ctx.fine_burst(steps)
        means, members = np.array([list(avg.mean)]), [ctx]
    out = {"means": as_type(means), "pos": [], "vel": [], "series": []}
    for c in members:
        pos, vel = c.get_state()
        out["pos"].append(as_type(pos))
        out["vel"].append(as_type(vel))
        out["series"].append(as_type(c.series(steps)))
    if kind == "ramp":
        out["mean_pos"] = as_type(ctx.mean_positions())
    return out


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
def _pairs(shape):
    """Unordered pairs within rc of the lattice block."""
    total = 0
    for i in range(-2, 3):
        for j in range(-2, 3):
            for k in range(-2, 3):
                for p in BASIS:
                    for q in BASIS:
                        t = (i + q[0] - p[0], j + q[1] - p[1], k + q[2] - p[2])
                        r2 = t[0] ** 2 + t[1] ** 2 + t[2] ** 2
                        if 0 < r2 < (RC / A0) ** 2 - 1e-9:
                            total += (max(0, shape[0] - abs(i)) * max(0, shape[1] - abs(j))
                                      * max(0, shape[2] - abs(k)))
    return total // 2


def work(case):
    """Per unordered pair 19 flop in the density and 41 in the force pass, per
    atom and step 33 (add, mul, div, sqrt 1, FMA 2).  Bytes: the state read
    once, and what the caller gets written once (forces and energies; or the
    new state, the mean positions, the sampled series)."""
    steps = case["steps"] * (3 if case["kind"] == "coarse" else 1)
    evals = steps + (3 if case["kind"] == "coarse" else 1) if case["kind"] != "forces" else 1
    flops = byts = 0.0
    for sh in _shapes(case):
        n = 4 * sh[0] * sh[1] * sh[2]
        flops += evals * (60.0 * _pairs(sh) + 33.0 * n)
        given = {"forces": 4, "ramp": 9}.get(case["kind"], 6)
        byts += (48.0 + given * (8.0 if case["prec"] == "fp64" else 4.0)) * n + 24.0 * steps
    return {"bytes": byts, "flops": flops}


# ---------------------------------------------------------------------------
# the same in 64 bits, in plain torch
# ---------------------------------------------------------------------------
def _equilibrium_c():
    """c that puts the perfect crystal under the cut potential in equilibrium."""
    sm = dn = dm = 0.0
    ac = A0 / RC
    for i in range(-3, 4):
        for j in range(-3, 4):
            for k in range(-3, 4):
                for q in BASIS:
                    t = (i + q[0], j + q[1], k + q[2])
                    r = A0 * math.sqrt(t[0] ** 2 + t[1] ** 2 + t[2] ** 2)
                    if r == 0.0 or not r < RC:
                        continue
                    s = A0 / r
                    sm += s ** PM - ac ** PM + PM / RC * ac ** PM * (r - RC)
                    dn += r * (-PN / r * s ** PN + PN / RC * ac ** PN)
                    dm += r * (-PM / r * s ** PM + PM / RC * ac ** PM)
    return math.sqrt(sm) * dn / dm


class _Exact:
    """Velocity Verlet of the cut Sutton-Chen EAM with fixed grips, float64."""

    SKIN, CHUNK = 1.2, 1 << 16

    def __init__(self, pos, vel, flag, shape, axis):
        dev = "cuda"
        self.x = torch.tensor(pos, device=dev)
        self.v = torch.tensor(vel, device=dev)
        self.mobile = torch.tensor(flag == 0, device=dev)[:, None]
        self.right = torch.tensor(flag == 2, device=dev)
        self.axis, self.L = axis, shape[axis] * A0
        area = 1.0
        for d in range(3):
            if d != axis:
                area *= shape[d] * A0
        self.t_fac = GPA / area
        self.c = _equilibrium_c()
        # eV/(A amu) -> A/fs^2 over two, times dt = 1 fs
        self.kick = 0.5 / (MASS * MV2)
        self.ref = None

    def lists(self):
        x, n, rl = self.x, len(self.x), RC + self.SKIN
        lo = x.min(0).values - 1e-3
        ic = ((x - lo) / rl).floor().long()
        nc = ic.max(0).values + 3
        ic = ic + 1                                  # a border of empty cells
        cid = (ic[:, 2] * nc[1] + ic[:, 1]) * nc[0] + ic[:, 0]
        order = torch.argsort(cid, stable=True)
        ncell = int(nc.prod())
        cnt = torch.bincount(cid, minlength=ncell)
        start = torch.cumsum(cnt, 0) - cnt
        occ = int(cnt.max())
        cells = torch.full((ncell, occ), n, device=x.device, dtype=torch.long)
        cells[cid[order], torch.arange(n, device=x.device) - start[cid[order]]] = order
        off = torch.tensor([(k * int(nc[1]) + j) * int(nc[0]) + i for k in (-1, 0, 1)
                            for j in (-1, 0, 1) for i in (-1, 0, 1)], device=x.device)
        far = torch.cat([x, torch.full((1, 3), 1e6, device=x.device, dtype=x.dtype)])
        rows, most = [], 0
        for a in range(0, n, 1 << 14):
            b = min(n, a + (1 << 14))
            cand = cells[cid[a:b, None] + off].reshape(b - a, -1)
            d = far[cand] - x[a:b, None]
            ok = ((d * d).sum(2) < rl * rl) & (cand != torch.arange(a, b, device=x.device)[:, None])
            k = int(ok.sum(1).max())
            idx = torch.where(ok, cand, n).sort(1).values[:, :k]
            rows.append(idx)
            most = max(most, k)
        self.idx = torch.full((n, most), n, device=x.device, dtype=torch.long)
        a = 0
        for r in rows:
            self.idx[a:a + len(r), :r.shape[1]] = r
            a += len(r)
        self.ref = x.clone()

    def forces(self):
        if self.ref is None or float((self.x - self.ref).square().sum(1).max()) > (0.5 * self.SKIN) ** 2:
            self.lists()
        x, n = self.x, len(self.x)
        far = torch.cat([x, torch.full((1, 3), 1e6, device=x.device, dtype=x.dtype)])
        ac = A0 / RC
        An, Am = ac ** PN, ac ** PM
        Bn, Bm = PN / RC * An, PM / RC * Am
        rho, en = torch.empty_like(x[:, 0]), torch.empty_like(x[:, 0])
        for p in (0, 1):
            if p:
                dB = torch.cat([-0.5 * EPS * self.c / rho.sqrt(), torch.zeros_like(rho[:1])])
                dB = torch.where(torch.isfinite(dB), dB, torch.zeros_like(dB))
                f = torch.empty_like(x)
            for a in range(0, n, self.CHUNK):
                j = self.idx[a:a + self.CHUNK]
                d = far[j] - x[a:a + self.CHUNK, None]
                r2 = (d * d).sum(2)
                inside = r2 < RC * RC
                r = torch.where(inside, r2, RC * RC).sqrt()
                s = A0 / r
                s6 = s ** PM
                s7 = s6 * s
                zero = torch.zeros_like(r)
                if not p:
                    rho[a:a + self.CHUNK] = torch.where(inside, s6 - Am + Bm * (r - RC), zero).sum(1)
                    en[a:a + self.CHUNK] = torch.where(inside, s7 - An + Bn * (r - RC), zero).sum(1)
                else:
                    g = EPS * (-PN * s7 / r + Bn)
                    g = g + (dB[a:a + self.CHUNK][:len(j), None] + dB[j]) * (-PM * s6 / r + Bm)
                    g = torch.where(inside, g / r, zero)
                    f[a:a + self.CHUNK] = (g[:, :, None] * d).sum(1)
        pe = 0.5 * EPS * en - EPS * self.c * rho.sqrt()
        return f, pe

    def observe(self, f, pe):
        k = 0.5 * MASS * MV2 * (self.v * self.v).sum()
        return torch.stack([k, pe.sum(), -self.t_fac * f[self.right, self.axis].sum()])

    def strain(self, d_eps):
        self.x[self.right, self.axis] += d_eps * self.L

    def burst(self, steps, ramp=0.0, mean_pos=None):
        series = []
        f, _ = self.forces()
        for _ in range(steps):
            self.v = torch.where(self.mobile, self.v + self.kick * f, self.v)
            self.x = self.x + torch.where(self.mobile, self.v, torch.zeros_like(self.v))
            if ramp:
                self.x[self.right, self.axis] += ramp * self.L
            f, pe = self.forces()
            self.v = torch.where(self.mobile, self.v + self.kick * f, self.v)
            series.append(self.observe(f, pe))
            if mean_pos is not None:
                mean_pos += self.x / steps
        return torch.stack(series)


def exact(case, seed):
    kind, steps, d = case["kind"], case["steps"], case["d_eps"]
    out = {"means": [], "pos": [], "vel": [], "series": []}
    for i, (shape, (pos, vel, flag)) in enumerate(zip(_shapes(case), _inputs(case, seed))):
        e = _Exact(pos, vel, flag, shape, case["axis"])
        if kind == "forces":
            f, pe = e.forces()
            return {"f": f, "pe": pe, "obs": e.observe(f, pe)}
        if kind == "coarse":
            rate, delta = 0.1 * d, 0.2
            m = []
            for inc in (rate * (1.0 - delta), rate * delta / 2, rate * delta / 2):
                e.strain(inc)
                series = e.burst(steps)
                m.append(series.mean(0))
            old = torch.tensor(_recorded_means(len(pos)), device=series.device)
            vd = (m[0] + 4.0 * m[1] + m[2]) / 6.0
            vp = (old[0] + 4.0 * old[1] + old[2]) / 6.0 + (old[2] - old[0]) / delta
            ev = (vp - vd).abs() / torch.maximum(vd.abs(), vd.new_tensor([1e-12, 1e-12, 0.05]))
            v = torch.where(ev < ev.new_tensor([0.01, 0.05, 0.01]), vp, vd)
            out["means"] = m + [v, vp, vd]
        else:
            if kind == "ramp":
                out["mean_pos"] = torch.zeros_like(e.x)
                series = e.burst(steps, d / steps, out["mean_pos"])
            else:
                e.strain(-d if i % 2 else d)
                series = e.burst(steps)
            out["means"].append(series.mean(0))
        out["pos"].append(e.x)
        out["vel"].append(e.v)
        out["series"].append(series)
    out["means"] = torch.stack(out["means"])
    return out
