"""The work a user of the peridynamic stepper has it do, as measurable cases.

Every forward case restarts a model from a given state (displacement and
velocity on the device, the step counter), advances it by a number of time
steps and reads the displacement, the velocity and the damage back into device
tensors: the calls of the outer loops that re-run one model many times.  The
adjoint cases record such a run and take the gradient of a loss of its final
state with respect to every bond's stiffness, the load and the initial state.

Bodies are cubic lattices, z fastest, pulled in x through 3-layer end slabs (or
loaded by body forces in the adjoint cases), optionally with every node moved
off the lattice and unequal volumes.  Notched bodies have a cut through the
bottom 30 % of their height at mid-span (absent bonds) and a crack grown
another 15 % above it (broken bonds).  The state is a strained body with a
smooth and a rough part and a velocity of a passing wave, its stretches far
enough below the critical one that nothing breaks while a pass runs, so that
a pass can be repeated from the same state.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2105_04150_gb300 as pd

DX = 1e-3                       # lattice spacing, m
RHO, DAMP, DT = 2400.0, 2.5e6, 1e-7
K_BULK = 3e10                   # Pa
SC = 1e-4                       # critical stretch
SC_LO, SC_HI, SC_SEED = 9e-5, 1.1e-4, 2105041502   # per-bond draw of the critical stretch
STEP0 = 100000                  # step the runs restart at (the slabs move slowly)
SLAB = 3


def _c(kind, name, **kw):
    c = dict(name=name, kind=kind, nx=0, ny=0, nz=0, steps=1, precision=64, jitter=0.0,
             delta=3.01, notch=False, hashed=False, vv=False, ramp=0, kr=0.0, state_based=False,
             graph=0, tune=False, count=0, n_lo=0, n_hi=0, strain=0.2)
    c.update(kw)
    return c


def listed():
    return [
        # The small verification bar of the tests, FP32, replayed in graphs: the
        # many short runs of a calibration, where launches and latency count.
        _c("step", "bar_f32_4k", nx=40, ny=10, nz=10, steps=100, precision=32, graph=50),
        # The same bar with the binding's defaults (FP64, direct launches).
        _c("step", "bar_f64_4k", nx=40, ny=10, nz=10, steps=50),
        # The benchmark beam: 1M nodes, notch, horizon pi dx, a critical stretch per
        # bond, FP32, autotuned as the benchmark does.
        _c("step", "beam_f32_1m", nx=300, ny=58, nz=58, steps=20, precision=32, delta=math.pi,
           notch=True, hashed=True, tune=True),
        # A large thin body (the benchmark plate's proportions at 2M nodes), FP32.
        _c("step", "plate_f32_2m", nx=354, ny=142, nz=40, steps=10, precision=32, notch=True,
           tune=True),
        # A body whose nodes are no lattice (a meshed part) with unequal volumes,
        # FP32: the general family layout.
        _c("step", "irregular_f32_250k", nx=100, ny=50, nz=50, steps=20, precision=32,
           jitter=0.25),
        # The notched beam in FP64, the precision of reference runs.
        _c("step", "beam_f64_220k", nx=180, ny=35, nz=35, steps=5, delta=math.pi, notch=True,
           hashed=True),
        # The same beam in double-word arithmetic (FP64-grade).
        _c("step", "beam_dw_220k", nx=180, ny=35, nz=35, steps=20, precision=48, delta=math.pi,
           notch=True, hashed=True),
        # The concrete examples: trilinear softening, velocity-Verlet and a smooth
        # start, FP64, an odd-sized notched beam.
        _c("step", "soft_vv_f64_30k", nx=95, ny=18, nz=18, steps=20, notch=True, vv=True,
           ramp=300, kr=4.0),
        # The state-based solid on a mid-sized bar, FP32.
        _c("step", "state_based_f32_135k", nx=150, ny=30, nz=30, steps=50, precision=32,
           notch=True, state_based=True),
        # Uncertainty quantification: independent bars and notched beams of 2k to 60k
        # nodes advanced together, FP32.
        _c("batch", "batch_f32_32", count=32, n_lo=2000, n_hi=60000, steps=10, precision=32),
        # Sensitivities of the 100k-node plate with a stiffness per bond, FP64.
        _c("adjoint", "adjoint_f64_100k", nx=250, ny=100, nz=4, steps=60, notch=True),
        # The same on a smaller plate in double-word arithmetic.
        _c("adjoint", "adjoint_dw_16k", nx=100, ny=40, nz=4, steps=100, precision=48, notch=True),
    ]


def _body(rng, n, ratio):
    """Lattice counts of about n nodes in all, nx about ratio times ny and nz."""
    a = (n / ratio) ** (1.0 / 3.0)
    ny = max(4, round(a * math.exp(rng.uniform(-0.2, 0.2))))
    nz = max(4, round(a * math.exp(rng.uniform(-0.2, 0.2))))
    return max(2 * SLAB + 4, round(n / (ny * nz))), ny, nz


def draw(rng):
    kind = rng.choice(["step", "step", "step", "step", "step", "batch", "adjoint"])
    if kind == "batch":
        lo = math.exp(rng.uniform(math.log(500.0), math.log(4000.0)))
        return {k: v for k, v in _c("batch", "", count=rng.randint(2, 32), n_lo=int(lo),
                                    n_hi=int(lo * rng.uniform(2.0, 15.0)),
                                    steps=rng.randint(3, 10),
                                    precision=rng.choice([32, 32, 48, 64])).items() if k != "name"}
    if kind == "adjoint":
        n = math.exp(rng.uniform(math.log(1500.0), math.log(8e4)))
        nz = rng.randint(3, 6)
        ny = max(6, round(math.sqrt(n / nz / 2.5) * math.exp(rng.uniform(-0.3, 0.3))))
        c = _c("adjoint", "", nx=max(8, round(n / (ny * nz))), ny=ny, nz=nz,
               steps=rng.randint(15, 60), notch=True, vv=rng.random() < 0.25,
               precision=rng.choice([64, 64, 48]))
        del c["name"]
        return c
    prec = rng.choice([32, 32, 48, 64, 64])
    top = {32: 1.2e6, 48: 3e5, 64: 2e5}[prec]
    n = math.exp(rng.uniform(math.log(800.0), math.log(top)))
    nx, ny, nz = _body(rng, n, rng.choice([1.0, 2.5, 4.0, 5.0]))
    form = rng.choice(["lattice", "lattice", "irregular", "soft", "state_based"])
    c = _c("step", "", nx=nx, ny=ny, nz=nz, precision=prec,
           steps=int(max(3, min(100, {32: 1.2e7, 48: 3e6, 64: 1e6}[prec] / n))),
           delta=rng.choice([3.01, math.pi]), notch=form != "irregular" and rng.random() < 0.7,
           hashed=rng.random() < 0.4, vv=rng.random() < 0.25, graph=rng.choice([0, 0, 10, 50]),
           strain=rng.uniform(0.05, 0.22))
    if form == "irregular":
        c["jitter"] = rng.uniform(0.02, 0.25)
    elif form == "soft":
        c["kr"] = rng.uniform(1.5, 4.0)
        c["ramp"] = rng.choice([0, 300])
    elif form == "state_based":
        c["state_based"] = True
    del c["name"]
    return c


# ---------------------------------------------------------------------------
# bodies and states

def _scale(case_rate, ramp, k):
    """Displacement scale after step k: the linear ramp, or the smooth start."""
    if ramp <= 0:
        return case_rate * k
    if k < ramp:
        t = k / ramp
        return case_rate * ramp * (t ** 4 - 0.6 * t ** 5)
    return case_rate * (k - 0.6 * ramp)


def _make(nx, ny, nz, case, seed, K=K_BULK, sc=SC):
    """Host arrays of one body and its state, from the seed alone."""
    rng = np.random.default_rng(seed)
    ix, iy, iz = (a.ravel() for a in np.meshgrid(np.arange(nx), np.arange(ny), np.arange(nz),
                                                 indexing="ij"))
    x = np.stack([ix, iy, iz], axis=1).astype(np.float64) * DX
    n = x.shape[0]
    b = dict(n=n, shape=(nx, ny, nz), K=K, sc=sc, delta=case["delta"] * DX,
             vol=np.full(n, DX ** 3), cut=None, crack=None)
    if case["jitter"] > 0.0:
        x += rng.uniform(-case["jitter"], case["jitter"], size=x.shape) * DX
        b["vol"] = DX ** 3 * rng.uniform(0.8, 1.2, size=n)
    b["x"] = x
    if case["notch"]:
        xm = (nx // 2 - 0.5) * DX
        far = 1e3 * DX
        if case["kind"] != "adjoint":       # bottom of the mid-span, over the full width
            z1, z2 = (0.3 * nz - 0.5) * DX, (0.45 * nz - 0.5) * DX
            b["cut"] = (0, xm, -far, far, -far, z1)
            b["crack"] = (0, xm, -far, far, z1, z2)
        else:                               # edge crack of a plate at half its width
            ym = (ny // 2 - 0.5) * DX
            b["cut"] = (1, ym, -far, (0.25 * nx - 0.5) * DX, -far, far)
    t = np.zeros((n, 3), np.uint8)
    g = np.zeros((n, 3))
    f = np.zeros((n, 3))
    s0 = sc if not case["hashed"] else SC_LO
    if case["kr"] >= 1.0:
        s0 /= case["kr"]
    eps = case["strain"] * s0
    length = (nx - 1 - 2 * (SLAB - 1)) * DX
    cen = 0.5 * (nx - 1) * DX
    ramp = case["ramp"]
    b["rate"] = 0.5 * eps * length / _scale(1.0, ramp, STEP0)
    if case["kind"] == "adjoint":
        f[iy < 2, 1], f[iy >= ny - 2, 1] = -1.0, 1.0
        b["rate"], b["load"] = 0.0, 8e6
    else:
        lo, hi = ix < SLAB, ix >= nx - SLAB
        t[lo, 0] = t[hi, 0] = 1
        g[lo, 0], g[hi, 0] = -1.0, 1.0
        b["load"] = 0.0
    b.update(type=t, disp=g, force=f)
    # linear strain between the slabs, smooth waves that end at them, and a rough
    # part of 1 %
    xr = np.clip((x[:, 0] - cen) / (0.5 * length), -1.0, 1.0)
    ph = rng.uniform(0.0, 2.0 * math.pi, size=(2, 3, 3))
    wl = 2.0 * math.pi / (max(nx, 8) * DX * np.array([0.5, 0.8, 1.3]))
    u = np.zeros((n, 3))
    v = np.zeros((n, 3))
    win = 1.0 - xr * xr if case["kind"] != "adjoint" else 1.0
    for a in range(3):
        k = np.roll(wl, a)
        for d in range(3):
            u[:, a] += 0.1 * eps / wl[0] * win * np.sin(k[d] * x[:, d] + ph[0, a, d])
            v[:, a] += 0.05 * eps * 3500.0 * win * np.sin(k[d] * x[:, d] + ph[1, a, d])
    u += eps * 0.01 * DX * rng.uniform(-1.0, 1.0, size=(n, 3))
    if case["kind"] != "adjoint":
        u[:, 0] += 0.5 * eps * length * xr
        u = np.where(t == 1, g * _scale(b["rate"], ramp, STEP0), u)
    b.update(u0=u, v0=v)
    return b


def _crossing(b, rect, xi, xj):
    """Bonds xi -> xj whose segment crosses the rectangle (axis, pos, lo, hi, lo, hi)."""
    ax, pos, la, ha, lb, hb = rect
    p, q = (k for k in range(3) if k != ax)
    d0, d1 = xi[..., ax] - pos, xj[..., ax] - pos
    t = d0 / (d0 - d1 + (d0 == d1))
    a = xi[..., p] + t * (xj[..., p] - xi[..., p])
    c = xi[..., q] + t * (xj[..., q] - xi[..., q])
    return ((d0 * d1) < 0) & (a >= la) & (a <= ha) & (c >= lb) & (c <= hb)


def _offsets(b):
    reach = 4 if b["vol"].min() != b["vol"].max() else 3
    r = range(-reach, reach + 1)
    return [(i, j, k) for i in r for j in r for k in r if (i, j, k) != (0, 0, 0)]


def _crack_pairs(b):
    """Node pairs of the bonds the grown crack has broken (one direction of each)."""
    nx, ny, nz = b["shape"]
    lim = b["delta"] * b["delta"]
    near = np.nonzero(np.abs(b["x"][:, 0] - b["crack"][1]) < 3.5 * DX)[0]
    near = near[b["x"][near, 2] < b["crack"][5] + 3.5 * DX]
    out = []
    at = np.stack(np.unravel_index(near, b["shape"]), axis=1)
    for o in _offsets(b):
        if o[0] <= 0 or DX * DX * (o[0] ** 2 + o[1] ** 2 + o[2] ** 2) > lim:
            continue
        to = at + np.array(o)
        ok = ((to >= 0) & (to < np.array(b["shape"]))).all(axis=1)
        i, t = near[ok], to[ok]
        j = (t[:, 0] * ny + t[:, 1]) * nz + t[:, 2]
        cut = _crossing(b, b["cut"], b["x"][i], b["x"][j])
        hit = _crossing(b, b["crack"], b["x"][i], b["x"][j]) & ~cut
        out.append(np.stack([i[hit], j[hit]], axis=1))
    return np.concatenate(out).astype(np.int64)


def _elastic(case, b):
    c = 18.0 * b["K"] / (math.pi * b["delta"] ** 4)
    return c, (b["K"], 0.5 * b["K"]) if case["state_based"] else None


def _kwargs(case, b):
    c, sb = _elastic(case, b)
    return dict(coords=b["x"], volumes=b["vol"], horizon=b["delta"], c=c, sc=b["sc"],
                sc_hash=(SC_SEED, SC_LO, SC_HI) if case["hashed"] else None,
                cuts=None if b["cut"] is None else [b["cut"]], bc_type=b["type"],
                bc_disp=b["disp"], bc_force=b["force"], disp_rate=b["rate"], load=b["load"],
                ramp_steps=case["ramp"], kr=case["kr"],
                trilinear=(2.0, 0.25) if case["kr"] > 2.0 else None, state_based=sb)


def _instances(case, seed):
    """The batch's bodies: bars 4:1:1 and notched beams 5:1:1, alternating; their
    sizes are the case's, their materials and states the seed's."""
    sizes = np.random.default_rng(case["n_lo"] * 64 + case["count"])
    rng = np.random.default_rng(seed + 77)
    out = []
    for k in range(case["count"]):
        n = math.exp(sizes.uniform(math.log(case["n_lo"]), math.log(case["n_hi"])))
        r = 4.0 + k % 2
        a = (n / r) ** (1.0 / 3.0)
        one = dict(case, kind="step", notch=k % 2 == 1)
        b = _make(max(10, round(r * a)), max(3, round(a)), max(4, round(a)), one, seed + k,
                  K=float(math.exp(rng.normal(math.log(K_BULK), 0.2))),
                  sc=float(math.exp(rng.normal(math.log(SC), 0.15))))
        out.append((one, b))
    rate = min(b["rate"] for _, b in out)
    for _, b in out:                        # one displacement rate for the whole batch
        b["disp"] = b["disp"] * (b["rate"] / rate)
        b["rate"] = rate
    return out


def _stiffness(case, b, c, off, idx):
    """A stiffness per directed bond, symmetric: 10 % variation of the bond midpoint."""
    rows = np.repeat(np.arange(b["n"]), np.diff(off))
    m = 0.5 * (b["x"][rows] + b["x"][idx])
    return c * _field(m[:, 0], m[:, 1], m[:, 2], np)


def _field(mx, my, mz, lib):
    w = 2.0 * math.pi / (17.0 * DX)
    return 1.0 + 0.1 * lib.sin(w * mx) * lib.cos(0.7 * w * my + 0.3) * lib.cos(0.4 * w * mz)


def _loss_grads(case, b, seed):
    rng = np.random.default_rng(seed + 5)
    return rng.normal(0.0, 1.0, size=(2, b["n"], 3)) * np.array([1.0, 1e-6]).reshape(2, 1, 1)


def prepare(case, seed):
    dev = torch.device("cuda")
    cfg = dict(dt=DT, damping=DAMP, density=RHO, precision=case["precision"],
               graph_steps=case["graph"], integrator=1 if case["vv"] else 0)
    if case["kind"] == "batch":
        bodies = _instances(case, seed)
        h = pd.pd_batch_create([_kwargs(c, b) for c, b in bodies], **cfg)
        offs = np.concatenate([[0], np.cumsum([b["n"] for _, b in bodies])])
        pairs = np.concatenate([np.zeros((0, 2), np.int64)] +
                               [_crack_pairs(b) + offs[k] for k, (_, b) in enumerate(bodies)
                                if b["crack"] is not None])
        u0 = np.concatenate([b["u0"] for _, b in bodies])
        v0 = np.concatenate([b["v0"] for _, b in bodies])
    else:
        b = _make(case["nx"], case["ny"], case["nz"], case, seed)
        h = pd.pd_create(**_kwargs(case, b), **cfg)
        pairs = _crack_pairs(b) if b["crack"] is not None else np.zeros((0, 2), np.int64)
        u0, v0 = b["u0"], b["v0"]
    m = pd.Model(handle=h)
    if len(pairs):
        m.remove_bonds(pairs)
    st = dict(case=case, model=m, u0=torch.from_numpy(u0).to(dev), v0=torch.from_numpy(v0).to(dev))
    if case["kind"] == "adjoint":
        off, idx = m.family()
        c, _ = _elastic(case, b)
        m.set_params(c, b["sc"], b["load"], b["rate"], _stiffness(case, b, c, off, idx))
        st["grads"] = [np.ascontiguousarray(g) for g in _loss_grads(case, b, seed)]
    if case["tune"]:
        m.autotune(10)
    n = u0.shape[0]
    st["u"], st["v"] = (torch.empty((n, 3), dtype=torch.float64, device=dev) for _ in range(2))
    st["phi"] = torch.empty(n, dtype=torch.float64, device=dev)
    return st


def run(st):
    case, m = st["case"], st["model"]
    m.set_state(st["u0"], st["v0"], step=STEP0)
    if case["kind"] == "adjoint":
        pd.pd_adjoint_forward(m.h, case["steps"])
        pd.pd_get_state(m.h, st["u"], st["v"])
        gc, gl, gu, gv = pd.pd_adjoint_backward(m.h, *st["grads"])
        return dict(u=st["u"], v=st["v"], dc=gc, dload=gl, du0=gu, dv0=gv)
    m.step(case["steps"])
    pd.pd_get_state(m.h, st["u"], st["v"])
    m.damage(st["phi"])
    return dict(u=st["u"], v=st["v"], phi=st["phi"])


def _counts(case):
    """(nodes, directed bonds) of a case, bonds by the lattice's family."""
    if case["kind"] == "batch":
        n = case["count"] * (case["n_hi"] - case["n_lo"]) / math.log(case["n_hi"] / case["n_lo"])
        return int(n), int(100 * n)
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    bonds = sum((nx - abs(i)) * (ny - abs(j)) * (nz - abs(k))
                for i in range(-3, 4) for j in range(-3, 4) for k in range(-3, 4)
                if 0 < i * i + j * j + k * k <= 9 and abs(i) < nx and abs(j) < ny and abs(k) < nz)
    return nx * ny * nz, bonds


def work(case):
    """Per step: each node's u and v read and written, a flag bit per bond read,
    and on bodies that are no lattice a neighbour id per bond; about 31 operations
    per directed bond (stretch, break test, force), 57 for the two loops of the
    state-based solid, 60 more for a reverse step.  Once per pass: the state in,
    the state and the damage out, or the gradients."""
    n, nb = _counts(case)
    small = case["precision"] == 32
    step_bytes = n * (72 if small else 96) + nb / 8 + (4 * nb if case["jitter"] > 0 else 0)
    flops = nb * (57.0 if case["state_based"] else 31.0)
    if case["kind"] == "adjoint":
        # the forward run, its recomputation, and the reverse steps with the
        # accumulated stiffness gradient
        return {"bytes": case["steps"] * (3 * step_bytes + 8 * nb) + 144 * n + 8 * nb,
                "flops": case["steps"] * nb * (2 * 31.0 + 60.0)}
    return {"bytes": case["steps"] * step_bytes + 104 * n, "flops": case["steps"] * flops}


# ---------------------------------------------------------------------------
# the same results in 64-bit torch

class _Exact:
    """One body on a grid padded by the stencil's reach; every bond quantity is
    formed offset by offset over all nodes, the stretch without cancellation."""

    def __init__(self, case, b, seed):
        self.case, self.b = case, b
        self.dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
        self.shape = b["shape"]
        offs = _offsets(b)
        self.R = max(abs(o[0]) for o in offs)
        self.x = self.grid(b["x"])
        self.vol = self.grid(b["vol"][:, None])
        inb = self.pad(torch.ones(self.shape + (1,), device=self.dev, dtype=torch.float64))
        xp, self.volp = self.pad(self.x), self.pad(self.vol)
        self.xp = xp
        self.off, self.fam, self.mask = [], [], []
        for o in offs:
            xj = self.at(xp, o)
            e = xj - self.x
            m = (torch.sqrt((e * e).sum(-1)) <= b["delta"]) & (self.at(inb, o)[..., 0] > 0)
            if b["cut"] is not None:
                m &= ~_crossing(b, b["cut"], self.x, xj)
            if not bool(m.any()):
                continue
            self.off.append(o)
            self.fam.append(m)
            self.mask.append(m & ~_crossing(b, b["crack"], self.x, xj)
                             if b["crack"] is not None else m)
        self.c, self.sb = _elastic(case, b)
        self.type = self.grid(b["type"].astype(np.float64)) > 0
        self.disp, self.force = self.grid(b["disp"]), self.grid(b["force"])
        self.u, self.v = self.grid(b["u0"]), self.grid(b["v0"])
        self.stiff = None
        if self.sb is not None:
            self.m = torch.zeros(self.shape + (1,), device=self.dev, dtype=torch.float64)
            for o, f in zip(self.off, self.fam):
                e = self.at(xp, o) - self.x
                self.m += ((e * e).sum(-1) * f).unsqueeze(-1) * self.at(self.volp, o)

    def grid(self, a):
        return torch.from_numpy(np.ascontiguousarray(a)).to(self.dev).reshape(
            self.shape + (a.shape[1],))

    def pad(self, g):
        R = self.R
        out = torch.zeros(tuple(s + 2 * R for s in self.shape) + (g.shape[-1],), device=self.dev,
                          dtype=torch.float64)
        out[R:-R, R:-R, R:-R] = g
        return out

    def at(self, p, o):
        R, s = self.R, self.shape
        return p[R + o[0]:R + o[0] + s[0], R + o[1]:R + o[1] + s[1], R + o[2]:R + o[2] + s[2]]

    def bond(self, k, u, up):
        """y, |xi|, |y|, |y|^2 - |xi|^2 across offset k (absent bonds: a unit bond)."""
        o, m = self.off[k], self.mask[k].unsqueeze(-1)
        e = torch.where(m, self.at(self.xp, o) - self.x, torch.ones_like(self.x))
        h = torch.where(m, self.at(up, o) - u, torch.zeros_like(u))
        y = e + h
        num = (h * (e + y)).sum(-1, keepdim=True)
        L2 = (e * e).sum(-1, keepdim=True)
        return y, torch.sqrt(L2), torch.sqrt(L2 + num), num, m

    def c_of(self, k):
        if self.stiff is None:
            return self.c
        mid = 0.5 * (self.x + self.at(self.xp, self.off[k]))
        return self.c * _field(mid[..., 0:1], mid[..., 1:2], mid[..., 2:3], torch)

    def forces(self, u):
        up = self.pad(u)
        F = torch.zeros_like(u)
        if self.sb is not None:
            K, G = self.sb
            th = torch.zeros_like(self.m)
            for k, o in enumerate(self.off):
                y, L, r, num, m = self.bond(k, u, up)
                th += torch.where(m, L * num / (L + r), torch.zeros_like(num)) * self.at(self.volp, o)
            th = 3.0 * th / self.m
            beta = 15.0 * G / self.m
            al = 3.0 * K * th / self.m - beta * th / 3.0
            alp, bep = self.pad(al), self.pad(beta)
            for k, o in enumerate(self.off):
                y, L, r, num, m = self.bond(k, u, up)
                t = (al + self.at(alp, o)) * L + (beta + self.at(bep, o)) * num / (L + r)
                F += torch.where(m, t * self.at(self.volp, o) / r, torch.zeros_like(t)) * y
            return F + self.b["load"] * self.force
        for k, o in enumerate(self.off):
            y, L, r, num, m = self.bond(k, u, up)
            f = self.c_of(k) * num / (L * (L + r)) * self.at(self.volp, o) / r
            F += torch.where(m, f, torch.zeros_like(f)) * y
        return F + self.b["load"] * self.force

    def run(self, keep=None):
        u, v, b, case = self.u, self.v, self.b, self.case
        a = None
        for k in range(STEP0, STEP0 + case["steps"]):
            if keep is not None:
                keep.append(u)
            s0, s1 = (_scale(b["rate"], case["ramp"], q) for q in (k, k + 1))
            if not case["vv"]:
                v = v + DT * (self.forces(u) - DAMP * v) / RHO
                u = u + DT * v
            else:
                if a is None:
                    a = (self.forces(u) - DAMP * v) / RHO
                half = v + 0.5 * DT * a
                u = u + DT * half
            u = torch.where(self.type, self.disp * s1, u)
            if case["vv"]:
                half = torch.where(self.type, self.disp * (s1 - s0) / DT, half)
                a = (self.forces(u) - DAMP * half) / RHO
                v = torch.where(self.type, half, half + 0.5 * DT * a)
            else:
                v = torch.where(self.type, self.disp * (s1 - s0) / DT, v)
        return u, v

    def damage(self):
        have = torch.zeros_like(self.vol)
        whole = torch.zeros_like(self.vol)
        for k, o in enumerate(self.off):
            vj = self.at(self.volp, o)
            have += vj * self.mask[k].unsqueeze(-1)
            whole += vj * self.fam[k].unsqueeze(-1)
        return torch.where(whole > 0, 1.0 - have / whole.clamp_min(1e-300), have).reshape(-1)

    def adjoint(self, keep, gu, gv):
        """Reverse of run() (no component is controlled in these cases)."""
        vv = self.case["vv"]
        N, dr = len(keep), DT / RHO
        damp = 1.0 - DT * DAMP / RHO
        ub, vb = self.grid(gu), self.grid(gv)
        dc = [torch.zeros_like(self.vol) for _ in self.off]
        dl = torch.zeros((), device=self.dev, dtype=torch.float64)

        def back(u, w):
            nonlocal dl
            up, wp = self.pad(u), self.pad(w)
            acc = torch.zeros_like(u)
            for k, o in enumerate(self.off):
                y, L, r, num, m = self.bond(k, u, up)
                vj = self.at(self.volp, o)
                s = num / (L * (L + r))
                d = self.vol * self.at(wp, o) - vj * w
                t = self.c_of(k) * (s / r * d + y * ((y * d).sum(-1, keepdim=True) / r ** 3))
                acc += torch.where(m, t, torch.zeros_like(t))
                g = dr * s * vj * (y * w).sum(-1, keepdim=True) / r
                dc[k] += torch.where(m, g, torch.zeros_like(g))
            dl = dl + dr * (self.force * w).sum()
            return dr * acc

        if vv:                       # the closing half kick forms v^N at u^N
            w = 0.5 * vb
            ub, vb = ub + back(self.uN, w), (1.0 + damp) * w
        for n in range(N - 1, -1, -1):
            first = vv and n == 0    # the opening half kick
            w = (0.5 if first else 1.0) * (vb + DT * ub)
            ub = ub + back(keep[n], w)
            vb = (1.0 + damp if first else damp) * w
        G = torch.stack([g.reshape(-1) for g in dc], dim=1)
        M = torch.stack([f.reshape(-1) for f in self.fam], dim=1)
        return G[M], dl, ub.reshape(-1, 3), vb.reshape(-1, 3)


def exact(case, seed):
    if case["kind"] == "batch":
        parts = []
        for one, b in _instances(case, seed):
            e = _Exact(one, b, seed)
            u, v = e.run()
            parts.append((u.reshape(-1, 3), v.reshape(-1, 3), e.damage()))
        u, v, phi = (torch.cat(p) for p in zip(*parts))
        return dict(u=u, v=v, phi=phi)
    b = _make(case["nx"], case["ny"], case["nz"], case, seed)
    e = _Exact(case, b, seed)
    if case["kind"] != "adjoint":
        u, v = e.run()
        return dict(u=u.reshape(-1, 3), v=v.reshape(-1, 3), phi=e.damage())
    e.stiff = True
    keep = []
    u, v = e.run(keep)
    e.uN = u
    dc, dl, du0, dv0 = e.adjoint(keep, *_loss_grads(case, b, seed))
    return dict(u=u.reshape(-1, 3), v=v.reshape(-1, 3), dc=dc.cpu().numpy(), dload=float(dl),
                du0=du0.cpu().numpy(), dv0=dv0.cpu().numpy())
