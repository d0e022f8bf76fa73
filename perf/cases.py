"""What this framework's speed is measured on: its own workloads, through its
public entry points.

Kinds of work (the "kind" of a case):

  step     a periodic box advanced `steps` velocity-Verlet steps, the state read
           into device tensors (Sim)
  round    a box whose state lives in page-locked host arrays between steps:
           upload, step, download (Sim; the end-to-end figure of bench.py)
  ensemble uneven replicas advanced together (Ensemble), every replica's state
           read into device tensors
  cube     the three-dimensional variant advanced `steps` steps, the state read
           to the host (Sim3)
  observe  one snapshot of a run: E(k), and where `nbins` > 0 the velocity
           correlation, T and the mean agent speed; with `field` the filtered
           velocity field and its vorticity too (Sim)
  observe3 the same snapshot of a cube (Sim3)
  fit      the surrogate's training: the loss and gradients of one member at
           the initial weights, `epochs` passes over `rows` rows, then the
           predictions for these rows (Surrogate)
  predict  the surrogate's answers for `rows` parameter rows (Surrogate)

Boxes start from the paper's initial condition (dimers at random centres and
orientations, bond at rest length) with thermal velocities and a smooth flow
on top, so that spectra and correlations have something to find.  Area
fraction phi means 2 phi L^2 agents in the benchmark's units (phi = 0.75 is bead
density 3) and 4 phi L^2 with the paper's own parameter set (4e4 phi at
L = 100); in a cube, phi is the bead density.
"""
import math

import numpy as np
import torch

from paper_1310_0998_gb300 import Ensemble, Sim, Sim3, Surrogate

# reduced units of the benchmark boxes, and the paper's own set
BASE = dict(a=25.0, gamma=4.5, kBT=1.0, rc=1.0, k_bond=100.0, r0=0.5, f_p=1.0, zeta=0.1, dt=0.01, mass=1.0)
PAPER = dict(a=1.5, gamma=8.0, kBT=0.05, rc=0.5, k_bond=1000.0, r0=0.75, f_p=1.0, zeta=0.5, dt=3.0e-3, mass=1.0)
NIN, NH, NOUT, MEMBERS = 4, 256, 40, 4


def listed():
    return [
        # the smallest box users step (tests, quick looks): launches and latency
        dict(name="step small box", kind="step", set="base", L=32.0, phi=0.25, steps=100),
        # one point of the paper's parameter study: dilute, r_c = 0.5, bonds longer than r_c
        dict(name="step paper box", kind="step", set="paper", L=100.0, phi=0.6, steps=50),
        # one point of the 256 x 256 parameter sweep
        dict(name="step sweep box", kind="step", set="base", L=256.0, phi=0.4, steps=20),
        # the headline box, 3,145,728 beads
        dict(name="step large box", kind="step", set="base", L=1024.0, phi=0.75, steps=10),
        # the headline box driven from host arrays, one step at a time
        dict(name="round trip large box", kind="round", set="base", L=1024.0, phi=0.75),
        # the uneven-replica ensemble of the parameter studies
        dict(name="ensemble 256", kind="ensemble", replicas=256, L_max=192.0, steps=50),
        # three dimensions, density 3, 786,432 beads
        dict(name="step cube", kind="cube", L=64.0, phi=3.0, steps=20),
        # the snapshot behind one training row of the surrogate (g out to L / 2: all pairs)
        dict(name="observe training box", kind="observe", L=48.0, phi=0.3, M=128, dr=0.25, nbins=96, field=False),
        # a snapshot of the headline box (g to r < 16: cell grid)
        dict(name="observe large box", kind="observe", L=1024.0, phi=0.75, M=128, dr=0.25, nbins=64, field=False),
        # a snapshot of the cube, with its field and vorticity
        dict(name="observe cube", kind="observe3", L=64.0, phi=3.0, M=64, dr=0.25, nbins=16, field=True),
        # two epochs of the surrogate's training set
        dict(name="fit", kind="fit", rows=2000, batch=64, epochs=2),
        # a large table of parameter points answered by the surrogate
        dict(name="predict", kind="predict", rows=4096),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _side(x):
    return max(4.0, round(x * 256.0) / 256.0)   # exact on the simulator's position grid


def draw(rng):
    kind = rng.choice(["step", "step", "step", "round", "ensemble", "cube", "observe", "observe", "observe3", "fit",
                       "predict"])
    if kind in ("step", "round"):
        phi = rng.uniform(0.05, 0.75)
        nd = _log(rng, 64, 1.5e6 if kind == "step" else 3e5)
        c = dict(kind=kind, set="paper" if rng.random() < 0.25 else "base", phi=phi)
        if c["set"] == "paper":
            phi = c["phi"] = rng.uniform(0.05, 0.8)
            c["L"] = _side(math.sqrt(min(nd, 64000) / (4.0 * phi)))
        else:
            c["L"] = _side(math.sqrt(nd / (2.0 * phi)))
            c.update(gamma=_log(rng, 0.5, 20.0), zeta=_log(rng, 0.005, 2.0), f_p=rng.uniform(0.5, 2.0),
                     noise=int(rng.random() < 0.15), wexp=1.0 if rng.random() < 0.15 else 0.0)
        if kind == "step":
            c["steps"] = max(1, min(100, int(_log(rng, 1, 100)), int(1.5e7 / nd)))
        return c
    if kind == "ensemble":
        return dict(kind=kind, replicas=int(_log(rng, 2, 256)), L_max=rng.uniform(48.0, 192.0),
                    steps=rng.randint(1, 50))
    if kind == "cube":
        L = _side(_log(rng, 6.0, 64.0))
        return dict(kind=kind, L=L, phi=rng.uniform(0.5, 3.0), steps=rng.randint(1, 20))
    if kind == "observe":
        L = _side(_log(rng, 24.0, 512.0))
        cells = rng.random() < 0.5
        rmax = _log(rng, 2.0, min(16.0, L / 3.2)) if cells or L > 128.0 else L / 2
        dr = rng.choice([0.125, 0.25, 0.5])
        phi = rng.uniform(0.1, 0.75)
        M = rng.choice([32, 64, 128, 256])
        if L * math.sqrt(10.0 / (2.0 * phi * L * L)) * M / L > 50.0:
            M = 32
        return dict(kind=kind, L=L, phi=phi, M=M, dr=dr, nbins=max(4, int(rmax / dr)), field=rng.random() < 0.5)
    if kind == "observe3":
        L = _side(_log(rng, 12.0, 64.0))
        return dict(kind=kind, L=L, phi=rng.uniform(1.0, 3.0), M=rng.choice([16, 32, 64]), dr=0.25,
                    nbins=rng.randint(8, 16), field=rng.random() < 0.5)
    if kind == "fit":
        rows, batch = int(_log(rng, 64, 4096)), rng.choice([16, 32, 64, 100, 128, 256])
        batch = min(batch, rows)
        return dict(kind=kind, rows=rows, batch=batch, epochs=max(1, min(4, 60 // max(1, rows // batch))))
    return dict(kind=kind, rows=int(_log(rng, 1, 262144)))


# ------------------------------------------------------------------ inputs ----
def _params(case):
    p = dict(PAPER if case.get("set") == "paper" else BASE)
    p.update({k: case[k] for k in ("gamma", "zeta", "f_p", "noise", "wexp") if k in case})
    return p


def _agents(case):
    if case["kind"] in ("cube", "observe3"):
        return max(8, int(round(0.5 * case["phi"] * case["L"] ** 3)))
    return max(8, int(round((4.0 if case.get("set") == "paper" else 2.0) * case["phi"] * case["L"] ** 2)))


def _gen(seed):
    return torch.Generator("cuda").manual_seed(int(seed) * 7919 + 11)


def _dimers(na, L, r0, dim, kBT, gen):
    """Positions [2 na, dim] float64 on the grid L 2^-32, velocities float32."""
    kw = dict(dtype=torch.float64, device="cuda", generator=gen)
    c = torch.rand(na, dim, **kw) * L
    n = torch.randn(na, dim, **kw)
    n = n / n.norm(dim=1, keepdim=True)
    x = torch.stack([c + 0.5 * r0 * n, c - 0.5 * r0 * n], 1).reshape(2 * na, dim)
    x = torch.remainder(torch.round(x * (2.0 ** 32 / L)), 2.0 ** 32) * (L / 2.0 ** 32)
    v = torch.randn(2 * na, dim, **kw) * math.sqrt(kBT)
    for d in range(dim):
        v[:, d] += 0.5 * torch.sin(2.0 * math.pi * (d + 2) * x[:, (d + 1) % dim] / L)
    return x.contiguous(), v.to(torch.float32).contiguous()


def _points(case, seed):
    """The replicas' boxes and parameters (the distribution of synth.ensemble_points), the same for every seed."""
    rng = np.random.default_rng(5)
    out = []
    for r in range(case["replicas"]):
        L = round(float(rng.uniform(32.0, max(40.0, case["L_max"]))) * 256.0) / 256.0
        phi = float(rng.uniform(0.05, 0.6))
        out.append(dict(BASE, L=L, n_beads=2 * max(8, int(round(2.0 * phi * L * L))), seed=int(seed), replica=r,
                        gamma=float(math.exp(rng.uniform(math.log(0.5), math.log(50.0)))),
                        zeta=float(math.exp(rng.uniform(math.log(0.005), math.log(2.0)))),
                        f_p=float(rng.uniform(0.5, 2.0))))
    return out


def _rows(case, seed):
    """Parameter rows in the ranges of synth.surrogate_points."""
    rng, n = np.random.default_rng(int(seed) + 9), case["rows"]
    return np.stack([rng.uniform(0.05, 0.6, n), np.exp(rng.uniform(math.log(0.5), math.log(50.0), n)),
                     np.exp(rng.uniform(math.log(0.005), math.log(2.0), n)), rng.uniform(0.5, 2.0, n)],
                    axis=1).astype(np.float32)


def _targets(X, seed):
    """Smooth statistics-like targets of the rows with a little noise."""
    rng = np.random.default_rng(int(seed) + 10)
    z = np.stack([X[:, 0] * 3.0, np.log(X[:, 1]) / 2.0, np.log(X[:, 2]) / 2.0, X[:, 3]], axis=1)
    return (np.tanh(z @ rng.standard_normal((4, NOUT))) * rng.uniform(0.5, 3.0, NOUT) +
            rng.standard_normal(NOUT) + 0.05 * rng.standard_normal((len(X), NOUT))).astype(np.float32)


def _weights(seed):
    """Members' weights as a trained network would have them, by size (padded as Surrogate.set_weights takes them)."""
    rng, out = np.random.default_rng(int(seed) + 12), []
    for _ in range(MEMBERS):
        W1, W3 = np.zeros((NH, 16), np.float32), np.zeros((48, NH), np.float32)
        W1[:, :NIN] = rng.standard_normal((NH, NIN)) * 0.5
        W3[:NOUT] = rng.standard_normal((NOUT, NH)) * 0.08
        b3 = np.zeros(48, np.float32)
        b3[:NOUT] = rng.standard_normal(NOUT) * 0.1
        out.append((W1, (rng.standard_normal(NH) * 0.3).astype(np.float32),
                    (rng.standard_normal((NH, NH)) * 0.08).astype(np.float32),
                    (rng.standard_normal(NH) * 0.1).astype(np.float32), W3, b3))
    return out


def _scaling(X, Y):
    """Mean and standard deviation of the network's inputs and targets."""
    z = np.stack([X[:, 0], np.log(X[:, 1]), np.log(X[:, 2]), X[:, 3]], axis=1).astype(np.float64)
    f = lambda a, b: (a.mean(0).astype(np.float32), np.maximum(a.std(0), b).astype(np.float32))  # noqa: E731
    return (*f(z, 1e-3), *f(Y.astype(np.float64), 1e-3))


def prepare(case, seed):
    kind = case["kind"]
    s = dict(case=case)
    if kind in ("step", "round", "observe"):
        na, p = _agents(case), _params(case)
        n = 2 * na
        x, v = _dimers(na, case["L"], p["r0"], 2, p["kBT"], _gen(seed))
        sim = s["sim"] = Sim(case["L"], n, seed=int(seed), **p)
        sim.set_state(x, v)
        if kind == "step":
            s["out"] = [torch.empty(n, 2, dtype=d, device="cuda") for d in (torch.float64, torch.float32, torch.float32)]
        if kind == "round":
            pin = lambda d: torch.empty(n, 2, dtype=d, pin_memory=True)  # noqa: E731
            s["in"], s["out"] = ([pin(d) for d in (torch.float64, torch.float32, torch.float32)] for _ in range(2))
            sim.get_state(*s["in"])
    elif kind == "ensemble":
        pts = _points(case, seed)
        ens = s["ens"] = Ensemble(pts)
        n = sum(p["n_beads"] for p in pts)
        s["out"] = [torch.empty(n, 2, dtype=d, device="cuda") for d in (torch.float64, torch.float32, torch.float32)]
        at, gen, s["views"] = 0, _gen(seed), []
        for r, p in enumerate(pts):
            x, v = _dimers(p["n_beads"] // 2, p["L"], p["r0"], 2, p["kBT"], gen)
            ens.replica(r).set_state(x, v)
            s["views"].append((ens.replica(r), [o[at:at + p["n_beads"]] for o in s["out"]]))
            at += p["n_beads"]
    elif kind in ("cube", "observe3"):
        na, p = _agents(case), _params(case)
        x, v = _dimers(na, case["L"], p["r0"], 3, p["kBT"], _gen(seed))
        sim = s["sim"] = Sim3(case["L"], 2 * na, seed=int(seed), **p)
        sim.set_positions(x.cpu().numpy(), v.cpu().numpy())
    else:
        X = _rows(case, seed)
        Y = _targets(X, seed)
        sur = s["sur"] = Surrogate(members=MEMBERS, max_rows=max(128, case["rows"]), seed=int(seed))
        for k, w in enumerate(_weights(seed)):
            sur.set_weights(k, w)
        sur.set_scaling(*_scaling(X, Y))
        s.update(X=X, Y=Y)
    return s


# ------------------------------------------------------------------- a pass ----
def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "step":
        s["sim"].step(case["steps"])
        s["sim"].get_state(*s["out"])
        return dict(zip("xvf", s["out"]))
    if kind == "round":
        s["sim"].set_state(*s["in"], step=0)
        s["sim"].step(1)
        s["sim"].get_state(*s["out"])
        return dict(zip("xvf", s["out"]))
    if kind == "ensemble":
        s["ens"].step(case["steps"])
        s["ens"].sync()
        for view, out in s["views"]:
            view.get_state(*out)
        return dict(zip("xvf", s["out"]))
    if kind == "cube":
        s["sim"].step(case["steps"])
        return dict(zip("xvf", s["sim"].get_state()[:3]))
    if kind in ("observe", "observe3"):
        sim = s["sim"]
        out = dict(E=sim.energy_spectrum(case["M"]))
        if case["nbins"]:
            out["g"], out["L_int"], out["num"], out["cnt"] = sim.velocity_correlation(case["dr"], case["nbins"])
        if kind == "observe":
            out["T"], out["speed"] = sim.temperature(), sim.agent_speed()
        else:
            out["T"] = sim.thermo()[4]
        if case["field"]:
            out["u"], out["n"] = sim.velocity_field(case["M"])
            out["omega"] = sim.vorticity(case["M"])
        return out
    if kind == "fit":
        sur, X, Y, b = s["sur"], s["X"], s["Y"], case["batch"]
        loss0, grads = sur.gradients(0, X[:b], Y[:b])
        loss = sur.fit(X, Y, epochs=case["epochs"], batch=b)
        mean, spread = sur.predict(X)
        return dict(loss0=loss0, grads=grads, loss=loss, mean=mean, spread=spread)
    mean, spread = s["sur"].predict(s["X"])
    return dict(mean=mean, spread=spread)


def work(case):
    """Steps: per bead and step 36 bytes (read X, Y, v, id, write X, Y, v; 52 in three dimensions), 110
    operations per interacting pair (Philox and force) and 70 per bead; the states and tables that come back
    once.  Correlation: 12 operations per pair inside r_max.  Surrogate: the matrix products."""
    kind = case["kind"]
    if kind in ("step", "round", "ensemble"):
        boxes = ([(p["n_beads"], p["L"], 1.0) for p in _points(case, 0)] if kind == "ensemble"
                 else [(2 * _agents(case), case["L"], _params(case)["rc"])])
        n = sum(b[0] for b in boxes)
        ops = sum(b[0] * (70.0 + 110.0 * 0.5 * math.pi * b[2] ** 2 * b[0] / b[1] ** 2) for b in boxes)
        k = case.get("steps", 1)
        return dict(bytes=36.0 * n * k + (64.0 if kind == "round" else 32.0) * n, flops=ops * k)
    if kind == "cube":
        n = 2 * _agents(case)
        return dict(bytes=(52.0 * case["steps"] + 48.0) * n,
                    flops=case["steps"] * n * (70.0 + 110.0 * 2.0 / 3.0 * math.pi * n / case["L"] ** 3))
    if kind in ("observe", "observe3"):
        na, d, M = _agents(case), 2 if kind == "observe" else 3, case["M"]
        r = min(case["nbins"] * case["dr"], case["L"] / 2)
        pairs = 0.5 * na * na / case["L"] ** d * (math.pi * r * r if d == 2 else 4.0 / 3.0 * math.pi * r ** 3)
        cells, field = M ** d, 1 if case["field"] else 0
        return dict(bytes=(32.0 if d == 2 else 64.0) * na * (2 + field) + 24.0 * case["nbins"] +
                    cells * field * 16.0 * d, flops=12.0 * pairs + cells * 5.0 * d * math.log2(M) * (d - 1) + 40.0 * na)
    mlp = 2.0 * (NIN * NH + NH * NH + NH * NOUT) * MEMBERS
    n = case["rows"]
    if kind == "predict":
        return dict(bytes=n * 4.0 * (NIN + 2 * NOUT) + 2.0 * mlp / 2.0, flops=n * mlp)
    steps = n // case["batch"] * case["epochs"]
    return dict(bytes=n * 4.0 * (NIN + NOUT) * (1 + case["epochs"]) + n * 4.0 * 2 * NOUT + steps * 14.0 * mlp,
                flops=steps * case["batch"] * 3.0 * mlp + n * mlp)


# -------------------------------------------------- the same in 64 bits ----
def _mulhilo(a, b):
    t = a * (b & 0xFFFF)
    u = a * (b >> 16) + (t >> 16)
    return u >> 16, ((u & 0xFFFF) << 16) | (t & 0xFFFF)


def _philox(c, k0, k1):
    c0, c1, c2, c3 = c
    for r in range(10):
        h0, l0 = _mulhilo(0xD2511F53, c0)
        h1, l1 = _mulhilo(0xCD9E8D57, c2)
        c0, c1, c2, c3 = h1 ^ c1 ^ k0, l1, h0 ^ c3 ^ k1, l0
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    return c0, c1


def _half_pairs(x, L, n, base, ncell, most=20_000_000):
    """Every pair of points in the same or adjacent cells of a periodic grid of n cells a side, once: chunks
    of (first, second) indexes.  L, n, base: numbers, or a value for each point."""
    dim = x.shape[1]
    c = (x / (L[:, None] if torch.is_tensor(L) else L) * (n[:, None] if torch.is_tensor(n) else n)).floor().long()
    top = (n[:, None] if torch.is_tensor(n) else torch.full_like(c[:, :1], n)) - 1
    c = torch.minimum(c.clamp_(min=0), top)
    m = top[:, 0] + 1

    def flat(q):
        f = q[:, dim - 1]
        for d in range(dim - 2, -1, -1):
            f = f * m + q[:, d]
        return f + base

    cell, order = torch.sort(flat(c))
    count = torch.bincount(cell, minlength=ncell)
    start = torch.cumsum(count, 0) - count
    c, m = c[order], m[order]
    base = base[order] if torch.is_tensor(base) else base
    me = torch.arange(len(x), device=x.device)
    for k in range(3 ** dim // 2, 3 ** dim):   # own cell, then the half of the others that comes after it
        off = [(k // 3 ** d) % 3 - 1 for d in range(dim)]
        if k == 3 ** dim // 2:
            first, num = me + 1, start[cell] + count[cell] - me - 1
        else:
            nb = flat(torch.stack([torch.remainder(c[:, d] + off[d], m) for d in range(dim)], 1))
            first, num = start[nb], count[nb]
        ends = torch.cumsum(num, 0)
        total, at = int(ends[-1]), 0
        while at < len(x) and total:
            done = int(ends[at - 1]) if at else 0
            to = max(at + 1, int(torch.searchsorted(ends, done + most, right=True)))
            nn = num[at:to]
            i = torch.repeat_interleave(me[at:to], nn)
            j = torch.arange(len(i), device=x.device) + torch.repeat_interleave(first[at:to] - (ends[at:to] - nn - done), nn)
            if len(i):
                yield order[i], order[j]
            at = to


def _at(a, i):
    return a[i] if torch.is_tensor(a) else a


def _minimg(d, L):
    L = L[:, None] if torch.is_tensor(L) else L
    return d - L * torch.round(d / L)


def _forces(x, v, step, q):
    """Total force on every bead; q: the parameters, numbers or a value for each bead."""
    col = lambda a: a[:, None] if torch.is_tensor(a) else a  # noqa: E731
    f = -col(q["zeta"]) * v
    d = _minimg(x[0::2] - x[1::2], _at(q["L"], slice(0, None, 2)))
    r = d.norm(dim=1, keepdim=True)
    u, t = d / r, -q["k_bond"] * (r - q["r0"])
    fp = col(_at(q["f_p"], slice(0, None, 2)))
    f[0::2] += (t + fp) * u
    f[1::2] += (fp - t) * u
    ids = q["ids"]
    for i, j in _half_pairs(x, q["L"], q["n"], q["base"], q["ncell"]):
        L = _at(q["L"], i)
        d = _minimg(x[i] - x[j], L)
        r2 = (d * d).sum(1)
        ok = (r2 < q["rc"] ** 2) & (r2 > 0) & (i != (j ^ 1))
        i, j, d, r = i[ok], j[ok], d[ok], r2[ok].sqrt()
        if not len(i):
            continue
        e, w = d / r[:, None], 1.0 - r / q["rc"]
        dve = ((v[i] - v[j]) * e).sum(1)
        a, b = ids[i], ids[j]
        c = (torch.minimum(a, b), torch.maximum(a, b), torch.full_like(a, step & 0xFFFFFFFF), torch.full_like(a, step >> 32))
        w0, w1 = _philox(c, q["key0"], _at(q["key1"], i))
        if q.get("noise"):
            z = torch.sqrt(-2.0 * torch.log(((w0 >> 8) + 0.5) * 2.0 ** -24)) * torch.cos(2.0 * math.pi * ((w1 >> 8) + 0.5) * 2.0 ** -24)
        else:
            z = math.sqrt(3.0) * (2 * (w0 >> 8) + 1 - 2 ** 24).double() * 2.0 ** -24
        g = _at(q["gamma"], i)
        sig = (2.0 * g * q["kBT"] / q["dt"]) ** 0.5
        ex = q.get("wexp") or 2.0
        F = (q["a"] * w - g * w ** ex * dve + sig * w ** (0.5 * ex) * z)[:, None] * e
        f.index_add_(0, i, F)
        f.index_add_(0, j, -F)
    return f


def _advance(x, v, q, steps):
    h, v = 0.5 * q["dt"] / q["mass"], v.double()
    f = _forces(x, v, 0, q)
    for s in range(1, steps + 1):
        v = v + h * f
        x = x + q["dt"] * v
        x = torch.remainder(x, q["L"][:, None] if torch.is_tensor(q["L"]) else q["L"])
        f = _forces(x, v, s, q)
        v = v + h * f
    return dict(x=x, v=v, f=f)


def _system(case, seed, dim):
    p, na = _params(case), _agents(case)
    x, v = _dimers(na, case["L"], p["r0"], dim, p["kBT"], _gen(seed))
    n = int(case["L"] / p["rc"])
    return x, v, dict(p, L=case["L"], n=n, base=0, ncell=n ** dim, ids=torch.arange(2 * na, device=x.device),
                      key0=int(seed) & 0xFFFFFFFF, key1=int(seed) >> 32)


def _window(c, L, M, half):
    """For each point, the grid indexes whose window may hold it and whether it does, axis by axis."""
    dx = L / M
    k = min(M, int(math.ceil(2.0 * half / dx)) + 3)
    i = torch.floor((c - half) / dx - 0.5)[..., None] + torch.arange(k, device=c.device, dtype=torch.float64) - 1.0
    d = (torch.remainder(i, M) + 0.5) * dx - c[..., None]
    return torch.remainder(i, M).long(), (d - L * torch.round(d / L)).abs() <= half


def _field(c, v, L, M):
    na, dim = c.shape
    half = 0.5 * L * (10.0 / na) ** (1.0 / dim)
    i, ok = _window(c, L, M, half)
    sums = torch.zeros(M ** dim, dim + 1, dtype=torch.float64, device=c.device)
    v1 = torch.cat([v, torch.ones_like(v[:, :1])], 1)
    k = i.shape[-1]
    for o in range(k ** dim):
        t = [(o // k ** d) % k for d in range(dim)]
        hit = torch.stack([ok[:, d, t[d]] for d in range(dim)]).all(0)
        g = sum(i[hit, d, t[d]] * M ** d for d in range(dim))
        sums.index_add_(0, g, v1[hit])
    n = sums[:, dim]
    u = torch.where(n[:, None] > 0, sums[:, :dim] / n.clamp(min=1.0)[:, None], torch.zeros_like(sums[:, :dim]))
    return u.reshape(*[M] * dim, dim), n.reshape(*[M] * dim)


def _exact_observe(case, seed):
    dim = 2 if case["kind"] == "observe" else 3
    x, v, q = _system(case, seed, dim)
    L, M, v = case["L"], case["M"], v.double()
    c = torch.remainder(x[1::2] + 0.5 * _minimg(x[0::2] - x[1::2], L), L)
    vc = 0.5 * (v[0::2] + v[1::2])
    na = len(c)
    u, n = _field(c, vc, L, M)
    Z = torch.fft.fftn(u.to(torch.complex128), dim=tuple(range(dim))) / M ** dim
    k = torch.fft.fftfreq(M, 1.0 / M, dtype=torch.float64, device=c.device)
    k2 = sum(k.reshape([-1 if d == e else 1 for e in range(dim)]) ** 2 for d in range(dim))
    sh = torch.round(torch.sqrt(k2)).long().flatten()
    E = torch.zeros(M * dim, dtype=torch.float64, device=c.device)
    E.index_add_(0, sh, (0.5 * Z.abs() ** 2).sum(-1).flatten())
    out = dict(E=E[1:M // 2 + 1])
    if case["nbins"]:
        dr, nb = case["dr"], case["nbins"]
        num = torch.zeros(nb, dtype=torch.float64, device=c.device)
        cnt = torch.zeros(nb, dtype=torch.float64, device=c.device)
        nv = int(L / (nb * dr * (1 + 1e-9)))
        pairs = _half_pairs(c, L, nv, 0, nv ** dim) if nv >= 3 else (
            (torch.arange(a, min(a + 500, na), device=c.device).repeat_interleave(na), torch.arange(na, device=c.device).repeat(min(500, na - a)))
            for a in range(0, na, 500))
        for i, j in pairs:
            if nv < 3:
                i, j = i[i < j], j[i < j]
            b = torch.floor(_minimg(c[i] - c[j], L).norm(dim=1) / dr).long()
            ok = b < nb
            i, j, b = i[ok], j[ok], b[ok]
            num += torch.bincount(b, (vc[i] * vc[j]).sum(1), nb)
            cnt += torch.bincount(b, minlength=nb)
        m2, v2 = float((vc.mean(0) ** 2).sum()), float((vc ** 2).sum(1).mean())
        g = torch.where(cnt > 0, (num / cnt - m2) / (v2 - m2), torch.full_like(num, math.nan))
        li, rp, gp = 0.0, 0.0, 1.0
        for b, gv in enumerate(g.tolist()):
            if gv == gv:
                r = (b + 0.5) * dr
                li, rp, gp = li + 0.5 * (gv + gp) * (r - rp), r, gv
        out.update(g=g, L_int=li, num=num, cnt=None)
    out["T"] = float((v ** 2).sum()) / (dim * (2.0 * na - 1.0))
    if dim == 2:
        out["speed"] = float(vc.norm(dim=1).mean())
    if case["field"]:
        D = lambda comp, axis: (torch.roll(u[..., comp], -1, axis) - torch.roll(u[..., comp], 1, axis)) * (M / (2.0 * L))  # noqa: E731
        out.update(u=u, n=n, omega=D(1, 1) - D(0, 0) if dim == 2 else
                   torch.stack([D(2, 1) - D(1, 0), D(0, 0) - D(2, 2), D(1, 2) - D(0, 1)], -1))
    return out


def _exact_mlp(case, seed):
    """Predictions, and for "fit" the loss and gradients of the first member at the initial weights."""
    dev = dict(dtype=torch.float64, device="cuda")
    X = _rows(case, seed)
    Y = _targets(X, seed)
    mx, sx, my, sy = (torch.tensor(a, **dev) for a in _scaling(X, Y))
    x, y = torch.tensor(X, **dev), torch.tensor(Y, **dev)
    z = (torch.stack([x[:, 0], x[:, 1].log(), x[:, 2].log(), x[:, 3]], 1) - mx) / sx
    net = lambda z, W: (torch.nn.functional.silu(torch.nn.functional.silu(z @ W[0].T + W[1]) @ W[2].T + W[3])  # noqa: E731
                        @ W[4].T + W[5])[:, :NOUT]
    if case["kind"] == "predict":
        o = torch.stack([net(z, [torch.tensor(a, **dev)[:, :NIN] if k == 0 else torch.tensor(a, **dev) for k, a in enumerate(w)])
                         for w in _weights(seed)]) * sy + my
        return dict(mean=o.mean(0), spread=o.std(0, unbiased=False))
    b = case["batch"]
    W = [torch.tensor(a, requires_grad=True, **dev) for a in _weights(seed)[0]]
    zp = torch.cat([z[:b], torch.zeros(b, 12, **dev)], 1)
    loss = ((net(zp, W) - (y[:b] - my) / sy) ** 2).mean()
    loss.backward()
    return dict(loss0=float(loss.detach()), grads=[w.grad for w in W], loss=None, mean=None, spread=None)


def exact(case, seed):
    kind = case["kind"]
    if kind in ("step", "round", "cube"):
        x, v, q = _system(case, seed, 3 if kind == "cube" else 2)
        return _advance(x, v, q, case.get("steps", 1))
    if kind == "ensemble":
        pts, gen = _points(case, seed), _gen(seed)
        xv = [_dimers(p["n_beads"] // 2, p["L"], p["r0"], 2, p["kBT"], gen) for p in pts]
        n = torch.tensor([p["n_beads"] for p in pts], device="cuda")
        per = lambda a, d=torch.float64: torch.tensor(a, dtype=d, device="cuda").repeat_interleave(n)  # noqa: E731
        side = [int(p["L"] / p["rc"]) for p in pts]
        cells = [0, *np.cumsum([s * s for s in side]).tolist()]
        q = dict(BASE, L=per([p["L"] for p in pts]), n=per(side, torch.int64), base=per(cells[:-1], torch.int64),
                 ncell=cells[-1], gamma=per([p["gamma"] for p in pts]), zeta=per([p["zeta"] for p in pts]),
                 f_p=per([p["f_p"] for p in pts]), key0=int(seed) & 0xFFFFFFFF,
                 key1=per([(int(seed) >> 32) ^ p["replica"] for p in pts], torch.int64),
                 ids=torch.cat([torch.arange(p["n_beads"], device="cuda") for p in pts]))
        return _advance(torch.cat([a for a, _ in xv]), torch.cat([b for _, b in xv]), q, case["steps"])
    return _exact_observe(case, seed) if kind in ("observe", "observe3") else _exact_mlp(case, seed)
