"""The work that users of this package have it do, as cases to be measured.

Every case is one suspension (or one batch of them) and one call of a user's
program on it:

  step     ``Suspension.step`` / ``Batch.step`` of a handle that stays on the
           GPU, then a read of the state and of the stress, as a run does
           between two outputs;
  forces   ``Suspension.forces``: one evaluation of the total force and torque
           at the present state;
  io       ``Suspension.step_io`` from and to pinned host buffers: the package
           inside another program that owns the state (a step per call);
  adjoint  ``Suspension.adjoint``: the gradient of the time-averaged viscosity
           over a rollout (the backward direction).

Sizes, radii, volume fractions and force settings are those of
``synth.SPECS``, ``synth.BATCH_SPECS`` and ``bench.py`` and the ranges between
them.  The packings are made here, on the GPU, from the seed alone: uniform
random centres and Jacobi sweeps that push overlapping spheres apart, with sums
taken in integers so that the same seed gives the same bytes everywhere.

In mixed precision forces, torques and accelerations are FP32 numbers, and
what is integrated from them and the stress carry their rounding: these
outputs are returned as the FP32 a user stores them in.  Positions, and every
output in FP64 precision, are returned as FP64.
"""
import math

import numpy as np
import torch

import paper_2108_01013_gb300 as dss

F64 = torch.float64

# Force settings: the lubrication range, and the electro-chemical forces of
# the paper's Tables 3 (repulsion), 4 (with attraction) and 5 (radius ratio 3).
FORCES = {
    "contact": dict(kn=1e4, dt=1e-4),
    "repulsion": dict(kn=1e4, dt=1e-4, f_er=10.0, lambda_d=0.05, delta_lub=0.10),
    "attraction": dict(kn=1e4, dt=1e-4, f_er=10.0, lambda_d=0.0225, hamaker=10.0 / 19.0 * 12.0 * 1e-4,
                       vdw_eps=0.01, delta_lub=0.25),
    "table5": dict(kn=4e5, kt=4e5 * 2.0 / 7.0, dt=1e-7, rho=1e-3, delta_lub=0.25, lub_cutoff_mode=1, f_er=1.0,
                   lambda_d=0.02, hamaker=12.0 * 1e-4 / 19.0, vdw_eps=0.01),
}
# Radii of a packing: the smallest cell edge the box has to hold four of is
# twice the largest (plus the range), which bounds n from below.
RADII = ("bidisperse", "ratio3", "loguniform")


def _case(name, kind, n, precision, steps, *, radii="bidisperse", phi=0.55, mu=0.5, forces="contact", wave=0.0,
          rolling=False, instances=1):
    c = dict(kind=kind, n=n, precision=precision, steps=steps, radii=radii, phi=phi, mu=mu, forces=forces, wave=wave,
             rolling=rolling, instances=instances)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest run in use: a thousand spheres in FP64 (validation
        # against the oracle, parameter studies); launches and latency
        _case("step_1k_fp64", "step", 1000, "fp64", 40, phi=0.50),
        # a mid-size mixed run of ragged size: less than one wave of warps
        _case("step_20k_mixed", "step", 20_011, "mixed", 40, phi=0.54),
        # the headline workload: 100k spheres, phi = 0.55, mu = 1, mixed precision
        _case("step_100k_mixed", "step", 100_000, "mixed", 20, phi=0.55, mu=1.0),
        # the same in FP64 precision
        _case("step_100k_fp64", "step", 100_000, "fp64", 10, phi=0.55, mu=1.0),
        # the polydisperse million: log-uniform radii, cells of 20 a_min
        _case("step_1m_poly_mixed", "step", 1_000_000, "mixed", 8, radii="loguniform", phi=0.50),
        # a flow-curve sweep: many suspensions of 500 to 20,000 spheres in one handle
        _case("batch_64_mixed", "step", 640_000, "mixed", 10, phi=0.50, instances=64),
        # double-layer repulsion: pairs listed out to one radius
        _case("repulsion_100k_mixed", "step", 100_000, "mixed", 10, phi=0.55, mu=1.0, forces="repulsion"),
        # Table 5: radius ratio 3, attraction out to four radii, wavy shear, rolling resistance
        _case("table5_65k_mixed", "step", 65_536, "mixed", 8, radii="ratio3", phi=0.50, mu=1.0, forces="table5",
              wave=20.0, rolling=True),
        # one evaluation of the forces (a coupling code, an analysis script), odd size
        _case("forces_50k_fp64", "forces", 50_021, "fp64", 1, phi=0.50),
        # a host program that owns the state: upload, one step, read back
        _case("io_100k_mixed", "io", 100_000, "mixed", 1, phi=0.55, mu=1.0),
        # the gradient of the mean viscosity of 20k spheres over 40 steps
        _case("adjoint_20k_mixed", "adjoint", 20_000, "mixed", 40, phi=0.54),
    ]


def draw(rng):
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    mu = rng.choice((0.0, 0.2, 0.5, 1.0))
    phi = round(rng.uniform(0.40, 0.56), 3)
    prec = rng.choice(("mixed", "mixed", "fp64"))
    what = rng.choice(("step", "step", "step", "poly", "batch", "echem", "table5", "forces", "io", "adjoint"))
    if what == "poly":
        n = size(5_000, 1_000_000 if prec == "mixed" else 250_000)
        return _case("", "step", n, prec, rng.randint(1, 8), radii="loguniform", phi=min(phi, 0.50), mu=mu)
    if what == "batch":
        k = size(2, 64)
        return _case("", "step", k * size(700, 10_000 if prec == "mixed" else 2_500), prec, rng.randint(1, 10), phi=phi,
                     mu=mu, instances=k)
    if what == "echem":
        f = rng.choice(("repulsion", "attraction"))
        n = size(6_000, 60_000 if f == "attraction" else 200_000)
        n = n // 4 if prec == "fp64" else n
        return _case("", "step", max(n, 6_000), prec, rng.randint(1, 8), phi=phi, mu=mu, forces=f,
                     rolling=rng.random() < 0.3)
    if what == "table5":
        n = size(12_000, 65_536 if prec == "mixed" else 16_000)
        return _case("", "step", n, prec, rng.randint(1, 6), radii="ratio3", phi=min(phi, 0.50), mu=mu, forces="table5",
                     wave=rng.choice((0.0, 20.0)), rolling=rng.random() < 0.5)
    if what == "forces":
        return _case("", "forces", size(500, 500_000 if prec == "mixed" else 150_000), prec, 1, phi=phi, mu=mu)
    if what == "io":
        return _case("", "io", size(500, 400_000 if prec == "mixed" else 150_000), prec, rng.randint(1, 3), phi=phi, mu=mu)
    if what == "adjoint":
        return _case("", "adjoint", size(1_000, 20_000), prec, rng.randint(5, 40), phi=phi, mu=mu)
    n = size(500, 800_000 if prec == "mixed" else 150_000)
    return _case("", "step", n, prec, rng.randint(1, 40 if n < 50_000 else 10), phi=phi, mu=mu,
                 rolling=rng.random() < 0.15)


# --------------------------------------------------------------------------
# inputs
# --------------------------------------------------------------------------
def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _sizes(case):
    """Particle counts of the instances: spread over a factor of 40 in a batch,
    as a sweep from 500 to 20,000 has it."""
    n, k = case["n"], case["instances"]
    if k == 1:
        return np.array([n], dtype=np.int64)
    w = np.linspace(1.0, 40.0, k)[np.random.RandomState(k).permutation(k)]
    free = n - 500 * k
    s = 500 + np.floor(max(free, 0) * w / w.sum()).astype(np.int64)
    s[-1] += max(n - int(s.sum()), 0)
    return s


def _radii(case, sizes, rng):
    out = []
    for n in sizes:
        n = int(n)
        if case["radii"] == "loguniform":
            a = np.exp(rng.rand(n) * math.log(10.0))
        else:
            large, frac = (1.4, 0.5) if case["radii"] == "bidisperse" else (3.0, (0.25 / 27.0) / (1.0 + 0.25 / 27.0))
            a = np.ones(n)
            a[:int(round(frac * n))] = large
            a = a[rng.permutation(n)]
        out.append(a)
    return out


def _ranges(first, last):
    """(p, q) for every p and every q in [first[p], last[p])."""
    cnt = (last - first).clamp_(min=0)
    p = torch.repeat_interleave(torch.arange(cnt.numel(), device=cnt.device), cnt)
    q = torch.arange(p.numel(), device=cnt.device) + (first - (cnt.cumsum(0) - cnt))[p]
    return p, q


def _near_pairs(x, a, inst, L, off, reach):
    """Index pairs i < j whose centres are within a_i + a_j + reach (plus a
    rounding margin) in boxes sheared by off along x: cells of the extended
    (ghost) boxes, each row of cells one range.  x (3, n), L and off per
    instance."""
    n, dev = a.numel(), a.device
    rc = float(2.0 * a.max()) + reach
    X, idx = x, torch.arange(n, device=dev)
    for d in (1, 0, 2):                      # images along y (sheared), then x, then z
        for s in (-1.0, 1.0):
            Lg = L[inst[idx[: X.shape[1]]]]
            m = ((X[d] > Lg - rc) if s < 0 else (X[d] < rc)) & (X[d] >= 0) & (X[d] < Lg)
            g = X[:, m].clone()
            g[d] += s * Lg[m]
            if d == 1:
                g[0] = torch.remainder(g[0] + s * off[inst[idx[m]]], Lg[m])
            X, idx = torch.cat([X, g], 1), torch.cat([idx, idx[m]])
    real = torch.arange(idx.numel(), device=dev) < n
    Lx = L + 2.0 * rc
    nc = torch.floor(Lx / rc).to(torch.int64)
    base = torch.cumsum(nc ** 3, 0) - nc ** 3
    k = inst[idx]
    c = torch.minimum(torch.floor((X + rc) * (nc[k] / Lx[k])).to(torch.int64).clamp_(min=0), nc[k] - 1)
    key = base[k] + (c[1] * nc[k] + c[2]) * nc[k] + c[0]
    key, order = torch.sort(key, stable=True)
    X, idx, real, c, k = X[:, order].contiguous(), idx[order], real[order], c[:, order], k[order]
    start = torch.searchsorted(key, torch.arange(int((nc ** 3).sum()) + 1, device=dev))
    me = torch.arange(idx.numel(), device=dev)
    A, m, w = a[idx], nc[k], nc[k]
    out = []
    for dy, dz in ((0, 0), (0, 1), (1, -1), (1, 0), (1, 1)):
        ok = (c[1] + dy < m) & (c[2] + dz >= 0) & (c[2] + dz < m)
        row = key + (dy * w + dz) * w - c[0]
        row = torch.where(ok, row, 0)
        hi = start[row + torch.minimum(c[0] + 1, m - 1) + 1]
        lo = me + 1 if (dy, dz) == (0, 0) else start[row + (c[0] - 1).clamp(min=0)]
        p, q = _ranges(lo, torch.where(ok, hi, lo))
        cut = A[p] + A[q] + reach
        r2 = sum((X[d][q] - X[d][p]) ** 2 for d in range(3))
        i, j = idx[p], idx[q]
        keep = (r2 < (cut * (1.0 + 1e-9)) ** 2) & torch.where(real[p] & real[q], True, torch.where(
            real[p], i < j, real[q] & (j < i)))
        i, j = i[keep], j[keep]
        out.append(torch.stack([torch.minimum(i, j), torch.maximum(i, j)]))
    return torch.cat(out, 1)


def _separation(x, L, off, i, j, inst):
    """Minimum image of x_j - x_i in the sheared boxes (3, p), and the y shift."""
    Lp = L[inst[i]]
    d = x[:, j] - x[:, i]
    sy = torch.where(d[1] > 0.5 * Lp, -1.0, torch.where(d[1] < -0.5 * Lp, 1.0, 0.0)).to(F64)
    dx = d[0] + sy * off[inst[i]]
    return torch.stack([dx - Lp * torch.round((dx / Lp).detach()), d[1] + sy * Lp,
                        d[2] - Lp * torch.round((d[2] / Lp).detach())]), sy


def _pack(a, inst, L, rng_seed, sweeps):
    """Centres of a random packing: uniform, then Jacobi sweeps in which each
    sphere moves away from those it overlaps by 0.8 of its share of the
    overlap (the larger moves less); candidates are listed anew every fourth
    sweep."""
    gen = torch.Generator(device="cpu").manual_seed(rng_seed)
    n, dev = a.numel(), a.device
    Lp = L[inst]
    x = torch.rand((3, n), generator=gen, dtype=F64).to(dev) * Lp
    off = torch.zeros_like(L)
    v = a ** 3
    for s in range(sweeps):
        if s % 4 == 0:
            i, j = _near_pairs(x, a, inst, L, off, 0.3)
            S, wi = a[i] + a[j], v[j] / (v[i] + v[j])
        r, _ = _separation(x, L, off, i, j, inst)
        rr = torch.sqrt((r * r).sum(0)).clamp_(min=1e-9)
        o = 0.8 * (S - rr).clamp_(min=0.0) / rr * r * float(1 << 40)
        mv = torch.zeros((3, n), dtype=torch.int64, device=dev)
        mv.index_add_(1, i, -torch.round(o * wi).to(torch.int64))
        mv.index_add_(1, j, torch.round(o * (1.0 - wi)).to(torch.int64))
        x = torch.remainder(x + mv.to(F64) / float(1 << 40), Lp)
        x = torch.where(x >= Lp, 0.0, x)
    return x


def _inputs(case, seed):
    sizes = _sizes(case)
    rng = np.random.RandomState(seed)
    radii = _radii(case, sizes, rng)
    K = len(sizes)
    phi = np.full(K, case["phi"])
    gdot = np.ones(K)
    if K > 1:      # a flow curve: every instance its own density and shear rate
        phi = rng.uniform(0.40, 0.56, K)
        gdot = np.exp(rng.uniform(math.log(1e-2), math.log(1e2), K))
    L = np.array([(4.0 / 3.0 * math.pi * float((r ** 3).sum()) / f) ** (1.0 / 3.0) for r, f in zip(radii, phi)])
    dev = _device()
    a = torch.from_numpy(np.concatenate(radii)).to(dev)
    inst = torch.repeat_interleave(torch.arange(K), torch.from_numpy(sizes)).to(dev)
    sweeps = 40 if case["radii"] == "loguniform" else 60
    x = _pack(a, inst, torch.from_numpy(L).to(dev), seed, sweeps)
    return dict(x=x, a=a, inst=inst, L=L, sizes=sizes, gdot=gdot)


def _settings(case):
    p = dict(FORCES[case["forces"]], mu=case["mu"])
    if case["wave"]:
        p.update(wave_amp=case["wave"], wave_n=1)
    if case["rolling"]:
        p["k_r"] = 0.05 * p["kn"]
    if case["kind"] == "adjoint":
        p["lub_taper"] = 0.2          # a differentiable lubrication cutoff
    return p


def prepare(case, seed):
    g = _inputs(case, seed)
    boxes = np.repeat(g["L"][:, None], 3, axis=1)
    p = dss.default_params(precision=case["precision"], **_settings(case))
    if case["instances"] > 1:
        h = dss.Batch(g["x"], g["a"], g["sizes"], boxes, g["gdot"], p)
    else:
        h = dss.Suspension(g["x"], g["a"], boxes[0], p)
    st = dict(case=case, handle=h)
    if case["kind"] == "io":
        st["host"] = [torch.empty((3, h.n), dtype=F64, pin_memory=True) for _ in range(5)]
        st["sigma"] = torch.empty(9, dtype=F64, pin_memory=True)
        h.get_state_into(*st["host"])
    if case["kind"] == "adjoint":
        st["weights"] = dss.viscosity_weights(case["steps"])
    return st


def _as_stored(case, v):
    """FP32 in mixed precision (see the module's comment)."""
    if case["precision"] != "mixed":
        return v
    return v.float() if isinstance(v, torch.Tensor) else np.asarray(v, dtype=np.float32)


def run(state):
    c, h = state["case"], state["handle"]
    if c["kind"] == "forces":
        F, T = h.forces()
        return dict(F=_as_stored(c, F), T=_as_stored(c, T))
    if c["kind"] == "io":
        h.step_io(state["host"], c["steps"], state["host"], state["sigma"])
        return dict(zip(("x", "u", "w", "al", "aw"), [state["host"][0]] + [_as_stored(c, v) for v in state["host"][1:]]),
                    sigma=_as_stored(c, state["sigma"]))
    if c["kind"] == "adjoint":
        r = h.adjoint(c["steps"], state["weights"], ckpt_every=20)
        return {k: _as_stored(c, v) for k, v in r.items()}
    h.step(c["steps"])
    out = h.state()
    out = {k: v if k == "x" else _as_stored(c, v) for k, v in out.items()}
    out["sigma"] = _as_stored(c, h.batch_stress()[0] if c["instances"] > 1 else h.stress())
    return out


def work(case):
    """Bytes: per particle and step the state read and written (x, u, w, a,
    id: 84 each way; FP32 or FP64 forces written; the integration's 288), the
    pair list written and read, the contact history (key and stretch) read and
    written, the cell table.  Flops: some 300 a listed pair and 9 a candidate
    of the half stencil.  Densities as in random packings of these sizes."""
    n = case["n"]
    pairs, cont, cells, cand = {"contact": (3.0, 1.5, 0.6, 24.0), "repulsion": (5.7, 1.5, 0.25, 55.0),
                                "attraction": (38.0, 1.5, 0.02, 600.0), "table5": (45.0, 1.5, 0.008, 1800.0)}[case["forces"]]
    if case["radii"] == "loguniform":
        pairs, cont, cells, cand = 1.2, 0.6, 0.14, 100.0
    f = 24.0 if case["precision"] == "mixed" else 48.0
    one = n * (168.0 + f + 8.0 * pairs + 64.0 * cont + 8.0 * cells)
    flops = n * (300.0 * pairs + 9.0 * cand)
    if case["kind"] == "forces":
        return dict(bytes=float(one), flops=float(flops))
    step = one + 288.0 * n
    if case["kind"] == "adjoint":      # forward, taped replay, reverse
        return dict(bytes=3.0 * case["steps"] * step, flops=5.0 * case["steps"] * flops)
    out = 240.0 * n if case["kind"] == "io" else 120.0 * n
    return dict(bytes=float(case["steps"] * step + out), flops=float(case["steps"] * flops))


# --------------------------------------------------------------------------
# the same in plain FP64 tensor operations
# --------------------------------------------------------------------------
def _dot(a, b):
    return (a * b).sum(0)


def _cross(a, b):
    return torch.stack([a[1] * b[2] - a[2] * b[1], a[2] * b[0] - a[0] * b[2], a[0] * b[1] - a[1] * b[0]])


class _Plain:
    """The model: lubrication (Eq. A2-A7), frictional contact with its history
    (Eq. 4-5), electro-chemical forces (Eq. 6-7), rolling resistance (App. B),
    drag (Eq. A1, with the wave of Eq. 17), the velocity-Verlet step of Eq. 15
    and the stress of Eq. 8-9."""

    def __init__(self, case, g):
        p = dict(kt=None, rho=1.0, eta0=1.0, a0=1.0, lub_eps=1e-3, delta_lub=0.05, lub_cutoff_mode=0, lub_taper=0.0,
                 f_er=0.0, lambda_d=0.05, hamaker=0.0, vdw_eps=0.01, wave_amp=0.0, wave_n=0, k_r=0.0)
        p.update(_settings(case))
        p["kt"] = 0.5 * p["kn"] if p["kt"] is None else p["kt"]
        self.p, self.a, self.inst, self.n = p, g["a"], g["inst"], g["a"].numel()
        dev = self.a.device
        self.L = torch.from_numpy(g["L"]).to(dev)
        self.gdot = torch.from_numpy(g["gdot"]).to(dev)
        self.th = {k: torch.tensor(float(v), dtype=F64, device=dev) for k, v in (
            ("kn", p["kn"]), ("kt", p["kt"]), ("gn", 1e-7 * p["kn"]), ("mu", p["mu"]), ("delta", p["delta_lub"]))}
        # the dashpot is 1e-7 k_n / gdot: gn is its value at gdot = 1
        self.wk = 2.0 * math.pi * p["wave_n"] / self.L
        self.m = 4.0 / 3.0 * math.pi * p["rho"] * self.a ** 3
        self.I = 0.4 * self.m * self.a ** 2
        self.range = max(20.0 * p["lambda_d"] if p["f_er"] > 0 else 0.0, 4.0 * p["a0"] if p["hamaker"] > 0 else 0.0)

    def offset(self, step):
        return torch.fmod(self.gdot * self.L * (step * self.p["dt"]), self.L)

    def flow(self, y, inst):
        """U_inf,x and its rate dU_inf,x/dy at heights y."""
        w, k = self.p["wave_amp"], self.wk[inst]
        return self.gdot[inst] * y + w * torch.sin(k * y), self.gdot[inst] + w * k * torch.cos(k * y)

    def forces(self, x, u, w, hist, step):
        p, a, inst, n, th = self.p, self.a, self.inst, self.n, self.th
        off = self.offset(step)
        mean = p["lub_cutoff_mode"] == 0     # the lubrication range: a share of the mean radius, or of a0
        with torch.no_grad():
            far = max(self.range, p["delta_lub"] * (float(a.max()) if mean else p["a0"]))
            i, j = _near_pairs(x.detach(), a, inst, self.L, off, far)
            r, _ = _separation(x.detach(), self.L, off, i, j, inst)
            S = a[i] + a[j]
            dl = p["delta_lub"] * (0.5 * S if mean else p["a0"])
            keep = (r * r).sum(0) < (S + torch.clamp(torch.as_tensor(dl, dtype=F64, device=a.device), min=self.range)) ** 2
            i, j = i[keep], j[keep]
            key, order = torch.sort(i * n + j)
            i, j = i[order], j[order]
        k = inst[i]
        r, sy = _separation(x, self.L, off, i, j, inst)
        A, B = a[i], a[j]
        S = A + B
        rr = torch.sqrt((r * r).sum(0))
        nn = r / rr
        d = rr - S
        gd, zero = self.gdot[k], torch.zeros_like(d)
        yj = x[1, j] + sy * self.L[k]
        Ui, ri = self.flow(x[1, i], k)
        Uj, rj = self.flow(yj, k)
        uj = torch.stack([u[0, j] + sy * gd * self.L[k], u[1, j], u[2, j]])
        wi, wj = w[:, i], w[:, j]
        Vi = torch.stack([u[0, i] - Ui, u[1, i], u[2, i]])
        Vj = torch.stack([uj[0] - Uj, uj[1], uj[2]])
        Wi = torch.stack([wi[0], wi[1], wi[2] + 0.5 * ri])
        Wj = torch.stack([wj[0], wj[1], wj[2] + 0.5 * rj])

        def tang(v):
            return v - _dot(nn, v) * nn

        # contact and its springs
        touch = d.detach() < 0.0
        c = touch.to(F64)
        xo, ro = torch.zeros_like(r), torch.zeros_like(r)
        if hist is not None and hist[0].numel():
            q = torch.searchsorted(hist[0], key).clamp_(max=hist[0].numel() - 1)
            hit = hist[0][q] == key
            xo = torch.where(hit, hist[1][:, q], 0.0)
            ro = torch.where(hit, hist[2][:, q], 0.0)
        du = uj - u[:, i]
        fn = th["kn"] * d + th["gn"] / gd * _dot(nn, du)
        xs = tang(xo) + p["dt"] * tang(du - _cross(A * wi + B * wj, nn))
        cap = th["mu"] * torch.abs(fn) / th["kt"]
        xm2 = _dot(xs, xs)
        slip = (torch.sqrt(xm2.detach()) > cap.detach()) & touch
        xs = xs * torch.where(slip, cap / torch.sqrt(torch.where(slip, xm2, 1.0)), 1.0)
        Ft = th["kt"] * xs
        Fc = c * (fn * nn + Ft)
        Tr, xr = zero, torch.zeros_like(xs)
        if p["k_r"] > 0.0:
            ab = 2.0 * A * B / S
            xr = tang(ro) + p["dt"] * ab * _cross(nn, wi - wj)
            capr, xrm2 = th["mu"] * torch.abs(fn) / p["k_r"], _dot(xr, xr)
            slip = (torch.sqrt(xrm2.detach()) > capr.detach()) & touch
            xr = xr * torch.where(slip, capr / torch.sqrt(torch.where(slip, xrm2, 1.0)), 1.0)
            Tr = c * ab * _cross(nn, p["k_r"] * xr)
        nf = c * _cross(nn, Ft)
        # electro-chemical forces
        if self.range > 0.0:
            ab = 2.0 * A * B / S
            m = zero
            if p["f_er"] > 0.0:
                m = m - torch.where(d < 20.0 * p["lambda_d"], p["f_er"] * ab / p["a0"]
                                    * torch.exp(-d.clamp(min=0.0) / p["lambda_d"]), zero)
            if p["hamaker"] > 0.0:
                m = m + torch.where(d < 4.0 * p["a0"], p["hamaker"] * ab / (12.0 * (d.clamp(min=0.0) ** 2 + (p["vdw_eps"] * ab) ** 2)), zero)
            Fc = Fc + m * nn
        # lubrication
        dl = th["delta"] * (0.5 * S if mean else p["a0"])
        on = (d.detach() < dl.detach()).to(F64)
        gap = torch.where(d.detach() < 0.0, zero, 2.0 * d / S) + p["lub_eps"]
        X, Y = on / gap, -on * torch.log(gap)
        AB = A * B
        xa = X * 2.0 * AB ** 2 / S ** 3
        ya = Y * (4.0 / 15.0) * AB * (2.0 * A * A + AB + 2.0 * B * B) / S ** 3
        ybi = -Y * (2.0 / 15.0) * A * AB * (4.0 * A + B) / S ** 2
        ybj = -Y * (2.0 / 15.0) * AB * B * (A + 4.0 * B) / S ** 2
        yci, ycj, ycx = (Y * f * AB / S for f in ((8.0 / 15.0) * A * A, (8.0 / 15.0) * B * B, (2.0 / 15.0) * AB))
        xg = X * 2.0 * AB ** 2 / S ** 2
        yg = Y * AB * (4.0 - 6.0 * AB / S ** 2) / 15.0
        yhi = Y * (2.0 * A * A * AB * (2.0 * A - B) + AB ** 2 * (7.0 * A + B)) / (15.0 * S ** 2)
        yhj = Y * (AB ** 2 * (A + 7.0 * B) + 2.0 * AB * B * B * (2.0 * B - A)) / (15.0 * S ** 2)
        dV, rate = Vi - Vj, 0.5 * (ri + rj)
        En = torch.stack([rate * nn[1], rate * nn[0], zero])
        P, np_ = rate * nn[0] * nn[1], _cross(nn, En)
        k6 = 6.0 * math.pi * p["eta0"]
        Fl = k6 * (xg * P * nn + yg * (En - 2.0 * P * nn) - xa * _dot(nn, dV) * nn - ya * tang(dV)
                   - ybi * _cross(nn, Wi) - ybj * _cross(nn, Wj))
        nV = _cross(nn, dV)
        Tli = k6 * (ybi * nV - yci * tang(Wi) - ycx * tang(Wj) + yhi * np_)
        Tlj = k6 * (ybj * nV - ycx * tang(Wi) - ycj * tang(Wj) + yhj * np_)
        if p["lub_taper"] > 0.0:
            t = ((dl - d) / (p["lub_taper"] * dl)).clamp(0.0, 1.0)
            s = t * t * (3.0 - 2.0 * t)
            Fl, Tli, Tlj = s * Fl, s * Tli, s * Tlj
        F = torch.zeros_like(x).index_add(1, i, Fc + Fl).index_add(1, j, -(Fc + Fl))
        T = torch.zeros_like(x).index_add(1, i, A * nf + Tr + Tli).index_add(1, j, B * nf - Tr + Tlj)
        # drag
        Ux, rx = self.flow(x[1], inst)
        fax = p["wave_amp"] * (a * self.wk[inst]) ** 2 / 6.0 * torch.sin(self.wk[inst] * x[1])
        k8 = 8.0 * math.pi * p["eta0"]
        F = F - k6 * a * torch.stack([u[0] - Ux + fax, u[1], u[2]])
        T = T - k8 * a ** 3 * torch.stack([w[0], w[1], w[2] + 0.5 * rx])
        # stress
        K = self.L.numel()
        S9 = (r[:, None] * Fc[None] + 0.5 * (r[:, None] * Fl[None] + Fl[:, None] * r[None])).reshape(9, -1)
        S9 = torch.zeros((9, K), dtype=F64, device=x.device).index_add(1, k, S9)
        ein = torch.zeros(K, dtype=F64, device=x.device).index_add(
            0, inst, (10.0 / 3.0) * math.pi * p["eta0"] * a ** 3 * rx)
        e = torch.zeros((9, 1), dtype=F64, device=x.device)
        e[1] = e[3] = 1.0
        sigma = (p["eta0"] * self.gdot * e + (ein * e + S9) / self.L ** 3).T
        t = touch.nonzero().squeeze(1)
        return F, T, sigma, (key[t], xs[:, t], xr[:, t])

    def start(self, x, u=None, w=None):
        if u is None:
            U, rate = self.flow(x[1], self.inst)
            z = torch.zeros_like(U)
            u, w = torch.stack([U, z, z]), torch.stack([z, z, -0.5 * rate])
        F, T, _, _ = self.forces(x, u, w, None, 0)
        return [x, u, w, F / self.m, T / self.I, None]

    def step(self, s, k):
        """The k-th step (1, 2, ...) and its stress."""
        x, u, w, al, aw, hist = s
        dt, L, inst = self.p["dt"], self.L[self.inst], self.inst
        x = x + dt * u + 0.5 * dt * dt * al
        u, w = u + 0.5 * dt * al, w + 0.5 * dt * aw
        v = x.detach()
        cr = torch.where(v[1] >= L, -1.0, torch.where(v[1] < 0.0, 1.0, 0.0)).to(F64)
        xx = x[0] + cr * self.offset(k)[inst]
        x = torch.stack([xx - L * torch.floor((xx / L).detach()), x[1] + cr * L,
                         x[2] - L * torch.floor((x[2] / L).detach())])
        u = torch.stack([u[0] + cr * self.gdot[inst] * L, u[1], u[2]])
        F, T, sigma, hist = self.forces(x, u, w, hist, k)
        al, aw = F / self.m, T / self.I
        return [x, u + 0.5 * dt * al, w + 0.5 * dt * aw, al, aw, hist], sigma


def _shaped(case, out):
    """As run() lays them out: the adjoint's results and sigma are host arrays."""
    sigma = out["sigma"].cpu()
    if case["kind"] == "io":
        return {k: v.cpu() for k, v in dict(out, sigma=sigma.reshape(9)).items()}
    return dict(out, sigma=sigma.reshape(3, 3) if case["instances"] == 1 else sigma.reshape(-1, 3, 3))


def exact(case, seed):
    g = _inputs(case, seed)
    m = _Plain(case, g)
    x = g["x"]
    if case["kind"] == "adjoint":
        W = torch.from_numpy(_mean_viscosity(case["steps"])).to(x.device)
        U, rate = m.flow(x[1], m.inst)
        z = torch.zeros_like(U)
        v = [t.detach().requires_grad_() for t in (x, torch.stack([U, z, z]), torch.stack([z, z, -0.5 * rate]))]
        th = {k: t.requires_grad_() for k, t in m.th.items()}
        s = m.start(*v)
        J = torch.zeros((), dtype=F64, device=x.device)
        for k in range(case["steps"]):
            s, sigma = m.step(s, k + 1)
            J = J + (W[k] * sigma[0]).sum()
        wrt = v + [th[k] for k in ("kn", "kt", "gn", "mu", "delta")]
        gr = [torch.zeros_like(t) if q is None else q for q, t in zip(
            torch.autograd.grad(J, wrt, allow_unused=True), wrt)]
        out = dict(zip(("x0", "u0", "w0"), [t.cpu().numpy() for t in gr[:3]]))
        # the initial accelerations come from the initial forces: what depends
        # on them is in x0, u0, w0, and they have no gradient of their own
        none = np.zeros_like(out["x0"])
        return dict(out, alpha0=none, beta0=none, J=np.asarray(J.item()), params=np.array([float(t) for t in gr[3:]]))
    with torch.no_grad():
        if case["kind"] == "forces":
            U, rate = m.flow(x[1], m.inst)
            z = torch.zeros_like(U)
            F, T, _, _ = m.forces(x, torch.stack([U, z, z]), torch.stack([z, z, -0.5 * rate]), None, 0)
            return dict(F=F, T=T)
        s = m.start(x)
        for k in range(case["steps"]):
            s, sigma = m.step(s, k + 1)
        return _shaped(case, dict(zip(("x", "u", "w", "al", "aw"), s), sigma=sigma))


def _mean_viscosity(steps):
    """sigma_xy averaged over the steps, over eta0 gdot = 1."""
    W = np.zeros((steps, 9))
    W[:, 1] = 1.0 / steps
    return W
