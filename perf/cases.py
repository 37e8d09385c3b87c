"""Workloads of the AAHRT operator pair and its solvers, for timing.

Every case is one pass through the public Python entry points (AahrtPlan and
the autograd wrappers): single operator applications (the layers of an
inversion), forward + adjoint pairs, the operator as a differentiable layer,
the stack of residual moveout, and whole sparse solves.  Sizes are those
of the generators in paper_2505_00387_gb300/synthetic.py (the 16 x 16 grid
cube, the paper-scale gather, the uneven-fold cube batch, the shared
geometry), of the benchmark, or odd ones in between.

A case's fields: `op` (forward, adjoint, pair, grad, solve, residual), `plan`
(single, batched, slowness, shared), the axes `nt`, `dt`, `nq`, `ntheta`, the
fold `ntr` (for batched plans folds are uniform in [lo, ntr]), `radius` (m, of
the disc the offsets fill), `ncube` / `ngather`, `interp`, and `iters`.
"""
import math

import numpy as np
import torch

from paper_2505_00387_gb300 import autograd
from paper_2505_00387_gb300.plan import AahrtPlan

P_MIN, P_MAX = 1.0 / 3500.0, 1.0 / 1500.0      # slowness range, s/m


def _case(name, op, plan="single", nt=1001, dt=0.004, nq=100, ntheta=36, ntr=2000,
          radius=3000.0, ncube=1, lo=200, interp="keys", iters=0):
    c = dict(op=op, plan=plan, nt=nt, dt=dt, nq=nq, ntheta=ntheta, ntr=ntr, radius=radius,
             ncube=ncube, lo=lo, interp=interp, iters=iters)
    return dict(c, name=name) if name else c


def listed():
    cube = dict(nt=256, nq=32, ntheta=8, ntr=256, radius=1000.0)
    batch = dict(plan="batched", nq=64, ntheta=24, ntr=3000)
    return [
        # one small cube modelled: the shortest call, bound by launches
        _case("cube_forward", "forward", **cube),
        # interactive sparse transform of one small cube
        _case("cube_solve", "solve", iters=20, **cube),
        # demigration / velocity stack of one paper-scale gather
        _case("gather_forward", "forward"),
        _case("gather_adjoint", "adjoint"),
        # velocity analysis: partial NMO, then the stack on the residual curvatures
        _case("gather_residual", "residual"),
        # the operator as a differentiable layer on a survey's odd sizes
        _case("gather_grad", "grad", nt=757, nq=61, ntheta=19, ntr=1237, interp="linear"),
        # the same gather on a uniform-slowness (non-uniform curvature) axis
        _case("slowness_pair", "pair", plan="slowness"),
        # one long record of the 8000-trace geometry (8192-sample frames)
        _case("long_pair", "pair", nt=2048, dt=0.002, nq=200, ntheta=72, ntr=8000,
              radius=4000.0),
        # cubes of uneven fold in one plan: modelling and stack of a survey line
        _case("batch_forward", "forward", ncube=32, **batch),
        _case("batch_adjoint", "adjoint", ncube=32, **batch),
        # production solve of a batch, every cube with its own step and threshold
        _case("batch_solve", "solve", ncube=16, iters=10, **batch),
        # gathers sharing one geometry on the tensor cores
        _case("shared_pair", "pair", plan="shared", nt=256, dt=0.016, nq=200, ntheta=72,
              ntr=8000, radius=4000.0, ncube=64),
    ]


def _log_int(rng, a, b):
    return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))


def draw(rng):
    plan = rng.choice(["single", "single", "single", "batched", "batched", "slowness", "shared"])
    op = rng.choice(["forward", "adjoint", "pair", "grad", "solve", "residual"])
    nt = _log_int(rng, 100, 1600)
    c = dict(nt=nt, dt=4.1 / nt, nq=_log_int(rng, 16, 200), ntheta=rng.randint(4, 72),
             ntr=_log_int(rng, 60, 6000), radius=rng.uniform(800.0, 3500.0),
             interp=rng.choice(["keys", "keys", "keys", "linear"]))
    if plan == "batched":
        c.update(ncube=rng.randint(2, 16), ntr=_log_int(rng, 250, 3000), nq=_log_int(rng, 16, 100),
                 ntheta=rng.randint(4, 36))
    elif plan == "shared":
        op = rng.choice(["forward", "adjoint", "pair"])
        c.update(ncube=rng.randint(5, 64), nt=min(nt, 300), ntr=_log_int(rng, 60, 3000))
        c["dt"] = 4.1 / c["nt"]
    if op == "solve":
        c["iters"] = rng.randint(3, 12)
    elif op == "residual" and plan == "slowness":
        op = "adjoint"
    return _case(None, op, plan=plan, **c)


# ---------------------------------------------------------------- geometry
def _offsets(case, seed):
    """Per cube (or the one geometry): (hx, hy) uniform in the disc, batched
    cubes with their own fold and a random azimuth sector."""
    rng = np.random.default_rng([seed, 11])
    folds = np.random.default_rng([case["ntr"], case["ncube"]])     # the same for every seed
    out = []
    for _ in range(case["ncube"] if case["plan"] == "batched" else 1):
        n, start, width = case["ntr"], 0.0, 2.0 * np.pi
        if case["plan"] == "batched":
            n = int(folds.integers(min(case["lo"], n), n + 1))
            start, width = rng.uniform(0.0, 2.0 * np.pi), np.deg2rad(rng.uniform(90.0, 360.0))
        r = case["radius"] * np.sqrt(rng.random(n))
        az = start + width * rng.random(n)
        out.append((r * np.cos(az), r * np.sin(az)))
    return out


def _q_axis(case):
    n = case["nq"]
    if case["plan"] == "slowness":
        return np.linspace(P_MIN, P_MAX, n) ** 2
    q = P_MIN ** 2 + (P_MAX ** 2 - P_MIN ** 2) / max(1, n - 1) * np.arange(n)
    return q - _q_ref(case)


def _q_ref(case):
    """Curvature removed by the partial NMO: the middle of the range."""
    return 0.5 * (P_MIN ** 2 + P_MAX ** 2) if case["op"] == "residual" else 0.0


class _Geometry:
    """What AahrtPlan.batched reads of a gather."""

    def __init__(self, case, hx, hy):
        q = _q_axis(case)
        self.nt = self.ntau = case["nt"]
        self.dt, self.nq, self.ntheta = case["dt"], case["nq"], case["ntheta"]
        self.q0, self.dq = float(q[0]), float(q[1] - q[0])
        self.hx, self.hy = hx, hy

    def kwargs(self):
        return dict(self.__dict__)


# ------------------------------------------------------------------ inputs
def _ricker(t, f):
    a = (math.pi * f * t) ** 2
    return (1.0 - 2.0 * a) * torch.exp(-a)


def _events(case, seed, tag):
    rng = np.random.default_rng([seed, tag])
    tmax = (case["nt"] - 1) * case["dt"]
    fny = 0.5 / case["dt"]
    for _ in range(30):
        yield (rng.uniform(0.05, 0.95) * tmax, rng.uniform(1600.0, 3300.0), rng.uniform(0.0, 0.2),
               rng.uniform(0.0, math.pi), min(rng.uniform(15.0, 40.0), 0.4 * fny),
               rng.uniform(0.5, 1.0) * (1.0 if rng.random() < 0.8 else -1.0))


def _curvature(th, v, an, axis):
    return torch.cos(th - axis) ** 2 / v ** 2 + torch.sin(th - axis) ** 2 / (v * (1 + an)) ** 2


def _data(case, seed, tag, hx, hy, dev):
    """A CMP gather [nt][trace]: Ricker events on elliptically anisotropic
    hyperbolae plus 10 % noise."""
    x, y = (torch.as_tensor(a, dtype=torch.float32, device=dev) for a in (hx, hy))
    t = torch.arange(case["nt"], device=dev, dtype=torch.float32)[:, None] * case["dt"]
    r2, az = x * x + y * y, torch.atan2(y, x)
    d = torch.zeros(case["nt"], x.numel(), device=dev)
    for tau, v, an, axis, f, amp in _events(case, seed, tag):
        d += amp * _ricker(t - torch.sqrt(tau * tau + _curvature(az, v, an, axis) * r2), f)
    return d + _noise(d, seed, tag, 0.1 * float(d.square().mean().sqrt()))


def _model(case, seed, tag, dev):
    """A Radon model [tau][q][theta] as an inversion holds it: sparse events
    on elliptical curvatures over a weak background."""
    n, q = case["ntheta"], _q_axis(case)
    th = torch.arange(n, device=dev) * (math.pi / n)
    t = torch.arange(case["nt"], device=dev, dtype=torch.float32)[:, None] * case["dt"]
    qa = torch.as_tensor(q, device=dev).contiguous()
    m = torch.zeros(case["nt"], case["nq"], n, device=dev)
    j = torch.arange(n, device=dev)
    for tau, v, an, axis, f, amp in _events(case, seed, tag):
        l = torch.searchsorted(qa, _curvature(th, v, an, axis).double()).clamp(0, case["nq"] - 1)
        m[:, l, j] += amp * _ricker(t - tau, f)
    return m + _noise(m, seed, tag, 0.02 * float(m.square().mean().sqrt()))


def _noise(like, seed, tag, level):
    g = torch.Generator(device=like.device).manual_seed(1000003 * seed + tag)
    return level * torch.randn(like.shape, device=like.device, generator=g)


def _inputs(case, seed, dev):
    """(model, data): flat float32 in the plan's layout (gathers fastest for
    the shared geometry), the ones the case does not read left None."""
    geo = _offsets(case, seed)
    need_m = case["op"] in ("forward", "pair", "grad")
    need_d = case["op"] in ("adjoint", "pair", "grad", "solve", "residual")
    tags = range(case["ncube"])
    m = [_model(case, seed, 100 + c, dev) for c in tags] if need_m else None
    d = None
    if need_d:
        d = [_data(case, seed, 5000 + c, *geo[c if len(geo) > 1 else 0], dev) for c in tags]
    if case["plan"] == "shared":
        m, d = (None if a is None else torch.stack(a, dim=-1).reshape(-1) for a in (m, d))
    else:
        m, d = (None if a is None else torch.cat([x.reshape(-1) for x in a]) for a in (m, d))
    return m, d


def _step(case, geo, weights):
    """A step length below 1 / ||L||^2 for each cube: ||L||^2 is at most about
    twice the number of curvatures times the largest azimuth weight of a slice."""
    return [0.4 / (case["nq"] * float(w.max())) for w in weights]


def _slice_weights(case, geo):
    out = []
    for hx, hy in geo:
        j0, j1, w0, w1 = _azimuth(case, hx, hy)
        out.append(np.bincount(j0, w0, case["ntheta"]) + np.bincount(j1, w1, case["ntheta"]))
    return out


def _round2(x):
    return float("%.2g" % x)


def prepare(case, seed):
    dev = torch.device("cuda")
    geo = _offsets(case, seed)
    gs = [_Geometry(case, hx, hy) for hx, hy in geo]
    if case["plan"] == "batched":
        plan = AahrtPlan.batched(gs, interp=case["interp"])
    else:
        kw = gs[0].kwargs()
        if case["plan"] == "slowness":
            kw["q_axis"] = _q_axis(case)
        elif case["plan"] == "shared":
            kw.update(ngather=case["ncube"], precision="split_bf16")
        plan = AahrtPlan(**kw, interp=case["interp"])
    m, d = _inputs(case, seed, dev)
    s = dict(op=case["op"], plan=plan, m=m, d=d, iters=case["iters"], q_ref=_q_ref(case))
    if case["op"] == "solve":
        g = plan.adjoint(d)
        n = len(geo)
        s["gamma"] = np.array(_step(case, geo, _slice_weights(case, geo)))
        s["lam"] = np.array([_round2(0.05 * float(g[c * (g.numel() // n):][:g.numel() // n]
                                                  .abs().max())) for c in range(n)])
    return s


def run(s):
    plan, op = s["plan"], s["op"]
    if op == "forward":
        return plan.forward(s["m"])
    if op == "adjoint":
        return plan.adjoint(s["d"])
    if op == "pair":
        return plan.forward(s["m"]), plan.adjoint(s["d"])
    if op == "grad":
        m = s["m"].detach().requires_grad_(True)
        d = autograd.radon(plan, m)
        d.backward(s["d"])
        return d, m.grad
    if op == "residual":
        return plan.adjoint(plan.partial_nmo(s["d"], s["q_ref"]))
    if len(s["gamma"]) == 1:
        m, _ = plan.sparse_solve(s["d"], float(s["lam"][0]), s["iters"], gamma=float(s["gamma"][0]),
                                 want_info=False)
    else:
        m, _ = plan.sparse_solve(s["d"], 0.0, s["iters"], per_cube=True,
                                 cube_gamma=s["gamma"].copy(), cube_lambda=s["lam"].copy(),
                                 want_info=False)
    return m


# -------------------------------------------------------------------- work
def work(case):
    """Bytes: model and data once per application that reads or writes them
    (per iteration of a solve: the two model-sized states read and written,
    the data read).  Flops: one real FFT per column and, per (bin, trace), the
    two azimuth slices' sums of seven kernel taps (the sum over all
    curvatures where the axis or the precision asks for it)."""
    nt, nq, nth = case["nt"], case["nq"], case["ntheta"]
    g = case["ncube"]
    ntr = case["ntr"] * g
    if case["plan"] == "batched":
        ntr = (min(case["lo"], case["ntr"]) + case["ntr"]) // 2 * g
    rho = P_MAX ** 2 * case["radius"] ** 2 / ((nt - 1) * case["dt"]) ** 2
    nfft = 1 << max(1, math.ceil(math.log2(2.0 * nt * (1.0 + rho))))
    m, d = nt * nq * nth * g, nt * ntr
    fft = 2.5 * nfft * math.log2(nfft) * (nq * nth * g + ntr)
    terms = nq if case["plan"] in ("shared", "slowness") else 7
    one = fft + (nfft // 2) * ntr * (2 * 4 * terms + 8)
    apps = {"pair": 2, "grad": 2, "solve": 2 * case["iters"]}.get(case["op"], 1)
    move = 2 * m + d / 2 if case["op"] == "solve" else m + d
    return {"bytes": 4.0 * apps * move, "flops": apps * one}


# ------------------------------------------------------------------- exact
def _azimuth(case, hx, hy):
    n = case["ntheta"]
    ph = np.mod(np.arctan2(hy, hx), np.pi) / (np.pi / n)
    j = np.floor(ph).astype(np.int64)
    f = ph - j
    f[j >= n] = 0.0
    j = np.where(j >= n, j - n, j).clip(0, n - 1)
    return j, (j + 1) % n, 1.0 - f, f


class _Operator:
    """L and its transpose for one cube in 64 bits, every sum written out:
    stretch, FFT, the DFT along q at k_q = f_k r^2 on the two neighbouring
    azimuths, band-limited synthesis, unstretch."""

    def __init__(self, case, hx, hy, r2max, dev):
        self.case, self.dev = case, dev
        nt, dt = case["nt"], case["dt"]
        q = _q_axis(case)
        tmax = (nt - 1) * dt
        rho = float(np.abs(q).max()) * r2max / (tmax * tmax)
        n = 1
        while n < math.ceil(2.0 * nt * (1.0 + rho)):
            n *= 2
        self.n, self.k = n, n // 2
        ns = int(math.floor((n - 2) / (1.0 + rho))) + 1
        ds = tmax * tmax / (ns - 1)
        self.S = self._taps(np.sqrt(np.arange(ns) * ds) / dt, nt)
        self.U = self._taps((np.arange(nt) * dt) ** 2 / ds, ns)
        self.ns = ns
        j0, _, w0, w1 = _azimuth(case, hx, hy)
        cyc = np.outer(hx * hx + hy * hy, q) / (n * ds)        # cycles per bin
        self.by_slice = []
        for j in range(case["ntheta"]):
            h = np.nonzero(j0 == j)[0]
            if h.size:
                w = torch.as_tensor(np.stack([w0[h], w1[h]], 1), device=dev)
                self.by_slice.append((j, (j + 1) % case["ntheta"], torch.as_tensor(h, device=dev), w,
                                      torch.as_tensor(cyc[h], device=dev)))
        self.ntr = hx.size

    def _taps(self, pos, n_in):
        base = np.floor(pos).astype(np.int64)
        linear = self.case["interp"] == "linear"
        idx = base[:, None] + np.arange(0 if linear else -1, 2 if linear else 3)
        x = np.abs(pos[:, None] - idx)
        if linear:
            w = np.maximum(0.0, 1.0 - x)
        else:
            w = np.where(x <= 1, 1.5 * x ** 3 - 2.5 * x ** 2 + 1,
                         np.where(x < 2, -0.5 * x ** 3 + 2.5 * x ** 2 - 4 * x + 2, 0.0))
        w = np.where((idx >= 0) & (idx < n_in), w, 0.0)
        rows = np.repeat(np.arange(pos.size), idx.shape[1])
        mat = torch.sparse_coo_tensor(np.stack([rows, idx.clip(0, n_in - 1).ravel()]), w.ravel(),
                                      (pos.size, n_in), dtype=torch.float64).coalesce()
        return mat.to(self.dev)

    def _phases(self, cyc):
        """exp(-2 pi i k cyc) for every bin: [bin][trace][q]."""
        b = 1 << ((self.k.bit_length() - 1) // 2)
        def cis(k):
            return torch.polar(torch.ones((), dtype=torch.float64, device=self.dev),
                               -2.0 * math.pi * torch.remainder(k[:, None, None] * cyc, 1.0))
        lo = cis(torch.arange(b, device=self.dev, dtype=torch.float64))
        hi = cis(b * torch.arange(self.k // b, device=self.dev, dtype=torch.float64))
        return (hi[:, None] * lo[None]).reshape(self.k, *cyc.shape)

    def _fft(self, x):              # real [n_in][col] -> bins [k][col]
        return torch.fft.rfft(x, n=self.n, dim=0)[:self.k]

    def _synth(self, X):            # Re X_0 + 2 Re sum_k X_k e^{+...}: [ns][col]
        full = torch.zeros(self.k + 1, X.shape[1], dtype=X.dtype, device=X.device)
        full[:self.k] = X
        return torch.fft.irfft(full, n=self.n, dim=0)[:self.ns] * self.n

    def forward(self, m):           # [ntau][nq][ntheta][g] -> [nt][ntr][g]
        _, nq, nth, g = m.shape
        X = self._fft(torch.sparse.mm(self.S, m.reshape(m.shape[0], -1))).reshape(self.k, nq, nth, g)
        Y = torch.zeros(self.k, self.ntr, g, dtype=X.dtype, device=X.device)
        for j, jn, h, w, cyc in self.by_slice:
            V = torch.matmul(self._phases(cyc), torch.cat([X[:, :, j], X[:, :, jn]], -1))
            Y[:, h] = V[..., :g] * w[:, :1] + V[..., g:] * w[:, 1:]
        del X
        d = torch.sparse.mm(self.U, self._synth(Y.reshape(self.k, -1) / self.n))
        return d.reshape(d.shape[0], self.ntr, g)

    def adjoint(self, d):           # [nt][ntr][g] -> [ntau][nq][ntheta][g]
        g, nq, nth = d.shape[2], self.case["nq"], self.case["ntheta"]
        Y = self._fft(torch.sparse.mm(self.U.t(), d.reshape(d.shape[0], -1)))
        Y = Y.reshape(self.k, self.ntr, g)
        X = torch.zeros(self.k, nq, nth, g, dtype=Y.dtype, device=Y.device)
        for j, jn, h, w, cyc in self.by_slice:
            y = Y[:, h]
            V = torch.matmul(self._phases(cyc).conj().transpose(1, 2),
                             torch.cat([y * w[:, :1], y * w[:, 1:]], -1))
            X[:, :, j] += V[..., :g]
            X[:, :, jn] += V[..., g:]
        del Y
        m = torch.sparse.mm(self.S.t(), self._synth(X.reshape(self.k, -1) / self.n))
        return m.reshape(m.shape[0], nq, nth, g)


def _soft(x, t):
    return torch.sign(x) * torch.clamp(x.abs() - t, min=0.0)


def _momentum(iters):
    t, out = 1.0, []
    for _ in range(iters):
        tn = 0.5 * (1.0 + math.sqrt(1.0 + 4.0 * t * t))
        out.append((t - 1.0) / tn)
        t = tn
    return out


def _iterate(op, d, gamma, lam, iters):
    """The FISTA iterate after `iters` steps from zero."""
    m = z = None
    for b in _momentum(iters):
        u = gamma * op.adjoint(d) if z is None else z + gamma * op.adjoint(d - op.forward(z))
        new = _soft(u, gamma * lam)
        z = new if m is None else new + b * (new - m)
        m = new
    return m


def _partial_nmo(case, d, hx, hy):
    """out(t_i, h) = in(sqrt(t_i^2 + q_ref r_h^2), h) by the plan's interpolation."""
    nt = case["nt"]
    c = torch.as_tensor(_q_ref(case) * (hx * hx + hy * hy) / case["dt"] ** 2, device=d.device)
    u = torch.sqrt(torch.arange(nt, device=d.device).double()[:, None] ** 2 + c)
    out = torch.zeros_like(d)
    for t in (0, 1) if case["interp"] == "linear" else (-1, 0, 1, 2):
        i = u.floor().long() + t
        x = (u - i).abs()
        if case["interp"] == "linear":
            w = 1.0 - x
        else:
            w = torch.where(x <= 1, 1.5 * x ** 3 - 2.5 * x ** 2 + 1,
                            -0.5 * x ** 3 + 2.5 * x ** 2 - 4 * x + 2)
        w = torch.where((i >= 0) & (i < nt), w, 0.0)
        out += w[..., None] * torch.gather(d, 0, i.clamp(0, nt - 1)[..., None].expand_as(d))
    return out


def exact(case, seed):
    dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
    geo = _offsets(case, seed)
    m, d = _inputs(case, seed, dev)
    nt, nq, nth, g = case["nt"], case["nq"], case["ntheta"], 1
    if case["plan"] == "shared":
        g = case["ncube"]
    r2max = max(float((hx * hx + hy * hy).max()) for hx, hy in geo)
    ops = [_Operator(case, hx, hy, r2max, dev) for hx, hy in geo]
    md = nt * nq * nth * g
    at = np.cumsum([0] + [nt * o.ntr * g for o in ops])

    def models(c):
        return m[c * md:(c + 1) * md].double().reshape(nt, nq, nth, g)

    def datas(c):
        return d[at[c]:at[c + 1]].double().reshape(nt, ops[c].ntr, g)

    def gathers(fn, x):      # a few gathers of the shared geometry at a time
        return torch.cat([fn(x[..., i:i + 8].contiguous()) for i in range(0, g, 8)], -1)

    def fwd():
        return torch.cat([gathers(o.forward, models(c)).reshape(-1) for c, o in enumerate(ops)])

    def adj():
        return torch.cat([gathers(o.adjoint, datas(c)).reshape(-1) for c, o in enumerate(ops)])

    if case["op"] == "forward":
        return fwd()
    if case["op"] == "adjoint":
        return adj()
    if case["op"] in ("pair", "grad"):
        return fwd(), adj()
    if case["op"] == "residual":
        return torch.cat([gathers(o.adjoint, _partial_nmo(case, datas(c), *geo[c])).reshape(-1)
                          for c, o in enumerate(ops)])
    out = []
    for c, (o, w) in enumerate(zip(ops, _slice_weights(case, geo))):
        gamma = _step(case, geo, [w])[0]
        lam = _round2(0.05 * float(o.adjoint(datas(c)).abs().max()))
        out.append(_iterate(o, datas(c), gamma, lam, case["iters"]).reshape(-1))
    return torch.cat(out)
