"""Performance cases: the calls a user of this framework makes, over the range of sizes they are made at.

Grids are the seeded synthetic ones of `gridgen` (inputs only, no power-flow
arithmetic); their sizes are the workloads of the tests and of the benchmark.
Every value below the grid (loads, states, outage order) comes from the seed.
"""
import functools
import math

import numpy as np
import torch

import gridgen
import paper_2603_28203_gb300 as dpf
from paper_2603_28203_gb300 import presets
from paper_2603_28203_gb300.autograd import dpf_loss
from paper_2603_28203_gb300.paramid import identify_branches
from paper_2603_28203_gb300.timeseries import TABLE3_T1

PREC = {"fp32": dpf.FP32, "fp64": dpf.FP64, "fp32r": dpf.FP32R}


def listed():
    return [
        # one operating point of a small grid evaluated: the smallest call, as an application's inner loop makes it
        dict(name="power_30x1_fp64", kind="power", n_bus=30, n_case=1, precision="fp64", outages=False),
        # what-if screening: the flows of every N-1 outage of the 2,000-bus grid at one state per case
        dict(name="power_2000x2379_fp32_n1", kind="power", n_bus=2000, n_case=2379, precision="fp32", outages=True),
        # the differentiable loss inside a PyTorch program (forward and backward, branch gradients with it)
        dict(name="autograd_118x24_fp64", kind="autograd", n_bus=118, n_case=24, precision="fp64"),
        # loss and voltage gradients of many states of the 10,000-bus grid
        dict(name="adjoint_10000x101_fp32", kind="adjoint", n_bus=10000, n_case=101, precision="fp32"),
        # Alg. 1 on one small grid in the oracle-faithful precision: latency of an iteration (a budget before the
        # last bits of the state decide the schedule, which at 1,000 iterations they do)
        dict(name="solve_30x1_fp64", kind="solve", n_bus=30, n_case=1, precision="fp64", start="flat", outages=False,
             specs=False, iters=250),
        # Alg. 1 on thousands of load variants of the 30-bus grid (Table 2)
        dict(name="solve_30x8192_fp32r", kind="solve", n_bus=30, n_case=8192, precision="fp32r", start="flat",
             outages=False, specs=True, iters=250),
        # the headline batch: every N-1 outage of the 2,000-bus grid from the base case's solution
        dict(name="solve_2000x2379_fp32r_n1", kind="solve", n_bus=2000, n_case=2379, precision="fp32r", start="base",
             outages=True, specs=False, iters=400),
        # one later window of the hourly series of the 10,000-bus grid (Table 3)
        dict(name="solve_10000x96_fp32_series", kind="solve", n_bus=10000, n_case=96, precision="fp32", start="dc",
             outages=False, specs=True, iters=300),
        # one large grid: node scaling
        dict(name="solve_100000x1_fp32", kind="solve", n_bus=100000, n_case=1, precision="fp32", start="flat",
             outages=False, specs=False, iters=300),
        # Newton-Raphson on every N-1 outage of the 2,000-bus grid
        dict(name="newton_2000x2379_fp32_n1", kind="newton", n_bus=2000, n_case=2379, precision="fp32", outages=True),
        # the DC approximation of the same batch
        dict(name="dc_2000x2379_n1", kind="dc", n_bus=2000, n_case=2379, tol=1e-10, outages=True),
        # branch parameters identified from 16 measured points of a batch of uneven grids
        dict(name="identify_16grids_x16_fp32", kind="identify", n_grid=16, n_case=16, precision="fp32", iters=20),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["power", "autograd", "adjoint", "solve", "solve", "solve", "newton", "dc", "identify"])
    if kind == "power" or kind == "adjoint":
        n = _log(rng, 30, 30000)
        k = _log(rng, 1, max(1, min(4000, 2_000_000 // n)))
        c = dict(kind=kind, n_bus=n, n_case=k, precision=rng.choice(["fp32", "fp32", "fp64"]))
        if kind == "power":
            c["outages"] = n <= 10000 and rng.random() < 0.5
        return c
    if kind == "autograd":
        n = _log(rng, 30, 3000)
        return dict(kind=kind, n_bus=n, n_case=_log(rng, 1, min(500, 300_000 // n)), precision=rng.choice(["fp32", "fp64"]))
    if kind == "solve":
        start = rng.choice(["flat", "base", "dc"])
        n = _log(rng, 30, {"flat": 60000, "base": 2000, "dc": 10000}[start])
        p = rng.choice(["fp32", "fp32r", "fp32r", "fp64"])
        k = _log(rng, 1, max(1, min(8000, (3_000_000 if p != "fp64" else 300_000) // n)))
        outages = start == "base" or (n <= 10000 and rng.random() < 0.3)
        return dict(kind=kind, n_bus=n, n_case=k, precision=p, start=start, outages=outages,
                    specs=start == "dc" or rng.random() < 0.5, iters=rng.randrange(100, 250))
    if kind == "newton":
        n = _log(rng, 30, 2500)
        return dict(kind=kind, n_bus=n, n_case=_log(rng, 1, max(1, min(3000, 2_000_000 // n))),
                    precision=rng.choice(["fp32", "fp64"]), outages=rng.random() < 0.7)
    if kind == "dc":
        n = _log(rng, 30, 4000)
        return dict(kind=kind, n_bus=n, n_case=_log(rng, 1, max(1, min(3000, 2_000_000 // n))), tol=1e-10,
                    outages=rng.random() < 0.7)
    return dict(kind=kind, n_grid=rng.randrange(2, 17), n_case=rng.randrange(2, 33), precision=rng.choice(["fp32", "fp64"]),
                iters=rng.randrange(5, 30))


# ---- inputs -----------------------------------------------------------------
@functools.lru_cache(maxsize=4)
def _grid_of(n_bus, n_grid):
    if n_grid:  # a block-diagonal batch of uneven grids
        sizes = gridgen.uneven_sizes(n_grid, 200, lo=300, hi=3000)
        return gridgen.concat_grids([gridgen.make_grid(int(n), 2000 + i, load_scale=0.1) for i, n in enumerate(sizes)])
    if n_bus == 30:
        return gridgen.config_grid("c1_30bus_fp64")
    return gridgen.make_grid(n_bus, 2, load_scale=0.1 if n_bus < 5000 else 0.05)


def _grid(case):
    return _grid_of(case.get("n_bus", 0), case.get("n_grid", 0))


@functools.lru_cache(maxsize=4)
def _secure_of(n_bus):
    return gridgen.n1_outages(_grid_of(n_bus, 0))


def _outages(case, rng):
    """Secure (non-bridge) outages in a seeded order, one per case."""
    ok = _secure_of(case["n_bus"])
    k = case["n_case"]
    return np.concatenate([rng.permutation(ok) for _ in range(-(-k // ok.size))])[:k].astype(np.int32)


def _branch_terms(g, gs=None, bs=None):
    """pi-model blocks (Y_ff, Y_ft = Y_tf, Y_tt) of every branch."""
    ys = 1.0 / (g.r + 1j * g.x) if gs is None else gs + 1j * bs
    tap = np.where(g.tap == 0, 1.0, g.tap)
    sh = 0.5j * g.b_ch
    return (ys + sh) / tap ** 2, -ys / tap, ys + sh


def _ell(n, f, t, off, diag):
    """Symmetric sparse matrix as (column, value) arrays [D][n], row i's entries down column i; pads are 0 at (i, i)."""
    rows, cols = np.concatenate([f, t]), np.concatenate([t, f])
    vals = np.concatenate([off, off])
    order = np.argsort(rows, kind="stable")
    rows, cols, vals = rows[order], cols[order], vals[order]
    start = np.searchsorted(rows, np.arange(n))
    slot = np.arange(rows.size) - start[rows]
    depth = 1 + (int(slot.max()) + 1 if rows.size else 0)
    idx = np.tile(np.arange(n), (depth, 1))
    val = np.zeros((depth, n), vals.dtype)
    val[0] = diag
    idx[1 + slot, rows], val[1 + slot, rows] = cols, vals
    return idx, val


def _ybus(g):
    ff, ft, tt = _branch_terms(g)
    diag = np.zeros(g.n_bus, complex)
    np.add.at(diag, g.f_bus, ff)
    np.add.at(diag, g.t_bus, tt)
    return _ell(g.n_bus, g.f_bus, g.t_bus, ft, diag)


def _mul(ell, x):
    idx, val = ell
    y = val[0][:, None] * x
    for d in range(1, idx.shape[0]):
        y = y + val[d][:, None] * x[idx[d]]
    return y


@functools.lru_cache(maxsize=4)
def _dc_angles(n_bus):
    """DC angles of the grid's own injections (conjugate gradients): a user's rough state of a large grid."""
    g = _grid_of(n_bus, 0)
    b = 1.0 / (g.x * np.where(g.tap == 0, 1.0, g.tap))
    diag = np.zeros(g.n_bus)
    np.add.at(diag, g.f_bus, b)
    np.add.at(diag, g.t_bus, b)
    ell = _ell(g.n_bus, g.f_bus, g.t_bus, -b, diag)
    free = (g.bus_type != gridgen.SLACK)[:, None]
    x = np.zeros((g.n_bus, 1))
    r = np.where(free, g.p_spec[:, None], 0.0)
    z = r / diag[:, None]
    p, rz, stop = z.copy(), float((r * z).sum()), 1e-10 * np.linalg.norm(r)
    for _ in range(4000):
        q = np.where(free, _mul(ell, p), 0.0)
        a = rz / float((p * q).sum())
        x, r = x + a * p, r - a * q
        if np.linalg.norm(r) <= stop:
            break
        z = r / diag[:, None]
        rz, old = float((r * z).sum()), rz
        p = z + (rz / old) * p
    return x[:, 0]


@functools.lru_cache(maxsize=4)
def _base_case(n_bus):
    """The solved grid without outage (dense Newton-Raphson): the start of its N-1 cases."""
    g = _grid_of(n_bus, 0)
    n = g.n_bus
    idx, val = _ybus(g)
    Y = np.zeros((n, n), complex)
    for d in range(idx.shape[0]):
        np.add.at(Y, (np.arange(n), idx[d]), val[d])
    va, vm = np.zeros(n), np.where(g.bus_type == gridgen.PQ, 1.0, g.vm_set)
    th, mg = np.flatnonzero(g.bus_type != gridgen.SLACK), np.flatnonzero(g.bus_type == gridgen.PQ)
    for _ in range(12):
        V = vm * np.exp(1j * va)
        I = Y @ V
        S = V * np.conj(I)
        f = np.concatenate([S.real[th] - g.p_spec[th], S.imag[mg] - g.q_spec[mg]])
        if np.abs(f).max() < 1e-10:
            break
        dth = 1j * V[:, None] * np.conj(np.diag(I) - Y * V[None, :])
        u = V / vm
        dvm = V[:, None] * np.conj(Y * u[None, :]) + np.diag(np.conj(I) * u)
        J = np.block([[dth.real[np.ix_(th, th)], dvm.real[np.ix_(th, mg)]],
                      [dth.imag[np.ix_(mg, th)], dvm.imag[np.ix_(mg, mg)]]])
        dx = np.linalg.solve(J, -f)
        va[th] += dx[: th.size]
        vm[mg] += dx[th.size:]
    else:  # no solution found: the flat state
        va, vm = np.zeros(n), np.where(g.bus_type == gridgen.PQ, 1.0, g.vm_set)
    return va, vm


def _inputs(case, seed):
    """The seeded values of a case, as numpy arrays in user bus order."""
    g = _grid(case)
    rng = np.random.default_rng([seed, 28203])
    k, n, d = case["n_case"], g.n_bus, {}
    kind = case["kind"]
    if case.get("outages"):
        d["outage"] = _outages(case, rng)
    if kind in ("power", "autograd", "adjoint", "identify"):  # operating points: angles of a loaded grid, |V| near 1
        swing = rng.uniform(-1, 1, (k, 3))
        d["va"] = 0.2 * (swing[:, :1] * g.pos[:, 0] + swing[:, 1:2] * g.pos[:, 1]) + 0.02 * rng.standard_normal((k, n))
        d["vm"] = 1.0 + 0.02 * rng.standard_normal((k, n))
    if kind in ("autograd", "newton", "dc") or case.get("specs"):
        if case.get("start") == "dc":  # consecutive hours of the load model
            d["p"], d["q"] = gridgen.time_series(g, k, seed % 100003, t0=seed % 8000)
        else:                          # load variants
            level = 1 + 0.05 * rng.uniform(-1, 1, (k, 1))
            d["p"], d["q"] = g.p_spec * level, g.q_spec * level
    if kind in ("autograd", "identify"):
        ys = 1.0 / (g.r * rng.uniform(0.9, 1.1, g.n_branch) + 1j * g.x * rng.uniform(0.9, 1.1, g.n_branch))
        d["g"], d["b"] = ys.real.copy(), ys.imag.copy()
    if kind == "identify":  # the injections measured at those points on the true grid
        V = (d["vm"] * np.exp(1j * d["va"])).T
        S = V * np.conj(_mul(_ybus(g), V))
        d["p"], d["q"] = np.ascontiguousarray(S.real.T), np.ascontiguousarray(S.imag.T)
    if kind == "solve" and case["start"] == "base":  # one estimated state shared by every case
        va, vm = _base_case(n)
        d["va_start"] = va + 1e-3 * rng.standard_normal(n)
        d["vm_start"] = vm + 1e-3 * rng.standard_normal(n)
    if kind == "solve" and case["start"] == "dc":  # a state per case
        d["va"] = _dc_angles(n) * rng.uniform(0.8, 1.2, (k, 1))
        d["vm"] = np.where(g.bus_type == gridgen.PQ, 0.99, g.vm_set) + 2e-3 * rng.standard_normal((k, n))
    if kind == "solve" and case["start"] == "flat" and not case["specs"]:
        d["vm_set"] = np.tile(g.vm_set, (k, 1)) * rng.uniform(0.99, 1.01, (k, 1))
    return d


def _settings(case):
    if case["start"] == "base":
        return dict(presets.N1_WARM, **presets.N1_TEST, flat_start=0)
    if case["start"] == "dc":
        return dict({k: v for k, v in TABLE3_T1.items() if k != "max_iter"}, check_every=25, flat_start=0)
    return dict(presets.TABLE2, lr=1e-2 if case["n_bus"] < 100 else 1e-3, check_every=25, flat_start=1)


def prepare(case, seed):
    g = _grid(case)
    d = {k: torch.tensor(np.ascontiguousarray(v), device="cuda") for k, v in _inputs(case, seed).items()}
    k, n, kind = case["n_case"], g.n_bus, case["kind"]
    y = dpf.dpf_build_ybus(g)
    s = dict(case=case, y=y, **d)
    if kind == "newton":
        s["nr"] = dpf.dpf_nr_create(y, k)
    else:
        s["ws"] = dpf.dpf_workspace_create(y, k)
    if kind in ("solve", "newton"):
        new = functools.partial(torch.empty, device="cuda")
        s["out"] = dict(va=new(k, n, dtype=torch.float64), vm=new(k, n, dtype=torch.float64),
                        iters=new(k, dtype=torch.int32), status=new(k, dtype=torch.int32))
        if kind == "solve":
            s["out"].update(max_mismatch=new(k, dtype=torch.float64), loss=new(k, dtype=torch.float64))
            s["opts"] = dpf.SolveOpts(precision=PREC[case["precision"]], max_iter=case["iters"], **_settings(case))
    return s


def run(s):
    case, y = s["case"], s["y"]
    kind, prec = case["kind"], PREC.get(case.get("precision"))
    if kind == "power":
        return dpf.dpf_power(y, s["ws"], s["va"], s["vm"], outage=s.get("outage"), precision=prec)
    if kind == "adjoint":
        return dpf.dpf_loss_backward(y, s["ws"], s["va"], s["vm"], precision=prec)
    if kind == "autograd":
        x = [s[k].detach().requires_grad_() for k in ("va", "vm", "p", "q", "g", "b")]
        loss = dpf_loss(x[0], x[1], y, s["ws"], x[2], x[3], x[4], x[5], precision=prec)
        return loss.detach(), torch.autograd.grad(loss, x)
    if kind == "identify":
        g, b, _ = identify_branches(y, s["ws"], s["va"], s["vm"], s["p"], s["q"], s["g"], s["b"], case["iters"],
                                    precision=prec)
        return g, b
    if kind == "dc":
        return dpf.dpf_dc_solve(y, s["ws"], case["n_case"], p_spec=s["p"], outage=s.get("outage"), tol=case["tol"])["va"]
    if kind == "newton":
        dpf.dpf_nr_solve(s["nr"], precision=prec, tol=1e-10, max_iter=10, n_case=case["n_case"], p_spec=s["p"],
                         q_spec=s["q"], outage=s.get("outage"), **s["out"])
        return s["out"]
    if case["start"] == "dc":  # (the solve overwrites its start)
        s["out"]["va"].copy_(s["va"])
        s["out"]["vm"].copy_(s["vm"])
    dpf.dpf_solve_batch(y, s["ws"], s["opts"], n_case=case["n_case"], p_spec=s.get("p"), q_spec=s.get("q"),
                        vm_set=s.get("vm_set"), outage=s.get("outage"), va_start=s.get("va_start"),
                        vm_start=s.get("vm_start"), **s["out"])
    return s["out"]


def work(case):
    g = _grid(case)
    n, m, k = g.n_bus, g.n_branch, case["n_case"]
    z = n + 2 * m  # nonzeros of Y_bus
    e, kind = n * k, case["kind"]
    fwd, adj = (8 * z + 30 * n) * k, (8 * z + 60 * n) * k  # flops of one pass over the batch
    grid = 20 * z + 16 * n
    if kind == "power":
        return dict(bytes=32 * e + grid, flops=fwd)
    if kind == "adjoint":
        return dict(bytes=32 * e + grid, flops=fwd + adj)
    if kind == "autograd":
        return dict(bytes=64 * e + 32 * m + grid, flops=fwd + adj + 40 * m * k)
    if kind == "identify":
        return dict(bytes=32 * e + 48 * m + grid, flops=case["iters"] * (fwd + 40 * m * k))
    if kind == "dc":  # sparse direct: a few operations per nonzero
        return dict(bytes=16 * e + grid, flops=20 * z * k)
    if kind == "newton":  # about five steps: mismatch, Jacobian, sparse factor
        return dict(bytes=32 * e + grid, flops=5 * (fwd + 60 * z * k))
    per = (16 if case["specs"] else 0) + (16 if case["start"] == "dc" else 0) + 16
    return dict(bytes=per * e + grid, flops=case["iters"] * (fwd + adj))


# ---- the same results in 64 bits --------------------------------------------
class _Grid64:
    """The equations on [N][K] complex128 tensors (case-minor), N-1 outages as per-case corrections."""

    def __init__(self, g, outage=None, gs=None, bs=None):
        t = lambda a: torch.as_tensor(np.ascontiguousarray(a), device="cuda")  # noqa: E731
        self.terms = [t(a) for a in _branch_terms(g, gs, bs)]
        ff, ft, tt = (a.cpu().numpy() for a in self.terms)
        diag = np.zeros(g.n_bus, complex)
        np.add.at(diag, g.f_bus, ff)
        np.add.at(diag, g.t_bus, tt)
        idx, val = _ell(g.n_bus, g.f_bus, g.t_bus, ft, diag)
        self.idx, self.val = t(idx), t(val)
        self.f, self.t = t(g.f_bus.astype(np.int64)), t(g.t_bus.astype(np.int64))
        ty = t(g.bus_type)[:, None]
        self.act, self.rea = (ty != gridgen.SLACK).double(), (ty == gridgen.PQ).double()
        self.m = float(self.act.sum() + self.rea.sum())
        self.out = None
        if outage is not None:
            o = t(outage.astype(np.int64))
            self.out = (self.f[o], self.t[o], *(a[o] for a in self.terms))

    def mul(self, x):
        y = self.val[0][:, None] * x
        for d in range(1, self.idx.shape[0]):
            y += self.val[d][:, None] * x[self.idx[d]]
        if self.out is not None:
            f, t, ff, ft, tt = self.out
            k = torch.arange(x.shape[1], device=x.device)
            xf, xt = x[f, k], x[t, k]
            y[f, k] -= ff * xf + ft * xt
            y[t, k] -= ft * xf + tt * xt
        return y

    def mismatch(self, V, p, q):
        I = self.mul(V)
        S = V * I.conj()
        return S, torch.complex((S.real - p) * self.act, (S.imag - q) * self.rea)

    def gradient(self, va, vm, p, q):
        V = torch.polar(torch.ones_like(va), va) * vm
        S, f = self.mismatch(V, p, q)
        c = f * (2.0 / self.m)
        w = c * V.conj()
        h = c.conj() * S + V * self.mul(w)
        loss = (f.real ** 2 + f.imag ** 2).sum(0) / self.m
        return loss, -h.imag * self.act, h.real / vm * self.rea, f, c, V, w


def _t(a):
    return torch.as_tensor(np.ascontiguousarray(a.T), device="cuda")


def _branch_grad(G, V, w, tap):
    it = torch.as_tensor(1.0 / np.where(tap == 0, 1.0, tap), device="cuda")
    wf, wt, vf, vt = w[G.f], w[G.t], V[G.f], V[G.t]
    e = (wf * vf).sum(1) * it ** 2 + (wt * vt).sum(1) - ((wf * vt).sum(1) + (wt * vf).sum(1)) * it
    return e.real, -e.imag


def exact(case, seed):
    g, d, kind = _grid(case), _inputs(case, seed), case["kind"]
    k, n = case["n_case"], g.n_bus
    p, q = (_t(d.get(x, y[None, :])) for x, y in (("p", g.p_spec), ("q", g.q_spec)))
    if kind == "power":
        G = _Grid64(g, d.get("outage"))
        S = G.mismatch(torch.polar(_t(d["vm"]), _t(d["va"])), 0.0, 0.0)[0]
        return S.real.T.contiguous(), S.imag.T.contiguous()
    if kind == "adjoint":
        L, ga, gm = _Grid64(g).gradient(_t(d["va"]), _t(d["vm"]), p, q)[:3]
        return dict(loss=L, d_va=ga.T.contiguous(), d_vm=gm.T.contiguous())
    if kind == "autograd":
        G = _Grid64(g, gs=d["g"], bs=d["b"])
        L, ga, gm, _, c, V, w = G.gradient(_t(d["va"]), _t(d["vm"]), p, q)
        return L.sum(), tuple(x.T.contiguous() for x in (ga, gm, -c.real, -c.imag)) + _branch_grad(G, V, w, g.tap)
    if kind == "identify":
        x = [torch.as_tensor(d[i], device="cuda") for i in ("g", "b")]
        scale = [a.abs() for a in x]
        mom = [[torch.zeros_like(a), torch.zeros_like(a)] for a in x]
        for t in range(1, case["iters"] + 1):
            G = _Grid64(g, gs=x[0].cpu().numpy(), bs=x[1].cpu().numpy())
            V, w = G.gradient(_t(d["va"]), _t(d["vm"]), p, q)[5:]
            for i, gr in enumerate(_branch_grad(G, V, w, g.tap)):
                mo = mom[i]
                mo[0], mo[1] = 0.9 * mo[0] + 0.1 * gr, 0.999 * mo[1] + 0.001 * gr * gr
                den = (mo[1] / (1 - 0.999 ** t)).sqrt() + 1e-8
                x[i] = x[i] - 3e-3 * scale[i] * (mo[0] / (1 - 0.9 ** t)) / den
        return tuple(x)
    if kind == "dc":
        return _exact_dc(g, p, d.get("outage"), k)
    if kind == "newton":
        return _exact_newton(g, d, p, q, k)
    return _exact_solve(case, g, d, p, q)


def _exact_dc(g, p, outage, k):
    n = g.n_bus
    b = 1.0 / (g.x * np.where(g.tap == 0, 1.0, g.tap))
    B = np.zeros((n, n))
    np.add.at(B, (g.f_bus, g.f_bus), b)
    np.add.at(B, (g.t_bus, g.t_bus), b)
    np.add.at(B, (g.f_bus, g.t_bus), -b)
    np.add.at(B, (g.t_bus, g.f_bus), -b)
    u = torch.as_tensor(np.flatnonzero(g.bus_type != gridgen.SLACK), device="cuda")
    inv = torch.zeros(n, n, dtype=torch.float64, device="cuda")
    inv[u[:, None], u] = torch.linalg.inv(torch.as_tensor(B, device="cuda")[u[:, None], u])
    x = inv @ p.expand(n, k)
    if outage is not None:  # Sherman-Morrison, the branch's susceptance taken out
        o = torch.as_tensor(outage.astype(np.int64), device="cuda")
        f, t, bl = (torch.as_tensor(a, device="cuda")[o] for a in (g.f_bus.astype(np.int64), g.t_bus.astype(np.int64), b))
        at = torch.arange(k, device="cuda")
        col = inv[:, f] - inv[:, t]
        x = x + col * (bl * (x[f, at] - x[t, at]) / (1 - bl * (col[f, at] - col[t, at])))
    return x.T.contiguous()


def _exact_newton(g, d, p, q, k):
    """Dense Newton-Raphson of every case; None where it takes too long."""
    n = g.n_bus
    th, mg = np.flatnonzero(g.bus_type != gridgen.SLACK), np.flatnonzero(g.bus_type == gridgen.PQ)
    size = th.size + mg.size
    if k * size ** 3 > 2e11 or k * n * n > 5e7:
        return None
    G = _Grid64(g, d.get("outage"))
    Y = torch.stack([G.mul(torch.eye(n, dtype=torch.complex128, device="cuda")[:, j:j + 1].expand(n, k)).T
                     for j in range(n)], 2)  # [k][n][n]
    th, mg = (torch.as_tensor(a, device="cuda") for a in (th, mg))
    va = torch.zeros(k, n, dtype=torch.float64, device="cuda")
    vm = torch.as_tensor(np.where(g.bus_type == gridgen.PQ, 1.0, g.vm_set), device="cuda").expand(k, n).clone()
    p, q = p.T.expand(k, n), q.T.expand(k, n)
    for _ in range(12):
        u = torch.polar(torch.ones_like(va), va)
        V = u * vm
        I = (Y @ V[:, :, None])[:, :, 0]
        S = V * I.conj()
        f = torch.cat([(S.real - p)[:, th], (S.imag - q)[:, mg]], 1)
        da = 1j * V[:, :, None] * (torch.diag_embed(I) - Y * V[:, None, :]).conj()
        dm = V[:, :, None] * (Y * u[:, None, :]).conj() + torch.diag_embed(I.conj() * u)
        J = torch.cat([torch.cat([da.real[:, th][:, :, th], dm.real[:, th][:, :, mg]], 2),
                       torch.cat([da.imag[:, mg][:, :, th], dm.imag[:, mg][:, :, mg]], 2)], 1)
        dx = torch.linalg.solve(J, -f)
        va[:, th] += dx[:, : th.numel()]
        vm[:, mg] += dx[:, th.numel():]
    if not bool((f.abs().max() < 1e-9)):  # a case without a solution has no exact value
        return None
    return dict(va=va, vm=vm, iters=None, status=None)


def _exact_solve(case, g, d, p, q):
    """Alg. 1 in 64 bits: Adam with the plateau schedule, every case on its own."""
    k, n = case["n_case"], g.n_bus
    depth = 1 + int(np.bincount(np.concatenate([g.f_bus, g.t_bus])).max())
    if case["iters"] * n * k * (2 * depth * 48 + 400) / 4e12 + case["iters"] * 2e-3 > 20:
        return None
    o = _settings(case)
    G = _Grid64(g, d.get("outage"))
    ty = torch.as_tensor(g.bus_type, device="cuda")[:, None]
    if case["start"] == "base":
        va, vm = (torch.as_tensor(d[x], device="cuda")[:, None].repeat(1, k) for x in ("va_start", "vm_start"))
    elif case["start"] == "dc":
        va, vm = _t(d["va"]), _t(d["vm"])
    else:
        va, vm = torch.zeros(n, k, dtype=torch.float64, device="cuda"), torch.ones(n, k, dtype=torch.float64, device="cuda")
    sets = _t(d["vm_set"]) if "vm_set" in d else torch.as_tensor(g.vm_set, device="cuda")[:, None].expand(n, k)
    vm = torch.where(ty == gridgen.PQ, vm, sets)
    va = torch.where(ty == gridgen.SLACK, torch.zeros_like(va), va)
    ma, sa, mm, sm = (torch.zeros_like(va) for _ in range(4))
    new = lambda v: torch.full((k,), float(v), dtype=torch.float64, device="cuda")  # noqa: E731
    lr, best, bad, cool, live = new(o["lr"]), new(math.inf), new(0), new(0), torch.ones(k, dtype=torch.bool, device="cuda")
    b1, b2, eps = o["beta1"], o["beta2"], o.get("eps", 1e-8)
    for t in range(1, case["iters"] + 1):
        loss, ga, gm, f = G.gradient(va, vm, p, q)[:4]
        if (t - 1) % o["check_every"] == 0:
            live &= ~(torch.maximum(f.real.abs().amax(0), f.imag.abs().amax(0)) <= 1e-6)
        ma, mm = b1 * ma + (1 - b1) * ga, b1 * mm + (1 - b1) * gm
        sa, sm = b2 * sa + (1 - b2) * ga * ga, b2 * sm + (1 - b2) * gm * gm
        step = lr / (1 - b1 ** t) * live
        root = 1 / math.sqrt(1 - b2 ** t)
        va = va - step * ma / (sa.sqrt() * root + eps)
        vm = vm - step * mm / (sm.sqrt() * root + eps)
        better = loss < best * (1 - o["threshold"])
        best = torch.where(better, loss, best)
        bad = torch.where(better, torch.zeros_like(bad), bad + 1)
        cooling = cool > 0
        cool = torch.where(cooling, cool - 1, cool)
        bad = torch.where(cooling, torch.zeros_like(bad), bad)
        drop = bad > o["patience"]
        lr = torch.where(drop & (lr * (1 - o["factor"]) > 1e-8), lr * o["factor"], lr)
        cool = torch.where(drop, torch.full_like(cool, float(o["cooldown"])), cool)
        bad = torch.where(drop, torch.zeros_like(bad), bad)
    loss, _, _, f = G.gradient(va, vm, p, q)[:4]
    worst = torch.maximum(f.real.abs().amax(0), f.imag.abs().amax(0))
    return dict(va=va.T.contiguous(), vm=vm.T.contiguous(), iters=None, status=None, max_mismatch=worst, loss=loss)
