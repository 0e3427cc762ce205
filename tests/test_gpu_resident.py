"""The on-chip form of the iterations (dpf_resident.cu) against the streaming
kernels: same options, same bits.

Timing the passes one by one (dpf_profile_enable) runs the streaming kernels,
so one solve with it and one without compare the two forms.  FP32 and refined
FP32 results have to agree to the bit, the plateau schedule (fed the FP32
loss) included; the FP64 on-chip form sums the loss in another order, which
only a schedule fed by it can see, so FP64 runs a constant rate.
"""
import numpy as np
import pytest

import gridgen

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2603_28203_gb300 as dpf  # noqa: E402

DEV = torch.device("cuda:0")


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import os
    from paper_2603_28203_gb300.build import LIB, build
    if not os.path.exists(LIB):
        build()
    dpf.lib()


def _grid(n):
    return gridgen.config_grid("c1_30bus_fp64") if n == 30 else gridgen.make_grid(n, 3, load_scale=0.1)


def _run(y, ws, K, opts, streaming, **kw):
    N = y.n_bus
    out = dict(va=torch.zeros((K, N), dtype=torch.float64, device=DEV),
               vm=torch.ones((K, N), dtype=torch.float64, device=DEV),
               iters=torch.zeros(K, dtype=torch.int32, device=DEV),
               status=torch.zeros(K, dtype=torch.int32, device=DEV),
               max_mismatch=torch.zeros(K, dtype=torch.float64, device=DEV))
    b = dict(n_case=K, **out, **kw)
    dpf.dpf_profile_enable(ws, streaming)
    dpf.dpf_solve_begin(y, ws, opts, **b)
    dpf.dpf_solve_iterate(ws, opts.max_iter)
    dpf.dpf_solve_end(ws, **b)
    torch.cuda.synchronize()
    n_fwd = dpf.dpf_kernel_times(ws)[2]
    dpf.dpf_profile_enable(ws, False)
    assert (n_fwd > 0) == streaming  # the two forms really ran
    return {k: v.cpu().numpy() for k, v in out.items()}


def _same(a, b):
    for k in a:
        assert np.array_equal(a[k], b[k], equal_nan=True), k


def _inputs(g, K, seed, specs, outages):
    rng = np.random.default_rng(seed)
    kw = {}
    if specs:
        sc = 1 + 0.1 * rng.uniform(-1, 1, (K, 1))
        kw["p_spec"] = torch.tensor(g.p_spec * sc, device=DEV)
        kw["q_spec"] = torch.tensor(g.q_spec * sc, device=DEV)
    if outages:
        ok = gridgen.n1_outages(g)
        o = np.resize(rng.permutation(ok), K).astype(np.int32)
        o[::7] = -1
        kw["outage"] = torch.tensor(o, device=DEV)
    return kw


# sizes around the edges of the forms: one row per lane (32), two (64), one
# CTA per case above, its largest grid (2,048); cases around a CTA's four, a
# warp's 32 and the two-case kernels' 64 (whose loss order differs)
@pytest.mark.parametrize("n,K", [(2, 1), (30, 1), (30, 70), (32, 5), (33, 64), (64, 33), (65, 2), (129, 40), (300, 100),
                                 (700, 1), (1000, 40), (1025, 9), (2000, 130), (2048, 3)])
@pytest.mark.parametrize("precision", ["fp32", "fp32r"])
def test_on_chip_equals_streaming(n, K, precision):
    g = gridgen.two_bus(0.3, 0.1, 0.01, 0.1) if n == 2 else _grid(n)
    y = dpf.dpf_build_ybus(g)
    ws = dpf.dpf_workspace_create(y, K)
    opts = dpf.SolveOpts(precision=getattr(dpf, precision.upper()), max_iter=63, check_every=20, lr=3e-3, patience=3,
                         cooldown=5, gate=1e-1)
    kw = _inputs(g, K, n + K, specs=K > 4, outages=n > 2 and K != 5)
    _same(_run(y, ws, K, opts, False, **kw), _run(y, ws, K, opts, True, **kw))


# larger grids with about one element per thread of the GPU: fewer row blocks
# than SMs (one case), one and two tiles, two-case tiles with a padded half,
# lanes < 32, more row blocks than 64 (two-level loss sum), two rounds of tasks
# per warp; the last is just above the range
@pytest.mark.parametrize("n,K", [(2049, 1), (2500, 33), (2500, 65), (5000, 3), (9001, 17), (40000, 1), (40000, 4),
                                 (160001, 1), (10000, 20)])
@pytest.mark.parametrize("precision", ["fp32", "fp32r"])
def test_whole_gpu_equals_streaming(n, K, precision):
    g = _grid(n)
    y = dpf.dpf_build_ybus(g)
    ws = dpf.dpf_workspace_create(y, K)
    opts = dpf.SolveOpts(precision=getattr(dpf, precision.upper()), max_iter=63, check_every=20, lr=3e-3, patience=3,
                         cooldown=5, gate=1e-1)
    kw = _inputs(g, K, n + K, specs=K > 4, outages=K != 5)
    _same(_run(y, ws, K, opts, False, **kw), _run(y, ws, K, opts, True, **kw))


@pytest.mark.parametrize("n,K", [(30, 1), (64, 40), (65, 3), (300, 150)])
def test_on_chip_equals_streaming_fp64(n, K):
    g = _grid(n)
    y = dpf.dpf_build_ybus(g)
    ws = dpf.dpf_workspace_create(y, K)
    opts = dpf.SolveOpts(precision=dpf.FP64, max_iter=45, check_every=20, lr=3e-3, sched=dpf.SCHED_CONST)
    kw = _inputs(g, K, n, specs=True, outages=True)
    _same(_run(y, ws, K, opts, False, **kw), _run(y, ws, K, opts, True, **kw))


@pytest.mark.parametrize("opt", [dpf.OPT_SGD, dpf.OPT_RMSPROP, dpf.OPT_ADAM])
@pytest.mark.parametrize("n", [30, 300, 3000])
def test_on_chip_optimisers_and_step_schedule(opt, n):
    g = _grid(n)
    K = 6
    y = dpf.dpf_build_ybus(g)
    ws = dpf.dpf_workspace_create(y, K)
    opts = dpf.SolveOpts(precision=dpf.FP32, max_iter=50, check_every=16, lr=1e-3, optimizer=opt, momentum=0.5,
                         sched=dpf.SCHED_STEP, step_size=7, gamma=0.8)
    kw = _inputs(g, K, 1, specs=True, outages=False)
    _same(_run(y, ws, K, opts, False, **kw), _run(y, ws, K, opts, True, **kw))


@pytest.mark.parametrize("precision", ["fp32", "fp32r"])
@pytest.mark.parametrize("n", [30, 300, 3000])
def test_on_chip_divergence(n, precision):
    """A case stops as diverged before the step its loss makes impossible: at
    once (NaN injections) or after some steps (a rate that overflows |V|);
    the other cases go on."""
    g = _grid(n)
    K = 5
    y = dpf.dpf_build_ybus(g)
    ws = dpf.dpf_workspace_create(y, K)
    kw = _inputs(g, K, 4, specs=True, outages=False)
    kw["p_spec"][2, n // 2] = float("nan")
    opts = dpf.SolveOpts(precision=getattr(dpf, precision.upper()), max_iter=40, check_every=10, lr=1e-2)
    a = _run(y, ws, K, opts, False, **kw)
    _same(a, _run(y, ws, K, opts, True, **kw))
    assert a["status"][2] == dpf.CASE_DIVERGED and a["iters"][2] == 0 and a["iters"][0] == 40
    kw = _inputs(g, K, 4, specs=True, outages=False)
    opts = dpf.SolveOpts(precision=opts.precision, max_iter=40, check_every=10, lr=3e8, sched=dpf.SCHED_STEP,
                         step_size=1, gamma=4.0)
    a = _run(y, ws, K, opts, False, **kw)
    _same(a, _run(y, ws, K, opts, True, **kw))
    assert (a["status"] == dpf.CASE_DIVERGED).all() and (a["iters"] > 0).all() and (a["iters"] < 40).all()


# ---- the DC solve on chip ------------------------------------------------------
def _dc_true_residual(g, va, p, ell):
    """|B' theta - P| / |P| over the non-slack rows in FP64."""
    b = 1.0 / (g.x * np.where(g.tap == 0, 1.0, g.tap))
    if ell >= 0:
        b = b.copy()
        b[ell] = 0.0
    flow = b * (va[g.f_bus] - va[g.t_bus])
    r = -p.copy()
    np.add.at(r, g.f_bus, flow)
    np.add.at(r, g.t_bus, -flow)
    u = g.bus_type != gridgen.SLACK
    return np.linalg.norm(r[u]) / np.linalg.norm(p[u])


# one thread per row pair up to 1,024 threads, and (more cases than SMs) four
# or eight rows per thread; a partial last slice, one warp, and the largest grid
@pytest.mark.parametrize("n,K", [(2, 1), (30, 3), (65, 200), (300, 400), (1000, 2), (2047, 200), (2048, 1)])
@pytest.mark.parametrize("tol", [1e-10, 1e-4])
def test_dc_on_chip_residual(n, K, tol):
    """Every case stops at the recurrence's |r| <= tol |r0|; the residual of the
    returned angles recomputed in FP64 differs from the recurrence's by
    rounding: a few hundred steps of 2^-47 (double-float) stay below the
    tolerance itself, of 2^-24 (FP32 vectors) below 10 tol as
    test_dc_fp32_vectors_at_a_loose_tolerance allows.  Equal cases give equal
    bits whatever SM runs them."""
    g = gridgen.two_bus(0.3, 0.1, 0.01, 0.1) if n == 2 else _grid(n)
    y = dpf.dpf_build_ybus(g)
    ws = dpf.dpf_workspace_create(y, K)
    rng = np.random.default_rng(n)
    P = g.p_spec * (1 + 0.1 * rng.uniform(-1, 1, (K, 1)))
    o = np.full(K, -1, np.int32)
    if n > 2:
        o = np.resize(rng.permutation(gridgen.n1_outages(g)), K).astype(np.int32)
        o[0] = -1
    P[K // 2], o[K // 2] = P[0], o[0]
    out = dpf.dpf_dc_solve(y, ws, K, p_spec=torch.tensor(P, device=DEV), outage=torch.tensor(o, device=DEV), tol=tol)
    va, rr = out["va"].cpu().numpy(), out["rel_residual"].cpu().numpy()
    it = out["iters"].cpu().numpy()
    assert (rr <= tol).all() and (it >= 1).all()
    assert np.array_equal(va[K // 2], va[0]) and it[K // 2] == it[0]
    for k in range(0, K, max(1, K // 12)):
        assert _dc_true_residual(g, va[k], P[k], int(o[k])) <= (2 if tol < 1e-5 else 10) * tol, k
    if it.max() > 2:  # the cap stops a case where it stands
        cap = dpf.dpf_dc_solve(y, ws, K, p_spec=torch.tensor(P, device=DEV), outage=torch.tensor(o, device=DEV),
                               tol=tol, max_iter=2)
        assert (cap["iters"].cpu().numpy() <= 2).all() and (cap["rel_residual"].cpu().numpy() > tol).any()


# ---- evaluation on chip --------------------------------------------------------
@pytest.mark.parametrize("n,K", [(2, 3), (31, 1), (33, 200), (513, 5), (1025, 160), (2048, 2)])
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_evaluation_on_chip_against_oracle(n, K, precision):
    """S_calc, loss and gradients at the edges of the slices and CTA sizes
    (one row per thread up to 1,024 threads; 512 where cases outnumber SMs).
    FP32 bars: a row's current carries |Y_ii| |V| 2^-24 times a few terms
    (|Y_ii| up to ~200), 1e-4; gradients 1e-4 of their largest entry."""
    import oracle
    from oracle.ybus import grid_ybus
    g = gridgen.two_bus(0.3, 0.1, 0.01, 0.1) if n == 2 else gridgen.make_grid(n, 3, load_scale=0.1)
    Y = grid_ybus(g)
    y = dpf.dpf_build_ybus(g)
    ws = dpf.dpf_workspace_create(y, 1)  # (an evaluation on chip needs no room in the workspace)
    rng = np.random.default_rng(n)
    va, vm = 0.1 * rng.standard_normal((K, n)), 1 + 0.03 * rng.standard_normal((K, n))
    P, Q = g.p_spec * rng.uniform(0.9, 1.1, (K, 1)), g.q_spec * rng.uniform(0.9, 1.1, (K, 1))
    t = lambda a: torch.tensor(a, device=DEV)  # noqa: E731
    prec = dict(fp32=dpf.FP32, fp64=dpf.FP64)[precision]
    tol = 1e-4 if precision == "fp32" else 1e-11
    p, q = dpf.dpf_power(y, ws, t(va), t(vm), precision=prec)
    out = dpf.dpf_loss_backward(y, ws, t(va), t(vm), t(P), t(Q), precision=prec,
                                want=("loss", "d_va", "d_vm", "d_p", "d_q"))
    for k in range(0, K, max(1, K // 5)):
        V = vm[k] * np.exp(1j * va[k])
        S = V * np.conj(Y @ V)
        assert np.abs(p[k].cpu().numpy() - S.real).max() <= tol * max(1, np.abs(S).max())
        assert np.abs(q[k].cpu().numpy() - S.imag).max() <= tol * max(1, np.abs(S).max())
        L, ga, gm = oracle.loss_grad(Y, va[k], vm[k], P[k], Q[k], g.bus_type)
        assert abs(out["loss"][k].item() - L) <= 1e-11 * L
        scale = max(np.abs(ga).max(), np.abs(gm).max())
        assert np.abs(out["d_va"][k].cpu().numpy() - ga).max() <= tol * scale
        assert np.abs(out["d_vm"][k].cpu().numpy() - gm).max() <= tol * scale
        act, rea, m = g.bus_type != gridgen.SLACK, g.bus_type == gridgen.PQ, (g.bus_type != 2).sum() + (g.bus_type == 0).sum()
        c = 2.0 / m * (np.where(act, S.real - P[k], 0) + 1j * np.where(rea, S.imag - Q[k], 0))
        assert np.abs(out["d_p"][k].cpu().numpy() + c.real).max() <= tol * np.abs(c).max()
        assert np.abs(out["d_q"][k].cpu().numpy() + c.imag).max() <= tol * np.abs(c).max()


def test_evaluation_on_chip_extreme_values():
    """The integer FP64 <-> FP32 conversions hand what they do not cover (zeros,
    subnormals, infinities, NaN, very small and large values) to the CUDA
    ones: |V| at bus 0 of a two-bus grid scales P there quadratically."""
    g = gridgen.two_bus(0.3, 0.1, 0.01, 0.1)
    y = dpf.dpf_build_ybus(g)
    ws = dpf.dpf_workspace_create(y, 1)
    ys = 1 / (g.r[0] + 1j * g.x[0])
    m = np.array([0.0, -0.0, 1e-310, 1e-45, 1e-30, 1e-19, -1.5, 3.0, 1e10, 1e18, np.inf, np.nan])
    va = np.zeros((m.size, 2))
    vm = np.stack([m, np.zeros(m.size)], 1)  # bus 1 at 0: P_0 = g |V_0|^2
    p, _ = dpf.dpf_power(y, ws, torch.tensor(va, device=DEV), torch.tensor(vm, device=DEV), precision=dpf.FP32)
    p = p.cpu().numpy()[:, 0]
    with np.errstate(all="ignore"):
        want = ys.real * m.astype(np.float32).astype(np.float64) ** 2
    for a, b in zip(p, want):
        if not np.isfinite(b):
            assert not np.isfinite(a)
        elif abs(b) < 1e-36:  # below FP32's normal range
            assert abs(a) <= 1e-36
        elif abs(b) < 3e38:
            assert abs(a - b) <= 1e-5 * abs(b)
