"""Grids with long rows (stars, dense and randomly meshed networks): their sliced
form of Y_bus may not fit shared memory, or is mostly padding."""
import dataclasses

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


def _star(n):
    g = gridgen.make_grid(n, 3, load_scale=0.05)
    hub = int(np.flatnonzero(g.bus_type == gridgen.SLACK)[0])
    rng, m = np.random.default_rng(1), n - 1
    r = rng.uniform(0.002, 0.02, m)
    return dataclasses.replace(g, f_bus=np.full(m, hub, np.int32), t_bus=np.delete(np.arange(n), hub).astype(np.int32),
                               r=r, x=10 * r, b_ch=np.zeros(m), tap=np.ones(m), shift=np.zeros(m))


def _grid(name):
    if name.startswith("star"):
        return _star(int(name[4:]))
    n, extra = (int(v) for v in name.split("+"))
    return gridgen.add_random_branches(gridgen.make_grid(n, 3, load_scale=0.05), extra, 1)


def _residual(g, va, p):
    """|B theta - P| / |P| over the non-slack rows in FP64."""
    flow = (va[g.f_bus] - va[g.t_bus]) / (g.x * np.where(g.tap == 0, 1.0, g.tap))
    r = -p.copy()
    np.add.at(r, g.f_bus, flow)
    np.add.at(r, g.t_bus, -flow)
    u = g.bus_type != gridgen.SLACK
    return np.linalg.norm(r[u]) / np.linalg.norm(p[u])


# sliced form of B: 243 KB (double-float), 712 / 427 KB, 249 KB, 232 KB; the
# last one just fits
@pytest.mark.parametrize("name", ["star700", "star2048", "150+10500", "300+10000", "300+9000"])
@pytest.mark.parametrize("tol", [1e-10, 1e-4])
@pytest.mark.parametrize("K", [2, 160])
def test_dc_of_a_dense_grid(name, tol, K):
    """A grid whose sliced B doesn't fit shared memory takes the streaming CG;
    bars as for the on-chip solve (test_dc_on_chip_residual): 2 tol in
    double-float, 10 tol in FP32."""
    g = _grid(name)
    y = dpf.dpf_build_ybus(g)
    ws = dpf.dpf_workspace_create(y, K)
    P = g.p_spec * (1 + 0.1 * np.random.default_rng(2).uniform(-1, 1, (K, 1)))
    Pt = torch.tensor(P, device=DEV)
    out = dpf.dpf_dc_solve(y, ws, K, p_spec=Pt, tol=tol)
    assert (out["rel_residual"].cpu().numpy() <= tol).all() and (out["iters"].cpu().numpy() >= 1).all()
    bar = (2 if tol < 1e-5 else 10) * tol
    va = out["va"].cpu().numpy()
    for k in range(0, K, max(1, K // 5)):
        assert _residual(g, va[k], P[k]) <= bar, k
    # the same start inside a solve
    res = dict(va=torch.zeros((K, g.n_bus), dtype=torch.float64, device=DEV),
               vm=torch.zeros((K, g.n_bus), dtype=torch.float64, device=DEV))
    dpf.dpf_solve_batch(y, ws, dpf.SolveOpts(precision=dpf.FP32R, max_iter=0, dc_start=1, dc_tol=tol), n_case=K,
                        p_spec=Pt, q_spec=torch.zeros_like(Pt), **res)
    for k in range(0, K, max(1, K // 5)):
        assert _residual(g, res["va"][k].cpu().numpy(), P[k]) <= bar, k


def _hub(n, degree):
    """make_grid with `degree` more branches at bus n // 2."""
    g = gridgen.make_grid(n, 3, load_scale=0.05)
    h = n // 2
    near = {h, *g.t_bus[g.f_bus == h], *g.f_bus[g.t_bus == h]}
    to = np.random.default_rng(0).permutation([i for i in range(n) if i not in near])[:degree]
    new = dict(f_bus=np.full(degree, h), t_bus=to, r=np.full(degree, 0.05), x=np.full(degree, 0.3),
               b_ch=np.zeros(degree), tap=np.ones(degree), shift=np.zeros(degree))
    return dataclasses.replace(g, **{k: np.concatenate([getattr(g, k), v.astype(getattr(g, k).dtype)])
                                     for k, v in new.items()})


@pytest.mark.parametrize("name,K,precision,chip", [("300+4800", 500, "FP32", True), ("300+4800", 1000, "FP32", False),
                                                   ("150+5000", 100, "FP32R", True), ("150+5000", 1000, "FP32R", False),
                                                   ("star300", 1000, "FP32", False), ("hub", 2400, "FP32", False),
                                                   ("hub", 1000, "FP32", True), ("star300", 1, "FP64", False),
                                                   ("60+1400", 1, "FP64", False), ("60+1400", 1000, "FP32", True)])
def test_iterations_of_dense_grids_run_where_they_are_faster(name, K, precision, chip):
    """A span of 20 iterations is one launch on chip, 40 streaming; FP32 gives
    the same bits either way."""
    if torch.cuda.get_device_properties(0).multi_processor_count != 152:
        pytest.skip("the limits count 152 SMs")
    g = _hub(1000, 160) if name == "hub" else _grid(name)
    y = dpf.dpf_build_ybus(g)
    ws = dpf.dpf_workspace_create(y, K)
    opts = dpf.SolveOpts(precision=getattr(dpf, precision), max_iter=40, check_every=20, lr=1e-3, use_graph=0)
    va = []
    for streaming in (False, True):
        out = dict(n_case=K, va=torch.zeros((K, g.n_bus), dtype=torch.float64, device=DEV),
                   vm=torch.ones((K, g.n_bus), dtype=torch.float64, device=DEV))
        dpf.dpf_profile_enable(ws, streaming)
        dpf.dpf_solve_begin(y, ws, opts, **out)
        before = dpf.dpf_kernel_launches(ws)
        dpf.dpf_solve_iterate(ws, 20)
        launches = dpf.dpf_kernel_launches(ws) - before
        assert (launches <= 6) == (chip and not streaming), launches
        dpf.dpf_solve_iterate(ws, 20)
        dpf.dpf_solve_end(ws, **out)
        va.append(out["va"])
    if precision != "FP64":
        assert torch.equal(va[0], va[1])


@pytest.mark.parametrize("name,K,tol,chip", [("1000+8000", 1000, 1e-4, True), ("1000+8000", 2400, 1e-4, False),
                                             ("300+4800", 1000, 1e-10, True), ("300+4800", 2400, 1e-10, False)])
def test_dc_of_dense_grids_runs_where_it_is_faster(name, K, tol, chip):
    """On chip a DC solve is one launch beside its set-up, streaming two per
    iteration; the residual bars are those of test_dc_of_a_dense_grid."""
    if torch.cuda.get_device_properties(0).multi_processor_count != 152:
        pytest.skip("the limits count 152 SMs")
    g = _grid(name)
    y = dpf.dpf_build_ybus(g)
    ws = dpf.dpf_workspace_create(y, K)
    P = g.p_spec * (1 + 0.1 * np.random.default_rng(2).uniform(-1, 1, (K, 1)))
    before = dpf.dpf_kernel_launches(ws)
    out = dpf.dpf_dc_solve(y, ws, K, p_spec=torch.tensor(P, device=DEV), tol=tol)
    assert (dpf.dpf_kernel_launches(ws) - before < 12) == chip
    assert (out["rel_residual"].cpu().numpy() <= tol).all()
    for k in range(0, K, K // 4):
        assert _residual(g, out["va"][k].cpu().numpy(), P[k]) <= (2 if tol < 1e-5 else 10) * tol, k


# more cases than SMs of grids that one warp holds: two rows per thread
@pytest.mark.parametrize("n", [5, 30, 33, 64])
@pytest.mark.parametrize("tol", [1e-10, 1e-4])
def test_dc_of_many_small_grids(n, tol):
    K = 700
    g = gridgen.make_grid(n, 3, load_scale=0.1)
    y = dpf.dpf_build_ybus(g)
    ws = dpf.dpf_workspace_create(y, K)
    P = g.p_spec * (1 + 0.1 * np.random.default_rng(n).uniform(-1, 1, (K, 1)))
    P[K - 1] = P[0]
    out = dpf.dpf_dc_solve(y, ws, K, p_spec=torch.tensor(P, device=DEV), tol=tol)
    va = out["va"].cpu().numpy()
    assert (out["rel_residual"].cpu().numpy() <= tol).all() and np.array_equal(va[0], va[K - 1])
    for k in range(0, K, 50):
        assert _residual(g, va[k], P[k]) <= (2 if tol < 1e-5 else 10) * tol, k


# rows of the hub staged in 20 to 75 KB beside the passes' static arrays
@pytest.mark.parametrize("n", [700, 1200, 1500, 1700, 2048, 3000])
@pytest.mark.parametrize("K", [1, 40])
def test_fp64_passes_of_a_star(n, K):
    """The streaming FP64 passes on a bus of n - 1 branches: one step of a solve
    from the flat start, against the oracle's S_calc through the mismatch."""
    import oracle
    from oracle.ybus import grid_ybus
    g = _star(n)
    y = dpf.dpf_build_ybus(g)
    ws = dpf.dpf_workspace_create(y, K)
    out = dict(n_case=K, va=torch.zeros((K, n), dtype=torch.float64, device=DEV),
               vm=torch.ones((K, n), dtype=torch.float64, device=DEV),
               loss=torch.zeros(K, dtype=torch.float64, device=DEV))
    dpf.dpf_solve_batch(y, ws, dpf.SolveOpts(precision=dpf.FP64, max_iter=3, check_every=2, lr=1e-4), **out)
    Y = grid_ybus(g)
    for k in (0, K - 1):
        va, vm = out["va"][k].cpu().numpy(), out["vm"][k].cpu().numpy()
        loss = oracle.loss_grad(Y, va, vm, g.p_spec, g.q_spec, g.bus_type)[0]
        assert abs(out["loss"][k].item() - loss) <= 1e-10 * loss


@pytest.mark.parametrize("name,K,precision,chip", [("star700", 342, "FP32", True), ("star700", 343, "FP32", False),
                                                   ("star700", 343, "FP64", False), ("14", 32768, "FP64", True),
                                                   ("14", 32769, "FP64", False), ("14", 32769, "FP32", False)])
def test_evaluations_run_where_they_are_faster(name, K, precision, chip):
    """Gradients by either route against the oracle; an evaluation on chip is
    one launch, streaming is more.  FP32 bars as in
    test_evaluation_on_chip_against_oracle, for |Y_ii| of a hub (700 x 100) by
    the sum's 350 pairs: 1e-3; without room in the workspace it stays on chip."""
    import oracle
    from oracle.ybus import grid_ybus
    g = _grid(name) if name != "14" else gridgen.make_grid(14, 3, load_scale=0.1)
    Y = grid_ybus(g)
    y = dpf.dpf_build_ybus(g)
    rng = np.random.default_rng(5)
    n, distinct = g.n_bus, 7
    va, vm = 0.05 * rng.standard_normal((distinct, n)), 1 + 0.02 * rng.standard_normal((distinct, n))
    at = np.arange(K) % distinct
    t = lambda a: torch.tensor(a[at], device=DEV)  # noqa: E731
    for room, on_chip in ((K, chip), (1, True)):
        ws = dpf.dpf_workspace_create(y, room)
        before = dpf.dpf_kernel_launches(ws)
        out = dpf.dpf_loss_backward(y, ws, t(va), t(vm), precision=getattr(dpf, precision))
        assert (dpf.dpf_kernel_launches(ws) - before == 1) == on_chip
        tol = 1e-3 if precision == "FP32" else 1e-10
        for k in (*range(distinct), K - 1):
            L, ga, gm = oracle.loss_grad(Y, va[at[k]], vm[at[k]], g.p_spec, g.q_spec, g.bus_type)
            assert abs(out["loss"][k].item() - L) <= 1e-10 * L
            scale = max(np.abs(ga).max(), np.abs(gm).max())
            assert np.abs(out["d_va"][k].cpu().numpy() - ga).max() <= tol * scale
            assert np.abs(out["d_vm"][k].cpu().numpy() - gm).max() <= tol * scale


@pytest.mark.parametrize("n,degree,K,whole", [(3000, 100, 4, True), (3000, 160, 4, False), (3000, 160, 1, False),
                                              (6000, 160, 1, True), (6000, 160, 2, False)])
def test_whole_gpu_iterations_of_a_hub(n, degree, K, whole):
    """A bus of more than about 128 branches runs streaming, with the same bits."""
    g = _hub(n, degree)
    y = dpf.dpf_build_ybus(g)
    ws = dpf.dpf_workspace_create(y, K)
    opts = dpf.SolveOpts(precision=dpf.FP32, max_iter=40, check_every=20, lr=1e-3, use_graph=0)
    va = []
    for streaming in (False, True):
        out = dict(n_case=K, va=torch.zeros((K, n), dtype=torch.float64, device=DEV),
                   vm=torch.ones((K, n), dtype=torch.float64, device=DEV))
        dpf.dpf_profile_enable(ws, streaming)
        dpf.dpf_solve_begin(y, ws, opts, **out)
        before = dpf.dpf_kernel_launches(ws)
        dpf.dpf_solve_iterate(ws, 20)
        assert (dpf.dpf_kernel_launches(ws) - before <= 6) == (whole and not streaming)
        dpf.dpf_solve_iterate(ws, 20)
        dpf.dpf_solve_end(ws, **out)
        va.append(out["va"])
    assert torch.equal(va[0], va[1])
