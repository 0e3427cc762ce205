"""Which kernels run a span of iterations: the two-pass kernels launch at least
twice per iteration, the on-chip and whole-GPU forms once per span.  A solve
that changes between them keeps its bits (FP32)."""
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


def _solve(y, K, precision, ce, spans, graph=0, streaming=False):
    """One solve stepped by `spans`; its outputs and the launches per span."""
    n = y.n_bus
    ws = dpf.dpf_workspace_create(y, K)
    rng = np.random.default_rng(1)
    g = _grid(n)
    sc = 1 + 0.1 * rng.uniform(-1, 1, (K, 1))
    out = dict(n_case=K, va=torch.zeros((K, n), dtype=torch.float64, device=DEV),
               vm=torch.ones((K, n), dtype=torch.float64, device=DEV),
               iters=torch.zeros(K, dtype=torch.int32, device=DEV),
               max_mismatch=torch.zeros(K, dtype=torch.float64, device=DEV),
               p_spec=torch.tensor(g.p_spec * sc, device=DEV), q_spec=torch.tensor(g.q_spec * sc, device=DEV))
    o = dpf.SolveOpts(precision=precision, max_iter=sum(spans), check_every=ce, lr=3e-3, patience=3, cooldown=4,
                      tol=1e-12, use_graph=graph)
    dpf.dpf_profile_enable(ws, streaming)
    dpf.dpf_solve_begin(y, ws, o, **out)
    launches = []
    for k in spans:
        before = dpf.dpf_kernel_launches(ws)
        dpf.dpf_solve_iterate(ws, k)
        launches.append(dpf.dpf_kernel_launches(ws) - before)
    dpf.dpf_solve_end(ws, **out)
    torch.cuda.synchronize()
    return {k: out[k].cpu().numpy() for k in ("va", "vm", "iters", "max_mismatch")}, launches


def _grid(n):
    return gridgen.make_grid(n, 3, load_scale=0.05)


# (check interval; long spans on chip, short ones streaming)
@pytest.mark.parametrize("n,K,precision,short,long", [(30, 8192, "FP32", 1, 2), (100, 2000, "FP32", 2, 3),
                                                      (300, 3000, "FP32R", 3, 4), (2000, 600, "FP32R", 7, 8),
                                                      (2000, 2379, "FP32R", 9, 10), (2000, 2379, "FP32", 5, 6),
                                                      (2500, 64, "FP32", 13, 14), (2500, 1, "FP32R", 1, 2)])
def test_short_spans_run_streaming(n, K, precision, short, long):
    y = dpf.dpf_build_ybus(_grid(n))
    prec = getattr(dpf, precision)
    ce = 20
    spans = [short, ce - short, long, ce - long, ce, 1]
    a, launches = _solve(y, K, prec, ce, spans)
    assert launches[0] >= 2 * short and launches[2] < 2 * long + 4
    assert launches[2] <= 6  # the test (five kernels) and one launch
    if ce - short >= long:
        assert launches[1] == 1
    assert launches[4] <= 6 and launches[5] >= (2 if short >= 1 else 1)
    b, _ = _solve(y, K, prec, ce, spans, streaming=True)
    for k in a:
        assert np.array_equal(a[k], b[k]), k


@pytest.mark.parametrize("n,K", [(2000, 2379), (2500, 64)])
def test_tests_after_every_iteration_run_streaming(n, K):
    """check_every = 1 through the graph path."""
    y = dpf.dpf_build_ybus(_grid(n))
    a, launches = _solve(y, K, dpf.FP32R, 1, [6], graph=1)
    assert launches[0] >= 6 * 3  # two passes and a test each
    b, _ = _solve(y, K, dpf.FP32R, 1, [6], streaming=True)
    for k in a:
        assert np.array_equal(a[k], b[k]), k


def test_few_cases_keep_the_on_chip_form_for_single_steps():
    y = dpf.dpf_build_ybus(_grid(300))
    _, launches = _solve(y, 20, dpf.FP32, 20, [20, 1, 1, 1])
    assert launches[2:] == [1, 1]


# the ends of the ranges in which whole warps of FP64 rows pay on 152 SMs, and
# FP32 batches that half fill their rows
@pytest.mark.parametrize("n,K,precision,chip", [
    (14, 1216, "FP64", True), (14, 1217, "FP64", False), (30, 5000, "FP64", True), (30, 8000, "FP64", False),
    (33, 608, "FP64", True), (33, 609, "FP64", False), (64, 1000, "FP64", True), (64, 1216, "FP64", False),
    (64, 1824, "FP64", True), (64, 2400, "FP64", False), (300, 300, "FP64", True), (300, 301, "FP64", False),
    (14, 32768, "FP32", True), (14, 32769, "FP32", False), (30, 40000, "FP32", True), (65, 16385, "FP32R", False)])
def test_many_cases_of_narrow_grids_run_streaming(n, K, precision, chip):
    if torch.cuda.get_device_properties(0).multi_processor_count != 152:
        pytest.skip("the limits count 152 SMs")
    y = dpf.dpf_build_ybus(_grid(n))
    _, launches = _solve(y, K, getattr(dpf, precision), 20, [20, 20])
    assert all((k <= 6) == chip for k in launches), launches


# Newton, FP32: CTAs of the shared-memory factor on 152 SMs (10, 5, 4, 4, 2, 2 an SM)
# in as many waves as pay; one case more goes to the global form
@pytest.mark.parametrize("n,most", [(30, 152 * 10 * 27 // 20), (118, 152 * 5 * 2), (200, 152 * 4 * 2),
                                    (256, 152 * 4 * 3), (300, 152 * 2 * 3), (600, 152 * 2 * 4)])
def test_newton_factor_leaves_shared_memory_with_many_cases(n, most):
    """A step in shared memory is two launches shorter than the global form
    (assembly and update are part of it)."""
    if torch.cuda.get_device_properties(0).multi_processor_count != 152:
        pytest.skip("the limits count 152 SMs")
    y = dpf.dpf_build_ybus(_grid(n))
    for K, chip in ((most, True), (most + 1, False)):
        nr = dpf.dpf_nr_create(y, K)
        out = {k: torch.ones((K, n), dtype=torch.float64, device=DEV) for k in ("va", "vm")}
        count, va = [], []
        for lanes in (0, 8):
            before = nr.stats()["launches"]
            dpf.dpf_nr_solve(nr, precision=dpf.FP32, tol=1e-9, max_iter=1, n_case=K, lanes=lanes, **out)
            count.append(nr.stats()["launches"] - before)
            va.append(out["va"].clone())
        assert count[1] - count[0] == (2 if chip else 0)
        assert torch.equal(va[0], va[1])
