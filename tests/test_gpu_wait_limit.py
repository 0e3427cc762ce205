"""A grid barrier of the whole-GPU iterations that gives up is an error of the
solve, whichever way it is driven; the next solve of the workspace is sound."""
import numpy as np
import pytest

import gridgen

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2603_28203_gb300 as dpf  # noqa: E402
from paper_2603_28203_gb300 import _abi  # noqa: E402

DEV = torch.device("cuda:0")


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import os
    from paper_2603_28203_gb300.build import LIB, build
    if not os.path.exists(LIB):
        build()
    dpf.lib()


@pytest.mark.parametrize("n,K", [(2500, 3), (40000, 1)])
def test_a_barrier_that_gives_up_ends_the_solve_with_an_error(n, K):
    """One poll is too few for CTAs that do not arrive together."""
    y = dpf.dpf_build_ybus(gridgen.make_grid(n, 3, load_scale=0.1))
    ws = dpf.dpf_workspace_create(y, K)
    opts = dpf.SolveOpts(precision=dpf.FP32, max_iter=60, check_every=20, lr=3e-3)
    out = dict(n_case=K, va=torch.zeros((K, n), dtype=torch.float64, device=DEV),
               vm=torch.ones((K, n), dtype=torch.float64, device=DEV))

    def solve():
        dpf.dpf_solve_batch(y, ws, opts, **out)
        return out["va"].cpu().numpy().copy()

    def stepped():
        dpf.dpf_solve_begin(y, ws, opts, **out)
        dpf.dpf_solve_iterate(ws, 60)
        dpf.dpf_solve_end(ws, **out)

    ref = solve()
    dpf.dpf_wait_limit(ws, 1)
    for run in (solve, stepped):
        with pytest.raises(dpf.DPFError) as e:
            run()
        assert e.value.code == _abi.DPF_E_CUDA and "barrier" in str(e.value)
    with pytest.raises(dpf.DPFError):  # the failed solve is over
        dpf.dpf_solve_iterate(ws, 20)
    dpf.dpf_solve_begin(y, ws, opts, **out)
    dpf.dpf_solve_iterate(ws, 20)
    with pytest.raises(dpf.DPFError):
        dpf.dpf_active_count(ws)
    dpf.dpf_wait_limit(ws)
    assert np.array_equal(solve(), ref)
    stepped()
    assert np.array_equal(out["va"].cpu().numpy(), ref)
