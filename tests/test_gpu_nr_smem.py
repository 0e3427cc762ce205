"""Newton-Raphson with one case's factor in shared memory against the
global-memory form (lanes > 0 forces that): every sum runs in the same order,
so the results agree to the bit.  Sizes around the CTA sizes (64, 256, 1,000
buses), dense grids whose pivots are larger than a stage of the schedule,
islands, and a single bus pair."""
import numpy as np
import pytest

import gridgen

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2603_28203_gb300 as dpf  # noqa: E402

DEV = torch.device("cuda:0")


def _grid(n, extra, islands):
    if n == 2:
        return gridgen.two_bus(0.1, 0.05, 0.01, 0.1)
    g = gridgen.make_grid(n, 3, load_scale=0.1)
    if extra:
        g = gridgen.add_random_branches(g, extra, 7)
    return gridgen.concat_grids([g, gridgen.make_grid(n // 2, 4, load_scale=0.1)]) if islands else g


@pytest.mark.parametrize("n,extra,islands", [(2, 0, False), (5, 0, False), (63, 0, False), (65, 0, False),
                                             (257, 0, True), (1001, 0, False), (40, 600, False), (100, 3000, False)])
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_shared_memory_form_has_the_global_form_s_bits(n, extra, islands, precision):
    g = _grid(n, extra, islands)
    outs = gridgen.n1_outages(g)[:2] if n > 2 else np.empty(0, np.int64)
    ids = np.array([-1, *outs], dtype=np.int32)
    K, N = ids.size, g.n_bus
    y = dpf.dpf_build_ybus(g)
    nr = dpf.dpf_nr_create(y, K)
    outage = torch.tensor(ids, device=DEV)
    runs = []
    for lanes in (0, 1):
        o = {k: torch.zeros((K, N), dtype=torch.float64, device=DEV) for k in ("va", "vm")}
        o.update({k: torch.zeros(K, dtype=torch.float64, device=DEV) for k in ("max_mismatch", "loss")})
        o.update({k: torch.zeros(K, dtype=torch.int32, device=DEV) for k in ("iters", "status")})
        dpf.dpf_nr_solve(nr, precision=dpf.FP32 if precision == "fp32" else dpf.FP64, tol=1e-9, max_iter=8,
                         n_case=K, outage=outage, lanes=lanes, **o)
        torch.cuda.synchronize()
        runs.append({k: v.cpu().numpy() for k, v in o.items()})
    assert (runs[0]["iters"] > 0).all()
    for k in runs[0]:
        np.testing.assert_array_equal(runs[0][k], runs[1][k])


def test_a_start_that_is_not_a_number_diverges_alone():
    """A case whose start holds a NaN diverges and the others are untouched."""
    g = gridgen.make_grid(120, 3, load_scale=0.1)
    K, N = 3, g.n_bus
    y = dpf.dpf_build_ybus(g)
    nr = dpf.dpf_nr_create(y, K)
    va = torch.zeros((K, N), dtype=torch.float64, device=DEV)
    vm = torch.ones((K, N), dtype=torch.float64, device=DEV)
    pq = int(np.flatnonzero(np.asarray(g.bus_type) == 0)[0])
    va[1, pq] = float("nan")
    status = torch.zeros(K, dtype=torch.int32, device=DEV)
    mm = torch.zeros(K, dtype=torch.float64, device=DEV)
    dpf.dpf_nr_solve(nr, precision=dpf.FP32, tol=1e-9, max_iter=8, flat_start=False, n_case=K, va=va, vm=vm,
                     status=status, max_mismatch=mm)
    torch.cuda.synchronize()
    assert status.tolist() == [dpf.CASE_CONVERGED, dpf.CASE_DIVERGED, dpf.CASE_CONVERGED]
    assert np.isnan(mm[1].item()) and (va[0] == va[2]).all()
