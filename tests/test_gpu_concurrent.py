"""Solves of different grids at the same time, from several threads or
interleaved in one: a kernel's shared-memory limit is common to all of them."""
import threading

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


class _Newton:
    def __init__(self, n, K):
        self.y = dpf.dpf_build_ybus(gridgen.make_grid(n, 3, load_scale=0.1))
        self.nr = dpf.dpf_nr_create(self.y, K)
        self.out = dict(n_case=K, va=torch.zeros((K, n), dtype=torch.float64, device=DEV),
                        vm=torch.ones((K, n), dtype=torch.float64, device=DEV))

    def __call__(self, stream):
        dpf.dpf_nr_solve(self.nr, precision=dpf.FP32, tol=1e-9, max_iter=8, stream=stream, **self.out)
        stream.synchronize()
        return self.out["va"].cpu().numpy()


class _Iterate(_Newton):
    def __init__(self, n, K):
        super().__init__(n, K)
        self.ws = dpf.dpf_workspace_create(self.y, K)
        self.opts = dpf.SolveOpts(precision=dpf.FP32R, max_iter=30, check_every=15, use_graph=0)

    def __call__(self, stream):
        dpf.dpf_solve_batch(self.y, self.ws, self.opts, stream=stream, **self.out)
        stream.synchronize()
        return self.out["va"].cpu().numpy()


class _Dc(_Iterate):
    def __call__(self, stream):
        return dpf.dpf_dc_solve(self.y, self.ws, self.out["n_case"], tol=1e-8, stream=stream)["va"].cpu().numpy()


# grids whose factor, sliced Y_bus or sliced B takes 60 KB to 200 KB of shared memory
@pytest.mark.parametrize("kind", [_Newton, _Iterate, _Dc])
def test_two_threads_with_different_grids(kind):
    solvers = [kind(n, 4) for n in (2000, 1000)]
    want = [s(torch.cuda.default_stream()).copy() for s in solvers]
    torch.cuda.synchronize()
    errors = []

    def work(i):
        try:
            stream = torch.cuda.Stream()
            with torch.cuda.stream(stream):
                for _ in range(60):
                    assert np.array_equal(solvers[i](stream), want[i])
        except BaseException as e:  # noqa: BLE001
            errors.append(e)

    threads = [threading.Thread(target=work, args=(i,)) for i in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not errors, errors[0]


def test_interleaved_solves_with_staged_windows():
    """Two streaming solves begun one after the other, then iterated: each V
    window keeps the shared memory it was given."""
    K, runs = 64, []
    for n in (10000, 2000, 4000):
        y = dpf.dpf_build_ybus(gridgen.make_grid(n, 3, load_scale=0.05))
        ws = dpf.dpf_workspace_create(y, K)
        out = dict(n_case=K, va=torch.zeros((K, n), dtype=torch.float64, device=DEV),
                   vm=torch.ones((K, n), dtype=torch.float64, device=DEV))
        runs.append((y, ws, out, dpf.SolveOpts(precision=dpf.FP32, max_iter=20, check_every=10, stage_v=1, pair_cases=0,
                                               use_graph=0)))
    want = []
    for y, ws, out, o in runs:
        dpf.dpf_solve_batch(y, ws, o, **out)
        want.append(out["va"].cpu().numpy().copy())
    for y, ws, out, o in runs:
        dpf.dpf_solve_begin(y, ws, o, **out)
    for y, ws, out, o in runs:
        dpf.dpf_solve_iterate(ws, 20)
    for (y, ws, out, o), w in zip(runs, want):
        dpf.dpf_solve_end(ws, **out)
        assert np.array_equal(out["va"].cpu().numpy(), w)
