"""Branch-parameter identification by gradient descent on the power mismatch.

The paper motivates DPF by end-to-end gradients from the power mismatches to
the simulation parameters, which "allows these parameters to be identified"
(abstract, Sec. 1), without an experiment.  Here: given K measured operating
points (V = |V| e^{j theta} and the injections P, Q at every bus), the series
admittances g + jb of every branch are adjusted by Adam to minimise the sum
over operating points of the DPF loss of Alg. 1 at those fixed voltages.
The operating points are staged once (dpf_paramid_begin); each step takes
the branch gradient from dpf_paramid_step (Y values rebuilt by k_ybus_values,
forward pass, branch adjoint k_edge_grad) and the step from dpf_adam_update;
the learning rate of each parameter is scaled by its starting magnitude, so a
step is a relative change of about `lr`.
"""
from __future__ import annotations

import ctypes as C

import torch

from . import _abi
from .dpf import Workspace, Ybus, _check, _ptr, _stream, dpf_paramid_begin, lib


def identify_branches(y: Ybus, ws: Workspace, va, vm, p, q, g0, b0, iters: int, lr: float = 3e-3,
                      betas=(0.9, 0.999), precision=_abi.FP32, record_every: int = 0, stream=None):
    """Returns (g, b, history); g0, b0 are [M] float64 CUDA tensors, the others [K][N]."""
    g = g0.clone()
    b = b0.clone()
    mg, vg, mb, vb = (torch.zeros_like(g0) for _ in range(4))
    sg, sb = g0.abs(), b0.abs()
    hist = []
    dpf_paramid_begin(y, ws, va, vm, p, q, precision=precision, stream=stream)
    # The loop's buffers do not change, so its calls (dpf_paramid_step, then
    # dpf_adam_update on g and on b) take arguments marshalled once: a step is
    # some 20 us of kernels, less than marshalling three calls afresh.
    L, h = lib(), _stream(stream)
    dg, db = (torch.empty(y.n_branch, dtype=torch.float64, device=g0.device) for _ in range(2))
    loss = torch.empty(int(va.shape[0]) if record_every else 0, dtype=torch.float64, device=g0.device)
    ptr = lambda t: C.c_void_p(_ptr(t))  # noqa: E731
    n, h = C.c_int32(int(g0.numel())), C.c_void_p(h)
    step = (y.handle, ws.handle, ptr(g), ptr(b), ptr(dg), ptr(db), None)
    adam = [(n, ptr(x), ptr(d), ptr(m), ptr(v), ptr(sc)) for x, d, m, v, sc in
            ((g, dg, mg, vg, sg), (b, db, mb, vb, sb))]
    rate = (C.c_double(lr), C.c_double(betas[0]), C.c_double(betas[1]), C.c_double(1e-8), h)
    for t in range(1, iters + 1):
        record = bool(record_every) and t % record_every == 0
        _check(L.dpf_paramid_step(*step, ptr(loss) if record else None, h))
        if record:
            hist.append((t, float(loss.sum().item())))
        for a in adam:
            _check(L.dpf_adam_update(*a, t, *rate))
    return g, b, hist
