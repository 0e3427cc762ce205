// On-chip form of the iterations (dpf_resident.cu): its launch parameters,
// shared with the host code that chooses it (dpf_api.cu).
#pragma once

#include "dpf_internal.h"

namespace dpf {

template <class R> struct IterArgs;

// Grids up to this many buses can run the on-chip form (a case's working set
// must fit one SM: 1,024 threads of two rows).
constexpr int RES_MAX_N = 2048;
constexpr int RES_WARP_N = 64;       // up to here one warp runs a case
constexpr int RES_TEAMS = 4;         // cases (warps) per CTA of the one-warp form

// Launch shape for one grid and precision.
struct ResShape {
  bool ok = false;
  bool warp = false;  // one warp per case
  int rpt = 1;        // rows per thread
  int T = 32;         // compute threads per case
  size_t smem = 0;
};

// The order in which the streaming kernels of the same options sum a case's
// loss (row blocks, warps, rows per warp), which the on-chip form repeats.
struct LossOrder {
  int gy, rpb, wpb, rpw, tile, nthr;
};

// Whether (and how) a solve of K cases runs on chip; smem_limit: opt-in shared
// memory per CTA.
ResShape res_shape(const dpf_ybus* y, int K, bool fp64, bool refined, const LossOrder& lo, size_t smem_limit);

// Enqueue n_it iterations of every active case (refined: DPF_FP32R); pdl:
// programmatic dependent launch.  Returns a cudaError_t.
template <class R>
int res_launch(const dpf_ybus* y, const IterArgs<R>& a, const ResShape& sh, const LossOrder& lo, int K, int n_it,
               bool refined, bool pdl, void* stream);

// Whole-GPU form of the FP32 iterations (dpf_grid.cu): one persistent launch
// per test interval for larger grids whose batch fits the SMs together.
struct GridShape {
  bool ok = false;
  int ctas = 0, warps = 0, workers = 0;
  int gx = 0;   // case tiles that hold cases
  int vb = 0;   // virtual blocks (case tile x row block) per CTA
  size_t smem = 0;
};
GridShape grid_shape(const dpf_ybus* y, int K, const LossOrder& lo, int lanes, size_t smem_limit);
// terms: 4 Kp floats; suspect: Kp words, zero between launches; bar: two words;
// err: set to 1 if a barrier gave up after `polls`.  Returns a cudaError_t.
constexpr int64_t GRID_POLLS = 1 << 20;  // of some 0.7 us: about a second
int grid_launch(const IterArgs<float>& a, const GridShape& g, const LossOrder& lo, int lanes, int K, int n_it,
                bool refined, float* terms, unsigned* suspect, unsigned* bar, int32_t* err, int64_t polls,
                void* stream);

// One interval of a solve with a whole-GPU shape: by `whole`, or by `streaming`
// (for good) where the driver refuses the cooperative launch.  grid_shape
// counts the device's SMs, of which a context or stream may have fewer (MPS, a
// green context); nothing of the interval has run when it is refused.  Both
// return a cudaError_t, `refused` clears the runtime's last error.
inline bool launch_refused(int e) {
  return e == 720 || e == 701 || e == 801;  // too large to be resident, out of resources, not supported
}
template <class Whole, class Cleared, class Streaming>
int whole_or_streaming(GridShape& g, Whole whole, Cleared refused, Streaming streaming) {
  if (g.ok) {
    const int e = whole();
    if (!launch_refused(e)) return e;
    refused();
    g = GridShape();
  }
  return streaming();
}

// On-chip form of the DC solve (dpf_dc_resident.cu): every case of the batch
// to its tolerance in one launch.
struct DcRes {
  int K, Kp, max_iter, spec_per_case;
  double tol, va_slack;
  const double* pspec;   // [N][Kp] or [N]
  const int32_t *of, *ot;
  const double *ob, *flow;
  double *x, *res;       // [N][Kp] FP64 solution; |r| / |r0| per case
  int32_t* iters;
};
// Launch shape for K cases (f32: FP32 vectors, else double-float); ok: the
// grid has the sliced form and one case fits the shared memory of an SM.
struct DcShape {
  bool ok = false;
  int rpt = 2;  // rows per thread
  int T = 32;   // threads
  size_t smem = 0;
};
DcShape dc_res_shape(const dpf_ybus* y, int K, bool f32);
// Returns a cudaError_t.
int dc_res_launch(const dpf_ybus* y, const DcRes& c, const DcShape& sh, bool f32, void* stream);

// Evaluation of whole cases on chip (dpf_eval.cu), one CTA per case: S_calc,
// or the loss and its adjoint.  Inputs and outputs are the caller's case-major
// arrays; outputs may be NULL.
struct EvalCall {
  int K, Kp;
  bool backward;
  const double *va, *vm, *p, *q;  // p, q NULL: the grid's
  const int32_t* outage;
  const void *val32, *val64;      // Y_bus values in the sliced form, NULL: as built
  double *o_p, *o_q;              // backward = false
  double *loss, *d_va, *d_vm, *d_p, *d_q;
  void *Vout, *Wout;              // V and w in the layout [N][Kp], or NULL
};
int eval_launch(const dpf_ybus* y, const EvalCall& c, bool fp64, void* stream);

}  // namespace dpf
