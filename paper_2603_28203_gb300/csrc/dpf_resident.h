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
  int min_span = 1;   // fewest iterations of a launch that pay
  size_t smem = 0;
};

// Whether K cases of n buses are few (or wide) enough for the on-chip form.
// FP64 is bound by the FP64 pipe, which the streaming kernels keep busy with
// live rows only, while here a warp of 32 or 64 rows costs the same whatever it
// holds: the form pays where an iteration is mostly latency.  100 iterations,
// tests every 25, streaming / on chip in ms (152 SMs: 4 cases per CTA, 3 CTAs
// per SM, so 608 cases are one CTA per SM and 1,824 a full wave):
//   one row per lane    9 x 3,000 2.8 / 4.1  14 x 1,824 2.8 / 3.3  24 x 3,000
//     4.0 / 4.1; but 30 x 1,500 3.1 / 2.4, 30 x 5,000 7.3 / 7.0, 30 x 8,000 9.1 / 10.7
//   two rows            33 x 600 2.5 / 1.6, 33 x 1,216 3.1 / 3.8, 33 x 8,000 10.4 /
//     16.9; 64 x 900 3.8 / 2.9, 64 x 1,216 3.9 / 4.3, 64 x 1,824 5.6 / 4.4, 64 x
//     2,400 6.3 / 7.1, 64 x 3,000 7.9 / 7.1, 64 x 4,000 9.8 / 11.2
//   one CTA per case    1 x 30 1.9 / 1.0, 1 x 300 2.3 / 1.9, 150 x 300 3.5 / 1.9,
//     300 x 320 5.4 / 3.3; but 1,000 x 300 11.3 / 12.5, 1 x 700 2.5 / 3.5
// FP32 pays over the whole range (1 x 30 1.2 / 0.33, 3,000 x 2,000 17.7 / 12.7)
// but for very many cases of a grid that half fills its rows: 50 iterations,
// 14 x 100,000 3.3 / 4.1, 33 x 50,000 3.2 / 3.4, 65 x 20,000 2.7 / 2.8.
inline bool res_pays(int n, long long K, bool fp64, int sms) {
  if (!fp64) {
    const int rows = n <= 32 ? 32 : n <= RES_WARP_N ? 64 : (n + 63) / 64 * 64;
    return 100 * n >= 55 * rows || K <= (n <= RES_WARP_N ? 32768 : 16384);
  }
  if (n > RES_WARP_N) return n <= 320 && K <= 300;
  const long long wave = 12ll * sms;
  if (n <= 32) return K <= 8 * sms || (n >= 28 && K <= 3 * wave);
  return K <= 4 * sms || (n >= 48 && K <= 7 * sms) ||
         (K <= 2 * wave && 100 * n * K >= 78 * 64 * wave * ((K + wave - 1) / wave));
}

// Whether K cases of a grid with long rows pay, from its sliced form (entry
// pairs in all slices, in the longest one).  FP32: where the staged matrix, not
// the threads, limits the CTAs of an SM (ctas < ctas_free), by the padded
// entries per row times the waves of CTAs (beyond some 16 both forms grow
// alike).  50 iterations, streaming / on chip in ms: 1,000 buses + 2,000
// branches x 2,400 (134) 4.5 / 4.4, 300 + 4,800 x 600 (156) 1.5 / 1.4, x 1,000
// (260) 1.8 / 2.2, 150 + 2,400 x 1,000 (133) 1.26 / 1.21, x 2,400 (316) 2.2 / 2.4,
// 1,000 with a bus of 160 branches x 2,400 (150) 5.2 / 6.4; 100 iterations, 150
// + 5,000 x 1,000 (507) 2.7 / 5.0, a star of 300 x 1,000 (224) 5.2 / 7.2.
// FP64: a CTA's longest slice is one warp's chain, and padding costs the FP64
// pipe: a star of 300 x 1 8.0 / 10.5, 60 + 1,400 x 1 4.0 / 4.4; but 300 with a bus
// of 160 branches x 1 3.6 / 3.3, 150 + 2,400 x 1 2.1 / 1.9.
inline bool res_pays_dense(int n, long long K, bool fp64, int sms, int pairs, int longest, int ctas, int ctas_free) {
  const long long padded = 64ll * pairs;  // entries
  if (fp64) return longest <= 100 && padded <= 50ll * n;
  if (ctas >= ctas_free) return true;
  const long long per_wave = (long long)sms * ctas;
  return padded * (K < 16 * per_wave ? K : 16 * per_wave) <= 145 * per_wave * n;
}

// A launch loads and stores every case's state in strided 8- and 16-byte
// pieces, which the iterations between have to earn: with tests (or the
// caller's steps) closer than this the streaming kernels are faster.  Time of
// 48 iterations, streaming / on chip, by the iterations per launch:
//   FP32R  2,000 x 2,379  2: 8.1 / 18.7 ms  6: 7.9 / 9.6   10: 7.9 / 7.8
//          2,000 x 600    2: 2.6 / 5.0      6: 2.4 / 2.6    8: 2.4 / 2.3
//          300 x 3,000    2: 2.1 / 2.8      4: 2.0 / 1.9
//          2,000 x 1      2: 0.87 / 0.91
//   FP32   2,000 x 2,379  2: 7.7 / 11.4     4: 7.6 / 8.1    6: faster
//          2,000 x 600    2: 2.5 / 3.1      4: 2.3 / 2.3
//          100 x 2,000    2: 1.08 / 1.20    3: 0.98 / 0.97
//          30 x 8,192     1: 1.6 / 1.8 ms
inline int res_min_span(int n, int K, bool fp64, bool refined) {
  const long long e = (long long)n * K;
  if (fp64) return n > 256 && K > 100 ? 3 : 1;  // 300 x 152, 2: 4.0 / 4.2 ms
  if (n <= RES_WARP_N) return e > 100000 ? 2 : 1;
  if (K <= 300 && n <= 512) return 1;
  if (refined) return e <= 250000 ? 3 : e <= 1000000 ? 4 : e <= 1300000 ? 8 : 10;
  return K <= 300 ? 2 : e <= 250000 ? 3 : e <= 1300000 ? 4 : 6;
}

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
  int min_span = 1;  // fewest iterations of a launch that pay
  size_t smem = 0;
};
// The same for the whole-GPU form: a launch costs some 2.6 us plus 0.2 us per
// case (the schedulers' state) more than an iteration streaming.  48
// iterations, FP32: 2,500 x 64, 4: 1.09 / 1.29 ms, 12: 1.06 / 1.08; 2,500 x 20,
// 4: 0.94 / 1.03, 8: 0.89 / 0.91; 10,000 x 16, 1: 1.51 / 1.72, 2: 1.28 / 1.26.
inline int grid_min_span(int K) { return 2 + K / 5; }
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
// grid has the sliced form, one case fits the shared memory of an SM and the
// batch is faster on chip.
struct DcShape {
  bool ok = false;
  int rpt = 2;  // rows per thread
  int T = 32;   // threads
  size_t smem = 0;
};
DcShape dc_res_shape(const dpf_ybus* y, int K, bool f32);
// The same question as res_pays_dense for the DC solve (ms, streaming / on
// chip).  To 1e-4, FP32: 1,000 buses + 8,000 branches x 1,000 (137) 0.81 / 0.71, x
// 2,400 (329) 1.2 / 1.5, 1,000 + 16,000 x 600 (147) 0.69 / 0.51, x 1,000 (245) 0.83 /
// 0.86, 300 + 10,000 x 1,000 (504) 0.57 / 0.64.  To 1e-10, double-float: 300 + 4,800
// x 1,000 (260) 1.30 / 0.83, x 2,400 (623) 1.70 / 1.79, 150 + 5,000 x 1,000 (507)
// 0.73 / 0.80, 1,000 + 8,000 x 2,400 (329) 3.4 / 2.3.
inline bool dc_pays(int n, long long K, bool f32, int sms, int pairs, int ctas, int ctas_free) {
  if (ctas >= ctas_free) return true;
  const long long per_wave = (long long)sms * ctas;
  return 64ll * pairs * (K < 16 * per_wave ? K : 16 * per_wave) <= (f32 ? 225 : 450) * per_wave * n;
}
// Returns a cudaError_t.
int dc_res_launch(const dpf_ybus* y, const DcRes& c, const DcShape& sh, bool f32, void* stream);

// Whether an evaluation of K cases pays on chip.  A CTA waits for its longest
// row's warp, and FP64 warps cost the same however few rows they hold; with many
// cases the streaming kernels hide both.  us, streaming / on chip, gradient
// FP32, FP64 and (last) S_calc FP64: 300 buses, one of 160 branches x 1,000 224 /
// 179, 299 / 260, 160 / 134, x 2,400 309 / 327, 432 / 498, 218 / 245; a star of
// 300 x 1,000 261 / 264, 319 / 400, 183 / 208; of 700 x 100 365 / 206, 452 / 287,
// 243 / 157, x 1,000 479 / 735, 627 / 1100, 328 / 555; 14 buses x 100,000 461 /
// 479, 601 / 803, 287 / 344, 33 x 50,000 480 / 447, 673 / 735, 326 / 323; FP64
// gradients of 2,000 buses, one of 160 branches x 1,000 785 / 865, one of 300 x
// 600 642 / 697.  S_calc in FP32 is faster on chip throughout.
inline bool eval_pays(int n, long long K, bool fp64, bool backward, int longest) {
  if (!fp64 && !backward) return true;
  const int rows = (n + 31) / 32 * 32;
  const int most = fp64 && backward && n > 1500 ? 80000 : 120000;
  return (longest <= 64 || longest * K <= most) && (100 * n >= 55 * rows || K <= 32768);
}

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
