// Batched Newton-Raphson power flow (Alg. 2) on the GPU, for the same batches
// dpf_solve_batch takes (one Y_bus, per-case injections and one outage each):
// the comparison solver of the paper and the second half of a hybrid in which
// Alg. 1 supplies the starting point (Sec. 5.4, Sec. 6).
//
// Per Newton iteration, for every case still iterating:
//   k_nr_volt      V = |V| e^{j theta} (FP64)
//   k_nr_eval      I = Y' V, S = V conj(I), f, right-hand side -f (FP64)
//   k_nr_partial   per case and chunk of rows: partial max |f| and ||f||^2
//   k_nr_check     per case max |f|, loss, stop test (the host reads the
//                  number of cases left)
//   k_nr_assemble  the 2x2 Jacobian blocks of Alg. 2 on the filled pattern
//   k_nr_lu        block LU, left-looking, level by level of the elimination
//                  tree, with the forward substitution L y = -f folded into
//                  the same level pass, then U dx = y back down the tree; one
//                  CTA per tile of cases, which syncs only its own threads:
//                  the cases are independent, so no CTA waits for another
//   k_nr_update    theta += dx_theta (pv, pq), |V| += dx_|V| (pq)
// or, where few cases iterate and a case's factor fits in shared memory,
// k_nr_lu_smem in the place of the last three.
// The factor and the triangular solves run in the factor precision (FP64, or
// FP32: GB300 issues FP32 FMA at many times its FP64 rate, and a Newton step
// solved to FP32 accuracy still converges, linearly at a rate of about
// cond(J) 2^-24 once quadratic convergence has run out); the mismatch, the
// stop test and the state are FP64 in both.
#include <cuda_runtime.h>
#include <stdio.h>
#include <string.h>

#include <algorithm>
#include <new>
#include <vector>

#include "dpf_internal.h"
#include "dpf_nr.h"
#include "dpf_smem.h"

using namespace dpf;

#define CK(call)                                                                              \
  do {                                                                                        \
    cudaError_t e_ = (call);                                                                  \
    if (e_ != cudaSuccess)                                                                    \
      return fail(e_ == cudaErrorMemoryAllocation ? DPF_E_OOM : DPF_E_CUDA, "%s: %s (%s:%d)", \
                  #call, cudaGetErrorString(e_), __FILE__, __LINE__);                         \
  } while (0)

#define CKLAUNCH()                                                                            \
  do {                                                                                        \
    cudaError_t e_ = cudaGetLastError();                                                      \
    if (e_ != cudaSuccess)                                                                    \
      return fail(DPF_E_CUDA, "kernel launch: %s (%s:%d)", cudaGetErrorString(e_), __FILE__, \
                  __LINE__);                                                                  \
  } while (0)

#define TRY(x)                   \
  do {                           \
    int s_ = (x);                \
    if (s_ != DPF_OK) return s_; \
  } while (0)

namespace {

constexpr uint8_t NR_PQ = 0, NR_SLACK = 2;  // bus types (pv = 1)
constexpr int NR_THREADS = 512;  // of k_nr_lu in FP32; half in FP64
constexpr int NR_SMEM_THREADS = 512;
constexpr int NR_CHUNKS = 16;  // row chunks of the per-case reduction

// 2x2 block: rows (P, Q), columns (theta, |V|), row-major.
template <class T>
struct alignas(4 * sizeof(T)) Blk {
  T a, b, c, d;
};

template <class T>
__device__ __forceinline__ Blk<T> ldb(const Blk<T>* p) {
  return *p;
}
template <>
__device__ __forceinline__ Blk<double> ldb(const Blk<double>* p) {
  const double2 u = reinterpret_cast<const double2*>(p)[0], v = reinterpret_cast<const double2*>(p)[1];
  return Blk<double>{u.x, u.y, v.x, v.y};
}
template <class T>
__device__ __forceinline__ void stb(Blk<T>* p, const Blk<T>& v) {
  *p = v;
}
template <>
__device__ __forceinline__ void stb(Blk<double>* p, const Blk<double>& v) {
  reinterpret_cast<double2*>(p)[0] = make_double2(v.a, v.b);
  reinterpret_cast<double2*>(p)[1] = make_double2(v.c, v.d);
}

// acc -= x y
template <class T>
__device__ __forceinline__ void msub(Blk<T>& acc, const Blk<T>& x, const Blk<T>& y) {
  acc.a = fma(-x.a, y.a, fma(-x.b, y.c, acc.a));
  acc.b = fma(-x.a, y.b, fma(-x.b, y.d, acc.b));
  acc.c = fma(-x.c, y.a, fma(-x.d, y.c, acc.c));
  acc.d = fma(-x.c, y.b, fma(-x.d, y.d, acc.d));
}
template <class T>
__device__ __forceinline__ Blk<T> mul(const Blk<T>& x, const Blk<T>& y) {
  return Blk<T>{fma(x.a, y.a, x.b * y.c), fma(x.a, y.b, x.b * y.d), fma(x.c, y.a, x.d * y.c),
                fma(x.c, y.b, x.d * y.d)};
}
// inverse of a 2x2 block; false if it is singular (or not finite)
template <class T>
__device__ __forceinline__ bool inv2(const Blk<T>& m, Blk<T>& r) {
  const T det = fma(m.a, m.d, -m.b * m.c);
  const T id = T(1) / det;
  r = Blk<T>{m.d * id, -m.b * id, -m.c * id, m.a * id};
  return det != T(0) && isfinite(id);
}

__device__ __forceinline__ double2 cmul(double2 x, double2 y) {
  return make_double2(fma(x.x, y.x, -x.y * y.y), fma(x.x, y.y, x.y * y.x));
}
__device__ __forceinline__ double2 cconj(double2 x) { return make_double2(x.x, -x.y); }
__device__ __forceinline__ double2 csub(double2 x, double2 y) { return make_double2(x.x - y.x, x.y - y.y); }

struct NrArgs {
  int N, K, Kp, C;
  double va_slack, tol, inv_m;
  int max_iter;
  // grid (device, internal order)
  const int32_t* rp;
  const int32_t* ycol;
  const double2* yval;
  const uint8_t* type;
  const double* p64;
  const double* q64;
  const double* vmset;
  const int32_t* perm;
  // schedule
  const int32_t* order;
  const int32_t* rank;
  const int32_t* frp;
  const int32_t* fcol;
  const int32_t* fdiag;
  const int32_t* ymap;
  int n_levels;
  const int32_t* lvl_ptr;
  const int4* targets;
  const int2* pairs;
  const int32_t* rlvl_ptr;
  const int4* rows;
  int64_t npos;
  const uint4* sstream;  // schedule of the shared-memory form (k_nr_lu_smem)
  const int2* schunk;
  const uint4* sent;
  const uint4* sdiag;
  int n_ent, n_chunk, chunk_units, ring_bytes;
  // state [N][Kp]
  double* th;
  double* vm;
  double2* V;
  double2* U;    // e^{j theta}: V = |V| U
  double2* I;
  double2* X;    // right-hand side / solution, by elimination step
  double* Ps;    // per-case specification or NULL
  double* Qs;
  void* F;       // [npos][Kp] blocks
  void* Dinv;    // [N][Kp] blocks
  // per case
  int32_t* of;
  int32_t* ot;
  double2* yff;
  double2* yft;
  double2* ytt;
  int32_t* active;
  int32_t* status;
  int32_t* iters;
  int32_t* bad;
  double* maxmis;
  double* loss;
  int32_t* n_active;
  double* pmax;  // [NR_CHUNKS][Kp] partials of the stop test
  double* psum;
  double* maxmis0;  // per case: max |f| and loss of the start
  double* loss0;
  int first;        // this evaluation is of the start
};

// Per case: outage data (pi-model block of the removed branch), state flags.
__global__ void k_nr_init(NrArgs a, const int32_t* __restrict__ outage, const int32_t* __restrict__ br_f,
                          const int32_t* __restrict__ br_t, const double* __restrict__ br_r,
                          const double* __restrict__ br_x, const double* __restrict__ br_bch,
                          const double* __restrict__ br_tap) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= a.Kp) return;
  a.active[k] = k < a.K ? 1 : 0;
  a.status[k] = DPF_CASE_MAX_ITER;
  a.iters[k] = 0;
  a.bad[k] = 0;
  a.maxmis[k] = 0.0;
  a.loss[k] = 0.0;
  const int ell = (k < a.K && outage) ? outage[k] : -1;
  if (ell < 0) {
    a.of[k] = -1;
    a.ot[k] = -1;
    return;
  }
  const double r = br_r[ell], x = br_x[ell], bch = br_bch[ell];
  const double tau = br_tap[ell] == 0.0 ? 1.0 : br_tap[ell];
  const double d = r * r + x * x, gs = r / d, bs = -x / d, t2 = tau * tau;
  a.of[k] = br_f[ell];
  a.ot[k] = br_t[ell];
  a.yff[k] = make_double2(gs / t2, (bs + 0.5 * bch) / t2);
  a.yft[k] = make_double2(-gs / tau, -bs / tau);
  a.ytt[k] = make_double2(gs, bs + 0.5 * bch);
}

// Inputs to the internal layout: start (flat or given, set-points enforced)
// and per-case specifications.
__global__ void k_nr_in(NrArgs a, const double* __restrict__ va_in, const double* __restrict__ vm_in,
                        const double* __restrict__ p_in, const double* __restrict__ q_in,
                        const double* __restrict__ vs_in, int flat) {
  const size_t n = (size_t)a.N * a.Kp;
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < n; e += (size_t)gridDim.x * blockDim.x) {
    const int i = (int)(e / a.Kp), k = (int)(e % a.Kp);
    const uint8_t t = __ldg(a.type + i);
    double th = 0.0, vm = 1.0;
    if (k < a.K) {
      const size_t u = (size_t)k * a.N + __ldg(a.perm + i);
      const double vs = vs_in ? vs_in[u] : __ldg(a.vmset + i);
      if (a.Ps) {
        a.Ps[e] = p_in[u];
        a.Qs[e] = q_in[u];
      }
      if (!flat) {
        th = va_in[u];
        vm = vm_in[u];
      }
      if (t == NR_SLACK) th = a.va_slack;
      if (t != NR_PQ) vm = vs;
    }
    a.th[e] = th;
    a.vm[e] = vm;
  }
}

__global__ void k_nr_volt(NrArgs a) {
  const size_t n = (size_t)a.N * a.Kp;
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < n; e += (size_t)gridDim.x * blockDim.x) {
    if (!a.active[e % a.Kp]) continue;
    double s, c;
    sincos(a.th[e], &s, &c);
    a.U[e] = make_double2(c, s);
    a.V[e] = make_double2(a.vm[e] * c, a.vm[e] * s);
  }
}

// Currents, power, mismatch f = [P_calc - P (pv, pq); Q_calc - Q (pq)] and
// the right-hand side -f by elimination step (0 for the identity rows).
__global__ void k_nr_eval(NrArgs a) {
  const size_t n = (size_t)a.N * a.Kp, Kp = a.Kp;
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < n; e += (size_t)gridDim.x * blockDim.x) {
    const int i = (int)(e / Kp), k = (int)(e % Kp);
    if (!a.active[k]) continue;
    double2 cur = make_double2(0.0, 0.0);
    const int p1 = __ldg(a.rp + i + 1);
    for (int p = __ldg(a.rp + i); p < p1; ++p) {
      const double2 y = __ldg(a.yval + p), v = a.V[(size_t)__ldg(a.ycol + p) * Kp + k];
      cur.x = fma(y.x, v.x, fma(-y.y, v.y, cur.x));
      cur.y = fma(y.x, v.y, fma(y.y, v.x, cur.y));
    }
    const int of = a.of[k], ot = a.ot[k];
    if (i == of || i == ot) {  // the outaged branch's share leaves Y_bus
      const double2 vf = a.V[(size_t)of * Kp + k], vt = a.V[(size_t)ot * Kp + k];
      const double2 d = (i == of) ? cmul(a.yff[k], vf) : cmul(a.yft[k], vf);
      const double2 d2 = (i == of) ? cmul(a.yft[k], vt) : cmul(a.ytt[k], vt);
      cur = csub(csub(cur, d), d2);
    }
    const double2 v = a.V[e];
    const double2 s = cmul(v, cconj(cur));
    const uint8_t t = __ldg(a.type + i);
    const double ps = a.Ps ? a.Ps[e] : __ldg(a.p64 + i), qs = a.Ps ? a.Qs[e] : __ldg(a.q64 + i);
    const double fp = (t != NR_SLACK) ? s.x - ps : 0.0;
    const double fq = (t == NR_PQ) ? s.y - qs : 0.0;
    a.I[e] = cur;
    a.X[(size_t)__ldg(a.rank + i) * Kp + k] = make_double2(-fp, -fq);
  }
}

// Per case and chunk of rows (32 cases x 8 row groups per CTA, fixed
// summation order): partial max |f| (NaN if any entry is NaN) and partial
// ||f||^2 from the right-hand side -f.  The maximum is taken on the bits of
// |f|, which order as the values do and put NaN above infinity: an FP64
// comparison holds the FP64 pipe as long as an FMA.
__device__ __forceinline__ unsigned long long abs_bits(double x) {
  return (unsigned long long)__double_as_longlong(x) & 0x7fffffffffffffffULL;
}
__device__ __forceinline__ double max_of_bits(unsigned long long m) {
  return __longlong_as_double(m > 0x7ff0000000000000ULL ? 0x7ff8000000000000LL : (long long)m);
}
__global__ void __launch_bounds__(256) k_nr_partial(NrArgs a) {
  __shared__ unsigned long long smax[8][32];
  __shared__ double ssum[8][32];
  const int lane = threadIdx.x & 31, g = threadIdx.x >> 5;
  const int k = blockIdx.x * 32 + lane;
  const bool on = k < a.K && a.active[k];
  const int rpc = (a.N + NR_CHUNKS - 1) / NR_CHUNKS;
  const int r0 = blockIdx.y * rpc, r1 = min(a.N, r0 + rpc);
  unsigned long long mx = 0;
  double sm = 0.0;
  if (on) {
#pragma unroll 4
    for (int r = r0 + g; r < r1; r += 8) {
      const double2 x = a.X[(size_t)r * a.Kp + k];
      mx = max(mx, max(abs_bits(x.x), abs_bits(x.y)));
      sm = fma(x.x, x.x, fma(x.y, x.y, sm));
    }
  }
  smax[g][lane] = mx;
  ssum[g][lane] = sm;
  __syncthreads();
  if (g != 0 || !on) return;
  mx = 0;
  sm = 0.0;
  for (int q = 0; q < 8; ++q) {
    mx = max(mx, smax[q][lane]);
    sm += ssum[q][lane];
  }
  a.pmax[(size_t)blockIdx.y * a.Kp + k] = max_of_bits(mx);
  a.psum[(size_t)blockIdx.y * a.Kp + k] = sm;
}

// Per case: max |f|, loss (1/m) ||f||^2 from the chunks' partials (fixed
// order) and the stop test of Alg. 2.
__global__ void k_nr_check(NrArgs a) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= a.K || !a.active[k]) return;
  double mx = 0.0, sm = 0.0;
  bool nan = false;
  for (int c = 0; c < NR_CHUNKS; ++c) {
    const double m = a.pmax[(size_t)c * a.Kp + k];
    nan = nan || !(m == m);
    mx = fmax(mx, m);
    sm += a.psum[(size_t)c * a.Kp + k];
  }
  if (nan) mx = __longlong_as_double(0x7ff8000000000000LL);
  a.maxmis[k] = mx;
  a.loss[k] = sm * a.inv_m;
  if (a.first) {
    a.maxmis0[k] = mx;
    a.loss0[k] = sm * a.inv_m;
  }
  if (a.bad[k] || nan || isinf(mx)) {
    a.status[k] = DPF_CASE_DIVERGED;
    a.active[k] = 0;
  } else if (mx <= a.tol) {
    a.status[k] = DPF_CASE_CONVERGED;
    a.active[k] = 0;
  } else if (a.iters[k] >= a.max_iter) {
    a.status[k] = DPF_CASE_MAX_ITER;
    a.active[k] = 0;
  } else {
    a.iters[k] += 1;  // a Newton step follows
    atomicAdd(a.n_active, 1);
  }
}

// Jacobian blocks (Alg. 2) at every position of the filled pattern, with
// u = e^{j theta} (so V = |V| u) and W = V_i conj(Y'_ij u_j):
//   i != j: dS_i/dtheta_j = -j |V|_j W,        dS_i/d|V|_j = W
//   i == j: dS_i/dtheta_i = j (S_i - |V|_i W), dS_i/d|V|_i = u_i conj(I_i) + W
// (the element rules of Alg. 2 with T = V_i conj(Y'_ij V_j) = |V|_j W; the
// division by |V|_j cancels, and none is left: an FP64 divide costs many
// issue slots here).  Computed in the factor's precision T (the FP64 state
// rounded once); rows P = Re, Q = Im; equations and unknowns Alg. 2 leaves
// out are zeroed, with a 1 on the diagonal.  Fill positions start at 0.  One
// thread per (block row, case) walks the row's positions.
template <class T>
struct Cx {
  T x, y;
};
template <class T>
__device__ __forceinline__ Cx<T> cx(double2 v) {
  return Cx<T>{(T)v.x, (T)v.y};
}
template <class T>
__device__ __forceinline__ Cx<T> mulc(Cx<T> a, Cx<T> b) {  // a conj(b)
  return Cx<T>{fma(a.x, b.x, a.y * b.y), fma(a.y, b.x, -a.x * b.y)};
}
template <class T>
__device__ __forceinline__ Cx<T> mul(Cx<T> a, Cx<T> b) {
  return Cx<T>{fma(a.x, b.x, -a.y * b.y), fma(a.x, b.y, a.y * b.x)};
}

// The block of bus pair (i, j) of case k with Y_bus value y: vi = V_i,
// uj = e^{j theta_j}, vmj = |V|_j, ii = I_i (read where i == j), bus types.
template <class T>
__device__ __forceinline__ Blk<T> jac_block(const NrArgs& a, int i, int j, double2 y, int k, int of, int ot, Cx<T> vi,
                                            Cx<T> uj, T vmj, Cx<T> ii, int ti, int tj) {
  if (of >= 0) {
    if (i == of && j == of) y = csub(y, a.yff[k]);
    else if (i == ot && j == ot) y = csub(y, a.ytt[k]);
    else if ((i == of && j == ot) || (i == ot && j == of)) y = csub(y, a.yft[k]);
  }
  const Cx<T> w = mulc(vi, mul(cx<T>(y), uj));
  T ba, bb, bc, bd;
  if (i != j) {
    ba = vmj * w.y;
    bc = -vmj * w.x;
    bb = w.x;
    bd = w.y;
  } else {
    const Cx<T> si = mulc(vi, ii);   // S_i
    const Cx<T> sdi = mulc(uj, ii);  // S_i / |V|_i
    ba = fma(vmj, w.y, -si.y);
    bc = fma(-vmj, w.x, si.x);
    bb = sdi.x + w.x;
    bd = sdi.y + w.y;
  }
  const bool rp = ti != NR_SLACK, rq = ti == NR_PQ, ct = tj != NR_SLACK, cv = tj == NR_PQ;
  Blk<T> b;
  b.a = (rp && ct) ? ba : T(0);
  b.b = (rp && cv) ? bb : T(0);
  b.c = (rq && ct) ? bc : T(0);
  b.d = (rq && cv) ? bd : T(0);
  if (i == j) {
    if (!rp) b.a = T(1);
    if (!rq) b.d = T(1);
  }
  return b;
}

// One block row of case k: its positions' blocks to dst[q * stride], with
// jac_block's arithmetic (called from here it cost the FP64 solve 2%).
template <class T>
__device__ __forceinline__ void assemble_row(const NrArgs& a, int r, int k, Blk<T>* __restrict__ dst, size_t stride) {
  const size_t Kp = a.Kp;
  const double2* __restrict__ U = a.U;
  const double* __restrict__ VM = a.vm;
  const int i = __ldg(a.order + r);
  const size_t ei = (size_t)i * Kp + k;
  const Cx<T> vi = cx<T>(a.V[ei]), ii = cx<T>(a.I[ei]);
  const Cx<T> si = mulc(vi, ii);             // S_i
  const Cx<T> sdi = mulc(cx<T>(U[ei]), ii);  // S_i / |V|_i
  const uint8_t ti = __ldg(a.type + i);
  const bool rp = ti != NR_SLACK, rq = ti == NR_PQ;
  const int of = a.of[k], ot = a.ot[k];
  const int q1 = __ldg(a.frp + r + 1);
  for (int q = __ldg(a.frp + r); q < q1; ++q) {
    const int j = __ldg(a.order + __ldg(a.fcol + q));
    const int yp = __ldg(a.ymap + q);
    Blk<T> b{T(0), T(0), T(0), T(0)};
    if (yp >= 0) {
      double2 y = __ldg(a.yval + yp);
      if (of >= 0) {
        if (i == of && j == of) y = csub(y, a.yff[k]);
        else if (i == ot && j == ot) y = csub(y, a.ytt[k]);
        else if ((i == of && j == ot) || (i == ot && j == of)) y = csub(y, a.yft[k]);
      }
      const size_t ej = (size_t)j * Kp + k;
      const Cx<T> w = mulc(vi, mul(cx<T>(y), cx<T>(U[ej])));
      const T vmj = (T)VM[ej];
      T ba, bb, bc, bd;
      if (i != j) {
        ba = vmj * w.y;
        bc = -vmj * w.x;
        bb = w.x;
        bd = w.y;
      } else {
        ba = fma(vmj, w.y, -si.y);
        bc = fma(-vmj, w.x, si.x);
        bb = sdi.x + w.x;
        bd = sdi.y + w.y;
      }
      const uint8_t tj = __ldg(a.type + j);
      const bool ct = tj != NR_SLACK, cv = tj == NR_PQ;
      b.a = (rp && ct) ? ba : T(0);
      b.b = (rp && cv) ? bb : T(0);
      b.c = (rq && ct) ? bc : T(0);
      b.d = (rq && cv) ? bd : T(0);
      if (i == j) {
        if (!rp) b.a = T(1);
        if (!rq) b.d = T(1);
      }
    }
    stb(dst + (size_t)q * stride, b);
  }
}

template <class T>
__global__ void k_nr_assemble(NrArgs a) {
  Blk<T>* F = static_cast<Blk<T>*>(a.F);
  const size_t n = (size_t)a.N * a.Kp, Kp = a.Kp;
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < n; e += (size_t)gridDim.x * blockDim.x) {
    const int r = (int)(e / Kp), k = (int)(e % Kp);
    if (a.active[k]) assemble_row(a, r, k, F + k, Kp);
  }
}

// Right-hand side / solution entries: FP64 pairs in global memory, pairs of
// the factor's type in shared memory.
template <class T>
__device__ __forceinline__ Cx<T> ldx(const double2* p) {
  const double2 v = *p;
  return Cx<T>{(T)v.x, (T)v.y};
}
template <class T>
__device__ __forceinline__ Cx<T> ldx(const Cx<T>* p) {
  return *p;
}
template <class T>
__device__ __forceinline__ void stx(double2* p, Cx<T> v) {
  *p = make_double2((double)v.x, (double)v.y);
}
template <class T>
__device__ __forceinline__ void stx(Cx<T>* p, Cx<T> v) {
  *p = v;
}

// acc minus the updates of one target: sum over its pairs of L(i,k) U(k,j)
template <class T>
__device__ __forceinline__ void apply_pairs(Blk<T>& acc, const Blk<T>* F, size_t fs, const int2* __restrict__ pairs,
                                            int p, int p1) {
  for (; p + 1 < p1; p += 2) {
    const int2 q0 = __ldg(pairs + p), q1 = __ldg(pairs + p + 1);
    const Blk<T> l0 = ldb(F + (size_t)q0.x * fs), u0 = ldb(F + (size_t)q0.y * fs);
    const Blk<T> l1 = ldb(F + (size_t)q1.x * fs), u1 = ldb(F + (size_t)q1.y * fs);
    msub(acc, l0, u0);
    msub(acc, l1, u1);
  }
  if (p < p1) {
    const int2 q0 = __ldg(pairs + p);
    msub(acc, ldb(F + (size_t)q0.x * fs), ldb(F + (size_t)q0.y * fs));
  }
}

// Block LU of one case and both triangular solves, in one pass per level of
// the elimination tree (leaves first) and one back down.  At level l every
// target position (i, j) whose pivot p = min(i, j) sits on level l takes
// its updates -L(i,k) U(k,j) from earlier pivots (all on lower levels, final
// after the previous level's barrier); an L position also forms its pivot's
// updated diagonal block D_p itself (a short list for this kind of grid) and
// stores L(i,p) = A(i,p) D_p^-1, so one barrier per level suffices; the
// diagonal target of row r stores D_r^-1 and the forward substitution
// y_r = b_r - sum_c L(r,c) y_c (its L columns are descendants: final).  The
// assembled diagonal blocks are only read.  Then, root first,
// x_r = D_r^-1 (y_r - sum_c U(r,c) x_c), in place in X.  Block q of the case
// is F[q * fs], the inverse diagonal of row r Dv[r * ds], its right-hand
// side X[r * xs]; this thread takes every S-th target from `slot` on.
template <class T, class XT>
__device__ __forceinline__ void lu_levels(const NrArgs& a, Blk<T>* F, size_t fs, Blk<T>* Dv, size_t ds, XT* X,
                                          size_t xs, int slot, int S, bool on, int32_t* bad) {
  for (int l = 0; l < a.n_levels; ++l) {
    const int t0 = __ldg(a.lvl_ptr + l), t1 = __ldg(a.lvl_ptr + l + 1);
    int t = t0 + slot;
    int4 na, nb;  // the schedule entry of this slot's next target, fetched one step ahead
    if (on && t < t1) {
      na = __ldg(a.targets + 2 * t);
      nb = __ldg(a.targets + 2 * t + 1);
    }
    if (on)
      for (; t < t1; t += S) {
        const int4 ta = na, tb = nb;
        if (t + S < t1) {
          na = __ldg(a.targets + 2 * (t + S));
          nb = __ldg(a.targets + 2 * (t + S) + 1);
        }
        Blk<T> acc = ldb(F + (size_t)ta.x * fs);
        apply_pairs(acc, F, fs, a.pairs, ta.y, ta.z);
        if (ta.w == NR_U) {
          stb(F + (size_t)ta.x * fs, acc);
          continue;
        }
        Blk<T> d = acc;
        if (ta.w == NR_L) {
          d = ldb(F + (size_t)tb.x * fs);
          apply_pairs(d, F, fs, a.pairs, tb.y, tb.z);
        }
        Blk<T> di;
        const bool ok = inv2(d, di);
        if (ta.w == NR_L) {
          stb(F + (size_t)ta.x * fs, mul(acc, di));
          continue;
        }
        if (!ok) *bad = 1;
        const int r = tb.w;
        stb(Dv + (size_t)r * ds, di);
        Cx<T> y = ldx<T>(X + (size_t)r * xs);
        const int q1 = ta.x;  // the row's L positions (from tb.x) precede its diagonal
        for (int q = tb.x; q < q1; ++q) {
          const Blk<T> m = ldb(F + (size_t)q * fs);
          const Cx<T> x = ldx<T>(X + (size_t)__ldg(a.fcol + q) * xs);
          y.x = fma(-m.a, x.x, fma(-m.b, x.y, y.x));
          y.y = fma(-m.c, x.x, fma(-m.d, x.y, y.y));
        }
        stx(X + (size_t)r * xs, y);
      }
    __syncthreads();
  }
  for (int l = a.n_levels - 1; l >= 0; --l) {
    const int t0 = __ldg(a.rlvl_ptr + l), t1 = __ldg(a.rlvl_ptr + l + 1);
    if (on)
      for (int t = t0 + slot; t < t1; t += S) {
        const int4 rw = __ldg(a.rows + t);  // {r, first U position, end of row}
        const int r = rw.x;
        Cx<T> y = ldx<T>(X + (size_t)r * xs);
        for (int q = rw.y; q < rw.z; ++q) {
          const Blk<T> m = ldb(F + (size_t)q * fs);
          const Cx<T> x = ldx<T>(X + (size_t)__ldg(a.fcol + q) * xs);
          y.x = fma(-m.a, x.x, fma(-m.b, x.y, y.x));
          y.y = fma(-m.c, x.x, fma(-m.d, x.y, y.y));
        }
        const Blk<T> di = ldb(Dv + (size_t)r * ds);
        stx(X + (size_t)r * xs, Cx<T>{fma(di.a, y.x, di.b * y.y), fma(di.c, y.x, di.d * y.y)});
      }
    __syncthreads();
  }
}

// Global-memory form: C cases per CTA are the lanes (their blocks adjacent),
// the remaining thread index is the slot.
template <class T>
__global__ void __launch_bounds__(sizeof(T) == 8 ? NR_THREADS / 2 : NR_THREADS) k_nr_lu(NrArgs a) {
  const int lane = threadIdx.x & (a.C - 1), slot = threadIdx.x / a.C, S = blockDim.x / a.C;
  const int k = blockIdx.x * a.C + lane;
  const bool on = k < a.K && a.active[k];
  if (!__syncthreads_or(on)) return;  // no case of this tile is iterating
  const size_t Kp = a.Kp;
  lu_levels(a, static_cast<Blk<T>*>(a.F) + k, Kp, static_cast<Blk<T>*>(a.Dinv) + k, Kp, a.X + k, Kp, slot, S, on,
            a.bad + k);
}

// Schedule of the shared-memory form: one stream of chunks, in 16-byte units.
// A chunk is a set of targets of one level, one per thread at most: first a
// record per target, then their lists in groups of 4 entries, filled up with
// the zero block (position npos) and the zero solution entry (row N), which
// change no bit of a sum.  Positions and rows are 16-bit fields (what fits in
// shared memory has fewer).
//   record {pos | x2 << 16, offset of its list in the chunk, groups, kind}
//   NR_U, NR_DIAG, NR_L: updates {L(i,k) | U(k,j) << 16} of position pos; an L
//     target is multiplied by its pivot's inverse at x2 after a barrier
//   NR_FWD: row x2's forward substitution {L position | column << 16}
//   NR_BACK: row x2's back substitution {U position | column << 16}, its
//     inverse diagonal at pos
//   chunk {first unit, targets | units to stage << 10, has L targets: bit 31};
//     no units: larger than a stage, read in place (a pivot with long lists)
// Block and vector targets don't share a warp.  A U target without updates has
// no record.  The pivots of a chunk are whole; one larger than a stage is
// split with its diagonal first.
//   entry {position, i | j << 16, types, Y_bus entry}: blocks off the diagonal
//   by Y_bus entry, diag {position, Y_bus entry, type} by bus
enum { NR_FWD = 3, NR_BACK = 4, NR_NONE = 5 };
constexpr int NR_STAGES = 4;  // chunks in shared memory: this one, the next ones on their way

__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

template <class T>
__device__ __forceinline__ void upd_group(Blk<T>& acc, const Blk<T>* F, uint4 g) {
  const Blk<T> l0 = ldb(F + (g.x & 0xffffu)), u0 = ldb(F + (g.x >> 16));
  const Blk<T> l1 = ldb(F + (g.y & 0xffffu)), u1 = ldb(F + (g.y >> 16));
  const Blk<T> l2 = ldb(F + (g.z & 0xffffu)), u2 = ldb(F + (g.z >> 16));
  const Blk<T> l3 = ldb(F + (g.w & 0xffffu)), u3 = ldb(F + (g.w >> 16));
  msub(acc, l0, u0);
  msub(acc, l1, u1);
  msub(acc, l2, u2);
  msub(acc, l3, u3);
}
template <class T>
__device__ __forceinline__ void sub_x(Cx<T>& y, const Blk<T>& m, const Cx<T>& x) {
  y.x = fma(-m.a, x.x, fma(-m.b, x.y, y.x));
  y.y = fma(-m.c, x.x, fma(-m.d, x.y, y.y));
}
template <class T>
__device__ __forceinline__ void sub_group(Cx<T>& y, const Blk<T>* F, const Cx<T>* X, uint4 g) {
  const Blk<T> m0 = ldb(F + (g.x & 0xffffu)), m1 = ldb(F + (g.y & 0xffffu));
  const Blk<T> m2 = ldb(F + (g.z & 0xffffu)), m3 = ldb(F + (g.w & 0xffffu));
  const Cx<T> x0 = X[g.x >> 16], x1 = X[g.y >> 16], x2 = X[g.z >> 16], x3 = X[g.w >> 16];
  sub_x(y, m0, x0);
  sub_x(y, m1, x1);
  sub_x(y, m2, x2);
  sub_x(y, m3, x3);
}

// One target (see the schedule above); true: `acc` is an L target's, to be
// multiplied by the inverse at position `x2`.
template <class T>
__device__ __forceinline__ bool smem_target(const uint4* __restrict__ p, uint4 r, uint4 g, Blk<T>* F, Cx<T>* X,
                                            Blk<T>& acc, int& pos, int& x2, int* bad) {
  const int n = (int)r.z, kind = (int)r.w;
  pos = r.x & 0xffffu;
  x2 = r.x >> 16;
  if (kind <= NR_L) {
    acc = ldb(F + pos);
    for (int i = 0; i < n; ++i) {
      const uint4 c = g;
      if (i + 1 < n) g = p[i + 1];
      upd_group(acc, F, c);
    }
    if (kind == NR_L) return true;
    if (kind == NR_DIAG) {
      Blk<T> di;
      if (!inv2(acc, di)) *bad = 1;
      acc = di;
    }
    stb(F + pos, acc);
  } else {
    Cx<T> y = X[x2];
    for (int i = 0; i < n; ++i) {
      const uint4 c = g;
      if (i + 1 < n) g = p[i + 1];
      sub_group(y, F, X, c);
    }
    if (kind == NR_BACK) {
      const Blk<T> d = ldb(F + pos);
      y = Cx<T>{fma(d.a, y.x, d.b * y.y), fma(d.c, y.x, d.d * y.y)};
    }
    X[x2] = y;
  }
  return false;
}

// Shared-memory form, for grids whose factor of one case fits: one CTA per
// case assembles its Jacobian straight into shared memory (the factor never
// goes to HBM), factorises and solves there by the levels of lu_levels (same
// sums in the same order: same bits), and updates theta and |V|.
//
// What bounds it is latency: a chain of 143 chunks for a 2,000-bus grid, most
// of the upper ones a warp's worth of targets, 1,440 cycles each (a target's
// loads from shared memory, the pivot's inverse, two barriers).  So the
// schedule arrives by cp.async some chunks ahead and never costs a trip to
// L2; a pivot's diagonal is updated and inverted once, not in each of its L
// targets; block and vector targets sit in different warps and don't take
// turns.  One case of 2,000 buses: 390 us with the schedule read from L2 by
// each thread and the diagonal updated per L target, 135 us so (assembly 29).
// 384 threads take 2% longer, 256 8%, 768 6%; 8 stages of 256 units 11%.
template <class T>
__global__ void __launch_bounds__(NR_SMEM_THREADS, 1) k_nr_lu_smem(NrArgs a) {
  extern __shared__ __align__(16) unsigned char nr_smem[];
  __shared__ int s_bad;
  const int k = blockIdx.x, tid = threadIdx.x, S = blockDim.x, N = a.N, C = a.n_chunk;
  if (!a.active[k]) return;  // the same for the whole CTA
  const int npos = (int)a.npos;
  Blk<T>* F = reinterpret_cast<Blk<T>*>(nr_smem);
  unsigned char* ring = reinterpret_cast<unsigned char*>(F + npos + 1);
  Cx<T>* X = reinterpret_cast<Cx<T>*>(ring + a.ring_bytes);
  int2* chunk = reinterpret_cast<int2*>(X + N + 1);
  const size_t Kp = a.Kp;

  // V in the place of X, e^{j theta} and |V| in that of the stages; four
  // buses' loads in flight
  Cx<T>* Us = reinterpret_cast<Cx<T>*>(ring);
  T* Ms = reinterpret_cast<T*>(Us + N);
  for (int i0 = tid; i0 < N; i0 += 4 * S) {
    double2 u[4], v[4];
    double m[4];
#pragma unroll
    for (int z = 0; z < 4; ++z) {
      const size_t e = (size_t)min(i0 + z * S, N - 1) * Kp + k;
      u[z] = a.U[e];
      v[z] = a.V[e];
      m[z] = a.vm[e];
    }
#pragma unroll
    for (int z = 0; z < 4; ++z)
      if (i0 + z * S < N) {
        Us[i0 + z * S] = cx<T>(u[z]);
        X[i0 + z * S] = cx<T>(v[z]);
        Ms[i0 + z * S] = (T)m[z];
      }
  }
  for (int q = tid; q <= npos; q += S) stb(F + q, Blk<T>{T(0), T(0), T(0), T(0)});
  for (int c = tid; c < C; c += S) chunk[c] = __ldg(a.schunk + c);
  if (tid == 0) {
    X[N] = Cx<T>{T(0), T(0)};
    s_bad = 0;
  }
  __syncthreads();
  {
    const int of = a.of[k], ot = a.ot[k];
    for (int q0 = tid; q0 < a.n_ent; q0 += 4 * S) {
      uint4 en[4];
      double2 y[4];
#pragma unroll
      for (int z = 0; z < 4; ++z) en[z] = __ldg(a.sent + min(q0 + z * S, a.n_ent - 1));
#pragma unroll
      for (int z = 0; z < 4; ++z) y[z] = __ldg(a.yval + en[z].w);
#pragma unroll
      for (int z = 0; z < 4; ++z)
        if (q0 + z * S < a.n_ent) {
          const int i = en[z].y & 0xffffu, j = en[z].y >> 16;
          stb(F + en[z].x, jac_block<T>(a, i, j, y[z], k, of, ot, X[i], Us[j], Ms[j], Cx<T>{T(0), T(0)}, en[z].z & 3,
                                        en[z].z >> 2));
        }
    }
    for (int i0 = tid; i0 < N; i0 += 4 * S) {
      uint4 dg[4];
      double2 ii[4], y[4];
#pragma unroll
      for (int z = 0; z < 4; ++z) {
        const int i = min(i0 + z * S, N - 1);
        dg[z] = __ldg(a.sdiag + i);
        ii[z] = a.I[(size_t)i * Kp + k];
      }
#pragma unroll
      for (int z = 0; z < 4; ++z) y[z] = __ldg(a.yval + dg[z].y);
#pragma unroll
      for (int z = 0; z < 4; ++z) {
        const int i = i0 + z * S;
        if (i < N)
          stb(F + dg[z].x, jac_block<T>(a, i, i, y[z], k, of, ot, X[i], Us[i], Ms[i], cx<T>(ii[z]), dg[z].z, dg[z].z));
      }
    }
  }
  __syncthreads();
  for (int r0 = tid; r0 < N; r0 += 4 * S) {
    double2 x[4];
#pragma unroll
    for (int z = 0; z < 4; ++z) x[z] = a.X[(size_t)min(r0 + z * S, N - 1) * Kp + k];
#pragma unroll
    for (int z = 0; z < 4; ++z)
      if (r0 + z * S < N) X[r0 + z * S] = cx<T>(x[z]);
  }
  uint4* stage = reinterpret_cast<uint4*>(ring);
  const int units = a.chunk_units;
  auto fetch = [&](int c, int at) {
    if (c < C) {
      const int2 ch = chunk[c];
      for (int u = tid; u < ((ch.y >> 10) & 0xffff); u += S) cp_async16(stage + at * units + u, a.sstream + ch.x + u);
    }
    cp_commit();
  };
#pragma unroll
  for (int c = 0; c < NR_STAGES - 1; ++c) fetch(c, c);
  // This thread's record of the next chunk and its list's first group are
  // read a chunk ahead: they don't depend on this chunk's results.
  const uint4 none = make_uint4(0, 0, 0, NR_NONE);
  uint4 rec = none, grp = none;
  const uint4* list = nullptr;
  auto look = [&](int2 ch, int at) {
    rec = none;
    if (tid < (ch.y & 1023)) {
      const uint4* base = ((ch.y >> 10) & 0xffff) ? stage + at * units : a.sstream + ch.x;
      rec = base[tid];
      list = base + rec.y;
      if (rec.z) grp = list[0];
    }
  };
  cp_wait<NR_STAGES - 2>();
  __syncthreads();
  int2 ch = chunk[0];
  look(ch, 0);
  int at = 0;
  for (int c = 0; c < C; ++c) {
    cp_wait<NR_STAGES - 3>();
    __syncthreads();  // chunk c + 1 has arrived; what the chunks before this one wrote is there
    int prev = at - 1, next = at + 1;
    if (prev < 0) prev = NR_STAGES - 1;
    if (next == NR_STAGES) next = 0;
    fetch(c + NR_STAGES - 1, prev);
    const uint4 r = rec, g = grp;
    const uint4* p = list;
    const int y = ch.y;
    if (c + 1 < C) {
      ch = chunk[c + 1];
      look(ch, next);
    }
    Blk<T> acc;
    int pos, x2;
    bool lower = false;
    if (r.w != NR_NONE) lower = smem_target(p, r, g, F, X, acc, pos, x2, &s_bad);
    if (y < 0) {
      __syncthreads();  // the pivots' inverses
      if (lower) stb(F + pos, mul(acc, ldb(F + x2)));
    }
    at = next;
  }
  __syncthreads();
  if (s_bad) {
    if (tid == 0) a.bad[k] = 1;
    return;
  }
  for (int r = tid; r < N; r += S) {
    const int i = __ldg(a.order + r);
    const uint8_t ty = __ldg(a.type + i);
    const size_t e = (size_t)i * Kp + k;
    if (ty != NR_SLACK) a.th[e] += (double)X[r].x;
    if (ty == NR_PQ) a.vm[e] += (double)X[r].y;
  }
}

// Shared memory the shared-memory form needs for one case: the factor, the
// stages (before the factorisation: e^{j theta} and |V|), X, the chunks.
template <class T>
size_t lu_ring_bytes(int n, int units) {
  return std::max((size_t)NR_STAGES * units * 16, ((size_t)n * 3 * sizeof(T) + 15) / 16 * 16);
}
template <class T>
size_t lu_smem_bytes(int64_t npos, int n, int units, int n_chunk) {
  return (size_t)(npos + 1) * sizeof(Blk<T>) + lu_ring_bytes<T>(n, units) + (size_t)(n + 1) * sizeof(Cx<T>) +
         (size_t)n_chunk * 8 + 64;  // 64: the static part
}

__global__ void k_nr_update(NrArgs a) {
  const size_t n = (size_t)a.N * a.Kp, Kp = a.Kp;
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < n; e += (size_t)gridDim.x * blockDim.x) {
    const int r = (int)(e / Kp), k = (int)(e % Kp);
    if (!a.active[k] || a.bad[k]) continue;
    const int i = __ldg(a.order + r);
    const uint8_t t = __ldg(a.type + i);
    const double2 dx = a.X[e];
    const size_t ei = (size_t)i * Kp + k;
    if (t != NR_SLACK) a.th[ei] += dx.x;
    if (t == NR_PQ) a.vm[ei] += dx.y;
  }
}

// Solution and per-case results to the caller's arrays (case-major, user bus
// order).  With `fallback`, a case that did not converge keeps the start the
// caller passed in va/vm, and its start's max |f| and loss are reported.
__global__ void k_nr_out(NrArgs a, double* __restrict__ va, double* __restrict__ vm, int fallback) {
  const size_t n = (size_t)a.N * a.Kp;
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < n; e += (size_t)gridDim.x * blockDim.x) {
    const int i = (int)(e / a.Kp), k = (int)(e % a.Kp);
    if (k >= a.K || (fallback && a.status[k] != DPF_CASE_CONVERGED)) continue;
    const size_t u = (size_t)k * a.N + __ldg(a.perm + i);
    va[u] = a.th[e];
    vm[u] = a.vm[e];
  }
}

__global__ void k_nr_case_out(NrArgs a, int32_t* iters, int32_t* status, double* maxmis, double* loss,
                              int fallback) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= a.K) return;
  const bool keep = fallback && a.status[k] != DPF_CASE_CONVERGED;
  if (iters) iters[k] = a.iters[k];
  if (status) status[k] = a.status[k];
  if (maxmis) maxmis[k] = keep ? a.maxmis0[k] : a.maxmis[k];
  if (loss) loss[k] = keep ? a.loss0[k] : a.loss[k];
}

template <class T>
int dalloc(T** p, size_t n) {
  *p = nullptr;
  if (n == 0) n = 1;
  cudaError_t e = cudaMalloc((void**)p, n * sizeof(T));
  if (e != cudaSuccess) {
    *p = nullptr;
    return fail(e == cudaErrorMemoryAllocation ? DPF_E_OOM : DPF_E_CUDA, "cudaMalloc(%zu bytes): %s",
                n * sizeof(T), cudaGetErrorString(e));
  }
  return DPF_OK;
}

template <class T>
void dfree(T*& p) {
  if (p) cudaFree((void*)p);
  p = nullptr;
}

template <class T>
int upload(T** dst, const std::vector<T>& src) {
  TRY(dalloc(dst, src.size()));
  if (!src.empty()) CK(cudaMemcpy(*dst, src.data(), src.size() * sizeof(T), cudaMemcpyHostToDevice));
  return DPF_OK;
}

int num_sms_nr() {
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  return sms > 0 ? sms : 1;
}

int grid_for(size_t n) { return (int)std::max<size_t>(1, std::min<size_t>((n + 255) / 256, (size_t)num_sms_nr() * 8)); }

}  // namespace

struct dpf_nr {
  const dpf_ybus* y = nullptr;
  int max_case = 0, Kp = 0;
  NrSymbolic sym;
  int64_t launches = 0;
  // schedule (device)
  int32_t *order = nullptr, *rank = nullptr, *frp = nullptr, *fcol = nullptr, *fdiag = nullptr,
          *ymap = nullptr, *lvl_ptr = nullptr, *rlvl_ptr = nullptr;
  int4* rows = nullptr;
  int4* targets = nullptr;
  int2* pairs = nullptr;
  // shared-memory form, if the grid has one
  uint4 *sstream = nullptr, *sent = nullptr, *sdiag = nullptr;  // in one allocation, sstream's
  int2* schunk = nullptr;
  int n_ent = 0, n_chunk = 0, smem_threads = 0, chunk_units = 0;
  // state
  double *th = nullptr, *vm = nullptr, *Ps = nullptr, *Qs = nullptr;
  double2 *V = nullptr, *U = nullptr, *I = nullptr, *X = nullptr;
  char* F = nullptr;
  char* Dinv = nullptr;
  int32_t *of = nullptr, *ot = nullptr, *active = nullptr, *status = nullptr, *iters = nullptr, *bad = nullptr,
          *n_active = nullptr;
  double2 *yff = nullptr, *yft = nullptr, *ytt = nullptr;
  double *maxmis = nullptr, *loss = nullptr, *pmax = nullptr, *psum = nullptr, *maxmis0 = nullptr,
         *loss0 = nullptr;
  int32_t* h_nact = nullptr;  // pinned
};

static void nr_release(dpf_nr* h) {
  dfree(h->order); dfree(h->rank); dfree(h->frp); dfree(h->fcol); dfree(h->fdiag);
  dfree(h->ymap); dfree(h->lvl_ptr); dfree(h->rlvl_ptr); dfree(h->rows); dfree(h->targets); dfree(h->pairs);
  dfree(h->sstream);
  dfree(h->th); dfree(h->vm); dfree(h->Ps); dfree(h->Qs); dfree(h->V); dfree(h->U); dfree(h->I); dfree(h->X);
  dfree(h->F); dfree(h->Dinv);
  dfree(h->of); dfree(h->ot); dfree(h->active); dfree(h->status); dfree(h->iters); dfree(h->bad);
  dfree(h->n_active); dfree(h->yff); dfree(h->yft); dfree(h->ytt); dfree(h->maxmis); dfree(h->loss); dfree(h->pmax); dfree(h->psum); dfree(h->maxmis0); dfree(h->loss0);
  if (h->h_nact) cudaFreeHost(h->h_nact);
  h->h_nact = nullptr;
}

static size_t smem_optin() {
  int dev = 0, v = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&v, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  return (size_t)v;
}

// The shared-memory form's schedule (above upd_group) from the analysis.  The
// order is free within a level: long lists come first, so that the lanes of a
// warp walk lists of like length.
static int nr_setup_smem(dpf_nr* h) {
  const NrSymbolic& s = h->sym;
  const dpf_ybus* y = h->y;
  const int n = s.n, npos = s.row_ptr[(size_t)n];
  const int S = n <= 64 ? 64 : n <= 256 ? 128 : n <= 1000 ? 256 : NR_SMEM_THREADS;
  const int units = std::min(4 * S, 512);
  const uint32_t pad_f = (uint32_t)npos | (uint32_t)npos << 16, pad_x = (uint32_t)npos | (uint32_t)n << 16;
  struct Item {
    uint32_t pos, x2, kind;
    std::vector<uint32_t> list;
  };
  auto pad = [](std::vector<uint32_t>& v, uint32_t p) {
    while (v.size() % 4) v.push_back(p);
  };
  std::vector<uint32_t> stream;
  std::vector<int2> chunks;
  auto vec = [](const Item* i) { return i->kind == NR_FWD || i->kind == NR_BACK; };
  // one chunk: block targets from the first thread on, vector targets from the next warp on
  auto emit = [&](std::vector<const Item*> its, bool staged) {
    std::stable_sort(its.begin(), its.end(), [&](const Item* a, const Item* b) {
      if (vec(a) != vec(b)) return vec(b);
      return a->list.size() > b->list.size();
    });
    static const Item none{0, 0, NR_NONE, {}};
    size_t nb = 0;
    bool lower = false;
    for (const Item* i : its) {
      nb += !vec(i);
      lower = lower || i->kind == NR_L;
    }
    if (nb < its.size()) its.insert(its.begin() + (long)nb, (32 - nb % 32) % 32, &none);
    const size_t base = stream.size();
    size_t at = its.size();
    for (const Item* i : its) {
      const uint32_t r[4] = {i->pos | i->x2 << 16, (uint32_t)at, (uint32_t)(i->list.size() / 4), i->kind};
      stream.insert(stream.end(), r, r + 4);
      at += r[2];
    }
    for (const Item* i : its) stream.insert(stream.end(), i->list.begin(), i->list.end());
    const uint32_t y = (uint32_t)its.size() | (staged ? (uint32_t)at << 10 : 0) | (lower ? 0x80000000u : 0);
    chunks.push_back(make_int2((int)(base / 4), (int)y));
  };
  // chunks of a level from its pivots (whole where they fit a stage)
  std::vector<std::vector<Item>> pivots;
  auto pack = [&] {
    std::vector<std::pair<size_t, size_t>> by_length;  // ~longest list, pivot
    for (size_t i = 0; i < pivots.size(); ++i) {
      size_t x = 0;
      for (const Item& it : pivots[i]) x = std::max(x, it.list.size());
      by_length.emplace_back(~x, i);
    }
    std::sort(by_length.begin(), by_length.end());
    const size_t most = (size_t)S - 32;  // 32: the fill between block and vector targets
    std::vector<const Item*> cur;
    size_t size = 0;
    auto flush = [&] {
      if (!cur.empty()) emit(cur, true);
      cur.clear();
      size = 0;
    };
    for (const auto& ip : by_length) {
      const std::vector<Item>& pv = pivots[ip.second];
      size_t u = pv.size();
      for (const Item& it : pv) u += it.list.size() / 4;
      if (u + 32 > (size_t)units || pv.size() > most) {
        flush();
        std::vector<const Item*> big;
        for (const Item& it : pv) big.push_back(&it);
        std::stable_sort(big.begin(), big.end(), [](const Item* a, const Item* b) {
          return (a->kind == NR_DIAG) > (b->kind == NR_DIAG);
        });
        for (size_t i = 0; i < big.size(); i += most)
          emit(std::vector<const Item*>(big.begin() + (long)i, big.begin() + (long)std::min(big.size(), i + most)), false);
        continue;
      }
      if (size + u + 32 > (size_t)units || cur.size() + pv.size() > most) flush();
      for (const Item& it : pv) cur.push_back(&it);
      size += u;
    }
    flush();
  };
  std::vector<int32_t> row_of((size_t)npos), slot((size_t)n, -1);
  for (int r = 0; r < n; ++r)
    for (int q = s.row_ptr[(size_t)r]; q < s.row_ptr[(size_t)r + 1]; ++q) row_of[(size_t)q] = r;
  for (int l = 0; l < s.n_levels; ++l) {
    pivots.clear();
    for (int t = s.lvl_ptr[(size_t)l]; t < s.lvl_ptr[(size_t)l + 1]; ++t) {
      const int32_t* w = &s.targets[(size_t)8 * t];
      Item it{(uint32_t)w[0], w[3] == NR_L ? (uint32_t)w[4] : 0, (uint32_t)w[3], {}};
      for (int p = w[1]; p < w[2]; ++p)
        it.list.push_back((uint32_t)s.pairs[2 * (size_t)p] | (uint32_t)s.pairs[2 * (size_t)p + 1] << 16);
      pad(it.list, pad_f);
      if (w[3] == NR_U && it.list.empty()) continue;
      const int p = std::min(row_of[(size_t)w[0]], s.col[(size_t)w[0]]);
      if (slot[(size_t)p] < 0) {
        slot[(size_t)p] = (int)pivots.size();
        pivots.emplace_back();
      }
      auto& pv = pivots[(size_t)slot[(size_t)p]];
      pv.push_back(std::move(it));
      if (w[3] != NR_DIAG || w[4] == w[0]) continue;
      Item fw{0, (uint32_t)w[7], NR_FWD, {}};
      for (int q = w[4]; q < w[0]; ++q) fw.list.push_back((uint32_t)q | (uint32_t)s.col[(size_t)q] << 16);
      pad(fw.list, pad_x);
      pv.push_back(std::move(fw));
    }
    pack();
  }
  for (int l = s.n_levels - 1; l >= 0; --l) {
    pivots.clear();
    for (int t = s.rlvl_ptr[(size_t)l]; t < s.rlvl_ptr[(size_t)l + 1]; ++t) {
      const int32_t* w = &s.rows[(size_t)4 * t];
      Item it{(uint32_t)s.diag[(size_t)w[0]], (uint32_t)w[0], NR_BACK, {}};
      for (int q = w[1]; q < w[2]; ++q) it.list.push_back((uint32_t)q | (uint32_t)s.col[(size_t)q] << 16);
      pad(it.list, pad_x);
      pivots.emplace_back(1, std::move(it));
    }
    pack();
  }
  if (stream.size() / 4 > 0x7fffffffu) return DPF_OK;
  // blocks by Y_bus entry, and the diagonal by bus
  std::vector<uint4> ent, dg((size_t)n);
  for (int r = 0; r < n; ++r)
    for (int q = s.row_ptr[(size_t)r]; q < s.row_ptr[(size_t)r + 1]; ++q) {
      const int yp = s.ymap[(size_t)q], i = s.order[(size_t)r], j = s.order[(size_t)s.col[(size_t)q]];
      const uint32_t ti = y->bus_type[(size_t)y->perm[(size_t)i]], tj = y->bus_type[(size_t)y->perm[(size_t)j]];
      if (yp < 0) continue;
      if (i == j) dg[(size_t)i] = make_uint4((uint32_t)q, (uint32_t)yp, ti, 0);
      else ent.push_back(make_uint4((uint32_t)q, (uint32_t)i | (uint32_t)j << 16, ti | tj << 2, (uint32_t)yp));
    }
  std::sort(ent.begin(), ent.end(), [](const uint4& a, const uint4& b) { return a.w < b.w; });
  // one allocation: the stream, entries and diagonal (16-byte units), the chunks
  const size_t ns = stream.size() / 4, ne = ent.size(), nc = chunks.size();
  std::vector<uint4> all(ns + ne + (size_t)n + (nc + 1) / 2);
  memcpy(all.data(), stream.data(), ns * 16);
  std::copy(ent.begin(), ent.end(), all.begin() + (long)ns);
  std::copy(dg.begin(), dg.end(), all.begin() + (long)(ns + ne));
  memcpy(all.data() + ns + ne + (size_t)n, chunks.data(), nc * 8);
  TRY(upload(&h->sstream, all));
  h->sent = h->sstream + ns;
  h->sdiag = h->sent + ne;
  h->schunk = reinterpret_cast<int2*>(h->sdiag + n);
  h->n_ent = (int)ent.size();
  h->n_chunk = (int)chunks.size();
  h->smem_threads = S;
  h->chunk_units = units;
  return DPF_OK;
}

static int nr_setup(dpf_nr* h) {
  const NrSymbolic& s = h->sym;
  const int n = s.n;
  const size_t npos = (size_t)s.row_ptr[n];
  TRY(upload(&h->order, s.order));
  TRY(upload(&h->rank, s.rank));
  TRY(upload(&h->frp, s.row_ptr));
  TRY(upload(&h->fcol, s.col));
  TRY(upload(&h->fdiag, s.diag));
  TRY(upload(&h->ymap, s.ymap));
  TRY(upload(&h->lvl_ptr, s.lvl_ptr));
  TRY(upload(&h->rlvl_ptr, s.rlvl_ptr));
  TRY(dalloc(&h->rows, s.rows.size() / 4));
  CK(cudaMemcpy(h->rows, s.rows.data(), s.rows.size() * 4, cudaMemcpyHostToDevice));
  TRY(dalloc(&h->targets, s.targets.size() / 4));  // two int4 per target
  CK(cudaMemcpy(h->targets, s.targets.data(), s.targets.size() * 4, cudaMemcpyHostToDevice));
  TRY(dalloc(&h->pairs, s.pairs.size() / 2));
  if (!s.pairs.empty()) CK(cudaMemcpy(h->pairs, s.pairs.data(), s.pairs.size() * 4, cudaMemcpyHostToDevice));
  if (lu_smem_bytes<float>((int64_t)npos, n, 0, 0) <= smem_optin()) TRY(nr_setup_smem(h));
  const int Kp = h->Kp;
  const size_t E = (size_t)n * Kp;
  TRY(dalloc(&h->th, E)); TRY(dalloc(&h->vm, E));
  TRY(dalloc(&h->Ps, E)); TRY(dalloc(&h->Qs, E));
  TRY(dalloc(&h->V, E)); TRY(dalloc(&h->U, E)); TRY(dalloc(&h->I, E)); TRY(dalloc(&h->X, E));
  TRY(dalloc(&h->F, npos * Kp * sizeof(Blk<double>)));
  TRY(dalloc(&h->Dinv, E * sizeof(Blk<double>)));
  TRY(dalloc(&h->of, Kp)); TRY(dalloc(&h->ot, Kp)); TRY(dalloc(&h->active, Kp)); TRY(dalloc(&h->status, Kp));
  TRY(dalloc(&h->iters, Kp)); TRY(dalloc(&h->bad, Kp)); TRY(dalloc(&h->n_active, 1));
  TRY(dalloc(&h->yff, Kp)); TRY(dalloc(&h->yft, Kp)); TRY(dalloc(&h->ytt, Kp));
  TRY(dalloc(&h->maxmis, Kp)); TRY(dalloc(&h->loss, Kp));
  TRY(dalloc(&h->pmax, (size_t)NR_CHUNKS * Kp)); TRY(dalloc(&h->psum, (size_t)NR_CHUNKS * Kp));
  TRY(dalloc(&h->maxmis0, Kp)); TRY(dalloc(&h->loss0, Kp));
  CK(cudaMallocHost((void**)&h->h_nact, sizeof(int32_t)));
  return DPF_OK;
}

extern "C" int dpf_nr_create(const dpf_ybus* y, int32_t max_case, dpf_nr** out) {
  dpf::Range nvtx_range("dpf_nr_create");
  clear_error();
  if (!y || !out || max_case <= 0) return fail(DPF_E_INVALID, "dpf_nr_create: NULL argument or max_case <= 0");
  *out = nullptr;
  if (!y->dev.ready) return fail(DPF_E_STATE, "dpf_nr_create: Y_bus not uploaded (dpf_ybus_upload)");
  dpf_nr* h = new (std::nothrow) dpf_nr;
  if (!h) return fail(DPF_E_OOM, "dpf_nr_create: host allocation");
  h->y = y;
  h->max_case = max_case;
  h->Kp = (max_case + 31) / 32 * 32;
  int rc = nr_symbolic(y, (int64_t)1 << 28, &h->sym);
  if (rc == DPF_OK && (int64_t)h->sym.row_ptr[y->n] * h->Kp > ((int64_t)1 << 40) / 32)
    rc = fail(DPF_E_UNSUPPORTED, "dpf_nr_create: factor storage too large");
  if (rc == DPF_OK) rc = nr_setup(h);
  if (rc != DPF_OK) {
    nr_release(h);
    delete h;
    return rc;
  }
  *out = h;
  return DPF_OK;
}

extern "C" int dpf_nr_free(dpf_nr* h) {
  if (!h) return DPF_OK;
  nr_release(h);
  delete h;
  return DPF_OK;
}

extern "C" int dpf_nr_stats(const dpf_nr* h, int64_t* n_pos, int64_t* n_pairs, int32_t* n_levels,
                            int64_t* launches) {
  clear_error();
  if (!h) return fail(DPF_E_INVALID, "dpf_nr_stats: NULL handle");
  if (n_pos) *n_pos = h->sym.row_ptr[h->sym.n];
  if (n_pairs) *n_pairs = (int64_t)h->sym.pairs.size() / 2;
  if (n_levels) *n_levels = h->sym.n_levels;
  if (launches) *launches = h->launches;
  return DPF_OK;
}

// CTAs of the shared-memory form an SM holds.
template <class T>
static int smem_ctas(int threads, size_t bytes, int* n) {
  CK(allow_smem(k_nr_lu_smem<T>, bytes));
  CK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(n, k_nr_lu_smem<T>, threads, bytes));
  return DPF_OK;
}

template <class T>
static int nr_iterate_linear(dpf_nr* h, const NrArgs& a, bool smem, cudaStream_t s) {
  if (smem) {
    const size_t bytes = lu_smem_bytes<T>(a.npos, a.N, a.chunk_units, a.n_chunk);
    k_nr_lu_smem<T><<<a.K, h->smem_threads, bytes, s>>>(a);
    CKLAUNCH();
    h->launches += 1;
    return DPF_OK;
  }
  k_nr_assemble<T><<<grid_for((size_t)a.N * a.Kp), 256, 0, s>>>(a);
  k_nr_lu<T><<<a.Kp / a.C, sizeof(T) == 8 ? NR_THREADS / 2 : NR_THREADS, 0, s>>>(a);
  k_nr_update<<<grid_for((size_t)a.N * a.Kp), 256, 0, s>>>(a);
  CKLAUNCH();
  h->launches += 3;
  return DPF_OK;
}

extern "C" void dpf_nr_default_opts(dpf_nr_opts* o) {
  if (!o) return;
  o->precision = DPF_FP64;
  o->tol = 1e-10;
  o->max_iter = 20;
  o->flat_start = 1;
  o->lanes = 0;
  o->fallback = 0;
}

extern "C" int dpf_nr_solve(dpf_nr* h, const dpf_batch* b, const dpf_nr_opts* o, void* stream) {
  dpf::Range nvtx_range("dpf_nr_solve");
  clear_error();
  if (!h || !b || !o) return fail(DPF_E_INVALID, "dpf_nr_solve: NULL argument");
  const int precision = o->precision, max_iter = o->max_iter, flat_start = o->flat_start;
  const double tol = o->tol;
  if (o->lanes < 0 || o->lanes > 32 || (o->lanes & (o->lanes - 1)))
    return fail(DPF_E_INVALID, "dpf_nr_solve: lanes must be 0 or a power of 2 up to 32");
  const dpf_ybus* y = h->y;
  const int K = b->n_case;
  if (K <= 0 || K > h->max_case) return fail(DPF_E_INVALID, "dpf_nr_solve: n_case %d outside 1..%d", K, h->max_case);
  if (b->host_io) return fail(DPF_E_INVALID, "dpf_nr_solve: device pointers only (host_io = 0)");
  if (!b->va || !b->vm) return fail(DPF_E_INVALID, "dpf_nr_solve: va and vm are required");
  if (b->va_start || b->vm_start) return fail(DPF_E_INVALID, "dpf_nr_solve: va_start / vm_start are not supported");
  if ((b->p_spec == nullptr) != (b->q_spec == nullptr))
    return fail(DPF_E_INVALID, "dpf_nr_solve: p_spec and q_spec are given together");
  if (precision != DPF_FP32 && precision != DPF_FP64)
    return fail(DPF_E_INVALID, "dpf_nr_solve: precision must be DPF_FP32 or DPF_FP64");
  if (!(tol >= 0.0) || max_iter < 0) return fail(DPF_E_INVALID, "dpf_nr_solve: tol >= 0 and max_iter >= 0");
  cudaStream_t s = (cudaStream_t)stream;
  if (b->outage) {
    std::vector<int32_t> ho(K);
    CK(cudaMemcpyAsync(ho.data(), b->outage, (size_t)K * 4, cudaMemcpyDeviceToHost, s));
    CK(cudaStreamSynchronize(s));
    for (int k = 0; k < K; ++k) {
      const int l = ho[k];
      if (l < -1 || l >= y->m) return fail(DPF_E_INVALID, "case %d: outage index %d out of range", k, l);
      if (l >= 0 && y->bridge[l]) return fail(DPF_E_ISLANDED, "case %d: removing branch %d islands the grid", k, l);
    }
  }
  const DeviceYbus& d = y->dev;
  const NrSymbolic& sym = h->sym;
  NrArgs a;
  memset(&a, 0, sizeof a);
  a.N = y->n;
  a.K = K;
  a.Kp = (K + 31) / 32 * 32;
  // cases per CTA: the C lanes of a slot share its schedule loads and read
  // C consecutive blocks (a 128-byte line: 8 in FP32, 4 in FP64); few enough cases per CTA
  // that every CTA of the batch is resident at once (each walks the whole tree:
  // a second wave would double the time).  ms for 2,379 cases of 2,000 buses
  // by threads and C: 512, 8 12.9; 256, 4 13.5; 128, 2 14.6; 256, 8 15.0;
  // 512, 4 15.7; 256, 2 16.4; 128, 4 16.5.
  const int C_fixed = o->lanes;
  auto lanes_for = [&](int n_active) {
    if (C_fixed) return C_fixed;
    int C = precision == DPF_FP64 ? 4 : 8;
    while (C > 1 && n_active / C < num_sms_nr()) C >>= 1;
    return C;
  };
  a.C = lanes_for(K);
  // The shared-memory form where one case's factor fits and the cases still
  // iterating are few: it takes a case in the least time, the global form the
  // most cases at a time (it hides one case's latency behind others; nr_smem_cases).
  // Both give the same bits; o->lanes > 0 forces the global form.
  const size_t need = precision == DPF_FP64 ? lu_smem_bytes<double>(sym.row_ptr[sym.n], y->n, h->chunk_units, h->n_chunk)
                                            : lu_smem_bytes<float>(sym.row_ptr[sym.n], y->n, h->chunk_units, h->n_chunk);
  const bool fits = o->lanes == 0 && h->sstream && need <= smem_optin();
  int smem_cases = 0;  // most cases the shared-memory form takes
  if (fits) {
    int per_sm = 0;
    if (precision == DPF_FP64) TRY(smem_ctas<double>(h->smem_threads, need, &per_sm));
    else TRY(smem_ctas<float>(h->smem_threads, need, &per_sm));
    smem_cases = nr_smem_cases(y->n, precision == DPF_FP64, num_sms_nr(), per_sm);
  }
  a.va_slack = y->va_slack;
  a.tol = tol;
  a.inv_m = y->m_loss > 0 ? 1.0 / y->m_loss : 0.0;
  a.max_iter = max_iter;
  a.rp = d.row_ptr;
  a.ycol = d.col;
  a.yval = d.val64;
  a.type = d.type;
  a.p64 = d.p64;
  a.q64 = d.q64;
  a.vmset = d.vmset;
  a.perm = d.perm;
  a.order = h->order;
  a.rank = h->rank;
  a.frp = h->frp;
  a.fcol = h->fcol;
  a.fdiag = h->fdiag;
  a.ymap = h->ymap;
  a.n_levels = sym.n_levels;
  a.lvl_ptr = h->lvl_ptr;
  a.targets = h->targets;
  a.pairs = h->pairs;
  a.rlvl_ptr = h->rlvl_ptr;
  a.rows = h->rows;
  a.sstream = h->sstream;
  a.schunk = h->schunk;
  a.sent = h->sent;
  a.sdiag = h->sdiag;
  a.n_ent = h->n_ent;
  a.n_chunk = h->n_chunk;
  a.chunk_units = h->chunk_units;
  a.ring_bytes = (int)(precision == DPF_FP64 ? lu_ring_bytes<double>(y->n, h->chunk_units)
                                             : lu_ring_bytes<float>(y->n, h->chunk_units));
  a.npos = sym.row_ptr[sym.n];
  a.th = h->th;
  a.vm = h->vm;
  a.V = h->V;
  a.U = h->U;
  a.I = h->I;
  a.X = h->X;
  a.Ps = b->p_spec ? h->Ps : nullptr;
  a.Qs = b->p_spec ? h->Qs : nullptr;
  a.F = h->F;
  a.Dinv = h->Dinv;
  a.of = h->of;
  a.ot = h->ot;
  a.yff = h->yff;
  a.yft = h->yft;
  a.ytt = h->ytt;
  a.active = h->active;
  a.status = h->status;
  a.iters = h->iters;
  a.bad = h->bad;
  a.maxmis = h->maxmis;
  a.loss = h->loss;
  a.n_active = h->n_active;
  a.pmax = h->pmax;
  a.psum = h->psum;
  a.maxmis0 = h->maxmis0;
  a.loss0 = h->loss0;
  const size_t E = (size_t)a.N * a.Kp;
  const int cb = (a.Kp + 255) / 256;
  k_nr_init<<<cb, 256, 0, s>>>(a, b->outage, d.br_f, d.br_t, d.br_r, d.br_x, d.br_bch, d.br_tap);
  k_nr_in<<<grid_for(E), 256, 0, s>>>(a, b->va, b->vm, b->p_spec, b->q_spec, b->vm_set, flat_start ? 1 : 0);
  CKLAUNCH();
  h->launches += 2;
  for (int it = 0;; ++it) {
    k_nr_volt<<<grid_for(E), 256, 0, s>>>(a);
    k_nr_eval<<<grid_for(E), 256, 0, s>>>(a);
    CK(cudaMemsetAsync(a.n_active, 0, 4, s));
    k_nr_partial<<<dim3(a.Kp / 32, NR_CHUNKS), 256, 0, s>>>(a);
    a.first = it == 0;
    k_nr_check<<<cb, 256, 0, s>>>(a);
    CKLAUNCH();
    h->launches += 4;
    CK(cudaMemcpyAsync(h->h_nact, a.n_active, 4, cudaMemcpyDeviceToHost, s));
    CK(cudaStreamSynchronize(s));
    if (*h->h_nact == 0 || it > max_iter) break;
    // few cases left: fewer cases per CTA, more slots per case (a shorter
    // walk for each; CTAs whose cases have all stopped return at once)
    a.C = lanes_for(*h->h_nact);
    const bool smem = *h->h_nact <= smem_cases;
    if (precision == DPF_FP64) TRY(nr_iterate_linear<double>(h, a, smem, s));
    else TRY(nr_iterate_linear<float>(h, a, smem, s));
  }
  const int fb = o->fallback && !flat_start;
  k_nr_out<<<grid_for(E), 256, 0, s>>>(a, b->va, b->vm, fb);
  k_nr_case_out<<<cb, 256, 0, s>>>(a, b->iters, b->status, b->max_mismatch, b->loss, fb);
  CKLAUNCH();
  h->launches += 2;
  return DPF_OK;
}
