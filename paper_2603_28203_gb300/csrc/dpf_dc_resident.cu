// On-chip form of the DC solve (dpf_dc.cuh) for grids of up to RES_MAX_N
// buses: one CTA per case runs the whole Jacobi-preconditioned CG.
//
// The streaming form launches two kernels per CG iteration over the whole
// batch and moves 96 bytes per element through HBM / L2 in each (48 in FP32).
// A case's vectors fit one SM, so here a CTA keeps x, r, the direction and
// 1 / B_ii in registers, the gathered copy of the direction and B (sliced
// ELL, see dpf_resident.cu) in shared memory, and stops when its own case has
// converged: no launch, no host test and no other case's iterations to wait
// for.  With the direction at hand q = B' p is formed directly (the streaming
// form carries it as a recurrence so that no CTA waits for another's p).
//
// Double-float sums: a product is added with a two-sum of the high words, its
// error terms collected in the low word and renormalised once per sum, about
// 2^-47 of the sum of the magnitudes.  The dot products and the step lengths
// are double-float as well (FP64 issue is dear here, and every warp forms
// them from the warps' partial sums).
// Error of the angles against a dense FP64 solve, rms over the batch relative
// to the largest angle, by the relative residual asked for (streaming form with
// FP64 scalars and q as a recurrence / here; cases x buses):
//             1e-4             1e-10              1e-14
//   3,000 x 30    1.3e-6 / 1.3e-6  1.8e-14 / 1.0e-14  1.8e-14 / 1.0e-14
//   1,000 x 300   1.3e-5 / 9.8e-6  6.8e-13 / 3.7e-13  6.2e-13 / 2.6e-13
//   1,000 x 1,000 3.5e-5 / 2.8e-5  2.6e-12 / 2.3e-12  1.3e-12 / 3.7e-13
//   400 x 2,000   1.3e-5 / 8.0e-6  3.8e-12 / 3.8e-12  6.6e-13 / 2.4e-13
// so the double-float scalars cost nothing (at 1e-10 and above the error is the
// stop test's); what the recurrence lost, the direct product keeps.  Totals in
// three floats took 20-39% longer, in fixed point 50-100%, with the same errors.
#include <cuda_runtime.h>

#include <algorithm>

#include "dpf_dc.cuh"
#include "dpf_resident.h"
#include "dpf_smem.h"

namespace dpf {

constexpr size_t DC_STATIC_SMEM = 1024;  // of k_dc_resident, at most

template <class T> struct DcResArgs {
  int N, K, Kp, T_, n_pair, n_slice, max_iter;
  const int32_t* rord;
  const int32_t* rpos;
  const int32_t* soff;
  const uint32_t* col2;
  const float4* bval;      // [pair][32] two entries (hi, lo)
  const int32_t* dpos;
  const float2* bcsr;      // B in CSR order (the diagonal of an outage's rows)
  const float2* dinv;      // 1 / B_ii by position
  const uint8_t* type;
  const double* pspec;
  int spec_per_case;
  double va_slack;
  const int32_t* of;
  const int32_t* ot;
  const double* ob;
  const double* flow;
  double* x;               // [N][Kp] solution
  double* res;
  int32_t* iters;
  double tol2;
};

// sum += a b, the sum an unnormalised (hi, lo) pair
__device__ __forceinline__ void acc_mul(float2& s, float2 a, float2 b) {
  const float p = __fmul_rn(a.x, b.x);
  float e = __fmaf_rn(a.x, b.x, -p);
  e = __fmaf_rn(a.x, b.y, e);
  e = __fmaf_rn(a.y, b.x, e);
  const float2 t = df_two_sum(s.x, p);
  s = make_float2(t.x, __fadd_rn(s.y, __fadd_rn(t.y, e)));
}
__device__ __forceinline__ void acc_mul(float& s, float a, float b) { s = fmaf(a, b, s); }
__device__ __forceinline__ float2 acc_done(float2 s) { return df_quick(s.x, s.y); }
__device__ __forceinline__ float acc_done(float s) { return s; }
// c + a b
template <class T> __device__ __forceinline__ T axpy(T a, T b, T c) {
  acc_mul(c, a, b);
  return acc_done(c);
}
// a dot product's partial as a double-float pair, and their sum
__device__ __forceinline__ float2 as_df(float2 v) { return v; }
__device__ __forceinline__ float2 as_df(float v) { return make_float2(v, 0.f); }
__device__ __forceinline__ float2 sum_df(float2 a, float2 b) {
  const float2 t = df_two_sum(a.x, b.x);
  return make_float2(t.x, __fadd_rn(t.y, __fadd_rn(a.y, b.y)));
}
__device__ __forceinline__ float2 shfl_sum(float2 v, int from) {
#pragma unroll
  for (int off = from; off > 0; off >>= 1)
    v = sum_df(v, make_float2(__shfl_xor_sync(0xffffffffu, v.x, off), __shfl_xor_sync(0xffffffffu, v.y, off)));
  return v;
}
template <class T> __device__ __forceinline__ T df_to(float2 v);
template <> __device__ __forceinline__ float2 df_to<float2>(float2 v) { return v; }
template <> __device__ __forceinline__ float df_to<float>(float2 v) { return v.x + v.y; }
template <class T> struct BPair;
template <> struct BPair<float2> { using V = float4; };
template <> struct BPair<float> { using V = float2; };
__device__ __forceinline__ void pair_of(float4 v, float2& a, float2& b) {
  a = make_float2(v.x, v.y);
  b = make_float2(v.z, v.w);
}
__device__ __forceinline__ void pair_of(float2 v, float& a, float& b) {
  a = v.x;
  b = v.y;
}
template <class T> __device__ __forceinline__ typename BPair<T>::V pair_to(float4 v);
template <> __device__ __forceinline__ float4 pair_to<float2>(float4 v) { return v; }
template <> __device__ __forceinline__ float2 pair_to<float>(float4 v) { return make_float2(v.x, v.z); }

// Every thread's rows are the positions tid + s * T.  What bounds it is issue
// of the (emulated) arithmetic, 286 instructions per 32 rows and iteration in
// double-float (issue 68%, FMA pipe 48%, shared memory 51%), 121 in FP32 (48%,
// 20%, 49%), a quarter of them the two reductions.  Milliseconds for
// 2,379 outages of a 2,000-bus grid to 1e-10 (double-float) and 1e-4 (FP32):
// streaming 119.5 and 48; four rows per thread and one CTA per SM 47.8 and
// 20.7; eight rows and two CTAs 57.7 (spills) and 15.8; two rows of 1,024
// threads 61.7 and 28.7.  A 64-register form of the first spills: 57.6.
template <class T, int RPT>
__global__ void __launch_bounds__(2048 / RPT, RPT == 8 ? 2 : 1) k_dc_resident(const DcResArgs<T> q) {
  using BV = typename BPair<T>::V;
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ float2 part[3][32];  // (the two reductions of an iteration use different rows)
  const int nt = q.T_, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = nt >> 5;
  BV* sb = reinterpret_cast<BV*>(smem);
  T* P = reinterpret_cast<T*>(sb + q.n_pair * 32);
  T* Pt = P + tid;       // this thread's rows: every nt-th position
  uint32_t* sc = reinterpret_cast<uint32_t*>(P + nt * RPT);
  __shared__ struct {  // of the case: out of the registers
    T ob, df, dt;        // b_l, 1 / B'_ii at the outage's rows
    float2 stop;         // tol^2 |r0|^2
    double rr0;
    int pf, pt;
  } cs;
  static_assert(sizeof part + sizeof cs <= DC_STATIC_SMEM, "static shared memory");
  const int k = blockIdx.x;
  const size_t Kp = (size_t)q.Kp;
  for (int t = tid; t < q.n_pair * 32; t += nt) {
    sb[t] = pair_to<T>(__ldg(q.bval + t));
    sc[t] = __ldg(q.col2 + t);
  }
  const int of = q.of ? q.of[k] : -1, ot = q.of ? q.ot[k] : -1;
  const T ob = df_cast<T>(q.ob[k]);
  const T zero = df_zero<T>();
  if (tid == 0) {
    cs.ob = ob;
    cs.pf = of >= 0 ? q.rpos[of] : 0;
    cs.pt = of >= 0 ? q.rpos[ot] : 0;
  }

  int sl[RPT];           // entry pairs of the rows' slices: first, count << 20
  T x[RPT], r[RPT];
  T di[RPT];             // 1 / B'_ii
  int bits = 0;          // 1 << s: unknown; 256 << s: the outage's from-row; 65536 << s: its to-row (s < 8)
#pragma unroll
  for (int s = 0; s < RPT; ++s) {
    const int pos = s * nt + tid, i = pos < q.N ? __ldg(q.rord + pos) : -1;
    sl[s] = 0;
    if ((pos >> 5) < q.n_slice) {
      const int a = __ldg(q.soff + (pos >> 5)), b = __ldg(q.soff + (pos >> 5) + 1);
      sl[s] = a | (b - a) << 20;
    }
    x[s] = r[s] = zero;
    if (i >= 0) {
      if (i == of) bits |= 256 << s;
      if (i == ot) bits |= 65536 << s;
      if (__ldg(q.type + i) == BUS_SLACK) {
        x[s] = df_cast<T>(q.va_slack);
      } else {
        bits |= 1 << s;
        const size_t e = (size_t)i * Kp + k;
        const double Pi = q.flow ? (i == of ? q.flow[k] : i == ot ? -q.flow[k] : 0.0)
                                 : (q.spec_per_case ? q.pspec[e] : q.pspec[i]);
        r[s] = df_cast<T>(Pi);
        if (i == of || i == ot) {  // 1 / B'_ii
          const T d = df_div(df_cast<T>(1.0), df_add(df_coef<T>(__ldg(q.bcsr + __ldg(q.dpos + i))), df_neg(ob)));
          (i == of ? cs.df : cs.dt) = d;
        }
      }
    }
    P[pos] = x[s];
  }
  __syncthreads();
  // (B' v)_row, v in P by position
  auto row = [&](int s) {
    T a = zero;
    int t = (sl[s] & 0xfffff) * 32 + lane;
    for (int n = sl[s] >> 20; n > 0; --n, t += 32) {
      const uint32_t cc = sc[t];
      T b0, b1;
      pair_of(sb[t], b0, b1);
      constexpr unsigned sh = sizeof(T) == 8 ? 0 : 1;  // columns are stored as position * 8
      acc_mul(a, b0, *reinterpret_cast<const T*>(reinterpret_cast<const unsigned char*>(P) + ((cc & 0xffffu) >> sh)));
      acc_mul(a, b1, *reinterpret_cast<const T*>(reinterpret_cast<const unsigned char*>(P) + (cc >> (16 + sh))));
    }
    a = acc_done(a);
    if (bits & (0x10100 << s)) {
      const T d = df_add(P[cs.pf], df_neg(P[cs.pt]));
      a = axpy((bits >> s) & 256 ? df_neg(cs.ob) : cs.ob, d, a);
    }
    return a;
  };
#pragma unroll
  for (int s = 0; s < RPT; ++s) {
    di[s] = zero;
    if (bits & (1 << s)) di[s] = df_coef<T>(__ldg(q.dinv + s * nt + tid));
    if (bits & (0x10100 << s)) di[s] = (bits >> s) & 256 ? cs.df : cs.dt;
  }
  // Sums of two per-thread values over the CTA, every thread gets them: the
  // halves of a warp exchange so that each carries one of the two.
  auto reduce2 = [&](float2& u, float2& v) {
    const bool lo = lane < 16;
    const float2 give = lo ? v : u;
    float2 a = sum_df(lo ? u : v, make_float2(__shfl_xor_sync(0xffffffffu, give.x, 16),
                                              __shfl_xor_sync(0xffffffffu, give.y, 16)));
    a = shfl_sum(a, 8);
    const float2 hi = make_float2(__shfl_sync(0xffffffffu, a.x, 16), __shfl_sync(0xffffffffu, a.y, 16));
    if (lane == 0) {
      part[0][warp] = a;
      part[1][warp] = hi;
    }
    __syncthreads();
    a = (lane & 15) < nw ? part[lane >> 4][lane & 15] : make_float2(0.f, 0.f);
    if (nw > 16) a = sum_df(a, 16 + (lane & 15) < nw ? part[lane >> 4][16 + (lane & 15)] : make_float2(0.f, 0.f));
    a = shfl_sum(a, 8);
    a = df_quick(a.x, a.y);
    u = make_float2(__shfl_sync(0xffffffffu, a.x, 0), __shfl_sync(0xffffffffu, a.y, 0));
    v = make_float2(__shfl_sync(0xffffffffu, a.x, 16), __shfl_sync(0xffffffffu, a.y, 16));
  };
  auto reduce1 = [&](float2& u) {
    u = shfl_sum(u, 16);
    if (lane == 0) part[2][warp] = u;
    __syncthreads();
    u = (lane & 15) < nw ? part[2][lane & 15] : make_float2(0.f, 0.f);
    if (nw > 16) u = sum_df(u, 16 + (lane & 15) < nw ? part[2][16 + (lane & 15)] : make_float2(0.f, 0.f));
    u = shfl_sum(u, 8);
    u = df_quick(u.x, u.y);
  };
  // r0 = P - B' x0, z0 = r0 / diag, p0 = z0
  float2 rz = make_float2(0.f, 0.f), rr = rz;
  T z[RPT];
  {
    T sz = zero, sr = zero;
#pragma unroll
    for (int s = 0; s < RPT; ++s) {
      const T b = row(s);
      z[s] = zero;
      if (bits & (1 << s)) {
        r[s] = df_add(r[s], df_neg(b));
        z[s] = df_mul(r[s], di[s]);
        acc_mul(sz, r[s], z[s]);
        acc_mul(sr, r[s], r[s]);
      }
    }
    rz = as_df(sz);
    rr = as_df(sr);
  }
  reduce2(rz, rr);  // (a barrier: every x0 has been gathered)
  if (tid == 0) {
    cs.rr0 = df_val(rr);
    cs.stop = df_from(q.tol2 * cs.rr0);
  }
#pragma unroll
  for (int s = 0; s < RPT; ++s) Pt[s * nt] = z[s];
  __syncthreads();

  int it = 0;
  for (;;) {
    T qv[RPT];
    T sum = zero;
#pragma unroll
    for (int s = 0; s < RPT; ++s) {
      qv[s] = row(s);
      acc_mul(sum, Pt[s * nt], qv[s]);  // (p = 0 off the unknowns)
    }
    float2 pq = as_df(sum);
    reduce1(pq);
    const float2 al = pq.x != 0.f ? df_div(rz, pq) : make_float2(0.f, 0.f);
    const T alpha = df_to<T>(al), nalpha = df_neg(alpha);
    T sz = zero, sr = zero;
#pragma unroll
    for (int s = 0; s < RPT; ++s) {
      if (bits & (1 << s)) {
        x[s] = axpy(alpha, Pt[s * nt], x[s]);
        r[s] = axpy(nalpha, qv[s], r[s]);
        z[s] = df_mul(r[s], di[s]);
        acc_mul(sz, r[s], z[s]);
        acc_mul(sr, r[s], r[s]);
      }
    }
    float2 rzn = as_df(sz);
    rr = as_df(sr);
    reduce2(rzn, rr);  // (a barrier: every p has been gathered)
    it += 1;
    // |r|^2 <= tol^2 |r0|^2, or broken down (NaN)
    const float2 stop = cs.stop;
    if (rr.x < stop.x || (rr.x == stop.x && rr.y <= stop.y) || !(rr.x == rr.x) || it >= q.max_iter) break;
    const T beta = df_to<T>(rz.x != 0.f ? df_div(rzn, rz) : make_float2(0.f, 0.f));
    rz = rzn;
#pragma unroll
    for (int s = 0; s < RPT; ++s) Pt[s * nt] = axpy(beta, Pt[s * nt], z[s]);
    __syncthreads();
  }
#pragma unroll
  for (int s = 0; s < RPT; ++s) {
    const int pos = s * nt + tid;
    if (pos < q.N) q.x[(size_t)__ldg(q.rord + pos) * Kp + k] = df_val(x[s]);
  }
  if (tid == 0) {
    q.iters[k] = it;
    q.res[k] = cs.rr0 > 0.0 ? sqrt(df_val(rr) / cs.rr0) : 0.0;
  }
}

// Rows per thread where cases outnumber SMs (the best of each type, see the kernel).
template <class T> constexpr int dc_many() { return sizeof(T) == 8 ? 4 : 8; }

DcShape dc_res_shape(const dpf_ybus* y, int K, bool f32) {
  DcShape sh;
  const DeviceYbus& d = y->dev;
  if (!d.res_rord) return sh;
  int dev = 0, sms = 1, lim = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  cudaDeviceGetAttribute(&lim, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  // more cases than SMs: many rows per thread; else two, the shorter iteration
  // (one case of 2,000 buses to 1e-10: 27.4 ms streaming, 3.9 ms), and for what
  // one warp holds
  sh.rpt = K > sms && y->n > 64 ? (f32 ? dc_many<float>() : dc_many<float2>()) : 2;
  sh.T = std::max(32, ((y->n + sh.rpt - 1) / sh.rpt + 31) / 32 * 32);
  const size_t v = f32 ? sizeof(float) : sizeof(float2);
  sh.smem = (size_t)d.res_pairs * 32 * (2 * v + 4) + (size_t)sh.T * sh.rpt * v;
  // B as sliced ELL is what may not fit: its slices are as long as their
  // longest row (a star of 700 buses takes 243 KB, a dense grid of 150 240 KB)
  if (sh.smem + DC_STATIC_SMEM > (size_t)lim) return sh;
  int most = 0;
  cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev);
  const int ctas = std::max(1, most / (int)(sh.smem + DC_STATIC_SMEM + 1024));
  const int ctas_free = std::max(1, std::min(32, (sh.rpt > 2 ? 512 : 1024) / sh.T));  // (128 or 64 registers a thread)
  sh.ok = dc_pays(y->n, K, f32, sms, d.res_pairs, ctas, ctas_free);
  return sh;
}

template <class T>
static int dc_res_t(const dpf_ybus* y, const DcRes& c, const DcShape& sh, cudaStream_t s) {
  const DeviceYbus& d = y->dev;
  DcResArgs<T> q;
  q.N = y->n;
  q.K = c.K;
  q.Kp = c.Kp;
  q.n_pair = d.res_pairs;
  q.n_slice = d.res_slices;
  q.max_iter = c.max_iter;
  q.rord = d.res_rord;
  q.rpos = d.res_rpos;
  q.soff = d.res_soff;
  q.col2 = d.res_col2;
  q.bval = d.res_bval;
  q.dpos = d.dpos;
  q.bcsr = d.dcval;
  q.dinv = d.res_dinv;
  q.type = d.type;
  q.pspec = c.pspec;
  q.spec_per_case = c.spec_per_case;
  q.va_slack = c.va_slack;
  q.of = c.of;
  q.ot = c.ot;
  q.ob = c.ob;
  q.flow = c.flow;
  q.x = c.x;
  q.res = c.res;
  q.iters = c.iters;
  q.tol2 = c.tol * c.tol;
  constexpr int many = dc_many<T>();
  q.T_ = sh.T;
  auto kern = sh.rpt == many ? k_dc_resident<T, many> : k_dc_resident<T, 2>;
  cudaError_t e = allow_smem(kern, sh.smem);
  if (e != cudaSuccess) return e;
  kern<<<c.K, q.T_, sh.smem, s>>>(q);
  return cudaGetLastError();
}

int dc_res_launch(const dpf_ybus* y, const DcRes& c, const DcShape& sh, bool f32, void* stream) {
  return f32 ? dc_res_t<float>(y, c, sh, (cudaStream_t)stream) : dc_res_t<float2>(y, c, sh, (cudaStream_t)stream);
}

}  // namespace dpf
