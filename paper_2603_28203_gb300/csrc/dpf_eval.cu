// Evaluation of whole cases on chip: S_calc (dpf_power) and the loss with its
// adjoint (dpf_loss_backward) for grids of up to RES_MAX_N buses, one CTA per
// case, one launch.
//
// The streaming form takes a batch through the case-minor workspace layout:
// transposes in, a full optimiser state nobody reads, one pass per kernel over
// HBM, widening and transposes out (11 to 20 launches).  A case's vectors are
// contiguous in the caller's arrays and fit one SM, so a CTA reads them once,
// runs both passes in shared memory and writes the results once.  Y_bus (the
// sliced ELL of dpf_resident.cu) is read through L1 / L2, shared by all cases.
//
// Conversions between FP64 and FP32 run as integer arithmetic: GB300 issues an
// FP64 instruction (the conversions among them) in 16 cycles per warp and SM,
// and splitting the two inputs into double-float pairs took eight of them per
// element, more than everything else of dpf_power together.
//
// The FP32 results are those of the streaming kernels to the bit (the same
// functions on the same operands, each row's products in the same order); FP64
// results and losses agree to rounding.
//
// S_calc of 2,379 FP32 cases of 2,000 buses: 281 us streaming, 110 here.  What
// bounds it is latency between the phases: two CTAs per SM (by registers) spend
// 6.5 of 20 warp cycles per issue on loads and 5.8 at barriers; issue 41%, DRAM
// 10%.  With a loss the FP64 pass binds (FP64 pipe 82%).  eval_pays says which
// batches the streaming kernels take.
#include <cuda_runtime.h>

#include <algorithm>

#include "dpf_kernels.cuh"
#include "dpf_resident.h"
#include "dpf_sell.cuh"
#include "dpf_smem.h"

namespace dpf {

template <class R> struct EvalArgs {
  using C = typename Prec<R>::C;
  int N, K, n_slice;
  size_t Kp;               // case stride of Vout / Wout
  const uint16_t* upos;    // user bus -> position
  const uint16_t* puser;   // position -> user bus
  const int32_t* rord;     // position -> internal row
  const uint8_t* type;     // by internal row
  const int32_t* soff;
  const uint32_t* col2;
  const ValPair<R>* val;
  const ValPair<double>* val64;  // FP32 with a loss
  const int32_t* rpos;
  const double *va, *vm, *p, *q;  // [K][N] user order (p, q may be NULL: the grid's)
  const R *gp, *gq;               // grid injections by internal row
  const double *gp64, *gq64;
  const int32_t* outage;
  const int32_t *br_f, *br_t;
  const double *br_r, *br_x, *br_bch, *br_tap;
  R inv_m2, m_half;
  double inv_m;
  // outputs (user order), each may be NULL
  double *o_p, *o_q;              // S_calc
  double *loss, *d_va, *d_vm, *d_p, *d_q;
  C *Vout, *Wout;                 // [N][Kp] internal layout (the branch adjoint's operands)
  // shared memory offsets (W, specification, c, |V|, FP64 V)
  unsigned w, s, c, m, v64;
};

// Working-precision state of one bus from the caller's FP64 (theta, |V|).
__device__ __forceinline__ void eval_volt(double va, double vm, float2& v, float& m, double2* v64) {
  const float2 th = split_df(va), mg = split_df(vm);
  v = volt(th, mg);
  m = mwork(mg);
  if (v64) {  // the master value, 48 bits, as the streaming FP64 pass sees it
    double s, c;
    sincos(mval(th), &s, &c);
    const double w = mval(mg);
    *v64 = make_double2(w * c, w * s);
  }
}
__device__ __forceinline__ void eval_volt(double va, double vm, double2& v, double& m, double2*) {
  v = volt(va, vm);
  m = vm;
}
// BWD: the adjoint pass; LOSS: the FP64 loss (in FP32 from an FP64 pass over
// the same state).
template <class R, bool BWD, bool LOSS>
__global__ void __launch_bounds__(sizeof(R) == 4 ? 1024 : 512, 1) k_eval_case(const EvalArgs<R> q) {
  using C = typename Prec<R>::C;
  constexpr bool V64 = LOSS && sizeof(R) == 4;
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ struct {
    int of, ot, pf, pt;
    C yff, yft, ytt;
    double2 ff, ft, tt;
  } out;
  __shared__ double lsum[32];
  C* V = reinterpret_cast<C*>(smem);
  C* W = reinterpret_cast<C*>(smem + q.w);
  C* S = reinterpret_cast<C*>(smem + q.s);
  C* Cc = reinterpret_cast<C*>(smem + q.c);
  R* M = reinterpret_cast<R*>(smem + q.m);
  double2* VV = reinterpret_cast<double2*>(smem + q.v64);
  const int tid = threadIdx.x, lane = tid & 31, T = blockDim.x, N = q.N, k = blockIdx.x;
  const size_t base = (size_t)k * N;
  if (tid == 0) {
    const int ell = q.outage ? q.outage[k] : -1;
    out.of = out.ot = -1;
    if (ell >= 0) {  // pi-model block of the outaged branch (as k_case_init)
      const double r = q.br_r[ell], x = q.br_x[ell], bch = q.br_bch[ell];
      const double tau = (q.br_tap[ell] == 0.0) ? 1.0 : q.br_tap[ell];
      const double d = r * r + x * x, gs = r / d, bs = -x / d, t2 = tau * tau;
      out.ff = make_double2(gs / t2, (bs + 0.5 * bch) / t2);
      out.ft = make_double2(-gs / tau, -bs / tau);
      out.tt = make_double2(gs, bs + 0.5 * bch);
      out.yff = mkc((R)out.ff.x, (R)out.ff.y);
      out.yft = mkc((R)out.ft.x, (R)out.ft.y);
      out.ytt = mkc((R)out.tt.x, (R)out.tt.y);
      out.of = q.br_f[ell];
      out.ot = q.br_t[ell];
      out.pf = q.rpos[out.of];
      out.pt = q.rpos[out.ot];
    }
  }
  for (int u = tid; u < N; u += T) {  // the case's state, into the order of the rows
    const int p = q.upos[u];
    C v;
    R m;
    eval_volt(__ldcs(q.va + base + u), __ldcs(q.vm + base + u), v, m, V64 ? VV + p : nullptr);
    V[p] = v;
    if constexpr (BWD) M[p] = m;
    if (q.p) S[p] = mkc(to_work(__ldcs(q.p + base + u), R(0)), to_work(__ldcs(q.q + base + u), R(0)));
  }
  __syncthreads();
  const int of = out.of, ot = out.ot, np = q.n_slice * 32;
  double sq = 0.0;
  for (int p = tid; p < np; p += T) {  // ---- forward
    const int sl = p >> 5;
    C I = sell_row_g<R>(q.val + lane, q.col2 + lane, __ldg(q.soff + sl) * 32, __ldg(q.soff + sl + 1) * 32, smem);
    if (p >= N) {
      if constexpr (BWD) W[p] = mkc(R(0), R(0));
      continue;
    }
    const int i = __ldg(q.rord + p), ty = __ldg(q.type + i);
    const C v = V[p];
    if (i == of) {
      cfms(I, out.yff, v);
      cfms(I, out.yft, V[out.pt]);
    } else if (i == ot) {
      cfms(I, out.yft, V[out.pf]);
      cfms(I, out.ytt, v);
    }
    const C s = power_of(v, I);
    if constexpr (!BWD) {
      W[p] = s;
    } else {
      const C sp = q.p ? S[p] : mkc(q.gp[i], q.gq[i]);
      const R dP = (ty != BUS_SLACK) ? s.x - sp.x : R(0);
      const R dQ = (ty == BUS_PQ) ? s.y - sp.y : R(0);
      if constexpr (LOSS && sizeof(R) == 8) sq += dP * dP + dQ * dQ;
      const R ca = q.inv_m2 * dP, cb = q.inv_m2 * dQ;
      Cc[p] = mkc(ca, cb);
      const C w = w_of(ca, cb, v);
      W[p] = w;
      S[p] = mkc(sp.x, ty == BUS_PV ? s.y : sp.y);  // Q_calc at pv buses, for the adjoint
      if (q.Wout) {
        q.Vout[(size_t)i * q.Kp + k] = v;
        q.Wout[(size_t)i * q.Kp + k] = w;
      }
    }
  }
  if constexpr (V64) {  // ---- the FP64 mismatch of the same state
    for (int p = tid; p < np; p += T) {
      const int sl = p >> 5;
      double2 I = make_double2(0.0, 0.0);
      const int e1 = __ldg(q.soff + sl + 1) * 32;
      for (int e = __ldg(q.soff + sl) * 32; e < e1; e += 32) {
        const uint32_t cc = __ldg(q.col2 + e + lane);
        const ValPair<double> y = ldg_pair(q.val64 + e + lane);
        cfma(I, y.a, VV[(cc & 0xffffu) >> 3]);
        cfma(I, y.b, VV[cc >> 19]);
      }
      if (p >= N) continue;
      const int i = __ldg(q.rord + p), ty = __ldg(q.type + i);
      const double2 v = VV[p];
      if (i == of) {
        cfms(I, out.ff, v);
        cfms(I, out.ft, VV[out.pt]);
      } else if (i == ot) {
        cfms(I, out.ft, VV[out.pf]);
        cfms(I, out.tt, v);
      }
      if (ty == BUS_SLACK) continue;
      // (the caller's FP64 injections again: S holds them rounded)
      const size_t e = base + q.puser[p];
      const double ps = q.p ? q.p[e] : q.gp64[i], qs = q.p ? q.q[e] : q.gq64[i];
      const double dP = fma(v.x, I.x, v.y * I.y) - ps;
      sq = fma(dP, dP, sq);
      if (ty == BUS_PQ) {
        const double dQ = fma(v.y, I.x, -(v.x * I.y)) - qs;
        sq = fma(dQ, dQ, sq);
      }
    }
  }
  if constexpr (LOSS) {
    for (int off = 16; off > 0; off >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, off);
    if (lane == 0) lsum[tid >> 5] = sq;
  }
  __syncthreads();
  if constexpr (LOSS)
    if (tid == 0) {
      double s = 0.0;
      for (int w = 0; w < (T >> 5); ++w) s += lsum[w];
      q.loss[k] = s * q.inv_m;
    }
  if constexpr (!BWD) {
    for (int u = tid; u < N; u += T) {
      const C s = W[q.upos[u]];
      if (q.o_p) __stcs(q.o_p + base + u, widen(s.x));
      if (q.o_q) __stcs(q.o_q + base + u, widen(s.y));
    }
  } else {
    if (q.d_va || q.d_vm) {
      for (int p = tid; p < np; p += T) {  // ---- adjoint; (dL/dtheta, dL/d|V|) into V's place
        const int sl = p >> 5;
        C z = sell_row_g<R>(q.val + lane, q.col2 + lane, __ldg(q.soff + sl) * 32, __ldg(q.soff + sl + 1) * 32,
                            smem + q.w);
        if (p >= N) continue;
        const int i = __ldg(q.rord + p), ty = __ldg(q.type + i);
        C g = mkc(R(0), R(0));
        if (ty != BUS_SLACK) {
          const C w = W[p], v = V[p], sp = S[p];
          if (i == of) {
            cfms(z, out.yff, w);
            cfms(z, out.yft, W[out.pt]);
          } else if (i == ot) {
            cfms(z, out.yft, W[out.pf]);
            cfms(z, out.ytt, w);
          }
          const C g0 = conj_c_s(w, v, ty, sp.x, sp.y, sp.y, q.m_half);
          const C h = adj_h(g0, v, z);
          g = mkc(-h.y, (ty == BUS_PQ) ? div_step(h.x, M[p]) : R(0));
        }
        V[p] = g;
      }
      __syncthreads();
    }
    for (int u = tid; u < N; u += T) {
      const int p = q.upos[u];
      const C g = V[p], c = Cc[p];
      if (q.d_va) __stcs(q.d_va + base + u, widen(g.x));
      if (q.d_vm) __stcs(q.d_vm + base + u, widen(g.y));
      if (q.d_p) __stcs(q.d_p + base + u, -widen(c.x));
      if (q.d_q) __stcs(q.d_q + base + u, -widen(c.y));
    }
  }
}

template <class R>
static int eval_t(const dpf_ybus* y, const EvalCall& c, cudaStream_t s) {
  using C = typename Prec<R>::C;
  const DeviceYbus& d = y->dev;
  EvalArgs<R> q;
  q.N = y->n;
  q.K = c.K;
  q.n_slice = d.res_slices;
  q.Kp = (size_t)c.Kp;
  q.upos = d.res_upos;
  q.puser = d.res_puser;
  q.rord = d.res_rord;
  q.rpos = d.res_rpos;
  q.type = d.type;
  q.soff = d.res_soff;
  q.col2 = d.res_col2;
  const void* v32 = c.val32 ? c.val32 : d.res_val32;
  const void* v64 = c.val64 ? c.val64 : d.res_val64;
  q.val = reinterpret_cast<const ValPair<R>*>(sizeof(R) == 4 ? v32 : v64);
  q.val64 = reinterpret_cast<const ValPair<double>*>(v64);
  q.va = c.va;
  q.vm = c.vm;
  q.p = c.p;
  q.q = c.q;
  if constexpr (sizeof(R) == 4) {
    q.gp = d.p32;
    q.gq = d.q32;
  } else {
    q.gp = d.p64;
    q.gq = d.q64;
  }
  q.gp64 = d.p64;
  q.gq64 = d.q64;
  q.outage = c.outage;
  q.br_f = d.br_f;
  q.br_t = d.br_t;
  q.br_r = d.br_r;
  q.br_x = d.br_x;
  q.br_bch = d.br_bch;
  q.br_tap = d.br_tap;
  q.inv_m2 = (R)(y->m_loss > 0 ? 2.0 / y->m_loss : 0.0);
  q.m_half = (R)(0.5 * y->m_loss);
  q.inv_m = y->m_loss > 0 ? 1.0 / y->m_loss : 0.0;
  q.o_p = c.o_p;
  q.o_q = c.o_q;
  q.loss = c.loss;
  q.d_va = c.d_va;
  q.d_vm = c.d_vm;
  q.d_p = c.d_p;
  q.d_q = c.d_q;
  q.Vout = (C*)c.Vout;
  q.Wout = (C*)c.Wout;
  const bool bwd = c.backward, loss = bwd && c.loss;
  const unsigned np = (unsigned)d.res_slices * 32u, cs = sizeof(C);
  q.w = np * cs;
  q.s = q.w + np * cs;
  q.c = q.s + (bwd || c.p ? np * cs : 0u);
  q.m = q.c + (bwd ? np * cs : 0u);
  q.v64 = q.m + (bwd ? np * (unsigned)sizeof(R) : 0u);
  const size_t smem = q.v64 + (loss && sizeof(R) == 4 ? np * 16u : 0u);
  auto kern = !bwd ? k_eval_case<R, false, false> : loss ? k_eval_case<R, true, true> : k_eval_case<R, true, false>;
  cudaError_t e = allow_smem(kern, smem);
  if (e != cudaSuccess) return e;
  int dev = 0, sms = 1;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  // fewer cases than SMs: one row per thread; else several CTAs per SM
  const int most = sizeof(R) == 8 || c.K > sms ? 512 : 1024;
  kern<<<c.K, std::min((int)np, most), smem, s>>>(q);
  return cudaGetLastError();
}

int eval_launch(const dpf_ybus* y, const EvalCall& c, bool fp64, void* stream) {
  return fp64 ? eval_t<double>(y, c, (cudaStream_t)stream) : eval_t<float>(y, c, (cudaStream_t)stream);
}

}  // namespace dpf
