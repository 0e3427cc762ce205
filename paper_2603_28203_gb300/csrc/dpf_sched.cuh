// What the on-chip and whole-GPU forms of the iterations share: a case's
// scheduler as one warp keeps it, the forward and adjoint arithmetic of one row.
#pragma once

#include "dpf_kernels.cuh"
#include "dpf_plateau.h"

namespace dpf {

// The scheduler of one case, run by one warp with its state in registers (the
// same decisions and values as sched_case).  FP64 issue is dear on GB300, so
// in FP32 solves a step takes two FP64 operations: lane 0 carries beta1^t,
// lane 1 beta2^t; the plateau test compares the FP32 loss sums and falls back
// to the FP64 comparison only near the threshold (dpf_plateau.h); the step schedule's power is taken when its exponent changes.
template <class R> struct ResSched {
  double lr, best, bt;    // bt: lane 0 beta1^t, lane 1 beta2^t
  float bsum;             // FP32: the loss sum behind `best` (< 0: best as loaded)
  float tsum;             // FP32: the bar of the next improvement (plateau_bar)
  R lrw;                  // lr in working precision
  int bad, cool, it;
  R step, isb;            // of the update numbered it + 1
  __device__ __forceinline__ void load(const SchedArgs<R>& s, int k, int lane) {
    lr = s.lr[k];
    lrw = (R)lr;
    best = s.best[k];
    bt = lane == 0 ? s.b1t[k] : s.b2t[k];
    bad = s.bad[k];
    cool = s.cool[k];
    it = s.iters[k];
    bsum = tsum = -1.f;
    step = isb = R(1);
  }
  // the powers of update it + 1 and its bias corrections (independent of the loss)
  __device__ __forceinline__ void terms(const SchedArgs<R>& s, int lane) {
    step = lrw;
    isb = R(1);
    bt *= lane == 0 ? s.beta1 : s.beta2;
    if (s.opt == OPT_ADAM) {
      const R om = R(1) - (R)bt;
      step = lrw / __shfl_sync(0xffffffffu, om, 0);
      isb = R(1) / sqrtT(__shfl_sync(0xffffffffu, om, 1));
    }
  }
  // the decision of sched_case on this iterate's loss
  __device__ __forceinline__ bool improved(const SchedArgs<R>& s, R lsum) {
    if constexpr (sizeof(R) == 4) {
      const int side = plateau_side(lsum, tsum);
      if (side) return side > 0;
      if (bsum >= 0.f) best = (double)bsum * s.inv_m;
    }
    return (double)lsum * s.inv_m < best * (1.0 - s.threshold);
  }
  __device__ __forceinline__ void feed(const SchedArgs<R>& s, R lsum) {
    it += 1;
    if (s.sched == SCHED_PLATEAU) {
      if (improved(s, lsum)) {
        if constexpr (sizeof(R) == 4) {
          bsum = lsum;
          tsum = plateau_bar(lsum, s.keep);
        } else {
          best = (double)lsum * s.inv_m;
        }
        bad = 0;
      } else {
        bad += 1;
      }
      if (cool > 0) { cool -= 1; bad = 0; }
      if (bad > s.patience) {
        const double nl = fmax(lr * s.factor, s.min_lr);
        if (lr - nl > 1e-8) lr = nl;
        lrw = (R)lr;
        cool = s.cooldown;
        bad = 0;
      }
    } else if (s.sched == SCHED_STEP && it % s.step_every == 0) {
      double gk = 1.0, base = s.gamma;
      for (int e = it / s.step_every; e > 0; e >>= 1) {
        if (e & 1) gk *= base;
        base *= base;
      }
      lr = s.lr0 * gk;
      lrw = (R)lr;
    }
  }
  // after the last step (bt is that step's power, step / isb its terms)
  __device__ __forceinline__ void store(const SchedArgs<R>& s, int k, int lane) {
    if (lane == 1) s.b2t[k] = bt;
    if (lane) return;
    s.lr[k] = lr;
    s.b1t[k] = bt;
    s.iters[k] = it;
    s.step_size[k] = step;
    s.isbc2[k] = isb;
    if (s.sched == SCHED_PLATEAU) {
      if (bsum >= 0.f) best = (double)bsum * s.inv_m;
      s.best[k] = best;
      s.bad[k] = bad;
      s.cool[k] = cool;
    }
  }
};

// One row of a case held by a thread: master values and moments.
template <class R> struct ResRow {
  typename Prec<R>::M th, vm;
  R m1, v1, m2, v2;
  __device__ __forceinline__ void load(const IterArgs<R>& a, size_t e) {
    const typename Prec<R>::MS ms = a.ms[e];
    th = ms_th(ms);
    vm = ms_vm(ms);
    const Mom<R> o = mom_load(a.os + e);
    m1 = o.m1;
    v1 = o.v1;
    m2 = o.m2;
    v2 = o.v2;
  }
  __device__ __forceinline__ void store(const IterArgs<R>& a, size_t e) const {
    a.ms[e] = ms_make(th, vm);
    mom_store(a.os + e, Mom<R>{m1, v1, m2, v2});
  }
};

// Adjoint of one row (the arithmetic of adj_finish) and the optimiser step;
// sp.y is Q_calc at pv buses.  Returns the new value of the gathered vector.
template <class R, bool REF, bool ADAM>
__device__ __forceinline__ typename Prec<R>::C res_adj(const IterArgs<R>& a, int ty, ResRow<R>& r,
                                                       typename Prec<R>::C x, typename Prec<R>::C w,
                                                       typename Prec<R>::C z, typename Prec<R>::C sp, R step, R isb) {
  using C = typename Prec<R>::C;
  const int opt = ADAM ? (int)OPT_ADAM : a.opt;
  C v = x, u;
  if constexpr (REF) v = volt(r.th, r.vm, u);
  const C g0 = conj_c_s(w, v, ty, sp.x, sp.y, sp.y, a.m_half);
  const C h = adj_h(g0, v, z);
  const R vm_old = mwork(r.vm);
  R d_th = R(0), d_vm = R(0);
  r.th = opt_update(opt, r.th, -h.y, r.m1, r.v1, a.beta1, a.beta2, step, isb, a.eps, a.mom, a.alpha, d_th);
  if (ty == BUS_PQ)
    r.vm = opt_update(opt, r.vm, div_step(h.x, vm_old), r.m2, r.v2, a.beta1, a.beta2, step, isb, a.eps, a.mom,
                      a.alpha, d_vm);
  if constexpr (REF) {
    const float2 dd = volt_change(u, vm_old, -d_th, -d_vm);
    return make_float2(x.x + dd.x, x.y + dd.y);
  } else {
    return volt(r.th, r.vm);
  }
}

// Forward epilogue of one row (the arithmetic of fwd_body): I = Y V (refined:
// Y dV) with the outage taken out, x the gathered vector's own value, sp the
// specification; returns (dP, dQ), w and Q_calc.
template <class R, bool REF>
__device__ __forceinline__ typename Prec<R>::C res_fwd(const IterArgs<R>& a, int ty, typename Prec<R>::C x,
                                                       typename Prec<R>::C I, typename Prec<R>::C sp, float2 vr,
                                                       float4 rf, typename Prec<R>::C& w, R& Q, float& mx, bool track) {
  using C = typename Prec<R>::C;
  C v;
  R dP, dQ;
  if constexpr (REF) {
    const float2 d = refined_mismatch(x, I, vr, rf, v);
    dP = (ty != BUS_SLACK) ? d.x : R(0);
    dQ = (ty == BUS_PQ) ? d.y : R(0);
    Q = d.y;
  } else {
    v = x;
    const C S = power_of(v, I);
    Q = S.y;
    dP = (ty != BUS_SLACK) ? S.x - sp.x : R(0);
    dQ = (ty == BUS_PQ) ? Q - sp.y : R(0);
  }
  const R ca = a.inv_m2 * dP, cb = a.inv_m2 * dQ;
  w = w_of(ca, cb, v);
  if (track) {  // max |f| (a NaN counts as infinity): only the last iteration before a test needs it
    const float am = fmaxf(fabsf((float)dP), fabsf((float)dQ));
    mx = (am != am) ? __int_as_float(0x7f800000) : fmaxf(mx, am);
  }
  return mkc(dP, dQ);
}

// The outaged branch's block out of acc at its two rows (bits of `end`: 1
// from-bus, 2 to-bus); xo: the operand at the other end.
template <class R, class C>
__device__ __forceinline__ void res_outage(const IterArgs<R>& a, int k, int end, C x, C xo, C& acc) {
  if (end & 1) {
    cfms(acc, a.yff[k], x);
    cfms(acc, a.yft[k], xo);
  } else {
    cfms(acc, a.yft[k], xo);
    cfms(acc, a.ytt[k], x);
  }
}

}  // namespace dpf
