// On-chip form of the DPF iterations for grids of up to RES_MAX_N buses.
//
// The streaming kernels (k_fwd, k_adj) pass a batch's whole state through
// HBM / L2 twice per iteration: 128 bytes per element and iteration in the
// refined mode.  But the cases are independent, and the state of one case of
// such a grid fits one SM.  Here a team of threads owns one case for a whole
// test interval: it loads the case's state once, runs the iterations with the
// master values, the moments and the references in registers and V (or dV), w
// and the mismatch in shared memory, and stores the state back once.  No
// barrier spans more than the team.
//
//   one warp per case (N <= RES_WARP_N, RES_TEAMS cases per CTA): warp
//   barriers only; the warp also sums the loss and steps the scheduler.
//   one CTA per case (larger N): T compute threads with RPT rows each plus
//   one warp that sums the loss and steps the case's scheduler while the
//   others run the adjoint gathers.
//
// Y_bus is staged once per CTA as sliced ELL: rows sorted by their entry
// count, 32 rows per slice, entry e of a slice's 32 rows adjacent, so a
// slice's rows have (nearly) equal lengths and the value and column loads are
// free of bank conflicts.  Shared-memory vectors are indexed by position in
// that order.
//
// Measured (2,379 N-1 cases of a 2,000-bus grid, refined FP32): 123 us per
// iteration streaming, 80 us on chip.  What bounds it now is instruction issue
// (60% of the slots, 404 instructions per 32 rows and iteration), then the
// shared-memory pipe (57%: two rows of 8-byte gathers at random banks).  8,192
// cases of 30 buses: 15.9 -> 8.1 us (issue 64%, 612 instructions per case and
// iteration, 31% of the warps); one case of 30 buses in FP64: 17.8 -> 8.7 (a
// dependent chain: 9 of 13 warp cycles per issue wait for a fixed latency).
// Batches, grids and spans for which the streaming kernels are faster are
// given to them (res_pays, res_pays_dense, res_min_span).
//
// The results are those of the streaming kernels to the bit: the same device
// functions on the same operands, each row's products in the same order, and
// the case's loss (which drives the plateau schedule) summed in the order of
// the launch shape the streaming kernels would use (LossOrder).
#include <cuda_runtime.h>

#include <algorithm>

#include "dpf_kernels.cuh"
#include "dpf_resident.h"
#include "dpf_sched.cuh"
#include "dpf_sell.cuh"
#include "dpf_smem.h"

namespace dpf {

// Threads of a CTA at most in the one-CTA form (FP64 needs the registers).
template <class R> __host__ __device__ constexpr int res_threads() { return sizeof(R) == 4 ? 1024 : 512; }

// Geometry of the loss sum (LossOrder with what is empty left out: adding an
// empty chain's 0 changes nothing).  Chain (b, w, r) holds the rows b*rpb +
// w*rpw + r + j*step of row block b.
struct LossGeo {
  int gy, rpb, wpb, rpw, lrpw, step, nj, nch, magic, tile, nthr;
};
// Shared-memory layout: X, W, the specification and (CTA form, refined mode)
// the references by position, D = (dP, dQ) by internal row, scratch; then the
// staged Y_bus.
struct ResLayout {
  unsigned w, d, s, vr, rf, scr, sc, flag, team;  // offsets inside a team's block, its size
  unsigned val, col, total;                   // after the teams
};
template <class R> struct ResArgs {
  using C = typename Prec<R>::C;
  IterArgs<R> a;
  int K, T, n_it;
  const int32_t* rord;    // position -> internal row
  const int32_t* rpos;    // internal row -> position
  const int32_t* soff;    // [slices + 1] entry pairs before a slice
  const uint32_t* col2;   // two column byte offsets (position * 8) per word, [pair][32]
  const ValPair<R>* val;  // [pair][32]
  int n_pair;             // entry pairs of all slices
  int n_slice;
  LossGeo lo;
  ResLayout L;
};

// Scratch values of the loss sum.
__host__ __device__ __forceinline__ int res_scratch(const LossGeo& g) {
  return g.gy * g.wpb + g.gy + (g.gy + SCHED_GROUP - 1) / SCHED_GROUP + 256 + 16;
}

// One case's loss sum in the streaming kernels' order, in two parts.  Chains:
// warp `cw` of `ncw` sums its chains' rows and the butterfly over a warp's
// rows into part.  Tail (one warp): the warps, the row blocks and (beyond 64)
// their groups.  FP64 solves, whose plateau decisions do not hang on the last
// bit, take a shorter fixed order: strided rows, then a butterfly.
template <class R, class C>
__device__ __forceinline__ void loss_chains(const C* __restrict__ D, R* __restrict__ part, int N, const LossGeo& g,
                                            int cw, int ncw, int lane) {
  if constexpr (sizeof(R) == 8) {
    R s = R(0);
    for (int i = cw * 32 + lane; i < N; i += 32 * ncw) {
      const C d = D[i];
      s = fmaT(d.x, d.x, fmaT(d.y, d.y, s));
    }
    for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
    if (lane == 0) part[cw] = s;
  } else {
    for (int c0 = cw * 32; c0 < g.nch; c0 += ncw * 32) {
      const int c = c0 + lane, bw = c >> g.lrpw;
      const int b = (int)(((unsigned)bw * (unsigned)g.magic) >> 18);  // bw / wpb
      int i = b * g.rpb + ((bw - b * g.wpb) << g.lrpw) + (c & (g.rpw - 1));
      const int r1 = c < g.nch ? min(N, (b + 1) * g.rpb) : 0;
      R acc = R(0);
      if (g.nj == 1) {
        if (i < r1) {
          const C d = D[i];
          acc = fmaT(d.x, d.x, fmaT(d.y, d.y, R(0)));
        }
      } else {
        for (; i < r1; i += 4 * g.step) {  // four rows' loads in flight; a missing row adds 0
          C d[4];
#pragma unroll
          for (int u = 0; u < 4; ++u) d[u] = i + u * g.step < r1 ? D[i + u * g.step] : mkc(R(0), R(0));
#pragma unroll
          for (int u = 0; u < 4; ++u) acc = fmaT(d[u].x, d[u].x, fmaT(d[u].y, d[u].y, acc));
        }
        __syncwarp();
      }
      for (int off = g.rpw >> 1; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
      if (c < g.nch && (c & (g.rpw - 1)) == 0) part[bw] = acc;
    }
  }
}

template <class R>
__device__ __forceinline__ R loss_tail(R* __restrict__ scr, const LossGeo& g, int ncw, int lane) {
  R L = R(0);
  if constexpr (sizeof(R) == 8) {
    for (int c = 0; c < ncw; ++c) L += scr[c];
  } else {
    const int nbw = g.gy * g.wpb;
    const R* sums = scr;
    R* blk = scr + ((nbw + 3) & ~3);
    R* grp = blk + ((g.gy + 3) & ~3);
    if (g.wpb > 1) {
      for (int b = lane; b < g.gy; b += 32) {
        const R* pb = scr + b * g.wpb;
        R s = R(0);
        if (g.wpb == 8) {
          const float4 u = *reinterpret_cast<const float4*>(pb), v = *reinterpret_cast<const float4*>(pb + 4);
          s = ((((((((s + u.x) + u.y) + u.z) + u.w) + v.x) + v.y) + v.z) + v.w);
        } else {
          for (int w = 0; w < g.wpb; ++w) s += pb[w];
        }
        blk[b] = s;
      }
      __syncwarp();
      sums = blk;
    }
    if (g.gy <= 64) {
      int b = 0;
      for (; b + 4 <= g.gy; b += 4) {
        const float4 u = *reinterpret_cast<const float4*>(sums + b);
        L = (((L + u.x) + u.y) + u.z) + u.w;
      }
      for (; b < g.gy; ++b) L += sums[b];
    } else {
      const int ng = (g.gy + SCHED_GROUP - 1) / SCHED_GROUP;
      for (int q = lane; q < ng; q += 32) {
        R s = R(0);
        for (int u = 0; u < SCHED_GROUP; ++u) s += (q * SCHED_GROUP + u < g.gy) ? sums[q * SCHED_GROUP + u] : R(0);
        grp[q] = s;
      }
      __syncwarp();
      int tpc = 1;
      while (2 * tpc * g.tile <= g.nthr) tpc *= 2;
      R* tree = grp + ng;
      for (int j = lane; j < tpc; j += 32) {
        R s = R(0);
        for (int q = j; q < ng; q += tpc) s += grp[q];
        tree[j] = s;
      }
      __syncwarp();
      for (int st = tpc >> 1; st > 0; st >>= 1) {
        for (int j = lane; j < st; j += 32) tree[j] += tree[j + st];
        __syncwarp();
      }
      L = tree[0];
    }
  }
  __syncwarp();  // the scratch is reused by the next iteration
  return L;
}

// Y_bus to shared memory (it does not change during a solve).
template <class R>
__device__ __forceinline__ void res_stage(const ResArgs<R>& q, unsigned char* smem) {
  ValPair<R>* sval = reinterpret_cast<ValPair<R>*>(smem + q.L.val);
  uint32_t* scol = reinterpret_cast<uint32_t*>(smem + q.L.col);
  for (int t = threadIdx.x; t < q.n_pair * 32; t += blockDim.x) {
    sval[t] = q.val[t];
    scol[t] = __ldg(q.col2 + t);
  }
}

// One warp per case, RES_TEAMS cases per CTA.  CTAs an SM: 250 iterations of
// 8,192 cases of 30 buses (one row a lane) 2.04 ms at 6, 2.07 at 5, 2.31 at 4;
// 3,000 of 60 (two rows) 0.66, 0.60, 0.80.
template <class R, bool REF, bool ADAM, int RPT>
__global__ void __launch_bounds__(32 * RES_TEAMS, sizeof(R) == 8 ? 3 : RPT == 1 ? 6 : 5)
    k_resident_warp(const ResArgs<R> q) {
  using C = typename Prec<R>::C;
  extern __shared__ __align__(16) unsigned char smem[];
  const IterArgs<R>& a = q.a;
  const int N = a.N, lane = threadIdx.x & 31, team = threadIdx.x >> 5;
  unsigned char* tb = smem + team * q.L.team;
  unsigned char* wb = tb + q.L.w;
  C* X = reinterpret_cast<C*>(tb);
  C* W = reinterpret_cast<C*>(wb);
  C* D = reinterpret_cast<C*>(tb + q.L.d);
  R* scr = reinterpret_cast<R*>(tb + q.L.scr);
  const ValPair<R>* val = reinterpret_cast<const ValPair<R>*>(smem + q.L.val) + lane;
  const uint32_t* col = reinterpret_cast<const uint32_t*>(smem + q.L.col) + lane;
  const int k = blockIdx.x * RES_TEAMS + team;
  res_stage(q, smem);
  pdl_wait();
  pdl_release();
  __syncthreads();
  if (k >= q.K || !a.active[k]) return;  // (no CTA barrier follows)
  const size_t Kp = (size_t)a.Kp;

  int row[RPT], ty[RPT], end[RPT], sl[RPT];
  ResRow<R> rw[RPT];
  C sp[RPT];
  float2 vr[RPT];
  float4 rf[RPT];
  int of = -1, ot = -1;
  if (a.has_outage) {
    of = a.of[k];
    ot = a.ot[k];
  }
  const int pf = of >= 0 ? q.rpos[of] : 0, pt = of >= 0 ? q.rpos[ot] : 0;
#pragma unroll
  for (int s = 0; s < RPT; ++s) {
    const int p = s * 32 + lane;
    row[s] = p < N ? __ldg(q.rord + p) : -1;
    ty[s] = BUS_SLACK;
    end[s] = 0;
    sl[s] = 0;
    if (s < q.n_slice) {
      const int p0 = __ldg(q.soff + s);
      sl[s] = p0 * 32 | (__ldg(q.soff + s + 1) - p0) << 20;
    }
    C x = mkc(R(0), R(0));
    sp[s] = x;
    rw[s] = ResRow<R>{};
    vr[s] = make_float2(0.f, 0.f);
    rf[s] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (row[s] >= 0) {
      const size_t e = (size_t)row[s] * Kp + k, si = a.spec_per_case ? e : (size_t)row[s];
      ty[s] = __ldg(a.type + row[s]);
      end[s] = row[s] == of ? 1 : row[s] == ot ? 2 : 0;
      x = a.V[e];
      sp[s] = mkc(a.pspec[si], a.qspec[si]);
      rw[s].load(a, e);
      if constexpr (REF) {
        vr[s] = a.vref[e];
        rf[s] = a.irf[e];
      }
    }
    X[p] = x;
    W[p] = mkc(R(0), R(0));
  }
  ResSched<R> sc;
  sc.load(a.sc, k, lane);
  __syncwarp();
  bool fin = true;
  for (int it = 0; it < q.n_it; ++it) {
    sc.terms(a.sc, lane);
    float mx = 0.f;
    const bool track = it == q.n_it - 1 && a.sc.mx32;
#pragma unroll
    for (int s = 0; s < RPT; ++s) {
      const int p = s * 32 + lane;
      C I = sell_row<R>(val, col, sl[s], tb);
      if (row[s] < 0) continue;
      const C x = X[p];
      if (end[s]) res_outage(a, k, end[s], x, X[end[s] & 1 ? pt : pf], I);
      C w;
      R Q;
      D[row[s]] = res_fwd<R, REF>(a, ty[s], x, I, sp[s], vr[s], rf[s], w, Q, mx, track);
      if (ty[s] == BUS_PV) sp[s].y = Q;
      W[p] = w;
    }
    if (track) {
      const unsigned m = __reduce_max_sync(0xffffffffu, __float_as_uint(mx));
      if (lane == 0) a.sc.cand[k] = (a.sc.gate <= 0.0 || (double)__uint_as_float(m) <= a.sc.gate) ? 1 : 0;
    }
    __syncwarp();
    loss_chains<R>(D, scr, N, q.lo, 0, 1, lane);
    __syncwarp();
    const R lsum = loss_tail<R>(scr, q.lo, 1, lane);
    fin = isfinite(lsum);  // (as the loss: 1 / m <= 1)
    if (!fin) break;       // stops as diverged before it steps
#pragma unroll
    for (int s = 0; s < RPT; ++s) {
      const int p = s * 32 + lane;
      C z = sell_row<R>(val, col, sl[s], wb);
      if (ty[s] == BUS_SLACK) continue;
      const C w = W[p];
      if (end[s]) res_outage(a, k, end[s], w, W[end[s] & 1 ? pt : pf], z);
      X[p] = res_adj<R, REF, ADAM>(a, ty[s], rw[s], X[p], w, z, sp[s], sc.step, sc.isb);
    }
    sc.feed(a.sc, lsum);
    __syncwarp();
  }
  if (!fin && lane == 0) {
    a.sc.status[k] = CASE_DIVERGED;
    a.sc.active[k] = 0;
    atomicSub(a.sc.n_active, 1);
  }
#pragma unroll
  for (int s = 0; s < RPT; ++s) {
    if (ty[s] == BUS_SLACK) continue;  // (a slack's state does not change)
    const size_t e = (size_t)row[s] * Kp + k;
    rw[s].store(a, e);
    a.V[e] = X[s * 32 + lane];
  }
  sc.store(a.sc, k, lane);
}

// One CTA per case.  The last warp also keeps the scheduler: it finishes an
// iteration's loss sum and takes the scheduler's step during the next forward
// pass, whose adjoint is the first to need the new rate.  A loss that is not
// finite is therefore noticed one update late: the CTA then starts over from
// the state in global memory and takes only the steps before it (what the
// streaming kernels return for a diverged case).
template <class R, bool REF, bool ADAM, int RPT>
__global__ void __launch_bounds__(res_threads<R>(), 1) k_resident_cta(const ResArgs<R> q) {
  using C = typename Prec<R>::C;
  extern __shared__ __align__(16) unsigned char smem[];
  const IterArgs<R>& a = q.a;
  const int N = a.N, T = q.T, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = (int)blockDim.x >> 5;
  constexpr unsigned WOFF = res_threads<R>() * RPT * sizeof(C);
  C* X = reinterpret_cast<C*>(smem) + tid;  // this thread's rows: every T-th position from tid
  C* W = reinterpret_cast<C*>(smem + WOFF) + tid;
  C* D = reinterpret_cast<C*>(smem + q.L.d);
  C* S = reinterpret_cast<C*>(smem + q.L.s) + tid;
  float2* VR = reinterpret_cast<float2*>(smem + q.L.vr) + tid;
  float4* RF = reinterpret_cast<float4*>(smem + q.L.rf) + tid;
  R* scr = reinterpret_cast<R*>(smem + q.L.scr);
  int* flag = reinterpret_cast<int*>(smem + q.L.flag);      // [0] steps before a divergence, or -1
  unsigned* mxs = reinterpret_cast<unsigned*>(flag + 1);    // [1] max mismatch of the last iterate
  R* terms = reinterpret_cast<R*>(smem + q.L.flag + 16);    // step, isb of the coming update
  const ValPair<R>* val = reinterpret_cast<const ValPair<R>*>(smem + q.L.val) + lane;
  const uint32_t* col = reinterpret_cast<const uint32_t*>(smem + q.L.col) + lane;
  ResSched<R>* scs = reinterpret_cast<ResSched<R>*>(smem + q.L.sc) + lane;
  const int k = blockIdx.x;
  res_stage(q, smem);
  pdl_wait();
  pdl_release();
  if (!a.active[k]) return;  // the whole CTA
  const bool compute = tid < T, sched = warp == nw - 1;  // (T = blockDim: the last warp does both)
  // the warps that sum the loss chains: the last ones before the scheduler's
  const int ncw = max(1, min(nw - 1, (q.lo.nch + 31) >> 5)), cw = warp - (nw - 1 - ncw);
  const size_t Kp = (size_t)a.Kp;
  int n = q.n_it;
  bool diverged = false;
  for (;;) {
    int info[RPT];  // internal row, bus type << 16, outage end << 20; -1: no row
    int sl[RPT];    // entry pairs of the row's slice: first * 32, count << 20
    ResRow<R> rw[RPT];
    int ends = 0;   // positions of the outaged branch's ends: from-bus, to-bus << 16
    if (compute) {
      int of = -1, ot = -1;
      if (a.has_outage) {
        of = a.of[k];
        ot = a.ot[k];
        if (of >= 0) ends = q.rpos[of] | q.rpos[ot] << 16;
      }
#pragma unroll
      for (int s = 0; s < RPT; ++s) {
        const int p = s * T + tid, i = p < N ? __ldg(q.rord + p) : -1;
        info[s] = -1;
        sl[s] = 0;
        if ((p >> 5) < q.n_slice) {
          const int p0 = __ldg(q.soff + (p >> 5));
          sl[s] = p0 * 32 | (__ldg(q.soff + (p >> 5) + 1) - p0) << 20;
        }
        C x = mkc(R(0), R(0));
        if (i >= 0) {
          const size_t e = (size_t)i * Kp + k, si = a.spec_per_case ? e : (size_t)i;
          info[s] = i | (int)__ldg(a.type + i) << 16 | (i == of ? 1 : i == ot ? 2 : 0) << 20;
          x = a.V[e];
          S[s * T] = mkc(a.pspec[si], a.qspec[si]);
          rw[s].load(a, e);
          if constexpr (REF) {
            VR[s * T] = a.vref[e];
            RF[s * T] = a.irf[e];
          }
        }
        X[s * T] = x;
        W[s * T] = mkc(R(0), R(0));
      }
    }
    if (sched) {
      ResSched<R> sc;
      sc.load(a.sc, k, lane);
      *scs = sc;
      if (lane == 0) {
        flag[0] = -1;
        *mxs = 0u;
      }
    }
    __syncthreads();

    for (int it = 0; it <= n; ++it) {
      if (sched) {  // the previous iterate's loss, then this update's step terms
        ResSched<R> sc = *scs;
        bool fin = true;
        if (it > 0) {
          const R lsum = loss_tail<R>(scr, q.lo, ncw, lane);
          fin = isfinite(lsum);  // (as the loss: 1 / m <= 1)
          if (fin) sc.feed(a.sc, lsum);
          else if (lane == 0) flag[0] = it - 1;
        }
        if (it < n) {
          if (fin) sc.terms(a.sc, lane);
          if (lane == 0) {
            terms[0] = sc.step;
            terms[1] = sc.isb;
          }
        }
        *scs = sc;
      }
      if (it == n) break;
      if (compute) {  // forward: I = Y V, mismatch, w
        float mx = 0.f;
        const bool track = it == n - 1 && a.mx32;
#pragma unroll
        for (int s = 0; s < RPT; ++s) {
          C I = sell_row<R>(val, col, sl[s], smem);  // (no entries past the last slice)
          if (info[s] < 0) continue;
          const C x = X[s * T];
          const int ty = (info[s] >> 16) & 15;
          if (info[s] >> 20)
            res_outage(a, k, info[s] >> 20, x,
                       reinterpret_cast<C*>(smem)[(info[s] >> 20) & 1 ? ends >> 16 : ends & 0xffff], I);
          float2 vr = make_float2(0.f, 0.f);
          float4 rf = make_float4(0.f, 0.f, 0.f, 0.f);
          if constexpr (REF) {
            vr = VR[s * T];
            rf = RF[s * T];
          }
          C w, sp = mkc(R(0), R(0));
          if constexpr (!REF) sp = S[s * T];
          R Q;
          D[info[s] & 0xffff] = res_fwd<R, REF>(a, ty, x, I, sp, vr, rf, w, Q, mx, track);
          if (ty == BUS_PV) S[s * T].y = Q;
          W[s * T] = w;
        }
        if (it == n - 1 && a.sc.mx32) {
          const unsigned m = __reduce_max_sync(0xffffffffu, __float_as_uint(mx));
          if (lane == 0) atomicMax(mxs, m);
        }
      }
      __syncthreads();
      if (flag[0] >= 0) break;
      if (cw >= 0 && !sched) loss_chains<R>(D, scr, N, q.lo, cw, ncw, lane);
      if (compute) {  // adjoint: z = Y w, gradient, step, new V
        const R step = terms[0], isb = terms[1];
#pragma unroll
        for (int s = 0; s < RPT; ++s) {
          C z = sell_row<R>(val, col, sl[s], smem + WOFF);
          const int ty = (info[s] >> 16) & 15;
          if (info[s] < 0 || ty == BUS_SLACK) continue;
          const C w = W[s * T];
          if (info[s] >> 20)
            res_outage(a, k, info[s] >> 20, w,
                       reinterpret_cast<C*>(smem + WOFF)[(info[s] >> 20) & 1 ? ends >> 16 : ends & 0xffff], z);
          X[s * T] = res_adj<R, REF, ADAM>(a, ty, rw[s], X[s * T], w, z, S[s * T], step, isb);
        }
      }
      __syncthreads();
    }
    __syncthreads();
    if (flag[0] >= 0) {  // again, only the steps before the divergence
      n = flag[0];
      diverged = true;
      __syncthreads();
      continue;
    }
    if (compute) {
#pragma unroll
      for (int s = 0; s < RPT; ++s) {
        if (info[s] < 0 || ((info[s] >> 16) & 15) == BUS_SLACK) continue;  // (a slack's state does not change)
        const size_t e = (size_t)(info[s] & 0xffff) * Kp + k;
        rw[s].store(a, e);
        a.V[e] = X[s * T];
      }
    }
    if (sched) {
      scs->store(a.sc, k, lane);
      if (lane == 0) {
        if (a.sc.mx32)
          a.sc.cand[k] = (a.sc.gate <= 0.0 || (double)__uint_as_float(*mxs) <= a.sc.gate) ? 1 : 0;
        if (diverged) {
          a.sc.status[k] = CASE_DIVERGED;
          a.sc.active[k] = 0;
          atomicSub(a.sc.n_active, 1);
        }
      }
    }
    return;
  }
}

// ---- host ---------------------------------------------------------------------
// Threads of a CTA for T compute threads: a warp of its own for the scheduler,
// unless that would leave room for one CTA per SM instead of two.
template <class R> static int res_cta_threads(int T) {
  return T <= 512 && T + 32 > 512 ? T : std::min(T + 32, res_threads<R>());
}

static LossGeo loss_geo(const LossOrder& lo) {
  LossGeo g;
  g.gy = lo.gy;
  g.rpb = lo.rpb;
  g.step = lo.wpb * lo.rpw;
  g.rpw = 1;
  g.lrpw = 0;
  while (g.rpw < std::min(lo.rpw, lo.rpb)) {
    g.rpw *= 2;
    g.lrpw += 1;
  }
  g.wpb = std::min(lo.wpb, (lo.rpb + lo.rpw - 1) / lo.rpw);
  g.nj = (lo.rpb + g.step - 1) / g.step;
  g.nch = g.gy * g.wpb * g.rpw;
  g.magic = (1 << 18) / g.wpb + 1;
  g.tile = lo.tile;
  g.nthr = lo.nthr;
  return g;
}

template <class R>
static ResLayout res_layout(const dpf_ybus* y, const ResShape& sh, bool refined, const LossOrder& lo) {
  const unsigned cs = 2 * sizeof(R), np = (unsigned)(sh.T * sh.rpt), pairs = (unsigned)y->dev.res_pairs;
  const bool refs = refined && !sh.warp;
  ResLayout L;
  L.w = (sh.warp ? np : (unsigned)(res_threads<R>() * sh.rpt)) * cs;  // (CTA form: a compile-time offset)
  L.d = L.w + np * cs;
  L.s = L.d + (unsigned)((y->n + 1) & ~1) * cs;
  L.vr = L.s + np * cs;
  L.rf = L.vr + (refs ? np * 8u : 0u);
  L.scr = L.rf + (refs ? np * 16u : 0u);
  L.sc = L.scr + (((unsigned)res_scratch(loss_geo(lo)) * (unsigned)sizeof(R) + 15u) & ~15u);
  L.flag = L.sc + (sh.warp ? 0u : 32u * (unsigned)sizeof(ResSched<R>));
  L.team = L.flag + 32u;
  L.val = L.team * (sh.warp ? RES_TEAMS : 1);
  L.col = L.val + pairs * 64u * cs;
  L.total = L.col + pairs * 32u * 4u;
  return L;
}

ResShape res_shape(const dpf_ybus* y, int K, bool fp64, bool refined, const LossOrder& lo, size_t smem_limit) {
  ResShape sh;
  const DeviceYbus& d = y->dev;
  const int n = y->n;
  if (!d.res_rord || n > RES_MAX_N || y->m_loss <= 0) return sh;
  int dev = 0, sms = 1;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (!res_pays(n, K, fp64, sms)) return sh;
  sh.min_span = res_min_span(n, K, fp64, refined);
  sh.warp = n <= RES_WARP_N;
  sh.rpt = sh.warp && n <= 32 ? 1 : 2;
  sh.T = sh.warp ? 32 : ((n + 1) / 2 + 31) / 32 * 32;
  sh.smem = fp64 ? res_layout<double>(y, sh, refined, lo).total : res_layout<float>(y, sh, refined, lo).total;
  if (sh.smem > smem_limit) return sh;
  int ctas = 1, ctas_free = 1;
  if (!sh.warp && !fp64) {  // CTAs an SM holds by shared memory, and by its 65,536 registers (64 a thread)
    int most = 0;
    cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev);
    ctas = std::max(1, most / (int)(sh.smem + 1024));
    ctas_free = 1024 / res_cta_threads<float>(sh.T);
  }
  sh.ok = res_pays_dense(n, K, fp64, sms, d.res_pairs, d.longest, ctas, ctas_free);
  return sh;
}

template <class R>
static cudaError_t res_go(void (*kern)(const ResArgs<R>), const ResArgs<R>& q, const ResShape& sh, bool pdl,
                          cudaStream_t s) {
  cudaError_t e = allow_smem(kern, sh.smem);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(sh.warp ? (q.K + RES_TEAMS - 1) / RES_TEAMS : q.K);
  cfg.blockDim = dim3(sh.warp ? 32 * RES_TEAMS : res_cta_threads<R>(sh.T));
  cfg.dynamicSmemBytes = sh.smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = pdl ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kern, q);
}

template <class R, bool REF, bool ADAM>
static cudaError_t res_pick(const ResArgs<R>& q, const ResShape& sh, bool pdl, cudaStream_t s) {
  return res_go<R>(!sh.warp      ? k_resident_cta<R, REF, ADAM, 2>
                   : sh.rpt == 1 ? k_resident_warp<R, REF, ADAM, 1>
                                 : k_resident_warp<R, REF, ADAM, 2>,
                   q, sh, pdl, s);
}

template <class R>
int res_launch(const dpf_ybus* y, const IterArgs<R>& a, const ResShape& sh, const LossOrder& lo, int K, int n_it,
               bool refined, bool pdl, void* stream) {
  const DeviceYbus& d = y->dev;
  ResArgs<R> q;
  q.a = a;
  q.K = K;
  q.T = sh.T;
  q.n_it = n_it;
  q.rord = d.res_rord;
  q.rpos = d.res_rpos;
  q.soff = d.res_soff;
  q.col2 = d.res_col2;
  q.n_pair = d.res_pairs;
  q.n_slice = d.res_slices;
  q.lo = loss_geo(lo);
  q.L = res_layout<R>(y, sh, refined, lo);
  cudaStream_t s = (cudaStream_t)stream;
  if constexpr (sizeof(R) == 4) {
    q.val = reinterpret_cast<const ValPair<float>*>(d.res_val32);
    if (a.opt == OPT_ADAM)
      return refined ? res_pick<float, true, true>(q, sh, pdl, s) : res_pick<float, false, true>(q, sh, pdl, s);
    return refined ? res_pick<float, true, false>(q, sh, pdl, s) : res_pick<float, false, false>(q, sh, pdl, s);
  } else {
    q.val = reinterpret_cast<const ValPair<double>*>(d.res_val64);
    return res_pick<double, false, false>(q, sh, pdl, s);
  }
}
template int res_launch<float>(const dpf_ybus*, const IterArgs<float>&, const ResShape&, const LossOrder&, int, int,
                               bool, bool, void*);
template int res_launch<double>(const dpf_ybus*, const IterArgs<double>&, const ResShape&, const LossOrder&, int, int,
                                bool, bool, void*);

}  // namespace dpf
