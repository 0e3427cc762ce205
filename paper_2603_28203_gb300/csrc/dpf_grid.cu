// Whole-GPU form of the FP32 iterations for grids above RES_MAX_N buses with
// about one element per thread of the GPU (see grid_shape): one persistent
// launch per test interval.
//
// The streaming kernels spend two launches per iteration on such batches, most
// of it launch and drain latency (one case of 100,000 buses: 17.3 us for 6 MB
// of state).  Here every SM runs one CTA that keeps its rows' master values
// and moments in shared memory for the whole interval; only V and w, which
// other SMs gather, live in L2 (read past L1, which is not coherent).  Two
// grid barriers (about 1.6 us each) separate the passes: 11.3 us.  What bounds
// it is the barriers and the chain of L2 reads of a pass (of 28 warp cycles per
// issue 15 are spent at a barrier, 7 on a load; issue 22%, L2 13%).
//
// Work is split as the streaming forward pass splits it: virtual blocks (case
// tile x row block) of `wpb` warps, dealt to the CTAs, a warp per virtual
// warp, so the loss partials and their order are the same and the results are
// the streaming kernels' to the bit.  One warp per case, somewhere in the
// grid, sums the case's partials during the adjoint pass and takes the
// scheduler's step for the next iteration.  A loss that may not be finite is
// flagged by the block that sees a partial above 1e30: only then do the
// adjoint's threads form the exact sum before they step.
//
// The barrier needs every CTA resident (a cooperative launch: the driver
// refuses what does not fit), and its wait gives up after a limit, sets an
// error flag and the CTA returns, as later launches of the solve do at once; the
// host reads the flag with the active count and at the solve's end.
#include <cuda_runtime.h>

#include <algorithm>

#include "dpf_kernels.cuh"
#include "dpf_resident.h"
#include "dpf_sched.cuh"
#include "dpf_smem.h"

namespace dpf {

struct GridArgs {
  IterArgs<float> a;
  int K, n_it, wpb, rpw, lanes, gy, gx, rpb;  // gx: case tiles that hold cases
  int vb_per_cta, workers;
  int tile, nthr;         // of the streaming scheduler (order of the group tree)
  float* terms;           // [2][2][Kp] step and 1 / sqrt(1 - beta2^t), by iteration parity
  unsigned* suspect;      // [Kp]
  unsigned* bar;          // arrivals of this launch, whether a case is suspect (both zeroed)
  int32_t* err;           // a barrier gave up (sticky for the solve)
  int polls;              // of a barrier before it gives up
};

constexpr int GRID_WARPS = 32;  // of a CTA at most

// Grid barrier number `gen` (1, 2, ...): 0 if it gave up, else 1 + the word
// beside the counter (whether any case is suspect).
__device__ __forceinline__ int grid_barrier(unsigned* bar, unsigned gen, int32_t* err, int polls) {
  __shared__ int ok;
  __syncthreads();
  if (threadIdx.x == 0) {
    const unsigned want = gen * gridDim.x;
    __threadfence();
    atomicAdd(bar, 1u);
    int n = 0;
    unsigned v;
    do {
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(bar) : "memory");
    } while (v < want && ++n < polls);
    ok = v >= want ? 1 + (int)__ldcg(bar + 1) : 0;
    if (!ok) *err = 1;
    __threadfence();
  }
  __syncthreads();
  return ok;
}

// The case's loss sum from its row blocks' partials, in the order of
// tile_sched: directly up to 64 blocks, else groups of SCHED_GROUP, then the
// strided tree over tpc <= 256 sums (lane l holds sums l, l + 32, ...).  One
// warp, all lanes get it.
__device__ __noinline__ float grid_loss(const float* __restrict__ part, int gy, int Kp, int k, int tile, int nthr,
                                           int lane) {
  if (gy <= 64) {
    float L = 0.f, v[2];
#pragma unroll
    for (int u = 0; u < 2; ++u) v[u] = lane + 32 * u < gy ? __ldcg(part + (size_t)(lane + 32 * u) * Kp + k) : 0.f;
    for (int b = 0; b < gy; ++b) L += __shfl_sync(0xffffffffu, b < 32 ? v[0] : v[1], b & 31);
    return L;
  }
  const int ng = (gy + SCHED_GROUP - 1) / SCHED_GROUP;
  int tpc = 1;
  while (2 * tpc * tile <= nthr) tpc *= 2;
  float v[8];
#pragma unroll
  for (int m = 0; m < 8; ++m) {
    const int j = lane + 32 * m;
    v[m] = 0.f;
    if (j < tpc)
      for (int q = j; q < ng; q += tpc) {
        float p[SCHED_GROUP], s = 0.f;
#pragma unroll
        for (int u = 0; u < SCHED_GROUP; ++u)
          p[u] = q * SCHED_GROUP + u < gy ? __ldcg(part + (size_t)(q * SCHED_GROUP + u) * Kp + k) : 0.f;
#pragma unroll
        for (int u = 0; u < SCHED_GROUP; ++u) s += p[u];
        v[m] += s;
      }
  }
#pragma unroll
  for (int st = 4; st > 0; st >>= 1)
    if (tpc > 32 * st)
#pragma unroll
      for (int m = 0; m < st; ++m) v[m] += v[m + st];
  for (int st = 16; st > 0; st >>= 1) {
    const float o = __shfl_down_sync(0xffffffffu, v[0], st);
    if (tpc > st) v[0] += o;
  }
  return __shfl_sync(0xffffffffu, v[0], 0);
}

// acc = sum of a row's padded entries times X (element offset col * Kp from
// this case's first), past L1; the order of row_spmv.
__device__ __forceinline__ float2 grid_row(const int4* __restrict__ ent, int p0, int p1, unsigned Kp,
                                           const float2* __restrict__ X) {
  float2 a0 = make_float2(0.f, 0.f), a1 = a0;
  for (int p = p0; p < p1; p += 4) {
    int4 e[4];
    float2 x[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) e[u] = __ldg(ent + p + u);
#pragma unroll
    for (int u = 0; u < 4; ++u) x[u] = __ldcg(X + (unsigned)e[u].x * Kp);
#pragma unroll
    for (int u = 0; u < 4; ++u)
      cfma((u & 1) ? a1 : a0, make_float2(__int_as_float(e[u].y), __int_as_float(e[u].z)), x[u]);
  }
  return make_float2(a0.x + a1.x, a0.y + a1.y);
}

template <bool REF, bool ADAM>
__global__ void __launch_bounds__(GRID_WARPS * 32, 1) k_grid_resident(const GridArgs q) {
  extern __shared__ __align__(16) unsigned char smem[];
  const IterArgs<float>& a = q.a;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = q.workers;
  const bool sched = warp == (int)(blockDim.x >> 5) - 1;  // the last warp keeps the schedulers (and may work too)
  const bool work = warp < nw;
  const int nvb = q.gx * q.gy, cells = q.rpb * q.lanes;  // elements of a virtual block
  float4* MS = reinterpret_cast<float4*>(smem);
  float4* OS = MS + (size_t)q.vb_per_cta * cells;
  float* red = reinterpret_cast<float*>(OS + (size_t)q.vb_per_cta * cells);  // [vb][wpb][lanes]
  const unsigned Kp = (unsigned)a.Kp;
  const int kl = lane & (q.lanes - 1), rsub = lane / q.lanes, step = q.wpb * q.rpw;
  // no case runs (the same for every CTA: nothing changes it before the first
  // barrier), or an earlier interval or another CTA of this one gave up (the
  // state is lost); one thread reads, so that the whole CTA leaves or none of it
  const int gone = threadIdx.x == 0 ? (__ldcg(a.n_active) == 0) | (__ldcg(q.err) != 0) : 0;
  if (__syncthreads_or(gone)) return;
  const int tasks = q.vb_per_cta * q.wpb;
  // task -> its case, rows i0, i0 + step, ... < r1, and the cell of row 0
  struct Task {
    int k, i0, r1, c;
    bool on;
  };
  auto task = [&](int t) {
    Task x;
    const int vb = t / q.wpb, w = t - vb * q.wpb, v = vb * (int)gridDim.x + (int)blockIdx.x;
    const int tile = v / q.gy, r0 = (v - tile * q.gy) * q.rpb;
    x.k = tile * q.lanes + kl;
    x.r1 = min(a.N, r0 + q.rpb);
    x.i0 = r0 + w * q.rpw + rsub;
    x.c = vb * cells - r0 * q.lanes + kl;
    x.on = v < nvb && x.k < q.K;
    return x;
  };
  // the specification; per case past L1, which keeps the rows of Y_bus
  auto spec = [&](unsigned i) {
    return a.spec_per_case ? make_float2(__ldcg(a.pspec + i), __ldcg(a.qspec + i))
                           : make_float2(__ldg(a.pspec + i), __ldg(a.qspec + i));
  };
  // state in; a case that is not active is left out of everything below
  // bit j: this lane's case of the warp's j-th task was active, and still runs
  unsigned act0 = 0, live;
  for (int t = warp, j = 0; work && t < tasks; t += nw, ++j) {
    const Task x = task(t);
    if (!x.on || !__ldcg(a.active + x.k)) continue;
    act0 |= 1u << j;
    for (int i = x.i0; i < x.r1; i += step) {
      const unsigned e = (unsigned)i * Kp + x.k;
      const int c = x.c + i * q.lanes;
      MS[c] = __ldcs(a.ms + e);
      const Mom<float> o = mom_load(a.os + e);
      OS[c] = make_float4(o.m1, o.v1, o.m2, o.v2);
    }
  }
  // schedulers: case k belongs to CTA k % gridDim (their state stays in global
  // memory between iterations, terms of iteration 0 first)
  auto owned = [&](auto&& f) {
    if (sched)
      for (int k = blockIdx.x; k < q.K; k += gridDim.x) f(k);
  };
  auto write_terms = [&](int k, int parity, const ResSched<float>& sc) {
    if (lane == 0) {
      q.terms[(size_t)(2 * parity) * Kp + k] = sc.step;
      q.terms[(size_t)(2 * parity + 1) * Kp + k] = sc.isb;
    }
  };
  owned([&](int k) {
    if (!__ldcg(a.active + k)) return;
    ResSched<float> sc;
    sc.load(a.sc, k, lane);
    sc.terms(a.sc, lane);
    sc.store(a.sc, k, lane);
    write_terms(k, 0, sc);
  });
  live = act0;
  unsigned gen = 0;
  for (int it = 0; it < q.n_it; ++it) {
    const bool last = it == q.n_it - 1;
    for (int t = warp, j = 0; work && t < tasks; t += nw, ++j) {  // ---- forward
      const Task x = task(t);
      const bool on = (live >> j) & 1;
      float acc = 0.f, mx = 0.f;
      if (on) {
        const int of = a.has_outage ? __ldg(a.of + x.k) : -1, ot = a.has_outage ? __ldg(a.ot + x.k) : -1;
        for (int i = x.i0; i < x.r1; i += step) {
          const unsigned e = (unsigned)i * Kp + x.k;
          const int ty = __ldg(a.type + i);
          const float2 xi = __ldcg(a.V + e);
          float2 vr = make_float2(0.f, 0.f), sp = vr;
          float4 rf = make_float4(0.f, 0.f, 0.f, 0.f);
          if constexpr (REF) {
            vr = __ldcg(a.vref + e);
            rf = __ldcg(a.irf + e);
          } else {
            sp = spec(a.spec_per_case ? e : (unsigned)i);
          }
          float2 I = grid_row(a.pent, __ldg(a.prp + i), __ldg(a.prp + i + 1), Kp, a.V + x.k), w;
          if (i == of) res_outage(a, x.k, 1, xi, __ldcg(a.V + (unsigned)ot * Kp + x.k), I);
          else if (i == ot) res_outage(a, x.k, 2, xi, __ldcg(a.V + (unsigned)of * Kp + x.k), I);
          float Q;
          const float2 d = res_fwd<float, REF>(a, ty, xi, I, sp, vr, rf, w, Q, mx, last);
          __stcg(a.W + e, w);
          if (ty == BUS_PV) __stcg(a.qpv + e, Q);
          acc = fmaf(d.x, d.x, fmaf(d.y, d.y, acc));
        }
      }
      for (int off = 16; off >= q.lanes; off >>= 1) {
        acc += __shfl_xor_sync(0xffffffffu, acc, off);
        mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, off));
      }
      if (lane < q.lanes) {
        red[t * q.lanes + lane] = acc;
        if (last && a.mx32 && on && mx > 0.f) atomicMax(a.mx32 + x.k, __float_as_uint(mx));
      }
    }
    __syncthreads();
    for (int t = threadIdx.x; t < q.vb_per_cta * q.lanes; t += blockDim.x) {  // the row blocks' partials
      const int vb = t / q.lanes, l = t - vb * q.lanes, v = vb * (int)gridDim.x + (int)blockIdx.x;
      const int tile = v / q.gy, k = tile * q.lanes + l;
      if (v >= nvb || k >= q.K) continue;
      float s = 0.f;
      for (int w = 0; w < q.wpb; ++w) s += red[(vb * q.wpb + w) * q.lanes + l];
      __stcg(a.loss_part + (size_t)(v - tile * q.gy) * Kp + k, s);
      if (!(s <= 1e30f)) {  // (below it the whole sum is finite)
        atomicOr(q.suspect + k, 1u);
        atomicOr(q.bar + 1, 1u);
      }
    }
    const int passed = grid_barrier(q.bar, ++gen, q.err, q.polls);
    if (!passed) return;
    const int par = it & 1;
    for (int t = warp, j = 0; work && t < tasks; t += nw, ++j) {  // ---- adjoint
      const Task x = task(t);
      bool on = (live >> j) & 1;
      const unsigned sus = on && passed > 1 ? __ldcg(q.suspect + x.k) : 0u;
      const float st = on ? __ldcg(q.terms + (unsigned)(2 * par) * Kp + x.k) : 0.f;
      const float isb = on ? __ldcg(q.terms + (unsigned)(2 * par + 1) * Kp + x.k) : 0.f;
      for (unsigned m = __ballot_sync(0xffffffffu, sus != 0u); m; m &= m - 1) {  // (rare) the exact verdict
        const int src = __ffs(m) - 1, k = __shfl_sync(0xffffffffu, x.k, src);
        const float L = grid_loss(a.loss_part, q.gy, a.Kp, k, q.tile, q.nthr, lane);
        if (lane == src && !isfinite(L)) on = false;  // it stops as diverged before it steps
      }
      if (!on) {
        live &= ~(1u << j);
        continue;
      }
      const int of = a.has_outage ? __ldg(a.of + x.k) : -1, ot = a.has_outage ? __ldg(a.ot + x.k) : -1;
      for (int i = x.i0; i < x.r1; i += step) {
        const int ty = __ldg(a.type + i);
        if (ty == BUS_SLACK) continue;
        const unsigned e = (unsigned)i * Kp + x.k;
        const float2 w = __ldcg(a.W + e), xv = __ldcg(a.V + e);
        float2 sp = spec(a.spec_per_case ? e : (unsigned)i);
        if (ty == BUS_PV) sp.y = __ldcg(a.qpv + e);
        float2 z = grid_row(a.pent, __ldg(a.prp + i), __ldg(a.prp + i + 1), Kp, a.W + x.k);
        if (i == of) res_outage(a, x.k, 1, w, __ldcg(a.W + (unsigned)ot * Kp + x.k), z);
        else if (i == ot) res_outage(a, x.k, 2, w, __ldcg(a.W + (unsigned)of * Kp + x.k), z);
        const int c = x.c + i * q.lanes;
        const float4 ms = MS[c], os = OS[c];
        ResRow<float> r;
        r.th = ms_th(ms);
        r.vm = ms_vm(ms);
        r.m1 = os.x;
        r.v1 = os.y;
        r.m2 = os.z;
        r.v2 = os.w;
        __stcg(a.V + e, res_adj<float, REF, ADAM>(a, ty, r, xv, w, z, sp, st, isb));
        MS[c] = ms_make(r.th, r.vm);
        OS[c] = make_float4(r.m1, r.v1, r.m2, r.v2);
      }
    }
    // ---- schedulers.  A case found diverged is switched off at once: the
    // adjoint's threads that read the flag early skip a step they skip anyway.
    owned([&](int k) {
      if (!__ldcg(a.active + k)) return;
      const float L = grid_loss(a.loss_part, q.gy, a.Kp, k, q.tile, q.nthr, lane);
      if (last && a.sc.mx32 && lane == 0) {
        a.sc.cand[k] = (a.sc.gate <= 0.0 || (double)__uint_as_float(__ldcg(a.mx32 + k)) <= a.sc.gate) ? 1 : 0;
        a.mx32[k] = 0u;
      }
      if (!isfinite(L)) {
        if (lane == 0) {
          a.sc.status[k] = CASE_DIVERGED;
          __stcg(a.sc.active + k, 0);
          atomicSub(a.sc.n_active, 1);
        }
        return;
      }
      ResSched<float> sc;
      sc.load(a.sc, k, lane);  // (the powers of this iteration's update, taken when its terms were)
      sc.feed(a.sc, L);
      if (!last) {
        sc.terms(a.sc, lane);
        write_terms(k, par ^ 1, sc);
      }
      sc.store(a.sc, k, lane);
    });
    if (!grid_barrier(q.bar, ++gen, q.err, q.polls)) return;
  }
  for (int t = warp, j = 0; work && t < tasks; t += nw, ++j) {  // state out
    if (!((act0 >> j) & 1)) continue;
    const Task x = task(t);
    for (int i = x.i0; i < x.r1; i += step) {
      const unsigned e = (unsigned)i * Kp + x.k;
      const int c = x.c + i * q.lanes;
      __stcs(a.ms + e, MS[c]);
      __stcs(reinterpret_cast<float4*>(a.os) + e, OS[c]);
    }
  }
  owned([&](int k) {
    if (lane == 0) q.suspect[k] = 0u;
  });
}

GridShape grid_shape(const dpf_ybus* y, int K, const LossOrder& lo, int lanes, size_t smem_limit) {
  GridShape g;
  if (y->n <= RES_MAX_N || y->m_loss <= 0) return g;
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  // About one element per thread of the GPU: there an iteration is launch and
  // drain latency.  us per iteration without the tests, streaming and here:
  // 1 x 100,000 buses 17.3 and 11.3, 1 x 20,000 13.2 and 9.5, 8 x 10,000 13.6
  // and 11.5, 16 x 10,000 15.6 and 13.0, 60 x 2,500 15.3 and 12.5, 4 x 40,000
  // 15.8 and 13.8.  With more elements per thread the gathers, which miss L1,
  // and issue bound both forms, and the gain shrinks: 2 x 100,000 18.9 and 17.7,
  // 96 x 10,000 32.5 and 29.5 with the limit lifted (it was set when this form
  // took 25.2 and 39.3 there; where it should lie now is not measured).
  if ((long long)y->n * K * 16 > (long long)sms * 1024 * 17) return g;
  // A long row is one lane's chain of reads past L1, with the whole GPU at the
  // barrier; the streaming kernels stage it in shared memory (one case: read it
  // through L1).  us per iteration, streaming and here, a bus of 160 and of 320
  // branches: 2 x 5,000 34.6 / 40.3, 55.5 / 71.6; 4 x 10,000 37.7 / 40.4, 61.0 / 83.7; 1 x
  // 2,500 35.2 / 36.9, 60.9 / 65.0; but 1 x 10,000 39.3 / 37.5, 67.0 / 63.6, and of 80
  // 12 x 10,000 28.4 / 25.3, 4 x 2,500 25.1 / 26.5.
  if (y->dev.longest > 64 && (K > 1 || y->n <= 5000)) return g;
  g.gx = (K + lanes - 1) / lanes;
  const long long nvb = (long long)g.gx * lo.gy;
  g.ctas = (int)std::min<long long>(sms, nvb);
  g.vb = (int)((nvb + g.ctas - 1) / g.ctas);
  const long long tasks = (long long)g.vb * lo.wpb;
  if (tasks > GRID_WARPS * 32) return g;
  const int rounds = (int)((tasks + GRID_WARPS - 1) / GRID_WARPS);
  g.workers = (int)((tasks + rounds - 1) / rounds);
  g.warps = std::min(GRID_WARPS, g.workers + 1);  // a warp of its own for the schedulers where one is free
  const long long bytes = (long long)g.vb * lanes * ((long long)lo.rpb * 32 + lo.wpb * 4);
  if (bytes > (long long)smem_limit - 1024) return g;  // (the barrier's flag)
  g.smem = (size_t)bytes;
  g.min_span = grid_min_span(K);
  g.ok = true;
  return g;
}

int grid_launch(const IterArgs<float>& a, const GridShape& g, const LossOrder& lo, int lanes, int K, int n_it,
                bool refined, float* terms, unsigned* suspect, unsigned* bar, int32_t* err, int64_t polls,
                void* stream) {
  cudaStream_t s = (cudaStream_t)stream;
  GridArgs q;
  q.a = a;
  q.K = K;
  q.n_it = n_it;
  q.wpb = lo.wpb;
  q.rpw = lo.rpw;
  q.lanes = lanes;
  q.gy = lo.gy;
  q.gx = g.gx;
  q.rpb = lo.rpb;
  q.vb_per_cta = g.vb;
  q.workers = g.workers;
  q.tile = lo.tile;
  q.nthr = lo.nthr;
  q.terms = terms;
  q.suspect = suspect;
  q.bar = bar;
  q.err = err;
  q.polls = (int)std::min<int64_t>(polls, 1 << 30);
  const bool adam = a.opt == OPT_ADAM;
  auto kern = refined ? (adam ? k_grid_resident<true, true> : k_grid_resident<true, false>)
                      : (adam ? k_grid_resident<false, true> : k_grid_resident<false, false>);
  cudaError_t e = allow_smem(kern, g.smem);
  if (e == cudaSuccess) e = cudaMemsetAsync(bar, 0, 2 * sizeof(unsigned), s);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(g.ctas);
  cfg.blockDim = dim3(g.warps * 32);
  cfg.dynamicSmemBytes = g.smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, q);
}

}  // namespace dpf
