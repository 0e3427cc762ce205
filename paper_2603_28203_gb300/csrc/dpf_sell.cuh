// Row products of the sliced ELL form of Y_bus (DeviceYbus::res_*): 32 rows
// per slice, entries in pairs, columns as byte offsets (position * 8).
#pragma once

#include "dpf_kernels.cuh"

namespace dpf {

// Two adjacent entries of a row: their values, one aligned access.
template <class R> struct __align__(16) ValPair { typename Prec<R>::C a, b; };

// sum_e val[e] x[col[e]] over a row's entry pairs: even entries into a0, odd
// into a1, as row_spmv does (pads: weight 0 on the row itself).
// slice: the first pair's index | the number of pairs << 20; val and col2
// point at this lane's entries.
template <class R>
__device__ __forceinline__ typename Prec<R>::C sell_row(const ValPair<R>* __restrict__ val,
                                                        const uint32_t* __restrict__ col2, int slice,
                                                        const unsigned char* __restrict__ X) {
  using C = typename Prec<R>::C;
  constexpr unsigned sc = sizeof(C) / 8;
  C a0 = mkc(R(0), R(0)), a1 = a0;
  val += slice & 0xfffff;
  col2 += slice & 0xfffff;
#pragma unroll 2
  for (int n = slice >> 20; n > 0; --n, val += 32, col2 += 32) {
    const uint32_t cc = *col2;
    const ValPair<R> y = *val;
    const C x0 = *reinterpret_cast<const C*>(X + (cc & 0xffffu) * sc);
    const C x1 = *reinterpret_cast<const C*>(X + (cc >> 16) * sc);
    cfma(a0, y.a, x0);
    cfma(a1, y.b, x1);
  }
  return mkc(a0.x + a1.x, a0.y + a1.y);
}

template <class R> __device__ __forceinline__ ValPair<R> ldg_pair(const ValPair<R>* p);
template <> __device__ __forceinline__ ValPair<float> ldg_pair<float>(const ValPair<float>* p) {
  const float4 t = __ldg(reinterpret_cast<const float4*>(p));
  return ValPair<float>{make_float2(t.x, t.y), make_float2(t.z, t.w)};
}
template <> __device__ __forceinline__ ValPair<double> ldg_pair<double>(const ValPair<double>* p) {
  const double2* t = reinterpret_cast<const double2*>(p);
  return ValPair<double>{__ldg(t), __ldg(t + 1)};
}

// The same with the entries in global memory (read-only, shared by all CTAs).
template <class R>
__device__ __forceinline__ typename Prec<R>::C sell_row_g(const ValPair<R>* __restrict__ val,
                                                          const uint32_t* __restrict__ col2, int p0, int p1,
                                                          const unsigned char* __restrict__ X) {
  using C = typename Prec<R>::C;
  constexpr unsigned sc = sizeof(C) / 8;
  C a0 = mkc(R(0), R(0)), a1 = a0;
  for (int p = p0; p < p1; p += 32) {
    const uint32_t cc = __ldg(col2 + p);
    const ValPair<R> y = ldg_pair(val + p);
    cfma(a0, y.a, *reinterpret_cast<const C*>(X + (cc & 0xffffu) * sc));
    cfma(a1, y.b, *reinterpret_cast<const C*>(X + (cc >> 16) * sc));
  }
  return mkc(a0.x + a1.x, a0.y + a1.y);
}

}  // namespace dpf
