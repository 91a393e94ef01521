#pragma once
#include "rmt_kernels.h"

namespace {

// All bodies of a step run in one launch per pass (grid row y = body): a body of its own takes 27 launches a
// step, most of them shorter than a launch, and streams beside each other overlap them only in part.  The
// passes of one step, with a stream per body and so: 20 bodies in 128^3 879 -> 446 us, 3 in 48^3 170 -> 121 us,
// 8 in 256^3 717 -> 554 us (FP32).  A block's body and its arrays, staged once:
template <typename T>
struct BandCtx {
  Body b;
  Band<T> a;
};
template <typename T>
__device__ __forceinline__ void load_ctx(const BandSet<T>& S, BandCtx<T>& c) {
  const int m = S.m0 + blockIdx.y;
  const int* bs = reinterpret_cast<const int*>(S.bodies ? S.bodies + m : &S.one);
  const int* as = reinterpret_cast<const int*>(S.bodies ? S.bands + m : &S.oneb);
  static_assert(sizeof(Body) % 4 == 0 && sizeof(Band<T>) % 4 == 0, "copied as words");
  for (int t = threadIdx.x; t < (int)(sizeof(Body) / 4); t += blockDim.x) reinterpret_cast<int*>(&c.b)[t] = bs[t];
  for (int t = threadIdx.x; t < (int)(sizeof(Band<T>) / 4); t += blockDim.x) reinterpret_cast<int*>(&c.a)[t] = as[t];
  __syncthreads();
}
template <typename T>
__device__ __forceinline__ Win band_win(const Geo& g, const BandSet<T>& S, const BandCtx<T>& c) {
  return make_win(g, S.in >= 0 ? c.a.bb + 6 * S.in : nullptr, 2);
}

}  // namespace
