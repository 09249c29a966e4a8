// Layout of the set network's flat parameter vector and the first layer, shared
// by its forward and backward kernels.
#pragma once
#include "km_internal.cuh"

namespace km {
namespace {

constexpr int H = kSetH;
constexpr int kTileP = 64;  // points per pooled sum (the number of points of a set is a multiple)

struct NetOff {  // offsets of the parameters in the flat vector
  int W1, b1, W2, b2, W3, b3, W4, b4, total;
};
__host__ __device__ inline NetOff net_off(int d, int k) {
  NetOff o;
  o.W1 = 0;
  o.b1 = o.W1 + H * d;
  o.W2 = o.b1 + H;
  o.b2 = o.W2 + H * H;
  o.W3 = o.b2 + H;
  o.b3 = o.W3 + H * H;
  o.W4 = o.b3 + H;
  o.b4 = o.W4 + k * d * H;
  o.total = o.b4 + k * d;
  return o;
}

// h1 of one point and unit (the same expression forward and backward).
__device__ __forceinline__ float h1_of(const float* s_w1, const float (&xv)[3], int u) {
  const float4 w = *reinterpret_cast<const float4*>(s_w1 + 4 * u);  // W1[u][0..2] (0 past d), b1[u]
  return fmaxf(fmaf(w.z, xv[2], fmaf(w.y, xv[1], fmaf(w.x, xv[0], w.w))), 0.f);
}
__device__ __forceinline__ void stage_w1(float* s_w1, const float* __restrict__ prm, const NetOff& o, int d, int tid,
                                         int nth) {
  for (int q = tid; q < 4 * H; q += nth) {
    const int u = q >> 2, j = q & 3;
    s_w1[q] = j == 3 ? prm[o.b1 + u] : j < d ? prm[o.W1 + u * d + j] : 0.f;
  }
}

}  // namespace
}  // namespace km
