// The k-means objective sum_i ||x_i - mu_{z_i}||^2 (the quantity Lloyd's
// iteration decreases; paper, section "The Lloyd's algorithm") of the
// current labels and centroids, in FP64: per point the squared distance with
// coordinates in order (no fused multiply-add), summed in a fixed order:
// thread t of a block adds points t, t + 256, ... of a 4096-point chunk, a
// tree adds the threads, and one block adds the chunk sums the same way.
#include <algorithm>

#include "km_internal.cuh"

namespace km {

namespace {

constexpr int kObjChunk = 4096;
constexpr int kObjThreads = 256;

// Sum of one value per thread, pairwise (t += t + 128, 64, ..., 1).
__device__ __forceinline__ double obj_tree(double v, double* s_red) {
  const int tid = threadIdx.x;
  s_red[tid] = v;
  __syncthreads();
  for (int w = kObjThreads / 2; w > 0; w >>= 1) {
    if (tid < w) s_red[tid] = __dadd_rn(s_red[tid], s_red[tid + w]);
    __syncthreads();
  }
  return s_red[0];
}

// One block per chunk.  (One warp per 65536 points, its distances added one
// after another by lane 0, is a chain of 65536 FP64 additions on 16 of 152
// SMs: 7.71 ms for 1e6 points in 3-D; the tree: 0.04 ms.  FP64 instructions
// bound it, 3 d + 1 a point.)
template <typename L>
__global__ void __launch_bounds__(kObjThreads) objective_kernel(const float* __restrict__ x, int64_t ld, int64_t n,
                                                                int d, const double* __restrict__ mu,
                                                                const L* __restrict__ z, double* __restrict__ part) {
  __shared__ double s_red[kObjThreads];
  const int64_t lo = (int64_t)blockIdx.x * kObjChunk, hi = min(lo + kObjChunk, n);
  double s = 0.0;
#pragma unroll 4
  for (int64_t i = lo + threadIdx.x; i < hi; i += kObjThreads) {
    const double* m = mu + (size_t)z[i] * d;
    double dv = 0.0;
    for (int j = 0; j < d; ++j) {
      const double t = __dsub_rn((double)x[(int64_t)j * ld + i], m[j]);
      dv = __dadd_rn(dv, __dmul_rn(t, t));
    }
    s = __dadd_rn(s, dv);
  }
  s = obj_tree(s, s_red);
  if (threadIdx.x == 0) part[blockIdx.x] = s;
}

__global__ void __launch_bounds__(kObjThreads) objective_sum_kernel(const double* __restrict__ part, int64_t nchunks,
                                                                    double* __restrict__ out) {
  __shared__ double s_red[kObjThreads];
  double s = 0.0;
#pragma unroll 8
  for (int64_t c = threadIdx.x; c < nchunks; c += kObjThreads) s = __dadd_rn(s, part[c]);
  s = obj_tree(s, s_red);
  if (threadIdx.x == 0) *out = s;
}

__global__ void widen_labels_kernel(const uint8_t* __restrict__ z8, int32_t* __restrict__ z, int64_t n) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    z[i] = z8[i];
}

}  // namespace

cudaError_t launch_widen_labels(const uint8_t* z8, int32_t* z, int64_t n, cudaStream_t st) {
  const int64_t blocks = std::max<int64_t>(1, std::min<int64_t>((n + 255) / 256, 8192));
  widen_labels_kernel<<<(unsigned)blocks, 256, 0, st>>>(z8, z, n);
  return cudaGetLastError();
}

int64_t objective_chunks(int64_t n) { return (n + kObjChunk - 1) / kObjChunk; }

cudaError_t launch_objective(const float* x, int64_t ld, int64_t n, int d, const double* mu, const int32_t* z,
                             const uint8_t* z8, double* part, double* out, cudaStream_t st) {
  const int64_t nch = objective_chunks(n);
  if (z8)
    objective_kernel<uint8_t><<<(unsigned)nch, kObjThreads, 0, st>>>(x, ld, n, d, mu, z8, part);
  else
    objective_kernel<int32_t><<<(unsigned)nch, kObjThreads, 0, st>>>(x, ld, n, d, mu, z, part);
  objective_sum_kernel<<<1, kObjThreads, 0, st>>>(part, nch, out);
  return cudaGetLastError();
}

}  // namespace km
