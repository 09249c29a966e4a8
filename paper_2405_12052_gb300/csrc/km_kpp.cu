// k-means++ seeding on the GPU (D^2 sampling, Arthur and Vassilvitskii
// 2007), the initialisation the configurations name for the start of
// Lloyd's algorithm (paper, section "The Lloyd's algorithm", step 1: initial
// centres).  The K uniforms are inputs, so a run is reproducible and the
// oracle can take the same ones.
//
// Pick 0 is floor(u_0 N).  Pick c >= 1: D^2_i = min over chosen centres
// of sum_j (x_ij - m_j)^2 in FP64 (coordinates in order, no fused
// multiply-add: the oracle's expression), total = sum_i D^2_i, target =
// u_c * total, and the pick is the first i whose running sum exceeds the
// target (the last point if none does).  The sums are taken over chunks of
// kKppChunk points (fixed-order tree per chunk), then over the chunk sums in
// order; so the pick equals a sequential scan's except when the target lies
// within FP64 rounding of a running-sum boundary.
#include "km_internal.cuh"

namespace km {

namespace {

constexpr int kKppChunk = 4096;
constexpr int kKppThreads = 256;

__device__ __forceinline__ double kpp_d2(const float* x, int64_t ld, int64_t i, int d, const double* m) {
  double acc = 0.0;
  for (int j = 0; j < d; ++j) {
    const double t = __dsub_rn((double)x[(int64_t)j * ld + i], m[j]);
    acc = __dadd_rn(acc, __dmul_rn(t, t));
  }
  return acc;
}

// An FP32 upper bound of a squared distance v >= 0 by integer arithmetic on
// its FP64 bits (a conversion would take the FP64 pipe): its leading 24 bits
// plus one ulp, at least 2^-126; from 2^127 on, +infinity.
__device__ __forceinline__ float kpp_up(double v) {
  const uint32_t hi = (uint32_t)__double2hiint(v), lo = (uint32_t)__double2loint(v);
  if (hi >= (1150u << 20)) return __uint_as_float(0x7f800000u);
  if (hi < (898u << 20)) return __uint_as_float(0x01000000u);
  return __uint_as_float((((hi - (896u << 20)) << 3) | (lo >> 29)) + 1u);
}

// D^2 against centre c (the minimum with the previous D^2 for c > 0) and the
// chunk sums.  One block per chunk; thread t sums points t, t + 256, ... of
// the chunk, then a fixed-order tree.
//
// FP64 instructions bound the plain form (11 a point and round: 2.73 ms a
// round for 1e8 points in 3-D, against 0.30 ms for reading the points and
// their D^2; with the screen below 0.71 ms on average over 31 rounds).  A centre is closer than the ones before for about 1 / c of the
// points only, so from the second centre on the distance is first formed in
// FP32: centres are points, so x - m is one rounding of the exact difference,
// and the FP32 sum is within (d + 2) 2^-24 relative of D^2 (plus underflow, at
// most d 2^-23 relative above 2^-126; KPP eps below covers both).  A point whose
// FP32 distance, reduced by that, is above its D^2 keeps it; the others are
// listed in shared memory and decided in FP64 by full warps (a warp that took
// them in place would pay the FP64 instructions for one lane in 32).  One
// FP64 addition a point is left, the chunk sum's, in the same order as before.
template <int D>
__global__ void __launch_bounds__(kKppThreads) kpp_d2_kernel(const float* __restrict__ x, int64_t ld, int64_t n,
                                                             int dd, const double* __restrict__ mu, int c,
                                                             double* __restrict__ d2, double* __restrict__ chunk_sum) {
  extern __shared__ __align__(16) double s_d2[];  // [kKppChunk]
  __shared__ double s_red[kKppThreads];
  __shared__ double s_m[D > 0 ? D : kMaxKppD];
  __shared__ float s_mf[D > 0 ? D : kMaxKppD];
  __shared__ unsigned short s_q[kKppChunk];
  __shared__ int s_n;
  const int d = D > 0 ? D : dd;
  const int tid = threadIdx.x, lane = tid & 31;
  if (tid < d) {
    s_m[tid] = mu[(size_t)c * d + tid];
    s_mf[tid] = (float)s_m[tid];  // exact: a centre is a point
  }
  if (tid == 0) s_n = 0;
  __syncthreads();
  const int64_t base = (int64_t)blockIdx.x * kKppChunk;
  const int m = (int)min((int64_t)kKppChunk, n - base);
  const float* xb = x + base;
  double* db = d2 + base;
  if (c == 0) {
    for (int q = tid; q < m; q += kKppThreads) {
      const double v = kpp_d2(x, ld, base + q, d, s_m);
      s_d2[q] = v;
      db[q] = v;
    }
  } else {
    const float keep = 1.f - (float)(3 * d + 8) * 0x1p-23f;
    float mf[D > 0 ? D : 1];
    if constexpr (D > 0) {
#pragma unroll
      for (int j = 0; j < D; ++j) mf[j] = s_mf[j];
    }
    // four rounds at a time, their loads issued before any is used
    constexpr int R = 4;
    for (int q0 = tid; q0 < kKppChunk; q0 += R * kKppThreads) {
      double v[R];
      float acc[R];
      if constexpr (D > 0) {
        float xv[R][D];
#pragma unroll
        for (int r = 0; r < R; ++r) {
          const int q = q0 + r * kKppThreads;
          v[r] = q < m ? db[q] : 0.0;
#pragma unroll
          for (int j = 0; j < D; ++j) xv[r][j] = q < m ? xb[(int64_t)j * ld + q] : 0.f;
        }
#pragma unroll
        for (int r = 0; r < R; ++r) {
          acc[r] = 0.f;
#pragma unroll
          for (int j = 0; j < D; ++j) {
            const float t = __fsub_rn(xv[r][j], mf[j]);
            acc[r] = __fmaf_rn(t, t, acc[r]);
          }
        }
      } else {
#pragma unroll
        for (int r = 0; r < R; ++r) {
          const int q = q0 + r * kKppThreads;
          v[r] = q < m ? db[q] : 0.0;
          acc[r] = 0.f;
        }
        for (int j = 0; j < d; ++j)
#pragma unroll
          for (int r = 0; r < R; ++r) {
            const int q = q0 + r * kKppThreads;
            const float t = __fsub_rn(q < m ? xb[(int64_t)j * ld + q] : 0.f, s_mf[j]);
            acc[r] = __fmaf_rn(t, t, acc[r]);
          }
      }
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const int q = q0 + r * kKppThreads;
        s_d2[q] = v[r];  // past m: 0, not read
        const bool need = q < m && !(acc[r] * keep > kpp_up(v[r]));
        const unsigned bal = __ballot_sync(0xffffffffu, need);
        if (bal) {
          int at = 0;
          if (lane == 0) at = atomicAdd(&s_n, __popc(bal));
          at = __shfl_sync(0xffffffffu, at, 0);
          if (need) s_q[at + __popc(bal & ((1u << lane) - 1u))] = (unsigned short)q;
        }
      }
    }
    __syncthreads();
    const int cnt = s_n;
    for (int e = tid; e < cnt; e += kKppThreads) {
      const int q = s_q[e];
      const double v = kpp_d2(x, ld, base + q, d, s_m);
      if (v < s_d2[q]) {
        s_d2[q] = v;
        db[q] = v;
      }
    }
  }
  __syncthreads();
  double acc = 0.0;
  for (int q = tid; q < m; q += kKppThreads) acc = __dadd_rn(acc, s_d2[q]);
  s_red[tid] = acc;
  __syncthreads();
  for (int w = kKppThreads / 2; w >= 32; w >>= 1) {
    if (tid < w) s_red[tid] = __dadd_rn(s_red[tid], s_red[tid + w]);
    __syncthreads();
  }
  if (tid < 32) {
    double t = s_red[tid];
#pragma unroll
    for (int w = 16; w > 0; w >>= 1) t = __dadd_rn(t, __shfl_down_sync(0xffffffffu, t, w));
    if (tid == 0) chunk_sum[blockIdx.x] = t;
  }
}

// Inclusive scan over the block's 1024 threads of one value each (warp scans,
// then the 32 warp totals): a fixed order.
__device__ __forceinline__ double block_scan(double v, double* s_w) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const double t = __shfl_up_sync(0xffffffffu, v, o);
    if (lane >= o) v = __dadd_rn(v, t);
  }
  __syncthreads();
  if (lane == 31) s_w[w] = v;
  __syncthreads();
  if (w == 0) {
    double t = s_w[lane];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const double u = __shfl_up_sync(0xffffffffu, t, o);
      if (lane >= o) t = __dadd_rn(t, u);
    }
    s_w[lane] = t;
  }
  __syncthreads();
  return w ? __dadd_rn(s_w[w - 1], v) : v;
}

// The first index whose running sum (before + the sums of v[0..i]) exceeds
// the target, or m: each thread adds a run of consecutive values, a block
// scan places the runs, and the first run that crosses is walked again.
// *below receives the running sum before that index.
__device__ int block_find(const double* __restrict__ v, int m, double before, double target, double* s_w,
                          double* below) {
  __shared__ int s_first;
  __shared__ int s_idx;
  __shared__ double s_below;
  const int run = (m + 1023) / 1024;
  const int lo = min(m, (int)threadIdx.x * run), hi = min(m, lo + run);
  double s = 0.0;
#pragma unroll 8
  for (int q = lo; q < hi; ++q) s = __dadd_rn(s, v[q]);
  if (threadIdx.x == 0) { s_first = 1024; s_idx = m; s_below = before; }
  const double incl = block_scan(s, s_w);
  if (hi > lo && __dadd_rn(before, incl) > target) atomicMin(&s_first, (int)threadIdx.x);
  // s_w is read by block_scan's last line in every thread before this barrier
  __syncthreads();
  const int f = s_first;
  // the running sum before run f: the inclusive sum of the run before it
  if ((int)threadIdx.x == f - 1) s_below = __dadd_rn(before, incl);
  __syncthreads();
  if ((int)threadIdx.x == f) {
    double b = s_below;
    int q = lo;
    for (; q < hi - 1; ++q) {  // the run's last value when rounding leaves none before it
      const double t = __dadd_rn(b, v[q]);
      if (t > target) break;
      b = t;
    }
    s_idx = q;
    s_below = b;
  }
  __syncthreads();
  *below = s_below;
  return s_idx;
}

// One block (1024 threads): the pick of round c and its coordinates.  The
// chunk sums are added in 32 segments, one per warp, the crossing segment is
// searched for its chunk and the chunk for its point.  (A Hillis-Steele scan
// of all chunk sums, two barriers per doubling: 157 us a round with 24414
// chunks; this: 25 us.)
__global__ void __launch_bounds__(1024) kpp_pick_kernel(const float* __restrict__ x, int64_t ld, int64_t n, int d,
                                                        const double* __restrict__ u, int c,
                                                        const double* __restrict__ chunk_sum, int nchunks,
                                                        const double* __restrict__ d2, double* mu, int64_t* idx) {
  __shared__ double s_w[32];
  __shared__ double s_seg[32];
  int64_t pick;
  if (c == 0) {
    pick = (int64_t)floor(u[0] * (double)n);
    if (pick >= n) pick = n - 1;
    if (pick < 0) pick = 0;
  } else {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int seg = (nchunks + 31) / 32;
    {
      const int hi = (int)min((int64_t)nchunks, (int64_t)(w + 1) * seg);
      double s = 0.0;
#pragma unroll 8
      for (int64_t q = (int64_t)w * seg + lane; q < hi; q += 32) s = __dadd_rn(s, chunk_sum[q]);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) s = __dadd_rn(s, __shfl_xor_sync(0xffffffffu, s, o));
      if (lane == 0) s_seg[w] = s;
    }
    __syncthreads();
    // every warp: the segments' running sums, the target and the segment
    double incl = s_seg[lane];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const double t = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl = __dadd_rn(incl, t);
    }
    const double target = __dmul_rn(u[c], __shfl_sync(0xffffffffu, incl, 31));
    const unsigned over = __ballot_sync(0xffffffffu, incl > target);
    if (over == 0u) {
      pick = n - 1;  // no running sum exceeds the target
    } else {
      const int f = __ffs((int)over) - 1;
      double before = f > 0 ? __shfl_sync(0xffffffffu, incl, f - 1) : 0.0;
      const int64_t s0 = (int64_t)f * seg;
      const int ms = (int)(min((int64_t)nchunks, s0 + seg) - s0);
      // the segment's last chunk when rounding leaves none in it
      const int64_t b = s0 + min(block_find(chunk_sum + s0, ms, before, target, s_w, &before), ms - 1);
      const int64_t i0 = b * kKppChunk;
      const int m = (int)min((int64_t)kKppChunk, n - i0);
      double unused;
      __syncthreads();
      pick = i0 + min(block_find(d2 + i0, m, before, target, s_w, &unused), m - 1);  // likewise its last point
    }
  }
  if ((int)threadIdx.x < d) mu[(size_t)c * d + threadIdx.x] = (double)x[(int64_t)threadIdx.x * ld + pick];
  if (threadIdx.x == 0) idx[c] = pick;
}

template <int D>
cudaError_t launch_d2(const float* x, int64_t ld, int64_t n, int d, const double* mu, int c, double* d2,
                      double* chunk_sum, int nch, cudaStream_t st) {
  kpp_d2_kernel<D><<<nch, kKppThreads, sizeof(double) * kKppChunk, st>>>(x, ld, n, d, mu, c, d2, chunk_sum);
  return cudaGetLastError();
}

}  // namespace

int64_t kpp_chunks(int64_t n) { return (n + kKppChunk - 1) / kKppChunk; }

cudaError_t launch_kmeanspp(const float* x, int64_t ld, int64_t n, int d, int k, const double* u, double* mu,
                            int64_t* idx, double* d2, double* chunk_sum, cudaStream_t st) {
  const int nch = (int)kpp_chunks(n);
  for (int c = 0; c < k; ++c) {
    if (c > 0) {
      cudaError_t e;
      switch (d) {
        case 1: e = launch_d2<1>(x, ld, n, d, mu, c - 1, d2, chunk_sum, nch, st); break;
        case 2: e = launch_d2<2>(x, ld, n, d, mu, c - 1, d2, chunk_sum, nch, st); break;
        case 3: e = launch_d2<3>(x, ld, n, d, mu, c - 1, d2, chunk_sum, nch, st); break;
        case 4: e = launch_d2<4>(x, ld, n, d, mu, c - 1, d2, chunk_sum, nch, st); break;
        default: e = launch_d2<0>(x, ld, n, d, mu, c - 1, d2, chunk_sum, nch, st); break;
      }
      if (e != cudaSuccess) return e;
    }
    kpp_pick_kernel<<<1, 1024, 0, st>>>(x, ld, n, d, u, c, chunk_sum, nch, d2, mu, idx);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace km
