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
constexpr int kKppThreads = 512;  // threads per block
constexpr int kKppSum = 256;      // threads whose points are added one after another

__device__ __forceinline__ double kpp_d2(const float* x, int64_t ld, int64_t i, int d, const double* m) {
  double acc = 0.0;
  for (int j = 0; j < d; ++j) {
    const double t = __dsub_rn((double)x[(int64_t)j * ld + i], m[j]);
    acc = __dadd_rn(acc, __dmul_rn(t, t));
  }
  return acc;
}

// Inclusive scan over the block's threads of one value each (warp scans, then
// the warp totals): a fixed order.
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
    double t = lane < kKppThreads / 32 ? s_w[lane] : 0.0;
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
// *below receives the running sum before that index.  v was written by other
// blocks of this launch: read past L1.
__device__ int block_find(const double* v, int m, double before, double target, double* s_w, double* below) {
  __shared__ int s_first;
  __shared__ int s_idx;
  __shared__ double s_below;
  const int run = (m + kKppThreads - 1) / kKppThreads;
  const int lo = min(m, (int)threadIdx.x * run), hi = min(m, lo + run);
  double s = 0.0;
#pragma unroll 8
  for (int q = lo; q < hi; ++q) s = __dadd_rn(s, __ldcg(v + q));
  if (threadIdx.x == 0) { s_first = kKppThreads; s_idx = m; s_below = before; }
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
      const double t = __dadd_rn(b, __ldcg(v + q));
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

// The pick of round c >= 1 (one block).  The chunk sums are added in one
// segment per warp, the crossing segment is searched for its chunk and the
// chunk for its point.  (A Hillis-Steele scan of all chunk sums, two barriers
// per doubling: 157 us a round with 24414 chunks; this, as a kernel of its
// own, 25 us, of which 4 were its launch.)
__device__ int64_t kpp_pick(int64_t n, double uc, const double* chunk_sum, int nchunks, const double* d2) {
  constexpr int kW = kKppThreads / 32;
  __shared__ double s_w[32];
  __shared__ double s_seg[32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int seg = (nchunks + kW - 1) / kW;
  {
    const int hi = (int)min((int64_t)nchunks, (int64_t)(w + 1) * seg);
    double s = 0.0;
#pragma unroll 8
    for (int64_t q = (int64_t)w * seg + lane; q < hi; q += 32) s = __dadd_rn(s, __ldcg(chunk_sum + q));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s = __dadd_rn(s, __shfl_xor_sync(0xffffffffu, s, o));
    if (lane == 0) s_seg[w] = s;
  }
  __syncthreads();
  // every warp: the segments' running sums, the target and the segment
  double incl = lane < kW ? s_seg[lane] : 0.0;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const double t = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl = __dadd_rn(incl, t);
  }
  const double target = __dmul_rn(uc, __shfl_sync(0xffffffffu, incl, 31));
  const unsigned over = __ballot_sync(0xffffffffu, lane < kW && incl > target);
  if (over == 0u) return n - 1;  // no running sum exceeds the target
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
  return i0 + min(block_find(d2 + i0, m, before, target, s_w, &unused), m - 1);  // likewise its last point
}

// Pick 0: floor(u_0 n).
__global__ void kpp_first_kernel(const float* __restrict__ x, int64_t ld, int64_t n, int d, const double* __restrict__ u,
                                 double* mu, int64_t* idx) {
  int64_t pick = (int64_t)floor(u[0] * (double)n);
  if (pick >= n) pick = n - 1;
  if (pick < 0) pick = 0;
  if ((int)threadIdx.x < d) mu[threadIdx.x] = (double)x[(int64_t)threadIdx.x * ld + pick];
  if (threadIdx.x == 0) idx[0] = pick;
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

// D^2 against centre c (the minimum with the previous D^2 for c > 0), the
// chunk sums and, in the block that finishes last (integer ticket), the pick
// of round c + 1.  One block per chunk; thread t < 256 sums points t, t + 256,
// ... of the chunk, then a fixed-order tree.
//
// FP64 instructions bound the plain form (11 a point and round: 2.73 ms a
// round for 1e8 points in 3-D, against 0.30 ms for reading the points and
// their D^2; with the screen below 0.66 ms on average over 31 rounds, 0.46 in the late ones).  A centre is closer than the ones before for about 1 / c of the
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
                                                             int dd, double* mu, int c, double* d2, double* chunk_sum,
                                                             int nchunks, const double* __restrict__ u, int64_t* idx,
                                                             unsigned int* ticket) {
  extern __shared__ __align__(16) double s_d2[];  // [kKppChunk]
  __shared__ double s_red[kKppSum];
  __shared__ bool s_last;
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
  if (tid < kKppSum) {
    double acc = 0.0;
    for (int q = tid; q < m; q += kKppSum) acc = __dadd_rn(acc, s_d2[q]);
    s_red[tid] = acc;
  }
  __syncthreads();
  for (int w = kKppSum / 2; w >= 32; w >>= 1) {
    if (tid < w) s_red[tid] = __dadd_rn(s_red[tid], s_red[tid + w]);
    __syncthreads();
  }
  if (tid < 32) {
    double t = s_red[tid];
#pragma unroll
    for (int w = 16; w > 0; w >>= 1) t = __dadd_rn(t, __shfl_down_sync(0xffffffffu, t, w));
    if (tid == 0) chunk_sum[blockIdx.x] = t;
  }
  __threadfence();
  __syncthreads();
  if (tid == 0) s_last = atomicAdd(ticket, 1u) == (unsigned)gridDim.x - 1u;
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  const int64_t pick = kpp_pick(n, u[c + 1], chunk_sum, nchunks, d2);
  if (tid < d) mu[(size_t)(c + 1) * d + tid] = (double)x[(int64_t)tid * ld + pick];
  if (tid == 0) {
    idx[c + 1] = pick;
    *ticket = 0u;
  }
}

}  // namespace

int64_t kpp_chunks(int64_t n) { return (n + kKppChunk - 1) / kKppChunk; }

cudaError_t launch_kmeanspp(const float* x, int64_t ld, int64_t n, int d, int k, const double* u, double* mu,
                            int64_t* idx, double* d2, double* chunk_sum, cudaStream_t st) {
  const int nch = (int)kpp_chunks(n);
  unsigned int* ticket = reinterpret_cast<unsigned int*>(chunk_sum + nch);
  cudaError_t e = cudaMemsetAsync(ticket, 0, sizeof(unsigned int), st);
  if (e != cudaSuccess) return e;
  kpp_first_kernel<<<1, kMaxKppD, 0, st>>>(x, ld, n, d, u, mu, idx);
  auto* fn = d == 1 ? kpp_d2_kernel<1> : d == 2 ? kpp_d2_kernel<2> : d == 3 ? kpp_d2_kernel<3>
           : d == 4 ? kpp_d2_kernel<4> : kpp_d2_kernel<0>;
  for (int c = 0; c + 1 < k; ++c) {
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    fn<<<nch, kKppThreads, sizeof(double) * kKppChunk, st>>>(x, ld, n, d, mu, c, d2, chunk_sum, nch, u, idx, ticket);
  }
  return cudaGetLastError();
}

}  // namespace km
