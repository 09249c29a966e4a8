// Reassignment and per-block sums for any d and K (paper, section "The
// Lloyd's algorithm", steps 2 and 3): an FP32 screen ||c~||^2 - 2 x~.c~ with a
// rigorous bound, the direct form and then FP64 in the oracle's order for the
// points it leaves open, exact fixed-point sums.
//
// Bound by FP32 multiply-adds, one per point, centroid and coordinate (1.02e9
// for N = 1e6, d = 16, K = 64: 27 us at one per lane and cycle; the direct
// form takes two operations), and by what a point costs beside them: its two
// smallest values over K and 2 d + 1 additions to the sums.  A block takes 256
// points against 64 centroids at a time (16 for few centroids), 32 coordinates of
// both in shared memory, 8 points x 8 centroids per thread: four 16-byte shared
// reads per 64 multiply-adds.  The two smallest values of a point are kept per thread over
// the centroid tiles and merged over its 8 threads at the end, each exchange
// halving the points a thread keeps.  Open points are decided by one warp each
// (lanes over centroids).  The sums go to 32-bit windows in shared memory (one or
// more per block, flushed every 512 points each) while those fit, else to the
// block's row by 64-bit global atomics.  N = 1e6, d = 16, K = 64: one point per
// thread and 64-bit atomics 572 us, direct form in tiles of 128 points 214
// us, this 170 us (ten steps of a run: 6.09, 2.36, 1.79 ms).
#include <type_traits>

#include "km_fast_common.cuh"

namespace km {

namespace {

constexpr int kGP = 256;              // points per tile
constexpr int kGC = 64;               // centroids per tile beyond kGSmallK
constexpr int kGSmallK = 40;          // up to here tiles of 16 centroids
constexpr int kGD = 32;               // coordinates staged at a time
constexpr int kGXS = kGP + 4;         // row strides of the staged tiles
constexpr int kGFlush = 2;            // point tiles per window between flushes (512 additions per bin)
constexpr size_t kGTwoMax = 66 * 1024;   // windows and totals with which two blocks stay on an SM
constexpr size_t kGManyMax = 32 * 1024;  // several windows take at most this

// Words of a window: odd, so that the windows' rows of one cluster lie in
// different banks.
__host__ __device__ __forceinline__ int generic_win_words(int d, int k) { return (k * (2 * d + 1)) | 1; }

__device__ __forceinline__ void top2_merge(float& best, float& second, int& kb, float ob, float os, int ok) {
  const bool take = ob < best || (ob == best && ok < kb);
  second = fminf(fminf(second, os), fmaxf(best, ob));
  best = fminf(best, ob);
  kb = take ? ok : kb;
}

// NC centroids a thread.  nwin windows (a power of two; 0: 64-bit atomics into the
// row), window lane mod nwin taking the point of that lane.
template <int NC>
__global__ void __launch_bounds__(kThreads, 2) assign_generic_kernel(GenericArgs a, int nwin, int tot_sh) {
  constexpr int GC = 8 * NC, GCS = GC + 4;
  constexpr bool MANY = NC < 8;  // more than one window
  // centroid of a tile that thread tx keeps as its c-th
  auto cent = [](int tx, int c) { return NC == 8 ? 4 * tx + (c & 3) + 32 * (c >> 2) : NC * tx + c; };
  extern __shared__ __align__(16) unsigned char smraw[];
  float* s_x = reinterpret_cast<float*>(smraw);       // [kGD][kGXS] x~ = fl(x - s) by coordinate
  float* s_c = s_x + kGD * kGXS;                      // [kGD][GCS] c~ by coordinate
  long long* s_tot = reinterpret_cast<long long*>(s_c + kGD * GCS);  // [k][d + 1] when tot_sh
  const int d = a.d, k = a.k, dp = d + 1, wn = 2 * d + 1;
  uint32_t* s_win = reinterpret_cast<uint32_t*>(s_tot + (tot_sh ? (size_t)k * dp : 0));  // [nwin][ws], k rows of 2 d + 1
  const int ws = generic_win_words(d, k);
  __shared__ float s_A[kGP];
  __shared__ int s_lab[kGP], s_q[kGP];
  __shared__ int s_qn, s_nflag, s_n64;
  if (a.ls->done && !a.ignore_done) return;
  const int tid = threadIdx.x, tx = tid & 7, ty = tid >> 3, lane = tid & 31, warp = tid >> 5;
  long long* row = a.partials + (size_t)blockIdx.x * k * dp;
  long long* tot = tot_sh ? s_tot : row;
  for (int q = tid; q < k * dp; q += kThreads) tot[q] = 0;
  for (int q = tid; q < nwin * ws; q += kThreads) s_win[q] = 0u;
  if (tid == 0) { s_qn = 0; s_nflag = 0; s_n64 = 0; }
  const DataConst dc = *a.dc;
  const float B_max = *a.B_max_ptr, sB = sqrtf(B_max);
  const int ktiles = (k + GC - 1) / GC, chunks = (d + kGD - 1) / kGD;
  const int64_t ntiles = (a.n + kGP - 1) / kGP;
  // Bound of the difference of two screen values against that of the exact
  // distances, per unit of A + B_max.  One value: the roundings of x~ and c~
  // (4.04 u), the d products and their sum (1.01 d u), ||c~||^2 (2.01 u), the
  // last multiply-add (2.02 u), and the oracle's FP64 rounding.
  const float evc = 2.04f * kU * ((float)d + 8.5f) + 2.f * kU64x * (float)(d + 1);
  __syncthreads();

  // the windows' sums of bin q = (cluster, column) into the block's totals
  auto flush = [&]() {
    __syncthreads();
    for (int q = tid; q < k * dp; q += kThreads) {
      const int c = q / dp, j = q - c * dp;
      const uint32_t* w = s_win + (size_t)c * wn;
      auto value = [&](const uint32_t* wb, uint32_t cnt) {
        if (j == d) return (long long)cnt;
        const int hi = (int)(wb[1 + j] - cnt * dc.bits_C_hi);  // exact: |sum| <= 2^30
        const int lo = (int)(wb[1 + d + j] - cnt * dc.bits_C_lo);
        return ((long long)hi << 22) + (long long)lo;
      };
      const uint32_t cnt = w[0];
      uint32_t any = cnt;
      long long v = value(w, cnt);
      for (int b = 1; b < (MANY ? nwin : 1); ++b) {
        const uint32_t* wb = w + (size_t)b * ws;
        any |= wb[0];
        v += value(wb, wb[0]);
      }
      if (any) tot[q] += v;
    }
    __syncthreads();
    for (int q = tid; q < nwin * ws; q += kThreads) s_win[q] = 0u;
    __syncthreads();
  };

  int since = 0;
  for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    const int64_t base = tile * kGP;
    const int np = (int)min((int64_t)kGP, a.n - base);
    float best[8], second[8], A = 0.f;  // A: of point tid
    int kb[8];
#pragma unroll
    for (int r = 0; r < 8; ++r) { best[r] = 3.0e38f; second[r] = 3.0e38f; kb[r] = 0; }
    for (int kt = 0; kt < ktiles; ++kt) {
      float acc[8][NC];  // points 8 ty + r, centroids cent(tx, c)
#pragma unroll
      for (int r = 0; r < 8; ++r)
#pragma unroll
        for (int c = 0; c < NC; ++c) acc[r][c] = 0.f;
      for (int ch = 0; ch < chunks; ++ch) {
        const int j0 = ch * kGD, nj = min(kGD, d - j0);
        __syncthreads();  // the tiles before are read no more
        if (kt == 0 || chunks > 1) {
#pragma unroll 4
          for (int j = 0; j < nj; ++j)
            s_x[j * kGXS + tid] =
                tid < np ? __fsub_rn(a.x[(int64_t)(j0 + j) * a.ld + base + tid], a.shift[j0 + j]) : 0.f;
        }
        if (ktiles > 1 || chunks > 1 || tile == blockIdx.x)
          for (int q = tid; q < nj * GC; q += kThreads) {
            const int c = q / nj, j = q - c * nj, cc = kt * GC + c;
            s_c[j * GCS + c] = cc < k ? a.ctil[(size_t)cc * d + j0 + j] : 0.f;
          }
        __syncthreads();
        if (kt == 0)
          for (int j = 0; j < nj; ++j) A = __fmaf_rn(s_x[j * kGXS + tid], s_x[j * kGXS + tid], A);
#pragma unroll 4
        for (int j = 0; j < nj; ++j) {
          const float4 x0 = *reinterpret_cast<const float4*>(s_x + j * kGXS + 8 * ty);
          const float4 x1 = *reinterpret_cast<const float4*>(s_x + j * kGXS + 8 * ty + 4);
          const float xv[8] = {x0.x, x0.y, x0.z, x0.w, x1.x, x1.y, x1.z, x1.w};
          alignas(16) float cw[NC];
          if constexpr (NC == 8) {
            *reinterpret_cast<float4*>(cw) = *reinterpret_cast<const float4*>(s_c + j * GCS + 4 * tx);
            *reinterpret_cast<float4*>(cw + 4) = *reinterpret_cast<const float4*>(s_c + j * GCS + 32 + 4 * tx);
          } else {
            *reinterpret_cast<float2*>(cw) = *reinterpret_cast<const float2*>(s_c + j * GCS + 2 * tx);
          }
#pragma unroll
          for (int r = 0; r < 8; ++r)
#pragma unroll
            for (int c = 0; c < NC; ++c) acc[r][c] = __fmaf_rn(xv[r], cw[c], acc[r][c]);
        }
      }
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        const int cc = kt * GC + cent(tx, c);
        if (cc >= k) continue;
        const float nc = __ldg(a.cnorm + cc);
#pragma unroll
        for (int r = 0; r < 8; ++r) {
          const float v = __fmaf_rn(-2.f, acc[r][c], nc);
          const bool less = v < best[r];
          second[r] = fminf(second[r], fmaxf(best[r], v));
          best[r] = fminf(best[r], v);
          kb[r] = less ? cc : kb[r];
        }
      }
    }
    s_A[tid] = A * 1.0001f;
    // merge over the 8 threads of a point group: each exchange halves the
    // points a thread keeps, so it ends with one
    auto merge_half = [&](auto half, int bit) {
      constexpr int H = decltype(half)::value;
      const bool up = tx & bit;
#pragma unroll
      for (int r = 0; r < H; ++r) {
        const float sb = up ? best[r] : best[r + H], ss = up ? second[r] : second[r + H];
        const int sk = up ? kb[r] : kb[r + H];
        const float ob = __shfl_xor_sync(0xffffffffu, sb, bit), os = __shfl_xor_sync(0xffffffffu, ss, bit);
        const int ok = __shfl_xor_sync(0xffffffffu, sk, bit);
        if (up) { best[r] = best[r + H]; second[r] = second[r + H]; kb[r] = kb[r + H]; }
        top2_merge(best[r], second[r], kb[r], ob, os, ok);
      }
    };
    merge_half(std::integral_constant<int, 4>{}, 4);
    merge_half(std::integral_constant<int, 2>{}, 2);
    merge_half(std::integral_constant<int, 1>{}, 1);
    __syncthreads();  // s_A
    {
      const int p = 8 * ty + tx;  // bits 4, 2, 1 of tx chose the point's half each time
      if (p < np) {
        bool clear = true;
        if (k > 1) {
          const float AB = s_A[p] + B_max, T0 = evc * AB + 1e-30f;  // 1e-30: underflowed products
          clear = second[0] - best[0] > T0 + a.tau * fmaxf(s_A[p] + second[0] + T0, 0.f);
        }
        s_lab[p] = kb[0];
        if (!clear) s_q[atomicAdd(&s_qn, 1)] = p;
      }
    }
    __syncthreads();
    const int qn = s_qn;
    for (int e = warp; e < qn; e += kWarps) {
      // direct form first, then FP64 where its bound leaves the point open
      const int p = s_q[e];
      const float* xp = a.x + base + p;
      float b1 = 3.0e38f, b2 = 3.0e38f;
      int k1 = 0;
      for (int c = lane; c < k; c += 32) {
        float dv = 0.f;
        for (int j = 0; j < d; ++j) {
          const float t = __fsub_rn(__fsub_rn(xp[(int64_t)j * a.ld], a.shift[j]), a.ctil[(size_t)c * d + j]);
          dv = __fmaf_rn(t, t, dv);
        }
        if (dv < b1) { b2 = b1; b1 = dv; k1 = c; }
        else if (dv < b2) b2 = dv;
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        const float ob = __shfl_xor_sync(0xffffffffu, b1, o), os = __shfl_xor_sync(0xffffffffu, b2, o);
        const int ok = __shfl_xor_sync(0xffffffffu, k1, o);
        top2_merge(b1, b2, k1, ob, os, ok);
      }
      const float Ap = s_A[p], sA = sqrtf(Ap), AB = Ap + B_max;
      const float e1 = direct_bound(b1, sA, sB, AB, d), e2 = direct_bound(b2, sA, sB, AB, d);
      const float lo2 = b2 - e2, hi1 = b1 + e1;
      int lab = k1;
      if (!((lo2 > hi1) && (lo2 - hi1 > a.tau * (b2 + e2)))) {  // the same in every lane
        double bd = 0.0;
        int k64 = -1;
        for (int c = lane; c < k; c += 32) {
          const double dd = d64_dyn(a.x, a.ld, base + p, d, a.mu + (size_t)c * d);
          if (k64 < 0 || dd < bd) { bd = dd; k64 = c; }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
          const double ob = __shfl_xor_sync(0xffffffffu, bd, o);
          const int ok = __shfl_xor_sync(0xffffffffu, k64, o);
          if (ok >= 0 && (k64 < 0 || ob < bd || (ob == bd && ok < k64))) { bd = ob; k64 = ok; }
        }
        lab = k64;
        if (lane == 0) atomicAdd(&s_n64, 1);
      }
      if (lane == 0) s_lab[p] = lab;
    }
    __syncthreads();
    if (tid == 0) { s_nflag += qn; s_qn = 0; }
    if (a.store_labels && tid < np) {
      if (a.labels8) a.labels8[base + tid] = (uint8_t)s_lab[tid];
      else a.labels[base + tid] = s_lab[tid];
    }
    // sums: a thread per point, coordinate after coordinate (coalesced)
    if (tid < np) {
      const int c = s_lab[tid];
      const float* xp = a.x + base + tid;
      if (nwin) {
        uint32_t* w = s_win + (size_t)(MANY ? lane & (nwin - 1) : 0) * ws + (size_t)c * wn;
        atomicAdd(w, 1u);
#pragma unroll 4
        for (int j = 0; j < d; ++j) {
          uint32_t bh, bl;
          split_limbs(xp[(int64_t)j * a.ld], dc.C_hi, dc.C_lo, bh, bl);
          atomicAdd(w + 1 + j, bh);
          atomicAdd(w + 1 + d + j, bl);
        }
      } else {
        unsigned long long* r = reinterpret_cast<unsigned long long*>(row) + (size_t)c * dp;
        atomicAdd(r + d, 1ull);
#pragma unroll 4
        for (int j = 0; j < d; ++j) {
          uint32_t bh, bl;
          split_limbs(xp[(int64_t)j * a.ld], dc.C_hi, dc.C_lo, bh, bl);
          const long long hi = (long long)(int)(bh - dc.bits_C_hi), lo = (long long)(int)(bl - dc.bits_C_lo);
          atomicAdd(r + j, (unsigned long long)((hi << 22) + lo));
        }
      }
    }
    if (nwin && ++since == (MANY ? kGFlush * nwin : kGFlush)) {
      flush();
      since = 0;
    }
  }
  if (nwin && since) flush();
  __syncthreads();
  if (tot_sh)
    for (int q = tid; q < k * dp; q += kThreads) row[q] = s_tot[q];
  if (tid == 0) {
    if (s_nflag) atomicAdd(&a.ls->flagged, (unsigned long long)s_nflag);
    if (s_n64) atomicAdd(&a.ls->fp64_decided, (unsigned long long)s_n64);
  }
}

// Where the sums go.  Windows while one takes at most 66 KB, with which two blocks
// stay on an SM (tiles 42 KB, static arrays 3 KB; N = 1e6, d = 32, K = 300, 78 KB of
// window: one block an SM 1.74 ms a step, 64-bit atomics into the block's row 1.16),
// the int64 totals beside them where both fit in that (d = 40, K = 130: 1.44 ms with
// totals in shared memory and one block, 1.09 with the row), else in the block's
// own row (read and written by one thread each).  With few clusters (K <= 40; at
// K = 64 they gained nothing) the lanes of a warp add to the same words, so a
// block has several windows, up to one per lane (d = 48, K = 2: 0.61 -> 0.48 ms a
// step), as far as they take 32 KB, and at most four per tile that the block
// takes (zeroing and flushing them).
// Tiles of 64 centroids are mostly padding for few: up to K = 40 tiles of 16
// (d = 48: K = 2 0.48 -> 0.25 ms a step, K = 5 0.51 -> 0.28, K = 40 0.60 -> 0.53).
struct GenericPlan {
  int nwin, tot_sh;
  size_t smem;
};
GenericPlan generic_plan(int d, int k, int64_t tiles_per_block) {
  const size_t win = ((size_t)k * (2 * (size_t)d + 1) | 1) * 4, tot = (size_t)k * (d + 1) * 8;
  GenericPlan g{};
  if (win <= kGTwoMax) {
    g.nwin = 1;
    g.tot_sh = win + tot <= kGTwoMax ? 1 : 0;
    const size_t t = g.tot_sh ? tot : 0;
    const int most = k <= kGSmallK ? (int)std::min<int64_t>(32, 4 * tiles_per_block) : 1;
    while (2 * g.nwin <= most && 2 * g.nwin * win <= kGManyMax && 2 * g.nwin * win + t <= kGTwoMax) g.nwin *= 2;
  }
  g.smem = sizeof(float) * kGD * (kGXS + (k <= kGSmallK ? 16 : kGC) + 4) + g.nwin * win + (g.tot_sh ? tot : 0);
  return g;
}

template <int NC>
int generic_blocks(size_t smem) {
  int nb = 0;
  if (allow_max_smem<assign_generic_kernel<NC>>() != cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, assign_generic_kernel<NC>, kThreads, smem) != cudaSuccess)
    return 1;
  return std::max(1, nb);
}
template <int NC>
cudaError_t generic_launch(int grid, const GenericPlan& g, cudaStream_t st, const GenericArgs& a) {
  cudaError_t e = allow_max_smem<assign_generic_kernel<NC>>();
  if (e != cudaSuccess) return e;
  assign_generic_kernel<NC><<<grid, kThreads, g.smem, st>>>(a, g.nwin, g.tot_sh);
  return cudaGetLastError();
}

}  // namespace

int64_t generic_grid(int64_t n, int d, int k, int sms) {
  const int64_t tiles = (n + kGP - 1) / kGP;
  const GenericPlan g = generic_plan(d, k, tiles);
  const int nb = k <= kGSmallK ? generic_blocks<2>(g.smem) : generic_blocks<8>(g.smem);
  return std::min<int64_t>(tiles, (int64_t)sms * nb);
}

cudaError_t launch_assign_generic(int grid, cudaStream_t st, const GenericArgs& a) {
  const GenericPlan g = generic_plan(a.d, a.k, ((a.n + kGP - 1) / kGP + grid - 1) / grid);
  return a.k <= kGSmallK ? generic_launch<2>(grid, g, st, a) : generic_launch<8>(grid, g, st, a);
}

}  // namespace km
