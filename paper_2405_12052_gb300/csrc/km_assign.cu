// Reassignment + per-block accumulation: the expectation step and the first
// half of the mean calculation of Lloyd's algorithm (paper, section "The
// Lloyd's algorithm", steps 2 and 3), fused in one pass over the points.
//
// assign_fast_kernel<D, KG, CT> (d <= 4, K <= 256) is the hot kernel: SoA
// point tiles staged by 16-byte cp.async copies; an FP32 screen on FFMA2
// chains over groups of 4 centroids, the group minima packed with the group
// index and a running top-2 updated two groups at a time; the winning group
// recomputed for the label and the runner-up; a flag test in units of the
// screen's binade; per-warp queues of flagged points re-decided in batches;
// exact integer sums in per-warp (or per-half-warp) shared windows flushed
// into the block's int64 totals.  KG > 0 fixes the number of groups at
// compile time (shift packing, unrolled screen); CT reads the screen table
// from the constant bank instead of shared memory (no vector registers and
// no shared-memory loads for the table; one context per device holds it).
#include "km_internal.cuh"
#include "km_fast_tile.cuh"

namespace km {

namespace {

template <int D, int KG, bool CT>
__global__ void __launch_bounds__(kThreads, KM_MINB) assign_fast_kernel(FastArgs a) {
  constexpr int DP = D + 1, WIN = 2 * D + 1, GS = FastSmem<D>::GS;
  extern __shared__ __align__(16) unsigned char smraw[];
  if (a.ls->done && !a.ignore_done) return;  // the loop already stopped (graph-driven runs)
  const int nbuf = a.nwin == 1 ? 1 : 2;
  FastSmem<D> sm(smraw, a.kpad, a.k, a.nwin, nbuf);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int k = a.k, kpad = KG > 0 ? 4 * KG : a.kpad;

  const IterConst ic = *a.ic;
  const DataConst dc = *a.dc;
  float s[D];
  unsigned long long s2[D];
#pragma unroll
  for (int j = 0; j < D; ++j) { s[j] = dc.s[j]; s2[j] = dup2(dc.s[j]); }

  const int nwin = a.nwin;
  uint32_t* wwarp = sm.win + (size_t)warp * nwin * (k + 1) * WIN;
  uint32_t* wmine = wwarp + (size_t)(nwin == 4 ? (lane >> 3) : nwin == 2 ? (lane >> 4) : 0) * (k + 1) * WIN;
  long long* acc = sm.acc;
  uint32_t* q = sm.queue + (size_t)warp * kWarpQueue;
  float* xb = sm.xbuf + (size_t)warp * nbuf * D * kWarpTile;
  const int wid = blockIdx.x * kWarps + warp;  // this warp's first tile
  const int wtot = gridDim.x * kWarps;         // tile stride
  const int ntiles = (int)a.ntiles;            // < 2^31 (N < 2^39)
  if (wid < ntiles) prefetch_tile<D>(a, xb, (int64_t)wid * kWarpTile, lane);

  for (int q2 = tid; q2 < kpad * DP; q2 += kThreads) {
    const unsigned long long v = a.tab2[q2];
    sm.tab[q2] = v;
    const int c = q2 / DP, j = q2 - c * DP;
    reinterpret_cast<float*>(sm.gtab + (size_t)(c >> 2) * GS + j)[c & 3] = __uint_as_float((uint32_t)v);
  }
  for (int q2 = tid; q2 < k * DP; q2 += kThreads) sm.acc[q2] = 0;
  if (sm.ctil)
    for (int q2 = tid; q2 < k; q2 += kThreads) sm.ctil[q2] = a.ctil[q2];
  for (int q2 = tid; q2 < kWarps * nwin * (k + 1) * WIN; q2 += kThreads) sm.win[q2] = 0u;
  if (tid < 2) sm.cnt[tid] = 0;
  __syncthreads();

  FastCtx cx;
  cx.L = (uint32_t)ic.L; cx.mul = ic.mul; cx.kmask = ic.mul - 1u;
  cx.ehi = __float_as_uint(ic.M) >> (32 - ic.L);
  cx.M = ic.M;
  {
    // ulp of the binade [2^eM, 2^(eM+1)) that holds every r: exact scaling
    const float ulp = __uint_as_float(__float_as_uint(ic.M) & 0x7f800000u) * 0x1p-23f;
    cx.c0 = ic.thr_c0 * ulp;
    cx.cA = (ic.thr_cA + ic.tau * ic.G) * ulp;
  }
  cx.tau = ic.tau;
  cx.chi2 = dup2(dc.C_hi); cx.clo2 = dup2(dc.C_lo);
  cx.k = k; cx.kpad = kpad;
  int qn = 0, nflag = 0, n64 = 0, since_flush = 0;
  int m = 0;  // this warp's local tile counter

  for (int tile = wid; tile < ntiles; tile += wtot, ++m) {
    const int64_t base = (int64_t)tile * kWarpTile;
    const float* xcur = xb + (nbuf == 2 ? (m & 1) : 0) * D * kWarpTile;
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    // each lane reads only the chunks it copied itself, so the next copy
    // needs no warp barrier
    if (nbuf == 2 && tile + wtot < ntiles)
      prefetch_tile<D>(a, xb + ((m + 1) & 1) * D * kWarpTile, (int64_t)(tile + wtot) * kWarpTile, lane);
    if (base + kWarpTile <= a.n)
      process_tile<D, KG, CT, true>(a, sm, cx, s2, xcur, base, m, lane, wmine, q, qn);
    else
      process_tile<D, KG, CT, false>(a, sm, cx, s2, xcur, base, m, lane, wmine, q, qn);
    if (nbuf == 1 && tile + wtot < ntiles) prefetch_tile<D>(a, xb, (int64_t)(tile + wtot) * kWarpTile, lane);
    // 8 lanes x 8 points x 8 tiles, 16 x 8 x 4 or 32 x 8 x 2: <= 512 additions per bin
    if (++since_flush == (nwin == 4 ? 8 : nwin == 2 ? 4 : 2)) {
      flush_windows<D>(wwarp, acc, k, nwin, lane, dc.bits_C_hi, dc.bits_C_lo);
      since_flush = 0;
    }
    if (qn > kWarpQueue - kWarpTile) {
      __syncwarp();
      drain_warp_queue<D>(a, sm, q, qn, wid, wtot, wwarp, wmine, acc, lane, s, dc, ic.B_max, ic.tau, n64);
      nflag += qn;
      qn = 0;
      since_flush = 0;
    }
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncwarp();
  if (qn > 0) {
    drain_warp_queue<D>(a, sm, q, qn, wid, wtot, wwarp, wmine, acc, lane, s, dc, ic.B_max, ic.tau, n64);
    nflag += qn;
  } else {
    flush_windows<D>(wwarp, acc, k, nwin, lane, dc.bits_C_hi, dc.bits_C_lo);
  }
  if (lane == 0 && nflag) atomicAdd(&sm.cnt[0], nflag);
  if (n64) atomicAdd(&sm.cnt[1], n64);
  __syncthreads();
  long long* out = a.partials + (size_t)blockIdx.x * k * DP;
  for (int q2 = tid; q2 < k * DP; q2 += kThreads) out[q2] = sm.acc[q2];
  if (tid == 0) {
    if (sm.cnt[0]) atomicAdd(&a.ls->flagged, (unsigned long long)sm.cnt[0]);
    if (sm.cnt[1]) atomicAdd(&a.ls->fp64_decided, (unsigned long long)sm.cnt[1]);
  }
}

}  // namespace

size_t fast_smem_bytes(int d, int kpad, int k, int nwin) {
  const int dp = d + 1, win = 2 * d + 1, gs = (dp & 1) ? dp : dp + 1;
  const int nbuf = nwin == 1 ? 1 : 2;
  size_t b = (size_t)kpad * dp * 8 + (size_t)(k * dp + (k * dp & 1)) * 8 + (size_t)(kpad / 4) * gs * 16 +
             (nbuf == 2 ? (size_t)k * 16 : 0) +
             (size_t)kWarps * nbuf * d * kWarpTile * 4 + (size_t)kWarps * kWarpQueue * 4 +
             (size_t)kWarps * nwin * (k + 1) * win * 4 + 16;
  return (b + 15) & ~size_t(15);
}

template <int D, int KG, bool CT>
static cudaError_t launch_fast_dk(int grid, size_t smem, cudaStream_t st, const FastArgs& a) {
  auto fn = assign_fast_kernel<D, KG, CT>;
  cudaError_t e = allow_max_smem<assign_fast_kernel<D, KG, CT>>();
  if (e != cudaSuccess) return e;
  if constexpr (CT) {
    e = cudaMemcpyToSymbolAsync(c_screen_tab, a.tab2, (size_t)a.kpad * (D + 1) * sizeof(unsigned long long), 0,
                                cudaMemcpyDeviceToDevice, st);
    if (e != cudaSuccess) return e;
  }
  fn<<<grid, kThreads, smem, st>>>(a);
  return cudaGetLastError();
}

template <int D, int KG, bool CT>
static int blocks_dk(size_t smem) {
  int nb = 0;
  allow_max_smem<assign_fast_kernel<D, KG, CT>>();
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, assign_fast_kernel<D, KG, CT>, kThreads, smem) !=
      cudaSuccess)
    return 1;
  return nb > 0 ? nb : 1;
}

// Instantiations: the constant-bank screen (compile-time group count, fully
// unrolled, shift packing) for 3-D data with K <= 32 in groups of 8; for 3-D
// data with kpad = 256, the shared-memory table with a compile-time group
// count (index packing by shifts, 1.5 % faster than the run-time count); a
// runtime loop over the shared-memory table otherwise.
#define KM_FAST_DISPATCH(FN, D, CT_OK, ...)                           \
  do {                                                                \
    if constexpr (D == 3) {                                           \
      if (kpad == 32) {                                               \
        if (CT_OK) return FN<D, 8, true>(__VA_ARGS__);                \
        return FN<D, 8, false>(__VA_ARGS__);                          \
      }                                                               \
      if (kpad == 256) return FN<D, 64, false>(__VA_ARGS__);          \
    }                                                                 \
    return FN<D, 0, false>(__VA_ARGS__);                              \
  } while (0)

template <int D>
static int blocks_d(size_t smem, int kpad, bool ct) {
  KM_FAST_DISPATCH(blocks_dk, D, ct, smem);
}

template <int D>
static cudaError_t launch_fast_d(int grid, size_t smem, cudaStream_t st, const FastArgs& a) {
  const int kpad = a.kpad;
  KM_FAST_DISPATCH(launch_fast_dk, D, a.const_tab != 0, grid, smem, st, a);
}

bool fast_has_const_table(int d, int kpad) { return d == 3 && kpad == 32; }

int fast_blocks_per_sm(int d, size_t smem, int kpad, bool ct) {
  switch (d) {
    case 1: return blocks_d<1>(smem, kpad, ct);
    case 2: return blocks_d<2>(smem, kpad, ct);
    case 3: return blocks_d<3>(smem, kpad, ct);
    default: return blocks_d<4>(smem, kpad, ct);
  }
}

cudaError_t launch_assign_fast(int d, int grid, size_t smem, cudaStream_t st, const FastArgs& a) {
  switch (d) {
    case 1: return launch_fast_d<1>(grid, smem, st, a);
    case 2: return launch_fast_d<2>(grid, smem, st, a);
    case 3: return launch_fast_d<3>(grid, smem, st, a);
    case 4: return launch_fast_d<4>(grid, smem, st, a);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace km
