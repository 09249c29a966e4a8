// Batched instances (d <= 3, K <= 64) through the fused kernel's tiles, points
// whose label cannot have changed skipped: the reassignment and sums of one
// step of every active instance (paper, section "The Lloyd's algorithm", steps
// 2 and 3).
//
// Tiles are runs of one instance's points, a multiple of 2048 long but the
// instance's last.  A block takes the next tile of the step's list when it is
// done with one (tiles cost from a few points to all of them times 64
// centroids), loads the instance's screen table, group table, re-check
// centroids and drift sums into shared memory, and its warps run run_pass
// (km_fast_tile.cuh) over the tile's 256-point warp-tiles.  In an instance's
// first step of a run every point is screened; afterwards a point is decided
// again only when its kept lower bound of sqrt(D2) - sqrt(D1) has been used up
// by its instance's moves (cum, written by the batch update; see km_run_fast.cu
// for the bound), so most steps read 5 bytes a point instead of comparing it
// with K centroids.  The tile's changes are added to the instance's totals with
// integer atomics, so the update divides the same sums as from all points.  The
// update also lists the tiles of the instances that go on.
//
// Bound by issue while many points are open (0.67 ms the first step), by the
// latency of a tile's dependent loads afterwards (about 90 us a step over 4.6e7
// points, 35 us at the memory's rate).  256 instances, 4.6e7 points, K 4 to 64,
// 300 steps: 150 -> 52 ms without the copy of the labels.  Slower: a separate
// kernel with 48 warps an SM that tests the bounds and lists open points for two
// more (69 ms: the points' second pass costs more than the first one gains); a
// warp per tile of an eighth (100 ms: the warps of an SM then run the tables and
// the code of several d and K at a time).
#include "km_fast_tile.cuh"

namespace km {

namespace {

constexpr int kBatchWinWords = 2 * (kBatchMaxK + 1) * 7;  // per warp: two windows of 65 bins of 7 words

// One instance's constants as the tile machinery takes them.
template <int D>
struct BatchTile {
  FastArgs a;
  FastCtx cx;
  DataConst dc;
  RunTile rt;
  float s[D];
  unsigned long long s2[D];
  float B_max;
  const double* mu;
  __device__ __forceinline__ BatchTile(const BatchArgs& ba, const BatchInst& bi, int inst, const float* cum, int first) {
    a = FastArgs{};
    a.x = ba.x + bi.x_off; a.ld = bi.n; a.n = bi.n; a.k = bi.k; a.kpad = bi.kpad; a.nwin = 2;
    const IterConst& ic = ba.ic[inst];
    dc = DataConst{};
#pragma unroll
    for (int j = 0; j < D; ++j) { s[j] = dc.s[j] = bi.s[j]; s2[j] = dup2(bi.s[j]); }
    dc.C_hi = bi.C_hi; dc.C_lo = bi.C_lo;
    dc.bits_C_hi = bi.bits_C_hi; dc.bits_C_lo = bi.bits_C_lo;
    cx.L = (uint32_t)ic.L; cx.mul = ic.mul; cx.kmask = ic.mul - 1u;
    cx.ehi = __float_as_uint(ic.M) >> (32 - ic.L);
    cx.M = ic.M;
    const float ulp = __uint_as_float(__float_as_uint(ic.M) & 0x7f800000u) * 0x1p-23f;
    cx.c0 = ic.thr_c0 * ulp;
    cx.cA = (ic.thr_cA + ic.tau * ic.G) * ulp;
    cx.tau = ic.tau;
    cx.chi2 = dup2(dc.C_hi); cx.clo2 = dup2(dc.C_lo);
    cx.k = bi.k; cx.kpad = bi.kpad;
    rt.slack = ba.slack + bi.p_off; rt.z = ba.z8 + bi.p_off; rt.cum = cum;
    rt.invs = 1.f / (ic.G * ulp);  // powers of two: exact
    rt.margin = 4e-13f * (sqrtf(bi.A_max) + 1e-20f);
    rt.first = first;
    B_max = ic.B_max;
    mu = ba.mu + bi.mu_off;
  }
};

// A tile's changes to its instance's totals: value = high 2^32 + low (the
// update carries the low word's excess over every step).
__device__ __forceinline__ void add_totals(const BatchArgs& ba, const BatchInst& bi, long long* acc, int cols, int from,
                                           int step) {
  unsigned long long* tot = ba.totals + 2 * bi.tot_off;
  for (int c = from; c < cols; c += step) {
    const long long v = acc[c];
    if (v) {
      if ((uint32_t)v) atomicAdd(tot + 2 * c, (unsigned long long)(uint32_t)v);
      if (v >> 32) atomicAdd(tot + 2 * c + 1, (unsigned long long)(v >> 32));
      acc[c] = 0;
    }
  }
}

template <int D>
__device__ __forceinline__ void batch_run_tile(const BatchArgs& ba, const int4& it, int first, unsigned char* raw,
                                               float* cum, int tid, int& nflag, int& n64) {
  constexpr int DP = D + 1, WIN = 2 * D + 1, GS = FastSmem<D>::GS;
  const int lane = tid & 31, warp = tid >> 5, inst = it.x;
  const FastSmem<3> f(raw, kBatchMaxK, kBatchMaxK, 2, 2);  // the regions of d = 3, K = 64 for every instance
  FastSmem<D> sm;
  sm.tab = f.tab; sm.acc = f.acc; sm.gtab = f.gtab; sm.ctil = f.ctil;
  const BatchInst& bi = ba.inst[inst];
  const int k = bi.k, kpad = bi.kpad;
  const unsigned long long* tab2 = ba.tab2 + bi.tab_off;
  for (int q = tid; q < kpad * DP; q += kThreads) {
    const unsigned long long v = tab2[q];
    sm.tab[q] = v;
    const int c = q / DP, j = q - c * DP;
    reinterpret_cast<float*>(sm.gtab + (size_t)(c >> 2) * GS + j)[c & 3] = __uint_as_float((uint32_t)v);
  }
  for (int q = tid; q < k; q += kThreads) {
    sm.ctil[q] = ba.ctil4[bi.k_off + q];
    cum[q] = first ? 0.f : ba.cum[bi.k_off + q];
  }
  const BatchTile<D> bt(ba, bi, inst, cum, first);
  __syncthreads();
  uint32_t* wwarp = f.win + (size_t)warp * kBatchWinWords;
  const int wt0 = it.y / kWarpTile;  // the tile's warp-tiles within the instance
  run_pass<D, 0, true>(bt.a, sm, bt.cx, bt.s2, bt.s, bt.dc, bt.rt, sm.ctil, bt.mu, bt.B_max, sm.acc,
                       f.queue + (size_t)warp * kWarpQueue, wwarp, wwarp + (lane >> 4) * (k + 1) * WIN,
                       f.xbuf + (size_t)warp * 2 * 3 * kWarpTile, 2, wt0 + warp, kWarps,
                       wt0 + (it.z + kWarpTile - 1) / kWarpTile, lane, nflag, n64);
  __syncthreads();
  add_totals(ba, bi, sm.acc, k * DP, tid, kThreads);
}

// mode: 0 as the instances' states say, 1 every instance in its first step, -1
// none (the tuner's timing).  work: [0] tiles listed, [1] tiles taken, [2]
// blocks done; the last block clears them for the next step's list.
__global__ void __launch_bounds__(kThreads, KM_MINB) batch_run_kernel(BatchArgs ba, int mode) {
  extern __shared__ __align__(16) unsigned char smraw[];
  __shared__ float s_cum[kBatchMaxK];
  __shared__ int s_next;
  const int tid = threadIdx.x;
  const int items = ba.work[0];
  if (tid == 0) s_next = items > 0 ? atomicAdd(ba.work + 1, 1) : 0;
  const FastSmem<3> f(smraw, kBatchMaxK, kBatchMaxK, 2, 2);
  for (int q = tid; q < kWarps * kBatchWinWords; q += kThreads) f.win[q] = 0u;
  for (int q = tid; q < kBatchMaxK * 4; q += kThreads) f.acc[q] = 0;
  __syncthreads();
  int nflag = 0, n64 = 0;
  while (true) {
    const int e = s_next;
    if (e >= items) break;
    int ne = 0;
    if (tid == 0) ne = atomicAdd(ba.work + 1, 1);  // on its way while this tile is worked on
    const int4 it = ba.tiles[ba.list[e]];
    const int d = ba.inst[it.x].d, first = mode > 0 || (mode == 0 && ba.state[it.x].first);
    if (d == 3) batch_run_tile<3>(ba, it, first, smraw, s_cum, tid, nflag, n64);
    else if (d == 2) batch_run_tile<2>(ba, it, first, smraw, s_cum, tid, nflag, n64);
    else batch_run_tile<1>(ba, it, first, smraw, s_cum, tid, nflag, n64);
    if (tid == 0) s_next = ne;  // read last before the tile's barriers
    __syncthreads();
  }
  for (int o = 16; o > 0; o >>= 1) n64 += __shfl_xor_sync(0xffffffffu, n64, o);
  if ((tid & 31) == 0) {
    if (nflag) atomicAdd(ba.flagged, (unsigned long long)nflag);
    if (n64) atomicAdd(ba.fp64, (unsigned long long)n64);
  }
  if (tid == 0) {
    __threadfence();
    if (atomicAdd(ba.work + 2, 1) == (int)gridDim.x - 1) {  // every block has read the list's length
      ba.work[0] = 0;
      ba.work[1] = 0;
      ba.work[2] = 0;
    }
  }
}

// Lists the tiles of the instances that are not done (mode != 0: of all), at
// the start of a run.
__global__ void __launch_bounds__(256) batch_list_kernel(BatchArgs ba, int mode) {
  const int t = blockIdx.x * 256 + threadIdx.x;
  const bool live = t < ba.ntiles && (mode != 0 || !ba.state[ba.tiles[t].x].done);
  const unsigned m = __ballot_sync(0xffffffffu, live);
  if (!m) return;
  int at = 0;
  if ((threadIdx.x & 31) == 0) at = atomicAdd(ba.work, __popc(m));
  at = __shfl_sync(0xffffffffu, at, 0);
  if (live) ba.list[at + __popc(m & ((1u << (threadIdx.x & 31)) - 1u))] = t;
}

// Byte labels (instances at 256-point boundaries) to the packed int32 labels.
__global__ void __launch_bounds__(256) batch_labels_kernel(const BatchInst* __restrict__ inst,
                                                           const uint8_t* __restrict__ z8,
                                                           int32_t* __restrict__ labels) {
  const BatchInst& bi = inst[blockIdx.y];
  const int64_t n = bi.n;
  const uint8_t* z = z8 + bi.p_off;
  int32_t* out = labels + bi.lab_off;
  for (int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x; i < n; i += (int64_t)gridDim.x * 256) out[i] = z[i];
}

size_t batch_run_smem() { return fast_smem_bytes(3, kBatchMaxK, kBatchMaxK, 2); }

}  // namespace

cudaError_t launch_batch_list(const BatchArgs& a, int mode, cudaStream_t st) {
  cudaError_t e = cudaMemsetAsync(a.work, 0, 3 * sizeof(int), st);
  if (e != cudaSuccess) return e;
  batch_list_kernel<<<(a.ntiles + 255) / 256, 256, 0, st>>>(a, mode);
  return cudaGetLastError();
}

cudaError_t launch_batch_run(const BatchArgs& a, int grid, int mode, cudaStream_t st) {
  const size_t smem = batch_run_smem();
  cudaError_t e = cudaFuncSetAttribute(batch_run_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  batch_run_kernel<<<grid, kThreads, smem, st>>>(a, mode);
  return cudaGetLastError();
}

cudaError_t launch_batch_labels(const BatchArgs& a, int count, int sms, cudaStream_t st) {
  // up to 65535 instances a launch (the grid's second dimension)
  for (int i0 = 0; i0 < count; i0 += 65535) {
    const int m = std::min(65535, count - i0);
    batch_labels_kernel<<<dim3((unsigned)std::max(1, std::min(64, 16 * sms / m + 1)), m), 256, 0, st>>>(a.inst + i0, a.z8,
                                                                                                       a.labels);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

int batch_run_blocks_per_sm() {
  const size_t smem = batch_run_smem();
  int nb = 0;
  cudaFuncSetAttribute(batch_run_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, batch_run_kernel, kThreads, smem) != cudaSuccess) return 1;
  return nb > 0 ? nb : 1;
}

}  // namespace km
