// A whole run of Lloyd's loop (d <= 4, K <= 256) in one cooperative kernel:
// reassignment, mean calculation, error and stop test of every step (paper,
// sections "The Lloyd's algorithm" and "Serial Lloyd's algorithm"), with the
// same labels, counts, centroids and errors as the step-by-step kernels.
//
// Two things bound the step-by-step loop.  Small sets: two kernels a step, 27
// us of launches, reductions through memory and one block's serial work for
// 1e5 points whose distances take 1 us.  Large sets: every step compares every
// point with every centroid (0.85 ms for 1e8 points, d = 3, K = 32), although
// after a few steps nearly all points keep their label by a wide margin.
//
// Here the grid stays resident.  Per step each block passes over its
// points, adds its sums to a small global table with integer atomics and
// waits for the other blocks once; then every block forms the new centroids,
// E, the stop test and the screen tables for itself (the same FP64 operations
// in the same order everywhere, so the same bits), which costs less than
// publishing one block's result behind a second wait.
//
// Skipping points.  When a point is decided, a rigorous lower bound of
// sqrt(D2) - sqrt(D1) is kept with it (D1 its squared distance to its centroid,
// D2 to any other; the bounds are the ones the flag test and the re-check
// already rest on).  When centroid k moves by delta_k, sqrt(D1) grows by at
// most delta_z and sqrt(D2) shrinks by at most the largest delta of the other
// centroids (triangle inequality; Hamerly 2010).  cum[z] adds those two per
// cluster and step, rounded up, so the point needs no distances while
//   slack - margin + cum[z] at its decision (rounded down) > cum[z] now,
// margin covering the FP64 rounding of the oracle's own distances.  Otherwise
// it is decided again from all K centroids: its label is then the FP64
// argmin as in every step.  The sums are exact integers, so taking a point
// out of its old cluster and adding it to the new one gives the same totals
// as adding all points again.  A step over points that keep their labels reads
// 5 bytes a point (0.5 GB for 1e8 points: 75 us at the memory's rate).  While the
// centroids move far nearly every point is open; the next step is then a first
// step again, in large sets the step kernels' (kSettled, kPlainMin).
//
// A 256-point warp-tile with more than kHeavy open points goes through the
// fused kernel's screen whole; fewer are listed and decided one per lane
// (run_pass in km_fast_tile.cuh, shared with the batched runs).
#include <algorithm>

#include "km_fast_tile.cuh"
#include "km_tables.cuh"
#include "km_i128.cuh"

namespace km {

namespace {

__device__ __forceinline__ unsigned long long run_clock() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
  return t;
}

// All blocks have arrived `target` times in all (monotone counter, one block's
// thread 0 per arrival).  Gives up after limit_ns; the result is the block's.
__device__ bool grid_wait(unsigned int* bar, unsigned int target, unsigned long long limit_ns) {
  __shared__ int s_ok;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) {
    atomicAdd(bar, 1u);
    int ok = 0;
    const unsigned long long t0 = run_clock();
    for (unsigned int spin = 0;; ++spin) {
      unsigned int v;
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(bar) : "memory");
      if (v >= target) { ok = 1; break; }
      if ((spin & 255u) == 255u && run_clock() - t0 > limit_ns) break;
    }
    __threadfence();
    s_ok = ok;
  }
  __syncthreads();
  return s_ok != 0;
}

// The block's own values: centroids, drift sums and tables (in shared memory
// when they fit beside the fused kernel's layout without costing a resident
// block, else in the block's slice of global memory).
struct RunPriv {
  double* mu;    // [k][D]
  float* cum;    // [k] drift so far, rounded up in every step
  float4* ctil;  // [k]
  __device__ RunPriv(unsigned char* p, int k, int D) {
    ctil = reinterpret_cast<float4*>(p);
    mu = reinterpret_cast<double*>(ctil + k);
    cum = reinterpret_cast<float*>(mu + (size_t)k * D);
  }
};

// KG as in the fused kernel (the table is read from shared memory: the
// constant bank cannot change while a kernel runs).
template <int D, int KG>
__global__ void __launch_bounds__(kThreads, KM_MINB) run_fast_kernel(RunArgs ra) {
  constexpr int DP = D + 1, WIN = 2 * D + 1, GS = FastSmem<D>::GS;
  extern __shared__ __align__(16) unsigned char smraw[];
  __shared__ IterConst s_ic;
  __shared__ double s_e2;
  __shared__ int s_empty;
  const FastArgs& a = ra.f;
  if (a.ls->done) return;  // written by block 0 only behind a wait for every block
  const int nbuf = a.nwin == 1 ? 1 : 2;
  FastSmem<D> sm(smraw, a.kpad, a.k, a.nwin, nbuf);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int k = a.k, kpad = KG > 0 ? 4 * KG : a.kpad, nwin = a.nwin;
  const int cols = k * DP;
  RunPriv pv(ra.priv_sh ? smraw + ra.priv_sh : ra.priv + (size_t)blockIdx.x * ra.priv_stride, k, D);
  // running totals of (cluster, coordinate): low word, high word, the cluster's count, unused
  long long* tot = ra.tot + (size_t)blockIdx.x * k * D * 4;
  // between the passes the point buffers hold the update's values
  double* s_df2 = reinterpret_cast<double*>(sm.xbuf);  // [k][D] squared moves
  double* sB = s_df2 + (size_t)k * D;                  // [k]
  double* s_red = sB + k;                              // [256]

  const DataConst dc = *a.dc;
  float s[D];
  unsigned long long s2[D];
#pragma unroll
  for (int j = 0; j < D; ++j) { s[j] = dc.s[j]; s2[j] = dup2(dc.s[j]); }
  const double grid_unit = __hiloint2double((1023 + dc.G0) << 20, 0);  // 2^G0
  const int iter0 = a.ls->iter, max_iter = a.ls->max_iter, e_mode = a.ls->e_mode;
  const double tol = a.ls->tol;

  uint32_t* wwarp = sm.win + (size_t)warp * nwin * (k + 1) * WIN;
  uint32_t* wmine = wwarp + (size_t)(nwin == 4 ? (lane >> 3) : nwin == 2 ? (lane >> 4) : 0) * (k + 1) * WIN;
  long long* acc = sm.acc;
  uint32_t* q = sm.queue + (size_t)warp * kWarpQueue;
  float* xb = sm.xbuf + (size_t)warp * nbuf * D * kWarpTile;
  // tiles are dealt over the blocks first, so few tiles still reach every SM
  const int wid = blockIdx.x + warp * gridDim.x;
  const int wtot = gridDim.x * kWarps;
  const int ntiles = (int)a.ntiles;

  for (int c = tid; c < k * D; c += kThreads) pv.mu[c] = ra.mu[c];
  for (int c = tid; c < k; c += kThreads) pv.cum[c] = ra.resume ? ra.cum0[c] : 0.f;
  for (int c = tid; c < 4 * k * D; c += kThreads) tot[c] = ra.resume ? ra.tot0[c] : 0;
  for (int c = tid; c < cols; c += kThreads) acc[c] = 0;
  for (int c = tid; c < kWarps * nwin * (k + 1) * WIN; c += kThreads) sm.win[c] = 0u;
  if (tid < 2) sm.cnt[tid] = 0;
  __syncthreads();
  auto tables = [&]() {  // screen tables of pv.mu (every thread)
    fast_screen_tables(pv.mu, dc.s, dc.A_max, k, D, kpad, ra.tie_rel, pv.ctil, &s_ic, sm.tab, sB, sm.gtab, GS);
    __syncthreads();
  };
  tables();

  bool first = !ra.resume;  // this step adds every point (the totals start from zero)
  for (int step = 0;; ++step) {
    FastCtx cx;
    RunTile rt;
    {
      const IterConst& ic = s_ic;
      cx.L = (uint32_t)ic.L; cx.mul = ic.mul; cx.kmask = ic.mul - 1u;
      cx.ehi = __float_as_uint(ic.M) >> (32 - ic.L);
      cx.M = ic.M;
      const float ulp = __uint_as_float(__float_as_uint(ic.M) & 0x7f800000u) * 0x1p-23f;
      cx.c0 = ic.thr_c0 * ulp;
      cx.cA = (ic.thr_cA + ic.tau * ic.G) * ulp;
      cx.tau = ic.tau;
      cx.chi2 = dup2(dc.C_hi); cx.clo2 = dup2(dc.C_lo);
      cx.k = k; cx.kpad = kpad;
      rt.invs = 1.f / (ic.G * ulp);  // powers of two: exact
    }
    rt.slack = ra.slack; rt.z = ra.z; rt.cum = pv.cum; rt.margin = ra.margin;
    rt.first = first;
    const float B_max = s_ic.B_max;
    int nflag = 0, n64 = 0;
    run_pass<D, KG, false>(a, sm, cx, s2, s, dc, rt, pv.ctil, pv.mu, B_max, acc, q, wwarp, wmine, xb, nbuf, wid, wtot,
                           ntiles, lane, nflag, n64);
    if (lane == 0 && nflag) atomicAdd(&sm.cnt[0], nflag);
    if (n64) atomicAdd(&sm.cnt[1], n64);
    __syncthreads();
    // the block's change of every column, split so that 64-bit words hold the
    // sums over all blocks: value = high 2^54 + low, |low| <= 2^53 (the high
    // part is mostly zero).  The table is kept kRep times, block b adding to
    // copy b % kRep: with one copy all blocks' atomics meet on the same words
    // (13 us a step for K = 32 once every block has changes)
    const int words = 2 * (cols + 2);
    unsigned long long* tab = ra.delta + (size_t)(step % 3) * ra.rep * words;
    unsigned long long* dl = tab + (size_t)((int)blockIdx.x % ra.rep) * words;
    for (int c = tid; c < cols; c += kThreads) {
      const long long v = acc[c];
      if (v) {
        const long long h = (v + (1ll << 53)) >> 54;
        atomicAdd(dl + 2 * c, (unsigned long long)(v - (h << 54)));
        if (h) atomicAdd(dl + 2 * c + 1, (unsigned long long)h);
        acc[c] = 0;
      }
    }
    if (tid < 2 && sm.cnt[tid]) {
      atomicAdd(dl + 2 * (cols + tid), (unsigned long long)sm.cnt[tid]);
      sm.cnt[tid] = 0;
    }
    if (tid == 0) s_empty = 0;
    if (!grid_wait(ra.bar, (unsigned)(step + 1) * gridDim.x + ra.wait_more, ra.wait_ns)) {
      if (tid == 0) a.ls->error = 3;
      return;
    }
    // this step's table was the one before last's; the last step's is read
    // by no block any more (all have arrived) and is added to again only after
    // the next wait: clear it
    {
      unsigned long long* old = ra.delta + (size_t)((step + 2) % 3) * ra.rep * words;
      for (int c = blockIdx.x * kThreads + tid; c < ra.rep * words; c += gridDim.x * kThreads) old[c] = 0ull;
    }
    // sum over the copies of the table's entry w: low and high words
    auto entry = [&](int w, long long& lo, long long& hi) {
      lo = 0;
      hi = 0;
#pragma unroll 4
      for (int r = 0; r < ra.rep; ++r) {
        const longlong2 v = __ldcg(reinterpret_cast<const longlong2*>(tab + (size_t)r * words + w));
        lo += v.x;
        hi += v.y;
      }
    };
    // centroids: a thread per (cluster, coordinate) keeps that column's running
    // total and its own copy of the cluster's count, so one round of loads and
    // one barrier do
    double e2p = 0.0;
    int empty = 0;
    for (int qd = tid; qd < k * D; qd += kThreads) {
      const int c = qd / D, j = qd - c * D;
      long long plo, phi, clo, chi;
      entry(2 * (c * DP + j), plo, phi);
      entry(2 * (c * DP + D), clo, chi);
      ulonglong2 pt = *reinterpret_cast<const ulonglong2*>(tot + 4 * qd);
      long long nn = tot[4 * qd + 2];
      if (first) { pt.x = 0ull; pt.y = 0ull; nn = 0; }
      nn += clo + (chi << 54);
      const double old = pv.mu[qd];
      unsigned long long tl = pt.x;
      long long th = (long long)pt.y;
      add128p(tl, th, (unsigned long long)phi << 54, phi >> 10);
      add128p(tl, th, (unsigned long long)plo, plo >> 63);
      *reinterpret_cast<ulonglong2*>(tot + 4 * qd) = make_ulonglong2(tl, (unsigned long long)th);
      tot[4 * qd + 2] = nn;
      double nw = old;
      // 2^G0 is a normal number and the product exact, as the update kernel's ldexp
      if (nn > 0) nw = __ddiv_rn(i128_to_double((long long)tl, th) * grid_unit, (double)nn);
      const double df = __dsub_rn(nw, old);
      const double dd = __dmul_rn(df, df);
      e2p = __dadd_rn(e2p, dd);
      s_df2[qd] = dd;
      pv.mu[qd] = nw;
      empty += j == 0 && nn == 0;
    }
    s_red[tid] = e2p;
    if (empty) atomicAdd(&s_empty, empty);
    __syncthreads();
    // E^2 by the update kernel's tree over 256 threads (levels that only add
    // zeros left out)
#pragma unroll
    for (int w = kThreads / 2; w >= 32; w >>= 1) {
      if (k * D <= w) continue;
      if (tid < w) s_red[tid] = __dadd_rn(s_red[tid], s_red[tid + w]);
      __syncthreads();
    }
    if (tid < 32) {
      double t = s_red[tid];
#pragma unroll
      for (int w = 16; w > 0; w >>= 1) t = __dadd_rn(t, __shfl_down_sync(0xffffffffu, t, w));
      if (tid == 0) s_e2 = t;
    }
    {
      // every warp forms the centroids' moves, rounded up, the largest with its
      // centroid and the second largest; thread c keeps centroid c's
      float m1 = -1.f, m2 = -1.f, mine = 0.f;
      int i1 = -1;
      for (int c = lane; c < k; c += 32) {
        double t = 0.0;
#pragma unroll
        for (int j = 0; j < D; ++j) t = __dadd_ru(t, s_df2[c * D + j]);
        const float v = sqrt_up(t);
        if (c == tid) mine = v;
        if (v > m1) { m2 = m1; m1 = v; i1 = c; }
        else if (v > m2) m2 = v;
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        const float p1 = __shfl_xor_sync(0xffffffffu, m1, o), p2 = __shfl_xor_sync(0xffffffffu, m2, o);
        const int pi = __shfl_xor_sync(0xffffffffu, i1, o);
        if (p1 > m1 || (p1 == m1 && pi < i1)) { m2 = fmaxf(m1, p2); m1 = p1; i1 = pi; }
        else m2 = fmaxf(m2, p1);
      }
      m2 = fmaxf(m2, 0.f);
      if (tid < k)  // k <= 256 threads
        pv.cum[tid] = fminf(__fadd_ru(pv.cum[tid], __fadd_ru(mine, tid == i1 ? m2 : m1)), kDriftMax);
    }
    tables();  // its barriers also publish s_e2 and the drift sums
    const double E2 = s_e2;
    const int iter = iter0 + step + 1;
    // sqrt(E2) < tol; the root itself only where E2 is not clearly above tol^2
    const bool conv = e_mode == 1 ? E2 < tol : !(tol <= 0.0) && E2 <= tol * tol * 1.001 + 1e-300 && sqrt(E2) < tol;
    const bool done = conv || iter >= max_iter;
    if (done || step + 1 == ra.steps) {
      // block 0 leaves the state of a stopped (or paused) loop
      if (blockIdx.x != 0) return;
      for (int c = tid; c < k * D; c += kThreads) {
        ra.mu[c] = pv.mu[c];
        if (c % D == 0) ra.counts[c / D] = tot[4 * c + 2];
      }
      for (int c = tid; c < k; c += kThreads) ra.cum0[c] = pv.cum[c];
      for (int c = tid; c < 4 * k * D; c += kThreads) ra.tot0[c] = tot[c];
      if (tid == 0) {
        LoopState* ls = a.ls;
        ls->E2 = E2;
        ls->E = sqrt(E2);
        ls->iter = iter;
        ls->empty = s_empty;
        if (conv) ls->converged = 1;
        long long nf, n6, unused;
        entry(2 * cols, nf, unused);
        entry(2 * cols + 2, n6, unused);
        ls->last_flagged = (unsigned long long)nf;
        ls->last_fp64 = (unsigned long long)n6;
        ls->last_overflowed = 0ull;
        ls->done = done ? 1 : 0;
      }
      // the step kernels' tables of the final centroids
      for (int c = tid; c < a.kpad * DP; c += kThreads) ra.tab_out[c] = sm.tab[c];
      for (int c = tid; c < k; c += kThreads) ra.ctil_out[c] = pv.ctil[c];
      if (tid == 0) *ra.ic_out = s_ic;
      return;
    }
    first = E2 > ra.restart_e2;  // the same in every block
    if (first) {
      // the next step reads no label and no slack: the drift starts over
      for (int c = tid; c < k; c += kThreads) pv.cum[c] = 0.f;
      __syncthreads();
    }
  }
}

__global__ void run_totals_kernel(int d, int k, const long long* __restrict__ tot0, long long* __restrict__ out) {
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= k * (d + 1)) return;
  const int c = q / (d + 1), j = q - c * (d + 1);
  const long long* t = tot0 + 4 * ((size_t)c * d + (j < d ? j : 0));
  out[2 * (size_t)q] = j < d ? t[0] : t[2];
  out[2 * (size_t)q + 1] = j < d ? t[1] : 0;
}

template <int D, int KG>
int run_blocks(size_t smem) {
  int nb = 0;
  if (allow_max_smem<run_fast_kernel<D, KG>>() != cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, run_fast_kernel<D, KG>, kThreads, smem) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return nb;
}

template <int D, int KG>
cudaError_t run_launch(int grid, size_t smem, cudaStream_t st, const RunArgs& a) {
  cudaError_t e = allow_max_smem<run_fast_kernel<D, KG>>();
  if (e != cudaSuccess) return e;
  void* args[] = {const_cast<RunArgs*>(&a)};
  return cudaLaunchCooperativeKernel(reinterpret_cast<void*>(run_fast_kernel<D, KG>), dim3(grid), dim3(kThreads), args,
                                     smem, st);
}

}  // namespace

// The instances of the fused kernel that read their table from shared memory.
// With the group count at run time in place of kpad = 32 and 256 (d = 3) a run is
// up to 3 % (K = 32; N = 1e5 to 4e6, 10 and 40 steps) and 1 % (K = 250) slower.
#define KM_RUN_DISPATCH(FN, d, kpad, ...)             \
  do {                                                \
    switch (d) {                                      \
      case 1: return FN<1, 0>(__VA_ARGS__);           \
      case 2: return FN<2, 0>(__VA_ARGS__);           \
      case 4: return FN<4, 0>(__VA_ARGS__);           \
      default: break;                                 \
    }                                                 \
    if ((kpad) == 32) return FN<3, 8>(__VA_ARGS__);   \
    if ((kpad) == 256) return FN<3, 64>(__VA_ARGS__); \
    return FN<3, 0>(__VA_ARGS__);                     \
  } while (0)

size_t run_priv_bytes(int d, int k) { return ((size_t)k * (16 + 8 * d + 4) + 15) & ~size_t(15); }

// Copies of the table of changes: as many as 16 KB a step hold, up to 8.
int run_rep(int d, int k) { return (int)std::max<size_t>(1, std::min<size_t>(8, 1024 / ((size_t)k * (d + 1) + 2))); }

int run_blocks_per_sm(int d, int kpad, size_t smem) { KM_RUN_DISPATCH(run_blocks, d, kpad, smem); }

cudaError_t launch_run_totals(int d, int k, const long long* tot0, long long* out, cudaStream_t st) {
  run_totals_kernel<<<(k * (d + 1) + 255) / 256, 256, 0, st>>>(d, k, tot0, out);
  return cudaGetLastError();
}

cudaError_t launch_run_fast(int d, int grid, size_t smem, cudaStream_t st, const RunArgs& a) {
  cudaError_t e = cudaMemsetAsync(a.delta, 0, run_delta_words(d, a.f.k, a.rep) * sizeof(unsigned long long), st);
  if (e != cudaSuccess) return e;
  KM_RUN_DISPATCH(run_launch, d, a.f.kpad, grid, smem, st, a);
}

}  // namespace km
