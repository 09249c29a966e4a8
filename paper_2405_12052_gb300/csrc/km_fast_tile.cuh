// The fused FP32 step's tile machinery (d <= 4, K <= 256), shared by the
// per-step kernel, the batched kernel and the whole-run kernel: shared-memory
// layout, point staging, the FFMA2 screen over groups of 4 centroids, the
// winning group's recompute, the flag test, labels and exact sums of one
// 256-point warp-tile, and the queue of points decided one by one.
#pragma once
#include "km_fast_common.cuh"

namespace km {

namespace {

constexpr int kGpUnroll = 1;  // the shared-memory-table screen keeps its group-pair loop rolled

// Shared memory of the fused kernel.  The windows, point buffers and queues
// are private to one warp; the int64 totals are the block's (windows are
// flushed into them with 64-bit shared atomics).  With one window per warp
// (large K) the points are single-buffered, so that two blocks fit on an SM.
template <int D>
struct FastSmem {
  static constexpr int DP = D + 1, WIN = 2 * D + 1;
  static constexpr int GS = (DP & 1) ? DP : DP + 1;  // float4 slots per group (odd: no bank conflicts)
  unsigned long long* tab;  // [kpad][DP] screen table, packed (a, a) pairs (block)
  long long* acc;           // [k][DP] int64 totals (block)
  float4* gtab;             // [kpad/4][GS] screen table by group: slot j = coefficient j of the 4 centroids
  float4* ctil;             // [k] fp32 centroids for the re-check (block; two-window layout only, else global)
  float* xbuf;              // [kWarps][nbuf][D][kWarpTile] points (double-buffered when nbuf = 2)
  uint32_t* queue;          // [kWarps][kWarpQueue] flagged points
  uint32_t* win;            // [kWarps][nwin][k+1][WIN] 32-bit windows (per 8 lanes when nwin = 4, per half-warp when 2); bin k discards
  int* cnt;                 // [2]: flagged, fp64-decided (block totals)
  FastSmem() = default;
  __device__ FastSmem(unsigned char* sm, int kpad, int k, int nwin, int nbuf) {
    tab = reinterpret_cast<unsigned long long*>(sm);
    acc = reinterpret_cast<long long*>(tab + (size_t)kpad * DP);
    gtab = reinterpret_cast<float4*>(acc + (size_t)k * DP + (k * DP & 1));
    ctil = nbuf == 2 ? gtab + (size_t)(kpad / 4) * GS : nullptr;
    xbuf = reinterpret_cast<float*>(gtab + (size_t)(kpad / 4) * GS + (nbuf == 2 ? k : 0));
    queue = reinterpret_cast<uint32_t*>(xbuf + (size_t)kWarps * nbuf * D * kWarpTile);
    win = queue + (size_t)kWarps * kWarpQueue;
    cnt = reinterpret_cast<int*>(win + (size_t)kWarps * nwin * (k + 1) * WIN);
  }
};

// Asynchronous copy of this lane's two 16-byte chunks of each coordinate row
// of warp-tile `base` (points base+4*lane.. and base+128+4*lane..) into a
// warp buffer; chunks past N are zero-filled and read nothing past N.
template <int D>
__device__ __forceinline__ void prefetch_tile(const FastArgs& a, float* xb, int64_t base, int lane) {
  if (base + kWarpTile <= a.n) {  // a full tile: no bounds logic
#pragma unroll
    for (int g = 0; g < kNG; ++g) {
      const int off = g * kGS + 4 * lane;
#pragma unroll
      for (int j = 0; j < D; ++j) {
        const float* src = a.x + (int64_t)j * a.ld + base + off;
        const uint32_t dst = (uint32_t)__cvta_generic_to_shared(xb + j * kWarpTile + off);
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src));
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
    return;
  }
#pragma unroll
  for (int g = 0; g < kNG; ++g) {
    const int off = g * kGS + 4 * lane;
    const int64_t i0 = base + off;
    const int64_t rem = a.n - i0;
    const int bytes = rem >= 4 ? 16 : (rem > 0 ? (int)rem * 4 : 0);
#pragma unroll
    for (int j = 0; j < D; ++j) {
      const float* src = a.x + (int64_t)j * a.ld + (bytes ? i0 : 0);
      const uint32_t dst = (uint32_t)__cvta_generic_to_shared(xb + j * kWarpTile + off);
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(bytes));
    }
  }
  asm volatile("cp.async.commit_group;" ::: "memory");
}

// Re-decide the points in this warp's queue (warp-level: lanes take
// entries; windows are flushed every 64 rounds with four windows per warp,
// 32 with two, 16 with one: <= 512 additions per bin).
template <int D>
__device__ void drain_warp_queue(const FastArgs& a, FastSmem<D>& sm, uint32_t* q, int qn, int wid,
                                 int wtot, uint32_t* wwarp, uint32_t* wmine, long long* acc, int lane,
                                 const float* s, const DataConst& dc, float B_max, float tau, int& n64) {
  flush_windows<D>(wwarp, acc, a.k, a.nwin, lane, dc.bits_C_hi, dc.bits_C_lo);
  const int rmask = a.nwin == 4 ? 63 : a.nwin == 2 ? 31 : 15;
  for (int r = 0, b = 0; b < qn; ++r, b += 32) {
    const int e = b + lane;
    if (e < qn) {
      const uint32_t loc = q[e];
      const int64_t tile = (int64_t)wid + (int64_t)(loc >> 8) * wtot;
      const int64_t i = tile * kWarpTile + (loc & 255u);
      float xo[D];
#pragma unroll
      for (int j = 0; j < D; ++j) xo[j] = a.x[(int64_t)j * a.ld + i];
      bool used64;
      const int kk = recheck_fast<D>(xo, s, sm.ctil ? sm.ctil : a.ctil, a.mu, a.k, B_max, tau, used64);
      n64 += used64 ? 1 : 0;
      if (a.store_labels) {
        if (a.labels8) a.labels8[i] = (uint8_t)kk;
        else a.labels[i] = kk;
      }
      accumulate_point<D>(wmine, kk, xo, dc.C_hi, dc.C_lo);
    }
    if ((r & rmask) == rmask) flush_windows<D>(wwarp, acc, a.k, a.nwin, lane, dc.bits_C_hi, dc.bits_C_lo);
  }
  flush_windows<D>(wwarp, acc, a.k, a.nwin, lane, dc.bits_C_hi, dc.bits_C_lo);
}

// Per-launch constants of the fused kernel, in registers.  The flag test is
// evaluated in units of r: a point is accepted when
//   r2 - r1 > c0 + A cA + tau (r2 - M),
// r1 <= r2 its two smallest screen values, A = ||x~||^2.  r2 - r1 and r2 - M
// are exact (one binade); c0 and cA are the ulp-unit constants of the update
// kernel times the binade's ulp (a power of two).
struct FastCtx {
  uint32_t mul, L, kmask, ehi;  // ehi: the top L bits shared by every r's bit pattern
  float M, c0, cA, tau;
  unsigned long long chi2, clo2;
  int k, kpad;
};

// bits(v) * 2^L + idx: the screen value with an index in its low L bits.
// With a compile-time L this is a shift and an add (integer ALU pipe).
template <int LB>
__device__ __forceinline__ float pack_idx(float v, const FastCtx& cx, uint32_t idx) {
  if constexpr (LB > 0) return __uint_as_float((__float_as_uint(v) << LB) + idx);
  else return __uint_as_float(imad(__float_as_uint(v), cx.mul, idx));
}
// The screen value r back from a packed value (one funnel shift).
template <int LB>
__device__ __forceinline__ float unpack_val(float w, const FastCtx& cx) {
  return __uint_as_float(__funnelshift_r(__float_as_uint(w), cx.ehi, LB > 0 ? LB : cx.L));
}

constexpr uint32_t kRecheck = 0x80000000u;  // whole-run queue entry that the screen has already flagged

// What the whole-run kernel keeps per point besides the label: z and the
// slack, a lower bound of sqrt(D2) - sqrt(D1) at the step that decided the
// point plus the drift of its cluster up to that step (see km_run_fast.cu).
struct RunTile {
  float* slack;      // [N]
  uint8_t* z;        // [N] labels
  const float* cum;  // [K] drift per cluster so far, rounded up (shared memory)
  float invs;        // 2^-sigma: screen units to squared distances
  float margin;      // least slack that counts (FP64 rounding of the oracle's distances)
  int first;         // 1: the first step (every point is added, none taken away)
};

// The slack of a point from its two smallest screen values v1, v2, its flag
// threshold T and A = ||x~||^2.  For every other centroid k the flag test's
// bound gives D_k - D_1 >= dl = (v2 - v1 - T) 2^-sigma, and D_1 <= d1, so
// sqrt(D_k) - sqrt(D_1) >= dl / (sqrt(d1 + dl) + sqrt(d1)) (decreasing in d1);
// the factors cover the roundings here (approximate roots and quotient, a few
// ulps) and of A.
__device__ __forceinline__ float sqrt_approx(float x) {
  float r;
  asm("sqrt.approx.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ float screen_slack(float v1, float v2, float T, float A, float M, const RunTile& rt,
                                              int label) {
  const float dl = (v2 - v1 - T) * rt.invs * 0.9999f;
  const float d1 = fmaxf(fmaf(v1 - M + T, rt.invs, A * 1.0001f), 0.f) * 1.0001f + 1e-37f;
  return __fadd_rd(__fdividef(dl * 0.9998f, sqrt_approx(d1 + dl) + sqrt_approx(d1)) - rt.margin, rt.cum[label]);
}

// Screen of one group of 4 centroids (table rows tr) for this lane's 8
// points: r = n_k + sum_j x~_j a_kj by one FFMA2 chain per pair of points,
// the group minimum by FMNMX3 + FMNMX, packed with the group's first index.
template <int D, int LB>
__device__ __forceinline__ void screen_group(const unsigned long long* tr, const unsigned long long (&X)[D][kPts / 2],
                                             uint32_t g4, const FastCtx& cx, float (&gm)[kPts]) {
  constexpr int DP = D + 1;
  unsigned long long T[4][DP];
  if constexpr (D <= 3) {
#pragma unroll
    for (int c = 0; c < 4; ++c)
#pragma unroll
      for (int j = 0; j < DP; ++j) T[c][j] = tr[c * DP + j];
  }
#pragma unroll
  for (int pp = 0; pp < kPts / 2; ++pp) {
    if constexpr (D > 3) {  // reloaded per pair of points: fewer live registers
#pragma unroll
      for (int c = 0; c < 4; ++c)
#pragma unroll
        for (int j = 0; j < DP; ++j) T[c][j] = tr[c * DP + j];
    }
    float v0[4], v1[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      unsigned long long r = T[c][D];
#pragma unroll
      for (int j = 0; j < D; ++j) r = ffma2(X[j][pp], T[c][j], r);
      unpack2(r, v0[c], v1[c]);
    }
    gm[2 * pp] = pack_idx<LB>(fminf(fmin3(v0[0], v0[1], v0[2]), v0[3]), cx, g4);
    gm[2 * pp + 1] = pack_idx<LB>(fminf(fmin3(v1[0], v1[1], v1[2]), v1[3]), cx, g4);
  }
}

// Screen table in the constant bank (one process-wide copy per device,
// kpad <= 64): the compile-time-unrolled screen reads its coefficients as
// uniform operands, so they take no vector registers and no shared-memory
// loads.  Written by a device-to-device copy before each launch that uses it.
__constant__ union {
  unsigned long long u[kConstTabWords];  // packed (a, a) pairs, as in the global table
  float f[2 * kConstTabWords];           // f[2 i] = the coefficient of pair i
} c_screen_tab;

// Running top-2 over groups, two groups at a time: with lo <= hi the pair's
// packed minima, m1' = min(m1, lo) and m2' = min(m2, hi, max(m1, lo)).
template <bool FIRST>
__device__ __forceinline__ void top2_pair(float (&m1)[kPts], float (&m2)[kPts], const float (&ga)[kPts],
                                          const float (&gb)[kPts]) {
#pragma unroll
  for (int p = 0; p < kPts; ++p) {
    const float lo = fminf(ga[p], gb[p]), hi = fmaxf(ga[p], gb[p]);
    if constexpr (FIRST) {
      m1[p] = lo;
      m2[p] = hi;
    } else {
      m2[p] = fmin3(m2[p], hi, fmaxf(m1[p], lo));
      m1[p] = fminf(m1[p], lo);
    }
  }
}

// Screen of groups G0/4 and G0/4 + 1 (centroids G0 .. G0 + 7) from the
// constant-bank table, one pair of points at a time: 8 FFMA2 chains, the two
// group minima per point, and the running top-2 update.  G0 is a
// compile-time constant after unrolling, so every table operand has a fixed
// offset.
template <int D, int LB, bool FIRST>
__device__ __forceinline__ void screen_pair_ct(int G0, const unsigned long long (&X)[D][kPts / 2], const FastCtx& cx,
                                               float (&m1)[kPts], float (&m2)[kPts]) {
  constexpr int DP = D + 1;
#pragma unroll
  for (int pp = 0; pp < kPts / 2; ++pp) {
    float a0[4], a1[4], b0[4], b1[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      unsigned long long ra = c_screen_tab.u[(G0 + c) * DP + D], rb = c_screen_tab.u[(G0 + 4 + c) * DP + D];
#pragma unroll
      for (int j = 0; j < D; ++j) {
        ra = ffma2(X[j][pp], c_screen_tab.u[(G0 + c) * DP + j], ra);
        rb = ffma2(X[j][pp], c_screen_tab.u[(G0 + 4 + c) * DP + j], rb);
      }
      unpack2(ra, a0[c], a1[c]);
      unpack2(rb, b0[c], b1[c]);
    }
    const float ga[2] = {pack_idx<LB>(fminf(fmin3(a0[0], a0[1], a0[2]), a0[3]), cx, (uint32_t)G0),
                         pack_idx<LB>(fminf(fmin3(a1[0], a1[1], a1[2]), a1[3]), cx, (uint32_t)G0)};
    const float gb[2] = {pack_idx<LB>(fminf(fmin3(b0[0], b0[1], b0[2]), b0[3]), cx, (uint32_t)G0 + 4u),
                         pack_idx<LB>(fminf(fmin3(b1[0], b1[1], b1[2]), b1[3]), cx, (uint32_t)G0 + 4u)};
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      const int p = 2 * pp + e;
      const float lo = fminf(ga[e], gb[e]), hi = fmaxf(ga[e], gb[e]);
      if constexpr (FIRST) {
        m1[p] = lo;
        m2[p] = hi;
      } else {
        m2[p] = fmin3(m2[p], hi, fmaxf(m1[p], lo));
        m1[p] = fminf(m1[p], lo);
      }
    }
  }
}

// One warp-tile: grouped screen, exact recompute of the winning group, flags,
// labels and exact sums.  FULL: all 256 points exist (no bounds checks).
// KG: groups of 4 centroids (kpad / 4) when fixed at compile time, else 0.
// RUN (whole-run kernel): also the slack of every point, and only the points
// whose label changed enter the sums (added to the new cluster, taken from the
// old one); a flagged point keeps its old label until the queue decides it.
template <int D, int KG, bool CT, bool FULL, bool RUN = false>
__device__ __forceinline__ void process_tile(const FastArgs& a, FastSmem<D>& sm, const FastCtx& cx,
                                             const unsigned long long* s2, const float* xcur, int64_t base,
                                             int m, int lane, uint32_t* wmine, uint32_t* q, int& qn,
                                             const RunTile* rt = nullptr) {
  constexpr int DP = D + 1, WIN = 2 * D + 1, GS = FastSmem<D>::GS;
  constexpr int LB = KG == 2 ? 3 : KG == 4 ? 4 : KG == 8 ? 5 : KG == 16 ? 6 : KG == 32 ? 7 : KG == 64 ? 8 : 0;
  static_assert(KG == 0 || LB > 0, "compile-time group counts: 2, 4, 8, 16, 32, 64");
  // this lane's points: base + g*128 + 4*lane + q, g in {0,1}, q in 0..3;
  // pair pp holds points 2pp, 2pp+1.  X = x~ = fl(x - s) per pair.
  unsigned long long X[D][kPts / 2];
#pragma unroll
  for (int g = 0; g < kNG; ++g)
#pragma unroll
    for (int j = 0; j < D; ++j) {
      const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(xcur + j * kWarpTile + g * kGS + 4 * lane);
      X[j][2 * g] = fsub2(v.x, s2[j]);
      X[j][2 * g + 1] = fsub2(v.y, s2[j]);
    }
  // Grouped screen over pairs of groups (kpad is a multiple of 8).
  float m1[kPts], m2[kPts];
  if constexpr (CT) {
    static_assert(KG > 0, "the constant-bank screen needs a compile-time group count");
    screen_pair_ct<D, LB, true>(0, X, cx, m1, m2);
#pragma unroll
    for (int gp = 1; gp < KG / 2; ++gp) screen_pair_ct<D, LB, false>(8 * gp, X, cx, m1, m2);
  } else {
    {
      float ga[kPts], gb[kPts];
      screen_group<D, LB>(sm.tab, X, 0u, cx, ga);
      screen_group<D, LB>(sm.tab + 4 * DP, X, 4u, cx, gb);
      top2_pair<true>(m1, m2, ga, gb);
    }
  }
  if constexpr (CT) {
  } else if constexpr (KG > 0) {
#pragma unroll kGpUnroll
    for (int gp = 1; gp < KG / 2; ++gp) {
      float ga[kPts], gb[kPts];
      screen_group<D, LB>(sm.tab + (size_t)(8 * gp) * DP, X, 8u * gp, cx, ga);
      screen_group<D, LB>(sm.tab + (size_t)(8 * gp + 4) * DP, X, 8u * gp + 4u, cx, gb);
      top2_pair<false>(m1, m2, ga, gb);
    }
  } else {
#pragma unroll 1
    for (int g8 = 8; g8 < cx.kpad; g8 += 8) {
      float ga[kPts], gb[kPts];
      screen_group<D, 0>(sm.tab + (size_t)g8 * DP, X, (uint32_t)g8, cx, ga);
      screen_group<D, 0>(sm.tab + (size_t)(g8 + 4) * DP, X, (uint32_t)g8 + 4u, cx, gb);
      top2_pair<false>(m1, m2, ga, gb);
    }
  }

  // Epilogue: the winning group is recomputed exactly (the same FMA chain,
  // two centroids per FFMA2), its values packed with the index within the
  // group; the label, the runner-up and the flag follow.
  // bin[p]: the label, or k (the discard bin of the sums) for a flagged or
  // padding point; a flagged point's label is written by the re-check.
  int lab[kPts];
  uint32_t fbits = 0u, dbits = 0u;  // flagged; not accumulated here
  float Ap[2];
  [[maybe_unused]] float slk[4];
#pragma unroll
  for (int p = 0; p < kPts; ++p) {
    if ((p & 1) == 0) {
      // A = ||x~||^2 exactly as the data scan that bounds it: x0*x0, then FMAs.
      unsigned long long a2 = ffma2(X[0][p >> 1], X[0][p >> 1], 0ull);
#pragma unroll
      for (int j = 1; j < D; ++j) a2 = ffma2(X[j][p >> 1], X[j][p >> 1], a2);
      unpack2(a2, Ap[0], Ap[1]);
    }
    const uint32_t gsel = __float_as_uint(m1[p]) & cx.kmask;  // the group's first index
    const ulonglong2* gt = reinterpret_cast<const ulonglong2*>(sm.gtab + (size_t)(gsel >> 2) * GS);
    float r0, r1, r2, r3;
    {
      const ulonglong2 nv = gt[D];
      unsigned long long rA = nv.x, rB = nv.y;
#pragma unroll
      for (int j = 0; j < D; ++j) {
        float lo, hi;
        unpack2(X[j][p >> 1], lo, hi);
        const unsigned long long xx = dup2((p & 1) ? hi : lo);
        const ulonglong2 cv = gt[j];
        rA = ffma2(xx, cv.x, rA);
        rB = ffma2(xx, cv.y, rB);
      }
      unpack2(rA, r0, r1);
      unpack2(rB, r2, r3);
    }
    const float w0 = pack_idx<LB>(r0, cx, 0u), w1 = pack_idx<LB>(r1, cx, 1u);
    const float w2 = pack_idx<LB>(r2, cx, 2u), w3 = pack_idx<LB>(r3, cx, 3u);
    const float lo01 = fminf(w0, w1), hi01 = fmaxf(w0, w1);
    const float lo23 = fminf(w2, w3), hi23 = fmaxf(w2, w3);
    const float best = fminf(lo01, lo23);
    const float sec = fmin3(fmaxf(lo01, lo23), fminf(hi01, hi23), m2[p]);
    lab[p] = (int)(gsel | (__float_as_uint(best) & 3u));
    const float v1 = unpack_val<LB>(best, cx), v2 = unpack_val<LB>(sec, cx);
    const float T = fmaf(cx.tau, v2 - cx.M, fmaf(Ap[p & 1], cx.cA, cx.c0));
    bool f = !(v2 - v1 > T);
    // a label outside 0..K-1 (only a padding centroid could give one) is
    // never trusted: the point goes to the re-check
    if (cx.k < cx.kpad) f = f || lab[p] >= cx.k;
    bool valid = true;
    if constexpr (!FULL) valid = base + (p >> 2) * kGS + 4 * lane + (p & 3) < a.n;
    fbits |= ((f && valid) ? 1u : 0u) << p;
    dbits |= ((f || !valid) ? 1u : 0u) << p;
    if constexpr (RUN) {
      slk[p & 3] = f ? -1.f : screen_slack(v1, v2, T, Ap[p & 1], cx.M, *rt, lab[p]);
      if ((p & 3) == 3) {
        const int64_t i0 = base + (p >> 2) * kGS + 4 * lane;
        if constexpr (FULL) {
          *reinterpret_cast<float4*>(rt->slack + i0) = make_float4(slk[0], slk[1], slk[2], slk[3]);
        } else {
#pragma unroll
          for (int e = 0; e < 4; ++e) if (i0 + e < a.n) rt->slack[i0 + e] = slk[e];
        }
      }
    }
  }
  if (__any_sync(0xffffffffu, fbits != 0u)) {
    const int nf = __popc(fbits);
    int incl = nf;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int t = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += t;
    }
    int at = qn + incl - nf;
    for (uint32_t fb = fbits; fb; fb &= fb - 1u) {
      const int p = __ffs(fb) - 1;
      q[at++] = (RUN ? kRecheck : 0u) | (uint32_t)(m << 8) | (uint32_t)((p >> 2) * kGS + 4 * lane + (p & 3));
    }
    qn += __shfl_sync(0xffffffffu, incl, 31);
  }
  if constexpr (RUN) {
    const bool first = rt->first != 0;
#pragma unroll
    for (int g = 0; g < kNG; ++g) {
      const int64_t i0 = base + g * kGS + 4 * lane;
      // old labels of this lane's 4 points; the new word keeps a flagged
      // point's (in the first step the queue writes it whatever it is)
      uint32_t ow = 0u, nw = 0u;
      if (!first) {
        if constexpr (FULL) ow = *reinterpret_cast<const uint32_t*>(rt->z + i0);
        else {
#pragma unroll
          for (int e = 0; e < 4; ++e) if (i0 + e < a.n) ow |= (uint32_t)rt->z[i0 + e] << (8 * e);
        }
      }
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int p = 4 * g + e;
        nw |= (((dbits >> p) & 1u) ? ow & (255u << (8 * e)) : (uint32_t)lab[p] << (8 * e));
      }
      if constexpr (FULL) *reinterpret_cast<uint32_t*>(rt->z + i0) = nw;
      else {
#pragma unroll
        for (int e = 0; e < 4; ++e) if (i0 + e < a.n) rt->z[i0 + e] = (uint8_t)(nw >> (8 * e));
      }
      if (!first && nw != ow) {  // changed labels only (a flagged or padding point keeps its byte)
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const uint32_t old = (ow >> (8 * e)) & 255u, now = (nw >> (8 * e)) & 255u;
          if (now == old) continue;
          uint32_t* wa = wmine + now * WIN;
          uint32_t* wo = wmine + old * WIN;
          atomicAdd(&wa[0], 1u);
          atomicSub(&wo[0], 1u);
#pragma unroll
          for (int j = 0; j < D; ++j) {
            uint32_t bh, bl;
            split_limbs(xcur[j * kWarpTile + g * kGS + 4 * lane + e], dup_lo(cx.chi2), dup_lo(cx.clo2), bh, bl);
            atomicAdd(&wa[1 + j], bh);
            atomicAdd(&wa[1 + D + j], bl);
            atomicSub(&wo[1 + j], bh);
            atomicSub(&wo[1 + D + j], bl);
          }
        }
      }
    }
    if (!first) return;
  } else
  // labels (flagged points are overwritten by the re-check)
  if (a.store_labels) {
#pragma unroll
    for (int g = 0; g < kNG; ++g) {
      const int64_t i0 = base + g * kGS + 4 * lane;
      if (a.labels8) {
        if constexpr (FULL) {
          const uint32_t w = __byte_perm(__byte_perm(lab[4 * g], lab[4 * g + 1], 0x0040),
                                         __byte_perm(lab[4 * g + 2], lab[4 * g + 3], 0x0040), 0x5410);
          *reinterpret_cast<uint32_t*>(a.labels8 + i0) = w;
        } else {
#pragma unroll
          for (int qq = 0; qq < 4; ++qq) if (i0 + qq < a.n) a.labels8[i0 + qq] = (uint8_t)lab[4 * g + qq];
        }
      } else if (FULL && !a.labels_unaligned) {
        *reinterpret_cast<int4*>(a.labels + i0) = make_int4(lab[4 * g], lab[4 * g + 1], lab[4 * g + 2], lab[4 * g + 3]);
      } else if constexpr (FULL) {
#pragma unroll
        for (int qq = 0; qq < 4; ++qq) a.labels[i0 + qq] = lab[4 * g + qq];
      } else {
#pragma unroll
        for (int qq = 0; qq < 4; ++qq) if (i0 + qq < a.n) a.labels[i0 + qq] = lab[4 * g + qq];
      }
    }
  }
  // Exact sums: limb splits on FADD2 pairs, then 32-bit shared atomics into
  // this half-warp's window; flagged and padding points go to the discard bin k.
#pragma unroll
  for (int g = 0; g < kNG; ++g)
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int p0 = 4 * g + 2 * h;
      uint32_t bh[D][2], bl[D][2];
#pragma unroll
      for (int j = 0; j < D; ++j) {
        const unsigned long long xv =
            *reinterpret_cast<const unsigned long long*>(xcur + j * kWarpTile + g * kGS + 4 * lane + 2 * h);
        const unsigned long long t = fadd2(xv, cx.chi2);
        const unsigned long long hh = fsub2(t, cx.chi2);
        const unsigned long long r = fsub2(xv, hh);
        const unsigned long long t2 = fadd2(r, cx.clo2);
        asm("mov.b64 {%0, %1}, %2;" : "=r"(bh[j][0]), "=r"(bh[j][1]) : "l"(t));
        asm("mov.b64 {%0, %1}, %2;" : "=r"(bl[j][0]), "=r"(bl[j][1]) : "l"(t2));
      }
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const int bn = ((dbits >> (p0 + e)) & 1u) ? cx.k : lab[p0 + e];
        uint32_t* wb = wmine + bn * WIN;
        atomicAdd(&wb[0], 1u);
#pragma unroll
        for (int j = 0; j < D; ++j) {
          atomicAdd(&wb[1 + j], bh[j][e]);
          atomicAdd(&wb[1 + D + j], bl[j][e]);
        }
      }
    }
}

// The screen, recompute and flag test of process_tile for one point per lane
// (coordinates xo), two centroids per FFMA2, the table read by groups from
// gtab (every lane reads the same address).  The same chains, so the same values
// and bounds.  Returns the label, or -1 when the point must be re-checked;
// *slack as in the whole-run kernel.
template <int D, int KG>
__device__ __forceinline__ int screen_point(const float4* gtab, const FastCtx& cx, const float* s, const float (&xo)[D],
                                            const RunTile& rt, float& slack) {
  constexpr int GS = FastSmem<D>::GS;
  constexpr int LB = KG == 8 ? 5 : KG == 64 ? 8 : 0;
  unsigned long long X[D];
  float xt[D], A = 0.f;
#pragma unroll
  for (int j = 0; j < D; ++j) {
    xt[j] = __fsub_rn(xo[j], s[j]);
    X[j] = dup2(xt[j]);
    A = __fmaf_rn(xt[j], xt[j], A);
  }
  auto group = [&](const float4* g4, float (&r)[4]) {
    const ulonglong2* gt = reinterpret_cast<const ulonglong2*>(g4);
    const ulonglong2 nv = gt[D];
    unsigned long long rA = nv.x, rB = nv.y;
#pragma unroll
    for (int j = 0; j < D; ++j) {
      const ulonglong2 cv = gt[j];
      rA = ffma2(X[j], cv.x, rA);
      rB = ffma2(X[j], cv.y, rB);
    }
    unpack2(rA, r[0], r[1]);
    unpack2(rB, r[2], r[3]);
  };
  auto gmin = [&](int g) {
    float r[4];
    group(gtab + (size_t)g * GS, r);
    return pack_idx<LB>(fminf(fmin3(r[0], r[1], r[2]), r[3]), cx, (uint32_t)(4 * g));
  };
  float m1, m2;
  {
    const float ga = gmin(0), gb = gmin(1);
    m1 = fminf(ga, gb);
    m2 = fmaxf(ga, gb);
  }
  const int ng = cx.kpad >> 2;
#pragma unroll 2
  for (int g = 2; g < ng; g += 2) {
    const float ga = gmin(g), gb = gmin(g + 1);
    const float lo = fminf(ga, gb), hi = fmaxf(ga, gb);
    m2 = fmin3(m2, hi, fmaxf(m1, lo));
    m1 = fminf(m1, lo);
  }
  const uint32_t gsel = __float_as_uint(m1) & cx.kmask;
  float r[4];
  group(gtab + (size_t)(gsel >> 2) * GS, r);
  const float w0 = pack_idx<LB>(r[0], cx, 0u), w1 = pack_idx<LB>(r[1], cx, 1u);
  const float w2 = pack_idx<LB>(r[2], cx, 2u), w3 = pack_idx<LB>(r[3], cx, 3u);
  const float lo01 = fminf(w0, w1), hi01 = fmaxf(w0, w1);
  const float lo23 = fminf(w2, w3), hi23 = fmaxf(w2, w3);
  const float best = fminf(lo01, lo23);
  const float sec = fmin3(fmaxf(lo01, lo23), fminf(hi01, hi23), m2);
  const int lab = (int)(gsel | (__float_as_uint(best) & 3u));
  const float v1 = unpack_val<LB>(best, cx), v2 = unpack_val<LB>(sec, cx);
  const float T = fmaf(cx.tau, v2 - cx.M, fmaf(A, cx.cA, cx.c0));
  if (!(v2 - v1 > T) || lab >= cx.k) return -1;
  slack = screen_slack(v1, v2, T, A, cx.M, rt, lab);
  return lab;
}

// Points of an instance are packed without padding, so the staging copies
// are 4 bytes each (rows need not be 16-byte aligned); past N, zero-filled.
template <int D>
__device__ __forceinline__ void prefetch_tile_any(const FastArgs& a, float* xb, int64_t base, int lane) {
#pragma unroll
  for (int g = 0; g < kNG; ++g)
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int off = g * kGS + 4 * lane + e;
      const int64_t i = base + off;
      const int bytes = i < a.n ? 4 : 0;
#pragma unroll
      for (int j = 0; j < D; ++j) {
        const float* src = a.x + (int64_t)j * a.ld + (bytes ? i : 0);
        const uint32_t dst = (uint32_t)__cvta_generic_to_shared(xb + j * kWarpTile + off);
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(src), "r"(bytes));
      }
    }
  asm volatile("cp.async.commit_group;" ::: "memory");
}

// A point's new label and slack; a changed label goes straight into the int64
// totals (few points change).
template <int D>
__device__ __forceinline__ void run_commit(const RunTile& rt, long long* acc, const DataConst& dc, int64_t i,
                                           const float (&xo)[D], int kk, int old, float sl) {
  constexpr int DP = D + 1;
  rt.slack[i] = sl;
  if (rt.first || kk != old) {
    rt.z[i] = (uint8_t)kk;
    unsigned long long* ta = reinterpret_cast<unsigned long long*>(acc + kk * DP);
    unsigned long long* to = reinterpret_cast<unsigned long long*>(acc + old * DP);
    atomicAdd(ta + D, 1ull);
    if (!rt.first) atomicAdd(to + D, ~0ull);
#pragma unroll
    for (int j = 0; j < D; ++j) {
      uint32_t bh, bl;
      split_limbs(xo[j], dc.C_hi, dc.C_lo, bh, bl);
      const long long v = ((long long)(int)(bh - dc.bits_C_hi) << 22) + (long long)(int)(bl - dc.bits_C_lo);
      atomicAdd(ta + j, (unsigned long long)v);
      if (!rt.first) atomicAdd(to + j, (unsigned long long)(-v));
    }
  }
}

// Re-check of nr queued points, one per lane.  Not inlined: few points come
// here, and the kernels' instructions should stay in the SM's cache.
template <int D>
__device__ __noinline__ int run_recheck(const float* x, int64_t ld, const float4* ctil, const double* mu, int k,
                                        const uint32_t* q, int nr, int64_t wid, int wtot, long long* acc, DataConst dc,
                                        float B_max, float tau, RunTile rt) {
  int n64 = 0;
  for (int e = threadIdx.x & 31; e < nr; e += 32) {
    const uint32_t loc = q[e];
    const int64_t i = (wid + (int64_t)((loc & ~kRecheck) >> 8) * wtot) * kWarpTile + (loc & 255u);
    float xo[D];
#pragma unroll
    for (int j = 0; j < D; ++j) xo[j] = x[(int64_t)j * ld + i];
    const int old = rt.z[i];
    bool used64;
    float sl;
    const int kk = recheck_fast<D>(xo, dc.s, ctil, mu, k, B_max, tau, used64, &sl);
    n64 += used64 ? 1 : 0;
    sl = used64 ? -1.f : __fadd_rd(sl - rt.margin, rt.cum[kk]);
    run_commit<D>(rt, acc, dc, i, xo, kk, old, sl);
  }
  return n64;
}

// Decide the queued points one per lane: by the screen, and the ones it flags
// (with kRecheck set, or all in the first step: flagged before) by the
// re-check.  The open points of a tile lie near cluster borders, where the
// screen flags some of nearly every 32, and the re-check takes three times the
// screen's instructions: so flagged points are gathered at the front of the
// queue and re-checked side by side afterwards.
template <int D, int KG>
__device__ __forceinline__ void run_drain(const FastArgs& a, const float4* gtab, const FastCtx& cx, const float4* ctil,
                                          const double* mu, uint32_t* q, int qn, int wid, int wtot, long long* acc,
                                          int lane, const float* s, const DataConst& dc, float B_max,
                                          const RunTile& rt, int& n64) {
  __syncwarp();
  int nr = 0;
  for (int b = 0; b < qn; b += 32) {
    const bool live = b + lane < qn;
    const uint32_t loc = live ? q[b + lane] : 0u;
    bool rec = live && (loc & kRecheck);
    if (live && !rec) {
      const int64_t i = ((int64_t)wid + (int64_t)(loc >> 8) * wtot) * kWarpTile + (loc & 255u);
      float xo[D];
#pragma unroll
      for (int j = 0; j < D; ++j) xo[j] = a.x[(int64_t)j * a.ld + i];
      const int old = rt.z[i];
      float sl;
      const int kk = screen_point<D, KG>(gtab, cx, s, xo, rt, sl);
      if (kk < 0) rec = true;
      else run_commit<D>(rt, acc, dc, i, xo, kk, old, sl);
    }
    const unsigned bal = __ballot_sync(0xffffffffu, rec);  // every lane holds its entry: the front may be written
    if (rec) q[nr + __popc(bal & ((1u << lane) - 1u))] = loc;
    nr += __popc(bal);
  }
  __syncwarp();
  if (nr > 0) n64 += run_recheck<D>(a.x, a.ld, ctil, mu, a.k, q, nr, wid, wtot, acc, dc, B_max, cx.tau, rt);
  __syncwarp();
}

// Open points of a 256-point tile: above kHeavy it is screened whole; above
// kStage its points are copied to shared memory (3 KB in whole lines, where
// gathering 12 bytes a point takes three 64-byte accesses) and the open ones
// decided from there; below, they are queued across tiles and gathered.
// Measured: 72, 96, 128, 160 for kHeavy give 11.5, 10.6, 10.0, 9.9 ms for a run of
// 1e8 points (K = 32, 37 steps) and 63, 61, 61, 61 ms for 256 instances.
constexpr int kHeavy = 160, kStage = 32;
constexpr int kQueueFull = kWarpQueue - kHeavy;  // entries from which the queue is emptied (a tile adds at most kHeavy)
static_assert(kQueueFull + 4 * kStage <= kWarpQueue, "a batch of tiles with few open points fits");

// One warp's part of a step that skips points (see km_run_fast.cu): warp-tiles
// wid, wid + wtot, ... below end of the points a.x (a.n of them).  Adds the
// changes to acc (int64, k x (D + 1)); nflag and n64 count the points decided
// again and those decided in FP64.  ANY: rows without 16-byte alignment.
// Tiles are tested four at a time, their slacks and labels (5 KB a warp)
// loaded together: 1e8 points that keep their labels took 150 us a step with
// one tile loaded ahead, 97 us with four.
template <int D, int KG, bool ANY>
__device__ __forceinline__ void run_pass(const FastArgs& a, FastSmem<D>& sm, const FastCtx& cx,
                                         const unsigned long long* s2, const float* s, const DataConst& dc,
                                         const RunTile& rt, const float4* ctil, const double* mu, float B_max,
                                         long long* acc, uint32_t* q, uint32_t* wwarp, uint32_t* wmine, float* xb,
                                         int nbuf, int wid, int wtot, int end, int lane, int& nflag, int& n64) {
  const int nwin = a.nwin;
  int qn = 0, since_flush = 0, m = 0, tile = wid;
  auto fetch = [&](float* dst, int t) {
    if constexpr (ANY) prefetch_tile_any<D>(a, dst, (int64_t)t * kWarpTile, lane);
    else prefetch_tile<D>(a, dst, (int64_t)t * kWarpTile, lane);
  };
  auto whole = [&](int t, int mt, const float* xcur) {
    const int64_t base = (int64_t)t * kWarpTile;
    if (base + kWarpTile <= a.n)
      process_tile<D, KG, false, true, true>(a, sm, cx, s2, xcur, base, mt, lane, wmine, q, qn, &rt);
    else
      process_tile<D, KG, false, false, true>(a, sm, cx, s2, xcur, base, mt, lane, wmine, q, qn, &rt);
    // at most 512 additions and 512 subtractions per bin between flushes
    if (++since_flush == (nwin == 4 ? 8 : nwin == 2 ? 4 : 2)) {
      flush_windows<D>(wwarp, acc, a.k, nwin, lane, dc.bits_C_hi, dc.bits_C_lo);
      since_flush = 0;
    }
  };
  if (rt.first) {
    // every point; the queue holds the flagged ones
    auto recheck = [&]() {
      __syncwarp();
      n64 += run_recheck<D>(a.x, a.ld, ctil, mu, a.k, q, qn, wid, wtot, acc, dc, B_max, cx.tau, rt);
      __syncwarp();
      nflag += qn;
      qn = 0;
    };
    if (tile < end) fetch(xb, tile);
    for (; tile < end; tile += wtot, ++m) {
      asm volatile("cp.async.wait_group 0;" ::: "memory");
      // each lane reads only the chunks it copied itself
      if (nbuf == 2 && tile + wtot < end) fetch(xb + ((m + 1) & 1) * D * kWarpTile, tile + wtot);
      whole(tile, m, xb + (nbuf == 2 ? (m & 1) : 0) * D * kWarpTile);
      if (nbuf == 1 && tile + wtot < end) fetch(xb, tile + wtot);
      if (qn > kWarpQueue - kWarpTile || (qn > 0 && tile + wtot >= end)) recheck();
    }
  } else {
    // batches of four tiles; u: the next of the current batch's tiles with
    // more than kStage open points (4: none left)
    uint32_t open = 0u;       // this lane's open points of such tiles: 8 bits per tile
    uint32_t n01 = 0u, n23 = 0u;  // open points of the batch's tiles, 16 bits each
    int u = 4, tb = 0, mb = 0;
    while (true) {
      if (u == 4 && tile < end) {
        open = 0u;
        {
          float4 sv[4][2];
          uint32_t zv[4][2];
#pragma unroll
          for (int v = 0; v < 4; ++v) {
            const int t = tile + v * wtot;
            const int64_t base = (int64_t)t * kWarpTile;
#pragma unroll
            for (int g = 0; g < 2; ++g) {
              const int64_t i0 = base + g * kGS + 4 * lane;
              sv[v][g] = make_float4(3.0e38f, 3.0e38f, 3.0e38f, 3.0e38f);  // past the end: never open
              zv[v][g] = 0u;
              if (t < end) {
                if (base + kWarpTile <= a.n) {
                  sv[v][g] = *reinterpret_cast<const float4*>(rt.slack + i0);
                  zv[v][g] = *reinterpret_cast<const uint32_t*>(rt.z + i0);
                } else {
                  float* sp = reinterpret_cast<float*>(&sv[v][g]);
#pragma unroll
                  for (int e = 0; e < 4; ++e)
                    if (i0 + e < a.n) {
                      sp[e] = rt.slack[i0 + e];
                      zv[v][g] |= (uint32_t)rt.z[i0 + e] << (8 * e);
                    }
                }
              }
            }
          }
#pragma unroll
          for (int v = 0; v < 4; ++v)
#pragma unroll
            for (int g = 0; g < 2; ++g) {
              const float sp[4] = {sv[v][g].x, sv[v][g].y, sv[v][g].z, sv[v][g].w};
#pragma unroll
              for (int e = 0; e < 4; ++e)
                open |= (sp[e] > rt.cum[(zv[v][g] >> (8 * e)) & 255u] ? 0u : 1u) << (8 * v + 4 * g + e);
            }
        }
        tb = tile;
        mb = m;
        tile += 4 * wtot;
        m += 4;
        if (__any_sync(0xffffffffu, open != 0u)) {
          n01 = __reduce_add_sync(0xffffffffu, (unsigned)__popc(open & 0xffu) | (unsigned)__popc(open & 0xff00u) << 16);
          n23 = __reduce_add_sync(0xffffffffu,
                                  (unsigned)__popc(open & 0xff0000u) | (unsigned)__popc(open & 0xff000000u) << 16);
          // the tiles with few open points, all four at once, into the queue
          uint32_t few = 0u, nfew = 0u;
#pragma unroll
          for (int v = 0; v < 4; ++v) {
            const uint32_t nv = ((v < 2 ? n01 : n23) >> (16 * (v & 1))) & 0xffffu;
            if (nv <= kStage) { few |= 0xffu << (8 * v); nfew += nv; }
            else u = min(u, v);
          }
          few &= open;
          open &= ~few;
          if (nfew) {  // at most 4 kStage: the queue has room (kQueueFull)
            const int nf = __popc(few);
            int incl = nf;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
              const int t = __shfl_up_sync(0xffffffffu, incl, o);
              if (lane >= o) incl += t;
            }
            int at = qn + incl - nf;
            for (; few; few &= few - 1u) {
              const int p = __ffs((int)few) - 1;
              q[at++] = (uint32_t)((mb + (p >> 3)) << 8) | (uint32_t)(((p >> 2) & 1) * kGS + 4 * lane + (p & 3));
            }
            qn += (int)nfew;
          }
        }
      }
      for (; u < 4; ++u) {
        const int total = (int)(((u < 2 ? n01 : n23) >> (16 * (u & 1))) & 0xffffu);
        if (total <= kStage) continue;
        const int t = tb + u * wtot;
        if (total > kHeavy) {
          if (qn > kWarpQueue - kWarpTile) break;  // empty the queue first
          fetch(xb, t);
          asm volatile("cp.async.wait_group 0;" ::: "memory");
          nflag += total + qn;
          whole(t, mb + u, xb);
          nflag -= qn;  // what it queued is counted when the queue is emptied
        } else {
          if (qn > kQueueFull) break;
          fetch(xb, t);
          uint32_t fb = (open >> (8 * u)) & 255u;
          const int nf = __popc(fb);
          int incl = nf;
#pragma unroll
          for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += v;
          }
          int at = qn + incl - nf;
          for (; fb; fb &= fb - 1u) {
            const int p = __ffs((int)fb) - 1;
            q[at++] = (uint32_t)((mb + u) << 8) | (uint32_t)((p >> 2) * kGS + 4 * lane + (p & 3));
          }
          asm volatile("cp.async.wait_group 0;" ::: "memory");
          __syncwarp();  // every lane's copies and queue entries
          int nr = qn;
          for (int b = qn; b < qn + total; b += 32) {
            const bool live = b + lane < qn + total;
            const uint32_t loc = live ? q[b + lane] : 0u;
            bool rec = false;
            if (live) {
              const int off = (int)(loc & 255u);
              const int64_t i = (int64_t)t * kWarpTile + off;
              float xo[D];
#pragma unroll
              for (int j = 0; j < D; ++j) xo[j] = xb[j * kWarpTile + off];
              const int old = rt.z[i];
              float sl;
              const int kk = screen_point<D, KG>(sm.gtab, cx, s, xo, rt, sl);
              if (kk < 0) rec = true;
              else run_commit<D>(rt, acc, dc, i, xo, kk, old, sl);
            }
            const unsigned bal = __ballot_sync(0xffffffffu, rec);
            if (rec) q[nr + __popc(bal & ((1u << lane) - 1u))] = loc | kRecheck;
            nr += __popc(bal);
          }
          nflag += total - (nr - qn);
          qn = nr;
          __syncwarp();  // the points are read no more
        }
      }
      const bool last = u == 4 && tile >= end;
      if (qn > 0 && (u < 4 || qn > kQueueFull || last)) {
        run_drain<D, KG>(a, sm.gtab, cx, ctil, mu, q, qn, wid, wtot, acc, lane, s, dc, B_max, rt, n64);
        nflag += qn;
        qn = 0;
      }
      if (last) break;
    }
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  if (since_flush) flush_windows<D>(wwarp, acc, a.k, nwin, lane, dc.bits_C_hi, dc.bits_C_lo);
}

}  // namespace
}  // namespace km
