// Screen tables of the fused assignment kernel from the current centroids,
// shared by the single-context update and the batched update (one block;
// every thread of the block calls it).
//
// For centroids mu (k x d, FP64), the data shift s and A_max >= max_i
// fl32 ||fl(x_i - s)||^2: c~_k = fl32(mu_k - s) (ctil4), B_k = ||c~_k||^2 in
// FP64, and the screen r_k = M + 2^sigma (||c~_k||^2 - 2 x~.c~_k) in one
// binade [2^eM, 2^(eM+1)) chosen so that an index of L = ceil(log2 kpad) bits
// packed below the value keeps positive floats in value order; the flag
// constants bound every rounding of the chain, of x~ and c~, and the
// oracle's own FP64 rounding (see the fused kernel).  tab2 holds, per
// centroid, d packed pairs (a_kj, a_kj) with a_kj = -2^(sigma+1) c~_kj and the
// pair (n_k, n_k), n_k = fl32(M + 2^sigma B_k); padding centroids k..kpad-1
// get zero coefficients and the largest value of the binade.
#pragma once
#include "km_internal.cuh"

namespace km {

// The FP64 pipe is slow and its chains long (this function, mostly one
// thread's FP64 constants, took 3.9 us of a small set's step), so beyond the
// difference mu - s the values are formed in FP32: B_k as an unevaluated sum
// of two floats (error below 2^-44 of B_k, where n_k keeps 2^-24), the flag
// constants with directed roundings or factors that cover theirs.  Every thread
// forms the constants for itself after one barrier.  gtab (may be null): the
// table by groups of 4 centroids as the fused kernel's epilogue reads it, GS
// float4 per group, slot j = coefficient j of the 4 centroids.
static __device__ void fast_screen_tables(const double* mu, const float* shift, float A_max, int k, int d, int kpad,
                                          double tie_rel, float4* ctil4, IterConst* ic_out,
                                          unsigned long long* tab2, double* sB_raw, float4* gtab = nullptr,
                                          int GS = 0) {
  const int tid = threadIdx.x + threadIdx.y * blockDim.x;
  const int nth = blockDim.x * blockDim.y, lane = tid & 31;
  float2* sB = reinterpret_cast<float2*>(sB_raw);  // [k] B_k = x + y
  for (int c = tid; c < k; c += nth) {
    float cv[4] = {0.f, 0.f, 0.f, 0.f};
    float bh = 0.f, bl = 0.f;
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (j < d) {
        cv[j] = __double2float_rn(__dsub_rn(mu[(size_t)c * d + j], (double)shift[j]));
        // exact product p + e, exact sum t + f
        const float p = __fmul_rn(cv[j], cv[j]), e = __fmaf_rn(cv[j], cv[j], -p);
        const float t = __fadd_rn(bh, p), q = __fsub_rn(t, bh);
        const float f = __fadd_rn(__fsub_rn(bh, __fsub_rn(t, q)), __fsub_rn(p, q));
        bh = t;
        bl = __fadd_rn(bl, __fadd_rn(e, f));
      }
    ctil4[c] = make_float4(cv[0], cv[1], cv[2], cv[3]);
    sB[c] = make_float2(bh, bl);
  }
  __syncthreads();
  // max B_k, rounded up (an overflow leaves +infinity: then every point is flagged)
  float bmax = 0.f;
  for (int c = lane; c < k; c += 32) bmax = fmaxf(bmax, sB[c].x);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) bmax = fmaxf(bmax, __shfl_xor_sync(0xffffffffu, bmax, o));
  bmax = __fmul_ru(bmax, 1.f + 0x1p-21f);
  int L = 1;
  while ((1 << L) < kpad) ++L;
  int E, half;   // biased exponent of the binade; 2^half: the largest |2^sigma W| allowed
  uint32_t frac;  // significand bits of M: 1.5, 1.25 or 1.375
  if (L <= 6) {
    const int base = 1 << (7 - L), step = 1 << (9 - L);
    E = base + ((127 - base) / step) * step;
    frac = 0x400000u;
    half = E - 128;
  } else if (L == 7) {
    E = 125; frac = 0x200000u; half = E - 129;
  } else {
    E = 126; frac = 0x300000u; half = E - 130;
  }
  const int eM = E - 127;
  const float M = __uint_as_float(((uint32_t)E << 23) | frac);
  // the largest sigma with 2^sigma P < 2^half, P in [2^e, 2^(e + 1))
  const float P = __fmul_ru(__fadd_ru(__fmul_ru(A_max, 1.f + 0x1p-20f), 2.f * bmax), 1.f + 0x1p-10f);
  const int e = (int)(__float_as_uint(P) >> 23) - 127;
  // squares so large that the scale leaves FP32's range (|x| from about 1e10 at
  // K = 8, 1e16 at K = 32 and 1e17 at K = 64): the values below leave the
  // binade, so every point is flagged
  const bool out = half - e - 1 < -120;
  const int sigma = max(-120, min(120, half - e - 1));
  auto pow2 = [](int x) {  // 2^x, +infinity or 0 outside the normal range
    return x > 127 ? __uint_as_float(0x7f800000u) : x < -126 ? 0.f : __uint_as_float((uint32_t)(x + 127) << 23);
  };
  if (tid == 0) {
    const float G = pow2(sigma - eM + 23), u = 0x1p-24f, u64x = 4.1f * 0x1p-53f, tau = __double2float_ru(tie_rel * (1.0 + 1e-4));
    IterConst ic;
    ic.M = M;
    ic.L = L;
    ic.mul = 1u << L;
    ic.bitsM_low = __float_as_uint(M) & ((1u << (32 - L)) - 1u);
    ic.G = G;
    ic.thr_c0 = out ? __uint_as_float(0x7f800000u) : ((float)(d + 3) + (8.002f * u + u64x * (float)(d + 1)) * bmax * G) * (1.f + 1.01e-4f);
    ic.thr_cA = (4.001f * u + u64x * (float)(d + 1)) * G * (1.f + 1.12e-4f);
    ic.tau = tau;
    ic.B_max = bmax;
    ic.pad[0] = ic.pad[1] = ic.pad[2] = 0.f;
    *ic_out = ic;
  }
  const float scale = -pow2(sigma + 1), s1 = pow2(sigma);
  const uint32_t dummy = ((uint32_t)E << 23) | (L <= 6 ? 0x7fffffu : 0x3fffffu);
  const int dp = d + 1;
  for (int c = tid; c < kpad; c += nth) {
    unsigned long long* row = tab2 + (size_t)c * dp;
    float4 cv4 = make_float4(0.f, 0.f, 0.f, 0.f);
    uint32_t nb = dummy;
    if (c < k) {
      cv4 = ctil4[c];
      const float2 B = sB[c];
      // n = fl(M + 2^sigma B): exact sum of M and 2^sigma B's high part, then the rest
      const float t = __fmul_rn(B.x, s1), h = __fadd_rn(M, t), q = __fsub_rn(h, M);
      const float f = __fadd_rn(__fsub_rn(M, __fsub_rn(h, q)), __fsub_rn(t, q));
      nb = __float_as_uint(__fadd_rn(h, __fmaf_rn(B.y, s1, f)));
    }
    const float cv[4] = {cv4.x, cv4.y, cv4.z, cv4.w};
    float* g = gtab ? reinterpret_cast<float*>(gtab + (size_t)(c >> 2) * GS) + (c & 3) : nullptr;
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (j < d) {
        const uint32_t b = c < k ? __float_as_uint(__fmul_rn(cv[j], scale)) : 0u;
        row[j] = ((unsigned long long)b << 32) | b;
        if (g) g[4 * j] = __uint_as_float(b);
      }
    row[d] = ((unsigned long long)nb << 32) | nb;
    if (g) g[4 * d] = __uint_as_float(nb);
  }
}

}  // namespace km
