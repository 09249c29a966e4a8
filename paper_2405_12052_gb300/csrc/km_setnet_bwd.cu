// Backward pass of the set network's per-point layers and their weight
// gradients on the 5th-gen tensor cores (tcgen05, BF16 operands, FP32
// accumulation in TMEM).
//
// dz2 = dg/S * [h2 > 0] is a set's vector times a 0/1 matrix M (the forward
// pass keeps its bits), so both products of the backward pass have an operand
// that BF16 holds exactly:
//   dh1^T[c][p] = sum_u V[c][u] M[p][u],  V[c][u] = dg_u/S W2[u][c]
//   T[u][c]     = sum_p M[p][u] h1[p][c],  dW2[u][c] = sum over sets dg_u/S T[u][c]
// and the other one, FP32, is split into three BF16 values whose sum is the FP32
// value (8 + 8 + 8 significand bits, to 2^-25 of it), so every product is exact
// and only the FP32 accumulation rounds.  T is read out and added in FP32
// registers after every 128 points: 24 accumulations of 16 products in a row
// (longer runs would add the tensor core's rounding up in one direction).
//
// Per 128-point tile of one set, 512 threads: M by point and by unit, and h1
// formed again from the standardised points, written to shared memory as
// 128-byte-swizzled K-major rows; one thread issues the MMAs (M = N = 128, K =
// 16) and commits them to mbarriers; meanwhile the second half of h1 is
// written, and dh1 is taken from TMEM with unit c in lane c, so a thread adds
// dW1[c], db1[c] over its 32 points in registers.  Each block takes a run of
// tiles and writes one partial gradient.
//
// The FP32 kernel it replaces was bound by 34.4e9 multiply-adds for 1M points
// (0.92 ms at one per lane and cycle; 1.65 ms).  Here the tensor work is 0.05 ms
// at the BF16 rate and the instructions that form and split the operands
// bound it: 0.29 ms.
#include <cuda_bf16.h>

#include <algorithm>

#include "km_setnet.cuh"
#include "km_tcgen05.cuh"

namespace km {

namespace {

constexpr int kBT = 128;                    // points per tile = units: M, N of every MMA
constexpr int kBlk = 128 * 128;             // bytes of a 128-row x 64-column operand block
constexpr int kBwThreads = 512;
// shared memory from the 1024-aligned base
constexpr int kOffV = 0;                    // [3 splits][2 K-blocks] V
constexpr int kOffM = kOffV + 6 * kBlk;     // [2 K-blocks] M by point
constexpr int kOffMt = kOffM + 2 * kBlk;    // M by unit, 64 points
constexpr int kOffH = kOffMt + kBlk;        // [3 splits] h1 by unit, 64 points
constexpr int kOffX = kOffH + 3 * kBlk;     // [128][4] points
constexpr int kOffBits = kOffX + kBT * 16;  // [128][4] bits of h2 > 0
constexpr int kOffDg = kOffBits + kBT * 16; // [128] dg / S
constexpr int kOffBar = kOffDg + 512;       // 4 mbarriers, TMEM address
constexpr int kBwSmem = kOffBar + 64 + 1024;

// D (128 x 128, f32) += A (128 x 16) B (128 x 16)^T, both BF16 and K-major
constexpr uint32_t kIdesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(kBT >> 3) << 17) | ((uint32_t)(kBT >> 4) << 24);

__device__ __forceinline__ void mma_bf16(uint32_t tmem, uint64_t ad, uint64_t bd, uint32_t acc) {
  asm volatile("{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\ntcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}"
               ::"r"(tmem), "l"(ad), "l"(bd), "r"(kIdesc), "r"(acc));
}
// 16-byte chunk ch (8 K-columns) of row r of a 64-column operand block
__device__ __forceinline__ uint32_t chunk_at(int r, int ch) { return (uint32_t)(r * 128 + ((ch ^ (r & 7)) << 4)); }

// Eight 0/1 values from the bits of b, as BF16.
__device__ __forceinline__ uint4 ones8(uint32_t b) {
  uint32_t w[4];
#pragma unroll
  for (int e = 0; e < 4; ++e) w[e] = ((b >> (2 * e)) & 1u) * 0x3F80u + ((b >> (2 * e + 1)) & 1u) * 0x3F800000u;
  return make_uint4(w[0], w[1], w[2], w[3]);
}
// v = s[0] + s[1] + s[2], each BF16 (rounded to nearest of what the ones
// before leave; the remainders are exact).
__device__ __forceinline__ void split8(const float (&v)[8], uint4 (&s)[3]) {
  uint32_t w[3][4];
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    float lo = v[2 * e], hi = v[2 * e + 1];
#pragma unroll
    for (int t = 0; t < 3; ++t) {
      const __nv_bfloat162 q = __floats2bfloat162_rn(lo, hi);
      const uint32_t b = *reinterpret_cast<const uint32_t*>(&q);
      w[t][e] = b;
      lo -= __uint_as_float(b << 16);
      hi -= __uint_as_float(b & 0xffff0000u);
    }
  }
#pragma unroll
  for (int t = 0; t < 3; ++t) s[t] = make_uint4(w[t][0], w[t][1], w[t][2], w[t][3]);
}

__global__ void __launch_bounds__(kBwThreads, 1) sn_bwd_points(const float* __restrict__ prm, int d, int k, int S,
                                                               int tiles_per_set, int64_t tiles,
                                                               const float* __restrict__ dG,
                                                               const float* __restrict__ xs,
                                                               const uint32_t* __restrict__ bits,
                                                               float* __restrict__ part, int* err) {
  extern __shared__ unsigned char raw[];
  unsigned char* sm = raw + ((1024u - ((uint32_t)__cvta_generic_to_shared(raw) & 1023u)) & 1023u);
  const uint32_t sb = (uint32_t)__cvta_generic_to_shared(sm);
  float4* s_x = reinterpret_cast<float4*>(sm + kOffX);
  uint32_t* s_bits = reinterpret_cast<uint32_t*>(sm + kOffBits);
  float* s_dg = reinterpret_cast<float*>(sm + kOffDg);
  uint32_t* s_tmem = reinterpret_cast<uint32_t*>(sm + kOffBar + 32);
  const NetOff o = net_off(d, k);
  const int tid = threadIdx.x, warp = tid >> 5, g = tid >> 7, i = tid & 127;  // unit i, group g of four
  auto bar = [&](int q) { return sb + kOffBar + 8 * q; };  // 0 T of half 0, 1 dh1, 2 T of half 1, 3 teardown
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     (uint32_t)__cvta_generic_to_shared(s_tmem)), "r"(256));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  if (tid == 0)
    for (int q = 0; q < 4; ++q) bar_init(bar(q), 1);
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *s_tmem;                       // dh1^T in columns 0..127, T in 128..255
  const uint32_t trow = tmem + ((uint32_t)(warp & 3) << 21);  // this warp's 32 lanes
  float4 w1;  // W1[i][0..2] (0 past d), b1[i]
  {
    float w[3];
    for (int j = 0; j < 3; ++j) w[j] = j < d ? prm[o.W1 + i * d + j] : 0.f;
    w1 = make_float4(w[0], w[1], w[2], prm[o.b1 + i]);
  }
  float acc2[32];  // dW2[i][32 g + q]
#pragma unroll
  for (int q = 0; q < 32; ++q) acc2[q] = 0.f;
  float gx = 0.f, gy = 0.f, gz = 0.f, gb = 0.f, gb2 = 0.f;  // dW1[i], db1[i] (points 32 g ..), db2[i] (this thread's chunks)
  const int64_t t0 = tiles * blockIdx.x / gridDim.x, t1 = tiles * (blockIdx.x + 1) / gridDim.x;
  // the next tile's points and bits, one word each per thread, on their way
  // while this tile is worked on (past a set's points: no bits)
  float nx = 0.f;
  uint32_t nb = 0u;
  auto prefetch = [&](int64_t t) {
    const int64_t set = t / tiles_per_set;
    const int p0 = (int)(t - set * tiles_per_set) * kBT, p = p0 + (tid >> 2), j = tid & 3;
    const bool live = p < S;
    nx = live && j < d ? xs[(set * S + p) * d + j] : 0.f;
    nb = live ? bits[(set * S + p) * 4 + j] : 0u;
  };
  if (t0 < t1) prefetch(t0);
  int64_t cur = -1;
  bool bad = false;
  uint32_t ph = 0u;
  for (int64_t t = t0; t < t1; ++t, ph ^= 1u) {
    const int64_t set = t / tiles_per_set;
    reinterpret_cast<float*>(s_x)[tid] = nx;
    s_bits[tid] = nb;
    if (set != cur && tid < H) s_dg[tid] = dG[set * H + tid] / (float)S;
    if (t + 1 < t1) prefetch(t + 1);
    __syncthreads();
    if (set != cur) {
      cur = set;
#pragma unroll 1
      for (int q = 0; q < 4; ++q) {
        const int c16 = 4 * g + q;  // chunk of 8 units u
        float v[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) v[e] = s_dg[8 * c16 + e] * prm[o.W2 + (8 * c16 + e) * H + i];
        uint4 sp[3];
        split8(v, sp);
#pragma unroll
        for (int r = 0; r < 3; ++r)
          *reinterpret_cast<uint4*>(sm + kOffV + (2 * r + (c16 >> 3)) * kBlk + chunk_at(i, c16 & 7)) = sp[r];
      }
    }
    const float dgi = s_dg[i];
    {
      // M by point: row i, units 32 g .. 32 g + 31
      const uint32_t b = s_bits[4 * i + g];
#pragma unroll
      for (int q = 0; q < 4; ++q)
        *reinterpret_cast<uint4*>(sm + kOffM + (g >> 1) * kBlk + chunk_at(i, 4 * (g & 1) + q)) = ones8(b >> (8 * q));
    }
    // M by unit and h1 by unit, 64 points: row i, chunks 2 g and 2 g + 1
    int cnt = 0;
    auto half = [&](int h) {
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const int ch = 2 * g + q, p0 = 64 * h + 8 * ch;
        uint32_t b = 0u;
        float v[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          b |= ((s_bits[4 * (p0 + e) + (i >> 5)] >> (i & 31)) & 1u) << e;
          const float4 x = s_x[p0 + e];
          v[e] = fmaxf(fmaf(w1.z, x.z, fmaf(w1.y, x.y, fmaf(w1.x, x.x, w1.w))), 0.f);
        }
        cnt += __popc(b);
        *reinterpret_cast<uint4*>(sm + kOffMt + chunk_at(i, ch)) = ones8(b);
        uint4 sp[3];
        split8(v, sp);
#pragma unroll
        for (int r = 0; r < 3; ++r) *reinterpret_cast<uint4*>(sm + kOffH + r * kBlk + chunk_at(i, ch)) = sp[r];
      }
    };
    auto mma_T = [&](int h) {
#pragma unroll
      for (int r = 2; r >= 0; --r)  // the small parts first
#pragma unroll
        for (int kk = 0; kk < 4; ++kk)
          mma_bf16(tmem + 128, sm_desc(sb + kOffMt + kk * 32), sm_desc(sb + kOffH + r * kBlk + kk * 32),
                   h > 0 || r < 2 || kk > 0 ? 1u : 0u);
    };
    half(0);
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // the rows -> the tensor core's view
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (tid == 0) {
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      mma_T(0);
      mma_commit(bar(0));
#pragma unroll
      for (int r = 2; r >= 0; --r)
#pragma unroll
        for (int kk = 0; kk < 8; ++kk)
          mma_bf16(tmem, sm_desc(sb + kOffV + (2 * r + (kk >> 2)) * kBlk + (kk & 3) * 32),
                   sm_desc(sb + kOffM + (kk >> 2) * kBlk + (kk & 3) * 32), r < 2 || kk > 0 ? 1u : 0u);
      mma_commit(bar(1));
    }
    __syncwarp();
    bad |= !wait_bar(bar(0), ph);  // the first half's rows may be overwritten
    half(1);
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    __syncthreads();
    if (tid == 0) {
      mma_T(1);
      mma_commit(bar(2));
    }
    __syncwarp();
    gb2 = fmaf(dgi, (float)cnt, gb2);
    bad |= !wait_bar(bar(1), ph);
    __syncwarp();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    {
      // dh1 of unit i and points 32 g .. 32 g + 31
      unsigned long long v[16];
      tmem_ld32(trow + 32 * g, v);
#pragma unroll
      for (int q = 0; q < 32; ++q) {
        const float4 x = s_x[32 * g + q];
        const float z = fmaf(w1.z, x.z, fmaf(w1.y, x.y, fmaf(w1.x, x.x, w1.w)));
        const float dh = __uint_as_float((uint32_t)(v[q >> 1] >> (32 * (q & 1))));
        const float dz = z > 0.f ? dh : 0.f;
        gx = fmaf(dz, x.x, gx);
        gy = fmaf(dz, x.y, gy);
        gz = fmaf(dz, x.z, gz);
        gb += dz;
      }
    }
    bad |= !wait_bar(bar(2), ph);
    __syncwarp();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    {
      unsigned long long v[16];
      tmem_ld32(trow + 128 + 32 * g, v);
#pragma unroll
      for (int q = 0; q < 32; ++q)
        acc2[q] = fmaf(dgi, __uint_as_float((uint32_t)(v[q >> 1] >> (32 * (q & 1)))), acc2[q]);
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");  // the accumulators may be rewritten
    if (__syncthreads_or(bad ? 1 : 0)) {
      if (tid == 0) { err[0] = 3; err[1] = 3; }  // a wait gave up: in this pass, and not yet reported
      break;
    }
  }
  // every MMA issued must complete before TMEM and shared memory are released
  if (tid == 0) {
    mma_commit(bar(3));
    wait_bar(bar(3), 0);
  }
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(256));
  float* out = part + (size_t)blockIdx.x * (H * H + H * d + 2 * H);
#pragma unroll
  for (int q = 0; q < 32; ++q) out[i * H + 32 * g + q] = acc2[q];
  // the four groups' sums of each unit, added in order
  float* s_g = reinterpret_cast<float*>(sm);  // [4][128][5]
  s_g[(g * H + i) * 5] = gx;
  s_g[(g * H + i) * 5 + 1] = gy;
  s_g[(g * H + i) * 5 + 2] = gz;
  s_g[(g * H + i) * 5 + 3] = gb;
  s_g[(g * H + i) * 5 + 4] = gb2;
  __syncthreads();
  for (int q = tid; q < 5 * H; q += kBwThreads) {
    float s = 0.f;
    for (int r = 0; r < 4; ++r) s += s_g[r * 5 * H + q];
    const int u = q / 5, j = q - 5 * u;
    if (j < 3) {
      if (j < d) out[H * H + u * d + j] = s;
    } else {
      out[H * H + H * d + (j - 3) * H + u] = s;
    }
  }
}

}  // namespace

int setnet_bwd_blocks(int B, int S) {
  return (int)std::min<int64_t>((int64_t)B * ((S + kBT - 1) / kBT), kSetBwdBlocks);
}

cudaError_t launch_setnet_bwd_points(const SetNetArgs& a, int blocks, cudaStream_t st) {
  cudaError_t e = cudaFuncSetAttribute(sn_bwd_points, cudaFuncAttributeMaxDynamicSharedMemorySize, kBwSmem);
  if (e != cudaSuccess) return e;
  const int tps = (a.S + kBT - 1) / kBT;
  sn_bwd_points<<<blocks, kBwThreads, kBwSmem, st>>>(a.prm, a.d, a.k, a.S, tps, (int64_t)a.B * tps, a.dG, a.xs, a.bits,
                                                    a.part, a.err);
  return cudaGetLastError();
}

}  // namespace km
