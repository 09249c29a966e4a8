// Learned initialiser: a set network that predicts K starting centres for
// Lloyd's algorithm from a sample of S points (the paper notes the result's
// dependence on the initial centres, section "The Lloyd's algorithm").
//
//   standardise  x' = (x - m) / s   (per set: per-coordinate mean and
//                population std of its S points; s = 1 where it is 0)
//   per point    h1 = relu(W1 x' + b1), h2 = relu(W2 h1 + b2)    (H = 128)
//   pool         g = mean_i h2_i
//   head         a3 = relu(W3 g + b3), p = W4 a3 + b4  (K x d, standardised)
//   loss         mean over sets of the symmetric Chamfer distance to the
//                standardised targets (ties: lowest index)
//
// FP32 throughout (the backward products on the tensor cores by exact three-way
// splits of their FP32 factor); every reduction runs in a fixed order (no float
// atomics), so a step is deterministic.  Kernels:
//   sn_standardize   one block per set
//   sn_fwd_points    64 or 256 points per block: h1 in shared memory, h2 by
//                    8x8 register tiles, the pooled sums of 64 points, and
//                    (training) one bit per h2 value, h2 > 0
//   sn_head          one block per set: pooling, head forward, loss and head
//                    backward to dg
//   sn_head_grad     dW3, dW4, db3, db4 and the loss, sets added in order
//   sn_bwd_points    (km_setnet_bwd.cu, tensor cores) dz2 = dg/S * [h2 > 0] from
//                    the bits, dz1 = (dz2 W2) * [h1 > 0], and each block's dW2
//                    = sum dz2 h1^T, dW1, db1, db2
//   sn_wgrad_reduce  adds the blocks' gradients in order
//   sn_adam          Adam with bias correction (Kingma and Ba 2015)
#include "km_setnet.cuh"

#include <algorithm>

namespace km {

namespace {

// Sum over the block's 256 threads of up to three values at once: the pairwise
// tree t += t + 128, 64, ..., 1 (the last five levels inside warp 0).
__device__ __forceinline__ void tree3(float (&v)[3], float (*s_red)[256], int d, int tid) {
  for (int j = 0; j < d; ++j) s_red[j][tid] = v[j];
  __syncthreads();
#pragma unroll
  for (int w = 128; w >= 32; w >>= 1) {
    if (tid < w)
      for (int j = 0; j < d; ++j) s_red[j][tid] += s_red[j][tid + w];
    __syncthreads();
  }
  if (tid < 32)
    for (int j = 0; j < d; ++j) {
      float t = s_red[j][tid];
#pragma unroll
      for (int w = 16; w > 0; w >>= 1) t += __shfl_down_sync(0xffffffffu, t, w);
      if (tid == 0) s_red[j][0] = t;
    }
  __syncthreads();
  for (int j = 0; j < d; ++j) v[j] = s_red[j][0];
  __syncthreads();
}

// One block per set; the d coordinates are summed together (one read of the
// set per pass instead of d; 26.7 -> 18.4 us for 256 sets of 4096 points).
__global__ void __launch_bounds__(256) sn_standardize(const float* __restrict__ x, const float* __restrict__ t,
                                                      int S, int d, int k, float* xs, float* ts, float* ms) {
  __shared__ float s_red[3][256];
  const int b = blockIdx.x, tid = threadIdx.x;
  const float* xb = x + (size_t)b * S * d;
  float m[3] = {0.f, 0.f, 0.f}, sd[3] = {0.f, 0.f, 0.f};
#pragma unroll 4
  for (int i = tid; i < S; i += 256)
#pragma unroll
    for (int j = 0; j < 3; ++j)
      if (j < d) m[j] += xb[(size_t)i * d + j];
  tree3(m, s_red, d, tid);
  for (int j = 0; j < d; ++j) m[j] = m[j] / (float)S;
#pragma unroll 4
  for (int i = tid; i < S; i += 256)
#pragma unroll
    for (int j = 0; j < 3; ++j)
      if (j < d) {
        const float u = xb[(size_t)i * d + j] - m[j];
        sd[j] = fmaf(u, u, sd[j]);
      }
  tree3(sd, s_red, d, tid);
  for (int j = 0; j < d; ++j) {
    const float q = sqrtf(sd[j] / (float)S);
    sd[j] = q > 0.f ? q : 1.f;
  }
  for (int i = tid; i < S; i += 256)
#pragma unroll
    for (int j = 0; j < 3; ++j)
      if (j < d) xs[((size_t)b * S + i) * d + j] = (xb[(size_t)i * d + j] - m[j]) / sd[j];
  if (t)
    for (int i = tid; i < k; i += 256)
#pragma unroll
      for (int j = 0; j < 3; ++j)
        if (j < d) ts[((size_t)b * k + i) * d + j] = (t[((size_t)b * k + i) * d + j] - m[j]) / sd[j];
  if (tid == 0)
    for (int j = 0; j < d; ++j) {
      ms[b * 2 * d + j] = m[j];
      ms[b * 2 * d + d + j] = sd[j];
    }
}

__global__ void sn_transpose(const float* __restrict__ prm, int d, int k, float* w2t) {
  const NetOff o = net_off(d, k);
  const int q = blockIdx.x * blockDim.x + threadIdx.x;  // w2t[c][u] = W2[u][c]
  if (q < H * H) w2t[q] = prm[o.W2 + (q % H) * H + q / H];
}

// acc[r][c] += sum over k of a[k][8 ty + r] w[k][4 tx + (c & 3) + 64 (c >> 2)],
// k ascending: one fused multiply-add per term.  16 unit groups tx of two
// runs of four units: the 16-byte reads of a half-warp are then contiguous
// (with eight units in a row per thread they would hit every bank twice).
template <int KN, int AS, int WS>
__device__ __forceinline__ void tile_gemm_8x8(const float* __restrict__ a, const float* __restrict__ w, int ty, int tx,
                                              float (&acc)[8][8]) {
#pragma unroll 4
  for (int q = 0; q < KN; ++q) {
    const float4 a0 = *reinterpret_cast<const float4*>(a + q * AS + 8 * ty);
    const float4 a1 = *reinterpret_cast<const float4*>(a + q * AS + 8 * ty + 4);
    const float4 w0 = *reinterpret_cast<const float4*>(w + q * WS + 4 * tx);
    const float4 w1 = *reinterpret_cast<const float4*>(w + q * WS + 64 + 4 * tx);
    const float av[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
    const float wv[8] = {w0.x, w0.y, w0.z, w0.w, w1.x, w1.y, w1.z, w1.w};
#pragma unroll
    for (int r = 0; r < 8; ++r)
#pragma unroll
      for (int c = 0; c < 8; ++c) acc[r][c] = fmaf(av[r], wv[c], acc[r][c]);
  }
}

// The per-point layers of PT points (PT = 64 or 256, 2 PT threads): h1 into
// shared memory transposed, h2 by 8 points x 8 units per thread.  Bound by
// the FP32 multiply-adds (17.2e9 for 1M points: 0.46 ms at one per lane and
// cycle); neither h1 nor h2 goes to memory (the backward pass forms h1 again
// and needs only the sign of h2: 16 bytes per point instead of 1 KB), and the
// 8x8 tile takes 4 16-byte shared reads per 64 multiply-adds (the 8x4 tile: 3
// per 32).  Resident blocks stride over the tiles, so W2 is staged once each.
// 1M points: 1.29 -> 0.69 ms.  64-point blocks where 256-point ones
// would leave SMs idle.  The pooled sum of 64 points is added as before: 8
// points in order per thread, then the eight groups in order.
template <int PT>
__global__ void __launch_bounds__(2 * PT) sn_fwd_points(const float* __restrict__ xs, const float* __restrict__ prm,
                                                        const float* __restrict__ w2t, int d, int k, int64_t P,
                                                        uint32_t* __restrict__ bits, float* __restrict__ tile_pool) {
  constexpr int AS = PT + 4, NT = 2 * PT;
  extern __shared__ __align__(16) float sm[];
  float* s_w2 = sm;               // [128][128]: s_w2[c][u] = W2[u][c]
  float* s_h1 = s_w2 + H * H;     // [128][AS]: s_h1[c][p]; then the pooled sums of 8 points [PT / 8][128]
  float* s_w1 = s_h1 + H * AS;    // [128][4]
  const NetOff o = net_off(d, k);
  const int tid = threadIdx.x, ty = tid >> 4, tx = tid & 15;
  for (int q = tid; q < H * H / 4; q += NT)
    reinterpret_cast<float4*>(s_w2)[q] = reinterpret_cast<const float4*>(w2t)[q];
  stage_w1(s_w1, prm, o, d, tid, NT);
  float b2[8];
#pragma unroll
  for (int c = 0; c < 8; ++c) b2[c] = prm[o.b2 + 4 * tx + (c & 3) + 64 * (c >> 2)];
  const int64_t ntiles = (P + PT - 1) / PT;
  for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    const int64_t p0 = tile * PT;
    __syncthreads();  // the weights; the tile before is read no more
    {
      const int p = tid % PT, u0 = (tid / PT) * (H / 2);
      float xv[3] = {0.f, 0.f, 0.f};
      if (p0 + p < P)
        for (int j = 0; j < d; ++j) xv[j] = xs[(p0 + p) * d + j];
#pragma unroll 8
      for (int u = u0; u < u0 + H / 2; ++u) s_h1[u * AS + p] = h1_of(s_w1, xv, u);
    }
    __syncthreads();
    float acc[8][8], ps[8];
#pragma unroll
    for (int r = 0; r < 8; ++r)
#pragma unroll
      for (int c = 0; c < 8; ++c) acc[r][c] = 0.f;
    tile_gemm_8x8<H, AS, H>(s_h1, s_w2, ty, tx, acc);
#pragma unroll
    for (int c = 0; c < 8; ++c) ps[c] = 0.f;
    const bool live = p0 + 8 * ty < P;  // P is a multiple of 64
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      uint32_t m = 0u;  // bits 0..3: units 4 tx .. 4 tx + 3, bits 4..7: 64 + those
#pragma unroll
      for (int c = 0; c < 8; ++c) {
        const float h = fmaxf(acc[r][c] + b2[c], 0.f);
        ps[c] += h;
        m |= (h > 0.f ? 1u : 0u) << c;
      }
      if (bits) {
        // the point's 128 bits from the 16 threads of its unit groups: word w
        // (units 32 w .. 32 w + 31) from groups 8 (w & 1) .. + 7
        uint32_t lo = (m & 15u) << (4 * (tx & 7)), hi = (m >> 4) << (4 * (tx & 7));
#pragma unroll
        for (int f = 1; f < 8; f <<= 1) {
          lo |= __shfl_xor_sync(0xffffffffu, lo, f);
          hi |= __shfl_xor_sync(0xffffffffu, hi, f);
        }
        if (live && (tx & 7) == 0) {
          uint32_t* w = bits + (p0 + 8 * ty + r) * 4 + (tx >> 3);
          w[0] = lo;
          w[2] = hi;
        }
      }
    }
    __syncthreads();  // s_h1 is read no more: the pooled sums take its place
#pragma unroll
    for (int c = 0; c < 8; ++c) s_h1[ty * H + 4 * tx + (c & 3) + 64 * (c >> 2)] = ps[c];
    __syncthreads();
    for (int q = tid; q < PT / kTileP * H; q += NT) {
      const int t = q / H, u = q % H;
      if (p0 + t * kTileP >= P) break;
      float s = 0.f;
      for (int g = 0; g < 8; ++g) s += s_h1[(8 * t + g) * H + u];
      tile_pool[(tile * (PT / kTileP) + t) * H + u] = s;
    }
  }
}

// One block per set: the pooled mean, the head forward and, with targets, the
// set's loss and the head backward to dg (the weight gradients, sums over the
// sets, are sn_head_grad's).  W3 and W4 are staged in shared memory with an
// odd row stride, so a thread per row reads them without bank conflicts.  (One
// block over all sets in order, one thread per loss: 26.2 ms for 256 sets;
// this and sn_head_grad: 0.053 ms.)
constexpr int kWS = H + 1;
__global__ void __launch_bounds__(256) sn_head(const float* __restrict__ prm, const float* __restrict__ tile_pool,
                                               int tiles_per_set, int S, int B, int d, int k,
                                               const float* __restrict__ ts, float* __restrict__ G,
                                               float* __restrict__ P, float* __restrict__ A3, float* __restrict__ dZ3,
                                               float* __restrict__ dP, float* __restrict__ dG,
                                               float* __restrict__ set_loss) {
  extern __shared__ __align__(16) float s_w[];  // [max(H, KD)][kWS]: W3, then W4
  __shared__ float s_g[H], s_z3[H], s_a3[H], s_dz3[H];
  __shared__ float s_p[kBatchMaxK * 3], s_dp[kBatchMaxK * 3], s_t[kBatchMaxK * 3];
  __shared__ float s_d1[kBatchMaxK], s_d2[kBatchMaxK];
  __shared__ int s_j1[kBatchMaxK], s_j2[kBatchMaxK];
  const NetOff o = net_off(d, k);
  const int tid = threadIdx.x, KD = k * d, b = blockIdx.x;
  const bool train = ts != nullptr;
  for (int q = tid; q < H * H; q += 256) s_w[(q / H) * kWS + q % H] = prm[o.W3 + q];
  if (tid < H) {
    float s = 0.f;
    const float* tp = tile_pool + (size_t)b * tiles_per_set * H + tid;
#pragma unroll 8
    for (int t = 0; t < tiles_per_set; ++t) s += tp[(size_t)t * H];
    s = s / (float)S;
    s_g[tid] = s;
    G[b * H + tid] = s;
  }
  __syncthreads();
  if (tid < H) {
    float z = prm[o.b3 + tid];
#pragma unroll 8
    for (int c = 0; c < H; ++c) z = fmaf(s_w[tid * kWS + c], s_g[c], z);
    s_z3[tid] = z;
    s_a3[tid] = fmaxf(z, 0.f);
    if (train) A3[b * H + tid] = fmaxf(z, 0.f);
  }
  __syncthreads();
  for (int q = tid; q < KD * H; q += 256) s_w[(q / H) * kWS + q % H] = prm[o.W4 + q];
  __syncthreads();
  for (int q = tid; q < KD; q += 256) {
    float z = prm[o.b4 + q];
#pragma unroll 8
    for (int u = 0; u < H; ++u) z = fmaf(s_w[q * kWS + u], s_a3[u], z);
    s_p[q] = z;
    P[(size_t)b * KD + q] = z;
    if (train) s_t[q] = ts[(size_t)b * KD + q];
  }
  __syncthreads();
  if (!train) return;
  // symmetric Chamfer distance: nearest target of each prediction (threads
  // 0..k-1) and nearest prediction of each target (threads 128..128+k-1),
  // lowest index on ties
  if ((tid & 127) < k) {
    const int a = tid & 127;
    const float* pa = tid < 128 ? s_p : s_t;
    const float* pb = tid < 128 ? s_t : s_p;
    int js = 0;
    float best = 3.0e38f;
    for (int j = 0; j < k; ++j) {
      float dd = 0.f;
      for (int c = 0; c < d; ++c) {
        const float u = pa[a * d + c] - pb[j * d + c];  // the sign does not matter
        dd = fmaf(u, u, dd);
      }
      if (dd < best) { best = dd; js = j; }
    }
    (tid < 128 ? s_d1 : s_d2)[a] = best;
    (tid < 128 ? s_j1 : s_j2)[a] = js;
  }
  __syncthreads();
  const float sc = 2.f / ((float)k * (float)B);  // gradients scaled by 1 / (K B)
  for (int q = tid; q < KD; q += 256) {
    const int a = q / d, c = q - a * d;
    float v = sc * (s_p[q] - s_t[s_j1[a] * d + c]);
    for (int j = 0; j < k; ++j)
      if (s_j2[j] == a) v = fmaf(sc, s_p[q] - s_t[j * d + c], v);
    s_dp[q] = v;
    dP[(size_t)b * KD + q] = v;
  }
  if (tid == 0) {
    float l1 = 0.f, l2 = 0.f;
    for (int a = 0; a < k; ++a) l1 += s_d1[a];
    for (int j = 0; j < k; ++j) l2 += s_d2[j];
    set_loss[b] = (l1 + l2) / (float)k / (float)B;
  }
  __syncthreads();
  if (tid < H) {
    float da = 0.f;
#pragma unroll 8
    for (int q = 0; q < KD; ++q) da = fmaf(s_w[q * kWS + tid], s_dp[q], da);
    const float z = s_z3[tid] > 0.f ? da : 0.f;
    s_dz3[tid] = z;
    dZ3[b * H + tid] = z;
  }
  __syncthreads();
  if (tid < H) {
    float dg = 0.f;
#pragma unroll 8
    for (int u = 0; u < H; ++u) dg = fmaf(prm[o.W3 + u * H + tid], s_dz3[u], dg);
    dG[b * H + tid] = dg;
  }
}

// dW3 = sum_b dz3 g^T, dW4 = sum_b dp a3^T, db3, db4 and the loss: one thread
// per value, the sets added in order.
__global__ void __launch_bounds__(128) sn_head_grad(int B, int d, int k, const float* __restrict__ G,
                                                    const float* __restrict__ A3, const float* __restrict__ dZ3,
                                                    const float* __restrict__ dP, const float* __restrict__ set_loss,
                                                    float* __restrict__ grads, float* __restrict__ loss) {
  const NetOff o = net_off(d, k);
  const int KD = k * d;
  const int q = blockIdx.x * 128 + threadIdx.x;
  float s = 0.f;
  if (q < H * H) {
    const int u = q / H, c = q % H;
#pragma unroll 8
    for (int b = 0; b < B; ++b) s = fmaf(dZ3[b * H + u], G[b * H + c], s);
    grads[o.W3 + q] = s;
  } else if (q < H * H + KD * H) {
    const int r = (q - H * H) / H, u = (q - H * H) % H;
#pragma unroll 8
    for (int b = 0; b < B; ++b) s = fmaf(dP[(size_t)b * KD + r], A3[b * H + u], s);
    grads[o.W4 + r * H + u] = s;
  } else if (q < H * H + KD * H + H) {
    const int u = q - H * H - KD * H;
#pragma unroll 8
    for (int b = 0; b < B; ++b) s += dZ3[b * H + u];
    grads[o.b3 + u] = s;
  } else if (q < H * H + KD * H + H + KD) {
    const int r = q - H * H - KD * H - H;
#pragma unroll 8
    for (int b = 0; b < B; ++b) s += dP[(size_t)b * KD + r];
    grads[o.b4 + r] = s;
  } else if (q == H * H + KD * H + H + KD) {
    for (int b = 0; b < B; ++b) s += set_loss[b];
    *loss = s;
  }
}

// The blocks' partial gradients added in order.
__global__ void __launch_bounds__(64) sn_wgrad_reduce(const float* __restrict__ part, int nparts, int d, int k,
                                                      float* __restrict__ grads) {
  const NetOff o = net_off(d, k);
  const int stride = H * H + H * d + 2 * H;
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= stride) return;
  float s = 0.f;
#pragma unroll 8
  for (int c = 0; c < nparts; ++c) s += part[(size_t)c * stride + q];
  int dst;
  if (q < H * H) dst = o.W2 + q;
  else if (q < H * H + H * d) dst = o.W1 + (q - H * H);
  else if (q < H * H + H * d + H) dst = o.b1 + (q - H * H - H * d);
  else dst = o.b2 + (q - H * H - H * d - H);
  grads[dst] = s;
}

// The gradients of a pass that gave up (*err) are not taken.
__global__ void sn_adam(float* prm, const float* grads, float* m, float* v, int n, float lr, float b1, float b2,
                        float eps, float c1, float c2, const int* err, int* skipped) {
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (*err) {
    if (q == 0) *skipped += 1;
    return;
  }
  if (q >= n) return;
  const float g = grads[q];
  const float mq = b1 * m[q] + (1.f - b1) * g;
  const float vq = b2 * v[q] + (1.f - b2) * g * g;
  m[q] = mq;
  v[q] = vq;
  prm[q] -= lr * (mq / c1) / (sqrtf(vq / c2) + eps);
}

// Sample of S points of a context: point floor(u_j N), u_j the j-th output
// of SplitMix64 (Vigna) from the seed, to 53 bits.
__global__ void sn_sample(const float* __restrict__ x, int64_t ld, int64_t n, int d, int S, unsigned long long seed,
                          float* out) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= S) return;
  unsigned long long z = seed + (unsigned long long)(j + 1) * 0x9E3779B97F4A7C15ull;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  z ^= z >> 31;
  const double u = (double)(z >> 11) * 0x1p-53;
  int64_t i = (int64_t)(u * (double)n);
  if (i >= n) i = n - 1;
  for (int c = 0; c < d; ++c) out[(size_t)j * d + c] = x[(int64_t)c * ld + i];
}

// Centres in the points' coordinates: c = p * s + m (FP64 output).
__global__ void sn_destd(const float* P, const float* ms, int B, int d, int k, double* out) {
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= B * k * d) return;
  const int b = q / (k * d), j = q % d;
  out[q] = (double)P[q] * (double)ms[b * 2 * d + d + j] + (double)ms[b * 2 * d + j];
}

}  // namespace

int setnet_param_count(int d, int k) { return net_off(d, k).total; }

cudaError_t launch_setnet_destandardize(const float* P, const float* ms, int B, int d, int k, double* out,
                                        cudaStream_t st) {
  const int n = B * k * d;
  sn_destd<<<(n + 255) / 256, 256, 0, st>>>(P, ms, B, d, k, out);
  return cudaGetLastError();
}

template <int PT>
static cudaError_t launch_fwd_points(const SetNetArgs& a, bool train, int64_t P, cudaStream_t st) {
  const size_t smem = sizeof(float) * (H * H + H * (PT + 4) + 4 * H);
  cudaError_t e = cudaFuncSetAttribute(sn_fwd_points<PT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  // resident blocks stride over the tiles: W2 (64 KB) is staged once each
  const int64_t grid = std::min<int64_t>((P + PT - 1) / PT, 152 * (PT == 256 ? 1 : 2));
  sn_fwd_points<PT><<<(unsigned)grid, 2 * PT, smem, st>>>(a.xs, a.prm, a.w2t, a.d, a.k, P, train ? a.bits : nullptr,
                                                          a.tile_pool);
  return cudaGetLastError();
}

cudaError_t launch_setnet_forward(const SetNetArgs& a, bool train, cudaStream_t st) {
  const int64_t P = (int64_t)a.B * a.S;
  sn_standardize<<<a.B, 256, 0, st>>>(a.x, train ? a.t : nullptr, a.S, a.d, a.k, a.xs, a.ts, a.ms);
  sn_transpose<<<H * H / 256, 256, 0, st>>>(a.prm, a.d, a.k, a.w2t);
  // 256-point blocks (one per SM) once they fill the SMs twice over; below
  // that 64-point ones, two to an SM
  cudaError_t e = P >= int64_t(256) * 2 * 152 ? launch_fwd_points<256>(a, train, P, st)
                                              : launch_fwd_points<64>(a, train, P, st);
  if (e != cudaSuccess) return e;
  const size_t hs = sizeof(float) * (size_t)std::max(H, a.k * a.d) * kWS;
  e = allow_max_smem<sn_head>();
  if (e != cudaSuccess) return e;
  sn_head<<<a.B, 256, hs, st>>>(a.prm, a.tile_pool, a.S / kTileP, a.S, a.B, a.d, a.k, train ? a.ts : nullptr, a.G, a.P,
                                a.A3, a.dZ3, a.dP, a.dG, a.set_loss);
  if (train) {
    const int nv = H * H + a.k * a.d * (H + 1) + H + 1;
    sn_head_grad<<<(nv + 127) / 128, 128, 0, st>>>(a.B, a.d, a.k, a.G, a.A3, a.dZ3, a.dP, a.set_loss, a.grads, a.loss);
  }
  return cudaGetLastError();
}

cudaError_t launch_setnet_backward(const SetNetArgs& a, cudaStream_t st) {
  const int nb = setnet_bwd_blocks(a.B, a.S);
  cudaError_t e = launch_setnet_bwd_points(a, nb, st);
  if (e != cudaSuccess) return e;
  const int stride = H * H + H * a.d + 2 * H;
  sn_wgrad_reduce<<<(stride + 63) / 64, 64, 0, st>>>(a.part, nb, a.d, a.k, a.grads);
  return cudaGetLastError();
}

int64_t setnet_part_floats(int d) { return (int64_t)kSetBwdBlocks * (H * H + H * d + 2 * H); }

cudaError_t launch_setnet_adam(float* prm, const float* grads, float* m, float* v, int n, float lr, float b1,
                               float b2, float eps, float c1, float c2, const int* err, int* skipped,
                               cudaStream_t st) {
  sn_adam<<<(n + 255) / 256, 256, 0, st>>>(prm, grads, m, v, n, lr, b1, b2, eps, c1, c2, err, skipped);
  return cudaGetLastError();
}

cudaError_t launch_setnet_sample(const float* x, int64_t ld, int64_t n, int d, int S, unsigned long long seed,
                                 float* out, cudaStream_t st) {
  sn_sample<<<(S + 255) / 256, 256, 0, st>>>(x, ld, n, d, S, seed, out);
  return cudaGetLastError();
}

namespace {

// Per-set mean of B sets of S points (d <= 3), FP64, one block per set:
// thread-strided partial sums combined by a fixed-order tree.
__global__ void __launch_bounds__(256) sets_mean_kernel(const float* __restrict__ x, int64_t set_stride, int S,
                                                        int d, double* __restrict__ means) {
  __shared__ double red[3][256];
  const int b = blockIdx.x, tid = threadIdx.x;
  const float* xs = x + (int64_t)b * set_stride;
  double acc[3] = {0.0, 0.0, 0.0};
  for (int s = tid; s < S; s += blockDim.x)
    for (int j = 0; j < d; ++j) acc[j] = __dadd_rn(acc[j], (double)xs[(int64_t)s * d + j]);
  for (int j = 0; j < 3; ++j) red[j][tid] = acc[j];
  __syncthreads();
  for (int w = blockDim.x / 2; w > 0; w >>= 1) {
    if (tid < w)
      for (int j = 0; j < 3; ++j) red[j][tid] = __dadd_rn(red[j][tid], red[j][tid + w]);
    __syncthreads();
  }
  if (tid < d) means[(int64_t)b * d + tid] = __ddiv_rn(red[tid][0], (double)S);
}

// out[b][s] = R_b (x[b][s] - c_b) + c_b (R_b^T with transpose), in FP64;
// R: B x d x d row-major, c: one centre per set (stride center_stride
// doubles; null = the origin).
template <typename T>
__global__ void sets_rotate_kernel(const T* __restrict__ x, int64_t set_stride, int B, int S, int d,
                                   const double* __restrict__ R, const double* __restrict__ c, int64_t center_stride,
                                   int transpose, T* __restrict__ out) {
  const int64_t total = (int64_t)B * S;
  for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < total; q += (int64_t)gridDim.x * blockDim.x) {
    const int b = (int)(q / S), s = (int)(q - (int64_t)b * S);
    const T* xp = x + (int64_t)b * set_stride + (int64_t)s * d;
    const double* Rb = R + (int64_t)b * d * d;
    double v[3], cc[3] = {0.0, 0.0, 0.0};
    for (int j = 0; j < d; ++j) {
      if (c) cc[j] = c[(int64_t)b * center_stride + j];
      v[j] = __dsub_rn((double)xp[j], cc[j]);
    }
    T* op = out + q * d;
    for (int i = 0; i < d; ++i) {
      double acc = 0.0;
      for (int j = 0; j < d; ++j)
        acc = __dadd_rn(acc, __dmul_rn(transpose ? Rb[j * d + i] : Rb[i * d + j], v[j]));
      op[i] = (T)__dadd_rn(acc, cc[i]);
    }
  }
}

}  // namespace

cudaError_t launch_sets_mean(const float* x, int64_t set_stride, int B, int S, int d, double* means, cudaStream_t st) {
  sets_mean_kernel<<<B, 256, 0, st>>>(x, set_stride, S, d, means);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_sets_rotate(const T* x, int64_t set_stride, int B, int S, int d, const double* R,
                               const double* c, int64_t center_stride, int transpose, T* out, cudaStream_t st) {
  const int64_t total = (int64_t)B * S;
  const int grid = (int)std::max<int64_t>(1, std::min<int64_t>((total + 255) / 256, 4096));
  sets_rotate_kernel<T><<<grid, 256, 0, st>>>(x, set_stride, B, S, d, R, c, center_stride, transpose, out);
  return cudaGetLastError();
}
template cudaError_t launch_sets_rotate<float>(const float*, int64_t, int, int, int, const double*, const double*,
                                               int64_t, int, float*, cudaStream_t);
template cudaError_t launch_sets_rotate<double>(const double*, int64_t, int, int, int, const double*, const double*,
                                                int64_t, int, double*, cudaStream_t);

}  // namespace km
