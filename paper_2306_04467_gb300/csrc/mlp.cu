// Training and evaluation kernels of the learned troubled-cell gate
// (24 -> 32 -> 32 -> 1, ReLU, sigmoid output), on BF16 tensor cores with FP32
// accumulation (mma.sync m16n8k16), and their C ABI (include/gks2l.h).
//
// k_mlp_grad: forward and backward of the logistic loss
//   L = sum_i pos_w y_i softplus(-s_i) + (1 - y_i) softplus(s_i)
// over a batch; each warp takes 16 samples at a time. Layer outputs stay in
// registers and are reused as the A operand of the next product; the weight
// gradients dW = dZ^T H are products over the batch dimension, read
// transposed from a per-warp shared-memory tile. Sums are FP32, in a fixed
// order (the warps of a block, then the blocks by a fixed tree): the gradient
// is the same from run to run.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cstdint>
#include <mutex>

#include "gks2l.h"
#include "launch.cuh"
#include "mlp.cuh"

using namespace gks2l;

namespace {

constexpr int TPB = 128;

__device__ __forceinline__ unsigned pack2(__nv_bfloat16 lo, __nv_bfloat16 hi) {
  __nv_bfloat162 v;
  v.x = lo;
  v.y = hi;
  return *reinterpret_cast<unsigned *>(&v);
}
__device__ __forceinline__ float bfr(float x) { return __bfloat162float(__float2bfloat16_rn(x)); }
__device__ __forceinline__ float softplus(float x) { return x > 0.f ? x + log1pf(expf(-x)) : log1pf(expf(x)); }
__device__ __forceinline__ float sigm(float x) { return 1.f / (1.f + expf(-x)); }

struct WarpTiles {
  __nv_bfloat16 X[16 * 32], H1[16 * 32], DZ2[16 * 32], DZ1[16 * 32];
};

// A fragment of T^T (m = column of T, k = row of T) from a bf16 [16][32] tile
__device__ __forceinline__ void load_a_t(unsigned a[4], const __nv_bfloat16 *T, int m0, int lane) {
  const int g = lane >> 2, c = (lane & 3) * 2;
  a[0] = pack2(T[c * 32 + m0 + g], T[(c + 1) * 32 + m0 + g]);
  a[1] = pack2(T[c * 32 + m0 + g + 8], T[(c + 1) * 32 + m0 + g + 8]);
  a[2] = pack2(T[(c + 8) * 32 + m0 + g], T[(c + 9) * 32 + m0 + g]);
  a[3] = pack2(T[(c + 8) * 32 + m0 + g + 8], T[(c + 9) * 32 + m0 + g + 8]);
}
// B fragment (k = row of T, n = column of T) from a bf16 [16][32] tile
__device__ __forceinline__ void load_b_t(unsigned b[2], const __nv_bfloat16 *T, int n0, int lane) {
  const int g = lane >> 2, c = (lane & 3) * 2;
  b[0] = pack2(T[c * 32 + n0 + g], T[(c + 1) * 32 + n0 + g]);
  b[1] = pack2(T[(c + 8) * 32 + n0 + g], T[(c + 9) * 32 + n0 + g]);
}

// Rows r0.. of X [n][24] into a warp's BF16 tile of ROWS rows (row stride LD
// elements, columns 24..31 already zero): each lane takes ROWS * 24 / 128
// 16-byte vectors, which lie in one row each. Rows past n become zero.
template <int ROWS> struct RowVecs {
  static constexpr int N = ROWS * MLP_IN / 4 / 32;
  float4 v[N];
};
template <int ROWS>
__device__ __forceinline__ void rows_load(RowVecs<ROWS> &t, const float *X, int n, int r0, int lane, bool aligned) {
  const long long have = ((long long)n - r0) * MLP_IN;   // values from r0 on
  const float *p = X + (size_t)r0 * MLP_IN;
#pragma unroll
  for (int i = 0; i < RowVecs<ROWS>::N; i++) {
    const int e = 4 * (lane + 32 * i);
    t.v[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (e < have) {
      if (aligned) t.v[i] = __ldg(reinterpret_cast<const float4 *>(p + e));
      else t.v[i] = make_float4(p[e], p[e + 1], p[e + 2], p[e + 3]);
    }
  }
}
__device__ __forceinline__ bool aligned16(const float *p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; }

// Each block writes its partial sums (NTRAIN gradients, then the loss) to
// part[block]; k_mlp_reduce adds them up in a fixed order, so the result does
// not depend on scheduling. At the usual batch (8192: 128 blocks, one tile of
// 16 samples per warp) the kernel is a chain of latencies: network to shared
// memory, rows, six small products, sums; so rows come as 16-byte vectors
// requested before the network is packed, and the warps' sums meet in shared
// memory, which leaves the reduction a quarter of the partials. A training
// step (gradient, reduction, Adam) of 8192 samples, steps queued: 32.1 -> 23.9 us,
// 21.4 with the reduction's launch chained; alone after a synchronisation 206 -> 195,
// most of it the partials' memory, which the default pool has given back.
constexpr int NPART = MLP_NTRAIN + 1;

__global__ void __launch_bounds__(TPB) k_mlp_grad(const float *X, const float *y, int n, const float *P, float pos_w,
                                                  float *part) {
  __shared__ MlpDev w;
  __shared__ WarpTiles tiles[TPB / 32];
  __shared__ float acc[NPART];
  const bool al = aligned16(X);
  RowVecs<16> rows;
  rows_load<16>(rows, X, n, (blockIdx.x * (TPB / 32) + (threadIdx.x >> 5)) * 16, threadIdx.x & 31, al);
  mlp_pack(w, P, 0.f, threadIdx.x, TPB);
  for (int i = threadIdx.x & 31; i < 16 * 4; i += 32)
    *reinterpret_cast<unsigned *>(&tiles[threadIdx.x >> 5].X[(i >> 2) * 32 + MLP_IN + 2 * (i & 3)]) = 0u;
  __syncthreads();
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int g = lane >> 2, c = (lane & 3) * 2;
  WarpTiles &S = tiles[wid];
  float gW1[2][4][4], gW2[2][4][4];
  float gb1[4][2], gb2[4][2], gw3[4][2], gb3 = 0.f, lsum = 0.f;
  for (int a = 0; a < 2; a++)
    for (int b = 0; b < 4; b++)
      for (int i = 0; i < 4; i++) gW1[a][b][i] = gW2[a][b][i] = 0.f;
  for (int b = 0; b < 4; b++)
    for (int i = 0; i < 2; i++) gb1[b][i] = gb2[b][i] = gw3[b][i] = 0.f;
  const int ntile = (n + 15) / 16;
  for (int t = blockIdx.x * (TPB / 32) + wid; t < ntile; t += gridDim.x * (TPB / 32)) {
    const int r0 = t * 16;
    if (t != (int)(blockIdx.x * (TPB / 32) + wid)) rows_load<16>(rows, X, n, r0, lane, al);
#pragma unroll
    for (int i = 0; i < RowVecs<16>::N; i++) {
      const int e = 4 * (lane + 32 * i), r = e / MLP_IN, k = e - r * MLP_IN;
      const float *v = reinterpret_cast<const float *>(&rows.v[i]);
      float x[4];
      for (int m = 0; m < 4; m++) x[m] = r0 + r < n ? (v[m] - w.mean[k + m]) * w.istd[k + m] : 0.f;
      uint2 q;
      q.x = pack_bf16(x[0], x[1]);
      q.y = pack_bf16(x[2], x[3]);
      *reinterpret_cast<uint2 *>(&S.X[r * 32 + k]) = q;
    }
    __syncwarp();
    // ---- forward
    float z1[4][4];
    for (int nt = 0; nt < 4; nt++)
      for (int i = 0; i < 4; i++) z1[nt][i] = 0.f;
    for (int ks = 0; ks < 2; ks++) {
      unsigned a[4];
      load_a(a, S.X, 32, 0, 16 * ks, lane);
      for (int nt = 0; nt < 4; nt++) {
        unsigned b[2];
        load_b_nk(b, w.w1, 32, 8 * nt, 16 * ks, lane);
        mma_bf16(z1[nt], a, b);
      }
    }
    unsigned a2[2][4];
    float m1[4][4];
    for (int nt = 0; nt < 4; nt++) {
      int col = 8 * nt + c;
      float p[4] = {z1[nt][0] + w.b1[col], z1[nt][1] + w.b1[col + 1], z1[nt][2] + w.b1[col], z1[nt][3] + w.b1[col + 1]};
      float h[4];
      for (int i = 0; i < 4; i++) {
        m1[nt][i] = p[i] > 0.f ? 1.f : 0.f;
        h[i] = fmaxf(p[i], 0.f);
      }
      a2[nt >> 1][2 * (nt & 1)] = pack_bf16(h[0], h[1]);
      a2[nt >> 1][2 * (nt & 1) + 1] = pack_bf16(h[2], h[3]);
      S.H1[g * 32 + col] = __float2bfloat16_rn(h[0]);
      S.H1[g * 32 + col + 1] = __float2bfloat16_rn(h[1]);
      S.H1[(g + 8) * 32 + col] = __float2bfloat16_rn(h[2]);
      S.H1[(g + 8) * 32 + col + 1] = __float2bfloat16_rn(h[3]);
    }
    float z2[4][4];
    for (int nt = 0; nt < 4; nt++)
      for (int i = 0; i < 4; i++) z2[nt][i] = 0.f;
    for (int ks = 0; ks < 2; ks++)
      for (int nt = 0; nt < 4; nt++) {
        unsigned b[2];
        load_b_nk(b, w.w2, 32, 8 * nt, 16 * ks, lane);
        mma_bf16(z2[nt], a2[ks], b);
      }
    float h2v[4][4], m2[4][4];
    float s0 = 0.f, s1 = 0.f;
    for (int nt = 0; nt < 4; nt++) {
      int col = 8 * nt + c;
      float p[4] = {z2[nt][0] + w.b2[col], z2[nt][1] + w.b2[col + 1], z2[nt][2] + w.b2[col], z2[nt][3] + w.b2[col + 1]};
      for (int i = 0; i < 4; i++) {
        m2[nt][i] = p[i] > 0.f ? 1.f : 0.f;
        h2v[nt][i] = bfr(fmaxf(p[i], 0.f));
      }
      s0 += h2v[nt][0] * w.w3[col] + h2v[nt][1] * w.w3[col + 1];
      s1 += h2v[nt][2] * w.w3[col] + h2v[nt][3] * w.w3[col + 1];
    }
    s0 += __shfl_xor_sync(0xffffffffu, s0, 1);
    s0 += __shfl_xor_sync(0xffffffffu, s0, 2);
    s1 += __shfl_xor_sync(0xffffffffu, s1, 1);
    s1 += __shfl_xor_sync(0xffffffffu, s1, 2);
    s0 += w.b3;
    s1 += w.b3;
    // ---- loss and its derivative in the logit, rows g and g + 8
    const int ra = r0 + g, rb = r0 + g + 8;
    const bool va = ra < n, vb = rb < n;
    const float ya = va ? y[ra] : 0.f, yb = vb ? y[rb] : 0.f;
    const float dsa = va ? (-pos_w * ya * sigm(-s0) + (1.f - ya) * sigm(s0)) : 0.f;
    const float dsb = vb ? (-pos_w * yb * sigm(-s1) + (1.f - yb) * sigm(s1)) : 0.f;
    if ((lane & 3) == 0) {
      if (va) lsum += pos_w * ya * softplus(-s0) + (1.f - ya) * softplus(s0);
      if (vb) lsum += pos_w * yb * softplus(-s1) + (1.f - yb) * softplus(s1);
      gb3 += dsa + dsb;
    }
    // ---- backward
    float dz2[4][4];
    unsigned ad[2][4];
    for (int nt = 0; nt < 4; nt++) {
      int col = 8 * nt + c;
      dz2[nt][0] = dsa * w.w3[col] * m2[nt][0];
      dz2[nt][1] = dsa * w.w3[col + 1] * m2[nt][1];
      dz2[nt][2] = dsb * w.w3[col] * m2[nt][2];
      dz2[nt][3] = dsb * w.w3[col + 1] * m2[nt][3];
      gw3[nt][0] += dsa * h2v[nt][0] + dsb * h2v[nt][2];
      gw3[nt][1] += dsa * h2v[nt][1] + dsb * h2v[nt][3];
      gb2[nt][0] += dz2[nt][0] + dz2[nt][2];
      gb2[nt][1] += dz2[nt][1] + dz2[nt][3];
      ad[nt >> 1][2 * (nt & 1)] = pack_bf16(dz2[nt][0], dz2[nt][1]);
      ad[nt >> 1][2 * (nt & 1) + 1] = pack_bf16(dz2[nt][2], dz2[nt][3]);
      S.DZ2[g * 32 + col] = __float2bfloat16_rn(dz2[nt][0]);
      S.DZ2[g * 32 + col + 1] = __float2bfloat16_rn(dz2[nt][1]);
      S.DZ2[(g + 8) * 32 + col] = __float2bfloat16_rn(dz2[nt][2]);
      S.DZ2[(g + 8) * 32 + col + 1] = __float2bfloat16_rn(dz2[nt][3]);
    }
    // dH1 = dZ2 W2: B element (k = out, n = in) = W2[k][n]
    float dh1[4][4];
    for (int nt = 0; nt < 4; nt++)
      for (int i = 0; i < 4; i++) dh1[nt][i] = 0.f;
    for (int ks = 0; ks < 2; ks++)
      for (int nt = 0; nt < 4; nt++) {
        const int k0 = 16 * ks + c, n0 = 8 * nt + g;
        unsigned b[2] = {pack2(w.w2[k0 * 32 + n0], w.w2[(k0 + 1) * 32 + n0]),
                         pack2(w.w2[(k0 + 8) * 32 + n0], w.w2[(k0 + 9) * 32 + n0])};
        mma_bf16(dh1[nt], ad[ks], b);
      }
    for (int nt = 0; nt < 4; nt++) {
      int col = 8 * nt + c;
      float d[4];
      for (int i = 0; i < 4; i++) d[i] = dh1[nt][i] * m1[nt][i];
      gb1[nt][0] += d[0] + d[2];
      gb1[nt][1] += d[1] + d[3];
      S.DZ1[g * 32 + col] = __float2bfloat16_rn(d[0]);
      S.DZ1[g * 32 + col + 1] = __float2bfloat16_rn(d[1]);
      S.DZ1[(g + 8) * 32 + col] = __float2bfloat16_rn(d[2]);
      S.DZ1[(g + 8) * 32 + col + 1] = __float2bfloat16_rn(d[3]);
    }
    __syncwarp();
    // weight gradients over the 16 samples: dW2 = dZ2^T H1, dW1 = dZ1^T X
    for (int mt = 0; mt < 2; mt++) {
      unsigned a[4], a1[4];
      load_a_t(a, S.DZ2, 16 * mt, lane);
      load_a_t(a1, S.DZ1, 16 * mt, lane);
      for (int nt = 0; nt < 4; nt++) {
        unsigned b[2], b1[2];
        load_b_t(b, S.H1, 8 * nt, lane);
        mma_bf16(gW2[mt][nt], a, b);
        load_b_t(b1, S.X, 8 * nt, lane);
        mma_bf16(gW1[mt][nt], a1, b1);
      }
    }
    __syncwarp();
  }
  // reduce the per-lane column partials over the eight row groups
  for (int nt = 0; nt < 4; nt++)
    for (int i = 0; i < 2; i++)
      for (int o = 4; o < 32; o <<= 1) {
        gb1[nt][i] += __shfl_xor_sync(0xffffffffu, gb1[nt][i], o);
        gb2[nt][i] += __shfl_xor_sync(0xffffffffu, gb2[nt][i], o);
        gw3[nt][i] += __shfl_xor_sync(0xffffffffu, gw3[nt][i], o);
      }
  for (int o = 1; o < 32; o <<= 1) {
    gb3 += __shfl_xor_sync(0xffffffffu, gb3, o);
    lsum += __shfl_xor_sync(0xffffffffu, lsum, o);
  }
  // the warps' sums in warp order, in shared memory
  for (int turn = 0; turn < TPB / 32; turn++) {
    if (wid == turn) {
      const bool first = turn == 0;
      auto put = [&](int i, float v) { acc[i] = first ? v : acc[i] + v; };
      if (lane < 4) {
        for (int nt = 0; nt < 4; nt++)
          for (int i = 0; i < 2; i++) {
            int col = 8 * nt + c + i;
            put(MLP_B1 + col, gb1[nt][i]);
            put(MLP_B2 + col, gb2[nt][i]);
            put(MLP_W3 + col, gw3[nt][i]);
          }
      }
      if (lane == 0) {
        put(MLP_B3, gb3);
        put(MLP_NTRAIN, lsum);
      }
      for (int mt = 0; mt < 2; mt++)
        for (int nt = 0; nt < 4; nt++)
          for (int i = 0; i < 4; i++) {
            int o = 16 * mt + g + (i >= 2 ? 8 : 0), in = 8 * nt + c + (i & 1);
            put(MLP_W2 + o * MLP_H + in, gW2[mt][nt][i]);
            if (in < MLP_IN) put(MLP_W1 + o * MLP_IN + in, gW1[mt][nt][i]);
          }
    }
    __syncthreads();
  }
  for (int i = threadIdx.x; i < NPART; i += TPB) part[(size_t)blockIdx.x * NPART + i] = acc[i];
}

// Sums of the blocks' partials: 32 values per block, each by eight threads
// over every eighth partial, then the eight in order (one thread per value
// over all partials is a serial chain of loads on eight blocks, 24 us at 512
// partials)
constexpr int RED_COLS = 32, RED_ROWS = 8;
__global__ void __launch_bounds__(RED_COLS *RED_ROWS) k_mlp_reduce(const float *part, int nparts, float *grads,
                                                                   float *loss_out) {
  dep_wait();
  __shared__ float s[RED_ROWS][RED_COLS];
  const int col = threadIdx.x % RED_COLS, row = threadIdx.x / RED_COLS, i = blockIdx.x * RED_COLS + col;
  float v = 0.f;
  if (i < NPART) {
#pragma unroll 8
    for (int w = row; w < nparts; w += RED_ROWS) v += part[(size_t)w * NPART + i];
  }
  s[row][col] = v;
  __syncthreads();
  if (row != 0 || i >= NPART) return;
  for (int r = 1; r < RED_ROWS; r++) v += s[r][col];
  if (i < MLP_NTRAIN) grads[i] = v;
  else *loss_out = v;
}

__global__ void k_mlp_adam(float *P, const float *G, float *M, float *V, int n, int step, float lr, float scale) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
  float gr = G[i] * scale;
  float m = b1 * M[i] + (1.f - b1) * gr;
  float v = b2 * V[i] + (1.f - b2) * gr * gr;
  M[i] = m;
  V[i] = v;
  float mh = m / (1.f - powf(b1, (float)step)), vh = v / (1.f - powf(b2, (float)step));
  P[i] -= lr * mh / (sqrtf(vh) + eps);
}

// logits with the inference image (normalisation folded into layer 1), the
// network the reconstruction runs. Bound by the samples' bytes: persistent
// blocks pack the network once, and each warp requests its next 32 rows as
// 16-byte vectors while the tensor cores work on the present ones:
// 77.5 -> 29.4 us for 1,000,003 samples (3.4 TB/s).
constexpr int FWD_BLOCKS_PER_SM = 4;
__global__ void __launch_bounds__(TPB, FWD_BLOCKS_PER_SM) k_mlp_forward(const float *X, int n, const float *P,
                                                                        float *logits) {
  constexpr int LD = 40;   // padded row stride of the feature tiles (bank spread)
  __shared__ MlpDev w;
  __shared__ __align__(16) __nv_bfloat16 Xs[TPB / 32][32 * LD];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int ntile = (n + 31) / 32, step = gridDim.x * (TPB / 32);
  const bool al = aligned16(X);
  int t = blockIdx.x * (TPB / 32) + wid;
  RowVecs<32> rows;
  if (t < ntile) rows_load<32>(rows, X, n, t * 32, lane, al);
  mlp_pack_folded(w, P, 0.f, threadIdx.x, TPB);
  for (int i = 0; i < 4; i++) *reinterpret_cast<unsigned *>(&Xs[wid][lane * LD + MLP_IN + 2 * i]) = 0u;
  __syncthreads();
  MlpFrags F;
  mlp_frags(F, w, lane);
  for (; t < ntile; t += step) {
#pragma unroll
    for (int i = 0; i < RowVecs<32>::N; i++) {
      const int e = 4 * (lane + 32 * i), r = e / MLP_IN, k = e - r * MLP_IN;
      uint2 q;
      q.x = pack_bf16(rows.v[i].x, rows.v[i].y);
      q.y = pack_bf16(rows.v[i].z, rows.v[i].w);
      *reinterpret_cast<uint2 *>(&Xs[wid][r * LD + k]) = q;
    }
    __syncwarp();
    if (t + step < ntile) rows_load<32>(rows, X, n, (t + step) * 32, lane, al);
    const float s = mlp_tile32(F, Xs[wid], LD, lane);
    if (t * 32 + lane < n) logits[t * 32 + lane] = s;
    __syncwarp();
  }
}

unsigned grid_for(int n, int per_block, int cap) {
  int b = (n + per_block - 1) / per_block;
  return (unsigned)(b < 1 ? 1 : (b > cap ? cap : b));
}

}  // namespace

namespace {

constexpr int MAX_DEV = 64;
struct PerDevice {
  std::once_flag once;
  int sms = 0;
};
PerDevice g_dev[MAX_DEV];

PerDevice *this_device() {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= MAX_DEV) return nullptr;
  PerDevice &D = g_dev[dev];
  std::call_once(D.once, [&] {
    if (cudaDeviceGetAttribute(&D.sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) D.sms = 0;
  });
  return D.sms > 0 ? &D : nullptr;
}

}  // namespace

extern "C" int gks2l_mlp_grad(const float *d_X, const float *d_y, int32_t n, const float *d_params, float pos_weight,
                              float *d_grads, float *d_loss, void *stream) {
  if (n <= 0 || !d_X || !d_y || !d_params || !d_grads || !d_loss) return GKS2L_EINVAL;
  cudaStream_t s = (cudaStream_t)stream;
  PerDevice *D = this_device();
  if (!D) return GKS2L_ECUDA;
  // one tile of 16 samples per warp while that fits two blocks per SM (what
  // the registers allow), then each warp loops
  const unsigned grid = grid_for(n, 16 * (TPB / 32), 2 * D->sms);
  const size_t bytes = (size_t)grid * NPART * sizeof(float);
  float *part = nullptr;
  if (cudaMallocAsync((void **)&part, bytes, s) != cudaSuccess) return GKS2L_ECUDA;
  k_mlp_grad<<<grid, TPB, 0, s>>>(d_X, d_y, n, d_params, pos_weight, part);
  launch(true, k_mlp_reduce, (NPART + RED_COLS - 1) / RED_COLS, RED_COLS * RED_ROWS, 0, s, part, (int)grid, d_grads,
         d_loss);
  const bool ok = cudaGetLastError() == cudaSuccess;
  if (cudaFreeAsync(part, s) != cudaSuccess || !ok) return GKS2L_ECUDA;
  return GKS2L_OK;
}

extern "C" int gks2l_mlp_adam(float *d_params, const float *d_grads, float *d_m, float *d_v, int32_t step, float lr,
                              float scale, void *stream) {
  if (!d_params || !d_grads || !d_m || !d_v || step <= 0) return GKS2L_EINVAL;
  k_mlp_adam<<<(MLP_NTRAIN + 255) / 256, 256, 0, (cudaStream_t)stream>>>(d_params, d_grads, d_m, d_v, MLP_NTRAIN,
                                                                          step, lr, scale);
  return cudaGetLastError() == cudaSuccess ? GKS2L_OK : GKS2L_ECUDA;
}

extern "C" int gks2l_mlp_forward(const float *d_X, int32_t n, const float *d_params, float *d_logits, void *stream) {
  if (n <= 0 || !d_X || !d_params || !d_logits) return GKS2L_EINVAL;
  PerDevice *D = this_device();
  if (!D) return GKS2L_ECUDA;
  k_mlp_forward<<<grid_for(n, 32 * (TPB / 32), FWD_BLOCKS_PER_SM * D->sms), TPB, 0, (cudaStream_t)stream>>>(
      d_X, n, d_params, d_logits);
  return cudaGetLastError() == cudaSuccess ? GKS2L_OK : GKS2L_ECUDA;
}
