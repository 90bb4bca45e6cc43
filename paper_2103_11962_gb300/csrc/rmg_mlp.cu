// Learned prolongator: a small MLP that maps a fine node's local operator to its interpolation
// weights, with hand-written training and inference kernels.
//
// Network: 27 features (padded to 32) -> 64 -> 64 -> 3, ReLU, ReLU, sigmoid. The three outputs
// are the weights a fine node takes from its right coarse neighbour along x, y and z (the left
// one gets 1 - w), so every predicted row of P sums to one and constants are preserved.
//
// Forward pass: BF16 tensor-core MMA (mma.sync m16n8k16, FP32 accumulate). Inference: each warp
// takes tiles of 16 samples. Training: a CTA of 16 warps takes 128 samples, a warp 16 rows and half
// of a layer's columns; backward pass on FP32 CUDA cores over the same tile, the weight gradients
// in registers, one atomic add per parameter per CTA. Adam updates FP32 master weights.
//
// Features of fine node n (9 per axis, zero along axes where n sits on a coarse index): for
// the line of three edges between its two coarse neighbours along the axis, log10 of the three
// composite conductances -A(p_e, p_e+1) and of the four composite diagonals, each divided by
// the node's own diagonal, then rem/3 and an active flag. Composite values are sums over the
// copies of a node, so co-located copies see the same features and get identical weights.
#include <cuda_bf16.h>

#include <algorithm>
#include <new>
#include <vector>

#include "rmg_hier.cuh"
#include "rmg_kernels.cuh"
#include "rmg_launch.cuh"

namespace rmg {
namespace {

constexpr int NF = 32, NH = 64, NOUT = 3;
constexpr int NPARAMS = NH * NF + NH + NH * NH + NH + NOUT * NH + NOUT;
constexpr int O_W1 = 0, O_B1 = O_W1 + NH * NF, O_W2 = O_B1 + NH, O_B2 = O_W2 + NH * NH,
              O_W3 = O_B2 + NH, O_B3 = O_W3 + NOUT * NH;
constexpr int kRows = 128, kThreads = 256;
constexpr int kGradThreads = 512;                          // k_mlp
// padded shared-memory strides (elements)
constexpr int SX = NF + 8, SH = NH + 8;

// The backward pass reads FP32 rows four values at a time: row strides are multiples of four.
constexpr int SXF = NF + 4, SHF = NH + 4;

struct MlpSmem {
  __nv_bfloat16 Xb[kRows * SX];
  __nv_bfloat16 W1b[NH * SX];
  __nv_bfloat16 H1b[kRows * SH];
  __nv_bfloat16 W2b[NH * SH];
  __nv_bfloat16 H2b[kRows * SH];
  __nv_bfloat16 W3b[8 * SH];
  float Xf[kRows * SXF];                 // the BF16-rounded X and H1 again as FP32
  float H1f[kRows * SHF];
  float W2f[NH * NH];
  float dZ3[kRows * 4];
  float dZ2[kRows * SHF];
  float dZ1[kRows * SHF];
  float W3f[4 * NH];                     // [j][k], row 3 zero
  float O[kRows * 4];
  float Y[kRows * 4];
  float M[kRows * 4];
  long long idx[kRows];                  // sample of every row, -1 past the last one
  float red[kGradThreads / 32];
};

__device__ __forceinline__ uint32_t pack2(const __nv_bfloat16* p) {
  return *reinterpret_cast<const uint32_t*>(p);    // two consecutive bf16 (4-byte aligned)
}

// acc[nt][4] += A[16 x K] * B[K x 8*NT] for one warp. A rows come from row-major bf16 smem
// (row stride lda, first row r0); B is given transposed: Bt[n][k] (row-major, stride ldb),
// which is how the layer weights are stored ([out][in]).
template <int NT, int K>
__device__ __forceinline__ void warp_mma(const __nv_bfloat16* A, int lda, int r0,
                                         const __nv_bfloat16* Bt, int ldb, float (&acc)[NT][4]) {
  const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
#pragma unroll
  for (int k0 = 0; k0 < K; k0 += 16) {
    const uint32_t a0 = pack2(A + (r0 + g) * lda + k0 + 2 * t);
    const uint32_t a1 = pack2(A + (r0 + g + 8) * lda + k0 + 2 * t);
    const uint32_t a2 = pack2(A + (r0 + g) * lda + k0 + 2 * t + 8);
    const uint32_t a3 = pack2(A + (r0 + g + 8) * lda + k0 + 2 * t + 8);
#pragma unroll
    for (int nt = 0; nt < NT; ++nt) {
      const uint32_t b0 = pack2(Bt + (nt * 8 + g) * ldb + k0 + 2 * t);
      const uint32_t b1 = pack2(Bt + (nt * 8 + g) * ldb + k0 + 2 * t + 8);
      asm volatile(
          "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 "
          "{%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};\n"
          : "+f"(acc[nt][0]), "+f"(acc[nt][1]), "+f"(acc[nt][2]), "+f"(acc[nt][3])
          : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
    }
  }
}

__device__ __forceinline__ unsigned long long mix64(unsigned long long z) {
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

__device__ __forceinline__ void red_add4(float* p, float a, float b, float c, float d) {
  asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};\n" ::"l"(p), "f"(a), "f"(b), "f"(c),
               "f"(d) : "memory");
}
__device__ __forceinline__ void red_add2(float* p, float a, float b) {
  asm volatile("red.global.add.v2.f32 [%0], {%1, %2};\n" ::"l"(p), "f"(a), "f"(b) : "memory");
}

// Gradient and loss over rows that are sampled or taken in order, in tiles of 128 samples.
//
// Bound by the FP32 pipe in the backward products (1.3M FMAs a tile). One FMA per two shared
// loads and a set of 6467 atomic adds per tile took 269 us for 65,573 samples; here every
// thread owns blocks of the outputs (4 x 4 of dW2, 4 x 2 of dW1, 4 x 4 of dZ1), loads its
// operands four at a time, and keeps the weight gradients of all its CTA's tiles in registers,
// so the atomic adds run once per CTA, and 16 warps hide each other's shared loads: 70 us (the
// whole call with its copies 313 -> 99 us; 105 with eight warps).
__global__ void __launch_bounds__(kGradThreads, 1)
k_mlp(const float* __restrict__ params, int n, long long ntiles, const float* __restrict__ feats,
      const float* __restrict__ labels, const float* __restrict__ mask, int sample,
      unsigned long long seed, float inv_norm, float* __restrict__ grads,
      float* __restrict__ loss) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  MlpSmem& S = *reinterpret_cast<MlpSmem*>(smem_raw);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int g = lane >> 2, t = lane & 3;

  // ---- stage weights (bf16 copies for the MMA, fp32 copies for the backward pass)
  for (int e = tid; e < NH * NF; e += kGradThreads)
    S.W1b[(e / NF) * SX + e % NF] = __float2bfloat16_rn(params[O_W1 + e]);
  for (int e = tid; e < NH * NH; e += kGradThreads) {
    const float w = params[O_W2 + e];
    S.W2b[(e / NH) * SH + e % NH] = __float2bfloat16_rn(w);
    S.W2f[e] = w;
  }
  for (int e = tid; e < 8 * NH; e += kGradThreads) {
    const int j = e / NH, k = e % NH;
    const float w = j < NOUT ? params[O_W3 + j * NH + k] : 0.f;
    S.W3b[j * SH + k] = __float2bfloat16_rn(w);
    if (j < 4) S.W3f[j * NH + k] = w;
  }
  // this thread's share of the gradients: over the rows of its half (64 rows from rh)
  // dW2[4 mg..][4 kg..] and dW1[4 mg..][2 kg..], over 16 rows column kq of dW3, db2 and db1
  const int rh = 64 * (tid >> 8), mg = (tid & 255) >> 4, kg = tid & 15;
  const int rq = 16 * (tid >> 6), kq = tid & 63;
  float gw2[4][4] = {}, gw1[4][2] = {}, gw3[NOUT] = {}, gb3 = 0.f, gb2 = 0.f, gb1 = 0.f;
  float lsum = 0.f;
  // persistent loop over tiles of 128 samples; the weights above are staged once per CTA
  for (long long tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
  const long long base = tile * kRows;
  __syncthreads();
  if (tid < kRows) {
    long long i = base + tid;
    if (sample)
      i = (long long)(mix64(seed + 0x9E3779B97F4A7C15ull * (unsigned long long)(i + 1)) %
                      (unsigned long long)n);
    else if (i >= n)
      i = -1;
    S.idx[tid] = i;
  }
  __syncthreads();
  // ---- stage the samples
  for (int e = tid; e < kRows * NF; e += kGradThreads) {
    const int r = e / NF, k = e % NF;
    const long long i = S.idx[r];
    const __nv_bfloat16 v = __float2bfloat16_rn(i >= 0 ? feats[i * NF + k] : 0.f);
    S.Xb[r * SX + k] = v;
    S.Xf[r * SXF + k] = __bfloat162float(v);
  }
  for (int e = tid; e < kRows * NOUT; e += kGradThreads) {
    const int r = e / NOUT, j = e % NOUT;
    const long long i = S.idx[r];
    S.Y[r * 4 + j] = i >= 0 ? labels[i * NOUT + j] : 0.f;
    S.M[r * 4 + j] = i >= 0 ? mask[i * NOUT + j] : 0.f;
  }
  __syncthreads();

  const int r0 = (warp & 7) * 16, c0 = 32 * (warp >> 3);   // rows and columns of the warp
  // ---- layer 1: H1 = relu(X W1^T + b1)
  {
    float acc[4][4] = {};
    warp_mma<4, NF>(S.Xb, SX, r0, S.W1b + c0 * SX, SX, acc);
#pragma unroll
    for (int nt = 0; nt < 4; ++nt) {
      const int c = c0 + nt * 8 + 2 * t;
      const float b0 = params[O_B1 + c], b1 = params[O_B1 + c + 1];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int r = r0 + g + 8 * h;
        const __nv_bfloat16 v0 = __float2bfloat16_rn(fmaxf(acc[nt][2 * h] + b0, 0.f));
        const __nv_bfloat16 v1 = __float2bfloat16_rn(fmaxf(acc[nt][2 * h + 1] + b1, 0.f));
        S.H1b[r * SH + c] = v0;
        S.H1b[r * SH + c + 1] = v1;
        *reinterpret_cast<float2*>(&S.H1f[r * SHF + c]) =
            make_float2(__bfloat162float(v0), __bfloat162float(v1));
      }
    }
  }
  __syncthreads();
  // ---- layer 2: H2 = relu(H1 W2^T + b2)
  {
    float acc[4][4] = {};
    warp_mma<4, NH>(S.H1b, SH, r0, S.W2b + c0 * SH, SH, acc);
#pragma unroll
    for (int nt = 0; nt < 4; ++nt) {
      const int c = c0 + nt * 8 + 2 * t;
      const float b0 = params[O_B2 + c], b1 = params[O_B2 + c + 1];
      S.H2b[(r0 + g) * SH + c] = __float2bfloat16_rn(fmaxf(acc[nt][0] + b0, 0.f));
      S.H2b[(r0 + g) * SH + c + 1] = __float2bfloat16_rn(fmaxf(acc[nt][1] + b1, 0.f));
      S.H2b[(r0 + g + 8) * SH + c] = __float2bfloat16_rn(fmaxf(acc[nt][2] + b0, 0.f));
      S.H2b[(r0 + g + 8) * SH + c + 1] = __float2bfloat16_rn(fmaxf(acc[nt][3] + b1, 0.f));
    }
  }
  __syncthreads();
  // ---- layer 3: O = sigmoid(H2 W3^T + b3) (8 padded output columns, 3 used)
  if (warp < 8) {
    float acc[1][4] = {};
    warp_mma<1, NH>(S.H2b, SH, r0, S.W3b, SH, acc);
    const int c = 2 * t;
    const float zz[4] = {acc[0][0], acc[0][1], acc[0][2], acc[0][3]};
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int row = r0 + g + (q >= 2 ? 8 : 0), col = c + (q & 1);
      if (col < NOUT) {
        const float z = zz[q] + params[O_B3 + col];
        S.O[row * 4 + col] = 1.f / (1.f + __expf(-z));
      }
    }
  }
  __syncthreads();

  // ---- backward (FP32)
  for (int e = tid; e < kRows * NOUT; e += kGradThreads) {
    const int r = e / NOUT, j = e % NOUT;
    const float o = S.O[r * 4 + j], m = S.M[r * 4 + j], d = o - S.Y[r * 4 + j];
    lsum += m * d * d;
    S.dZ3[r * 4 + j] = 2.f * m * d * inv_norm * o * (1.f - o);
  }
  __syncthreads();
  // dZ2 = (dZ3 W3) * [H2 > 0], and column kq of dW3, db2 over 16 rows
  {
    const float w0 = S.W3f[kq], w1 = S.W3f[NH + kq], w2 = S.W3f[2 * NH + kq];
#pragma unroll 4
    for (int r = rq; r < rq + 16; ++r) {
      const float d0 = S.dZ3[r * 4], d1 = S.dZ3[r * 4 + 1], d2 = S.dZ3[r * 4 + 2];
      const float h = __bfloat162float(S.H2b[r * SH + kq]);
      gw3[0] = fmaf(d0, h, gw3[0]);
      gw3[1] = fmaf(d1, h, gw3[1]);
      gw3[2] = fmaf(d2, h, gw3[2]);
      const float z = h > 0.f ? fmaf(d2, w2, fmaf(d1, w1, d0 * w0)) : 0.f;
      S.dZ2[r * SHF + kq] = z;
      gb2 += z;
    }
    if (kq < NOUT)
      for (int r = rq; r < rq + 16; ++r) gb3 += S.dZ3[r * 4 + kq];
  }
  __syncthreads();
  // dW2 += dZ2^T H1
#pragma unroll 4
  for (int r = rh; r < rh + 64; ++r) {
    const float4 z = *reinterpret_cast<const float4*>(&S.dZ2[r * SHF + 4 * mg]);
    const float4 h = *reinterpret_cast<const float4*>(&S.H1f[r * SHF + 4 * kg]);
    const float zv[4] = {z.x, z.y, z.z, z.w}, hv[4] = {h.x, h.y, h.z, h.w};
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
      for (int b = 0; b < 4; ++b) gw2[a][b] = fmaf(zv[a], hv[b], gw2[a][b]);
  }
  // dZ1 = (dZ2 W2) * [H1 > 0]: rows r4 .. r4 + 3, columns 4 kg ..
  {
    const int r4 = 4 * (tid >> 4);
    float acc[4][4] = {};
#pragma unroll 2
    for (int m = 0; m < NH; m += 4) {
      float4 w[4];
#pragma unroll
      for (int q = 0; q < 4; ++q)
        w[q] = *reinterpret_cast<const float4*>(&S.W2f[(m + q) * NH + 4 * kg]);
#pragma unroll
      for (int a = 0; a < 4; ++a) {
        const float4 z = *reinterpret_cast<const float4*>(&S.dZ2[(r4 + a) * SHF + m]);
        const float zv[4] = {z.x, z.y, z.z, z.w};
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          acc[a][0] = fmaf(zv[q], w[q].x, acc[a][0]);
          acc[a][1] = fmaf(zv[q], w[q].y, acc[a][1]);
          acc[a][2] = fmaf(zv[q], w[q].z, acc[a][2]);
          acc[a][3] = fmaf(zv[q], w[q].w, acc[a][3]);
        }
      }
    }
#pragma unroll
    for (int a = 0; a < 4; ++a) {
      const int at = (r4 + a) * SHF + 4 * kg;
      const float4 h = *reinterpret_cast<const float4*>(&S.H1f[at]);
      *reinterpret_cast<float4*>(&S.dZ1[at]) =
          make_float4(h.x > 0.f ? acc[a][0] : 0.f, h.y > 0.f ? acc[a][1] : 0.f,
                      h.z > 0.f ? acc[a][2] : 0.f, h.w > 0.f ? acc[a][3] : 0.f);
    }
  }
  __syncthreads();
  // dW1 += dZ1^T X, db1
#pragma unroll 4
  for (int r = rh; r < rh + 64; ++r) {
    const float4 z = *reinterpret_cast<const float4*>(&S.dZ1[r * SHF + 4 * mg]);
    const float2 x = *reinterpret_cast<const float2*>(&S.Xf[r * SXF + 2 * kg]);
    const float zv[4] = {z.x, z.y, z.z, z.w};
#pragma unroll
    for (int a = 0; a < 4; ++a) {
      gw1[a][0] = fmaf(zv[a], x.x, gw1[a][0]);
      gw1[a][1] = fmaf(zv[a], x.y, gw1[a][1]);
    }
  }
#pragma unroll 4
  for (int r = rq; r < rq + 16; ++r) gb1 += S.dZ1[r * SHF + kq];
  }  // tiles

  // ---- this CTA's sums
#pragma unroll
  for (int a = 0; a < 4; ++a) {
    red_add4(&grads[O_W2 + (4 * mg + a) * NH + 4 * kg], gw2[a][0], gw2[a][1], gw2[a][2],
             gw2[a][3]);
    red_add2(&grads[O_W1 + (4 * mg + a) * NF + 2 * kg], gw1[a][0], gw1[a][1]);
  }
#pragma unroll
  for (int j = 0; j < NOUT; ++j) atomicAdd(&grads[O_W3 + j * NH + kq], gw3[j]);
  atomicAdd(&grads[O_B2 + kq], gb2);
  atomicAdd(&grads[O_B1 + kq], gb1);
  if (kq < NOUT) atomicAdd(&grads[O_B3 + kq], gb3);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) lsum += __shfl_xor_sync(0xffffffffu, lsum, o);
  if (lane == 0) S.red[warp] = lsum;
  __syncthreads();
  if (tid == 0) {
    float sum = 0.f;
    for (int w = 0; w < kGradThreads / 32; ++w) sum += S.red[w];
    atomicAdd(loss, sum * inv_norm);
  }
}

// Inference: the forward pass of k_mlp (same BF16 roundings, same MMA sequence, same
// epilogues, so the same outputs) with each warp working through its own tiles of 16 samples.
// Without the backward buffers a block needs 44 KB of shared memory instead of k_mlp's, so
// more blocks share an SM, and no block-wide barrier stands between a warp's tiles.
constexpr int kWarpRows = 16;
struct MlpInferSmem {
  __nv_bfloat16 W1b[NH * SX];
  __nv_bfloat16 W2b[NH * SH];
  __nv_bfloat16 W3b[8 * SH];
  __nv_bfloat16 Xb[kThreads / 32][kWarpRows * SX];
  __nv_bfloat16 Hb[kThreads / 32][kWarpRows * SH];  // layer-1 output, then layer 2's in place
};

__global__ void __launch_bounds__(kThreads)
k_mlp_infer(const float* __restrict__ params, int n, const float* __restrict__ feats,
            float* __restrict__ out) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  MlpInferSmem& S = *reinterpret_cast<MlpInferSmem*>(smem_raw);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int g = lane >> 2, t = lane & 3;
  for (int e = tid; e < NH * NF; e += kThreads)
    S.W1b[(e / NF) * SX + e % NF] = __float2bfloat16_rn(params[O_W1 + e]);
  for (int e = tid; e < NH * NH; e += kThreads)
    S.W2b[(e / NH) * SH + e % NH] = __float2bfloat16_rn(params[O_W2 + e]);
  for (int e = tid; e < 8 * NH; e += kThreads) {
    const int j = e / NH, k = e % NH;
    S.W3b[j * SH + k] = __float2bfloat16_rn(j < NOUT ? params[O_W3 + j * NH + k] : 0.f);
  }
  __syncthreads();
  __nv_bfloat16* X = S.Xb[warp];
  __nv_bfloat16* H = S.Hb[warp];
  const long long tiles = ((long long)n + kWarpRows - 1) / kWarpRows;
  for (long long tile = (long long)blockIdx.x * (kThreads / 32) + warp; tile < tiles;
       tile += (long long)gridDim.x * (kThreads / 32)) {
    const long long base = tile * kWarpRows;
    __syncwarp();                                  // the previous tile's reads are done
    for (int e = lane; e < kWarpRows * NF; e += 32) {
      const int r = e / NF, k = e % NF;
      const long long i = base + r;
      X[r * SX + k] = __float2bfloat16_rn(i < n ? feats[i * NF + k] : 0.f);
    }
    __syncwarp();
    {
      float acc[8][4] = {};
      warp_mma<8, NF>(X, SX, 0, S.W1b, SX, acc);
#pragma unroll
      for (int nt = 0; nt < 8; ++nt) {
        const int c = nt * 8 + 2 * t;
        const float b0 = params[O_B1 + c], b1 = params[O_B1 + c + 1];
        H[g * SH + c] = __float2bfloat16_rn(fmaxf(acc[nt][0] + b0, 0.f));
        H[g * SH + c + 1] = __float2bfloat16_rn(fmaxf(acc[nt][1] + b1, 0.f));
        H[(g + 8) * SH + c] = __float2bfloat16_rn(fmaxf(acc[nt][2] + b0, 0.f));
        H[(g + 8) * SH + c + 1] = __float2bfloat16_rn(fmaxf(acc[nt][3] + b1, 0.f));
      }
    }
    __syncwarp();
    {
      float acc[8][4] = {};
      warp_mma<8, NH>(H, SH, 0, S.W2b, SH, acc);
      __syncwarp();                                // layer 1's values are all read
#pragma unroll
      for (int nt = 0; nt < 8; ++nt) {
        const int c = nt * 8 + 2 * t;
        const float b0 = params[O_B2 + c], b1 = params[O_B2 + c + 1];
        H[g * SH + c] = __float2bfloat16_rn(fmaxf(acc[nt][0] + b0, 0.f));
        H[g * SH + c + 1] = __float2bfloat16_rn(fmaxf(acc[nt][1] + b1, 0.f));
        H[(g + 8) * SH + c] = __float2bfloat16_rn(fmaxf(acc[nt][2] + b0, 0.f));
        H[(g + 8) * SH + c + 1] = __float2bfloat16_rn(fmaxf(acc[nt][3] + b1, 0.f));
      }
    }
    __syncwarp();
    {
      float acc[1][4] = {};
      warp_mma<1, NH>(H, SH, 0, S.W3b, SH, acc);
      const int c = 2 * t;
      const float zz[4] = {acc[0][0], acc[0][1], acc[0][2], acc[0][3]};
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int row = g + (q >= 2 ? 8 : 0), col = c + (q & 1);
        const long long i = base + row;
        if (col < NOUT && i < n) {
          const float z = zz[q] + params[O_B3 + col];
          out[i * NOUT + col] = 1.f / (1.f + __expf(-z));
        }
      }
    }
  }
}

__global__ void k_adam(int np, float* __restrict__ p, const float* __restrict__ gr,
                       float* __restrict__ m, float* __restrict__ v, float lr, float b1, float b2,
                       float eps, float c1, float c2) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < np; i += gridDim.x * blockDim.x) {
    const float gg = gr[i];
    const float mi = b1 * m[i] + (1.f - b1) * gg;
    const float vi = b2 * v[i] + (1.f - b2) * gg * gg;
    m[i] = mi;
    v[i] = vi;
    p[i] -= lr * (mi * c1) / (sqrtf(vi * c2) + eps);
  }
}

// What the features read of a level: the region stencils and, for nodes with several copies, the
// composite couplings in comp[0..3] (centre, +x, +y, +z; written at the shared nodes only).
struct FeatArgs {
  const double* coef;
  const uint8_t* mult;
  double* comp[4];
};

// Composite coupling number p (0: centre, 1..3: +x, +y, +z) of stencil KIND, or -1.
template <int KIND>
__device__ __forceinline__ int feature_slot(int p) {
  return p == 0 ? Sten<KIND>::CENTER : sten_slot<KIND>(p == 1, p == 2, p == 3);
}

// The composite couplings of the shared nodes, one thread per copy: sums over the copies in
// ascending slot order.
template <int KIND>
__global__ void __launch_bounds__(256)
k_shared_couplings(int nslots, int n_r, const int* __restrict__ sgrp,
                   const int* __restrict__ gptr, const int* __restrict__ gslot, FeatArgs A) {
  for (int q = blockIdx.x * blockDim.x + threadIdx.x; q < nslots; q += gridDim.x * blockDim.x) {
    const int grp = sgrp[q], n = gslot[q], a = gptr[grp], e = gptr[grp + 1];
    double s[4] = {};
    for (int k = a; k < e; ++k)
#pragma unroll
      for (int p = 0; p <= Sten<KIND>::DIM; ++p)
        s[p] += A.coef[(size_t)feature_slot<KIND>(p) * n_r + gslot[k]];
#pragma unroll
    for (int p = 0; p <= Sten<KIND>::DIM; ++p) A.comp[p][n] = s[p];
  }
}

// The 27 features of regional node n (layout described at the top of the file) and zeros up to
// NF. Nearly every warp holds a few nodes of an interface: the copies' couplings come from
// k_shared_couplings, so that reading a shared node is one load from another array and the warp
// does not wait for a walk over the copies at each of the 21 values (that walk inside the
// one-pass kernel took it to 1244 us, slower than the three kernels it replaced).
template <int KIND>
__device__ __forceinline__ void node_features(const Grid& G, const FeatArgs& A, const RegionDev& R,
                                              int n, int li, float (&f)[NF]) {
  using St = Sten<KIND>;
  int x[3];
  decode(li, R, x[0], x[1], x[2]);
  const int stride[3] = {1, R.nx, R.nx * R.ny};
  const int len[3] = {R.nx, R.ny, R.nz};
  auto coupling = [&](int p, int m, bool single) {
    return single ? A.coef[(size_t)feature_slot<KIND>(p) * G.n_r + m] : A.comp[p][m];
  };
  const double dn = coupling(0, n, A.mult[n] == 1);
  const double dref = dn > 0.0 ? dn : 1.0;
  const double inv_ref = 1.0 / dref;            // one FP64 division per node, not 21
#pragma unroll
  for (int q = 0; q < NF; ++q) f[q] = 0.f;
#pragma unroll
  for (int a = 0; a < St::DIM; ++a) {
    int rem = x[a] % 3;
    if (rem && x[a] - rem + 3 > len[a] - 1) rem = 0;   // no right coarse node in the region
    if (!rem) continue;
    const int p0 = n - rem * stride[a];
    double k[3], d[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int m = p0 + i * stride[a];
      const bool single = A.mult[m] == 1;
      if (i < 3) k[i] = coupling(a + 1, m, single);
      d[i] = coupling(0, m, single);
    }
    // ratios in FP64, logarithms in FP32 (the features are FP32 network inputs)
#pragma unroll
    for (int e = 0; e < 3; ++e)
      f[9 * a + e] = fminf(log10f(fmaxf((float)(-k[e] * inv_ref), 1e-12f)), 2.f);
#pragma unroll
    for (int i = 0; i < 4; ++i)
      f[9 * a + 3 + i] = fminf(log10f(fmaxf((float)(d[i] * inv_ref), 1e-12f)), 12.f);
    f[9 * a + 7] = rem == 1 ? (float)(1.0 / 3.0) : (float)(2.0 / 3.0);
    f[9 * a + 8] = 1.f;
  }
}

// Features of every regional node of a level, one 128-byte row per node (16-byte stores when the
// caller's array allows them).
template <int KIND>
__global__ void __launch_bounds__(kTile)
k_features(Grid G, FeatArgs A, float* __restrict__ feats) {
  const bool aligned = (reinterpret_cast<uintptr_t>(feats) & 15) == 0;
  RMG_FOR_NODES(G)
    float f[NF];
    node_features<KIND>(G, A, R, n, li, f);
    if (!aligned) {
#pragma unroll
      for (int q = 0; q < NF; ++q) feats[(size_t)n * NF + q] = f[q];
      continue;
    }
    float4* row = reinterpret_cast<float4*>(feats + (size_t)n * NF);
#pragma unroll
    for (int q = 0; q < NF / 4; ++q)
      row[q] = make_float4(f[4 * q], f[4 * q + 1], f[4 * q + 2], f[4 * q + 3]);
  RMG_END_FOR_NODES
}

// Interpolation weights of a level in one pass: features, network and weights of 32 consecutive
// nodes at a time per warp, the features going to the MMA through shared memory (the BF16 rows
// of k_mlp_infer, the same operations in the same order). Nothing but the coefficients is read
// and nothing but the weights written; as three kernels the features (128 bytes a node) went
// through memory with 4-byte stores 128 bytes apart, and that was most of the time: 939 us for
// 2.54M nodes of a 7-point level, 300 us in this form. The FP64 pipe bounds it now (a product
// and a conversion per ratio, about 28 ratios a node, and one division).
struct WeightsSmem {
  __nv_bfloat16 W1b[NH * SX];
  __nv_bfloat16 W2b[NH * SH];
  __nv_bfloat16 W3b[8 * SH];
  __nv_bfloat16 Xb[kTile / 32][32 * SX];
  __nv_bfloat16 Hb[kTile / 32][16 * SH];   // layer-1 output of 16 nodes, then layer 2's in place
};

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
  const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&v);
}

// H = relu(acc + bias) as BF16 rows g and g + 8 of a 16-row tile.
__device__ __forceinline__ void store_relu(__nv_bfloat16* H, const float (&acc)[8][4],
                                           const float* __restrict__ bias, int g, int t) {
#pragma unroll
  for (int nt = 0; nt < 8; ++nt) {
    const int c = nt * 8 + 2 * t;
    const float b0 = bias[c], b1 = bias[c + 1];
    *reinterpret_cast<uint32_t*>(&H[g * SH + c]) =
        pack_bf16(fmaxf(acc[nt][0] + b0, 0.f), fmaxf(acc[nt][1] + b1, 0.f));
    *reinterpret_cast<uint32_t*>(&H[(g + 8) * SH + c]) =
        pack_bf16(fmaxf(acc[nt][2] + b0, 0.f), fmaxf(acc[nt][3] + b1, 0.f));
  }
}

template <int KIND>
__global__ void __launch_bounds__(kTile)
k_learned_weights(Grid G, FeatArgs A, const float* __restrict__ params, float* __restrict__ wr) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  WeightsSmem& S = *reinterpret_cast<WeightsSmem*>(smem_raw);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int g = lane >> 2, t = lane & 3;
  for (int e = tid; e < NH * NF; e += kTile)
    S.W1b[(e / NF) * SX + e % NF] = __float2bfloat16_rn(params[O_W1 + e]);
  for (int e = tid; e < NH * NH; e += kTile)
    S.W2b[(e / NH) * SH + e % NH] = __float2bfloat16_rn(params[O_W2 + e]);
  for (int e = tid; e < 8 * NH; e += kTile) {
    const int j = e / NH, k = e % NH;
    S.W3b[j * SH + k] = __float2bfloat16_rn(j < NOUT ? params[O_W3 + j * NH + k] : 0.f);
  }
  __syncthreads();
  __nv_bfloat16* X = S.Xb[warp];
  __nv_bfloat16* H = S.Hb[warp];
  for (int ti = blockIdx.x; ti < G.ntiles; ti += gridDim.x) {
    const Tile tile = G.tiles[ti];
    const RegionDev R = G.regions[tile.region];
    const int l0 = tile.start + warp * 32;             // first node of the warp in the region
    const int nodes = min(32, R.nx * R.ny * R.nz - l0);
    if (nodes <= 0) continue;
    float f[NF];
    if (lane < nodes) {
      node_features<KIND>(G, A, R, R.off + l0 + lane, l0 + lane, f);
    } else {
#pragma unroll
      for (int q = 0; q < NF; ++q) f[q] = 0.f;
    }
    __syncwarp();                                      // the previous tile's reads are done
    uint4* row = reinterpret_cast<uint4*>(&X[lane * SX]);
#pragma unroll
    for (int q = 0; q < NF / 8; ++q)
      row[q] = make_uint4(pack_bf16(f[8 * q], f[8 * q + 1]), pack_bf16(f[8 * q + 2], f[8 * q + 3]),
                          pack_bf16(f[8 * q + 4], f[8 * q + 5]),
                          pack_bf16(f[8 * q + 6], f[8 * q + 7]));
    __syncwarp();
    for (int r0 = 0; r0 < nodes; r0 += 16) {
      {
        float acc[8][4] = {};
        warp_mma<8, NF>(X, SX, r0, S.W1b, SX, acc);
        __syncwarp();                                  // the last 16 nodes' layer 2 is read
        store_relu(H, acc, params + O_B1, g, t);
      }
      __syncwarp();
      {
        float acc[8][4] = {};
        warp_mma<8, NH>(H, SH, 0, S.W2b, SH, acc);
        __syncwarp();                                  // layer 1's values are all read
        store_relu(H, acc, params + O_B2, g, t);
      }
      __syncwarp();
      float acc[1][4] = {};
      warp_mma<1, NH>(H, SH, 0, S.W3b, SH, acc);
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int i = r0 + g + (q >= 2 ? 8 : 0), col = 2 * t + (q & 1);
        if (col >= NOUT || i >= nodes) continue;
        const float z = acc[0][q] + params[O_B3 + col];
        const bool active = __bfloat162float(X[i * SX + 9 * col + 8]) > 0.5f;
        wr[(size_t)col * G.n_r + R.off + l0 + i] = active ? 1.f / (1.f + __expf(-z)) : 0.f;
      }
    }
  }
}

}  // namespace
}  // namespace rmg

using namespace rmg;

struct rmg_mlp {
  rmg_ctx* ctx = nullptr;
  DBuf<float> p, g, m, v, loss;
  int steps_done = 0;
};

namespace {
template <class F>
rmg_status mlp_guard(rmg_ctx* ctx, F&& f) {
  if (!ctx) return RMG_ERR_ARG;
  try {
    RMG_CUDA(cudaSetDevice(ctx->c.device));
    f();
    ctx->c.last_error.clear();
    return RMG_OK;
  } catch (const Error& e) {
    ctx->c.last_error = e.what();
    return e.status;
  } catch (const std::exception& e) {
    ctx->c.last_error = e.what();
    return RMG_ERR_CUDA;
  }
}

void mlp_infer(rmg_mlp* net, int n, const float* feats, float* out) {
  Ctx& c = net->ctx->c;
  const int smem = (int)sizeof(MlpInferSmem);
  RMG_CUDA(cudaFuncSetAttribute(k_mlp_infer, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
  int per_sm = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_mlp_infer, kThreads, smem) !=
      cudaSuccess) {
    cudaGetLastError();
    per_sm = 1;
  }
  const long long warps = ((long long)n + kWarpRows - 1) / kWarpRows;
  const long long want = (warps + kThreads / 32 - 1) / (kThreads / 32);
  const int blocks = (int)std::max<long long>(
      1, std::min<long long>(want, (long long)c.nsm * std::max(1, per_sm)));
  k_mlp_infer<<<blocks, kThreads, smem, c.stream>>>(net->p.get(), n, feats, out);
  RMG_LAUNCHED();
}

// Gradient (into net->g) and loss over `rows` rows. The shared memory of k_mlp leaves one CTA
// per SM, so one CTA per SM strides over the tiles.
void mlp_backward(rmg_mlp* net, int n, const float* feats, const float* labels, const float* mask,
                  int sample, int rows, unsigned long long seed, float inv_norm, float* loss) {
  Ctx& c = net->ctx->c;
  const int smem = (int)sizeof(MlpSmem);
  RMG_CUDA(cudaFuncSetAttribute(k_mlp, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
  const long long tiles = ((long long)rows + kRows - 1) / kRows;
  const int blocks = (int)std::min<long long>(tiles, (long long)c.nsm);
  k_mlp<<<blocks, kGradThreads, smem, c.stream>>>(net->p.get(), n, tiles, feats, labels, mask, sample,
                                             seed, inv_norm, net->g.get(), loss);
  RMG_LAUNCHED();
}

// Room for the couplings of the level's shared nodes in the PCG work vectors: calls that use those
// synchronise before they return, so that nothing of theirs is in flight on any stream (a cycle's
// own vectors may be: rmg_vcycle_apply returns once queued). Every level has a place of its own,
// so that features of different levels may be formed on different streams. The finest level takes
// four whole vectors; DIM + 1 arrays of each of the others fit one (3D: level l + 1 has at most an
// eighth of the nodes of level l, and 4 (1/8 + 1/64 + ..) < 1; 2D: 3 (1/4 + 1/16 + ..) < 1).
template <int KIND>
FeatArgs feat_args(const Hier& h, int level) {
  const Level& L = *h.lv[level];
  FeatArgs A{L.coef.get(), L.mult.get(), {h.x.get(), h.p.get(), h.q.get(), h.tmp.get()}};
  if (level > 0) {
    double* at = h.zold.get();
    for (int l = 1; l < level; ++l) at += (size_t)(L.dim + 1) * h.lv[l]->n_r;
    for (int p = 0; p < 4; ++p) A.comp[p] = at + (size_t)std::min(p, L.dim) * L.n_r;
  }
  if (L.nslots) {
    k_shared_couplings<KIND><<<persistent_grid(*h.c, (L.nslots + 255) / 256), 256, 0,
                               h.c->stream>>>(L.nslots, L.n_r, L.sgrp.get(), L.gptr.get(),
                                              L.gslot.get(), A);
    RMG_LAUNCHED();
  }
  return A;
}

template <int KIND>
void learned_weights(const rmg_mlp& net, const Hier& h, int level, float* wr) {
  const Ctx& c = *h.c;
  const Level& L = *h.lv[level];
  const FeatArgs A = feat_args<KIND>(h, level);
  const Grid G = L.grid();
  const int smem = (int)sizeof(WeightsSmem);
  const int per_sm = resident_per_sm_smem((const void*)k_learned_weights<KIND>, smem);
  k_learned_weights<KIND><<<persistent_grid(c, G.ntiles, per_sm), kTile, smem, c.stream>>>(
      G, A, net.p.get(), wr);
  RMG_LAUNCHED();
}
}  // namespace

extern "C" {

int rmg_mlp_num_params(void) { return NPARAMS; }

rmg_status rmg_mlp_create(rmg_ctx* ctx, const float* init_params, rmg_mlp** out) {
  if (!out) return RMG_ERR_ARG;
  *out = nullptr;
  rmg_mlp* net = new (std::nothrow) rmg_mlp();
  if (!net) return RMG_ERR_NOMEM;
  net->ctx = ctx;
  rmg_status st = mlp_guard(ctx, [&] {
    RMG_REQUIRE(init_params, RMG_ERR_ARG, "init_params is NULL");
    net->p.alloc(NPARAMS); net->g.alloc(NPARAMS + 1); net->m.alloc(NPARAMS); net->v.alloc(NPARAMS);
    RMG_CUDA(cudaMemcpy(net->p.get(), init_params, NPARAMS * sizeof(float), cudaMemcpyHostToDevice));
    RMG_CUDA(cudaMemset(net->m.get(), 0, NPARAMS * sizeof(float)));
    RMG_CUDA(cudaMemset(net->v.get(), 0, NPARAMS * sizeof(float)));
  });
  if (st != RMG_OK) {
    delete net;
    return st;
  }
  *out = net;
  return RMG_OK;
}

void rmg_mlp_destroy(rmg_mlp* net) { delete net; }

rmg_status rmg_mlp_get_params(rmg_mlp* net, float* params) {
  if (!net || !params) return RMG_ERR_ARG;
  return mlp_guard(net->ctx, [&] {
    RMG_CUDA(cudaStreamSynchronize(net->ctx->c.stream));
    RMG_CUDA(cudaMemcpy(params, net->p.get(), NPARAMS * sizeof(float), cudaMemcpyDeviceToHost));
  });
}

rmg_status rmg_mlp_forward(rmg_mlp* net, int n, const float* feats, float* out) {
  if (!net) return RMG_ERR_ARG;
  return mlp_guard(net->ctx, [&] {
    RMG_REQUIRE(n > 0 && feats && out, RMG_ERR_ARG, "bad arguments");
    mlp_infer(net, n, feats, out);
  });
}

rmg_status rmg_mlp_gradient(rmg_mlp* net, int n, const float* feats, const float* labels,
                            const float* mask, float* grad, float* loss) {
  if (!net) return RMG_ERR_ARG;
  return mlp_guard(net->ctx, [&] {
    RMG_REQUIRE(n > 0 && feats && labels && mask && grad && loss, RMG_ERR_ARG, "bad arguments");
    Ctx& c = net->ctx->c;
    // gradient and loss side by side (g has room for both): one memset and one copy back
    RMG_CUDA(cudaMemsetAsync(net->g.get(), 0, (NPARAMS + 1) * sizeof(float), c.stream));
    mlp_backward(net, n, feats, labels, mask, 0, n, 0, 1.f / (3.f * n), net->g.get() + NPARAMS);
    std::vector<float> host(NPARAMS + 1);
    RMG_CUDA(cudaMemcpyAsync(host.data(), net->g.get(), (NPARAMS + 1) * sizeof(float),
                             cudaMemcpyDeviceToHost, c.stream));
    RMG_CUDA(cudaStreamSynchronize(c.stream));
    std::copy(host.begin(), host.begin() + NPARAMS, grad);
    *loss = host[NPARAMS];
  });
}

rmg_status rmg_mlp_train(rmg_mlp* net, int n, const float* feats, const float* labels,
                         const float* mask, int steps, int batch, float lr,
                         unsigned long long seed, float* loss_history) {
  if (!net) return RMG_ERR_ARG;
  return mlp_guard(net->ctx, [&] {
    RMG_REQUIRE(n > 0 && feats && labels && mask && steps > 0, RMG_ERR_ARG, "bad arguments");
    RMG_REQUIRE(batch >= kRows && batch % kRows == 0, RMG_ERR_ARG, "batch must be a multiple of 128");
    Ctx& c = net->ctx->c;
    net->loss.ensure((size_t)steps);
    RMG_CUDA(cudaMemsetAsync(net->loss.get(), 0, sizeof(float) * steps, c.stream));
    const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
    for (int s = 0; s < steps; ++s) {
      RMG_CUDA(cudaMemsetAsync(net->g.get(), 0, NPARAMS * sizeof(float), c.stream));
      mlp_backward(net, n, feats, labels, mask, 1, batch,
                   seed * 0x100000001B3ull + (unsigned long long)(net->steps_done + s) * batch,
                   1.f / (3.f * batch), net->loss.get() + s);
      const int t = net->steps_done + s + 1;
      const float c1 = 1.f / (1.f - powf(b1, (float)t)), c2 = 1.f / (1.f - powf(b2, (float)t));
      k_adam<<<(NPARAMS + 255) / 256, 256, 0, c.stream>>>(NPARAMS, net->p.get(), net->g.get(),
                                                         net->m.get(), net->v.get(), lr, b1, b2,
                                                         eps, c1, c2);
      RMG_LAUNCHED();
    }
    net->steps_done += steps;
    RMG_CUDA(cudaStreamSynchronize(c.stream));
    if (loss_history)
      RMG_CUDA(cudaMemcpy(loss_history, net->loss.get(), sizeof(float) * steps,
                          cudaMemcpyDeviceToHost));
  });
}

rmg_status rmg_hier_mlp_features(rmg_hier* hh, int level, float* feats) {
  if (!hh) return RMG_ERR_ARG;
  return mlp_guard(hh->h.layout->ctx, [&] {
    Hier& h = hh->h;
    RMG_REQUIRE(level >= 0 && level < h.levels() && feats, RMG_ERR_ARG, "bad arguments");
    Level& L = *h.lv[level];
    const Grid G = L.grid();
    const int gb = persistent_grid(*h.c, G.ntiles);
#define RMG_FEAT(K)                                                                            \
  {                                                                                            \
    const FeatArgs A = feat_args<K>(h, level);                                                 \
    k_features<K><<<gb, kTile, 0, h.c->stream>>>(G, A, feats);                                 \
  }
    switch (L.kind) {
      case 5: RMG_FEAT(5); break;
      case 7: RMG_FEAT(7); break;
      case 9: RMG_FEAT(9); break;
      default: RMG_FEAT(27); break;
    }
#undef RMG_FEAT
    RMG_LAUNCHED();
  });
}

rmg_status rmg_hier_mlp_weights(rmg_hier* hh, int level, rmg_mlp* net, float* wr) {
  if (!hh || !net) return RMG_ERR_ARG;
  return mlp_guard(hh->h.layout->ctx, [&] {
    Hier& h = hh->h;
    RMG_REQUIRE(level >= 0 && level < h.levels() && wr, RMG_ERR_ARG, "bad arguments");
    switch (h.lv[level]->kind) {
      case 5: learned_weights<5>(*net, h, level, wr); break;
      case 7: learned_weights<7>(*net, h, level, wr); break;
      case 9: learned_weights<9>(*net, h, level, wr); break;
      default: learned_weights<27>(*net, h, level, wr); break;
    }
  });
}

}  // extern "C"
