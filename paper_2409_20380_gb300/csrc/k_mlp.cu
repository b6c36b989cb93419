// Learned proposal (the learned form of the data-driven predictor of Section 3.2): a 64 -> 256 -> 256 -> 32
// multilayer perceptron with GELU, BF16 weights and activations and FP32 accumulation on the tensor cores,
// forward and backward passes, Adam, and the kernels that tie it to the time step: input features per
// (region, case), the proposal's coefficient correction, the per-case choice between the proposal and the
// plain data-driven guess (smaller initial residual wins), and the collection of training samples.
//
// Parameter layout (FP32 master copy, also the gradient layout): W1 [256][64], b1 [256], W2 [256][256],
// b2 [256], W3 [32][256], b3 [32].  Layer l computes Z_l = A_{l-1} W_l^T + b_l, A_l = GELU(Z_l) (l < 3).
#include <cuda_bf16.h>

#include <cmath>
#include <mutex>
#include <string>

#include "fem_internal.cuh"

using namespace fem;
typedef __nv_bfloat16 bf16;

namespace {

constexpr int kL0 = 64, kL1 = 256, kL2 = 256, kL3 = 32;
// A residual-space sample: the upper triangle of W (row by row) and w, in age order.
constexpr int kNTri = kL3 * (kL3 + 1) / 2;
constexpr int kNRes = kNTri + kL3;
static_assert(kNRes == FEM_MLP_RES, "residual sample size");
constexpr int64_t kOffW1 = 0;
constexpr int64_t kOffB1 = kOffW1 + (int64_t)kL1 * kL0;
constexpr int64_t kOffW2 = kOffB1 + kL1;
constexpr int64_t kOffB2 = kOffW2 + (int64_t)kL2 * kL1;
constexpr int64_t kOffW3 = kOffB2 + kL2;
constexpr int64_t kOffB3 = kOffW3 + (int64_t)kL3 * kL2;
constexpr int64_t kNParams = kOffB3 + kL3;
static_assert(kNParams == 90656, "parameter count of the 64-256-256-32 network");

__device__ __forceinline__ float gelu_f(float z) { return 0.5f * z * (1.0f + erff(z * 0.70710678118654752f)); }
__device__ __forceinline__ float gelu_grad_f(float z) {
  return 0.5f * (1.0f + erff(z * 0.70710678118654752f)) + z * 0.39894228040143268f * expf(-0.5f * z * z);
}

// ------------------------------------------------------------------------------------------------------
// The network on the tensor cores (BF16 mma.sync m16n8k16, FP32 accumulation).  Everything but the weight
// gradients is local to a sample, so one kernel takes a block of kRows samples through the forward pass, the
// loss and the backward pass with the activations in shared memory and the GELU derivatives in registers (a
// thread owns the same entries of a layer on the way forward and back), and a second kernel forms the three
// weight gradients.  What bounds both is latency (2.2 GFLOP a training pass at 4096 samples, ~2 us of tensor
// time), so passes and launches are what is saved: 4096 samples took 246 us in 13 launches (three column sums of
// 60 us on 1 to 8 blocks among them), and take 46 us in 2 launches now (66,560 samples: 3332 -> 330 us; forward
// alone at 4096: 37 -> 10 us).  32 samples a block (128 blocks at 4096) leave the
// tensor cores mostly idle either way; tcgen05's smallest tile (128 rows) would leave 120 of 152 SMs without work.
// Weights come straight from L2 in the order of the MMA's B fragments (k_pack): 16 bytes a lane cover 32 of K
// for 8 output columns, so no shared-memory staging and no barrier between K steps.
// ------------------------------------------------------------------------------------------------------
constexpr int kRows = 32;                      // samples a block (two m16 tiles)
constexpr int kNBias = kL1 + kL2 + kL3;
constexpr int kMlpBlock = 256;                 // 8 warps: 32 of a layer's 256 columns each
constexpr int kSX = kL0 + 8, kSA = kL1 + 8, kSD = kL3 + 8;   // padded rows (16 bytes mod 128: conflict-free ldmatrix)

__device__ __forceinline__ void mma_bf16_16816(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};\n"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void ldsm4(uint32_t (&r)[4], const bf16* p) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"((uint32_t)__cvta_generic_to_shared(p)));
}
__device__ __forceinline__ void ldsm4t(uint32_t (&r)[4], const bf16* p) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"((uint32_t)__cvta_generic_to_shared(p)));
}

// acc[mt][j] = rows 16 mt .. +15 of A (shared, row stride ld) times 8 columns nt0 + j of the packed weights P.
template <int K, int MT, int NT>
__device__ __forceinline__ void layer_mma(const bf16* A, int ld, const uint4* __restrict__ P, int nt0,
                                          float (&acc)[MT][NT][4]) {
  const int lane = threadIdx.x & 31;
  const bf16* a0 = A + (lane & 15) * ld + (lane >> 4) * 8;
#pragma unroll
  for (int m = 0; m < MT; ++m)
#pragma unroll
    for (int j = 0; j < NT; ++j)
#pragma unroll
      for (int e = 0; e < 4; ++e) acc[m][j][e] = 0.0f;
#pragma unroll
  for (int kp = 0; kp < K / 32; ++kp) {
    uint4 b[NT];
#pragma unroll
    for (int j = 0; j < NT; ++j) b[j] = __ldg(P + ((nt0 + j) * (K / 32) + kp) * 32 + lane);
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
      for (int m = 0; m < MT; ++m) {
        uint32_t a[4];
        ldsm4(a, a0 + m * 16 * ld + kp * 32 + h * 16);
#pragma unroll
        for (int j = 0; j < NT; ++j) mma_bf16_16816(acc[m][j], a, h ? b[j].z : b[j].x, h ? b[j].w : b[j].y);
      }
  }
}

struct MlpPass {
  const float* x;          // [n_src][64]
  const int32_t* idx;      // rows of the batch (null: row r is sample r)
  int64_t n_src, B, Mpad;  // samples, rows of the batch, rows of the workspace (multiple of kRows)
  const uint4 *P1, *P2, *P3, *P3T, *P2T;   // packed weights
  const float* th;         // FP32 parameters (biases)
  int* bad;                // set where a sample index is out of range (the row is zero)
  float* out;              // forward only: [B][32]
  const float* t;          // training: [n_src][32] targets, or residual-space samples [n_src][kNRes]
  bf16 *X0, *A1, *A2, *dZ1, *dZ2, *dZ3;    // training: row-major, for the weight gradients
  float* bsum;             // training: [blocks][kNBias] bias gradients of each block's samples (b1, b2, b3)
  double* loss;
};

// entry (mt, j, e) of a thread's accumulators: row 16 mt + gq + 8 (e >> 1), column 32 warp + 8 j + 2 tq + (e & 1)
template <int MODE>   // 0 forward only, 1 training (mean squared error), 2 training (residual space)
__global__ void __launch_bounds__(kMlpBlock) k_mlp_pass(MlpPass g) {
  __shared__ __align__(16) bf16 sX[kRows * kSX];
  __shared__ __align__(16) bf16 sA[kRows * kSA];     // A1, then dZ1
  __shared__ __align__(16) bf16 sB[kRows * kSA];     // A2, then dZ2
  __shared__ __align__(16) bf16 sD[kRows * kSD];     // dZ3
  __shared__ float sO[kRows][kL3 + 1];
  __shared__ float sr[kMlpBlock / 32][kL3];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, gq = lane >> 2, tq = lane & 3;
  const int64_t row0 = (int64_t)blockIdx.x * kRows;
  float* bsum = g.bsum + (size_t)blockIdx.x * kNBias;
  auto sample = [&](int r) -> int64_t {   // source row of batch row row0 + r, -1: none
    const int64_t b = row0 + r;
    if (b >= g.B) return -1;
    const int64_t sr_ = g.idx ? (int64_t)g.idx[b] : b;
    return sr_ >= 0 && sr_ < g.n_src ? sr_ : -1;
  };
#pragma unroll
  for (int u = 0; u < kRows * kL0 / kMlpBlock; ++u) {
    const int i = tid + u * kMlpBlock, r = i / kL0, c = i % kL0;
    const int64_t sr_ = sample(r);
    sX[r * kSX + c] = __float2bfloat16_rn(sr_ >= 0 ? g.x[sr_ * kL0 + c] : 0.0f);
    if (sr_ < 0 && c == 0 && row0 + r < g.B) atomicExch(g.bad, 1);
  }
  __syncthreads();
  float acc[2][4][4], g1[2][4][4], g2[2][4][4];
  // z + bias -> GELU into dst (BF16), its derivative into gd
  auto act = [&](const float* bias, bf16* dst, float (&gd)[2][4][4]) {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int c = 32 * warp + 8 * j + 2 * tq;
      const float b0 = __ldg(bias + c), b1 = __ldg(bias + c + 1);
#pragma unroll
      for (int m = 0; m < 2; ++m)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const float z0 = acc[m][j][2 * h] + b0, z1 = acc[m][j][2 * h + 1] + b1;
          if (MODE) gd[m][j][2 * h] = gelu_grad_f(z0), gd[m][j][2 * h + 1] = gelu_grad_f(z1);
          *reinterpret_cast<__nv_bfloat162*>(dst + (16 * m + gq + 8 * h) * kSA + c) =
              __floats2bfloat162_rn(gelu_f(z0), gelu_f(z1));
        }
    }
  };
  // a [kRows][W] tile of shared memory to rows row0 .. of a row-major matrix, 16 bytes a thread
  auto put = [&](const bf16* src, int ld, int W, bf16* dst) {
    for (int i = tid; i < kRows * W / 8; i += kMlpBlock) {
      const int r = i / (W / 8), c = (i % (W / 8)) * 8;
      *reinterpret_cast<uint4*>(dst + (row0 + r) * W + c) = *reinterpret_cast<const uint4*>(src + r * ld + c);
    }
  };
  layer_mma<kL0, 2, 4>(sX, kSX, g.P1, 4 * warp, acc);
  act(g.th + kOffB1, sA, g1);
  if (MODE) put(sX, kSX, kL0, g.X0);
  __syncthreads();
  layer_mma<kL1, 2, 4>(sA, kSA, g.P2, 4 * warp, acc);
  act(g.th + kOffB2, sB, g2);
  if (MODE) put(sA, kSA, kL1, g.A1);
  __syncthreads();
  {   // layer 3: warp w takes rows 16 (w & 1) .. and columns 8 (w >> 1) ..
    float o[1][1][4];
    const int m = warp & 1, j = warp >> 1;
    layer_mma<kL2, 1, 1>(sB + m * 16 * kSA, kSA, g.P3, j, o);
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int r = 16 * m + gq + 8 * (e >> 1), c = 8 * j + 2 * tq + (e & 1);
      sO[r][c] = o[0][0][e] + __ldg(g.th + kOffB3 + c);
    }
  }
  if (MODE) put(sB, kSA, kL2, g.A2);
  __syncthreads();
  if (MODE == 0) {
    for (int i = tid; i < kRows * kL3; i += kMlpBlock) {
      const int r = i / kL3, c = i % kL3;
      if (row0 + r < g.B) g.out[(row0 + r) * kL3 + c] = sO[r][c];
    }
    return;
  }
  // loss and dL/dout: a warp takes four rows, a lane one output; sO becomes dL/dout in FP32
  double sq = 0.0;
#pragma unroll
  for (int u = 0; u < kRows / 8; ++u) {
    const int r = warp * (kRows / 8) + u;
    const int64_t sr_ = sample(r);
    float d = 0.0f;
    if (MODE == 1) {
      if (sr_ >= 0) {
        const float scale = 2.0f / ((float)g.B * kL3);
        const float diff = sO[r][lane] - g.t[sr_ * kL3 + lane];
        d = scale * diff;
        sq += (double)diff * diff;
      }
    } else if (sr_ >= 0) {
      // residual space: with the row's sample (W upper triangular, w), r = W d - w, loss += ||r||^2,
      // dL/dd = 2 W^T r / B (row i of the packed triangle starts at 32 i - i (i - 1) / 2)
      const float* S = g.t + sr_ * kNRes;
      const int off = lane * kL3 - lane * (lane - 1) / 2;
      float ri = -S[kNTri + lane];
      for (int j = lane; j < kL3; ++j) ri = fmaf(S[off + j - lane], sO[r][j], ri);
      __syncwarp();
      sr[warp][lane] = ri;
      sq += (double)ri * ri;
      __syncwarp();
      for (int i = 0; i <= lane; ++i) d = fmaf(S[i * kL3 - i * (i - 1) / 2 + lane - i], sr[warp][i], d);
      d *= 2.0f / (float)g.B;
      __syncwarp();
    }
    sO[r][lane] = d;
    sD[r * kSD + lane] = __float2bfloat16_rn(d);
  }
  for (int o = 16; o > 0; o >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
  if (lane == 0 && sq != 0.0) atomicAdd(g.loss, sq);
  __syncthreads();
  if (warp == 0) {
    float c = 0.0f;
#pragma unroll 8
    for (int r = 0; r < kRows; ++r) c += sO[r][lane];
    bsum[kL1 + kL2 + lane] = c;
  }
  put(sD, kSD, kL3, g.dZ3);
  // dZ = (dZ_next W) * GELU'(Z): BF16 into dst, the FP32 column sums (bias gradient) into gb
  auto back = [&](const float (&gd)[2][4][4], bf16* dst, float* gb) {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int c = 32 * warp + 8 * j + 2 * tq;
      float s0 = 0.0f, s1 = 0.0f;
#pragma unroll
      for (int m = 0; m < 2; ++m)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const float v0 = acc[m][j][2 * h] * gd[m][j][2 * h], v1 = acc[m][j][2 * h + 1] * gd[m][j][2 * h + 1];
          s0 += v0, s1 += v1;
          *reinterpret_cast<__nv_bfloat162*>(dst + (16 * m + gq + 8 * h) * kSA + c) = __floats2bfloat162_rn(v0, v1);
        }
#pragma unroll
      for (int o = 4; o < 32; o <<= 1) {
        s0 += __shfl_xor_sync(0xffffffffu, s0, o);
        s1 += __shfl_xor_sync(0xffffffffu, s1, o);
      }
      if (gq == 0) gb[c] = s0, gb[c + 1] = s1;
    }
  };
  layer_mma<kL3, 2, 4>(sD, kSD, g.P3T, 4 * warp, acc);
  back(g2, sB, bsum + kL1);      // (rows past the batch have dL/dout = 0, so their dZ is zero)
  __syncthreads();
  put(sB, kSA, kL2, g.dZ2);
  layer_mma<kL2, 2, 4>(sB, kSA, g.P2T, 4 * warp, acc);
  back(g1, sA, bsum);
  __syncthreads();
  put(sA, kSA, kL1, g.dZ1);
}

// Weight gradients: C[m][n] += sum_b P[b][m] Q[b][n] over the batch rows b, 64 x 64 tiles of the three outputs
// (dW2 = dZ2^T A1: 16 tiles; dW1 = dZ1^T X0: 4; dW3 = dZ3^T A2, as its transpose A2^T dZ3 with 32 columns: 4),
// each with its batch split over gridDim.y blocks that add into the zeroed gradient (so that the grid covers the
// SMs twice; from 512 samples on, so that smaller batches have one writer and repeat bitwise).  The blocks behind the
// tiles sum the bias gradients of the pass's blocks, 32 columns each, in a fixed order.  Both operands lie row-major by sample: ldmatrix.trans turns them.  A block stages 32 samples at a
// time, double-buffered by cp.async.
constexpr int kWgStride = 72;                  // BF16 values a staged row of 64 (144 bytes: conflict-free)
struct MlpWgrad {
  const bf16 *X0, *A1, *A2, *dZ1, *dZ2, *dZ3;
  const float* bsum;
  float* grad;
  int steps;                                   // batch rows / 32, the blocks of the pass
};
constexpr int kWgTiles = 24;
static_assert(kRows == 32 && kNBias % 32 == 0, "one row of bias sums a step, 32 columns a block");
__global__ void __launch_bounds__(128) k_mlp_wgrad(MlpWgrad g) {
  __shared__ __align__(16) bf16 sP[2][32 * kWgStride], sQ[2][32 * kWgStride];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, gq = lane >> 2, tq = lane & 3;
  const int tile = blockIdx.x;
  if (tile >= kWgTiles) {
    if (blockIdx.y) return;
    float* sb = reinterpret_cast<float*>(sP);  // [4][32]
    const int c = (tile - kWgTiles) * 32 + lane;
    float s = 0.0f;
    for (int b = warp; b < g.steps; b += 4) s += g.bsum[(size_t)b * kNBias + c];
    sb[tid] = s;
    __syncthreads();
    const int64_t off = c < kL1 ? kOffB1 + c : c < kL1 + kL2 ? kOffB2 + c - kL1 : kOffB3 + c - kL1 - kL2;
    if (warp == 0) g.grad[off] = (sb[lane] + sb[lane + 32]) + (sb[lane + 64] + sb[lane + 96]);
    return;
  }
  const bf16 *P, *Q;
  float* C;
  int ldp, ldq, nq = 64, rs, cs;               // C[m * rs + n * cs]
  if (tile < 16) {
    P = g.dZ2 + (tile >> 2) * 64, Q = g.A1 + (tile & 3) * 64, ldp = kL2, ldq = kL1, rs = kL1, cs = 1;
    C = g.grad + kOffW2 + (tile >> 2) * 64 * kL1 + (tile & 3) * 64;
  } else if (tile < 20) {
    P = g.dZ1 + (tile - 16) * 64, Q = g.X0, ldp = kL1, ldq = kL0, rs = kL0, cs = 1;
    C = g.grad + kOffW1 + (tile - 16) * 64 * kL0;
  } else {
    P = g.A2 + (tile - 20) * 64, Q = g.dZ3, ldp = kL2, ldq = kL3, nq = 32, rs = 1, cs = kL2;
    C = g.grad + kOffW3 + (tile - 20) * 64;
  }
  const int k0 = (int)((int64_t)g.steps * blockIdx.y / gridDim.y), k1 = (int)((int64_t)g.steps * (blockIdx.y + 1) / gridDim.y);
  auto cp16 = [](bf16* dst, const bf16* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
  };
  auto stage = [&](int k, int b) {
    const int64_t r0 = (int64_t)k * 32;
    for (int i = tid; i < 32 * 8; i += 128) {
      const int r = i >> 3, c = (i & 7) * 8;
      cp16(sP[b] + r * kWgStride + c, P + (r0 + r) * ldp + c);
      if (c < nq) cp16(sQ[b] + r * kWgStride + c, Q + (r0 + r) * ldq + c);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  float acc[8][4];
#pragma unroll
  for (int j = 0; j < 8; ++j)
#pragma unroll
    for (int e = 0; e < 4; ++e) acc[j][e] = 0.0f;
  if (k0 < k1) stage(k0, 0);
  const int mi = lane >> 3, lr = lane & 7;
  for (int k = k0; k < k1; ++k) {
    const int b = (k - k0) & 1;
    if (k + 1 < k1) {
      stage(k + 1, b ^ 1);
      asm volatile("cp.async.wait_group 1;" ::: "memory");
    } else {
      asm volatile("cp.async.wait_group 0;" ::: "memory");
    }
    __syncthreads();
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      uint32_t a[4];
      ldsm4t(a, sP[b] + (16 * h + lr + (mi >> 1) * 8) * kWgStride + 16 * warp + (mi & 1) * 8);
#pragma unroll
      for (int jj = 0; jj < 4; ++jj) {
        if (16 * jj >= nq) break;
        uint32_t q[4];
        ldsm4t(q, sQ[b] + (16 * h + lr + (mi & 1) * 8) * kWgStride + 16 * jj + (mi >> 1) * 8);
        mma_bf16_16816(acc[2 * jj], a, q[0], q[1]);
        mma_bf16_16816(acc[2 * jj + 1], a, q[2], q[3]);
      }
    }
    __syncthreads();
  }
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    if (8 * j >= nq) break;
#pragma unroll
    for (int e = 0; e < 4; ++e)
      atomicAdd(C + (16 * warp + gq + 8 * (e >> 1)) * rs + (8 * j + 2 * tq + (e & 1)) * cs, acc[j][e]);
  }
}

__global__ void k_adam(float* __restrict__ th, float* __restrict__ m, float* __restrict__ v,
                       const float* __restrict__ g, int64_t n, float lr, float b1, float b2, float eps, float bc1,
                       float bc2) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.0f - b1) * gi;
    const float vi = b2 * v[i] + (1.0f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    th[i] -= lr * (mi / bc1) / (sqrtf(vi / bc2) + eps);
  }
}

// The weights in BF16 in the order of the MMA's B fragments: for output columns 8 nt .. +7 and 32 of K (kp), lane
// (gq = lane / 4, tq = lane % 4) holds at P[(nt * K / 32 + kp) * 32 + lane] the values W[8 nt + gq][32 kp + 8 i +
// 2 tq + {0, 1}], i = 0 .. 3.  W1, W2, W3 for the forward pass; W3^T, W2^T for the backward one.
__global__ void k_pack(const float* __restrict__ th, bf16* P1, bf16* P2, bf16* P3, bf16* P3T, bf16* P2T) {
  constexpr int n1 = kL1 * kL0, n2 = kL2 * kL1, n3 = kL3 * kL2;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n1 + 2 * n2 + 2 * n3; i += gridDim.x * blockDim.x) {
    int o = i, K = kL0, n = 0, k = 0;
    bf16* P = P1;
    int which = 0;
    if (o >= n1) o -= n1, which = 1, P = P2, K = kL1;
    if (which == 1 && o >= n2) o -= n2, which = 2, P = P3, K = kL2;
    if (which == 2 && o >= n3) o -= n3, which = 3, P = P3T, K = kL3;
    if (which == 3 && o >= n3) o -= n3, which = 4, P = P2T, K = kL2;
    const int v = o & 7, lane = (o >> 3) & 31, blk = o >> 8;       // 8 values a lane, 32 lanes a block
    n = (blk / (K / 32)) * 8 + (lane >> 2);
    k = (blk % (K / 32)) * 32 + (v >> 1) * 8 + (lane & 3) * 2 + (v & 1);
    const int64_t src = which == 0   ? kOffW1 + n * kL0 + k
                        : which == 1 ? kOffW2 + n * kL1 + k
                        : which == 2 ? kOffW3 + n * kL2 + k
                        : which == 3 ? kOffW3 + k * kL2 + n      // W3^T[n][k] = W3[k][n]
                                     : kOffW2 + k * kL1 + n;     // W2^T[n][k] = W2[k][n]
    P[o] = __float2bfloat16_rn(th[src]);
  }
}

int grid_of(int64_t n) {
  int64_t g = (n + 255) / 256;
  return (int)(g < 1 ? 1 : (g > wide_grid_cap() ? wide_grid_cap() : g));
}

}  // namespace

// ------------------------------------------------------------------------------------------------------
// The network object.
// ------------------------------------------------------------------------------------------------------
struct fem_mlp {
  int device = 0;
  cudaStream_t s = nullptr;
  float *th = nullptr, *m = nullptr, *v = nullptr, *grad = nullptr;
  int64_t t = 0;                       // Adam steps taken
  bf16 *P1 = nullptr, *P2 = nullptr, *P3 = nullptr, *P3T = nullptr, *P2T = nullptr;   // packed weights (k_pack)
  int64_t cap = 0;                     // rows of the training workspace (multiple of kRows)
  bf16 *X0 = nullptr, *A1 = nullptr, *A2 = nullptr, *dZ1 = nullptr, *dZ2 = nullptr, *dZ3 = nullptr;
  float* bsum = nullptr;
  int64_t out_cap = 0;                 // rows of OUT
  float* OUT = nullptr;
  double* loss_acc = nullptr;
  int* bad = nullptr;                  // set by a kernel that met a sample index out of range
  std::mutex mu;

  void free_ws() {
    for (void* p : {(void*)X0, (void*)A1, (void*)A2, (void*)dZ1, (void*)dZ2, (void*)dZ3, (void*)bsum})
      if (p) cudaFree(p);
    X0 = A1 = A2 = dZ1 = dZ2 = dZ3 = nullptr;
    bsum = nullptr;
    cap = 0;
  }
  ~fem_mlp() {
    free_ws();
    for (void* p : {(void*)th, (void*)m, (void*)v, (void*)grad, (void*)P1, (void*)P2, (void*)P3, (void*)P3T,
                    (void*)P2T, (void*)OUT, (void*)loss_acc, (void*)bad})
      if (p) cudaFree(p);
  }
};

namespace {

#define CE(x)                                 \
  do {                                        \
    cudaError_t e_ = (x);                     \
    if (e_ != cudaSuccess) return e_;         \
  } while (0)

template <typename T>
cudaError_t alloc_n(T** p, int64_t n) {
  return cudaMalloc((void**)p, sizeof(T) * (size_t)(n > 0 ? n : 1));
}

// Training workspace of `rows` rows (a multiple of kRows).
cudaError_t ensure_cap(fem_mlp* n, int64_t rows) {
  if (rows <= n->cap) return cudaSuccess;
  // the old workspace may still be read by work queued on another stream
  CE(cudaDeviceSynchronize());
  n->free_ws();
  cudaError_t e = cudaSuccess;
  auto A = [&](auto** p, int64_t k) {
    if (e == cudaSuccess) e = alloc_n(p, k);
  };
  A(&n->X0, rows * kL0); A(&n->A1, rows * kL1); A(&n->A2, rows * kL2);
  A(&n->dZ1, rows * kL1); A(&n->dZ2, rows * kL2); A(&n->dZ3, rows * kL3);
  A(&n->bsum, rows / kRows * kNBias);
  if (e != cudaSuccess) {
    cudaGetLastError();
    n->free_ws();
    return e;
  }
  n->cap = rows;
  return cudaSuccess;
}

// OUT for `rows` rows.
cudaError_t ensure_out(fem_mlp* n, int64_t rows) {
  if (rows <= n->out_cap) return cudaSuccess;
  CE(cudaDeviceSynchronize());      // (the old buffer may still be read by work queued on another stream)
  if (n->OUT) cudaFree(n->OUT);
  n->OUT = nullptr, n->out_cap = 0;
  CE(alloc_n(&n->OUT, rows * kL3));
  n->out_cap = rows;
  return cudaSuccess;
}

// Whether the results of `out` may overwrite values of `in` that other blocks still read.
bool overlap(const void* out, size_t out_bytes, const void* in, size_t in_bytes) {
  const uintptr_t a = reinterpret_cast<uintptr_t>(out), b = reinterpret_cast<uintptr_t>(in);
  return a < b + in_bytes && b < a + out_bytes;
}

cudaError_t pack_weights(fem_mlp* n, cudaStream_t s) {
  k_pack<<<grid_of(kNParams + kL2 * kL1), 256, 0, s>>>(n->th, n->P1, n->P2, n->P3, n->P3T, n->P2T);
  return cudaGetLastError();
}

MlpPass pass_args(const fem_mlp* n, const float* x, const int32_t* idx, int64_t n_src, int64_t B) {
  MlpPass g{};
  g.x = x, g.idx = idx, g.n_src = n_src, g.B = B, g.Mpad = ((B + kRows - 1) / kRows) * kRows;
  g.P1 = (const uint4*)n->P1, g.P2 = (const uint4*)n->P2, g.P3 = (const uint4*)n->P3;
  g.P3T = (const uint4*)n->P3T, g.P2T = (const uint4*)n->P2T;
  g.th = n->th, g.bad = n->bad;
  return g;
}

// out [B][32] = network of the B rows of x.
cudaError_t forward(fem_mlp* n, const float* x, int64_t B, float* out, cudaStream_t s) {
  MlpPass g = pass_args(n, x, nullptr, B, B);
  g.out = out;
  k_mlp_pass<0><<<(unsigned)(g.Mpad / kRows), kMlpBlock, 0, s>>>(g);
  return cudaGetLastError();
}

// Loss (added to n->loss_acc) and its gradient into grad, over B rows (gathered through idx if given) of x and
// the targets t (residual: residual-space samples).
cudaError_t loss_grad(fem_mlp* n, const float* x, const float* t, const int32_t* idx, int64_t n_src, int64_t B,
                      float* grad, cudaStream_t s, bool residual) {
  MlpPass g = pass_args(n, x, idx, n_src, B);
  CE(ensure_cap(n, g.Mpad));
  CE(cudaMemsetAsync(grad, 0, sizeof(float) * kNParams, s));
  g.t = t, g.bsum = n->bsum, g.loss = n->loss_acc;
  g.X0 = n->X0, g.A1 = n->A1, g.A2 = n->A2, g.dZ1 = n->dZ1, g.dZ2 = n->dZ2, g.dZ3 = n->dZ3;
  const unsigned blocks = (unsigned)(g.Mpad / kRows);
  if (residual)
    k_mlp_pass<2><<<blocks, kMlpBlock, 0, s>>>(g);
  else
    k_mlp_pass<1><<<blocks, kMlpBlock, 0, s>>>(g);
  CE(cudaGetLastError());
  // 24 tiles; the batch split so that the grid covers the SMs twice, at least 8 of the 32-row steps a block
  MlpWgrad w{n->X0, n->A1, n->A2, n->dZ1, n->dZ2, n->dZ3, n->bsum, grad, (int)(g.Mpad / 32)};
  int split = (2 * sm_count() + kWgTiles - 1) / kWgTiles;
  if (split > w.steps / 8) split = w.steps / 8;
  k_mlp_wgrad<<<dim3(kWgTiles + kNBias / 32, split < 1 ? 1 : split), 128, 0, s>>>(w);
  return cudaGetLastError();
}

cudaError_t adam(fem_mlp* n, double lr, cudaStream_t s) {
  n->t += 1;
  const double b1 = 0.9, b2 = 0.999;
  const float bc1 = (float)(1.0 - std::pow(b1, (double)n->t)), bc2 = (float)(1.0 - std::pow(b2, (double)n->t));
  k_adam<<<grid_of(kNParams), 256, 0, s>>>(n->th, n->m, n->v, n->grad, kNParams, (float)lr, (float)b1, (float)b2,
                                           1e-8f, bc1, bc2);
  CE(cudaGetLastError());
  return pack_weights(n, s);
}

// ------------------------------------------------------------------------------------------------------
// Kernels of the time step.
// ------------------------------------------------------------------------------------------------------

// Input features of row R * rpad + c: (source - centroid_R) / L, (f0 - 5) / 3, asinh of the predictor's
// coefficients in age order (newest pair first), zeros.  Pad rows up to Mpad are zero.
__global__ void k_features(PredView p, int n_pairs, const float4* __restrict__ case_src,
                           const float* __restrict__ centroid, float inv_extent, int64_t Mpad, float* __restrict__ F) {
  const int64_t rows = (int64_t)p.n_regions * p.rpad;
  const int64_t total = Mpad * kL0;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t row = i / kL0;
    const int j = (int)(i % kL0);
    float v = 0.0f;
    if (row < rows) {
      const int R = (int)(row / p.rpad), c = (int)(row % p.rpad);
      if (j < 3) {
        const float4 sp = case_src[c];
        const float s3[3] = {sp.x, sp.y, sp.z};
        v = (s3[j] - centroid[R * 3 + j]) * inv_extent;
      } else if (j == 3) {
        v = case_src[c].w;
      } else if (j < 4 + n_pairs) {
        const int a = n_pairs - 1 - (j - 4);
        const double c = p.w[row * kMaxSlots + a];
        v = isfinite(c) ? (float)asinh(c) : 0.0f;     // bounded input for nearly collinear snapshots
      }
    }
    F[i] = v;
  }
}

// Coefficient correction of the proposal in slot order (column a of Y is e^{it-n+a}):  dw_a = out[n-1-a].
__global__ void k_coef_delta(int64_t rows, int n_pairs, const float* __restrict__ out, double* __restrict__ dw) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < rows * kMaxSlots;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t row = i / kMaxSlots;
    const int a = (int)(i % kMaxSlots);
    dw[i] = a < n_pairs ? (double)out[row * kL3 + (n_pairs - 1 - a)] : 0.0;
  }
}

__global__ void k_to_f32(int64_t n, const double* __restrict__ x, float* __restrict__ y) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    y[i] = (float)x[i];
}

// Per case: squared norm of the proposal's initial residual r0 - A dy (free DOFs); the proposal is taken
// where it is smaller than the plain guess's.  The last block updates the case's solver state.
__global__ void __launch_bounds__(kVecBlock) k_choose(MeshView m, int rpad, int rshift, const float* __restrict__ r32,
                                                      const float* __restrict__ qd, Reducer red, CgCase* outer,
                                                      int* n_active, double tol, double inner_max, double aim,
                                                      int ncase, int* __restrict__ choose,
                                                      long long* __restrict__ counts) {
  double rr = 0.0;
  const int64_t total = m.N << rshift;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t n = i >> rshift;
    const int c = (int)(i & (rpad - 1));
    const uint8_t f = m.freemask[n];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      if (!dof_free(f, k)) continue;
      const int64_t id = (n * 3 + k) * rpad + c;
      const double v = (double)r32[id] - (double)qd[id];
      rr += v * v;
    }
  }
  double vals[1] = {rr};
  if (block_reduce_last<1>(vals, rpad, red)) {
    if (threadIdx.x < rpad) {
      const int c = threadIdx.x;
      CgCase& s = outer[c];
      const double rrc = red.out[c];
      const bool take = c < ncase && s.status == FEM_OK && s.bb > 0.0 && isfinite(rrc) && rrc < s.rr;
      choose[c] = take ? 1 : 0;
      if (take) {
        s.rr = rrc;
        s.relres = sqrt(rrc / s.bb);
        s.relres0 = s.relres;
        s.active = rrc >= tol * tol * s.bb ? 1 : 0;
        s.inner_tol = inner_target(aim, s.relres, inner_max);
      }
      if (c < ncase && s.bb > 0.0) atomicAdd(reinterpret_cast<unsigned long long*>(counts + (take ? 0 : 1)), 1ull);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      int na = 0;
      for (int c = 0; c < rpad; ++c) na += outer[c].active;
      *n_active = na;
    }
  }
}

__global__ void k_apply(int64_t n, int rpad, const int* __restrict__ choose, float* __restrict__ r32,
                        const float* __restrict__ qd, double* __restrict__ guess, const double* __restrict__ dy) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    if (!choose[i & (rpad - 1)]) continue;
    r32[i] -= qd[i];
    guess[i] += dy[i];
  }
}

// Training samples of one step: features F (computed at prediction time) and targets c* - c in age
// order, for the real cases; rows are appended at row0 in (region, case) order.  A target with a
// non-finite entry or one above kTargetClip in magnitude is written as zero (no correction).
constexpr double kTargetClip = 100.0;

__global__ void k_collect(int n_regions, int rpad, int ncase, int n_pairs, const float* __restrict__ F,
                          const double* __restrict__ w_best, const double* __restrict__ w_pred, int64_t row0,
                          float* __restrict__ x_out, float* __restrict__ t_out) {
  const int64_t rows = (int64_t)n_regions * ncase;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < rows * (kL0 + 1);
       i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t row = i / (kL0 + 1);
    const int j = (int)(i % (kL0 + 1));
    const int R = (int)(row / ncase), c = (int)(row % ncase);
    const int64_t src = (int64_t)R * rpad + c;
    if (j < kL0) {
      x_out[(row0 + row) * kL0 + j] = F[src * kL0 + j];
    } else {
      float t[kL3];
      bool ok = true;
#pragma unroll
      for (int k = 0; k < kL3; ++k) {
        double d = 0.0;
        if (k < n_pairs) {
          const int a = n_pairs - 1 - k;
          d = w_best[src * kMaxSlots + a] - w_pred[src * kMaxSlots + a];
        }
        ok = ok && isfinite(d) && fabs(d) <= kTargetClip;
        t[k] = (float)d;
      }
#pragma unroll
      for (int k = 0; k < kL3; ++k) t_out[(row0 + row) * kL3 + k] = ok ? t[k] : 0.0f;
    }
  }
}

// Per case c: ||e||^2 of the step's correction over all regions, sum_R G_R[new][new] (one block per case,
// fixed summation order).
__global__ void __launch_bounds__(256) k_case_e2(PredView p, int slot_new, double* __restrict__ e2) {
  __shared__ double part[256];
  const int c = blockIdx.x;
  double acc = 0.0;
  for (int R = threadIdx.x; R < p.n_regions; R += blockDim.x)
    acc += p.gram[(((int64_t)R * p.rpad + c) * kMaxSlots + slot_new) * kMaxSlots + slot_new];
  part[threadIdx.x] = acc;
  __syncthreads();
  for (int h = blockDim.x / 2; h > 0; h >>= 1) {
    if ((int)threadIdx.x < h) part[threadIdx.x] += part[threadIdx.x + h];
    __syncthreads();
  }
  if (threadIdx.x == 0) e2[c] = part[0];
}

// Residual-space training samples of one step (one warp per region and real case): the features F of the
// step's prediction, and (W, w) of the region's share ||Y_R (c + d) - e_R||^2 / ||e||^2 of the relative error
// of the case's corrected guess of the correction, from the ring Gram after e = e^it is pushed (||e||^2 of the
// whole case from k_case_e2).  In age order (index k: the pair whose output is e^{it-1-k}) the Gram of Y_R is
// factored R^T R by the same right-looking Cholesky with the column-drop rule as the predictor (pivot <=
// tau^2 G_kk drops column k: its row of R is zero); then z = R^{-T} Y_R^T e_R, W = R / ||e||,
// w = (z - R c) / ||e||.  A sample of a case with ||e|| = 0, or with a non-finite value, is zero.
__global__ void __launch_bounds__(32) k_collect_res(PredView p, const int* __restrict__ y_slots, int n, int slot_new,
                                                    double tau, int ncase, const double* __restrict__ e2case,
                                                    const float* __restrict__ F, int64_t row0,
                                                    float* __restrict__ x_out, float* __restrict__ s_out) {
  const int R = blockIdx.x / ncase, c = blockIdx.x % ncase;
  const int lane = threadIdx.x;
  constexpr int LD = kMaxSlots;
  __shared__ double L[kMaxSlots * LD];
  __shared__ double inv[kMaxSlots];
  const int64_t src = (int64_t)R * p.rpad + c;
  const int64_t row = row0 + (int64_t)R * ncase + c;
  for (int j = lane; j < kL0; j += 32) x_out[row * kL0 + j] = F[src * kL0 + j];
  const double* G = p.gram + src * kMaxSlots * kMaxSlots;
  const int yk = lane < n ? y_slots[n - 1 - lane] : 0;
  for (int i = 0; i < n; ++i) {
    const int yi = __shfl_sync(0xffffffffu, yk, i);
    if (lane < n) L[i * LD + lane] = G[yi * kMaxSlots + yk];
  }
  const double rhs = lane < n ? G[yk * kMaxSlots + slot_new] : 0.0;
  const double d0 = lane < n ? G[yk * kMaxSlots + yk] : 0.0;
  const double E = e2case[c];
  __syncwarp();
  for (int j = 0; j < n; ++j) {
    const double djj = L[j * LD + j];
    const double d0j = __shfl_sync(0xffffffffu, d0, j);
    const bool keep = d0j > 0.0 && djj > tau * tau * d0j && isfinite(djj);
    const double ip = keep ? rsqrt(djj) : 0.0;
    __syncwarp();
    if (lane > j && lane < n) L[lane * LD + j] = keep ? L[lane * LD + j] * ip : 0.0;
    if (lane == j) {
      L[j * LD + j] = keep ? djj * ip : 0.0;
      inv[j] = ip;
    }
    __syncwarp();
    if (keep && lane > j && lane < n) {   // lane i updates row i of the trailing block: L_ik -= L_ij L_kj
      const double lij = L[lane * LD + j];
      for (int k = j + 1; k <= lane; ++k) L[lane * LD + k] = fma(-lij, L[k * LD + j], L[lane * LD + k]);
    }
    __syncwarp();
  }
  double z = rhs;   // forward substitution R^T z = Y^T e (dropped columns give 0)
  for (int j = 0; j < n; ++j) {
    const double zr = __shfl_sync(0xffffffffu, z, j);
    const double zj = inv[j] != 0.0 ? zr * inv[j] : 0.0;
    if (lane == j) z = zj;
    if (lane > j && lane < n) z -= L[lane * LD + j] * zj;
  }
  const double ck = lane < n ? p.w[src * kMaxSlots + (n - 1 - lane)] : 0.0;
  double v = z;     // v_i = z_i - sum_{j >= i} R_ij c_j with R_ij = L_ji
  for (int j = 0; j < n; ++j) {
    const double cj = __shfl_sync(0xffffffffu, ck, j);
    if (lane <= j && lane < n) v -= L[j * LD + lane] * cj;
  }
  double sc = (E > 0.0 && isfinite(E)) ? rsqrt(E) : 0.0;
  if (__any_sync(0xffffffffu, !isfinite(v * sc))) sc = 0.0;
  float* so = s_out + row * kNRes;
  for (int i = 0; i < kL3; ++i) {
    const int off = i * kL3 - i * (i - 1) / 2;
    for (int j = i + lane; j < kL3; j += 32)
      so[off + j - i] = (sc != 0.0 && i < n && j < n) ? (float)(L[j * LD + i] * sc) : 0.0f;
  }
  so[kNTri + lane] = (sc != 0.0 && lane < n) ? (float)(v * sc) : 0.0f;
}

}  // namespace

// ------------------------------------------------------------------------------------------------------
// Internal entry points used by the time step.
// ------------------------------------------------------------------------------------------------------
namespace fem {

cudaError_t mlp_features(const PredView& p, int n_pairs, const float4* case_src, const float* centroid,
                         float inv_extent, float* F, cudaStream_t s) {
  const int64_t Mp = (((int64_t)p.n_regions * p.rpad + 63) / 64) * 64;
  k_features<<<grid_of(Mp * kL0), 256, 0, s>>>(p, n_pairs, case_src, centroid, inv_extent, Mp, F);
  return cudaGetLastError();
}

cudaError_t mlp_propose(fem_mlp* net, const float* F, int64_t rows, int n_pairs, double* dw, cudaStream_t s) {
  std::lock_guard<std::mutex> lk(net->mu);
  CE(ensure_out(net, rows));
  CE(forward(net, F, rows, net->OUT, s));
  k_coef_delta<<<grid_of(rows * kMaxSlots), 256, 0, s>>>(rows, n_pairs, net->OUT, dw);
  return cudaGetLastError();
}

cudaError_t mlp_to_f32(int64_t n, const double* x, float* y, cudaStream_t s) {
  k_to_f32<<<grid_of(n), 256, 0, s>>>(n, x, y);
  return cudaGetLastError();
}

cudaError_t mlp_choose(const MeshView& m, int rpad, const float* r32, const float* qd, Reducer red, CgCase* outer,
                       int* n_active, double tol, double inner_max, double aim, int ncase, int* choose,
                       long long* counts, cudaStream_t s) {
  int rs = 0;
  while ((1 << rs) < rpad) ++rs;
  int64_t items = m.N << rs;
  int grid = (int)((items + kVecBlock - 1) / kVecBlock);
  if (grid > vec_grid_cap()) grid = vec_grid_cap();
  if (grid < 1) grid = 1;
  k_choose<<<grid, kVecBlock, 0, s>>>(m, rpad, rs, r32, qd, red, outer, n_active, tol, inner_max, aim, ncase,
                                      choose, counts);
  return cudaGetLastError();
}

cudaError_t mlp_apply(int64_t n, int rpad, const int* choose, float* r32, const float* qd, double* guess,
                      const double* dy, cudaStream_t s) {
  k_apply<<<grid_of(n), 256, 0, s>>>(n, rpad, choose, r32, qd, guess, dy);
  return cudaGetLastError();
}

cudaError_t mlp_collect(int n_regions, int rpad, int ncase, int n_pairs, const float* F, const double* w_best,
                        const double* w_pred, int64_t row0, float* x_out, float* t_out, cudaStream_t s) {
  const int64_t rows = (int64_t)n_regions * ncase;
  k_collect<<<grid_of(rows * (kL0 + 1)), 256, 0, s>>>(n_regions, rpad, ncase, n_pairs, F, w_best, w_pred, row0,
                                                        x_out, t_out);
  return cudaGetLastError();
}

cudaError_t mlp_collect_res(const PredView& p, const int* y_slots, int n_pairs, int slot_new, double tau, int ncase,
                            const float* F, int64_t row0, float* x_out, float* s_out, double* e2, cudaStream_t s) {
  k_case_e2<<<ncase, 256, 0, s>>>(p, slot_new, e2);
  k_collect_res<<<p.n_regions * ncase, 32, 0, s>>>(p, y_slots, n_pairs, slot_new, tau, ncase, e2, F, row0, x_out,
                                                   s_out);
  return cudaGetLastError();
}

int mlp_device(const fem_mlp* n) { return n->device; }

}  // namespace fem

// ------------------------------------------------------------------------------------------------------
// C ABI
// ------------------------------------------------------------------------------------------------------
#define MCU(x)                                                                                 \
  do {                                                                                         \
    cudaError_t e_ = (x);                                                                      \
    if (e_ != cudaSuccess) {                                                                   \
      cudaGetLastError();                                                                      \
      return set_error(FEM_ERR_CUDA, std::string(#x ": ") + cudaGetErrorString(e_));           \
    }                                                                                          \
  } while (0)

extern "C" {

fem_status fem_mlp_create(const float* params, void* stream, fem_mlp** out) {
  if (!params || !out) return set_error(FEM_ERR_ARG, "fem_mlp_create: null argument");
  *out = nullptr;
  fem_mlp* n = new fem_mlp();
  n->s = (cudaStream_t)stream;
  cudaGetDevice(&n->device);
  cudaError_t e = cudaSuccess;
  auto A = [&](auto** p, int64_t k) {
    if (e == cudaSuccess) e = alloc_n(p, k);
  };
  A(&n->th, kNParams); A(&n->m, kNParams); A(&n->v, kNParams); A(&n->grad, kNParams);
  A(&n->P1, (int64_t)kL1 * kL0); A(&n->P2, (int64_t)kL2 * kL1); A(&n->P2T, (int64_t)kL2 * kL1);
  A(&n->P3, (int64_t)kL3 * kL2); A(&n->P3T, (int64_t)kL3 * kL2); A(&n->loss_acc, 1); A(&n->bad, 1);
  if (e != cudaSuccess) {
    cudaGetLastError();
    delete n;
    return set_error(FEM_ERR_OOM, "fem_mlp_create: device allocation failed");
  }
  e = cudaMemcpyAsync(n->th, params, sizeof(float) * kNParams, cudaMemcpyHostToDevice, n->s);
  if (e == cudaSuccess) e = cudaMemsetAsync(n->m, 0, sizeof(float) * kNParams, n->s);
  if (e == cudaSuccess) e = cudaMemsetAsync(n->v, 0, sizeof(float) * kNParams, n->s);
  if (e == cudaSuccess) e = cudaMemsetAsync(n->bad, 0, sizeof(int), n->s);
  if (e == cudaSuccess) e = pack_weights(n, n->s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(n->s);
  if (e != cudaSuccess) {
    cudaGetLastError();
    delete n;
    return set_error(FEM_ERR_CUDA, std::string("fem_mlp_create: ") + cudaGetErrorString(e));
  }
  *out = n;
  return FEM_OK;
}

fem_status fem_mlp_destroy(fem_mlp* n) {
  if (!n) return FEM_OK;
  cudaStreamSynchronize(n->s);
  delete n;
  return FEM_OK;
}

fem_status fem_mlp_get_params(fem_mlp* n, float* params) {
  if (!n || !params) return set_error(FEM_ERR_ARG, "fem_mlp_get_params: null argument");
  MCU(cudaMemcpyAsync(params, n->th, sizeof(float) * kNParams, cudaMemcpyDeviceToHost, n->s));
  MCU(cudaStreamSynchronize(n->s));
  return FEM_OK;
}

fem_status fem_mlp_forward(fem_mlp* n, const float* x_dev, int64_t B, float* out_dev) {
  if (!n || (B > 0 && (!x_dev || !out_dev)) || B < 0) return set_error(FEM_ERR_ARG, "fem_mlp_forward: bad argument");
  if (B == 0) return FEM_OK;
  std::lock_guard<std::mutex> lk(n->mu);
  const size_t bytes = sizeof(float) * kL3 * B;
  const bool apart = !overlap(out_dev, bytes, x_dev, sizeof(float) * kL0 * B);
  if (!apart) MCU(ensure_out(n, B));
  MCU(forward(n, x_dev, B, apart ? out_dev : n->OUT, n->s));
  if (!apart) MCU(cudaMemcpyAsync(out_dev, n->OUT, bytes, cudaMemcpyDeviceToDevice, n->s));
  return FEM_OK;
}


static fem_status mlp_loss_grad_any(fem_mlp* n, const float* x_dev, const float* t_dev, int64_t B, float* grad_dev,
                                    double* loss_out, bool residual) {
  clear_error();
  if (!n || !x_dev || !t_dev || B <= 0) return set_error(FEM_ERR_ARG, "fem_mlp_loss_grad: bad argument");
  std::lock_guard<std::mutex> lk(n->mu);
  MCU(cudaMemsetAsync(n->loss_acc, 0, sizeof(double), n->s));
  // (grad_dev may lie in the inputs' memory: it is written once they have been read)
  const size_t gbytes = sizeof(float) * kNParams;
  const bool apart = grad_dev && !overlap(grad_dev, gbytes, x_dev, sizeof(float) * kL0 * B) &&
                     !overlap(grad_dev, gbytes, t_dev, sizeof(float) * (residual ? kNRes : kL3) * B);
  MCU(loss_grad(n, x_dev, t_dev, nullptr, B, B, apart ? grad_dev : n->grad, n->s, residual));
  if (grad_dev && !apart) MCU(cudaMemcpyAsync(grad_dev, n->grad, gbytes, cudaMemcpyDeviceToDevice, n->s));
  double acc = 0.0;
  MCU(cudaMemcpyAsync(&acc, n->loss_acc, sizeof(double), cudaMemcpyDeviceToHost, n->s));
  MCU(cudaStreamSynchronize(n->s));
  if (loss_out) *loss_out = residual ? acc / (double)B : acc / ((double)B * kL3);
  return FEM_OK;
}

static fem_status mlp_train_any(fem_mlp* n, const float* x_dev, const float* t_dev, int64_t n_samples,
                                const int32_t* order_dev, int n_updates, int batch, double lr, double* loss_out,
                                bool residual) {
  clear_error();
  if (!n || !x_dev || !t_dev || !order_dev || n_samples <= 0 || n_updates < 0 || batch <= 0 || !(lr > 0.0))
    return set_error(FEM_ERR_ARG, "fem_mlp_train: bad argument");
  std::lock_guard<std::mutex> lk(n->mu);
  MCU(cudaMemsetAsync(n->bad, 0, sizeof(int), n->s));
  for (int u = 0; u < n_updates; ++u) {
    const int32_t* idx = order_dev + (int64_t)u * batch;
    if (loss_out) MCU(cudaMemsetAsync(n->loss_acc, 0, sizeof(double), n->s));
    MCU(loss_grad(n, x_dev, t_dev, idx, n_samples, batch, n->grad, n->s, residual));
    if (loss_out) {
      double acc = 0.0;
      MCU(cudaMemcpyAsync(&acc, n->loss_acc, sizeof(double), cudaMemcpyDeviceToHost, n->s));
      MCU(cudaStreamSynchronize(n->s));
      loss_out[u] = residual ? acc / (double)batch : acc / ((double)batch * kL3);
    }
    MCU(adam(n, lr, n->s));
  }
  int bad = 0;
  MCU(cudaMemcpyAsync(&bad, n->bad, sizeof(int), cudaMemcpyDeviceToHost, n->s));
  MCU(cudaStreamSynchronize(n->s));
  if (bad) return set_error(FEM_ERR_ARG, "fem_mlp_train: a sample index was outside [0, n_samples)");
  return FEM_OK;
}

fem_status fem_mlp_loss_grad(fem_mlp* n, const float* x_dev, const float* t_dev, int64_t B, float* grad_dev,
                             double* loss_out) {
  return mlp_loss_grad_any(n, x_dev, t_dev, B, grad_dev, loss_out, false);
}

fem_status fem_mlp_loss_grad_residual(fem_mlp* n, const float* x_dev, const float* s_dev, int64_t B, float* grad_dev,
                                      double* loss_out) {
  return mlp_loss_grad_any(n, x_dev, s_dev, B, grad_dev, loss_out, true);
}

fem_status fem_mlp_train(fem_mlp* n, const float* x_dev, const float* t_dev, int64_t n_samples,
                         const int32_t* order_dev, int n_updates, int batch, double lr, double* loss_out) {
  return mlp_train_any(n, x_dev, t_dev, n_samples, order_dev, n_updates, batch, lr, loss_out, false);
}

fem_status fem_mlp_train_residual(fem_mlp* n, const float* x_dev, const float* s_dev, int64_t n_samples,
                                  const int32_t* order_dev, int n_updates, int batch, double lr, double* loss_out) {
  return mlp_train_any(n, x_dev, s_dev, n_samples, order_dev, n_updates, batch, lr, loss_out, true);
}

}  // extern "C"
