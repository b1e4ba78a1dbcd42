// Learned starting value for the Riemann star pressure: the 6 -> 64 -> 64 -> 1
// SiLU perceptron on BF16 tensor cores (tcgen05, accumulators in tensor
// memory), its training (forward, backward, Adam), and the data path that
// feeds it (face-state harvest, exact p* targets, feature normalisation).
// The paper has no such component; see learned.cuh for the specification.
//
// Tiles are 128 samples (faces): sample t of the tile is row t of every MMA and
// lane t of tensor memory.  The forward kernel has a thread per sample (4 warps),
// the gradient kernel two, which split the columns (8 warps).
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <string>
#include <vector>

#include "amm_internal.cuh"
#include "learned.cuh"
#include "riemann.cuh"
#include "tc.cuh"

namespace amm {

constexpr int MLP_TILE = 128;
constexpr int NP_W1 = MLP_HID * MLP_IN, NP_B1 = MLP_HID, NP_W2 = MLP_HID * MLP_HID, NP_B2 = MLP_HID, NP_W3 = MLP_HID;
constexpr int OFF_W1 = 0, OFF_B1 = OFF_W1 + NP_W1, OFF_W2 = OFF_B1 + NP_B1, OFF_B2 = OFF_W2 + NP_W2,
              OFF_W3 = OFF_B2 + NP_B2, OFF_B3 = OFF_W3 + NP_W3, NPARAMS = OFF_B3 + 1;

__device__ __forceinline__ float silu(float z) { return z / (1.0f + __expf(-z)); }

// parameter i of the FP32 master vector into the kernels' weights (BF16
// matrices, FP32 biases; the padding columns of W1 stay zero)
__device__ __forceinline__ void mlp_pack_one(int i, float x, MlpDevice* out) {
  if (i < OFF_B1)
    out->W1[i / MLP_IN * 16 + i % MLP_IN] = __float2bfloat16_rn(x);
  else if (i < OFF_W2)
    out->b1[i - OFF_B1] = x;
  else if (i < OFF_B2)
    out->W2[i - OFF_W2] = __float2bfloat16_rn(x);
  else if (i < OFF_W3)
    out->b2[i - OFF_B2] = x;
  else if (i < OFF_B3)
    out->W3[i - OFF_W3] = __float2bfloat16_rn(x);
  else
    out->b3 = x;
}

__global__ void k_mlp_pack(const float* p, MlpDevice* out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < NPARAMS) mlp_pack_one(i, p[i], out);
}

// Shared-memory image of one CTA's operands
struct MlpSmem {
  alignas(1024) uint8_t a1[MLP_TILE * 16 * 2];        // X      [128 x 16]
  alignas(1024) uint8_t a2[MLP_TILE * MLP_HID * 2];   // H1     [128 x 64]
  alignas(1024) uint8_t b1[MLP_HID * 16 * 2];         // W1     [64 x 16]
  alignas(1024) uint8_t b2[MLP_HID * MLP_HID * 2];    // W2     [64 x 64]
  float bias1[MLP_HID], bias2[MLP_HID], w3[MLP_HID];
  float bias3;
  uint64_t mbar;
  uint32_t tmem;
  uint32_t ok;
};

// weights into the K-major core-matrix layout
__device__ __forceinline__ void load_weights(MlpSmem& s, const MlpDevice* M) {
  for (int i = threadIdx.x; i < MLP_HID * 16; i += blockDim.x) {
    const int o = i / 16, k = i % 16;
    *reinterpret_cast<__nv_bfloat16*>(s.b1 + tc::kmajor_offset(o, k, 16)) = M->W1[i];
  }
  for (int i = threadIdx.x; i < MLP_HID * MLP_HID; i += blockDim.x) {
    const int o = i / MLP_HID, k = i % MLP_HID;
    *reinterpret_cast<__nv_bfloat16*>(s.b2 + tc::kmajor_offset(o, k, MLP_HID)) = M->W2[i];
  }
  for (int i = threadIdx.x; i < MLP_HID; i += blockDim.x) {
    s.bias1[i] = M->b1[i];
    s.bias2[i] = M->b2[i];
    s.w3[i] = __bfloat162float(M->W3[i]);
  }
  if (threadIdx.x == 0) s.bias3 = M->b3;
}

// Forward pass of one tile; x[6] in, returns y.  Called by all 128 threads;
// uses tensor-memory columns [0,64) and [64,128) of s.tmem.  `phase` is the
// mbarrier parity of the first of the two waits (the second uses phase^1).
// On a wait timeout s.ok is cleared and y is 0.
__device__ __forceinline__ float mlp_tile_forward(MlpSmem& s, const float* x, uint32_t phase) {
  const int t = threadIdx.x;
  const int warp = t >> 5;
  {
    float row[16] = {x[0], x[1], x[2], x[3], x[4], x[5], 0, 0, 0, 0, 0, 0, 0, 0, 0, 0};
    tc::st_bf16x8(s.a1, tc::kmajor_offset(t, 0, 16), row);
    tc::st_bf16x8(s.a1, tc::kmajor_offset(t, 8, 16), row + 8);
  }
  tc::fence_async_smem();
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  if (t == 0) {
    const uint64_t ad = tc::kmajor_desc(tc::smem_addr(s.a1), 16);
    const uint64_t bd = tc::kmajor_desc(tc::smem_addr(s.b1), 16);
    tc::mma_bf16(s.tmem, ad, bd, tc::make_idesc(128, 64), false);
    tc::mma_commit(&s.mbar);
  }
  if (!tc::mbar_wait(&s.mbar, phase)) s.ok = 0;
  tc::fence_after_sync();
  // layer 1 epilogue: h1 = silu(z1 + b1) -> A2
#pragma unroll
  for (int c = 0; c < 4; c++) {
    float z[16];
    tc::tmem_ld16(tc::tmem_lane_addr(s.tmem, warp, 16 * c), z);
#pragma unroll
    for (int j = 0; j < 16; j++) z[j] = silu(z[j] + s.bias1[16 * c + j]);
    tc::st_bf16x8(s.a2, tc::kmajor_offset(t, 16 * c, MLP_HID), z);
    tc::st_bf16x8(s.a2, tc::kmajor_offset(t, 16 * c + 8, MLP_HID), z + 8);
  }
  tc::fence_async_smem();
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  if (t == 0) {
#pragma unroll
    for (int kb = 0; kb < MLP_HID / 16; kb++) {
      const uint64_t ad = tc::kmajor_desc(tc::smem_addr(s.a2) + 256 * kb, MLP_HID);
      const uint64_t bd = tc::kmajor_desc(tc::smem_addr(s.b2) + 256 * kb, MLP_HID);
      tc::mma_bf16(s.tmem + 64, ad, bd, tc::make_idesc(128, 64), kb > 0);
    }
    tc::mma_commit(&s.mbar);
  }
  if (!tc::mbar_wait(&s.mbar, phase ^ 1u)) s.ok = 0;
  tc::fence_after_sync();
  float y = s.bias3;
#pragma unroll
  for (int c = 0; c < 4; c++) {
    float z[16];
    tc::tmem_ld16(tc::tmem_lane_addr(s.tmem, warp, 64 + 16 * c), z);
#pragma unroll
    for (int j = 0; j < 16; j++) y += s.w3[16 * c + j] * silu(z[j] + s.bias2[16 * c + j]);
  }
  return s.ok ? y : 0.0f;
}

// batched inference: one 128-sample tile per CTA
__global__ void __launch_bounds__(MLP_TILE) k_mlp_forward(const MlpDevice* M, const float* x, int64_t m, float* y,
                                                         unsigned* status) {
  extern __shared__ uint8_t smem_raw[];
  MlpSmem& s = *reinterpret_cast<MlpSmem*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const int t = threadIdx.x;
  if (t < 32) tc::tmem_alloc(&s.tmem, 128);
  if (t == 0) {
    tc::mbar_init(&s.mbar, 1);
    s.ok = 1;
  }
  load_weights(s, M);
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const int64_t row = (int64_t)blockIdx.x * MLP_TILE + t;
  float xi[6] = {0, 0, 0, 0, 0, 0};
  if (row < m)
    for (int j = 0; j < 6; j++) xi[j] = x[row * 6 + j];
  const float yo = mlp_tile_forward(s, xi, 0);
  if (row < m) y[row] = yo;
  tc::fence_before_sync();
  __syncthreads();
  if (t == 0 && !s.ok) atomicOr(status, (unsigned)ST_TIMEOUT);
  if (t < 32) tc::tmem_dealloc(s.tmem, 128);
}


// ---------------------------------------------------------------- training
// Gradient kernel.  A CTA of 8 warps takes tiles of 128 samples; sample r is
// row r of every MMA and lane r of tensor memory, and the two warps that can
// read a quadrant of 32 lanes split the 64 columns.  Two CTAs share an SM
// (208 of 256 tensor-memory columns and 63 KB each), so one computes
// element-wise while the other waits for its tensor cores.
//
// What bounds it: the element-wise passes (two exponentials and two
// reciprocals per hidden unit and sample, about 20 FP32 instructions) and the
// barriers between the five stages of a tile; the tensor pipe is nearly idle.
// So every sigmoid is taken once, its derivative kept in registers; the column
// sums (bias and output-weight gradients, FP32) are a warp butterfly that
// halves the columns a lane carries, 31 shuffles for 32 columns, accumulated
// in a register per lane over the CTA's tiles; and the weight gradients read
// the activations and deltas where the forward and backward MMAs left them, as
// MN-major operands, instead of from transposed copies.
// 2^20 samples: 2.05 ms with one CTA of 4 warps per SM, serial column sums and
// transposed copies; 0.16 ms now (a step at 2048 samples: 70 us, 16 now).
constexpr int TR_THREADS = 256;
constexpr int TR_HX = 80;    // columns of the activation tile: H1 | X
constexpr int TR_DZ = 128;   // columns of the delta tile: dZ2 | dZ1

struct TrainSmem {
  alignas(1024) uint8_t hx[MLP_TILE * TR_HX * 2];     // [H1 (64) | X (16)]   [128 x 80]
  alignas(1024) uint8_t dz[MLP_TILE * TR_DZ * 2];     // [dZ2 (64) | dZ1 (64)] [128 x 128]
  alignas(1024) uint8_t b1[MLP_HID * 16 * 2];         // W1       [64 x 16]
  alignas(1024) uint8_t b2[MLP_HID * MLP_HID * 2];    // W2       [64 x 64]
  float bias1[MLP_HID], bias2[MLP_HID], w3[MLP_HID];
  float ysum[2][MLP_TILE];
  float colsum[4][3][MLP_HID];                        // per quadrant: dW3, db2, db1
  float lsum[4], dsum[4];
  uint64_t mbar;
  uint32_t tmem;
  uint32_t ok;
};

// TMEM columns: [0,64) Z1, [64,128) Z2 then dH1, [128,208) weight gradients
constexpr int TC_Z1 = 0, TC_Z2 = 64, TC_DH1 = 64, TC_DW = 128, TC_COLS = 256;

__device__ __forceinline__ void tr_sync() {
  tc::fence_async_smem();
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
}

// sums over the warp's 32 rows of v[0..31] (destroyed): lane l gets column l's
__device__ __forceinline__ float tr_colsum(float* v) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const bool up = (lane & o) != 0;
#pragma unroll
    for (int j = 0; j < o; j++) {
      const float keep = up ? v[j + o] : v[j], send = up ? v[j] : v[j + o];
      v[j] = keep + __shfl_xor_sync(0xffffffffu, send, o);
    }
  }
  return v[0];
}

// 32 columns of row t from column c0 of a K-major tile with K columns, as BF16
__device__ __forceinline__ void tr_store32(uint8_t* tile, int t, int c0, int K, const float* v) {
#pragma unroll
  for (int q = 0; q < 4; q++) tc::st_bf16x8(tile, tc::kmajor_offset(t, c0 + 8 * q, K), v + 8 * q);
}

// the larger; a NaN if either is one
__device__ __forceinline__ float max_nan(float a, float b) {
  float m;
  asm("max.NaN.f32 %0, %1, %2;" : "=f"(m) : "f"(a), "f"(b));
  return m;
}

// silu(z) = z / q with q = 1 + exp(-z), and its derivative s (1 + z (1 - s)), s = 1 / q.
// The hardware's reciprocal (good to an ulp) and the product z s are corrected with their
// remainders, which leaves both quotients the nearest floats but for rare ties: 4
// multiply-adds.  A step of 2^20 samples: 182 us; 162 with neither corrected, at a quarter
// more error of the output weights' gradients than rounded divisions have, which take 252.
// Below -87 (where both are under 2e-36) z is held there: exp(87) keeps 1 / q normal.
__device__ __forceinline__ void silu_both(float zz, float& h, float& d) {
  const float z = max_nan(zz, -87.0f);
  const float q = 1.0f + __expf(-z), r = approx_rcp(q);
  const float s = __fmaf_rn(__fmaf_rn(-q, r, 1.0f), r, r), a = z * s;
  h = __fmaf_rn(__fmaf_rn(-a, q, z), s, a);
  d = s * __fmaf_rn(z, 1.0f - s, 1.0f);
}

// Gradient of L = sum over the batch of (y - t)^2 / n_total with respect to
// every parameter; each CTA processes tiles blockIdx.x, blockIdx.x+gridDim.x,
// ... of the batch and writes its partial sums to part[blockIdx.x][NPARAMS+1]
// (the last entry is its share of the loss).
__global__ void __launch_bounds__(TR_THREADS, 2) k_mlp_grads(const MlpDevice* M, const float* x, const float* tgt,
                                                            const int* idx, int64_t n, float inv_n, float* part,
                                                            unsigned* status) {
  extern __shared__ uint8_t smem_raw[];
  TrainSmem& s = *reinterpret_cast<TrainSmem*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const int t = threadIdx.x;
  const int warp = t >> 5, lane = t & 31;
  const int quad = warp & 3, half = warp >> 2;   // tensor-memory lanes 32 quad.., columns 32 half..
  const int row = 32 * quad + lane;              // the sample of the tile
  const int c0 = 32 * half;
  if (t < 32) tc::tmem_alloc(&s.tmem, TC_COLS);
  if (t == 0) {
    tc::mbar_init(&s.mbar, 1);
    s.ok = 1;
  }
  // weights into the operand layout, 16 bytes (8 columns) at a time
  const uint4* w1 = reinterpret_cast<const uint4*>(M->W1);
  const uint4* w2 = reinterpret_cast<const uint4*>(M->W2);
  if (t < MLP_HID * 2) *reinterpret_cast<uint4*>(s.b1 + tc::kmajor_offset(t / 2, 8 * (t % 2), 16)) = w1[t];
  for (int i = t; i < MLP_HID * MLP_HID / 8; i += TR_THREADS)
    *reinterpret_cast<uint4*>(s.b2 + tc::kmajor_offset(i / 8, 8 * (i % 8), MLP_HID)) = w2[i];
  if (t < MLP_HID) {
    s.bias1[t] = M->b1[t];
    s.bias2[t] = M->b2[t];
    s.w3[t] = __bfloat162float(M->W3[t]);
  }
  const float bias3 = M->b3;
  tr_sync();
  const uint32_t tm = s.tmem;
  const uint32_t hx = tc::smem_addr(s.hx), dz = tc::smem_addr(s.dz), sb1 = tc::smem_addr(s.b1), sb2 = tc::smem_addr(s.b2);
  const uint32_t idesc64 = tc::make_idesc(128, 64);
  const int64_t tiles = (n + MLP_TILE - 1) / MLP_TILE;
  float a_w3 = 0.0f, a_b2 = 0.0f, a_b1 = 0.0f;   // column c0 + lane, this quadrant's rows
  float a_loss = 0.0f, a_b3 = 0.0f;              // this row (half 0)
  uint32_t phase = 0;
  bool first = true;
  auto wait = [&] {
    if (!tc::mbar_wait(&s.mbar, phase)) s.ok = 0;
    phase ^= 1u;
    tc::fence_after_sync();
  };
  for (int64_t tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
    const int64_t r = tile * MLP_TILE + row;
    const bool valid = r < n;
    const int64_t src = valid ? (idx ? (int64_t)idx[r] : r) : 0;
    float xi[16] = {0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0};
    float ti = 0.0f;
    if (valid) {
      if (half == 0) {
#pragma unroll
        for (int j = 0; j < MLP_IN; j++) xi[j] = x[src * MLP_IN + j];
      }
      ti = tgt[src];
    }
    // the previous tile's weight-gradient MMAs still read the tiles
    if (!first) wait();
    if (half == 0) {
      tc::st_bf16x8(s.hx, tc::kmajor_offset(row, 64, TR_HX), xi);
      tc::st_bf16x8(s.hx, tc::kmajor_offset(row, 72, TR_HX), xi + 8);
    }
    tr_sync();
    if (t == 0) {
      tc::mma_bf16(tm + TC_Z1, tc::kmajor_desc(hx + 8 * 128, TR_HX), tc::kmajor_desc(sb1, 16), idesc64, false);
      tc::mma_commit(&s.mbar);
    }
    wait();
    // H1 = silu(Z1 + b1), its derivative kept
    float d1[32];
    {
      float z[32];
      tc::tmem_ld32(tc::tmem_lane_addr(tm, quad, TC_Z1 + c0), z);
#pragma unroll
      for (int j = 0; j < 32; j++) {
        silu_both(z[j] + s.bias1[c0 + j], z[j], d1[j]);
      }
      tr_store32(s.hx, row, c0, TR_HX, z);
    }
    tr_sync();
    if (t == 0) {
#pragma unroll
      for (int kb = 0; kb < 4; kb++)
        tc::mma_bf16(tm + TC_Z2, tc::kmajor_desc(hx + 256 * kb, TR_HX), tc::kmajor_desc(sb2 + 256 * kb, MLP_HID), idesc64,
                     kb > 0);
      tc::mma_commit(&s.mbar);
    }
    wait();
    // y from both halves' columns, residual, dy = 2 (y - t) / n_total
    float h2[32], d2[32];
    tc::tmem_ld32(tc::tmem_lane_addr(tm, quad, TC_Z2 + c0), h2);
    {
      float y = 0.0f;
#pragma unroll
      for (int j = 0; j < 32; j++) {
        const float w = s.w3[c0 + j];
        silu_both(h2[j] + s.bias2[c0 + j], h2[j], d2[j]);
        d2[j] *= w;
        y += w * h2[j];
      }
      s.ysum[half][row] = y;
    }
    __syncthreads();
    const float res = valid ? (bias3 + s.ysum[0][row] + s.ysum[1][row] - ti) : 0.0f;
    const float dy = 2.0f * res * inv_n;
    if (half == 0) {
      a_loss += res * res * inv_n;
      a_b3 += dy;
    }
    // dW3 = sum dy h2; dZ2 = dy w3 silu'(Z2 + b2), db2 = sum dZ2 in FP32 (the
    // BF16 copy is for the tensor core)
#pragma unroll
    for (int j = 0; j < 32; j++) {
      h2[j] *= dy;
      d2[j] *= dy;
    }
    tr_store32(s.dz, row, c0, TR_DZ, d2);
    tr_sync();
    // dH1 = dZ2 W2 (W2's tile read along its rows), over Z2, which is read
    if (t == 0) {
#pragma unroll
      for (int kb = 0; kb < 4; kb++)
        tc::mma_bf16(tm + TC_DH1, tc::kmajor_desc(dz + 256 * kb, TR_DZ), tc::mnmajor_desc(sb2 + 2048 * kb, MLP_HID),
                     idesc64 | tc::IDESC_B_MN, kb > 0);
      tc::mma_commit(&s.mbar);
    }
    a_w3 += tr_colsum(h2);
    a_b2 += tr_colsum(d2);
    wait();
    // dZ1 = dH1 silu'(Z1 + b1), db1 = sum dZ1
    {
      float z[32];
      tc::tmem_ld32(tc::tmem_lane_addr(tm, quad, TC_DH1 + c0), z);
#pragma unroll
      for (int j = 0; j < 32; j++) z[j] *= d1[j];
      tr_store32(s.dz, row, 64 + c0, TR_DZ, z);
      tr_sync();
      // weight gradients: D[128 x 80] += [dZ2 | dZ1]^T [H1 | X], both tiles
      // read along their rows; waited for before the tiles are written again
      if (t == 0) {
#pragma unroll
        for (int kb = 0; kb < MLP_TILE / 16; kb++)
          tc::mma_bf16(tm + TC_DW, tc::mnmajor_desc(dz + 2 * (TR_DZ / 8) * 128 * kb, TR_DZ),
                       tc::mnmajor_desc(hx + 2 * (TR_HX / 8) * 128 * kb, TR_HX),
                       tc::make_idesc(128, TR_HX) | tc::IDESC_A_MN | tc::IDESC_B_MN, !(first && kb == 0));
        tc::mma_commit(&s.mbar);
      }
      a_b1 += tr_colsum(z);
    }
    first = false;
  }
  if (!first) wait();
  // partial gradients of this CTA (it has a tile: the grid is at most their number)
  float* out = part + (size_t)blockIdx.x * (NPARAMS + 1);
  {
    // rows 0..63 x columns 0..63: dW2[o][i]; rows 64..127 x columns 64..69: dW1[i][j]
    float z[32];
    if (quad < 2) {
      tc::tmem_ld32(tc::tmem_lane_addr(tm, quad, TC_DW + c0), z);
#pragma unroll
      for (int j = 0; j < 32; j++) out[OFF_W2 + row * MLP_HID + c0 + j] = first ? 0.0f : z[j];
    } else if (half == 0) {
      tc::tmem_ld16(tc::tmem_lane_addr(tm, quad, TC_DW + 64), z);
#pragma unroll
      for (int j = 0; j < MLP_IN; j++) out[OFF_W1 + (row - 64) * MLP_IN + j] = first ? 0.0f : z[j];
    }
  }
  s.colsum[quad][0][c0 + lane] = a_w3;
  s.colsum[quad][1][c0 + lane] = a_b2;
  s.colsum[quad][2][c0 + lane] = a_b1;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    a_loss += __shfl_xor_sync(0xffffffffu, a_loss, o);
    a_b3 += __shfl_xor_sync(0xffffffffu, a_b3, o);
  }
  if (half == 0 && lane == 0) {
    s.lsum[quad] = a_loss;
    s.dsum[quad] = a_b3;
  }
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  if (t < 3 * MLP_HID) {
    const int a = t / MLP_HID, c = t % MLP_HID;
    const int off = a == 0 ? OFF_W3 : (a == 1 ? OFF_B2 : OFF_B1);
    out[off + c] = (s.colsum[0][a][c] + s.colsum[1][a][c]) + (s.colsum[2][a][c] + s.colsum[3][a][c]);
  }
  if (t == TR_THREADS - 1) {
    out[OFF_B3] = (s.dsum[0] + s.dsum[1]) + (s.dsum[2] + s.dsum[3]);
    out[NPARAMS] = (s.lsum[0] + s.lsum[1]) + (s.lsum[2] + s.lsum[3]);
    if (!s.ok) atomicOr(status, (unsigned)ST_TIMEOUT);
  }
  if (t < 32) tc::tmem_dealloc(tm, TC_COLS);
}

// The CTAs' partial gradients added in a fixed order (bit reproducible) and,
// for a training step (lr > 0), Adam (Kingma & Ba) on the FP32 master
// parameters and their BF16 copies: one launch where the sum, the step and a
// one-CTA repack took three (20 us of a 110 us step at 2048 samples).  32
// parameters per CTA; 8 groups of threads share a parameter's partials.
struct AdamStep {
  float *p, *m, *v;
  MlpDevice* packed;
  float lr, b1, b2, eps, c1, c2;
};
constexpr int RED_PARAMS = 32, RED_GROUPS = 8;
__global__ void __launch_bounds__(RED_PARAMS * RED_GROUPS) k_mlp_reduce(const float* part, int nparts, float* grads,
                                                                      AdamStep st) {
  __shared__ float red[RED_GROUPS][RED_PARAMS];
  const int lane = threadIdx.x % RED_PARAMS, g = threadIdx.x / RED_PARAMS;
  const int i = blockIdx.x * RED_PARAMS + lane;
  float a = 0.0f;
  if (i <= NPARAMS) {
    int c = g;
    for (; c + 7 * RED_GROUPS < nparts; c += 8 * RED_GROUPS) {
      float q[8];
#pragma unroll
      for (int u = 0; u < 8; u++) q[u] = part[(size_t)(c + u * RED_GROUPS) * (NPARAMS + 1) + i];
#pragma unroll
      for (int u = 0; u < 8; u++) a += q[u];
    }
    for (; c < nparts; c += RED_GROUPS) a += part[(size_t)c * (NPARAMS + 1) + i];
  }
  red[g][lane] = a;
  __syncthreads();
  if (g != 0 || i > NPARAMS) return;
#pragma unroll
  for (int q = 1; q < RED_GROUPS; q++) a += red[q][lane];
  grads[i] = a;
  if (st.lr > 0.0f && i < NPARAMS) {
    const float mi = st.b1 * st.m[i] + (1.0f - st.b1) * a;
    const float vi = st.b2 * st.v[i] + (1.0f - st.b2) * a * a;
    st.m[i] = mi;
    st.v[i] = vi;
    const float p = st.p[i] - st.lr * (mi / st.c1) / (sqrtf(vi / st.c2) + st.eps);
    st.p[i] = p;
    mlp_pack_one(i, p, st.packed);
  }
}

// normalised features and pbar from face states (rhoL, uL, pL, rhoR, uR, pR)
__global__ void k_mlp_features(double gamma, int64_t m, const float* st, float* x, float* pbar, float* pts,
                               float* ratio) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= m) return;
  const float* s = st + 6 * i;
  if (pts || ratio) {
    // the two-shock estimate the proposal corrects, and the compression
    // measure of the gate, in FP32 as the flux kernel takes them
    const GasC<float> G(gamma);
    const float cL = sqrtf(G.g * s[2] / s[0]), cR = sqrtf(G.g * s[5] / s[3]);
    const float ppv = linearised_pstar(s[0], s[1], s[2], cL, s[3], s[4], s[5], cR);
    if (pts) pts[i] = two_shock_pstar(s[0], s[1], s[2], s[3], s[4], s[5], ppv, G);
    if (ratio) ratio[i] = ppv / fmaxf(s[2], s[5]);
  }
  const float rb = 0.5f * (s[0] + s[3]);
  const float pb = 0.5f * (s[2] + s[5]);
  const float cb = sqrtf((float)gamma * pb / rb);
  float* o = x + 6 * i;
  o[0] = logf(s[0] / rb);
  o[1] = logf(s[2] / pb);
  o[2] = s[1] / cb;
  o[3] = logf(s[3] / rb);
  o[4] = logf(s[5] / pb);
  o[5] = s[4] / cb;
  if (pbar) pbar[i] = pb;
}

// exact star pressure in FP64 (Newton from the standard guess to tol); NaN
// where the states generate vacuum (no star region)
__global__ void k_riemann_pstar(double gamma, int64_t m, const float* st, double tol, int maxit, float* pstar) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= m) return;
  const float* s = st + 6 * i;
  const double rL = s[0], uL = s[1], pL = s[2], rR = s[3], uR = s[4], pR = s[5];
  const GasC<double> G(gamma);
  const double cL = sqrt(gamma * pL / rL), cR = sqrt(gamma * pR / rR);
  if (!(rL > 0.0) || !(rR > 0.0) || !(pL > 0.0) || !(pR > 0.0) || G.two_gm1 * (cL + cR) <= uR - uL) {
    pstar[i] = __int_as_float(0x7fc00000);
    return;
  }
  RiemannInfo info{0, 0, 0, 0};
  double us;
  const double p0 = standard_guess(rL, uL, pL, cL, rR, uR, pR, cR, G);
  const double p = newton_pstar(p0, rL, uL, pL, cL, rR, uR, pR, cR, G, tol, tol, maxit, info, us);
  pstar[i] = info.fail ? __int_as_float(0x7fc00000) : (float)p;
}

// training target of each face state: log(p* / p_TS), the correction of the
// two-shock estimate (FP32, as the flux kernel forms it) that takes it to the
// exact star pressure (FP64 Newton to tol); NaN without a star region
__global__ void k_mlp_targets(double gamma, int64_t m, const float* st, double tol, int maxit, float* target) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= m) return;
  const float* s = st + 6 * i;
  const double rL = s[0], uL = s[1], pL = s[2], rR = s[3], uR = s[4], pR = s[5];
  const GasC<double> G(gamma);
  const double cL = sqrt(gamma * pL / rL), cR = sqrt(gamma * pR / rR);
  if (!(rL > 0.0) || !(rR > 0.0) || !(pL > 0.0) || !(pR > 0.0) || G.two_gm1 * (cL + cR) <= uR - uL) {
    target[i] = __int_as_float(0x7fc00000);
    return;
  }
  RiemannInfo info{0, 0, 0, 0};
  double us;
  const double p0 = standard_guess(rL, uL, pL, cL, rR, uR, pR, cR, G);
  const double p = newton_pstar(p0, rL, uL, pL, cL, rR, uR, pR, cR, G, tol, tol, maxit, info, us);
  const GasC<float> Gf(gamma);
  const float cLf = sqrtf(Gf.g * s[2] / s[0]), cRf = sqrtf(Gf.g * s[5] / s[3]);
  const float ppv = linearised_pstar(s[0], s[1], s[2], cLf, s[3], s[4], s[5], cRf);
  const float pts = two_shock_pstar(s[0], s[1], s[2], s[3], s[4], s[5], ppv, Gf);
  target[i] = (info.fail || !(pts > 0.0f)) ? __int_as_float(0x7fc00000) : (float)log(p / (double)pts);
}

}  // namespace amm

// ============================================================ C ABI
struct amm_mlp {
  double gamma = 5.0 / 3.0;
  cudaStream_t stream = nullptr;
  char* block = nullptr;              // holds the arrays below but `partial`
  float* params = nullptr;            // FP32 master parameters [NPARAMS]
  amm::MlpDevice* packed = nullptr;   // BF16 weights for the kernels
  unsigned* status = nullptr;
  // training state
  float* adam_m = nullptr;
  float* adam_v = nullptr;
  float* grads = nullptr;             // [NPARAMS]
  float* partial = nullptr;           // per-CTA gradient partials
  int partial_ctas = 0;
  int64_t adam_t = 0;
  std::string err;
};

namespace {
int mfail(amm_mlp* m, int code, const std::string& msg) {
  if (m) m->err = msg;
  return code;
}
#define MCU(call)                                                                          \
  do {                                                                                     \
    cudaError_t e_ = (call);                                                               \
    if (e_ != cudaSuccess) return mfail(m, AMM_ERR_CUDA, std::string(#call) + ": " + cudaGetErrorString(e_)); \
  } while (0)

size_t mlp_smem_bytes() { return sizeof(amm::MlpSmem) + 1024; }
size_t train_smem_bytes() { return sizeof(amm::TrainSmem) + 1024; }

// Allocates the handle's arrays, all in one block, and clears them before it returns.
// (cudaMemset runs on the legacy stream, which a non-blocking stream of the handle is not
// ordered after: behind other work there the clear could land on weights already set.  On
// the handle's stream it would be taken into a graph that the caller captures.)
cudaError_t alloc_cleared(amm_mlp* m) {
  size_t bytes = 0;
  const auto part = [&](size_t b) {
    const size_t at = bytes;
    bytes += (b + 255) / 256 * 256;
    return at;
  };
  const size_t np = sizeof(float) * (amm::NPARAMS + 1);
  const size_t packed = part(sizeof(amm::MlpDevice)), params = part(np), adam_m = part(np), adam_v = part(np), grads = part(np),
               status = part(sizeof(unsigned));
  cudaError_t e = cudaMalloc(&m->block, bytes);
  if (e != cudaSuccess) return e;
  cudaStream_t st = nullptr;
  if ((e = cudaStreamCreateWithFlags(&st, cudaStreamNonBlocking)) != cudaSuccess) return e;
  e = cudaMemsetAsync(m->block, 0, bytes, st);
  const cudaError_t w = cudaStreamSynchronize(st);
  cudaStreamDestroy(st);
  m->packed = reinterpret_cast<amm::MlpDevice*>(m->block + packed);
  m->params = reinterpret_cast<float*>(m->block + params);
  m->adam_m = reinterpret_cast<float*>(m->block + adam_m);
  m->adam_v = reinterpret_cast<float*>(m->block + adam_v);
  m->grads = reinterpret_cast<float*>(m->block + grads);
  m->status = reinterpret_cast<unsigned*>(m->block + status);
  return e != cudaSuccess ? e : w;
}

int ensure_train(amm_mlp* m, int ctas) {
  if (m->partial_ctas < ctas) {
    if (m->partial) cudaFree(m->partial);
    m->partial = nullptr;
    MCU(cudaMalloc(&m->partial, sizeof(float) * (amm::NPARAMS + 1) * (size_t)ctas));
    m->partial_ctas = ctas;
  }
  return AMM_OK;
}

// gradients of the batch into m->grads (device), loss in m->grads[NPARAMS];
// lr > 0: also an Adam step with them
int run_grads(amm_mlp* m, const float* x, const float* t, const int* idx, int64_t n, float lr) {
  int dev = 0, sms = 148;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const int64_t tiles = (n + amm::MLP_TILE - 1) / amm::MLP_TILE;
  const int ctas = (int)std::min<int64_t>(tiles, 2 * (int64_t)sms);   // two per SM
  int rc = ensure_train(m, ctas);
  if (rc != AMM_OK) return rc;
  amm::k_mlp_grads<<<ctas, amm::TR_THREADS, train_smem_bytes(), m->stream>>>(m->packed, x, t, idx, n, 1.0f / (float)n,
                                                                          m->partial, m->status);
  MCU(cudaGetLastError());
  amm::AdamStep st{m->params, m->adam_m, m->adam_v, m->packed, lr, 0.9f, 0.999f, 1e-8f, 1.0f, 1.0f};
  if (lr > 0.0f) {
    m->adam_t++;
    st.c1 = 1.0f - powf(st.b1, (float)m->adam_t);
    st.c2 = 1.0f - powf(st.b2, (float)m->adam_t);
  }
  amm::k_mlp_reduce<<<(amm::NPARAMS + amm::RED_PARAMS) / amm::RED_PARAMS, amm::RED_PARAMS * amm::RED_GROUPS, 0,
                      m->stream>>>(m->partial, ctas, m->grads, st);
  MCU(cudaGetLastError());
  return AMM_OK;
}
}  // namespace

extern "C" {

int amm_mlp_create(amm_mlp** out, double gamma, void* stream) {
  if (!out || !(gamma > 1.0)) return AMM_ERR_INVALID_ARG;
  *out = nullptr;
  amm_mlp* m = new amm_mlp();
  m->gamma = gamma;
  m->stream = (cudaStream_t)stream;
  auto bail = [&](int rc) {
    if (m->block) cudaFree(m->block);
    delete m;
    return rc;
  };
  if (alloc_cleared(m) != cudaSuccess) return bail(AMM_ERR_CUDA);
  if (cudaFuncSetAttribute(amm::k_mlp_forward, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)mlp_smem_bytes()) !=
      cudaSuccess)
    return bail(AMM_ERR_CUDA);
  if (cudaFuncSetAttribute(amm::k_mlp_grads, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)train_smem_bytes()) !=
      cudaSuccess)
    return bail(AMM_ERR_CUDA);
  *out = m;
  return AMM_OK;
}

void amm_mlp_destroy(amm_mlp* m) {
  if (!m) return;
  cudaStreamSynchronize(m->stream);
  void* ptrs[] = {m->block, m->partial};
  for (void* p : ptrs)
    if (p) cudaFree(p);
  delete m;
}

const char* amm_mlp_last_error(const amm_mlp* m) { return m ? m->err.c_str() : "null handle"; }

int amm_mlp_num_params(void) { return amm::NPARAMS; }

int amm_mlp_set_params(amm_mlp* m, const float* params) {
  if (!m || !params) return mfail(m, AMM_ERR_INVALID_ARG, "null argument");
  for (int i = 0; i < amm::NPARAMS; i++)
    if (!std::isfinite(params[i])) return mfail(m, AMM_ERR_INVALID_ARG, "non-finite parameter");
  MCU(cudaMemcpyAsync(m->params, params, sizeof(float) * amm::NPARAMS, cudaMemcpyHostToDevice, m->stream));
  amm::k_mlp_pack<<<(amm::NPARAMS + 255) / 256, 256, 0, m->stream>>>(m->params, m->packed);
  MCU(cudaGetLastError());
  MCU(cudaStreamSynchronize(m->stream));
  return AMM_OK;
}

int amm_mlp_get_params(amm_mlp* m, float* params) {
  if (!m || !params) return mfail(m, AMM_ERR_INVALID_ARG, "null argument");
  MCU(cudaMemcpyAsync(params, m->params, sizeof(float) * amm::NPARAMS, cudaMemcpyDeviceToHost, m->stream));
  MCU(cudaStreamSynchronize(m->stream));
  return AMM_OK;
}

int amm_mlp_forward(amm_mlp* m, const float* x_device, int64_t n, float* y_device) {
  if (!m || !x_device || !y_device || n < 1) return mfail(m, AMM_ERR_INVALID_ARG, "bad argument");
  const int64_t tiles = (n + amm::MLP_TILE - 1) / amm::MLP_TILE;
  amm::k_mlp_forward<<<(unsigned)tiles, amm::MLP_TILE, mlp_smem_bytes(), m->stream>>>(m->packed, x_device, n,
                                                                                     y_device, m->status);
  MCU(cudaGetLastError());
  unsigned st = 0;
  MCU(cudaMemcpyAsync(&st, m->status, sizeof(st), cudaMemcpyDeviceToHost, m->stream));
  MCU(cudaStreamSynchronize(m->stream));
  if (st) return mfail(m, AMM_ERR_TIMEOUT, "tensor-core wait timed out");
  return AMM_OK;
}

int amm_mlp_grads(amm_mlp* m, const float* x_device, const float* t_device, const int32_t* idx_device, int64_t n,
                  float* grads, float* loss) {
  if (!m || !x_device || !t_device || n < 1 || !grads) return mfail(m, AMM_ERR_INVALID_ARG, "bad argument");
  int rc = run_grads(m, x_device, t_device, idx_device, n, 0.0f);
  if (rc != AMM_OK) return rc;
  std::vector<float> g(amm::NPARAMS + 1);
  unsigned st = 0;
  MCU(cudaMemcpyAsync(g.data(), m->grads, sizeof(float) * g.size(), cudaMemcpyDeviceToHost, m->stream));
  MCU(cudaMemcpyAsync(&st, m->status, sizeof(st), cudaMemcpyDeviceToHost, m->stream));
  MCU(cudaStreamSynchronize(m->stream));
  if (st) return mfail(m, AMM_ERR_TIMEOUT, "tensor-core wait timed out");
  for (int i = 0; i < amm::NPARAMS; i++) grads[i] = g[i];
  if (loss) *loss = g[amm::NPARAMS];
  return AMM_OK;
}

int amm_mlp_train_step(amm_mlp* m, const float* x_device, const float* t_device, const int32_t* idx_device, int64_t n,
                       float lr, float* loss_device) {
  if (!m || !x_device || !t_device || n < 1 || !(lr > 0.0f)) return mfail(m, AMM_ERR_INVALID_ARG, "bad argument");
  int rc = run_grads(m, x_device, t_device, idx_device, n, lr);
  if (rc != AMM_OK) return rc;
  if (loss_device)
    MCU(cudaMemcpyAsync(loss_device, m->grads + amm::NPARAMS, sizeof(float), cudaMemcpyDeviceToDevice, m->stream));
  return AMM_OK;
}

int amm_mlp_sync(amm_mlp* m) {
  if (!m) return AMM_ERR_INVALID_ARG;
  unsigned st = 0;
  MCU(cudaMemcpyAsync(&st, m->status, sizeof(st), cudaMemcpyDeviceToHost, m->stream));
  MCU(cudaStreamSynchronize(m->stream));
  if (st) return mfail(m, AMM_ERR_TIMEOUT, "tensor-core wait timed out");
  return AMM_OK;
}

int amm_mlp_attach(amm_ctx* c, const amm_mlp* m) {
  if (!c || !m) return AMM_ERR_INVALID_ARG;
  if (c->opt.precision != AMM_FP32_LEARNED) {
    c->err = "amm_mlp_attach: the context is not of the FP32 learned form";
    return AMM_ERR_INVALID_ARG;
  }
  if (!c->mlp && cudaMalloc(&c->mlp, sizeof(amm::MlpDevice)) != cudaSuccess) {
    c->err = "amm_mlp_attach: cudaMalloc failed";
    return AMM_ERR_CUDA;
  }
  // the list of faces past the proposal's gate (room for every face)
  if (!c->defer_list && (cudaMalloc((void**)&c->defer_list, sizeof(int2) * (size_t)std::max<int64_t>(c->nf_cap, 1)) !=
                             cudaSuccess ||
                         cudaMalloc((void**)&c->defer_count, sizeof(unsigned)) != cudaSuccess)) {
    c->err = "amm_mlp_attach: cudaMalloc failed";
    return AMM_ERR_CUDA;
  }
  if (cudaMemcpyAsync(c->mlp, m->packed, sizeof(amm::MlpDevice), cudaMemcpyDeviceToDevice, m->stream) != cudaSuccess ||
      cudaStreamSynchronize(m->stream) != cudaSuccess || amm::prepare_flux_learned() != cudaSuccess) {
    c->err = "amm_mlp_attach: copy failed";
    return AMM_ERR_CUDA;
  }
  c->mlp_loaded = true;
  if (c->graph) {
    cudaGraphExecDestroy(c->graph);
    c->graph = nullptr;
  }
  return AMM_OK;
}

int amm_mlp_features(double gamma, int64_t n, const float* states_device, float* x_device, float* pbar_device,
                     float* pts_device, float* ratio_device, void* stream) {
  if (!(gamma > 1.0) || n < 1 || !states_device || !x_device) return AMM_ERR_INVALID_ARG;
  amm::k_mlp_features<<<(unsigned)((n + 255) / 256), 256, 0, (cudaStream_t)stream>>>(
      gamma, n, states_device, x_device, pbar_device, pts_device, ratio_device);
  return cudaGetLastError() == cudaSuccess ? AMM_OK : AMM_ERR_CUDA;
}

int amm_mlp_targets(double gamma, int64_t n, const float* states_device, double tol, float* target_device,
                    void* stream) {
  if (!(gamma > 1.0) || n < 1 || !states_device || !target_device || !(tol > 0.0)) return AMM_ERR_INVALID_ARG;
  amm::k_mlp_targets<<<(unsigned)((n + 255) / 256), 256, 0, (cudaStream_t)stream>>>(gamma, n, states_device, tol, 200,
                                                                                   target_device);
  return cudaGetLastError() == cudaSuccess ? AMM_OK : AMM_ERR_CUDA;
}

int amm_riemann_pstar(double gamma, int64_t n, const float* states_device, double tol, float* pstar_device,
                      void* stream) {
  if (!(gamma > 1.0) || n < 1 || !states_device || !pstar_device || !(tol > 0.0)) return AMM_ERR_INVALID_ARG;
  amm::k_riemann_pstar<<<(unsigned)((n + 255) / 256), 256, 0, (cudaStream_t)stream>>>(gamma, n, states_device, tol,
                                                                                     200, pstar_device);
  return cudaGetLastError() == cudaSuccess ? AMM_OK : AMM_ERR_CUDA;
}

}  // extern "C"
