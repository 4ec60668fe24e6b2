// mlp.cu -- training and stand-alone inference of the learned reconstruction weights on the
// tensor cores (BF16 operands, FP32 accumulation), and Adam on FP32 master parameters.
//
// Loss of a batch of n stencils: mean_b (sum_k omega_k qhat_k - that_b)^2, with x, qhat and the
// target that in the normalised units of each stencil (x = (v - v_2)/amp).  The backward pass
// propagates through softmax, the four dense layers and gelu; weight gradients
// dW_l = dZ_l^T H_{l-1} are tensor-core products over the samples that a block has at a time, each
// warp accumulating its quarter of every matrix, added to the global FP32 gradient with one atomic
// per parameter and block.
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>
#include <stdio.h>

#include "ibfsa_internal.h"
#include "mlp_tile.cuh"

namespace ibfsa {
namespace mlp {

// training state (device): floats [master | m | v | grad] (NPAD each), loss, then the packed image
constexpr int NPAD = 2432;
constexpr size_t OFF_MASTER = 0, OFF_M = NPAD, OFF_V = 2 * NPAD, OFF_GRAD = 3 * NPAD,
                 OFF_LOSS = 4 * NPAD;
constexpr size_t STATE_FLOATS = 4 * NPAD + 64;
constexpr size_t OFF_IMAGE_BYTES = STATE_FLOATS * sizeof(float);
constexpr size_t STATE_BYTES = OFF_IMAGE_BYTES + PACKED_BYTES;

constexpr int TRAIN_WARPS = 4, TRAIN_BLOCKS = 4;  // warps of a block, blocks of a multiprocessor

__device__ __forceinline__ float bf16r(float x) {
  return __bfloat162float(__float2bfloat16_rn(x));
}

// packed image from the FP32 master parameters (all parameters rounded to bf16)
__global__ void k_pack(const float *__restrict__ th, unsigned char *__restrict__ img) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  __nv_bfloat16 *W1 = (__nv_bfloat16 *)(img + OFF_W1), *W2 = (__nv_bfloat16 *)(img + OFF_W2);
  __nv_bfloat16 *W3 = (__nv_bfloat16 *)(img + OFF_W3), *W4 = (__nv_bfloat16 *)(img + OFF_W4);
  __nv_bfloat16 *W2T = (__nv_bfloat16 *)(img + OFF_W2T), *W3T = (__nv_bfloat16 *)(img + OFF_W3T);
  __nv_bfloat16 *W4T = (__nv_bfloat16 *)(img + OFF_W4T);
  float *B1 = (float *)(img + OFF_B1), *B2 = (float *)(img + OFF_B2);
  float *B3 = (float *)(img + OFF_B3), *B4 = (float *)(img + OFF_B4);
  if (i < 32 * 16) {  // W1 [32][16]
    int r = i / 16, c = i % 16;
    W1[i] = __float2bfloat16_rn(c < 5 ? th[P_W1 + r * 5 + c] : 0.f);
  }
  if (i < 32 * 32) {
    int r = i / 32, c = i % 32;
    W2[i] = __float2bfloat16_rn(th[P_W2 + i]);
    W3[i] = __float2bfloat16_rn(th[P_W3 + i]);
    W2T[i] = __float2bfloat16_rn(th[P_W2 + c * 32 + r]);
    W3T[i] = __float2bfloat16_rn(th[P_W3 + c * 32 + r]);
  }
  if (i < 8 * 32) {  // W4 [8][32]
    int r = i / 32;
    W4[i] = __float2bfloat16_rn(r < 3 ? th[P_W4 + i] : 0.f);
  }
  if (i < 32 * 16) {  // W4T [32][16]: row = hidden unit, col = logit
    int r = i / 16, c = i % 16;
    W4T[i] = __float2bfloat16_rn(c < 3 ? th[P_W4 + c * 32 + r] : 0.f);
  }
  if (i < 32) {
    B1[i] = bf16r(th[P_B1 + i]);
    B2[i] = bf16r(th[P_B2 + i]);
    B3[i] = bf16r(th[P_B3 + i]);
  }
  if (i < 8) B4[i] = i < 3 ? bf16r(th[P_B4 + i]) : 0.f;
}

// --- backward pass --------------------------------------------------------------------------
// A warp's tile as the weight gradients read it, sample by sample: dz1, dz2, dz3, h1, h2, h3
// (rows of 32 units in 80 bytes) and a last matrix of the inputs (columns 0..7) and dz4 (8..15) in
// rows of 48 bytes.  With these strides 8 rows x 16 bytes lie in 32 different banks.
constexpr int ROW32 = 80, ROWX = 48, MAT = 16 * ROW32;
constexpr int DZ = 0, HID = 3 * MAT, XZ = 6 * MAT, TILE_BYTES = XZ + 16 * ROWX;

// a 16x32 operand (two k-step A fragments) into rows of 80 bytes
__device__ __forceinline__ void put32(unsigned char *m, const uint32_t A[2][4], int g, int t) {
#pragma unroll
  for (int s = 0; s < 2; s++)
#pragma unroll
    for (int r = 0; r < 4; r++)
      *reinterpret_cast<uint32_t *>(m + (g + 8 * (r & 1)) * ROW32 + 32 * s + 16 * (r >> 1) + 4 * t) =
          A[s][r];
}

// 16 samples x 16 columns, transposed on the way: v[0] columns 0..7 and v[1] columns 8..15 of
// samples 0..7, v[2] and v[3] of samples 8..15: v is the A operand (columns x samples), and
// (v[0], v[2]) and (v[1], v[3]) are B operands (samples x columns).
__device__ __forceinline__ void get16(uint32_t v[4], const unsigned char *m, int row_bytes,
                                      int lane) {
  const uint32_t a = (uint32_t)__cvta_generic_to_shared(
      m + ((lane & 7) + 8 * (lane >> 4)) * row_bytes + 16 * ((lane >> 3) & 1));
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];\n"
               : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3])
               : "r"(a)
               : "memory");
}

// dH (16 x 32) = dZ (16 x 32) W (32 x 32), W given transposed (row = input unit)
__device__ __forceinline__ void backprop32(float dh[4][4], const uint32_t A[2][4],
                                           const unsigned char *img, int offWT, int g, int t) {
#pragma unroll
  for (int j = 0; j < 4; j++) {
    dh[j][0] = dh[j][1] = dh[j][2] = dh[j][3] = 0.f;
#pragma unroll
    for (int s = 0; s < 2; s++) {
      uint32_t w0 = ldw(img, offWT, LD32, 8 * j + g, 16 * s + 2 * t);
      uint32_t w1 = ldw(img, offWT, LD32, 8 * j + g, 16 * s + 2 * t + 8);
      mma16816(dh[j], A[s], w0, w1);
    }
  }
}

__device__ __forceinline__ void pack_C_as_A(const float c[4][4], uint32_t A[2][4]) {
#pragma unroll
  for (int s = 0; s < 2; s++) {
    A[s][0] = pack2(c[2 * s][0], c[2 * s][1]);
    A[s][1] = pack2(c[2 * s][2], c[2 * s][3]);
    A[s][2] = pack2(c[2 * s + 1][0], c[2 * s + 1][1]);
    A[s][3] = pack2(c[2 * s + 1][2], c[2 * s + 1][3]);
  }
}

// the sum over the 16 samples of one of a 16x32 tile's columns, another for each lane: column
// 8 (2 bit2(g) + bit1(g)) + 2t + bit0(g).  Halving: a lane sends the half that it does not keep.
__device__ __forceinline__ float column_sum(const float c[4][4], int lane) {
  float v[8];
#pragma unroll
  for (int j = 0; j < 4; j++) {
    v[2 * j] = c[j][0] + c[j][2];
    v[2 * j + 1] = c[j][1] + c[j][3];
  }
#pragma unroll
  for (int h = 4; h > 0; h >>= 1) {
    const bool up = lane & (4 * h);
#pragma unroll
    for (int k = 0; k < h; k++) {
      const float keep = up ? v[k + h] : v[k], send = up ? v[k] : v[k + h];
      v[k] = keep + __shfl_xor_sync(0xffffffffu, send, 4 * h);
    }
  }
  return v[0];
}

// loads one stencil row (raw values), its normalised form, candidates and normalised target
__device__ __forceinline__ bool load_row(const float *S, const float *T, int n, unsigned m, float x[5],
                                         float q[3], float &tn) {
  float v[5] = {0.f, 0.f, 0.f, 0.f, 0.f};
  bool ok = m < (unsigned)n;
  if (ok)
#pragma unroll
    for (int j = 0; j < 5; j++) v[j] = S[(size_t)m * 5 + j];
  float amp = normalise(v, x);
  candidates(x, q);
  tn = 0.f;
  bool live = amp > 1e-30f;  // the same cut as normalise: no overflow from denormal amplitudes
  if (ok && T && live) tn = (T[m] - v[2]) / amp;
  return ok && live;
}

// Bound by what a warp issues (2600 instructions for 16 samples, half of them the 1536 tanh) at the
// latency of its chain of small products, tanh and exchanges: the issue slots are 51 % taken, 24
// bytes a sample are read.  Accumulators of whole matrices took 100 registers a thread, 4 or 8 warps
// a multiprocessor, and shared-memory atomics to sum over a block's warps.  Here a warp takes 16
// samples through the network and back, leaves its operands in shared memory, and after a barrier
// accumulates a quarter of each matrix over the block's 64 samples: 20 registers, 16 warps a
// multiprocessor, and no sum over warps but that of the biases.  65,536 samples: 47 -> 22 us.
__global__ void __launch_bounds__(32 * TRAIN_WARPS, TRAIN_BLOCKS)
    k_train(const unsigned char *__restrict__ gimg, int n, const float *__restrict__ S,
            const float *__restrict__ T, float inv_n, float *__restrict__ grad,
            float *__restrict__ loss) {
  __shared__ __align__(16) unsigned char img[STAGED_BYTES];
  __shared__ __align__(16) unsigned char tiles_of[TRAIN_WARPS][TILE_BYTES];
  stage_image<true>(img, gimg);
  __syncthreads();
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, g = lane >> 2, t = lane & 3;
  // this warp's share: units 16 (w/2).. x inputs 16 (w%2).. of dW3 and dW2; half w%2 of dW1
  // (warps 0, 1) or of dW4, there as h3^T dz4 (warps 2, 3)
  float a3[2][4] = {}, a2[2][4] = {}, ax[4] = {};
  float db1 = 0.f, db2 = 0.f, db3 = 0.f, db4a = 0.f, db4b = 0.f, lsum = 0.f;
  const int groups = n / (16 * TRAIN_WARPS) + (n % (16 * TRAIN_WARPS) != 0);
  for (int group = blockIdx.x; group < groups; group += gridDim.x) {
    unsigned char *my = tiles_of[w];
    float dz[4][4], z1[4][4], z2[4][4], z3[4][4];
    uint32_t A[2][4];
    float d4a[3] = {0.f, 0.f, 0.f}, d4b[3] = {0.f, 0.f, 0.f};
    {
      // rows past n come as zeros and with no residual
      const unsigned ma = ((unsigned)group * TRAIN_WARPS + w) * 16 + g, mb = ma + 8;
      float xa[5], xb[5], qa[3], qb[3], ta, tb, z4[4], wa[3], wb[3];
      bool va = load_row(S, T, n, ma, xa, qa, ta), vb = load_row(S, T, n, mb, xb, qb, tb);
      uint32_t A0[2];
      input_fragment(xa, xb, t, A0);
      *reinterpret_cast<uint32_t *>(my + XZ + g * ROWX + 4 * t) = A0[0];
      *reinterpret_cast<uint32_t *>(my + XZ + (g + 8) * ROWX + 4 * t) = A0[1];
      dense8(z1, A0, img, g, t);
      gelu_pack<true>(z1, A);
      put32(my + HID, A, g, t);
      dense32(z2, A, img, S_W2, S_B2, g, t);
      gelu_pack<true>(z2, A);
      put32(my + HID + MAT, A, g, t);
      dense32(z3, A, img, S_W3, S_B3, g, t);
      gelu_pack<true>(z3, A);
      put32(my + HID + 2 * MAT, A, g, t);
      logits(z4, A, img, g, t);
      softmax3(z4, wa, wb);
      // loss and d(logits) for rows g and g+8 (lane t == 0 holds the weights)
      if (t == 0) {
        float fa = wa[0] * qa[0] + wa[1] * qa[1] + wa[2] * qa[2];
        float fb = wb[0] * qb[0] + wb[1] * qb[1] + wb[2] * qb[2];
        float ra = va ? fa - ta : 0.f, rb = vb ? fb - tb : 0.f;
        lsum += ra * ra + rb * rb;
        float dfa = 2.f * ra * inv_n, dfb = 2.f * rb * inv_n;
        float sa = 0.f, sb = 0.f;
#pragma unroll
        for (int k = 0; k < 3; k++) {
          sa += wa[k] * dfa * qa[k];
          sb += wb[k] * dfb * qb[k];
        }
#pragma unroll
        for (int k = 0; k < 3; k++) {
          d4a[k] = wa[k] * (dfa * qa[k] - sa);
          d4b[k] = wb[k] * (dfb * qb[k] - sb);
        }
      }
    }
    // dz4 in C layout of the 16x8 logit tile: lane t holds logits 2t, 2t+1
    {
      float x2 = __shfl_sync(0xffffffffu, d4a[2], lane & ~3);
      float y2 = __shfl_sync(0xffffffffu, d4b[2], lane & ~3);
      float c0 = t == 0 ? d4a[0] : (t == 1 ? x2 : 0.f), c1 = t == 0 ? d4a[1] : 0.f;
      float c2 = t == 0 ? d4b[0] : (t == 1 ? y2 : 0.f), c3 = t == 0 ? d4b[1] : 0.f;
      db4a += c0 + c2;
      db4b += c1 + c3;
      const uint32_t u0 = pack2(c0, c1), u1 = pack2(c2, c3);
      *reinterpret_cast<uint32_t *>(my + XZ + g * ROWX + 16 + 4 * t) = u0;
      *reinterpret_cast<uint32_t *>(my + XZ + (g + 8) * ROWX + 16 + 4 * t) = u1;
      // dh3 = dz4 W4
#pragma unroll
      for (int j = 0; j < 4; j++) {
        dz[j][0] = dz[j][1] = dz[j][2] = dz[j][3] = 0.f;
        mma1688(dz[j], u0, u1, ldw(img, S_W4T, LD8, 8 * j + g, 2 * t));
      }
    }
#pragma unroll
    for (int j = 0; j < 4; j++)
#pragma unroll
      for (int r = 0; r < 4; r++) dz[j][r] *= z3[j][r];  // z now holds gelu's derivative
    pack_C_as_A(dz, A);
    put32(my + DZ + 2 * MAT, A, g, t);
    db3 += column_sum(dz, lane);
    backprop32(dz, A, img, S_W3T, g, t);
#pragma unroll
    for (int j = 0; j < 4; j++)
#pragma unroll
      for (int r = 0; r < 4; r++) dz[j][r] *= z2[j][r];
    pack_C_as_A(dz, A);
    put32(my + DZ + MAT, A, g, t);
    db2 += column_sum(dz, lane);
    backprop32(dz, A, img, S_W2T, g, t);
#pragma unroll
    for (int j = 0; j < 4; j++)
#pragma unroll
      for (int r = 0; r < 4; r++) dz[j][r] *= z1[j][r];
    pack_C_as_A(dz, A);
    put32(my + DZ, A, g, t);
    db1 += column_sum(dz, lane);
    __syncthreads();
#pragma unroll
    for (int k = 0; k < TRAIN_WARPS; k++) {
      const unsigned char *m = tiles_of[k];
      const int unit = 32 * (w >> 1), input = 32 * (w & 1);  // bytes
      uint32_t a[4], b[4];
      get16(a, m + DZ + 2 * MAT + unit, ROW32, lane);
      get16(b, m + HID + MAT + input, ROW32, lane);
      mma16816(a3[0], a, b[0], b[2]);
      mma16816(a3[1], a, b[1], b[3]);
      get16(a, m + DZ + MAT + unit, ROW32, lane);
      get16(b, m + HID + input, ROW32, lane);
      mma16816(a2[0], a, b[0], b[2]);
      mma16816(a2[1], a, b[1], b[3]);
      get16(a, m + (w < 2 ? DZ : HID + 2 * MAT) + input, ROW32, lane);
      get16(b, m + XZ, ROWX, lane);
      mma16816(ax, a, w < 2 ? b[0] : b[1], w < 2 ? b[2] : b[3]);
    }
    __syncthreads();
  }
  // ---- the block's gradient, in the place of the tiles, then added to the global one
  float *acc = reinterpret_cast<float *>(tiles_of);
  float(*dbs)[128] = reinterpret_cast<float(*)[128]>(acc + NPAD);
  static_assert(sizeof(float) * (NPAD + 128 * TRAIN_WARPS) <= TRAIN_WARPS * TILE_BYTES, "");
  // C element r of a product: row g (+8 with r & 2), column 2t (+1 with r & 1)
#pragma unroll
  for (int r = 0; r < 4; r++) {
    const int row = g + 8 * (r >> 1), col = 2 * t + (r & 1);
#pragma unroll
    for (int k = 0; k < 2; k++) {
      const int i = (16 * (w >> 1) + row) * 32 + 16 * (w & 1) + 8 * k + col;
      acc[P_W3 + i] = a3[k][r];
      acc[P_W2 + i] = a2[k][r];
    }
    const int unit = 16 * (w & 1) + row;
    if (w < 2 && col < 5) acc[P_W1 + unit * 5 + col] = ax[r];
    if (w >= 2 && col < 3) acc[P_W4 + col * 32 + unit] = ax[r];
  }
  const int column = 8 * (lane >> 3) + 2 * t + ((lane >> 2) & 1);  // of column_sum
  dbs[w][column] = db1;
  dbs[w][32 + column] = db2;
  dbs[w][64 + column] = db3;
  for (int o = 4; o < 32; o <<= 1) {
    db4a += __shfl_xor_sync(0xffffffffu, db4a, o);
    db4b += __shfl_xor_sync(0xffffffffu, db4b, o);
    lsum += __shfl_xor_sync(0xffffffffu, lsum, o);
  }
  if (lane < 2) {  // lane t of g = 0: logits 2t, 2t+1
    dbs[w][96 + 2 * lane] = db4a;
    dbs[w][97 + 2 * lane] = db4b;
  }
  if (lane == 0) dbs[w][100] = lsum;
  __syncthreads();
  if (threadIdx.x < 101) {
    float s = 0.f;
#pragma unroll
    for (int k = 0; k < TRAIN_WARPS; k++) s += dbs[k][threadIdx.x];
    const int l = threadIdx.x >> 5, u = threadIdx.x & 31;
    if (threadIdx.x == 100)
      atomicAdd(loss, s * inv_n);
    else if (l < 3 || u < 3)
      acc[(l == 0 ? P_B1 : l == 1 ? P_B2 : l == 2 ? P_B3 : P_B4) + u] = s;
  }
  __syncthreads();
  for (int i = threadIdx.x; i < NPARAM; i += blockDim.x) atomicAdd(&grad[i], acc[i]);
}

__global__ void k_adam(float *__restrict__ th, float *__restrict__ m, float *__restrict__ v,
                       const float *__restrict__ grad, float lr, float b1, float b2, float eps,
                       float c1, float c2) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= NPARAM) return;
  float gi = grad[i];
  float mi = b1 * m[i] + (1.f - b1) * gi;
  float vi = b2 * v[i] + (1.f - b2) * gi * gi;
  m[i] = mi;
  v[i] = vi;
  th[i] -= lr * (mi * c1) / (sqrtf(vi * c2) + eps);
}

// stand-alone inference: face values, weights and (with targets) the mean squared loss
__global__ void __launch_bounds__(256) k_eval(const unsigned char *__restrict__ gimg, int n,
                                              const float *__restrict__ S,
                                              const float *__restrict__ T, float *__restrict__ face,
                                              float *__restrict__ omega, float inv_n,
                                              float *__restrict__ loss) {
  __shared__ __align__(16) unsigned char img[STAGED_BYTES];
  stage_image<false>(img, gimg);
  __syncthreads();
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, g = lane >> 2, t = lane & 3;
  const int warps = blockDim.x >> 5;
  float lsum = 0.f;
  for (int tile = blockIdx.x * warps + w; tile < (n + 15) / 16; tile += gridDim.x * warps) {
    int ma = tile * 16 + g, mb = ma + 8;
    float xa[5], xb[5], qa[3], qb[3], ta, tb;
    bool va = load_row(S, T, n, ma, xa, qa, ta), vb = load_row(S, T, n, mb, xb, qb, tb);
    float z[4][4], z4[4], wa[3], wb[3];
    uint32_t A0[2], A[2][4];
    input_fragment(xa, xb, t, A0);
    dense8(z, A0, img, g, t);
    gelu_pack<false>(z, A);
    dense32(z, A, img, S_W2, S_B2, g, t);
    gelu_pack<false>(z, A);
    dense32(z, A, img, S_W3, S_B3, g, t);
    gelu_pack<false>(z, A);
    logits(z4, A, img, g, t);
    softmax3(z4, wa, wb);
    if (t == 0) {
      float fa = wa[0] * qa[0] + wa[1] * qa[1] + wa[2] * qa[2];
      float fb = wb[0] * qb[0] + wb[1] * qb[1] + wb[2] * qb[2];
      if (ma < n) {
        float v2 = S[(size_t)ma * 5 + 2], amp = 0.f;
        for (int j = 0; j < 5; j++) amp = fmaxf(amp, fabsf(S[(size_t)ma * 5 + j] - v2));
        if (face) face[ma] = v2 + amp * fa;
        if (omega)
          for (int k = 0; k < 3; k++) omega[(size_t)ma * 3 + k] = wa[k];
        if (va && T) lsum += (fa - ta) * (fa - ta);
      }
      if (mb < n) {
        float v2 = S[(size_t)mb * 5 + 2], amp = 0.f;
        for (int j = 0; j < 5; j++) amp = fmaxf(amp, fabsf(S[(size_t)mb * 5 + j] - v2));
        if (face) face[mb] = v2 + amp * fb;
        if (omega)
          for (int k = 0; k < 3; k++) omega[(size_t)mb * 3 + k] = wb[k];
        if (vb && T) lsum += (fb - tb) * (fb - tb);
      }
    }
  }
  for (int o = 16; o > 0; o >>= 1) lsum += __shfl_xor_sync(0xffffffffu, lsum, o);
  if (loss && lane == 0) atomicAdd(loss, lsum * inv_n);
}

}  // namespace mlp

size_t mlp_image_offset() { return mlp::OFF_IMAGE_BYTES; }
size_t mlp_image_bytes() { return mlp::PACKED_BYTES; }

}  // namespace ibfsa

using namespace ibfsa;
using namespace ibfsa::mlp;

extern "C" {

size_t ibfsa_mlp_state_bytes(void) { return STATE_BYTES; }

static int cerr(cudaError_t e, const char *what) {
  if (e == cudaSuccess) return IBFSA_OK;
  char msg[256];
  snprintf(msg, sizeof(msg), "%s: %s", what, cudaGetErrorString(e));
  record_error(msg);
  return IBFSA_ERR_CUDA;
}

int ibfsa_mlp_init(void *d_state, const float *params, void *stream) {
  if (!d_state || !params) {
    record_error("ibfsa_mlp_init: NULL argument");
    return IBFSA_ERR_ARG;
  }
  cudaStream_t st = (cudaStream_t)stream;
  float *s = (float *)d_state;
  cudaError_t e = cudaMemsetAsync(s, 0, STATE_FLOATS * sizeof(float), st);
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(s + OFF_MASTER, params, NPARAM * sizeof(float), cudaMemcpyDefault, st);
  if (e == cudaSuccess) {
    k_pack<<<4, 256, 0, st>>>(s + OFF_MASTER, (unsigned char *)d_state + OFF_IMAGE_BYTES);
    e = cudaGetLastError();
  }
  return cerr(e, "ibfsa_mlp_init");
}

int ibfsa_mlp_train_step(void *d_state, int n, const float *stencils, const float *targets,
                         float lr, int step, void *stream) {
  if (!d_state || n <= 0 || !stencils || !targets || step < 1) {
    record_error("ibfsa_mlp_train_step: bad argument");
    return IBFSA_ERR_ARG;
  }
  cudaStream_t st = (cudaStream_t)stream;
  float *s = (float *)d_state;
  unsigned char *img = (unsigned char *)d_state + OFF_IMAGE_BYTES;
  cudaError_t e = cudaMemsetAsync(s + OFF_GRAD, 0, (NPAD + 64) * sizeof(float), st);
  if (e != cudaSuccess) return cerr(e, "ibfsa_mlp_train_step");
  int blocks = n / (16 * TRAIN_WARPS) + (n % (16 * TRAIN_WARPS) != 0);
  if (blocks > 152 * TRAIN_BLOCKS) blocks = 152 * TRAIN_BLOCKS;
  k_train<<<blocks, 32 * TRAIN_WARPS, 0, st>>>(img, n, stencils, targets, 1.f / (float)n,
                                                s + OFF_GRAD, s + OFF_LOSS);
  if ((e = cudaGetLastError()) != cudaSuccess) return cerr(e, "ibfsa_mlp_train_step");
  if (lr > 0.f) {
    const float b1 = 0.9f, b2 = 0.999f;
    float c1 = 1.f / (1.f - powf(b1, (float)step)), c2 = 1.f / (1.f - powf(b2, (float)step));
    k_adam<<<(NPARAM + 255) / 256, 256, 0, st>>>(s + OFF_MASTER, s + OFF_M, s + OFF_V,
                                                 s + OFF_GRAD, lr, b1, b2, 1e-8f, c1, c2);
    if ((e = cudaGetLastError()) != cudaSuccess) return cerr(e, "ibfsa_mlp_train_step");
    k_pack<<<4, 256, 0, st>>>(s + OFF_MASTER, img);
    e = cudaGetLastError();
  }
  return cerr(e, "ibfsa_mlp_train_step");
}

int ibfsa_mlp_read(const void *d_state, float *params, float *grad, float *loss, void *stream) {
  if (!d_state) {
    record_error("ibfsa_mlp_read: NULL state");
    return IBFSA_ERR_ARG;
  }
  cudaStream_t st = (cudaStream_t)stream;
  const float *s = (const float *)d_state;
  cudaError_t e = cudaSuccess;
  if (params) e = cudaMemcpyAsync(params, s + OFF_MASTER, NPARAM * 4, cudaMemcpyDefault, st);
  if (e == cudaSuccess && grad) e = cudaMemcpyAsync(grad, s + OFF_GRAD, NPARAM * 4, cudaMemcpyDefault, st);
  if (e == cudaSuccess && loss) e = cudaMemcpyAsync(loss, s + OFF_LOSS, 4, cudaMemcpyDefault, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  return cerr(e, "ibfsa_mlp_read");
}

int ibfsa_mlp_eval(const void *d_state, int n, const float *stencils, const float *targets,
                   float *face, float *omega, float *loss, void *stream) {
  if (!d_state || n < 0 || (n > 0 && !stencils)) {
    record_error("ibfsa_mlp_eval: bad argument");
    return IBFSA_ERR_ARG;
  }
  if (n == 0) return IBFSA_OK;
  cudaStream_t st = (cudaStream_t)stream;
  cudaError_t e = cudaSuccess;
  if (loss) e = cudaMemsetAsync(loss, 0, sizeof(float), st);
  if (e != cudaSuccess) return cerr(e, "ibfsa_mlp_eval");
  int tiles = (n + 15) / 16;
  int blocks = (tiles + 7) / 8;
  if (blocks > 152 * 8) blocks = 152 * 8;
  k_eval<<<blocks, 256, 0, st>>>((const unsigned char *)d_state + OFF_IMAGE_BYTES, n, stencils,
                                 targets, face, omega, 1.f / (float)n, loss);
  return cerr(cudaGetLastError(), "ibfsa_mlp_eval");
}

}  // extern "C"
