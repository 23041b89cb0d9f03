// bp_mlp.cu -- MLP surrogate of the per-halo ICM solve (not in the paper).
//
// Network 6 -> 128 -> 128 -> 128 -> 3 with GELU hidden activations, mapping halo
// features (log10 M, log10 c, z, eps_*, f_*, eps_DM; normalised) to the solved model
// (ln r_f/r_vir, ln T r_vir/(G M), ln rho0/rho_s; normalised).
//
//  training (FP32):  k_forward (all four layers of a tile of rows), k_backward (data and
//                    weight gradients of a tile, all layers; one set of weight-gradient
//                    partials per CTA) + k_sum_partials (fixed order), k_adam
//  inference:        k_infer_tc, all four layers fused per 128-row tile, BF16 weights and
//                    activations, FP32 accumulation; the two 128 x 128 layers on the
//                    tensor cores (tcgen05, accumulator in tensor memory)
//  helpers:          k_features, k_targets, k_mse
// The surrogate solve (bp_solve_halos_surrogate) decodes the prediction into the seed of
// the FP32 pre-solve of bp_solve_halos_ex, whose FP64 Newton and residual gate follow (the
// rejected halos get the full solve).
#include <cuda_bf16.h>

#include <algorithm>
#include <vector>

#include "bp_internal.cuh"
#include "bp_tc.cuh"

namespace {

constexpr int IN = BP_MLP_IN, HID = BP_MLP_HID, OUT = BP_MLP_OUT;
constexpr int OFF_W1 = 0, OFF_B1 = OFF_W1 + HID * IN, OFF_W2 = OFF_B1 + HID,
              OFF_B2 = OFF_W2 + HID * HID, OFF_W3 = OFF_B2 + HID, OFF_B3 = OFF_W3 + HID * HID,
              OFF_W4 = OFF_B3 + HID, OFF_B4 = OFF_W4 + OUT * HID, NPAR = OFF_B4 + OUT;
static_assert(NPAR == BP_MLP_NPARAMS, "parameter count");
// bf16 weight buffer: W1, W2, W3, W4 back to back
constexpr int WB_W1 = 0, WB_W2 = WB_W1 + HID * IN, WB_W3 = WB_W2 + HID * HID,
              WB_W4 = WB_W3 + HID * HID, NWB = WB_W4 + OUT * HID;
static_assert(NWB == BP_MLP_NWEIGHTS, "weight count");
// cache per row: Z1, A1, Z2, A2, Z3, A3
constexpr int CZ1 = 0, CA1 = HID, CZ2 = 2 * HID, CA2 = 3 * HID, CZ3 = 4 * HID, CA3 = 5 * HID;
static_assert(6 * HID == BP_MLP_CACHE_PER_ROW, "cache layout");

__device__ __forceinline__ float gelu(float x) {
  return 0.5f * x * (1.0f + erff(x * 0.70710678118654752f));
}
__device__ __forceinline__ float gelu_grad(float x) {
  // d/dx [x Phi(x)] = Phi(x) + x phi(x)
  float cdf = 0.5f * (1.0f + erff(x * 0.70710678118654752f));
  float pdf = 0.39894228040143268f * expf(-0.5f * x * x);
  return cdf + x * pdf;
}

// ---------------------------------------------------------------- FP32 training kernels
// One CTA of 8 warps per SM, persistent over tiles of 32 rows, with W2 and W3 in shared memory
// ([out][in], rows padded to 132 floats: the lanes' 16-byte reads hit all banks whether they
// run over outputs or inputs).  Warp w owns rows 4 w .. 4 w + 3 of the tile through every layer,
// so the layers need no CTA barrier; a lane computes 4 rows x 4 outputs (or inputs) and reads 8
// 16-byte words of shared memory per 64 multiply-adds.  Bound by latency at one tile per SM: 8
// warps use 26 to 30% of the issue slots and wait for the weights and the cache (shared-memory
// reads keep their pipe 25% busy).
// Measured at 4096 rows (one training step of 17 launches took 398 us: the weight gradients ran
// on 16 CTAs, each layer was a launch, and every activation went through global memory twice):
// k_forward 20 us (68 us as four launches), k_backward + k_sum_partials 40 us (296 us as
// 13 launches).  32 rows per tile puts 128 tiles on 152 SMs at the training batch of 4096.
constexpr int MT_ROWS = 32, MT_THREADS = 256;
// Tiles whose weight gradients are added up in registers before they go into the CTA's partials:
// one chain of FP32 additions over all of a CTA's rows loses bits as its root (4e6 rows, terms of
// random sign: 4.1e-6 relative, 6.8e-7 with this, at 18.0 instead of 16.9 ms).  512 rows are fewer
// additions in a row than the 256 rows and then n / 256 partials of gradients formed in chunks, for
// every n.
constexpr int MT_FOLD = 16;
constexpr int LDW = HID + 4;  // padded row length in shared memory

struct MtForward {
  float w2[HID][LDW], w3[HID][LDW];
  float a[2][MT_ROWS][LDW];  // activations of the layer before and of this one
  float w1[HID][IN], w4[OUT][HID];
  float b1[HID], b2[HID], b3[HID], b4[4];
};
struct MtBackward {
  float w2[HID][LDW], w3[HID][LDW];
  float d[3][MT_ROWS][LDW];  // gradients of the pre-activations of layers 3, 2, 1
  float a[MT_ROWS][LDW];     // activations the weight gradient takes
  float x[MT_ROWS][8], dy[MT_ROWS][4];
  float w4[OUT][HID];
};

// a [HID][HID] matrix into padded shared rows (16-byte loads when src allows them)
__device__ __forceinline__ void mt_load_w(float (*dst)[LDW], const float* __restrict__ src) {
  if ((reinterpret_cast<uintptr_t>(src) & 15) == 0) {
    for (int q = threadIdx.x; q < HID * HID / 4; q += MT_THREADS)
      *reinterpret_cast<float4*>(&dst[q >> 5][4 * (q & 31)]) =
          __ldg(reinterpret_cast<const float4*>(src) + q);
  } else {
    for (int q = threadIdx.x; q < HID * HID; q += MT_THREADS) dst[q >> 7][q & 127] = src[q];
  }
}

// acc[r][j] += sum_k in[r][k] w[lane + 32 j][k] for the warp's four rows
__device__ __forceinline__ void mt_gemm_nt(const float (*in)[LDW], const float (*w)[LDW], int lane,
                                           float (&acc)[4][4]) {
#pragma unroll 4
  for (int k = 0; k < HID; k += 4) {
    float4 xv[4], wv[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) xv[r] = *reinterpret_cast<const float4*>(&in[r][k]);
#pragma unroll
    for (int j = 0; j < 4; ++j) wv[j] = *reinterpret_cast<const float4*>(&w[lane + 32 * j][k]);
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        acc[r][j] = fmaf(xv[r].x, wv[j].x, acc[r][j]);
        acc[r][j] = fmaf(xv[r].y, wv[j].y, acc[r][j]);
        acc[r][j] = fmaf(xv[r].z, wv[j].z, acc[r][j]);
        acc[r][j] = fmaf(xv[r].w, wv[j].w, acc[r][j]);
      }
  }
}

// acc[r][j] += sum_o d[r][o] w[o][4 lane + j] for the warp's four rows
__device__ __forceinline__ void mt_gemm_nn(const float (*d)[LDW], const float (*w)[LDW], int lane,
                                           float (&acc)[4][4]) {
#pragma unroll 2
  for (int o = 0; o < HID; o += 4) {
    float dv[4][4];
#pragma unroll
    for (int r = 0; r < 4; ++r)
      *reinterpret_cast<float4*>(dv[r]) = *reinterpret_cast<const float4*>(&d[r][o]);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const float4 wv = *reinterpret_cast<const float4*>(&w[o + q][4 * lane]);
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        acc[r][0] = fmaf(dv[r][q], wv.x, acc[r][0]);
        acc[r][1] = fmaf(dv[r][q], wv.y, acc[r][1]);
        acc[r][2] = fmaf(dv[r][q], wv.z, acc[r][2]);
        acc[r][3] = fmaf(dv[r][q], wv.w, acc[r][3]);
      }
    }
  }
}

__global__ void __launch_bounds__(MT_THREADS, 1)
    k_forward(int64_t n, const float* __restrict__ X, const float* __restrict__ par,
              float* __restrict__ Y, float* __restrict__ cache) {
  extern __shared__ __align__(16) unsigned char mt_raw[];
  MtForward& S = *reinterpret_cast<MtForward*>(mt_raw);
  const int tid = threadIdx.x, w = tid >> 5, lane = tid & 31;
  constexpr int LC = BP_MLP_CACHE_PER_ROW;
  mt_load_w(S.w2, par + OFF_W2);
  mt_load_w(S.w3, par + OFF_W3);
  for (int q = tid; q < HID * IN; q += MT_THREADS) (&S.w1[0][0])[q] = par[OFF_W1 + q];
  for (int q = tid; q < OUT * HID; q += MT_THREADS) (&S.w4[0][0])[q] = par[OFF_W4 + q];
  for (int q = tid; q < HID; q += MT_THREADS) {
    S.b1[q] = par[OFF_B1 + q];
    S.b2[q] = par[OFF_B2 + q];
    S.b3[q] = par[OFF_B3 + q];
  }
  if (tid < OUT) S.b4[tid] = par[OFF_B4 + tid];
  __syncthreads();
  for (int64_t t = blockIdx.x; t * MT_ROWS < n; t += gridDim.x) {
    const int64_t row0 = t * MT_ROWS + 4 * w;  // this warp's first row
    float acc[4][4];
    // pre-activation + bias and activation of one layer: to the cache and the next layer
    auto emit = [&](const float* b, int cz, int ca, float (*out)[LDW]) {
#pragma unroll
      for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const int o = lane + 32 * j;
          const float z = acc[r][j] + b[o], av = gelu(z);
          if (row0 + r < n) {
            cache[(row0 + r) * LC + cz + o] = z;
            cache[(row0 + r) * LC + ca + o] = av;
          }
          out[r][o] = av;
        }
      __syncwarp();
    };
    float(*a0)[LDW] = &S.a[0][4 * w];
    float(*a1)[LDW] = &S.a[1][4 * w];
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      float x[IN];
#pragma unroll
      for (int i = 0; i < IN; ++i) x[i] = row0 + r < n ? X[(row0 + r) * IN + i] : 0.f;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        float v = 0.f;
#pragma unroll
        for (int i = 0; i < IN; ++i) v = fmaf(x[i], S.w1[lane + 32 * j][i], v);
        acc[r][j] = v;
      }
    }
    emit(S.b1, CZ1, CA1, a0);
    auto clear = [&]() {
#pragma unroll
      for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[r][j] = 0.f;
    };
    clear();
    mt_gemm_nt(a0, S.w2, lane, acc);
    emit(S.b2, CZ2, CA2, a1);
    clear();
    mt_gemm_nt(a1, S.w3, lane, acc);
    emit(S.b3, CZ3, CA3, a0);
    // layer 4: lanes over the inputs, a fixed shuffle tree over the lanes
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
      for (int o = 0; o < OUT; ++o) {
        float v = 0.f;
#pragma unroll
        for (int j = 0; j < 4; ++j) v = fmaf(a0[r][lane + 32 * j], S.w4[o][lane + 32 * j], v);
#pragma unroll
        for (int q = 16; q > 0; q >>= 1) v += __shfl_xor_sync(0xffffffffu, v, q);
        if (lane == 0 && row0 + r < n) Y[(row0 + r) * OUT + o] = v + S.b4[o];
      }
    __syncwarp();
  }
}

// The weight gradient of a 128 x 128 layer over the tile's rows: thread (og, ig) owns outputs
// 4 og + {0..3}, 64 + 4 og + {0..3} and the same of the inputs
__device__ __forceinline__ void mt_wgrad(const float (*d)[LDW], const float (*a)[LDW], int og,
                                         int ig, float (&acc)[8][8]) {
#pragma unroll 2
  for (int r = 0; r < MT_ROWS; ++r) {
    float dv[8], av[8];
    *reinterpret_cast<float4*>(dv) = *reinterpret_cast<const float4*>(&d[r][4 * og]);
    *reinterpret_cast<float4*>(dv + 4) = *reinterpret_cast<const float4*>(&d[r][64 + 4 * og]);
    *reinterpret_cast<float4*>(av) = *reinterpret_cast<const float4*>(&a[r][4 * ig]);
    *reinterpret_cast<float4*>(av + 4) = *reinterpret_cast<const float4*>(&a[r][64 + 4 * ig]);
#pragma unroll
    for (int p = 0; p < 8; ++p)
#pragma unroll
      for (int q = 0; q < 8; ++q) acc[p][q] = fmaf(dv[p], av[q], acc[p][q]);
  }
}

__global__ void __launch_bounds__(MT_THREADS, 1)
    k_backward(int64_t n, const float* __restrict__ X, const float* __restrict__ par,
               const float* __restrict__ cache, const float* __restrict__ dY,
               float* __restrict__ P) {
  extern __shared__ __align__(16) unsigned char mt_raw[];
  MtBackward& S = *reinterpret_cast<MtBackward*>(mt_raw);
  const int tid = threadIdx.x, w = tid >> 5, lane = tid & 31;
  const int og = tid >> 4, ig = tid & 15;
  const int c = tid & (HID - 1), half = tid >> 7;  // column and half of the small gradients
  constexpr int LC = BP_MLP_CACHE_PER_ROW;
  mt_load_w(S.w2, par + OFF_W2);
  mt_load_w(S.w3, par + OFF_W3);
  for (int q = tid; q < OUT * HID; q += MT_THREADS) (&S.w4[0][0])[q] = par[OFF_W4 + q];
  float g3[8][8], g2[8][8];  // this thread's part of dW3 and dW2
#pragma unroll
  for (int p = 0; p < 8; ++p)
#pragma unroll
    for (int q = 0; q < 8; ++q) g3[p][q] = g2[p][q] = 0.f;
  // dW1 (inputs 3 half ..), dW4 (outputs 0, 1 of half 0, output 2 of half 1), biases: half 0
  // holds db3 and db1 of column c, half 1 db2 and (threads 128 ..) db4
  float g1[3] = {0.f, 0.f, 0.f}, g4[2] = {0.f, 0.f}, gb[2] = {0.f, 0.f};
  float* out = P + (int64_t)blockIdx.x * NPAR;
  int held = 0;         // tiles in the registers
  bool folded = false;  // out holds the tiles before them
  for (int64_t t = blockIdx.x; t * MT_ROWS < n; t += gridDim.x) {
    const int64_t base = t * MT_ROWS;
    const int64_t row0 = base + 4 * w;
    __syncthreads();  // the tile before is done with the shared arrays
    for (int q = tid; q < MT_ROWS * 8; q += MT_THREADS) {
      const int r = q >> 3, i = q & 7;
      S.x[r][i] = (i < IN && base + r < n) ? X[(base + r) * IN + i] : 0.f;
      if (i < 4) S.dy[r][i] = (i < OUT && base + r < n) ? dY[(base + r) * OUT + i] : 0.f;
    }
    // rows of cached activations, and of pre-activations' GELU' (zeros past the end)
    auto load_a = [&](int ca) {
#pragma unroll
      for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int j = 0; j < 4; ++j)
          S.a[4 * w + r][lane + 32 * j] =
              row0 + r < n ? cache[(row0 + r) * LC + ca + lane + 32 * j] : 0.f;
    };
    float z[4][4];  // pre-activations of columns 4 lane + j
    auto load_z = [&](int cz) {
#pragma unroll
      for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int j = 0; j < 4; ++j)
          z[r][j] = row0 + r < n ? cache[(row0 + r) * LC + cz + 4 * lane + j] : 0.f;
    };
    load_a(CA3);
    load_z(CZ3);
    __syncthreads();
    // layer 4 back to the pre-activations of layer 3
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        float v = 0.f;
#pragma unroll
        for (int o = 0; o < OUT; ++o) v = fmaf(S.dy[4 * w + r][o], S.w4[o][4 * lane + j], v);
        S.d[0][4 * w + r][4 * lane + j] = v * gelu_grad(z[r][j]);
      }
    // dW4, db4
    for (int r = 0; r < MT_ROWS; ++r) {
      const float av = S.a[r][c];
      g4[0] = fmaf(S.dy[r][2 * half], av, g4[0]);
      if (half == 0) g4[1] = fmaf(S.dy[r][1], av, g4[1]);
      else if (c < OUT) gb[1] += S.dy[r][c];
    }
    load_z(CZ2);
    __syncthreads();
    load_a(CA2);
    float acc[4][4];
    auto back = [&](int l, const float (*wt)[LDW]) {  // layer 3 - l to the pre-activations before
#pragma unroll
      for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[r][j] = 0.f;
      mt_gemm_nn(&S.d[l][4 * w], wt, lane, acc);
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        float4 v;
        v.x = acc[r][0] * gelu_grad(z[r][0]);
        v.y = acc[r][1] * gelu_grad(z[r][1]);
        v.z = acc[r][2] * gelu_grad(z[r][2]);
        v.w = acc[r][3] * gelu_grad(z[r][3]);
        *reinterpret_cast<float4*>(&S.d[l + 1][4 * w + r][4 * lane]) = v;
      }
    };
    back(0, S.w3);
    load_z(CZ1);
    __syncthreads();
    mt_wgrad(S.d[0], S.a, og, ig, g3);
    for (int r = 0; r < MT_ROWS; ++r) gb[0] += S.d[half][r][c];  // db3, db2
    back(1, S.w2);
    __syncthreads();
    load_a(CA1);
    __syncthreads();
    mt_wgrad(S.d[1], S.a, og, ig, g2);
    for (int r = 0; r < MT_ROWS; ++r) {
      const float dv = S.d[2][r][c];
#pragma unroll
      for (int i = 0; i < 3; ++i) g1[i] = fmaf(dv, S.x[r][3 * half + i], g1[i]);
      if (half == 0) gb[1] += dv;  // db1
    }
    if (++held < MT_FOLD && (t + gridDim.x) * MT_ROWS < n) continue;
    // into the CTA's partials (a row's loads before its stores, which may alias them)
    auto put = [&](int k, float& v) {
      out[k] = folded ? out[k] + v : v;
      v = 0.f;
    };
    auto put_rows = [&](int off, float (&g)[8][8]) {
#pragma unroll
      for (int p = 0; p < 8; ++p) {
        float* row = out + off + ((p < 4 ? 0 : 60) + 4 * og + p) * HID + 4 * ig;
        float before[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) before[q] = folded ? row[(q < 4 ? 0 : 60) + q] : 0.f;
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          row[(q < 4 ? 0 : 60) + q] = before[q] + g[p][q];
          g[p][q] = 0.f;
        }
      }
    };
    put_rows(OFF_W3, g3);
    put_rows(OFF_W2, g2);
#pragma unroll
    for (int i = 0; i < 3; ++i) put(OFF_W1 + c * IN + 3 * half + i, g1[i]);
    put(OFF_W4 + 2 * half * HID + c, g4[0]);
    if (half == 0) {
      put(OFF_W4 + HID + c, g4[1]);
      put(OFF_B3 + c, gb[0]);
      put(OFF_B1 + c, gb[1]);
    } else {
      put(OFF_B2 + c, gb[0]);
      if (c < OUT) put(OFF_B4 + c, gb[1]);
    }
    held = 0;
    folded = true;
  }
}

// grad[j] = the sum of the CTAs' partials: four threads per parameter, each a contiguous range
// of the CTAs in order, then their sums in a fixed tree
constexpr int SP_THREADS = 256, SP_COLS = SP_THREADS / 4;
__global__ void __launch_bounds__(SP_THREADS)
    k_sum_partials(const float* __restrict__ P, int ncta, float* __restrict__ grad) {
  __shared__ float s[4][SP_COLS];
  const int col = threadIdx.x % SP_COLS, q = threadIdx.x / SP_COLS;
  const int j = blockIdx.x * SP_COLS + col;
  const int per = (ncta + 3) / 4, c0 = q * per, c1 = min(ncta, c0 + per);
  float v = 0.f;
  if (j < NPAR) {
#pragma unroll 8
    for (int k = c0; k < c1; ++k) v += P[(int64_t)k * NPAR + j];
  }
  s[q][col] = v;
  __syncthreads();
  if (q == 0 && j < NPAR) grad[j] = (s[0][col] + s[1][col]) + (s[2][col] + s[3][col]);
}

__global__ void k_adam(int np, float* __restrict__ p, const float* __restrict__ g,
                       float* __restrict__ m, float* __restrict__ v, float lr, float b1, float b2,
                       float eps, float c1, float c2) {
  int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= np) return;
  float gj = g[j];
  float mj = b1 * m[j] + (1.f - b1) * gj;
  float vj = b2 * v[j] + (1.f - b2) * gj * gj;
  m[j] = mj;
  v[j] = vj;
  p[j] -= lr * (mj * c1) / (sqrtf(vj * c2) + eps);
}

__global__ void k_to_bf16(const float* __restrict__ p, __nv_bfloat16* __restrict__ wb) {
  int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= NWB) return;
  int src;
  if (j < WB_W2) src = OFF_W1 + j;
  else if (j < WB_W3) src = OFF_W2 + (j - WB_W2);
  else if (j < WB_W4) src = OFF_W3 + (j - WB_W3);
  else src = OFF_W4 + (j - WB_W4);
  wb[j] = __float2bfloat16_rn(p[src]);
}

// ---------------------------------------------------------------- tensor-core inference
// BF16 inference: a persistent CTA of 256 threads takes 128 rows at a time.  Layer 1 (6
// inputs) runs on the CUDA cores and writes its BF16 activations straight into the A operand
// of layer 2 (K-major, 128-byte swizzle, two K blocks of 64 inputs, 16 KB each).  Layers 2
// and 3 are one 128 x 128 x 128 tcgen05 GEMM each (kind::f16, BF16 operands) against W2 and
// W3, staged once per CTA in the same layout as the B operand, with the FP32 accumulator in
// tensor memory.  Their epilogues (bias, GELU, rounding to BF16) read it back, warp w taking
// rows 32 (w % 4) .. + 31 and columns 64 (w / 4) .. + 63; layer 4 (3 outputs, FP32 sums of
// BF16 activations times BF16 weights) is folded into layer 3's epilogue.  Every mbarrier
// wait is bounded; a timeout sets *err and stops the CTA.
constexpr int TI_M = 128, TI_THREADS = 256;
constexpr int TI_KB = TI_M * 128;  // bytes of one K block (128 rows x 64 BF16)
constexpr uint32_t TI_COLS = 128;
constexpr uint32_t TI_IDESC = bptc::idesc_bf16(TI_M, HID);
constexpr uint32_t TI_WAIT_POLLS = 1u << 26;
constexpr uint64_t TI_WAIT_NS = 2000000000ull;  // 2 s

struct alignas(1024) TiSmem {
  unsigned char w2[2 * TI_KB];
  unsigned char w3[2 * TI_KB];
  unsigned char act[2 * TI_KB];
  float w1[HID * IN];
  float b1[HID], b2[HID], b3[HID];
  float w4[OUT * HID];
  float b4[4];
  float ypart[2][TI_M][OUT];  // layer-4 sums of the two column halves
  uint64_t mbar;
  uint32_t tmem;
};

// byte offset of the 16-byte chunk holding inputs 8 q .. 8 q + 7 (q < 16) of row r
__device__ __forceinline__ int ti_chunk(int r, int q) {
  return (q >> 3) * TI_KB + (r >> 3) * 1024 + (r & 7) * 128 + (((q & 7) ^ (r & 7)) << 4);
}

__device__ __forceinline__ uint4 pack8_bf16(const float* v) {
  uint4 u;
  uint32_t* wd = reinterpret_cast<uint32_t*>(&u);
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const __nv_bfloat162 t = __floats2bfloat162_rn(v[2 * j], v[2 * j + 1]);
    wd[j] = *reinterpret_cast<const uint32_t*>(&t);
  }
  return u;
}

__device__ __forceinline__ float bf16_round(float v) {
  return __bfloat162float(__float2bfloat16_rn(v));
}

__global__ void __launch_bounds__(TI_THREADS) k_infer_tc(int64_t n, const float* __restrict__ X,
                                                         const __nv_bfloat16* __restrict__ wb,
                                                         const float* __restrict__ par,
                                                         float* __restrict__ Y, int* err) {
  using namespace bptc;
  extern __shared__ unsigned char ti_raw[];
  TiSmem& S = *reinterpret_cast<TiSmem*>(((uintptr_t)ti_raw + 1023) & ~(uintptr_t)1023);
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const int64_t ntiles = (n + TI_M - 1) / TI_M;
  if (w == 0) {
    tmem_alloc(&S.tmem, TI_COLS);
    tmem_relinquish();
  }
  if (tid == 0) {
    mbar_init(&S.mbar, 1);
    fence_mbar_init();
  }
  // W2, W3 ([out][in], 16-byte chunks of 8 inputs) into the B-operand layout; the rest FP32
  const uint4* w2g = reinterpret_cast<const uint4*>(wb + WB_W2);
  const uint4* w3g = reinterpret_cast<const uint4*>(wb + WB_W3);
  for (int c = tid; c < HID * 16; c += TI_THREADS) {
    const int o = c >> 4, q = c & 15;
    *reinterpret_cast<uint4*>(S.w2 + ti_chunk(o, q)) = w2g[c];
    *reinterpret_cast<uint4*>(S.w3 + ti_chunk(o, q)) = w3g[c];
  }
  for (int i = tid; i < HID * IN; i += TI_THREADS) S.w1[i] = __bfloat162float(wb[WB_W1 + i]);
  for (int i = tid; i < OUT * HID; i += TI_THREADS) S.w4[i] = __bfloat162float(wb[WB_W4 + i]);
  for (int i = tid; i < HID; i += TI_THREADS) {
    S.b1[i] = par[OFF_B1 + i];
    S.b2[i] = par[OFF_B2 + i];
    S.b3[i] = par[OFF_B3 + i];
  }
  if (tid < OUT) S.b4[tid] = par[OFF_B4 + tid];
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tm = S.tmem;
  const int qw = w & 3, hw = w >> 2;  // this warp's TMEM lane quarter and column half
  const uint32_t t_rows = tm + ((uint32_t)(32 * qw) << 16);
  const int er = 32 * qw + lane;                      // epilogue row
  const int r1 = tid & (TI_M - 1), h1 = tid >> 7;     // layer-1 row and output half
  uint32_t phase = 0;
  bool ok = true;
  for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    const int64_t row0 = tile * TI_M;
    {  // layer 1: row r1, outputs 64 h1 .. 64 h1 + 63
      const int64_t row = row0 + r1;
      float x[IN];
#pragma unroll
      for (int i = 0; i < IN; ++i) x[i] = bf16_round(row < n ? X[row * IN + i] : 0.f);
      for (int g = 0; g < 8; ++g) {
        float a[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const int o = 64 * h1 + 8 * g + j;
          float acc = 0.f;
#pragma unroll
          for (int i = 0; i < IN; ++i) acc = fmaf(x[i], S.w1[o * IN + i], acc);
          a[j] = gelu(acc + S.b1[o]);
        }
        *reinterpret_cast<uint4*>(S.act + ti_chunk(r1, 8 * h1 + g)) = pack8_bf16(a);
      }
    }
    for (int layer = 0; layer < 2; ++layer) {  // layers 2 and 3
      fence_proxy_async_smem();  // the activations, written by the threads, to the MMA
      tc_fence_before();
      __syncthreads();
      tc_fence_after();
      if (tid == 0) {
        const unsigned char* Bw = layer == 0 ? S.w2 : S.w3;
#pragma unroll
        for (int kb = 0; kb < 2; ++kb) {
          const uint64_t da = desc_sw128(smem_u32(S.act + kb * TI_KB));
          const uint64_t db = desc_sw128(smem_u32(Bw + kb * TI_KB));
#pragma unroll
          for (int ks = 0; ks < 4; ++ks)  // K step of 16 BF16 = 32 bytes: + 2 in the address
            mma_f16(tm, da + 2 * ks, db + 2 * ks, TI_IDESC, (kb | ks) ? 1u : 0u);
        }
        mma_commit(&S.mbar);
      }
      bool got = mbar_wait_bounded(&S.mbar, phase, TI_WAIT_POLLS, TI_WAIT_NS);
      got = __syncthreads_and(got) != 0;
      if (!got) {
        if (tid == 0) atomicExch(err, 1);
        ok = false;
        break;
      }
      phase ^= 1u;
      tc_fence_after();
      const float* bias = layer == 0 ? S.b2 : S.b3;
      float y0 = 0.f, y1 = 0.f, y2 = 0.f;
#pragma unroll
      for (int c16 = 0; c16 < 4; ++c16) {
        const int col0 = 64 * hw + 16 * c16;
        float v[16];
        tmem_ld16(t_rows + (uint32_t)col0, v);
        tmem_wait_ld();
        float a[16];
#pragma unroll
        for (int j = 0; j < 16; ++j) a[j] = bf16_round(gelu(v[j] + bias[col0 + j]));
        if (layer == 0) {
          *reinterpret_cast<uint4*>(S.act + ti_chunk(er, col0 / 8)) = pack8_bf16(a);
          *reinterpret_cast<uint4*>(S.act + ti_chunk(er, col0 / 8 + 1)) = pack8_bf16(a + 8);
        } else {
#pragma unroll
          for (int j = 0; j < 16; ++j) {
            y0 = fmaf(a[j], S.w4[col0 + j], y0);
            y1 = fmaf(a[j], S.w4[HID + col0 + j], y1);
            y2 = fmaf(a[j], S.w4[2 * HID + col0 + j], y2);
          }
        }
      }
      if (layer == 1) {
        S.ypart[hw][er][0] = y0;
        S.ypart[hw][er][1] = y1;
        S.ypart[hw][er][2] = y2;
      }
    }
    if (!ok) break;
    tc_fence_before();
    __syncthreads();
    if (tid < TI_M && row0 + tid < n) {
      const int64_t row = row0 + tid;
#pragma unroll
      for (int o = 0; o < OUT; ++o)
        Y[row * OUT + o] = (S.ypart[0][tid][o] + S.ypart[1][tid][o]) + S.b4[o];
    }
  }
  // a timed-out batch may still be running: wait for it (bounded) before releasing TMEM
  if (!ok) mbar_wait_bounded(&S.mbar, phase, TI_WAIT_POLLS, TI_WAIT_NS);
  tc_fence_before();
  __syncthreads();
  if (w == 0) tmem_dealloc(tm, TI_COLS);
}

// Launches the tensor-core inference (at most two CTAs per SM: 128 TMEM columns each and
// ~100 KB of shared memory) and queues the read-back of its timeout flag into
// h_pinned[7]; infer_check reads it after a synchronisation.
int infer_tc(bp_ctx* ctx, int64_t n, const float* x, const uint16_t* wb, const float* par,
             float* y) {
  if (n <= 0) return BP_OK;
  if (((uintptr_t)wb & 15) != 0)
    return bp_fail(ctx, BP_EINVAL, "mlp inference: BF16 weights not 16-byte aligned");
  const size_t smem = sizeof(TiSmem) + 1024;
  BP_CUDA(ctx, cudaFuncSetAttribute(k_infer_tc, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)smem));
  BP_CUDA(ctx, cudaFuncSetAttribute(k_infer_tc, cudaFuncAttributePreferredSharedMemoryCarveout,
                                    100));
  const int64_t ntiles = (n + TI_M - 1) / TI_M;
  const int64_t grid = std::min<int64_t>(ntiles, (int64_t)ctx->num_sms * 2);
  BP_CUDA(ctx, cudaMemsetAsync(ctx->d_flags + 1, 0, sizeof(int), ctx->stream));
  k_infer_tc<<<(unsigned)grid, TI_THREADS, smem, ctx->stream>>>(
      n, x, reinterpret_cast<const __nv_bfloat16*>(wb), par, y, ctx->d_flags + 1);
  BP_LAUNCH_CHECK(ctx, "mlp infer (tensor cores)");
  BP_CUDA(ctx, cudaMemcpyAsync(ctx->h_pinned + 7, ctx->d_flags + 1, sizeof(int),
                               cudaMemcpyDeviceToHost, ctx->stream));
  return BP_OK;
}
// after a synchronisation of the stream: did an inference wait time out?
int infer_check(bp_ctx* ctx) {
  if (*reinterpret_cast<const int*>(ctx->h_pinned + 7))
    return bp_fail(ctx, BP_ETIMEOUT, "mlp inference: a tensor-core wait timed out");
  return BP_OK;
}

// norm layout: [0..8] means of the 6 features and 3 targets, [9..17] their scales
__global__ void k_features(int64_t n, const double* __restrict__ M, const double* __restrict__ c,
                           const double* __restrict__ z, const double* __restrict__ prm,
                           const float* __restrict__ norm, float* __restrict__ X,
                           const float* __restrict__ hull, int* __restrict__ outside) {
  // the scales' reciprocals once per block: the kernel is bound by the FP64 pipe, and six
  // divisions per halo were a third of it (3e6 halos: 490 us, 740 us before)
  __shared__ double s_inv[IN];
  if (threadIdx.x < IN) s_inv[threadIdx.x] = 1.0 / norm[9 + threadIdx.x];
  __syncthreads();
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  double f[IN];
  f[0] = log10(M[i]);
  f[1] = log10(c[i]);
  f[2] = z[i];
  f[3] = prm ? prm[i] : 3.97e-6;
  f[4] = prm ? prm[n + i] : 0.026;
  f[5] = prm ? prm[2 * n + i] : 0.0;
  int out = 0;
  for (int k = 0; k < IN; ++k) {
    float v = (float)((f[k] - norm[k]) * s_inv[k]);
    if (!(v >= hull[k] && v <= hull[IN + k])) out = 1;
    X[i * IN + k] = v;
  }
  if (outside) outside[i] = out;
}

__global__ void k_targets(int64_t n, const double* __restrict__ model,
                          const float* __restrict__ norm, float* __restrict__ T) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  auto F = [&](int f) { return model[(int64_t)f * n + i]; };
  double rv = F(BP_M_RVIR), GM = bpc::G * F(BP_M_MVIR);
  double t[OUT] = {log(F(BP_M_RF) / rv), log(F(BP_M_T) * rv / GM), log(F(BP_M_RHO0) / F(BP_M_RHOS))};
  for (int k = 0; k < OUT; ++k) T[i * OUT + k] = (float)((t[k] - norm[IN + k]) / norm[9 + IN + k]);
}

// dY = 2 (Y - T) / (n OUT); per-block partial sums of the squared error
__global__ void k_mse(int64_t n, const float* __restrict__ Y, const float* __restrict__ T,
                      float* __restrict__ dY, float* __restrict__ part) {
  __shared__ float red[256];
  int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  float e2 = 0.f;
  if (j < n * OUT) {
    float d = Y[j] - T[j];
    dY[j] = 2.f * d / (float)(n * OUT);
    e2 = d * d;
  }
  red[threadIdx.x] = e2;
  __syncthreads();
  for (int s = 128; s > 0; s >>= 1) {
    if (threadIdx.x < s) red[threadIdx.x] += red[threadIdx.x + s];
    __syncthreads();
  }
  if (threadIdx.x == 0) part[blockIdx.x] = red[0];
}

// decoded prediction -> starting point of the FP64 solve; outside the hull -> NaN
__global__ void k_decode_guess(int64_t n, const float* __restrict__ Y,
                               const float* __restrict__ norm, const int* __restrict__ outside,
                               double* __restrict__ guess, unsigned long long* n_outside) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  double g0 = (double)Y[i * OUT + 0] * norm[9 + IN + 0] + norm[IN + 0];
  double g1 = (double)Y[i * OUT + 1] * norm[9 + IN + 1] + norm[IN + 1];
  if (outside[i]) {
    g0 = g1 = NAN;
    atomicAdd(n_outside, 1ull);  // an integer count: the same whatever the order
  }
  guess[i] = g0;
  guess[n + i] = g1;
}

// CTAs of the training kernels: one per tile of rows, at most one per SM
unsigned mt_grid(const bp_ctx* ctx, int64_t n) {
  return (unsigned)std::min<int64_t>((n + MT_ROWS - 1) / MT_ROWS, ctx->num_sms);
}

int check_n(bp_ctx* ctx, int64_t n, const char* who) {
  if (n < 0) return bp_fail(ctx, BP_EINVAL, "%s: n < 0", who);
  if (n > (int64_t)1 << 31) return bp_fail(ctx, BP_ERANGE, "%s: n above 2^31", who);
  return BP_OK;
}

}  // namespace

extern "C" {

int bp_mlp_forward(bp_ctx* ctx, int64_t n, const float* params, const float* x, float* y,
                   float* cache) {
  if (!ctx) return BP_EINVAL;
  int r = check_n(ctx, n, "bp_mlp_forward");
  if (r || n == 0) return r;
  if (!params || !x || !y || !cache) return bp_fail(ctx, BP_EINVAL, "bp_mlp_forward: null pointer");
  BP_CUDA(ctx, cudaFuncSetAttribute(k_forward, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)sizeof(MtForward)));
  k_forward<<<mt_grid(ctx, n), MT_THREADS, sizeof(MtForward), ctx->stream>>>(n, x, params, y,
                                                                            cache);
  BP_LAUNCH_CHECK(ctx, "mlp forward");
  return BP_OK;
}

int bp_mlp_backward(bp_ctx* ctx, int64_t n, const float* params, const float* x,
                    const float* cache, const float* dy, float* grad) {
  if (!ctx) return BP_EINVAL;
  int r = check_n(ctx, n, "bp_mlp_backward");
  if (r) return r;
  if (!params || !x || !cache || !dy || !grad)
    return bp_fail(ctx, BP_EINVAL, "bp_mlp_backward: null pointer");
  if (n == 0) {
    BP_CUDA(ctx, cudaMemsetAsync(grad, 0, NPAR * sizeof(float), ctx->stream));
    return BP_OK;
  }
  const unsigned grid = mt_grid(ctx, n);
  float* part;  // weight-gradient partials, one set per CTA
  if ((r = bp_ws(ctx, WS_MISC2, (size_t)grid * NPAR * sizeof(float), (void**)&part))) return r;
  BP_CUDA(ctx, cudaFuncSetAttribute(k_backward, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)sizeof(MtBackward)));
  k_backward<<<grid, MT_THREADS, sizeof(MtBackward), ctx->stream>>>(n, x, params, cache, dy, part);
  BP_LAUNCH_CHECK(ctx, "mlp backward");
  k_sum_partials<<<(NPAR + SP_COLS - 1) / SP_COLS, SP_THREADS, 0, ctx->stream>>>(part, (int)grid,
                                                                               grad);
  BP_LAUNCH_CHECK(ctx, "mlp gradient sums");
  return BP_OK;
}

int bp_mlp_adam(bp_ctx* ctx, float* params, const float* grad, float* m, float* v, int64_t step,
                double lr, double beta1, double beta2, double eps) {
  if (!ctx) return BP_EINVAL;
  if (!params || !grad || !m || !v || step < 1)
    return bp_fail(ctx, BP_EINVAL, "bp_mlp_adam: arguments");
  double c1 = 1.0 / (1.0 - pow(beta1, (double)step));
  double c2 = 1.0 / (1.0 - pow(beta2, (double)step));
  k_adam<<<(NPAR + 255) / 256, 256, 0, ctx->stream>>>(NPAR, params, grad, m, v, (float)lr,
                                                      (float)beta1, (float)beta2, (float)eps,
                                                      (float)c1, (float)c2);
  BP_LAUNCH_CHECK(ctx, "adam");
  return BP_OK;
}

int bp_mlp_to_bf16(bp_ctx* ctx, const float* params, uint16_t* weights_bf16) {
  if (!ctx) return BP_EINVAL;
  if (!params || !weights_bf16) return bp_fail(ctx, BP_EINVAL, "bp_mlp_to_bf16: null pointer");
  k_to_bf16<<<(NWB + 255) / 256, 256, 0, ctx->stream>>>(params, (__nv_bfloat16*)weights_bf16);
  BP_LAUNCH_CHECK(ctx, "to bf16");
  return BP_OK;
}

int bp_mlp_infer_bf16(bp_ctx* ctx, int64_t n, const uint16_t* weights_bf16, const float* params,
                      const float* x, float* y) {
  if (!ctx) return BP_EINVAL;
  int r = check_n(ctx, n, "bp_mlp_infer_bf16");
  if (r || n == 0) return r;
  if (!weights_bf16 || !params || !x || !y)
    return bp_fail(ctx, BP_EINVAL, "bp_mlp_infer_bf16: null pointer");
  if ((r = infer_tc(ctx, n, x, weights_bf16, params, y))) return r;
  BP_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
  return infer_check(ctx);
}

int bp_mlp_features(bp_ctx* ctx, int64_t n, const double* Mvir, const double* c, const double* z,
                    const double* params, const float* norm, float* x) {
  if (!ctx) return BP_EINVAL;
  int r = check_n(ctx, n, "bp_mlp_features");
  if (r || n == 0) return r;
  if (!Mvir || !c || !z || !norm || !x) return bp_fail(ctx, BP_EINVAL, "bp_mlp_features: null");
  // no hull test here: an all-inclusive hull
  float* hull;
  if ((r = bp_ws(ctx, WS_MISC3, 2 * IN * sizeof(float), (void**)&hull))) return r;
  float h[2 * IN];
  for (int k = 0; k < IN; ++k) {
    h[k] = -INFINITY;
    h[IN + k] = INFINITY;
  }
  BP_CUDA(ctx, cudaMemcpyAsync(hull, h, sizeof(h), cudaMemcpyHostToDevice, ctx->stream));
  k_features<<<(unsigned)((n + 255) / 256), 256, 0, ctx->stream>>>(n, Mvir, c, z, params, norm, x,
                                                                   hull, nullptr);
  BP_LAUNCH_CHECK(ctx, "features");
  BP_CUDA(ctx, cudaStreamSynchronize(ctx->stream));  // the host staging buffer h
  return BP_OK;
}

int bp_mlp_targets(bp_ctx* ctx, int64_t n, const double* model, const float* norm, float* t) {
  if (!ctx) return BP_EINVAL;
  int r = check_n(ctx, n, "bp_mlp_targets");
  if (r || n == 0) return r;
  if (!model || !norm || !t) return bp_fail(ctx, BP_EINVAL, "bp_mlp_targets: null pointer");
  k_targets<<<(unsigned)((n + 255) / 256), 256, 0, ctx->stream>>>(n, model, norm, t);
  BP_LAUNCH_CHECK(ctx, "targets");
  return BP_OK;
}

int bp_mlp_mse(bp_ctx* ctx, int64_t n, const float* y, const float* t, float* dy, double* loss) {
  if (!ctx) return BP_EINVAL;
  int r = check_n(ctx, n, "bp_mlp_mse");
  if (r || n == 0) return r;
  if (!y || !t || !dy) return bp_fail(ctx, BP_EINVAL, "bp_mlp_mse: null pointer");
  int64_t ne = n * OUT;
  unsigned nb = (unsigned)((ne + 255) / 256);
  float* part;
  if ((r = bp_ws(ctx, WS_MISC3, (size_t)nb * sizeof(float), (void**)&part))) return r;
  k_mse<<<nb, 256, 0, ctx->stream>>>(n, y, t, dy, part);
  BP_LAUNCH_CHECK(ctx, "mse");
  if (loss) {
    std::vector<float> h(nb);
    BP_CUDA(ctx, cudaMemcpyAsync(h.data(), part, nb * sizeof(float), cudaMemcpyDeviceToHost,
                                 ctx->stream));
    BP_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
    double s = 0;
    for (unsigned k = 0; k < nb; ++k) s += h[k];
    *loss = s / (double)ne;
  }
  return BP_OK;
}

int bp_solve_halos_surrogate(bp_ctx* ctx, int64_t n, const double* Mvir, const double* c,
                             const double* z, const double* params, const uint16_t* weights_bf16,
                             const float* mlp_params, const float* norm, const float* hull,
                             int polish_iter, double gate, double* model, int32_t* status,
                             double resid_tol) {
  if (!ctx) return BP_EINVAL;
  int r = check_n(ctx, n, "bp_solve_halos_surrogate");
  if (r || n == 0) return r;
  if (!Mvir || !c || !z || !weights_bf16 || !mlp_params || !norm || !hull || !model || !status)
    return bp_fail(ctx, BP_EINVAL, "bp_solve_halos_surrogate: null pointer");
  if (!(gate > 0)) return bp_fail(ctx, BP_EINVAL, "bp_solve_halos_surrogate: gate must be > 0");
  char* base;
  size_t bx = (size_t)n * IN * 4, by = (size_t)n * OUT * 4, bo = (size_t)n * 4,
         bg = (size_t)n * 2 * 8;
  if ((r = bp_ws(ctx, WS_MISC2, bx + by + bo + bg + 1024, (void**)&base))) return r;
  float* x = (float*)base;
  float* y = (float*)(base + ((bx + 255) / 256) * 256);
  int* outside = (int*)((char*)y + ((by + 255) / 256) * 256);
  double* guess = (double*)((char*)outside + ((bo + 255) / 256) * 256);
  bp_phase_begin(ctx, BP_PH_SURROGATE);
  k_features<<<(unsigned)((n + 255) / 256), 256, 0, ctx->stream>>>(n, Mvir, c, z, params, norm, x,
                                                                   hull, outside);
  BP_LAUNCH_CHECK(ctx, "features");
  if ((r = infer_tc(ctx, n, x, weights_bf16, mlp_params, y))) return r;
  unsigned long long* n_out = (unsigned long long*)(ctx->d_counter + 6);
  BP_CUDA(ctx, cudaMemsetAsync(n_out, 0, sizeof(int64_t), ctx->stream));
  k_decode_guess<<<(unsigned)((n + 255) / 256), 256, 0, ctx->stream>>>(n, y, norm, outside, guess,
                                                                      n_out);
  BP_LAUNCH_CHECK(ctx, "decode guess");
  BP_CUDA(ctx, cudaMemcpyAsync(ctx->h_pinned + 6, n_out, sizeof(int64_t), cudaMemcpyDeviceToHost,
                               ctx->stream));
  bp_phase_end(ctx, BP_PH_SURROGATE);
  // the prediction seeds the FP32 pre-solve; the halos outside the hull take its default
  // start (the plain solve), and count as fallbacks with those the gate rejects
  r = bp_solve_halos_ex(ctx, n, Mvir, c, z, params, guess, polish_iter > 0 ? polish_iter : 4,
                        gate, model, status,
                        polish_iter > 0 ? BP_SOLVE_FP64_SEEDED : BP_SOLVE_FP32_GATED, resid_tol);
  if (r == BP_OK || r == BP_ENOCONV) {  // the solve synchronised: the counts have arrived
    ctx->last_fallback += ctx->h_pinned[6];
    const int t = infer_check(ctx);
    if (t) return t;
  }
  return r;
}

}  // extern "C"
