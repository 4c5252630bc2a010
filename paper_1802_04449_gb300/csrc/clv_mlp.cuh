// clv_mlp.cuh -- learned initial guess for the primitive root solve.
//
// Not part of the paper: a 10 -> 64 -> 64 -> 4 SiLU network maps features of
// a cell's ideal part (E, M) and its spatial shear components to
// (eps/E, v^x, v^y, v^eta); |v| seeds the Newton solve.  Inference runs on the
// tensor cores (BF16 mma.sync m16n8k16, FP32 accumulate) inside the recovery
// kernel; training runs in FP32 with the kernels below.
//
// Features of a cell (the same definition is used for the training samples):
//   x0 = (ln E - kLnEShift) / kLnEScale,  x1..3 = M^{x,y,eta} / E,
//   x4..9 = pi~^{xx, xy, x eta, yy, y eta, eta eta} / E, clamped to [-4, 4].
// Parameters are packed W1 (64x10) | b1 | W2 (64x64) | b2 | W3 (4x64) | b3.
#pragma once
#include <cuda_bf16.h>

#include "clv_device.cuh"
#include "clv_launch.cuh"

namespace clv {

constexpr int kMlpIn = 10, kMlpHid = 64, kMlpOut = 4;
constexpr int kMlpParams = kMlpHid * kMlpIn + kMlpHid + kMlpHid * kMlpHid + kMlpHid + kMlpOut * kMlpHid + kMlpOut;
constexpr int kOffW1 = 0, kOffB1 = kOffW1 + kMlpHid * kMlpIn, kOffW2 = kOffB1 + kMlpHid,
              kOffB2 = kOffW2 + kMlpHid * kMlpHid, kOffW3 = kOffB2 + kMlpHid, kOffB3 = kOffW3 + kMlpOut * kMlpHid;
constexpr float kLnEShift = -5.0f, kLnEScale = 5.0f, kFeatClamp = 4.0f;

// Tensor-core copy of the network: BF16 weights padded to the mma tiles
// (W1 64x16, W2 64x64, W3 8x64) and FP32 biases (64, 64, 8).
constexpr int kMlpW1e = 64 * 16, kMlpW2e = 64 * 64, kMlpW3e = 8 * 64;
constexpr int kMlpBf16Elems = kMlpW1e + kMlpW2e + kMlpW3e;      // 5632
constexpr int kMlpBiasElems = 64 + 64 + 8;                       // 136
constexpr size_t kMlpDeviceBytes = kMlpBf16Elems * 2 + kMlpBiasElems * 4;

// Shared-memory copy: rows padded by 8 BF16 (16 bytes) so that the eight rows
// a fragment load touches fall in distinct banks.
constexpr int kMlpS1 = 16 + 8, kMlpS2 = 64 + 8, kMlpSX = 16 + 8;   // row strides (BF16)
constexpr int kMlpSW1 = 64 * kMlpS1, kMlpSW2 = 64 * kMlpS2, kMlpSW3 = 8 * kMlpS2;
constexpr int kMlpSmemW = kMlpSW1 + kMlpSW2 + kMlpSW3;             // BF16 elements

// Cooperative copy of the network from global (compact) to shared (padded).
__device__ __forceinline__ void mlp_load_smem(const void* mlp, __nv_bfloat16* s_w, float* s_b) {
  const unsigned* gw = reinterpret_cast<const unsigned*>(mlp);   // BF16 pairs
  const float* gb = reinterpret_cast<const float*>(reinterpret_cast<const __nv_bfloat16*>(mlp) + kMlpBf16Elems);
  unsigned* sw = reinterpret_cast<unsigned*>(s_w);
  for (int i = threadIdx.x; i < kMlpBf16Elems / 2; i += blockDim.x) {
    int d;
    if (i < kMlpW1e / 2) d = (i >> 3) * (kMlpS1 / 2) + (i & 7);
    else if (i < (kMlpW1e + kMlpW2e) / 2) { const int j = i - kMlpW1e / 2; d = kMlpSW1 / 2 + (j >> 5) * (kMlpS2 / 2) + (j & 31); }
    else { const int j = i - (kMlpW1e + kMlpW2e) / 2; d = (kMlpSW1 + kMlpSW2) / 2 + (j >> 5) * (kMlpS2 / 2) + (j & 31); }
    sw[d] = gw[i];
  }
  for (int i = threadIdx.x; i < kMlpBiasElems; i += blockDim.x) s_b[i] = gb[i];
}

// silu(z) = z sigmoid(z) = z (1 + tanh(z / 2)) / 2: one hardware tanh
// (tanh.approx.f32, max relative error ~2^-11) instead of an exponential and
// a reciprocal.
__device__ __forceinline__ float tanh_approx(float x) {
  float y;
  asm("tanh.approx.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float silu(float z) {
  const float hz = 0.5f * z;
  return fmaf(hz, tanh_approx(hz), hz);
}

template <typename R>
__device__ __forceinline__ void mlp_features(R E, R Mx, R My, R Me, const R* pij, float* x) {
  const float iE = 1.0f / float(E);
  x[0] = (__logf(float(E)) - kLnEShift) * (1.0f / kLnEScale);
  x[1] = float(Mx) * iE;
  x[2] = float(My) * iE;
  x[3] = float(Me) * iE;
#pragma unroll
  for (int k = 0; k < 6; ++k) x[4 + k] = fminf(kFeatClamp, fmaxf(-kFeatClamp, float(pij[k]) * iE));
}

__device__ __forceinline__ unsigned pack_bf16(float lo, float hi) {
  const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const unsigned*>(&v);
}

__device__ __forceinline__ void mma_bf16(float (&d)[4], unsigned a0, unsigned a1, unsigned a2, unsigned a3,
                                         unsigned b0, unsigned b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};\n"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// Four 8x8 BF16 matrices from shared memory: lane l gives the row address of
// row l & 7 of matrix l >> 3 (16 bytes, 16-byte aligned); register j of lane
// l receives elements (l >> 2, 2 (l & 3) .. + 1) of matrix j.
__device__ __forceinline__ void ldmatrix_x4(unsigned (&r)[4], const void* row_addr) {
  const unsigned a = (unsigned)__cvta_generic_to_shared(row_addr);
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];\n"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(a));
}

// Forward pass of 16 cells (rows of xs, bf16 [16][kMlpSX] in shared memory)
// on one warp; writes the 4 outputs of each row to ys ([16][4] floats).
// s_w: the padded shared copy (mlp_load_smem); bias: b1[64] b2[64] b3[8].
// Fragments come from ldmatrix: the B fragments (b0, b1) of n-tile n and k
// tile kk are the 8x8 blocks (rows n*8.., columns kk*16 and kk*16 + 8) of the
// row-major [out][in] weights.
__device__ __forceinline__ void mlp_tile16(const __nv_bfloat16* xs, const __nv_bfloat16* s_w, const float* bias,
                                           float* ys, int lane) {
  const int g = lane >> 2, t = lane & 3;
  const int mi = lane >> 3, mr = lane & 7;   // matrix and row this lane addresses
  const __nv_bfloat16* w1 = s_w;
  const __nv_bfloat16* w2 = s_w + kMlpSW1;
  const __nv_bfloat16* w3 = s_w + kMlpSW1 + kMlpSW2;
  // A: rows 0-7 / 8-15 x columns 0-7 / 8-15 -> a0 (r0-7,c0-7) a1 (r8-15,c0-7) a2 (r0-7,c8-15) a3 (r8-15,c8-15)
  unsigned a[4];
  ldmatrix_x4(a, xs + (mr + 8 * (mi & 1)) * kMlpSX + 8 * (mi >> 1));
  // layer 1: 16x16 . 16x64; n-tiles in pairs: matrices (nt, c0-7) (nt, c8-15) (nt+1, c0-7) (nt+1, c8-15)
  float h[8][4];
#pragma unroll
  for (int np = 0; np < 4; ++np) {
    unsigned b[4];
    ldmatrix_x4(b, w1 + ((2 * np + (mi >> 1)) * 8 + mr) * kMlpS1 + 8 * (mi & 1));
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int nt = 2 * np + u;
      const float bl = bias[nt * 8 + 2 * t], bh = bias[nt * 8 + 2 * t + 1];
      h[nt][0] = bl; h[nt][1] = bh; h[nt][2] = bl; h[nt][3] = bh;
      mma_bf16(h[nt], a[0], a[1], a[2], a[3], b[2 * u], b[2 * u + 1]);
#pragma unroll
      for (int r = 0; r < 4; ++r) h[nt][r] = silu(h[nt][r]);
    }
  }
  // layer 2: 16x64 . 64x64 (accumulators of two n-tiles form one k-tile of A)
  float h2[8][4];
#pragma unroll
  for (int nt = 0; nt < 8; ++nt) {
    const float bl = bias[64 + nt * 8 + 2 * t], bh = bias[64 + nt * 8 + 2 * t + 1];
    h2[nt][0] = bl; h2[nt][1] = bh; h2[nt][2] = bl; h2[nt][3] = bh;
  }
#pragma unroll
  for (int kk = 0; kk < 4; ++kk) {
    const unsigned a0 = pack_bf16(h[2 * kk][0], h[2 * kk][1]), a1 = pack_bf16(h[2 * kk][2], h[2 * kk][3]);
    const unsigned a2 = pack_bf16(h[2 * kk + 1][0], h[2 * kk + 1][1]), a3 = pack_bf16(h[2 * kk + 1][2], h[2 * kk + 1][3]);
#pragma unroll
    for (int np = 0; np < 4; ++np) {
      unsigned b[4];
      ldmatrix_x4(b, w2 + ((2 * np + (mi >> 1)) * 8 + mr) * kMlpS2 + kk * 16 + 8 * (mi & 1));
      mma_bf16(h2[2 * np], a0, a1, a2, a3, b[0], b[1]);
      mma_bf16(h2[2 * np + 1], a0, a1, a2, a3, b[2], b[3]);
    }
  }
#pragma unroll
  for (int nt = 0; nt < 8; ++nt)
#pragma unroll
    for (int r = 0; r < 4; ++r) h2[nt][r] = silu(h2[nt][r]);
  // layer 3: 16x64 . 64x8 (outputs 4..7 are padding); k-tiles in pairs:
  // matrices (kk, c0-7) (kk, c8-15) (kk+1, c0-7) (kk+1, c8-15) of W3's 8 rows
  float y[4];
  {
    const float bl = bias[128 + 2 * t], bh = bias[128 + 2 * t + 1];
    y[0] = bl; y[1] = bh; y[2] = bl; y[3] = bh;
  }
#pragma unroll
  for (int kp = 0; kp < 2; ++kp) {
    unsigned b[4];
    ldmatrix_x4(b, w3 + mr * kMlpS2 + (2 * kp + (mi >> 1)) * 16 + 8 * (mi & 1));
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int kk = 2 * kp + u;
      const unsigned a0 = pack_bf16(h2[2 * kk][0], h2[2 * kk][1]), a1 = pack_bf16(h2[2 * kk][2], h2[2 * kk][3]);
      const unsigned a2 = pack_bf16(h2[2 * kk + 1][0], h2[2 * kk + 1][1]),
                     a3 = pack_bf16(h2[2 * kk + 1][2], h2[2 * kk + 1][3]);
      mma_bf16(y, a0, a1, a2, a3, b[2 * u], b[2 * u + 1]);
    }
  }
  if (t < 2) {
    ys[g * 4 + 2 * t] = y[0];
    ys[g * 4 + 2 * t + 1] = y[1];
    ys[(g + 8) * 4 + 2 * t] = y[2];
    ys[(g + 8) * 4 + 2 * t + 1] = y[3];
  }
}

// ---------------------------------------------------------------------------
// Training (FP32).  A block of 256 threads takes chunks of kMlpChunk (64)
// samples: the layers and their transposes are 64 x 64 products over the
// chunk held in shared memory (feature-major rows of kMlpLd floats), a 4 x 4
// register tile per thread in packed FP32x2 arithmetic; the 64 x 64 product
// over the samples that is the gradient of W2 and the dot products of the
// other parameters stay in registers over all chunks of the block.
// Bound: shared-memory latency between the barriers of a chunk; 109 KB of
// shared memory and 128 registers keep two blocks on an SM, so one's products
// cover the other's barriers.  Before, one thread ran one sample with its
// activations in local memory, and the gradient phase read one column per
// lane (32-way bank conflicts).  Ten iterations of 32,768 samples: 2.95 ms
// before, 0.49 ms now (GB300).
// ---------------------------------------------------------------------------
constexpr int kMlpChunk = 64, kMlpGradThreads = 256;
constexpr int kMlpLd = kMlpChunk + 4;   // adjacent rows start 16 bytes apart modulo the 128-byte bank period

__device__ __forceinline__ unsigned long long mix64(unsigned long long z) {
  // splitmix64 finaliser (Steele, Lea, Flood 2014)
  z += 0x9e3779b97f4a7c15ull;
  z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
  z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
  return z ^ (z >> 31);
}

// sample index of slot j of a batch: uniform in [0, n) from (seed, iter, j);
// seed = 0 selects the identity (slot j -> sample j) for full-batch gradients
__device__ __forceinline__ long long batch_index(unsigned long long seed, int iter, long long j, long long n) {
  if (seed == 0) return j;
  return (long long)(mix64(seed ^ ((unsigned long long)iter << 32) ^ (unsigned long long)j) % (unsigned long long)n);
}

// Gradient of the loss over a batch, deterministically: the launch has a
// fixed number of blocks (at most kMlpGradBlocks); block b takes the chunks
// of kMlpChunk samples b, b + gridDim.x, ... in order and leaves their
// parameter gradients and loss in its own row of `partial`
// ([gridDim.x][kMlpParams + 1], loss last), which mlp_reduce_kernel adds up
// in a fixed order.  No atomics: the same inputs give the same bits.
constexpr int kMlpGradBlocks = 256;
constexpr int kMlpPartialRow = kMlpParams + 1;

// shared memory of the gradient kernel, in floats (every offset a multiple of 4)
constexpr int kMlpSmW1 = 0;                                   // W1 transposed [10][64]
constexpr int kMlpSmW2 = kMlpSmW1 + kMlpIn * kMlpHid;         // W2 [64][64]
constexpr int kMlpSmW2t = kMlpSmW2 + kMlpHid * kMlpHid;       // W2 transposed [64][kMlpLd]
constexpr int kMlpSmW3 = kMlpSmW2t + kMlpHid * kMlpLd;        // W3 [4][64]
constexpr int kMlpSmB = kMlpSmW3 + kMlpOut * kMlpHid;         // b1 [64] b2 [64] b3 [4]
constexpr int kMlpSmX = kMlpSmB + 2 * kMlpHid + kMlpOut;      // [11][kMlpLd]: features, then ones
constexpr int kMlpSmDY = kMlpSmX + (kMlpIn + 1) * kMlpLd;     // [4][kMlpLd]
constexpr int kMlpSmYt = kMlpSmDY + kMlpOut * kMlpLd;         // [4][kMlpLd] targets
constexpr int kMlpSmH1 = kMlpSmYt + kMlpOut * kMlpLd;         // [64][kMlpLd] each
constexpr int kMlpSmH2 = kMlpSmH1 + kMlpHid * kMlpLd;
constexpr int kMlpSmD1 = kMlpSmH2 + kMlpHid * kMlpLd;         // silu'(z), then the gradient of z
constexpr int kMlpSmD2 = kMlpSmD1 + kMlpHid * kMlpLd;
constexpr int kMlpSmFloats = kMlpSmD2 + kMlpHid * kMlpLd;
constexpr size_t mlp_grad_smem_bytes() { return (size_t)kMlpSmFloats * sizeof(float); }

// acc[a][0..1] += sum_k w[k * wld + i0 + a] * x[k * kMlpLd + s0 .. s0 + 3] for
// the thread's features i0 .. i0 + 3 and samples s0 .. s0 + 3 (pairs of samples)
template <int K>
__device__ __forceinline__ void mlp_tile_product(const float* w, int wld, const float* x, int i0, int s0,
                                                 float2 (&acc)[4][2]) {
#pragma unroll 8
  for (int k = 0; k < K; ++k) {
    const float4 a = *reinterpret_cast<const float4*>(w + k * wld + i0);
    const float4 v = *reinterpret_cast<const float4*>(x + k * kMlpLd + s0);
    const float2 lo = make_float2(v.x, v.y), hi = make_float2(v.z, v.w);
    const float wa[4] = {a.x, a.y, a.z, a.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float2 ww = make_float2(wa[i], wa[i]);
      acc[i][0] = __ffma2_rn(ww, lo, acc[i][0]);
      acc[i][1] = __ffma2_rn(ww, hi, acc[i][1]);
    }
  }
}

// h = silu(z) and silu'(z) of the thread's 4 x 4 tile to H and D
__device__ __forceinline__ void mlp_store_silu(const float2 (&z)[4][2], float* H, float* D, int i0, int s0) {
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const float zz[4] = {z[i][0].x, z[i][0].y, z[i][1].x, z[i][1].y};
    float h[4], d[4];
#pragma unroll
    for (int s = 0; s < 4; ++s) {
      const float sg = 1.0f / (1.0f + expf(-zz[s]));
      h[s] = zz[s] * sg;
      d[s] = sg * (1.0f + zz[s] * (1.0f - sg));
    }
    *reinterpret_cast<float4*>(H + (i0 + i) * kMlpLd + s0) = make_float4(h[0], h[1], h[2], h[3]);
    *reinterpret_cast<float4*>(D + (i0 + i) * kMlpLd + s0) = make_float4(d[0], d[1], d[2], d[3]);
  }
}

// D (silu' on entry) times the thread's 4 x 4 tile, in place
__device__ __forceinline__ void mlp_scale_tile(const float2 (&a)[4][2], float* D, int i0, int s0) {
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    float4* d = reinterpret_cast<float4*>(D + (i0 + i) * kMlpLd + s0);
    const float4 v = *d;
    *d = make_float4(v.x * a[i][0].x, v.y * a[i][0].y, v.z * a[i][1].x, v.w * a[i][1].y);
  }
}

static __global__ void __launch_bounds__(kMlpGradThreads, 2) mlp_grad_kernel(const float* params,
                                                                  const float* __restrict__ X,
                                                                  const float* __restrict__ Y, long long n,
                                                                  long long batch, unsigned long long seed, int iter,
                                                                  float* __restrict__ partial) {
  release_next_kernel();
  enter_step_kernel();
  extern __shared__ __align__(16) float sm[];
  __shared__ long long s_idx[kMlpChunk];   // sample of each slot of the chunk, -1 past the batch
  __shared__ float s_red[kMlpGradThreads / 32][2];
  float *sW1 = sm + kMlpSmW1, *sW2 = sm + kMlpSmW2, *sW2t = sm + kMlpSmW2t, *sW3 = sm + kMlpSmW3, *sB = sm + kMlpSmB;
  float *sX = sm + kMlpSmX, *sDY = sm + kMlpSmDY, *sYt = sm + kMlpSmYt;
  float *sH1 = sm + kMlpSmH1, *sH2 = sm + kMlpSmH2, *sD1 = sm + kMlpSmD1, *sD2 = sm + kMlpSmD2;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  for (int i = tid; i < kMlpIn * kMlpHid; i += kMlpGradThreads) sW1[(i % kMlpIn) * kMlpHid + i / kMlpIn] = params[kOffW1 + i];
  for (int i = tid; i < kMlpHid * kMlpHid; i += kMlpGradThreads) {
    const float w = params[kOffW2 + i];
    sW2[i] = w;
    sW2t[(i & 63) * kMlpLd + (i >> 6)] = w;
  }
  for (int i = tid; i < kMlpOut * kMlpHid; i += kMlpGradThreads) sW3[i] = params[kOffW3 + i];
  if (tid < kMlpHid) {
    sB[tid] = params[kOffB1 + tid];
    sB[kMlpHid + tid] = params[kOffB2 + tid];
  }
  if (tid < kMlpOut) sB[2 * kMlpHid + tid] = params[kOffB3 + tid];
  if (tid < kMlpLd) sX[kMlpIn * kMlpLd + tid] = 1.0f;
  // tile of the layer products: a warp covers 16 features x 32 samples
  const int i0 = 4 * ((wid >> 1) * 4 + (lane >> 3)), s0 = 4 * ((wid & 1) * 8 + (lane & 7));
  // tile of the W2 gradient: rows ti + 16 a (outputs) and tk + 16 b (inputs)
  const int ti = (wid & 1) * 8 + (lane & 7), tk = (wid >> 1) * 4 + (lane >> 3);
  float2 g2[4][4], gs[4];   // even and odd samples
#pragma unroll
  for (int a = 0; a < 4; ++a) {
    gs[a] = make_float2(0.f, 0.f);
#pragma unroll
    for (int b = 0; b < 4; ++b) g2[a][b] = make_float2(0.f, 0.f);
  }
  float loss = 0.0f, gb3 = 0.0f;
  const float inv_b = 1.0f / (float)batch;
  const long long nchunk = (batch + kMlpChunk - 1) / kMlpChunk;
  auto index_chunk = [&](long long chunk) {   // threads 0 .. 63
    const long long j = chunk * kMlpChunk + tid;
    s_idx[tid] = j < batch ? batch_index(seed, iter, j, n) : -1ll;
  };
  // the chunk's features and targets on their way to shared memory: element
  // tid + 256 r of the 64 x 10 features, element tid of the 64 x 4 targets
  float xr[3], yr;
  auto fetch_chunk = [&]() {
#pragma unroll
    for (int r = 0; r < 3; ++r) {
      const int e = tid + r * kMlpGradThreads;
      xr[r] = 0.0f;
      if (e < kMlpChunk * kMlpIn) {
        const long long s = s_idx[e / kMlpIn];
        if (s >= 0) xr[r] = X[s * kMlpIn + e % kMlpIn];
      }
    }
    const long long s = s_idx[tid >> 2];
    yr = s >= 0 ? Y[s * kMlpOut + (tid & 3)] : 0.0f;
  };
  if (tid < kMlpChunk) index_chunk(blockIdx.x);
  __syncthreads();
  fetch_chunk();
  for (long long chunk = blockIdx.x; chunk < nchunk; chunk += gridDim.x) {
    const bool more = chunk + gridDim.x < nchunk;
#pragma unroll
    for (int r = 0; r < 3; ++r) {
      const int e = tid + r * kMlpGradThreads;
      if (e < kMlpChunk * kMlpIn) sX[(e % kMlpIn) * kMlpLd + e / kMlpIn] = xr[r];
    }
    sYt[(tid & 3) * kMlpLd + (tid >> 2)] = yr;
    __syncthreads();
    if (more && tid < kMlpChunk) index_chunk(chunk + gridDim.x);   // every thread is past its fetch
    auto bias_tile = [&](const float* b, float2 (&z)[4][2]) {
#pragma unroll
      for (int i = 0; i < 4; ++i) z[i][0] = z[i][1] = make_float2(b[i0 + i], b[i0 + i]);
    };
    {
      float2 z[4][2];
      bias_tile(sB, z);
      mlp_tile_product<kMlpIn>(sW1, kMlpHid, sX, i0, s0, z);
      mlp_store_silu(z, sH1, sD1, i0, s0);
    }
    __syncthreads();
    if (more) fetch_chunk();
    {
      float2 z[4][2];
      bias_tile(sB + kMlpHid, z);
      mlp_tile_product<kMlpHid>(sW2t, kMlpLd, sH1, i0, s0, z);
      mlp_store_silu(z, sH2, sD2, i0, s0);
    }
    __syncthreads();
    {   // output o of sample s, its residual and the loss
      const int o = tid >> 6, s = tid & 63;
      float a[4] = {sB[2 * kMlpHid + o], 0.f, 0.f, 0.f};
#pragma unroll 4
      for (int k = 0; k < kMlpHid; k += 4)
#pragma unroll
        for (int q = 0; q < 4; ++q) a[q] = fmaf(sW3[o * kMlpHid + k + q], sH2[(k + q) * kMlpLd + s], a[q]);
      const bool valid = chunk * kMlpChunk + s < batch;
      const float r = valid ? ((a[0] + a[1]) + (a[2] + a[3])) - sYt[o * kMlpLd + s] : 0.0f;
      const float dy = 2.0f * r * inv_b;
      sDY[o * kMlpLd + s] = dy;
      loss = fmaf(r, r, loss);
      gb3 += dy;
    }
    __syncthreads();
    {   // gradient of z2
      float2 a[4][2];
#pragma unroll
      for (int i = 0; i < 4; ++i) a[i][0] = a[i][1] = make_float2(0.f, 0.f);
      mlp_tile_product<kMlpOut>(sW3, kMlpHid, sDY, i0, s0, a);
      mlp_scale_tile(a, sD2, i0, s0);
    }
    __syncthreads();
    {   // gradient of z1
      float2 a[4][2];
#pragma unroll
      for (int i = 0; i < 4; ++i) a[i][0] = a[i][1] = make_float2(0.f, 0.f);
      mlp_tile_product<kMlpHid>(sW2, kMlpHid, sD2, i0, s0, a);
      mlp_scale_tile(a, sD1, i0, s0);
    }
    // W2: needs only the gradient of z2 and h1
#pragma unroll 2
    for (int s = 0; s < kMlpChunk; s += 4) {
      float4 u[4], v[4];
#pragma unroll
      for (int a = 0; a < 4; ++a) u[a] = *reinterpret_cast<const float4*>(sD2 + (ti + 16 * a) * kMlpLd + s);
#pragma unroll
      for (int b = 0; b < 4; ++b) v[b] = *reinterpret_cast<const float4*>(sH1 + (tk + 16 * b) * kMlpLd + s);
#pragma unroll
      for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) {
          g2[a][b] = __ffma2_rn(make_float2(u[a].x, u[a].y), make_float2(v[b].x, v[b].y), g2[a][b]);
          g2[a][b] = __ffma2_rn(make_float2(u[a].z, u[a].w), make_float2(v[b].z, v[b].w), g2[a][b]);
        }
    }
    __syncthreads();
    // the other parameters: dot product q = tid + 256 r is row q & 63 of
    // dz1 with feature q >> 6 (10: ones, the bias b1), of dz2 with ones (11:
    // b2), or of h2 with the output gradient (q >> 6) - 12 (W3)
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const int k = (tid >> 6) + 4 * r, i = tid & 63;
      const float* u = (k < 11 ? sD1 : k == 11 ? sD2 : sH2) + i * kMlpLd;
      const float* v = k < 12 ? sX + (k < kMlpIn ? k : kMlpIn) * kMlpLd : sDY + (k - 12) * kMlpLd;
#pragma unroll 4
      for (int s = 0; s < kMlpChunk; s += 4) {
        const float4 x = *reinterpret_cast<const float4*>(u + s), y = *reinterpret_cast<const float4*>(v + s);
        gs[r] = __ffma2_rn(make_float2(x.x, x.y), make_float2(y.x, y.y), gs[r]);
        gs[r] = __ffma2_rn(make_float2(x.z, x.w), make_float2(y.z, y.w), gs[r]);
      }
    }
    __syncthreads();   // the next chunk overwrites the activations
  }
  // the block's row: every entry by one thread
  float* row = partial + (size_t)blockIdx.x * kMlpPartialRow;
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) row[kOffW2 + (ti + 16 * a) * kMlpHid + tk + 16 * b] = g2[a][b].x + g2[a][b].y;
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    const int k = (tid >> 6) + 4 * r, i = tid & 63;
    const int p = k < kMlpIn ? kOffW1 + i * kMlpIn + k : k == 10 ? kOffB1 + i : k == 11 ? kOffB2 + i
                                                                : kOffW3 + (k - 12) * kMlpHid + i;
    row[p] = gs[r].x + gs[r].y;
  }
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) {
    loss += __shfl_down_sync(0xffffffffu, loss, d);
    gb3 += __shfl_down_sync(0xffffffffu, gb3, d);
  }
  if (lane == 0) { s_red[wid][0] = loss; s_red[wid][1] = gb3; }
  __syncthreads();
  if (tid < kMlpOut) row[kOffB3 + tid] = s_red[2 * tid][1] + s_red[2 * tid + 1][1];
  if (tid == kMlpOut) {
    float a = 0.0f;
    for (int w = 0; w < kMlpGradThreads / 32; ++w) a += s_red[w][0];
    row[kMlpParams] = a / (float)batch;
  }
}

// Adam state of a training run (Kingma & Ba 2015); params = nullptr: gradient only
struct MlpAdam {
  float *params, *m, *v;
  int step;
  float lr;
};

// grad = sum of the partial rows (loss likewise), then the Adam step of the
// parameter.  A block takes 32 columns; its kMlpReduceGroups warps sum every
// kMlpReduceGroups-th row in order (coalesced), and the first warp adds the
// warps' sums in order.
constexpr int kMlpReduceGroups = 16;
static __global__ void __launch_bounds__(32 * kMlpReduceGroups) mlp_reduce_kernel(const float* partial,
                                                                                 int nblocks, float* grad,
                                                                                 float* loss, const MlpAdam ad) {
  release_next_kernel();
  enter_step_kernel();
  __shared__ float s[kMlpReduceGroups][33];
  const int lane = threadIdx.x & 31, g = threadIdx.x >> 5;
  const int p = blockIdx.x * 32 + lane;
  float a = 0.0f;
  if (p < kMlpPartialRow)
#pragma unroll 8
    for (int b = g; b < nblocks; b += kMlpReduceGroups) a += partial[(size_t)b * kMlpPartialRow + p];
  s[g][lane] = a;
  __syncthreads();
  if (g > 0 || p >= kMlpPartialRow) return;
#pragma unroll
  for (int w = 1; w < kMlpReduceGroups; ++w) a += s[w][lane];
  if (p == kMlpParams) {
    *loss = a;
    return;
  }
  grad[p] = a;
  if (!ad.params) return;
  const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
  const float mi = b1 * ad.m[p] + (1.0f - b1) * a;
  const float vi = b2 * ad.v[p] + (1.0f - b2) * a * a;
  ad.m[p] = mi;
  ad.v[p] = vi;
  const float mh = mi / (1.0f - powf(b1, (float)ad.step));
  const float vh = vi / (1.0f - powf(b2, (float)ad.step));
  ad.params[p] -= ad.lr * mh / (sqrtf(vh) + eps);
}

}  // namespace clv
