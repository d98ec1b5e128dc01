// Learned Davidson preconditioner: training (FP32 CUDA cores) and inference
// (BF16 hidden layer on the tensor cores) kernels.  The definitions are stated
// in mlp.hpp.
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <random>
#include <vector>

#include "device_once.hpp"
#include "kernels_tma.hpp"
#include "mlp.hpp"
#include "ptx.cuh"

namespace gbdmrg {

namespace {

constexpr double PAIR_CLIP = 100.0;
constexpr double DEN_EPS = 1e-8;

// SplitMix64 finaliser (Steele, Lea & Flood, OOPSLA 2014): a counter-based
// hash used to draw sample indices
__host__ __device__ inline uint64_t splitmix64(uint64_t x) {
  uint64_t z = x + 0x9E3779B97F4A7C15ULL;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ULL;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBULL;
  return z ^ (z >> 31);
}

__device__ __forceinline__ float gelu_f(float x) { return 0.5f * x * (1.0f + erff(x * 0.70710678118654752f)); }

// d/dx [x Phi(x)] = Phi(x) + x phi(x)
__device__ __forceinline__ float gelu_grad_f(float x) {
  return 0.5f * (1.0f + erff(x * 0.70710678118654752f)) + x * expf(-0.5f * x * x) * 0.39894228040143268f;
}

// barrier of 256 threads that returns whether p holds for all of them
template <int ID>
__device__ __forceinline__ bool vote_256(bool p) {
  int r;
  asm volatile(
      "{\n .reg .pred p, q;\n setp.ne.b32 p, %1, 0;\n barrier.cta.red.and.pred q, %2, 256, p;\n"
      " selp.s32 %0, 1, 0, q;\n}\n"
      : "=r"(r)
      : "r"((int)p), "n"(ID)
      : "memory");
  return r != 0;
}

__device__ __forceinline__ bool is_weight(long p) {
  return p < MLP_OFF_B1 || (p >= MLP_OFF_W2 && p < MLP_OFF_B2) || (p >= MLP_OFF_W3 && p < MLP_OFF_B3);
}

__device__ __forceinline__ void quantize_one(long p, const float* w, float* wq, __nv_bfloat16* w2b) {
  const float x = w[p];
  const __nv_bfloat16 b = __float2bfloat16_rn(x);
  wq[p] = is_weight(p) ? __bfloat162float(b) : x;
  if (p >= MLP_OFF_W2 && p < MLP_OFF_B2) w2b[p - MLP_OFF_W2] = b;
}

__global__ void quantize_kernel(const float* __restrict__ w, float* __restrict__ wq, __nv_bfloat16* __restrict__ w2b) {
  for (long p = (long)blockIdx.x * blockDim.x + threadIdx.x; p < MLP_NPARAMS; p += (long)gridDim.x * blockDim.x)
    quantize_one(p, w, wq, w2b);
}

// Adam on every parameter.  The gradient of W2 is the sum of `nparts` partial sums (in a
// fixed order); the other gradients are read from g and cleared for the next step.
__global__ void adam_kernel(float* __restrict__ w, float* __restrict__ g, const float* __restrict__ part, int nparts,
                            float* __restrict__ m, float* __restrict__ v, float lr, float b1, float b2, float c1,
                            float c2, float eps, float* __restrict__ wq, __nv_bfloat16* __restrict__ w2b) {
  for (long p = (long)blockIdx.x * blockDim.x + threadIdx.x; p < MLP_NPARAMS; p += (long)gridDim.x * blockDim.x) {
    float gg = 0.f;
    if (p >= MLP_OFF_W2 && p < MLP_OFF_B2) {
      for (int q = 0; q < nparts; ++q) gg += part[(long)q * MLP_H * MLP_H + p - MLP_OFF_W2];
    } else {
      gg = g[p];
      g[p] = 0.f;
    }
    const float mm = b1 * m[p] + (1.0f - b1) * gg;
    const float vv = b2 * v[p] + (1.0f - b2) * gg * gg;
    m[p] = mm;
    v[p] = vv;
    w[p] -= lr * (mm / c1) / (sqrtf(vv / c2) + eps);
    quantize_one(p, w, wq, w2b);
  }
}

__global__ void sum_parts_kernel(const float* __restrict__ part, int nparts, float* __restrict__ g) {
  for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < MLP_H * MLP_H; p += gridDim.x * blockDim.x) {
    float s = 0.f;
    for (int q = 0; q < nparts; ++q) s += part[(long)q * MLP_H * MLP_H + p];
    g[p] = s;
  }
}

// Training numerics, one kernel for the forward pass and (GRAD) everything of the backward
// pass except dL/dW2: a thread block takes 32 samples at a time, with W2 (BF16 values, 128 KB)
// resident in shared memory, so that the 256-wide activations never leave the SM but for h1 and
// dL/da2, which the dL/dW2 product needs.  Bound by the FP32 multiply-adds of the two 32 x 256
// x 256 products: a thread holds 8 samples x 4 neurons, per 8 columns 16 broadcast and 4 row
// loads (16 bytes; rows of 528 bytes, conflict-free for the forward product that runs along a
// row and for the backward one that runs down the columns) for 256 multiply-adds.  Sums over
// the samples (dL/dW3, db2, dW1, db1) stay in registers over all tiles of a block and are added
// atomically once.
// Measured (4 steps of 4096 samples with Adam): one 64 x 64 SGEMM and one element-wise kernel per
// operation 4.36 ms, this kernel, the dL/dW2 product and Adam 0.53 ms.
constexpr int TR_ROWS = 32, TR_THREADS = 256;
constexpr int TR_W2_LD = MLP_H + 8;  // BF16 elements per row of W2
constexpr int TR_ACT_LD = MLP_H + 4;  // floats per row of activations
struct TrSmem {
  __nv_bfloat16 w2[MLP_H * TR_W2_LD];
  float act[TR_ROWS * TR_ACT_LD];  // h1, then dL/da2
  float F[TR_ROWS][8];
  float P[TR_ROWS], T[TR_ROWS], g2[2][TR_ROWS], dg[TR_ROWS];
};

// the sample of row s: s itself, or (draw) an element of [0, n) drawn by the hash
__device__ __forceinline__ long train_sample(long s, long n, uint64_t key, bool draw) {
  return draw ? (long)(splitmix64(key + (uint64_t)s) % (uint64_t)n) : s;
}

template <bool GRAD>
__global__ void __launch_bounds__(TR_THREADS, 1)
    train_kernel(long rows, long n, uint64_t key, int draw, const float* __restrict__ F, const float* __restrict__ P,
                 const float* __restrict__ T, const float* __restrict__ wq, const __nv_bfloat16* __restrict__ w2b,
                 float* __restrict__ g_out, float* __restrict__ H1, float* __restrict__ dA2, double scale,
                 double* __restrict__ loss, float* __restrict__ grad) {
  extern __shared__ __align__(16) uint8_t tr_raw[];
  TrSmem& sm = *reinterpret_cast<TrSmem*>(tr_raw);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int half = warp & 1, rg = warp >> 1;  // neurons half * 128 + ..., samples rg * 8 + ...
  for (int e = tid; e < MLP_H * (MLP_H / 8); e += TR_THREADS) {
    const int j = e / (MLP_H / 8), q = e % (MLP_H / 8);
    *reinterpret_cast<uint4*>(&sm.w2[j * TR_W2_LD + q * 8]) = *reinterpret_cast<const uint4*>(w2b + j * MLP_H + q * 8);
  }
  float w1[MLP_F], b1 = wq[MLP_OFF_B1 + tid];
#pragma unroll
  for (int k = 0; k < MLP_F; ++k) w1[k] = wq[MLP_OFF_W1 + tid * MLP_F + k];
  float sw3[4] = {0, 0, 0, 0}, sb2[4] = {0, 0, 0, 0}, sb1[4] = {0, 0, 0, 0}, sw1[4][MLP_F];
#pragma unroll
  for (int c = 0; c < 4; ++c)
#pragma unroll
    for (int k = 0; k < MLP_F; ++k) sw1[c][k] = 0.f;
  double lsum = 0.0;
  float gsum = 0.f;
  const float b3 = wq[MLP_OFF_B3];
  for (long r0 = (long)blockIdx.x * TR_ROWS; r0 < rows; r0 += (long)gridDim.x * TR_ROWS) {
    const int nr = (int)min((long)TR_ROWS, rows - r0);
    __syncthreads();
    if (tid < TR_ROWS) {
      const long s = tid < nr ? train_sample(r0 + tid, n, key, draw != 0) : -1;
#pragma unroll
      for (int k = 0; k < MLP_F; ++k) sm.F[tid][k] = s >= 0 ? F[s * MLP_F + k] : 0.f;
      if (GRAD) {
        sm.P[tid] = s >= 0 ? P[s] : 0.f;
        sm.T[tid] = s >= 0 ? T[s] : 0.f;
      }
    }
    __syncthreads();
    for (int i = 0; i < TR_ROWS; ++i) {  // neuron tid of layer 1
      float a = 0.f;
#pragma unroll
      for (int k = 0; k < MLP_F; ++k) a = fmaf(sm.F[i][k], w1[k], a);
      const float h = gelu_f(a + b1);
      sm.act[i * TR_ACT_LD + tid] = h;
      if (GRAD && i < nr) H1[(r0 + i) * MLP_H + tid] = h;
    }
    __syncthreads();
    // a2[i][j] = sum_k h1[i][k] W2[j][k], j = half * 128 + c * 32 + lane
    float acc[8][4];
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
      for (int c = 0; c < 4; ++c) acc[i][c] = 0.f;
    for (int k0 = 0; k0 < MLP_H; k0 += 8) {
      uint4 wv[4];
#pragma unroll
      for (int c = 0; c < 4; ++c)
        wv[c] = *reinterpret_cast<const uint4*>(&sm.w2[(half * 128 + c * 32 + lane) * TR_W2_LD + k0]);
#pragma unroll
      for (int kh = 0; kh < 2; ++kh) {
        float4 a[8];
#pragma unroll
        for (int i = 0; i < 8; ++i)
          a[i] = *reinterpret_cast<const float4*>(&sm.act[(rg * 8 + i) * TR_ACT_LD + k0 + 4 * kh]);
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          const uint32_t u0 = kh ? wv[c].z : wv[c].x, u1 = kh ? wv[c].w : wv[c].y;
          const float w0 = __uint_as_float(u0 << 16), w1_ = __uint_as_float(u0 & 0xffff0000u);
          const float w2 = __uint_as_float(u1 << 16), w3 = __uint_as_float(u1 & 0xffff0000u);
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            acc[i][c] = fmaf(a[i].x, w0, acc[i][c]);
            acc[i][c] = fmaf(a[i].y, w1_, acc[i][c]);
            acc[i][c] = fmaf(a[i].z, w2, acc[i][c]);
            acc[i][c] = fmaf(a[i].w, w3, acc[i][c]);
          }
        }
      }
    }
    // g = b3 + W3 . gelu(a2 + b2)
    float gp[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) gp[i] = 0.f;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const int j = half * 128 + c * 32 + lane;
      const float b2 = wq[MLP_OFF_B2 + j], w3 = wq[MLP_OFF_W3 + j];
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        acc[i][c] += b2;
        gp[i] = fmaf(w3, gelu_f(acc[i][c]), gp[i]);
      }
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) {
#pragma unroll
      for (int o = 16; o; o >>= 1) gp[i] += __shfl_xor_sync(0xffffffffu, gp[i], o);
      if (lane == 0) sm.g2[half][rg * 8 + i] = gp[i];
    }
    __syncthreads();
    if (tid < nr) {
      const float g = sm.g2[0][tid] + sm.g2[1][tid] + b3;
      if (!GRAD) {
        g_out[r0 + tid] = g;
      } else {
        // e = (1 + g) P - T, dL/dg = 2 e P / rows
        const float e = (1.0f + g) * sm.P[tid] - sm.T[tid];
        const float dg = 2.0f * e * sm.P[tid] / (float)rows;
        sm.dg[tid] = dg;
        lsum += (double)e * e;
        gsum += dg;
      }
    } else if (GRAD && tid < TR_ROWS) {
      sm.dg[tid] = 0.f;
    }
    if constexpr (GRAD) {
      __syncthreads();
      // dL/da2 = dg W3 gelu'(a2), into shared memory in the place of h1
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const int j = half * 128 + c * 32 + lane;
        const float w3 = wq[MLP_OFF_W3 + j];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const int r = rg * 8 + i;
          const float dg = sm.dg[r], a = acc[i][c];
          const float d = dg * w3 * gelu_grad_f(a);
          sw3[c] = fmaf(dg, gelu_f(a), sw3[c]);
          sb2[c] += d;
          sm.act[r * TR_ACT_LD + j] = d;
          if (r < nr) dA2[(r0 + r) * MLP_H + j] = d;
        }
      }
      __syncthreads();
      // dL/dh1[i][k] = sum_j dL/da2[i][j] W2[j][k], k = half * 128 + lane * 4 + c
#pragma unroll
      for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int c = 0; c < 4; ++c) acc[i][c] = 0.f;
      for (int j0 = 0; j0 < MLP_H; j0 += 4) {
        float4 a[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) a[i] = *reinterpret_cast<const float4*>(&sm.act[(rg * 8 + i) * TR_ACT_LD + j0]);
#pragma unroll
        for (int jj = 0; jj < 4; ++jj) {
          const uint2 u = *reinterpret_cast<const uint2*>(&sm.w2[(j0 + jj) * TR_W2_LD + half * 128 + lane * 4]);
          const float w0 = __uint_as_float(u.x << 16), w1_ = __uint_as_float(u.x & 0xffff0000u);
          const float w2 = __uint_as_float(u.y << 16), w3 = __uint_as_float(u.y & 0xffff0000u);
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const float d = jj == 0 ? a[i].x : jj == 1 ? a[i].y : jj == 2 ? a[i].z : a[i].w;
            acc[i][0] = fmaf(d, w0, acc[i][0]);
            acc[i][1] = fmaf(d, w1_, acc[i][1]);
            acc[i][2] = fmaf(d, w2, acc[i][2]);
            acc[i][3] = fmaf(d, w3, acc[i][3]);
          }
        }
      }
      // dL/da1 = dL/dh1 gelu'(a1), a1 formed again from the features
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const int k = half * 128 + lane * 4 + c;
        float w[MLP_F];
#pragma unroll
        for (int q = 0; q < MLP_F; ++q) w[q] = wq[MLP_OFF_W1 + k * MLP_F + q];
        const float b = wq[MLP_OFF_B1 + k];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const int r = rg * 8 + i;
          float a = 0.f;
#pragma unroll
          for (int q = 0; q < MLP_F; ++q) a = fmaf(sm.F[r][q], w[q], a);
          const float d = acc[i][c] * gelu_grad_f(a + b);
          sb1[c] += d;
#pragma unroll
          for (int q = 0; q < MLP_F; ++q) sw1[c][q] = fmaf(d, sm.F[r][q], sw1[c][q]);
        }
      }
    }
  }
  if constexpr (GRAD) {
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const int j = half * 128 + c * 32 + lane, k = half * 128 + lane * 4 + c;
      atomicAdd(grad + MLP_OFF_W3 + j, sw3[c]);
      atomicAdd(grad + MLP_OFF_B2 + j, sb2[c]);
      atomicAdd(grad + MLP_OFF_B1 + k, sb1[c]);
#pragma unroll
      for (int q = 0; q < MLP_F; ++q) atomicAdd(grad + MLP_OFF_W1 + k * MLP_F + q, sw1[c][q]);
    }
    if (warp == 0) {
#pragma unroll
      for (int o = 16; o; o >>= 1) {
        lsum += __shfl_xor_sync(0xffffffffu, lsum, o);
        gsum += __shfl_xor_sync(0xffffffffu, gsum, o);
      }
      if (lane == 0) {
        atomicAdd(loss, lsum * scale);
        atomicAdd(grad + MLP_OFF_B3, gsum);
      }
    }
  }
}

// dL/dW2[j][k] = sum_s dA2[s][j] H1[s][k]: 128 x 128 outputs per block over `per` samples, one
// partial sum per blockIdx.z (added by the reader).  FP32-bound: 8 x 8 outputs per thread, 16
// samples staged at a time, double-buffered; enough sample ranges that the grid fills the GPU.
constexpr int DW_T = 128, DW_K = 16;
__global__ void __launch_bounds__(256) dw2_kernel(long rows, long per, const float* __restrict__ dA2,
                                                  const float* __restrict__ H1, float* __restrict__ part) {
  __shared__ __align__(16) float As[2][DW_K][DW_T], Bs[2][DW_K][DW_T];
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  const int j0 = blockIdx.y * DW_T, k0 = blockIdx.x * DW_T;
  const long s0 = (long)blockIdx.z * per, s1 = min(rows, s0 + per);
  float acc[8][8];
#pragma unroll
  for (int p = 0; p < 8; ++p)
#pragma unroll
    for (int q = 0; q < 8; ++q) acc[p][q] = 0.f;
  float4 ra[2], rb[2];
  auto fetch = [&](long s) {  // two float4 of each operand per thread
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int e = tid + 256 * u, r = e >> 5, c = (e & 31) * 4;
      const bool in = s + r < s1;
      ra[u] = in ? *reinterpret_cast<const float4*>(dA2 + (s + r) * MLP_H + j0 + c) : make_float4(0, 0, 0, 0);
      rb[u] = in ? *reinterpret_cast<const float4*>(H1 + (s + r) * MLP_H + k0 + c) : make_float4(0, 0, 0, 0);
    }
  };
  auto put = [&](int b) {
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int e = tid + 256 * u, r = e >> 5, c = (e & 31) * 4;
      *reinterpret_cast<float4*>(&As[b][r][c]) = ra[u];
      *reinterpret_cast<float4*>(&Bs[b][r][c]) = rb[u];
    }
  };
  fetch(s0);
  put(0);
  __syncthreads();
  int b = 0;
  for (long s = s0; s < s1; s += DW_K, b ^= 1) {
    const bool more = s + DW_K < s1;
    if (more) fetch(s + DW_K);
#pragma unroll
    for (int r = 0; r < DW_K; ++r) {
      float a[8], w[8];
      *reinterpret_cast<float4*>(a) = *reinterpret_cast<const float4*>(&As[b][r][ty * 4]);
      *reinterpret_cast<float4*>(a + 4) = *reinterpret_cast<const float4*>(&As[b][r][64 + ty * 4]);
      *reinterpret_cast<float4*>(w) = *reinterpret_cast<const float4*>(&Bs[b][r][tx * 4]);
      *reinterpret_cast<float4*>(w + 4) = *reinterpret_cast<const float4*>(&Bs[b][r][64 + tx * 4]);
#pragma unroll
      for (int p = 0; p < 8; ++p)
#pragma unroll
        for (int q = 0; q < 8; ++q) acc[p][q] = fmaf(a[p], w[q], acc[p][q]);
    }
    if (more) put(b ^ 1);
    __syncthreads();
  }
  float* out = part + (long)blockIdx.z * MLP_H * MLP_H;
#pragma unroll
  for (int p = 0; p < 8; ++p) {
    const int j = j0 + (p < 4 ? ty * 4 + p : 64 + ty * 4 + p - 4);
#pragma unroll
    for (int q = 0; q < 8; q += 4)
      *reinterpret_cast<float4*>(out + (long)j * MLP_H + k0 + (q ? 64 : 0) + tx * 4) =
          make_float4(acc[p][q], acc[p][q + 1], acc[p][q + 2], acc[p][q + 3]);
  }
}

// ------------------------------------------------------------ inference

__device__ void features(long i, const double* __restrict__ r, const double* __restrict__ d, double theta, double rn,
                         long n, const long* __restrict__ boff, int nb, const double* __restrict__ bsum,
                         const double* __restrict__ bmean, float* f) {
  int lo = 0, hi = nb - 1;  // the block b with boff[b] <= i < boff[b + 1]
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (boff[mid] <= i)
      lo = mid;
    else
      hi = mid - 1;
  }
  const double sqn = sqrt((double)n);
  const double delta = d[i] - theta;
  f[0] = (float)(r[i] * sqn / rn);
  f[1] = (float)asinh(delta);
  f[2] = (float)(delta / (delta * delta + 0.01));
  const double sz = (double)(boff[lo + 1] - boff[lo]);
  f[3] = (float)asinh(sqrt(bsum[lo] / sz) * sqn / rn);
  f[4] = (float)asinh(bmean[lo] - theta);
}

__device__ __forceinline__ double diag_correction(double r, double d, double theta) {
  double den = theta - d;
  if (fabs(den) < DEN_EPS) den = den < 0 ? -DEN_EPS : DEN_EPS;
  return r / den;
}

// The network applied to n elements, 128 at a time, in one kernel.  MODE 0: g of given
// features; MODE 1: t = (1 + g) r / (theta - d) with the features formed here.
//   warps 0-7   layer 1: two threads per element write h1 = gelu(W1 f + b1) in BF16 into the A
//               operand (128 x 256, 64 KB)
//   warp 16     one thread issues the 16 tcgen05.mma (M = 128, N = 256, K = 16) of the tile
//               against W2 (256 x 256 BF16, 128 KB, loaded once per block)
//   warps 8-15  g = W3 . gelu(z + b2) + b3 from the accumulator (two threads per element)
// Both operands lie in shared memory in column groups of 8 (K-major without swizzle), two
// accumulators of 256 columns.  Bound by the 512 erff per element on the CUDA cores (about
// 65 us for 200,000 elements at full rate); h1 and z never leave the SM.  Every wait is bounded:
// on timeout the block raises its abort flag and sets err.
// Measured (200,000 elements): layer 1, the tensor-core layer and the output as three kernels
// through 300 MB of intermediates 0.86-1.24 ms, this kernel 0.155 ms.
constexpr int IN_ROWS = 128, IN_THREADS = 544;
constexpr int IN_A_BYTES = IN_ROWS * MLP_H * 2, IN_B_BYTES = MLP_H * MLP_H * 2;
struct InSmem {
  __align__(128) uint8_t a[IN_A_BYTES], b[IN_B_BYTES];
  float w1[MLP_F + 1][MLP_H];  // columns of W1, then b1
  float b2[MLP_H], w3[MLP_H];
  float f[IN_ROWS][MLP_F];
  float part[2][IN_ROWS];
  uint64_t a_full, d_full[2], d_empty[2];
  uint32_t tmem;
  int abort;
};

template <int MODE>
__global__ void __launch_bounds__(IN_THREADS, 1)
    infer_kernel(long n, const float* __restrict__ F, const double* __restrict__ r, const double* __restrict__ d,
                 double theta, double rn, const long* __restrict__ boff, int nb, const double* __restrict__ bsum,
                 const double* __restrict__ bmean, const float* __restrict__ wq, const __nv_bfloat16* __restrict__ w2b,
                 float* __restrict__ g_out, double* __restrict__ t_out, int* __restrict__ flag, int* __restrict__ err) {
  extern __shared__ __align__(128) uint8_t in_raw[];
  InSmem& sm = *reinterpret_cast<InSmem*>(in_raw);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (warp == 8) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_u32(&sm.tmem)),
                 "r"(512));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::);
  }
  if (tid == 0) {
    mbar_init(&sm.a_full, 256);
    for (int i = 0; i < 2; ++i) {
      mbar_init(&sm.d_full[i], 1);
      mbar_init(&sm.d_empty[i], 256);
    }
    sm.abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::);
  }
  // W2: row = output neuron; column group q of all rows is contiguous
  for (int e = tid; e < MLP_H * (MLP_H / 8); e += IN_THREADS) {
    const int j = e % MLP_H, q = e / MLP_H;
    *reinterpret_cast<uint4*>(sm.b + (q * MLP_H + j) * 16) = *reinterpret_cast<const uint4*>(w2b + j * MLP_H + q * 8);
  }
  for (int e = tid; e < MLP_F * MLP_H; e += IN_THREADS) sm.w1[e % MLP_F][e / MLP_F] = wq[MLP_OFF_W1 + e];
  for (int j = tid; j < MLP_H; j += IN_THREADS) {
    sm.w1[MLP_F][j] = wq[MLP_OFF_B1 + j];
    sm.b2[j] = wq[MLP_OFF_B2 + j];
    sm.w3[j] = wq[MLP_OFF_W3 + j];
  }
  asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::);
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;\n" ::);
  const uint32_t tmem = sm.tmem;
  volatile int* abort_flag = &sm.abort;
  const long ntiles = (n + IN_ROWS - 1) / IN_ROWS;
  int it = 0;  // tiles of this block done by this role
  bool ok = true;
  if (warp < 8) {
    const int row = tid & 127, half = tid >> 7;
    for (long tl = blockIdx.x; tl < ntiles && ok; tl += gridDim.x, ++it) {
      const long e = tl * IN_ROWS + row;
      float f[MLP_F];
      if (MODE == 0) {
#pragma unroll
        for (int k = 0; k < MLP_F; ++k) f[k] = e < n ? F[e * MLP_F + k] : 0.f;
      } else {
        if (half == 0) {
          float fe[MLP_F] = {0.f, 0.f, 0.f, 0.f, 0.f};
          if (e < n) features(e, r, d, theta, rn, n, boff, nb, bsum, bmean, fe);
#pragma unroll
          for (int k = 0; k < MLP_F; ++k) sm.f[row][k] = fe[k];
        }
        asm volatile("bar.sync 2, 256;\n" ::: "memory");
#pragma unroll
        for (int k = 0; k < MLP_F; ++k) f[k] = sm.f[row][k];
      }
      // the previous tile's products have read the operand
      if (it > 0) ok = mbar_wait(&sm.d_full[(it - 1) & 1], (uint32_t)(((it - 1) >> 1) & 1), abort_flag);
      ok = vote_256<3>(ok);
      if (!ok) break;
      for (int q = half * 16; q < half * 16 + 16; ++q) {
        float a[8];
        auto row8 = [&](int k, float (&x)[8]) {
          *reinterpret_cast<float4*>(x) = *reinterpret_cast<const float4*>(&sm.w1[k][q * 8]);
          *reinterpret_cast<float4*>(x + 4) = *reinterpret_cast<const float4*>(&sm.w1[k][q * 8 + 4]);
        };
        row8(MLP_F, a);
#pragma unroll
        for (int k = 0; k < MLP_F; ++k) {
          float x[8];
          row8(k, x);
#pragma unroll
          for (int u = 0; u < 8; ++u) a[u] = fmaf(x[u], f[k], a[u]);
        }
        uint32_t w[4];
#pragma unroll
        for (int u = 0; u < 8; u += 2) {
          const __nv_bfloat162 b = __floats2bfloat162_rn(gelu_f(a[u]), gelu_f(a[u + 1]));
          w[u / 2] = *reinterpret_cast<const uint32_t*>(&b);
        }
        *reinterpret_cast<uint4*>(sm.a + (q * IN_ROWS + row) * 16) = make_uint4(w[0], w[1], w[2], w[3]);
      }
      asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
      mbar_arrive(&sm.a_full);
    }
  } else if (warp == 16) {
    if (lane == 0) {
      const uint32_t al = (smem_u32(sm.a) >> 4) | (uint32_t)IN_ROWS << 16;
      const uint32_t bl = (smem_u32(sm.b) >> 4) | (uint32_t)MLP_H << 16;
      const uint32_t id = tm_idesc_bf16(MLP_H, false);
      for (long tl = blockIdx.x; tl < ntiles && ok; tl += gridDim.x, ++it) {
        ok = mbar_wait(&sm.a_full, (uint32_t)(it & 1), abort_flag);
        if (ok && it >= 2) ok = mbar_wait(&sm.d_empty[it & 1], (uint32_t)(((it >> 1) - 1) & 1), abort_flag);
        if (!ok) break;
        asm volatile("tcgen05.fence::after_thread_sync;\n" ::);
        const uint32_t dd = tmem + (uint32_t)((it & 1) * MLP_H);
        for (int kk = 0; kk < MLP_H / 16; ++kk) {
          const uint32_t accum = kk > 0;
          asm volatile(
              "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
              " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(dd),
              "l"(sdesc_groups(al + kk * 2 * IN_ROWS)), "l"(sdesc_groups(bl + kk * 2 * MLP_H)), "r"(id), "r"(accum));
        }
        asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(
            smem_u32(&sm.d_full[it & 1])));
      }
    }
  } else {
    const int half = (warp - 8) >> 2, row = (warp & 3) * 32 + lane;
    const float b3 = wq[MLP_OFF_B3];
    for (long tl = blockIdx.x; tl < ntiles && ok; tl += gridDim.x, ++it) {
      const long e = tl * IN_ROWS + row;
      ok = mbar_wait(&sm.d_full[it & 1], (uint32_t)((it >> 1) & 1), abort_flag);
      ok = __all_sync(0xffffffffu, ok);
      asm volatile("tcgen05.fence::after_thread_sync;\n" ::);
      float acc[4] = {0.f, 0.f, 0.f, 0.f};
      if (ok) {
#pragma unroll 1
        for (int c0 = half * 128; c0 < half * 128 + 128; c0 += 32) {
          uint32_t v[32];
          tmem_ld32(tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)((it & 1) * MLP_H + c0), v);
#pragma unroll
          for (int u = 0; u < 32; u += 4) {
            const float4 w = *reinterpret_cast<const float4*>(&sm.w3[c0 + u]);
            const float4 b = *reinterpret_cast<const float4*>(&sm.b2[c0 + u]);
            acc[0] = fmaf(w.x, gelu_f(__uint_as_float(v[u]) + b.x), acc[0]);
            acc[1] = fmaf(w.y, gelu_f(__uint_as_float(v[u + 1]) + b.y), acc[1]);
            acc[2] = fmaf(w.z, gelu_f(__uint_as_float(v[u + 2]) + b.z), acc[2]);
            acc[3] = fmaf(w.w, gelu_f(__uint_as_float(v[u + 3]) + b.w), acc[3]);
          }
        }
      }
      asm volatile("tcgen05.fence::before_thread_sync;\n" ::);
      mbar_arrive(&sm.d_empty[it & 1]);
      const float s = (acc[0] + acc[1]) + (acc[2] + acc[3]);
      if (half == 1) sm.part[it & 1][row] = s;
      ok = vote_256<1>(ok);  // one warp's timeout ends the role for all
      if (ok && half == 0 && e < n) {
        const float g = s + sm.part[it & 1][row] + b3;
        if (MODE == 0) {
          g_out[e] = g;
        } else {
          if (!isfinite(g)) atomicExch(flag, 1);
          t_out[e] = (1.0 + (double)g) * diag_correction(r[e], d[e], theta);
        }
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::);
  __syncthreads();
  if (tid == 0 && sm.abort) atomicExch(err, 1);
  if (warp == 8) {
    __syncwarp();
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::);
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(512));
  }
}

// per block: sum of v^2 (mode 0) or mean of v (mode 1)
__global__ void block_reduce_kernel(const double* __restrict__ v, const long* __restrict__ boff, int nb,
                                    double* __restrict__ out, int mode) {
  __shared__ double sh[8];
  for (int b = blockIdx.x; b < nb; b += gridDim.x) {
    const long o0 = boff[b], o1 = boff[b + 1];
    double s = 0.0;
    for (long e = o0 + threadIdx.x; e < o1; e += blockDim.x) {
      const double x = v[e];
      s += mode == 0 ? x * x : x;
    }
    for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
      double S = 0.0;
      for (int i = 0; i < (int)(blockDim.x >> 5); ++i) S += sh[i];
      out[b] = mode == 0 ? S : (o1 > o0 ? S / (double)(o1 - o0) : 0.0);
    }
    __syncthreads();
  }
}

__global__ void dot_kernel(long n, const double* __restrict__ a, const double* __restrict__ b,
                           double* __restrict__ out) {
  __shared__ double sh[8];
  double s = 0.0;
  for (long e = (long)blockIdx.x * blockDim.x + threadIdx.x; e < n; e += (long)gridDim.x * blockDim.x)
    s += a[e] * b[e];
  for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    double S = 0.0;
    for (int i = 0; i < (int)(blockDim.x >> 5); ++i) S += sh[i];
    atomicAdd(out, S);
  }
}

__global__ void tau_kernel(long n, const double* __restrict__ psi, double inv_c, const double* __restrict__ x,
                           double* __restrict__ tau) {
  for (long e = (long)blockIdx.x * blockDim.x + threadIdx.x; e < n; e += (long)gridDim.x * blockDim.x)
    tau[e] = psi[e] * inv_c - x[e];
}

__global__ void pairs_kernel(long ns, uint64_t seed, long n, const double* __restrict__ r, const double* __restrict__ d,
                             double theta, double rn, const long* __restrict__ boff, int nb,
                             const double* __restrict__ bsum, const double* __restrict__ bmean,
                             const double* __restrict__ tau, double sc, float* __restrict__ F, float* __restrict__ P,
                             float* __restrict__ T, long* __restrict__ idx) {
  for (long q = (long)blockIdx.x * blockDim.x + threadIdx.x; q < ns; q += (long)gridDim.x * blockDim.x) {
    const long i = (long)(splitmix64(seed + (uint64_t)q) % (uint64_t)n);
    float f[MLP_F];
    features(i, r, d, theta, rn, n, boff, nb, bsum, bmean, f);
#pragma unroll
    for (int k = 0; k < MLP_F; ++k) F[q * MLP_F + k] = f[k];
    P[q] = (float)fmin(PAIR_CLIP, fmax(-PAIR_CLIP, diag_correction(r[i], d[i], theta) * sc));
    T[q] = (float)fmin(PAIR_CLIP, fmax(-PAIR_CLIP, tau[i] * sc));
    if (idx) idx[q] = i;
  }
}

constexpr int SM_COUNT = 152;

inline int blocks_for(long n, int threads = 256, int cap = 4096) {
  long b = (n + threads - 1) / threads;
  return (int)std::max<long>(1, std::min<long>(b, cap));
}

}  // namespace

// ------------------------------------------------------------ host side

Mlp::~Mlp() {
  // the arrays are freed on the network's stream: release them before it goes
  for (DArr<float>* a : {&w, &wq, &grad, &am, &av, &H1, &dA2, &part}) a->release();
  w2b.release();
  err.release();
  acc.release();
  if (stream) cudaStreamSynchronize(stream);
  if (own_stream && stream) cudaStreamDestroy(stream);
}

void MlpScratchDeleter::operator()(MlpScratch* p) const { delete p; }

static void mlp_requantize(Mlp& m) {
  quantize_kernel<<<blocks_for(MLP_NPARAMS), 256, 0, m.stream>>>(m.w.p, m.wq.p, m.w2b.p);
  count_launches(1);
  cuda_check(cudaGetLastError(), "quantize");
}

void mlp_init(Mlp& m, uint64_t seed, cudaStream_t s) {
  if (!s) {
    cuda_check(cudaStreamCreateWithFlags(&m.stream, cudaStreamNonBlocking), "stream create");
    m.own_stream = true;
  } else {
    m.stream = s;
  }
  std::vector<float> h(MLP_NPARAMS, 0.0f);
  std::mt19937_64 rng(seed);
  std::normal_distribution<float> n1(0.0f, 1.0f / std::sqrt((float)MLP_F)), n2(0.0f, 1.0f / std::sqrt((float)MLP_H));
  for (long p = MLP_OFF_W1; p < MLP_OFF_B1; ++p) h[p] = n1(rng);
  for (long p = MLP_OFF_W2; p < MLP_OFF_B2; ++p) h[p] = n2(rng);
  // W3 = 0, b3 = 0: the untrained network is the diagonal preconditioner
  m.w.alloc(MLP_NPARAMS, m.stream);
  m.wq.alloc(MLP_NPARAMS, m.stream);
  m.w2b.alloc((size_t)MLP_H * MLP_H, m.stream);
  m.grad.alloc(MLP_NPARAMS, m.stream);
  m.am.alloc(MLP_NPARAMS, m.stream);
  m.av.alloc(MLP_NPARAMS, m.stream);
  m.err.alloc(1, m.stream);
  m.acc.alloc(4, m.stream);
  cuda_check(cudaMemsetAsync(m.err.p, 0, sizeof(int), m.stream), "memset");
  mlp_set_params(m, h.data());
}

void mlp_set_params(Mlp& m, const float* host) {
  cuda_check(cudaMemcpyAsync(m.w.p, host, MLP_NPARAMS * sizeof(float), cudaMemcpyHostToDevice, m.stream), "h2d");
  cuda_check(cudaMemsetAsync(m.am.p, 0, MLP_NPARAMS * sizeof(float), m.stream), "memset");
  cuda_check(cudaMemsetAsync(m.av.p, 0, MLP_NPARAMS * sizeof(float), m.stream), "memset");
  m.adam_t = 0;
  mlp_requantize(m);
  cuda_check(cudaStreamSynchronize(m.stream), "sync");
}

void mlp_get_params(Mlp& m, float* host) {
  cuda_check(cudaMemcpyAsync(host, m.w.p, MLP_NPARAMS * sizeof(float), cudaMemcpyDeviceToHost, m.stream), "d2h");
  cuda_check(cudaStreamSynchronize(m.stream), "sync");
}

// sample ranges of the dL/dW2 product: four 128 x 128 output tiles each, enough for the GPU but
// at least 64 samples long
static int dw2_parts(long rows) { return (int)std::max<long>(1, std::min<long>(SM_COUNT / 4, rows / 64)); }

static void ensure_cap(Mlp& m, long B) {
  if (B <= m.cap) return;
  m.cap = 0;  // until all of them are there
  m.H1.alloc((size_t)B * MLP_H, m.stream);
  m.dA2.alloc((size_t)B * MLP_H, m.stream);
  m.part.alloc((size_t)dw2_parts(B) * MLP_H * MLP_H, m.stream);
  m.cap = B;
}

template <bool GRAD>
static void launch_train(Mlp& m, long rows, long n, uint64_t key, bool draw, const float* F, const float* P,
                         const float* T, float* g, double scale, double* loss_acc) {
  static DeviceOnce once;
  if (!allow_shared_memory(once, train_kernel<GRAD>, (int)sizeof(TrSmem))) throw Error(ST_ECUDA, "mlp: shared memory attribute");
  const int grid = (int)std::min<long>((rows + TR_ROWS - 1) / TR_ROWS, SM_COUNT);
  train_kernel<GRAD><<<grid, TR_THREADS, sizeof(TrSmem), m.stream>>>(rows, n, key, draw ? 1 : 0, F, P, T, m.wq.p,
                                                                     m.w2b.p, g, m.H1.p, m.dA2.p, scale, loss_acc,
                                                                     m.grad.p);
  count_launches(1);
}

// forward + backward of `rows` samples (drawn from F, P, T [n] with `key`, or the samples
// themselves); the gradient except dL/dW2 is added to m.grad, dL/dW2 left as partial sums
// (their number is returned), loss * scale added to *loss_acc
static int step_grad(Mlp& m, const float* F, const float* P, const float* T, long rows, long n, uint64_t key, bool draw,
                     double scale, double* loss_acc) {
  launch_train<true>(m, rows, n, key, draw, F, P, T, nullptr, scale, loss_acc);
  int np = dw2_parts(rows);
  const long per = ((rows + np - 1) / np + DW_K - 1) / DW_K * DW_K;
  np = (int)((rows + per - 1) / per);
  dw2_kernel<<<dim3(MLP_H / DW_T, MLP_H / DW_T, np), 256, 0, m.stream>>>(rows, per, m.dA2.p, m.H1.p, m.part.p);
  count_launches(1);
  cuda_check(cudaGetLastError(), "mlp gradient");
  return np;
}

double mlp_loss_grad(Mlp& m, const float* F, const float* P, const float* T, long n) {
  if (n <= 0) throw Error(ST_EINVAL, "no samples");
  ensure_cap(m, n);
  cuda_check(cudaMemsetAsync(m.acc.p, 0, sizeof(double), m.stream), "memset");
  cuda_check(cudaMemsetAsync(m.grad.p, 0, MLP_NPARAMS * sizeof(float), m.stream), "memset");
  const int np = step_grad(m, F, P, T, n, n, 0, false, 1.0 / (double)n, m.acc.p);
  sum_parts_kernel<<<blocks_for((long)MLP_H * MLP_H), 256, 0, m.stream>>>(m.part.p, np, m.grad.p + MLP_OFF_W2);
  count_launches(1);
  cuda_check(cudaGetLastError(), "mlp gradient");
  double L = 0;
  cuda_check(cudaMemcpyAsync(&L, m.acc.p, sizeof(double), cudaMemcpyDeviceToHost, m.stream), "d2h");
  cuda_check(cudaStreamSynchronize(m.stream), "sync");
  return L;
}

template <int MODE>
static void launch_infer(Mlp& m, long n, const float* F, const double* r, const double* d, double theta, double rn,
                         const MlpScratch* s, float* g, double* t, cudaStream_t st) {
  static DeviceOnce once;
  if (!allow_shared_memory(once, infer_kernel<MODE>, (int)sizeof(InSmem))) throw Error(ST_ECUDA, "mlp: shared memory attribute");
  const int grid = (int)std::min<long>((n + IN_ROWS - 1) / IN_ROWS, SM_COUNT);
  infer_kernel<MODE><<<grid, IN_THREADS, sizeof(InSmem), st>>>(
      n, F, r, d, theta, rn, s ? s->boff.p : nullptr, s ? s->nb : 0, s ? s->bsum.p : nullptr, s ? s->bmean.p : nullptr,
      m.wq.p, m.w2b.p, g, t, s ? s->flag.p : nullptr, m.err.p);
  count_launches(1);
  cuda_check(cudaGetLastError(), "mlp inference");
}

void mlp_forward(Mlp& m, const float* F, long n, float* g, bool inference) {
  if (n <= 0) return;
  cudaStream_t s = m.stream;
  if (!inference) {
    launch_train<false>(m, n, n, 0, false, F, nullptr, nullptr, g, 0.0, nullptr);
    cuda_check(cudaGetLastError(), "mlp forward");
    cuda_check(cudaStreamSynchronize(s), "sync");
    return;
  }
  launch_infer<0>(m, n, F, nullptr, nullptr, 0, 1, nullptr, g, nullptr, s);
  int h = 0;
  cuda_check(cudaMemcpyAsync(&h, m.err.p, sizeof(int), cudaMemcpyDeviceToHost, s), "d2h");
  cuda_check(cudaStreamSynchronize(s), "sync");
  if (h) throw Error(ST_ETIMEOUT, "tensor-core GEMM: a bounded wait ran out");
}

void mlp_train(Mlp& m, const float* F, const float* P, const float* T, long n, int epochs, int batch, float lr,
               uint64_t seed, double* first, double* last) {
  if (n <= 0 || epochs <= 0 || batch <= 0) throw Error(ST_EINVAL, "mlp_train: empty data or schedule");
  ensure_cap(m, batch);
  cudaStream_t s = m.stream;
  const long spe = (n + batch - 1) / batch;  // steps per epoch
  cuda_check(cudaMemsetAsync(m.acc.p, 0, 4 * sizeof(double), s), "memset");
  cuda_check(cudaMemsetAsync(m.grad.p, 0, MLP_NPARAMS * sizeof(float), s), "memset");
  const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
  for (int ep = 0; ep < epochs; ++ep) {
    double* lacc = m.acc.p + (ep == 0 ? 0 : ep == epochs - 1 ? 1 : 2);
    for (long st = 0; st < spe; ++st) {
      const uint64_t key = splitmix64(seed + (uint64_t)(ep * spe + st));
      const int np = step_grad(m, F, P, T, batch, n, key, true, 1.0 / ((double)batch * (double)spe), lacc);
      ++m.adam_t;
      const float c1 = 1.0f - std::pow(b1, (float)m.adam_t), c2 = 1.0f - std::pow(b2, (float)m.adam_t);
      adam_kernel<<<blocks_for(MLP_NPARAMS), 256, 0, s>>>(m.w.p, m.grad.p, m.part.p, np, m.am.p, m.av.p, lr, b1,
                                                          b2, c1, c2, eps, m.wq.p, m.w2b.p);
      count_launches(1);
    }
  }
  cuda_check(cudaGetLastError(), "mlp train");
  double h[2];
  cuda_check(cudaMemcpyAsync(h, m.acc.p, 2 * sizeof(double), cudaMemcpyDeviceToHost, s), "d2h");
  cuda_check(cudaStreamSynchronize(s), "sync");
  if (first) *first = h[0];
  if (last) *last = epochs == 1 ? h[0] : h[1];
}

// ------------------------------------------------------------ per-problem scratch

void mlp_scratch_build(MlpScratch& s, const Mlp* m, const PsiLayout& P, cudaStream_t st) {
  s.n = P.nnz;
  s.nb = (int)P.blocks.size();
  std::vector<long> off(s.nb + 1);
  for (int b = 0; b < s.nb; ++b) off[b] = P.blocks[b].off;
  off[s.nb] = P.nnz;
  s.boff.upload(off, st);
  s.bsum.alloc(std::max(1, s.nb), st);
  s.bmean.alloc(std::max(1, s.nb), st);
  s.flag.alloc(1, st);
  if (!m || s.n == 0) {
    cuda_check(cudaStreamSynchronize(st), "sync");
    return;
  }
  s.network = true;
  cuda_check(cudaStreamSynchronize(st), "sync");
}

void mlp_scratch_set_diag(MlpScratch& s, const double* d, cudaStream_t st) {
  if (s.nb == 0) return;
  block_reduce_kernel<<<std::min(s.nb, 4096), 256, 0, st>>>(d, s.boff.p, s.nb, s.bmean.p, 1);
  count_launches(1);
  cuda_check(cudaGetLastError(), "block mean");
}

bool mlp_precondition(Mlp& m, MlpScratch& s, const double* r, const double* d, double theta, double rnorm, double* t,
                      cudaStream_t st) {
  if (s.n == 0) return true;
  if (!s.network) throw Error(ST_ESTATE, "learned preconditioner: scratch built without the network");
  block_reduce_kernel<<<std::min(s.nb, 4096), 256, 0, st>>>(r, s.boff.p, s.nb, s.bsum.p, 0);
  count_launches(1);
  cuda_check(cudaMemsetAsync(s.flag.p, 0, sizeof(int), st), "memset");
  launch_infer<1>(m, s.n, nullptr, r, d, theta, rnorm, &s, nullptr, t, st);
  int h[2] = {0, 0};
  cuda_check(cudaMemcpyAsync(&h[0], s.flag.p, sizeof(int), cudaMemcpyDeviceToHost, st), "d2h");
  cuda_check(cudaMemcpyAsync(&h[1], m.err.p, sizeof(int), cudaMemcpyDeviceToHost, st), "d2h");
  cuda_check(cudaStreamSynchronize(st), "sync");
  if (h[1]) throw Error(ST_ETIMEOUT, "tensor-core GEMM: a bounded wait ran out");
  return h[0] == 0;
}

long mlp_make_pairs(MlpScratch& s, const double* x, const double* r, const double* d, double theta, double rnorm,
                    const double* psi, long ns, uint64_t seed, float* F, float* P, float* T, long* idx,
                    double min_overlap, cudaStream_t st) {
  if (ns <= 0 || s.n == 0) return 0;
  if ((long)s.tmp.n < s.n) s.tmp.alloc(s.n, st);
  DArr<double> dd;
  dd.alloc(2, st);
  cuda_check(cudaMemsetAsync(dd.p, 0, 2 * sizeof(double), st), "memset");
  dot_kernel<<<blocks_for(s.n, 256, 1024), 256, 0, st>>>(s.n, x, psi, dd.p);
  count_launches(1);
  double c = 0;
  cuda_check(cudaMemcpyAsync(&c, dd.p, sizeof(double), cudaMemcpyDeviceToHost, st), "d2h");
  cuda_check(cudaStreamSynchronize(st), "sync");
  if (!(std::fabs(c) > 0) || std::fabs(c) < min_overlap) return 0;
  tau_kernel<<<blocks_for(s.n), 256, 0, st>>>(s.n, psi, 1.0 / c, x, s.tmp.p);
  dot_kernel<<<blocks_for(s.n, 256, 1024), 256, 0, st>>>(s.n, s.tmp.p, s.tmp.p, dd.p + 1);
  block_reduce_kernel<<<std::min(s.nb, 4096), 256, 0, st>>>(r, s.boff.p, s.nb, s.bsum.p, 0);
  count_launches(3);
  double tn2 = 0;
  cuda_check(cudaMemcpyAsync(&tn2, dd.p + 1, sizeof(double), cudaMemcpyDeviceToHost, st), "d2h");
  cuda_check(cudaStreamSynchronize(st), "sync");
  if (!(tn2 > 0)) return 0;
  const double sc = std::sqrt((double)s.n) / std::sqrt(tn2);
  pairs_kernel<<<blocks_for(ns), 256, 0, st>>>(ns, seed, s.n, r, d, theta, rnorm, s.boff.p, s.nb, s.bsum.p,
                                               s.bmean.p, s.tmp.p, sc, F, P, T, idx);
  count_launches(1);
  cuda_check(cudaGetLastError(), "pairs");
  cuda_check(cudaStreamSynchronize(st), "sync");
  return ns;
}

}  // namespace gbdmrg
