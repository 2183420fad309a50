// ls_mlp.cuh -- training kernels of the donor-proposal MLP (FP32 master weights).
//
// Network: 8 inputs (7 window match fractions, one zero slot) -> 256 -> 256 -> 1, ReLU between
// layers.  Loss: half mean squared error between the score and the label.  FP32 throughout.  The loss
// and b3's gradient are double sums, b1's and b2's two-float sums; those of W1 and w3 are two-float sums over the
// CTAs and plain FP32 within one, W2's plain FP32 in chains of at most a split's rows (128, or B / 76 at 152 SMs).  Against
// float64 the gradient is within 3e-8 to 7e-8 of its norm for batches of 2048 to 40000 rows (1.3e-7 for 256).
//
// One gradient is three launches:
//   mlp_rows_kernel    tiles of up to 64 rows: both layers forward, the loss, dZ2, dH1 = dZ2 W2^T and the
//                      gradients of W1, b1, b2, w3, b3 (one partial per CTA); only H1 and dZ2 go to memory
//   mlp_dw2_kernel     H1^T dZ2 in 128 x 128 tiles, split over the rows
//   mlp_update_kernel  the partials' sums in a fixed order, and the Adam update or the gradient itself
// What bounds them is the FP32 pipe (3 x 2 x 65536 FLOP per row): packed FFMA2 on an 8 x 8 tile of
// outputs per thread, both operands from shared memory.  A CTA holds whole rows of the hidden layers, so
// nothing but H1 and dZ2 is written between the layers, and its time goes with its rows: the tile is 2, 4,
// 6, 7 or 8 rows a warp, whichever has the fewest rows in the fullest SM (two CTAs each).  Two CTAs leave 128
// registers a thread, beyond which the epilogues of 6, 7 and 8 rows spill 216, 380 and 540 bytes.
// Twenty training steps of 16384 / 2048 rows: 195.7 / 33.9 -> 3.4 / 1.5 ms (before: naive 16 x 16 GEMM
// tiles, one thread per column sum, twelve launches, seven allocations and a synchronisation a step; with
// 64-row tiles and a serial sum of the partials 4.0 ms at 16384).
//
// Inference uses the BF16 MMA kernel of ls_mlp_tc.cuh.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

namespace lsk {

constexpr int kMlpIn = 8;
// packed parameter vector (host and device FP32): W1 [8][256] (input x unit), b1 [256],
// W2 [256][256], b2 [256], w3 [256], b3
constexpr int kOffW1 = 0;
constexpr int kOffB1 = kOffW1 + kMlpIn * 256;
constexpr int kOffW2 = kOffB1 + 256;
constexpr int kOffB2 = kOffW2 + 256 * 256;
constexpr int kOffW3 = kOffB2 + 256;
constexpr int kOffB3 = kOffW3 + 256;
constexpr int kMlpParams = kOffB3 + 1;

constexpr int kTrRows = 64;      // most rows per tile of mlp_rows_kernel
constexpr int kTrThreads = 256;  // 8 warps: warp w holds RW rows from RW w, lane q columns 4q.. and 128 + 4q..
constexpr int kTrK = 16;         // weight rows per staged chunk
// dynamic shared memory: hidden tile [64][256], two weight chunks [16][256]
constexpr int kTrSmem = (kTrRows * 256 + 2 * kTrK * 256) * 4;
// a CTA's partial: dW1 [8][256], then [256] each: db1 (sum, error), db2 (sum, error), dw3
constexpr int kTrPart = 256 * (kMlpIn + 5);
constexpr int kDwTile = 128, kDwStages = 3;  // mlp_dw2_kernel
constexpr int kDwSmem = kDwStages * 2 * kTrK * kDwTile * 4;

__host__ __device__ inline uint64_t splitmix_at(uint64_t seed, uint64_t k) {  // k-th output (k >= 1) of the stream
  uint64_t z = seed + k * 0x9e3779b97f4a7c15ull;
  z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
  z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
  return z ^ (z >> 31);
}

struct MlpBatch {
  const float* X;    // [n_src][8]
  const float* y;    // [n_src]
  long long n_src;
  int B;             // rows of the batch
  int drawn;         // 1: row r of the batch is splitmix_at(seed, first + r + 1) % n_src, 0: row r
  uint64_t seed, first;
  const float* p;    // parameters
  const float* w2t;  // [256][256] W2 transposed
  float* H1;         // [B][256]
  float* dZ2;        // [B][256]
  float* part;       // [grid][kTrPart]
  double* partd;     // [grid][2]: sums of (s - y)^2 / 2 and of ds
};

__device__ __forceinline__ void mlp_cp16(void* dst, const void* src, bool valid) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src),
               "r"(valid ? 16 : 0)
               : "memory");
}
__device__ __forceinline__ void mlp_cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int K>
__device__ __forceinline__ void mlp_cp_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(K) : "memory");
}
// (s, e) += v with the exact error of the addition kept in e
__device__ __forceinline__ void two_sum(float& s, float& e, float v) {
  const float t = __fadd_rn(s, v), b = __fsub_rn(t, s);
  e = __fadd_rn(e, __fadd_rn(__fsub_rn(s, __fsub_rn(t, b)), __fsub_rn(v, b)));
  s = t;
}

// acc[r][.] += A[RW warp + r][k] Bg[k][columns of the lane], k < 256: A in shared memory, Bg [256][256]
// in global memory staged through the two chunks at Wc.  Starts and ends with a CTA barrier behind it.
template <int RW>
__device__ __forceinline__ void mlp_tile_gemm(const float* A, const float* __restrict__ Bg, float* Wc, float2 (&acc)[RW][4]) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  auto stage = [&](int c) {
    float* d = Wc + (c & 1) * kTrK * 256;
#pragma unroll
    for (int i = 0; i < kTrK * 64 / kTrThreads; ++i) {
      const int e = 4 * (tid + i * kTrThreads);
      mlp_cp16(d + e, Bg + (size_t)c * kTrK * 256 + e, true);
    }
    mlp_cp_commit();
  };
#pragma unroll
  for (int r = 0; r < RW; ++r)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[r][j] = make_float2(0.f, 0.f);
  stage(0);
#pragma unroll 1
  for (int c = 0; c < 256 / kTrK; ++c) {
    mlp_cp_wait<0>();
    __syncthreads();  // chunk c is complete, and everyone is done with the chunk the next copies overwrite
    if (c + 1 < 256 / kTrK) stage(c + 1);
    const float* b = Wc + (c & 1) * kTrK * 256 + 4 * lane;
    const float* a = A + (RW * warp) * 256 + c * kTrK;
#pragma unroll
    for (int k = 0; k < kTrK; k += 2) {
      float2 av[RW];
#pragma unroll
      for (int r = 0; r < RW; ++r) av[r] = *reinterpret_cast<const float2*>(a + r * 256 + k);
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const float4 b0 = *reinterpret_cast<const float4*>(b + (k + q) * 256);
        const float4 b1 = *reinterpret_cast<const float4*>(b + (k + q) * 256 + 128);
#pragma unroll
        for (int r = 0; r < RW; ++r) {
          const float v = q ? av[r].y : av[r].x;
          const float2 vv = make_float2(v, v);
          acc[r][0] = __ffma2_rn(vv, make_float2(b0.x, b0.y), acc[r][0]);
          acc[r][1] = __ffma2_rn(vv, make_float2(b0.z, b0.w), acc[r][1]);
          acc[r][2] = __ffma2_rn(vv, make_float2(b1.x, b1.y), acc[r][2]);
          acc[r][3] = __ffma2_rn(vv, make_float2(b1.z, b1.w), acc[r][3]);
        }
      }
    }
  }
  __syncthreads();
}

template <int RW>
__global__ void __launch_bounds__(kTrThreads, 2) mlp_rows_kernel(const MlpBatch m) {
  constexpr int ROWS = 8 * RW;
  extern __shared__ __align__(16) float tr_smem[];
  float* A = tr_smem;                  // [ROWS][256]: H1, then dZ2
  float* Wc = A + kTrRows * 256;       // weight chunks; between the products, scratch of the column sums
  __shared__ float Xs[ROWS][kMlpIn];
  __shared__ float ys[ROWS];
  __shared__ double redd[8][2];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int row0 = RW * warp;
  auto col = [&](int j) { return (j >> 2) * 128 + 4 * lane + (j & 3); };  // j-th of the lane's 8 columns
  const float* p = m.p;
  float* part = m.part + (size_t)blockIdx.x * kTrPart;
  double lsum = 0.0, dsum = 0.0;  // lanes < RW: row row0 + lane of every tile
  bool first = true;
  for (long long r0 = (long long)blockIdx.x * ROWS; r0 < m.B; r0 += (long long)gridDim.x * ROWS, first = false) {
    const int rows = (int)min((long long)ROWS, m.B - r0);
    for (int e = tid; e < ROWS * kMlpIn; e += kTrThreads) {
      const int r = e / kMlpIn, k = e % kMlpIn;
      long long src = r0 + r;
      if (m.drawn) src = (long long)(splitmix_at(m.seed, m.first + (uint64_t)src + 1) % (uint64_t)m.n_src);
      Xs[r][k] = r < rows ? m.X[src * kMlpIn + k] : 0.0f;
      if (k == 0) ys[r] = r < rows ? m.y[src] : 0.0f;
    }
    __syncthreads();
    {  // layer 1: thread = hidden unit
      float w1[kMlpIn];
#pragma unroll
      for (int k = 0; k < kMlpIn; ++k) w1[k] = p[kOffW1 + k * 256 + tid];
      const float b1 = p[kOffB1 + tid];
#pragma unroll 4
      for (int r = 0; r < ROWS; ++r) {
        float z = 0.0f;
#pragma unroll
        for (int k = 0; k < kMlpIn; ++k) z = fmaf(Xs[r][k], w1[k], z);
        const float h = fmaxf(z + b1, 0.0f);
        A[r * 256 + tid] = h;
        if (r < rows) m.H1[(size_t)(r0 + r) * 256 + tid] = h;
      }
    }
    __syncthreads();
    uint32_t live[2] = {0u, 0u};  // H1 > 0 at this thread's outputs of the last product, bit 4 r + j
#pragma unroll
    for (int r = 0; r < RW; ++r)
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const float4 v = *reinterpret_cast<const float4*>(A + (row0 + r) * 256 + 128 * h + 4 * lane);
        live[h] |= ((v.x > 0.f ? 1u : 0u) | (v.y > 0.f ? 2u : 0u) | (v.z > 0.f ? 4u : 0u) | (v.w > 0.f ? 8u : 0u)) << (4 * r);
      }
    float2 acc[RW][4];
    mlp_tile_gemm(A, p + kOffW2, Wc, acc);  // Z2 before its bias
    {
      // score, loss and ds of the warp's rows, dZ2 into A; column sums of dZ2 (db2) and of ds H2 (dw3)
      const float b3 = p[kOffB3];
      float ds[RW];
#pragma unroll
      for (int r = 0; r < RW; ++r) {
        float s = 0.0f;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          float2& z2 = acc[r][j >> 1];
          float& z = (j & 1) ? z2.y : z2.x;
          z += p[kOffB2 + col(j)];
          s = fmaf(fmaxf(z, 0.0f), p[kOffW3 + col(j)], s);
        }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
        const float d = (s + b3) - ys[row0 + r];
        ds[r] = row0 + r < rows ? d / (float)m.B : 0.0f;
        if (lane == r && row0 + r < rows) {
          lsum += 0.5 * (double)d * (double)d;
          dsum += (double)ds[r];
        }
      }
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const float w3 = p[kOffW3 + col(j)];
        float g3 = 0.0f, gs = 0.0f, ge = 0.0f;
#pragma unroll
        for (int r = 0; r < RW; ++r) {
          float& z = (j & 1) ? acc[r][j >> 1].y : acc[r][j >> 1].x;
          g3 = fmaf(ds[r], fmaxf(z, 0.0f), g3);
          z = z > 0.0f ? ds[r] * w3 : 0.0f;
          two_sum(gs, ge, z);
        }
        Wc[warp * 256 + col(j)] = g3;
        Wc[(8 + warp) * 256 + col(j)] = gs;
        Wc[(16 + warp) * 256 + col(j)] = ge;
      }
#pragma unroll
      for (int r = 0; r < RW; ++r)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const float4 v = make_float4(acc[r][2 * h].x, acc[r][2 * h].y, acc[r][2 * h + 1].x, acc[r][2 * h + 1].y);
          *reinterpret_cast<float4*>(A + (row0 + r) * 256 + 128 * h + 4 * lane) = v;
          if (row0 + r < rows) *reinterpret_cast<float4*>(m.dZ2 + (size_t)(r0 + row0 + r) * 256 + 128 * h + 4 * lane) = v;
        }
      __syncthreads();
      float* o = part + kMlpIn * 256 + tid;  // db1 (2 x 256), db2 (2 x 256), dw3 (256)
      float g3 = first ? 0.0f : o[4 * 256], gs = first ? 0.0f : o[2 * 256], ge = first ? 0.0f : o[3 * 256];
#pragma unroll
      for (int w = 0; w < 8; ++w) {
        g3 += Wc[w * 256 + tid];
        two_sum(gs, ge, Wc[(8 + w) * 256 + tid]);
        ge += Wc[(16 + w) * 256 + tid];
      }
      o[4 * 256] = g3;
      o[2 * 256] = gs;
      o[3 * 256] = ge;
      __syncthreads();
    }
    mlp_tile_gemm(A, m.w2t, Wc, acc);  // dH1
    {
      // dZ1; its column sums (db1) and products with the inputs (dW1) meet over the warps in A and Wc
      float* S = A;
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        float gs = 0.0f, ge = 0.0f, gw[kMlpIn];
#pragma unroll
        for (int k = 0; k < kMlpIn; ++k) gw[k] = 0.0f;
#pragma unroll
        for (int r = 0; r < RW; ++r) {
          const float a = (j & 1) ? acc[r][j >> 1].y : acc[r][j >> 1].x;
          const float z = (live[j >> 2] >> (4 * r + (j & 3))) & 1u ? a : 0.0f;
          two_sum(gs, ge, z);
#pragma unroll
          for (int k = 0; k < kMlpIn; ++k) gw[k] = fmaf(Xs[row0 + r][k], z, gw[k]);
        }
#pragma unroll
        for (int k = 0; k < kMlpIn; ++k) S[(8 * k + warp) * 256 + col(j)] = gw[k];
        S[(64 + warp) * 256 + col(j)] = gs;
        S[(72 + warp) * 256 + col(j)] = ge;
      }
      __syncthreads();
      float* o = part + tid;
#pragma unroll
      for (int k = 0; k < kMlpIn; ++k) {
        float g = first ? 0.0f : o[k * 256];
#pragma unroll
        for (int w = 0; w < 8; ++w) g += S[(8 * k + w) * 256 + tid];
        o[k * 256] = g;
      }
      float gs = first ? 0.0f : o[kMlpIn * 256], ge = first ? 0.0f : o[(kMlpIn + 1) * 256];
#pragma unroll
      for (int w = 0; w < 8; ++w) {
        two_sum(gs, ge, S[(64 + w) * 256 + tid]);
        ge += S[(72 + w) * 256 + tid];
      }
      o[kMlpIn * 256] = gs;
      o[(kMlpIn + 1) * 256] = ge;
      __syncthreads();  // before the next tile overwrites Xs and A
    }
  }
#pragma unroll
  for (int off = 4; off > 0; off >>= 1) {
    lsum += __shfl_xor_sync(0xffffffffu, lsum, off);
    dsum += __shfl_xor_sync(0xffffffffu, dsum, off);
  }
  if (lane == 0) {
    redd[warp][0] = lsum;
    redd[warp][1] = dsum;
  }
  __syncthreads();
  if (tid < 2) {
    double t = 0.0;
    for (int w = 0; w < 8; ++w) t += redd[w][tid];
    m.partd[2 * blockIdx.x + tid] = t;
  }
}

// Partial dW2 of the rows [blockIdx.y rows, ..): out[blockIdx.y][k][n] = sum_r H1[r][k] dZ2[r][n], one
// 128 x 128 quarter per blockIdx.x.  `rows` is a multiple of kTrK.
__global__ void __launch_bounds__(256, 2) mlp_dw2_kernel(const float* __restrict__ H1, const float* __restrict__ dZ2, int B,
                                                         int rows, float* __restrict__ out) {
  extern __shared__ __align__(16) float dw_smem[];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int k0 = (blockIdx.x >> 1) * kDwTile, n0 = (blockIdx.x & 1) * kDwTile;
  const int r_begin = blockIdx.y * rows, r_end = min(B, r_begin + rows);
  const int nchunk = (r_end - r_begin + kTrK - 1) / kTrK;
  auto stage = [&](int c) {
    float* a = dw_smem + (c % kDwStages) * 2 * kTrK * kDwTile;
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const int e = tid + i * 256, r = e >> 5, x = 4 * (e & 31), gr = r_begin + c * kTrK + r;
      const bool in = gr < r_end;
      const size_t o = (size_t)(in ? gr : r_begin) * 256 + x;
      mlp_cp16(a + r * kDwTile + x, H1 + o + k0, in);
      mlp_cp16(a + (kTrK + r) * kDwTile + x, dZ2 + o + n0, in);
    }
  };
  float2 acc[8][4];
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = make_float2(0.f, 0.f);
#pragma unroll
  for (int c = 0; c < kDwStages - 1; ++c) {
    if (c < nchunk) stage(c);
    mlp_cp_commit();
  }
  const int ka = 32 * (warp & 3) + 4 * (lane >> 3), nb = 64 * (warp >> 2) + 4 * (lane & 7);
#pragma unroll 1
  for (int c = 0; c < nchunk; ++c) {
    mlp_cp_wait<kDwStages - 2>();
    __syncthreads();
    if (c + kDwStages - 1 < nchunk) stage(c + kDwStages - 1);
    mlp_cp_commit();
    const float* a = dw_smem + (c % kDwStages) * 2 * kTrK * kDwTile;
    const float* b = a + kTrK * kDwTile;
#pragma unroll 4
    for (int r = 0; r < kTrK; ++r) {
      const float4 a0 = *reinterpret_cast<const float4*>(a + r * kDwTile + ka);
      const float4 a1 = *reinterpret_cast<const float4*>(a + r * kDwTile + ka + 16);
      const float4 b0 = *reinterpret_cast<const float4*>(b + r * kDwTile + nb);
      const float4 b1 = *reinterpret_cast<const float4*>(b + r * kDwTile + nb + 32);
      const float av[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const float2 vv = make_float2(av[i], av[i]);
        acc[i][0] = __ffma2_rn(vv, make_float2(b0.x, b0.y), acc[i][0]);
        acc[i][1] = __ffma2_rn(vv, make_float2(b0.z, b0.w), acc[i][1]);
        acc[i][2] = __ffma2_rn(vv, make_float2(b1.x, b1.y), acc[i][2]);
        acc[i][3] = __ffma2_rn(vv, make_float2(b1.z, b1.w), acc[i][3]);
      }
    }
  }
  float* o = out + (size_t)blockIdx.y * 65536;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    float* oi = o + (size_t)(k0 + ka + (i & 3) + 16 * (i >> 2)) * 256 + n0 + nb;
    *reinterpret_cast<float4*>(oi) = make_float4(acc[i][0].x, acc[i][0].y, acc[i][1].x, acc[i][1].y);
    *reinterpret_cast<float4*>(oi + 32) = make_float4(acc[i][2].x, acc[i][2].y, acc[i][3].x, acc[i][3].y);
  }
}

struct MlpUpdate {
  const float* partw;   // [splits][65536]
  int splits;
  const float* part;    // [ctas][kTrPart]
  const double* partd;  // [ctas][2]
  int ctas;
  float* g;             // gradient out (null: Adam update of p instead)
  double* loss;         // loss sum out (may be null)
  float *p, *m, *v, *w2t;
  float lr, b1, b2, c1, c2, eps;
};

// The gradient of every parameter from the partials, in a fixed order, and its Adam update:
// m = b1 m + (1-b1) g; v = b2 v + (1-b2) g^2; p -= lr * mhat / (sqrt(vhat) + eps).  Blocks 0..255: 256 weights
// of W2 each (four threads of 16-byte loads per quad, each a quarter of the splits); 256..343: 32 parameters of
// W1, b1, b2 and w3 each (8 threads a parameter, pairs of floats joined in double); the last block: b3 and the
// loss.
constexpr int kUpdBlocks = 256 + 11 * 256 / 32 + 1;
__global__ void __launch_bounds__(256) mlp_update_kernel(const MlpUpdate u) {
  const int tid = threadIdx.x;
  auto apply = [&](int e, float gi) {
    if (u.g) {
      u.g[e] = gi;
      return;
    }
    const float mi = u.b1 * u.m[e] + (1.0f - u.b1) * gi;
    const float vi = u.b2 * u.v[e] + (1.0f - u.b2) * gi * gi;
    u.m[e] = mi;
    u.v[e] = vi;
    const float pn = u.p[e] - u.lr * (mi / u.c1) / (sqrtf(vi / u.c2) + u.eps);
    u.p[e] = pn;
    if (e >= kOffW2 && e < kOffB2) u.w2t[((e - kOffW2) & 255) * 256 + ((e - kOffW2) >> 8)] = pn;
  };
  if (blockIdx.x < 256) {
    __shared__ float4 part[4][64];
    const int q = tid & 63, grp = tid >> 6;
    float4 g = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 8
    for (int s = grp; s < u.splits; s += 4) {
      const float4 v = *reinterpret_cast<const float4*>(u.partw + (size_t)s * 65536 + blockIdx.x * 256 + 4 * q);
      g.x += v.x;
      g.y += v.y;
      g.z += v.z;
      g.w += v.w;
    }
    part[grp][q] = g;
    __syncthreads();
    const float* f = reinterpret_cast<const float*>(&part[0][0]) + tid;
    apply(kOffW2 + blockIdx.x * 256 + tid, (f[0] + f[256]) + (f[512] + f[768]));
    return;
  }
  if (blockIdx.x + 1 < gridDim.x) {
    __shared__ double red[8][33];
    const int q = (blockIdx.x - 256) * 32 + (tid & 31), sec = q >> 8, c = q & 255;  // sec 0..7 W1, 8 b1, 9 b2, 10 w3
    const int o0 = (sec < 9 ? sec : sec == 9 ? kMlpIn + 2 : kMlpIn + 4) * 256 + c;
    const bool pair = sec == 8 || sec == 9;  // (sum, error)
    float ps = 0.0f, pe = 0.0f;
    for (int b0 = tid >> 5; b0 < u.ctas; b0 += 64) {  // eight CTAs' loads ahead of their sums
      float v[8], w[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const int b = b0 + 8 * k;
        const float* o = u.part + (size_t)min(b, u.ctas - 1) * kTrPart + o0;
        v[k] = b < u.ctas ? o[0] : 0.0f;
        w[k] = pair && b < u.ctas ? o[256] : 0.0f;
      }
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        two_sum(ps, pe, v[k]);
        pe += w[k];
      }
    }
    red[tid >> 5][tid & 31] = (double)ps + (double)pe;
    __syncthreads();
    if (tid < 32) {
      double t = 0.0;
      for (int k = 0; k < 8; ++k) t += red[k][tid];
      apply(sec < 8 ? kOffW1 + q : (sec == 8 ? kOffB1 : sec == 9 ? kOffB2 : kOffW3) + c, (float)t);
    }
    return;
  }
  __shared__ double rd[256][2];
  double l = 0.0, d = 0.0;
  for (int b = tid; b < u.ctas; b += 256) {
    l += u.partd[2 * b];
    d += u.partd[2 * b + 1];
  }
  rd[tid][0] = l;
  rd[tid][1] = d;
  __syncthreads();
  for (int h = 128; h > 0; h >>= 1) {
    if (tid < h) {
      rd[tid][0] += rd[tid + h][0];
      rd[tid][1] += rd[tid + h][1];
    }
    __syncthreads();
  }
  if (tid == 0) {
    if (u.loss) *u.loss = rd[0][0];
    apply(kOffB3, (float)rd[0][1]);
  }
}

// W2 transposed, for the first gradient of a call
__global__ void mlp_transpose_kernel(const float* __restrict__ w2, float* __restrict__ w2t) {
  __shared__ float t[32][33];
  for (int k = threadIdx.y; k < 32; k += 8) t[k][threadIdx.x] = w2[(blockIdx.y * 32 + k) * 256 + blockIdx.x * 32 + threadIdx.x];
  __syncthreads();
  for (int k = threadIdx.y; k < 32; k += 8) w2t[(blockIdx.x * 32 + k) * 256 + blockIdx.y * 32 + threadIdx.x] = t[threadIdx.x][k];
}

}  // namespace lsk
