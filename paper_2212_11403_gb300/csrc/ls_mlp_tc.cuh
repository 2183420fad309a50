// ls_mlp_tc.cuh -- the proposal network's scorer on the fifth-generation tensor cores (tcgen05).
//
// scores[r] = w3 . relu(W2^T relu(W1^T x_r + b1) + b2) + b3 for n rows of BF16 features, in tiles
// of 128 rows, one persistent CTA of 18 warps per SM.  Both products run on the tensor cores,
// issued by one thread, FP32 accumulators in tensor memory:
//   layer 1: one tcgen05.mma (M = 128, N = 256, K = 16: the 7 features zero-padded) of the feature
//            tile by W1;
//   layer 2: sixteen tcgen05.mma (M = 128, N = 256, K = 16 each) of the BF16 hidden tile by W2.
// The CUDA cores only move data between them: epilogue 1 reads the layer-1 accumulator back with
// tcgen05.ld, adds b1, applies ReLU while rounding to BF16 (one cvt.rn.relu.bf16x2 per pair) and
// writes the hidden tile into shared memory; epilogue 2 reads the layer-2 accumulator, adds b2,
// applies ReLU and takes the dot product with w3 in FP32 (warp w: TMEM lanes 32 (w % 4).. = rows,
// columns of half w / 4; the halves meet through shared memory).
//
// Pipeline: the warps have roles (8 for epilogue 1, 8 for epilogue 2, one issues the tensor-core work,
// one loads features) and meet only at mbarriers.  Two 256-column accumulators in tensor memory (512
// columns): tile t uses buffer t % 2 for both of its layers.  Layer 2 runs over the hidden tile's four
// 64-column atoms and releases each as it is done with it, so that epilogue 1 of tile t+1 refills atom
// by atom behind it; tile t+1's layer 1 is issued between tile t's atoms (after kTcNext of them), by
// when epilogue 2 has drained its buffer.  The tensor pipe needs
// 2176 cycles a tile and its operands 1632 of the shared memory's; a tile takes about 3800 (before, with
// one set of warps for both epilogues and the biases in shared memory: 4500).  12.64 M BF16 rows:
// 1.50 -> 1.26 ms; 2 M float rows: 248 us after a conversion pass of 88 us -> 207 us with none.  Issuing
// the next layer 1 after one or three atoms instead of two costs 2 and 6 % more.
//
// Operand layouts (shared memory, K-major).  W2^T and the hidden tile: 128-byte swizzle, a matrix of
// R rows x 256 BF16 columns is four 64-column atoms of R rows x 128 bytes, row r of an atom at byte
// 128 r, its 16-byte chunk c stored at chunk c ^ (r % 8), atoms on 1024-byte boundaries (the
// hardware's swizzle XORs address bits 4-6 with bits 7-9); the k-th 16-column slice is atom k / 4
// shifted by 32 (k % 4) bytes, 8-row groups 1024 bytes apart.  W1^T and the feature tile (16
// columns): no swizzle, 8-row x 16-byte core matrices, the two along K 128 bytes apart and
// consecutive 8-row groups 256 bytes apart.
//
// The network's parameters are staged once per CTA.  Every wait has a time limit; on a timeout the
// CTA records it in *err, stops, waits for its tensor-core work and frees its tensor memory.
#pragma once

#include <cstdint>
#include <type_traits>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

namespace lsk {

constexpr int kTcThreads = 576;                    // warps 0-7 epilogue 1, 8-15 epilogue 2, 16 issue, 17 features
constexpr int kTcNext = 2;                         // atoms of layer 2 issued before the next tile's layer 1
constexpr int kTcRows = 128;                       // rows per tile (M)
constexpr int kTcCols = 256;                       // hidden units (N of both layers, K of layer 2)
constexpr int kTcB = 0;                            // W2^T as the B operand: 4 atoms x 256 rows x 128 B
constexpr int kTcA = kTcB + 4 * kTcCols * 128;     // hidden tile as the A operand: 4 atoms x 128 rows x 128 B
constexpr int kTcW1 = kTcA + 4 * kTcRows * 128;    // W1^T as the B operand of layer 1: 256 rows x 32 B
constexpr int kTcX = kTcW1 + kTcCols * 32;         // two feature tiles as the A operand of layer 1: 128 rows x 32 B
constexpr int kTcPart = kTcX + 2 * kTcRows * 32;    // partial scores of the second column half [128]
constexpr int kTcBar = kTcPart + kTcRows * 4;       // mbarriers (8 B each), then tensor-memory address and abort flag
enum TcBar { kBarX = 0, kBarXFree = 2, kBarZ1 = 4, kBarA = 5, kBarAFree = 6, kBarZ2 = 10, kBarZFree = 12, kBarDone = 14, kTcBars = 15 };
constexpr int kTcBytes = kTcBar + kTcBars * 8 + 8;
constexpr int kTcSmem = kTcBytes + 1024;           // + alignment of the base to 1024 bytes
constexpr int kTcTmemCols = 2 * kTcCols;           // two accumulators

__device__ __forceinline__ uint32_t tc_smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ uint32_t tc_pack_bf16(float lo, float hi) {  // round to nearest even
  const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&v);
}

// shared-memory matrix descriptor: K-major, 128-byte swizzle, 8-row groups 1024 bytes apart
__device__ __forceinline__ uint64_t tc_desc(uint32_t saddr) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);  // start address
  d |= (uint64_t)1 << 16;                    // leading-dimension offset (unused for this layout)
  d |= (uint64_t)(1024 >> 4) << 32;          // stride-dimension offset
  d |= (uint64_t)1 << 46;                    // descriptor version
  d |= (uint64_t)2 << 61;                    // swizzle: 128 bytes
  return d;
}

// shared-memory matrix descriptor: K-major, no swizzle, 8-row x 16-byte core matrices, the next
// core matrix along K 128 bytes on, the next 8-row group 256 bytes on (a 16-column operand)
__device__ __forceinline__ uint64_t tc_desc_k16(uint32_t saddr) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);  // start address
  d |= (uint64_t)(128 >> 4) << 16;           // leading-dimension (K) offset
  d |= (uint64_t)(256 >> 4) << 32;           // stride-dimension (M/N) offset
  d |= (uint64_t)1 << 46;                    // descriptor version; swizzle field 0: none
  return d;
}
// byte offset of the 16-byte chunk c (columns 8c..8c+7) of row r in that layout
__device__ __forceinline__ uint32_t tc_off_k16(int r, int c) {
  return (uint32_t)((r >> 3) * 256 + c * 128 + (r & 7) * 16);
}

// (relu(lo), relu(hi)) rounded to BF16, lo in the low half
__device__ __forceinline__ uint32_t tc_relu_bf16x2(float lo, float hi) {
  uint32_t d;
  asm("cvt.rn.relu.bf16x2.f32 %0, %1, %2;" : "=r"(d) : "f"(hi), "f"(lo));
  return d;
}

// instruction descriptor of kind::f16: D FP32, A and B BF16, both K-major, N = 256, M = 128
constexpr uint32_t kTcIdesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(kTcCols >> 3) << 17) |
                              ((uint32_t)(kTcRows >> 4) << 24);

__device__ __forceinline__ void tc_mma(uint32_t dtmem, uint64_t adesc, uint64_t bdesc, uint32_t accumulate) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(dtmem),
      "l"(adesc), "l"(bdesc), "r"(kTcIdesc), "r"(accumulate)
      : "memory");
}

__device__ __forceinline__ bool tc_mbar_test(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}

__device__ __forceinline__ uint64_t tc_now_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// 32 consecutive accumulator columns of this thread's lane: requested by tc_ld32, there after
// tc_ld_wait (which carries the registers, so nothing reads them before the load has landed)
__device__ __forceinline__ void tc_ld32(uint32_t taddr, uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
      "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]),
        "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]),
        "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]),
        "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr));
}
__device__ __forceinline__ void tc_ld_wait(uint32_t (&r)[32]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
                 "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]),
                 "+r"(r[15]), "+r"(r[16]), "+r"(r[17]), "+r"(r[18]), "+r"(r[19]), "+r"(r[20]), "+r"(r[21]),
                 "+r"(r[22]), "+r"(r[23]), "+r"(r[24]), "+r"(r[25]), "+r"(r[26]), "+r"(r[27]), "+r"(r[28]),
                 "+r"(r[29]), "+r"(r[30]), "+r"(r[31])
               :
               : "memory");
}

// byte offset of element (row, col) of a K-major, 128-byte-swizzled operand with R rows
__device__ __forceinline__ uint32_t tc_off(int R, int row, int col) {
  const int atom = col >> 6, chunk = (col >> 3) & 7;
  return (uint32_t)(atom * R * 128 + row * 128 + ((chunk ^ (row & 7)) << 4) + ((col & 7) << 1));
}

// The FP32 vectors are kernel parameters: the epilogues read them through the constant bank, because
// the shared memory's bandwidth is taken by the tensor cores' operands (96 of 128 bytes a cycle) and
// the hidden tile.
struct MlpTcDev {
  float b1[kTcCols], b2[kTcCols], w3[kTcCols];
  float b3;
  const __nv_bfloat16* w1t;  // [256][16]  w1t[n][k] = W1[k][n]
  const __nv_bfloat16* w2t;  // [256][256] w2t[n][k] = W2[k][n]
  int* err;                  // set to 1 when a wait ran out of time
};

// the same, suspended in hardware for a short time while the phase is not complete (a nanosleep between
// polls overslept the handovers between the roles by 0.15 us a tile)
__device__ __forceinline__ bool tc_mbar_try(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}

// wait for phase `parity` of an mbarrier for at most ~2 s; on a timeout the CTA's abort flag makes every
// other wait give up too
__device__ __forceinline__ bool tc_wait(uint32_t bar, uint32_t parity, volatile int* abort) {
  if (tc_mbar_try(bar, parity)) return true;
  const uint64_t t0 = tc_now_ns();
  while (!tc_mbar_try(bar, parity)) {
    if (*abort) return false;
    if (tc_now_ns() - t0 > 2000000000ull) {
      *abort = 1;
      return false;
    }
  }
  return true;
}
// the same answer in every lane of the warp
__device__ __forceinline__ bool tc_wait_warp(uint32_t bar, uint32_t parity, volatile int* abort) {
  return __all_sync(0xffffffffu, tc_wait(bar, parity, abort));
}
__device__ __forceinline__ void tc_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

__device__ __forceinline__ void tc_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}

// Features of row r as eight BF16 values.  Rows are 8 BF16 values (16-byte aligned), or 8 floats.
__device__ __forceinline__ uint4 tc_row(const __nv_bfloat16* X, long long r) {
  return *reinterpret_cast<const uint4*>(X + (size_t)r * 8);
}
__device__ __forceinline__ uint4 tc_row(const float* X, long long r) {
  const float* x = X + (size_t)r * 8;
  float v[8];
  if ((reinterpret_cast<uintptr_t>(X) & 15) == 0) {
    const float4 a = *reinterpret_cast<const float4*>(x), b = *reinterpret_cast<const float4*>(x + 4);
    v[0] = a.x, v[1] = a.y, v[2] = a.z, v[3] = a.w, v[4] = b.x, v[5] = b.y, v[6] = b.z, v[7] = b.w;
  } else {
#pragma unroll
    for (int k = 0; k < 8; ++k) v[k] = x[k];
  }
  return make_uint4(tc_pack_bf16(v[0], v[1]), tc_pack_bf16(v[2], v[3]), tc_pack_bf16(v[4], v[5]), tc_pack_bf16(v[6], v[7]));
}

template <class T>
__global__ void __launch_bounds__(kTcThreads, 1) mlp_score_tc_kernel(const __grid_constant__ MlpTcDev m, const T* __restrict__ X,
                                                                     long long n, float* __restrict__ scores) {
  extern __shared__ unsigned char tc_raw[];
  const uint32_t raw = tc_smem_u32(tc_raw);
  unsigned char* sm = tc_raw + (((raw + 1023u) & ~1023u) - raw);  // 1024-byte aligned base
  const uint32_t base = tc_smem_u32(sm);
  float* part = reinterpret_cast<float*>(sm + kTcPart);
  uint32_t* tslot = reinterpret_cast<uint32_t*>(sm + kTcBar + kTcBars * 8);
  volatile int* abort = reinterpret_cast<volatile int*>(sm + kTcBar + kTcBars * 8 + 4);
  auto bar = [&](int k) { return base + kTcBar + 8 * (uint32_t)k; };
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

  // stage W2^T (swizzled), W1^T (16 columns, no swizzle); columns 8..15 of the feature tiles
  // stay zero
  for (int e = tid; e < kTcCols * kTcCols / 8; e += kTcThreads) {
    const int row = e >> 5, c8 = (e & 31) << 3;  // row n of W2^T, first of 8 columns k
    const uint4 v = *reinterpret_cast<const uint4*>(m.w2t + (size_t)row * kTcCols + c8);
    *reinterpret_cast<uint4*>(sm + kTcB + tc_off(kTcCols, row, c8)) = v;
  }
  for (int e = tid; e < kTcCols * 2; e += kTcThreads) {
    const int row = e >> 1, c = e & 1;
    *reinterpret_cast<uint4*>(sm + kTcW1 + tc_off_k16(row, c)) = *reinterpret_cast<const uint4*>(m.w1t + row * 16 + 8 * c);
  }
  for (int e = tid; e < 2 * kTcRows; e += kTcThreads)
    *reinterpret_cast<uint4*>(sm + kTcX + (e >> 7) * kTcRows * 32 + tc_off_k16(e & 127, 1)) = make_uint4(0u, 0u, 0u, 0u);
  if (tid == 0) {
    *abort = 0;
    for (int k = 0; k < kTcBars; ++k) {
      // arrivals: one per epilogue-1 warp (A), one per epilogue-2 warp (ZFree), else one
      const uint32_t count = (k == kBarA || k == kBarZFree || k == kBarZFree + 1) ? 8u : 1u;
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar(k)), "r"(count) : "memory");
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 16) {  // two 256-column accumulators (128 lanes x FP32)
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(tc_smem_u32(tslot)),
                 "r"(kTcTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // the staged weights, to the tensor cores
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tslot;
  const long long ntile = (n + kTcRows - 1) / kTcRows;
  const long long G = gridDim.x;
  const int count = (int)((ntile - blockIdx.x + G - 1) / G);  // tiles of this CTA: blockIdx.x, + G, ...
  auto tile = [&](int i) { return blockIdx.x + (long long)i * G; };
  // this thread's accumulator lane (= row of the tile)
  const int erow = 32 * (warp & 3) + lane;
  const uint32_t lane_off = (uint32_t)(32 * (warp & 3)) << 16;

  // epilogue 1: b1, ReLU, BF16 into the hidden tile (the A operand of layer 2); warps 0-3 take the first
  // 32 columns of each atom (HALF 0), warps 4-7 the others.  The half is a compile-time argument so
  // that every constant has a fixed address.
  auto epilogue1 = [&](auto half) {
    constexpr int HALF = decltype(half)::value;
    for (int i = 0; i < count; ++i) {
      const uint32_t d = tmem + (uint32_t)((i & 1) * kTcCols);
      if (!tc_wait_warp(bar(kBarZ1), (uint32_t)i & 1u, abort)) return;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      uint32_t r[2][32];  // the next columns are requested before the current ones are worked on
      tc_ld32(d + lane_off + (uint32_t)(32 * HALF), r[0]);
#pragma unroll
      for (int a = 0; a < 4; ++a) {
        const int c0 = 64 * a + 32 * HALF;
        const uint32_t(&v)[32] = r[a & 1];
        tc_ld_wait(r[a & 1]);
        if (a < 3) tc_ld32(d + lane_off + (uint32_t)(c0 + 64), r[(a + 1) & 1]);
        uint4 pk[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          uint32_t w[4];
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const int k = 8 * q + 2 * e;
            const float2 h = __fadd2_rn(make_float2(__uint_as_float(v[k]), __uint_as_float(v[k + 1])),
                                        make_float2(m.b1[c0 + k], m.b1[c0 + k + 1]));
            w[e] = tc_relu_bf16x2(h.x, h.y);
          }
          pk[q] = make_uint4(w[0], w[1], w[2], w[3]);
        }
        // the previous tile's layer 2 has read the atom
        if (i > 0 && !tc_wait_warp(bar(kBarAFree + a), (uint32_t)(i - 1) & 1u, abort)) return;
#pragma unroll
        for (int q = 0; q < 4; ++q) *reinterpret_cast<uint4*>(sm + kTcA + tc_off(kTcRows, erow, c0 + 8 * q)) = pk[q];
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncwarp();
      if (lane == 0) tc_arrive(bar(kBarA));
    }
  };
  // epilogue 2: b2, ReLU and the dot product with w3; warps 8-11 take columns 0..127 (HALF 0), warps
  // 12-15 the others, and the halves meet in shared memory
  auto epilogue2 = [&](auto half) {
    constexpr int HALF = decltype(half)::value;
    for (int i = 0; i < count; ++i) {
      const uint32_t d = tmem + (uint32_t)((i & 1) * kTcCols);
      const bool ok = tc_wait(bar(kBarZ2 + (i & 1)), (uint32_t)(i >> 1) & 1u, abort);
      uint32_t all;  // one answer for the eight warps, which also orders the reads of part before its next writes
      asm volatile(
          "{\n .reg .pred p, q;\n setp.ne.u32 p, %1, 0;\n barrier.cta.red.and.pred q, 1, 256, p;\n selp.u32 %0, 1, 0, q;\n}\n"
          : "=r"(all)
          : "r"(ok ? 1u : 0u)
          : "memory");
      if (!all) return;
      __syncwarp();
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      float2 acc[4] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f), make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
      uint32_t r[2][32];
      tc_ld32(d + lane_off + (uint32_t)(128 * HALF), r[0]);
#pragma unroll
      for (int b = 0; b < 4; ++b) {
        const int c0 = 128 * HALF + 32 * b;
        const uint32_t(&v)[32] = r[b & 1];
        tc_ld_wait(r[b & 1]);
        if (b < 3) {
          tc_ld32(d + lane_off + (uint32_t)(c0 + 32), r[(b + 1) & 1]);
        } else {  // the accumulator has been read: it may take a later tile's layer 1
          asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
          __syncwarp();
          if (lane == 0) tc_arrive(bar(kBarZFree + (i & 1)));
        }
#pragma unroll
        for (int k = 0; k < 32; k += 4) {
          const int c = c0 + k;
          const float2 h01 = __fadd2_rn(make_float2(__uint_as_float(v[k]), __uint_as_float(v[k + 1])),
                                        make_float2(m.b2[c], m.b2[c + 1]));
          const float2 h23 = __fadd2_rn(make_float2(__uint_as_float(v[k + 2]), __uint_as_float(v[k + 3])),
                                        make_float2(m.b2[c + 2], m.b2[c + 3]));
          acc[(k >> 2) & 1] = __ffma2_rn(make_float2(fmaxf(h01.x, 0.f), fmaxf(h01.y, 0.f)),
                                         make_float2(m.w3[c], m.w3[c + 1]), acc[(k >> 2) & 1]);
          acc[2 + ((k >> 2) & 1)] = __ffma2_rn(make_float2(fmaxf(h23.x, 0.f), fmaxf(h23.y, 0.f)),
                                               make_float2(m.w3[c + 2], m.w3[c + 3]), acc[2 + ((k >> 2) & 1)]);
        }
      }
      const float s = ((acc[0].x + acc[0].y) + (acc[1].x + acc[1].y)) + ((acc[2].x + acc[2].y) + (acc[3].x + acc[3].y));
      if (HALF == 1) part[erow] = s;
      asm volatile("barrier.cta.sync 1, 256;" ::: "memory");
      const long long er = tile(i) * kTcRows + erow;
      if (HALF == 0 && er < n) scores[er] = (s + part[erow]) + m.b3;
    }
  };
  if (warp < 4) {
    epilogue1(std::integral_constant<int, 0>{});
  } else if (warp < 8) {
    epilogue1(std::integral_constant<int, 1>{});
  } else if (warp < 12) {
    epilogue2(std::integral_constant<int, 0>{});
  } else if (warp < 16) {
    epilogue2(std::integral_constant<int, 1>{});
  } else if (warp == 16) {
    if (lane == 0) {  // tensor-core issue: layer 1 of a tile into accumulator i % 2, layer 2 likewise
      auto layer1 = [&](int i) -> bool {
        if (!tc_wait(bar(kBarX + (i & 1)), (uint32_t)(i >> 1) & 1u, abort)) return false;
        if (i >= 2 && !tc_wait(bar(kBarZFree + (i & 1)), (uint32_t)((i >> 1) - 1) & 1u, abort)) return false;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        tc_mma(tmem + (uint32_t)((i & 1) * kTcCols), tc_desc_k16(base + kTcX + (uint32_t)((i & 1) * kTcRows * 32)),
               tc_desc_k16(base + kTcW1), 0u);
        tc_commit(bar(kBarZ1));
        tc_commit(bar(kBarXFree + (i & 1)));
        return true;
      };
      bool ok = layer1(0);
      for (int i = 0; ok && i < count; ++i) {
        const uint32_t d = tmem + (uint32_t)((i & 1) * kTcCols);
        if (!(ok = tc_wait(bar(kBarA), (uint32_t)i & 1u, abort))) break;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll 1
        for (int a = 0; a < 4; ++a) {
          if (a == kTcNext && i + 1 < count && !(ok = layer1(i + 1))) break;
#pragma unroll
          for (int k = 0; k < 4; ++k)  // 16 columns = 32 bytes within the atom
            tc_mma(d, tc_desc(base + kTcA + (uint32_t)(a * kTcRows * 128 + k * 32)),
                   tc_desc(base + kTcB + (uint32_t)(a * kTcCols * 128 + k * 32)), a + k > 0 ? 1u : 0u);
          tc_commit(bar(kBarAFree + a));
        }
        if (ok) tc_commit(bar(kBarZ2 + (i & 1)));
      }
      // nothing is in flight when the tensor memory is freed
      tc_commit(bar(kBarDone));
      if (!tc_wait(bar(kBarDone), 0u, abort)) {
        const uint64_t t0 = tc_now_ns();
        while (!tc_mbar_test(bar(kBarDone), 0u) && tc_now_ns() - t0 < 2000000000ull) __nanosleep(100);
      }
    }
    __syncwarp();
  } else {  // features: four rows a lane, rows beyond n as zero
    for (int i = 0; i < count; ++i) {
      uint4 v[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const long long r = tile(i) * kTcRows + 32 * q + lane;
        v[q] = r < n ? tc_row(X, r) : make_uint4(0u, 0u, 0u, 0u);
      }
      if (i >= 2 && !tc_wait_warp(bar(kBarXFree + (i & 1)), (uint32_t)((i >> 1) - 1) & 1u, abort)) break;
#pragma unroll
      for (int q = 0; q < 4; ++q)
        *reinterpret_cast<uint4*>(sm + kTcX + (i & 1) * kTcRows * 32 + tc_off_k16(32 * q + lane, 0)) = v[q];
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      __syncwarp();
      if (lane == 0) tc_arrive(bar(kBarX + (i & 1)));
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  if (tid == 0 && *abort) atomicExch(m.err, 1);
  if (warp == 16)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTcTmemCols) : "memory");
}

}  // namespace lsk
