// ls_propose.cuh -- donor proposal for the sparse recursions: window match-count features, a
// first-stage pre-filter and top-K (the MLP scorer on the tensor cores is in ls_mlp_tc.cuh).
//
// Windows hold 256 consecutive loci.  For haplotypes i, j and window w the feature is the match
// count m_ij^w = n_w - popcount(h_i^w XOR h_j^w) (n_w = loci in the window).  Stage 1 keeps, for
// target i and window w, the C donors with the smallest mismatch sum over windows w-1..w+1 (ties
// to the lower donor id, never i itself).  Stage 2 scores each candidate with the MLP on the
// match fractions m^{w+d}/n_{w+d}, d = -3..3 (windows clamped to the range), and keeps the K best
// (ties to the lower id).  Sets are written in ascending donor order.
#pragma once

#include <cstdint>
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

namespace lsk {

constexpr int kPropWS = 256;       // loci per window
constexpr int kFeat = 16;          // inputs of layer 1 on the tensor cores (one k-step; a feature row holds the first 8)
constexpr int kFeatUsed = 7;
constexpr int kHidden = 256;

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
  const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&v);
}

// Haplotype-major window bits: hw[(w*N + i)*8 + k] bit b = allele of haplotype i at locus
// w*256 + 32k + b (0 beyond L).  grid (ceil(N/32), 8, Wn), one warp: a 32 x 32 bit transpose by
// ballots.
__global__ void hapmajor_kernel(const uint32_t* __restrict__ bits, int row_words, int N, int L,
                                uint32_t* __restrict__ hw) {
  const int g = blockIdx.x, k = blockIdx.y, w = blockIdx.z, lane = threadIdx.x;
  const int l = w * kPropWS + 32 * k + lane;
  const uint32_t word = l < L ? bits[(size_t)l * row_words + g] : 0u;
  uint32_t mine = 0u;
#pragma unroll
  for (int h = 0; h < 32; ++h) {
    const uint32_t b = __ballot_sync(0xffffffffu, (word >> h) & 1u);
    if (lane == h) mine = b;
  }
  const int i = 32 * g + lane;
  if (i < N) hw[((size_t)w * N + i) * 8 + k] = mine;
}

// Mismatch counts of one window, min(popcount, 255) as bytes: M[i*Np + j] (columns up to Np are written).
// 64 x 64 pairs per block of 256 threads, 4 x 4 per thread with both sides' words in registers; the counts
// are symmetric, so a block off the diagonal also writes the tile's mirror image and half the blocks have
// nothing to do.  Bound by the shared memory (94 % busy: a warp's lanes read rows of B 128 bytes apart, on the same
// banks), then by the population counts (16 a cycle and SM, eight a pair).  N = 12345: 305 -> 162 us a window
// (before, every pair counted twice with one 4-byte shared load per word).
__global__ void __launch_bounds__(256) mismatch_kernel(const uint32_t* __restrict__ hw, int N, int Np, uint8_t* __restrict__ M) {
  if (blockIdx.y > blockIdx.x) return;
  __shared__ __align__(16) uint32_t A[64][8], B[64][8];
  __shared__ uint32_t mir[64][17];  // the mirrored tile, four counts a word
  const int i0 = blockIdx.y * 64, j0 = blockIdx.x * 64, tid = threadIdx.x;
  {
    const int r = tid >> 2, k = 2 * (tid & 3);
    const uint2 z = make_uint2(0u, 0u);
    *reinterpret_cast<uint2*>(&A[r][k]) = i0 + r < N ? *reinterpret_cast<const uint2*>(hw + (size_t)(i0 + r) * 8 + k) : z;
    *reinterpret_cast<uint2*>(&B[r][k]) = j0 + r < N ? *reinterpret_cast<const uint2*>(hw + (size_t)(j0 + r) * 8 + k) : z;
  }
  __syncthreads();
  const int ti = tid >> 4, tj = tid & 15;
  uint32_t a[4][8], row[4] = {0u, 0u, 0u, 0u};
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    const uint4 lo = *reinterpret_cast<const uint4*>(&A[4 * ti + r][0]), hi = *reinterpret_cast<const uint4*>(&A[4 * ti + r][4]);
    a[r][0] = lo.x, a[r][1] = lo.y, a[r][2] = lo.z, a[r][3] = lo.w, a[r][4] = hi.x, a[r][5] = hi.y, a[r][6] = hi.z, a[r][7] = hi.w;
  }
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    const uint4 lo = *reinterpret_cast<const uint4*>(&B[4 * tj + c][0]), hi = *reinterpret_cast<const uint4*>(&B[4 * tj + c][4]);
    const uint32_t b[8] = {lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z, hi.w};
    uint32_t col = 0u;
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      int m = 0;
#pragma unroll
      for (int k = 0; k < 8; ++k) m += __popc(a[r][k] ^ b[k]);
      const uint32_t v = (uint32_t)min(m, 255);
      row[r] |= v << (8 * c);
      col |= v << (8 * r);
    }
    mir[4 * tj + c][ti] = col;
  }
#pragma unroll
  for (int r = 0; r < 4; ++r)
    if (i0 + 4 * ti + r < N) *reinterpret_cast<uint32_t*>(M + (size_t)(i0 + 4 * ti + r) * Np + j0 + 4 * tj) = row[r];
  if (blockIdx.x == blockIdx.y) return;
  __syncthreads();
  const int r = tid >> 2, q = 4 * (tid & 3);
  if (j0 + r < N)
    *reinterpret_cast<uint4*>(M + (size_t)(j0 + r) * Np + i0 + 4 * q) = make_uint4(mir[r][q], mir[r][q + 1], mir[r][q + 2], mir[r][q + 3]);
}

// Stage 1 for one window, one block (256 threads) per target i: the C donors with the smallest
// mismatch sum over the available windows among w-1..w+1 (score <= 765), ties to the lower id,
// written in ascending id order (target i's row at cand + i cstride) together with their features
// (match fractions of windows w-3..w+3, clamped).  Ms[d] = count matrix of window w+d-3 (clamped), nv[d] its locus count.
struct Stage1Args {
  const uint8_t* Ms[7];
  float inv_nv[7];
  int use[3];  // whether windows w-1, w, w+1 exist
};

// Targets with N <= kS1MaxN donors: a thread keeps the scores of 4 x 16 donors in registers as
// binary16 pairs 1024 + score (exact: scores are below 1024), finds the threshold by bisecting its ten
// bits (two packed operations per pair and bit), and the block compacts the selected ids with two
// scans; features are then read by position, consecutive threads on ascending ids.  The count rows are
// read once for the scores and once for the features, in whole lines; what bounds it is that traffic and
// the bisection's arithmetic.  N = 12345, C = 1024: 1330 -> 387 us a window (stage1_hist_kernel, whose
// shared-memory histogram costs one atomic per donor and whose features are 7 scattered bytes per
// selected donor).
constexpr int kS1Iter = 4;                        // chunks of 16 donors per thread
constexpr int kS1MaxN = 16 * kS1Iter * 1024;      // 1024 threads

template <int NT>  // largest block size: warps = ceil(N / 2048) at the launch
__global__ void __launch_bounds__(NT) stage1_kernel(Stage1Args a, int N, int Np, int C, int32_t* __restrict__ cand,
                                                    size_t cstride, __nv_bfloat16* __restrict__ feat,
                                                    float* __restrict__ feat32) {
  __shared__ int cnt_s[2][32];
  __shared__ uint2 scan_s[32];
  const int i = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nt = blockDim.x, nw = nt >> 5;
  const uint8_t* r0 = a.use[0] ? a.Ms[2] + (size_t)i * Np : nullptr;
  const uint8_t* r1 = a.Ms[3] + (size_t)i * Np;
  const uint8_t* r2 = a.use[2] ? a.Ms[4] + (size_t)i * Np : nullptr;
  // sc[t][2m], sc[t][2m + 1]: donors (4m, 4m + 2) and (4m + 1, 4m + 3) of chunk t, low half first
  uint32_t sc[kS1Iter][8];
#pragma unroll
  for (int t = 0; t < kS1Iter; ++t) {
    const int j0 = 16 * (t * nt + tid);
#pragma unroll
    for (int m = 0; m < 8; ++m) sc[t][m] = 0x64006400u;
    auto add = [&](const uint8_t* r) {
      const uint4 v = *reinterpret_cast<const uint4*>(r + j0);  // rows are 16-byte multiples (Np a multiple of 64)
      const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        sc[t][2 * m] += w[m] & 0x00ff00ffu;
        sc[t][2 * m + 1] += (w[m] >> 8) & 0x00ff00ffu;
      }
    };
    if (j0 < N) {
      if (r0) add(r0);
      add(r1);
      if (r2) add(r2);
    }
    if (j0 + 16 > N || (unsigned)(i - j0) < 16u) {  // donors beyond N and the target: never below a threshold
#pragma unroll
      for (int k = 0; k < 16; ++k)
        if (j0 + k >= N || j0 + k == i) sc[t][2 * (k >> 2) + (k & 1)] |= (k & 2) ? 0x67ff0000u : 0x67ffu;
    }
  }
  // T: the largest t with #{score < t} < C; n_lt = #{score < T}.  A t with #{score < t} = C ends the
  // search (nothing is taken at the threshold then).
  int T = 0, n_lt = 0;
  for (int bit = 512, ph = 0; bit; bit >>= 1, ph ^= 1) {
    const int t = T | bit;
    const uint32_t tt = (uint32_t)(0x6400 + t) * 0x10001u;
    const __half2 th = *reinterpret_cast<const __half2*>(&tt);
    __half2 c0 = __float2half2_rn(0.0f), c1 = c0;  // counts of at most 32 per half: exact
#pragma unroll
    for (int q = 0; q < kS1Iter; ++q)
#pragma unroll
      for (int m = 0; m < 8; m += 2) {
        c0 = __hadd2(c0, __hlt2(*reinterpret_cast<const __half2*>(&sc[q][m]), th));
        c1 = __hadd2(c1, __hlt2(*reinterpret_cast<const __half2*>(&sc[q][m + 1]), th));
      }
    c0 = __hadd2(c0, c1);
    const int mine = (int)(__low2float(c0) + __high2float(c0));
    const int wsum = __reduce_add_sync(0xffffffffu, mine);
    if (lane == 0) cnt_s[ph][warp] = wsum;
    __syncthreads();
    const int n = __reduce_add_sync(0xffffffffu, lane < nw ? cnt_s[ph][lane] : 0);
    if (n <= C) {
      T = t;
      n_lt = n;
    }
    if (n == C) break;
  }
  const int need_eq = C - n_lt;
  // donors below / at the threshold, 16 bits per chunk
  uint32_t ltm[kS1Iter], eqm[kS1Iter];
#pragma unroll
  for (int t = 0; t < kS1Iter; ++t) {
    ltm[t] = eqm[t] = 0u;
#pragma unroll
    for (int k = 0; k < 16; ++k) {
      const int s = (int)((sc[t][2 * (k >> 2) + (k & 1)] >> ((k & 2) ? 16 : 0)) & 0xffffu) - 0x6400;
      ltm[t] |= (s < T ? 1u : 0u) << k;
      eqm[t] |= (s == T && s < 1023 ? 1u : 0u) << k;
    }
  }
  // exclusive prefixes over the block of four 16-bit counts per thread (chunk t of every thread comes
  // before chunk t + 1 of any), and the block totals
  auto scan = [&](const uint32_t (&m)[kS1Iter], int (&pre)[kS1Iter]) -> int {
    const uint2 own = make_uint2(__popc(m[0]) | (__popc(m[1]) << 16), __popc(m[2]) | (__popc(m[3]) << 16));
    uint2 x = own;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const uint32_t ya = __shfl_up_sync(0xffffffffu, x.x, off), yb = __shfl_up_sync(0xffffffffu, x.y, off);
      if (lane >= off) {
        x.x += ya;
        x.y += yb;
      }
    }
    __syncthreads();  // the previous scan's words have been read
    if (lane == 31) scan_s[warp] = x;
    __syncthreads();
    const uint2 v = lane < nw ? scan_s[lane] : make_uint2(0u, 0u);
    const uint32_t ta = __reduce_add_sync(0xffffffffu, v.x), tb = __reduce_add_sync(0xffffffffu, v.y);
    const uint32_t wa = __reduce_add_sync(0xffffffffu, lane < warp ? v.x : 0u);
    const uint32_t wb = __reduce_add_sync(0xffffffffu, lane < warp ? v.y : 0u);
    const uint32_t pa = wa + x.x - own.x, pb = wb + x.y - own.y;
    const int t0 = (int)(ta & 0xffffu), t1 = (int)(ta >> 16), t2 = (int)(tb & 0xffffu), t3 = (int)(tb >> 16);
    pre[0] = (int)(pa & 0xffffu);
    pre[1] = t0 + (int)(pa >> 16);
    pre[2] = t0 + t1 + (int)(pb & 0xffffu);
    pre[3] = t0 + t1 + t2 + (int)(pb >> 16);
    return t0 + t1 + t2 + t3;
  };
  int pre[kS1Iter];
  scan(eqm, pre);
  uint32_t selm[kS1Iter];  // equal scores are taken in ascending id until need_eq of them are in
#pragma unroll
  for (int t = 0; t < kS1Iter; ++t) {
    selm[t] = ltm[t];
    for (uint32_t m = eqm[t]; m && pre[t] < need_eq; m &= m - 1u, ++pre[t]) selm[t] |= m & (~m + 1u);
  }
  const int nsel = min(scan(selm, pre), C);
  int32_t* ci = cand + i * cstride;
#pragma unroll
  for (int t = 0; t < kS1Iter; ++t) {
    int pos = pre[t];
    for (uint32_t m = selm[t]; m; m &= m - 1u, ++pos) ci[pos] = 16 * (t * nt + tid) + __ffs(m) - 1;
  }
  for (int q = nsel + tid; q < C; q += nt) ci[q] = -1;  // fewer than C donors (C >= N)
  if (!feat && !feat32) return;
  __syncthreads();  // the block's ids are visible to all its threads
  for (int q = tid; q < nsel; q += nt) {
    const int j = ci[q];
    float f[kFeatUsed];
#pragma unroll
    for (int d = 0; d < kFeatUsed; ++d) f[d] = 1.0f - (float)a.Ms[d][(size_t)i * Np + j] * a.inv_nv[d];
    if (feat) {
      uint4 lo;
      lo.x = pack_bf16(f[0], f[1]);
      lo.y = pack_bf16(f[2], f[3]);
      lo.z = pack_bf16(f[4], f[5]);
      lo.w = pack_bf16(f[6], 0.0f);
      *reinterpret_cast<uint4*>(feat + ((size_t)i * C + q) * 8) = lo;
    }
    if (feat32) {
      float* fo = feat32 + ((size_t)i * C + q) * 8;
#pragma unroll
      for (int d = 0; d < 8; ++d) fo[d] = d < kFeatUsed ? f[d] : 0.0f;
    }
  }
}

// The same for any N, with a histogram of the scores in shared memory: beyond kS1MaxN donors, which the
// registers of one block cannot hold.
__global__ void __launch_bounds__(256) stage1_hist_kernel(Stage1Args a, int N, int Np, int C, int32_t* __restrict__ cand,
                                                     size_t cstride,
                                                     __nv_bfloat16* __restrict__ feat, float* __restrict__ feat32) {
  constexpr int NB = 768, NT = 256, V = 16;  // score bins, threads, donors per thread per pass step
  __shared__ int hist[8][NB];                // one histogram per warp (fewer colliding atomics)
  __shared__ int scan_s[8];
  __shared__ int thr_s, need_eq_s;
  const int i = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  // the three windows' rows of target i (16-byte aligned: Np is a multiple of 64)
  const uint8_t* r0 = a.use[0] ? a.Ms[2] + (size_t)i * Np : nullptr;
  const uint8_t* r1 = a.use[1] ? a.Ms[3] + (size_t)i * Np : nullptr;
  const uint8_t* r2 = a.use[2] ? a.Ms[4] + (size_t)i * Np : nullptr;
  auto load16 = [](const uint8_t* r, int j0) -> uint4 {
    return r ? *reinterpret_cast<const uint4*>(r + j0) : make_uint4(0u, 0u, 0u, 0u);
  };
  auto byte_of = [](const uint4& v, int k) -> int {
    const uint32_t w = k < 4 ? v.x : (k < 8 ? v.y : (k < 12 ? v.z : v.w));
    return (int)((w >> (8 * (k & 3))) & 255u);
  };
  // exclusive prefix of v over the block (thread order) and the block total; two barriers
  auto block_scan = [&](int v, int& total) -> int {
    int x = v;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, x, off);
      if (lane >= off) x += y;
    }
    if (lane == 31) scan_s[warp] = x;
    __syncthreads();
    int wpre = 0, tot = 0;
#pragma unroll
    for (int w2 = 0; w2 < 8; ++w2) {
      const int s = scan_s[w2];
      wpre += w2 < warp ? s : 0;
      tot += s;
    }
    __syncthreads();
    total = tot;
    return wpre + x - v;
  };

  for (int b = tid; b < 8 * NB; b += NT) (&hist[0][0])[b] = 0;
  if (tid == 0) {
    thr_s = NB - 1;  // fewer than C donors: every donor is below the threshold
    need_eq_s = 0;
  }
  __syncthreads();
  for (int j0 = V * tid; j0 < N; j0 += V * NT) {
    const uint4 a0 = load16(r0, j0), a1 = load16(r1, j0), a2 = load16(r2, j0);
#pragma unroll
    for (int k = 0; k < V; ++k) {
      const int j = j0 + k;
      if (j < N && j != i) atomicAdd(&hist[warp][byte_of(a0, k) + byte_of(a1, k) + byte_of(a2, k)], 1);
    }
  }
  __syncthreads();
  // threshold: the smallest T with #{score <= T} >= C; thread t owns bins 3t .. 3t+2
  {
    int c[3];
#pragma unroll
    for (int e = 0; e < 3; ++e) {
      int s = 0;
#pragma unroll
      for (int w2 = 0; w2 < 8; ++w2) s += hist[w2][3 * tid + e];
      c[e] = s;
    }
    int total;
    int acc = block_scan(c[0] + c[1] + c[2], total);
#pragma unroll
    for (int e = 0; e < 3; ++e) {
      if (acc < C && acc + c[e] >= C) {
        thr_s = 3 * tid + e;
        need_eq_s = C - acc;
      }
      acc += c[e];
    }
  }
  __syncthreads();
  const int T = thr_s, need_eq = need_eq_s;
  int base_sel = 0, eq_seen = 0;
  for (int jc = 0; jc < N; jc += V * NT) {  // the same trip count in every thread (block scans inside)
    const int j0 = jc + V * tid;
    uint32_t ltm = 0u, eqm = 0u;  // donors of this thread's 16 below / at the threshold
    if (j0 < N) {
      const uint4 a0 = load16(r0, j0), a1 = load16(r1, j0), a2 = load16(r2, j0);
#pragma unroll
      for (int k = 0; k < V; ++k) {
        const int j = j0 + k;
        const int sc = (j < N && j != i) ? byte_of(a0, k) + byte_of(a1, k) + byte_of(a2, k) : 1 << 30;
        ltm |= (sc < T ? 1u : 0u) << k;
        eqm |= (sc == T ? 1u : 0u) << k;
      }
    }
    // equal scores are taken in ascending j until need_eq of them are in
    int eq_tot;
    int r = eq_seen + block_scan(__popc(eqm), eq_tot);
    uint32_t selm = ltm;
    for (uint32_t m = eqm; m; m &= m - 1u) {
      if (r < need_eq) selm |= m & (~m + 1u);
      ++r;
    }
    int sel_tot;
    int pos = base_sel + block_scan(__popc(selm), sel_tot);
    for (uint32_t m = selm; m; m &= m - 1u, ++pos) {
      if (pos >= C) break;
      const int j = j0 + __ffs(m) - 1;
      cand[i * cstride + pos] = j;
      float f[kFeatUsed];
#pragma unroll
      for (int d = 0; d < kFeatUsed; ++d) f[d] = 1.0f - (float)a.Ms[d][(size_t)i * Np + j] * a.inv_nv[d];
      if (feat) {
        __nv_bfloat16* fo = feat + ((size_t)i * C + pos) * 8;
#pragma unroll
        for (int d = 0; d < 8; ++d) fo[d] = __float2bfloat16_rn(d < kFeatUsed ? f[d] : 0.0f);
      }
      if (feat32) {
        float* fo = feat32 + ((size_t)i * C + pos) * 8;
#pragma unroll
        for (int d = 0; d < 8; ++d) fo[d] = d < kFeatUsed ? f[d] : 0.0f;
      }
    }
    base_sel += sel_tot;
    eq_seen += eq_tot;
  }
  // fewer than C donors (C >= N): pad with -1
  for (int q = base_sel + tid; q < C; q += NT) cand[i * cstride + q] = -1;
}

// Stage 2, one warp per target: the K best of C candidates by score (higher first, ties to the lower
// id; -1 entries score -3e38 and lose ties), written to idx[(i*Wn + w)*K ...] in ascending id order.
// Stage 1 hands the candidates over in ascending id order with the -1 entries last, so position order
// is id order and nothing has to be sorted: the K-th largest score is found by bisection over the 32
// bits of an order-preserving integer key held in registers (V keys a lane, key v of lane q is
// candidate 32 v + q), and the selected candidates are compacted in position order by ballots.  It is
// bound by the latency of its loads with few warps in flight, then by the compares; no barrier.  12345 targets, C = 1024, K = 512: 988 -> 173 us a
// window (before: two bitonic sorts in shared memory per target; 246 us without the shared leading
// bits and the early end).
template <int V>
__global__ void __launch_bounds__(256) topk_kernel(const int32_t* __restrict__ cand, const float* __restrict__ scores, int N,
                                                   int C, int K, int Wn, int w, int32_t* __restrict__ idx) {
  const int lane = threadIdx.x & 31;
  const int i = blockIdx.x * 8 + (threadIdx.x >> 5);
  if (i >= N) return;
  const int32_t* ci = cand + (size_t)i * C;
  uint32_t key[V];
#pragma unroll
  for (int v = 0; v < V; ++v) {
    const int q = 32 * v + lane;
    key[v] = 0u;  // beyond C: below every key of a candidate
    if (q < C) {
      const float f = (ci[q] >= 0 ? scores[(size_t)i * C + q] : -3.0e38f) + 0.0f;  // -0 becomes +0: they tie
      const uint32_t u = __float_as_uint(f);
      key[v] = u ^ ((u >> 31) ? 0xffffffffu : 0x80000000u);
    }
  }
  // T becomes the largest value with #{key >= T} >= K (the K-th largest key), or any value with
  // #{key >= T} = K.  The bits that the smallest and the largest candidate key share are T's too.
  uint32_t kmin = 0xffffffffu, kmax = 0u;
#pragma unroll
  for (int v = 0; v < V; ++v) {
    if (32 * v + lane < C) kmin = min(kmin, key[v]);
    kmax = max(kmax, key[v]);
  }
  kmin = __reduce_min_sync(0xffffffffu, kmin);
  kmax = __reduce_max_sync(0xffffffffu, kmax);
  const int shared_bits = __clz(kmin ^ kmax);
  uint32_t T = shared_bits ? kmax & ~(0xffffffffu >> shared_bits) : 0u;
  if (shared_bits == 32) T = kmax;
#pragma unroll 1
  for (uint32_t bit = shared_bits == 32 ? 0u : 0x80000000u >> shared_bits; bit; bit >>= 1) {
    const uint32_t t = T | bit;
    int c[4] = {0, 0, 0, 0};
#pragma unroll
    for (int v = 0; v < V; ++v) c[v & 3] += key[v] >= t ? 1 : 0;
    const int n = __reduce_add_sync(0xffffffffu, (c[0] + c[1]) + (c[2] + c[3]));
    if (n >= K) T = t;
    if (n == K) break;
  }
  int above = 0;
#pragma unroll
  for (int v = 0; v < V; ++v) above += key[v] > T ? 1 : 0;
  int need = K - __reduce_add_sync(0xffffffffu, above);  // entries equal to T to take, in position order
  const uint32_t lt = (1u << lane) - 1u;
  int32_t* out = idx + ((size_t)i * Wn + w) * K;
  int base = 0;
#pragma unroll
  for (int v = 0; v < V; ++v) {
    const int q = 32 * v + lane;
    const uint32_t eq = __ballot_sync(0xffffffffu, key[v] == T && q < C);
    const bool sel = key[v] > T || (((eq >> lane) & 1u) && __popc(eq & lt) < need);
    need -= min(need, __popc(eq));
    const uint32_t m = __ballot_sync(0xffffffffu, sel);
    if (sel) out[base + __popc(m & lt)] = ci[q];
    base += __popc(m);
  }
}

// Training labels of the stage-1 candidates of one window, one thread per (target, candidate):
// y = 1 + log10(max(p_ij, floor)) / 12 with p_ij the dense posterior of candidate j for target i
// (row-major P [N][N]); 0 for padding (-1) and NaN for an id outside [0, N).
__global__ void label_kernel(const float* __restrict__ P, const int32_t* __restrict__ cand, int N, int C, float floor,
                             float* __restrict__ y) {
  const long long n = (long long)N * C;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x) {
    const int j = cand[e];
    float v = 0.0f;
    if (j >= N) v = __int_as_float(0x7fc00000);
    else if (j >= 0) v = 1.0f + log10f(fmaxf(P[(size_t)(e / C) * N + j], floor)) * (1.0f / 12.0f);
    y[e] = v;
  }
}

}  // namespace lsk
