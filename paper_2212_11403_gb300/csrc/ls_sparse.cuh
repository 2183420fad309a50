// ls_sparse.cuh -- the LS recursions restricted to proposed donor sets.
//
// For target i and window w (WS consecutive loci) the copying state ranges over a set S_i^w of at
// most K donors (ascending ids, -1 padding at the end).  The prior keeps its dense value
// pi = 1/(N-1): recombination mass that would go to donors outside the set is dropped, so donors
// in the set follow exactly the dense recursions (Eq. fwd1 / Eq. bck1) up to a common factor per
// target and locus.  A transition from locus l (window w) to l+1 (window w') continues only for
// donors in both sets:
//   forward:  alpha'_k = theta_k ((1-rho) a_k [k in S] + rho pi),  a = alpha / sum_{S} alpha,
//   backward: beta_j   = (1-rho) [j in S'] t_j / S + rho,  t = theta beta,  S = pi sum_{k in S'} t_k,
// so the backward is the adjoint of the forward and p ~ alpha beta over S_i^w is the posterior of
// the restricted chain.  The normalised forward mass on donors that leave the set at a window
// change is the in-set check: its maximum per target is reported ("lost"), and targets above a
// tolerance are recomputed densely by the caller.
//
// Outside pool (pool = 1): the donors outside the set are carried as one aggregate state o (their
// total forward mass, or their total t = theta beta backward) with the average emission of the
// outside donors at each locus (from the locus' allele count minus the set's own matches):
//   o <- theta_out (c o) + r sum_{j out} theta_j,   theta_out = sum_{j out} theta_j / |out|,
// and the normalisers become set sum + o, as in the dense chain.  At a window change the mass of
// donors leaving the set joins the pool and each entering donor takes the pool's average.  The
// posterior is the pooled chain's own: its normaliser adds the pool's forward mass times the mean
// backward value of the outside donors, and each outside donor receives an equal share of the
// pool's posterior mass (an estimate, reported apart from the set donors' values).
//
// One warp per target, slot s of lane q <-> set index 32 s + q (coalesced set loads and stores).  Loci
// run in blocks of 64.  At the start of a block (and at a window change) a lane loads the block's 64
// bits of each of its donors from the haplotype-major words (8 bytes of a 32-byte sector), XORs them
// with the target's and transposes them in registers to one word per locus and 32 slots, bit s = slot
// s differs from the target; the words wait in shared memory, and the outside donors' emissions at the
// block's loci are worked out a locus per lane.  A locus then needs its words, a packed FFMA2 and FADD2
// per pair of slots and one predicated multiply per slot, and its logarithm is taken with 31 others.
// Emissions are divided by b = max(1-mu, mu) throughout, f in {1, min(1-mu, mu)/b}: the factor cancels in
// every ratio of the chain, and the log-likelihood gets the sum of log b back at the end (multiplying
// it into c and r would round 1 - rho the same way at every locus).  Padding slots take the smaller
// factor; they start at 0 when their window starts and so hold one common value xs, which the row sum
// subtracts.  The per-locus constants of the next block are copied with cp.async while the current one runs.
//
// Bound by the dependent chain of a locus (row sum, division, multiply, add), so what counts is the warps that
// cover it: 128 registers and 12.8 KB a warp leave four a scheduler (bits are gathered and transposed 16 slots
// at a time for that).  N = 20003, L = 2000, K = 3 x 512: forward / backward 32.3 / 30.2 -> 14.5 / 14.7 ms
// (before: one word and one bit test, select and count per slot and locus, set ids in registers, two warps a
// scheduler; with three warps, transposing 32 slots at a time, 17.4 / 17.5).
//
// Short windows are bound by the window changes.  The lookups of eight slots run side by side in a fixed number of
// steps, only the part of a block that the window reaches is worked out, and variants of few slots take five or
// six CTAs per SM (72 to 96 registers): N = 10000, L = 1024, K = 256, windows of 4 / 16 / 64 / 256 loci 29.3 / 9.8 /
// 4.5 / 3.6 -> 14.3 / 5.2 / 3.2 / 3.0 ms with sets as they are (before the blocks of 64 loci 15.7 / 6.8 / 4.9 / 4.5),
// 92 / 23.8 / 8.7 / 5.6 -> 49 / 13.3 / 6.5 / 5.3 ms widened; the run of N = 20003 above 32.2 -> 29.3 ms in all.
#pragma once

#include <cstdint>
#include <type_traits>
#include <cuda_runtime.h>

namespace lsk {

constexpr int kSparseWarps = 4;   // targets per CTA (four to six CTAs per SM)
constexpr int kSparseChunk = 64;  // loci per block: two 32-bit haplotype-major words per donor
constexpr int kSparseScal = 4;    // per-locus constants staged per block: 1-rho, rho, n1, emission ratio

struct SparseParams {
  const uint32_t* hw;    // [ceil(L/256)][N][8] haplotype-major words: bit b of word k of (w, j) is
                         // haplotype j at locus 256 w + 32 k + b (0 beyond L)
  int N, L;
  int K;                 // set entries per target and window
  int WS;                // loci per window
  int Wn;                // windows, ceil(L / WS)
  const int32_t* idx;    // [N][Wn][K] donor ids, ascending, -1 padding at the end
  const float* omr;      // [L-1] 1 - rho
  const float* rho;      // [L-1] rho
  const float* ratio;    // [L] the smaller of 1 - mu and mu over the larger; negative where the larger is mu
  double log_base;       // sum over the loci of the logarithm of the larger
  int t_begin, t_count;
  int n_store;
  int store_loci[64];    // processing order
  int store_slot[64];
  float* store;          // [slots][N][K]: forward writes alpha, backward overwrites it with p
  double* logs;          // [N] forward: log-likelihood of the restricted chain (may be null)
  float* lost;           // [N] forward: max normalised mass on leaving donors (may be null)
  uint32_t* status;      // [N] status bits (may be null)
  const int32_t* n1;     // [L] haplotypes carrying allele 1 at each locus (outside pool only)
  int pool;              // 1: carry the donors outside the set as one pooled state (below)
  float* poolf;          // [slots][N] forward: the pool's mass at the store loci (pool = 1)
  float* share;          // [slots][N] backward: posterior of one outside donor (pool = 1)
  float* pout;           // [slots][N] backward: posterior mass of all outside donors (may be null)
};

// posterior products alpha * (beta * 2^100): exact scaling that cancels in the normalisation and
// keeps products of small alpha and beta above FP32's underflow
constexpr float kSparseProdScale = 0x1p100f;

// Words per lane and locus (bit s of word g: slot 32 g + s), the second one of 16 bits where a lane has 48
// slots; bytes per warp of a block's words [64][32 lanes] (32-bit), [64][32 lanes] (16-bit), whose place the
// copies of the old set (ids and values) take at a window change.
__host__ __device__ constexpr int sparse_groups(int ks) { return (ks + 31) / 32; }
__host__ __device__ constexpr int sparse_warp_bytes(int ks) {
  const int words = kSparseChunk * 128 + (ks > 32 ? kSparseChunk * 64 : 0);
  return words > 256 * ks ? words : 256 * ks;
}
constexpr int kSparsePool = 2 * kSparseChunk;  // floats per warp: the outside donors' summed and mean emission per locus
// two buffers of per-locus constants and the per-warp regions
__host__ __device__ constexpr int sparse_smem_bytes(int ks) {
  return 2 * kSparseScal * kSparseChunk * 4 + kSparseWarps * (kSparsePool * 4 + sparse_warp_bytes(ks));
}

__device__ __forceinline__ void cp_async4(void* dst, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait1() { asm volatile("cp.async.wait_group 1;" ::: "memory"); }

#ifndef LS_SPARSE_PARAMS_ONLY  // the kernels live in ls_sparse.cu only

// Two 16 x 16 bit transpositions at once: the low half of m[c] becomes the bits c of the low halves of all
// m[r], the high half those of the high halves
__device__ __forceinline__ void transpose16x2(uint32_t (&m)[16]) {
#pragma unroll
  for (int st = 0; st < 4; ++st) {
    const int j = 8 >> st;
    const uint32_t mask = st == 0 ? 0x00ff00ffu : st == 1 ? 0x0f0f0f0fu : st == 2 ? 0x33333333u : 0x55555555u;
#pragma unroll
    for (int k = 0; k < 16; ++k)
      if (!(k & j)) {
        const uint32_t lo = (m[k] & mask) | ((m[k + j] & mask) << j);
        const uint32_t hi = ((m[k] >> j) & mask) | (m[k + j] & ~mask);
        m[k] = lo;
        m[k + j] = hi;
      }
  }
}

template <int DIR, int KS>
__global__ void __launch_bounds__(kSparseWarps * 32, KS == 8 ? 6 : KS == 4 ? 5 : 4) ls_sparse_kernel(const __grid_constant__ SparseParams p) {
  static_assert(KS % 2 == 0, "slots come in pairs");
  constexpr float eps = 2.220446049250313e-16f;
  constexpr int INF_ID = 0x7fffffff;
  constexpr int CH = kSparseChunk, NG = sparse_groups(KS), NT = kSparseWarps * 32;
  extern __shared__ __align__(16) unsigned char smem[];
  float* scal = reinterpret_cast<float*>(smem);  // [2][kSparseScal][CH]
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  float* pool_e = scal + 2 * kSparseScal * CH + warp * kSparsePool;  // [64] sums, [64] means
  unsigned char* mine = smem + (2 * kSparseScal * CH + kSparseWarps * kSparsePool) * 4 + warp * sparse_warp_bytes(KS);
  uint32_t* words = reinterpret_cast<uint32_t*>(mine) + lane;                     // [locus] x 32 lanes
  uint16_t* words2 = reinterpret_cast<uint16_t*>(mine + kSparseChunk * 128) + lane;  // 48 slots: the last 16
  auto word_at = [&](int kr, int g) -> uint32_t { return g == 0 ? words[32 * kr] : (uint32_t)words2[32 * kr]; };
  int* sid = reinterpret_cast<int*>(mine);                     // window changes: the old set's ids and values
  float* sval = reinterpret_cast<float*>(mine) + 32 * KS;
  const int i_raw = p.t_begin + blockIdx.x * kSparseWarps + warp;
  const bool active = i_raw < p.t_begin + p.t_count;
  const int i = active ? i_raw : p.t_begin;  // idle warps shadow a valid target and write nothing
  const int K = p.K, L = p.L, N = p.N;
  const float pi = 1.0f / (float)(N - 1);  // dense uniform prior

  float2 x2[KS / 2];  // slots 2k and 2k + 1
  auto X = [&](int s) -> float& { return (s & 1) ? x2[s >> 1].y : x2[s >> 1].x; };
  float xs = 0.0f;
  int cur_w = -1;
  int n_enter = 0, nset = 0;  // set entries are indices 0 .. nset - 1
  uint32_t pad[NG];           // bit s: slot 32 g + s is padding
  auto warp_sum = [&](float v) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    return v;
  };
  auto set_entry = [&](int w, int s) -> int {
    const int q = 32 * s + lane;
    return q < K ? p.idx[((size_t)i * p.Wn + w) * K + q] : -1;
  };
  // the words of block b (loci 64 b .. 64 b + 63) for the current set, and the outside donors' emissions
  // (sc: the block's constants), where the window reaches: 32 loci at a time transposed, eight stored, the emissions
  // of each
  auto gather = [&](int b, const float* sc) {
    const int first = max(cur_w * p.WS - CH * b, 0), last = min(p.WS - (CH * b - cur_w * p.WS), CH);  // [first, last)
    __syncwarp();
    const uint32_t* hwb = p.hw + (size_t)(b >> 2) * N * 8 + 2 * (b & 3);
    const uint2 tw = *reinterpret_cast<const uint2*>(hwb + (size_t)i * 8);
#pragma unroll 1
    for (int g = 0; g < (KS + 15) / 16; ++g) {  // 16 slots at a time
      uint32_t lo[16], hi[16];
#pragma unroll
      for (int s = 0; s < 16; ++s) {
        lo[s] = hi[s] = 0u;
        if (s < KS) {
          const int id = set_entry(cur_w, 16 * g + s);
          uint2 v = make_uint2(~tw.x, ~tw.y);  // padding differs everywhere
          if (id >= 0) v = *reinterpret_cast<const uint2*>(hwb + (size_t)id * 8);
          lo[s] = v.x ^ tw.x;
          hi[s] = v.y ^ tw.y;
        }
      }
      // group g's 16 bits: halves of the 32-bit words, or the 16-bit words
      const int step = g < 2 ? 64 : 32;
      uint16_t* dst = g < 2 ? reinterpret_cast<uint16_t*>(words) + g : words2;
      auto put = [&](uint32_t (&m)[16], int k0) {
        transpose16x2(m);
#pragma unroll
        for (int q = 0; q < 32; q += 8) {  // eight loci at a time
          if (k0 + q + 8 <= first || k0 + q >= last) continue;
#pragma unroll
          for (int k = q; k < q + 8; ++k) {
            const uint32_t v = k < 16 ? m[k & 15] & 0xffffu : m[k & 15] >> 16;
            if (KS <= 16) words[32 * (k0 + k)] = v;
            else dst[(k0 + k) * step] = (uint16_t)v;
          }
        }
      };
      if (first < 32) put(lo, 0);
      if (last > 32) put(hi, 32);
    }
    if (p.pool) {
      const int nout = N - 1 - nset;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int k0 = max(first - 32 * h, 0), k1 = min(last - 32 * h, 32);
        if (k0 >= k1) continue;
        int mis = 0;  // slots (padding included) that differ from the target at locus 32 h + lane
#pragma unroll 8
        for (int k = k0; k < k1; ++k) {
          int n = 0;
#pragma unroll
          for (int g = 0; g < NG; ++g) n += __popc(word_at(32 * h + k, g));
          n = __reduce_add_sync(0xffffffffu, n);
          if (lane == k) mis = n;
        }
        const int kr = 32 * h + lane;
        const int n1 = __float_as_int(sc[2 * CH + kr]);
        const int mtot = (((h ? tw.y : tw.x) >> lane) & 1u ? n1 : N - n1) - 1;  // matching donors, the target excluded
        const int mout = min(max(mtot - (32 * KS - mis), 0), nout);
        const float q = sc[3 * CH + kr];
        const float thsum = signbit(q) ? -q * (float)mout + (float)(nout - mout) : (float)mout + q * (float)(nout - mout);
        pool_e[kr] = thsum;
        pool_e[CH + kr] = nout > 0 ? thsum / (float)nout : 0.0f;
      }
      __syncwarp();
    }
  };
  // exact sum of the set's values, in the order the window map sums them
  auto set_sum = [&]() -> float {
    float v = 0.0f;
#pragma unroll
    for (int s = 0; s < KS; ++s) v += 32 * s + lane < nset ? X(s) : 0.0f;
    return warp_sum(v);
  };
  // enter window w: map the values of the old set onto the new one (`fill` for new donors); returns
  // the mapped total, and the number of entering donors and of set entries
  auto enter = [&](int w, bool map, float fill) -> float {
    __syncwarp();
    if (map) {
#pragma unroll
      for (int s = 0; s < KS; ++s) {
        const int id = set_entry(cur_w, s);
        sid[32 * s + lane] = id >= 0 ? id : INF_ID;
        sval[32 * s + lane] = X(s);
      }
      __syncwarp();
    }
    float mapped = 0.0f;
    int ne = 0, nv = 0;
    constexpr int SB = KS < 8 ? KS : 8;  // slots looked up side by side
#pragma unroll
    for (int s0 = 0; s0 < KS; s0 += SB) {
      int id[SB], pos[SB];  // pos: entries of the old set below id (at most 32 KS - 1 counted)
#pragma unroll
      for (int q = 0; q < SB; ++q) {
        id[q] = set_entry(w, s0 + q);
        pos[q] = 0;
      }
      if (map) {
#pragma unroll 1
        for (int step = KS == 48 ? 1024 : 16 * KS; step > 0; step >>= 1)
#pragma unroll
          for (int q = 0; q < SB; ++q)
            if ((KS != 48 || pos[q] + step < 32 * KS) && sid[pos[q] + step - 1] < id[q]) pos[q] += step;
      }
#pragma unroll
      for (int q = 0; q < SB; ++q) {
        float v = 0.0f;
        if (map && id[q] >= 0) {
          if (sid[pos[q]] == id[q]) {
            v = sval[pos[q]];
            mapped += v;
          } else {
            v = fill;
            ++ne;
          }
        }
        nv += id[q] >= 0;
        X(s0 + q) = v;
      }
    }
    __syncwarp();
    cur_w = w;
    xs = 0.0f;  // every padding slot restarts at 0
    n_enter = __reduce_add_sync(0xffffffffu, ne);
    nset = __reduce_add_sync(0xffffffffu, nv);
#pragma unroll
    for (int g = 0; g < NG; ++g) {
      const int have = min(max((nset - lane + 31) / 32 - 32 * g, 0), 32);  // this lane's set entries in the group
      pad[g] = have == 32 ? 0u : 0xffffffffu << have;
    }
    return warp_sum(mapped);
  };

  double logacc = 0.0;
  float keep = 1.0f;      // lane k: the normaliser of the k-th locus since the last fold
  int nkeep = 0;
  uint32_t stb = 0u;
  // the kept normalisers: status bits, and (forward) their logarithms summed with an exact error term per
  // addition into the double accumulator
  auto fold = [&]() {
    if (keep < 1.17549435e-38f) stb |= 1u;      // LS_STATUS_UNDERFLOW
    if (!(keep <= 3.40282347e+38f)) stb |= 2u;  // LS_STATUS_OVERFLOW (infinite or NaN)
    if (DIR == 0) {
      float v = logf(keep), e = 0.0f;
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) {
        const float vo = __shfl_xor_sync(0xffffffffu, v, off), eo = __shfl_xor_sync(0xffffffffu, e, off);
        const float t = __fadd_rn(v, vo), bb = __fsub_rn(t, v);
        e = __fadd_rn(__fadd_rn(e, eo), __fadd_rn(__fsub_rn(v, __fsub_rn(t, bb)), __fsub_rn(vo, bb)));
        v = t;
      }
      logacc += (double)v + (double)e;
    }
    keep = 1.0f;
    nkeep = 0;
  };
  float lost_max = 0.0f;
  float sum_prev = 1.0f;  // forward: sum alpha; backward: sum t (set plus pool)
  float opool = 0.0f;     // outside pool (pool = 1)
  int store_next = 0;
  // blocks of CH loci aligned to multiples of CH, in processing order
  const int nb = (L + CH - 1) / CH;
  auto blk_of = [&](int t) { return DIR == 0 ? t : nb - 1 - t; };
  auto issue = [&](int t) {
    const int base = CH * blk_of(t), nrows = min(CH, L - base);
    for (int e = threadIdx.x; e < kSparseScal * CH; e += NT) {
      const int f = e / CH, k = e % CH, l = base + k;
      if (k >= nrows) continue;
      const int m = DIR == 0 ? l - 1 : l;  // interval entering locus l in processing order
      float* d = scal + ((t & 1) * kSparseScal + f) * CH + k;
      if (f == 0 && m >= 0 && m < L - 1) cp_async4(d, p.omr + m);
      else if (f == 1 && m >= 0 && m < L - 1) cp_async4(d, p.rho + m);
      else if (f == 2 && p.n1) cp_async4(d, p.n1 + l);
      else if (f == 3) cp_async4(d, p.ratio + l);
    }
  };
  issue(0);
  cp_async_commit();
  for (int t = 0; t < nb; ++t) {
    const int b = blk_of(t), base = CH * b, nrows = min(CH, L - base);
    __syncthreads();  // every warp is done with block t-1, whose buffer the next copies reuse
    if (t + 1 < nb) issue(t + 1);
    cp_async_commit();
    cp_async_wait1();  // this thread's copies of block t have landed
    __syncthreads();   // and everyone's
    const float* sc = scal + (t & 1) * kSparseScal * CH;
    bool need_gather = true;
    // One locus.  EV (compile-time) marks the event steps: the block's first (the words are
    // gathered), a window change and a store locus; the other steps run a copy without those
    // branches.
    auto body = [&](const int jj, auto evc) {
      constexpr bool EV = decltype(evc)::value;
      const int kr = DIR == 0 ? jj : nrows - 1 - jj;  // locus l = base + kr
      const int l = base + kr;
      float c, r;
      const int w = EV ? l / p.WS : cur_w;
      if (EV && cur_w < 0) {  // initial locus: alpha = theta pi ; t = theta (beta = 1)
        enter(w, false, 0.0f);
        need_gather = true;
        c = 0.0f;
        r = DIR == 0 ? pi : 1.0f;
      } else {
        if (EV && w != cur_w) {
          const float s_set = set_sum();
          const int nout_old = N - 1 - nset;
          const float fill = (p.pool && nout_old > 0) ? opool / (float)nout_old : 0.0f;
          const float mapped = enter(w, true, fill);
          if (DIR == 0 && s_set > 0.0f) lost_max = fmaxf(lost_max, 1.0f - mapped / s_set);
          if (p.pool) opool = fmaxf(opool + (s_set - mapped) - (float)n_enter * fill, 0.0f);
          need_gather = true;
        }
        const float om = sc[kr], rh = sc[CH + kr];  // interval entering locus l
        if (DIR == 0) {
          c = om / sum_prev;
          r = rh * pi;
        } else {
          // S = pi sum_{k in S'} t_k over the set of locus l+1 (the transition's target set)
          c = om / (pi * sum_prev);
          r = rh;
        }
      }
      if (EV && need_gather) {
        gather(b, sc);
        need_gather = false;
      }
      const bool is_store = EV && store_next < p.n_store && p.store_loci[store_next] == l;
      float* srow = is_store ? p.store + ((size_t)p.store_slot[store_next] * N + i) * K : nullptr;
      if (DIR == 1 && is_store) {
        // posterior: alpha (stored by the forward) times beta = c t + r over the set, plus (pool) the
        // pool's forward mass times the outside donors' mean backward value c (o / n_out) + r
        constexpr float S = kSparseProdScale;
        float zb = 0.0f;
#pragma unroll
        for (int q = 0; q < KS; ++q) {
          const int sq = 32 * q + lane;
          if (sq < nset) zb += srow[sq] * (fmaf(c, X(q), r) * S);
        }
        zb = warp_sum(zb);
        const int nout = N - 1 - nset;
        const size_t so = (size_t)p.store_slot[store_next] * N + i;
        const float zp = (p.pool && nout > 0) ? p.poolf[so] * (fmaf(c, opool / (float)nout, r) * S) : 0.0f;
        const float z = zb + zp;
        const float inv = z > 0.0f ? 1.0f / z : 0.0f;
#pragma unroll
        for (int q = 0; q < KS; ++q) {
          const int sq = 32 * q + lane;
          if (active && sq < K)
            srow[sq] = sq >= nset ? 0.0f : (z > 0.0f ? srow[sq] * (fmaf(c, X(q), r) * S) * inv : eps);
        }
        if (p.pool && active && lane == 0) p.share[so] = (nout > 0 && z > 0.0f) ? zp * inv / (float)nout : 0.0f;
        if (p.pout && active && lane == 0) p.pout[so] = z > 0.0f ? zp * inv : 0.0f;
      }
      const float qr = sc[3 * CH + kr], ur = fabsf(qr);
      const uint32_t flip = signbit(qr) ? 0xffffffffu : 0u;  // mu > 1/2: the matches carry the smaller factor
      const float2 C2 = make_float2(c, c), R2 = make_float2(r, r);
      float2 acc[4] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f), make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
#pragma unroll
      for (int g = 0; g < NG; ++g) {
        const uint32_t wd = word_at(kr, g);
        const uint32_t sm = (wd ^ flip) | pad[g];
#pragma unroll
        for (int s = 0; s < 32; s += 2) {
          const int k = (32 * g + s) >> 1;
          if (32 * g + s < KS) {
            float2 u = __ffma2_rn(C2, x2[k], R2);
            if ((sm >> s) & 1u) u.x = __fmul_rn(u.x, ur);
            if ((sm >> (s + 1)) & 1u) u.y = __fmul_rn(u.y, ur);
            x2[k] = u;
            acc[k & 3] = __fadd2_rn(acc[k & 3], u);
          }
        }
      }
      xs = __fmul_rn(__fmaf_rn(c, xs, r), ur);  // padding slots: always the smaller factor
      acc[0] = __fadd2_rn(__fadd2_rn(acc[0], acc[2]), __fadd2_rn(acc[1], acc[3]));
      float tot = warp_sum(acc[0].x + acc[0].y) - (float)(32 * KS - nset) * xs;
      if (p.pool) {
        opool = pool_e[CH + kr] * (c * opool) + r * pool_e[kr];
        tot += opool;
      }
      if (is_store) {
        if (DIR == 0) {
#pragma unroll
          for (int q = 0; q < KS; ++q) {
            const int sq = 32 * q + lane;
            if (active && sq < K) srow[sq] = sq < nset ? X(q) : 0.0f;
          }
          if (p.pool && active && lane == 0) p.poolf[(size_t)p.store_slot[store_next] * N + i] = opool;
        }
        ++store_next;
      }
      if (lane == nkeep) keep = tot;
      if (++nkeep == 32) fold();
      sum_prev = tot;
    };
    for (int jj = 0; jj < nrows;) {
      body(jj++, std::true_type{});
      // the next event in this block: a window change (the first step whose locus lies outside the
      // current window) or a store locus
      int ev = nrows;
      const int wlo = cur_w * p.WS, whi = wlo + p.WS;  // the current window's loci [wlo, whi)
      const int lb = DIR == 0 ? whi : wlo - 1;         // the first locus beyond it, in processing order
      if (lb >= base && lb < base + nrows) ev = min(ev, DIR == 0 ? lb - base : nrows - 1 - (lb - base));
      if (store_next < p.n_store) {
        const int ks = p.store_loci[store_next] - base;
        if (ks >= 0 && ks < nrows) ev = min(ev, DIR == 0 ? ks : nrows - 1 - ks);
      }
      for (; jj < ev; ++jj) body(jj, std::false_type{});
    }
  }
  fold();
  stb = __reduce_or_sync(0xffffffffu, stb);
  if (active && lane == 0) {
    if (DIR == 0 && p.logs) p.logs[i] = logacc + p.log_base;
    if (DIR == 0 && p.lost) p.lost[i] = lost_max;
    if (p.status && stb) atomicOr(p.status + i, stb);
  }
}

// SparseParams::ratio
__global__ void emission_kernel(const float* __restrict__ thm, const float* __restrict__ thx, int L, float* __restrict__ ratio) {
  const int l = blockIdx.x * blockDim.x + threadIdx.x;
  if (l >= L) return;
  const float a = thm[l], b = thx[l];
  ratio[l] = a < b ? -__fdiv_rn(a, b) : __fdiv_rn(b, a);  // 1 - mu and mu: the larger is at least 1/2
}

// Half distances -log(max(p, eps))/2 of the sparse posteriors into dense [D][N][N] rows.  Every
// entry of row i is first set to the outside donors' estimate: the half distance of the pool's
// share (share != null), stored NEGATED so that it stays distinguishable (its sign bit, -0.0
// included), or NaN without a pool; then the set's donors get their own half distances (>= 0).
// grid (N, D), 256 threads.
__global__ void sparse_hdist_kernel(const float* __restrict__ P, const int32_t* __restrict__ idx, int N, int K, int Wn,
                                    const int* __restrict__ win_of_slot, const float* __restrict__ share,
                                    float* __restrict__ h) {
  constexpr float eps = 2.220446049250313e-16f;
  const int i = blockIdx.x, k = blockIdx.y;
  const int w = win_of_slot[k];
  const int32_t* ids = idx + ((size_t)i * Wn + w) * K;
  const float* pr = P + ((size_t)k * N + i) * K;
  float* hr = h + ((size_t)k * N + i) * N;
  // -log(p)/2 >= 0 for p <= 1: computed as |log(p)/2| so that p = 1 gives +0.0 (chain values keep
  // the sign bit clear); estimates are stored as -|log(share)/2| (sign bit set, -0.0 included)
  const float est =
      share ? -fabsf(0.5f * logf(fminf(fmaxf(share[(size_t)k * N + i], eps), 1.0f))) : __int_as_float(0xffffffff);
  for (int j = threadIdx.x; j < N; j += blockDim.x) hr[j] = j == i ? 0.0f : est;
  __syncthreads();
  for (int q = threadIdx.x; q < K; q += blockDim.x) {
    const int j = ids[q];
    if (j >= 0 && j < N && j != i) hr[j] = fabsf(0.5f * logf(fminf(fmaxf(pr[q], eps), 1.0f)));
  }
}

// d = |h| + |h^T| in place over D stacked N x N matrices of half distances, with trust bits:
// bit j of word j/32 of mask row i (mask [D][N][wpr], wpr = ceil(N/32)) is 1 where both halves are
// chain values (sign bit clear) and either both targets have dense rows (dense_row[i] and
// dense_row[j]) or d_ij <= d_trust.  A NaN half (no pool) leaves d NaN and the bit 0.  Tiles as in
// symmetrize_kernel; a warp holds 32 consecutive columns of one row, so one ballot gives a word.
// A warp takes a row of 32 columns at a time and eight rows of both tiles, whose 16 loads go out ahead of
// the first use; the dense flags of the tiles' rows are read once (N = 20003, two matrices: 3.26 -> 1.90
// ms, 3.4 TB/s).
__global__ void __launch_bounds__(128) symmetrize_trust_kernel(float* __restrict__ d, int N, const uint8_t* __restrict__ dense_row,
                                                               float d_trust, uint32_t* __restrict__ mask, int wpr) {
  const int bx = blockIdx.x, by = blockIdx.y;
  if (bx > by) return;
  float* m = d + (size_t)blockIdx.z * N * N;
  uint32_t* mk = mask ? mask + (size_t)blockIdx.z * N * wpr : nullptr;
  __shared__ float A[32][33], B[32][33];
  const int tx = threadIdx.x, ty = threadIdx.y;  // 32 x 4
  const int ca = by * 32 + tx, cb = bx * 32 + tx;  // this lane's column in tile (bx, by) and in (by, bx)
  float va[8], vb[8];
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const int k = ty + 4 * q, ra = bx * 32 + k, rb = by * 32 + k;
    va[q] = (ra < N && ca < N) ? m[(size_t)ra * N + ca] : 0.0f;
    vb[q] = (rb < N && cb < N) ? m[(size_t)rb * N + cb] : 0.0f;
  }
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    A[ty + 4 * q][tx] = va[q];
    B[ty + 4 * q][tx] = vb[q];
  }
  // bit k: row (= column) 32 bx + k, respectively 32 by + k, has a dense row
  const uint32_t dx = __ballot_sync(0xffffffffu, cb < N && dense_row[cb]), dy = __ballot_sync(0xffffffffu, ca < N && dense_row[ca]);
  __syncthreads();
  auto one = [&](int row, int col, float a, float b, bool dense) {
    const bool in = row < N && col < N;
    const float v = row == col ? 0.0f : fabsf(a) + fabsf(b);
    const bool chain = !signbit(a) && !signbit(b) && v == v;
    if (in) m[(size_t)row * N + col] = v;
    const uint32_t word = __ballot_sync(0xffffffffu, in && row != col && chain && (dense || v <= d_trust));
    if (mk && tx == 0 && row < N) mk[(size_t)row * wpr + (col >> 5)] = word;
  };
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const int k = ty + 4 * q;
    one(bx * 32 + k, ca, va[q], B[tx][k], (dx >> k) & (dy >> tx) & 1u);
    if (bx != by) one(by * 32 + k, cb, vb[q], A[tx][k], (dy >> k) & (dx >> tx) & 1u);
  }
}

// Dense fallback rows: products alpha^l t^l (t = theta beta, the dense backward's decode product)
// of nf listed targets ([D][nf][N]) divided by theta^l (the locus' alleles from the packed rows,
// decode locus of slot k in dloci[k]) and normalised into half distances of rows tlist[r] of h
// ([D][N][N]).  grid (nf, D), 256 threads.
__global__ void dense_rows_hdist_kernel(const float* __restrict__ prod, int nf, int N, const int* __restrict__ tlist,
                                        const uint32_t* __restrict__ bits, int row_words, const float* __restrict__ thm,
                                        const float* __restrict__ thx, const int* __restrict__ dloci,
                                        float* __restrict__ h) {
  constexpr float eps = 2.220446049250313e-16f;
  const int r = blockIdx.x, k = blockIdx.y;
  const int i = tlist[r];
  const int l = dloci[k];
  const uint32_t* row = bits + (size_t)l * row_words;
  const uint32_t ai = (row[i >> 5] >> (i & 31)) & 1u;
  const float im = thm[l] > 0.0f ? 1.0f / thm[l] : 0.0f, ix = thx[l] > 0.0f ? 1.0f / thx[l] : 0.0f;
  const float* a0 = prod + ((size_t)k * nf + r) * N;
  auto a = [&](int j) { return a0[j] * ((((row[j >> 5] >> (j & 31)) & 1u) == ai) ? im : ix); };
  float s = 0.0f;
  for (int j = threadIdx.x; j < N; j += blockDim.x)
    if (j != i) s += a(j);
  __shared__ float red[32];
  for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x < 32) {
    float v = threadIdx.x < (blockDim.x >> 5) ? red[threadIdx.x] : 0.0f;
    for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    if (threadIdx.x == 0) red[0] = v;
  }
  __syncthreads();
  const float Z = red[0];
  const float invZ = Z > 0.0f ? 1.0f / Z : 0.0f;
  float* o = h + ((size_t)k * N + i) * N;
  for (int j = threadIdx.x; j < N; j += blockDim.x) {
    const float q = Z > 0.0f ? a(j) * invZ : eps;
    o[j] = j == i ? 0.0f : fabsf(0.5f * logf(fminf(fmaxf(q, eps), 1.0f)));  // +0.0 at q = 1 (a chain value)
  }
}

// Widened sets: U^w = S^w u S^{w+1} (span 1) or S^{w-1} u S^w u S^{w+1} (span 2), missing windows
// empty.  A donor proposed for window w+1 is already carried through window w, so it enters with
// a window of history; with span 2 a donor proposed for window w also stays through w+1, so the
// forward mass of donors about to mismatch decays inside the chain instead of being cut at the
// window change.  U has (span + 1) K entries, ascending, -1 padded.  One warp per (target, window) with a
// bitmap of the donors in shared memory: the lists' bits are set, and the words are read off 32 at a
// time, each lane writing its word's donors behind those of the lanes before it.  N = 20003, 8 windows,
// K = 512: 3.45 -> 0.40 ms (before, one thread merged the lists; a merge by binary searches in shared
// memory took 4.8 ms).
__global__ void lookahead_sets_kernel(const int32_t* __restrict__ idx, int N, int Wn, int K, int span, int32_t* __restrict__ U) {
  extern __shared__ uint32_t look_smem[];  // per warp: the bitmap, ceil(N / 32) words
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = (N + 31) / 32;
  const long long t = (long long)blockIdx.x * (blockDim.x >> 5) + warp;
  if (t >= (long long)N * Wn) return;
  uint32_t* map = look_smem + warp * nw;
  const int w = (int)(t % Wn);
  for (int q = lane; q < nw; q += 32) map[q] = 0u;
  __syncwarp();
  for (int v = span >= 2 ? -1 : 0; v <= 1; ++v) {
    if (w + v < 0 || w + v >= Wn) continue;
    const int32_t* list = idx + (t + v) * K;
    for (int q = lane; q < K; q += 32) {
      const int j = list[q];
      if (j >= 0 && j < N) atomicOr(map + (j >> 5), 1u << (j & 31));
    }
  }
  __syncwarp();
  const int width = (span + 1) * K;
  int32_t* u = U + t * width;
  int base = 0;
  for (int q0 = 0; q0 < nw; q0 += 32) {
    uint32_t m = q0 + lane < nw ? map[q0 + lane] : 0u;
    const int n = __popc(m);
    int pre = n;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, pre, off);
      if (lane >= off) pre += y;
    }
    int pos = base + pre - n;
    for (; m; m &= m - 1u) u[pos++] = 32 * (q0 + lane) + __ffs(m) - 1;
    base += __shfl_sync(0xffffffffu, pre, 31);
  }
  for (int q = base + lane; q < width; q += 32) u[q] = -1;
}

// Haplotypes carrying allele 1 at each locus: one warp per row, popcount of the first N bits.
__global__ void row_ones_kernel(const uint32_t* __restrict__ bits, int row_words, int N, int L, int32_t* __restrict__ n1) {
  const long long wid = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (wid >= L) return;
  const uint32_t* r = bits + (size_t)wid * row_words;
  int c = 0;
  for (int k = lane; 32 * k < N; k += 32) {
    uint32_t v = r[k];
    const int rem = N - 32 * k;
    if (rem < 32) v &= (1u << rem) - 1u;
    c += __popc(v);
  }
  c = __reduce_add_sync(0xffffffffu, c);
  if (lane == 0) n1[wid] = c;
}

#endif  // LS_SPARSE_PARAMS_ONLY

}  // namespace lsk
