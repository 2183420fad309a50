// ls_row.cuh -- kernels that take one table row per CTA and hold it in registers: single steps of a
// table, and posteriors / half distances of a row.
//
// Both are bound by memory: a row is read once, stays in registers across its reductions and is
// written once, in quads on 16-byte boundaries: thread t of nt holds E4 quads, t, t + nt, ..  Rows that do
// not start on a boundary (SHIFT: N not a multiple of four) begin with the quad that holds their first
// element; the parts of the first and last quad outside the row are left alone, and a quad's bits are
// funnel-shifted out of two words.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

#include "ls_aux.cuh"

namespace lsk {

constexpr int kRowMaxThreads = 512;
constexpr int kRowMaxN = 40 * kRowMaxThreads - 3;  // single steps (E4 = 10); three elements for the shift
constexpr int kRowMidPostN = 20 * kRowMaxThreads - 3;  // posteriors of 20 elements a thread (E4 = 5)
constexpr int kRowMaxPostN = 64 * kRowMaxThreads - 3;  // posteriors (E4 = 16)

// sum over the CTA, the same value in every thread; buf holds 32 floats and alternates between calls
__device__ __forceinline__ float row_sum(float v, float* buf) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
  if (nw == 1) return v;
  if (lane == 0) buf[warp] = v;
  __syncthreads();
  v = lane < nw ? buf[lane] : 0.0f;
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
  return v;
}

// The quads of a row: `at(e)` is the position of the first element of this thread's e-th quad
template <bool SHIFT>
struct RowQuads {
  int N, mis;  // mis: elements between the boundary before the row and the row
  __device__ RowQuads(int n, const float* row) : N(n), mis(SHIFT ? (int)((reinterpret_cast<uintptr_t>(row) >> 2) & 3) : 0) {}
  __device__ int at(int e) const { return 4 * ((int)threadIdx.x + e * (int)blockDim.x) - mis; }
  __device__ bool in(int pos) const { return !SHIFT || (unsigned)pos < (unsigned)N; }  // element of a quad with at(e) < N
  __device__ bool whole(int pos) const { return !SHIFT || (pos >= 0 && pos + 4 <= N); }
  __device__ void load(const float* row, int pos, float (&v)[4]) const {
    if (whole(pos)) {
      const float4 q = __ldcs(reinterpret_cast<const float4*>(row + pos));
      v[0] = q.x, v[1] = q.y, v[2] = q.z, v[3] = q.w;
      return;
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) v[k] = in(pos + k) ? __ldcs(row + pos + k) : 0.0f;
  }
  __device__ void store(float* row, int pos, const float (&v)[4]) const {
    if (whole(pos)) {
      __stcs(reinterpret_cast<float4*>(row + pos), make_float4(v[0], v[1], v[2], v[3]));
      return;
    }
#pragma unroll
    for (int k = 0; k < 4; ++k)
      if (in(pos + k)) __stcs(row + pos + k, v[k]);
  }
  // bit k: element pos + k of a packed row (which ends in at least one spare word)
  __device__ uint32_t bits(const uint32_t* b, int pos) const {
    if (!SHIFT) return b[pos >> 5] >> (pos & 31);
    if (pos < 0) return b[0] << -pos;
    return funnel(b[pos >> 5], b[(pos >> 5) + 1], (uint32_t)(pos & 31));
  }
};

// A few steps of a table (uniform prior; PropParams as for ls_prop_kernel, without alpha_dec and
// tlist), one target per CTA.  The register-tile kernel loads and saves its tile through shared memory
// element by element; a table moved by one locus is all load and save, so this kernel takes calls of
// few steps.  N = 10000, one locus forward / backward: 658 / 520 -> 158 / 186 us (0.8 GB moved, 75 / 63 % of
// the measured copy rate); the two reductions between load and save are what keeps it from the rest.
template <int DIR, int E4, bool SHIFT>
__global__ void __launch_bounds__(kRowMaxThreads) row_steps_kernel(const PropParams p) {
  __shared__ float buf[2][32];
  const int N = p.N, i = p.t_begin + blockIdx.x, row = i - p.tab_t0;
  float* state = p.state + (size_t)row * N;
  const RowQuads<SHIFT> P(N, state);
  float x[E4][4];
  int ph = 0;
  // forty elements of a thread are summed in four parts: in one, the additions round the same way in every thread of an
  // even row (N = 10000, four single steps: relative error of alpha 1.8e-7 against 9.6e-8 of the register-tile kernel;
  // now 6.9e-8).  Up to twenty, one sum is no further off than that kernel's (N = 2100 to 5117: 1.1e-7 against 1.3e-7)
  constexpr int PARTS = E4 <= 5 ? 1 : 4;
  auto total = [&](const float (&s)[PARTS]) {
    ph ^= 1;
    if constexpr (PARTS == 4) return row_sum((s[0] + s[1]) + (s[2] + s[3]), buf[ph]);
    else return row_sum(s[0], buf[ph]);
  };
  float sig_prev = 1.0f;
  {
    float s[PARTS] = {};
#pragma unroll
    for (int e = 0; e < E4; ++e) {
      const int pos = P.at(e);
#pragma unroll
      for (int k = 0; k < 4; ++k) x[e][k] = 0.0f;
      if (p.load_state && pos < N) P.load(state, pos, x[e]);
#pragma unroll
      for (int k = 0; k < 4; ++k) s[k % PARTS] += x[e][k];
    }
    if (p.load_state && DIR == 0) sig_prev = total(s);
  }
  double lg = 0.0;
  uint32_t sts = 0u;
  int store_next = 0;
  for (int step = 0; step < p.n_steps; ++step) {
    const int l = DIR == 0 ? p.l_first + step : p.l_first - step;
    const bool last = step + 1 == p.n_steps;
    float c, r, sg = 1.0f;
    if (step == 0 && p.init) {
      c = 0.0f;
      r = DIR == 0 ? p.pi_u : 1.0f;  // alpha^0 = theta pi ; beta^{L-1} = 1
    } else if (step == 0 && DIR == 1) {
      c = 1.0f;  // backward resume: x = theta^l beta^l from the stored beta
      r = 0.0f;
    } else {
      const int m = DIR == 0 ? l - 1 : l;
      c = __fdividef(p.omr[m], sig_prev);
      r = p.rr[m];
      sg = sig_prev;
    }
    const bool store_here = store_next < p.n_store && p.store_loci[store_next] == l;
    float* out = store_here ? p.store + ((size_t)p.store_slot[store_next] * p.state_rows + row) * N : nullptr;
    store_next += store_here ? 1 : 0;
    const uint32_t* bits = p.bits2 + (size_t)l * p.rw2;
    const uint32_t inv = (bits[i >> 5] >> (i & 31)) & 1u ? 0u : 0xffffffffu;  // match = bit ^ inv
    const float tm = p.thm[l], tx = p.thx[l];
    float s[PARTS] = {};
#pragma unroll
    for (int e = 0; e < E4; ++e) {
      const int pos = P.at(e);
      if (pos < N) {
        const uint32_t w = P.bits(bits, pos) ^ inv;
        float b[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          b[k] = pos + k == i || !P.in(pos + k) ? 0.0f : fmaf(c, x[e][k], r);  // alpha before its emission, or beta
          x[e][k] = ((w >> k) & 1u ? tm : tx) * b[k];
          s[k % PARTS] += x[e][k];
        }
        const float(&v)[4] = DIR == 0 ? x[e] : b;
        if (out && SHIFT) {  // a stored row need not lie on the boundaries of the table's
#pragma unroll
          for (int k = 0; k < 4; ++k)
            if (P.in(pos + k)) out[pos + k] = v[k];
        } else if (out) {
          P.store(out, pos, v);
        }
        if (last && p.save_state) P.store(state, pos, v);
      }
    }
    if (DIR == 0 || !last) {
      const float sig = total(s) * (DIR == 0 ? 1.0f : p.pi_u);
      if (DIR == 0) sg = sig;
      sig_prev = sig;
    }
    if (sg < 1.17549435e-38f) sts |= 1u;      // LS_STATUS_UNDERFLOW
    if (!(sg <= 3.40282347e+38f)) sts |= 2u;  // LS_STATUS_OVERFLOW
    lg += (double)logf(sg);
  }
  if (threadIdx.x == 0) {
    if (p.logs) p.logs[row] = (p.init ? 0.0 : p.logs[row]) + lg;
    if (p.status && sts) atomicOr(p.status + row, sts);
  }
}

// Eq. postprob of one row per CTA, the row's products held in registers between their sum and their use.
// DEC = 0: products alpha (beta 2^100) of caller-held rows (target t0 + r), written as p (mode 0) or as
// half distances -log(max(p, eps))/2 (mode 1).  DEC = 1: the products alpha t 2^100 that the backward
// pass left in out at D decode loci ([D][N][N], row i = recipient i), t = theta beta, are divided by their
// emission theta^l (1 - mu where the donor carries the target's allele at l, mu elsewhere; a zero theta
// means alpha = 0 too, and the entry is 0) and replaced by half distances.  A zero normaliser gives p =
// eps for every donor (Sec. 2.2); the target's own entry is 0.  Bound by memory (posteriors at N = 10000: 204 us,
// 5.9 TB/s; before, with the rows read twice, 442 us) and, with distances, by the logarithms too.
struct PostArgs {
  const float *alpha, *beta;  // DEC 0; DEC 1: null and, where out holds alpha alone, the backward's t 2^100
  float* out;
  int N, t0, mode;
  const uint32_t* bits;       // DEC 1: packed rows
  int row_words;
  const float *thm, *thx;
  DecodeLoci dl;
};

template <int DEC, int E4, bool SHIFT>
__global__ void __launch_bounds__(kRowMaxThreads) row_posterior_kernel(const __grid_constant__ PostArgs a) {
  constexpr float eps = 2.220446049250313e-16f;
  __shared__ float buf[32];
  const int N = a.N, r = blockIdx.x, i = DEC ? r : a.t0 + r;
  float* o = a.out + ((size_t)(DEC ? blockIdx.y : 0) * (DEC ? N : 0) + r) * N;
  const RowQuads<SHIFT> P(N, o);
  const uint32_t* bits = nullptr;
  uint32_t inv = 0u;
  float im = 0.0f, ix = 0.0f;
  if (DEC) {
    const int l = a.dl.l[blockIdx.y];
    bits = a.bits + (size_t)l * a.row_words;
    inv = (bits[i >> 5] >> (i & 31)) & 1u ? 0u : 0xffffffffu;
    im = a.thm[l] > 0.0f ? 1.0f / a.thm[l] : 0.0f;
    ix = a.thx[l] > 0.0f ? 1.0f / a.thx[l] : 0.0f;
  }
  float q[E4][4];
  float s = 0.0f;
#pragma unroll
  for (int e = 0; e < E4; ++e) {
    const int pos = P.at(e);
#pragma unroll
    for (int k = 0; k < 4; ++k) q[e][k] = 0.0f;
    if (pos < N) {
      if (DEC) {
        P.load(o, pos, q[e]);
        if (a.beta) {
          float t[4];
          P.load(a.beta + (o - a.out), pos, t);
#pragma unroll
          for (int k = 0; k < 4; ++k) q[e][k] *= t[k];
        }
        const uint32_t w = P.bits(bits, pos) ^ inv;
#pragma unroll
        for (int k = 0; k < 4; ++k) q[e][k] *= (w >> k) & 1u ? im : ix;
      } else {
        float b[4];
        P.load(a.alpha + (size_t)r * N, pos, q[e]);
        P.load(a.beta + (size_t)r * N, pos, b);
#pragma unroll
        for (int k = 0; k < 4; ++k) q[e][k] *= b[k] * kProdScale;
      }
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        if (pos + k == i || !P.in(pos + k)) q[e][k] = 0.0f;
        s += q[e][k];
      }
    }
  }
  const float Z = row_sum(s, buf);
  const float invZ = Z > 0.0f ? 1.0f / Z : 0.0f;
#pragma unroll
  for (int e = 0; e < E4; ++e) {
    const int pos = P.at(e);
    if (pos < N) {
      float v[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const float p = Z > 0.0f ? q[e][k] * invZ : eps;
        v[k] = pos + k == i ? 0.0f : (DEC || a.mode == 1 ? -0.5f * logf(fmaxf(p, eps)) : p);
      }
      P.store(o, pos, v);
    }
  }
}

}  // namespace lsk
