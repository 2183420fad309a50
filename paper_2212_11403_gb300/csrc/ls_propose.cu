// ls_propose.cu -- C ABI of the learned donor proposal: window features, the MLP (training and
// BF16 inference) and the proposal of per-window donor sets for ls_sparse_run_all.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "ls.h"
#include "ls_internal.h"
#include "ls_mlp.cuh"
#include "ls_propose.cuh"
#include "ls_mlp_tc.cuh"

struct ls_mlp {
  int device = 0;
  float* p = nullptr;       // [kMlpParams] FP32 master weights
  float* g = nullptr;       // gradient
  float* m = nullptr;       // Adam moments
  float* v = nullptr;
  long long t = 0;          // Adam step count
  __nv_bfloat16* w1t = nullptr;  // [256][16]
  __nv_bfloat16* w2t = nullptr;  // [256][256]
  std::vector<float> vec;        // host copy of b1, b2, w3, b3 (parameters of the scorer kernel)
  int* err = nullptr;            // device word: a scorer wait ran out of time
};

namespace {

template <class... A>
int fail(int code, const char* fmt, A... a) {
  return ls_fail(code, fmt, a...);
}
int dev_alloc(void*, void** p, size_t n) { return ls_dev_alloc(p, n); }

#define TRY(x)                                                                                 \
  do {                                                                                         \
    cudaError_t e_ = (x);                                                                      \
    if (e_ != cudaSuccess) return fail(LS_ERR_CUDA, "%s: %s", #x, cudaGetErrorString(e_));     \
  } while (0)

// BF16 transposed copies for the MMA kernel
__global__ void mlp_refresh_kernel(const float* __restrict__ p, __nv_bfloat16* __restrict__ w1t,
                                   __nv_bfloat16* __restrict__ w2t) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e < 256 * 256) {
    const int n = e >> 8, k = e & 255;
    w2t[e] = __float2bfloat16_rn(p[lsk::kOffW2 + k * 256 + n]);
  }
  if (e < 256 * lsk::kFeat) {
    const int n = e >> 4, k = e & 15;
    w1t[e] = __float2bfloat16_rn(k < lsk::kMlpIn ? p[lsk::kOffW1 + k * 256 + n] : 0.0f);
  }
}

int refresh(ls_mlp* m) {
  mlp_refresh_kernel<<<256, 256>>>(m->p, m->w1t, m->w2t);
  TRY(cudaGetLastError());
  m->vec.resize(3 * 256 + 1);
  TRY(cudaMemcpy(m->vec.data(), m->p + lsk::kOffB1, sizeof(float) * 256, cudaMemcpyDeviceToHost));
  TRY(cudaMemcpy(m->vec.data() + 256, m->p + lsk::kOffB2, sizeof(float) * 513, cudaMemcpyDeviceToHost));
  return LS_OK;
}

// Scores of n feature rows (8 BF16 values, or 8 floats, each) on the tensor cores (persistent CTAs, one
// per SM).
template <class T>
int launch_scores(const ls_mlp* m, const T* X, long long n, float* scores, int nsm, cudaStream_t s) {
  TRY(cudaFuncSetAttribute(lsk::mlp_score_tc_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, lsk::kTcSmem));
  lsk::MlpTcDev d;
  memcpy(d.b1, m->vec.data(), sizeof d.b1);
  memcpy(d.b2, m->vec.data() + 256, sizeof d.b2);
  memcpy(d.w3, m->vec.data() + 512, sizeof d.w3);
  d.b3 = m->vec[768];
  d.w1t = m->w1t;
  d.w2t = m->w2t;
  d.err = m->err;
  const long long tiles = (n + lsk::kTcRows - 1) / lsk::kTcRows;
  const int grid = (int)std::min<long long>(nsm, tiles);
  lsk::mlp_score_tc_kernel<T><<<grid, lsk::kTcThreads, lsk::kTcSmem, s>>>(d, X, n, scores);
  TRY(cudaGetLastError());
  return LS_OK;
}

// the error word of the scorer: LS_ERR_DEVICE (and cleared) when a wait ran out of time
int scorer_status(const ls_mlp* m, cudaStream_t s) {
  int h = 0;
  TRY(cudaMemcpyAsync(&h, m->err, sizeof(int), cudaMemcpyDeviceToHost, s));
  TRY(cudaStreamSynchronize(s));
  if (h) {
    cudaMemsetAsync(m->err, 0, sizeof(int), s);
    return fail(LS_ERR_DEVICE, "a wait of the tensor-core scorer ran out of time");
  }
  return LS_OK;
}

uint64_t splitmix(uint64_t& s) {
  uint64_t z = (s += 0x9e3779b97f4a7c15ull);
  z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
  z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
  return z ^ (z >> 31);
}

unsigned blocks(long long n, int t = 256) { return (unsigned)((n + t - 1) / t); }

// Scratch of the gradient of up to B rows and its launches.
struct GradWork {
  int ctas = 0, splits = 0, split_rows = 0, rw = 8;  // rw: rows per warp of mlp_rows_kernel
  float *H1, *dZ2, *part, *partw, *w2t;
  double *partd, *loss;
  int setup(const ls_mlp* m, CallScratch& b, int B, int nloss, cudaStream_t s) {
    int nsm = 0, rc;
    TRY(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, m->device));
    // two CTAs per SM; the tile with the fewest rows in the fullest one
    long long best = -1;
    for (int w : {8, 7, 6, 4, 2}) {
      const long long tiles = (B + 8ll * w - 1) / (8 * w), rows = (tiles + 2 * nsm - 1) / (2 * nsm) * w;
      if (best >= 0 && rows >= best) continue;
      best = rows;
      rw = w;
      ctas = (int)std::min<long long>(2 * nsm, tiles);
    }
    TRY(rows_kernel([](auto k) { return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, lsk::kTrSmem); }));
    // four quarter tiles of dW2 per split, two CTAs per SM, at least 128 rows a split
    const int most = std::max(1, 2 * nsm / 4);
    split_rows = std::max(128, (int)((B + (long long)most - 1) / most));
    split_rows = (split_rows + lsk::kTrK - 1) / lsk::kTrK * lsk::kTrK;
    splits = (int)((B + (long long)split_rows - 1) / split_rows);
    if ((rc = b.get(&H1, (size_t)B * 256)) || (rc = b.get(&dZ2, (size_t)B * 256)) ||
        (rc = b.get(&part, (size_t)ctas * lsk::kTrPart)) || (rc = b.get(&partw, (size_t)splits * 65536)) ||
        (rc = b.get(&w2t, 65536)) || (rc = b.get(&partd, 2 * (size_t)ctas)) || (rc = b.get(&loss, nloss)))
      return rc;
    lsk::mlp_transpose_kernel<<<dim3(8, 8), dim3(32, 8), 0, s>>>(m->p + lsk::kOffW2, w2t);
    TRY(cudaGetLastError());
    return LS_OK;
  }
  // f applied to the rows kernel of rw rows a warp
  template <class F>
  cudaError_t rows_kernel(F f) const {
    switch (rw) {
      case 2: return f(lsk::mlp_rows_kernel<2>);
      case 4: return f(lsk::mlp_rows_kernel<4>);
      case 6: return f(lsk::mlp_rows_kernel<6>);
      case 7: return f(lsk::mlp_rows_kernel<7>);
      default: return f(lsk::mlp_rows_kernel<8>);
    }
  }
  // gradient of the batch (its rows and source in mb), then into u.g or, with u.g null, an Adam update
  int run(const ls_mlp* m, lsk::MlpBatch mb, lsk::MlpUpdate u, cudaStream_t s) const {
    mb.p = m->p;
    mb.w2t = w2t;
    mb.H1 = H1;
    mb.dZ2 = dZ2;
    mb.part = part;
    mb.partd = partd;
    TRY(rows_kernel([&](auto k) {
      k<<<ctas, lsk::kTrThreads, lsk::kTrSmem, s>>>(mb);
      return cudaGetLastError();
    }));
    lsk::mlp_dw2_kernel<<<dim3(4, splits), 256, lsk::kDwSmem, s>>>(H1, dZ2, mb.B, split_rows, partw);
    u.partw = partw;
    u.splits = splits;
    u.part = part;
    u.partd = partd;
    u.ctas = ctas;
    u.w2t = w2t;
    lsk::mlp_update_kernel<<<lsk::kUpdBlocks, 256, 0, s>>>(u);
    TRY(cudaGetLastError());
    return LS_OK;
  }
};

}  // namespace

extern "C" {

int ls_mlp_create(const float* params, uint64_t seed, ls_mlp** out) {
  if (!out) return fail(LS_ERR_ARG, "null output");
  ls_mlp* m = new ls_mlp;
  cudaGetDevice(&m->device);
  const size_t P = lsk::kMlpParams;
  int rc;
  if ((rc = dev_alloc(nullptr, (void**)&m->p, sizeof(float) * P)) || (rc = dev_alloc(nullptr, (void**)&m->g, sizeof(float) * P)) ||
      (rc = dev_alloc(nullptr, (void**)&m->m, sizeof(float) * P)) || (rc = dev_alloc(nullptr, (void**)&m->v, sizeof(float) * P)) ||
      (rc = dev_alloc(nullptr, (void**)&m->w1t, 2 * 256 * lsk::kFeat)) || (rc = dev_alloc(nullptr, (void**)&m->w2t, 2 * 256 * 256)) ||
      (rc = dev_alloc(nullptr, (void**)&m->err, sizeof(int)))) {
    cudaFree(m->p);
    cudaFree(m->g);
    cudaFree(m->m);
    cudaFree(m->v);
    cudaFree(m->w1t);
    cudaFree(m->w2t);
    delete m;
    return rc;
  }
  cudaMemset(m->err, 0, sizeof(int));
  std::vector<float> h(P, 0.0f);
  if (params) {
    memcpy(h.data(), params, sizeof(float) * P);
  } else {
    // He-uniform initialisation from a seeded splitmix64 stream; biases 0
    uint64_t s = seed;
    auto uni = [&]() { return (float)((double)(splitmix(s) >> 11) * (1.0 / 9007199254740992.0)) * 2.0f - 1.0f; };
    const float a1 = std::sqrt(6.0f / 7.0f), a2 = std::sqrt(6.0f / 256.0f), a3 = std::sqrt(3.0f / 256.0f);
    for (int k = 0; k < 7; ++k)
      for (int n = 0; n < 256; ++n) h[lsk::kOffW1 + k * 256 + n] = a1 * uni();
    for (int e = 0; e < 256 * 256; ++e) h[lsk::kOffW2 + e] = a2 * uni();
    for (int e = 0; e < 256; ++e) h[lsk::kOffW3 + e] = a3 * uni();
  }
  cudaMemcpy(m->p, h.data(), sizeof(float) * P, cudaMemcpyHostToDevice);
  cudaMemset(m->m, 0, sizeof(float) * P);
  cudaMemset(m->v, 0, sizeof(float) * P);
  if ((rc = refresh(m))) {
    ls_tmp_hold(m->device);
    ls_mlp_destroy(m);
    return rc;
  }
  ls_tmp_hold(m->device);
  *out = m;
  return LS_OK;
}

int ls_mlp_destroy(ls_mlp* m) {
  if (!m) return fail(LS_ERR_ARG, "null network");
  cudaSetDevice(m->device);
  cudaFree(m->p);
  cudaFree(m->g);
  cudaFree(m->m);
  cudaFree(m->v);
  cudaFree(m->w1t);
  cudaFree(m->w2t);
  cudaFree(m->err);
  ls_tmp_release(m->device);
  delete m;
  return LS_OK;
}

int ls_mlp_get(const ls_mlp* m, float* params) {
  if (!m || !params) return fail(LS_ERR_ARG, "null argument");
  TRY(cudaMemcpy(params, m->p, sizeof(float) * lsk::kMlpParams, cudaMemcpyDeviceToHost));
  return LS_OK;
}

int ls_mlp_set(ls_mlp* m, const float* params) {
  if (!m || !params) return fail(LS_ERR_ARG, "null argument");
  TRY(cudaMemcpy(m->p, params, sizeof(float) * lsk::kMlpParams, cudaMemcpyHostToDevice));
  return refresh(m);
}

int ls_mlp_forward(const ls_mlp* m, const float* X, int64_t n, float* scores, ls_stream_t stream) {
  if (!m || (n > 0 && (!X || !scores))) return fail(LS_ERR_ARG, "null argument");
  if (n <= 0) return LS_OK;
  cudaStream_t s = (cudaStream_t)stream;
  int nsm = 0, rc;
  TRY(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, m->device));
  if ((rc = launch_scores(m, X, n, scores, nsm, s))) return rc;
  return scorer_status(m, s);
}

int ls_mlp_grad(ls_mlp* m, const float* X, const float* y, int32_t n, float* grad, double* loss, ls_stream_t stream) {
  if (!m || !X || !y || n < 1) return fail(LS_ERR_ARG, "bad arguments");
  cudaStream_t s = (cudaStream_t)stream;
  CallScratch b(s);
  GradWork gw;
  int rc = gw.setup(m, b, n, 1, s);
  if (rc) return rc;
  lsk::MlpBatch mb = {};
  mb.X = X;
  mb.y = y;
  mb.n_src = n;
  mb.B = n;
  lsk::MlpUpdate u = {};
  u.g = m->g;
  u.loss = gw.loss;
  if ((rc = gw.run(m, mb, u, s))) return rc;
  double l = 0.0;
  TRY(cudaMemcpyAsync(&l, gw.loss, sizeof(double), cudaMemcpyDeviceToHost, s));
  TRY(cudaStreamSynchronize(s));
  if (loss) *loss = l / n;
  if (grad) TRY(cudaMemcpy(grad, m->g, sizeof(float) * lsk::kMlpParams, cudaMemcpyDeviceToHost));
  return LS_OK;
}

int ls_mlp_train(ls_mlp* m, const float* X, const float* y, int64_t n, int32_t steps, int32_t batch, float lr,
                 uint64_t seed, double* loss_out, ls_stream_t stream) {
  if (!m || !X || !y || n < 1 || steps < 0 || batch < 1) return fail(LS_ERR_ARG, "bad arguments");
  cudaStream_t s = (cudaStream_t)stream;
  CallScratch b(s);
  GradWork gw;
  const int ntail = std::min(steps, std::max(1, steps / 10));  // the steps whose losses are averaged
  int rc = gw.setup(m, b, batch, ntail, s);
  if (rc) return rc;
  lsk::MlpBatch mb = {};
  mb.X = X;
  mb.y = y;
  mb.n_src = n;
  mb.B = batch;
  mb.drawn = 1;
  mb.seed = seed;
  for (int it = 0; it < steps; ++it) {
    mb.first = (uint64_t)it * (uint64_t)batch;
    ++m->t;
    lsk::MlpUpdate u = {};
    const int k = it - (steps - ntail);
    u.loss = k >= 0 ? gw.loss + k : nullptr;
    u.p = m->p;
    u.m = m->m;
    u.v = m->v;
    u.lr = lr;
    u.b1 = 0.9f;
    u.b2 = 0.999f;
    u.c1 = 1.0f - std::pow(0.9f, (float)m->t);
    u.c2 = 1.0f - std::pow(0.999f, (float)m->t);
    u.eps = 1e-8f;
    if ((rc = gw.run(m, mb, u, s))) return rc;
  }
  std::vector<double> tail(std::max(ntail, 1), 0.0);
  if (ntail) TRY(cudaMemcpyAsync(tail.data(), gw.loss, sizeof(double) * ntail, cudaMemcpyDeviceToHost, s));
  TRY(cudaStreamSynchronize(s));
  double t = 0.0;
  for (int k = 0; k < ntail; ++k) t += tail[k] / batch;
  if (loss_out) *loss_out = ntail ? t / ntail : 0.0;
  return refresh(m);
}

}  // extern "C"

namespace {
struct PropWork {
  int N = 0, L = 0, Wn = 0, Np = 0;
  uint32_t* hw = nullptr;
  uint8_t* ring[7] = {};
  int ring_w[7] = {-1, -1, -1, -1, -1, -1, -1};
  std::vector<int> nv;
};

int prop_setup(ls_ctx* c, CallScratch& b, PropWork& pw, cudaStream_t s) {
  pw.N = c->N;
  pw.L = c->L;
  pw.Wn = (c->L + lsk::kPropWS - 1) / lsk::kPropWS;
  pw.Np = lsk::round_up(c->N, 64);
  int rc;
  if ((rc = b.get(&pw.hw, (size_t)pw.Wn * pw.N * 8))) return rc;
  for (int k = 0; k < 7; ++k)
    if ((rc = b.get(&pw.ring[k], (size_t)pw.N * pw.Np))) return rc;
  lsk::hapmajor_kernel<<<dim3((pw.N + 31) / 32, 8, pw.Wn), 32, 0, s>>>(c->bits, c->row_words, pw.N, pw.L, pw.hw);
  TRY(cudaGetLastError());
  pw.nv.resize(pw.Wn);
  for (int w = 0; w < pw.Wn; ++w) pw.nv[w] = std::min(lsk::kPropWS, pw.L - w * lsk::kPropWS);
  return LS_OK;
}

int ensure(PropWork& pw, int w, cudaStream_t s) {
  const int slot = w % 7;
  if (pw.ring_w[slot] == w) return LS_OK;
  const int nb = pw.Np / 64;
  lsk::mismatch_kernel<<<dim3(nb, (pw.N + 63) / 64), 256, 0, s>>>(pw.hw + (size_t)w * pw.N * 8, pw.N, pw.Np, pw.ring[slot]);
  TRY(cudaGetLastError());
  pw.ring_w[slot] = w;
  return LS_OK;
}

int stage1(PropWork& pw, int w, int C, int32_t* cand, size_t cstride, __nv_bfloat16* feat, float* feat32,
           cudaStream_t s) {
  for (int d = -3; d <= 3; ++d) {
    const int ww = std::min(std::max(w + d, 0), pw.Wn - 1);
    int rc = ensure(pw, ww, s);
    if (rc) return rc;
  }
  lsk::Stage1Args a;
  for (int d = 0; d < 7; ++d) {
    const int ww = std::min(std::max(w + d - 3, 0), pw.Wn - 1);
    a.Ms[d] = pw.ring[ww % 7];
    a.inv_nv[d] = 1.0f / (float)pw.nv[ww];
  }
  a.use[0] = w - 1 >= 0;
  a.use[1] = 1;
  a.use[2] = w + 1 < pw.Wn;
  // one block per target, 2048 donors a warp; the histogram kernel beyond the largest block's registers
  const int threads = 32 * ((pw.N + 2047) / 2048);
  if (threads <= 256) lsk::stage1_kernel<256><<<pw.N, threads, 0, s>>>(a, pw.N, pw.Np, C, cand, cstride, feat, feat32);
  else if (threads <= 1024) lsk::stage1_kernel<1024><<<pw.N, threads, 0, s>>>(a, pw.N, pw.Np, C, cand, cstride, feat, feat32);
  else lsk::stage1_hist_kernel<<<pw.N, 256, 0, s>>>(a, pw.N, pw.Np, C, cand, cstride, feat, feat32);
  TRY(cudaGetLastError());
  return LS_OK;
}

// the K best of C scored candidates per target: C / 32 keys a lane, rounded up to a power of two
int topk(const int32_t* cand, const float* scores, int N, int C, int K, int Wn, int w, int32_t* idx, cudaStream_t s) {
  const unsigned grid = blocks(N, 8);
  if (C <= 128) lsk::topk_kernel<4><<<grid, 256, 0, s>>>(cand, scores, N, C, K, Wn, w, idx);
  else if (C <= 256) lsk::topk_kernel<8><<<grid, 256, 0, s>>>(cand, scores, N, C, K, Wn, w, idx);
  else if (C <= 512) lsk::topk_kernel<16><<<grid, 256, 0, s>>>(cand, scores, N, C, K, Wn, w, idx);
  else if (C <= 1024) lsk::topk_kernel<32><<<grid, 256, 0, s>>>(cand, scores, N, C, K, Wn, w, idx);
  else lsk::topk_kernel<64><<<grid, 256, 0, s>>>(cand, scores, N, C, K, Wn, w, idx);
  TRY(cudaGetLastError());
  return LS_OK;
}
}  // namespace

extern "C" {

int ls_propose_window(ls_ctx* ctx, int32_t C, int32_t w, int32_t* cand_out, float* feat_out, ls_stream_t stream) {
  if (!ctx || C < 1 || !cand_out) return fail(LS_ERR_ARG, "bad arguments");
  cudaSetDevice(ctx->device);
  cudaStream_t s = (cudaStream_t)stream;
  CallScratch b(s);
  PropWork pw;
  int rc = prop_setup(ctx, b, pw, s);
  if (rc) return rc;
  if (w < 0 || w >= pw.Wn) return fail(LS_ERR_ARG, "window %d outside [0, %d)", w, pw.Wn);
  if ((rc = stage1(pw, w, C, cand_out, C, nullptr, feat_out, s))) return rc;
  TRY(cudaStreamSynchronize(s));
  return LS_OK;
}

int ls_propose_labels(ls_ctx* ctx, const float* P, const int32_t* cand, int32_t C, float* y_out, ls_stream_t stream) {
  if (!ctx || !P || !cand || !y_out || C < 1) return fail(LS_ERR_ARG, "bad arguments");
  cudaSetDevice(ctx->device);
  cudaStream_t s = (cudaStream_t)stream;
  lsk::label_kernel<<<8 * ctx->num_sms, 256, 0, s>>>(P, cand, ctx->N, C, 1e-12f, y_out);
  TRY(cudaGetLastError());
  TRY(cudaStreamSynchronize(s));
  return LS_OK;
}

int ls_propose(ls_ctx* ctx, int32_t C, int32_t K, const ls_mlp* mlp, int32_t* idx_out, ls_stream_t stream) {
  if (!ctx || K < 1 || K > 512 || !idx_out) return fail(LS_ERR_ARG, "bad arguments (1 <= K <= 512)");
  if (mlp && (C < K || C > 2048)) return fail(LS_ERR_ARG, "need K <= C <= 2048 candidates for the MLP stage");
  cudaSetDevice(ctx->device);
  cudaStream_t s = (cudaStream_t)stream;
  CallScratch b(s);
  PropWork pw;
  int rc = prop_setup(ctx, b, pw, s);
  if (rc) return rc;
  const int N = pw.N, Wn = pw.Wn;
  int32_t* cand = nullptr;
  __nv_bfloat16* feat = nullptr;
  float* scores = nullptr;
  if (mlp && ((rc = b.get(&cand, (size_t)N * C)) || (rc = b.get(&feat, (size_t)N * C * 8)) ||
              (rc = b.get(&scores, (size_t)N * C))))
    return rc;
  for (int w = 0; w < Wn; ++w) {
    if (!mlp) {  // stage 1's K candidates are the set, already in ascending id order
      if ((rc = stage1(pw, w, K, idx_out + (size_t)w * K, (size_t)Wn * K, nullptr, nullptr, s))) return rc;
      continue;
    }
    if ((rc = stage1(pw, w, C, cand, C, feat, nullptr, s))) return rc;
    if ((rc = launch_scores(mlp, feat, (long long)N * C, scores, ctx->num_sms, s))) return rc;
    if ((rc = topk(cand, scores, N, C, K, Wn, w, idx_out, s))) return rc;
  }
  TRY(cudaStreamSynchronize(s));
  return mlp ? scorer_status(mlp, s) : LS_OK;
}

}  // extern "C"

// haplotype-major words of the packed rows: hw [ceil(L/256)][N][8] (the sparse recursions read
// their donors' bits from it)
cudaError_t ls_launch_hapmajor(const uint32_t* bits, int row_words, int N, int L, uint32_t* hw, cudaStream_t s) {
  const int Wn = (L + lsk::kPropWS - 1) / lsk::kPropWS;
  lsk::hapmajor_kernel<<<dim3((N + 31) / 32, 8, Wn), 32, 0, s>>>(bits, row_words, N, L, hw);
  return cudaGetLastError();
}
