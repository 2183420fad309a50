// ls_internal.h -- host-side structures shared by the libls translation units.
#pragma once

#include <algorithm>
#include <cstdint>
#include <mutex>
#include <vector>

#include <cuda_runtime.h>

#include "ls_prop.cuh"

// One compiled variant of the propagation kernel: TPW targets per CTA, W warps, KQ quads per lane
// (forward and backward instantiations).
struct PropKernelInfo {
  int tpw, w, kq;
  int pim;  // prior-matrix variant: 1 FP32 prior values, 2 bfloat16 (0: uniform prior)
  int st;   // 1: statistic-pass variant (launch's dir argument picks ST 1 or ST 2)
  const void* func[2];
  cudaError_t (*launch)(int dir, const lsk::PropParams& p, int grid, int smem, cudaStream_t s);
  int (*smem_bytes)(int rw2);
  bool (*serves)(int N);
  int cpt = 1;  // CTAs per target (2: a thread-block cluster of two CTAs shares one target)
  int pi16 = 0; // 1: holds the prior matrix on chip as bfloat16 (needs the BF16 prior format)
  // a variant with a slower rival in long runs only: loci per row transfer from which it is the faster one, by
  // direction and by kind of mu (scalar, per locus); 0: never; null: no such rival
  const short (*even)[2] = nullptr;
};

// a variant that serves a context, the dynamic shared memory it takes there and the CTAs an SM holds
struct PropCand {
  const PropKernelInfo* k;
  int smem, per_sm;
};
// Upper bound on compiled variants (the registry is a fixed list; the candidates sit in fixed arrays so that the
// allocation-free pipeline shares the planner).
constexpr int kMaxCand = 64;

void ls_register_prop_kernels(std::vector<PropKernelInfo>& out);

// shared by the translation units: set the thread's error message and return code; device
// allocation with LS_ERR_OOM on failure
int ls_fail(int code, const char* fmt, ...);
int ls_dev_alloc(void** p, size_t bytes);

// Scratch of one call, from a pool per device: allocated and freed in the order of the call's stream, so that
// a call neither waits for the device twice nor maps its gigabytes anew each time (a gradient of 2.4 GB
// scratch spent 2.5 of 11.7 ms in cudaMalloc and cudaFree).  The pool keeps at most kTmpKeep bytes between
// calls and gives everything back when the last context and network of the device is destroyed.
// ls_tmp_hold / ls_tmp_release count those; the pool is safe with any threads and streams.
constexpr size_t kTmpKeep = (size_t)4 << 30;
int ls_tmp_alloc(void** p, size_t bytes, cudaStream_t s);
void ls_tmp_free(void* p, cudaStream_t s);
void ls_tmp_hold(int device);
void ls_tmp_release(int device);

// Scratch of one call.  What goes beyond kTmpKeep is the call's own allocation: from the pool it would be
// mapped and unmapped by every call, which takes longer (a gradient with 16 GB of scratch at N = 9000: 62.2
// against 48.3 ms, a proposal at N = 60000: 76.1 against 48.8 ms).
struct CallScratch {
  cudaStream_t s;
  std::vector<void*> pooled, own;
  size_t taken = 0;
  explicit CallScratch(cudaStream_t stream) : s(stream) {}
  CallScratch(const CallScratch&) = delete;
  ~CallScratch() {
    for (void* p : pooled) ls_tmp_free(p, s);
    if (!own.empty()) cudaStreamSynchronize(s);
    for (void* p : own) cudaFree(p);
  }
  template <class T>
  int get(T** p, size_t n) {
    const size_t bytes = sizeof(T) * std::max<size_t>(n, 1);
    const bool pool = taken + bytes <= kTmpKeep;
    const int rc = pool ? ls_tmp_alloc((void**)p, bytes, s) : ls_dev_alloc((void**)p, bytes);
    if (rc) return rc;
    if (pool) taken += bytes;
    (pool ? pooled : own).push_back(*p);
    return 0;
  }
};

namespace lsk {
struct SparseParams;
}
cudaError_t ls_launch_sparse(int dir, const lsk::SparseParams& p, cudaStream_t s);
cudaError_t ls_launch_row_ones(const uint32_t* bits, int row_words, int N, int L, int32_t* n1, cudaStream_t s);
cudaError_t ls_launch_emission(const float* thm, const float* thx, int L, float* ratio, cudaStream_t s);
cudaError_t ls_launch_hapmajor(const uint32_t* bits, int row_words, int N, int L, uint32_t* hw, cudaStream_t s);
cudaError_t ls_launch_lookahead(const int32_t* idx, int N, int Wn, int K, int span, int32_t* U, cudaStream_t s);
cudaError_t ls_launch_sparse_hdist(const float* P, const int32_t* idx, int N, int K, int Wn, const int* win_of_slot,
                                   const float* share, int D, float* h, cudaStream_t s);
cudaError_t ls_launch_symmetrize_trust(float* d, int N, int D, const uint8_t* dense_row, float d_trust, uint32_t* mask,
                                       cudaStream_t s);
cudaError_t ls_launch_dense_rows_hdist(const float* prod, int nf, int N, const int* tlist, const uint32_t* bits,
                                       int row_words, const float* thm, const float* thx, const int* dloci, int D, float* h,
                                       cudaStream_t s);

struct ls_ctx {
  int device = 0;
  int N = 0, L = 0, row_words = 0;
  uint32_t* bits = nullptr;       // [L][row_words], the packed cache
  uint32_t* bits2 = nullptr;      // [L][rw2], every row doubled (2N bits) for the propagation kernel
  int rw2 = 0;
  size_t bytes = 0;               // device bytes owned
  // parameters
  bool have_params = false;
  uint64_t hash = 0;
  float* omr = nullptr;           // [L-1] 1 - rho
  float* rr_f = nullptr;          // [L-1] rho * pi (forward)
  float* rr_b = nullptr;          // [L-1] rho (backward)
  float* thm = nullptr;           // [L] 1 - mu
  float* thx = nullptr;           // [L] mu
  float* Pi = nullptr;            // [N][N] prior matrix copy (null: uniform)
  int prior_bf16 = 0;             // LS_PRIOR_BF16: Pi rounded to bfloat16 by ls_set_params
  float pi_u = 0.0f;
  int mu_vec = 0;                 // mu given per locus
  std::vector<double> rho_h, mu_h;  // host copies (the gradient's constant terms)
  // scratch (log scales and status words that no call reads back)
  double* logs_scratch = nullptr; // [N]
  uint32_t* status_scratch = nullptr;  // [N]
  int* err = nullptr;             // device error word
  float* dscratch = nullptr;      // host-output staging for ls_run_all
  size_t dscratch_bytes = 0;
  int num_sms = 0;
  int ntables = 0;
  // profiling of ls_run_all phases
  bool profile = false;
  bool profiled = false;
  cudaEvent_t ev[5] = {nullptr, nullptr, nullptr, nullptr, nullptr};
  // side stream for the tail launch of a main/tail plan and for the backward of small data sets (fork/join
  // events on the caller's stream; the mutex keeps each record and its wait together)
  cudaStream_t side = nullptr;
  cudaEvent_t fork_ev = nullptr, join_ev = nullptr;
  std::mutex side_mu;
  // the variants that serve the context, by prior kind (none, FP32, BF16), from the first plan on
  struct {
    int n = -1;
    PropCand c[kMaxCand];
  } cand[3];
  std::mutex cand_mu;
  int launches[4] = {0, 0, 0, 0};
};

struct ls_ckpt {
  ls_ctx* ctx = nullptr;
  int dtype = 0;
  int t_from = 0, t_to = 0;
  std::vector<int> loci;     // c_0 < c_1 < ... < c_{K-1}
  uint64_t hash = 0;
  void* data = nullptr;      // [K][T][N] float or binary16
  float* scale = nullptr;    // [K][T] (binary16 only)
  double* logs = nullptr;    // [K][T]
  size_t bytes = 0;
};

struct ls_table {
  ls_ctx* ctx = nullptr;
  int kind = 0;
  int t_from = 0, t_to = 0;
  int locus = -1;
  uint64_t hash = 0;
  float* state = nullptr;   // [T][N]
  double* logs = nullptr;   // [T]
};
