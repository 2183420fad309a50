// ls_prop_inst.cu -- compiled variants of the propagation kernel and their registry.
//
// A variant is (TPW targets per CTA, W warps, KQ quads of 4 donor slots per lane); a CTA covers
// W * 32 / TPW slices of up to 4*KQ donors.  PropCfg::serves(N) decides which variants fit a
// given N; the host planner picks the one with the fewest CTA waves x slots per lane.  Variants
// are spread over translation units (LS_INST_GROUP) so the build compiles them in parallel.
#include "ls_internal.h"
#include "ls_hyb.cuh"

namespace {

template <int TPW, int W, int KQ, int PIM>
cudaError_t launch_prop(int dir, const lsk::PropParams& p, int grid, int smem, cudaStream_t s) {
  if (dir == 0) lsk::ls_prop_kernel<0, TPW, W, KQ, PIM, 0><<<grid, W * 32, smem, s>>>(p);
  else lsk::ls_prop_kernel<1, TPW, W, KQ, PIM, 0><<<grid, W * 32, smem, s>>>(p);
  return cudaGetLastError();
}

// statistic passes (forward only): dir selects ST 1 (0) or ST 2 (1)
template <int TPW, int W, int KQ>
cudaError_t launch_stat(int which, const lsk::PropParams& p, int grid, int smem, cudaStream_t s) {
  if (which == 0) lsk::ls_prop_kernel<0, TPW, W, KQ, 0, 1><<<grid, W * 32, smem, s>>>(p);
  else lsk::ls_prop_kernel<0, TPW, W, KQ, 0, 2><<<grid, W * 32, smem, s>>>(p);
  return cudaGetLastError();
}

template <int TPW, int W, int KQ, int PIM>
int smem_prop(int rw2) {
  return lsk::PropCfg<TPW, W, KQ>::layout(rw2, PIM).total;
}

template <int TPW, int W, int KQ>
bool serves_prop(int N) {
  return lsk::PropCfg<TPW, W, KQ>::serves(N);
}

// grid = number of targets; CL CTAs (a thread-block cluster when CL = 2) per target
template <int QS, int CL, int PIM>
cudaError_t launch_hyb(int dir, const lsk::PropParams& p, int grid, int smem, cudaStream_t s) {
  if (CL == 1) {
    if (dir == 0) lsk::ls_hyb_kernel<0, QS, 1, PIM><<<grid, lsk::kHybThreads, smem, s>>>(p);
    else lsk::ls_hyb_kernel<1, QS, 1, PIM><<<grid, lsk::kHybThreads, smem, s>>>(p);
    return cudaGetLastError();
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(CL * grid), 1, 1);
  cfg.blockDim = dim3(lsk::kHybThreads, 1, 1);
  cfg.dynamicSmemBytes = (size_t)smem;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = CL;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  if (dir == 0) return cudaLaunchKernelEx(&cfg, lsk::ls_hyb_kernel<0, QS, CL, PIM>, p);
  return cudaLaunchKernelEx(&cfg, lsk::ls_hyb_kernel<1, QS, CL, PIM>, p);
}
template <int QS, int PIM>
int smem_hyb(int) {
  return lsk::HybCfg<QS, PIM>::smem_bytes();
}
template <int QS, int CL, int PIM>
bool serves_hyb(int N) {
  return lsk::HybCfg<QS, PIM>::serves(N, CL);
}

// Wide tiles (one target per CTA of 8 warps, the whole state in 24, 28, .., 40 quads of registers a lane) against the
// large-N kernel (16 warps, state in registers and shared memory).  In us for eight targets an SM, tile / large-N:
//   N                     24576        28672        32768        36864        40960
//   forward, a locus      5.76 / 7.17  6.45 / 7.50  7.02 / 8.26  7.53 / 9.69  8.14 / 10.52
//   with mu per locus     7.51 / 7.34  7.84 / 7.85  8.38 / 8.28  8.67 / 9.47  9.07 / 10.15
//   backward, a locus     5.99 / 6.91  6.54 / 7.45  8.25 / 7.89  8.35 / 9.04  8.77 / 10.27
//   with mu per locus     7.77 / 7.33  7.49 / 7.94  8.78 / 8.43  9.03 / 9.25  10.12 / 10.28
//   load and save a row   158 / 131    204 / 148    207 / 160    253 / 181    255 / 201
// and decode products cost the tile more (N = 28672, L = 64, 8 decode loci: backward 37.0 / 29.4 ms; L = 200: 57.4 /
// 59.0; N = 26000, L = 100, 4 decode loci: 60.6 / 56.6 in all), so the tile needs enough loci per row transfer.
constexpr short kWideEven[5][2][2] = {{{10, 0}, {30, 0}}, {{14, 0}, {40, 400}}, {{10, 0}, {0, 0}}, {{10, 22}, {45, 80}}, {{8, 14}, {30, 90}}};

}  // namespace

// large-N variants: one target per CTA of 16 warps, 12 quads per thread in registers and QS in
// shared memory
#define LS_REGHX(QS, CL, P)                                                                         \
  out.push_back(PropKernelInfo{1, lsk::kHybThreads / 32, lsk::kHybQR + QS, P, 0,                    \
                               {(const void*)lsk::ls_hyb_kernel<0, QS, CL, P>, (const void*)lsk::ls_hyb_kernel<1, QS, CL, P>}, \
                               launch_hyb<QS, CL, P>, smem_hyb<QS, P>, serves_hyb<QS, CL, P>, CL, P})
#define LS_REGH(QS) LS_REGHX(QS, 1, 0)
// a cluster of two CTAs (on two SMs) per target: N in (57344, 2 x 2048 (12 + QS)]
#define LS_REGH2(QS) LS_REGHX(QS, 2, 0)
// prior matrix, held on chip as bfloat16 (the BF16 prior format): N in (20480, 53248] with one CTA,
// (53248, 2 x 2048 (12 + QS)] with a cluster of two
#define LS_REGHP(QS) LS_REGHX(QS, 1, 1)
#define LS_REGH2P(QS) LS_REGHX(QS, 2, 1)

#define LS_REGP(T, Wp, K, P)                                                                        \
  out.push_back(PropKernelInfo{T, Wp, K, P, 0,                                                      \
                               {(const void*)lsk::ls_prop_kernel<0, T, Wp, K, P, 0>,                \
                                (const void*)lsk::ls_prop_kernel<1, T, Wp, K, P, 0>},               \
                               launch_prop<T, Wp, K, P>, smem_prop<T, Wp, K, P>, serves_prop<T, Wp, K>, 1, P == 2})
#define LS_REG(T, Wp, K) LS_REGP(T, Wp, K, 0)
// one target per CTA of 8 warps with the whole state in registers, up to 160 slots a lane
#define LS_REGW(K)                                                                                  \
  LS_REG(1, 8, K);                                                                                  \
  out.back().even = kWideEven[(K - 24) / 4]
// statistic-pass variants: func[0] = ST 1, func[1] = ST 2
#define LS_REGS(T, Wp, K)                                                                           \
  out.push_back(PropKernelInfo{T, Wp, K, 0, 1,                                                      \
                               {(const void*)lsk::ls_prop_kernel<0, T, Wp, K, 0, 1>,                \
                                (const void*)lsk::ls_prop_kernel<0, T, Wp, K, 0, 2>},               \
                               launch_stat<T, Wp, K>, smem_prop<T, Wp, K, 0>, serves_prop<T, Wp, K>})

#if LS_INST_GROUP == 0
void ls_register_group0(std::vector<PropKernelInfo>& out) {
  // 4 targets per CTA, two CTAs per SM: N up to 5120
  LS_REG(4, 4, 40);
  LS_REG(4, 8, 20);
}
#elif LS_INST_GROUP == 1
void ls_register_group1(std::vector<PropKernelInfo>& out) {
  LS_REG(4, 4, 32);
  LS_REG(4, 4, 24);
  LS_REG(4, 4, 16);
}
#elif LS_INST_GROUP == 2
void ls_register_group2(std::vector<PropKernelInfo>& out) {
  // 8 targets per CTA for N up to 2560
  LS_REG(8, 4, 40);
  LS_REG(8, 4, 32);
  LS_REG(8, 4, 24);
}
#elif LS_INST_GROUP == 3
void ls_register_group3(std::vector<PropKernelInfo>& out) {
  LS_REG(8, 4, 16);
  LS_REG(8, 4, 8);
  LS_REG(8, 4, 4);
  LS_REG(8, 4, 2);
}
#elif LS_INST_GROUP == 4
void ls_register_group4(std::vector<PropKernelInfo>& out) {
  // 2 or 1 targets per CTA: larger N and short tails
  LS_REG(2, 4, 40);
  LS_REG(1, 4, 40);
  LS_REG(1, 4, 32);
}
#elif LS_INST_GROUP == 5
void ls_register_group5(std::vector<PropKernelInfo>& out) {
  LS_REG(1, 4, 24);
  LS_REG(1, 4, 16);
  LS_REG(1, 4, 8);
  LS_REG(1, 4, 1);
}
#elif LS_INST_GROUP == 6
void ls_register_group6(std::vector<PropKernelInfo>& out) {
  // prior-matrix variants: one target per CTA covers every N up to 20480
  LS_REGP(1, 4, 1, 1);
  LS_REGP(1, 4, 8, 1);
  LS_REGP(1, 4, 16, 1);
  LS_REGP(1, 4, 24, 1);
}
#elif LS_INST_GROUP == 7
void ls_register_group7(std::vector<PropKernelInfo>& out) {
  LS_REGP(1, 4, 32, 1);
  LS_REGP(1, 4, 40, 1);
  LS_REGP(1, 8, 20, 1);
  LS_REGP(8, 4, 16, 1);
}
#elif LS_INST_GROUP == 10
void ls_register_group10(std::vector<PropKernelInfo>& out) {
  // two-CTA clusters: N in (57344, 81920]
  LS_REGH2(4);
  LS_REGH2(8);
}
#elif LS_INST_GROUP == 11
void ls_register_group11(std::vector<PropKernelInfo>& out) {
  // N in (81920, 114688]
  LS_REGH2(12);
  LS_REGH2(13);
  LS_REGH2(16);
}
#elif LS_INST_GROUP == 12
void ls_register_group12(std::vector<PropKernelInfo>& out) {
  // one target per CTA of 8 warps with the whole state in registers: N in (16384, 40960], where kWideEven says so
  // beyond 20480; N <= 20480 runs faster with two CTAs of 4 warps an SM
  LS_REGW(24);
  LS_REGW(28);
  LS_REGW(32);
}
#elif LS_INST_GROUP == 21
void ls_register_group21(std::vector<PropKernelInfo>& out) {
  LS_REGW(36);
  LS_REGW(40);
}
#elif LS_INST_GROUP == 22
void ls_register_group22(std::vector<PropKernelInfo>& out) {
  // register + shared-memory state, N in (20480, 40960]
  LS_REGH(0);
  LS_REGH(2);
  LS_REGH(4);
  LS_REGH(6);
  LS_REGH(8);
}
#elif LS_INST_GROUP == 13
void ls_register_group13(std::vector<PropKernelInfo>& out) {
  // N in (40960, 57344]
  LS_REGH(10);
  LS_REGH(12);
  LS_REGH(13);
  LS_REGH(14);
  LS_REGH(16);
}
#elif LS_INST_GROUP == 16
void ls_register_group16(std::vector<PropKernelInfo>& out) {
  // prior matrix held as bfloat16 (the BF16 prior format), N up to 20480
  LS_REGP(1, 4, 1, 2);
  LS_REGP(1, 4, 8, 2);
  LS_REGP(1, 4, 16, 2);
  LS_REGP(1, 4, 24, 2);
}
#elif LS_INST_GROUP == 17
void ls_register_group17(std::vector<PropKernelInfo>& out) {
  LS_REGP(1, 4, 32, 2);
  LS_REGP(1, 4, 40, 2);
  LS_REGP(1, 8, 20, 2);
  LS_REGP(8, 4, 16, 2);
}
#elif LS_INST_GROUP == 14
void ls_register_group14(std::vector<PropKernelInfo>& out) {
  // prior matrix (BF16 format), one CTA per target: N in (20480, 53248]
  LS_REGHP(0);
  LS_REGHP(4);
  LS_REGHP(8);
  LS_REGHP(14);
}
#elif LS_INST_GROUP == 15
void ls_register_group15(std::vector<PropKernelInfo>& out) {
  // prior matrix (BF16 format), two-CTA clusters: N in (53248, 106496]
  LS_REGH2P(4);
  LS_REGH2P(8);
  LS_REGH2P(14);
}
#elif LS_INST_GROUP == 18
void ls_register_group18(std::vector<PropKernelInfo>& out) {
  // one warp per target for N up to 1024: small data sets are bound by the latency of a locus, and a
  // single warp needs no CTA barrier and no exchange through shared memory (N = 64 / 200 / 500: 0.242 /
  // 0.250 / 0.261 us per locus against 0.285 / 0.269 / 0.293 for the best four-warp variants).  Beyond
  // 1024 the four-warp variants are faster (N = 2000: 0.69 against 0.89 us, N = 5000: 3.76 against 3.92).
  LS_REG(1, 1, 8);
  LS_REG(1, 1, 4);
  LS_REG(1, 1, 2);
  LS_REG(1, 1, 1);
}
#elif LS_INST_GROUP == 8
void ls_register_group8(std::vector<PropKernelInfo>& out) {
  // statistic passes of the adjoint (uniform prior): two tiles per lane.  With many targets, as many per CTA as
  // keep a lane's slices long, because the work per locus that does not scale with the slice is the larger
  // part of a short one (N = 2003, L = 1999, one target of 16 slots a lane against four of 63: 7.8 / 8.5 ->
  // 3.7 / 3.3 ms for the two passes).  One target per CTA serves every N up to 10240 too: it is the faster
  // tile where the targets would not fill the GPU otherwise, and the one that fits any scratch ceiling.
  LS_REGS(1, 4, 1);
  LS_REGS(1, 4, 8);
  LS_REGS(8, 4, 4);
  LS_REGS(8, 4, 8);
}
#elif LS_INST_GROUP == 9
void ls_register_group9(std::vector<PropKernelInfo>& out) {
  LS_REGS(1, 4, 16);
  LS_REGS(1, 4, 20);
}
#elif LS_INST_GROUP == 19
void ls_register_group19(std::vector<PropKernelInfo>& out) {
  LS_REGS(8, 4, 16);
  LS_REGS(4, 4, 16);
}
#elif LS_INST_GROUP == 20
void ls_register_group20(std::vector<PropKernelInfo>& out) {
  LS_REGS(4, 4, 20);
  LS_REGS(2, 4, 16);
  LS_REGS(2, 4, 20);
}
#endif
