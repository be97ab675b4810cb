// GEMM for passes of hundreds to thousands of token rows (the prefill): host-side interface.
#pragma once
#include "tma_maps.cuh"

namespace spec {

enum WideEpi {
  WIDE_RESID = 0,    // x[r][o] (+)= acc; hb = bf16(x * gain[o]); per-128-feature sums of squares; optional taps
  WIDE_QKV = 1,      // scale, rotate q and k by the row's position, store q, write K/V into the paged cache (head_dim 128)
  WIDE_SWIGLU = 2,   // two weights (gate, up): act = bf16(silu(scale*g) * scale*u)
  WIDE_BF16 = 3,     // out_b[r][o] = bf16(acc)
  WIDE_F32 = 4,      // out_f32[r][o] = scale * acc
  WIDE_ARGMAX = 5    // per (128 features, row) best (value, index); optional fp32 logits (scale * acc)
};

struct WideGemmArgs {
  // out[r][o] = sum_i x[r][i] * w[o][i]; x has x_rows allocated rows of which the first `rows` are computed
  const bf16 *x = nullptr;
  int rows = 0, x_rows = 0, I = 0;
  const bf16 *w[3] = {nullptr, nullptr, nullptr};   // [O[j]][I]
  int O[3] = {0, 0, 0};
  int nw = 1;
  // per-row scale of the input: rsqrt(sum_t ssq_in[t * ssq_ld + r] / k_in + eps); nullptr: 1
  const float *ssq_in = nullptr;
  int ssq_in_tiles = 0, ssq_ld = 0, k_in = 1;
  float eps = 0.0f;
  // WIDE_RESID (O[0] = width of the residual stream)
  float *xres = nullptr;
  const bf16 *gain = nullptr;
  bf16 *hb = nullptr;
  float *ssq_out = nullptr;     // [ceil(O/128)][ssq_ld]
  bf16 *taps = nullptr;         // [rows][3*O], slot s written when bit s of tap_mask is set
  int tap_mask = 0;
  int resid_add = 1;
  // WIDE_QKV: w = {wq, wk, wv}, or {wk, wv} when only the cache is to be written (nw = 2)
  const float2 *cs = nullptr;   // [rows][64] (cos, sin)
  const int32_t *slot = nullptr;   // [rows] cache row page * G * page_size + offset of the row's K/V; -1: none is written
  const int32_t *seq = nullptr, *kvpos = nullptr;   // without `slot`: the row's sequence (-1: padding, q = 0) and cache position
  PageMap pm = {nullptr, 0, 0, 0};
  bf16 *q = nullptr;            // [rows][H][128]
  KvPool pool = {nullptr, nullptr};
  int H = 0, G = 0, page_size = 0;
  // WIDE_SWIGLU
  bf16 *act = nullptr;          // [rows][O[0]]
  // WIDE_BF16
  bf16 *out_b = nullptr;
  int ldo = 0;
  // WIDE_F32, the logits of WIDE_ARGMAX (may be null there)
  float *out_f32 = nullptr;     // row pitch ldo
  // WIDE_ARGMAX
  float *best_val = nullptr;    // [ceil(O/128)][best_ld]
  int32_t *best_idx = nullptr;
  int best_ld = 0;
  // Form of the kernel, 0: the plan's choice.  WIDE_SWIGLU: features per tile (a multiple of 16 in 64..256), else K slices
  // (1..4, for the epilogues that split; 1 also selects the persistent gate/up kernel).  `used` receives what ran.
  int form = 0;
  int *used = nullptr;
  // launch
  int32_t *status = nullptr;
  bool pdl = false;
  unsigned long long *stamp = nullptr;   // profiling aid (see KernelStamp)
};

// Test hook of the calling thread's launches: in launches of one of the three kernels the first CTA never receives its first
// activation tile, and the waits of the launch give up after 2000 polls.
enum WideTest { WIDE_TEST_OFF = 0, WIDE_TEST_PERSISTENT = 1, WIDE_TEST_SPLIT = 2, WIDE_TEST_GATE_UP = 3 };
extern thread_local int tl_wide_test;

constexpr int WIDE_ROWS = 256;      // token rows per tile
// what the launch's time goes with, in k-blocks (64 elements of the contraction, 0.27 us) of a tile
long long wide_gemm_cost(WideEpi epi, const int *O, int nw, int I, int row_tiles);
// whether a launch takes these widths and alignments
bool wide_gemm_supported(WideEpi epi, const WideGemmArgs &a);
// Returns 0 or a negative code (-1: not supported).
int wide_gemm_launch(TmaMaps *g, WideEpi epi, const WideGemmArgs &a, cudaStream_t s);

}  // namespace spec
