// Causal paged GQA attention for long runs of query positions (prefill, training-time test): host-side interface.
#pragma once
#include <cuda.h>

#include "common.cuh"

namespace spec {

constexpr int CAUSAL_TILE = 128;       // query positions per tile; a CTA works on two tiles

// One block of query rows of one sequence: rows row0 .. row0 + nrows - 1 of q are positions pos0 .. of sequence seq.  With
// an even number of query heads per KV head a block holds up to 128 rows (a CTA takes two heads of it), otherwise 256.
struct CausalBlock {
  int32_t row0, nrows, seq, pos0;
  int32_t tok0, len, pad0, pad1;       // prefill: where the sequence's prompt starts in the concatenated ids, and its length
};
inline int causal_block_rows(int group) { return group % 2 == 0 ? CAUSAL_TILE : 2 * CAUSAL_TILE; }

// head_dim 128, page sizes 16 / 32 / 64
bool causal_attn_supported(int head_dim, int page_size);

struct CausalArgs {
  const bf16 *q = nullptr;             // [q_rows][H][128], q_rows allocated rows
  int q_rows = 0;
  KvPool pool = {nullptr, nullptr};    // [pages][G][page_size][128]
  PageMap pm = {nullptr, 0, 0, 0};
  bf16 *out = nullptr;                 // [rows][H][128]
  int H = 0, G = 0;
  const CausalBlock *blocks = nullptr; // device, longest context first; nullptr: one sequence of T rows at position 0
  int n_blocks = 0, T = 0;
  // extra keys on the diagonal (training-time test): kd / vd [J][T][G][128], lse [T][H] (optional); blocks == nullptr only
  const bf16 *kd = nullptr, *vd = nullptr;
  int J = 0;
  float *lse = nullptr;
  int32_t *status = nullptr;
};
// Test hook of the calling thread's launches.  LATE: the softmax warps pause for tens of microseconds before they wait for
// the last contraction of their tile, which is complete long before they look.  WITHHOLD: the first CTA never receives its
// queries and gives up after 2000 polls.
enum CausalTest { CAUSAL_TEST_OFF = 0, CAUSAL_TEST_LATE = 1, CAUSAL_TEST_WITHHOLD = 2 };
extern thread_local int tl_causal_test;

// Returns 0 or a negative code.
int launch_causal_attn(const CausalArgs &a, cudaStream_t s);

}  // namespace spec
