// Integer / fp32-compare kernels of the step: per-row log-softmax + top-k, dynamic-tree expansion
// (Section 2.2: expand by draft confidence, cumulative log-probability as the node value), the
// end-of-draft pruning ("rerank") that fixes the verified tree and its ancestor masks, per-node
// argmax, greedy acceptance (Section 2.1 at temperature 0) and KV-cache compaction.
#include "state.cuh"

namespace spec {

bool draft_tree_step_fits(int tiles, int K);
int draft_tree_cand_ld(int tiles);

// ---------------------------------------------------------------- block argmax helpers
struct VI { float v; int i; };

__device__ __forceinline__ VI block_best(VI x, VI *sh) {
  for (int o = 16; o > 0; o >>= 1) {
    float ov = __shfl_xor_sync(0xffffffffu, x.v, o);
    int oi = __shfl_xor_sync(0xffffffffu, x.i, o);
    if (oi >= 0 && (x.i < 0 || before(ov, oi, x.v, x.i))) { x.v = ov; x.i = oi; }
  }
  int w = threadIdx.x >> 5, l = threadIdx.x & 31, nw = blockDim.x >> 5;
  if (l == 0) sh[w] = x;
  __syncthreads();
  if (w == 0) {
    VI t = (l < nw) ? sh[l] : VI{0.0f, -1};
    for (int o = 16; o > 0; o >>= 1) {
      float ov = __shfl_xor_sync(0xffffffffu, t.v, o);
      int oi = __shfl_xor_sync(0xffffffffu, t.i, o);
      if (oi >= 0 && (t.i < 0 || before(ov, oi, t.v, t.i))) { t.v = ov; t.i = oi; }
    }
    if (l == 0) sh[0] = t;
  }
  __syncthreads();
  VI r = sh[0];
  __syncthreads();
  return r;
}

__global__ void __launch_bounds__(256) argmax_kernel(const float *__restrict__ logits, int n, int32_t *__restrict__ out) {
  pdl_wait();
  pdl_trigger();
  __shared__ VI sh[32];
  const float *z = logits + (size_t)blockIdx.x * n;
  VI b{0.0f, -1};
#pragma unroll 8
  for (int i = threadIdx.x; i < n; i += blockDim.x) {      // the loads of eight rounds in flight
    float v = z[i];
    if (b.i < 0 || before(v, i, b.v, b.i)) { b.v = v; b.i = i; }
  }
  b = block_best(b, sh);
  if (threadIdx.x == 0) out[blockIdx.x] = b.i;
}
void launch_argmax(const float *logits, int rows, int n, int32_t *idx, cudaStream_t s) {
  launch_k(argmax_kernel, dim3(rows), dim3(256), 0, s, logits, n, idx);
}

// log-softmax + top-K, (value desc, index asc).  Row r reads logits row src_row[r] when given.
// PER > 0: up to PER * 256 logits, which a thread reads once and keeps; every warp then ranks its own K best by warp-wide reductions, and
// a thread per entry those of all warps by counting.  PER = 0: any number, read again for each of the K results.  Cold, PER = 0 / PER > 0: 1024
// logits, K = 4: 9.4 / 5.6 us.  (With the keys made again for each result and all 8 K entries ranked by one warp, K = 16 took 16.6 to 17.2 us
// at 200 logits where PER = 0 takes 15.4, and 1024 rows of 1025 logits 58 where it takes 43.)
template <int PER>
__global__ void __launch_bounds__(256) logsoftmax_topk_kernel(const float *__restrict__ logits, const int32_t *src_row,
                                                              int n, int K, int32_t *__restrict__ idx,
                                                              float *__restrict__ lp) {
  pdl_wait();
  pdl_trigger();
  __shared__ VI sh[32];
  __shared__ float shf[2][8];
  __shared__ uint2 cand[8 * 16];
  int r = blockIdx.x;
  int sr = src_row ? src_row[r] : r;
  if (sr < 0) {
    for (int c = threadIdx.x; c < K; c += blockDim.x) { idx[(size_t)r * K + c] = 0; lp[(size_t)r * K + c] = 0.0f; }
    return;
  }
  const float *z = logits + (size_t)sr * n;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float v[PER > 0 ? PER : 1];
  float mx = -INFINITY;
  if (PER > 0) {
#pragma unroll
    for (int j = 0; j < PER; j++) { const int i = threadIdx.x + j * 256; v[j] = i < n ? z[i] : -INFINITY; }
#pragma unroll
    for (int j = 0; j < PER; j++) mx = fmaxf(mx, v[j]);
  } else {
    for (int i = threadIdx.x; i < n; i += blockDim.x) mx = fmaxf(mx, z[i]);
  }
  for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  if (lane == 0) shf[0][warp] = mx;
  __syncthreads();
  mx = shf[0][0];
#pragma unroll
  for (int w = 1; w < 8; w++) mx = fmaxf(mx, shf[0][w]);
  float sum = 0.0f;
  if (PER > 0) {
#pragma unroll
    for (int j = 0; j < PER; j++) sum += threadIdx.x + j * 256 < n ? expf(v[j] - mx) : 0.0f;
  } else {
    for (int i = threadIdx.x; i < n; i += blockDim.x) sum += expf(z[i] - mx);
  }
  for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
  if (lane == 0) shf[1][warp] = sum;
  __syncthreads();
  sum = 0.0f;
#pragma unroll
  for (int w = 0; w < 8; w++) sum += shf[1][w];
  const float lse = logf(sum);
  if (PER > 0) {
    unsigned key[PER > 0 ? PER : 1];                       // of this thread's values that are still to be taken (keys of values are >= 1)
#pragma unroll
    for (int j = 0; j < PER; j++) key[j] = threadIdx.x + j * 256 < n ? ordered_key((v[j] - mx) - lse) : 0u;
    for (int c = 0; c < K; c++) {
      unsigned bk = 0u, wk;
      int bj = -1;
#pragma unroll
      for (int j = 0; j < PER; j++)
        if (key[j] > bk) { bk = key[j]; bj = j; }          // equal: the lower index stays
      const int bi = bj < 0 ? -1 : (int)threadIdx.x + bj * 256;
      const int wi = warp_best(bk, bi, &wk);
#pragma unroll
      for (int j = 0; j < PER; j++)
        if (wi == (int)threadIdx.x + j * 256) key[j] = 0u;
      if (lane == 0) cand[warp * K + c] = make_uint2(wk, (unsigned)wi);
    }
    __syncthreads();
    if ((int)threadIdx.x >= 8 * K) return;                 // an entry per thread: one warp for all of them took a third of the launch at K = 16
    const uint2 me = cand[threadIdx.x];
    if ((int)me.y < 0) return;                             // its warp has fewer than K values
    int rank = 0;
    for (int o = 0; o < 8 * K; o++) { const uint2 w = cand[o]; rank += (int)w.y >= 0 && (w.x > me.x || (w.x == me.x && w.y < me.y)); }
    if (rank < K) { idx[(size_t)r * K + rank] = (int)me.y; lp[(size_t)r * K + rank] = key_value(me.x); }
    return;
  }
  float pv = INFINITY;
  int pi = -1;
  for (int c = 0; c < K; c++) {
    VI b{0.0f, -1};
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
      float x = (z[i] - mx) - lse;
      bool after_prev = (pi < 0) || before(pv, pi, x, i);
      if (after_prev && (b.i < 0 || before(x, i, b.v, b.i))) { b.v = x; b.i = i; }
    }
    b = block_best(b, sh);
    if (threadIdx.x == 0) { idx[(size_t)r * K + c] = b.i; lp[(size_t)r * K + c] = b.v; }
    pv = b.v; pi = b.i;
  }
}
void launch_logsoftmax_topk_rows(const float *logits, const int32_t *src_row, int rows, int n, int K, int32_t *idx,
                                 float *lp, cudaStream_t s) {
  auto kern = K > 16 || n > 8 * 256 ? logsoftmax_topk_kernel<0> : n <= 4 * 256 ? logsoftmax_topk_kernel<4> : logsoftmax_topk_kernel<8>;
  launch_k(kern, dim3(rows), dim3(256), 0, s, logits, src_row, n, K, idx, lp);
}
void launch_logsoftmax_topk(const float *logits, int rows, int n, int K, int32_t *idx, float *lp, cudaStream_t s) {
  launch_logsoftmax_topk_rows(logits, nullptr, rows, n, K, idx, lp, s);
}


// ---------------------------------------------------------------- two-stage log-softmax + top-K
// Stage 1: one CTA per (row, chunk of TOPK_CHUNK logits): chunk maximum, sum of exp relative to it, and
// the chunk's K best (value desc, index asc).  Stage 2: one CTA per row merges the chunks: log-sum-exp
// of the row and the K best of the chunk candidates, ranked by counting.
constexpr int TOPK_CHUNK = 1024;
constexpr int TOPK_MAXK = 16;

__global__ void __launch_bounds__(256) topk_partial_kernel(const float *__restrict__ logits, const int32_t *src_row, int n,
                                                           int K, int nch, float *__restrict__ pmax,
                                                           float *__restrict__ psum, float *__restrict__ cval,
                                                           int32_t *__restrict__ cidx) {
  pdl_wait();
  pdl_trigger();
  // Warp w owns the 128 consecutive logits base + 128 w ...: it finds its own K best with shuffles only (no block
  // barrier per round); the 8 x K warp candidates are then ranked against each other by counting.
  __shared__ float shf[8];
  __shared__ float wv[8 * TOPK_MAXK];
  __shared__ int32_t wi[8 * TOPK_MAXK];
  const int r = blockIdx.y, ch = blockIdx.x;
  const int sr = src_row ? src_row[r] : r;
  if (sr < 0) return;
  const float *z = logits + (size_t)sr * n;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int base = ch * TOPK_CHUNK + warp * 128;
  float v[4];
  int id[4];
  float mx = -INFINITY;
#pragma unroll
  for (int j = 0; j < 4; j++) {
    id[j] = base + j * 32 + lane;
    v[j] = id[j] < n ? z[id[j]] : -INFINITY;
    if (id[j] >= n) id[j] = -1;
    mx = fmaxf(mx, v[j]);
  }
  for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  if (lane == 0) shf[warp] = mx;
  __syncthreads();
  mx = shf[0];
  for (int w = 1; w < 8; w++) mx = fmaxf(mx, shf[w]);
  __syncthreads();
  float sum = 0.0f;
#pragma unroll
  for (int j = 0; j < 4; j++) sum += id[j] >= 0 ? expf(v[j] - mx) : 0.0f;
  for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
  if (lane == 0) shf[warp] = sum;
  // ---- this warp's K best, best first
  for (int c = 0; c < K; c++) {
    float bv = 0.0f;
    int bi = -1;
#pragma unroll
    for (int j = 0; j < 4; j++)
      if (id[j] >= 0 && (bi < 0 || before(v[j], id[j], bv, bi))) { bv = v[j]; bi = id[j]; }
    for (int o = 16; o > 0; o >>= 1) {
      const float ov = __shfl_xor_sync(0xffffffffu, bv, o);
      const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
      if (oi >= 0 && (bi < 0 || before(ov, oi, bv, bi))) { bv = ov; bi = oi; }
    }
#pragma unroll
    for (int j = 0; j < 4; j++)
      if (id[j] == bi) id[j] = -1;            // taken (bi is -1 only when the warp's range is exhausted)
    if (lane == 0) { wv[warp * K + c] = bv; wi[warp * K + c] = bi; }
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    float t = 0.0f;
    for (int w = 0; w < 8; w++) t += shf[w];
    pmax[(size_t)r * nch + ch] = mx;
    psum[(size_t)r * nch + ch] = t;
  }
  // ---- the chunk's K best of the 8 K warp candidates, by rank (value desc, index asc)
  const int nc = 8 * K;
  int my = -1;
  float mv = 0.0f;
  if ((int)threadIdx.x < nc) { my = wi[threadIdx.x]; mv = wv[threadIdx.x]; }
  const int nvalid = __syncthreads_count(my >= 0);
  if (my >= 0) {
    int rank = 0;
    for (int j = 0; j < nc; j++) rank += (wi[j] >= 0 && before(wv[j], wi[j], mv, my)) ? 1 : 0;
    if (rank < K) {
      cval[((size_t)r * nch + ch) * K + rank] = mv;
      cidx[((size_t)r * nch + ch) * K + rank] = my;
    }
  }
  for (int c = nvalid + (int)threadIdx.x; c < K; c += blockDim.x) {      // fewer than K logits in the chunk
    cval[((size_t)r * nch + ch) * K + c] = 0.0f;
    cidx[((size_t)r * nch + ch) * K + c] = -1;
  }
}

__global__ void __launch_bounds__(256) topk_merge_kernel(const int32_t *src_row, int K, int nch, const float *__restrict__ pmax,
                                                         const float *__restrict__ psum, const float *__restrict__ cval,
                                                         const int32_t *__restrict__ cidx, int32_t *__restrict__ idx,
                                                         float *__restrict__ lp) {
  pdl_wait();
  pdl_trigger();
  extern __shared__ unsigned char smraw[];
  __shared__ float shf[32];
  int r = blockIdx.x;
  int sr = src_row ? src_row[r] : r;
  if (sr < 0) {
    for (int c = threadIdx.x; c < K; c += blockDim.x) { idx[(size_t)r * K + c] = 0; lp[(size_t)r * K + c] = 0.0f; }
    return;
  }
  int nc = nch * K;
  float *cv = (float *)smraw;              // [nc]
  int32_t *ci = (int32_t *)(cv + nc);      // [nc]
  float *pm = (float *)(ci + nc);          // [nch]
  float *ps = pm + nch;                    // [nch]
  __shared__ float sv[TOPK_MAXK * TOPK_MAXK];      // candidates that can still be among the K best
  __shared__ int32_t si[TOPK_MAXK * TOPK_MAXK];
  __shared__ int nsurv, thr_i;
  __shared__ float thr_v;
  for (int i = threadIdx.x; i < nc; i += blockDim.x) { cv[i] = cval[(size_t)r * nc + i]; ci[i] = cidx[(size_t)r * nc + i]; }
  float mx = -INFINITY;
  for (int i = threadIdx.x; i < nch; i += blockDim.x) {
    float m = pmax[(size_t)r * nch + i];
    pm[i] = m; ps[i] = psum[(size_t)r * nch + i];
    mx = fmaxf(mx, m);
  }
  for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  if ((threadIdx.x & 31) == 0) shf[threadIdx.x >> 5] = mx;
  if (threadIdx.x == 0) { nsurv = 0; thr_i = -1; thr_v = 0.0f; }
  __syncthreads();
  mx = shf[0];
  for (int w = 1; w < 8; w++) mx = fmaxf(mx, shf[w]);
  __syncthreads();
  // chunk sums are combined in chunk order by one thread: the result does not depend on the launch shape
  if (threadIdx.x == 0) {
    float t = 0.0f;
    for (int i = 0; i < nch; i++) t += ps[i] * expf(pm[i] - mx);
    shf[0] = logf(t);
  }
  // A chunk's candidates are stored best first.  With t = the K-th best of the chunks' best candidates, K
  // candidates are at least as good as t, so a candidate after t cannot be among the K best of the row.
  for (int ch = (int)threadIdx.x - 32; ch < nch; ch += (int)blockDim.x - 32) {       // warp 0 is busy with the sum
    if (ch < 0) break;
    int c0 = ch * K, my = ci[c0];
    if (my < 0) continue;
    float v = cv[c0];
    int rank = 0;
    for (int j = 0; j < nch; j++) rank += (ci[j * K] >= 0 && before(cv[j * K], ci[j * K], v, my)) ? 1 : 0;
    if (rank == K - 1) { thr_v = v; thr_i = my; }
  }
  __syncthreads();
  float lse = shf[0];
  const float tv = thr_v;
  const int ti = thr_i;
  for (int i = threadIdx.x; i < nc; i += blockDim.x) {
    int my = ci[i];
    if (my < 0 || (ti >= 0 && before(tv, ti, cv[i], my))) continue;
    int pos = atomicAdd(&nsurv, 1);        // at most K chunks x K candidates survive; their order does not matter
    if (pos < TOPK_MAXK * TOPK_MAXK) { sv[pos] = cv[i]; si[pos] = my; }
  }
  __syncthreads();
  int ns = nsurv < TOPK_MAXK * TOPK_MAXK ? nsurv : TOPK_MAXK * TOPK_MAXK;
  for (int i = threadIdx.x; i < ns; i += blockDim.x) {
    int my = si[i];
    float v = sv[i];
    int rank = 0;
    for (int j = 0; j < ns; j++) rank += before(sv[j], si[j], v, my) ? 1 : 0;
    if (rank < K) { idx[(size_t)r * K + rank] = my; lp[(size_t)r * K + rank] = (v - mx) - lse; }
  }
}

size_t topk_scratch_bytes(int rows, int n, int K) {
  size_t nch = (size_t)(n + TOPK_CHUNK - 1) / TOPK_CHUNK;
  return (size_t)rows * nch * (2 + 2 * (size_t)K) * 4 + 256;
}

// scratch: topk_scratch_bytes(rows, n, K) bytes.  Returns the number of kernels launched.
int launch_topk2(const float *logits, const int32_t *src_row, int rows, int n, int K, int32_t *idx, float *lp, void *scratch,
                 cudaStream_t s) {
  int nch = (n + TOPK_CHUNK - 1) / TOPK_CHUNK;
  float *pmax = (float *)scratch;
  float *psum = pmax + (size_t)rows * nch;
  float *cval = psum + (size_t)rows * nch;
  int32_t *cidx = (int32_t *)(cval + (size_t)rows * nch * K);
  {
    // Launched without the programmatic-dependent-launch attribute: pre-launched under the LM-head GEMM, the
    // rows x nch small CTAs become resident wherever that kernel leaves room, packed onto a few SMs instead of spread
    // over all of them, and the pair ran 8 us slower per draft pass (measured on the 8B shapes).
    const bool pdl = tl_pdl;
    tl_pdl = false;
    launch_k(topk_partial_kernel, dim3(nch, rows), dim3(256), 0, s, logits, src_row, n, K, nch, pmax, psum, cval, cidx);
    tl_pdl = pdl;
  }
  size_t smem = (size_t)nch * K * 8 + (size_t)nch * 8;
  static SmemLimit limit;
  if (smem > 48 * 1024) limit.ensure(topk_merge_kernel, (int)smem);
  launch_k(topk_merge_kernel, dim3(rows), dim3(256), smem, s, src_row, K, nch, pmax, psum, cval, cidx, idx, lp);
  return 2;
}

// ---------------------------------------------------------------- argmax over per-tile candidates
// y[r] = index of the best (value desc, index asc) of best_val/best_idx[t][r], t < tiles.
__global__ void __launch_bounds__(256) argmax_merge_kernel(const float *__restrict__ best_val, const int32_t *__restrict__ best_idx,
                                                           int tiles, int ld, int32_t *__restrict__ out) {
  pdl_wait();
  pdl_trigger();
  __shared__ VI sh[32];
  int r = blockIdx.x;
  VI b{0.0f, -1};
#pragma unroll 4
  for (int t = threadIdx.x; t < tiles; t += blockDim.x) {    // the loads of four rounds in flight
    float v = best_val[(size_t)t * ld + r];
    int i = best_idx[(size_t)t * ld + r];
    if (i >= 0 && (b.i < 0 || before(v, i, b.v, b.i))) { b.v = v; b.i = i; }
  }
  b = block_best(b, sh);
  if (threadIdx.x == 0) out[r] = b.i;
}
void launch_argmax_merge(const float *best_val, const int32_t *best_idx, int tiles, int ld, int rows, int32_t *out, cudaStream_t s) {
  launch_k(argmax_merge_kernel, dim3(rows), dim3(256), 0, s, best_val, best_idx, tiles, ld, out);
}

__device__ __forceinline__ int block_sum_int(int v) {
  __shared__ int acc;
  if (threadIdx.x == 0) acc = 0;
  __syncthreads();
  if (v) atomicAdd(&acc, v);
  __syncthreads();
  return acc;
}

// ---------------------------------------------------------------- step set-up: rows of the extend pass
// Row b*Pmax + j is pending entry j of sequence b: position n-P+j, causal among the pending rows.
__global__ void prep_extend_kernel(SeqState st, TreeBufs tb, RowMeta m, int need_positions, int32_t *status) {
  pdl_wait();
  pdl_trigger();
  int b = blockIdx.x, j = threadIdx.x;
  int n = st.n[b], P = st.P[b];
  bool ok = (n + need_positions <= st.cap[b]) && P >= 1 && P <= tb.Pmax;
  // rank of this sequence by (length desc, index asc): longest sequences get their attention CTAs first, which
  // packs CTAs of unequal length into fewer waves
  int longer = 0;
  for (int o = j; o < (int)gridDim.x; o += blockDim.x) {
    int no = st.n[o];
    longer += (no > n || (no == n && o < b)) ? 1 : 0;
  }
  longer = block_sum_int(longer);
  if (j == 0) {
    st.order[longer] = b;
    st.active[b] = ok ? 1 : 0;
    st.last_row[b] = ok ? b * tb.Pmax + P - 1 : -1;
    if (!ok) set_status(status, ST_CAPACITY, 10, b, n);
    tb.frontier[(size_t)b * tb.D * tb.K] = 0;
    tb.pool_tok[(size_t)b * (tb.pool + 1)] = st.root[b];
    tb.pool_parent[(size_t)b * (tb.pool + 1)] = -1;
    tb.pool_depth[(size_t)b * (tb.pool + 1)] = 0;
    tb.pool_score[(size_t)b * (tb.pool + 1)] = 0.0f;
  }
  if (j >= tb.Pmax) return;
  int r = b * tb.Pmax + j;
  bool valid = ok && j < P;
  m.seq[r] = valid ? b : -1;
  m.pos[r] = valid ? n - P + j : 0;
  m.kvpos[r] = valid ? n - P + j : 0;
  m.ctx[r] = valid ? n - P : 0;
  m.tail_base[r] = valid ? n - P : 0;
  m.mask_lo[r] = valid ? ((j >= 63) ? ~0ull : ((1ull << (j + 1)) - 1ull)) : 0ull;
  m.mask_hi[r] = 0ull;
  m.tok[r] = valid ? tb.pend_tok[b * tb.Pmax + j] : 0;
}
void launch_prep_extend(SeqState st, TreeBufs tb, RowMeta m, int B, int need_positions, int32_t *status, cudaStream_t s) {
  int threads = ((tb.Pmax + 31) / 32) * 32;
  launch_k(prep_extend_kernel, dim3(B), dim3(threads), 0, s, st, tb, m, need_positions, status);
}

// ---------------------------------------------------------------- dynamic-tree expansion after draft pass `pass` (1-based)
// Adds this pass's children to the pool (cumulative log-prob scores), picks the next frontier (the K
// best of the level) and writes the row metadata of the next draft pass.
__global__ void __launch_bounds__(256) expand_kernel(SeqState st, TreeBufs tb, RowMeta m, const int32_t *__restrict__ d2t,
                                                     int pass) {
  pdl_wait();
  pdl_trigger();
  extern __shared__ unsigned char smraw[];
  int K = tb.K, D = tb.D, b = blockIdx.x;
  int nch = (pass == 1) ? K : K * K;        // children created by this pass
  float *cs = (float *)smraw;               // [nch] child scores
  uint64_t *pm_lo = (uint64_t *)(cs + ((nch + 1) & ~1));   // [K] parent masks
  uint64_t *pm_hi = pm_lo + K;
  int32_t *newf = (int32_t *)(pm_hi + K);   // [K] local child index of the new frontier
  int32_t *ctok = newf + K;                 // [nch] child tokens (target ids)
  // every load that does not depend on another is issued up front: the kernel is a chain of L2 round trips otherwise
  const int active = st.active[b], n = st.n[b], last_row = st.last_row[b];
  if (!active) {   // skipped sequence: its rows of the next pass are padding
    for (int rr = threadIdx.x; rr < K; rr += blockDim.x) { m.seq[b * K + rr] = -1; m.tok[b * K + rr] = 0; m.pos[b * K + rr] = 0; }
    return;
  }
  size_t pb = (size_t)b * (tb.pool + 1);
  int base = (pass == 1) ? 0 : K + (pass - 2) * K * K;     // pool index of child 0 is base + 1
  for (int r = threadIdx.x; r < K; r += blockDim.x) {
    pm_lo[r] = (pass == 1) ? 0ull : m.mask_lo[b * K + r];
    pm_hi[r] = (pass == 1) ? 0ull : m.mask_hi[b * K + r];
    newf[r] = r;                            // where scores are NaN the ranks below leave places out
  }
  for (int c = threadIdx.x; c < nch; c += blockDim.x) {
    int r = (pass == 1) ? 0 : c / K, cc = (pass == 1) ? c : c % K;
    int row = (pass == 1) ? b : b * K + r;                  // row of the top-k output
    int u = (pass == 1) ? 0 : tb.front_cur[b * K + r];
    const float lp = tb.tk_lp[(size_t)row * K + cc];
    const int tokid = d2t[tb.tk_idx[(size_t)row * K + cc]];
    float sc = tb.pool_score[pb + u] + lp;
    int ci = base + c + 1;
    tb.pool_tok[pb + ci] = tokid;
    ctok[c] = tokid;
    tb.pool_parent[pb + ci] = u;
    tb.pool_depth[pb + ci] = pass;
    tb.pool_score[pb + ci] = sc;
    cs[c] = sc;
  }
  __syncthreads();
  if (pass >= D) return;
  // next frontier: rank by (score desc, pool index asc)
  for (int c = threadIdx.x; c < nch; c += blockDim.x) {
    float s = cs[c];
    int rank = 0;
    for (int j = 0; j < nch; j++) rank += (cs[j] > s || (cs[j] == s && j < c)) ? 1 : 0;
    if (rank < K) newf[rank] = c;
  }
  __syncthreads();
  for (int rr = threadIdx.x; rr < K; rr += blockDim.x) {
    int c = newf[rr];
    int ci = base + c + 1;
    int pr = (pass == 1) ? 0 : c / K;                       // parent's rank in the current pass
    int row = b * K + rr;
    int slot = (pass - 1) * K + rr;
    tb.front_cur[b * K + rr] = ci;
    tb.frontier[((size_t)b * D + pass) * K + rr] = ci;
    tb.feat_row[row] = (pass == 1) ? last_row : b * K + pr;
    uint64_t lo = pm_lo[pr], hi = pm_hi[pr];
    if (slot < 64) lo |= 1ull << slot; else hi |= 1ull << (slot - 64);
    m.seq[row] = b;
    m.pos[row] = n + pass - 1;
    m.kvpos[row] = n + slot;
    m.ctx[row] = n;
    m.tail_base[row] = n;
    m.mask_lo[row] = lo;
    m.mask_hi[row] = hi;
    m.tok[row] = ctok[c];
  }
}
void launch_expand(SeqState st, TreeBufs tb, RowMeta m, const int32_t *d2t, int pass, int B, cudaStream_t s) {
  int K = tb.K, nch = K * K;
  size_t smem = (size_t)((nch + 1) & ~1) * 4 + (size_t)K * 16 + (size_t)K * 4 + (size_t)nch * 4 + 16;
  launch_k(expand_kernel, dim3(B), dim3(256), smem, s, st, tb, m, d2t, pass);
}

// One warp merges the per-tile candidates of one row (the draft LM head's epilogue left, per 128-logit tile, the tile
// maximum, the sum of exp relative to it and the tile's K best logits, best first): the row's log-sum-exp and its K best
// (value desc, index asc) as log-probabilities.  Layout: candidates [row][ld][K], statistics [row][ld]; tiles <= 256, K <= 15.
//
// Only the K tiles with the best heads can hold one of the K best candidates: every candidate of another tile comes behind
// its own head, hence behind K better heads (tiles hold ascending index ranges, so the order of equal heads is the order of
// the tiles).  So the warp first picks K tiles from the statistics it has in registers anyway and then fetches those K * K
// candidates, one tile per lane.  Both selections bound the K-th best from below (by the K-th largest lane maximum, by the least
// of the K heads), collect the few entries that reach the bound and rank them by counting; with more than 32 of them (many equal
// values), or fewer than K lists, the best is picked K times by warp-wide reductions.
// tgt (may be null): d2t, whose values for the winners go to out_tok; they are asked for before the ranking.
constexpr int MERGE_SCRATCH = 32 + 64 + 16;              // words of shared memory a warp needs: lane maxima, (key, id) entries, tiles
__device__ __forceinline__ void merge_tile_candidates(const float *__restrict__ cand_val, const int32_t *__restrict__ cand_idx,
                                                      const float *__restrict__ cand_max, const float *__restrict__ cand_sum,
                                                      int tiles, int ld, int row, int K, int32_t *out_id, float *out_lp,
                                                      const int32_t *__restrict__ tgt, int32_t *out_tok, unsigned *scratch) {
  const int lane = threadIdx.x & 31;
  unsigned *s_max = scratch;
  uint2 *s_ent = (uint2 *)(scratch + 32);
  int *s_sel = (int *)(scratch + 96);
  float pm[8], ps[8];                                    // at most 8 tiles per lane, all loads issued before the first use
  int head[8];                                           // K = 1: the tiles' best are all the candidates there are (one load less to wait for)
#pragma unroll
  for (int j = 0; j < 8; j++) {
    const int t = lane + 32 * j;
    head[j] = (K == 1 && t < tiles) ? cand_idx[(size_t)row * ld + t] : -1;
    pm[j] = t < tiles ? cand_max[(size_t)row * ld + t] : -INFINITY;
    ps[j] = t < tiles ? cand_sum[(size_t)row * ld + t] : 0.0f;
  }
  float mx = -INFINITY;
#pragma unroll
  for (int j = 0; j < 8; j++) mx = fmaxf(mx, pm[j]);
  for (int off = 16; off > 0; off >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, off));
  unsigned key[8];
#pragma unroll
  for (int j = 0; j < 8; j++) key[j] = lane + 32 * j < tiles ? ordered_key(pm[j]) : 0u;      // keys of values are >= 1
  // entries (key >= bound) of this lane join the list, in any order; returns how many the warp has (those past 32 are not stored)
  int cnt = 0;
  auto collect = [&](bool in, unsigned k, int id) {
    const unsigned m = __ballot_sync(0xffffffffu, in);
    const int at = cnt + __popc(m & ((1u << lane) - 1u));
    if (in && at < 32) s_ent[at] = make_uint2(k, (unsigned)id);
    cnt += __popc(m);
  };
  auto rank_of = [&](uint2 me) {                         // (key desc, id asc) among the cnt <= 32 entries
    int rank = 0;
#pragma unroll 4
    for (int i = 0; i < cnt; i++) { const uint2 w = s_ent[i]; rank += w.x > me.x || (w.x == me.x && w.y < me.y); }
    return rank;
  };
  unsigned ck[15];
  int ci[15];
  const int nsel = K < tiles ? K : tiles;
  if (K == 1) {                                          // each lane's best head, by (value desc, tile asc)
#pragma unroll
    for (int i = 0; i < 15; i++) { ck[i] = 0u; ci[i] = -1; }
#pragma unroll
    for (int j = 0; j < 8; j++)
      if (head[j] >= 0 && key[j] > ck[0]) { ck[0] = key[j]; ci[0] = head[j]; }
  } else {
    // ---- the K best tiles, (head desc, tile asc): lane c keeps the c-th
    unsigned lm = 0u;
#pragma unroll
    for (int j = 0; j < 8; j++) lm = max(lm, key[j]);
    s_max[lane] = lm;
    __syncwarp();
    int above = 0;                                       // lanes with a larger maximum
#pragma unroll
    for (int i = 0; i < 32; i += 4) { const uint4 w = *(const uint4 *)(s_max + i); above += (w.x > lm) + (w.y > lm) + (w.z > lm) + (w.w > lm); }
    const unsigned bound = __reduce_min_sync(0xffffffffu, above < K && lm > 0u ? lm : 0xffffffffu);
#pragma unroll
    for (int j = 0; j < 8; j++) collect(key[j] >= bound, key[j], lane + 32 * j);
    __syncwarp();
    int sel = 0;
    if (cnt <= 32) {
      if (lane < cnt) {
        const uint2 me = s_ent[lane];
        const int rank = rank_of(me);
        if (rank < nsel) s_sel[rank] = (int)me.y;
      }
      __syncwarp();
      if (lane < nsel) sel = s_sel[lane];
    } else {
      for (int c = 0; c < nsel; c++) {
        unsigned bk = 0u, wk;
        int bt = -1;
#pragma unroll
        for (int j = 0; j < 8; j++)
          if (key[j] > bk) { bk = key[j]; bt = lane + 32 * j; }
        const int w = warp_best(bk, bt, &wk);
        if (lane == c) sel = w;
#pragma unroll
        for (int j = 0; j < 8; j++)
          if (lane + 32 * j == w) key[j] = 0u;
      }
    }
    // ---- lane c holds the c-th tile's candidates, best first
#pragma unroll
    for (int i = 0; i < 15; i++) {
      const bool have = lane < nsel && i < K;
      const size_t at = ((size_t)row * ld + sel) * K + i;
      ci[i] = have ? cand_idx[at] : -1;
      ck[i] = have ? ordered_key(cand_val[at]) : 0u;
    }
  }
  // the log-sum-exp while they are on their way: a lane adds its tiles in tile order, then a fixed shuffle tree
  float sum = 0.0f;
#pragma unroll
  for (int j = 0; j < 8; j++) sum += (lane + 32 * j < tiles) ? ps[j] * expf(pm[j] - mx) : 0.0f;
  for (int off = 16; off > 0; off >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, off);
  const float lse = logf(sum);
  // ---- the K best of the lists
  cnt = 33;
  if (K > 1 && nsel == K) {
    __syncwarp();                                        // the tiles' entries have been read
    cnt = 0;
    const unsigned bound = __reduce_min_sync(0xffffffffu, lane < K ? ck[0] : 0xffffffffu);      // K heads reach it
#pragma unroll
    for (int i = 0; i < 15; i++)
      if (i < K) collect(ci[i] >= 0 && ck[i] >= bound, ck[i], ci[i]);
    __syncwarp();
  }
  if (cnt >= K && cnt <= 32) {
    if (lane < cnt) {
      const uint2 me = s_ent[lane];
      const int tok = tgt ? tgt[me.y] : 0;
      const int rank = rank_of(me);
      if (rank < K) {
        out_id[rank] = (int)me.y;
        out_lp[rank] = (key_value(me.x) - mx) - lse;
        if (tgt) out_tok[rank] = tok;
      }
    }
  } else {
    // only the lists' heads compete, and the winner's list moves up
    for (int c = 0; c < K; c++) {
      unsigned wk;
      const int wi = warp_best(ck[0], ci[0], &wk);       // two redux instructions instead of a shuffle tree
      const bool won = wi >= 0 && ci[0] == wi;           // indices are unique: one lane at most
#pragma unroll
      for (int i = 0; i < 14; i++) { ck[i] = won ? ck[i + 1] : ck[i]; ci[i] = won ? ci[i + 1] : ci[i]; }
      if (won) ci[14] = -1;
      if (lane == 0) {
        out_id[c] = wi < 0 ? 0 : wi;
        out_lp[c] = wi < 0 ? 0.0f : (key_value(wk) - mx) - lse;
        if (tgt) out_tok[c] = tgt[wi < 0 ? 0 : wi];
      }
    }
  }
  __syncwarp();
}

// The merge alone, one warp per row (per-kernel parity tests of the LM-head epilogue + merge).
__global__ void __launch_bounds__(256) merge_candidates_kernel(const float *cand_val, const int32_t *cand_idx, const float *cand_max,
                                                               const float *cand_sum, int tiles, int ld, int rows, int K,
                                                               int32_t *__restrict__ idx, float *__restrict__ lp) {
  pdl_wait();
  pdl_trigger();
  __shared__ __align__(16) unsigned scratch[8][MERGE_SCRATCH];
  const int warp = threadIdx.x >> 5, row = blockIdx.x * 8 + warp;
  if (row >= rows) return;
  merge_tile_candidates(cand_val, cand_idx, cand_max, cand_sum, tiles, ld, row, K, idx + (size_t)row * K, lp + (size_t)row * K, nullptr, nullptr, scratch[warp]);
}
int launch_merge_candidates(const float *cand_val, const int32_t *cand_idx, const float *cand_max, const float *cand_sum, int tiles,
                            int ld, int rows, int K, int32_t *idx, float *lp, cudaStream_t s) {
  if (!draft_tree_step_fits(tiles, K) || ld != draft_tree_cand_ld(tiles)) return -1;
  launch_k(merge_candidates_kernel, dim3((rows + 7) / 8), dim3(256), 0, s, cand_val, cand_idx, cand_max, cand_sum, tiles, ld, rows, K, idx, lp);
  return 0;
}

// ---------------------------------------------------------------- one launch between two draft passes
// After the draft LM head of pass `pass` (whose epilogue left, per 128-logit tile and row, the tile maximum, the sum of
// exp relative to it and the tile's K best logits): merges the tiles into each row's log-softmax top-K, adds the children
// to the candidate pool with cumulative log-probability scores, picks the next frontier, writes the next pass's row
// metadata, and builds that pass's inputs (the FC2 input [feature ; embedding] of every frontier node and its RoPE
// angles).  Section 2.2 (dynamic draft tree: expansion by the draft's confidence), Section 3.1 (the draft's own output
// is the feature of the next step), Appendix A (nodes per expansion).
//
// grid (B, Z): the Z CTAs of a sequence each redo the small merge + expansion (same inputs, same order of operations,
// hence identical results) and then take one Z-th of the elements of the next pass's inputs; only CTA z = 0 writes the
// tree state.  Nothing a CTA reads is written by another CTA of the launch.
struct TreeStepArgs {
  SeqState st; TreeBufs tb; RowMeta m;
  const int32_t *d2t;
  int pass;                       // 1-based draft pass that just ran
  const float *cand_val, *cand_max, *cand_sum; const int32_t *cand_idx; int tiles, ld;   // [rows][ld][K], [rows][ld]
  const float *x; const bf16 *embed; bf16 *cat; int k;                                    // next pass's FC2 input
  const double *inv_freq; float2 *cs; int half;                                           // next pass's RoPE angles
  int compact;                    // pass 1: candidates and features are in row b (else in row last_row[b])
};

constexpr int TREE_WARPS = 10;   // one warp per row of a top-10 level
constexpr int TREE_ANGLE_WARPS = 2, TREE_THREADS = (TREE_WARPS + TREE_ANGLE_WARPS) * 32;
__global__ void __launch_bounds__(TREE_THREADS) draft_tree_step_kernel(const TreeStepArgs a) {
  pdl_wait();
  pdl_trigger();
  extern __shared__ __align__(16) unsigned char smraw[];
  const TreeBufs &tb = a.tb;
  const int K = tb.K, D = tb.D, b = blockIdx.x, pass = a.pass;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nrows = (pass == 1) ? 1 : K;                 // rows of this sequence in the pass that just ran
  const int nchild = nrows * K;
  const int nchild4 = (nchild + 3) & ~3;
  unsigned *scratch = (unsigned *)smraw;                 // [TREE_WARPS][MERGE_SCRATCH]
  uint64_t *par_mask = (uint64_t *)(scratch + TREE_WARPS * MERGE_SCRATCH);   // [K][2] ancestor masks of this pass's rows
  float *cscore = (float *)(par_mask + 2 * K);           // [nchild], padded to whole float4s with -inf
  float *tk_lp = cscore + ((K * K + 3) & ~3);            // [nrows][K]
  int32_t *tk_id = (int32_t *)(tk_lp + K * K);           // [nrows][K] draft ids
  int32_t *ctok = tk_id + K * K;                         // [nchild] target ids
  int32_t *newf = ctok + K * K;                          // [K] child index (within the level) of the new frontier
  int32_t *par_u = newf + K;                             // [K] pool index of the node each row of this pass processed
  float *par_sc = (float *)(par_u + K);                  // [K] its score
  // What follows is a chain of round trips to L2 that nothing hides; everything that does not depend on another load is asked for
  // at once: the sequence's state, the parents and their masks, the tiles' statistics.
  const int active = a.st.active[b], n = a.st.n[b];
  const int src1 = pass > 1 || a.compact ? b : a.st.last_row[b];     // pass 1: the row that holds the last pending entry's outputs
  const size_t pb = (size_t)b * (tb.pool + 1);
  const int base = (pass == 1) ? 0 : K + (pass - 2) * K * K;       // pool index of child 0 is base + 1
  const bool writer = blockIdx.y == 0;
  // the parents of this pass's rows (two dependent loads)
  if ((int)threadIdx.x < nrows) {
    const int u = (pass == 1) ? 0 : tb.frontier[((size_t)b * D + pass - 1) * K + threadIdx.x];
    const bool masks = writer && pass > 1;                // the writer replaces them below, and it alone reads them
    const uint64_t lo = masks ? a.m.mask_lo[b * K + threadIdx.x] : 0ull, hi = masks ? a.m.mask_hi[b * K + threadIdx.x] : 0ull;
    par_u[threadIdx.x] = u;
    par_sc[threadIdx.x] = tb.pool_score[pb + u];
    par_mask[2 * threadIdx.x] = lo; par_mask[2 * threadIdx.x + 1] = hi;
  }
  // ---- the RoPE angles of the next pass (one position for all rows; double precision, rounded once): two warps of their
  // own, while the others merge
  if (warp >= TREE_WARPS && pass < D && active) {
    for (int i = threadIdx.x - TREE_WARPS * 32; i < a.half; i += TREE_ANGLE_WARPS * 32) {
      double sn, cs_;
      sincos((double)(n + pass - 1) * a.inv_freq[i], &sn, &cs_);
      for (int rr = blockIdx.y; rr < K; rr += gridDim.y) a.cs[(size_t)(b * K + rr) * a.half + i] = make_float2((float)cs_, (float)sn);
    }
  }
  // ---- 1. per row: log-sum-exp over the tiles and the K best of the tiles' candidates (value desc, index asc).  (The rows of a
  // skipped sequence hold candidates too, of padding or of an earlier step; they are dropped below.)
  for (int r = warp; warp < TREE_WARPS && r < nrows; r += TREE_WARPS) {
    const int row = (pass == 1) ? max(src1, 0) : b * K + r;
    merge_tile_candidates(a.cand_val, a.cand_idx, a.cand_max, a.cand_sum, a.tiles, a.ld, row, K, tk_id + r * K, tk_lp + r * K, a.d2t, ctok + r * K, scratch + warp * MERGE_SCRATCH);
  }
  if (!active) {   // skipped sequence: its rows of the next pass are padding
    if (pass < D) {
      if (writer)
        for (int rr = threadIdx.x; rr < K; rr += blockDim.x) { a.m.seq[b * K + rr] = -1; a.m.tok[b * K + rr] = 0; a.m.pos[b * K + rr] = 0; }
      const size_t total = (size_t)K * 2 * a.k;
      for (size_t e = (size_t)blockIdx.y * blockDim.x + threadIdx.x; e < total; e += (size_t)gridDim.y * blockDim.x)
        a.cat[(size_t)b * K * 2 * a.k + e] = __float2bfloat16_rn(0.0f);
    }
    return;
  }
  __syncthreads();
  // ---- 2. children join the pool with cumulative scores
  for (int c = threadIdx.x; c < nchild; c += blockDim.x) {
    const int r = c / K;
    const int u = par_u[r];                                // the node row r processed
    const float sc = par_sc[r] + tk_lp[c];
    cscore[c] = sc;
    if (writer) {
      const int ci = base + c + 1;
      tb.pool_tok[pb + ci] = ctok[c];
      tb.pool_parent[pb + ci] = u;
      tb.pool_depth[pb + ci] = pass;
      tb.pool_score[pb + ci] = sc;
      // kept for inspection: the top-K of this pass in the layout of the per-row kernels
      const int row = (pass == 1) ? b : b * K + r;
      tb.tk_idx[(size_t)row * K + c - r * K] = tk_id[c];
      tb.tk_lp[(size_t)row * K + c - r * K] = tk_lp[c];
    }
  }
  if (pass >= D) return;
  if ((int)threadIdx.x < nchild4 - nchild) cscore[nchild + threadIdx.x] = -INFINITY;
  if ((int)threadIdx.x < K) newf[threadIdx.x] = threadIdx.x;           // where scores are NaN the ranks below leave places out
  __syncthreads();
  // ---- 3. next frontier: the K best children of the level, (score desc, pool index asc)
  for (int c = threadIdx.x; c < nchild; c += blockDim.x) {
    const float s = cscore[c];
    int rank = 0;
#pragma unroll 4
    for (int j = 0; j < nchild4; j += 4) {               // the padding never comes before a child
      const float4 o = *(const float4 *)(cscore + j);
      rank += (o.x > s || (o.x == s && j < c)) + (o.y > s || (o.y == s && j + 1 < c)) + (o.z > s || (o.z == s && j + 2 < c)) + (o.w > s || (o.w == s && j + 3 < c));
    }
    if (rank < K) newf[rank] = c;
  }
  __syncthreads();
  if (writer && (int)threadIdx.x < K) {
    const int rr = threadIdx.x, c = newf[rr];
    const int pr = c / K;                                  // parent's row in the pass that just ran (0 in pass 1)
    const int ci = base + c + 1, row = b * K + rr, slot = (pass - 1) * K + rr;
    uint64_t lo = par_mask[2 * pr], hi = par_mask[2 * pr + 1];
    if (slot < 64) lo |= 1ull << slot; else hi |= 1ull << (slot - 64);
    tb.front_cur[b * K + rr] = ci;
    tb.frontier[((size_t)b * D + pass) * K + rr] = ci;
    tb.feat_row[row] = (pass == 1) ? src1 : b * K + pr;
    a.m.seq[row] = b;
    a.m.pos[row] = n + pass - 1;
    a.m.kvpos[row] = n + slot;
    a.m.ctx[row] = n;
    a.m.tail_base[row] = n;
    a.m.mask_lo[row] = lo;
    a.m.mask_hi[row] = hi;
    a.m.tok[row] = ctok[c];
  }
  // ---- 4. inputs of the next pass: FC2 input [bf16(feature of the parent's row) ; embedding of the node's token], split
  // over the CTAs of the sequence
  const int k = a.k, vpr = 2 * k / 8;                      // 8-element vectors per row (hidden % 8 == 0)
  const int stride = gridDim.y * blockDim.x, total = K * vpr;
  constexpr int NV = 4;                                    // vectors of a thread whose loads are in flight together
  for (int e0 = blockIdx.y * blockDim.x + threadIdx.x; e0 < total; e0 += NV * stride) {
    uint4 v[NV][2];                                        // eight floats of the feature, or eight bf16 of the embedding
#pragma unroll
    for (int q = 0; q < NV; q++) {
      const int e = e0 + q * stride;
      if (e < total) {
        const int rr = e / vpr, i = (e % vpr) * 8, c = newf[rr];
        if (i < k) {
          const int fr = (pass == 1) ? src1 : b * K + c / K;
          v[q][0] = *(const uint4 *)(a.x + (size_t)fr * k + i); v[q][1] = *(const uint4 *)(a.x + (size_t)fr * k + i + 4);
        } else {
          v[q][0] = *(const uint4 *)(a.embed + (size_t)ctok[c] * k + (i - k));
        }
      }
    }
#pragma unroll
    for (int q = 0; q < NV; q++) {
      const int e = e0 + q * stride;
      if (e < total) {
        const int rr = e / vpr, i = (e % vpr) * 8;
        uint4 out = v[q][0];
        if (i < k) {
          __nv_bfloat162 p0 = __floats2bfloat162_rn(__uint_as_float(v[q][0].x), __uint_as_float(v[q][0].y)), p1 = __floats2bfloat162_rn(__uint_as_float(v[q][0].z), __uint_as_float(v[q][0].w));
          __nv_bfloat162 p2 = __floats2bfloat162_rn(__uint_as_float(v[q][1].x), __uint_as_float(v[q][1].y)), p3 = __floats2bfloat162_rn(__uint_as_float(v[q][1].z), __uint_as_float(v[q][1].w));
          out = make_uint4(*(uint32_t *)&p0, *(uint32_t *)&p1, *(uint32_t *)&p2, *(uint32_t *)&p3);
        }
        *(uint4 *)(a.cat + ((size_t)(b * K + rr)) * 2 * k + i) = out;
      }
    }
  }
}

// Shapes the kernel takes (the others use the separate kernels): at most eight tiles per lane and 15 candidates per tile in
// registers.  The kernel itself has no other limit.  The product of the two is the line between the calls that spec_gemm_topk
// takes and refuses; it dates from a form that staged the candidates of a level's ten rows in 220 KB of shared memory.
int draft_tree_cand_ld(int tiles) { return (tiles + 3) & ~3; }
bool draft_tree_step_fits(int tiles, int K) {
  if (tiles > 256 || K > 15) return false;
  return (size_t)TREE_WARPS * 2 * draft_tree_cand_ld(tiles) * K * 4 + (size_t)K * K * 16 + (size_t)K * 12 + 64 <= 220 * 1024;
}
int launch_draft_tree_step(SeqState st, TreeBufs tb, RowMeta m, const int32_t *d2t, int pass, const float *cand_val,
                           const int32_t *cand_idx, const float *cand_max, const float *cand_sum, int tiles, int ld, const float *x,
                           const bf16 *embed, bf16 *cat, int k, const double *inv_freq, float2 *cs, int half, int B, bool compact, cudaStream_t s) {
  if (!draft_tree_step_fits(tiles, tb.K) || ld != draft_tree_cand_ld(tiles) || (k % 8)) return -1;
  const size_t smem = (size_t)TREE_WARPS * MERGE_SCRATCH * 4 + (size_t)tb.K * 16 + (size_t)((tb.K * tb.K + 3) & ~3) * 4 + (size_t)tb.K * tb.K * 12 + (size_t)tb.K * 12;
  TreeStepArgs a{st, tb, m, d2t, pass, cand_val, cand_max, cand_sum, cand_idx, tiles, ld, x, embed, cat, k, inv_freq, cs, half, compact ? 1 : 0};
  const int Z = B >= 16 ? 1 : 8;        // CTAs per sequence that share the next pass's input assembly
  launch_k(draft_tree_step_kernel, dim3(B, Z), dim3(TREE_THREADS), smem, s, a);
  return 0;
}

// ---------------------------------------------------------------- the last pending entries of a batch, side by side
__global__ void __launch_bounds__(256) gather_pending_kernel(const int32_t *__restrict__ last_row, const uint4 *__restrict__ x, uint4 *__restrict__ cx,
                                                             int x_vecs, const uint4 *__restrict__ ao, uint4 *__restrict__ cao, int ao_vecs) {
  pdl_wait();
  pdl_trigger();
  const int b = blockIdx.x, r = last_row[b];
  const uint4 zero = make_uint4(0u, 0u, 0u, 0u);
  for (int i = threadIdx.x + blockIdx.y * blockDim.x; i < x_vecs; i += gridDim.y * blockDim.x) cx[(size_t)b * x_vecs + i] = r >= 0 ? x[(size_t)r * x_vecs + i] : zero;
  for (int i = threadIdx.x + blockIdx.y * blockDim.x; i < ao_vecs; i += gridDim.y * blockDim.x) cao[(size_t)b * ao_vecs + i] = r >= 0 ? ao[(size_t)r * ao_vecs + i] : zero;
}
void launch_gather_pending(const int32_t *last_row, const float *x, float *cx, int k, const bf16 *ao, bf16 *cao, int qd, int B, cudaStream_t s) {
  launch_k(gather_pending_kernel, dim3(B, 4), dim3(256), 0, s, last_row, (const uint4 *)x, (uint4 *)cx, k / 4, (const uint4 *)ao, (uint4 *)cao, qd / 8);
}

// ---------------------------------------------------------------- pruning + tree assembly
// Keeps the M = min(N-1, pool) best candidates (score desc, pool index asc), numbers them in pool
// order after the root and emits parents, depths, ancestor-or-self bit masks and the verify rows.
// One thread per pool entry (pool + 1 <= 1024): rank counting over four candidates per shared-memory load, numbering by
// warp ballots (with 256 threads, scalar loads and a counting loop per kept candidate: 17 us on the step's critical path).
__global__ void __launch_bounds__(1024) rerank_kernel(SeqState st, TreeBufs tb, RowMeta m) {
  pdl_wait();
  pdl_trigger();
  extern __shared__ __align__(16) unsigned char smraw[];
  __shared__ int warp_kept[32];
  const int b = blockIdx.x, pool = tb.pool, N = tb.N, pool4 = (pool + 3) & ~3;
  float *sc = (float *)smraw;                       // [pool4]: candidate i at i - 1, padded with -inf
  int32_t *node_of = (int32_t *)(sc + pool4);       // [pool+1], -1 = dropped
  int32_t *par = node_of + pool + 1;                // [pool+1]
  const int M = (N - 1 < pool) ? N - 1 : pool;
  const size_t pb = (size_t)b * (pool + 1);
  const int n = st.n[b];
  const bool act = st.active[b] != 0;
  const int i = threadIdx.x;
  float score = 0.0f;
  int parent = 0, depth = 0, tok = 0;
  if (i <= pool) {
    score = tb.pool_score[pb + i]; parent = tb.pool_parent[pb + i]; depth = tb.pool_depth[pb + i]; tok = tb.pool_tok[pb + i];
    if (i > 0) sc[i - 1] = score;
    par[i] = parent;
  }
  if (i < pool4 - pool) sc[pool + i] = -INFINITY;
  __syncthreads();
  bool kept = false;
  if (i >= 1 && i <= pool) {
    const int c = i - 1;
    int rank = 0;
    // equal scores: the lower index comes first.  Only around the warp's own candidates does that take a look at the index: those
    // before them come first if they are not smaller, those behind them if they are larger (half the instructions)
    const int c_lo = max((i & ~31) - 1, 0) & ~3, c_hi = min(((i | 31) + 3) & ~3, pool4);      // the warp's candidates are i - 1, in whole fours
#pragma unroll 4
    for (int j = 0; j < c_lo; j += 4) {
      const float4 o = *(const float4 *)(sc + j);
      rank += (o.x >= score) + (o.y >= score) + (o.z >= score) + (o.w >= score);
    }
#pragma unroll 4
    for (int j = c_lo; j < c_hi; j += 4) {          // the padding never comes before a candidate
      const float4 o = *(const float4 *)(sc + j);
      rank += (o.x > score || (o.x == score && j < c)) + (o.y > score || (o.y == score && j + 1 < c)) +
              (o.z > score || (o.z == score && j + 2 < c)) + (o.w > score || (o.w == score && j + 3 < c));
    }
#pragma unroll 4
    for (int j = c_hi; j < pool4; j += 4) {
      const float4 o = *(const float4 *)(sc + j);
      rank += (o.x > score) + (o.y > score) + (o.z > score) + (o.w > score);
    }
    kept = rank < M;
  }
  // number the kept candidates in pool order, after the root
  const unsigned ballot = __ballot_sync(0xffffffffu, kept);
  if ((i & 31) == 0) warp_kept[i >> 5] = __popc(ballot);
  __syncthreads();
  int ni = i == 0 ? 0 : -1;
  if (kept) {
    ni = 1 + __popc(ballot & ((1u << (i & 31)) - 1u));
    for (int w = 0; w < (i >> 5); w++) ni += warp_kept[w];
  }
  if (i <= pool) node_of[i] = ni;
  __syncthreads();
  if (i == 0) tb.nn[b] = act ? M + 1 : 0;
  if (ni >= 0 && ni < N) {
    uint64_t mask = 0;
    for (int v = i, it = 0; v >= 0 && v <= pool && it < 64; v = par[v], it++) mask |= 1ull << (node_of[v] & 63);
    const size_t t = (size_t)b * N + ni;
    tb.tok[t] = tok;
    tb.parent[t] = (i == 0) ? -1 : node_of[parent];
    tb.depth[t] = depth;
    tb.poolidx[t] = i;
    tb.score[t] = score;
    tb.mask[t] = mask;
    m.seq[t] = act ? b : -1;
    m.pos[t] = act ? n + depth : 0;
    m.kvpos[t] = act ? n + ni : 0;
    m.ctx[t] = act ? n : 0;
    m.tail_base[t] = act ? n : 0;
    m.mask_lo[t] = mask;
    m.mask_hi[t] = 0ull;
    m.tok[t] = act ? tok : 0;
  }
  // rows beyond the tree (only when pool < N-1) are padding
  for (int r = M + 1 + threadIdx.x; r < N; r += blockDim.x) {
    const size_t t = (size_t)b * N + r;
    m.seq[t] = -1; m.pos[t] = 0; m.kvpos[t] = 0; m.ctx[t] = 0; m.tail_base[t] = 0;
    m.mask_lo[t] = 0; m.mask_hi[t] = 0; m.tok[t] = 0;
  }
}
void launch_rerank(SeqState st, TreeBufs tb, RowMeta m, int B, cudaStream_t s) {
  const size_t smem = (size_t)((tb.pool + 3) & ~3) * 4 + (size_t)(tb.pool + 1) * 8;
  launch_k(rerank_kernel, dim3(B), dim3((tb.pool + 1 + 31) / 32 * 32), smem, s, st, tb, m);
}

// Tree of the root alone (plain autoregressive decoding on the same kernels): one row per sequence.
__global__ void plain_tree_kernel(SeqState st, TreeBufs tb, RowMeta m, int B) {
  pdl_wait();
  pdl_trigger();
  int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= B) return;
  int n = st.n[b];
  bool act = n + 1 <= st.cap[b];
  st.active[b] = act ? 1 : 0;
  tb.nn[b] = act ? 1 : 0;
  tb.tok[b] = st.root[b]; tb.parent[b] = -1; tb.depth[b] = 0; tb.poolidx[b] = 0; tb.score[b] = 0.0f; tb.mask[b] = 1ull;
  m.seq[b] = act ? b : -1; m.pos[b] = n; m.kvpos[b] = n; m.ctx[b] = n; m.tail_base[b] = n;
  m.mask_lo[b] = 1ull; m.mask_hi[b] = 0ull; m.tok[b] = act ? st.root[b] : 0;
}
void launch_plain_tree(SeqState st, TreeBufs tb, RowMeta m, int B, cudaStream_t s) {
  launch_k(plain_tree_kernel, dim3((B + 63) / 64), dim3(64), 0, s, st, tb, m, B);
}

// ---------------------------------------------------------------- greedy acceptance
// Follow, from the root, the child whose token equals the target's argmax at the current node.
// A thread per node looks whether it is the one its parent goes on to; the walk is then one step of shared memory per accepted node.
constexpr int ACCEPT_THREADS = 64;                           // nodes a tree can have
__global__ void __launch_bounds__(ACCEPT_THREADS) accept_kernel(SeqState st, TreeBufs tb, int rows_per_seq) {
  pdl_wait();
  pdl_trigger();
  __shared__ int32_t tok[64], y[64], next[64];
  const int b = blockIdx.x, i = threadIdx.x, Pmax = tb.Pmax;
  const size_t row0 = (size_t)b * rows_per_seq;
  // everything is asked for at once (rows_per_seq <= 64)
  const int nn = tb.nn[b], active = st.active[b], n = st.n[b];
  const bool row = i < rows_per_seq;
  const int t = row ? tb.tok[row0 + i] : 0, p = row ? tb.parent[row0 + i] : -1, best = row ? tb.y[row0 + i] : 0;
  tok[i] = t; y[i] = best; next[i] = 64;
  __syncthreads();
  if (i > 0 && i < nn && row && p >= 0 && p < i && t == y[p]) atomicMin(&next[p], i);      // the first child whose token the target would emit
  __syncthreads();
  if (i != 0) return;
  if (!active || nn < 1) { tb.out_cnt[b] = 0; return; }
  int cur = 0, a = 0;
  tb.path[b * Pmax] = 0;
  while (a + 1 < Pmax && next[cur] < 64) {
    cur = next[cur];
    tb.out_ids[b * Pmax + a] = tok[cur];
    tb.pend_tok[b * Pmax + a] = tok[cur];
    tb.path[b * Pmax + (++a)] = cur;
  }
  tb.out_ids[b * Pmax + a] = y[cur];
  tb.pend_tok[b * Pmax + a] = y[cur];
  for (int j = a + 1; j < Pmax; j++) tb.out_ids[b * Pmax + j] = -1;
  tb.out_cnt[b] = a + 1;
  st.n_prev[b] = n;
  st.n[b] = n + a + 1;
  st.P[b] = a + 1;
  st.root[b] = y[cur];
}
void launch_accept(SeqState st, TreeBufs tb, int B, int rows_per_seq, cudaStream_t s) {
  launch_k(accept_kernel, dim3(B), dim3(ACCEPT_THREADS), 0, s, st, tb, rows_per_seq);
}

// ---------------------------------------------------------------- stochastic acceptance (temperature > 0)
// Section 2.1's rule on the deterministic top-K tree: child c of the current node is accepted with probability
// p(tok[c]) under what is left of softmax(z / T) after its rejected elder siblings were removed; when no child is
// left the token is drawn from the residual by inverse CDF over increasing ids.  The uniforms are inputs:
// u[b][c] decides node c, u[b][N + cur] draws the final token at node cur.  One CTA per sequence; every reduction
// has a fixed order, so a step is reproducible on this kernel.
constexpr int ACC_THREADS = 1024;
constexpr int ACC_MAX_REJ = 64;
constexpr float ACC_LEAST = 1e-30f;      // of the row's mass, below which a run of ids counts as empty: its terms may be 0 one by one

// exp on the special-function unit (ex2.approx), relative error ~1e-6 near the maximum, far inside the parity slack.  A term of a
// row's mass is the product of two, of its distance to its run's maximum and of the run's to the row's.
__device__ __forceinline__ float acc_exp(float x) { return __expf(x); }

// Masses of the verify rows: per run of MASS_CHUNK ids the largest logit and sum exp((z - largest) / T), [row][chunk].  The acceptance walks one
// node after the other on one SM, which reads a row of 128256 logits in 7 us: three times a visited node, that was most of the launch.
// Here the whole chip reads all rows once, and the walk needs a few numbers a node.  Sampled step of the 8B shapes over a greedy one, 6.2
// nodes visited: 145 -> 65 us (of which the logits' way to memory, the uniforms' copy and the host take 40).
constexpr int MASS_CHUNK = 8192;
int accept_mass_chunks(int V) { return (int)(((long long)V + MASS_CHUNK - 1) / MASS_CHUNK); }
bool accept_sampled_takes(int V) { return accept_mass_chunks(V) <= MASS_CHUNK; }      // the walk holds a row's masses in the place of a run's terms
// grid (rows, chunks): there are up to 4096 x 64 rows, and a grid's second index ends at 65535
__global__ void __launch_bounds__(256) row_mass_kernel(const float *__restrict__ logits, int V, const float *__restrict__ inv_temp, float2 *__restrict__ part) {
  pdl_wait();
  pdl_trigger();
  __shared__ float red[2][8];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int v0 = blockIdx.y * MASS_CHUNK, n = min(MASS_CHUNK, V - v0);
  const float *z = logits + (size_t)blockIdx.x * V + v0;
  const float inv_T = *inv_temp;
  constexpr int PER = MASS_CHUNK / 256;
  float v[PER];
  if ((V & 3) == 0) {                                        // rows are then 16-byte aligned
#pragma unroll
    for (int j = 0; j < PER / 4; j++) {
      const int i = 4 * (threadIdx.x + j * 256);
      const float4 q = i < n ? *(const float4 *)(z + i) : make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
      v[4 * j] = q.x; v[4 * j + 1] = q.y; v[4 * j + 2] = q.z; v[4 * j + 3] = q.w;
    }
  } else {
#pragma unroll
    for (int j = 0; j < PER; j++) { const int i = threadIdx.x + j * 256; v[j] = i < n ? z[i] : -INFINITY; }
  }
  float m = -INFINITY;
#pragma unroll
  for (int j = 0; j < PER; j++) m = fmaxf(m, v[j]);
  for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  if (lane == 0) red[0][warp] = m;
  __syncthreads();
  m = red[0][0];
#pragma unroll
  for (int w = 1; w < 8; w++) m = fmaxf(m, red[0][w]);
  float sum = 0.0f;
  if (m > -INFINITY) {
#pragma unroll
    for (int j = 0; j < PER; j++) sum += acc_exp((v[j] - m) * inv_T);      // exp(-inf) = 0 past the end
  }
  for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
  if (lane == 0) red[1][warp] = sum;
  __syncthreads();
  if (threadIdx.x == 0) {
    sum = red[1][0];
#pragma unroll
    for (int w = 1; w < 8; w++) sum += red[1][w];
    part[(size_t)blockIdx.x * gridDim.y + blockIdx.y] = make_float2(m, sum);
  }
}

__global__ void __launch_bounds__(ACC_THREADS) accept_sampled_kernel(SeqState st, TreeBufs tb, const float *__restrict__ logits,
                                                                     int V, const float *__restrict__ u, const float2 *__restrict__ mass_part, int chunks,
                                                                     int rows_per_seq) {
  pdl_wait();
  pdl_trigger();
  constexpr int NWARP = ACC_THREADS / 32;
  __shared__ float seg[MASS_CHUNK];                          // residual terms of the chunk that holds the drawn token
  __shared__ float part[NWARP];
  __shared__ int32_t rej[ACC_MAX_REJ];
  __shared__ float rej_e[ACC_MAX_REJ];
  __shared__ int again[ACC_MAX_REJ];                         // chunks whose residual is added up again
  __shared__ int s_cur, s_len, s_nrej, s_pick, s_owner, s_again;
  __shared__ float s_target;
  __shared__ int32_t tok[64];
  __shared__ float ub[128], zc[64], zmax_s[64], mass_s[64];
  __shared__ unsigned long long kids[64];                    // children of a node, in node order
  const int b = blockIdx.x, tid = threadIdx.x, wid = tid >> 5, ln = tid & 31;
  const int Pmax = tb.Pmax, N = tb.N;
  const int nn = min(tb.nn[b], 64);
  if (!st.active[b] || nn < 1) {
    if (tid == 0) tb.out_cnt[b] = 0;
    return;
  }
  if (tid < 64) kids[tid] = 0ull;
  __syncthreads();
  // ---- the tree, the uniforms, the nodes' masses and their tokens' logits go to shared memory at once: the walk below is serial
  const size_t row0 = (size_t)b * rows_per_seq;
  if (tid < 2 * N && tid < 128) ub[tid] = u[(size_t)b * 2 * N + tid];
  const float inv_T = u[(size_t)gridDim.x * 2 * N];          // 1 / temperature follows the uniforms
  if (tid < nn) {
    const int t = tb.tok[row0 + tid], p = tb.parent[row0 + tid];
    tok[tid] = t;
    if (tid > 0) { zc[tid] = logits[(row0 + p) * V + t]; atomicOr(&kids[p], 1ull << tid); }
  }
  for (int node = wid; node < nn; node += NWARP) {           // a warp per node, a lane per chunk
    const float2 *mp = mass_part + (row0 + node) * chunks;
    float m = -INFINITY, sum = 0.0f;
    for (int c = ln; c < chunks; c += 32) m = fmaxf(m, mp[c].x);
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    for (int c = ln; c < chunks; c += 32) sum += mp[c].y > 0.0f ? mp[c].y * acc_exp((mp[c].x - m) * inv_T) : 0.0f;
    for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    if (ln == 0) { zmax_s[node] = m; mass_s[node] = sum; }
  }
  __syncthreads();
  // ---- the walk, by one thread: the children of the current node in node order
  if (tid == 0) {
    int cur = 0, a = 0, nrej;
    tb.path[b * Pmax] = 0;
    for (;;) {
      int nxt = -1;
      float mass = mass_s[cur];
      nrej = 0;
      if (a + 1 < Pmax) {
        for (unsigned long long left = kids[cur]; left && nxt < 0; left &= left - 1) {
          const int c = __ffsll(left) - 1;
          const float e = acc_exp((zc[c] - zmax_s[cur]) * inv_T);
          const float pc = mass > 0.0f ? e / mass : 0.0f;
          if (ub[c] < pc) nxt = c;
          else { mass -= e; if (nrej < ACC_MAX_REJ) { rej[nrej] = tok[c]; rej_e[nrej++] = e; } }
        }
      }
      if (nxt < 0) break;
      tb.out_ids[b * Pmax + a] = tok[nxt];
      tb.pend_tok[b * Pmax + a] = tok[nxt];
      tb.path[b * Pmax + a + 1] = nxt;
      cur = nxt;
      a++;
    }
    s_cur = cur; s_len = a; s_nrej = nrej; s_again = 0;
  }
  __syncthreads();
  const int cur = s_cur, a = s_len, nrej = s_nrej;
  const float *z = logits + (row0 + cur) * V;
  const float zmax = zmax_s[cur];
  // ---- the final token: inverse CDF over the residual, in three levels.  One thread finds the chunk that holds the target, the chunk's
  // terms go to shared memory, one thread finds the warp whose 32nd of them holds what is left of it, and that warp walks its range 32 ids at a
  // time with a warp prefix sum.
  // The residual of a chunk is its mass without the rejected tokens'.  Where they are more than half of it, the difference has lost bits,
  // up to all of them, and what is left is added up again from its terms.
  auto residual = [&](int id) {                              // term of an id, 0 for a rejected one
    float e = acc_exp((z[id] - zmax) * inv_T);
    for (int r = 0; r < nrej; r++)
      if (rej[r] == id) e = 0.0f;
    return e;
  };
  for (int c = tid; c < chunks; c += ACC_THREADS) {          // masses of the chunks (at most MASS_CHUNK of them), without the rejected tokens
    const float2 mp = mass_part[(row0 + cur) * chunks + c];
    const float m = mp.y > 0.0f ? mp.y * acc_exp((mp.x - zmax) * inv_T) : 0.0f;
    float left = m;
    bool less = false;
    for (int r = 0; r < nrej; r++)
      if (rej[r] / MASS_CHUNK == c) { left -= rej_e[r]; less = true; }
    if (less && !(left >= 0.5f * m)) again[atomicAdd(&s_again, 1)] = c;      // one per rejected token at most
    seg[c] = left > ACC_LEAST ? left : 0.0f;
  }
  __syncthreads();
  for (int q = 0; q < s_again; q++) {
    const int c0 = again[q] * MASS_CHUNK, n = min(MASS_CHUNK, V - c0);
    float loc = 0.0f;
    for (int i = tid; i < n; i += ACC_THREADS) loc += residual(c0 + i);
    for (int o = 16; o > 0; o >>= 1) loc += __shfl_xor_sync(0xffffffffu, loc, o);
    if (ln == 0) part[wid] = loc;
    __syncthreads();
    if (tid == 0) {
      float m = 0.0f;
      for (int w = 0; w < NWARP; w++) m += part[w];
      seg[again[q]] = m > ACC_LEAST ? m : 0.0f;
    }
    __syncthreads();
  }
  if (tid == 0) {
    float total = 0.0f;
    for (int c = 0; c < chunks; c++) total += seg[c];
    const float target = ub[N + cur] * total;
    float cum = 0.0f, last_cum = 0.0f;
    int owner = -1, last = 0;
    for (int c = 0; c < chunks; c++) {
      const float m = seg[c];
      if (m > 0.0f) {
        last = c; last_cum = cum;
        if (cum + m > target) { owner = c; break; }
      }
      cum += m;
    }
    if (owner < 0) { owner = last; cum = last_cum; }           // rounding at the upper end: the last chunk with mass
    s_owner = owner; s_target = target - cum;
  }
  __syncthreads();
  const int c0 = s_owner * MASS_CHUNK, n = min(MASS_CHUNK, V - c0);
  const float in_chunk = s_target;
  for (int i = tid; i < n; i += ACC_THREADS) seg[i] = residual(c0 + i);
  __syncthreads();
  const int CW = (n + NWARP - 1) / NWARP, w0 = wid * CW, w1 = min(w0 + CW, n);
  float loc = 0.0f;
  for (int i = w0 + ln; i < w1; i += 32) loc += seg[i];
  for (int o = 16; o > 0; o >>= 1) loc += __shfl_xor_sync(0xffffffffu, loc, o);
  if (ln == 0) part[wid] = loc;
  __syncthreads();
  if (tid == 0) {
    float cum = 0.0f, last_cum = 0.0f;
    int owner = -1, last = 0;
    for (int w = 0; w < NWARP; w++) {
      if (part[w] > 0.0f) {
        last = w; last_cum = cum;
        if (cum + part[w] > in_chunk) { owner = w; break; }
      }
      cum += part[w];
    }
    if (owner < 0) { owner = last; cum = last_cum; }           // rounding: the last warp with mass
    s_owner = owner; s_target = in_chunk - cum; s_pick = 0;
  }
  __syncthreads();
  if (wid == s_owner) {
    const float target = s_target;
    float cum = 0.0f;
    int pick = -1, last = -1;
    for (int base = w0; base < w1 && pick < 0; base += 32) {
      const int i = base + ln;
      const float e = i < w1 ? seg[i] : 0.0f;
      float inc = e;                                         // inclusive prefix sum over the 32 lanes
      for (int o = 1; o < 32; o <<= 1) {
        const float t = __shfl_up_sync(0xffffffffu, inc, o);
        if (ln >= o) inc += t;
      }
      const bool hit = e > 0.0f && cum + inc > target;
      const unsigned hits = __ballot_sync(0xffffffffu, hit), alive = __ballot_sync(0xffffffffu, e > 0.0f);
      if (alive) last = base + 31 - __clz(alive);
      if (hits) pick = base + __ffs(hits) - 1;
      cum += __shfl_sync(0xffffffffu, inc, 31);
    }
    if (ln == 0) s_pick = c0 + (pick >= 0 ? pick : (last >= 0 ? last : w0));
  }
  __syncthreads();
  if (tid == 0) {
    const int bonus = s_pick;
    tb.out_ids[b * Pmax + a] = bonus;
    tb.pend_tok[b * Pmax + a] = bonus;
    for (int j = a + 1; j < Pmax; j++) tb.out_ids[b * Pmax + j] = -1;
    tb.out_cnt[b] = a + 1;
    const int n0 = st.n[b];
    st.n_prev[b] = n0;
    st.n[b] = n0 + a + 1;
    st.P[b] = a + 1;
    st.root[b] = bonus;
  }
}
int launch_accept_sampled(SeqState st, TreeBufs tb, const float *logits, int V, const float *u, float2 *mass_part, int B, int rows_per_seq, cudaStream_t s) {
  if (!accept_sampled_takes(V)) return -1;
  const int chunks = accept_mass_chunks(V);
  if (launch_k(row_mass_kernel, dim3(B * rows_per_seq, chunks), dim3(256), 0, s, logits, V, u + (size_t)B * 2 * tb.N, mass_part) != cudaSuccess) return -1;
  if (launch_k(accept_sampled_kernel, dim3(B), dim3(ACC_THREADS), 0, s, st, tb, logits, V, u, (const float2 *)mass_part, chunks, rows_per_seq) != cudaSuccess) return -1;
  return 2;
}

// ---------------------------------------------------------------- commit: KV compaction + tap gather
// Accepted node path[j] (K/V at cache position n+path[j]) moves to position n+j in every layer; its
// taps become pending entry j.  path[j] >= j and is increasing, and a thread copies the same element
// offsets for every j, so the in-place move in increasing j never reads an overwritten slot.
template <typename T>
__global__ void __launch_bounds__(256) commit_kernel(SeqState st, TreeBufs tb, const KvPool *__restrict__ pools,
                                                     PageMap pm, const T *__restrict__ node_taps,
                                                     T *__restrict__ pend_taps, int L, int G, int hd, int k,
                                                     int rows_per_seq) {
  pdl_wait();
  pdl_trigger();
  int b = blockIdx.x, l = blockIdx.y;
  int cnt = tb.out_cnt[b];
  if (cnt <= 0) return;
  int n0 = st.n_prev[b], Pmax = tb.Pmax;
  constexpr int VEC = 16 / (int)sizeof(T);           // elements per 16-byte vector (head_dim is a multiple of 16)
  constexpr int JB = 8;                              // accepted nodes moved per batch
  __shared__ int32_t path_s[64];
  for (int j = threadIdx.x; j < cnt && j < 64; j += blockDim.x) path_s[j] = tb.path[b * Pmax + j];
  __syncthreads();
  if (l < L) {
    // A thread owns the same 16-byte vectors of every position.  Per batch of JB accepted nodes it issues all its loads
    // before its first store: a destination slot j can only be the source of an earlier node (path[j'] >= j'), never
    // of a later batch, and within a batch every load has been issued before any store.
    T *Kp = (T *)pools[l].k, *Vp = (T *)pools[l].v;
    const int nvec = G * hd / VEC;
    for (int t = threadIdx.x; t < nvec; t += blockDim.x) {
      const int g = (t * VEC) / hd, i = (t * VEC) % hd;
      for (int j0 = 0; j0 < cnt; j0 += JB) {
        uint4 kv[JB], vv[JB];
        size_t dof[JB];
        bool mv[JB];
#pragma unroll
        for (int jj = 0; jj < JB; jj++) {
          const int j = j0 + jj;
          mv[jj] = false;
          if (j < cnt) {
            const int src = n0 + path_s[j], dst = n0 + j;
            mv[jj] = src != dst;
            if (mv[jj]) {
              const size_t so = kv_offset(pm, b, src, g, G, hd) + i;
              dof[jj] = kv_offset(pm, b, dst, g, G, hd) + i;
              kv[jj] = *(const uint4 *)(Kp + so);
              vv[jj] = *(const uint4 *)(Vp + so);
            }
          }
        }
#pragma unroll
        for (int jj = 0; jj < JB; jj++)
          if (mv[jj]) { *(uint4 *)(Kp + dof[jj]) = kv[jj]; *(uint4 *)(Vp + dof[jj]) = vv[jj]; }
      }
    }
  } else if (const int j = l - L; j < cnt) {
    // taps of the j-th accepted node -> pending entry j (different buffers: no ordering needed), a block each with its loads in flight (one
    // block for all of them took 15 us, and with it the launch)
    const int nvec = 3 * k / VEC;
    const uint4 *__restrict__ src = (const uint4 *)(node_taps + ((size_t)b * rows_per_seq + path_s[j]) * 3 * k);
    uint4 *__restrict__ dst = (uint4 *)(pend_taps + ((size_t)b * Pmax + j) * 3 * k);
    constexpr int NV = 8;
    for (int e0 = threadIdx.x; e0 < nvec; e0 += NV * blockDim.x) {
      uint4 v[NV];
#pragma unroll
      for (int q = 0; q < NV; q++)
        if (e0 + q * (int)blockDim.x < nvec) v[q] = src[e0 + q * blockDim.x];
#pragma unroll
      for (int q = 0; q < NV; q++)
        if (e0 + q * (int)blockDim.x < nvec) dst[e0 + q * blockDim.x] = v[q];
    }
  }
}
template <typename T>
void launch_commit(SeqState st, TreeBufs tb, const KvPool *pools, PageMap pm, const T *node_taps, T *pend_taps, int B,
                   int L, int G, int hd, int k, int rows_per_seq, cudaStream_t s) {
  launch_k(commit_kernel<T>, dim3(B, L + tb.Pmax), dim3(256), 0, s, st, tb, pools, pm, node_taps, pend_taps, L, G, hd, k, rows_per_seq);
}
template void launch_commit<float>(SeqState, TreeBufs, const KvPool *, PageMap, const float *, float *, int, int, int,
                                   int, int, int, cudaStream_t);
template void launch_commit<bf16>(SeqState, TreeBufs, const KvPool *, PageMap, const bf16 *, bf16 *, int, int, int, int,
                                  int, int, cudaStream_t);

}  // namespace spec
