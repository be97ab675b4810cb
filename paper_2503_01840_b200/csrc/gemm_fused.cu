// Weight-streaming bf16 GEMM with fused epilogues for sm_100a.
//
//   out[r][o] = sum_i x[r][i] * w[o][i],  rows <= 256 token rows, weights far larger than the L2.
//
// The contraction is HBM-bound (every weight byte is read once per launch), so the kernel is built
// around keeping many weight bytes in flight per SM and wasting no extra pass over the result:
//
//  * swap-AB mapping: the weight tile (128 output features x 64 k, K-major, 128-byte swizzle) is the
//    UMMA M side, the token rows the N side (NT = 16/64/128/256), the fp32 accumulator sits in TMEM;
//  * warp 0 streams tiles with TMA through a ring of shared-memory stages, warp 1 issues tcgen05.mma; both walk their
//    loops as converged warps and one lane chosen by elect.sync issues (the issuing warp, not shared memory or HBM,
//    is what limits a single CTA: see ubench/issue_loop.cu);
//  * split-K: the S slices of one feature tile form a thread-block cluster.  Each CTA parks its
//    accumulator in its own shared memory and every CTA reduces a share of the rows by reading its
//    peers' copies through distributed shared memory, in slice order (deterministic, no atomics, no
//    round trip of partial sums through global memory);
//  * the epilogue that follows the reduction is the consumer's work: residual add + bf16 copy scaled
//    by the next norm's gain + RMSNorm statistics (+ feature taps); RoPE + q store + paged K/V write;
//    SiLU(gate)*up (gate and up tiles of a feature range in one CTA); per-tile argmax; per-tile top-K.  RMSNorm of the input is applied as a per-row scale in the
//    epilogue (the normalisation factor is a row constant, so it commutes with the contraction);
//  * programmatic dependent launch: the producer prefetches the first weight tiles (which never depend
//    on the previous kernel) before griddepcontrol.wait, so the pipeline is full when the activations
//    become valid.
//
// Every mbarrier wait is bounded; on timeout the CTA records it, skips its arithmetic, still takes part
// in the cluster barriers (so its peers are not left waiting), frees its TMEM and exits.
#include <cuda.h>
#include <stdio.h>

#include <algorithm>

#include "gemm_fused.cuh"
#include "tcgen05_ptx.cuh"

namespace spec {

namespace {

using namespace tc;

constexpr int MAX_STAGES = 16;
constexpr int CHUNK = 64;                       // rows reduced per epilogue round (tiles of up to 64 rows)
constexpr int MAX_CHUNK = 256;                  // wider tiles take as many rows per round as the free ring holds
constexpr int A_BYTES = TILE_M * TILE_K * 2;    // one weight tile of a stage

struct alignas(64) FusedParams {
  CUtensorMap map_w[3];
  CUtensorMap map_x;
  int tiles0, tiles1;          // tile index ranges of the weights: [0,tiles0) w0, [tiles0,tiles1) w1, rest w2
  int O[3];
  int nrt;                                 // gemm_swiglu_pair_kernel: rows of its MMAs, the rows there are in whole 16s
  int rows, KB, S, stages, ctrl_off;       // S = K slices = cluster size (CTA pairs: half of it)
  int chunk;                               // rows per epilogue round
  const float *ssq_in; int ssq_in_tiles, ssq_ld; float inv_k_in, eps;
  float *out_f32; int ldo;
  float *xres; const bf16 *gain; bf16 *hb; float *ssq_out; bf16 *taps; int tap_mask, resid_add;
  const float2 *cs; RowMeta m; bf16 *q; KvPool pool; PageMap pm; int H, G, hd;
  bf16 *act;
  int vec;                                 // EPI_RESID: the gains, EPI_SWIGLU: act, EPI_F32: out_f32 take vector accesses
  float *best_val; int32_t *best_idx; int best_ld;
  int topk; float *cand_val, *cand_max, *cand_sum; int32_t *cand_idx; int cand_ld; const int32_t *want_rows; int n_want;
  int32_t *status;
  unsigned long long *stamp;
  unsigned spin;               // polls before a wait gives up
  int withhold;                // test hook: CTA 0 leaves out the activation load of its first k-block
};

__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// norm gains of features f .. f + 3; they are the caller's, who owes them no alignment beyond their own two bytes
__device__ __forceinline__ float4 load_gain4(const FusedParams &p, int f) {
  const bf16 *g = p.gain + f;
  if (!p.vec) return make_float4(to_f32(g[0]), to_f32(g[1]), to_f32(g[2]), to_f32(g[3]));
  const uint2 u = *(const uint2 *)g;
  const float2 g01 = __bfloat1622float2(*(const __nv_bfloat162 *)&u.x), g23 = __bfloat1622float2(*(const __nv_bfloat162 *)&u.y);
  return make_float4(g01.x, g01.y, g23.x, g23.y);
}
__device__ __forceinline__ uint2 pack4(float4 v) {
  __nv_bfloat162 a = __floats2bfloat162_rn(v.x, v.y), b = __floats2bfloat162_rn(v.z, v.w);
  return make_uint2(*(uint32_t *)&a, *(uint32_t *)&b);
}
__device__ __forceinline__ float silu_mul(float g, float u) { return (g / (1.0f + expf(-g))) * u; }

__device__ __forceinline__ uint32_t ld_peer_u32(uint32_t local_addr, uint32_t rank) {
  uint32_t ra, v;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(local_addr), "r"(rank));
  asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(ra) : "memory");
  return v;
}

// 16-byte load from a cluster address (a CTA's own shared-memory address is one too).  Deliberately without a "memory"
// clobber: consecutive loads stay in program order (volatile) but do not wait for one another, so a thread keeps several
// remote requests in flight.
__device__ __forceinline__ float4 ld_cluster4(uint32_t addr) {
  float4 v;
  asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr));
  return v;
}
// Sums over the cluster's K slices of up to N rows of this warp (row0, row0 + step, .. up to last; four features a lane), added
// in slice order: red is this CTA's dump [row][128], slice i is cluster member first + i * stride.  All remote loads are in
// flight before the first sum (S <= 8), and only what is needed crosses the SM-to-SM fabric, which moves 3 TB/s in all: rows
// past the last are not read, the CTA's own slice comes from its own shared memory.
template <int N>
__device__ __forceinline__ void sum_slices(const float *red, int row0, int step, int last, int lane, int S, int own, int first, int stride, float4 (&v)[N]) {
  float4 t[N][8];
  auto fetch = [&](int j) {
    const uint32_t la = smem_u32(&red[(row0 + j * step) * TILE_M + lane * 4]);
#pragma unroll
    for (int i = 0; i < 8; i++)
      if (i < S) t[j][i] = ld_cluster4(i == own ? la : mapa_u32(la, (uint32_t)(first + i * stride)));
  };
  if (row0 + (N - 1) * step <= last) {       // the usual case without a branch per row
#pragma unroll
    for (int j = 0; j < N; j++) fetch(j);
  } else {
#pragma unroll
    for (int j = 0; j < N - 1; j++)
      if (row0 + j * step <= last) fetch(j);
  }
#pragma unroll
  for (int j = 0; j < N; j++) {
    v[j] = t[j][0];
#pragma unroll
    for (int i = 1; i < 8; i++)
      if (i < S) { v[j].x += t[j][i].x; v[j].y += t[j][i].y; v[j].z += t[j][i].z; v[j].w += t[j][i].w; }
  }
}
// the values are there: nothing after this point (asm volatile) is issued before the loads they come from have returned
template <int N>
__device__ __forceinline__ void arrived(const float4 (&v)[N]) {
#pragma unroll
  for (int j = 0; j < N; j++) asm volatile("" ::"f"(v[j].x), "f"(v[j].y), "f"(v[j].z), "f"(v[j].w));
}

// PAIR (EPI_SWIGLU only): the CTA streams the gate tile AND the up tile of its 128 features for its K slice, both
// MMAs of a k-block share one activation tile, and the two accumulators sit side by side in tensor memory.
//
// MIX (EPI_SWIGLU only): one 128-row weight tile made of 64 gate features and the 64 up features of the same range, the whole
// contraction in one CTA.  It takes the place of PAIR with two K slices: the same number of CTAs, but no cluster, no parked
// partial sums and no exchange through distributed shared memory, which cost 5 us of a launch at 60 rows (the launch is bound by
// the weight stream, and what comes after the last k-block is not hidden by it).  8B shapes, inside the replayed step: 46.6 ->
// 41.7 us at 60 rows, 38.0 -> 34.5 at 10, 43.8 -> 40.2 at 40; 13B shapes at 50 rows 52.6 -> 47.3; C2 step 4.950 -> 4.775 ms.  The
// activation k-block is read once per 64 features instead of 128 (1.5 bytes from L2 per weight byte at 60 rows against 1.25).
//
// DUO (256-row tiles; EPI_F32 / EPI_RESID / EPI_QKV): two neighbouring feature tiles run as a CTA pair (cta_group::2).
// Each CTA streams its own weight tile but only HALF of the activation k-block (128 of the 256 rows); the even CTA issues
// one M = 256 MMA per k-step that reads both CTAs' shared memory, and each CTA's tensor memory receives the accumulator
// of its own tile.  At 256 rows the activation k-block (32 KB) is twice a weight tile, so the shared-memory fill traffic
// per weight byte drops from 3 x to 2 x, which is what bounds the loop at this width.  The cluster is (2, S): x = the
// pair, y = the K slices; the reduction runs over the members with the same x.
// Threads per CTA: 128; the 256-row tiles run 256, so that two threads share a feature when the accumulator is dumped and twice
// as many warps take rows afterwards (the epilogue of a 256-row tile is as long as its main loop).  So do the top-K and the gate/up
// epilogues from 64-row tiles on, whose arithmetic per value (selection, exponential and division) is long enough to share:
// top-K at 40 rows 70 -> 66 us, gate/up at 60 rows 41.5 -> 40.7.  They need two CTAs per SM as the others do, hence the bound on
// registers (without it top-K at 40 rows takes 82 us, the 70B gate/up 208 us instead of 147).
constexpr int fused_threads(int nt, int epi) { return ((epi == EPI_TOPK || epi == EPI_SWIGLU) && nt >= 64) || (nt == 256 && (epi == EPI_F32 || epi == EPI_RESID || epi == EPI_QKV)) ? 256 : 128; }

template <int NT, int EPI, bool PAIR = false, bool DUO = false, bool MIX = false>
__global__ void __launch_bounds__(fused_threads(NT, EPI), EPI == EPI_TOPK || EPI == EPI_SWIGLU ? 2 : 1) gemm_fused_kernel(const __grid_constant__ FusedParams p) {
  constexpr int THREADS = fused_threads(NT, EPI), NH = THREADS / 128;
  static_assert((EPI == EPI_SWIGLU) == (PAIR || MIX), "two weight tiles per CTA exist for the gate/up epilogue only");
  static_assert(!MIX || (EPI == EPI_SWIGLU && !PAIR && !DUO), "tiles of 64 gate and 64 up features exist for the gate/up epilogue only");
  static_assert(!DUO || (NT == 256 && !PAIR && (EPI == EPI_F32 || EPI == EPI_RESID || EPI == EPI_QKV)), "CTA pairs serve the 256-row tiles");
  constexpr int A_TILES = PAIR ? 2 : 1;
  constexpr int F_TILE = MIX ? TILE_M / 2 : TILE_M;            // output features of a tile
  constexpr int B_BYTES = (DUO ? NT / 2 : NT) * TILE_K * 2;
  constexpr int STAGE = A_TILES * A_BYTES + B_BYTES;
  constexpr int TMEM_COLS = (A_TILES * NT < 32) ? 32 : A_TILES * NT;
  static_assert(TMEM_COLS <= 512, "accumulators must fit the tensor memory");

  extern __shared__ unsigned char smem_raw[];
  unsigned char *tiles = (unsigned char *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  unsigned char *ctrl = tiles + p.ctrl_off;
  uint64_t *full = (uint64_t *)ctrl;
  uint64_t *empty = full + MAX_STAGES;
  uint64_t *acc_bar = empty + MAX_STAGES;
  uint32_t *tmem_slot = (uint32_t *)(acc_bar + 1);
  volatile uint32_t *abort_flag = tmem_slot + 1;
  volatile int *n_issued = (volatile int *)(tmem_slot + 2), *n_consumed = (volatile int *)(tmem_slot + 3);   // stage loads issued / seen complete
  float *inv_s = (float *)(ctrl + 512);          // [256] per-row input scale
  float *wpart = inv_s + 256;                    // [4][MAX_CHUNK] per-warp partial sums / argmax exchange
  int32_t *slot_s = (int32_t *)wpart, *seq_s = slot_s + 256;   // EPI_QKV: element offset / hd of every row's K/V slot (-1: none), its sequence

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int stages = p.stages, S = p.S;
  const uint32_t crank = (S > 1 || DUO) ? cluster_rank() : 0u;
  const int xr = DUO ? (int)(crank & 1u) : 0;                 // DUO: position in the CTA pair (0 issues the MMAs)
  const int slice = DUO ? (int)(crank >> 1) : (int)crank;     // K slice = rank among the CTAs that share this feature tile
  const int kb0 = (int)(((long long)slice * p.KB) / S), kb1 = (int)(((long long)(slice + 1) * p.KB) / S);
  const int nkb = kb1 - kb0;
  int mi = 0, tm = blockIdx.x;                   // weight index and tile within that weight
  if (EPI != EPI_SWIGLU) {
    if (tm >= p.tiles1) { mi = 2; tm -= p.tiles1; }
    else if (tm >= p.tiles0) { mi = 1; tm -= p.tiles0; }
  }

  if (threadIdx.x == 0) {
    for (int i = 0; i < stages; i++) { mbar_init(&full[i], 1); mbar_init(&empty[i], 1); }
    mbar_init(acc_bar, 1);
    *abort_flag = 0;
    *n_issued = 0; *n_consumed = 0;
    // pairs rely on cluster ranks running x first (rank = x + 2 y): checked, never assumed
    if (DUO && ((crank & 1u) != (blockIdx.x & 1u) || (int)(crank >> 1) != (int)(blockIdx.y % (unsigned)S))) {
      *abort_flag = 1;
      set_status(p.status, ST_TIMEOUT, 234, blockIdx.x, (int)crank);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  // The weight tiles do not depend on the previous kernel, and nobody but this warp has to be there for them: the ring is
  // filled with them before the block's first barrier and the tensor-memory allocation.
  const int npre = nkb < stages ? nkb : stages;
  const uint64_t pol = l2_policy_evict_first();
  if (!DUO && warp == 0) {
    __syncwarp();
    if (elect_one()) {
      for (int i = 0; i < npre; i++) {
        unsigned char *a = tiles + i * STAGE;
        mbar_expect_tx(&full[i], STAGE);
        tma_load_2d_hint(a, &p.map_w[mi], (kb0 + i) * TILE_K, tm * F_TILE, &full[i], pol);
        if (MIX) tma_load_2d_hint(a + A_BYTES / 2, &p.map_w[1], (kb0 + i) * TILE_K, tm * F_TILE, &full[i], pol);
        if (PAIR) tma_load_2d_hint(a + A_BYTES, &p.map_w[1], (kb0 + i) * TILE_K, tm * TILE_M, &full[i], pol);
      }
      tma_prefetch_map(&p.map_x);
    }
    __syncwarp();
  }
  if (warp == 1) {   // TMEM allocation is a whole-warp operation (pairs: the same warp of both CTAs, same slot offset)
    if (DUO) {
      asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(TMEM_COLS)
                   : "memory");
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    } else {
      asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(TMEM_COLS)
                   : "memory");
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  if (DUO) cluster_sync_all(); else __syncthreads();   // pairs: the partner's barriers must exist before anything signals them
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem_base = *tmem_slot;
  // EPI_QKV lets its dependents start only once it is past its own wait: whatever earlier kernels of the stream wrote is then
  // complete, and the attention kernel that follows reads it (row metadata, page table, cached context) before it waits itself.
  if (EPI != EPI_QKV) pdl_trigger();

  if (DUO && *abort_flag) {
    pdl_wait();            // wrong cluster layout: nothing is loaded or issued; the epilogue below writes nothing
  } else if (DUO && warp == 0) {
    // ---- producer of a CTA pair: own weight tile + own half of the activation rows; every byte of both CTAs is counted
    // on the even CTA's full barrier (it alone announces the byte count: one arrival per phase).
    const CUtensorMap *mw0 = &p.map_w[mi];
    const uint32_t lead = crank & ~1u;
    if (elect_one())
      for (int i = 0; i < npre; i++) {
        if (xr == 0) mbar_expect_tx(&full[i], 2 * STAGE);
        tma_load_2d_pair_hint(tiles + i * STAGE, mw0, (kb0 + i) * TILE_K, tm * TILE_M, mapa_u32(smem_u32(&full[i]), lead), pol);
      }
    __syncwarp();
    pdl_wait();
    if (EPI == EPI_QKV) pdl_trigger();
    if (elect_one()) {
      if (p.stamp) atomicMin(p.stamp, global_ns());
      for (int i = 0; i < npre; i++)
        tma_load_2d_pair(tiles + i * STAGE + A_BYTES, &p.map_x, (kb0 + i) * TILE_K, xr * (NT / 2), mapa_u32(smem_u32(&full[i]), lead));
    }
    __syncwarp();
    // steady state: stage and phase advance by increments (no divisions), nothing but the wait and the copies per k-block
    int i = npre, st = 0;
    uint32_t ph = 0;
    for (; i < nkb; i++) {
      if (!mbar_wait_warp(&empty[st], ph, p.spin)) { *abort_flag = 1; set_status(p.status, ST_TIMEOUT, 230, blockIdx.x, i); break; }
      if (elect_one()) {
        unsigned char *a = tiles + st * STAGE;
        const uint32_t fb = mapa_u32(smem_u32(&full[st]), lead);
        if (xr == 0) mbar_expect_tx(&full[st], 2 * STAGE);
        tma_load_2d_pair_hint(a, mw0, (kb0 + i) * TILE_K, tm * TILE_M, fb, pol);
        tma_load_2d_pair(a + A_BYTES, &p.map_x, (kb0 + i) * TILE_K, xr * (NT / 2), fb);
      }
      __syncwarp();
      if (++st == stages) { st = 0; ph ^= 1u; }
    }
    if (lane == 0) *n_issued = i;
  } else if (!DUO && warp == 0) {
    // ---- producer warp (all lanes walk the loop, the elected lane issues); the ring already holds weight tiles
    const CUtensorMap *mw0 = &p.map_w[mi];
    pdl_wait();
    if (EPI == EPI_QKV) pdl_trigger();
    if (elect_one()) {
      if (p.stamp) atomicMin(p.stamp, global_ns());
      const bool hold = p.withhold && blockIdx.x == 0 && blockIdx.y == 0;     // test hook: the first stage never completes
      for (int i = hold ? 1 : 0; i < npre; i++) tma_load_2d(tiles + i * STAGE + A_TILES * A_BYTES, &p.map_x, (kb0 + i) * TILE_K, 0, &full[i]);
    }
    __syncwarp();
    int i = npre, st = 0;             // the loop runs only when the prefill used every stage: it restarts at stage 0
    uint32_t ph = 0;
    for (; i < nkb; i++) {
      if (!mbar_wait_warp(&empty[st], ph, p.spin)) { *abort_flag = 1; set_status(p.status, ST_TIMEOUT, 200, blockIdx.x, i); break; }
      if (elect_one()) {
        unsigned char *a = tiles + st * STAGE;
        mbar_expect_tx(&full[st], STAGE);
        tma_load_2d_hint(a, mw0, (kb0 + i) * TILE_K, tm * F_TILE, &full[st], pol);
        if (MIX) tma_load_2d_hint(a + A_BYTES / 2, &p.map_w[1], (kb0 + i) * TILE_K, tm * F_TILE, &full[st], pol);
        if (PAIR) tma_load_2d_hint(a + A_BYTES, &p.map_w[1], (kb0 + i) * TILE_K, tm * TILE_M, &full[st], pol);
        tma_load_2d(a + A_TILES * A_BYTES, &p.map_x, (kb0 + i) * TILE_K, 0, &full[st]);
      }
      __syncwarp();
      if (++st == stages) { st = 0; ph ^= 1u; }
    }
    if (lane == 0) *n_issued = i;
  } else {
    pdl_wait();
    if (EPI == EPI_QKV) pdl_trigger();
    if (DUO && warp == 1) {
      // ---- MMA issuer of a CTA pair (even CTA only): M = 256 over both CTAs' weight tiles, N = both activation halves
      if (xr == 0) {
        constexpr uint32_t idesc = umma_idesc_m(NT, 2 * TILE_M);
        const uint32_t pair_lead = crank;                        // this (even) CTA and its partner crank + 1
        const uint32_t partner_base = ld_peer_u32(smem_u32(tmem_slot), crank | 1u);
        if (partner_base != tmem_base) { *abort_flag = 1; set_status(p.status, ST_TIMEOUT, 233, blockIdx.x, (int)partner_base); }
        const uint64_t desc0 = umma_desc_sw128(smem_u32(tiles));
        int i = 0, st = 0;
        uint32_t ph = 0, ready = 0;
        if (!*abort_flag)
          for (; i < nkb; i++) {
            if (!ready && !mbar_wait_warp(&full[st], ph, p.spin)) { *abort_flag = 1; set_status(p.status, ST_TIMEOUT, 231, blockIdx.x, i); break; }
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint64_t da = desc0 + (uint64_t)((st * STAGE) >> 4);
            int nst = st + 1;
            uint32_t nph = ph;
            if (nst == stages) { nst = 0; nph ^= 1u; }
            if (elect_one()) {
#pragma unroll
              for (int j = 0; j < TILE_K / UMMA_K; j++) umma_bf16_pair(tmem_base, da + 2 * j, da + (A_BYTES >> 4) + 2 * j, idesc, (i | j) ? 1u : 0u);
              umma_commit_pair(&empty[st], pair_lead);      // frees the stage in both CTAs
            }
            __syncwarp();
            ready = mbar_test_warp(&full[nst], nph) ? 1u : 0u;
            st = nst; ph = nph;
          }
        if (lane == 0) *n_consumed = i;
        __syncwarp();
        if (!*abort_flag && elect_one()) umma_commit_pair(acc_bar, pair_lead);   // both accumulators complete
      }
    } else if (!DUO && warp == 1) {
      // ---- MMA issuer warp (all lanes walk the loop, the elected lane issues)
      // The issuing warp is what limits a CTA's streaming rate, so the loop is kept to a non-blocking look at the
      // barrier (the blocking wait only when the stage is not full yet), one fence, four MMAs and the commit.
      constexpr uint32_t idesc = umma_idesc(NT);
      const uint64_t desc0 = umma_desc_sw128(smem_u32(tiles));
      int i = 0, st = 0;
      uint32_t ph = 0, ready = 0;
      for (; i < nkb; i++) {
        if (!ready && !mbar_wait_warp(&full[st], ph, p.spin)) { *abort_flag = 1; set_status(p.status, ST_TIMEOUT, 201, blockIdx.x, i); break; }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint64_t da = desc0 + (uint64_t)((st * STAGE) >> 4), db = da + (uint64_t)((A_TILES * A_BYTES) >> 4);
        int nst = st + 1;
        uint32_t nph = ph;
        if (nst == stages) { nst = 0; nph ^= 1u; }
        if (elect_one()) {
#pragma unroll
          for (int j = 0; j < TILE_K / UMMA_K; j++) {      // a K = 16 step advances the descriptors by 32 bytes = 2 units
            umma_bf16(tmem_base, da + 2 * j, db + 2 * j, idesc, (i | j) ? 1u : 0u);
            if (PAIR) umma_bf16(tmem_base + NT, da + (A_BYTES >> 4) + 2 * j, db + 2 * j, idesc, (i | j) ? 1u : 0u);   // the up accumulator
          }
          umma_commit(&empty[st]);      // frees the stage once these MMAs have read it
        }
        __syncwarp();
        ready = mbar_test_warp(&full[nst], nph) ? 1u : 0u;      // a cheap look at the next stage: mostly spares the wait
        st = nst; ph = nph;
      }
      if (lane == 0) *n_consumed = i;
      if (elect_one()) umma_commit(acc_bar);           // accumulator complete
    } else if (warp >= 2) {
      // ---- per-row scale of the input: rsqrt(mean square + eps) from the producer kernel's per-tile sums
      for (int r = threadIdx.x - 64; r < p.rows; r += THREADS - 64) {
        float sc = 1.0f;
        if (p.ssq_in) {
          float ss = 0.0f;
          for (int t = 0; t < p.ssq_in_tiles; t++) ss += p.ssq_in[(size_t)t * p.ssq_ld + r];
          sc = 1.0f / sqrtf(ss * p.inv_k_in + p.eps);
        }
        inv_s[r] = sc;
      }
      // ---- cache slot of every row: a chain of three dependent loads (sequence, position, page), here under the main loop
      if (EPI == EPI_QKV)
        for (int row = threadIdx.x - 64; row < p.rows; row += THREADS - 64) {
          const int seq = p.m.seq[row];
          int slot = -1;
          if (seq >= 0 && mi > 0) {
            const int kvpos = p.m.kvpos[row];
            if (kvpos < 0 || kvpos / p.pm.page_size >= p.pm.pages_per_seq) {
              set_status(p.status, ST_BOUNDS, 1, row, kvpos);
            } else {
              const int page = p.pm.table[(size_t)seq * p.pm.pages_per_seq + kvpos / p.pm.page_size];
              if (page < 0 || page >= p.pm.num_pages) set_status(p.status, ST_BOUNDS, 2, row, page);
              else slot = (page * p.G) * p.pm.page_size + (kvpos % p.pm.page_size);   // + head * page_size below
            }
          }
          slot_s[row] = slot;
          seq_s[row] = seq;
        }
    }
  }
  __syncthreads();

  // ---- what the epilogue reads from global memory besides the accumulator: the first batch of rows is requested here, so
  // that it arrives during the wait, the dump and the cluster's exchange
  const int CH = (NT <= CHUNK || EPI == EPI_ARGMAX) ? CHUNK : p.chunk;   // rows per epilogue round; a constant for the narrow tiles
  const int f = threadIdx.x & (TILE_M - 1);          // feature of the tile = tensor-memory lane (a warp reads lanes 32 (warp % 4) ..)
  const int hw = threadIdx.x >> 7;                   // 0, or with 256 threads which half of the columns
  const int o = tm * TILE_M + f;                     // output feature within weight mi
  constexpr bool ROWWISE = EPI == EPI_RESID || EPI == EPI_QKV || EPI == EPI_F32 || PAIR;
  constexpr int NW = THREADS / 32;
  constexpr int IT = NT <= 16 || PAIR ? 1 : NT == 64 ? 3 : 2;   // ROWWISE: rows a warp has in flight (60 rows, 7 slices: a CTA's share is one batch)
  const int fo = tm * TILE_M + lane * 4;             // ROWWISE: a warp takes whole rows, a lane four features of the tile
  const bool fok = fo < p.O[mi];
  const int half = EPI == EPI_QKV ? p.hd >> 1 : 0, qi = EPI == EPI_QKV ? fo & (p.hd - 1) : 0;   // EPI_QKV: features qi .. + 3 of their head
  float4 xin[EPI == EPI_RESID ? IT : 1], cs[EPI == EPI_QKV ? 2 * IT : 1];
  auto request = [&](int row, int last) {            // rows row, row + NW, .. up to last
#pragma unroll
    for (int j = 0; j < IT; j++) {
      const int r = row + j * NW;
      if (EPI == EPI_RESID) xin[j] = (fok && p.resid_add && r <= last) ? *(const float4 *)(p.xres + (size_t)r * p.O[0] + fo) : make_float4(0.f, 0.f, 0.f, 0.f);
      if (EPI == EPI_QKV) {
        const bool rot = fok && mi < 2 && r <= last;
        const float4 *c = (const float4 *)(p.cs + (size_t)r * half + (qi & (half - 1)));
        cs[2 * j] = rot ? c[0] : make_float4(1.f, 0.f, 1.f, 0.f);
        cs[2 * j + 1] = rot ? c[1] : make_float4(1.f, 0.f, 1.f, 0.f);
      }
    }
  };
  float4 gn = make_float4(0.f, 0.f, 0.f, 0.f);
  if (EPI == EPI_RESID || EPI == EPI_QKV) {
    const int nrow = p.rows < CH ? p.rows : CH, per = (nrow + S - 1) / S, last = slice * per + per < nrow ? slice * per + per : nrow;
    request(slice * per + warp, last - 1);
    if (EPI == EPI_RESID && fok) gn = load_gain4(p, fo);
  }

  // ---- wait for the accumulator (one bounded wait per warp)
  int good = 0;
  if (lane == 0) {
    bool ok = *abort_flag ? false : mbar_wait(acc_bar, 0, p.spin);    // after an abort the accumulator never completes
    if (!ok && !*abort_flag) { *abort_flag = 1; set_status(p.status, ST_TIMEOUT, 202, blockIdx.x, slice); }
    good = (ok && !*abort_flag) ? 1 : 0;
  }
  good = __shfl_sync(0xffffffffu, good, 0);
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");

  // ---- epilogue, CH rows at a time.  The stage ring is free now (every load landed, every MMA that
  // read it completed) and is reused: red = this CTA's accumulator, sumb = this CTA's rows after the cluster sum.
  float *red = (float *)tiles;                       // [CH][128]
  float *red_u = red + CH * TILE_M;                  // PAIR: the up accumulator, [CH][128]
  float *sumb = red + CH * TILE_M;                   // EPI_TOPK: this CTA's rows after the cluster sum, [rows][128]
  for (int c0 = 0; c0 < p.rows; c0 += CH) {
    const int nrow = (p.rows - c0 < CH) ? p.rows - c0 : CH;
    if (good) {
#pragma unroll 1
      for (int cc = hw * (CH / NH); cc < (hw + 1) * (CH / NH) && c0 + cc < NT; cc += 16) {
        if (cc >= nrow) break;
        uint32_t v[16];
        tmem_ld16(tmem_base + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)(c0 + cc), v);
#pragma unroll
        for (int j = 0; j < 16; j++) red[(cc + j) * TILE_M + f] = __uint_as_float(v[j]);
        if (PAIR) {
          tmem_ld16(tmem_base + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)(NT + c0 + cc), v);
#pragma unroll
          for (int j = 0; j < 16; j++) red_u[(cc + j) * TILE_M + f] = __uint_as_float(v[j]);
        }
      }
    }
    if (S > 1) cluster_sync_all(); else __syncthreads();
    const int per = (nrow + S - 1) / S;
    const int r0 = (slice * per < nrow) ? slice * per : nrow, r1 = (r0 + per < nrow) ? r0 + per : nrow;   // r0 <= r1
    const int first = DUO ? xr : 0, stride = DUO ? 2 : 1;                                                  // cluster ranks of the K slices

    if (ROWWISE) {
      // Reduction and epilogue in one pass over registers: a warp takes whole rows (IT at a time), a lane four features.  What
      // follows the last k-block is a chain of latencies that nothing hides.  With a thread per feature walking the rows, after
      // the sums had gone through shared memory, the epilogue alone took 2.4 us of the O launch at 60 rows (9 rows per CTA), as
      // long as the reduction.  8B shapes inside the replayed step, 60 rows: O 12.3 -> 10.9 us, down 24.0 -> 22.7, QKV 14.1 ->
      // 12.7 (its cache slots, three dependent loads, are now looked up under the main loop); 10 rows: QKV 11.0 -> 10.3.
      const int nb = max(1, (r1 - r0 + IT * NW - 1) / (IT * NW));          // uniform over the CTA
      for (int b = 0; b < nb; b++) {
        const int rb = r0 + b * IT * NW + warp;
        if (c0 > 0 || b > 0) request(c0 + rb, c0 + r1 - 1);
        float4 v[IT], u[PAIR ? IT : 1];
        if (rb < r1) {                       // uniform over the warp
          sum_slices<IT>(red, rb, NW, r1 - 1, lane, S, slice, first, stride, v);
          arrived(v);
          if constexpr (PAIR) { sum_slices<IT>(red_u, rb, NW, r1 - 1, lane, S, slice, first, stride, u); arrived(u); }
        }
        // this CTA has everything it needs from its peers: announce it now and wait only at the end of the round
        if (S > 1 && b == nb - 1) asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
#pragma unroll
        for (int j = 0; j < IT; j++) {
          const int r = rb + j * NW, row = c0 + r;
          if (r >= r1 || !good) continue;    // uniform over the warp
          float4 a = v[j];
          if (EPI == EPI_RESID) {
            float sq = 0.0f;
            if (fok) {
              a.x += xin[j].x; a.y += xin[j].y; a.z += xin[j].z; a.w += xin[j].w;
              const size_t xi = (size_t)row * p.O[0] + fo;
              *(float4 *)(p.xres + xi) = a;
              *(uint2 *)(p.hb + xi) = pack4(make_float4(a.x * gn.x, a.y * gn.y, a.z * gn.z, a.w * gn.w));
              if (p.tap_mask) {
                const uint2 tb = pack4(a);
#pragma unroll
                for (int s = 0; s < 3; s++)
                  if ((p.tap_mask >> s) & 1) *(uint2 *)(p.taps + (size_t)row * 3 * p.O[0] + (size_t)s * p.O[0] + fo) = tb;
              }
              sq = (a.x * a.x + a.y * a.y) + (a.z * a.z + a.w * a.w);
            }
            for (int off = 16; off > 0; off >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, off);
            if (lane == 0) p.ssq_out[(size_t)tm * p.ssq_ld + row] = sq;
          } else if (EPI == EPI_QKV) {
            const float sc = inv_s[row];
            a.x *= sc; a.y *= sc; a.z *= sc; a.w *= sc;
            if (mi < 2) {                    // rotate-half RoPE: the partner features qi ^ half are half / 4 lanes away (hd >= 8)
              float4 w;
              w.x = __shfl_xor_sync(0xffffffffu, a.x, half >> 2); w.y = __shfl_xor_sync(0xffffffffu, a.y, half >> 2);
              w.z = __shfl_xor_sync(0xffffffffu, a.z, half >> 2); w.w = __shfl_xor_sync(0xffffffffu, a.w, half >> 2);
              if (qi < half) { w.x = -w.x; w.y = -w.y; w.z = -w.z; w.w = -w.w; }
              const float4 c = cs[2 * j], d = cs[2 * j + 1];
              a = make_float4(a.x * c.x + w.x * c.y, a.y * c.z + w.y * c.w, a.z * d.x + w.z * d.y, a.w * d.z + w.w * d.w);
            }
            if (!fok) continue;
            const int head = fo / p.hd;
            if (mi == 0) {
              if (seq_s[row] < 0) a = make_float4(0.f, 0.f, 0.f, 0.f);
              *(uint2 *)(p.q + ((size_t)row * p.H + head) * p.hd + qi) = pack4(a);
            } else if (slot_s[row] >= 0) {
              bf16 *kv = (bf16 *)(mi == 1 ? p.pool.k : p.pool.v);
              *(uint2 *)(kv + ((size_t)slot_s[row] + (size_t)head * p.pm.page_size) * p.hd + qi) = pack4(a);
            }
          } else if (EPI == EPI_F32) {
            const float sc = inv_s[row];
            float *dst = p.out_f32 + (size_t)row * p.ldo + fo;
            a.x *= sc; a.y *= sc; a.z *= sc; a.w *= sc;
            if (p.vec && fo + 3 < p.O[0]) *(float4 *)dst = a;
            else {
              const float e[4] = {a.x, a.y, a.z, a.w};
#pragma unroll
              for (int z = 0; z < 4; z++)
                if (fo + z < p.O[0]) dst[z] = e[z];
            }
          } else if constexpr (PAIR) {
            const float sc = inv_s[row];
            const float e[4] = {silu_mul(a.x * sc, u[j].x * sc), silu_mul(a.y * sc, u[j].y * sc), silu_mul(a.z * sc, u[j].z * sc), silu_mul(a.w * sc, u[j].w * sc)};
            bf16 *dst = p.act + (size_t)row * p.O[0] + fo;
            if (p.vec && fo + 3 < p.O[0]) *(uint2 *)dst = pack4(make_float4(e[0], e[1], e[2], e[3]));
            else {
#pragma unroll
              for (int z = 0; z < 4; z++)
                if (fo + z < p.O[0]) dst[z] = __float2bfloat16_rn(e[z]);
            }
          }
        }
      }
    } else if (MIX) {
      // red[row] = 64 gate values, then the 64 up values of the same features: a warp takes four rows at a time, a lane two features
      const int o2 = tm * F_TILE + 2 * lane;
      if (good)
        for (int rb = warp; rb < nrow; rb += 4 * NW) {
          float2 g[4], u[4];
#pragma unroll
          for (int j = 0; j < 4; j++) {
            const int r = min(rb + NW * j, nrow - 1);
            const float sc = inv_s[c0 + r];
            g[j] = *(const float2 *)&red[r * TILE_M + 2 * lane]; u[j] = *(const float2 *)&red[r * TILE_M + TILE_M / 2 + 2 * lane];
            g[j].x *= sc; g[j].y *= sc; u[j].x *= sc; u[j].y *= sc;
          }
#pragma unroll
          for (int j = 0; j < 4; j++) { g[j].x = silu_mul(g[j].x, u[j].x); g[j].y = silu_mul(g[j].y, u[j].y); }
#pragma unroll
          for (int j = 0; j < 4; j++) {
            const int r = rb + NW * j;
            bf16 *dst = p.act + (size_t)(c0 + r) * p.O[0] + o2;
            if (r >= nrow || o2 >= p.O[0]) continue;
            if (p.vec) *(__nv_bfloat162 *)dst = __floats2bfloat162_rn(g[j].x, g[j].y);
            else {
              dst[0] = __float2bfloat16_rn(g[j].x);
              if (o2 + 1 < p.O[0]) dst[1] = __float2bfloat16_rn(g[j].y);
            }
          }
        }
    } else if (EPI == EPI_TOPK) {
      const float *src = red + r0 * TILE_M;            // S == 1: the accumulator dump is the sum
      if (S > 1) {
        for (int r = r0 + warp; r < r1; r += NW) {
          float4 v[1];
          sum_slices<1>(red, r, NW, r1 - 1, lane, S, slice, first, stride, v);
          *(float4 *)&sumb[(r - r0) * TILE_M + lane * 4] = v[0];
        }
        __syncthreads();
        src = sumb;
        asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
      }
      unsigned char *want = (unsigned char *)wpart;                // [256]: rows that need candidates (a list made by an earlier kernel)
      if (p.want_rows) {
        for (int t = threadIdx.x; t < 256; t += THREADS) want[t] = 0;
        __syncthreads();
        for (int t = threadIdx.x; t < p.n_want; t += THREADS) { const int wr = p.want_rows[t]; if (wr >= 0 && wr < 256) want[wr] = 1; }
        __syncthreads();
      }
      if (good && p.out_f32 && o < p.O[0])
        for (int r = r0 + hw; r < r1; r += NH) p.out_f32[(size_t)(c0 + r) * p.ldo + o] = src[(r - r0) * TILE_M + f] * inv_s[c0 + r];
      // One warp takes four rows at a time: four independent dependency chains in straight-line code (a CTA has four warps,
      // eight from 64-row tiles on: nothing else hides the latencies).  Lane l holds features l, l+32, l+64, l+96 of the tile as order-preserving keys.  The
      // K-th largest of the 32 lane maxima bounds the tile's K-th best value from below, and few values reach it (K to about
      // 1.5 K): those are collected and ranked by counting, so that the K results leave in one store.  In the
      // replayed step, 32000 x 4096, against picking the best K times by a warp-wide reduction: K = 10 49.3 -> 44.4 us at 10 rows,
      // 76.7 -> 54.7 at 40; K = 1 60.0 -> 50.5 at 64 rows (one exchange for the four rows' sums).
      const int K = p.topk;
      unsigned *sk = (unsigned *)(sumb + (S > 1 ? per : 0) * TILE_M) + warp * 4 * 96;   // per row of the batch: [32] lane maxima, [32] (key, id)
      const int nv = min(4, max(0, (p.O[0] - tm * TILE_M - lane + 31) / 32));          // features of this lane that exist
      for (int rb = r0 + warp; rb < r1; rb += 4 * NW) {
        unsigned key[4][4], lm[4];
        bool act[4];
        float mx[4], sum[4];
#pragma unroll
        for (int q = 0; q < 4; q++) {
          const int r = rb + NW * q, row = c0 + r;
          const int rs = r < r1 ? r : r0;                                  // a row that exists (results are masked)
          act[q] = good && r < r1 && (!p.want_rows || want[row < 256 ? row : 255]);     // uniform over the warp
          const float sc = inv_s[c0 + rs];
          float v[4];
#pragma unroll
          for (int j2 = 0; j2 < 4; j2++) v[j2] = j2 < nv ? src[(rs - r0) * TILE_M + lane + 32 * j2] * sc : -INFINITY;
          mx[q] = key_value(__reduce_max_sync(0xffffffffu, ordered_key(fmaxf(fmaxf(v[0], v[1]), fmaxf(v[2], v[3])))));   // NaN: ignored
          sum[q] = 0.0f;
          lm[q] = 0u;
#pragma unroll
          for (int j2 = 0; j2 < 4; j2++) {
            key[q][j2] = ordered_key(v[j2]);
            if (j2 < nv) { lm[q] = max(lm[q], key[q][j2]); sum[q] += expf(v[j2] - mx[q]); }
          }
        }
        // sums over the lanes, the four rows in one exchange: afterwards lanes 8 q .. hold row q
        {
          const bool u1 = lane & 16, u2 = lane & 8;
          const float a = (u1 ? sum[2] : sum[0]) + __shfl_xor_sync(0xffffffffu, u1 ? sum[0] : sum[2], 16);
          const float b = (u1 ? sum[3] : sum[1]) + __shfl_xor_sync(0xffffffffu, u1 ? sum[1] : sum[3], 16);
          float t = (u2 ? b : a) + __shfl_xor_sync(0xffffffffu, u2 ? a : b, 8);
          for (int off = 4; off > 0; off >>= 1) t += __shfl_xor_sync(0xffffffffu, t, off);
          // row-major: all candidates / statistics of a row are contiguous, so that the merge fetches a row in one go
          const int q = lane >> 3;
          if ((lane & 7) == 0 && (q == 0 ? act[0] : q == 1 ? act[1] : q == 2 ? act[2] : act[3])) {
            const size_t at = (size_t)(c0 + rb + NW * q) * p.cand_ld + blockIdx.x;
            p.cand_max[at] = q == 0 ? mx[0] : q == 1 ? mx[1] : q == 2 ? mx[2] : mx[3];
            p.cand_sum[at] = t;
          }
        }
        const size_t slot0 = ((size_t)(c0 + rb) * p.cand_ld + blockIdx.x) * K, slot4 = (size_t)NW * p.cand_ld * K;     // slot of row q: slot0 + q slot4
        if (K == 1) {                            // the maximum itself
#pragma unroll
          for (int q = 0; q < 4; q++) {
            const unsigned m = __reduce_max_sync(0xffffffffu, lm[q]);
            int id = -1;
#pragma unroll
            for (int j2 = 3; j2 >= 0; j2--)
              if (j2 < nv && key[q][j2] == m) id = tm * TILE_M + lane + 32 * j2;
            const unsigned w = __reduce_min_sync(0xffffffffu, (unsigned)id);
            if (act[q] && lane == 0) { p.cand_val[slot0 + q * slot4] = key_value(m); p.cand_idx[slot0 + q * slot4] = (int)w; }
          }
          continue;
        }
#pragma unroll
        for (int q = 0; q < 4; q++) {
          sk[q * 96 + lane] = lm[q];
          *(uint2 *)&sk[q * 96 + 32 + 2 * lane] = make_uint2(0u, 0x7fffffffu);     // an entry that ranks behind every value
        }
        __syncwarp();
        int above[4] = {0, 0, 0, 0};             // lane maxima larger than the lane's own
#pragma unroll
        for (int i = 0; i < 8; i++)
#pragma unroll
          for (int q = 0; q < 4; q++) {
            const uint4 w = *(const uint4 *)&sk[q * 96 + 4 * i];
            above[q] += (w.x > lm[q]) + (w.y > lm[q]) + (w.z > lm[q]) + (w.w > lm[q]);
          }
        int cnt[4];
#pragma unroll
        for (int q = 0; q < 4; q++) {
          // (with fewer than K lanes that have a feature each of them has one, and all are candidates)
          const unsigned bound = __reduce_min_sync(0xffffffffu, above[q] < K && nv > 0 ? lm[q] : 0xffffffffu);
          cnt[q] = 0;
#pragma unroll
          for (int j2 = 0; j2 < 4; j2++) {
            const bool in = j2 < nv && key[q][j2] >= bound;
            const unsigned m = __ballot_sync(0xffffffffu, in);
            const int at = cnt[q] + __popc(m & ((1u << lane) - 1u));
            if (in && at < 32) *(uint2 *)&sk[q * 96 + 32 + 2 * at] = make_uint2(key[q][j2], (unsigned)(tm * TILE_M + lane + 32 * j2));
            cnt[q] += __popc(m);
          }
        }
        __syncwarp();
        const int most = min(32, max(max(cnt[0], cnt[1]), max(cnt[2], cnt[3])));
        uint2 me[4];
        int rank[4] = {0, 0, 0, 0};
#pragma unroll
        for (int q = 0; q < 4; q++) me[q] = *(const uint2 *)&sk[q * 96 + 32 + 2 * lane];
#pragma unroll 4
        for (int i = 0; i < most; i++)
#pragma unroll
          for (int q = 0; q < 4; q++) {
            const uint2 w = *(const uint2 *)&sk[q * 96 + 32 + 2 * i];
            rank[q] += w.x > me[q].x || (w.x == me[q].x && w.y < me[q].y);
          }
#pragma unroll
        for (int q = 0; q < 4; q++) {
          if (!act[q]) continue;                 // uniform over the warp
          const size_t slot = slot0 + q * slot4;
          if (cnt[q] <= 32) {
            if (lane < cnt[q] && rank[q] < K) { p.cand_val[slot + rank[q]] = key_value(me[q].x); p.cand_idx[slot + rank[q]] = (int)me[q].y; }
            if (lane >= cnt[q] && lane < K) { p.cand_val[slot + lane] = 0.0f; p.cand_idx[slot + lane] = -1; }       // tile exhausted
          } else {                               // many equal values: the best of what is left, K times
            unsigned taken = 0u;
            for (int c = 0; c < K; c++) {
              unsigned bk = 0u;
              int bi = -1;
#pragma unroll
              for (int j2 = 0; j2 < 4; j2++) {
                const bool better = j2 < nv && !(taken >> j2 & 1u) && (bi < 0 || key[q][j2] > bk);      // equal: the lower feature stays
                bk = better ? key[q][j2] : bk;
                bi = better ? tm * TILE_M + lane + 32 * j2 : bi;
              }
              unsigned wk;
              const int wi = warp_best(bk, bi, &wk);
              if (wi >= 0 && bi == wi) taken |= 1u << ((wi - tm * TILE_M) >> 5);
              if (lane == 0) { p.cand_val[slot + c] = wi < 0 ? 0.0f : key_value(wk); p.cand_idx[slot + c] = wi; }
            }
          }
        }
        __syncwarp();
      }
    } else {   // EPI_ARGMAX
      if (good && p.out_f32 && o < p.O[0])
        for (int r = r0; r < r1; r++) p.out_f32[(size_t)(c0 + r) * p.ldo + o] = red[r * TILE_M + f] * inv_s[c0 + r];
      // thread t scans half of the tile's features for row t % 64, starting at a row-dependent feature
      // so that the 32 rows of a warp touch 32 different banks
      const int row = threadIdx.x & (CHUNK - 1), hf = threadIdx.x >> 6;
      float bv = 0.0f;
      int bi = -1;
      if (row < nrow) {
        for (int j = 0; j < 64; j++) {
          int ff = hf * 64 + ((j + row) & 63), oo = tm * TILE_M + ff;
          float v = red[row * TILE_M + ff];
          if (oo < p.O[0] && (bi < 0 || v > bv || (v == bv && oo < bi))) { bv = v; bi = oo; }
        }
      }
      if (hf == 1) { wpart[row] = bv; wpart[CHUNK + row] = __int_as_float(bi); }
      __syncthreads();
      if (hf == 0 && row < nrow && good) {
        float ov = wpart[row];
        int oi = __float_as_int(wpart[CHUNK + row]);
        if (oi >= 0 && (bi < 0 || ov > bv || (ov == bv && oi < bi))) { bv = ov; bi = oi; }
        p.best_val[(size_t)blockIdx.x * p.best_ld + c0 + row] = bv;
        p.best_idx[(size_t)blockIdx.x * p.best_ld + c0 + row] = bi;
      }
    }
    // peers may still be reading this CTA's red; nobody overwrites or leaves before all are done
    if (S > 1) asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); else __syncthreads();
  }
  if (*abort_flag && threadIdx.x == 0 && xr == 0) {
    // gave up on a wait: no bulk copy may still be landing in this CTA's shared memory when it exits.  Every stage
    // load that was issued and not seen complete is waited for (bounded; a load that was never issued runs the wait out).
    // (Pairs: the even CTA's barriers count both CTAs' bytes, and the odd CTA leaves only after the barrier below.)
    for (int i = *n_consumed; i < *n_issued; i++) mbar_wait(&full[i % stages], (i / stages) & 1, p.spin);
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  if (DUO) cluster_sync_all(); else __syncthreads();   // pairs: neither CTA frees tensor memory the other's MMAs may still use
  if (warp == 1) {
    if (DUO) asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(TMEM_COLS) : "memory");
    else asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(TMEM_COLS) : "memory");
  }
  if (p.stamp && threadIdx.x == 0) atomicMin(p.stamp + 1, ~global_ns());
}

// ----------------------------------------------------------------------------------------------
// Gate/up GEMM with SiLU(gate) * up for wide row tiles (129..256 token rows).  At this width the k-block of activations
// (32 KB) is twice a weight tile, and re-reading it from L2 for every weight tile is what bounds the loop.  Here ONE CTA
// owns the gate tile AND the up tile of the same 128 features: both MMAs of a k-block share one activation tile
// (64 KB per stage instead of 96), the two accumulators fill the tensor memory (2 x 256 columns), and since a thread
// then holds gate and up of its feature for every row the activation is applied straight from the accumulators:
// no cluster, no shared-memory round trip.
// DUO: two neighbouring feature tiles as a CTA pair (cta_group::2, cluster of 2): each CTA streams its own gate and up
// tile and HALF of the activation rows, the even CTA issues one M = 256 MMA per accumulator and k-step (fill bytes per
// k-block 48 KB instead of 64 KB per CTA, four stages instead of three).
// PAIR_THREADS threads: several threads share a feature (tensor-memory lane) and split the rows in the epilogue, which
// converts 2 x 256 accumulator columns per feature (with 128 threads it took a quarter of the launch).
// It serves spec_gemm_swiglu, and passes under the pair switch of the split-K kernel: the passes' own gate/up above 128 rows is the
// row-major kernel's (gemm_wide.cu), which is ahead at every row count (the table is beside row_major in api.cu).
constexpr int PAIR_THREADS = 512, PAIR_GROUPS = PAIR_THREADS / 128;
template <int NT, bool DUO = false>
__global__ void __launch_bounds__(PAIR_THREADS) gemm_swiglu_pair_kernel(const __grid_constant__ FusedParams p) {
  const int xrows = DUO ? p.nrt / 2 : p.nrt, STAGE = 2 * A_BYTES + xrows * TILE_K * 2;     // activation rows of this CTA, bytes of a stage
  constexpr int TMEM_COLS = 2 * NT;
  static_assert(TMEM_COLS <= 512, "two accumulators must fit the tensor memory");
  extern __shared__ unsigned char smem_raw[];
  unsigned char *tiles = (unsigned char *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  unsigned char *ctrl = tiles + p.ctrl_off;
  uint64_t *full = (uint64_t *)ctrl;
  uint64_t *empty = full + MAX_STAGES;
  uint64_t *acc_bar = empty + MAX_STAGES;
  uint32_t *tmem_slot = (uint32_t *)(acc_bar + 1);
  volatile uint32_t *abort_flag = tmem_slot + 1;
  volatile int *n_issued = (volatile int *)(tmem_slot + 2), *n_consumed = (volatile int *)(tmem_slot + 3);
  float *inv_s = (float *)(ctrl + 512);          // [256] per-row input scale

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int stages = p.stages, KB = p.KB;
  const int tm = blockIdx.x;                     // feature tile (of gate and of up)
  const uint32_t crank = DUO ? cluster_rank() : 0u;
  const int xr = (int)(crank & 1u);              // DUO: position in the pair (0 issues the MMAs)

  if (threadIdx.x == 0) {
    for (int i = 0; i < stages; i++) { mbar_init(&full[i], 1); mbar_init(&empty[i], 1); }
    mbar_init(acc_bar, 1);
    *abort_flag = 0;
    *n_issued = 0; *n_consumed = 0;
    if (DUO && crank != (blockIdx.x & 1u)) { *abort_flag = 1; set_status(p.status, ST_TIMEOUT, 224, blockIdx.x, (int)crank); }   // pairs = (even, odd) tile
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    if (DUO) {
      asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(TMEM_COLS)
                   : "memory");
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    } else {
      asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(TMEM_COLS)
                   : "memory");
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  if (DUO) cluster_sync_all(); else __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem_base = *tmem_slot;
  pdl_trigger();

  if (DUO && *abort_flag) {
    pdl_wait();
  } else if (DUO && warp == 0) {
    // ---- producer warp of a CTA pair: every byte of both CTAs is counted on the even CTA's full barrier
    const uint64_t pol = l2_policy_evict_first();
    const int npre = KB < stages ? KB : stages;
    if (elect_one())
      for (int i = 0; i < npre; i++) {
        unsigned char *a = tiles + i * STAGE;
        const uint32_t fb = mapa_u32(smem_u32(&full[i]), 0u);
        if (xr == 0) mbar_expect_tx(&full[i], 2 * STAGE);
        tma_load_2d_pair_hint(a, &p.map_w[0], i * TILE_K, tm * TILE_M, fb, pol);
        tma_load_2d_pair_hint(a + A_BYTES, &p.map_w[1], i * TILE_K, tm * TILE_M, fb, pol);
      }
    __syncwarp();
    pdl_wait();
    if (elect_one()) {
      if (p.stamp) atomicMin(p.stamp, global_ns());
      for (int i = 0; i < npre; i++)
        tma_load_2d_pair(tiles + i * STAGE + 2 * A_BYTES, &p.map_x, i * TILE_K, xr * xrows, mapa_u32(smem_u32(&full[i]), 0u));
    }
    __syncwarp();
    int i = npre, st = 0;
    uint32_t ph = 0;
    for (; i < KB; i++) {
      if (!mbar_wait_warp(&empty[st], ph, p.spin)) { *abort_flag = 1; set_status(p.status, ST_TIMEOUT, 225, blockIdx.x, i); break; }
      if (elect_one()) {
        unsigned char *a = tiles + st * STAGE;
        const uint32_t fb = mapa_u32(smem_u32(&full[st]), 0u);
        if (xr == 0) mbar_expect_tx(&full[st], 2 * STAGE);
        tma_load_2d_pair_hint(a, &p.map_w[0], i * TILE_K, tm * TILE_M, fb, pol);
        tma_load_2d_pair_hint(a + A_BYTES, &p.map_w[1], i * TILE_K, tm * TILE_M, fb, pol);
        tma_load_2d_pair(a + 2 * A_BYTES, &p.map_x, i * TILE_K, xr * xrows, fb);
      }
      __syncwarp();
      if (++st == stages) { st = 0; ph ^= 1u; }
    }
    if (lane == 0) *n_issued = i;
  } else if (!DUO && warp == 0) {
    // ---- producer warp (the elected lane issues): the weight tiles do not depend on the previous kernel
    const uint64_t pol = l2_policy_evict_first();
    const int npre = KB < stages ? KB : stages;
    if (elect_one())
      for (int i = 0; i < npre; i++) {
        unsigned char *a = tiles + i * STAGE;
        mbar_expect_tx(&full[i], STAGE);
        tma_load_2d_hint(a, &p.map_w[0], i * TILE_K, tm * TILE_M, &full[i], pol);
        tma_load_2d_hint(a + A_BYTES, &p.map_w[1], i * TILE_K, tm * TILE_M, &full[i], pol);
      }
    __syncwarp();
    pdl_wait();
    if (elect_one()) {
      if (p.stamp) atomicMin(p.stamp, global_ns());
      for (int i = 0; i < npre; i++) tma_load_2d(tiles + i * STAGE + 2 * A_BYTES, &p.map_x, i * TILE_K, 0, &full[i]);
    }
    __syncwarp();
    int i = npre, st = 0;
    uint32_t ph = 0;
    for (; i < KB; i++) {
      if (!mbar_wait_warp(&empty[st], ph, p.spin)) { *abort_flag = 1; set_status(p.status, ST_TIMEOUT, 220, blockIdx.x, i); break; }
      if (elect_one()) {
        unsigned char *a = tiles + st * STAGE;
        mbar_expect_tx(&full[st], STAGE);
        tma_load_2d_hint(a, &p.map_w[0], i * TILE_K, tm * TILE_M, &full[st], pol);
        tma_load_2d_hint(a + A_BYTES, &p.map_w[1], i * TILE_K, tm * TILE_M, &full[st], pol);
        tma_load_2d(a + 2 * A_BYTES, &p.map_x, i * TILE_K, 0, &full[st]);
      }
      __syncwarp();
      if (++st == stages) { st = 0; ph ^= 1u; }
    }
    if (lane == 0) *n_issued = i;
  } else {
    pdl_wait();
    if (DUO && warp == 1) {
      // ---- MMA issuer warp of a CTA pair (even CTA only): M = 256 over both CTAs' gate tiles, then both up tiles
      if (xr == 0) {
        const uint32_t idesc = umma_idesc_m(p.nrt, 2 * TILE_M);
        const uint32_t partner_base = ld_peer_u32(smem_u32(tmem_slot), 1u);
        if (partner_base != tmem_base) { *abort_flag = 1; set_status(p.status, ST_TIMEOUT, 226, blockIdx.x, (int)partner_base); }
        const uint64_t desc0 = umma_desc_sw128(smem_u32(tiles));
        int i = 0, st = 0;
        uint32_t ph = 0, ready = 0;
        if (!*abort_flag)
          for (; i < KB; i++) {
            if (!ready && !mbar_wait_warp(&full[st], ph, p.spin)) { *abort_flag = 1; set_status(p.status, ST_TIMEOUT, 227, blockIdx.x, i); break; }
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint64_t dg = desc0 + (uint64_t)((st * STAGE) >> 4), du = dg + (A_BYTES >> 4), db = dg + ((2 * A_BYTES) >> 4);
            int nst = st + 1;
            uint32_t nph = ph;
            if (nst == stages) { nst = 0; nph ^= 1u; }
            if (elect_one()) {
#pragma unroll
              for (int j = 0; j < TILE_K / UMMA_K; j++) {
                umma_bf16_pair(tmem_base, dg + 2 * j, db + 2 * j, idesc, (i | j) ? 1u : 0u);
                umma_bf16_pair(tmem_base + NT, du + 2 * j, db + 2 * j, idesc, (i | j) ? 1u : 0u);
              }
              umma_commit_pair(&empty[st], 0u);
            }
            __syncwarp();
            ready = mbar_test_warp(&full[nst], nph) ? 1u : 0u;
            st = nst; ph = nph;
          }
        if (lane == 0) *n_consumed = i;
        __syncwarp();
        if (!*abort_flag && elect_one()) umma_commit_pair(acc_bar, 0u);
      }
    } else if (!DUO && warp == 1) {
      // ---- MMA issuer warp (the elected lane issues): gate accumulator at column 0, up accumulator at column NT
      const uint32_t idesc = umma_idesc(p.nrt);
      const uint64_t desc0 = umma_desc_sw128(smem_u32(tiles));
      int i = 0, st = 0;
      uint32_t ph = 0, ready = 0;
      for (; i < KB; i++) {
        if (!ready && !mbar_wait_warp(&full[st], ph, p.spin)) { *abort_flag = 1; set_status(p.status, ST_TIMEOUT, 221, blockIdx.x, i); break; }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint64_t dg = desc0 + (uint64_t)((st * STAGE) >> 4), du = dg + (A_BYTES >> 4), db = dg + ((2 * A_BYTES) >> 4);
        int nst = st + 1;
        uint32_t nph = ph;
        if (nst == stages) { nst = 0; nph ^= 1u; }
        if (elect_one()) {
#pragma unroll
          for (int j = 0; j < TILE_K / UMMA_K; j++) {
            umma_bf16(tmem_base, dg + 2 * j, db + 2 * j, idesc, (i | j) ? 1u : 0u);
            umma_bf16(tmem_base + NT, du + 2 * j, db + 2 * j, idesc, (i | j) ? 1u : 0u);
          }
          umma_commit(&empty[st]);
        }
        __syncwarp();
        ready = mbar_test_warp(&full[nst], nph) ? 1u : 0u;
        st = nst; ph = nph;
      }
      if (lane == 0) *n_consumed = i;
      __syncwarp();
      if (elect_one()) umma_commit(acc_bar);
    } else if (warp >= 2) {
      for (int r = threadIdx.x - 64; r < p.rows; r += PAIR_THREADS - 64) {
        float sc = 1.0f;
        if (p.ssq_in) {
          float ss = 0.0f;
          for (int t = 0; t < p.ssq_in_tiles; t++) ss += p.ssq_in[(size_t)t * p.ssq_ld + r];
          sc = 1.0f / sqrtf(ss * p.inv_k_in + p.eps);
        }
        inv_s[r] = sc;
      }
    }
  }
  __syncthreads();

  int good = 0;
  if (lane == 0) {
    bool ok = *abort_flag ? false : mbar_wait(acc_bar, 0, p.spin);
    if (!ok && !*abort_flag) { *abort_flag = 1; set_status(p.status, ST_TIMEOUT, 222, blockIdx.x, 0); }
    good = (ok && !*abort_flag) ? 1 : 0;
  }
  good = __shfl_sync(0xffffffffu, good, 0);
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");

  // ---- epilogue: thread = feature f (tensor-memory lane), 16 rows (columns) of both accumulators at a time
  const int o = tm * TILE_M + (threadIdx.x & (TILE_M - 1));
  const int hw = threadIdx.x >> 7;               // which share of the rows (accumulator columns) this thread converts: every fourth 16
  if (good) {
#pragma unroll 1
    for (int cc = hw * 16; cc < p.rows; cc += PAIR_GROUPS * 16) {
      uint32_t g[16], u[16];
      tmem_ld16(tmem_base + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)cc, g);
      tmem_ld16(tmem_base + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)(NT + cc), u);
      if (o < p.O[0]) {
#pragma unroll
        for (int j = 0; j < 16; j++) {
          const int row = cc + j;
          if (row < p.rows) {
            const float sc = inv_s[row];
            const float gv = __uint_as_float(g[j]) * sc, uv = __uint_as_float(u[j]) * sc;
            p.act[(size_t)row * p.O[0] + o] = __float2bfloat16_rn((gv / (1.0f + expf(-gv))) * uv);
          }
        }
      }
    }
  }
  if (*abort_flag && threadIdx.x == 0 && xr == 0) {      // no bulk copy may still be landing when the CTA exits
    for (int i = *n_consumed; i < *n_issued; i++) mbar_wait(&full[i % stages], (i / stages) & 1, p.spin);
  }

  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  if (DUO) cluster_sync_all(); else __syncthreads();   // pairs: neither CTA frees tensor memory the other's MMAs may still use
  if (warp == 1) {
    if (DUO) asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(TMEM_COLS) : "memory");
    else asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(TMEM_COLS) : "memory");
  }
  if (p.stamp && threadIdx.x == 0) atomicMin(p.stamp + 1, ~global_ns());
}

// ---------------------------------------------------------------------------------------------- host side
int pick_nt(int rows) { return rows <= 16 ? 16 : rows <= 64 ? 64 : rows <= 128 ? 128 : 256; }

constexpr int TOPK_BYTES = 8 * 4 * 96 * 4;   // EPI_TOPK: selection scratch of up to eight warps
constexpr int NUM_SMS = 148;
constexpr int SMEM_ONE = 200 * 1024;      // ring budget with one CTA per SM
constexpr int SMEM_TWO = 104 * 1024;      // ring budget that lets two CTAs share an SM

struct Plan { int nt, tiles, S, stages, smem, ctrl_off, KB, chunk; bool pair, duo, mix; };

// K slices per feature tile.  An SM streams at a capped rate whether one or two CTAs feed it, so the time
// of a launch goes with (CTAs on the busiest SM) x (k-blocks per CTA + a fixed cost per CTA); two CTAs per SM
// are needed to hide one CTA's MMA and epilogue time behind the other's loads.
int g_target_ctas = 222;   // measured best on the 8B shapes (1.5 CTAs per SM)
constexpr int MAX_CLUSTER = 8;    // portable cluster sizes only: size 9 (non-portable) measured 20 % slower per step

// force_two: plan a wide tile (whose full ring takes the SM) as two CTAs per SM with two-stage rings
constexpr int NUM_GPCS = 8;
constexpr int MAX_BUMPED_CTAS = 266;   // 90 % of the 296 CTA slots: fuller grids fail to place all their clusters
// duo: neighbouring feature tiles as CTA pairs (clusters of 2 x Sk members; the stage holds half of the activation rows)
Plan make_plan(FusedEpi epi, const FusedGemmArgs &a, bool force_two = false, bool duo = false) {
  Plan pl;
  pl.duo = duo;
  pl.nt = pick_nt(a.rows);
  pl.KB = (a.I + TILE_K - 1) / TILE_K;
  pl.tiles = fused_gemm_tiles(epi, a);
  // gate/up up to 128 rows: gate and up features in one CTA (beyond: the pair kernel without K split)
  pl.pair = epi == EPI_SWIGLU && pl.nt <= 128;
  // Where pairs of whole tiles would be split in two over K (89 to 148 of them), tiles of 64 + 64 features give as many CTAs
  // without a cluster.  With fewer pairs (more K slices) the halved tiles alone would leave SMs idle; with more, one slice per
  // pair already fills the chip and reads the activations half as often (70B shapes: 224 pairs).
  pl.mix = pl.pair && a.split == 0 && a.stages == 0 && (g_target_ctas + pl.tiles / 2) / pl.tiles == 2;
  if (pl.mix) { pl.pair = false; pl.tiles = (a.O[0] + TILE_M / 2 - 1) / (TILE_M / 2); }
  const int stage = (pl.pair ? 2 : 1) * A_BYTES + (duo ? pl.nt / 2 : pl.nt) * TILE_K * 2;
  const int smax = MAX_CLUSTER / (duo ? 2 : 1);
  const bool wide = duo || SMEM_TWO / stage < (pl.pair ? 2 : 3);     // 256-row tiles: the ring of one CTA takes the SM
  const bool one_per_sm = wide && !force_two;
  const int target = one_per_sm ? NUM_SMS : g_target_ctas;   // one wave
  int Sk = 1;
  if (epi != EPI_ARGMAX) {
    Sk = one_per_sm ? target / std::max(1, pl.tiles)  // never more CTAs than SMs
                    : (target + pl.tiles / 2) / std::max(1, pl.tiles);   // nearest to the target CTA count
    Sk = std::max(1, std::min(Sk, smax));
    Sk = std::max(1, std::min(Sk, pl.KB / 4));
  }
  // One more K slice when that shortens the longest per-SM queue (CTAs per SM x k-blocks per CTA: with 64 tiles
  // of the 70B shapes, 4 slices make 256 CTAs of 112 k-blocks against 192 of 150) and every cluster can still be
  // placed in the first wave: a cluster lives inside one GPC, and with two CTAs per SM a GPC of at least 16 SMs holds 32 / S clusters of S CTAs.  (The
  // occupancy query counts one CTA per SM for these launches, so the bound is spelled out here.)
  if (!one_per_sm && epi != EPI_ARGMAX && a.split == 0) {
    auto queue = [&](int sk) { return ((pl.tiles * sk + NUM_SMS - 1) / NUM_SMS) * ((pl.KB + sk - 1) / sk); };
    const int up = Sk + 1, s_up = up;
    // only up to clusters of 4: with 7 -> 8 slices on the 8B shapes the longer reduction and the fuller grid (less
    // room for the next launch's early CTAs) cost more than the shorter queue saves (+2.6 % per step, measured)
    if (s_up <= 4 && up <= smax && up <= pl.KB / 4 && pl.tiles * s_up <= MAX_BUMPED_CTAS && pl.tiles <= NUM_GPCS * (32 / s_up) &&
        queue(up) < queue(Sk)) {
      Sk = up;
    }
  }
  if (pl.mix) Sk = 1;
  if (a.split > 0) Sk = std::max(1, std::min(std::min(a.split, smax), pl.KB));
  pl.S = Sk;
  // more tiles than SMs and a ring that fills the SM: two CTAs with two stages each beat two waves of one
  const int budget = !wide ? SMEM_TWO : ((force_two || pl.tiles * Sk > NUM_SMS) ? 2 * stage : SMEM_ONE);
  int stages = std::max(2, std::min(MAX_STAGES, budget / stage));
  if (a.stages > 0) stages = std::max(2, std::min(std::min(a.stages, MAX_STAGES), (220 * 1024) / stage));
  int per_slice = (pl.KB + Sk - 1) / Sk;
  stages = std::max(2, std::min(stages, per_slice));
  pl.stages = stages;
  // rows per epilogue round: accumulator dump [chunk][128] + this CTA's reduced rows; wide tiles take the most rows
  // the stage ring (free by then) holds, which saves cluster barriers
  auto epi_bytes = [&](int ch) {
    const int mine = epi == EPI_TOPK && pl.S > 1 ? (ch + pl.S - 1) / pl.S : 0;
    return ((pl.pair ? 2 : 1) * ch + mine) * TILE_M * 4 + (epi == EPI_TOPK ? TOPK_BYTES : 0);
  };
  pl.chunk = CHUNK;
  if (epi != EPI_ARGMAX)
    for (int ch = MAX_CHUNK; ch > CHUNK; ch >>= 1)
      if (ch <= pl.nt && epi_bytes(ch) <= std::max(stages * stage, 2 * CHUNK * TILE_M * 4)) { pl.chunk = ch; break; }
  pl.ctrl_off = (std::max(stages * stage, std::max(epi_bytes(pl.chunk), 2 * CHUNK * TILE_M * 4)) + 1023) & ~1023;
  pl.smem = pl.ctrl_off + 512 + 256 * 4 + 4 * MAX_CHUNK * 4 + 1024 /*alignment slack*/;
  return pl;
}

template <int NT, int EPI, bool PAIR = false, bool DUO = false, bool MIX = false>
int launch_inst(const FusedParams &p, const Plan &pl, bool pdl, cudaStream_t s) {
  static SmemLimit limit;
  if (!limit.ensure(gemm_fused_kernel<NT, EPI, PAIR, DUO, MIX>, pl.smem)) return -6;
  if (pl.S * (DUO ? 2 : 1) > 8 || (DUO && (pl.tiles & 1))) return -1;   // portable cluster sizes only; pairs need an even tile count
  if (!launch_allowed()) return 0;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(pl.tiles, pl.S, 1);
  cfg.blockDim = dim3(fused_threads(NT, EPI), 1, 1);
  cfg.dynamicSmemBytes = pl.smem;
  cfg.stream = s;
  cudaLaunchAttribute at[2];
  int na = 0;
  if (pl.S > 1 || DUO) {
    at[na].id = cudaLaunchAttributeClusterDimension;
    at[na].val.clusterDim.x = DUO ? 2 : 1; at[na].val.clusterDim.y = pl.S; at[na].val.clusterDim.z = 1;
    na++;
  }
  if (pdl) {
    at[na].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[na].val.programmaticStreamSerializationAllowed = 1;
    na++;
  }
  cfg.attrs = at;
  cfg.numAttrs = na;
  return cudaLaunchKernelEx(&cfg, gemm_fused_kernel<NT, EPI, PAIR, DUO, MIX>, p) == cudaSuccess ? 0 : -6;
}

// clusters of the plan's shape that can be resident at once (0: unknown)
template <int NT, int EPI>
int resident_clusters_inst(const Plan &pl) {
  static int cached_smem = -1, cached_S = -1, cached_n = 0;
  if (cached_smem == pl.smem && cached_S == pl.S) return cached_n;
  if (cudaFuncSetAttribute(gemm_fused_kernel<NT, EPI>, cudaFuncAttributeMaxDynamicSharedMemorySize, pl.smem) != cudaSuccess) return 0;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(pl.tiles, pl.S, 1);
  cfg.blockDim = dim3(fused_threads(NT, EPI), 1, 1);
  cfg.dynamicSmemBytes = pl.smem;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = 1; at[0].val.clusterDim.y = pl.S; at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  int n = 0;
  if (cudaOccupancyMaxActiveClusters(&n, gemm_fused_kernel<NT, EPI>, &cfg) != cudaSuccess) { cudaGetLastError(); n = 0; }
  cached_smem = pl.smem; cached_S = pl.S; cached_n = n;
  return n;
}
int resident_clusters_wide(FusedEpi epi, const Plan &pl) {
  if (pl.nt != 256) return 0;
  switch (epi) {
    case EPI_F32: return resident_clusters_inst<256, EPI_F32>(pl);
    case EPI_RESID: return resident_clusters_inst<256, EPI_RESID>(pl);
    case EPI_QKV: return resident_clusters_inst<256, EPI_QKV>(pl);
    default: return 0;
  }
}

template <int EPI>
int launch_epi(const FusedParams &p, const Plan &pl, bool pdl, cudaStream_t s) {
  switch (pl.nt) {
    case 16: return launch_inst<16, EPI>(p, pl, pdl, s);
    case 64: return launch_inst<64, EPI>(p, pl, pdl, s);
    case 128: return launch_inst<128, EPI>(p, pl, pdl, s);
    default: return launch_inst<256, EPI>(p, pl, pdl, s);
  }
}
int launch_swiglu_mix(const FusedParams &p, const Plan &pl, bool pdl, cudaStream_t s) {
  switch (pl.nt) {
    case 16: return launch_inst<16, EPI_SWIGLU, false, false, true>(p, pl, pdl, s);
    case 64: return launch_inst<64, EPI_SWIGLU, false, false, true>(p, pl, pdl, s);
    case 128: return launch_inst<128, EPI_SWIGLU, false, false, true>(p, pl, pdl, s);
    default: return -1;                // the pair kernel's
  }
}
int launch_swiglu_pair(const FusedParams &p, const Plan &pl, bool pdl, cudaStream_t s) {
  switch (pl.nt) {
    case 16: return launch_inst<16, EPI_SWIGLU, true>(p, pl, pdl, s);
    case 64: return launch_inst<64, EPI_SWIGLU, true>(p, pl, pdl, s);
    case 128: return launch_inst<128, EPI_SWIGLU, true>(p, pl, pdl, s);
    default: return -1;                // the pair kernel's
  }
}

}  // namespace

void fused_gemm_set_target_ctas(int n) { g_target_ctas = n; }
// 256-row tiles of neighbouring feature tiles as CTA pairs.  Bit 0: the split-K kernel (measured no faster: off); bit 1: the
// gate/up kernel (gate/up launch -1 %, C3 step -0.6 %: on)
namespace { int g_pairs = 0, g_pairs_swiglu = 1; }
int fused_gemm_pairs() { return g_pairs; }
void fused_gemm_set_pairs(int on) { g_pairs = on & 1; g_pairs_swiglu = (on >> 1) & 1; }

int fused_gemm_tiles(FusedEpi epi, const FusedGemmArgs &a) {
  if (epi == EPI_SWIGLU) return (a.O[0] + TILE_M - 1) / TILE_M;
  int t = 0;
  for (int j = 0; j < a.nw; j++) t += (a.O[j] + TILE_M - 1) / TILE_M;
  return t;
}

bool fused_gemm_supported(FusedEpi epi, const FusedGemmArgs &a) {
  if (a.rows < 1 || a.rows > 256 || a.I < 8 || (a.I % 8) != 0 || ((uintptr_t)a.x & 15)) return false;
  int need = epi == EPI_QKV ? 3 : epi == EPI_SWIGLU ? 2 : 1;
  if (a.nw != need) return false;
  for (int j = 0; j < a.nw; j++)
    if (!a.w[j] || ((uintptr_t)a.w[j] & 15) || a.O[j] < 1) return false;
  // gate/up beyond 128 rows is the pair kernel's, which has one slice and a ring of its own
  if (epi == EPI_SWIGLU && (a.O[0] != a.O[1] || (a.rows > 128 && (a.split || a.stages)))) return false;
  if (epi == EPI_RESID && (a.O[0] & 7)) return false;
  if (epi == EPI_TOPK && (a.topk < 1 || a.topk > 16 || !a.cand_val || !a.cand_idx || !a.cand_max || !a.cand_sum || a.cand_ld < (a.O[0] + TILE_M - 1) / TILE_M)) return false;
  if (epi == EPI_QKV) {
    if (a.hd < 8 || a.hd > TILE_M || (a.hd & (a.hd - 1))) return false;
    if (a.O[0] != a.H * a.hd || a.O[1] != a.G * a.hd || a.O[2] != a.G * a.hd) return false;
  }
  return true;
}

int fused_gemm_launch(TmaMaps *g, FusedEpi epi, const FusedGemmArgs &a, cudaStream_t s) {
  if (!g || !fused_gemm_supported(epi, a)) return -1;
  Plan pl = make_plan(epi, a);
  // 256 rows: CTA pairs when every weight's tile count is even (pairs never straddle two weights)
  bool duo = g_pairs && pl.nt == 256 && (epi == EPI_F32 || epi == EPI_RESID || epi == EPI_QKV);
  for (int j = 0; j < a.nw; j++) duo = duo && (a.O[j] % (2 * TILE_M)) == 0;
  if (duo) pl = make_plan(epi, a, false, true);
  if (!duo && pl.nt == 256 && pl.S > 1 && a.split == 0 && a.stages == 0 && pl.tiles * pl.S <= NUM_SMS) {
    // clusters are placed inside one GPC: a grid that counts fewer CTAs than SMs can still need a second wave
    const int fit = resident_clusters_wide(epi, pl);
    if (fit > 0 && pl.tiles > fit) pl = make_plan(epi, a, true);
  }
  FusedParams p;
  memset(&p, 0, sizeof p);
  for (int j = 0; j < a.nw; j++) {
    const CUtensorMap *mw = tma_maps_get(g, a.w[j], a.O[j], a.I, pl.mix ? TILE_M / 2 : TILE_M);
    if (!mw) return -6;
    p.map_w[j] = *mw;
    p.O[j] = a.O[j];
  }
  const CUtensorMap *mx = tma_maps_get(g, a.x, a.rows, a.I, duo ? pl.nt / 2 : pl.nt);   // pairs: each CTA loads half of the rows
  if (!mx) return -6;
  p.map_x = *mx;
  p.tiles0 = (a.O[0] + TILE_M - 1) / TILE_M;
  p.tiles1 = p.tiles0 + (a.nw > 1 ? (a.O[1] + TILE_M - 1) / TILE_M : 0);
  p.rows = a.rows; p.KB = pl.KB; p.S = pl.S; p.stages = pl.stages; p.ctrl_off = pl.ctrl_off; p.chunk = pl.chunk;
  p.ssq_in = a.ssq_in; p.ssq_in_tiles = a.ssq_in_tiles; p.ssq_ld = a.ssq_ld; p.inv_k_in = 1.0f / (float)a.k_in; p.eps = a.eps;
  p.out_f32 = a.out_f32; p.ldo = a.ldo;
  p.xres = a.xres; p.gain = a.gain; p.hb = a.hb; p.ssq_out = a.ssq_out; p.taps = a.tap_mask ? a.taps : nullptr;
  p.tap_mask = a.taps ? a.tap_mask : 0; p.resid_add = a.resid_add;
  p.cs = a.cs; p.m = a.m; p.q = a.q; p.pool = a.pool; p.pm = a.pm; p.H = a.H; p.G = a.G; p.hd = a.hd;
  p.act = a.act;
  const uintptr_t va = epi == EPI_RESID ? (uintptr_t)a.gain : epi == EPI_SWIGLU ? (uintptr_t)a.act | (unsigned)(a.O[0] * 2) : (uintptr_t)a.out_f32 | (unsigned)(a.ldo * 4);
  p.vec = (va & (epi == EPI_F32 ? 15 : 7)) == 0;
  p.best_val = a.best_val; p.best_idx = a.best_idx; p.best_ld = a.best_ld;
  p.topk = a.topk; p.cand_val = a.cand_val; p.cand_max = a.cand_max; p.cand_sum = a.cand_sum; p.cand_idx = a.cand_idx;
  p.cand_ld = a.cand_ld; p.want_rows = a.want_rows; p.n_want = a.n_want;
  p.status = a.status;
  p.stamp = a.stamp;
  p.spin = a.spin_limit ? a.spin_limit : SPIN_LIMIT;
  p.withhold = a.withhold ? 1 : 0;
  if (epi == EPI_SWIGLU && pl.nt == 256) {
    // wide rows: one CTA per (gate tile, up tile) pair sharing the activation tiles; optionally two such CTAs as a
    // CTA pair that also share the activation k-block (each loads half of the rows)
    const bool duo2 = g_pairs_swiglu && (p.tiles0 % 2) == 0;
    p.nrt = (a.rows + 15) & ~15;                 // N of an MMA is a multiple of 16
    const int xrows = duo2 ? p.nrt / 2 : p.nrt, stage2 = 2 * A_BYTES + xrows * TILE_K * 2;
    const CUtensorMap *mxh = tma_maps_get(g, a.x, a.rows, a.I, xrows);
    if (!mxh) return -6;
    p.map_x = *mxh;
    p.stages = std::max(2, std::min(SMEM_ONE / stage2, pl.KB));
    p.S = 1;
    p.ctrl_off = (p.stages * stage2 + 1023) & ~1023;
    const int smem = p.ctrl_off + 512 + 256 * 4 + 1024;
    static SmemLimit limit, limit_duo;
    if (!(duo2 ? limit_duo.ensure(gemm_swiglu_pair_kernel<256, true>, smem) : limit.ensure(gemm_swiglu_pair_kernel<256>, smem))) return -6;
    if (!launch_allowed()) return 0;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(p.tiles0, 1, 1);
    cfg.blockDim = dim3(PAIR_THREADS, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at[2];
    int na = 0;
    if (duo2) {
      at[na].id = cudaLaunchAttributeClusterDimension;
      at[na].val.clusterDim.x = 2; at[na].val.clusterDim.y = 1; at[na].val.clusterDim.z = 1;
      na++;
    }
    if (a.pdl) {
      at[na].id = cudaLaunchAttributeProgrammaticStreamSerialization;
      at[na].val.programmaticStreamSerializationAllowed = 1;
      na++;
    }
    cfg.attrs = at;
    cfg.numAttrs = na;
    if (duo2) return cudaLaunchKernelEx(&cfg, gemm_swiglu_pair_kernel<256, true>, p) == cudaSuccess ? 0 : -6;
    return cudaLaunchKernelEx(&cfg, gemm_swiglu_pair_kernel<256>, p) == cudaSuccess ? 0 : -6;
  }
  if (duo) {
    switch (epi) {
      case EPI_F32: return launch_inst<256, EPI_F32, false, true>(p, pl, a.pdl, s);
      case EPI_RESID: return launch_inst<256, EPI_RESID, false, true>(p, pl, a.pdl, s);
      default: return launch_inst<256, EPI_QKV, false, true>(p, pl, a.pdl, s);
    }
  }
  switch (epi) {
    case EPI_F32: return launch_epi<EPI_F32>(p, pl, a.pdl, s);
    case EPI_RESID: return launch_epi<EPI_RESID>(p, pl, a.pdl, s);
    case EPI_QKV: return launch_epi<EPI_QKV>(p, pl, a.pdl, s);
    case EPI_SWIGLU: return pl.mix ? launch_swiglu_mix(p, pl, a.pdl, s) : launch_swiglu_pair(p, pl, a.pdl, s);
    case EPI_TOPK: return launch_epi<EPI_TOPK>(p, pl, a.pdl, s);
    default: return launch_epi<EPI_ARGMAX>(p, pl, a.pdl, s);
  }
}

}  // namespace spec
