// bf16 GEMM with fused epilogues for many token rows (prefill), sm_100a.
//
//   out[r][o] = sum_i x[r][i] * w[o][i],  hundreds to thousands of rows
//
// From about 215 rows on the contraction is bound by the tensor pipe, no longer by the weight stream, so this kernel is
// the mirror image of the weight-streaming one (gemm_fused.cu): token rows are the UMMA M side, features the N side.
//
//  * a CTA pair (cta_group::2) owns a tile of 256 rows x 256 features: each CTA stages its own 128 rows and half of the
//    features per 64-element k-block (32 KB, six stages), so a k-block costs 64 bytes of shared-memory fill per tensor
//    cycle, which the L2 can deliver; one M = 256, N = 256 MMA per 16 elements;
//  * the kernel is persistent (one pair per two SMs, tiles dealt out in order, row tiles fastest so that the pairs that
//    run together share their weights in L2), and the 512 tensor-memory columns hold two accumulators: the epilogue of a
//    tile runs under the main loop of the next one;
//  * a thread of the epilogue owns one token row (tensor-memory lane), so the RMSNorm factor, the cache slot and the RoPE
//    row are one value per thread; the values cross to row-contiguous order through 4 KB of shared memory per warp, so
//    that every global access of the epilogue moves whole 64- or 128-byte runs.
//
// Measured with the packing of prompts into passes (one B200, whole requests, before: one prompt at a time in passes of 256
// rows on the weight-streaming kernel): 64 prompts of 64..768 tokens, 8 layers of the 8B shapes, 24 chain steps 306 -> 156 ms;
// 56 prompts of 16..96 tokens, 16 layers 268 -> 104 ms; 16384 tokens, 32 layers 535 -> 292 ms.
//
// Every mbarrier wait is bounded and answers a warp as one; on a time-out the CTA records it, stops, waits (bounded) for the copies in flight, keeps
// its cluster barriers and frees its tensor memory.
#include <cuda.h>
#include <string.h>

#include <algorithm>

#include "gemm_wide.cuh"
#include "tcgen05_ptx.cuh"

namespace spec {

thread_local int tl_wide_test = WIDE_TEST_OFF;

namespace {

using namespace tc;

constexpr int W_HALF = 128;                               // rows of a CTA / features of a half tile
constexpr int W_A_BYTES = W_HALF * TILE_K * 2;            // 16 KB: the CTA's rows of a k-block
constexpr int W_STAGE = 2 * W_A_BYTES;                    // + its half of the features
constexpr int W_STAGES = 6;
constexpr int W_EPI_WARPS = 8;                            // two per quarter of the tensor-memory lanes: one per half tile
constexpr int W_THREADS = (W_EPI_WARPS + 2) * 32;
constexpr int W_STG = 32 * 128;                           // staging bytes per epilogue warp: 32 rows x 128 B
constexpr int W_CTRL = 256;
constexpr int W_SMEM = W_STAGES * W_STAGE + W_EPI_WARPS * W_STG + W_CTRL + 1024 /*alignment slack*/;
constexpr int W_PAIRS = 74;                               // 148 SMs

struct alignas(64) WideParams {
  CUtensorMap map_x, map_w[3];
  int rows, KB, m_tiles, n_tiles;
  int half;                      // rows of a CTA: 128, or with one row tile half of the rows there are (split and gate/up kernel)
  int h0, h1;                    // half tiles [0,h0) belong to w0, [h0,h1) to w1, the rest to w2
  int O[3];
  int kind0;                     // WIDE_QKV: what w0 is (0 q, 1 k)
  const float *ssq_in; int ssq_in_tiles, ssq_ld; float inv_k_in, eps;
  float *xres; const bf16 *gain; int gain_vec; bf16 *hb; float *ssq_out; bf16 *taps; int tap_mask, resid_add;
  const float2 *cs; const int32_t *slot, *seq, *kvpos; PageMap pm; bf16 *q; bf16 *kp, *vp; int H, G, page_size;
  bf16 *act;
  bf16 *out_b; int ldo;
  float *out_f32;
  float *best_val; int32_t *best_idx; int best_ld;
  int fpt, stages;               // gate/up kernel with tiles of a chosen width: features per tile, ring stages
  int32_t *status;
  unsigned long long *stamp;
  int hold;                      // test hook: block 0 leaves out the activations of its first k-block
  uint32_t spin;                 // polls before a wait gives up
};

// cache row of a row's K/V (-1: none); seq: the row's sequence, negative for padding (1 where the caller gave slots: a real row)
__device__ __forceinline__ int row_slot(const WideParams &p, int row, int *seq) {
  if (p.slot) { *seq = 1; return p.slot[row]; }
  *seq = p.seq[row];
  if (*seq < 0) return -1;
  const int kvpos = p.kvpos[row];
  if (kvpos < 0 || kvpos / p.pm.page_size >= p.pm.pages_per_seq) { set_status(p.status, ST_BOUNDS, 1, row, kvpos); return -1; }
  const int page = p.pm.table[(size_t)*seq * p.pm.pages_per_seq + kvpos / p.pm.page_size];
  if (page < 0 || page >= p.pm.num_pages) { set_status(p.status, ST_BOUNDS, 2, row, page); return -1; }
  return page * p.G * p.pm.page_size + kvpos % p.pm.page_size;
}
__device__ __forceinline__ float row_scale(const WideParams &p, int row) {
  if (!p.ssq_in) return 1.0f;
  float ss = 0.0f;
#pragma unroll 8
  for (int u = 0; u < p.ssq_in_tiles; u++) ss += p.ssq_in[(size_t)u * p.ssq_ld + row];
  return 1.0f / sqrtf(ss * p.inv_k_in + p.eps);
}

// norm gains of features f .. f + 3; they are the caller's, who owes them no alignment beyond their own two bytes
__device__ __forceinline__ float4 load_gain(const WideParams &p, int f) {
  const bf16 *g = p.gain + f;
  if (!p.gain_vec) return make_float4(to_f32(g[0]), to_f32(g[1]), to_f32(g[2]), to_f32(g[3]));
  const uint2 u = *(const uint2 *)g;
  const float2 g01 = __bfloat1622float2(*(const __nv_bfloat162 *)&u.x), g23 = __bfloat1622float2(*(const __nv_bfloat162 *)&u.y);
  return make_float4(g01.x, g01.y, g23.x, g23.y);
}

__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// one arrival on an mbarrier of the cluster (shared::cluster address), releasing this thread's earlier work
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t addr) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(addr) : "memory");
}
// bounded wait for arrivals that come from both CTAs of the pair (cluster-scope acquire)
__device__ __forceinline__ bool mbar_wait_cluster(uint64_t *bar, uint32_t parity, uint32_t limit) {
  const uint32_t addr = smem_u32(bar);
  for (uint32_t it = 0; it < limit; it++) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(addr), "r"(parity)
        : "memory");
    if (ok) return true;
  }
  return false;
}
// 32 consecutive columns of this thread's tensor-memory lane; tmem_ld_wait() before the values are used
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&v)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, %17, %18, "
      "%19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]), "=r"(v[9]),
        "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]), "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]),
        "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]), "=r"(v[24]), "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]),
        "=r"(v[30]), "=r"(v[31])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t pack2(float a, float b) {
  __nv_bfloat162 v = __floats2bfloat162_rn(a, b);
  return *(uint32_t *)&v;
}
__device__ __forceinline__ uint2 pack4(float4 v) { return make_uint2(pack2(v.x, v.y), pack2(v.z, v.w)); }

// 32 values of every lane's own row -> row-contiguous order: afterwards lane l holds, in t[i], columns 4 (l % 8) .. + 3 of
// row 4 i + l / 8.  stg: the warp's 4 KB, 16-byte chunks swizzled by the row.
__device__ __forceinline__ void transpose32(unsigned char *stg, int lane, const uint32_t (&v)[32], float4 (&t)[8]) {
#pragma unroll
  for (int j = 0; j < 8; j++)
    *(uint4 *)(stg + lane * 128 + ((j ^ (lane & 7)) << 4)) = make_uint4(v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3]);
  __syncwarp();
#pragma unroll
  for (int i = 0; i < 8; i++) {
    const int r = i * 4 + (lane >> 3);
    t[i] = *(const float4 *)(stg + r * 128 + (((lane & 7) ^ (r & 7)) << 4));
  }
  __syncwarp();
}

template <int EPI>
__global__ void __launch_bounds__(W_THREADS, 1) gemm_wide_kernel(const __grid_constant__ WideParams p) {
  extern __shared__ unsigned char smem_raw[];
  unsigned char *ring = (unsigned char *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  unsigned char *stg_all = ring + W_STAGES * W_STAGE;
  uint64_t *full = (uint64_t *)(stg_all + W_EPI_WARPS * W_STG);
  uint64_t *empty = full + W_STAGES;
  uint64_t *tfull = empty + W_STAGES, *tempty = tfull + 2;
  uint32_t *tmem_slot = (uint32_t *)(tempty + 2);
  volatile uint32_t *abort_flag = tmem_slot + 1;
  volatile int *n_issued = (volatile int *)(tmem_slot + 2), *n_consumed = (volatile int *)(tmem_slot + 3);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  uint32_t crank;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(crank));
  const int xr = (int)(crank & 1u);
  const int pair = blockIdx.x >> 1, n_pairs = gridDim.x >> 1;
  const int ntiles = p.m_tiles * p.n_tiles, KB = p.KB;

  if (threadIdx.x == 0) {
    for (int i = 0; i < W_STAGES; i++) { mbar_init(&full[i], 1); mbar_init(&empty[i], 1); }
    for (int i = 0; i < 2; i++) { mbar_init(&tfull[i], 1); mbar_init(&tempty[i], 2 * W_EPI_WARPS); }
    *abort_flag = 0;
    *n_issued = 0; *n_consumed = 0;
    // the pair is (even, odd) blocks with ranks 0, 1: checked, never assumed
    if (crank != (blockIdx.x & 1u)) { *abort_flag = 1; set_status(p.status, ST_TIMEOUT, 244, blockIdx.x, (int)crank); }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == W_EPI_WARPS + 1) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(512) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  cluster_sync_all();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem_base = *tmem_slot;        // 512 columns: the whole tensor memory, so both CTAs start at column 0
  if (EPI != WIDE_QKV) pdl_trigger();            // WIDE_QKV: after the wait, see gemm_fused_kernel

  if (warp == W_EPI_WARPS) {
    // ================================================================ producer (converged warp, the elected lane issues)
    const uint64_t pol = l2_policy_evict_first();
    int issued = 0, st = 0;
    uint32_t ph = 1;                             // a stage's first use needs no wait: the preceding phase counts as complete
    bool ok = !__any_sync(0xffffffffu, *abort_flag != 0), first = true;
    for (int t = pair; t < ntiles && ok; t += n_pairs) {
      const int mt = t % p.m_tiles, nt = t / p.m_tiles;
      int mi = 0, tm = nt;
      if (EPI == WIDE_SWIGLU) mi = xr;
      else {
        tm = 2 * nt + xr;
        if (tm >= p.h1) { mi = 2; tm -= p.h1; }
        else if (tm >= p.h0) { mi = 1; tm -= p.h0; }
      }
      const CUtensorMap *mw = &p.map_w[mi];
      const int wrow = tm * W_HALF, xrow = mt * WIDE_ROWS + xr * W_HALF;
      int kb = 0;
      if (first) {
        // the weights do not depend on the previous kernel: fill the ring with them, then wait for the activations
        first = false;
        const int npre = KB < W_STAGES ? KB : W_STAGES;
        if (elect_one())
          for (int i = 0; i < npre; i++) {
            if (xr == 0) mbar_expect_tx(&full[i], 2 * W_STAGE);
            tma_load_2d_pair_hint(ring + i * W_STAGE + W_A_BYTES, mw, i * TILE_K, wrow, mapa_u32(smem_u32(&full[i]), 0u), pol);
          }
        __syncwarp();
        pdl_wait();
        if (EPI == WIDE_QKV) pdl_trigger();
        if (elect_one())
          for (int i = p.hold && blockIdx.x == 0 ? 1 : 0; i < npre; i++) tma_load_2d_pair(ring + i * W_STAGE, &p.map_x, i * TILE_K, xrow, mapa_u32(smem_u32(&full[i]), 0u));
        __syncwarp();
        kb = npre; issued = npre;
        if (npre == W_STAGES) ph = 0; else st = npre;
      }
      for (; kb < KB; kb++) {
        if (!mbar_wait_warp(&empty[st], ph, p.spin)) { *abort_flag = 1; set_status(p.status, ST_TIMEOUT, 240, blockIdx.x, t); ok = false; break; }
        if (elect_one()) {
          unsigned char *a = ring + st * W_STAGE;
          const uint32_t fb = mapa_u32(smem_u32(&full[st]), 0u);
          if (xr == 0) mbar_expect_tx(&full[st], 2 * W_STAGE);
          const int kx = kb * TILE_K;
          tma_load_2d_pair_hint(a + W_A_BYTES, mw, kx, wrow, fb, pol);
          tma_load_2d_pair(a, &p.map_x, kx, xrow, fb);
        }
        __syncwarp();
        issued++;
        if (++st == W_STAGES) { st = 0; ph ^= 1u; }
      }
    }
    if (first) pdl_wait();
    if (lane == 0) *n_issued = issued;
  } else if (warp == W_EPI_WARPS + 1) {
    // ================================================================ MMA issuer (even CTA only)
    pdl_wait();
    if (EPI == WIDE_QKV) pdl_trigger();
    if (xr == 0 && !__any_sync(0xffffffffu, *abort_flag != 0)) {
      constexpr uint32_t idesc = umma_idesc_m(256, 256);
      const uint64_t desc0 = umma_desc_sw128(smem_u32(ring));
      int consumed = 0, st = 0, it = 0;
      uint32_t ph = 0, ready = 0;
      bool ok = true;
      for (int t = pair; t < ntiles && ok; t += n_pairs, it++) {
        const int acc = it & 1, use = it >> 1;
        if (use > 0) {                           // both CTAs' epilogues have emptied this accumulator
          const bool w = mbar_wait_cluster(&tempty[acc], (uint32_t)((use - 1) & 1), p.spin);
          if (!__all_sync(0xffffffffu, w)) { *abort_flag = 1; set_status(p.status, ST_TIMEOUT, 241, blockIdx.x, t); break; }
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        }
        const uint32_t d = tmem_base + (uint32_t)(acc * 256);
        for (int kb = 0; kb < KB; kb++) {
          if (!ready && !mbar_wait_warp(&full[st], ph, p.spin)) { *abort_flag = 1; set_status(p.status, ST_TIMEOUT, 242, blockIdx.x, t); ok = false; break; }
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          const uint64_t da = desc0 + (uint64_t)((st * W_STAGE) >> 4), db = da + (W_A_BYTES >> 4);
          int nst = st + 1;
          uint32_t nph = ph;
          if (nst == W_STAGES) { nst = 0; nph ^= 1u; }
          if (elect_one()) {
#pragma unroll
            for (int j = 0; j < TILE_K / UMMA_K; j++) umma_bf16_pair(d, da + 2 * j, db + 2 * j, idesc, (kb | j) ? 1u : 0u);
            umma_commit_pair(&empty[st], 0u);    // frees the stage in both CTAs
            if (kb == KB - 1) umma_commit_pair(&tfull[acc], 0u);
          }
          __syncwarp();
          consumed++;
          ready = mbar_test_warp(&full[nst], nph) ? 1u : 0u;
          st = nst; ph = nph;
        }
      }
      if (lane == 0) *n_consumed = consumed;
    }
  } else {
    // ================================================================ epilogue: thread = token row, warp / 4 = half tile
    pdl_wait();
    if (EPI == WIDE_QKV) pdl_trigger();
    if (p.stamp && threadIdx.x == 0) atomicMin(p.stamp, global_ns());
    unsigned char *stg = stg_all + warp * W_STG;
    const int quarter = warp & 3, half = warp >> 2;
    const int sub = lane >> 3, c4 = (lane & 7) * 4;              // place in row-contiguous order: rows 4 i + sub, columns c4 ..
    int it = 0;
    for (int t = pair; t < ntiles; t += n_pairs, it++) {
      const int acc = it & 1, use = it >> 1;
      const int mt = t % p.m_tiles, nt = t / p.m_tiles;
      const int row_w = mt * WIDE_ROWS + xr * W_HALF + quarter * 32;        // first row of the warp
      const int row = row_w + lane;
      const bool any_row = row_w < p.rows;
      const float inv = row < p.rows ? row_scale(p, row) : 1.0f;
      int slot = -1, seq = -1;
      if (EPI == WIDE_QKV && row < p.rows) slot = row_slot(p, row, &seq);
      // everything that does not depend on the accumulator is requested before the wait for it
      float4 xin[8];
      const int fo0 = nt * 256 + half * 128;                     // WIDE_RESID / WIDE_BF16: first feature of the warp
      if (EPI == WIDE_RESID && p.resid_add && any_row) {
#pragma unroll
        for (int i = 0; i < 8; i++) {
          const int gr = row_w + i * 4 + sub, f = fo0 + c4;
          xin[i] = (gr < p.rows && f < p.O[0]) ? *(const float4 *)(p.xres + (size_t)gr * p.O[0] + f) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
      }
      const bool ok = __all_sync(0xffffffffu, mbar_wait_warp(&tfull[acc], (uint32_t)(use & 1), p.spin) && !*abort_flag);
      if (!ok) {
        if (lane == 0) { *abort_flag = 1; set_status(p.status, ST_TIMEOUT, 243, blockIdx.x, t); }
        break;
      }
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const uint32_t ta = tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(acc * 256);
      if (EPI == WIDE_RESID || EPI == WIDE_BF16 || EPI == WIDE_F32) {
        float sq[8];
#pragma unroll
        for (int i = 0; i < 8; i++) sq[i] = 0.0f;
#pragma unroll
        for (int c = 0; c < 4; c++) {
          uint32_t v[32];
          tmem_ld32(ta + half * 128 + c * 32, v);
          float4 a[8];
          transpose32(stg, lane, v, a);
          const int f = fo0 + c * 32 + c4;
          const bool fok = f < p.O[0];
          if (EPI == WIDE_F32) {
#pragma unroll
            for (int i = 0; i < 8; i++) {
              const int r = i * 4 + sub, gr = row_w + r;
              const float sc = __shfl_sync(0xffffffffu, inv, r);
              if (gr < p.rows && fok) *(float4 *)(p.out_f32 + (size_t)gr * p.ldo + f) = make_float4(a[i].x * sc, a[i].y * sc, a[i].z * sc, a[i].w * sc);
            }
          } else if (EPI == WIDE_BF16) {
#pragma unroll
            for (int i = 0; i < 8; i++) {
              const int gr = row_w + i * 4 + sub;
              if (gr < p.rows && fok) *(uint2 *)(p.out_b + (size_t)gr * p.ldo + f) = pack4(a[i]);
            }
          } else {
            float4 xn[8];                         // the next 32 columns of the residual, in flight during this round
            if (c < 3 && p.resid_add && any_row) {
#pragma unroll
              for (int i = 0; i < 8; i++) {
                const int gr = row_w + i * 4 + sub;
                xn[i] = (gr < p.rows && f + 32 < p.O[0]) ? *(const float4 *)(p.xres + (size_t)gr * p.O[0] + f + 32) : make_float4(0.f, 0.f, 0.f, 0.f);
              }
            }
            float4 gn = make_float4(0.f, 0.f, 0.f, 0.f);
            if (fok) gn = load_gain(p, f);
#pragma unroll
            for (int i = 0; i < 8; i++) {
              const int gr = row_w + i * 4 + sub;
              float4 o = a[i];
              if (p.resid_add) { o.x += xin[i].x; o.y += xin[i].y; o.z += xin[i].z; o.w += xin[i].w; }
              if (gr < p.rows && fok) {
                const size_t xi = (size_t)gr * p.O[0] + f;
                *(float4 *)(p.xres + xi) = o;
                *(uint2 *)(p.hb + xi) = pack4(make_float4(o.x * gn.x, o.y * gn.y, o.z * gn.z, o.w * gn.w));
                if (p.tap_mask) {
                  const uint2 tb = pack4(o);
#pragma unroll
                  for (int s = 0; s < 3; s++)
                    if ((p.tap_mask >> s) & 1) *(uint2 *)(p.taps + (size_t)gr * 3 * p.O[0] + (size_t)s * p.O[0] + f) = tb;
                }
                sq[i] += (o.x * o.x + o.y * o.y) + (o.z * o.z + o.w * o.w);
              }
              if (c < 3) xin[i] = xn[i];
            }
          }
        }
        if (EPI == WIDE_RESID) {
#pragma unroll
          for (int i = 0; i < 8; i++) {
            float s = sq[i];
            for (int off = 4; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
            const int gr = row_w + i * 4 + sub;
            if ((lane & 7) == 0 && gr < p.rows && fo0 < p.O[0]) p.ssq_out[(size_t)(fo0 >> 7) * p.ssq_ld + gr] = s;
          }
        }
      } else if (EPI == WIDE_SWIGLU) {
        // this warp: gate columns 64 half .. + 63, up columns 128 + the same, of features 128 nt + 64 half ..
        const int f0 = nt * 128 + half * 64;
#pragma unroll
        for (int c = 0; c < 2; c++) {
          if (!any_row) break;                                   // uniform over the warp
          uint32_t g[32], u[32];
          tmem_ld32(ta + half * 64 + c * 32, g);
          tmem_ld32(ta + 128 + half * 64 + c * 32, u);
#pragma unroll
          for (int j = 0; j < 4; j++) {
            uint32_t w[4];
#pragma unroll
            for (int e = 0; e < 4; e++) {
              float r[2];
#pragma unroll
              for (int z = 0; z < 2; z++) {
                // (a lane without a row divides 1: see gemm_wide_swiglu_kernel)
                const float gv = row < p.rows ? __uint_as_float(g[8 * j + 2 * e + z]) * inv : 1.0f, uv = __uint_as_float(u[8 * j + 2 * e + z]) * inv;
                r[z] = (gv / (1.0f + expf(-gv))) * uv;
              }
              w[e] = pack2(r[0], r[1]);
            }
            *(uint4 *)(stg + lane * 128 + (((c * 4 + j) ^ (lane & 7)) << 4)) = make_uint4(w[0], w[1], w[2], w[3]);
          }
        }
        __syncwarp();
        const int f = f0 + (lane & 7) * 8;
#pragma unroll
        for (int i = 0; i < 8; i++) {
          const int r = i * 4 + sub, gr = row_w + r;
          if (gr < p.rows && f < p.O[0])
            *(uint4 *)(p.act + (size_t)gr * p.O[0] + f) = *(const uint4 *)(stg + r * 128 + (((lane & 7) ^ (r & 7)) << 4));
        }
        __syncwarp();
      } else if (EPI == WIDE_ARGMAX) {
        // the thread scans its row's 128 features in order: the first of equal values wins (lowest index)
        const int f0 = nt * 256 + half * 128;
        float bv = 0.0f;
        int bi = -1;
#pragma unroll
        for (int c = 0; c < 4; c++) {
          uint32_t v[32];
          tmem_ld32(ta + half * 128 + c * 32, v);
#pragma unroll
          for (int e = 0; e < 32; e++) {
            const float x = __uint_as_float(v[e]);
            const bool better = f0 + c * 32 + e < p.O[0] && (bi < 0 || x > bv);
            bv = better ? x : bv;
            bi = better ? f0 + c * 32 + e : bi;
          }
          if (p.out_f32) {
            float4 a[8];
            transpose32(stg, lane, v, a);
            const int f = f0 + c * 32 + c4;
#pragma unroll
            for (int i = 0; i < 8; i++) {
              const int r = i * 4 + sub, gr = row_w + r;
              const float sc = __shfl_sync(0xffffffffu, inv, r);
              if (gr < p.rows && f < p.O[0]) {
                float *dst = p.out_f32 + (size_t)gr * p.ldo + f;
                const float o[4] = {a[i].x * sc, a[i].y * sc, a[i].z * sc, a[i].w * sc};
#pragma unroll
                for (int z = 0; z < 4; z++)
                  if (f + z < p.O[0]) dst[z] = o[z];
              }
            }
          }
        }
        if (row < p.rows && f0 < p.O[0]) {
          p.best_val[(size_t)(f0 >> 7) * p.best_ld + row] = bv;
          p.best_idx[(size_t)(f0 >> 7) * p.best_ld + row] = bi;
        }
      } else {   // WIDE_QKV: the half tile is one head of q, k or v
        int mi = 0, tm = 2 * nt + half;
        if (tm >= p.h1) { mi = 2; tm -= p.h1; }
        else if (tm >= p.h0) { mi = 1; tm -= p.h0; }
        const int kind = mi + p.kind0;
        const bool head_ok = tm * 128 < p.O[mi];
        bf16 *kv = kind == 1 ? p.kp : p.vp;
#pragma unroll
        for (int c = 0; c < 2; c++) {
          float4 a[8], b[8];
          {
            uint32_t v[32];
            tmem_ld32(ta + half * 128 + c * 32, v);
            transpose32(stg, lane, v, a);
            tmem_ld32(ta + half * 128 + 64 + c * 32, v);
            transpose32(stg, lane, v, b);
          }
#pragma unroll
          for (int i = 0; i < 8; i++) {
            const int r = i * 4 + sub, gr = row_w + r;
            const float sc = __shfl_sync(0xffffffffu, inv, r);
            const int sl = __shfl_sync(0xffffffffu, slot, r), sq = __shfl_sync(0xffffffffu, seq, r);
            if (gr >= p.rows || !head_ok) continue;
            float4 lo = make_float4(a[i].x * sc, a[i].y * sc, a[i].z * sc, a[i].w * sc);
            float4 hi = make_float4(b[i].x * sc, b[i].y * sc, b[i].z * sc, b[i].w * sc);
            if (kind < 2) {                       // rotate-half RoPE: feature j pairs with j + 64
              const float4 c0 = *(const float4 *)(p.cs + (size_t)gr * 64 + c * 32 + c4), c1 = *(const float4 *)(p.cs + (size_t)gr * 64 + c * 32 + c4 + 2);
              const float4 l = lo, h = hi;
              lo = make_float4(l.x * c0.x - h.x * c0.y, l.y * c0.z - h.y * c0.w, l.z * c1.x - h.z * c1.y, l.w * c1.z - h.w * c1.w);
              hi = make_float4(h.x * c0.x + l.x * c0.y, h.y * c0.z + l.y * c0.w, h.z * c1.x + l.z * c1.y, h.w * c1.z + l.w * c1.w);
            }
            bf16 *dst = nullptr;
            if (kind == 0) {
              dst = p.q + ((size_t)gr * p.H + tm) * 128;
              if (sq < 0) lo = hi = make_float4(0.f, 0.f, 0.f, 0.f);      // padding row
            } else if (sl >= 0) dst = kv + ((size_t)sl + (size_t)tm * p.page_size) * 128;
            if (dst) {
              *(uint2 *)(dst + c * 32 + c4) = pack4(lo);
              *(uint2 *)(dst + 64 + c * 32 + c4) = pack4(hi);
            }
          }
        }
      }
      // the accumulator may be overwritten: one arrival per warp on the even CTA's barrier
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncwarp();
      if (lane == 0) mbar_arrive_cluster(mapa_u32(smem_u32(&tempty[acc]), 0u));
    }
  }
  __syncthreads();
  if (*abort_flag && threadIdx.x == 0 && xr == 0) {
    // no bulk copy may still be landing when the pair exits (the even CTA's barriers count both CTAs' bytes)
    for (int i = *n_consumed; i < *n_issued; i++) mbar_wait(&full[i % W_STAGES], (uint32_t)((i / W_STAGES) & 1), p.spin);
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  cluster_sync_all();
  if (warp == W_EPI_WARPS + 1) asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512) : "memory");
  if (p.stamp && threadIdx.x == 0) atomicMin(p.stamp + 1, ~global_ns());
}

// ------------------------------------------------------------------------------------------------
// The same contraction with the K range split over S CTA pairs, for launches that have fewer tiles than the chip has pairs
// (16 tiles of a 4096-wide residual at 256 rows): the 2 S CTAs of a tile are one cluster (rank = position in the pair + 2 x
// slice).  Every CTA parks its accumulator (128 rows x 256 features, fp32, 128 KB) in its own shared memory, which the ring
// no longer needs, and takes an S-th of its ROWS from all slices through distributed shared memory, in slice order
// (deterministic); a warp handles one row of a half tile per step, a lane four consecutive features, so the epilogue's
// global accesses are whole rows of 256 or 512 bytes, the row's sum of squares is one warp sum, and RoPE's partner feature
// is sixteen lanes away.
constexpr int WS_DUMP = 2 * W_HALF * W_HALF * 4;               // 128 KB
constexpr int WS_SMEM = W_STAGES * W_STAGE + 2 * W_HALF * 4 + W_HALF * 4 + W_CTRL + 1024;
constexpr int WS_EPI_WARPS = 16, WS_THREADS = (WS_EPI_WARPS + 2) * 32;      // parking and reduction are latency chains: 16 warps, not 8
static_assert(WS_DUMP <= W_STAGES * W_STAGE, "the accumulator is parked in the ring");

__device__ __forceinline__ float4 ld_peer4(uint32_t local_addr, uint32_t rank) {      // several may be in flight (no memory clobber)
  float4 v;
  asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(mapa_u32(local_addr, rank)));
  return v;
}

// FEW: at most 96 rows per CTA
template <int EPI, int S, bool FEW>
__global__ void __launch_bounds__(WS_THREADS, 1) gemm_wide_split_kernel(const __grid_constant__ WideParams p) {
  extern __shared__ unsigned char smem_raw[];
  unsigned char *ring = (unsigned char *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  float *inv_s = (float *)(ring + W_STAGES * W_STAGE);         // [128] scale of this CTA's rows
  int *slot_s = (int *)(inv_s + W_HALF), *seq_s = slot_s + W_HALF;
  uint64_t *full = (uint64_t *)(seq_s + W_HALF);
  uint64_t *empty = full + W_STAGES;
  uint64_t *acc_bar = empty + W_STAGES;
  uint32_t *tmem_slot = (uint32_t *)(acc_bar + 1);
  volatile uint32_t *abort_flag = tmem_slot + 1;
  volatile int *n_issued = (volatile int *)(tmem_slot + 2), *n_consumed = (volatile int *)(tmem_slot + 3);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  uint32_t crank;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(crank));
  const int xr = (int)(crank & 1u), slice = (int)(crank >> 1);
  const uint32_t lead = crank & ~1u;
  const int t = blockIdx.x / (2 * S), mt = t % p.m_tiles, nt = t / p.m_tiles;
  const int kb0 = (int)(((long long)slice * p.KB) / S), kb1 = (int)(((long long)(slice + 1) * p.KB) / S), nkb = kb1 - kb0;
  const int row_c = mt * WIDE_ROWS + xr * p.half;              // first row of this CTA
  const int nrow = min(max(p.rows - row_c, 0), p.half);
  const uint32_t fill = 2u * (uint32_t)(p.half * TILE_K * 2 + W_A_BYTES);      // bytes of a stage, both CTAs

  if (threadIdx.x == 0) {
    for (int i = 0; i < W_STAGES; i++) { mbar_init(&full[i], 1); mbar_init(&empty[i], 1); }
    mbar_init(acc_bar, 1);
    *abort_flag = 0;
    *n_issued = 0; *n_consumed = 0;
    if ((int)crank != (int)(blockIdx.x % (2u * (unsigned)S))) { *abort_flag = 1; set_status(p.status, ST_TIMEOUT, 254, blockIdx.x, (int)crank); }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == WS_EPI_WARPS + 1) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(256) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  cluster_sync_all();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem_base = *tmem_slot;
  if (EPI != WIDE_QKV) pdl_trigger();            // WIDE_QKV: after the wait, see gemm_fused_kernel

  if (warp == WS_EPI_WARPS) {
    // ---- producer: own rows and own half of the features; all bytes are counted on the even CTA's barrier
    int mi = 0, tm = 2 * nt + xr;
    if (tm >= p.h1) { mi = 2; tm -= p.h1; }
    else if (tm >= p.h0) { mi = 1; tm -= p.h0; }
    const CUtensorMap *mw = &p.map_w[mi];
    const uint64_t pol = l2_policy_evict_first();
    const bool dead = __any_sync(0xffffffffu, *abort_flag != 0), hold = p.hold && blockIdx.x == 0;      // hold: test hook
    const int npre = dead ? 0 : nkb < W_STAGES ? nkb : W_STAGES;
    if (elect_one())
      for (int i = 0; i < npre; i++) {
        if (xr == 0) mbar_expect_tx(&full[i], fill);
        tma_load_2d_pair_hint(ring + i * W_STAGE + W_A_BYTES, mw, (kb0 + i) * TILE_K, tm * W_HALF, mapa_u32(smem_u32(&full[i]), lead), pol);
      }
    __syncwarp();
    pdl_wait();
    if (EPI == WIDE_QKV) pdl_trigger();
    if (elect_one()) {
      if (p.stamp) atomicMin(p.stamp, global_ns());
      for (int i = hold ? 1 : 0; i < npre; i++) tma_load_2d_pair(ring + i * W_STAGE, &p.map_x, (kb0 + i) * TILE_K, row_c, mapa_u32(smem_u32(&full[i]), lead));
    }
    __syncwarp();
    int i = npre, st = 0;
    uint32_t ph = 0;
    if (!dead)
      for (; i < nkb; i++) {
        if (!mbar_wait_warp(&empty[st], ph, p.spin)) { *abort_flag = 1; set_status(p.status, ST_TIMEOUT, 250, blockIdx.x, i); break; }
        if (elect_one()) {
          unsigned char *a = ring + st * W_STAGE;
          const uint32_t fb = mapa_u32(smem_u32(&full[st]), lead);
          if (xr == 0) mbar_expect_tx(&full[st], fill);
          const int kx = (kb0 + i) * TILE_K;
          tma_load_2d_pair_hint(a + W_A_BYTES, mw, kx, tm * W_HALF, fb, pol);
          tma_load_2d_pair(a, &p.map_x, kx, row_c, fb);
        }
        __syncwarp();
        if (++st == W_STAGES) { st = 0; ph ^= 1u; }
      }
    if (lane == 0) *n_issued = i;
  } else if (warp == WS_EPI_WARPS + 1) {
    pdl_wait();
    if (EPI == WIDE_QKV) pdl_trigger();
    if (xr == 0 && !__any_sync(0xffffffffu, *abort_flag != 0)) {
      constexpr uint32_t idesc = umma_idesc_m(256, 256);
      uint32_t partner_base;
      asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(partner_base) : "r"(mapa_u32(smem_u32(tmem_slot), crank | 1u)) : "memory");
      bool ok = partner_base == tmem_base;
      if (!ok) { *abort_flag = 1; set_status(p.status, ST_TIMEOUT, 253, blockIdx.x, (int)partner_base); }
      const uint64_t desc0 = umma_desc_sw128(smem_u32(ring));
      int i = 0, st = 0;
      uint32_t ph = 0, ready = 0;
      for (; ok && i < nkb; i++) {
        if (!ready && !mbar_wait_warp(&full[st], ph, p.spin)) { *abort_flag = 1; set_status(p.status, ST_TIMEOUT, 251, blockIdx.x, i); ok = false; break; }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint64_t da = desc0 + (uint64_t)((st * W_STAGE) >> 4), db = da + (W_A_BYTES >> 4);
        int nst = st + 1;
        uint32_t nph = ph;
        if (nst == W_STAGES) { nst = 0; nph ^= 1u; }
        if (elect_one()) {
#pragma unroll
          for (int j = 0; j < TILE_K / UMMA_K; j++) umma_bf16_pair(tmem_base, da + 2 * j, db + 2 * j, idesc, (i | j) ? 1u : 0u);
          umma_commit_pair(&empty[st], lead);
        }
        __syncwarp();
        ready = mbar_test_warp(&full[nst], nph) ? 1u : 0u;
        st = nst; ph = nph;
      }
      if (lane == 0) *n_consumed = i;
      __syncwarp();
      if (ok && elect_one()) umma_commit_pair(acc_bar, lead);
    }
  } else {
    pdl_wait();
    if (EPI == WIDE_QKV) pdl_trigger();
    if ((int)threadIdx.x < nrow) {                             // per-row values of this CTA's rows
      inv_s[threadIdx.x] = row_scale(p, row_c + threadIdx.x);
      if (EPI == WIDE_QKV) {
        int seq;
        slot_s[threadIdx.x] = row_slot(p, row_c + threadIdx.x, &seq);
        seq_s[threadIdx.x] = seq;
      }
    }
    // ---- accumulator -> shared memory: [half][row][128 floats], 16-byte chunks swizzled by the row
    const bool ok = __all_sync(0xffffffffu, mbar_wait_warp(acc_bar, 0, p.spin) && !*abort_flag);
    if (!ok) {
      if (lane == 0) set_status(p.status, ST_TIMEOUT, 252, blockIdx.x, slice);
      *abort_flag = 1;
    } else if ((warp & 3) * 32 < nrow) {
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const int r = (warp & 3) * 32 + lane, half = warp >> 3, c0 = (warp >> 2 & 1) * 2;      // four warps per quarter: 64 columns each
      unsigned char *dst = ring + (half * W_HALF + r) * 512;
#pragma unroll
      for (int c = 0; c < 2; c++) {
        uint32_t v[32];
        tmem_ld32(tmem_base + ((uint32_t)((warp & 3) * 32) << 16) + half * 128 + (c0 + c) * 32, v);
#pragma unroll
        for (int j = 0; j < 8; j++)
          *(uint4 *)(dst + ((((c0 + c) * 8 + j) ^ (r & 7)) << 4)) = make_uint4(v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3]);
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  cluster_sync_all();
  const bool good = !*abort_flag;                              // (a CTA that gave up stores nothing; its peers read stale sums, the status says so)

  if (warp < WS_EPI_WARPS) {
    const int per = (nrow + S - 1) / S, r0 = min(slice * per, nrow), r1 = min(r0 + per, nrow);
    const int half = warp & 1, sub = warp >> 1;                // eight warps per half tile, every eighth row each
    const int fo = nt * 256 + half * 128 + lane * 4;           // WIDE_RESID / WIDE_F32: first of the lane's features
    int mi = 0, tm = 2 * nt + half;
    if (EPI == WIDE_QKV) {
      if (tm >= p.h1) { mi = 2; tm -= p.h1; }
      else if (tm >= p.h0) { mi = 1; tm -= p.h0; }
    }
    const int kind = mi + p.kind0;
    const bool fok = good && (EPI == WIDE_QKV ? tm * 128 < p.O[mi] : fo < p.O[0]);
    float4 gn = make_float4(0.f, 0.f, 0.f, 0.f);
    if (EPI == WIDE_RESID && fok) gn = load_gain(p, fo);
    // rows in flight per warp: a share in one batch (two with two slices), of 128 rows or of at most 96
    constexpr int RB = FEW ? (S == 3 ? 4 : 3) : S == 3 ? 6 : 4;
    for (int rb = r0 + sub; rb < r1; rb += 8 * RB) {
      float4 xin[RB];
#pragma unroll
      for (int j = 0; j < RB; j++) {
        const int r = rb + 8 * j;
        xin[j] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (EPI == WIDE_RESID && p.resid_add && fok && r < r1) xin[j] = *(const float4 *)(p.xres + (size_t)(row_c + r) * p.O[0] + fo);
      }
      float4 v[S][RB];                                         // every remote load of the batch is in flight before the first sum
#pragma unroll
      for (int s = 0; s < S; s++)
#pragma unroll
        for (int j = 0; j < RB; j++) {
          const int r = min(rb + 8 * j, r1 - 1);
          v[s][j] = ld_peer4(smem_u32(ring + (half * W_HALF + r) * 512 + ((lane ^ (r & 7)) << 4)), (uint32_t)(xr + 2 * s));
        }
#pragma unroll
      for (int s = 1; s < S; s++)
#pragma unroll
        for (int j = 0; j < RB; j++) { v[0][j].x += v[s][j].x; v[0][j].y += v[s][j].y; v[0][j].z += v[s][j].z; v[0][j].w += v[s][j].w; }
#pragma unroll
      for (int j = 0; j < RB; j++) {
        const int r = rb + 8 * j, gr = row_c + r;
        if (r >= r1) continue;                                 // uniform over the warp
        float4 o = v[0][j];
        if (EPI == WIDE_RESID) {
          float sq = 0.0f;
          if (fok) {
            o.x += xin[j].x; o.y += xin[j].y; o.z += xin[j].z; o.w += xin[j].w;
            const size_t xi = (size_t)gr * p.O[0] + fo;
            *(float4 *)(p.xres + xi) = o;
            *(uint2 *)(p.hb + xi) = pack4(make_float4(o.x * gn.x, o.y * gn.y, o.z * gn.z, o.w * gn.w));
            if (p.tap_mask) {
              const uint2 tb = pack4(o);
#pragma unroll
              for (int s = 0; s < 3; s++)
                if ((p.tap_mask >> s) & 1) *(uint2 *)(p.taps + (size_t)gr * 3 * p.O[0] + (size_t)s * p.O[0] + fo) = tb;
            }
            sq = (o.x * o.x + o.y * o.y) + (o.z * o.z + o.w * o.w);
          }
          for (int off = 16; off > 0; off >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, off);
          if (lane == 0 && fok) p.ssq_out[(size_t)(fo >> 7) * p.ssq_ld + gr] = sq;
        } else if (EPI == WIDE_QKV) {
          const float sc = inv_s[r];
          const int sl = slot_s[r], sq = seq_s[r];
          o.x *= sc; o.y *= sc; o.z *= sc; o.w *= sc;
          float4 w;                                            // the partner features (i ^ 64): lane ^ 16
          w.x = __shfl_xor_sync(0xffffffffu, o.x, 16); w.y = __shfl_xor_sync(0xffffffffu, o.y, 16);
          w.z = __shfl_xor_sync(0xffffffffu, o.z, 16); w.w = __shfl_xor_sync(0xffffffffu, o.w, 16);
          if (!fok) continue;
          if (kind < 2) {
            const float4 c0 = *(const float4 *)(p.cs + (size_t)gr * 64 + (lane & 15) * 4), c1 = *(const float4 *)(p.cs + (size_t)gr * 64 + (lane & 15) * 4 + 2);
            if (lane < 16) o = make_float4(o.x * c0.x - w.x * c0.y, o.y * c0.z - w.y * c0.w, o.z * c1.x - w.z * c1.y, o.w * c1.z - w.w * c1.w);
            else o = make_float4(o.x * c0.x + w.x * c0.y, o.y * c0.z + w.y * c0.w, o.z * c1.x + w.z * c1.y, o.w * c1.z + w.w * c1.w);
          }
          if (kind == 0) {
            if (sq < 0) o = make_float4(0.f, 0.f, 0.f, 0.f);   // padding row
            *(uint2 *)(p.q + ((size_t)gr * p.H + tm) * 128 + lane * 4) = pack4(o);
          } else if (sl >= 0) {
            *(uint2 *)((kind == 1 ? p.kp : p.vp) + ((size_t)sl + (size_t)tm * p.page_size) * 128 + lane * 4) = pack4(o);
          }
        } else if (fok) {                                      // WIDE_F32
          const float sc = inv_s[r];
          *(float4 *)(p.out_f32 + (size_t)gr * p.ldo + fo) = make_float4(o.x * sc, o.y * sc, o.z * sc, o.w * sc);
        }
      }
    }
  }
  if (*abort_flag && threadIdx.x == 0 && xr == 0)              // no bulk copy may still be landing when the cluster exits
    for (int i = *n_consumed; i < *n_issued; i++) mbar_wait(&full[i % W_STAGES], (uint32_t)((i / W_STAGES) & 1), p.spin);
  cluster_sync_all();                                          // peers may still be reading this CTA's accumulator
  if (warp == WS_EPI_WARPS + 1) asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(256) : "memory");
  if (p.stamp && threadIdx.x == 0) atomicMin(p.stamp + 1, ~global_ns());
}

// ------------------------------------------------------------------------------------------------
// Gate/up GEMM with tiles of a chosen width: 2 x fpt accumulator columns (gate, up) per CTA pair instead of 2 x 128.  The
// 112 tiles of the 8B shapes are 1.5 waves of 74 pairs at one row tile, i.e. two; 69 tiles of 208 features are one, a k-block
// then costs 832 tensor cycles instead of 2 x 512 and the activations are read 69 times instead of 112.  Two accumulators of
// this width fill the tensor memory, so the epilogue is not hidden by a next tile: taken only where the waves say so
// (plan_swiglu).  A thread of the epilogue owns a row and writes 16 features = one 32-byte sector at a time.
constexpr int WG_MAX_FPT = 256;
__global__ void __launch_bounds__(WS_THREADS, 1) gemm_wide_swiglu_kernel(const __grid_constant__ WideParams p) {
  extern __shared__ unsigned char smem_raw[];
  unsigned char *ring = (unsigned char *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  const int fpt = p.fpt, b_bytes = fpt / 2 * 128, stage = W_A_BYTES + 2 * b_bytes, stages = p.stages;
  uint64_t *full = (uint64_t *)(ring + stages * stage);
  uint64_t *empty = full + 8, *tfull = empty + 8, *tempty = tfull + 1;
  uint32_t *tmem_slot = (uint32_t *)(tempty + 1);
  volatile uint32_t *abort_flag = tmem_slot + 1;
  volatile int *n_issued = (volatile int *)(tmem_slot + 2), *n_consumed = (volatile int *)(tmem_slot + 3);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  uint32_t crank;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(crank));
  const int xr = (int)(crank & 1u);
  const int pair = blockIdx.x >> 1, n_pairs = gridDim.x >> 1;
  const int ntiles = p.m_tiles * p.n_tiles, KB = p.KB;
  const uint32_t fill = 2u * (uint32_t)(p.half * TILE_K * 2 + 2 * b_bytes);    // bytes of a stage, both CTAs

  if (threadIdx.x == 0) {
    for (int i = 0; i < stages; i++) { mbar_init(&full[i], 1); mbar_init(&empty[i], 1); }
    mbar_init(tfull, 1);
    mbar_init(tempty, 2 * WS_EPI_WARPS);
    *abort_flag = 0;
    *n_issued = 0; *n_consumed = 0;
    if (crank != (blockIdx.x & 1u)) { *abort_flag = 1; set_status(p.status, ST_TIMEOUT, 264, blockIdx.x, (int)crank); }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == WS_EPI_WARPS + 1) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(512) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  cluster_sync_all();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem_base = *tmem_slot;
  pdl_trigger();

  if (warp == WS_EPI_WARPS) {
    // ---- producer: own rows, and the own half of the tile's gate and up features
    const uint64_t pol = l2_policy_evict_first();
    int issued = 0, st = 0;
    uint32_t ph = 1;
    bool ok = !__any_sync(0xffffffffu, *abort_flag != 0), first = true;
    for (int t = pair; t < ntiles && ok; t += n_pairs) {
      const int mt = t % p.m_tiles, nt = t / p.m_tiles;
      const int wrow = nt * fpt + xr * (fpt / 2), xrow = mt * WIDE_ROWS + xr * p.half;
      int kb = 0;
      if (first) {
        first = false;
        const int npre = KB < stages ? KB : stages;
        if (elect_one())
          for (int i = 0; i < npre; i++) {
            const uint32_t fb = mapa_u32(smem_u32(&full[i]), 0u);
            if (xr == 0) mbar_expect_tx(&full[i], fill);
            tma_load_2d_pair_hint(ring + i * stage + W_A_BYTES, &p.map_w[0], i * TILE_K, wrow, fb, pol);
            tma_load_2d_pair_hint(ring + i * stage + W_A_BYTES + b_bytes, &p.map_w[1], i * TILE_K, wrow, fb, pol);
          }
        __syncwarp();
        pdl_wait();
        if (elect_one())
          for (int i = p.hold && blockIdx.x == 0 ? 1 : 0; i < npre; i++) tma_load_2d_pair(ring + i * stage, &p.map_x, i * TILE_K, xrow, mapa_u32(smem_u32(&full[i]), 0u));
        __syncwarp();
        kb = npre; issued = npre;
        if (npre == stages) ph = 0; else st = npre;
      }
      for (; kb < KB; kb++) {
        if (!mbar_wait_warp(&empty[st], ph, p.spin)) { *abort_flag = 1; set_status(p.status, ST_TIMEOUT, 260, blockIdx.x, t); ok = false; break; }
        if (elect_one()) {
          unsigned char *a = ring + st * stage;
          const uint32_t fb = mapa_u32(smem_u32(&full[st]), 0u);
          if (xr == 0) mbar_expect_tx(&full[st], fill);
          const int kx = kb * TILE_K;
          tma_load_2d_pair_hint(a + W_A_BYTES, &p.map_w[0], kx, wrow, fb, pol);
          tma_load_2d_pair_hint(a + W_A_BYTES + b_bytes, &p.map_w[1], kx, wrow, fb, pol);
          tma_load_2d_pair(a, &p.map_x, kx, xrow, fb);
        }
        __syncwarp();
        issued++;
        if (++st == stages) { st = 0; ph ^= 1u; }
      }
    }
    if (first) pdl_wait();
    if (lane == 0) *n_issued = issued;
  } else if (warp == WS_EPI_WARPS + 1) {
    pdl_wait();
    if (xr == 0 && !__any_sync(0xffffffffu, *abort_flag != 0)) {
      const uint32_t idesc = umma_idesc_m(fpt, 256);
      const uint64_t desc0 = umma_desc_sw128(smem_u32(ring));
      int consumed = 0, st = 0, it = 0;
      uint32_t ph = 0, ready = 0;
      bool ok = true;
      for (int t = pair; t < ntiles && ok; t += n_pairs, it++) {
        if (it > 0) {
          const bool w = mbar_wait_cluster(tempty, (uint32_t)((it - 1) & 1), p.spin);
          if (!__all_sync(0xffffffffu, w)) { *abort_flag = 1; set_status(p.status, ST_TIMEOUT, 261, blockIdx.x, t); break; }
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        }
        for (int kb = 0; kb < KB; kb++) {
          if (!ready && !mbar_wait_warp(&full[st], ph, p.spin)) { *abort_flag = 1; set_status(p.status, ST_TIMEOUT, 262, blockIdx.x, t); ok = false; break; }
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          const uint64_t da = desc0 + (uint64_t)((st * stage) >> 4), dg = da + (W_A_BYTES >> 4), du = dg + (uint64_t)(b_bytes >> 4);
          int nst = st + 1;
          uint32_t nph = ph;
          if (nst == stages) { nst = 0; nph ^= 1u; }
          if (elect_one()) {
#pragma unroll
            for (int j = 0; j < TILE_K / UMMA_K; j++) {
              umma_bf16_pair(tmem_base, da + 2 * j, dg + 2 * j, idesc, (kb | j) ? 1u : 0u);
              umma_bf16_pair(tmem_base + 256, da + 2 * j, du + 2 * j, idesc, (kb | j) ? 1u : 0u);
            }
            umma_commit_pair(&empty[st], 0u);
            if (kb == KB - 1) umma_commit_pair(tfull, 0u);
          }
          __syncwarp();
          consumed++;
          ready = mbar_test_warp(&full[nst], nph) ? 1u : 0u;
          st = nst; ph = nph;
        }
      }
      if (lane == 0) *n_consumed = consumed;
    }
  } else {
    pdl_wait();
    if (p.stamp && threadIdx.x == 0) atomicMin(p.stamp, global_ns());
    const int quarter = warp & 3, part = warp >> 2;
    int it = 0;
    for (int t = pair; t < ntiles; t += n_pairs, it++) {
      const int mt = t % p.m_tiles, nt = t / p.m_tiles;
      const int lr = quarter * 32 + lane, row = mt * WIDE_ROWS + xr * p.half + lr;
      const bool mine = lr < p.half && row < p.rows;             // the other lanes' accumulators hold zeros or anything
      const float inv = mine ? row_scale(p, row) : 1.0f;
      const bool ok = __all_sync(0xffffffffu, mbar_wait_warp(tfull, (uint32_t)(it & 1), p.spin) && !*abort_flag);
      if (!ok) {
        if (lane == 0) { *abort_flag = 1; set_status(p.status, ST_TIMEOUT, 263, blockIdx.x, t); }
        break;
      }
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const uint32_t ta = tmem_base + ((uint32_t)(quarter * 32) << 16);
      const int runs = __any_sync(0xffffffffu, mine) ? fpt / 16 : 0;
#pragma unroll 1
      for (int c = part; c < runs; c += 4) {                 // the four warps of a quarter take alternate runs of 16 features
        uint32_t g[16], u[16], w[8];
        tmem_ld16(ta + c * 16, g);
        tmem_ld16(ta + 256 + c * 16, u);
#pragma unroll
        for (int e = 0; e < 8; e++) {
          float r[2];
#pragma unroll
          for (int z = 0; z < 2; z++) {
            // (A lane without a row divides 1: zeros and the like send the whole warp through the division's slow path, 8 us of a launch.)
            const float gv = mine ? __uint_as_float(g[2 * e + z]) * inv : 1.0f, uv = __uint_as_float(u[2 * e + z]) * inv;
            r[z] = (gv / (1.0f + expf(-gv))) * uv;
          }
          w[e] = pack2(r[0], r[1]);
        }
        const int f = nt * fpt + c * 16;
        bf16 *dst = p.act + (size_t)row * p.O[0] + f;
        if (mine && f < p.O[0]) *(uint4 *)dst = make_uint4(w[0], w[1], w[2], w[3]);
        if (mine && f + 8 < p.O[0]) *(uint4 *)(dst + 8) = make_uint4(w[4], w[5], w[6], w[7]);
      }
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncwarp();
      if (lane == 0) mbar_arrive_cluster(mapa_u32(smem_u32(tempty), 0u));
    }
  }
  __syncthreads();
  if (*abort_flag && threadIdx.x == 0 && xr == 0)
    for (int i = *n_consumed; i < *n_issued; i++) mbar_wait(&full[i % stages], (uint32_t)((i / stages) & 1), p.spin);
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  cluster_sync_all();
  if (warp == WS_EPI_WARPS + 1) asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512) : "memory");
  if (p.stamp && threadIdx.x == 0) atomicMin(p.stamp + 1, ~global_ns());
}

int n_tiles_of(WideEpi epi, const int *O, int nw) {
  if (epi == WIDE_SWIGLU) return (O[0] + 127) / 128;
  int h = 0;
  for (int j = 0; j < nw; j++) h += (O[j] + 127) / 128;
  return (h + 1) / 2;
}

void set_test(WideParams &p, WideTest kernel) {
  p.hold = tl_wide_test == kernel;
  p.spin = p.hold ? 2000u : SPIN_LIMIT;
}

template <int EPI>
int launch_wide(WideParams &p, bool pdl, cudaStream_t s) {
  set_test(p, WIDE_TEST_PERSISTENT);
  static SmemLimit limit;
  if (!limit.ensure(gemm_wide_kernel<EPI>, W_SMEM)) return -6;
  if (!launch_allowed()) return 0;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(2 * std::min(W_PAIRS, p.m_tiles * p.n_tiles), 1, 1);
  cfg.blockDim = dim3(W_THREADS, 1, 1);
  cfg.dynamicSmemBytes = W_SMEM;
  cfg.stream = s;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = 2; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
  at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = pdl ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, gemm_wide_kernel<EPI>, p) == cudaSuccess ? 0 : -6;
}

template <int EPI, int S, bool FEW>
int launch_split_inst(WideParams &p, bool pdl, cudaStream_t s) {
  set_test(p, WIDE_TEST_SPLIT);
  static SmemLimit limit;
  if (!limit.ensure(gemm_wide_split_kernel<EPI, S, FEW>, WS_SMEM)) return -6;
  if (!launch_allowed()) return 0;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(2 * S * p.m_tiles * p.n_tiles, 1, 1);
  cfg.blockDim = dim3(WS_THREADS, 1, 1);
  cfg.dynamicSmemBytes = WS_SMEM;
  cfg.stream = s;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = 2 * S; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
  at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = pdl ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, gemm_wide_split_kernel<EPI, S, FEW>, p) == cudaSuccess ? 0 : -6;
}
template <int EPI>
int launch_split(WideParams &p, int S, bool pdl, cudaStream_t s) {
  const bool few = p.half <= 96;
  switch (S) {
    case 2: return few ? launch_split_inst<EPI, 2, true>(p, pdl, s) : launch_split_inst<EPI, 2, false>(p, pdl, s);
    case 3: return few ? launch_split_inst<EPI, 3, true>(p, pdl, s) : launch_split_inst<EPI, 3, false>(p, pdl, s);
    default: return few ? launch_split_inst<EPI, 4, true>(p, pdl, s) : launch_split_inst<EPI, 4, false>(p, pdl, s);
  }
}

int launch_swiglu(WideParams &p, bool pdl, cudaStream_t s) {
  set_test(p, WIDE_TEST_GATE_UP);
  const int stage = W_A_BYTES + p.fpt * 128;
  p.stages = std::min(8, (W_SMEM - W_CTRL - 1024) / stage);
  static SmemLimit limit;
  if (!limit.ensure(gemm_wide_swiglu_kernel, W_SMEM)) return -6;
  if (!launch_allowed()) return 0;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(2 * std::min(W_PAIRS, p.m_tiles * p.n_tiles), 1, 1);
  cfg.blockDim = dim3(WS_THREADS, 1, 1);
  cfg.dynamicSmemBytes = p.stages * stage + W_CTRL + 1024;
  cfg.stream = s;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = 2; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
  at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = pdl ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, gemm_wide_swiglu_kernel, p) == cudaSuccess ? 0 : -6;
}

// Measured at 168 to 256 rows in the replayed step of the 8B shapes (weight-streaming kernel -> this one): QKV 26.7 -> 18.3 us, O 18.5 ->
// 17.8, down 33.4 -> 33 (168 rows); 31.7 -> 18.9, 22 -> 17.9, 38 -> 33 (240 rows); LM head 276 -> 180.
// Whole requests with 129, 144 and 160 rows a step (4 layers, 12 steps, their prefill included): 32.1 -> 26.4 ms, 31.8 -> 26.4, 36.4 -> 28.8.
// Clusters of 2 S CTAs (one CTA per SM) that are resident at once: a cluster lives inside one GPC, and this chip's GPCs hold
// 33, 22 and 15 clusters of 4, 6 and 8.  Constants: on a chip cut otherwise the plan may take one wave for two, no result changes.
constexpr int W_MAX_SPLIT = 4;
constexpr int W_FIT[W_MAX_SPLIT + 1] = {0, W_PAIRS, 33, 22, 15};
// What a launch costs beside its k-blocks, in k-blocks: the epilogue of the last tile (persistent kernel), or parking,
// cluster barrier, reduction and epilogue (split kernel)
constexpr int W_COST_TAIL = 12, W_COST_SPLIT = 18;
// K slices of a launch and its cost
long long plan_split(WideEpi epi, int tiles, int KB, int *S) {
  long long best = (long long)((tiles + W_PAIRS - 1) / W_PAIRS) * KB + W_COST_TAIL;
  *S = 1;
  if (epi != WIDE_RESID && epi != WIDE_QKV && epi != WIDE_F32) return best;
  for (int sk = 2; sk <= W_MAX_SPLIT; sk++) {
    if (KB / sk < 4) break;
    const long long c = (long long)((tiles + W_FIT[sk] - 1) / W_FIT[sk]) * ((KB + sk - 1) / sk + W_COST_SPLIT);
    if (c < best) { best = c; *S = sk; }
  }
  return best;
}

// Gate/up: features per tile of the launch (0: the persistent kernel with 128) and its cost.  A k-block of a tile fetches 128 rows of
// activations and f of weights per CTA, and that fill bounds it: its time goes with 96 + f, not with f, so narrow tiles cost more than their
// share.  Row-major kernel alone at 168 rows, own choice of the older estimate (f / 128) / of this one (us): F 14336 57.6 / 57.6, 13824 x
// 5120 83.2 / 62.1, 13824 x 4096 71.4 / 53.2, 11008 57.7 / 47.0, 16384 64.1 / 61.8, 28672 x 8192 227.8 / 198.4.  The persistent kernel hides its
// epilogues; with one row tile its waves are bound by the fill too (a third on top: F 14336 68, 18432 x 6144 96 against 95 with 256).  512 rows,
// older choice / this one: F 14336 80: 132.7 / persistent: 103.8, 11008 80: 106.8 / 82.4; 768 rows 11008 64: 155.9 / 108.3.
long long plan_swiglu(int F, int KB, int m_tiles, int *fpt) {
  const int t128 = (F + 127) / 128 * m_tiles;
  long long best = (long long)((t128 + W_PAIRS - 1) / W_PAIRS) * KB + W_COST_TAIL;
  if (m_tiles == 1) best = best * 4 / 3;
  *fpt = 0;
  for (int f = 64; f <= WG_MAX_FPT; f += 16) {       // N of an M = 256 MMA is a multiple of 16
    const int tiles = (F + f - 1) / f * m_tiles;
    const long long c = (long long)((tiles + W_PAIRS - 1) / W_PAIRS) * ((long long)KB * (96 + f) / 160 + W_COST_TAIL * f / 128);
    if (c < best) { best = c; *fpt = f; }
  }
  return best;
}

}  // namespace

long long wide_gemm_cost(WideEpi epi, const int *O, int nw, int I, int row_tiles) {
  int S;
  if (epi == WIDE_SWIGLU) return plan_swiglu(O[0], (I + TILE_K - 1) / TILE_K, row_tiles, &S);
  return plan_split(epi, n_tiles_of(epi, O, nw) * row_tiles, (I + TILE_K - 1) / TILE_K, &S);
}

// The epilogues store four or eight features at a time (only the argmax one's logits are stored one by one).
bool wide_gemm_supported(WideEpi epi, const WideGemmArgs &a) {
  if (a.rows < 1 || a.rows > a.x_rows || a.I < 8 || (a.I % 8) || ((uintptr_t)a.x & 15)) return false;
  if (a.nw < 1 || a.nw > 3 || (epi == WIDE_SWIGLU && (a.nw != 2 || a.O[0] != a.O[1])) || (epi == WIDE_QKV && a.nw < 2)) return false;
  for (int j = 0; j < a.nw; j++)
    if (!a.w[j] || ((uintptr_t)a.w[j] & 15) || a.O[j] < 1 || (epi != WIDE_ARGMAX && (a.O[j] % 8))) return false;
  if (a.form && a.form != 1) {
    if (epi == WIDE_SWIGLU ? a.form < 64 || a.form > WG_MAX_FPT || (a.form % 16) : a.form < 1 || a.form > W_MAX_SPLIT || a.form > (a.I + TILE_K - 1) / TILE_K)
      return false;
    if (epi == WIDE_BF16 || epi == WIDE_ARGMAX) return false;
  }
  return epi != WIDE_F32 || ((a.ldo % 4) == 0 && ((uintptr_t)a.out_f32 & 15) == 0);
}

int wide_gemm_launch(TmaMaps *g, WideEpi epi, const WideGemmArgs &a, cudaStream_t s) {
  if (!g || !wide_gemm_supported(epi, a)) return -1;
  WideParams p;
  memset(&p, 0, sizeof p);
  for (int j = 0; j < a.nw; j++) {
    const CUtensorMap *mw = tma_maps_get(g, a.w[j], a.O[j], a.I, W_HALF);
    if (!mw) return -6;
    p.map_w[j] = *mw;
    p.O[j] = a.O[j];
  }
  p.rows = a.rows; p.KB = (a.I + TILE_K - 1) / TILE_K;
  p.m_tiles = (a.rows + WIDE_ROWS - 1) / WIDE_ROWS; p.n_tiles = n_tiles_of(epi, a.O, a.nw);
  p.half = W_HALF;
  p.h0 = a.nw > 1 ? (a.O[0] + 127) / 128 : 1 << 30;
  p.h1 = a.nw > 2 ? p.h0 + (a.O[1] + 127) / 128 : 1 << 30;
  p.kind0 = a.nw == 3 ? 0 : 1;
  p.ssq_in = a.ssq_in; p.ssq_in_tiles = a.ssq_in_tiles; p.ssq_ld = a.ssq_ld; p.inv_k_in = 1.0f / (float)a.k_in; p.eps = a.eps;
  p.xres = a.xres; p.gain = a.gain; p.gain_vec = ((uintptr_t)a.gain & 7) == 0; p.hb = a.hb; p.ssq_out = a.ssq_out; p.taps = a.taps; p.tap_mask = a.taps ? a.tap_mask : 0; p.resid_add = a.resid_add;
  p.cs = a.cs; p.slot = a.slot; p.q = a.q; p.kp = (bf16 *)a.pool.k; p.vp = (bf16 *)a.pool.v; p.H = a.H; p.page_size = a.page_size;
  p.seq = a.seq; p.kvpos = a.kvpos; p.pm = a.pm; p.G = a.G;
  p.act = a.act; p.out_b = a.out_b; p.ldo = a.ldo; p.out_f32 = a.out_f32; p.status = a.status; p.stamp = a.stamp;
  p.best_val = a.best_val; p.best_idx = a.best_idx; p.best_ld = a.best_ld;
  int S = 1;
  if (epi == WIDE_SWIGLU) {
    plan_swiglu(a.O[0], p.KB, p.m_tiles, &p.fpt);
    if (a.form) p.fpt = a.form == 1 ? 0 : a.form;
    if (a.used) *a.used = p.fpt ? p.fpt : 1;
  } else {
    plan_split(epi, p.m_tiles * p.n_tiles, p.KB, &S);
    if (a.form) S = a.form;
    if (a.used) *a.used = S;
  }
  // One row tile of the split and the gate/up kernel is shared evenly: with 168 rows each CTA of a pair fetches, parks and adds up 88 or 80 of them
  // instead of 128 or 40 (in whole groups of eight, as the operand lies in shared memory).  Replayed step, 8B shapes (us, before -> now):
  // 132 rows QKV 19.6 -> 17.7, O 17.4 -> 15.3, down 32.9 -> 31.0; 168 rows 19.6 -> 18.1, 18.6 -> 16.3, 34.5 -> 31.9; 192 rows 20.5 -> 18.7,
  // 18.3 -> 16.1, 34.8 -> 32.4; 240 rows the same.
  if (p.m_tiles == 1 && (S > 1 || p.fpt)) p.half = std::min(W_HALF, ((a.rows + 1) / 2 + 7) & ~7);
  const CUtensorMap *mx = tma_maps_get(g, a.x, a.x_rows, a.I, p.half);
  if (!mx) return -6;
  p.map_x = *mx;
  if (epi == WIDE_SWIGLU) {
    if (p.fpt) {
      for (int j = 0; j < 2; j++) {
        const CUtensorMap *mw = tma_maps_get(g, a.w[j], a.O[j], a.I, p.fpt / 2);
        if (!mw) return -6;
        p.map_w[j] = *mw;
      }
      p.n_tiles = (a.O[0] + p.fpt - 1) / p.fpt;
      return launch_swiglu(p, a.pdl, s);
    }
  }
  if (S > 1) {
    switch (epi) {
      case WIDE_RESID: return launch_split<WIDE_RESID>(p, S, a.pdl, s);
      case WIDE_QKV: return launch_split<WIDE_QKV>(p, S, a.pdl, s);
      default: return launch_split<WIDE_F32>(p, S, a.pdl, s);
    }
  }
  switch (epi) {
    case WIDE_RESID: return launch_wide<WIDE_RESID>(p, a.pdl, s);
    case WIDE_QKV: return launch_wide<WIDE_QKV>(p, a.pdl, s);
    case WIDE_F32: return launch_wide<WIDE_F32>(p, a.pdl, s);
    case WIDE_ARGMAX: return launch_wide<WIDE_ARGMAX>(p, a.pdl, s);
    case WIDE_SWIGLU: return launch_wide<WIDE_SWIGLU>(p, a.pdl, s);
    default: return launch_wide<WIDE_BF16>(p, a.pdl, s);
  }
}

}  // namespace spec

extern "C" int spec_debug_wide_gemm(int32_t kernel) {
  if (kernel < spec::WIDE_TEST_OFF || kernel > spec::WIDE_TEST_GATE_UP) return -1;
  spec::tl_wide_test = kernel;
  return 0;
}
