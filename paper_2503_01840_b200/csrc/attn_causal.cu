// Causal paged attention on the fifth-generation tensor cores, head_dim 128 (sm_100a): the prefill's attention and the
// dense part of training-time-test attention.
//
// A query at position i attends keys 0..i of its sequence, read from the paged cache.  4 hd flops and one exponential per
// (query, key, head): the tensor pipe (512 cycles for each of the two 128 x 128 x 128 contractions) and the special-function
// unit (16 ex2 per cycle and SM: 1024 cycles per 128 x 128 scores) take the same time, so both have to run all the time:
//
//  * a CTA owns TWO query tiles of 128 positions that share every K and V tile: two heads of the same KV head (even
//    groups, same positions, so both tiles have the same key range), or two consecutive blocks of positions (odd groups);
//  * the scores of a query tile are taken 64 keys at a time into two alternating buffers of tensor memory.  The tile's
//    softmax warpgroup (thread = query row) reads a buffer, writes P (bf16) over it, and O += P V takes P straight from
//    tensor memory; behind each P V the scores two steps ahead go into the buffer it freed.  So the scores of the next step
//    are ready when a warpgroup comes for them, and no contraction lies on its path from one softmax to the next;
//  * each tile has an MMA-issuing warp of its own (one warp for both spent 1200 of 2230 cycles per 64-key step on waits,
//    commits and issue while the softmax waited for it);
//  * a row whose reference maximum moves (see CA_EARLY; rare after the first steps) waits for its last P V and rescales its O;
//    no other step waits for one;
//  * only the steps that cross the diagonal are masked;
//  * the diagonal entries of training-time test come through the K and V rings as further tiles (row = position), whose
//    dot products the softmax threads take from shared memory.
//
// Measured (one B200, T = 8192, 32 / 8 heads, 3 diagonal entries per row): 0.494 ms = 1110 TFLOP/s of causal flops (0.48 ms
// without diagonal entries) called in a row on the same inputs.  Earlier forms, in a row: one 128-key score buffer per tile and
// one issuer 0.67 ms; the same with an issuer per tile and P V in two halves 0.59; two 64-key buffers and one issuer 0.68; with
// an issuer each 0.536.  A 64-key step of both tiles takes 1470 cycles: shared memory delivers the operands of its MMAs and takes
// in the next tiles in 1250 (a 128 x 64 x 16 MMA reads 6 KB and takes 48 cycles, 32 with A in tensor memory), the exponentials
// take 1024, and the two softmax warps of a scheduler, which run in step, leave the special-function unit idle for the rest of
// theirs.  That rest was 580 cycles and is 450: one vote and one branch decide whether a reference moves, additions and multiply-adds
// go two at a time.
// Not better (same call, ms): the two warps' exponentials by turns 0.488 to 0.498; the next step's scores loaded, and their
// maximum taken, under this step's exponentials 0.59 to 0.62 (they come too late for it); an eighth to a third of the
// exponentials by a polynomial on the multiply-add pipe 0.493 to 0.514; half of Q in tensor memory with one score buffer 0.575; the next
// step's scores asked for before this step's P is known to be written 0.494 too, and 3 to 5 % slower where softmax alone is the bound (500
// positions of 16 heads 18.7 against 17.9 us, 2500 of 16 / 4 heads 44.3 against 43.1): two loads into the same registers want copies.
//
// Every wait is bounded.  On a time-out the CTA winds down; a prefill's status words record it, and training-time test, which
// has none, gets NaN in the rows (and normalisers) it could not finish.
#include <math.h>
#include <string.h>

#include "../../include/spec_b200.h"
#include "attn_causal.cuh"
#include "tcgen05_ptx.cuh"
#include "attn_fast.cuh"
#include "attn_maps.cuh"

namespace spec {

thread_local int tl_causal_test = CAUSAL_TEST_OFF;

namespace {

using tc::elect_one;
using tc::mbar_expect_tx;
using tc::mbar_init;
using tc::mbar_wait;
using tc::mbar_wait_warp;
using tc::smem_u32;

constexpr int CA_HD = 128, CA_T = CAUSAL_TILE, CA_KS = 64;      // keys per softmax step
constexpr int CA_TILE = CA_T * CA_HD * 2;          // 32 KB: a Q, K or V tile
constexpr int CA_HALF = CA_T * 128;                // 16 KB: 64 of the 128 dimensions of a tile
constexpr int CA_STAGES = 2;                       // K tiles and V tiles in flight (each)
constexpr int CA_CTRL = 256;
constexpr int CA_SMEM = (2 + 2 * CA_STAGES) * CA_TILE + CA_CTRL + 1024;
// Two softmax warpgroups and one with the TMA warp and the MMA warps.  384 threads start with 168 registers each (64512 in
// all); the softmax holds a row's 128 scores, so its 256 threads take 208 and the other 128 go down to 88 (64512 again).
constexpr int CA_THREADS = 384, CA_REGS_SOFTMAX = 208, CA_REGS_ISSUE = 88;
static_assert(256 * CA_REGS_SOFTMAX + 128 * CA_REGS_ISSUE <= CA_THREADS * 168, "register shares must fit what the block is launched with");
constexpr int CA_MAX_DIAG = 8;
// How closely a row's reference maximum follows its maximum.  P is bf16, so the error of an output comes from the row's
// largest probabilities; it is least when those lie at or just below 1, i.e. when the reference is the maximum.  The prefill
// moves the reference by jumps beyond 2^CA_FAR only (each costs a rescaled O; the rounding of a layer's activations hides the
// difference).  Training-time test follows jumps beyond 2^CA_NEAR while the maximum settles, in a row's first CA_EARLY steps.
// Sequences of at most CA_BRIEF positions have few and therefore large probabilities: they follow closely throughout and
// divide by the sum of the rounded ones, which O sums, so that the rounding of a large one partly cancels (a kernel of its own:
// the second sum costs 5 to 8 % wherever it stands).
// Relative error against fp64 in 1e-3 (the bf16 output alone is 1.66) and time.  T = 8192, 32 / 8 heads, 3 diagonal entries:
// jumps of 2^8 only 2.175, 551 us; this 2.141, 539; 2^1 throughout 2.123, 588; rounded sum and 2^0.5 in the first 8 steps 2.125,
// 582.  T = 512, 32 / 8 heads, 3 entries: 2^8 only 2.073, 26 us; 2^0.5 in the first 4 steps 2.034, 26; this 2.011, 29.  T = 256,
// 16 / 16 heads: 1.958, 1.927 and 1.903, 19 us each.
constexpr int CA_EARLY = 4, CA_BRIEF = 512;
constexpr float CA_NEAR = 0.5f, CA_FAR = 8.0f;

struct CausalParams {
  PageMap pm;
  bf16 *out;
  int H, G, T, J;
  const CausalBlock *blocks;
  const bf16 *kd, *vd;
  float *lse;
  int narrow;                      // out / kd / vd are only 8-byte aligned: the diagonal entries are read row by row instead
  int32_t *status;
  int test;                        // test hook, see CausalTest
  uint32_t spin;                   // polls before a wait gives up
};

// eight elements of a row that starts on an 8-byte boundary
__device__ __forceinline__ uint4 ld_row8(const bf16 *p) {
  const uint2 a = *(const uint2 *)p, b = *(const uint2 *)(p + 4);
  return make_uint4(a.x, a.y, b.x, b.y);
}
__device__ __forceinline__ void mbar_arrive(uint64_t *bar) { asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory"); }
__device__ __forceinline__ float ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {      // two multiply-adds in one instruction, each rounded like fmaf
  float2 r;
  asm("{\n\t.reg .b64 a, b, c, d;\n\tmov.b64 a, {%2, %3};\n\tmov.b64 b, {%4, %5};\n\tmov.b64 c, {%6, %7};\n\tfma.rn.f32x2 d, a, b, c;\n\tmov.b64 {%0, %1}, d;\n\t}"
      : "=f"(r.x), "=f"(r.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
  return r;
}
__device__ __forceinline__ float2 add2(float2 a, float2 b) {
  float2 r;
  asm("{\n\t.reg .b64 a, b, d;\n\tmov.b64 a, {%2, %3};\n\tmov.b64 b, {%4, %5};\n\tadd.rn.f32x2 d, a, b;\n\tmov.b64 {%0, %1}, d;\n\t}"
      : "=f"(r.x), "=f"(r.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return r;
}
__device__ __forceinline__ uint32_t pack2(float lo, float hi) {
  __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *(uint32_t *)&v;
}
__device__ __forceinline__ void load_3d(void *dst, const CUtensorMap *map, int c0, int c1, int c2, uint64_t *bar) {
  asm volatile("cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], [%2];" ::"r"(smem_u32(dst)),
               "l"(map), "r"(smem_u32(bar)), "r"(c0), "r"(c1), "r"(c2)
               : "memory");
}
__device__ __forceinline__ void load_4d(void *dst, const CUtensorMap *map, int c0, int c1, int c2, int c3, uint64_t *bar) {
  asm volatile("cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6}], [%2];" ::"r"(smem_u32(dst)),
               "l"(map), "r"(smem_u32(bar)), "r"(c0), "r"(c1), "r"(c2), "r"(c3)
               : "memory");
}
// D += A B with A (128 x 16 bf16, two elements per column) in tensor memory
__device__ __forceinline__ void umma_ts(uint32_t tmem_d, uint32_t tmem_a, uint64_t db, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}" ::"r"(tmem_d),
      "r"(tmem_a), "l"(db), "r"(idesc), "r"(accumulate)
      : "memory");
}
__device__ __forceinline__ uint64_t desc_mn(uint32_t saddr, uint32_t lbo) {      // MN-major operand, 128-byte swizzle
  return (uint64_t)((saddr & 0x3FFFF) >> 4) | ((uint64_t)(lbo >> 4) << 16) | ((uint64_t)(1024 >> 4) << 32) | ((uint64_t)1 << 46) | ((uint64_t)2 << 61);
}
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float *f) {     // no wait
  uint32_t *v = (uint32_t *)f;
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, %17, %18, "
      "%19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]), "=r"(v[9]),
        "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]), "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]),
        "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]), "=r"(v[24]), "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]),
        "=r"(v[30]), "=r"(v[31])
      : "r"(taddr));
}
// values that a tmem_ld32 put out, from here on: behind the wait for them, nothing that uses them moves to before it
__device__ __forceinline__ void pin32(float *f) {
  asm volatile("" : "+f"(f[0]), "+f"(f[1]), "+f"(f[2]), "+f"(f[3]), "+f"(f[4]), "+f"(f[5]), "+f"(f[6]), "+f"(f[7]), "+f"(f[8]), "+f"(f[9]), "+f"(f[10]), "+f"(f[11]),
                    "+f"(f[12]), "+f"(f[13]), "+f"(f[14]), "+f"(f[15]));
  asm volatile("" : "+f"(f[16]), "+f"(f[17]), "+f"(f[18]), "+f"(f[19]), "+f"(f[20]), "+f"(f[21]), "+f"(f[22]), "+f"(f[23]), "+f"(f[24]), "+f"(f[25]), "+f"(f[26]),
                    "+f"(f[27]), "+f"(f[28]), "+f"(f[29]), "+f"(f[30]), "+f"(f[31]));
}
__device__ __forceinline__ void tmem_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tmem_st32(uint32_t taddr, const uint32_t *v) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, %17, %18, "
      "%19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, %32};" ::"r"(taddr),
      "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]), "r"(v[8]), "r"(v[9]), "r"(v[10]),
      "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15]), "r"(v[16]), "r"(v[17]), "r"(v[18]), "r"(v[19]), "r"(v[20]), "r"(v[21]),
      "r"(v[22]), "r"(v[23]), "r"(v[24]), "r"(v[25]), "r"(v[26]), "r"(v[27]), "r"(v[28]), "r"(v[29]), "r"(v[30]), "r"(v[31])
      : "memory");
}
__device__ __forceinline__ void tmem_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ float2 bf2(uint32_t u) { return __bfloat1622float2(*(const __nv_bfloat162 *)&u); }

// DIAG: the diagonal keys of training-time test are folded in (J may be 0) and the log-normaliser is written.  BRIEF: see CA_BRIEF
template <bool DIAG, bool BRIEF>
__global__ void __launch_bounds__(CA_THREADS, 1) attn_causal_kernel(const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_k,
                                                           const __grid_constant__ CUtensorMap map_v, const __grid_constant__ CUtensorMap map_kd,
                                                           const __grid_constant__ CUtensorMap map_vd, const __grid_constant__ CausalParams p) {
  pdl_trigger();
  pdl_wait();
  extern __shared__ unsigned char smem_raw[];
  unsigned char *sQ = (unsigned char *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);   // two tiles [hd half][128 rows][128 B]
  unsigned char *sK = sQ + 2 * CA_TILE, *sV = sK + CA_STAGES * CA_TILE;
  uint64_t *kfull = (uint64_t *)(sV + CA_STAGES * CA_TILE), *kempty = kfull + CA_STAGES, *vfull = kempty + CA_STAGES, *vempty = vfull + CA_STAGES;
  uint64_t *q_bar = vempty + CA_STAGES, *s_bar = q_bar + 1, *p_bar = s_bar + 4, *o_bar = p_bar + 4, *d_bar = o_bar + 2;     // s, p: [tile][buffer]; o, d: [tile]
  uint32_t *tmem_slot = (uint32_t *)(d_bar + 2);
  volatile uint32_t *abort_flag = tmem_slot + 1;
  volatile int *n_filled = (volatile int *)(tmem_slot + 2);     // [0] K tiles, [1] V tiles requested

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int grp = p.H / p.G;
  const bool two_heads = (grp & 1) == 0;
  int row0, nrows, seq, pos0;
  if (p.blocks) {
    const CausalBlock b = p.blocks[blockIdx.y];
    row0 = b.row0; nrows = b.nrows; seq = b.seq; pos0 = b.pos0;
  } else {                                          // one sequence of T rows; the longest key ranges first
    const int br = two_heads ? CA_T : 2 * CA_T;
    row0 = ((int)gridDim.y - 1 - (int)blockIdx.y) * br;
    nrows = min(br, p.T - row0); seq = 0; pos0 = row0;
  }
  const int head0 = two_heads ? 2 * blockIdx.x : blockIdx.x;
  const int g = head0 / grp;
  // tile t of the CTA: rows, first position, 64-key steps
  const int rows_0 = min(nrows, CA_T), rows_1 = two_heads ? rows_0 : max(0, nrows - CA_T);
  const int off_1 = two_heads ? 0 : CA_T;
  const int n0 = (pos0 + rows_0 + CA_KS - 1) / CA_KS, n1 = rows_1 > 0 ? (pos0 + off_1 + rows_1 + CA_KS - 1) / CA_KS : 0;
  const int n = max(n0, n1), nkt = (n + 1) / 2;     // steps, 128-key tiles
  const bool diag_ring = DIAG && p.J > 0 && !p.narrow;
  const int nb = two_heads ? 1 : 2;                 // ring tiles per diagonal step: both query tiles' rows, or one each

  if (threadIdx.x == 0) {
    for (int i = 0; i < CA_STAGES; i++) { mbar_init(&kfull[i], 1); mbar_init(&kempty[i], 2); mbar_init(&vfull[i], 1); mbar_init(&vempty[i], 2); }
    mbar_init(q_bar, 1);
    for (int i = 0; i < 4; i++) { mbar_init(&s_bar[i], 1); mbar_init(&p_bar[i], 4); }
    for (int i = 0; i < 2; i++) { mbar_init(&o_bar[i], 1); mbar_init(&d_bar[i], 1); }
    *abort_flag = 0;
    n_filled[0] = n_filled[1] = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 9) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(512) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem_base = *tmem_slot;            // S / P of tile t, buffer u at column 128 t + 64 u, O at 256 + 128 t

  if (warp >= 8) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(CA_REGS_ISSUE));
    if (warp == 8) {
      // ================================================================ TMA warp
      const int ps = p.pm.page_size, ppt = CA_T / ps;          // pages per key tile: 8, 4 or 2
      const int32_t *tbl = p.pm.table + (size_t)seq * p.pm.pages_per_seq;
      const int fallback = tbl[0];                             // keys past the last page are masked; they still need a valid source
      const bool hold = p.test == CAUSAL_TEST_WITHHOLD && blockIdx.x == 0 && blockIdx.y == 0;
      if (elect_one()) {
        mbar_expect_tx(q_bar, 2 * CA_TILE);
        if (!hold)
#pragma unroll
        for (int t = 0; t < 2; t++)
#pragma unroll
          for (int h = 0; h < 2; h++)
            load_3d(sQ + t * CA_TILE + h * CA_HALF, &map_q, 64 * h, two_heads ? head0 + t : head0, row0 + (two_heads ? 0 : t * CA_T), q_bar);
      }
      __syncwarp();
      auto page_of = [&](int j) {                              // lane's page of key tile j
        const int ip = j * ppt + lane;
        int page = (lane < ppt && ip < p.pm.pages_per_seq) ? tbl[ip] : -1;
        if (page < 0 || page >= p.pm.num_pages) page = fallback;
        return (page * p.G + g) * ps;
      };
      // one ring tile: wait for its stage, then request it (whole warp; the elected lane issues)
      auto fill = [&](int kv, int j, auto issue) {
        const int st = j % CA_STAGES;
        uint64_t *fb = kv ? &vfull[st] : &kfull[st], *eb = kv ? &vempty[st] : &kempty[st];
        if (!mbar_wait_warp(eb, (uint32_t)((j / CA_STAGES) & 1) ^ 1u, p.spin)) {
          *abort_flag = 1;
          if (p.status) set_status(p.status, ST_TIMEOUT, 430 + kv, blockIdx.y, j);
        } else if (elect_one()) {
          mbar_expect_tx(fb, CA_TILE);
          issue((kv ? sV : sK) + st * CA_TILE, fb);
          n_filled[kv] = j + 1;
        }
        __syncwarp();
        return !__any_sync(0xffffffffu, *abort_flag != 0);      // one answer for the warp, whoever gives up meanwhile
      };
      int cur = page_of(0);
      bool ok = true;
      for (int j = 0; j < nkt && ok; j++) {
        const int nxt = j + 1 < nkt ? page_of(j + 1) : 0;
        int row[8];
#pragma unroll
        for (int i = 0; i < 8; i++) row[i] = __shfl_sync(0xffffffffu, cur, i);
#pragma unroll
        for (int kv = 0; kv < 2; kv++)
          ok = ok && fill(kv, j, [&](unsigned char *d, uint64_t *fb) {
#pragma unroll
                 for (int i = 0; i < 8; i++) {
                   if (i >= ppt) break;
#pragma unroll
                   for (int h = 0; h < 2; h++) load_3d(d + h * CA_HALF + i * ps * 128, kv ? &map_v : &map_k, 0, row[i], h, fb);
                 }
               });
        cur = nxt;
      }
      if (DIAG && diag_ring) {
        // The diagonal steps' entries: all keys (their dot products come first), then all values, by turns through the two
        // rings, so that all four stages are in flight in either phase (see diag_entry)
        const int total = p.J * nb;
        for (int e = 0; e < 2 * total && ok; e++) {
          const int x = e < total ? e : e - total;
          ok = fill(e & 1, nkt + (e >> 1), [&](unsigned char *d, uint64_t *fb) {
#pragma unroll
            for (int h = 0; h < 2; h++) load_4d(d + h * CA_HALF, e < total ? &map_kd : &map_vd, 64 * h, g, row0 + (x % nb) * CA_T, x / nb, fb);
          });
        }
      }
    } else if (warp <= 10) {
      // ================================================================ MMA warps: one per query tile
      // Both release every K and V tile, also those their own query tile has no keys in: they wait for it to land like the
      // other one.
      const int t = warp - 9, nt = t ? n1 : n0;
      constexpr uint32_t idesc_s = tc::umma_idesc(CA_KS);                   // both operands K-major, N = 64 keys
      constexpr uint32_t idesc_o = tc::umma_idesc(CA_HD) | (1u << 16);      // B (the V tile) MN-major, N = 128 dimensions
      const uint64_t dq = tc::umma_desc_sw128(smem_u32(sQ + t * CA_TILE)), dk = tc::umma_desc_sw128(smem_u32(sK));
      const uint64_t dv = desc_mn(smem_u32(sV), CA_HALF);
      const uint32_t ts = tmem_base + t * 128, to = tmem_base + 256 + t * 128;
      // step i: half i % 2 of key tile i / 2, buffer i % 2
      auto part = [&](int i) { return (uint64_t)((((i >> 1) % CA_STAGES) * CA_TILE + (i & 1) * (CA_KS * 128)) >> 4); };
      auto issue_s = [&](int i) {
        const uint64_t kd = dk + part(i);
#pragma unroll
        for (int kk = 0; kk < 8; kk++) {
          const uint64_t o = (uint64_t)(((kk >> 2) * CA_HALF + (kk & 3) * 32) >> 4);
          tc::umma_bf16(ts + (i & 1) * CA_KS, dq + o, kd + o, idesc_s, kk ? 1u : 0u);
        }
        tc::umma_commit(&s_bar[t * 2 + (i & 1)]);
      };
      bool ok = mbar_wait_warp(q_bar, 0, p.spin) && mbar_wait_warp(&kfull[0], 0, p.spin);
      if (!ok) { *abort_flag = 1; if (p.status) set_status(p.status, ST_TIMEOUT, 432, blockIdx.y, t); }
      if (ok) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        if (elect_one()) {
          for (int i = 0; i < 2; i++)
            if (i < nt) issue_s(i);
          tc::umma_commit(&kempty[0]);
        }
        __syncwarp();
        for (int i = 0; i < n; i++) {
          const int st = (i >> 1) % CA_STAGES, st2 = ((i + 2) >> 1) % CA_STAGES;
          if (!(i & 1)) {                              // a new V tile, and the K tile of the scores that follow it
            ok = mbar_wait_warp(&vfull[st], (uint32_t)(((i >> 1) / CA_STAGES) & 1), p.spin);
            if (ok && i + 2 < n) ok = mbar_wait_warp(&kfull[st2], (uint32_t)((((i + 2) >> 1) / CA_STAGES) & 1), p.spin);
          }
          if (ok && i < nt) ok = mbar_wait_warp(&p_bar[t * 2 + (i & 1)], (uint32_t)((i >> 1) & 1), p.spin);
          if (!ok) { *abort_flag = 1; if (p.status) set_status(p.status, ST_TIMEOUT, 433, blockIdx.y, i); break; }
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          if (elect_one()) {
            if (i < nt) {
              const uint64_t vd = dv + part(i);
#pragma unroll
              for (int kk = 0; kk < 4; kk++)           // 16 keys: 8 columns of P, 16 rows of V
                umma_ts(to, ts + (i & 1) * CA_KS + kk * 8, vd + (uint64_t)((kk * 16 * 128) >> 4), idesc_o, (i | kk) ? 1u : 0u);
              tc::umma_commit(&o_bar[t]);
              if (i == nt - 1) tc::umma_commit(&d_bar[t]);
            }
            if (i + 2 < nt) issue_s(i + 2);
            // the tiles whose last use has been issued
            if ((i & 1) || i == n - 1) tc::umma_commit(&vempty[st]);
            if (i + 2 < n && ((i & 1) || i + 2 == n - 1)) tc::umma_commit(&kempty[st2]);
          }
          __syncwarp();
        }
      }
    }
  } else {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(CA_REGS_SOFTMAX));
    // ================================================================ softmax: thread = query row = tensor-memory lane
    const int t = warp >> 2, lr = threadIdx.x & 127;
    const int nt = t ? n1 : n0, nr = t ? rows_1 : rows_0;
    const int head = two_heads ? head0 + t : head0;
    const int trow = row0 + (t ? off_1 : 0), pos = pos0 + (t ? off_1 : 0) + lr;      // first row of the tile, this thread's position
    const uint32_t lanes = (uint32_t)((warp & 3) * 32) << 16;
    const uint32_t my_s = tmem_base + lanes + (uint32_t)(t * 128), my_o = tmem_base + lanes + 256u + (uint32_t)(t * 128);
    const float sc = rsqrtf((float)CA_HD) * 1.4426950408889634f;                     // softmax scale folded into exp2
    float mx = -INFINITY, l = 0.0f, lrnd = 0.0f;                  // sums of the probabilities and (BRIEF) of the rounded ones
    bool alive = true;
    auto gave_up = [&](int site, int i) {
      if (lane == 0) { *abort_flag = 1; if (p.status) set_status(p.status, ST_TIMEOUT, site, blockIdx.y, i); }
      alive = false;
    };
    float nb_ = 0.0f;                                            // the reference maximum in the exponent (0 while there is none)
    for (int i = 0; i < nt; i++) {
      if (!mbar_wait_warp(&s_bar[t * 2 + (i & 1)], (uint32_t)((i >> 1) & 1), p.spin)) { gave_up(435, i); break; }
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      float s[CA_KS];
      tmem_ld32(my_s + (uint32_t)((i & 1) * CA_KS), s);
      tmem_ld32(my_s + (uint32_t)((i & 1) * CA_KS + 32), s + 32);
      tmem_ld_wait();
      pin32(s);
      pin32(s + 32);
      const int k0 = i * CA_KS;
      if (k0 + CA_KS - 1 > pos - lane) {                         // uniform over the warp: its first row does not see the whole step
        const int lim = pos - k0;                                // keys 0..lim of the step
#pragma unroll
        for (int e = 0; e < CA_KS; e++) s[e] = e <= lim ? s[e] : -INFINITY;
      }
      float m4[4] = {s[0], s[1], s[2], s[3]};
#pragma unroll
      for (int e = 4; e < CA_KS; e += 4) {
#pragma unroll
        for (int z = 0; z < 4; z++) m4[z] = fmaxf(m4[z], s[e + z]);
      }
      const float tm = fmaxf(fmaxf(m4[0], m4[1]), fmaxf(m4[2], m4[3]));
      // the reference maximum moves when the step's exceeds it by more than this in the exponent (training-time test: those of
      // the warp's other rows then move along)
      const float jump = DIAG && (BRIEF || i < CA_EARLY) ? CA_NEAR : CA_FAR;
      const bool far = (tm - mx) * sc > jump;
      if (__any_sync(0xffffffffu, far)) {                        // rare after a row's first steps: all that a moving reference costs is in here
        float f = 1.0f;
        if ((DIAG || far) && tm > mx) {
          f = (mx == -INFINITY) ? 1.0f : ex2((mx - tm) * sc);
          mx = tm;
          nb_ = mx * sc;
        }
        l *= f;
        lrnd *= f;
        if (i > 0 && __any_sync(0xffffffffu, f != 1.0f)) {       // the P V of the last step must be complete before O is rescaled
          if (!mbar_wait_warp(&o_bar[t], (uint32_t)((i - 1) & 1), p.spin)) { gave_up(438, i); break; }
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll 1
          for (int c = 0; c < 4; c++) {
            float o[32];
            tmem_ld32(my_o + c * 32, o);
            tmem_ld_wait();
#pragma unroll
            for (int e = 0; e < 32; e++) o[e] *= f;
            tmem_st32(my_o + c * 32, (uint32_t *)o);
          }
        }
      }
      float2 rs[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
      const float2 sc2 = make_float2(sc, sc), nb2 = make_float2(-nb_, -nb_);
      uint32_t pk[32];
#pragma unroll
      for (int e = 0; e < 32; e++) {
        const float2 x = fma2(make_float2(s[2 * e], s[2 * e + 1]), sc2, nb2), pr = make_float2(ex2(x.x), ex2(x.y));
        rs[e & 1] = add2(rs[e & 1], pr);
        pk[e] = pack2(pr.x, pr.y);
      }
      tmem_st32(my_s + (uint32_t)((i & 1) * CA_KS), pk);
      l += (rs[0].x + rs[0].y) + (rs[1].x + rs[1].y);
      if (BRIEF) {
#pragma unroll
        for (int z = 0; z < 2; z++) rs[z] = make_float2(0.f, 0.f);
#pragma unroll
        for (int e = 0; e < 32; e++) rs[e & 1] = add2(rs[e & 1], bf2(pk[e]));
        lrnd += (rs[0].x + rs[0].y) + (rs[1].x + rs[1].y);
      }
      tmem_st_wait();
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncwarp();
      if (lane == 0) mbar_arrive(&p_bar[t * 2 + (i & 1)]);
    }
    if (alive && nt > 0) {
      // All P V of the tile.  A barrier of its own: the scores of the last step only tell that the P V two steps earlier is
      // complete, so o_bar can be up to two phases behind, and a warp that comes late finds it two phases further, where
      // its parity says the same.
      if (p.test == CAUSAL_TEST_LATE) __nanosleep(50000);
      const bool ok = __all_sync(0xffffffffu, mbar_wait_warp(&d_bar[t], 0, p.spin) && !*abort_flag);
      if (!ok) { if (lane == 0) { *abort_flag = 1; if (p.status) set_status(p.status, ST_TIMEOUT, 436, blockIdx.y, nt); } alive = false; }
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    }
    unsigned char *qt = sQ + t * CA_TILE;                        // this row's 16-byte chunk c: half c / 8, row lr, chunk (c % 8) ^ (lr % 8)
    auto chunk = [](unsigned char *tile, int r, int c) { return (uint4 *)(tile + (c >> 3) * CA_HALF + r * 128 + (((c & 7) ^ (r & 7)) << 4)); };
    const bool rv = lr < nr;
    float fo = 1.0f, wd[CA_MAX_DIAG];
    size_t doff = 0;
    const size_t dstep = (size_t)p.T * p.G * CA_HD;
    // Diagonal entry e of this CTA sits in ring e % 2, place nkt + e / 2.  The two query tiles share an entry where they are
    // two heads, and take alternate ones (one ring each) where they are two blocks of positions.  Both tiles have to be
    // through with their keys first: a wait for place j of a ring means something only when the use of its stage before that
    // (place j - 2, maybe keys of the other tile alone) has landed.
    // With keys in one ring, values in the other and both tiles in step after every entry, an entry took the latency of a load
    // (1.5 us).  With few heads that is on the critical path: 4 heads, 7 steps, T = 2048 63 us then, 57 now; T = 512 39, 33.
    if (DIAG && diag_ring) asm volatile("bar.sync 3, 256;" ::: "memory");
    auto diag_wait = [&](int e) -> unsigned char * {
      const int st = (nkt + (e >> 1)) % CA_STAGES;
      const bool ok = mbar_wait_warp((e & 1) ? &vfull[st] : &kfull[st], (uint32_t)(((nkt + (e >> 1)) / CA_STAGES) & 1), p.spin);
      if (!ok) { if (lane == 0) { *abort_flag = 1; if (p.status) set_status(p.status, ST_TIMEOUT, 439, blockIdx.y, e); } alive = false; }
      return ((e & 1) ? sV : sK) + st * CA_TILE;
    };
    auto diag_done = [&](int e) {                                // the tile's threads are done with it: its place may be filled again
      asm volatile("bar.sync %0, 128;" ::"r"(1 + t) : "memory");
      if (lr == 0) {                                             // two arrivals per place, as from the MMA warps
        uint64_t *eb = (e & 1) ? &vempty[(nkt + (e >> 1)) % CA_STAGES] : &kempty[(nkt + (e >> 1)) % CA_STAGES];
        mbar_arrive(eb);
        if (!two_heads) mbar_arrive(eb);
      }
    };
    if (DIAG) {
      doff = ((size_t)(rv ? trow + lr : 0) * p.G + g) * CA_HD;
      float d[CA_MAX_DIAG];
#pragma unroll
      for (int s = 0; s < CA_MAX_DIAG; s++) d[s] = 0.0f;
      auto dot8 = [](const uint4 &a, const uint4 &b) {
        const float2 a0 = bf2(a.x), a1 = bf2(a.y), a2 = bf2(a.z), a3 = bf2(a.w), b0 = bf2(b.x), b1 = bf2(b.y), b2 = bf2(b.z), b3 = bf2(b.w);
        return ((a0.x * b0.x + a0.y * b0.y) + (a1.x * b1.x + a1.y * b1.y)) + ((a2.x * b2.x + a2.y * b2.y) + (a3.x * b3.x + a3.y * b3.y));
      };
      if (diag_ring) {
#pragma unroll
        for (int s = 0; s < CA_MAX_DIAG; s++)
          if (s < p.J) {
            const int e = two_heads ? s : 2 * s + t;
            unsigned char *kt = diag_wait(e);
            if (alive) {
#pragma unroll 4
              for (int c = 0; c < 16; c++) d[s] += dot8(*chunk(qt, lr, c), *chunk(kt, lr, c));
            }
            diag_done(e);
          }
      } else if (p.J > 0 && alive && nt > 0) {
#pragma unroll 2
        for (int c = 0; c < 16; c++) {
          const uint4 qv = *chunk(qt, lr, c);
#pragma unroll
          for (int s = 0; s < CA_MAX_DIAG; s++)
            if (s < p.J) d[s] += dot8(qv, ld_row8(p.kd + s * dstep + doff + c * 8));
        }
      }
      float M = mx;
#pragma unroll
      for (int s = 0; s < CA_MAX_DIAG; s++)
        if (s < p.J) M = fmaxf(M, d[s]);
      fo = mx == -INFINITY ? 0.0f : ex2((mx - M) * sc);          // every causal score -inf: the row has no causal part
      l *= fo;
      lrnd *= fo;
#pragma unroll
      for (int s = 0; s < CA_MAX_DIAG; s++) {
        wd[s] = s < p.J ? exp2f((d[s] - M) * sc) : 0.0f;
        l += wd[s];
        lrnd += wd[s];
      }
      if (p.lse && rv && alive && nt > 0) p.lse[(size_t)(trow + lr) * p.H + head] = logf(l) + M * rsqrtf((float)CA_HD);
    }
    const float div = BRIEF ? lrnd : l, inv = div > 0.0f ? 1.0f / div : 0.0f;
    __syncwarp();                                                // every lane has read its q row: the tile becomes the output staging
    auto add8 = [](float *o, float w, const uint4 &v) {
      const float2 v0 = bf2(v.x), v1 = bf2(v.y), v2 = bf2(v.z), v3 = bf2(v.w);
      o[0] += w * v0.x; o[1] += w * v0.y; o[2] += w * v1.x; o[3] += w * v1.y; o[4] += w * v2.x; o[5] += w * v2.y; o[6] += w * v3.x; o[7] += w * v3.y;
    };
    auto put32 = [&](int c, const float *o) {
#pragma unroll
      for (int u = 0; u < 4; u++)
        *chunk(qt, lr, c * 4 + u) = make_uint4(pack2(o[u * 8] * inv, o[u * 8 + 1] * inv), pack2(o[u * 8 + 2] * inv, o[u * 8 + 3] * inv),
                                               pack2(o[u * 8 + 4] * inv, o[u * 8 + 5] * inv), pack2(o[u * 8 + 6] * inv, o[u * 8 + 7] * inv));
    };
    if (DIAG && diag_ring) {
      float o[CA_HD];                                            // the whole row in registers: every step's values pass by once
      if (alive && nt > 0) {
#pragma unroll
        for (int c = 0; c < 4; c++) tmem_ld32(my_o + c * 32, o + c * 32);
        tmem_ld_wait();
#pragma unroll
        for (int e = 0; e < CA_HD; e++) o[e] *= fo;
      }
#pragma unroll 1
      for (int s = 0; s < p.J; s++) {
        const int e = p.J * nb + (two_heads ? s : 2 * s + t);
        unsigned char *vt = diag_wait(e);
        if (alive && nt > 0) {
          float w = 0.0f;
#pragma unroll
          for (int z = 0; z < CA_MAX_DIAG; z++) w = z == s ? wd[z] : w;
#pragma unroll
          for (int c = 0; c < 16; c++) add8(o + c * 8, w, *chunk(vt, lr, c));
        }
        diag_done(e);
      }
      if (alive && nt > 0) {
#pragma unroll
        for (int c = 0; c < 4; c++) put32(c, o + c * 32);
      }
    } else if (alive && nt > 0) {
#pragma unroll 1
      for (int c = 0; c < 4; c++) {
        float o[32];
        tmem_ld32(my_o + c * 32, o);
        tmem_ld_wait();
        if (DIAG) {
#pragma unroll
          for (int e = 0; e < 32; e++) o[e] *= fo;
#pragma unroll
          for (int s = 0; s < CA_MAX_DIAG; s++)
            if (s < p.J) {
#pragma unroll
              for (int u = 0; u < 4; u++) add8(o + u * 8, wd[s], ld_row8(p.vd + s * dstep + doff + c * 32 + u * 8));
            }
        }
        put32(c, o);
      }
    }
    __syncwarp();
    // A warp that gave up: where there are no status words to say so, its rows are NaN, never what the buffer held before.
    if (nt > 0 && (alive || !p.status)) {
      if (DIAG && !alive && p.lse && rv) p.lse[(size_t)(trow + lr) * p.H + head] = __int_as_float(0x7fffffff);
      // a warp's 32 rows, two whole rows (256 bytes each) per instruction
      const int rw = (warp & 3) * 32;
#pragma unroll 4
      for (int i = 0; i < 16; i++) {
        const int r = rw + 2 * i + (lane >> 4), c = lane & 15;
        if (r < nr) {
          bf16 *dst = p.out + ((size_t)(trow + r) * p.H + head) * CA_HD + c * 8;
          const uint4 v = alive ? *chunk(qt, r, c) : make_uint4(~0u, ~0u, ~0u, ~0u);
          if (DIAG && p.narrow) { *(uint2 *)dst = make_uint2(v.x, v.y); *(uint2 *)(dst + 4) = make_uint2(v.z, v.w); }
          else *(uint4 *)dst = v;
        }
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (*abort_flag && threadIdx.x == 0) {            // no copy may still be landing when the CTA exits
    mbar_wait(q_bar, 0, p.spin);
    for (int kv = 0; kv < 2; kv++)
      for (int j = max(0, n_filled[kv] - CA_STAGES); j < n_filled[kv]; j++) mbar_wait(kv ? &vfull[j % CA_STAGES] : &kfull[j % CA_STAGES], (uint32_t)((j / CA_STAGES) & 1), p.spin);
  }
  if (warp == 9) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512) : "memory");
}

}  // namespace

bool causal_attn_supported(int head_dim, int page_size) { return head_dim == CA_HD && (page_size == 16 || page_size == 32 || page_size == 64); }

int launch_causal_attn(const CausalArgs &a, cudaStream_t s) {
  if (a.J > CA_MAX_DIAG || a.H % a.G) return -1;
  const int grp = a.H / a.G;
  const CUtensorMap *mk = kv_map(a.pool.k, a.pm.num_pages, a.G, a.pm.page_size, CA_HD, 1), *mv = kv_map(a.pool.v, a.pm.num_pages, a.G, a.pm.page_size, CA_HD, 1);
  CUtensorMap mq, mkd, mvd;
  memset(&mkd, 0, sizeof mkd);
  memset(&mvd, 0, sizeof mvd);
  if (!mk || !mv || !q_map(&mq, a.q, a.q_rows, a.H, CA_T)) return -6;
  CausalParams p;
  memset(&p, 0, sizeof p);
  p.pm = a.pm; p.out = a.out; p.H = a.H; p.G = a.G; p.T = a.T; p.J = a.J; p.blocks = a.blocks; p.kd = a.kd; p.vd = a.vd; p.lse = a.lse;
  p.narrow = (((uintptr_t)a.out | (uintptr_t)a.kd | (uintptr_t)a.vd) & 15) ? 1 : 0;
  if (a.J > 0 && !p.narrow && (!diag_map(&mkd, a.kd, a.J, a.T, a.G, CA_T) || !diag_map(&mvd, a.vd, a.J, a.T, a.G, CA_T))) return -6;
  p.status = a.status;
  p.test = tl_causal_test;
  p.spin = p.test == CAUSAL_TEST_WITHHOLD ? 2000u : tc::SPIN_LIMIT;
  const int br = causal_block_rows(grp);
  dim3 grid(grp % 2 == 0 ? a.H / 2 : a.H, a.blocks ? a.n_blocks : (a.T + br - 1) / br);
  static SmemLimit limit[3];
  const int form = a.blocks ? 0 : a.T > CA_BRIEF ? 1 : 2;
  auto kern = form == 0 ? attn_causal_kernel<false, false> : form == 1 ? attn_causal_kernel<true, false> : attn_causal_kernel<true, true>;
  if (!limit[form].ensure(kern, CA_SMEM)) return -6;
  launch_k(kern, grid, dim3(CA_THREADS), (size_t)CA_SMEM, s, mq, *mk, *mv, mkd, mvd, p);
  return 0;
}

}  // namespace spec

// ------------------------------------------------------------------------------------------------
// Training-time-test attention (Section 3.2, the figure of the attention masks during training-time test).
//
// While the draft model is trained, its own outputs are fed back for further simulated steps.  At simulated step j a
// query at slot i sees the ORIGINAL sequence causally (keys 0..i of the native step: an ordinary lower-triangular mask)
// and, of every earlier simulated step s = 1..j, only the entry at its own slot i (a diagonal mask).  The diagonal part is
// j dot products per (slot, head): the causal kernel computes them as such after the key loop, when the row's statistics
// and its O are at hand, and folds them into the same softmax.  Nothing passes through global memory in between, so the
// call needs no scratch; the parameter stays in the interface.
extern "C" size_t spec_ttt_attention_scratch_bytes(int32_t T, int32_t n_heads, int32_t n_kv_heads, int32_t head_dim) {
  if (T < 1 || n_heads < 1 || n_kv_heads < 1 || n_heads % n_kv_heads || head_dim != 128) return 0;
  return 256;
}

extern "C" int spec_debug_causal(int32_t mode) {
  if (mode < spec::CAUSAL_TEST_OFF || mode > spec::CAUSAL_TEST_WITHHOLD) return SPEC_ERR_INVALID_CFG;
  spec::tl_causal_test = mode;
  return SPEC_OK;
}

extern "C" int spec_ttt_attention(const void *q, const void *k_pool, const void *v_pool, const int32_t *page_table,
                                  int32_t pages_per_seq, int32_t page_size, const void *k_diag, const void *v_diag, int32_t n_steps,
                                  void *out, float *lse, int32_t T, int32_t H, int32_t G, int32_t hd, void *scratch, void *stream) {
  using namespace spec;
  if (!q || !k_pool || !v_pool || !page_table || !out || !scratch || (n_steps > 0 && (!k_diag || !v_diag))) return SPEC_ERR_NULL;
  if (T < 1 || H < 1 || G < 1 || H % G || n_steps < 0 || n_steps > CA_MAX_DIAG) return SPEC_ERR_INVALID_CFG;
  if (!causal_attn_supported(hd, page_size) || (long long)pages_per_seq * page_size < T) return SPEC_ERR_UNSUPPORTED;
  CausalArgs a;
  a.q = (const bf16 *)q; a.q_rows = T;
  a.pool = KvPool{(void *)k_pool, (void *)v_pool};
  a.pm = PageMap{page_table, pages_per_seq, page_size, 1 << 20};
  a.out = (bf16 *)out; a.H = H; a.G = G; a.T = T;
  a.kd = n_steps ? (const bf16 *)k_diag : nullptr; a.vd = n_steps ? (const bf16 *)v_diag : nullptr; a.J = n_steps; a.lse = lse;
  if (launch_causal_attn(a, (cudaStream_t)stream)) return SPEC_ERR_CUDA;
  attn_fast_forget_maps();
  return cudaGetLastError() == cudaSuccess ? SPEC_OK : SPEC_ERR_CUDA;
}
