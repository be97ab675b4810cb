// Plain CUDA-core GEMM: out[r][o] = sum_i x[r][i] * w[o][i], fp32 accumulation with FMA.
// This is the fp32 model's GEMM (tensor-core tf32 would not hold a 1e-4 bound) and a debugging
// stand-in for the tcgen05 kernel on bf16 models.
#include <algorithm>

#include "common.cuh"

namespace spec {

template <typename T>
__global__ void __launch_bounds__(256) gemm_ref_kernel(const T *__restrict__ x, const T *__restrict__ w,
                                                       float *__restrict__ out, int rows, int O, int I, int ldo) {
  pdl_wait();
  pdl_trigger();
  constexpr int BM = 64, BN = 64, BK = 16;
  __shared__ float xs[BK][BM + 1];
  __shared__ float ws[BK][BN + 1];
  int r0 = blockIdx.y * BM, o0 = blockIdx.x * BN;
  int tx = threadIdx.x % 16, ty = threadIdx.x / 16;   // tx -> o, ty -> r
  float acc[4][4];
#pragma unroll
  for (int a = 0; a < 4; a++)
#pragma unroll
    for (int b = 0; b < 4; b++) acc[a][b] = 0.0f;
  for (int i0 = 0; i0 < I; i0 += BK) {
    for (int e = threadIdx.x; e < BM * BK; e += 256) {
      int rr = e / BK, kk = e % BK;
      int r = r0 + rr, i = i0 + kk;
      xs[kk][rr] = (r < rows && i < I) ? to_f32(x[(size_t)r * I + i]) : 0.0f;
      int o = o0 + rr;
      ws[kk][rr] = (o < O && i < I) ? to_f32(w[(size_t)o * I + i]) : 0.0f;
    }
    __syncthreads();
#pragma unroll
    for (int kk = 0; kk < BK; kk++) {
      float xv[4], wv[4];
#pragma unroll
      for (int a = 0; a < 4; a++) xv[a] = xs[kk][ty * 4 + a];
#pragma unroll
      for (int b = 0; b < 4; b++) wv[b] = ws[kk][tx * 4 + b];
#pragma unroll
      for (int a = 0; a < 4; a++)
#pragma unroll
        for (int b = 0; b < 4; b++) acc[a][b] = fmaf(xv[a], wv[b], acc[a][b]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int a = 0; a < 4; a++) {
    int r = r0 + ty * 4 + a;
    if (r >= rows) continue;
#pragma unroll
    for (int b = 0; b < 4; b++) {
      int o = o0 + tx * 4 + b;
      if (o < O) out[(size_t)r * ldo + o] = acc[a][b];
    }
  }
}

// The fp32 model's GEMM for few rows.  Its launches are bound by latency, not by bytes or flops (4 rows of a 256 x 256
// weight are 0.5 MFLOP): the tile kernel above walks the contraction in dependent steps of 16 elements with two block
// barriers each, 40 to 80 us per launch.  Here a warp owns C output features for R rows and splits the CONTRACTION over its
// lanes (four consecutive elements each, 128 per step, all loads of a step in flight together); the R * C lane sums are
// added up by a halving exchange (each step swaps half of the values, 31 or 63 shuffles in all instead of five per value).
// Launches of 4 rows x 256..768: 72 -> 5 to 7.5 us under a profiler (cold); a step of the tiny model 1.87 -> 0.32 ms with the
// attention kernel's key split and programmatic dependent launch.
// Several weights that share the input run in one launch (q, k, v; gate, up): feature o belongs to w0 below o1, to w1 below
// o2, else to w2.
struct SkinnyWeights { const float *w0, *w1, *w2; int o1, o2; };
// KS: the block's four warps take the same features and a quarter of the contraction each (added up through shared memory): a
// warp then walks 128 elements of every 512 instead of all.  Taken from 384 elements on (three dependent steps of loads) while the
// blocks, four times as many, are resident together, and where they take two or three waves from the length on at which the shorter
// walk is worth them (launch_skinny).  Tiny request of ten steps 2.76 -> 2.48 ms.
template <int R, int C, bool KS>
__global__ void __launch_bounds__(128) gemm_skinny_kernel(const float *__restrict__ x, SkinnyWeights sw, float *__restrict__ out, int rows,
                                                          int O, int I, int ldo) {
  pdl_wait();
  pdl_trigger();
  constexpr int NV = R * C;
  const int lane = threadIdx.x & 31;
  const int warp = threadIdx.x >> 5, o0 = (KS ? blockIdx.x : blockIdx.x * 4 + warp) * C, r0 = blockIdx.y * R;
  if (o0 >= O) return;
  const float *wr[C];
#pragma unroll
  for (int c = 0; c < C; c++) {
    const int o = min(o0 + c, O - 1);                 // a feature past the end repeats the last one (not stored)
    wr[c] = o < sw.o1 ? sw.w0 + (size_t)o * I : o < sw.o2 ? sw.w1 + (size_t)(o - sw.o1) * I : sw.w2 + (size_t)(o - sw.o2) * I;
  }
  float v[NV];
#pragma unroll
  for (int e = 0; e < NV; e++) v[e] = 0.0f;
#pragma unroll 2
  for (int k = (KS ? warp * 128 : 0) + lane * 4; k < I; k += KS ? 512 : 128) {        // I % 4 == 0
    float4 w[C];
#pragma unroll
    for (int c = 0; c < C; c++) w[c] = *(const float4 *)(wr[c] + k);
#pragma unroll
    for (int r = 0; r < R; r++) {
      const float4 a = *(const float4 *)(x + (size_t)min(r0 + r, rows - 1) * I + k);
#pragma unroll
      for (int c = 0; c < C; c++) v[r * C + c] = fmaf(a.x, w[c].x, fmaf(a.y, w[c].y, fmaf(a.z, w[c].z, fmaf(a.w, w[c].w, v[r * C + c]))));
    }
  }
  // halving exchange: afterwards lane l holds the sums of values l * NV / 32 ..
#pragma unroll
  for (int step = 0; step < 5; step++) {
    const int off = 16 >> step, half = NV >> (step + 1);
    const bool up = lane & off;
#pragma unroll
    for (int i = 0; i < half; i++) {
      const float keep = up ? v[i + half] : v[i], send = up ? v[i] : v[i + half];
      v[i] = keep + __shfl_xor_sync(0xffffffffu, send, off);
    }
  }
  if constexpr (KS) {
    __shared__ float part[3][NV];
    if (warp)
#pragma unroll
      for (int i = 0; i < NV / 32; i++) part[warp - 1][lane * (NV / 32) + i] = v[i];
    __syncthreads();
    if (warp) return;
#pragma unroll
    for (int i = 0; i < NV / 32; i++) {
      const int e = lane * (NV / 32) + i;
      v[i] = (v[i] + part[0][e]) + (part[1][e] + part[2][e]);
    }
  }
#pragma unroll
  for (int i = 0; i < NV / 32; i++) {
    const int e = lane * (NV / 32) + i, r = r0 + e / C, o = o0 + e % C;
    if (r < rows && o < O) out[(size_t)r * ldo + o] = v[i];
  }
}

// The same kernel with what surrounds it in a decoder layer: RMSNorm on the way in (the pending partial result is added to the
// residual stream, the norm's factor is applied to the finished sums, the sum of squares comes out of the same loop) and RoPE
// with the cache write, or SiLU(gate) * up, on the way out.  A warp's features come in pairs (rotation partners j and j + hd / 2
// of a head, gate and up), which end in neighbouring lanes.  The new residual rows go to a buffer of their own (the last block does
// nothing else): other blocks still read the old one.  A step of the tiny model is a chain of dependent launches of 4 to
// 5 us each, so what counts is their number: five a layer instead of nine,
// 48 a step instead of 76: a request of ten steps 3.06 -> 2.76 ms.  (With a branch per row around the added partial result, and the cache
// slot looked up in front of the loop, it was 3.34: every load must be on its way before the first is used.)
struct NormIn {
  const float *x, *add;        // [rows][I]; add may be null
  float *x_out, *taps;         // x + add (may be null: unchanged); feature taps [rows][3 I], slots by tap_mask
  int tap_mask;
  const float *gain;
  float eps;
};
enum { NOUT_PLAIN = 0, NOUT_QKV = 1, NOUT_SWIGLU = 2 };
struct NormOut {
  float *out; int ldo;                                   // NOUT_PLAIN; NOUT_SWIGLU: act [rows][pairs]
  const float2 *cs; RowMeta m; float *q, *kp, *vp; PageMap pm; int H, G, hd; int32_t *status;   // NOUT_QKV
};
template <int R, int C, int OUT, bool ADD>
__global__ void __launch_bounds__(128) gemm_norm_kernel(NormIn in, SkinnyWeights sw, NormOut no, int rows, int O, int I) {
  pdl_wait();
  pdl_trigger();
  constexpr int NV = R * C, P = C / 2;
  static_assert(NV == 32, "every lane ends with one value");
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int u0 = (blockIdx.x * 4 + warp) * (OUT == NOUT_PLAIN ? C : P), units = OUT == NOUT_PLAIN ? O : O / 2;    // features, or pairs of features
  if (blockIdx.x + 1 == gridDim.x) {                   // the new residual rows and the taps: the last block
    if (in.x_out || in.tap_mask)
      for (int i = threadIdx.x; i < rows * (I / 4); i += 128) {
        const int r = i / (I / 4), k = i % (I / 4) * 4;
        const size_t at = (size_t)r * I + k;
        float4 a = *(const float4 *)(in.x + at);
        if (ADD) { const float4 b = *(const float4 *)(in.add + at); a.x += b.x; a.y += b.y; a.z += b.z; a.w += b.w; }
        if (in.x_out) *(float4 *)(in.x_out + at) = a;
#pragma unroll
        for (int s = 0; s < 3; s++)
          if ((in.tap_mask >> s) & 1) *(float4 *)(in.taps + (size_t)r * 3 * I + (size_t)s * I + k) = a;
      }
    return;
  }
  if (u0 >= units) return;
  const int half = OUT == NOUT_QKV ? no.hd >> 1 : 1;
  const float *wr[C];
#pragma unroll
  for (int c = 0; c < C; c++) {
    const int u = min(u0 + (OUT == NOUT_PLAIN ? c : c % P), units - 1);           // past the end: repeats the last (not stored)
    const int o = OUT == NOUT_PLAIN ? u : OUT == NOUT_QKV ? u / half * no.hd + u % half + (c >= P ? half : 0) : u + (c >= P ? units : 0);
    wr[c] = o < sw.o1 ? sw.w0 + (size_t)o * I : o < sw.o2 ? sw.w1 + (size_t)(o - sw.o1) * I : sw.w2 + (size_t)(o - sw.o2) * I;
  }
  // where this lane's value goes: row lane / C, feature (or pair member) lane % C
  const int row = lane / C, c_own = lane % C, unit = u0 + (OUT == NOUT_PLAIN ? c_own : c_own % P);
  const bool mine = row < rows && unit < units;
  float2 cs = make_float2(1.0f, 0.0f);
  int head = 0, seq = -1, kvpos = 0;
  if (OUT == NOUT_QKV && mine) {                       // not used before the sums are there
    head = unit / half;
    seq = no.m.seq[row];
    kvpos = no.m.kvpos[row];
    if (head < no.H + no.G) cs = no.cs[(size_t)row * half + unit % half];
  }
  float v[NV], sq[R];
#pragma unroll
  for (int e = 0; e < NV; e++) v[e] = 0.0f;
#pragma unroll
  for (int r = 0; r < R; r++) sq[r] = 0.0f;
#pragma unroll 1
  for (int k = lane * 4; k < I; k += 128) {           // I % 4 == 0
    float4 w[C];
#pragma unroll
    for (int c = 0; c < C; c++) w[c] = *(const float4 *)(wr[c] + k);
    const float4 g = *(const float4 *)(in.gain + k);
#pragma unroll
    for (int r = 0; r < R; r++) {
      const size_t at = (size_t)min(r, rows - 1) * I + k;
      float4 a = *(const float4 *)(in.x + at);
      if (ADD) { const float4 b = *(const float4 *)(in.add + at); a.x += b.x; a.y += b.y; a.z += b.z; a.w += b.w; }
      sq[r] = fmaf(a.x, a.x, fmaf(a.y, a.y, fmaf(a.z, a.z, fmaf(a.w, a.w, sq[r]))));
      a.x *= g.x; a.y *= g.y; a.z *= g.z; a.w *= g.w;
#pragma unroll
      for (int c = 0; c < C; c++) v[r * C + c] = fmaf(a.x, w[c].x, fmaf(a.y, w[c].y, fmaf(a.z, w[c].z, fmaf(a.w, w[c].w, v[r * C + c]))));
    }
  }
  int page = -1;                                       // cache page of the row, on its way during the exchange
  const bool in_cache = OUT == NOUT_QKV && mine && seq >= 0 && head >= no.H;
  if (in_cache) {
    if (kvpos < 0 || kvpos / no.pm.page_size >= no.pm.pages_per_seq) { set_status(no.status, ST_BOUNDS, 1, row, kvpos); page = -2; }
    else page = no.pm.table[(size_t)seq * no.pm.pages_per_seq + kvpos / no.pm.page_size];
  }
  // halving exchange of the sums (cf. gemm_skinny_kernel), and of the squares down to the lane's own row
#pragma unroll
  for (int step = 0; step < 5; step++) {
    const int off = 16 >> step, hv = NV >> (step + 1), hr = R >> (step + 1);
    const bool up = lane & off;
#pragma unroll
    for (int i = 0; i < hv; i++) {
      const float keep = up ? v[i + hv] : v[i], send = up ? v[i] : v[i + hv];
      v[i] = keep + __shfl_xor_sync(0xffffffffu, send, off);
    }
    if (hr >= 1) {
#pragma unroll
      for (int i = 0; i < hr; i++) {
        const float keep = up ? sq[i + hr] : sq[i], send = up ? sq[i] : sq[i + hr];
        sq[i] = keep + __shfl_xor_sync(0xffffffffu, send, off);
      }
    } else sq[0] += __shfl_xor_sync(0xffffffffu, sq[0], off);
  }
  const float inv = 1.0f / sqrtf(sq[0] / (float)I + in.eps);
  if (OUT == NOUT_PLAIN) {
    if (mine) no.out[(size_t)row * no.ldo + unit] = v[0] * inv;
    return;
  }
  // a: first member of the pair (feature j, gate), b: second (j + hd / 2, up)
  const float own = v[0] * inv, other = __shfl_xor_sync(0xffffffffu, own, P);
  const bool second = c_own >= P;
  const float a = second ? other : own, b = second ? own : other;
  if (mine && OUT == NOUT_SWIGLU && !second) no.out[(size_t)row * units + unit] = (a / (1.0f + expf(-a))) * b;
  if (OUT == NOUT_SWIGLU || !mine) return;
  const int j = unit % half;
  float *kv = nullptr;
  if (in_cache && page != -2) {
    if (page < 0 || page >= no.pm.num_pages) set_status(no.status, ST_BOUNDS, 2, row, page);
    else kv = (head < no.H + no.G ? no.kp : no.vp) + (((size_t)page * no.G + (head - no.H) % no.G) * no.pm.page_size + kvpos % no.pm.page_size) * no.hd;
  }
  float *dst = head < no.H ? no.q + ((size_t)row * no.H + head) * no.hd : kv;
  if (!dst) return;
  float oa = a * cs.x - b * cs.y, ob = b * cs.x + a * cs.y;
  if (head < no.H && seq < 0) oa = ob = 0.0f;           // padding row
  dst[second ? j + half : j] = second ? ob : oa;
}

// When the warp-per-feature kernel is taken: up to 32 rows every weight is read once; up to 256 rows while the weights fit the
// L2 comfortably (they are read once per 32 rows); and in either case only where it is the shorter one.  Its time goes with
// (rows padded to a group) x features x (contraction + 192: the exchange costs as much as 192 elements), spread over the chip
// from a few thousand warps on; the tile kernel's goes with the contraction alone until its 64 x 64 tiles fill the chip (256 of
// them).  The line is a fit to both kernels' times at 900 shapes of 1 to 256 rows, 64 to 128256 features, 16 to 4096 elements (tile / this
// kernel, us, binding included): 256 x 4096 x 64 13.3 / 29.2, x 256 39.4 / 43.6, x 512 72 / 68, x 1024 138 / 125; 64 x 4096 x
// 64 11.5 / 11.8, x 256 31 / 14.7; 32 x 128256 x 64 54 / 99, 4 x 4096 x 256 29 / 12.
static bool skinny_ok(const float *x, const float *w, int rows, int O, int I) {
  if ((I & 3) || (((uintptr_t)x | (uintptr_t)w) & 15)) return false;
  if (rows > 256 || (rows > 32 && (long long)O * I > (4 << 20))) return false;
  const int padded = rows <= 4 ? 4 : rows <= 8 ? 8 : rows <= 16 ? 16 : (rows + 31) / 32 * 32;
  const double tiles = (double)((O + 63) / 64) * ((rows + 63) / 64);
  return (double)padded * O * (I + 192) <= 1.31e6 * I * std::max(1.0, tiles / 256);
}
static void launch_skinny(const float *x, SkinnyWeights sw, float *out, int rows, int O, int I, int ldo, cudaStream_t s) {
  // resident: blocks of the form that the chip holds (by registers); two, three: contraction from which KS may take as many waves of
  // them.  Whole / shared contraction, us: 4 rows x 2048 x 384 (256 blocks) 3.1 / 2.5, x 4096 (512) x 512 3.8 / 3.9, x 1024 5.6 / 4.8, x 8192
  // (1024) x 1024 6.4 / 6.8; 8 rows x 4096 (1024) x 384 3.9 / 4.0, x 512 5.0 / 4.4; 16 rows x 1024 (512) x 384 3.7 / 3.3, x 2048 (1024) x 384
  // 4.1 / 4.7, x 512 5.3 / 4.8; 32 rows x 1024 (512) x 384 4.2 / 4.5, x 512 5.2 / 4.8, x 2048 (1024) x 1024 10.7 / 11.9; 64 rows x 688 (688)
  // x 768 8.5 / 8.8, x 1024 10.5 / 10.0.
  auto go = [&](auto kern, auto split, int R, int C, int resident, int two, int three) {
    const int groups = (rows + R - 1) / R, blocks = (O + C - 1) / C * groups, waves = (blocks + resident - 1) / resident;
    if (blocks <= 1184 && I >= (waves == 1 ? 384 : waves == 2 ? two : waves == 3 ? three : I + 1))
      launch_k(split, dim3((O + C - 1) / C, groups), dim3(128), 0, s, x, sw, out, rows, O, I, ldo);
    else launch_k(kern, dim3((O + 4 * C - 1) / (4 * C), groups), dim3(128), 0, s, x, sw, out, rows, O, I, ldo);
  };
  if (rows <= 4) go(gemm_skinny_kernel<4, 8, false>, gemm_skinny_kernel<4, 8, true>, 4, 8, 444, 1024, 1536);
  else if (rows <= 8) go(gemm_skinny_kernel<8, 4, false>, gemm_skinny_kernel<8, 4, true>, 8, 4, 592, 512, 512);
  else if (rows <= 16) go(gemm_skinny_kernel<16, 2, false>, gemm_skinny_kernel<16, 2, true>, 16, 2, 444, 384, 512);
  else go(gemm_skinny_kernel<32, 2, false>, gemm_skinny_kernel<32, 2, true>, 32, 2, 296, 512, 1024);
}

template <int OUT>
static void launch_norm(const NormIn &in, const SkinnyWeights &sw, const NormOut &no, int rows, int O, int I, cudaStream_t s) {
  auto go = [&](auto kern, int C) { launch_k(kern, dim3((O + 4 * C - 1) / (4 * C) + 1), dim3(128), 0, s, in, sw, no, rows, O, I); };
  auto pick = [&](auto k4, auto k8, auto k16) { if (rows <= 4) go(k4, 8); else if (rows <= 8) go(k8, 4); else go(k16, 2); };
  if (in.add) pick(gemm_norm_kernel<4, 8, OUT, true>, gemm_norm_kernel<8, 4, OUT, true>, gemm_norm_kernel<16, 2, OUT, true>);
  else pick(gemm_norm_kernel<4, 8, OUT, false>, gemm_norm_kernel<8, 4, OUT, false>, gemm_norm_kernel<16, 2, OUT, false>);
}
// Every warp norms all rows for its own two to eight features, so what the launches saved cost grows with rows x contraction.  Steps
// of fp32 models of four layers, separate kernels / these, us: 8 rows 302 / 239 at hidden 256, 317 / 283 at 512, 472 / 436 at 1024, 2239 /
// 2183 at 4096; 16 rows 254 / 250 at 64, 297 / 290 at 256, 324 / 338 at 320, 326 / 349 at 512, 608 / 681 at 1024; 24 rows 264 / 286 at
// hidden 64 already, 32 rows 372 / 584 at 512, 4910 / 12690 at 4096.
bool gemm_norm_ok(const float *const *w, int nw, const float *gain, int rows, int O, int I) {
  if (((uintptr_t)gain & 15) || rows > (I <= 256 ? 16 : 8)) return false;
  for (int j = 0; j < nw; j++)
    if (!skinny_ok(nullptr, w[j], rows, O, I)) return false;
  return true;
}
void launch_norm_gemm(const float *x, const float *add, float *x_out, float *taps, int tap_mask, const float *gain, float eps, const float *w, float *out,
                      int rows, int O, int I, cudaStream_t s) {
  launch_norm<NOUT_PLAIN>(NormIn{x, add, x_out, taps, tap_mask, gain, eps}, SkinnyWeights{w, w, w, O, O}, NormOut{out, O}, rows, O, I, s);
}
void launch_norm_swiglu(const float *x, const float *add, float *x_out, const float *gain, float eps, const float *w_gate, const float *w_up, float *act,
                        int rows, int F, int I, cudaStream_t s) {
  launch_norm<NOUT_SWIGLU>(NormIn{x, add, x_out, nullptr, 0, gain, eps}, SkinnyWeights{w_gate, w_up, w_up, F, 2 * F}, NormOut{act, F}, rows, 2 * F, I, s);
}
void launch_norm_qkv(const float *x, const float *add, float *x_out, float *taps, int tap_mask, const float *gain, float eps, const float *wq,
                     const float *wk, const float *wv, const float2 *cs, RowMeta m, float *q, KvPool pool, PageMap pm, int rows, int H, int G, int hd,
                     int I, int32_t *status, cudaStream_t s) {
  const int o1 = H * hd, o2 = o1 + G * hd;
  launch_norm<NOUT_QKV>(NormIn{x, add, x_out, taps, tap_mask, gain, eps}, SkinnyWeights{wq, wk, wv, o1, o2},
                        NormOut{nullptr, 0, cs, m, q, (float *)pool.k, (float *)pool.v, pm, H, G, hd, status}, rows, o2 + G * hd, I, s);
}

template <typename T>
static void launch_tiles(const T *x, const T *w, float *out, int rows, int O, int I, int ldo, cudaStream_t s) {
  dim3 grid((O + 63) / 64, (rows + 63) / 64);
  launch_k(gemm_ref_kernel<T>, dim3(grid), dim3(256), 0, s, x, w, out, rows, O, I, ldo);
}
template <> void launch_gemm_ref<float>(const float *x, const float *w, float *out, int rows, int O, int I, int ldo, cudaStream_t s) {
  if (skinny_ok(x, w, rows, O, I)) launch_skinny(x, SkinnyWeights{w, w, w, O, O}, out, rows, O, I, ldo, s);
  else launch_tiles(x, w, out, rows, O, I, ldo, s);
}
template <> void launch_gemm_ref<bf16>(const bf16 *x, const bf16 *w, float *out, int rows, int O, int I, int ldo, cudaStream_t s) {
  launch_tiles(x, w, out, rows, O, I, ldo, s);
}
template <typename T>
int launch_gemm_ref_cat(const T *x, const T *const (&w)[3], const int (&O)[3], int nw, float *out, int rows, int I, int ldo, cudaStream_t s) {
  if constexpr (sizeof(T) == 4) {
    bool ok = true;
    for (int j = 0; j < nw; j++) ok = ok && skinny_ok(x, w[j], rows, O[j], I);
    if (ok) {
      const int o1 = O[0], o2 = o1 + O[1];
      launch_skinny(x, SkinnyWeights{w[0], w[1], nw > 2 ? w[2] : w[1], o1, nw > 2 ? o2 : 1 << 30}, out, rows, nw > 2 ? o2 + O[2] : o2, I, ldo, s);
      return 1;
    }
  }
  int col = 0;
  for (int j = 0; j < nw; j++) { launch_gemm_ref<T>(x, w[j], out + col, rows, O[j], I, ldo, s); col += O[j]; }
  return nw;
}
template int launch_gemm_ref_cat<float>(const float *, const float *const (&)[3], const int (&)[3], int, float *, int, int, int, cudaStream_t);
template int launch_gemm_ref_cat<bf16>(const bf16 *, const bf16 *const (&)[3], const int (&)[3], int, float *, int, int, int, cudaStream_t);

}  // namespace spec
