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
template <int R, int C>
__global__ void __launch_bounds__(128) gemm_skinny_kernel(const float *__restrict__ x, SkinnyWeights sw, float *__restrict__ out, int rows,
                                                          int O, int I, int ldo) {
  pdl_wait();
  pdl_trigger();
  constexpr int NV = R * C;
  const int lane = threadIdx.x & 31;
  const int o0 = (blockIdx.x * 4 + (threadIdx.x >> 5)) * C, r0 = blockIdx.y * R;
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
  for (int k = lane * 4; k < I; k += 128) {           // I % 4 == 0
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
#pragma unroll
  for (int i = 0; i < NV / 32; i++) {
    const int e = lane * (NV / 32) + i, r = r0 + e / C, o = o0 + e % C;
    if (r < rows && o < O) out[(size_t)r * ldo + o] = v[i];
  }
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
  auto go = [&](auto kern, int R, int C) { launch_k(kern, dim3((O + 4 * C - 1) / (4 * C), (rows + R - 1) / R), dim3(128), 0, s, x, sw, out, rows, O, I, ldo); };
  if (rows <= 4) go(gemm_skinny_kernel<4, 8>, 4, 8);
  else if (rows <= 8) go(gemm_skinny_kernel<8, 4>, 8, 4);
  else if (rows <= 16) go(gemm_skinny_kernel<16, 2>, 16, 2);
  else go(gemm_skinny_kernel<32, 2>, 32, 2);
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
