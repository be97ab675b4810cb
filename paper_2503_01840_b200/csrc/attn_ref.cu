// Plain tree-masked paged GQA attention (Section 2.2 "tree attention"): one CTA per (row, query head),
// two-pass softmax with the scores in shared memory.  Used by the fp32 model and as a debugging
// stand-in for the tensor-core kernel on bf16 models.
#include "common.cuh"

#include <algorithm>

namespace spec {

// four consecutive elements; VEC: one 16-byte (fp32) or 8-byte (bf16) load, for rows that start on such a boundary
template <bool VEC> __device__ __forceinline__ float4 load4(const float *p) {
  if (VEC) return *(const float4 *)p;
  return make_float4(p[0], p[1], p[2], p[3]);
}
template <bool VEC> __device__ __forceinline__ float4 load4(const bf16 *p) {
  if (VEC) {
    const uint2 u = *(const uint2 *)p;
    const float2 a = __bfloat1622float2(*(const __nv_bfloat162 *)&u.x), b = __bfloat1622float2(*(const __nv_bfloat162 *)&u.y);
    return make_float4(a.x, a.y, b.x, b.y);
  }
  return make_float4(to_f32(p[0]), to_f32(p[1]), to_f32(p[2]), to_f32(p[3]));
}

// A launch of a wave or two is bound by latency: a row attends tens to hundreds of keys.  So there (AHEAD) are four dependent round
// trips and no more for up to 8192 / head_dim keys: metadata, page ids, K and V rows together, output.  Four threads share a key's dot product
// (256 keys a round, their page ids and then their rows requested at once), and a thread's first V_AHEAD values, whose addresses need no
// score, are requested before the scores.  The value pass splits the keys over the threads that are left beside hd / 4 dimension groups.
// Tiny fp32 model, replayed step with the register-resident top-K: 214 -> 189 us at 64 tokens,
// 275 -> 213 at 250, 386 -> 253 at 600.
// That takes 128 registers and 256 threads, two CTAs an SM.  A larger grid is bound by the requests in flight on the whole chip and wants
// the 40 registers and 128 threads of the form without reading ahead, eleven CTAs an SM.
template <bool AHEAD> struct ArShape {
  static constexpr int THREADS = AHEAD ? 256 : 128, KEY_ROUNDS = AHEAD ? 4 : 1, V_AHEAD = AHEAD ? 8 : 0, PER_SM = AHEAD ? 2 : 10;
  static constexpr int STATIC_SMEM = (AHEAD ? 2 : 1) * (THREADS / 32) * (int)sizeof(float);      // red
};
template <typename T, bool VEC, bool AHEAD>
__global__ void __launch_bounds__(ArShape<AHEAD>::THREADS, ArShape<AHEAD>::PER_SM) attn_ref_kernel(const T *__restrict__ q, KvPool pool, PageMap pm, RowMeta m,
                                                       int tail_len, T *__restrict__ out, int H, int G, int hd) {
  constexpr int AR_THREADS = ArShape<AHEAD>::THREADS, V_AHEAD = ArShape<AHEAD>::V_AHEAD;
  pdl_wait();
  pdl_trigger();
  extern __shared__ __align__(16) float smem[];
  float *qs = smem;            // [hd]
  float *sc = smem + hd;       // [ctx + tail_len]
  float4 *part = (float4 *)smem;   // [AR_THREADS], over both once they are done with
  __shared__ float red[AHEAD ? 2 : 1][AR_THREADS / 32];
  const int r = blockIdx.x, h = blockIdx.y, g = h / (H / G);
  const int seq = m.seq[r], ctx = m.ctx[r], tb = m.tail_base[r];
  const uint64_t mlo = m.mask_lo[r], mhi = m.mask_hi[r];
  for (int i = threadIdx.x; i < hd; i += AR_THREADS) qs[i] = to_f32(q[((size_t)r * H + h) * hd + i]);
  T *o = out + ((size_t)r * H + h) * hd;
  if (seq < 0) {
    for (int i = threadIdx.x; i < hd; i += AR_THREADS) o[i] = from_f32<T>(0.0f);
    return;
  }
  const int nk = ctx + tail_len, ps = pm.page_size, psh = (ps & (ps - 1)) == 0 ? __ffs(ps) - 1 : -1;
  const T *Kp = (const T *)pool.k, *Vp = (const T *)pool.v;
  const int32_t *tbl = pm.table + (size_t)seq * pm.pages_per_seq;
  // first element of the row of a position, from its page
  auto page_of = [&](int pos) { return tbl[psh >= 0 ? pos >> psh : pos / ps]; };
  auto row_at = [&](int page, int pos) { return (((size_t)page * G + g) * ps + (psh >= 0 ? pos & (ps - 1) : pos % ps)) * hd; };
  auto pos_of = [&](int j) { return j < ctx ? j : tb + (j - ctx); };
  auto visible = [&](int j) {
    const int t = j - ctx;
    return j < nk && (t < 0 || (t < 64 ? ((mlo >> t) & 1ull) : ((mhi >> (t - 64)) & 1ull)));
  };
  const int n_dim = hd >> 2;
  const int n_grp = n_dim <= AR_THREADS ? AR_THREADS / n_dim : 0, dim = n_grp ? threadIdx.x % n_dim : 0, grp = n_grp ? threadIdx.x / n_dim : 0;
  const bool has_v = n_grp && grp < n_grp;               // thread = (four dimensions, every n_grp-th key)
  // ---- page ids of the first keys and of this thread's first values, then those values
  constexpr int KR = ArShape<AHEAD>::KEY_ROUNDS;         // rounds of AR_THREADS / 4 keys in flight
  const int sub = threadIdx.x & 3, key0 = threadIdx.x >> 2;
  int kpage[KR];
  auto key_pages = [&](int j0) {
#pragma unroll
    for (int u = 0; u < KR; u++) {
      const int j = j0 + u * (AR_THREADS / 4) + key0;
      kpage[u] = visible(j) ? page_of(pos_of(j)) : -1;
    }
  };
  key_pages(0);
  float4 vv[AHEAD ? V_AHEAD : 1];
  if constexpr (AHEAD) {
    int vpage[V_AHEAD];
#pragma unroll
    for (int u = 0; u < V_AHEAD; u++) {
      const int j = grp + u * n_grp;
      vpage[u] = has_v && visible(j) ? page_of(pos_of(j)) : -1;
    }
#pragma unroll
    for (int u = 0; u < V_AHEAD; u++) vv[u] = vpage[u] >= 0 ? load4<VEC>(Vp + row_at(vpage[u], pos_of(grp + u * n_grp)) + dim * 4) : make_float4(0.f, 0.f, 0.f, 0.f);
  }
  __syncthreads();
  const float scale = 1.0f / sqrtf((float)hd);
  float mx = -INFINITY;
  for (int j0 = 0; j0 < nk; j0 += KR * (AR_THREADS / 4)) {      // all four threads of a key take part
    if (j0 > 0) key_pages(j0);
    const T *kr[KR];
    float d[KR];
#pragma unroll
    for (int u = 0; u < KR; u++) {
      kr[u] = kpage[u] >= 0 ? Kp + row_at(kpage[u], pos_of(j0 + u * (AR_THREADS / 4) + key0)) : nullptr;
      d[u] = 0.0f;
    }
#pragma unroll 4
    for (int i = sub * 4; i < hd; i += 16) {              // hd is a multiple of 16
      const float4 b = *(const float4 *)(qs + i);
#pragma unroll
      for (int u = 0; u < KR; u++)
        if (kr[u]) {
          const float4 a = load4<VEC>(kr[u] + i);
          d[u] = fmaf(b.x, a.x, fmaf(b.y, a.y, fmaf(b.z, a.z, fmaf(b.w, a.w, d[u]))));
        }
    }
#pragma unroll
    for (int u = 0; u < KR; u++) {
      const int j = j0 + u * (AR_THREADS / 4) + key0;
      float t = d[u] + __shfl_xor_sync(0xffffffffu, d[u], 1);
      t += __shfl_xor_sync(0xffffffffu, t, 2);
      const float s = kpage[u] >= 0 ? t * scale : -INFINITY;
      if (sub == 0 && j < nk) sc[j] = s;
      mx = fmaxf(mx, s);
    }
  }
  for (int off = 16; off > 0; off >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, off));
  if ((threadIdx.x & 31) == 0) red[0][threadIdx.x >> 5] = mx;
  __syncthreads();
  mx = red[0][0];
#pragma unroll
  for (int w = 1; w < AR_THREADS / 32; w++) mx = fmaxf(mx, red[0][w]);
  constexpr int SUMS = AHEAD ? 1 : 0;                     // (without reading ahead the sums take the maxima's place)
  if (!AHEAD) __syncthreads();
  float sum = 0.0f;
  for (int j = threadIdx.x; j < nk; j += AR_THREADS) {
    float e = (sc[j] == -INFINITY) ? 0.0f : expf(sc[j] - mx);
    sc[j] = e;
    sum += e;
  }
  for (int off = 16; off > 0; off >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, off);
  if ((threadIdx.x & 31) == 0) red[SUMS][threadIdx.x >> 5] = sum;
  __syncthreads();
  sum = red[SUMS][0];
#pragma unroll
  for (int w = 1; w < AR_THREADS / 32; w++) sum += red[SUMS][w];
  const float inv = 1.0f / sum;
  if (!n_grp) {                                           // more groups of four dimensions than threads: a thread takes several, over all keys
    for (int dm = threadIdx.x; dm < n_dim; dm += AR_THREADS) {
      float4 acc = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
#pragma unroll 4
      for (int j = 0; j < nk; j++) {
        const float p = sc[j];
        if (p == 0.0f) continue;
        const float4 a = load4<VEC>(Vp + row_at(page_of(pos_of(j)), pos_of(j)) + dm * 4);
        acc.x = fmaf(p, a.x, acc.x); acc.y = fmaf(p, a.y, acc.y); acc.z = fmaf(p, a.z, acc.z); acc.w = fmaf(p, a.w, acc.w);
      }
      o[dm * 4] = from_f32<T>(acc.x * inv); o[dm * 4 + 1] = from_f32<T>(acc.y * inv);
      o[dm * 4 + 2] = from_f32<T>(acc.z * inv); o[dm * 4 + 3] = from_f32<T>(acc.w * inv);
    }
    return;
  }
  float4 acc = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
  if (has_v) {
#pragma unroll
    for (int u = 0; u < V_AHEAD; u++) {
      const int j = grp + u * n_grp;
      const float p = j < nk ? sc[j] : 0.0f;
      if (p == 0.0f) continue;                            // a hidden key counts nothing, whatever its value holds
      acc.x = fmaf(p, vv[u].x, acc.x); acc.y = fmaf(p, vv[u].y, acc.y); acc.z = fmaf(p, vv[u].z, acc.z); acc.w = fmaf(p, vv[u].w, acc.w);
    }
#pragma unroll 4
    for (int j = grp + V_AHEAD * n_grp; j < nk; j += n_grp) {
      const float p = sc[j];
      if (p == 0.0f) continue;
      const float4 a = load4<VEC>(Vp + row_at(page_of(pos_of(j)), pos_of(j)) + dim * 4);
      acc.x = fmaf(p, a.x, acc.x); acc.y = fmaf(p, a.y, acc.y); acc.z = fmaf(p, a.z, acc.z); acc.w = fmaf(p, a.w, acc.w);
    }
  }
  __syncthreads();
  part[threadIdx.x] = acc;
  __syncthreads();
  if ((int)threadIdx.x < n_dim) {
    for (int e = 1; e < n_grp; e++) {
      const float4 a = part[e * n_dim + threadIdx.x];
      acc.x += a.x; acc.y += a.y; acc.z += a.z; acc.w += a.w;
    }
    o[threadIdx.x * 4] = from_f32<T>(acc.x * inv); o[threadIdx.x * 4 + 1] = from_f32<T>(acc.y * inv);
    o[threadIdx.x * 4 + 2] = from_f32<T>(acc.z * inv); o[threadIdx.x * 4 + 3] = from_f32<T>(acc.w * inv);
  }
}

// Whether a launch reads ahead: up to two waves of that form, two CTAs an SM (registers).  Above, the form with ten CTAs an SM is faster, up to
// 2.6 times, as long as shared memory (a score for every key that the caller allows for) holds more than three of them.  Called in a row on
// the same few caches, us, reading ahead / not: fp32 hd 64, 240 CTAs 6.9 / 7.4 with 20 keys, 13.0 / 20.8 with 250, 34 / 67 with 1000; 512 CTAs 11.0 / 7.3,
// 23.2 / 21.1, 55 / 54 with 800; 640 CTAs 15.0 / 7.3, 31.8 / 21.6, 79 / 56; 960 CTAs 18.8 / 7.9, 39.6 / 23.1, 125 / 72; bf16 hd 96, 1920 CTAs 39 / 16,
// 107 / 64, 312 / 218.  In a step, whose weights have pushed the cache out of L2, the line lies higher, ms a step with two waves / one: hidden 1024,
// 512 CTAs .749 / .768 at 40 tokens, .932 / .978 at 400; 576 CTAs .890 / .903, 1.075 / 1.125; three waves / two: 640 CTAs .915 / .896, 1.125 / 1.137;
// 768 CTAs .941 / .927, 1.174 / 1.161; bf16 hd 32, 768 CTAs .471 / .439.
// 1920 CTAs of bf16 hd 96, 250 keys of 6000 / 12000 / 16000 / 24000 allowed for: 106 / 65, 107 / 110, 107 / 134, 107 / 184 us.
bool attn_ref_reads_ahead(int rows, int H, int hd, int max_keys) {
  const size_t smem = ((size_t)max_keys + hd) * sizeof(float);
  if (smem + ArShape<true>::STATIC_SMEM > 227 * 1024) return false;      // the last dozen keys that an SM can hold are for the smaller one
  return (long long)rows * H <= 2 * 148 * ArShape<true>::PER_SM || 228 * 1024 / (smem + ArShape<false>::STATIC_SMEM + 1024) <= 3;
}

template <typename T, bool VEC, bool AHEAD>
void launch_attn_ref_form(const T *q, KvPool pool, PageMap pm, RowMeta m, int tail_len, T *out, int rows, int H, int G, int hd, int max_keys, cudaStream_t s) {
  constexpr int threads = ArShape<AHEAD>::THREADS;
  const size_t smem = std::max(((size_t)max_keys + hd) * sizeof(float), threads * sizeof(float4));
  static SmemLimit limit;
  if (smem > 48 * 1024) limit.ensure(attn_ref_kernel<T, VEC, AHEAD>, (int)smem);
  launch_k(attn_ref_kernel<T, VEC, AHEAD>, dim3(rows, H), dim3(threads), smem, s, q, pool, pm, m, tail_len, out, H, G, hd);
}

template <typename T>
void launch_attn_ref(const T *q, KvPool pool, PageMap pm, RowMeta m, int tail_len, T *out, int rows, int H, int G,
                     int hd, int max_keys, cudaStream_t s) {
  const bool vec = (((uintptr_t)pool.k | (uintptr_t)pool.v) & (4 * sizeof(T) - 1)) == 0;      // rows are multiples of 16 elements
  const bool ahead = attn_ref_reads_ahead(rows, H, hd, max_keys);
  auto launch = ahead ? (vec ? launch_attn_ref_form<T, true, true> : launch_attn_ref_form<T, false, true>)
                      : (vec ? launch_attn_ref_form<T, true, false> : launch_attn_ref_form<T, false, false>);
  launch(q, pool, pm, m, tail_len, out, rows, H, G, hd, max_keys, s);
}
template void launch_attn_ref<float>(const float *, KvPool, PageMap, RowMeta, int, float *, int, int, int, int, int,
                                     cudaStream_t);
template void launch_attn_ref<bf16>(const bf16 *, KvPool, PageMap, RowMeta, int, bf16 *, int, int, int, int, int,
                                    cudaStream_t);

}  // namespace spec
