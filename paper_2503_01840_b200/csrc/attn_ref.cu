// Plain tree-masked paged GQA attention (Section 2.2 "tree attention"): one CTA per (row, query head),
// two-pass softmax with the scores in shared memory.  Used by the fp32 model and as a debugging
// stand-in for the tensor-core kernel on bf16 models.
#include "common.cuh"

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

// Bound by latency (a row attends tens to hundreds of keys): four threads share a key's dot product, so that a key row is
// read in 64-byte runs with all its loads in flight, and the value pass splits the KEYS over the threads that are left
// beside hd / 4 dimension groups instead of walking them one after the other (70 keys, 16 CTAs: 45 -> 14 us, cold).
template <typename T, bool VEC>
__global__ void __launch_bounds__(128) attn_ref_kernel(const T *__restrict__ q, KvPool pool, PageMap pm, RowMeta m,
                                                       int tail_len, T *__restrict__ out, int H, int G, int hd) {
  pdl_wait();
  pdl_trigger();
  extern __shared__ __align__(16) float smem[];
  float *qs = smem;            // [hd]
  float *sc = smem + hd;       // [ctx + tail_len]
  float4 *part = (float4 *)smem;   // [128], over both once they are done with
  __shared__ float red[4];
  const int r = blockIdx.x, h = blockIdx.y, g = h / (H / G);
  const int seq = m.seq[r];
  T *o = out + ((size_t)r * H + h) * hd;
  if (seq < 0) {
    for (int i = threadIdx.x; i < hd; i += blockDim.x) o[i] = from_f32<T>(0.0f);
    return;
  }
  const int ctx = m.ctx[r], tb = m.tail_base[r];
  const uint64_t mlo = m.mask_lo[r], mhi = m.mask_hi[r];
  const int nk = ctx + tail_len;
  const T *Kp = (const T *)pool.k, *Vp = (const T *)pool.v;
  for (int i = threadIdx.x; i < hd; i += blockDim.x) qs[i] = to_f32(q[((size_t)r * H + h) * hd + i]);
  __syncthreads();
  const float scale = 1.0f / sqrtf((float)hd);
  float mx = -INFINITY;
  const int sub = threadIdx.x & 3;
  for (int j0 = 0; j0 < nk; j0 += 32) {                  // 32 keys per round: all four threads of a key take part
    const int j = j0 + (threadIdx.x >> 2);
    bool vis = j < nk;
    int pos = j;
    if (j >= ctx) {
      const int t = j - ctx;
      vis = vis && (t < 64 ? ((mlo >> t) & 1ull) : ((mhi >> (t - 64)) & 1ull));
      pos = tb + t;
    }
    float d = 0.0f;
    if (vis) {
      const T *kr = Kp + kv_offset(pm, seq, pos, g, G, hd);
#pragma unroll 4
      for (int i = sub * 4; i < hd; i += 16) {            // hd is a multiple of 16
        const float4 a = load4<VEC>(kr + i), b = *(const float4 *)(qs + i);
        d = fmaf(b.x, a.x, fmaf(b.y, a.y, fmaf(b.z, a.z, fmaf(b.w, a.w, d))));
      }
    }
    d += __shfl_xor_sync(0xffffffffu, d, 1);
    d += __shfl_xor_sync(0xffffffffu, d, 2);
    const float s = vis ? d * scale : -INFINITY;
    if (sub == 0 && j < nk) sc[j] = s;
    mx = fmaxf(mx, s);
  }
  for (int off = 16; off > 0; off >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, off));
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = mx;
  __syncthreads();
  mx = fmaxf(fmaxf(red[0], red[1]), fmaxf(red[2], red[3]));
  __syncthreads();
  float sum = 0.0f;
  for (int j = threadIdx.x; j < nk; j += blockDim.x) {
    float e = (sc[j] == -INFINITY) ? 0.0f : expf(sc[j] - mx);
    sc[j] = e;
    sum += e;
  }
  for (int off = 16; off > 0; off >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, off);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = sum;
  __syncthreads();
  sum = red[0] + red[1] + red[2] + red[3];
  const float inv = 1.0f / sum;
  const int n_dim = hd >> 2;
  if (n_dim > 128) {                                      // more groups of four dimensions than threads: a thread takes several, over all keys
    for (int dim = threadIdx.x; dim < n_dim; dim += 128) {
      float4 acc = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
#pragma unroll 4
      for (int j = 0; j < nk; j++) {
        const float p = sc[j];
        if (p == 0.0f) continue;
        const int pos = j < ctx ? j : tb + (j - ctx);
        const float4 a = load4<VEC>(Vp + kv_offset(pm, seq, pos, g, G, hd) + dim * 4);
        acc.x = fmaf(p, a.x, acc.x); acc.y = fmaf(p, a.y, acc.y); acc.z = fmaf(p, a.z, acc.z); acc.w = fmaf(p, a.w, acc.w);
      }
      o[dim * 4] = from_f32<T>(acc.x * inv); o[dim * 4 + 1] = from_f32<T>(acc.y * inv);
      o[dim * 4 + 2] = from_f32<T>(acc.z * inv); o[dim * 4 + 3] = from_f32<T>(acc.w * inv);
    }
    return;
  }
  // values: thread = (four dimensions, every n_grp-th key)
  const int n_grp = 128 / n_dim, dim = threadIdx.x % n_dim, grp = threadIdx.x / n_dim;
  float4 acc = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
  if (grp < n_grp) {
#pragma unroll 4
    for (int j = grp; j < nk; j += n_grp) {
      const float p = sc[j];
      if (p == 0.0f) continue;
      const int pos = j < ctx ? j : tb + (j - ctx);
      const float4 a = load4<VEC>(Vp + kv_offset(pm, seq, pos, g, G, hd) + dim * 4);
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

size_t attn_ref_smem_bytes(int max_keys, int hd) {
  const size_t n = ((size_t)max_keys + hd) * sizeof(float);
  return n < 128 * sizeof(float4) ? 128 * sizeof(float4) : n;
}

template <typename T>
void launch_attn_ref(const T *q, KvPool pool, PageMap pm, RowMeta m, int tail_len, T *out, int rows, int H, int G,
                     int hd, int max_keys, cudaStream_t s) {
  size_t smem = attn_ref_smem_bytes(max_keys, hd);
  const bool vec = (((uintptr_t)pool.k | (uintptr_t)pool.v) & (4 * sizeof(T) - 1)) == 0;      // rows are multiples of 16 elements
  auto kern = vec ? attn_ref_kernel<T, true> : attn_ref_kernel<T, false>;
  static size_t configured[4] = {0, 0, 0, 0};
  int which = (sizeof(T) == 4 ? 0 : 1) + (vec ? 2 : 0);
  if (smem > 48 * 1024 && smem > configured[which]) {
    cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    configured[which] = smem;
  }
  launch_k(kern, dim3(rows, H), dim3(128), smem, s, q, pool, pm, m, tail_len, out, H, G, hd);
}
template void launch_attn_ref<float>(const float *, KvPool, PageMap, RowMeta, int, float *, int, int, int, int, int,
                                     cudaStream_t);
template void launch_attn_ref<bf16>(const bf16 *, KvPool, PageMap, RowMeta, int, bf16 *, int, int, int, int, int,
                                    cudaStream_t);

}  // namespace spec
