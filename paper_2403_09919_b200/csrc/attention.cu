// Tree-masked attention of the verification forward (Sections 3.3, 3.4).
//
// Row m of sequence b attends the cache slots [0, n_cache[m]) of its sequence and, under tree
// attention, the packed rows j whose bit is set in its mask row; those rows' K/V were written
// to the provisional slots n_cache[m] + j by the rotary kernel, so every key is read from the
// cache.  One CTA per (row, head); each warp walks a strided share of the keys with an online
// softmax and the warps' partial results are merged in shared memory.  Bound by latency: a warp takes ATT_UNROLL keys at
// a time (their K and V requested together, one pass over the running maximum), and everything that the launches ahead
// of the chain wrote -- row tables, tree mask -- is read before the wait.
#include "rd_internal.cuh"
#include "pdl.cuh"

namespace rd {

constexpr int ATT_WARPS = 4;
constexpr int ATT_UNROLL = 4;

// E consecutive elements.  Coherent loads (the rows of this pass were written by the launch before, which may still have
// been running when this CTA started; the acquire of the wait drops what the L1 held from before it) that do keep
// lines in the L1: the rows of a prompt that share an SM read the same keys.
template <int E> __device__ __forceinline__ void load_e(const float* p, float (&v)[E]) {
  if constexpr (E == 2) { const float2 t = __ldca(reinterpret_cast<const float2*>(p)); v[0] = t.x; v[1] = t.y; }
  else { const float4 t = __ldca(reinterpret_cast<const float4*>(p)); v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w; }
}
template <int E> __device__ __forceinline__ void load_e(const __nv_bfloat16* p, float (&v)[E]) {
#pragma unroll
  for (int e = 0; e < E; e += 2) {
    const uint32_t t = __ldca(reinterpret_cast<const unsigned int*>(p + e));
    v[e] = __uint_as_float(t << 16); v[e + 1] = __uint_as_float(t & 0xffff0000u);
  }
}

template <typename T, int HD>
__global__ void __launch_bounds__(ATT_WARPS * 32) attention_kernel(const float* qkv, const T* kc, const T* vc,
                                                                   T* __restrict__ out, RowTables rt, Dims dm, ChainSync cs) {
  chain_begin(cs);
  constexpr int E = HD / 32;  // elements per lane
  __shared__ int32_t tree_slot[1024];
  __shared__ int n_tree_sh;
  __shared__ float sh_m[ATT_WARPS], sh_l[ATT_WARPS], sh_acc[ATT_WARPS][HD];
  const bool early = cs.signal_ptr != nullptr && cs.wait_ptr != nullptr;
  if (!early) chain_wait_cta(cs);
  const int m = blockIdx.x, h = blockIdx.y;
  if (m >= *rt.m_total) {
    if (early) chain_wait_cta(cs);
    chain_exit(cs);
    return;
  }
  const int b = rt.seq[m];
  const int n_cache = rt.n_cache[m];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;

  if (w == 0) {   // the slots of the row's tree keys, in ascending order: a mask word per lane (MW <= 32)
    uint32_t bits = rt.mask && lane < dm.MW ? rt.mask[((size_t)b * dm.NMAX + rt.local[m]) * dm.MW + lane] : 0u;
    const int room = dm.max_ctx - n_cache - lane * 32;   // bits from here on name slots past the cache
    if (room < 32) bits &= room > 0 ? (1u << room) - 1u : 0u;
    int at = __popc(bits);
    const int mine = at;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, at, o);
      if (lane >= o) at += v;
    }
    if (lane == 31) n_tree_sh = at;
    for (at -= mine; bits; bits &= bits - 1) tree_slot[at++] = n_cache + lane * 32 + __ffs(bits) - 1;
  }
  if (early) chain_wait_cta(cs);
  __syncthreads();
  const int n_keys = n_cache + n_tree_sh;

  float q[E];
  load_e<E>(qkv + (size_t)m * 3 * dm.d + h * HD + lane * E, q);
  const float scale = rsqrtf((float)HD);
#pragma unroll
  for (int e = 0; e < E; ++e) q[e] *= scale;

  const size_t head_base = ((size_t)b * dm.H + h) * dm.max_ctx * HD + lane * E;
  float mx = -INFINITY, l = 0.f, acc[E];
#pragma unroll
  for (int e = 0; e < E; ++e) acc[e] = 0.f;
  for (int j0 = w; j0 < n_keys; j0 += ATT_WARPS * ATT_UNROLL) {
    float k[ATT_UNROLL][E], v[ATT_UNROLL][E], s[ATT_UNROLL];
#pragma unroll
    for (int u = 0; u < ATT_UNROLL; ++u) {
      const int j = min(j0 + u * ATT_WARPS, n_keys - 1);
      const size_t at = head_base + (size_t)(j < n_cache ? j : tree_slot[j - n_cache]) * HD;
      load_e<E>(kc + at, k[u]);
      load_e<E>(vc + at, v[u]);
    }
    float nm = mx;
#pragma unroll
    for (int u = 0; u < ATT_UNROLL; ++u) {
      s[u] = 0.f;
#pragma unroll
      for (int e = 0; e < E; ++e) s[u] = fmaf(q[e], k[u][e], s[u]);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) s[u] += __shfl_xor_sync(0xffffffffu, s[u], o);
      if (j0 + u * ATT_WARPS >= n_keys) s[u] = -INFINITY;
      nm = fmaxf(nm, s[u]);
    }
    const float corr = __expf(mx - nm);   // 0 in the first pass; the batch's first key exists
    l *= corr;
#pragma unroll
    for (int e = 0; e < E; ++e) acc[e] *= corr;
#pragma unroll
    for (int u = 0; u < ATT_UNROLL; ++u) {
      const float p = j0 + u * ATT_WARPS < n_keys ? __expf(s[u] - nm) : 0.f;
      l += p;
#pragma unroll
      for (int e = 0; e < E; ++e) acc[e] = fmaf(p, v[u][e], acc[e]);
    }
    mx = nm;
  }
  if (lane == 0) { sh_m[w] = mx; sh_l[w] = l; }
#pragma unroll
  for (int e = 0; e < E; ++e) sh_acc[w][lane * E + e] = acc[e];
  __syncthreads();
  if (w == 0) {
    float gm = -INFINITY;
#pragma unroll
    for (int i = 0; i < ATT_WARPS; ++i) gm = fmaxf(gm, sh_m[i]);
    float gl = 0.f, o[E];
#pragma unroll
    for (int e = 0; e < E; ++e) o[e] = 0.f;
#pragma unroll
    for (int i = 0; i < ATT_WARPS; ++i) {
      const float c = (sh_m[i] == -INFINITY) ? 0.f : __expf(sh_m[i] - gm);
      gl += sh_l[i] * c;
#pragma unroll
      for (int e = 0; e < E; ++e) o[e] += sh_acc[i][lane * E + e] * c;
    }
    const float inv = gl > 0.f ? 1.f / gl : 0.f;
#pragma unroll
    for (int e = 0; e < E; ++e) out[(size_t)m * dm.d + h * HD + lane * E + e] = from_f<T>(o[e] * inv);
  }
  chain_exit(cs);
}

cudaError_t launch_attention(int dtype, const float* qkv, const void* kcache, const void* vcache, void* out_t,
                             const RowTables& rt, const Dims& dm, int m_max, Chain* chain, cudaStream_t st) {
  dim3 grid(m_max, dm.H);
  const ChainSync cs = chain ? chain->link(grid.x * grid.y, true) : ChainSync{nullptr, 0u, nullptr, nullptr, nullptr};
#define RD_ATT(T, HD) launch_pdl(attention_kernel<T, HD>, grid, ATT_WARPS * 32, 0, st, qkv, (const T*)kcache, (const T*)vcache, (T*)out_t, rt, dm, cs)
  if (dtype == RD_DTYPE_FP32) {
    if (dm.hd == 64) RD_ATT(float, 64); else if (dm.hd == 128) RD_ATT(float, 128); else return cudaErrorInvalidValue;
  } else {
    if (dm.hd == 64) RD_ATT(__nv_bfloat16, 64); else if (dm.hd == 128) RD_ATT(__nv_bfloat16, 128); else return cudaErrorInvalidValue;
  }
#undef RD_ATT
  return cudaGetLastError();
}

}  // namespace rd
