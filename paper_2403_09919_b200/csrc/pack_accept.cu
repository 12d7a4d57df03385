// Dynamic tree attention packing (Section 3.3, Appendix A.1) and greedy acceptance with KV-cache
// compaction (Section 3.4).  Integer work on at most a few thousand entries per sequence: one CTA
// per sequence, everything staged in shared memory, no host involvement.
#include <mutex>

#include "rd_internal.cuh"
#include "pdl.cuh"

namespace rd {

// ---------------------------------------------------------------- pack
// beam' = [root | beam] is [BW][C], C = L+1.  Thread (i, j):
//   owner(i,j) = the first candidate k <= i with beam'[k][0..j] == beam'[i][0..j]   (dedup_prefix)
//   keep(i,j)  = owner == i; packed index = exclusive scan of keep in row-major order (pack_beam)
//   unpack[i][j] = packed index of (owner, j); pos = ctx + j; parent = unpack[i][j-1];
//   mask row = bits unpack[i][0..j].
constexpr int PACK_MAX_ENTRIES = 1024;

__global__ void __launch_bounds__(1024) pack_kernel(const int32_t* __restrict__ beams, const int32_t* __restrict__ root,
                                                     const int32_t* __restrict__ ctx, rd_packed out, Dims dm, int no_tree) {
  pdl_enter();
  __shared__ int32_t tok[PACK_MAX_ENTRIES];
  __shared__ int32_t owner[PACK_MAX_ENTRIES];
  __shared__ int32_t scan[PACK_MAX_ENTRIES];
  __shared__ int32_t warp_tot[32];
  const int b = blockIdx.x, BW = dm.BW, L = dm.L, C = L + 1, E = BW * C;
  const int t = threadIdx.x;
  const int i = t / C, j = t - i * C;
  if (t < E) tok[t] = (j == 0) ? root[b] : beams[((size_t)b * BW + i) * L + (j - 1)];
  __syncthreads();
  int keep = 0, own = 0;
  if (t < E) {
    if (no_tree) {
      own = (j == 0) ? 0 : i;
    } else {
      own = i;
      for (int k = 0; k < i; ++k) {
        bool same = true;
        for (int c = 1; c <= j; ++c) same = same && (tok[k * C + c] == tok[i * C + c]);  // column 0 is the shared root
        if (same) { own = k; break; }
      }
    }
    keep = (own == i);
    owner[t] = own;
  }
  // exclusive scan of keep over t (row-major order)
  const int lane = t & 31, w = t >> 5;
  int incl = keep;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int v = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += v;
  }
  if (lane == 31) warp_tot[w] = incl;
  __syncthreads();
  if (w == 0) {
    int v = warp_tot[lane];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int u = __shfl_up_sync(0xffffffffu, v, o);
      if (lane >= o) v += u;
    }
    warp_tot[lane] = v;  // inclusive totals
  }
  __syncthreads();
  const int excl = incl - keep + (w > 0 ? warp_tot[w - 1] : 0);
  if (t < E) scan[t] = excl;
  const int N = warp_tot[31];
  __syncthreads();

  const size_t rb = (size_t)b * dm.NMAX;
  // padding rows first (disjoint from kept rows)
  for (int n = N + t; n < dm.NMAX; n += blockDim.x) {
    out.tokens[rb + n] = 0;
    out.pos[rb + n] = 0;
    out.parent[rb + n] = -1;
    for (int wd = 0; wd < dm.MW; ++wd) out.mask[(rb + n) * dm.MW + wd] = 0u;
  }
  if (t == 0) out.n[b] = N;
  if (t < E) {
    const int u = scan[owner[t] * C + j];
    out.unpack[((size_t)b * BW + i) * C + j] = u;
    if (keep) {
      out.tokens[rb + excl] = tok[t];
      out.pos[rb + excl] = ctx[b] + j;
      out.parent[rb + excl] = (j == 0) ? -1 : scan[owner[i * C + j - 1] * C + j - 1];
      uint32_t* mr = out.mask + (rb + excl) * dm.MW;
      for (int wd = 0; wd < dm.MW; ++wd) mr[wd] = 0u;
      for (int c = 0; c <= j; ++c) {
        const int a = scan[owner[i * C + c] * C + c];
        mr[a >> 5] |= 1u << (a & 31);
      }
    }
  }
}

cudaError_t launch_pack(const int32_t* beams, const int32_t* root, const int32_t* ctx, const rd_packed& out,
                        const Dims& dm, int B, int no_tree, cudaStream_t st) {
  launch_pdl(pack_kernel, B, 1024, 0, st, beams, root, ctx, out, dm, no_tree);
  return cudaGetLastError();
}

// ---------------------------------------------------------------- accept
// a_i = longest j with beam[i][j'] == llm_argmax[unpack[i][j']] for all j' < j; a = max_i a_i, best = the
// lowest such i; bonus = llm_argmax[unpack[best][a]]; next h = hidden[unpack[best][a]].
// Saves the old context length for the compaction kernel and advances ctx by 1 + a.
// Latency: a candidate's nodes and the LLM's tokens at them are requested ACCEPT_BATCH at a time, so that a walk of five
// tokens costs three round trips to the L2 (nodes, tokens, the hidden row) and not one per node and token.
constexpr int ACCEPT_BATCH = 8;
__global__ void __launch_bounds__(256) accept_kernel(const int32_t* __restrict__ beams, rd_packed pk,
                                                      const int32_t* __restrict__ argmax, const float* __restrict__ hidden,
                                                      const int32_t* __restrict__ seq_off,
                                                      int32_t* ctx, int32_t* root, float* h, rd_accept_out out,
                                                      int32_t* n_accept_ws, int32_t* best_ws, int32_t* ctx_prev, Dims dm,
                                                      int* status) {
  pdl_enter();
  __shared__ int sh_a[8], sh_i[8];
  __shared__ int s_node, s_bonus;
  const int b = blockIdx.x, BW = dm.BW, L = dm.L, C = L + 1;
  const size_t rb = (size_t)b * dm.NMAX;
  int a = -1, bi = 0x7fffffff, node = 0, bonus = 0;   // the best of this thread's candidates, where it ends and the token there
  bool bad = false;
  for (int i = threadIdx.x; i < BW; i += blockDim.x) {
    const int32_t* up = pk.unpack + ((size_t)b * BW + i) * C;
    const int32_t* bm = beams + ((size_t)b * BW + i) * L;
    int ai = 0, an = 0, at = 0;
    bool bad_end = false;
    for (bool go = true; go;) {
      int nd[ACCEPT_BATCH], tk[ACCEPT_BATCH], want[ACCEPT_BATCH];
      const int j0 = ai;
#pragma unroll
      for (int k = 0; k < ACCEPT_BATCH; ++k) {
        nd[k] = j0 + k <= L ? up[j0 + k] : 0;
        want[k] = j0 + k < L ? bm[j0 + k] : 0;
      }
#pragma unroll
      for (int k = 0; k < ACCEPT_BATCH; ++k) tk[k] = argmax[rb + (nd[k] >= 0 && nd[k] < dm.NMAX ? nd[k] : 0)];
#pragma unroll
      for (int k = 0; k < ACCEPT_BATCH; ++k) {
        if (!go) continue;
        an = nd[k]; at = tk[k];
        if (an < 0 || an >= dm.NMAX) {   // (tk is the token at node 0) behind the last token only the winner's node counts
          if (j0 + k < L) atomicOr(status, DEV_ERR_INDEX_RANGE);
          else bad_end = true;
          an = 0; go = false;
        } else if (j0 + k == L || want[k] != at) go = false;
        else ++ai;
      }
    }
    if (ai > a || (ai == a && i < bi)) { a = ai; bi = i; node = an; bonus = at; bad = bad_end; }
  }
  const int mine = bi;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const int oa = __shfl_xor_sync(0xffffffffu, a, o), oi = __shfl_xor_sync(0xffffffffu, bi, o);
    if (oa > a || (oa == a && oi < bi)) { a = oa; bi = oi; }
  }
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  if (lane == 0) { sh_a[w] = a; sh_i[w] = bi; }
  __syncthreads();
  a = sh_a[0]; bi = sh_i[0];
  for (int k = 1; k < (int)(blockDim.x >> 5); ++k)
    if (sh_a[k] > a || (sh_a[k] == a && sh_i[k] < bi)) { a = sh_a[k]; bi = sh_i[k]; }
  if (mine == bi) {   // one thread holds the winner
    s_node = node; s_bonus = bonus;
    if (bad) atomicOr(status, DEV_ERR_INDEX_RANGE);
  }
  __syncthreads();
  if (out.tokens)
    for (int j = threadIdx.x; j < C; j += blockDim.x)
      out.tokens[(size_t)b * C + j] = j < a ? beams[((size_t)b * BW + bi) * L + j] : (j == a ? s_bonus : -1);
  if (threadIdx.x == 0) {
    if (out.n_accept) out.n_accept[b] = a;
    if (out.best) out.best[b] = bi;
    n_accept_ws[b] = a;
    best_ws[b] = bi;
    const int c = ctx[b];
    ctx_prev[b] = c;
    ctx[b] = c + 1 + a;
    root[b] = s_bonus;
  }
  // hidden rows: padded [B][NMAX], or compact (sequence b's first row is seq_off[b])
  const float* src = hidden + (seq_off ? (size_t)seq_off[b] + s_node : rb + s_node) * dm.d;
  for (int i = threadIdx.x; i < dm.d; i += blockDim.x) h[(size_t)b * dm.d + i] = src[i];
}

// Compaction: the accepted path's K/V rows move from provisional slots ctx + unpack[best][j] to
// ctx + j, j = 1..a.  Sources are strictly increasing and never below their destination.  A thread owns one 16-byte
// piece of a head's row for the whole path and moves it in batches, every load of a batch before its stores (a later
// batch's sources lie above this batch's destinations), so the kernel is one or two round trips long; moving element by
// element, row after row, it was up to a hundred of them in series (33B shape, 24 layers, batch 4, paths of up to five:
// two steps 34.5 -> 33.9 ms together with the batched walk above; 13B, one sequence: 19.1 -> 18.7 ms).
constexpr int COMPACT_BATCH = 8;
__global__ void __launch_bounds__(256) compact_kv_kernel(char* __restrict__ kv, int es, rd_packed pk,
                                                          const int32_t* __restrict__ n_accept,
                                                          const int32_t* __restrict__ best,
                                                          const int32_t* __restrict__ ctx_prev, Dims dm, int* status) {
  pdl_enter();
  const int b = blockIdx.x, plane = blockIdx.y;  // plane = layer*2 + {0:K, 1:V}
  const int a = n_accept[b];
  if (a <= 0) return;
  const int c0 = ctx_prev[b], C = dm.L + 1;
  const int32_t* up = pk.unpack + ((size_t)b * dm.BW + best[b]) * C;
  const int per_head = dm.hd * es / 16;                    // 16-byte pieces of a head's row
  const int piece = blockIdx.z * blockDim.x + threadIdx.x;
  const bool active = piece < dm.H * per_head;
  const int hh = active ? piece / per_head : 0, x = active ? piece - hh * per_head : 0;
  const size_t row = (size_t)dm.hd * es;
  char* head = kv + (((size_t)plane * dm.B + b) * dm.H + hh) * (size_t)dm.max_ctx * row + (size_t)x * 16;
  for (int j0 = 1; j0 <= a; j0 += COMPACT_BATCH) {
    int node[COMPACT_BATCH];
    uint4 v[COMPACT_BATCH];
    bool ok = true;
#pragma unroll
    for (int k = 0; k < COMPACT_BATCH; ++k) node[k] = j0 + k <= a ? up[j0 + k] : j0 + k;
#pragma unroll
    for (int k = 0; k < COMPACT_BATCH; ++k) {
      const int j = j0 + k;
      if (j <= a && (node[k] < j || c0 + node[k] >= dm.max_ctx)) ok = false;
      if (!ok || j > a) node[k] = j;                       // not moved: past the path, or behind an index out of range
      if (active && node[k] != j) v[k] = *reinterpret_cast<const uint4*>(head + (size_t)(c0 + node[k]) * row);
    }
#pragma unroll
    for (int k = 0; k < COMPACT_BATCH; ++k)
      if (active && node[k] != j0 + k) *reinterpret_cast<uint4*>(head + (size_t)(c0 + j0 + k) * row) = v[k];
    if (!ok) {
      if (threadIdx.x == 0) atomicOr(status, DEV_ERR_INDEX_RANGE);
      return;
    }
  }
}

// seq_off: hidden holds compact rows (sequence b's first at seq_off[b]); nullptr: padded [B][NMAX].
cudaError_t launch_accept(int dtype, const int32_t* beams, const rd_packed& pk, const int32_t* argmax,
                          const float* hidden, const int32_t* seq_off, void* kcache, int32_t* ctx, int32_t* root, float* h,
                          const rd_accept_out& out, int32_t* n_accept_ws, int32_t* best_ws, int32_t* ctx_prev,
                          const Dims& dm, int B, int* status, cudaStream_t st) {
  launch_pdl(accept_kernel, B, 256, 0, st, beams, pk, argmax, hidden, seq_off, ctx, root, h, out, n_accept_ws, best_ws, ctx_prev, dm,
                                   status);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  const int es = dtype == RD_DTYPE_FP32 ? 4 : 2;
  const int pieces = dm.H * dm.hd * es / 16;   // a head's row is 128 bytes or a multiple of it
  launch_pdl(compact_kv_kernel, dim3(B, dm.n_layers * 2, (pieces + 255) / 256), 256, 0, st, (char*)kcache, es, pk, n_accept_ws, best_ws,
             ctx_prev, dm, status);
  return cudaGetLastError();
}

// ---------------------------------------------------------------- scratch that needs no allocation
// The accept and compaction kernels hand three small per-sequence values to each other (accepted
// length, best candidate, previous context length).  redrafter_accept keeps them in the caller's
// workspace; redrafter_accept_static keeps them here, in memory that is part of the loaded library,
// for callers that cannot allocate.  Every GPU that loads the library holds these 48 KB until exit.
constexpr int ACCEPT_STATIC_MAX_BATCH = 4096;
static __device__ __align__(256) int32_t g_accept_scratch[3 * ACCEPT_STATIC_MAX_BATCH];

int accept_static_max_batch() { return ACCEPT_STATIC_MAX_BATCH; }

// Device address of the static scratch on the CURRENT device.  In host code the array's name is only a
// handle for the runtime, not an address a kernel can use, so the address is asked for once per device
// and remembered.
cudaError_t accept_static_scratch(int32_t** n_accept, int32_t** best, int32_t** ctx_prev) {
  constexpr int MAX_DEVICES = 64;
  static int32_t* base[MAX_DEVICES] = {};
  static std::mutex mu;   // host threads may make their first call on a device at the same time
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= MAX_DEVICES) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lock(mu);
  if (base[dev] == nullptr) {
    void* p = nullptr;
    e = cudaGetSymbolAddress(&p, g_accept_scratch);
    if (e != cudaSuccess) return e;
    base[dev] = static_cast<int32_t*>(p);
  }
  *n_accept = base[dev];
  *best = base[dev] + ACCEPT_STATIC_MAX_BATCH;
  *ctx_prev = base[dev] + 2 * ACCEPT_STATIC_MAX_BATCH;
  return cudaSuccess;
}

}  // namespace rd
