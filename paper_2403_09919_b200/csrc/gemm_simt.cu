// CUDA-core projection y[m][n] = sum_k A[m][k] W[n][k], with the function that follows it applied to the sums.
//
// Used for the fp32 configuration (no tensor-core path for fp32 operands is wanted there: the point of that
// configuration is tight parity) and for bf16 with RD_FLAG_FORCE_SIMT.  Its models are small, so a step is a chain of
// launches of a few microseconds and what bounds it is their number and the hand-over from one to the next: the
// projections take the RMSNorm in front of them and the residual, rotary, SwiGLU or activation behind them along (five
// launches per layer where there were nine) and hand over through the same counters as the tensor-core path (chain.cuh).
//
// One warp owns one weight row -- two, where the function needs both: the halves of a rotary pair, gate and up -- and keeps
// MT running sums, so a weight is read once per MT activation rows; these go through shared memory SIMT_CHUNK columns
// at a time, once for the CTA's eight warps.  The first chunk's weights are requested before the wait.  What a row's
// sums are does not depend on MT or on the other rows, so that verification and autoregressive steps agree bit for bit.
// Measured on the fp32 configuration (d = 256, 2 layers), calls back to back between two events, against one kernel per
// function and grid dependencies: a step of 14 rows 271 -> 177 us, a 64-token prompt 153 -> 88, 16 prompts of 300 tokens 3.19
// -> 2.83 ms (the prompts with what their row tables no longer cost, see prefill_rows_kernel).
#include "rd_internal.cuh"
#include "pdl.cuh"

namespace rd {

constexpr int SIMT_WARPS = 8;
constexpr int SIMT_CHUNK = 512;   // columns of the activation rows in shared memory at a time
// Launches bounded by more rows than this are bound by the CTAs an SM can hold and by the activations' way out of shared
// memory: they request weights as they are needed (64 registers, four CTAs, though 8 to 84 bytes a
// thread spill: with three CTAs and no spills 16 prompts of 300 tokens take 3.77 ms instead of 2.83) and give a warp two
// weight rows always.
// Requesting ahead throughout: 16 prompts of 300 tokens 3.67 ms instead of 2.94; a line at 16 rows instead of 64: steps of
// 17 to 41 rows 2 % slower.
constexpr int SIMT_FEW_ROWS = 64;

template <typename T> struct Vec;
template <> struct Vec<float> {
  static constexpr int N = 4;
  __device__ static __forceinline__ void unpack(const uint4& t, float (&v)[4]) {
    v[0] = __uint_as_float(t.x); v[1] = __uint_as_float(t.y); v[2] = __uint_as_float(t.z); v[3] = __uint_as_float(t.w);
  }
};
template <> struct Vec<__nv_bfloat16> {
  static constexpr int N = 8;
  __device__ static __forceinline__ void unpack(const uint4& t, float (&v)[8]) {
    const uint32_t w[4] = {t.x, t.y, t.z, t.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      v[2 * i] = __uint_as_float(w[i] << 16);
      v[2 * i + 1] = __uint_as_float(w[i] & 0xffff0000u);
    }
  }
};

// grid (ceil(items / 8), ceil(m_max / MT)), block 256.  PRE: a chunk's weights are requested ahead, the first chunk's before
// the wait; otherwise as they are needed, for the sake of more resident CTAs.
template <typename T, int MT, int EPI, bool PRE>
__global__ void __launch_bounds__(SIMT_WARPS * 32, PRE ? 2 : 4) gemm_simt_kernel(SimtOperands p, SimtEpilogue e, Dims dm, ChainSync cs) {
  chain_begin(cs);
  constexpr int VN = Vec<T>::N, NV = SIMT_CHUNK / (32 * VN);   // elements per weight vector, vectors per lane and chunk
  constexpr bool PAIR = EPI == SIMT_ROPE || EPI == SIMT_SWIGLU;   // an item is a pair of weight rows
  constexpr bool TWO = !PRE && !PAIR;                             // ... or the warp takes two items, 8 apart
  constexpr int NR = PAIR || TWO ? 2 : 1;
  __shared__ __align__(16) float sA[MT][SIMT_CHUNK];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int m0 = blockIdx.y * MT;
  const int half = dm.hd >> 1;
  const int item = blockIdx.x * (TWO ? 2 * SIMT_WARPS : SIMT_WARPS) + warp;
  // the item's weight rows: n1 and, with NR == 2, n2 (past the end: the last item's, computed and dropped)
  const int it = min(item, p.items - 1);
  const int n1 = EPI == SIMT_ROPE ? (it / half) * dm.hd + it % half : it;
  const int n2 = EPI == SIMT_ROPE ? n1 + half : EPI == SIMT_SWIGLU ? it + e.F : min(item + SIMT_WARPS, p.items - 1);
  auto load_w = [&](int n, int k) {
    return k < p.K ? __ldg(reinterpret_cast<const uint4*>((const T*)p.W + (size_t)n * p.K + k)) : make_uint4(0u, 0u, 0u, 0u);
  };
  uint4 wv[NR][NV];
  auto load_chunk = [&](int k0) {
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      wv[0][v] = load_w(n1, k0 + (v * 32 + lane) * VN);
      if (NR == 2) wv[NR - 1][v] = load_w(n2, k0 + (v * 32 + lane) * VN);
    }
  };
  if (PRE) load_chunk(0);
  chain_wait_cta(cs);
  const int M = *p.m_total;
  if (m0 >= M) {
    chain_exit(cs);
    return;
  }
  const int rows = min(MT, M - m0);
  float acc[NR][MT];
#pragma unroll
  for (int q = 0; q < NR; ++q)
#pragma unroll
    for (int r = 0; r < MT; ++r) acc[q][r] = 0.f;
  for (int k0 = 0; k0 < p.K; k0 += SIMT_CHUNK) {
    if (k0 > 0) {
      __syncthreads();   // every warp is done with the previous chunk
      if (PRE) load_chunk(k0);
    }
    // the chunk's activations (written by the preceding launches: read past the L1)
    if (p.norm_gain) {
      // fp32 rows of the residual stream, one warp per row: the row fits the chunk (K <= SIMT_CHUNK)
      for (int r = warp; r < MT; r += SIMT_WARPS) {
        float4 x[SIMT_CHUNK / 128];
        float ss = 0.f;
#pragma unroll
        for (int v = 0; v < SIMT_CHUNK / 128; ++v) {
          const int k = (v * 32 + lane) * 4;
          x[v] = r < rows && k < p.K ? __ldcg(reinterpret_cast<const float4*>((const float*)p.A + (size_t)(m0 + r) * p.lda + k))
                                     : make_float4(0.f, 0.f, 0.f, 0.f);
          ss += x[v].x * x[v].x + x[v].y * x[v].y + x[v].z * x[v].z + x[v].w * x[v].w;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
        const float rs = rsqrtf(ss / (float)p.K + p.eps);
        const T* gain = (const T*)p.norm_gain;
#pragma unroll
        for (int v = 0; v < SIMT_CHUNK / 128; ++v) {
          const int k = (v * 32 + lane) * 4;
          float4 y = make_float4(0.f, 0.f, 0.f, 0.f);
          if (k < p.K) {   // rounded to the storage type, as a vector that feeds a projection is
            y.x = to_f<T>(from_f<T>(x[v].x * rs * to_f<T>(gain[k])));
            y.y = to_f<T>(from_f<T>(x[v].y * rs * to_f<T>(gain[k + 1])));
            y.z = to_f<T>(from_f<T>(x[v].z * rs * to_f<T>(gain[k + 2])));
            y.w = to_f<T>(from_f<T>(x[v].w * rs * to_f<T>(gain[k + 3])));
          }
          *reinterpret_cast<float4*>(&sA[r][k]) = y;
        }
      }
    } else {
      constexpr int PER_ROW = SIMT_CHUNK / VN;
#pragma unroll
      for (int i = threadIdx.x; i < MT * PER_ROW; i += SIMT_WARPS * 32) {
        const int r = i / PER_ROW, kk = (i % PER_ROW) * VN;
        uint4 t = make_uint4(0u, 0u, 0u, 0u);
        if (k0 + kk / (32 * VN) * (32 * VN) >= p.K) continue;   // columns that no vector reads
        if (r < rows && k0 + kk < p.K) t = __ldcg(reinterpret_cast<const uint4*>((const T*)p.A + (size_t)(m0 + r) * p.lda + k0 + kk));
        float v[VN];
        Vec<T>::unpack(t, v);
#pragma unroll
        for (int j = 0; j < VN; j += 4) *reinterpret_cast<float4*>(&sA[r][kk + j]) = make_float4(v[j], v[j + 1], v[j + 2], v[j + 3]);
      }
    }
    __syncthreads();
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      if (k0 + v * 32 * VN >= p.K) break;   // nothing but padding from here on
      float w[NR][VN];
#pragma unroll
      for (int q = 0; q < NR; ++q) Vec<T>::unpack(PRE ? wv[q][v] : load_w(q ? n2 : n1, k0 + (v * 32 + lane) * VN), w[q]);
#pragma unroll
      for (int r = 0; r < MT; ++r) {
#pragma unroll
        for (int j = 0; j < VN; j += 4) {
          const float4 a = *reinterpret_cast<const float4*>(&sA[r][(v * 32 + lane) * VN + j]);
#pragma unroll
          for (int q = 0; q < NR; ++q) {
            acc[q][r] = fmaf(a.x, w[q][j], acc[q][r]);
            acc[q][r] = fmaf(a.y, w[q][j + 1], acc[q][r]);
            acc[q][r] = fmaf(a.z, w[q][j + 2], acc[q][r]);
            acc[q][r] = fmaf(a.w, w[q][j + 3], acc[q][r]);
          }
        }
      }
    }
  }
  // Sums over the lanes, MT rows at once: each of the first steps keeps half of the rows and hands the other half to the
  // partner lane, so a row's sum (partners 16, 8, 4, 2, 1 lanes apart, whatever MT is) ends up in lane row * (32 / MT).
  constexpr int LPR = 32 / MT;
  const int r_mine = lane / LPR;
#pragma unroll
  for (int q = 0; q < NR; ++q) {
#pragma unroll
    for (int o = 16, n = MT / 2; o > 0; o >>= 1, n >>= 1) {
      if (n > 0) {
        const bool upper = lane & o;
#pragma unroll
        for (int i = 0; i < MT / 2; ++i)
          if (i < n) {
            const float keep = upper ? acc[q][i + n] : acc[q][i], give = upper ? acc[q][i] : acc[q][i + n];
            acc[q][i] = keep + __shfl_xor_sync(0xffffffffu, give, o);
          }
      } else {
        acc[q][0] += __shfl_xor_sync(0xffffffffu, acc[q][0], o);
      }
    }
  }
  const float y1 = acc[0][0], y2 = acc[NR - 1][0];
  if (item < p.items && lane % LPR == 0 && r_mine < rows) {
    const size_t m = (size_t)(m0 + r_mine);
    auto finish = [&](int n, float y) {
      float* dst = e.out_f + m * e.ld + n;
      if (EPI == SIMT_RAW) {
        *dst = y;
      } else if (EPI == SIMT_RESIDUAL) {   // x += y
        *dst = __ldcg(dst) + y;
      } else {                             // (residual) + SiLU(y + bias), as fp32 and in the storage type
        const float rv = e.resid ? __ldcg(e.resid + m * e.ld_resid + n) : 0.f;
        const float z = rv + silu_f(y + to_f<T>(((const T*)e.bias)[n]));
        *dst = z;
        ((T*)e.out_t)[m * e.ld + n] = from_f<T>(z);
      }
    };
    if (!PAIR) {
      finish(n1, y1);
      if (TWO && item + SIMT_WARPS < p.items) finish(n2, y2);
    } else if (EPI == SIMT_SWIGLU) {
      ((T*)e.out_t)[m * e.F + item] = from_f<T>(silu_f(y1) * y2);
    } else {                             // rotary embedding of Q and K (pairs i, i + hd/2); K and V go to the row's cache slot
      const int part = n1 / dm.d, o = n1 - part * dm.d, h = o / dm.hd, x = o - h * dm.hd;
      const float2 c = part < 2 ? e.table[m * half + x] : make_float2(1.f, 0.f);
      const float a = part < 2 ? y1 * c.x - y2 * c.y : y1, b = part < 2 ? y2 * c.x + y1 * c.y : y2;
      if (part == 0) {                   // the attention kernel reads the rotated Q as fp32
        e.out_f[m * e.ld + n1] = a;
        e.out_f[m * e.ld + n2] = b;
      } else {
        const int slot = e.slot[m];
        if (slot >= 0 && slot < dm.max_ctx) {
          T* dst = (T*)(part == 1 ? e.kcache : e.vcache) + (((size_t)e.seq[m] * dm.H + h) * dm.max_ctx + slot) * dm.hd + x;
          dst[0] = from_f<T>(a);
          dst[half] = from_f<T>(b);
        } else if (o == 0) {
          atomicOr(e.status, DEV_ERR_CAPACITY);
        }
      }
    }
  }
  chain_exit(cs);
}

// K a multiple of 4 (fp32) or 8 (bf16), rows of A and W 16-byte aligned.
cudaError_t launch_gemm_simt(int dtype, int epi, const SimtOperands& p, const SimtEpilogue& e, const Dims& dm, int m_max, Chain* chain,
                             cudaStream_t st) {
  if (p.norm_gain && p.K > SIMT_CHUNK) return cudaErrorInvalidValue;
  if (m_max <= 0) return cudaSuccess;
  const int mt = m_max <= 2 ? 2 : m_max <= 4 ? 4 : 8;
  const int per_cta = m_max <= SIMT_FEW_ROWS || epi == SIMT_ROPE || epi == SIMT_SWIGLU ? SIMT_WARPS : 2 * SIMT_WARPS;
  const dim3 grid((p.items + per_cta - 1) / per_cta, (m_max + mt - 1) / mt);
  // the first launch of a chain starts after everything before it has completed (see launch_ordered)
  const bool first = chain && chain->enabled && chain->prev_ptr == nullptr;
  const ChainSync cs = chain ? chain->link(grid.x * grid.y, true) : ChainSync{nullptr, 0u, nullptr, nullptr, nullptr};
  auto go = [&](auto kernel) {
    if (first) launch_ordered(kernel, grid, SIMT_WARPS * 32, 0, st, p, e, dm, cs);
    else launch_pdl(kernel, grid, SIMT_WARPS * 32, 0, st, p, e, dm, cs);
  };
#define RD_SIMT_MT(T, EPI)                                                    \
  if (mt == 2) go(gemm_simt_kernel<T, 2, EPI, true>);                           \
  else if (mt == 4) go(gemm_simt_kernel<T, 4, EPI, true>);                      \
  else if (m_max <= SIMT_FEW_ROWS) go(gemm_simt_kernel<T, 8, EPI, true>);       \
  else go(gemm_simt_kernel<T, 8, EPI, false>)
#define RD_SIMT(EPI) \
  if (dtype == RD_DTYPE_FP32) { RD_SIMT_MT(float, EPI); } else { RD_SIMT_MT(__nv_bfloat16, EPI); }
  switch (epi) {
    case SIMT_RAW: RD_SIMT(SIMT_RAW); break;
    case SIMT_RESIDUAL: RD_SIMT(SIMT_RESIDUAL); break;
    case SIMT_SWIGLU: RD_SIMT(SIMT_SWIGLU); break;
    case SIMT_ACT: RD_SIMT(SIMT_ACT); break;
    case SIMT_ROPE: RD_SIMT(SIMT_ROPE); break;
    default: return cudaErrorInvalidValue;
  }
#undef RD_SIMT
#undef RD_SIMT_MT
  return cudaGetLastError();
}

int simt_norm_max_k() { return SIMT_CHUNK; }

GemmOut simt_out(float* raw, int ld) {
  GemmOut g{};
  g.raw = raw; g.partial = nullptr; g.ld = ld; g.nkb = 1; g.n_tiles = 1; g.mt = 1; g.grid = 1; g.m_tiles_max = 1;
  return g;
}

}  // namespace rd
