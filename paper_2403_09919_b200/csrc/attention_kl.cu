// Attention with the keys on the tensor-memory lanes, for passes of a few dozen rows per sequence (Sections 3.3, 3.4):
// head dimension 128, bf16 operands, fp32 accumulation in tensor memory.
//
// The 128-row kernel (attention_t5.cu) gives every query row a lane, so a decode step's 20 to 90 rows leave half of each
// matrix instruction, of the softmax and of the tensor memory to padding, and its set-up and tail are those of a full tile.
// Here both products are transposed, so that the rows are the N of the instruction, which comes in steps of 16:
//   S^T = K Q^T      A = chunk of 128 keys straight from the cache (K-major), B = the tile's rows (K-major, converted once
//                    from the fp32 rows of the rotary kernel), D: lane = key, column = row;
//   softmax          sixteen warps, four per lane quarter with a quarter of the columns each: a thread has one key and those
//                    rows.  A row's reference maximum is moved only when a score exceeds it by 2^32 (one vote per chunk): the
//                    maximum over the keys lies across the lanes, and finding it for every chunk would cost more than the
//                    exponentials.  With the maximum as reference the largest weight would be exactly one; here it is rounded
//                    like the rest, which alone would make the output less exact than the other kernels' (2.3e-3 against
//                    1.9 to 2.1e-3, scores of deviation 1.5).  So every weight goes in two parts, itself in bf16 and
//                    what that rounding left, again in bf16 (to 2^-17 together; 1.65e-3, the rounding of the output);
//   O^T += V^T P^T   A = V chunk as it lies in the cache ([key][dim], MN-major), B = the weights and behind them their
//                    remainders as further columns, written to shared memory as [16 rows][key] lines of 32 bytes (MN-major,
//                    32-byte swizzle), D: lane = dimension, column = row, and again for the remainders; the output adds the two.
//
// A tile is (head, sequence, up to 96 of its rows); a sequence with more rows is cut into equal tiles.  One CTA per SM takes
// its tiles one after the other (longest sequences first): K and V come through two rings of 16 KB slots (half of a chunk's
// dimensions of K, half of its keys of V) that the producer keeps filled across the tiles' ends, and the next tile's first
// scores are formed while the one before is written out.
// Roles: warp 0 = TMA producer, warps 1 and 2 = MMA issuers of the scores and of the output (the whole warp runs the loop, an
// elected lane issues), warp 3 lays out the CTA's tiles and clears the values behind their last keys, warps 4..19 = softmax and
// output.  Every wait is bounded (one second), as in attention_t5.cu; a warp that gives up still takes part in the named barriers
// until all of its part have seen it.
//
// What bounds it: the copies where every SM has tiles (7B, 16 sequences of 1024 tokens and 52 rows: 69 us a launch for 309 MB, 4.5 TB/s
// or 0.69 of the measured copy rate, tensor pipe 18 %; without the remainders 16 of 256 to 2048 tokens took 70 us, 95 in the 64- and
// 128-row kernels), else a chunk's chain of hand-overs
// (scores 0.25 us, weights 0.35 to 0.6 us by columns, the product; 0.8 to 1.5 us a chunk) and, in the first, the code's fetch.
// The remainders take 0.3 % of a 7B step (30 rows, 512 tokens), 0.4 to 0.9 of the 7B calls, 1.5 of the batch-16 step and 2 of
// 4 x 4096 tokens at 33B, most of it for forming and storing them (doubled columns alone: 0.3 %).  One buffer of weights
// instead of two for tiles of 64 rows and more, which leaves the rings half as much again: 7B batch 16 33.4 -> 33.9 ms, 33B 32.2 -> 32.6.
// Tried before: two smaller CTAs per SM (half the copies under way each: 2 to 5 % behind), the loop run once over nothing before
// the wait (no gain), a common ring for K and V, copies that stay in the L2 (16 sequences 444 -> 450 us a layer, 4 single rows
// 120 -> 124).  96 registers (640 threads), 68 bytes of them spilled in the widest tiles.
#include "pdl.cuh"
#include "rd_internal.cuh"
#include "tcgen05.cuh"

namespace rd {

namespace {

constexpr int KL_ROWS = 96;            // most rows of a tile
constexpr int KL_KEYS = 128;           // keys per chunk (TMEM lanes)
constexpr int KL_HD = 128;
constexpr int KL_PARTS = 4;            // parts of a tile's columns, four softmax warps each
constexpr int KL_SOFT = 128 * KL_PARTS;
constexpr int KL_THREADS = 128 + KL_SOFT;
constexpr uint32_t KL_SLOT = 16384;    // ring slot: 64 dimensions of 128 keys (K), 64 keys of 128 dimensions (V)
constexpr int KL_MAX_SLOTS = 12;
constexpr uint32_t KL_TMEM = 512;      // columns: two score buffers of 128, the output from 256 (twice a tile's columns)
constexpr int KL_MAX_TILES = 32;       // tiles of a CTA
constexpr uint32_t KL_SMEM = 227 * 1024;
constexpr float KL_SLACK = 32.0f;      // log2 by which a score may exceed its row's reference (values beyond 2^80 could overflow the sums)
constexpr float KL_LOW = 64.0f;        // ... and its largest may stay below it

// K^T-major operands: see tcgen05.cuh for the K-major one.  MN-major, 128-byte swizzle: 64 elements per line, 8 keys 1024 bytes
// apart, the next 64 elements `lbo` bytes further.
__device__ __forceinline__ uint64_t desc_mn128(uint32_t addr, uint32_t lbo) {
  return (uint64_t)((addr & 0x3FFFFu) >> 4) | ((uint64_t)(lbo >> 4) << 16) | (64ull << 32) | (1ull << 46) | (2ull << 61);
}
// MN-major, 32-byte swizzle: 16 elements per line, 8 keys 256 bytes apart, the next 16 elements `lbo` bytes further.
__device__ __forceinline__ uint64_t desc_mn32(uint32_t addr, uint32_t lbo) {
  return (uint64_t)((addr & 0x3FFFFu) >> 4) | ((uint64_t)(lbo >> 4) << 16) | (16ull << 32) | (1ull << 46) | (6ull << 61);
}
__device__ __forceinline__ void tmem_ld8_nowait(uint32_t taddr, float* r) {
  uint32_t u[8];
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(u[0]), "=r"(u[1]), "=r"(u[2]), "=r"(u[3]), "=r"(u[4]), "=r"(u[5]), "=r"(u[6]), "=r"(u[7])
               : "r"(taddr));
#pragma unroll
  for (int j = 0; j < 8; ++j) r[j] = __uint_as_float(u[j]);
}
// Keys and values are read once a pass and leave the L2 first: what the launches hand to each other stays in it.
__device__ __forceinline__ uint64_t evict_first() {
  uint64_t pol;
  asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
  return pol;
}
__device__ __forceinline__ void load_box_2d(uint32_t dst, const CUtensorMap* map, uint32_t bar, int x, int y, uint64_t pol) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, {%3, %4}], [%2], %5;" ::"r"(dst),
      "l"(map), "r"(bar), "r"(x), "r"(y), "l"(pol)
      : "memory");
}
__device__ __forceinline__ void load_box_3d(uint32_t dst, const CUtensorMap* map, uint32_t bar, int x, int y, int z, uint64_t pol) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, {%3, %4, %5}], [%2], %6;" ::"r"(dst),
      "l"(map), "r"(bar), "r"(x), "r"(y), "r"(z), "l"(pol)
      : "memory");
}
__device__ __forceinline__ void tmem_ld4_nowait(uint32_t taddr, float* r) {
  uint32_t u[4];
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(u[0]), "=r"(u[1]), "=r"(u[2]), "=r"(u[3]) : "r"(taddr));
#pragma unroll
  for (int j = 0; j < 4; ++j) r[j] = __uint_as_float(u[j]);
}
__device__ __forceinline__ void tmem_st4(uint32_t taddr, const float* r) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1, %2, %3, %4};" ::"r"(taddr), "r"(__float_as_uint(r[0])),
               "r"(__float_as_uint(r[1])), "r"(__float_as_uint(r[2])), "r"(__float_as_uint(r[3]))
               : "memory");
}
// Barrier over `n` threads that also tells whether any of them brought `v`.
template <int n>
__device__ __forceinline__ bool bar_any(int id, bool v) {
  uint32_t r;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t"
      "setp.ne.u32 p, %2, 0;\n\t"
      "barrier.cta.red.or.pred q, %1, %3, p;\n\t"
      "selp.u32 %0, 1, 0, q;\n\t}"
      : "=r"(r)
      : "r"(id), "r"((uint32_t)v), "n"(n)
      : "memory");
  return r != 0;
}
template <int n>
__device__ __forceinline__ void bar_sync(int id) { asm volatile("barrier.cta.sync %0, %1;" ::"r"(id), "n"(n) : "memory"); }
// N values per lane (4 or 8) reduced over the lanes: afterwards lane i (and i + N, ...) holds the result of value i mod N.  A
// butterfly that halves the values a lane holds: nine shuffles for eight, where a warp-wide reduction each took five times as
// long (redux.sync of floats).
template <int N, class Op>
__device__ __forceinline__ float lanes_reduce(const float* v, int lane, Op op) {
  float a[4], b[2];
  const bool u4 = lane & 4, u2 = lane & 2, u1 = lane & 1;
#pragma unroll
  for (int i = 0; i < 4; ++i) a[i] = N == 4 ? v[i] : op(u4 ? v[(4 + i) & (N - 1)] : v[i], __shfl_xor_sync(0xffffffffu, u4 ? v[i] : v[(4 + i) & (N - 1)], 4));
#pragma unroll
  for (int i = 0; i < 2; ++i) b[i] = op(u2 ? a[2 + i] : a[i], __shfl_xor_sync(0xffffffffu, u2 ? a[i] : a[2 + i], 2));
  float r = op(u1 ? b[1] : b[0], __shfl_xor_sync(0xffffffffu, u1 ? b[0] : b[1], 1));
  if (N == 4) r = op(r, __shfl_xor_sync(0xffffffffu, r, 4));
  r = op(r, __shfl_xor_sync(0xffffffffu, r, 8));
  return op(r, __shfl_xor_sync(0xffffffffu, r, 16));
}
// COLS columns over the lanes, one result per column to dst.
template <int COLS, class Op>
__device__ __forceinline__ void columns_reduce(const float* v, int lane, float* dst, Op op) {
#pragma unroll
  for (int i = 0; i + 8 <= COLS; i += 8) {
    const float r = lanes_reduce<8>(v + i, lane, op);
    if (lane < 8) dst[i + lane] = r;
  }
  if (COLS % 8) {
    const float r = lanes_reduce<4>(v + COLS / 8 * 8, lane, op);
    if (lane < 4) dst[COLS / 8 * 8 + lane] = r;
  }
}
__device__ __forceinline__ void mul2(float& x, float& y, float f) {   // both by f, one instruction
  asm("{\n\t.reg .b64 a, b;\n\tmov.b64 a, {%0, %1};\n\tmov.b64 b, {%2, %2};\n\tmul.rn.f32x2 a, a, b;\n\tmov.b64 {%0, %1}, a;\n\t}"
      : "+f"(x), "+f"(y) : "f"(f));
}
__device__ __forceinline__ void fma2(float& x, float& y, float f, float u, float v) {   // both times f, plus u and v
  asm("{\n\t.reg .b64 a, b, c;\n\tmov.b64 a, {%0, %1};\n\tmov.b64 b, {%2, %2};\n\tmov.b64 c, {%3, %4};\n\tfma.rn.f32x2 a, a, b, c;\n\tmov.b64 {%0, %1}, a;\n\t}"
      : "+f"(x), "+f"(y) : "f"(f), "f"(u), "f"(v));
}
__device__ __forceinline__ void add2(float& x, float& y, float u, float v) {
  asm("{\n\t.reg .b64 a, b;\n\tmov.b64 a, {%0, %1};\n\tmov.b64 b, {%2, %3};\n\tadd.rn.f32x2 a, a, b;\n\tmov.b64 {%0, %1}, a;\n\t}"
      : "+f"(x), "+f"(y) : "f"(u), "f"(v));
}
// The issuing instructions under a predicate, so that a pass of the loop with nothing to issue fetches its code.
__device__ __forceinline__ void umma_if(bool on, uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "setp.ne.b32 q, %5, 0;\n\t"
      "@q tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(acc), "r"((uint32_t)on)
      : "memory");
}
__device__ __forceinline__ void commit_if(bool on, uint32_t bar) {
  asm volatile(
      "{\n\t.reg .pred q;\n\t"
      "setp.ne.b32 q, %1, 0;\n\t"
      "@q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t}" ::"r"(bar),
      "r"((uint32_t)on)
      : "memory");
}

struct KlParams {
  const float* qkv;            // [M][3d] fp32, Q rotated in place by the rotary kernel
  __nv_bfloat16* out;          // [M][d]
  RowTables rt;
  const int32_t* seq_off;
  const int32_t* seq_order;    // the launch's sequences, longest key extent first, or nullptr (index order)
  const uint32_t* mask_t;      // the tree mask with rows and columns exchanged: [B][NMAX][MW], bit r of node j's words: row r attends j
  Dims dm;
  int n_seq, n_tiles;          // tiles of the launch: heads x sequences x row tiles (bound)
  int32_t* status;
  ChainSync cs;
};

struct KlTile {
  int b, head, row0, rel_row0, nrows;      // sequence, head, first row (of the pass, of the sequence), rows
  int seq_rows, tree_base, kext, nc_min;   // nc_min: every row attends the keys below it
  int old_keys;                            // keys below this are older than the pass
  int pad[2];
};
// Shared memory in front of the operands.
struct KlShared {
  unsigned long long bars[48];
  uint32_t tmem;
  volatile int abort_flag;
  int n_tiles, rows_max;
  KlTile tiles[KL_MAX_TILES];
  alignas(16) float nref[KL_ROWS];   // minus the reference maximum of every row (base 2, scaled)
  alignas(16) float corr[KL_ROWS];   // factor by which a moved reference scales what was summed before; at the end 1 / sum
  float red[4][KL_ROWS];          // per lane quarter: row maxima of a chunk; at the end the rows' sums
  uint32_t vis[1];                // [chunks from the first that some row does not attend whole][part][key]: rows that attend the key
};
// S_* to PV_*: by chunk parity
enum { KB_FULL = 0, KB_EMPTY = KL_MAX_SLOTS, KB_Q = 2 * KL_MAX_SLOTS, KB_S_FULL, KB_S_EMPTY = KB_S_FULL + 2, KB_P_FULL = KB_S_EMPTY + 2,
       KB_PV_DONE = KB_P_FULL + 2, KB_TAIL = KB_PV_DONE + 2, KB_COUNT = KB_TAIL + KL_MAX_SLOTS };
static_assert(KB_COUNT <= 48, "barriers");

// Chunks of a tile that some row may not attend whole: as many as the tree (or a causal tile) touches.
__host__ __device__ constexpr int kl_vis_chunks(int nmax) { return ((nmax > KL_ROWS ? nmax : KL_ROWS) + KL_KEYS - 1) / KL_KEYS + 1; }
__host__ __device__ constexpr uint32_t kl_front_bytes(int nmax) {
  return ((uint32_t)sizeof(KlShared) + (uint32_t)(kl_vis_chunks(nmax) * KL_PARTS * KL_KEYS) * 4u + 1023u) & ~1023u;
}

// What the softmax warps share.
struct KlCtx {
  KlShared* sm;
  uint32_t bar0, tmem;
  uint8_t *sQ, *sP;
  bool early;
};

// The softmax and output warps: every tile of the CTA in tiles of N = 4 COLS columns.
template <int COLS>
__device__ __forceinline__ void kl_softmax(const KlParams& p, const KlCtx& t, const int n_tiles) {
  constexpr int N = KL_PARTS * COLS;
  constexpr uint32_t WEIGHT_BYTES = 2 * N * 256u;   // a chunk's weights and their remainders
  KlShared* sm = t.sm;
  const int st = (int)threadIdx.x - 128, tip = st & 127;   // thread of the softmax warps, of this part
  const int lane = threadIdx.x & 31, q4 = (st >> 5) & 3, part = st >> 7;
  const int key_lane = q4 * 32 + lane;
  const int col0 = part * COLS, MW = p.dm.MW;
  const int part_bar = 1 + part;
  constexpr int ALL_BAR = 1 + KL_PARTS;
  const float scale2 = rsqrtf((float)KL_HD) * 1.4426950408889634f;   // 1/sqrt(hd) * log2(e)
  auto bar = [&](int i) { return t.bar0 + 8u * i; };
  auto wait_all = [&](uint32_t b, uint32_t parity) {
    return __all_sync(0xffffffffu, mbar_wait(b, parity, &sm->abort_flag, p.status)) != 0;
  };
  const uint32_t tm = t.tmem + ((uint32_t)(q4 * 32) << 16) + (uint32_t)col0;
  const uint32_t o_addr = tm + 256u;
  uint8_t* const p_line = t.sP + key_lane * 32;
  const uint32_t p_swz = (uint32_t)((key_lane >> 2) & 1);
  uint32_t* const vis0 = sm->vis + part * KL_KEYS + key_lane;
  // For every key of the chunks that some row of a tile does not attend whole, the rows that do (a thread reads the words that
  // it wrote itself).  A row attends the keys below its extent -- under the tree mask the context, else one key more than the row
  // before it -- and the nodes of its mask row.  Columns past the rows hold zeros and are never read.
  auto lay_out = [&](const KlTile& tl) {
    const int mc0 = tl.nc_min / KL_KEYS;
    for (int c = mc0; c * KL_KEYS < tl.kext; ++c) {
      const int key = c * KL_KEYS + key_lane, j = key - tl.tree_base;
      uint32_t w;
      if (p.mask_t) {
        w = j < 0 ? 0xffffffffu : 0u;
        if (j >= 0 && j < tl.seq_rows) {
          const uint32_t* bits = p.mask_t + ((size_t)tl.b * p.dm.NMAX + j) * MW;
          const int r = tl.rel_row0 + col0, wd = r >> 5;
          w = __funnelshift_r(wd < MW ? bits[wd] : 0u, wd + 1 < MW ? bits[wd + 1] : 0u, r & 31);
        }
      } else {
        const int from = j + 1 - col0;   // first column that attends the key
        w = from <= 0 ? 0xffffffffu : from < 32 ? 0xffffffffu << from : 0u;
      }
      const int past = tl.nrows - col0;   // columns from here on
      vis0[(c - mc0) * KL_PARTS * KL_KEYS] = w | (past <= 0 ? 0xffffffffu : past < 32 ? 0xffffffffu << past : 0u);
    }
    if (tip < COLS) sm->nref[col0 + tip] = 0.f;
  };
  lay_out(sm->tiles[0]);

  int j0 = 0;   // chunks of the tiles before this one
  for (int k = -1; k < n_tiles; ++k) {   // (-1: only the first tile's rows are fetched)
    const KlTile& tl = sm->tiles[max(k, 0)];
    const int n_chunks = k < 0 ? 0 : (tl.kext + KL_KEYS - 1) / KL_KEYS, mc0 = tl.nc_min / KL_KEYS;
    float l[COLS];
#pragma unroll
    for (int i = 0; i < COLS; ++i) l[i] = 0.f;
    // The rows' references start at zero, which serves any row with a score of at least -KL_LOW (one key whose scores all are
    // settles it for its part), and move when a score exceeds one by KL_SLACK.  A row that attends no key of the first chunks
    // (`none`, of the row that this thread keeps the reference of) takes its reference from the first that it does attend: until
    // then its part looks at every chunk's maxima (`hollow`).
    bool ok = true, moved = false, none = true, hollow = false;
    for (int c = 0; c < n_chunks; ++c) {
      const int j = j0 + c;
      const uint32_t ph = (uint32_t)((j >> 1) & 1);
      const bool masked = c >= mc0;
      const uint32_t seen = masked ? vis0[(c - mc0) * KL_PARTS * KL_KEYS] : 0xffffffffu;
      if (ok) ok = wait_all(bar(KB_S_FULL + (j & 1)), ph);
      tc_fence_after();
      float sc[COLS];
      bool far = true;   // a score too large for its row's reference (or a wait that gave up)
      if (ok) {
        const uint32_t s_addr = tm + (uint32_t)(j & 1) * 128u;
#pragma unroll
        for (int g = 0; g + 8 <= COLS; g += 8) tmem_ld8_nowait(s_addr + g, sc + g);
        if (COLS % 8) tmem_ld4_nowait(s_addr + COLS / 8 * 8, sc + COLS / 8 * 8);
        tmem_ld_wait();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(bar(KB_S_EMPTY + (j & 1)));
        if (masked) {   // by selection: masked scores may be anything
#pragma unroll
          for (int i = 0; i < COLS; ++i) sc[i] = ((seen >> i) & 1u) ? sc[i] : -INFINITY;
        }
        // to base 2: 1/sqrt(hd) * log2(e)
        if (!moved) {
#pragma unroll
          for (int i = 0; i < COLS; i += 2) mul2(sc[i], sc[i + 1], scale2);
        } else {
#pragma unroll
          for (int i = 0; i < COLS; i += 4) {
            const float4 n = *reinterpret_cast<const float4*>(&sm->nref[col0 + i]);
            fma2(sc[i], sc[i + 1], scale2, n.x, n.y);
            fma2(sc[i + 2], sc[i + 3], scale2, n.z, n.w);
          }
        }
        float mx = sc[0];
#pragma unroll
        for (int i = 1; i < COLS; ++i) mx = fmaxf(mx, sc[i]);
        far = mx > KL_SLACK;
      }
      bool move = bar_any<128>(part_bar, far) || hollow;
      if (c == 0) {
        float low = sc[0];
#pragma unroll
        for (int i = 1; i < COLS; ++i) low = fminf(low, sc[i]);
        move = !bar_any<128>(part_bar, ok && low >= -KL_LOW) || move;
        none = move;
      }
      if (move) {
        // references move: the maximum of every column over the chunk's keys
        if (bar_any<128>(part_bar, !ok)) { ok = false; break; }
        columns_reduce<COLS>(sc, lane, &sm->red[q4][col0], [](float x, float y) { return fmaxf(x, y); });
        bar_sync<128>(part_bar);
        if (tip < COLS) {
          const int r = col0 + tip;
          // by how much row r's reference rises (at its first keys it may also fall); a row without keys so far keeps its own
          const float m = fmaxf(fmaxf(sm->red[0][r], sm->red[1][r]), fmaxf(sm->red[2][r], sm->red[3][r]));
          const float up = m == -INFINITY ? 0.f : none ? m : fmaxf(m, 0.f);
          sm->corr[r] = -up;
          sm->nref[r] -= up;
          none = none && m == -INFINITY;
        }
        moved = true;
        hollow = bar_any<128>(part_bar, tip < COLS && none);
#pragma unroll
        for (int i = 0; i < COLS; ++i) {
          const float down = sm->corr[col0 + i];
          sc[i] += down;
          l[i] *= fast_exp2(fminf(down, 0.f));   // (where the reference falls, its factor has no bound, and the sums are zero)
        }
        if (c > 0) {
          // O is complete through the chunk before this one and waits for this one's weights
          ok = wait_all(bar(KB_PV_DONE + ((j - 1) & 1)), (uint32_t)(((j - 1) >> 1) & 1));
          if (ok) {
            tc_fence_after();
#pragma unroll 1
            for (int i = 0; i < COLS; i += 4) {
              float o[4], r[4];
              tmem_ld4_nowait(o_addr + i, o);
              tmem_ld4_nowait(o_addr + N + i, r);
              tmem_ld_wait();
#pragma unroll
              for (int n = 0; n < 4; ++n) {
                const float f = fast_exp2(fminf(sm->corr[col0 + i + n], 0.f));
                o[n] *= f; r[n] *= f;
              }
              tmem_st4(o_addr + i, o);
              tmem_st4(o_addr + N + i, r);
            }
            tmem_st_wait();
          }
        }
      }
      // this chunk's buffer of weights is free once the product of the chunk before last has read it
      if (ok && j >= 2) ok = wait_all(bar(KB_PV_DONE + (j & 1)), ph ^ 1u);
      if (ok) {
        // four weights at a time, and what their rounding left of them (exact in fp32) rounded again
        uint8_t* const line = p_line + (uint32_t)(j & 1) * WEIGHT_BYTES;
        uint32_t hi[4], lo[4];
#pragma unroll
        for (int i = 0; i < COLS; i += 4) {
          const int col = col0 + i, at = COLS % 8 ? 0 : (i & 4) / 2;
#pragma unroll
          for (int n = 0; n < 4; n += 2) {
            const float x = fast_exp2(sc[i + n]), y = fast_exp2(sc[i + n + 1]);   // 2^(-inf) = 0
            add2(l[i + n], l[i + n + 1], x, y);
            const uint32_t h = pack_bf16(x, y);
            float rx = __uint_as_float(h << 16), ry = __uint_as_float(h & 0xffff0000u);
            fma2(rx, ry, -1.f, x, y);
            hi[at + n / 2] = h; lo[at + n / 2] = pack_bf16(rx, ry);
          }
          uint8_t* const to = line + (col >> 4) * (KL_KEYS * 32) + ((((uint32_t)(col >> 3) & 1u) ^ p_swz) << 4);
          if (COLS % 8) {
            *reinterpret_cast<uint2*>(to + (col & 4) * 2) = make_uint2(hi[0], hi[1]);
            *reinterpret_cast<uint2*>(to + N * 256 + (col & 4) * 2) = make_uint2(lo[0], lo[1]);
          } else if (i & 4) {
            *reinterpret_cast<uint4*>(to) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
            *reinterpret_cast<uint4*>(to + N * 256) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
          }
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(bar(KB_P_FULL + (j & 1)));
      }
    }
    if (bar_any<KL_SOFT>(ALL_BAR, !ok)) return;   // also: everybody is through with this tile's tables

    // ---- the next tile's rows: requested here, converted once this tile's sums are formed (its scores all are, so that their
    // operand's buffer is free)
    const bool more = k + 1 < n_tiles;
    const KlTile& nx = sm->tiles[more ? k + 1 : 0];
    const int cq = st & 15;
    constexpr int STEP = KL_SOFT / 16, PASSES = (N + STEP - 1) / STEP;
    float4 a[PASSES][2];
    if (more) {
      if (k < 0) {
        if (st == 0 && t.early) chain_wait_thread(p.cs);
        bar_sync<KL_SOFT>(ALL_BAR);
      }
#pragma unroll
      for (int i = 0; i < PASSES; ++i) {
        const int r = min((st >> 4) + i * STEP, nx.nrows - 1);
        const float* q = p.qkv + (size_t)(nx.row0 + r) * 3 * p.dm.d + nx.head * KL_HD + cq * 8;
        a[i][0] = __ldcg(reinterpret_cast<const float4*>(q)); a[i][1] = __ldcg(reinterpret_cast<const float4*>(q + 4));
      }
    }
    // ---- this tile's sums over the keys of all lanes
    if (k >= 0) {
      columns_reduce<COLS>(l, lane, &sm->red[q4][col0], [](float x, float y) { return x + y; });
      bar_sync<128>(part_bar);
      if (tip < COLS) {
        const int r = col0 + tip;
        const float sum = (sm->red[0][r] + sm->red[1][r]) + (sm->red[2][r] + sm->red[3][r]);
        sm->corr[r] = sum == 0.f ? 0.f : 1.f / sum;   // a row without keys is zero, one of NaN stays so
      }
    }
    if (more) {   // Q -> bf16, K-major swizzled: 16-byte chunk i of row r lands at chunk i ^ (r & 7) of its 128-byte line
      uint8_t* q_dst = t.sQ + (size_t)(cq >> 3) * N * 128;
#pragma unroll
      for (int i = 0; i < PASSES; ++i) {
        const int r = (st >> 4) + i * STEP;
        const uint4 v = make_uint4(pack_bf16(a[i][0].x, a[i][0].y), pack_bf16(a[i][0].z, a[i][0].w), pack_bf16(a[i][1].x, a[i][1].y),
                                   pack_bf16(a[i][1].z, a[i][1].w));
        if (N % STEP == 0 || r < N)
          *reinterpret_cast<uint4*>(q_dst + r * 128 + (((cq & 7) ^ (r & 7)) << 4)) = r < nx.nrows ? v : make_uint4(0u, 0u, 0u, 0u);
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      __syncwarp();
      if (lane == 0) mbar_arrive(bar(KB_Q));
    }
    bar_sync<KL_SOFT>(ALL_BAR);
    if (more && k >= 0) lay_out(nx);
    if (k < 0) continue;

    // ---- output: lane = dimension, column = row; neighbouring lanes swap so that each stores two dimensions of one row
    j0 += n_chunks;
    if (wait_all(bar(KB_PV_DONE + ((j0 - 1) & 1)), (uint32_t)(((j0 - 1) >> 1) & 1))) {
      tc_fence_after();
      const int odd = lane & 1, nrows = tl.nrows;
      __nv_bfloat16* o = p.out + (size_t)(tl.row0 + col0 + odd) * p.dm.d + tl.head * KL_HD + q4 * 32 + (lane & ~1);
      float ov[4], rv[4];
      tmem_ld4_nowait(o_addr, ov);
      tmem_ld4_nowait(o_addr + N, rv);
#pragma unroll 1
      for (int i = 0; i < COLS; i += 4) {
        float v[4];
        tmem_ld_wait();
        if (col0 + i >= nrows) break;   // the same for the whole warp
#pragma unroll
        for (int n = 0; n < 4; ++n) v[n] = ov[n] + rv[n];
        if (i + 4 < COLS) {
          tmem_ld4_nowait(o_addr + i + 4, ov);
          tmem_ld4_nowait(o_addr + N + i + 4, rv);
        }
#pragma unroll
        for (int n = 0; n < 4; n += 2) {
          const float2 inv = *reinterpret_cast<const float2*>(&sm->corr[col0 + i + n]);
          const float x = v[n] * inv.x, y = v[n + 1] * inv.y;
          const float other = __shfl_xor_sync(0xffffffffu, odd ? x : y, 1);
          if (col0 + i + n + odd < nrows) *reinterpret_cast<uint32_t*>(o + (size_t)(i + n) * p.dm.d) = odd ? pack_bf16(other, y) : pack_bf16(x, other);
        }
      }
      tc_fence_before();
    }
    bar_sync<128>(part_bar);   // the part is done with the sums, and its references of the next tile are laid out
  }
}

__global__ void __launch_bounds__(KL_THREADS, 1)
    attention_kl_kernel(const __grid_constant__ CUtensorMap map_k, const __grid_constant__ CUtensorMap map_v, const KlParams p) {
  extern __shared__ uint8_t smem_raw[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  uint8_t* gen = smem_raw + (base - raw);
  KlShared* sm = reinterpret_cast<KlShared*>(gen);
  const uint32_t bar0 = base;   // KlShared starts with the barriers
  auto bar = [&](int i) { return bar0 + 8u * i; };
  const Dims& dm = p.dm;

  // Tensor memory first, before the dependents may start.
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&sm->tmem)), "r"(KL_TMEM) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  chain_begin(p.cs);
  // Inside a chain the row tables, the mask and older cache entries may be read before the wait; Q and this pass's K and V
  // come from the kernel right before this one.
  const bool early = p.cs.signal_ptr != nullptr;
  if (!early) chain_wait_cta(p.cs);
  if (warp == 0 && lane == 0) {
    asm volatile("prefetch.tensormap [%0];" ::"l"(&map_k) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(&map_v) : "memory");
    for (int s = 0; s < KL_MAX_SLOTS; ++s) { mbar_init(bar(KB_FULL + s), 1); mbar_init(bar(KB_EMPTY + s), 1); mbar_init(bar(KB_TAIL + s), 1); }
    mbar_init(bar(KB_Q), KL_SOFT / 32);
    for (int s = 0; s < 2; ++s) {
      mbar_init(bar(KB_S_FULL + s), 1); mbar_init(bar(KB_S_EMPTY + s), KL_SOFT / 32);
      mbar_init(bar(KB_P_FULL + s), KL_SOFT / 32); mbar_init(bar(KB_PV_DONE + s), 1);
    }
    sm->abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  } else if (warp == 3) {
    // ---- the CTA's tiles, one per lane
    const int G = (int)gridDim.x;
    // (up to 32 sequences, lane by lane: their order, first rows and rows, and the keys below their first row's extent)
    const bool few = p.n_seq <= 32;
    int s_order = lane, s_row0 = 0, s_rows = 0, s_nc = 0;
    if (few && lane < p.n_seq) {
      if (p.seq_order) s_order = p.seq_order[lane];
      s_row0 = p.seq_off[lane];
      s_rows = p.seq_off[lane + 1] - s_row0;
      if (s_rows > 0) s_nc = p.rt.n_cache[s_row0];
    }
    // rows that a tile may have: as few as leave every tile a CTA of its own (narrow tiles take less time per chunk), else the most.
    // (The launch has as many CTAs as there are tiles of the most rows, so a sequence whose bound is one such tile is never cut.)
    int most = KL_ROWS, first = 0, count = 0;   // first, count: of this lane's sequence, when tiles are that narrow
    if (few)
      for (int m = 32; m < KL_ROWS && most == KL_ROWS; m += 16) {
        count = (s_rows + m - 1) / m;
        first = count;
        for (int d = 1; d < 32; d <<= 1) { const int v = __shfl_up_sync(0xffffffffu, first, d); if (lane >= d) first += v; }
        if (__shfl_sync(0xffffffffu, first, 31) * dm.H <= G) most = m;
        first -= count;
      }
    KlTile tl;
    tl.nrows = 0; tl.kext = 0;
    int h = 0, b = -1, rb = 0;
    if (most < KL_ROWS) {
      const int sr = (int)blockIdx.x / dm.H;
      h = (int)blockIdx.x - sr * dm.H;
      const int owner = __ffs(__ballot_sync(0xffffffffu, sr >= first && sr < first + count)) - 1;
      rb = sr - __shfl_sync(0xffffffffu, first, max(owner, 0));
      if (lane == 0) b = owner;
    } else {
      // the launch's tiles are ordered by row tile (unused ones come last), sequence (longest first) and head, and dealt out in
      // turn, every other round backwards
      const int i = lane * G + ((lane & 1) ? G - 1 - (int)blockIdx.x : (int)blockIdx.x);
      int bi = 0;
      if (i < p.n_tiles) {
        const int sr = i / dm.H;
        h = i - sr * dm.H; rb = sr / p.n_seq;
        b = bi = sr - rb * p.n_seq;
      }
      if (few) bi = __shfl_sync(0xffffffffu, s_order, bi);
      else if (b >= 0 && p.seq_order) bi = p.seq_order[b];
      if (b >= 0) b = bi;
    }
    int seq_row0 = __shfl_sync(0xffffffffu, s_row0, max(b, 0) & 31), seq_rows = __shfl_sync(0xffffffffu, s_rows, max(b, 0) & 31);
    int nc_seq = __shfl_sync(0xffffffffu, s_nc, max(b, 0) & 31);
    if (b >= 0) {
      if (!few) {
        seq_row0 = p.seq_off[b]; seq_rows = p.seq_off[b + 1] - seq_row0;
        if (seq_rows > 0) nc_seq = p.rt.n_cache[seq_row0];
      }
      const int n = (seq_rows + most - 1) / most;
      if (rb < n) {
        const int rows = ((seq_rows + n - 1) / n + 15) & ~15;
        const bool tree = p.rt.mask != nullptr;
        tl.b = b; tl.head = h; tl.rel_row0 = rb * rows; tl.row0 = seq_row0 + rb * rows;
        tl.nrows = min(rows, seq_rows - rb * rows); tl.seq_rows = seq_rows;
        if (tl.nrows > 0) {
          // without a tree every row attends one key more than the row before it
          tl.tree_base = tree ? nc_seq : nc_seq + tl.rel_row0;
          tl.kext = min(tree ? nc_seq + seq_rows : tl.tree_base + tl.nrows - 1, dm.max_ctx);
          tl.nc_min = min(tl.tree_base, tl.kext);
          tl.old_keys = !early ? 0 : tree ? nc_seq : nc_seq - 1;
        }
      }
    }
    const bool some = tl.nrows > 0 && tl.kext > 0;
    const uint32_t all = __ballot_sync(0xffffffffu, some);
    if (some) sm->tiles[__popc(all & ((1u << lane) - 1u))] = tl;
    const int rows_max = __reduce_max_sync(0xffffffffu, tl.nrows);
    if (lane == 0) { sm->n_tiles = __popc(all); sm->rows_max = rows_max; }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = sm->tmem;
  const int n_tiles = sm->n_tiles;
  // ---- operands behind KlShared, sized for the CTA's largest tile: its rows, two buffers of weights and remainders, and ring slots.  K and V
  // have rings of their own because each is read by a warp of its own: in a common ring one reader could be a lap ahead of the
  // other, and a barrier's parity would mistake the laps.  V has a chunk's two slots more: the scores run two chunks ahead of
  // the output, so that K's slots come free as much earlier, and with the copies in turn, K a chunk ahead, both rings are full
  // of copies under way.
  const int N = max(16, (sm->rows_max + 15) & ~15);
  const uint32_t tile_bytes = (uint32_t)N * 256u;
  const uint32_t sQ = base + kl_front_bytes(dm.NMAX), sP = sQ + tile_bytes, ring = sP + 4u * tile_bytes;
  const int n_slots = min(KL_MAX_SLOTS, (int)((raw + KL_SMEM - ring) / KL_SLOT)), v_slots = n_slots / 2 + 1, k_slots = n_slots - v_slots;
  // second 64 keys of a chunk: multiplied only if some row attends one of them
  auto both_halves = [&](int kext, int c) { return kext - c * KL_KEYS > KL_KEYS / 2; };

  if (warp == 0) {
    // ===================== TMA producer =====================
    if (lane == 0 && n_tiles > 0) {
      const uint64_t pol = evict_first();
      bool ok = true, waited = false;
      int ks = 0, vs = 0;
      uint32_t k_ph = 0, v_ph = 0;
      auto take = [&](int slot, uint32_t ph, bool old) {   // a free slot; waits for the launch before this one at the first keys that it wrote
        if (!waited && !old) {
          if (early) chain_wait_thread(p.cs);
          chain_fence_async_reads();
          waited = true;
        }
        ok = ok && mbar_wait(bar(KB_EMPTY + slot), ph ^ 1u, &sm->abort_flag, p.status);
        return ok;
      };
      for (int k = 0; k < n_tiles && ok; ++k) {
        const KlTile& tl = sm->tiles[k];
        const int kext = tl.kext, old_keys = tl.old_keys, n_chunks = (kext + KL_KEYS - 1) / KL_KEYS;
        const int key_row0 = (tl.b * dm.H + tl.head) * dm.max_ctx;   // first row of this (sequence, head) in the cache plane
        auto load_k = [&](int c) {
          for (int dh = 0; dh < 2; ++dh) {
            if (!take(ks, k_ph, (c + 1) * KL_KEYS <= old_keys)) return;
            const uint32_t fb = bar(KB_FULL + ks);
            mbar_expect_tx(fb, KL_SLOT);
            load_box_2d(ring + (uint32_t)ks * KL_SLOT, &map_k, fb, dh * 64, key_row0 + c * KL_KEYS, pol);
            if (++ks == k_slots) { ks = 0; k_ph ^= 1u; }
          }
        };
        auto load_v = [&](int c) {
          for (int kh = 0; kh < (both_halves(kext, c) ? 2 : 1); ++kh) {
            const int slot = k_slots + vs;
            if (!take(slot, v_ph, (c + 1) * KL_KEYS <= old_keys)) return;
            // (the values that the extent ends among are full when warp 3 has cleared the rest)
            const uint32_t fb = bar((c * 2 + kh + 1) * 64 > kext ? KB_TAIL + slot : KB_FULL + slot);
            mbar_expect_tx(fb, KL_SLOT);
            load_box_3d(ring + (uint32_t)slot * KL_SLOT, &map_v, fb, 0, key_row0 + c * KL_KEYS + kh * 64, 0, pol);
            if (++vs == v_slots) { vs = 0; v_ph ^= 1u; }
          }
        };
        // (K a chunk ahead of V, also across the tiles' ends: V's slots come free later)
        if (k == 0) load_k(0);
        for (int c = 0; c < n_chunks && ok; ++c) {
          if (c + 1 < n_chunks) load_k(c + 1);
          if (ok) load_v(c);
        }
        if (ok && k + 1 < n_tiles) {
          const KlTile& nx = sm->tiles[k + 1];
          const int nx_row0 = (nx.b * dm.H + nx.head) * dm.max_ctx;
          for (int dh = 0; dh < 2; ++dh) {
            if (!take(ks, k_ph, KL_KEYS <= nx.old_keys)) break;
            const uint32_t fb = bar(KB_FULL + ks);
            mbar_expect_tx(fb, KL_SLOT);
            load_box_2d(ring + (uint32_t)ks * KL_SLOT, &map_k, fb, dh * 64, nx_row0, pol);
            if (++ks == k_slots) { ks = 0; k_ph ^= 1u; }
          }
        }
      }
      if (!ok || sm->abort_flag) {  // give the copies already issued time to land before the CTA's shared memory is released
        const unsigned long long t0 = now_ns();
        while (now_ns() - t0 < 2000000ull) __nanosleep(1000);
      }
    }
  } else if (warp == 1 || warp == 2) {
    // ===================== MMA issuers: scores (warp 1) and output (warp 2) =====================
    // Two warps, because a chunk's sixteen instructions with their waits take one warp 1.3 us, longer than its softmax.
    if (n_tiles > 0) {
      uint32_t leader;
      asm volatile("{\n\t.reg .pred P;\n\telect.sync _|P, 0xffffffff;\n\tselp.u32 %0, 1, 0, P;\n\t}" : "=r"(leader));
      auto wait_warp = [&](uint32_t b, uint32_t parity) {
        return __all_sync(0xffffffffu, mbar_wait(b, parity, &sm->abort_flag, p.status)) != 0;
      };
      const int slot0 = warp == 1 ? 0 : k_slots, slot_end = warp == 1 ? k_slots : n_slots;
      int slot = slot0;
      uint32_t ph = 0;
      auto next = [&]() { if (++slot == slot_end) { slot = slot0; ph ^= 1u; } };
      bool ok = true;
      int j0 = 0;   // chunks of the tiles before this one
      const uint32_t idesc_qk = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(KL_KEYS >> 4) << 24);
      const uint32_t idesc_pv = idesc_qk + ((uint32_t)(N >> 3) << 17) | (1u << 15) | (1u << 16);   // N doubled (weights and remainders), both operands MN-major; M = 128 head dimensions
      const uint64_t q_desc = desc_kmajor(sQ);
      for (int k = 0; k < n_tiles && ok; ++k) {
        const KlTile& tl = sm->tiles[k];
        const int kext = tl.kext, n_chunks = (kext + KL_KEYS - 1) / KL_KEYS;
        // (chunk -1 of the first tile issues nothing: it fetches the loop's code while Q is on its way)
        if (warp == 1) {
          for (int c = k ? 0 : -1; c < n_chunks && ok; ++c) {
            const int j = j0 + c;
            const bool live = c >= 0, on = live && leader;
            if (c == 0) ok = wait_warp(bar(KB_Q), (uint32_t)(k & 1));
            if (live && ok) ok = wait_warp(bar(KB_S_EMPTY + (j & 1)), (uint32_t)((j >> 1) & 1) ^ 1u);
            const uint32_t d = tmem + (uint32_t)(j & 1) * 128u;
#pragma unroll 1
            for (int dh = 0; dh < 2 && ok; ++dh) {
              if (live) {
                ok = wait_warp(bar(KB_FULL + slot), ph);
                if (!ok) break;
              }
              tc_fence_after();
              const uint64_t kd = desc_kmajor(ring + (uint32_t)slot * KL_SLOT);
              const uint64_t qd = q_desc + (uint64_t)((uint32_t)dh * (uint32_t)N * 128u >> 4);
#pragma unroll
              for (int kk = 0; kk < 4; ++kk) umma_if(on, d, kd + (uint64_t)(kk * 2), qd + (uint64_t)(kk * 2), idesc_qk, (dh | kk) ? 1u : 0u);
              commit_if(on, bar(KB_EMPTY + slot));
              commit_if(on && dh, bar(KB_S_FULL + (j & 1)));
              __syncwarp();
              if (live) next();
            }
          }
        } else {
          const uint32_t d_o = tmem + 256u;
          for (int c = k ? 0 : -1; c < n_chunks && ok; ++c) {
            const int j = j0 + c;
            const bool live = c >= 0, on = live && leader;
            const int halves = both_halves(kext, c) ? 2 : 1;
            if (live) ok = wait_warp(bar(KB_P_FULL + (j & 1)), (uint32_t)((j >> 1) & 1));
            const uint64_t p_desc = desc_mn32(sP + (uint32_t)(j & 1) * 2u * tile_bytes, KL_KEYS * 32);
#pragma unroll 1
            for (int kh = 0; kh < halves && ok; ++kh) {
              if (live) {
                ok = wait_warp(bar(KB_FULL + slot), ph);
                if (!ok) break;
              }
              tc_fence_after();
              const uint64_t vd = desc_mn128(ring + (uint32_t)slot * KL_SLOT, KL_SLOT / 2);
#pragma unroll
              for (int kk = 0; kk < 4; ++kk)   // 16 keys: 2048 bytes of V, 512 of the weights
                umma_if(on, d_o, vd + (uint64_t)(kk * 128), p_desc + (uint64_t)((kh * 4 + kk) * 32), idesc_pv, (c | kh | kk) ? 1u : 0u);
              commit_if(on, bar(KB_EMPTY + slot));
              commit_if(on && kh == halves - 1, bar(KB_PV_DONE + (j & 1)));
              __syncwarp();
              if (live) next();
            }
          }
        }
        j0 += n_chunks;
      }
    }
  } else if (warp == 3) {
    // ===================== the end of every tile's values =====================
    // Keys past the extent have weights of zero, but their slots may hold anything (and the box that crosses the last slot another
    // head's or sequence's values), and zero times that has to be zero.  A warp of its own: the issuing one would do it between the
    // weights of two chunks (which cost the 7B step 0.4 %, this 0.2).
    int v_used = 0;       // V slots filled by the tiles before, in the ring's order
    uint32_t tail_ph = 0;
    bool ok = true;
    for (int k = 0; k < n_tiles && ok; ++k) {
      const int kext = sm->tiles[k].kext, rows = kext & 63;   // of the last half chunk
      v_used += (kext + 63) >> 6;
      if (rows == 0) continue;
      const int slot = k_slots + (v_used - 1) % v_slots;
      ok = __all_sync(0xffffffffu, mbar_wait(bar(KB_TAIL + slot), (tail_ph >> slot) & 1u, &sm->abort_flag, p.status)) != 0;
      if (!ok) break;
      tail_ph ^= 1u << slot;
      uint4* const v = reinterpret_cast<uint4*>(gen + (ring - base) + (size_t)slot * KL_SLOT);   // [2 halves of the dimensions][64 keys][8]
      for (int i = rows * 8 + lane; i < 64 * 8; i += 32) v[i] = v[64 * 8 + i] = make_uint4(0u, 0u, 0u, 0u);
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      __syncwarp();
      if (lane == 0) mbar_arrive(bar(KB_FULL + slot));
    }
  } else if (warp >= 4) {
    // ===================== softmax and output =====================
    if (n_tiles > 0) {
      const KlCtx t{sm, bar0, tmem, gen + (sQ - base), gen + (sP - base), early};
      switch (N >> 4) {
        case 1: kl_softmax<4>(p, t, n_tiles); break;
        case 2: kl_softmax<8>(p, t, n_tiles); break;
        case 3: kl_softmax<12>(p, t, n_tiles); break;
        case 4: kl_softmax<16>(p, t, n_tiles); break;
        case 5: kl_softmax<20>(p, t, n_tiles); break;
        default: kl_softmax<24>(p, t, n_tiles); break;
      }
    }
  }
  // a CTA without tiles still waits for its predecessor before it reports completion
  if (n_tiles == 0 && threadIdx.x == 0) chain_wait_thread(p.cs);
  // ---- teardown: everyone meets, then the allocating warp frees the tensor memory
  tc_fence_before();
  __syncthreads();
  chain_exit(p.cs);
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(KL_TMEM) : "memory");
  }
}

}  // namespace

int attn_kl_row_tiles(int rows) { return (rows + KL_ROWS - 1) / KL_ROWS; }
// Tiles of the most rows leave either ring a chunk (K two slots, V three).
bool attn_kl_supported(int hd, int NMAX) {
  return hd == KL_HD && 1024 + kl_front_bytes(NMAX) + 5u * KL_ROWS * 256u + 5u * KL_SLOT <= KL_SMEM;
}

cudaError_t attn_kl_prepare(int hd) {
  if (hd != KL_HD) return cudaSuccess;
  return cudaFuncSetAttribute(attention_kl_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)KL_SMEM);
}

// map_k: tensor map of the layer's K plane ([sequences * heads * max_ctx rows][128 dims], box 128 rows x 64 dims); map_v: of its V
// plane as [2 halves][rows][64 dims], box 2 x 64 x 64: a slot is one copy.
// One CTA per SM, or more where a CTA would have more tiles than its table holds.
cudaError_t launch_attention_kl(const void* map_k, const void* map_v, const float* qkv, void* out, const RowTables& rt,
                                const int32_t* seq_off, const int32_t* seq_order, const uint32_t* mask_t, const Dims& dm, int n_seq, int row_tiles, int n_sms,
                                int32_t* status, Chain* chain, cudaStream_t st) {
  if (!attn_kl_supported(dm.hd, dm.NMAX)) return cudaErrorInvalidValue;
  const int n_tiles = dm.H * n_seq * row_tiles;
  int grid = (n_tiles + KL_MAX_TILES - 1) / KL_MAX_TILES;
  if (grid < n_sms) grid = n_tiles < n_sms ? n_tiles : n_sms;
  KlParams p;
  p.qkv = qkv; p.out = (__nv_bfloat16*)out; p.rt = rt; p.seq_off = seq_off; p.seq_order = seq_order; p.mask_t = rt.mask ? mask_t : nullptr; p.dm = dm; p.n_seq = n_seq;
  p.n_tiles = n_tiles; p.status = status;
  p.cs = chain ? chain->link((unsigned)grid) : ChainSync{nullptr, 0u, nullptr, status, nullptr};
  launch_pdl(attention_kl_kernel, dim3(grid), KL_THREADS, KL_SMEM, st, *(const CUtensorMap*)map_k, *(const CUtensorMap*)map_v, p);
  return cudaGetLastError();
}

}  // namespace rd
