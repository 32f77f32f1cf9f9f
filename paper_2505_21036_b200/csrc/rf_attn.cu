// Pattern-masked FlashAttention forward on tcgen05 / TMEM / TMA (Eq. 1-2 with the masks of Sec. 3.2).
//
// An item of work is two adjacent 128-row query tiles of one head (two "streams"); a CTA walks the union of
// their KV-tile lists, so every K/V tile fetched by TMA feeds up to two S = Q K^T and two O += P V
// contractions.  A CTA works off one item after another: its own, then those of CTAs that have not started yet, which it
// takes over through cluster launch control.  The TMA and MMA warps run on into the next item while the softmax
// warps write out the last one: per item that hides what a CTA of its own pays for its start, its Q and first K, its first
// scores and its end, 6 to 9 us (24 heads, 8448 tokens, D = 128: 83 us an item, 490 -> 480 us a call; 48 heads,
// 17 776 tokens, D = 64: 130 us an item, 2930 -> 2700 us masked, 5590 -> 5210 dense, most of it from the issuing
// thread's shorter code).  Warp roles:
//   warps 0-3  softmax of stream 0   (one thread per query row, TMEM lane = row)
//   warps 4-7  softmax of stream 1
//   warp  8    TMA producer: Q once per item, K and V tiles into two shared-memory rings (V of tile u and K of
//              tile u + 1 as a pair under one full / one empty mbarrier)
//   warp  9    MMA issuer: tcgen05.mma, accumulators in TMEM (S0, S1, O0, O1)
//   warp  10   one thread fetches items and publishes them in shared memory
//   (warp 11 only fills the third warpgroup, which hands its registers to the softmax warpgroups)
// Per listed tile and stream: S lands in TMEM, the softmax warps read their rows (tcgen05.ld), keep a
// running maximum in fp32, write P as packed bf16 back into TMEM (tcgen05.st: on top of the S
// columns at D = 96 / 128, into spare columns at D = 64) and the MMA warp multiplies it with V straight
// from TMEM.  V carries one column more, of ones: O's column D is the sum of a row's weights of one tile as rounded to bf16, the
// ones that are multiplied with V; the softmax warps take it out tile by tile, and the sum over the tiles normalises O (which makes
// O an exact convex combination of V rows with slightly perturbed weights: the rounding of a dominant weight cancels instead of
// scaling the output row).  The running maximum is raised lazily (see kRaise), in which case the softmax warp itself
// rescales its rows of O in TMEM; the final O / l and the log-sum-exp do not depend on it.
// PARTIAL tiles apply the exact element mask of the head's pattern; FULL tiles skip it.
#include <algorithm>

#include "rf_attn_common.cuh"

namespace {

using namespace sm100;
using namespace rf_attn;

constexpr int kThreads = kWsThreads;        // 3 warpgroups: softmax 0, softmax 1, {TMA, MMA, items, 1 idle warp}
constexpr int kTmaWarp = 8, kMmaWarp = 9, kItemWarp = 10;
constexpr int kItemSlots = 2, kItemWords = 12, kItemReaders = 9;   // readers: eight softmax warps and the TMA thread
constexpr uint32_t kMore = 4, kLast = 8;   // of a tile record, see the TMA producer
constexpr int kAskAhead = 4;   // tiles an item's longer list has left when the next item is asked for: 8 us or more, an answer takes about one
// What bounds the loop: a stream is the chain scores -> softmax -> P V -> Q K^T, so what counts is how few dependent
// operations stand between the scores' arrival and the hand-over of P, and, once the board is at its power limit (every long
// call), the energy of a tile, a sixth of which are the softmax warps' instructions.  At D = 96 / 128 the first kSpec weights
// are taken while the tile's maximum is being found and the first half of P is stored and multiplied under the second half's
// exponentials; at D = 64 the maximum comes first.  The row sums of the rounded weights were 192 of a row's 512 instructions a tile
// (two to widen a pair, one to add it); the tensor pipe takes them in 16 columns more of P V (128 cycles beside 2048 a pair of
// tiles at D = 128).  Repeated calls at the power limit, before and after: dense 24 heads, 8448 tokens, D = 128 870 -> 841 us;
// 24 heads, 119 056 tokens 73.8 -> 71.7 ms; 48 heads, 5082 tokens, D = 96 2530 -> 2415 us; 48 heads, 17 776 tokens,
// D = 64 2900 -> 2763 us masked, 5340 -> 4990 dense.
// Column D holds one tile's sum only: it is read and cleared before the next P is handed over, and the tiles are added up in fp32.
// An accumulator of the whole row cuts every weight off at the last place of the sum so far: beside one key of weight 1, 2^18
// keys of 2^-19 lost 2.1e-3 of the row's weight in it; with the sums by tile the error is what the outputs' rounding leaves, 5e-5, as it
// is with all sums added up by the softmax warps, whose outputs are within rel 6e-5.  It costs a load and a store of one column a
// tile: sixteen shapes, 0.993 to 1.010 times as fast as without.
// Without lse the sum of the unrounded weights is left out (a template: dense D = 64 5.74 -> 5.59 ms).
// Lazy rescaling of the running maximum: it is raised once a tile's maximum exceeds it by kRaise (log2 units; all rows
// of the warp more than kRaiseMargin above theirs then raise it together).  A tile's weights thus sum to 2^32 at most;
// bf16 P and the fp32 sums carry the same relative precision at every exponent and 2^32 times the longest row is far
// from overflow, so O / l and the log-sum-exp do not depend on how stale the running maximum is.
constexpr float kLazyRaise = 32.0f;         // D = 64: the maximum comes before the weights there
constexpr float kRaise = 25.0f, kRaiseMargin = 8.0f;
constexpr int kSpec = 32;                   // weights taken before the tile's maximum is known

constexpr size_t kL2Bytes = 48u << 20;      // K and V of the heads worked on at the same time: well inside the 126 MB L2

struct Maps { CUtensorMap m[8]; };

template <int D>
struct Cfg {
  static constexpr int KB = (D + 63) / 64;            // 64-column (128-byte) blocks per row
  // first column of the second block.  Q and K of D = 96 are fetched as columns [0,64) and [64,128): the TMA box
  // reaches past the tensor's 96 columns and the missing ones arrive as zeros; they are never read
  // (Q K^T runs 6 k-steps).  V has blocks of its own, see VBOX.
  static constexpr int COL1 = 64;
  static constexpr uint32_t BLK = 128 * 128;          // bytes of one 128-row x 64-col bf16 block
  static constexpr uint32_t TILE = KB * BLK;          // bytes of one 128-row tile
  // At D = 64 O is narrow enough for P of both streams to have TMEM columns of its own (with the row sums' columns that
  // makes all 512): a stream's next scores are computed during the softmax of its current tile, once both streams
  // have read theirs (S0 and S1 share columns).  At D = 96 / 128 P lives on top of the S columns it was computed from.
  static constexpr bool S_EARLY = D == 64;
  static constexpr int NK = D == 64 ? 3 : 2;          // K ring depth
  static constexpr int NV = D == 64 ? 3 : 2;          // V ring depth
  // byte offset, inside a tile, of the 16 columns of k-step ks of the Q K^T contraction
  static __host__ __device__ constexpr uint32_t koff(int ks) {
    return ks < 4 ? (uint32_t)ks * 32u : BLK + (uint32_t)(ks - 4) * 32u;
  }
  // V, the MN-major operand of P V, lies in blocks of VBOX columns; behind its D columns stands a block whose first column
  // is one and whose others are zero, so that O's column D is a tile's row sum of the weights (see the softmax).  At D = 96
  // blocks of 32 columns (64-byte swizzle) put that block next to column 95.
  static constexpr int VBOX = D == 96 ? 32 : 64;
  static constexpr uint32_t VROW = VBOX * 2, VBLK = 128 * VROW, VLOAD = D / VBOX * VBLK, VTILE = VLOAD + VBLK;
  static constexpr int NPV = D + 16;                  // columns of O += P V
  // P is handed over in parts, part p the keys [cut(p), cut(p + 1)): P V of the first half runs under the exponentials of the
  // second.  (At D = 64 P V is not on a stream's chain, and half as a part of its own costs more than it hides: dense 8500 ->
  // 9010 kcycles a call; parts of 96 + 32 or 64 + 32 + 32 keys at D = 96 / 128 are up to 4 % behind the halves.)
  static constexpr int PARTS = D == 64 ? 1 : 2;
  static __host__ __device__ constexpr int cut(int p) { return p * (BN / PARTS); }
  // Byte offset of the 16-byte chunk c of a row of such a block; chunks 0 and 1 are the 16 columns P V takes.
  static __host__ __device__ constexpr uint32_t vchunk(int row, int c) { return row * VROW + ((VBOX == 64 ? c ^ (row & 7) : c ^ ((row >> 1) & 3)) << 4); }
  static constexpr uint32_t Q = 0;
  static constexpr uint32_t K0 = Q + 2 * TILE;
  static constexpr uint32_t V0 = K0 + NK * TILE;
  static constexpr uint32_t BAR = V0 + NV * VTILE;
  // barrier slots (8 bytes each)
  // V of tile u and K of tile u + 1 travel as a pair: they are wanted in the same iteration of the MMA warp and
  // released by it together, so one full and one empty barrier per pair (B_F, B_E) serve both; K of the first
  // tile has its own two (B_K0 landed, B_K0E consumed).
  static_assert(NK == NV, "K and V rings advance together");
  static constexpr int NP = NV;
  static constexpr int B_Q = 0, B_K0 = 1, B_K0E = 2, B_F = 3, B_E = B_F + NP, B_SF = B_E + NP,
                       B_PF = B_SF + 2, B_OF = B_PF + 2 * PARTS, B_SE = B_OF + 2 /* S read, not at D = 96 */, B_QE = B_SE + 2 /* Q consumed */,
                       B_REQ = B_QE + 1, B_CLC = B_REQ + 1, B_IF = B_CLC + 1, B_IE = B_IF + kItemSlots, B_COUNT = B_IE + kItemSlots;
  static constexpr uint32_t MISC = BAR + 8 * ((B_COUNT + 7) / 8 * 8);
  static constexpr uint32_t ITEM = MISC + 64;         // kItemSlots items of kItemWords words, then the launch-control answer
  static constexpr uint32_t ANSWER = ITEM + kItemSlots * kItemWords * 4;
  static constexpr uint32_t RECORD = ANSWER + 16;     // tile records: one per ring slot, then the first tile's
  static constexpr uint32_t TOTAL = RECORD + 4 * (NP + 1);
  static constexpr uint32_t ALLOC = TOTAL + 1024;     // slack for manual 1024-byte alignment
  static_assert(ALLOC <= 227 * 1024, "shared memory of a CTA");
  // TMEM columns.  The row sums' 16 columns a stream do not fit beside two whole S at D = 64 and 128, so S0 and S1 share 32
  // columns there (P lies outside them): a stream's scores are computed once the other stream has read its own.
  static constexpr bool S_SHARED = D != 96;
  static constexpr uint32_t S_COL0 = 0, S_COL1 = S_SHARED ? 96 : 128, S_END = S_COL1 + 128, TMEM_COLS = 512;
  static constexpr uint32_t P_COL0 = S_EARLY ? S_END : S_COL0, P_COL1 = S_EARLY ? S_END + 64 : S_COL1 + 64;   // packed bf16, 64 columns
  static constexpr uint32_t O_COL0 = S_EARLY ? S_END + 128 : S_END, O_COL1 = O_COL0 + NPV;
  static_assert(O_COL1 + NPV <= TMEM_COLS, "TMEM columns");
};

// One item of work: two adjacent query tiles of one head.
// (or, of a split one, a piece: n0 and n1 entries of the two lists from b0 and b1 on)
struct Item { int bh, qt0, cls, n0, n1, window, b0, b1; };

// Which item the CTA of index `lin` of the grid stands for.  Heads are taken in groups whose K and V fit the L2 cache
// together (one head at a time where they are long); inside a group the last pair of query tiles of every head comes
// first: the text rows list every tile and are the longest items, while the first pairs list the fewest (the windows of
// Spatial and Temporal heads are cut at the ends), so the SMs run out of work with short items.
__device__ __forceinline__ void place_item(uint64_t lin, int group, int heads, int pairs, int& bh, int& pair) {
  const uint64_t per = (uint64_t)group * pairs;
  const int g0 = (int)(lin / per) * group;
  const uint32_t r = (uint32_t)(lin % per), in = min(group, heads - g0);
  bh = g0 + (int)(r % in);
  pair = pairs - 1 - (int)(r / in);
}

// What a unit of the grid is: an item, or one piece of an item that may be split.
struct Unit { int bh, pair, piece, most, tiles, slot, split; };
__device__ __forceinline__ void place_unit(uint64_t lin, const RfAttnArgs& a, Unit& un) {
  const RfSplit& sp = a.sp;
  const int heads = a.g.B * a.g.H, pairs = rf_cdiv(a.g.nQ, 2);
  un.piece = 0;
  un.most = 1;
  un.tiles = un.slot = un.split = 0;
  if (!sp.on) {
    place_item(lin, a.heads_l2, heads, pairs, un.bh, un.pair);
    return;
  }
  const uint32_t u = (uint32_t)lin;
  if (u < sp.n_text) {                                  // pairs with text rows
    const int item = (int)(u / sp.kt);
    un.most = sp.kt; un.tiles = sp.lt; un.piece = (int)(u % sp.kt); un.slot = (int)u; un.split = item;
    un.bh = item % heads;
    un.pair = pairs - 1 - item / heads;
    return;
  }
  int item = (int)(u - sp.n_text), row;
  if (item >= (int)sp.first_tail) {                     // the tail: from row0 on, row by row
    const int t = item - (int)sp.first_tail, i = t / sp.kr, head = sp.head_row0 + i;
    un.most = sp.kr; un.tiles = sp.lr; un.piece = t % sp.kr;
    un.slot = (int)(sp.kt > 1 ? sp.n_text : 0) + t;
    un.split = (sp.kt > 1 ? heads * sp.text_pairs : 0) + i;
    row = sp.row0 + head / heads;
    un.bh = head % heads;
  } else {                                              // whole items: in groups of heads as in place_item
    int g0 = 0, in, n;
    for (;; g0 += a.heads_l2, item -= n) {
      in = min(a.heads_l2, heads - g0);
      n = in * sp.row0 + min(max(sp.head_row0 - g0, 0), in);
      if (item < n) break;
    }
    row = item / in;
    un.bh = g0 + item % in;
  }
  un.pair = pairs - sp.text_pairs - 1 - row;
}

// 16 and 32 bf16 columns of an output row.
__device__ __forceinline__ void store_sector(uint4* dst, const uint32_t* v, bool o32) {
  if (o32) {
    st_global_v8(dst, v);
  } else {
    dst[0] = make_uint4(v[0], v[1], v[2], v[3]);
    dst[1] = make_uint4(v[4], v[5], v[6], v[7]);
  }
}
__device__ __forceinline__ void store_columns(uint4* dst, const uint32_t* v, bool o32) {
  store_sector(dst, v, o32);
  store_sector(dst + 2, v + 8, o32);
}

// Where this thread's row of an item goes.
struct Row {
  uint4* o;
  size_t at;       // row of [B*H][N]
  bool inside;     // false: past the sequence
  bool o32;        // a thread writes its row alone, so a warp's store touches 32 rows: whole 32-byte sectors where O allows it
};
__device__ __forceinline__ Row output_row(const RfAttnArgs& a, const int* iw, int j, int row_in_tile) {
  const RfGeom& g = a.g;
  const int r = (iw[1] + j) * BM + row_in_tile;
  int tok = r;
  if (iw[2] == RF_TEMPORAL && g.permute && r < g.Nv) tok = (r % g.T) * g.S + r / g.T;
  Row row;
  row.inside = r < g.N && rf_in_bounds(tok, g.N, a.dev_status);
  row.at = (size_t)iw[0] * g.N + min(tok, g.N - 1);
  row.o = reinterpret_cast<uint4*>(a.o + row.at * g.D);
  row.o32 = (reinterpret_cast<uintptr_t>(a.o) & 31u) == 0;
  return row;
}

// One warp's 32 rows of a piece of a split item: O and the sums go to the workspace as they are, and the last warp to
// arrive at these rows joins the pieces.  They are taken in order, so the bits do not depend on who does it.  Out of
// line: the loop over the tiles has no register to spare.
template <int D, bool LSE>
__device__ __noinline__ void leave_piece(const RfAttnArgs& a, const int* iw, uint32_t t_o, int warp, int lane, float m_run, float l_run,
                                         float l_exact, bool has_o) {
  constexpr size_t kRows = (size_t)(D / 4 + 1) * BM;          // float4 of one piece of one stream
  const int j = warp >> 2, row_in_tile = (warp & 3) * 32 + lane, pieces = iw[8];
  // (the warp as a whole)
  if (iw[1] + j >= a.g.nQ || !rf_in_bounds(iw[9], a.sp.n_slots, a.dev_status) ||
      !rf_in_bounds(iw[10] * 8 + warp, a.sp.n_tickets, a.dev_status))
    return;
  float4* first = reinterpret_cast<float4*>(a.pieces) + ((size_t)(iw[9] - iw[11]) * 2 + j) * kRows + row_in_tile;
  float4* mine = first + (size_t)iw[11] * 2 * kRows;
  if (has_o) {
#pragma unroll 1
    for (int c = 0; c < D / 32; ++c) {
      uint32_t v[32];
      tmem_ld32(t_o + c * 32, v);
      tc_wait_ld();
#pragma unroll
      for (int i = 0; i < 8; ++i)
        __stcg(mine + (c * 8 + i) * BM, make_float4(__uint_as_float(v[4 * i]), __uint_as_float(v[4 * i + 1]),
                                                    __uint_as_float(v[4 * i + 2]), __uint_as_float(v[4 * i + 3])));
    }
  }
  __stcg(mine + (D / 4) * BM, make_float4(m_run, l_run, l_exact, has_o ? 1.f : 0.f));
  __threadfence();
  __syncwarp();
  int32_t* ticket = a.tickets + iw[10] * 8 + warp;
  int before = 0;
  if (lane == 0) before = atomicAdd(ticket, 1);
  if (__shfl_sync(0xffffffffu, before, 0) != pieces - 1) return;
  __threadfence();
  const Row row = output_row(a, iw, j, row_in_tile);
  // half a row at a time, so that all loads of a piece are under way together
  constexpr int kCols = D == 64 ? 64 : D / 2;
#pragma unroll 1
  for (int c0 = 0; c0 < D; c0 += kCols) {
    float m = -INFINITY, l = 0.f, l_all = 0.f;
    bool any = false;                                          // some piece lists a tile for these rows
    float4 acc[kCols / 4];
#pragma unroll
    for (int i = 0; i < kCols / 4; ++i) acc[i] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 1
    for (int p = 0; p < pieces; ++p) {
      const float4* at = first + p * 2 * kRows;
      const float4 st = __ldcg(at + (D / 4) * BM);
      float4 o[kCols / 4];
#pragma unroll
      for (int i = 0; i < kCols / 4; ++i) o[i] = __ldcg(at + (c0 / 4 + i) * BM);
      if (st.w == 0.f) continue;                               // listed no tile: its O was never written
      any = true;
      // where one side has no maximum its O and sums are zero (or not numbers): they are added as they are
      float keep = 1.f, w = 1.f;
      if (st.x > m) {
        if (m > -INFINITY) keep = ex2(m - st.x);
        m = st.x;
      } else if (st.x > -INFINITY) {
        w = ex2(st.x - m);
      }
      l = l * keep + st.y * w;
      l_all = l_all * keep + st.z * w;
#pragma unroll
      for (int i = 0; i < kCols / 4; ++i) {
        acc[i].x = acc[i].x * keep + o[i].x * w;
        acc[i].y = acc[i].y * keep + o[i].y * w;
        acc[i].z = acc[i].z * keep + o[i].z * w;
        acc[i].w = acc[i].w * keep + o[i].w * w;
      }
    }
    if (!row.inside || !any) continue;
    const float inv = l > 0.f ? 1.f / l : 0.f;
#pragma unroll
    for (int q = 0; q < kCols / 16; ++q) {
      uint32_t v[8];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        v[2 * i] = pack_bf16(acc[q * 4 + i].x * inv, acc[q * 4 + i].y * inv);
        v[2 * i + 1] = pack_bf16(acc[q * 4 + i].z * inv, acc[q * 4 + i].w * inv);
      }
      store_sector(row.o + c0 / 8 + q * 2, v, row.o32);
    }
    if (LSE && c0 == 0) a.lse[row.at] = (m + log2f(l_all)) * 0.6931471805599453f;
  }
}

// This thread's row of O times alpha (warp-collective).
__device__ __forceinline__ void rescale_columns(uint32_t t_o, float alpha) {
  uint32_t v[32];
  tmem_ld32(t_o, v);
  tc_wait_ld();
#pragma unroll
  for (int i = 0; i < 32; ++i) v[i] = __float_as_uint(__uint_as_float(v[i]) * alpha);
  tmem_st32(t_o, v);
}
template <int D>
__device__ __forceinline__ void rescale_o(uint32_t t_o, float alpha) {
  tc_fence_after();
#pragma unroll
  for (int c = 0; c < D; c += 32) rescale_columns(t_o + c, alpha);
  tc_wait_st();
  tc_fence_before();
}
// The same out of line, for D = 96 / 128: rare as it is, the scores then stay in registers around it and the loop over the
// tiles is free of spills.  (At D = 64, inline, 16 bytes are spilt; out of line none, but 48 heads of 17 776 tokens took 5013 us
// instead of 4932 dense and 2676 instead of 2639 all Textural.)
template <int D>
__device__ __noinline__ void rescale_o_call(uint32_t t_o, float alpha) {
  tc_fence_after();
#pragma unroll 1
  for (int c = 0; c < D; c += 32) rescale_columns(t_o + c, alpha);
  tc_wait_st();
  tc_fence_before();
}

// This thread's row of scores, and the masked ones of a PARTIAL tile set to -inf.
__device__ __forceinline__ void load_scores(uint32_t t_s, uint32_t (&s)[BN]) {
  tmem_ld32(t_s, *reinterpret_cast<uint32_t(*)[32]>(&s[0]));
  tmem_ld32(t_s + 32, *reinterpret_cast<uint32_t(*)[32]>(&s[32]));
  tmem_ld32(t_s + 64, *reinterpret_cast<uint32_t(*)[32]>(&s[64]));
  tmem_ld32(t_s + 96, *reinterpret_cast<uint32_t(*)[32]>(&s[96]));
  tc_wait_ld();
}
__device__ __forceinline__ void mask_scores(const uint4* keep, uint32_t (&s)[BN]) {
  const uint4 kw = *keep;
  const uint32_t w[4] = {kw.x, kw.y, kw.z, kw.w};
#pragma unroll
  for (int c = 0; c < BN; ++c)
    if (!((w[c >> 5] >> (c & 31)) & 1u)) s[c] = 0xff800000u;  // -inf
}

// Weights of the key columns [C0, C1) of a tile: 2^(score * sc - m), packed to bf16; with LSE also their sum before rounding.
template <int C0, int C1, bool LSE>
__device__ __forceinline__ void take_weights(const uint32_t (&s)[BN], uint32_t (&pk)[BN / 2], float2& la, float2 sc2, float2 mneg) {
#pragma unroll
  for (int c = C0; c < C1; c += 4) {
    float2 e0 = __ffma2_rn(make_float2(__uint_as_float(s[c]), __uint_as_float(s[c + 1])), sc2, mneg);
    float2 e1 = __ffma2_rn(make_float2(__uint_as_float(s[c + 2]), __uint_as_float(s[c + 3])), sc2, mneg);
    e0.x = ex2(e0.x); e0.y = ex2(e0.y);
    e1.x = ex2(e1.x); e1.y = ex2(e1.y);
    pk[c / 2] = pack_bf16(e0.x, e0.y);
    pk[c / 2 + 1] = pack_bf16(e1.x, e1.y);
    if (LSE) la = __fadd2_rn(la, __fadd2_rn(e0, e1));
  }
}

// The packed weights of the key columns [C0, C1) into P.  Eight registers at a time: longer stores want that many consecutive
// registers, which costs moves (24 heads, 8448 tokens, dense, D = 128: 1153 kcycles a call with 32, 1112 with 16, 1108 with 8).
template <int C0, int C1>
__device__ __forceinline__ void store_weights(uint32_t t_p, const uint32_t (&pk)[BN / 2]) {
#pragma unroll
  for (int c = C0 / 2; c < C1 / 2; c += 8) tmem_st8(t_p + c, *reinterpret_cast<const uint32_t(*)[8]>(&pk[c]));
}

template <int D, bool LSE>
__global__ void __launch_bounds__(kThreads, 1) rf_attn_kernel(const __grid_constant__ Maps maps, const __grid_constant__ RfAttnArgs a) {
  using C = Cfg<D>;
  constexpr int KB = C::KB;
  constexpr uint32_t IDESC_S = idesc_bf16(BM, BN, 0);
  constexpr uint32_t IDESC_PV = idesc_bf16(BM, C::NPV, 1);

  extern __shared__ uint8_t smem_raw[];
  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  uint8_t* base_ptr = smem_raw + (base - smem_u32(smem_raw));
  auto bar = [&](int slot) -> uint32_t { return base + C::BAR + 8u * slot; };
  volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(base_ptr + C::MISC);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(base_ptr + C::MISC + 8);

  const RfGeom& g = a.g;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  int* items = reinterpret_cast<int*>(base_ptr + C::ITEM);
  volatile uint32_t* records = reinterpret_cast<volatile uint32_t*>(base_ptr + C::RECORD);

  if (tid == 0) {
    mbar_init(bar(C::B_Q), 1);
    mbar_init(bar(C::B_K0), 1);
    mbar_init(bar(C::B_K0E), 1);
    for (int s = 0; s < C::NP; ++s) { mbar_init(bar(C::B_F + s), 1); mbar_init(bar(C::B_E + s), 1); }
    for (int j = 0; j < 2; ++j) {
      mbar_init(bar(C::B_SF + j), 1);
      for (int p = 0; p < C::PARTS; ++p) mbar_init(bar(C::B_PF + j * C::PARTS + p), 4);   // one arrival per softmax warp
      mbar_init(bar(C::B_OF + j), 1);
      mbar_init(bar(C::B_SE + j), 4);
    }
    mbar_init(bar(C::B_QE), 1);
    mbar_init(bar(C::B_REQ), 1);
    mbar_init(bar(C::B_CLC), 1);
    for (int i = 0; i < kItemSlots; ++i) { mbar_init(bar(C::B_IF + i), 1); mbar_init(bar(C::B_IE + i), kItemReaders); }
    *abort_flag = 0;
    mbar_init_fence();
  }
  for (int i = tid; i < C::NV * BN * 2; i += kThreads) {   // the 16 columns behind V's: one, then zeros
    const int v = i / (BN * 2), row = i / 2 % BN, c = i % 2;
    *reinterpret_cast<uint4*>(base_ptr + C::V0 + v * C::VTILE + C::VLOAD + C::vchunk(row, c)) = make_uint4(c == 0 ? 0x3f80u : 0u, 0u, 0u, 0u);
  }
  fence_proxy_async_smem();
  if (warp == kTmaWarp) {
    if (lane < 8) prefetch_tmap(&maps.m[lane]);
    __syncwarp();
    tmem_alloc(smem_u32(const_cast<uint32_t*>(tmem_slot)), C::TMEM_COLS);
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  const WaitCtx wc{abort_flag, a.dev_status};
  rf_grid_wait();

  // The i-th item of this CTA.  False: there is none (or a wait was abandoned).
  auto take = [&](int i, Item& im, int waited) -> bool {
    const int slot = i % kItemSlots;
    if (!mbar_wait_long(bar(C::B_IF + slot), (i / kItemSlots) & 1, wc, waited)) return false;
    const int* w = items + slot * kItemWords;
    im.bh = w[0]; im.qt0 = w[1]; im.cls = w[2]; im.n0 = w[3]; im.n1 = w[4]; im.window = w[5]; im.b0 = w[6]; im.b1 = w[7];
    return im.bh >= 0;
  };
  auto lists = [&](const Item& im) -> Lists {
    Lists L;
    L.lkv = rf_kv_len(g, im.cls);
    L.listed = a.head_class != nullptr;
    L.n0 = im.n0;
    L.n1 = im.n1;
    L.first = im.b0;
    L.l0 = L.listed ? a.kv_tile + ((size_t)im.bh * g.nQ + im.qt0) * g.nKmax + im.b0 : nullptr;
    L.l1 = L.listed ? a.kv_tile + ((size_t)im.bh * g.nQ + min(im.qt0 + 1, g.nQ - 1)) * g.nKmax + im.b1 : nullptr;
    return L;
  };

  if (warp >= 8) {
  RF_SETMAXNREG_DEC();
  if (warp == kItemWarp) {
    // ------------------------------------------------------------ items: the own one, then those of CTAs not started yet
    if (lane == 0) {
      uint32_t x = blockIdx.x, y = blockIdx.y, asked = 0;
      bool more = true;
      // asks for another unit of work; false: there is none
      auto ask = [&]() -> bool {
        fence_proxy_async_smem();
        mbar_expect_tx(bar(C::B_CLC), 16);
        clc_request(base + C::ANSWER, bar(C::B_CLC));
        const bool ok = mbar_wait(bar(C::B_CLC), asked & 1, wc) && clc_answer(base + C::ANSWER, x, y);
        ++asked;
        return ok;
      };
      for (int i = 0;; ++i) {
        const int slot = i % kItemSlots;
        int* w = items + slot * kItemWords;
        if (i >= kItemSlots) mbar_wait(bar(C::B_IE + slot), ((i / kItemSlots) - 1) & 1, wc);
        int n0 = 0, n1 = 0;
        for (; more; more = ask()) {
          Unit un;
          place_unit((uint64_t)y * gridDim.x + x, a, un);
          const int bh = un.bh, qt0 = 2 * un.pair, qt1 = qt0 + 1;
          int cls = RF_DENSE, window = -1;
          if (a.head_class != nullptr) {
            cls = a.head_class[bh];
            if (cls < 0 || cls > 3) {
              rf_report(a.dev_status, RF_ERR_INVALID_ARG);
              cls = RF_DENSE;
            }
            if (a.head_window != nullptr) window = a.head_window[bh];
            n0 = a.count[(size_t)bh * g.nQ + qt0];
            n1 = qt1 < g.nQ ? a.count[(size_t)bh * g.nQ + qt1] : 0;
            // a schedule that was not built for this shape could hold any count: the checking build refuses to walk past a row
            if (!rf_in_bounds(n0, g.nKmax + 1, a.dev_status)) n0 = 0;
            if (!rf_in_bounds(n1, g.nKmax + 1, a.dev_status)) n1 = 0;
          } else {
            n0 = rf_cdiv(rf_kv_len(g, cls), BN);
            n1 = qt1 < g.nQ ? n0 : 0;
          }
          // Nothing is written for a pair whose lists are both empty (a schedule that the tile builder did not write).  It is
          // not published either: the TMA thread holds back the last V of the item before while it looks for the next tile,
          // so with two slots an empty item in between would wait for that V and keep it waiting.  (Below, a piece has at
          // least one entry of the longer list, so no published item is empty.)
          if (n0 == 0 && n1 == 0) continue;
          int b0 = 0, b1 = 0, k = 1;
          if (un.most > 1) {
            const int u = max(n0, n1);
            k = 4 * u > 5 * un.tiles ? min(rf_cdiv(u, un.tiles), un.most) : 1;   // up to a quarter more stays in one piece
            if (un.piece >= k) continue;
            b0 = n0 * un.piece / k;                                              // (at most 32 waves: the products are small)
            b1 = n1 * un.piece / k;
            n0 = n0 * (un.piece + 1) / k - b0;
            n1 = n1 * (un.piece + 1) / k - b1;
          }
          w[0] = bh; w[1] = qt0; w[2] = cls; w[3] = n0; w[4] = n1; w[5] = window; w[6] = b0; w[7] = b1;
          w[8] = k; w[9] = un.slot; w[10] = un.split; w[11] = un.piece;
          break;
        }
        if (!more) {
          w[0] = -1;
          rf_grid_trigger();
        }
        mbar_arrive(bar(C::B_IF + slot));
        if (!more) break;
        // not before the TMA warp has nearly worked the item off: an item taken early would wait here while other SMs idle
        more = mbar_wait_long(bar(C::B_REQ), i & 1, wc, n0 + n1) && ask();
      }
    }
  } else if (warp == kTmaWarp) {
    // ------------------------------------------------------------ TMA producer
    // The CTA's items are one sequence of tiles: the last tile's V of an item travels with the first K of the next one.
    if (lane == 0) {
      Item im;
      Lists L;
      Merge mg;
      int item = -1, tile = 0, ntile = 0, uses, listed = 0;   // listed: tiles of the item at most
      bool asked = true;
      const CUtensorMap *map_k = nullptr, *map_v = nullptr;
      // moves on to the next item; Q is fetched by the caller
      auto advance = [&](int& t) -> bool {
        if (!asked) mbar_arrive(bar(C::B_REQ));
        ++item;
        if (!take(item, im, listed)) return false;
        mbar_arrive(bar(C::B_IE + item % kItemSlots));
        asked = false;
        L = lists(im);
        mg.start(L);
        listed = im.n0 + im.n1;
        const bool perm = im.cls == RF_TEMPORAL && g.permute, tex = im.cls == RF_TEXTURAL;
        map_k = &maps.m[perm ? 4 : (tex ? 6 : 1)];
        map_v = &maps.m[perm ? 5 : (tex ? 7 : 2)];
        return mg.next(L, t, uses);      // (an item lists a tile)
      };
      auto load_q = [&]() {
        const CUtensorMap* map_q = &maps.m[im.cls == RF_TEMPORAL && g.permute ? 3 : 0];
        mbar_expect_tx(bar(C::B_Q), 2 * C::TILE);
#pragma unroll
        for (int j = 0; j < 2; ++j)
#pragma unroll
          for (int kb = 0; kb < KB; ++kb)
            tma_load_3d(base + C::Q + j * C::TILE + kb * C::BLK, map_q, kb * C::COL1, (im.qt0 + j) * BM, im.bh, bar(C::B_Q));
      };
      bool has = advance(tile);
      // A tile's record: which streams list it, whether it ends its item; 0 ends the sequence.  It is published with the
      // barrier its K is counted on, so the MMA thread walks no lists.
      auto record = [&](bool any) -> uint32_t { return any ? uses | kMore | (mg.left(L) == 0 ? kLast : 0u) : 0u; };
      records[C::NP] = record(has);
      if (!has) mbar_arrive(bar(C::B_K0));
      if (has) {
        load_q();
        mbar_expect_tx(bar(C::B_K0), C::TILE);
#pragma unroll
        for (int kb = 0; kb < KB; ++kb)
          tma_load_3d(base + C::K0 + kb * C::BLK, map_k, kb * C::COL1, tile * BN, im.bh, bar(C::B_K0));
      }
      int nq = 1;      // Q tiles loaded
      for (int u = 0; has; ++u) {
        if (!asked && mg.left(L) <= kAskAhead) {
          mbar_arrive(bar(C::B_REQ));
          asked = true;
        }
        const CUtensorMap* cur_v = map_v;
        const int cur_bh = im.bh;
        bool has_nxt = mg.next(L, ntile, uses), new_item = false;
        if (!has_nxt) has_nxt = new_item = advance(ntile);
        const int ps = u % C::NP, ksn = (u + 1) % C::NK;
        // pair u reuses the V slot of pair u - NP and the K slot that pair filled; the first tile's K slot
        // comes round at u = NK - 1
        if (u >= C::NP) mbar_wait(bar(C::B_E + ps), ((u / C::NP) - 1) & 1, wc);
        else if (has_nxt && ksn == 0) mbar_wait(bar(C::B_K0E), 0, wc);
        records[ps] = record(has_nxt);
        mbar_expect_tx(bar(C::B_F + ps), has_nxt ? C::VLOAD + C::TILE : C::VLOAD);
#pragma unroll
        for (int vb = 0; vb < D / C::VBOX; ++vb)
          tma_load_3d(base + C::V0 + ps * C::VTILE + vb * C::VBLK, cur_v, vb * C::VBOX, tile * BN, cur_bh, bar(C::B_F + ps));
        if (has_nxt) {
#pragma unroll
          for (int kb = 0; kb < KB; ++kb)
            tma_load_3d(base + C::K0 + ksn * C::TILE + kb * C::BLK, map_k, kb * C::COL1, ntile * BN, im.bh, bar(C::B_F + ps));
        }
        if (new_item) {
          mbar_wait(bar(C::B_QE), (nq - 1) & 1, wc);   // the item before has taken its last scores
          load_q();
          ++nq;
        }
        has = has_nxt;
        tile = ntile;
      }
    }
  } else if (warp == kMmaWarp) {
    // ------------------------------------------------------------ MMA issuer
    // elect.sync tells the compiler that one thread issues, which shortens what stands between two instructions: D = 96 /
    // 128 2 to 3 % faster (24 heads, 32 896 tokens, dense 11.92 -> 11.69 and 10.81 -> 10.54 ms).  At D = 64, where the
    // streams' distance from one another counts for more, the plain branch is the faster one (dense, 48 heads, 17 776
    // tokens: 5.09 against 5.44 ms).
    if (C::S_EARLY ? lane == 0 : elect_one()) {
      // Descriptors differ only in their 14-bit start-address field: keep the constant words in
      // registers and add the byte offset (>> 4) per k-step.
      constexpr uint32_t DESC_HI = (1024u >> 4) | (1u << 14) | (2u << 29);      // SBO 1024 B, version 1, 128B swizzle
      constexpr uint32_t DESC_HI_V = C::VBOX == 64 ? DESC_HI : (512u >> 4) | (1u << 14) | (4u << 29);   // SBO 512 B, 64B swizzle
      constexpr uint32_t LO_KMAJOR = 1u << 16;                                    // LBO field unused for K-major
      constexpr uint32_t LO_VMAJOR = (C::VBLK >> 4) << 16;                        // LBO = one block of columns
      auto desc = [](uint32_t lo) -> uint64_t { return ((uint64_t)DESC_HI << 32) | lo; };
      auto desc_v = [](uint32_t lo) -> uint64_t { return ((uint64_t)DESC_HI_V << 32) | lo; };
      const uint32_t q_lo = ((base + C::Q) >> 4) | LO_KMAJOR, k_lo = ((base + C::K0) >> 4) | LO_KMAJOR;
      const uint32_t v_lo = ((base + C::V0) >> 4) | LO_VMAJOR;
      auto issue_s = [&](int j, int ks) {
        uint32_t a0 = q_lo + j * (C::TILE >> 4);
        const uint32_t b0 = k_lo + ks * (C::TILE >> 4);
        asm volatile("" : "+r"(a0));   // the descriptors of Q are added up here, not kept in (spilled) registers
        // the accumulate flag is a compile-time constant: the issuing thread blocks on every MMA, so each
        // instruction between two of them is idle tensor time
        const uint32_t t_d = tmem_base + (j ? C::S_COL1 : C::S_COL0);
        mma_ss_c<false>(t_d, desc(a0), desc(b0), IDESC_S);
#pragma unroll
        for (int k = 1; k < D / 16; ++k)
          mma_ss_c<true>(t_d, desc(a0 + (C::koff(k) >> 4)), desc(b0 + (C::koff(k) >> 4)), IDESC_S);
        tc_commit(bar(C::B_SF + j));
      };
      // waits for the parts of P (par: the parity they are handed over with) and issues their share of O += P V
      auto issue_pv = [&](int j, int vs, uint32_t acc, uint32_t par) {
        const uint32_t b0 = v_lo + vs * (C::VTILE >> 4);
        const uint32_t t_p = tmem_base + (j ? C::P_COL1 : C::P_COL0), t_o = tmem_base + (j ? C::O_COL1 : C::O_COL0);
#pragma unroll
        for (int p = 0; p < C::PARTS; ++p) {
          mbar_wait(bar(C::B_PF + j * C::PARTS + p), par, wc);
          tc_fence_after();
#pragma unroll
          for (int k = C::cut(p) / 16; k < C::cut(p + 1) / 16; ++k) {
            if (k == 0) mma_ts(t_o, t_p, desc_v(b0), IDESC_PV, acc);
            else mma_ts_c<true>(t_o, t_p + k * 8, desc_v(b0 + k * (16 * C::VROW >> 4)), IDESC_PV);
          }
        }
        tc_commit(bar(C::B_OF + j));
      };
      // one bit per stream
      uint32_t pv_par = 0;               // parity of the P V bursts issued
      uint32_t s_par = 3;                // parity of the S tiles issued, less one
      // Until the columns of S_j may be written: where P lies elsewhere the stream has read its last scores (else its last P V,
      // issued before, says so), where S0 and S1 share columns the other stream has too.
      auto s_free = [&](int j) {
        if (C::S_EARLY) mbar_wait(bar(C::B_SE + j), (s_par >> j) & 1, wc);
        if (C::S_SHARED) mbar_wait(bar(C::B_SE + (j ^ 1)), (s_par >> (j ^ 1)) & 1, wc);
        if (C::S_EARLY || C::S_SHARED) tc_fence_after();
        s_par ^= 1u << j;
      };
      uint32_t acc = 0;                  // the stream's next P V adds to O (clear: it opens an item)
      uint32_t cur = 0, nq = 0;          // the current tile's record; Q tiles taken
      if (mbar_wait(bar(C::B_K0), 0, wc)) cur = records[C::NP];
      if (cur & kMore) {
        mbar_wait(bar(C::B_Q), 0, wc);
        ++nq;
        tc_fence_after();
        if (cur & 1) { s_free(0); issue_s(0, 0); }
        if (cur & 2) { s_free(1); issue_s(1, 0); }
        tc_commit(bar(C::B_K0E));
        if (cur & kLast) tc_commit(bar(C::B_QE));
      }
      for (int u = 0; cur & kMore; ++u) {
        const int vs = u % C::NV, ksn = (u + 1) % C::NK;
        // the TMA barrier first (V of this tile and K of the next): the data has normally landed long ago, and
        // checking here keeps it out of the gap between a stream's P arriving and its MMAs being issued
        if (!mbar_wait(bar(C::B_F + vs), (u / C::NP) & 1, wc)) break;   // abandoned: the record may never come
        const uint32_t nxt = records[vs];
        if (cur & kLast) {
          // An item ends.  Both P V go first, then the next item's first scores (its O is not written before the softmax
          // warps have read this item's: their P of the new item follows their reads).
#pragma unroll 1
          for (int j = 0; j < 2; ++j) {
            if (cur & (1 << j)) {
              issue_pv(j, vs, (acc >> j) & 1, (pv_par >> j) & 1);
              pv_par ^= 1u << j;
            }
          }
          acc = 0;
          if (nxt & kMore) {
            mbar_wait(bar(C::B_Q), nq & 1, wc);
            ++nq;
#pragma unroll 1
            for (int j = 0; j < 2; ++j) {
              if (nxt & (1 << j)) {
                s_free(j);
                tc_fence_after();
                issue_s(j, ksn);
              }
            }
          }
        } else if constexpr (C::S_EARLY) {
          // Per stream: the next tile's scores (S is free as soon as the softmax warps have read the current
          // one), then O += P V of the current tile.  Stream 1's next scores are thus only issued once stream 0
          // has delivered its P: the two streams settle half a tile apart and take turns at the MUFU unit
          // instead of sitting in their exponentials at the same time.
#pragma unroll
          for (int j = 0; j < 2; ++j) {
            if (nxt & (1 << j)) {
              s_free(j);
              issue_s(j, ksn);
            }
            if (cur & (1 << j)) {
              issue_pv(j, vs, (acc >> j) & 1, (pv_par >> j) & 1);
              acc |= 1u << j;
              pv_par ^= 1u << j;
            }
          }
        } else {
#pragma unroll
          for (int j = 0; j < 2; ++j) {
            if (cur & (1 << j)) {
              issue_pv(j, vs, (acc >> j) & 1, (pv_par >> j) & 1);
              acc |= 1u << j;
              pv_par ^= 1u << j;
            }
            if (nxt & (1 << j)) {
              s_free(j);
              issue_s(j, ksn);
            }
          }
        }
        if ((nxt & (kMore | kLast)) == (kMore | kLast)) tc_commit(bar(C::B_QE));   // the item's last scores are under way
        tc_commit(bar(C::B_E + vs));
        cur = nxt;
      }
    }
  }
  } else {
    RF_SETMAXNREG_INC();
    // ------------------------------------------------------------ softmax + epilogue, one thread per query row
    const int j = warp >> 2;                       // stream
    const int row_in_tile = tid & 127;
    const uint32_t lane_sel = (uint32_t)((warp & 3) * 32) << 16;
    const uint32_t t_s = tmem_base + lane_sel + (j ? C::S_COL1 : C::S_COL0);
    const uint32_t t_o = tmem_base + lane_sel + (j ? C::O_COL1 : C::O_COL0);
    const float sc = a.scale_log2;
    // this row's keep words of a PARTIAL tile, in the part of V's first block of ones that nothing reads
    uint4* keep = reinterpret_cast<uint4*>(base_ptr + C::V0 + C::VLOAD + C::vchunk(row_in_tile, 2 + j));
    uint32_t done = 0;         // tiles of this stream in the items before: the barriers' phases run on
    Item im;
    im.n0 = im.n1 = 0;
    // (a warp leaves as a whole: after an abandoned wait its lanes may differ in what they saw)
    for (int item = 0; __all_sync(0xffffffffu, take(item, im, im.n0 + im.n1)); ++item) {
    const int n = j == 0 ? im.n0 : im.n1;
    const int32_t* list = a.head_class != nullptr ? a.kv_tile + ((size_t)im.bh * g.nQ + min(im.qt0 + j, g.nQ - 1)) * g.nKmax : nullptr;
    const RowMask rmask = make_row_mask(g, im.cls, im.window, min((im.qt0 + j) * BM + row_in_tile, g.N - 1));
    float m_run = -INFINITY;   // running maximum, log2 domain (score * sc)
    float l_run = 0.f;         // sum of the weights as rounded to bf16, the ones P V multiplies: normalises O (the last tile's are in O's column D)
    float l_exact = 0.f;       // sum of the unrounded weights: the log-sum-exp (LSE only)

    const int begin = j == 0 ? im.b0 : im.b1, end = begin + n;
    bool opens = true;         // the stream's first tile of the item (or piece)
    for (int t = begin; t < end; ++t, ++done, opens = false) {
      const uint32_t entry = list != nullptr ? (uint32_t)list[t] : dense_entry(t, g.N);
      // The keep words of a PARTIAL tile do not depend on its scores: they are worked out before the wait for the
      // scores, where a stream spends a third of its time anyway, and wait in shared memory (four registers live
      // through the exponentials cost every tile 3 %).
      bool partial = (entry & RF_PARTIAL_BIT) != 0;
      if (partial) {
        uint32_t w[4];
        rmask.tile_bits((int)(entry & ~RF_PARTIAL_BIT) * BN, w);
        partial = __any_sync(0xffffffffu, (w[0] & w[1] & w[2] & w[3]) != 0xffffffffu);   // a warp's rows may keep it whole
        *keep = make_uint4(w[0], w[1], w[2], w[3]);
      }
      mbar_wait(bar(C::B_SF + j), done & 1, wc);
      tc_fence_after();
      uint32_t s[128];
      // the sum of the last tile's weights, whose P V (D = 96 / 128) these scores were issued after
      uint32_t l_tile;
      if constexpr (!C::S_EARLY) l_tile = tmem_ld1(t_o + D);
      load_scores(t_s, s);
      if constexpr (!C::S_EARLY) l_run = opens ? 0.f : l_run + __uint_as_float(l_tile);
      if constexpr (C::S_SHARED) {   // S is handed back at once: its columns are the other stream's too, or (D = 64) its own next scores'
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(bar(C::B_SE + j));
      }
      if (partial) mask_scores(keep, s);
      if constexpr (C::S_EARLY) {
        // The scores are gone from TMEM, so the exact row maximum comes first and the exponentials are
        // taken once; the running maximum is raised only when the tile exceeds it by kLazyRaise.
        float mx0 = -INFINITY, mx1 = -INFINITY;
#pragma unroll
        for (int c = 0; c < 128; c += 4) {
          mx0 = fmaxf(mx0, fmaxf(__uint_as_float(s[c]), __uint_as_float(s[c + 1])));
          mx1 = fmaxf(mx1, fmaxf(__uint_as_float(s[c + 2]), __uint_as_float(s[c + 3])));
        }
        const float m_tile = fmaxf(mx0, mx1) * sc;
        const bool raise = m_tile > m_run + kLazyRaise || (m_run == -INFINITY && m_tile > -INFINITY);
        const bool any_raise = __any_sync(0xffffffffu, raise);
        float alpha = 1.f;
        if (raise) {
          alpha = ex2(m_run - m_tile);   // 0 when m_run = -inf
          m_run = m_tile;
          l_run *= alpha;
          if (LSE) l_exact *= alpha;
        }
        // P V of the previous tile reads the P columns this tile is about to overwrite, and O may only be
        // rescaled once everything issued into it has landed.  The wait sits in front of the P store (the
        // exponentials of this tile run under the previous tile's P V); it also keeps this stream at most
        // one tile ahead of the MMA warp, which tracks the P barrier by phase parity.
        bool o_landed = opens;
        if (!opens && any_raise) {
          mbar_wait(bar(C::B_OF + j), (done - 1) & 1, wc);
          o_landed = true;
          rescale_o<D>(t_o, alpha);
        }
        const float m_use = m_run == -INFINITY ? 0.f : m_run;
        const float2 sc2 = make_float2(sc, sc), mneg = make_float2(-m_use, -m_use);
        float2 la = make_float2(0.f, 0.f);
        uint32_t pk[64];
        take_weights<0, BN, LSE>(s, pk, la, sc2, mneg);
        if (LSE) l_exact += la.x + la.y;
        if (!o_landed) mbar_wait(bar(C::B_OF + j), (done - 1) & 1, wc);
        tc_fence_after();
        l_tile = tmem_ld1(t_o + D);   // the sum of the last tile's weights; cleared for this tile's
        {
          const uint32_t t_p = tmem_base + lane_sel + (j ? C::P_COL1 : C::P_COL0);
          uint32_t(&p0)[32] = *reinterpret_cast<uint32_t(*)[32]>(&pk[0]);
          uint32_t(&p1)[32] = *reinterpret_cast<uint32_t(*)[32]>(&pk[32]);
          tmem_st32(t_p, p0);
          tmem_st32(t_p + 32, p1);
          tc_wait_ld();
          tmem_st1(t_o + D, 0u);
          tc_wait_st();
        }
        l_run = opens ? 0.f : l_run + __uint_as_float(l_tile) * alpha;
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(bar(C::B_PF + j));
        continue;
      }
      // The first kSpec weights are taken against the running maximum of the previous tiles while the tile's own
      // maximum is being found; only if it exceeds the running one by kRaise (a row's first tile, rare after it) is
      // the running maximum raised, O rescaled and the weights taken so far taken again.
      uint32_t pk[64];
      float2 la = make_float2(0.f, 0.f);
      const float2 sc2 = make_float2(sc, sc);
      float m_use = m_run == -INFINITY ? 0.f : m_run;
      take_weights<0, kSpec, LSE>(s, pk, la, sc2, make_float2(-m_use, -m_use));
      float mx0 = -INFINITY, mx1 = -INFINITY;
#pragma unroll
      for (int c = 0; c < 128; c += 4) {
        mx0 = fmaxf(mx0, fmaxf(__uint_as_float(s[c]), __uint_as_float(s[c + 1])));
        mx1 = fmaxf(mx1, fmaxf(__uint_as_float(s[c + 2]), __uint_as_float(s[c + 3])));
      }
      const float m_tile = fmaxf(mx0, mx1) * sc;
      if (__any_sync(0xffffffffu, m_tile > m_run + kRaise)) {
        float alpha = 1.f;
        if (m_tile > m_run + kRaiseMargin) {
          alpha = ex2(m_run - m_tile);   // 0 when m_run = -inf
          m_run = m_tile;
          l_run *= alpha;
          if (LSE) l_exact *= alpha;
        }
        if (!opens) {
          // O of the previous tiles must be complete before it is rescaled
          mbar_wait(bar(C::B_OF + j), (done - 1) & 1, wc);
          rescale_o_call<D>(t_o, alpha);
        }
        m_use = m_run == -INFINITY ? 0.f : m_run;
        la = make_float2(0.f, 0.f);
        take_weights<0, kSpec, LSE>(s, pk, la, sc2, make_float2(-m_use, -m_use));
      }
      const uint32_t t_p = tmem_base + lane_sel + (j ? C::P_COL1 : C::P_COL0);
      const float2 mneg = make_float2(-m_use, -m_use);
      static_assert(C::S_EARLY || C::PARTS == 2, "the first half is handed over under the exponentials of the second");
      take_weights<kSpec, 64, LSE>(s, pk, la, sc2, mneg);
      store_weights<0, 64>(t_p, pk);
      tmem_st1(t_o + D, 0u);     // the column of this tile's sum
      take_weights<64, 80, LSE>(s, pk, la, sc2, mneg);
      tc_wait_st();              // the store has had these exponentials' time
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(bar(C::B_PF + j * C::PARTS));
      take_weights<80, BN, LSE>(s, pk, la, sc2, mneg);
      store_weights<64, BN>(t_p, pk);
      tc_wait_st();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(bar(C::B_PF + j * C::PARTS + 1));
      if (LSE) l_exact += la.x + la.y;
    }

    if (n > 0) {
      mbar_wait(bar(C::B_OF + j), (done - 1) & 1, wc);
      tc_fence_after();
    }
    if (n > 0) {
      const uint32_t l_tile = tmem_ld1(t_o + D);
      tc_wait_ld();
      l_run += __uint_as_float(l_tile);
    }
    // the item's words are read again here: kept in registers they would be in the way of the scores
    const int* iw = items + (item % kItemSlots) * kItemWords;
    if (iw[8] > 1) {
      leave_piece<D, LSE>(a, iw, t_o, warp, lane, m_run, l_run, l_exact, n > 0);
    } else if (n > 0) {
      const Row row = output_row(a, iw, j, row_in_tile);
      const float inv = l_run > 0.f ? 1.f / l_run : 0.f;
#pragma unroll
      for (int c = 0; c < D / 32; ++c) {
        uint32_t v[32];
        tmem_ld32(t_o + c * 32, v);   // warp-collective: rows past N take part, they just do not store
        tc_wait_ld();
        if (row.inside) {
#pragma unroll
          for (int i = 0; i < 16; ++i) v[i] = pack_bf16(__uint_as_float(v[2 * i]) * inv, __uint_as_float(v[2 * i + 1]) * inv);
          store_columns(row.o + c * 4, v, row.o32);
        }
      }
      if (LSE && row.inside) a.lse[row.at] = (m_run + log2f(l_exact)) * 0.6931471805599453f;
    }
    tc_fence_before();   // O has been read: the next P hand-over lets it be overwritten
    __syncwarp();
    if (lane == 0) mbar_arrive(bar(C::B_IE + item % kItemSlots));
    }
  }

  tc_fence_before();
  __syncthreads();
  if (warp == kTmaWarp) {
    if (*abort_flag) __nanosleep(20000);  // let abandoned copies land before shared memory is released
    __syncwarp();
    tmem_dealloc(tmem_base, C::TMEM_COLS);
  }
}

template <int D, bool LSE>
rf_status launch(RfAttnArgs a, const CUtensorMap* maps, cudaStream_t st) {
  static bool configured[64] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return RF_ERR_CUDA;
  if (dev >= 0 && dev < 64 && !configured[dev]) {
    if (!rf_regs_ok(rf_attn_kernel<D, LSE>)) return RF_ERR_UNSUPPORTED;   // setmaxnreg.inc could never be granted
    if (cudaFuncSetAttribute(rf_attn_kernel<D, LSE>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Cfg<D>::ALLOC) != cudaSuccess)
      return RF_ERR_CUDA;
    configured[dev] = true;
  }
  Maps m;
  for (int i = 0; i < 8; ++i) m.m[i] = maps[i];
  const size_t kv_bytes = (size_t)a.g.N * D * 2 * sizeof(__nv_bfloat16);
  a.heads_l2 = (int)std::min<size_t>(std::max<size_t>(kL2Bytes / kv_bytes, 1), (size_t)a.g.B * a.g.H);
  // one CTA a unit of work; running CTAs take over what has not started
  const dim3 grid = a.sp.on ? dim3(a.sp.n_units) : dim3(rf_cdiv(a.g.nQ, 2), a.g.B * a.g.H);
  return rf_launch(rf_attn_kernel<D, LSE>, grid, kThreads, Cfg<D>::ALLOC, st, m, a) == cudaSuccess ? RF_OK : RF_ERR_CUDA;
}
template <int D>
rf_status launch(const RfAttnArgs& a, const CUtensorMap* maps, cudaStream_t st) {
  return a.lse != nullptr ? launch<D, true>(a, maps, st) : launch<D, false>(a, maps, st);
}

}  // namespace

// Self-test of the bounded-wait machinery every kernel here relies on: one warp waits on an mbarrier that
// nothing ever arrives at.  The wait must give up after limit_ns, raise the CTA's abort flag, report
// RF_ERR_TIMEOUT to *dev_status, let a second wait return at once, and the kernel must exit normally.
__global__ void rf_selftest_timeout_kernel(int32_t* dev_status, uint64_t limit_ns, int32_t* waits_returned) {
  __shared__ __align__(8) uint64_t barrier;
  __shared__ int abort_flag;
  const uint32_t bar = sm100::smem_u32(&barrier);
  if (threadIdx.x == 0) {
    sm100::mbar_init(bar, 1);
    abort_flag = 0;
    sm100::mbar_init_fence();
  }
  __syncthreads();
  sm100::WaitCtx wc{&abort_flag, dev_status, limit_ns};
  const bool first = sm100::mbar_wait(bar, 0, wc);    // runs out
  const bool second = sm100::mbar_wait(bar, 0, wc);   // returns at once: the CTA has given up
  if (threadIdx.x == 0) *waits_returned = (first ? 1 : 0) + (second ? 2 : 0) + (abort_flag ? 4 : 0);
}

rf_status rf_launch_selftest_timeout(int32_t* dev_status, uint64_t limit_ns, int32_t* waits_returned, cudaStream_t st) {
  rf_selftest_timeout_kernel<<<1, 32, 0, st>>>(dev_status, limit_ns, waits_returned);
  return cudaGetLastError() == cudaSuccess ? RF_OK : RF_ERR_CUDA;
}

rf_status rf_launch_attention(const RfAttnArgs& a, const CUtensorMap* maps, cudaStream_t st) {
  switch (a.g.D) {
    case 64: return launch<64>(a, maps, st);
    case 96: return launch<96>(a, maps, st);
    case 128: return launch<128>(a, maps, st);
  }
  return RF_ERR_UNSUPPORTED;
}
