// Block-mask / tile-schedule builder and the token reordering gathers.
//
// The pattern masks of Sec. 3.2 (Spatial: Eq. 3, Temporal, Textural: Eq. 4-5) are evaluated in
// closed form per tile: a tile's query slots and key slots each cover a contiguous range of
// frames (Spatial), of in-frame positions (Temporal in position-major order) or a cyclic range
// of positions (Temporal in original order), so "some pair kept" and "all pairs kept" reduce to
// distances between at most two intervals per side.
#include <algorithm>

#include "rf_decide.cuh"

namespace {

struct Iv { int lo, hi; };  // closed interval

// Positions (index mod S) covered by slots [a0, a1) of the original order: one or two intervals.
__device__ __forceinline__ int cyclic_intervals(int a0, int a1, int S, Iv out[2]) {
  if (a1 - a0 >= S) { out[0] = {0, S - 1}; return 1; }
  int s = a0 % S, e = (a1 - 1) % S;
  if (s <= e) { out[0] = {s, e}; return 1; }
  out[0] = {s, S - 1};
  out[1] = {0, e};
  return 2;
}

// 2-D in-frame window between two runs of consecutive positions A = [a0, a1] and B = [b0, b1] (row-major positions
// of a frame of width W): `any` - some pair (p in A, p' in B) has |dy| <= wy and |dx| <= wx; `all` - every pair has.
// A run of positions is up to three rectangles (a partial first row, whole rows, a partial last row); between two
// rectangles the smallest and largest |dy| and |dx| follow from the interval ends.
struct Rect { int y0, y1, x0, x1; };
__device__ __forceinline__ int run_rects(int p0, int p1, int W, Rect out[3]) {
  const int ya = p0 / W, xa = p0 - ya * W, yb = p1 / W, xb = p1 - yb * W;
  if (ya == yb) { out[0] = {ya, ya, xa, xb}; return 1; }
  int n = 0;
  out[n++] = {ya, ya, xa, W - 1};
  if (yb - ya > 1) out[n++] = {ya + 1, yb - 1, 0, W - 1};
  out[n++] = {yb, yb, 0, xb};
  return n;
}
__device__ void window2d(const Iv& A, const Iv& B, int W, int wy, int wx, bool& any, bool& all) {
  Rect ra[3], rb[3];
  const int na = run_rects(A.lo, A.hi, W, ra), nb = run_rects(B.lo, B.hi, W, rb);
  for (int i = 0; i < na; ++i)
    for (int j = 0; j < nb; ++j) {
      const int gy = max(max(rb[j].y0 - ra[i].y1, ra[i].y0 - rb[j].y1), 0), gx = max(max(rb[j].x0 - ra[i].x1, ra[i].x0 - rb[j].x1), 0);
      const int sy = max(ra[i].y1 - rb[j].y0, rb[j].y1 - ra[i].y0), sx = max(ra[i].x1 - rb[j].x0, rb[j].x1 - ra[i].x0);
      any = any || (gy <= wy && gx <= wx);
      all = all && (sy <= wy && sx <= wx);
    }
}

// 0: empty, 1: PARTIAL, 2: FULL.  Tile (a, b) of a head of class cls.
__device__ int tile_flag(const RfGeom& g, int cls, int a, int b) {
  const int Lkv = rf_kv_len(g, cls);
  const int r0 = a * g.BM, r1 = min(r0 + g.BM, g.N);
  const int u0 = b * g.BN, u1 = min(u0 + g.BN, Lkv);
  if (r0 >= r1 || u0 >= u1) return 0;
  const bool full_width = (b + 1) * g.BN <= Lkv;
  bool any = true, all = true;
  if (cls == RF_SPATIAL || cls == RF_TEMPORAL) {
    const int Nv = g.Nv;
    const bool text_row = r1 > Nv, text_col = u1 > Nv;
    const bool video_part = r0 < Nv && u0 < Nv;
    bool vv_any = false, vv_all = true;
    if (video_part) {
      const int rv1 = min(r1, Nv), uv1 = min(u1, Nv);
      if (cls == RF_TEMPORAL && g.t2d) {
        // 2-D in-frame window: the tile's query and key slots each cover one run of positions (position-major
        // order) or a run that may wrap round the frame's end (original order)
        Iv R[2], C[2];
        int nr, nc;
        if (g.permute) {
          R[0] = {r0 / g.T, (rv1 - 1) / g.T};
          C[0] = {u0 / g.T, (uv1 - 1) / g.T};
          nr = nc = 1;
        } else {
          nr = cyclic_intervals(r0, rv1, g.S, R);
          nc = cyclic_intervals(u0, uv1, g.S, C);
        }
        for (int i = 0; i < nr; ++i)
          for (int j = 0; j < nc; ++j) window2d(R[i], C[j], g.Wf, g.wy, g.wx, vv_any, vv_all);
      } else if (cls == RF_SPATIAL || g.permute) {
        // contiguous ranges of frames (Spatial) or of positions (position-major Temporal)
        const int unit = cls == RF_SPATIAL ? g.S : g.T;
        const int w = cls == RF_SPATIAL ? g.wf : g.ws;
        const int ra = r0 / unit, rb = (rv1 - 1) / unit, ca = u0 / unit, cb = (uv1 - 1) / unit;
        vv_any = max(max(ca - rb, ra - cb), 0) <= w;
        vv_all = max(rb - ca, cb - ra) <= w;
        if (cls == RF_SPATIAL && g.key_first) {
          // keys of frame 0 are kept for every query: the tile is non-empty if it reaches into frame 0, and all of
          // it is kept if the window holds for its keys of the other frames (if it has any)
          vv_any = vv_any || ca == 0;
          vv_all = cb == 0 || max(rb - max(ca, 1), cb - ra) <= w;
        }
      } else {
        Iv R[2], C[2];
        const int nr = cyclic_intervals(r0, rv1, g.S, R), nc = cyclic_intervals(u0, uv1, g.S, C);
        for (int i = 0; i < nr; ++i)
          for (int j = 0; j < nc; ++j) {
            vv_any = vv_any || max(max(C[j].lo - R[i].hi, R[i].lo - C[j].hi), 0) <= g.ws;
            vv_all = vv_all && max(R[i].hi - C[j].lo, C[j].hi - R[i].lo) <= g.ws;
          }
      }
    }
    any = text_row || text_col || vv_any;
    all = vv_all;
  }
  if (!any) return 0;
  return (all && full_width) ? 2 : 1;
}

// One warp per (query tile a, head): flags for 32 key tiles at a time, ordered compaction by ballot.
// No block-level synchronisation; eight rows per CTA.
struct TileArrays {
  int32_t* count;
  int32_t* kv_tile;
  uint32_t* bitmap;
  int32_t* kv_len;
};
__device__ __forceinline__ void build_row(RfGeom& g, int cls, int window, int a, int bh, int lane, const TileArrays& out, int32_t* dev_status) {
  if (cls == RF_SPATIAL && window >= 0) g.wf = min(window, g.T);     // dynamic bandwidth: this head's own window; past the
  if (cls == RF_TEMPORAL && window >= 0) g.ws = min(window, g.S);    // extent the mask is the same, and nothing overflows
  const int Lkv = rf_kv_len(g, cls);
  const int nK = rf_cdiv(Lkv, g.BN);
  if (a == 0 && lane == 0 && rf_in_bounds(bh, (size_t)g.B * g.H, dev_status)) out.kv_len[bh] = Lkv;
  int32_t* row = out.kv_tile + ((size_t)bh * g.nQ + a) * g.nKmax;
  const int words = rf_cdiv(g.nKmax, 32);
  uint32_t* brow = out.bitmap ? out.bitmap + ((size_t)bh * g.nQ + a) * words : nullptr;
  int base = 0;
  for (int b0 = 0; b0 < words * 32; b0 += 32) {
    const int b = b0 + lane;
    const int f = (b < nK) ? tile_flag(g, cls, a, b) : 0;
    const unsigned m = __ballot_sync(0xffffffffu, f != 0);
    if (brow && lane == 0 && rf_in_bounds(b0 >> 5, words, dev_status)) brow[b0 >> 5] = m;
    if (f != 0) {
      const int slot = base + __popc(m & ((1u << lane) - 1));
      if (rf_in_bounds(slot, g.nKmax, dev_status)) row[slot] = (int32_t)((uint32_t)b | (f == 1 ? RF_PARTIAL_BIT : 0u));
    }
    base += __popc(m);
  }
  if (lane == 0 && rf_in_bounds((size_t)bh * g.nQ + a, (size_t)g.B * g.H * g.nQ, dev_status)) out.count[(size_t)bh * g.nQ + a] = base;
}
__global__ void __launch_bounds__(256) rf_build_tiles_kernel(RfGeom g, const int32_t* head_class, const int32_t* head_window,
                                                              const TileArrays out, int32_t* dev_status) {
  const int lane = threadIdx.x & 31;
  const int a = blockIdx.x * 8 + (threadIdx.x >> 5), bh = blockIdx.y;
  rf_grid_trigger();
  rf_grid_wait();
  if (a >= g.nQ) return;   // whole warp
  int cls = head_class[bh];
  if (cls < 0 || cls > 3) {
    if (lane == 0) rf_report(dev_status, RF_ERR_INVALID_ARG);
    cls = RF_DENSE;
  }
  build_row(g, cls, head_window != nullptr ? head_window[bh] : -1, a, bh, lane, out, dev_status);
}

// Reordered copies for heads whose coordinate space is not the original one.
//   Temporal + permute: Q, K, V  -> slot pos*T + frame (text rows keep their index)
//   Textural:           K, V     -> frame*nC + rank(pos) for kept positions, text after T*nC
// A byte mover: what bounds it is how many 16-byte vectors are under way.  A thread moves its column of kGatherRows rows
// of two or three tensors, all loads before the first store; the CTAs of a head (grid.y) share its rows.  Temporal heads are
// walked in source order, Textural heads in the order of the kept rows: the k-th kept position of a frame follows in closed form
// (any tau consecutive frame rows keep W positions between them), so no thread visits a row that is not copied and no table has
// to be built first.  48 heads, 17 776 tokens, D = 64, all Textural: 133 -> 44 us (221 MB); 24 heads, 8448 tokens, D = 128,
// 8/8/8: 41 -> 25 us (139 MB).
constexpr int kGatherRows = 4;
struct Copies {
  const uint4 *q, *k, *v;
  uint4 *wq, *wk, *wv;
  int32_t* tickets;          // of the attention kernel: they start at zero
  int n_tickets;
};
__device__ __forceinline__ void clear_tickets(const Copies& io, int block, int blocks) {
  for (int i = block * 256 + threadIdx.x; i < io.n_tickets; i += blocks * 256) io.tickets[i] = 0;
}
// CTA `block` of the `blocks` that share head bh.
__device__ __forceinline__ void gather_rows(const RfGeom& g, int cls, int bh, int block, int blocks, const Copies& io, int32_t* dev_status) {
  const uint4 *q = io.q, *k = io.k, *v = io.v;
  uint4 *wq = io.wq, *wk = io.wk, *wv = io.wv;
  const bool perm = cls == RF_TEMPORAL && g.permute;
  const bool tex = cls == RF_TEXTURAL;
  if (!perm && !tex) return;
  const int vec = g.D / 8;  // uint4 per row
  const int rows_per_step = 256 / vec;
  const int lr = threadIdx.x / vec, c = threadIdx.x % vec;
  if (lr >= rows_per_step) return;
  const size_t head_off = (size_t)bh * g.N * vec + c;
  const int rows = perm ? g.N : g.LkvTex, video = perm ? g.Nv : g.T * g.nC;
  for (long long i0 = (long long)block * rows_per_step * kGatherRows + lr; i0 < rows;
       i0 += (long long)blocks * rows_per_step * kGatherRows) {
    int src[kGatherRows], dst[kGatherRows];
    bool on[kGatherRows];
#pragma unroll
    for (int r = 0; r < kGatherRows; ++r) {
      const long long at = i0 + r * rows_per_step;
      on[r] = at < rows;
      const int i = on[r] ? (int)at : 0;
      src[r] = dst[r] = i;
      if (i >= video) {
        src[r] = g.Nv + (i - video);
      } else if (perm) {
        const int f = i / g.S, p = i - f * g.S;
        dst[r] = p * g.T + f;
      } else {
        const int f = i / g.nC, rank = i - f * g.nC;
        const int band = rank / g.Wf;          // tau frame rows each
        int x = rank - band * g.Wf, y = 0;
        for (int kept; x >= (kept = y < g.Wf ? (g.Wf - y + g.tau - 1) / g.tau : 0); ++y) x -= kept;
        src[r] = f * g.S + (band * g.tau + y) * g.Wf + y + x * g.tau;
      }
      on[r] = on[r] && rf_in_bounds(dst[r], rows, dev_status);
    }
    uint4 tq[kGatherRows], tk[kGatherRows], tv[kGatherRows];
#pragma unroll
    for (int r = 0; r < kGatherRows; ++r) {
      if (!on[r]) continue;
      const size_t s = head_off + (size_t)src[r] * vec;
      if (perm) tq[r] = q[s];
      tk[r] = k[s];
      tv[r] = v[s];
    }
#pragma unroll
    for (int r = 0; r < kGatherRows; ++r) {
      if (!on[r]) continue;
      const size_t d = head_off + (size_t)dst[r] * vec;
      if (perm) wq[d] = tq[r];
      wk[d] = tk[r];
      wv[d] = tv[r];
    }
  }
}

__global__ void __launch_bounds__(256) rf_gather_kernel(RfGeom g, const int32_t* head_class, const Copies io, int32_t* dev_status) {
  rf_grid_trigger();
  rf_grid_wait();
  if (blockIdx.y == 0) clear_tickets(io, blockIdx.x, gridDim.x);
  gather_rows(g, head_class[blockIdx.y], blockIdx.y, blockIdx.x, gridDim.x, io, dev_status);
}

// Decision, schedule and copies in one launch: the first CTAs of a head build its tile lists, the others copy.  A warp's own
// decision costs it one round of loads (a few sums per recall); what it saves is two launches' hand-over, and the lists are
// built beside the copies, which wait for memory.
__global__ void __launch_bounds__(256) rf_prepare_kernel(RfGeom g, const RfDecision dec, const TileArrays out, const Copies io, int tile_blocks,
                                                          int32_t* dev_status) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, bh = blockIdx.y;
  const bool lists = (int)blockIdx.x < tile_blocks;
  rf_grid_trigger();
  rf_grid_wait();
  if (!lists && bh == 0) clear_tickets(io, blockIdx.x - tile_blocks, gridDim.x - tile_blocks);
  const int a = blockIdx.x * 8 + warp;
  if (lists && a >= g.nQ) return;   // whole warp
  const RfHead h = rf_decide(dec, bh, lane, lists && a == 0);
  if (lists) build_row(g, h.failed ? RF_DENSE : h.cls, h.window, a, bh, lane, out, dev_status);
  else gather_rows(g, h.cls, bh, blockIdx.x - tile_blocks, gridDim.x - tile_blocks, io, dev_status);
}

__global__ void __launch_bounds__(256) rf_zero_kernel(int32_t* words, int n) {
  rf_grid_trigger();
  rf_grid_wait();
  for (int i = blockIdx.x * 256 + threadIdx.x; i < n; i += gridDim.x * 256) words[i] = 0;
}

}  // namespace

cudaError_t rf_launch_zero(int32_t* words, int n, cudaStream_t st) {
  return rf_launch(rf_zero_kernel, dim3(rf_cdiv(n, 1024)), 256, 0, st, words, n);
}

cudaError_t rf_launch_build_tiles(const RfGeom& g, const int32_t* head_class, const int32_t* head_window, int32_t* count,
                                  int32_t* kv_tile, uint32_t* bitmap, int32_t* kv_len, int32_t* dev_status, cudaStream_t st) {
  return rf_launch(rf_build_tiles_kernel, dim3(rf_cdiv(g.nQ, 8), g.B * g.H), 256, 0, st, g, head_class, head_window,
                   TileArrays{count, kv_tile, bitmap, kv_len}, dev_status);
}

namespace {
int gather_blocks(const RfGeom& g) { return rf_cdiv(g.N, 256 / (g.D / 8) * kGatherRows); }
Copies copies(const __nv_bfloat16* q, const __nv_bfloat16* k, const __nv_bfloat16* v, __nv_bfloat16* wq, __nv_bfloat16* wk,
              __nv_bfloat16* wv, int32_t* tickets, int n_tickets) {
  return Copies{(const uint4*)q, (const uint4*)k, (const uint4*)v, (uint4*)wq, (uint4*)wk, (uint4*)wv, tickets, n_tickets};
}
}  // namespace

cudaError_t rf_launch_gather(const RfGeom& g, const int32_t* head_class, const __nv_bfloat16* q,
                             const __nv_bfloat16* k, const __nv_bfloat16* v, __nv_bfloat16* wq, __nv_bfloat16* wk,
                             __nv_bfloat16* wv, int32_t* tickets, int n_tickets, int32_t* dev_status, cudaStream_t st) {
  return rf_launch(rf_gather_kernel, dim3(gather_blocks(g), g.B * g.H), 256, 0, st, g, head_class,
                   copies(q, k, v, wq, wk, wv, tickets, n_tickets), dev_status);
}

cudaError_t rf_launch_prepare(const RfGeom& g, const RfDecision& dec, int32_t* count, int32_t* kv_tile, uint32_t* bitmap,
                              int32_t* kv_len, const __nv_bfloat16* q, const __nv_bfloat16* k, const __nv_bfloat16* v,
                              __nv_bfloat16* wq, __nv_bfloat16* wk, __nv_bfloat16* wv, int32_t* tickets, int n_tickets,
                              int32_t* dev_status, cudaStream_t st) {
  const int heads = g.B * g.H, tile_blocks = rf_cdiv(g.nQ, 8);
  // A head's copying CTAs are fixed before its class is known; those of a head that copies nothing leave at once.  Two CTAs share an
  // SM (registers).  Three CTAs an SM over all heads at least, so that each pays for its decision once and walks on (24 heads, 8448
  // tokens, D = 128: 508 us a call, 517 with one CTA per step), and up to four times as many while each still has four steps,
  // so that a few reordered heads of many spread over the SMs too.  us a call without and with the second half of the rule: 48 heads, 17 776
  // tokens, D = 64, all reordered 1396 and 1378, one 1621 and 1615; 24 heads, 8448 tokens, D = 128, all 327 and 322, eight 368 and
  // 363.  Calls of few steps keep their share: more CTAs cost them 1 to 3 % (24 heads, 2457 tokens, D = 96: 71.9, with twice as many 74.1).
  // Three CTAs to an SM (80 registers) gained 1 % in some calls and lost as much in others (3 heads, 7476 tokens, D = 96: 113.5 and
  // 115.6).
  const int share = rf_cdiv(148 * 3, heads), steps = gather_blocks(g);
  const int blocks = std::min(steps, std::max(share, std::min(rf_cdiv(steps, 4), 4 * share)));
  return rf_launch(rf_prepare_kernel, dim3(tile_blocks + blocks, heads), 256, 0, st, g, dec, TileArrays{count, kv_tile, bitmap, kv_len},
                   copies(q, k, v, wq, wk, wv, tickets, n_tickets), tile_blocks, dev_status);
}
