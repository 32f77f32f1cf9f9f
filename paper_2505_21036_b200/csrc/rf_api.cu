// C ABI of the RainFusion CUDA path: argument validation, workspace layout, tensor-map encoding.
#include <algorithm>
#include <math.h>
#include <string.h>

#include "rf_common.cuh"

namespace {

constexpr size_t kAlign = 256;
inline size_t align_up(size_t x) { return (x + kAlign - 1) / kAlign * kAlign; }
inline bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }
inline bool pow2(int x) { return x > 0 && (x & (x - 1)) == 0; }

// The kernels pack a frame row and column into one word for the 2-D Temporal window.
rf_status check_2d(const rf_shape* s, const rf_params* p) {
  if (p->temporal_window_2d == 1 && (s->frame_h >= 32768 || s->frame_w >= 32768)) return RF_ERR_UNSUPPORTED;
  return RF_OK;
}

rf_status check_shape(const rf_shape* s) {
  if (s == nullptr) return RF_ERR_INVALID_ARG;
  if (s->B < 1 || s->H < 1 || s->T < 1 || s->frame_h < 1 || s->frame_w < 1 || s->L_text < 0) return RF_ERR_INVALID_ARG;
  if (s->D < 8 || s->D % 8 != 0) return RF_ERR_INVALID_ARG;
  const long long n = (long long)s->T * s->frame_h * s->frame_w + s->L_text;
  if (n > (1ll << 30) || (long long)s->B * s->H > 65535) return RF_ERR_UNSUPPORTED;
  return RF_OK;
}

rf_status check_params(const rf_params* p) {
  if (p == nullptr) return RF_ERR_INVALID_ARG;
  if (p->frame_window < 0 || p->spatial_window < 0 || p->textural_stride < 1 || p->sample_stride < 1)
    return RF_ERR_INVALID_ARG;
  if (p->sample_mode != RF_SAMPLE_ALG1 && p->sample_mode != RF_SAMPLE_GLOBAL) return RF_ERR_INVALID_ARG;
  if (!(p->alpha > 0.f && p->alpha <= 1.f)) return RF_ERR_INVALID_ARG;
  if (!pow2(p->block_m) || !pow2(p->block_n) || p->block_m < 16 || p->block_n < 16) return RF_ERR_INVALID_ARG;
  if (p->temporal_permute != 0 && p->temporal_permute != 1) return RF_ERR_INVALID_ARG;
  if (p->two_mask != 0 && p->two_mask != 1) return RF_ERR_INVALID_ARG;
  if (p->spatial_key_first_frame != 0 && p->spatial_key_first_frame != 1) return RF_ERR_INVALID_ARG;
  if (p->temporal_window_2d != 0 && p->temporal_window_2d != 1) return RF_ERR_INVALID_ARG;
  if (p->temporal_window_2d == 1 && (p->temporal_window_y < 0 || p->temporal_window_x < 0)) return RF_ERR_INVALID_ARG;
  return RF_OK;
}

// Kept tokens per frame of the checkerboard set C (Eq. 4).
int checkerboard_count(int Hf, int Wf, int tau) {
  int n = 0;
  for (int r = 0; r < tau; ++r) {
    const int rows = r < Hf ? (Hf - r + tau - 1) / tau : 0;
    const int cols = r < Wf ? (Wf - r + tau - 1) / tau : 0;
    n += rows * cols;
  }
  return n;
}

RfGeom make_geom(const rf_shape* s, int wf, int ws, int tau, int bm, int bn, int permute) {
  RfGeom g;
  g.B = s->B; g.H = s->H; g.D = s->D;
  g.T = s->T; g.Hf = s->frame_h; g.Wf = s->frame_w; g.S = s->frame_h * s->frame_w;
  g.Nv = g.T * g.S; g.L = s->L_text; g.N = g.Nv + g.L;
  // Windows past the extent and strides past the frame's longer side give the same masks as the extent itself
  // (every frame / position within reach; y mod tau = y and x mod tau = x); clamping keeps the kernels' index
  // arithmetic ((f + w_f + 1) * S, p + w_s, loops over tau) inside int range for any caller value.
  g.wf = wf < g.T ? wf : g.T;
  g.ws = ws < g.S ? ws : g.S;
  g.tau = tau < (g.Hf > g.Wf ? g.Hf : g.Wf) ? tau : (g.Hf > g.Wf ? g.Hf : g.Wf);
  tau = g.tau;
  g.nC = checkerboard_count(g.Hf, g.Wf, tau);
  g.LkvTex = g.T * g.nC + g.L;
  g.BM = bm; g.BN = bn;
  g.nQ = rf_cdiv(g.N, bm);
  g.nKmax = rf_cdiv(g.N, bn);
  g.permute = permute;
  g.two_mask = 0;
  g.key_first = 0;
  g.t2d = g.wy = g.wx = 0;
  return g;
}
RfGeom make_geom(const rf_shape* s, const rf_params* p) {
  RfGeom g = make_geom(s, p->frame_window, p->spatial_window, p->textural_stride, p->block_m, p->block_n, p->temporal_permute);
  g.two_mask = p->two_mask;
  g.key_first = p->spatial_key_first_frame;
  g.t2d = p->temporal_window_2d;
  g.wy = g.t2d ? (p->temporal_window_y < g.Hf ? p->temporal_window_y : g.Hf) : 0;   // past the frame: same mask
  g.wx = g.t2d ? (p->temporal_window_x < g.Wf ? p->temporal_window_x : g.Wf) : 0;
  return g;
}

size_t tensor_bytes(const RfGeom& g) { return align_up((size_t)g.B * g.H * g.N * g.D * sizeof(__nv_bfloat16)); }

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                                  const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn() {
  static EncodeTiledFn fn = nullptr;
  if (fn == nullptr) {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult qres;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &qres) != cudaSuccess ||
        qres != cudaDriverEntryPointSuccess)
      return nullptr;
    fn = reinterpret_cast<EncodeTiledFn>(p);
  }
  return fn;
}

// bf16 [heads][rows (stride head_rows)][D] viewed as a 3-D tensor, box = 64 columns x 128 rows, 128B swizzle.
bool encode_map(CUtensorMap* m, const void* ptr, int D, int rows, int head_rows, int heads) {
  return rf_encode_rows_map(m, ptr, D, rows, (size_t)D * 2, (size_t)head_rows * D * 2, heads);
}
// The same for V: at D = 96 in boxes of 32 columns.
bool encode_v_map(CUtensorMap* m, const void* ptr, int D, int rows, int head_rows, int heads) {
  return rf_encode_rows_map(m, ptr, D, rows, (size_t)D * 2, (size_t)head_rows * D * 2, heads, D == 96 ? 32 : 64);
}

// The workspace: the reordered copies of Q, K and V, the pieces of split items, ARM's scratch.  The offsets depend on the
// shape alone, so that calls whose other parameters differ find the same things in the same places.
size_t split_offset(const RfGeom& g) { return 3 * tensor_bytes(g); }
size_t arm_offset(const RfGeom& g) { return split_offset(g) + rf_split_bytes(rf_split_plan(g, true, g.B * g.H, 0), g.D); }
size_t arm_bytes(const RfGeom& g, const rf_params* p) {
  return align_up(rf_arm_scratch_floats(g, p->sample_stride, RF_MAX_BANDWIDTHS) * sizeof(float));
}
// The pieces are no necessity: a block that lacks the room for them (one sized for a larger shape that needs none, say) does
// for the copies and ARM's scratch, and the items stay whole.
size_t least_bytes(const RfGeom& g, const rf_params* p) { return 3 * tensor_bytes(g) + arm_bytes(g, p); }
float* arm_scratch(const RfGeom& g, const rf_params* p, void* ws, size_t ws_bytes) {
  const size_t at = ws_bytes >= arm_offset(g) + arm_bytes(g, p) ? arm_offset(g) : split_offset(g);
  return reinterpret_cast<float*>(static_cast<uint8_t*>(ws) + at);
}
void set_split(RfAttnArgs* a, const RfSplit& sp, uint8_t* at) {
  a->sp = sp;
  a->tickets = sp.on ? reinterpret_cast<int32_t*>(at) : nullptr;
  a->pieces = sp.on ? reinterpret_cast<float*>(at + rf_split_ticket_bytes(sp)) : nullptr;
}

rf_status check_attn_shape(const rf_shape* s) {
  rf_status st = check_shape(s);
  if (st != RF_OK) return st;
  if (s->D != 64 && s->D != 96 && s->D != 128) return RF_ERR_UNSUPPORTED;
  return RF_OK;
}

}  // namespace

bool rf_encode_rows_map(CUtensorMap* m, const void* ptr, int D, int rows, size_t row_stride_bytes,
                        size_t head_stride_bytes, int heads, int box_columns) {
  EncodeTiledFn fn = encode_fn();
  if (fn == nullptr) return false;
  cuuint64_t dims[3] = {(cuuint64_t)D, (cuuint64_t)rows, (cuuint64_t)heads};
  cuuint64_t strides[2] = {(cuuint64_t)row_stride_bytes, (cuuint64_t)head_stride_bytes};
  cuuint32_t box[3] = {(cuuint32_t)box_columns, 128, 1};
  cuuint32_t estr[3] = {1, 1, 1};
  return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(ptr), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, box_columns == 64 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

rf_status rf_checked_geom(const rf_shape* shape, const rf_params* params, RfGeom* out) {
  rf_status st = check_shape(shape);
  if (st != RF_OK) return st;
  st = check_params(params);
  if (st != RF_OK) return st;
  st = check_2d(shape, params);
  if (st != RF_OK) return st;
  *out = make_geom(shape, params);
  return RF_OK;
}

namespace {
// What the host can see wrong with the arguments of a sparse attention call.
rf_status check_sparse_attn(const rf_shape* shape, const rf_params* params, const void* q, const void* k, const void* v,
                            const int32_t* head_class, const int32_t* head_window, const rf_schedule* sched, const void* o,
                            const void* ws, size_t ws_bytes) {
  rf_status st = check_attn_shape(shape);
  if (st != RF_OK) return st;
  st = check_params(params);
  if (st != RF_OK) return st;
  st = check_2d(shape, params);
  if (st != RF_OK) return st;
  if (params->block_m != 128 || params->block_n != 128) return RF_ERR_UNSUPPORTED;
  if (q == nullptr || k == nullptr || v == nullptr || o == nullptr || head_class == nullptr || sched == nullptr ||
      sched->count == nullptr || sched->kv_tile == nullptr || ws == nullptr)
    return RF_ERR_INVALID_ARG;
  if (!aligned16(q) || !aligned16(k) || !aligned16(v) || !aligned16(o) ||
      (reinterpret_cast<uintptr_t>(ws) & (kAlign - 1)) != 0)
    return RF_ERR_INVALID_ARG;
  if (head_window != nullptr && params->temporal_window_2d) return RF_ERR_UNSUPPORTED;
  const RfGeom g = make_geom(shape, params);
  if (ws_bytes < least_bytes(g, params)) return RF_ERR_WORKSPACE_TOO_SMALL;
  return sched->nQ == g.nQ && sched->nKmax == g.nKmax ? RF_OK : RF_ERR_INVALID_ARG;
}

// Where the copies of a sparse attention call come from: made by it, left in the workspace by rf_reorder_tokens, or made in one
// launch with the decision over the classes and the tile schedule.
enum class Copies { kMake, kMade, kPrepare };
// Shared by rf_sparse_attn_fwd(_plus), rf_sparse_attn_reordered and rf_sparse_call.
rf_status sparse_attn_impl(const rf_shape* shape, const rf_params* params, const void* q, const void* k, const void* v,
                           const int32_t* head_class, const int32_t* head_window, const rf_schedule* sched, void* o,
                           float* lse, void* ws, size_t ws_bytes, int32_t* dev_status, void* cuda_stream, Copies from,
                           int heads_total, int head0, const RfDecision* dec = nullptr) {
  const rf_status st = check_sparse_attn(shape, params, q, k, v, head_class, head_window, sched, o, ws, ws_bytes);
  if (st != RF_OK) return st;
  const RfGeom g = make_geom(shape, params);
  cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);

  uint8_t* w = static_cast<uint8_t*>(ws);
  __nv_bfloat16* wq = reinterpret_cast<__nv_bfloat16*>(w);
  __nv_bfloat16* wk = reinterpret_cast<__nv_bfloat16*>(w + tensor_bytes(g));
  __nv_bfloat16* wv = reinterpret_cast<__nv_bfloat16*>(w + 2 * tensor_bytes(g));

  CUtensorMap maps[RF_ATTN_MAPS];
  const int heads = g.B * g.H;
  bool ok = encode_map(&maps[0], q, g.D, g.N, g.N, heads) && encode_map(&maps[1], k, g.D, g.N, g.N, heads) &&
            encode_v_map(&maps[2], v, g.D, g.N, g.N, heads) && encode_map(&maps[3], wq, g.D, g.N, g.N, heads) &&
            encode_map(&maps[4], wk, g.D, g.N, g.N, heads) && encode_v_map(&maps[5], wv, g.D, g.N, g.N, heads) &&
            encode_map(&maps[6], wk, g.D, g.LkvTex, g.N, heads) && encode_v_map(&maps[7], wv, g.D, g.LkvTex, g.N, heads);
  if (!ok) return RF_ERR_CUDA;

  RfAttnArgs a;
  const bool room = ws_bytes >= rf_group_workspace_bytes(shape, params, heads_total, head0);
  set_split(&a, room ? rf_split_plan(g, true, heads_total, head0) : RfSplit{}, w + split_offset(g));
  bool clear = a.sp.on;   // whatever ran on this workspace before, the tickets begin at zero
  if (from == Copies::kPrepare) {
    // a group's tickets may lie where ARM's sums do (its pieces were not part of the workspace's layout)
    const uintptr_t t0 = reinterpret_cast<uintptr_t>(a.tickets), t1 = t0 + a.sp.n_tickets * sizeof(int32_t);
    const bool apart = t1 <= reinterpret_cast<uintptr_t>(dec->glb) || t0 > reinterpret_cast<uintptr_t>(dec->arm_flag);
    cudaError_t e = rf_launch_prepare(g, *dec, sched->count, sched->kv_tile, sched->bitmap, sched->kv_len,
                                      static_cast<const __nv_bfloat16*>(q), static_cast<const __nv_bfloat16*>(k),
                                      static_cast<const __nv_bfloat16*>(v), wq, wk, wv, a.tickets, clear && apart ? (int)a.sp.n_tickets : 0,
                                      dev_status, stream);
    if (e != cudaSuccess) return RF_ERR_CUDA;
    clear = clear && !apart;
  } else if (from == Copies::kMake) {
    cudaError_t e = rf_launch_gather(g, head_class, static_cast<const __nv_bfloat16*>(q),
                                     static_cast<const __nv_bfloat16*>(k), static_cast<const __nv_bfloat16*>(v), wq, wk, wv,
                                     a.tickets, (int)a.sp.n_tickets, dev_status, stream);
    if (e != cudaSuccess) return RF_ERR_CUDA;
    clear = false;
  }
  if (clear && rf_launch_zero(a.tickets, (int)a.sp.n_tickets, stream) != cudaSuccess) return RF_ERR_CUDA;

  a.g = g;
  a.head_class = head_class;
  a.head_window = head_window;
  a.count = sched->count;
  a.kv_tile = sched->kv_tile;
  a.o = static_cast<__nv_bfloat16*>(o);
  a.lse = lse;
  a.dev_status = dev_status;
  a.scale_log2 = 1.4426950408889634f / sqrtf((float)g.D);
  return rf_launch_attention(a, maps, stream);
}
}  // namespace

// ------------------------------------------------------------------------------------------------
// The plan of split items (see RfSplit).  Costs are counted in tiles of an item (about 2 us): a unit of work costs its
// tiles and kUnit more, joining pieces kJoin, and a piece kPiece (its O through the L2 twice, over all SMs).  Leaving a
// piece takes 5 to 7 us against 2 to 3 for writing O out, so a piece needs tiles enough to pay for it: four where SMs
// would otherwise stay idle, more in a call of more items than SMs, whose last wave is not empty to begin with (masked
// calls most, as their items' lengths differ and fill each other's gaps).  Measured, whole calls: 27 items of 9 tiles (3
// heads, 2146 tokens, D = 96) 56.8 -> 48.0 us; 42 items of 14 230 -> 203; 205 items of 41 321 -> 273; 360 dense items of 30
// 183 -> 173; with pieces of 4 tiles 192 items of 12 became slower (83 -> 91), with text rows' pairs alone split 84 items
// of 7 too (99 -> 102).
// ------------------------------------------------------------------------------------------------
RfSplit rf_split_plan(const RfGeom& g, bool sparse, int heads_total, int head0) {
  constexpr int W = 148;                                // SMs, one CTA each
  constexpr long long kMostWaves = 32, kMostSlots = 384;
  constexpr double kUnit = 2.5, kJoin = 2.0, kPiece = 0.02;
  RfSplit sp = {};
  const int heads = g.B * g.H;
  const int nK = rf_cdiv(g.N, 128), pairs = rf_cdiv(rf_cdiv(g.N, 128), 2);
  const long long items = (long long)heads_total * pairs;
  if (items > kMostWaves * W) return sp;
  const int least = items < W ? 4 : (sparse ? 16 : 8);  // tiles a piece has at least
  const int usual = sparse ? (nK + 1) / 2 : nK;         // tiles an item lists: the patterns keep about half
  sp.text_pairs = sparse ? pairs - g.Nv / 256 : 0;
  const long long tail = std::min(items % W, (long long)heads_total * (pairs - sp.text_pairs));
  sp.kr = 1;
  double best = 1e30;
  for (int k = 1; k <= 8 && tail > 0; ++k) {
    if (k > 1 && (usual < least * k || tail * k > kMostSlots)) break;
    const double cost = (double)((tail * k + W - 1) / W) * ((double)usual / k + kUnit) + (k > 1 ? kJoin + kPiece * tail * k : 0.0);
    if (cost < best) { best = cost; sp.kr = k; }
  }
  sp.lr = rf_cdiv(usual, sp.kr);
  sp.kt = 1;
  sp.lt = items < W ? sp.lr : usual;
  const long long text = (long long)heads_total * sp.text_pairs;
  if (sp.kr == 1) return RfSplit{};
  if (text > 0 && items < 3 * W && text * rf_cdiv(nK, sp.lt) + tail * sp.kr <= kMostSlots) sp.kt = rf_cdiv(nK, sp.lt);
  sp.on = 1;
  if (sp.kt == 1) sp.text_pairs = 0;
  // the items of this group of heads
  const long long t0 = (long long)heads_total * (pairs - sp.text_pairs) - tail;
  sp.row0 = (int)(t0 / heads_total);
  sp.head_row0 = (int)std::min<long long>(std::max<long long>(t0 % heads_total - head0, 0), heads);
  sp.n_text = (uint32_t)(heads * sp.text_pairs * sp.kt);
  sp.first_tail = (uint32_t)(sp.row0 * heads + sp.head_row0);
  const uint32_t n_tail = (uint32_t)(heads * (pairs - sp.text_pairs)) - sp.first_tail;
  sp.n_units = sp.n_text + sp.first_tail + n_tail * sp.kr;
  sp.n_slots = (sp.kt > 1 ? sp.n_text : 0) + n_tail * sp.kr;
  sp.n_tickets = 8 * ((sp.kt > 1 ? heads * sp.text_pairs : 0) + n_tail);
  return sp;
}
size_t rf_split_ticket_bytes(const RfSplit& sp) { return align_up(sp.n_tickets * sizeof(int32_t)); }
size_t rf_split_bytes(const RfSplit& sp, int D) {
  return sp.on ? rf_split_ticket_bytes(sp) + align_up((size_t)sp.n_slots * 2 * 128 * (D + 4) * sizeof(float)) : 0;
}

size_t rf_group_workspace_bytes(const rf_shape* shape, const rf_params* params, int heads_total, int head0) {
  if (check_shape(shape) != RF_OK || check_params(params) != RF_OK) return 0;
  const RfGeom g = make_geom(shape, params);
  // (a group's pieces may reach into ARM's scratch, which is done with by then)
  return std::max(arm_offset(g) + arm_bytes(g, params), split_offset(g) + rf_split_bytes(rf_split_plan(g, true, heads_total, head0), g.D));
}

size_t rf_least_workspace_bytes(const rf_shape* shape, const rf_params* params) {
  return check_shape(shape) == RF_OK && check_params(params) == RF_OK ? least_bytes(make_geom(shape, params), params) : 0;
}

namespace {
rf_status check_arm(const rf_shape* shape, const rf_params* params, bool plus) {
  rf_status st = check_shape(shape);
  if (st != RF_OK) return st;
  st = check_params(params);
  if (st != RF_OK) return st;
  st = check_2d(shape, params);
  if (st != RF_OK) return st;
  if (shape->D != 64 && shape->D != 96 && shape->D != 128) return RF_ERR_UNSUPPORTED;
  return plus && params->temporal_window_2d ? RF_ERR_UNSUPPORTED : RF_OK;   // a bandwidth has no 2-D meaning defined here
}

// ARM with the fixed windows (n_bandwidths = 0) or candidate bandwidths; later: see rf_launch_arm.
rf_status arm_call(const rf_shape* shape, const rf_params* params, const float* bandwidths, int32_t n_bandwidths, const void* q,
                   const void* k, int32_t* head_class, int32_t* head_window, float* recall, void* ws, size_t ws_bytes,
                   int32_t* dev_status, void* cuda_stream, RfDecision* later = nullptr, bool selftest_abandon = false) {
  const bool plus = n_bandwidths != 0;
  const rf_status st = check_arm(shape, params, plus);
  if (st != RF_OK) return st;
  if (plus && (bandwidths == nullptr || n_bandwidths < 1 || n_bandwidths > RF_MAX_BANDWIDTHS)) return RF_ERR_INVALID_ARG;
  if (q == nullptr || k == nullptr || head_class == nullptr || (plus && head_window == nullptr) || ws == nullptr) return RF_ERR_INVALID_ARG;
  if (!aligned16(q) || !aligned16(k) || (reinterpret_cast<uintptr_t>(ws) & (kAlign - 1)) != 0) return RF_ERR_INVALID_ARG;
  const RfGeom g = make_geom(shape, params);
  if (ws_bytes < least_bytes(g, params)) return RF_ERR_WORKSPACE_TOO_SMALL;
  int ws_list[RF_MAX_BANDWIDTHS] = {g.ws}, wf_list[RF_MAX_BANDWIDTHS] = {g.wf};
  for (int i = 0; i < n_bandwidths; ++i) {
    const float b = bandwidths[i];
    if (!(b > 0.f && b <= 1.f) || (i > 0 && b <= bandwidths[i - 1])) return RF_ERR_INVALID_ARG;
    wf_list[i] = (int)floor((double)b * g.T);
    ws_list[i] = (int)floor((double)b * g.S);
  }
  float* scratch = arm_scratch(g, params, ws, ws_bytes);
  cudaError_t e = rf_launch_arm(g, params->sample_mode, params->sample_stride, params->alpha, plus ? n_bandwidths : 1, ws_list, wf_list,
                                static_cast<const __nv_bfloat16*>(q), static_cast<const __nv_bfloat16*>(k), head_class,
                                plus ? head_window : nullptr, plus ? nullptr : recall, plus ? recall : nullptr, scratch, dev_status,
                                static_cast<cudaStream_t>(cuda_stream), selftest_abandon, later);
  return e == cudaSuccess ? RF_OK : RF_ERR_CUDA;
}
}  // namespace

rf_status rf_sparse_call_group(const rf_shape* shape, const rf_params* params, const float* bandwidths, int32_t n_bandwidths,
                               const void* q, const void* k, const void* v, int32_t* head_class, int32_t* head_window,
                               rf_schedule* sched, void* o, float* lse, void* ws, size_t ws_bytes, int32_t* dev_status,
                               void* cuda_stream, int heads_total, int head0, bool selftest_abandon) {
  if (n_bandwidths < 0) return RF_ERR_INVALID_ARG;
  if (n_bandwidths == 0) head_window = nullptr;
  // ARM checks its own arguments before it launches; what the steps after it would refuse is refused here
  rf_status st = check_sparse_attn(shape, params, q, k, v, head_class, head_window, sched, o, ws, ws_bytes);
  if (st == RF_OK && sched->kv_len == nullptr) st = RF_ERR_INVALID_ARG;
  if (st != RF_OK) return st;
  RfDecision dec;
  st = arm_call(shape, params, bandwidths, n_bandwidths, q, k, head_class, head_window, nullptr, ws, ws_bytes, dev_status, cuda_stream, &dec,
                selftest_abandon);
  if (st != RF_OK) return st;
  return sparse_attn_impl(shape, params, q, k, v, head_class, head_window, sched, o, lse, ws, ws_bytes, dev_status, cuda_stream,
                          Copies::kPrepare, heads_total, head0, &dec);
}

extern "C" {

int32_t rf_bounds_checked(void) {
#ifdef RF_BOUNDS_CHECK
  return 1;
#else
  return 0;
#endif
}

const char* rf_status_string(rf_status s) {
  switch (s) {
    case RF_OK: return "ok";
    case RF_ERR_INVALID_ARG: return "invalid argument";
    case RF_ERR_UNSUPPORTED: return "unsupported shape or parameter";
    case RF_ERR_WORKSPACE_TOO_SMALL: return "workspace too small";
    case RF_ERR_CUDA: return "CUDA error";
    case RF_ERR_TIMEOUT: return "device-side wait timed out";
    case RF_ERR_STATIC_SCRATCH_TOO_SMALL:
      return "problem needs more scratch than the library's built-in array holds (use the workspace entry point)";
    case RF_ERR_BOUNDS: return "a kernel of the bounds-checking build was about to index outside an array";
  }
  return "unknown status";
}

rf_status rf_schedule_dims(const rf_shape* shape, const rf_params* params, int32_t* nQ, int32_t* nKmax) {
  rf_status st = check_shape(shape);
  if (st != RF_OK) return st;
  st = check_params(params);
  if (st != RF_OK) return st;
  st = check_2d(shape, params);
  if (st != RF_OK) return st;
  const RfGeom g = make_geom(shape, params);
  if (nQ) *nQ = g.nQ;
  if (nKmax) *nKmax = g.nKmax;
  return RF_OK;
}

size_t rf_workspace_bytes(const rf_shape* shape, const rf_params* params) {
  return check_shape(shape) == RF_OK ? rf_group_workspace_bytes(shape, params, shape->B * shape->H, 0) : 0;
}

rf_status rf_arm_classify(const rf_shape* shape, const rf_params* params, const void* q, const void* k,
                          int32_t* head_class, float* recall, void* ws, size_t ws_bytes, int32_t* dev_status,
                          void* cuda_stream) {
  return arm_call(shape, params, nullptr, 0, q, k, head_class, nullptr, recall, ws, ws_bytes, dev_status, cuda_stream);
}

rf_status rf_selftest_arm_abandoned(const rf_shape* shape, const rf_params* params, const void* q, const void* k,
                                    int32_t* head_class, void* ws, size_t ws_bytes, int32_t* dev_status, void* cuda_stream) {
  return arm_call(shape, params, nullptr, 0, q, k, head_class, nullptr, nullptr, ws, ws_bytes, dev_status, cuda_stream, nullptr, true);
}

rf_status rf_arm_classify_plus(const rf_shape* shape, const rf_params* params, const float* bandwidths,
                               int32_t n_bandwidths, const void* q, const void* k, int32_t* head_class,
                               int32_t* head_window, float* recall, void* ws, size_t ws_bytes, int32_t* dev_status,
                               void* cuda_stream) {
  if (n_bandwidths < 1) {
    // (0 selects the fixed windows in arm_call)
    const rf_status st = check_arm(shape, params, true);
    return st != RF_OK ? st : RF_ERR_INVALID_ARG;
  }
  return arm_call(shape, params, bandwidths, n_bandwidths, q, k, head_class, head_window, recall, ws, ws_bytes, dev_status, cuda_stream);
}

rf_status rf_build_block_mask(const rf_shape* shape, const rf_params* params, const int32_t* head_class,
                              rf_schedule* out, int32_t* dev_status, void* cuda_stream) {
  return rf_build_block_mask_plus(shape, params, head_class, nullptr, out, dev_status, cuda_stream);
}

rf_status rf_build_block_mask_plus(const rf_shape* shape, const rf_params* params, const int32_t* head_class,
                                   const int32_t* head_window, rf_schedule* out, int32_t* dev_status, void* cuda_stream) {
  rf_status st = check_shape(shape);
  if (st != RF_OK) return st;
  st = check_params(params);
  if (st != RF_OK) return st;
  st = check_2d(shape, params);
  if (st != RF_OK) return st;
  if (head_window != nullptr && params->temporal_window_2d) return RF_ERR_UNSUPPORTED;
  if (head_class == nullptr || out == nullptr || out->count == nullptr || out->kv_tile == nullptr || out->kv_len == nullptr)
    return RF_ERR_INVALID_ARG;
  const RfGeom g = make_geom(shape, params);
  if (out->nQ != g.nQ || out->nKmax != g.nKmax) return RF_ERR_INVALID_ARG;
  cudaError_t e = rf_launch_build_tiles(g, head_class, head_window, out->count, out->kv_tile, out->bitmap, out->kv_len,
                                        dev_status, static_cast<cudaStream_t>(cuda_stream));
  return e == cudaSuccess ? RF_OK : RF_ERR_CUDA;
}

rf_status rf_sparse_attn_fwd(const rf_shape* shape, const rf_params* params, const void* q, const void* k,
                             const void* v, const int32_t* head_class, const rf_schedule* sched, void* o, float* lse,
                             void* ws, size_t ws_bytes, int32_t* dev_status, void* cuda_stream) {
  return rf_sparse_attn_fwd_plus(shape, params, q, k, v, head_class, nullptr, sched, o, lse, ws, ws_bytes, dev_status,
                                 cuda_stream);
}

rf_status rf_sparse_attn_fwd_plus(const rf_shape* shape, const rf_params* params, const void* q, const void* k,
                                  const void* v, const int32_t* head_class, const int32_t* head_window,
                                  const rf_schedule* sched, void* o, float* lse, void* ws, size_t ws_bytes,
                                  int32_t* dev_status, void* cuda_stream) {
  return sparse_attn_impl(shape, params, q, k, v, head_class, head_window, sched, o, lse, ws, ws_bytes, dev_status,
                          cuda_stream, Copies::kMake, shape != nullptr ? shape->B * shape->H : 0, 0);
}

rf_status rf_sparse_attn_reordered(const rf_shape* shape, const rf_params* params, const void* q, const void* k,
                                   const void* v, const int32_t* head_class, const int32_t* head_window,
                                   const rf_schedule* sched, void* o, float* lse, void* ws, size_t ws_bytes,
                                   int32_t* dev_status, void* cuda_stream) {
  return sparse_attn_impl(shape, params, q, k, v, head_class, head_window, sched, o, lse, ws, ws_bytes, dev_status,
                          cuda_stream, Copies::kMade, shape != nullptr ? shape->B * shape->H : 0, 0);
}

rf_status rf_sparse_call(const rf_shape* shape, const rf_params* params, const float* bandwidths, int32_t n_bandwidths, const void* q,
                         const void* k, const void* v, int32_t* head_class, int32_t* head_window, rf_schedule* sched, void* o,
                         float* lse, void* ws, size_t ws_bytes, int32_t* dev_status, void* cuda_stream) {
  return rf_sparse_call_group(shape, params, bandwidths, n_bandwidths, q, k, v, head_class, head_window, sched, o, lse, ws, ws_bytes,
                              dev_status, cuda_stream, shape != nullptr ? shape->B * shape->H : 0, 0);
}

rf_status rf_selftest_sparse_call_abandoned(const rf_shape* shape, const rf_params* params, const float* bandwidths, int32_t n_bandwidths,
                                            const void* q, const void* k, const void* v, int32_t* head_class, int32_t* head_window,
                                            rf_schedule* sched, void* o, float* lse, void* ws, size_t ws_bytes, int32_t* dev_status,
                                            void* cuda_stream) {
  return rf_sparse_call_group(shape, params, bandwidths, n_bandwidths, q, k, v, head_class, head_window, sched, o, lse, ws, ws_bytes,
                              dev_status, cuda_stream, shape != nullptr ? shape->B * shape->H : 0, 0, true);
}

rf_status rf_selftest_wait_timeout(int32_t* dev_status, int32_t limit_ms, int32_t* waits_returned, void* cuda_stream) {
  if (dev_status == nullptr || waits_returned == nullptr || limit_ms < 1 || limit_ms > 1000) return RF_ERR_INVALID_ARG;
  return rf_launch_selftest_timeout(dev_status, (uint64_t)limit_ms * 1000000ull, waits_returned,
                                    static_cast<cudaStream_t>(cuda_stream));
}

rf_status rf_reorder_tokens(const rf_shape* shape, const rf_params* params, const void* q, const void* k,
                            const void* v, const int32_t* head_class, void* ws, size_t ws_bytes, void* cuda_stream) {
  rf_status st = check_shape(shape);
  if (st != RF_OK) return st;
  st = check_params(params);
  if (st != RF_OK) return st;
  st = check_2d(shape, params);
  if (st != RF_OK) return st;
  if (shape->D > 2048) return RF_ERR_UNSUPPORTED;   // a row is at most one CTA's 256 vectors of 16 bytes
  if (q == nullptr || k == nullptr || v == nullptr || head_class == nullptr || ws == nullptr) return RF_ERR_INVALID_ARG;
  if (!aligned16(q) || !aligned16(k) || !aligned16(v) || (reinterpret_cast<uintptr_t>(ws) & (kAlign - 1)) != 0)
    return RF_ERR_INVALID_ARG;
  const RfGeom g = make_geom(shape, params);
  if (ws_bytes < least_bytes(g, params)) return RF_ERR_WORKSPACE_TOO_SMALL;
  uint8_t* w = static_cast<uint8_t*>(ws);
  cudaError_t e = rf_launch_gather(g, head_class, static_cast<const __nv_bfloat16*>(q), static_cast<const __nv_bfloat16*>(k),
                                   static_cast<const __nv_bfloat16*>(v), reinterpret_cast<__nv_bfloat16*>(w),
                                   reinterpret_cast<__nv_bfloat16*>(w + tensor_bytes(g)),
                                   reinterpret_cast<__nv_bfloat16*>(w + 2 * tensor_bytes(g)), nullptr, 0, nullptr,
                                   static_cast<cudaStream_t>(cuda_stream));
  return e == cudaSuccess ? RF_OK : RF_ERR_CUDA;
}

size_t rf_dense_workspace_bytes(const rf_shape* shape) {
  if (check_attn_shape(shape) != RF_OK) return 0;
  return rf_split_bytes(rf_split_plan(make_geom(shape, 0, 0, 1, 128, 128, 0), false, shape->B * shape->H, 0), shape->D);
}

rf_status rf_dense_attn_fwd_split(const rf_shape* shape, const void* q, const void* k, const void* v, void* o, float* lse,
                                  void* scratch, size_t scratch_bytes, int32_t* dev_status, void* cuda_stream) {
  rf_status st = check_attn_shape(shape);
  if (st != RF_OK) return st;
  if (q == nullptr || k == nullptr || v == nullptr || o == nullptr) return RF_ERR_INVALID_ARG;
  if (!aligned16(q) || !aligned16(k) || !aligned16(v) || !aligned16(o)) return RF_ERR_INVALID_ARG;
  const RfGeom g = make_geom(shape, 0, 0, 1, 128, 128, 0);
  CUtensorMap maps[RF_ATTN_MAPS];
  const int heads = g.B * g.H;
  bool ok = encode_map(&maps[0], q, g.D, g.N, g.N, heads) && encode_map(&maps[1], k, g.D, g.N, g.N, heads) &&
            encode_v_map(&maps[2], v, g.D, g.N, g.N, heads);
  if (!ok) return RF_ERR_CUDA;
  for (int i = 3; i < 8; ++i) maps[i] = maps[i % 3];
  RfAttnArgs a;
  const RfSplit sp = rf_split_plan(g, false, heads, 0);
  const bool split = sp.on && scratch != nullptr && (reinterpret_cast<uintptr_t>(scratch) & (kAlign - 1)) == 0 &&
                     scratch_bytes >= rf_split_bytes(sp, g.D);
  set_split(&a, split ? sp : RfSplit{}, static_cast<uint8_t*>(scratch));
  if (split && rf_launch_zero(a.tickets, (int)sp.n_tickets, static_cast<cudaStream_t>(cuda_stream)) != cudaSuccess) return RF_ERR_CUDA;
  a.g = g;
  a.head_class = nullptr;
  a.head_window = nullptr;
  a.count = nullptr;
  a.kv_tile = nullptr;
  a.o = static_cast<__nv_bfloat16*>(o);
  a.lse = lse;
  a.dev_status = dev_status;
  a.scale_log2 = 1.4426950408889634f / sqrtf((float)g.D);
  return rf_launch_attention(a, maps, static_cast<cudaStream_t>(cuda_stream));
}

rf_status rf_dense_attn_fwd(const rf_shape* shape, const void* q, const void* k, const void* v, void* o, float* lse,
                            void* ws, size_t ws_bytes, int32_t* dev_status, void* cuda_stream) {
  (void)ws;
  (void)ws_bytes;
  return rf_dense_attn_fwd_split(shape, q, k, v, o, lse, nullptr, 0, dev_status, cuda_stream);
}

}  // extern "C"
