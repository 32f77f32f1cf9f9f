// Shared host/device definitions of the RainFusion CUDA path (sm_100a only).
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/rainfusion.h"

#define RF_PARTIAL_BIT 0x80000000u

// Geometry and pattern parameters as the kernels see them (passed by value).
struct RfGeom {
  int B, H, D;
  int T, Hf, Wf, S;      // frames, frame height/width, tokens per frame
  int Nv, L, N;          // video tokens, text tokens, all tokens
  int wf, ws, tau;       // frame window, spatial window, checkerboard stride
  int nC;                // kept tokens per frame for the Textural pattern
  int LkvTex;            // key slots of a Textural head: T*nC + L
  int BM, BN, nQ, nKmax; // block mask tile and its extents
  int permute;           // Temporal heads in position-major order
  int two_mask;          // ARM decides between Spatial and Temporal only (ablation of Sec. 4.4)
  int key_first;         // Spatial heads also keep every key of frame 0 (a key frame, Sec. 3.2)
  int t2d, wy, wx;       // Temporal heads keep the 2-D in-frame window |dy| <= wy, |dx| <= wx instead of the band ws
};

// Device-side error reporting: first error wins, kernels never trap.
__device__ __forceinline__ void rf_report(int32_t* dev_status, int code) {
  if (dev_status != nullptr) atomicCAS(dev_status, 0, code);
}

// Index check of the bounds-checking build: true when idx < limit; otherwise RF_ERR_BOUNDS is reported and the
// caller skips the access.  Compiles to `true` in the normal build.
#ifdef RF_BOUNDS_CHECK
__device__ __forceinline__ bool rf_in_bounds(unsigned long long idx, unsigned long long limit, int32_t* dev_status) {
  if (idx < limit) return true;
  rf_report(dev_status, RF_ERR_BOUNDS);
  return false;
}
#else
__device__ __forceinline__ bool rf_in_bounds(unsigned long long, unsigned long long, int32_t*) { return true; }
#endif

__host__ __device__ __forceinline__ int rf_cdiv(int a, int b) { return (a + b - 1) / b; }

// Number of key slots of a head of class `cls`.
__host__ __device__ __forceinline__ int rf_kv_len(const RfGeom& g, int cls) {
  return cls == RF_TEXTURAL ? g.LkvTex : g.N;
}

// Programmatic dependent launch.  Every kernel of the path is launched so that its CTAs may become resident, and set up
// what depends on no global memory, while the kernel before it in the stream drains; rf_grid_wait then waits until all of
// that kernel's writes are visible.  All threads of a kernel call it before their first access to global memory.
// Inputs are plain pointers: const __restrict__ or __ldg would promise that they do not change while the kernel runs, and it
// runs from before the wait, so such a load need not stay behind it.
// rf_grid_trigger lets the next kernel's CTAs come in as soon as every CTA of this one has called it or ended.
__device__ __forceinline__ void rf_grid_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void rf_grid_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
// While an RfPlainLaunches is alive, its thread launches without the attribute: see rf_host_pipeline_run.
inline thread_local int rf_plain_launches = 0;
struct RfPlainLaunches {
  RfPlainLaunches() { ++rf_plain_launches; }
  ~RfPlainLaunches() { --rf_plain_launches; }
};
template <typename... P, typename... A>
inline cudaError_t rf_launch(void (*kernel)(P...), dim3 grid, unsigned block, size_t smem, cudaStream_t st, const A&... args) {
  cudaLaunchConfig_t c = {};
  c.gridDim = grid;
  c.blockDim = dim3(block);
  c.dynamicSmemBytes = smem;
  c.stream = st;
  cudaLaunchAttribute at;
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  c.attrs = &at;
  c.numAttrs = rf_plain_launches > 0 ? 0 : 1;
  return cudaLaunchKernelEx(&c, kernel, static_cast<P>(args)...);
}

// Launchers implemented in the .cu files (host).
// head_window (nullable): per-head window replacing g.wf (Spatial heads) / g.ws (Temporal heads)
cudaError_t rf_launch_build_tiles(const RfGeom& g, const int32_t* head_class, const int32_t* head_window, int32_t* count,
                                  int32_t* kv_tile, uint32_t* bitmap, int32_t* kv_len, int32_t* dev_status, cudaStream_t st);
cudaError_t rf_launch_gather(const RfGeom& g, const int32_t* head_class, const __nv_bfloat16* q,
                             const __nv_bfloat16* k, const __nv_bfloat16* v, __nv_bfloat16* wq, __nv_bfloat16* wk,
                             __nv_bfloat16* wv, int32_t* tickets, int n_tickets, int32_t* dev_status, cudaStream_t st);
// Algorithm 1's decision (or the dynamic-bandwidth one) over the score kernel's sums; see rf_decide in rf_decide.cuh.
struct RfDecision {
  int nb, nb_user;            // window slots per pattern, candidates among them
  int n_loc, n_glb;           // rows of the first-frame and of the stride sample
  int t_loc, t_glb, t_pad;    // score CTAs (128 rows each) of a head per sample
  int local_t;                // the Temporal recall comes from the first-frame sample
  int two_mask;
  float alpha;
  int ws[RF_MAX_BANDWIDTHS], wf[RF_MAX_BANDWIDTHS];
  const double *loc, *glb;    // [B*H][2*nb+1][t_pad]: sums of the rows' recalls
  const int32_t* arm_flag;
  int32_t* head_class;
  int32_t* head_window;       // null: plain Algorithm 1
  float* recall;
  float* recall_plus;
  int32_t* dev_status;
};
// The tile schedule and the reordered copies of a call whose classes are not decided yet: every warp takes the decision of its
// head itself and one of them writes it out.  One launch for what rf_launch_build_tiles, rf_launch_gather and the decision
// kernel do.
cudaError_t rf_launch_prepare(const RfGeom& g, const RfDecision& dec, int32_t* count, int32_t* kv_tile, uint32_t* bitmap,
                              int32_t* kv_len, const __nv_bfloat16* q, const __nv_bfloat16* k, const __nv_bfloat16* v,
                              __nv_bfloat16* wq, __nv_bfloat16* wk, __nv_bfloat16* wv, int32_t* tickets, int n_tickets,
                              int32_t* dev_status, cudaStream_t st);
// nb candidate windows per pattern (ws_list for Temporal, wf_list for Spatial, ascending).  head_window == nullptr:
// plain Algorithm 1 on the first candidate (recall: [B,H,3] or null).  Otherwise dynamic bandwidth: head_window
// receives each head's chosen window, recall_plus ([B,H,2,nb] or null) the candidates' recalls.
// dev_status (nullable) receives RF_ERR_TIMEOUT if a wait inside the score kernel ran out; head_class is then -1.
// selftest_abandon: the score kernel is not launched; its failure flag is set instead, as if a wait had run out.
// later (nullable): the decision is not launched but left there for rf_launch_prepare.
cudaError_t rf_launch_arm(const RfGeom& g, int sample_mode, int omega, float alpha, int nb, const int* ws_list,
                          const int* wf_list, const __nv_bfloat16* q, const __nv_bfloat16* k, int32_t* head_class,
                          int32_t* head_window, float* recall, float* recall_plus, float* scratch, int32_t* dev_status,
                          cudaStream_t st, bool selftest_abandon = false, RfDecision* later = nullptr);
// Floats of ARM scratch.  The sums of the rows' recalls lie at its end, before RF_ARM_FLAG_FLOATS whose first word records a
// wait that ran out inside the score kernel (cleared by every call at the start of its first kernel).  The size allows for a float
// per sampled row and mask, of which a sum takes a 64th: the entry points accept and refuse callers' blocks, and
// rf_arm_classify_noalloc shapes, by it.
#define RF_ARM_FLAG_FLOATS 64
size_t rf_arm_scratch_floats(const RfGeom& g, int omega, int nb);
// Tensor map over bf16 rows: [heads][rows][D] with the given row and head strides in bytes (multiples of 16),
// box = 64 (or 32) columns x 128 rows, swizzled by the box's row of 128 (64) bytes, zero fill past `rows`.
bool rf_encode_rows_map(CUtensorMap* m, const void* ptr, int D, int rows, size_t row_stride_bytes,
                        size_t head_stride_bytes, int heads, int box_columns = 64);
// Validates shape and parameters as the entry points do and fills the kernel-side geometry.
rf_status rf_checked_geom(const rf_shape* shape, const rf_params* params, RfGeom* out);

// Split items.  An item of the attention kernel is a pair of query tiles of one head; one CTA per SM works items off, so a
// call of a few hundred items ends with most SMs idle, and one of fewer items than SMs never fills them.  The items of
// the last, partial wave (all of them when there are fewer items than SMs) are therefore cut into pieces of their tile
// lists, and so are the pairs with text rows, whose lists are twice as long as the others', when there are at most three
// waves.  A piece leaves its unnormalised O and its sums in the workspace; whoever finishes last joins them.  The plan
// depends on the whole call's shape alone (and on the item's own list), so that a call made in groups of heads gives
// the same bits as the call made at once.
struct RfSplit {
  int on;                    // 0: one unit of work per item, in the order of place_item
  int text_pairs;            // pairs of query tiles that may hold text rows (the last ones of a head): the first units
  int kt, lt;                // pieces such an item has at most, tiles of a piece
  int kr, lr;                // the same for the tail items
  uint32_t n_text;           // units of the pairs with text rows
  int row0, head_row0;       // the other items lie in rows (one item per head), last pairs first: the tail is the rows from
                             // row0 on, of row0 itself the heads from head_row0 on
  uint32_t first_tail;       // the items that stay whole come before the tail
  uint32_t n_units, n_slots, n_tickets;
};
RfSplit rf_split_plan(const RfGeom& g, bool sparse, int heads_total, int head0);
// Bytes of the split region: the tickets (one word per piece-joining warp, zero when a call begins), then the pieces.
size_t rf_split_ticket_bytes(const RfSplit& sp);
size_t rf_split_bytes(const RfSplit& sp, int D);
cudaError_t rf_launch_zero(int32_t* words, int n, cudaStream_t st);

struct RfAttnArgs {
  RfGeom g;
  const int32_t* head_class;  // nullptr: every head Dense, implicit full tile list
  const int32_t* head_window; // nullable: per-head window replacing g.wf (Spatial) / g.ws (Temporal)
  const int32_t* count;
  const int32_t* kv_tile;
  __nv_bfloat16* o;
  float* lse;
  int32_t* dev_status;
  float scale_log2;           // log2(e) / sqrt(D)
  RfSplit sp;
  int32_t* tickets;           // [n_tickets], zero
  float* pieces;              // [n_slots][2 streams][D/4 + 1][128 rows] float4: O, then {m, l, l exact, has O}
  int heads_l2 = 1;           // heads whose items are interleaved (filled by the launcher)
};
// Tensor maps: [0..2] Q/K/V in original order, [3..5] the workspace copies with N rows per head
// (position-major Q/K/V of Temporal heads), [6..7] workspace K/V with LkvTex rows per head (Textural).
constexpr int RF_ATTN_MAPS = 8;
rf_status rf_launch_attention(const RfAttnArgs& a, const CUtensorMap* maps, cudaStream_t st);
// A call for heads [head0, head0 + B*H) of one of heads_total heads that is made in groups; the workspace needs
// rf_group_workspace_bytes, or rf_least_workspace_bytes if no item is to be split.
size_t rf_least_workspace_bytes(const rf_shape* shape, const rf_params* params);
size_t rf_group_workspace_bytes(const rf_shape* shape, const rf_params* params, int heads_total, int head0);
rf_status rf_sparse_call_group(const rf_shape* shape, const rf_params* params, const float* bandwidths, int32_t n_bandwidths,
                               const void* q, const void* k, const void* v, int32_t* head_class, int32_t* head_window,
                               rf_schedule* sched, void* o, float* lse, void* ws, size_t ws_bytes, int32_t* dev_status,
                               void* cuda_stream, int heads_total, int head0, bool selftest_abandon = false);
rf_status rf_launch_selftest_timeout(int32_t* dev_status, uint64_t limit_ns, int32_t* waits_returned, cudaStream_t st);
