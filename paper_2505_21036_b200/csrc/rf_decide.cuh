// The decision over the recalls of a head (Algorithm 1, Sec. 3.3; or the smallest qualifying bandwidth).
#pragma once

#include "rf_common.cuh"

struct RfHead { int cls, window, failed; };

// One warp, all of it; every warp that asks gets the same answer (fixed order of additions).  write: also stores class, window
// and recalls.
//   plain (head_window == nullptr, nb = 1): Algorithm 1.
//   dynamic bandwidth: a pattern qualifies if any candidate window reaches alpha, Temporal before Spatial;
//   the head takes the smallest qualifying window (candidates ascend); Textural heads get window -1.
__device__ __forceinline__ RfHead rf_decide(const RfDecision& d, int bh, int lane, bool write) {
  RfHead h;
  h.cls = h.window = -1;
  h.failed = *d.arm_flag;
  write = write && lane == 0;
  if (h.failed != 0) {
    // the score kernel gave up a wait: its rows are incomplete, no class may come out of them
    if (lane == 0) rf_report(d.dev_status, h.failed);
    if (write) {
      d.head_class[bh] = -1;
      if (d.head_window != nullptr) d.head_window[bh] = -1;
    }
    return h;
  }
  const int nm = 2 * d.nb + 1;
  // mean recall of mask k: Temporal windows, then Spatial ones, then Textural
  auto recall = [&](int k) -> float {
    const bool local = k < d.nb && d.local_t;
    const double* src = (local ? d.loc : d.glb) + ((size_t)bh * nm + k) * d.t_pad;
    const int tiles = local ? d.t_loc : d.t_glb;
    double sum = 0.0;
    for (int i = lane; i < tiles; i += 32) sum += src[i];
    for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    return (float)(sum / (local ? d.n_loc : d.n_glb));
  };
  if (d.head_window == nullptr) {
    const float rt = recall(0), rs = recall(d.nb);
    if (d.recall != nullptr) {
      const float rc = recall(2 * d.nb);   // (the score kernel sums it whenever recalls are asked for)
      if (write) { d.recall[bh * 3] = rt; d.recall[bh * 3 + 1] = rs; d.recall[bh * 3 + 2] = rc; }
    }
    // Algorithm 1; with only two masks (ablation) a head that reaches alpha with neither takes the larger recall
    const int otherwise = d.two_mask ? (rt >= rs ? RF_TEMPORAL : RF_SPATIAL) : RF_TEXTURAL;
    h.cls = rt >= d.alpha ? RF_TEMPORAL : (rs >= d.alpha ? RF_SPATIAL : otherwise);
    if (write) d.head_class[bh] = h.cls;
    return h;
  }
  int first_t = -1, first_s = -1;        // windows of the first candidates that reach alpha
  float widest_t = 0.f, widest_s = 0.f;
  // of the kernel's nb slots the caller's nb_user candidates are the first; the others stay empty
  for (int i = 0; i < d.nb_user; ++i) {
    const float rt = recall(i), rs = recall(d.nb + i);
    if (first_t < 0 && rt >= d.alpha) first_t = d.ws[i];
    if (first_s < 0 && rs >= d.alpha) first_s = d.wf[i];
    widest_t = rt;
    widest_s = rs;
    if (write && d.recall_plus != nullptr) {
      d.recall_plus[(bh * 2) * d.nb_user + i] = rt;
      d.recall_plus[(bh * 2 + 1) * d.nb_user + i] = rs;
    }
  }
  if (first_t >= 0) {
    h.cls = RF_TEMPORAL;
    h.window = first_t;
  } else if (first_s >= 0) {
    h.cls = RF_SPATIAL;
    h.window = first_s;
  } else if (d.two_mask) {               // nothing qualifies: the larger recall at the widest candidate, with that bandwidth
    const bool t = widest_t >= widest_s;
    h.cls = t ? RF_TEMPORAL : RF_SPATIAL;
    h.window = t ? d.ws[d.nb_user - 1] : d.wf[d.nb_user - 1];
  } else {
    h.cls = RF_TEXTURAL;
  }
  if (write) {
    d.head_class[bh] = h.cls;
    d.head_window[bh] = h.window;
  }
  return h;
}
