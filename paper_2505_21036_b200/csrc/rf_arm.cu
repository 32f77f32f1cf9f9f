// ARM: Adaptive Recognition Module (Sec. 3.3, Eq. 6, Algorithm 1).
//
// The sampled score matrix S' = Q' K'^T / sqrt(d) is a dense contraction, so it runs on tcgen05 like the
// attention kernel, minus everything that concerns V: one CTA takes one 128-row tile of sampled queries of one
// head and walks all 128-key tiles of the sample.  Sampled rows are fetched straight from Q and K by TMA through
// tensor maps whose row stride is omega tokens (no gather pass).  Warp roles:
//   warps 0-3 / 4-7  softmax statistics of the even / odd key tiles (one thread per sampled query row)
//   warp 8           TMA producer: the Q tile once, then K tiles into a shared-memory ring
//   warp 9           MMA issuer; S is double-buffered in TMEM (2 x 128 columns), a buffer per warpgroup
// The kernel is bound by its exponentials (one per score; 1024 cycles of the exponential pipe per warp and tile) once
// enough warps hide the chain load -> maximum -> exponentials -> sums of each other's tiles: two CTAs share an SM
// (half of its TMEM, shared memory and registers each), so a sub-partition holds four softmax warps and one CTA's start
// runs beside the other's tiles.  A thread holds 64 scores at a time and takes the first half from TMEM twice (maximum,
// then exponentials).  Measured against one CTA per SM with two warps a sub-partition, 128 scores a thread and two
// query tiles a CTA (rf_arm_classify alone, us): 24 heads, samples of 1024 39.1 -> 29.4; 48 heads, 1170 and 1350, D = 64
// 94.7 -> 71.5; 24 heads, 3300 and 3600 258 -> 217; with three candidate windows, 1920 and 2040 169 -> 121; with the
// per-key table (both recalls on the stride sample, 867 of 86 400 tokens) 38.4 -> 31.2.
// Per tile a softmax thread updates an online softmax (running maximum, total mass) plus the masked masses
// Algorithm 1 needs: the share of the row kept by the sampled Temporal / Spatial (/ Textural, when recalls are
// requested) mask; the two warpgroups' statistics of a row are joined at the end.
// On the first-frame sample positions equal sample indices, and on the stride sample frames grow
// with the sample index, so a row's kept keys form one index interval: half tiles wholly inside or outside
// it for all 32 rows of a warp cost nothing extra (which they are is worked out before the scores arrive), those
// an edge crosses use a 64-bit keep word per row.  Only the Temporal mask on the stride sample (RF_SAMPLE_GLOBAL) and the Textural diagnostic
// need per-key attributes, computed cooperatively per tile.
// With the first frame as a key frame of Spatial heads (Sec. 3.2: adjacent or key frames) the Spatial masks keep,
// in addition, the sampled keys of frame 0, a prefix of the stride sample.
// A CTA leaves the sums of its rows' recalls in scratch (in double and in a fixed order, so that they do not depend on the
// schedule); whoever needs the classes next adds a head's few sums up and takes Algorithm 1's decision: the decision kernel here,
// or every warp of the kernel that builds the schedule and the copies, which saves a call two launches (3 heads, 272
// tokens 31.2 -> 27.5 us a call; 10 heads, 3668 tokens 80.7 -> 77.3; 3 heads, 7476 tokens 120.4 -> 113.5).  The n x n score matrix is never written.
// A bounded wait that runs out is recorded in a flag word at the end of the scratch (cleared by the score
// kernel as it starts); the decision then gives class -1 for every head instead of a class computed from
// unwritten rows, and passes the code on to the caller's status word.  The tile builder and the attention
// kernel report a class outside 0..3 through their own status, so the failure cannot go unnoticed even by a
// caller that gave ARM no status pointer.
#include "rf_decide.cuh"
#include "rf_sm100.cuh"

namespace {

using namespace sm100;

constexpr int ARM_TILE = 128;
constexpr int ARM_HALF = 64;               // scores a thread holds at a time
constexpr int ARM_THREADS = 320;           // softmax of even tiles, of odd tiles, TMA, MMA
constexpr int ARM_TMA_WARP = 8, ARM_MMA_WARP = 9;
constexpr float kLeast = -1e38f;           // scores times log2(e) / sqrt(D), at most 0.18, stay above -6.2e37

struct ArmMaps { CUtensorMap q[2], k[2]; };   // per sample: 0 = stride sample, 1 = first-frame sample

constexpr int ARM_MAX_NB = RF_MAX_BANDWIDTHS;   // candidate windows per pattern (1 for plain Algorithm 1)

struct ArmSample {
  int n;          // sampled tokens
  int stride;     // token index of sample m is m * stride
  int tiles;      // CTAs per head: ceil(n / 128)
  int want_t;     // accumulate the Temporal masses on this sample
  int want_s;     // accumulate the Spatial masses on this sample
  double* out;    // [B*H][2*NB+1][t_pad]: Temporal per window, Spatial per window, Textural
};
struct ArmWindows { int ws[ARM_MAX_NB], wf[ARM_MAX_NB], n; };   // candidate spatial (Temporal) / frame (Spatial) windows

template <int D>
struct ArmCfg {
  static constexpr int KB = (D + 63) / 64;
  static constexpr int COL1 = 64;   // D = 96: the second 64-column box reaches past the tensor and is zero-filled
  static constexpr uint32_t BLK = 128 * 128;
  static constexpr uint32_t TILE = KB * BLK;
  static constexpr int NK = D == 64 ? 4 : 2;
  static constexpr uint32_t Q = 0;
  static constexpr uint32_t K0 = Q + TILE;
  static constexpr uint32_t BAR = K0 + NK * TILE;
  static constexpr int B_Q = 0, B_KF = 1, B_KE = B_KF + NK, B_SF = B_KE + NK, B_SE = B_SF + 2, B_COUNT = B_SE + 2;
  static constexpr uint32_t MISC = BAR + 8 * ((B_COUNT + 7) / 8 * 8);
  static constexpr uint32_t ATTR = MISC + 64;                    // int [8 warps][2][128]: key position / checkerboard flag
  static constexpr uint32_t JOIN = ATTR + 8 * 2 * 128 * 4;       // float [masks + 2][128]: the odd tiles' statistics
  static constexpr uint32_t TOTAL = JOIN + (2 * ARM_MAX_NB + 3) * 128 * 4;
  static constexpr uint32_t ALLOC = TOTAL + 1024;
  static_assert(2 * (ALLOC + 1024) <= 228 * 1024, "two CTAs exceed the shared memory of an SM");
  static __host__ __device__ constexpr uint32_t koff(int ks) {
    return ks < 4 ? (uint32_t)ks * 32u : BLK + (uint32_t)(ks - 4) * 32u;
  }
};

__device__ __forceinline__ float ex2f(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ uint32_t bits_below(int n) { return n >= 32 ? 0xffffffffu : ((1u << n) - 1u); }
// Bits of the half tile starting at key u0 that fall in the key interval [a, b).
__device__ __forceinline__ void interval_bits(uint32_t (&w)[2], int u0, int a, int b) {
  a = max(a - u0, 0);
  b = min(b - u0, ARM_HALF);
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    const int lo = min(max(a - 32 * k, 0), 32), hi = min(max(b - 32 * k, 0), 32);
    w[k] |= hi > lo ? (bits_below(hi) & ~bits_below(lo)) : 0u;
  }
}
__device__ __forceinline__ void load_half(uint32_t t_s, uint32_t (&s)[ARM_HALF]) {
  tmem_ld32(t_s, *reinterpret_cast<uint32_t(*)[32]>(&s[0]));
  tmem_ld32(t_s + 32, *reinterpret_cast<uint32_t(*)[32]>(&s[32]));
  tc_wait_ld();
}
// Keys past the sample score -inf; returns the largest of the others (or mx).
__device__ __forceinline__ float half_max(uint32_t (&s)[ARM_HALF], int u0, int n, float mx) {
  if (u0 + ARM_HALF > n) {
#pragma unroll
    for (int c = 0; c < ARM_HALF; ++c)
      if (u0 + c >= n) s[c] = 0xff800000u;
  }
  float m0 = mx, m1 = -INFINITY;
#pragma unroll
  for (int c = 0; c < ARM_HALF; c += 4) {
    m0 = fmaxf(m0, fmaxf(__uint_as_float(s[c]), __uint_as_float(s[c + 1])));
    m1 = fmaxf(m1, fmaxf(__uint_as_float(s[c + 2]), __uint_as_float(s[c + 3])));
  }
  return fmaxf(m0, m1);
}
// Exponentials in place, 2^(score * sc - m); returns their sum.
__device__ __forceinline__ float half_exp(uint32_t (&s)[ARM_HALF], float sc, float m) {
  const float2 sc2 = make_float2(sc, sc), mneg = make_float2(-m, -m);
  float2 la = make_float2(0.f, 0.f), lb = make_float2(0.f, 0.f);
#pragma unroll
  for (int c = 0; c < ARM_HALF; c += 4) {
    float2 e0 = __ffma2_rn(make_float2(__uint_as_float(s[c]), __uint_as_float(s[c + 1])), sc2, mneg);
    float2 e1 = __ffma2_rn(make_float2(__uint_as_float(s[c + 2]), __uint_as_float(s[c + 3])), sc2, mneg);
    e0.x = ex2f(e0.x); e0.y = ex2f(e0.y);
    e1.x = ex2f(e1.x); e1.y = ex2f(e1.y);
    la = __fadd2_rn(la, e0);
    lb = __fadd2_rn(lb, e1);
    s[c] = __float_as_uint(e0.x); s[c + 1] = __float_as_uint(e0.y);
    s[c + 2] = __float_as_uint(e1.x); s[c + 3] = __float_as_uint(e1.y);
  }
  return (la.x + la.y) + (lb.x + lb.y);
}

// Sum of the weights whose key's attribute (table in shared memory, 16-byte aligned) is kept; four chains of additions.
template <typename F>
__device__ __forceinline__ float table_sum(const uint32_t (&s)[ARM_HALF], const int* table, F kept) {
  const int4* t = reinterpret_cast<const int4*>(table);
  float p0 = 0.f, p1 = 0.f, p2 = 0.f, p3 = 0.f;
#pragma unroll
  for (int c = 0; c < ARM_HALF; c += 4) {
    const int4 a = t[c / 4];
    p0 += kept(a.x) ? __uint_as_float(s[c]) : 0.f;
    p1 += kept(a.y) ? __uint_as_float(s[c + 1]) : 0.f;
    p2 += kept(a.z) ? __uint_as_float(s[c + 2]) : 0.f;
    p3 += kept(a.w) ? __uint_as_float(s[c + 3]) : 0.f;
  }
  return (p0 + p1) + (p2 + p3);
}

template <int D, int NB, bool TEX>
__global__ void __launch_bounds__(ARM_THREADS, 2) rf_arm_kernel(const __grid_constant__ ArmMaps maps, const RfGeom g,
                                                                const ArmSample sm0, const ArmSample sm1,
                                                                const ArmWindows win, int t_pad, float scale_log2,
                                                                int32_t* arm_flag) {
  using C = ArmCfg<D>;
  constexpr uint32_t IDESC_S = idesc_bf16(128, 128, 0);
  extern __shared__ uint8_t smem_raw[];
  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  uint8_t* base_ptr = smem_raw + (base - smem_u32(smem_raw));
  auto bar = [&](int slot) -> uint32_t { return base + C::BAR + 8u * slot; };
  volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(base_ptr + C::MISC);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(base_ptr + C::MISC + 8);

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int bh = blockIdx.y;
  // blockIdx.x enumerates the CTAs of the stride sample first, then those of the first-frame sample
  const bool second = (int)blockIdx.x >= sm0.tiles;
  const ArmSample& sm = second ? sm1 : sm0;
  const int which = second ? 1 : 0;
  const int qt = second ? blockIdx.x - sm0.tiles : blockIdx.x;
  const int n = sm.n, stride = sm.stride;
  const int nt = rf_cdiv(n, ARM_TILE);
  const CUtensorMap* map_q = &maps.q[which];
  const CUtensorMap* map_k = &maps.k[which];
  // positions equal sample indices only while the sample is contiguous and stays inside the first frame
  // (the 2-D in-frame window is not an interval of the sample index, so it always takes the per-key table)
  const bool t_generic = sm.want_t && (stride != 1 || n > g.S || g.t2d);    // needs per-key positions

  if (tid == 0) {
    mbar_init(bar(C::B_Q), 1);
    for (int s = 0; s < C::NK; ++s) { mbar_init(bar(C::B_KF + s), 1); mbar_init(bar(C::B_KE + s), 1); }
    for (int s = 0; s < 2; ++s) { mbar_init(bar(C::B_SF + s), 1); mbar_init(bar(C::B_SE + s), 4); }
    *abort_flag = 0;
    mbar_init_fence();
  }
  if (warp == ARM_TMA_WARP) {
    if (lane == 0) { prefetch_tmap(map_q); prefetch_tmap(map_k); }
    __syncwarp();
    tmem_alloc(smem_u32(const_cast<uint32_t*>(tmem_slot)), 2 * ARM_TILE);
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  const WaitCtx wc{abort_flag, arm_flag};
  rf_grid_trigger();
  rf_grid_wait();
#ifndef RF_BOUNDS_CHECK
  // The call's failure flag is cleared here and not by a launch of its own: the first wait that can raise it runs out
  // two seconds from now.  (The bounds-checking build, whose reports come at once, clears it before the launch.)
  if (blockIdx.x == 0 && blockIdx.y == 0 && tid == 0) *arm_flag = 0;
#endif

  // Masks k = 0..NB-1: Temporal with window win.ws[k]; k = NB..2NB-1: Spatial with win.wf[k-NB];
  // k = 2NB: Textural.  Band masks keep one key interval per row in sample-index space.
  constexpr int NM = 2 * NB + 1;
  // The running maximum starts at a finite value below any finite score: a tile whose scores are all -inf (a key that is -inf
  // where the query is not zero) then adds nothing, instead of -inf - -inf.
  float mx = kLeast, l_all = 0.f;
  float l_m[NM];
#pragma unroll
  for (int k = 0; k < NM; ++k) l_m[k] = 0.f;
  float* join = reinterpret_cast<float*>(base_ptr + C::JOIN) + (tid & 127);
  const int m = qt * ARM_TILE + (tid & 127);                   // sampled row of a softmax thread

  if (warp == ARM_TMA_WARP) {
    if (lane == 0) {
      mbar_expect_tx(bar(C::B_Q), C::TILE);
#pragma unroll
      for (int kb = 0; kb < C::KB; ++kb)
        tma_load_3d(base + C::Q + kb * C::BLK, map_q, kb * C::COL1, qt * ARM_TILE, bh, bar(C::B_Q));
      for (int u = 0; u < nt; ++u) {
        const int ks = u % C::NK;
        if (u >= C::NK) mbar_wait(bar(C::B_KE + ks), ((u / C::NK) - 1) & 1, wc);
        mbar_expect_tx(bar(C::B_KF + ks), C::TILE);
#pragma unroll
        for (int kb = 0; kb < C::KB; ++kb)
          tma_load_3d(base + C::K0 + ks * C::TILE + kb * C::BLK, map_k, kb * C::COL1, u * ARM_TILE, bh, bar(C::B_KF + ks));
      }
    }
  } else if (warp == ARM_MMA_WARP) {
    if (lane == 0) {
      constexpr uint32_t DESC_HI = (1024u >> 4) | (1u << 14) | (2u << 29);
      auto desc = [](uint32_t lo) -> uint64_t { return ((uint64_t)DESC_HI << 32) | lo; };
      const uint32_t q_lo = ((base + C::Q) >> 4) | (1u << 16), k_lo = ((base + C::K0) >> 4) | (1u << 16);
      mbar_wait(bar(C::B_Q), 0, wc);
      for (int u = 0; u < nt; ++u) {
        const int ks = u % C::NK, b = u & 1;
        mbar_wait(bar(C::B_KF + ks), (u / C::NK) & 1, wc);
        if (u >= 2) mbar_wait(bar(C::B_SE + b), ((u >> 1) - 1) & 1, wc);
        tc_fence_after();
        const uint32_t b0 = k_lo + ks * (C::TILE >> 4);
#pragma unroll
        for (int k = 0; k < D / 16; ++k)
          mma_ss(tmem_base + b * ARM_TILE, desc(q_lo + (C::koff(k) >> 4)), desc(b0 + (C::koff(k) >> 4)), IDESC_S, k > 0);
        tc_commit(bar(C::B_SF + b));
        tc_commit(bar(C::B_KE + ks));
      }
    }
  } else {
    const int grp = warp >> 2;                                 // even or odd key tiles
    const int tok = min(m, n - 1) * stride;
    const int rf = tok / g.S, rp = tok - rf * g.S;
    const int ry = rp / g.Wf, rx = rp - ry * g.Wf;
    int slo[NB], shi[NB];                                      // Spatial: stride sample, frames grow with the index
#pragma unroll
    for (int i = 0; i < NB; ++i) {
      slo[i] = rf_cdiv(max(rf - win.wf[i], 0) * g.S, stride);
      shi[i] = rf_cdiv((rf + win.wf[i] + 1) * g.S, stride);
    }
    // Spatial masks with the first frame as key frame also keep the sampled keys of frame 0: a prefix
    // [0, pre) of the stride sample, the same for every row
    const int pre = g.key_first ? rf_cdiv(g.S, stride) : 0;
    const uint32_t t_s = tmem_base + ((uint32_t)((warp & 3) * 32) << 16) + grp * ARM_TILE;
    int* attr_p = reinterpret_cast<int*>(base_ptr + C::ATTR) + warp * 256;           // per-warp tables
    int* attr_c = attr_p + 128;
    const bool by_table_t = sm.want_t && t_generic;

    for (int u = grp; u < nt; u += 2) {
      const int u0 = u * ARM_TILE;
      if (by_table_t || TEX) {
        // per-key attributes of the tile, four keys per lane, into this warp's table
        __syncwarp();
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int c = lane * 4 + i;
          const int ktok = min(u0 + c, n - 1) * stride;
          const int kp = ktok % g.S;
          const int y = kp / g.Wf, x = kp - y * g.Wf;
          attr_p[c] = g.t2d ? ((y << 16) | x) : kp;    // frame dimensions stay below 2^15 with the 2-D window
          attr_c[c] = (y % g.tau) == (x % g.tau);
        }
        __syncwarp();
      }
      // Per mask and half tile, two bits: 2 - the half lies inside the row's kept interval for the whole warp (its sum
      // is added), 0 - outside it (nothing), 1 - an edge crosses it, or the mask goes by the table.
      uint32_t cls[2];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int c0 = u0 + h * ARM_HALF, c1 = min(c0 + ARM_HALF, n);
        uint32_t bits = 0;
        if (c0 < n) {
#pragma unroll
          for (int i = 0; i < NB; ++i) {
            if (i >= win.n) break;                   // slots past the caller's candidates stay empty
            if (sm.want_t) {
              const bool in = rp - win.ws[i] <= c0 && c1 <= rp + win.ws[i] + 1;
              const bool out = c1 <= rp - win.ws[i] || rp + win.ws[i] + 1 <= c0;
              bits |= (t_generic ? 1u : (__all_sync(0xffffffffu, in) ? 2u : (__all_sync(0xffffffffu, out) ? 0u : 1u))) << (2 * i);
            }
            if (sm.want_s) {
              const bool in = (slo[i] <= c0 && c1 <= shi[i]) || c1 <= pre, out = (c1 <= slo[i] || shi[i] <= c0) && c0 >= pre;
              bits |= (__all_sync(0xffffffffu, in) ? 2u : (__all_sync(0xffffffffu, out) ? 0u : 1u)) << (2 * (NB + i));
            }
          }
          if (TEX) bits |= 1u << (4 * NB);
        }
        cls[h] = bits;
      }

      mbar_wait(bar(C::B_SF + grp), (u >> 1) & 1, wc);
      tc_fence_after();
      uint32_t s[ARM_HALF];
      load_half(t_s, s);
      float top = half_max(s, u0, n, -INFINITY);
      load_half(t_s + ARM_HALF, s);
      top = half_max(s, u0 + ARM_HALF, n, top);
      const float m_new = fmaxf(mx, top * scale_log2);
      const float corr = ex2f(mx - m_new);
      l_all *= corr;
#pragma unroll
      for (int k = 0; k < NM; ++k) l_m[k] *= corr;
      mx = m_new;
#pragma unroll 1
      for (int h = 1; h >= 0; --h) {
        const int c0 = u0 + h * ARM_HALF;
        if (h == 0) {
          load_half(t_s, s);
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(bar(C::B_SE + grp));   // the buffer may be refilled
          half_max(s, c0, n, -INFINITY);                    // (for the keys past the sample)
        }
        const float bs = half_exp(s, scale_log2, mx);
        l_all += bs;
        const uint32_t bits = h ? cls[1] : cls[0];
#pragma unroll
        for (int k = 0; k < NM; ++k)
          if (((bits >> (2 * k)) & 3u) == 2u) l_m[k] += bs;
        if ((bits & 0x55555555u) == 0) continue;
#pragma unroll 1
        for (int k = 0; k < NM; ++k) {
          if (((bits >> (2 * k)) & 3u) != 1u) continue;
          const bool is_t = k < NB, is_x = k == 2 * NB;
          float add = 0.f;
          if (is_x) {
            add = table_sum(s, attr_c + h * ARM_HALF, [](int a) { return a != 0; });
          } else if (is_t && t_generic) {
            int wk = 0;
#pragma unroll
            for (int i = 0; i < NB; ++i)
              if (i == k) wk = win.ws[i];
            if (g.t2d) {
              const int wy = g.wy, wx = g.wx;
              add = table_sum(s, attr_p + h * ARM_HALF, [=](int a) { return abs((a >> 16) - ry) <= wy && abs((a & 0xffff) - rx) <= wx; });
            } else {
              const int off = wk - rp;                           // |position - rp| <= wk
              const uint32_t span = 2u * (uint32_t)wk;
              add = table_sum(s, attr_p + h * ARM_HALF, [=](int a) { return (uint32_t)(a + off) <= span; });
            }
          } else {
            int klo = 0, khi = 0;
#pragma unroll
            for (int i = 0; i < NB; ++i) {
              if (i == k) { klo = rp - win.ws[i]; khi = rp + win.ws[i] + 1; }
              if (NB + i == k) { klo = slo[i]; khi = shi[i]; }
            }
            uint32_t w[2] = {0, 0};
            interval_bits(w, c0, klo, khi);
            if (!is_t && pre > c0) interval_bits(w, c0, 0, pre);
#pragma unroll
            for (int c = 0; c < ARM_HALF; ++c)
              if ((w[c >> 5] >> (c & 31)) & 1u) add += __uint_as_float(s[c]);
          }
#pragma unroll
          for (int i = 0; i < NM; ++i)
            if (i == k) l_m[i] += add;
        }
      }
    }
    if (grp == 1) {
      join[0] = mx;
      join[128] = l_all;
#pragma unroll
      for (int k = 0; k < NM; ++k) join[(2 + k) * 128] = l_m[k];
    }
  }

  __syncthreads();
  double* part = reinterpret_cast<double*>(base_ptr + C::ATTR);   // [masks][4 warps]; the tables are done with
  auto wanted = [&](int k) { return k == 2 * NB ? TEX : (k < NB ? sm.want_t != 0 : sm.want_s != 0); };
  if (warp < 4) {
    const float m1 = join[0], top = fmaxf(mx, m1);
    const float f0 = ex2f(mx - top), f1 = ex2f(m1 - top);        // no odd tile: m1 = kLeast, factor 0
    const float inv = 1.f / (l_all * f0 + join[128] * f1);
#pragma unroll
    for (int k = 0; k < NM; ++k) {
      if (!wanted(k)) continue;
      double sum = m < n ? (double)((l_m[k] * f0 + join[(2 + k) * 128] * f1) * inv) : 0.0;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
      if (lane == 0) part[k * 4 + warp] = sum;
    }
  }

  tc_fence_before();
  __syncthreads();
  if (tid < NM && wanted(tid) && rf_in_bounds(qt, t_pad, arm_flag))
    sm.out[((size_t)bh * NM + tid) * t_pad + qt] = (part[tid * 4] + part[tid * 4 + 1]) + (part[tid * 4 + 2] + part[tid * 4 + 3]);
  if (warp == ARM_TMA_WARP) {
    if (*abort_flag) __nanosleep(20000);
    __syncwarp();
    tmem_dealloc(tmem_base, 2 * ARM_TILE);
  }
}

// One warp per head.
__global__ void __launch_bounds__(32) rf_arm_decide_kernel(const RfDecision d) {
  rf_grid_trigger();
  rf_grid_wait();
  rf_decide(d, blockIdx.x, threadIdx.x, true);
}

// Self-test only: stands in for a score kernel whose wait ran out.
__global__ void rf_arm_set_flag_kernel(int32_t* arm_flag, int code) {
  rf_grid_wait();
  *arm_flag = code;
}

template <int D, int NB, bool TEX>
cudaError_t launch_arm_t(const ArmMaps& maps, const RfGeom& g, const ArmSample& s0, const ArmSample& s1,
                         const ArmWindows& win, int t_pad, int32_t* arm_flag, cudaStream_t st) {
  static bool configured[64] = {};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev >= 0 && dev < 64 && !configured[dev]) {
    e = cudaFuncSetAttribute(rf_arm_kernel<D, NB, TEX>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ArmCfg<D>::ALLOC);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(rf_arm_kernel<D, NB, TEX>, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
    if (e != cudaSuccess) return e;
    configured[dev] = true;
  }
  dim3 grid(s0.tiles + s1.tiles, g.B * g.H);
  const float scale_log2 = 1.4426950408889634f / sqrtf((float)D);
  return rf_launch(rf_arm_kernel<D, NB, TEX>, grid, ARM_THREADS, ArmCfg<D>::ALLOC, st, maps, g, s0, s1, win, t_pad, scale_log2, arm_flag);
}

template <int D>
cudaError_t launch_arm_n(bool plus, bool tex, const ArmMaps& maps, const RfGeom& g, const ArmSample& s0,
                         const ArmSample& s1, const ArmWindows& win, int t_pad, int32_t* arm_flag, cudaStream_t st) {
  if (plus) return launch_arm_t<D, ARM_MAX_NB, false>(maps, g, s0, s1, win, t_pad, arm_flag, st);
  return tex ? launch_arm_t<D, 1, true>(maps, g, s0, s1, win, t_pad, arm_flag, st)
             : launch_arm_t<D, 1, false>(maps, g, s0, s1, win, t_pad, arm_flag, st);
}

int arm_n_pad(const RfGeom& g, int omega) {
  const int n_glb = rf_cdiv(g.Nv, omega);
  const int n = n_glb > g.S ? n_glb : g.S;
  return (n + 63) / 64 * 64;
}

}  // namespace

size_t rf_arm_scratch_floats(const RfGeom& g, int omega, int nb) {
  return (size_t)2 * g.B * g.H * (2 * nb + 1) * arm_n_pad(g, omega) + RF_ARM_FLAG_FLOATS;
}

cudaError_t rf_launch_arm(const RfGeom& g, int sample_mode, int omega, float alpha, int nb, const int* ws_list,
                          const int* wf_list, const __nv_bfloat16* q, const __nv_bfloat16* k, int32_t* head_class,
                          int32_t* head_window, float* recall, float* recall_plus, float* scratch, int32_t* dev_status,
                          cudaStream_t st, bool selftest_abandon, RfDecision* later) {
  const bool plus = head_window != nullptr;
  const int NB = plus ? ARM_MAX_NB : 1;           // windows the kernel has room for; it evaluates the first nb
  if (nb < 1 || nb > NB) return cudaErrorInvalidValue;
  ArmWindows win;
  win.n = nb;
  for (int i = 0; i < ARM_MAX_NB; ++i) {
    win.ws[i] = ws_list[i < nb ? i : nb - 1];
    win.wf[i] = wf_list[i < nb ? i : nb - 1];
  }
  const int n_pad = arm_n_pad(g, omega);
  const int n_glb = rf_cdiv(g.Nv, omega), n_loc = g.S;
  const int heads = g.B * g.H;
  const int t_glb = rf_cdiv(n_glb, ARM_TILE), t_loc = rf_cdiv(n_loc, ARM_TILE), t_pad = t_glb > t_loc ? t_glb : t_loc;
  float* end = scratch + (size_t)2 * heads * (2 * NB + 1) * n_pad;
  int32_t* arm_flag = reinterpret_cast<int32_t*>(end);
  const size_t sums = (size_t)heads * (2 * NB + 1) * t_pad;     // of one sample; t_pad <= n_pad / 64, so both fit
  double* sums_loc = reinterpret_cast<double*>(end) - sums;
  double* sums_glb = sums_loc - sums;
  const bool alg1 = sample_mode == RF_SAMPLE_ALG1;
  const bool tex = !plus && recall != nullptr;   // the Textural recall is a diagnostic: Algorithm 1 does not use it
  const size_t row_bytes = (size_t)g.D * 2, head_bytes = (size_t)g.N * g.D * 2;
  ArmMaps maps;
  bool ok = rf_encode_rows_map(&maps.q[0], q, g.D, n_glb, row_bytes * omega, head_bytes, heads) &&
            rf_encode_rows_map(&maps.k[0], k, g.D, n_glb, row_bytes * omega, head_bytes, heads) &&
            rf_encode_rows_map(&maps.q[1], q, g.D, n_loc, row_bytes, head_bytes, heads) &&
            rf_encode_rows_map(&maps.k[1], k, g.D, n_loc, row_bytes, head_bytes, heads);
  if (!ok) return cudaErrorUnknown;
  ArmSample s0, s1;
  s0.n = n_glb; s0.stride = omega; s0.tiles = t_glb;
  s0.want_t = alg1 ? 0 : 1; s0.want_s = 1; s0.out = sums_glb;
  s1.n = n_loc; s1.stride = 1; s1.tiles = alg1 ? t_loc : 0;
  s1.want_t = 1; s1.want_s = 0; s1.out = sums_loc;
  cudaError_t e = cudaSuccess;
#ifdef RF_BOUNDS_CHECK
  e = cudaMemsetAsync(arm_flag, 0, sizeof(int32_t), st);
  if (e != cudaSuccess) return e;
#endif
  if (selftest_abandon) {
    e = rf_launch(rf_arm_set_flag_kernel, dim3(1), 1, 0, st, arm_flag, (int)RF_ERR_TIMEOUT);
  } else
  switch (g.D) {
    case 64: e = launch_arm_n<64>(plus, tex, maps, g, s0, s1, win, t_pad, arm_flag, st); break;
    case 96: e = launch_arm_n<96>(plus, tex, maps, g, s0, s1, win, t_pad, arm_flag, st); break;
    case 128: e = launch_arm_n<128>(plus, tex, maps, g, s0, s1, win, t_pad, arm_flag, st); break;
    default: e = cudaErrorInvalidValue;
  }
  if (e != cudaSuccess) return e;
  RfDecision d;
  d.nb = NB; d.nb_user = nb;
  d.n_loc = n_loc; d.n_glb = n_glb;
  d.t_loc = t_loc; d.t_glb = t_glb; d.t_pad = t_pad;
  d.local_t = alg1;
  d.two_mask = g.two_mask;
  d.alpha = alpha;
  for (int i = 0; i < ARM_MAX_NB; ++i) { d.ws[i] = win.ws[i]; d.wf[i] = win.wf[i]; }
  d.loc = sums_loc; d.glb = sums_glb;
  d.arm_flag = arm_flag;
  d.head_class = head_class; d.head_window = head_window;
  d.recall = recall; d.recall_plus = recall_plus;
  d.dev_status = dev_status;
  if (later != nullptr) {
    *later = d;
    return cudaSuccess;
  }
  return rf_launch(rf_arm_decide_kernel, dim3(heads), 32, 0, st, d);
}

// ------------------------------------------------------------------------------------------------
// Entry point for callers that can neither pass a workspace nor allocate one: ARM's scratch is a
// fixed array in this library's device image.
// ------------------------------------------------------------------------------------------------
static __device__ __align__(256) float g_arm_static_scratch[RF_ARM_STATIC_SCRATCH_FLOATS];

namespace {
// Device address of g_arm_static_scratch per device.  In host code the array's name is only a
// handle for the runtime, not a pointer a kernel may use; the address comes from cudaGetSymbolAddress
// with the device in question current.
float* static_scratch_ptr(int dev, cudaError_t* err) {
  static float* ptrs[64] = {};
  *err = cudaSuccess;
  if (dev < 0 || dev >= 64) { *err = cudaErrorInvalidDevice; return nullptr; }
  if (ptrs[dev] == nullptr) {
    void* p = nullptr;
    *err = cudaGetSymbolAddress(&p, g_arm_static_scratch);
    if (*err != cudaSuccess) return nullptr;
    ptrs[dev] = static_cast<float*>(p);
  }
  return ptrs[dev];
}
}  // namespace

extern "C" rf_status rf_arm_classify_noalloc(const rf_shape* shape, const rf_params* params, const void* q,
                                             const void* k, int32_t* head_class, float* recall, int32_t* dev_status,
                                             void* cuda_stream) {
  RfGeom g;
  rf_status st = rf_checked_geom(shape, params, &g);
  if (st != RF_OK) return st;
  if (g.D != 64 && g.D != 96 && g.D != 128) return RF_ERR_UNSUPPORTED;
  if (q == nullptr || k == nullptr || head_class == nullptr) return RF_ERR_INVALID_ARG;
  if ((reinterpret_cast<uintptr_t>(q) & 15u) != 0 || (reinterpret_cast<uintptr_t>(k) & 15u) != 0) return RF_ERR_INVALID_ARG;
  if (rf_arm_scratch_floats(g, params->sample_stride, 1) > (size_t)RF_ARM_STATIC_SCRATCH_FLOATS)
    return RF_ERR_STATIC_SCRATCH_TOO_SMALL;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return RF_ERR_CUDA;
  cudaError_t e;
  float* scratch = static_scratch_ptr(dev, &e);
  if (scratch == nullptr) return RF_ERR_CUDA;
  e = rf_launch_arm(g, params->sample_mode, params->sample_stride, params->alpha, 1, &g.ws, &g.wf,
                    static_cast<const __nv_bfloat16*>(q), static_cast<const __nv_bfloat16*>(k), head_class, nullptr, recall,
                    nullptr, scratch, dev_status, static_cast<cudaStream_t>(cuda_stream));
  return e == cudaSuccess ? RF_OK : RF_ERR_CUDA;
}
