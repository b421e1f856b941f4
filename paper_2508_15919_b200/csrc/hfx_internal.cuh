// Internal declarations shared by the kernels of the scheduler library.
// Integer nanoseconds everywhere; nothing here is floating point.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "hfx.h"

#define HFX_MAX_CLASSES 64
#define HFX_MAX_REPLICAS 65536
#define HFX_MAX_ROWS (INT64_C(1) << 27)

// phases of the key (2 bits)
#define PH_RUNNING 0
#define PH_QUEUED 1
#define PH_INACTIVE 3

// kinds of a regrouped record
#define KIND_RUNNING 0  // in flight
#define KIND_QUEUED 1   // arrived and waiting
#define KIND_FUTURE 2   // QUEUED but not arrived yet (only matters for the idle clock jump)
#define KIND_DEAD 3     // DONE, REJECTED or a row with bad data

#define ROWFLAG_BADREP 4  // row bound to no replica (bucket R)

// "no bound" marker of a slack base
#define BASE_UNBOUNDED INT64_MAX

// Scheduler constants, passed by value to every kernel (lives in the constant bank).
struct HfxParams {
  int64_t c0, c1, c2, d0, d1, d2;
  int64_t ttft[HFX_MAX_CLASSES];
  int64_t tpot[HFX_MAX_CLASSES];
  uint8_t prio[HFX_MAX_CLASSES];
  int32_t n_classes;
  int32_t n_replicas;
  int32_t budget_mode;
  int32_t weight_max;
  int32_t first_fit;      // admission variant: every request is tried against what is left of the budget
};

// One row after regrouping by replica: everything the per-replica kernel needs, 32 bytes
// (one L2 sector), so that kernel never goes back to the table for reads.
struct __align__(32) HfxRec {
  int64_t base;      // slack before the per-replica shift (see ReplicaPlan); the final 48-bit key for a queued row on a
                     // colocated / prefill replica; arrival for KIND_FUTURE
  int32_t req_id;
  int32_t row;
  int32_t prompt;
  int32_t gen;
  int32_t output_len;
  uint8_t cls, kind, prio, pad;
};
static_assert(sizeof(HfxRec) == 32, "record is one 32-byte sector");

// Compact record of an ACTIVE row as the tile front end leaves it (16 bytes, a uint4):
//   x, y  slack base (int64, as HfxRec::base); for a queued row on a colocated / prefill replica the row's final
//         48-bit key (phase | prio | clamped slack) instead, which needs nothing from the running batch
//   z     prompt_len<25> | kind<1> (KIND_RUNNING / KIND_QUEUED) | prio<6>
//   w     gen<25> | class<6>
// The row index travels beside it (16-bit index inside the tile); req_id and output_len are fetched
// from the table by the few paths that need them.
#define CREC_LEN_MASK 0x1ffffffu
#define CREC_KIND_SHIFT 25
#define CREC_PRIO_SHIFT 26
#define CREC_CLS_SHIFT 25
#define HFX_FRONT_SMEM (220 * 1024)      // dynamic shared memory the tile kernel may use

#include <vector>

enum { KSLOT_COUNT = 0, KSLOT_COLSCAN, KSLOT_OFFSETS, KSLOT_REGROUP, KSLOT_SEG_SMALL, KSLOT_SEG_MED, KSLOT_BIG, KSLOT_SIM, KSLOT_SCALE, KSLOT_FRONT, KSLOT_DISPATCH, KSLOT_SLOMAP, KSLOT_PD, KSLOT_METRICS };

// tiling of the front end: one tile per block, at most 8192 rows (16-bit indices inside a tile)
#define HFX_TILE_ROWS_MAX 8192
#define HFX_TILE_MATRIX_MAX (INT64_C(8) << 20)   // entries of the tile matrix (64 MiB), the tiles of one round of the SMs left out
#define HFX_TILE_REPLICAS_MAX 4095               // replicas whose counters fit in shared memory (12-bit bucket ids)
// Replicas up to which a tile notes the next arrival of each (8 bytes a replica, over the tile's slots); beyond them an idle replica's rows are
// looked through instead.  1 M rows, with notes / without: ten steps over 1024 replicas 695 / 709 us, 2048 993 / 967, 3000 1260 / 1193, 4095
// 1770 / 1552 (the matrix of notes is written and read in every step, and from about 2600 replicas on it makes the tiles lower); three ticks of the
// scaling loop, whose replicas have long lists of finished rows, 1024 1351 / 1670, 2048 1929 / 2215, 3000 2413 / 2253, 4094 3435 / 2578.
#define HFX_NEXT_REPLICAS_MAX 2047
#define HFX_WAIT_LIMIT (1u << 22)                // polls of a grid barrier before the kernel gives up (about two seconds)

struct HfxBracket { cudaEvent_t a, b; int slot; };

struct hfx_sched {
  HfxParams p;
  int64_t max_rows;
  int n_sm;
  cudaStream_t stream;
  int64_t launches;
  int profiling;
  std::vector<HfxBracket> *brackets;
  // device
  hfx_replica_cfg *d_cfg;   // [R]
  uint8_t *d_mode;          // [R] replica modes, one byte each
  uint32_t *d_status;       // sticky status word
  uint32_t *d_seg_count;    // [R+2] rows per replica (+ the bad-replica bucket R)      (fallback front end)
  uint32_t *d_act_count;    // [R+2] active rows (in flight or in the visible queue) per replica    (fallback)
  uint32_t *d_seg_begin;    // [R+2] exclusive prefix of d_seg_count                      (fallback)
  uint32_t *d_cursor;       // [2][R+2] fill cursors of the fallback regroup (active, inactive)
  uint8_t *d_rowflag;       // [max_rows] kind of every row (KIND_*), ROWFLAG_BADREP for a bad replica id
  uint32_t *d_flags;        // [4],[5] "ordered" of the tile front end by parity
  HfxRec *d_rec;            // [max_rows] contiguous records: written by the fallback regroup, or gathered from the
                            // slabs by the blocks of larger replicas
  uint64_t *d_big_hi;       // sort scratch of oversize segments
  uint32_t *d_big_lo;
  // tile front end (see hfx_front.cu)
  uint4 *d_slab_rec;        // [tiles_max * tile_rows] records of active rows, tile-major
  uint16_t *d_slab_idx;     // [tiles_max * tile_rows] local row indices, tile-major, grouped by replica
  uint2 *d_M;               // [tiles_max][R+1] where each replica's rows sit in a tile's slabs
  int64_t *d_next;          // [tiles_max][R+1] earliest arrival still to come of each replica in a tile (up to HFX_NEXT_REPLICAS_MAX replicas)
  uint16_t *d_inact;        // [tiles_max][front_inact_ld(R+1)] inactive rows of each replica in a tile
  unsigned long long *d_tot;// [2][R+2] rows | active rows << 32 per replica, by parity
  int32_t tiles_max;        // matrix rows allocated (0: fallback front end only)
  uint32_t tot_parity;      // which half of d_tot / which "ordered" word the next tile front end uses
  int64_t horizon;          // commit horizon of the following steps (INT64_MAX: none)
  uint32_t wait_limit;      // polls of a device-side wait (HFX_WAIT_LIMIT unless set)
  int front_enabled;        // 0: use the fallback front end (global counters) even where the tile front end fits
  void *dispatch_ws;                   // workspace of hfx_dispatch_step, allocated by its first call
  unsigned char *d_sim_scratch;        // rows of long traces in hfx_sim_run (allocated by the first call that needs it)
  size_t sim_scratch_bytes;
  unsigned long long *d_att;           // totals of hfx_attainment, zero between its calls (in the allocation of d_flags)
  void *d_slo;                         // per-priority table of hfx_slo_map
  uint32_t slo_parity;                 // which copy of its first rows the next call uses
  void *d_pd;                          // moved counter, wake-up times and busy flags of hfx_pd_migrate, zero between its calls
  bool pd_unsettled;                   // a call launched its first kernel and not the second, which clears them
};

// ---- latency predictor -------------------------------------------------------------------
__device__ __forceinline__ int64_t dev_Ep(const HfxParams &p, int64_t t) { return p.c0 + p.c1 * t + p.c2 * t * t; }
__device__ __forceinline__ int64_t dev_Ed(const HfxParams &p, int64_t b, int64_t kv) { return p.d0 + p.d1 * b + p.d2 * kv; }

__device__ __forceinline__ int64_t dev_clamp_slack(int64_t s) {
  return s < HFX_SLACK_MIN ? HFX_SLACK_MIN : (s > HFX_SLACK_MAX ? HFX_SLACK_MAX : s);
}

// phase<2> | prio<6> | (clamp(slack) + 2^39)<40>  -- the low 48 bits of the key
__device__ __forceinline__ uint64_t dev_key48(int phase, int prio, int64_t slack) {
  return ((uint64_t)phase << 46) | ((uint64_t)prio << 40) | (uint64_t)(dev_clamp_slack(slack) + (INT64_C(1) << 39));
}

// Per-replica quantities of one step, computed once per replica.
struct ReplicaPlan {
  int64_t now, mat, start;
  int64_t n_run, sum_kv, n_eff, kv_eff;
  int64_t tpot_eff;   // strictest TPOT of the running batch (HFX_INF if none)
  int64_t e_d;
  int64_t budget;
  int64_t shift_run;  // slack of a running row = base - shift_run      (now + E_d)
  int64_t shift_q;    // slack of a queued row  = base - shift_q        (earliest start; + predicted TPOT base on DECODE)
  int64_t tpot_q0;    // predicted TPOT of a queued row = tpot_q0 + d2 * (prompt_len + gen)
  int32_t mode, token_cap, batch_cap;
};

// Largest E_p with 2 E_p + k E_d <= TTFT, k = E_p / (TPOT - E_d)  (worst-case TTFT bound
// behind Eq. 3).  HFX_INF without a TTFT bound, -1 when TPOT <= E_d.
__device__ inline int64_t dev_epmax(int64_t min_ttft, bool decoding, int64_t min_tpot, int64_t e_d) {
  if (min_ttft == HFX_INF) return HFX_INF;
  if (!decoding) return min_ttft / 2;
  if (min_tpot <= e_d) return -1;
  const uint64_t x = (uint64_t)min_ttft, y = (uint64_t)(min_tpot - e_d), den = (uint64_t)(2 * min_tpot - e_d);
  if (__umul64hi(x, y) == 0) return (int64_t)((x * y) / den);     // the product fits 64 bits (the usual case)
  return (int64_t)(((unsigned __int128)x * y) / den);
}

// Largest n in [0, cap] with E_p(n) <= epmax (Eq. 3 on the general prefill model), 0 if none.
__device__ inline int64_t dev_nsafe(const HfxParams &p, int64_t epmax, int64_t cap) {
  if (epmax == HFX_INF) return cap;
  if (dev_Ep(p, 0) > epmax) return 0;
  int64_t lo = 0, hi = cap;
  while (lo < hi) {
    int64_t mid = lo + (hi - lo + 1) / 2;
    if (dev_Ep(p, mid) <= epmax) lo = mid; else hi = mid - 1;
  }
  return lo;
}

__device__ inline int64_t dev_min_over_mask(const int64_t *v, uint64_t mask) {
  int64_t m = HFX_INF;
  while (mask) {
    int c = __ffsll((long long)mask) - 1;
    mask &= mask - 1;
    if (v[c] > 0 && v[c] < m) m = v[c];
  }
  return m;
}

// Dispatching step 2 for one replica: E_d of the running batch and the safe budget.
__device__ inline void dev_plan(const HfxParams &p, const hfx_replica_cfg &cfg, int64_t now, int64_t mat,
                                int64_t n_run, int64_t sum_kv, uint64_t mask_run, uint64_t mask_q,
                                ReplicaPlan &pl) {
  pl.now = now; pl.mat = mat; pl.start = now > mat ? now : mat;
  pl.mode = cfg.mode; pl.token_cap = cfg.token_cap; pl.batch_cap = cfg.batch_cap;
  pl.n_run = n_run; pl.sum_kv = sum_kv;
  const int64_t min_tpot = dev_min_over_mask(p.tpot, mask_run);
  const int64_t min_ttft = dev_min_over_mask(p.ttft, mask_q);
  const int64_t min_tpot_q = dev_min_over_mask(p.tpot, mask_q);
  const bool prefill = cfg.mode == HFX_PREFILL;
  pl.n_eff = prefill ? 0 : n_run;
  pl.kv_eff = prefill ? 0 : sum_kv;
  pl.tpot_eff = prefill ? HFX_INF : min_tpot;
  pl.e_d = pl.n_eff > 0 ? dev_Ed(p, pl.n_eff, pl.kv_eff) : 0;
  int64_t budget;
  if (cfg.mode == HFX_DECODE) {
    const int64_t T = (n_run > 0 && min_tpot < HFX_INF) ? min_tpot : min_tpot_q;
    if (p.budget_mode == HFX_BUDGET_CAP_ONLY || T == HFX_INF) budget = HFX_INF;
    else {
      const int64_t room = T - dev_Ed(p, n_run, sum_kv);
      budget = room > 0 ? room : 0;
    }
  } else {
    const int64_t cap_left = cfg.token_cap - pl.n_eff > 0 ? cfg.token_cap - pl.n_eff : 0;
    int64_t n_safe;
    if (p.budget_mode == HFX_BUDGET_CAP_ONLY) n_safe = cfg.token_cap;
    else n_safe = dev_nsafe(p, dev_epmax(min_ttft, pl.n_eff > 0 && pl.tpot_eff < HFX_INF, pl.tpot_eff, pl.e_d), cfg.token_cap);
    budget = n_safe < cap_left ? n_safe : cap_left;
  }
  if (now < mat) budget = 0;
  pl.budget = budget;
  pl.tpot_q0 = dev_Ed(p, pl.n_eff + 1, pl.kv_eff);
  pl.shift_run = now + pl.e_d;
  pl.shift_q = pl.start + (cfg.mode == HFX_DECODE ? pl.tpot_q0 : 0);
}

// The same plan computed by a whole warp (all 32 lanes call with the same arguments and get the same
// result).  The class minima come from tables in shared memory; the largest safe n comes from a 32-way search
// on the bound itself, E_p(n) * (2 TPOT - E_d) <= TTFT * (TPOT - E_d), compared in 128 bits: for
// integer E_p that is the same set of n as E_p(n) <= floor(TTFT (TPOT - E_d) / (2 TPOT - E_d)), and no
// division is needed.
// Strictest SLO of a set of classes: every class has a rank by its bound (HFX_MAX_CLASSES: none) and the bounds are kept by
// rank, so it is a minimum over small integers (one reduction) and a look.
struct ClassTab {
  int64_t ttft[HFX_MAX_CLASSES + 1], tpot[HFX_MAX_CLASSES + 1];      // by rank; the last one: unbounded
  uint8_t rank_ttft[HFX_MAX_CLASSES], rank_tpot[HFX_MAX_CLASSES];
};
// (threads 0 .. HFX_MAX_CLASSES of a block; the block synchronises before use)
__device__ __forceinline__ void class_tab_init(const HfxParams &p, ClassTab &t, int tid) {
  if (tid == HFX_MAX_CLASSES) { t.ttft[tid] = HFX_INF; t.tpot[tid] = HFX_INF; }
  if (tid >= HFX_MAX_CLASSES) return;
  const int64_t a = tid < p.n_classes ? p.ttft[tid] : 0, b = tid < p.n_classes ? p.tpot[tid] : 0;
  int ra = 0, rb = 0;
  for (int k = 0; k < p.n_classes; k++) {
    const int64_t x = p.ttft[k], y = p.tpot[k];
    ra += x > 0 && (x < a || (x == a && k < tid)) ? 1 : 0;
    rb += y > 0 && (y < b || (y == b && k < tid)) ? 1 : 0;
  }
  t.rank_ttft[tid] = (uint8_t)(a > 0 ? ra : HFX_MAX_CLASSES); t.rank_tpot[tid] = (uint8_t)(b > 0 ? rb : HFX_MAX_CLASSES);
  if (a > 0) t.ttft[ra] = a;
  if (b > 0) t.tpot[rb] = b;
}
__device__ __forceinline__ int64_t warp_min_over_mask(const int64_t *by_rank, const uint8_t *rank, uint64_t mask, int lane) {
  const uint32_t x = (mask >> lane) & 1ull ? rank[lane] : HFX_MAX_CLASSES, y = (mask >> (lane + 32)) & 1ull ? rank[lane + 32] : HFX_MAX_CLASSES;
  return by_rank[__reduce_min_sync(0xffffffffu, x < y ? x : y)];
}

// Largest n in [0, cap] with E_p(n) * den <= num (num = nh:nl as 128 bits, den > 0), 0 if none.
__device__ inline int64_t warp_nsafe(const HfxParams &p, uint64_t nh, uint64_t nl, uint64_t den, int64_t cap, int lane) {
  auto fits = [&](int64_t n) {
    const uint64_t ep = (uint64_t)dev_Ep(p, n);
    const uint64_t ph = __umul64hi(ep, den), pl = ep * den;
    return ph < nh || (ph == nh && pl <= nl);
  };
  if (!fits(0)) return 0;
  int64_t lo = 0, hi = cap;          // fits(lo); the answer lies in [lo, hi]
  while (lo < hi) {
    const int64_t step = (int64_t)(((uint64_t)(hi - lo) + 31u) >> 5);
    const int64_t cand = lo + (int64_t)(lane + 1) * step;
    const int m = __popc(__ballot_sync(0xffffffffu, cand <= hi && fits(cand)));     // E_p is monotone: the ones that fit are a prefix
    const int64_t nlo = lo + (int64_t)m * step;
    int64_t nhi = lo + (int64_t)(m + 1) * step - 1;
    if (nhi > hi) nhi = hi;
    lo = nlo; hi = nhi;
  }
  return lo;
}

__device__ inline void warp_plan(const HfxParams &p, const ClassTab &tab, const hfx_replica_cfg &cfg, int64_t now, int64_t mat, int64_t n_run, int64_t sum_kv,
                                 uint64_t mask_run, uint64_t mask_q, ReplicaPlan &pl, int lane) {
  pl.now = now; pl.mat = mat; pl.start = now > mat ? now : mat;
  pl.mode = cfg.mode; pl.token_cap = cfg.token_cap; pl.batch_cap = cfg.batch_cap;
  pl.n_run = n_run; pl.sum_kv = sum_kv;
  const int64_t min_tpot = warp_min_over_mask(tab.tpot, tab.rank_tpot, mask_run, lane);
  const bool prefill = cfg.mode == HFX_PREFILL;
  pl.n_eff = prefill ? 0 : n_run;
  pl.kv_eff = prefill ? 0 : sum_kv;
  pl.tpot_eff = prefill ? HFX_INF : min_tpot;
  pl.e_d = pl.n_eff > 0 ? dev_Ed(p, pl.n_eff, pl.kv_eff) : 0;
  int64_t budget = 0;
  if (now >= mat) {      // before maturity the instance is protected: no budget to work out
    if (cfg.mode == HFX_DECODE) {
      const int64_t T = (n_run > 0 && min_tpot < HFX_INF) ? min_tpot : warp_min_over_mask(tab.tpot, tab.rank_tpot, mask_q, lane);
      if (p.budget_mode == HFX_BUDGET_CAP_ONLY || T == HFX_INF) budget = HFX_INF;
      else {
        const int64_t room = T - dev_Ed(p, n_run, sum_kv);
        budget = room > 0 ? room : 0;
      }
    } else {
      const int64_t cap_left = cfg.token_cap - pl.n_eff > 0 ? cfg.token_cap - pl.n_eff : 0;
      int64_t n_safe;
      if (p.budget_mode == HFX_BUDGET_CAP_ONLY) n_safe = cfg.token_cap;
      else {
        const int64_t min_ttft = warp_min_over_mask(tab.ttft, tab.rank_ttft, mask_q, lane);
        const bool decoding = pl.n_eff > 0 && pl.tpot_eff < HFX_INF;
        if (min_ttft == HFX_INF) n_safe = cfg.token_cap;
        else if (!decoding) n_safe = warp_nsafe(p, 0, (uint64_t)min_ttft, 2, cfg.token_cap, lane);     // 2 E_p <= TTFT
        else if (pl.tpot_eff <= pl.e_d) n_safe = 0;
        else {
          const uint64_t x = (uint64_t)min_ttft, y = (uint64_t)(pl.tpot_eff - pl.e_d);
          n_safe = warp_nsafe(p, __umul64hi(x, y), x * y, (uint64_t)(2 * pl.tpot_eff - pl.e_d), cfg.token_cap, lane);
        }
      }
      budget = n_safe < cap_left ? n_safe : cap_left;
    }
  }
  pl.budget = budget;
  pl.tpot_q0 = dev_Ed(p, pl.n_eff + 1, pl.kv_eff);
  pl.shift_run = now + pl.e_d;
  pl.shift_q = pl.start + (cfg.mode == HFX_DECODE ? pl.tpot_q0 : 0);
}

// Dispatching step 4: maturity time after admitting adm_count requests of adm_cost in total.
__device__ inline int64_t dev_maturity_next(const HfxParams &p, const ReplicaPlan &pl, int64_t adm_count,
                                            int64_t adm_cost, int64_t adm_kv, int64_t *lp_out) {
  int64_t lp = 0, mat_next = pl.mat;
  if (pl.mode == HFX_DECODE) {
    if (pl.now >= pl.mat && pl.n_run + adm_count > 0)
      mat_next = pl.now + dev_Ed(p, pl.n_run + adm_count, pl.sum_kv + adm_kv);
  } else if (adm_count > 0) {
    lp = dev_Ep(p, adm_cost);
    if (pl.mode == HFX_PREFILL) mat_next = pl.now + lp;
    else {
      uint64_t k = 0;
      if (pl.n_eff > 0 && pl.tpot_eff < HFX_INF && pl.tpot_eff > pl.e_d) {
        const uint64_t d = (uint64_t)(pl.tpot_eff - pl.e_d);
        k = ((uint64_t)lp + d - 1) / d;
      }
      // now + lp + k * e_d, saturating at HFX_TIME_MAX (the product may need more than 64 bits)
      const uint64_t ed = (uint64_t)pl.e_d, prod = k * ed;
      const int64_t t = pl.now + lp;                              // |now| <= 2^56, lp < 2^61
      if (__umul64hi(k, ed) != 0 || prod >= (UINT64_C(1) << 63)) mat_next = HFX_TIME_MAX;
      else mat_next = (int64_t)prod > HFX_TIME_MAX - t ? HFX_TIME_MAX : t + (int64_t)prod;
    }
  }
  *lp_out = lp;
  return mat_next;
}

// ---- warp / block primitives ----------------------------------------------------------------
__device__ __forceinline__ int64_t warp_sum_i64(int64_t v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
// the same for values in [0, 2^46): two narrow reductions instead of ten shuffles
__device__ __forceinline__ int64_t warp_sum_wide(int64_t v) {
  return (int64_t)__reduce_add_sync(0xffffffffu, (uint32_t)v & 0xfffffu) + ((int64_t)__reduce_add_sync(0xffffffffu, (uint32_t)(v >> 20)) << 20);
}
__device__ __forceinline__ int64_t warp_min_i64(int64_t v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) { int64_t w = __shfl_xor_sync(0xffffffffu, v, o); v = w < v ? w : v; }
  return v;
}
__device__ __forceinline__ uint64_t warp_or_u64(uint64_t v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v |= __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ int64_t warp_incl_scan_i64(int64_t v, int lane) {
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) { int64_t w = __shfl_up_sync(0xffffffffu, v, o); if (lane >= o) v += w; }
  return v;
}
__device__ __forceinline__ int32_t warp_incl_scan_i32(int32_t v, int lane) {
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) { int32_t w = __shfl_up_sync(0xffffffffu, v, o); if (lane >= o) v += w; }
  return v;
}

// Compare-exchange of sort items, ascending: `hi` alone (items carry their tie-break in the low
// bits) or the 96-bit pair (hi, lo).
template <bool WIDE>
__device__ __forceinline__ void cmp_swap(uint64_t *hi, uint32_t *lo, int i, int j) {
  const uint64_t hi_i = hi[i], hi_j = hi[j];
  if (WIDE) {
    const uint32_t lo_i = lo[i], lo_j = lo[j];
    if (hi_i > hi_j || (hi_i == hi_j && lo_i > lo_j)) { hi[i] = hi_j; hi[j] = hi_i; lo[i] = lo_j; lo[j] = lo_i; }
  } else if (hi_i > hi_j) { hi[i] = hi_j; hi[j] = hi_i; }
}

// First-fit admission along an order of n places, by one warp (all 32 lanes call).  cost_of(q) is the
// cost of the candidate at place q, or -1 where there is none; every candidate is tried in order against
// what is left of `budget` and of `room` (how many more may be taken) and taken if it fits; decide(q, taken)
// is called once for every place.  32 places at a time: the first lane that still fits starts a run, the
// run ends at the first lane that no longer fits behind it (that lane is refused for good), the lanes after
// it are tried again with what is left then.
struct FirstFit { int64_t used = 0, taken = 0; };

template <typename CostF, typename DecideF>
__device__ __forceinline__ void warp_first_fit_32(FirstFit &f, int64_t base, int64_t n, int64_t budget, int64_t room, int lane, CostF cost_of, DecideF decide) {
  const int64_t q = base + lane;
  const int64_t c = q < n ? cost_of(q) : -1;
  uint32_t pending = __ballot_sync(0xffffffffu, c >= 0);
  bool mine = false;
  while (pending) {
    const int64_t rem = budget - f.used, left = room - f.taken;
    const bool me = (pending >> lane) & 1u;
    const uint32_t fit = left > 0 ? __ballot_sync(0xffffffffu, me && c <= rem) : 0u;
    if (!fit) break;
    const int l0 = __ffs(fit) - 1;
    const bool in = me && lane >= l0;
    const int64_t pre = warp_incl_scan_i64(in ? c : 0, lane);
    const int32_t pcnt = warp_incl_scan_i32(in ? 1 : 0, lane);
    const bool ok = in && pre <= rem && (int64_t)pcnt <= left;
    const uint32_t bad = __ballot_sync(0xffffffffu, in && !ok);
    const int l1 = bad ? __ffs(bad) - 1 : 32;            // the run is the pending lanes in [l0, l1)
    const bool take = in && lane < l1;
    if (take) mine = true;
    const uint32_t tm = __ballot_sync(0xffffffffu, take);
    const int last = 31 - __clz(tm);                      // tm has lane l0 at least
    f.used += __shfl_sync(0xffffffffu, pre, last);
    f.taken += __shfl_sync(0xffffffffu, pcnt, last);
    pending = l1 >= 31 ? 0u : (pending & ~((2u << l1) - 1u));
  }
  if (q < n) decide(q, mine);
}

template <typename CostF, typename DecideF>
__device__ __forceinline__ void warp_first_fit(int64_t n, int64_t budget, int64_t room, int lane, CostF cost_of, DecideF decide) {
  FirstFit f;
  for (int64_t base = 0; base < n; base += 32) warp_first_fit_32(f, base, n, budget, room, lane, cost_of, decide);
}

// The same where the smallest cost of every 32 places (HFX_INF: no candidate) is known: only the 32s in which something may
// still fit are looked at, and decide is called for their places alone.
template <typename CostF, typename DecideF>
__device__ __forceinline__ void warp_first_fit(int64_t n, const int64_t *min32, int64_t budget, int64_t room, int lane, CostF cost_of, DecideF decide) {
  FirstFit f;
  const int n32 = (int)((n + 31) >> 5);
  for (int k = 0; k < n32 && f.taken < room;) {
    const uint32_t some = __ballot_sync(0xffffffffu, k + lane < n32 && min32[k + lane] <= budget - f.used);
    if (!some) { k += 32; continue; }
    k += __ffs(some) - 1;
    warp_first_fit_32(f, (int64_t)k * 32, n, budget, room, lane, cost_of, decide);
    k++;
  }
}

// The code of a runtime call.  A failed call's error is read here: left behind, the next call's check would find it.
inline int cuda_rc(cudaError_t e) {
  if (e == cudaSuccess) return HFX_OK;
  cudaGetLastError();
  return HFX_E_CUDA;
}

// Brackets one kernel launch with events when profiling is on; counts the launch either way.
struct KernelScope {
  hfx_sched *s; HfxBracket br; bool on; cudaStream_t st;
  KernelScope(hfx_sched *s_, int slot, cudaStream_t stream = nullptr) : s(s_), on(false), st(stream ? stream : s_->stream) {
    s->launches++;
    if (s->profiling && s->brackets) {
      br.slot = slot;
      if (cudaEventCreate(&br.a) == cudaSuccess && cudaEventCreate(&br.b) == cudaSuccess) {
        cudaEventRecord(br.a, st);
        on = true;
      }
    }
  }
  ~KernelScope() {
    if (on) { cudaEventRecord(br.b, st); s->brackets->push_back(br); }
  }
};

// ---- kernel argument blocks ------------------------------------------------------------------
// the fallback front end (global counters; tables with more replicas than the tile front end takes)
struct RegroupArgs {
  const int32_t *replica_id; const uint8_t *class_id; const uint8_t *state; const int32_t *prompt_len;
  const int32_t *output_len; const int32_t *gen; const int64_t *arrival; const int64_t *first_token;
  const int32_t *req_id; const int32_t *weight;
  const int64_t *now; const int64_t *mat; const hfx_replica_cfg *cfg; const uint8_t *mode;
  int64_t *pred_ttft;    // optional output
  int64_t n;
  // per-row outputs written by the regroup itself
  int64_t *slack; int64_t *pred_tpot; uint64_t *key; int32_t *order; uint8_t *admit; int32_t *admitted_rows;
  uint32_t commit;
};

// the tile front end
// entries per row of the matrix of inactive rows (rows start on 16 bytes)
__host__ __device__ constexpr int front_inact_ld(int R1) { return (R1 + 7) & ~7; }

struct FrontArgs {
  const int32_t *replica_id; const uint8_t *class_id; const uint8_t *state; const int32_t *prompt_len; const int32_t *gen;
  const int64_t *arrival; const int64_t *first_token; const int32_t *req_id; const int32_t *weight;
  const int64_t *now; const int64_t *mat; const uint8_t *mode;
  int64_t n; int32_t tile_rows; int32_t n_tiles; int32_t by_warp;
  // per-row outputs, written in row order
  int64_t *slack; int64_t *pred_ttft; int64_t *pred_tpot; uint64_t *key; uint8_t *admit; uint8_t *rowflag;
  // the slabs
  uint4 *slab_rec; uint16_t *slab_idx; uint2 *M; int64_t *next; uint16_t *inact; unsigned long long *tot; unsigned long long *tot_next;
  uint32_t *ordered; uint32_t *ordered_next; uint32_t *status;
};

struct SegArgs {
  // read-only table columns (fetched by row where a path needs them)
  const int64_t *arrival; const int32_t *req_id; const int32_t *output_len;
  // table columns written by COMMIT
  uint8_t *state; int32_t *gen; int64_t *first_token; int64_t *last_token; int64_t *finish;
  // replica state
  int64_t *now; int64_t *mat; const hfx_replica_cfg *cfg;
  // outputs
  int64_t *slack; int64_t *pred_tpot; uint64_t *key; int32_t *order; int32_t *seg_off; uint8_t *admit; int32_t *admitted_rows;
  int64_t *budget; int64_t *e_d; int32_t *n_run; int64_t *sum_kv; int64_t *adm_cost; int32_t *adm_count;
  int64_t *maturity_next;
  uint32_t flags;
  int64_t horizon;           // a replica whose clock is past it sits the commit out
};

// host-side launchers implemented in the .cu files
void hfx_front_shape(const hfx_sched *s, int64_t n, int32_t *tile_rows, int32_t *n_tiles);
int hfx_launch_front(hfx_sched *s, const FrontArgs &fa);
int hfx_launch_regroup(hfx_sched *s, const RegroupArgs &ra, int32_t *seg_off);
int hfx_launch_replicas(hfx_sched *s, const SegArgs &sa, int64_t n, bool slabs);
int hfx_launch_step(hfx_sched *s, const hfx_table *t, const hfx_replica_state *st, const hfx_step_out *o, uint32_t flags);
int hfx_launch_dispatch(hfx_sched *s, const hfx_table *t, int64_t now_ns, const int64_t *maturity, const hfx_dispatch_out *o,
                        int32_t cap_max, bool d_stage);
void hfx_dispatch_release(hfx_sched *s);
void hfx_sim_release(hfx_sched *s);
int hfx_launch_slo_map(hfx_sched *s, int32_t n_prio, const hfx_slo_window *win, const hfx_slo_bounds *b, int64_t *last_queue,
                       const int32_t *pending, const int32_t *new_prio, int64_t n_new, int64_t *ttft_out, int64_t *tpot_out);
size_t hfx_slomap_workspace_bytes();
int hfx_launch_pd_migrate(hfx_sched *s, const hfx_table *t, int32_t *replica_id, int64_t *now, const int32_t *pair, int64_t x0,
                          int64_t x1, int32_t *n_moved);
size_t hfx_pd_workspace_bytes(int n_replicas);
size_t hfx_attainment_workspace_bytes();
int hfx_launch_attainment(hfx_sched *s, const hfx_table *t, int64_t *out);
int hfx_launch_fleet_apply(hfx_sched *s, int64_t now, const int32_t *decision, const int64_t *used_blocks,
                           const int64_t *cold, const hfx_fleet *f, int64_t *clock, int64_t *maturity, int64_t *cost);
int hfx_launch_dispatch_bind(hfx_sched *s, int64_t n, int64_t now, const int32_t *assign, const int32_t *adm_count,
                             int32_t *replica_id, int64_t *clock);
