// hfx_dispatch_step: the four dispatching steps of Sec. 3.3.1 over a shared global queue, for every
// colocated or P-stage instance whose maturity time has come, in maturity order; and, on a scheduler with
// D-stage instances, the same steps for the D stage (the Migrator): the queue of prefilled requests, the D instances
// in maturity order, budgets and costs in time.  Neither stage needs anything of the other's result, so both go
// through the same four launches: the two queues are ordered as one, the stage above the priority.
//
//   k_disp_scan     one streaming pass over the table: the running batch of every instance (count, context tokens,
//                   classes), slack of the rows of either queue, those rows as 16-byte items (stage, priority, slack | tie | row)
//   k_disp_sort     cooperative, a block per SM: E_d and budget of every instance, the matured instances by (maturity,
//                   index), the queue in order, the running totals of its costs and entries
//   k_disp_chain    a block per stage: one warp hands consecutive runs of the queue to the instances in order; then the new
//                   maturity times
//   k_disp_assign   the request -> instance binding of every dispatched row; counters cleared for the next call
#include <new>
#include <string.h>

#include "hfx_internal.cuh"

#define SCAN_THREADS 1024
#define SCAN_THREADS_FEW 256
#define SCAN_SMEM_REPLICAS 512      // up to here a block adds up the running batches in shared memory first: with few instances the
                                    // global counters queue up (R x blocks counters are flushed, so not for large fleets)
#define SCAN_SMEM_ROWS 32768        // rows per block up to which its 32-bit sums cannot overflow
#define SORT_THREADS 1024
#define DISP_CLASSES 128            // stage<1> | priority<6>
#define DISP_SAMPLES 2048           // items of the sample at most; one in 64 of the queue
#define DISP_STEP 4                 // samples per splitter interval
#define DISP_SPLITS (DISP_SAMPLES / DISP_STEP + 3 * DISP_CLASSES)
#define DISP_SUB 8                  // bins an interval is divided into evenly
#define DISP_BINS (DISP_SPLITS * DISP_SUB)
#define DISP_SMALL 4096             // a queue of so many entries is ordered by comparing all with all
#define DISP_TILE 4096              // queue entries a block orders at a time (whole bins: up to the fullest bin more, DISP_TILE_MAX in all)
#define DISP_TILE_MAX (DISP_TILE + 1024)
#define DISP_TILE_MIN 512
#define DISP_BIN_MAX (DISP_TILE_MAX - DISP_TILE_MIN)      // fuller bins send the queue to the radix sort
#define DISP_FINE 4096              // bins of a tile
// Items of a fine bin that are compared all with all; a fuller one (slacks crowded beside a gap, equal ones whose ids share their leading bits) goes
// through a sorting network of the block.  40,960 rows, so many of them within 2 ns, compared / network: 200 67.0 / 61.8 us, 1000 205 / 72, 3000 857 /
// 117, 4500 1884 / 162.  Many bins of a hundred (100,000 equal slacks, ids of 256 front ends): 66.8 us, with the line at 64 items 137.
#define DISP_FINE_MAX 128
#define DISP_TILES_CHAIN 1024       // tiles whose totals the chain adds up itself; beyond them they are added to the running totals
#define SORT_SMEM (DISP_TILE_MAX * 22 + (DISP_FINE + 4) * 4 + (DISP_BINS + 4) * 4 + DISP_SPLITS * 16)
#define VAL_FITS 0x80000000u        // on an ordered row: some instance's budget reaches it (the others are passed over)
#define CHAIN_THREADS 1024
#define CHAIN_CHUNK 4096            // running totals staged in shared memory at a time
#define CHAIN_WIN 256               // and held in registers by the walking warp, eight per lane
#define CHAIN_BATCH 24              // instances between two looks at whether all went well: as many as the windows before held,
#define CHAIN_BATCH_MIN 4           // between these two
#define ASSIGN_THREADS 256

// words of the control block, zero between calls unless noted
enum { CTL_QMASK = 0, CTL_DMASK, CTL_FALLS, CTL_BMAX0, CTL_BMAX1, CTL_BARRIER, CTL_N0, CTL_N1, CTL_NM0, CTL_NM1, CTL_TAKEN0, CTL_TAKEN1, CTL_ABORT, CTL_ITEMS,
       CTL_IDMAX, CTL_IDMIN_INV, CTL_TILE_ROWS, CTL_TILES,
       CTL_CLASSES = 32, CTL_WORDS = CTL_CLASSES + DISP_CLASSES };
// (minima are kept inverted, so that everything starts at 0; CTL_CLASSES: per class the upper 32 bits of the largest slack, behind them all those of the smallest, inverted)

struct DispWork {
  uint4 *item[2];            // [rows] items (key<47> in x, y; id in z; row in w): [1] as the scan leaves them, [0] by bin
  uint64_t *sorted;          // [DISP_SAMPLES] a sample's places in the order: (stage, priority)<7> | slack<40> | leading bits of the tie<16>
  uint32_t *rank;            // [rows] bin of an item << 16 | place in it
  uint32_t *val;             // [rows] rows of the queue in order, VAL_FITS
  int64_t *prefix;           // [rows] running total of the costs inside a tile (entries that fit some instance)
  int32_t *prefix_cnt;       // [rows] running count of those entries
  int64_t *tile_sum;         // [2][tiles] totals of a tile: cost, entries
  uint32_t *tile_edge;       // [tiles + 1] where each tile starts
  uint32_t *hist;            // [blocks][256] digit counts of a radix pass
  // zero between calls
  uint32_t *n_run; unsigned long long *sum_kv; unsigned long long *mask_run;      // [R]
  unsigned long long *ctl; uint32_t *bin_cnt;
  ReplicaPlan *plan;         // [R]
  int64_t *ord_budget; int32_t *ord_room; int32_t *ord_id;      // [R] matured instances in order, stage 0, then stage 1
  int32_t *run_end;                                               // [R] where its run ends in its stage's queue
  int32_t R, tiles_max;
  uint32_t wait_limit;       // polls of a grid barrier before the kernel gives up
};

struct DispArgs {
  const int32_t *replica_id; const uint8_t *class_id; const uint8_t *state; const int32_t *prompt_len; const int32_t *gen;
  const int64_t *arrival; const int32_t *req_id; const int32_t *weight; const int64_t *first_token;
  int64_t n; int64_t now; int32_t cap_max;
  int32_t d_stage;           // the scheduler has D-stage instances: the Migrator's stage runs too
  int32_t rounds;            // of the scan over the table
  const int64_t *maturity; const hfx_replica_cfg *cfg; const uint8_t *mode;
  // outputs
  int32_t *assign; int32_t *queue_order; int32_t *n_queue; int32_t *inst_order; int32_t *n_mature; int64_t *slack;
  int64_t *budget; int64_t *e_d; int32_t *n_run; int64_t *sum_kv; int64_t *adm_cost; int32_t *adm_count; int64_t *maturity_next;
  uint32_t *status;
};

__device__ __forceinline__ uint64_t item_key(const uint4 x) { return ((uint64_t)x.y << 32) | x.x; }

// what a queue entry takes of an instance's budget: prompt tokens (first stage), decode time d1 + d2 kv (D stage)
__device__ __forceinline__ int64_t disp_cost(const HfxParams &p, const DispArgs &a, uint32_t row, int stage) {
  const int64_t x = a.prompt_len[row];
  return stage ? p.d1 + p.d2 * (x + a.gen[row]) : x;
}

// ------------------------------------------------------------------------------------------------
// k_disp_scan.  Bound by the columns it reads and the three outputs it initialises (54 bytes a row).  Four rows per
// thread with 16-byte loads; a block reserves room for the items of a round of rows with one global atomic (their order
// does not matter: the tie word settles it).
// ------------------------------------------------------------------------------------------------
template <int threads>
__global__ void __launch_bounds__(threads, 1) k_disp_scan(const HfxParams p, const DispArgs a, const DispWork w) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  uint32_t *s_run = reinterpret_cast<uint32_t *>(smem_raw);      // [4 R] requests in flight, context low / high part; (if R is small)
  unsigned long long *s_mask = reinterpret_cast<unsigned long long *>(s_run + 4 * (size_t)p.n_replicas);      // [R]
  __shared__ int64_t s_ttft[HFX_MAX_CLASSES], s_tpot[HFX_MAX_CLASSES];
  __shared__ uint8_t s_prio[HFX_MAX_CLASSES];
  __shared__ uint32_t s_up[2 * DISP_CLASSES];      // of every class the largest slack's upper 32 bits; the smallest's, inverted
  __shared__ uint32_t s_count, s_base, s_idmax, s_idmin_inv;
  __shared__ unsigned long long s_qmask, s_dmask;
  const int tid = threadIdx.x, lane = tid & 31, R = p.n_replicas;
  const bool own = R <= SCAN_SMEM_REPLICAS && (int64_t)a.rounds * threads * 4 <= SCAN_SMEM_ROWS;
  for (int c = tid; c < HFX_MAX_CLASSES; c += threads) {
    s_ttft[c] = c < p.n_classes ? p.ttft[c] : 0;
    s_tpot[c] = c < p.n_classes ? p.tpot[c] : 0;
    s_prio[c] = c < p.n_classes ? p.prio[c] : 63;
  }
  if (own) for (int i = tid; i < R; i += threads) { s_run[4 * i] = 0; s_run[4 * i + 1] = 0; s_run[4 * i + 2] = 0; s_mask[i] = 0; }
  static_assert(threads >= 2 * DISP_CLASSES, "a thread for every bound");
  if (tid < 2 * DISP_CLASSES) s_up[tid] = 0;
  if (tid == 0) { s_count = 0; s_idmax = 0; s_idmin_inv = 0; s_qmask = 0; s_dmask = 0; }
  __syncthreads();
  uint32_t bad = 0;
  unsigned long long qmask = 0, dmask = 0;
  bool falls = false;
  uint32_t idmax = 0, idmin_inv = 0;

  // the item's key of a row, 0 if it is in neither queue; its slack
  auto do_row = [&](int64_t i, int32_t rid, uint32_t cls, uint32_t st, int32_t prompt, int32_t gen, int32_t weight, int64_t arrival,
                    int64_t &slack) -> uint64_t {
    slack = 0;
    bool ok = true;
    if (cls >= (uint32_t)p.n_classes) { bad |= HFX_ST_BAD_CLASS; ok = false; }
    if ((uint32_t)prompt > HFX_MAX_TOKENS || (uint32_t)gen > HFX_MAX_TOKENS) { bad |= HFX_ST_BAD_LEN; ok = false; }
    if (!ok || st > HFX_RUNNING) return 0;
    int stage = 0;
    if (st == HFX_RUNNING) {
      if ((uint32_t)rid >= (uint32_t)R) { bad |= HFX_ST_BAD_REPLICA; return 0; }
      const int64_t kv = (int64_t)prompt + gen;
      if (own) {
        atomicAdd(&s_run[4 * rid], 1u); atomicAdd(&s_run[4 * rid + 1], (uint32_t)kv & 0xffffu); atomicAdd(&s_run[4 * rid + 2], (uint32_t)(kv >> 16));
        if (!((s_mask[rid] >> cls) & 1ull)) atomicOr(&s_mask[rid], 1ull << cls);
      } else {
        atomicAdd(&w.n_run[rid], 1u); atomicAdd(&w.sum_kv[rid], (unsigned long long)kv); atomicOr(&w.mask_run[rid], 1ull << cls);
      }
      // a prefilled request: in flight on a P-stage instance, its first token produced by now
      if (!a.d_stage || a.mode[rid] != HFX_PREFILL) return 0;
      const int64_t ft = a.first_token[i];
      if (ft > a.now) return 0;
      const int64_t tpot = s_tpot[cls];
      slack = tpot > 0 ? ft + ((int64_t)gen + 1) * tpot - a.now - dev_Ed(p, 1, kv) : HFX_SLACK_MAX;
      dmask |= 1ull << cls;
      stage = 1;
    } else {
      if (arrival > a.now || prompt > a.cap_max) return 0;
      const int64_t ttft = s_ttft[cls];
      slack = ttft > 0 ? ttft - ((a.now - arrival) + dev_Ep(p, prompt)) : HFX_SLACK_MAX;
      qmask |= 1ull << cls;
    }
    uint32_t prio = s_prio[cls];
    if (p.weight_max > 0) prio = weight >= p.weight_max ? 0 : (weight <= p.weight_max - 62 ? 62 : p.weight_max - weight);
    return (1ull << 47) | ((uint64_t)(stage * 64 + prio) << 40) | (uint64_t)(dev_clamp_slack(slack) + (INT64_C(1) << 39));      // (bit 47 marks it; stored without)
  };
  auto item_of = [&](uint64_t key, int64_t i, int32_t id) -> uint4 {
    const uint32_t uid = (uint32_t)id ^ 0x80000000u;
    idmax = uid > idmax ? uid : idmax; idmin_inv = ~uid > idmin_inv ? ~uid : idmin_inv;
    const uint32_t cl = (uint32_t)(key >> 40) & 127u, up = (uint32_t)(key >> 8);      // (few rows raise a bound: mostly two loads)
    if (up > s_up[cl]) atomicMax(&s_up[cl], up);
    if (~up > s_up[DISP_CLASSES + cl]) atomicMax(&s_up[DISP_CLASSES + cl], ~up);
    return make_uint4((uint32_t)key, (uint32_t)(key >> 32) & 0x7fffu, uid, (uint32_t)i);
  };

  const int64_t n4 = a.n >> 2;
  for (int64_t v0 = (int64_t)blockIdx.x * threads; v0 < n4; v0 += (int64_t)gridDim.x * threads) {
    const int64_t v = v0 + tid;
    uint64_t key[4] = {0, 0, 0, 0};
    int4 id = make_int4(0, 0, 0, 0);
    if (v < n4) {
      const int4 rid = __ldg(reinterpret_cast<const int4 *>(a.replica_id) + v);
      const uchar4 cls = __ldg(reinterpret_cast<const uchar4 *>(a.class_id) + v), st = __ldg(reinterpret_cast<const uchar4 *>(a.state) + v);
      const int4 pr = __ldg(reinterpret_cast<const int4 *>(a.prompt_len) + v), ge = __ldg(reinterpret_cast<const int4 *>(a.gen) + v);
      const longlong2 ar0 = __ldg(reinterpret_cast<const longlong2 *>(a.arrival) + 2 * v), ar1 = __ldg(reinterpret_cast<const longlong2 *>(a.arrival) + 2 * v + 1);
      int4 we = make_int4(0, 0, 0, 0);
      if (a.weight) we = __ldg(reinterpret_cast<const int4 *>(a.weight) + v);
      id = __ldg(reinterpret_cast<const int4 *>(a.req_id) + v);
      if (!(id.x < id.y && id.y < id.z && id.z < id.w && (4 * v + 4 >= a.n || id.w < __ldg(a.req_id + 4 * v + 4)))) falls = true;
      int64_t sl[4];
      key[0] = do_row(4 * v, rid.x, cls.x, st.x, pr.x, ge.x, we.x, ar0.x, sl[0]);
      key[1] = do_row(4 * v + 1, rid.y, cls.y, st.y, pr.y, ge.y, we.y, ar0.y, sl[1]);
      key[2] = do_row(4 * v + 2, rid.z, cls.z, st.z, pr.z, ge.z, we.z, ar1.x, sl[2]);
      key[3] = do_row(4 * v + 3, rid.w, cls.w, st.w, pr.w, ge.w, we.w, ar1.y, sl[3]);
      longlong2 *slp = reinterpret_cast<longlong2 *>(a.slack) + 2 * v;
      slp[0] = make_longlong2(sl[0], sl[1]); slp[1] = make_longlong2(sl[2], sl[3]);
      reinterpret_cast<int4 *>(a.assign)[v] = make_int4(-1, -1, -1, -1);
      reinterpret_cast<int4 *>(a.queue_order)[v] = make_int4(-1, -1, -1, -1);
    }
    // room for the block's items: my warp's share of it, then its place among all items
    uint32_t m[4], mine = 0, before = 0;
#pragma unroll
    for (int k = 0; k < 4; k++) { m[k] = __ballot_sync(0xffffffffu, key[k] != 0); mine += __popc(m[k]); before += __popc(m[k] & ((1u << lane) - 1u)); }
    uint32_t at = 0;
    if (lane == 0 && mine) at = atomicAdd(&s_count, mine);
    __syncthreads();
    if (tid == 0) { s_base = s_count ? (uint32_t)atomicAdd(&w.ctl[CTL_ITEMS], (unsigned long long)s_count) : 0u; s_count = 0; }
    __syncthreads();
    if (mine) {
      at = s_base + __shfl_sync(0xffffffffu, at, 0) + before;
      if (key[0]) w.item[1][at++] = item_of(key[0], 4 * v, id.x);
      if (key[1]) w.item[1][at++] = item_of(key[1], 4 * v + 1, id.y);
      if (key[2]) w.item[1][at++] = item_of(key[2], 4 * v + 2, id.z);
      if (key[3]) w.item[1][at++] = item_of(key[3], 4 * v + 3, id.w);
    }
  }
  if (blockIdx.x == gridDim.x - 1 && tid < 4) {      // at most three rows are left
    const int64_t i = (n4 << 2) + tid;
    if (i < a.n) {
      int64_t sl;
      const int32_t id = a.req_id[i];
      if (i + 1 < a.n && !(id < a.req_id[i + 1])) falls = true;
      const uint64_t key = do_row(i, a.replica_id[i], a.class_id[i], a.state[i], a.prompt_len[i], a.gen[i], a.weight ? a.weight[i] : 0, a.arrival[i], sl);
      a.slack[i] = sl; a.assign[i] = -1; a.queue_order[i] = -1;
      if (key) w.item[1][atomicAdd(&w.ctl[CTL_ITEMS], 1ull)] = item_of(key, i, id);
    }
  }
  if (bad) atomicOr(a.status, bad);
  qmask = ((uint64_t)__reduce_or_sync(0xffffffffu, (uint32_t)(qmask >> 32)) << 32) | __reduce_or_sync(0xffffffffu, (uint32_t)qmask);
  dmask = ((uint64_t)__reduce_or_sync(0xffffffffu, (uint32_t)(dmask >> 32)) << 32) | __reduce_or_sync(0xffffffffu, (uint32_t)dmask);
  idmax = __reduce_max_sync(0xffffffffu, idmax); idmin_inv = __reduce_max_sync(0xffffffffu, idmin_inv);
  if (lane == 0) {
    if (qmask) atomicOr(&s_qmask, qmask);
    if (dmask) atomicOr(&s_dmask, dmask);
    atomicMax(&s_idmax, idmax); atomicMax(&s_idmin_inv, idmin_inv);
  }
  const int any_falls = __syncthreads_or(falls);
  if (tid == 0) {
    if (s_qmask) atomicOr(&w.ctl[CTL_QMASK], s_qmask);
    if (s_dmask) atomicOr(&w.ctl[CTL_DMASK], s_dmask);
    if (any_falls) w.ctl[CTL_FALLS] = 1;
    atomicMax(&w.ctl[CTL_IDMAX], (unsigned long long)s_idmax); atomicMax(&w.ctl[CTL_IDMIN_INV], (unsigned long long)s_idmin_inv);
  }
  if (tid < 2 * DISP_CLASSES && s_up[tid]) atomicMax(reinterpret_cast<uint32_t *>(w.ctl + CTL_CLASSES) + tid, s_up[tid]);
  if (own)
    for (int r = tid; r < R; r += threads)
      if (s_run[4 * r]) {
        atomicAdd(&w.n_run[r], s_run[4 * r]);
        atomicAdd(&w.sum_kv[r], (unsigned long long)s_run[4 * r + 1] + ((unsigned long long)s_run[4 * r + 2] << 16));
        atomicOr(&w.mask_run[r], s_mask[r]);
      }
}

// ------------------------------------------------------------------------------------------------
// k_disp_sort.  Four phases between grid barriers (the launch is cooperative, so every block is resident; a barrier that
// is not reached in time makes every block return with HFX_ST_TIMEOUT and CTL_ABORT raised; the kernels behind it then hand out
// nothing: the queue, its running totals and the tiles may be unwritten).
//   0  plan of every instance and its place in the maturity order, a warp per instance; the sample in order, a warp
//      per sampled item counting the smaller ones.  Of a queue of up to DISP_SMALL entries all are sampled, and phases 1 and 2 fall away
//      (with bins / so: 300 rows over 2 instances 45.6 / 33.3 us, 2000 over 8 47.6 / 35.3, 8000 over 16, half of them queued, 51.7 / 43.0)
//   1  every item's bin, and its place in it from a global counter.  Every fourth sample of a (stage, priority) starts an
//      interval, an interval is divided evenly into eight bins by slack and tie (so equal slacks spread by tie).  1 M rows over 1024 instances, 60,013
//      and 150,000 rows: every eighth and sixteen 210, 62, 68 us, every fourth and eight 205, 59, 64, every second and eight 221, 63, 68 (each block
//      adds up all bins)
//   2  items to their bins; a fuller bin makes the tiles lower, one of more than DISP_BIN_MAX items (slacks crowded closer than the sample
//      sees) sends the whole queue to a radix sort instead, 22 us a pass at 500 K entries.  (With the line at 1024 items the gaps between the classes of one
//      priority do that: 500,001 rows with weights 324 us, 126 so)
//   3  tiles of whole bins in shared memory: every bin divided further, about one item to a fine bin, an item's place in
//      its fine bin by counting, in a full one by a sorting network; rows out in order, running totals
// An item is moved once (into its bin) where the radix passes moved it eleven times.  A queue of 471 K entries in 148 blocks takes 58 us by the GPU's clock:
// sample and plans 8, splitters 5, bins 14, their starts 3, moving 4, tiles 10.5, running totals 8.5, three barriers of 1.5; one of 42 K 30.
// ------------------------------------------------------------------------------------------------
__device__ __forceinline__ bool grid_barrier(unsigned long long *ctl, uint32_t *status, uint32_t limit, uint32_t &round, uint32_t *s_ok) {
  round++;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) {
    const unsigned long long target = (unsigned long long)round * gridDim.x;
    uint32_t ok = 1;
    if (atomicAdd(&ctl[CTL_BARRIER], 1ull) + 1 < target) {
      uint32_t polls = 0;
      volatile unsigned long long *v = ctl;
      while (v[CTL_BARRIER] < target)
        if (++polls > limit || v[CTL_ABORT]) { ok = 0; break; }
    }
    if (!ok) { ctl[CTL_ABORT] = 1; atomicOr(status, HFX_ST_TIMEOUT); }
    __threadfence();
    *s_ok = ok;
  }
  __syncthreads();
  return *s_ok != 0;
}

// block-wide exclusive prefix of x; *total = the block's sum.  s_part: 33 words, may be reused after the next barrier
template <typename T>
__device__ __forceinline__ T block_prefix(T x, T *s_part, T *total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  T v = x;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) { const T y = __shfl_up_sync(0xffffffffu, v, o); if (lane >= o) v += y; }
  __syncthreads();
  if (lane == 31) s_part[warp] = v;
  __syncthreads();
  if (warp == 0) {
    T s = lane < (int)(blockDim.x >> 5) ? s_part[lane] : T(0);
    const T own = s;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) { const T y = __shfl_up_sync(0xffffffffu, s, o); if (lane >= o) s += y; }
    s_part[lane] = s - own;
    if (lane == 31) s_part[32] = s;
  }
  __syncthreads();
  *total = s_part[32];
  return s_part[warp] + v - x;
}

// two of them behind the same barriers: x and c become the prefixes, all_x and all_c the sums
__device__ __forceinline__ void block_prefix2(int64_t &x, uint32_t &c, int64_t *s_part64, uint32_t *s_part, int64_t *all_x, uint32_t *all_c) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int64_t v = x;
  uint32_t u = c;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int64_t y = __shfl_up_sync(0xffffffffu, v, o);
    const uint32_t z = __shfl_up_sync(0xffffffffu, u, o);
    if (lane >= o) { v += y; u += z; }
  }
  __syncthreads();
  if (lane == 31) { s_part64[warp] = v; s_part[warp] = u; }
  __syncthreads();
  if (warp == 0) {
    const bool in = lane < (int)(blockDim.x >> 5);
    int64_t s = in ? s_part64[lane] : 0;
    uint32_t t = in ? s_part[lane] : 0u;
    const int64_t own = s;
    const uint32_t own_c = t;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int64_t y = __shfl_up_sync(0xffffffffu, s, o);
      const uint32_t z = __shfl_up_sync(0xffffffffu, t, o);
      if (lane >= o) { s += y; t += z; }
    }
    s_part64[lane] = s - own; s_part[lane] = t - own_c;
    if (lane == 31) { s_part64[32] = s; s_part[32] = t; }
  }
  __syncthreads();
  *all_x = s_part64[32]; *all_c = s_part[32];
  x = s_part64[warp] + v - x;
  c = s_part[warp] + u - c;
}

// Puts the items idx[0 .. n) of a tile in order, all threads of the block: a bitonic network with ascending comparators (mirrored first
// sub-stage), so that places behind n need not exist.  What bounds it is the items' scattered places in shared memory: what lies within 32
// places is exchanged in registers, two wider sub-stages at a time by a thread with four places.
struct TileEntry { uint64_t key; uint32_t tie; uint16_t at; };
__device__ __noinline__ void tile_network(uint16_t *idx, int n, const uint4 *s_item, bool by_id) {
  const int lane = threadIdx.x & 31;
  auto load = [&](int i) -> TileEntry {
    TileEntry e = {~0ull, ~0u, 0};
    if (i < n) { e.at = idx[i]; const uint4 x = s_item[e.at]; e.key = item_key(x); e.tie = by_id ? x.z : x.w; }
    return e;
  };
  auto less = [](const TileEntry &x, const TileEntry &y) { return x.key < y.key || (x.key == y.key && x.tie < y.tie); };
  auto exchange = [&](TileEntry &x, TileEntry &y) { if (less(y, x)) { const TileEntry z = x; x = y; y = z; } };
  auto within_warps = [&](bool all) {      // merges of up to 32, or the last five sub-stages of a wider one
    for (int i = threadIdx.x; (i & ~31) < n; i += blockDim.x) {
      TileEntry e = load(i);
      auto exchange_lanes = [&](int mask) {
        TileEntry o;
        o.key = __shfl_xor_sync(0xffffffffu, e.key, mask); o.tie = __shfl_xor_sync(0xffffffffu, e.tie, mask);
        o.at = (uint16_t)__shfl_xor_sync(0xffffffffu, (uint32_t)e.at, mask);
        if (lane < (lane ^ mask) ? less(o, e) : less(e, o)) e = o;
      };
      for (int k = all ? 2 : 32; k <= 32; k <<= 1) {
        if (all) exchange_lanes(k - 1);
        for (int h = all ? k >> 2 : k >> 1; h > 0; h >>= 1) exchange_lanes(h);
      }
      if (i < n) idx[i] = e.at;
    }
    __syncthreads();
  };
  int n_pad = 32;
  while (n_pad < n) n_pad <<= 1;
  within_warps(true);
  for (int k = 64; k <= n_pad; k <<= 1) {
    const int hk = k >> 1;
    for (int t = threadIdx.x; t < n_pad >> 1; t += blockDim.x) {
      const int off = t & (hk - 1), i = 2 * (t - off) + off, j = i + k - 1 - 2 * off;
      if (j < n) {
        const TileEntry x = load(i), y = load(j);
        if (less(y, x)) { idx[i] = y.at; idx[j] = x.at; }
      }
    }
    __syncthreads();
    int h = k >> 2;
    for (; h > 32; h >>= 2) {
      const int q = h >> 1;
      for (int t = threadIdx.x; t < n_pad >> 2; t += blockDim.x) {
        const int off = t & (q - 1), i = 4 * (t - off) + off;
        if (i + q >= n) continue;      // (one place at most)
        TileEntry e0 = load(i), e1 = load(i + q), e2 = load(i + h), e3 = load(i + h + q);
        exchange(e0, e2); exchange(e1, e3); exchange(e0, e1); exchange(e2, e3);
        idx[i] = e0.at; idx[i + q] = e1.at;
        if (i + h < n) idx[i + h] = e2.at;
        if (i + h + q < n) idx[i + h + q] = e3.at;
      }
      __syncthreads();
    }
    if (h == 32) {
      for (int t = threadIdx.x; t < n_pad >> 1; t += blockDim.x) {
        const int i = 2 * t - (t & 31);
        if (i + 32 < n) {
          const TileEntry x = load(i), y = load(i + 32);
          if (less(y, x)) { idx[i] = y.at; idx[i + 32] = x.at; }
        }
      }
      __syncthreads();
    }
    within_warps(false);
  }
}

#define ITEMS_AT_ONCE 4      // items a thread has in flight in the passes over the queue

static_assert(DISP_BINS % SORT_THREADS == 0 && DISP_BINS >= DISP_SPLITS * DISP_SUB && DISP_FINE <= 8192, "bins");
__global__ void __launch_bounds__(SORT_THREADS, 1) k_disp_sort(const HfxParams p, const DispArgs a, const DispWork w) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  uint4 *s_item = reinterpret_cast<uint4 *>(smem_raw);                           // [DISP_TILE_MAX]
  uint32_t *s_row = reinterpret_cast<uint32_t *>(s_item + DISP_TILE_MAX);           // [DISP_TILE_MAX] rows in order
  uint16_t *s_ord = reinterpret_cast<uint16_t *>(s_row + DISP_TILE_MAX);            // [DISP_TILE_MAX] items by fine bin
  uint32_t *s_fine = reinterpret_cast<uint32_t *>(s_ord + DISP_TILE_MAX);           // [DISP_FINE + 4] items per fine bin, then where it starts
  uint32_t *s_start = s_fine + DISP_FINE + 4;                                     // [DISP_BINS + 4] where each bin starts
  uint64_t *s_split = reinterpret_cast<uint64_t *>(s_start + DISP_BINS + 4);        // [DISP_SPLITS] where each interval starts
  uint64_t *s_scale = s_split + DISP_SPLITS;                                      // [DISP_SPLITS] bins per unit<45>, in units of 2^shift, shift<6>
  uint64_t *s_sample = reinterpret_cast<uint64_t *>(smem_raw);                          // [DISP_SMALL] the sample, or the whole of a small queue (before the items are there)
  static_assert(DISP_SMALL >= DISP_SAMPLES && DISP_SMALL <= DISP_TILE && DISP_SMALL * 8 + 4096 * 8 <= SORT_SMEM, "and the instances' maturities behind it");
  int64_t *s_mat = reinterpret_cast<int64_t *>(s_sample + DISP_SMALL);                // [R] maturity of every instance, HFX_INF if it has not come
  uint32_t *s_wc = reinterpret_cast<uint32_t *>(smem_raw);                              // [32][256] (radix passes)
  __shared__ ClassTab s_tab;
  __shared__ uint32_t s_class[DISP_CLASSES], s_r0[DISP_CLASSES + 1];      // first interval | intervals << 16; first sample
  __shared__ uint32_t s_part[33];
  __shared__ int64_t s_part64[33];
  __shared__ unsigned long long s_bmax[2];
  __shared__ uint32_t s_nm[2], s_n1, s_ok, s_digit[256];
  __shared__ uint32_t s_n_full, s_full[DISP_TILE_MAX / DISP_FINE_MAX];      // fine bins beyond DISP_FINE_MAX
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, R = p.n_replicas;
  uint32_t round = 0;
  cudaTriggerProgrammaticLaunchCompletion();

  const uint32_t n_all = (uint32_t)w.ctl[CTL_ITEMS];
  // the sample: every (n_all / n_samples)-th item (they lie in runs of consecutive rows, so the table is sampled evenly)
  const uint32_t n_want = n_all / 64 > 256 ? (n_all / 64 < DISP_SAMPLES ? n_all / 64 : DISP_SAMPLES) : 256;
  const bool small = n_all <= DISP_SMALL;
  const int n_samples = (int)(small ? n_all : n_want);
  const bool by_id = w.ctl[CTL_FALLS] != 0;
  // an item's tie word (request id, or the row where ids rise with the rows), and its 16 leading bits
  const uint32_t id_lo = ~(uint32_t)w.ctl[CTL_IDMIN_INV], tie_span = by_id ? (uint32_t)w.ctl[CTL_IDMAX] - id_lo : (uint32_t)(a.n - 1);
  const int tie_bits = 32 - __clz(tie_span), tie_shift = tie_bits > 16 ? tie_bits - 16 : 0;
  auto tie_of = [&](const uint4 &x) -> uint32_t { return by_id ? x.z : x.w; };
  auto place_of = [&](const uint4 &x) -> uint64_t { return (item_key(x) << 16) | ((by_id ? x.z - id_lo : x.w) >> tie_shift); };

  // ---- 0: instances; the sample in order -------------------------------------------------------------------------
  class_tab_init(p, s_tab, tid);
  for (int r = tid; r < R; r += SORT_THREADS) {
    const int64_t m = a.maturity[r];
    s_mat[r] = m <= a.now ? m : HFX_INF;
  }
  const uint32_t apart = n_all / (uint32_t)(n_samples > 0 ? n_samples : 1), over = n_all - apart * (uint32_t)n_samples;
  for (int k = tid; k < n_samples; k += SORT_THREADS) s_sample[k] = place_of(w.item[1][(uint32_t)k * apart + (uint32_t)k * over / (uint32_t)n_samples]);      // (k n_all / n_samples)
  if (tid < 2) { s_bmax[tid] = 0; s_nm[tid] = 0; }
  if (tid == 0) s_n1 = 0;
  __syncthreads();
  const int gw = warp * gridDim.x + blockIdx.x, n_gw = gridDim.x * (SORT_THREADS / 32);      // the warps of the grid, one of every block after the other
  for (int k = gw; k < n_samples; k += n_gw) {
    const uint64_t x = s_sample[k];
    uint32_t r = 0;
#pragma unroll 4
    for (int i = lane; i < n_samples; i += 32) r += s_sample[i] < x || (s_sample[i] == x && i < k) ? 1u : 0u;
    if (small && tie_shift > 0)      // places equal in the leading bits of the tie
      for (int i = lane; i < n_samples; i += 32)
        if (s_sample[i] == x && i != k) {
          const bool ahead = tie_of(w.item[1][i]) < tie_of(w.item[1][k]);
          if (ahead != (i < k)) r += ahead ? 1u : ~0u;
        }
    r = __reduce_add_sync(0xffffffffu, r);
    if (lane == 0) {
      if (!small) w.sorted[r] = x;
      else { w.rank[r] = w.item[1][k].w; if (x >> 62) atomicAdd(&s_n1, 1u); }      // the row in its place; (bit 46 of the key: the D stage)
    }
  }
  for (int r = n_gw - 1 - gw; r < R; r += n_gw) {
    const hfx_replica_cfg cfg = a.cfg[r];
    const int64_t mat = a.maturity[r];
    const int64_t n_run = (int64_t)w.n_run[r], sum_kv = (int64_t)w.sum_kv[r];
    const uint64_t mask_run = w.mask_run[r];
    const int stage = cfg.mode == HFX_DECODE;
    uint32_t before = 0, first = 0;      // matured instances of my stage in front of me; matured ones of the first stage
    if (mat <= a.now) {
#pragma unroll 4
      for (int r2 = lane; r2 < R; r2 += 32) {
        const int64_t m2 = s_mat[r2];
        const bool ahead = m2 < mat || (m2 == mat && r2 < r);
        if (!a.d_stage) before += ahead ? 1u : 0u;
        else if (m2 != HFX_INF) {
          const int s2 = a.mode[r2] == HFX_DECODE;
          before += s2 == stage && ahead ? 1u : 0u;
          first += s2 ? 0u : 1u;
        }
      }
      before = __reduce_add_sync(0xffffffffu, before); first = __reduce_add_sync(0xffffffffu, first);
    }
    ReplicaPlan pl;
    warp_plan(p, s_tab, cfg, a.now, mat, n_run, sum_kv, mask_run, w.ctl[stage ? CTL_DMASK : CTL_QMASK], pl, lane);
    if (lane == 0) {
      w.plan[r] = pl;
      a.budget[r] = pl.budget; a.e_d[r] = pl.e_d; a.n_run[r] = (int32_t)pl.n_run; a.sum_kv[r] = pl.sum_kv;
      a.adm_cost[r] = 0; a.adm_count[r] = 0; a.maturity_next[r] = mat;
      if (mat <= a.now) {
        const uint32_t k = before + (stage ? first : 0u);      // the D instances are listed behind the first stage's
        int64_t room = INT32_MAX;
        if (pl.batch_cap != 0) { room = (int64_t)pl.batch_cap - pl.n_eff; room = room > 0 ? room : 0; }
        w.ord_id[k] = r;
        w.ord_budget[k] = pl.budget < (INT64_C(1) << 62) ? pl.budget : (INT64_C(1) << 62);      // (a D-stage budget may be unbounded; the totals stay far below)
        w.ord_room[k] = (int32_t)(room < INT32_MAX ? room : INT32_MAX);
        a.inst_order[k] = r;
        atomicAdd(&s_nm[stage], 1u);
        if (pl.budget > 0) atomicMax(&s_bmax[stage], (unsigned long long)pl.budget);
      }
    }
  }
  __syncthreads();
  if (tid < 2) {
    if (s_nm[tid]) atomicAdd(&w.ctl[CTL_NM0 + tid], (unsigned long long)s_nm[tid]);
    if (s_bmax[tid]) atomicMax(&w.ctl[CTL_BMAX0 + tid], s_bmax[tid]);
  }
  if (small && tid == 0 && s_n1) atomicAdd(&w.ctl[CTL_N1], (unsigned long long)s_n1);
  if (!grid_barrier(w.ctl, a.status, w.wait_limit, round, &s_ok)) return;

  // ---- 1: bins -------------------------------------------------------------------------------------------------
  if (blockIdx.x == 0) {
    const int nm0 = (int)__ldcg(w.ctl + CTL_NM0), nm1 = (int)__ldcg(w.ctl + CTL_NM1);
    for (int k = nm0 + nm1 + tid; k < R; k += SORT_THREADS) a.inst_order[k] = -1;
    if (tid == 0) { a.n_mature[0] = nm0; a.n_mature[1] = nm1; }
  }
  if (!small) {
  for (int k = tid; k < n_samples; k += SORT_THREADS) s_sample[k] = __ldcg(w.sorted + k);
  __syncthreads();
  if (tid <= DISP_CLASSES) {      // the first sample of every class
    int b = 0;
#pragma unroll
    for (int h = DISP_SAMPLES; h > 0; h >>= 1) if (b + h <= n_samples && (uint32_t)(s_sample[b + h - 1] >> 56) < (uint32_t)tid) b += h;
    s_r0[tid] = (uint32_t)b;
  }
  __syncthreads();
  if (warp == 0) {      // intervals of every class: one per DISP_STEP samples, one more at either end up to the class's bounds
    uint32_t c[DISP_CLASSES / 32], sum = 0;
#pragma unroll
    for (int e = 0; e < DISP_CLASSES / 32; e++) {
      const int k = lane * (DISP_CLASSES / 32) + e;
      const uint32_t n = s_r0[k + 1] - s_r0[k];
      c[e] = n ? (n + DISP_STEP - 1) / DISP_STEP + 2 : 1u;
      sum += c[e];
    }
    uint32_t run = (uint32_t)warp_incl_scan_i32((int32_t)sum, lane) - sum;
#pragma unroll
    for (int e = 0; e < DISP_CLASSES / 32; e++) {
      const int k = lane * (DISP_CLASSES / 32) + e;
      s_class[k] = run | (c[e] << 16);
      run += c[e];
    }
  }
  __syncthreads();
  }
  auto scale_of = [&](uint64_t span) -> uint64_t {
    const int bits = 64 - __clzll((long long)span), sh = bits > 32 ? bits - 32 : 0;
    return (((uint64_t)DISP_SUB << 32) / ((span >> sh) + 1)) | ((uint64_t)sh << 56);
  };
  const uint32_t *bounds = reinterpret_cast<const uint32_t *>(w.ctl + CTL_CLASSES);
  auto lowest = [&](uint32_t cl) { return (uint64_t)(~bounds[DISP_CLASSES + cl]) << 24; };
  auto highest = [&](uint32_t cl) { return ((uint64_t)bounds[cl] << 24) | 0xffffffull; };
  if (!small) {
  if (tid < DISP_CLASSES && s_r0[tid + 1] == s_r0[tid]) {      // a class the sample missed
    s_split[s_class[tid] & 0xffffu] = lowest(tid); s_scale[s_class[tid] & 0xffffu] = scale_of(highest(tid) > lowest(tid) ? highest(tid) - lowest(tid) : 0);
  }
  for (int k = tid; k < n_samples; k += SORT_THREADS) {
    const uint64_t x = s_sample[k], v = x & ((1ull << 56) - 1);
    const uint32_t cl = (uint32_t)(x >> 56), r0 = s_r0[cl], r1 = s_r0[cl + 1], i = (uint32_t)k - r0, k0 = s_class[cl] & 0xffffu;
    if (i % DISP_STEP == 0) {
      const uint64_t span = s_sample[(uint32_t)k + DISP_STEP < r1 ? (uint32_t)k + DISP_STEP : r1 - 1] - x;
      s_split[k0 + 1 + i / DISP_STEP] = v; s_scale[k0 + 1 + i / DISP_STEP] = scale_of(span);
      if (i == 0) { s_split[k0] = lowest(cl); s_scale[k0] = scale_of(v - lowest(cl)); }
    }
    if ((uint32_t)k == r1 - 1) {
      const uint32_t at = k0 + (s_class[cl] >> 16) - 1;
      s_split[at] = v; s_scale[at] = scale_of(highest(cl) - v);
    }
  }
  __syncthreads();
  }
  // the bin of an item, and how far into it the item lies (in units of 2^-32)
  auto bin_of = [&](const uint4 &x, uint32_t &frac) -> uint32_t {
    const uint64_t pl = place_of(x), v = pl & ((1ull << 56) - 1);
    const uint32_t ci = s_class[(uint32_t)(pl >> 56) & 127u], n = ci >> 16;
    uint32_t k = ci & 0xffffu;
    for (uint32_t len = n; len > 1;) {      // the last interval of the class that starts at or below v
      const uint32_t half = len >> 1;
      if (s_split[k + half] <= v) k += half;
      len -= half;
    }
    const uint64_t lo = s_split[k], sc = s_scale[k], f = sc & ((1ull << 45) - 1);
    const uint64_t d = v > lo ? ((v - lo) >> (sc >> 56)) : 0ull;
    const bool beyond = d >> 32 || __umul64hi(d << 32, f) >= DISP_SUB;      // (only by the rounding of the scale)
    const uint64_t at = d * f;
    frac = beyond ? ~0u : (uint32_t)at;
    return k * DISP_SUB + (beyond ? DISP_SUB - 1 : (uint32_t)(at >> 32));
  };
  const uint32_t per = (n_all + gridDim.x - 1) / gridDim.x;
  const uint32_t lo = blockIdx.x * per < n_all ? blockIdx.x * per : n_all, hi = lo + per < n_all ? lo + per : n_all;      // this block's items
  if (!small) {
    {
    uint32_t n1 = 0;
    for (uint32_t q0 = lo + tid; q0 < hi; q0 += ITEMS_AT_ONCE * SORT_THREADS) {
      uint4 x[ITEMS_AT_ONCE];
      uint32_t rk[ITEMS_AT_ONCE];
#pragma unroll
      for (int e = 0; e < ITEMS_AT_ONCE; e++) { const uint32_t q = q0 + e * SORT_THREADS; if (q < hi) x[e] = w.item[1][q]; }
#pragma unroll
      for (int e = 0; e < ITEMS_AT_ONCE; e++) { const uint32_t q = q0 + e * SORT_THREADS; if (q < hi) { uint32_t fr; const uint32_t bn = bin_of(x[e], fr), k = atomicAdd(&w.bin_cnt[bn], 1u); rk[e] = (bn << 16) | (k < 0xffffu ? k : 0xffffu); n1 += x[e].y >> 14; } }      // (bit 46: the D stage)
#pragma unroll
      for (int e = 0; e < ITEMS_AT_ONCE; e++) { const uint32_t q = q0 + e * SORT_THREADS; if (q < hi) w.rank[q] = rk[e]; }
    }
    n1 = __reduce_add_sync(0xffffffffu, n1);
    if (lane == 0 && n1) atomicAdd(&s_n1, n1);
    }
    __syncthreads();
    if (tid == 0 && s_n1) atomicAdd(&w.ctl[CTL_N1], (unsigned long long)s_n1);
    if (!grid_barrier(w.ctl, a.status, w.wait_limit, round, &s_ok)) return;
  }

  // ---- 2: items to their bins ------------------------------------------------------------------------------------
  const uint32_t n1 = (uint32_t)__ldcg(w.ctl + CTL_N1), n0 = n_all - n1;
  uint32_t fullest = 0;
  if (!small) {
    constexpr int PER = DISP_BINS / SORT_THREADS;
    static_assert(DISP_BINS % SORT_THREADS == 0, "every thread sums the same number of bins");
    uint32_t c[PER], sum = 0, big = 0;
#pragma unroll
    for (int e = 0; e < PER; e++) { c[e] = __ldcg(w.bin_cnt + tid * PER + e); sum += c[e]; big = c[e] > big ? c[e] : big; }
    uint32_t all, run = block_prefix<uint32_t>(sum, s_part, &all);
#pragma unroll
    for (int e = 0; e < PER; e++) { s_start[tid * PER + e] = run; run += c[e]; }
    if (tid == 0) s_start[DISP_BINS] = all;
    big = __reduce_max_sync(0xffffffffu, big);
    if (lane == 0) s_digit[warp] = big;      // (not s_part, which the warp's lanes have just read)
    __syncthreads();
    fullest = __reduce_max_sync(0xffffffffu, s_digit[lane]);
    __syncthreads();
  }
  const bool binned = !small && fullest <= DISP_BIN_MAX;
  if (binned) {
    for (uint32_t q0 = lo + tid; q0 < hi; q0 += ITEMS_AT_ONCE * SORT_THREADS) {
      uint4 x[ITEMS_AT_ONCE];
      uint32_t rk[ITEMS_AT_ONCE];
#pragma unroll
      for (int e = 0; e < ITEMS_AT_ONCE; e++) { const uint32_t q = q0 + e * SORT_THREADS; if (q < hi) { x[e] = w.item[1][q]; rk[e] = w.rank[q]; } }
#pragma unroll
      for (int e = 0; e < ITEMS_AT_ONCE; e++) { const uint32_t q = q0 + e * SORT_THREADS; if (q < hi) { const uint32_t bn = rk[e] >> 16; w.item[0][s_start[bn] + (rk[e] & 0xffffu)] = x[e]; } }
    }
    if (!grid_barrier(w.ctl, a.status, w.wait_limit, round, &s_ok)) return;
  } else if (!small) {
    // radix sort, 8 bits a pass: the tie word, then the key (47 bits).  A block counts the digits of its share, adds up the
    // counts of the blocks before it, and places its items 1024 at a time in order.  Blocks of 2048 items at least, the others only keep step:
    // every block adds up the counts of all (us, all blocks of the grid / so: 40,960 entries 207 / 162, 65,536 218 / 177, 131,072 242 / 211).
    const uint32_t want = (n_all + 2047) / 2048, blocks = want < gridDim.x ? want : gridDim.x, share = (n_all + blocks - 1) / blocks;
    const uint32_t lo = blockIdx.x * share < n_all ? blockIdx.x * share : n_all, hi = lo + share < n_all ? lo + share : n_all;
    for (int pass = 0; pass < 10; pass++) {
      const uint4 *src = w.item[(pass & 1) ^ 1];
      uint4 *dst = w.item[pass & 1];
      auto digit = [&](const uint4 &x) -> uint32_t { return pass < 4 ? (tie_of(x) >> (8 * pass)) & 255u : (uint32_t)(item_key(x) >> (8 * (pass - 4))) & 255u; };
      if (tid < 256) s_digit[tid] = 0;
      __syncthreads();
      for (uint32_t q = lo + tid; q < hi; q += SORT_THREADS) atomicAdd(&s_digit[digit(__ldcg(src + q))], 1u);
      __syncthreads();
      if (tid < 256) w.hist[blockIdx.x * 256 + tid] = s_digit[tid];
      if (!grid_barrier(w.ctl, a.status, w.wait_limit, round, &s_ok)) return;
      {
        uint32_t before = 0, total = 0;
        if (tid < 256)
#pragma unroll 4
          for (int b = 0; b < (int)blocks; b++) { const uint32_t c = __ldcg(w.hist + b * 256 + tid); total += c; if (b < (int)blockIdx.x) before += c; }
        uint32_t all;
        const uint32_t start = block_prefix<uint32_t>(total, s_part, &all);
        if (tid < 256) s_digit[tid] = start + before;
      }
      __syncthreads();
      for (uint32_t q0 = lo; q0 < hi; q0 += SORT_THREADS) {
        for (int i = tid; i < 32 * 256; i += SORT_THREADS) s_wc[i] = 0;
        __syncthreads();
        const uint32_t q = q0 + tid;
        const bool in = q < hi;
        uint4 x = make_uint4(0, 0, 0, 0);
        if (in) x = __ldcg(src + q);
        const uint32_t d = in ? digit(x) : 256u;
        const uint32_t same = __match_any_sync(0xffffffffu, d);
        if (in && lane == __ffs(same) - 1) s_wc[warp * 256 + d] = __popc(same);
        __syncthreads();
        if (tid < 256) {
          uint32_t run = s_digit[tid];
          for (int k = 0; k < 32; k++) { const uint32_t c = s_wc[k * 256 + tid]; s_wc[k * 256 + tid] = run; run += c; }
          s_digit[tid] = run;
        }
        __syncthreads();
        if (in) dst[s_wc[warp * 256 + d] + __popc(same & ((1u << lane) - 1u))] = x;
        __syncthreads();
      }
      if (!grid_barrier(w.ctl, a.status, w.wait_limit, round, &s_ok)) return;
    }
  }

  // ---- 3: rows in order, running totals inside every tile -----------------------------------------------------------
  // tiles: no higher than leaves room for the fullest bin, and the same number of them for every block (819 K entries in 200 tiles of
  // 4096 were two rounds of 148 blocks: 38 us for ordering them, 27 in 296 tiles)
  const uint32_t room = binned && fullest > DISP_TILE_MAX - DISP_TILE ? DISP_TILE_MAX - fullest : DISP_TILE;
  const uint32_t per_block = (per + room - 1) / room, share = (per + per_block - 1) / (per_block ? per_block : 1u);
  const uint32_t tile_rows = share > DISP_TILE_MIN && !small ? share : DISP_TILE_MIN;
  const uint32_t tiles = (n_all + tile_rows - 1) / tile_rows;
  const int64_t bmax0 = (int64_t)__ldcg(w.ctl + CTL_BMAX0), bmax1 = (int64_t)__ldcg(w.ctl + CTL_BMAX1);
  const uint4 *ordered = w.item[binned ? 0 : 1];      // (ten passes end where they began)
  auto bin_edge = [&](uint32_t x) -> uint32_t {      // the first bin that starts at or behind x
    constexpr int K = DISP_BINS / 1024;      // (32 parts of 32 parts of K bins, a look of the warp at each; every warp searches for itself)
    const int full = __popc(__ballot_sync(0xffffffffu, s_start[(lane + 1) * 32 * K - 1] < x));
    if (full == 32) return DISP_BINS;
    int b = full * 32 * K;
    b += __popc(__ballot_sync(0xffffffffu, s_start[b + (lane + 1) * K - 1] < x)) * K;
    return (uint32_t)(b + __popc(__ballot_sync(0xffffffffu, lane < K && s_start[b + (lane < K ? lane : 0)] < x)));
  };
  if (blockIdx.x == 0 && tid == 0) {
    a.n_queue[0] = (int32_t)n0; a.n_queue[1] = (int32_t)n1;
    w.ctl[CTL_N0] = n0; w.ctl[CTL_TILE_ROWS] = tile_rows; w.ctl[CTL_TILES] = tiles;
    w.tile_edge[tiles] = n_all;
  }
  for (uint32_t t = blockIdx.x; t < tiles; t += gridDim.x) {
    const uint32_t x0 = t * tile_rows, x1 = x0 + tile_rows < n_all ? x0 + tile_rows : n_all;
    const uint32_t b0 = binned ? bin_edge(x0) : 0u, b1 = binned ? bin_edge(x1) : 0u;      // whole bins
    const uint32_t e0 = binned ? s_start[b0] : x0, n = (binned ? s_start[b1] : x1) - e0;
    constexpr int IPT = (DISP_TILE_MAX + SORT_THREADS - 1) / SORT_THREADS;
    if (binned) {
      // fine bins: an even share of them for every bin of the tile, in the bin by how far into it an item lies
      // (the last tile ends with the last bin that holds anything: the empty bins behind it, half of them all, would leave its items few fine bins,
      // and the grid waits for its block)
      const uint32_t nb = b1 - b0;
      const int lg = nb <= DISP_FINE ? 31 - __clz(DISP_FINE / (nb > 1 ? nb : 1u)) : 0, down = nb <= DISP_FINE ? 0 : 32 - __clz((nb - 1) / DISP_FINE);      // (a tile of many empty bins: several to a fine one)
      uint32_t fp[IPT];      // fine bin << 16 | place in it (by arrival)
      for (uint32_t i = tid; i < DISP_FINE; i += SORT_THREADS) s_fine[i] = 0;
      if (tid == 0) s_n_full = 0;
      __syncthreads();
#pragma unroll
      for (int e = 0; e < IPT; e++) {
        const uint32_t i = tid + e * SORT_THREADS;
        if (i < n) {
          uint4 x = __ldcg(ordered + e0 + i);
          uint32_t fr;
          const uint32_t fb = (((bin_of(x, fr) - b0) << lg) | (lg ? fr >> (32 - lg) : 0u)) >> down;
          x.y |= fb << 15;      // (the fine bin above the key: the same for all that are compared)
          s_item[i] = x;
          fp[e] = (fb << 16) | atomicAdd(&s_fine[fb], 1u);
        }
      }
      __syncthreads();
      {
        constexpr int FPT = DISP_FINE / SORT_THREADS;
        uint32_t c[FPT], sum = 0, all;
#pragma unroll
        for (int e = 0; e < FPT; e++) { c[e] = s_fine[tid * FPT + e]; sum += c[e]; if (c[e] > DISP_FINE_MAX) s_full[atomicAdd(&s_n_full, 1u)] = tid * FPT + e; }
        uint32_t run = block_prefix<uint32_t>(sum, s_part, &all);
#pragma unroll
        for (int e = 0; e < FPT; e++) { s_fine[tid * FPT + e] = run; run += c[e]; }
        if (tid == 0) s_fine[DISP_FINE] = all;
      }
      __syncthreads();
#pragma unroll
      for (int e = 0; e < IPT; e++) { const uint32_t i = tid + e * SORT_THREADS; if (i < n) s_ord[s_fine[fp[e] >> 16] + (fp[e] & 0xffffu)] = (uint16_t)i; }
      __syncthreads();
#pragma unroll
      for (int e = 0; e < IPT; e++) {
        const uint32_t i = tid + e * SORT_THREADS;
        if (i < n) {
          const uint4 x = s_item[i];
          const uint32_t g0 = s_fine[fp[e] >> 16], g1 = s_fine[(fp[e] >> 16) + 1], tie = tie_of(x);
          const uint64_t key = item_key(x);
          uint32_t place = g0;
          if (g1 > g0 + DISP_FINE_MAX) continue;
          if (g1 > g0 + 1)
            for (uint32_t k = g0; k < g1; k++) {
              const uint4 y = s_item[s_ord[k]];
              const uint64_t ky = item_key(y);
              place += ky < key || (ky == key && tie_of(y) < tie) ? 1u : 0u;
            }
          s_row[place] = x.w;
        }
      }
      for (uint32_t k = 0; k < s_n_full; k++) {
        const uint32_t g0 = s_fine[s_full[k]], g1 = s_fine[s_full[k] + 1];
        tile_network(s_ord + g0, (int)(g1 - g0), s_item, by_id);
        for (uint32_t i = g0 + tid; i < g1; i += SORT_THREADS) s_row[i] = s_item[s_ord[i]].w;
      }
    } else
      for (uint32_t i = tid; i < n; i += SORT_THREADS) s_row[i] = small ? __ldcg(w.rank + e0 + i) : __ldcg(ordered + e0 + i).w;
    __syncthreads();
    // costs of my consecutive places; entries that no instance's budget reaches count nothing
    const uint32_t ipt = (n + SORT_THREADS - 1) / SORT_THREADS, i0 = tid * ipt < n ? tid * ipt : n, mine = i0 + ipt < n ? ipt : n - i0;
    int64_t c[IPT], cost = 0, all_cost;
    uint32_t cnt = 0, all_cnt;
#pragma unroll
    for (int e = 0; e < IPT; e++) { c[e] = -1; if (e < (int)mine) c[e] = disp_cost(p, a, s_row[i0 + e], e0 + i0 + e >= n0); }
#pragma unroll
    for (int e = 0; e < IPT; e++) {
      if (c[e] > (e0 + i0 + e >= n0 ? bmax1 : bmax0)) c[e] = -1;
      if (c[e] >= 0) { cost += c[e]; cnt++; }
    }
    block_prefix2(cost, cnt, s_part64, s_part, &all_cost, &all_cnt);
    int64_t run = cost;
    int32_t run_cnt = (int32_t)cnt;
#pragma unroll
    for (int e = 0; e < IPT; e++)
      if (e < (int)mine) {
        if (c[e] >= 0) { run += c[e]; run_cnt++; s_row[i0 + e] |= VAL_FITS; }
        w.prefix[e0 + i0 + e] = run; w.prefix_cnt[e0 + i0 + e] = run_cnt;
      }
    if (tid == 0) { w.tile_sum[t] = all_cost; w.tile_sum[w.tiles_max + t] = (int64_t)all_cnt; w.tile_edge[t] = e0; }
    __syncthreads();
    for (uint32_t i = tid; i < n; i += SORT_THREADS) { const uint32_t v = s_row[i]; w.val[e0 + i] = v; a.queue_order[e0 + i] = (int32_t)(v & ~VAL_FITS); }
    __syncthreads();
  }
  if (tiles <= DISP_TILES_CHAIN) return;
  // more tiles than the chain adds up by itself: their totals into the running totals
  if (!grid_barrier(w.ctl, a.status, w.wait_limit, round, &s_ok)) return;
  for (uint32_t t = blockIdx.x; t < tiles; t += gridDim.x) {
    const uint32_t e0 = __ldcg(w.tile_edge + t), e1 = __ldcg(w.tile_edge + t + 1);
    int64_t base = 0, base_cnt = 0, all_base, all_base_cnt;
    for (uint32_t t2 = tid; t2 < t; t2 += SORT_THREADS) { base += __ldcg(w.tile_sum + t2); base_cnt += __ldcg(w.tile_sum + w.tiles_max + t2); }
    block_prefix<int64_t>(base, s_part64, &all_base);
    block_prefix<int64_t>(base_cnt, s_part64, &all_base_cnt);
    for (uint32_t q = e0 + tid; q < e1; q += SORT_THREADS) { w.prefix[q] += all_base; w.prefix_cnt[q] += (int32_t)all_base_cnt; }
    __syncthreads();
  }
}

// ------------------------------------------------------------------------------------------------
// k_disp_chain: dispatching step 3, a block per stage.  Every instance starts where the one before it stopped, so the
// walk is one warp's serial recurrence  limit = base + budget -> entries within the limit -> base,  and what counts is its
// latency.  The warp holds the running totals of 256 entries in registers, eight per lane, as 32-bit distances from the
// chunk's start: the new base is the largest total within the limit, one maximum over the lanes (22 cycles), and nothing
// else is on the recurrence.  A batch of instances is done in a loop without a further branch (a short loop: what the single warp
// executes has to come from its first instruction cache, unrolled it took three times as long); then it is looked at whether
// the last of them reached the end of the window: what is in front of the first that did stands, that one is tried again from a fresh
// window or, if it started this one, searched for (32 ways).  A batch is as long as the windows before allowed, or four instances longer: runs
// are of three entries or of a hundred, and a third of the instances takes nothing where one prompt keeps them all waiting (eight instances
// always / sixteen / so, 1 M rows: 700 instances 162 / 162 / 153 us a call, 1024 205 / 240 / 205, 4096 633 / 842 / 620).
// The other warps meanwhile stage the next chunk of totals in shared memory and look up where the runs of the chunk before ended (the entries up to
// a base are those within it).  Then all threads: what every instance took, dispatching step 4 (its new maturity time).  1024 instances, 472 K entries of which
// 22 K are taken: 107 us by the GPU's clock, 98 of them the walk.
// ------------------------------------------------------------------------------------------------
// longest m in [lo, hi] with fits(m), given fits(lo) and fits monotone; whole warp
template <typename F>
__device__ __forceinline__ int64_t warp_longest(int64_t lo, int64_t hi, int lane, F fits) {
  while (lo < hi) {
    const int64_t step = (hi - lo + 31) / 32;
    const int64_t cand = lo + (int64_t)(lane + 1) * step;
    const int f = __popc(__ballot_sync(0xffffffffu, cand <= hi && fits(cand)));      // the lanes that fit are a prefix
    const int64_t nlo = lo + (int64_t)f * step;
    int64_t nhi = lo + (int64_t)(f + 1) * step - 1;
    if (nhi > hi) nhi = hi;
    lo = nlo; hi = nhi;
  }
  return lo;
}

// One batch of the walk.  rel / rc: totals and counts of the window's entries (eight per lane, in order), ~0 where there is
// none; b, c: totals at the cursor, then behind the last instance; lane i gets the totals behind instance i.
template <bool COUNTS>
__device__ __forceinline__ void chain_batch(const uint32_t *rel, const uint32_t *rc, const uint32_t *s_bud, const uint32_t *s_room, uint32_t &b, uint32_t &c, int lane,
                                            int batch, uint32_t &at_b, uint32_t &at_c) {
  uint32_t bud = s_bud[0], room = COUNTS ? s_room[0] : 0u;
#pragma unroll 2
  for (int i = 0; i < batch; i++) {
    const uint32_t lim = b + bud, lc = c + room;
    bud = s_bud[i + 1];                      // (one more than the batch: the arrays are padded)
    if (COUNTS) room = s_room[i + 1];
    uint32_t top[8], topc[8];
#pragma unroll
    for (int j = 0; j < 8; j++) {
      const bool ok = rel[j] <= lim && (!COUNTS || rc[j] <= lc);
      top[j] = ok ? rel[j] : 0u; topc[j] = COUNTS && ok ? rc[j] : 0u;
    }
#pragma unroll
    for (int h = 4; h > 0; h >>= 1)
#pragma unroll
      for (int j = 0; j < h; j++) { top[j] = max(top[j], top[j + h]); topc[j] = max(topc[j], topc[j + h]); }
    b = max(b, __reduce_max_sync(0xffffffffu, top[0]));
    if (COUNTS) c = max(c, __reduce_max_sync(0xffffffffu, topc[0]));
    if (lane == i) { at_b = b; at_c = c; }
  }
}

__global__ void __launch_bounds__(CHAIN_THREADS) k_disp_chain(const HfxParams p, const DispArgs a, const DispWork w) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  constexpr int BUF = CHAIN_CHUNK + CHAIN_WIN + 8;
  uint32_t *s_rel = reinterpret_cast<uint32_t *>(smem_raw);                       // [2][BUF] totals, as distances from the chunk's start
  uint32_t *s_cnt = s_rel + 2 * BUF;                                              // [2][BUF] counts, likewise
  int64_t *s_base = reinterpret_cast<int64_t *>(s_cnt + 2 * BUF);                 // [DISP_TILES_CHAIN] totals in front of each tile
  uint32_t *s_basec = reinterpret_cast<uint32_t *>(s_base + DISP_TILES_CHAIN);    // [DISP_TILES_CHAIN]
  uint32_t *s_edge = s_basec + DISP_TILES_CHAIN;                                  // [DISP_TILES_CHAIN + 1] where each tile starts
  uint32_t *s_bud = s_edge + DISP_TILES_CHAIN + 4;                                // [R + CHAIN_BATCH + 1] budgets, clamped to 2^31 - 1
  uint32_t *s_room = s_bud + p.n_replicas + CHAIN_BATCH + 1;                          // [R + CHAIN_BATCH]
  uint32_t *s_tb = s_room + p.n_replicas + CHAIN_BATCH + 1;                           // [R + CHAIN_BATCH] totals behind an instance's run, from the start of the
  uint32_t *s_tc = s_tb + p.n_replicas + CHAIN_BATCH + 1;                             // [R + CHAIN_BATCH] chunk in which it ended; counts likewise
  __shared__ int s_k, s_capped, s_clamped;      // (any batch cap; any budget of 31 bits or more)
  __shared__ int64_t s_cursor, s_part64[33], s_b0[2], s_c0[2];      // totals at the start of the chunks
  __shared__ uint32_t s_part[33];
  const int tid = threadIdx.x, lane = tid & 31, stage = blockIdx.x;
  if (tid == 0) { s_k = 0; s_cursor = 0; s_capped = 0; s_clamped = 0; }
  cudaTriggerProgrammaticLaunchCompletion();
  cudaGridDependencySynchronize();
  const int nm0 = (int)w.ctl[CTL_NM0], nm = stage ? (int)w.ctl[CTL_NM1] : nm0, koff = stage ? nm0 : 0;
  const int64_t n0 = (int64_t)w.ctl[CTL_N0], qoff = stage ? n0 : 0, nq = stage ? (int64_t)w.ctl[CTL_N1] : n0;
  const uint32_t tiles = (uint32_t)w.ctl[CTL_TILES], tile_rows = (uint32_t)w.ctl[CTL_TILE_ROWS];
  if (w.ctl[CTL_ABORT]) return;                // (TAKEN stays 0)
  const bool by_tile = tiles <= DISP_TILES_CHAIN;      // the running totals start anew in every tile
  if (by_tile) {
    constexpr int PER = DISP_TILES_CHAIN / CHAIN_THREADS;
    int64_t x[PER], sum = 0, all;
    uint32_t y[PER], sumc = 0, allc;
#pragma unroll
    for (int e = 0; e < PER; e++) {
      const uint32_t t = tid * PER + e;
      x[e] = t < tiles ? w.tile_sum[t] : 0; y[e] = t < tiles ? (uint32_t)w.tile_sum[w.tiles_max + t] : 0u;
      sum += x[e]; sumc += y[e];
    }
    for (uint32_t t = tid; t <= tiles; t += CHAIN_THREADS) s_edge[t] = w.tile_edge[t];
    int64_t run = sum;
    uint32_t runc = sumc;
    block_prefix2(run, runc, s_part64, s_part, &all, &allc);
#pragma unroll
    for (int e = 0; e < PER; e++) { s_base[tid * PER + e] = run; s_basec[tid * PER + e] = runc; run += x[e]; runc += y[e]; }
  }
  __syncthreads();
  // the running totals behind q entries of both queues together
  auto total_at = [&](int64_t q, int64_t &cost, int64_t &cnt) {
    cost = 0; cnt = 0;
    if (q <= 0) return;
    cost = w.prefix[q - 1]; cnt = w.prefix_cnt[q - 1];
    if (by_tile) {
      uint32_t t = (uint32_t)(q - 1) / tile_rows;      // (tile t starts at or a little behind t * tile_rows)
      while (s_edge[t] > (uint32_t)(q - 1)) t--;
      cost += s_base[t]; cnt += s_basec[t];
    }
  };
  const int64_t *budgets = w.ord_budget + koff;
  const int32_t *rooms = w.ord_room + koff;
  bool capped = false, wide = false;
  for (int k = tid; k <= nm + CHAIN_BATCH; k += CHAIN_THREADS) {
    const int64_t b = k < nm ? budgets[k] : 0;
    const int32_t r = k < nm ? rooms[k] : 0;
    s_bud[k] = b < 0x7fffffff ? (uint32_t)b : 0x7fffffffu;
    s_room[k] = (uint32_t)r;
    capped = capped || (k < nm && r != INT32_MAX);
    wide = wide || b >= 0x7fffffff;
  }
  if (capped) s_capped = 1;
  if (wide) s_clamped = 1;
  // chunk c and the window behind it, as distances from the totals at the chunk's start
  auto stage_chunk = [&](int64_t c, int first, int step) {
    const int64_t lo = c * CHAIN_CHUNK;
    int64_t b0, c0;
    total_at(qoff + lo, b0, c0);
    uint32_t *rel = s_rel + (c & 1) * BUF, *cnt = s_cnt + (c & 1) * BUF;
    if (first == 0) { s_b0[c & 1] = b0; s_c0[c & 1] = c0; }
#pragma unroll 4
    for (int i = first; i < BUF; i += step) {
      rel[i] = ~0u; cnt[i] = ~0u;
      if (lo + i < nq) {
        int64_t x, y;
        total_at(qoff + lo + i + 1, x, y);
        const uint64_t d = (uint64_t)(x - b0);
        rel[i] = d < 0xffffffffull ? (uint32_t)d : ~0u;
        cnt[i] = (uint32_t)(y - c0);
      }
    }
  };
  stage_chunk(0, tid, CHAIN_THREADS);
  int64_t c = 0, base = 0, base_cnt = 0;      // base: totals at the cursor (the walking warp's)
  if (tid < 32) total_at(qoff, base, base_cnt);
  int k_found = 0;      // instances whose run's end has been looked up
  // the ends of the runs of instances [k0, k1), which lie in chunk cc
  auto look_up = [&](int64_t cc, int k0, int k1, int first, int step) {
    const uint32_t *r = s_rel + (cc & 1) * BUF, *n = s_cnt + (cc & 1) * BUF;
    for (int k = k0 + first; k < k1; k += step) {
      const uint32_t b = s_tb[k], x = s_tc[k];
      if (b == ~0u) continue;      // (noted by the search itself)
      int lo = 0, hi = BUF;
      while (lo < hi) { const int mid = (lo + hi) >> 1; if (r[mid] <= b && n[mid] <= x) lo = mid + 1; else hi = mid; }
      w.run_end[koff + k] = (int32_t)(cc * CHAIN_CHUNK + lo);
    }
  };
  int64_t before = -1;      // the chunk walked before this one, while it is still staged
  for (;;) {
    __syncthreads();
    const int k_now = s_k;
    const int64_t cursor = s_cursor;
    __syncthreads();      // (the walking warp writes the next ones while the others are at work: everyone has read these)
    if (k_now >= nm || cursor >= nq) break;
    if (cursor / CHAIN_CHUNK != c) {      // not the chunk that was staged ahead (a long run)
      if (before >= 0) { look_up(before, k_found, k_now, tid, CHAIN_THREADS); k_found = k_now; before = -1; }
      c = cursor / CHAIN_CHUNK;
      __syncthreads();
      stage_chunk(c, tid, CHAIN_THREADS);
      __syncthreads();
    }
    if (tid >= 32) {
      if (before >= 0) look_up(before, k_found, k_now, tid - 32, CHAIN_THREADS - 32);
      asm volatile("bar.sync 1, %0;" ::"n"(CHAIN_THREADS - 32) : "memory");      // (the chunk ahead goes where the one before lies)
      if ((c + 1) * CHAIN_CHUNK < nq) stage_chunk(c + 1, tid - 32, CHAIN_THREADS - 32);
    } else {
      const int64_t lo = c * CHAIN_CHUNK;
      const int n_here = (int)(nq - lo < CHAIN_CHUNK ? nq - lo : CHAIN_CHUNK);
      const uint32_t *s_r = s_rel + (c & 1) * BUF, *s_c = s_cnt + (c & 1) * BUF;
      const bool counts = s_capped != 0;
      const int64_t b0 = s_b0[c & 1], c0 = s_c0[c & 1];
      const int n_more = (int)(nq - lo < BUF + CHAIN_WIN ? nq - lo : BUF + CHAIN_WIN) - CHAIN_WIN;      // windows that start in front of it are not the last one
      int k = k_now, cur = (int)(cursor - lo);
      int64_t jumped = -1;                   // the cursor behind a run that left the chunk
      const bool clamped = s_clamped != 0;
      int batch = CHAIN_BATCH_MIN + 4;       // as many as the last windows held, or four more
      bool long_runs = false;                // the last run went on behind the window: no use in trying the next one in it
      uint32_t b = base - b0 < 0x7fffffff ? (uint32_t)(base - b0) : 0x7fffffffu, cc = (uint32_t)(base_cnt - c0);      // totals at the cursor, from the chunk's start
      int w0 = cur & ~7;                     // the window's start, at most seven entries in front of the cursor (they are within every limit)
      while (k < nm && w0 < n_here) {
        int good = 0;
        if (!long_runs) {
          uint32_t rel[8], rc[8], tb = 0, tc = 0, nb = b, nc = cc;
          { const uint4 x = reinterpret_cast<const uint4 *>(s_r + w0)[2 * lane], y = reinterpret_cast<const uint4 *>(s_r + w0)[2 * lane + 1];
            rel[0] = x.x; rel[1] = x.y; rel[2] = x.z; rel[3] = x.w; rel[4] = y.x; rel[5] = y.y; rel[6] = y.z; rel[7] = y.w; }
          const uint32_t last = __shfl_sync(0xffffffffu, rel[7], 31);
          if (counts) {
            const uint4 x = reinterpret_cast<const uint4 *>(s_c + w0)[2 * lane], y = reinterpret_cast<const uint4 *>(s_c + w0)[2 * lane + 1];
            rc[0] = x.x; rc[1] = x.y; rc[2] = x.z; rc[3] = x.w; rc[4] = y.x; rc[5] = y.y; rc[6] = y.z; rc[7] = y.w;
            chain_batch<true>(rel, rc, s_bud + k, s_room + k, nb, nc, lane, batch, tb, tc);
          } else chain_batch<false>(rel, rc, s_bud + k, s_room + k, nb, nc, lane, batch, tb, tc);
          // What stands: the answers in front of the first one that reaches the window's last entry (its run may go on behind
          // it), or whose totals or budget do not fit 32 bits.
          const bool more = w0 < n_more;
          good = batch;
          if ((more && nb >= last) || nb >= 0x7fffffffu || k + batch > nm || clamped) {
            const uint32_t my_bud = s_bud[k + (lane < batch ? lane : 0)];
            good = __ffs((int)__ballot_sync(0xffffffffu, lane >= batch || k + lane >= nm || (more && tb >= last) || tb >= 0x7fffffffu || my_bud == 0x7fffffffu)) - 1;
            nb = __shfl_sync(0xffffffffu, tb, good > 0 ? good - 1 : 0);
            nc = __shfl_sync(0xffffffffu, tc, good > 0 ? good - 1 : 0);
          }
          batch = good == batch ? min(batch + 4, CHAIN_BATCH) : max(good, CHAIN_BATCH_MIN);
          if (lane < good) { s_tb[k + lane] = tb; s_tc[k + lane] = counts ? tc : ~0u; }
          if (good) {      // the lanes that hold an entry within the last base: all but the last of them hold nothing else
            b = nb; cc = nc; k += good;
            const int lanes = __popc(__ballot_sync(0xffffffffu, rel[0] <= nb && (!counts || rc[0] <= nc)));
            w0 += lanes > 1 ? 8 * (lanes - 1) : 0;
          }
        }
        if (good == 0) {      // a run longer than the window: searched for among the staged totals, then in memory
          cur = w0;                           // the cursor itself: behind the entries within the base
          { const uint32_t in = __ballot_sync(0xffffffffu, lane < 9 && s_r[w0 + lane] <= b && (!counts || s_c[w0 + lane] <= cc)); cur += __ffs((int)~in) - 1; }
          const int64_t at = lo + cur;
          const int avail = (int)(nq - lo < BUF ? nq - lo : BUF) - cur;
          const uint32_t bud = s_bud[k], lim = b + bud, lc = counts ? cc + s_room[k] : 0xfffffffeu;
          int64_t m = 0;
          const bool narrow = b < 0x7fffffffu && bud < 0x7fffffffu;
          if (narrow) m = warp_longest(0, avail, lane, [&](int64_t x) { return s_r[cur + x - 1] <= lim && s_c[cur + x - 1] <= lc; });
          long_runs = m >= CHAIN_WIN / 2;
          if (!narrow || (m == avail && at + avail < nq)) {
            total_at(qoff + at, base, base_cnt);
            const int64_t limit = base + budgets[k], limit_cnt = base_cnt + rooms[k];
            m = warp_longest(m, nq - at, lane, [&](int64_t x) { int64_t y, z; total_at(qoff + at + x, y, z); return y <= limit && z <= limit_cnt; });
          }
          if (lane == 0) { w.run_end[koff + k] = (int32_t)(at + m); s_tb[k] = ~0u; }
          k++;
          if (cur + m >= n_here) { jumped = at + m; break; }
          cur += (int)m;
          w0 = cur & ~7;
          if (m > 0 && s_r[cur - 1] < 0x7fffffffu) { b = s_r[cur - 1]; cc = s_c[cur - 1]; }
          else if (m > 0) {
            total_at(qoff + lo + cur, base, base_cnt);
            b = base - b0 < 0x7fffffff ? (uint32_t)(base - b0) : 0x7fffffffu; cc = (uint32_t)(base_cnt - c0);
          }
        }
      }
      if (jumped < 0) {                       // the cursor: behind the entries within the base, which end within the next 264
        int hi = w0 + CHAIN_WIN + 8 < BUF ? w0 + CHAIN_WIN + 8 : BUF;
        cur = (int)warp_longest(w0, hi, lane, [&](int64_t x) { return s_r[x - 1] <= b && (!counts || s_c[x - 1] <= cc); });
        jumped = lo + cur;
      }
      total_at(qoff + jumped, base, base_cnt);
      if (lane == 0) { s_k = k; s_cursor = jumped; }
    }
    if (before >= 0) k_found = k_now;
    before = c;
    c++;      // the chunk staged ahead
  }
  const int done = s_k;
  if (before >= 0) look_up(before, k_found, done, tid, CHAIN_THREADS);
  for (int k = done + tid; k < nm; k += CHAIN_THREADS) w.run_end[koff + k] = (int32_t)s_cursor;
  __syncthreads();
  // what every instance took, from the running totals at the ends of its run; its new maturity time
  for (int k = tid; k < nm; k += CHAIN_THREADS) {
    const int r = w.ord_id[koff + k];
    const int64_t st = k > 0 ? w.run_end[koff + k - 1] : 0, en = w.run_end[koff + k];
    int64_t cost = 0, taken = 0;
    if (en > st) {
      int64_t x0, x1, y0, y1;
      total_at(qoff + st, x0, y0); total_at(qoff + en, x1, y1);
      cost = x1 - x0; taken = y1 - y0;
      a.adm_cost[r] = cost;
      a.adm_count[r] = (int32_t)taken;
    }
    if (stage || taken > 0) {
      const ReplicaPlan pl = w.plan[r];
      int64_t lp = 0;
      // (D stage: the enlarged batch's E_d counts d2 per token of context, which is the run's cost less d1 per request)
      if (!stage) a.maturity_next[r] = dev_maturity_next(p, pl, taken, cost, 0, &lp);
      else if (pl.n_run + taken > 0) a.maturity_next[r] = pl.now + p.d0 + p.d1 * pl.n_run + p.d2 * pl.sum_kv + cost;
    }
  }
  if (tid == 0) w.ctl[CTL_TAKEN0 + stage] = (unsigned long long)s_cursor;
}

// ------------------------------------------------------------------------------------------------
// k_disp_assign: the request -> instance binding, a thread per queue place that was handed out (its instance is the first one
// whose run ends behind it; entries that were passed over stay).  The counters that a call adds up into are cleared
// here for the next one (the control words have a copy per parity).
// ------------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(ASSIGN_THREADS) k_disp_assign(const DispArgs a, const DispWork w, unsigned long long *ctl_next) {
  cudaGridDependencySynchronize();
  const int64_t n0 = (int64_t)w.ctl[CTL_N0], t0 = (int64_t)w.ctl[CTL_TAKEN0], t1 = a.d_stage ? (int64_t)w.ctl[CTL_TAKEN1] : 0;
  const int nm0 = (int)w.ctl[CTL_NM0], nm1 = (int)w.ctl[CTL_NM1];
  const int64_t gid = (int64_t)blockIdx.x * ASSIGN_THREADS + threadIdx.x, stride = (int64_t)gridDim.x * ASSIGN_THREADS;
  if (w.ctl[CTL_ABORT]) {      // the order was given up: nothing was handed out (t0 = t1 = 0), and the lists are reported empty
    for (int64_t i = gid; i < a.n; i += stride) a.queue_order[i] = -1;
    for (int64_t r = gid; r < w.R; r += stride) a.inst_order[r] = -1;
    if (gid < 2) { a.n_queue[gid] = 0; a.n_mature[gid] = 0; }
  }
  for (int64_t i = gid; i < t0 + t1; i += stride) {
    const int stage = i >= t0;
    const int64_t q = stage ? n0 + (i - t0) : i;      // place in the numbering of both queues
    const int32_t rel = (int32_t)(stage ? i - t0 : i);
    const int32_t *end = w.run_end + (stage ? nm0 : 0);
    int lo = 0, hi = stage ? nm1 : nm0;               // the first k with end[k] > rel
    while (lo < hi) { const int mid = (lo + hi) >> 1; if (end[mid] <= rel) lo = mid + 1; else hi = mid; }
    const uint32_t v = w.val[q];
    if (v & VAL_FITS) a.assign[v & ~VAL_FITS] = w.ord_id[(stage ? nm0 : 0) + lo];
  }
  for (int64_t r = gid; r < w.R; r += stride) { w.n_run[r] = 0; w.sum_kv[r] = 0; w.mask_run[r] = 0; }
  for (int64_t b = gid; b < DISP_BINS; b += stride) w.bin_cnt[b] = 0;
  for (int64_t k = gid; k < CTL_WORDS; k += stride) ctl_next[k] = 0;
}

// ------------------------------------------------------------------------------------------------
// host side
// ------------------------------------------------------------------------------------------------
// unsettled: a call launched some of its kernels and not the last one, so the counters are not as the next call wants to find them
struct hfx_dispatch_ws { DispWork w; unsigned char *mem; size_t zero; unsigned long long *ctl[2]; uint32_t parity; bool unsettled; };

static size_t chain_smem(int R) { return (size_t)(CHAIN_CHUNK + CHAIN_WIN + 8) * 16 + (size_t)DISP_TILES_CHAIN * 16 + 16 + ((size_t)R + CHAIN_BATCH + 1) * 16; }
static size_t scan_smem(int R) { return R <= SCAN_SMEM_REPLICAS ? (size_t)R * 24 : 0; }
// threads of a block of the scan of n rows, and blocks: small blocks while an SM has one at most (always 1024 threads, whose rows in flight meet in a few
// instances' counters / so: 20,000 rows 53.8 / 51.7 us, 60,013 61.2 / 59.3, 150,000 66.1 / 64.0)
static int scan_threads(const hfx_sched *s, int64_t n) { return n <= (int64_t)s->n_sm * 4 * SCAN_THREADS_FEW ? SCAN_THREADS_FEW : SCAN_THREADS; }
static int scan_blocks(const hfx_sched *s, int64_t n) {
  const int64_t want = (n / 4 + scan_threads(s, n) - 1) / scan_threads(s, n);
  return (int)(want < 1 ? 1 : (want < s->n_sm ? want : s->n_sm));
}
int hfx_dispatch_configure() {
  if (cudaFuncSetAttribute(k_disp_chain, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)chain_smem(4096)) != cudaSuccess ||
      cudaFuncSetAttribute(k_disp_sort, cudaFuncAttributeMaxDynamicSharedMemorySize, SORT_SMEM) != cudaSuccess)
    return HFX_E_CUDA;
  return HFX_OK;
}

void hfx_dispatch_release(hfx_sched *s) {
  if (!s->dispatch_ws) return;
  hfx_dispatch_ws *d = reinterpret_cast<hfx_dispatch_ws *>(s->dispatch_ws);
  cudaFree(d->mem);
  cudaGetLastError();
  delete d;
  s->dispatch_ws = nullptr;
}

static int disp_workspace(hfx_sched *s, hfx_dispatch_ws **out) {
  if (s->dispatch_ws) { *out = reinterpret_cast<hfx_dispatch_ws *>(s->dispatch_ws); return HFX_OK; }
  hfx_dispatch_ws *d = new (std::nothrow) hfx_dispatch_ws();
  if (!d) return HFX_E_NOMEM;
  memset(d, 0, sizeof(*d));
  DispWork &w = d->w;
  const size_t rows = (size_t)s->max_rows, R = (size_t)s->p.n_replicas;
  w.R = s->p.n_replicas;
  w.tiles_max = (int)(rows / DISP_TILE_MIN) + 2;
  size_t used = 0;
  auto part = [&](size_t bytes) { const size_t at = used; used += (bytes + 255) & ~(size_t)255; return at; };
  // what has to be zero between calls, first
  const size_t o_run = part(4 * R), o_kv = part(8 * R), o_mask = part(8 * R), o_ctl = part(8 * CTL_WORDS), o_ctl2 = part(8 * CTL_WORDS), o_bin = part(4 * DISP_BINS);
  const size_t zero = used;
  const size_t o_i0 = part(16 * rows), o_i1 = part(16 * rows), o_sort = part(8 * DISP_SAMPLES), o_rank = part(4 * rows), o_val = part(4 * rows),
               o_pre = part(8 * rows), o_cnt = part(4 * rows), o_ts = part(16 * (size_t)w.tiles_max), o_te = part(4 * ((size_t)w.tiles_max + 1)), o_hist = part(1024 * (size_t)s->n_sm),
               o_plan = part(sizeof(ReplicaPlan) * R), o_ob = part(8 * R), o_or = part(4 * R), o_oi = part(4 * R), o_re = part(4 * R);
  unsigned char *m = nullptr;
  if (cudaMalloc(&m, used) != cudaSuccess) { cudaGetLastError(); delete d; return HFX_E_NOMEM; }
  if (cudaMemsetAsync(m, 0, zero, s->stream) != cudaSuccess) { cudaGetLastError(); cudaFree(m); delete d; return HFX_E_CUDA; }
  d->mem = m; d->zero = zero;
  w.n_run = reinterpret_cast<uint32_t *>(m + o_run); w.sum_kv = reinterpret_cast<unsigned long long *>(m + o_kv); w.mask_run = reinterpret_cast<unsigned long long *>(m + o_mask);
  d->ctl[0] = reinterpret_cast<unsigned long long *>(m + o_ctl); d->ctl[1] = reinterpret_cast<unsigned long long *>(m + o_ctl2);
  w.bin_cnt = reinterpret_cast<uint32_t *>(m + o_bin);
  w.item[0] = reinterpret_cast<uint4 *>(m + o_i0); w.item[1] = reinterpret_cast<uint4 *>(m + o_i1);
  w.sorted = reinterpret_cast<uint64_t *>(m + o_sort); w.tile_edge = reinterpret_cast<uint32_t *>(m + o_te);
  w.rank = reinterpret_cast<uint32_t *>(m + o_rank); w.val = reinterpret_cast<uint32_t *>(m + o_val); w.prefix = reinterpret_cast<int64_t *>(m + o_pre);
  w.prefix_cnt = reinterpret_cast<int32_t *>(m + o_cnt); w.tile_sum = reinterpret_cast<int64_t *>(m + o_ts); w.hist = reinterpret_cast<uint32_t *>(m + o_hist);
  w.plan = reinterpret_cast<ReplicaPlan *>(m + o_plan); w.ord_budget = reinterpret_cast<int64_t *>(m + o_ob);
  w.ord_room = reinterpret_cast<int32_t *>(m + o_or); w.ord_id = reinterpret_cast<int32_t *>(m + o_oi); w.run_end = reinterpret_cast<int32_t *>(m + o_re);
  s->dispatch_ws = d;
  *out = d;
  return HFX_OK;
}

int hfx_launch_dispatch(hfx_sched *s, const hfx_table *t, int64_t now_ns, const int64_t *maturity, const hfx_dispatch_out *o,
                        int32_t cap_max, bool d_stage) {
  hfx_dispatch_ws *d = nullptr;
  int rc = disp_workspace(s, &d);
  if (rc != HFX_OK) return rc;
  DispWork &w = d->w;
  cudaStream_t st = s->stream;
  const int R = s->p.n_replicas;
  const int64_t n = t->n_rows;
  if (d->unsettled && cudaMemsetAsync(d->mem, 0, d->zero, st) != cudaSuccess) { cudaGetLastError(); return HFX_E_CUDA; }
  d->unsettled = true;
  const uint32_t par = d->parity;
  d->parity ^= 1u;
  w.ctl = d->ctl[par];
  w.wait_limit = s->wait_limit;
  DispArgs a;
  a.replica_id = t->replica_id; a.class_id = t->class_id; a.state = t->state; a.prompt_len = t->prompt_len; a.gen = t->gen;
  a.arrival = t->arrival_ns; a.req_id = t->req_id; a.weight = s->p.weight_max > 0 ? t->weight : nullptr;
  a.first_token = t->first_token_ns; a.d_stage = d_stage ? 1 : 0; a.mode = s->d_mode;
  a.n = n; a.now = now_ns; a.cap_max = cap_max; a.maturity = maturity; a.cfg = s->d_cfg;
  a.assign = o->assign; a.queue_order = o->queue_order; a.n_queue = o->n_queue; a.inst_order = o->inst_order;
  a.n_mature = o->n_mature; a.slack = o->slack_ns; a.budget = o->budget; a.e_d = o->e_d_ns; a.n_run = o->n_run;
  a.sum_kv = o->sum_kv; a.adm_cost = o->adm_cost; a.adm_count = o->adm_count; a.maturity_next = o->maturity_next;
  a.status = s->d_status;
  const int blocks = scan_blocks(s, n);
  const int threads = scan_threads(s, n);
  a.rounds = (int32_t)((n / 4 + (int64_t)threads * blocks - 1) / ((int64_t)threads * blocks));
  // blocks of the cooperative kernel: a warp per entry of a small queue, which a larger table may hold too, and tiles of 512 entries (a barrier takes
  // 1.5 us with 30 and with 148 blocks).  4090 entries queued: 8300 rows 17 blocks 83.2 us, 128 42.3, 20,000 rows 40 blocks 54.6, 128 42.4; most of
  // 16,000 rows queued 32 blocks 53.2, 128 53.3, 60,013 118 55.0, 128 55.4
  int64_t want = (n < DISP_SMALL ? n + 31 : DISP_SMALL) / 32, want_r = (R + 31) / 32;
  if (want < (n + 511) / 512) want = (n + 511) / 512;
  if (want < want_r) want = want_r;
  const int grid = (int)(want < 1 ? 1 : (want < s->n_sm ? want : s->n_sm));
  cudaLaunchAttribute attr[1];
  cudaLaunchConfig_t cfg;
  memset(&cfg, 0, sizeof(cfg));
  cfg.stream = st;
  {
    KernelScope ks(s, KSLOT_DISPATCH);
    cfg.gridDim = dim3(blocks); cfg.blockDim = dim3(threads); cfg.dynamicSmemBytes = scan_smem(R);
    const cudaError_t e = threads == SCAN_THREADS ? cudaLaunchKernelEx(&cfg, k_disp_scan<SCAN_THREADS>, s->p, a, w) : cudaLaunchKernelEx(&cfg, k_disp_scan<SCAN_THREADS_FEW>, s->p, a, w);
    if (e != cudaSuccess) { cudaGetLastError(); return HFX_E_CUDA; }
  }
  cfg.attrs = attr; cfg.numAttrs = 1;
  {
    KernelScope ks(s, KSLOT_DISPATCH);
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.gridDim = dim3(grid); cfg.blockDim = dim3(SORT_THREADS); cfg.dynamicSmemBytes = SORT_SMEM;
    if (cudaLaunchKernelEx(&cfg, k_disp_sort, s->p, a, w) != cudaSuccess) { cudaGetLastError(); return HFX_E_CUDA; }
  }
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;      // set up while the kernel before drains
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.numAttrs = s->profiling ? 0 : 1;
  {
    KernelScope ks(s, KSLOT_DISPATCH);
    cfg.gridDim = dim3(d_stage ? 2 : 1); cfg.blockDim = dim3(CHAIN_THREADS); cfg.dynamicSmemBytes = chain_smem(R);
    const cudaError_t e = cudaLaunchKernelEx(&cfg, k_disp_chain, s->p, a, w);
    if (e != cudaSuccess) { cudaGetLastError(); return HFX_E_CUDA; }
  }
  {
    KernelScope ks(s, KSLOT_DISPATCH);
    int64_t want_a = (n + ASSIGN_THREADS * 4 - 1) / (ASSIGN_THREADS * 4);
    want_a = want_a < 8 ? 8 : (want_a < s->n_sm * 2 ? want_a : s->n_sm * 2);
    cfg.gridDim = dim3((unsigned)want_a); cfg.blockDim = dim3(ASSIGN_THREADS); cfg.dynamicSmemBytes = 0;
    if (cudaLaunchKernelEx(&cfg, k_disp_assign, a, w, d->ctl[par ^ 1u]) != cudaSuccess) { cudaGetLastError(); return HFX_E_CUDA; }
  }
  d->unsettled = false;
  return cudaGetLastError() == cudaSuccess ? HFX_OK : HFX_E_CUDA;
}
