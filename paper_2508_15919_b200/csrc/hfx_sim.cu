// hfx_sim_run: batched trace-driven simulation, one warp per trace.
//
// The scheduler iteration (visible set, aggregates of the running batch, E_d, safe budget, most-urgent-first
// admission, maturity, commit, clock advance) is a serial recurrence with little work in it, so what bounds it is
// the latency of one iteration.  A warp holds the whole state of its trace in registers (clock, maturity, list
// lengths, class counts with one class per lane) and never meets a block barrier; what an iteration has to look
// at is bounded by what changed:
//   - a window of 32 rows is held in registers (one row per lane, the window behind it already asked for), so
//     "has anything arrived?" is a comparison with the next arrival time, and a row that has arrived simply
//     waits there (the box); when the window moves on, what is left of it joins a list sorted by (prio, slack base,
//     id), which is the order of the queue at any later time (all slacks fall together);
//   - a running request's finish iteration is fixed at admission; the first 128 of them are in registers, four a lane, what else their
//     end needs in shared memory, and the smallest one is kept, so nobody is looked at in an iteration that finishes nobody
//   - the budget is solved for once a decision (sim_budget), and not at all while nothing of the queue can fit: after a decision that
//     admitted nothing E_d only grows until a request arrives, finishes or is admitted.  Admission takes the most urgent requests from the
//     list's end and the window, whose rows were put in order of urgency when it opened, until one no longer fits;
//   - iterations in which nothing arrives, finishes or is admitted are taken 32 at a time: the clock after j of
//     them is now + j E_d + d2 n_run j (j - 1) / 2 (every request in flight adds one token of context), lane j
//     forms it and a ballot finds the first one that something happens in.  Before maturity the stretch ends at maturity.
// What bounds it is one dependent chain per trace.  B200, one trace of 256 rows, 2000 iterations: 756 us with the running batch in a list in
// memory and comparisons of 128-bit products in place of the budget, 653 so (5.6 cycles to a warp instruction, half of them the latency of the one
// in front); 4096 traces of 2048 rows, 10,000 iterations 21.3 and 15.0 ms (loads waited 2.5 of 9 cycles an instruction there, rows of the queue and the
// batch scattered over sectors of L1 and L2).
// A row takes 19 bytes: 16 side by side, which are one look at it (slack base while queued, admission and finish iteration while running; prompt length
// and priority; output length), a byte (class and state) and one list entry (the queue from the front of the list array, what the
// registers do not hold of the running batch from its back: a row is in one of them at most).
#include "hfx_internal.cuh"

#define SIM_SMEM_ROWS 10240          // longest trace whose rows are kept in shared memory (19 bytes each)
#define SIM_BYTES_PER_ROW 16           // besides the 3 bytes of list, class and state
#define SIM_RUN_REGS 128             // requests in flight whose finish iteration is in a register (four a lane); more of them are in a list
#define SIM_BINS 256                 // bins of the percentile selection (8 bits a pass)
#define SIM_HEAD_BYTES(nc) ((((size_t)(nc) * 40 + 16 + SIM_BINS * 4) + 15) & ~(size_t)15)     // in front of the rows: TTFT and TPOT by class and by rank, the bins, two counters per class
#define SIM_LIST_BYTES(nc, cap) (SIM_HEAD_BYTES(nc) + (size_t)(cap) * 2)      // what is in shared memory wherever the rows are
#define SIM_NOTES_BYTES(cap) (SIM_RUN_REGS * 8 + (size_t)(cap))               // notes of the running batch, classes and states: in shared memory, or behind the rows in scratch
#define SIM_OUTLEN_CAP (1 << 30)   // output lengths are clamped here when the finish iteration is formed
#define SIM_PARKED (SIM_BINS * 2)   // admitted requests of an iteration that are noted in shared memory (over the bins)
// Most traces worked on at once per SM with the rows in scratch: what the registers of a warp (119 a thread, a quarter of the file per
// scheduler) let in.  4096 traces of 2048 rows: 8 a SM 25.7 ms, 12 20.5, 16 15.1.
// (Four classes: up to 3760 rows; of longer traces shared memory holds fewer, or as many as their lists alone let in, see LONG.)
#define SIM_SCRATCH_PER_SM 16

#define SIM_SM_BYTES (227 * 1024)    // shared memory of an SM, of which every block takes 1 KB for itself
#define SIM_BLOCK_BYTES 1024

// the byte of a row: class<6> | state<2>; the word of a row: prompt_len<25> | prio<6>
#define ROW_CLS(x) ((x) & 0x3fu)
#define ROW_STATE(x) ((x) >> 6)
#define ROW_BYTE(cls, st) ((uint8_t)((cls) | ((st) << 6)))
#define ROW_PROMPT(w) ((int32_t)((w) & 0x1ffffffu))
#define ROW_PRIO(w) ((w) >> 25)

struct SimArgs {
  const uint8_t *class_id; const int32_t *prompt_len; const int32_t *output_len; const int64_t *arrival;
  const int32_t *req_id; const int32_t *weight;
  uint8_t *state; int32_t *gen; int64_t *first_token; int64_t *last_token; int64_t *finish;
  const int32_t *trace_off; const hfx_replica_cfg *cfg;
  int32_t n_traces, iters, cap_rows;
  // outputs
  int32_t *iters_executed, *finished, *rejected, *attained;
  int64_t *ttft_p50, *ttft_p99, *tpot_p50, *tpot_p99, *now_out;
};

#define FULL 0xffffffffu

// A field of the rows: of 16-byte rows, of which one sector holds all that an admission asks of a queued row, or a column of its own.
template <typename T, int STRIDE>
struct SimField {
  unsigned char *at;
  __device__ __forceinline__ T &operator[](int i) const { return *reinterpret_cast<T *>(at + STRIDE * (size_t)i); }
};

// The nearest-rank percentile of n non-negative values: 8 bits a pass from the highest byte in use, the warp counting the
// values that share the prefix found so far.  All lanes call; all get the result.
template <typename V>
__device__ int64_t warp_percentile(const V v, int n, int pct, uint32_t *bins, int lane) {
  if (n == 0) return -1;
  int64_t k = ((int64_t)pct * n + 99) / 100;
  if (k < 1) k = 1;
  uint32_t rank = (uint32_t)k;               // 1-based
  uint64_t all = 0;
  for (int i = lane; i < n; i += 32) all |= (uint64_t)v[i];
  all = warp_or_u64(all);
  int shift = all ? ((63 - __clzll((long long)all)) & ~7) : 0;
  uint64_t prefix = 0;                       // the bits above `shift + 8` of the answer
  for (;; shift -= 8) {
    for (int i = lane; i < SIM_BINS; i += 32) bins[i] = 0;
    __syncwarp();
    for (int i = lane; i < n; i += 32) {
      const uint64_t x = (uint64_t)v[i];
      if (shift == 56 || (x >> (shift + 8)) == prefix) atomicAdd(&bins[(uint32_t)(x >> shift) & 255u], 1u);
    }
    __syncwarp();
    uint32_t c[8], sum = 0;                  // lane l holds the bins 8 l .. 8 l + 7
#pragma unroll
    for (int e = 0; e < 8; e++) { c[e] = bins[lane * 8 + e]; sum += c[e]; }
    const uint32_t inc = (uint32_t)warp_incl_scan_i32((int32_t)sum, lane);
    const int l = __ffs(__ballot_sync(FULL, inc >= rank)) - 1;
    uint32_t before = inc - sum, d = 0;
#pragma unroll
    for (int e = 0; e < 8; e++) if (before + c[e] < rank && d == (uint32_t)e) { before += c[e]; d = e + 1; }
    d = __shfl_sync(FULL, d, l); before = __shfl_sync(FULL, before, l);
    rank -= before;
    prefix = (prefix << 8) | (uint64_t)(l * 8 + d);
    __syncwarp();
    if (shift == 0) return (int64_t)prefix;
  }
}

// one row of the arrival window, as a lane holds it
struct SimRow { int64_t arr; int32_t prompt, weight; uint32_t cls, id; int32_t len; };

__device__ __forceinline__ SimRow sim_load_row(const SimArgs &a, int64_t g, bool in) {
  SimRow r;
  r.arr = HFX_INF; r.prompt = -1; r.weight = 0; r.cls = 0; r.id = 0; r.len = 0;
  if (in) {
    r.arr = a.arrival[g]; r.prompt = a.prompt_len[g]; r.cls = a.class_id[g]; r.id = (uint32_t)a.req_id[g] ^ 0x80000000u; r.len = a.output_len[g];
    if (a.weight) r.weight = a.weight[g];
  }
  return r;
}

// Largest n in [0, cap] with E_p(n) den <= ttft y, 0 if there is none (ttft, y, den > 0; the whole warp calls).  The bound is solved for n in
// single precision, and lanes settle the 32 values around the answer exactly; where all of them or none hold it is searched for.
// (Comparisons of 128-bit products only, without the answer, were 50 instructions each, several to an admission.)
__device__ __forceinline__ uint32_t sim_budget(const HfxParams &p, int64_t ttft, int64_t y, int64_t den, uint32_t cap, int lane) {
  const uint64_t nh = __umul64hi((uint64_t)ttft, (uint64_t)y), nl = (uint64_t)ttft * (uint64_t)y;
  const float c1 = (float)p.c1, x = __fdividef((float)ttft * (float)y, (float)den) - (float)p.c0;
  const float est = x > 0.0f ? __fdividef(2.0f * x, c1 + __fsqrt_rn(c1 * c1 + 4.0f * (float)p.c2 * x)) : 0.0f;
  const uint32_t g = est < (float)cap ? (uint32_t)est : cap;
  const uint32_t first = g > 15u ? g - 15u : 0u, n = first + (uint32_t)lane;
  const uint64_t ep = (uint64_t)p.c0 + ((uint64_t)p.c1 + (uint64_t)p.c2 * n) * n;
  const uint64_t h = __umul64hi(ep, (uint64_t)den), l = ep * (uint64_t)den;
  const uint32_t m = __ballot_sync(FULL, n <= cap && (h < nh || (h == nh && l <= nl)));      // (E_p does not fall: the ones that hold are the first)
  if ((m == 0u && first > 0u) || (m == FULL && first + 31u < cap)) return (uint32_t)warp_nsafe(p, nh, nl, (uint64_t)den, (int64_t)cap, lane);
  return m ? first + (uint32_t)__popc(m) - 1u : 0u;
}

// SCRATCH: the 16 bytes of every row live in the block's part of a global scratch buffer, only list, classes, states and notes in
// shared memory.  The live rows then come from L1 most of the time, and more than twice as many traces are resident: what
// a batch of more traces than shared memory holds needs, since a warp by itself issues in one cycle of eight.
// LONG (with SCRATCH): classes, states and notes live there too, shared memory holds the list alone, and more of the traces that are too
// long for SIM_SCRATCH_PER_SM of them are resident.  Long traces have long queues, of which an iteration looks at prompts and priorities along
// the list, so the fields of a row are columns here: entries that are neighbours in the list often share a sector.
// Traces x rows, three iterations a row, ms, lists with classes and notes in shared memory / LONG / LONG with rows of 16 bytes: 2368 x 4096
// 30.8 / 18.7 / 19.3, 3552 x 6144 77.2 / 60.9 / 78.6, 3552 x 8192 124.5 / 90.5 / 127.9, 888 x 16,384 (30,000 iterations) 905 / 649 / 748, 296 x
// 56,000 (20,000) 104.7 / 62.3.
template <bool SCRATCH, bool LONG>
__global__ void __launch_bounds__(32) k_sim(const HfxParams p, const SimArgs a, uint32_t *__restrict__ work_counter,
                                            uint32_t *__restrict__ status, unsigned char *__restrict__ scratch) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int cap = a.cap_rows;
  const int nc = p.n_classes;
  int64_t *c_ttft = reinterpret_cast<int64_t *>(smem_raw), *c_tpot = c_ttft + nc;      // by class
  int64_t *s_ttft = c_tpot + nc, *s_tpot = s_ttft + nc + 1;                           // by rank
  uint32_t *s_bins = reinterpret_cast<uint32_t *>(s_tpot + nc + 1);
  uint16_t *s_park = reinterpret_cast<uint16_t *>(s_bins);      // [SIM_PARKED] the requests admitted in an iteration
  int32_t *s_cq = reinterpret_cast<int32_t *>(s_bins + SIM_BINS), *s_cr = s_cq + nc;      // requests in the queue's list / in flight per class
  uint16_t *s_q = reinterpret_cast<uint16_t *>(smem_raw + SIM_HEAD_BYTES(nc) + (LONG ? 0 : SIM_RUN_REGS * 8));
  unsigned char *rows_mem = SCRATCH ? scratch + (size_t)blockIdx.x * ((size_t)cap * SIM_BYTES_PER_ROW + (LONG ? SIM_NOTES_BYTES(cap) : 0))
                                    : smem_raw + SIM_LIST_BYTES(nc, cap) + SIM_NOTES_BYTES(cap);
  unsigned char *run_mem = LONG ? rows_mem + (size_t)cap * SIM_BYTES_PER_ROW : smem_raw + SIM_HEAD_BYTES(nc);
  uint8_t *s_byte = LONG ? run_mem + SIM_RUN_REGS * 8 : reinterpret_cast<uint8_t *>(s_q + cap);      // class | state << 6
  const SimField<int64_t, LONG ? 8 : 16> s_slot = {rows_mem};             // slack base in the queue; finish iteration | admission iteration << 32 in the batch; later the TTFT, then the TPOT samples
  const SimField<uint32_t, LONG ? 4 : 16> s_word = {rows_mem + (LONG ? 8 * (size_t)cap : 8)};      // prompt_len | prio << 25
  const SimField<int32_t, LONG ? 4 : 16> s_len = {rows_mem + (LONG ? 12 * (size_t)cap : 12)};      // output length
  // One list array for both lists: from the front the queue's list (row indices, the least urgent first), from the back the
  // running batch (RUN(s), unordered)
  uint32_t *s_rinfo = reinterpret_cast<uint32_t *>(run_mem);      // [SIM_RUN_REGS] requests in flight by slot: row | class << 16
  int32_t *s_rctx = reinterpret_cast<int32_t *>(s_rinfo + SIM_RUN_REGS);                // [SIM_RUN_REGS] prompt length less the admission iteration
#define RUN(s) s_q[cap - 1 - (s)]
  const int lane = threadIdx.x;
  const uint32_t lt = (1u << lane) - 1u;
  // Strictest SLO over the classes that have requests: every class has a rank by its bound (nc: none), the bounds are kept
  // by rank, so the strictest one of a set is a minimum over small integers (lane c looks at classes c and c + 32).
  uint32_t rt0 = nc, rt1 = nc, rp0 = nc, rp1 = nc;
#pragma unroll
  for (int h = 0; h < 2; h++) {
    const int c = lane + 32 * h;
    if (c < nc) {
      const int64_t tc = p.ttft[c], pc = p.tpot[c];
      uint32_t rt = 0, rp = 0;
      for (int k = 0; k < nc; k++) {
        const int64_t tk = p.ttft[k], pk = p.tpot[k];
        rt += tk > 0 && (tk < tc || (tk == tc && k < c));
        rp += pk > 0 && (pk < pc || (pk == pc && k < c));
      }
      if (tc > 0) { s_ttft[rt] = tc; if (h == 0) rt0 = rt; else rt1 = rt; }
      if (pc > 0) { s_tpot[rp] = pc; if (h == 0) rp0 = rp; else rp1 = rp; }
      c_ttft[c] = tc; c_tpot[c] = pc;
    }
  }
  if (lane == 0) { s_ttft[nc] = HFX_INF; s_tpot[nc] = HFX_INF; }
  const int64_t d2 = p.d2;

  for (;;) {
    int j = 0;
    if (lane == 0) j = (int)atomicAdd(work_counter, 1u);
    j = __shfl_sync(FULL, j, 0);
    if (j >= a.n_traces) return;
    const int32_t b = a.trace_off[j];
    const int m = a.trace_off[j + 1] - b;
    const hfx_replica_cfg cfg = a.cfg[j];
    for (int i = lane; i < m; i += 32) s_byte[i] = ROW_BYTE(0u, HFX_QUEUED);
    for (int c = lane; c < nc; c += 32) { s_cq[c] = 0; s_cr[c] = 0; }
    __syncwarp();

    int64_t now = 0, mat = 0, sum_kv = 0;
    int nq = 0, nr = 0, it = 0;
    int n_list = 0;                           // requests in flight that are in the list (the others have a slot each)
    int32_t r_fin[SIM_RUN_REGS / 32];         // finish iteration of the request in slot lane + 32 k (INT32_MAX: none)
#pragma unroll
    for (int k = 0; k < SIM_RUN_REGS / 32; k++) r_fin[k] = INT32_MAX;
    int32_t min_prompt = INT32_MAX;           // a lower bound of the shortest prompt in the queue: lowered by every arrival, made exact
                                              // when the whole queue has been looked at (an admission can only raise the true value)
    int32_t next_fin = INT32_MAX;             // the earliest finish iteration in the running batch
    int64_t min_ttft = HFX_INF, min_tpot = HFX_INF;
    int64_t base_lo = HFX_INF, base_hi = INT64_MIN;      // bounds of the finite slack bases in the queue
    // the requests admitted in an iteration: the first ones in shared memory, the rest (tiny prompts) in the trace's gen
    // column, which is written when the trace is over
    auto park = [&](int k, int row) { if (k < SIM_PARKED) s_park[k] = (uint16_t)row; else a.gen[(int64_t)b + k] = row; };
    auto parked = [&](int k) -> int { return k < SIM_PARKED ? (int)s_park[k] : a.gen[(int64_t)b + k]; };
    auto id_of = [&](int row) -> uint32_t { return (uint32_t)__ldg(a.req_id + b + row) ^ 0x80000000u; };

    // The window: rows wb .. wb + 31.  Lane l holds the arrival of row wb + l, and word, class and slack base of the l-th most urgent row of
    // them, row wb + src (an order that no later decision changes, found once when the window opens: the most urgent of a set of lanes is
    // its lowest one).  pend, by arrival: the valid ones that have not arrived; box, by urgency: those that have arrived and wait (the
    // young part of the queue stays here; what is left of it joins the sorted list when the window moves on).
    int wb = 0;
    SimRow w = sim_load_row(a, (int64_t)b + lane, lane < m);
    SimRow wn = sim_load_row(a, (int64_t)b + 32 + lane, 32 + lane < m);
    uint32_t word = 0, pend = 0, box = 0, wrank = 0, wcls = 0;
    int src = 0, wlen = 0;
    int64_t base = BASE_UNBOUNDED;            // slack base, ttft_slo + arrival - E_p(prompt_len): the slack at any later decision is the base minus the earliest start
    auto put_row = [&](int row) {
      if (LONG) { s_slot[row] = base; s_word[row] = word; s_len[row] = wlen; }
      else *reinterpret_cast<uint4 *>(&s_slot[row]) = make_uint4((uint32_t)(uint64_t)base, (uint32_t)((uint64_t)base >> 32), word, (uint32_t)wlen);
    };
    auto open_window = [&]() {
      const bool ok = wb + lane < m && w.cls < (uint32_t)nc && w.prompt >= 0 && w.prompt <= HFX_MAX_TOKENS;
      uint32_t prio = 64u, wd = 0;            // (rows with bad data come last)
      int64_t be = BASE_UNBOUNDED;
      if (ok) {
        if (p.weight_max > 0) {
          const int64_t x = (int64_t)p.weight_max - w.weight;
          prio = (uint32_t)(x < 0 ? 0 : (x > 62 ? 62 : x));
        } else prio = p.prio[w.cls];
        wd = (uint32_t)w.prompt | (prio << 25);
        const int64_t ttft = c_ttft[w.cls];
        if (ttft > 0) be = ttft + w.arr - dev_Ep(p, w.prompt);
      }
      pend = __ballot_sync(FULL, ok);
      const bool bounded = ok && be != BASE_UNBOUNDED;
      const int64_t lo = warp_min_i64(bounded ? be : HFX_INF), hi = ~warp_min_i64(bounded ? ~be : HFX_INF);
      base_lo = lo < base_lo ? lo : base_lo; base_hi = hi > base_hi ? hi : base_hi;
      // Rows of the window that are more urgent than mine, by (prio, base, id).  The bases are taken as 56 bits beside the priority; where one
      // does not fit, or two rows are equal in it, the whole comparison is made.
      const int64_t narrow = be == BASE_UNBOUNDED ? (INT64_C(1) << 56) : be;
      const uint64_t k = ((uint64_t)prio << 57) + (uint64_t)(narrow + (INT64_C(1) << 56));
      bool whole = narrow < -(INT64_C(1) << 56) || (be != BASE_UNBOUNDED && narrow >= (INT64_C(1) << 56));
      int place = 0, same = 0;
#pragma unroll 8
      for (int l = 0; l < 32; l++) {
        const uint64_t x = __shfl_sync(FULL, k, l);
        place += x < k ? 1 : 0; same += x == k ? 1 : 0;
      }
      whole = __any_sync(FULL, whole || same > 1);
      if (whole) {
        place = 0;
        for (int l = 0; l < 32; l++) {
          const uint32_t pr = __shfl_sync(FULL, prio, l), id = __shfl_sync(FULL, w.id, l);
          const int64_t x = __shfl_sync(FULL, be, l);
          const bool first = id < w.id || (id == w.id && l < lane);
          place += pr < prio || (pr == prio && (x < be || (x == be && first))) ? 1 : 0;
        }
      }
      s_park[place] = (uint16_t)lane;         // (no admission is under way)
      __syncwarp();
      src = s_park[lane];
      __syncwarp();
      word = __shfl_sync(FULL, wd, src); base = __shfl_sync(FULL, be, src); wcls = __shfl_sync(FULL, w.cls, src); wlen = __shfl_sync(FULL, w.len, src);
      wrank = __shfl_sync(FULL, rt0, wcls & 31u);
      if (nc > 32) { const uint32_t r1 = __shfl_sync(FULL, rt1, wcls & 31u); if (wcls >= 32u) wrank = r1; }
    };
    // The box joins the list: every waiting row finds its place by a binary search of its own and its rank among the
    // others, then the more urgent entries move up, 32 at a time from the top down.
    auto merge_box = [&]() {
      const bool me = (box >> lane) & 1u;
      const int row = wb + src;
      const uint32_t prio = ROW_PRIO(word);
      if (me) {
        put_row(row); s_byte[row] = ROW_BYTE(wcls, HFX_QUEUED);
        atomicAdd(&s_cq[wcls], 1);
      }
      int pos = 0;                            // entries of the list that are less urgent than mine
      for (int hi = nq; __any_sync(FULL, pos < hi);) {
        if (pos < hi) {
          const int mid = (pos + hi) >> 1, i = s_q[mid];
          const uint32_t pr = ROW_PRIO(s_word[i]);
          const int64_t be = s_slot[i];
          bool less = pr > prio || (pr == prio && be > base);
          if (me && pr == prio && be == base) less = id_of(i) > id_of(row);
          if (less) pos = mid + 1; else hi = mid;
        }
      }
      const int rank = __popc(box & ~((2u << lane) - 1u));      // those of the box that are less urgent
      for (int c0 = (nq - 1) & ~31; nq > 0 && c0 >= 0; c0 -= 32) {
        const int e = c0 + lane;
        const uint32_t below = __ballot_sync(FULL, me && pos <= c0), in = __ballot_sync(FULL, me && pos > c0 && pos <= c0 + 31);
        if ((below | in) == 0) break;         // (the places below are none either)
        const uint16_t v = e < nq ? s_q[e] : (uint16_t)0;
        int up = __popc(below);
        for (uint32_t x = in; x; x &= x - 1) up += __shfl_sync(FULL, pos, __ffs(x) - 1) <= e ? 1 : 0;
        __syncwarp();
        if (e < nq && up) s_q[e + up] = v;
        __syncwarp();
      }
      if (me) s_q[pos + rank] = (uint16_t)row;
      nq += __popc(box);
      box = 0;
      __syncwarp();
    };
    auto advance_window = [&]() {             // to the next window that has a valid row, if there is one
      while (pend == 0 && wb + 32 < m) {
        if (box) merge_box();
        wb += 32;
        w = wn;
        wn = sim_load_row(a, (int64_t)b + wb + 32 + lane, wb + 32 + lane < m);
        open_window();
      }
    };
    auto strictest_q = [&]() -> int64_t {      // TTFT, over the queue
      uint32_t x = ((box >> lane) & 1u) ? wrank : (uint32_t)nc;
      if (lane < nc && s_cq[lane] > 0) x = rt0 < x ? rt0 : x;
      if (lane + 32 < nc && s_cq[lane + 32] > 0) x = rt1 < x ? rt1 : x;
      return s_ttft[__reduce_min_sync(FULL, x)];
    };
    open_window();
    advance_window();
    int64_t next_arr = pend ? __shfl_sync(FULL, w.arr, __ffs(pend) - 1) : HFX_INF;
    bool blocked = false;                     // nothing of the queue fits the budget until a request arrives, finishes or is admitted: E_d only grows

    while (it < a.iters) {
      // ---- 1. arrivals: the rows with arrival <= now join the queue -------------------------------------------
      bool over_any = false;                  // an oversize prompt arrived: its TTFT counts in this iteration only
      int64_t ttft_it = min_ttft;             // the strictest TTFT of this iteration
      if (next_arr <= now) {
        uint32_t over_rank = nc;
        do {
          // (a trace that is not sorted by arrival is a caller error: the rows behind one that has not arrived wait for it)
          const uint32_t late = pend & ~__ballot_sync(FULL, w.arr <= now);
          const uint32_t come = late ? pend & ((1u << (__ffs(late) - 1)) - 1u) : pend;
          const bool me = (come >> src) & 1u, over = me && ROW_PROMPT(word) > cfg.token_cap;
          const uint32_t om = __ballot_sync(FULL, over);
          const int32_t shortest = (int32_t)__reduce_min_sync(FULL, me && !over ? (uint32_t)ROW_PROMPT(word) : 0x7fffffffu);
          min_prompt = shortest < min_prompt ? shortest : min_prompt;
          if (om) {                           // never served: rejected at this iteration's commit
            if (over) s_byte[wb + src] = ROW_BYTE(wcls, HFX_REJECTED);
            const uint32_t r = __reduce_min_sync(FULL, over ? wrank : (uint32_t)nc);
            over_rank = r < over_rank ? r : over_rank;
            over_any = true;
          }
          box |= __ballot_sync(FULL, me && !over);
          pend &= ~come;
          if (pend == 0) advance_window();
          next_arr = pend ? __shfl_sync(FULL, w.arr, __ffs(pend) - 1) : HFX_INF;
        } while (next_arr <= now);
        blocked = false;
        min_ttft = strictest_q();
        ttft_it = min_ttft;
        if (over_any) { const int64_t x = s_ttft[over_rank]; ttft_it = x < ttft_it ? x : ttft_it; }
      }

      // ---- 2. plan: E_d of the running batch, the safe budget (Eq. 3) as a bound on E_p ----------------------
      // The budget is the largest n <= cap_left with E_p(n) den <= num, 0 if there is none (and before maturity: then only a zero-token prompt fits it).
      const int64_t e_d = nr > 0 ? dev_Ed(p, nr, sum_kv) : 0;
      uint32_t budget = 0;
      bool scan = false;
      if (!blocked && (nq > 0 || box)) {
        if (now >= mat) {
          budget = cfg.token_cap - nr > 0 ? (uint32_t)(cfg.token_cap - nr) : 0u;
          if (p.budget_mode != HFX_BUDGET_CAP_ONLY && ttft_it != HFX_INF) {
            const bool decoding = nr > 0 && min_tpot < HFX_INF;      // 2 E_p <= TTFT while nothing decodes
            const int64_t y = decoding ? min_tpot - e_d : 1, den = decoding ? 2 * min_tpot - e_d : 2;
            budget = y > 0 ? sim_budget(p, ttft_it, y, den, budget, lane) : 0u;
          }
        }
        scan = (uint32_t)min_prompt <= budget;            // otherwise the shortest prompt does not fit: nothing is admitted
      }

      // ---- 3. admission: the most urgent requests that fit alone, until one fails ----------------------------
      uint32_t adm_cost = 0;
      int adm_cnt = 0;
      if (scan) {
        const int64_t start = now > mat ? now : mat;
        // The queue's order is (prio, slack base, id), which is the order of the keys as long as no slack is clamped; the
        // bounds of the bases say when one might be.
        auto clamped = [&]() { return base_lo - start < HFX_SLACK_MIN || (base_hi != INT64_MIN && base_hi - start >= HFX_SLACK_MAX); };
        bool by_key = false;
        if (clamped()) {                      // (the bounds may be those of requests that are not in the queue)
          if (box) merge_box();
          int64_t lo = HFX_INF, hi = INT64_MIN;
          for (int s = lane; s < nq; s += 32) {
            const int64_t x = s_slot[s_q[s]];
            if (x != BASE_UNBOUNDED) { lo = x < lo ? x : lo; hi = x > hi ? x : hi; }
          }
          if (((pend >> src) & 1u) && base != BASE_UNBOUNDED) { lo = base < lo ? base : lo; hi = base > hi ? base : hi; }
          base_lo = warp_min_i64(lo); base_hi = ~warp_min_i64(~hi);
          by_key = clamped();
        }
        int low = nq;                         // the lowest place of the list that has been looked at
        bool from_list = false;
        auto room = [&]() { return cfg.batch_cap == 0 || nr + adm_cnt < cfg.batch_cap; };
        if (!by_key) {
          // Two ordered sources: the list from the most urgent entry down, 32 entries at a time, and the box, whose lanes are in
          // order of urgency too.
          const int32_t wp = ROW_PROMPT(word);
          uint32_t bm = box & __ballot_sync(FULL, (uint32_t)wp <= budget), fm = 0;      // rows that fit alone: in the box; in the list's chunk
          int32_t lmin = (box >> lane) & 1u ? wp : INT32_MAX;
          int q = 0, i = 0, left = nq;
          uint32_t wd = 0;
          int64_t list_base = 0;
          bool stop = !room();
          while (!stop) {
            while (fm == 0 && left > 0) {     // the next chunk of the list
              q = left - 1 - lane;
              i = 0; wd = 0;
              if (q >= 0) {
                i = s_q[q];
                if (LONG) wd = s_word[i];
                else {
                  const uint4 x = *reinterpret_cast<const uint4 *>(&s_slot[i]);
                  wd = x.z; list_base = (int64_t)(((uint64_t)x.y << 32) | x.x);
                }
                lmin = ROW_PROMPT(wd) < lmin ? ROW_PROMPT(wd) : lmin;
              }
              fm = __ballot_sync(FULL, q >= 0 && (uint32_t)ROW_PROMPT(wd) <= budget);
              left = left > 32 ? left - 32 : 0;
              low = left;
            }
            if (fm == 0 && bm == 0) break;    // every row that fits has been looked at
            const int fl = __ffs(fm) - 1, bl = __ffs(bm) - 1;
            bool list = bm == 0;
            if (fm && bm) {
              const uint32_t pr = __shfl_sync(FULL, ROW_PRIO(wd), fl), b_prio = __shfl_sync(FULL, ROW_PRIO(word), bl);
              if (pr != b_prio) list = pr < b_prio;
              else {
                const int64_t x = LONG ? s_slot[__shfl_sync(FULL, i, fl)] : __shfl_sync(FULL, list_base, fl), b_base = __shfl_sync(FULL, base, bl);
                list = x < b_base;
                if (x == b_base) list = id_of(__shfl_sync(FULL, i, fl)) < id_of(wb + __shfl_sync(FULL, src, bl));
              }
            }
            const uint32_t c = (uint32_t)ROW_PROMPT(__shfl_sync(FULL, list ? wd : word, list ? fl : bl));
            if (adm_cost + c <= budget) {
              if (list) {
                if (lane == fl) { park(adm_cnt, i); s_q[q] = 0xffffu; atomicSub(&s_cq[ROW_CLS(s_byte[i])], 1); }      // (row numbers stay below 0xffff)
                from_list = true;
              } else {
                if (lane == bl) { park(adm_cnt, wb + src); put_row(wb + src); s_byte[wb + src] = ROW_BYTE(wcls, HFX_QUEUED); }
                box &= ~(1u << bl);
              }
              adm_cost += c; adm_cnt += 1;
              stop = !room();
            } else stop = !p.first_fit || adm_cost + (uint32_t)min_prompt > budget;      // (first fit: can what is left take the shortest prompt?)
            if (list) fm &= fm - 1; else bm &= bm - 1;
          }
          if (left == 0 && !stop) min_prompt = (int32_t)__reduce_min_sync(FULL, (uint32_t)lmin);      // every entry was looked at
        } else {
          // a walk over the list for every extraction, with the clamped keys (the box is empty)
          low = 0; from_list = true;
          // slack of a queued request: ttft_slo - (start - arrival) - E_p(prompt_len) = base - start
          auto key_of = [&](uint32_t wd, int64_t base) -> uint64_t {
            const int64_t sl = base != BASE_UNBOUNDED ? dev_clamp_slack(base - start) : HFX_SLACK_MAX;
            return ((uint64_t)ROW_PRIO(wd) << 40) | (uint64_t)(sl + (INT64_C(1) << 39));
          };
          while (room()) {
            uint64_t bk = ~0ull;
            uint32_t bid = ~0u;
            int bs = -1;
            int32_t lmin = INT32_MAX;
            for (int s = lane; s < nq; s += 32) {
              const uint16_t i = s_q[s];
              if (i == 0xffffu) continue;
              const uint32_t wd = s_word[i];
              lmin = ROW_PROMPT(wd) < lmin ? ROW_PROMPT(wd) : lmin;
              if ((p.first_fit ? adm_cost : 0u) + (uint32_t)ROW_PROMPT(wd) > budget) continue;
              const uint64_t k = key_of(wd, s_slot[i]);
              const uint32_t id = (uint32_t)__ldg(a.req_id + b + i) ^ 0x80000000u;
              if (k < bk || (k == bk && id < bid)) { bk = k; bid = id; bs = s; }
            }
            min_prompt = (int32_t)__reduce_min_sync(FULL, (uint32_t)lmin);
            // the smallest key (46 bits: the upper 32, then the lower 14), then the lowest id
            const uint32_t top = __reduce_min_sync(FULL, bs >= 0 ? (uint32_t)(bk >> 14) : ~0u);
            bool cand = bs >= 0 && (uint32_t)(bk >> 14) == top;
            const uint32_t low14 = __reduce_min_sync(FULL, cand ? (uint32_t)bk & 0x3fffu : ~0u);
            cand = cand && ((uint32_t)bk & 0x3fffu) == low14;
            const uint32_t least = __reduce_min_sync(FULL, cand ? bid : ~0u);
            const uint32_t win = __ballot_sync(FULL, cand && bid == least);
            if (win == 0) break;              // no eligible request left
            const int slot = __shfl_sync(FULL, bs, __ffs(win) - 1);
            const int i = s_q[slot];
            const uint32_t pr = (uint32_t)ROW_PROMPT(s_word[i]);
            if (adm_cost + pr > budget) break;
            __syncwarp();
            if (lane == 0) { s_q[slot] = 0xffffu; park(adm_cnt, i); atomicSub(&s_cq[ROW_CLS(s_byte[i])], 1); }
            __syncwarp();
            adm_cost += pr; adm_cnt += 1;
          }
        }
        // the list closes up over the places of the admitted requests
        if (from_list) {
          __syncwarp();
          int to = low;
          for (int s0 = low; s0 < nq; s0 += 32) {
            const uint16_t v = s0 + lane < nq ? s_q[s0 + lane] : (uint16_t)0xffffu;
            const uint32_t vm = __ballot_sync(FULL, v != 0xffffu);
            __syncwarp();
            if (v != 0xffffu) s_q[to + __popc(vm & lt)] = v;      // (never beyond the places read so far)
            to += __popc(vm);
            __syncwarp();
          }
          nq = to;
        }
        if (nq == 0 && box == 0) min_prompt = INT32_MAX;
        // An admitted request is noted by the lane that holds it, and the commit reads the notes with other lanes (shuffles and
        // ballots between the two do not order memory).
        if (adm_cnt > 0) __syncwarp();
      }
      blocked = adm_cnt == 0 && now >= mat && !over_any;

      // ---- a stretch of iterations in which nothing arrives, finishes or is admitted -------------------------
      if (adm_cnt == 0 && nr > 0 && it < next_fin) {
        const int64_t j1 = lane + 1, grow = d2 * nr;
        const int64_t at = now + j1 * e_d + grow * (j1 * lane / 2);          // the clock after j1 of them
        const int32_t left = (a.iters < next_fin ? a.iters : next_fin) - it; // iterations that may still be plain
        // iteration it + j1 is plain too?  (an oversize arrival tightened this iteration's budget: look again at the next one)
        const bool more = j1 < left && at < next_arr && (now >= mat || at < mat) && !over_any;
        const uint32_t plain = __ballot_sync(FULL, more);
        const int steps = (plain | 0x80000000u) == FULL ? 32 : __ffs((int)~plain);      // this iteration and the run of plain ones behind it
        now = __shfl_sync(FULL, at, steps - 1);
        sum_kv += (int64_t)nr * steps;
        it += steps;
        continue;
      }

      // ---- 4. maturity and the iteration's clock -------------------------------------------------------------
      const int64_t lp = adm_cnt > 0 ? dev_Ep(p, adm_cost) : 0;
      const int64_t t1 = now + lp, t2 = t1 + e_d;
      if (adm_cnt > 0) {
        ReplicaPlan pl;
        pl.now = now; pl.mat = mat; pl.mode = HFX_COLOCATED; pl.n_run = nr; pl.sum_kv = sum_kv; pl.n_eff = nr; pl.tpot_eff = min_tpot; pl.e_d = e_d;
        int64_t lp_ = 0;
        mat = dev_maturity_next(p, pl, adm_cnt, adm_cost, 0, &lp_);
      }
      const bool worked = adm_cnt > 0 || nr > 0;
      bool run_changed = false;

      // ---- 5. commit ---------------------------------------------------------------------------------------------
      // running batch: one more token each; a request finishes when gen + 1 reaches output_len.  Finished ones leave the
      // list, which is closed up in place.
      sum_kv += nr;
      if (it >= next_fin) {
        int32_t nf = INT32_MAX;
#pragma unroll
        for (int k = 0; k < SIM_RUN_REGS / 32; k++) {
          const bool done = it >= r_fin[k];
          const uint32_t dm = __ballot_sync(FULL, done);
          if (dm) {
            uint32_t ctx = 0;
            if (done) {
              const uint32_t info = s_rinfo[32 * k + lane], cls = info >> 16;
              const int i = info & 0xffffu;
              s_byte[i] = ROW_BYTE(cls, HFX_DONE);
              a.finish[(int64_t)b + i] = t2;
              atomicSub(&s_cr[cls], 1);
              ctx = (uint32_t)(s_rctx[32 * k + lane] + it);      // leaves with the context it has after this step
              r_fin[k] = INT32_MAX;
            }
            sum_kv -= (int64_t)__reduce_add_sync(FULL, ctx & 0xffffu) + ((int64_t)__reduce_add_sync(FULL, ctx >> 16) << 16);
            nr -= __popc(dm);
          }
          nf = r_fin[k] < nf ? r_fin[k] : nf;
        }
        __syncwarp();                         // (an admission of this iteration writes the notes of the freed slots, which have just been read, with other lanes)
        int kept = 0;
        for (int s0 = 0; s0 < n_list; s0 += 32) {
          const int s = s0 + lane;
          const bool in = s < n_list;
          const int i = in ? RUN(s) : 0;
          const int64_t slot = in ? s_slot[i] : 0;
          const int32_t fin = (int32_t)(uint32_t)slot;
          const bool done = in && it >= fin;
          uint32_t ctx = 0;
          if (done) {
            const uint32_t cls = ROW_CLS(s_byte[i]);
            s_byte[i] = ROW_BYTE(cls, HFX_DONE);
            a.finish[(int64_t)b + i] = t2;
            atomicSub(&s_cr[cls], 1);
            ctx = (uint32_t)(ROW_PROMPT(s_word[i]) + (it - (int32_t)(slot >> 32)));
          }
          const uint32_t dm = __ballot_sync(FULL, done), km = __ballot_sync(FULL, in && !done);
          __syncwarp();
          if (dm) sum_kv -= (int64_t)__reduce_add_sync(FULL, ctx & 0xffffu) + ((int64_t)__reduce_add_sync(FULL, ctx >> 16) << 16);
          if (in && !done) {
            RUN(kept + __popc(km & lt)) = (uint16_t)i;      // (never beyond the places read so far)
            nf = fin < nf ? fin : nf;
          }
          kept += __popc(km);
          nr -= __popc(dm);
          __syncwarp();
        }
        n_list = kept;
        next_fin = (int32_t)__reduce_min_sync(FULL, (uint32_t)nf);
        run_changed = true;
      }
      // admitted requests: first token at t1; those that go on decoding join the running list
      if (adm_cnt > 0) {
        int32_t nf = INT32_MAX;
        for (int e0 = 0; e0 < adm_cnt; e0 += 32) {
          const bool here = e0 + lane < adm_cnt;
          const int i = here ? parked(e0 + lane) : 0;
          bool goes_on = false;
          uint32_t kv = 0;
          int32_t fin = 0;
          const uint32_t cls = here ? ROW_CLS(s_byte[i]) : 0u;
          if (here) {
            const int32_t ol = s_len[i];
            a.first_token[(int64_t)b + i] = t1;
            if (ol <= 1) { s_byte[i] = ROW_BYTE(cls, HFX_DONE); a.finish[(int64_t)b + i] = t1; }
            else {
              goes_on = true;
              s_byte[i] = ROW_BYTE(cls, HFX_RUNNING);
              atomicAdd(&s_cr[cls], 1);
              fin = it + (ol < SIM_OUTLEN_CAP ? ol : SIM_OUTLEN_CAP) - 1;
              s_slot[i] = (int64_t)(uint32_t)fin | ((int64_t)it << 32);
              nf = fin < nf ? fin : nf;
              kv = (uint32_t)ROW_PROMPT(s_word[i]);
            }
          }
          uint32_t gm = __ballot_sync(FULL, goes_on);
          sum_kv += __reduce_add_sync(FULL, kv);
          nr += __popc(gm);
          // to the free slots, one after the other; the rest to the list
#pragma unroll
          for (int k = 0; k < SIM_RUN_REGS / 32; k++) {
            if (gm == 0) break;
            for (uint32_t fm = __ballot_sync(FULL, r_fin[k] == INT32_MAX); gm && fm; gm &= gm - 1, fm &= fm - 1) {
              const int from = __ffs(gm) - 1, to = __ffs(fm) - 1;
              const int32_t f = __shfl_sync(FULL, fin, from);
              if (lane == to) r_fin[k] = f;
              if (lane == from) { s_rinfo[32 * k + to] = (uint32_t)i | (cls << 16); s_rctx[32 * k + to] = (int32_t)kv - it; }
            }
          }
          if ((gm >> lane) & 1u) RUN(n_list + __popc(gm & lt)) = (uint16_t)i;
          n_list += __popc(gm);
          __syncwarp();
        }
        nf = (int32_t)__reduce_min_sync(FULL, (uint32_t)nf);
        next_fin = nf < next_fin ? nf : next_fin;
        run_changed = true;
        min_ttft = strictest_q();
      }
      if (run_changed) {
        blocked = false;
        __syncwarp();
        uint32_t x = lane < nc && s_cr[lane] > 0 ? rp0 : (uint32_t)nc;
        if (lane + 32 < nc && s_cr[lane + 32] > 0) x = rp1 < x ? rp1 : x;
        min_tpot = s_tpot[__reduce_min_sync(FULL, x)];
      }

      // ---- 6. the clock --------------------------------------------------------------------------------------------
      if (worked) now = t2;
      else {                                  // idle: to the next event; without one the trace is over
        int64_t ev = mat > now ? mat : HFX_INF;
        ev = next_arr < ev ? next_arr : ev;
        if (ev == HFX_INF) break;
        now = ev;
      }
      it++;
    }
    const int executed = it;

    // ---- per-request outputs and per-trace metrics ------------------------------------------
    __syncwarp();
    int fin = 0, rej = 0, att = 0, n_ttft = 0;
    uint32_t bad = 0;
    for (int i0 = 0; i0 < m; i0 += 32) {
      const int i = i0 + lane;
      const int64_t g = (int64_t)b + i;
      int64_t ttft = -1;
      if (i < m) {
        const uint32_t byte = s_byte[i], cls = a.class_id[g];
        const int st = ROW_STATE(byte);
        const int32_t prompt = a.prompt_len[g], outlen = a.output_len[g];
        if (cls >= (uint32_t)nc) bad |= HFX_ST_BAD_CLASS;
        if (prompt < 0 || prompt > HFX_MAX_TOKENS) bad |= HFX_ST_BAD_LEN;
        int32_t gen = 0;
        int64_t first = -1, last = -1;
        if (st == HFX_RUNNING || st == HFX_DONE) {
          first = a.first_token[g];
          ttft = first - a.arrival[g];
          if (st == HFX_DONE) {
            gen = outlen > 1 ? outlen - 1 : 0; last = a.finish[g];
            fin++;
            const int64_t tp = outlen > 1 ? (last - first) / (outlen - 1) : 0;
            const int64_t ttft_slo = c_ttft[cls], tpot_slo = c_tpot[cls];
            if ((ttft_slo <= 0 || ttft <= ttft_slo) && (tpot_slo <= 0 || tp <= tpot_slo)) att++;
          } else {
            gen = executed - 1 - (int32_t)(s_slot[i] >> 32);
            last = gen > 0 ? now : first;
          }
        } else {
          a.first_token[g] = -1;
          if (st == HFX_REJECTED) rej++;
        }
        a.last_token[g] = last;
        if (st != HFX_DONE) a.finish[g] = -1;
        a.state[g] = (uint8_t)st;
        a.gen[g] = gen;
      }
      // the TTFT samples, closed up over the slots of rows already looked at (their order does not matter)
      const uint32_t sm = __ballot_sync(FULL, ttft >= 0);
      __syncwarp();                           // (a request still in flight has had its admission iteration read from a slot that is written now)
      if (ttft >= 0) s_slot[n_ttft + __popc(sm & lt)] = ttft;
      n_ttft += __popc(sm);
      __syncwarp();
    }
    if (bad) atomicOr(status, bad);
    fin = (int)__reduce_add_sync(FULL, (uint32_t)fin); rej = (int)__reduce_add_sync(FULL, (uint32_t)rej); att = (int)__reduce_add_sync(FULL, (uint32_t)att);
    const int64_t ttft50 = warp_percentile(s_slot, n_ttft, 50, s_bins, lane), ttft99 = warp_percentile(s_slot, n_ttft, 99, s_bins, lane);
    __syncwarp();
    int n_tpot = 0;
    for (int i0 = 0; i0 < m; i0 += 32) {
      const int i = i0 + lane;
      const int64_t g = (int64_t)b + i;
      int64_t tpot = -1;
      if (i < m && ROW_STATE(s_byte[i]) == HFX_DONE) {
        const int32_t outlen = a.output_len[g];
        if (outlen > 1) tpot = (a.finish[g] - a.first_token[g]) / (outlen - 1);
      }
      const uint32_t sm = __ballot_sync(FULL, tpot >= 0);
      if (tpot >= 0) s_slot[n_tpot + __popc(sm & lt)] = tpot;
      n_tpot += __popc(sm);
    }
    __syncwarp();
    const int64_t tpot50 = warp_percentile(s_slot, n_tpot, 50, s_bins, lane), tpot99 = warp_percentile(s_slot, n_tpot, 99, s_bins, lane);
    if (lane == 0) {
      a.iters_executed[j] = executed;
      a.finished[j] = fin; a.rejected[j] = rej; a.attained[j] = att;
      a.ttft_p50[j] = ttft50; a.ttft_p99[j] = ttft99; a.tpot_p50[j] = tpot50; a.tpot_p99[j] = tpot99;
      if (a.now_out) a.now_out[j] = now;
    }
    __syncwarp();
  }
}

int hfx_sim_configure() {
  if (cudaFuncSetAttribute(k_sim<false, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, SIM_SMEM_ROWS * SIM_BYTES_PER_ROW + (int)(SIM_LIST_BYTES(HFX_MAX_CLASSES, SIM_SMEM_ROWS) + SIM_NOTES_BYTES(SIM_SMEM_ROWS))) != cudaSuccess ||
      cudaFuncSetAttribute(k_sim<true, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, SIM_SM_BYTES - SIM_BLOCK_BYTES) != cudaSuccess ||
      cudaFuncSetAttribute(k_sim<true, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, SIM_SM_BYTES - SIM_BLOCK_BYTES) != cudaSuccess)
    return HFX_E_CUDA;
  return HFX_OK;
}

void hfx_sim_release(hfx_sched *s) {
  cudaFree(s->d_sim_scratch);
  s->d_sim_scratch = nullptr; s->sim_scratch_bytes = 0;
}

// `trace_off` is already on the device (copied by the caller of this launcher); max_rows is the
// longest trace, known on the host.
int hfx_launch_sim_kernel(hfx_sched *s, const hfx_table *t, const int32_t *d_trace_off, int32_t n_traces,
                          int32_t max_trace_rows, int32_t iters, const hfx_sim_out *o, uint32_t *d_work_counter) {
  SimArgs a;
  a.class_id = t->class_id; a.prompt_len = t->prompt_len; a.output_len = t->output_len; a.arrival = t->arrival_ns;
  a.req_id = t->req_id; a.weight = s->p.weight_max > 0 ? t->weight : nullptr;
  a.state = t->state; a.gen = t->gen; a.first_token = t->first_token_ns; a.last_token = t->last_token_ns;
  a.finish = t->finish_ns; a.trace_off = d_trace_off; a.cfg = s->d_cfg;
  a.n_traces = n_traces; a.iters = iters;
  int cap = (max_trace_rows + 15) & ~15;
  if (cap < 16) cap = 16;
  a.cap_rows = cap;
  a.iters_executed = o->iters_executed; a.finished = o->finished; a.rejected = o->rejected; a.attained = o->attained;
  a.ttft_p50 = o->ttft_p50_ns; a.ttft_p99 = o->ttft_p99_ns; a.tpot_p50 = o->tpot_p50_ns; a.tpot_p99 = o->tpot_p99_ns;
  a.now_out = o->now_ns;
  const size_t rows_bytes = (size_t)cap * SIM_BYTES_PER_ROW, list_bytes = SIM_LIST_BYTES(s->p.n_classes, cap), notes_bytes = SIM_NOTES_BYTES(cap);
  const size_t sm_bytes = SIM_SM_BYTES, block_bytes = SIM_BLOCK_BYTES;
  int rc = cuda_rc(cudaMemsetAsync(d_work_counter, 0, sizeof(uint32_t), s->stream));
  if (rc != HFX_OK) return rc;
  int per_sm = cap <= SIM_SMEM_ROWS ? (int)(sm_bytes / (rows_bytes + list_bytes + notes_bytes + block_bytes)) : 0;
  if (per_sm > 32) per_sm = 32;
  auto in_scratch = [&](size_t smem) { const int x = (int)(sm_bytes / (smem + block_bytes)); return x < SIM_SCRATCH_PER_SM ? x : SIM_SCRATCH_PER_SM; };
  int per_sm_scratch = in_scratch(list_bytes + notes_bytes);
  // LONG where it saves a round of traces: in the same number of rounds fewer at a time are the quicker ones (3000 traces of 5120 rows, two
  // rounds of 12 or 16 an SM: 42.2 ms with classes and notes in shared memory, 45.7 without)
  auto rounds = [&](int each) { return (n_traces + s->n_sm * each - 1) / (s->n_sm * each); };
  const bool long_rows = rounds(in_scratch(list_bytes)) < rounds(per_sm_scratch);
  if (long_rows) per_sm_scratch = in_scratch(list_bytes);
  // Rows in shared memory (the shorter latency) while that keeps every trace resident, or as many as scratch would.  Traces of 2048 rows,
  // shared memory / scratch: 444 5.64 / 5.89 ms, 740 (five a SM) 5.90 / 6.45, 1036 (scratch) 6.7; 4096 of 512 rows 3.89 / 4.07, of 256 1.89 / 2.00.
  bool in_smem = per_sm > 0 && (n_traces <= s->n_sm * per_sm || per_sm >= per_sm_scratch);
  // otherwise the rows of every resident block in a scratch buffer, allocated when first needed
  int grid = s->n_sm * per_sm_scratch;
  if (grid > n_traces) grid = n_traces;
  const size_t need = (rows_bytes + (long_rows ? notes_bytes : 0)) * (size_t)grid;
  if (!in_smem && s->sim_scratch_bytes < need) {
    // Inside a stream capture the stream cannot be waited for: traces that shared memory can hold stay there, fewer at a time.
    cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
    rc = cuda_rc(cudaStreamIsCapturing(s->stream, &capture));
    if (rc != HFX_OK) return rc;
    in_smem = capture != cudaStreamCaptureStatusNone && per_sm > 0;
    if (!in_smem) {
      rc = cuda_rc(cudaStreamSynchronize(s->stream));
      if (rc != HFX_OK) return rc;
      cudaFree(s->d_sim_scratch);
      s->d_sim_scratch = nullptr; s->sim_scratch_bytes = 0;
      if (cudaMalloc(&s->d_sim_scratch, need) != cudaSuccess) { cudaGetLastError(); return HFX_E_NOMEM; }
      s->sim_scratch_bytes = need;
    }
  }
  if (in_smem) {
    grid = s->n_sm * per_sm;
    if (grid > n_traces) grid = n_traces;
  }
  {
    KernelScope ks(s, KSLOT_SIM);
    if (in_smem) k_sim<false, false><<<grid, 32, rows_bytes + list_bytes + notes_bytes, s->stream>>>(s->p, a, d_work_counter, s->d_status, nullptr);
    else if (long_rows) k_sim<true, true><<<grid, 32, list_bytes, s->stream>>>(s->p, a, d_work_counter, s->d_status, s->d_sim_scratch);
    else k_sim<true, false><<<grid, 32, list_bytes + notes_bytes, s->stream>>>(s->p, a, d_work_counter, s->d_status, s->d_sim_scratch);
  }
  return cudaGetLastError() == cudaSuccess ? HFX_OK : HFX_E_CUDA;
}
