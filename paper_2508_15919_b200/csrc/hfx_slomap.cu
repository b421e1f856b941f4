// hfx_slo_map: priority-based SLO mapping (Sec. 3.3.2).  Requests that carry only a priority get
// their TTFT / TPOT targets from a sliding window of completed requests.
//
//   k_slo_window   Every priority p asks for one record of the window ordered by TTFT and one of it ordered by TPOT, at index
//                  base + offset, base = C_0 + ... + C_{p-1}, offset = floor((p + 1) C_p / (N + 1)).  So the window is not
//                  sorted: for every record the smaller ones are counted (4096 x 4096 comparisons over the whole GPU are short;
//                  ordering the window twice by one block was 114 us, the whole call takes 17.1 us now, 9.7 with a window of
//                  64: its two launches), and a record whose rank somebody asked for is
//                  noted.  Other blocks of the same launch find the first request (lowest row) of every priority: only
//                  it sees the queueing-delay correction, the later ones find the delay it left behind
//   k_slo_assign   per request: correction, contention-aware clamp, the two targets
#include <string.h>

#include "hfx_internal.cuh"

#define SLO_WINDOW_MAX 4096
#define SLO_THREADS 256
#define SLO_WIN_THREADS 1024
#define SLO_WIN_RECORDS 32      // records a block ranks
#define SLO_WARP_RECORDS 4      // of them at a time in a warp

struct SloTable {          // per priority, HFX_MAX_CLASSES entries each
  unsigned long long first_row[2][HFX_MAX_CLASSES];      // two copies used in turn: a call clears the next one's (~0: none)
  int64_t ref_ttft[HFX_MAX_CLASSES], ref_tpot[HFX_MAX_CLASSES], ref_queue[HFX_MAX_CLASSES], delta[HFX_MAX_CLASSES];
  int32_t higher_pending[HFX_MAX_CLASSES];
  int32_t w_valid;
};

struct SloArgs {
  const int32_t *win_prio; const int64_t *win_ttft; const int64_t *win_tpot; const int64_t *win_queue; int32_t w;
  const int64_t *ttft_min, *ttft_max, *ttft_min_relaxed, *tpot_min, *tpot_max, *tpot_min_relaxed;
  int64_t *last_queue; const int32_t *pending; const int32_t *new_prio; int64_t n_new;
  int64_t *ttft_out, *tpot_out;
  int32_t n_prio, win_blocks, par; SloTable *tab; uint32_t *status;
};

__global__ void __launch_bounds__(SLO_WIN_THREADS) k_slo_window(const SloArgs a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  uint64_t *s_ttft = reinterpret_cast<uint64_t *>(smem_raw), *s_tpot = s_ttft + a.w;      // [w] values, biased to unsigned order; ~0 on a bad record
  __shared__ uint32_t s_C[HFX_MAX_CLASSES];
  __shared__ uint32_t s_idx[HFX_MAX_CLASSES];
  __shared__ uint32_t s_first[HFX_MAX_CLASSES];
  __shared__ uint32_t s_rank[2 * SLO_WIN_RECORDS];
  const int N = a.n_prio, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  cudaTriggerProgrammaticLaunchCompletion();
  if ((int)blockIdx.x >= a.win_blocks) {      // the first request of every priority: row numbers relative to the block's first row
    const int64_t lo = (int64_t)(blockIdx.x - a.win_blocks) * SLO_WIN_THREADS;
    if (tid < N) s_first[tid] = ~0u;
    __syncthreads();
    const int32_t pr = lo + tid < a.n_new ? a.new_prio[lo + tid] : -1;
    const bool ok = pr >= 0 && pr < N;
    const uint32_t same = __match_any_sync(0xffffffffu, ok ? pr : -1);
    if (ok && lane == __ffs(same) - 1) atomicMin(&s_first[pr], (uint32_t)tid);
    __syncthreads();
    if (tid < N && s_first[tid] != ~0u) atomicMin(&a.tab->first_row[a.par][tid], (unsigned long long)(lo + s_first[tid]));
    return;
  }
  if (tid < HFX_MAX_CLASSES) s_C[tid] = 0;
  if (tid < 2 * SLO_WIN_RECORDS) s_rank[tid] = 0;
  __syncthreads();
  // the whole window into shared memory; valid records per priority
  uint32_t bad = 0;
#pragma unroll
  for (int r = 0; r < SLO_WINDOW_MAX / SLO_WIN_THREADS; r++) {
    const int j = r * SLO_WIN_THREADS + tid;
    if (j - lane >= a.w) break;               // (whole warps)
    const bool in = j < a.w;
    const int32_t pr = in ? a.win_prio[j] : -1;
    const int64_t t = in ? a.win_ttft[j] : 0, q = in ? a.win_tpot[j] : 0;
    const bool ok = pr >= 0 && pr < N;
    const uint32_t same = __match_any_sync(0xffffffffu, ok ? pr : -1);      // (priorities are few: a warp's are counted together)
    if (ok && lane == __ffs(same) - 1) atomicAdd(&s_C[pr], (uint32_t)__popc(same));
    if (!in) break;
    if (!ok) bad |= HFX_ST_BAD_CLASS;
    s_ttft[j] = ok ? (uint64_t)t ^ (1ull << 63) : ~0ull;
    s_tpot[j] = ok ? (uint64_t)q ^ (1ull << 63) : ~0ull;
  }
  __syncthreads();
  if (tid < N) {      // the index that priority tid asks for
    uint32_t base = 0, all = 0;
    for (int i = 0; i < N; i++) { if (i < tid) base += s_C[i]; all += s_C[i]; }
    const uint32_t offset = (uint32_t)(((uint64_t)(tid + 1) * s_C[tid]) / (uint64_t)(N + 1));
    uint32_t idx = base + offset;
    if (all > 0 && idx > all - 1) idx = all - 1;
    s_idx[tid] = idx;
    if (blockIdx.x == 0) {
      int hp = 0;      // a higher priority pending?
      for (int i = 0; i < tid; i++) hp |= a.pending[i] > 0;
      a.tab->higher_pending[tid] = hp;
      if (tid == 0) a.tab->w_valid = (int32_t)all;
    }
  }
  // (all entries: the call that used the other copy, or the one that will, may have more priorities than this one)
  if (blockIdx.x == 0 && tid < HFX_MAX_CLASSES) a.tab->first_row[a.par ^ 1][tid] = ~0ull;
  if (bad && blockIdx.x == 0) atomicOr(a.status, bad);
  __syncthreads();
  // Ranks among the valid records, ties by position.  A warp counts for four neighbouring records, so a value read from
  // shared memory serves four comparisons (one record per warp is bound by those reads); four warps share a group of
  // records, a quarter of the window each.
  const int j0 = (int)blockIdx.x * SLO_WIN_RECORDS + (warp & 7) * SLO_WARP_RECORDS;
  auto valid = [&](int k) { return a.win_prio[k] >= 0 && a.win_prio[k] < N; };
  if (j0 < a.w) {
    const int chunks = (a.w + 31) >> 5, per = (chunks + 3) >> 2, c0 = (warp >> 3) * per, c1 = c0 + per < chunks ? c0 + per : chunks, cj = j0 >> 5;
    auto count = [&](const uint64_t *v, uint32_t *rank) {
      uint64_t x[SLO_WARP_RECORDS];
      uint32_t r[SLO_WARP_RECORDS];
#pragma unroll
      for (int e = 0; e < SLO_WARP_RECORDS; e++) { x[e] = j0 + e < a.w ? v[j0 + e] : 0; r[e] = 0; }
      const int front = cj < c1 ? (cj > c0 ? cj : c0) : c1;      // chunks in front of the records' own: there an equal value counts
#pragma unroll 4
      for (int c = c0; c < front; c++) {
        const uint64_t y = v[c * 32 + lane];
#pragma unroll
        for (int e = 0; e < SLO_WARP_RECORDS; e++) if (y <= x[e]) r[e]++;
      }
      if (cj >= c0 && cj < c1) {
        const int k = cj * 32 + lane;
        const uint64_t y = k < a.w ? v[k] : ~0ull;
#pragma unroll
        for (int e = 0; e < SLO_WARP_RECORDS; e++) if (y < x[e] || (y == x[e] && k < j0 + e)) r[e]++;
      }
#pragma unroll 4
      for (int c = front > cj ? front : cj + 1; c < c1; c++) {
        const int k = c * 32 + lane;
        const uint64_t y = k < a.w ? v[k] : ~0ull;      // (bad records are ~0 too: never smaller)
#pragma unroll
        for (int e = 0; e < SLO_WARP_RECORDS; e++) if (y < x[e]) r[e]++;
      }
#pragma unroll
      for (int e = 0; e < SLO_WARP_RECORDS; e++) {
        if (x[e] == ~0ull) {      // the largest value there is: bad records look equal to it
          r[e] = 0;
          for (int k = c0 * 32 + lane; k < c1 * 32 && k < a.w; k += 32) r[e] += v[k] < x[e] || (k < j0 + e && valid(k)) ? 1u : 0u;
        }
        const uint32_t all = __reduce_add_sync(0xffffffffu, r[e]);
        if (lane == 0) atomicAdd(&rank[(warp & 7) * SLO_WARP_RECORDS + e], all);
      }
    };
    count(s_ttft, s_rank);
    count(s_tpot, s_rank + SLO_WIN_RECORDS);
  }
  __syncthreads();
  const int j = (int)blockIdx.x * SLO_WIN_RECORDS + warp;      // a record per warp: has some priority asked for its ranks?
  if (j >= a.w || !valid(j)) return;
  const uint64_t t = s_ttft[j], q = s_tpot[j];
  const uint32_t rt = s_rank[warp], rq = s_rank[SLO_WIN_RECORDS + warp];
  for (int p = lane; p < N; p += 32) {
    if (s_idx[p] == rt) {
      const int64_t wait = a.win_queue[j];
      a.tab->ref_ttft[p] = (int64_t)(t ^ (1ull << 63));
      a.tab->ref_queue[p] = wait;
      a.tab->delta[p] = wait - a.last_queue[p];
    }
    if (s_idx[p] == rq) a.tab->ref_tpot[p] = (int64_t)(q ^ (1ull << 63));
  }
}

__global__ void __launch_bounds__(SLO_THREADS) k_slo_assign(const SloArgs a) {
  cudaGridDependencySynchronize();      // set up while k_slo_window runs
  const int w = a.tab->w_valid;
  uint32_t bad = 0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < a.n_new; i += (int64_t)gridDim.x * blockDim.x) {
    const int32_t pr = a.new_prio[i];
    int64_t ttft = 0, tpot = 0;
    if (pr < 0 || pr >= a.n_prio) bad |= HFX_ST_BAD_CLASS;
    else {
      ttft = a.ttft_max[pr]; tpot = a.tpot_max[pr];
      if (w > 0) {
        const bool first = a.tab->first_row[a.par][pr] == (unsigned long long)i;
        ttft = a.tab->ref_ttft[pr] - (first ? a.tab->delta[pr] : 0);
        tpot = a.tab->ref_tpot[pr];
        if (first) a.last_queue[pr] = a.tab->ref_queue[pr];      // (the others read the delay from the table)
      }
      const bool hp = a.tab->higher_pending[pr] != 0;
      const int64_t lo_t = hp ? a.ttft_min[pr] : a.ttft_min_relaxed[pr], hi_t = a.ttft_max[pr];
      const int64_t lo_p = hp ? a.tpot_min[pr] : a.tpot_min_relaxed[pr], hi_p = a.tpot_max[pr];
      ttft = ttft < lo_t ? lo_t : (ttft > hi_t ? hi_t : ttft);
      tpot = tpot < lo_p ? lo_p : (tpot > hi_p ? hi_p : tpot);
    }
    a.ttft_out[i] = ttft;
    a.tpot_out[i] = tpot;
  }
  if (bad) atomicOr(a.status, bad);
}

int hfx_slomap_configure() {
  if (cudaFuncSetAttribute(k_slo_window, cudaFuncAttributeMaxDynamicSharedMemorySize, 16 * SLO_WINDOW_MAX) != cudaSuccess)
    return HFX_E_CUDA;
  return HFX_OK;
}

int hfx_launch_slo_map(hfx_sched *s, int32_t n_prio, const hfx_slo_window *win, const hfx_slo_bounds *b, int64_t *last_queue,
                       const int32_t *pending, const int32_t *new_prio, int64_t n_new, int64_t *ttft_out, int64_t *tpot_out) {
  SloArgs a;
  a.win_prio = win->prio; a.win_ttft = win->ttft_ns; a.win_tpot = win->tpot_ns; a.win_queue = win->queue_ns; a.w = win->w;
  a.ttft_min = b->ttft_min_ns; a.ttft_max = b->ttft_max_ns; a.ttft_min_relaxed = b->ttft_min_relaxed_ns;
  a.tpot_min = b->tpot_min_ns; a.tpot_max = b->tpot_max_ns; a.tpot_min_relaxed = b->tpot_min_relaxed_ns;
  a.last_queue = last_queue; a.pending = pending; a.new_prio = new_prio; a.n_new = n_new;
  a.ttft_out = ttft_out; a.tpot_out = tpot_out; a.n_prio = n_prio;
  a.tab = reinterpret_cast<SloTable *>(s->d_slo); a.status = s->d_status;
  a.par = (int32_t)s->slo_parity;
  a.win_blocks = win->w > 0 ? (win->w + SLO_WIN_RECORDS - 1) / SLO_WIN_RECORDS : 1;
  cudaLaunchConfig_t cfg;
  memset(&cfg, 0, sizeof(cfg));
  cfg.stream = s->stream;
  {
    KernelScope ks(s, KSLOT_SLOMAP);
    cfg.gridDim = dim3((unsigned)(a.win_blocks + (n_new + SLO_WIN_THREADS - 1) / SLO_WIN_THREADS)); cfg.blockDim = dim3(SLO_WIN_THREADS);
    cfg.dynamicSmemBytes = 16 * (size_t)(win->w > 0 ? win->w : 1);
    if (cudaLaunchKernelEx(&cfg, k_slo_window, a) != cudaSuccess) { cudaGetLastError(); return HFX_E_CUDA; }
  }
  s->slo_parity ^= 1u;      // (once the kernel that uses one copy and clears the other is on its way)
  if (n_new > 0) {
    int grid = (int)((n_new + SLO_THREADS - 1) / SLO_THREADS);
    if (grid > s->n_sm * 8) grid = s->n_sm * 8;
    KernelScope ks(s, KSLOT_SLOMAP);
    cfg.gridDim = dim3(grid); cfg.blockDim = dim3(SLO_THREADS); cfg.dynamicSmemBytes = 0;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = s->profiling ? 0 : 1;
    if (cudaLaunchKernelEx(&cfg, k_slo_assign, a) != cudaSuccess) { cudaGetLastError(); return HFX_E_CUDA; }
  }
  return cudaGetLastError() == cudaSuccess ? HFX_OK : HFX_E_CUDA;
}

size_t hfx_slomap_workspace_bytes() { return sizeof(SloTable); }
