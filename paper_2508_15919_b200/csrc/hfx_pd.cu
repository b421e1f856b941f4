// hfx_pd_migrate: hand-off of prefilled requests from the P instances to their partner D instances in
// the disaggregated mode (Sec. 3.3.1 "Disaggregated Mode"); with hfx_sched_step + HFX_COMMIT it couples
// the two stages.
//
//   k_pd_rows    one streaming pass: a request RUNNING on a P instance whose KV transfer
//                (x0 + x1 * prompt_len after its first token) has ended by its partner's clock becomes
//                QUEUED on the partner; otherwise it bids for the partner's wake-up time.  Rows that
//                keep a D instance occupied (in flight, or queued and arrived) mark it busy.
//   k_pd_clock   a D instance that is not busy is woken at the earliest end of a transfer to it.
// A row that moves makes its new instance busy in the same pass, so the two kernels need no third; k_pd_clock leaves the
// wake-up times, busy marks and the count as the next call wants to find them (all zero).  Both are set up while the
// kernel before them drains.  Bound by launches and the pass's loads: a round of committed step
// and hand-off over 1 M rows takes 56.7 us, 61.3 with a third kernel that set the marks up and one row to a thread.
#include "hfx_internal.cuh"

#define PD_THREADS 256

struct PdArgs {
  int32_t *replica_id; const uint8_t *class_id; uint8_t *state; const int32_t *prompt_len; const int32_t *gen;
  const int64_t *arrival; const int64_t *first_token; int64_t n;
  int64_t *now; const int32_t *pair; const uint8_t *mode; int64_t x0, x1;
  unsigned long long *wake; uint32_t *busy; uint32_t *moved; int32_t *n_moved; uint32_t *status;
};

// wake-up times are kept so that the largest is the earliest and zero is never
__device__ __forceinline__ unsigned long long wake_of(int64_t t) { return ~((unsigned long long)t ^ (1ull << 63)); }

__global__ void __launch_bounds__(PD_THREADS) k_pd_rows(const HfxParams p, const PdArgs a) {
  cudaTriggerProgrammaticLaunchCompletion();
  cudaGridDependencySynchronize();
  const int R = p.n_replicas;
  uint32_t bad = 0, moved = 0;
  auto do_row = [&](int64_t i, int32_t r, uint32_t cls, uint32_t st, int32_t prompt, int32_t gen) {
    if (r == -1 && st == HFX_QUEUED) return;       // still in the global queue
    if (r < 0 || r >= R) { bad |= HFX_ST_BAD_REPLICA; return; }
    bool ok = true;
    if (cls >= (uint32_t)p.n_classes) { bad |= HFX_ST_BAD_CLASS; ok = false; }
    if (prompt < 0 || prompt > HFX_MAX_TOKENS || gen < 0 || gen > HFX_MAX_TOKENS) { bad |= HFX_ST_BAD_LEN; ok = false; }
    if (!ok) return;
    const int mode = a.mode[r];
    if (mode == HFX_DECODE) {
      if ((st == HFX_RUNNING || (st == HFX_QUEUED && a.arrival[i] <= a.now[r])) && a.busy[r] == 0) atomicExch(&a.busy[r], 1u);
    } else if (mode == HFX_PREFILL && st == HFX_RUNNING) {
      const int32_t d = a.pair[r];
      if (d < 0 || d >= R || a.mode[d] != HFX_DECODE) { bad |= HFX_ST_BAD_REPLICA; return; }
      const int64_t ready = a.first_token[i] + a.x0 + a.x1 * (int64_t)prompt;
      if (ready <= a.now[d]) {
        a.replica_id[i] = d;
        a.state[i] = HFX_QUEUED;
        if (a.arrival[i] <= a.now[d]) atomicExch(&a.busy[d], 1u);      // prefilled and arrived: it occupies the D instance's queue
        moved++;
      } else atomicMax(&a.wake[d], wake_of(ready));
    }
  };
  // four rows to a thread, a load per column (the columns start on 16 bytes)
  const int64_t nvec = a.n >> 2, stride = (int64_t)gridDim.x * blockDim.x, first = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  for (int64_t v = first; v < nvec; v += stride) {
    const int4 r = reinterpret_cast<const int4 *>(a.replica_id)[v];
    const uchar4 cls = reinterpret_cast<const uchar4 *>(a.class_id)[v], st = reinterpret_cast<const uchar4 *>(a.state)[v];
    const int4 pr = reinterpret_cast<const int4 *>(a.prompt_len)[v], ge = reinterpret_cast<const int4 *>(a.gen)[v];
    do_row(4 * v, r.x, cls.x, st.x, pr.x, ge.x);
    do_row(4 * v + 1, r.y, cls.y, st.y, pr.y, ge.y);
    do_row(4 * v + 2, r.z, cls.z, st.z, pr.z, ge.z);
    do_row(4 * v + 3, r.w, cls.w, st.w, pr.w, ge.w);
  }
  if (const int64_t i = 4 * nvec + first; i < a.n) do_row(i, a.replica_id[i], a.class_id[i], a.state[i], a.prompt_len[i], a.gen[i]);
  moved = __reduce_add_sync(0xffffffffu, moved);
  if (moved && (threadIdx.x & 31) == 0) atomicAdd(a.moved, moved);
  if (bad) atomicOr(a.status, bad);
}

__global__ void __launch_bounds__(PD_THREADS) k_pd_clock(const HfxParams p, const PdArgs a) {
  cudaTriggerProgrammaticLaunchCompletion();
  cudaGridDependencySynchronize();
  const int d = blockIdx.x * blockDim.x + threadIdx.x;
  if (d == 0) { if (a.n_moved) *a.n_moved = (int32_t)*a.moved; *a.moved = 0; }
  if (d >= p.n_replicas || a.mode[d] != HFX_DECODE) return;      // (only DECODE instances are ever marked)
  const unsigned long long w = a.wake[d];
  const int64_t t = (int64_t)(~w ^ (1ull << 63));
  if (a.busy[d] == 0 && w != 0 && t > a.now[d]) a.now[d] = t;
  a.wake[d] = 0; a.busy[d] = 0;
}

size_t hfx_pd_workspace_bytes(int n_replicas) { return 16 + (size_t)n_replicas * 16; }

int hfx_launch_pd_migrate(hfx_sched *s, const hfx_table *t, int32_t *replica_id, int64_t *now, const int32_t *pair, int64_t x0,
                          int64_t x1, int32_t *n_moved) {
  const int R = s->p.n_replicas;
  PdArgs a;
  unsigned char *ws = reinterpret_cast<unsigned char *>(s->d_pd);
  a.moved = reinterpret_cast<uint32_t *>(ws);
  a.wake = reinterpret_cast<unsigned long long *>(ws + 16);
  a.busy = reinterpret_cast<uint32_t *>(ws + 16 + (size_t)R * 8);
  a.replica_id = replica_id; a.class_id = t->class_id; a.state = t->state; a.prompt_len = t->prompt_len; a.gen = t->gen;
  a.arrival = t->arrival_ns; a.first_token = t->first_token_ns; a.n = t->n_rows;
  a.now = now; a.pair = pair; a.mode = s->d_mode; a.x0 = x0; a.x1 = x1; a.n_moved = n_moved; a.status = s->d_status;
  cudaStream_t st = s->stream;
  cudaLaunchConfig_t cfg;
  memset(&cfg, 0, sizeof(cfg));
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.blockDim = dim3(PD_THREADS); cfg.stream = st; cfg.attrs = attr; cfg.numAttrs = s->profiling ? 0 : 1;
  cudaError_t e = cudaSuccess;
  if (s->pd_unsettled) e = cudaMemsetAsync(s->d_pd, 0, hfx_pd_workspace_bytes(R), st);
  if (e == cudaSuccess) {
    s->pd_unsettled = true;
    KernelScope ks(s, KSLOT_PD);
    int64_t grid = ((t->n_rows >> 2) + PD_THREADS - 1) / PD_THREADS;
    if (grid > s->n_sm * 8) grid = s->n_sm * 8;
    if (grid < 1) grid = 1;
    cfg.gridDim = dim3((unsigned)grid);
    e = cudaLaunchKernelEx(&cfg, k_pd_rows, s->p, a);
  }
  if (e == cudaSuccess) {
    KernelScope ks(s, KSLOT_PD);
    cfg.gridDim = dim3((unsigned)((R + PD_THREADS - 1) / PD_THREADS));
    e = cudaLaunchKernelEx(&cfg, k_pd_clock, s->p, a);
  }
  if (e == cudaSuccess) s->pd_unsettled = false;
  return cuda_rc(e);
}
