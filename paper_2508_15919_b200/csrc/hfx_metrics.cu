// hfx_attainment: SLO attainment over a request table (Problem Definition, Eq. 2) per SLO class and in
// total, with the sums behind the mean TTFT and the mean end-to-end time.
//
// One streaming pass, two neighbouring rows per thread and round (the widest loads that leave a warp's rows of an 8-byte
// column contiguous), bound by the 46 bytes it reads per row.  Up to eight
// classes a thread keeps every class's totals in registers (the four counts packed into one word, the two sums), which
// costs a few predicated additions per row and class; more classes are totalled per warp, one class of the warp at a time.
// (Shared-memory atomics per row and field, as before, queue up behind each other: there are few classes.  1,048,576
// rows, 4 classes: 187 us with them, 14.7 us now.)  Blocks add their totals to an accumulator of the scheduler once; the last one writes
// the output and clears the accumulator for the next call.
#include "hfx_internal.cuh"

#define ATT_THREADS 256
#define ATT_FIELDS 6
// Classes whose totals a thread keeps in registers: eight, in an instance of its own up to four.  1,048,576 rows, calls back to back: up to four
// classes 13.4 - 15.3 us with room for four, 21.4 - 23.4 with room for eight (registers, and additions for classes that are not there),
// 19.3 - 39.9 per warp; five to eight 23.6 - 25.3 in registers, 46 - 66 per warp; per warp 72 for nine, 182 for sixty-four.
#define ATT_REG_CLASSES 8

struct AttArgs {
  const uint8_t *class_id; const uint8_t *state; const int32_t *prompt_len; const int32_t *output_len; const int32_t *gen;
  const int64_t *arrival; const int64_t *first_token; const int64_t *last_token; const int64_t *finish;
  int64_t n; int64_t *out; unsigned long long *acc; uint32_t *status;      // acc: HFX_MAX_CLASSES x ATT_FIELDS totals, then the count of finished blocks
};

// what one row adds: counts (requests | DONE << 16 | attained << 32 | REJECTED << 48), TTFT, E2E
struct AttRow { uint32_t cls; unsigned long long counts, ttft, e2e; };

__device__ __forceinline__ AttRow att_row(const int64_t *s_ttft, const int64_t *s_tpot, uint32_t K, uint32_t cls, uint32_t st, int32_t prompt, int32_t gen,
                                          int32_t outlen, int64_t arrival, int64_t first, int64_t last, int64_t finish, uint32_t &bad) {
  AttRow r;
  r.cls = cls; r.counts = 0; r.ttft = 0; r.e2e = 0;
  bool ok = true;
  if (cls >= K) { bad |= HFX_ST_BAD_CLASS; ok = false; }
  if ((uint32_t)prompt > HFX_MAX_TOKENS || (uint32_t)gen > HFX_MAX_TOKENS) { bad |= HFX_ST_BAD_LEN; ok = false; }
  if (!ok) return r;
  r.counts = 1;
  if (st == HFX_REJECTED) r.counts |= 1ull << 48;
  if (st == HFX_RUNNING || st == HFX_DONE) r.ttft = (unsigned long long)(first - arrival);
  if (st == HFX_DONE) {
    const int64_t ttft_slo = s_ttft[cls], tpot_slo = s_tpot[cls], x = last - first;
    // floor(x / (outlen - 1)) <= tpot_slo without the division: x < (tpot_slo + 1) (outlen - 1); 0 for outlen <= 1
    bool tp = true;
    if (tpot_slo > 0 && outlen > 1 && x > 0) {
      const uint64_t t = (uint64_t)tpot_slo + 1, d = (uint64_t)(outlen - 1);
      tp = __umul64hi(t, d) != 0 || (uint64_t)x < t * d;
    }
    r.counts |= 1ull << 16;
    r.e2e = (unsigned long long)(finish - arrival);
    if ((ttft_slo <= 0 || first - arrival <= ttft_slo) && tp) r.counts |= 1ull << 32;
  }
  return r;
}

// KR classes in registers (0: totals per warp, any number of classes)
template <int KR>
__global__ void __launch_bounds__(ATT_THREADS) k_attainment(const HfxParams p, const AttArgs a) {
  __shared__ unsigned long long s_acc[KR > 0 ? 1 : HFX_MAX_CLASSES * ATT_FIELDS], s_warp[ATT_THREADS / 32][KR > 0 ? KR * ATT_FIELDS : 1];
  __shared__ int64_t s_ttft[HFX_MAX_CLASSES], s_tpot[HFX_MAX_CLASSES];
  __shared__ bool s_last;
  const int K = p.n_classes, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (KR == 0) for (int k = threadIdx.x; k < K * ATT_FIELDS; k += blockDim.x) s_acc[k] = 0;
  for (int k = threadIdx.x; k < K; k += blockDim.x) { s_ttft[k] = p.ttft[k]; s_tpot[k] = p.tpot[k]; }
  __syncthreads();
  uint32_t bad = 0;
  constexpr int KN = KR > 0 ? KR : 1;
  unsigned long long counts[KN], ttft[KN], e2e[KN];
#pragma unroll
  for (int c = 0; c < KN; c++) { counts[c] = 0; ttft[c] = 0; e2e[c] = 0; }
  auto spill = [&](int c, unsigned long long n, unsigned long long t, unsigned long long e) {      // totals of class c into the block's
#pragma unroll
    for (int f = 0; f < 4; f++) { const unsigned long long x = (n >> (16 * f)) & 0xffffull; if (x) atomicAdd(&s_acc[c * ATT_FIELDS + f], x); }
    if (t) atomicAdd(&s_acc[c * ATT_FIELDS + 4], t);
    if (e) atomicAdd(&s_acc[c * ATT_FIELDS + 5], e);
  };
  auto add = [&](const AttRow &r) {
    if (KR > 0) {
#pragma unroll
      for (int c = 0; c < KN; c++) if (r.cls == (uint32_t)c) { counts[c] += r.counts; ttft[c] += r.ttft; e2e[c] += r.e2e; }
    } else {      // (whole warps call)
      uint32_t todo = __ballot_sync(0xffffffffu, r.counts != 0);
      while (todo) {
        const uint32_t c = __shfl_sync(0xffffffffu, r.cls, __ffs(todo) - 1);
        const bool me = r.counts != 0 && r.cls == c;
        const uint32_t mask = __ballot_sync(0xffffffffu, me);
        todo &= ~mask;
        unsigned long long n = 0;
#pragma unroll
        for (int f = 0; f < 4; f++) n |= (unsigned long long)__popc(__ballot_sync(0xffffffffu, me && ((r.counts >> (16 * f)) & 1ull))) << (16 * f);
        const unsigned long long t = (unsigned long long)warp_sum_i64(me ? (int64_t)r.ttft : 0), e = (unsigned long long)warp_sum_i64(me ? (int64_t)r.e2e : 0);
        if (lane == 0) spill((int)c, n, t, e);
      }
    }
  };
  auto one = [&](int64_t i) {
    AttRow r;
    r.cls = 0; r.counts = 0; r.ttft = 0; r.e2e = 0;
    if (i < a.n) r = att_row(s_ttft, s_tpot, (uint32_t)K, a.class_id[i], a.state[i], a.prompt_len[i], a.gen[i], a.output_len[i], a.arrival[i], a.first_token[i],
                             a.last_token[i], a.finish[i], bad);
    add(r);
  };
  const int64_t n2 = a.n >> 1;
#pragma unroll 2
  for (int64_t v0 = (int64_t)blockIdx.x * blockDim.x; v0 < n2; v0 += (int64_t)gridDim.x * blockDim.x) {
    const int64_t v = v0 + threadIdx.x;
    AttRow x, y;
    x.cls = 0; x.counts = 0; x.ttft = 0; x.e2e = 0;
    y = x;
    if (v < n2) {
      const uchar2 cls = __ldg(reinterpret_cast<const uchar2 *>(a.class_id) + v), st = __ldg(reinterpret_cast<const uchar2 *>(a.state) + v);
      const int2 pr = __ldg(reinterpret_cast<const int2 *>(a.prompt_len) + v), ge = __ldg(reinterpret_cast<const int2 *>(a.gen) + v);
      const int2 ol = __ldg(reinterpret_cast<const int2 *>(a.output_len) + v);
      const longlong2 ar = __ldg(reinterpret_cast<const longlong2 *>(a.arrival) + v), ft = __ldg(reinterpret_cast<const longlong2 *>(a.first_token) + v);
      const longlong2 la = __ldg(reinterpret_cast<const longlong2 *>(a.last_token) + v), fi = __ldg(reinterpret_cast<const longlong2 *>(a.finish) + v);
      x = att_row(s_ttft, s_tpot, (uint32_t)K, cls.x, st.x, pr.x, ge.x, ol.x, ar.x, ft.x, la.x, fi.x, bad);
      y = att_row(s_ttft, s_tpot, (uint32_t)K, cls.y, st.y, pr.y, ge.y, ol.y, ar.y, ft.y, la.y, fi.y, bad);
    }
    add(x);
    add(y);
  }
  if (blockIdx.x == 0 && threadIdx.x < 32) one((n2 << 1) + threadIdx.x);      // at most one row is left
  if (bad) atomicOr(a.status, bad);
  if (KR > 0) {
    // a thread's counts stay below 2^16 (the grid is sized so); a warp's are widened before they are added up
#pragma unroll
    for (int c = 0; c < KN; c++) {
      uint32_t n[4];
#pragma unroll
      for (int f = 0; f < 4; f++) n[f] = __reduce_add_sync(0xffffffffu, (uint32_t)(counts[c] >> (16 * f)) & 0xffffu);
      const unsigned long long t = (unsigned long long)warp_sum_i64((int64_t)ttft[c]), e = (unsigned long long)warp_sum_i64((int64_t)e2e[c]);
      if (lane < ATT_FIELDS) s_warp[warp][c * ATT_FIELDS + lane] = lane == 0 ? n[0] : lane == 1 ? n[1] : lane == 2 ? n[2] : lane == 3 ? n[3] : lane == 4 ? t : e;
    }
    __syncthreads();
    for (int k = threadIdx.x; k < K * ATT_FIELDS; k += blockDim.x) {
      unsigned long long x = 0;
#pragma unroll
      for (int w = 0; w < ATT_THREADS / 32; w++) x += s_warp[w][k];
      if (x) atomicAdd(&a.acc[k], x);
    }
  } else {
    __syncthreads();
    for (int k = threadIdx.x; k < K * ATT_FIELDS; k += blockDim.x)
      if (s_acc[k]) atomicAdd(&a.acc[k], s_acc[k]);
  }
  __threadfence();
  __syncthreads();
  unsigned long long *done = a.acc + HFX_MAX_CLASSES * ATT_FIELDS;
  if (threadIdx.x == 0) s_last = atomicAdd(done, 1ull) == (unsigned long long)gridDim.x - 1;
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  for (int k = threadIdx.x; k < ATT_FIELDS; k += blockDim.x) {      // the totals
    unsigned long long x = 0;
    for (int c = 0; c < K; c++) x += __ldcg(a.acc + c * ATT_FIELDS + k);
    a.out[K * ATT_FIELDS + k] = (int64_t)x;
  }
  __syncthreads();
  for (int k = threadIdx.x; k < K * ATT_FIELDS; k += blockDim.x) { a.out[k] = (int64_t)__ldcg(a.acc + k); a.acc[k] = 0; }
  if (threadIdx.x == 0) *done = 0;
}

size_t hfx_attainment_workspace_bytes() { return sizeof(unsigned long long) * (HFX_MAX_CLASSES * ATT_FIELDS + 1); }

int hfx_launch_attainment(hfx_sched *s, const hfx_table *t, int64_t *out) {
  AttArgs a;
  a.class_id = t->class_id; a.state = t->state; a.prompt_len = t->prompt_len; a.output_len = t->output_len; a.gen = t->gen;
  a.arrival = t->arrival_ns; a.first_token = t->first_token_ns; a.last_token = t->last_token_ns; a.finish = t->finish_ns;
  a.n = t->n_rows; a.out = out; a.acc = s->d_att; a.status = s->d_status;
  // up to four blocks per SM, so a thread sees far fewer than 2^16 of the at most 2^27 rows (its counts are 16 bits wide)
  int64_t want = (t->n_rows / 2 + ATT_THREADS - 1) / ATT_THREADS;
  int grid = (int)(want < (int64_t)s->n_sm * 4 ? want : (int64_t)s->n_sm * 4);
  if (grid < 1) grid = 1;
  KernelScope ks(s, KSLOT_METRICS);
  if (s->p.n_classes <= 4) k_attainment<4><<<grid, ATT_THREADS, 0, s->stream>>>(s->p, a);
  else if (s->p.n_classes <= ATT_REG_CLASSES) k_attainment<ATT_REG_CLASSES><<<grid, ATT_THREADS, 0, s->stream>>>(s->p, a);
  else k_attainment<0><<<grid, ATT_THREADS, 0, s->stream>>>(s->p, a);
  return cudaGetLastError() == cudaSuccess ? HFX_OK : HFX_E_CUDA;
}
