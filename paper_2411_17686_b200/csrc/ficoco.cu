// C ABI of libficoco: context, plans, argument validation and kernel launches.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>
#include <limits.h>
#include <stdlib.h>
#include <string.h>

#include <algorithm>
#include <new>
#include <mutex>
#include <vector>

#include "../../include/ficoco.h"
#include "common.cuh"
#include "correlate_plan.h"
#include "filter_plan.h"
#include "kernels_correlate.cuh"
#include "kernels_correlate_umma.cuh"
#include "kernels_correlate_umma_f32.cuh"
#include "kernels_filter.cuh"
#include "kernels_filter_fused.cuh"
#include "kernels_merge.cuh"
#include "kernels_relation.cuh"
#include "plan_tables.h"

using namespace ficoco;

namespace {

constexpr int N_PLANS = 16;
constexpr int PART_PER_TOKEN = 64;   // partial top-list entries budgeted per token row
constexpr int OUT_ROWS_PER_CTA = 16;  // the merge kernel's work table is sized for this many (wide rows: fewer)

size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

// host-buffer entry points: image groups pipelined over upload / kernels / download
constexpr int HOST_MAX_GROUPS = 8;
constexpr size_t HOST_GROUP_BYTES = 8u << 20;   // at least this many token bytes per group

struct PlanKey {
  int mode;  // 0 = V, 1 = L
  int dtype, batch, dim, n_text, has_cls, max_targets, avg;
  int rel = 0;  // 0: cosine relation of the tokens; 1 / 2: caller-supplied relation, by row / by column
  int conv = 0; // 1: "convergent correlation" ablation (one additional token per image, no merging)
  double eps;
  std::vector<int> ntok, keep, gh, gw;
  bool operator==(const PlanKey& o) const {
    return mode == o.mode && dtype == o.dtype && batch == o.batch && dim == o.dim &&
           n_text == o.n_text && has_cls == o.has_cls && max_targets == o.max_targets && avg == o.avg && rel == o.rel && conv == o.conv &&
           eps == o.eps && ntok == o.ntok && keep == o.keep && gh == o.gh && gw == o.gw;
  }
};

struct Plan {
  bool valid = false;
  unsigned long long stamp = 0;
  PlanKey key;
  // device tables (one behind the other in the slot)
  size_t table_bytes = 0;
  ImgDesc* d_desc = nullptr;
  WorkItem* d_rows = nullptr;
  WorkItem* d_corr = nullptr;
  WorkItem* d_out = nullptr;
  int n_rows = 0, n_corr = 0, n_out = 0;
  size_t m_smem = 0;            // shared memory of a merge CTA: the input rows of its output rows
  // totals and maxima used to size launches and inspection copies
  int tot_patch = 0, tot_src = 0, tot_tgt = 0, tot_out_rows = 0;
  int max_np = 0, max_tgt = 0, max_src = 0, max_rc = 0, max_nwin_cells = 0, max_list = 0;
  // fused persistent filter kernel
  bool fused = false;
  int* d_ctafirst = nullptr;
  int* d_out_cu = nullptr;      // device int32[batch + 1]: first output row of every image, then the total
  int f_grid = 0, f_nstage = 0, f_vpl = 0;
  size_t f_smem = 0;
  // tensor-core correlate (bf16, hidden size a multiple of 64, FiCoCo-V)
  bool need_finalize = false;   // some image merges nothing: its per-token counts are zeroed by a kernel
  bool umma = false;
  bool um_f32 = false;          // fp32 tokens split into three bf16 terms (k_correlate_umma_f32)
  bool uf_small = false;        // fp32 tiles of 32 x 32 instead of 128 x 64
  int um_b_bytes = 0, uf_stg_off = 0;     // uf_stg_off: where the slots for fp32 values lie
  int um_stage_bytes = 0, um_a_bytes = 0, um_tmem_cols = 0, um_nstage = 0, um_ksub = 1, um_text_off = 0;
  bool um_text_late = false;
  size_t um_smem = 0;
  std::vector<ImgDesc> h_desc;
};

// ---- what the last step on a stream wrote ------------------------------------------------------
// The filter grid of a step may start under the tail of the merge grid of the step launched
// before it on the same stream.  That is only sound when the new step does not read what the
// older one is still writing, so the output spans of the last step are remembered per
// (device, stream), over all contexts of the process; a step whose inputs touch them, or whose
// stream has no record, is launched fully serialized.
struct Span {
  const char* lo = nullptr;
  const char* hi = nullptr;
};
inline Span span_of(const void* ptr, size_t bytes) {
  Span s;
  if (ptr != nullptr && bytes > 0) { s.lo = (const char*)ptr; s.hi = s.lo + bytes; }
  return s;
}
inline bool spans_overlap(const Span& a, const Span& b) {
  return a.lo != nullptr && b.lo != nullptr && a.lo < b.hi && b.lo < a.hi;
}
constexpr int N_TAILS = 16, N_SPANS = 4;
struct StreamTail {
  bool used = false;
  int device = 0;
  cudaStream_t st = nullptr;
  Span out[N_SPANS];
  unsigned long long stamp = 0;
};
std::mutex g_tail_mu;
StreamTail g_tail[N_TAILS];
unsigned long long g_tail_clock = 0;

bool inputs_clear_of_last_outputs(int device, cudaStream_t st, const Span* in, int n_in) {
  std::lock_guard<std::mutex> lk(g_tail_mu);
  for (int i = 0; i < N_TAILS; ++i) {
    const StreamTail& t = g_tail[i];
    if (!t.used || t.device != device || t.st != st) continue;
    for (int a = 0; a < n_in; ++a)
      for (int b = 0; b < N_SPANS; ++b)
        if (spans_overlap(in[a], t.out[b])) return false;
    return true;
  }
  return false;
}

void record_last_outputs(int device, cudaStream_t st, const Span* out, int n_out) {
  std::lock_guard<std::mutex> lk(g_tail_mu);
  int slot = -1;
  for (int i = 0; i < N_TAILS && slot < 0; ++i)
    if (g_tail[i].used && g_tail[i].device == device && g_tail[i].st == st) slot = i;
  if (slot < 0) {
    slot = 0;
    for (int i = 0; i < N_TAILS; ++i) {
      if (!g_tail[i].used) { slot = i; break; }
      if (g_tail[i].stamp < g_tail[slot].stamp) slot = i;
    }
  }
  StreamTail& t = g_tail[slot];
  t.used = true;
  t.device = device;
  t.st = st;
  t.stamp = ++g_tail_clock;
  for (int b = 0; b < N_SPANS; ++b) t.out[b] = b < n_out ? out[b] : Span();
}

}  // namespace

__global__ void k_launch_probe() {}

struct ficoco_ctx {
  int device = 0;
  long long max_tokens = 0;
  int max_dim = 0, max_batch = 0, max_text = 0;
  int last_cuda = 0;
  int launches = 0;
  unsigned long long clock = 0;

  char* d_base = nullptr;
  size_t d_bytes = 0;
  // scratch arrays
  float* rn = nullptr;
  float* partial = nullptr;
  float* msum = nullptr;     // [B][max_dim] column sums of the unfused filter
  float* s_raw = nullptr;
  float* s_pen = nullptr;
  int* S_idx = nullptr;
  int* T_idx = nullptr;
  float* part_val = nullptr;
  int* part_idx = nullptr;
  int* corr_cnt = nullptr;
  int* e_tgt = nullptr;     // compact per-image entry arrays, L slots per discarded token
  float* e_w = nullptr;
  float* e_c = nullptr;
  float* tau = nullptr;
  float* tmean = nullptr;
  unsigned* status = nullptr;
  int* tile_cnt = nullptr;  // per source tile: column splits of the correlate kernel that are done
  int* img_cnt = nullptr;   // two sets of 3 * max_batch per-image counters of the fused filter kernel
  unsigned long long epoch = 0;          // fused filter launches so far (its parity picks the counter set)
  int last_parity = 0;                   // counter set of the latest fused filter launch
  unsigned long long wait_ns = WAIT_NS_DEFAULT;   // bound of every device-side wait
  int dbg_extra_arrivals = 0;            // testing hook: arrivals the fused filter waits for that never come
  int num_sms = 0;
  bool coop_ok = false;
  bool coop_pdl_ok = false;  // a cooperative grid may also be a programmatic dependent
  char* plan_slots = nullptr;
  size_t slot_bytes = 0;
  int cap_rows = 0, cap_corr = 0, cap_out = 0;
  long long cap_part = 0;

  char* h_stage = nullptr;  // pinned, slot_bytes
  Plan plans[N_PLANS];
  Plan* last_plan = nullptr;

  // optional per-kernel timing (events recorded between launches)
  bool prof_on = false;
  std::vector<cudaEvent_t> prof_ev;
  size_t prof_used = 0;
  std::vector<int> prof_name;            // per recorded event: index into prof_acc, -1 = end of call
  struct ProfAcc { const char* name; double ms; long long launches; };
  std::vector<ProfAcc> prof_acc;

  // grow-only intermediates of ficoco_v_reduce_schedule: tokens / positions ping-pong, kept indices per step
  char* sch_base = nullptr;
  size_t sch_bytes = 0;

  // grow-only staging for the host-buffer entry points
  char* hs_dev = nullptr;
  size_t hs_dev_bytes = 0;
  cudaStream_t hs_stream = nullptr;
  cudaStream_t hs_run = nullptr, hs_out = nullptr;   // kernels / downloads of the host entry points
  cudaEvent_t hs_ev[2 * HOST_MAX_GROUPS] = {};
};

#define CUDA_TRY(ctx, expr)                                  \
  do {                                                       \
    cudaError_t e__ = (expr);                                \
    if (e__ != cudaSuccess) {                                \
      (ctx)->last_cuda = (int)e__;                           \
      return FICOCO_ERR_CUDA;                                \
    }                                                        \
  } while (0)

namespace {

// Record an event in front of the kernel about to be launched (name) or at the end of a
// call (nullptr).  The time between two consecutive events is attributed to the first.
void prof_tick(ficoco_ctx* c, cudaStream_t st, const char* name) {
  if (!c->prof_on) return;
  if (c->prof_used == c->prof_ev.size()) {
    cudaEvent_t e;
    if (cudaEventCreate(&e) != cudaSuccess) return;
    c->prof_ev.push_back(e);
  }
  int idx = -1;
  if (name) {
    for (size_t i = 0; i < c->prof_acc.size(); ++i)
      if (c->prof_acc[i].name == name) idx = (int)i;
    if (idx < 0) { c->prof_acc.push_back({name, 0.0, 0}); idx = (int)c->prof_acc.size() - 1; }
  }
  cudaEventRecord(c->prof_ev[c->prof_used], st);
  if (c->prof_name.size() <= c->prof_used) c->prof_name.resize(c->prof_used + 1);
  c->prof_name[c->prof_used] = idx;
  ++c->prof_used;
}

void prof_flush(ficoco_ctx* c) {
  if (c->prof_used == 0) return;
  cudaDeviceSynchronize();
  for (size_t i = 0; i + 1 < c->prof_used; ++i) {
    const int idx = c->prof_name[i];
    if (idx < 0) continue;
    float ms = 0.f;
    if (cudaEventElapsedTime(&ms, c->prof_ev[i], c->prof_ev[i + 1]) == cudaSuccess) {
      c->prof_acc[idx].ms += ms;
      c->prof_acc[idx].launches += 1;
    }
  }
  c->prof_used = 0;
}

}  // namespace

extern "C" int ficoco_profile(ficoco_ctx* c, int enable) {
  if (!c) return FICOCO_ERR_INVALID_ARG;
  cudaSetDevice(c->device);
  c->prof_used = 0;
  c->prof_acc.clear();
  c->prof_on = enable != 0;
  return FICOCO_OK;
}

extern "C" int ficoco_profile_read(ficoco_ctx* c, int index, char* name, int name_cap, double* total_ms,
                                   long long* launches) {
  if (!c || index < 0 || !name || name_cap < 2 || !total_ms || !launches) return FICOCO_ERR_INVALID_ARG;
  cudaSetDevice(c->device);
  prof_flush(c);
  if (index >= (int)c->prof_acc.size()) return FICOCO_ERR_INVALID_ARG;
  strncpy(name, c->prof_acc[index].name, name_cap - 1);
  name[name_cap - 1] = 0;
  *total_ms = c->prof_acc[index].ms;
  *launches = c->prof_acc[index].launches;
  return FICOCO_OK;
}

extern "C" const char* ficoco_strerror(int code) {
  switch (code) {
    case FICOCO_OK: return "ok";
    case FICOCO_ERR_INVALID_ARG: return "invalid argument";
    case FICOCO_ERR_UNSUPPORTED: return "unsupported dtype, size or quantile level";
    case FICOCO_ERR_KEEP_RANGE: return "keep count out of range";
    case FICOCO_ERR_WORKSPACE: return "problem exceeds the sizes given to ficoco_create";
    case FICOCO_ERR_CUDA: return "CUDA runtime error";
    case FICOCO_ERR_TIMEOUT: return "device-side wait timed out";
    case FICOCO_ERR_CAPTURE: return "a new plan cannot be uploaded during stream capture";
    case FICOCO_ERR_GRID: return "grid smaller than the number of alive patches";
    case FICOCO_ERR_STATIC_LIMIT:
      return "problem exceeds the fixed scratch of the allocation-free entry point "
             "(at most 64 images, dim 2048, 32768 patch tokens in total)";
    default: return "unknown error";
  }
}

extern "C" void ficoco_default_params(ficoco_params* p) {
  if (!p) return;
  p->lambda_ = 0.35;
  p->beta = 0.6;
  p->gamma = 0.6;
  p->eps = 0.998;
  p->penalty_coef = 2.0;
  p->window = 2;
  p->max_targets = -1;
  p->flags = FICOCO_HAS_CLS | FICOCO_LOCAL_PENALTY;
  p->reserved = 0;
}

#ifdef FICOCO_PHASE_TIMERS
// Phase timestamps of the most recent launch of every instrumented kernel (profiling builds only).
extern "C" int ficoco_phase_read(void* host_dst, size_t bytes) {
  if (cudaDeviceSynchronize() != cudaSuccess) return FICOCO_ERR_CUDA;
  const size_t n = sizeof(unsigned long long) * PH_KERNELS * PH_CTAS * PH_SLOTS;
  if (cudaMemcpyFromSymbol(host_dst, g_phase_ts, bytes < n ? bytes : n) != cudaSuccess) return FICOCO_ERR_CUDA;
  // start the next run from empty records
  static const unsigned long long zeros[PH_SLOTS * 64] = {0};
  for (size_t o = 0; o < n; o += sizeof(zeros))
    if (cudaMemcpyToSymbol(g_phase_ts, zeros, sizeof(zeros), o) != cudaSuccess) return FICOCO_ERR_CUDA;
  const unsigned zn[PH_KERNELS] = {0};
  return cudaMemcpyToSymbol(g_phase_n, zn, sizeof(zn)) == cudaSuccess ? FICOCO_OK : FICOCO_ERR_CUDA;
}
#endif

extern "C" int ficoco_last_cuda_error(const ficoco_ctx* ctx) { return ctx ? ctx->last_cuda : 0; }
extern "C" int ficoco_debug_waits(ficoco_ctx* c, long long wait_ns, int extra_arrivals) {
  if (!c || wait_ns < 0 || extra_arrivals < 0) return FICOCO_ERR_INVALID_ARG;
  c->wait_ns = wait_ns > 0 ? (unsigned long long)wait_ns : WAIT_NS_DEFAULT;
  c->dbg_extra_arrivals = extra_arrivals;
  return FICOCO_OK;
}
__global__ void k_barrier_wait(unsigned long long wait_ns, unsigned long long* cycles) {
  __shared__ uint64_t bar;
  mbar_init(&bar, 1);
  const unsigned long long t0 = sm_cycles();
  mbar_wait(&bar, 0, wait_ns);
  *cycles = sm_cycles() - t0;
}
extern "C" int ficoco_debug_barrier_wait(ficoco_ctx* c, long long* cycles) {
  if (!c || !cycles) return FICOCO_ERR_INVALID_ARG;
  CUDA_TRY(c, cudaSetDevice(c->device));
  unsigned long long* d = reinterpret_cast<unsigned long long*>(c->status + 2);   // spare bytes behind the status word
  k_barrier_wait<<<1, 1>>>(c->wait_ns, d);
  CUDA_TRY(c, cudaMemcpy(cycles, d, sizeof(*d), cudaMemcpyDeviceToHost));
  return FICOCO_OK;
}
extern "C" int ficoco_last_launch_count(const ficoco_ctx* ctx) { return ctx ? ctx->launches : 0; }

extern "C" int ficoco_create(ficoco_ctx** out, int device, long long max_tokens, int max_dim,
                             int max_batch, int max_text) {
  if (!out || max_tokens <= 0 || max_dim <= 0 || max_batch <= 0 || max_text < 0 || device < 0)
    return FICOCO_ERR_INVALID_ARG;
  if (max_tokens > (1ll << 26) || max_dim > 16384) return FICOCO_ERR_UNSUPPORTED;
  ficoco_ctx* c = new (std::nothrow) ficoco_ctx();
  if (!c) return FICOCO_ERR_INVALID_ARG;
  c->device = device;
  c->max_tokens = max_tokens;
  c->max_dim = max_dim;
  c->max_batch = max_batch;
  c->max_text = max_text;
  cudaError_t e = cudaSetDevice(device);
  if (e != cudaSuccess) { delete c; return FICOCO_ERR_CUDA; }

  const size_t T = (size_t)max_tokens, B = (size_t)max_batch;
  {
    int v = 0;
    cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, device);
    c->num_sms = v > 0 ? v : 1;
    v = 0;
    cudaDeviceGetAttribute(&v, cudaDevAttrCooperativeLaunch, device);
    c->coop_ok = v != 0;
    // Does the runtime take a cooperative launch that also carries programmatic stream
    // serialization?  One empty grid answers it; a refusal only turns the overlap off.
    if (c->coop_ok) {
      cudaLaunchConfig_t cfg = {};
      cfg.gridDim = dim3(1);
      cfg.blockDim = dim3(32);
      cudaLaunchAttribute at[2];
      at[0].id = cudaLaunchAttributeCooperative;
      at[0].val.cooperative = 1;
      at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
      at[1].val.programmaticStreamSerializationAllowed = 1;
      cfg.attrs = at;
      cfg.numAttrs = 2;
      const cudaError_t pe = cudaLaunchKernelEx(&cfg, k_launch_probe);
      const cudaError_t se = cudaDeviceSynchronize();
      c->coop_pdl_ok = pe == cudaSuccess && se == cudaSuccess;
      if (!c->coop_pdl_ok) cudaGetLastError();
    }
  }
  c->cap_rows = (int)(MAX_CHUNKS * B);
  if (c->cap_rows < c->num_sms + (int)B + 8) c->cap_rows = c->num_sms + (int)B + 8;
  // (bf16 tiles of 64 x 256 tokens, the largest that leave room for 101 text tokens: at most n * n / (4 * 64 * 256) +
  // n / 64 + n / 256 + 1 of an image of n tokens)
  const size_t n_most = T < (size_t)MAX_IMG_TOKENS ? T : MAX_IMG_TOKENS;
  c->cap_corr = (int)std::max<size_t>(2 * (T / CBM + B) + 2048, T * n_most / (2 * UM * UN_MAX) + T / 32 + B + 64);
  // (wide rows: no more of them per merge CTA than its shared memory takes, fp32 being the widest)
  const size_t out_rows = std::min<size_t>(OUT_ROWS_PER_CTA, std::max<size_t>(1, MSTAGE_BYTES / ((size_t)max_dim * 4)));
  c->cap_out = (int)(T / out_rows + B + 2 * c->num_sms);
  c->cap_part = (long long)T * PART_PER_TOKEN;
  c->slot_bytes = align_up(plan_tables(B * sizeof(ImgDesc), sizeof(WorkItem), c->cap_rows, c->cap_corr, c->cap_out,
                                       c->num_sms + 2, B + 1).bytes, 256);

  size_t off = 0;
  auto carve = [&](size_t bytes) { size_t o = off; off += align_up(bytes, 256); return o; };
  const size_t o_rn = carve(T * 4), o_partial = carve((size_t)c->cap_rows * max_dim * 4);
  const size_t o_msum = carve((size_t)B * max_dim * 4);
  const size_t o_icnt = carve(6 * B * 4);
  const size_t o_tcnt = carve((size_t)c->cap_corr * 4);

  const size_t o_sraw = carve(T * 4), o_spen = carve(T * 4);
  const size_t o_S = carve(T * 4), o_T = carve(T * 4);
  const size_t o_pv = carve((size_t)c->cap_part * 4), o_pi = carve((size_t)c->cap_part * 4);
  const size_t o_cc = carve(T * 4), o_ct = carve(T * KCAP * 4), o_cw = carve(T * KCAP * 4);
  const size_t o_c = carve(T * KCAP * 4), o_tau = carve(T * 4);
  const size_t o_tm = carve(max_text > 0 ? T * (size_t)max_text * 4 : 256);
  const size_t o_st = carve(256);
  const size_t o_pl = carve(c->slot_bytes * N_PLANS);
  c->d_bytes = off;
  e = cudaMalloc((void**)&c->d_base, c->d_bytes);
  if (e != cudaSuccess) { c->last_cuda = (int)e; delete c; return FICOCO_ERR_CUDA; }
  e = cudaMemset(c->d_base, 0, c->d_bytes);
  if (e == cudaSuccess) e = cudaMallocHost((void**)&c->h_stage, c->slot_bytes);
  if (e != cudaSuccess) { cudaFree(c->d_base); delete c; return FICOCO_ERR_CUDA; }
  char* b = c->d_base;
  c->rn = (float*)(b + o_rn); c->partial = (float*)(b + o_partial); c->msum = (float*)(b + o_msum);
  c->s_raw = (float*)(b + o_sraw); c->s_pen = (float*)(b + o_spen);
  c->S_idx = (int*)(b + o_S); c->T_idx = (int*)(b + o_T);
  c->part_val = (float*)(b + o_pv); c->part_idx = (int*)(b + o_pi);
  c->corr_cnt = (int*)(b + o_cc); c->e_tgt = (int*)(b + o_ct); c->e_w = (float*)(b + o_cw);
  c->e_c = (float*)(b + o_c); c->tau = (float*)(b + o_tau);
  c->tmean = (float*)(b + o_tm); c->status = (unsigned*)(b + o_st);
  c->img_cnt = (int*)(b + o_icnt);
  c->tile_cnt = (int*)(b + o_tcnt);

  c->plan_slots = b + o_pl;

  // kernels that may need more than 48 KB of dynamic shared memory
  cudaFuncSetAttribute(k_select<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
  cudaFuncSetAttribute(k_select<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
  {
    const int um_smem_max = 221 * 1024;
#define FICOCO_UMMA_ATTR(LC)                                                                                  \
    cudaFuncSetAttribute(k_correlate_umma<LC, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, um_smem_max);     \
    cudaFuncSetAttribute(k_correlate_umma<LC, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize, um_smem_max);     \
    cudaFuncSetAttribute(k_correlate_umma<LC, 4>, cudaFuncAttributeMaxDynamicSharedMemorySize, um_smem_max)
    FICOCO_UMMA_ATTR(2); FICOCO_UMMA_ATTR(4); FICOCO_UMMA_ATTR(16);
#undef FICOCO_UMMA_ATTR
#define FICOCO_UF32_ATTR(LC)                                                                                       \
    cudaFuncSetAttribute(k_correlate_umma_f32<LC, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, um_smem_max); \
    cudaFuncSetAttribute(k_correlate_umma_f32<LC, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, um_smem_max)
    FICOCO_UF32_ATTR(2); FICOCO_UF32_ATTR(4); FICOCO_UF32_ATTR(16);
#undef FICOCO_UF32_ATTR
  }
  {
#define FICOCO_FUSED_ATTR(TT, V) \
    cudaFuncSetAttribute(k_filter_fused<TT, V>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)F_SMEM)
    FICOCO_FUSED_ATTR(float, 1); FICOCO_FUSED_ATTR(float, 2); FICOCO_FUSED_ATTR(float, 4);
    FICOCO_FUSED_ATTR(float, 5); FICOCO_FUSED_ATTR(float, 6); FICOCO_FUSED_ATTR(float, 7); FICOCO_FUSED_ATTR(float, 8);
    FICOCO_FUSED_ATTR(__nv_bfloat16, 1); FICOCO_FUSED_ATTR(__nv_bfloat16, 2); FICOCO_FUSED_ATTR(__nv_bfloat16, 4);
    FICOCO_FUSED_ATTR(__nv_bfloat16, 5); FICOCO_FUSED_ATTR(__nv_bfloat16, 6); FICOCO_FUSED_ATTR(__nv_bfloat16, 7);
#undef FICOCO_FUSED_ATTR
  }
  cudaFuncSetAttribute(k_merge_rows<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)MSTAGE_BYTES);
  cudaFuncSetAttribute(k_merge_rows<__nv_bfloat16>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)MSTAGE_BYTES);
  cudaFuncSetAttribute(k_correlate_simt<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SIMT_ALONE_BYTES);
  cudaFuncSetAttribute(k_correlate_simt<__nv_bfloat16>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SIMT_ALONE_BYTES);
  // Two merge CTAs need 184 KB of shared memory.  Left to itself the SM stays at the largest carve-out when the correlate
  // kernel has set it, and the 28 KB of L1 that leaves slow the streaming kernels of the next step, which start beside
  // the merge (16 FiCoCo-L sequences, correlate CTAs of 205 KB: head mean 15.5 -> 17.4 us, column sums 18.9 -> 20.9,
  // step 108 us instead of 102).  76 % is the 196 KB setting.
  cudaFuncSetAttribute(k_merge_rows<float>, cudaFuncAttributePreferredSharedMemoryCarveout, 76);
  cudaFuncSetAttribute(k_merge_rows<__nv_bfloat16>, cudaFuncAttributePreferredSharedMemoryCarveout, 76);
  // The kernels in front of them ask for 100 KB, which suits what they stream and lets them start beside their
  // neighbours; what the driver picks by itself depends on the neighbours (256 x 577 tokens: column sums 74 or 98 us, the
  // step 315 or 339; relation map: the step 41.8 or 44.8; 28 and 57 % like 43).
  {
    auto carve = [](auto* kernel, int percent = 43) { cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, percent); };
#define FICOCO_COLSUM_CARVE(V) carve(k_colsum<float, V, true>); carve(k_colsum<__nv_bfloat16, V, true>)
    FICOCO_COLSUM_CARVE(1); FICOCO_COLSUM_CARVE(2); FICOCO_COLSUM_CARVE(4); FICOCO_COLSUM_CARVE(5); FICOCO_COLSUM_CARVE(8);
#undef FICOCO_COLSUM_CARVE
    carve(k_score_rel); carve(k_correlate_rel<2>); carve(k_correlate_rel<4>); carve(k_correlate_rel<16>);
    carve(k_select<true>); carve(k_select<false>);
    // The wide column sums with the head mean have up to 128 KB of loads in flight per SM, which L1 has to hold: as much L1 as
    // there is (16 FiCoCo-L sequences of 4096 91.7 us, four 51.5; the driver's choice 93.4 and 53.0, 100 KB 101.2 and 57.7).
    carve(k_colsum_wide<float, 2, 8>, 0); carve(k_colsum_wide<float, 4, 4>, 0);
    carve(k_colsum_wide<__nv_bfloat16, 2, 8>, 0); carve(k_colsum_wide<__nv_bfloat16, 4, 4>, 0);
  }
  cudaFuncSetAttribute(k_score<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, 96 * 1024);
  cudaFuncSetAttribute(k_score<__nv_bfloat16>, cudaFuncAttributeMaxDynamicSharedMemorySize, 96 * 1024);
  if (cudaGetLastError() != cudaSuccess) { ficoco_destroy(c); return FICOCO_ERR_CUDA; }
  *out = c;
  return FICOCO_OK;
}

extern "C" int ficoco_destroy(ficoco_ctx* c) {
  if (!c) return FICOCO_ERR_INVALID_ARG;
  cudaSetDevice(c->device);
  cudaDeviceSynchronize();
  if (c->d_base) cudaFree(c->d_base);
  if (c->h_stage) cudaFreeHost(c->h_stage);
  if (c->hs_dev) cudaFree(c->hs_dev);
  if (c->sch_base) cudaFree(c->sch_base);
  if (c->hs_stream) cudaStreamDestroy(c->hs_stream);
  if (c->hs_run) cudaStreamDestroy(c->hs_run);
  if (c->hs_out) cudaStreamDestroy(c->hs_out);
  for (int i = 0; i < 2 * HOST_MAX_GROUPS; ++i)
    if (c->hs_ev[i]) cudaEventDestroy(c->hs_ev[i]);
  for (cudaEvent_t e : c->prof_ev) cudaEventDestroy(e);
  delete c;
  return FICOCO_OK;
}

// ---------------------------------------------------------------------------------------
// Plans
// ---------------------------------------------------------------------------------------
namespace {

int build_plan(ficoco_ctx* c, Plan* p, const PlanKey& key, int slot) {
  const int B = key.batch;
  const int cls = key.mode == 0 ? key.has_cls : 0;
  const int tail = key.mode == 1 ? key.n_text : 0;
  p->h_desc.assign(B, ImgDesc());
  std::vector<WorkItem> rows, corr, outw;
  long long row0 = 0, patch0 = 0, out0 = 0, src0 = 0, tgt0 = 0, ent0 = 0, part0 = 0, chunk0 = 0, rel0 = 0;
  p->max_np = p->max_tgt = p->max_src = p->max_rc = p->max_nwin_cells = p->max_list = 0;
  p->need_finalize = false;
  // tensor-core correlate: bf16 tokens, hidden size a multiple of 64.  FiCoCo-L adds its text term
  // in the epilogue from weights staged in shared memory.  With up to 101 text tokens tiles of 64 x 256, for which the work
  // tables are sized, leave room for two stages of operands; sequences with more take the SIMT kernel.
  p->umma = key.dtype == FICOCO_BF16 && key.dim % UKB == 0 &&
            (key.mode == 0 || key.n_text <= UM_TEXT_MAX);
  // fp32 tokens (FiCoCo-V): the same tiling with narrower column tiles, operands split into bf16 terms
  p->um_f32 = key.dtype == FICOCO_FP32 && key.dim % UKB == 0 && key.mode == 0;
  if (p->um_f32) p->umma = true;
  p->uf_small = false;
  if (key.rel) p->umma = p->um_f32 = false;           // C is read from the supplied matrix, not contracted
  int un_max = p->um_f32 ? UF_COLS : UN_MAX;          // accumulator columns per CTA
  int tile_rows_max = p->umma ? UM : CBM;             // source rows per correlate CTA
  if (key.rel) {
    // a warp of the relation correlate takes one discarded token at a time and is bound by the
    // latency of its gathers: small tiles put more rows in flight (as far as the work table goes)
    auto strips = [&](int t) {
      long long n = 0;
      for (int b = 0; b < B; ++b) n += (key.ntok[b] - cls - tail - key.keep[b] + t - 1) / t;
      return n;
    };
    tile_rows_max = 16;
    while (tile_rows_max < CBM && strips(tile_rows_max) + 2 * c->num_sms > c->cap_corr) tile_rows_max *= 2;
  }
  const int col_granule = p->umma ? 16 : CBN;
  int um_a_rows = 8, um_cols = 16;

  // first pass: sizes
  for (int b = 0; b < B; ++b) {
    ImgDesc& d = p->h_desc[b];
    const int ntok = key.ntok[b];
    const int np = ntok - cls - tail;
    if (np < 1) return FICOCO_ERR_INVALID_ARG;
    if (np > MAX_IMG_TOKENS) return FICOCO_ERR_UNSUPPORTED;
    const int keep = key.keep[b];
    if (keep < 0 || keep > np) return FICOCO_ERR_KEEP_RANGE;
    d.n_cls = cls; d.np = np; d.n_tgt = keep; d.n_src = np - keep; d.n_tail = tail;
    d.n_extra = (key.conv && np - keep > 0) ? 1 : 0;
    d.gh = key.gh[b]; d.gw = key.gw[b];
    if (key.mode == 0) {
      if (d.gh < 1 || d.gw < 1) return FICOCO_ERR_INVALID_ARG;
      if ((long long)d.gh * d.gw < np) return FICOCO_ERR_GRID;
      if ((long long)d.gh * d.gw > 20000) return FICOCO_ERR_UNSUPPORTED;
    }
    int L = 0;
    float frac = 0.f;
    if (key.max_targets != 0 && d.n_src > 0 && d.n_tgt > 0) {
      if (key.max_targets > 0) {
        L = key.max_targets < d.n_tgt ? key.max_targets : d.n_tgt;
      } else {
        const double q = key.eps * (double)(d.n_tgt - 1);
        const double lo = floor(q);
        L = d.n_tgt - (int)lo;
        frac = (float)(q - lo);
      }
      if (L > KCAP) return FICOCO_ERR_UNSUPPORTED;
    }
    d.list_len = L;
    d.frac = frac;
    d.avg = key.avg;
    if (L > p->max_list) p->max_list = L;
  }
  // ---- fused filter kernel: piece size and feasibility -------------------------------------
  const int esz = key.dtype == FICOCO_BF16 ? 2 : 4;
  const int f_nvec = key.dim / (16 / esz);
  p->f_vpl = (f_nvec + 31) / 32;
  p->fused = c->coop_ok && p->f_vpl <= 8 && !key.rel;
  int f_rc = 0, f_cap = 0;
  if (p->fused) {
    std::vector<int> nps(B);
    long long total = 0;
    for (int b = 0; b < B; ++b) total += nps[b] = p->h_desc[b].np;
    const PieceDeal best = best_deal(nps.data(), B, c->num_sms, c->cap_rows, F_MAXWON);
    f_rc = best.rc;
    f_cap = best.cap;
    // A deal that comes out uneven leaves SMs idle through both passes; from about 64 MB of tokens on three plain
    // kernels then make up for their launches and the second read.  Whole step, fused / unfused, both paths forced:
    //   rows of up to 1024 values, uneven and large: 1.00 to 1.20 (768, 1024 in bf16, 85 to 300 images of 256 to 2304
    //   tokens; 192 batches on the kernels before these: 1.065 in the mean of 30, even ones 1.003 of 94);
    //   1280 values, uneven and large: 0.97 to 1.07;
    //   six and seven vectors a lane in bf16 (1344 to 1792 values, 48 batches of one to 256 images): 0.88 to 0.99, for one
    //   image 1.01 to 1.05;
    //   eight (1800 to 2048 values, one to 256 images of 576 tokens, four of 2880), where a warp of the fused kernel held one
    //   row at a time and spilled: 1.00 to 1.16 from 1984 on; 0.955 to 1.00 at 1856 and 1920 from 18 000 tokens on and for
    //   large images, up to 1.09 below; 0.995 to 1.38 where the hidden size is no multiple of 64.  They have no fused kernel.
    const bool wide_bf16 = esz == 2 && p->f_vpl >= 6;
    const bool uneven = best.cost * 100 > (best.even + F_PIECE_ROWS) * 122LL && total * key.dim * esz > 64LL * 1024 * 1024;
    if (best.cost < 0 || (wide_bf16 ? p->f_vpl == 8 : uneven)) p->fused = false;
    // shared memory: ring stages of 16 rows (the selection works in them), the fold area, a score per row of a piece
    const size_t stage = (size_t)FROWS * key.dim * esz, fixed = (size_t)FFOLD * key.dim * 4 + (size_t)best.max_piece * 4 + 256;
    int ns = F_SMEM > fixed ? (int)((F_SMEM - fixed) / stage) : 0;
    if (ns > F_MAXSTAGE) ns = F_MAXSTAGE;
    size_t sel_need = 0;
    for (int b = 0; b < B; ++b) {
      const int np = p->h_desc[b].np, cells = key.mode == 0 ? p->h_desc[b].gh * p->h_desc[b].gw : 0;
      sel_need = std::max(sel_need, np <= SEL_SMALL_MAX ? select_small_bytes(np, cells) : select_work_bytes(np, cells));
    }
    if (ns < 2 || sel_need > (size_t)ns * stage) p->fused = false;
    p->f_nstage = ns;
    p->f_smem = (size_t)ns * stage + fixed;
  }
  // Unfused filter, rows of up to 256 vectors: chunks of at least 64 rows that make about three and a half waves of
  // two CTAs per SM, so that the last wave costs little and the folds at their ends do not either (256 x 577 tokens,
  // whole step: 64 rows 348 us, 144 rows 341, 576 rows in less than one wave 349).
  int u_rc = 0;
  if (!p->fused && p->f_vpl <= 8 && !key.rel) {
    auto count = [&](int rc) {
      long long n = 0;
      for (int b = 0; b < B; ++b) n += (p->h_desc[b].np + rc - 1) / rc;
      return n;
    };
    u_rc = 64;
    while (u_rc < 1024 && count(u_rc) > std::max(7 * c->num_sms, B)) u_rc += 8;
  }

  // ---- correlate tiling ---------------------------------------------------------------------
  int cols_max = p->umma ? un_max : INT_MAX;
  auto split_cols = [&](int n_tgt, int ns) { return split_columns(n_tgt, ns, cols_max, col_granule); };
  int want_split = 1;
  if (p->umma && !p->um_f32) {
    std::vector<int> n_src(B), n_tgt(B), len(B);
    for (int b = 0; b < B; ++b) {
      n_src[b] = p->h_desc[b].n_src;
      n_tgt[b] = p->h_desc[b].n_tgt;
      len[b] = p->h_desc[b].list_len;
    }
    const Tiling t = best_tiling(distinct_shapes(n_src.data(), n_tgt.data(), len.data(), B), key.dim, tail, c->num_sms,
                                 c->cap_corr, c->cap_part);
    tile_rows_max = t.rows;
    want_split = t.splits;
  } else {
    // As many splits as give every SM two CTAs, no more than eight with fp32 tiles; a grid of fp32 tiles of
    // 32 x 32 that needs no second CTA on any SM is taken instead (47.0 -> 43.0 us for 64 x 512 entries; twice as many
    // entries as fit: the larger tiles are ahead).
    long long strips = 0;
    for (int b = 0; b < B; ++b)
      if (p->h_desc[b].list_len > 0) strips += (p->h_desc[b].n_src + tile_rows_max - 1) / tile_rows_max;
    if (strips > 0) want_split = (int)std::min(std::max(2LL * c->num_sms / strips, 1LL), p->um_f32 ? 8LL : (long long)NSPLIT_MAX);
    long long n_ctas = 0, entries = 0;
    for (int b = 0; b < B; ++b) {
      const ImgDesc& d = p->h_desc[b];
      if (d.list_len == 0) continue;
      const int ns = (d.n_tgt + UF_SMALL - 1) / UF_SMALL;
      n_ctas += (long long)((d.n_src + UF_SMALL - 1) / UF_SMALL) * ns;
      entries += (long long)d.n_src * ns * d.list_len;
    }
    if (p->um_f32 && n_ctas <= c->num_sms && n_ctas <= c->cap_corr && entries <= c->cap_part) {
      p->uf_small = true;
      tile_rows_max = cols_max = um_a_rows = um_cols = UF_SMALL;     // (full tiles)
      want_split = 1;
    }
  }

  // Output rows per merge CTA: the fewest that make one wave of two CTAs per SM, or else as many as the shared
  // memory for their input rows takes, evened out over the waves.
  int out_rows_cta = 1;
  {
    const size_t row_b = (size_t)key.dim * (key.dtype == FICOCO_BF16 ? 2 : 4);
    const int most = (int)std::min<size_t>(MROWS, std::max<size_t>(1, MSTAGE_BYTES / row_b));
    const long long slots = 2LL * c->num_sms;
    auto n_out_ctas = [&](int r) {
      long long n = 0;
      for (int b = 0; b < B; ++b) n += (cls + key.keep[b] + p->h_desc[b].n_extra + tail + r - 1) / r;
      return n;
    };
    const long long waves = (n_out_ctas(most) + slots - 1) / slots;
    while (out_rows_cta < most && (n_out_ctas(out_rows_cta) > waves * slots || n_out_ctas(out_rows_cta) > c->cap_out)) ++out_rows_cta;
    p->m_smem = out_rows_cta * row_b;
  }
  for (int b = 0; b < B; ++b) {
    ImgDesc& d = p->h_desc[b];
    d.row0 = (int)row0; d.patch0 = (int)patch0; d.out_row0 = (int)out0;
    d.src0 = (int)src0; d.tgt0 = (int)tgt0; d.ent0 = (int)ent0; d.part0 = (int)part0;
    d.attn0 = 0;  // set by the caller-specific code below
    d.rel0 = rel0;
    rel0 += (long long)d.np * d.np;
    // row chunks (fused filter: equal pieces of at most f_rc rows)
    int rc = (d.np + MAX_CHUNKS - 1) / MAX_CHUNKS;
    rc = (rc + 7) / 8 * 8;
    // unfused filter: chunks of about 256 KB of token rows (at most 64 rows; 32 rows of 4096 bf16), so
    // that wide rows still give every SM several CTAs
    int rc_floor = (int)(262144 / ((size_t)key.dim * (key.dtype == FICOCO_BF16 ? 2 : 4))) / 8 * 8;
    rc_floor = rc_floor < 8 ? 8 : (rc_floor > 64 ? 64 : rc_floor);
    if (rc < rc_floor) rc = rc_floor;
    if (u_rc > 0 && d.np > 0) rc = std::max(rc, piece_rows(d.np, u_rc));
    if (p->fused) {
      if (d.np > 0) rc = piece_rows(d.np, f_rc);
    }
    d.n_chunks = (d.np + rc - 1) / rc;
    d.chunk0 = (int)chunk0;
    for (int k = 0; k < d.n_chunks; ++k) {
      WorkItem w; w.img = b; w.r0 = k * rc; w.nrows = (d.np - w.r0 < rc) ? d.np - w.r0 : rc; w.aux = k;
      rows.push_back(w);
    }
    if (rc > p->max_rc) p->max_rc = rc;
    // correlate
    d.nsplit = 1; d.cols_per_split = d.n_tgt > 0 ? d.n_tgt : 1;
    if (d.list_len == 0 && d.n_src > 0) p->need_finalize = true;
    if (d.list_len > 0) {
      const int cps = split_cols(d.n_tgt, want_split), ns = (d.n_tgt + cps - 1) / cps;
      d.nsplit = ns; d.cols_per_split = cps;
      // source tiles of equal size (rounded to 8 rows)
      const int trows = tile_height(d.n_src, tile_rows_max);
      if (trows > um_a_rows) um_a_rows = trows;
      if (cps > um_cols) um_cols = cps;
      for (int s0 = 0; s0 < d.n_src; s0 += trows)
        for (int sp = 0; sp < ns; ++sp) {
          WorkItem w; w.img = b; w.r0 = s0; w.nrows = (d.n_src - s0 < trows) ? d.n_src - s0 : trows; w.aux = sp;
          corr.push_back(w);
        }
      part0 += (long long)d.n_src * ns * d.list_len;
      ent0 += (long long)d.n_src * d.list_len;
    }
    // output rows
    const int orows = d.n_cls + d.n_tgt + d.n_extra + d.n_tail;
    const int n_cta = (orows + out_rows_cta - 1) / out_rows_cta;
    for (int k = 0; k < n_cta; ++k) {            // rows k, k + n_cta, k + 2 n_cta, ...
      WorkItem w; w.img = b; w.r0 = k; w.nrows = (orows - k + n_cta - 1) / n_cta; w.aux = n_cta;
      outw.push_back(w);
    }
    row0 += key.ntok[b]; patch0 += d.np; out0 += orows; src0 += d.n_src; tgt0 += d.n_tgt;
    chunk0 += d.n_chunks;
    if (d.np > p->max_np) p->max_np = d.np;
    if (d.n_tgt > p->max_tgt) p->max_tgt = d.n_tgt;
    if (d.n_src > p->max_src) p->max_src = d.n_src;
    if (key.mode == 0 && d.gh * d.gw > p->max_nwin_cells) p->max_nwin_cells = d.gh * d.gw;
  }
  if (row0 > c->max_tokens || B > c->max_batch || key.dim > c->max_dim || tail > c->max_text)
    return FICOCO_ERR_WORKSPACE;
  // ---- fused filter kernel: pieces -> CTAs, shared memory -----------------------------------
  std::vector<int> cta_first;
  if (p->fused) {
    cta_first.push_back(0);
    int acc = 0, items = 0;                            // (the same deal)
    for (size_t i = 0; i < rows.size(); ++i) {
      if (items > 0 && (acc + rows[i].nrows > f_cap || items >= F_MAXWON)) {
        cta_first.push_back((int)i);
        acc = items = 0;
      }
      acc += rows[i].nrows;
      ++items;
    }
    cta_first.push_back((int)rows.size());
    p->f_grid = (int)cta_first.size() - 1;
  }
  if (!p->fused && rows.size() > (size_t)MAX_CHUNKS * B) return FICOCO_ERR_UNSUPPORTED;
  if ((int)rows.size() > c->cap_rows || (int)corr.size() > c->cap_corr || (int)outw.size() > c->cap_out ||
      part0 > c->cap_part)
    return FICOCO_ERR_WORKSPACE;
  p->tot_patch = (int)patch0; p->tot_src = (int)src0; p->tot_tgt = (int)tgt0; p->tot_out_rows = (int)out0;
  p->n_rows = (int)rows.size(); p->n_corr = (int)corr.size(); p->n_out = (int)outw.size();
  if (p->um_f32) {
    p->um_a_bytes = um_a_rows * 128;
    p->um_b_bytes = (um_cols + 15) / 16 * 16 * 128;
    p->um_tmem_cols = 32;
    while (p->um_tmem_cols < 6 * (p->um_b_bytes / 128)) p->um_tmem_cols *= 2;   // six partial products per entry
    p->um_smem = uf_smem(p->uf_small, p->um_a_bytes, p->um_b_bytes);
    if (p->uf_small) {
      p->uf_stg_off = (int)(p->um_smem - 1024);
      p->um_smem += UF_SLOTS * UF_SLOT;
    }
    if (um_a_rows > UM || um_cols > UF_COLS || p->um_smem > 220 * 1024) return FICOCO_ERR_UNSUPPORTED;
  } else if (p->umma) {
    const UmRing r = um_ring(um_a_rows, um_cols, (long long)corr.size(), key.dim, tail, list_capacity(p->max_list), c->num_sms);
    if (r.nstage == 0) return FICOCO_ERR_UNSUPPORTED;
    p->um_a_bytes = um_a_rows * 128;
    p->um_tmem_cols = 32;
    while (p->um_tmem_cols < um_cols) p->um_tmem_cols *= 2;
    p->um_nstage = r.nstage;
    p->um_ksub = r.ksub;
    p->um_stage_bytes = r.stage_bytes;
    p->um_text_off = r.text_off;
    p->um_text_late = r.text_late;
    p->um_smem = r.smem;
  }

  char* slot_dev = c->plan_slots + (size_t)slot * c->slot_bytes;
  p->d_desc = (ImgDesc*)slot_dev;
  const PlanTables at = plan_tables(B * sizeof(ImgDesc), sizeof(WorkItem), rows.size(), corr.size(), outw.size(),
                                    cta_first.size(), B + 1);
  if (at.bytes > c->slot_bytes) return FICOCO_ERR_WORKSPACE;
  p->table_bytes = at.bytes;
  p->d_rows = (WorkItem*)(slot_dev + at.rows);
  p->d_corr = (WorkItem*)(slot_dev + at.corr);
  p->d_out = (WorkItem*)(slot_dev + at.out);
  p->d_ctafirst = (int*)(slot_dev + at.cta_first);
  p->d_out_cu = (int*)(slot_dev + at.out_cu);
  {
    int* ocu = (int*)(c->h_stage + at.out_cu);
    for (int b = 0; b < B; ++b) ocu[b] = p->h_desc[b].out_row0;
    ocu[B] = p->tot_out_rows;
  }
  p->key = key;
  auto fill = [&](size_t to, const void* from, size_t bytes) { if (bytes) memcpy(c->h_stage + to, from, bytes); };
  fill(at.cta_first, cta_first.data(), cta_first.size() * sizeof(int));
  fill(at.rows, rows.data(), rows.size() * sizeof(WorkItem));
  fill(at.corr, corr.data(), corr.size() * sizeof(WorkItem));
  fill(at.out, outw.data(), outw.size() * sizeof(WorkItem));
  return FICOCO_OK;
}

// Finds or builds the plan for `key`.  heads_or_text scales the attention block offsets:
// V: image b's block starts at H * patch0 floats; L: at M * b * N floats of the head-mean
// block t.
int get_plan(ficoco_ctx* c, const PlanKey& key, long long attn_rows, cudaStream_t stream, Plan** out) {
  ++c->clock;
  for (int i = 0; i < N_PLANS; ++i)
    if (c->plans[i].valid && c->plans[i].key == key) {
      // attention offsets depend on the head count, which is not part of the key
      bool same = true;
      for (int b = 0; b < key.batch && same; ++b)
        same = c->plans[i].h_desc[b].attn0 == attn_rows * c->plans[i].h_desc[b].patch0;
      if (same) {
        c->plans[i].stamp = c->clock;
        *out = &c->plans[i];
        return FICOCO_OK;
      }
      c->plans[i].valid = false;
    }
  cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
  CUDA_TRY(c, cudaStreamIsCapturing(stream, &cs));
  if (cs != cudaStreamCaptureStatusNone) return FICOCO_ERR_CAPTURE;
  int slot = 0;
  for (int i = 0; i < N_PLANS; ++i) {
    if (!c->plans[i].valid) { slot = i; break; }
    if (c->plans[i].stamp < c->plans[slot].stamp) slot = i;
  }
  // the staging buffer and the slot may still be read by work enqueued earlier
  CUDA_TRY(c, cudaStreamSynchronize(stream));
  Plan* p = &c->plans[slot];
  p->valid = false;
  int rc = build_plan(c, p, key, slot);
  if (rc != FICOCO_OK) return rc;
  for (int b = 0; b < key.batch; ++b) p->h_desc[b].attn0 = attn_rows * p->h_desc[b].patch0;
  memcpy(c->h_stage, p->h_desc.data(), key.batch * sizeof(ImgDesc));
  CUDA_TRY(c, cudaMemcpyAsync(c->plan_slots + (size_t)slot * c->slot_bytes, c->h_stage, p->table_bytes,
                              cudaMemcpyHostToDevice, stream));
  CUDA_TRY(c, cudaStreamSynchronize(stream));
  p->valid = true;
  p->stamp = c->clock;
  *out = p;
  return FICOCO_OK;
}

// Launch with programmatic stream serialization: the grid may be staged while the kernel before
// it in the stream is still running; the kernel itself waits (grid_dep_wait) before it reads
// anything that kernel wrote.  Takes a launch's set-up off the stream (about 1.5 us per kernel).
template <class... KArgs, class... Args>
cudaError_t launch_dependent(void (*kernel)(KArgs...), dim3 grid, int block, size_t smem, cudaStream_t st,
                             Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, KArgs(args)...);
}

template <class T, int VPL>
cudaError_t launch_filter_fused(ficoco_ctx* c, const Plan* p, const T* tok, int D, const float* attn,
                                int attn_rows, float cA, const int* pos, int window, float coef, int penalty,
                                int* kept_idx, int* pos_out, float* scores_out, int overlap_prev,
                                cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(p->f_grid);
  cfg.blockDim = dim3(F_NCONS);
  cfg.dynamicSmemBytes = p->f_smem;
  cfg.stream = st;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeCooperative;
  at[0].val.cooperative = 1;
  at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = (c->coop_pdl_ok && overlap_prev) ? 2 : 1;   // 1: inputs independent of the step before; 2: fed by it
  c->last_parity = (int)(c->epoch++ & 1);
  const size_t set = 3 * (size_t)c->max_batch;
  return cudaLaunchKernelEx(&cfg, k_filter_fused<T, VPL>, tok, D, (const ImgDesc*)p->d_desc,
                            (const WorkItem*)p->d_rows, (const int*)p->d_ctafirst, c->rn, c->partial, attn,
                            attn_rows, cA, c->s_raw, c->img_cnt + c->last_parity * set, p->key.batch, pos, window, coef,
                            penalty, c->s_pen, scores_out, c->S_idx, c->T_idx, kept_idx, pos_out, c->status,
                            p->f_nstage, c->img_cnt + (1 - c->last_parity) * set, (int)set, c->wait_ns,
                            c->dbg_extra_arrivals, (c->coop_pdl_ok && overlap_prev == 2) ? 1 : 0);
}

template <class T, int VPL>
void launch_colsum_fused(ficoco_ctx* c, const Plan* p, const T* tok, int D, cudaStream_t st) {
  constexpr int E = VecTraits<T>::E;
  launch_dependent(k_colsum<T, VPL, true>, dim3(p->n_rows, 1), 256, 4 * VPL * 32 * E * sizeof(float), st,
      tok, D, p->d_desc, p->d_rows, c->rn, c->partial);
}

// Runs the whole reduce step for tokens of type T.  `attn` is the per-head CLS attention
// (V) or the head-mean text->vision block (L); `attn_rows` its number of rows per image.
template <class T>
int run_step(ficoco_ctx* c, const Plan* p, const T* tok, int D, const float* attn, int attn_rows,
             float cA, const int* pos, int window, float coef, int penalty, const float* tmean, int M,
             float gamma, T* out_tokens, int* kept_idx, int* pos_out, float* scores_out,
             cudaStream_t st, bool back_to_back, const float* rel = nullptr, const float* t2v = nullptr,
             int t2v_heads = 0) {
  constexpr int E = VecTraits<T>::E;
  const int nvec = D / E;
  const int vpl = (nvec + 31) / 32;
  const size_t in_rows = (size_t)p->tot_patch + (size_t)p->key.batch * (p->key.has_cls + (p->key.mode == 1 ? p->key.n_text : 0));
  const Span in_spans[3] = {span_of(tok, in_rows * D * sizeof(T)),
                            span_of(attn, (size_t)attn_rows * p->tot_patch * sizeof(float)),
                            span_of(pos, (size_t)p->tot_patch * sizeof(int))};
  const Span out_spans[N_SPANS] = {span_of(out_tokens, (size_t)p->tot_out_rows * D * sizeof(T)),
                                   span_of(kept_idx, (size_t)p->tot_out_rows * sizeof(int)),
                                   span_of(pos_out, (size_t)p->tot_tgt * sizeof(int)),
                                   span_of(scores_out, (size_t)p->tot_patch * sizeof(float))};
  const Span rel_span = span_of(rel, rel ? (size_t)p->h_desc.back().rel0 * 4 + (size_t)p->h_desc.back().np * p->h_desc.back().np * 4 : 0);
  for (int o = 0; o < N_SPANS; ++o) {
    for (int i = 0; i < 3; ++i)
      if (spans_overlap(out_spans[o], in_spans[i])) return FICOCO_ERR_INVALID_ARG;
    if (spans_overlap(out_spans[o], rel_span)) return FICOCO_ERR_INVALID_ARG;
  }
  // How the filter grid starts.  1: it may read its inputs under the tail of the step before (only when the caller
  // vouches for what sits in front of this step); 2: launched early, so that its CTAs are in place and set up, but
  // reads only once whatever is in front of it on the stream is complete.
  const int overlap_prev = back_to_back && inputs_clear_of_last_outputs(c->device, st, in_spans, 3) ? 1 : 2;
  record_last_outputs(c->device, st, out_spans, N_SPANS);
  const bool wide = !p->fused && !rel && vpl > 8 && nvec <= 1024;   // rows of 257 .. 1024 16-byte vectors: CTA-wide rows
  // FiCoCo-L: head mean of the text->vision attention, in the grid of the column sums where rows are CTA-wide
  const int mn = t2v ? M * p->max_np : 0;
  const int head_ctas = p->key.batch * head_mean_parts(mn, head_mean_values(t2v, c->tmean, mn), wide ? 256 : HM_THREADS);
  if (t2v && !wide) {
    prof_tick(c, st, "head_mean");
    launch_dependent(k_head_mean, dim3(head_ctas), HM_THREADS, 0, st, t2v, t2v_heads, mn, c->tmean);
    c->launches += 1;
  }
  if (p->fused) {
    prof_tick(c, st, "filter_fused");
    cudaError_t fe;
#define FICOCO_FUSED_GO(V) fe = launch_filter_fused<T, V>(c, p, tok, D, attn, attn_rows, cA, pos, window, coef, \
                                                          penalty, kept_idx, pos_out, scores_out, overlap_prev, st)
    if (vpl <= 1) FICOCO_FUSED_GO(1);
    else if (vpl <= 2) FICOCO_FUSED_GO(2);
    else if (vpl <= 4) FICOCO_FUSED_GO(4);
    else if (vpl <= 5) FICOCO_FUSED_GO(5);
    else if (vpl <= 6) FICOCO_FUSED_GO(6);
    else if (vpl <= 7) FICOCO_FUSED_GO(7);
    else if constexpr (sizeof(T) == 4) FICOCO_FUSED_GO(8);
    else return FICOCO_ERR_UNSUPPORTED;                // (never planned)
#undef FICOCO_FUSED_GO
    if (fe != cudaSuccess) { c->last_cuda = (int)fe; return FICOCO_ERR_CUDA; }
    c->launches += 1;
  } else {
  if (rel) {
    prof_tick(c, st, "score_relation");
    launch_dependent(k_score_rel, dim3(p->n_rows), 256, (size_t)p->max_rc * sizeof(float), st,
        rel, p->d_desc, p->d_rows, attn, attn_rows, cA, p->key.rel == 2 ? 1 : 0, c->s_raw);
    c->launches += 1;
  } else {
  prof_tick(c, st, (vpl <= 8 || wide) ? "colsum" : "rownorm");
  if (vpl <= 8) {
    if (vpl <= 1) launch_colsum_fused<T, 1>(c, p, tok, D, st);
    else if (vpl <= 2) launch_colsum_fused<T, 2>(c, p, tok, D, st);
    else if (vpl <= 4) launch_colsum_fused<T, 4>(c, p, tok, D, st);
    else if (vpl <= 5) launch_colsum_fused<T, 5>(c, p, tok, D, st);
    else launch_colsum_fused<T, 8>(c, p, tok, D, st);
    c->launches += 1;
  } else if (wide) {
#define FICOCO_WIDE_GO(NV, RB)                                                                              \
  launch_dependent(k_colsum_wide<T, NV, RB>, dim3(p->n_rows + head_ctas), 256, 0, st, tok, D, p->d_desc, p->d_rows, \
                   c->rn, c->partial, p->n_rows, t2v, t2v_heads, mn, c->tmean)
    if (nvec <= 512) FICOCO_WIDE_GO(2, 8);
    else FICOCO_WIDE_GO(4, 4);
#undef FICOCO_WIDE_GO
    c->launches += 1;
  } else {
    launch_dependent(k_rownorm<T>, dim3(p->n_rows), 256, 0, st,
      tok, D, p->d_desc, p->d_rows, c->rn);
    prof_tick(c, st, "colsum");
    const int slabs = (nvec + 255) / 256;
    launch_dependent(k_colsum<T, 8, false>, dim3(p->n_rows, slabs), 256, 4 * 8 * 32 * E * sizeof(float), st,
        tok, D, p->d_desc, p->d_rows, c->rn, c->partial);
    c->launches += 2;
  }
  prof_tick(c, st, "score");
  launch_dependent(k_msum, dim3(p->key.batch, (D + 255) / 256), 256, 0, st,
      D, p->d_desc, c->partial, c->msum);
  if (wide && nvec <= 512)
    launch_dependent(k_score_wide<T, 2, 8>, dim3(p->n_rows), 256, (size_t)9 * p->max_rc * sizeof(float), st,
        tok, D, p->d_desc, p->d_rows, c->rn, c->msum, attn, attn_rows, cA, c->s_raw);
  else if (wide)
    launch_dependent(k_score_wide<T, 4, 4>, dim3(p->n_rows), 256, (size_t)9 * p->max_rc * sizeof(float), st,
        tok, D, p->d_desc, p->d_rows, c->rn, c->msum, attn, attn_rows, cA, c->s_raw);
#define FICOCO_SCORE_GO(V) \
  launch_dependent(k_score_rows<T, V>, dim3(p->n_rows), 256, (size_t)9 * p->max_rc * sizeof(float), st, \
      tok, D, p->d_desc, p->d_rows, c->rn, c->msum, attn, attn_rows, cA, c->s_raw)
  else if (vpl <= 1) FICOCO_SCORE_GO(1);
  else if (vpl <= 2) FICOCO_SCORE_GO(2);
  else if (vpl <= 4) FICOCO_SCORE_GO(4);
  else if (vpl <= 5) FICOCO_SCORE_GO(5);
  else if (vpl <= 8) FICOCO_SCORE_GO(8);
#undef FICOCO_SCORE_GO
  else
    launch_dependent(k_score<T>, dim3(p->n_rows), 256, (size_t)(D + 9 * p->max_rc) * sizeof(float), st,
        tok, D, p->d_desc, p->d_rows, c->rn, c->msum, attn, attn_rows, cA, c->s_raw);
  c->launches += 2;
  }
  const int sel_cells = penalty ? p->max_nwin_cells : 0;
  const size_t small_smem = select_small_bytes(std::min(p->max_np, SEL_SMALL_MAX), sel_cells) + 16;
  const size_t sel_smem = p->max_np <= SEL_SMALL_MAX ? small_smem : std::max(small_smem, select_work_bytes(p->max_np, sel_cells) + 16);
  prof_tick(c, st, "select");
  launch_dependent(p->max_np <= SEL_SMALL_MAX ? k_select<true> : k_select<false>, dim3(p->key.batch), SEL_THREADS, sel_smem,
                   st, p->d_desc, c->s_raw, pos, window, coef, penalty, c->s_pen, scores_out, c->S_idx, c->T_idx, kept_idx,
                   pos_out, c->status);
  c->launches += 1;
  }
  if (p->n_corr > 0) {
    if (rel) {
      prof_tick(c, st, "correlate_relation");
      int rel_cols = 1;
      for (const ImgDesc& d : p->h_desc)
        if (d.list_len > 0 && d.cols_per_split > rel_cols) rel_cols = d.cols_per_split;
#define FICOCO_REL_GO(LC)                                                                              \
  launch_dependent(k_correlate_rel<LC>, dim3(p->n_corr), 256, (size_t)rel_cols * sizeof(int), st,       \
                   rel, p->d_desc, p->d_corr, c->S_idx, c->T_idx, c->part_val,                          \
                                                 c->part_idx, c->tile_cnt, c->corr_cnt, c->tau, c->e_tgt,    \
                                                 c->e_w, c->e_c, c->status)
      if (p->max_list <= 2) FICOCO_REL_GO(2);
      else if (p->max_list <= 4) FICOCO_REL_GO(4);
      else FICOCO_REL_GO(16);
#undef FICOCO_REL_GO
    } else if (p->um_f32 && sizeof(T) == 4) {
      prof_tick(c, st, "correlate_umma_f32");
      const float* tk = reinterpret_cast<const float*>(tok);
#define FICOCO_UF32_LAUNCH(LC)                                                                         \
  launch_dependent(p->uf_small ? k_correlate_umma_f32<LC, true> : k_correlate_umma_f32<LC, false>, dim3(p->n_corr), UTHREADS, p->um_smem, st, tk, D,                                                                  \
      (const ImgDesc*)p->d_desc, (const WorkItem*)p->d_corr, (const float*)c->rn,                       \
      (const int*)c->S_idx, (const int*)c->T_idx, c->part_val, c->part_idx, c->status,                 \
      p->um_a_bytes, p->um_b_bytes, p->uf_stg_off, p->um_tmem_cols, c->tile_cnt, c->corr_cnt, c->tau, c->e_tgt, \
      c->e_w, c->e_c, c->wait_ns)
      if (p->max_list <= 2) FICOCO_UF32_LAUNCH(2);
      else if (p->max_list <= 4) FICOCO_UF32_LAUNCH(4);
      else FICOCO_UF32_LAUNCH(16);
#undef FICOCO_UF32_LAUNCH
    } else if (p->umma && sizeof(T) == 2) {
      prof_tick(c, st, "correlate_umma");
      const __nv_bfloat16* tk = reinterpret_cast<const __nv_bfloat16*>(tok);
#define FICOCO_UMMA_LAUNCH(LC, KS)                                                                      \
  launch_dependent(k_correlate_umma<LC, KS>, dim3(p->n_corr), UTHREADS, p->um_smem, st, tk, D,                   \
      (const ImgDesc*)p->d_desc, (const WorkItem*)p->d_corr, (const float*)c->rn,                       \
      (const int*)c->S_idx, (const int*)c->T_idx, c->part_val, c->part_idx, c->status, p->um_nstage,    \
      p->um_stage_bytes, p->um_a_bytes, p->um_tmem_cols, c->tile_cnt, c->corr_cnt, c->tau, c->e_tgt, \
      c->e_w, c->e_c, tmean, M, p->max_np, gamma, p->um_text_off, p->um_text_late ? 1 : 0, c->wait_ns)
#define FICOCO_UMMA_STAGES(LC)                                                                         \
  do {                                                                                                 \
    if (p->um_ksub == 4) FICOCO_UMMA_LAUNCH(LC, 4);                                                     \
    else if (p->um_ksub == 2) FICOCO_UMMA_LAUNCH(LC, 2);                                                     \
    else FICOCO_UMMA_LAUNCH(LC, 1);                                                                     \
  } while (0)
      if (p->max_list <= 2) FICOCO_UMMA_STAGES(2);
      else if (p->max_list <= 4) FICOCO_UMMA_STAGES(4);
      else FICOCO_UMMA_STAGES(16);
#undef FICOCO_UMMA_STAGES
#undef FICOCO_UMMA_LAUNCH
    } else {
      prof_tick(c, st, "correlate_simt");
      // The CTAs are placed while the filter grid still holds most SMs, two to each of the others.  A grid that needs no
      // second CTA on any SM asks for shared memory that keeps a second one off (4 x 576 tokens of 1000, 100 CTAs: whole step
      // 116 -> 89 us; 44 FiCoCo-L sequences of 99 + 34 fp32 tokens of 1024, 88 CTAs: 119 -> 90).
      launch_dependent(k_correlate_simt<T>, dim3(p->n_corr), 256, p->n_corr <= c->num_sms ? SIMT_ALONE_BYTES : 0, st,
      tok, D, p->d_desc, p->d_corr, c->rn, c->S_idx,
                                                     c->T_idx, tmean, M, gamma, c->part_val, c->part_idx,
                                                     c->tile_cnt, c->corr_cnt, c->tau,
                                                     c->e_tgt, c->e_w, c->e_c, c->status);
    }
    c->launches += 1;
  }
  if (p->max_src > 0 && p->need_finalize) {
    prof_tick(c, st, "finalize");
    launch_dependent(k_finalize_src, dim3(p->key.batch, (p->max_src + 255) / 256), 256, 0, st,
        p->d_desc, c->corr_cnt, c->tau);
    c->launches += 1;
  }
  prof_tick(c, st, "merge_compact");
  launch_dependent(k_merge_rows<T>, dim3(p->n_out), MTHREADS, p->m_smem, st, tok, D, (const ImgDesc*)p->d_desc,
                   (const WorkItem*)p->d_out, (const int*)c->S_idx, (const int*)c->T_idx,
                   (const int*)c->e_tgt, (const float*)c->e_w, out_tokens, c->status,
                   p->fused ? c->img_cnt + (size_t)c->last_parity * 3 * c->max_batch : (int*)nullptr,
                   p->fused ? 3 * c->max_batch : 0, c->wait_ns);
  c->launches += 1;
  if (p->key.conv) {
    prof_tick(c, st, "convergent_token");
    launch_dependent(k_convergent_token<T>, dim3(p->key.batch), 256, 0, st,
      tok, D, p->d_desc, c->S_idx, out_tokens, c->status);
    c->launches += 1;
  }
  prof_tick(c, st, nullptr);
  if (c->prof_used > 60000) prof_flush(c);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) { c->last_cuda = (int)e; return FICOCO_ERR_CUDA; }
  return FICOCO_OK;
}

int check_common(const ficoco_params* prm, int dtype, int batch, int dim, int heads, const void* tokens,
                 const void* out_tokens) {
  if (!prm || !tokens || !out_tokens) return FICOCO_ERR_INVALID_ARG;
  if (batch < 1 || dim < 1 || heads < 1) return FICOCO_ERR_INVALID_ARG;
  if (dtype != FICOCO_FP32 && dtype != FICOCO_BF16) return FICOCO_ERR_UNSUPPORTED;
  const int e = dtype == FICOCO_BF16 ? 8 : 4;
  if (dim % e != 0) return FICOCO_ERR_UNSUPPORTED;
  if (((uintptr_t)tokens & 15) || ((uintptr_t)out_tokens & 15)) return FICOCO_ERR_INVALID_ARG;
  if (!(prm->eps >= 0.0 && prm->eps <= 1.0) || prm->window < 1) return FICOCO_ERR_INVALID_ARG;
  return FICOCO_OK;
}

}  // namespace

namespace {
int v_reduce_impl(ficoco_ctx* c, const ficoco_v_args* a, const ficoco_params* prm, void* cuda_stream,
                  const float* rel, int rel_mode, bool plan_only = false) {
  if (!c || !a) return FICOCO_ERR_INVALID_ARG;
  // planning needs the shapes only: stand-ins for the data pointers pass the checks
  static const long long dummy[2] = {0, 0};
  int rc = check_common(prm, a->dtype, a->batch, a->dim, a->heads, plan_only ? (const void*)dummy : a->tokens,
                        plan_only ? (const void*)dummy : (const void*)a->out_tokens);
  if (rc) return rc;
  if (!a->grid_h || !a->grid_w || !a->keep) return FICOCO_ERR_INVALID_ARG;
  if (!plan_only && (!a->attn || !a->kept_idx)) return FICOCO_ERR_INVALID_ARG;
  if ((a->n_grid != 1 && a->n_grid != a->batch) || (a->n_keep != 1 && a->n_keep != a->batch))
    return FICOCO_ERR_INVALID_ARG;
  if (!a->seqlens && a->n_tokens < 1) return FICOCO_ERR_INVALID_ARG;
  if (a->batch > c->max_batch) return FICOCO_ERR_WORKSPACE;
  cudaStream_t st = (cudaStream_t)cuda_stream;
  CUDA_TRY(c, cudaSetDevice(c->device));

  PlanKey key;
  key.mode = 0; key.dtype = a->dtype; key.batch = a->batch; key.dim = a->dim; key.n_text = 0;
  key.has_cls = (prm->flags & FICOCO_HAS_CLS) ? 1 : 0;
  key.max_targets = prm->max_targets < 0 ? -1 : prm->max_targets;
  key.avg = (prm->flags & FICOCO_AVERAGE_COMPRESSION) ? 1 : 0;
  key.conv = (prm->flags & FICOCO_CONVERGENT) ? 1 : 0;
  if (key.conv) key.max_targets = 0;               // nothing is merged into the preserved tokens
  key.rel = rel_mode;
  key.eps = prm->eps;
  key.ntok.resize(a->batch); key.keep.resize(a->batch); key.gh.resize(a->batch); key.gw.resize(a->batch);
  for (int b = 0; b < a->batch; ++b) {
    key.ntok[b] = a->seqlens ? a->seqlens[b] : a->n_tokens;
    key.keep[b] = a->keep[a->n_keep == 1 ? 0 : b];
    key.gh[b] = a->grid_h[a->n_grid == 1 ? 0 : b];
    key.gw[b] = a->grid_w[a->n_grid == 1 ? 0 : b];
  }
  Plan* p = nullptr;
  rc = get_plan(c, key, a->heads, st, &p);
  if (rc) return rc;
  if (plan_only) return FICOCO_OK;
  c->last_plan = p;
  c->launches = 0;
  if (a->out_cu_seqlens)       // prefix of the output rows per image, from the plan's device copy
    CUDA_TRY(c, cudaMemcpyAsync(a->out_cu_seqlens, p->d_out_cu, (size_t)(a->batch + 1) * sizeof(int),
                                cudaMemcpyDeviceToDevice, st));
  const int penalty = (prm->flags & FICOCO_LOCAL_PENALTY) ? 1 : 0;
  const bool b2b = (prm->flags & FICOCO_BACK_TO_BACK) != 0;
  if (a->dtype == FICOCO_BF16)
    return run_step<__nv_bfloat16>(c, p, (const __nv_bfloat16*)a->tokens, a->dim, a->attn, a->heads,
                                   (float)prm->lambda_, a->pos, prm->window, (float)prm->penalty_coef,
                                   penalty, nullptr, 0, 1.0f, (__nv_bfloat16*)a->out_tokens, a->kept_idx,
                                   a->pos_out, a->scores_out, st, b2b, rel);
  return run_step<float>(c, p, (const float*)a->tokens, a->dim, a->attn, a->heads, (float)prm->lambda_,
                         a->pos, prm->window, (float)prm->penalty_coef, penalty, nullptr, 0, 1.0f,
                         (float*)a->out_tokens, a->kept_idx, a->pos_out, a->scores_out, st, b2b, rel);
}
}  // namespace

extern "C" int ficoco_v_reduce(ficoco_ctx* c, const ficoco_v_args* a, const ficoco_params* prm,
                               void* cuda_stream) {
  return v_reduce_impl(c, a, prm, cuda_stream, nullptr, 0);
}

extern "C" int ficoco_v_plan(ficoco_ctx* c, const ficoco_v_args* a, const ficoco_params* prm, void* cuda_stream) {
  return v_reduce_impl(c, a, prm, cuda_stream, nullptr, 0, true);
}

extern "C" int ficoco_v_reduce_relation(ficoco_ctx* c, const ficoco_v_args* a, const float* relation,
                                        int by_column, const ficoco_params* prm, void* cuda_stream) {
  if (!relation || ((uintptr_t)relation & 3)) return FICOCO_ERR_INVALID_ARG;
  return v_reduce_impl(c, a, prm, cuda_stream, relation, by_column ? 2 : 1);
}

// kept_idx of a schedule: the chain of the steps' kept indices, last step first.
// kidx[s] : [B, rows_s] row indices into step s's input rows (rows_s = c + keep[s]).
struct ComposeArgs {
  const int* kidx[8];
  int rows[8];
  int n_steps;
};
__global__ void k_compose_kept(ComposeArgs a, int batch, int* __restrict__ out) {
  grid_dep_wait();        // launched under the tail of the last step's merge grid
  grid_dep_launch();
  const int rows_last = a.rows[a.n_steps - 1];
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= batch * rows_last) return;
  const int b = i / rows_last;
  int idx = a.kidx[a.n_steps - 1][i];
  for (int s = a.n_steps - 2; s >= 0 && idx >= 0; --s) idx = a.kidx[s][(size_t)b * a.rows[s] + idx];
  out[i] = idx;
}

extern "C" int ficoco_v_reduce_schedule(ficoco_ctx* c, const ficoco_v_args* first, int n_steps, const int* keep,
                                        const float* const* attn, const ficoco_params* prm, void* cuda_stream) {
  if (!c || !first || !keep || !attn || !prm) return FICOCO_ERR_INVALID_ARG;
  if (n_steps < 1 || n_steps > 8) return FICOCO_ERR_INVALID_ARG;
  if (first->seqlens || (prm->flags & FICOCO_CONVERGENT)) return FICOCO_ERR_UNSUPPORTED;
  if (first->batch < 1 || first->n_tokens < 1 || first->dim < 1 || !first->out_tokens || !first->kept_idx)
    return FICOCO_ERR_INVALID_ARG;
  if (first->dtype != FICOCO_FP32 && first->dtype != FICOCO_BF16) return FICOCO_ERR_UNSUPPORTED;
  const int cls = (prm->flags & FICOCO_HAS_CLS) ? 1 : 0;
  const size_t es = first->dtype == FICOCO_BF16 ? 2 : 4;
  const int B = first->batch;
  int np = first->n_tokens - cls;
  for (int s = 0; s < n_steps; ++s) {
    if (!attn[s]) return FICOCO_ERR_INVALID_ARG;
    if (keep[s] < 0 || keep[s] > np) return FICOCO_ERR_KEEP_RANGE;
    np = keep[s];
  }
  if (n_steps == 1) {
    ficoco_v_args a = *first;
    a.attn = attn[0]; a.keep = keep; a.n_keep = 1; a.scores_out = nullptr;
    return ficoco_v_reduce(c, &a, prm, cuda_stream);
  }
  cudaStream_t st = (cudaStream_t)cuda_stream;
  CUDA_TRY(c, cudaSetDevice(c->device));
  // intermediates: tokens and positions ping-pong (A holds the outputs of even steps, B of odd
  // ones), kept indices of every step
  const size_t rows0 = (size_t)B * (cls + keep[0]), rows1 = (size_t)B * (cls + keep[1 < n_steps ? 1 : 0]);
  const size_t tokA = align_up(rows0 * first->dim * es, 256), tokB = align_up(rows1 * first->dim * es, 256);
  const size_t posA = align_up((size_t)B * keep[0] * 4 + 4, 256), posB = align_up((size_t)B * keep[1] * 4 + 4, 256);
  size_t kid_bytes = 0;
  for (int s = 0; s < n_steps; ++s) kid_bytes += align_up((size_t)B * (cls + keep[s]) * 4, 256);
  const size_t need = tokA + tokB + posA + posB + kid_bytes;
  if (need > c->sch_bytes) {
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    CUDA_TRY(c, cudaStreamIsCapturing(st, &cs));
    if (cs != cudaStreamCaptureStatusNone) return FICOCO_ERR_CAPTURE;
    CUDA_TRY(c, cudaDeviceSynchronize());
    if (c->sch_base) { cudaFree(c->sch_base); c->sch_base = nullptr; c->sch_bytes = 0; }
    CUDA_TRY(c, cudaMalloc((void**)&c->sch_base, need));
    c->sch_bytes = need;
  }
  char* tok_buf[2] = {c->sch_base, c->sch_base + tokA};
  int* pos_buf[2] = {(int*)(c->sch_base + tokA + tokB), (int*)(c->sch_base + tokA + tokB + posA)};
  ComposeArgs ca = {};
  ca.n_steps = n_steps;
  char* kp = c->sch_base + tokA + tokB + posA + posB;
  for (int s = 0; s < n_steps; ++s) {
    ca.kidx[s] = (const int*)kp;
    ca.rows[s] = cls + keep[s];
    kp += align_up((size_t)B * (cls + keep[s]) * 4, 256);
  }
  ficoco_params ps = *prm;
  int total_launches = 0;
  np = first->n_tokens - cls;
  for (int s = 0; s < n_steps; ++s) {
    const bool last = s + 1 == n_steps;
    ficoco_v_args a = *first;
    a.seqlens = nullptr;
    a.n_tokens = cls + np;
    a.attn = attn[s];
    a.keep = &keep[s];
    a.n_keep = 1;
    a.scores_out = nullptr;
    if (s > 0) {
      a.tokens = tok_buf[(s - 1) & 1];
      a.pos = pos_buf[(s - 1) & 1];
      ps.flags |= FICOCO_BACK_TO_BACK;              // the kernel in front of this step is the library's own
    }
    a.out_tokens = last ? first->out_tokens : (void*)tok_buf[s & 1];
    a.pos_out = last ? first->pos_out : pos_buf[s & 1];
    a.kept_idx = (int*)ca.kidx[s];
    const int rc = ficoco_v_reduce(c, &a, &ps, cuda_stream);
    if (rc) return rc;
    total_launches += c->launches;
    np = keep[s];
  }
  const int n_out = B * (cls + keep[n_steps - 1]);
  launch_dependent(k_compose_kept, dim3((n_out + 255) / 256), 256, 0, st, ca, B, first->kept_idx);
  c->launches = total_launches + 1;
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) { c->last_cuda = (int)e; return FICOCO_ERR_CUDA; }
  return FICOCO_OK;
}

extern "C" int ficoco_l_reduce(ficoco_ctx* c, const ficoco_l_args* a, const ficoco_params* prm,
                               void* cuda_stream) {
  if (!c || !a) return FICOCO_ERR_INVALID_ARG;
  int rc = check_common(prm, a->dtype, a->batch, a->dim, a->heads, a->tokens, a->out_tokens);
  if (rc) return rc;
  if (!a->attn_t2v || !a->keep || !a->kept_idx) return FICOCO_ERR_INVALID_ARG;
  if (a->n_vision < 1 || a->n_text < 1) return FICOCO_ERR_INVALID_ARG;
  if (a->n_keep != 1 && a->n_keep != a->batch) return FICOCO_ERR_INVALID_ARG;
  if (a->batch > c->max_batch || a->n_text > c->max_text) return FICOCO_ERR_WORKSPACE;
  cudaStream_t st = (cudaStream_t)cuda_stream;
  CUDA_TRY(c, cudaSetDevice(c->device));

  PlanKey key;
  key.mode = 1; key.dtype = a->dtype; key.batch = a->batch; key.dim = a->dim; key.n_text = a->n_text;
  key.has_cls = 0;
  key.max_targets = prm->max_targets < 0 ? -1 : prm->max_targets;
  key.avg = (prm->flags & FICOCO_AVERAGE_COMPRESSION) ? 1 : 0;
  key.conv = (prm->flags & FICOCO_CONVERGENT) ? 1 : 0;
  if (key.conv) key.max_targets = 0;
  key.eps = prm->eps;
  key.ntok.assign(a->batch, a->n_vision + a->n_text);
  key.keep.resize(a->batch);
  key.gh.assign(a->batch, 1); key.gw.assign(a->batch, a->n_vision);
  for (int b = 0; b < a->batch; ++b) key.keep[b] = a->keep[a->n_keep == 1 ? 0 : b];
  Plan* p = nullptr;
  rc = get_plan(c, key, a->n_text, st, &p);
  if (rc) return rc;
  c->last_plan = p;
  c->launches = 0;
  if (a->dtype == FICOCO_BF16)
    return run_step<__nv_bfloat16>(c, p, (const __nv_bfloat16*)a->tokens, a->dim, c->tmean, a->n_text,
                                   (float)prm->beta, nullptr, 1, 1.0f, 0, c->tmean, a->n_text,
                                   (float)prm->gamma, (__nv_bfloat16*)a->out_tokens, a->kept_idx, nullptr,
                                   a->scores_out, st, false, nullptr, a->attn_t2v, a->heads);
  return run_step<float>(c, p, (const float*)a->tokens, a->dim, c->tmean, a->n_text, (float)prm->beta,
                         nullptr, 1, 1.0f, 0, c->tmean, a->n_text, (float)prm->gamma,
                         (float*)a->out_tokens, a->kept_idx, nullptr, a->scores_out, st, false, nullptr, a->attn_t2v,
                         a->heads);
}

extern "C" int ficoco_status(ficoco_ctx* c, void* cuda_stream, int* device_status) {
  if (!c || !device_status) return FICOCO_ERR_INVALID_ARG;
  cudaStream_t st = (cudaStream_t)cuda_stream;
  CUDA_TRY(c, cudaSetDevice(c->device));
  unsigned v = 0;
  CUDA_TRY(c, cudaMemcpyAsync(&v, c->status, 4, cudaMemcpyDeviceToHost, st));
  CUDA_TRY(c, cudaMemsetAsync(c->status, 0, 4, st));
  CUDA_TRY(c, cudaStreamSynchronize(st));
  if (v & STATUS_TIMEOUT) {
    // a kernel gave up half-way: its per-image counters may be left non-zero
    CUDA_TRY(c, cudaMemsetAsync(c->img_cnt, 0, 6 * (size_t)c->max_batch * sizeof(int), st));
    CUDA_TRY(c, cudaMemsetAsync(c->tile_cnt, 0, (size_t)c->cap_corr * sizeof(int), st));
    CUDA_TRY(c, cudaStreamSynchronize(st));
  }
  *device_status = (int)v;
  return FICOCO_OK;
}

extern "C" int ficoco_inspect(ficoco_ctx* c, int what, void* host_dst, size_t bytes, size_t* bytes_avail) {
  if (!c || !c->last_plan) return FICOCO_ERR_INVALID_ARG;
  const Plan* p = c->last_plan;
  const void* src = nullptr;
  size_t n = 0;
  switch (what) {
    case FICOCO_INSPECT_RNORM: src = c->rn; n = (size_t)p->tot_patch * 4; break;
    case FICOCO_INSPECT_SCORE_RAW: src = c->s_raw; n = (size_t)p->tot_patch * 4; break;
    case FICOCO_INSPECT_SCORE: src = c->s_pen; n = (size_t)p->tot_patch * 4; break;
    case FICOCO_INSPECT_SRC_IDX: src = c->S_idx; n = (size_t)p->tot_src * 4; break;
    case FICOCO_INSPECT_TGT_IDX: src = c->T_idx; n = (size_t)p->tot_tgt * 4; break;
    case FICOCO_INSPECT_CORR_CNT: src = c->corr_cnt; n = (size_t)p->tot_src * 4; break;
    case FICOCO_INSPECT_CORR_TGT: src = c->e_tgt; n = (size_t)p->tot_src * KCAP * 4; break;
    case FICOCO_INSPECT_CORR_W: src = c->e_w; n = (size_t)p->tot_src * KCAP * 4; break;
    case FICOCO_INSPECT_CORR_C: src = c->e_c; n = (size_t)p->tot_src * KCAP * 4; break;
    case FICOCO_INSPECT_TAU: src = c->tau; n = (size_t)p->tot_src * 4; break;
    default: return FICOCO_ERR_INVALID_ARG;
  }
  if (bytes_avail) *bytes_avail = n;
  if (!host_dst || bytes == 0) return FICOCO_OK;
  CUDA_TRY(c, cudaSetDevice(c->device));
  CUDA_TRY(c, cudaDeviceSynchronize());
  if (what == FICOCO_INSPECT_CORR_TGT || what == FICOCO_INSPECT_CORR_W || what == FICOCO_INSPECT_CORR_C) {
    // the device keeps L slots per discarded token; widen to KCAP per token for the caller
    long long tot_ent = 0;
    for (const ImgDesc& d : p->h_desc) tot_ent += (long long)d.n_src * d.list_len;
    std::vector<int> compact((size_t)tot_ent + 1);
    if (tot_ent) CUDA_TRY(c, cudaMemcpy(compact.data(), src, (size_t)tot_ent * 4, cudaMemcpyDeviceToHost));
    std::vector<int> wide((size_t)p->tot_src * KCAP, what == FICOCO_INSPECT_CORR_TGT ? -1 : 0);
    for (const ImgDesc& d : p->h_desc)
      for (int s = 0; s < d.n_src; ++s)
        for (int k = 0; k < d.list_len; ++k)
          wide[(size_t)(d.src0 + s) * KCAP + k] = compact[(size_t)d.ent0 + (size_t)s * d.list_len + k];
    memcpy(host_dst, wide.data(), bytes < n ? bytes : n);
    return FICOCO_OK;
  }
  CUDA_TRY(c, cudaMemcpy(host_dst, src, bytes < n ? bytes : n, cudaMemcpyDeviceToHost));
  return FICOCO_OK;
}

// ---------------------------------------------------------------------------------------
// Host-buffer entry points
// ---------------------------------------------------------------------------------------
namespace {

int ensure_staging(ficoco_ctx* c, size_t dev_bytes) {
  if (!c->hs_stream) CUDA_TRY(c, cudaStreamCreateWithFlags(&c->hs_stream, cudaStreamNonBlocking));
  if (!c->hs_run) CUDA_TRY(c, cudaStreamCreateWithFlags(&c->hs_run, cudaStreamNonBlocking));
  if (!c->hs_out) CUDA_TRY(c, cudaStreamCreateWithFlags(&c->hs_out, cudaStreamNonBlocking));
  for (int i = 0; i < 2 * HOST_MAX_GROUPS; ++i)
    if (!c->hs_ev[i]) CUDA_TRY(c, cudaEventCreateWithFlags(&c->hs_ev[i], cudaEventDisableTiming));
  if (dev_bytes > c->hs_dev_bytes) {
    if (c->hs_dev) { CUDA_TRY(c, cudaDeviceSynchronize()); cudaFree(c->hs_dev); c->hs_dev = nullptr; }
    CUDA_TRY(c, cudaMalloc((void**)&c->hs_dev, dev_bytes));
    c->hs_dev_bytes = dev_bytes;
  }
  return FICOCO_OK;
}

struct Carver {
  char* base;
  size_t off = 0;
  explicit Carver(char* b) : base(b) {}
  template <class U> U* take(size_t bytes) { U* p = (U*)(base + off); off += align_up(bytes, 256); return p; }
};

}  // namespace

extern "C" int ficoco_v_reduce_host(ficoco_ctx* c, const ficoco_v_args* h, const ficoco_params* prm) {
  if (!c || !h || !prm) return FICOCO_ERR_INVALID_ARG;
  if (!h->tokens || !h->attn || !h->keep || !h->out_tokens || !h->kept_idx || h->batch < 1 || h->dim < 1 ||
      h->heads < 1 || (h->n_keep != 1 && h->n_keep != h->batch))
    return FICOCO_ERR_INVALID_ARG;
  if (h->dtype != FICOCO_FP32 && h->dtype != FICOCO_BF16) return FICOCO_ERR_UNSUPPORTED;
  const int cls = (prm->flags & FICOCO_HAS_CLS) ? 1 : 0;
  const size_t es = h->dtype == FICOCO_BF16 ? 2 : 4;
  const int B = h->batch;
  // prefix sums over images: input rows, patch tokens, output rows, preserved tokens
  std::vector<long long> p_rows(B + 1, 0), p_patch(B + 1, 0), p_orow(B + 1, 0), p_kept(B + 1, 0);
  for (int b = 0; b < B; ++b) {
    const int n = h->seqlens ? h->seqlens[b] : h->n_tokens;
    const int k = h->keep[h->n_keep == 1 ? 0 : b];
    if (n < cls + 1 || k < 0 || k > n - cls) return FICOCO_ERR_KEEP_RANGE;
    p_rows[b + 1] = p_rows[b] + n;
    p_patch[b + 1] = p_patch[b] + n - cls;
    p_orow[b + 1] = p_orow[b] + cls + k + (((prm->flags & FICOCO_CONVERGENT) && n - cls - k > 0) ? 1 : 0);
    p_kept[b + 1] = p_kept[b] + k;
  }
  const long long rows = p_rows[B], patches = p_patch[B], orows = p_orow[B], kept = p_kept[B];
  if (rows > c->max_tokens) return FICOCO_ERR_WORKSPACE;
  CUDA_TRY(c, cudaSetDevice(c->device));
  const size_t b_tok = (size_t)rows * h->dim * es, b_attn = (size_t)patches * h->heads * 4;
  const size_t b_pos = h->pos ? (size_t)patches * 4 : 0;
  const size_t b_out = (size_t)orows * h->dim * es, b_kidx = (size_t)orows * 4;
  const size_t b_posout = h->pos_out ? (size_t)kept * 4 : 0, b_sc = h->scores_out ? (size_t)patches * 4 : 0;
  const size_t total = align_up(b_tok, 256) + align_up(b_attn, 256) + align_up(b_pos, 256) +
                       align_up(b_out, 256) + align_up(b_kidx, 256) + align_up(b_posout, 256) +
                       align_up(b_sc, 256) + 256;
  int rc = ensure_staging(c, total);
  if (rc) return rc;
  Carver dv(c->hs_dev);
  char* d_tok = dv.take<char>(b_tok);
  char* d_attn = dv.take<char>(b_attn);
  char* d_pos = dv.take<char>(b_pos);
  char* d_out = dv.take<char>(b_out);
  char* d_kidx = dv.take<char>(b_kidx);
  char* d_po = dv.take<char>(b_posout);
  char* d_sc = dv.take<char>(b_sc);

  // Images are independent, so the batch goes through in groups of images: the upload of a
  // group, the kernels of the group before it and the download of the one before that run at
  // the same time on three streams (PCIe carries both directions at once).  Every group has its
  // own slice of the staging area, so nothing is reused while in flight.
  int n_groups = (int)(b_tok / HOST_GROUP_BYTES);
  if (n_groups > HOST_MAX_GROUPS) n_groups = HOST_MAX_GROUPS;
  if (n_groups > B) n_groups = B;
  if (n_groups < 1) n_groups = 1;
  cudaStream_t s_in = c->hs_stream, s_run = c->hs_run, s_out = c->hs_out;
  if (n_groups == 1) s_run = s_out = s_in;
  const size_t row_b = (size_t)h->dim * es;
  int launches = 0;
  rc = FICOCO_OK;
  auto group_begin = [&](int g) { return (int)((long long)B * g / n_groups); };
  // all uploads first: they depend on nothing, and queued ahead of everything else they never
  // sit behind a download that is itself waiting for kernels
  for (int g = 0; g < n_groups && rc == FICOCO_OK; ++g) {
    const int b0 = group_begin(g), b1 = group_begin(g + 1);
    const size_t o_tok = (size_t)p_rows[b0] * row_b, n_tok = (size_t)(p_rows[b1] - p_rows[b0]) * row_b;
    const size_t o_at = (size_t)p_patch[b0] * h->heads * 4, n_at = (size_t)(p_patch[b1] - p_patch[b0]) * h->heads * 4;
    const size_t o_ps = (size_t)p_patch[b0] * 4, n_ps = (size_t)(p_patch[b1] - p_patch[b0]) * 4;
    cudaError_t e = cudaMemcpyAsync(d_tok + o_tok, (const char*)h->tokens + o_tok, n_tok, cudaMemcpyHostToDevice, s_in);
    if (e == cudaSuccess)
      e = cudaMemcpyAsync(d_attn + o_at, (const char*)h->attn + o_at, n_at, cudaMemcpyHostToDevice, s_in);
    if (e == cudaSuccess && h->pos)
      e = cudaMemcpyAsync(d_pos + o_ps, (const char*)h->pos + o_ps, n_ps, cudaMemcpyHostToDevice, s_in);
    if (e == cudaSuccess && n_groups > 1) e = cudaEventRecord(c->hs_ev[2 * g], s_in);
    if (e != cudaSuccess) { c->last_cuda = (int)e; rc = FICOCO_ERR_CUDA; }
  }
  for (int g = 0; g < n_groups && rc == FICOCO_OK; ++g) {
    const int b0 = group_begin(g), b1 = group_begin(g + 1);
    const size_t o_tok = (size_t)p_rows[b0] * row_b;
    const size_t o_at = (size_t)p_patch[b0] * h->heads * 4;
    const size_t o_ps = (size_t)p_patch[b0] * 4, n_ps = (size_t)(p_patch[b1] - p_patch[b0]) * 4;
    const size_t o_out = (size_t)p_orow[b0] * row_b, n_out = (size_t)(p_orow[b1] - p_orow[b0]) * row_b;
    const size_t o_ki = (size_t)p_orow[b0] * 4, n_ki = (size_t)(p_orow[b1] - p_orow[b0]) * 4;
    const size_t o_po = (size_t)p_kept[b0] * 4, n_po = (size_t)(p_kept[b1] - p_kept[b0]) * 4;
    cudaError_t e = cudaSuccess;
    if (n_groups > 1) e = cudaStreamWaitEvent(s_run, c->hs_ev[2 * g], 0);
    if (e != cudaSuccess) { c->last_cuda = (int)e; rc = FICOCO_ERR_CUDA; break; }
    ficoco_v_args a = *h;
    a.batch = b1 - b0;
    a.tokens = d_tok + o_tok;
    a.attn = (const float*)(d_attn + o_at);
    a.pos = h->pos ? (const int*)(d_pos + o_ps) : nullptr;
    if (h->seqlens) a.seqlens = h->seqlens + b0;
    if (h->n_keep != 1) { a.keep = h->keep + b0; a.n_keep = b1 - b0; }
    if (h->n_grid != 1) { a.grid_h = h->grid_h + b0; a.grid_w = h->grid_w + b0; a.n_grid = b1 - b0; }
    a.out_tokens = d_out + o_out;
    a.kept_idx = (int*)(d_kidx + o_ki);
    a.pos_out = h->pos_out ? (int*)(d_po + o_po) : nullptr;
    a.scores_out = h->scores_out ? (float*)(d_sc + o_ps) : nullptr;
    rc = ficoco_v_reduce(c, &a, prm, s_run);
    if (rc) break;
    launches += c->launches;
    if (n_groups > 1) {
      e = cudaEventRecord(c->hs_ev[2 * g + 1], s_run);
      if (e == cudaSuccess) e = cudaStreamWaitEvent(s_out, c->hs_ev[2 * g + 1], 0);
    }
    if (e == cudaSuccess)
      e = cudaMemcpyAsync((char*)h->out_tokens + o_out, d_out + o_out, n_out, cudaMemcpyDeviceToHost, s_out);
    if (e == cudaSuccess)
      e = cudaMemcpyAsync((char*)h->kept_idx + o_ki, d_kidx + o_ki, n_ki, cudaMemcpyDeviceToHost, s_out);
    if (e == cudaSuccess && h->pos_out)
      e = cudaMemcpyAsync((char*)h->pos_out + o_po, d_po + o_po, n_po, cudaMemcpyDeviceToHost, s_out);
    if (e == cudaSuccess && h->scores_out)
      e = cudaMemcpyAsync((char*)h->scores_out + o_ps, d_sc + o_ps, n_ps, cudaMemcpyDeviceToHost, s_out);
    if (e != cudaSuccess) { c->last_cuda = (int)e; rc = FICOCO_ERR_CUDA; }
  }
  // drain all three streams whatever happened, so that no copy outlives the call
  const cudaError_t e1 = cudaStreamSynchronize(s_in), e2 = cudaStreamSynchronize(s_run),
                    e3 = cudaStreamSynchronize(s_out);
  if (rc) return rc;
  if (e1 != cudaSuccess || e2 != cudaSuccess || e3 != cudaSuccess) {
    c->last_cuda = (int)(e1 != cudaSuccess ? e1 : e2 != cudaSuccess ? e2 : e3);
    return FICOCO_ERR_CUDA;
  }
  c->launches = launches;
  return FICOCO_OK;
}

extern "C" int ficoco_l_reduce_host(ficoco_ctx* c, const ficoco_l_args* h, const ficoco_params* prm) {
  if (!c || !h || !prm) return FICOCO_ERR_INVALID_ARG;
  if (!h->tokens || !h->attn_t2v || !h->keep || !h->out_tokens || !h->kept_idx || h->batch < 1 ||
      h->dim < 1 || h->heads < 1 || h->n_vision < 1 || h->n_text < 1 ||
      (h->n_keep != 1 && h->n_keep != h->batch))
    return FICOCO_ERR_INVALID_ARG;
  if (h->dtype != FICOCO_FP32 && h->dtype != FICOCO_BF16) return FICOCO_ERR_UNSUPPORTED;
  const size_t es = h->dtype == FICOCO_BF16 ? 2 : 4;
  const int B = h->batch;
  std::vector<long long> p_orow(B + 1, 0);
  for (int b = 0; b < B; ++b) {
    const int k = h->keep[h->n_keep == 1 ? 0 : b];
    if (k < 0 || k > h->n_vision) return FICOCO_ERR_KEEP_RANGE;
    p_orow[b + 1] = p_orow[b] + k + h->n_text + (((prm->flags & FICOCO_CONVERGENT) && h->n_vision - k > 0) ? 1 : 0);
  }
  const long long orows = p_orow[B];
  const long long rows = (long long)B * (h->n_vision + h->n_text);
  if (rows > c->max_tokens) return FICOCO_ERR_WORKSPACE;
  CUDA_TRY(c, cudaSetDevice(c->device));
  const size_t seq_tok = (size_t)(h->n_vision + h->n_text) * h->dim * es;      // bytes per sequence
  const size_t seq_attn = (size_t)h->heads * h->n_text * h->n_vision * 4;
  const size_t seq_sc = (size_t)h->n_vision * 4;
  const size_t row_b = (size_t)h->dim * es;
  const size_t b_tok = seq_tok * B, b_attn = seq_attn * B;
  const size_t b_out = (size_t)orows * row_b, b_kidx = (size_t)orows * 4;
  const size_t b_sc = h->scores_out ? seq_sc * B : 0;
  const size_t total = align_up(b_tok, 256) + align_up(b_attn, 256) + align_up(b_out, 256) +
                       align_up(b_kidx, 256) + align_up(b_sc, 256) + 256;
  int rc = ensure_staging(c, total);
  if (rc) return rc;
  Carver dv(c->hs_dev);
  char* d_tok = dv.take<char>(b_tok);
  char* d_attn = dv.take<char>(b_attn);
  char* d_out = dv.take<char>(b_out);
  char* d_kidx = dv.take<char>(b_kidx);
  char* d_sc = dv.take<char>(b_sc);

  // Sequences are independent: groups of sequences go through upload, kernels and download on three
  // streams, as in ficoco_v_reduce_host (every group has its own slice of the staging area).
  int n_groups = (int)((b_tok + b_attn) / HOST_GROUP_BYTES);
  if (n_groups > HOST_MAX_GROUPS) n_groups = HOST_MAX_GROUPS;
  if (n_groups > B) n_groups = B;
  if (n_groups < 1) n_groups = 1;
  cudaStream_t s_in = c->hs_stream, s_run = c->hs_run, s_out = c->hs_out;
  if (n_groups == 1) s_run = s_out = s_in;
  int launches = 0;
  rc = FICOCO_OK;
  auto group_begin = [&](int g) { return (int)((long long)B * g / n_groups); };
  for (int g = 0; g < n_groups && rc == FICOCO_OK; ++g) {
    const int b0 = group_begin(g), b1 = group_begin(g + 1);
    cudaError_t e = cudaMemcpyAsync(d_tok + seq_tok * b0, (const char*)h->tokens + seq_tok * b0, seq_tok * (b1 - b0),
                                    cudaMemcpyHostToDevice, s_in);
    if (e == cudaSuccess)
      e = cudaMemcpyAsync(d_attn + seq_attn * b0, (const char*)h->attn_t2v + seq_attn * b0, seq_attn * (b1 - b0),
                          cudaMemcpyHostToDevice, s_in);
    if (e == cudaSuccess && n_groups > 1) e = cudaEventRecord(c->hs_ev[2 * g], s_in);
    if (e != cudaSuccess) { c->last_cuda = (int)e; rc = FICOCO_ERR_CUDA; }
  }
  for (int g = 0; g < n_groups && rc == FICOCO_OK; ++g) {
    const int b0 = group_begin(g), b1 = group_begin(g + 1);
    const size_t o_out = (size_t)p_orow[b0] * row_b, n_out = (size_t)(p_orow[b1] - p_orow[b0]) * row_b;
    const size_t o_ki = (size_t)p_orow[b0] * 4, n_ki = (size_t)(p_orow[b1] - p_orow[b0]) * 4;
    cudaError_t e = cudaSuccess;
    if (n_groups > 1) e = cudaStreamWaitEvent(s_run, c->hs_ev[2 * g], 0);
    if (e != cudaSuccess) { c->last_cuda = (int)e; rc = FICOCO_ERR_CUDA; break; }
    ficoco_l_args a = *h;
    a.batch = b1 - b0;
    a.tokens = d_tok + seq_tok * b0;
    a.attn_t2v = (const float*)(d_attn + seq_attn * b0);
    if (h->n_keep != 1) { a.keep = h->keep + b0; a.n_keep = b1 - b0; }
    a.out_tokens = d_out + o_out;
    a.kept_idx = (int*)(d_kidx + o_ki);
    a.scores_out = h->scores_out ? (float*)(d_sc + seq_sc * b0) : nullptr;
    rc = ficoco_l_reduce(c, &a, prm, s_run);
    if (rc) break;
    launches += c->launches;
    if (n_groups > 1) {
      e = cudaEventRecord(c->hs_ev[2 * g + 1], s_run);
      if (e == cudaSuccess) e = cudaStreamWaitEvent(s_out, c->hs_ev[2 * g + 1], 0);
    }
    if (e == cudaSuccess)
      e = cudaMemcpyAsync((char*)h->out_tokens + o_out, d_out + o_out, n_out, cudaMemcpyDeviceToHost, s_out);
    if (e == cudaSuccess)
      e = cudaMemcpyAsync((char*)h->kept_idx + o_ki, d_kidx + o_ki, n_ki, cudaMemcpyDeviceToHost, s_out);
    if (e == cudaSuccess && h->scores_out)
      e = cudaMemcpyAsync((char*)h->scores_out + seq_sc * b0, d_sc + seq_sc * b0, seq_sc * (b1 - b0),
                          cudaMemcpyDeviceToHost, s_out);
    if (e != cudaSuccess) { c->last_cuda = (int)e; rc = FICOCO_ERR_CUDA; }
  }
  // drain all three streams whatever happened, so that no copy outlives the call
  const cudaError_t e1 = cudaStreamSynchronize(s_in), e2 = cudaStreamSynchronize(s_run),
                    e3 = cudaStreamSynchronize(s_out);
  if (rc) return rc;
  if (e1 != cudaSuccess || e2 != cudaSuccess || e3 != cudaSuccess) {
    c->last_cuda = (int)(e1 != cudaSuccess ? e1 : e2 != cudaSuccess ? e2 : e3);
    return FICOCO_ERR_CUDA;
  }
  c->launches = launches;
  return FICOCO_OK;
}
