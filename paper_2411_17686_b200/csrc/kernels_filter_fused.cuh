// Filter stage as one persistent kernel (Eq. 1, local penalty, top-N^S selection).
//
// Launched cooperatively with one CTA per SM at most, so all CTAs are co-resident.  Every CTA
// owns a fixed list of "pieces" (consecutive patch rows of one image), of which each of its 16 warps
// takes a sixteenth and streams it through a shared-memory ring of its own (bulk copies, TMA).
//   pass 1  rn_i = 1/||x_i||, column sums of the normalised rows -> one partial per piece;
//           the piece's image counter is bumped;
//   pass 2  (the rows still in the rings from there, the others, now L2-resident, with 16-byte loads, several rows in
//           flight per warp) once all pieces of the image are in:
//           v_i = rn_i (x_i . sum of partials) / Np,  s_i = cA v_i - (1 - cA) a_i;
//   select  every CTA that scored a piece waits until all of the image's scores are in, runs the selection on the whole
//           image and writes the outputs of its own tokens.
// The inter-CTA waits are polls of per-image counters, bounded by elapsed time (wait_ns).  The
// counters ([0, B) pieces through pass 1, [B, 2B) pieces scored) exist twice; a launch uses the set of its parity and
// zeroes the whole other one, whatever its batch, behind its wait, so a step that ended before its merge cannot leave counts
// behind for the step after the next.  The set a launch
// used is cleared by the merge grid of the same step (which runs once the filter grid is complete
// and before a later filter grid can start), so launches replayed from CUDA graphs, whose
// parities are fixed at capture, find their set clean in whatever order they run.
//
// What bounds it: the read of the rows with 16 warps to convert and add them up (pass 1: 32 x 577 rows of 1024 bf16 take
// 7 us, 5.2 TB/s), then trips to L2 of 0.7 to 1.2 us one behind the other.  So the heads of the attention, the other
// pieces' column sums (half of the threads half of the pieces each) and the first rows and norms of pass 2 are each one
// trip, asked for before what they do not depend on is waited for; the plan is read under the tail of the grid before;
// the mean direction sits in registers, sums of four rows are folded together, and fp32 work goes two at a time.
// Phases, before / now: attention 2.1 / 1.1 us, column sums of 18 pieces 2.8 / 1.0, scores of 144 rows 6.9 / 5.2,
// publication of the scores 1.9 / 0.8.  Whole step: 16 ragged images 100.5 -> 92.0, one fp32 image 50.4 -> 47.1, 8 x 2881
// tokens 132.2 -> 130.7, 32 x 577 the same.
#pragma once
#include "async_ops.cuh"
#include "common.cuh"
#include "kernels_filter.cuh"

namespace ficoco {

constexpr int FWARPS = 16;
constexpr int FROWS = FWARPS;     // rows of a ring stage: one per warp
constexpr int FFOLD = 8;          // rows of the fold buffer (warps w and w + 8 share a row)
constexpr int F_NCONS = 512;
constexpr int F_MAXSTAGE = 16;
constexpr int F_MAXWON = 32;      // pieces per CTA
constexpr size_t F_SMEM = 216 * 1024;   // dynamic shared memory at most
// what is static beside it: the rings' barriers, the selections' tables, the pieces and their images, a flag
constexpr size_t F_STATIC = sizeof(uint64_t) * FWARPS * F_MAXSTAGE + sizeof(SelectShared) + sizeof(SelectSmallShared) +
                            F_MAXWON * (sizeof(WorkItem) + sizeof(ImgDesc)) + 128;
static_assert(F_SMEM + F_STATIC <= 227 * 1024, "a CTA of the fused filter does not fit an SM: no context could be created");
static_assert(F_NCONS == SEL_SMALL_THREADS, "the selection is written for the threads of this kernel");

__device__ __forceinline__ int ld_acquire(const int* p) {
  int v;
  asm volatile("ld.acquire.gpu.global.b32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// Poll until *p >= need.  Gives up after limit_ns, or at once when another CTA has already
// raised STATUS_TIMEOUT (its pieces will never arrive).  One thread calls this.
__device__ __forceinline__ bool poll_count(const int* p, int need, unsigned long long limit_ns,
                                           const unsigned* status) {
  unsigned long long t0 = 0;
  for (;;) {
    if (ld_acquire(p) >= need) return true;
    const unsigned long long t = sm_cycles();
    if (t0 == 0) t0 = t;
    else if (t - t0 > 2 * limit_ns) return false;
    if (*reinterpret_cast<const volatile unsigned*>(status) & STATUS_TIMEOUT) return false;
    __nanosleep(32);
  }
}

// The mean direction m (one float per column) is kept in shared memory so that a warp reads it
// without bank conflicts: with 8 columns per 16-byte vector, floats 0-3 of vector v live in plane
// A at 4v and floats 4-7 in plane B at 4(nvec + v); with 4 columns per vector there is one plane.
template <int E>
__device__ __forceinline__ int msum_slot(int c, int nvec) {
  const int v = c / E, e = c % E;
  return (e < 4 ? 0 : 4 * nvec) + 4 * v + (e & 3);
}

// Sums of four values over the warp in six shuffles: lanes 8 r .. 8 r + 7 end up with the sum of v[r].
__device__ __forceinline__ float warp_sum4(const float (&v)[4], int lane) {
  const bool hi = lane & 16, odd = lane & 8;
  float a = hi ? v[2] : v[0], b = hi ? v[3] : v[1];
  a += __shfl_xor_sync(0xFFFFFFFFu, hi ? v[0] : v[2], 16);
  b += __shfl_xor_sync(0xFFFFFFFFu, hi ? v[1] : v[3], 16);
  float c = odd ? b : a;
  c += __shfl_xor_sync(0xFFFFFFFFu, odd ? a : b, 8);
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) c += __shfl_xor_sync(0xFFFFFFFFu, c, o);
  return c;
}

template <class T, int VPL>
__global__ void __launch_bounds__(F_NCONS, 1) k_filter_fused(
    const T* __restrict__ tokens, int D, const ImgDesc* __restrict__ desc,
    const WorkItem* __restrict__ pieces, const int* __restrict__ cta_first,
    float* __restrict__ rn, float* __restrict__ partial, const float* __restrict__ attn, int H, float cA,
    float* __restrict__ s_raw, int* __restrict__ cnt, int B,
    const int* __restrict__ pos, int window, float coef, int penalty, float* __restrict__ s_pen,
    float* __restrict__ scores_out, int* __restrict__ S_idx, int* __restrict__ T_idx,
    int* __restrict__ kept_idx, int* __restrict__ pos_out, unsigned* __restrict__ status,
    int nstage, int* __restrict__ other_cnt, int n_other, unsigned long long wait_ns, int dbg_extra_arrivals,
    int dep_wait_first) {
  constexpr int E = VecTraits<T>::E;
  constexpr int F_P2B = VPL <= 4 ? 4 : VPL <= 5 ? 2 : 1;   // rows a warp has in flight from L2 in pass 2
  extern __shared__ __align__(128) unsigned char fs_raw[];
  __shared__ uint64_t full_bar[FWARPS][F_MAXSTAGE];
  __shared__ SelectShared sel_sh;
  __shared__ SelectSmallShared sel_small_sh;
  // All CTAs of this grid are co-resident, so the next grid may be staged right away: its blocks
  // take over SMs as blocks of this grid exit and park until this grid has completed.
  grid_dep_launch();
  FICOCO_PHASE_BEGIN(0);
  __shared__ int failed;
  __shared__ WorkItem w_s[F_MAXWON];          // this CTA's pieces and their images
  __shared__ ImgDesc d_s[F_MAXWON];

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int row_bytes = D * (int)sizeof(T);
  const int stage_bytes = FROWS * row_bytes;
  const int nvec = D / E;
  unsigned char* ring = fs_raw;
  float* fold = reinterpret_cast<float*>(fs_raw + (size_t)nstage * stage_bytes);   // [FFOLD][D], msum aliases fold[0]
  float* a_s = fold + (size_t)FFOLD * D;                                            // a float per row of the largest piece
  const int p_begin = cta_first[blockIdx.x], p_end = cta_first[blockIdx.x + 1];
  if (lane < nstage) mbar_init(&full_bar[warp][lane], 1);
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  if (tid == 0) failed = 0;
  // (plan data: looked up once, under the tail of the grid before)
  for (int i = warp; i < p_end - p_begin; i += F_NCONS / 32) {
    const WorkItem w = pieces[p_begin + i];
    static_assert(sizeof(ImgDesc) % 4 == 0 && sizeof(ImgDesc) / 4 <= 32, "a lane copies a word of the descriptor");
    if (lane == 0) w_s[i] = w;
    if (lane < sizeof(ImgDesc) / 4)
      reinterpret_cast<uint32_t*>(&d_s[i])[lane] = reinterpret_cast<const uint32_t*>(desc + w.img)[lane];
  }
  __syncthreads();
  // A step fed from the outputs of the step before it on the stream (a progressive schedule) is
  // still launched early, so that its blocks are in place and set up when that step ends, but
  // must not touch the tokens before then.
  if (dep_wait_first) grid_dep_wait();

  // Every warp has a ring of its own for its sixteenth of a piece's rows (G = ceil(rows / 16) consecutive ones; a warp's
  // rows end where the piece does).  Lane 0 asks for the first row and for as many behind it as fit here, then, once the
  // warp has read a row, for the one that takes its place.  A copy of several rows completes on the barrier of its first
  // slot and the others' complete without one: slots are read in order.  (One ring of 16-row copies for all, filled by a
  // producer warp: the warps advance in step, and a 17th warp leaves 96 registers a thread instead of 128; filled by a
  // consumer, which every 32 KB copy keeps for half a microsecond, or row by row from the start, 80 copies of 54 cycles:
  // 32 x 577 tokens 60.8 and 59.7 us.)
  int issued = 0, ip = p_begin, ig = 0;            // rows asked for; piece and number of the next one
  unsigned char* my_ring = ring + (size_t)warp * nstage * row_bytes;
  auto issue = [&](int most) {
    if (ip >= p_end) return;
    const WorkItem& w = w_s[ip - p_begin];
    const ImgDesc& d = d_s[ip - p_begin];
    const int G = (w.nrows + FROWS - 1) / FROWS, r = warp * G + ig, n = min(most, G - ig), have = max(0, min(n, w.nrows - r));
    const int s = issued % nstage;
    if (have > 0) {
      mbar_expect_tx(&full_bar[warp][s], (uint32_t)(have * row_bytes));
      bulk_load(my_ring + (size_t)s * row_bytes, tokens + (size_t)(d.row0 + d.n_cls + w.r0 + r) * D,
                (uint32_t)(have * row_bytes), &full_bar[warp][s]);
    }
    for (int j = have > 0 ? 1 : 0; j < n; ++j) mbar_arrive(&full_bar[warp][s + j]);
    issued += n;
    ig += n;
    if (ig >= G) { ig = 0; ++ip; }
  };
  if (lane == 0) {
    issue(1);
    while (issued < nstage && ip < p_end) issue(nstage - issued);
  }
  __syncwarp();

  FICOCO_PHASE(0, 1);
  int seq = 0;
  bool ok = true;
  // Head mean of the attention of a piece's rows, the heads' loads in flight together (four at a time by the compiler's own
  // choice kept the first warps from pass 1 for 2 us on 32 x 577 tokens, 4 us on 16 ragged images).
  auto attn_means = [&](const WorkItem& w, const ImgDesc& d) {
    const float inv_h = 1.0f / (float)H;
    for (int r = tid; r < w.nrows; r += F_NCONS) {
      const float* a = attn + d.attn0 + w.r0 + r;
      float t = 0.f;
      for (int h0 = 0; h0 < H; h0 += 16) {
        float q[16];
#pragma unroll
        for (int j = 0; j < 16; ++j) q[j] = h0 + j < H ? __ldg(a + (size_t)(h0 + j) * d.np) : 0.f;
#pragma unroll
        for (int j = 0; j < 16; ++j) t += q[j];
      }
      a_s[r] = t * inv_h;
    }
  };
  // That of the first piece depends on nothing this kernel computes: it is fetched now, while the ring fills, instead of
  // between the two passes.
  if (p_begin < p_end) attn_means(w_s[0], d_s[0]);
  // pass 1: norms and column sums
  for (int pi = p_begin; pi < p_end; ++pi) {
    const WorkItem& w = w_s[pi - p_begin];
    const ImgDesc& d = d_s[pi - p_begin];
    float2 acc[VPL][E / 2];
#pragma unroll
    for (int k = 0; k < VPL; ++k)
#pragma unroll
      for (int e = 0; e < E / 2; ++e) acc[k][e] = make_float2(0.f, 0.f);
    const int G1 = (w.nrows + FROWS - 1) / FROWS;
    for (int g = 0; g < G1; ++g, ++seq) {
      const int s = seq % nstage;
      ok = __all_sync(0xFFFFFFFFu, ok && mbar_wait(&full_bar[warp][s], (seq / nstage) & 1, wait_ns));
      const int r = warp * G1 + g;
      if (r < w.nrows) {
        const unsigned char* rp = my_ring + (size_t)s * row_bytes;
        uint4 u[VPL];
        float2 ssk[VPL];
#pragma unroll
        for (int k = 0; k < VPL; ++k) {
          const int v = lane + 32 * k;
          u[k] = v < nvec ? *reinterpret_cast<const uint4*>(rp + (size_t)v * 16) : make_uint4(0, 0, 0, 0);
        }
#pragma unroll
        for (int k = 0; k < VPL; ++k) {
          float2 f[E / 2];
          unpack2(u[k], f, (const T*)nullptr);
          ssk[k] = make_float2(0.f, 0.f);
#pragma unroll
          for (int e = 0; e < E / 2; ++e) ssk[k] = fma2(f[e], f[e], ssk[k]);
        }
        float ss = 0.f;
#pragma unroll
        for (int k = 0; k < VPL; ++k) ss += ssk[k].x + ssk[k].y;
        ss = warp_sum(ss);
        const float s1 = ss > 0.f ? 1.0f / sqrtf(ss) : 0.f;
        if (lane == 0) rn[d.patch0 + w.r0 + r] = s1;
        const float2 s2 = make_float2(s1, s1);
#pragma unroll
        for (int k = 0; k < VPL; ++k) {
          float2 f[E / 2];
          unpack2(u[k], f, (const T*)nullptr);
#pragma unroll
          for (int e = 0; e < E / 2; ++e) acc[k][e] = fma2(f[e], s2, acc[k][e]);
        }
      }
      __syncwarp();
      if (lane == 0 && ok) issue(1);
      __syncwarp();
    }
    // fold the 16 warps in a fixed order -> partial of this piece: warps 0-7 store, warps 8-15
    // add into the row of warp - 8, then the 8 rows are summed per column
#pragma unroll
    for (int half = 0; half < 2; ++half) {
      if (warp / FFOLD == half) {
#pragma unroll
        for (int k = 0; k < VPL; ++k) {
          const int v = lane + 32 * k;
          if (v < nvec) {
            float4* dst = reinterpret_cast<float4*>(fold + (size_t)(warp % FFOLD) * D + (size_t)v * E);
#pragma unroll
            for (int q = 0; q < E / 4; ++q) {
              float4 x = half ? dst[q] : make_float4(0.f, 0.f, 0.f, 0.f);
              x.x += acc[k][2 * q].x; x.y += acc[k][2 * q].y; x.z += acc[k][2 * q + 1].x; x.w += acc[k][2 * q + 1].y;
              dst[q] = x;
            }
          }
        }
      }
      cta_sync(1, F_NCONS);
    }
    float* pout = partial + (size_t)(d.chunk0 + w.aux) * D;
    for (int c = tid; c < D; c += F_NCONS) {
      float t = 0.f;
#pragma unroll
      for (int ww = 0; ww < FFOLD; ++ww) t += fold[(size_t)ww * D + c];
      pout[c] = t;
    }
    cta_sync(1, F_NCONS);
    if (tid == 0) red_release_add(&cnt[w.img], 1);   // pairs with the ld.acquire poll of pass 2
  }
  if (!ok && lane == 0) {
    atomicOr(status, STATUS_TIMEOUT);
    failed = 1;
    // no copy outlives the CTA
    for (int q = max(0, issued - nstage); q < issued; ++q) mbar_wait(&full_bar[warp][q % nstage], (q / nstage) & 1, wait_ns);
  }
  __syncwarp();
  FICOCO_PHASE(0, 2);

  // pass 2: scores.  The last `nstage` row groups of pass 1 are still in the ring and are read
  // from there (only when every wait of pass 1 succeeded); the older ones are L2-resident and
  // are read with plain loads.
  const int first_kept = ok ? seq - nstage : seq;   // rows numbered >= this are in shared memory
  int seq2 = 0;
  for (int pi = p_begin; pi < p_end; ++pi) {
    const WorkItem& w = w_s[pi - p_begin];
    const ImgDesc& d = d_s[pi - p_begin];
    const int seq_piece = seq2;                     // number of the warp's first row of this piece
    const int nrows = w.nrows;
    const T* base = tokens + (size_t)(d.row0 + d.n_cls + w.r0) * D;
    // Row g of this warp is row warp * G + g of the piece.  Those below g_res were overwritten in the ring and come from
    // L2; the others are still in shared memory.
    const int G = (nrows + FROWS - 1) / FROWS;
    const int g_res = min(G, max(0, first_kept - seq_piece));
    seq2 += G;
    // The first rows from L2 and the norms of the warp's rows (lane l: row l) are asked for before the
    // other pieces' column sums are waited for: they depend on nothing but this CTA.
    uint4 ub[F_P2B][VPL];
    auto load_row = [&](int g, uint4 (&u)[VPL]) {
      const int r = warp * G + g;
      const bool on = g < g_res && r < nrows;
#pragma unroll
      for (int k = 0; k < VPL; ++k) {
        const int v = lane + 32 * k;
        u[k] = (on && v < nvec) ? ld16_now(base + (size_t)r * D + (size_t)v * E) : make_uint4(0, 0, 0, 0);
      }
    };
#pragma unroll
    for (int j = 0; j < F_P2B; ++j) load_row(j, ub[j]);
    const int row_l = warp * G + lane;
    const float rn_l = (lane < G && row_l < nrows) ? ld_now(rn + d.patch0 + w.r0 + row_l) : 0.f;
    if (tid == 0 && !poll_count(&cnt[w.img], d.n_chunks + dbg_extra_arrivals, wait_ns, status)) {
      atomicOr(status, STATUS_TIMEOUT);
      failed = 1;
    }
    if (pi == p_begin) FICOCO_PHASE(0, 3);
    if (pi > p_begin) attn_means(w, d);
    cta_sync(1, F_NCONS);
    // Column sums of the image: half of the threads adds the first half of the pieces, the others the second, four columns
    // and twelve pieces in flight each, so that up to 24 pieces are one trip to L2.
    {
      const int half = tid >> 8, nh = (d.n_chunks + 1) / 2, k_lo = half * nh, k_hi = min(d.n_chunks, k_lo + nh);
      for (int c = 4 * (tid & 255); c < D; c += 4 * 256) {
        float4 t = make_float4(0.f, 0.f, 0.f, 0.f);
        #pragma unroll 1
        for (int k0 = k_lo; k0 < k_hi; k0 += 12) {
          float4 q[12];
#pragma unroll
          for (int k = 0; k < 12; ++k)
            q[k] = k0 + k < k_hi ? __ldcg(reinterpret_cast<const float4*>(partial + (size_t)(d.chunk0 + k0 + k) * D + c))
                                 : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
          for (int k = 0; k < 12; ++k) { t.x += q[k].x; t.y += q[k].y; t.z += q[k].z; t.w += q[k].w; }
        }
        *reinterpret_cast<float4*>(fold + (size_t)half * D + msum_slot<E>(c, nvec)) = t;
      }
    }
    cta_sync(1, F_NCONS);
    if (pi == p_begin) FICOCO_PHASE(0, 4);
    // The lane's columns of the mean direction, for all its rows.  (Read from shared memory with every pair of rows, they
    // were half of this pass's shared-memory traffic.)
    float2 m[VPL][E / 2];
#pragma unroll
    for (int k = 0; k < VPL; ++k) {
      const int vv = lane + 32 * k < nvec ? lane + 32 * k : 0;
#pragma unroll
      for (int e = 0; e < E; e += 4) {
        const float* at = fold + 4 * (e / 4 * nvec + vv);
        const float4 ma = *reinterpret_cast<const float4*>(at), mb = *reinterpret_cast<const float4*>(at + D);
        m[k][e / 2] = make_float2(ma.x + mb.x, ma.y + mb.y);
        m[k][e / 2 + 1] = make_float2(ma.z + mb.z, ma.w + mb.w);
      }
    }
    const float inv_np = 1.0f / (float)d.np;
    float* s_out = s_raw + d.patch0 + w.r0;
    // Rows g .. g + 3 of the warp (from `end` on: nothing), their dot products summed over the warp together.
    auto finish_rows = [&](int g, int end, const float (&dot)[4]) {
      const float t = warp_sum4(dot, lane);
      g += lane >> 3;
      const int r = warp * G + g;
      const float k = __shfl_sync(0xFFFFFFFFu, rn_l, g & 31);
      if ((lane & 7) == 0 && g < end && r < nrows) {
        const float rnv = g < 32 ? k : __ldcg(rn + d.patch0 + w.r0 + r);
        s_out[r] = cA * (t * rnv * inv_np) - (1.0f - cA) * a_s[r];
      }
    };
    auto add_dot = [&](const uint4& u, int k, float2& dot) {
      float2 f[E / 2];
      unpack2(u, f, (const T*)nullptr);
#pragma unroll
      for (int e = 0; e < E / 2; ++e) dot = fma2(f[e], m[k][e], dot);
    };
    // the rows in the ring, four at a time, while the first ones from L2 are in flight (lines without a row: garbage that
    // nothing stores)
    #pragma unroll 1
    for (int g = g_res; g < G; g += 4) {
      const unsigned char* rp[4];
      float2 dot2[4];
      float dot[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        rp[j] = my_ring + (size_t)((seq_piece + min(g + j, G - 1)) % nstage) * row_bytes;
        dot2[j] = make_float2(0.f, 0.f);
      }
#pragma unroll
      for (int k = 0; k < VPL; ++k) {
        const int v = lane + 32 * k;
        if (v < nvec) {
#pragma unroll
          for (int j = 0; j < 4; ++j) add_dot(*reinterpret_cast<const uint4*>(rp[j] + (size_t)v * 16), k, dot2[j]);
        }
      }
      __syncwarp();
#pragma unroll
      for (int j = 0; j < 4; ++j) dot[j] = dot2[j].x + dot2[j].y;
      finish_rows(g, G, dot);
    }
    // the others, the registers of a batch filled again as soon as it is done
    #pragma unroll 1
    for (int g0 = 0; g0 < g_res; g0 += F_P2B) {
      float dot[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        dot[j] = 0.f;
        if (j < F_P2B) {
          float2 dot2 = make_float2(0.f, 0.f);
#pragma unroll
          for (int k = 0; k < VPL; ++k) add_dot(ub[j][k], k, dot2);
          dot[j] = dot2.x + dot2.y;
        }
      }
#pragma unroll
      for (int j = 0; j < F_P2B; ++j) load_row(g0 + F_P2B + j, ub[j]);
      finish_rows(g0, min(g_res, g0 + F_P2B), dot);
    }
    cta_sync(1, F_NCONS);
    if (tid == 0) red_release_add(&cnt[B + w.img], 1);   // releases this piece's scores; the selection polls for all of them
  }
  cta_sync(1, F_NCONS);

  FICOCO_PHASE(0, 5);
  // Without dep_wait_first (the caller states that what sits in front is a step of this library) the kernel has by now
  // written only scratch that no grid but a filter or correlate grid reads, and those of that step had ended before its
  // merge let this grid in.  The index lists and outputs written below are read by that merge: wait for it, also after a
  // wait that ran out, since the grid behind this one waits for this one alone.
  grid_dep_wait();
  // the counters of the launch before, complete by now, are zeroed for the launch after (see the top)
  if (blockIdx.x == 0)
    for (int i = tid; i < n_other; i += F_NCONS) other_cnt[i] = 0;
  if (failed) return;
  FICOCO_PHASE(0, 6);
  // selections (the ring is idle now and serves as work area), image by image over this CTA's pieces
  int pi = p_begin;
  #pragma unroll 1
  while (pi < p_end) {
    const WorkItem& w0 = w_s[pi - p_begin];
    const ImgDesc& d = d_s[pi - p_begin];
    int pj = pi, hi = w0.r0;
    while (pj < p_end && w_s[pj - p_begin].img == w0.img) { hi = w_s[pj - p_begin].r0 + w_s[pj - p_begin].nrows; ++pj; }
    const bool small = d.np <= SEL_SMALL_MAX;
    if (small) select_small_prepare(d, penalty, ring, tid);
    else select_image_prepare(d, penalty, ring, sel_sh, tid);
    if (tid == 0 && !poll_count(&cnt[B + w0.img], d.n_chunks, wait_ns, status)) {
      atomicOr(status, STATUS_TIMEOUT);
      failed = 1;
    }
    cta_sync(1, F_NCONS);
    if (failed) return;
    FICOCO_PHASE(0, 7);
    // (the counters are not reset here: the next launch zeroes this launch's set, see the top)
    if (small)
      select_small(d, s_raw, pos, window, coef, penalty, s_pen, scores_out, S_idx, T_idx, kept_idx, pos_out,
                   status, ring, sel_small_sh, tid, 1, w0.r0, hi);
    else
      select_image(d, s_raw, pos, window, coef, penalty, s_pen, scores_out, S_idx, T_idx, kept_idx, pos_out,
                   status, ring, sel_sh, tid, 1, w0.r0, hi);
    if (pj < p_end) cta_sync(1, F_NCONS);         // the work area is used again by the next image
    pi = pj;
  }
  FICOCO_PHASE(0, 8);
}

}  // namespace ficoco
