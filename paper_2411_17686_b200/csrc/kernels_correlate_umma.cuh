// Correlate stage on the 5th-generation tensor cores (bf16 tokens; FiCoCo-V, and FiCoCo-L with its
// text-bridged term added in the epilogue).
//
// One CTA owns a tile of discarded tokens (rows of the accumulator, one TMEM lane each) and
// one column split (<= 256 preserved tokens) of one image; two CTAs share an SM:
//   warps 0-3, 5-8  gather the token rows with 16-byte cp.async into a ring of 128B-swizzled,
//              K-major shared-memory tiles (64, 128 or 256 bf16 of the hidden dimension per stage);
//   warp  4    allocates TMEM and issues tcgen05.mma (elect.sync, M = 128, N = columns rounded to 16,
//              K = 16 per instruction, fp32 accumulation of exact bf16 products);
//   warps 0-3, 5-8  afterwards read TMEM lanes back with tcgen05.ld (warps 0-3 the lower half
//              of the columns, warps 5-8 the upper half of the same lanes), scale by
//              rn_i * rn_j to cosines and keep each row's L <= LCAP largest entries in registers.
// Rows / columns past the valid range are never loaded: their shared memory is garbage that
// only reaches accumulator rows / columns the epilogue ignores.
// Every wait is bounded; on a timeout the CTA raises STATUS_TIMEOUT, drains its copies,
// frees its TMEM and returns.
//
// What bounds the k-loop: large tiles, the rate at which copies fill shared memory (66 to 79 bytes per cycle and SM at
// 360 and 192 rows per CTA); small ones, the instructions of a stage (waits, addresses, arrivals: about 400 cycles a
// warp), as a stage costs the same with its copies or its MMAs left out.  So a copy is predicated instead of branched
// around, a stage takes up to four k-blocks, the descriptors are made from the ring's address as it is (a shuffle
// "to make it uniform" put 47 cycles on every MMA, 31 without), and row indices and norms are asked for as soon as the
// lists exist.  k-loop of one FiCoCo-L sequence (80 rows per CTA, 64 k-blocks) 15.4 -> 10 us, of one image of 144 tokens
// 3.5 -> 2.2, of 32 x 577 tokens 5.6 -> 5.8, of 16 sequences 16.6 -> 13.
// Taken back: one arrival per warp after waiting for its copies (one sequence 17 to 28 us: the loop then runs at the
// latency of a copy), groups of warps that fill different stages with the row offsets in shared memory (10 us there, but
// 8 x 2881 tokens 12 -> 15), up to four accumulators in turn (the same).
#pragma once
#include <limits.h>
#include <math_constants.h>
#include "async_ops.cuh"
#include "common.cuh"
#include "correlate_plan.h"
#include "kernels_correlate.cuh"

namespace ficoco {

constexpr int UTHREADS = 288;    // warps 0-3 and 5-8 gather + epilogue, warp 4 MMA
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// K-major, 128-byte swizzle: rows of 128 bytes, 8-row groups 1024 bytes apart.
__device__ __forceinline__ uint64_t umma_smem_desc(uint32_t saddr) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);   // start address, 16-byte units
  d |= (uint64_t)1 << 16;                      // leading byte offset (unused for swizzled K-major)
  d |= (uint64_t)(1024 >> 4) << 32;            // stride byte offset between 8-row groups
  d |= (uint64_t)1 << 46;                      // descriptor version for sm_100
  d |= (uint64_t)2 << 61;                      // SWIZZLE_128B
  return d;
}
// kind::f16 instruction descriptor: D fp32, A and B bf16, both K-major, M = 128, N = n.
__device__ __forceinline__ uint32_t umma_idesc_bf16(int n) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(UM >> 4) << 24);
}
// umma_bf16 and umma_commit are called by a whole converged warp with uniform arguments; one elected lane
// issues.  (Called from a branch that only one lane takes, the same instructions cost 74 cycles per MMA and 175
// per commit to issue, because every operand travels from that lane to the uniform registers; called by the warp
// they cost 14-37 and 35: with four MMAs and a commit per k-block that was most of the k-loop.)
__device__ __forceinline__ void umma_bf16(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                          uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t"
      "elect.sync _|q, 0xFFFFFFFF;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "@q tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(d_tmem), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate) : "memory");
}
__device__ __forceinline__ void umma_commit(uint64_t* bar) {
  asm volatile(
      "{\n\t.reg .pred q;\n\t"
      "elect.sync _|q, 0xFFFFFFFF;\n\t"
      "@q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t}"
      ::"r"(smem_u32(bar)) : "memory");
}
// The same value in every lane, so that the compiler keeps it in uniform registers.
__device__ __forceinline__ uint32_t warp_uniform(uint32_t x) { return __shfl_sync(0xFFFFFFFFu, x, 0); }
__device__ __forceinline__ void tmem_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr) : "memory");
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

// 16 consecutive accumulator columns of this thread's TMEM lane; completes at tmem_ld_wait().
__device__ __forceinline__ void tmem_ld16_issue(uint32_t taddr, uint32_t* r) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr) : "memory");
}

// Takes t (column c) into a descending list of LCAP entries.  Branch-free: entry k changes when t > v[k], and then
// to the entry above it where that one changed as well, else to t.  '>' keeps the lower column first among equal
// values because columns arrive in ascending order; a NaN is never taken.
template <int LCAP>
__device__ __forceinline__ void toplist_take(float t, int c, float (&v)[LCAP], int (&ix)[LCAP]) {
  if constexpr (LCAP > 4) {      // more predicates than there are registers for: the displaced entry moves down
    bool in = false;
#pragma unroll
    for (int k = 0; k < LCAP; ++k) {
      in = in || t > v[k];
      const float tv = v[k];
      const int ti = ix[k];
      v[k] = in ? t : tv; ix[k] = in ? c : ti;
      t = in ? tv : t; c = in ? ti : c;
    }
    return;
  }
  bool p[LCAP];
#pragma unroll
  for (int k = 0; k < LCAP; ++k) p[k] = t > v[k];
#pragma unroll
  for (int k = LCAP - 1; k > 0; --k) {
    v[k] = p[k] ? (p[k - 1] ? v[k - 1] : t) : v[k];
    ix[k] = p[k] ? (p[k - 1] ? ix[k - 1] : c) : ix[k];
  }
  v[0] = p[0] ? t : v[0];
  ix[0] = p[0] ? c : ix[0];
}

// Top list of one accumulator row over the columns [c_lo, c_hi) (multiples of 16).  The code is
// kept small on purpose (a rolled loop over 16-column TMEM loads): it runs once per CTA, so a
// long unrolled body would be paid for in instruction-cache misses.  What bounds it is the number of
// instructions per entry: the row's own factor rs > 0 does not change the order of a row's entries and is
// applied to the list alone, padding columns carry a NaN in rnT instead of being compared with the column
// count, and the insertion is the one above (about 20 instructions per entry for four-entry lists, 40 before).
// v / ix: descending list, -inf / INT_MAX in empty slots.  Warp-collective (tcgen05.ld).
// FiCoCo-L adds the text-bridged term: tS (this row's text->vision weights, element k at
// tS[k * s_stride]) and tT ([M][t_stride], one row per text token over the CTA's columns) sit in
// shared memory; C = gamma * cosine + t_scale * sum_k tS_k tT_kc.  tT == nullptr: FiCoCo-V.
template <int LCAP>
__device__ __forceinline__ void epilogue_scan(uint32_t tmem_lane, int c_lo, int c_hi, int col_begin, float rs,
                                              const float* rnT, float (&v)[LCAP], int (&ix)[LCAP], const float* tS,
                                              int s_stride, const float* tT, int t_stride, int M, float gamma,
                                              float t_scale) {
#pragma unroll
  for (int k = 0; k < LCAP; ++k) { v[k] = -CUDART_INF_F; ix[k] = INT_MAX; }
  if (tT == nullptr) {
    #pragma unroll 1
    for (int c0 = c_lo; c0 < c_hi; c0 += 16) {
      uint32_t r[16];
      tmem_ld16(tmem_lane + (uint32_t)c0, r);
#pragma unroll
      for (int j = 0; j < 16; ++j) toplist_take<LCAP>(rnT[c0 + j] * __uint_as_float(r[j]), col_begin + c0 + j, v, ix);
    }
#pragma unroll
    for (int k = 0; k < LCAP; ++k)
      if (ix[k] != INT_MAX) v[k] *= rs;
    return;
  }
  #pragma unroll 1
  for (int c0 = c_lo; c0 < c_hi; c0 += 16) {
    uint32_t r[16];
    tmem_ld16_issue(tmem_lane + (uint32_t)c0, r);
    float tx[16];
#pragma unroll
    for (int j = 0; j < 16; ++j) tx[j] = 0.f;
    #pragma unroll 4
    for (int k = 0; k < M; ++k) {
      const float a = tS[(size_t)k * s_stride];
      const float4* q = reinterpret_cast<const float4*>(tT + (size_t)k * t_stride + c0);
#pragma unroll
      for (int j4 = 0; j4 < 4; ++j4) {
        const float4 t4 = q[j4];
        tx[4 * j4 + 0] = fmaf(a, t4.x, tx[4 * j4 + 0]);
        tx[4 * j4 + 1] = fmaf(a, t4.y, tx[4 * j4 + 1]);
        tx[4 * j4 + 2] = fmaf(a, t4.z, tx[4 * j4 + 2]);
        tx[4 * j4 + 3] = fmaf(a, t4.w, tx[4 * j4 + 3]);
      }
    }
    tmem_ld_wait();
#pragma unroll
    for (int j = 0; j < 16; ++j)
      toplist_take<LCAP>(gamma * ((rs * rnT[c0 + j]) * __uint_as_float(r[j])) + t_scale * tx[j], col_begin + c0 + j, v, ix);
  }
}

// Dynamic shared memory: [1024-aligned] ring of nstage stages, each KSUB k-blocks of an A tile (a_bytes: the
// valid source rows rounded up to 8, x 128 B) followed by a B tile (column rows x 128 B).  An
// MMA always reads 128 A rows; rows past a_bytes alias the B tile (or the slack the host adds
// behind the ring) and only feed accumulator rows that are never read.  FiCoCo-L's text weights lie text_off bytes behind
// the ring's start and are gathered ahead of the operands; with text_late they lie in the ring, behind the lists that the
// epilogue hands over there, and are gathered when the accumulator is complete.
template <int LCAP, int KSUB>
__global__ void __launch_bounds__(UTHREADS, 2) k_correlate_umma(
    const __nv_bfloat16* __restrict__ tokens, int D, const ImgDesc* __restrict__ desc,
    const WorkItem* __restrict__ work, const float* __restrict__ rn,
    const int* __restrict__ S_idx, const int* __restrict__ T_idx,
    float* __restrict__ part_val, int* __restrict__ part_idx, unsigned* __restrict__ status,
    int nstage, int stage_bytes, int a_bytes, int tmem_cols, int* __restrict__ img_done, int* __restrict__ corr_cnt,
    float* __restrict__ tau_out, int* __restrict__ e_tgt, float* __restrict__ e_w, float* __restrict__ e_c,
    const float* __restrict__ tmean, int M, int NV, float gamma, int text_off, int text_late, unsigned long long wait_ns) {
  extern __shared__ unsigned char um_raw[];
  __shared__ uint64_t full_bar[UM_STAGES], empty_bar[UM_STAGES], acc_bar;
  __shared__ uint32_t tmem_base_s;
  __shared__ float rnT[UN_MAX];
  __shared__ int failed, acc_committed, is_last, dead;

  FICOCO_PHASE_BEGIN(1);
  const WorkItem w = work[blockIdx.x];
  const ImgDesc d = desc[w.img];
  const int L = d.list_len;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int col_begin = w.aux * d.cols_per_split;
  const int ncols = min(d.n_tgt, col_begin + d.cols_per_split) - col_begin;   // 1..256
  const int n_pad = (ncols + 15) & ~15;
  const int nk = D / UKB, nkb = (nk + KSUB - 1) / KSUB;   // 64-element k-blocks, stages
  const uint32_t ring = (smem_u32(um_raw) + 1023u) & ~1023u;

  if (tid == 0) {
    for (int s = 0; s < nstage; ++s) { mbar_init(&full_bar[s], 256); mbar_init(&empty_bar[s], 1); }
    mbar_init(&acc_bar, 1);
    failed = 0;
    acc_committed = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 4) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                 ::"r"(smem_u32(&tmem_base_s)), "r"((uint32_t)tmem_cols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  // Everything above touches only launch-constant plan data and this CTA's own resources, so it
  // may run while the filter grid is still finishing; the index lists and norms it wrote are
  // read below.
  FICOCO_PHASE(1, 1);
  grid_dep_wait();
  grid_dep_launch();
  FICOCO_PHASE(1, 2);
  // Producer pt copies chunk (pt & 7) of rows (pt >> 3) + 32 i of the A tile and of the B tile, in every k-block
  // of the stage.  Byte offsets of the rows stay in registers and the swizzled destination advances by a constant
  // (32 rows = 4 KB).  A warp's four rows lie in one group of eight, so its number of copies is the same for all
  // lanes once the tile is rounded up to whole groups (the last row again in the rows added).  A thread looks its rows
  // up by itself, all of them at once; list entries are range-checked, so those of a step that gave up do no harm.
  const int pt = warp < 4 ? tid : tid - 32;
  const int chunk = pt & 7;
  const int rsub = pt >> 3;           // 0..31
  const int rgrp = (int)warp_uniform((uint32_t)(rsub >> 3) * 8);
  const int nA = (((w.nrows + 7) & ~7) - rgrp + 31) / 32, nB = (((ncols + 7) & ~7) - rgrp + 31) / 32;
  const int* Sl = S_idx + d.src0 + w.r0;
  const int* Tl = T_idx + d.tgt0 + col_begin;
  uint32_t offA[UM / 32], offB[UN_MAX / 32];
  const int row = ((warp & 3) << 5) + lane;       // accumulator row (TMEM lane) of this thread's epilogue
  const bool row_valid = row < w.nrows;
  int my_row = 0, my_col = -1;
  if (warp != 4) {
#pragma unroll
    for (int i = 0; i < UM / 32; ++i) offA[i] = i < nA ? (uint32_t)Sl[min(rsub + 32 * i, w.nrows - 1)] : 0u;
#pragma unroll
    for (int i = 0; i < UN_MAX / 32; ++i) offB[i] = i < nB ? (uint32_t)Tl[min(rsub + 32 * i, ncols - 1)] : 0u;
    if (row_valid) my_row = Sl[row];
    if (pt < ncols) my_col = Tl[pt];
  }
  // A filter grid that gave up left no valid index lists: do nothing but give the TMEM back.
  if (tid == 0) dead = (*reinterpret_cast<const volatile unsigned*>(status) & STATUS_TIMEOUT) ? 1 : 0;
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = tmem_base_s;
  if (dead) {
    if (warp == 4)
      asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"((uint32_t)tmem_cols)
                   : "memory");
    return;
  }
  FICOCO_PHASE(1, 3);

  if (warp != 4) {
    // ---------------- producers (all eight epilogue warps): gather rows, 16 bytes per copy -------
#pragma unroll
    for (int i = 0; i < UM / 32; ++i)
      offA[i] = ((uint32_t)checked_index((int)offA[i], d.np, status) * (uint32_t)D + chunk * 8) * 2u;
#pragma unroll
    for (int i = 0; i < UN_MAX / 32; ++i)
      offB[i] = ((uint32_t)checked_index((int)offB[i], d.np, status) * (uint32_t)D + chunk * 8) * 2u;
    const uint32_t dsw = (uint32_t)((rsub >> 3) * 1024 + (rsub & 7) * 128 + ((chunk ^ (rsub & 7)) << 4));
    const uint32_t kblock_bytes = (uint32_t)stage_bytes / KSUB;
    const char* src = reinterpret_cast<const char*>(tokens + (size_t)(d.row0 + d.n_cls) * D);
    // norms of this thread's column and of its accumulator row: asked for here, used in the epilogue
    const float rn_col = my_col >= 0 ? rn[d.patch0 + checked_index(my_col, d.np, status)] : CUDART_NAN_F;
    const float rs = row_valid ? rn[d.patch0 + checked_index(my_row, d.np, status)] : 0.f;
    // FiCoCo-L: the head-mean text->vision weights of the tile's columns and rows, a warp per eighth of the text.  (Gathered
    // behind the k-loop, eight at a time through registers, and for 128 rows whatever the tile, they took 4 of the 7 us
    // between accumulator and lists: one sequence of 576 + 64 tokens.)
    const int s_stride = (w.nrows + 7) & ~7;
    float* tT = tmean != nullptr ? reinterpret_cast<float*>(um_raw + (ring - smem_u32(um_raw)) + text_off) : nullptr;
    float* tSb = tT + (size_t)M * n_pad;
    auto gather_text = [&]() {
      const float* tb = tmean + (size_t)w.img * M * NV;
      #pragma unroll 1
      for (int j = lane; j < n_pad + s_stride; j += 32) {       // a column or a row of the tile
        const bool col = j < n_pad;
        const int at = col ? j : j - n_pad;
        if (at >= (col ? ncols : w.nrows)) continue;
        const float* from = tb + checked_index(col ? Tl[at] : Sl[at], d.np, status);
        const uint32_t to = smem_u32((col ? tT : tSb) + at), step = (uint32_t)(col ? n_pad : s_stride) * 4u;
        #pragma unroll 4
        for (int k = pt >> 5; k < M; k += 8) cp_async4(to + (uint32_t)k * step, from + (size_t)k * NV);
      }
    };
    if (tmean != nullptr && !text_late) gather_text();
    bool ok = true;
    // Each thread's copies of a stage arrive on its barrier when they have landed, so a producer never waits
    // for its own copies and the whole ring is in flight; the MMA warp orders the two proxies (below).
    int s = 0;
    uint32_t par = 1;
    #pragma unroll 1
    for (int kb = 0; kb < nkb; ++kb, src += KSUB * UKB * 2) {
      if (kb >= nstage) ok = mbar_wait(&empty_bar[s], par, wait_ns);
      if (!ok) break;
      const uint32_t a0 = ring + (uint32_t)s * stage_bytes + dsw;
      const uint32_t b0 = a0 + (uint32_t)a_bytes;
      const int nsub = KSUB == 1 ? 1 : min(KSUB, nk - KSUB * kb);    // k-blocks of this stage
#pragma unroll
      for (int i = 0; i < UM / 32; ++i) {
        const char* p = src + offA[i];
#pragma unroll
        for (int j = 0; j < KSUB; ++j) cp_async16_if(i < nA && (KSUB == 1 || j < nsub), a0 + j * kblock_bytes + i * 4096, p + j * (UKB * 2));
      }
#pragma unroll
      for (int i = 0; i < UN_MAX / 32; ++i) {
        const char* p = src + offB[i];
#pragma unroll
        for (int j = 0; j < KSUB; ++j) cp_async16_if(i < nB && (KSUB == 1 || j < nsub), b0 + j * kblock_bytes + i * 4096, p + j * (UKB * 2));
      }
      cp_async_arrive(&full_bar[s]);
      if (++s == nstage) { s = 0; par ^= 1u; }
    }
    FICOCO_PHASE(1, 4);
    rnT[pt] = rn_col;                                  // NaN in a padding column: no list takes its products
    if (!ok) { atomicOr(status, STATUS_TIMEOUT); failed = 1; }
    bool acc_ok = ok && mbar_wait(&acc_bar, 0, wait_ns);
    FICOCO_PHASE(1, 5);
    if (!acc_ok) { atomicOr(status, STATUS_TIMEOUT); failed = 1; cp_async_wait_all(); }
    acc_ok = __all_sync(0xFFFFFFFFu, acc_ok);          // tcgen05.ld below is warp-collective
    tc_fence_after();
    const float t_scale = tmean != nullptr ? (1.0f - gamma) / (float)M : 0.f;
    if (tmean != nullptr) {
      if (text_late && acc_ok) gather_text();          // (the accumulator is complete: nothing reads or fills the ring)
      cp_async_wait_all();
    }
    cta_sync(1, 256);                                  // norms and text weights are in shared memory
    // ---------------- epilogue: lane = accumulator row ---------------------------------------
    // Warps 0-3 scan the lower half of the columns, warps 5-8 (the same TMEM lanes) the upper half, whose lists come
    // back through the (now idle) operand ring.
    const int c_mid = ((n_pad / 16 + 1) / 2) * 16;
    const bool lower = warp < 4;
    float v[LCAP];
    int ix[LCAP];
    if (acc_ok && (warp & 3) * 32 < w.nrows)
      epilogue_scan<LCAP>(tmem_base + ((uint32_t)((warp & 3) * 32) << 16), lower ? 0 : c_mid, lower ? c_mid : n_pad,
                          col_begin, rs, rnT, v, ix, tSb + min(row, s_stride - 1), s_stride, tT, n_pad, M, gamma, t_scale);
    else {
#pragma unroll
      for (int k = 0; k < LCAP; ++k) { v[k] = -CUDART_INF_F; ix[k] = INT_MAX; }
    }
    float* hv = reinterpret_cast<float*>(um_raw + (ring - smem_u32(um_raw)));
    int* hi = reinterpret_cast<int*>(hv + UM * LCAP);
    if (!lower) {
#pragma unroll
      for (int k = 0; k < LCAP; ++k) { hv[row * LCAP + k] = v[k]; hi[row * LCAP + k] = ix[k]; }
    }
    cta_sync(1, 256);                                  // helper lists are in shared memory
    if (lower) {
      #pragma unroll 1                               // rolled: the body is a full insertion
      for (int e = 0; e < L; ++e) {
        float cv = hv[row * LCAP + e];
        int ci = hi[row * LCAP + e];
        bool shift = ci == INT_MAX;                // empty helper slot: nothing to insert
        if (!shift) {
#pragma unroll
          for (int k = 0; k < LCAP; ++k)
            if (k < L && (shift || toplist_better(cv, ci, v[k], ix[k]))) {
              const float tv = v[k]; const int ti = ix[k];
              v[k] = cv; ix[k] = ci; cv = tv; ci = ti;
              shift = true;
            }
        }
      }
      if (row_valid) {
        const size_t o = (size_t)d.part0 + ((size_t)(w.r0 + row) * d.nsplit + w.aux) * L;
#pragma unroll
        for (int k = 0; k < LCAP; ++k)
          if (k < L) {
            part_val[o + k] = v[k];
            part_idx[o + k] = ix[k] == INT_MAX ? -1 : ix[k];
          }
      }
    }
  } else {
    // ---------------- MMA issuer (the whole warp, one elected lane per instruction) -------------
    const uint32_t idesc = umma_idesc_bf16(n_pad);
    const uint32_t u_tmem = warp_uniform(tmem_base);
    const uint32_t kblock_bytes = (uint32_t)stage_bytes / KSUB;
    bool m_ok = true;
    int s = 0;
    uint32_t par = 0;
    #pragma unroll 1
    for (int kb = 0; kb < nkb; ++kb) {
      m_ok = __all_sync(0xFFFFFFFFu, mbar_wait(&full_bar[s], par, wait_ns));
      if (!m_ok) break;
      // the operands were written through the generic proxy (cp.async) and are read through the async
      // proxy: this fence sits between the two on the path that the barrier orders
      fence_proxy_async();
      tc_fence_after();
#pragma unroll
      for (int j = 0; j < KSUB; ++j) {
        if (j > 0 && KSUB * kb + j >= nk) break;
        const uint32_t a0 = ring + (uint32_t)s * stage_bytes + j * kblock_bytes;
        const uint64_t ad = umma_smem_desc(a0), bd = umma_smem_desc(a0 + (uint32_t)a_bytes);
#pragma unroll
        for (int k4 = 0; k4 < UKB / 16; ++k4) {
          const uint32_t acc = (kb > 0 || j > 0 || k4 > 0) ? 1u : 0u;
          umma_bf16(u_tmem, ad + (uint64_t)(k4 * 2), bd + (uint64_t)(k4 * 2), idesc, acc);
        }
      }
      umma_commit(&empty_bar[s]);      // frees the stage once these MMAs have read it
      if (++s == nstage) { s = 0; par ^= 1u; }
    }
    if (m_ok) umma_commit(&acc_bar);   // accumulator complete
    if (lane == 0) {
      if (m_ok) acc_committed = 1;
      else { atomicOr(status, STATUS_TIMEOUT); failed = 1; }
    }
    __syncwarp();
  }

  FICOCO_PHASE(1, 6);
  tc_fence_before();
  __syncthreads();
  FICOCO_PHASE(1, 7);
  if (warp == 4) {
    if (failed) {
      // MMAs may still be in flight: give them a bounded time to drain before freeing TMEM
      if (!acc_committed) umma_commit(&acc_bar);
      mbar_wait(&acc_bar, 0, wait_ns);
      __syncwarp();
    }
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"((uint32_t)tmem_cols)
                 : "memory");
  }
  correlate_tail<LCAP>(d, w, (int)blockIdx.x - w.aux, img_done, part_val, part_idx, corr_cnt, tau_out, e_tgt, e_w, e_c,
                       &is_last);
  FICOCO_PHASE(1, 8);
}

}  // namespace ficoco
