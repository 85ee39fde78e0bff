// Compress + compact (Eq. 2 and the last step of Algorithm 1 / 2).
#pragma once
#include "async_ops.cuh"
#include "common.cuh"

namespace ficoco {

constexpr int MTHREADS = 512;
constexpr int MWARPS = MTHREADS / 32;
constexpr int MROWS = 64;      // most output rows a CTA takes (a lane looks after two in the scan)
constexpr int MLIST = 1024;    // sources a CTA files in shared memory
constexpr int MDEPTH = 6;      // source rows a warp has in flight
constexpr size_t MSTAGE_BYTES = 70 * 1024;   // input rows of a CTA's output rows kept in shared memory (two CTAs per SM)

// Compress + compact.  A CTA owns a few output rows of one image, the ones `stride` apart from its first: targets
// with many sources lie close together (neighbouring patches look alike), and dealt out like cards they load the
// CTAs of an image about alike (16 ragged images: the busiest CTA 38 us after its start, 14 in the median, when the
// rows of a CTA were consecutive).
//   rows    the input rows of its output rows are fetched into shared memory by bulk copies (TMA) as soon as the
//           index lists exist, i.e. under the tail of the correlate grid;
//   file    the image's (source -> target) entries that hit its rows are filed into per-row lists in shared
//           memory, ordered by discarded token, so that every fp32 sum has one fixed order and no atomics touch
//           floats; one pass over the entries, four loads in flight per thread;
//   copies  a row that nothing is folded into leaves by a bulk store from shared memory: no thread touches it;
//   merge   out_j = (x_j + sum_{i in I_j} alpha_ij x_i) / (1 + sum alpha_ij), rounded once.  (slices of 32
//           vectors) x (own rows and sources, in list order) form one sequence of which every warp takes an equal
//           segment, MDEPTH source rows in flight: rows with one source and hubs with dozens cost what their
//           elements cost.  A group cut by the end of a segment is left in pieces in shared memory, which are
//           added in order.
// What bounds it is the latency of its few dependent trips to L2; the split into 16 warps and the host's choice of
// one wave of CTAs where possible keep them few: 32 x 577 -> 289 rows of 1024 went from 25 us (a scan per 16 rows,
// copies and hub rows by warps, two waves of CTAs) to 20 us, 16 ragged images keeping 1/9 from 48 to 28 us.
// If the CTA's rows receive more than MLIST sources in total, a slow in-order rescan is used.
template <class T>
__global__ void __launch_bounds__(MTHREADS, 2) k_merge_rows(
    const T* __restrict__ tokens, int D, const ImgDesc* __restrict__ desc,
    const WorkItem* __restrict__ work, const int* __restrict__ S_idx, const int* __restrict__ T_idx,
    const int* __restrict__ e_tgt, const float* __restrict__ e_w, T* __restrict__ out,
    int index_before_wait, unsigned* __restrict__ status, int* __restrict__ filter_cnt, int n_filter_cnt,
    unsigned long long wait_ns) {
  constexpr int E = VecTraits<T>::E;
  constexpr int PW = E + 1;                      // a piece: E sums and the weight of a lane, lanes side by side
  extern __shared__ __align__(128) unsigned char stage[];     // [rows][row bytes]
  __shared__ int cnt[MROWS], gbeg[MROWS + 1], beg[MROWS + 1], srow_s[MROWS];
  __shared__ int m_e[MLIST], bucket[MLIST];
  __shared__ unsigned short m_rs[MLIST];         // row << 10 | slot inside the row's bucket
  __shared__ uint2 el[MLIST + MROWS];            // weight, row << 16 | source token (the group's own row: anything)
  __shared__ float fold[MWARPS * PW * 32];
  __shared__ uint64_t row_bar;
  __shared__ int n_match, dead;
  FICOCO_PHASE_BEGIN(2);
  const WorkItem w = work[blockIdx.x];
  const ImgDesc d = desc[w.img];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int nvec = D / E, row_bytes = D * (int)sizeof(T);
  const int L = d.list_len;
  const int stride = w.aux;                      // row r of the CTA is output row w.r0 + r * stride of the image
  const float inv_stride = 1.0f / (float)stride;
  const int n_ent = d.n_src * L;
  const T* pbase = tokens + (size_t)(d.row0 + d.n_cls) * D;

  if (tid < MROWS) cnt[tid] = 0;
  if (tid == 0) n_match = 0;
  // When the grid before this one is a correlate grid, the filter grid (which wrote T_idx) had
  // completed before this grid could start, so the rows may be looked up and fetched under that
  // grid's tail; otherwise wait first.
  if (!index_before_wait) grid_dep_wait();
  if (warp == 0) {
    // input row of every output row (CLS / preserved token / trailing text row; -1: the additional token, which
    // k_convergent_token writes)
    if (lane == 0) {
      mbar_init(&row_bar, 1);
      asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    int srow[2], n = 0;
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const int r = lane + 32 * j, orow = w.r0 + r * stride;
      srow[j] = -1;
      if (r < w.nrows) {
        if (orow < d.n_cls) srow[j] = orow;
        else if (orow < d.n_cls + d.n_tgt) srow[j] = d.n_cls + checked_index(T_idx[d.tgt0 + orow - d.n_cls], d.np, status);
        else if (orow >= d.n_cls + d.n_tgt + d.n_extra) srow[j] = d.n_cls + d.np + (orow - d.n_cls - d.n_tgt - d.n_extra);
        srow_s[r] = srow[j];
        n += srow[j] >= 0 ? 1 : 0;
      }
    }
    n = __reduce_add_sync(0xFFFFFFFFu, n);
    if (lane == 0) mbar_expect_tx(&row_bar, (uint32_t)n * (uint32_t)row_bytes);
    __syncwarp();
#pragma unroll
    for (int j = 0; j < 2; ++j)
      if (srow[j] >= 0)
        bulk_load(stage + (size_t)(lane + 32 * j) * row_bytes, tokens + (size_t)(d.row0 + srow[j]) * D, (uint32_t)row_bytes,
                  &row_bar);
  }
  __syncthreads();
  if (index_before_wait) grid_dep_wait();
  // The filter grid of this step is complete: its per-image counters are cleared for whichever launch
  // uses that set next (launches replayed from graphs need not alternate between the two sets).  The
  // stores are fenced and the CTA synchronised before it releases the dependent grid.
  if (filter_cnt != nullptr && blockIdx.x == 0) {
    for (int i = tid; i < n_filter_cnt; i += MTHREADS) filter_cnt[i] = 0;
    __threadfence();
    __syncthreads();
  }
  grid_dep_launch();   // correlate is complete: the next step's filter may stream its rows under our tail
  FICOCO_PHASE(2, 1);
  // a step whose filter or correlate grid gave up has no valid index lists: write nothing
  if (tid == 0) dead = (*reinterpret_cast<const volatile unsigned*>(status) & STATUS_TIMEOUT) ? 1 : 0;
  // ---- file the entries that hit this CTA's rows ----------------------------------------------------
  for (int e0 = tid; e0 < n_ent; e0 += 4 * MTHREADS) {
    int t[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) t[i] = e0 + MTHREADS * i < n_ent ? e_tgt[d.ent0 + e0 + MTHREADS * i] : -1;
#pragma unroll
    for (int i = 0; i < 4; ++i)
      if (t[i] >= 0) {
        // (exact: for numbers below 2^13 the quotient of o + 1/2 stays away from the whole numbers)
        const int o = d.n_cls + t[i] - w.r0, r = __float2int_rd(((float)o + 0.5f) * inv_stride);
        if (o < 0 || r * stride != o || r >= w.nrows) continue;
        const int slot = atomicAdd(&cnt[r], 1), k = atomicAdd(&n_match, 1);
        if (k < MLIST) {
          m_e[k] = e0 + MTHREADS * i;
          m_rs[k] = (unsigned short)(r << 10 | (slot & 1023));
        }
      }
  }
  __syncthreads();
  const int total = n_match;
  const bool fits = total <= MLIST;
  bool rows_ok = true;
  if (dead) {
    mbar_wait(&row_bar, 0, wait_ns);             // no copy outlives the CTA
    return;
  }
  if (warp == 0) {
    // starts of the buckets, and of the groups (own row + sources) of the rows that have sources
    const int c0 = cnt[2 * lane], c1 = cnt[2 * lane + 1];
    const int g0 = c0 > 0 ? c0 + 1 : 0, g1 = c1 > 0 ? c1 + 1 : 0;
    int inc = (c0 + c1) << 16 | (g0 + g1);       // (both totals stay below 2^15 where they are used)
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int n = __shfl_up_sync(0xFFFFFFFFu, inc, o);
      if (lane >= o) inc += n;
    }
    const int exc = inc - ((c0 + c1) << 16 | (g0 + g1));
    beg[2 * lane] = exc >> 16; beg[2 * lane + 1] = (exc >> 16) + c0;
    gbeg[2 * lane] = exc & 0xFFFF; gbeg[2 * lane + 1] = (exc & 0xFFFF) + g0;
    if (lane == 31) { beg[MROWS] = inc >> 16; gbeg[MROWS] = inc & 0xFFFF; }
  }
  __syncthreads();
  int my_src[MLIST / MTHREADS];
  float my_w[MLIST / MTHREADS];
  if (fits && total > 0) {
#pragma unroll
    for (int q = 0; q < MLIST / MTHREADS; ++q) {
      const int i = tid + MTHREADS * q;
      if (i < total) {
        const int e = m_e[i], rs = m_rs[i];
        my_src[q] = S_idx[d.src0 + e / L];
        my_w[q] = e_w[d.ent0 + e];
        bucket[beg[rs >> 10] + (rs & 1023)] = e;
      }
    }
    if (tid < w.nrows && cnt[tid] > 0) el[gbeg[tid]] = make_uint2(__float_as_uint(1.0f), (uint32_t)tid << 16);
    __syncthreads();
    // the list of a row is ordered by entry, i.e. by discarded token
#pragma unroll
    for (int q = 0; q < MLIST / MTHREADS; ++q) {
      const int i = tid + MTHREADS * q;
      if (i < total) {
        const int e = m_e[i], r = m_rs[i] >> 10, b = beg[r], n = cnt[r];
        int rank = 0;
        for (int k = 0; k < n; ++k) rank += bucket[b + k] < e ? 1 : 0;
        el[gbeg[r] + 1 + rank] = make_uint2(__float_as_uint(my_w[q]), (uint32_t)r << 16 | (uint32_t)checked_index(my_src[q], d.np, status));
      }
    }
    __syncthreads();
  }
  FICOCO_PHASE(2, 2);
  rows_ok = mbar_wait(&row_bar, 0, wait_ns);
  if (!rows_ok) { atomicOr(status, STATUS_TIMEOUT); return; }
  // ---- rows without sources leave shared memory as they came ------------------------------------------
  if (warp == 0) {
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const int r = lane + 32 * j;
      if (r < w.nrows && cnt[r] == 0 && srow_s[r] >= 0)
        asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;"
                     ::"l"(out + (size_t)(d.out_row0 + w.r0 + r * stride) * D), "r"(smem_u32(stage + (size_t)r * row_bytes)), "r"(row_bytes)
                     : "memory");
    }
    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
  }
  FICOCO_PHASE(2, 3);
  // ---- rows with sources ------------------------------------------------------------------------------
  if (fits && total > 0) {
    const int n_el = gbeg[MROWS], n_all = n_el * ((nvec + 31) / 32);
    auto seg = [&](int k) { return (int)((long long)n_all * k / MWARPS); };
    const int p_hi = seg(warp + 1);
    float* piece = fold + warp * PW * 32 + lane;
    float acc[E], den = 0.f;
    int tail = -1;                               // where a group that goes on behind the segment began
    #pragma unroll 1
    for (int p = seg(warp); p < p_hi;) {
      const int sl = p / n_el, e0 = p - sl * n_el, r = (int)(el[e0].y >> 16);
      const int start = gbeg[r], end = start + 1 + cnt[r], e_hi = min(end, e0 + (p_hi - p));
      const int v = 32 * sl + lane;
      const bool on = v < nvec;
      const T* col = pbase + (size_t)(on ? v : 0) * E;
      int e = e0;
      if (e0 == start) {
        unpack(*reinterpret_cast<const uint4*>(stage + (size_t)r * row_bytes + (size_t)(on ? v : 0) * 16), acc, (const T*)nullptr);
        den = 1.0f;
        ++e;
      } else {
        den = 0.f;
#pragma unroll
        for (int q = 0; q < E; ++q) acc[q] = 0.f;
      }
      #pragma unroll 1
      for (; e < e_hi; e += MDEPTH) {
        uint4 u[MDEPTH];
#pragma unroll
        for (int j = 0; j < MDEPTH; ++j)         // (past the end: the last row again, weight 0)
          u[j] = ldg16(col + (size_t)(el[min(e + j, e_hi - 1)].y & 0xFFFFu) * D);
#pragma unroll
        for (int j = 0; j < MDEPTH; ++j) {
          const float a = e + j < e_hi ? __uint_as_float(el[e + j].x) : 0.f;
          float x[E];
          unpack(u[j], x, (const T*)nullptr);
          den += a;
#pragma unroll
          for (int q = 0; q < E; ++q) acc[q] = fmaf(a, x[q], acc[q]);
        }
      }
      if (e0 == start && e_hi < end) {           // stays in registers: it is the last piece of the segment
        tail = p;
        break;
      }
      if (e0 == start) {
        const float inv = 1.0f / den;
#pragma unroll
        for (int q = 0; q < E; ++q) acc[q] *= inv;
        if (on) st_stream16(reinterpret_cast<uint4*>(out + (size_t)(d.out_row0 + w.r0 + r * stride) * D) + v, pack(acc, (const T*)nullptr));
      } else {
#pragma unroll
        for (int q = 0; q < E; ++q) piece[q * 32] = acc[q];
        piece[E * 32] = den;
      }
      p += e_hi - e0;
    }
    FICOCO_PHASE(2, 4);
    __syncthreads();
    if (tail >= 0) {
      // add the pieces of the segments that the group reaches
      const int sl = tail / n_el, r = (int)(el[tail - sl * n_el].y >> 16), end = sl * n_el + gbeg[r] + 1 + cnt[r];
      const int v = 32 * sl + lane;
      for (int k = warp + 1; k < MWARPS && seg(k) < end; ++k) {
        if (seg(k) == seg(k + 1)) continue;
        const float* x = fold + k * PW * 32 + lane;
        den += x[E * 32];
#pragma unroll
        for (int q = 0; q < E; ++q) acc[q] += x[q * 32];
      }
      const float inv = 1.0f / den;
#pragma unroll
      for (int q = 0; q < E; ++q) acc[q] *= inv;
      if (v < nvec)
        st_stream16(reinterpret_cast<uint4*>(out + (size_t)(d.out_row0 + w.r0 + r * stride) * D) + v, pack(acc, (const T*)nullptr));
    }
  } else if (total > 0) {
    // too many sources for shared memory: walk the entries in order (ascending source)
    #pragma unroll 1
    for (int r = warp; r < w.nrows; r += MWARPS) {
      if (cnt[r] == 0) continue;
      const int tp = w.r0 + r * stride - d.n_cls;
      float wsum = 0.f;
      for (int e = 0; e < n_ent; ++e)
        if (e_tgt[d.ent0 + e] == tp) wsum += e_w[d.ent0 + e];
      const float den = 1.0f + wsum;
      for (int v = lane; v < nvec; v += 32) {
        float acc[E];
        unpack(*reinterpret_cast<const uint4*>(stage + (size_t)r * row_bytes + (size_t)v * 16), acc, (const T*)nullptr);
        for (int e = 0; e < n_ent; ++e) {
          if (e_tgt[d.ent0 + e] != tp) continue;
          const T* x0 = pbase + (size_t)checked_index(S_idx[d.src0 + e / L], d.np, status) * D;
          float f[E];
          unpack(ldg16(x0 + (size_t)v * E), f, (const T*)nullptr);
          const float a0 = e_w[d.ent0 + e];
#pragma unroll
          for (int q = 0; q < E; ++q) acc[q] = fmaf(a0, f[q], acc[q]);
        }
#pragma unroll
        for (int q = 0; q < E; ++q) acc[q] = acc[q] / den;
        st_stream16(reinterpret_cast<uint4*>(out + (size_t)(d.out_row0 + w.r0 + r * stride) * D) + v, pack(acc, (const T*)nullptr));
      }
    }
  }
  if (warp == 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");   // the stores have read shared memory
  FICOCO_PHASE(2, 5);
}

// Ablation "convergent correlation" (Sec. "Correlation-based Information Recycling": all discarded
// tokens merge into one additional token): the plain mean of an image's discarded rows, written
// behind the image's preserved rows.  One CTA per image; warp w sums the discarded rows w, w + 8,
// ... in ascending order, the eight partial sums are added in warp order (fp32, fixed order),
// scaled by 1 / N^S and rounded once.  Columns are processed in slabs of 128 vectors.
template <class T>
__global__ void __launch_bounds__(256) k_convergent_token(
    const T* __restrict__ tokens, int D, const ImgDesc* __restrict__ desc, const int* __restrict__ S_idx,
    T* __restrict__ out, const unsigned* __restrict__ status) {
  constexpr int E = VecTraits<T>::E;
  __shared__ float part[8][128 * E];
  const ImgDesc d = desc[blockIdx.x];
  grid_dep_wait();
  grid_dep_launch();
  if (!d.n_extra || (*status & STATUS_TIMEOUT)) return;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int nvec = D / E;
  const T* pbase = tokens + (size_t)(d.row0 + d.n_cls) * D;
  T* dst = out + (size_t)(d.out_row0 + d.n_cls + d.n_tgt) * D;
  const float inv = 1.0f / (float)d.n_src;
  #pragma unroll 1
  for (int c0 = 0; c0 < nvec; c0 += 128) {
    float acc[4][E];
#pragma unroll
    for (int k = 0; k < 4; ++k)
#pragma unroll
      for (int q = 0; q < E; ++q) acc[k][q] = 0.f;
    #pragma unroll 1
    for (int s = warp; s < d.n_src; s += 8) {
      const T* row = pbase + (size_t)S_idx[d.src0 + s] * D;
      uint4 u[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const int v = c0 + lane + 32 * k;
        u[k] = v < nvec ? ldg16(row + (size_t)v * E) : make_uint4(0, 0, 0, 0);
      }
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        float f[E];
        unpack(u[k], f, (const T*)nullptr);
#pragma unroll
        for (int q = 0; q < E; ++q) acc[k][q] += f[q];
      }
    }
#pragma unroll
    for (int k = 0; k < 4; ++k)
#pragma unroll
      for (int q = 0; q < E; ++q) part[warp][(lane + 32 * k) * E + q] = acc[k][q];
    __syncthreads();
    if (tid < 128 && c0 + tid < nvec) {
      float o[E];
#pragma unroll
      for (int q = 0; q < E; ++q) {
        float t = 0.f;
#pragma unroll
        for (int wv = 0; wv < 8; ++wv) t += part[wv][tid * E + q];
        o[q] = t * inv;
      }
      reinterpret_cast<uint4*>(dst)[c0 + tid] = pack(o, (const T*)nullptr);
    }
    __syncthreads();
  }
}

}  // namespace ficoco
