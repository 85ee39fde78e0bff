// Compress + compact (Eq. 2 and the last step of Algorithm 1 / 2).
#pragma once
#include "async_ops.cuh"
#include "common.cuh"

namespace ficoco {

constexpr int MTHREADS = 512;
constexpr int MWARPS = MTHREADS / 32;
constexpr int MROWS = 64;      // most output rows a CTA takes (a lane looks after two in the scan)
constexpr int MLIST = 1024;    // sources a CTA files in shared memory
constexpr int MDEPTH = 6;      // loads a lane has in flight; rows with more sources than that go first
constexpr int MUNITS = 640;    // (row with sources, part of it) units of a CTA
constexpr size_t MSTAGE_BYTES = 70 * 1024;   // input rows of a CTA's output rows kept in shared memory (two CTAs per SM)
static_assert(MSTAGE_BYTES / 128 + MROWS <= MUNITS, "every unit of a CTA needs an entry");

// A warp walks a row's list over 512 bytes of the row, a long list over 128: its lanes then form MGROUPS groups of
// eight, group k takes the sources k, k + MGROUPS, ... and the groups' sums are added at the end, which puts four times
// as many sources in flight.  Which of the two it is, and with it the order of the sum, follows the list and the
// hidden size alone (rows of 16 parts and more give every warp one as they are).
constexpr int MLONG = 12 * MDEPTH, MGROUPS = 4;
__device__ __forceinline__ bool list_long(int n, int row_bytes) { return n > MLONG && row_bytes <= 512 * (MWARPS - 1); }
__device__ __forceinline__ int list_parts(int n, int row_bytes) {
  return n == 0 ? 0 : list_long(n, row_bytes) ? (row_bytes + 127) / 128 : (row_bytes + 511) / 512;
}
// The groups' sums: (0 + 1) + (2 + 3), in every lane.
template <int E>
__device__ __forceinline__ void add_groups(float (&acc)[E], float& den) {
#pragma unroll
  for (int o = 32 / MGROUPS; o < 32; o <<= 1) {
    den += __shfl_xor_sync(0xFFFFFFFFu, den, o);
#pragma unroll
    for (int q = 0; q < E; ++q) acc[q] += __shfl_xor_sync(0xFFFFFFFFu, acc[q], o);
  }
}

// Byte `off` of row `own` (shared memory) plus its sources, 16 bytes per lane; lanes past the row's end idle.  LONG: as
// one of MGROUPS groups of lanes, the `first`-th; a function of its own, so that the usual lists keep their registers
// and instructions.
template <class T, bool LONG>
__device__ __forceinline__ void merge_list(const unsigned char* own, const uint2* list, int n, const unsigned char* image,
                                           unsigned char* dst, int off, int first, int row_bytes) {
  constexpr int E = VecTraits<T>::E, STEP = LONG ? MGROUPS : 1;
  const bool on = off < row_bytes;
  if (!on) off = 0;
  float acc[E], den = first == 0 ? 1.0f : 0.0f;
  unpack(*reinterpret_cast<const uint4*>(own + off), acc, (const T*)nullptr);
  if (LONG && first != 0) {
#pragma unroll
    for (int q = 0; q < E; ++q) acc[q] = 0.f;
  }
  image += off;
  #pragma unroll 1
  for (int e = first; e < n; e += MDEPTH * STEP) {
    uint4 u[MDEPTH];
#pragma unroll
    for (int j = 0; j < MDEPTH; ++j) u[j] = ldg16(image + list[min(e + j * STEP, n - 1)].y);   // (past the end: the last row)
#pragma unroll
    for (int j = 0; j < MDEPTH; ++j)
      if (e + j * STEP < n) {
        const float a = __uint_as_float(list[e + j * STEP].x);
        float x[E];
        unpack(u[j], x, (const T*)nullptr);
        den += a;
#pragma unroll
        for (int q = 0; q < E; ++q) acc[q] = fmaf(a, x[q], acc[q]);
      }
  }
  if (LONG) {
    __syncwarp();
    add_groups(acc, den);
  }
  const float inv = 1.0f / den;
#pragma unroll
  for (int q = 0; q < E; ++q) acc[q] *= inv;
  if (on && first == 0) st_stream16(reinterpret_cast<uint4*>(dst + off), pack(acc, (const T*)nullptr));
}
template <class T>
__device__ __noinline__ void merge_long_list(const unsigned char* own, const uint2* list, int n, const unsigned char* image,
                                             unsigned char* dst, int part, int lane, int row_bytes) {
  merge_list<T, true>(own, list, n, image, dst, (8 * part + (lane & 7)) * 16, lane >> 3, row_bytes);
}

// Compress + compact.  A CTA owns a few output rows of one image, the ones `stride` apart from its first: targets
// with many sources lie close together (neighbouring patches look alike), and dealt out like cards they load the
// CTAs of an image about alike (16 ragged images: the busiest CTA 38 us after its start, 14 in the median, when the
// rows of a CTA were consecutive).
//   rows    the input rows of its output rows are fetched into shared memory by bulk copies (TMA) that the last warp asks
//           for as soon as the correlate grid is complete, while the others file the entries (asked for under that grid's
//           tail, ahead of the wait, which nothing promises to be sound: relation map 42.0 us instead of 43.1, 16 FiCoCo-L
//           sequences 93.4 and 94.0, but 32 x 577 58.9 and 58.4, 256 x 577 318 and 315; by a warp that files as well:
//           0.7 and 5 us more on the last two);
//   file    the image's (source -> target) entries that hit its rows are filed into per-row lists in shared
//           memory, ordered by discarded token; no atomics touch floats; one pass over the entries, four loads in
//           flight per thread of the other 15 warps;
//   copies  a row that nothing is folded into leaves by a bulk store from shared memory: no thread touches it;
//   merge   out_j = (x_j + sum_{i in I_j} alpha_ij x_i) / (1 + sum alpha_ij), rounded once.  A unit is one row and
//           512 bytes of it, or 128 where its list is long; a warp adds the row's sources, several of them in flight,
//           and draws its next unit from a counter.  Rows with many sources go first.
// The order of every fp32 sum follows its row's list alone, whatever else the CTA owns: an output row is the same bits
// alone, in a batch of any size and in a group of a batch.
// What bounds it is the latency of its few dependent trips to L2; the split into 16 warps and the host's choice of
// one wave of CTAs where possible keep them few: 32 x 577 -> 289 rows of 1024 went from 25 us (a scan per 16 rows,
// copies and hub rows by warps, two waves of CTAs) to 18 us, 16 ragged images keeping 1/9 from 48 to 30 us.  (Equal
// segments of the sequence slices x sources per warp, with a list cut wherever a segment ended, are balanced better
// where a CTA has one long list, but the order of a sum then follows the rows per CTA and with them the batch: whole
// step 100.6 us instead of 102.9 for 16 ragged images, but 61.2 and 59.7 for 32 x 577, 138 and 135 for 8 x 2881, 112.7
// and 105.5 for 16 FiCoCo-L sequences, 53.4 and 44.5 with a relation map, as the pieces took a barrier, 18 KB of shared
// memory and another pass.  Long lists like the others: 16 ragged images of up to 4096 tokens 105.5 us instead of 99.6;
// long from 36 sources on: 100.4.  One function for both kinds, the number of groups a variable: 8 x 2881 tokens 138 us
// instead of 135.  8 or 10 sources in flight: the same.)
// If the CTA's rows receive more than MLIST sources in total, a slow in-order rescan is used.
template <class T>
__global__ void __launch_bounds__(MTHREADS, 2) k_merge_rows(
    const T* __restrict__ tokens, int D, const ImgDesc* __restrict__ desc,
    const WorkItem* __restrict__ work, const int* __restrict__ S_idx, const int* __restrict__ T_idx,
    const int* __restrict__ e_tgt, const float* __restrict__ e_w, T* __restrict__ out,
    unsigned* __restrict__ status, int* __restrict__ filter_cnt, int n_filter_cnt,
    unsigned long long wait_ns) {
  constexpr int E = VecTraits<T>::E;
  extern __shared__ __align__(128) unsigned char stage[];     // [rows][row bytes]
  __shared__ int cnt[MROWS], beg[MROWS], ubeg[MROWS], srow_s[MROWS];
  __shared__ int m_e[MLIST], bucket[MLIST];
  __shared__ unsigned short m_rs[MLIST];         // row << 10 | slot inside the row's bucket
  __shared__ uint2 el[MLIST];                    // weight, byte offset of the source row in its image
  __shared__ unsigned short unit[MUNITS];        // row << 8 | part
  __shared__ uint64_t row_bar;
  __shared__ int n_match, n_unit, next_unit, dead;
  FICOCO_PHASE_BEGIN(2);
  const WorkItem w = work[blockIdx.x];
  const ImgDesc d = desc[w.img];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int row_bytes = D * (int)sizeof(T);
  const int L = d.list_len;
  const int stride = w.aux;                      // row r of the CTA is output row w.r0 + r * stride of the image
  const float inv_stride = 1.0f / (float)stride;
  const int n_ent = d.n_src * L;
  if (tid < MROWS) cnt[tid] = 0;
  if (tid == 0) {
    n_match = 0;
    next_unit = MWARPS;
    mbar_init(&row_bar, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  grid_dep_wait();
  const T* pbase = tokens + (size_t)(d.row0 + d.n_cls) * D;
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
  if (warp == MWARPS - 1) {
    // input row of every output row (CLS / preserved token / trailing text row; -1: the additional token, which
    // k_convergent_token writes)
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
  // ---- file the entries that hit this CTA's rows ----------------------------------------------------
  constexpr int FILERS = MTHREADS - 32;
  for (int e0 = tid; e0 < n_ent && tid < FILERS; e0 += 4 * FILERS) {
    int t[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) t[i] = e0 + FILERS * i < n_ent ? e_tgt[d.ent0 + e0 + FILERS * i] : -1;
#pragma unroll
    for (int i = 0; i < 4; ++i)
      if (t[i] >= 0) {
        // (exact: for numbers below 2^13 the quotient of o + 1/2 stays away from the whole numbers)
        const int o = d.n_cls + t[i] - w.r0, r = __float2int_rd(((float)o + 0.5f) * inv_stride);
        if (o < 0 || r * stride != o || r >= w.nrows) continue;
        const int slot = atomicAdd(&cnt[r], 1), k = atomicAdd(&n_match, 1);
        if (k < MLIST) {
          m_e[k] = e0 + FILERS * i;
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
    // starts of the lists, and of the units of the rows that have sources: those with many first
    const int c0 = cnt[2 * lane], c1 = cnt[2 * lane + 1];
    const int u0 = list_parts(c0, row_bytes) << (c0 > MDEPTH ? 16 : 0);
    const int u1 = list_parts(c1, row_bytes) << (c1 > MDEPTH ? 16 : 0);
    int ci = c0 + c1, ui = u0 + u1;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int nc = __shfl_up_sync(0xFFFFFFFFu, ci, o), nu = __shfl_up_sync(0xFFFFFFFFu, ui, o);
      if (lane >= o) { ci += nc; ui += nu; }
    }
    const int all = __shfl_sync(0xFFFFFFFFu, ui, 31), many = all >> 16;
    const int ux = ui - u0 - u1, uy = ui - u1;
    beg[2 * lane] = ci - c0 - c1; beg[2 * lane + 1] = ci - c1;
    ubeg[2 * lane] = c0 > MDEPTH ? ux >> 16 : many + (ux & 0xFFFF);
    ubeg[2 * lane + 1] = c1 > MDEPTH ? uy >> 16 : many + (uy & 0xFFFF);
    if (lane == 0) n_unit = many + (all & 0xFFFF);
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
    for (int r = warp; r < w.nrows; r += MWARPS)
      for (int k = lane; k < list_parts(cnt[r], row_bytes); k += 32) unit[ubeg[r] + k] = (unsigned short)(r << 8 | k);
    __syncthreads();
    // the list of a row is ordered by entry, i.e. by discarded token
#pragma unroll
    for (int q = 0; q < MLIST / MTHREADS; ++q) {
      const int i = tid + MTHREADS * q;
      if (i < total) {
        const int e = m_e[i], r = m_rs[i] >> 10, b = beg[r], n = cnt[r];
        int rank = 0;
        for (int k = 0; k < n; ++k) rank += bucket[b + k] < e ? 1 : 0;
        el[b + rank] = make_uint2(__float_as_uint(my_w[q]), (uint32_t)checked_index(my_src[q], d.np, status) * (uint32_t)row_bytes);
      }
    }
    __syncthreads();
  }
  FICOCO_PHASE(2, 2);
  rows_ok = mbar_wait(&row_bar, 0, wait_ns);
  if (!rows_ok) {
    atomicOr(status, STATUS_TIMEOUT);
    mbar_wait(&row_bar, 0, wait_ns);             // (as above)
    return;
  }
  // ---- rows without sources leave shared memory as they came ------------------------------------------
  if (warp == 0) {
    const uint64_t policy = l2_evict_first();
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const int r = lane + 32 * j;
      if (r < w.nrows && cnt[r] == 0 && srow_s[r] >= 0)
        bulk_store_streaming(out + (size_t)(d.out_row0 + w.r0 + r * stride) * D, stage + (size_t)r * row_bytes,
                             (uint32_t)row_bytes, policy);
    }
    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
  }
  FICOCO_PHASE(2, 3);
  // ---- rows with sources ------------------------------------------------------------------------------
  if (fits && total > 0) {
    #pragma unroll 1
    for (int u = warp; u < n_unit;) {
      const int r = unit[u] >> 8, part = unit[u] & 255;
      const unsigned char* own = stage + (size_t)r * row_bytes;
      const unsigned char* image = reinterpret_cast<const unsigned char*>(pbase);
      unsigned char* dst = reinterpret_cast<unsigned char*>(out + (size_t)(d.out_row0 + w.r0 + r * stride) * D);
      if (list_long(cnt[r], row_bytes)) merge_long_list<T>(own, el + beg[r], cnt[r], image, dst, part, lane, row_bytes);
      else merge_list<T, false>(own, el + beg[r], cnt[r], image, dst, (32 * part + lane) * 16, 0, row_bytes);
      if (lane == 0) u = atomicAdd(&next_unit, 1);
      u = __shfl_sync(0xFFFFFFFFu, u, 0);
    }
    FICOCO_PHASE(2, 4);
  } else if (total > 0) {
    // too many sources for shared memory: walk the entries in order (ascending source).  Sums and quotient as in
    // merge_list, because whether a CTA comes here follows its other rows.
    #pragma unroll 1
    for (int r = warp; r < w.nrows; r += MWARPS) {
      const int n = cnt[r], tp = w.r0 + r * stride - d.n_cls;
      const bool is_long = list_long(n, row_bytes);
      const int width = is_long ? 32 / MGROUPS : 32, first = lane / width;
      #pragma unroll 1
      for (int part = 0; part < list_parts(n, row_bytes); ++part) {
        int off = (part * width + (lane & (width - 1))) * 16;
        const bool on = off < row_bytes;
        if (!on) off = 0;
        float acc[E], den = first == 0 ? 1.0f : 0.0f;
        unpack(*reinterpret_cast<const uint4*>(stage + (size_t)r * row_bytes + off), acc, (const T*)nullptr);
        if (first != 0) {
#pragma unroll
          for (int q = 0; q < E; ++q) acc[q] = 0.f;
        }
        int k = 0;
        for (int e = 0; e < n_ent; ++e) {
          if (e_tgt[d.ent0 + e] != tp) continue;
          if (is_long && k++ % MGROUPS != first) continue;
          const T* x0 = pbase + (size_t)checked_index(S_idx[d.src0 + e / L], d.np, status) * D;
          float f[E];
          unpack(ldg16(reinterpret_cast<const unsigned char*>(x0) + off), f, (const T*)nullptr);
          const float a0 = e_w[d.ent0 + e];
          den += a0;
#pragma unroll
          for (int q = 0; q < E; ++q) acc[q] = fmaf(a0, f[q], acc[q]);
        }
        __syncwarp();
        if (is_long) add_groups(acc, den);
        const float inv = 1.0f / den;
#pragma unroll
        for (int q = 0; q < E; ++q) acc[q] *= inv;
        if (on && first == 0)
          st_stream16(reinterpret_cast<uint4*>(reinterpret_cast<unsigned char*>(out + (size_t)(d.out_row0 + w.r0 + r * stride) * D) + off),
                      pack(acc, (const T*)nullptr));
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
