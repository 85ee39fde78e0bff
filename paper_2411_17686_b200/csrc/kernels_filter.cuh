// Filter stage (Eq. 1, local penalty, top-N^S selection).
//
// Every kernel of a step is launched under the tail of the grid before it (programmatic stream serialization): it
// reads its plan entries, which are constants, then waits for that grid to be complete and only then lets the next
// one in.  All else that it reads or writes it touches behind its own wait: nothing promises a grid that what lies before its
// predecessor is visible to it any earlier.
#pragma once
#include <math_constants.h>
#include <type_traits>
#include "async_ops.cuh"
#include "common.cuh"

namespace ficoco {

// ---------------------------------------------------------------------------------------
// Row norms.  One warp per vision token: rn_i = 1 / ||x_i||.  Used alone when the hidden
// size is too wide for the fused kernel below.
// ---------------------------------------------------------------------------------------
template <class T>
__global__ void __launch_bounds__(256) k_rownorm(const T* __restrict__ tokens, int D,
                                                 const ImgDesc* __restrict__ desc,
                                                 const WorkItem* __restrict__ work,
                                                 float* __restrict__ rn) {
  constexpr int E = VecTraits<T>::E;
  const WorkItem w = work[blockIdx.x];
  const ImgDesc d = desc[w.img];
  grid_dep_wait();
  grid_dep_launch();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int nvec = D / E;
  for (int r = warp; r < w.nrows; r += 8) {
    const T* row = tokens + (size_t)(d.row0 + d.n_cls + w.r0 + r) * D;
    float ss = 0.f;
    for (int v0 = lane; v0 < nvec; v0 += 32 * 8) {     // eight 16-byte loads in flight per lane
      uint4 u[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const int v = v0 + 32 * k;
        u[k] = v < nvec ? ldg16(row + (size_t)v * E) : make_uint4(0, 0, 0, 0);
      }
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        float f[E];
        unpack(u[k], f, (const T*)nullptr);
#pragma unroll
        for (int e = 0; e < E; ++e) ss = fmaf(f[e], f[e], ss);
      }
    }
    ss = warp_sum(ss);
    if (lane == 0) rn[d.patch0 + w.r0 + r] = ss > 0.f ? 1.0f / sqrtf(ss) : 0.f;
  }
}

// ---------------------------------------------------------------------------------------
// Column sums of the normalised tokens: partial[chunk][d] = sum_{i in chunk} rn_i x_id.
// The row mean of the cosine relation is x_hat_i . (1/N) sum_j x_hat_j, so this vector is
// all the first term of Eq. 1 needs.  One CTA per row chunk; a warp owns whole rows, each
// lane the 16-byte vectors lane, lane+32, ... of the column slab [c0, c0 + VPL*32*E).
// FUSED: the CTA also computes rn (requires the slab to cover the full row).
// Warps are folded into shared memory one after the other, so the result does not depend
// on scheduling.
// ---------------------------------------------------------------------------------------
template <class T, int VPL, bool FUSED>
__global__ void __launch_bounds__(256) k_colsum(const T* __restrict__ tokens, int D,
                                                const ImgDesc* __restrict__ desc,
                                                const WorkItem* __restrict__ work,
                                                float* __restrict__ rn,
                                                float* __restrict__ partial) {
  constexpr int E = VecTraits<T>::E;
  extern __shared__ __align__(16) float sm_acc[];  // [4][VPL * 32 * E]
  const WorkItem w = work[blockIdx.x];
  const ImgDesc d = desc[w.img];
  grid_dep_wait();
  grid_dep_launch();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int slab = blockIdx.y;
  const int c0 = slab * (VPL * 32 * E);
  const int nvec = (min(D - c0, VPL * 32 * E)) / E;

  float acc[VPL][E];
#pragma unroll
  for (int k = 0; k < VPL; ++k)
#pragma unroll
    for (int e = 0; e < E; ++e) acc[k][e] = 0.f;

  const T* base = tokens + (size_t)(d.row0 + d.n_cls + w.r0) * D + c0;
  float* rn_out = rn + d.patch0 + w.r0;

  #pragma unroll 1
  for (int r = warp; r < w.nrows; r += 16) {
    const int r2 = r + 8;
    const bool has2 = r2 < w.nrows;
    uint4 u[VPL], u2[VPL];
#pragma unroll
    for (int k = 0; k < VPL; ++k) {
      const int v = lane + 32 * k;
      u[k] = (v < nvec) ? ldg16(base + (size_t)r * D + (size_t)v * E) : make_uint4(0, 0, 0, 0);
    }
#pragma unroll
    for (int k = 0; k < VPL; ++k) {
      const int v = lane + 32 * k;
      u2[k] = (has2 && v < nvec) ? ldg16(base + (size_t)r2 * D + (size_t)v * E) : make_uint4(0, 0, 0, 0);
    }
    float s1, s2;
    if (FUSED) {
      float ss = 0.f, ss2 = 0.f;
#pragma unroll
      for (int k = 0; k < VPL; ++k) {
        float f[E];
        unpack(u[k], f, (const T*)nullptr);
#pragma unroll
        for (int e = 0; e < E; ++e) ss = fmaf(f[e], f[e], ss);
        unpack(u2[k], f, (const T*)nullptr);
#pragma unroll
        for (int e = 0; e < E; ++e) ss2 = fmaf(f[e], f[e], ss2);
      }
      ss = warp_sum(ss);
      ss2 = warp_sum(ss2);
      s1 = ss > 0.f ? 1.0f / sqrtf(ss) : 0.f;
      s2 = ss2 > 0.f ? 1.0f / sqrtf(ss2) : 0.f;
      if (lane == 0) {
        rn_out[r] = s1;
        if (has2) rn_out[r2] = s2;
      }
    } else {
      s1 = rn_out[r];
      s2 = has2 ? rn_out[r2] : 0.f;
    }
#pragma unroll
    for (int k = 0; k < VPL; ++k) {
      float f[E];
      unpack(u[k], f, (const T*)nullptr);
#pragma unroll
      for (int e = 0; e < E; ++e) acc[k][e] = fmaf(f[e], s1, acc[k][e]);
      unpack(u2[k], f, (const T*)nullptr);
#pragma unroll
      for (int e = 0; e < E; ++e) acc[k][e] = fmaf(f[e], s2, acc[k][e]);
    }
  }

  // fold the 8 warps in a fixed order: warps 0-3 store, warps 4-7 add to the row of warp - 4, then four rows per column
  // (one warp after the other took eight barriers: 256 x 577 tokens of 1024 in chunks of 64 rows 103 us, now 72)
  constexpr int WIDTH = VPL * 32 * E;
#pragma unroll
  for (int half = 0; half < 2; ++half) {
    if ((warp >> 2) == half) {
#pragma unroll
      for (int k = 0; k < VPL; ++k) {
        float4* dst = reinterpret_cast<float4*>(sm_acc + (size_t)(warp & 3) * WIDTH + (size_t)(lane + 32 * k) * E);
#pragma unroll
        for (int q = 0; q < E / 4; ++q) {
          float4 x = half ? dst[q] : make_float4(0.f, 0.f, 0.f, 0.f);
          x.x += acc[k][4 * q]; x.y += acc[k][4 * q + 1]; x.z += acc[k][4 * q + 2]; x.w += acc[k][4 * q + 3];
          dst[q] = x;
        }
      }
    }
    __syncthreads();
  }
  float* out = partial + (size_t)(d.chunk0 + w.aux) * D + c0;
  for (int i = threadIdx.x; i < nvec * E; i += 256)
    out[i] = (sm_acc[i] + sm_acc[WIDTH + i]) + (sm_acc[2 * WIDTH + i] + sm_acc[3 * WIDTH + i]);
}

// ---------------------------------------------------------------------------------------
// Eq. 1 (and the FiCoCo-L score): s_i = cA * v_i - (1 - cA) * a_i with
//   v_i = rn_i * (x_i . msum) / Np,   msum = the image's column sums (k_msum),
//   a_i = (1/H) sum_h attn[h, i]      (FiCoCo-L: H = M rows of the head-mean block t).
// One CTA per row chunk, one warp per token for the dot product.
// ---------------------------------------------------------------------------------------
// Column sums of every image: msum[b, c] = sum over the image's row chunks, in chunk order.
__global__ void __launch_bounds__(256) k_msum(int D, const ImgDesc* __restrict__ desc,
                                              const float* __restrict__ partial, float* __restrict__ msum) {
  const ImgDesc d = desc[blockIdx.x];
  grid_dep_wait();
  grid_dep_launch();
  const int c = blockIdx.y * 256 + threadIdx.x;
  if (c >= D) return;
  float s = 0.f;
  const float* q0 = partial + (size_t)d.chunk0 * D + c;
  auto add = [&](auto n) {                         // this many chunks' loads in flight
    constexpr int N = decltype(n)::value;
    for (int k0 = 0; k0 < d.n_chunks; k0 += N) {
      float q[N];
#pragma unroll
      for (int k = 0; k < N; ++k) q[k] = k0 + k < d.n_chunks ? q0[(size_t)(k0 + k) * D] : 0.f;
#pragma unroll
      for (int k = 0; k < N; ++k) s += q[k];
    }
  };
  // (a sequence's 18 chunks as one trip: 16 sequences of 4096 take 4.4 us, 6.0 eight at a time; 256 images of 4 chunks
  // 2 us more with 24 at a time)
  if (d.n_chunks <= 8) add(std::integral_constant<int, 8>());
  else add(std::integral_constant<int, 24>());
  msum[(size_t)blockIdx.x * D + c] = s;
}

// Mean over the H attention rows of the chunk's tokens, a_i = (1/H) sum_h attn[h, i], by all 256 threads:
// warp q adds rows q, q + 8, ... for 32 tokens per lane trip (eight loads in flight), the eight partial sums
// of a token are then added in warp order.  `part` holds 8 * nrows floats.
__device__ __forceinline__ void attn_mean_rows(const float* __restrict__ a0, int H, int np, int nrows,
                                               float* part, int tid) {
  const int lane = tid & 31, warp = tid >> 5;
  for (int r = lane; r < nrows; r += 32) {
    float s = 0.f;
    for (int h0 = warp; h0 < H; h0 += 64) {
      float q[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) q[j] = h0 + 8 * j < H ? __ldg(a0 + (size_t)(h0 + 8 * j) * np + r) : 0.f;
#pragma unroll
      for (int j = 0; j < 8; ++j) s += q[j];
    }
    part[warp * nrows + r] = s;
  }
}

// Rows of up to 256 vectors.  Bound by the read of the tokens, so a warp keeps two rows in flight while it works on
// the two before them: the mean direction sits in registers (a lane owns the same columns of every row), and nothing
// else is fetched inside the loop.  The chunks are taken last to first: a batch larger than the L2 cache leaves its
// last images there when the column sums are done.  (One row per warp at a time, the direction in shared memory and
// the norm read behind every dot product: 256 x 577 rows of 1024, 302 MB, took 139 us, now 63.)
template <class T, int VPL>
__global__ void __launch_bounds__(256, VPL <= 5 ? 2 : 1) k_score_rows(const T* __restrict__ tokens, int D,
                                                                      const ImgDesc* __restrict__ desc,
                                                                      const WorkItem* __restrict__ work,
                                                                      const float* __restrict__ rn,
                                                                      const float* __restrict__ msum_all,
                                                                      const float* __restrict__ attn, int H, float cA,
                                                                      float* __restrict__ s_raw) {
  constexpr int E = VecTraits<T>::E;
  extern __shared__ float vrow[];  // v[nrows], attention partial sums [8][nrows]
  const WorkItem w = work[gridDim.x - 1 - blockIdx.x];
  const ImgDesc d = desc[w.img];
  grid_dep_wait();
  grid_dep_launch();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int nvec = D / E;
  const T* base = tokens + (size_t)(d.row0 + d.n_cls + w.r0) * D;
  uint4 next[2][VPL];
  auto fetch = [&](int r) {
#pragma unroll
    for (int j = 0; j < 2; ++j)
#pragma unroll
      for (int k = 0; k < VPL; ++k) {
        const int v = lane + 32 * k;
        next[j][k] = (r + 8 * j < w.nrows && v < nvec) ? ldg16(base + (size_t)(r + 8 * j) * D + (size_t)v * E)
                                                       : make_uint4(0, 0, 0, 0);
      }
  };
  fetch(warp);
  float m[VPL][E];
#pragma unroll
  for (int k = 0; k < VPL; ++k) {
    const int v = lane + 32 * k;
#pragma unroll
    for (int e = 0; e < E; e += 4) {
      const float4 q = v < nvec ? __ldcg(reinterpret_cast<const float4*>(msum_all + (size_t)w.img * D + (size_t)v * E + e))
                                : make_float4(0.f, 0.f, 0.f, 0.f);
      m[k][e] = q.x; m[k][e + 1] = q.y; m[k][e + 2] = q.z; m[k][e + 3] = q.w;
    }
  }
  float* part = vrow + w.nrows;
  attn_mean_rows(attn + d.attn0 + w.r0, H, d.np, w.nrows, part, threadIdx.x);
  #pragma unroll 1
  for (int r = warp; r < w.nrows; r += 16) {
    uint4 u[2][VPL];
#pragma unroll
    for (int j = 0; j < 2; ++j)
#pragma unroll
      for (int k = 0; k < VPL; ++k) u[j][k] = next[j][k];
    fetch(r + 16);
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      float dot = 0.f;
#pragma unroll
      for (int k = 0; k < VPL; ++k) {
        float f[E];
        unpack(u[j][k], f, (const T*)nullptr);
#pragma unroll
        for (int e = 0; e < E; ++e) dot = fmaf(f[e], m[k][e], dot);
      }
      dot = warp_sum(dot);
      if (lane == 0 && r + 8 * j < w.nrows) vrow[r + 8 * j] = dot;
    }
  }
  const float inv_np = 1.0f / (float)d.np, inv_h = 1.0f / (float)H;
  const float rn_first = threadIdx.x < w.nrows ? __ldcg(rn + d.patch0 + w.r0 + threadIdx.x) : 0.f;
  __syncthreads();
  for (int r = threadIdx.x; r < w.nrows; r += 256) {
    float s = 0.f;
#pragma unroll
    for (int q = 0; q < 8; ++q) s += part[q * w.nrows + r];
    const float k = r == threadIdx.x ? rn_first : __ldcg(rn + d.patch0 + w.r0 + r);
    s_raw[d.patch0 + w.r0 + r] = cA * (vrow[r] * k * inv_np) - (1.0f - cA) * (s * inv_h);
  }
}

template <class T>
__global__ void __launch_bounds__(256) k_score(const T* __restrict__ tokens, int D,
                                               const ImgDesc* __restrict__ desc,
                                               const WorkItem* __restrict__ work,
                                               const float* __restrict__ rn,
                                               const float* __restrict__ msum_all,
                                               const float* __restrict__ attn, int H, float cA,
                                               float* __restrict__ s_raw) {
  constexpr int E = VecTraits<T>::E;
  extern __shared__ float sm[];  // msum[D], v[nrows], attention partial sums [8][nrows]
  const WorkItem w = work[blockIdx.x];
  const ImgDesc d = desc[w.img];
  grid_dep_wait();
  grid_dep_launch();
  float* msum = sm;
  float* vrow = sm + D;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;

  for (int c = threadIdx.x; c < D; c += 256) msum[c] = msum_all[(size_t)w.img * D + c];
  __syncthreads();

  const int nvec = D / E;
  const float inv_np = 1.0f / (float)d.np;
  for (int r = warp; r < w.nrows; r += 8) {
    const T* row = tokens + (size_t)(d.row0 + d.n_cls + w.r0 + r) * D;
    float dot = 0.f;
    for (int v0 = lane; v0 < nvec; v0 += 32 * 8) {     // eight 16-byte loads in flight per lane
      uint4 u[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const int v = v0 + 32 * k;
        u[k] = v < nvec ? ldg16(row + (size_t)v * E) : make_uint4(0, 0, 0, 0);
      }
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const int v = v0 + 32 * k;
        if (v < nvec) {
          float f[E];
          unpack(u[k], f, (const T*)nullptr);
          const float* m = msum + (size_t)v * E;
#pragma unroll
          for (int e = 0; e < E; ++e) dot = fmaf(f[e], m[e], dot);
        }
      }
    }
    dot = warp_sum(dot);
    if (lane == 0) vrow[r] = dot * rn[d.patch0 + w.r0 + r] * inv_np;
  }
  __syncthreads();

  const float inv_h = 1.0f / (float)H;
  float* part = vrow + w.nrows;
  attn_mean_rows(attn + d.attn0 + w.r0, H, d.np, w.nrows, part, threadIdx.x);
  __syncthreads();
  for (int r = threadIdx.x; r < w.nrows; r += 256) {
    float s = 0.f;
#pragma unroll
    for (int q = 0; q < 8; ++q) s += part[q * w.nrows + r];
    s_raw[d.patch0 + w.r0 + r] = cA * vrow[r] - (1.0f - cA) * (s * inv_h);
  }
}

// ---------------------------------------------------------------------------------------
// FiCoCo-L: head mean of the text->vision attention, t[b, k, i] = (1/H) sum_h A[b, h, k, i].
// The M * N values of a sequence are cut into parts, one CTA per part; heads are added in order, so many at a time that the
// loads are in flight together.  Where everything is aligned a thread takes four values, else one (12 sequences of 722 + 19
// tokens of 2048 57.5 us, four single values 61.5).  In a grid of its own (narrow rows) small CTAs of few registers start
// beside what the grid before still holds: 128 threads and eight heads; whole step, 35 sequences of 214 + 80 of 1024 50.7 us
// (256 threads and 16 heads 53.3), 32 of 1000 + 100 of 2048 251.6 (257.2).  Beside the column sums, whose registers are taken
// anyway, 256 threads and 16 heads.
// ---------------------------------------------------------------------------------------
__host__ __device__ __forceinline__ int head_mean_values(const float* attn, const float* t, int MN) {   // of a thread
  return ((MN & 3) == 0 && (reinterpret_cast<uintptr_t>(attn) & 15) == 0 && (reinterpret_cast<uintptr_t>(t) & 15) == 0) ? 4 : 1;
}
// CTAs of `threads` threads for a sequence
__host__ __device__ __forceinline__ int head_mean_parts(int MN, int values, int threads) { return (MN + values * threads - 1) / (values * threads); }

template <int NT, int HF>
__device__ __forceinline__ void head_mean_part(const float* __restrict__ attn, int H, int MN, int part,
                                               float* __restrict__ t) {
  const int values = head_mean_values(attn, t, MN), per_seq = head_mean_parts(MN, values, NT), b = part / per_seq;
  const int i = (part % per_seq * NT + (int)threadIdx.x) * values;
  const float inv_h = 1.0f / (float)H;
  const float* src = attn + (size_t)b * H * MN + i;
  float* dst = t + (size_t)b * MN + i;
  if (i >= MN) return;
  if (values == 4) {
    float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int h0 = 0; h0 < H; h0 += HF) {
      float4 a[HF];
#pragma unroll
      for (int q = 0; q < HF; ++q)
        a[q] = h0 + q < H ? __ldg(reinterpret_cast<const float4*>(src + (size_t)(h0 + q) * MN))
                          : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int q = 0; q < HF; ++q) { s.x += a[q].x; s.y += a[q].y; s.z += a[q].z; s.w += a[q].w; }
    }
    *reinterpret_cast<float4*>(dst) = make_float4(s.x * inv_h, s.y * inv_h, s.z * inv_h, s.w * inv_h);
    return;
  }
  float s = 0.f;
  for (int h0 = 0; h0 < H; h0 += 16) {
    float a[16];
#pragma unroll
    for (int q = 0; q < 16; ++q) a[q] = ld_now(src + (size_t)min(h0 + q, H - 1) * MN);
#pragma unroll
    for (int q = 0; q < 16; ++q) s += h0 + q < H ? a[q] : 0.f;
  }
  *dst = s * inv_h;
}

constexpr int HM_THREADS = 128;
__global__ void __launch_bounds__(HM_THREADS) k_head_mean(const float* __restrict__ attn, int H, int MN, float* __restrict__ t) {
  grid_dep_wait();
  grid_dep_launch();
  head_mean_part<HM_THREADS, 8>(attn, H, MN, blockIdx.x, t);
}

// ---------------------------------------------------------------------------------------
// Wide rows (more than 256 16-byte vectors: hidden 4096 in bf16): a row no longer fits one
// warp's registers, so the CTA's 256 threads own the row's column vectors (NV each) and rows
// go through in batches of RB.  A per-row sum is folded lane -> warp -> the 8 warps in order.
//   k_colsum_wide: row norms and the chunk's column sums of the normalised rows in one read;
//                  every thread keeps the sums of its own columns, so there is no fold at the end.  FiCoCo-L's head mean,
//                  which shares nothing with them, is taken by other CTAs of the same grid, so that the two reads of
//                  memory run into one another (behind one another: 16 sequences of 4096 92.1 us, one 50.4, eight of 3584
//                  74.9).  As two grids, the second without a wait ahead of its reads, it was 90.9, 45.1 and 68.4, but a
//                  grid is promised to see what the grid it waits for wrote, not what grids before that one did.
//   k_score_wide:  Eq. 1 with the image's column sums held in registers; a batch's rows are asked for under the barrier of
//                  the batch before, the first ones and the attention ahead of everything (16 sequences of 4096: with
//                  the overlap of head mean and column sums the step 101.3 -> 93.1 us, one sequence 49.4 -> 45.0)
// ---------------------------------------------------------------------------------------
template <class T, int NV, int RB>
__device__ __forceinline__ void wide_load(const T* __restrict__ base, int D, int nvec, int r0, int nrows, int tid,
                                          uint4 (&u)[RB][NV]) {
  constexpr int E = VecTraits<T>::E;
#pragma unroll
  for (int j = 0; j < RB; ++j)
#pragma unroll
    for (int k = 0; k < NV; ++k) {
      const int v = tid + 256 * k;
      u[j][k] = (r0 + j < nrows && v < nvec) ? ld16_now(base + (size_t)(r0 + j) * D + (size_t)v * E) : make_uint4(0, 0, 0, 0);
    }
}

__device__ __forceinline__ float fold8(const float* r) {
  const float4 a = *reinterpret_cast<const float4*>(r), b = *reinterpret_cast<const float4*>(r + 4);
  return ((((((a.x + a.y) + a.z) + a.w) + b.x) + b.y) + b.z) + b.w;
}

template <class T, int NV, int RB>
__global__ void __launch_bounds__(256, 2) k_colsum_wide(const T* __restrict__ tokens, int D,
                                                     const ImgDesc* __restrict__ desc,
                                                     const WorkItem* __restrict__ work,
                                                     float* __restrict__ rn_out, float* __restrict__ partial,
                                                     int n_rows, const float* __restrict__ t2v, int H, int MN,
                                                     float* __restrict__ t) {
  constexpr int E = VecTraits<T>::E;
  __shared__ __align__(16) float red[2][RB][8];
  // The CTAs behind the first n_rows take the head mean: what takes longest comes first (head mean first: 10 sequences of 4096
  // 74.0 instead of 70.2 us, 32 164.9 and 161.8, eight of 3584 70.9 and 67.5; only 16 of 4096, whose rows fill the GPU once,
  // the other way round, 89.0 and 91.7).
  const bool rows_here = (int)blockIdx.x < n_rows;
  const WorkItem w = work[rows_here ? blockIdx.x : 0];
  const ImgDesc d = desc[w.img];
  grid_dep_wait();
  grid_dep_launch();
  if (!rows_here) {
    head_mean_part<256, 16>(t2v, H, MN, (int)blockIdx.x - n_rows, t);
    return;
  }
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int nvec = D / E;
  const T* base = tokens + (size_t)(d.row0 + d.n_cls + w.r0) * D;
  float* rn = rn_out + d.patch0 + w.r0;
  float acc[NV][E];
#pragma unroll
  for (int k = 0; k < NV; ++k)
#pragma unroll
    for (int e = 0; e < E; ++e) acc[k][e] = 0.f;

  int par = 0;
  for (int r0 = 0; r0 < w.nrows; r0 += RB, par ^= 1) {
    uint4 u[RB][NV];
    wide_load<T, NV, RB>(base, D, nvec, r0, w.nrows, tid, u);
#pragma unroll
    for (int j = 0; j < RB; ++j) {
      float ss = 0.f;
#pragma unroll
      for (int k = 0; k < NV; ++k) {
        float f[E];
        unpack(u[j][k], f, (const T*)nullptr);
#pragma unroll
        for (int e = 0; e < E; ++e) ss = fmaf(f[e], f[e], ss);
      }
      ss = warp_sum(ss);
      if (lane == 0) red[par][j][warp] = ss;
    }
    __syncthreads();   // one barrier per batch: the next batch writes the other half of `red`
#pragma unroll
    for (int j = 0; j < RB; ++j) {
      const float tot = fold8(red[par][j]);
      const float sc = tot > 0.f ? 1.0f / sqrtf(tot) : 0.f;
      if (tid == j && r0 + j < w.nrows) rn[r0 + j] = sc;
#pragma unroll
      for (int k = 0; k < NV; ++k) {
        float f[E];
        // unpack again rather than keep the batch's converted values in registers across the barrier
        asm volatile("" : "+r"(u[j][k].x), "+r"(u[j][k].y), "+r"(u[j][k].z), "+r"(u[j][k].w));
        unpack(u[j][k], f, (const T*)nullptr);
#pragma unroll
        for (int e = 0; e < E; ++e) acc[k][e] = fmaf(f[e], sc, acc[k][e]);
      }
    }
  }
  float* out = partial + (size_t)(d.chunk0 + w.aux) * D;
#pragma unroll
  for (int k = 0; k < NV; ++k) {
    const int v = tid + 256 * k;
    if (v < nvec) {
#pragma unroll
      for (int e = 0; e < E; e += 4)
        *reinterpret_cast<float4*>(out + (size_t)v * E + e) = make_float4(acc[k][e], acc[k][e + 1], acc[k][e + 2], acc[k][e + 3]);
    }
  }
}

template <class T, int NV, int RB>
__global__ void __launch_bounds__(256) k_score_wide(const T* __restrict__ tokens, int D,
                                                    const ImgDesc* __restrict__ desc,
                                                    const WorkItem* __restrict__ work,
                                                    const float* __restrict__ rn,
                                                    const float* __restrict__ msum_all,
                                                    const float* __restrict__ attn, int H, float cA,
                                                    float* __restrict__ s_raw) {
  constexpr int E = VecTraits<T>::E;
  extern __shared__ float vrow[];  // v[nrows], attention partial sums [8][nrows]
  __shared__ __align__(16) float red[2][RB][8];
  const WorkItem w = work[blockIdx.x];
  const ImgDesc d = desc[w.img];
  grid_dep_wait();
  grid_dep_launch();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int nvec = D / E;
  const T* base = tokens + (size_t)(d.row0 + d.n_cls + w.r0) * D;
  // the first rows are in flight under everything up to the loop, the next ones under each barrier
  uint4 u[RB][NV];
  wide_load<T, NV, RB>(base, D, nvec, 0, w.nrows, tid, u);
  float m[NV][E];
#pragma unroll
  for (int k = 0; k < NV; ++k) {
    const int v = tid + 256 * k;
#pragma unroll
    for (int e = 0; e < E; e += 4) {
      const float4 q = v < nvec ? __ldcg(reinterpret_cast<const float4*>(msum_all + (size_t)w.img * D + (size_t)v * E + e))
                                : make_float4(0.f, 0.f, 0.f, 0.f);
      m[k][e] = q.x; m[k][e + 1] = q.y; m[k][e + 2] = q.z; m[k][e + 3] = q.w;
    }
  }
  const float inv_np = 1.0f / (float)d.np;
  float* part = vrow + w.nrows;
  attn_mean_rows(attn + d.attn0 + w.r0, H, d.np, w.nrows, part, tid);
  int par = 0;
  for (int r0 = 0; r0 < w.nrows; r0 += RB, par ^= 1) {
#pragma unroll
    for (int j = 0; j < RB; ++j) {
      float dot = 0.f;
#pragma unroll
      for (int k = 0; k < NV; ++k) {
        float f[E];
        unpack(u[j][k], f, (const T*)nullptr);
#pragma unroll
        for (int e = 0; e < E; ++e) dot = fmaf(f[e], m[k][e], dot);
      }
      dot = warp_sum(dot);
      if (lane == 0) red[par][j][warp] = dot;
    }
    if (r0 + RB < w.nrows) wide_load<T, NV, RB>(base, D, nvec, r0 + RB, w.nrows, tid, u);
    __syncthreads();
    if (tid < RB && r0 + tid < w.nrows)
      vrow[r0 + tid] = fold8(red[par][tid]) * rn[d.patch0 + w.r0 + r0 + tid] * inv_np;
  }
  __syncthreads();

  const float inv_h = 1.0f / (float)H;
  for (int r = tid; r < w.nrows; r += 256) {
    float s = 0.f;
#pragma unroll
    for (int q = 0; q < 8; ++q) s += part[q * w.nrows + r];
    s_raw[d.patch0 + w.r0 + r] = cA * vrow[r] - (1.0f - cA) * (s * inv_h);
  }
}

// ---------------------------------------------------------------------------------------
// Threshold of the k largest of np keys (0 < k < np): `nthr` threads (tid 0 .. nthr - 1, barrier `bar`) count the keys
// above three trial values at a time until exactly k keys are.  KPT keys per thread sit in registers, so a round is a
// few compares, a warp reduction and one barrier.  The trial values quarter the interval of the scores, not of the
// keys: the scores of an image are spread over their range, so the gap between the k-th and the next one is usually
// met after five or six rounds, while the keys of floats around zero would take more than twice as many.  (A radix
// select over 8-bit digits took 2.7 us for 576 keys and 8 us for 2880: histogram atomics, two to four passes.)
// need_eq < 0: every key >= thr is selected; otherwise the keys > thr and the need_eq lowest-indexed ones equal to it.
// `cnt`: [2][3][32] ints of shared memory.  kmin / kmax: smallest and largest key.
// ---------------------------------------------------------------------------------------
__device__ __forceinline__ float key_score(uint32_t key) {   // inverse of order_key
  return __uint_as_float((key & 0x80000000u) ? key & 0x7FFFFFFFu : ~key);
}
template <int KPT>
__device__ __forceinline__ void select_threshold(const uint32_t (&key)[KPT], int k, uint32_t kmin, uint32_t kmax, int* cnt,
                                                 int tid, int nthr, int bar, uint32_t& thr, int& need_eq) {
  const int lane = tid & 31, warp = tid >> 5, nwarp = nthr >> 5;
  // count(>= lo) >= k > count(>= hi)
  uint32_t lo = kmin, hi = kmax;
  int above = 0;                       // count(>= hi); hi starts as "above the largest key"
  bool open = true;
  int par = 0;
  #pragma unroll 1
  for (;;) {
    const uint32_t top = open ? hi : hi - 1u;        // largest trial value
    if (top == lo) break;
    uint32_t mid[3];
    {
      const float a = key_score(lo), b = key_score(top);
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        const uint32_t by_key = lo + 1u + (uint32_t)((((unsigned long long)(top - lo - 1u)) * (j + 1)) >> 2);
        const float v = a + (b - a) * (0.25f * (j + 1));
        const uint32_t m = order_key(v);
        mid[j] = (m > lo && m <= top) ? m : by_key;  // (not finite, or nothing between the two: by key)
      }
      // (ascending in every case that matters: a trial value out of order only repeats work)
    }
    int n[3] = {0, 0, 0};
#pragma unroll
    for (int q = 0; q < KPT; ++q)
#pragma unroll
      for (int j = 0; j < 3; ++j) n[j] += key[q] >= mid[j] ? 1 : 0;
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      n[j] = __reduce_add_sync(0xFFFFFFFFu, n[j]);
      if (lane == 0) cnt[(3 * par + j) * 32 + warp] = n[j];
    }
    cta_sync(bar, nthr);
#pragma unroll
    for (int j = 0; j < 3; ++j) n[j] = __reduce_add_sync(0xFFFFFFFFu, lane < nwarp ? cnt[(3 * par + j) * 32 + lane] : 0);
    par ^= 1;                          // the next round's counts go to the other half: one barrier per round is enough
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      if (n[j] == k) { thr = mid[j]; need_eq = -1; return; }
      if (n[j] > k) { if (mid[j] > lo) lo = mid[j]; }
      else if (open || mid[j] < hi) { hi = mid[j]; above = n[j]; open = false; }
    }
  }
  thr = lo;
  need_eq = k - above;
}

// Positions that occur more than once: the map keeps whichever token was written last, so until nothing changes any
// more a token that beats the one its cell holds (higher score, lower index on equal scores) takes its place.  Every
// round leaves each contested cell with a better token, so the rounds end, with the best one, whatever the order of
// the writes; where all positions differ there is one round, a read per token and a barrier.  pos_of(i, k): position of
// token i, the thread's k-th.
template <class Cell, class PosOf>
__device__ __forceinline__ void settle_cells(Cell* cell, int cells, const float* sc, PosOf pos_of, int np, int tid, int nthr,
                                             int bar) {
  volatile Cell* map = cell;
  bool again;
  do {
    again = false;
    #pragma unroll 1
    for (int i = tid, k = 0; i < np; i += nthr, ++k) {
      const int p = pos_of(i, k);
      if (p < 0 || p >= cells) continue;
      const int holder = map[p];
      if (holder == i) continue;
      const uint32_t mine = order_key(sc[i] + 0.0f), theirs = order_key(sc[holder] + 0.0f);
      if (mine > theirs || (mine == theirs && i < holder)) { map[p] = (Cell)i; again = true; }
    }
  } while (cta_sync_or(bar, nthr, again));
}

// Token whose score is largest in window `wdx` of `nwc` per grid row (lower token index on equal scores), -1: none alive.
// cell: token of every grid cell, NONE where there is none; sc: scores.
template <class Cell, Cell NONE>
__device__ __forceinline__ int window_best(const Cell* cell, const float* sc, int gh, int gw, int window, int nwc, int wdx) {
  const int r0 = (wdx / nwc) * window, c0 = (wdx % nwc) * window;
  int best = -1;
  float bs = 0.f;
  if (window == 2) {                               // the four cells and their scores as two trips, not eight
    Cell t[4];
    float v[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int r = r0 + (j >> 1), c = c0 + (j & 1);
      t[j] = r < gh && c < gw ? cell[r * gw + c] : NONE;
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) v[j] = t[j] != NONE ? sc[t[j]] : 0.f;
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (t[j] != NONE && (best < 0 || v[j] > bs || (v[j] == bs && (int)t[j] < best))) { best = t[j]; bs = v[j]; }
    return best;
  }
  const int r1 = min(gh, r0 + window), c1 = min(gw, c0 + window);
  #pragma unroll 1
  for (int r = r0; r < r1; ++r)
    #pragma unroll 1
    for (int c = c0; c < c1; ++c) {
      const Cell t = cell[r * gw + c];
      if (t == NONE) continue;
      const float v = sc[t];
      if (best < 0 || v > bs || (v == bs && (int)t < best)) { best = t; bs = v; }
    }
  return best;
}

// ---------------------------------------------------------------------------------------
// Local penalty + top-N^S selection of one image by 512 threads (hardware barrier `bar`).
//   1. a grid-cell -> token map lets one thread per window pick the window's maximum (lower token index on
//      equal scores) and multiply it in place;
//   2. a histogram of the scores over SEL_BINS equal parts of their range finds the part that the threshold lies in (a
//      few tokens of thousands); its tokens, listed, are ranked among themselves.  Where they are more than the list
//      takes (scores that are mostly equal, or not finite), a search over the value range takes over;
//      ties at the threshold go to the lower index;
//   3. ballots and one scan turn the membership flags into ascending index lists S and T, the kept
//      row indices and the surviving grid positions.
// Only the outputs of tokens w_lo <= i < w_hi are written (plus the CLS / trailing entries of kept_idx when w_lo == 0), so
// the CTAs that scored an image can each run the selection and write their own slice.  select_image_prepare() clears the
// work area; a barrier (or any inter-CTA wait that ends in one) must separate it from select_image().
// What bounds it is the chain of barriers and shared-memory trips, and instruction fetch, as the code runs once: loops are
// rolled (eight tokens per thread in registers, everything unrolled: 13 us).  2880 tokens, on the CTA that scored the image's last
// piece alone and with sixteen keys per thread in a search of the value range: 17.6 us, of which threshold 6.5, keys 3.6,
// windows 2.0, lists 3.2; now 11 (whole step of 8 x 2881 tokens 130.7 -> 123 us, 16 ragged images 92 -> 85.5).  As a kernel of
// its own, 512 threads for an image instead of 1024 and the histogram instead of the search: 8 x 2880 tokens 22.2 -> 14.2 us,
// 8 x 4096 22.6 -> 15.6 (FiCoCo-L); with relation maps the step of 4 x 1152 47.0 -> 37.0, of 2 x 3000 84.1 -> 77.4.
// ---------------------------------------------------------------------------------------
constexpr int SEL_THREADS = 512;
constexpr int SEL_BINS = 4 * SEL_THREADS;
constexpr int SEL_LIST = 512;      // tokens of one part that are ranked among themselves

__host__ __device__ inline size_t select_work_bytes(int np, int cells) {
  return (size_t)np * 4 + 16 + SEL_BINS * sizeof(int) + (size_t)cells * 2 + 64;
}

struct SelectShared {
  int group[MAX_IMG_TOKENS / 32];
  uint32_t list[SEL_LIST];
  uint32_t wmin[16], wmax[16];
  int wsum[16];
  int cnt[192];
  int n_list, part, rest, in_part, need_eq;
  uint32_t thr;
};

struct SelectWork {
  float* sc;             // [np] scores (penalised in place)
  int* hist;             // [SEL_BINS]
  unsigned short* cell;  // [gh * gw] token of every grid cell, 0xFFFF: none
};
__device__ __forceinline__ SelectWork select_layout(unsigned char* work, int np) {
  SelectWork w;
  w.sc = reinterpret_cast<float*>(work);
  w.hist = reinterpret_cast<int*>((reinterpret_cast<uintptr_t>(work + (size_t)np * 4) + 15) & ~(uintptr_t)15);
  w.cell = reinterpret_cast<unsigned short*>(w.hist + SEL_BINS);
  return w;
}

__device__ __forceinline__ void select_image_prepare(const ImgDesc& d, int penalty, unsigned char* work, SelectShared& sh, int tid) {
  const SelectWork w = select_layout(work, d.np);
  *reinterpret_cast<int4*>(w.hist + 4 * tid) = make_int4(0, 0, 0, 0);
  if (tid == 0) sh.n_list = 0;
  if (penalty) {
    const int cells = d.gh * d.gw;
    #pragma unroll 1
    for (int i = tid; i < cells; i += SEL_THREADS) w.cell[i] = 0xFFFFu;
  }
}

// Threshold by a search over the value range, for images whose scores are mostly equal or not finite.
__device__ __noinline__ void select_threshold_search(const float* sc, int np, int k, uint32_t kmin, uint32_t kmax,
                                                     SelectShared& sh, int tid, int bar) {
  constexpr int KPT = MAX_IMG_TOKENS / SEL_THREADS;
  uint32_t key[KPT], thr;
  int need_eq;
#pragma unroll
  for (int q = 0; q < KPT; ++q) key[q] = tid + SEL_THREADS * q < np ? max(1u, order_key(sc[tid + SEL_THREADS * q] + 0.0f)) : 0u;
  select_threshold<KPT>(key, k, kmin, kmax, sh.cnt, tid, SEL_THREADS, bar, thr, need_eq);
  if (tid == 0) {
    sh.thr = need_eq < 0 ? thr - 1u : thr;         // all keys > thr - 1, none at the threshold
    sh.need_eq = max(need_eq, 0);
  }
  cta_sync(bar, SEL_THREADS);
}

__device__ __noinline__ void select_image(
    const ImgDesc& d, const float* s_raw, const int* __restrict__ pos, int window, float coef,
    int penalty, float* __restrict__ s_pen, float* __restrict__ scores_out, int* __restrict__ S_idx,
    int* __restrict__ T_idx, int* __restrict__ kept_idx, int* __restrict__ pos_out,
    unsigned* __restrict__ status, unsigned char* work, SelectShared& sh, int tid, int bar, int w_lo, int w_hi) {
  constexpr int NT = SEL_THREADS;
  const int np = d.np, lane = tid & 31, warp = tid >> 5;
  const SelectWork wk = select_layout(work, np);
  float* sc = wk.sc;
  const int cells = d.gh * d.gw;
  #pragma unroll 1
  for (int i0 = tid; i0 < np; i0 += 8 * NT) {      // eight tokens' loads in flight per thread
    float a[8];
    int p[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const int i = i0 + NT * j;
      a[j] = i < np ? __ldcg(s_raw + d.patch0 + i) : 0.f;
      p[j] = i < np && pos ? pos[d.patch0 + i] : i;
    }
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const int i = i0 + NT * j;
      if (i >= np) break;
      sc[i] = a[j];
      if (penalty) {
        if (p[j] >= 0 && p[j] < cells) wk.cell[p[j]] = (unsigned short)i;
        else atomicOr(status, STATUS_POS_RANGE);
      }
    }
  }
  cta_sync(bar, NT);

  // ---- local penalty: one thread per window ------------------------------------------------
  if (penalty) {
    if (pos) settle_cells(wk.cell, cells, sc, [&](int i, int) { return pos[d.patch0 + i]; }, np, tid, NT, bar);
    const int nwc = (d.gw + window - 1) / window, nwr = (d.gh + window - 1) / window;
    #pragma unroll 1
    for (int wdx = tid; wdx < nwc * nwr; wdx += NT) {
      const int best = window_best<unsigned short, 0xFFFFu>(wk.cell, sc, d.gh, d.gw, window, nwc, wdx);
      if (best >= 0) sc[best] *= coef;               // windows are disjoint: nobody else touches this token
    }
    cta_sync(bar, NT);
  }

  // ---- range of the keys -------------------------------------------------------------------
  uint32_t kmin = 0xFFFFFFFFu, kmax = 0u;
  #pragma unroll 2
  for (int i = tid; i < np; i += NT) {
    const float s = sc[i] + 0.0f;                  // -0 and +0 are one score
    if (i >= w_lo && i < w_hi) {
      s_pen[d.patch0 + i] = s;
      if (scores_out) scores_out[d.patch0 + i] = s;
    }
    const uint32_t key = max(1u, order_key(s));
    kmin = min(kmin, key);
    kmax = max(kmax, key);
  }
  const int k = d.n_src;
  uint32_t thr = 0;       // threshold key
  int need_eq = 0;        // how many keys equal to thr are selected (lowest indices)
  if (k > 0 && k < np) {
    kmin = __reduce_min_sync(0xFFFFFFFFu, kmin);
    kmax = __reduce_max_sync(0xFFFFFFFFu, kmax);
    if (lane == 0) { sh.wmin[warp] = kmin; sh.wmax[warp] = kmax; }
    cta_sync(bar, NT);
    kmin = __reduce_min_sync(0xFFFFFFFFu, sh.wmin[lane & 15]);
    kmax = __reduce_max_sync(0xFFFFFFFFu, sh.wmax[lane & 15]);
    // ---- histogram over the value range (the part of a score does not fall as the score rises) ----
    const float lo = key_score(kmin), range = key_score(kmax) - lo;
    const float scale = range > 0.f && range < CUDART_MAX_NORMAL_F ? (float)(SEL_BINS - 1) / range : 0.f;
    auto part_of = [&](float s) { return max(0, min(SEL_BINS - 1, (int)__fmul_rn(__fsub_rn(s + 0.0f, lo), scale))); };
    #pragma unroll 2
    for (int i = tid; i < np; i += NT) atomicAdd(&wk.hist[part_of(sc[i])], 1);
    cta_sync(bar, NT);
    // thread t: parts SEL_BINS - 1 - 4 t and the three below; running counts from the top
    const int4 h4 = *reinterpret_cast<const int4*>(wk.hist + SEL_BINS - 4 - 4 * tid);
    const int h[4] = {h4.w, h4.z, h4.y, h4.x}, sum = h4.x + h4.y + h4.z + h4.w;
    int inc = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int n = __shfl_up_sync(0xFFFFFFFFu, inc, o);
      if (lane >= o) inc += n;
    }
    if (lane == 31) sh.wsum[warp] = inc;
    cta_sync(bar, NT);
    int run = __reduce_add_sync(0xFFFFFFFFu, lane < warp ? sh.wsum[lane & 15] : 0) + inc - sum;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      if (run < k && run + h[j] >= k) { sh.part = SEL_BINS - 1 - 4 * tid - j; sh.rest = k - run; sh.in_part = h[j]; }
      run += h[j];
    }
    cta_sync(bar, NT);
    const int in_part = sh.in_part, rest = sh.rest, at = sh.part;
    if (in_part <= SEL_LIST) {
      #pragma unroll 2
      for (int i = tid; i < np; i += NT)
        if (part_of(sc[i]) == at) sh.list[atomicAdd(&sh.n_list, 1)] = max(1u, order_key(sc[i] + 0.0f));
      cta_sync(bar, NT);
      // the rest-th largest of the list: every entry counts the ones above it and the ones not below it
      if (tid < in_part) {
        const uint32_t mine = sh.list[tid];
        int above = 0, not_below = 0;
        #pragma unroll 4
        for (int j = 0; j < in_part; ++j) {
          above += sh.list[j] > mine ? 1 : 0;
          not_below += sh.list[j] >= mine ? 1 : 0;
        }
        if (above < rest && not_below >= rest) { sh.thr = mine; sh.need_eq = rest - above; }   // (equal entries: the same)
      }
      cta_sync(bar, NT);
    } else {
      select_threshold_search(sc, np, k, kmin, kmax, sh, tid, bar);
    }
    thr = sh.thr;
    need_eq = sh.need_eq;
  }

  // ---- ordered compaction into S and T ------------------------------------------------------
  // 32 tokens per warp and trip: ballots give the members among them, one scan over the groups' packed counts
  // (greater-than in the high half, equal in the low half) what lies before each group.
  const int nw = (np + 31) / 32;
  auto members = [&](int g, unsigned& gt, unsigned& eq) {
    const int i = 32 * g + lane;
    const uint32_t key = i < np ? max(1u, order_key(sc[i] + 0.0f)) : 0u;
    gt = __ballot_sync(0xFFFFFFFFu, i < np && (k >= np || (k > 0 && key > thr)));
    eq = __ballot_sync(0xFFFFFFFFu, i < np && k > 0 && k < np && key == thr);
  };
  #pragma unroll 2
  for (int g = warp; g < nw; g += NT / 32) {
    unsigned gt, eq;
    members(g, gt, eq);
    if (lane == 0) sh.group[g] = __popc(gt) << 16 | __popc(eq);
  }
  cta_sync(bar, NT);
  if (warp == 0) {
    constexpr int PER = MAX_IMG_TOKENS / 32 / 32;
    int c[PER], sum = 0;
#pragma unroll
    for (int j = 0; j < PER; ++j) { c[j] = PER * lane + j < nw ? sh.group[PER * lane + j] : 0; sum += c[j]; }
    int inc = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int n = __shfl_up_sync(0xFFFFFFFFu, inc, o);
      if (lane >= o) inc += n;
    }
    int run = inc - sum;
#pragma unroll
    for (int j = 0; j < PER; ++j) {
      if (PER * lane + j < nw) sh.group[PER * lane + j] = run;
      run += c[j];
    }
  }
  cta_sync(bar, NT);
  #pragma unroll 1
  for (int g = (w_lo >> 5) + warp; 32 * g < w_hi; g += NT / 32) {
    const int i = 32 * g + lane;
    unsigned gt, eq;
    members(g, gt, eq);
    if (i < w_lo || i >= w_hi) continue;
    const unsigned lt = (1u << lane) - 1u;
    const int before = sh.group[g];
    const int gt_before = (before >> 16) + __popc(gt & lt), eq_before = (before & 0xFFFF) + __popc(eq & lt);
    const int sel_rank = gt_before + min(eq_before, need_eq);   // selected tokens before i
    if ((gt >> lane & 1u) || ((eq >> lane & 1u) && eq_before < need_eq)) {
      S_idx[d.src0 + sel_rank] = i;
    } else {
      const int tp = i - sel_rank;
      T_idx[d.tgt0 + tp] = i;
      kept_idx[d.out_row0 + d.n_cls + tp] = d.n_cls + i;
      if (pos_out) pos_out[d.tgt0 + tp] = pos ? pos[d.patch0 + i] : i;
    }
  }
  if (w_lo == 0) {
    #pragma unroll 1
    for (int i = tid; i < d.n_cls; i += NT) kept_idx[d.out_row0 + i] = i;
    #pragma unroll 1
    for (int i = tid; i < d.n_tail; i += NT)
      kept_idx[d.out_row0 + d.n_cls + d.n_tgt + d.n_extra + i] = d.n_cls + np + i;
    if (tid == 0 && d.n_extra) kept_idx[d.out_row0 + d.n_cls + d.n_tgt] = -1;
  }
}

// ---------------------------------------------------------------------------------------
// The same step for images of up to SEL_SMALL_MAX tokens by exactly 512 threads, two tokens per
// thread held in registers, built for a short critical path (seven or eight barriers, no
// contended atomics):
//   1. scores and grid positions are loaded once; a grid-cell -> token map in shared memory lets
//      one thread per window pick the window's maximum (lower token index on equal scores) and
//      multiply it in place;
//   2. keys are made dense: key - min key, shifted so that the largest has its top bit set, so the
//      first radix digit already spreads the tokens over its 256 bins (raw fp32 keys of one
//      image share sign and exponent and would all hit one bin); every warp reads the histogram
//      and finds the digit by itself, so a pass costs one barrier; passes that could only see
//      zero bits are skipped;
//   3. membership flags become ascending positions with two ballots per warp and one 32-entry
//      table of per-warp counts.
// Only the outputs of tokens w_lo <= i < w_hi are written (plus the CLS / trailing entries of
// kept_idx when w_lo == 0), so the CTAs that scored an image can each run the selection and
// write their own slice.  select_small_prepare() zeroes the work area; a barrier (or any
// inter-CTA wait that ends in one) must separate it from select_small().
// ---------------------------------------------------------------------------------------
constexpr int SEL_SMALL_MAX = 1024;
constexpr int SEL_SMALL_THREADS = SEL_THREADS;

struct SelectSmallShared {
  uint32_t wmin[16], wmax[16];
  int cnt[32];
};

__host__ __device__ inline size_t select_small_bytes(int np, int cells) {
  return (size_t)np * 8 + 16 + 4 * 256 * sizeof(int) + (size_t)cells * 2 + 16;
}

struct SelectSmallWork {
  float* sc;        // [np] scores (penalised in place)
  uint32_t* nk;     // [np] dense keys
  int* hist;        // [4][256]
  short* cell;      // [gh * gw] token of every grid cell, -1 = no alive token
};
__device__ __forceinline__ SelectSmallWork select_small_layout(unsigned char* work, int np) {
  SelectSmallWork w;
  w.sc = reinterpret_cast<float*>(work);
  w.nk = reinterpret_cast<uint32_t*>(work + (size_t)np * 4);
  w.hist = reinterpret_cast<int*>((reinterpret_cast<uintptr_t>(work + (size_t)np * 8) + 15) & ~(uintptr_t)15);
  w.cell = reinterpret_cast<short*>(w.hist + 4 * 256);
  return w;
}

__device__ __forceinline__ void select_small_prepare(const ImgDesc& d, int penalty, unsigned char* work, int tid) {
  const SelectSmallWork w = select_small_layout(work, d.np);
  w.hist[tid] = 0;
  w.hist[tid + SEL_SMALL_THREADS] = 0;
  if (penalty) {
    const int cells = d.gh * d.gw;
    #pragma unroll 1
    for (int c = tid; c < cells; c += SEL_SMALL_THREADS) w.cell[c] = -1;
  }
}

__device__ __noinline__ void select_small(
    const ImgDesc& d, const float* s_raw, const int* __restrict__ pos, int window, float coef,
    int penalty, float* __restrict__ s_pen, float* __restrict__ scores_out, int* __restrict__ S_idx,
    int* __restrict__ T_idx, int* __restrict__ kept_idx, int* __restrict__ pos_out,
    unsigned* __restrict__ status, unsigned char* work, SelectSmallShared& sh, int tid, int bar,
    int w_lo, int w_hi) {
  constexpr int NT = SEL_SMALL_THREADS;
  const int np = d.np, lane = tid & 31, warp = tid >> 5;
  const SelectSmallWork wk = select_small_layout(work, np);
  const int cells = d.gh * d.gw;
  float s[2];
  int pp[2];
  bool on[2];
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    const int i = tid + NT * q;
    on[q] = i < np;
    s[q] = on[q] ? __ldcg(s_raw + d.patch0 + i) : 0.f;
    pp[q] = on[q] ? (pos ? pos[d.patch0 + i] : i) : -1;
  }
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    const int i = tid + NT * q;
    if (!on[q]) continue;
    wk.sc[i] = s[q];
    if (penalty) {
      if (pp[q] >= 0 && pp[q] < cells) wk.cell[pp[q]] = (short)i;
      else atomicOr(status, STATUS_POS_RANGE);
    }
  }
  cta_sync(bar, NT);

  // ---- local penalty: one thread per window ------------------------------------------------
  if (penalty) {
    if (pos) settle_cells(wk.cell, cells, wk.sc, [&](int, int k) { return k == 0 ? pp[0] : pp[1]; }, np, tid, NT, bar);
    const int nwc = (d.gw + window - 1) / window, nwr = (d.gh + window - 1) / window;
    #pragma unroll 1
    for (int wdx = tid; wdx < nwc * nwr; wdx += NT) {
      const int best = window_best<short, -1>(wk.cell, wk.sc, d.gh, d.gw, window, nwc, wdx);
      if (best >= 0) wk.sc[best] *= coef;            // windows are disjoint: nobody else touches this token
    }
    cta_sync(bar, NT);
  }

  // ---- keys, their range, dense keys -----------------------------------------------------------
  uint32_t key[2];
  uint32_t kmin = 0xFFFFFFFFu, kmax = 0u;
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    const int i = tid + NT * q;
    if (on[q]) {
      s[q] = wk.sc[i] + 0.0f;                      // -0 and +0 are one score
      key[q] = order_key(s[q]);
      kmin = min(kmin, key[q]);
      kmax = max(kmax, key[q]);
      if (i >= w_lo && i < w_hi) {
        s_pen[d.patch0 + i] = s[q];
        if (scores_out) scores_out[d.patch0 + i] = s[q];
      }
    } else {
      key[q] = 0u;
    }
  }
  kmin = __reduce_min_sync(0xFFFFFFFFu, kmin);
  kmax = __reduce_max_sync(0xFFFFFFFFu, kmax);
  if (lane == 0) { sh.wmin[warp] = kmin; sh.wmax[warp] = kmax; }
  cta_sync(bar, NT);
  {
    const uint32_t a = sh.wmin[lane & 15], b = sh.wmax[lane & 15];
    kmin = __reduce_min_sync(0xFFFFFFFFu, a);
    kmax = __reduce_max_sync(0xFFFFFFFFu, b);
  }
  const int k = d.n_src;
  const uint32_t range = kmax - kmin;
  const int sh_l = range ? __clz(range) : 0;
  uint32_t nk[2];
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    nk[q] = range ? (key[q] - kmin) << sh_l : 0u;
    if (on[q]) wk.nk[tid + NT * q] = nk[q];
  }

  // ---- radix select on the dense keys: the n_src-th largest -------------------------------------
  uint32_t thr = 0;      // threshold (dense key)
  int need_eq = 0;       // how many of the keys equal to thr are selected (lowest indices)
  int c_eq = 0;          // how many keys equal thr
  uint32_t thr_mask = 0xFFFFFFFFu;   // digits of the dense keys the passes have looked at
  if (k > 0 && k < np) {
    const int npass = range ? (32 - sh_l + 7) / 8 : 1;   // the low sh_l bits of every dense key are zero
    uint32_t prefix = 0, mask = 0;
    int remaining = k;
    #pragma unroll 1
    for (int pass = 0; pass < npass; ++pass) {
      const int shift = 24 - 8 * pass;
      int* h = wk.hist + 256 * pass;
#pragma unroll
      for (int q = 0; q < 2; ++q)
        if (on[q] && (nk[q] & mask) == prefix) atomicAdd(&h[(nk[q] >> shift) & 255], 1);
      cta_sync(bar, NT);
      // every warp: lane l owns bins 255-8l .. 248-8l (descending); find where the running count
      // from the top reaches `remaining`
      int c[8], tot = 0;
      {
        const int4 lo = *reinterpret_cast<const int4*>(h + 248 - 8 * lane);
        const int4 hi = *reinterpret_cast<const int4*>(h + 252 - 8 * lane);
        c[0] = hi.w; c[1] = hi.z; c[2] = hi.y; c[3] = hi.x;
        c[4] = lo.w; c[5] = lo.z; c[6] = lo.y; c[7] = lo.x;
      }
#pragma unroll
      for (int j = 0; j < 8; ++j) tot += c[j];
      int inc = tot;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int n = __shfl_up_sync(0xFFFFFFFFu, inc, o);
        if (lane >= o) inc += n;
      }
      const int before = inc - tot;
      const bool mine = before < remaining && inc >= remaining;
      int digit = 0, rem_new = 0, ceq_new = 0;
      if (mine) {
        int cum = before;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          if (cum < remaining && cum + c[j] >= remaining) {
            digit = 255 - 8 * lane - j;
            rem_new = remaining - cum;
            ceq_new = c[j];
          }
          cum += c[j];
        }
      }
      const int src = __ffs(__ballot_sync(0xFFFFFFFFu, mine)) - 1;   // exactly one lane (0 < remaining <= total)
      digit = __shfl_sync(0xFFFFFFFFu, digit, src);
      remaining = __shfl_sync(0xFFFFFFFFu, rem_new, src);
      c_eq = __shfl_sync(0xFFFFFFFFu, ceq_new, src);
      prefix |= (uint32_t)digit << shift;
      mask |= 0xFFu << shift;
      if (remaining == c_eq) break;    // every key that shares these digits is selected: no need to tell them apart
    }
    thr = prefix;
    need_eq = remaining;
    thr_mask = mask;
  }

  // ---- membership ---------------------------------------------------------------------------------
  bool sel[2];
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    const int i = tid + NT * q;
    if (!on[q]) sel[q] = false;
    else if (k <= 0) sel[q] = false;
    else if (k >= np) sel[q] = true;
    else if ((nk[q] & thr_mask) != thr) sel[q] = (nk[q] & thr_mask) > thr;
    else if (need_eq >= c_eq) sel[q] = true;
    else {
      // equal scores straddle the boundary: the lowest indices among them are taken
      // (all passes were made, so the mask covers every bit that is set in any key)
      int before = 0;
      #pragma unroll 1
      for (int j = 0; j < i; ++j) before += wk.nk[j] == thr ? 1 : 0;
      sel[q] = before < need_eq;
    }
  }

  // ---- ascending positions ------------------------------------------------------------------------
  const unsigned b0 = __ballot_sync(0xFFFFFFFFu, sel[0]), b1 = __ballot_sync(0xFFFFFFFFu, sel[1]);
  if (lane == 0) { sh.cnt[warp] = __popc(b0); sh.cnt[16 + warp] = __popc(b1); }
  cta_sync(bar, NT);
  {
    const int mycnt = sh.cnt[lane];
    int inc = mycnt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int n = __shfl_up_sync(0xFFFFFFFFu, inc, o);
      if (lane >= o) inc += n;
    }
    const int excl = inc - mycnt;                 // selected tokens in the 32-token groups before group `lane`
    const unsigned lt = (1u << lane) - 1u;
    const int rank0 = __shfl_sync(0xFFFFFFFFu, excl, warp) + __popc(b0 & lt);
    const int rank1 = __shfl_sync(0xFFFFFFFFu, excl, 16 + warp) + __popc(b1 & lt);
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const int i = tid + NT * q;
      if (!on[q] || i < w_lo || i >= w_hi) continue;
      const int rank = q ? rank1 : rank0;          // selected tokens with a lower index
      if (sel[q]) {
        S_idx[d.src0 + rank] = i;
      } else {
        const int tp = i - rank;
        T_idx[d.tgt0 + tp] = i;
        kept_idx[d.out_row0 + d.n_cls + tp] = d.n_cls + i;
        if (pos_out) pos_out[d.tgt0 + tp] = pp[q];
      }
    }
  }
  if (w_lo == 0) {
    #pragma unroll 1
    for (int i = tid; i < d.n_cls; i += NT) kept_idx[d.out_row0 + i] = i;
    #pragma unroll 1
    for (int i = tid; i < d.n_tail; i += NT)
      kept_idx[d.out_row0 + d.n_cls + d.n_tgt + d.n_extra + i] = d.n_cls + np + i;
    if (tid == 0 && d.n_extra) kept_idx[d.out_row0 + d.n_cls + d.n_tgt] = -1;
  }
}

// One CTA per image.  SMALL: no image has more than SEL_SMALL_MAX tokens.
template <bool SMALL>
__global__ void __launch_bounds__(SEL_THREADS, 2) k_select(const ImgDesc* __restrict__ desc,
                                                           const float* __restrict__ s_raw,
                                                           const int* __restrict__ pos, int window, float coef,
                                                           int penalty, float* __restrict__ s_pen,
                                                           float* __restrict__ scores_out,
                                                           int* __restrict__ S_idx, int* __restrict__ T_idx,
                                                           int* __restrict__ kept_idx, int* __restrict__ pos_out,
                                                           unsigned* __restrict__ status) {
  extern __shared__ __align__(16) unsigned char sm_raw[];
  const ImgDesc d = desc[blockIdx.x];
  const int tid = threadIdx.x;
  if (SMALL || d.np <= SEL_SMALL_MAX) {
    __shared__ SelectSmallShared shs;
    select_small_prepare(d, penalty, sm_raw, tid);
    grid_dep_wait();
    grid_dep_launch();
    __syncthreads();
    select_small(d, s_raw, pos, window, coef, penalty, s_pen, scores_out, S_idx, T_idx, kept_idx, pos_out,
                 status, sm_raw, shs, tid, 0, 0, d.np);
    return;
  }
  if constexpr (!SMALL) {
    __shared__ SelectShared sh;
    select_image_prepare(d, penalty, sm_raw, sh, tid);
    grid_dep_wait();
    grid_dep_launch();
    __syncthreads();
    select_image(d, s_raw, pos, window, coef, penalty, s_pen, scores_out, S_idx, T_idx, kept_idx, pos_out,
                 status, sm_raw, sh, tid, 0, 0, d.np);
  }
}

}  // namespace ficoco
