// Shared device-side definitions: per-image descriptors, work items, vector loads.
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>
#include "correlate_plan.h"

namespace ficoco {

constexpr int MAX_CHUNKS = 64;      // row chunks per image for the column-sum partials
constexpr int MAX_IMG_TOKENS = 8192;
constexpr unsigned STATUS_POS_RANGE = 1u;

// One image (FiCoCo-V) or sequence (FiCoCo-L) of the batch.  All offsets are in elements of
// the array they index, counted over the whole packed batch.
struct alignas(16) ImgDesc {
  int row0;        // first token row in `tokens`
  int n_cls;       // leading pass-through rows (CLS)
  int np;          // alive vision tokens
  int n_src;       // N^S, discarded
  int n_tgt;       // N^T, preserved
  int n_tail;      // trailing pass-through rows (text)
  int n_extra;     // 1: one additional output row after the preserved tokens ("convergent correlation" ablation)
  int gh, gw;      // original patch grid
  int patch0;      // offset in per-vision-token arrays
  int out_row0;    // first output row (also offset in kept_idx)
  int src0;        // offset in per-discarded-token arrays
  int tgt0;        // offset in per-preserved-token arrays
  int ent0;        // offset in the (target, source, weight) entry arrays
  int part0;       // offset in the partial top-list arrays
  int list_len;    // L: entries of the top list needed for tau_i (0 = no merging)
  float frac;      // interpolation weight of the quantile
  int nsplit;      // column splits of the correlate step
  int cols_per_split;
  int chunk0;      // first row chunk (column-sum partials)
  int n_chunks;
  int avg;         // 1: every alpha_ij is 1 ("average compression" ablation)
  long long attn0; // offset (floats) of this image's attention block
  long long rel0;  // offset (floats) of this image's [Np, Np] relation block (relation mode)
};

struct WorkItem {
  int img;
  int r0;      // first row (patch / source slot / output row) inside the image
  int nrows;
  int aux;     // row chunks: chunk index inside the image; correlate: column split; output rows: distance of a CTA's rows
};

// ---------------------------------------------------------------------------------------
// 16-byte vector access, converted to fp32 lanes
// ---------------------------------------------------------------------------------------
template <class T> struct VecTraits;
template <> struct VecTraits<float> { static constexpr int E = 4; };
template <> struct VecTraits<__nv_bfloat16> { static constexpr int E = 8; };

__device__ __forceinline__ void unpack(const uint4& u, float (&f)[4], const float*) {
  f[0] = __uint_as_float(u.x); f[1] = __uint_as_float(u.y);
  f[2] = __uint_as_float(u.z); f[3] = __uint_as_float(u.w);
}
__device__ __forceinline__ void unpack(const uint4& u, float (&f)[8], const __nv_bfloat16*) {
  f[0] = __uint_as_float(u.x << 16); f[1] = __uint_as_float(u.x & 0xFFFF0000u);
  f[2] = __uint_as_float(u.y << 16); f[3] = __uint_as_float(u.y & 0xFFFF0000u);
  f[4] = __uint_as_float(u.z << 16); f[5] = __uint_as_float(u.z & 0xFFFF0000u);
  f[6] = __uint_as_float(u.w << 16); f[7] = __uint_as_float(u.w & 0xFFFF0000u);
}

// The same as pairs of neighbours, for the two-wide fp32 instructions of sm_100 (each half rounded like the one-wide one).
__device__ __forceinline__ void unpack2(const uint4& u, float2 (&f)[2], const float*) {
  f[0] = make_float2(__uint_as_float(u.x), __uint_as_float(u.y));
  f[1] = make_float2(__uint_as_float(u.z), __uint_as_float(u.w));
}
__device__ __forceinline__ void unpack2(const uint4& u, float2 (&f)[4], const __nv_bfloat16*) {
  f[0] = make_float2(__uint_as_float(u.x << 16), __uint_as_float(u.x & 0xFFFF0000u));
  f[1] = make_float2(__uint_as_float(u.y << 16), __uint_as_float(u.y & 0xFFFF0000u));
  f[2] = make_float2(__uint_as_float(u.z << 16), __uint_as_float(u.z & 0xFFFF0000u));
  f[3] = make_float2(__uint_as_float(u.w << 16), __uint_as_float(u.w & 0xFFFF0000u));
}
__device__ __forceinline__ float2 fma2(const float2& a, const float2& b, const float2& c) {
  unsigned long long d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d)
      : "l"(reinterpret_cast<const unsigned long long&>(a)), "l"(reinterpret_cast<const unsigned long long&>(b)),
        "l"(reinterpret_cast<const unsigned long long&>(c)));
  return reinterpret_cast<const float2&>(d);
}

__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi) {
  __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<uint32_t*>(&v);
}
__device__ __forceinline__ uint4 pack(const float (&f)[4], const float*) {
  return make_uint4(__float_as_uint(f[0]), __float_as_uint(f[1]), __float_as_uint(f[2]), __float_as_uint(f[3]));
}
__device__ __forceinline__ uint4 pack(const float (&f)[8], const __nv_bfloat16*) {
  return make_uint4(pack_bf16x2(f[0], f[1]), pack_bf16x2(f[2], f[3]), pack_bf16x2(f[4], f[5]), pack_bf16x2(f[6], f[7]));
}

__device__ __forceinline__ uint4 ldg16(const void* p) { return __ldg(reinterpret_cast<const uint4*>(p)); }
// Loads that are issued where they stand (the compiler moves a plain load of constant data to its first use, behind the
// waits that it is meant to be in flight under).
__device__ __forceinline__ uint4 ld16_now(const void* p) {
  uint4 v;
  asm volatile("ld.global.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
  return v;
}
__device__ __forceinline__ float ld_now(const float* p) {
  float v;
  asm volatile("ld.global.cg.f32 %0, [%1];" : "=f"(v) : "l"(p));
  return v;
}

// Streaming store (st.global.cs) for the output rows.  A step's token rows, read by all three of its kernels, plus its
// output rows are about as much as L2 keeps.  32 x 577 tokens of 1024, DRAM reads of correlate and merge in the running
// step: 0.64 and 0.18 MB where inputs are used again, 1.50 and 0.47 with ordinary stores; on cycled inputs 0.3 MB both ways.
__device__ __forceinline__ void st_stream16(uint4* p, const uint4& v) { __stcs(p, v); }

// A token index read from an index list of the step, as a row offset inside its image: anything
// outside [0, np) (lists left behind by a step that went wrong) raises STATUS_INDEX and becomes 0,
// so that no gather leaves the image.
__device__ __forceinline__ int checked_index(int idx, int np, unsigned* status) {
  if ((unsigned)idx >= (unsigned)np) {
    atomicOr(status, 8u);
    return 0;
  }
  return idx;
}

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
  return v;
}

// Order-preserving map fp32 -> uint32 (larger float <=> larger key).
__device__ __forceinline__ uint32_t order_key(float s) {
  uint32_t u = __float_as_uint(s);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

// Barrier over the first `n` threads of the CTA (n a multiple of 32) on hardware barrier `id`;
// cta_sync(0, blockDim.x) is __syncthreads().
__device__ __forceinline__ void cta_sync(int id, int n) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(n) : "memory");
}

// The same barrier; true for all threads when `pred` is true for any.
__device__ __forceinline__ bool cta_sync_or(int id, int n, bool pred) {
  uint32_t any;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t"
      "setp.ne.u32 p, %3, 0;\n\t"
      "barrier.cta.red.or.pred q, %1, %2, p;\n\t"
      "selp.u32 %0, 1, 0, q;\n\t}"
      : "=r"(any) : "r"(id), "r"(n), "r"((uint32_t)pred) : "memory");
  return any != 0;
}

// Sorted top list (descending value, ties: lower index first).
__device__ __forceinline__ bool toplist_better(float val, int idx, float v_last, int i_last) {
  return val > v_last || (val == v_last && idx < i_last);
}
__device__ __forceinline__ void toplist_insert(float* v, int* ix, int L, float val, int idx) {
  int p = L - 1;
  while (p > 0 && toplist_better(val, idx, v[p - 1], ix[p - 1])) {
    v[p] = v[p - 1];
    ix[p] = ix[p - 1];
    --p;
  }
  v[p] = val;
  ix[p] = idx;
}

}  // namespace ficoco
