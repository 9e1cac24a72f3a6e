// Restart rotary positional encoding over the packed batch (Section 3.2, Algorithm 1 (RESTART-PE)).
// Each row's position is its bin-local row index minus the start row of the prompt it belongs
// to; Q and K rows are rotated in place. HBM-bound: every element is read once and written once.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <type_traits>

#include "pp_internal.h"

namespace pp {
namespace {

constexpr int kRopeThreads = 256;
constexpr int kRopeRows = 4;        // packed rows per block
constexpr int kMaxHalf = 64;        // head_dim / 2 at most

struct RopeFreq {
  double inv_freq[kMaxHalf];        // theta_j = base^(-2j/D), computed in double on the host
};

__device__ __forceinline__ float2 bf2_to_f2(uint32_t u) {
  __nv_bfloat162 h = *reinterpret_cast<__nv_bfloat162*>(&u);
  return __bfloat1622float2(h);
}
__device__ __forceinline__ uint32_t f2_to_bf2(float a, float b) {
  __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<uint32_t*>(&h);
}

// Rotates the 8 (lower, upper) pairs held in two 16-byte vectors.
__device__ __forceinline__ void rotate8(uint4& lo, uint4& hi, const float* cs, const float* sn) {
  uint32_t* l = reinterpret_cast<uint32_t*>(&lo);
  uint32_t* h = reinterpret_cast<uint32_t*>(&hi);
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const float2 a = bf2_to_f2(l[i]);
    const float2 b = bf2_to_f2(h[i]);
    const float c0 = cs[2 * i], c1 = cs[2 * i + 1], s0 = sn[2 * i], s1 = sn[2 * i + 1];
    // written with explicit fma/mul so that every kernel that rotates gives the same bits
    l[i] = f2_to_bf2(__fmaf_rn(a.x, c0, -__fmul_rn(b.x, s0)), __fmaf_rn(a.y, c1, -__fmul_rn(b.y, s1)));
    h[i] = f2_to_bf2(__fmaf_rn(b.x, c0, __fmul_rn(a.x, s0)), __fmaf_rn(b.y, c1, __fmul_rn(a.y, s1)));
  }
}

// Largest |row|^2 per head, for the bound on the scores that the attention kernel uses (shared-stream
// mode): a (row, head) is held by kLanes neighbouring lanes, each with the sum of squares of its part in
// `part` (>= 0; all lanes of the warp call). Non-negative floats order like their bit patterns.
template <int kLanes>
__device__ __forceinline__ void note_norm(float part, bool real, uint32_t* s_max_of_head) {
#pragma unroll
  for (int o = kLanes / 2; o > 0; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
  if (real && (threadIdx.x & (kLanes - 1)) == 0) atomicMax(s_max_of_head, __float_as_uint(part));
}
__device__ __forceinline__ float sum_squares(const uint4& lo, const uint4& hi) {
  const uint32_t w[8] = {lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z, hi.w};
  float a = 0.f, b = 0.f;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const float2 f = bf2_to_f2(w[i]);
    a = fmaf(f.x, f.x, a);
    b = fmaf(f.y, f.y, b);
  }
  return a + b;
}

// Largest |x| of bf16 pairs, a NaN if there is one.
__device__ __forceinline__ __nv_bfloat162 max_abs(__nv_bfloat162 m, const uint4& x) {
  const uint32_t w[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
  for (int i = 0; i < 4; ++i) m = __hmax2_nan(m, __habs2(*reinterpret_cast<const __nv_bfloat162*>(&w[i])));
  return m;
}
// ... of a warp into *s_max as bits, which order like the values and a NaN above all
__device__ __forceinline__ void note_max_abs(__nv_bfloat162 m2, uint32_t* s_max) {
  const uint32_t bits = *reinterpret_cast<const uint32_t*>(&m2);
  const uint32_t m = __reduce_max_sync(0xffffffffu, max(bits >> 16, bits & 0xffffu));
  if ((threadIdx.x & 31) == 0) atomicMax(s_max, m);
}
// A block's maxima to global memory: s_max[0 .. n) to out[0 .. n), s_max[n] to *out_v.
__device__ __forceinline__ void publish_ranges(const uint32_t* s_max, int n, uint32_t* out, uint32_t* out_v) {
  __syncthreads();
  for (int h = threadIdx.x; h <= n; h += kRopeThreads) {
    uint32_t* dst = h < n ? out + h : out_v;
    if (s_max[h] > __ldcg(dst)) atomicMax(dst, s_max[h]);
  }
}

// Where a kernel finds the segment tables in the prefill table. (One parameter instead of three: each costs a launch about 0.1 us of
// host time, which is what a small batch takes.)
struct SegTables {
  int32_t bin_seg_ptr, bin_used, seg_start;
};

// kRange (shared-stream mode): norms, [Hkv] then [Hq] words, receive the largest |k|^2 / |q|^2 of each head, and the
// word kValueFromNorms before them the largest |v| of the real rows of v (null: not wanted). Reading V here costs its bytes (four prompts of 3000 to 4096
// tokens on 32 / 32 heads of 128, three calls: 638 -> 655 us; as a kernel of its own 633 -> 664).
// counter: null, or the work counter to reset for the attention kernel.
template <int D, bool kRange, class Table>
__global__ void __launch_bounds__(kRopeThreads, 6)
rope_kernel(__nv_bfloat16* __restrict__ q, __nv_bfloat16* __restrict__ k, const __nv_bfloat16* v, uint32_t* norms,
            int32_t* counter, const __grid_constant__ Table tab, SegTables seg, int32_t n_bins, int32_t capacity, int32_t n_q_heads,
            int32_t n_kv_heads, const __grid_constant__ RopeFreq freq) {
  constexpr int kHalf = D / 2;
  constexpr int kUnitsPerHead = kHalf / 8;          // 16-byte vector pairs per head
  __shared__ int32_t s_pos[kRopeRows];              // restart position, -1 for padding rows
  __shared__ float s_cos[kRopeRows][kHalf];
  __shared__ float s_sin[kRopeRows][kHalf];
  __shared__ uint32_t s_norm[kMaxNormHeads + 1];    // [Hkv] of k, then [Hq] of q, then v

  pdl_launch_dependents();      // the attention kernel may set up while this one runs
  if (Table::kUploaded) pdl_wait();
  const int64_t row0 = (int64_t)blockIdx.x * kRopeRows;
  const int64_t n_rows = (int64_t)n_bins * capacity;
  const int tid = threadIdx.x;

  const int n_heads = n_q_heads + n_kv_heads;
  if (kRange)
    for (int h = tid; h <= n_heads; h += kRopeThreads) s_norm[h] = 0u;
  if (tid < kRopeRows) {
    const int64_t row = row0 + tid;
    int32_t pos = -1;
    if (row < n_rows) {
      const int32_t b = (int32_t)(row / capacity);
      const int32_t t = (int32_t)(row - (int64_t)b * capacity);
      if (t < tab.i32(seg.bin_used + b)) {
        // last segment of bin b whose start row is <= t
        int32_t lo = tab.i32(seg.bin_seg_ptr + b), hi = tab.i32(seg.bin_seg_ptr + b + 1) - 1;
        while (lo < hi) {
          const int32_t mid = (lo + hi + 1) >> 1;
          if (tab.i32(seg.seg_start + mid) <= t) lo = mid; else hi = mid - 1;
        }
        pos = t - tab.i32(seg.seg_start + lo);
      }
    }
    s_pos[tid] = pos;
  }
  __syncthreads();

  if (tid < kRopeRows * kHalf) {
    const int r = tid / kHalf, j = tid % kHalf;
    const int32_t pos = s_pos[r];
    float sn = 0.f, cs = 1.f;
    if (pos > 0) {
      // angle in double, reduced to [-pi, pi] before the single-precision sincos, so that the
      // argument error stays ~1e-7 rad even at positions of several 10^4
      const double ang = (double)pos * freq.inv_freq[j];
      const double n = rint(ang * 0.15915494309189535);                 // 1 / (2 pi)
      double red = fma(-n, 6.283185307179586, ang);
      red = fma(-n, 2.4492935982947064e-16, red);                      // low part of 2 pi
      sincosf((float)red, &sn, &cs);
    }
    s_cos[r][j] = cs;
    s_sin[r][j] = sn;
  }
  pdl_wait();
  if (counter && blockIdx.x == 0 && tid == 0) *counter = 0;
  __syncthreads();

  const int units_per_row = n_heads * kUnitsPerHead;
  const int units = kRopeRows * units_per_row;
  for (int u0 = 0; u0 < units; u0 += kRopeThreads) {          // whole warps: the norms are summed across lanes
    const int u = u0 + tid;
    const int r = u / units_per_row;
    const int w = u - r * units_per_row;
    const int32_t pos = u < units ? s_pos[r] : -1;
    const int head = w / kUnitsPerHead;
    const int c = w - head * kUnitsPerHead;
    const int64_t row = row0 + r;
    const bool is_q = head < n_q_heads;
    float n2 = 0.f;
    if (pos > 0 || (kRange && pos == 0)) {                     // padding rows are skipped, position 0 is the identity
      __nv_bfloat16* p = is_q ? q + (row * n_q_heads + head) * D : k + (row * n_kv_heads + (head - n_q_heads)) * D;
      uint4 lo = *reinterpret_cast<const uint4*>(p + c * 8);
      uint4 hi = *reinterpret_cast<const uint4*>(p + kHalf + c * 8);
      if (kRange) n2 = sum_squares(lo, hi);
      if (pos > 0) {
        rotate8(lo, hi, &s_cos[r][c * 8], &s_sin[r][c * 8]);
        *reinterpret_cast<uint4*>(p + c * 8) = lo;
        *reinterpret_cast<uint4*>(p + kHalf + c * 8) = hi;
      }
    }
    if (kRange) note_norm<kUnitsPerHead>(n2, pos >= 0, s_norm + (is_q ? n_kv_heads + head : head - n_q_heads));
  }
  if (kRange) {
    if (v) {
      constexpr int kAtOnce = 4;
      const int vecs = n_kv_heads * (D / 8);
      __nv_bfloat162 m = __float2bfloat162_rn(0.f);
      for (int u0 = tid; u0 < kRopeRows * vecs; u0 += kAtOnce * kRopeThreads) {
        uint4 val[kAtOnce];
#pragma unroll
        for (int i = 0; i < kAtOnce; ++i) {
          const int u = u0 + i * kRopeThreads, r = u / vecs;
          val[i] = u < kRopeRows * vecs && s_pos[r] >= 0 ? reinterpret_cast<const uint4*>(v)[row0 * vecs + u] : make_uint4(0u, 0u, 0u, 0u);
        }
#pragma unroll
        for (int i = 0; i < kAtOnce; ++i) m = max_abs(m, val[i]);
      }
      note_max_abs(m, s_norm + n_heads);
    }
    publish_ranges(s_norm, n_heads, norms, norms + kValueFromNorms);
  }
}

// cos/sin of position * theta_j for every position of a bin, laid out [j / 2][pos][j % 2] as
// (cos, sin) pairs, so that threads working on consecutive rows (positions) read consecutive
// 16-byte pieces. Read by the fused kernels.
__global__ void __launch_bounds__(256)
rope_table_kernel(float2* __restrict__ table, int32_t capacity, int32_t half,
                  const __grid_constant__ RopeFreq freq) {
  pdl_launch_dependents();      // the fused K/V kernel may set up while this one runs
  const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= (int64_t)capacity * half) return;
  const int32_t pos = (int32_t)(idx / half), j = (int32_t)(idx - (int64_t)pos * half);
  float sn = 0.f, cs = 1.f;
  if (pos > 0) {      // same arithmetic as rope_kernel, so both give identical bits
    const double ang = (double)pos * freq.inv_freq[j];
    const double n = rint(ang * 0.15915494309189535);
    double red = fma(-n, 6.283185307179586, ang);
    red = fma(-n, 2.4492935982947064e-16, red);
    sincosf((float)red, &sn, &cs);
  }
  table[((size_t)(j >> 1) * capacity + pos) * 2 + (j & 1)] = make_float2(cs, sn);
}

// (The kernels here read what a kernel in front may still be writing when they start, q, k, v and the cos/sin table, through
// ordinary loads, not through the read-only path.)
//
// Fused K rotation + UNPACK (Algorithm 1 (RESTART-PE to UNPACK) in one pass over K and V): every real packed
// row of K is rotated (cos/sin from the table), written back to the packed tensor (the attention
// kernel reads it there) and into its prompt's K cache; the V row is copied into the V cache.
struct SegExt {                    // per-segment arrays appended to the prefill table
  int32_t off_true_len, off_cap, off_cache_off;   // int32 offsets into the table (cache_off: int64 data)
};

// Packed rows per block of the fused K/V kernel: 8 where a row of K is several KB (many KV heads), 32
// where it is at most 2 KB, so that a block always has tens of KB to move for its set-up cost.
constexpr int kRuRowsWide = 8, kRuRowsNarrow = 32;
constexpr int kRuNarrowRowElems = 1024;   // n_kv_heads * D up to which a row counts as narrow
// ... and only where that still gives every SM a few blocks: a few hundred rows in blocks of 32 leave most of the chip
// idle (448 rows of 4 heads, D = 64: 14 blocks; with 56 blocks of 8 rows and the table as a parameter 5.8 -> 3.3 us).
constexpr int64_t kRuNarrowRows = 32 * kSms * 4;
constexpr int kRuV = 8;      // 16-byte V copies in flight per thread
constexpr int kRuK = 2;      // (lower, upper) K pairs in flight per thread
// kRange: the norms and the largest |v| are wanted (shared-stream mode).
template <int D, int kRuRows, bool kRange, class Table>
__global__ void __launch_bounds__(kRopeThreads)
rope_unpack_kernel(__nv_bfloat16* __restrict__ k, const __nv_bfloat16* v, uint32_t* norms,
                   int32_t* counter, __nv_bfloat16* __restrict__ k_cache, __nv_bfloat16* __restrict__ v_cache,
                   const __grid_constant__ Table tab, SegTables seg, SegExt ext, const float2* rope_table,
                   int32_t n_bins, int32_t capacity, int32_t n_kv_heads) {
  constexpr int kHalf = D / 2;
  constexpr int kPairUnits = kHalf / 8;             // (lower, upper) 16-byte pairs per head
  constexpr int kVecs = D / 8;                      // 16-byte vectors per head
  __shared__ int32_t s_pos[kRuRows];              // restart position, -1 for padding rows
  __shared__ int64_t s_dst[kRuRows];              // cache element offset of (head 0, this position); -1: not cached
  __shared__ int64_t s_head_stride[kRuRows];      // cache_cap * D
  __shared__ float4 s_tab[kRuRows][D / 4];          // (cos, sin) of j = 2g, 2g + 1 at each row's position
  __shared__ uint32_t s_norm[kMaxNormHeads + 1];    // largest |k|^2 of the block's rows, per KV head, then their largest |v|

  pdl_launch_dependents();      // the attention kernel may set up while this one runs
  if (Table::kUploaded) pdl_wait();
  const int64_t row0 = (int64_t)blockIdx.x * kRuRows;
  const int64_t n_rows = (int64_t)n_bins * capacity;
  const int tid = threadIdx.x;
  if (kRange)
    for (int h = tid; h <= n_kv_heads; h += kRopeThreads) s_norm[h] = 0u;
  if (tid < kRuRows) {
    const int64_t row = row0 + tid;
    int32_t pos = -1;
    int64_t dst = -1, stride = 0;
    if (row < n_rows) {
      const int32_t b = (int32_t)(row / capacity);
      const int32_t t = (int32_t)(row - (int64_t)b * capacity);
      if (t < tab.i32(seg.bin_used + b)) {
        int32_t lo = tab.i32(seg.bin_seg_ptr + b), hi = tab.i32(seg.bin_seg_ptr + b + 1) - 1;
        while (lo < hi) {
          const int32_t mid = (lo + hi + 1) >> 1;
          if (tab.i32(seg.seg_start + mid) <= t) lo = mid; else hi = mid - 1;
        }
        pos = t - tab.i32(seg.seg_start + lo);
        if (pos < tab.i32(ext.off_true_len + lo)) {   // rows past the prompt's true length are not cached
          stride = (int64_t)tab.i32(ext.off_cap + lo) * D;
          dst = tab.i64(ext.off_cache_off, lo) + (int64_t)pos * D;
        }
      }
    }
    s_pos[tid] = pos;
    s_dst[tid] = dst;
    s_head_stride[tid] = stride;
  }
  __syncthreads();
  pdl_wait();                   // the rotation table is written by the kernel before this one
  if (counter && blockIdx.x == 0 && tid == 0) *counter = 0;
  // each row's D/2 (cos, sin) pairs once, for all heads: D/4 16-byte loads per row, one per thread
  for (int u = tid; u < kRuRows * (D / 4); u += kRopeThreads) {
    const int r = u / (D / 4), g = u - r * (D / 4);
    const int32_t pos = s_pos[r];
    if (pos > 0) s_tab[r][g] = reinterpret_cast<const float4*>(rope_table)[(size_t)g * (size_t)capacity + pos];
  }

  // V rows first: plain 16-byte copies, kRuV in flight per thread (rows that are attended to but not cached are
  // read for their largest value only)
  const int units_v = v ? n_kv_heads * kVecs : 0;
  __nv_bfloat162 my_v_max = __float2bfloat162_rn(0.f);
  for (int u0 = tid; u0 < kRuRows * units_v; u0 += kRuV * kRopeThreads) {
    uint4 val[kRuV];
    int64_t dsts[kRuV];
#pragma unroll
    for (int i = 0; i < kRuV; ++i) {
      const int u = u0 + i * kRopeThreads;
      dsts[i] = -1;
      if (u < kRuRows * units_v) {
        const int r = u / units_v, w = u - r * units_v;
        if (s_dst[r] >= 0 || (kRange && s_pos[r] >= 0)) {
          const int head = w / kVecs, c = w - head * kVecs;
          val[i] = *reinterpret_cast<const uint4*>(v + ((row0 + r) * n_kv_heads + head) * D + c * 8);
          dsts[i] = !kRange || s_dst[r] >= 0 ? s_dst[r] + head * s_head_stride[r] + c * 8 : -2;
        }
      }
    }
#pragma unroll
    for (int i = 0; i < kRuV; ++i) {
      if (dsts[i] >= 0) *reinterpret_cast<uint4*>(v_cache + dsts[i]) = val[i];
      if (kRange && dsts[i] != -1) my_v_max = max_abs(my_v_max, val[i]);
    }
  }
  __syncthreads();
  // K rows: rotate, write back to the packed tensor and into the cache; two pairs in flight
  const int units_k = n_kv_heads * kPairUnits;
  for (int base_u = 0; base_u < kRuRows * units_k; base_u += kRuK * kRopeThreads) {   // whole warps (norms)
    const int u0 = base_u + tid;
    uint4 lo[kRuK], hi[kRuK];
    int rr[kRuK], hh[kRuK], cc[kRuK];
#pragma unroll
    for (int i = 0; i < kRuK; ++i) {
      const int u = u0 + i * kRopeThreads;
      rr[i] = -1;
      hh[i] = 0;
      if (u < kRuRows * units_k) {
        const int r = u / units_k, w = u - r * units_k;
        if (s_pos[r] >= 0) {
          rr[i] = r; hh[i] = w / kPairUnits; cc[i] = w - hh[i] * kPairUnits;
          const __nv_bfloat16* base = k + ((row0 + r) * n_kv_heads + hh[i]) * D;
          lo[i] = *reinterpret_cast<const uint4*>(base + cc[i] * 8);
          hi[i] = *reinterpret_cast<const uint4*>(base + kHalf + cc[i] * 8);
        }
      }
    }
#pragma unroll
    for (int i = 0; i < kRuK; ++i) {
      if (kRange) note_norm<kPairUnits>(rr[i] < 0 ? 0.f : sum_squares(lo[i], hi[i]), rr[i] >= 0, s_norm + hh[i]);
      if (rr[i] < 0) continue;
      const int r = rr[i], head = hh[i], c = cc[i];
      const int32_t pos = s_pos[r];
      __nv_bfloat16* base = k + ((row0 + r) * n_kv_heads + head) * D;
      if (pos > 0) {
        float cs[8], sn[8];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const float4 t4 = s_tab[r][c * 4 + q];
          cs[2 * q] = t4.x; sn[2 * q] = t4.y; cs[2 * q + 1] = t4.z; sn[2 * q + 1] = t4.w;
        }
        rotate8(lo[i], hi[i], cs, sn);
        *reinterpret_cast<uint4*>(base + c * 8) = lo[i];
        *reinterpret_cast<uint4*>(base + kHalf + c * 8) = hi[i];
      }
      if (s_dst[r] >= 0) {
        __nv_bfloat16* cd = k_cache + s_dst[r] + head * s_head_stride[r];
        *reinterpret_cast<uint4*>(cd + c * 8) = lo[i];
        *reinterpret_cast<uint4*>(cd + kHalf + c * 8) = hi[i];
      }
    }
  }
  if (kRange) {
    note_max_abs(my_v_max, s_norm + n_kv_heads);
    publish_ranges(s_norm, n_kv_heads, norms, norms + kValueFromNorms);
  }
}

// The largest |v| of the occupied rows where no rotation kernel of the call has read V (attention alone). HBM-bound.
// grid = (bins, slices of a bin).
constexpr int kRangeVecs = 8;      // 16-byte loads in flight per thread
__global__ void __launch_bounds__(kRopeThreads)
value_range_kernel(const uint4* v, const TableInMemory tab, int32_t off_bin_used, int32_t capacity, int32_t vec_per_row,
                   uint32_t* v_max) {
  __shared__ uint32_t s_max;
  if (threadIdx.x == 0) s_max = 0u;
  pdl_launch_dependents();
  pdl_wait();
  __syncthreads();
  const int64_t n = (int64_t)tab.i32(off_bin_used + blockIdx.x) * vec_per_row;
  const uint4* src = v + (int64_t)blockIdx.x * capacity * vec_per_row;
  const int64_t stride = (int64_t)gridDim.y * kRopeThreads;
  __nv_bfloat162 m = __float2bfloat162_rn(0.f);
  for (int64_t at = (int64_t)blockIdx.y * kRopeThreads + threadIdx.x; at < n; at += kRangeVecs * stride) {
    uint4 val[kRangeVecs];
#pragma unroll
    for (int i = 0; i < kRangeVecs; ++i) val[i] = at + i * stride < n ? src[at + i * stride] : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
    for (int i = 0; i < kRangeVecs; ++i) m = max_abs(m, val[i]);
  }
  note_max_abs(m, &s_max);
  publish_ranges(&s_max, 0, nullptr, v_max);
}

// Where the kernels leave the norms and the largest |v|: words of the table, or null where nothing uses them.
uint32_t* norm_words(const pp_attn_params& p, int32_t* d_table, const TableLayout& L) {
  return tracks_ranges(p, L) ? reinterpret_cast<uint32_t*>(d_table + L.norms) : nullptr;
}

RopeFreq make_freq(const pp_attn_params& p) {
  RopeFreq freq;
  const int half = p.head_dim / 2;
  for (int j = 0; j < kMaxHalf; ++j)
    freq.inv_freq[j] = j < half ? pow((double)p.rope_base, -2.0 * j / (double)p.head_dim) : 0.0;
  return freq;
}

template <class Table>
int launch_rope_unpack_t(const pp_attn_params& p, int32_t* d_table, const TableLayout& L, const Table& tab, int32_t* counter,
                         const SegExt& ext, const void* rope_table, void* k, const void* v, void* k_cache, void* v_cache,
                         cudaStream_t s) {
  const int64_t n_rows = (int64_t)p.n_bins * p.capacity;
  const bool narrow = p.n_kv_heads * p.head_dim <= kRuNarrowRowElems && n_rows >= kRuNarrowRows;
  const int rows = narrow ? kRuRowsNarrow : kRuRowsWide;
  const unsigned grid = (unsigned)((n_rows + rows - 1) / rows);
  auto launch = [&](auto kernel) {
    return launch_dependent(kernel, dim3(grid), dim3(kRopeThreads), 0, s, (__nv_bfloat16*)k, (const __nv_bfloat16*)v,
                            norm_words(p, d_table, L), counter, (__nv_bfloat16*)k_cache, (__nv_bfloat16*)v_cache, tab,
                            SegTables{L.bin_seg_ptr, L.bin_used, L.seg_start}, ext, (const float2*)rope_table, p.n_bins, p.capacity,
                            p.n_kv_heads);
  };
  cudaError_t e;
  const auto launch_d = [&](auto range) {
    constexpr bool kRange = decltype(range)::value;
    if (p.head_dim == 128)
      return narrow ? launch(rope_unpack_kernel<128, kRuRowsNarrow, kRange, Table>) : launch(rope_unpack_kernel<128, kRuRowsWide, kRange, Table>);
    return narrow ? launch(rope_unpack_kernel<64, kRuRowsNarrow, kRange, Table>) : launch(rope_unpack_kernel<64, kRuRowsWide, kRange, Table>);
  };
  if constexpr (Table::kUploaded)           // (tables as parameters: independent mode only)
    e = tracks_ranges(p, L) ? launch_d(std::true_type{}) : launch_d(std::false_type{});
  else
    e = launch_d(std::false_type{});
  return e == cudaSuccess ? PP_OK : note_cuda_error((int)e, "rope+unpack kernel launch");
}

template <class Table>
int launch_rope_t(const pp_attn_params& p, int32_t* d_table, const TableLayout& L, const Table& tab, int32_t* counter, void* q,
                  void* k, const void* v, cudaStream_t s) {
  const RopeFreq freq = make_freq(p);
  const int64_t n_rows = (int64_t)p.n_bins * p.capacity;
  const unsigned grid = (unsigned)((n_rows + kRopeRows - 1) / kRopeRows);
  auto launch = [&](auto kernel) {
    return launch_dependent(kernel, dim3(grid), dim3(kRopeThreads), 0, s, (__nv_bfloat16*)q, (__nv_bfloat16*)k, (const __nv_bfloat16*)v,
                            norm_words(p, d_table, L), counter, tab, SegTables{L.bin_seg_ptr, L.bin_used, L.seg_start}, p.n_bins,
                            p.capacity, p.n_q_heads, p.n_kv_heads, freq);
  };
  const auto launch_d = [&](auto range) {
    constexpr bool kRange = decltype(range)::value;
    return p.head_dim == 128 ? launch(rope_kernel<128, kRange, Table>) : launch(rope_kernel<64, kRange, Table>);
  };
  cudaError_t e;
  if constexpr (Table::kUploaded)           // (tables as parameters: independent mode only)
    e = tracks_ranges(p, L) ? launch_d(std::true_type{}) : launch_d(std::false_type{});
  else
    e = launch_d(std::false_type{});
  return e == cudaSuccess ? PP_OK : note_cuda_error((int)e, "rope kernel launch");
}

}  // namespace

bool tracks_ranges(const pp_attn_params& p, const TableLayout& L) {
  return !L.independent_slots && p.n_q_heads + p.n_kv_heads <= kMaxNormHeads;
}

int launch_value_range(const pp_attn_params& p, int32_t* d_table, const TableLayout& L, const void* v, void* stream) {
  const int32_t vec_per_row = p.n_kv_heads * p.head_dim / 8;
  // about four blocks per SM, but no slice of a bin shorter than one pass of a block
  const int64_t per_bin = ((int64_t)p.capacity * vec_per_row + kRopeThreads * kRangeVecs - 1) / (kRopeThreads * kRangeVecs);
  const int64_t wanted = (4 * kSms + (int64_t)p.n_bins - 1) / p.n_bins;
  const unsigned slices = (unsigned)std::min<int64_t>(std::min(per_bin, wanted), 65535);
  const cudaError_t e = launch_dependent(value_range_kernel, dim3((unsigned)p.n_bins, slices), dim3(kRopeThreads), 0,
                                         static_cast<cudaStream_t>(stream), static_cast<const uint4*>(v), TableInMemory{d_table},
                                         L.bin_used, p.capacity, vec_per_row, norm_words(p, d_table, L) + kValueFromNorms);
  return e == cudaSuccess ? PP_OK : note_cuda_error((int)e, "value range kernel launch");
}

int launch_rope_table(const pp_attn_params& p, void* table, void* stream) {
  const RopeFreq freq = make_freq(p);
  const int half = p.head_dim / 2;
  const int64_t n = (int64_t)p.capacity * half;
  rope_table_kernel<<<(unsigned)((n + 255) / 256), 256, 0, static_cast<cudaStream_t>(stream)>>>(
      static_cast<float2*>(table), p.capacity, half, freq);
  const cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? PP_OK : note_cuda_error((int)e, "rope table kernel launch");
}

int launch_rope_unpack(const pp_attn_params& p, int32_t* d_table, const TableLayout& L, const int32_t* inline_table,
                       int32_t off_true_len, int32_t off_cap, int32_t off_cache_off, const void* rope_table,
                       void* k, const void* v, void* k_cache, void* v_cache, void* stream) {
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const SegExt ext{off_true_len, off_cap, off_cache_off};
  if (inline_table)      // the per-segment arrays lie behind the work list, the cache offsets last
    return launch_rope_unpack_t(p, d_table, L, inline_copy(inline_table, (size_t)off_cache_off + 2 * (size_t)inline_table[kHeaderSegments]),
                                d_table + kHeaderCounter, ext, rope_table, k, v, k_cache, v_cache, s);
  return launch_rope_unpack_t(p, d_table, L, TableInMemory{d_table}, nullptr, ext, rope_table, k, v, k_cache, v_cache, s);
}

int launch_rope(const pp_attn_params& p, int32_t* d_table, const TableLayout& L, const int32_t* inline_table, void* q, void* k,
                const void* v, void* stream) {
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  if (inline_table)
    return launch_rope_t(p, d_table, L, inline_copy(inline_table, (size_t)L.total_ints), d_table + kHeaderCounter, q, k, v, s);
  return launch_rope_t(p, d_table, L, TableInMemory{d_table}, nullptr, q, k, v, s);
}

}  // namespace pp
