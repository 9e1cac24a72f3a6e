// One generation step over the per-prompt caches that UNPACK produced (Section 7 of the prepacking
// paper, "prepacking for generation"): the caches are never padded, so the step reads exactly the
// keys and values every prompt has. Two kernels:
//   decode_kernel            one CTA per (chunk of a prompt's cached keys, KV head): rotates the query heads of
//                            that KV head by the new token's position (= tokens cached so far), scores, online
//                            softmax and P V over the chunk; the CTA of a prompt's last chunk also rotates the
//                            new key, appends k' and v to the caches and attends to them. A prompt of one
//                            chunk gets its O at once, the others leave (m, l, o) of every chunk.
//   decode_combine_kernel    merges the chunks of those prompts into O (launched only if there are any)
//
// Bound: HBM, K and V of every cached token are read once. The arithmetic therefore runs on the tensor cores
// through mma.m16n8k16 with the query heads of a KV head as the N = 8 columns (absent ones are zero): with
// four heads per KV head the dot products of a warp per key row, each summed over 32 lanes by five shuffles,
// took 541 us for 240 k cached tokens, 3.6 times what their 983 MB take to copy. Fragments are read straight
// from global memory (no shared memory in between): the order of the contraction index is free as long as
// both operands use the same, so a thread's 16-byte piece of a K row serves two products, and its 16-byte
// pieces of four V rows (paired with byte permutes) serve eight. P is split into three bf16 numbers (24 bits
// of it), so P V is as exact as with P in fp32.
// Measured, whole step (D = 128): 256 prompts, 240 k cached tokens, 32 / 8 heads 568 -> 165-172 us (decode_kernel 157 us,
// 6.3 TB/s, 97 % of the copy peak); 64 prompts, 17.5 k tokens, 32 / 32 heads 76 -> 59 us (57.5 us); ten prompts, 1009
// tokens 38.5 -> 12.7 us, where the latencies in front of the first product count: the search for the prompt and
// the angles run while the kernel before is finishing (programmatic dependent launch), and the loads of q, k
// and the first keys and values are all issued before any is waited for (16.0 us without the two).
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cfloat>
#include <cmath>

#include "pp_internal.h"

namespace pp {
namespace {

constexpr int kDecodeThreads = 128;     // 4 warps per CTA
constexpr int kDecodeWarps = kDecodeThreads / 32;
constexpr int kMaxGroup = 8;            // query heads per KV head: the N of the tensor-core product
constexpr int kTileKeys = 16;           // keys per warp and step: the M of the score product

// What the kernels know about a prompt. For up to kInlineMany prompts the entries travel in the kernel's
// parameters (a launch takes up to 32 KB of them), so that a step needs no table upload, a copy and a gap in
// the stream in front of it; beyond that they are read from the workspace.
struct DecodePrompt {
  int64_t cache_off;                    // elements
  int32_t length, cap;                  // tokens cached so far, rows of the block
};
struct DecodeArgs {
  const __nv_bfloat16 *q_new, *k_new, *v_new;
  __nv_bfloat16 *o, *k_cache, *v_cache;
  float2* part_ml;                      // [chunk][Hq] (m, l), m in scaled log2 units
  float* part_o;                        // [chunk][Hq][D]
  const DecodePrompt* prompts;          // [k], chunk_ptr: read where the parameters do not hold them
  const int32_t* chunk_ptr;             // [k + 1] first chunk of every prompt
  int32_t n_prompts, n_q_heads, n_kv_heads, group, chunk_keys;
  float scale_log2;
  double inv_freq[64];                  // theta_j = base^(-2j/D), computed in double on the host
};
template <int N>
struct DecodeInline {
  DecodePrompt prompts[N];
  int32_t chunk_ptr[N + 1];
};
template <>
struct DecodeInline<0> {};
constexpr int kInlineFew = 32, kInlineMany = 512;

template <int N>
__device__ __forceinline__ int32_t chunk_ptr_at(const DecodeArgs& a, const DecodeInline<N>& in, int i) {
  if constexpr (N > 0) return in.chunk_ptr[i]; else return __ldg(a.chunk_ptr + i);
}
template <int N>
__device__ __forceinline__ DecodePrompt prompt_at(const DecodeArgs& a, const DecodeInline<N>& in, int i) {
  if constexpr (N > 0) return in.prompts[i]; else return a.prompts[i];
}

__device__ __forceinline__ void mma16816(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                         uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
// 8 x 8 transpose of 16-bit elements across the warp
__device__ __forceinline__ uint32_t transpose8x8(uint32_t x) {
  uint32_t y;
  asm volatile("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(y) : "r"(x));
  return y;
}
// Read once, so not kept in L1. And, like all tensors here, not through the read-only path: this kernel may have started before
// the one in front of it has written them (the rows it appends to the caches, the new token).
__device__ __forceinline__ uint4 load16(const __nv_bfloat16* p) {
  uint4 v;
  asm volatile("ld.global.L1::no_allocate.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
  return v;
}
__device__ __forceinline__ float ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ uint32_t word_of(const uint4& v, int i) { return i == 0 ? v.x : i == 1 ? v.y : i == 2 ? v.z : v.w; }

// Fragments of one 16-key step of a warp. Lane = 4 g + t. K: rows g and g + 8, 16-byte pieces t, t + 4, ...
// of a row. V: rows 2t, 2t + 1, 2t + 8, 2t + 9, the 16-byte piece g of a row (and, at D = 128, piece g + 8).
template <int D>
struct StepK { uint4 r[2][D / 32]; };
template <int D>
struct StepV { uint4 r[4][D / 64]; };

template <int D>
__device__ __forceinline__ void load_k(StepK<D>& f, const __nv_bfloat16* base, int key, int last, int g, int t) {
#pragma unroll
  for (int x = 0; x < 2; ++x) {
    const __nv_bfloat16* p = base + (int64_t)min(key + g + 8 * x, last) * D + 8 * t;   // rows past the chunk: a row of it
#pragma unroll
    for (int i = 0; i < D / 32; ++i) f.r[x][i] = load16(p + 32 * i);
  }
}
template <int D>
__device__ __forceinline__ void load_v(StepV<D>& f, const __nv_bfloat16* base, int key, int last, int g, int t) {
#pragma unroll
  for (int x = 0; x < 4; ++x) {
    const __nv_bfloat16* p = base + (int64_t)min(key + 2 * t + (x & 1) + 8 * (x >> 1), last) * D + 8 * g;
#pragma unroll
    for (int i = 0; i < D / 64; ++i) f.r[x][i] = load16(p + 64 * i);
  }
}

// A maximum over nothing. Finite, so that a score of -inf (a key with an infinite element) weighs nothing beside it.
constexpr float kNoScore = -FLT_MAX;

// The rows past the last real one are copies of it, whose weight is 0: no part of O, not as 0 times an infinity either.
template <int D>
__device__ __forceinline__ void clear_past(StepV<D>& f, int n_real, int t) {
#pragma unroll
  for (int x = 0; x < 4; ++x)
    if (2 * t + (x & 1) + 8 * (x >> 1) >= n_real) {
#pragma unroll
      for (int i = 0; i < D / 64; ++i) f.r[x][i] = make_uint4(0u, 0u, 0u, 0u);
    }
}

template <int D>
struct Softmax {
  float m[2] = {kNoScore, kNoScore};      // running maximum of query heads 2t and 2t + 1 (all lanes of equal t agree)
  float l[2] = {0.f, 0.f};                // this thread's keys' share of the running sum
  float acc[D / 16][4];                   // O^T: product j, rows d (see pv), columns = heads 2t, 2t + 1
};

// Scores of 16 keys against 8 query heads (c: keys g, g + 8 by heads 2t, 2t + 1).
template <int D>
__device__ __forceinline__ void scores(float (&c)[4], const StepK<D>& f, const uint4 (&q)[D / 32]) {
  c[0] = c[1] = c[2] = c[3] = 0.f;
#pragma unroll
  for (int i = 0; i < D / 32; ++i) {
    mma16816(c, f.r[0][i].x, f.r[1][i].x, f.r[0][i].y, f.r[1][i].y, q[i].x, q[i].y);
    mma16816(c, f.r[0][i].z, f.r[1][i].z, f.r[0][i].w, f.r[1][i].w, q[i].z, q[i].w);
  }
}

// Online softmax over the 16 keys (those at or past n_real are hidden); leaves P in c.
template <int D>
__device__ __forceinline__ void softmax_step(Softmax<D>& s, float (&c)[4], float scale, int n_real, int g) {
#pragma unroll
  for (int x = 0; x < 4; ++x) c[x] = g + 8 * (x >> 1) < n_real ? c[x] * scale : -INFINITY;
  float mx[2];
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    mx[h] = fmaxf(c[h], c[2 + h]);
#pragma unroll
    for (int o = 4; o < 32; o <<= 1) mx[h] = fmaxf(mx[h], __shfl_xor_sync(0xffffffffu, mx[h], o));
  }
  if (__any_sync(0xffffffffu, mx[0] > s.m[0] || mx[1] > s.m[1])) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const float m_new = fmaxf(s.m[h], mx[h]);
      const float alpha = ex2(s.m[h] - m_new);           // 0 on the first step
      s.m[h] = m_new;
      s.l[h] *= alpha;
#pragma unroll
      for (int j = 0; j < D / 16; ++j) { s.acc[j][h] *= alpha; s.acc[j][2 + h] *= alpha; }
    }
  }
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    c[h] = ex2(c[h] - s.m[h]);
    c[2 + h] = ex2(c[2 + h] - s.m[h]);
    s.l[h] += c[h] + c[2 + h];
  }
}

// (a, b) cut to bf16, a in the low half.
__device__ __forceinline__ uint32_t truncate_bf16x2(float a, float b) {
  uint32_t y;
  asm("cvt.rz.bf16x2.f32 %0, %1, %2;" : "=r"(y) : "f"(b), "f"(a));
  return y;
}

// O^T += V^T P. Product j: row g is d = 8g + j, row g + 8 is d = 64 + 8g + j (D = 128) or 8g + 4 + j (D = 64).
template <int D>
__device__ __forceinline__ void pv(Softmax<D>& s, const StepV<D>& f, const float (&p)[4]) {
  // P in three parts of 8 bits, cut and not rounded, so that none is negative, and none of a weight above 0 (which is at least
  // 2^-126) is 0: an infinite value then gives an infinity and not a NaN, a finite one up to 2^-125 of itself too much.
  uint32_t b[3][2];
  float r[4] = {p[0], p[1], p[2], p[3]};
  uint32_t least[2];
#pragma unroll
  for (int x = 0; x < 2; ++x) least[x] = (p[2 * x] > 0.f ? 0x0080u : 0u) | (p[2 * x + 1] > 0.f ? 0x00800000u : 0u);
#pragma unroll
  for (int part = 0; part < 3; ++part)
#pragma unroll
    for (int x = 0; x < 2; ++x) {
      const uint32_t cut = truncate_bf16x2(r[2 * x], r[2 * x + 1]);
      const __nv_bfloat162 v = *reinterpret_cast<const __nv_bfloat162*>(&cut);
      const __nv_bfloat162 w = part == 0 ? v : __hmax2_nan(v, *reinterpret_cast<const __nv_bfloat162*>(&least[x]));
      b[part][x] = transpose8x8(*reinterpret_cast<const uint32_t*>(&w));
      const float2 back = __bfloat1622float2(v);
      r[2 * x] -= back.x;
      r[2 * x + 1] -= back.y;
    }
#pragma unroll
  for (int j = 0; j < D / 16; ++j) {
    uint32_t a[4];
#pragma unroll
    for (int x = 0; x < 4; ++x) {      // a0: row g, keys 2t, 2t + 1; a1: row g + 8; a2, a3: the same for keys 2t + 8, 2t + 9
      const int e = (D == 128) ? j : j + 4 * (x & 1), piece = (D == 128) ? (x & 1) : 0;
      const uint32_t k0 = word_of(f.r[2 * (x >> 1)][piece], e >> 1), k1 = word_of(f.r[2 * (x >> 1) + 1][piece], e >> 1);
      a[x] = __byte_perm(k0, k1, (e & 1) ? 0x7632 : 0x5410);
    }
#pragma unroll
    for (int part = 2; part >= 0; --part) mma16816(s.acc[j], a[0], a[1], a[2], a[3], b[part][0], b[part][1]);
  }
}

template <int D, int N>
__global__ void __launch_bounds__(kDecodeThreads, D == 128 ? 3 : 4)
decode_kernel(const __grid_constant__ DecodeArgs a, const __grid_constant__ DecodeInline<N> in) {
  constexpr int kHalf = D / 2;
  __shared__ float s_cos[kHalf], s_sin[kHalf];
  __shared__ __align__(16) __nv_bfloat16 s_q[kMaxGroup + 1][D];       // rotated query heads, then the rotated new key
  __shared__ float s_m[kDecodeWarps][kMaxGroup], s_l[kDecodeWarps][kMaxGroup];
  __shared__ float s_o[kDecodeWarps][kMaxGroup][D];
  const int chunk = blockIdx.x, kvh = blockIdx.y, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int g = lane >> 2, t = lane & 3;
  // An uploaded table is not read before the work in front is done; nor by the combine kernel, which looks at it before its own
  // wait and therefore must not start earlier.
  if constexpr (N == 0) pdl_wait();
  pdl_launch_dependents();              // the combine kernel may set up while this one runs
  int lo = 0, hi = a.n_prompts - 1;     // last prompt whose first chunk is <= chunk
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (chunk_ptr_at(a, in, mid) <= chunk) lo = mid; else hi = mid - 1;
  }
  const int i = lo;
  const int c0 = chunk_ptr_at(a, in, i), n_chunks = chunk_ptr_at(a, in, i + 1) - c0;
  const DecodePrompt pr = prompt_at(a, in, i);
  const int key0 = (chunk - c0) * a.chunk_keys, key_end = min(key0 + a.chunk_keys, pr.length);
  const bool last_chunk = chunk - c0 == n_chunks - 1;
  const int64_t base = pr.cache_off + (int64_t)kvh * pr.cap * D;
  const __nv_bfloat16 *kb = a.k_cache + base, *vb = a.v_cache + base;

  // Everything up to here, and the angles, come from the parameters alone (up to kInlineMany prompts): with a
  // programmatic dependent launch this runs while the kernel before this one is finishing.
  if (tid < kHalf) {      // the position is >= 1; same reduction as the prefill kernels
    const double ang = (double)pr.length * a.inv_freq[tid];
    const double n = rint(ang * 0.15915494309189535);
    double red = fma(-n, 6.283185307179586, ang);
    red = fma(-n, 2.4492935982947064e-16, red);
    float sn, cs;
    sincosf((float)red, &sn, &cs);
    s_cos[tid] = cs;
    s_sin[tid] = sn;
  }
  pdl_wait();
  // heads of the group, zeros for the absent ones, and the new key; four (j, j + D/2) pairs at a time. These and
  // the first step's K and V are all on their way before any of them is used.
  constexpr int kRotUnits = (kMaxGroup + 1) * (kHalf / 4), kRotTrips = (kRotUnits + kDecodeThreads - 1) / kDecodeThreads;
  uint2 lo2[kRotTrips], hi2[kRotTrips];
#pragma unroll
  for (int x = 0; x < kRotTrips; ++x) {
    const int u = tid + x * kDecodeThreads, h = u / (kHalf / 4), j = 4 * (u - h * (kHalf / 4));
    lo2[x] = hi2[x] = make_uint2(0u, 0u);
    if (u < kRotUnits && (h < a.group || (h == kMaxGroup && last_chunk))) {
      const __nv_bfloat16* src = h == kMaxGroup ? a.k_new + ((int64_t)i * a.n_kv_heads + kvh) * D
                                                : a.q_new + ((int64_t)i * a.n_q_heads + kvh * a.group + h) * D;
      lo2[x] = *reinterpret_cast<const uint2*>(src + j);
      hi2[x] = *reinterpret_cast<const uint2*>(src + j + kHalf);
    }
  }
  StepK<D> fk;
  StepV<D> fv;
  int key = key0 + kTileKeys * warp;
  if (key < key_end) {
    load_k<D>(fk, kb, key, key_end - 1, g, t);
    load_v<D>(fv, vb, key, key_end - 1, g, t);
  }
  __syncthreads();
#pragma unroll
  for (int x = 0; x < kRotTrips; ++x) {
    const int u = tid + x * kDecodeThreads, h = u / (kHalf / 4), j = 4 * (u - h * (kHalf / 4));
    if (u >= kRotUnits) break;
    uint32_t* l32 = reinterpret_cast<uint32_t*>(&lo2[x]);
    uint32_t* h32 = reinterpret_cast<uint32_t*>(&hi2[x]);
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      const float2 p = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&l32[e]));
      const float2 y = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&h32[e]));
      const float ca = s_cos[j + 2 * e], sa = s_sin[j + 2 * e], cb = s_cos[j + 2 * e + 1], sb = s_sin[j + 2 * e + 1];
      const __nv_bfloat162 rl = __floats2bfloat162_rn(__fmaf_rn(p.x, ca, -__fmul_rn(y.x, sa)), __fmaf_rn(p.y, cb, -__fmul_rn(y.y, sb)));
      const __nv_bfloat162 rh = __floats2bfloat162_rn(__fmaf_rn(y.x, ca, __fmul_rn(p.x, sa)), __fmaf_rn(y.y, cb, __fmul_rn(p.y, sb)));
      l32[e] = *reinterpret_cast<const uint32_t*>(&rl);
      h32[e] = *reinterpret_cast<const uint32_t*>(&rh);
    }
    *reinterpret_cast<uint2*>(&s_q[h][j]) = lo2[x];
    *reinterpret_cast<uint2*>(&s_q[h][j + kHalf]) = hi2[x];
  }
  __syncthreads();
  uint4 q[D / 32];        // head g, the pieces of a row that this thread's K pieces meet
#pragma unroll
  for (int x = 0; x < D / 32; ++x) q[x] = *reinterpret_cast<const uint4*>(&s_q[g][8 * t + 32 * x]);

  Softmax<D> s;
#pragma unroll
  for (int j = 0; j < D / 16; ++j)
#pragma unroll
    for (int x = 0; x < 4; ++x) s.acc[j][x] = 0.f;
  float c[4];
  // K of the next 16 keys is loaded as soon as the scores of these are there, V after its product, so a warp
  // has 4 to 8 KB in flight (D = 128), three CTAs of four warps per SM 48 to 96 KB.
  while (key < key_end) {
    scores<D>(c, fk, q);
    const int next = key + kTileKeys * kDecodeWarps;
    if (next < key_end) load_k<D>(fk, kb, next, key_end - 1, g, t);
    softmax_step<D>(s, c, a.scale_log2, key_end - key, g);
    if (key_end - key < kTileKeys) clear_past<D>(fv, key_end - key, t);
    pv<D>(s, fv, c);
    if (next < key_end) load_v<D>(fv, vb, next, key_end - 1, g, t);
    key = next;
  }
  if (last_chunk && warp == 0) {        // the new token, as a step with one real key
    const __nv_bfloat16* vn = a.v_new + ((int64_t)i * a.n_kv_heads + kvh) * D;
#pragma unroll
    for (int x = 0; x < 2; ++x)
#pragma unroll
      for (int y = 0; y < D / 32; ++y)
        fk.r[x][y] = x == 0 && g == 0 ? *reinterpret_cast<const uint4*>(&s_q[kMaxGroup][8 * t + 32 * y]) : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
    for (int x = 0; x < 4; ++x)
#pragma unroll
      for (int y = 0; y < D / 64; ++y)
        fv.r[x][y] = x == 0 && t == 0 ? *reinterpret_cast<const uint4*>(vn + 8 * g + 64 * y) : make_uint4(0u, 0u, 0u, 0u);
    scores<D>(c, fk, q);
    softmax_step<D>(s, c, a.scale_log2, 1, g);
    pv<D>(s, fv, c);
    // and its rows of the caches
    const int64_t row = base + (int64_t)pr.length * D;
    if (lane < D / 8) {
      *reinterpret_cast<uint4*>(a.k_cache + row + 8 * lane) = *reinterpret_cast<const uint4*>(&s_q[kMaxGroup][8 * lane]);
      *reinterpret_cast<uint4*>(a.v_cache + row + 8 * lane) = *reinterpret_cast<const uint4*>(vn + 8 * lane);
    }
  }
  // merge the four warps (one without keys has m = kNoScore, l = 0)
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    float l = s.l[h];
#pragma unroll
    for (int o = 4; o < 32; o <<= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
    const int head = 2 * t + h;
    if (head < a.group) {
      if (g == 0) { s_m[warp][head] = s.m[h]; s_l[warp][head] = l; }
#pragma unroll
      for (int j = 0; j < D / 16; ++j) {
        s_o[warp][head][8 * g + j] = s.acc[j][h];
        s_o[warp][head][(D == 128 ? 64 + 8 * g : 8 * g + 4) + j] = s.acc[j][2 + h];
      }
    }
  }
  __syncthreads();
  for (int u = tid; u < a.group * D; u += kDecodeThreads) {
    const int h = u / D, d = u - h * D;
    float mm = s_m[0][h];
#pragma unroll
    for (int w = 1; w < kDecodeWarps; ++w) mm = fmaxf(mm, s_m[w][h]);
    float ll = 0.f, oo = 0.f;
#pragma unroll
    for (int w = 0; w < kDecodeWarps; ++w) {
      const float f = ex2(s_m[w][h] - mm);
      ll += s_l[w][h] * f;
      oo += s_o[w][h][d] * f;
    }
    const int head = kvh * a.group + h;
    if (n_chunks == 1) {
      a.o[((int64_t)i * a.n_q_heads + head) * D + d] = __float2bfloat16_rn(oo / ll);
    } else {
      const int64_t at = (int64_t)chunk * a.n_q_heads + head;
      if (d == 0) a.part_ml[at] = make_float2(mm, ll);
      a.part_o[at * D + d] = oo;
    }
  }
}

// One warp per (prompt, query head); prompts of one chunk are done already.
template <int D, int N>
__global__ void __launch_bounds__(kDecodeThreads)
decode_combine_kernel(const __grid_constant__ DecodeArgs a, const __grid_constant__ DecodeInline<N> in) {
  constexpr int E = D / 32;             // consecutive elements per lane
  const int i = blockIdx.x, head = blockIdx.y * kDecodeWarps + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  const int c0 = chunk_ptr_at(a, in, i), c1 = chunk_ptr_at(a, in, i + 1);
  if (c1 - c0 < 2 || head >= a.n_q_heads) return;
  pdl_wait();                           // the partial results come from the kernel before this one
  float mm = kNoScore, ll = 0.f, oo[E];
#pragma unroll
  for (int e = 0; e < E; ++e) oo[e] = 0.f;
  for (int base = c0; base < c1; base += 32) {           // 32 chunks at a time: one (m, l) per lane
    const int n = min(32, c1 - base);
    const float2 ml = lane < n ? a.part_ml[(int64_t)(base + lane) * a.n_q_heads + head] : make_float2(kNoScore, 0.f);
    float m_new = ml.x;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m_new = fmaxf(m_new, __shfl_xor_sync(0xffffffffu, m_new, o));
    m_new = fmaxf(mm, m_new);
    const float alpha = ex2(mm - m_new), f = ex2(ml.x - m_new);
    mm = m_new;
    float l = ml.y * f;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
    ll = ll * alpha + l;
#pragma unroll
    for (int e = 0; e < E; ++e) oo[e] *= alpha;
    const float* src = a.part_o + ((int64_t)base * a.n_q_heads + head) * D + E * lane;
    const int64_t stride = (int64_t)a.n_q_heads * D;
#pragma unroll 8
    for (int c = 0; c < n; ++c) {
      const float fc = __shfl_sync(0xffffffffu, f, c);
      float p[E];
      if constexpr (E == 4) {
        const float4 x = *reinterpret_cast<const float4*>(src + c * stride);
        p[0] = x.x; p[1] = x.y; p[2] = x.z; p[3] = x.w;
      } else {
        const float2 x = *reinterpret_cast<const float2*>(src + c * stride);
        p[0] = x.x; p[1] = x.y;
      }
#pragma unroll
      for (int e = 0; e < E; ++e) oo[e] += p[e] * fc;
    }
  }
  uint32_t r[E / 2];
#pragma unroll
  for (int e = 0; e < E / 2; ++e) {
    const __nv_bfloat162 x = __floats2bfloat162_rn(oo[2 * e] / ll, oo[2 * e + 1] / ll);
    r[e] = *reinterpret_cast<const uint32_t*>(&x);
  }
  __nv_bfloat16* dst = a.o + ((int64_t)i * a.n_q_heads + head) * D + E * lane;
  if constexpr (E == 4) *reinterpret_cast<uint2*>(dst) = make_uint2(r[0], r[1]);
  else *reinterpret_cast<uint32_t*>(dst) = r[0];
}

// Keys per chunk. Enough (chunk, KV head) CTAs for about four rounds of the three per SM that run at once, so that
// the last round is a small part of the whole; at least one 16-key step for each of the four warps, at most 512 keys (a
// CTA's set-up is then a few per cent of its loads), or 1024 where those make the four rounds too; and more only where a
// very long prompt would otherwise be cut into more pieces than one warp merges quickly. 1024 against 512, whole steps:
// 256 prompts, 240 k cached tokens, 32 / 8 heads 176 -> 169 us, of 893 tokens each 165 -> 156, 32 / 4 heads, 256 of 1786 180 ->
// 165, 16 heads of 64, 256 of 867 168 -> 152; 0.90 to 1.007 on ten more (768 keys as 1024, 1536 and 2048 1 to 4 % longer). Below
// that line even chunks of 513 to 1023 keys made 0.92 to 1.005 of the time of 512 on 25 batches and 1.02 on one (100 prompts of
// 777 tokens on 16 heads of 64): not the same way everywhere, so those batches keep 512.
constexpr int64_t kChunkCtasWanted = kSms * 3 * 4;
constexpr int kMostChunksPerPrompt = 64;

struct DecodeLayout {
  size_t chunk_ptr_off, table_bytes;    // table: prompts, chunk_ptr (uploaded where they do not fit the parameters)
  size_t ml_off, o_off, total_bytes;
  int64_t n_chunks;
  int32_t chunk_keys;
};
int32_t decode_chunk_keys(const pp_attn_params& p, const int32_t* lengths, int32_t k) {
  int64_t total = 0;
  int32_t longest = 0;
  for (int32_t i = 0; i < k; ++i) {
    total += lengths[i];
    longest = std::max(longest, lengths[i]);
  }
  const int64_t unit = kTileKeys * kDecodeWarps;
  const int64_t even = total * p.n_kv_heads / kChunkCtasWanted;
  int64_t keys = even >= 1024 ? 1024 : std::min<int64_t>(std::max<int64_t>(even, 1), 512);
  keys = std::max<int64_t>(keys, ((int64_t)longest + kMostChunksPerPrompt - 1) / kMostChunksPerPrompt);
  return (int32_t)((keys + unit - 1) / unit * unit);
}
DecodeLayout decode_layout(const pp_attn_params& p, const int32_t* lengths, int32_t k, int32_t chunk_keys) {
  DecodeLayout L;
  L.chunk_keys = chunk_keys;
  L.n_chunks = 0;
  for (int32_t i = 0; i < k; ++i) L.n_chunks += ((int64_t)lengths[i] + chunk_keys - 1) / chunk_keys;
  auto up = [](size_t x) { return (x + 255) & ~size_t(255); };
  L.chunk_ptr_off = (size_t)k * sizeof(DecodePrompt);
  L.table_bytes = L.chunk_ptr_off + ((size_t)k + 1) * sizeof(int32_t);
  L.ml_off = up(L.table_bytes);
  L.o_off = up(L.ml_off + (size_t)L.n_chunks * p.n_q_heads * sizeof(float2));
  L.total_bytes = L.o_off + (size_t)L.n_chunks * p.n_q_heads * p.head_dim * sizeof(float);
  return L;
}

void fill_table(const DecodeLayout& L, const int32_t* lengths, int32_t k, const int64_t* cache_off,
                const int32_t* cache_cap, DecodePrompt* prompts, int32_t* chunk_ptr) {
  int32_t c = 0;
  for (int32_t i = 0; i < k; ++i) {
    prompts[i] = DecodePrompt{cache_off[i], lengths[i], cache_cap[i]};
    chunk_ptr[i] = c;
    c += (int32_t)(((int64_t)lengths[i] + L.chunk_keys - 1) / L.chunk_keys);
  }
  chunk_ptr[k] = c;
}

template <int D, int N>
cudaError_t launch_decode(const DecodeArgs& a, const DecodeInline<N>& in, const DecodeLayout& L, cudaStream_t s) {
  const dim3 chunks((unsigned)L.n_chunks, (unsigned)a.n_kv_heads);
  const cudaError_t first = launch_dependent(decode_kernel<D, N>, chunks, dim3(kDecodeThreads), 0, s, a, in);
  if (first != cudaSuccess || L.n_chunks == a.n_prompts) return first;       // one chunk each: O is complete
  const dim3 grid((unsigned)a.n_prompts, (unsigned)((a.n_q_heads + kDecodeWarps - 1) / kDecodeWarps));
  const cudaError_t e = launch_dependent(decode_combine_kernel<D, N>, grid, dim3(kDecodeThreads), 0, s, a, in);
  return e;
}
template <int N>
cudaError_t launch_decode_d(int head_dim, const DecodeArgs& a, const DecodeInline<N>& in, const DecodeLayout& L, cudaStream_t s) {
  return head_dim == 128 ? launch_decode<128, N>(a, in, L, s) : launch_decode<64, N>(a, in, L, s);
}
template <int N>
cudaError_t launch_decode_inline(int head_dim, const DecodeArgs& a, const DecodeLayout& L, const int32_t* lengths, int32_t k,
                                 const int64_t* cache_off, const int32_t* cache_cap, cudaStream_t s) {
  DecodeInline<N> in;
  fill_table(L, lengths, k, cache_off, cache_cap, in.prompts, in.chunk_ptr);
  return launch_decode_d(head_dim, a, in, L, s);
}

int check_decode_params(const pp_attn_params* p) {
  if (!p) return PP_ERR_INVALID_ARG;
  if (p->n_q_heads < 1 || p->n_kv_heads < 1) return PP_ERR_INVALID_ARG;
  if (p->head_dim != 64 && p->head_dim != 128) return PP_ERR_UNSUPPORTED;
  if (p->n_q_heads % p->n_kv_heads != 0 || p->n_q_heads / p->n_kv_heads > kMaxGroup) return PP_ERR_UNSUPPORTED;
  if (p->n_kv_heads > 65535 || p->n_q_heads > 65535) return PP_ERR_UNSUPPORTED;
  if (!(p->rope_base > 0.f) || p->softmax_scale < 0.f) return PP_ERR_INVALID_ARG;
  return PP_OK;
}

}  // namespace
}  // namespace pp

extern "C" size_t pp_decode_workspace_bytes(const pp_attn_params* params, const int32_t* lengths, int32_t k) {
  if (pp::check_decode_params(params) != PP_OK || !lengths || k < 1) return 0;
  for (int32_t i = 0; i < k; ++i)
    if (lengths[i] < 1) return 0;
  // Where a step takes chunks of 1024 keys there is room for chunks of 512: the same prompts a few tokens shorter, across
  // the line between the two, then fit a workspace that was sized for the longer ones. (Not across the smaller steps of
  // the chunks below 512.)
  const int32_t keys = pp::decode_chunk_keys(*params, lengths, k);
  return pp::decode_layout(*params, lengths, k, keys == 1024 ? 512 : keys).total_bytes;
}

extern "C" int pp_decode_step(const pp_attn_params* params, const int32_t* lengths, int32_t k,
                              const void* q_new, const void* k_new, const void* v_new, void* o,
                              void* k_cache, void* v_cache, const int64_t* cache_off, const int32_t* cache_cap,
                              void* workspace, void* host_workspace, size_t workspace_bytes, void* stream) {
  int st = pp::check_decode_params(params);
  if (st != PP_OK) return st;
  if (!lengths || k < 1 || !q_new || !k_new || !v_new || !o || !k_cache || !v_cache || !cache_off || !cache_cap ||
      !workspace || !host_workspace)
    return PP_ERR_INVALID_ARG;
  auto al = [](const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; };
  if (!al(q_new) || !al(k_new) || !al(v_new) || !al(o) || !al(k_cache) || !al(v_cache) ||
      (reinterpret_cast<uintptr_t>(workspace) & 255u))
    return PP_ERR_ALIGNMENT;
  for (int32_t i = 0; i < k; ++i) {
    if (lengths[i] < 1 || cache_cap[i] <= lengths[i]) return PP_ERR_LENGTH;     // room for one more token
    if (cache_off[i] < 0) return PP_ERR_INVALID_ARG;
    if (cache_off[i] % 8 != 0) return PP_ERR_ALIGNMENT;
  }
  const pp::DecodeLayout L = pp::decode_layout(*params, lengths, k, pp::decode_chunk_keys(*params, lengths, k));
  if (L.n_chunks > INT32_MAX / 4) return PP_ERR_UNSUPPORTED;
  if (workspace_bytes < L.total_bytes) return PP_ERR_BUFFER_TOO_SMALL;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  char* ws = static_cast<char*>(workspace);
  pp::DecodeArgs a;
  a.q_new = static_cast<const __nv_bfloat16*>(q_new);
  a.k_new = static_cast<const __nv_bfloat16*>(k_new);
  a.v_new = static_cast<const __nv_bfloat16*>(v_new);
  a.o = static_cast<__nv_bfloat16*>(o);
  a.k_cache = static_cast<__nv_bfloat16*>(k_cache);
  a.v_cache = static_cast<__nv_bfloat16*>(v_cache);
  a.part_ml = reinterpret_cast<float2*>(ws + L.ml_off);
  a.part_o = reinterpret_cast<float*>(ws + L.o_off);
  a.prompts = reinterpret_cast<const pp::DecodePrompt*>(ws);
  a.chunk_ptr = reinterpret_cast<const int32_t*>(ws + L.chunk_ptr_off);
  a.n_prompts = k;
  a.n_q_heads = params->n_q_heads;
  a.n_kv_heads = params->n_kv_heads;
  a.group = params->n_q_heads / params->n_kv_heads;
  a.chunk_keys = L.chunk_keys;
  const float scale = params->softmax_scale > 0.f ? params->softmax_scale : 1.0f / sqrtf((float)params->head_dim);
  a.scale_log2 = scale * 1.4426950408889634f;
  const int half = params->head_dim / 2;
  for (int j = 0; j < 64; ++j)
    a.inv_freq[j] = j < half ? pow((double)params->rope_base, -2.0 * j / (double)params->head_dim) : 0.0;
  cudaError_t e;
  if (k <= pp::kInlineFew) {
    e = pp::launch_decode_inline<pp::kInlineFew>(params->head_dim, a, L, lengths, k, cache_off, cache_cap, s);
  } else if (k <= pp::kInlineMany) {
    e = pp::launch_decode_inline<pp::kInlineMany>(params->head_dim, a, L, lengths, k, cache_off, cache_cap, s);
  } else {
    char* h = static_cast<char*>(host_workspace);
    pp::fill_table(L, lengths, k, cache_off, cache_cap, reinterpret_cast<pp::DecodePrompt*>(h),
                   reinterpret_cast<int32_t*>(h + L.chunk_ptr_off));
    e = cudaMemcpyAsync(workspace, host_workspace, L.table_bytes, cudaMemcpyHostToDevice, s);
    if (e != cudaSuccess) return pp::note_cuda_error((int)e, "decode table upload");
    e = pp::launch_decode_d(params->head_dim, a, pp::DecodeInline<0>{}, L, s);
  }
  return e == cudaSuccess ? PP_OK : pp::note_cuda_error((int)e, "decode kernel launch");
}
