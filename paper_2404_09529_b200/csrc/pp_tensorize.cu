// TENSORIZE (Algorithm 1 (TENSORIZE)) on the device, for the host-buffer entry point: rows of a
// token-major tensor [T, H, D] (prompts back to back in original order) are scattered into the packed
// [R, M, H, D] layout, or gathered back from it. A row is H * D contiguous elements on both sides, so
// this is a row permutation by 16-byte copies; it lets the host side move each tensor with one large
// copy instead of one copy per prompt.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <type_traits>

#include "pp_internal.h"

namespace pp {
namespace {

constexpr int kTzThreads = 256;
constexpr int kTzTokens = 8;    // tokens per block

// map: int64 tok_prefix[n_prompts + 1] (first token of each prompt), then int64 first_row[n_prompts]
// (flat packed row of each prompt's first token).
template <bool kToPacked>
__global__ void __launch_bounds__(kTzThreads)
tensorize_kernel(uint4* __restrict__ packed, uint4* __restrict__ tokens, const int64_t* __restrict__ map,
                 int32_t n_prompts, int64_t total_tokens, int32_t vec_per_row) {
  __shared__ int64_t s_row[kTzTokens];
  const int64_t tok0 = (int64_t)blockIdx.x * kTzTokens;
  if (threadIdx.x < kTzTokens) {
    const int64_t tok = tok0 + threadIdx.x;
    int64_t row = -1;
    if (tok < total_tokens) {
      int32_t lo = 0, hi = n_prompts - 1;           // last prompt whose first token is <= tok
      while (lo < hi) {
        const int32_t mid = (lo + hi + 1) >> 1;
        if (map[mid] <= tok) lo = mid; else hi = mid - 1;
      }
      row = map[n_prompts + 1 + lo] + (tok - map[lo]);
    }
    s_row[threadIdx.x] = row;
  }
  __syncthreads();
  const int units = kTzTokens * vec_per_row;
  for (int u0 = threadIdx.x; u0 < units; u0 += 4 * kTzThreads) {
    uint4 val[4];
    int64_t dst[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int u = u0 + i * kTzThreads;
      dst[i] = -1;
      if (u < units) {
        const int t = u / vec_per_row, w = u - t * vec_per_row;
        const int64_t row = s_row[t];
        if (row >= 0) {
          const int64_t p = row * vec_per_row + w, q = (tok0 + t) * vec_per_row + w;
          val[i] = kToPacked ? tokens[q] : packed[p];
          dst[i] = kToPacked ? p : q;
        }
      }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
      if (dst[i] >= 0) (kToPacked ? packed : tokens)[dst[i]] = val[i];
  }
}

// Zeroes the padding rows [bin_used[b], capacity) of every bin of up to three packed tensors (the
// attention kernels want finite values there); grid = (bins, row chunks).
struct PadTensors {
  uint4* base[3];
  int32_t vec_per_row[3];
};
__global__ void __launch_bounds__(kTzThreads)
zero_pad_rows_kernel(PadTensors t, const int64_t* __restrict__ bin_used, int32_t capacity) {
  const int32_t b = blockIdx.x;
  const int64_t used = bin_used[b];
  const int64_t pad_rows = capacity - used;
  for (int i = 0; i < 3; ++i) {
    if (!t.base[i]) continue;
    const int64_t n = pad_rows * t.vec_per_row[i];
    uint4* dst = t.base[i] + ((int64_t)b * capacity + used) * t.vec_per_row[i];
    for (int64_t u = (int64_t)blockIdx.y * kTzThreads + threadIdx.x; u < n; u += (int64_t)gridDim.y * kTzThreads)
      dst[u] = make_uint4(0u, 0u, 0u, 0u);
  }
}

// A batch in mapped (pinned) host memory: the rows are read and written over the bus by the kernel itself, so one
// launch takes the place of three copies, the zeroing and three scatters (or of a gather and a copy). For a small
// batch those are a queue of 2 us operations (see launch_host_rows); the bus runs at 51 GB/s up and 52 GB/s down this
// way against 55 and 53 of the copy engines.
struct RowTable {
  int32_t off_bin_seg_ptr, off_bin_used, off_seg_start, off_cache_off;
  int32_t capacity, kv_elems;                  // kv_elems: n_kv_heads * head_dim, one token of a token-major cache
  int32_t rows_per_block;                      // at most kTzTokens
  int64_t n_rows;
};
template <bool kToPacked, class Table>
__global__ void __launch_bounds__(kTzThreads)
host_rows_kernel(HostRows h, RowTable m, int32_t q_vec, int32_t kv_vec, const __grid_constant__ Table tab) {
  __shared__ int64_t s_tok[kTzTokens];           // token of each packed row, -1 for padding
  if (!kToPacked && Table::kUploaded) pdl_wait();
  const int64_t row0 = (int64_t)blockIdx.x * m.rows_per_block;
  if (threadIdx.x < m.rows_per_block) {
    const int64_t row = row0 + threadIdx.x;
    int64_t tok = -1;
    if (row < m.n_rows) {
      const int32_t b = (int32_t)(row / m.capacity);
      const int32_t t = (int32_t)(row - (int64_t)b * m.capacity);
      if (t < tab.i32(m.off_bin_used + b)) {
        int32_t lo = tab.i32(m.off_bin_seg_ptr + b), hi = tab.i32(m.off_bin_seg_ptr + b + 1) - 1;
        while (lo < hi) {                        // last prompt that starts at or before the row
          const int32_t mid = (lo + hi + 1) >> 1;
          if (tab.i32(m.off_seg_start + mid) <= t) lo = mid; else hi = mid - 1;
        }
        tok = tab.i64(m.off_cache_off, lo) / m.kv_elems + (t - tab.i32(m.off_seg_start + lo));
      }
    }
    s_tok[threadIdx.x] = tok;
  }
  if (!kToPacked) pdl_wait();
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    if (kToPacked) *h.status = 0; else *h.host_status = *h.status;
  }
  __syncthreads();
  const int per_row = kToPacked ? q_vec + 2 * kv_vec : q_vec;
  const int rows = (int)(m.n_rows - row0 < m.rows_per_block ? m.n_rows - row0 : m.rows_per_block);
  for (int u0 = threadIdx.x; u0 < rows * per_row; u0 += 4 * kTzThreads) {
    uint4 val[4];
    uint4* dst[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int u = u0 + i * kTzThreads;
      dst[i] = nullptr;
      if (u < rows * per_row) {
        const int r = u / per_row, w = u - r * per_row;
        const int64_t tok = s_tok[r], row = row0 + r;
        if (kToPacked) {
          const int which = w < q_vec ? 0 : w < q_vec + kv_vec ? 1 : 2;
          const int vec = which == 0 ? q_vec : kv_vec, c = w - (which == 0 ? 0 : which == 1 ? q_vec : q_vec + kv_vec);
          const uint4* src = static_cast<const uint4*>(which == 0 ? h.q_host : which == 1 ? h.k_host : h.v_host);
          dst[i] = static_cast<uint4*>(which == 0 ? h.q : which == 1 ? h.k : h.v) + row * vec + c;
          val[i] = tok >= 0 ? src[tok * vec + c] : make_uint4(0u, 0u, 0u, 0u);
        } else if (tok >= 0) {
          dst[i] = static_cast<uint4*>(h.o_host) + tok * q_vec + w;
          val[i] = static_cast<const uint4*>(h.o)[row * q_vec + w];
        }
      }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
      if (dst[i]) *dst[i] = val[i];
  }
}


// A table read from mapped host memory. A bus read takes 1 to 2 us whatever its size, so all of a thread's reads are
// issued together, and before the wait for the kernel in front, whose end they overlap.
constexpr int kUploadThreads = 128, kUploadVecs = 4;
__global__ void __launch_bounds__(kUploadThreads)
upload_kernel(uint4* dst, const uint4* src, int32_t n_vec, int32_t tail_words) {
  const int32_t at = blockIdx.x * (kUploadThreads * kUploadVecs) + threadIdx.x;
  uint4 val[kUploadVecs];
#pragma unroll
  for (int i = 0; i < kUploadVecs; ++i)
    if (at + i * kUploadThreads < n_vec) val[i] = __ldcv(src + at + i * kUploadThreads);
  uint32_t word = 0;
  const bool tail = blockIdx.x == 0 && (int)threadIdx.x < tail_words;
  if (tail) word = __ldcv(reinterpret_cast<const uint32_t*>(src + n_vec) + threadIdx.x);
  pdl_wait();                   // the kernel in front may still read the table that was here
#pragma unroll
  for (int i = 0; i < kUploadVecs; ++i)
    if (at + i * kUploadThreads < n_vec) dst[at + i * kUploadThreads] = val[i];
  if (tail) reinterpret_cast<uint32_t*>(dst + n_vec)[threadIdx.x] = word;
}

}  // namespace

int launch_upload(void* dst, const void* src, size_t bytes, void* stream) {
  const int32_t n_vec = (int32_t)(bytes / 16);
  const unsigned grid = (unsigned)(n_vec / (kUploadThreads * kUploadVecs) + 1);
  const cudaError_t e = launch_dependent(upload_kernel, dim3(grid), dim3(kUploadThreads), 0, static_cast<cudaStream_t>(stream),
                                         static_cast<uint4*>(dst), static_cast<const uint4*>(src), n_vec, (int32_t)(bytes % 16 / 4));
  return e == cudaSuccess ? PP_OK : note_cuda_error((int)e, "table upload");
}

int launch_host_rows(bool to_packed, const pp_attn_params& p, int32_t* d_table, const TableLayout& L, const int32_t* inline_table,
                     int32_t off_cache_off, const HostRows& rows, void* stream) {
  RowTable m{L.bin_seg_ptr, L.bin_used, L.seg_start, off_cache_off, p.capacity, p.n_kv_heads * p.head_dim, 1,
             (int64_t)p.n_bins * p.capacity};
  // a bus read takes 1 to 2 us, so few rows are spread over as many blocks as there are
  while (m.rows_per_block < kTzTokens && m.n_rows > (int64_t)m.rows_per_block * kSms * 2) m.rows_per_block *= 2;
  const dim3 grid((unsigned)((m.n_rows + m.rows_per_block - 1) / m.rows_per_block)), block(kTzThreads);
  const int32_t q_vec = p.n_q_heads * p.head_dim / 8, kv_vec = m.kv_elems / 8;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  auto launch = [&](const auto& tab) {
    using Table = std::decay_t<decltype(tab)>;
    if (!to_packed) return launch_dependent(host_rows_kernel<false, Table>, grid, block, 0, s, rows, m, q_vec, kv_vec, tab);
    host_rows_kernel<true, Table><<<grid, block, 0, s>>>(rows, m, q_vec, kv_vec, tab);
    return cudaGetLastError();
  };
  const cudaError_t e = inline_table ? launch(inline_copy(inline_table, (size_t)off_cache_off + 2 * (size_t)inline_table[kHeaderSegments]))
                                     : launch(TableInMemory{d_table});
  return e == cudaSuccess ? PP_OK : note_cuda_error((int)e, "host rows kernel launch");
}

int launch_zero_pad_rows(void* q, void* k, void* v, int32_t q_row_bytes, int32_t kv_row_bytes,
                         const int64_t* d_bin_used, int32_t n_bins, int32_t capacity, void* stream) {
  PadTensors t;
  t.base[0] = static_cast<uint4*>(q); t.base[1] = static_cast<uint4*>(k); t.base[2] = static_cast<uint4*>(v);
  t.vec_per_row[0] = q_row_bytes / 16; t.vec_per_row[1] = t.vec_per_row[2] = kv_row_bytes / 16;
  zero_pad_rows_kernel<<<dim3((unsigned)n_bins, 8), kTzThreads, 0, static_cast<cudaStream_t>(stream)>>>(
      t, d_bin_used, capacity);
  const cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? PP_OK : note_cuda_error((int)e, "padding-row kernel launch");
}

int launch_tensorize(bool to_packed, void* packed, void* tokens, const int64_t* d_map, int32_t n_prompts,
                     int64_t total_tokens, int32_t row_bytes, void* stream) {
  if (total_tokens <= 0) return PP_OK;
  const unsigned grid = (unsigned)((total_tokens + kTzTokens - 1) / kTzTokens);
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  if (to_packed)
    tensorize_kernel<true><<<grid, kTzThreads, 0, s>>>(static_cast<uint4*>(packed), static_cast<uint4*>(tokens),
                                                       d_map, n_prompts, total_tokens, row_bytes / 16);
  else
    tensorize_kernel<false><<<grid, kTzThreads, 0, s>>>(static_cast<uint4*>(packed), static_cast<uint4*>(tokens),
                                                        d_map, n_prompts, total_tokens, row_bytes / 16);
  const cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? PP_OK : note_cuda_error((int)e, "tensorize kernel launch");
}

}  // namespace pp
