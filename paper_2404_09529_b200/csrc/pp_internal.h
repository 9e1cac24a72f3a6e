// Internal declarations shared by the translation units of the prepack-b200 library.
#ifndef PREPACK_B200_PP_INTERNAL_H_
#define PREPACK_B200_PP_INTERNAL_H_

#include <cstddef>
#include <cstdint>

#include "../../include/pp.h"

namespace pp {

constexpr int kTileM = 128;      // query rows per work item (tcgen05 MMA M)
constexpr int kTileN = 128;      // key rows per inner step (tcgen05 MMA N of Q.K^T), shared-stream mode
constexpr int kTileNShort = 64;  // the same in independent-slot mode (short work items)
constexpr int kHeaderInts = 16;  // table header, see build_prefill_tables
constexpr int kHeaderSegments = 4;   // header word with the number of segments
constexpr int kHeaderCounter = 10;   // header word the persistent CTAs draw work indices from
constexpr int kHeaderValueMax = 11;  // header word with the largest |v| (bf16 bits), shared-stream mode; zero in the uploaded table
constexpr int kValueFromNorms = kHeaderValueMax - kHeaderInts;   // that word seen from the norms, which follow the header
constexpr int kItemInts = 16;
constexpr int kSms = 148;        // multiprocessors of a B200, for rules that split work (and size workspaces) on the host alike
                                 // whether or not a device is there; the persistent kernel asks the device
constexpr int kMaxFold = 8;      // most query heads of one KV head folded into the rows of a query tile
constexpr int kMaxNormHeads = 512;   // Hq + Hkv up to which the rotation kernels track the norms (shared memory)

// One entry of the attention work list: two query-tile slots sharing one key/value tile stream.
struct WorkItem {
  int32_t bin;
  int32_t kv_row0;      // first key row of the stream (multiple of the mode's key tile)
  int32_t n_kv_tiles;   // key tiles in the stream
  int32_t q_row0[2];    // first query row of each slot; -1 = slot unused
  int32_t jb1;          // slot 1 takes part in key tiles [jb1, n_kv_tiles)
  int32_t je0;          // slot 0 takes part in key tiles [0, je0)
  int32_t cost;         // (slot, key tile) steps, for longest-first ordering
  int32_t bin_used;     // occupied rows of the bin
  int32_t seg_end;      // one past the bin's last segment index
  int32_t key_lo[2];    // start row of the prompt that holds the slot's first query row
  int32_t seg_first[2]; // segment index of that prompt
  int32_t single_seg;   // bit t set: all real rows of slot t belong to that one prompt
  int32_t reserved;
};

// Offsets (in int32 units) of the blocks inside the prefill table that is built on the host and
// copied to the device workspace.
struct TableLayout {
  int32_t norms = 0;        // [Hkv + Hq] largest |k|^2 per KV head and |q|^2 per query head (float bits), filled by the
                            // rotation kernels (shared-stream mode); zero in the uploaded table
  int32_t bin_seg_ptr = 0;  // [R+1]
  int32_t bin_used = 0;     // [R]   occupied rows per bin
  int32_t seg_start = 0;    // [k]   bin-local first row of each segment
  int32_t items = 0;        // [n_items] WorkItem, longest first
  int32_t n_items = 0;
  int32_t total_ints = 0;
  bool independent_slots = false;   // items are single tiles, drawn by each slot on its own
  bool pair_rows = false;           // shared-stream mode: the two slots are consecutive row tiles of one head
  int64_t rows_used = 0;            // occupied rows of all bins
  int32_t n_segments = 0;           // prompts
  int32_t fold = 1;                 // independent mode: query heads folded into a query tile (128 / fold bin rows each)
};

int validate_packing(int32_t n_bins, int32_t capacity, const int32_t* bin_seg_ptr,
                     const int32_t* seg_start, const int32_t* seg_len, int32_t k);
size_t prefill_table_ints(int32_t n_bins, int32_t capacity, int32_t k, int32_t n_q_heads, int32_t n_kv_heads);
int32_t max_fold(int32_t group);   // largest power of two <= kMaxFold that divides the GQA group
int build_prefill_tables(int32_t n_bins, int32_t capacity, const int32_t* bin_seg_ptr,
                         const int32_t* seg_start, const int32_t* seg_len, int32_t k, int32_t n_q_heads,
                         int32_t n_kv_heads, int32_t* out, size_t out_ints, TableLayout* layout);

// Records a failed CUDA call for pp_last_cuda_error(); returns PP_ERR_CUDA.
int note_cuda_error(int cuda_error, const char* what);

// Kernel launchers (device pointers, stream = cudaStream_t as void*). Return a PP_* status.
// Rotates q and k in place; in the shared-stream mode it also leaves the largest |k|^2 and |q|^2 of every
// head (L.norms) and, unless v is null, the largest |v| (kHeaderValueMax) in the table.
// inline_table (here and below): null, or the host copy of a table that was not uploaded and travels in the
// kernel's parameters; the rotation kernel then resets the work counter in d_table.
int launch_rope(const pp_attn_params& p, int32_t* d_table, const TableLayout& L, const int32_t* inline_table, void* q, void* k,
                const void* v, void* stream);
// rope_table: device [D/4][capacity][2] (cos, sin) pairs, or null. When given, q holds the raw
// queries and the kernel rotates each Q tile in shared memory before use. have_norms: a rotation kernel
// of the same call has filled the norms of the table (of the keys, and without rope_table of the queries).
// caches: null, or the per-prompt V caches, which the kernel fills from the V tiles it loads (independent mode, head_dim
// 128, as many KV heads as query heads).
struct CacheFill {
  void* v_cache;
  int32_t off_true_len, off_cap, off_cache_off;   // per-segment arrays inside the table, as for launch_rope_unpack
};
int launch_attention(const pp_attn_params& p, int32_t* d_table, const TableLayout& L, const int32_t* inline_table,
                     const void* q, const void* k, const void* v, void* o, const void* rope_table,
                     bool have_norms, const CacheFill* caches, int32_t* device_status, void* stream);
// Whether the kernels leave norms and the largest |v| in the table and use them: shared-stream mode, and as many heads
// as the rotation kernels' shared memory has room for.
bool tracks_ranges(const pp_attn_params& p, const TableLayout& L);
// Largest |v| of the packed batch into the table (kHeaderValueMax), where no rotation kernel of the call has read v.
int launch_value_range(const pp_attn_params& p, int32_t* d_table, const TableLayout& L, const void* v, void* stream);
// Fused K rotation + UNPACK; the three offsets locate per-segment arrays inside the table
// (true length, cache capacity: int32; cache element offset: int64). v null: the V caches are filled elsewhere.
// In the shared-stream mode (v is not null there) it also leaves the largest |k|^2 of every KV head (L.norms) and the
// largest |v| (kHeaderValueMax) in the table.
int launch_rope_unpack(const pp_attn_params& p, int32_t* d_table, const TableLayout& L, const int32_t* inline_table,
                       int32_t off_true_len, int32_t off_cap, int32_t off_cache_off, const void* rope_table,
                       void* k, const void* v, void* k_cache, void* v_cache, void* stream);
// Fills rope_table for positions 0 .. capacity-1.
int launch_rope_table(const pp_attn_params& p, void* table, void* stream);
int launch_unpack(const pp_attn_params& p, const int32_t* d_table, int32_t k, int64_t total_tokens,
                  const void* k_rot, const void* v, void* k_cache, void* v_cache, void* stream);

// Row scatter (to_packed) / gather between a token-major tensor [T, row_bytes] and the packed layout.
// d_map: device int64 tok_prefix[n_prompts + 1] followed by first_row[n_prompts].
int launch_tensorize(bool to_packed, void* packed, void* tokens, const int64_t* d_map, int32_t n_prompts,
                     int64_t total_tokens, int32_t row_bytes, void* stream);

// Token-major tensors in mapped host memory <-> packed tensors, by packed row (the row's token is found in the prefill
// table: the cache offsets of its prompt are those of token-major caches). to_packed: q, k, v into the packed tensors,
// padding rows zeroed, *status zeroed. Back: O into the host tensor, *status copied to *host_status.
struct HostRows {
  void *q, *k, *v, *o;                         // packed
  const void *q_host, *k_host, *v_host;
  void* o_host;
  int32_t *status, *host_status;
};
int launch_host_rows(bool to_packed, const pp_attn_params& p, int32_t* d_table, const TableLayout& L, const int32_t* inline_table,
                     int32_t off_cache_off, const HostRows& rows, void* stream);

// Zeroes rows [bin_used[b], capacity) of every bin of the packed q / k / v (null pointers are skipped).
int launch_zero_pad_rows(void* q, void* k, void* v, int32_t q_row_bytes, int32_t kv_row_bytes,
                         const int64_t* d_bin_used, int32_t n_bins, int32_t capacity, void* stream);

int launch_bounded_wait_selftest(int32_t* device_status, uint64_t limit_ns, void* stream);

// A table in mapped host memory (both addresses on 16-byte boundaries) into device memory, up to kUploadKernelBytes.
constexpr size_t kUploadKernelBytes = size_t(1) << 20;
int launch_upload(void* dst, const void* src, size_t bytes, void* stream);

// Unpack table (int32 units): header 4 ints, then token_prefix[k+1], bin_of[k], off_of[k],
// cache_cap[k], cache_off as int64[k] (8-byte aligned).
size_t unpack_table_bytes(int32_t k);

// A table of at most this many ints is not uploaded but handed to the kernels as a parameter (independent mode:
// the shared-stream mode wants words of it zeroed in memory). Without the copy, the gap behind it and the wait
// for it a step of 8 prompts on 4 heads takes 13.5 us instead of 16.9, one of 16 prompts on 32 heads 54 instead
// of 65 (the rotation kernel's look-ups then run under the end of the kernel before). But the block is copied whole at every
// launch of a call that uses it. Steps of n prompts of 16 to 128 tokens on 4 / 4 heads of 64 with a block of 448, 896,
// 1792, 3584 and 7168 ints (us): n = 8 (140 ints) 14.0, 14.2, 14.9, 16.7, 20.5; n = 32 (584) 16.8, 15.4, 16.2, 17.8, 21.5;
// n = 64 (1088) 17.8, 18.0, 17.0, 18.8, 23.9; n = 160 (2628) 26.1, 26.1, 26.1, 23.2, 26.1.
// On 32 / 32 heads of 128, where the kernels are longer than the host: n = 24 (492) 34.0, 31.9, 32.0, 32.0, 32.8; n = 64 (1144)
// 74.1, 73.5, 71.4, 71.4, 71.5.
constexpr int kInlineInts = 896;

#ifdef __CUDACC__
// The prefill table as the kernels see it.
struct TableInMemory {
  static constexpr bool kUploaded = true;      // by a kernel, perhaps: nothing may be read before pdl_wait()
  const int32_t* p;
  __device__ __forceinline__ int32_t i32(int i) const { return __ldg(p + i); }
  __device__ __forceinline__ int4 i128(int i) const { return __ldg(reinterpret_cast<const int4*>(p + i)); }
  __device__ __forceinline__ int64_t i64(int base, int i) const { return __ldg(reinterpret_cast<const long long*>(p + base) + i); }
};
struct alignas(16) TableInline {
  static constexpr bool kUploaded = false;
  int32_t w[kInlineInts];
  __device__ __forceinline__ int32_t i32(int i) const { return w[i]; }
  __device__ __forceinline__ int4 i128(int i) const { return *reinterpret_cast<const int4*>(w + i); }
  __device__ __forceinline__ int64_t i64(int base, int i) const { return *reinterpret_cast<const int64_t*>(w + base + 2 * i); }
};

inline TableInline inline_copy(const int32_t* table, size_t ints) {
  TableInline t;
  for (size_t i = 0; i < (ints < (size_t)kInlineInts ? ints : (size_t)kInlineInts); ++i) t.w[i] = table[i];
  return t;
}

// Programmatic dependent launch. A kernel of the path that is launched with launch_dependent() may
// start while the kernel before it in the stream is still finishing: its blocks are scheduled once
// every block of that kernel has called pdl_launch_dependents() (or exited), run their set-up, and
// block in pdl_wait() until that kernel has completed and its writes are visible. Work queued
// before that kernel has completed by then in any case. Launched the ordinary way, both calls
// do nothing.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

template <typename... KArgs, typename... Args>
inline cudaError_t launch_dependent(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream,
                                    Args&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}
#endif  // __CUDACC__

}  // namespace pp

#endif  // PREPACK_B200_PP_INTERNAL_H_
