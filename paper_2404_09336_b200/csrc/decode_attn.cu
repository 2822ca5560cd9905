// Split-KV decode attention over a KV index list (ssa_decode_attn_sparse) or
// over the full context (ssa_decode_attn_dense).
//
// Pass 1 (decode_partial_kernel): grid (chunk, head, request).  A block owns
// `chunk` consecutive entries of the request's index list (dense: `chunk`
// consecutive positions).  A cache row of D 16-bit values is read by a group
// of D/16 lanes, 32 bytes per lane (one 256-bit load where the cache is
// 32-byte aligned, else two 128-bit loads), so a warp covers 32/(D/16) rows
// per load and every 32-byte sector of a selected row is fetched exactly once.
// A warp keeps a tile of kU such loads of K and kU of V in flight, then
// reduces the kU dot products across each lane group with shuffles and folds
// them into a running (max, sum, accumulator) triple - the online form of the
// softmax.  The arithmetic is packed: two fp32 lanes per FMA (fma.rn.f32x2).
// Lane groups never talk to one another until the block ends, where their
// triples are combined through shared memory.  With one chunk per request the
// block normalises and stores the output itself; otherwise it stores the
// unnormalised triple to the workspace and
// Pass 2 (decode_merge_kernel) combines the chunks of one (request, head).
//
// The attended rows of a block come from one of four sources (kMode): every
// position (dense), a slice of the request's index list, a run of entries
// of the request's blocked (block index, bitmask) list, whose set bits the
// block expands into positions in shared memory before reading any row, or
// the request's span list itself, which the block sorts and merges in shared
// memory and turns into positions by arithmetic (no index list anywhere).
#include <algorithm>
#include <atomic>
#include <type_traits>

#include "fetch_index.cuh"
#include "span_merge.cuh"
#include "ssa_common.cuh"

namespace ssa {

#ifndef SSA_WARPS
#define SSA_WARPS 4
#endif
#ifndef SSA_U
#define SSA_U 4
#endif
#ifndef SSA_MIN_BLOCKS
#define SSA_MIN_BLOCKS 4
#endif

constexpr int kSmallBlock = SSA_WARPS; // warps per block in pass 1, where blocks are many; see block_warps for larger ones
constexpr int kWarpSlots = SSA_WARPS * SSA_MIN_BLOCKS;   // warps of an SM
constexpr int kMaxChunk = 512;         // index entries staged per block
constexpr int kMaxWideChunk = 1024;    // ... of more than kSmallBlock warps
__host__ __device__ constexpr int staged_entries(int warps) { return warps > kSmallBlock ? kMaxWideChunk : kMaxChunk; }
constexpr int kMaskChunk = 512;        // positions a block expands from bitmasks
enum { kDense = 0, kIndex = 1, kBlockMask = 2, kSpans = 3 };

struct DecodeParams {
  const void* q_host;       // kHostQ only: the query rows in page-locked host memory the device addresses; every
                            // block fetches its own row across the bus and leaves a copy at q
  const void* q;
  const void* k;
  const void* v;
  const int32_t* ctx_lens;
  const int32_t* index;     // sparse only
  const int32_t* counts;    // list lengths: index entries or listed blocks (NULL selects the dense count)
  const int32_t* block_idx; // blocked list only
  const uint32_t* block_mask;
  int32_t block_size, block_stride;
  const int32_t* span_offsets;  // span lists only: [B+1]
  const int2* spans;            //   (start, end) pairs
  int32_t span_cap;             //   spans taken per request (<= kDirectSpans)
  int32_t spans_readable;       //   pairs that may be read from `spans` on before their offsets can be trusted (0: none)
  int32_t* index_out;           //   optional copy of the positions, [B, index_stride]
  int32_t* counts_out;          //   optional number of positions per request
  int32_t* ws_counts;           //   the same for the second pass (when n_chunks > 1)
  void* out;
  float* lse;
  float* ws_acc;            // [B*H*n_chunks, D]
  float2* ws_ml;            // [B*H*n_chunks]  (max in log2 units, sum)
  uint32_t* dev_status;
  int64_t q_sb, q_sh, k_sb, k_sh, v_sb, v_sh, o_sb, o_sh;
  uint32_t k_row_bytes, v_row_bytes;   // token stride of the cache in bytes
  int32_t H, max_ctx, index_stride, max_selected, chunk, n_chunks, out_f32, early_release;
  int32_t early_blocks, guess_blocks;   // see plan_early
  int16_t early_rows, early_warps;
  int32_t kv_group;         // query heads per K/V head (1: multi-head attention)
  int16_t warps;            // warps of a one-head block
  uint8_t share_rows;       // row-sharing kernel (otherwise one query head per block)
  uint8_t gqa_wide;         // row-sharing kernel, one large block per SM
  int32_t head_splits;      // row-sharing kernel: blocks that share the heads of a group, heads_per_block each
  int32_t heads_per_block;
  int32_t even_blocks;      // row-sharing kernel over full contexts: blocks that share the rows evenly (0: fixed chunks)
  int32_t even_factor;      // ... unless the lengths make slices of `chunk` rows the better cut (even_by_slices)
  int32_t B;
  // paged cache (page_table != nullptr): logical position t of request b is row
  // page_table[b * page_table_stride + (t >> page_shift)] << page_shift | (t & page_mask) of the pool
  const int32_t* page_table;
  int32_t page_table_stride, page_shift, page_mask, n_pages;
  float scale_log2;         // softmax scale * log2(e)
};

// Number of list entries (dense: positions) of request b, clamped to what the
// host sized the launch for.
__device__ __forceinline__ void request_sizes(const DecodeParams& p, int b, int& n, int& c,
                                              uint32_t& flags) {
  n = p.ctx_lens[b];
  if (n > p.max_ctx) { n = p.max_ctx; flags |= SSA_DEV_BAD_COUNT; }
  if (n < 0) n = 0;
  if (p.counts) {
    c = p.counts[b];
    if (c > p.max_selected) { c = p.max_selected; flags |= SSA_DEV_BAD_COUNT; }
    if (c < 0) c = 0;
  } else {
    c = n;
  }
}

template <typename T>
__device__ __forceinline__ void store_out(const DecodeParams& p, int b, int h, int d, float val) {
  const int64_t o = (int64_t)b * p.o_sb + (int64_t)h * p.o_sh + d;
  if (p.out_f32) reinterpret_cast<float*>(p.out)[o] = val;
  else reinterpret_cast<T*>(p.out)[o] = from_float<T>(val);
}

// Element d of a finished row and, with d = 0, its lse.  No attended row (L is exactly 0): zeros and -inf.  A NaN among
// the scores has made L a NaN, which must reach both.
template <typename T>
__device__ __forceinline__ void store_row_value(const DecodeParams& p, int b, int h, int d, float M, float L, float A) {
  store_out<T>(p, b, h, d, L == 0.f ? 0.f : A / L);
  if (d == 0 && p.lse) p.lse[(int64_t)b * p.H + h] = L == 0.f ? neg_inf() : (M + log2f(L)) * kLn2;
}

// The same for elements d..d + 3, d a multiple of four (rows start on 16 bytes: check_desc).
template <typename T>
__device__ __forceinline__ void store_row_values(const DecodeParams& p, int b, int h, int d, float M, float L, const float (&A)[4]) {
  const int64_t o = (int64_t)b * p.o_sb + (int64_t)h * p.o_sh + d;
  float r[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) r[i] = L == 0.f ? 0.f : A[i] / L;
  if (p.out_f32) {
    *reinterpret_cast<float4*>(reinterpret_cast<float*>(p.out) + o) = make_float4(r[0], r[1], r[2], r[3]);
  } else {
    const T x[4] = {from_float<T>(r[0]), from_float<T>(r[1]), from_float<T>(r[2]), from_float<T>(r[3])};
    uint2 w;
    w.x = (uint32_t)*reinterpret_cast<const uint16_t*>(&x[0]) | (uint32_t)*reinterpret_cast<const uint16_t*>(&x[1]) << 16;
    w.y = (uint32_t)*reinterpret_cast<const uint16_t*>(&x[2]) | (uint32_t)*reinterpret_cast<const uint16_t*>(&x[3]) << 16;
    *reinterpret_cast<uint2*>(reinterpret_cast<T*>(p.out) + o) = w;
  }
  if (d == 0 && p.lse) p.lse[(int64_t)b * p.H + h] = L == 0.f ? neg_inf() : (M + log2f(L)) * kLn2;
}

// A lane's piece of a cache row: 16 values as eight pairs.  16-bit storage: 32 bytes, a pair per word; 8-bit
// storage: 16 bytes in w[0..3], two pairs per word.
struct Piece { uint32_t w[8]; };

// A cache row is used once per launch, so the 256-bit loads mark its lines evict-first in L2 as well: they then
// do not push out what is re-read (index lists, query rows, partial results).  Measured: 4-5 % off every workload
// (cfg 2 attention 32.4 -> 30.7 us, full context at cfg 2 105 -> 100.5 us); prefetch-size hints on top: nothing.
// (The qualifier exists for 256-bit loads only, so the 128-bit fallback keeps the default L2 policy.)
template <bool kAligned32, bool kFp8 = false>
__device__ __forceinline__ void load_piece(Piece& r, const char* p) {
  if (kFp8) {
    const uint4 a = ld_stream_16B(p);
    r.w[0] = a.x; r.w[1] = a.y; r.w[2] = a.z; r.w[3] = a.w;
    r.w[4] = 0u; r.w[5] = 0u; r.w[6] = 0u; r.w[7] = 0u;
  } else if (kAligned32) {
    asm volatile("ld.global.nc.L1::no_allocate.L2::evict_first.v8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(r.w[0]), "=r"(r.w[1]), "=r"(r.w[2]), "=r"(r.w[3]),
                   "=r"(r.w[4]), "=r"(r.w[5]), "=r"(r.w[6]), "=r"(r.w[7])
                 : "l"(p));
  } else {
    const uint4 a = ld_stream_16B(p), b = ld_stream_16B(p + 16);
    r.w[0] = a.x; r.w[1] = a.y; r.w[2] = a.z; r.w[3] = a.w;
    r.w[4] = b.x; r.w[5] = b.y; r.w[6] = b.z; r.w[7] = b.w;
  }
}

// Pair i (0..7) of a piece as two floats.
template <typename T>
__device__ __forceinline__ float2 piece_pair(const Piece& r, int i) {
  if constexpr (kIsFp8<T>) return e4m3x2_to_float2(r.w[i >> 1] >> ((i & 1) * 16));
  else return unpack2<T>(r.w[i]);
}

__device__ __forceinline__ void zero_piece(Piece& r) {
#pragma unroll
  for (int i = 0; i < 8; ++i) r.w[i] = 0u;
}

// Over the lanes of a warp that hold the same dims (lane groups of kLanesPerRow): largest value, sum.
template <int kLanesPerRow>
__device__ __forceinline__ float lane_groups_max(float v) {
#pragma unroll
  for (int o = kLanesPerRow; o < 32; o <<= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}
template <int kLanesPerRow>
__device__ __forceinline__ float lane_groups_sum(float v) {
#pragma unroll
  for (int o = kLanesPerRow; o < 32; o <<= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
// Lanes kBit apart hold 2 N pairs of the same dims: the sums of the first N to the lane without that bit, of the last to the other.
template <int kBit, int N>
__device__ __forceinline__ void halve_between(float2 (&out)[N], const float2 (&in)[2 * N], int lane) {
  const bool upper = lane & kBit;
#pragma unroll
  for (int i = 0; i < N; ++i) {
    const float2 keep = upper ? in[i + N] : in[i], give = upper ? in[i] : in[i + N];
    out[i].x = keep.x + __shfl_xor_sync(0xffffffffu, give.x, kBit);
    out[i].y = keep.y + __shfl_xor_sync(0xffffffffu, give.y, kBit);
  }
}

// Called before grid_dependency_wait() by each of the first p.early_warps warps of a block: they ask for the first p.early_rows rows of the
// block in L2, by the lists as they stand.  Neighbouring lanes take the
// sectors of a row: with a row per lane the requests took four times as long to issue.  (Lists, counts, lengths and page tables are
// read where the host says they are, and no further; what they name is checked against max_ctx and n_pages.)
// kSpans: the warp has the request's runs in `runs` (runs_p of them, n and c positions).
template <typename T, int D, int kMode, bool kPaged>
__device__ __forceinline__ void prefetch_early(const DecodeParams& p, int b, int kvh, int start, int warp,
                                               const WarpRuns* runs = nullptr, int runs_p = 0, int n_of_spans = 0, int c_of_spans = 0) {
  constexpr int kSectors = D * (int)sizeof(T) / 32, kRows = 32 / kSectors;   // of a row; rows an instruction covers
  const int lane = threadIdx.x & 31;
  const char* const krows =
      reinterpret_cast<const char*>(reinterpret_cast<const T*>(p.k) + (int64_t)b * p.k_sb + (int64_t)kvh * p.k_sh);
  const char* const vrows =
      reinterpret_cast<const char*>(reinterpret_cast<const T*>(p.v) + (int64_t)b * p.v_sb + (int64_t)kvh * p.v_sh);
  const bool listed = kMode == kIndex && (!kPaged || p.index != nullptr);
  const int n = kMode == kSpans ? n_of_spans : min(load_early(p.ctx_lens + b), p.max_ctx);
  const int c = kMode == kSpans ? c_of_spans : min(p.counts ? load_early(p.counts + b) : n, p.max_selected);
  const int rows = min(p.early_rows, min(p.chunk, p.max_selected - start));
  for (int r0 = 32 * warp; r0 < rows; r0 += 32 * p.early_warps) {
    const int r = r0 + lane;
    int pos = -1;
    if (r < rows) {
      if constexpr (kMode == kSpans) pos = start + r < c ? span_position(*runs, runs_p, start + r) : -1;
      else pos = listed ? load_early(p.index + (int64_t)b * p.index_stride + start + r) : start + r;
      if (start + r >= c) pos = -1;
    }
    if (pos < 0 || pos >= n) pos = -1;
    if (kPaged && pos >= 0) {
      const int page = load_early(p.page_table + (int64_t)b * p.page_table_stride + (pos >> p.page_shift));
      pos = (unsigned)page < (unsigned)p.n_pages ? (page << p.page_shift) | (pos & p.page_mask) : -1;
    }
#pragma unroll
    for (int i = 0; i < 32; i += kRows) {
      const int row = __shfl_sync(0xffffffffu, pos, i + lane / kSectors);
      if (row >= 0) {
        prefetch_sector(krows + (uint64_t)(uint32_t)row * p.k_row_bytes + lane % kSectors * 32);
        prefetch_sector(vrows + (uint64_t)(uint32_t)row * p.v_row_bytes + lane % kSectors * 32);
      }
    }
  }
}

// kPaged (index lists only): positions are translated through the page table while they are staged, and a
// missing list stands for 0, 1, 2, ...; kept out of the unpaged instantiations so that they stay as they are.
// kHostQ (index lists, one chunk per request): the query rows are still in page-locked host memory.  Each block
// asks for its row (D/8 threads, 16 bytes each) before anything else, so that the trip across the bus overlaps
// the block's start-up, shares it through shared memory and writes the device copy the caller expects at q.
// kWarps: see block_warps.
// kGuess (span lists): the lists are merged before the wait (see plan_early for who does without).
template <typename T, int D, int kMode, bool kAligned32, bool kPaged = false, bool kHostQ = false, int kWarps = kSmallBlock,
          bool kGuess = kMode == kSpans>
__global__ void __launch_bounds__(kWarps * 32, kWarpSlots / kWarps)
decode_partial_kernel(const DecodeParams p) {
  constexpr int kThreads = kWarps * 32, kStage = staged_entries(kWarps);
  constexpr int kIdxPerThread = kStage / kThreads;
  constexpr bool kWide = kWarps > kSmallBlock;
  static_assert(!kPaged || kMode == kIndex, "a paged cache is read through staged positions");
  static_assert(!kHostQ || (kMode == kIndex && !kPaged), "host-resident queries: plain index lists only");
  using TQ = typename Storage<T>::Query;              // type of the query rows and of a stored output
  constexpr bool kFp8 = kIsFp8<T>;
  constexpr int kU = kFp8 ? 2 * SSA_U : SSA_U;        // pieces in flight per lane and tensor; 8-bit ones are half as large
  constexpr bool kSparse = kMode != kDense;           // positions come from shared memory
  constexpr int kLanesPerRow = D / 16;                // 32-byte pieces per row
  constexpr int kRowsPerLoad = 32 / kLanesPerRow;     // rows one warp-wide load covers
  constexpr int kTileRows = kRowsPerLoad * kU;        // rows per warp per iteration
  constexpr int kGroups = kWide ? kWarps : kWarps * kRowsPerLoad;   // triples the block combines
  static_assert(kThreads >= D, "the epilogue uses one thread per output element");
  static_assert(kStage == kIdxPerThread * kThreads && (32 * kIdxPerThread) % kTileRows == 0, "a warp stages whole tiles");
  static_assert(kMaskChunk / 32 <= 32 && kMaskChunk / 32 >= kWarps, "a lane per word of the bitmasks");

  __shared__ int32_t s_idx[kSparse ? kStage : 1];
  __shared__ __align__(16) float s_acc[kGroups][D];
  __shared__ float s_m[kGroups], s_l[kGroups];
  __shared__ typename std::conditional<kMode == kSpans, SpanRuns, int>::type s_runs;
  __shared__ typename std::conditional<kMode == kSpans, WarpRuns, int>::type s_wruns[kMode == kSpans ? kWarps : 1];
  __shared__ uint4 s_qrow[kHostQ ? D / 8 : 1];

  const int chunk_id = blockIdx.x, h = blockIdx.y, b = blockIdx.z;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int col = lane % kLanesPerRow, sub = lane / kLanesPerRow;
  const int start = chunk_id * p.chunk;

  // (kHostQ: the query row, across the bus, comes first.  Blocked lists have mostly been made by the launch in front, which
  // leaves no time, and take two trips: 52 requests of 32 heads, six rows each, 14.0 / 16.0 us)
  if constexpr ((kMode == kIndex || kMode == kDense) && kWarps == kSmallBlock && !kHostQ)
    if (warp < p.early_warps && blockIdx.x + gridDim.x * (blockIdx.y + gridDim.y * blockIdx.z) < (unsigned)p.early_blocks)
      prefetch_early<T, D, kMode, kPaged>(p, b, h / p.kv_group, start, warp);
  // span lists of up to 32: blocks that wait merge them meanwhile, and see afterwards whether that still holds
  const bool warp_merge = kMode == kSpans && p.span_cap <= 32;
  int warp_runs = 1;                                  // span_cap rounded up to a power of two
  while (warp_merge && warp_runs < p.span_cap) warp_runs <<= 1;
  EarlySpans guess;
  guess.there = false;
  if constexpr (kGuess) {
    const unsigned block = blockIdx.x + gridDim.x * (blockIdx.y + gridDim.y * blockIdx.z);
    if (warp_merge && p.spans_readable > 0 && block < (unsigned)p.guess_blocks) {
      guess = merge_spans_early(s_wruns[warp], p.span_offsets, p.spans, p.spans_readable, p.ctx_lens, p.max_ctx, b, p.span_cap, warp_runs);
      if (guess.there && warp < p.early_warps && block < (unsigned)p.early_blocks)
        prefetch_early<T, D, kSpans, false>(p, b, h / p.kv_group, start, warp, &s_wruns[warp], warp_runs, guess.n,
                                            min(guess.total, p.max_selected));
    }
  }
  grid_dependency_wait();
  if (p.early_release) grid_launch_dependents();      // small grid: let the next kernel's blocks move in now

  uint4 q_word = make_uint4(0u, 0u, 0u, 0u);          // kHostQ: this thread's 16 bytes of the query row
  if constexpr (kHostQ) {
    if (tid < D / 8)
      q_word = *(reinterpret_cast<const uint4*>(reinterpret_cast<const TQ*>(p.q_host) + (int64_t)b * p.q_sb +
                                                (int64_t)h * p.q_sh) + tid);
  }

  // Everything the block needs before it can request cache rows is loaded
  // here in one go: sizes, its slice of the index list, the query row.
  // A warp stages exactly the list entries of its own tiles (entry i of the
  // warp's share is row staged_row(i) of the block), so staging needs no block
  // barrier, only a warp one.
  auto staged_row = [&](int i) {
    return warp * kTileRows + (i / kTileRows) * (kWarps * kTileRows) + (i % kTileRows);
  };
  int32_t raw[kIdxPerThread];
  if (kMode == kIndex) {
    const bool listed = !kPaged || p.index != nullptr;
    const int32_t* row = listed ? p.index + (int64_t)b * p.index_stride + start : nullptr;
#pragma unroll
    for (int j = 0; j < kIdxPerThread; ++j) {
      const int r = staged_row(lane + 32 * j);
      raw[j] = (r < p.chunk && start + r < p.max_selected) ? (listed ? __ldg(row + r) : start + r) : -1;
    }
  }
  Piece qraw;                                         // re-read by every warp and chunk of the head: plain L2 policy
  if constexpr (!kHostQ) {
    const char* qp = reinterpret_cast<const char*>(
        reinterpret_cast<const TQ*>(p.q) + (int64_t)b * p.q_sb + (int64_t)h * p.q_sh + col * 16);
    const uint4 a = ld_stream_16B(qp), c4 = ld_stream_16B(qp + 16);
    qraw.w[0] = a.x; qraw.w[1] = a.y; qraw.w[2] = a.z; qraw.w[3] = a.w;
    qraw.w[4] = c4.x; qraw.w[5] = c4.y; qraw.w[6] = c4.z; qraw.w[7] = c4.w;
  }

  // span lists: where the request's list is; with up to 32 spans every lane asks for "its" span right away (a
  // fixed-stride table needs no offsets, so the spans then arrive together with the sizes and the query)
  int span_first = 0, span_n = 0;
  int2 my_span = make_int2(0, 0);
  if constexpr (kMode == kSpans) {
    if (guess.there && lane < guess.S) my_span = load_now(p.spans + guess.first + lane);
    if (p.span_offsets) {
      span_first = load_now(p.span_offsets + b);
      span_n = load_now(p.span_offsets + b + 1) - span_first;
    } else {
      span_first = b * p.span_cap;
      span_n = p.span_cap;
    }
    if (!kGuess && warp_merge && lane < min(span_n, p.span_cap)) my_span = load_now(p.spans + span_first + lane);
  }
  // blocked lists: every warp takes all words of the block's entries, one per lane (those beyond the list are ignored below)
  int mask_block = -1;
  uint32_t mask_word = 0u;
  if constexpr (kMode == kBlockMask) {
    const int wpb = p.block_size / 32, entry = start + lane / wpb;
    if (lane < p.chunk * wpb && entry < p.max_selected) {
      const int64_t at = (int64_t)b * p.block_stride + entry;
      mask_block = __ldg(p.block_idx + at);
      mask_word = __ldg(p.block_mask + at * wpb + lane % wpb);
    }
  }
  uint32_t flags = 0;
  int n, c;
  request_sizes(p, b, n, c, flags);
  if constexpr (kMode == kSpans) {
    if (kGuess && warp_merge && !guess.there && lane < min(span_n, p.span_cap))
      my_span = load_now(p.spans + span_first + lane);
    // the request's spans -> disjoint ascending runs in shared memory (every block of the request repeats this)
    int total;
    if (warp_merge && still_the_spans(guess, span_first, span_n, n, my_span)) {
      total = guess.total;
      flags |= guess.flags;
    } else if (warp_merge) {                          // up to 32 spans: every warp merges them for itself, no barrier
      if (guess.there && lane < min(span_n, p.span_cap)) my_span = load_now(p.spans + span_first + lane);
      int S = max(span_n, 0);
      if (S > p.span_cap) { S = p.span_cap; flags |= SSA_DEV_TOO_MANY_SPANS; }
      total = merge_spans_warp(s_wruns[warp], my_span, S, warp_runs, n, flags);
    } else {
      total = merge_spans_block<kThreads>(s_runs, p.spans + span_first, span_n, p.span_cap, n);
      if (tid == 0) flags |= s_runs.flags;
    }
    c = min(total, p.max_selected);
    if (total > p.max_selected) flags |= SSA_DEV_OVERFLOW;
  }
  if (start >= c && chunk_id > 0) return;             // chunk 0 always reports
  int cnt = max(0, min(p.chunk, c - start));          // list entries of this block; rows, except for bitmasks

  if constexpr (kMode == kBlockMask) {
    // The set bits of the listed blocks -> positions, in list order: a scan over the words' counts, and a word at a time
    // per warp.  One trip to memory and one barrier; with the words read 32 positions a warp at a time, four trips and
    // eight barriers, short lists waited longer for this than for their rows (64 requests x 32 heads, 1024 of 2048 rows:
    // 175.0 -> 170.5 us; 3 x 8, at most 314 rows: both kernels 5.7 -> 5.2 us).
    const int wpb = p.block_size / 32;
    int base = 0;
    if (lane >= cnt * wpb) {
      mask_word = 0u;
    } else {
      uint32_t in = 0u;                               // bits inside the context
      if (mask_block >= 0 && mask_block <= (n - 1) / p.block_size) {
        base = mask_block * p.block_size + (lane % wpb) * 32;
        const int left = n - base;
        in = left >= 32 ? 0xffffffffu : left > 0 ? (1u << left) - 1u : 0u;
      }
      if (mask_word & ~in) flags |= SSA_DEV_BAD_INDEX;
      mask_word &= in;
    }
    const int own = __popc(mask_word);
    int upto = own;
#pragma unroll
    for (int o = 1; o < kMaskChunk / 32; o <<= 1) {
      const int up = __shfl_up_sync(0xffffffffu, upto, o);
      if (lane >= o) upto += up;
    }
    cnt = __shfl_sync(0xffffffffu, upto, kMaskChunk / 32 - 1);
#pragma unroll
    for (int w = warp; w < kMaskChunk / 32; w += kWarps) {
      const uint32_t word = __shfl_sync(0xffffffffu, mask_word, w);
      const int at = __shfl_sync(0xffffffffu, upto - own, w), first = __shfl_sync(0xffffffffu, base, w);
      if ((word >> lane) & 1u) s_idx[at + __popc(word & ((1u << lane) - 1u))] = first + lane;
    }
    __syncthreads();
  }
  if constexpr (kMode == kSpans) {
    // positions of this warp's tiles, by arithmetic on the runs; head 0 leaves a copy for callers that want the list
    int32_t* row = (h == 0 && p.index_out) ? p.index_out + (int64_t)b * p.index_stride + start : nullptr;
#pragma unroll
    for (int j = 0; j < kIdxPerThread; ++j) {
      const int r = staged_row(lane + 32 * j);
      if (r < cnt) {
        const int v = warp_merge ? span_position(s_wruns[warp], warp_runs, start + r) : span_position(s_runs, start + r);
        s_idx[r] = v;
        if (row) row[r] = v;
      }
    }
    __syncwarp();
    if (chunk_id == 0 && h == 0 && tid == 0) {
      if (p.counts_out) p.counts_out[b] = c;
      if (p.ws_counts) p.ws_counts[b] = c;
    }
  }
  bool any_bad = false;                               // warp-uniform: an entry of this warp's tiles is out of range
  if (kMode == kIndex) {
    bool bad = false;
#pragma unroll
    for (int j = 0; j < kIdxPerThread; ++j) {
      const int r = staged_row(lane + 32 * j);
      if (r < cnt) {
        int v = raw[j];
        if (v < 0 || v >= n) {
          v = -1; flags |= SSA_DEV_BAD_INDEX; bad = true;
        } else if (kPaged) {                          // logical position -> row of the pool
          const int page = __ldg(p.page_table + (int64_t)b * p.page_table_stride + (v >> p.page_shift));
          if ((unsigned)page < (unsigned)p.n_pages) v = (page << p.page_shift) | (v & p.page_mask);
          else { v = -1; flags |= SSA_DEV_BAD_INDEX; bad = true; }
        }
        s_idx[r] = v;
      }
    }
    any_bad = __any_sync(0xffffffffu, bad) != 0;      // also orders the stores before the warp's reads
    __syncwarp();
  }
  if (p.dev_status && h == 0) {
    const uint32_t f = (tid == 0 && chunk_id == 0) ? flags : (flags & SSA_DEV_BAD_INDEX);
    if (f) atomicOr(p.dev_status, f);
  }

  const char* kbase = reinterpret_cast<const char*>(
      reinterpret_cast<const T*>(p.k) + (int64_t)b * p.k_sb + (int64_t)(h / p.kv_group) * p.k_sh + col * 16);
  const char* vbase = reinterpret_cast<const char*>(
      reinterpret_cast<const T*>(p.v) + (int64_t)b * p.v_sb + (int64_t)(h / p.kv_group) * p.v_sh + col * 16);

  // Requests the K and V rows of the warp's tile that starts at row t of the block; returns whether the tile needs
  // the predicated path (a ragged tail or entries that were skipped).
  Piece kr[kU], vr[kU];
  float s[kU];
  auto request_tile = [&](int t) -> bool {
    // full tiles without bad entries take the unpredicated path
    const bool checked = any_bad || (t + kTileRows > cnt);
    if (!checked) {
#pragma unroll
      for (int u = 0; u < kU; ++u) {
        const int r = t + u * kRowsPerLoad + sub;
        const uint32_t pos = (uint32_t)(kSparse ? s_idx[r] : start + r);
        load_piece<kAligned32, kFp8>(kr[u], kbase + (uint64_t)pos * p.k_row_bytes);
        load_piece<kAligned32, kFp8>(vr[u], vbase + (uint64_t)pos * p.v_row_bytes);
      }
    } else {
#pragma unroll
      for (int u = 0; u < kU; ++u) {
        const int r = t + u * kRowsPerLoad + sub;
        int pos = -1;
        if (r < cnt) pos = kSparse ? s_idx[r] : start + r;
        if (pos >= 0) {
          load_piece<kAligned32, kFp8>(kr[u], kbase + (uint64_t)(uint32_t)pos * p.k_row_bytes);
          load_piece<kAligned32, kFp8>(vr[u], vbase + (uint64_t)(uint32_t)pos * p.v_row_bytes);
          s[u] = 0.f;
        } else {
          zero_piece(kr[u]);
          zero_piece(vr[u]);
          s[u] = neg_inf();                           // marks the row as masked
        }
      }
    }
    return checked;
  };
  bool pre_issued = false, pre_checked = false;
  if constexpr (kHostQ) {
    // the first tile's rows are requested before the block waits for its query row
    if (warp * kTileRows < cnt) {
      pre_checked = request_tile(warp * kTileRows);
      pre_issued = true;
    }
    // the row has crossed the bus by now (or is about to): share it, and leave the device copy
    if (tid < D / 8) {
      s_qrow[tid] = q_word;
      *(reinterpret_cast<uint4*>(const_cast<TQ*>(reinterpret_cast<const TQ*>(p.q)) + (int64_t)b * p.q_sb +
                                 (int64_t)h * p.q_sh) + tid) = q_word;
    }
    __syncthreads();                                  // one chunk per request: every block gets here
    const uint4 a = s_qrow[2 * col], c4 = s_qrow[2 * col + 1];
    qraw.w[0] = a.x; qraw.w[1] = a.y; qraw.w[2] = a.z; qraw.w[3] = a.w;
    qraw.w[4] = c4.x; qraw.w[5] = c4.y; qraw.w[6] = c4.z; qraw.w[7] = c4.w;
  }
  float2 q2[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    q2[i] = unpack2<TQ>(qraw.w[i]);
    q2[i].x *= p.scale_log2;
    q2[i].y *= p.scale_log2;
  }
  float m = neg_inf(), l = 0.f;
  float2 acc[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) acc[i] = make_float2(0.f, 0.f);

  for (int t = warp * kTileRows; t < cnt; t += kWarps * kTileRows) {
    bool checked;
    if (kHostQ && pre_issued) {                         // the warp's first tile is already on its way
      checked = pre_checked;
      pre_issued = false;
    } else {
      checked = request_tile(t);
    }
    float mt = neg_inf();
#pragma unroll
    for (int u = 0; u < kU; ++u) {
      float2 d2 = make_float2(0.f, 0.f);
#pragma unroll
      for (int i = 0; i < 8; ++i) d2 = fma2(q2[i], piece_pair<T>(kr[u], i), d2);
      float d = d2.x + d2.y;
#pragma unroll
      for (int o = kLanesPerRow / 2; o > 0; o >>= 1) d += __shfl_xor_sync(0xffffffffu, d, o);
      s[u] = checked ? d + s[u] : d;                  // -inf stays -inf
      mt = max_or_nan(mt, s[u]);
    }
    const float m_new = max_or_nan(m, mt);
    if (m_new != neg_inf()) {                           // (a NaN among the scores: m stays, the weights become NaN)
      if (m_new > m) {                                // rare after the first tiles
        const float alpha = fast_exp2(m - m_new);     // m = -inf gives 0
        l *= alpha;
#pragma unroll
        for (int i = 0; i < 8; ++i) { acc[i].x *= alpha; acc[i].y *= alpha; }
        m = m_new;
      }
#pragma unroll
      for (int u = 0; u < kU; ++u) {
        const float pw = fast_exp2(s[u] - m);         // masked rows give 0
        l += pw;
        const float2 pw2 = make_float2(pw, pw);
#pragma unroll
        for (int i = 0; i < 8; ++i) acc[i] = fma2(pw2, piece_pair<T>(vr[u], i), acc[i]);
      }
    }
  }

  // all cache rows of this block have been read: the next kernel of the stream
  // may start filling the SMs this grid is leaving
  if (!p.early_release) grid_launch_dependents();

  // combine the lane groups of the block
  if constexpr (kWide) {
    // first those of a warp, each lane ending up with its share of the warp's sum
    const float top = lane_groups_max<kLanesPerRow>(m);
    const float w = (m > neg_inf()) ? fast_exp2(m - top) : 0.f;
    l = lane_groups_sum<kLanesPerRow>(l * w);
#pragma unroll
    for (int i = 0; i < 8; ++i) { acc[i].x *= w; acc[i].y *= w; }
    float2 part4[4], part2[2];
    halve_between<16>(part4, acc, lane);
    halve_between<8>(part2, part4, lane);
    const int d = col * 16 + ((lane & 16) ? 8 : 0) + ((lane & 8) ? 4 : 0);
    if constexpr (kLanesPerRow == 8) {
      *reinterpret_cast<float4*>(&s_acc[warp][d]) = make_float4(part2[0].x, part2[0].y, part2[1].x, part2[1].y);
    } else {
      float2 part1[1];
      halve_between<4>(part1, part2, lane);
      *reinterpret_cast<float2*>(&s_acc[warp][d + ((lane & 4) ? 2 : 0)]) = part1[0];
    }
    if (lane == 0) { s_m[warp] = top; s_l[warp] = l; }
  } else {
    const int g = warp * kRowsPerLoad + sub;
#pragma unroll
    for (int i = 0; i < 4; ++i)
      *reinterpret_cast<float4*>(&s_acc[g][col * 16 + 4 * i]) =
          make_float4(acc[2 * i].x, acc[2 * i].y, acc[2 * i + 1].x, acc[2 * i + 1].y);
    if (col == 0) { s_m[g] = m; s_l[g] = l; }
  }
  __syncthreads();
  if (tid < D) {
    float M = neg_inf();
#pragma unroll
    for (int i = 0; i < kGroups; ++i) M = fmaxf(M, s_m[i]);
    float L = 0.f, A = 0.f;
#pragma unroll
    for (int i = 0; i < kGroups; ++i) {
      const float w = (s_m[i] > neg_inf()) ? fast_exp2(s_m[i] - M) : 0.f;
      L = fmaf(s_l[i], w, L);
      A = fmaf(s_acc[i][tid], w, A);
    }
    if (p.n_chunks == 1) {
      store_row_value<TQ>(p, b, h, tid, M, L, A);
    } else {
      const int64_t slot = ((int64_t)b * p.H + h) * p.n_chunks + chunk_id;
      p.ws_acc[slot * D + tid] = A;
      if (tid == 0) p.ws_ml[slot] = make_float2(M, L);
    }
  }
}

// Pass 2.  The kernel is pure latency (a few KB per block), so everything it may need is requested in one go,
// before the request's list length is known: the (max, sum) pairs of all n_chunks slots and the first eight
// accumulator rows.  Slots of chunks that do not exist were never written; what is read from them is not used.
constexpr int kMergeStage = 512;       // (max, sum) pairs staged in shared memory; more chunks: read in place
constexpr int kMergeAhead = 8;         // accumulator rows requested before the sizes are known

template <typename T, int D>
__global__ void __launch_bounds__(D)
decode_merge_kernel(const DecodeParams p) {
  __shared__ float2 s_ml[kMergeStage];
  const int h = blockIdx.x, b = blockIdx.y, d = threadIdx.x;
  grid_dependency_wait();
  grid_launch_dependents();
  const int64_t base = ((int64_t)b * p.H + h) * p.n_chunks;
  const bool staged = p.n_chunks <= kMergeStage;
  if (staged)
    for (int k = d; k < p.n_chunks; k += D) s_ml[k] = p.ws_ml[base + k];
  float ahead[kMergeAhead];
#pragma unroll
  for (int k = 0; k < kMergeAhead; ++k) ahead[k] = k < p.n_chunks ? p.ws_acc[(base + k) * D + d] : 0.f;
  uint32_t flags = 0;
  int n, c;
  request_sizes(p, b, n, c, flags);
  const int ns = c > 0 ? (c + p.chunk - 1) / p.chunk : 1;
  __syncthreads();
  auto pair = [&](int k) { return staged ? s_ml[k] : p.ws_ml[base + k]; };
  float M = neg_inf();
  for (int k = 0; k < ns; ++k) M = fmaxf(M, pair(k).x);
  float L = 0.f, A = 0.f;
#pragma unroll
  for (int k = 0; k < kMergeAhead; ++k) {
    if (k < ns) {
      const float2 ml = pair(k);
      const float w = (ml.x > neg_inf()) ? fast_exp2(ml.x - M) : 0.f;
      L = fmaf(ml.y, w, L);
      A = fmaf(ahead[k], w, A);
    }
  }
  for (int k0 = kMergeAhead; k0 < ns; k0 += kMergeAhead) {   // long requests: eight rows per trip
    float rows[kMergeAhead];
#pragma unroll
    for (int j = 0; j < kMergeAhead; ++j) rows[j] = k0 + j < ns ? p.ws_acc[(base + k0 + j) * D + d] : 0.f;
#pragma unroll
    for (int j = 0; j < kMergeAhead; ++j) {
      if (k0 + j < ns) {
        const float2 ml = pair(k0 + j);
        const float w = (ml.x > neg_inf()) ? fast_exp2(ml.x - M) : 0.f;
        L = fmaf(ml.y, w, L);
        A = fmaf(rows[j], w, A);
      }
    }
  }
  store_row_value<T>(p, b, h, d, M, L, A);
}

}  // namespace ssa

#include "decode_gqa.cuh"

namespace ssa {

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
// share: row-sharing kernel; wide: one large row-sharing block per SM; even_blocks: that many blocks with even shares of
// the rows (0: chunks)
// warps: of a one-head block
struct Plan { int chunk, n_chunks; size_t acc_bytes, total_bytes; bool share, wide; int even_blocks, warps; };

// Grouped query heads that the kernel which reads a K/V row once for many heads can serve.
static bool can_share_rows(const ssa_attn_desc* d) {
  const int group = d->H_kv > 0 ? d->H / d->H_kv : 1;
  return d->D == 128 && group >= 2;
}

// A row-sharing block serves up to kGqaHeads heads; larger groups (several query tokens per head) take several blocks per
// chunk, side by side in the grid, so that all but the first find the rows in L2.  One head per block instead reads every
// row from L2 once per head (us, one head per block / row-sharing, 32 heads on each of 4 K/V heads, bf16): 3 requests of
// 12897 rows 194 / 34, 8 of 2000 listed rows 88 / 20, 24 of 40 14.7 / 6.3.  (Small launches: one_head_blocks_pay.)
static int head_splits(const ssa_attn_desc* d) { return (d->H / d->H_kv + kGqaHeads - 1) / kGqaHeads; }

// Warps of a one-head block that takes up to `rows` rows, in a launch of `blocks`.  A warp has sixteen rows of 128 16-bit
// values on their way at a time (as many bytes of others) and takes about 1.1 us a turn, however few other warps there are.
// A launch that leaves the SMs room therefore gets blocks of two or four times the warps, as far as the rows give each of
// them a turn.  Four warps / this, us, 16-bit rows of 128 in index lists: 32 heads x 80 rows 4.1 / 3.1, x 256 rows 6.4 / 4.2;
// 148 heads x 200 rows 6.8 / 5.1, x 512 rows 11.7 / 7.9; 296 heads x 200 rows 8.1 / 7.3, x 512 rows 14.1 / 12.3.  16-bit rows
// of 64: 32 x 160 rows 3.2 / 2.7, 148 x 512 7.0 / 5.6, 296 x 512 9.6 / 8.7; 8-bit rows of 128: 32 x 160 3.8 / 3.3, 148 x 512
// 8.6 / 7.3, 296 x 512 10.9 / 10.0; of 64: 148 x 512 4.7 / 3.8, 296 x 400 6.7 / 6.6.
static int block_warps(const ssa_attn_desc* d, long long blocks, int rows) {
  const int turn = 16 * (128 / d->D) * (d->kv_dtype == SSA_FP8_E4M3 ? 2 : 1);
  int warps = kSmallBlock;
  while (warps < kWarpSlots && rows > warps * turn && blocks * 2 * warps <= (long long)kWarpSlots * sm_count()) warps *= 2;
  return warps;
}

// Bytes of the partial results (accumulator row, maximum and sum) of `triples` (row, chunk) pairs, and of the accumulators.
static size_t triples_bytes(const ssa_attn_desc* d, size_t triples, size_t* acc_bytes) {
  *acc_bytes = (triples * d->D * sizeof(float) + 255) / 256 * 256;
  return *acc_bytes + (triples * sizeof(float2) + 255) / 256 * 256;
}

// full: contexts that are read as they lie, without a list or a page table.
static bool make_plan(const ssa_attn_desc* d, int max_selected, bool share, bool full, Plan* pl) {
  if (!d || d->B <= 0 || d->H <= 0 || max_selected <= 0) return false;
  if (d->D != 64 && d->D != 128) return false;
  const long long out_units = (long long)d->B * d->H;                  // triples per chunk
  const long long units = share ? (long long)d->B * d->H_kv * head_splits(d) : out_units;   // blocks per chunk
  // The second pass costs about as much as two rounds of a block, so a request is split only when that buys
  // parallelism: one chunk whenever the list fits a block's staging area and either every SM gets a block or
  // the list is short anyway; otherwise 256-entry chunks, halved while the grid has under two blocks per SM.
  // Large blocks (block_warps) stage up to 1024 entries, and taking a list of 257..1024 whole is better from a fifth of a
  // block per SM on, as far as 768 rows of 128 (16-bit ones are three turns of sixteen warps), and from two fifths on beyond
  // that (us, chunks / whole: 32 heads x 300 rows 4.9 / 4.4, x 700 6.7 / 6.5, but x 820 7.1 / 7.7 and x 1024 8.0 / 8.3; 48 x 820
  // 7.9 / 8.2, 64 x 820 8.8 / 8.6, 80 x 820 10.7 / 9.2, 296 x 820 24.6 / 21.1, but 8 x 820 5.7 / 6.7; 8-bit rows, 32 x 700 6.6 /
  // 6.3, x 1024 7.2 / 7.4; 32 x 1024 rows of 64 8.8 / 4.9); over an 8-bit cache, whose rows are fewer turns, not where a second
  // block would leave most SMs idle (160 x 1024 12.2 / 13.5), nor for grouped heads, whose lines (one_head_blocks_pay) were
  // measured with chunks.
  const long long sms = sm_count();
  const long long want = sms * 2;
  int chunk = 256, sized_for = 0;
  if (max_selected <= kMaxChunk && (units >= sms || max_selected <= 256)) chunk = kMaxChunk;
  else if (!share && max_selected <= staged_entries(block_warps(d, units, max_selected)) && units <= want &&
           5 * units >= (max_selected * d->D <= 768 * 128 ? sms : 2 * sms) &&
           (d->kv_dtype != SSA_FP8_E4M3 || (d->H == d->H_kv && (units <= sms || 5 * units >= 7 * sms))))
    chunk = kMaxWideChunk;
  // Longer chunks where there are blocks enough without (us, 256 / 512 entries; 32 heads a request).  Rows of 128 16-bit values:
  // lists and page tables gain, most of all where they are ragged (a paged context of 64 x 2048 307 / 304, of 64 x 512..2048 181 /
  // 177; 72 requests of up to 1024, every eighth full, 49.6 / 47.1, 64 44.9 / 43.7), but below 27 chunks of 512 per SM as often lose
  // (44 of them 34.6 / 35.0, 36 30.2 / 30.9; 56 41.2 / 40.3).  Contexts read as they lie do only in the longest launches (64 x 1024
  // 151 / 154, 32 x 512..2048 97 / 99, 32 x 4096 292 / 295; 32 x 8192 602 / 601, 32 x 2048..8192 395 / 388, on another GPU 581 / 584
  // and 384 / 384).  Rows of half the bytes, or less, are half a chunk: 8-bit, 32 x 900 49.7 / 47.4, 64 94 / 87, 16-bit of 64 52 / 51
  // (40) and 81 / 78 (fewer would make one-kernel steps of some that gain nothing by it: 24 x 600, 8-bit, 31.6 / 33.3); contexts
  // read as they lie from 20 chunks per SM on (rows of 64: 32 x 1024 42.7 / 45.0, 48 x 256..1024 42.7 / 41.5; 8-bit, 64 x 1024 90 / 86).
  else if (const long long long_chunks = units * ((max_selected + kMaxChunk - 1) / kMaxChunk);
           !share && (d->D == 64 || d->kv_dtype == SSA_FP8_E4M3
                          ? max_selected > kMaxChunk && units > 6 * sms && (!full || long_chunks >= 20 * sms)
                          : max_selected > 768 && long_chunks >= (full ? 80 : 27) * sms)) {
    sized_for = chunk;                                   // (the workspace asked for stays that of chunks of 256)
    chunk = kMaxChunk;
  }
  else while (chunk > 64 && units * ((max_selected + chunk - 1) / chunk) < want) chunk >>= 1;
  pl->share = share;
  pl->wide = false;
  if (share && 2 * units > sms && units <= sms && max_selected <= 2048) {
    // One unit for most SMs and a short list: the whole list is one large block's work, and the second pass
    // (about 3 us in the stream) is not needed (32 query heads over 4 K/V heads, 32 requests, 819 rows: 15.2 vs
    // 18.0 us).  With fewer units (2 K/V heads: 64) too many SMs would idle: 15.2 vs 14.4 us with four chunks.
    pl->wide = true;
    chunk = (max_selected + 63) / 64 * 64;
  } else if (share) {
    // The row-sharing kernel leaves G triples per chunk, its blocks stream (a ring of tiles per warp) and two of
    // them fit an SM: about one block per resident slot, i.e. as few chunks as keep the SMs busy (measured,
    // B*H_kv = 64..256, context 8192: within 3 % of the best split for groups of 4, 8 and 16 heads).  Ragged batches
    // would rather have shorter chunks (17 requests of 1001..8190 rows, 16 heads: 62 instead of 73 us with chunks of
    // 1024), batches of like lengths pay for them (all 8190: 102 instead of 90 us), and the host knows no lengths;
    // full contexts are therefore cut on the device (make_even), lists keep this split.
    const long long target = sms * 2;
    long long n = target / units;                              // rounded down: never one block over a full wave
    n = std::max<long long>(1, std::min<long long>(n, (max_selected + 255) / 256));
    chunk = (int)(((max_selected + n - 1) / n + 63) / 64 * 64);
  }
  pl->even_blocks = 0;
  int n_chunks = (max_selected + chunk - 1) / chunk;
  if (n_chunks == 1) chunk = (max_selected + 31) / 32 * 32;
  pl->warps = block_warps(d, units * n_chunks, chunk);
  pl->chunk = chunk;
  pl->n_chunks = n_chunks;
  pl->total_bytes = triples_bytes(d, (size_t)out_units * n_chunks, &pl->acc_bytes);
  size_t acc = 0;
  if (sized_for > 0) pl->total_bytes = triples_bytes(d, (size_t)out_units * ((max_selected + sized_for - 1) / sized_for), &acc);
  return true;
}

// The plan every workspace holds: grouped heads share rows.
static bool make_plan(const ssa_attn_desc* d, int max_selected, Plan* pl) {
  return make_plan(d, max_selected, d && can_share_rows(d), false, pl);
}

// Small launches over an 8-bit cache, grouped heads: a row-sharing block starts up slower (ring, Q fragments), combines G
// heads one after the other and converts every row; with few rows per block that outweighs reading them G times (from
// L2).  The lines below were measured over groups of 2, 4, 8, 12 and 16, 8..1600 query heads in all, lists of 40..8000
// rows and full contexts, by the product of heads and rows (us with one head per block / row-sharing): 1 request, 32
// heads over 2, 40 rows 2.6 / 5.0; 32 over 8: 160 rows 4.3 / 4.7, 820 rows 7.2 / 7.0; 8 requests of 32 over 4, 160 rows
// 4.9 / 5.6, 500 rows 8.0 / 8.9, 37 such requests 20.6 / 8.8; 8 of 32 over 2, 500 rows 7.7 / 11.7.  Never where only
// sharing saves the second pass, nor beyond one wave of blocks - except in groups of two, which then take two waves either
// way (48 requests of 16 over 8, 40 rows 6.7 / 7.5).  Groups of more than kGqaHeads over 16-bit rows follow the lines of the
// large groups: 1 request, 20 heads over 1, 3000 rows 8.3 / 9.4, 12000 rows 17.9 / 12.0; 2 requests of 96 over 4, 300 rows
// 6.9 / 8.0, 2000 rows 20.6 / 11.7.
static bool one_head_blocks_pay(const ssa_attn_desc* d, int max_selected, const Plan& shared, const Plan& single) {
  if ((d->kv_dtype != SSA_FP8_E4M3 && head_splits(d) == 1) || (shared.n_chunks == 1 && single.n_chunks > 1)) return false;
  const int group = d->H / d->H_kv;
  const long long heads = (long long)d->B * d->H, rows = heads * max_selected, sms = sm_count();
  if (group == 2 && single.n_chunks == 1 && heads > SSA_MIN_BLOCKS * sms) return rows <= 100000;
  if (heads * single.n_chunks > SSA_MIN_BLOCKS * sms) return false;
  if (single.n_chunks > 1) return rows <= (group <= 4 ? 20000 : group <= 8 ? 70000 : 130000);
  if (group > 8) return rows <= 160000;
  if (group <= 4) return rows <= 40000;
  return rows <= (shared.n_chunks > 1 ? 135000 : heads <= 2 * sms ? 75000 : 48000);
}

// The plan of a call with a workspace of ws_bytes: one head per block where that pays and the workspace, which callers may
// have sized by another bound, holds its partial results; otherwise the plan above.  (Above kGqaHeads heads per K/V head
// that is also the plan for a workspace too small for the one above.)
static bool choose_plan(const ssa_attn_desc* d, int max_selected, size_t ws_bytes, Plan* pl, bool full = false) {
  if (!make_plan(d, max_selected, d && can_share_rows(d), full, pl)) return false;
  Plan single;
  if (pl->share && make_plan(d, max_selected, false, full, &single) && single.total_bytes <= ws_bytes &&
      (one_head_blocks_pay(d, max_selected, *pl, single) || (head_splits(d) > 1 && pl->total_bytes > ws_bytes)))
    *pl = single;
  return true;
}

// Workspace with which choose_plan has its choice.  Where launches of more units are cut into fewer chunks than they were with
// four-warp blocks of one head (lists taken whole, row-sharing blocks above kGqaHeads heads), it also holds what fewer requests
// and shorter lists of the same geometry need, so that one size asked for the largest batch still serves all: one head per
// block, chunks of 256, and, as halving ends once there are two blocks per SM, fewer than four per SM of 64 rows or more;
// row-sharing blocks, two per SM at most, of 256 rows or more.
static size_t plan_bytes(const ssa_attn_desc* d, int max_selected) {
  Plan pl, chosen;
  if (!make_plan(d, max_selected, &pl) || !choose_plan(d, max_selected, SIZE_MAX, &chosen)) return 0;
  const long long rows = (long long)d->B * d->H, sms = sm_count();
  auto cut = [&](int chunk) { return rows * ((max_selected + chunk - 1) / chunk); };
  long long triples = 0;
  if (!pl.share) {
    if (max_selected > kMaxChunk) triples = cut(256);
    if (max_selected > 256) triples = std::max(triples, std::min(4 * sms, cut(64)));
  } else if (head_splits(d) > 1) {
    const long long per_block = (d->H / d->H_kv + head_splits(d) - 1) / head_splits(d);
    triples = std::min(2 * sms * per_block, cut(256));
  }
  size_t acc = 0;
  return std::max({pl.total_bytes, chosen.total_bytes, triples_bytes(d, (size_t)triples, &acc)});
}

// Full contexts read by the row-sharing kernel: cut on the device over one block per resident slot, if the lengths of all
// requests fit a block's scan and the workspace, which callers may have sized by an index list's bound, holds the results.
static size_t even_bytes(const ssa_attn_desc* d, int blocks, size_t* acc_bytes) {
  return triples_bytes(d, (size_t)2 * blocks * (d->H / d->H_kv), acc_bytes);
}

static int even_blocks_wanted(const ssa_attn_desc* d, const Plan& pl) {
  // Only where the fixed plan has a second pass too (about 3 us): one unit per SM at most, hence few requests.
  if (!pl.share || pl.wide || pl.n_chunks == 1 || d->B > kEvenMaxBatch) return 0;
  const long long units = (long long)d->B * d->H_kv, pieces = ((long long)d->max_ctx + kEvenRows - 1) / kEvenRows;
  if (units * pieces > 0xffffffll) return 0;                         // rows and pieces stay far inside 32 bits
  const long long blocks = 2ll * sm_count() / head_splits(d), share = units * d->max_ctx / blocks;
  // Below 1024 rows per share, were all contexts as long as the cache, there is nothing to win against the scan of the
  // lengths in front of the first rows (the lengths themselves may be shorter: even_by_slices).
  if (share < 1024) return 0;
  // Nine and more heads over 16-bit rows (two-warp teams) start up dearer: where two slices per unit fill the chip anyway,
  // shares have to be longer.  16 heads, 136 units, us with fixed slices / equal shares: caches of 4096 rows, all full 52.9
  // / 60.4, 1024..4096 rows 42.2 / 41.1, 0..4096 rows 41.9 / 47.9; of 8190 rows 91.3 / 99.0, 2047..8190 rows 77.1 / 65.7.
  if (d->H / d->H_kv > 8 && d->kv_dtype != SSA_FP8_E4M3 && share < 2304 && pl.n_chunks == 2 && 16 * units > 7 * blocks)
    return 0;
  return (int)blocks;
}

static void make_even(const ssa_attn_desc* d, size_t ws_bytes, Plan* pl) {
  const int blocks = even_blocks_wanted(d, *pl);
  size_t acc = 0;
  if (blocks == 0 || even_bytes(d, blocks, &acc) > ws_bytes) return;
  pl->even_blocks = blocks;
  pl->acc_bytes = acc;
}

// Blocked lists: a block of the grid expands as many list entries as fit kMaskChunk positions.
static bool make_plan_blockmask(const ssa_attn_desc* d, int block_size, int max_blocks, Plan* pl) {
  if (!d || d->B <= 0 || d->H <= 0 || max_blocks <= 0) return false;
  if (d->D != 64 && d->D != 128) return false;
  if (block_size != 32 && block_size != 64 && block_size != 128 && block_size != 256) return false;
  const long long units = (long long)d->B * d->H;
  pl->share = pl->wide = false;
  pl->even_blocks = 0;
  pl->chunk = kMaskChunk / block_size;
  pl->n_chunks = (max_blocks + pl->chunk - 1) / pl->chunk;
  pl->warps = block_warps(d, units * pl->n_chunks, std::min(pl->chunk, max_blocks) * block_size);
  pl->total_bytes = triples_bytes(d, (size_t)units * pl->n_chunks, &pl->acc_bytes);
  return true;
}

static bool aligned16(const void* p) { return reinterpret_cast<uintptr_t>(p) % 16 == 0; }

static int32_t check_desc(const ssa_attn_desc* d) {
  if (d->B <= 0 || d->H <= 0 || d->max_ctx <= 0 || d->B > 65535 || d->H > 65535) return SSA_ERR_SHAPE;
  if (d->D != 64 && d->D != 128) return SSA_ERR_UNSUPPORTED;
  if (d->H_kv <= 0 || d->H % d->H_kv != 0) return SSA_ERR_UNSUPPORTED;
  const bool fp8 = d->kv_dtype == SSA_FP8_E4M3;
  if (d->kv_dtype != SSA_F16 && d->kv_dtype != SSA_BF16 && !fp8) return SSA_ERR_DTYPE;
  const int32_t q_dtype = fp8 ? SSA_BF16 : d->kv_dtype;            // queries over an 8-bit cache are bf16
  if (d->out_dtype != q_dtype && d->out_dtype != SSA_F32) return SSA_ERR_DTYPE;
  const int64_t qo_strides[] = {d->q_stride_b, d->q_stride_h, d->o_stride_b, d->o_stride_h};
  const int64_t kv_strides[] = {d->k_stride_b, d->k_stride_t, d->k_stride_h, d->v_stride_b, d->v_stride_t, d->v_stride_h};
  for (int64_t s : qo_strides) {
    if (s < 0) return SSA_ERR_SHAPE;
    if (s % 8 != 0) return SSA_ERR_ALIGN;
  }
  for (int64_t s : kv_strides) {                                   // 16 bytes: 8 16-bit or 16 8-bit elements
    if (s < 0) return SSA_ERR_SHAPE;
    if (s % (fp8 ? 16 : 8) != 0) return SSA_ERR_ALIGN;
  }
  if (d->k_stride_t >= (1ll << 31) || d->v_stride_t >= (1ll << 31)) return SSA_ERR_SHAPE;
  return SSA_OK;
}

template <typename T, int D>
static int32_t launch(const DecodeParams& p, int B, int mode, bool aligned32, cudaStream_t st) {
  cudaEvent_t ev_b, ev_e;
  take_kernel_events(&ev_b, &ev_e);
  dim3 grid((unsigned)p.n_chunks, (unsigned)p.H, (unsigned)B);
  void (*kernel)(const DecodeParams);
  using TQ = typename Storage<T>::Query;
  constexpr bool kFp8 = kIsFp8<T>;
  size_t dynamic_smem = 0;
  unsigned block_threads = 0;
  const bool share = p.share_rows;
  if constexpr (D == 128) {
    if (share) {
      grid.x *= (unsigned)p.head_splits;
      grid.y = (unsigned)(p.H / p.kv_group);            // one block, or head_splits, per K/V head
      auto pick = [&](auto hi_tag, auto wide_tag, auto split_tag) {
        constexpr bool kHi = decltype(hi_tag)::value, kWide = decltype(wide_tag)::value, kSplit = decltype(split_tag)::value;
        using Shape = GqaShape<T, kHi, kWide>;
        block_threads = Shape::kWarps * 32;
        dynamic_smem = Shape::kSmemBytes;
        if constexpr (!kWide) {
          if (p.even_blocks > 0) {
            kernel = decode_partial_gqa_kernel<T, kDense, kHi, false, true, kSplit>;
            return;
          }
        }
        kernel = mode == kIndex   ? decode_partial_gqa_kernel<T, kIndex, kHi, kWide, false, kSplit>
                 : mode == kSpans ? decode_partial_gqa_kernel<T, kSpans, kHi, kWide, false, kSplit>
                                  : decode_partial_gqa_kernel<T, kDense, kHi, kWide, false, kSplit>;
      };
      constexpr std::true_type yes;
      constexpr std::false_type no;
      if (p.head_splits > 1) p.gqa_wide ? pick(yes, yes, yes) : pick(yes, no, yes);   // nine heads a block at least
      else if (p.heads_per_block > 8) p.gqa_wide ? pick(yes, yes, no) : pick(yes, no, no);
      else p.gqa_wide ? pick(no, yes, no) : pick(no, no, no);
      if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dynamic_smem) != cudaSuccess)
        return SSA_ERR_CUDA;
      if (p.even_blocks > 0) grid = dim3((unsigned)(p.even_blocks * p.head_splits));
    }
  }
  if (!share) {
    if ((mode == kIndex || mode == kSpans) && p.chunk > staged_entries(p.warps)) return SSA_ERR_SHAPE;   // (no plan does)
    auto pick = [&](auto aligned_tag, auto warps_tag) {
      constexpr bool kA = decltype(aligned_tag)::value;
      constexpr int kW = decltype(warps_tag)::value;
      block_threads = kW * 32;
      if constexpr (!kFp8) {
        if (p.q_host) {                                 // run() has checked: index lists, one chunk, no paging
          kernel = decode_partial_kernel<T, D, kIndex, kA, false, true, kW>;
          return;
        }
      }
      kernel = mode == kIndex ? (p.page_table ? decode_partial_kernel<T, D, kIndex, kA, true, false, kW>
                                              : decode_partial_kernel<T, D, kIndex, kA, false, false, kW>)
               : mode == kBlockMask ? decode_partial_kernel<T, D, kBlockMask, kA, false, false, kW>
               : mode == kSpans     ? decode_partial_kernel<T, D, kSpans, kA, false, false, kW>
                                    : decode_partial_kernel<T, D, kDense, kA, false, false, kW>;
      if constexpr (D == 128 && !kFp8 && kW > kSmallBlock)
        if (mode == kSpans && p.guess_blocks == 0) kernel = decode_partial_kernel<T, D, kSpans, kA, false, false, kW, false>;
    };
    auto by_warps = [&](auto aligned_tag) {
      if (p.warps == kWarpSlots) pick(aligned_tag, std::integral_constant<int, kWarpSlots>{});
      else if (p.warps > kSmallBlock) pick(aligned_tag, std::integral_constant<int, 2 * kSmallBlock>{});
      else pick(aligned_tag, std::integral_constant<int, kSmallBlock>{});
    };
    // (8-bit rows are read in 16-byte pieces: one instantiation)
    if (!kFp8 && aligned32) by_warps(std::bool_constant<!kFp8>{});
    else by_warps(std::false_type{});
  }
  if (ev_b) cudaEventRecord(ev_b, st);
  cudaError_t err = launch_pdl_smem(kernel, grid, dim3(block_threads), dynamic_smem, st, p);
  if (ev_e) cudaEventRecord(ev_e, st);
  if (err != cudaSuccess || cudaGetLastError() != cudaSuccess) return SSA_ERR_CUDA;
  int launches = 1;
  if (share && p.even_blocks > 0) {
    const int heads = std::min(p.kv_group, kEvenMergeHeads), splits = (p.kv_group + kEvenMergeHeads - 1) / kEvenMergeHeads;
    err = launch_pdl(decode_merge_even_kernel<TQ>, dim3((unsigned)(p.H / p.kv_group * splits), (unsigned)B),
                     dim3((unsigned)(D * heads)), st, p);
    if (err != cudaSuccess || cudaGetLastError() != cudaSuccess) return SSA_ERR_CUDA;
    ++launches;
  } else if (p.n_chunks > 1) {
    DecodeParams pm = p;
    if (mode == kSpans) pm.counts = p.ws_counts;        // the first pass left the list lengths there
    err = launch_pdl(decode_merge_kernel<TQ, D>, dim3((unsigned)p.H, (unsigned)B), dim3(D), st, pm);
    if (err != cudaSuccess || cudaGetLastError() != cudaSuccess) return SSA_ERR_CUDA;
    ++launches;
  }
  note_launches(launches);
  return SSA_OK;
}

// A request's attended set in the blocked encoding (mode kBlockMask).
struct BlockList { const int32_t* block_idx; const uint32_t* block_mask; int32_t block_size; };

// The span lists themselves (mode kSpans), with the optional copies of what they expand to.
struct SpanLists { const int32_t* span_offsets; const int32_t* spans; int32_t span_cap; int32_t* index_out;
                   int32_t* counts_out; };

static size_t counts_bytes(const ssa_attn_desc* d) { return ((size_t)d->B * sizeof(int32_t) + 255) / 256 * 256; }

// Which blocks use the time before grid_dependency_wait(), and how (prefetch_early).  Launches follow one another, and the blocks
// of one move in while the last blocks of the one in front drain, 3..7 us before they may begin; the memory system is half idle
// then, and altogether so for two microseconds more, until the lists have arrived and name the first rows.  What is asked for in
// L2 meanwhile should fill that gap and no more, since the blocks in front still wait for their own rows.
// One head per block: blocks of kSmallBlock warps, five of eight that fit the chip (the others come too late to gain by it), two
// turns of rows each, by one warp.  us, 64 requests of 32 heads over 141 listed rows: none 28.5, so 27.0; 592 blocks with one
// turn 26.9, with two 28.3, 370 with four 28.2, all four warps asking 28.1; 16 x 32 heads x 200 rows 12.1 / 10.0, 37 x 32 x 100
// 15.0 / 13.1, 20 x 32 x 400 28.3 / 27.0.  A launch of a wave or less over lists of one turn has nothing to gain (16 x 32 x 40
// 4.55 / 4.65; 37 x 32 x 40 9.1 / 8.2), nor have the shortest lists behind an index launch (61 x 32 x 15 14.2 / 14.4) and launches
// of larger blocks, two per SM at most (7 requests of 8 heads and up to 900 rows 11.7 / 13.2).
// Behind a merge launch, which is soon over, never more than 128 rows: two turns of 8-bit rows, or of rows of 64, are a whole chunk
// of 256 (without / two turns / 128 rows; steps over 8-bit rows, 30 spans, 7 x 8 heads 12.2 / 13.4 / 11.8, 1 x 32 12.1 / 13.4 / 11.9;
// index lists of 2000 of them, 16 x 8 heads 20.3 / 19.0 / 18.2).  Lists of one chunk keep two turns (16 x 32 heads of 64, 400 rows,
// 11.8 / 10.3 / 10.7).  Span lists, which are merged first, are late as it is: one turn where all blocks begin at once (without / two
// turns / one; 4 x 8 heads, 30 spans of 45, 11.5 / 11.2 / 10.1, 7 x 8, 19 spans, 11.7 / 11.6 / 10.4; but 14 x 8, 30 spans of 110, 33.3 /
// 31.1 / 31.6).  Index lists keep two there (7 x 8 heads, 2000 rows, 15.4 / 13.1 / 14.0), which lose behind an index launch: references
// of 8 requests, 8 heads, 14.8 / 15.9 / 14.8; the call does not know what is in front of it.
// Row-sharing launches are a wave: three of four blocks, the rows that fill the rings, by four warps, or what these ask for at once
// where there are fewer blocks than SMs.  us, 32 heads over 8, 32 requests of 820 rows 21.9 / 18.6, of 400 13.6 / 11.2, 8-bit rows
// 15.6 / 14.1; 4 requests of 820 9.2 / 8.7, of 100 4.9 / 4.9; one warp asking 19.4 for the first of these, for 512 rows 20.3; 2 full contexts of 300 rows, 12
// heads, 7.8 / 7.9: these, and whoever else is few, have no lists to wait for.  (Not
// groups above sixteen, whose registers are short.)
// Span lists of up to 32 are merged before the wait by every block that fits the chip, and by the others as before: checking
// that the list is still the same takes one trip, reading and merging it two and 0.4 us.  us, one-kernel steps, merged after / before
// the wait: 16 requests, 32 heads, three spans of 40: 10.9 / 8.9, 48 x 8 heads, 14 of 20: 13.7 / 12.3, 4 x 8, six of 20 5.1 / 4.6.
// In blocks of 8 and 16 warps over 16-bit rows of 128 the turns come out slower where the kernel has the code to do so, which lists
// of more than 384 rows lose by unless merging more than 16 spans takes longer: 8 requests of 32 heads, two of them full contexts of
// up to 1024, 16.0 / 17.5, 32 units of up to 514 rows, 3 spans, 7.0 / 7.4; but 64 of 264 rows, 10 spans, 6.2 / 5.6, of 664, 30 spans, 8.4 /
// 8.0.  These have a kernel without it.
// What then is left for row-sharing blocks to prefetch in pays for lists of one chunk that take them longest: 32 heads over 8, 32
// requests of six spans of 100 15.9 / 13.3, 8-bit rows 12.4 / 11.4; but with a merge launch in front, which is short, 4 requests of
// 14 spans 10.0 / 11.0, and 16 of three, 8-bit rows, 7.3 / 7.6.
static void plan_early(const ssa_attn_desc* d, const Plan& pl, int max_selected, int mode, DecodeParams* p) {
  const int sms = sm_count(), turn = kSmallBlock * 16 * (128 / d->D) * (d->kv_dtype == SSA_FP8_E4M3 ? 2 : 1);
  const bool few = (long long)d->B * d->H_kv * pl.n_chunks < sms;
  p->early_blocks = 0;
  p->early_warps = pl.share ? 4 : 1;
  const bool one_turn = mode == kSpans && (long long)d->B * d->H * pl.n_chunks <= SSA_MIN_BLOCKS * sms;
  p->early_rows = pl.share ? (few ? 128 : 192) : pl.n_chunks == 1 ? 2 * turn : std::min(one_turn ? turn : 2 * turn, 128);
  const bool in_time = mode == kSpans ? pl.n_chunks == 1 && max_selected * (d->kv_dtype == SSA_FP8_E4M3 ? 1 : 2) >= 600
                                      : mode != kDense || !few;
  if (pl.share) p->early_blocks = in_time ? sms * 3 / 2 : 0;
  else if (pl.warps == kSmallBlock && (max_selected > turn || (2 * max_selected > turn &&
                                                               (long long)d->B * d->H * pl.n_chunks > SSA_MIN_BLOCKS * sms)))
    p->early_blocks = sms * SSA_MIN_BLOCKS * 5 / 8;
  const bool long_turns = !pl.share && pl.warps > kSmallBlock && d->D == 128 && d->kv_dtype != SSA_FP8_E4M3;
  p->guess_blocks = long_turns && p->span_cap <= 16 && std::min(pl.chunk, max_selected) > 384 ? 0
                    : pl.share ? 2 * sms : kWarpSlots / pl.warps * sms;
  Allocation known = {};
  p->spans_readable = mode == kSpans && p->guess_blocks > 0 ? readable_entries<int2>(p->spans, &known) : 0;
}

// mode kDense: index/counts unused.  kIndex: the index list.  kBlockMask: `counts`
// are the numbers of listed blocks, `index_stride` the list capacity in blocks,
// `max_selected` the host bound on listed blocks, `bl` the lists.  kSpans: `sl`
// the span lists, `index_stride` the pitch of sl->index_out; the workspace then
// ends with one int32 per request (list lengths for the second pass).
static int32_t run(const ssa_attn_desc* d, const void* q, const void* k, const void* v,
                   const int32_t* ctx_lens, const int32_t* index, int32_t index_stride,
                   const int32_t* counts, int32_t max_selected, void* out, float* lse,
                   void* ws, size_t ws_bytes, uint32_t* dev_status, void* stream, int mode,
                   const BlockList* bl = nullptr, const ssa_paging* pg = nullptr,
                   const SpanLists* sl = nullptr, const void* q_host = nullptr) {
  // a paged cache is read through the staged-positions path; without a list the positions are 0 .. ctx_len-1
  const bool dense_paged = pg && mode == kDense;
  if (dense_paged) mode = kIndex;
  const bool sparse = mode == kIndex;
  if (!d || !q || !k || !v || !ctx_lens || !out) return SSA_ERR_NULL;
  if (sparse && !dense_paged && (!index || !counts)) return SSA_ERR_NULL;
  if (pg) {
    if (!pg->page_table) return SSA_ERR_NULL;
    if (mode == kBlockMask) return SSA_ERR_UNSUPPORTED;
    if (pg->page_size <= 0 || (pg->page_size & (pg->page_size - 1)) != 0 || pg->n_pages <= 0 ||
        pg->page_table_stride <= 0 || (long long)pg->n_pages * pg->page_size > 0x7fffffffll ||
        (long long)pg->page_table_stride * pg->page_size < d->max_ctx)
      return SSA_ERR_SHAPE;
  }
  if (mode == kBlockMask && (!bl || !bl->block_idx || !bl->block_mask || !counts)) return SSA_ERR_NULL;
  if (mode == kSpans) {
    if (!sl || !sl->spans) return SSA_ERR_NULL;           // no offsets: a fixed-stride table
    if (pg) return SSA_ERR_UNSUPPORTED;
    if (reinterpret_cast<uintptr_t>(sl->spans) % 8 != 0) return SSA_ERR_ALIGN;
  }
  const int32_t rc = check_desc(d);
  if (rc != SSA_OK) return rc;
  if (dense_paged) {
    max_selected = d->max_ctx;
    index_stride = d->max_ctx;
  } else if (mode == kSpans) {
    if (max_selected <= 0 || sl->span_cap <= 0 || sl->span_cap > kDirectSpans) return SSA_ERR_CAPACITY;
    if (sl->index_out && max_selected > index_stride) return SSA_ERR_CAPACITY;
  } else if (mode != kDense) {
    if (index_stride <= 0 || max_selected <= 0 || max_selected > index_stride) return SSA_ERR_CAPACITY;
  } else {
    max_selected = d->max_ctx;
  }
  if (!aligned16(q) || !aligned16(k) || !aligned16(v) || !aligned16(out) || !aligned16(ws)) return SSA_ERR_ALIGN;
  Plan pl;
  const size_t list_bytes = mode == kSpans ? counts_bytes(d) : 0;
  if (mode == kBlockMask) {
    if (bl->block_size != 32 && bl->block_size != 64 && bl->block_size != 128 && bl->block_size != 256)
      return SSA_ERR_UNSUPPORTED;
    if (!make_plan_blockmask(d, bl->block_size, max_selected, &pl)) return SSA_ERR_SHAPE;
  } else if (!choose_plan(d, max_selected, ws_bytes - std::min(ws_bytes, list_bytes), &pl, mode == kDense)) {
    return SSA_ERR_SHAPE;
  }
  if (!ws || ws_bytes < pl.total_bytes + list_bytes) return SSA_ERR_WORKSPACE;
  if (mode == kDense) make_even(d, ws_bytes, &pl);

  if (q_host && !(mode == kIndex && !pg && !dense_paged && pl.n_chunks == 1 && !pl.share &&
                  d->kv_dtype != SSA_FP8_E4M3 && aligned16(q_host)))
    return SSA_ERR_UNSUPPORTED;
  DecodeParams p;
  p.q_host = q_host;
  p.span_offsets = mode == kSpans ? sl->span_offsets : nullptr;
  p.spans = mode == kSpans ? reinterpret_cast<const int2*>(sl->spans) : nullptr;
  p.span_cap = mode == kSpans ? sl->span_cap : 0;
  p.index_out = mode == kSpans ? sl->index_out : nullptr;
  p.counts_out = mode == kSpans ? sl->counts_out : nullptr;
  p.ws_counts = mode == kSpans ? reinterpret_cast<int32_t*>(reinterpret_cast<char*>(ws) + pl.total_bytes) : nullptr;
  p.q = q; p.k = k; p.v = v;
  p.ctx_lens = ctx_lens;
  p.index = sparse && !dense_paged ? index : nullptr;
  p.counts = mode != kDense && mode != kSpans && !dense_paged ? counts : nullptr;
  p.page_table = pg ? pg->page_table : nullptr;
  p.page_table_stride = pg ? pg->page_table_stride : 0;
  p.n_pages = pg ? pg->n_pages : 0;
  p.page_mask = pg ? pg->page_size - 1 : 0;
  p.page_shift = 0;
  while (pg && (1 << p.page_shift) < pg->page_size) ++p.page_shift;
  p.block_idx = mode == kBlockMask ? bl->block_idx : nullptr;
  p.block_mask = mode == kBlockMask ? bl->block_mask : nullptr;
  p.block_size = mode == kBlockMask ? bl->block_size : 0;
  p.block_stride = mode == kBlockMask ? index_stride : 0;
  p.out = out; p.lse = lse;
  p.ws_acc = reinterpret_cast<float*>(ws);
  p.ws_ml = reinterpret_cast<float2*>(reinterpret_cast<char*>(ws) + pl.acc_bytes);
  p.dev_status = dev_status;
  p.q_sb = d->q_stride_b; p.q_sh = d->q_stride_h;
  p.kv_group = d->H / d->H_kv;
  p.k_sb = pg ? 0 : d->k_stride_b; p.k_sh = d->k_stride_h;      // a pool has no batch dimension
  p.v_sb = pg ? 0 : d->v_stride_b; p.v_sh = d->v_stride_h;
  const int kv_bytes = d->kv_dtype == SSA_FP8_E4M3 ? 1 : 2;
  p.k_row_bytes = (uint32_t)(d->k_stride_t * kv_bytes);
  p.v_row_bytes = (uint32_t)(d->v_stride_t * kv_bytes);
  p.o_sb = d->o_stride_b; p.o_sh = d->o_stride_h;
  p.H = d->H; p.max_ctx = d->max_ctx;
  p.index_stride = index_stride; p.max_selected = max_selected;
  p.chunk = pl.chunk; p.n_chunks = pl.n_chunks;
  p.share_rows = pl.share ? 1 : 0;
  p.warps = pl.warps;
  p.head_splits = pl.share ? head_splits(d) : 1;
  p.heads_per_block = (p.kv_group + p.head_splits - 1) / p.head_splits;
  p.gqa_wide = pl.wide ? 1 : 0;
  p.even_blocks = pl.even_blocks;
  p.even_factor = d->kv_dtype == SSA_FP8_E4M3 ? 5 : 6;
  p.B = d->B;
  p.out_f32 = d->out_dtype == SSA_F32;
  // A grid of a few waves releases the next kernel at once (its blocks wait on
  // chip instead of being launched after the drain); a long grid does so only
  // as its blocks finish, so that waiting blocks do not crowd out its own.
  p.early_release = pl.even_blocks == 0 &&
                    (long long)d->B * d->H * pl.n_chunks <= (long long)sm_count() * SSA_MIN_BLOCKS * 6;
  plan_early(d, pl, max_selected, mode, &p);
  const float scale = d->scale > 0.f ? d->scale : 1.0f / sqrtf((float)d->D);
  p.scale_log2 = scale * kLog2e;

  // one 256-bit load per lane needs every cache row piece on a 32-byte boundary
  const bool a32 = reinterpret_cast<uintptr_t>(k) % 32 == 0 && reinterpret_cast<uintptr_t>(v) % 32 == 0 &&
                   p.k_sb % 16 == 0 && d->k_stride_t % 16 == 0 && d->k_stride_h % 16 == 0 &&
                   p.v_sb % 16 == 0 && d->v_stride_t % 16 == 0 && d->v_stride_h % 16 == 0;
  cudaStream_t st = (cudaStream_t)stream;
  if (d->kv_dtype == SSA_FP8_E4M3)
    return d->D == 128 ? launch<Fp8E4M3, 128>(p, d->B, mode, false, st) : launch<Fp8E4M3, 64>(p, d->B, mode, false, st);
  if (d->kv_dtype == SSA_BF16)
    return d->D == 128 ? launch<__nv_bfloat16, 128>(p, d->B, mode, a32, st)
                       : launch<__nv_bfloat16, 64>(p, d->B, mode, a32, st);
  return d->D == 128 ? launch<__half, 128>(p, d->B, mode, a32, st) : launch<__half, 64>(p, d->B, mode, a32, st);
}

int32_t one_kernel_span_limit() { return kDirectSpans; }

// ssa_decode_attn_sparse with the query rows still in page-locked host memory that the device addresses (q_host,
// laid out like q): every block fetches its own row across the bus and writes the device copy at q.  Offered
// where host_queries_pay() says so.
int32_t decode_attn_sparse_host_queries(const ssa_attn_desc* desc, void* q, const void* q_host, const void* k_cache,
                                        const void* v_cache, const int32_t* ctx_lens, const int32_t* index,
                                        int32_t index_stride, const int32_t* counts, int32_t max_selected, void* out,
                                        float* lse, void* workspace, size_t workspace_bytes, uint32_t* dev_status,
                                        void* stream) {
  if (!q_host) return SSA_ERR_NULL;
  return run(desc, q, k_cache, v_cache, ctx_lens, index, index_stride, counts, max_selected, out, lse, workspace,
             workspace_bytes, dev_status, stream, kIndex, nullptr, nullptr, nullptr, q_host);
}

// One chunk per request (every row then crosses the bus once) and one head per block over a 16-bit cache, by the plan that the
// call with this workspace will take.
bool host_queries_pay(const ssa_attn_desc* d, int32_t max_selected, size_t ws_bytes) {
  Plan pl;
  if (!d || check_desc(d) != SSA_OK || !choose_plan(d, max_selected, ws_bytes, &pl)) return false;
  return pl.n_chunks == 1 && !pl.share && d->kv_dtype != SSA_FP8_E4M3;
}

// Every block of the span-list kernel repeats the merge of its request's spans (about a microsecond per wave
// of blocks when a warp can do it alone), the index kernel does it once per request but costs a launch of its
// own (about 3 us exposed): one kernel up to three waves of blocks.
bool one_kernel_step_pays(const ssa_attn_desc* d, int32_t max_selected, int32_t max_spans, size_t ws_bytes) {
  Plan pl;
  if (max_spans <= 0 || max_spans > 32 || !d || check_desc(d) != SSA_OK) return false;
  if (!choose_plan(d, max_selected, ws_bytes - std::min(ws_bytes, counts_bytes(d)), &pl)) return false;
  if (ws_bytes < pl.total_bytes + counts_bytes(d)) return false;
  const long long units = pl.share ? (long long)d->B * d->H_kv * head_splits(d) : (long long)d->B * d->H;
  return units * pl.n_chunks <= 3ll * SSA_MIN_BLOCKS * sm_count();
}

// Scratch of ssa_decode_attn_sparse_noalloc: part of the library's device image.
// In host code the name `g_static_scratch` is only a handle for
// cudaGetSymbolAddress, never a device address to pass to a kernel.
static __device__ __align__(256) unsigned char g_static_scratch[SSA_STATIC_SCRATCH_BYTES];

// Device address of the array on the current device (its primary context), looked up once per device; threads
// that race on the first call all store the same value.  The address does not survive cudaDeviceReset.
static void* static_scratch_address() {
  constexpr int kMaxDevices = 64;
  static std::atomic<void*> address[kMaxDevices];
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return nullptr;
  void* ptr = address[dev].load(std::memory_order_acquire);
  if (!ptr) {
    if (cudaGetSymbolAddress(&ptr, g_static_scratch) != cudaSuccess || !ptr) return nullptr;
    address[dev].store(ptr, std::memory_order_release);
  }
  return ptr;
}

}  // namespace ssa

extern "C" {

int32_t ssa_decode_attn_sparse_noalloc(const ssa_attn_desc* desc, const void* q, const void* k_cache,
                                       const void* v_cache, const int32_t* ctx_lens, const int32_t* index,
                                       int32_t index_stride, const int32_t* counts, int32_t max_selected,
                                       void* out, float* lse, uint32_t* dev_status, void* stream) {
  // the checks of ssa_decode_attn_sparse in its order, so that a bad call gets the same status from both
  if (!desc || !q || !k_cache || !v_cache || !ctx_lens || !out || !index || !counts) return SSA_ERR_NULL;
  const int32_t rc = ssa::check_desc(desc);
  if (rc != SSA_OK) return rc;
  if (index_stride <= 0 || max_selected <= 0 || max_selected > index_stride) return SSA_ERR_CAPACITY;
  if (!ssa::aligned16(q) || !ssa::aligned16(k_cache) || !ssa::aligned16(v_cache) || !ssa::aligned16(out))
    return SSA_ERR_ALIGN;
  ssa::Plan pl;
  // (groups above kGqaHeads are taken as far as their one-head-per-block plan fits, like multi-head calls)
  const bool share = ssa::can_share_rows(desc) && ssa::head_splits(desc) == 1;
  if (!ssa::make_plan(desc, max_selected, share, false, &pl)) return SSA_ERR_SHAPE;
  if (pl.total_bytes > SSA_STATIC_SCRATCH_BYTES) return SSA_ERR_WORKSPACE;   // beyond the built-in scratch
  void* scratch = ssa::static_scratch_address();
  if (!scratch) return SSA_ERR_CUDA;
  return ssa::run(desc, q, k_cache, v_cache, ctx_lens, index, index_stride, counts, max_selected, out, lse,
                  scratch, SSA_STATIC_SCRATCH_BYTES, dev_status, stream, ssa::kIndex);
}

// Layout of the workspace of ssa_decode_attn_spans: the partial results of the split pass, one int32 per
// request, and - only when the request may have more spans than a block merges in shared memory and the
// list is expanded by ssa_spans_to_index first - room for the index lists.
static size_t spans_index_pitch(int32_t max_selected) { return ((size_t)max_selected + 31) / 32 * 32; }

size_t ssa_decode_spans_workspace_bytes(const ssa_attn_desc* desc, int32_t max_selected, int32_t max_spans) {
  if (!desc || max_spans <= 0 || ssa::check_desc(desc) != SSA_OK) return 0;
  size_t need = ssa::plan_bytes(desc, max_selected);
  if (need == 0) return 0;
  need += ssa::counts_bytes(desc);
  if (max_spans > ssa::kDirectSpans) need += (size_t)desc->B * spans_index_pitch(max_selected) * sizeof(int32_t);
  return need;
}

int32_t ssa_decode_attn_spans(const ssa_attn_desc* desc, const void* q, const void* k_cache, const void* v_cache,
                              const int32_t* ctx_lens, const int32_t* span_offsets, const int32_t* spans,
                              int32_t max_spans, int32_t max_selected, void* out, float* lse, int32_t* index_out,
                              int32_t index_stride, int32_t* counts_out, void* workspace, size_t workspace_bytes,
                              uint32_t* dev_status, void* stream) {
  if (!desc || !spans) return SSA_ERR_NULL;
  if (max_spans <= 0) return SSA_ERR_CAPACITY;
  if (!span_offsets && max_spans > ssa::kDirectSpans) return SSA_ERR_UNSUPPORTED;
  if (max_spans <= ssa::kDirectSpans) {
    const ssa::SpanLists sl = {span_offsets, spans, max_spans, index_out, counts_out};
    return ssa::run(desc, q, k_cache, v_cache, ctx_lens, nullptr, index_stride, nullptr, max_selected, out, lse,
                    workspace, workspace_bytes, dev_status, stream, ssa::kSpans, nullptr, nullptr, &sl);
  }
  // More spans per request than a block merges on chip: expand the lists once (into the caller's buffers
  // when given, else into the workspace) and attend through them.
  if (!q || !k_cache || !v_cache || !ctx_lens || !out) return SSA_ERR_NULL;
  const int32_t rc = ssa::check_desc(desc);
  if (rc != SSA_OK) return rc;
  ssa::Plan pl;
  if (max_selected <= 0 || (index_out && max_selected > index_stride)) return SSA_ERR_CAPACITY;
  const size_t list_bytes = ssa::counts_bytes(desc) + (size_t)desc->B * spans_index_pitch(max_selected) * sizeof(int32_t);
  if (!ssa::choose_plan(desc, max_selected, workspace_bytes - std::min(workspace_bytes, list_bytes), &pl)) return SSA_ERR_SHAPE;
  if (!workspace || workspace_bytes < pl.total_bytes + list_bytes) return SSA_ERR_WORKSPACE;
  if (!ssa::aligned16(workspace)) return SSA_ERR_ALIGN;
  const size_t partial_bytes = (workspace_bytes - list_bytes) / 256 * 256;
  char* ws = static_cast<char*>(workspace);
  int32_t* counts = counts_out ? counts_out : reinterpret_cast<int32_t*>(ws + partial_bytes);
  int32_t* index = index_out ? index_out : reinterpret_cast<int32_t*>(ws + partial_bytes + ssa::counts_bytes(desc));
  const int32_t pitch = index_out ? index_stride : (int32_t)spans_index_pitch(max_selected);
  const int32_t cap = max_spans < SSA_MAX_SPANS_PER_SEQ ? max_spans : SSA_MAX_SPANS_PER_SEQ;
  const int32_t rc2 = ssa::spans_to_index_capped(span_offsets, spans, ctx_lens, desc->B, index, pitch, max_selected,
                                                 cap, counts, dev_status, (cudaStream_t)stream);
  if (rc2 != SSA_OK) return rc2;
  return ssa::run(desc, q, k_cache, v_cache, ctx_lens, index, pitch, counts, max_selected, out, lse, workspace,
                  partial_bytes, dev_status, stream, ssa::kIndex);
}

// Several query tokens per head: (head, token) pairs become the heads of a wider descriptor over the same cache
// heads, so that the kernel for grouped query heads reads every selected row once for all of them.
static int32_t widen_for_tokens(const ssa_attn_desc* desc, int32_t n_q, int64_t q_stride_t, int64_t o_stride_t,
                                ssa_attn_desc* wide) {
  if (!desc) return SSA_ERR_NULL;
  if (n_q <= 0 || (long long)desc->H * n_q > 65535) return SSA_ERR_SHAPE;
  if (desc->q_stride_h != (int64_t)n_q * q_stride_t || desc->o_stride_h != (int64_t)n_q * o_stride_t)
    return SSA_ERR_UNSUPPORTED;                          // the rows of one head must lie side by side
  *wide = *desc;
  wide->H = desc->H * n_q;
  wide->q_stride_h = q_stride_t;
  wide->o_stride_h = o_stride_t;
  return SSA_OK;
}

size_t ssa_decode_multiq_workspace_bytes(const ssa_attn_desc* desc, int32_t n_q, int32_t max_selected) {
  ssa_attn_desc wide;
  if (!desc || widen_for_tokens(desc, n_q, desc->q_stride_h / (n_q > 0 ? n_q : 1),
                                desc->o_stride_h / (n_q > 0 ? n_q : 1), &wide) != SSA_OK)
    return 0;
  return ssa_decode_workspace_bytes(&wide, max_selected);
}

int32_t ssa_decode_attn_sparse_multiq(const ssa_attn_desc* desc, int32_t n_q, int64_t q_stride_t, int64_t o_stride_t,
                                      const void* q, const void* k_cache, const void* v_cache,
                                      const int32_t* ctx_lens, const int32_t* index, int32_t index_stride,
                                      const int32_t* counts, int32_t max_selected, void* out, float* lse,
                                      void* workspace, size_t workspace_bytes, uint32_t* dev_status, void* stream) {
  ssa_attn_desc wide;
  const int32_t rc = widen_for_tokens(desc, n_q, q_stride_t, o_stride_t, &wide);
  if (rc != SSA_OK) return rc;
  return ssa::run(&wide, q, k_cache, v_cache, ctx_lens, index, index_stride, counts, max_selected, out, lse,
                  workspace, workspace_bytes, dev_status, stream, ssa::kIndex);
}

int32_t ssa_decode_attn_dense_multiq(const ssa_attn_desc* desc, int32_t n_q, int64_t q_stride_t, int64_t o_stride_t,
                                     const void* q, const void* k_cache, const void* v_cache,
                                     const int32_t* ctx_lens, void* out, float* lse, void* workspace,
                                     size_t workspace_bytes, uint32_t* dev_status, void* stream) {
  ssa_attn_desc wide;
  const int32_t rc = widen_for_tokens(desc, n_q, q_stride_t, o_stride_t, &wide);
  if (rc != SSA_OK) return rc;
  return ssa::run(&wide, q, k_cache, v_cache, ctx_lens, nullptr, 0, nullptr, 0, out, lse, workspace,
                  workspace_bytes, dev_status, stream, ssa::kDense);
}

size_t ssa_decode_blockmask_workspace_bytes(const ssa_attn_desc* desc, int32_t block_size, int32_t max_blocks) {
  ssa::Plan pl;
  if (!desc || ssa::check_desc(desc) != SSA_OK || !ssa::make_plan_blockmask(desc, block_size, max_blocks, &pl))
    return 0;
  return pl.total_bytes;
}

int32_t ssa_decode_attn_blockmask(const ssa_attn_desc* desc, const void* q, const void* k_cache,
                                  const void* v_cache, const int32_t* ctx_lens, const int32_t* block_idx,
                                  const uint32_t* block_mask, int32_t block_stride, const int32_t* block_counts,
                                  int32_t block_size, int32_t max_blocks, void* out, float* lse,
                                  void* workspace, size_t workspace_bytes, uint32_t* dev_status, void* stream) {
  const ssa::BlockList bl = {block_idx, block_mask, block_size};
  return ssa::run(desc, q, k_cache, v_cache, ctx_lens, nullptr, block_stride, block_counts, max_blocks, out, lse,
                  workspace, workspace_bytes, dev_status, stream, ssa::kBlockMask, &bl);
}

size_t ssa_decode_workspace_bytes(const ssa_attn_desc* desc, int32_t max_selected) {
  ssa::Plan pl;
  if (!desc || ssa::check_desc(desc) != SSA_OK || !ssa::make_plan(desc, max_selected, &pl)) return 0;
  const size_t need = ssa::plan_bytes(desc, max_selected);
  if (max_selected < desc->max_ctx) return need;
  size_t acc = 0;                                        // the bound of a full context: room for even shares as well
  return std::max(need, ssa::even_bytes(desc, ssa::even_blocks_wanted(desc, pl), &acc));
}

int32_t ssa_decode_attn_sparse(const ssa_attn_desc* desc, const void* q, const void* k_cache,
                               const void* v_cache, const int32_t* ctx_lens, const int32_t* index,
                               int32_t index_stride, const int32_t* counts, int32_t max_selected,
                               void* out, float* lse, void* workspace, size_t workspace_bytes,
                               uint32_t* dev_status, void* stream) {
  return ssa::run(desc, q, k_cache, v_cache, ctx_lens, index, index_stride, counts, max_selected, out,
                  lse, workspace, workspace_bytes, dev_status, stream, ssa::kIndex);
}

int32_t ssa_decode_attn_dense(const ssa_attn_desc* desc, const void* q, const void* k_cache,
                              const void* v_cache, const int32_t* ctx_lens, void* out, float* lse,
                              void* workspace, size_t workspace_bytes, uint32_t* dev_status,
                              void* stream) {
  return ssa::run(desc, q, k_cache, v_cache, ctx_lens, nullptr, 0, nullptr, 0, out, lse, workspace,
                  workspace_bytes, dev_status, stream, ssa::kDense);
}

int32_t ssa_decode_attn_sparse_paged(const ssa_attn_desc* desc, const void* q, const void* k_pool,
                                     const void* v_pool, const ssa_paging* paging, const int32_t* ctx_lens,
                                     const int32_t* index, int32_t index_stride, const int32_t* counts,
                                     int32_t max_selected, void* out, float* lse, void* workspace,
                                     size_t workspace_bytes, uint32_t* dev_status, void* stream) {
  if (!paging) return SSA_ERR_NULL;
  return ssa::run(desc, q, k_pool, v_pool, ctx_lens, index, index_stride, counts, max_selected, out, lse,
                  workspace, workspace_bytes, dev_status, stream, ssa::kIndex, nullptr, paging);
}

int32_t ssa_decode_attn_dense_paged(const ssa_attn_desc* desc, const void* q, const void* k_pool,
                                    const void* v_pool, const ssa_paging* paging, const int32_t* ctx_lens,
                                    void* out, float* lse, void* workspace, size_t workspace_bytes,
                                    uint32_t* dev_status, void* stream) {
  if (!paging) return SSA_ERR_NULL;
  return ssa::run(desc, q, k_pool, v_pool, ctx_lens, nullptr, 0, nullptr, 0, out, lse, workspace,
                  workspace_bytes, dev_status, stream, ssa::kDense, nullptr, paging);
}

}  // extern "C"
