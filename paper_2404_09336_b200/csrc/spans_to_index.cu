// Span list -> sorted duplicate-free KV index list (ssa_spans_to_index).
//
// One thread block per (output slice, request).  The block
//   1. loads the request's spans, clamps them to [0, ctx_len) and packs each
//      non-empty one into a 64-bit key (start << 32 | end);
//   2. sorts the keys by start: up to 32 spans by rank counting inside one
//      warp (shuffles only), up to 256 by rank counting in shared memory, more
//      by a bitonic network in shared memory;
//   3. has one warp walk the sorted spans 32 at a time with two shuffle
//      scans: a running maximum of the span ends seen so far, which trims
//      each span to the part no earlier span covers, and a prefix sum of the
//      trimmed lengths, which gives every span its offset in the output;
//   4. writes its slice of the output: slot k finds its span by binary
//      search over the offsets, so the stores are coalesced and balanced
//      however uneven the spans are.
// Blocks of one request repeat steps 1-3 (a few microseconds) instead of
// communicating.
//
// ssa_refs_to_index runs the same kernel with another step 1: one warp
// resolves the request's references into spans (as ssa_refs_to_spans does) and
// packs them straight into the keys in shared memory, so the span list never
// goes through global memory and the step is one launch instead of two.
// The kernel is a chain of trips to memory.  Resolving walks references,
// anchors and lines, each naming the next; the block therefore first copies
// the request's tables to shared memory in one trip (up to kTable entries
// each): 16 requests of 4..50 spans 9.0 -> 4.2 us, 2 of them 6.0 -> 3.3 us (with the
// ranking of up to 256 spans and the shorter slices; span lists 3.3 -> 2.3 us, 64 of
// 3..6 spans 2.6 -> 2.4 us).
#include <algorithm>

#include "fetch_index.cuh"
#include "refs_resolve.cuh"

namespace ssa {

constexpr int kIdxThreads = 128;
constexpr int kMaxSpans = SSA_MAX_SPANS_PER_SEQ;   // power of two
constexpr int kRankSpans = 2 * kIdxThreads;        // most spans ranked by counting: two per thread
constexpr int kTable = 512;                        // most entries of an anchor table that are copied to shared memory
constexpr int kEarlyBlocks = 4;                    // per SM: the first of a launch guess
constexpr unsigned long long kEmptyKey = 0xffffffffffffffffull;

// Where the spans of a request come from: a span list in global memory, or the anchor tables.
struct SpanSource {
  const int32_t* span_offsets;
  const int32_t* spans;
  const int32_t* ctx_lens;
  ssa_anchor_tables tables;
  // entries that may be read from these on before their offsets can be trusted (0: none); for blocks below early_blocks
  int32_t spans_readable, lines_readable, anchors_readable, refs_readable, early_blocks;
};

// kFetch: rows of the grid from first_row on do not expand a request but copy n16 16-byte words from page-locked
// host memory to the device (the step's inputs), while the other rows read their span lists straight from
// that host memory: the fetch of a decode step's inputs and its index expansion overlap in one launch.
struct FetchJob {
  uint4* dst;
  const uint4* src;
  size_t n16;
  int32_t first_row;
};

template <bool kFromRefs, bool kFetch = false>
__global__ void __launch_bounds__(kIdxThreads)
spans_to_index_kernel(const SpanSource src, int32_t* __restrict__ index,
                      int32_t index_stride, int32_t slice, int32_t* __restrict__ counts,
                      uint32_t* __restrict__ dev_status, const FetchJob job,
                      int32_t capacity, int32_t span_cap, const Spare<24>) {
  // index_stride: distance between the rows of `index`; capacity <= index_stride: most positions a list keeps;
  // span_cap <= kMaxSpans: most spans a request may have
  if (kFetch && (int)blockIdx.y >= job.first_row) {
    grid_dependency_wait();                      // the destination may still be read by the previous kernel
    const size_t n_threads = (size_t)(gridDim.y - job.first_row) * gridDim.x * kIdxThreads;
    size_t i = ((size_t)(blockIdx.y - job.first_row) * gridDim.x + blockIdx.x) * kIdxThreads + threadIdx.x;
    for (; i + n_threads < job.n16; i += 2 * n_threads) {   // two requests in flight per thread
      const uint4 a = job.src[i], c = job.src[i + n_threads];
      job.dst[i] = a;
      job.dst[i + n_threads] = c;
    }
    if (i < job.n16) job.dst[i] = job.src[i];
    return;
  }
  __shared__ __align__(16) unsigned long long keys[kMaxSpans];
  __shared__ __align__(16) int32_t new_start[kMaxSpans];
  __shared__ __align__(16) int32_t offs[kMaxSpans + 1];
  __shared__ uint32_t s_flags;
  __shared__ int s_resolved;
  constexpr int kWords = kFromRefs ? kRefWords : 3;
  __shared__ int32_t s_words[kWords];
  const int32_t* __restrict__ spans = src.spans;

  const int b = blockIdx.y;
  const int tid = threadIdx.x;
  // Steps 1-3 run while the kernel in front drains, on the lists as they stand, and again only if they have changed by then:
  // seeing that they have not takes one trip to memory, the steps two or three and half a microsecond.  Spans to lists and
  // attention, 64 requests 28.8 -> 28.1 us; references and attention, 2 requests of ~25 spans 11.6 -> 9.5, 36 of ~38, 8 heads,
  // 23.9 -> 21.3, 16 of 2 to 50, 32 heads, 41.6 -> 40.5; 51 of ~20, behind a merge, 89.6 -> 88.1.
  bool guess = !kFetch && (int)(blockIdx.y * gridDim.x + blockIdx.x) < src.early_blocks;
  if (!guess) grid_dependency_wait();   // dependents are released when this grid completes: blocks of a large
                                        // attention grid parked on the SMs during this kernel slowed it down
  int2* const guess_room = reinterpret_cast<int2*>(keys + 2 * kRankSpans);
  static_assert(2 * kRankSpans * 8 + kTable * 20 <= kMaxSpans * 8, "a guess's copies lie behind its keys and starts");
  // The words that say where the request's list or tables lie, and its context, decide about barriers below.  The kernel in
  // front may be writing them, so that threads could see different ones: for a guess one warp reads them, once, and hands them out.
  auto word_at = [&](int i) -> const int32_t* {
    if constexpr (kFromRefs) return ref_word(src.tables, b, i);
    else return i == 0 ? src.ctx_lens + b : src.span_offsets + b + (i - 1);
  };
  if (guess) {
    if (tid < kWords) s_words[tid] = load_early(word_at(tid));
    __syncthreads();
  }
  int P;
  while (true) {
    auto load = [&](auto* p) { return !kFetch && guess ? load_early(p) : load_now(p); };
    auto word = [&](int i) { return !kFetch && guess ? s_words[i] : load_now(word_at(i)); };
    RefTables r = {};
    if constexpr (kFromRefs) r = locate_refs(word);
    const int n = max(kFromRefs ? r.current.y : word(0), 0);
    uint32_t flags = 0;
    if (tid == 0) s_flags = 0;

    // clamp a span to the context and pack it; empty spans get the sentinel
    auto pack = [&](int2 se) -> unsigned long long {
      if (se.x < 0 || se.x > se.y) flags |= SSA_DEV_BAD_SPAN;
      if (se.y > n) flags |= SSA_DEV_CLIPPED;
      const int s = max(se.x, 0), e = min(se.y, n);
      return e > s ? ((unsigned long long)(uint32_t)s << 32) | (uint32_t)e : kEmptyKey;
    };

    int first = 0, S;
    int2 raw[2] = {make_int2(0, 0), make_int2(0, 0)};   // spans tid and tid + kIdxThreads of a list of up to kRankSpans
    if constexpr (kFromRefs) {
      // 1 (references): warp 0 resolves them and leaves the packed spans, unsorted, in keys[0, S)
      static_assert(4 * kTable <= kMaxSpans, "the copies lie in arrays that step 3 fills");
      struct Copied {
        int2 *lines, *refs;
        int32_t* anchors;
        __device__ __forceinline__ int2 line(int i) const { return lines[i]; }
        __device__ __forceinline__ int2 ref(int i) const { return refs[i]; }
        __device__ __forceinline__ int anchor(int i) const { return anchors[i]; }
      };
      const RefsInMemory far(src.tables, r);
      // (a guess needs its copies for the comparison: behind the keys of a list of up to kRankSpans, where nothing else comes)
      int2* const room = guess ? guess_room : reinterpret_cast<int2*>(new_start);
      const Copied near = {room, room + kTable, guess ? reinterpret_cast<int32_t*>(room + 2 * kTable) : offs};
      const bool copied = r.n_lines <= kTable && r.n_anchors <= kTable && r.n_refs <= kTable;
      if (guess && !(copied && r.l0 >= 0 && r.a0 >= 0 && r.r0 >= 0 && r.l0 <= src.lines_readable - r.n_lines &&
                     r.a0 <= src.anchors_readable - r.n_anchors && r.r0 <= src.refs_readable - r.n_refs)) {
        grid_dependency_wait();                         // no guess; the same for all threads, as r is
        guess = false;
        continue;
      }
      if (copied) {
        for (int i = tid; i < max(max(r.n_lines, r.n_anchors), r.n_refs); i += kIdxThreads) {
          int2 line = make_int2(0, 0), ref = line;        // all three requested before any is stored
          int anchor = 0;
          if (i < r.n_lines) line = load(far.lines + i);
          if (i < r.n_anchors) anchor = load(far.anchors + i);
          if (i < r.n_refs) ref = load(far.refs + i);
          if (i < r.n_lines) near.lines[i] = line;
          if (i < r.n_anchors) near.anchors[i] = anchor;
          if (i < r.n_refs) near.refs[i] = ref;
        }
        __syncthreads();
      }
      if (tid < 32) {
        auto put = [&](int at, int2 span) {
          if (at < (guess ? kRankSpans : kMaxSpans)) keys[at] = pack(span);
        };
        const int resolved = copied ? resolve_refs_warp(r, near, tid, flags, put) : resolve_refs_warp(r, far, tid, flags, put);
        if (tid == 0) s_resolved = resolved;
      }
      __syncthreads();
      S = s_resolved;
      if (guess && S > kRankSpans) {
        __syncthreads();                                // every thread has read s_resolved
        grid_dependency_wait();
        guess = false;
        continue;
      }
    } else {
      first = word(1);
      S = word(2) - first;
      if (guess && !(first >= 0 && S >= 0 && S <= min(span_cap, kRankSpans) && first <= src.spans_readable - S)) {
        grid_dependency_wait();
        guess = false;
        continue;
      }
    }
    if (S < 0) S = 0;
    if (S > span_cap) { S = span_cap; flags |= SSA_DEV_TOO_MANY_SPANS; }
    P = (max(S, 1) + 31) & ~31;
    if (S > kRankSpans)
      for (P = 2 * kRankSpans; P < S;) P <<= 1;
    if constexpr (!kFromRefs) {
      if (S <= kRankSpans) {
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          const int i = tid + k * kIdxThreads;
          if (i < S) raw[k] = load(reinterpret_cast<const int2*>(spans) + first + i);
          if (guess && i < S) guess_room[i] = raw[k];
        }
      }
      __syncthreads();                                    // s_flags
    }

    auto load_key = [&](int i) -> unsigned long long {
      if (i >= S) return kEmptyKey;
      if (kFromRefs) return keys[i];
      if (S <= kRankSpans) return pack(raw[i / kIdxThreads]);   // i is tid or tid + kIdxThreads
      return pack(reinterpret_cast<const int2*>(spans)[first + i]);
    };

    if (P == 32) {
      // 1+2 (up to 32 spans, the usual case): one warp ranks its starts with shuffles, no block barrier needed.  (The ends do
      // not order: the walk of step 3 trims by the largest end so far.)
      if (tid < 32) {
        const unsigned long long key = load_key(tid);
        if (kFromRefs) __syncwarp();                  // every lane has read its key before any is overwritten
        const uint32_t start = (uint32_t)(key >> 32);
        int rank = 0;
        for (int j = 0; j < S; ++j) {
          const uint32_t sj = __shfl_sync(0xffffffffu, start, j);
          rank += (sj < start || (sj == start && j < tid)) ? 1 : 0;
        }
        keys[tid < S ? rank : tid] = key;
        __syncwarp();
      }
    } else if (P <= kRankSpans) {
      uint32_t* starts = reinterpret_cast<uint32_t*>(keys + kRankSpans);   // the unsorted starts, read four at a time
      unsigned long long key[2];
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        const int i = tid + k * kIdxThreads;
        key[k] = i < P ? load_key(i) : kEmptyKey;
        if (i < P) starts[i] = (uint32_t)(key[k] >> 32);
      }
      __syncthreads();                                // also: every key of the references has been read
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        const int i = tid + k * kIdxThreads;
        if (i < P) {
          const uint32_t start = (uint32_t)(key[k] >> 32);
          int rank = 0;
          for (int j = 0; j < P; j += 4) {
            const uint4 s4 = *reinterpret_cast<const uint4*>(starts + j);
            rank += (s4.x < start || (s4.x == start && j < i)) ? 1 : 0;
            rank += (s4.y < start || (s4.y == start && j + 1 < i)) ? 1 : 0;
            rank += (s4.z < start || (s4.z == start && j + 2 < i)) ? 1 : 0;
            rank += (s4.w < start || (s4.w == start && j + 3 < i)) ? 1 : 0;
          }
          keys[rank] = key[k];
        }
      }
      __syncthreads();
    } else {
      // 1. load, clamp, pack (references: the keys are in place, only the padding is missing)
      for (int i = tid; i < P; i += kIdxThreads)
        if (!kFromRefs || i >= S) keys[i] = load_key(i);
      __syncthreads();
      // 2. bitonic sort, ascending by (start, end); empty keys sink to the end
      for (int k = 2; k <= P; k <<= 1) {
        for (int j = k >> 1; j > 0; j >>= 1) {
          for (int i = tid; i < P; i += kIdxThreads) {
            const int ixj = i ^ j;
            if (ixj > i) {
              const unsigned long long a = keys[i], c = keys[ixj];
              const bool up = (i & k) == 0;
              if ((a > c) == up) { keys[i] = c; keys[ixj] = a; }
            }
          }
          __syncthreads();
        }
      }
    }

    // 3. trim against the running maximum end and prefix-sum the lengths
    bool changed = false;
    if (tid < 32) {
      int run_max = 0, run_sum = 0;
      for (int base = 0; base < P; base += 32) {
        const unsigned long long key = keys[base + tid];
        const bool live = key != kEmptyKey;
        const int s = live ? (int)(key >> 32) : 0;
        const int e = live ? (int)(uint32_t)key : 0;
        int mx = e;                                   // inclusive max-scan of ends
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
          const int o = __shfl_up_sync(0xffffffffu, mx, d);
          if (tid >= d) mx = max(mx, o);
        }
        int prev = __shfl_up_sync(0xffffffffu, mx, 1);
        prev = (tid == 0) ? run_max : max(prev, run_max);
        const int ns = max(s, prev);
        const int len = live ? max(e - ns, 0) : 0;
        int sum = len;                                // inclusive sum-scan of lengths
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
          const int o = __shfl_up_sync(0xffffffffu, sum, d);
          if (tid >= d) sum += o;
        }
        new_start[base + tid] = ns;
        offs[base + tid] = run_sum + sum - len;
        run_max = max(run_max, __shfl_sync(0xffffffffu, mx, 31));
        run_sum += __shfl_sync(0xffffffffu, sum, 31);
      }
      if (tid == 0) offs[P] = run_sum;
    } else if (!kFetch && guess) {
      // Meanwhile the other warps see whether the guess still holds, so that its trip is not one more where there was no time in
      // front of the wait.  us, references and attention behind an elementwise kernel, compared after the lists have been made /
      // meanwhile / without guesses: 1 request of 32 heads 16.6 / 15.3 / 14.8, 9 29.2 / 28.6 / 28.0; between such calls 6 of 8 heads
      // 13.6 / 12.9 / 13.4.
      grid_dependency_wait();
      const int t = tid - 32;
      constexpr int kStep = kIdxThreads - 32;
      changed = t < kWords && load_now(word_at(t)) != s_words[t];
      if constexpr (kFromRefs) {
        const RefsInMemory far(src.tables, r);
        const int2 *lines = guess_room, *refs = guess_room + kTable;
        const int32_t* anchors = reinterpret_cast<const int32_t*>(guess_room + 2 * kTable);
        for (int i = t; i < max(max(r.n_lines, r.n_anchors), r.n_refs); i += kStep) {
          int2 line = make_int2(0, 0), ref = line;
          int anchor = 0;
          if (i < r.n_lines) line = load_now(far.lines + i);
          if (i < r.n_anchors) anchor = load_now(far.anchors + i);
          if (i < r.n_refs) ref = load_now(far.refs + i);
          changed |= i < r.n_lines && (line.x != lines[i].x || line.y != lines[i].y);
          changed |= i < r.n_anchors && anchor != anchors[i];
          changed |= i < r.n_refs && (ref.x != refs[i].x || ref.y != refs[i].y);
        }
      } else {
        const int2* list = reinterpret_cast<const int2*>(spans) + first;
        for (int i = t; i < S; i += kStep) {
          const int2 now = load_now(list + i), then = guess_room[i];
          changed |= now.x != then.x || now.y != then.y;
        }
      }
    }
    if (flags) atomicOr(&s_flags, flags);
    if (kFetch || !guess) {
      __syncthreads();
      break;
    }
    grid_dependency_wait();
    guess = false;
    if (!__syncthreads_or(changed)) break;
  }

  const int total = offs[P];
  const int c = min(total, capacity);
  if (blockIdx.x == 0 && tid == 0) {
    counts[b] = c;
    uint32_t f = s_flags;
    if (total > capacity) f |= SSA_DEV_OVERFLOW;
    if (f && dev_status) atomicOr(dev_status, f);
  }

  // 4. write this block's slice of the list
  const int k_end = min(c, (int)(blockIdx.x + 1) * slice);
  int32_t* row = index + (size_t)b * index_stride;
  for (int k = blockIdx.x * slice + tid; k < k_end; k += kIdxThreads) {
    int lo = 0, hi = P;                             // last i with offs[i] <= k
    while (hi - lo > 1) {
      const int mid = (lo + hi) >> 1;
      if (offs[mid] <= k) lo = mid; else hi = mid;
    }
    row[k] = new_start[lo] + (k - offs[lo]);
  }
}

// Entries of a list that one block writes, and the blocks per request (at most 32): 512 entries each, or fewer while that
// leaves the launch within one block per SM, where repeating steps 1-3 costs nothing and a thread writes its entries one
// after the other.
static int32_t slice_of(int32_t B, int32_t capacity, int* slices) {
  int entries = 512;
  while (entries > kIdxThreads && (long long)B * ((capacity + entries / 2 - 1) / (entries / 2)) <= sm_count()) entries /= 2;
  *slices = std::min((capacity + entries - 1) / entries, 32);
  return (capacity + *slices - 1) / *slices;
}

// ssa_spans_to_index with the span lists read from page-locked host memory (host_* are host addresses the
// device can use), fused with the copy of `bytes` bytes from src (the same kind of memory) to dst (device).  (No guess: two
// readings across the bus, 43 -> 92 us.)
int32_t fetch_and_index(const int32_t* host_span_offsets, const int32_t* host_spans, const int32_t* host_ctx_lens,
                        int32_t B, int32_t* index, int32_t index_stride, int32_t* counts, uint32_t* dev_status,
                        void* dst, const void* src, size_t bytes, cudaStream_t stream) {
  if (!host_span_offsets || !host_spans || !host_ctx_lens || !index || !counts || !dst || !src) return SSA_ERR_NULL;
  if (B <= 0 || index_stride <= 0) return SSA_ERR_SHAPE;
  if (reinterpret_cast<uintptr_t>(host_spans) % 8 != 0 || bytes % 16 != 0 ||
      reinterpret_cast<uintptr_t>(dst) % 16 != 0 || reinterpret_cast<uintptr_t>(src) % 16 != 0)
    return SSA_ERR_ALIGN;
  int slices = (index_stride + 511) / 512;
  if (slices > 32) slices = 32;
  const int32_t slice = (index_stride + slices - 1) / slices;
  const size_t n16 = bytes / 16;
  const size_t per_row = (size_t)slices * kIdxThreads * 2;            // two words per thread
  const int copy_rows = (int)std::min<size_t>((n16 + per_row - 1) / per_row, (size_t)sm_count() * 8);
  if (B + copy_rows > 65535) return SSA_ERR_SHAPE;
  SpanSource s = {};
  s.span_offsets = host_span_offsets; s.spans = host_spans; s.ctx_lens = host_ctx_lens;
  FetchJob job = {reinterpret_cast<uint4*>(dst), reinterpret_cast<const uint4*>(src), n16, B};
  dim3 grid((unsigned)slices, (unsigned)(B + std::max(copy_rows, 1)));
  const cudaError_t err = launch_pdl(spans_to_index_kernel<false, true>, grid, dim3(kIdxThreads), stream, s,
                                     index, index_stride, slice, counts, dev_status, job, index_stride, kMaxSpans, Spare<24>{});
  if (err != cudaSuccess || cudaGetLastError() != cudaSuccess) return SSA_ERR_CUDA;
  note_launches(1);
  return SSA_OK;
}

// ssa_spans_to_index with two more bounds: a list keeps at most `capacity` <= index_stride positions and a
// request at most `span_cap` <= SSA_MAX_SPANS_PER_SEQ spans.
int32_t spans_to_index_capped(const int32_t* span_offsets, const int32_t* spans, const int32_t* ctx_lens, int32_t B,
                              int32_t* index, int32_t index_stride, int32_t capacity, int32_t span_cap,
                              int32_t* counts, uint32_t* dev_status, cudaStream_t stream) {
  if (!span_offsets || !spans || !ctx_lens || !index || !counts) return SSA_ERR_NULL;
  if (B <= 0 || B > 65535 || index_stride <= 0) return SSA_ERR_SHAPE;
  if (capacity <= 0 || capacity > index_stride || span_cap <= 0 || span_cap > kMaxSpans) return SSA_ERR_CAPACITY;
  if (reinterpret_cast<uintptr_t>(spans) % 8 != 0) return SSA_ERR_ALIGN;
  int slices;
  const int32_t slice = slice_of(B, capacity, &slices);
  dim3 grid((unsigned)slices, (unsigned)B);
  SpanSource src = {};
  src.span_offsets = span_offsets; src.spans = spans; src.ctx_lens = ctx_lens;
  Allocation known = {};
  src.spans_readable = readable_entries<int2>(spans, &known);
  src.early_blocks = src.spans_readable > 0 ? kEarlyBlocks * sm_count() : 0;
  const cudaError_t err = launch_pdl(spans_to_index_kernel<false>, grid, dim3(kIdxThreads), stream, src, index,
                                     index_stride, slice, counts, dev_status, FetchJob{}, capacity, span_cap, Spare<24>{});
  if (err != cudaSuccess || cudaGetLastError() != cudaSuccess) return SSA_ERR_CUDA;
  note_launches(1);
  return SSA_OK;
}

}  // namespace ssa

extern "C" int32_t ssa_spans_to_index(const int32_t* span_offsets, const int32_t* spans,
                                      const int32_t* ctx_lens, int32_t B, int32_t* index,
                                      int32_t index_stride, int32_t* counts,
                                      uint32_t* dev_status, void* stream) {
  return ssa::spans_to_index_capped(span_offsets, spans, ctx_lens, B, index, index_stride, index_stride,
                                    ssa::kMaxSpans, counts, dev_status, (cudaStream_t)stream);
}

extern "C" int32_t ssa_refs_to_index(const ssa_anchor_tables* tables, int32_t B, int32_t* index,
                                     int32_t index_stride, int32_t* counts, uint32_t* dev_status,
                                     void* stream) {
  if (!index || !counts) return SSA_ERR_NULL;
  const int32_t rc = ssa::check_anchor_tables(tables);
  if (rc != SSA_OK) return rc;
  if (B <= 0 || B > 65535 || index_stride <= 0) return SSA_ERR_SHAPE;
  int slices;
  const int32_t slice = ssa::slice_of(B, index_stride, &slices);
  dim3 grid((unsigned)slices, (unsigned)B);
  ssa::SpanSource src = {};
  src.tables = *tables;
  ssa::Allocation known = {};
  src.lines_readable = ssa::readable_entries<int2>(tables->lines, &known);
  src.anchors_readable = ssa::readable_entries<int32_t>(tables->anchor_line, &known);
  src.refs_readable = ssa::readable_entries<int2>(tables->refs, &known);
  // (tables elsewhere than in one allocation of device memory, across the bus for instance, are not read twice)
  const bool readable = src.lines_readable > 0 && src.anchors_readable > 0 && src.refs_readable > 0;
  src.early_blocks = readable ? ssa::kEarlyBlocks * ssa::sm_count() : 0;
  const cudaError_t err = ssa::launch_pdl(ssa::spans_to_index_kernel<true>, grid, dim3(ssa::kIdxThreads),
                                          (cudaStream_t)stream, src, index, index_stride, slice, counts,
                                          dev_status, ssa::FetchJob{}, index_stride, ssa::kMaxSpans, ssa::Spare<24>{});
  if (err != cudaSuccess || cudaGetLastError() != cudaSuccess) return SSA_ERR_CUDA;
  ssa::note_launches(1);
  return SSA_OK;
}
