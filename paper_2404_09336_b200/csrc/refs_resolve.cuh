// Resolution of one request's references into token spans, shared by
// ssa_refs_to_spans (spans written to global memory) and ssa_refs_to_index
// (spans kept in shared memory and expanded at once).
#pragma once
#include "ssa_common.cuh"

namespace ssa {

// Where request b's tables begin and how long they are, and its first two spans.
struct RefTables {
  int l0, n_lines, a0, n_anchors, r0, n_refs;
  int2 prefix, current;                     // the instruction prefix and the line being generated
};
// They follow from nine words: one trip to memory.
constexpr int kRefWords = 9;
__device__ __forceinline__ const int32_t* ref_word(const ssa_anchor_tables& t, int b, int i) {
  switch (i) {
    case 0: return t.line_offsets + b;
    case 1: return t.line_offsets + b + 1;
    case 2: return t.anchor_offsets + b;
    case 3: return t.anchor_offsets + b + 1;
    case 4: return t.ref_offsets + b;
    case 5: return t.ref_offsets + b + 1;
    case 6: return t.prefix_len + b;
    case 7: return t.line_start + b;
    default: return t.ctx_lens + b;
  }
}
// word(i): the value of the i-th.
template <typename Word>
__device__ __forceinline__ RefTables locate_refs(Word word) {
  RefTables r;
  r.l0 = word(0);
  r.n_lines = max(word(1) - r.l0, 0);
  r.a0 = word(2);
  r.n_anchors = max(word(3) - r.a0, 0);
  r.r0 = word(4);
  r.n_refs = max(word(5) - r.r0, 0);
  r.prefix = make_int2(0, word(6));
  r.current = make_int2(word(7), word(8));
  return r;
}

// The tables as they lie in global memory.
struct RefsInMemory {
  const int2 *lines, *refs;
  const int32_t* anchors;
  __device__ __forceinline__ RefsInMemory(const ssa_anchor_tables& t, const RefTables& r)
      : lines(reinterpret_cast<const int2*>(t.lines) + r.l0), refs(reinterpret_cast<const int2*>(t.refs) + r.r0),
        anchors(t.anchor_line + r.a0) {}
  __device__ __forceinline__ int2 line(int i) const { return __ldg(lines + i); }
  __device__ __forceinline__ int2 ref(int i) const { return __ldg(refs + i); }
  __device__ __forceinline__ int anchor(int i) const { return __ldg(anchors + i); }
};

// Called by all 32 lanes of one warp for one request.  Span 0 is the
// instruction prefix, span 1 the line being generated; then the lanes take the
// references 32 at a time: each lane resolves one (lo, hi) pair to a first
// line and a count of lines, a shuffle prefix sum turns the counts into output
// positions, and the lane hands its spans to put(position, span).  Returns the
// number of spans the request resolves to (put decides what to do with
// positions beyond its capacity).  `tables`: RefsInMemory, or a copy of what
// that shows.
template <typename Tables, typename Put>
__device__ __forceinline__ int resolve_refs_warp(const RefTables& r, const Tables& tables, int lane, uint32_t& flags,
                                                 Put put) {
  const int n_lines = r.n_lines, n_anchors = r.n_anchors, n_refs = r.n_refs;
  if (lane == 0) {
    put(0, r.prefix);
    put(1, r.current);
  }
  int written = 2;
  for (int base = 0; base < n_refs; base += 32) {
    // this lane's reference: anchors [first, first + count) or one earlier line
    int first = 0, count = 0;
    bool by_anchor = false;
    if (base + lane < n_refs) {
      const int2 ref = tables.ref(base + lane);
      if (ref.x == ref.y && ref.x < 0) {
        if (n_lines + ref.x >= 0) { first = n_lines + ref.x; count = 1; }
        else flags |= SSA_DEV_BAD_REF;
      } else if (ref.x >= 0 && ref.x <= ref.y) {
        // anchors past the end of the table do not exist: flag them and walk only the ones that do, so the
        // work per reference is bounded by the table whatever the pair says
        int hi = ref.y;
        if (hi >= n_anchors) { hi = n_anchors - 1; flags |= SSA_DEV_BAD_REF; }
        first = ref.x;
        count = max(hi - ref.x + 1, 0);
        by_anchor = true;
      } else {
        flags |= SSA_DEV_BAD_REF;
      }
    }
    // anchors that do not resolve are dropped, so count what each lane really emits (table reads four at a
    // time: a lane's walk over its anchors is a chain of dependent-looking loads otherwise)
    int emit = 0;
    if (by_anchor) {
      for (int a = first; a < first + count; a += 4) {
        int li[4];
#pragma unroll
        for (int k = 0; k < 4; ++k)
          li[k] = (a + k < first + count && a + k < n_anchors) ? tables.anchor(a + k) : -1;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          if (a + k >= first + count) break;
          if (li[k] >= 0 && li[k] < n_lines) ++emit; else flags |= SSA_DEV_BAD_REF;
        }
      }
    } else {
      emit = count;
    }
    int incl = emit;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const int o = __shfl_up_sync(0xffffffffu, incl, d);
      if (lane >= d) incl += o;
    }
    int at = written + incl - emit;
    if (by_anchor) {
      for (int a = first; a < first + count; a += 4) {
        int li[4];
        int2 span[4];
#pragma unroll
        for (int k = 0; k < 4; ++k)
          li[k] = (a + k < first + count && a + k < n_anchors) ? tables.anchor(a + k) : -1;
#pragma unroll
        for (int k = 0; k < 4; ++k)
          span[k] = (li[k] >= 0 && li[k] < n_lines) ? tables.line(li[k]) : make_int2(0, 0);
#pragma unroll
        for (int k = 0; k < 4; ++k)
          if (li[k] >= 0 && li[k] < n_lines) put(at++, span[k]);
      }
    } else if (count == 1) {
      put(at, tables.line(first));
    }
    written += __shfl_sync(0xffffffffu, incl, 31);
  }
  return written;
}

// Host-side check of the tables shared by both entry points.
inline int32_t check_anchor_tables(const ssa_anchor_tables* t) {
  if (!t) return SSA_ERR_NULL;
  if (!t->line_offsets || !t->lines || !t->anchor_offsets || !t->anchor_line || !t->ref_offsets || !t->refs ||
      !t->prefix_len || !t->line_start || !t->ctx_lens)
    return SSA_ERR_NULL;
  if (reinterpret_cast<uintptr_t>(t->lines) % 8 || reinterpret_cast<uintptr_t>(t->refs) % 8) return SSA_ERR_ALIGN;
  return SSA_OK;
}

}  // namespace ssa
