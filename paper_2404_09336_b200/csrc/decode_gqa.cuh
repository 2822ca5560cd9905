// Pass 1 of the decode attention for grouped query heads (G = H / H_kv >= 2
// query heads share one K/V head, D = 128; also several query tokens per
// head, which are served the same way): one block per (chunk, K/V head,
// request) reads every selected row ONCE and serves all G heads; above
// sixteen heads (kGqaHeads) several blocks share them.
//
// With G heads per row the work per byte is G times that of multi-head
// attention and the packed-FMA path of decode_partial_kernel runs out of issue
// slots before it runs out of HBM bandwidth, so here the two contractions go
// to the tensor cores.  The shapes are far too small for tcgen05 tiles (G x 16
// rows x 128), so they are warp-level mma.sync.m16n8k16 (16-bit inputs, fp32
// accumulation) with the N dimension holding eight query heads:
//   S^T[16 rows, 8 heads] = K_tile . Q^T : A = K tile (16 rows), B = Q
//                           (registers, loaded once);
//   O^T[16 dims, 8 heads] += V_tile^T . P^T : A = V tile, transposed, B = P
//                           from the accumulators of S, transposed by movmatrix.
// Groups of up to eight heads take one head tile, larger ones two (kHi): with
// the heads in the M dimension instead, a group of up to eight heads paid for
// sixteen, twice the matrix instructions.
// 16-bit tiles come out of shared memory with ldmatrix (.trans for V).  8-bit
// rows (e4m3) are read with plain 16-byte loads and converted to fp16 in
// registers, exactly, one instruction per pair; their bf16 query rows become
// fp16 times a power of two of their own (scaled_query), or, where that would
// lose a bit, stay bf16 against rows of K in bf16.  Which lane holds
// which dimension is free as long as Q (for K) and the output (for V) follow,
// so a lane takes whole 16-byte pieces of a row.
// The rows travel global -> shared memory by asynchronous 16-byte copies
// (cp.async, evict-first in L2) into a ring of tiles that every team of warps
// (one warp per head tile, GqaShape) keeps for itself, and the fragments come
// out of that ring.  The bytes in flight are set by the ring (three tiles of
// 16 rows x (K + V), 24 KB per team; 8-bit rows with up to eight heads: twice
// the teams with 12 KB; 96 KB per block, two blocks per SM), not by fragment
// registers, and a team works on one tile while its next two are on their way;
// a team waits for itself, no block barrier sits inside the tile loop.  (An
// earlier version loaded the fragments straight from global memory into
// registers, one tile in flight per warp: 5-15 % slower on long lists.)
//
// Shared-memory tiles are [16 rows][256 bytes] with the 16-byte chunk index
// XOR-ed with (row & 7), so that the eight row addresses of an ldmatrix hit
// eight different bank groups; [16 rows][128 bytes] for 8-bit rows (below).
// The softmax weights are the fp32 accumulators of S; they enter the second
// contraction as a 16-bit value plus a 16-bit residual (two mma passes), so
// the result keeps fp32-level accuracy instead of the 2^-9 of a bf16 weight.
// Over an 8-bit cache they are fp16 pairs of 2^13 times the weight: 22 bits
// for the large ones and an absolute error below 2^-37 of the largest for the
// rest; above sixteen heads (kSplit) further terms hold the rest as well.
// Included by decode_attn.cu after DecodeParams and its helpers.
#pragma once

namespace ssa {

template <typename T>
__device__ __forceinline__ uint32_t pack2(float lo, float hi);
template <>
__device__ __forceinline__ uint32_t pack2<__nv_bfloat16>(float lo, float hi) {
  const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&v);
}
template <>
__device__ __forceinline__ uint32_t pack2<__half>(float lo, float hi) {
  const __half2 v = __floats2half2_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&v);
}

// D(16x8, fp32) = A(16x16) . B(16x8) + C, 16-bit inputs of type T.
template <typename T>
__device__ __forceinline__ void mma_16816(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                          uint32_t b0, uint32_t b1, const float (&c)[4]);
template <>
__device__ __forceinline__ void mma_16816<__nv_bfloat16>(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2,
                                                         uint32_t a3, uint32_t b0, uint32_t b1,
                                                         const float (&c)[4]) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
               "{%10,%11,%12,%13};"
               : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
               : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1), "f"(c[0]), "f"(c[1]), "f"(c[2]), "f"(c[3]));
}
template <>
__device__ __forceinline__ void mma_16816<__half>(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                                  uint32_t b0, uint32_t b1, const float (&c)[4]) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
               "{%10,%11,%12,%13};"
               : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
               : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1), "f"(c[0]), "f"(c[1]), "f"(c[2]), "f"(c[3]));
}

constexpr int kGqaRows = 16;            // rows per warp per iteration
constexpr int kGqaHeads = 16;           // two head tiles of the mma's N = 8: most query heads one block serves
// floats per head row of the block-level combine, dim d at d + 2 (d / 16): lanes that hold dims 16 apart (8-bit rows)
// or one apart (16-bit rows) and heads two apart store to different banks
constexpr int kGqaPitch = 148;
__device__ __forceinline__ int gqa_column(int d) { return d + 2 * (d >> 4); }

// Warps and ring of a block.  A team of warps shares one ring of tiles: one warp for up to eight heads, two - one per
// head tile - for more (one warp with both head tiles had twice the instructions per tile in one dependent stream,
// and with eight such warps per SM that stream, not the memory, was what a tile waited for).  Four teams with 24 KB
// each make a block, two blocks fit an SM; 8-bit rows, whose tiles are half as large and cost more instructions
// (conversions), take twice the teams with half the ring.  Wide blocks have twice the teams, one block per SM.
template <typename T, bool kHi, bool kWide>
struct GqaShape {
  static constexpr int kTeam = kHi ? 2 : 1;
  static constexpr int kRingBytes = (kIsFp8<T> && !kHi ? 12 : 24) * 1024;
  static constexpr int kSmemBytes = (kWide ? 192 : 96) * 1024;
  static constexpr int kTeams = kSmemBytes / kRingBytes;
  static constexpr int kWarps = kTeam * kTeams;
  static constexpr int kDenseWindow = kHi ? 1024 : kIsFp8<T> ? 512 : 256;   // see below
};
// A chunk is worked through in windows: for lists, the block's warps meet and stage the next window's positions; over
// a full context, each team lets its ring run empty.  Short windows keep the teams on neighbouring rows, which the
// memory system rewards, long ones keep more in flight.  Measured with windows of 256 / 512 / 1024 rows, full context:
// 4 heads, 32 requests of 8192: 152 / 158 / 158 us; 16 heads, 26 x 3287: 62.8 / 61.4 / 60.3 us, 17 requests of
// 1001..8190: 75.8 / 74.0 / 72.7 us, 17 x 8190: 89.2 / 92.2 / 93.4 us.  8-bit rows have twice the teams: 512.
constexpr int kStagedWindow = 512;                       // list entries staged at a time ...
constexpr int kStagedShortList = 1024;                   // ... unless the whole chunk fits this many: then one window

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// 16-byte asynchronous copy global -> shared, not kept in L1, evict-first in L2.
__device__ __forceinline__ void cp_async_16(uint32_t dst, const void* src, uint64_t policy) {
  asm volatile("cp.async.cg.shared.global.L2::cache_hint [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "l"(policy) : "memory");
}
// The same; src_bytes = 0 writes zeros.
__device__ __forceinline__ void cp_async_16_or_zero(uint32_t dst, const void* src, uint32_t src_bytes, uint64_t policy) {
  asm volatile("cp.async.cg.shared.global.L2::cache_hint [%0], [%1], 16, %2, %3;"
               ::"r"(dst), "l"(src), "r"(src_bytes), "l"(policy)
               : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int kPending>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(kPending) : "memory"); }

__device__ __forceinline__ void ldmatrix_x4(uint32_t (&r)[4], uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(addr));
}
__device__ __forceinline__ void ldmatrix_x4_trans(uint32_t (&r)[4], uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(addr));
}

// 8x8 transpose of 16-bit values across a warp (lane 4r + c holds columns 2c, 2c + 1 of row r).
__device__ __forceinline__ uint32_t transpose8x8(uint32_t v) {
  uint32_t r;
  asm("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(r) : "r"(v));
  return r;
}

__device__ __forceinline__ uint4 lds_16B(uint32_t addr) {
  uint4 r;
  asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(r.x), "=r"(r.y), "=r"(r.z), "=r"(r.w) : "r"(addr) : "memory");
  return r;
}

// Two e4m3 values (low 16 bits) -> two fp16 or two bf16 (both exact).
template <typename T>
__device__ __forceinline__ uint32_t e4m3x2_to_16bit(uint32_t pair);
template <>
__device__ __forceinline__ uint32_t e4m3x2_to_16bit<__half>(uint32_t pair) {
  uint32_t h2;
  asm("cvt.rn.f16x2.e4m3x2 %0, %1;" : "=r"(h2) : "h"((unsigned short)pair));
  return h2;
}
template <>
__device__ __forceinline__ uint32_t e4m3x2_to_16bit<__nv_bfloat16>(uint32_t pair) {
  const float2 f = e4m3x2_to_float2(pair);
  return pack2<__nv_bfloat16>(f.x, f.y);
}
// A query row over an 8-bit cache: sixteen bf16 values of each of eight neighbouring lanes -> fp16 values times 2^k, the
// largest in [2^14, 2^15).  Returns what turns its scores into log2 units, scale_log2 2^-k, or 0 where that is no normal
// number or a bit may be lost (exponents more than 31 apart): such a row is for bf16 scores.  (With bf16 queries the rows of
// K have to become bf16, by way of two fp32 values: four instructions per pair instead of one.  us, four heads on each of 8
// K/V heads: 32 requests of 819 rows 16.98 -> 16.38, 17 full contexts of 8190 rows 57.2 -> 52.5.  The values are the same and
// the powers of two cancel: same bits.)
__device__ __forceinline__ float scaled_query(uint4& lo, uint4& hi, float scale_log2) {
  uint32_t w[8] = {lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z, hi.w};
  uint32_t most = 0u, least = 0xffffffffu;              // largest finite, smallest other than 0 (less 1): bits of bf16 values
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const uint32_t a = w[i] & 0x7fffu, b = (w[i] >> 16) & 0x7fffu;
    most = max(most, max(a < 0x7f80u ? a : 0u, b < 0x7f80u ? b : 0u));
    least = min(least, min(a - 1u, b - 1u));
  }
#pragma unroll
  for (int o = 1; o < 8; o <<= 1) most = max(most, __shfl_xor_sync(0xffffffffu, most, o));
  const int up = most == 0u ? 127 : min(268 - (int)(most >> 7), 253);   // biased exponents of 2^k and, below, of 2^-k
  const float scale = __int_as_float(up << 23);
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const float2 f = unpack2<__nv_bfloat16>(w[i]);
    w[i] = pack2<__half>(f.x * scale, f.y * scale);
  }
  lo = make_uint4(w[0], w[1], w[2], w[3]);
  hi = make_uint4(w[4], w[5], w[6], w[7]);
  const float unit = scale_log2 * __int_as_float((254 - up) << 23);
  // (the last bit of a value lies 7 below its exponent, that of fp16 numbers at 2^-24, the largest value at 2^14 or above)
  const bool lost = most != 0u && (int)(most >> 7) - max((int)((least + 1u) >> 7), 1) > 31 ||
                    !(unit >= 1.17549435e-38f && unit <= 3.40282347e38f);
  const uint32_t row_lost = __ballot_sync(0xffffffffu, lost) >> (threadIdx.x & 24) & 0xffu;
  return row_lost ? 0.f : unit;
}

// 8-bit tiles, [16 rows][128 B]: 16-byte chunk `chunk` of a row.  The XOR keeps the eight lanes that a 16-byte
// shared load serves at a time on different banks: K reads take chunks 0-3 (4-7) of two neighbouring rows, V reads
// chunks 2i, 2i + 1 of rows 0, 2, 4, 6 (1, 3, 5, 7).
__device__ __forceinline__ uint32_t tile8_offset_k(int row, int chunk) {
  return (uint32_t)(row * 128 + ((chunk ^ ((row & 1) << 2)) << 4));
}
__device__ __forceinline__ uint32_t tile8_offset_v(int row, int chunk) {
  return (uint32_t)(row * 128 + ((chunk ^ (row & 6)) << 4));
}

// byte offset of 16-byte chunk `chunk` of row `row` inside a swizzled [16][256 B] tile
__device__ __forceinline__ uint32_t tile_offset(int row, int chunk) {
  return (uint32_t)(row * 256 + ((chunk ^ (row & 7)) << 4));
}

// ---- full contexts cut on the device ----
// A full-context launch whose blocks each own a fixed slice of one request lasts as long as its longest slice, and the
// host, which sizes the slices, knows only the longest context the cache can hold.  Here the device cuts the work: the
// rows of all units (request x K/V head, in that order), in pieces of kEvenRows, form one line, block i of the launch
// takes the i-th of equal shares of it, whatever units these belong to, and a unit that one share holds whole is
// finished on the spot; the others leave a partial result per share for decode_merge_even_kernel.  A block has at most
// two of those: slot 2 i for a unit that began in an earlier share, 2 i + 1 for one that begins in its own.  Lengths that
// gain nothing from that are read in the host's slices, by the same kernel (even_by_slices).
// What bounded fixed slices was their last blocks.  Microseconds, fixed slices / as the device decides (equal shares
// alone), caches of 8190 rows: 17 requests, 4 heads on each of 8 K/V heads: 2047..8190 rows 62.8 / 58.3, all 8190 rows
// 85.3 / 86.5 (87.0), 511..585 rows 14.2 / 14.2; 68 requests, 16 heads on each of 2 K/V heads: 77.1 / 65.7, 91.3 / 94.8
// (99.0), 18.1 / 20.8 (22.0).
constexpr int kEvenRows = 64;
constexpr int kEvenMinPieces = 4;                        // no share below 256 rows: block start-up would outweigh it
constexpr int kEvenMaxBatch = 256;                       // requests whose lengths a block scans in shared memory

__device__ __forceinline__ int even_rows(const DecodeParams& p, int n) { return max(0, min(n, p.max_ctx)); }
// a request without rows still has a piece: its output is written as zeros
__device__ __forceinline__ int even_pieces(int rows) { return max(1, (rows + kEvenRows - 1) / kEvenRows); }
__device__ __forceinline__ int even_share(const DecodeParams& p, int total) {
  return max(kEvenMinPieces, (total + p.even_blocks - 1) / p.even_blocks);
}
// Whether the host's slices (p.chunk rows, p.n_chunks per unit, one per block) serve these lengths better: a share that
// ends one unit and begins the next starts up and combines twice, which pays only where the longest slice is longer than
// a share by more than that costs, and over 16-bit rows, where memory bounds the blocks that are left as well, by more
// than a fifth.  Fitted to both cuts measured over 1184 launches: groups of 2..16, 40..148 units, caches of 3000..16000
// rows, lengths alike, ragged and far below the cache; the better cut is missed by 0.5 % on average (16-bit), 0.3 % (8-bit).
__device__ __forceinline__ bool even_by_slices(const DecodeParams& p, int total, int longest) {
  return 5 * min(p.chunk / kEvenRows, longest) <= p.even_factor * even_share(p, total) + 25;
}

// Lengths of the requests and, over all before each, the pieces of one K/V head.
struct EvenLine { int32_t rows[kEvenMaxBatch], before[kEvenMaxBatch + 1], warp_sum[32], warp_most[32]; };

// The lengths -> line.rows, and their sum and maximum in pieces of one K/V head.  Thread t looks after requests
// [t per, (t + 1) per); returns the pieces in front of those.
// kEarly: by the lengths as they stand before grid_dependency_wait().
template <int kThreads, bool kEarly>
__device__ __forceinline__ int sum_even_line(EvenLine& line, const DecodeParams& p, uint32_t& flags, int& total,
                                             int& longest) {
  constexpr int kWarps = kThreads / 32;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int per = (p.B + kThreads - 1) / kThreads, first = tid * per;
  int own = 0, most = 0;
  for (int b = first; b < min(first + per, p.B); ++b) {
    const int n = kEarly ? load_early(p.ctx_lens + b) : load_now(p.ctx_lens + b), rows = even_rows(p, n);
    if (n > p.max_ctx) flags |= SSA_DEV_BAD_COUNT;
    line.rows[b] = rows;
    own += even_pieces(rows);
    most = max(most, even_pieces(rows));
  }
  int sum = own;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int up = __shfl_up_sync(0xffffffffu, sum, o);
    if (lane >= o) sum += up;
  }
  most = __reduce_max_sync(0xffffffffu, most);
  if (lane == 31) { line.warp_sum[warp] = sum; line.warp_most[warp] = most; }
  __syncthreads();
  int at = sum - own;
  total = longest = 0;
#pragma unroll
  for (int w = 0; w < kWarps; ++w) {
    const int s = line.warp_sum[w];
    if (w < warp) at += s;
    total += s;
    longest = max(longest, line.warp_most[w]);
  }
  return at;
}

template <int kThreads>
__device__ __forceinline__ void scan_even_line(EvenLine& line, const DecodeParams& p, int at) {
  const int per = (p.B + kThreads - 1) / kThreads, first = threadIdx.x * per;
  for (int b = first; b < min(first + per, p.B); ++b) {
    line.before[b] = at;
    at += even_pieces(line.rows[b]);
  }
  __syncthreads();
}

// What block chunk_id of the launch begins with: a request, a K/V head, a row, and its pieces [piece, piece_end) (of the line, or
// of the slice).  False if nothing.  kEarly: sum_even_line's.
struct EvenCut { int b, kvh, start, piece, piece_end; };
template <int kThreads, bool kEarly>
__device__ __forceinline__ bool cut_even(EvenLine& line, const DecodeParams& p, int chunk_id, EvenCut& c, uint32_t& flags) {
  const int kv_heads = p.H / p.kv_group;
  int total, longest;
  const int at = sum_even_line<kThreads, kEarly>(line, p, flags, total, longest);
  total *= kv_heads;
  if (even_by_slices(p, total, longest)) {
    const int unit = chunk_id / p.n_chunks, slice = chunk_id - unit * p.n_chunks;
    if (unit >= p.B * kv_heads) return false;
    c.b = unit / kv_heads;
    c.kvh = unit - c.b * kv_heads;
    c.start = slice * p.chunk;
    c.piece = 0;
    c.piece_end = min(p.chunk / kEvenRows, even_pieces(line.rows[c.b]) - c.start / kEvenRows);
    return c.piece_end > 0;
  }
  const int share = even_share(p, total);
  if ((int64_t)chunk_id * share >= total) return false;
  c.piece = chunk_id * share;
  c.piece_end = min(total - c.piece, share) + c.piece;
  scan_even_line<kThreads>(line, p, at);
  c.b = 0;                                               // the last request that begins at or before the share
  for (int step = kEvenMaxBatch / 2; step > 0; step >>= 1)
    if (c.b + step < p.B && line.before[c.b + step] * kv_heads <= c.piece) c.b += step;
  const int in_request = c.piece - line.before[c.b] * kv_heads, of_unit = even_pieces(line.rows[c.b]);
  c.kvh = in_request / of_unit;
  c.start = (in_request - c.kvh * of_unit) * kEvenRows;
  return true;
}

// What the rows of V whose value at `v` is not finite add to it: infinities of their sign, or a NaN.  Called by one thread for
// its dim where the split weights (kSplit) have made a NaN of it; the scores as the kernel has them, the weights whole.
template <typename T, typename Position>
__device__ __forceinline__ float sum_of_infinities(const T* q, const char* k, uint32_t k_row_bytes, const char* v,
                                                uint32_t v_row_bytes, int rows, Position position, float scale_log2, float top) {
  constexpr int kAhead = 8;
  float A = 0.f;
  for (int r0 = 0; r0 < rows; r0 += kAhead) {
    int pos[kAhead];
    float value[kAhead];
#pragma unroll
    for (int i = 0; i < kAhead; ++i) {
      pos[i] = r0 + i < rows ? position(r0 + i) : -1;
      value[i] = pos[i] >= 0 ? to_float(*reinterpret_cast<const T*>(v + (uint64_t)(uint32_t)pos[i] * v_row_bytes)) : 0.f;
    }
#pragma unroll 1
    for (int i = 0; i < kAhead; ++i) {
      if (fabsf(value[i]) <= 3.40282347e38f) continue;
      const T* const row = reinterpret_cast<const T*>(k + (uint64_t)(uint32_t)pos[i] * k_row_bytes);
      float score = 0.f;
      for (int d = 0; d < 128; ++d) score = fmaf(to_float(q[d]), to_float(row[d]), score);
      A = fmaf(fast_exp2(score * scale_log2 - top), value[i], A);
    }
  }
  return A;
}

// kWide serves launches with at most one unit (request x K/V head) per SM and short lists: a whole list is then one
// block's work, no second pass.
// kEven (full contexts): even shares, see above; the grid is (even_blocks * head_splits, 1, 1).
// kSplit: groups of more than kGqaHeads heads; head_splits blocks, side by side, serve heads_per_block of them each.  One
// head per block, which served them before, has fp32 weights and an error of a row against 64 bits of 1.5..2.6e-7; smaller
// groups have 1.4..3.2e-6.  So here tiles are summed on their own, as 8-bit rows have it anyway; bf16 weights enter whole, in
// three terms; fp16 ones in two (2^-23 of a weight; their exponential itself is good to 2^-22) and, far below the largest
// one, as many more as they have bits; and the k-steps of fp16 scores are added outside the tensor cores.  Errors then, over
// N(0, 1) in fp16 / bf16 / 8 bits: 16 x 4096 rows 2.0 / 2.0 / 1.8e-7 (one head per block 2.1 / 2.0 / 2.0e-7), 24 x 2000
// 2.0 / 2.0 / 1.8e-7 (2.0 / 2.0 / 1.9), 24 x 40 1.2 / 1.2 / 1.1e-7 (1.5); only past some 6000 rows per block the running
// sums, each of one team, show: 2.7 / 2.7 / 2.6e-7 over 17 x 8 K/V heads of 8190 rows (2.2e-7).  Time, us: 24 requests, 128
// heads over 4, 2000 rows 48.0 / 50.5 / 52.6; with queries twice and six times as large, whose many small weights take the
// further terms, 57.9 and 79.0 in fp16, 65.7 and 95.6 over 8 bits; one head per block 258 / 253 / 231.
template <typename T, int kMode, bool kHi, bool kWide, bool kEven = false, bool kSplit = false>
__global__ void __launch_bounds__(GqaShape<T, kHi, kWide>::kWarps * 32, kWide ? 1 : 2)
decode_partial_gqa_kernel(const DecodeParams p) {
  using Shape = GqaShape<T, kHi, kWide>;
  constexpr int kWarps = Shape::kWarps, kThreads = kWarps * 32;
  constexpr int kTeam = Shape::kTeam, kTeams = Shape::kTeams;
  constexpr int D = 128;
  constexpr bool kSparse = kMode != kDense;
  constexpr bool kFp8 = kIsFp8<T>;
  using TQ = typename Storage<T>::Query;                // type of the query rows and of a stored output
  using TP = typename std::conditional<kFp8, __half, T>::type;   // type of the weights in the second contraction
  constexpr bool kHalfWeights = std::is_same<TP, __half>::value;
  constexpr float kUp = kFp8 || (kSplit && kHalfWeights) ? 8192.f : 1.f;   // weights (and all they enter) are scaled by this in the loop
  constexpr int kTileBytes = kGqaRows * (kFp8 ? 128 : 256);      // one tensor's tile
  constexpr int kStagedDepth = Shape::kRingBytes / (2 * kTileBytes);
  constexpr int kLiveHeads = 8 * kTeam;
  static_assert(!kEven || (kMode == kDense && !kWide), "even shares are for full contexts");
  static_assert(kThreads % D == 0, "128 threads finish a head");
  static_assert(kMode == kDense || kMode == kIndex || kMode == kSpans,
                "blocked lists take the one-head-per-block kernel");
  static_assert(kLiveHeads * kGqaPitch * 4 <= Shape::kRingBytes, "the combine reuses the ring");

  extern __shared__ __align__(1024) unsigned char s_ring[];
  __shared__ int32_t s_idx[kSparse ? kStagedShortList : 1];
  __shared__ __align__(128) unsigned char s_qtile[kGqaHeads * 256];   // Q of the group, swizzled like a row tile
  __shared__ float s_m[kTeams][kLiveHeads], s_l[kTeams][kLiveHeads];
  __shared__ float s_unit[kFp8 ? kGqaHeads : 1];         // 8-bit rows: of a head's scaled query row (scaled_query)
  __shared__ typename std::conditional<kMode == kSpans, SpanRuns, int>::type s_runs;
  __shared__ typename std::conditional<kMode == kSpans, WarpRuns, int>::type s_wruns[kMode == kSpans ? kWarps : 1];
  __shared__ typename std::conditional<kEven, EvenLine, int>::type s_line;

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int g = lane >> 2, j = lane & 3;
  const int team = warp / kTeam, ht = warp % kTeam;     // ht: the eight heads of the block's that are this warp's
  const int G = p.kv_group;
  // the block serves the part-th heads_per_block heads of the group
  const int chunk_id = kSplit ? blockIdx.x / p.head_splits : blockIdx.x, part = kSplit ? blockIdx.x - chunk_id * p.head_splits : 0;
  const int h0 = kSplit ? part * p.heads_per_block : 0, heads = kSplit ? min(p.heads_per_block, G - h0) : G;

  const unsigned block = blockIdx.x + gridDim.x * (blockIdx.y + gridDim.y * blockIdx.z);
  const bool warp_merge = kMode == kSpans && p.span_cap <= 32;
  int runs = 1;                                        // span_cap rounded up to a power of two
  while (warp_merge && runs < p.span_cap) runs <<= 1;
  EarlySpans guess;                                    // (see decode_partial_kernel)
  guess.there = false;
  if constexpr (kMode == kSpans) {
    if (warp_merge && p.spans_readable > 0 && block < (unsigned)p.guess_blocks) {
      guess = merge_spans_early(s_wruns[warp], p.span_offsets, p.spans, p.spans_readable, p.ctx_lens, p.max_ctx, blockIdx.z, p.span_cap, runs);
      if (!kSplit && guess.there && warp < p.early_warps && block < (unsigned)p.early_blocks)
        prefetch_early<T, D, kSpans, false>(p, blockIdx.z, blockIdx.y, blockIdx.x * p.chunk, warp, &s_wruns[warp], runs, guess.n,
                                            min(guess.total, p.max_selected));
    }
  } else if constexpr (!kEven && !kSplit)
    if (warp < p.early_warps && block < (unsigned)p.early_blocks) {
      if (kMode == kIndex && p.page_table) prefetch_early<T, D, kIndex, true>(p, blockIdx.z, blockIdx.y, blockIdx.x * p.chunk, warp);
      else prefetch_early<T, D, kMode, false>(p, blockIdx.z, blockIdx.y, blockIdx.x * p.chunk, warp);
    }
  if constexpr (!kEven) {
    grid_dependency_wait();
    if (p.early_release) grid_launch_dependents();
  }
  uint32_t flags = 0;
  int kvh = blockIdx.y, b = blockIdx.z, start = chunk_id * p.chunk;
  int piece = 0, piece_end = 0;                        // kEven: what is left of this block's share
  if constexpr (kEven) {
    if (block < (unsigned)p.early_blocks) {
      // (34 requests of 5000 rows, 8 heads on each of 4 K/V heads: 58.2 -> 57.2 us; 15 of 7972, two tokens, 78.4 -> 77.1)
      uint32_t unused = 0;
      EvenCut guessed;                                 // (nothing of it is used behind the wait)
      if (cut_even<kThreads, true>(s_line, p, chunk_id, guessed, unused) && warp < p.early_warps && part == 0)
        prefetch_early<T, D, kDense, false>(p, guessed.b, guessed.kvh, guessed.start, warp);
      __syncthreads();                                 // the lengths are gathered anew
    }
    grid_dependency_wait();
    if (p.early_release) grid_launch_dependents();
    EvenCut c;
    if (!cut_even<kThreads, false>(s_line, p, chunk_id, c, flags)) return;
    b = c.b;
    kvh = c.kvh;
    start = c.start;
    piece = c.piece;
    piece_end = c.piece_end;
  }

  while (true) {                                       // kEven: once per unit of the share; else once
    // One round trip for everything that does not depend on the list length: the first kStagedShortList list
    // entries of the chunk (within the host's bound, so inside the caller's row) and the group's query rows.
    constexpr int kAhead = kStagedShortList / kThreads;
    int32_t ahead[kAhead];
    const bool listed = kMode == kIndex && p.index != nullptr;
    if (listed) {
      const int32_t* row = p.index + (int64_t)b * p.index_stride + start;
#pragma unroll
      for (int jj = 0; jj < kAhead; ++jj) {
        const int i = tid + jj * kThreads;
        ahead[jj] = (i < p.chunk && start + i < p.max_selected) ? __ldg(row + i) : -1;
      }
    }
    uint4 q_lo = make_uint4(0u, 0u, 0u, 0u), q_hi = make_uint4(0u, 0u, 0u, 0u);
    {
      const int row = tid >> 3, c0 = (tid & 7) * 2;     // 16 rows x 8 threads; further threads have no part
      if (row < heads) {
        const TQ* src =
            reinterpret_cast<const TQ*>(p.q) + (int64_t)b * p.q_sb + (int64_t)(kvh * G + h0 + row) * p.q_sh + 8 * c0;
        q_lo = ld_stream_16B(src);
        q_hi = ld_stream_16B(src + 8);
      }
    }
    // span lists: up to 32 spans are merged by every warp for itself, which needs no barrier (one warp for the block, us: 32
    // requests of 819 rows, four heads on each of 8 K/V heads over an 8-bit cache 17.75 -> 16.98, 20 requests of 5199 or 316
    // rows over a 16-bit one 79.4 -> 72.2); a lane asks for "its" span right away
    int span_first = 0, span_n = 0;
    int2 my_span = make_int2(0, 0);
    if constexpr (kMode == kSpans) {
      if (guess.there && lane < guess.S) my_span = load_now(p.spans + guess.first + lane);
      span_first = p.span_offsets ? load_now(p.span_offsets + b) : b * p.span_cap;
      span_n = p.span_offsets ? load_now(p.span_offsets + b + 1) - span_first : p.span_cap;
    }
    // (8-bit rows: in front of the sizes.  32 requests, 32 heads over 8: 15.05 us, 15.33 behind them, 16-bit rows, 17 requests, 12.92
    // and 12.32)
    auto ask_span = [&]() {
      if (warp_merge && !guess.there && lane < min(span_n, p.span_cap)) my_span = load_now(p.spans + span_first + lane);
    };
    if (kMode == kSpans && kFp8) ask_span();
    int n, c;
    if constexpr (kEven) n = c = s_line.rows[b];
    else request_sizes(p, b, n, c, flags);
    if constexpr (kMode == kSpans) {
      if (!kFp8) ask_span();
      int total;
      if (warp_merge && still_the_spans(guess, span_first, span_n, n, my_span)) {
        total = guess.total;
        flags |= guess.flags;
      } else if (warp_merge) {
        if (guess.there && lane < min(span_n, p.span_cap)) my_span = load_now(p.spans + span_first + lane);
        int S = max(span_n, 0);
        if (S > p.span_cap) { S = p.span_cap; flags |= SSA_DEV_TOO_MANY_SPANS; }
        total = merge_spans_warp(s_wruns[warp], my_span, S, runs, n, flags);
      } else {
        total = merge_spans_block<kThreads>(s_runs, p.spans + span_first, span_n, p.span_cap, n);
        if (tid == 0) flags |= s_runs.flags;
      }
      c = min(total, p.max_selected);
      if (total > p.max_selected) flags |= SSA_DEV_OVERFLOW;
      if (chunk_id == 0 && kvh == 0 && part == 0 && tid == 0) {
        if (p.counts_out) p.counts_out[b] = c;
        if (p.ws_counts) p.ws_counts[b] = c;
      }
    }
    if (!kEven && start >= c && chunk_id > 0) return;
    const int most = kEven ? min(piece_end - piece, (c + kEvenRows - 1) / kEvenRows) * kEvenRows : p.chunk;
    const int cnt = max(0, min(most, c - start));

    // position -> what the tile loop uses: -1 for an entry outside the context, the pool row for a paged cache
    auto checked = [&](int v) {
      if (v < 0 || v >= n) {
        flags |= SSA_DEV_BAD_INDEX;
        return -1;
      }
      if (p.page_table) {
        const int page = __ldg(p.page_table + (int64_t)b * p.page_table_stride + (v >> p.page_shift));
        if ((unsigned)page < (unsigned)p.n_pages) return (page << p.page_shift) | (v & p.page_mask);
        flags |= SSA_DEV_BAD_INDEX;
        return -1;
      }
      return v;
    };
    auto stage_window = [&](int w0, int wn) {
      if constexpr (kMode == kSpans) {
        int32_t* out = (kvh == 0 && part == 0 && p.index_out) ? p.index_out + (int64_t)b * p.index_stride + start + w0 : nullptr;
        for (int i = tid; i < wn; i += kThreads) {
          const int v = warp_merge ? span_position(s_wruns[warp], runs, start + w0 + i) : span_position(s_runs, start + w0 + i);
          s_idx[i] = v;
          if (out) out[i] = v;
        }
        return;
      }
      if (listed && w0 == 0) {                             // the entries requested ahead cover any first window
#pragma unroll
        for (int jj = 0; jj < kAhead; ++jj) {
          const int i = tid + jj * kThreads;
          if (i < wn) s_idx[i] = checked(ahead[jj]);
        }
        return;
      }
      const int32_t* row = listed ? p.index + (int64_t)b * p.index_stride + start + w0 : nullptr;
      for (int i = tid; i < wn; i += kThreads)             // no list: the position itself (a paged full context)
        s_idx[i] = checked(row ? __ldg(row + i) : start + w0 + i);
    };
    // the cache row of entry i of the block, -1 if there is none
    auto position = [&](int i) {
      if constexpr (kMode == kSpans)
        return warp_merge ? span_position(s_wruns[warp], runs, start + i) : span_position(s_runs, start + i);
      else if constexpr (kMode == kIndex)
        return checked(listed ? __ldg(p.index + (int64_t)b * p.index_stride + start + i) : start + i);
      else
        return start + i;
    };
    // a list chunk of up to kStagedShortList entries is one window (no meeting in mid-chunk); longer ones go by 512
    const int window = kSparse ? (cnt <= kStagedShortList ? kStagedShortList : kStagedWindow) : Shape::kDenseWindow;
    if (kSparse) stage_window(0, min(cnt, window));
    // the group's query rows -> shared memory (rows of heads that do not exist are zero)
    auto store_q = [&]() {
      if (tid < kGqaHeads * 8) {
        const int row = tid >> 3, c0 = (tid & 7) * 2;
        if constexpr (kFp8) {
          const float unit = scaled_query(q_lo, q_hi, p.scale_log2);
          if (c0 == 0) s_unit[row] = unit;
        }
        *reinterpret_cast<uint4*>(s_qtile + tile_offset(row, c0)) = q_lo;
        *reinterpret_cast<uint4*>(s_qtile + tile_offset(row, c0 + 1)) = q_hi;
      }
    };
    if (kSparse) {
      store_q();
      __syncthreads();                                   // the first window is staged
    }
    uint64_t policy;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(policy));
    const char* kbase = reinterpret_cast<const char*>(
        reinterpret_cast<const T*>(p.k) + (int64_t)b * p.k_sb + (int64_t)kvh * p.k_sh);
    const char* vbase = reinterpret_cast<const char*>(
        reinterpret_cast<const T*>(p.v) + (int64_t)b * p.v_sb + (int64_t)kvh * p.v_sh);
    const uint32_t ring = smem_u32(s_ring) + team * Shape::kRingBytes;
    // this lane's part in copying a tile: its 16 bytes of every row, and where they go in the first row it copies
    constexpr int kRowBytes = kFp8 ? 128 : 256, kChunks = kRowBytes / 16, kRowsPerCopy = 32 / kChunks;
    const char* kcol = kbase + (lane % kChunks) * 16;
    const char* vcol = vbase + (lane % kChunks) * 16;
    const int copy_row = ht * (kGqaRows / kTeam) + lane / kChunks;
    const uint32_t copy_k = kFp8 ? tile8_offset_k(copy_row, lane % kChunks) : tile_offset(copy_row, lane % kChunks);
    const uint32_t copy_v = kFp8 ? tile8_offset_v(copy_row, lane % kChunks) : tile_offset(copy_row, lane % kChunks);
    // this lane's part in reading one: fragment addresses are these, XOR-ed with a multiple of 32 (or 64) bytes
    const uint32_t read_k = kFp8 ? tile8_offset_k(g, j) : tile_offset(lane & 15, lane >> 4);
    const uint32_t read_v = kFp8 ? tile8_offset_v(2 * j, g) : tile_offset((lane >> 4) * 8 + (lane & 7), (lane >> 3) & 1);

    // Running softmax state of heads 8 ht + 2 j + {0, 1}, the same in all lanes of equal j; the sums are per lane until
    // the end.  o[t][e]: head 8 ht + 2 j + (e & 1), dim 16 t + g + 8 (e >> 1) (8-bit rows: 16 g + 2 t + (e >> 1)).
    float m[2] = {neg_inf(), neg_inf()}, l[2] = {0.f, 0.f}, o[8][4];
#pragma unroll
    for (int t = 0; t < 8; ++t) { o[t][0] = 0.f; o[t][1] = 0.f; o[t][2] = 0.f; o[t][3] = 0.f; }
    // B fragments of Q for the eight k-steps: registers for the whole block's life.  8-bit rows: k-step ks of lane
    // (g, j) is dims 64 (ks / 4) + 16 j + 4 (ks % 4) + 0..3 of head g, the order its K pieces come in.
    uint32_t qb[8][2];
    float score_scale[2] = {p.scale_log2, p.scale_log2};   // of heads 8 ht + 2 j + {0, 1}
    bool bf16_scores = false;                              // 8-bit rows: a query row of this warp is not for fp16
    auto load_q = [&]() {
      const uint32_t base = smem_u32(s_qtile);
      if constexpr (kFp8) {
        bf16_scores = __any_sync(0xffffffffu, s_unit[8 * ht + (lane & 7)] == 0.f) != 0;
        if (!bf16_scores) {
#pragma unroll
          for (int e = 0; e < 2; ++e) score_scale[e] = s_unit[8 * ht + 2 * j + e];
        }
        const int head = 8 * ht + g;
        const TQ* const row = reinterpret_cast<const TQ*>(p.q) + (int64_t)b * p.q_sb + (int64_t)(kvh * G + h0 + head) * p.q_sh;
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          const int chunk = 8 * (c >> 1) + 2 * j + (c & 1);
          uint4 w;
          if (!bf16_scores) w = lds_16B(base + tile_offset(head, chunk));
          else w = head < heads ? ld_stream_16B(row + 8 * chunk) : make_uint4(0u, 0u, 0u, 0u);
          qb[2 * c][0] = w.x; qb[2 * c][1] = w.y;
          qb[2 * c + 1][0] = w.z; qb[2 * c + 1][1] = w.w;
        }
      } else {
#pragma unroll
        for (int ks = 0; ks < 8; ks += 2) {
          uint32_t w[4];
          ldmatrix_x4(w, base + tile_offset(8 * ht + (lane & 7), 2 * ks + (lane >> 3)));
          qb[ks][0] = w[0]; qb[ks][1] = w[1];
          qb[ks + 1][0] = w[2]; qb[ks + 1][1] = w[3];
        }
      }
    };
    auto team_sync = [&]() {
      __syncwarp();
      if constexpr (kTeam > 1) asm volatile("bar.sync %0, %1;" ::"r"(1 + team), "n"(kTeam * 32) : "memory");
    };

    for (int w0 = 0; w0 < cnt; w0 += window) {
      const int wn = min(window, cnt - w0);
      if (kSparse && w0 > 0) {
        __syncthreads();                                 // every warp is done with the previous window
        stage_window(w0, wn);
        __syncthreads();
      } else if (w0 > 0) {
        team_sync();                                     // the ring is filled anew: no lane still reads the last tiles
      }
      const int first_row = team * kGqaRows;
      const int nk = wn > first_row ? (wn - first_row + kTeams * kGqaRows - 1) / (kTeams * kGqaRows) : 0;
      // position of row (lane & 15) of this team's k-th tile, -1 if there is none
      auto tile_pos = [&](int k) {
        const int r = first_row + k * (kTeams * kGqaRows) + (lane & 15);
        return r < wn ? (kSparse ? s_idx[r] : start + w0 + r) : -1;
      };
      // Requests tile k of the window (if it exists) into the slot at `slot`; always closes a copy group.  Returns which
      // of its sixteen rows exist.
      auto request = [&](int k, uint32_t slot) -> uint32_t {
        uint32_t live = 0u;
        if (k < nk) {
          const int my_pos = tile_pos(k);
          live = __ballot_sync(0xffffffffu, my_pos >= 0) & 0xffffu;
          const uint32_t dk = slot + copy_k, dv = slot + kTileBytes + copy_v;
          // (the warps of a team copy the rows in turns; from one copy of a lane to its next only XOR-ed bits and a
          // constant change in the address)
          constexpr int kCopies = kGqaRows / kRowsPerCopy / kTeam;
          auto to_k = [&](int i) { return (kFp8 ? dk : dk ^ ((2 * i & 7) << 4)) + i * (kRowsPerCopy * kRowBytes); };
          auto to_v = [&](int i) { return (dv ^ ((kRowsPerCopy * i & 7) << 4)) + i * (kRowsPerCopy * kRowBytes); };
          if (live == 0xffffu) {                         // warp-uniform
#pragma unroll
            for (int i = 0; i < kCopies; ++i) {
              const uint32_t pos = __shfl_sync(0xffffffffu, my_pos, kRowsPerCopy * i + copy_row);
              cp_async_16(to_k(i), kcol + (uint64_t)pos * p.k_row_bytes, policy);
              cp_async_16(to_v(i), vcol + (uint64_t)pos * p.v_row_bytes, policy);
            }
          } else {
            // rows that do not exist are zero.  (Most tiles of a short list are such tiles: rolled, launches of 40..2500
            // rows were 0.7 % slower on average and those of one request up to 9 %.  Where registers are at their limit -
            // two-warp teams, 8-bit rows cut on the device: 3 % - unrolling loses.)
#pragma unroll (kHi || (kFp8 && kEven) ? 1 : kCopies)
            for (int i = 0; i < kCopies; ++i) {
              const int pos = __shfl_sync(0xffffffffu, my_pos, kRowsPerCopy * i + copy_row);
              const uint64_t row = pos >= 0 ? (uint64_t)(uint32_t)pos : 0ull;
              cp_async_16_or_zero(to_k(i), kcol + row * p.k_row_bytes, pos >= 0 ? 16u : 0u, policy);
              cp_async_16_or_zero(to_v(i), vcol + row * p.v_row_bytes, pos >= 0 ? 16u : 0u, policy);
            }
          }
        }
        cp_async_commit();
        return live;
      };
      uint32_t lives[kStagedDepth];                      // rows of tiles k, k + 1, ... (registers: shifted by one per tile)
#pragma unroll
      for (int k = 0; k < kStagedDepth - 1; ++k) lives[k] = request(k, ring + k * (2 * kTileBytes));
      if (w0 == 0) {                                     // (the query is not needed before the first tiles are requested)
        if (!kSparse) {
          store_q();
          __syncthreads();
        }
        load_q();
      }
      constexpr uint32_t kRingBytes = kStagedDepth * 2 * kTileBytes;
      uint32_t kt = ring, refill = ring + kRingBytes - 2 * kTileBytes;   // slots of tile k and of tile k + depth - 1
      auto after = [&](uint32_t slot) { return slot + 2 * kTileBytes == ring + kRingBytes ? ring : slot + 2 * kTileBytes; };
      for (int k = 0; k < nk; ++k, kt = after(kt), refill = after(refill)) {
        team_sync();                                     // the slot about to be refilled has been read by every lane
        lives[kStagedDepth - 1] = request(k + kStagedDepth - 1, refill);
        cp_async_wait<kStagedDepth - 1>();               // tile k has landed (for this lane's copies) ...
        team_sync();                                     // ... and for every other lane's
        const uint32_t live = lives[0];
#pragma unroll
        for (int i = 0; i + 1 < kStagedDepth; ++i) lives[i] = lives[i + 1];
        if (live == 0u) continue;                        // warp-uniform: nothing to add
        const uint32_t ka = kt + read_k, va = kt + kTileBytes + read_v;

        // S^T = K . Q^T: lane (g, j) gets rows g (s[0..1]) and g + 8 (s[2..3]) of heads 2 j and 2 j + 1
        // (two sums of four k-steps each: half the length of the dependent chain)
        float s[4] = {0.f, 0.f, 0.f, 0.f}, s_odd[4] = {0.f, 0.f, 0.f, 0.f};
        if constexpr (kFp8) {
          // (rows of K in bf16 are rare and stay out of the way of the usual loop: rolled for one-warp teams and marked unlikely
          // over full contexts, where registers are tightest: 32 requests of 820 rows, four heads on each of 8 K/V heads, 14.7 us
          // unrolled, 13.1 so; two-warp teams would lose a tenth by it)
          auto scores = [&](auto type) {
            using TS = decltype(type);
#pragma unroll (!kHi && std::is_same<TS, __nv_bfloat16>::value ? 1 : 2)
            for (int half = 0; half < 2; ++half) {
              const uint4 lo = lds_16B(ka ^ (half << 6)), hi = lds_16B((ka ^ (half << 6)) + 8 * kRowBytes);
              const uint32_t a[4] = {lo.x, lo.y, lo.z, lo.w}, c[4] = {hi.x, hi.y, hi.z, hi.w};
#pragma unroll
              for (int i = 0; i < 4; ++i) {
                const uint32_t a0 = e4m3x2_to_16bit<TS>(a[i]), a1 = e4m3x2_to_16bit<TS>(c[i]);
                const uint32_t a2 = e4m3x2_to_16bit<TS>(a[i] >> 16), a3 = e4m3x2_to_16bit<TS>(c[i] >> 16);
                const uint32_t b0 = half == 0 ? qb[i][0] : qb[4 + i][0], b1 = half == 0 ? qb[i][1] : qb[4 + i][1];
                float (&sum)[4] = (i & 1) ? s_odd : s;
                mma_16816<TS>(sum, a0, a1, a2, a3, b0, b1, sum);
              }
            }
          };
          if (kMode == kDense && !kHi ? __builtin_expect(bf16_scores, false) : bf16_scores) scores(__nv_bfloat16());   // warp-uniform
          else scores(__half());
        } else {
#pragma unroll
          for (int ks = 0; ks < 8; ++ks) {
            uint32_t a[4];
            ldmatrix_x4(a, ka ^ (ks << 5));
            float (&sum)[4] = (ks & 1) ? s_odd : s;
            if constexpr (kSplit && kHalfWeights) {
              // (products of fp16 values fill the sum's 24 bits and the tensor cores truncate: k-steps are added here)
              float step[4] = {0.f, 0.f, 0.f, 0.f};
              mma_16816<TQ>(step, a[0], a[1], a[2], a[3], qb[ks][0], qb[ks][1], step);
#pragma unroll
              for (int e = 0; e < 4; ++e) sum[e] += step[e];
            } else {
              mma_16816<TQ>(sum, a[0], a[1], a[2], a[3], qb[ks][0], qb[ks][1], sum);
            }
          }
        }
#pragma unroll
        for (int e = 0; e < 4; ++e) s[e] = (s[e] + s_odd[e]) * score_scale[e & 1];
        if (live != 0xffffu) {                           // warp-uniform; a masked row's score is -inf
          const bool live_lo = (live >> g) & 1u, live_hi = (live >> (g + 8)) & 1u;
#pragma unroll
          for (int e = 0; e < 2; ++e) {
            s[e] = live_lo ? s[e] : neg_inf();
            s[2 + e] = live_hi ? s[2 + e] : neg_inf();
          }
        }
        if (__any_sync(0xffffffffu, fmaxf(s[0], s[2]) > m[0] || fmaxf(s[1], s[3]) > m[1])) {
#pragma unroll
          for (int e = 0; e < 2; ++e) {                  // rare after the first tiles
            float mt = fmaxf(s[e], s[2 + e]);
            mt = fmaxf(mt, __shfl_xor_sync(0xffffffffu, mt, 4));
            mt = fmaxf(mt, __shfl_xor_sync(0xffffffffu, mt, 8));
            mt = fmaxf(mt, __shfl_xor_sync(0xffffffffu, mt, 16));
            const float mn = fmaxf(m[e], mt);
            if (mn > m[e]) {
              const float alpha = fast_exp2(m[e] - mn);
              l[e] *= alpha;
#pragma unroll
              for (int t = 0; t < 8; ++t) { o[t][e] *= alpha; o[t][2 + e] *= alpha; }
              m[e] = mn;
            }
          }
        }
        // weights, split into a 16-bit value and a 16-bit residual (kSplit: bf16 into three terms, with which nothing of them
        // is left), transposed into B fragments of P^T[16 rows, 8 heads]
        uint32_t pa[2], pr[2], pl[2];
        bool small = false;                              // kSplit: a weight whose fp16 terms have less than 23 bits
        // (a maximum of -inf: no finite score yet, every weight is 0)
        const float r0 = m[0] > neg_inf() ? m[0] : 0.f, r1 = m[1] > neg_inf() ? m[1] : 0.f;
#pragma unroll
        for (int half = 0; half < 2; ++half) {
          const float w0 = fast_exp2(s[2 * half] - r0) * kUp, w1 = fast_exp2(s[2 * half + 1] - r1) * kUp;   // -inf gives 0
          l[0] += w0;
          l[1] += w1;
          const uint32_t w = pack2<TP>(w0, w1);
          const float2 back = unpack2<TP>(w);
          pa[half] = transpose8x8(w);
          const uint32_t rest = pack2<TP>(w0 - back.x, w1 - back.y);
          pr[half] = transpose8x8(rest);
          if constexpr (kSplit && !kHalfWeights) {
            const float2 mid = unpack2<TP>(rest);
            pl[half] = transpose8x8(pack2<TP>((w0 - back.x) - mid.x, (w1 - back.y) - mid.y));
          }
          if constexpr (kSplit && kHalfWeights)          // 0 < weight < 1/4 (and not a NaN), by the bits
            small |= __float_as_uint(w0) - 1u < 0x3e7fffffu || __float_as_uint(w1) - 1u < 0x3e7fffffu;
        }
        // fragments of V^T, sixteen dims at a time
        auto for_dims = [&](auto use) {
          if constexpr (kFp8) {
            const uint4 v0 = lds_16B(va), v1 = lds_16B(va + kRowBytes);                          // rows 2 j, 2 j + 1
            const uint4 v2 = lds_16B(va + 8 * kRowBytes), v3 = lds_16B(va + 9 * kRowBytes);      // rows 2 j + 8, 2 j + 9
            const uint32_t x0[4] = {v0.x, v0.y, v0.z, v0.w}, x1[4] = {v1.x, v1.y, v1.z, v1.w};
            const uint32_t x2[4] = {v2.x, v2.y, v2.z, v2.w}, x3[4] = {v3.x, v3.y, v3.z, v3.w};
#pragma unroll
            for (int t = 0; t < 8; ++t) {
              // bytes 2 (t & 1) and 2 (t & 1) + 1 of both rows of a pair, interleaved
              const uint32_t sel = (t & 1) ? 0x7362u : 0x5140u;
              const uint32_t lo = __byte_perm(x0[t >> 1], x1[t >> 1], sel), hi = __byte_perm(x2[t >> 1], x3[t >> 1], sel);
              const uint32_t a[4] = {e4m3x2_to_16bit<__half>(lo), e4m3x2_to_16bit<__half>(lo >> 16),
                                     e4m3x2_to_16bit<__half>(hi), e4m3x2_to_16bit<__half>(hi >> 16)};
              use(t, a);
            }
          } else {
#pragma unroll
            for (int t = 0; t < 8; ++t) {
              uint32_t a[4];                             // dims 16t..+7, 16t+8..+15 of rows 0-7; the same of rows 8-15
              ldmatrix_x4_trans(a, va ^ (t << 5));
              use(t, a);
            }
          }
        };
        if constexpr (kSplit && kHalfWeights) {
          // Weights below 2^-15 of the largest, of which the terms hold less, down to nothing at 2^-38: further terms, the
          // first 2^24 up and each next 2^11, until nothing is left (nine reach the last bit of the smallest normal one).
          if (__any_sync(0xffffffffu, small)) {          // warp-uniform; costs a tile of such rows about half a tile per term
            float left[4];
#pragma unroll
            for (int e = 0; e < 4; e += 2) {
              const float w0 = fast_exp2(s[e] - r0) * kUp, w1 = fast_exp2(s[e + 1] - r1) * kUp;
              const float2 first = unpack2<TP>(pack2<TP>(w0, w1));
              const float2 second = unpack2<TP>(pack2<TP>(w0 - first.x, w1 - first.y));
              left[e] = (w0 - first.x) - second.x;
              left[e + 1] = (w1 - first.y) - second.y;
            }
            float up = 16777216.f, unit = 1.f;
#pragma unroll 1
            for (int term = 0; term < 9; ++term) {
              const bool some = fabsf(left[0]) > 0.f || fabsf(left[1]) > 0.f || fabsf(left[2]) > 0.f || fabsf(left[3]) > 0.f;
              if (!__any_sync(0xffffffffu, some)) break;
              unit /= up;
              uint32_t more[2];
#pragma unroll
              for (int half = 0; half < 2; ++half) {
                const float w0 = left[2 * half] * up, w1 = left[2 * half + 1] * up;
                const uint32_t w = pack2<TP>(w0, w1);
                const float2 back = unpack2<TP>(w);
                more[half] = transpose8x8(w);
                left[2 * half] = w0 - back.x;
                left[2 * half + 1] = w1 - back.y;
              }
              for_dims([&](int t, const uint32_t (&a)[4]) {
                float sum[4] = {0.f, 0.f, 0.f, 0.f};
                mma_16816<TP>(sum, a[0], a[1], a[2], a[3], more[0], more[1], sum);
#pragma unroll
                for (int e = 0; e < 4; ++e) o[t][e] = fmaf(sum[e], unit, o[t][e]);
              });
              up = 2048.f;
            }
          }
        }
        // O^T += V^T . P^T
        for_dims([&](int t, const uint32_t (&a)[4]) {
          if constexpr (kFp8 || kSplit) {
            // (the tile's own sum first, rounded to nearest into the running one: the tensor cores truncate, which over
            // a long list would cost more than the weights' split)
            float sum[4] = {0.f, 0.f, 0.f, 0.f};
            if constexpr (kSplit && !kHalfWeights) mma_16816<TP>(sum, a[0], a[1], a[2], a[3], pl[0], pl[1], sum);
            mma_16816<TP>(sum, a[0], a[1], a[2], a[3], pr[0], pr[1], sum);
            mma_16816<TP>(sum, a[0], a[1], a[2], a[3], pa[0], pa[1], sum);
#pragma unroll
            for (int e = 0; e < 4; ++e) o[t][e] += sum[e];
          } else {
            mma_16816<TP>(o[t], a[0], a[1], a[2], a[3], pa[0], pa[1], o[t]);
            mma_16816<TP>(o[t], a[0], a[1], a[2], a[3], pr[0], pr[1], o[t]);
          }
        });
      }
      cp_async_wait<0>();                                // only empty groups can be pending here
    }
    if (p.dev_status && kvh == 0 && part == 0) {
      const uint32_t f = ((kEven || tid == 0) && chunk_id == 0) ? flags : (flags & SSA_DEV_BAD_INDEX);
      if (f) atomicOr(p.dev_status, f);
    }

    // pieces of this unit that the share ends with or goes on behind
    int unit_pieces = 0, taken = 0;
    if constexpr (kEven) {
      unit_pieces = even_pieces(s_line.rows[b]);
      taken = min(unit_pieces - start / kEvenRows, piece_end - piece);
    }
    if (!p.early_release && (!kEven || piece + taken == piece_end)) grid_launch_dependents();

    // per-warp triples -> shared memory (the ring is free now)
    __syncthreads();
    // [kTeams][kLiveHeads][kGqaPitch]
    float (*s_acc)[kLiveHeads][kGqaPitch] = reinterpret_cast<float (*)[kLiveHeads][kGqaPitch]>(s_ring);
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      const int head = 8 * ht + 2 * j + e;
      float sum = l[e];
      sum += __shfl_xor_sync(0xffffffffu, sum, 4);
      sum += __shfl_xor_sync(0xffffffffu, sum, 8);
      sum += __shfl_xor_sync(0xffffffffu, sum, 16);
      if (g == 0) { s_m[team][head] = m[e]; s_l[team][head] = sum / kUp; }
#pragma unroll
      for (int t = 0; t < 8; ++t) {
        if constexpr (kFp8) {
          *reinterpret_cast<float2*>(&s_acc[team][head][gqa_column(16 * g + 2 * t)]) =
              make_float2(o[t][e] / kUp, o[t][2 + e] / kUp);
        } else {
          s_acc[team][head][gqa_column(16 * t + g)] = o[t][e] / kUp;
          s_acc[team][head][gqa_column(16 * t + g + 8)] = o[t][2 + e] / kUp;
        }
      }
    }
    __syncthreads();
    // Where the result of head i of the block goes when others have to be merged with it.
    auto slot_of = [&](int i) {
      return kEven ? (int64_t)(2 * chunk_id + (start == 0 ? 1 : 0)) * G + h0 + i
                   : ((int64_t)b * p.H + kvh * G + h0 + i) * p.n_chunks + chunk_id;
    };
    const bool whole = kEven ? taken == unit_pieces : p.n_chunks == 1;
    bool infinite = false;                               // kSplit: an infinity in V left a NaN
    {
      // A warp finishes a head, a lane its dims 4 x..4 x + 3: one round of heads where one thread per dim took a round per head
      // and block of 128 threads.  us: 32 requests, 12 heads on each of 8 K/V heads, 100 rows 6.0 -> 5.0, 4 heads, 300 rows 9.0 ->
      // 8.5; 8-bit rows, 8 heads on each of 4, 820 rows 10.7 -> 10.2.
      const int x4 = lane * 4, col4 = gqa_column(x4);
      for (int i = warp; i < heads; i += kWarps) {
        float top[kTeams], M = neg_inf(), L = 0.f;
        float2 lo[kTeams], hi[kTeams];
#pragma unroll
        for (int w = 0; w < kTeams; ++w) {
          top[w] = s_m[w][i];
          lo[w] = *reinterpret_cast<const float2*>(&s_acc[w][i][col4]);
          hi[w] = *reinterpret_cast<const float2*>(&s_acc[w][i][col4 + 2]);
        }
#pragma unroll
        for (int w = 0; w < kTeams; ++w) M = fmaxf(M, top[w]);
        float A[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int w = 0; w < kTeams; ++w) {
          const float wgt = top[w] > neg_inf() ? fast_exp2(top[w] - M) : 0.f;
          L = fmaf(s_l[w][i], wgt, L);
          A[0] = fmaf(lo[w].x, wgt, A[0]);
          A[1] = fmaf(lo[w].y, wgt, A[1]);
          A[2] = fmaf(hi[w].x, wgt, A[2]);
          A[3] = fmaf(hi[w].y, wgt, A[3]);
        }
        if constexpr (kSplit && !kFp8) {
          const float all = (A[0] + A[1]) + (A[2] + A[3]);
          infinite |= all != all && L == L;
        }
        if (whole) {
          store_row_values<TQ>(p, b, kvh * G + h0 + i, x4, M, L, A);
        } else {
          *reinterpret_cast<float4*>(p.ws_acc + slot_of(i) * D + x4) = make_float4(A[0], A[1], A[2], A[3]);
          if (x4 == 0) p.ws_ml[slot_of(i)] = make_float2(M, L);
        }
      }
    }
    if constexpr (kSplit && !kFp8) {
      // The heads again, a thread per dim: a NaN that an infinity has left is put right.  (A pass of its own: what it needs would
      // cost the one above 0.3 us per launch.)
      if (__syncthreads_or(infinite)) {
        const int d = tid % D;
        for (int i = tid / D; i < heads; i += kThreads / D) {
          const int h = kvh * G + h0 + i;
          float M = neg_inf();
#pragma unroll
          for (int w = 0; w < kTeams; ++w) M = fmaxf(M, s_m[w][i]);
          float L = 0.f, A = 0.f;
#pragma unroll
          for (int w = 0; w < kTeams; ++w) {
            const float wgt = (s_m[w][i] > neg_inf()) ? fast_exp2(s_m[w][i] - M) : 0.f;
            L = fmaf(s_l[w][i], wgt, L);
            A = fmaf(s_acc[w][i][gqa_column(d)], wgt, A);
          }
          if (A == A || L != L) continue;
          const TQ* const q_row = reinterpret_cast<const TQ*>(p.q) + (int64_t)b * p.q_sb + (int64_t)h * p.q_sh;
          A = M > neg_inf() ? sum_of_infinities<T>(q_row, kbase, p.k_row_bytes, vbase + d * sizeof(T), p.v_row_bytes, cnt,
                                                   position, p.scale_log2, M)
                            : 0.f;
          if (whole) store_row_value<TQ>(p, b, h, d, M, L, A);
          else p.ws_acc[slot_of(i) * D + d] = A;
        }
      }
    }
    if constexpr (!kEven) break;
    piece += taken;
    if (piece >= piece_end) break;
    start = 0;                                           // the next unit of the line
    if (++kvh == p.H / G) { kvh = 0; ++b; }
    __syncthreads();                                     // ring, query rows and triples are free again
  }
}

// Pass 2 of full contexts cut on the device: the query heads of a unit that more than one block read, kEvenMergeHeads per
// block: one per block works the cut out twice as often, four leave fewer and larger blocks to squeeze in behind the first
// pass (17..68 requests, groups of 4..16: 1 % of the whole call slower on average).  What depends on the lengths alone is
// worked out before the wait: the launch this grid waits for has itself waited for whatever wrote them.  (A note of each
// unit's blocks left by the first pass instead: 0.6 % faster for groups above eight, 1.7 % slower for the others.)
constexpr int kEvenMergeHeads = 2;
template <typename TQ>
__global__ void __launch_bounds__(128 * kEvenMergeHeads)
decode_merge_even_kernel(const DecodeParams p) {
  constexpr int D = 128;
  __shared__ int s_before[4 * kEvenMergeHeads], s_total[4 * kEvenMergeHeads], s_longest[4 * kEvenMergeHeads];
  const int G = p.kv_group, kv_heads = p.H / G, splits = (G + kEvenMergeHeads - 1) / kEvenMergeHeads;
  const int kvh = blockIdx.x / splits, b = blockIdx.y, tid = threadIdx.x, d = tid % D;
  const int i = (blockIdx.x - kvh * splits) * kEvenMergeHeads + tid / D;     // head of the group
  int before = 0, total = 0, longest = 0;
  const int own = even_pieces(even_rows(p, __ldcg(p.ctx_lens + b)));
  for (int k = tid; k < p.B; k += blockDim.x) {
    const int pieces = even_pieces(even_rows(p, __ldcg(p.ctx_lens + k)));
    total += pieces;
    longest = max(longest, pieces);
    if (k < b) before += pieces;
  }
  before = __reduce_add_sync(0xffffffffu, before);
  total = __reduce_add_sync(0xffffffffu, total);
  longest = __reduce_max_sync(0xffffffffu, longest);
  if ((tid & 31) == 0) { s_before[tid >> 5] = before; s_total[tid >> 5] = total; s_longest[tid >> 5] = longest; }
  __syncthreads();
  before = total = longest = 0;
  for (int w = 0; w < (int)blockDim.x / 32; ++w) {
    before += s_before[w];
    total += s_total[w];
    longest = max(longest, s_longest[w]);
  }
  total *= kv_heads;
  int first, last;
  if (even_by_slices(p, total, longest)) {
    first = (b * kv_heads + kvh) * p.n_chunks;
    last = first + (own - 1) / (p.chunk / kEvenRows);
  } else {
    const int share = even_share(p, total), at = before * kv_heads + kvh * own;
    first = at / share;
    last = (at + own - 1) / share;
  }
  grid_dependency_wait();
  grid_launch_dependents();
  if (first == last || i >= G) return;                 // (the block that read it has stored it)
  const int h = kvh * G + i;
  float M = neg_inf(), L = 0.f, A = 0.f;
  for (int k0 = first; k0 <= last; k0 += kMergeAhead) {
    float2 ml[kMergeAhead];
    float row[kMergeAhead];
#pragma unroll
    for (int k = 0; k < kMergeAhead; ++k) {
      const bool there = k0 + k <= last;
      const int64_t slot = (int64_t)(2 * (k0 + k) + (k0 + k == first ? 1 : 0)) * G + i;
      ml[k] = there ? p.ws_ml[slot] : make_float2(neg_inf(), 0.f);
      row[k] = there ? p.ws_acc[slot * D + d] : 0.f;
    }
    float top = M;
#pragma unroll
    for (int k = 0; k < kMergeAhead; ++k) top = fmaxf(top, ml[k].x);
    const float keep = M > neg_inf() ? fast_exp2(M - top) : 0.f;
    L *= keep;
    A *= keep;
    M = top;
#pragma unroll
    for (int k = 0; k < kMergeAhead; ++k) {
      const float w = ml[k].x > neg_inf() ? fast_exp2(ml[k].x - M) : 0.f;
      L = fmaf(ml[k].y, w, L);
      A = fmaf(row[k], w, A);
    }
  }
  store_row_value<TQ>(p, b, h, d, M, L, A);
}

}  // namespace ssa
