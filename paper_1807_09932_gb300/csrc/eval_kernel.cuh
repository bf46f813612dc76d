// Population evaluator: scores every candidate of a population against every row.
//
// What it computes (arXiv 1807.09932, Methods, "Handling missing values"): a row follows a
// candidate (c_1..c_L) when its values satisfy the "greater or equal" relation along the
// candidate's column order; a row with a missing value in one of those columns no longer counts
// when exclusion is on; with the negative-trend option a non-increasing row also follows. The
// output is each candidate's matched-row count and, optionally, its row bitmap.
//
// How (GB300): the rank codes are stored as bit planes (see ebic_internal.h): word (c, p, w) holds
// bit p of column c's code for the 32 rows of bitmap word w. A lane owns one bitmap word of a
// candidate and compares two columns 32 rows at a time, bit-serially from the lowest plane:
//   ge <- majority(b_p, ~a_p, ge)
// one three-input logic operation per plane, after which ge has the bit of every row with
// b >= a. The chain's AND is the bitmap word itself, in its final bit order, so it is stored and
// popcounted as it is. A compare of 32 rows costs NB operations and NB shared-memory words
// (NB = 7 for 64 columns, 8 for 200, 9 for 457).
//   * exclusion by code: a missing value has code 0, below every real rank (1..C). A
//     non-decreasing chain that contains a 0 starts with it, a non-increasing one ends with it,
//     so starting from first >= 1 (the OR of its planes) and, for decreasing trends, ending with
//     last >= 1 removes exactly the rows with a missing value among the candidate's columns;
//   * the walk stops when no row of the warp's words follows any more: a random chain of 8
//     columns matches one row in 40,320, so a candidate of 64 columns ends after about 7.
//
// Row tiles of TS slabs are contiguous in memory and are staged by one bulk copy each
// (cp.async.bulk, completion on an mbarrier; every wait is bounded by the global timer), two
// stages deep. A persistent grid of one CTA per SM divides the work units evenly: a unit is
// 1/1024 of an item (candidate chunk, row tile), so a CTA's first and last item may be a part of
// a chunk's candidates and every CTA gets the same share whatever the number of tiles. The
// chunk's column lists are staged in shared memory; the CTA's warps take candidates from a
// counter, and move on to the next item without waiting for each other: the last warp to leave
// a stage has it refilled.
//
// What bounds it: instruction issue and shared-memory reads (128 bytes per clock and SM), 4 NB / 32
// bytes per row and column walked. One warp covers one candidate over 32 or 64 words where a tile has
// them (eval_wide_tile; up to 104 columns by default); other matrices put several candidates into a
// warp, those of more than 208 columns, whose slabs are 8, 4 or 2 words high, 4 to 16, whose reads
// then meet in banks by chance (2 to 3 wavefronts instead of one).
// Measured, counts and bitmaps of 1,600 candidates, against packed byte and half compares of
// every column (the form before): 436,444 x 64, 2-16 columns 251 -> 142 us; 20,000 x 200, 2-20
// columns, both trends 66 -> 26 us; 50,021 x 457, 2-64 columns 487 -> 76 us.
#pragma once

#include <atomic>

#include "device_common.cuh"
#include "ebic_internal.h"

namespace ebic {

// The comparison b >= a of 32 rows after one more plane, from the lowest plane up.
__device__ __forceinline__ uint32_t ge_step(uint32_t b, uint32_t a, uint32_t ge) {
  return (b & ~a) | (ge & (b | ~a));
}

// Shape of a staged tile as the walk sees it. NB and T are compile-time in the single-population
// evaluator; 0 takes them from the struct (the batch, whose requests differ).
struct TileShape {
  int planes;           // bit planes of a code
  int words;            // words (of 32 rows) per slab: T
  int slabs;            // slabs in the tile: TS
  uint32_t pitch;       // bytes from slab to slab
};

template <int NB, int T>
struct Walk {
  static constexpr int kPlanes = NB ? NB : kMaxPlanes;
  const TileShape sh;
  __device__ __forceinline__ int planes() const { return NB ? NB : sh.planes; }
  __device__ __forceinline__ int words() const { return T ? T : sh.words; }
  __device__ __forceinline__ void load(const uint8_t* base, uint32_t col,
                                       uint32_t (&v)[kPlanes]) const {
    const uint8_t* p0 = base + col * (uint32_t)(planes() * words() * 4);
#pragma unroll
    for (int p = 0; p < kPlanes; ++p)
      v[p] = NB || p < planes() ? *reinterpret_cast<const uint32_t*>(p0 + p * words() * 4) : 0u;
  }
  // rows with y >= x
  __device__ __forceinline__ uint32_t ge(const uint32_t (&y)[kPlanes],
                                         const uint32_t (&x)[kPlanes]) const {
    uint32_t g = y[0] | ~x[0];
#pragma unroll
    for (int p = 1; p < kPlanes; ++p)
      if (NB || p < planes()) g = ge_step(y[p], x[p], g);
    return g;
  }
  static __device__ __forceinline__ uint32_t present(const uint32_t (&v)[kPlanes]) {
    uint32_t o = v[0];
#pragma unroll
    for (int p = 1; p < kPlanes; ++p) o |= v[p];  // (planes past the last are zero)
    return o;
  }

  // The bitmap words of one candidate, the whole warp's, for the lane's WPL words of the tile (word i
  // at base + i * apart; in[i]: it is a row's). Columns two at a time and a last one by itself.
  template <bool NEG, int WPL>
  __device__ __forceinline__ void chain_one(const uint8_t* base, uint32_t apart,
                                            const bool (&in)[WPL], const uint16_t* ccols, int L,
                                            uint32_t (&out)[WPL]) const {
    uint32_t a[WPL][kPlanes], b[WPL][kPlanes], acc[WPL], dec[WPL];
    uint32_t n0 = ccols[0];
#pragma unroll
    for (int i = 0; i < WPL; ++i) load(base + i * apart, n0, a[i]);
    // (the list is read ahead of the columns: past a candidate's end lies the next one or the
    // chunk's slack, and what is read there is never used)
    n0 = ccols[1];
    uint32_t n1 = ccols[2];
    uint32_t any = 0u;
#pragma unroll
    for (int i = 0; i < WPL; ++i) {
      acc[i] = in[i] ? present(a[i]) : 0u;
      dec[i] = NEG && in[i] ? ~0u : 0u;
      any |= acc[i] | dec[i];
    }
    int k = 1;
    while (k + 1 < L && __any_sync(0xFFFFFFFFu, any != 0u)) {
      const uint32_t c0 = n0, c1 = n1;
      n0 = ccols[k + 2];
      n1 = ccols[k + 3];
      any = 0u;
#pragma unroll
      for (int i = 0; i < WPL; ++i) {
        load(base + i * apart, c0, b[i]);
        const uint32_t up = ge(b[i], a[i]), dn = NEG ? ge(a[i], b[i]) : 0u;
        load(base + i * apart, c1, a[i]);
        acc[i] &= up & ge(a[i], b[i]);
        if (NEG) dec[i] &= dn & ge(b[i], a[i]);
        any |= acc[i] | (NEG ? dec[i] : 0u);
      }
      k += 2;
    }
    if (k + 1 == L) {  // (after an early end k + 1 < L: nothing follows any more)
#pragma unroll
      for (int i = 0; i < WPL; ++i) {
        load(base + i * apart, n0, b[i]);
        acc[i] &= ge(b[i], a[i]);
        if (NEG) dec[i] &= ge(a[i], b[i]);
        if (NEG) dec[i] &= present(b[i]);
      }
    } else if (NEG) {
#pragma unroll
      for (int i = 0; i < WPL; ++i) dec[i] &= present(a[i]);
    }
#pragma unroll
    for (int i = 0; i < WPL; ++i) out[i] = NEG ? acc[i] | dec[i] : acc[i];
  }

  // The candidate's bitmap word for the lane's word of the tile (`base`: that word of column 0's
  // plane 0); 0 for a lane without a candidate (L 0, list not read past its first entry). The
  // warp's lanes walk several candidates at once: a lane past its own end compares its last column
  // with itself, and the walk goes on while a lane has rows left and columns to go.
  template <bool NEG>
  __device__ __forceinline__ uint32_t chain(const uint8_t* base, const uint16_t* ccols,
                                            int L) const {
    const int last = L > 0 ? L - 1 : 0;
    uint32_t a[kPlanes], b[kPlanes];
    load(base, ccols[0], a);
    uint32_t acc = L > 0 ? present(a) : 0u, dec = L > 0 ? ~0u : 0u;
    uint32_t n0 = ccols[min(1, last)], n1 = ccols[min(2, last)];
    for (int k = 1; __any_sync(0xFFFFFFFFu, k < L && (NEG ? acc | dec : acc) != 0u); k += 2) {
      load(base, n0, b);
      n0 = ccols[min(k + 2, last)];
      const uint32_t up = ge(b, a), dn = NEG ? ge(a, b) : 0u;
      load(base, n1, a);
      n1 = ccols[min(k + 3, last)];
      acc &= up & ge(a, b);
      if (NEG) dec &= dn & ge(b, a);
    }
    return NEG ? acc | (dec & present(a)) : acc;
  }
};

__device__ __forceinline__ uint32_t lower_bound_u32(const uint32_t* a, uint32_t n, uint64_t v) {
  uint32_t lo = 0, hi = n;
  while (lo < hi) {
    const uint32_t mid = lo + (hi - lo) / 2;
    if ((uint64_t)a[mid] < v) lo = mid + 1; else hi = mid;
  }
  return lo;
}

// eval_tile where the warp has one candidate at a time: slabs of 16 words in tiles of 32 words (WPL 1)
// or 64 (WPL 2: each lane has two words, so that the walk's steps and votes serve 2,048 rows). An odd
// last column is compared by itself, and the list is read without bounds. Counts of 3,000
// candidates of 2-10 columns, calls queued one behind the other, through eval_tile's walk and through
// this one: 100,000 x 20 113 and 74 us, 400,000 x 52 433 and 297, 400,000 x 100 407 and 292 (the packed
// byte compares at their best 91, 344 and 327); 436,444 x 64, 1,600 of 2-16 columns with bitmaps 189
// and 144.
template <int NB, int WPL, bool NEG, class Take>
__device__ __forceinline__ void eval_wide_tile(const TileShape& sh, const uint8_t* stage,
                                               const uint16_t* ccols, const uint16_t* coffs,
                                               uint32_t lo, uint32_t c1, int64_t first_word,
                                               int64_t n_words, uint32_t* counts,
                                               uint32_t* bitmaps, int lane, Take take) {
  const Walk<NB, 16> walk{sh};
  const uint8_t* base = stage + (uint32_t)(lane >> 4) * sh.pitch + (uint32_t)(lane & 15) * 4u;
  bool in[WPL];  // (past the last word the stage may hold another tile's slabs)
#pragma unroll
  for (int i = 0; i < WPL; ++i) in[i] = first_word + lane + 32 * i < n_words;
  for (uint32_t c = take(); c < c1; c = take()) {
    const int o = coffs[c], L = coffs[c + 1] - o;
    uint32_t x[WPL], cnt = 0;
    walk.template chain_one<NEG, WPL>(base, 2u * sh.pitch, in, ccols + o, L, x);
#pragma unroll
    for (int i = 0; i < WPL; ++i) {
      cnt += __popc(x[i]);
      if (bitmaps && in[i])
        bitmaps[(size_t)(lo + c) * (size_t)n_words + first_word + lane + 32 * i] = x[i];
    }
    cnt = __reduce_add_sync(0xFFFFFFFFu, cnt);
    if (lane == 0 && cnt) atomicAdd(&counts[lo + c], cnt);
  }
}

// Candidates [c0, c1) of a staged chunk on one staged tile, those that `take()` hands the warp
// (its first candidate of 32 / SEG, warp-uniform; >= c1 ends). A warp's lanes cover SEG words of
// each of 32 / SEG candidates, SEG = the tile's words up to 32; a taller tile takes several
// passes. first_word: the tile's first bitmap word.
template <int NB, int T, bool NEG, class Take>
__device__ __forceinline__ void eval_tile(const TileShape& sh, const uint8_t* stage,
                                          const uint16_t* ccols, const uint16_t* coffs,
                                          uint32_t lo, uint32_t c1, int64_t first_word,
                                          int64_t n_words, uint32_t* counts, uint32_t* bitmaps,
                                          int lane, Take take) {
  const Walk<NB, T> walk{sh};
  const int t = walk.words();
  const int tile_words = t * sh.slabs;
  const int seg = tile_words < 32 ? tile_words : 32;  // a power of two
  const int li = lane & (seg - 1);
  const uint32_t sub = (uint32_t)lane / (uint32_t)seg;
  for (uint32_t c = take(); c < c1; c = take()) {
    const uint32_t ci = c + sub;
    const bool live = ci < c1;
    const int o = live ? coffs[ci] : 0;
    const int L = live ? coffs[ci + 1] - o : 0;
    uint32_t cnt = 0;
    for (int w0 = 0; w0 < tile_words; w0 += seg) {
      const int w = w0 + li;  // the lane's word of the tile
      const uint8_t* base = stage + (uint32_t)(w / t) * sh.pitch + (uint32_t)(w & (t - 1)) * 4u;
      // (past the last word the stage may hold another tile's slabs)
      const bool in = live && first_word + w < n_words;
      const uint32_t x = walk.template chain<NEG>(base, ccols + o, in ? L : 0);
      cnt += __popc(x);
      if (bitmaps && in)
        bitmaps[(size_t)(lo + ci) * (size_t)n_words + first_word + w] = x;
    }
    if (seg == 32) {
      cnt = __reduce_add_sync(0xFFFFFFFFu, cnt);
    } else {
      for (int d = seg >> 1; d > 0; d >>= 1) cnt += __shfl_xor_sync(0xFFFFFFFFu, cnt, d);
    }
    if (li == 0 && live && cnt) atomicAdd(&counts[lo + ci], cnt);
  }
}

// 32 warps: the walk's registers (two columns' planes and the addresses) fit in 64 per thread, and
// the warps hide each other's shared-memory latency.
constexpr int kEvalThreads = 1024;
constexpr int kEvalWarps = kEvalThreads / 32;
constexpr uint32_t kItemUnits = 1024;  // work units per item

// Shared-memory plan (dynamic): [stage 0][stage 1][chunk columns][chunk offsets]
// WPL 0: tiles whose warps walk several candidates at once (eval_tile).
template <int NB, int T, int WPL, bool NEG>
__global__ void __launch_bounds__(kEvalThreads, 1) eval_population_kernel(const EvalArgs a) {
  extern __shared__ __align__(128) uint8_t smem[];
  __shared__ __align__(8) uint64_t full_bar[2];
  __shared__ uint32_t next_s[2], done_s[2];  // per stage: next candidate, warps that have left
  __shared__ uint32_t chunk_info[3];
  __shared__ uint32_t dead_s;                // a wait expired
  __shared__ uint32_t issued_s;              // items whose copy was issued
  const int tid = threadIdx.x, lane = tid & 31;
  const int64_t n_tiles = (a.slabs + a.ts - 1) / a.ts;
  const TileShape sh{a.planes, a.slab_high, a.ts, a.pitch_bytes};
  uint8_t* const stage0 = smem;
  uint8_t* const stage1 = smem + a.stage_bytes;
  uint16_t* const ccols = reinterpret_cast<uint16_t*>(smem + 2 * (size_t)a.stage_bytes);
  uint16_t* const coffs = ccols + a.chunk_cols + kChunkSlack;

  // one thread: a tile's slabs into stage s (the last tile may have fewer)
  auto issue = [&](int64_t tile, int s) {
    const int64_t q0 = tile * a.ts;
    const int64_t n = a.slabs - q0 < a.ts ? a.slabs - q0 : a.ts;
    const uint32_t bytes = (uint32_t)(n - 1) * a.pitch_bytes + a.slab_bytes;
    dev::mbar_arrive_expect_tx(&full_bar[s], bytes);
    dev::bulk_load(s ? stage1 : stage0,
                   reinterpret_cast<const uint8_t*>(a.ranks) + (size_t)q0 * a.pitch_bytes, bytes,
                   &full_bar[s]);
  };
  if (tid == 0) {
    dev::mbar_init(&full_bar[0], 1);
    dev::mbar_init(&full_bar[1], 1);
    dev::fence_barrier_init();
    next_s[0] = next_s[1] = done_s[0] = done_s[1] = 0u;
    dead_s = 0u;
  }
  // this CTA's units, from the population's column total (an input of the call, complete before
  // the preparation started; of a rejected list only the split is arbitrary, never a tile)
  const uint32_t total = a.cand_offsets[a.n_cand];
  const uint64_t n_chunks = ((uint64_t)total + a.chunk_cols - 1) / a.chunk_cols;
  const uint64_t units = n_chunks * (uint64_t)n_tiles * kItemUnits;  // < 2^26 * 2^26 * 2^10
  const uint64_t per = units / gridDim.x, rem = units % gridDim.x;
  const uint64_t u0 = per * blockIdx.x + (blockIdx.x < rem ? blockIdx.x : rem);
  const uint64_t u1 = u0 + per + (blockIdx.x < rem ? 1u : 0u);
  if (u0 >= u1) {
    // (waits all the same: with a total of 0, in a rejected list, no CTA has work, and the grid must
    // not end before the preparation, whose outputs the next operation in the stream reads)
    dev::pdl_wait();
    return;
  }
  const uint64_t i0 = u0 / kItemUnits, i1 = (u1 + kItemUnits - 1) / kItemUnits;
  __syncthreads();  // the barriers are set up
  if (tid == 0) {  // the first tiles are on their way while the preparation ends
    issue((int64_t)(i0 % n_tiles), 0);
    if (i0 + 1 < i1) issue((int64_t)((i0 + 1) % n_tiles), 1);
    issued_s = i0 + 1 < i1 ? 2u : 1u;
  }
  dev::pdl_wait();  // the preparation (list check, zeroed counts) is complete and visible
  if (*reinterpret_cast<const volatile uint32_t*>(a.err) != 0) {  // invalid input
    if (tid == 0)
      for (uint32_t n = 0; n < issued_s; ++n)
        dev::mbar_wait_bounded(&full_bar[n], 0u, a.timeout_ns);
    return;
  }

  uint64_t cur_chunk = ~0ull;
  uint32_t lo = 0, nc = 0;
  const uint32_t group = 32u / (uint32_t)min(32, sh.words * sh.slabs);  // candidates per warp
  bool dead = false;
  for (uint64_t it = i0; it < i1; ++it) {
    const uint64_t k = it / n_tiles;
    const int64_t tile = (int64_t)(it - k * n_tiles);
    const uint32_t n = (uint32_t)(it - i0);
    const int s = (int)(n & 1u);
    if (k != cur_chunk) {
      // stage the column lists of the candidates whose first column lies in
      // [k*CC, (k+1)*CC): at most CC candidates and CC+63 columns
      __syncthreads();
      if (tid < 2) {
        const uint64_t v = (k + tid) * (uint64_t)a.chunk_cols;
        const uint32_t c = v == 0 ? 0u
                           : v >= total ? a.n_cand
                                        : lower_bound_u32(a.cand_offsets, a.n_cand, v);
        chunk_info[tid] = c;
        if (tid == 0) chunk_info[2] = a.cand_offsets[c];
      }
      __syncthreads();
      lo = chunk_info[0];
      const uint32_t hi = chunk_info[1], c0 = chunk_info[2];
      nc = hi - lo;
      const uint32_t span = a.cand_offsets[hi] - c0;
      for (uint32_t i = tid; i < span; i += kEvalThreads) ccols[i] = a.cand_cols[c0 + i];
      for (uint32_t i = tid; i <= nc; i += kEvalThreads)
        coffs[i] = (uint16_t)(a.cand_offsets[lo + i] - c0);
      __syncthreads();
      cur_chunk = k;
    }
    if (!dead && !dev::mbar_wait_bounded(&full_bar[s], (n >> 1) & 1u, a.timeout_ns)) dead = true;
    dead = __any_sync(0xFFFFFFFFu, dead);
    if (!dead) {
      // this CTA's share of the item's candidates
      const uint32_t s0 = it == i0 ? (uint32_t)(u0 - i0 * kItemUnits) : 0u;
      const uint32_t s1 = it + 1 == i1 ? (uint32_t)(u1 - it * kItemUnits) : kItemUnits;
      const uint32_t c0 = (uint32_t)((uint64_t)nc * s0 / kItemUnits);
      const uint32_t c1 = (uint32_t)((uint64_t)nc * s1 / kItemUnits);
      auto take = [&]() {
        uint32_t u = 0;
        if (lane == 0) u = atomicAdd(&next_s[s], group);
        return c0 + __shfl_sync(0xFFFFFFFFu, u, 0);
      };
      const int64_t first_word = tile * a.ts * sh.words;
      if constexpr (WPL > 0)
        eval_wide_tile<NB, WPL, NEG>(sh, s ? stage1 : stage0, ccols, coffs, lo, c1, first_word,
                                     a.words, a.counts, a.bitmaps, lane, take);
      else
        eval_tile<NB, T, NEG>(sh, s ? stage1 : stage0, ccols, coffs, lo, c1, first_word, a.words,
                              a.counts, a.bitmaps, lane, take);
    }
    // the last warp to leave the stage has it refilled (its release of the counter orders every
    // warp's reads of the stage before the copy)
    __syncwarp();
    if (lane == 0) {
      if (dead) dead_s = 1u;
      if (dev::atom_add_acq_rel(&done_s[s], 1u) == (uint32_t)kEvalWarps - 1u) {
        next_s[s] = 0u;
        done_s[s] = 0u;
        if (it + 2 < i1 && !dead) {
          dev::fence_proxy_async();
          issue((int64_t)((it + 2) % n_tiles), s);
          issued_s = n + 3u;
        }
      }
    }
  }
  __syncthreads();
  if (tid == 0 && dead_s) {
    atomicOr(a.err_out, kErrTimeout);
    atomicOr(a.status, kErrTimeout);
    // wait, again bounded, for the copies that may still be in flight into this CTA's memory
    for (uint32_t d = 0; d < 2 && d < issued_s; ++d) {
      const uint32_t n = issued_s - 1u - d;
      dev::mbar_wait_bounded(&full_bar[n & 1u], (n >> 1) & 1u, a.timeout_ns);
    }
  }
}

}  // namespace ebic
