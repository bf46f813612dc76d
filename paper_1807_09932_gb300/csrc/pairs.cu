// Pair-table evaluation: an exact alternative encoding of the same trend rule, with the archive
// overlaps of the fitness optionally computed in the same pass.
//
// For a loaded matrix, the pair table holds one row bitmap per ordered column pair (a, b):
//   T[a*C + b] = rows where a is not missing and code[b] >= code[a]   (a != b)
//   T[a*C + a] = rows where a is not missing
// It is built once per matrix from the bit planes (pair_build_kernel). Then, for a candidate (c_1..c_L), with the "greater or equal" relation of arXiv
// 1807.09932 (Methods, "Handling missing values"):
//   increasing: AND_i T[c_i*C + c_{i+1}]       (each factor also says c_i is present; c_L is
//               present because code[c_L] >= code[c_{L-1}] >= 1)
//   decreasing: AND_i T[c_{i+1}*C + c_i]       (each factor says c_{i+1} is present and
//               code[c_i] >= code[c_{i+1}]; so c_1 is present too)
//   L = 1:      T[c_1*C + c_1]
// so a candidate costs one 32-bit AND per 32 rows per column, streamed from the table.
//
// Table rows are stored with a stride of ceil(W / 512) * 512 words whose padding words are zero,
// so a lane reads four consecutive words of each 128-word part of an item with one 16-byte load
// and never tests a bound: a padding word ANDs to zero and counts nothing.
//
// Work order: items are (range of 512 words = 16,384 rows, group of 28 or 24 candidates, one per
// warp of a block), taken
// round-robin by a persistent grid in range-major order, so all CTAs work on the same few row
// ranges at a time and the table rows of those ranges stay in L2 while every candidate reads
// them; each table word comes from HBM about once per evaluation. A CTA's items are fixed
// (round-robin), but its warps take the items' candidates in order from a counter of the CTA as
// each warp becomes free, so a warp that drew short candidates takes more of them. The
// preparation kernel has already turned the candidate into its term list (the table-row offsets
// of its consecutive pairs), which the warp loads while it walks its previous candidate. The
// chain goes two pairs per step, each step keeping eight 512-byte warp loads in flight (two
// pairs x four parts; with negative trends one pair, both orders); the next candidate's first
// step is prefetched into L2 before the epilogue (a prefetch holds no registers), and the
// preparation kernel, which builds the term lists while DRAM is otherwise idle, prefetches every
// candidate's first step in the first two ranges, the rows of the pass's first wave. A part stops
// loading once all its words are zero and the walk
// stops when all are: long chains match no row of most ranges. Larger items amortise the
// per-item work (the term list, the reductions and atomics of the epilogue) over more rows.
//
// Fused overlaps (the fitness's o(c, a) = popcount(M_c & M_a), Methods, "Handling missing
// values" and the archive rule of the fitness): the warp that has just built a candidate's words
// of an item ANDs them with the archive members' words of the same rows (archive rows padded to
// the same stride) and adds the popcounts, so candidate bitmaps never go through HBM. Items
// where the candidate matches no row are skipped, and so are archive members that the caller
// does not need (those sharing no column with the candidate cannot penalise it). By the number
// of non-zero words in the item: up to 12 are walked by a lane per member (no reductions); up
// to 32 are compacted to one per lane and members go two per warp reduction; denser items
// take the wanted members two at a time over all words.
#include <type_traits>

#include "pair_chain.cuh"

namespace ebic {
namespace {

using namespace pairdev;

template <bool NEG, bool BITMAPS, bool OVERLAP, int WARPS>
__global__ void __launch_bounds__(WARPS * 32, 1) pair_eval_kernel(const PairArgs p) {
  // per warp: 128 words for the coalesced bitmap store, or its compacted non-zero words
  __shared__ __align__(16) uint32_t stage[WARPS][kRangeWords];
  __shared__ uint32_t next_unit;  // the CTA's next (item, candidate) unit
  if (threadIdx.x == 0) next_unit = 0u;
  dev::pdl_wait();     // the preparation (checks, zeroed outputs) is complete and visible
  dev::pdl_trigger();  // the finalize launch may be scheduled now; it waits for this grid itself
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  // the preparation's verdicts (per block, or the call's error word), requested here and checked
  // once the warp's first term list is requested too: the two loads are in flight together, and
  // no table row is read before the check
  uint32_t f = 0;
  if (p.flags) {
    for (uint32_t i = lane; i < p.n_flags; i += 32) f |= p.flags[i];
  } else if (lane == 0) {
    f = *reinterpret_cast<const volatile uint32_t*>(p.err);
  }
  __syncthreads();  // next_unit is set
  pair_items<NEG, BITMAPS, OVERLAP, kParts, WARPS>(p, stage[warp], &next_unit, [&]() {
    f = __reduce_or_sync(0xFFFFFFFFu, f);
    if (p.flags && blockIdx.x == 0 && threadIdx.x == 0) *p.err_out = f;  // CTA 0 records it
    return f == 0u;  // else invalid input: nothing is evaluated
  });
}

// A generation's scores in one launch after the preparation, for matrices and populations that a
// wave or two of warps covers: a warp per 128-word part of a candidate, all of a candidate's warps
// in one block, which therefore has its whole count and overlaps in shared memory and computes
// its fitness itself. Against the pass above and its finalize launch there are no global
// counters, one launch less, and the chain of a short walk is not cut into steps of two terms:
// a warp keeps eight terms of its one part in flight (four of each direction with negative
// trends), so a chain of up to nine columns waits for memory once. Bound by those round trips:
// list, rows, archive rows.
// A member's own row count is taken along with the overlap, from the same words, and only where
// the candidate has rows at all.
constexpr int kScoreMembers = 4;   // archive members whose words are in flight together
constexpr int kScoreCands = 8;     // most candidates per block

// The overlaps of the warp's words x (words 4 * lane .. of a part) with the wanted archive members, and
// the members' own rows in these words, added to over[] and rows[] (shared). arch: member 0's words
// of the part. SEG lanes per member: bitmaps of at most 32 words fill 8 lanes, and the warp then takes
// 4 members side by side (all overlaps with 64 members, 16,000 candidates on
// 1,000 rows: 63 us, one member at a time 109, the pass and its finalize 71).
template <int SEG>
__device__ __forceinline__ void member_overlaps(uint4 x, const uint32_t* arch, uint64_t stride,
                                                uint64_t members, uint32_t* over, uint32_t* rows,
                                                int lane) {
  constexpr int kSide = 32 / SEG;
  const int li = lane % SEG, side = lane / SEG;
  if constexpr (SEG < 32) {
    x.x = __shfl_sync(0xFFFFFFFFu, x.x, li);
    x.y = __shfl_sync(0xFFFFFFFFu, x.y, li);
    x.z = __shfl_sync(0xFFFFFFFFu, x.z, li);
    x.w = __shfl_sync(0xFFFFFFFFu, x.w, li);
  }
  arch += 4 * li;
  for (uint64_t left = members; left;) {  // warp-uniform
    int m[kScoreMembers];
    uint4 v[kScoreMembers];
#pragma unroll
    for (int k = 0; k < kScoreMembers; ++k) {
      m[k] = -1;
#pragma unroll
      for (int s = 0; s < kSide; ++s) {
        if (left && s == side) m[k] = __ffsll((long long)left) - 1;
        left &= left - 1ull;
      }
      v[k] = m[k] >= 0 ? __ldg(reinterpret_cast<const uint4*>(arch + (uint64_t)m[k] * stride))
                       : make_uint4(0u, 0u, 0u, 0u);
    }
#pragma unroll
    for (int k = 0; k < kScoreMembers; ++k) {
      // both sums are at most 4,096
      uint32_t r = popc4(and4(x, v[k])) | (popc4(v[k]) << 16);
      if constexpr (SEG == 32) {
        r = __reduce_add_sync(0xFFFFFFFFu, r);
      } else {
#pragma unroll
        for (int d = SEG / 2; d > 0; d >>= 1) r += __shfl_xor_sync(0xFFFFFFFFu, r, d);
      }
      if (li == 0 && r) {
        atomicAdd(&over[m[k]], r & 0xFFFFu);
        atomicAdd(&rows[m[k]], r >> 16);
      }
    }
  }
}

template <bool NEG, int SEG>
__global__ void __launch_bounds__(kScoreWarps * 32)
    pair_score_kernel(const PairArgs p, const ScoreArgs f, int parts) {
  __shared__ uint32_t count_s[kScoreCands];
  __shared__ uint32_t over_s[kScoreCands][kPairMaxArch];  // overlap with each member
  __shared__ uint32_t rows_s[kScoreCands][kPairMaxArch];  // the member's own rows
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int team = warp / parts, part = warp - team * parts;
  const uint32_t cand = blockIdx.x * (blockDim.x / (32u * parts)) + team;
  const bool live = cand < p.n_cand;
  for (int i = threadIdx.x; i < kScoreCands * kPairMaxArch; i += blockDim.x) {
    (&over_s[0][0])[i] = 0u;
    (&rows_s[0][0])[i] = 0u;
  }
  if (threadIdx.x < kScoreCands) count_s[threadIdx.x] = 0u;
  // (inputs of the call, complete before the preparation started)
  const uint32_t L = live ? f.offsets[cand + 1] - f.offsets[cand] : 1u;
  dev::pdl_wait();  // the preparation is complete and visible
  uint32_t bad = 0;
  for (uint32_t i = lane; i < p.n_flags; i += 32) bad |= p.flags[i];
  Terms t;
  uint64_t members = 0;
  if (live) {
    load_terms<NEG>(p, cand, lane, t);
    if (p.n_arch)
      members = p.score ? p.score[cand] : p.n_arch >= 64 ? ~0ull : (1ull << p.n_arch) - 1ull;
  }
  bad = __reduce_or_sync(0xFFFFFFFFu, bad);
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    *p.err_out = bad;
    if (f.err_mirror) *f.err_mirror = bad;
  }
  if (bad) return;  // the whole grid: invalid input, nothing is evaluated
  __syncthreads();  // the shared sums are zero
  const uint32_t word = (uint32_t)part * kRangeWords + 4u * lane;
  uint4 x[1] = {make_uint4(0u, 0u, 0u, 0u)};
  if (live) {
    const uint32_t ones = (uint32_t)((uint64_t)p.C * p.C * p.stride);
    const bool any = pair_chain<NEG, 1>(t, p.table, word, ones, lane, x);
    if (any) {
      const uint32_t c = __reduce_add_sync(0xFFFFFFFFu, popc4(x[0]));
      if (lane == 0) atomicAdd(&count_s[team], c);
    }
    if (p.bitmaps) {
      uint32_t* out = p.bitmaps + (uint64_t)cand * (uint64_t)p.bitmap_stride + word;
      const uint32_t v[4] = {x[0].x, x[0].y, x[0].z, x[0].w};
#pragma unroll
      for (int j = 0; j < 4; ++j)
        if (word + j < (uint64_t)p.W) out[j] = v[j];
    }
  }
  __syncthreads();
  const uint32_t n = count_s[team];
  if (n) {
    const uint32_t* arch = p.arch + part * kRangeWords;
    member_overlaps<SEG>(x[0], arch, p.stride, members, over_s[team], rows_s[team], lane);
  }
  __syncthreads();
  if (part != 0 || !live) return;
  // q(a) >= q(c) of the members sharing a column decides which overlaps count
  const uint32_t shift = (L < 33u ? L : 33u) - 1u;
  const uint64_t qc = (uint64_t)n << shift;
  const uint64_t share = p.n_arch ? f.share[cand] : 0ull;
  uint32_t best = 0;
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const uint32_t a = lane + 32u * h;
    if (a >= p.n_arch) continue;
    const uint32_t o = over_s[team][a];
    const uint32_t al = f.arch_offsets[a + 1] - f.arch_offsets[a];
    const uint64_t qa = (uint64_t)rows_s[team][a] << ((al < 33u ? al : 33u) - 1u);
    if (((share >> a) & 1ull) && qa >= qc && o > best) best = o;
    if (o) p.overlaps[(uint64_t)cand * p.ov_stride + a] = o;  // (zeroed by the preparation)
  }
  best = __reduce_max_sync(0xFFFFFFFFu, best);
  if (lane == 0) {
    p.counts[cand] = n;
    if (f.counts_mirror) f.counts_mirror[cand] = n;
    f.fitness[cand] = (uint64_t)(n - best) << shift;
  }
}

// The pair table from the bit planes: a lane has two neighbouring bitmap words, a warp kBuildA
// columns a, whose planes it keeps in registers; columns b pass through shared memory, kBuildB at
// a time and two buffers deep (cp.async), and each serves all of the block's columns a. A table
// word is the comparison b >= a over the planes (one operation each, as ge_step) AND the rows where
// a is present; for b = a that leaves "a present". Rows past the matrix read as code 0, so the
// padding words come out zero, and every word of the table is written by one store, 256 bytes a
// warp.
// Bound by those stores (C * C rows of the padded width) with the logic pipe close behind (NB
// operations per word: for NB = 9, 5 cycles of an SM per 128 bytes, 6 of its share of HBM), so
// everything else per word is kept small: two words per lane halve the address arithmetic, four
// columns a per warp the shared reads. Measured (library events, which add some 5 us): 50,021 x 457
// (1.7 GB) 450 us, 436,444 x 64 (226 MB) 70 us, 20,000 x 200 51 us; without FOLD 485, 76 and 58;
// one word per lane and eight columns a 566 and 76; run through the evaluator as a population of
// all pairs (with the table zeroed first) 3,670 and 355.
constexpr int kBuildWarps = 8;
constexpr int kBuildA = 4;                         // columns a per warp
constexpr int kBuildB = 16;                        // columns b per buffer
constexpr int kBuildCols = kBuildWarps * kBuildA;  // columns a per block
constexpr int kBuildWords = 64;                    // words of a block's range

// FOLD (columns < 2^NB - 1, so that no code has every bit set): a row where a is missing is given
// the code with every bit set in a, which no b reaches, instead of a mask at the end: one operation
// of NB + 1 less.
template <int NB, bool FOLD>
__global__ void __launch_bounds__(kBuildWarps * 32, 2)
    pair_build_kernel(const uint32_t* __restrict__ ranks, int C, int T, uint32_t pitch_words,
                      int64_t slabs, int64_t word0, uint32_t* __restrict__ table, uint32_t stride,
                      uint32_t groups_a, uint32_t groups_b, int b_per_block) {
  extern __shared__ __align__(16) uint2 bs[];  // [2][kBuildB][NB][32]
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  // block = (range of words, group of columns a, group of columns b), the last fastest
  const uint32_t gb = blockIdx.x % groups_b, rest = blockIdx.x / groups_b;
  const int a0 = (int)(rest % groups_a) * kBuildCols + warp * kBuildA;
  const int b0 = (int)gb * b_per_block, b1 = min(C, b0 + b_per_block);
  const uint32_t word = rest / groups_a * (uint32_t)kBuildWords + 2u * lane;
  // (slabs are 2, 4, 8 or 16 words high: both of the lane's words lie in one)
  const int64_t q = (word0 + word) / T;
  const bool in = q < slabs;
  const uint32_t* const src = ranks + (in ? (size_t)q * pitch_words + (word0 + word) % T : 0);
  // columns b of one buffer; past the matrix (rows or columns) zeros are written instead
  auto stage = [&](int b, int buf) {
    for (int i = warp; i < kBuildB * NB; i += kBuildWarps) {
      const int c = b + i / NB, p = i % NB;
      uint2* dst = bs + (buf * kBuildB * NB + i) * 32 + lane;
      const bool ok = in && c < b1;
      const uint32_t* g = ok ? src + ((size_t)c * NB + p) * T : src;
      asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(dev::smem_addr(dst)),
                   "l"(__cvta_generic_to_global(g)), "r"(ok ? 8 : 0)
                   : "memory");
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  stage(b0, 0);
  if (blockIdx.x == 0 && threadIdx.x < kOnesWords)  // the all-ones row after the table
    table[(uint64_t)C * C * stride + threadIdx.x] = ~0u;
  uint2 na[kBuildA][NB], here[kBuildA];  // columns a: planes inverted, rows present
#pragma unroll
  for (int k = 0; k < kBuildA; ++k) {
    here[k] = make_uint2(0u, 0u);
#pragma unroll
    for (int p = 0; p < NB; ++p) {
      uint2 v = make_uint2(0u, 0u);
      if (in && a0 + k < C)
        v = __ldg(reinterpret_cast<const uint2*>(src + ((size_t)(a0 + k) * NB + p) * T));
      na[k][p] = make_uint2(~v.x, ~v.y);
      here[k].x |= v.x;
      here[k].y |= v.y;
    }
    if (FOLD)
#pragma unroll
      for (int p = 0; p < NB; ++p) {
        na[k][p].x &= here[k].x;
        na[k][p].y &= here[k].y;
      }
  }
  uint32_t* out = table + ((uint64_t)a0 * C + b0) * stride + word;
  const uint64_t next_a = (uint64_t)C * stride;
  int buf = 0;
  for (int b = b0; b < b1; b += kBuildB, buf ^= 1) {
    stage(b + kBuildB, buf ^ 1);  // (past the last column: zeros, never used)
    asm volatile("cp.async.wait_group 1;" ::: "memory");
    __syncthreads();
    const uint2* row = bs + buf * kBuildB * NB * 32 + lane;
    const int n = min(kBuildB, b1 - b);
    for (int j = 0; j < n; ++j, out += stride, row += NB * 32) {
      uint2 v[NB];
#pragma unroll
      for (int p = 0; p < NB; ++p) v[p] = row[p * 32];
#pragma unroll
      for (int k = 0; k < kBuildA; ++k) {
        uint2 g = make_uint2(v[0].x | na[k][0].x, v[0].y | na[k][0].y);
#pragma unroll
        for (int p = 1; p < NB; ++p) {
          g.x = (v[p].x & na[k][p].x) | (g.x & (v[p].x | na[k][p].x));
          g.y = (v[p].y & na[k][p].y) | (g.y & (v[p].y | na[k][p].y));
        }
        if (!FOLD) {
          g.x &= here[k].x;
          g.y &= here[k].y;
        }
        if (a0 + k < C) *reinterpret_cast<uint2*>(out + k * next_a) = g;
      }
    }
    __syncthreads();  // the buffer is refilled in the next round
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
}

template <bool NEG, bool BITMAPS, int WARPS>
cudaError_t launch_variant(const PairArgs& p, int grid, bool pdl, cudaStream_t s) {
  if (p.arch)
    return launch_maybe_pdl(pdl, pair_eval_kernel<NEG, BITMAPS, true, WARPS>, dim3(grid),
                            dim3(WARPS * 32), 0, s, p);
  if constexpr (BITMAPS && WARPS != kPairWarps)
    return cudaErrorInvalidValue;  // (launch_pair_eval takes kPairWarps)
  else
    return launch_maybe_pdl(pdl, pair_eval_kernel<NEG, BITMAPS, false, WARPS>, dim3(grid),
                            dim3(WARPS * 32), 0, s, p);
}

}  // namespace

cudaError_t launch_pair_eval(const PairArgs& p, bool negative, int grid, bool pdl,
                             cudaStream_t s) {
  if (p.n_cand == 0) return cudaSuccess;
  if (p.arch && p.n_arch > (uint32_t)kPairMaxArch) return cudaErrorInvalidValue;
  if (p.stride % kItemWords != 0 || (int64_t)p.stride < p.W) return cudaErrorInvalidValue;
  if ((uint64_t)p.C * (uint64_t)p.C * p.stride > 0xFFFFFFFFull) return cudaErrorInvalidValue;
  if (p.arch && (p.ov_stride % 2 != 0 || p.ov_stride < p.n_arch)) return cudaErrorInvalidValue;
  count_launch();
  const bool bm = p.bitmaps != nullptr;
  // 28 warps where 72 registers suffice (increasing trends: 4 % off 65,535 candidates, 1 % off
  // 1,600 on 436,444 x 64 against 24; 20 and 32 warps were slower; both trends need 80), and where
  // the fullest SM then has fewer items to go through. With as many items, or none to spare, the
  // items of 28 candidates only take longer: calls with 24 and 28 warps, 20,000 rows, 1,600 candidates
  // 13.0 and 13.7 us, 30,000 rows 13.1 and 13.9, 12,000 rows, 6,000 candidates 17.2 and 18.3. Without an
  // archive the writing of bitmaps takes longer with 28: 436,444 x 64, 1,600 of 2-6 columns 46.0 and
  // 47.9.
  auto rounds = [&](uint32_t warps) {
    const uint64_t items = (uint64_t)((p.W + kItemWords - 1) / kItemWords) *
                           ((p.n_cand + (uint64_t)warps - 1) / warps);
    return (items + grid - 1) / grid;
  };
  const bool wide = !negative && (p.arch || !bm) && rounds(28) < rounds(kPairWarps);
  if (negative)
    return bm ? launch_variant<true, true, kPairWarps>(p, grid, pdl, s)
              : launch_variant<true, false, kPairWarps>(p, grid, pdl, s);
  if (wide)
    return bm ? launch_variant<false, true, 28>(p, grid, pdl, s)
              : launch_variant<false, false, 28>(p, grid, pdl, s);
  return bm ? launch_variant<false, true, kPairWarps>(p, grid, pdl, s)
            : launch_variant<false, false, kPairWarps>(p, grid, pdl, s);
}

// Where the pass's items of four parts are mostly empty and its finalize launch costs more than the
// work, up to some waves of warps; beyond, its order, which keeps a range's rows in L1 and L2 for
// all candidates, counts for more. The members make the line: a warp here goes over every member
// whose overlap is wanted, the pass drops most of a sparse candidate's work before it gets to them.
// Wanted are all (`all`: the caller reads every overlap) or those that share a column, 18 / cols of
// them taken as typical. Measured, calls queued one behind the other, the pass's time over this
// kernel's at its side of the line and past it:
//   one part: 1.06-1.66 throughout for 33 to 128 words; up to 32 words with 64 members wanted 1.02 at
//     6,000 candidates, 0.95 at 10,000;
//   two parts: without members 1.18 at 12,000 warps, 1.04 at 20,000; 20 wanted 1.24 at 3,200, 1.00 at
//     12,000, 0.92 at 20,000; 64 wanted 1.19 at 3,200, 0.87 at 6,000;
//   three to eight parts: without members 1.12 at 9,000 warps, 0.97 at 12,000; 20 wanted 1.08 at 4,800,
//     0.99 at 5,600, 0.92 at 8,000, 0.75 at 12,800; 64 wanted 1.23 at 3,200, 1.05 at 4,000, 0.94 at
//     4,800, 0.58 at 12,800.
// One trend over more than two parts stays with the pass.
static int64_t wanted_members(uint32_t n_arch, bool all, int32_t cols) {
  return all || cols <= 18 ? n_arch : (int64_t)n_arch * 18 / cols;
}

bool pair_score_fits(int64_t W, uint32_t n_cand, bool negative, uint32_t n_arch, bool all,
                     int32_t cols) {
  const int64_t parts = (W + kRangeWords - 1) / kRangeWords, warps = (int64_t)n_cand * parts;
  const int64_t wanted = wanted_members(n_arch, all, cols);
  if (parts == 1) return warps <= (W <= 32 && wanted > 32 ? 8000 : 32000);
  if (parts > (negative ? kScoreWarps : 2)) return false;
  return warps <= 3200 + (parts == 2 ? 153600 : 75600) / (12 + wanted);
}

cudaError_t launch_pair_score(const PairArgs& p, const ScoreArgs& f, bool negative, bool pdl,
                              cudaStream_t s) {
  const int parts = (int)((p.W + kRangeWords - 1) / kRangeWords);
  // several candidates per block while their warps are few
  const int cands = parts >= kScoreCands ? 1 : kScoreCands / parts;
  const unsigned blocks = (unsigned)(((uint64_t)p.n_cand + cands - 1) / cands);
  // (a few members are in flight together anyway)
  const bool side = p.W <= 32 && wanted_members(p.n_arch, !p.score, p.C) > 2 * kScoreMembers;
  auto kern = negative ? (side ? pair_score_kernel<true, 8> : pair_score_kernel<true, 32>)
                       : (side ? pair_score_kernel<false, 8> : pair_score_kernel<false, 32>);
  count_launch();
  return launch_maybe_pdl(pdl, kern, dim3(blocks), dim3(32 * parts * cands), 0, s, p, f, parts);
}

cudaError_t launch_pair_build(const Layout& L, const uint32_t* ranks, uint32_t* table,
                              uint32_t stride, int64_t word0, int num_sms, cudaStream_t s) {
  const uint32_t ga = (L.cols + kBuildCols - 1) / kBuildCols;
  const uint64_t outer = (uint64_t)(stride / kBuildWords) * ga;
  // all columns b in one block where that fills the GPU several times over, else fewer
  int per = (L.cols + kBuildB - 1) / kBuildB * kBuildB;
  while (per > kBuildB && outer * ((L.cols + per - 1) / per) < 6ull * num_sms)
    per = (per / 2 + kBuildB - 1) / kBuildB * kBuildB;
  const uint32_t gb = (L.cols + per - 1) / per;
  const uint64_t blocks = outer * gb;
  if (blocks > 0x7FFFFFFFull) return cudaErrorInvalidConfiguration;
  auto go = [&](auto nb) {
    const size_t smem = (size_t)2 * kBuildB * nb() * 32 * sizeof(uint2);
    auto kern = L.cols < (1 << nb()) - 1 ? pair_build_kernel<nb(), true>
                                         : pair_build_kernel<nb(), false>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)smem);
    if (e != cudaSuccess) return e;
    count_launch();
    kern<<<(unsigned)blocks, kBuildWarps * 32, smem, s>>>(
        ranks, L.cols, L.slab_high, L.pitch_bytes / 4, L.slabs, word0, table, stride, ga, gb, per);
    return cudaGetLastError();
  };
  switch (L.planes) {
    case 1: return go(std::integral_constant<int, 1>());
    case 2: return go(std::integral_constant<int, 2>());
    case 3: return go(std::integral_constant<int, 3>());
    case 4: return go(std::integral_constant<int, 4>());
    case 5: return go(std::integral_constant<int, 5>());
    case 6: return go(std::integral_constant<int, 6>());
    case 7: return go(std::integral_constant<int, 7>());
    case 8: return go(std::integral_constant<int, 8>());
    case 9: return go(std::integral_constant<int, 9>());
    case 10: return go(std::integral_constant<int, 10>());
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace ebic
