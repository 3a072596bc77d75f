// Quantised fast path of the fused select kernel for tree ensembles (Model A).
//
// Repack (host, at model-create time)
//   A split "x[f] < thr" only needs to know how many of feature f's distinct thresholds are
//   <= x. With the thresholds of f sorted, bin(x) = #{j : thr_j <= x}, and
//   x < thr_j  <=>  bin(x) <= j  exactly. A feature's thresholds are cut into slices of 127; a
//   "row" is one slice, a pair's byte in that row the number of the slice's thresholds that are
//   <= x (0..127), and a node one 32-bit word (row offset, index within the slice). A feature
//   with thousands of distinct thresholds (an ensemble trained by exact greedy splitting) simply
//   owns more rows; the tile geometry follows the row count (see FastGeom). Trees are padded to
//   complete trees of the ensemble's depth D and stored in chunks, each chunk laid out level by
//   level ([level][tree][node]) followed by its leaves, so that a chunk is one contiguous block
//   a CTA copies into shared memory with one bulk async copy. The nodes of the top levels are
//   also kept as (row offset, replicated threshold) pairs that travel as a kernel parameter,
//   i.e. through the constant bank.
//   A partition split on a categorical field ("level in S goes right") joins the same scheme
//   through rank rows: a row whose byte is the rank of the pair's level in a fixed ordering of
//   the field's levels, chosen so that S or its complement is the set of ranks >= c; the node
//   then is the ordinary "bin <= c - 1 goes left", with its children exchanged for a complement.
//
// Hoisting
//   Rows are grouped by what their feature depends on. Candidate-only rows (given the
//   problem's element types) are quantised once per call by cand_rows_kernel into a table
//   indexed by (type combination, candidate); problem-only rows once per CTA; only the
//   per-pair rows are computed and searched for every pair - or, in a batch of problems, once
//   per (problem, class of candidates that look alike to the per-pair columns) and copied
//   (see MemoView).
//
// Other entries into the same walk
//   few candidate blocks (a single problem, a short list): the machine's CTAs share out the trees of all
//   blocks evenly (split walk); scoring call (ks_score): tiles are quantised
//   from given feature rows by tile_rows_kernel and the scores are stored instead of ranked.
//
// Kernel (an item = one problem x up to NC candidates; a CTA of THREADS threads serves one item,
// or - batch form of the geometries with one CTA per SM - a run of items: one candidate block
// for problem after problem, whose candidate-only rows it keeps in the tile)
//   phase A  fill the [row][candidate] byte tile. A 32-bit word of a row holds the four
//            candidates that share a lane slot, so a warp's byte loads of any mix of rows
//            touch 32 distinct banks and one word load serves four candidates;
//   phase B  stream the ensemble through rings of two shared-memory buffers (cp.async.bulk +
//            mbarrier, bounded waits). Thread (w, g) owns the four candidates of word w and
//            walks group g's share of the trees: the chunks of its ring (see ring_count), and of
//            those the trees that fall to it when two groups share a ring. The top levels are evaluated for all four
//            candidates at once, node by node, with byte-parallel arithmetic on whole words;
//            below that each candidate follows its own path: a' = 2 a + k0 (+ 4 to go right), a
//            multiply-add plus a predicated add;
//   phase C  add the groups' partial scores, rank the block's keys, write a partial top-k list.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <climits>
#include <cstring>
#include <limits>
#include <new>
#include <vector>

#include "ks_features.cuh"
#include "ks_gbdt_quant.cuh"
#include "ks_internal.h"
#include "ks_memo.cuh"
#include "ks_topk.cuh"

namespace ks {

namespace {

constexpr int kBufBytes = 16 * 1024;   // one tree-chunk buffer (twice that where the shared memory allows)
constexpr int kCombos = 16;            // dtype_ab x dtype_d

constexpr int kSmCount = 148;           // SMs of the one device this library is built for (sm_100a)
// Chunk rings of a CTA with G tree groups: every ring has kNBuf buffers and serves G / rings groups,
// which share out the trees of its chunks; ring r takes the chunks r, r + rings, ... A ring of
// its own per group means that only the group's warps meet at a buffer's release, for the same
// shared memory and the same trees per thread and chunk (config 1, two groups: 55.3 -> 54.4 ms);
// four groups do best with two rings (config 2: 132.4 ms with four rings, 131.6 with one, 129.3 with two).
__host__ __device__ constexpr int ring_count(int groups) { return groups <= 2 ? groups : 2; }
constexpr int kNBuf = 2;                // buffers of a ring (four of 8 KB and three of 12 KB measured slower)
// shared memory map (byte offsets from the dynamic shared base): the rings' chunk buffers, then the tile
constexpr int kOffBuf0 = 0;

// Split walk: where there are too few candidate blocks for whole rounds of the machine's CTAs, the blocks'
// trees lie on one line, block after block, and every CTA takes an equal stretch of it. A stretch's ends fall
// inside blocks: such a part's sums go to memory, and the last CTA to arrive at a block (atomic counter,
// nobody waits) adds its parts in order and ranks it. In a single-problem call the last block overall
// merges the lists and writes the final result. Where a block is cut depends on where it lies, a
// candidate's score must not (equal candidates tie, whatever their places): a chunk's trees are added up in
// floats, in a fixed order, and the chunks' sums as doubles that are multiples of one power of two (`grid`, see
// sum_grid), so that every sum of them is exact, in any order. An ensemble whose leaves spread too far for that has
// no grid: all blocks are cut alike then.
//
// The line is measured in trees, a block's beginning with `fill` trees' worth for its tile; a CTA that starts
// inside a block fills its tile too, but that holds for nearly all of them. Trees are dealt in units of
// one chunk a ring. CTA c begins at the unit that holds point c * total / gridDim.x.
struct SplitArgs {
  int units;            // of a block; 0: CTAs take whole blocks
  int unit, fill;       // trees of a unit, and what filling a tile counts for
  int blocks;
  int step, rest;       // total / CTAs, and the remainder
  double grid;          // added and subtracted, it rounds a chunk's sum to a multiple of its lowest bit; or 0
  double* scores;       // [CTAs][2][NC]: sums of a CTA's first and last part
  int* words;           // the context's device words: arrival counters, by the first CTA of a block (reset by their last users), kWordWalk
  int32_t* out_idx;     // single-problem form only: [k] final result (device-visible, may be
  float* out_score;     // mapped host memory); null when a merge kernel follows
  const uint8_t* tiles; // tiles built in front: [blocks][rows][NC] (tile_rows_kernel), or the per-pair rows alone (tile_pairs_kernel)
  const uint8_t* cand_tiles;  // the candidate-only rows of the latter, or null
  int* out_seq;         // single-problem form: receives `seq` once the k results are written
  int seq;
  float* score_out;     // scoring call (ks_score): the scores of the block's rows go here, no ranking
  int repeat;           // floor measurement only: passes over the resident chunks
};
// (32 bits hold a launch's trees, see split_fits)
__host__ __device__ __forceinline__ int split_block(const SplitArgs& s) { return s.fill + s.units * s.unit; }
// first unit (of all blocks') of CTA c of n
__host__ __device__ __forceinline__ int split_start(const SplitArgs& s, int c, int n) {
  const int len = split_block(s), x = c * s.step + c * s.rest / n, block = x / len, in = x - block * len - s.fill;
  return block * s.units + (in > 0 ? in / s.unit : 0);
}
// (a n - 1) / total; in 32 bits where they hold the product, as a division in 64 takes half a microsecond
__host__ __device__ __forceinline__ int split_quotient(int a, int n, int total) {
  if (total < (1 << 21)) return static_cast<int>((static_cast<unsigned>(a) * static_cast<unsigned>(n) - 1u) / static_cast<unsigned>(total));
  return static_cast<int>((static_cast<long long>(a) * n - 1) / total);
}
// the CTAs that hold the first and the last unit of a block: the largest c whose start is not behind it
__host__ __device__ __forceinline__ int split_first(const SplitArgs& s, int block, int n) {
  const int len = split_block(s);
  return split_quotient(block * len + s.fill + s.unit, n, s.blocks * len);
}
__host__ __device__ __forceinline__ int split_last(const SplitArgs& s, int block, int n) {
  const int len = split_block(s);
  return split_quotient((block + 1) * len, n, s.blocks * len);
}

// ------------------------------------------------------------------------------------------
// candidate-only rows, once per call
// ------------------------------------------------------------------------------------------

__global__ void combo_mask_kernel(const ks_problem* __restrict__ p, int P, unsigned* __restrict__ mask) {
  unsigned m = 0;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < P; i += gridDim.x * blockDim.x) {
    const ks_problem pr = load_problem(p + i);
    m |= 1u << ((pr.dtype_ab & 3) * 4 + (pr.dtype_d & 3));
  }
  m = __reduce_or_sync(0xFFFFFFFFu, m);
  if ((threadIdx.x & 31) == 0 && m) atomicOr(mask, m);
}

// A block of 256 threads stages the thresholds once and takes kBlock candidates of one type combination
// after the other: kBlock threads evaluate the candidate-only columns, all search (256 / kBlock threads
// a candidate, a column after the other), and the records, put together in shared memory, leave as whole
// lines. What bounds it is latency: of the searches, and of fetching the instructions, so the columns
// are a loop and not 29 copies of the search. kBlock = 64 where C leaves the machine idle (2,048
// candidates: 30 us with one thread a candidate and byte stores, 11 us), else 256, which evaluates with
// every thread. combo0: the only combination (grid y = 1), or -1: blockIdx.y.
constexpr int kCandThreads = 256;
template <int kBlockCands>
__global__ void __launch_bounds__(kCandThreads)
cand_rows_kernel(ks_gpu_desc desc, const ks_candidate* __restrict__ c, int C, const unsigned* mask_ptr, int combo0,
                 FastView fv, uint8_t* __restrict__ out, MemoView memo, int thr_cap, int* ctx_words) {
  extern __shared__ __align__(16) float s_cthr[];  // thresholds of the candidate-only features, values, records
  __shared__ FeatQ s_fq[64];
  const int combo = combo0 >= 0 ? combo0 : blockIdx.y, tid = threadIdx.x;
  if (ctx_words && blockIdx.x == 0 && blockIdx.y == 0 && tid == 0) ctx_words[kWordWalk] = 0;
  if (mask_ptr && !((*mask_ptr >> combo) & 1u)) return;
  const float* T = stage_thresholds(fv, fv.thr_cand0, fv.thr_prob0 - fv.thr_cand0, s_cthr, thr_cap) - fv.thr_cand0;
  if (tid < 64) s_fq[tid] = fv.feat[tid];
  float* s_val = s_cthr + (thr_cap > 0 ? (thr_cap + 3) / 4 * 4 : 0);  // [column][candidate]
  // records an odd number of words apart: no two threads of a warp on one bank
  const int words = fv.cand_rec / 4, stride = words | 1, me = tid % kBlockCands;
  uint32_t* recs = reinterpret_cast<uint32_t*>(s_val + kCandCols * kBlockCands);
  uint8_t* rec = reinterpret_cast<uint8_t*>(recs + me * stride);
  ks_problem fake{};
  fake.m = fake.n = fake.k = 1;
  fake.dtype_ab = static_cast<uint8_t>(combo >> 2);
  fake.dtype_d = static_cast<uint8_t>(combo & 3);
  for (int base = blockIdx.x * kBlockCands; base < C; base += gridDim.x * kBlockCands) {
    if (tid < kBlockCands) {
      const int i = base + tid < C ? base + tid : C - 1;
      ProblemTerms t;
      problem_terms(fake, desc, t);
      const ks_candidate cand = load_candidate(c + i);
      featurize_pair(t, cand, desc, [&](int col, float v) {
        if (feat_class(col) == 1) s_val[cand_slot(col) * kBlockCands + tid] = v;
      });
      if (memo.keys && base + tid < C)
        memo.cls[static_cast<size_t>(combo) * C + i] = memo_assign(memo, combo, i, cand, resources(t, cand, desc).b_eff);
    }
    __syncthreads();
    const int first = fv.n_pair_rows;
#pragma unroll 1
    for (int q = tid / kBlockCands; q < kCandCols; q += kCandThreads / kBlockCands) {
      const FeatQ& f = s_fq[cand_col(q)];
      quantise(f, T + f.thr0, s_val[q * kBlockCands + me], false,
               [&](int row, uint8_t b) { rec[KS_IDX(row - first, fv.cand_rec)] = b; });
    }
    __syncthreads();
    const int n = min(kBlockCands, C - base);
    uint32_t* dst = reinterpret_cast<uint32_t*>(out + (static_cast<size_t>(combo) * C + base) * fv.cand_rec);
    for (int w = tid; w < n * words; w += kCandThreads) dst[w] = recs[w / words * stride + w % words];
    __syncthreads();
  }
}

// Packs the occupied slots of every type combination's table, so that the per-problem kernel runs full
// warps over classes only. `keys` then holds a slot's place. A thread a slot, an atomic operation a warp
// (one block for all of a combination's slots took 7 us for half as many).
__global__ void __launch_bounds__(256)
memo_compact_kernel(MemoView memo) {
  const int combo = blockIdx.y, slot = blockIdx.x * 256 + threadIdx.x, lane = threadIdx.x & 31;
  unsigned long long& key = memo.keys[static_cast<size_t>(combo) * kMemoCap + slot];
  const bool used = key != 0ull;
  const unsigned all = __ballot_sync(0xFFFFFFFFu, used);
  if (all == 0u) return;
  int first = 0;
  if (lane == 0) first = atomicAdd(memo.count + combo, __popc(all));
  const int j = __shfl_sync(0xFFFFFFFFu, first, 0) + __popc(all & ((1u << lane) - 1u));
  if (!used) return;
  memo.dense[static_cast<size_t>(combo) * kMemoCap + j] = slot;
  key = j;  // (the key is not needed any more)
}

// Per problem: the tile bytes of the per-pair rows of every class, from the class's member, plus
// (last block of a row) the problem's own terms and the tile bytes of its problem-only rows.
// grid (kMemoCap / 256, problem lanes): block (x, y) serves classes 256 x .. 256 x + 255 of the
// problems y, y + gridDim.y, ... of the batch, so the thresholds are staged once per block.
// `p` points at the batch's first problem; record (problem within the batch, slot) is written.
// Dynamic shared memory: the staged thresholds (thr_cap floats), then 256 records.
constexpr int kProbRec = kFastMaxProbRows + 128;  // problem-only rows, then the ProblemTerms
static_assert(sizeof(ProblemTerms) <= 128, "problem record");

__global__ void __launch_bounds__(256)
pair_table_kernel(ks_gpu_desc desc, const ks_problem* __restrict__ p, int n_prob,
                  const ks_candidate* __restrict__ c, FastView fv, MemoView memo, int thr_cap, const int* path, int* words, int C,
                  int most_classes) {
  extern __shared__ __align__(16) float s_pthr[];  // thresholds of the per-pair features, then the records
  __shared__ ProblemTerms s_pt;
  __shared__ FeatQ s_fq[64];
  __shared__ float s_pf[64];
  const int tid = threadIdx.x;
  // the select kernel that follows may start its own set-up now (it waits for this grid to finish
  // before it reads the tables)
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  // (also) precedes the select kernel, whose CTAs leave at once when the class walk
  // (ks_gbdt_classes.cu) serves the call; that one then writes the partial lists
  const bool skip = path && *path == 1;
  if (blockIdx.x == 0 && tid == 0) words[kWordWalk] = skip ? kLeaveServed : 0;
  if (skip) return;
  int most = 0;
  for (int q = 0; q < kMemoCombos; ++q) {
    const int n = memo.count[q];
    if (n <= most_classes) {
      most = max(most, n);
    } else {
      // a type combination of too many classes: its candidates have none for the walk, which evaluates their columns in place
      for (int i = blockIdx.x * 256 + tid; i < C; i += gridDim.x * 256) memo.cls[static_cast<size_t>(q) * C + i] = kNoClass;
    }
  }
  // An item is (block of 256 classes, problem); the blocks of the grid deal the items among
  // themselves, so that the work is even whatever the number of classes. The item of class
  // block 0 also writes its problem's own record (problem-only rows and terms).
  const int class_blocks = most > 0 ? (most + 255) / 256 : 1;
  const int n_items = class_blocks * n_prob;
  if (static_cast<int>(blockIdx.x) >= n_items) return;
  const float* T = stage_thresholds(fv, 0, fv.thr_cand0, s_pthr, thr_cap);
  uint8_t* my_rec = reinterpret_cast<uint8_t*>(s_pthr + (thr_cap > 0 ? (thr_cap + 3) / 4 * 4 : 0)) +
                    static_cast<size_t>(tid) * fv.pair_rec;
  if (tid < 64) s_fq[tid] = fv.feat[tid];
  int max_thr = -1;  // the longest threshold list among the per-pair columns (found after the first barrier)
  for (int item = blockIdx.x; item < n_items; item += gridDim.x) {
    const int prob = item / class_blocks, j = (item % class_blocks) * 256 + tid;
    const bool first_block = item % class_blocks == 0;
    const ks_problem pr = load_problem(p + prob);
    const int combo = (pr.dtype_ab & 3) * 4 + (pr.dtype_d & 3);
    const int n_classes = memo.count[combo];
    __syncthreads();  // the previous item's terms are no longer read (and the staging is complete)
    if (tid == 0) {
      problem_terms(pr, desc, s_pt);
      if (first_block) problem_columns(s_pt, [&](int col, float v) { s_pf[col] = v; });
    }
    __syncthreads();
    if (first_block) {
      // once per problem, for all its CTAs: the problem-only rows and the problem's terms
      uint8_t* out = const_cast<uint8_t*>(fv.prob_tab) + static_cast<size_t>(prob) * kProbRec;
      if (tid < KS_F && feat_class(tid) == 0) {
        const FeatQ& q = s_fq[tid];
        const int first = fv.n_pair_rows + fv.n_cand_rows;
        quantise(q, fv.thr + q.thr0, s_pf[tid], false,
                 [&](int row, uint8_t b) { out[KS_IDX(row - first, kFastMaxProbRows)] = b; });
      }
      if (tid < static_cast<int>(sizeof(ProblemTerms) / 4))
        reinterpret_cast<uint32_t*>(out + kFastMaxProbRows)[tid] = reinterpret_cast<const uint32_t*>(&s_pt)[tid];
    }
    if (j >= n_classes || n_classes > most_classes) continue;
    if (max_thr < 0) {
      max_thr = 0;
#pragma unroll
      for (int i = 0; i < kPairCols; ++i) max_thr = max(max_thr, static_cast<int>(s_fq[pair_col(i)].nthr));
    }
    const int slot = memo.dense[static_cast<size_t>(combo) * kMemoCap + j];
    const ks_candidate cand = load_candidate(c + memo.reps[static_cast<size_t>(combo) * kMemoCap + slot]);
    const long long b_eff = resources(s_pt, cand, desc).b_eff;
    float vals[kPairCols];
    pair_columns<true>(s_pt, cand, desc, b_eff, [&](int col, float v) { vals[pair_slot(col)] = v; });
    quantise_pair_columns(s_fq, T, vals, max_thr, [&](int row, uint8_t b) { my_rec[KS_IDX(row, fv.pair_rec)] = b; });
    // the record leaves as whole 16-byte words (it is a multiple of 16 bytes, and so is its place)
    uint4* dst = reinterpret_cast<uint4*>(static_cast<uint8_t*>(memo.tab) +
                                          (static_cast<size_t>(prob) * kMemoCap + slot) * fv.pair_rec);
    const uint4* src = reinterpret_cast<const uint4*>(my_rec);
    for (int q = 0; q < fv.pair_rec / 16; ++q) dst[q] = src[q];
  }
}

// ------------------------------------------------------------------------------------------
// split walks: the whole tile of every (problem, candidate block), once per call
// ------------------------------------------------------------------------------------------

// The rows of one column in 32 words of a tile: x holds the column's values for the lane's four
// candidates. The four searches halve the same interval in step, four instructions a probe and no bound to
// test; slices are cut from pairs of 16-bit counts (a model on this path has fewer than 48 K thresholds) and
// a rank is one byte permutation. A NaN goes right at every numeric split (x < t is false), like +inf.
__device__ __forceinline__ void tile_column(const FeatQ& q, float4 x, uint32_t thr, int n_rows, int W, uint32_t* out) {
  const float v[4] = {x.x, x.y, x.z, x.w};
  if (q.nslice) {
    // the thresholds <= v end at an address in [at, at + 4 n]; !(T > v) holds for a NaN too
    const uint32_t first = thr + 4 * q.thr0;
    uint32_t at[4] = {first, first, first, first};
    const auto probe = [&](uint32_t step) {
      float t[4];
#pragma unroll
      for (int b = 0; b < 4; ++b) t[b] = lds_f32(at[b] + step - 4);
#pragma unroll
      for (int b = 0; b < 4; ++b)
        if (!(t[b] > v[b])) at[b] += step;
    };
    int n = q.nthr;
    for (; n > 1; n -= n >> 1) probe(4u * (n >> 1));
    if (n == 1) probe(4);
    uint32_t lo = (at[0] - first) / 4 | (at[1] - first) / 4 << 16, hi = (at[2] - first) / 4 | (at[3] - first) / 4 << 16;
    for (int s = 0; s < q.nslice; ++s) {
      const uint32_t a = __vminu2(lo, kSlice * 0x00010001u), b = __vminu2(hi, kSlice * 0x00010001u);
      lo -= a;
      hi -= b;
      out[static_cast<size_t>(KS_IDX(q.row0 + s, n_rows)) * W] = 0x80808080u | __byte_perm(a, b, 0x6420);
    }
  }
  if (q.nrank) {
    // a selector per candidate: its level code picks a byte of the rank word, any other value a zero
    uint32_t sel = 0;
#pragma unroll
    for (int b = 0; b < 4; ++b) sel |= min(static_cast<unsigned>(__float2int_rz(v[b])), 4u) << (4 * b);
    for (int k = 0; k < q.nrank; ++k)
      out[static_cast<size_t>(KS_IDX(q.row0 + q.nslice + k, n_rows)) * W] =
          0x80808080u | __byte_perm(*reinterpret_cast<const uint32_t*>(q.rank[k]), 0u, sel);
  }
}

// What a walk copies its tiles from: the per-pair rows of every (problem, candidate block), the candidate-only
// rows of every block once per type combination in use (at the first problem that has it), and every problem's
// record (problem-only rows, then that first problem).
struct PairTiles {
  uint8_t* pair;  // [P][blocks][pair rows][NC]
  uint8_t* cand;  // [P][blocks][candidate rows][NC]
  uint8_t* prob;  // [P][kProbRec]
};
inline PairTiles pair_tiles(const GbdtModel& g, int P, int nblk, uint8_t* mem) {
  const auto up = [](size_t v) { return (v + 255) / 256 * 256; };
  PairTiles t;
  t.pair = mem;
  t.cand = t.pair + up(static_cast<size_t>(P) * nblk * g.n_pair_rows * g.block_cands);
  t.prob = t.cand + up(static_cast<size_t>(P) * nblk * g.n_cand_rows * g.block_cands);
  return t;
}

// An item is 128 candidates (32 words of a tile) of one problem; a block takes a run of items, so that the
// thresholds are staged once and a problem's terms evaluated once or twice. Two threads share a
// candidate's columns; then a warp takes every eighth column, four candidates a lane, and stores whole
// lines, in the layout phase A would produce. The first problem of a type combination also brings the
// candidate-only columns, for all that have it, and the first item of a problem its problem-only rows.
// Two more forms serve a prepared catalogue, whose candidates are taken in `order`: without `tiles.pair` the candidate-only
// rows of all 16 type combinations, once; without `tiles.cand` a call's per-pair rows and record, which then names the
// combination. Slots past the catalogue get the last candidate's bytes (they are not ranked). Also clears the abort flag
// (this kernel precedes the select kernel). What bounds it is the issue of the searches beside the
// latency of the columns' divisions. One problem x 61,140 candidates, 500 trees: 18 us (21 with the candidate-only columns
// for every problem, four searches of the problem-only ones in every lane and a last item for some blocks; a thread that
// wrote its candidate's bytes one by one took 72); 64 x 2,048: 30 -> 16.
constexpr int kTileRows = 128, kTileCols = kPairCols + kCandCols;
// Thresholds that fit beside 64 columns of a block's rows and the static part (49,152). The walk's own tile
// geometries hold 376 rows of 127 at most, 47,752.
constexpr int kTileMaxThr = (227 * 1024 - 3072) / 4 - 64 * kTileRows;
static_assert(kTileMaxThr >= 376 * kSlice, "every ensemble of the regular geometries");

__global__ void __launch_bounds__(256, 4)
tile_pairs_kernel(const __grid_constant__ ks_gpu_desc desc, const ks_problem* __restrict__ p, ks_problem p_value, int use_value, int P,
                  const ks_candidate* __restrict__ c, int C, const int* __restrict__ order, FastView fv, int W, int groups,
                  PairTiles tiles, int* words) {
  extern __shared__ __align__(16) float s_x[];  // [kTileCols][kTileRows], then the thresholds of every feature
  __shared__ ProblemTerms s_pt;
  __shared__ FeatQ s_fq[64];
  __shared__ float s_pf[64];
  __shared__ int s_first;
  float* s_thr = s_x + kTileCols * kTileRows;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");  // (the walk waits for this grid before it reads the tiles)
  if (words && blockIdx.x == 0 && tid == 0) words[kWordWalk] = 0;
  const bool cand_only = !tiles.pair, prepared = !tiles.cand;
  const long long n_items = static_cast<long long>(P) * groups;
  const int begin = static_cast<int>(n_items * blockIdx.x / gridDim.x);
  const int end = static_cast<int>(n_items * (blockIdx.x + 1) / gridDim.x);
  // A problem's terms and columns (the logarithms by threads of their own), and the first problem of its combination.
  // Between two barriers.
  const auto fetch = [&](int prob) {
    ks_problem pr = use_value ? p_value : load_problem(p + prob);
    if (cand_only) {  // "problem" stands for a type combination
      pr.dtype_ab = static_cast<uint8_t>(prob >> 2);
      pr.dtype_d = static_cast<uint8_t>(prob & 3);
    }
    return pr;
  };
  const auto evaluate = [&](int prob) {
    if (tid < 128 && (tid & 31) == 0) {
      const ks_problem pr = fetch(prob);
      if (tid == 0) {
        problem_terms<false>(pr, desc, s_pt);
        problem_columns(s_pt, [&](int col, float v) { if (col > 2) s_pf[col] = v; });
      } else {
        s_pf[warp - 1] = log2_dim(warp == 1 ? pr.m : (warp == 2 ? pr.n : pr.k));
      }
    } else if (tid >= 128) {
      const ks_problem pr = fetch(prob);
      int first = prepared ? (pr.dtype_ab & 3) * 4 + (pr.dtype_d & 3) : prob;
      if (!use_value)
        for (int q = tid - 128; q < first; q += 128) {
          const ks_problem other = load_problem(p + q);
          if ((other.dtype_ab & 3) == (pr.dtype_ab & 3) && (other.dtype_d & 3) == (pr.dtype_d & 3)) first = q;
        }
      first = __reduce_min_sync(0xFFFFFFFFu, first);
      if (lane == 0) atomicMin(&s_first, first);
    }
  };
  int held = begin / groups;
  if (tid == 0) s_first = INT_MAX;
  if (tid < 64) s_fq[tid] = fv.feat[tid];
  __syncthreads();
  if (begin < end) evaluate(held);
  stage_thresholds(fv, 0, fv.n_thr, s_thr, fv.n_thr);
  const uint32_t thr = smem_u32(s_thr);
  for (int item = begin; item < end; ++item) {
    const int prob = item / groups, g = item - prob * groups;
    __syncthreads();  // the columns of the item before have been read
    if (prob != held) {
      if (tid == 0) s_first = INT_MAX;
      __syncthreads();
      evaluate(prob);
      held = prob;
      __syncthreads();
    }
    if (g == 0 && !cand_only) {
      uint8_t* rec = tiles.prob + static_cast<size_t>(prob) * kProbRec;
      if (tid < KS_F && feat_class(tid) == 0) {
        const FeatQ& q = s_fq[tid];
        const int first = fv.n_pair_rows + fv.n_cand_rows;
        quantise(q, s_thr + q.thr0, s_pf[tid], false, [&](int row, uint8_t b) { rec[KS_IDX(row - first, kFastMaxProbRows)] = b; });
      }
      if (tid == 64) *reinterpret_cast<int*>(rec + kFastMaxProbRows) = s_first;
    }
    const bool with_cand = s_first == prob && !prepared;
    const int row = tid % kTileRows, place = min(g * kTileRows + row, C - 1);
    const ks_candidate cand = load_candidate(c + (order ? __ldg(order + place) : place));
    const long long b_eff = resources(s_pt, cand, desc).b_eff;
    if (cand_only)
      ;
    else if (tid < kTileRows)
      pair_columns<true>(s_pt, cand, desc, b_eff, [&](int col, float v) { if (col <= 32) s_x[pair_slot(col) * kTileRows + row] = v; });
    else
      pair_columns<true>(s_pt, cand, desc, b_eff, [&](int col, float v) { if (col > 32) s_x[pair_slot(col) * kTileRows + row] = v; });
    if (with_cand) {
      const auto put = [&](int col, float v) {
        if (col < KS_F && feat_class(col) == 1) s_x[(kPairCols + cand_slot(col)) * kTileRows + row] = v;
      };
      if (tid < kTileRows) featurize_pair(s_pt, cand, desc, [&](int col, float v) { if (col <= 49) put(col, v); });
      else featurize_pair(s_pt, cand, desc, [&](int col, float v) { if (col > 49) put(col, v); });
    }
    __syncthreads();
    const int in_block = g * 32 / W, word = g * 32 - in_block * W + lane;
    const size_t block = static_cast<size_t>(prob) * (groups * 32 / W) + in_block;
    uint32_t* pair_out = reinterpret_cast<uint32_t*>(tiles.pair) + block * fv.n_pair_rows * W + word;
    // (rows are counted over the whole tile: the candidate-only ones follow the per-pair ones)
    uint32_t* cand_out = reinterpret_cast<uint32_t*>(tiles.cand) + block * fv.n_cand_rows * W + word - static_cast<ptrdiff_t>(fv.n_pair_rows) * W;
#pragma unroll 1
    for (int slot = warp + (cand_only ? kPairCols : 0); slot < (with_cand ? kTileCols : kPairCols); slot += 8) {
      const bool is_pair = slot < kPairCols;
      const float4 x = *reinterpret_cast<const float4*>(s_x + slot * kTileRows + 4 * lane);
      tile_column(s_fq[is_pair ? pair_col(slot) : cand_col(slot - kPairCols)], x, thr, fv.n_rows, W, is_pair ? pair_out : cand_out);
    }
  }
}

// ------------------------------------------------------------------------------------------
// scoring call: tiles from feature rows
// ------------------------------------------------------------------------------------------

// ks_score with a qualifying ensemble: quantise feature rows into the tile layout of phase A. A block
// brings 128 rows (32 words of a tile) into shared memory by whole sectors and column by column, the next
// ones on their way in registers meanwhile; a warp then takes every 16th column, four rows a lane, and
// stores whole lines. The walk kernel copies the tiles as in a split walk and writes the scores instead of
// ranking. Slots past the last row get the last row's bytes (their scores are not stored). Also clears the abort flag.
//
// What bounds it is the searches' chains of shared-memory loads and their issue. A million rows, 500 trees of depth 8: 166 us (260 MB of rows and 180 MB of tiles: 68 us); a thread
// reading 16 bytes of its four rows at a time and searching row by row took 405 us.
constexpr int kTileWarps = 16;

__global__ void __launch_bounds__(kTileWarps * 32, 2)
tile_rows_kernel(const float* __restrict__ feat, int64_t rows, FastView fv, uint8_t* __restrict__ tiles, int W,
                 int groups, int* words) {
  extern __shared__ __align__(16) float s_x[];  // [64][kTileRows], then the thresholds of every feature
  __shared__ FeatQ s_fq[64];
  float* s_thr = s_x + 64 * kTileRows;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");  // (the walk waits for this grid before it reads the tiles)
  if (blockIdx.x == 0 && threadIdx.x == 0) words[kWordWalk] = 0;
  stage_thresholds(fv, 0, fv.n_thr, s_thr, fv.n_thr);
  if (threadIdx.x < 64) s_fq[threadIdx.x] = fv.feat[threadIdx.x];
  const uint32_t thr = smem_u32(s_thr);
  const int per_block = W / 32;
  // a warp reads 64 bytes of each of eight rows at a time; row r of a column stands at r ^ 8 (column / 4 % 4),
  // which keeps four rows together and puts a warp's 32 stores on different banks
  const int r = 8 * warp + lane / 4, q0 = lane & 3;
  float4 f[4];
  const auto fetch = [&](int g) {
    const int64_t row = static_cast<int64_t>(g) * kTileRows + r;
    const float4* src = reinterpret_cast<const float4*>(feat + (row < rows ? row : rows - 1) * KS_F_PAD) + q0;
#pragma unroll
    for (int i = 0; i < 4; ++i) f[i] = __ldg(src + 4 * i);
  };
  fetch(blockIdx.x);
  for (int g = blockIdx.x; g < groups; g += gridDim.x) {
    __syncthreads();  // the columns of the group before have been read
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      float* to = s_x + 4 * (q0 + 4 * i) * kTileRows + (r ^ 8 * q0);
      to[0] = f[i].x; to[kTileRows] = f[i].y; to[2 * kTileRows] = f[i].z; to[3 * kTileRows] = f[i].w;
    }
    __syncthreads();
    if (g + gridDim.x < groups) fetch(g + gridDim.x);
    const int block = g / per_block, word = (g - block * per_block) * 32 + lane;
    uint32_t* out = reinterpret_cast<uint32_t*>(tiles) + static_cast<size_t>(block) * fv.n_rows * W + word;
#pragma unroll 1
    for (int col = warp; col < KS_F; col += kTileWarps) {
      const float4 x = *reinterpret_cast<const float4*>(s_x + col * kTileRows + (4 * lane ^ 8 * (col / 4 & 3)));
      tile_column(s_fq[col], x, thr, fv.n_rows, W, out);
    }
  }
}

// ------------------------------------------------------------------------------------------
// phase A
// ------------------------------------------------------------------------------------------

// Sixteen rows of four neighbouring candidates: q[r] holds candidate r's bytes of rows row0 ..
// row0 + 15 (a 16-byte vector of its record). Byte r of a tile word is candidate r, so every
// group of four rows is a 4 x 4 byte transpose (eight byte permutes) and four word stores.
__device__ __forceinline__ void scatter_vectors(const uint4 (&q)[4], int row0, int n, unsigned char* word0, int NC) {
  const uint32_t w[4][4] = {{q[0].x, q[0].y, q[0].z, q[0].w},
                            {q[1].x, q[1].y, q[1].z, q[1].w},
                            {q[2].x, q[2].y, q[2].z, q[2].w},
                            {q[3].x, q[3].y, q[3].z, q[3].w}};
#pragma unroll
  for (int g = 0; g < 4; ++g) {
    const int row = row0 + 4 * g;
    if (row >= n) break;
    const uint32_t lo_ab = __byte_perm(w[0][g], w[1][g], 0x5140u), lo_cd = __byte_perm(w[2][g], w[3][g], 0x5140u);
    const uint32_t hi_ab = __byte_perm(w[0][g], w[1][g], 0x7362u), hi_cd = __byte_perm(w[2][g], w[3][g], 0x7362u);
    const uint32_t out[4] = {__byte_perm(lo_ab, lo_cd, 0x5410u), __byte_perm(lo_ab, lo_cd, 0x7632u),
                             __byte_perm(hi_ab, hi_cd, 0x5410u), __byte_perm(hi_ab, hi_cd, 0x7632u)};
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (row + j < n) *reinterpret_cast<uint32_t*>(word0 + static_cast<size_t>(row + j) * NC) = out[j];
  }
}

// Fills the tile: candidate-only rows from the per-call table, problem-only rows from s_pbin,
// per-pair rows from the memo record of the candidate's class or computed here. Slots past the
// end of the segment get a neutral byte so that word-wise arithmetic on the tile never borrows
// across bytes. A thread serves the four candidates of one tile word (byte r of the word is
// candidate r): it fetches their records sixteen rows at a time and stores whole words; the
// THREADS / (NC / 4) threads that share a word deal the records' vectors among themselves.
template <int THREADS, int NC>
__device__ __noinline__ void fill_tile(const ks_gpu_desc& desc, const ProblemTerms& pt,
                                       const ks_candidate* __restrict__ c, const FastView& fv,
                                       const int64_t* __restrict__ seg_off, const int32_t* __restrict__ seg_idx,
                                       int C, int64_t lo, int64_t start, int64_t stop, const float* T,
                                       const FeatQ* s_fq, const uint8_t* s_pbin, unsigned char* tile, int prob,
                                       unsigned* s_cid, bool reuse) {
  constexpr int W = NC / 4, PARTS = THREADS / W;
  const int tid = threadIdx.x;
  const int combo = pt.dtype_ab * 4 + pt.dtype_d;
  // `reuse`: the tile still holds the candidate-only rows of these very candidates (the CTA's last
  // item was the same candidate block under the same element types), and s_cid their classes.
  // problem-only rows: one byte for the whole row
  {
    unsigned char* dst = tile + static_cast<size_t>(fv.n_pair_rows + fv.n_cand_rows) * NC;
    for (int i = tid; i < fv.n_prob_rows * (NC / 16); i += THREADS) {
      const uint32_t b = s_pbin[i / (NC / 16)] * 0x01010101u;
      reinterpret_cast<uint4*>(dst)[i] = make_uint4(b, b, b, b);
    }
  }
  const int word = tid % W, part = tid / W;
  unsigned char* word0 = tile + 4 * word;
  int ci[4];
  unsigned cid[4];
  bool lone = false;  // one of this word's candidates has no record of per-pair rows
  if (reuse) {
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      ci[r] = start + 4 * word + r < stop ? 0 : -1;  // (the pool index itself is not needed again)
      cid[r] = s_cid[4 * word + r];
      lone |= ci[r] >= 0 && cid[r] == kNoClass;
    }
  } else {
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const int64_t row = start + 4 * word + r;
      ci[r] = row < stop ? (seg_idx ? seg_idx[lo + row] : static_cast<int>(row)) : -1;
    }
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      cid[r] = (ci[r] >= 0 && fv.pair_class) ? __ldg(fv.pair_class + static_cast<size_t>(combo) * C + ci[r]) : kNoClass;
      lone |= ci[r] >= 0 && cid[r] == kNoClass;
      if (s_cid && part == 0) s_cid[4 * word + r] = cid[r];
    }
  }
  const uint4 neutral = make_uint4(0x80808080u, 0x80808080u, 0x80808080u, 0x80808080u);
  const int cand_vecs = (fv.n_cand_rows + 15) / 16, pair_vecs = (fv.n_pair_rows + 15) / 16;
  const uint8_t* cand_rec[4];
  const uint8_t* pair_rec[4];
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    cand_rec[r] = ci[r] >= 0 ? fv.cand_rows + (static_cast<size_t>(combo) * C + KS_IDX(ci[r], C)) * fv.cand_rec : nullptr;
    pair_rec[r] = cid[r] != kNoClass
                      ? fv.pair_tab + (static_cast<size_t>(prob) * kMemoCap + KS_IDX(cid[r], kMemoCap)) * fv.pair_rec
                      : nullptr;
  }
  // kBatch vectors of the four candidates are fetched before the first is stored, so that a thread
  // waits for the memory once per batch, not once per vector
  constexpr int kBatch = 1;
#pragma unroll 1
  for (int v0 = (reuse ? cand_vecs : 0) + part; v0 < cand_vecs + pair_vecs; v0 += kBatch * PARTS) {
    uint4 q[kBatch][4];
#pragma unroll
    for (int j = 0; j < kBatch; ++j) {
      const int v = v0 + j * PARTS;
      if (v >= cand_vecs + pair_vecs) break;
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        const uint8_t* rec = v < cand_vecs ? cand_rec[r] : pair_rec[r];
        q[j][r] = rec ? __ldg(reinterpret_cast<const uint4*>(rec) + (v < cand_vecs ? v : v - cand_vecs)) : neutral;
      }
    }
#pragma unroll
    for (int j = 0; j < kBatch; ++j) {
      const int v = v0 + j * PARTS;
      if (v >= cand_vecs + pair_vecs) break;
      if (v < cand_vecs) scatter_vectors(q[j], 16 * v, fv.n_cand_rows, word0 + static_cast<size_t>(fv.n_pair_rows) * NC, NC);
      else scatter_vectors(q[j], 16 * (v - cand_vecs), fv.n_pair_rows, word0, NC);
    }
  }
  // candidates without a record (no memo in this call, no class, or a class table that was full): their
  // per-pair columns are computed here, after the word stores that cover their bytes
  if (!__syncthreads_or(lone)) return;
  if (!lone) return;
#pragma unroll 1
  for (int r = part % 4; r < 4; r += (PARTS < 4 ? PARTS : 4)) {
    if (ci[r] < 0 || cid[r] != kNoClass) continue;
    unsigned char* my = word0 + r;
    const int64_t row = start + 4 * word + r;
    const ks_candidate cand = load_candidate(c + (seg_idx ? seg_idx[lo + row] : static_cast<int>(row)));
    pair_columns<true>(pt, cand, desc, resources(pt, cand, desc).b_eff, [&](int col, float v) {
      const FeatQ& q = s_fq[col];
      quantise(q, T + q.thr0, v, false, [&](int row, uint8_t b) { my[KS_IDX(row, fv.n_pair_rows) * NC] = b; });
    });
  }
}

// ------------------------------------------------------------------------------------------
// the kernel
// ------------------------------------------------------------------------------------------

// Bounded wait for a tile that is copied in one piece: the thread is suspended by the barrier itself, for as long as the
// hardware sees fit, so the bound is a time: half a microsecond a probe of `limit`. (To sleep here as mbar_wait_bounded
// does costs a single call 2 us of 96.)
__device__ __forceinline__ bool tile_wait(uint32_t bar, uint32_t parity, int limit, volatile int* fail) {
  const long long begin = clock64(), most = static_cast<long long>(limit) * 1000;
  while (!mbar_try_wait(bar, parity))
    if (*fail || clock64() - begin > most) return false;
  return true;
}

// bytes of `a` where the top bit of the matching byte of `m` is set, else bytes of `b`
__device__ __forceinline__ uint32_t byte_select(uint32_t m, uint32_t a, uint32_t b) {
  const uint32_t f = __byte_perm(m, 0u, 0xBA98u);  // top bit of every byte replicated over the byte
  return (a & f) | (b & ~f);
}

// one path step of one walk: fetch the node, fetch the candidate's byte, move to the child:
// next = 2 a + k0 (+ 4 when the candidate goes right)
#ifndef KS_DEBUG_BOUNDS
__device__ __forceinline__ uint32_t path_step(uint32_t a, uint32_t cb_r, uint32_t k0, uint32_t, uint32_t, uint32_t) {
  uint32_t nx;
  asm volatile(
      "{\n"
      " .reg .u32 n, x, m;\n"
      " .reg .pred p;\n"
      " ld.shared.u32 n, [%1];\n"
      " shr.u32 m, n, 8;\n"
      " add.u32 m, m, %2;\n"
      " ld.shared.u8 x, [m];\n"
      " and.b32 n, n, 255;\n"
      " setp.gt.u32 p, x, n;\n"
      " mad.lo.u32 %0, %1, 2, %3;\n"
      " @p add.u32 %0, %0, 4;\n"
      "}\n"
      : "=r"(nx)
      : "r"(a), "r"(cb_r), "r"(k0));
  return nx;
}
#else
// checked build: the node address must lie in the chunk buffer, the byte address in the tile
__device__ __forceinline__ uint32_t path_step(uint32_t a, uint32_t cb_r, uint32_t k0, uint32_t buf,
                                              uint32_t tile0, uint32_t tile_bytes) {
  a = buf + static_cast<uint32_t>(KS_IDX((a - buf) >> 2, 2 * kBufBytes / 4)) * 4u;
  const uint32_t n = lds_u32(a);
  uint32_t m = (n >> 8) + cb_r;
  m = tile0 + static_cast<uint32_t>(KS_IDX(m - tile0, tile_bytes));
  uint32_t x;
  asm volatile("ld.shared.u8 %0, [%1];" : "=r"(x) : "r"(m));
  return 2u * a + k0 + (x > (n & 255u) ? 4u : 0u);
}
#endif

// L levels evaluated word-wise; NP path levels unrolled (-1: runtime count); kCompact: the top
// levels' constants travel as one 32-bit word per node (row offset << 8 | j + 1) instead of a
// (row offset, replicated j + 1) pair, so that twice as many trees keep their word-wise levels.
// THREADS threads rank NC candidates: NC / 4 words times THREADS / (NC / 4) tree groups.
// kSplit: the CTAs share out the blocks' trees (SplitArgs); a form of its own, since what it keeps slowed the
// other by 2 %.
// kShared: the top levels come from the chunk in shared memory, not from the parameters. That takes three more
// shared-memory wavefronts and seven more instructions a tree (5 % of the walk), but a launch costs the host 7 us
// where 28 KB of parameters make it 21; see takes_shared_top.
// kFloor (measurement only): the walk without its chunk rings. Every tree group's first kNBuf
// chunks are copied once and stay resident; the group walks them again and again (sl.repeat
// times as many chunk walks as it has chunks), never waits, releases or refills, so the time per
// pass is that of the gather and instruction stream of the walk alone, at the occupancy and tile
// size of the real kernel.
template <bool kShared>
struct TopArg {
  FastTopParams p;
};
template <>
struct TopArg<true> {};

template <int L, int NP, bool kCompact, int THREADS, int NC, bool kSplit, bool kShared = false, bool kFloor = false>
__global__ void __launch_bounds__(THREADS, THREADS <= 256 ? 2 : 1)
select_fast_kernel(ks_gpu_desc desc, const ks_problem* __restrict__ p, ks_problem p_value, int use_value,
                   const ks_candidate* __restrict__ c, int P, int C, int nblk, int rows_per_cta,
                   const int64_t* __restrict__ seg_off, const int32_t* __restrict__ seg_idx, FastView fv,
                   int k, unsigned long long* __restrict__ partial, int* __restrict__ status,
                   SplitArgs sl, int n_items, const __grid_constant__ TopArg<kShared> top) {
  constexpr int W = NC / 4;        // words per tile row = lane slots
  constexpr int G = THREADS / W;   // tree groups
  constexpr int RG = ring_count(G);  // chunk rings
  constexpr int GPR = G / RG;        // groups that share a ring (and split the trees of its chunks)
  static_assert(THREADS % W == 0 && W % 32 == 0 && G >= 1, "tile geometry");
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ ProblemTerms s_pt;
  __shared__ unsigned long long s_warp[THREADS / 32 * KS_MAX_K];
  __shared__ unsigned long long s_list[KS_MAX_K];
  __shared__ __align__(8) unsigned long long s_bar[kNBuf * RG + 1];  // [ring][buffer], then the tile's
  __shared__ FeatQ s_fq[64];
  __shared__ uint8_t s_pbin[kFastMaxProbRows];
  __shared__ float s_pfeat[64];
  __shared__ int s_fail, s_last, s_done[kNBuf * RG], s_abort, s_pending[kNBuf * RG], s_parts[3];
  // the classes of the candidates whose candidate-only rows the tile holds (one-CTA forms only:
  // there a CTA serves one candidate block for many problems in a row, see below)
  __shared__ unsigned s_cid[THREADS > 256 && NC == 1024 ? NC : 1];

  const int tid = threadIdx.x;
  const int kOffTile = kNBuf * RG * fv.buf_bytes;  // every ring has kNBuf buffers
  const uint32_t sbase = smem_u32(smem);
  const uint32_t bar0 = smem_u32(&s_bar[0]);  // barrier of buffer b: bar0 + 8 b
  const bool tiles_given = sl.tiles != nullptr;  // the tiles were built in front: no feature work here
  if (tid == 0) {
    for (int b = 0; b <= kNBuf * RG; ++b) mbar_init(bar0 + 8u * b, 1);
    s_fail = 0;
    for (int b = 0; b < kNBuf * RG; ++b) s_done[b] = s_pending[b] = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (tid < 64) s_fq[tid] = fv.feat[tid];
  __syncthreads();
  uint32_t phases = 0;  // bit b: parity of buffer b's barrier
  const int word = tid % W, grp = tid / W;
  volatile int* v_fail = &s_fail;

  // An item is one (problem, candidate block). The batch form of a geometry that holds one CTA per SM is
  // launched with one CTA per SM, so that a CTA's set-up and the gap between two CTAs are paid
  // once, not per item; so is a split walk, whose CTAs take parts of items. Two CTAs per SM hide each
  // other's gaps: there a batch is launched with one CTA per item.
  // A CTA (of the 1,024-candidate forms) that serves many items of a dense batch takes a run of
  // consecutive items in the order (candidate block, problem): successive items then are the same
  // candidates for another problem, and while the element types stay the same their
  // candidate-only rows (and classes) stay in place. (The 512-candidate form serves segmented
  // batches in the benchmark; compiled with this path it ran them 2 % slower, so it keeps the
  // plain order.)
  const int grid = static_cast<int>(gridDim.x), cta = static_cast<int>(blockIdx.x);
  constexpr bool split = kSplit;
  const bool block_major = NC == 1024 && grid < n_items && !seg_off && !tiles_given;
  const int per_cta = (n_items + grid - 1) / grid;
  int unit = split ? split_start(sl, cta, grid) : 0;  // a split walk: the next unit
  const int unit_first = unit, unit_end = split ? split_start(sl, cta + 1, grid) : 0;
  int first_item = block_major ? cta * per_cta : cta, item_step = block_major ? 1 : grid;
  int last_item = block_major ? (first_item + per_cta < n_items ? first_item + per_cta : n_items) : n_items;
  if (split) {
    first_item = unit / sl.units;
    item_step = 1;
    last_item = (unit_end + sl.units - 1) / sl.units;
  }
  int held_chunk = -1, held_combo = -1;  // what the tile's candidate-only rows belong to
  uint32_t tile_phase = 0;
  // everything above is independent of the kernel in front (the per-problem tables): when this
  // grid was launched as its programmatic dependent, wait for that grid here
  asm volatile("griddepcontrol.wait;" ::: "memory");
#pragma unroll 1
  for (int item = first_item; item < last_item; item += item_step) {
  const int prob = block_major ? item % P : item / nblk;
  const int chunk = block_major ? item / P : item % nblk;
  // rows of this problem: lo = where its scores sit in per-row arrays; lo_idx = where its pool
  // indices start in seg_idx (per-problem segments, or - without offsets - one ranking order of
  // the whole catalogue shared by every problem)
  int64_t lo, len, lo_idx;
  if (seg_off) {
    lo = lo_idx = seg_off[prob];
    len = seg_off[prob + 1] - lo;
  } else {
    lo = static_cast<int64_t>(prob) * C;
    lo_idx = 0;
    len = C;
  }
  // chunks of the ensemble this CTA walks
  int ch_begin = 0, ch_end = fv.n_chunks;
  const bool first_part = unit == unit_first;
  if (split) {
    const int block0 = item * sl.units;
    ch_begin = (unit - block0) * RG;
    unit = unit_end < block0 + sl.units ? unit_end : block0 + sl.units;
    ch_end = (unit - block0) * RG < fv.n_chunks ? (unit - block0) * RG : fv.n_chunks;
  }
  const bool whole = ch_begin == 0 && ch_end == fv.n_chunks;
  __syncthreads();  // the item before this one is finished with the shared state
  if (tid == 0) {
    if (!fv.prob_tab && !tiles_given) {
      problem_terms(use_value ? p_value : load_problem(p + prob), desc, s_pt);
      problem_columns(s_pt, [&](int col, float v) { s_pfeat[col] = v; });
    }
    s_abort = *reinterpret_cast<volatile int*>(sl.words + kWordWalk);
  }
  if (tid < KS_MAX_K) s_list[tid] = 0ull;
  if (fv.prob_tab) {
    const uint8_t* rec = fv.prob_tab + static_cast<size_t>(prob) * kProbRec;
    for (int i = tid; i < fv.n_prob_rows; i += THREADS) s_pbin[i] = __ldcg(rec + i);
    if (tid < static_cast<int>(sizeof(ProblemTerms) / 4))
      reinterpret_cast<uint32_t*>(&s_pt)[tid] = __ldcg(reinterpret_cast<const uint32_t*>(rec + kFastMaxProbRows) + tid);
  }
  __syncthreads();
  if (s_abort) {  // a wait ran out in an earlier CTA of this call, which fails, or the class walk serves the call: leave at once
    if (s_abort == kLeaveFailed && tid == 0 && status) atomicExch(status, KS_ERR_TIMEOUT);
    if (tid < k && partial) partial[(static_cast<size_t>(prob) * nblk + chunk) * k + tid] = 0ull;
    return;
  }
  if (!tiles_given && !fv.prob_tab && tid < KS_F && feat_class(tid) == 0) {
    const int first = fv.n_pair_rows + fv.n_cand_rows;
    const FeatQ& q = s_fq[tid];
    quantise(q, fv.thr + q.thr0, s_pfeat[tid], false,
             [&](int row, uint8_t b) { s_pbin[KS_IDX(row - first, kFastMaxProbRows)] = b; });
  }

  bool ranked = !sl.score_out;
  for (int64_t start = static_cast<int64_t>(chunk) * rows_per_cta; start < len;
       start += static_cast<int64_t>(nblk) * rows_per_cta) {
    const int64_t stop = (start + rows_per_cta < len) ? start + rows_per_cta : len;
    // ---- phase A ---------------------------------------------------------------------------------
    __syncthreads();
    // (asked where it is used: kept over the walk's loop it costs a walk of whole blocks up to 1.8 %)
    const auto starved = [&] { return split ? fv.starve == kStarveAll || (fv.starve == kStarveOdd && (cta & 1)) : fv.starve != 0; };
    // The first chunks are on their way while the tile is filled, where the fill leaves the chunk buffers alone.
    const auto start_rings = [&] {
      // ring g takes the chunks ch_begin + g, ch_begin + g + RG, ... through its own buffers
      for (int g = 0; g < RG; ++g)
        for (int b = 0; b < kNBuf && ch_begin + g + b * RG < ch_end; ++b) {
          const int rb = g * kNBuf + b;
          // test hook: a barrier armed for more bytes than its copy brings never completes
          mbar_expect_tx(bar0 + 8u * rb, fv.chunk_bytes + (starved() ? 16 : 0));
          bulk_copy_g2s(sbase + kOffBuf0 + rb * fv.buf_bytes,
                        reinterpret_cast<const char*>(fv.chunks) + static_cast<size_t>(ch_begin + g + b * RG) * fv.chunk_bytes,
                        fv.chunk_bytes, bar0 + 8u * rb);
          s_pending[rb] = 1;
        }
    };
    const bool early = tiles_given || fv.pair_class;
    if (early && tid == 0) {
      fence_async_proxy();
      if (tiles_given) {
        // the block's tile was built in front, in one piece or two
        const uint32_t bar = bar0 + 8u * (kNBuf * RG);
        const uint32_t bytes = static_cast<uint32_t>(sl.cand_tiles ? fv.n_pair_rows : fv.n_rows) * NC;
        const uint32_t more = sl.cand_tiles ? static_cast<uint32_t>(fv.n_cand_rows) * NC : 0u;
        asm volatile("fence.proxy.async.global;" ::: "memory");  // (written by ordinary stores of the kernel in front)
        mbar_expect_tx(bar, bytes + more + (fv.starve == kStarveTiles ? 16 : 0));  // (test hook, as below)
        if (bytes) bulk_copy_g2s(sbase + kOffTile, sl.tiles + (static_cast<size_t>(prob) * nblk + chunk) * bytes, bytes, bar);
        // (the record's terms are the first problem of the combination here)
        if (more) {
          const size_t first = KS_IDX(*reinterpret_cast<const int*>(&s_pt), P > kCombos ? P : kCombos);
          bulk_copy_g2s(sbase + kOffTile + bytes, sl.cand_tiles + (first * nblk + chunk) * more, more, bar);
        }
      }
      start_rings();
    }
    bool tile_late = false;
    if (tiles_given) {
      if (sl.cand_tiles) {  // problem-only rows: one byte for the whole row
        unsigned char* dst = smem + kOffTile + static_cast<size_t>(fv.n_pair_rows + fv.n_cand_rows) * NC;
        for (int i = tid; i < fv.n_prob_rows * (NC / 16); i += THREADS) {
          const uint32_t b = s_pbin[i / (NC / 16)] * 0x01010101u;
          reinterpret_cast<uint4*>(dst)[i] = make_uint4(b, b, b, b);
        }
      }
      if (!tile_wait(bar0 + 8u * (kNBuf * RG), tile_phase, fv.wait_limit, v_fail)) {
        tile_late = true;
        if (!*v_fail) {
          s_fail = 1;
          atomicExch(sl.words + kWordWalk, kLeaveFailed);
          if (status) atomicExch(status, KS_ERR_TIMEOUT);
        }
      }
      tile_phase ^= 1u;
    } else {
      // thresholds of the per-pair features: into the idle chunk buffers when they fit
      const float* T = stage_thresholds(fv, 0, fv.thr_cand0, reinterpret_cast<float*>(smem + kOffBuf0),
                                        fv.pair_class ? 0 : kNBuf * RG * fv.buf_bytes / 4);
      __syncthreads();
      const int combo = s_pt.dtype_ab * 4 + s_pt.dtype_d;
      const bool reuse = THREADS > 256 && block_major && fv.pair_class && chunk == held_chunk && combo == held_combo;
      fill_tile<THREADS, NC>(desc, s_pt, c, fv, seg_off, seg_idx, C, lo_idx, start, stop, T, s_fq, s_pbin,
                             smem + kOffTile, prob, THREADS > 256 && block_major ? s_cid : nullptr, reuse);
      held_chunk = chunk;
      held_combo = combo;
    }
    __syncthreads();  // tile complete; the threshold table is no longer needed

    // ---- phase B ---------------------------------------------------------------------------------
    if (!early && tid == 0) {
      fence_async_proxy();
      start_rings();
    }
    float score[4] = {0.0f, 0.0f, 0.0f, 0.0f};
    double sums[4] = {0.0, 0.0, 0.0, 0.0};  // split walk: of the chunks' sums
    const uint32_t cb = sbase + kOffTile + word * 4;
    const int tpc = fv.tpc, grp_trees = (tpc + GPR - 1) / GPR;
    const int np = NP >= 0 ? NP : fv.depth - L;
    constexpr int kTop = (1 << L) - 1;
    const int ring = grp / GPR;
    // the groups of a ring share out the trees of its chunks
    const int t_first = (grp % GPR) * grp_trees;
    const int t_count = t_first + grp_trees <= tpc ? grp_trees : (tpc > t_first ? tpc - t_first : 0);
#ifdef KS_DEBUG_BOUNDS
    const uint32_t tile0 = sbase + kOffTile, tile_bytes = static_cast<uint32_t>(fv.n_rows) * NC;
#else
    constexpr uint32_t tile0 = 0, tile_bytes = 0;
#endif
    // this ring's chunks: n_mine of them; the floor form walks its first kNBuf again and again
    const int n_mine = ch_end - ch_begin > ring ? (ch_end - ch_begin - ring + RG - 1) / RG : 0;
    const int n_walks = kFloor ? n_mine * sl.repeat : n_mine;
#pragma unroll 1
    for (int it = 0; it < n_walks; ++it) {
      const int b = it % kNBuf, rb = ring * kNBuf + b;
      const int ch = ch_begin + ring + (kFloor ? b : it) * RG;  // the chunk whose trees are walked
      const uint32_t bar = bar0 + 8u * rb;
      const uint32_t par = (phases >> b) & 1u;
      // A wait that runs out ends the walk of this CTA: the buffer was never filled, so it is not
      // read; the call fails, and the CTAs that start later leave at once.
      if (!kFloor || it < kNBuf) {
        if (*v_fail || !mbar_wait_bounded(bar, par, fv.wait_limit, v_fail)) {
          if (!*v_fail) {
            s_fail = 1;
            atomicExch(sl.words + kWordWalk, kLeaveFailed);
            if (status) atomicExch(status, KS_ERR_TIMEOUT);
          }
          break;
        }
        phases ^= 1u << b;
      }
      const uint32_t buf = sbase + kOffBuf0 + rb * fv.buf_bytes;
      // With A_l the shared address of a walk's node at level l, A_{l+1} = 2 A_l + (4 tpc - buf)
      // + 4 bit for every level, and after the last level A points at the walk's leaf.
      const uint32_t k0 = 4u * tpc - buf;  // modulo 2^32, like the additions it enters
      const uint32_t lvlL = buf + 4u * tpc * kTop;  // first node of level L
#pragma unroll 4
      for (int tt = 0; tt < t_count; ++tt) {
        const int t = t_first + tt;
        uint32_t a[4];
        if (L == 0) {
#pragma unroll
          for (int r = 0; r < 4; ++r) a[r] = buf + 4u * t;
        } else {
          // Word-wise evaluation of the top L levels for the four candidates of this word.
          // A tile byte is 0x80 | bin and a node constant (j + 1) in every byte, so byte r of
          // d[n] keeps its top bit iff candidate r goes right at node n; no byte borrows.
          uint32_t d[kTop > 0 ? kTop : 1];
          if constexpr (kShared) {
            // (the nodes of a level lie side by side, aligned since a chunk's trees are a multiple of four). A node's low
            // byte is v = 0x80 | j: byte r of tile + 0x7F.. - v.. is 0x80 + bin - (j + 1), as below.
            uint32_t n[7];
            n[0] = lds_u32(buf + 4u * t);
            lds_u64(buf + 4u * tpc + 8u * t, n[1], n[2]);
            lds_u128(buf + 12u * tpc + 16u * t, n[3], n[4], n[5], n[6]);
#pragma unroll
            for (int i = 0; i < 7; ++i)
              d[i] = lds_u32(cb + static_cast<uint32_t>(KS_IDX(n[i] >> 8, fv.n_rows * NC))) + 0x7F7F7F7Fu - __byte_perm(n[i], 0u, 0u);
          } else if constexpr (kCompact) {
            const uint32_t* tw = reinterpret_cast<const uint32_t*>(top.p.w) +
                                 static_cast<size_t>(KS_IDX(ch * tpc + t, 2 * kFastTopPairs / (kTop > 0 ? kTop : 1))) * kTop;
#pragma unroll
            for (int n = 0; n < kTop; ++n) {
              const uint32_t v = tw[n];
              d[n] = lds_u32(cb + static_cast<uint32_t>(KS_IDX(v >> 8, fv.n_rows * NC))) - __byte_perm(v, 0u, 0u);
            }
          } else {
            const uint2* tw = top.p.w + static_cast<size_t>(KS_IDX(ch * tpc + t, kFastTopPairs / (kTop > 0 ? kTop : 1))) * kTop;
#pragma unroll
            for (int n = 0; n < kTop; ++n)
              d[n] = lds_u32(cb + static_cast<uint32_t>(KS_IDX(tw[n].x, fv.n_rows * NC))) - tw[n].y;
          }
          uint32_t x = d[0] & 0x80808080u;  // path bits: level 0 in bit 7 of each byte, ...
          if (L >= 2) {
            const uint32_t s1 = byte_select(d[0], d[2], d[1]);
            x |= (s1 >> 1) & 0x40404040u;
            if (L >= 3) {
              const uint32_t sa = byte_select(s1, d[4], d[3]);
              const uint32_t sb = byte_select(s1, d[6], d[5]);
              const uint32_t s2 = byte_select(d[0], sb, sa);
              x |= (s2 >> 2) & 0x20202020u;
            }
          }
          // byte r of x holds candidate r's node index at level L in its top L bits (the rest
          // is zero), so x >> (6 - L) holds 4 * index in every byte
          const uint32_t y = x >> (6 - L);
          const uint32_t tbase = lvlL + (static_cast<uint32_t>(t) << (L + 2));
#pragma unroll
          for (int r = 0; r < 4; ++r) a[r] = tbase + __byte_perm(y, 0u, 0x4440u + r);
        }
        if (NP >= 0) {
#pragma unroll
          for (int l = 0; l < (NP >= 0 ? NP : 0); ++l)
#pragma unroll
            for (int r = 0; r < 4; ++r) a[r] = path_step(a[r], cb + r, k0, buf, tile0, tile_bytes);
        } else {
#pragma unroll 1
          for (int l = 0; l < np; ++l)
#pragma unroll
            for (int r = 0; r < 4; ++r) a[r] = path_step(a[r], cb + r, k0, buf, tile0, tile_bytes);
        }
#pragma unroll
        for (int r = 0; r < 4; ++r) {
#ifdef KS_DEBUG_BOUNDS
          a[r] = buf + 4u * static_cast<uint32_t>(KS_IDX((a[r] - buf) >> 2, fv.buf_bytes / 4));
#endif
          score[r] += lds_f32(a[r]);
        }
      }
      if (split) {
#pragma unroll
        for (int r = 0; r < 4; ++r) {
          sums[r] += __dsub_rn(__dadd_rn(static_cast<double>(score[r]), sl.grid), sl.grid);
          score[r] = 0.0f;
        }
      }
      // Release the buffer without a block-wide barrier: every warp of the group counts itself
      // out, and the last one to leave refills the buffer (nobody waits; warps may run a chunk ahead).
      __syncwarp();
      if (!kFloor && (tid & 31) == 0) {
        if (atomicAdd(&s_done[rb], 1) == THREADS / 32 / RG - 1) {
          s_done[rb] = 0;
          s_pending[rb] = 0;
          if (ch + kNBuf * RG < ch_end && !*v_fail) {
            fence_async_proxy();
            mbar_expect_tx(bar, fv.chunk_bytes + (starved() ? 16 : 0));
            bulk_copy_g2s(buf, reinterpret_cast<const char*>(fv.chunks) +
                                   static_cast<size_t>(KS_IDX(ch + kNBuf * RG, fv.n_chunks)) * fv.chunk_bytes,
                          fv.chunk_bytes, bar);
            s_pending[rb] = 1;
          }
        }
      }
    }
    __syncthreads();  // all walks are done: the buffers are free
    if (kFloor && tid < kNBuf * RG && !*v_fail) s_pending[tid] = 0;  // copied once, landed, never refilled
    if (*v_fail) {
      // The call has failed. Before this CTA gives its shared memory back, give the copies that
      // may still be in flight the time to land (bounded again); the test hook's copies land in
      // full although their barriers never complete, so there a short pause stands in for it.
      const auto let_land = [&](uint32_t bar, uint32_t parity, bool hooked) {
        if (!hooked) mbar_wait_bounded(bar, parity, fv.wait_limit, &s_abort /* stays 0 */);
        else
          for (int i = 0; i < 64; ++i) __nanosleep(kSleepNs);
      };
      if (word == 0 && grp % GPR == 0) {  // one thread per ring, for its ring's buffers (it knows their parities)
        for (int b = 0; b < kNBuf; ++b)
          if (s_pending[ring * kNBuf + b]) let_land(bar0 + 8u * (ring * kNBuf + b), (phases >> b) & 1u, starved());
        if (tile_late && ring == 0) let_land(bar0 + 8u * (kNBuf * RG), tile_phase ^ 1u, fv.starve == kStarveTiles);
      }
      __syncthreads();
      if (tid < k && partial) partial[(static_cast<size_t>(prob) * nblk + chunk) * k + tid] = 0ull;
      return;
    }

    // ---- phase C ---------------------------------------------------------------------------------
    // this thread's sum over the groups, in a fixed order; the buffers are idle now
    float total[4];
    if (split) {
      double* s_part = reinterpret_cast<double*>(smem + kOffBuf0);  // [G - 1][4][W]
      if (grp > 0) {
#pragma unroll
        for (int r = 0; r < 4; ++r) s_part[((grp - 1) * 4 + r) * W + word] = sums[r];
      }
      __syncthreads();
      if (grp == 0) {
#pragma unroll
        for (int r = 0; r < 4; ++r)
          for (int g = 1; g < G; ++g) sums[r] += s_part[((g - 1) * 4 + r) * W + word];
      }
      if (!whole) {
        // publish this part's sums, let the last arrival finish the block
        double2* to = reinterpret_cast<double2*>(sl.scores + (2 * static_cast<size_t>(cta) + (first_part ? 0 : 1)) * NC + 4 * word);
        if (grp == 0) {
          __stcg(to, make_double2(sums[0], sums[1]));
          __stcg(to + 1, make_double2(sums[2], sums[3]));
        }
        __threadfence();
        __syncthreads();
        if (tid == 0) {
          const int c0 = split_first(sl, item, grid), n = split_last(sl, item, grid) - c0 + 1;
          s_parts[0] = c0;
          s_parts[1] = n;
          s_parts[2] = split_start(sl, c0, grid) < item * sl.units ? 1 : 0;  // its last part
          s_last = atomicAdd(sl.words + c0, 1) == n - 1;
          if (s_last) sl.words[c0] = 0;  // nobody else touches this counter again in this launch
        }
        __syncthreads();
        if (!s_last) {
          ranked = false;
          continue;
        }
        __threadfence();
        if (grp == 0) {
          // parts 0 .. n - 1: the first CTA's first or last one, the others' first
          const double* from = sl.scores + 2 * static_cast<size_t>(s_parts[0]) * NC + 4 * word;
          const int n = s_parts[1], second = s_parts[2] * NC;
          sums[0] = sums[1] = sums[2] = sums[3] = 0.0;
          for (int q0 = 0; q0 < n; q0 += 4) {
            double2 u[4], v[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              const double2* p2 = reinterpret_cast<const double2*>(from + 2 * static_cast<size_t>(q0 + q) * NC + (q0 + q == 0 ? second : 0));
              u[q] = q0 + q < n ? __ldcg(p2) : make_double2(0.0, 0.0);
              v[q] = q0 + q < n ? __ldcg(p2 + 1) : make_double2(0.0, 0.0);
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              sums[0] += u[q].x; sums[1] += u[q].y; sums[2] += v[q].x; sums[3] += v[q].y;
            }
          }
        }
      }
#pragma unroll
      for (int r = 0; r < 4; ++r) total[r] = static_cast<float>(sums[r]);
    } else {
      float* s_part = reinterpret_cast<float*>(smem + kOffBuf0);  // [G - 1][4][W]
      if (grp > 0) {
#pragma unroll
        for (int r = 0; r < 4; ++r) s_part[((grp - 1) * 4 + r) * W + word] = score[r];
      }
      __syncthreads();
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        total[r] = score[r];
        if (grp == 0)
          for (int g = 1; g < G; ++g) total[r] += s_part[((g - 1) * 4 + r) * W + word];
      }
    }
    if (sl.score_out) {
      // scoring call: the scores are the result (same order of additions as the ranking path)
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        const int64_t row = start + 4 * word + r;
        if (grp == 0 && row < stop) sl.score_out[lo + row] = (fv.base + total[r]) + 0.0f;
      }
      continue;
    }
    unsigned long long keys[5];
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      keys[r] = 0ull;
      // byte r of word `word` is row 4 word + r of the block
      const int64_t row = start + 4 * word + r;
      if (grp == 0 && row < stop) {
        keys[r] = make_key((fv.base + total[r]) + 0.0f, seg_idx ? seg_idx[lo_idx + row] : static_cast<int>(row));
      }
    }
    keys[4] = tid < k ? s_list[tid] : 0ull;
    __syncthreads();
    block_topk<5>(keys, k, s_warp, s_list);
  }
  if (!ranked) continue;
  if (tid < k)
    partial[KS_IDX((static_cast<size_t>(prob) * nblk + chunk) * k + tid, static_cast<size_t>(P) * nblk * k)] = s_list[tid];
  if (sl.out_idx) {
    // single-problem form: the last block to finish merges the per-block lists
    __threadfence();
    __syncthreads();
    if (tid == 0) s_last = atomicAdd(sl.words + kMaxShares, 1) == nblk - 1;
    __syncthreads();
    if (!s_last) continue;
    __threadfence();
    // the whole CTA ranks the nblk * k keys (each key is read once)
    const int n_keys = nblk * k;
    __syncthreads();
    if (tid < KS_MAX_K) s_list[tid] = 0ull;
    for (int base = 0; base < n_keys; base += 2 * THREADS) {
      unsigned long long keys[3];
      keys[0] = base + tid < n_keys ? __ldcg(partial + base + tid) : 0ull;
      keys[1] = base + THREADS + tid < n_keys ? __ldcg(partial + base + THREADS + tid) : 0ull;
      __syncthreads();
      keys[2] = tid < k ? s_list[tid] : 0ull;
      __syncthreads();
      block_topk<3>(keys, k, s_warp, s_list);
    }
    if (tid < k) {
      sl.out_idx[tid] = key_index(s_list[tid]);
      sl.out_score[tid] = key_score(s_list[tid]);
      __threadfence_system();
    }
    __syncthreads();
    if (tid == 0) {
      sl.words[kMaxShares] = 0;
      if (sl.out_seq) {  // the results are in place: tell the host, which polls this word
        __threadfence_system();
        *reinterpret_cast<volatile int*>(sl.out_seq) = sl.seq;
      }
    }
  }
  }  // items
}

}  // namespace

// ------------------------------------------------------------------------------------------
// host: repack
// ------------------------------------------------------------------------------------------

// The orderings of L levels used by rank rows (lowest rank first).
static const int* partition_perm(int L, int q) {
  static const int p2[1][4] = {{0, 1, 0, 0}};
  static const int p3[2][4] = {{0, 1, 2, 0}, {0, 2, 1, 0}};
  static const int p4[3][4] = {{0, 1, 2, 3}, {1, 3, 0, 2}, {1, 2, 0, 3}};
  return L == 2 ? p2[q] : (L == 3 ? p3[q] : p4[q]);
}
// How a membership mask is tested: levels of rank >= cut in ordering `perm` go right, or, with
// `swap`, go left (the mask is the complement of that upper set).
struct PartitionCode {
  int perm, cut;
  bool swap;
};
static std::vector<PartitionCode> partition_codes(int L) {
  const int n_perm = L == 2 ? 1 : (L == 3 ? 2 : 3);
  const uint32_t full = (1u << L) - 1;
  std::vector<PartitionCode> code(full + 1, PartitionCode{-1, 0, false});
  for (int q = 0; q < n_perm; ++q)
    for (int c = 1; c < L; ++c) {
      uint32_t up = 0;
      for (int r = c; r < L; ++r) up |= 1u << partition_perm(L, q)[r];
      if (code[up].perm < 0) code[up] = PartitionCode{q, c, false};
      if (code[full ^ up].perm < 0) code[full ^ up] = PartitionCode{q, c, true};
    }
  return code;
}

// Tile geometry by the number of rows: the [row][candidate] tile and the two chunk buffers have to
// fit the shared memory of one SM (228 KiB, 1 KiB of it reserved per CTA; a CTA's own limit is
// 227 KiB including its static part). What was measured to matter on one ensemble: (i) four trees
// or more per thread and chunk, which the compiler interleaves (13 %); (ii) up to 128 registers
// per thread - the 64-register forms (two CTAs of 512 threads) ran 54 to 63 ms on the same
// ensemble depending on how unrelated code around the loop happened to be compiled, and one CTA
// of 512 threads gained 15 % from the larger budget; (iii) two CTAs per SM, so that one CTA's
// tile fill and ranking overlap the other's walk, when the tile leaves room for them; sixteen
// walking warps per SM saturate the walk, eight do not. Hence, in order of preference: two CTAs
// of 256 threads x 1,024 candidates (eight trees per thread and chunk; up to 74 rows); one CTA of
// 512 threads x 1,024 candidates with 32 KB chunk buffers (eight trees per thread and chunk; up
// to 156 rows); two CTAs of 256 threads x 512 candidates; one CTA of 512 threads x 1,024
// candidates with 16 KB buffers (up to 188 rows) or x 512 candidates (up to 376 rows). Every CTA
// streams the whole ensemble, so a halved block doubles that traffic (two CTAs of 256 threads x
// 256 candidates measured slower than one CTA of 512 x 512; two CTAs of 128 x 512 and one CTA of
// 256 x 1,024 have too few warps). More rows than 376: the general kernel.
// KS_FAST_GEOMETRY="threads,candidates,buffer KiB" overrides the choice (a tuning aid; a geometry
// that does not fit is refused). With buffers of 8 KB more rows fit than the kernels that build tiles
// in front of the walk can stage thresholds for (kTileMaxThr): such an ensemble takes the general kernel.
struct Geometry {
  int threads, cands, buf_bytes, ctas_per_sm;
};
static size_t geometry_smem(const Geometry& g, int n_rows) {
  // static shared memory of the kernel, with slack (the one-CTA forms keep a class per candidate)
  const size_t stat = 2560 + static_cast<size_t>(g.threads) / 32 * KS_MAX_K * 8 + 256 + (g.threads > 256 && g.cands == 1024 ? 4 * g.cands : 0);
  return static_cast<size_t>(kNBuf) * g.buf_bytes + static_cast<size_t>(n_rows) * g.cands + stat;
}
static bool geometry_fits(const Geometry& g, int n_rows) {
  const size_t per_cta = geometry_smem(g, n_rows);
  if (per_cta > 227 * 1024) return false;
  return g.ctas_per_sm * (per_cta + 1024) <= 228 * 1024;
}
static bool geometry_known(int t, int c) {
  return (t == 512 && c == 1024) || (t == 256 && c == 512) || (t == 512 && c == 512) || (t == 256 && c == 1024);
}
static bool pick_geometry(int n_rows, Geometry* out) {
  if (const char* env = std::getenv("KS_FAST_GEOMETRY")) {
    int t = 0, c = 0, kb = 0;
    if (std::sscanf(env, "%d,%d,%d", &t, &c, &kb) == 3 && geometry_known(t, c) && kb >= 8 && kb <= 64) {
      Geometry g{t, c, kb * 1024, 2};
      if (!geometry_fits(g, n_rows)) g.ctas_per_sm = 1;
      if (geometry_fits(g, n_rows)) {
        *out = g;
        return true;
      }
    }
  }
  const Geometry order[] = {{256, 1024, kBufBytes, 2},     {512, 1024, 2 * kBufBytes, 1}, {256, 512, kBufBytes, 2},
                            {512, 1024, kBufBytes, 1},     {512, 512, 2 * kBufBytes, 1},  {512, 512, kBufBytes, 1}};
  for (const Geometry& g : order)
    if (geometry_fits(g, n_rows)) {
      *out = g;
      return true;
    }
  return false;
}

// What rounds a chunk's sum to a multiple of u, a power of two of which no sum of one leaf a tree has more than
// 2^51: 1.5 * 2^52 u. Sums of such multiples are exact. The rounding, at most B 2^-52 with B the sum of the trees' largest
// leaves, is none where every leaf is a multiple of u already; it is far below the last bit of any float score where the
// leaves are of one scale (`even`: fixed_point_shift's B <= 200 V, so at most V 2^-44 a chunk where a float holds V to
// 2^-25). Else 0.
static double sum_grid(int n_trees, const int64_t* off, const ks_node_host* nodes, bool even) {
  double largest = 0.0;
  int low = INT_MAX, e = 0;  // exponent of the lowest bit of any leaf
  for (int t = 0; t < n_trees; ++t) {
    float top = 0.0f;
    for (int64_t i = off[t]; i < off[t + 1]; ++i) {
      const float v = std::fabs(nodes[i].thr_or_leaf);
      if (nodes[i].feat != 0xFFFF || v == 0.0f) continue;
      top = std::max(top, v);
      uint32_t bits;  // (by its bits: frexp and ldexp for every leaf took 2.2 ms of 500 trees of depth 8, this 0.1)
      std::memcpy(&bits, &v, 4);
      const int exponent = static_cast<int>(bits >> 23);  // 0: subnormal
      const uint32_t digits = (bits & 0x7FFFFFu) | (exponent ? 0x800000u : 0u);
      low = std::min(low, std::max(exponent, 1) - 150 + __builtin_ctz(digits));
    }
    largest += top;
  }
  std::frexp(1.001 * largest, &e);  // (< 2^e; a chunk's float sum rounds up by less than a thousandth)
  return even || low >= e - 51 ? std::ldexp(1.5, e + 1) : 0.0;
}

cudaError_t build_fast_gbdt(GbdtModel& m, int n_trees, const int64_t* off, const ks_node_host* nodes) {
  m.fast = false;
  if (n_trees < 1 || m.max_depth < 1 || m.max_depth > kFastMaxDepth) return cudaSuccess;
  const int D = m.max_depth;
  // distinct thresholds per feature, sliced into rows of at most 127
  std::vector<std::vector<float>> thr(KS_F);
  // Partition splits: "level in S goes right" becomes a bin comparison on a rank row. A rank row
  // orders the field's levels by one of a few fixed permutations; S (or its complement, with the
  // node's children exchanged) is then the set of levels of rank >= c for some c, i.e. the
  // ordinary test "bin <= c - 1 goes left". The permutations below reach every proper subset of
  // 2, 3 and 4 levels up to complement.
  std::vector<std::vector<PartitionCode>> part(KS_F);  // per feature: code of every mask
  bool perm_used[KS_F][3] = {};
  for (int64_t i = 0; i < off[n_trees]; ++i) {
    const ks_node_host& nd = nodes[i];
    if (nd.feat == 0xFFFF) continue;
    if (nd.kind == KS_NODE_PARTITION) {
      const int L = categorical_levels(nd.feat);
      if (L == 0) return cudaSuccess;
      if (part[nd.feat].empty()) part[nd.feat] = partition_codes(L);
      uint32_t mask;
      std::memcpy(&mask, &nd.thr_or_leaf, 4);
      if (mask == 0 || mask >= (1u << L)) return cudaSuccess;
      if (mask != (1u << L) - 1) perm_used[nd.feat][part[nd.feat][mask].perm] = true;
    } else {
      thr[nd.feat].push_back(nd.thr_or_leaf);
    }
  }
  FeatQ fq[64];
  std::memset(fq, 0, sizeof(fq));
  int rank_row[KS_F][3];  // row offset (within the feature's rows) of each permutation in use
  int n_rows = 0, n_class[3] = {0, 0, 0}, thr_class[3] = {0, 0, 0};
  for (int f = 0; f < KS_F; ++f) {
    auto& v = thr[f];
    std::sort(v.begin(), v.end());
    v.erase(std::unique(v.begin(), v.end()), v.end());
    if (v.size() > 65000) return cudaSuccess;
    const int n_slices = static_cast<int>((v.size() + kSlice - 1) / kSlice);
    int cnt = n_slices, n_rank = 0;
    for (int q = 0; q < 3; ++q) {
      rank_row[f][q] = perm_used[f][q] ? cnt++ : -1;
      if (perm_used[f][q]) {
        const int L = categorical_levels(f);
        for (int r = 0; r < L; ++r) fq[f].rank[n_rank][partition_perm(L, q)[r]] = static_cast<uint8_t>(r);
        ++n_rank;
      }
    }
    fq[f].nthr = static_cast<uint16_t>(v.size());
    fq[f].nslice = static_cast<uint16_t>(n_slices);
    fq[f].nrank = static_cast<uint16_t>(n_rank);
    n_class[feat_class(f)] += cnt;
    thr_class[feat_class(f)] += static_cast<int>(v.size());
    n_rows += cnt;
  }
  Geometry geom{};
  if (n_rows == 0 || !pick_geometry(n_rows, &geom)) return cudaSuccess;  // generic path
  if (thr_class[0] + thr_class[1] + thr_class[2] > kTileMaxThr) return cudaSuccess;
  if (n_class[0] > kFastMaxProbRows || n_class[1] > kFastMaxCandRec) return cudaSuccess;
  const int NC = geom.cands, threads = geom.threads;
  // rows and thresholds ordered: per-pair, candidate-only, problem-only features
  std::vector<float> table;
  int next = 0;
  for (int cls : {2, 1, 0}) {
    for (int f = 0; f < KS_F; ++f) {
      if (feat_class(f) != cls) continue;
      fq[f].row0 = static_cast<uint16_t>(next);
      fq[f].thr0 = static_cast<uint32_t>(table.size());
      table.insert(table.end(), thr[f].begin(), thr[f].end());
      next += fq[f].nslice + fq[f].nrank;
    }
  }
  if (table.empty()) table.push_back(0.0f);
  const int G = threads / (NC / 4);
  const int per_tree_words = (2 << D) - 1;
  // A chunk is what one ring's buffer holds (the geometry's buffer size is shared out among the
  // rings); ring r takes the chunks r, r + rings, ..., and the groups of a ring split a chunk's trees.
  const int rings = ring_count(G), gpr = G / rings;
  const int group_buf = geom.buf_bytes / rings / 16 * 16;
  int tpc = group_buf / (per_tree_words * 4) / gpr * gpr;
  if (tpc < gpr) return cudaSuccess;
  // At least sixteen chunks a ring, so that a split walk's units are not coarse, but no fewer than eight trees a thread, which
  // hide a chunk's beginning and end (100 trees of depth 6 in chunks of 32: 64 x 2,048 from host memory 122 us, of 8 112).
  // A multiple of four a thread, by which the walk is unrolled, and no more padding than the top levels' constants have
  // room for (500 trees of depth 6, 128 slots, in chunks of 31, 527 with the padding, whose constants take the compact form:
  // 31 x 62,000 2,070 us and 300 x 3,900 1,231; in chunks of 28 1,434 and 987).
  const auto top_form = [&](int t) {
    const int64_t pairs = static_cast<int64_t>((n_trees + t - 1) / t) * t * 7;
    return pairs <= kFastTopPairs ? 2 : pairs <= 2 * kFastTopPairs ? 1 : 0;
  };
  for (int t = std::max(8, n_trees / (16 * rings) / 4 * 4); t >= 8; t -= 4)
    if (t * gpr < tpc && top_form(t * gpr) >= top_form(tpc)) {
      tpc = t * gpr;
      break;
    }
  if (tpc > (n_trees + G - 1) / G * gpr) tpc = (n_trees + G - 1) / G * gpr;  // a small ensemble: one short chunk per ring
  const int n_chunks = (n_trees + tpc - 1) / tpc;
  const int chunk_words = (tpc * per_tree_words + 3) / 4 * 4;  // bulk copies move multiples of 16 bytes
  if (chunk_words * 4 > group_buf) return cudaSuccess;
  int L = D < 3 ? D : 3;  // levels whose nodes travel as kernel-parameter constants
  while (L > 0 && static_cast<int64_t>(n_chunks) * tpc * ((1 << L) - 1) > kFastTopPairs) --L;
  // three levels in the compact form (one word per node) when the pair form would leave fewer
  bool compact = false;
  if (L < 3 && D >= 3 && static_cast<int64_t>(n_chunks) * tpc * 7 <= 2 * kFastTopPairs) {
    L = 3;
    compact = true;
  }
  const int n_top = (1 << L) - 1;
  std::vector<uint32_t> chunks(static_cast<size_t>(n_chunks) * chunk_words);
  FastTopParams* top = new (std::nothrow) FastTopParams();
  if (!top) return cudaErrorMemoryAllocation;
  m.h_top = top;  // (freed with the model)
  const uint32_t always_left = 0xFFu;  // row 0, threshold 127: no byte (0x80 | bin) exceeds 0xFF
  for (int ch = 0; ch < n_chunks; ++ch) {
    uint32_t* base = chunks.data() + static_cast<size_t>(ch) * chunk_words;
    float* leaves = reinterpret_cast<float*>(base + tpc * ((1 << D) - 1));
    for (int tt = 0; tt < tpc; ++tt) {
      const int t = ch * tpc + tt;
      std::vector<int> src(1, t < n_trees ? 0 : -1);
      std::vector<float> carry(1, 0.0f);  // leaf value carried below an original leaf
      for (int l = 0; l < D; ++l) {
        uint32_t* lvl = base;
        for (int q = 0; q < l; ++q) lvl += tpc << q;
        std::vector<int> nsrc(2 << l);
        std::vector<float> ncarry(2 << l);
        for (int i = 0; i < (1 << l); ++i) {
          uint32_t word = always_left;
          uint2 tw = make_uint2(0u, 128u * 0x01010101u);
          int ls = -1, rs = -1;
          float lc = carry[i], rc = carry[i];
          if (src[i] >= 0) {
            const ks_node_host& nd = nodes[off[t] + src[i]];
            if (nd.feat == 0xFFFF) {
              lc = rc = nd.thr_or_leaf;
            } else {
              uint32_t row, jl;
              bool swap = false, always_right = false;
              if (nd.kind == KS_NODE_PARTITION) {
                uint32_t mask;
                std::memcpy(&mask, &nd.thr_or_leaf, 4);
                if (mask == (1u << categorical_levels(nd.feat)) - 1) {
                  always_right = true;  // every level is a member
                  row = 0;
                  jl = 127;
                } else {
                  const PartitionCode pc = part[nd.feat][mask];
                  row = fq[nd.feat].row0 + rank_row[nd.feat][pc.perm];
                  jl = pc.cut - 1;
                  swap = pc.swap;
                }
              } else {
                const auto& v = thr[nd.feat];
                const int j = static_cast<int>(std::lower_bound(v.begin(), v.end(), nd.thr_or_leaf) - v.begin());
                row = fq[nd.feat].row0 + j / kSlice;
                jl = j % kSlice;
              }
              ls = nd.left;
              rs = nd.left + 1;
              if (always_right) {
                ls = rs;  // the walk always goes left here: put the right subtree on both sides
              } else {
                word = (row * NC) << 8 | (0x80u | jl);
                tw = make_uint2(row * NC, (jl + 1) * 0x01010101u);
                if (swap) std::swap(ls, rs);
              }
            }
          }
          lvl[tt * (1 << l) + i] = word;
          if (l < L) {
            const size_t at = static_cast<size_t>(t) * n_top + ((1 << l) - 1) + i;
            if (compact) reinterpret_cast<uint32_t*>(top->w)[at] = (tw.x << 8) | (tw.y & 0xFFu);
            else top->w[at] = tw;
          }
          nsrc[2 * i] = ls;
          nsrc[2 * i + 1] = rs;
          ncarry[2 * i] = lc;
          ncarry[2 * i + 1] = rc;
        }
        src.swap(nsrc);
        carry.swap(ncarry);
      }
      for (int i = 0; i < (1 << D); ++i) {
        float v = carry[i];
        if (src[i] >= 0) v = nodes[off[t] + src[i]].thr_or_leaf;
        leaves[tt * (1 << D) + i] = v;
      }
    }
  }
  cudaError_t e = cudaMalloc(reinterpret_cast<void**>(&m.d_qnodes), chunks.size() * 4);
  if (e == cudaSuccess) e = cudaMemcpy(m.d_qnodes, chunks.data(), chunks.size() * 4, cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMalloc(reinterpret_cast<void**>(&m.d_qthr), table.size() * 4);
  if (e == cudaSuccess) e = cudaMemcpy(m.d_qthr, table.data(), table.size() * 4, cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMalloc(reinterpret_cast<void**>(&m.d_qfeat), sizeof(fq));
  if (e == cudaSuccess) e = cudaMemcpy(m.d_qfeat, fq, sizeof(fq), cudaMemcpyHostToDevice);
  if (e != cudaSuccess) return e;
  m.fixed_shift = fixed_point_shift(n_trees, off, nodes);
  m.sum_grid = sum_grid(n_trees, off, nodes, m.fixed_shift != kNoFixed);
  m.class_words = class_tree_words(n_trees, off, nodes);
  m.top_levels = L;
  m.top_compact = compact;
  m.fast = true;
  m.fast_depth = D;
  m.fast_threads = threads;
  m.block_cands = NC;
  m.buf_bytes = group_buf;
  m.ctas_per_sm = geom.ctas_per_sm;
  m.n_qrows = n_rows;
  m.n_pair_rows = n_class[2];
  m.n_cand_rows = n_class[1];
  m.n_prob_rows = n_class[0];
  m.n_qthr = thr_class[0] + thr_class[1] + thr_class[2];
  m.thr_cand0 = thr_class[2];
  m.thr_prob0 = thr_class[2] + thr_class[1];
  m.tpc = tpc;
  m.n_chunks = n_chunks;
  m.chunk_bytes = chunk_words * 4;
  return cudaSuccess;
}

void free_fast_gbdt(GbdtModel& m) {
  delete m.h_top;
  m.h_top = nullptr;
}

// ------------------------------------------------------------------------------------------
// launcher
// ------------------------------------------------------------------------------------------

// Blocks per problem: full tiles of the model's block size. A block's cost does not depend on how
// many of its slots are live, so an under-filled machine is filled by splitting the trees over
// several CTAs per block (split walk) rather than by shorter blocks.
void fast_tiling(const GbdtModel& g, int P, int64_t per_problem, int* nblk, int* rows_per_cta) {
  int64_t n = (per_problem + g.block_cands - 1) / g.block_cands;
  if (n < 1) n = 1;
  (void)P;
  *nblk = static_cast<int>(n);
  *rows_per_cta = g.block_cands;
}

size_t fast_tiles_bytes(const GbdtModel& g, int P, int nblk) {
  return reinterpret_cast<size_t>(pair_tiles(g, P, nblk, nullptr).prob) + static_cast<size_t>(P) * kProbRec;
}

size_t fast_scratch_bytes(const GbdtModel& g, int C) {
  return 256 + static_cast<size_t>(kCombos) * C * cand_rec_bytes(g);
}

// Memo of the per-pair rows (see MemoView): for every dense batch that is not split (a split walk takes whole
// tiles, see tile_pairs_kernel) and for segmented batches of 32 problems or more. (Dense batches of 3 to 31 problems come here from
// 1,924 blocks on: 16 x 150,000 grid candidates, 500 trees, 2,802 us without records, 2,240 with; 50 trees 760 and 469.) The
// table is held for at most `fast_memo_batch` problems at a time (512 MiB of
// records); a larger call is served batch by batch. 0 = not used.
size_t memo_fixed_bytes(int C) {
  return static_cast<size_t>(kMemoCombos) * kMemoCap * (sizeof(unsigned long long) + 2 * sizeof(int)) + 256 +
         (static_cast<size_t>(kMemoCombos) * C * sizeof(unsigned) + 255) / 256 * 256;
}
MemoView memo_view(void* mem, int C) {
  char* m = static_cast<char*>(mem);
  const size_t slots = static_cast<size_t>(kMemoCombos) * kMemoCap;
  MemoView v{};
  v.keys = reinterpret_cast<unsigned long long*>(m);
  v.count = reinterpret_cast<int*>(m + slots * sizeof(unsigned long long));
  v.dense = reinterpret_cast<int*>(m + slots * sizeof(unsigned long long) + 256);
  v.reps = v.dense + slots;
  v.cls = reinterpret_cast<unsigned*>(v.reps + slots);
  v.tab = m + memo_fixed_bytes(C);
  return v;
}
cudaError_t memo_clear(const MemoView& memo, cudaStream_t stream) {
  // (the counts lie behind the keys)
  return cudaMemsetAsync(memo.keys, 0, static_cast<size_t>(kMemoCombos) * (kMemoCap * sizeof(unsigned long long) + sizeof(int)), stream);
}
cudaError_t memo_compact(const MemoView& memo, cudaStream_t stream) {
  memo_compact_kernel<<<dim3(kMemoCap / 256, kMemoCombos), 256, 0, stream>>>(memo);
  return cudaGetLastError();
}

int fast_memo_batch(const GbdtModel& g, int P, bool segmented, bool lean) {
  if (P < (segmented || lean ? kMemoMinProblems : kMemoMinDense) || g.n_pair_rows < 1 || g.n_pair_rows > kFastMaxPairRec) return 0;
  const size_t per_problem = static_cast<size_t>(kMemoCap) * pair_rec_bytes(g);
  int64_t batch = static_cast<int64_t>(kMemoTableBytes / per_problem);
  if (batch < kMemoMinProblems) batch = kMemoMinProblems;
  if (lean) batch = kMemoMinProblems / 2;
  return static_cast<int>(batch < P ? batch : P);
}

size_t fast_memo_bytes(const GbdtModel& g, int P, int C, bool segmented, bool lean) {
  const int batch = fast_memo_batch(g, P, segmented, lean);
  if (batch == 0 || C < 1) return 0;
  return memo_fixed_bytes(C) + static_cast<size_t>(batch) * (static_cast<size_t>(kMemoCap) * pair_rec_bytes(g) + kProbRec);
}

// Copying a tile takes 2 to 3 us, where a tree of eight levels takes a block of 1,024 candidates 0.25 us.
constexpr int kFillCopy = 10;

// A split walk of `blocks` candidate blocks: the line of
// trees (see SplitArgs) and the CTAs that share it, one for every place of the machine unless a stretch
// would be shorter than a tile and a unit. Returns the CTAs; without units, whole blocks do as well.
// Measured: 61,140 candidates x 500 trees (60 blocks, one CTA an SM) on 120 CTAs in equal slices 79 us, on 148 by
// stretches 68; 96,000 candidates (94 blocks), 282 CTAs in two rounds 114, now 84; a million given rows (977
// blocks, 6.6 rounds) 930, now 896.
static int split_plan(const GbdtModel& g, int64_t blocks, SplitArgs* s) {
  const int fill = kFillCopy;
  const int rings = ring_count(g.fast_threads / (g.block_cands / 4));
  s->units = (g.n_chunks + rings - 1) / rings;
  s->unit = rings * g.tpc;
  s->fill = fill;
  s->blocks = static_cast<int>(blocks);
  const auto deal = [&](int64_t ctas) {
    const int64_t total = blocks * split_block(*s);
    s->step = static_cast<int>(total / ctas);
    s->rest = static_cast<int>(total % ctas);
    return static_cast<int>(ctas);
  };
  const int64_t len = split_block(*s), slots = static_cast<int64_t>(g.ctas_per_sm) * kSmCount;
  // Whole rounds that are nearly full are left as they are (293 blocks of 300,000 given rows: split 4 % slower).
  const int64_t rounds = (blocks + slots - 1) / slots;
  if (rounds > 1 && 20 * blocks >= 19 * rounds * slots) {
    s->units = 0;
    return 0;
  }
  // The last CTA of a block reads all its parts, 0.1 us each: 32 at most (one block of 1,000 trees: 125 parts 93 us the
  // whole call, 32 parts 80).
  constexpr int64_t kParts = 32;
  const int64_t most = std::max<int64_t>(1, std::min({blocks * len / (fill + s->unit), slots, kParts * blocks}));
  // Stretches that end where blocks do spare the second tile and the second part of most CTAs (some 4 us):
  // an equal number of CTAs a block, where that keeps nearly all of them busy, or where the sums ask for it.
  s->grid = g.sum_grid;
  const int64_t each = std::min<int64_t>({slots / blocks, s->units, kParts});
  if (each >= 1) {
    const int64_t aligned = (s->units + each - 1) / each * s->unit;
    const int64_t shared = (blocks * len / most - fill + s->unit - 1) / s->unit * s->unit + fill + 16;
    if (aligned <= shared || g.sum_grid == 0.0) {
      s->fill = 0;
      return deal(blocks * each);
    }
  }
  if (g.sum_grid == 0.0) {
    s->units = 0;
    return 0;
  }
  return deal(most);
}
// Whether a dense walk of so many blocks is split: where whole blocks would leave part of the machine idle,
// in the only round of CTAs or in the last of a few. Measured against whole blocks that fill their tiles in
// the walk (500 trees, 256 bins): 7 problems x 61,140 valid candidates (420 blocks) 533 -> 455 us, 31 x 61,140 (1,860) 2,117 ->
// 1,900, 64 x 9,000 grid candidates (576) 695 -> 595. From 32 problems on a catalogue in similarity order with class
// records is the alternative: 100 x 9,000 (900 blocks) 1,110 -> 934, 32 x 60,000 (1,888) 1,879 -> 1,959. Which of the two wins up
// to eight rounds was measured at 50, 200, 500 and 1,000 trees of depth 6 to 8 under the three laws: split walks, on grid pools 0.51
// to 0.99 of the time with records (full rounds of 592 and 888 blocks 1.01 to 1.02), on the valid pool, whose classes hold
// few members, 0.28 to 0.85; only 500 trees of depth 8 with a threshold of its own at every node lose at 1,152 grid blocks
// (1,215 -> 1,281 us; 1,855 -> 1,254 at the same size on the valid pool). A problem looks through those
// before it for its type combination, so there may not be very many. A single call of more blocks than the machine
// holds at once keeps whole blocks (310,000 candidates, 500 trees 610 us): its tiles would be 43 MB and more of workspace.
constexpr int kSplitBlocks = 13 * kSmCount, kSplitBlocksMemo = 8 * kSmCount, kSplitProblems = 512;
static bool split_fits(const GbdtModel& g, int64_t blocks) {  // (a line of trees is counted in 32 bits)
  return blocks * (static_cast<int64_t>(g.n_chunks + 2) * g.tpc + 64) < int64_t{1} << 30;
}
bool fast_splits(const GbdtModel& g, int P, int nblk, bool one_round) {
  const int64_t blocks = static_cast<int64_t>(P) * nblk;
  one_round |= g.sum_grid == 0.0;  // (blocks that are all cut alike share one round of CTAs)
  return split_fits(g, blocks) && P >= 1 && P <= kSplitProblems && blocks < (one_round ? g.ctas_per_sm * kSmCount : P < kMemoMinProblems ? kSplitBlocks : kSplitBlocksMemo) && g.n_chunks > ring_count(g.fast_threads / (g.block_cands / 4));
}
size_t fast_split_bytes(const GbdtModel& g) { return sizeof(double) * 2 * 2 * kSmCount * g.block_cands; }
static_assert(2 * kSmCount <= kMaxShares, "an arrival counter for every CTA");

// A prepared catalogue: the candidate-only rows of its tiles for every type combination, and a call's scratch.
size_t fast_prepared_rows_bytes(const GbdtModel& g, int nblk) {
  return (static_cast<size_t>(kCombos) * nblk * g.n_cand_rows * g.block_cands + 255) / 256 * 256;
}
size_t fast_prepared_call_bytes(const GbdtModel& g, int nblk) {
  return (static_cast<size_t>(nblk) * g.n_pair_rows * g.block_cands + 255) / 256 * 256 + kProbRec;
}

namespace {

struct WalkArgs {
  ks_gpu_desc desc;
  const ks_problem* d_p;
  ks_problem pv;
  int uv;
  const ks_candidate* d_c;
  int P, C, nblk, rows_per_cta;
  const int64_t* seg_off;
  const int32_t* seg_idx;
  FastView fv;
  int k;
  unsigned long long* partial;
  int* status;
  SplitArgs sl;
  int split_ctas;  // of a split walk
  const FastTopParams* top;
  cudaStream_t stream;
  int dependent;  // launched right behind the kernel whose tables it reads
};

template <int L, int NP, bool kCompact, int THREADS, int NC, bool kSplit, bool kShared = false, bool kFloor = false>
cudaError_t launch_form(const WalkArgs& a) {
  const size_t smem = static_cast<size_t>(kNBuf) * ring_count(THREADS / (NC / 4)) * a.fv.buf_bytes +
                      static_cast<size_t>(a.fv.n_rows) * NC;
  auto kernel = &select_fast_kernel<L, NP, kCompact, THREADS, NC, kSplit, kShared, kFloor>;
  cudaError_t e = ensure_dynamic_smem(reinterpret_cast<const void*>(kernel), smem);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg{};
  // One CTA per item; or - batch form of the geometries that hold one CTA per SM - one CTA per SM, each
  // serving many items; or a split walk's CTAs. (Two persistent CTAs on an SM run in step, so that both fill
  // and rank at the same time and neither hides the other's: measured 6 % slower than one CTA per item.)
  const int64_t n_items = static_cast<int64_t>(a.P) * a.nblk;
  const bool persistent = THREADS > 256 && !a.sl.tiles;
  const int64_t slots = kSmCount;
  cfg.gridDim = dim3(static_cast<unsigned>(kSplit ? a.split_ctas : (persistent && n_items > slots ? slots : n_items)));
  cfg.blockDim = dim3(THREADS);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = a.stream;
  // behind a table kernel the grid is launched as its programmatic dependent: its CTAs may start
  // their set-up while that kernel still runs, and wait for it (griddepcontrol.wait) before they
  // read its tables
  cudaLaunchAttribute attr{};
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &attr;
  cfg.numAttrs = a.dependent ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kernel, a.desc, a.d_p, a.pv, a.uv, a.d_c, a.P, a.C, a.nblk, a.rows_per_cta,
                            a.seg_off, a.seg_idx, a.fv, a.k, a.partial, a.status, a.sl, static_cast<int>(n_items),
                            *reinterpret_cast<const TopArg<kShared>*>(a.top));
}

template <int L, int NP, bool kCompact, int THREADS, int NC>
cudaError_t launch_ln(const WalkArgs& a) {
  return launch_form<L, NP, kCompact, THREADS, NC, false>(a);
}

// Split walks take the top levels from the chunk where the launch would keep the GPU waiting, i.e. behind the tiles
// of few blocks (10 to 14 us): 500 candidates, 500 trees, prepared 46.5 -> 42 us, 60,000 95.5 -> 97.5. And where the
// parameters hold fewer than three levels of the ensemble.
bool takes_shared_top(const GbdtModel& g, const WalkArgs& a) {
  if (g.fast_depth < 3 || g.tpc % 4 != 0) return false;
  return g.top_levels < 3 || g.top_compact || (!a.sl.score_out && a.sl.blocks < 50);
}

// the instantiation for a model's top levels and depth, within one tile geometry
template <int THREADS, int NC>
cudaError_t launch_walk_geom(const GbdtModel& g, const WalkArgs& a) {
  const int L = g.top_levels, np = g.fast_depth - L;
  if (a.sl.units > 0) {
    if (takes_shared_top(g, a)) {
      if (g.fast_depth == 8) return launch_form<3, 5, false, THREADS, NC, true, true>(a);
      if (g.fast_depth == 7) return launch_form<3, 4, false, THREADS, NC, true, true>(a);
      if (g.fast_depth == 6) return launch_form<3, 3, false, THREADS, NC, true, true>(a);
      return launch_form<3, -1, false, THREADS, NC, true, true>(a);
    }
    if (L == 3 && !g.top_compact) {
      if (np == 5) return launch_form<3, 5, false, THREADS, NC, true>(a);
      if (np == 4) return launch_form<3, 4, false, THREADS, NC, true>(a);
      if (np == 3) return launch_form<3, 3, false, THREADS, NC, true>(a);
      return launch_form<3, -1, false, THREADS, NC, true>(a);
    }
    return launch_form<0, -1, false, THREADS, NC, true>(a);
  }
  if (g.top_compact) {
    if (np == 5) return launch_ln<3, 5, true, THREADS, NC>(a);
    if (np == 4) return launch_ln<3, 4, true, THREADS, NC>(a);
    return launch_ln<3, -1, true, THREADS, NC>(a);
  }
  if (L == 3 && np == 5) return launch_ln<3, 5, false, THREADS, NC>(a);
  if (THREADS == 512 && NC == 1024) {  // the shapes met so far only in small ensembles
    if (L == 2 && np == 6) return launch_ln<2, 6, false, 512, 1024>(a);
    if (L == 2 && np == 5) return launch_ln<2, 5, false, 512, 1024>(a);  // the paper-sized ensemble: 916 trees of depth 7
  }
  if (L == 3 && np == 4) return launch_ln<3, 4, false, THREADS, NC>(a);
  if (L == 3 && np == 3) return launch_ln<3, 3, false, THREADS, NC>(a);
  if (L == 3) return launch_ln<3, -1, false, THREADS, NC>(a);
  if (L == 2) return launch_ln<2, -1, false, THREADS, NC>(a);
  if (L == 1) return launch_ln<1, -1, false, THREADS, NC>(a);
  return launch_ln<0, -1, false, THREADS, NC>(a);
}

// The floor measurement exists for the two geometries and the ensemble shape of the benchmark's
// first configuration (three word-wise levels, five path levels, top constants as pairs).
cudaError_t launch_walk_floor(const GbdtModel& g, const WalkArgs& a) {
  if (g.top_compact || g.top_levels != 3 || g.fast_depth != 8 || g.block_cands != 1024 ||
      g.n_chunks < kNBuf * ring_count(g.fast_threads / 256))  // every ring needs its kNBuf resident chunks
    return cudaErrorNotSupported;
  if (g.fast_threads == 512) return launch_form<3, 5, false, 512, 1024, false, false, true>(a);
  return launch_form<3, 5, false, 256, 1024, false, false, true>(a);
}

cudaError_t launch_walk(const GbdtModel& g, const WalkArgs& a) {
  if (g.fast_threads == 512 && g.block_cands == 1024) return launch_walk_geom<512, 1024>(g, a);
  if (g.fast_threads == 512) return launch_walk_geom<512, 512>(g, a);
  if (g.block_cands == 512) return launch_walk_geom<256, 512>(g, a);
  return launch_walk_geom<256, 1024>(g, a);
}

// Dynamic shared memory for `count` staged thresholds: all of them when they fit, else none (the
// kernel then searches the global array). Returns the capacity in floats to pass to the kernel.
int staged_floats(int count, size_t* bytes) {
  constexpr int kCap = 48 * 1024;  // floats: 192 KB
  const int cap = count <= kCap ? (count > 0 ? count : 1) : 0;
  *bytes = static_cast<size_t>(cap > 0 ? cap : 1) * sizeof(float);
  return cap;
}

}  // namespace

// combo >= 0: only that type combination; else those of the mask, or all (null).
static cudaError_t launch_cand_rows(const ks_gpu_desc& desc, const GbdtModel& g, const ks_candidate* d_c, int C,
                                    const unsigned* d_mask, int combo, const FastView& fv, uint8_t* d_rows,
                                    const MemoView& memo, int* words, cudaStream_t stream, int64_t* launches) {
  const int count = g.thr_prob0 - g.thr_cand0, block = C < 8192 ? 64 : 256;
  const size_t own = static_cast<size_t>(block) * (cand_rec_bytes(g) + 4 + 4 * kCandCols);
  size_t thr = (static_cast<size_t>(count) + 3) / 4 * 16;
  int cap = count > 0 ? count : 1;
  if (thr + own > 200 * 1024) cap = 0, thr = 0;  // (the global array is searched in place)
  const size_t smem = std::max<size_t>(thr, 16) + own;
  auto kernel = block == 64 ? &cand_rows_kernel<64> : &cand_rows_kernel<256>;
  cudaError_t e = ensure_dynamic_smem(reinterpret_cast<const void*>(kernel), smem);
  if (e != cudaSuccess) return e;
  kernel<<<dim3(std::min((C + block - 1) / block, 2 * kSmCount), combo >= 0 ? 1 : kCombos), kCandThreads, smem, stream>>>(
      desc, d_c, C, d_mask, combo, fv, d_rows, memo, cap, words);
  ++*launches;
  return cudaGetLastError();
}

// The tile kernel in one of its forms, see there.
static cudaError_t launch_tile_pairs(const ks_gpu_desc& desc, const GbdtModel& g, const ks_problem* d_p, const ks_problem& pv, int uv,
                                     int P, const ks_candidate* d_c, int C, const int* order, int nblk, const PairTiles& tiles,
                                     int* words, cudaStream_t stream, int64_t* launches) {
  const size_t smem = sizeof(float) * (kTileCols * kTileRows + g.n_qthr);
  cudaError_t e = ensure_dynamic_smem(reinterpret_cast<const void*>(&tile_pairs_kernel), smem);
  if (e != cudaSuccess) return e;
  const int W = g.block_cands / 4, groups = nblk * (W / 32);
  const int resident = std::max<int>(1, std::min<int>(4, 226 * 1024 / (smem + 4096)));
  tile_pairs_kernel<<<std::min(P * groups, resident * kSmCount), 256, smem, stream>>>(
      desc, d_p, pv, uv, P, d_c, C, order, make_view(g, nullptr), W, groups, tiles, words);
  ++*launches;
  return cudaGetLastError();
}

// Prepared catalogue: the candidate-only rows of its tiles, in the catalogue's order, for every type combination,
// computed once for a (catalogue, model) pair.
cudaError_t fast_prepare(const ks_gpu_desc& desc, const GbdtModel& g, const ks_candidate* d_c, int C, int nblk, void* d_rows,
                         const int* order, cudaStream_t stream, int64_t* launches) {
  if (g.n_cand_rows == 0) return cudaSuccess;
  ks_problem any{};
  any.m = any.n = any.k = 1;
  return launch_tile_pairs(desc, g, nullptr, any, 1, kCombos, d_c, C, order, nblk, PairTiles{nullptr, static_cast<uint8_t*>(d_rows), nullptr},
                           nullptr, stream, launches);
}

// Problems per launch when a call is served in batches of at most `cap`. In the launch form
// with one CTA per SM every launch runs its items in rounds of kSmCount, and a last round that
// is nearly empty still takes a whole item's time; a batch a little below the cap can save a
// round per launch (4,096 problems x 32 blocks in batches of 226 instead of 227: 889 rounds
// instead of 903: 133.3 -> 130.7 ms). Picks the size within an eighth below the cap that needs
// the fewest rounds. (With two CTAs per SM, one per item, the hardware hands out the items and
// the same rule measured 0.6 % slower: not applied there.)
static int balanced_step(const GbdtModel& g, int P, int cap, int nblk) {
  if (P <= cap || g.ctas_per_sm != 1 || cap < 16) return cap;
  int best = cap;
  int64_t best_rounds = INT64_MAX;
  for (int n = cap; n >= cap - cap / 8; --n) {
    int64_t rounds = 0;
    for (int first = 0; first < P; first += n) {
      const int64_t items = static_cast<int64_t>(P - first < n ? P - first : n) * nblk;
      rounds += (items + kSmCount - 1) / kSmCount;
    }
    if (rounds < best_rounds) {
      best_rounds = rounds;
      best = n;
    }
  }
  return best;
}

cudaError_t launch_select_fast(const ks_gpu_desc& desc, const GbdtModel& g, const ks_problem* d_p,
                               const ks_problem* p_by_value, int P, const ks_candidate* d_c, int C,
                               int nblk, int rows_per_cta, const int64_t* seg_off, const int32_t* seg_idx,
                               int k, unsigned long long* partial, void* scratch, int* status,
                               cudaStream_t stream, int64_t* launches, cudaEvent_t ev_begin,
                               const FastSplit* split, void* memo_mem, const FastWait* wait,
                               const FastPrepared* prep, const int32_t* perm, const ClassCall* classes) {
  WalkArgs a{};
  a.desc = desc;
  if (p_by_value) a.pv = *p_by_value;
  a.uv = p_by_value != nullptr;
  a.d_c = d_c;
  a.C = C;
  a.nblk = nblk;
  a.rows_per_cta = rows_per_cta;
  a.seg_idx = seg_idx;
  a.k = k;
  a.status = status;
  a.top = g.h_top;
  a.stream = stream;
  FastView& fv = a.fv;
  fv = make_view(g, wait);
  unsigned* d_mask = static_cast<unsigned*>(scratch);
  uint8_t* d_rows = static_cast<uint8_t*>(scratch) + 256;
  fv.cand_rows = d_rows;
  if (!seg_off && perm) a.seg_idx = perm;  // dense form ranked in the given order of the catalogue
  MemoView memo{};
  int memo_batch = (memo_mem && !p_by_value && C > 0) ? fast_memo_batch(g, P, seg_off != nullptr, wait->lean) : 0;
  if (memo_batch > 0) memo = memo_view(memo_mem, C);
  // candidate-only rows for the type combinations in use
  cudaError_t e = cudaSuccess;
  const bool tiles_mode = !prep && split && split->tiles && !seg_off;
  if (!prep && !a.uv && !tiles_mode) {
    e = cudaMemsetAsync(d_mask, 0, sizeof(unsigned), stream);
    if (e != cudaSuccess) return e;
    combo_mask_kernel<<<P >= 4096 ? 16 : 1, 256, 0, stream>>>(d_p, P, d_mask);
    ++*launches;
  }
  // shared memory of the table kernel: the per-pair thresholds when they fit beside its 256 records
  size_t pthr_bytes = 0;
  int pthr_cap = staged_floats(g.thr_cand0, &pthr_bytes);
  {
    const size_t rec_bytes = static_cast<size_t>(256) * pair_rec_bytes(g);
    size_t thr_part = pthr_cap > 0 ? static_cast<size_t>((pthr_cap + 3) / 4 * 4) * sizeof(float) : 0;
    if (thr_part + rec_bytes > 200 * 1024) {
      pthr_cap = 0;
      thr_part = 0;
    }
    pthr_bytes = thr_part + rec_bytes + 16;
  }
  if (prep) {
    const PairTiles tiles{prep->call, nullptr, prep->call + fast_prepared_call_bytes(g, nblk) - kProbRec};
    e = launch_tile_pairs(desc, g, d_p, a.pv, a.uv, P, d_c, C, perm, nblk, tiles, wait->words, stream, launches);
    if (e != cudaSuccess) return e;
    fv.prob_tab = tiles.prob;
    a.sl.cand_tiles = prep->cand_rows;
  } else if (tiles_mode) {
    const PairTiles tiles = pair_tiles(g, P, nblk, split->tiles);
    if (C > 0) {
      e = launch_tile_pairs(desc, g, d_p, a.pv, a.uv, P, d_c, C, nullptr, nblk, tiles, wait->words, stream, launches);
    } else {  // (nobody is ranked: any bytes with the top bit, and an index in range)
      e = cudaMemsetAsync(split->tiles, 0x80, tiles.prob - split->tiles, stream);
      if (e == cudaSuccess) e = cudaMemsetAsync(tiles.prob, 0, static_cast<size_t>(P) * kProbRec, stream);
    }
    if (e != cudaSuccess) return e;
    fv.prob_tab = tiles.prob;
    a.sl.cand_tiles = tiles.cand;
  } else if (C > 0) {
    if (memo.keys) {
      e = memo_clear(memo, stream);
      if (e != cudaSuccess) return e;
    }
    e = launch_cand_rows(desc, g, d_c, C, a.uv ? nullptr : d_mask,
                         a.uv ? (a.pv.dtype_ab & 3) * 4 + (a.pv.dtype_d & 3) : -1, fv, d_rows, memo, wait->words, stream,
                         launches);
    if (e != cudaSuccess) return e;
    if (memo.keys) {
      e = ensure_dynamic_smem(reinterpret_cast<const void*>(&pair_table_kernel), pthr_bytes);
      if (e != cudaSuccess) return e;
      e = memo_compact(memo, stream);
      if (e != cudaSuccess) return e;
      ++*launches;
      fv.pair_class = memo.cls;
      fv.pair_tab = static_cast<const uint8_t*>(memo.tab);
      fv.prob_tab = fv.pair_tab + static_cast<size_t>(memo_batch) * kMemoCap * pair_rec_bytes(g);
    }
  }
  if (C == 0) {  // no kernel in front of the walk: the word that a failed call may have left is cleared here
    e = cudaMemsetAsync(wait->words + kWordWalk, 0, sizeof(int), stream);
    if (e != cudaSuccess) return e;
  }
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  if (ev_begin) cudaEventRecord(ev_begin, stream);
  const int* path = nullptr;  // device word: whether the class walk serves the call
  if (classes) {
    e = prepare_classes(desc, g, d_p, P, d_c, C, *classes, stream, launches, wait, &path);
    if (e != cudaSuccess) return e;
  }

  a.sl.words = wait->words;
  if (split) {
    a.sl.scores = split->scores;
    a.sl.out_idx = split->out_idx;
    a.sl.out_score = split->out_score;
    a.sl.tiles = prep ? prep->call : split->tiles;  // (per-pair rows first)
    a.sl.out_seq = split->out_seq;
    a.sl.seq = split->seq;
  }
  // problems in batches when the memo's table does not hold them all at once
  const int step = memo.keys ? balanced_step(g, P, memo_batch, nblk) : P;
  // A table that holds more classes than a problem has candidates is evaluated for nothing: the tiles of a short segment
  // are filled in place then. Up to 4,096 classes a problem's table is done sooner, spread over the machine,
  // than a block fills its tile. Mixed types, 500 trees of depth 8 (200, 256 bins): 300 segments of 700
  // out of 61,085 valid candidates (10,785 classes) 1,955 -> 707 us (1,328 -> 403), 1,000 of 300 6,016 -> 1,937 (3,864 ->
  // 786); out of 60,000 grid ones, with records 732 (410) and in place 680 (329), but 32 x 700 244 (151) and 267 (149).
  const int most_classes = seg_off ? std::max(4096, nblk * rows_per_cta) : kMemoCap;
  for (int first = 0; first < P; first += step) {
    const int n = P - first < step ? P - first : step;
    if (memo.keys) {
      // as many blocks as the machine holds at once (two per SM by registers, fewer when the staged
      // thresholds take more than half an SM's shared memory); never more blocks than items
      const int64_t table_items = static_cast<int64_t>(kMemoCap / 256) * n;
      const int64_t table_slots = static_cast<int64_t>(kSmCount) * (2 * (pthr_bytes + 4096) <= 227 * 1024 ? 2 : 1);
      pair_table_kernel<<<static_cast<unsigned>(table_items < table_slots ? table_items : table_slots), 256, pthr_bytes,
                          stream>>>(
          desc, d_p + first, n, d_c, fv, memo, pthr_cap, path, wait->words, C, most_classes);
      ++*launches;
    }
    a.dependent = memo.keys != nullptr || ((tiles_mode || prep) && !ev_begin);  // (no event stands between the two)
    a.d_p = d_p ? d_p + first : nullptr;
    a.P = n;
    a.seg_off = seg_off ? seg_off + first : nullptr;
    a.partial = partial + static_cast<size_t>(first) * nblk * k;
    if (split) a.split_ctas = split_plan(g, static_cast<int64_t>(n) * nblk, &a.sl);
    if (a.sl.units > 0) ++*wait->splits;
    e = launch_walk(g, a);
    ++*launches;
    if (e != cudaSuccess) return e;
  }
  if (classes)
    return launch_classes(desc, g, P, d_c, C, d_rows, seg_off, seg_idx, nblk, rows_per_cta, k, partial, *classes, status,
                          stream, launches, wait);
  return cudaSuccess;
}

// ks_score on the quantised path. Rows are taken in batches so that the tiles (n_rows bytes per
// row) stay a bounded workspace; every batch is one tile launch and one walk launch.
constexpr int64_t kScoreBatchRows = 4096 * 1024;

size_t score_fast_scratch_bytes(const GbdtModel& g, int64_t rows) {
  int64_t blocks = (std::min(rows, kScoreBatchRows) + g.block_cands - 1) / g.block_cands;
  return (static_cast<size_t>(blocks) * g.n_qrows * g.block_cands + 255) / 256 * 256 + fast_split_bytes(g);
}

cudaError_t launch_score_fast(const ks_gpu_desc& desc, const GbdtModel& g, const float* d_feat, int64_t rows,
                              float* d_scores, void* scratch, int* status, cudaStream_t stream,
                              int64_t* launches, const FastWait* wait, int floor_repeat) {
  WalkArgs a{};
  a.desc = desc;
  a.uv = 1;
  a.P = 1;
  a.rows_per_cta = g.block_cands;
  a.status = status;
  a.top = g.h_top;
  a.stream = stream;
  a.fv = make_view(g, wait);
  uint8_t* tiles = static_cast<uint8_t*>(scratch);
  // (at most kTileMaxThr thresholds, 192 KB)
  const size_t smem = sizeof(float) * (64 * kTileRows + g.n_qthr);
  cudaError_t e = ensure_dynamic_smem(reinterpret_cast<const void*>(&tile_rows_kernel), smem);
  if (e != cudaSuccess) return e;
  for (int64_t first = 0; first < rows; first += kScoreBatchRows) {
    const int64_t n = rows - first < kScoreBatchRows ? rows - first : kScoreBatchRows;
    const int nblk = static_cast<int>((n + g.block_cands - 1) / g.block_cands);
    const int W = g.block_cands / 4, groups = nblk * (W / 32);
    const int resident = 2 * (smem + 3072) <= 227 * 1024 ? 2 : 1;
    tile_rows_kernel<<<std::min(groups, resident * kSmCount), kTileWarps * 32, smem, stream>>>(
        d_feat + first * KS_F_PAD, n, a.fv, tiles, W, groups, wait->words);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    a.C = static_cast<int>(n);
    a.nblk = nblk;
    a.sl = SplitArgs{};
    if (floor_repeat == 0 && (g.ctas_per_sm == 1 || nblk < 2 * kSmCount) && split_fits(g, nblk)) {
      a.split_ctas = split_plan(g, nblk, &a.sl);
      a.sl.scores = reinterpret_cast<double*>(tiles + score_fast_scratch_bytes(g, std::min(rows, kScoreBatchRows)) - fast_split_bytes(g));
    }
    if (a.sl.units > 0) ++*wait->splits;
    a.sl.words = wait->words;
    a.dependent = 1;
    a.sl.tiles = tiles;
    a.sl.score_out = d_scores + first;
    a.sl.repeat = floor_repeat;
    *launches += 2;
    e = floor_repeat > 0 ? launch_walk_floor(g, a) : launch_walk(g, a);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

#ifdef KS_DEBUG_BOUNDS
int fast_bounds_line() {
  int v = 0;
  cudaMemcpyFromSymbol(&v, g_bounds_line, sizeof(int));
  return v ? v : class_bounds_line();
}
void fast_bounds_clear() {
  const int z = 0;
  cudaMemcpyToSymbol(g_bounds_line, &z, sizeof(int));
  class_bounds_clear();
}
#else
int fast_bounds_line() { return -1; }
void fast_bounds_clear() {}
#endif

}  // namespace ks
