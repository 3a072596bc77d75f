// Tree ensembles on a large batch: one walk for all candidates of a class.
//
// What bounds the walk of ks_gbdt_fast.cu is that every candidate follows its own path: eight
// dependent node visits a tree, two shared-memory gathers each. In a cross-product catalogue that
// work repeats itself. Candidates that agree in (T_M, T_N, T_K, stages, c_M, c_N) and in their
// resident-block count - a class - have the same per-pair columns for every problem; they differ in
// candidate-only columns alone, and which way a candidate turns at such a node does not depend on
// the problem. So the ensemble is compiled for a class and run for all problems:
//
//   compile  every tree is restricted to the class. A candidate-only node at which all members turn
//            the same way disappears (46 % of the nodes test such a column). Where the members part,
//            the walk has to visit both sides, one after the other: the leaves of the first side get
//            the second side as their continuation, so that a tree stays one chain of node and leaf
//            visits without a stack, and the last leaf of a tree continues at the next tree. A leaf
//            carries the set of members that reach it as the number of an accumulator (bucket).
//   run      a thread is a problem: it follows the chain through node words (per-pair and problem-only
//            rows) and adds leaf values to its buckets.
//   finish   a member's score is the sum of the buckets whose set it belongs to.
//
// A class of 36 members (the mean of the 60,000-candidate catalogue) costs about 5.7 node and 1.8
// leaf visits a tree where its members took 288 node visits; a class of one still saves the
// candidate-only nodes. Compiling costs as much as some 60 problems, hence the batch.
//
// Leaf values are summed as 32-bit integers in units of a power of two (see fixed_point_shift), so a
// sum does not depend on its order: candidates that end in the same leaves have equal scores in
// whatever classes they are, and how many threads share a problem changes nothing.
//
// Scores go to a plane [candidate][problem] (coalesced: a warp is 32 problems) and are ranked by a
// kernel of their own, one thread per problem and share of the candidates.
//
// Words of a compiled tree (4 bytes, offsets in bytes relative to the chunk buffer they run in):
//   node   row << 24 | threshold index << 16 | right child's offset | 1: it is a leaf | 2: the left
//          child (always the next word) is a leaf
//   leaf   value; bucket << 16 | continuation's offset | 1: it is a leaf | 2: the chunk ends here
#include <cub/device/device_radix_sort.cuh>

#include <algorithm>
#include <cmath>
#include <vector>

#include "ks_gbdt_quant.cuh"
#include "ks_topk.cuh"

namespace ks {
namespace {

constexpr int kSlots = 128;         // problems of a CTA
constexpr int kT = 512;             // its threads: four or more share a problem, each with its own trees
constexpr int kMembers = 64;        // candidates compiled together
constexpr int kBufWords = 4096;     // one of the two chunk buffers
constexpr int kMinProg = 256;       // words of a compiled tree on average, for the size of the program's memory
constexpr int kMaxTreeWords = 1536; // ... and the longest
constexpr int kHash = 1024;         // distinct member sets a class may have
constexpr int kPool = 4096;         // terms of the sets that take several buckets
constexpr int kMaxTerms = 24;
constexpr int kSplitRows = 64, kSplitValues = 8;  // rows whose member sets are tabulated
constexpr int kMaxBuckets = 112;
constexpr int kMaxTrees = 1024;     // <= kHash: arrays of the member sets are used again for the trees
constexpr int kMaxChunks = 640;     // kMaxTrees full trees of depth 8 (768 words) take 615
constexpr unsigned kLeaf = 1u, kLeftLeaf = 2u, kEnd = 2u;  // low bits of a code
constexpr uint32_t kRootLeaf = 0x8000u;
constexpr int kBufBytes = 4 * kBufWords;  // a power of two: a buffer starts at a multiple, so that an offset is or-ed in
constexpr int kRunCut = 4096;
constexpr int kSms = 148;
constexpr int kProbBytes = kFastMaxProbRows + 128;  // problem-only bytes, then the problem's terms
constexpr size_t kPlaneBytes = size_t(1) << 30;   // scores held at a time

// What one launch works on. `seg` of a batch: problems of one element-type combination.
struct ClassArgs {
  FastView fv;
  int nc_shift;               // log2 of the candidates per tile row that the model's node words count in
  int n_trees;
  float scale, unscale;       // leaf values are summed as integers: multiples of `unscale`
  int n_buckets, tile_rows;   // accumulators per problem; rows of the tile (per-pair, then problem-only)
  const ks_candidate* c;
  int C, P;
  const int* order;           // [C] catalogue positions in similarity order
  const int2* units;          // (first position in `order`, candidates)
  int* counters;              // [0] units, [1] 1: this path serves the call, [2] work counter, [3] 1: a wait ran out, [8..25) first problem of every combination
  const int* prob_order;      // [P] problems by combination and size
  const uint8_t* prob_tab;    // [P][kProbBytes], in that order
  uint8_t* programs;          // per CTA: [n_trees][32] uint4 (sets of the leaves), [n_trees * prog_words] words
  int prog_words;
  float* plane;               // [C][pitch]
  int pitch, first, count;    // problems first .. first + count - 1 of the order
  int* status;
};

// ------------------------------------------------------------------------------------------
// preparation of a call
// ------------------------------------------------------------------------------------------

__device__ __forceinline__ bool same_group(const ks_candidate& a, const ks_candidate& b) {
  return a.tile_m == b.tile_m && a.tile_n == b.tile_n && a.tile_k == b.tile_k && a.stages == b.stages &&
         a.cluster_m == b.cluster_m && a.cluster_n == b.cluster_n;
}

// Runs of candidates that agree in the six knobs, cut into units of at most kMembers.
__global__ void __launch_bounds__(256)
units_kernel(const ks_candidate* __restrict__ c, int C, const int* __restrict__ order, int2* __restrict__ units,
             int* __restrict__ counters) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= C) return;
  // a run also ends at every multiple of kRunCut, so that no thread walks a whole catalogue
  const ks_candidate me = load_candidate(c + order[i]);
  if (i % kRunCut != 0 && same_group(me, load_candidate(c + order[i - 1]))) return;
  int start = i, j = i + 1;
  for (;; ++j) {
    const bool more = j < C && j % kRunCut != 0 && same_group(me, load_candidate(c + order[j]));
    if (!more || j - start == kMembers) {
      units[atomicAdd(counters, 1)] = make_int2(start, j - start);
      start = j;
    }
    if (!more) break;
  }
}

// Sort key of a problem: element-type combination, then the octaves of M, N, K interleaved, so that
// the lanes of a warp take similar paths.
__device__ __forceinline__ unsigned problem_key(const ks_problem& pr) {
  const unsigned q[3] = {static_cast<unsigned>(__log2f(static_cast<float>(pr.m)) * 6.4f) & 127u,
                         static_cast<unsigned>(__log2f(static_cast<float>(pr.n)) * 6.4f) & 127u,
                         static_cast<unsigned>(__log2f(static_cast<float>(pr.k)) * 6.4f) & 127u};
  unsigned key = (pr.dtype_ab & 3) * 4 + (pr.dtype_d & 3);
  for (int b = 6; b >= 0; --b)
    for (int d = 0; d < 3; ++d) key = key << 1 | ((q[d] >> b) & 1u);
  return key;
}
__global__ void problem_keys_kernel(const ks_problem* __restrict__ p, int P, unsigned* __restrict__ keys,
                                    int* __restrict__ idx) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= P) return;
  keys[i] = problem_key(load_problem(p + i));
  idx[i] = i;
}
// Keys and order of up to kCountProblems problems in one launch: a problem's place is the number of keys
// before its own. P comparisons a thread, four a load: 6 us for 267 problems, where the
// keys and the radix sort of one block take 18.
constexpr int kCountProblems = 4096;
__global__ void __launch_bounds__(256)
problem_order_kernel(const ks_problem* __restrict__ p, int P, unsigned* __restrict__ keys, int* __restrict__ order) {
  __shared__ __align__(16) unsigned s_key[kCountProblems];
  const int padded = (P + 3) / 4 * 4;
  for (int i = threadIdx.x; i < padded; i += blockDim.x) s_key[i] = i < P ? problem_key(load_problem(p + i)) : ~0u;
  __syncthreads();
  const int me = blockIdx.x * blockDim.x + threadIdx.x;
  if (me >= P) return;
  const unsigned key = s_key[me];
  int place = 0;
  for (int i = 0; i < padded; i += 4) {
    const uint4 other = *reinterpret_cast<const uint4*>(s_key + i);
    place += (other.x < key || (other.x == key && i < me)) + (other.y < key || (other.y == key && i + 1 < me)) +
             (other.z < key || (other.z == key && i + 2 < me)) + (other.w < key || (other.w == key && i + 3 < me));
  }
  keys[place] = key;
  order[place] = me;
}
constexpr int kProblemKeyBits = 25;

// One block of 64 threads per problem: terms and problem-only bytes, in sorted order; and where
// each combination begins.
__global__ void __launch_bounds__(64)
problem_rows_kernel(ks_gpu_desc desc, const ks_problem* __restrict__ p, int P, const int* __restrict__ prob_order,
                    const unsigned* __restrict__ keys, FastView fv, uint8_t* __restrict__ tab, int* __restrict__ counters) {
  __shared__ ProblemTerms s_pt;
  __shared__ float s_pf[64];
  const int i = blockIdx.x, tid = threadIdx.x;
  if (tid == 0) {
    const int combo = static_cast<int>(keys[i] >> 21), prev = i > 0 ? static_cast<int>(keys[i - 1] >> 21) : -1;
    for (int q = prev + 1; q <= combo; ++q) counters[8 + q] = i;
    if (i == P - 1)
      for (int q = combo + 1; q <= 16; ++q) counters[8 + q] = P;
    problem_terms(load_problem(p + prob_order[i]), desc, s_pt);
    problem_columns(s_pt, [&](int col, float v) { s_pf[col] = v; });
  }
  __syncthreads();
  uint8_t* out = tab + static_cast<size_t>(i) * kProbBytes;
  if (tid < KS_F && feat_class(tid) == 0) {
    const FeatQ q = fv.feat[tid];
    const int first = fv.n_pair_rows + fv.n_cand_rows;
    quantise(q, fv.thr + q.thr0, s_pf[tid], false,
             [&](int row, uint8_t b) { out[KS_IDX(row - first, kFastMaxProbRows)] = b & 0x7F; });
  }
  if (tid < static_cast<int>(sizeof(ProblemTerms) / 4))
    reinterpret_cast<uint32_t*>(out + kFastMaxProbRows)[tid] = reinterpret_cast<const uint32_t*>(&s_pt)[tid];
}

// Rounds that n problems take when a round serves kSlots / s of them.
__host__ __device__ constexpr int rounds_of(int n, int s) { return (n * s + kSlots - 1) / kSlots; }

// The cost of this walk for `n` problems of one element-type combination, in pairs that their own walks
// take as long for (see choose_path_kernel).
__host__ __device__ constexpr int64_t walk_cost(int64_t units, int n) {
  return units * 13 / 10 * (static_cast<int64_t>(rounds_of(n, 1)) * 900 + 3600);
}
__host__ __device__ constexpr bool walk_pays(int64_t cost, int64_t pairs) { return cost + cost / 10 < pairs; }

// Chooses between this path and the per-candidate walk, on the device, where the number of units is
// known. In clocks of one of two CTAs on an SM, a tree: a candidate's own walk takes 1.0 (52.9 ms for
// 1,024 x 60,000 pairs and 500 trees); a class 900 for every round of problem slots and 3,600 to be
// compiled (measured on the same batch: 1,712 classes, 1.3 a unit, 8 rounds, 17 ms). The line is put a
// tenth to the safe side.
__global__ void choose_path_kernel(int64_t pairs, int* counters, int* served) {
  const int64_t units = counters[0];
  int64_t cost = 0;
  for (int q = 0; q < 16; ++q) {
    const int n = counters[9 + q] - counters[8 + q];
    if (n > 0) cost += walk_cost(units, n);
  }
  counters[1] = walk_pays(cost, pairs) ? 1 : 0;
  *served += counters[1];
}

// ------------------------------------------------------------------------------------------
// compilation
// ------------------------------------------------------------------------------------------

// Shared state of a CTA. The arrays of the compilation lie in the part of the dynamic shared
// memory that holds the tile and the buckets afterwards.
struct BuildShared {
  unsigned long long key[kHash];  // member sets, 0: free
  unsigned weight[kHash];         // how often a walk is expected to meet the set
  unsigned chain[kHash];          // its buckets: first term of the pool << 8 | number of terms, or 0: its members one by one
  uint8_t pool[kPool];            // terms: bucket, top bit: subtract
  uint8_t terms[kT / 32][kMaxTerms];
  int occupied[kHash];
  int n_occupied, n_pool;
  int scan[kT / 32];
  uint8_t lo[kFastMaxCandRec], hi[kFastMaxCandRec];      // smallest and largest member byte of a candidate-only row
  uint8_t bytes[kFastMaxCandRec][kMembers];              // member bytes of the candidate-only rows
  // rows at which members part: the members above each of their distinct bytes
  unsigned long long split_set[kSplitRows][kSplitValues];
  uint8_t split_index[kSplitRows][128];                  // threshold index -> which of them
  uint8_t split_of[kFastMaxCandRec];                     // a row's place among them, 0xFF: not tabulated
  int n_split;
};

__device__ __forceinline__ int hash_of(unsigned long long key) {
  return static_cast<int>((key * 0x9E3779B97F4A7C15ull) >> 54);
}
// slot of a member set, inserting it; -1 when the table is full
__device__ __forceinline__ int set_slot(BuildShared* b, unsigned long long key) {
  int h = hash_of(key);
  for (int probe = 0; probe < 128; ++probe) {
    // (most sets are there already, and an exchange that a whole warp asks for is served lane by lane)
    unsigned long long prev = *reinterpret_cast<volatile unsigned long long*>(&b->key[h]);
    if (prev == 0ull) prev = atomicCAS(&b->key[h], 0ull, key);
    if (prev == 0ull || prev == key) return h;
    h = (h + 1) & (kHash - 1);
  }
  return -1;
}

// Members whose byte of candidate-only row r exceeds j (bytes are 0..127; padding repeats member 0).
__device__ __forceinline__ unsigned long long members_right(const BuildShared* b, int r, unsigned j) {
  const uint32_t* w = reinterpret_cast<const uint32_t*>(b->bytes[r]);
  const uint32_t sub = (j + 1) * 0x01010101u;
  unsigned long long m = 0ull;
#pragma unroll
  for (int q = 0; q < kMembers / 4; ++q) {
    const uint32_t t = ((w[q] | 0x80808080u) - sub) & 0x80808080u;  // top bit: byte > j
    m |= static_cast<unsigned long long>((t >> 7) * 0x10204080u >> 28) << (4 * q);
  }
  return m;
}

// The same for a threshold index j between the row's smallest and largest byte, from the table where
// the row is in it.
__device__ __forceinline__ unsigned long long members_above(const BuildShared* b, int r, unsigned j) {
  const unsigned e = b->split_of[r];
  if (e == 0xFFu) return members_right(b, r, j);
  return b->split_set[e][b->split_index[e][j]];
}

// ------------------------------------------------------------------------------------------
// the kernel
// ------------------------------------------------------------------------------------------

// Exclusive prefix sum over the CTA; `total` receives the sum. All threads call.
__device__ __forceinline__ int block_scan(int v, int* s_part, int* total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int incl = v;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const int u = __shfl_up_sync(0xFFFFFFFFu, incl, d);
    if (lane >= d) incl += u;
  }
  __syncthreads();
  if (lane == 31) s_part[warp] = incl;
  __syncthreads();
  int before = 0, sum = 0;
  for (int w = 0; w < kT / 32; ++w) {
    if (w < warp) before += s_part[w];
    sum += s_part[w];
  }
  *total = sum;
  return before + incl - v;
}

// Gives every member set its accumulators. The full set is bucket 0. When all sets fit, each has
// its own; else the single members have one each, so that any set can be written, and the rest
// goes to the sets that are met most often; any other set becomes a sum of disjoint sets that have
// one, largest first, or a superset less such a sum, whichever is shorter. Everything is decided by
// (weight, set), so the sums do not depend on the order of insertion.
__device__ void assign_buckets(BuildShared* b, int n_buckets, int m, unsigned long long full, unsigned long long* s_sets) {
  const int tid = threadIdx.x;
  if (tid == 0) b->n_occupied = b->n_pool = 0;
  for (int i = tid; i < n_buckets; i += kT) s_sets[i] = 0ull;
  __syncthreads();
  for (int i = tid; i < kHash; i += kT)
    if (b->key[i]) b->occupied[atomicAdd(&b->n_occupied, 1)] = i;
  __syncthreads();
  const int n = b->n_occupied;
  const bool all = n + 1 <= n_buckets;
  const int reserved = all ? 1 : 1 + m;  // the full set, and the single members
  if (tid == 0) s_sets[0] = full;
  if (!all && tid < m) s_sets[1 + tid] = 1ull << tid;
  for (int e = tid; e < n; e += kT) {
    const int me = b->occupied[e];
    const unsigned long long k = b->key[me];
    const unsigned w = b->weight[me];
    int bucket = -1;
    if (k == full) {
      bucket = 0;
    } else if (!all && __popcll(k) == 1) {
      bucket = 1 + __ffsll(static_cast<long long>(k)) - 1;
    } else {
      int rank = 0;
      for (int q = 0; q < n; ++q) {
        const int o = b->occupied[q];
        const unsigned long long ko = b->key[o];
        if (ko == full || (!all && __popcll(ko) == 1)) continue;
        const unsigned wo = b->weight[o];
        rank += wo > w || (wo == w && ko < k);
      }
      if (reserved + rank < n_buckets) bucket = reserved + rank;
    }
    b->chain[me] = bucket >= 0 ? 0x80000000u | static_cast<unsigned>(bucket) : 0u;
    if (bucket >= 0) s_sets[bucket] = k;
  }
  __syncthreads();
  // a warp per set, its lanes the buckets
  const int lane = tid & 31;
  for (int e = tid >> 5; e < n; e += kT / 32) {
    const int me = b->occupied[e];
    uint8_t* terms = b->terms[tid >> 5];
    int cnt = 0;
    if (b->chain[me] & 0x80000000u) {  // a bucket of its own
      if (lane == 0) terms[0] = static_cast<uint8_t>(b->chain[me]);
      cnt = 1;
    } else {
      // largest subsets first, either of the set or of what its smallest superset has too much
      const unsigned long long k = b->key[me];
      auto pick = [&](unsigned long long rest, bool around) {  // bucket: largest inside `rest`, or smallest around it
        int best = 0;
        for (int q = lane; q < n_buckets; q += 32) {
          const unsigned long long x = s_sets[q];
          if (x == 0ull || (around ? rest & ~x : x & ~rest)) continue;
          best = max(best, (around ? 128 - __popcll(x) : __popcll(x)) << 8 | (255 - q));
        }
        return 255 - (__reduce_max_sync(0xFFFFFFFFu, best) & 0xFF);
      };
      auto cover = [&](unsigned long long rest, int from, unsigned sign) {  // terms from .. ; returns their end, or more than kMaxTerms
        int c = from;
        while (rest && c <= kMaxTerms) {
          const int q = pick(rest, false);
          if (lane == 0 && c < kMaxTerms) terms[c] = static_cast<uint8_t>(q | sign);
          rest ^= s_sets[q];
          ++c;
        }
        return c;
      };
      cnt = cover(k, 0, 0u);
      if (cnt > 2) {
        const int around = pick(k, true);
        const int with_less = cover(s_sets[around] ^ k, 1, 0x80u);  // (overwrites)
        if (with_less <= cnt) {
          if (lane == 0) terms[0] = static_cast<uint8_t>(around);
          cnt = with_less;
        } else {
          cnt = cover(k, 0, 0u);
        }
      }
    }
    __syncwarp();
    int at = 0;
    if (lane == 0 && cnt <= kMaxTerms) at = atomicAdd(&b->n_pool, cnt);
    at = __shfl_sync(0xFFFFFFFFu, at, 0);
    const bool fits = cnt <= kMaxTerms && at + cnt <= kPool;
    if (fits && lane < cnt) b->pool[at + lane] = terms[lane];
    if (lane == 0) b->chain[me] = fits ? static_cast<unsigned>(at) << 8 | static_cast<unsigned>(cnt) : 0u;
    __syncwarp();
  }
  __syncthreads();
}

// terms of a set; without a chain: its members one by one (possible when they have buckets)
__device__ __forceinline__ int chain_length(unsigned chain, unsigned long long set) {
  return chain ? static_cast<int>(chain & 0xFFu) : __popcll(set);
}

// Which members turn right at a node, and whether it stays a node of the compiled tree (`real`: it
// tests a per-pair or problem-only row; `above` then means nothing).
struct NodeView {
  unsigned long long above;
  uint32_t head;  // row of the tile << 8 | threshold index
  bool real;
};
__device__ __forceinline__ NodeView view_node(const ClassArgs& a, const BuildShared* b, uint32_t word) {
  const FastView& fv = a.fv;
  NodeView n;
  const unsigned j = word & 0xFFu, jj = j & 0x7Fu;
  const int row = static_cast<int>(word >> 8) >> a.nc_shift, r = row - fv.n_pair_rows;
  n.real = j != 0xFFu && !(r >= 0 && r < fv.n_cand_rows);  // 0xFF: everybody goes left
  n.head = static_cast<uint32_t>(r >= 0 ? row - fv.n_cand_rows : row) << 8 | jj;
  n.above = 0ull;
  if (!n.real && j != 0xFFu) {
    if (b->lo[r] > jj) n.above = ~0ull;
    else if (b->hi[r] > jj) n.above = members_above(b, r, jj);
  }
  return n;
}
__device__ __forceinline__ unsigned long long shfl64(unsigned long long v, int src) {
  return __shfl_sync(0xFFFFFFFFu, v, src);
}

// A warp works on one tree. Lane h < 31 holds node h of the five top levels (heap order), and every
// lane the subtree below node `lane` of level 5: 2^SUB - 1 nodes, 2^SUB leaves, in registers. What
// travels between levels goes through shuffles; nothing is stacked or stored.
__device__ __forceinline__ const uint32_t* top_word(const FastView& fv, int t, int lane) {
  const uint32_t* base = fv.chunks + static_cast<size_t>(t / fv.tpc) * (fv.chunk_bytes / 4);
  const int tt = t % fv.tpc, l = 31 - __clz(lane + 1);
  return base + fv.tpc * ((1 << l) - 1) + (tt << l) + (lane + 1 - (1 << l));
}
// The lane's subtree: nodes 0 .. N - 1 in heap order (level d of it has 2^d; its level SUB are the
// leaves). A level's words lie side by side, so they are fetched as one vector or two where the chunk's
// tree count keeps them aligned.
template <int N>
__device__ __forceinline__ void load_subtree(const FastView& fv, int t, int lane, uint32_t (&v)[N]) {
  const uint32_t* base = fv.chunks + static_cast<size_t>(t / fv.tpc) * (fv.chunk_bytes / 4);
  const int tt = t % fv.tpc;
  const bool aligned = (fv.tpc & 3) == 0;
#pragma unroll
  for (int d = 0; (1 << d) - 1 < N; ++d) {
    const int l = 5 + d;
    const uint32_t* p = base + fv.tpc * ((1 << l) - 1) + (tt << l) + (lane << d);
    if (d == 1 && aligned) {
      const uint2 q = __ldg(reinterpret_cast<const uint2*>(p));
      v[1 < N ? 1 : 0] = q.x; v[2 < N ? 2 : 0] = q.y;
    } else if (d >= 2 && aligned) {
#pragma unroll
      for (int x = 0; x < (1 << d) / 4; ++x) {
        const uint4 q = __ldg(reinterpret_cast<const uint4*>(p) + x);
        const int k = (1 << d) - 1 + 4 * x;
        v[k < N ? k : 0] = q.x; v[k + 1 < N ? k + 1 : 0] = q.y; v[k + 2 < N ? k + 2 : 0] = q.z; v[k + 3 < N ? k + 3 : 0] = q.w;
      }
    } else {
#pragma unroll
      for (int x = 0; x < (1 << d); ++x) v[(1 << d) - 1 + x < N ? (1 << d) - 1 + x : 0] = __ldg(p + x);
    }
  }
}
// lane that holds the left child of top node h: of the level-5 subtrees for h >= 15, else a top node
__device__ __forceinline__ int left_lane(int h) { return h >= 15 ? 2 * (h - 15) : 2 * h + 1; }

// First pass: the member set of every leaf, entered into the table; ids[lane] receives the table
// slots of the lane's leaves (0xFFFF: nobody gets there), sh_tree[t] the number of nodes that stay
// (and kRootLeaf). False: the table is full.
template <int SUB>
__device__ bool find_sets(const ClassArgs& a, BuildShared* b, unsigned long long full, int t, uint4* ids, uint32_t* sh_tree) {
  constexpr int NL = 1 << SUB;
  const FastView& fv = a.fv;
  const int lane = threadIdx.x & 31;
  unsigned long long mask = lane == 0 ? full : 0ull;
  unsigned count = 0;  // nodes that stay above this one
  uint32_t words[NL > 1 ? NL - 1 : 1];
  const uint32_t top_node = __ldg(top_word(fv, t, lane < 31 ? lane : 0));
  load_subtree(fv, t, lane, words);
  NodeView top{};
  if (lane < 31) top = view_node(a, b, top_node);
  const int parent = lane > 0 ? (lane - 1) >> 1 : 0;
  for (int l = 0; l < 4; ++l) {  // level l to level l + 1
    const unsigned long long lm = shfl64(top.real ? mask : mask & ~top.above, parent);
    const unsigned long long rm = shfl64(top.real ? mask : mask & top.above, parent);
    const unsigned c = __shfl_sync(0xFFFFFFFFu, count + (top.real ? 1u : 0u), parent);
    if (31 - __clz(lane + 1) == l + 1) {
      mask = (lane & 1) ? lm : rm;
      count = c;
    }
  }
  unsigned n_real = lane < 31 && top.real && mask != 0ull;
  const int above5 = 15 + (lane >> 1);  // the lane's subtree hangs below this node
  const unsigned long long lm = shfl64(top.real ? mask : mask & ~top.above, above5);
  const unsigned long long rm = shfl64(top.real ? mask : mask & top.above, above5);
  const unsigned c5 = __shfl_sync(0xFFFFFFFFu, count + (top.real ? 1u : 0u), above5);
  unsigned long long m[2 * NL - 1];
  unsigned c[2 * NL - 1];
  m[0] = (lane & 1) ? rm : lm;
  c[0] = c5;
#pragma unroll
  for (int k = 0; k < NL - 1; ++k) {
    const NodeView n = view_node(a, b, words[k]);
    m[2 * k + 1] = n.real ? m[k] : m[k] & ~n.above;
    m[2 * k + 2] = n.real ? m[k] : m[k] & n.above;
    c[2 * k + 1] = c[2 * k + 2] = c[k] + (n.real ? 1u : 0u);
    n_real += n.real && m[k] != 0ull;
  }
  uint32_t w[4] = {0xFFFFFFFFu, 0xFFFFFFFFu, 0xFFFFFFFFu, 0xFFFFFFFFu};
  bool fits = true;
  unsigned first = 0xFFFFu;  // nodes above the lane's first living leaf
#pragma unroll
  for (int k = NL - 1; k >= 0; --k) {
    const unsigned long long set = m[NL - 1 + k];
    if (set == 0ull) continue;
    const int id = set_slot(b, set);
    if (id < 0) {
      fits = false;
      continue;
    }
    first = c[NL - 1 + k];
    atomicAdd(&b->weight[id], 4096u >> first);
    w[k >> 1] = (k & 1) ? (w[k >> 1] & 0xFFFFu) | static_cast<uint32_t>(id) << 16 : (w[k >> 1] & 0xFFFF0000u) | static_cast<uint32_t>(id);
  }
  ids[lane] = make_uint4(w[0], w[1], w[2], w[3]);
  n_real = __reduce_add_sync(0xFFFFFFFFu, n_real);
  const unsigned living = __ballot_sync(0xFFFFFFFFu, first != 0xFFFFu);
  const unsigned above_first = __shfl_sync(0xFFFFFFFFu, first, __ffs(living) - 1);
  if (lane == 0) sh_tree[t] = n_real | (above_first == 0u ? kRootLeaf : 0u);
  return __all_sync(0xFFFFFFFFu, fits);
}

// Second pass: words of the tree, with the sets that take several buckets.
__device__ int tree_words(const BuildShared* b, const uint4* ids, int n_real) {
  const uint4 q = ids[threadIdx.x & 31];
  const uint32_t w[4] = {q.x, q.y, q.z, q.w};
  int n = 0;
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const unsigned id = (w[k >> 1] >> (16 * (k & 1))) & 0xFFFFu;
    if (id != 0xFFFFu) n += 2 * chain_length(b->chain[id], b->key[id]);
  }
  return n_real + __reduce_add_sync(0xFFFFFFFFu, n);
}

// Third pass: writes the words. Depth first: the left child right behind its node; where the members
// part, the left side first, and the right side is what its leaves continue at. `at`: offset of the
// tree in its chunk; `next_tree`: where its last leaf continues.
template <int SUB>
__device__ void write_tree(const ClassArgs& a, const BuildShared* b, int t, const uint4* ids, uint32_t* out, unsigned at,
                           unsigned next_tree) {
  constexpr int NL = 1 << SUB, NN = 2 * NL - 1;
  constexpr uint32_t kNone = 0xFFFFu;  // continuation of the tree's last leaves
  const FastView& fv = a.fv;
  const int lane = threadIdx.x & 31;
  const uint4 q = ids[lane];
  const uint32_t idw[4] = {q.x, q.y, q.z, q.w};
  auto id_of = [&](int k) { return (idw[k >> 1] >> (16 * (k & 1))) & 0xFFFFu; };
  uint32_t words[NN];  // nodes and leaves
  load_subtree(fv, t, lane, words);
  const uint32_t top_node = __ldg(top_word(fv, t, lane < 31 ? lane : 0));
  // per node: words of its subtree << 1 | it begins with a leaf
  uint32_t size[NN], head[NL];
  bool real[NL];
#pragma unroll
  for (int k = 0; k < NL; ++k) {
    const unsigned id = id_of(k);
    size[NL - 1 + k] = id != 0xFFFFu ? static_cast<uint32_t>(2 * chain_length(b->chain[id], b->key[id])) << 1 | 1u : 0u;
  }
  auto join = [](bool is_real, uint32_t l, uint32_t r) -> uint32_t {
    const uint32_t words = (l >> 1) + (r >> 1);
    if (words == 0) return 0u;
    return is_real ? (words + 1) << 1 : words << 1 | ((l >> 1) ? l & 1u : r & 1u);
  };
  auto row_of = [&](uint32_t word, uint32_t& hd) {  // (as view_node, without the members)
    const unsigned j = word & 0xFFu;
    const int row = static_cast<int>(word >> 8) >> a.nc_shift, r = row - fv.n_pair_rows;
    hd = static_cast<uint32_t>(r >= 0 ? row - fv.n_cand_rows : row) << 8 | (j & 0x7Fu);
    return j != 0xFFu && !(r >= 0 && r < fv.n_cand_rows);
  };
#pragma unroll
  for (int k = NL - 2; k >= 0; --k) {
    real[k] = row_of(words[k], head[k]);
    size[k] = join(real[k], size[2 * k + 1], size[2 * k + 2]);
  }
  uint32_t top_head = 0, top_size = 0, top_l = 0, top_r = 0;
  const bool top_real = lane < 31 && row_of(top_node, top_head);
  for (int l = 4; l >= 0; --l) {  // bottom up
    const uint32_t from = l == 4 ? size[0] : top_size;
    const int src = left_lane(lane < 31 ? lane : 0) & 31;
    const uint32_t lw = __shfl_sync(0xFFFFFFFFu, from, src), rw = __shfl_sync(0xFFFFFFFFu, from, (src + 1) & 31);
    if (lane < 31 && 31 - __clz(lane + 1) == l) {
      top_l = lw;
      top_r = rw;
      top_size = join(top_real, lw, rw);
    }
  }
  // top down: place << 16 | continuation
  auto code = [](uint32_t place, uint32_t sz) { return 4u * place | (sz & 1u); };
  auto place_left = [](bool is_real, uint32_t mine, uint32_t l, uint32_t r, uint32_t code_r) -> uint32_t {
    const uint32_t place = (mine >> 16) + (is_real ? 1u : 0u);
    return place << 16 | (!is_real && l != 0u && r != 0u ? code_r : mine & 0xFFFFu);
  };
  auto place_right = [](bool is_real, uint32_t mine, uint32_t l) -> uint32_t {
    return ((mine >> 16) + (is_real ? 1u : 0u) + (l >> 1)) << 16 | (mine & 0xFFFFu);
  };
  auto emit = [&](bool is_real, uint32_t hd, uint32_t mine, uint32_t sz, uint32_t l, uint32_t right) {
    if (is_real && sz != 0u) out[mine >> 16] = hd << 16 | (right + at) | ((l & 1u) ? kLeftLeaf : 0u);
  };
  uint32_t mine = kNone, lp = 0, rp = 0;
  const int parent = lane > 0 ? (lane - 1) >> 1 : 0;
  for (int l = 0; l < 5; ++l) {
    if (31 - __clz(lane + 1) == l) {
      rp = place_right(top_real, mine, top_l);
      lp = place_left(top_real, mine, top_l, top_r, code(rp >> 16, top_r));
      emit(top_real, top_head, mine, top_size, top_l, code(rp >> 16, top_r));
    }
    if (l == 4) break;
    const uint32_t fl = __shfl_sync(0xFFFFFFFFu, lp, parent), fr = __shfl_sync(0xFFFFFFFFu, rp, parent);
    if (31 - __clz(lane + 1) == l + 1) mine = (lane & 1) ? fl : fr;
  }
  const int above5 = 15 + (lane >> 1);
  const uint32_t fl = __shfl_sync(0xFFFFFFFFu, lp, above5), fr = __shfl_sync(0xFFFFFFFFu, rp, above5);
  uint32_t place[NN];
  place[0] = (lane & 1) ? fr : fl;
#pragma unroll
  for (int k = 0; k < NL - 1; ++k) {
    const uint32_t r = place_right(real[k], place[k], size[2 * k + 1]);
    place[2 * k + 2] = r;
    place[2 * k + 1] = place_left(real[k], place[k], size[2 * k + 1], size[2 * k + 2], code(r >> 16, size[2 * k + 2]));
    emit(real[k], head[k], place[k], size[k], size[2 * k + 1], code(r >> 16, size[2 * k + 2]));
  }
#pragma unroll
  for (int k = 0; k < NL; ++k) {
    const unsigned id = id_of(k);
    const uint32_t me = place[NL - 1 + k], cont = me & 0xFFFFu, pos = me >> 16;
    const uint32_t value = static_cast<uint32_t>(__float2int_rn(__uint_as_float(words[NL - 1 + k]) * a.scale));
    const unsigned last = cont == kNone ? next_tree : cont + at;
    unsigned chain = 1u;
    if (id != 0xFFFFu) {
      chain = b->chain[id];
      const unsigned term = chain ? b->pool[chain >> 8] : static_cast<unsigned>(__ffsll(static_cast<long long>(b->key[id])));
      out[pos] = value;  // (the first term is never one to subtract)
      out[pos + 1] = term << 16 | (chain_length(chain, b->key[id]) > 1 ? (4u * (pos + 2) | kLeaf) + at : last);
    }
    // the other terms of a set that takes several buckets: one lane each
    for (unsigned multi = __ballot_sync(0xFFFFFFFFu, (chain & 0xFFu) != 1u); multi; multi &= multi - 1) {
      const int src = __ffs(multi) - 1;
      const unsigned ch = __shfl_sync(0xFFFFFFFFu, chain, src), sid = __shfl_sync(0xFFFFFFFFu, id, src);
      const uint32_t p0 = __shfl_sync(0xFFFFFFFFu, pos, src), v0 = __shfl_sync(0xFFFFFFFFu, value, src);
      const unsigned l0 = __shfl_sync(0xFFFFFFFFu, last, src);
      const int n = chain_length(ch, b->key[sid]);
      for (int x = lane + 1; x < n; x += 32) {
        unsigned term;
        if (ch) {
          term = b->pool[(ch >> 8) + x];
        } else {  // its members one by one
          unsigned long long set = b->key[sid];
          for (int y = 0; y < x; ++y) set &= set - 1;
          term = static_cast<unsigned>(__ffsll(static_cast<long long>(set)));
        }
        const uint32_t p = p0 + 2 * x;
        out[p] = term & 0x80u ? 0u - v0 : v0;
        out[p + 1] = (term & 0x7Fu) << 16 | (x + 1 < n ? (4u * (p + 2) | kLeaf) + at : l0);
      }
    }
  }
}

template <int SUB>
__device__ bool find_all_sets(const ClassArgs& a, BuildShared* b, unsigned long long full, uint4* ids, uint32_t* sh_tree) {
  bool fits = true;
  for (int t = threadIdx.x >> 5; t < a.n_trees && fits; t += kT / 32) fits = find_sets<SUB>(a, b, full, t, ids + 32 * t, sh_tree);
  return fits;
}

struct ClassShared {  // what the run keeps of the compilation, and the CTA's own state
  unsigned long long sets[kMaxBuckets];  // members of every bucket
  uint16_t chunk_tree[kMaxChunks + 1];   // first tree of every chunk
  uint32_t chunk_word[kMaxChunks];       // its first word in the program
  uint32_t tree[kMaxTrees];              // words (a multiple of 4) << 16 | kRootLeaf | first word in its chunk
  int cand[kMembers];                    // the unit's candidates
  int b_eff[kMembers];
  int member[kMembers];                  // the class's members (candidates)
  ks_candidate rep;                      // one of them
  unsigned long long bar[2];
  FeatQ fq[64];
  int item, fail, build_fail, n_words, max_words, n_chunks, done[2], pending[2], abort;
};

// Compiles the ensemble for the m members of sh.member; false: does not fit (fewer members would).
__device__ bool compile_class(const ClassArgs& a, ClassShared& sh, BuildShared* b, int m, int combo, int S, uint4* ids, uint32_t* prog, uint32_t* stage) {
  const int tid = threadIdx.x;
  const FastView& fv = a.fv;
  const unsigned long long full = m == 64 ? ~0ull : (1ull << m) - 1ull;
  for (int i = tid; i < kHash; i += kT) {
    b->key[i] = 0ull;
    b->weight[i] = 0u;
  }
  // member bytes of the candidate-only rows
  const int vecs = (fv.n_cand_rows + 15) / 16;
  for (int i = tid; i < kMembers * vecs; i += kT) {
    const int mem = i % kMembers, v = i / kMembers;
    const int c = sh.member[mem < m ? mem : 0];
    const uint4 q = __ldg(reinterpret_cast<const uint4*>(fv.cand_rows + (static_cast<size_t>(combo) * a.C + c) * fv.cand_rec) + v);
    const uint32_t w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
    for (int x = 0; x < 16; ++x)
      if (16 * v + x < fv.n_cand_rows) b->bytes[16 * v + x][mem] = static_cast<uint8_t>(w[x / 4] >> (8 * (x % 4))) & 0x7F;
  }
  if (tid == 0) {
    sh.build_fail = 0;
    sh.max_words = 0;
    b->n_split = 0;
  }
  __syncthreads();
  for (int r = tid; r < fv.n_cand_rows; r += kT) {
    int lo = 127, hi = 0;
    for (int x = 0; x < m; ++x) {
      const int v = b->bytes[r][x];
      lo = min(lo, v);
      hi = max(hi, v);
    }
    b->lo[r] = static_cast<uint8_t>(lo);
    b->hi[r] = static_cast<uint8_t>(hi);
    unsigned e = 0xFFu;
    if (lo < hi) {
      uint8_t value[kSplitValues];
      int n = 0;
      int next = lo;
      while (next < 128 && n < kSplitValues) {  // the distinct bytes in ascending order
        value[n++] = static_cast<uint8_t>(next);
        int above = 128;
        for (int x = 0; x < m; ++x) {
          const int v = b->bytes[r][x];
          if (v > next && v < above) above = v;
        }
        next = above;
      }
      const int at = next == 128 ? atomicAdd(&b->n_split, 1) : kSplitRows;
      if (at < kSplitRows) {
        e = static_cast<unsigned>(at);
        for (int q = 0; q < n; ++q) {
          b->split_set[e][q] = members_right(b, r, value[q]);
          for (int x = value[q]; x < (q + 1 < n ? value[q + 1] : 128); ++x) b->split_index[e][x] = static_cast<uint8_t>(q);
        }
      }
    }
    b->split_of[r] = static_cast<uint8_t>(e);
  }
  __syncthreads();
  bool fits;
  switch (fv.depth) {
    case 5: fits = find_all_sets<0>(a, b, full, ids, sh.tree); break;
    case 6: fits = find_all_sets<1>(a, b, full, ids, sh.tree); break;
    case 7: fits = find_all_sets<2>(a, b, full, ids, sh.tree); break;
    default: fits = find_all_sets<3>(a, b, full, ids, sh.tree);
  }
  if (!fits) sh.build_fail = 1;
  __syncthreads();
  if (sh.build_fail) return false;
  assign_buckets(b, a.n_buckets, m, full, sh.sets);
  for (int t = tid >> 5; t < a.n_trees; t += kT / 32) {
    const uint32_t got = sh.tree[t];
    const int words = (tree_words(b, ids + 32 * t, static_cast<int>(got & 0x7FFFu)) + 3) & ~3;
    __syncwarp();
    if ((tid & 31) == 0) {
      sh.tree[t] = static_cast<uint32_t>(words) << 16 | (got & kRootLeaf);
      if (words > kMaxTreeWords) sh.build_fail = 1;
      atomicMax(&sh.max_words, words);
    }
  }
  __syncthreads();
  if (sh.build_fail) return false;
  // Trees are laid end to end and cut into chunks by their starts: a chunk takes the trees that
  // begin within kBufWords - (longest tree) words of one another.
  const int span = kBufWords - sh.max_words;
  int carry = 0;
  for (int t0 = 0; t0 < a.n_trees; t0 += kT) {
    const int t = t0 + tid;
    int total;
    const int at = carry + block_scan(t < a.n_trees ? static_cast<int>(sh.tree[t] >> 16) : 0, b->scan, &total);
    const int prev = at - (t > 0 && t < a.n_trees ? static_cast<int>(sh.tree[t - 1] >> 16) : 0);  // start of the tree before
    if (t < a.n_trees && at / span < kMaxChunks && (t == 0 || at / span != prev / span)) {
      sh.chunk_tree[at / span] = static_cast<uint16_t>(t);
      b->occupied[at / span] = at;  // (free again) where the chunk's words begin
    }
    if (t < a.n_trees) b->weight[t] = static_cast<unsigned>(at);  // (free again) where the tree begins
    if (t == a.n_trees - 1) {
      sh.n_chunks = at / span + 1;
      sh.n_words = at + static_cast<int>(sh.tree[t] >> 16);
      if (at / span + 1 > kMaxChunks || sh.n_words > a.n_trees * a.prog_words) sh.build_fail = 1;
      else sh.chunk_tree[at / span + 1] = static_cast<uint16_t>(a.n_trees);
    }
    carry += total;
  }
  __syncthreads();
  if (sh.build_fail) return false;
  // the code that leads to tree t (of chunk ch): its first word
  auto code_of = [&](int t, int ch) {
    return t < sh.chunk_tree[ch + 1]
               ? 4u * (b->weight[t] - static_cast<unsigned>(b->occupied[ch])) | (sh.tree[t] & kRootLeaf ? kLeaf : 0u) : kEnd;
  };
  // (a tree's words are put together in the idle chunk buffers and leave as whole lines)
  constexpr int kStage = 2 * kBufWords / (kT / 32);
  for (int t = tid >> 5; t < a.n_trees; t += kT / 32) {
    const int ch = static_cast<int>(b->weight[t]) / span, words = static_cast<int>(sh.tree[t] >> 16);
    const unsigned at = 4u * (b->weight[t] - static_cast<unsigned>(b->occupied[ch]));
    uint32_t* dst = prog + b->weight[t];
    uint32_t* out = words <= kStage ? stage + (tid >> 5) * kStage : dst;
    switch (fv.depth) {
      case 5: write_tree<0>(a, b, t, ids + 32 * t, out, at, code_of(t + S, ch)); break;
      case 6: write_tree<1>(a, b, t, ids + 32 * t, out, at, code_of(t + S, ch)); break;
      case 7: write_tree<2>(a, b, t, ids + 32 * t, out, at, code_of(t + S, ch)); break;
      default: write_tree<3>(a, b, t, ids + 32 * t, out, at, code_of(t + S, ch));
    }
    if (words <= kStage) {
      __syncwarp();
      for (int i = tid & 31; i < words / 4; i += 32) reinterpret_cast<uint4*>(dst)[i] = reinterpret_cast<const uint4*>(out)[i];
      __syncwarp();
    }
  }
  for (int i = tid; i < sh.n_chunks; i += kT) sh.chunk_word[i] = static_cast<uint32_t>(b->occupied[i]);
  asm volatile("fence.proxy.async;" ::: "memory");  // the chunks are read by bulk copies
  __threadfence();
  __syncthreads();
  // what the copies need of a tree: its words, and where it begins in its chunk
  for (int t = tid; t < a.n_trees; t += kT)
    sh.tree[t] = (sh.tree[t] & (0xFFFF0000u | kRootLeaf)) | (b->weight[t] - static_cast<unsigned>(b->occupied[b->weight[t] / span]));
  __syncthreads();
  return true;
}

// Bounded wait for a chunk: the chunks are a few microseconds apart, so a thread that waits is
// suspended by the barrier itself, not put to sleep for a fixed time.
__device__ __forceinline__ bool chunk_wait(uint32_t bar, uint32_t parity, int limit, volatile int* fail) {
  for (int i = 0; i < limit; ++i) {
    if (mbar_try_wait(bar, parity)) return true;
    if ((i & 63) == 63 && *fail) return false;
  }
  return false;
}

// Shared memory of a CTA without what the alignment of its buffers takes.
__host__ __device__ constexpr uint32_t walk_smem(int tile_rows, int n_buckets) {
  return 2u * kBufBytes + static_cast<uint32_t>(tile_rows) * kSlots + static_cast<uint32_t>(n_buckets) * 4u * kSlots;
}

// Copies chunk `ch` of the program into a buffer; one thread calls.
__device__ __forceinline__ void copy_chunk(const ClassShared& sh, const uint32_t* prog, int ch, uint32_t dst, uint32_t bar,
                                           int starve) {
  const uint32_t last = sh.tree[sh.chunk_tree[ch + 1] - 1], bytes = ((last & 0x7FFFu) + (last >> 16)) * 4u;
  fence_async_proxy();
  mbar_expect_tx(bar, bytes + (starve ? 16u : 0u));
  bulk_copy_g2s(dst, prog + sh.chunk_word[ch], bytes, bar);
}

// Follows this thread's chain through a chunk. `tile`: address of the thread's byte in row 0;
// `bucket`: of its first accumulator. Rows are kSlots bytes apart, buckets 4 kSlots. A round is two node
// visits for the threads that stand at a node and an addition for those that then stand at a leaf
// (2.7 nodes lie between two leaves on average), all under predicates: the threads of a warp are at
// different places of their trees, and branches around the parts cost more than the parts. The
// addition is atomic, since the threads that share a problem share its buckets.
__device__ __forceinline__ void run_chunk(uint32_t buf, unsigned code, uint32_t tile, uint32_t bucket, int rows, int n_buckets) {
  if (code & kEnd) return;
  uint32_t p = buf | (code & 0xFFFCu), leaf = code & kLeaf;
#ifndef KS_DEBUG_BOUNDS
  (void)rows;
  (void)n_buckets;
#define KS_NODE_VISIT                          \
  " @!L ld.shared.u32 n, [%0];\n"              \
  " prmt.b32 a, n, 0, 0x4443;\n"               \
  " mad.lo.u32 a, a, %5, %3;\n"                \
  " @!L ld.shared.u8 x, [a];\n"                \
  " prmt.b32 j, n, 0, 0x4442;\n"               \
  " setp.gt.u32 R, x, j;\n"                    \
  " lop3.b32 t, n, 0xFFFC, %2, 0xEA;\n"        \
  " add.u32 a, %0, 4;\n"                       \
  " selp.u32 m, 1, 2, R;\n"                    \
  " and.b32 m, n, m;\n"                        \
  " @!L selp.u32 %0, t, a, R;\n"               \
  " @!L setp.ne.u32 L, m, 0;\n"
  asm volatile(
      "{\n"
      " .reg .pred L, R, E;\n"
      " .reg .u32 n, a, x, j, t, m, v, w;\n"
      " mov.u32 n, 0;\n mov.u32 x, 0;\n mov.u32 w, 0;\n"
      " setp.ne.u32 L, %1, 0;\n"
      "AGAIN_%=:\n" KS_NODE_VISIT KS_NODE_VISIT
      " @L ld.shared.u32 v, [%0];\n"
      " @L ld.shared.u32 w, [%0 + 4];\n"
      " prmt.b32 a, w, 0, 0x4432;\n"
      " mad.lo.u32 a, a, %6, %4;\n"
      " @L red.shared.add.u32 [a], v;\n"
      " @L lop3.b32 %0, w, 0xFFFC, %2, 0xEA;\n"
      " and.b32 t, w, 2;\n"
      " and.b32 m, w, 1;\n"
      " setp.ne.and.u32 E, t, 0, L;\n"
      " @L setp.ne.u32 L, m, 0;\n"
      " @!E bra AGAIN_%=;\n"
      "}\n"
      : "+r"(p)
      : "r"(leaf), "r"(buf), "r"(tile), "r"(bucket), "n"(kSlots), "n"(4 * kSlots)
      : "memory");
#undef KS_NODE_VISIT
#else
  // checked build: every index against its range, and a limit on the rounds
  for (int steps = 0; KS_IDX(steps, 1 << 16) == steps; ++steps) {
    if (!leaf) {
      uint32_t n = lds_u32(buf + static_cast<uint32_t>(KS_IDX((p - buf) >> 2, kBufWords)) * 4u);
      n = static_cast<uint32_t>(KS_IDX(n >> 24, rows)) << 24 | (n & 0xFFFFFFu);
      uint32_t x;
      asm volatile("ld.shared.u8 %0, [%1];" : "=r"(x) : "r"((n >> 24) * kSlots + tile));
      const bool right = x > ((n >> 16) & 0xFFu);
      leaf = n & (right ? kLeaf : kLeftLeaf);
      p = right ? buf | (n & 0xFFFCu) : p + 4u;
    }
    if (leaf) {
      p = buf + static_cast<uint32_t>(KS_IDX((p - buf) >> 2, kBufWords - 1)) * 4u;
      const uint32_t v = lds_u32(p), w = lds_u32(p + 4u);
      atomicAdd(reinterpret_cast<uint32_t*>(__cvta_shared_to_generic(bucket + static_cast<uint32_t>(KS_IDX(w >> 16, n_buckets)) * (4u * kSlots))), v);
      if (w & kEnd) return;
      p = buf | (w & 0xFFFCu);
      leaf = w & kLeaf;
    }
  }
#endif
}

__global__ void __launch_bounds__(kT, 2)
class_walk_kernel(ks_gpu_desc desc, const __grid_constant__ ClassArgs a) {
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ ClassShared sh;
  const int tid = threadIdx.x, lane = tid & 31;
  if (a.counters[1] != 1) return;  // the per-candidate walk serves this call
  const FastView& fv = a.fv;
  uint32_t dyn;
  asm("mov.u32 %0, %%dynamic_smem_size;" : "=r"(dyn));
  const uint32_t sbase = smem_u32(smem);
  // two chunk buffers at multiples of their size, the tile, the buckets
  const uint32_t buf0 = (sbase + kBufBytes - 1) & ~static_cast<uint32_t>(kBufBytes - 1);
  unsigned char* tile = smem + (buf0 - sbase) + 2 * kBufBytes;
  uint32_t* buckets = reinterpret_cast<uint32_t*>(tile + static_cast<size_t>(a.tile_rows) * kSlots);
  BuildShared* build = reinterpret_cast<BuildShared*>(tile);
  uint4* ids = reinterpret_cast<uint4*>(a.programs + static_cast<size_t>(blockIdx.x) * a.n_trees * (512 + 4 * static_cast<size_t>(a.prog_words)));
  uint32_t* prog = reinterpret_cast<uint32_t*>(ids + 32 * static_cast<size_t>(a.n_trees));
  const uint32_t bar0 = smem_u32(&sh.bar[0]);
  volatile int* v_fail = &sh.fail;
  if (tid == 0) {
    mbar_init(bar0, 1);
    mbar_init(bar0 + 8u, 1);
    sh.fail = 0;
    sh.done[0] = sh.done[1] = 0;
    sh.pending[0] = sh.pending[1] = 0;
    sh.abort = *reinterpret_cast<volatile int*>(a.counters + 3);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (tid < 64) sh.fq[tid] = fv.feat[tid];
  __syncthreads();
  if (sh.abort) {  // a wait ran out in an earlier CTA of this call, which fails
    if (tid == 0 && a.status) atomicExch(a.status, KS_ERR_TIMEOUT);
    return;
  }
  if (buf0 - sbase + walk_smem(a.tile_rows, a.n_buckets) > dyn) {  // (the host's allowance for the alignment is too small)
    if (tid == 0 && a.status) atomicExch(a.status, KS_ERR_UNSUPPORTED);
    return;
  }
  uint32_t phases = 0;
  const int n_units = a.counters[0];
  const int last = a.first + a.count;
  for (;;) {
    // ---- the next item: a class of a unit (the fourth takes the rest) for the problems of one combination
    if (tid == 0) sh.item = atomicAdd(a.counters + 2, 1);
    __syncthreads();
    int item = sh.item;
    int combo = -1, p_begin = 0, p_end = 0;
    for (int q = 0; q < 16; ++q) {
      const int lo = max(a.counters[8 + q], a.first), hi = min(a.counters[9 + q], last);
      if (lo >= hi) continue;
      if (item < 4 * n_units) {
        combo = q;
        p_begin = lo;
        p_end = hi;
        break;
      }
      item -= 4 * n_units;
    }
    __syncthreads();
    if (combo < 0) break;
    const int2 unit = a.units[item >> 2];
    const int which = item & 3;
    const int n_prob = p_end - p_begin;
    // problems of a round: kSlots, or fewer with more threads to each, whichever takes less time
    int s_best = 1;
    for (int s = 2; s <= 4; s *= 2)
      if (rounds_of(n_prob, s) * s_best < rounds_of(n_prob, s_best) * s) s_best = s;
    const int n_slots = kSlots / s_best, S = kT / n_slots;
    if (tid < unit.y) {
      const int c = a.order[unit.x + tid];
      sh.cand[tid] = c;
      ProblemTerms t;  // the resident-block count depends on the element sizes alone
      t.bA = bytes_ab(combo >> 2);
      t.bD = bytes_d(combo & 3);
      sh.b_eff[tid] = static_cast<int>(resources(t, load_candidate(a.c + c), desc).b_eff);
    }
    __syncthreads();
    unsigned long long todo = unit.y == 64 ? ~0ull : (1ull << unit.y) - 1ull;
    int cap = min(kMembers, (a.n_buckets - 2) * 3 / 4);  // single members take a bucket each when sets have to share
    unsigned long long rest = 0ull;  // members of the class at hand that are still to be done
    for (int nth = 0;;) {
      // the unit's classes one after the other, whole: this item's, or passed over
      while (!rest && todo) {
        const int first_b = sh.b_eff[__ffsll(static_cast<long long>(todo)) - 1];
        unsigned long long all = 0ull;
        for (int i = 0; i < unit.y; ++i)
          if (((todo >> i) & 1ull) && sh.b_eff[i] == first_b) all |= 1ull << i;
        todo &= ~all;
        if (nth == which || (which == 3 && nth > 3)) rest = all;
        ++nth;
      }
      if (!rest) break;
      const int b_eff = sh.b_eff[__ffsll(static_cast<long long>(rest)) - 1];
      // all of it, or a piece that can be compiled together
      unsigned long long cls = 0ull;
      int m = 0;
      for (unsigned long long left = rest; left && m < cap; left &= left - 1) {
        cls |= left & (0ull - left);
        ++m;
      }
      __syncthreads();
      if (tid < kMembers && ((cls >> tid) & 1ull)) {
        const int at = __popcll(cls & ((1ull << tid) - 1ull));
        sh.member[at] = sh.cand[tid];
        if (at == 0) sh.rep = load_candidate(a.c + sh.cand[tid]);
      }
      __syncthreads();
      if (!compile_class(a, sh, build, m, combo, S, ids, prog, reinterpret_cast<uint32_t*>(tile - 2 * kBufBytes))) {
        __syncthreads();
        if (m <= 1) {  // cannot happen: a single member never parts
          if (tid == 0 && a.status) atomicExch(a.status, KS_ERR_UNSUPPORTED);
          return;
        }
        cap = max(1, min(cap, m) / 2);  // fewer members have fewer sets and fewer second sides
        continue;
      }
      rest &= ~cls;
      const int n_chunks = sh.n_chunks;

      for (int p0 = p_begin; p0 < p_end; p0 += n_slots) {
        const int share = tid / n_slots, q = tid % n_slots, pi = p0 + q;
        const int place = (q & 31) * 4 + (q >> 5);  // the lanes of a warp touch 32 different words of a row
        // ---- tile: per-pair and problem-only bytes of every problem --------------------------------
        const float* T = stage_thresholds(fv, 0, fv.thr_cand0, reinterpret_cast<float*>(buckets), a.n_buckets * kSlots);
        __syncthreads();
        // the columns' values, [column][slot] in the idle chunk buffers ...
        float* values = reinterpret_cast<float*>(tile - 2 * kBufBytes);
        const uint8_t* rec = a.prob_tab + static_cast<size_t>(min(pi, p_end - 1)) * kProbBytes;
        if (share == 0) {
          ProblemTerms pt;
          const uint32_t* src = reinterpret_cast<const uint32_t*>(rec + kFastMaxProbRows);
          uint32_t* dst = reinterpret_cast<uint32_t*>(&pt);
#pragma unroll
          for (int i = 0; i < static_cast<int>(sizeof(ProblemTerms) / 4); ++i) dst[i] = __ldg(src + i);
          pair_columns<true>(pt, sh.rep, desc, b_eff, [&](int col, float v) { values[pair_slot(col) * kSlots + q] = v; });
        }
        // ... (the other threads copy the problem-only bytes) ...
        for (int r = share - 1; r >= 0 && r < (fv.n_prob_rows + 3) / 4; r += S - 1) {
          const uint32_t w = __ldg(reinterpret_cast<const uint32_t*>(rec) + r);
#pragma unroll
          for (int x = 0; x < 4; ++x)
            if (4 * r + x < fv.n_prob_rows) tile[(fv.n_pair_rows + 4 * r + x) * kSlots + place] = static_cast<uint8_t>(w >> (8 * x));
        }
        __syncthreads();
        // ... and their bytes, a column at a time
        for (int i = share; i < kPairCols; i += S) {
          const FeatQ& f = sh.fq[pair_col(i)];
          quantise(f, T + f.thr0, values[i * kSlots + q], false,
                   [&](int row, uint8_t byte) { tile[KS_IDX(row, a.tile_rows) * kSlots + place] = byte & 0x7F; });
        }
        __syncthreads();
        // ---- run -----------------------------------------------------------------------------------
        if (tid == 0)
          for (int ch = 0; ch < 2 && ch < n_chunks; ++ch) {
            copy_chunk(sh, prog, ch, buf0 + ch * kBufBytes, bar0 + 8u * ch, fv.starve);
            sh.pending[ch] = 1;
          }
        for (int i = tid; i < a.n_buckets * (kSlots / 4); i += kT) reinterpret_cast<uint4*>(buckets)[i] = make_uint4(0, 0, 0, 0);
        __syncthreads();
        const bool live = pi < p_end;
        for (int ch = 0; ch < n_chunks; ++ch) {
          const int b = ch & 1;
          const uint32_t bar = bar0 + 8u * b, buf = buf0 + b * kBufBytes;
          const bool here = !*v_fail && chunk_wait(bar, (phases >> b) & 1u, fv.wait_limit, v_fail);
          if (!__all_sync(0xFFFFFFFFu, here)) {  // the warp gives up together
            if (!*v_fail) {
              sh.fail = 1;
              atomicExch(a.counters + 3, 1);
              if (a.status) atomicExch(a.status, KS_ERR_TIMEOUT);
            }
            break;
          }
          phases ^= 1u << b;
          if (live) {
            const int t = sh.chunk_tree[ch] + share;  // the share's first tree of the chunk
            const uint32_t w = sh.tree[t < a.n_trees ? t : 0];
            run_chunk(buf, t < sh.chunk_tree[ch + 1] ? 4u * (w & 0x7FFFu) | (w & kRootLeaf ? kLeaf : 0u) : kEnd,
                      smem_u32(tile) + place, smem_u32(buckets) + q * 4, a.tile_rows, a.n_buckets);
          }
          __syncwarp();
          if (lane == 0 && atomicAdd(&sh.done[b], 1) == kT / 32 - 1) {  // the last warp to leave the buffer fills it again
            sh.done[b] = sh.pending[b] = 0;
            if (ch + 2 < n_chunks && !*v_fail) {
              copy_chunk(sh, prog, ch + 2, buf, bar, fv.starve);
              sh.pending[b] = 1;
            }
          }
        }
        __syncthreads();
        if (*v_fail) {  // give copies in flight the time to land, then leave
          if (tid == 0) {
            for (int b = 0; b < 2; ++b) {
              if (!sh.pending[b]) continue;
              if (fv.starve) {
                for (int i = 0; i < 64; ++i) __nanosleep(kSleepNs);
              } else {
                mbar_wait_bounded(bar0 + 8u * b, (phases >> b) & 1u, fv.wait_limit, &sh.abort);
              }
            }
          }
          __syncthreads();
          return;
        }
        // ---- finish: every member's score --------------------------------------------------------
        // membership as factors of 32 members at a time, in the idle chunk buffers: [bucket][32]
        uint32_t* factor = reinterpret_cast<uint32_t*>(tile - 2 * kBufBytes);
        for (int m0 = 0; m0 < m; m0 += 32) {
          __syncthreads();
          for (int i = tid; i < a.n_buckets * 32; i += kT)
            factor[i] = static_cast<uint32_t>(sh.sets[i / 32] >> (m0 + i % 32)) & 1u;
          __syncthreads();
          if (!live) continue;
          for (int i0 = share * 8; i0 < 32 && m0 + i0 < m; i0 += 8 * S) {
            uint32_t acc[8] = {0u, 0u, 0u, 0u, 0u, 0u, 0u, 0u};
            for (int b = 0; b < a.n_buckets; ++b) {
              const uint32_t v = buckets[b * kSlots + q];
              const uint4 f0 = reinterpret_cast<const uint4*>(factor + b * 32 + i0)[0];
              const uint4 f1 = reinterpret_cast<const uint4*>(factor + b * 32 + i0)[1];
              acc[0] += v * f0.x; acc[1] += v * f0.y; acc[2] += v * f0.z; acc[3] += v * f0.w;
              acc[4] += v * f1.x; acc[5] += v * f1.y; acc[6] += v * f1.z; acc[7] += v * f1.w;
            }
#pragma unroll
            for (int i = 0; i < 8; ++i)
              if (m0 + i0 + i < m)
                a.plane[static_cast<size_t>(sh.member[m0 + i0 + i]) * a.pitch + (pi - a.first)] =
                    (fv.base + __int2float_rn(static_cast<int>(acc[i])) * a.unscale) + 0.0f;
          }
        }
        __syncthreads();  // before the buffers are filled again
      }
      // hand the program's memory from the copies back to ordinary stores
      asm volatile("fence.proxy.async;" ::: "memory");
      __syncthreads();
    }
  }
}

// ------------------------------------------------------------------------------------------
// ranking of the score plane
// ------------------------------------------------------------------------------------------

// One thread ranks one problem against block y's share of its candidates, in a sorted list of k keys
// in shared memory ([k][threads]). A warp reads 32 neighbouring scores of the plane per candidate.
constexpr int kRankThreads = 128;
__global__ void __launch_bounds__(kRankThreads)
class_rank_kernel(const float* __restrict__ plane, int pitch, int first, int count, const int* __restrict__ prob_order,
                  const int* __restrict__ counters, int C, const int64_t* __restrict__ seg_off,
                  const int32_t* __restrict__ seg_idx, int rows, int k, unsigned long long* __restrict__ partial) {
  extern __shared__ unsigned long long s_keys[];
  if (counters[1] != 1) return;
  const int tid = threadIdx.x, q = blockIdx.x * kRankThreads + tid, nblk = gridDim.y;
  if (q >= count) return;
  unsigned long long* list = s_keys + tid;
  for (int j = 0; j < k; ++j) list[j * kRankThreads] = 0ull;
  const int prob = prob_order[first + q];
  const int64_t lo = seg_off ? seg_off[prob] : 0;
  const int64_t len = seg_off ? seg_off[prob + 1] - lo : C;
  unsigned long long worst = 0ull;
  auto insert = [&](unsigned long long key) {
    if (key <= worst) return;
    int j = k - 1;
    while (j > 0) {
      const unsigned long long up = list[(j - 1) * kRankThreads];
      if (up >= key) break;
      list[j * kRankThreads] = up;
      --j;
    }
    list[j * kRankThreads] = key;
    worst = list[(k - 1) * kRankThreads];
  };
  const float* col = plane + q;
  for (int64_t start = static_cast<int64_t>(blockIdx.y) * rows; start < len; start += static_cast<int64_t>(nblk) * rows) {
    const int64_t stop = start + rows < len ? start + rows : len;
    constexpr int kAhead = 8;
    for (int64_t r = start; r < stop; r += kAhead) {
      int c[kAhead];
      float v[kAhead];
#pragma unroll
      for (int i = 0; i < kAhead; ++i) c[i] = r + i < stop ? (seg_idx ? __ldg(seg_idx + lo + r + i) : static_cast<int>(r) + i) : -1;
#pragma unroll
      for (int i = 0; i < kAhead; ++i) v[i] = c[i] >= 0 ? __ldcs(col + static_cast<size_t>(c[i]) * pitch) : 0.0f;
#pragma unroll
      for (int i = 0; i < kAhead; ++i)
        if (c[i] >= 0) insert(make_key(v[i], c[i]));
    }
  }
  unsigned long long* out = partial + (static_cast<size_t>(prob) * nblk + blockIdx.y) * k;
  for (int j = 0; j < k; ++j) out[j] = list[j * kRankThreads];
}

size_t up256(size_t v) { return (v + 255) / 256 * 256; }

// Buckets of a CTA: what its half of an SM's shared memory holds beside the chunk buffers and the
// tile. (Two CTAs: one compiles or fills its tile while the other walks.)
constexpr int kCtas = 2;
// up to here a buffer's alignment may cost: the CTA's shared memory starts with 1 KB of the system's and
// the static part
constexpr int kAlignRoom = kBufBytes - 1024 - static_cast<int>(sizeof(ClassShared)) + 512;
int bucket_count(int tile_rows) {
  const int64_t room = 228 * 1024 / kCtas - 1024 - static_cast<int64_t>(sizeof(ClassShared)) - kAlignRoom - 2 * kBufBytes -
                       static_cast<int64_t>(tile_rows) * kSlots;
  const int64_t n = room / (4 * kSlots);
  return static_cast<int>(n < kMaxBuckets ? n : kMaxBuckets);
}
size_t program_bytes(const GbdtModel& g) {
  return static_cast<size_t>(kCtas) * kSms * g.n_trees * (512 + 4 * static_cast<size_t>(std::max(kMinProg, g.class_words)));
}
int batch_problems(int P, int C) {
  const int64_t n = static_cast<int64_t>(kPlaneBytes / (4 * static_cast<size_t>(C))) / kSlots * kSlots;
  return static_cast<int>(std::min<int64_t>(n, P));  // (classes_apply: at least kSlots fit)
}
size_t problem_sort_bytes(int P) {
  size_t bytes = 0;
  cub::DeviceRadixSort::SortPairs(nullptr, bytes, static_cast<const unsigned*>(nullptr), static_cast<unsigned*>(nullptr),
                                  static_cast<const int*>(nullptr), static_cast<int*>(nullptr), P, 0, kProblemKeyBits);
  return bytes;
}

}  // namespace

// Leaf values as integers: the shift s with |leaf| * 2^s rounded to an integer, such that no sum of one
// leaf a tree leaves 32 bits. A leaf is then off by at most 2^-(s+1), where adding it to a float sum of
// size S is off by up to 2^-25 S. With B the sum of the trees' largest leaves (2^s > 2^30 / B) and V the
// standard deviation of a sum whose every tree ends in a random leaf, the integer sum is the more
// accurate one while B <= 200 V: its error is at most B 2^-31 / sqrt(3) a leaf in the mean square,
// 0.29 * 200 / 64 = 0.9 of the float's V 2^-25. (500 trees of normal leaves: B = 63 V; 1,000: 89 V.)
// kNoFixed for any other ensemble.
int fixed_point_shift(int n_trees, const int64_t* off, const ks_node_host* nodes) {
  double largest = 0.0, variance = 0.0;
  for (int t = 0; t < n_trees; ++t) {
    double top = 0.0, sum = 0.0, squares = 0.0;
    int64_t n = 0;
    for (int64_t i = off[t]; i < off[t + 1]; ++i) {
      if (nodes[i].feat != 0xFFFF) continue;
      const double v = nodes[i].thr_or_leaf;
      top = std::max(top, std::fabs(v));
      sum += v;
      squares += v * v;
      ++n;
    }
    largest += top;
    variance += squares / n - (sum / n) * (sum / n);
  }
  if (!(largest > 0.0) || !(largest <= 200.0 * std::sqrt(std::max(variance, 0.0)))) return kNoFixed;
  // rounding adds half a unit a tree at most
  int s = 0;
  std::frexp(static_cast<double>((1u << 31) - 1 - n_trees) / largest, &s);
  --s;
  return s >= -100 && s <= 100 ? s : kNoFixed;
}

// Words that the largest tree may take when it is compiled for a single candidate: a candidate-only
// node leaves one of its subtrees (whichever is larger), any other both. A multiple of 32.
int class_tree_words(int n_trees, const int64_t* off, const ks_node_host* nodes) {
  int most = 0;
  std::vector<int> words;
  bool drops[64];  // columns whose nodes leave one subtree
  for (int f = 0; f < 64; ++f) drops[f] = f < KS_F && feat_class(f) == 1;
  for (int t = 0; t < n_trees; ++t) {
    const int64_t n = off[t + 1] - off[t];
    words.assign(static_cast<size_t>(n), 2);
    for (int64_t i = n - 1; i >= 0; --i) {  // children come after their parent
      const ks_node_host& nd = nodes[off[t] + i];
      if (nd.feat == 0xFFFF) continue;
      const int l = words[nd.left], r = words[nd.left + 1];
      words[i] = drops[nd.feat & 63] ? std::max(l, r) : 1 + l + r;
    }
    most = std::max(most, words[0]);
  }
  return (most + 31) / 32 * 32;
}

// Batches this path may serve (whether it does is decided on the device, where the number of units is
// known): enough problems to pay for compiling even if every unit were full (more than 100), enough
// candidates for classes to have members and few enough for a round of problems' scores to fit the plane,
// and a model whose words fit the compiled form. A batch refused here costs nothing; one refused on the
// device has paid for its preparation and for the memory.
bool classes_apply(const GbdtModel& g, int P, int C, int64_t pairs) {
  if (!g.fast || P < 1 || C < 4096 || pairs / P < 2048 || C > static_cast<int64_t>(kPlaneBytes / (4 * kSlots))) return false;
  if (!walk_pays(walk_cost((C + kMembers - 1) / kMembers, P), pairs)) return false;
  if (g.fast_depth < 5 || g.fast_depth > 8 || g.n_trees > kMaxTrees || g.fixed_shift == kNoFixed) return false;
  const int rows = g.n_pair_rows + g.n_prob_rows;
  if (rows > 255 || g.n_pair_rows < 1) return false;
  return walk_smem(rows, bucket_count(rows)) - 2 * kBufBytes >= sizeof(BuildShared);
}

// units | counters | problem keys, indices (twice, for the sort) | sort workspace | problem rows |
// programs | score plane
size_t classes_scratch_bytes(const GbdtModel& g, int P, int C) {
  return up256(sizeof(int2) * C) + 256 + 4 * up256(sizeof(int) * P) + up256(problem_sort_bytes(P)) +
         up256(static_cast<size_t>(P) * kProbBytes) + up256(program_bytes(g)) +
         up256(sizeof(float) * static_cast<size_t>(C) * batch_problems(P, C)) + 256;
}

namespace {
// The parts of a call's scratch memory.
struct ClassScratch {
  int2* units;
  int* counters;
  unsigned *keys_in, *keys;
  int *idx_in, *order;
  void* sort_mem;
  uint8_t *prob_tab, *programs;
  float* plane;
};
ClassScratch class_scratch(const GbdtModel& g, int P, int C, void* mem) {
  char* q = static_cast<char*>(mem);
  auto take = [&](size_t bytes) {
    char* at = q;
    q += up256(bytes);
    return at;
  };
  ClassScratch s;
  s.units = reinterpret_cast<int2*>(take(sizeof(int2) * C));
  s.counters = reinterpret_cast<int*>(take(256));
  s.keys_in = reinterpret_cast<unsigned*>(take(sizeof(int) * P));
  s.keys = reinterpret_cast<unsigned*>(take(sizeof(int) * P));
  s.idx_in = reinterpret_cast<int*>(take(sizeof(int) * P));
  s.order = reinterpret_cast<int*>(take(sizeof(int) * P));
  s.sort_mem = take(problem_sort_bytes(P));
  s.prob_tab = reinterpret_cast<uint8_t*>(take(static_cast<size_t>(P) * kProbBytes));
  s.programs = reinterpret_cast<uint8_t*>(take(program_bytes(g)));
  s.plane = reinterpret_cast<float*>(q);
  return s;
}
}  // namespace

cudaError_t prepare_classes(const ks_gpu_desc& desc, const GbdtModel& g, const ks_problem* d_p, int P,
                            const ks_candidate* d_c, int C, const ClassCall& call, cudaStream_t stream,
                            int64_t* launches, const FastWait* wait, const int** path) {
  const ClassScratch s = class_scratch(g, P, C, call.scratch);
  *path = s.counters + 1;
  cudaError_t e = cudaMemsetAsync(s.counters, 0, 256, stream);
  if (e != cudaSuccess) return e;
  units_kernel<<<(C + 255) / 256, 256, 0, stream>>>(d_c, C, call.order, s.units, s.counters);
  if (P <= kCountProblems) {
    problem_order_kernel<<<(P + 255) / 256, 256, 0, stream>>>(d_p, P, s.keys, s.order);
  } else {
    problem_keys_kernel<<<(P + 255) / 256, 256, 0, stream>>>(d_p, P, s.keys_in, s.idx_in);
    size_t sort_bytes = problem_sort_bytes(P);
    e = cub::DeviceRadixSort::SortPairs(s.sort_mem, sort_bytes, s.keys_in, s.keys, s.idx_in, s.order, P, 0,
                                        kProblemKeyBits, stream);
    if (e != cudaSuccess) return e;
  }
  problem_rows_kernel<<<P, 64, 0, stream>>>(desc, d_p, P, s.order, s.keys, make_view(g, nullptr), s.prob_tab, s.counters);
  choose_path_kernel<<<1, 1, 0, stream>>>(call.pairs, s.counters, wait->words + kWordServed);
  *launches += 4;
  return cudaGetLastError();
}

cudaError_t launch_classes(const ks_gpu_desc& desc, const GbdtModel& g, int P, const ks_candidate* d_c, int C,
                           const uint8_t* cand_rows, const int64_t* seg_off, const int32_t* seg_idx, int nblk,
                           int rows_per_block, int k, unsigned long long* partial, const ClassCall& call, int* status,
                           cudaStream_t stream, int64_t* launches, const FastWait* wait) {
  const ClassScratch s = class_scratch(g, P, C, call.scratch);
  ClassArgs a{};
  a.fv = make_view(g, wait);
  a.fv.cand_rows = cand_rows;
  a.nc_shift = 0;
  while ((1 << a.nc_shift) < g.block_cands) ++a.nc_shift;
  a.n_trees = g.n_trees;
  a.scale = std::ldexp(1.0f, g.fixed_shift);
  a.unscale = std::ldexp(1.0f, -g.fixed_shift);
  a.tile_rows = g.n_pair_rows + g.n_prob_rows;
  a.n_buckets = bucket_count(a.tile_rows);
  a.prog_words = std::max(kMinProg, g.class_words);
  a.c = d_c;
  a.C = C;
  a.P = P;
  a.order = call.order;
  a.units = s.units;
  a.counters = s.counters;
  a.prob_order = s.order;
  a.prob_tab = s.prob_tab;
  a.programs = s.programs;
  a.plane = s.plane;
  a.status = status;
  a.pitch = batch_problems(P, C);
  const size_t smem = kAlignRoom + walk_smem(a.tile_rows, a.n_buckets);
  cudaError_t e = ensure_dynamic_smem(reinterpret_cast<const void*>(&class_walk_kernel), smem);
  if (e != cudaSuccess) return e;
  for (int first = 0; first < P; first += a.pitch) {
    a.first = first;
    a.count = std::min(a.pitch, P - first);
    if (first > 0) {
      e = cudaMemsetAsync(s.counters + 2, 0, sizeof(int), stream);
      if (e != cudaSuccess) return e;
    }
    class_walk_kernel<<<kCtas * kSms, kT, smem, stream>>>(desc, a);
    class_rank_kernel<<<dim3((a.count + kRankThreads - 1) / kRankThreads, nblk), kRankThreads,
                        sizeof(unsigned long long) * k * kRankThreads, stream>>>(
        a.plane, a.pitch, first, a.count, s.order, s.counters, C, seg_off, seg_idx, rows_per_block, k, partial);
    *launches += 2;
  }
  return cudaGetLastError();
}

#ifdef KS_DEBUG_BOUNDS
int class_bounds_line() {
  int v = 0;
  cudaMemcpyFromSymbol(&v, g_bounds_line, sizeof(int));
  return v;
}
void class_bounds_clear() {
  const int z = 0;
  cudaMemcpyToSymbol(g_bounds_line, &z, sizeof(int));
}
#else
int class_bounds_line() { return -1; }
void class_bounds_clear() {}
#endif

}  // namespace ks
