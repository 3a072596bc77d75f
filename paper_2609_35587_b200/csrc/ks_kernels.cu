// Generic kernels of libks: the standalone feature map, the standalone scorers, the generic
// fused featurize + score + top-k kernel (any tree shape), the linear scorer and the
// per-problem merge of partial top-k lists. The quantised fast path for complete trees lives
// in ks_gbdt_fast.cu.
#include <cuda_bf16.h>

#include <algorithm>

#include <cstdlib>
#include <cstring>
#include <new>

#include "ks_features.cuh"
#include "ks_internal.h"
#include "ks_memo.cuh"
#include "ks_topk.cuh"

namespace ks {

// ------------------------------------------------------------------------------------------
// block -> (problem, chunk) mapping shared by the pair kernels
// ------------------------------------------------------------------------------------------

struct PairMap {
  int P, C, nblk;           // nblk blocks per problem
  int rows_per_block;       // rows one block covers per pass
  const int64_t* seg_off;   // null = dense
  const int32_t* seg_idx;
};

__device__ __forceinline__ void segment_of(const PairMap& m, int prob, int64_t& lo, int64_t& len) {
  if (m.seg_off) {
    lo = m.seg_off[prob];
    len = m.seg_off[prob + 1] - lo;
  } else {
    lo = static_cast<int64_t>(prob) * m.C;
    len = m.C;
  }
}

__device__ __forceinline__ int pool_index(const PairMap& m, int64_t lo, int64_t r) {
  return m.seg_off ? m.seg_idx[lo + r] : static_cast<int>(r);
}

// ------------------------------------------------------------------------------------------
// ks_featurize: one thread per pair, rows staged through shared memory for coalesced stores
// ------------------------------------------------------------------------------------------

// The 13 problem-only columns are the same in every row of a block; the other 50 are staged, which
// leaves room for four blocks an SM, and a row leaves as one 256-byte store of the warp (lane l writes
// columns 2 l and 2 l + 1). A block takes several slabs of a problem's rows, since its one thread that
// evaluates the problem's terms keeps the others waiting. 300 problems x 7,000 rows: 147 us with all 64
// columns staged, 4-byte stores and a block per 256 rows, 117 us like this (the stores alone: 85 us).
constexpr int kStaged = kCandCols + kPairCols, kStagedStride = kStaged + 1;  // (odd: rows start on different banks)
__host__ __device__ constexpr int staged_slot(int col) {
  return feat_class(col) == 1 ? cand_slot(col) : kCandCols + pair_slot(col);
}

template <bool kAligned>  // out starts on an 8-byte boundary (tested per store: 122 us instead of 117)
__global__ void __launch_bounds__(kBlock, 4)
featurize_kernel(const __grid_constant__ ks_gpu_desc desc, const ks_problem* __restrict__ p,
                 const ks_candidate* __restrict__ c, PairMap map, float* __restrict__ out) {
  extern __shared__ float s_tile[];  // [kBlock][kStagedStride]
  __shared__ ProblemTerms s_pt;
  __shared__ float s_pc[64];
  const int prob = blockIdx.x / map.nblk, chunk = blockIdx.x % map.nblk;
  int64_t lo, len;
  segment_of(map, prob, lo, len);
  if (threadIdx.x == 0) {
    problem_terms(p[prob], desc, s_pt);
    problem_columns(s_pt, [&](int col, float v) { s_pc[col] = v; });
    s_pc[KS_F] = 0.0f;
  }
  __syncthreads();
  // every warp stages and stores its own 32 rows, so that one warp's stores overlap another's
  // arithmetic without block-wide barriers
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  float* w_tile = s_tile + warp * 32 * kStagedStride;
  const int c0 = 2 * lane, c1 = 2 * lane + 1;
  const bool fixed0 = feat_class(c0) == 0, fixed1 = c1 == KS_F || feat_class(c1) == 0;
  const float v0 = fixed0 ? s_pc[c0] : 0.0f, v1 = fixed1 ? s_pc[c1] : 0.0f;
  const int at0 = fixed0 ? 0 : staged_slot(c0), at1 = fixed1 ? 0 : staged_slot(c1);
  for (int64_t start = static_cast<int64_t>(chunk) * kBlock; start < len;
       start += static_cast<int64_t>(map.nblk) * kBlock) {
    const int64_t w0 = start + warp * 32;  // first row of this warp
    if (w0 >= len) break;
    if (w0 + lane < len) {
      const ks_candidate cand = load_candidate(c + pool_index(map, lo, w0 + lane));
      float* row = w_tile + lane * kStagedStride;
      featurize_pair(s_pt, cand, desc, [&](int col, float v) {
        if (col < KS_F && feat_class(col) != 0) row[staged_slot(col)] = v;
      });
    }
    __syncwarp();
    const int n_rows = (len - w0 < 32) ? static_cast<int>(len - w0) : 32;
    float* dst = out + (lo + w0) * kRow + c0;
#pragma unroll 8
    for (int r = 0; r < n_rows; ++r) {
      const float a = w_tile[r * kStagedStride + at0], b = w_tile[r * kStagedStride + at1];
      const float2 v = make_float2(fixed0 ? v0 : a, fixed1 ? v1 : b);
      if (kAligned) {
        __stcs(reinterpret_cast<float2*>(dst + r * kRow), v);
      } else {
        __stcs(dst + r * kRow, v.x);
        __stcs(dst + r * kRow + 1, v.y);
      }
    }
    __syncwarp();
  }
}

// Dense form (every problem against the whole pool). The work is cut into items of 32
// candidates x 1 problem, ordered candidate slab first, and every warp of the grid takes a
// contiguous run of items of equal length (to within one), so that no SM idles in a last
// partial wave. A lane keeps its candidate, the candidate-only columns and the candidate's
// resident-block count in registers while the problems of the run change (re-evaluated only
// when the element-type combination does); the problem-only terms and columns come from a
// table written once per call. Only the per-pair columns are arithmetic per pair. Same
// functions, same operands: the rows are bit-identical to featurize_pair's.
struct ProblemEntry {
  ProblemTerms t;
  float pc[16];  // the problem-only columns, in column order
};

__global__ void __launch_bounds__(128)
problem_table_kernel(ks_gpu_desc desc, const ks_problem* __restrict__ p, int P, ProblemEntry* __restrict__ tab) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= P) return;
  ProblemEntry e;
  problem_terms(p[i], desc, e.t);
  ks_candidate dummy{};
  dummy.tile_m = dummy.tile_n = dummy.tile_k = 64;
  dummy.stages = dummy.cluster_m = dummy.cluster_n = 1;
#pragma unroll
  for (int q = 0; q < 16; ++q) e.pc[q] = 0.0f;
  featurize_pair(e.t, dummy, desc, [&](int col, float v) {
    if (feat_class(col) == 0) e.pc[prob_slot(col)] = v;
  });
  tab[i] = e;
}

__global__ void __launch_bounds__(kBlock, 3)
featurize_dense_kernel(ks_gpu_desc desc, const ProblemEntry* __restrict__ tab, const ks_candidate* __restrict__ c,
                       int P, int C, float* __restrict__ out) {
  extern __shared__ float s_tile[];  // [kBlock][65], one 32-row slab per warp
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  float* row = s_tile + (warp * 32 + lane) * 65;
  const float* w_tile = s_tile + warp * 32 * 65;
  const int64_t n_warps = static_cast<int64_t>(gridDim.x) * (kBlock / 32);
  const int64_t me = static_cast<int64_t>(blockIdx.x) * (kBlock / 32) + warp;
  const int64_t total = static_cast<int64_t>((C + 31) / 32) * P;
  const int64_t i_end = total * (me + 1) / n_warps;
  ks_candidate cand{};
  float cc[29];
  long long b_eff = 1;
  int slab_prev = -1, combo_prev = -1, w0 = 0, n_rows = 0;
  bool live = false;
#pragma unroll 1
  for (int64_t i = total * me / n_warps; i < i_end; ++i) {
    const int slab = static_cast<int>(i / P), prob = static_cast<int>(i - static_cast<int64_t>(slab) * P);
    if (slab != slab_prev) {
      slab_prev = slab;
      combo_prev = -1;
      w0 = slab * 32;
      n_rows = C - w0 < 32 ? C - w0 : 32;
      live = lane < n_rows;
      cand = c[live ? w0 + lane : C - 1];
    }
    const ProblemEntry& e = tab[prob];
    const ProblemTerms t = e.t;
    const int combo = t.dtype_ab * 4 + t.dtype_d;
    if (combo != combo_prev) {  // the same for every lane
      combo_prev = combo;
      b_eff = resources(t, cand, desc).b_eff;
      featurize_pair(t, cand, desc, [&](int col, float v) {
        if (feat_class(col) == 1) cc[cand_slot(col)] = v;
      });
    }
#pragma unroll
    for (int col = 0; col < KS_F; ++col) {
      if (feat_class(col) == 1) row[col] = cc[cand_slot(col)];
      if (feat_class(col) == 0) row[col] = __ldg(&e.pc[prob_slot(col)]);
    }
    row[KS_F] = 0.0f;
    pair_columns<true>(t, cand, desc, b_eff, [&](int col, float v) { row[col] = v; });
    __syncwarp();
    float* dst = out + (static_cast<int64_t>(prob) * C + w0) * kRow;
    for (int q = lane; q < n_rows * kRow; q += 32) __stcs(dst + q, w_tile[(q >> 6) * 65 + (q & 63)]);
    __syncwarp();
  }
}

// ------------------------------------------------------------------------------------------
// generic tree walk: nodes from global memory (read-only path), features from a shared tile
// laid out [column][thread] so that a warp's reads of one column are conflict-free
// ------------------------------------------------------------------------------------------

__device__ __forceinline__ DevNode load_node(const DevNode* p) {
  const uint2 u = __ldg(reinterpret_cast<const uint2*>(p));
  DevNode n;
  n.v = __uint_as_float(u.x);
  n.feat = static_cast<uint16_t>(u.y & 0xFFFFu);
  n.left = static_cast<uint16_t>(u.y >> 16);
  return n;
}

// returns base + sum of leaves; optionally records the leaf node index of every tree
__device__ __forceinline__ float walk_ensemble(const DevNode* __restrict__ nodes,
                                               const int* __restrict__ roots, int n_trees, float base,
                                               const float* s_cols /* [64][kBlock], this thread's lane */,
                                               uint16_t* leaf_out) {
  float s = base;
  for (int t = 0; t < n_trees; ++t) {
    const DevNode* tree = nodes + roots[t];
    int i = 0;
    DevNode nd = load_node(tree);
#pragma unroll 1
    for (int d = 0; d <= KS_MAX_DEPTH && nd.feat != 0xFFFFu; ++d) {
      const float x = s_cols[(nd.feat & 0x7FFFu) * kBlock];
      int right;
      if (nd.feat & 0x8000u) {  // partition split: v's bits are the set of levels that go right
        const unsigned code = static_cast<unsigned>(__float2int_rz(x));
        right = code < 32u ? (__float_as_uint(nd.v) >> code) & 1u : 0;
      } else {
        right = x < nd.v ? 0 : 1;
      }
      i = nd.left + right;
      nd = load_node(tree + i);
    }
    if (leaf_out) leaf_out[t] = static_cast<uint16_t>(i);
    s += nd.v;
  }
  return s;
}

__global__ void __launch_bounds__(kBlock)
score_gbdt_kernel(const DevNode* __restrict__ nodes, const int* __restrict__ roots, int n_trees,
                  float base, const float* __restrict__ feat, int64_t rows, float* __restrict__ scores,
                  uint16_t* __restrict__ leaf_idx) {
  extern __shared__ float s_cols[];  // [64][kBlock]
  const int64_t r = static_cast<int64_t>(blockIdx.x) * kBlock + threadIdx.x;
  if (r < rows) {
    const float4* src = reinterpret_cast<const float4*>(feat + r * kRow);
#pragma unroll 4
    for (int q = 0; q < kRow / 4; ++q) {
      const float4 v = __ldg(src + q);
      s_cols[(4 * q + 0) * kBlock + threadIdx.x] = v.x;
      s_cols[(4 * q + 1) * kBlock + threadIdx.x] = v.y;
      s_cols[(4 * q + 2) * kBlock + threadIdx.x] = v.z;
      s_cols[(4 * q + 3) * kBlock + threadIdx.x] = v.w;
    }
    const float s = walk_ensemble(nodes, roots, n_trees, base, s_cols + threadIdx.x,
                                  leaf_idx ? leaf_idx + r * n_trees : nullptr);
    scores[r] = s + 0.0f;
  }
}

// ------------------------------------------------------------------------------------------
// ks_score with the linear scorer (one weight layer): one thread per row
// ------------------------------------------------------------------------------------------

// The model's input positions in order: weight (bf16), mean, deviation, by value.
struct LinearRow {
  float w[KS_F_ONEHOT], mu[KS_F_ONEHOT], sigma[KS_F_ONEHOT];
  float bias;
};

template <bool kOneHot>
__global__ void __launch_bounds__(kBlock)
score_linear_kernel(const __grid_constant__ LinearRow m, const float* __restrict__ feat, int64_t rows,
                    float* __restrict__ scores) {
  const int64_t r = static_cast<int64_t>(blockIdx.x) * kBlock + threadIdx.x;
  if (r >= rows) return;
  const float4* src = reinterpret_cast<const float4*>(feat + r * kRow);
  float x[kRow];
#pragma unroll
  for (int q = 0; q < kRow / 4; ++q) {
    const float4 v = __ldg(src + q);
    x[4 * q] = v.x; x[4 * q + 1] = v.y; x[4 * q + 2] = v.z; x[4 * q + 3] = v.w;
  }
  float acc = 0.0f;
#pragma unroll
  for (int pos = 0; pos < (kOneHot ? 73 : KS_F); ++pos) {
    float v;
    if (!kOneHot) {
      v = x[pos];
    } else if (pos < 59) {  // the columns other than 5, 9, 17, 18 in order, then the level indicators
      v = x[pos + (pos >= 5) + (pos >= 8) + 2 * (pos >= 15)];
    } else {
      const int q = pos - 59;  // operand type 0..3, activation 4..6, kernel sched 7..10, epilogue sched 11..13
      const int col = q < 4 ? 5 : (q < 7 ? 9 : (q < 11 ? 17 : 18));
      const int level = q < 4 ? q : (q < 7 ? q - 4 : (q < 11 ? q - 7 : q - 11));
      v = __float2int_rz(x[col]) == level ? 1.0f : 0.0f;
    }
    if (!isfinite(v)) v = 0.0f;
    acc = fmaf(m.w[pos], __bfloat162float(__float2bfloat16_rn(__fdiv_rn(__fsub_rn(v, m.mu[pos]), m.sigma[pos]))), acc);
  }
  scores[r] = (acc + m.bias) + 0.0f;
}

// ------------------------------------------------------------------------------------------
// generic fused select: featurize a sub-tile of kBlock pairs into shared memory, score it,
// keep one key per thread per sub-tile, rank the block's keys, write a partial top-k list.
// ------------------------------------------------------------------------------------------

template <bool kStatic>  // tree ensemble, or the static sampling score (no feature tile)
__global__ void __launch_bounds__(kBlock)
select_generic_kernel(ks_gpu_desc desc, const ks_problem* __restrict__ p, ks_problem p_value,
                      int use_value, const ks_candidate* __restrict__ c, PairMap map, int sub_tiles,
                      const DevNode* __restrict__ nodes, const int* __restrict__ roots, int n_trees,
                      float base, int k, unsigned long long* __restrict__ partial /* [P][nblk][k] */) {
  extern __shared__ __align__(16) unsigned char s_raw[];
  float* s_cols = reinterpret_cast<float*>(s_raw);  // [64][kBlock]
  __shared__ ProblemTerms s_pt;
  __shared__ unsigned long long s_warp[kBlock / 32 * KS_MAX_K];
  __shared__ unsigned long long s_list[KS_MAX_K];

  const int prob = blockIdx.x / map.nblk, chunk = blockIdx.x % map.nblk;
  int64_t lo, len;
  segment_of(map, prob, lo, len);
  if (threadIdx.x == 0) problem_terms(use_value ? p_value : p[prob], desc, s_pt);
  if (threadIdx.x < KS_MAX_K) s_list[threadIdx.x] = 0ull;
  __syncthreads();

  const int64_t pass_rows = static_cast<int64_t>(sub_tiles) * kBlock;
  for (int64_t start = static_cast<int64_t>(chunk) * pass_rows; start < len;
       start += static_cast<int64_t>(map.nblk) * pass_rows) {
    unsigned long long keys[kSubTilesMax + 1];
#pragma unroll
    for (int s = 0; s <= kSubTilesMax; ++s) keys[s] = 0ull;
    // carry the list of the previous pass in as extra keys
    if (threadIdx.x < k) keys[kSubTilesMax] = s_list[threadIdx.x];
#pragma unroll 1
    for (int s = 0; s < sub_tiles; ++s) {
      const int64_t r = start + static_cast<int64_t>(s) * kBlock + threadIdx.x;
      const bool live = r < len;
      int idx = 0;
      __syncthreads();  // previous sub-tile's readers are done with s_cols
      float score = 0.0f;
      if (live) {
        idx = pool_index(map, lo, r);
        const ks_candidate cand = c[idx];
        if (kStatic) {
          score = static_score(s_pt, cand, desc);
        } else {
          float* col0 = s_cols + threadIdx.x;
          featurize_pair(s_pt, cand, desc, [&](int col, float v) { col0[col * kBlock] = v; });
          score = walk_ensemble(nodes, roots, n_trees, base, s_cols + threadIdx.x, nullptr);
        }
      }
      const unsigned long long key = live ? make_key(score + 0.0f, idx) : 0ull;
#pragma unroll
      for (int q = 0; q < kSubTilesMax; ++q)
        if (q == s) keys[q] = key;
    }
    block_topk<kSubTilesMax + 1>(keys, k, s_warp, s_list);
  }
  if (threadIdx.x < k)
    partial[(static_cast<size_t>(prob) * map.nblk + chunk) * k + threadIdx.x] = s_list[threadIdx.x];
}

// ------------------------------------------------------------------------------------------
// linear scorer (one weight layer): s = b + sum_j w_j * bf16((x_j - mu_j) / sigma_j). The sum
// splits by what a column depends on: the candidate-only part is formed once per call and
// candidate (per element-type combination), the problem-only part once per block, and only the
// 21 per-pair columns are evaluated per pair, without a feature tile.
// ------------------------------------------------------------------------------------------

__device__ __forceinline__ float ridge_term(const RidgeParams& prm, int col, float v) {
  if (!isfinite(v)) v = 0.0f;
  const float x = __bfloat162float(__float2bfloat16_rn(__fdiv_rn(__fsub_rn(v, prm.mu[col]), prm.sigma[col])));
  return prm.w[col] * x;
}
__device__ __forceinline__ float ridge_level(const float (&lut)[4], float v) {
  const int code = __float2int_rz(v);
  return (code >= 0 && code < 4) ? lut[code] : 0.0f;
}

// the candidate-only part of the sum, and the resident-block count
__device__ __forceinline__ float ridge_candidate_sum(const ks_gpu_desc& desc, const RidgeParams& prm, int combo,
                                                     const ks_candidate& cand, long long& b_eff) {
  ks_problem fake{};
  fake.m = fake.n = fake.k = 1;
  fake.dtype_ab = static_cast<uint8_t>(combo >> 2);
  fake.dtype_d = static_cast<uint8_t>(combo & 3);
  ProblemTerms t;
  problem_terms(fake, desc, t);
  float s = 0.0f;
  featurize_pair(t, cand, desc, [&](int col, float v) {
    if (feat_class(col) != 1) return;
    s += ridge_term(prm, col, v);
    if (col == 17) s += ridge_level(prm.lut17, v);
    if (col == 18) s += ridge_level(prm.lut18, v);
  });
  b_eff = resources(t, cand, desc).b_eff;
  return s;
}

// per (type combination, candidate): (candidate-only part of the sum, resident-block count)
__global__ void __launch_bounds__(256)
ridge_cand_kernel(ks_gpu_desc desc, const ks_candidate* __restrict__ c, int C, const unsigned* mask_ptr,
                  const __grid_constant__ RidgeParams prm, float2* __restrict__ out, MemoView memo) {
  const int combo = blockIdx.y;
  if (!((*mask_ptr >> combo) & 1u)) return;
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= C) return;
  const ks_candidate cand = c[i];
  long long b_eff;
  const float s = ridge_candidate_sum(desc, prm, combo, cand, b_eff);
  out[static_cast<size_t>(combo) * C + i] = make_float2(s, static_cast<float>(b_eff));
  if (memo.keys) memo.cls[static_cast<size_t>(combo) * C + i] = memo_assign(memo, combo, i, cand, b_eff);
}

// What a problem brings: its terms, and the bias + problem-only part of the sum; and the combinations
// in use.
struct RidgeProblem {
  ProblemTerms t;
  float sum;
  int combo;
};
__global__ void __launch_bounds__(128)
ridge_problem_kernel(ks_gpu_desc desc, const ks_problem* __restrict__ p, ks_problem p_value, int use_value, int P,
                     const __grid_constant__ RidgeParams prm, RidgeProblem* __restrict__ out, unsigned* __restrict__ mask) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  unsigned m = 0;
  if (i < P) {
    RidgeProblem e;
    problem_terms(use_value ? p_value : p[i], desc, e.t);
    e.combo = e.t.dtype_ab * 4 + e.t.dtype_d;
    float s = prm.bias;
    problem_columns(e.t, [&](int col, float v) {
      s += ridge_term(prm, col, v);
      if (col == 5) s += ridge_level(prm.lut5, v);
      if (col == 9) s += ridge_level(prm.lut9, v);
    });
    e.sum = s;
    out[i] = e;
    m = 1u << e.combo;
  }
  // (the whole warp: which of its threads run together after the arithmetic above is not given)
  m = __reduce_or_sync(0xFFFFFFFFu, m);
  if ((threadIdx.x & 31) == 0 && m) atomicOr(mask, m);
}

// With classes: a candidate's second word, so far its resident-block count b, becomes the number of
// its class among the classes in use, or -b when it has none (memo_compact left the numbers in `keys`) or its type
// combination has more than `most`.
__global__ void __launch_bounds__(256)
ridge_pack_kernel(int C, const unsigned* __restrict__ mask, MemoView memo, float2* __restrict__ tab, int most) {
  const int combo = blockIdx.y, i = blockIdx.x * blockDim.x + threadIdx.x;
  if (!((*mask >> combo) & 1u) || i >= C) return;
  const unsigned slot = memo.cls[static_cast<size_t>(combo) * C + i];
  float& y = tab[static_cast<size_t>(combo) * C + i].y;
  const int v = slot == kNoClass || memo.count[combo] > most ? -static_cast<int>(y) : static_cast<int>(memo.keys[static_cast<size_t>(combo) * kMemoCap + slot]);
  y = __int_as_float(v);
}

// Per (problem, class): the per-pair part of the sum, from the class's member (classes: ks_memo.cuh).
// grid (a few, P); record j of a problem is its j-th class. Not where there are more than `most`.
__global__ void __launch_bounds__(256)
ridge_pair_kernel(ks_gpu_desc desc, const RidgeProblem* __restrict__ problems, const ks_candidate* __restrict__ c,
                  const __grid_constant__ RidgeParams prm, MemoView memo, int most) {
  __shared__ ProblemTerms s_pt;
  const int prob = blockIdx.y, combo = problems[prob].combo;
  const int n_classes = memo.count[combo];
  if (n_classes > most) return;
  if (threadIdx.x < sizeof(ProblemTerms) / 4)
    reinterpret_cast<uint32_t*>(&s_pt)[threadIdx.x] = reinterpret_cast<const uint32_t*>(&problems[prob].t)[threadIdx.x];
  __syncthreads();
  for (int j = blockIdx.x * 256 + threadIdx.x; j < n_classes; j += gridDim.x * 256) {
    const int slot = memo.dense[static_cast<size_t>(combo) * kMemoCap + j];
    const ks_candidate cand = load_candidate(c + memo.reps[static_cast<size_t>(combo) * kMemoCap + slot]);
    float pair = 0.0f;
    pair_columns<true>(s_pt, cand, desc, resources(s_pt, cand, desc).b_eff,
                       [&](int col, float v) { pair += ridge_term(prm, col, v); });
    static_cast<float*>(memo.tab)[static_cast<size_t>(prob) * kMemoCap + j] = pair;
  }
}

// the per-pair part in place, for a candidate without a class (out of line: it would cost a kernel
// half its resident warps)
__device__ __noinline__ float ridge_pair_in_place(const ks_gpu_desc& desc, const ProblemTerms& t, const ks_candidate* c,
                                                  long long b_eff, const RidgeParams& prm) {
  float pair = 0.0f;
  pair_columns<true>(t, load_candidate(c), desc, b_eff, [&](int col, float v) { pair += ridge_term(prm, col, v); });
  return pair;
}

// Segmented batches, and batches of few problems: a block ranks one problem against its share of the
// candidates. What bounds it is the instructions a pair takes, so the class sums are gathered from
// shared memory, and a warp keeps a running top-k list (one key a lane): a score that does not reach
// the best k-th score any of the block's warps has seen costs no more than the comparison. (Ranking
// eight keys a thread from scratch, with sums from L2, took three times as long.)
constexpr int kRidgeThreads = 512;
constexpr int kRidgeClasses = 2048;  // classes whose sums are staged; the others are fetched from L2
// kClasses: with the class tables; without them (few problems) every pair is evaluated in place.
template <bool kClasses>
__global__ void __launch_bounds__(kRidgeThreads, kClasses ? 2 : 1)
select_ridge_kernel(const __grid_constant__ ks_gpu_desc desc, const RidgeProblem* __restrict__ problems, const ks_candidate* __restrict__ c,
                    PairMap map, const float2* __restrict__ cand_tab, const __grid_constant__ RidgeParams prm, int k,
                    unsigned long long* __restrict__ partial /* [P][nblk][k] */, MemoView memo) {
  __shared__ float s_tab[kClasses ? kRidgeClasses : 1];
  __shared__ ProblemTerms s_pt;  // (without classes)
  __shared__ unsigned s_bar;     // upper word of a key below which nothing can make the list
  // The upper words of a warp's best key and (for k > 16) its second best, in one 64-bit word: another warp
  // sees both from before or both from after an update, so no candidate counts twice in the bar.
  __shared__ unsigned long long s_best[kRidgeThreads / 32];
  __shared__ unsigned long long s_list[kRidgeThreads / 32][32];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int prob = blockIdx.x / map.nblk, chunk = blockIdx.x % map.nblk;
  const int combo = problems[prob].combo;
  const float sum = problems[prob].sum;
  const float* tab = static_cast<const float*>(memo.tab) + static_cast<size_t>(prob) * kMemoCap;
  unsigned long long top = 0ull;
  if (kClasses) {
    const int n = min(memo.count[combo], kRidgeClasses);
    for (int j = tid; j < n; j += kRidgeThreads) s_tab[j] = __ldg(tab + j);
  }
  if (!kClasses && tid < static_cast<int>(sizeof(ProblemTerms) / 4))
    reinterpret_cast<uint32_t*>(&s_pt)[tid] = reinterpret_cast<const uint32_t*>(&problems[prob].t)[tid];
  if (tid == 0) s_bar = 0u;
  if (tid < kRidgeThreads / 32) s_best[tid] = 0ull;
  __syncthreads();
  int64_t lo, len;
  segment_of(map, prob, lo, len);
  const int64_t share = (len + map.nblk - 1) / map.nblk, stop = min(len, share * (chunk + 1));
  const float2* cand = cand_tab + static_cast<size_t>(combo) * map.C;
  // a candidate's record is fetched one round ahead
  auto row_index = [&](int64_t r) { return r < stop ? pool_index(map, lo, r) : 0; };
  const int64_t r_first = share * chunk + warp * 32 + lane;
  int next_idx = row_index(r_first);
  float2 next = __ldg(cand + next_idx);
  for (int64_t r = r_first; r - lane < stop; r += kRidgeThreads) {
    const bool live = r < stop;
    const int idx = next_idx;
    const float2 t = next;
    next_idx = row_index(r + kRidgeThreads);
    next = __ldg(cand + next_idx);
    const int cls = __float_as_int(t.y);
    float pair = 0.0f;
    if (kClasses && cls >= 0) {
      pair = cls < kRidgeClasses ? s_tab[cls] : __ldg(tab + cls);
    } else if (kClasses) {
      pair = ridge_pair_in_place(desc, problems[prob].t, c + idx, -static_cast<long long>(cls), prm);
    } else {
      pair_columns<true>(s_pt, load_candidate(c + idx), desc, static_cast<long long>(t.y),
                         [&](int col, float v) { pair += ridge_term(prm, col, v); });
    }
    const float score = ((sum + t.x) + pair) + 0.0f;
    if (__any_sync(0xFFFFFFFFu, live && sortable(score) >= *const_cast<volatile unsigned*>(&s_bar))) {
      warp_topk_insert(top, live ? make_key(score, idx) : 0ull, k);
      // The k-th largest of the warps' best keys bounds the k-th best score from below (each is a
      // candidate of its own), far better than any one warp's k-th.
      constexpr int kWarps = kRidgeThreads / 32;
      volatile unsigned long long* best = s_best;
      const unsigned mine = static_cast<unsigned>(top >> 32), after = __shfl_sync(0xFFFFFFFFu, mine, 1);
      if (lane == 0) best[warp] = static_cast<unsigned long long>(mine) << 32 | (k > kWarps ? after : 0u);
      __syncwarp();
      const unsigned long long two = lane < kWarps ? best[lane] : 0ull;
      const unsigned first = static_cast<unsigned>(two >> 32), second = static_cast<unsigned>(two);
      int ahead = 0, ahead2 = 0;  // of the two: keys that are at least as good
#pragma unroll
      for (int i = 0; i < kWarps; ++i) ahead += __shfl_sync(0xFFFFFFFFu, first, i) >= first;
      unsigned bar = ahead >= k ? first : 0u;
      if (k > kWarps) {
#pragma unroll
        for (int i = 0; i < kWarps; ++i) {
          const unsigned f = __shfl_sync(0xFFFFFFFFu, first, i), s = __shfl_sync(0xFFFFFFFFu, second, i);
          ahead += s >= first;
          ahead2 += (f >= second) + (s >= second);
        }
        bar = max(ahead >= k ? first : 0u, ahead2 >= k ? second : 0u);
      }
      bar = __reduce_max_sync(0xFFFFFFFFu, bar);
      if (lane == 0) atomicMax(&s_bar, bar);
    }
  }
  s_list[warp][lane] = top;
  __syncthreads();
  if (warp == 0) {
    for (int w = 1; w < kRidgeThreads / 32; ++w) warp_topk_insert(top, s_list[w][lane], k);
    if (lane < k) partial[(static_cast<size_t>(prob) * map.nblk + chunk) * k + lane] = top;
  }
}

// ---- dense batches: the classes of the catalogue, their members and their largest sums ----
//
// The score ((problem + candidate) + pair) rounds after every addition, and rounding keeps the order: among
// the members of a class (equal pair part, see ks_memo.cuh) the one with the largest candidate part has the
// largest score. So a problem ranks its classes by that score first, and only a class whose best
// member reaches the k-th best of them is looked into: about k classes of 36 members instead of 60,000 pairs.
// What is not a number or infinite is outside this order: such a class is always looked into.
//
// Slots of a combination's table: a power of two above the 10,785 classes of the valid search space. A
// candidate without a slot (more classes than slots) is kept in a list of its own and always evaluated.
constexpr int kRidgeCap = 16384;
struct RidgeClass {  // 32 bytes
  ks_candidate member;
  float best;   // largest candidate-only sum of the class; not finite: look into it
  int b_eff;
  int first, count;  // its members in the list
};
struct RidgeMember {
  int idx;
  float sum;  // candidate-only part
};
// What a call keeps, per type combination. The first four are cleared in front of a call.
struct RidgeTables {
  unsigned* mask;            // combinations in use (with the clearing of the next two)
  unsigned long long* keys;  // [16][kRidgeCap], 0 = free
  uint2* stat;               // [16][kRidgeCap + 1] (largest sum as a sortable word, members); the last entry: without a class
  int* n;                    // [16] (classes, their members)
  int* rep;                  // [16][kRidgeCap] one member
  uint2* place;              // [16][C] (slot, place among its members)
  float* sum;                // [16][C] candidate-only part
  int* first;                // [16][kRidgeCap] where a slot's members begin in the list (those without a class end it)
  RidgeClass* cls;           // [16][kRidgeCap]
  RidgeMember* list;         // [16][C]
  float* pair;               // [blocks][kRidgeCap] a block's per-pair parts
};

// A class's largest sum: order-preserving, with everything that is not finite above all.
__device__ __forceinline__ unsigned ridge_bound_word(float s) { return isfinite(s) ? sortable(s) : 0xFFFFFFFFu; }

// per (type combination, candidate): the candidate-only part of the sum, and its class
__global__ void __launch_bounds__(256)
ridge_members_kernel(const __grid_constant__ ks_gpu_desc desc, const ks_candidate* __restrict__ c, int C,
                     const __grid_constant__ RidgeParams prm, RidgeTables t) {
  const int combo = blockIdx.y, i = blockIdx.x * blockDim.x + threadIdx.x;
  if (!((*t.mask >> combo) & 1u) || i >= C) return;
  const ks_candidate cand = load_candidate(c + i);
  long long b_eff;
  const float s = ridge_candidate_sum(desc, prm, combo, cand, b_eff);
  const size_t at = static_cast<size_t>(combo) * kRidgeCap;
  const unsigned slot = memo_slot<kRidgeCap>(t.keys + at, t.rep + at, i, cand, b_eff);
  uint2* stat = t.stat + static_cast<size_t>(combo) * (kRidgeCap + 1) + min(slot, static_cast<unsigned>(kRidgeCap));
  atomicMax(&stat->x, ridge_bound_word(s));
  t.place[static_cast<size_t>(combo) * C + i] = make_uint2(slot, atomicAdd(&stat->y, 1u));
  t.sum[static_cast<size_t>(combo) * C + i] = s;
}

__device__ __noinline__ float ridge_lone_pair(const ks_gpu_desc& desc, const ProblemTerms& t, const ks_candidate* c,
                                              const RidgeParams& prm) {
  return ridge_pair_in_place(desc, t, c, resources(t, load_candidate(c), desc).b_eff, prm);
}

// Packs the classes of every combination and gives each its part of the list: a thread a slot, two atomic
// operations a block. (One block for all of a combination's slots took 40 us for 1,700 classes and 100 for 10,785.)
__global__ void __launch_bounds__(256)
ridge_classes_kernel(const __grid_constant__ ks_gpu_desc desc, const ks_candidate* __restrict__ c, RidgeTables t) {
  __shared__ int s_n, s_members, s_cls0, s_first0;
  const int combo = blockIdx.y, slot = blockIdx.x * 256 + threadIdx.x;
  if (!((*t.mask >> combo) & 1u)) return;
  if (threadIdx.x == 0) s_n = s_members = 0;
  __syncthreads();
  const uint2 st = t.stat[static_cast<size_t>(combo) * (kRidgeCap + 1) + slot];
  int j = 0, first = 0;
  if (st.y != 0u) {
    j = atomicAdd(&s_n, 1);
    first = atomicAdd(&s_members, static_cast<int>(st.y));
  }
  __syncthreads();
  if (threadIdx.x == 0 && s_n > 0) {
    s_cls0 = atomicAdd(t.n + 2 * combo, s_n);
    s_first0 = atomicAdd(t.n + 2 * combo + 1, s_members);
  }
  __syncthreads();
  if (st.y == 0u) return;
  const size_t at = static_cast<size_t>(combo) * kRidgeCap;
  ProblemTerms pt;  // the resident-block count depends on the element sizes alone
  pt.bA = bytes_ab(combo >> 2);
  pt.bD = bytes_d(combo & 3);
  RidgeClass r;
  r.member = load_candidate(c + t.rep[at + slot]);
  r.best = st.x == 0xFFFFFFFFu ? __uint_as_float(0x7FC00000u) : key_score(static_cast<unsigned long long>(st.x) << 32);
  r.b_eff = static_cast<int>(resources(pt, r.member, desc).b_eff);
  r.first = s_first0 + first;
  r.count = static_cast<int>(st.y);
  t.first[at + slot] = r.first;
  t.cls[at + s_cls0 + j] = r;
}

__global__ void __launch_bounds__(256)
ridge_list_kernel(int C, RidgeTables t) {
  const int combo = blockIdx.y, i = blockIdx.x * blockDim.x + threadIdx.x;
  if (!((*t.mask >> combo) & 1u) || i >= C) return;
  const size_t at = static_cast<size_t>(combo) * C;
  const uint2 p = t.place[at + i];
  const int first = p.x == kNoClass ? C - static_cast<int>(t.stat[static_cast<size_t>(combo) * (kRidgeCap + 1) + kRidgeCap].y)
                                    : t.first[static_cast<size_t>(combo) * kRidgeCap + p.x];
  t.list[at + first + p.y] = RidgeMember{i, t.sum[at + i]};
}

// A block ranks a problem's share y of the classes (gridDim.y shares); blocks take problem after problem.
// First every thread evaluates its classes and keeps its best one: the k-th largest of these bounds the k-th
// best score from below (they are candidates of their own). Then the classes that reach it are looked into,
// a warp a class. What bounds it is the arithmetic of the per-pair columns, once per (problem, class), so the
// blocks are small: seven of 128 threads an SM serve 1,024 problems in one even round. 1,024 x 60,000 pairs: the
// whole call 115 us, of it 75 here; every pair added up and compared, from a table of the pair parts, 279.
constexpr int kRidgeRankThreads = 128, kRidgeRankBlocks = 7;
__global__ void __launch_bounds__(kRidgeRankThreads, kRidgeRankBlocks)
ridge_rank_kernel(const __grid_constant__ ks_gpu_desc desc, const RidgeProblem* __restrict__ problems, int P,
                  const ks_candidate* __restrict__ c, int C, const __grid_constant__ RidgeParams prm, int k, RidgeTables t,
                  unsigned long long* __restrict__ partial /* [P][gridDim.y][k], or null: the lists are the result */,
                  int32_t* __restrict__ out_idx, float* __restrict__ out_score) {
  constexpr int kWarps = kRidgeRankThreads / 32;
  __shared__ RidgeProblem s_p;
  __shared__ unsigned long long s_warp[kWarps * KS_MAX_K], s_list[KS_MAX_K];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  float* pair_of = t.pair + static_cast<size_t>(blockIdx.y * gridDim.x + blockIdx.x) * kRidgeCap;
  for (int prob = blockIdx.x; prob < P; prob += gridDim.x) {
    __syncthreads();  // the problem before is finished with
    static_assert(sizeof(RidgeProblem) % 4 == 0 && sizeof(RidgeProblem) / 4 <= kRidgeRankThreads, "one word a thread");
    if (tid < static_cast<int>(sizeof(RidgeProblem) / 4))
      reinterpret_cast<uint32_t*>(&s_p)[tid] = __ldg(reinterpret_cast<const uint32_t*>(problems + prob) + tid);
    __syncthreads();
    const int n = t.n[2 * s_p.combo];
    const int begin = static_cast<int>(static_cast<int64_t>(n) * blockIdx.y / gridDim.y);
    const int end = static_cast<int>(static_cast<int64_t>(n) * (blockIdx.y + 1) / gridDim.y);
    const RidgeClass* cls = t.cls + static_cast<size_t>(s_p.combo) * kRidgeCap;
    const float sum = s_p.sum;
    unsigned long long best = 0ull;
    for (int j = begin + tid; j < end; j += kRidgeRankThreads) {
      const ks_candidate cand = load_candidate(&cls[j].member);
      float pair = 0.0f;
      pair_columns<true>(s_p.t, cand, desc, static_cast<long long>(cls[j].b_eff),
                         [&](int col, float v) { pair += ridge_term(prm, col, v); });
      pair_of[j] = pair;
      const float bound = ((sum + cls[j].best) + pair) + 0.0f;
      if (isfinite(bound)) best = max(best, make_key(bound, j));
    }
    unsigned long long one[1] = {best};
    block_topk<1>(one, k, s_warp, s_list);
    const unsigned bar = static_cast<unsigned>(s_list[k - 1] >> 32);
    unsigned long long mine = 0ull;  // the warp's running list
    const RidgeMember* list = t.list + static_cast<size_t>(s_p.combo) * C;
    for (int j0 = begin + 32 * warp; j0 < end; j0 += kRidgeRankThreads) {
      const int j = j0 + lane;
      float pair = 0.0f;
      int first = 0, count = 0;
      bool look = false;
      if (j < end) {
        pair = pair_of[j];
        const float bound = ((sum + cls[j].best) + pair) + 0.0f;
        look = !isfinite(bound) || sortable(bound) >= bar;
        if (look) {
          first = cls[j].first;
          count = cls[j].count;
        }
      }
      for (unsigned todo = __ballot_sync(0xFFFFFFFFu, look); todo; todo &= todo - 1) {
        const int src = __ffs(todo) - 1;
        const int f = __shfl_sync(0xFFFFFFFFu, first, src), m = __shfl_sync(0xFFFFFFFFu, count, src);
        const float q = __shfl_sync(0xFFFFFFFFu, pair, src);
        for (int i = lane; i - lane < m; i += 32) {
          unsigned long long key = 0ull;
          if (i < m) {
            const RidgeMember e = list[f + i];
            key = make_key(((sum + e.sum) + q) + 0.0f, e.idx);
            if (static_cast<unsigned>(key >> 32) < bar) key = 0ull;
          }
          warp_topk_insert(mine, key, k);
        }
      }
    }
    // candidates without a class: dealt to the blocks and warps like the classes
    const int lone = static_cast<int>(t.stat[static_cast<size_t>(s_p.combo) * (kRidgeCap + 1) + kRidgeCap].y);
    const int lone_at = C - lone;
    for (int i0 = 32 * (blockIdx.y * kWarps + warp); i0 < lone; i0 += 32 * kWarps * gridDim.y) {
      unsigned long long key = 0ull;
      if (i0 + lane < lone) {
        const RidgeMember e = list[lone_at + i0 + lane];
        key = make_key(((sum + e.sum) + ridge_lone_pair(desc, s_p.t, c + e.idx, prm)) + 0.0f, e.idx);
      }
      warp_topk_insert(mine, key, k);
    }
    one[0] = mine;
    block_topk<1>(one, k, s_warp, s_list);
    if (tid < k) {
      if (partial) {
        partial[(static_cast<size_t>(prob) * gridDim.y + blockIdx.y) * k + tid] = s_list[tid];
      } else {
        out_idx[static_cast<size_t>(prob) * k + tid] = key_index(s_list[tid]);
        out_score[static_cast<size_t>(prob) * k + tid] = key_score(s_list[tid]);
      }
    }
  }
}


// Blocks a problem of the kernels above takes.
// Of the class form: as many as the machine holds at once; a block has a thread for each of the valid search
// space's 10,785 classes then.
static int ridge_rank_shares(int P) {
  return static_cast<int>(std::max<int64_t>(1, std::min<int64_t>(64, kRidgeRankBlocks * 148 / P)));
}
static int ridge_rank_grid(int P) {
  return static_cast<int>(std::min<int64_t>(P, kRidgeRankBlocks * 148 / ridge_rank_shares(P)));
}
// Of the candidate form: as many as fill the machine once (two blocks of 512 threads an SM), with about 512
// candidates each at least.
static int ridge_blocks(int P, int64_t per_problem) {
  const int64_t most = std::max<int64_t>(1, (per_problem + 511) / 512);
  return static_cast<int>(std::min(most, std::max<int64_t>(1, 2 * 148 / P)));
}
// Dense batches go by classes where that many pairs take longer one by one than the class tables do: 60,000
// grid candidates 55 us whatever the (few) problems, in place 87 for 24 and 106 for 32; 61,140 valid candidates (10,785
// classes) 89 and 95, in place 88 and 108; 5,000 candidates 52, in place 45 for 64 and 58 for 128. Valid candidates are
// less alike: 30 x 20,000 of them 73 us, in place 54, 30 x 45,000 84 and 82 (mixed types 99 and 87), 30 x 60,000 86 and 99 (102 and
// 109), so batches of fewer than 32 problems go by classes from there on.
static bool ridge_by_classes(int P, int C, bool segmented, bool lean) {
  return !segmented && !lean && P >= 30 && static_cast<int64_t>(P) * C >= (P < 32 ? 1800000 : 600000);
}

// ------------------------------------------------------------------------------------------
// merge: ranks the nblk * k partial keys of a problem
// ------------------------------------------------------------------------------------------

// A warp (kWarps = 1, eight problems a block) or a block of eight warps ranks a problem's keys, each
// read once into the warp's running list; a block's lists are merged by its first warp. (One warp that
// read the keys again for each of the k ranks took 19 us for the 1,480 keys of a single problem.)
template <int kWarps>
__global__ void __launch_bounds__(kBlock)
topk_merge_kernel(const unsigned long long* __restrict__ partial, int P, int n_keys, int k,
                  int32_t* __restrict__ out_idx, float* __restrict__ out_score, HostNotice notice) {
  asm volatile("griddepcontrol.wait;" ::: "memory");  // (launched as the dependent of the kernel in front)
  __shared__ unsigned long long s_list[kWarps][32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int prob = kWarps == 1 ? blockIdx.x * (kBlock / 32) + warp : blockIdx.x, part = kWarps == 1 ? 0 : warp;
  if (prob >= P) return;
  const unsigned long long* keys = partial + static_cast<size_t>(prob) * n_keys;
  unsigned long long mine = 0ull;
  for (int i0 = part * 128; i0 < n_keys; i0 += kWarps * 128) {
    unsigned long long v[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) v[q] = i0 + 32 * q + lane < n_keys ? keys[i0 + 32 * q + lane] : 0ull;
#pragma unroll
    for (int q = 0; q < 4; ++q) warp_topk_insert(mine, v[q], k);
  }
  if (kWarps > 1) {
    s_list[part][lane] = mine;
    __syncthreads();
    if (warp != 0) return;
    for (int w = 1; w < kWarps; ++w) warp_topk_insert(mine, s_list[w][lane], k);
  }
  if (lane < k) {
    out_idx[static_cast<size_t>(prob) * k + lane] = key_index(mine);
    out_score[static_cast<size_t>(prob) * k + lane] = key_score(mine);
  }
  if (notice.word) {  // (a single problem)
    __threadfence_system();
    __syncwarp();
    if (lane == 0) *static_cast<volatile int*>(notice.word) = notice.seq;
  }
}

// A block per problem while that leaves the machine room, else a warp.
static cudaError_t launch_merge(const unsigned long long* partial, int P, int n_keys, int k, int32_t* d_topk_idx,
                                float* d_topk_score, cudaStream_t stream, int64_t* launches, const HostNotice* notice = nullptr, bool timed = false) {
  constexpr int kPer = kBlock / 32;
  const bool blocks = P <= 8 * 148 && n_keys > 128;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(blocks ? P : (P + kPer - 1) / kPer);
  cfg.blockDim = dim3(kBlock);
  cfg.stream = stream;
  cudaLaunchAttribute attr{};
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &attr;
  cfg.numAttrs = timed ? 0 : 1;  // (an event stands between it and the kernel in front)
  if (launches) ++*launches;
  return cudaLaunchKernelEx(&cfg, blocks ? &topk_merge_kernel<kPer> : &topk_merge_kernel<1>, partial, P, n_keys, k, d_topk_idx,
                            d_topk_score, notice ? *notice : HostNotice{nullptr, 0});
}

// Merge of ranked lists (the exchange step of a candidate-split selection): per problem, n
// (index, score) entries gathered from several partial top-k lists, index -1 = empty; the k best
// by (score descending, index ascending) go to the output. One warp per problem.
__global__ void __launch_bounds__(kBlock)
merge_lists_kernel(const int32_t* __restrict__ in_idx, const float* __restrict__ in_score, int P, int n, int k,
                   int32_t* __restrict__ out_idx, float* __restrict__ out_score) {
  const int warp = (blockIdx.x * kBlock + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  if (warp >= P) return;
  const int32_t* idx = in_idx + static_cast<size_t>(warp) * n;
  const float* sc = in_score + static_cast<size_t>(warp) * n;
  unsigned long long prev = ~0ull;
  for (int j = 0; j < k; ++j) {
    unsigned long long best = 0ull;
    for (int i = lane; i < n; i += 32) {
      const unsigned long long v = idx[i] >= 0 ? make_key(sc[i] + 0.0f, idx[i]) : 0ull;
      if (v < prev && v > best) best = v;
    }
    best = warp_max_u64(best);
    if (lane == 0) {
      out_idx[static_cast<size_t>(warp) * k + j] = key_index(best);
      out_score[static_cast<size_t>(warp) * k + j] = key_score(best);
    }
    prev = best;
  }
}

cudaError_t launch_merge_lists(const int32_t* d_idx, const float* d_score, int P, int n, int k, int32_t* d_out_idx,
                               float* d_out_score, cudaStream_t stream, int64_t* launches) {
  merge_lists_kernel<<<(P * 32 + kBlock - 1) / kBlock, kBlock, 0, stream>>>(d_idx, d_score, P, n, k, d_out_idx,
                                                                           d_out_score);
  ++*launches;
  return cudaGetLastError();
}

// ------------------------------------------------------------------------------------------
// launchers
// ------------------------------------------------------------------------------------------

static PairMap make_map(int P, int C, int64_t pairs, const int64_t* seg_off, const int32_t* seg_idx,
                        int rows_per_block) {
  PairMap m;
  m.P = P;
  m.C = C;
  m.seg_off = seg_off;
  m.seg_idx = seg_idx;
  m.rows_per_block = rows_per_block;
  const int64_t per_problem = seg_off ? (P > 0 ? (pairs + P - 1) / P : 0) : C;
  m.nblk = static_cast<int>(per_problem > 0 ? (per_problem + rows_per_block - 1) / rows_per_block : 1);
  if (m.nblk < 1) m.nblk = 1;
  return m;
}

cudaError_t launch_featurize(const ks_gpu_desc& desc, const ks_problem* d_p, int P,
                             const ks_candidate* d_c, int C, const int64_t* d_seg_off,
                             const int32_t* d_seg_idx, int64_t pairs, float* d_out, void* scratch,
                             cudaStream_t stream, int64_t* launches) {
  if (P == 0 || pairs == 0) return cudaSuccess;
  const PairMap map = make_map(P, C, pairs, d_seg_off, d_seg_idx, kBlock);
  const size_t smem = sizeof(float) * kBlock * 65;
  if (!d_seg_off && C > 0 && scratch) {
    cudaError_t e = ensure_dynamic_smem(reinterpret_cast<const void*>(&featurize_dense_kernel), smem);
    if (e != cudaSuccess) return e;
    ProblemEntry* tab = static_cast<ProblemEntry*>(scratch);
    problem_table_kernel<<<(P + 127) / 128, 128, 0, stream>>>(desc, d_p, P, tab);
    const int64_t total = static_cast<int64_t>((C + 31) / 32) * P;
    int64_t grid = (total + kBlock / 32 - 1) / (kBlock / 32);
    if (grid > 3 * 148) grid = 3 * 148;  // three resident blocks per SM
    featurize_dense_kernel<<<static_cast<unsigned>(grid), kBlock, smem, stream>>>(desc, tab, d_c, P, C, d_out);
    *launches += 2;
    return cudaGetLastError();
  }
  // about four blocks for every place on the machine, each with several slabs of a problem's rows
  // (one for every place 146 us, two 125, eight 126)
  PairMap some = map;
  some.nblk = static_cast<int>(std::min<int64_t>(map.nblk, std::max<int64_t>(1, (4 * 4 * 148 + P - 1) / P)));
  const size_t staged = sizeof(float) * kBlock * kStagedStride;
  const auto kernel = (reinterpret_cast<uintptr_t>(d_out) & 7u) == 0 ? &featurize_kernel<true> : &featurize_kernel<false>;
  cudaError_t e = ensure_dynamic_smem(reinterpret_cast<const void*>(kernel), staged);
  if (e != cudaSuccess) return e;
  kernel<<<static_cast<unsigned>(static_cast<int64_t>(P) * some.nblk), kBlock, staged, stream>>>(
      desc, d_p, d_c, some, d_out);
  ++*launches;
  return cudaGetLastError();
}

cudaError_t launch_score_gbdt(const GbdtModel& m, const float* d_feat, int64_t rows, float* d_scores,
                              uint16_t* d_leaf_idx, cudaStream_t stream, int64_t* launches) {
  if (rows == 0) return cudaSuccess;
  const size_t smem = sizeof(float) * kRow * kBlock;
  cudaError_t e = ensure_dynamic_smem(reinterpret_cast<const void*>(&score_gbdt_kernel), smem);
  if (e != cudaSuccess) return e;
  score_gbdt_kernel<<<static_cast<unsigned>((rows + kBlock - 1) / kBlock), kBlock, smem, stream>>>(
      m.d_nodes, m.d_roots, m.n_trees, m.base, d_feat, rows, d_scores, d_leaf_idx);
  ++*launches;
  return cudaGetLastError();
}

static float bf16_bits_host(uint16_t b) {
  const uint32_t u = static_cast<uint32_t>(b) << 16;
  float f;
  std::memcpy(&f, &u, 4);
  return f;
}
static float round_bf16_host(float v) {
  uint32_t u;
  std::memcpy(&u, &v, 4);
  if ((u & 0x7F800000u) == 0x7F800000u) return v;
  u += 0x7FFFu + ((u >> 16) & 1u);
  u &= 0xFFFF0000u;
  std::memcpy(&v, &u, 4);
  return v;
}

cudaError_t build_ridge(MlpModel& m, const uint16_t* h_w, const float* h_b, const float* h_mu,
                        const float* h_sigma) {
  if (m.n_layers != 1) return cudaSuccess;
  RidgeParams* r = new (std::nothrow) RidgeParams();
  if (!r) return cudaErrorMemoryAllocation;
  std::memset(r, 0, sizeof(*r));
  for (int j = 0; j < 64; ++j) r->sigma[j] = 1.0f;
  r->bias = h_b[0];
  if (m.widths[0] == KS_F_PAD) {
    for (int j = 0; j < KS_F; ++j) {
      r->w[j] = bf16_bits_host(h_w[j]);
      r->mu[j] = h_mu[j];
      r->sigma[j] = h_sigma[j];
    }
  } else {  // one-hot form: kept columns in ascending order, then the level indicators
    int pos = 0;
    for (int j = 0; j < KS_F; ++j) {
      if (j == 5 || j == 9 || j == 17 || j == 18) continue;
      r->w[j] = bf16_bits_host(h_w[pos]);
      r->mu[j] = h_mu[pos];
      r->sigma[j] = h_sigma[pos];
      ++pos;
    }
    float* luts[4] = {r->lut5, r->lut9, r->lut17, r->lut18};
    const int levels[4] = {4, 3, 4, 3};
    for (int f = 0; f < 4; ++f) {
      for (int lv = 0; lv < levels[f]; ++lv) {  // the field is at level lv: one indicator is 1
        float s = 0.0f;
        for (int q = 0; q < levels[f]; ++q) {
          const float x = round_bf16_host(((q == lv ? 1.0f : 0.0f) - h_mu[pos + q]) / h_sigma[pos + q]);
          s += bf16_bits_host(h_w[pos + q]) * x;
        }
        luts[f][lv] = s;
      }
      pos += levels[f];
    }
  }
  m.h_ridge = r;
  LinearRow* q = new (std::nothrow) LinearRow();
  if (!q) return cudaErrorMemoryAllocation;
  m.h_linear = q;
  for (int j = 0; j < m.widths[0]; ++j) {
    q->w[j] = bf16_bits_host(h_w[j]);
    q->mu[j] = h_mu[j];
    q->sigma[j] = h_sigma[j];
  }
  q->bias = h_b[0];
  return cudaSuccess;
}

void free_ridge(MlpModel& m) {
  delete m.h_ridge;
  m.h_ridge = nullptr;
  delete m.h_linear;
  m.h_linear = nullptr;
}

cudaError_t launch_score_linear(const MlpModel& m, const float* d_feat, int64_t rows, float* d_scores,
                                cudaStream_t stream, int64_t* launches) {
  if (rows == 0) return cudaSuccess;
  const unsigned grid = static_cast<unsigned>((rows + kBlock - 1) / kBlock);
  if (m.widths[0] == KS_F_ONEHOT) score_linear_kernel<true><<<grid, kBlock, 0, stream>>>(*m.h_linear, d_feat, rows, d_scores);
  else score_linear_kernel<false><<<grid, kBlock, 0, stream>>>(*m.h_linear, d_feat, rows, d_scores);
  ++*launches;
  return cudaGetLastError();
}

size_t ridge_scratch_bytes(int P, int C) {
  return 256 + (sizeof(float2) * 16 * static_cast<size_t>(C) + 255) / 256 * 256 + (sizeof(RidgeProblem) * static_cast<size_t>(P) + 255) / 256 * 256;
}
// classes and the per-(problem, class) sums of a segmented batch (0: not used)
static size_t ridge_memo_bytes(int P, int C, bool segmented) {
  if (!segmented || P < kMemoMinProblems || P > kMemoMaxProblems || C < 1) return 0;
  return memo_fixed_bytes(C) + sizeof(float) * static_cast<size_t>(P) * kMemoCap;
}
// The parts of the class form's memory; `cleared` receives the bytes at its beginning that a call clears.
static size_t ridge_tables(int P, int C, void* mem, RidgeTables* t, size_t* cleared) {
  size_t at = 0;
  const auto take = [&](size_t bytes) {
    char* q = static_cast<char*>(mem) + at;
    at += (bytes + 255) / 256 * 256;
    return q;
  };
  const size_t slots = static_cast<size_t>(16) * kRidgeCap, all = static_cast<size_t>(16) * C;
  t->mask = reinterpret_cast<unsigned*>(take(256));
  t->keys = reinterpret_cast<unsigned long long*>(take(slots * sizeof(unsigned long long)));
  t->stat = reinterpret_cast<uint2*>(take((slots + 16) * sizeof(uint2)));
  t->n = reinterpret_cast<int*>(take(32 * sizeof(int)));
  *cleared = at;
  t->rep = reinterpret_cast<int*>(take(slots * sizeof(int)));
  t->place = reinterpret_cast<uint2*>(take(all * sizeof(uint2)));
  t->sum = reinterpret_cast<float*>(take(all * sizeof(float)));
  t->first = reinterpret_cast<int*>(take(slots * sizeof(int)));
  t->cls = reinterpret_cast<RidgeClass*>(take(slots * sizeof(RidgeClass)));
  t->list = reinterpret_cast<RidgeMember*>(take(all * sizeof(RidgeMember)));
  t->pair = reinterpret_cast<float*>(take(static_cast<size_t>(ridge_rank_grid(P)) * ridge_rank_shares(P) * kRidgeCap * sizeof(float)));
  return at;
}

static int pick_sub_tiles(int P, int64_t per_problem) {
  for (int s = kSubTilesMax; s > 1; s >>= 1) {
    const int64_t nblk = (per_problem + static_cast<int64_t>(s) * kBlock - 1) / (static_cast<int64_t>(s) * kBlock);
    if (static_cast<int64_t>(P) * nblk >= 4 * 148) return s;
  }
  return 1;
}

static int64_t per_problem_rows(int P, int C, int64_t pairs, bool segmented) {
  return segmented ? (P > 0 ? (pairs + P - 1) / P : 0) : C;
}

// Dense walks that are split: few blocks, and not for the walk of whole classes to serve.
static bool select_splits(const GbdtModel& g, int P, int C, int64_t pairs, int nblk, bool segmented, bool lean) {
  return !segmented && fast_splits(g, P, nblk, lean) && (lean || !classes_apply(g, P, C, pairs));
}

size_t select_partial_bytes(const ks_model& model, int P, int C, int64_t pairs, bool segmented, int k, bool lean) {
  const int64_t per = per_problem_rows(P, C, pairs, segmented);
  if (model.kind == 0 && model.gbdt.fast) {
    int nblk, rows;
    fast_tiling(model.gbdt, P, per, &nblk, &rows);
    const size_t part = (static_cast<size_t>(P) * nblk * k * sizeof(unsigned long long) + 255) / 256 * 256;
    if (select_splits(model.gbdt, P, C, pairs, nblk, segmented, lean)) {
      return part + fast_split_bytes(model.gbdt) + 512 +
             std::max(fast_scratch_bytes(model.gbdt, C), fast_tiles_bytes(model.gbdt, P, nblk));
    }
    const size_t memo = (fast_memo_bytes(model.gbdt, P, C, segmented, lean) + 255) / 256 * 256;
    // a dense batch is ranked in similarity order of the catalogue (ks_order.cu)
    const bool classes = memo > 0 && !lean && classes_apply(model.gbdt, P, C, pairs);
    const size_t order = (memo > 0 && P >= kOrderMinProblems && (!segmented || classes))
                             ? (order_scratch_bytes(C) + 255) / 256 * 256 : 0;
    return part + (fast_scratch_bytes(model.gbdt, C) + 255) / 256 * 256 + memo + order +
           (classes ? classes_scratch_bytes(model.gbdt, P, C) : 0);
  }
  if (model.kind == 1 && model.mlp.tc) {
    const int nblk = mlp_tc_blocks_per_problem(P, per);
    const size_t part = (static_cast<size_t>(P) * nblk * k * sizeof(unsigned long long) + 255) / 256 * 256;
    return part + mlp_tc_scratch_bytes(C);
  }
  if (model.kind == 1 && model.mlp.wide) {
    const size_t part = static_cast<size_t>(P) * wide_rank_blocks(per) * k * sizeof(unsigned long long);
    return (part + 255) / 256 * 256 + wide_scratch_bytes(model.mlp, P, pairs, lean);
  }
  if (model.kind == 1 && model.mlp.h_ridge) {
    if (ridge_by_classes(P, C, segmented, lean)) {
      RidgeTables t;
      size_t cleared;
      const size_t part = static_cast<size_t>(P) * ridge_rank_shares(P) * k * sizeof(unsigned long long);
      return (part + 255) / 256 * 256 + ridge_tables(P, C, nullptr, &t, &cleared) + sizeof(RidgeProblem) * static_cast<size_t>(P);
    }
    const size_t part = static_cast<size_t>(P) * ridge_blocks(P, per) * k * sizeof(unsigned long long);
    return (part + 255) / 256 * 256 + ridge_scratch_bytes(P, C) + ridge_memo_bytes(P, C, segmented);
  }
  const int st = pick_sub_tiles(P, per);
  int64_t nblk = (per + static_cast<int64_t>(st) * kBlock - 1) / (static_cast<int64_t>(st) * kBlock);
  if (nblk < 1) nblk = 1;
  return static_cast<size_t>(P) * nblk * k * sizeof(unsigned long long);
}

cudaError_t launch_select(const ks_gpu_desc& desc, const ks_model& model, const ks_problem* d_p,
                          const ks_problem* p_by_value, int P, const ks_candidate* d_c, int C,
                          const int64_t* d_seg_off, const int32_t* d_seg_idx, int64_t pairs, int k,
                          void* d_partial, int32_t* d_topk_idx, float* d_topk_score,
                          cudaStream_t stream, int64_t* launches, int* d_status, cudaEvent_t ev_begin,
                          cudaEvent_t ev_end, const FastWait* wait, const HostNotice* notice) {
  if (P == 0) return cudaSuccess;
  const int64_t per = per_problem_rows(P, C, pairs, d_seg_off != nullptr);
  if (model.kind == 0 && model.gbdt.fast) {
    int nblk, rows;
    fast_tiling(model.gbdt, P, per, &nblk, &rows);
    unsigned long long* part = static_cast<unsigned long long*>(d_partial);
    const size_t part_bytes = (static_cast<size_t>(P) * nblk * k * sizeof(unsigned long long) + 255) / 256 * 256;
    // an under-filled machine: the CTAs share out the blocks' trees (dense form only, where a block covers
    // its rows in one pass)
    const bool splits = select_splits(model.gbdt, P, C, pairs, nblk, d_seg_off != nullptr, wait->lean);  // as sized
    char* mem = static_cast<char*>(d_partial) + part_bytes;
    FastSplit split{};
    // the parts of a block share a tile that is built in front of them; behind the tiles, their sums
    split.tiles = reinterpret_cast<uint8_t*>(mem);
    split.scores = reinterpret_cast<double*>(mem + fast_tiles_bytes(model.gbdt, P, nblk));
    // the memo of the per-pair rows sits behind the per-call table (batches of whole-ensemble CTAs only)
    void* memo_mem = (splits || p_by_value || fast_memo_bytes(model.gbdt, P, C, d_seg_off != nullptr, wait->lean) == 0)
                         ? nullptr
                         : mem + (fast_scratch_bytes(model.gbdt, C) + 255) / 256 * 256;
    // a dense batch of problems: rank the catalogue in similarity order (neighbouring candidates
    // then take similar paths through the trees); the order sits behind the memo
    const int32_t* perm = nullptr;
    ClassCall classes{pairs, nullptr, nullptr};
    const bool use_classes = memo_mem && !wait->lean && classes_apply(model.gbdt, P, C, pairs);
    if (memo_mem && P >= kOrderMinProblems && C > 0 && (!d_seg_off || use_classes)) {
      char* order_mem = static_cast<char*>(memo_mem) + (fast_memo_bytes(model.gbdt, P, C, d_seg_off != nullptr, wait->lean) + 255) / 256 * 256;
      cudaError_t eo = launch_catalogue_order(d_c, C, order_mem, stream, launches);
      if (eo != cudaSuccess) return eo;
      if (!d_seg_off) perm = reinterpret_cast<const int32_t*>(order_mem);
      classes.order = reinterpret_cast<const int*>(order_mem);
      classes.scratch = order_mem + (order_scratch_bytes(C) + 255) / 256 * 256;
    }
    cudaError_t e = launch_select_fast(desc, model.gbdt, d_p, p_by_value, P, d_c, C, nblk, rows, d_seg_off,
                                       d_seg_idx, k, part, mem, d_status,
                                       stream, launches, ev_begin, splits && !p_by_value ? &split : nullptr, memo_mem, wait,
                                       nullptr, perm, use_classes ? &classes : nullptr);
    if (e != cudaSuccess) return e;
    if (ev_end) cudaEventRecord(ev_end, stream);
    return launch_merge(part, P, nblk * k, k, d_topk_idx, d_topk_score, stream, launches, notice, ev_end != nullptr);
  }
  if (model.kind == 1 && model.mlp.tc) {
    const int nblk = mlp_tc_blocks_per_problem(P, per);
    unsigned long long* part = static_cast<unsigned long long*>(d_partial);
    const size_t part_bytes = (static_cast<size_t>(P) * nblk * k * sizeof(unsigned long long) + 255) / 256 * 256;
    cudaError_t e = launch_select_mlp_tc(desc, model.mlp, d_p, p_by_value, P, d_c, C, nblk, d_seg_off, d_seg_idx, k,
                                         part, static_cast<char*>(d_partial) + part_bytes, d_status, stream,
                                         launches, ev_begin, wait);
    if (e != cudaSuccess) return e;
    if (ev_end) cudaEventRecord(ev_end, stream);
    return launch_merge(part, P, nblk * k, k, d_topk_idx, d_topk_score, stream, launches, notice, ev_end != nullptr);
  }
  if (model.kind == 1 && model.mlp.wide) {
    const int nblk = wide_rank_blocks(per);
    unsigned long long* part = static_cast<unsigned long long*>(d_partial);
    const size_t part_bytes = (static_cast<size_t>(P) * nblk * k * sizeof(unsigned long long) + 255) / 256 * 256;
    cudaError_t e = launch_select_wide(desc, model.mlp, d_p, p_by_value, P, d_c, C, nblk, d_seg_off, d_seg_idx, pairs, k,
                                       part, static_cast<char*>(d_partial) + part_bytes, d_status, stream, launches,
                                       ev_begin, wait);
    if (e != cudaSuccess) return e;
    if (ev_end) cudaEventRecord(ev_end, stream);
    return launch_merge(part, P, nblk * k, k, d_topk_idx, d_topk_score, stream, launches, notice, ev_end != nullptr);
  }
  if (model.kind == 1 && model.mlp.h_ridge) {
    const RidgeParams& prm = *model.mlp.h_ridge;
    ks_problem pv{};
    if (p_by_value) pv = *p_by_value;
    if (ridge_by_classes(P, C, d_seg_off != nullptr, wait->lean)) {
      const int shares = ridge_rank_shares(P);
      unsigned long long* partial = static_cast<unsigned long long*>(d_partial);
      char* mem = static_cast<char*>(d_partial) + (static_cast<size_t>(P) * shares * k * sizeof(unsigned long long) + 255) / 256 * 256;
      RidgeTables t;
      size_t cleared;
      RidgeProblem* d_prob = reinterpret_cast<RidgeProblem*>(mem + ridge_tables(P, C, mem, &t, &cleared));
      cudaError_t e = cudaMemsetAsync(mem, 0, cleared, stream);
      if (e != cudaSuccess) return e;
      const dim3 all((C + 255) / 256, 16);
      ridge_problem_kernel<<<(P + 127) / 128, 128, 0, stream>>>(desc, d_p, pv, p_by_value != nullptr, P, prm, d_prob, t.mask);
      ridge_members_kernel<<<all, 256, 0, stream>>>(desc, d_c, C, prm, t);
      ridge_classes_kernel<<<dim3(kRidgeCap / 256, 16), 256, 0, stream>>>(desc, d_c, t);
      ridge_list_kernel<<<all, 256, 0, stream>>>(C, t);
      if (ev_begin) cudaEventRecord(ev_begin, stream);
      ridge_rank_kernel<<<dim3(ridge_rank_grid(P), shares), kRidgeRankThreads, 0, stream>>>(
          desc, d_prob, P, d_c, C, prm, k, t, shares > 1 ? partial : nullptr, d_topk_idx, d_topk_score);
      *launches += 5;
      e = cudaGetLastError();
      if (e != cudaSuccess) return e;
      if (ev_end) cudaEventRecord(ev_end, stream);
      return shares > 1 ? launch_merge(partial, P, shares * k, k, d_topk_idx, d_topk_score, stream, launches, nullptr, ev_end != nullptr) : cudaSuccess;
    }
    // per-call tables of what a problem, a candidate and (segments) a class bring, then the kernel that adds
    // and ranks
    PairMap map = make_map(P, C, pairs, d_seg_off, d_seg_idx, kBlock);
    map.nblk = ridge_blocks(P, per);
    unsigned long long* partial = static_cast<unsigned long long*>(d_partial);
    const size_t part_bytes = (static_cast<size_t>(P) * map.nblk * k * sizeof(unsigned long long) + 255) / 256 * 256;
    char* mem = static_cast<char*>(d_partial) + part_bytes;
    unsigned* d_mask = reinterpret_cast<unsigned*>(mem);
    float2* d_tab = reinterpret_cast<float2*>(mem + 256);
    RidgeProblem* d_prob =
        reinterpret_cast<RidgeProblem*>(mem + 256 + (sizeof(float2) * 16 * static_cast<size_t>(C) + 255) / 256 * 256);
    cudaError_t e = cudaMemsetAsync(d_mask, 0, sizeof(unsigned), stream);
    if (e != cudaSuccess) return e;
    ridge_problem_kernel<<<(P + 127) / 128, 128, 0, stream>>>(desc, d_p, pv, p_by_value != nullptr, P, prm, d_prob, d_mask);
    ++*launches;
    MemoView memo{};
    if (ridge_memo_bytes(P, C, d_seg_off != nullptr) != 0) {  // (never for a single problem)
      memo = memo_view(mem + ridge_scratch_bytes(P, C), C);
      e = memo_clear(memo, stream);
      if (e != cudaSuccess) return e;
    }
    if (C > 0) {
      ridge_cand_kernel<<<dim3((C + 255) / 256, 16), 256, 0, stream>>>(desc, d_c, C, d_mask, prm, d_tab, memo);
      ++*launches;
      if (memo.keys) {
        e = memo_compact(memo, stream);
        if (e != cudaSuccess) return e;
        // As for trees (ks_gbdt_fast.cu): a problem of a short segment does not pay for all of the pool's classes. Mixed types,
        // 61,085 valid candidates: 1,000 segments of 300 643 -> 109 us, of 4,000 710 -> 251, 300 of 8,000 299 -> 224.
        const int most = static_cast<int>(std::max<int64_t>(4096, per));
        ridge_pack_kernel<<<dim3((C + 255) / 256, 16), 256, 0, stream>>>(C, d_mask, memo, d_tab, most);
        // enough blocks for 2,048 classes a problem; they loop over more
        ridge_pair_kernel<<<dim3(P < 512 ? 8 : 2, P), 256, 0, stream>>>(desc, d_prob, d_c, prm, memo, most);
        *launches += 3;
      }
    }
    if (ev_begin) cudaEventRecord(ev_begin, stream);
    auto kernel = memo.keys ? &select_ridge_kernel<true> : &select_ridge_kernel<false>;
    kernel<<<static_cast<unsigned>(static_cast<int64_t>(P) * map.nblk), kRidgeThreads, 0, stream>>>(
        desc, d_prob, d_c, map, d_tab, prm, k, partial, memo);
    ++*launches;
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    if (ev_end) cudaEventRecord(ev_end, stream);
    return launch_merge(partial, P, map.nblk * k, k, d_topk_idx, d_topk_score, stream, launches, notice, ev_end != nullptr);
  }
  const int st = pick_sub_tiles(P, per);
  const PairMap map = make_map(P, C, pairs, d_seg_off, d_seg_idx, st * kBlock);
  unsigned long long* partial = static_cast<unsigned long long*>(d_partial);
  const unsigned grid = static_cast<unsigned>(static_cast<int64_t>(P) * map.nblk);
  ks_problem pv{};
  if (p_by_value) pv = *p_by_value;
  cudaError_t e;
  if (ev_begin) cudaEventRecord(ev_begin, stream);
  if (model.kind == 2) {
    select_generic_kernel<true><<<grid, kBlock, 0, stream>>>(desc, d_p, pv, p_by_value != nullptr, d_c, map, st, nullptr,
                                                             nullptr, 0, 0.0f, k, partial);
  } else {
    const GbdtModel& g = model.gbdt;
    const size_t smem = sizeof(float) * kRow * kBlock;
    e = ensure_dynamic_smem(reinterpret_cast<const void*>(&select_generic_kernel<false>), smem);
    if (e != cudaSuccess) return e;
    select_generic_kernel<false><<<grid, kBlock, smem, stream>>>(desc, d_p, pv, p_by_value != nullptr, d_c, map, st,
                                                                 g.d_nodes, g.d_roots, g.n_trees, g.base, k, partial);
  }
  ++*launches;
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  if (ev_end) cudaEventRecord(ev_end, stream);
  return launch_merge(partial, P, map.nblk * k, k, d_topk_idx, d_topk_score, stream, launches, notice, ev_end != nullptr);
}


// Generic tree select with caller-provided node arrays and partial-list storage (dense form).
int64_t select_generic_partial_keys(int P, int C, int k) {
  const int st = pick_sub_tiles(P, C);
  const PairMap map = make_map(P, C, static_cast<int64_t>(P) * C, nullptr, nullptr, st * kBlock);
  return static_cast<int64_t>(P) * map.nblk * k;
}

cudaError_t launch_select_generic_trees(const ks_gpu_desc& desc, const DevNode* d_nodes, const int* d_roots,
                                        int n_trees, float base, const ks_problem* d_p, int P,
                                        const ks_candidate* d_c, int C, int k, unsigned long long* partial,
                                        int32_t* d_topk_idx, float* d_topk_score, cudaStream_t stream) {
  const int st = pick_sub_tiles(P, C);
  const PairMap map = make_map(P, C, static_cast<int64_t>(P) * C, nullptr, nullptr, st * kBlock);
  const size_t smem = sizeof(float) * kRow * kBlock;
  cudaError_t e = ensure_dynamic_smem(reinterpret_cast<const void*>(&select_generic_kernel<false>), smem);
  if (e != cudaSuccess) return e;
  select_generic_kernel<false><<<static_cast<unsigned>(static_cast<int64_t>(P) * map.nblk), kBlock, smem, stream>>>(
      desc, d_p, ks_problem{}, 0, d_c, map, st, d_nodes, d_roots, n_trees, base, k, partial);
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  return launch_merge(partial, P, map.nblk * k, k, d_topk_idx, d_topk_score, stream, nullptr);
}

size_t featurize_scratch_bytes(int P) { return sizeof(ProblemEntry) * static_cast<size_t>(P > 0 ? P : 1); }

}  // namespace ks
