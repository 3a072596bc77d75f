// Device-side pieces shared by the two kernels that walk the quantised form of a tree ensemble
// (ks_gbdt_fast.cu, ks_gbdt_classes.cu): barriers and copies, the search that turns a feature value
// into the bytes of its rows, and the view of a model.
#pragma once

#include <cstddef>
#include <cstdint>

#include "ks_features.cuh"
#include "ks_internal.h"

namespace ks {
namespace {

constexpr int kSlice = 127;            // thresholds per row: a byte is 0x80 | (0..127)
constexpr unsigned kSleepNs = 1200;    // asked-for sleep between two probes of a chunk barrier (400 to 2500 measured alike)

#ifdef KS_DEBUG_BOUNDS
// Checked build: every index formed from data (tile byte, node, chunk, record, partial list) is
// compared with its range; a violation records its source line in this word and uses element 0.
__device__ int g_bounds_line;
__device__ __forceinline__ long long checked_index(long long i, long long n, int line) {
  if (i < 0 || i >= n) {
    atomicCAS(&g_bounds_line, 0, line);
    return 0;
  }
  return i;
}
#define KS_IDX(i, n) checked_index(static_cast<long long>(i), static_cast<long long>(n), __LINE__)
#else
#define KS_IDX(i, n) (i)
#endif

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ void mbar_init(uint32_t bar, int count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count));
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_test_wait(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}
// The same, but the thread may be suspended by the barrier for some time.
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}
// Bounded wait: one probe, then sleep-and-probe (measured faster than the blocking try_wait with
// or without a time hint); gives up after `limit` probes, or as soon as another warp of the CTA
// has given up (`fail`), and reports false.
__device__ __forceinline__ bool mbar_wait_bounded(uint32_t bar, uint32_t parity, int limit, volatile int* fail) {
  if (mbar_test_wait(bar, parity)) return true;
  for (int i = 0; i < limit; ++i) {
    __nanosleep(kSleepNs);
    if (mbar_test_wait(bar, parity)) return true;
    if ((i & 63) == 63 && *fail) return false;
  }
  return false;
}
__device__ __forceinline__ void bulk_copy_g2s(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
      "l"(src), "r"(bytes), "r"(bar)
      : "memory");
}
__device__ __forceinline__ void fence_async_proxy() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

__device__ __forceinline__ uint32_t lds_u32(uint32_t addr) {
  uint32_t v;
  asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(addr));
  return v;
}
__device__ __forceinline__ void lds_u64(uint32_t addr, uint32_t& a, uint32_t& b) {
  asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(a), "=r"(b) : "r"(addr));
}
__device__ __forceinline__ void lds_u128(uint32_t addr, uint32_t& a, uint32_t& b, uint32_t& c, uint32_t& d) {
  asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(a), "=r"(b), "=r"(c), "=r"(d) : "r"(addr));
}
__device__ __forceinline__ float lds_f32(uint32_t addr) {
  float v;
  asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(addr));
  return v;
}

// #{j < n : T[j] <= v} over n sorted thresholds.
__device__ __forceinline__ int count_le(const float* T, int n, float v) {
  int pos = 0;
  for (int s = n > 0 ? 1 << (31 - __clz(n)) : 0; s >= 1; s >>= 1) {
    const int np = pos + s;
    if (np <= n && T[np - 1] <= v) pos = np;
  }
  return pos;
}

// Tile bytes of one feature value: slice s of the feature's thresholds gets the number of its
// thresholds that are <= v, i.e. the overall count less 127 s clamped to 0..127; a rank row gets
// the rank of the level code v. `T` is the feature's own sorted threshold array. With
// `nan_right` a NaN takes the last bin of every slice (x < t is false: it goes right).
// `pos` is the count of the feature's thresholds that are <= v (unused for a feature without slices).
template <typename Put>
__device__ __forceinline__ void emit_rows(const FeatQ& q, int pos, float v, Put put) {
  if (q.nslice) {
    for (int s = 0; s < q.nslice; ++s) {
      int b = pos - kSlice * s;
      b = b < 0 ? 0 : (b > kSlice ? kSlice : b);
      put(q.row0 + s, static_cast<uint8_t>(0x80 | b));
    }
  }
  if (q.nrank) {
    const int code = __float2int_rz(v);
    for (int r = 0; r < q.nrank; ++r)
      put(q.row0 + q.nslice + r, static_cast<uint8_t>(0x80 | ((code >= 0 && code < 4) ? q.rank[r][code] : 0)));
  }
}
template <typename Put>
__device__ __forceinline__ void quantise(const FeatQ& q, const float* T, float v, bool nan_right, Put put) {
  const int pos = q.nslice ? ((nan_right && v != v) ? q.nthr : count_le(T, q.nthr, v)) : 0;
  emit_rows(q, pos, v, put);
}

// All per-pair columns of one pair at once: the binary searches advance in step (one probe of
// every column per round), so that a thread has 21 independent loads in flight instead of one
// dependent chain after the other. `T` is the staged (or global) array of per-pair thresholds.
template <typename Put>
__device__ __forceinline__ void quantise_pair_columns(const FeatQ* s_fq, const float* T, const float (&v)[kPairCols],
                                                      int max_thr, Put put) {
  int pos[kPairCols];
#pragma unroll
  for (int i = 0; i < kPairCols; ++i) pos[i] = 0;
  for (int s = max_thr > 0 ? 1 << (31 - __clz(max_thr)) : 0; s >= 1; s >>= 1) {
#pragma unroll
    for (int i = 0; i < kPairCols; ++i) {
      const FeatQ& q = s_fq[pair_col(i)];
      const int np = pos[i] + s;
      if (np <= q.nthr && T[q.thr0 + np - 1] <= v[i]) pos[i] = np;
    }
  }
#pragma unroll
  for (int i = 0; i < kPairCols; ++i) emit_rows(s_fq[pair_col(i)], pos[i], v[i], put);
}

struct FastView {
  int n_rows, n_pair_rows, n_cand_rows, n_prob_rows;  // rows are ordered pair, candidate, problem
  int depth, n_chunks, chunk_bytes, tpc;
  int n_thr, thr_cand0, thr_prob0;  // thresholds in all, and where the candidate-only / problem-only features' begin
  int cand_rec, pair_rec;           // bytes per record of the per-call tables (multiples of 16)
  int wait_limit, starve;           // probes a chunk wait may take; test hook: arm the barrier for bytes that never come
  int buf_bytes;                    // size of one chunk buffer in shared memory
  float base;
  const uint32_t* chunks;      // [n_chunks][chunk_bytes / 4]
  const float* thr;            // [n_thr] sorted thresholds, feature after feature (per-pair features first)
  const FeatQ* feat;           // [64] rows and thresholds of each feature column
  const uint8_t* cand_rows;    // [kCombos][C][cand_rec] quantised candidate-only rows
  const unsigned* pair_class;  // [kCombos][C] class of every candidate, or null (no memo)
  const uint8_t* pair_tab;     // [P][kMemoCap][pair_rec] per-pair tile bytes of every (problem, class)
  const uint8_t* prob_tab;     // [P][kProbRec] tile bytes of the problem-only rows and the problem's terms, or null
};

// Thresholds of a range of features into shared memory when they fit `cap` floats, else the
// global array is searched in place. Returns the pointer that stands for fv.thr + first.
__device__ __forceinline__ const float* stage_thresholds(const FastView& fv, int first, int count, float* s_thr,
                                                         int cap) {
  if (count > cap) return fv.thr + first;
  const int vec = (first & 3) == 0 ? count / 4 : 0;  // whole 16-byte words when the source is aligned like s_thr
  for (int i = threadIdx.x; i < vec; i += blockDim.x)
    reinterpret_cast<float4*>(s_thr)[i] = __ldg(reinterpret_cast<const float4*>(fv.thr + first) + i);
  for (int i = 4 * vec + threadIdx.x; i < count; i += blockDim.x) s_thr[i] = __ldg(fv.thr + first + i);
  return s_thr;
}

inline int cand_rec_bytes(const GbdtModel& g) { return g.n_cand_rows > 0 ? (g.n_cand_rows + 15) / 16 * 16 : 16; }
inline int pair_rec_bytes(const GbdtModel& g) { return (g.n_pair_rows + 15) / 16 * 16; }

inline FastView make_view(const GbdtModel& g, const FastWait* wait) {
  FastView fv{};
  fv.n_rows = g.n_qrows;
  fv.n_pair_rows = g.n_pair_rows;
  fv.n_cand_rows = g.n_cand_rows;
  fv.n_prob_rows = g.n_prob_rows;
  fv.depth = g.fast_depth;
  fv.n_chunks = g.n_chunks;
  fv.chunk_bytes = g.chunk_bytes;
  fv.tpc = g.tpc;
  fv.n_thr = g.n_qthr;
  fv.thr_cand0 = g.thr_cand0;
  fv.thr_prob0 = g.thr_prob0;
  fv.cand_rec = cand_rec_bytes(g);
  fv.pair_rec = pair_rec_bytes(g);
  fv.wait_limit = wait && wait->limit > 0 ? wait->limit : kFastWaitLimit;
  fv.starve = wait ? wait->starve : 0;
  fv.buf_bytes = g.buf_bytes;
  fv.base = g.base;
  fv.chunks = g.d_qnodes;
  fv.thr = g.d_qthr;
  fv.feat = g.d_qfeat;
  return fv;
}

}  // namespace
}  // namespace ks
