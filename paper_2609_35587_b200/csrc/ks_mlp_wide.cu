// Tensor-core path for feed-forward rankers (Model B) of any width and depth the ABI accepts
// (hidden widths 64 .. 1,024 in steps of 64, up to five hidden layers, both input forms): the
// shapes that do not fit the resident-weights kernel of ks_mlp_tc.cu, the shipped ranker
// 64-1024-1024-512-256-1 among them.
//
// What bounds it: 3.5 MFLOP per pair against 128 bytes of input, so the tensor cores. A layer of
// 1,024 units does not fit shared memory as an operand (128 rows x 1,024 x 2 bytes = 256 KB), so
// both operands stream: two CTAs share one 256-row tile (cta_group::2), each holding its own 128
// rows of A and half of B, which is 32 KB a CTA for 64 of K (16.8 MFLOP) - half of what a CTA of
// its own would fetch. The rows of a tile never leave its pair: the pair takes 256 rows through
// all layers, writes every layer's activations to a scratch of its own that stays in L2 (2 x
// 128 x width x 2 bytes a CTA, 76 MB in all at width 1,024) and reads them back as the next
// layer's A. No CTA waits for another pair. The next layer's first K blocks only need the first
// column tiles of the layer before, so the epilogue of a layer's last tile runs under the next
// layer's MMAs.
// Measured on 16 x 60,000 pairs of the shipped shape (3.4 TFLOP): 4.8 ms a call, of it 4.3 ms in
// the layers (790 TFLOP/s, 0.56 of cuBLAS's sustained rate); a tile MLP on the CUDA cores took
// 440 ms. This kernel is the only one for these shapes. What is left of the gap is the operands' way from L2
// (a K block brings 128 flop a byte, so the sustained rate would need 10.9 TB/s) and the parts that a
// layer's sums are taken in (see part_count; 3.8 ms a call without them). Taking
// two row blocks in turn, so that one's epilogues run under the other's MMAs, measured 4.34 ms for 4.18.
//
// Operand images: K-major with 128-byte swizzle, blocks of [rows][64 of K]: element (row, k) of a
// block sits at row * 128 + (((k / 8) ^ (row % 8)) * 16) + (k % 8) * 2. Inputs, activations and
// weights are kept in global memory in exactly this form, so that a TMA box of [rows][64] is a
// contiguous copy and an epilogue thread writes its row's 128 bytes itself.
#include <cuda.h>
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <new>
#include <vector>

#include "ks_features.cuh"
#include "ks_internal.h"
#include "ks_topk.cuh"

namespace ks {

// Standardisation of the model's input positions, by value.
struct WideInput {
  float mu[KS_F_ONEHOT], sigma[KS_F_ONEHOT];
  int onehot;
};

struct WideMlp {
  int n_hidden = 0;
  int kblocks[KS_MLP_MAX_LAYERS] = {0};  // 64-wide K blocks of every hidden layer
  int width[KS_MLP_MAX_LAYERS] = {0};    // its units
  int wrow[KS_MLP_MAX_LAYERS] = {0};     // first 128-byte row of its weights in the image
  int max_kb = 1;                        // widest stored activation, in K blocks
  int image_rows = 0;
  uint8_t* d_image = nullptr;  // weights, then biases (fp32, 1,024 a layer) and the last layer's weights (fp32)
  float b_last = 0.0f;
  WideInput input;
};

namespace {

constexpr int kThreads = 384;      // warp 0 loads, warp 1 issues MMAs, warps 4..11 are the epilogue
constexpr int kRegs = 168, kRegsFew = 56, kRegsEpilogue = 224;  // a thread's registers at launch, and after the split
static_assert(128 * kRegsFew + 256 * kRegsEpilogue <= kThreads * kRegs, "the split hands out what the block was launched with");
constexpr int kRowsCta = 128, kRowsPair = 256;
constexpr int kStages = 6;
constexpr int kBlockBytes = kRowsCta * 128;        // [128 rows][64 of K] bf16
constexpr int kStageBytes = 2 * kBlockBytes;       // A block, B half block
constexpr int kMaxHidden = KS_MLP_MAX_LAYERS - 1;
constexpr int kMaxBiasBytes = (kMaxHidden + 1) * KS_MLP_MAX_WIDTH * 4;
constexpr int kSmemWide = 1024 + kStages * kStageBytes + kMaxBiasBytes;
constexpr int kPairs = 74;                         // CTA pairs the machine holds (148 SMs)
constexpr int64_t kBatchRows = int64_t{55} * kPairs * kRowsPair;  // rows per launch: whole rounds of all pairs (1.04 M)
constexpr int64_t kScorePairs = 64 * kBatchRows;  // scores held at a time (267 MB)
// ... where the memory for that cannot be had (at most 19 MB in all)
constexpr int64_t kLeanRows = 8 * kRowsPair, kLeanScorePairs = 512 * kLeanRows;
constexpr int64_t batch_rows(bool lean) { return lean ? kLeanRows : kBatchRows; }
constexpr int64_t score_pairs(bool lean) { return lean ? kLeanScorePairs : kScorePairs; }
constexpr int kTileN = 256;

// Parts that a layer's K is summed in. The tensor core adds to its fp32 accumulator by truncation, so that
// what a sum loses grows with the number of its MMAs (16 of K each) and with its size, where additions that
// round lose the square root of their number: measured, a sum over 64 of K has 1.27 times the error of the
// same sum in sequence, one over 1,024 1.66 times (as scores, against 64 bits). So an accumulator takes a
// part of K, and the epilogue adds the parts, which rounds. In the square, p parts of b blocks of 64 lose
// 1.6 b^3 / p^2 where the sequence loses b^2: p is the smallest with 2 p^2 >= 3 b. What a part costs is
// reading its accumulator: 128 KB an SM from TMEM, some 2,300 clocks, beside the 2,000 to 4,600 that its
// MMAs and operands take (16 x 60,000 pairs of the shipped shape: 3.8 ms in one part, 4.8 like this, of it 0.15
// for the two parts of the first layer; parts cut within a block 5.4). Error of that shape, root mean square
// over 320,000 rows: 3.8e-4 in sequence, 6.4e-4 in one part, 3.6e-4 like this.
constexpr int part_count(int kblocks) {
  int p = 1;
  while (2 * p * p < 3 * kblocks) ++p;
  return p;
}

struct WideArgs {
  int n_hidden;
  int kblocks[kMaxHidden], parts[kMaxHidden], width[kMaxHidden], wrow[kMaxHidden];
  int act_kb;                // K blocks per activation buffer
  const float* consts;       // biases [n_hidden][1024], last layer's weights [1024]
  float b_last;
  uint8_t* act;              // [CTAs][2][act_kb][128][128 bytes]
  float* scores;
  int64_t rows;
  int wait_limit, starve;
  int* leave;   // the context's word kWordWide: raised by a CTA whose wait ran out, cleared by the input kernel in front
  int* status;
};

__device__ __forceinline__ uint32_t smem_addr(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ void bar_init(uint32_t bar, int count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count));
}
__device__ __forceinline__ void bar_expect(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void bar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
// arrives at a barrier of either CTA of the pair (cluster address)
__device__ __forceinline__ void bar_arrive_cluster(uint32_t cluster_bar) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(cluster_bar) : "memory");
}
__device__ __forceinline__ bool bar_try(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n"
      " selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}
__device__ __forceinline__ uint32_t to_cluster(uint32_t addr, uint32_t rank) {
  uint32_t r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
// box of [rows][64] into this CTA's shared memory; completes on a barrier of either CTA of the pair
__device__ __forceinline__ void tma_load(uint32_t dst, const CUtensorMap* map, int row, uint32_t cluster_bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes.cta_group::2 "
      "[%0], [%1, {%2, %3}], [%4];" ::"r"(dst),
      "l"(map), "r"(0), "r"(row), "r"(cluster_bar)
      : "memory");
}
__device__ __forceinline__ void fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// shared-memory matrix descriptor: K-major, 128-byte swizzle, groups of eight rows 1,024 bytes apart
__device__ __forceinline__ uint64_t operand_desc(uint32_t saddr) {
  return static_cast<uint64_t>((saddr >> 4) & 0x3FFFu) | (1ull << 16) | (64ull << 32) | (1ull << 46) | (2ull << 61);
}
// D fp32, A and B bf16, K-major, M = 256 over the pair, N = n
__device__ __forceinline__ uint32_t instr_desc(int n) {
  return (1u << 4) | (1u << 7) | (1u << 10) | (static_cast<uint32_t>(n >> 3) << 17) | ((256u >> 4) << 24);
}
__device__ __forceinline__ void mma_pair(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d),
      "l"(a), "l"(b), "r"(idesc), "r"(accumulate)
      : "memory");
}
// arrives at the same barrier of both CTAs once the MMAs issued so far are complete
__device__ __forceinline__ void commit_pair(uint32_t bar) {
  asm volatile(
      "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(bar),
      "h"(static_cast<uint16_t>(3))
      : "memory");
}
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];\n"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
        "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
        "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr));
}
// the loaded registers pass through, so that no use of them moves above the wait
__device__ __forceinline__ void tmem_wait(uint32_t (&r)[32]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
                 "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]),
                 "+r"(r[15]), "+r"(r[16]), "+r"(r[17]), "+r"(r[18]), "+r"(r[19]), "+r"(r[20]), "+r"(r[21]),
                 "+r"(r[22]), "+r"(r[23]), "+r"(r[24]), "+r"(r[25]), "+r"(r[26]), "+r"(r[27]), "+r"(r[28]),
                 "+r"(r[29]), "+r"(r[30]), "+r"(r[31])
               :
               : "memory");
}
// ReLU of both, rounded to bf16; of what is not a number 0 (x > 0 is false; cvt's own .relu keeps it)
__device__ __forceinline__ uint32_t bf16_relu2(float lo, float hi) {
  uint32_t d;
  asm("{\n .reg .b32 t;\n cvt.rn.bf16x2.f32 t, %1, %2;\n max.bf16x2 %0, t, %3;\n}\n" : "=r"(d) : "f"(hi), "f"(lo), "r"(0));
  return d;
}

// barrier of the eight epilogue warps that also says whether `v` holds for all their threads
__device__ __forceinline__ bool epilogue_and(bool v) {
  uint32_t r;
  asm volatile(
      "{\n .reg .pred p, q;\n setp.ne.u32 p, %1, 0;\n barrier.cta.red.and.pred q, 1, 256, p;\n selp.u32 %0, 1, 0, q;\n}\n"
      : "=r"(r)
      : "r"(static_cast<uint32_t>(v))
      : "memory");
  return r != 0;
}

// ------------------------------------------------------------------------------------------
// the input rows: features (or given rows), standardised, rounded to bf16, in operand form
// ------------------------------------------------------------------------------------------

// One thread builds one row and writes its 128 (one-hot form: 256) bytes. Rows past the last one up
// to the end of their 256-row tile are zero.
template <bool kOneHot>
__device__ __forceinline__ void store_input_row(const WideInput& in, const float (&x)[KS_F_PAD], bool live, int64_t row,
                                                uint8_t* image) {
  constexpr int kKb = kOneHot ? 2 : 1;
  uint8_t* base = image + (row / kRowsCta) * (kKb * kBlockBytes) + (row % kRowsCta) * 128;
  const int sw = static_cast<int>(row & 7);
#pragma unroll
  for (int chunk = 0; chunk < 8 * kKb; ++chunk) {
    uint32_t w[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      float v[2];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int pos = chunk * 8 + 2 * q + h;
        float f = 0.0f;
        bool used;
        if (!kOneHot) {
          used = pos < KS_F;
          if (used) f = x[pos < KS_F ? pos : 0];
        } else {
          // the columns other than 5, 9, 17, 18 in order, then the level indicators of those four
          used = pos < 73;
          if (pos < 59) {
            f = x[pos + (pos >= 5) + (pos >= 8) + 2 * (pos >= 15)];
          } else if (used) {
            const int p = pos - 59;
            const int col = p < 4 ? 5 : (p < 7 ? 9 : (p < 11 ? 17 : 18));
            const int level = p < 4 ? p : (p < 7 ? p - 4 : (p < 11 ? p - 7 : p - 11));
            f = __float2int_rz(x[col]) == level ? 1.0f : 0.0f;
          }
        }
        if (used) {
          if (!isfinite(f)) f = 0.0f;
          f = __fdiv_rn(__fsub_rn(f, in.mu[pos]), in.sigma[pos]);
        }
        v[h] = (used && live) ? f : 0.0f;
      }
      const __nv_bfloat162 t = __floats2bfloat162_rn(v[0], v[1]);
      w[q] = *reinterpret_cast<const uint32_t*>(&t);
    }
    *reinterpret_cast<uint4*>(base + (chunk / 8) * kBlockBytes + (((chunk & 7) ^ sw) * 16)) =
        make_uint4(w[0], w[1], w[2], w[3]);
  }
}

__global__ void __launch_bounds__(128)
wide_terms_kernel(ks_gpu_desc desc, const ks_problem* __restrict__ p, ks_problem p_value, int use_value, int P,
                  ProblemTerms* __restrict__ terms) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < P) problem_terms(use_value ? p_value : load_problem(p + i), desc, terms[i]);
}

// rows first .. first + n - 1 of the call's pairs
template <bool kOneHot>
__global__ void __launch_bounds__(128)
wide_pair_rows_kernel(ks_gpu_desc desc, const ProblemTerms* __restrict__ terms, int P, const ks_candidate* __restrict__ c,
                      int C, const int64_t* __restrict__ seg_off, const int32_t* __restrict__ seg_idx, int64_t first,
                      int64_t n, int64_t n_padded, const __grid_constant__ WideInput in, uint8_t* __restrict__ image, int* leave) {
  if (blockIdx.x == 0 && threadIdx.x == 0) *leave = 0;
  const int64_t r = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (r >= n_padded) return;
  float x[KS_F_PAD];
#pragma unroll
  for (int q = 0; q < KS_F_PAD; ++q) x[q] = 0.0f;
  const bool live = r < n;
  if (live) {
    const int64_t pair = first + r;
    int prob, idx;
    if (seg_off) {
      int lo = 0, hi = P - 1;  // the last problem whose segment starts at or before the pair
      while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (seg_off[mid] <= pair) lo = mid;
        else hi = mid - 1;
      }
      prob = lo;
      idx = seg_idx[pair];
    } else {
      prob = static_cast<int>(pair / C);
      idx = static_cast<int>(pair - static_cast<int64_t>(prob) * C);
    }
    const ProblemTerms t = terms[prob];
    featurize_pair(t, load_candidate(c + idx), desc, [&](int col, float v) { x[col] = v; });
  }
  store_input_row<kOneHot>(in, x, live, r, image);
}

template <bool kOneHot>
__global__ void __launch_bounds__(128)
wide_given_rows_kernel(const float* __restrict__ feat, int64_t n, int64_t n_padded,
                       const __grid_constant__ WideInput in, uint8_t* __restrict__ image, int* leave) {
  if (blockIdx.x == 0 && threadIdx.x == 0) *leave = 0;
  const int64_t r = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (r >= n_padded) return;
  float x[KS_F_PAD];
  const float4* src = reinterpret_cast<const float4*>(feat + (r < n ? r : 0) * KS_F_PAD);
#pragma unroll
  for (int q = 0; q < KS_F_PAD / 4; ++q) {
    const float4 v = __ldg(src + q);
    x[4 * q] = v.x; x[4 * q + 1] = v.y; x[4 * q + 2] = v.z; x[4 * q + 3] = v.w;
  }
  store_input_row<kOneHot>(in, x, r < n, r, image);
}

// ------------------------------------------------------------------------------------------
// the layers
// ------------------------------------------------------------------------------------------

__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kThreads, 1)
mlp_wide_kernel(const __grid_constant__ WideArgs a, const __grid_constant__ CUtensorMap map_x,
                const __grid_constant__ CUtensorMap map_act, const __grid_constant__ CUtensorMap map_w32,
                const __grid_constant__ CUtensorMap map_w64, const __grid_constant__ CUtensorMap map_w96,
                const __grid_constant__ CUtensorMap map_w128) {
  extern __shared__ unsigned char smem_raw[];
  // full[kStages] (the leader's are used), empty[kStages], accumulator full[2] and read out[2] (the
  // leader's), a stored column tile of the layer before [4]
  __shared__ __align__(8) unsigned long long s_bar[2 * kStages + 8];
  __shared__ uint32_t s_tmem;
  __shared__ float s_half[2][kRowsCta];
  __shared__ int s_fail, s_abort;

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t rank = blockIdx.x & 1;  // CTA of the pair; 0 issues the MMAs
  const int pair = blockIdx.x >> 1, n_pairs = gridDim.x >> 1;
  unsigned char* smem = smem_raw + ((1024u - (smem_addr(smem_raw) & 1023u)) & 1023u);
  float* s_const = reinterpret_cast<float*>(smem + kStages * kStageBytes);
  const uint32_t bar0 = smem_addr(&s_bar[0]);
  auto bar_full = [&](int s) { return bar0 + 8u * s; };
  auto bar_empty = [&](int s) { return bar0 + 8u * (kStages + s); };
  auto bar_acc = [&](int i) { return bar0 + 8u * (2 * kStages + i); };
  auto bar_read = [&](int i) { return bar0 + 8u * (2 * kStages + 2 + i); };
  auto bar_stored = [&](int i) { return bar0 + 8u * (2 * kStages + 4 + i); };

  if (tid == 0) {
    s_abort = *reinterpret_cast<volatile int*>(a.leave);
    if (s_abort && a.status) atomicExch(a.status, KS_ERR_TIMEOUT);
    s_fail = 0;
    for (int s = 0; s < kStages; ++s) {
      bar_init(bar_full(s), 1);
      bar_init(bar_empty(s), 1);
    }
    for (int i = 0; i < 2; ++i) {
      bar_init(bar_acc(i), 1);
      bar_init(bar_read(i), 16);  // eight epilogue warps of each CTA
    }
    for (int i = 0; i < 4; ++i) bar_init(bar_stored(i), 8);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 2) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(&s_tmem)), "r"(512)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  for (int i = tid; i < (a.n_hidden + 1) * KS_MLP_MAX_WIDTH / 4; i += kThreads)
    reinterpret_cast<float4*>(s_const)[i] = __ldg(reinterpret_cast<const float4*>(a.consts) + i);
  fence_before();
  __syncthreads();
  cluster_sync();  // both CTAs' barriers exist before either is used
  fence_after();
  const uint32_t tmem = s_tmem;
  const uint32_t sbase = smem_addr(smem);
  const int64_t n_blocks = (a.rows + kRowsPair - 1) / kRowsPair;
  volatile int* v_fail = &s_fail;

  // Bounded wait; after the first that runs out every role of the CTA leaves its loop (the pair's
  // other CTA runs into its own limit), and CTAs that start later run no tile.
  auto wait_ok = [&](uint32_t bar, uint32_t parity) {
    for (int i = 0; i < a.wait_limit; ++i) {
      if (bar_try(bar, parity)) return true;
      if ((i & 63) == 63 && *v_fail) return false;
    }
    *v_fail = 1;
    atomicExch(a.leave, kLeaveFailed);
    if (a.status) atomicExch(a.status, KS_ERR_TIMEOUT);
    return false;
  };

  const int64_t b_first = s_abort ? n_blocks : pair;
  // the epilogue keeps 128 sums a thread: it takes the registers that the first four warps do without
  if (warp < 4) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kRegsFew));
    if (warp == 0) {
      // ---------------------------------- loads -------------------------------------------------------
      if (lane == 0) {
        const uint32_t stage0 = sbase;
        uint32_t it = 0, ph_stored = 0;
        bool ok = true;
        for (int64_t blk = b_first; blk < n_blocks && ok; blk += n_pairs) {
          for (int l = 0; l < a.n_hidden && ok; ++l) {
            const int kbs = a.kblocks[l], width = a.width[l];
            for (int n0 = 0; n0 < width && ok; n0 += kTileN) {
              const int nt = width - n0 < kTileN ? width - n0 : kTileN;
              const CUtensorMap* mw = nt == 256 ? &map_w128 : (nt == 192 ? &map_w96 : (nt == 128 ? &map_w64 : &map_w32));
              const int wrow = a.wrow[l] + n0 * kbs + static_cast<int>(rank) * (nt / 2);
              for (int kb = 0; kb < kbs; ++kb) {
                if (l > 0 && n0 == 0 && (kb & 3) == 0) {
                  // the column tile of the layer before that holds these K blocks is stored
                  const int t = kb >> 2;
                  if (!(ok = wait_ok(bar_stored(t), (ph_stored >> t) & 1u))) break;
                  ph_stored ^= 1u << t;
                  asm volatile("fence.proxy.async;" ::: "memory");
                }
                const int s = static_cast<int>(it % kStages);
                if (!(ok = wait_ok(bar_empty(s), ((it / kStages) & 1u) ^ 1u))) break;
                const uint32_t full = to_cluster(bar_full(s), 0);
                if (rank == 0) bar_expect(bar_full(s), 2u * (kBlockBytes + nt / 2 * 128));
                if (!a.starve) {  // test hook: without the copies the waits on this barrier run out
                  const uint32_t dst = stage0 + s * kStageBytes;
                  if (l == 0) tma_load(dst, &map_x, static_cast<int>(((blk * 2 + rank) * kbs + kb) * kRowsCta), full);
                  else tma_load(dst, &map_act, static_cast<int>(((blockIdx.x * 2 + (l & 1)) * a.act_kb + kb) * kRowsCta), full);
                  tma_load(dst + kBlockBytes, mw, wrow + kb * nt, full);
                }
                ++it;
              }
            }
          }
        }
      }
      __syncwarp();
    } else if (warp == 1) {
      // ---------------------------------- MMAs --------------------------------------------------------
      if (rank == 0 && lane == 0) {
        uint32_t it = 0, part = 0;
        bool ok = true;
        for (int64_t blk = b_first; blk < n_blocks && ok; blk += n_pairs) {
          for (int l = 0; l < a.n_hidden && ok; ++l) {
            const int kbs = a.kblocks[l], parts = a.parts[l], width = a.width[l];
            for (int n0 = 0; n0 < width && ok; n0 += kTileN) {
              const int nt = width - n0 < kTileN ? width - n0 : kTileN;
              const uint32_t idesc = instr_desc(nt);
              for (int j = 0; j < parts && ok; ++j, ++part) {
                const uint32_t acc = part & 1u;
                if (!(ok = wait_ok(bar_read(acc), ((part >> 1) & 1u) ^ 1u))) break;
                fence_after();
                // whole blocks, or (a layer of one block) 32 of K
                const int first = kbs > 1 ? 4 * (kbs * j / parts) : 4 * j / parts;
                const int stop = kbs > 1 ? 4 * (kbs * (j + 1) / parts) : 4 * (j + 1) / parts;
                for (int u = first; u < stop; u = (u | 3) + 1) {
                  const int s = static_cast<int>(it % kStages);
                  if ((u & 3) == 0) {  // (a block that the part before has begun is there)
                    if (!(ok = wait_ok(bar_full(s), (it / kStages) & 1u))) break;
                    fence_after();
                  }
                  const uint64_t da = operand_desc(sbase + s * kStageBytes);
                  const uint64_t db = operand_desc(sbase + s * kStageBytes + kBlockBytes);
#pragma unroll
                  for (int k16 = 0; k16 < 4; ++k16)  // 32 bytes on in K: two units of the address field
                    if (k16 >= (u & 3) && (u & ~3) + k16 < stop)
                      mma_pair(tmem + acc * 256u, da + 2u * k16, db + 2u * k16, idesc, (u & ~3) + k16 > first);
                  if ((u | 3) < stop) {
                    commit_pair(bar_empty(s));
                    ++it;
                  }
                }
                if (ok) commit_pair(bar_acc(acc));
              }
            }
          }
        }
      }
      __syncwarp();
    }
  } else {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kRegsEpilogue));
    // ---------------------------------- epilogue ----------------------------------------------------
    // warp w owns lanes 32 (w % 4) .. and one half of a tile's columns
    const int quarter = warp & 3, half = (warp - 4) >> 2;
    const int trow = quarter * 32 + lane;
    const uint32_t tmem_row = tmem + (static_cast<uint32_t>(quarter * 32) << 16);
    int pending = -1;  // column tile whose rows are written but not yet announced
    auto publish = [&]() {
      if (pending < 0) return;
      // the rows are written; what the loading thread issues next must see them
      __threadfence();
      asm volatile("fence.proxy.async;" ::: "memory");
      __syncwarp();
      if (lane == 0) bar_arrive(bar_stored(pending));
      pending = -1;
    };
    uint32_t part = 0, blk_par = 0;  // s_half is written for every other block in turn
    bool ok = true;
    for (int64_t blk = b_first; blk < n_blocks && ok; blk += n_pairs, blk_par ^= 1u) {
      float score = 0.0f;
      for (int l = 0; l < a.n_hidden && ok; ++l) {
        const int parts = a.parts[l], width = a.width[l];
        const bool last = l + 1 == a.n_hidden;
        const float* bias = s_const + l * KS_MLP_MAX_WIDTH;
        const float* w_last = s_const + a.n_hidden * KS_MLP_MAX_WIDTH;
        uint8_t* out = a.act + (static_cast<size_t>(blockIdx.x * 2 + ((l + 1) & 1)) * a.act_kb) * kBlockBytes + trow * 128;
        for (int n0 = 0; n0 < width && ok; n0 += kTileN) {
          const int nt = width - n0 < kTileN ? width - n0 : kTileN;
          const int cols = nt / 2, c_first = half * cols;  // this warp's columns of the tile: 32 to 128
          const uint32_t tmem_mine = tmem_row + c_first;
          float sum[kTileN / 2];  // over the parts of K
          for (int j = 0; j < parts; ++j, ++part) {
            const uint32_t acc = part & 1u;
            if (!(ok = __all_sync(0xFFFFFFFFu, wait_ok(bar_acc(acc), (part >> 1) & 1u)))) break;
            fence_after();
#pragma unroll
            for (int c0 = 0; c0 < kTileN / 2; c0 += 32) {
              if (c0 >= cols) break;
              uint32_t r[32];
              tmem_ld32(tmem_mine + acc * 256u + c0, r);
              tmem_wait(r);
              if (j == 0) {
#pragma unroll
                for (int q = 0; q < 32; ++q) sum[c0 + q] = __uint_as_float(r[q]);
              } else {
#pragma unroll
                for (int q = 0; q < 32; ++q) sum[c0 + q] += __uint_as_float(r[q]);
              }
            }
            fence_before();
            if (lane == 0) bar_arrive_cluster(to_cluster(bar_read(acc), 0));
            publish();
          }
          if (!ok) break;
#pragma unroll
          for (int c0 = 0; c0 < kTileN / 2; c0 += 32) {
            if (c0 >= cols) break;
            const int col = n0 + c_first + c0;
            const float4* b4 = reinterpret_cast<const float4*>(bias + col);
            uint32_t h[16];
#pragma unroll
            for (int q = 0; q < 8; ++q) {
              const float4 b = b4[q];
              h[2 * q] = bf16_relu2(sum[c0 + 4 * q] + b.x, sum[c0 + 4 * q + 1] + b.y);
              h[2 * q + 1] = bf16_relu2(sum[c0 + 4 * q + 2] + b.z, sum[c0 + 4 * q + 3] + b.w);
            }
            if (!last) {
              uint8_t* dst = out + static_cast<size_t>(col >> 6) * kBlockBytes;
#pragma unroll
              for (int q = 0; q < 4; ++q)
                *reinterpret_cast<uint4*>(dst + ((((col & 63) >> 3) + q) ^ (trow & 7)) * 16) =
                    make_uint4(h[4 * q], h[4 * q + 1], h[4 * q + 2], h[4 * q + 3]);
            } else {
              const float4* w4 = reinterpret_cast<const float4*>(w_last + col);
#pragma unroll
              for (int q = 0; q < 8; ++q) {
                const float4 w = w4[q];
                score = fmaf(__uint_as_float(h[2 * q] << 16), w.x, score);
                score = fmaf(__uint_as_float(h[2 * q] & 0xFFFF0000u), w.y, score);
                score = fmaf(__uint_as_float(h[2 * q + 1] << 16), w.z, score);
                score = fmaf(__uint_as_float(h[2 * q + 1] & 0xFFFF0000u), w.w, score);
              }
            }
          }
          if (!last) {
            // Announced behind the next part's accumulator, so that its MMAs do not wait for these stores: that
            // part needs nothing of this tile, but where the tile is all of the layer.
            pending = n0 / kTileN;
            if (width <= kTileN) publish();
          }
        }
      }
      // The two halves of the row's columns meet here; a failed wait of any warp ends the loop of
      // all of them in the same round.
      if (half == 1) s_half[blk_par][trow] = score;
      ok = epilogue_and(ok && !*v_fail);
      if (half == 0 && ok) {
        const int64_t row = blk * kRowsPair + rank * kRowsCta + trow;
        if (row < a.rows) a.scores[row] = ((score + s_half[blk_par][trow]) + a.b_last) + 0.0f;
      }
    }
  }
  // after a failure: time for the copies and MMAs in flight to end
  if (*v_fail)
    for (int i = 0; i < 64; ++i) __nanosleep(2000);
  __syncthreads();
  cluster_sync();
  if (warp == 2)
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
}

// ------------------------------------------------------------------------------------------
// ranking of stored scores
// ------------------------------------------------------------------------------------------

constexpr int kRankRows = 8 * kBlock;  // scores one block ranks at a time

// Block (problem, chunk) ranks its share of the problem's scores among the pairs first ..
// first + count - 1, whose scores `scores` holds, and merges them into its partial list (`fresh`:
// the list is empty). Every call with more pairs than the score buffer holds is ranked in rounds.
__global__ void __launch_bounds__(kBlock)
rank_scores_kernel(const float* __restrict__ scores, int64_t first, int64_t count, int fresh, int C, int nblk,
                   const int64_t* __restrict__ seg_off, const int32_t* __restrict__ seg_idx, int k,
                   unsigned long long* __restrict__ partial) {
  __shared__ unsigned long long s_warp[kBlock / 32 * KS_MAX_K];
  __shared__ unsigned long long s_list[KS_MAX_K];
  const int prob = blockIdx.x / nblk, chunk = blockIdx.x % nblk;
  const int64_t lo = seg_off ? seg_off[prob] : static_cast<int64_t>(prob) * C;
  const int64_t len = seg_off ? seg_off[prob + 1] - lo : C;
  const int64_t r_begin = first > lo ? first - lo : 0, r_end = first + count - lo < len ? first + count - lo : len;
  if (!fresh && r_begin >= r_end) return;
  unsigned long long* list = partial + (static_cast<size_t>(prob) * nblk + chunk) * k;
  if (threadIdx.x < KS_MAX_K) s_list[threadIdx.x] = !fresh && threadIdx.x < k ? list[threadIdx.x] : 0ull;
  __syncthreads();
  for (int64_t start = static_cast<int64_t>(chunk) * kRankRows; start < r_end;
       start += static_cast<int64_t>(nblk) * kRankRows) {
    if (start + kRankRows <= r_begin) continue;
    unsigned long long keys[9];
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int64_t r = start + q * kBlock + threadIdx.x;
      keys[q] = r >= r_begin && r < r_end
                    ? make_key(scores[lo + r - first], seg_idx ? seg_idx[lo + r] : static_cast<int>(r)) : 0ull;
    }
    keys[8] = threadIdx.x < k ? s_list[threadIdx.x] : 0ull;
    __syncthreads();
    block_topk<9>(keys, k, s_warp, s_list);
  }
  if (threadIdx.x < k) list[threadIdx.x] = s_list[threadIdx.x];
}

size_t up(size_t v) { return (v + 1023) / 1024 * 1024; }

// ------------------------------------------------------------------------------------------
// host
// ------------------------------------------------------------------------------------------

using EncodeTiled = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                 const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                 CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiled encode_tiled() {
  static const EncodeTiled fn = [] {
    void* f = nullptr;
    cudaDriverEntryPointQueryResult res;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000, cudaEnableDefault, &res) != cudaSuccess ||
        res != cudaDriverEntryPointSuccess)
      f = nullptr;
    return reinterpret_cast<EncodeTiled>(f);
  }();
  return fn;
}

// [rows][64] bf16, boxes of `box_rows` rows; the images are swizzled in memory, so the copy is plain
cudaError_t make_map(CUtensorMap* map, void* base, int64_t rows, int box_rows) {
  const EncodeTiled fn = encode_tiled();
  if (!fn) return cudaErrorNotSupported;
  const cuuint64_t dims[2] = {64, static_cast<cuuint64_t>(rows)};
  const cuuint64_t strides[1] = {128};
  const cuuint32_t box[2] = {64, static_cast<cuuint32_t>(box_rows)};
  const cuuint32_t step[2] = {1, 1};
  return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, base, dims, strides, box, step, CU_TENSOR_MAP_INTERLEAVE_NONE,
            CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS
             ? cudaSuccess
             : cudaErrorInvalidValue;
}

size_t image_bytes(const WideMlp& w, int64_t rows) {
  return static_cast<size_t>((rows + kRowsPair - 1) / kRowsPair) * 2 * kBlockBytes * w.kblocks[0];
}
int pairs_used(int64_t rows) {
  const int64_t n_blocks = (rows + kRowsPair - 1) / kRowsPair;
  return static_cast<int>(n_blocks < kPairs ? n_blocks : kPairs);
}
// two activation buffers for each CTA of a launch over `rows` rows
int64_t act_rows(const WideMlp& w, int64_t rows) {
  return static_cast<int64_t>(2 * pairs_used(rows)) * 2 * w.max_kb * kRowsCta;
}

// the layers over `rows` rows whose operand image is at `image`
cudaError_t launch_layers(const WideMlp& w, uint8_t* image, uint8_t* act, int64_t rows, float* scores, int* status,
                          const FastWait* wait, cudaStream_t stream) {
  WideArgs a{};
  a.n_hidden = w.n_hidden;
  for (int l = 0; l < w.n_hidden; ++l) {
    a.kblocks[l] = w.kblocks[l];
    a.parts[l] = part_count(w.kblocks[l]);
    a.width[l] = w.width[l];
    a.wrow[l] = w.wrow[l];
  }
  a.act_kb = w.max_kb;
  a.consts = reinterpret_cast<const float*>(w.d_image + static_cast<size_t>(w.image_rows) * 128);
  a.b_last = w.b_last;
  a.act = act;
  a.scores = scores;
  a.rows = rows;
  a.wait_limit = wait->limit > 0 ? wait->limit : kMlpWaitLimit;
  a.starve = wait->starve;
  a.leave = wait->words + kWordWide;
  a.status = status;
  const int64_t n_blocks = (rows + kRowsPair - 1) / kRowsPair;
  CUtensorMap mx, ma, mw[4];
  cudaError_t e = make_map(&mx, image, n_blocks * 2 * kRowsCta * w.kblocks[0], kRowsCta);
  if (e == cudaSuccess) e = make_map(&ma, act, act_rows(w, rows), kRowsCta);
  for (int i = 0; i < 4 && e == cudaSuccess; ++i) e = make_map(&mw[i], w.d_image, w.image_rows, 32 * (i + 1));
  if (e == cudaSuccess) e = ensure_dynamic_smem(reinterpret_cast<const void*>(&mlp_wide_kernel), kSmemWide);
  if (e != cudaSuccess) return e;
  mlp_wide_kernel<<<2 * pairs_used(rows), kThreads, kSmemWide, stream>>>(a, mx, ma, mw[0], mw[1], mw[2], mw[3]);
  return cudaGetLastError();
}

}  // namespace

// Builds the weight image of a ranker with at least one hidden layer.
cudaError_t build_wide_mlp(MlpModel& m, const uint16_t* const* h_w, const float* const* h_b, const float* h_mu,
                           const float* h_sigma) {
  if (m.n_layers < 2) return cudaSuccess;
  cudaFuncAttributes attr{};  // the register split is made for this count
  cudaError_t ea = cudaFuncGetAttributes(&attr, reinterpret_cast<const void*>(&mlp_wide_kernel));
  if (ea != cudaSuccess) return ea;
  if (attr.numRegs != kRegs) return cudaErrorInvalidKernelImage;
  WideMlp* w = new (std::nothrow) WideMlp();
  if (!w) return cudaErrorMemoryAllocation;
  m.wide = w;
  w->n_hidden = m.n_layers - 1;
  int rows = 0;
  for (int l = 0; l < w->n_hidden; ++l) {
    w->kblocks[l] = (m.widths[l] + 63) / 64;
    w->width[l] = m.widths[l + 1];
    w->wrow[l] = rows;
    rows += w->kblocks[l] * w->width[l];
    if (l + 1 < w->n_hidden) w->max_kb = std::max(w->max_kb, w->width[l] / 64);
  }
  w->image_rows = rows;
  w->b_last = h_b[m.n_layers - 1][0];
  w->input.onehot = m.widths[0] == KS_F_ONEHOT;
  for (int j = 0; j < KS_F_ONEHOT; ++j) {
    w->input.mu[j] = j < m.widths[0] ? h_mu[j] : 0.0f;
    w->input.sigma[j] = j < m.widths[0] ? h_sigma[j] : 1.0f;
  }
  const size_t const_floats = static_cast<size_t>(w->n_hidden + 1) * KS_MLP_MAX_WIDTH;
  std::vector<uint8_t> img(static_cast<size_t>(rows) * 128 + const_floats * 4, 0);
  float* consts = reinterpret_cast<float*>(img.data() + static_cast<size_t>(rows) * 128);
  for (int l = 0; l < w->n_hidden; ++l) {
    const int in = m.widths[l], width = w->width[l], kbs = w->kblocks[l];
    for (int n = 0; n < width; ++n) {
      const int n0 = n / kTileN * kTileN, nt = std::min(kTileN, width - n0);
      const int half = (n - n0) / (nt / 2), r = (n - n0) % (nt / 2);
      for (int kb = 0; kb < kbs; ++kb) {
        // block (column tile, K block, half): nt / 2 rows of 128 bytes
        uint8_t* dst = img.data() + (static_cast<size_t>(w->wrow[l]) + static_cast<size_t>(n0) * kbs + kb * nt + half * (nt / 2) + r) * 128;
        const uint16_t* src = h_w[l] + static_cast<size_t>(n) * in + kb * 64;
        const int chunks = std::min(64, in - kb * 64) / 8;
        for (int c = 0; c < chunks; ++c) std::memcpy(dst + (c ^ (r & 7)) * 16, src + 8 * c, 16);
      }
    }
    std::memcpy(consts + static_cast<size_t>(l) * KS_MLP_MAX_WIDTH, h_b[l], sizeof(float) * width);
  }
  for (int n = 0; n < m.widths[m.n_layers - 1]; ++n) {
    const uint32_t u = static_cast<uint32_t>(h_w[m.n_layers - 1][n]) << 16;
    std::memcpy(consts + static_cast<size_t>(w->n_hidden) * KS_MLP_MAX_WIDTH + n, &u, 4);
  }
  cudaError_t e = cudaMalloc(reinterpret_cast<void**>(&w->d_image), img.size());
  if (e == cudaSuccess) e = cudaMemcpy(w->d_image, img.data(), img.size(), cudaMemcpyHostToDevice);
  return e;
}

void free_wide_mlp(MlpModel& m) {
  if (!m.wide) return;
  cudaFree(m.wide->d_image);
  delete m.wide;
  m.wide = nullptr;
}

int wide_rank_blocks(int64_t per_problem) {
  const int64_t n = (per_problem + kRankRows - 1) / kRankRows;
  return static_cast<int>(n < 1 ? 1 : n);
}

// problem terms | scores of a round's pairs | operand image of a batch | activations
size_t wide_scratch_bytes(const MlpModel& m, int P, int64_t pairs, bool lean) {
  const int64_t batch = std::min(pairs, batch_rows(lean));
  return up(sizeof(ProblemTerms) * static_cast<size_t>(P > 0 ? P : 1)) + up(sizeof(float) * static_cast<size_t>(std::min(pairs, score_pairs(lean)))) +
         up(image_bytes(*m.wide, batch)) + static_cast<size_t>(act_rows(*m.wide, batch)) * 128 + 1024;
}

cudaError_t launch_select_wide(const ks_gpu_desc& desc, const MlpModel& m, const ks_problem* d_p,
                               const ks_problem* p_by_value, int P, const ks_candidate* d_c, int C, int nblk,
                               const int64_t* seg_off, const int32_t* seg_idx, int64_t pairs, int k,
                               unsigned long long* partial, void* scratch, int* status, cudaStream_t stream,
                               int64_t* launches, cudaEvent_t ev_begin, const FastWait* wait) {
  const WideMlp& w = *m.wide;
  const int64_t batch = batch_rows(wait->lean), round = score_pairs(wait->lean);
  char* q = reinterpret_cast<char*>((reinterpret_cast<uintptr_t>(scratch) + 1023) / 1024 * 1024);
  ProblemTerms* terms = reinterpret_cast<ProblemTerms*>(q);
  q += up(sizeof(ProblemTerms) * static_cast<size_t>(P));
  float* scores = reinterpret_cast<float*>(q);
  q += up(sizeof(float) * static_cast<size_t>(std::min(pairs, round)));
  uint8_t* image = reinterpret_cast<uint8_t*>(q);
  q += up(image_bytes(w, std::min(pairs, batch)));
  uint8_t* act = reinterpret_cast<uint8_t*>(q);
  ks_problem pv{};
  if (p_by_value) pv = *p_by_value;
  wide_terms_kernel<<<(P + 127) / 128, 128, 0, stream>>>(desc, d_p, pv, p_by_value != nullptr, P, terms);
  ++*launches;
  if (ev_begin) cudaEventRecord(ev_begin, stream);
  int64_t first = 0;
  do {  // a round: the scores of so many pairs, then their ranking
    const int64_t round0 = first, round_end = std::min(pairs, round0 + round);
    for (; first < round_end; first += batch) {
      const int64_t n = std::min(round_end - first, batch), padded = (n + kRowsPair - 1) / kRowsPair * kRowsPair;
      const unsigned grid = static_cast<unsigned>((padded + 127) / 128);
      if (w.input.onehot)
        wide_pair_rows_kernel<true><<<grid, 128, 0, stream>>>(desc, terms, P, d_c, C, seg_off, seg_idx, first, n, padded,
                                                              w.input, image, wait->words + kWordWide);
      else
        wide_pair_rows_kernel<false><<<grid, 128, 0, stream>>>(desc, terms, P, d_c, C, seg_off, seg_idx, first, n,
                                                               padded, w.input, image, wait->words + kWordWide);
      cudaError_t e = cudaGetLastError();
      if (e == cudaSuccess) e = launch_layers(w, image, act, n, scores + (first - round0), status, wait, stream);
      if (e != cudaSuccess) return e;
      *launches += 2;
    }
    rank_scores_kernel<<<static_cast<unsigned>(static_cast<int64_t>(P) * nblk), kBlock, 0, stream>>>(
        scores, round0, round_end - round0, round0 == 0, C, nblk, seg_off, seg_idx, k, partial);
    ++*launches;
  } while (first < pairs);
  return cudaGetLastError();
}

size_t score_wide_scratch_bytes(const MlpModel& m, int64_t rows, bool lean) {
  const int64_t batch = std::min(rows, batch_rows(lean));
  return up(image_bytes(*m.wide, batch)) + static_cast<size_t>(act_rows(*m.wide, batch)) * 128 + 1024;
}

cudaError_t launch_score_wide(const MlpModel& m, const float* d_feat, int64_t rows, float* d_scores, void* scratch,
                              int* status, cudaStream_t stream, int64_t* launches, const FastWait* wait) {
  const WideMlp& w = *m.wide;
  const int64_t batch = batch_rows(wait->lean);
  uint8_t* image = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(scratch) + 1023) / 1024 * 1024);
  uint8_t* act = image + up(image_bytes(w, std::min(rows, batch)));
  for (int64_t first = 0; first < rows; first += batch) {
    const int64_t n = std::min(rows - first, batch), padded = (n + kRowsPair - 1) / kRowsPair * kRowsPair;
    const unsigned grid = static_cast<unsigned>((padded + 127) / 128);
    const float* x = d_feat + first * KS_F_PAD;
    if (w.input.onehot) wide_given_rows_kernel<true><<<grid, 128, 0, stream>>>(x, n, padded, w.input, image, wait->words + kWordWide);
    else wide_given_rows_kernel<false><<<grid, 128, 0, stream>>>(x, n, padded, w.input, image, wait->words + kWordWide);
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) e = launch_layers(w, image, act, n, d_scores + first, status, wait, stream);
    if (e != cudaSuccess) return e;
    *launches += 2;
  }
  return cudaSuccess;
}

}  // namespace ks
