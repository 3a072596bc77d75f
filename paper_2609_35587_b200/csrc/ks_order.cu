// Similarity order of a candidate catalogue.
//
// The quantised tree kernel keeps the four candidates of a tile word in one thread and can share
// one walk among them for as long as they take the same turns. They do so the more often the
// more alike they are, so the catalogue is ranked in an order in which neighbours differ in as
// few knobs as possible: sorted by (T_M, T_N, T_K, stages, c_M, c_N, kernel schedule, epilogue
// schedule, tile scheduler, instruction shape), most significant first. In a cross-product
// catalogue the four candidates of a word then differ only in the tile scheduler and the
// instruction shape. The order changes nothing in the results: ranking keys carry the pool index.
//
// The sort of a large catalogue is a library primitive (cub::DeviceRadixSort) outside the hot loop:
// about 0.1 % of a batch step, and done once for a prepared catalogue. A small one is ordered by counting.
#include <cub/device/device_radix_sort.cuh>

#include "ks_features.cuh"
#include "ks_internal.h"

namespace ks {

namespace {

__device__ __forceinline__ unsigned long long order_key(const ks_candidate& k) {
  unsigned long long key = k.tile_m & 0xFFFu;
  key = (key << 12) | (k.tile_n & 0xFFFu);
  key = (key << 12) | (k.tile_k & 0xFFFu);
  key = (key << 4) | (k.stages & 0xFu);
  key = (key << 5) | (k.cluster_m & 0x1Fu);
  key = (key << 5) | (k.cluster_n & 0x1Fu);
  key = (key << 2) | (k.kernel_sched & 3u);
  key = (key << 2) | (k.epi_sched & 3u);
  key = (key << 1) | (k.tile_sched & 1u);
  key = (key << 1) | (k.instr_n != k.tile_n ? 1u : 0u);
  return key;
}

__global__ void order_keys_kernel(const ks_candidate* __restrict__ c, int C, unsigned long long* __restrict__ keys,
                                  int* __restrict__ idx) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= C) return;
  keys[i] = order_key(load_candidate(c + i));
  idx[i] = i;
}

// Up to kCountMax candidates: a candidate's place is the number of keys before its own (of equal ones the
// earlier comes first, as in the stable sort). A block places 32 candidates, each of its warps against an
// eighth of the keys. The radix sort takes a pass of one block for every eight bits of the key here, seven
// times 9 us: 4,883 candidates 72 us with its keys, 27 like this.
constexpr int kCountMax = 8192;
__global__ void __launch_bounds__(256)
order_count_kernel(const ks_candidate* __restrict__ c, int C, int* __restrict__ order) {
  extern __shared__ __align__(16) unsigned long long s_key[];  // C rounded up to 16
  __shared__ int s_place[32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, padded = (C + 15) / 16 * 16;
  for (int i = threadIdx.x; i < padded; i += 256) s_key[i] = i < C ? order_key(load_candidate(c + i)) : ~0ull;
  if (threadIdx.x < 32) s_place[threadIdx.x] = 0;
  __syncthreads();
  const int me = blockIdx.x * 32 + lane;
  if (me < C) {
    const unsigned long long key = s_key[me];
    const int share = padded / 8, begin = warp * share;  // (a multiple of two)
    int place = 0;
#pragma unroll 4
    for (int j = begin; j < begin + share; j += 2) {
      const ulonglong2 other = *reinterpret_cast<const ulonglong2*>(s_key + j);
      place += (other.x < key + (j < me)) + (other.y < key + (j + 1 < me));
    }
    atomicAdd(&s_place[lane], place);
  }
  __syncthreads();
  if (warp == 0 && me < C) order[s_place[lane]] = me;
}

constexpr int kKeyBits = 56;

size_t align256(size_t v) { return (v + 255) / 256 * 256; }

size_t cub_temp_bytes(int C) {
  size_t bytes = 0;
  cub::DeviceRadixSort::SortPairs(nullptr, bytes, static_cast<const unsigned long long*>(nullptr),
                                  static_cast<unsigned long long*>(nullptr), static_cast<const int*>(nullptr),
                                  static_cast<int*>(nullptr), C, 0, kKeyBits);
  return bytes;
}

}  // namespace

// scratch layout: order (the result, first) | keys in | keys out | indices in | sort workspace
size_t order_scratch_bytes(int C) {
  if (C < 1) return 0;
  return align256(sizeof(int) * C) + 2 * align256(sizeof(unsigned long long) * C) + align256(sizeof(int) * C) +
         align256(cub_temp_bytes(C));
}

// Writes the catalogue positions in similarity order to the front of `scratch` (C int32).
cudaError_t launch_catalogue_order(const ks_candidate* d_c, int C, void* scratch, cudaStream_t stream,
                                   int64_t* launches) {
  char* base = static_cast<char*>(scratch);
  int* order = reinterpret_cast<int*>(base);
  if (C <= kCountMax) {
    const size_t smem = sizeof(unsigned long long) * ((C + 15) / 16 * 16);
    cudaError_t e = ensure_dynamic_smem(reinterpret_cast<const void*>(&order_count_kernel), smem);
    if (e != cudaSuccess) return e;
    order_count_kernel<<<(C + 31) / 32, 256, smem, stream>>>(d_c, C, order);
    *launches += 1;
    return cudaGetLastError();
  }
  base += align256(sizeof(int) * C);
  unsigned long long* keys_in = reinterpret_cast<unsigned long long*>(base);
  base += align256(sizeof(unsigned long long) * C);
  unsigned long long* keys_out = reinterpret_cast<unsigned long long*>(base);
  base += align256(sizeof(unsigned long long) * C);
  int* idx_in = reinterpret_cast<int*>(base);
  base += align256(sizeof(int) * C);
  size_t temp = cub_temp_bytes(C);
  order_keys_kernel<<<(C + 255) / 256, 256, 0, stream>>>(d_c, C, keys_in, idx_in);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  e = cub::DeviceRadixSort::SortPairs(base, temp, keys_in, keys_out, idx_in, order, C, 0, kKeyBits, stream);
  *launches += 1;  // the key kernel (the sort launches the library's own kernels)
  return e;
}

}  // namespace ks
