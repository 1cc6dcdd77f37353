// Copies between a caller's dense device arrays and the padded planes of a
// lattice, and the reset of a whole set, each one launch.
#include <algorithm>

#include "lbm_internal.h"

namespace lbm {
namespace {

// A warp copies pieces of 32 x kUnroll words of V, one row's pieces after
// the other; V is the widest word that both sides' addresses and strides
// allow.  Bound by memory: 1.2 GB of populations each way (8192 x 4096 FP32)
// in 365 us (6.6 TB/s), where the strided device-to-device copy of the
// runtime takes 1,230; BF16 rows of 7001 cells (two-byte words), 0.44 GB each
// way, 200 against 530.  A small lattice costs its launch: nine planes of 128 x
// 64 cells 13 us with the call, 44 as nine copies.
constexpr int kUnroll = 4;

template <class V>
__global__ void __launch_bounds__(256) k_copy_planes(const PlaneCopy c, int chunks, int tasks) {
  const int lane = threadIdx.x & 31, warps = gridDim.x * 8;
  const int width = (int)(c.width / sizeof(V));
  for (int t = blockIdx.x * 8 + (threadIdx.x >> 5); t < tasks; t += warps) {
    const int row = t / chunks, x0 = (t - row * chunks) * (32 * kUnroll) + lane;
    const int plane = row / c.rows, y = row - plane * c.rows;
    const V* src = reinterpret_cast<const V*>(static_cast<const char*>(c.src) + plane * c.src_plane + y * c.src_pitch);
    V* dst = reinterpret_cast<V*>(static_cast<char*>(c.dst) + plane * c.dst_plane + y * c.dst_pitch);
    V v[kUnroll];
#pragma unroll
    for (int u = 0; u < kUnroll; ++u)
      if (x0 + 32 * u < width) v[u] = src[x0 + 32 * u];
#pragma unroll
    for (int u = 0; u < kUnroll; ++u)
      if (x0 + 32 * u < width) dst[x0 + 32 * u] = v[u];
  }
}

template <class V>
cudaError_t copy_as(const PlaneCopy& c, cudaStream_t stream) {
  const long long chunks = ((long long)(c.width / sizeof(V)) + 32 * kUnroll - 1) / (32 * kUnroll);
  const long long tasks = chunks * c.rows * c.planes;
  if (tasks >= 1ll << 30) return cudaErrorInvalidValue;
  const long long blocks = (tasks + 7) / 8;
  k_copy_planes<V><<<(int)(blocks < 152 * 16 ? blocks : 152 * 16), 256, 0, stream>>>(c, (int)chunks, (int)tasks);
  count_launches(1);
  return cudaGetLastError();
}

// Entry blockIdx.y of the list: copied, or zeroed where it has no source.
__global__ void __launch_bounds__(256) k_fill_list(const FillEntry* __restrict__ list) {
  const FillEntry e = list[blockIdx.y];
  const bool wide = ((uintptr_t)e.dst | (uintptr_t)e.src) % 16 == 0;
  const size_t words = wide ? e.bytes / 16 : 0;
  const size_t first = (size_t)blockIdx.x * blockDim.x + threadIdx.x, stride = (size_t)gridDim.x * blockDim.x;
  for (size_t i = first; i < words; i += stride)
    static_cast<uint4*>(e.dst)[i] = e.src ? static_cast<const uint4*>(e.src)[i] : make_uint4(0, 0, 0, 0);
  for (size_t i = words * 16 + first; i < e.bytes; i += stride)
    static_cast<uint8_t*>(e.dst)[i] = e.src ? static_cast<const uint8_t*>(e.src)[i] : (uint8_t)0;
}

}  // namespace

cudaError_t launch_copy_planes(const PlaneCopy& c, cudaStream_t stream) {
  if (c.planes < 1 || c.rows < 1 || c.width < 1) return cudaSuccess;
  const size_t all = (uintptr_t)c.src | (uintptr_t)c.dst | c.src_pitch | c.dst_pitch | c.src_plane | c.dst_plane |
                     c.width;
  if (all % 16 == 0) return copy_as<uint4>(c, stream);
  if (all % 8 == 0) return copy_as<uint2>(c, stream);
  if (all % 4 == 0) return copy_as<uint32_t>(c, stream);
  if (all % 2 == 0) return copy_as<uint16_t>(c, stream);
  return copy_as<uint8_t>(c, stream);
}

// Blocks an entry: 8 fill the device from some 300 entries on (the 256
// candidates have 768); fewer entries share 16 blocks per SM, and an entry of
// many MB gets a block per MB of its own, whatever stands beside it.  Reset of
// two members of 8192 x 4096 cells 2.20 ms (1.11 each alone; 3.98 with 8 blocks
// an entry), of one of 4096 x 2048 beside the 256 candidates 0.92 (1.43), of
// the 256 alone 0.68 (0.71).
cudaError_t launch_fill_list(const FillEntry* list, int n, size_t largest, int sm_count, cudaStream_t stream) {
  const size_t most = (size_t)16 * sm_count;
  const size_t blocks = std::min(most, std::max({(size_t)8, (most + n - 1) / n, largest >> 20}));
  k_fill_list<<<dim3((unsigned)blocks, n), 256, 0, stream>>>(list);
  count_launches(1);
  return cudaGetLastError();
}

}  // namespace lbm
