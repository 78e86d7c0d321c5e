// A user's kernels on the device API whose value functions return something
// the element type is only explicitly convertible from, and count their calls.
// They include only the public header.
#include <cuda_runtime.h>
#include <stdint.h>

#include "gga_device.cuh"

namespace {

struct Id {
  uint32_t v;
  Id() = default;
  __device__ explicit Id(uint32_t x) : v(x) {}
};

enum class Tag : unsigned long long {};

// Thread t of block l pushes 3 elements l * 1000 + 10 t + k per round, by a
// staged cursor, an unstaged one and a rounds cursor of 2.
template <class T>
__global__ void __launch_bounds__(128) push_typed(const gga_dev_view* v, uint32_t R) {
  __shared__ gga::PushShared sh, sh2;
  __shared__ gga::RoundsShared<2> rs;
  __shared__ uint4 stage[512];
  const uint32_t base = blockIdx.x * 1000u + threadIdx.x * 10u;
  const auto value = [=](uint32_t k) { return base + k; };
  const auto value_r = [=](uint32_t, uint32_t k) { return base + k; };
  {
    gga::BlockPusher<T> p(v, blockIdx.x, sh, stage, sizeof(stage));
    for (uint32_t r = 0; r < R; ++r) p.push(3u, value);
    p.flush();
  }
  {
    gga::BlockPusher<T> p(v, blockIdx.x, sh2);
    for (uint32_t r = 0; r < R; ++r) p.push(3u, value);
  }
  __syncthreads();
  gga::RoundsPusher<T, 2> p(v, blockIdx.x, rs, stage, sizeof(stage));
  const uint32_t c[2] = {3u, 3u};
  p.push(c, value_r);
  p.template push<3>(c, value_r);
  gga::block_push_rounds<T, 2>(v, blockIdx.x, c, value_r);
  gga::block_push_back<T>(v, blockIdx.x, 3u, value);
}

// Every thread pushes 5 elements in each of 3 rounds per call, up to `limit`;
// `calls` counts the calls of the value function.
__global__ void __launch_bounds__(128) push_counted(const gga_dev_view* v, uint64_t limit, int staged, unsigned long long* calls,
                                                    uint32_t* kept) {
  __shared__ gga::RoundsShared<3> rs;
  __shared__ uint4 stage[2048];
  gga::RoundsPusher<uint32_t, 3> p(v, blockIdx.x, rs, staged ? stage : nullptr, staged ? sizeof(stage) : 0, limit);
  const uint32_t c[3] = {5u, 5u, 5u};
  uint32_t n = 0;
  for (int i = 0; i < 3; ++i) {
    uint32_t k = 0;
    p.push(c, [&](uint32_t kr, uint32_t m) {
      atomicAdd(calls, 1ull);
      return kr * 100u + m;
    }, &k);
    n += k;
  }
  if (threadIdx.x == 0) kept[blockIdx.x] = n;
}

int launched() { return cudaGetLastError() == cudaSuccess ? 0 : 5; }

}  // namespace

extern "C" {

int user_push_typed(const void* view, uint32_t L, uint32_t T, uint32_t R, uint32_t E, void* stream) {
  const gga_dev_view* v = static_cast<const gga_dev_view*>(view);
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  if (E == 4) push_typed<Id><<<L, T, 0, st>>>(v, R);
  else push_typed<Tag><<<L, T, 0, st>>>(v, R);
  return launched();
}

int user_push_counted(const void* view, uint32_t L, uint32_t T, uint64_t limit, int staged, unsigned long long* calls,
                      uint32_t* kept, void* stream) {
  push_counted<<<L, T, 0, static_cast<cudaStream_t>(stream)>>>(static_cast<const gga_dev_view*>(view), limit, staged,
                                                               calls, kept);
  return launched();
}

}  // extern "C"
