// gga_batch_grow.cuh -- the growth kernel of a batch, one instance per
// payload size and count distribution (a "form").  Each form is a kernel of
// its own, run beside the others: with all twelve inlined into one kernel it
// spilled 2.2 KB of registers and took three and a half minutes to compile,
// at the same speed.
#pragma once

#include "gga_gen.cuh"

namespace gga {

// Threads per block, virtual threads per thread (T <= kBatchThreads *
// kBatchKV = 1024; a block draws for ceil(T / kBatchThreads) of them) and
// resident blocks per SM.  Drawing for all four whatever T was, arrays of T = 256
// took 1300 us where it now takes 550 (300 arrays of lognormal sizes).
constexpr int kBatchThreads = 256;
constexpr int kBatchKV = 4;
constexpr int kBatchMinBlocks = 4;
constexpr uint32_t kBatchStageBytes = 40960;
constexpr uint32_t kBatchMaxRounds = 1u << 20;
constexpr int kBatchLaunches = 24;   // a cluster and a block kernel per (payload size, distribution)
// Blocks of a cluster.  An LFVector's rounds follow one another, so one block
// grows a large one in one long chain of passes: for 1024 arrays of lognormal
// sizes (2.1e8 elements) the longest chains, 256 passes, took 1.9 ms while the
// blocks' average load is a third of that.  The largest items (chosen in
// gga_batch_create) are therefore grown by whole clusters, one pass
// of kBatchCluster times the rounds at a time; the others by single blocks,
// which take the SMs as the clusters finish.  Measured on GB300 for that
// batch, growth with its reads and flattens: 2.19 ms by single blocks, 1.36
// with clusters of 4 (1.25 now), 1.37 of 8 (a larger part of the last pass is
// clipped), 1.96 of 2; blocks of 512 threads with two virtual threads per thread
// and clusters of 4: 1.54.  (Of the 1.25 ms 0.2 are the reads and flattens.)
constexpr int kBatchCluster = 4;

struct BatchJob {
  ArrayView v;
  GenParams g;
  uint64_t target;
};

struct BatchItem {
  uint32_t job;
  uint32_t l;
};

// Rounds per pass.  Bernoulli and uniform counts stage their elements,
// batch_staged rounds at a time (at T = 1024 threads and one element per thread
// and round 32 KB of the 40 KB stage), the others 4-byte marks.
constexpr int kBatchRounds = 8;
constexpr int batch_staged(int E, uint32_t dist) { return dist > GGA_DIST_UNIFORM3 ? kBatchRounds : 32 / E; }

// Grow LFVector l of job J to its share of the target: rounds of in-thread
// insertions in passes of K (grow_passes in gga_gen.cuh), clipped at the
// target, by this block (C = 1) or by its cluster.  All threads call it.
template <int E, int DIST, int C>
__device__ __forceinline__ void grow_item(const BatchJob* __restrict__ jobs, const BatchItem* __restrict__ items,
                                          uint32_t it, BatchJob& s_job, GenShared& sh, uint4* stage) {
  const BatchItem item = items[it];
  if (threadIdx.x < sizeof(BatchJob) / 8)
    reinterpret_cast<unsigned long long*>(&s_job)[threadIdx.x] =
        reinterpret_cast<const unsigned long long*>(jobs + item.job)[threadIdx.x];
  __syncthreads();
  const ArrayView& v = s_job.v;
  const uint64_t target = s_job.target / v.L + (item.l < s_job.target % v.L ? 1 : 0);
  bool done;
  const uint32_t drawn = grow_passes<E, kBatchRounds, kBatchKV, DIST, C, batch_staged(E, DIST), true>(
      v, s_job.g, item.l, kBatchMaxRounds, target, sh, stage, kBatchStageBytes / E, &done);
  if (threadIdx.x == 0 && !done && drawn >= kBatchMaxRounds) latch_error(v.status, GGA_ERR_TIMEOUT);
  __syncthreads();
}

// Items taken from *ticket, longest chains first: by blocks, or (the cluster
// kernel) by the blocks of a cluster together.
template <int E, int DIST>
__global__ void __launch_bounds__(kBatchThreads, kBatchMinBlocks)
    batch_grow_kernel(const BatchJob* __restrict__ jobs, const BatchItem* __restrict__ items, uint32_t n_items,
                      uint32_t* ticket) {
  extern __shared__ uint4 s_stage4[];
  __shared__ GenShared sh;
  __shared__ uint32_t s_item;
  // The item's job (its view and draws) in shared memory: the pass loop
  // reads these fields over and over, and from here they are shared-memory
  // loads instead of global ones.
  __shared__ __align__(16) BatchJob s_job;
  static_assert(sizeof(BatchJob) % 8 == 0 && sizeof(BatchJob) / 8 <= kBatchThreads, "job copied in 8-byte words");
  while (true) {
    if (threadIdx.x == 0) s_item = atomicAdd(ticket, 1u);
    __syncthreads();
    const uint32_t it = s_item;
    if (it >= n_items) break;
    grow_item<E, DIST, 1>(jobs, items, it, s_job, sh, s_stage4);
  }
}

template <int E, int DIST>
__global__ void __cluster_dims__(kBatchCluster, 1, 1) __launch_bounds__(kBatchThreads, kBatchMinBlocks)
    batch_cluster_kernel(const BatchJob* __restrict__ jobs, const BatchItem* __restrict__ items, uint32_t n_items,
                         uint32_t* ticket) {
  extern __shared__ uint4 s_stage4[];
  __shared__ GenShared sh;
  __shared__ uint32_t s_item[2];
  __shared__ __align__(16) BatchJob s_job;
  cluster_barrier();   // every block of the cluster runs: its shared memory may be written
  // s_item alternates: block 0 stores the next ticket of the same slot two
  // items later, after a barrier the peers reach past their read of it.
  for (uint32_t par = 0;; par ^= 1u) {
    if (threadIdx.x == 0 && cluster_rank() == 0) {
      const uint32_t it = atomicAdd(ticket, 1u);
      for (uint32_t q = 0; q < kBatchCluster; ++q) cluster_store(&s_item[par], q, it);
    }
    cluster_barrier();
    const uint32_t it = s_item[par];
    if (it >= n_items) break;
    grow_item<E, DIST, kBatchCluster>(jobs, items, it, s_job, sh, s_stage4);
  }
}

struct BatchLaunch {
  uint32_t form;      // payload index * 4 + distribution
  bool clusters;
  const BatchJob* jobs;
  const BatchItem* items;
  uint32_t n_items;
  uint32_t* ticket;
  unsigned grid;
};

// Instantiated per payload size in gga_batch_e*.cu.
template <int E>
void launch_batch_form(const BatchLaunch& a, cudaStream_t st);
// Resident blocks per SM of a form's kernels (and their shared memory set).
template <int E>
int batch_blocks_per_sm(uint32_t form, bool clusters);

#ifdef GGA_BATCH_E
typedef void (*BatchKernel)(const BatchJob*, const BatchItem*, uint32_t, uint32_t*);

static BatchKernel batch_kernel_of(uint32_t form, bool clusters) {
  constexpr int E = GGA_BATCH_E;
  switch (form & 3u) {
    case GGA_DIST_BERNOULLI:
      return clusters ? batch_cluster_kernel<E, GGA_DIST_BERNOULLI> : batch_grow_kernel<E, GGA_DIST_BERNOULLI>;
    case GGA_DIST_UNIFORM3:
      return clusters ? batch_cluster_kernel<E, GGA_DIST_UNIFORM3> : batch_grow_kernel<E, GGA_DIST_UNIFORM3>;
    case GGA_DIST_GEOMETRIC:
      return clusters ? batch_cluster_kernel<E, GGA_DIST_GEOMETRIC> : batch_grow_kernel<E, GGA_DIST_GEOMETRIC>;
    default:
      return clusters ? batch_cluster_kernel<E, GGA_DIST_POISSON> : batch_grow_kernel<E, GGA_DIST_POISSON>;
  }
}

template <>
void launch_batch_form<GGA_BATCH_E>(const BatchLaunch& a, cudaStream_t st) {
  batch_kernel_of(a.form, a.clusters)<<<a.grid, kBatchThreads, kBatchStageBytes, st>>>(a.jobs, a.items, a.n_items,
                                                                                        a.ticket);
}

template <>
int batch_blocks_per_sm<GGA_BATCH_E>(uint32_t form, bool clusters) {
  BatchKernel kern = batch_kernel_of(form, clusters);
  cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(kBatchStageBytes));
  int per_sm = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kBatchThreads, kBatchStageBytes) != cudaSuccess ||
      per_sm < 1)
    per_sm = 1;
  return per_sm;
}
#endif

}  // namespace gga
