// gga_batch.cu -- many GGArrays grown in one persistent launch.
//
// A batch is a list of jobs: an array, the draws of its counts and values
// (as gga_insert_generated), and a target size.  gga_batch_grow runs one
// persistent kernel per form (payload size and count distribution) over its
// (array, LFVector) items, longest first, taken from atomic tickets
// (gga_batch_grow.cuh): a block -- a cluster of blocks for the longest --
// grows its LFVector in passes of several rounds: every thread draws its
// counts, a block scan gives positions, counts are clipped at the LFVector's
// target by the same scan, the leader reserves and allocates, the block
// stages the pass and writes it with 128-bit stores (Algorithm 1 with thread
// coarsening).  The forms run side by side, a form's blocks taking the SMs as
// an earlier one's finish.  Then one kernel folds the pool pops and finalizes
// every array.  Nothing allocates and nothing waits on the host, so the whole
// step can be captured in a CUDA graph and replayed (gga_batch_capture /
// gga_batch_replay).
#include <algorithm>
#include <new>
#include <vector>

#include "gga_batch_grow.cuh"

namespace gga {
namespace {

// The prefix sums of every job's array, one block each.  After a growth
// (pools given) the blocks also fold the grow kernel's pops into the pools'
// queue heads -- a batch has no more pools than jobs -- and reset the tickets
// for the next run.
__global__ void __launch_bounds__(256) batch_finalize_kernel(const BatchJob* __restrict__ jobs,
                                                             PoolState* const* pools, uint32_t n_pools,
                                                             uint32_t* tickets) {
  __shared__ FinalizeShared sh;
  if (pools) {
    if (blockIdx.x < n_pools) ring_fixup_class(pools[blockIdx.x], threadIdx.x);
    if (blockIdx.x == 0 && threadIdx.x < kBatchLaunches) tickets[threadIdx.x] = 0;
  }
  finalize_block(jobs[blockIdx.x].v, nullptr, nullptr, nullptr, 1, sh);
}

// Every bucket of every item back to its pool's queue; sizes to zero.
__global__ void batch_clear_kernel(const BatchJob* __restrict__ jobs, const BatchItem* __restrict__ items) {
  const BatchItem item = items[blockIdx.x];
  const ArrayView& v = jobs[item.job].v;
  const uint64_t l = item.l;
  for (uint32_t b = threadIdx.x; b < static_cast<uint32_t>(kMaxBuckets); b += blockDim.x) {
    uint64_t* slot = v.buckets + l * kMaxBuckets + b;
    const uint64_t a = *slot;
    if (a) {
      if (!ring_push(v.pool, class_of(bucket_len(b, v.log2B) * v.E), a)) latch_error(v.status, GGA_ERR_INVALID);
      *slot = 0;
    }
  }
  if (threadIdx.x == 0) {
    v.sizes[l] = 0;
    v.nbuckets[l] = 0;
  }
}

}  // namespace
}  // namespace gga

struct gga_batch_t {
  gga::BatchJob* jobs;
  gga::BatchItem* items;      // form by form
  gga::PoolState** pools;
  uint32_t* tickets;          // one per launch
  uint32_t n_jobs, n_items, n_pools;
  uint32_t n_launches;
  gga::BatchLaunch launch[gga::kBatchLaunches];
  // Streams of the second and later launches, forked from and joined to the
  // caller's stream by events.
  cudaStream_t side[gga::kBatchLaunches];
  cudaEvent_t fork, join[gga::kBatchLaunches];
  cudaGraphExec_t graph;
  bool has_graph;
};

namespace {

// Rounds that draw an LFVector of `target` elements.
double expected_rounds(const gga::BatchJob& J, uint64_t target) {
  const double per_round = static_cast<double>(J.g.mean) * J.v.T;
  return per_round > 0 ? std::min(static_cast<double>(target) / per_round + 1, 1e12) : 1e12;
}

// Its cost in microseconds of a whole GB300 per 2^24 draws and elements, from
// generated insertions of means 0.5 and 1 at T = 1024 (idle threads draw too).
// The forms' shares of the chip follow it: by passes, which hold two to eight
// rounds, 300 arrays of the three payloads took 492 us (T = 1024, uniform
// counts, 131K elements per LFVector), by cost 262.
double expected_cost(const gga::BatchJob& J, uint64_t target, double rounds) {
  const uint32_t kv = (J.v.T + gga::kBatchThreads - 1) / gga::kBatchThreads;
  const double draw = J.g.dist > GGA_DIST_UNIFORM3 ? 70 : 40;
  const double elem = J.v.E == 4 ? 15 : (J.v.E == 8 ? 22 : 35);
  return rounds * gga::kBatchThreads * kv * draw + static_cast<double>(target) * elem;
}

void launch_form(const gga::BatchLaunch& a, cudaStream_t st) {
  switch (a.form >> 2) {
    case 0: gga::launch_batch_form<4>(a, st); break;
    case 1: gga::launch_batch_form<8>(a, st); break;
    default: gga::launch_batch_form<16>(a, st); break;
  }
}

int blocks_per_sm(uint32_t form, bool clusters) {
  return form >> 2 == 0 ? gga::batch_blocks_per_sm<4>(form, clusters)
                        : (form >> 2 == 1 ? gga::batch_blocks_per_sm<8>(form, clusters)
                                          : gga::batch_blocks_per_sm<16>(form, clusters));
}

int batch_grow(gga_batch_t* b, cudaStream_t st) {
  bool ok = true;
  uint32_t started = 0;
  if (b->n_launches > 1) ok = cudaEventRecord(b->fork, st) == cudaSuccess;
  for (uint32_t i = 0; i < b->n_launches && ok; ++i) {
    cudaStream_t s = i == 0 ? st : b->side[i];
    if (i) ok = cudaStreamWaitEvent(s, b->fork, 0) == cudaSuccess;
    if (!ok) break;   // the launch would not wait for what comes before
    launch_form(b->launch[i], s);
    started = i + 1;
    if (i) ok = cudaEventRecord(b->join[i], s) == cudaSuccess;
  }
  for (uint32_t i = 1; i < started && ok; ++i) ok = cudaStreamWaitEvent(st, b->join[i], 0) == cudaSuccess;
  if (!ok) {
    // Growth kernels may be running that `st` does not wait for: what follows a
    // growth is launched when they are done (a stream that is captured runs
    // none, and its capture fails).
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(st, &cap) != cudaSuccess || cap != cudaStreamCaptureStatusNone) return GGA_ERR_CUDA;
    for (uint32_t i = 1; i < started; ++i)
      if (cudaStreamSynchronize(b->side[i]) != cudaSuccess) return GGA_ERR_CUDA;
  }
  if (b->n_jobs)
    gga::batch_finalize_kernel<<<b->n_jobs, 256, 0, st>>>(b->jobs, b->pools, b->n_pools, b->tickets);
  return cudaGetLastError() == cudaSuccess && ok ? GGA_OK : GGA_ERR_CUDA;
}

int batch_clear(gga_batch_t* b, cudaStream_t st) {
  if (b->n_items) gga::batch_clear_kernel<<<b->n_items, 64, 0, st>>>(b->jobs, b->items);
  if (b->n_jobs) gga::batch_finalize_kernel<<<b->n_jobs, 256, 0, st>>>(b->jobs, nullptr, 0, nullptr);
  return cudaGetLastError() == cudaSuccess ? GGA_OK : GGA_ERR_CUDA;
}

}  // namespace

extern "C" {

int gga_batch_create(const gga_batch_job* jobs, uint32_t n_jobs, void* stream, gga_batch* out) {
  if (!out || (n_jobs && !jobs)) return GGA_ERR_INVALID;
  *out = nullptr;
  struct Item {
    uint32_t form;
    double rounds, cost;
    gga::BatchItem it;
  };
  std::vector<gga::BatchJob> hj(n_jobs);
  std::vector<Item> hi;
  std::vector<gga::PoolState*> hp;
  int num_sms = 0;
  for (uint32_t j = 0; j < n_jobs; ++j) {
    gga::InsertScratch ins;
    int dev = 0;
    if (!gga::handle_parts(jobs[j].array, &hj[j].v, &ins, &dev, &num_sms)) return GGA_ERR_INVALID;
    const gga_gen_spec& sp = jobs[j].spec;
    if (sp.dist > GGA_DIST_POISSON || sp.n_thresholds > GGA_MAX_THRESHOLDS ||
        (sp.dist == GGA_DIST_POISSON && sp.n_thresholds == 0))
      return GGA_ERR_INVALID;
    hj[j].g = gga::make_gen_params(sp);
    hj[j].target = jobs[j].target;
    const uint32_t L = hj[j].v.L, E = hj[j].v.E;
    const uint32_t form = (E == 4 ? 0u : (E == 8 ? 4u : 8u)) + sp.dist;
    for (uint32_t l = 0; l < L; ++l) {
      const uint64_t tl = jobs[j].target / L + (l < jobs[j].target % L ? 1 : 0);
      if (!tl) continue;
      const double rounds = expected_rounds(hj[j], tl);
      hi.push_back({form, rounds, expected_cost(hj[j], tl, rounds), gga::BatchItem{j, l}});
    }
    if (std::find(hp.begin(), hp.end(), hj[j].v.pool) == hp.end()) hp.push_back(hj[j].v.pool);
  }
  // Form by form, longest chains first: the tickets then balance
  // the tail.
  std::stable_sort(hi.begin(), hi.end(), [](const Item& a, const Item& b) {
    return a.form != b.form ? a.form < b.form : a.rounds > b.rounds;
  });
  std::vector<gga::BatchItem> items(hi.size());
  double sum = 0;
  for (size_t i = 0; i < hi.size(); ++i) {
    items[i] = hi[i].it;
    sum += hi[i].cost;
  }

  gga_batch_t* b = new (std::nothrow) gga_batch_t();   // zeroed
  if (!b) return GGA_ERR_CUDA;
  b->n_jobs = n_jobs;
  b->n_items = static_cast<uint32_t>(items.size());
  b->n_pools = static_cast<uint32_t>(hp.size());
  // A form's items grown by clusters (`big`, the first ones): those whose
  // chain is long enough for the cluster's larger passes -- four of them, or
  // one while the items leave three quarters of the blocks idle -- and that
  // cost more than a quarter of a block's average load over the whole batch.
  // (The rest then ends within a quarter of that load.)  Measured on GB300, four
  // / one: 30 arrays of 32 to 131K elements per LFVector at T = 1024, uniform
  // counts, 117 / 63 us; 300 arrays at T = 256 462 / 629.
  struct Form {
    uint32_t id, first, n, big;
    double cost, big_cost;
  };
  std::vector<Form> forms;
  double big_sum = 0;
  const uint64_t blocks = static_cast<uint64_t>(std::max(num_sms, 1)) * gga::kBatchMinBlocks;
  const double least = (hi.size() * 4 <= blocks ? 1 : 4) * gga::kBatchCluster * gga::kBatchRounds;
  for (uint32_t i = 0; i < b->n_items; ++i) {
    if (forms.empty() || forms.back().id != hi[i].form) forms.push_back({hi[i].form, i, 0, 0, 0, 0});
    Form& f = forms.back();
    if (f.big == f.n && hi[i].rounds >= least && hi[i].cost * 4 > sum / static_cast<double>(blocks)) {
      ++f.big;
      f.big_cost += hi[i].cost;
      big_sum += hi[i].cost;
    }
    ++f.n;
    f.cost += hi[i].cost;
  }
  // The form with most work first.
  std::stable_sort(forms.begin(), forms.end(), [](const Form& x, const Form& y) { return x.cost > y.cost; });
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  int rc = GGA_OK;
  if (cudaMalloc(&b->jobs, sizeof(gga::BatchJob) * (n_jobs ? n_jobs : 1)) != cudaSuccess ||
      cudaMalloc(&b->items, sizeof(gga::BatchItem) * (items.empty() ? 1 : items.size())) != cudaSuccess ||
      cudaMalloc(&b->pools, sizeof(gga::PoolState*) * (hp.empty() ? 1 : hp.size())) != cudaSuccess ||
      cudaMalloc(&b->tickets, gga::kBatchLaunches * sizeof(uint32_t)) != cudaSuccess)
    rc = GGA_ERR_CUDA;
  if (rc == GGA_OK &&
      ((n_jobs && cudaMemcpyAsync(b->jobs, hj.data(), sizeof(gga::BatchJob) * n_jobs, cudaMemcpyHostToDevice, st) !=
                      cudaSuccess) ||
       (!items.empty() && cudaMemcpyAsync(b->items, items.data(), sizeof(gga::BatchItem) * items.size(),
                                          cudaMemcpyHostToDevice, st) != cudaSuccess) ||
       (!hp.empty() && cudaMemcpyAsync(b->pools, hp.data(), sizeof(gga::PoolState*) * hp.size(),
                                       cudaMemcpyHostToDevice, st) != cudaSuccess) ||
       cudaMemsetAsync(b->tickets, 0, gga::kBatchLaunches * sizeof(uint32_t), st) != cudaSuccess ||
       cudaStreamSynchronize(st) != cudaSuccess))
    rc = GGA_ERR_CUDA;
  // The cluster kernels first, then the block kernels.
  for (int clusters = 1; clusters >= 0; --clusters) {
    for (size_t k = 0; k < forms.size() && rc == GGA_OK; ++k) {
      const Form& f = forms[k];
      const uint32_t n = clusters ? f.big : f.n - f.big, unit = clusters ? gga::kBatchCluster : 1;
      if (n == 0) continue;
      // As many units as are resident at once -- for the cluster kernels the
      // form's share of them by its cost, so that every form's longest
      // chains start at once -- or as there are items.
      uint64_t fit = static_cast<uint64_t>(num_sms) * blocks_per_sm(f.id, clusters != 0) / unit;
      if (clusters) fit = static_cast<uint64_t>(static_cast<double>(fit) * (f.big_cost / big_sum) + 0.5);
      const uint32_t i = b->n_launches++;
      b->launch[i] = gga::BatchLaunch{f.id, clusters != 0, b->jobs, b->items + f.first + (clusters ? 0 : f.big),
                                      n, b->tickets + i, static_cast<uint32_t>(std::max<uint64_t>(1, std::min<uint64_t>(fit, n))) * unit};
      if (i && (cudaStreamCreateWithFlags(&b->side[i], cudaStreamNonBlocking) != cudaSuccess ||
                cudaEventCreateWithFlags(&b->join[i], cudaEventDisableTiming) != cudaSuccess))
        rc = GGA_ERR_CUDA;
    }
  }
  if (rc == GGA_OK && b->n_launches > 1 && cudaEventCreateWithFlags(&b->fork, cudaEventDisableTiming) != cudaSuccess)
    rc = GGA_ERR_CUDA;
  if (rc != GGA_OK) {
    gga_batch_destroy(b);
    return rc;
  }
  *out = b;
  return GGA_OK;
}

int gga_batch_grow(gga_batch b, void* stream) {
  if (!b) return GGA_ERR_INVALID;
  return batch_grow(b, static_cast<cudaStream_t>(stream));
}

int gga_batch_clear(gga_batch b, void* stream) {
  if (!b) return GGA_ERR_INVALID;
  return batch_clear(b, static_cast<cudaStream_t>(stream));
}

int gga_batch_capture(gga_batch b, void* stream) {
  if (!b || !stream) return GGA_ERR_INVALID;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  if (b->has_graph) {
    cudaGraphExecDestroy(b->graph);
    b->has_graph = false;
  }
  cudaGraph_t g;
  if (cudaStreamBeginCapture(st, cudaStreamCaptureModeThreadLocal) != cudaSuccess) return GGA_ERR_CUDA;
  int rc = batch_clear(b, st);
  if (rc == GGA_OK) rc = batch_grow(b, st);
  if (cudaStreamEndCapture(st, &g) != cudaSuccess) return GGA_ERR_CUDA;
  if (rc != GGA_OK) {
    cudaGraphDestroy(g);
    return rc;
  }
  const cudaError_t e = cudaGraphInstantiate(&b->graph, g, 0);
  cudaGraphDestroy(g);
  if (e != cudaSuccess) return GGA_ERR_CUDA;
  b->has_graph = true;
  return GGA_OK;
}

int gga_batch_replay(gga_batch b, void* stream) {
  if (!b || !b->has_graph) return GGA_ERR_INVALID;
  return cudaGraphLaunch(b->graph, static_cast<cudaStream_t>(stream)) == cudaSuccess ? GGA_OK : GGA_ERR_CUDA;
}

int gga_batch_destroy(gga_batch b) {
  if (!b) return GGA_ERR_INVALID;
  int rc = GGA_OK;
  if (cudaDeviceSynchronize() != cudaSuccess) rc = GGA_ERR_CUDA;
  if (b->has_graph) cudaGraphExecDestroy(b->graph);
  for (int i = 0; i < gga::kBatchLaunches; ++i) {
    if (b->side[i]) cudaStreamDestroy(b->side[i]);
    if (b->join[i]) cudaEventDestroy(b->join[i]);
  }
  if (b->fork) cudaEventDestroy(b->fork);
  if (b->jobs) cudaFree(b->jobs);
  if (b->items) cudaFree(b->items);
  if (b->pools) cudaFree(b->pools);
  if (b->tickets) cudaFree(b->tickets);
  delete b;
  return rc;
}

}  // extern "C"
