// gga_twophase.cu -- the two-phase case study (Sec. VI-D) on the GGArray.
//
// Insertion phase: an application kernel grows the array from inside the
// kernel.  Every parent record spawns Geometric(1/2) - 1 children that the
// kernel push_backs into the parent's own LFVector (Algorithm 1 called by the
// application, with thread coarsening).  Work phase: the array is flattened
// (gga_flatten) and a streaming kernel updates the contiguous copy.
//
// Records are 16 bytes {uint64 id, float pos, float vel}.  The count of the
// parent at local index j of LFVector l in generation `gen` is the number of
// trailing one bits of SplitMix64 draw ((gen << 48) | (offsets[l] + j)) + 1 of
// the stream seeded with `seed`; children follow parent order, a parent's
// children consecutively, and child k of a parent is the parent with
// id = ((gen + 1) << 56) | (l << 40) | (the child's LFVector-local index).
#include "gga_core.cuh"
#include "gga_gen.cuh"

namespace gga {

int launch_finalize(const ArrayView& v, cudaStream_t st);

namespace {

// The mixing function of SplitMix64 on a state z (states of consecutive keys
// are GOLDEN apart).
constexpr uint64_t kSpawnGolden = 0x9E3779B97F4A7C15ull;

__device__ __forceinline__ uint64_t spawn_mix(uint64_t z) {
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

// Geometric(1/2) - 1: trailing one bits of h, at most 63.
__device__ __forceinline__ uint32_t trailing_ones(uint64_t h) {
  const uint32_t lo = static_cast<uint32_t>(__clz(static_cast<int>(__brev(~static_cast<uint32_t>(h)))));
  if (lo < 32) return lo;
  return min(63u, 32u + static_cast<uint32_t>(__clz(static_cast<int>(__brev(~static_cast<uint32_t>(h >> 32))))));
}

__device__ __forceinline__ uint32_t warp_scan_packed(uint32_t v) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t n = __shfl_up_sync(0xffffffffu, v, o);
    if (lane >= o) v += n;
  }
  return v;
}

constexpr int kSpawnP = 8;             // parents per thread per pass (coarsening)
constexpr uint32_t kSpawnGroup = 1024; // parents whose children are kept or dropped together

// An LFVector of the growth, by one block.  A warp takes 32 * kSpawnP consecutive parents of a
// pass, 32 at a time, so its children are one run of the LFVector, round
// after round, and the block needs one total per warp: one block barrier per
// pass, after which every thread knows where its warp's run starts and
// whether the pass stays inside the allocated buckets (only when it does
// not, warp 0 allocates behind a second barrier).
//
// The children of 32 parents are written by the warp together, lane i taking
// children i, i + 32, ...: the parents with children leave their pos and vel
// in shared memory in order, one warp-wide OR of the bits of their first
// children gives the heads among 32 children, and a child's parent is the
// number of heads up to it.  Consecutive lanes store consecutive children.
//
// The kernel reads 16 bytes per parent and writes 16 per child; what kept it
// from that rate were instructions and waits (a five-step shuffle search per
// child, 64-bit bucket math per parent and child, three barriers per pass
// over 1024 threads, one block per SM).  Measured on GB300 for the last of 8
// generations from 2^20 records (2^27 parents, as many children, 1024
// LFVectors; 4.3 GB): 1.04 ms before, 0.80 now (0.63 at the copy rate); with the
// children's loop unrolled over the rounds 1.07 (instruction-cache misses).
template <int NT>
__device__ __forceinline__ void spawn_lfv(const ArrayView& v, uint32_t l, uint32_t gen, uint64_t seed, int only_newborn,
                                          uint64_t* born) {
  constexpr int P = kSpawnP, KP = P / 2, NW = NT / 32;
  constexpr uint32_t kPass = NT * P;
  static_assert(kPass % kSpawnGroup == 0, "whole groups of parents per pass");
  extern __shared__ uint2 s_pv[];            // [NW][32 P] pos and vel of the warps' parents with children;
                                             // then [NW][32 P] uint32: every parent's count and offset
  __shared__ alignas(16) uint32_t s_wt[2][NW];   // the warps' children, by pass parity
  __shared__ uint64_t s_tab[kMaxBuckets];    // the LFVector's bucket table (copy)
  __shared__ uint32_t s_nb;

  const uint32_t t = threadIdx.x, lane = t & 31, w = t >> 5;
  const uint32_t upto = 0xffffffffu >> (31 - lane);          // lanes 0 .. lane
  uint2* const my_pv = s_pv + w * (32 * P);
  uint32_t* const my_ce = reinterpret_cast<uint32_t*>(s_pv + NT * P) + w * (32 * P);
  const uint64_t* bk = v.buckets + static_cast<uint64_t>(l) * kMaxBuckets;
  const uint64_t s = v.sizes[l];                       // parents end here
  const uint64_t first = only_newborn ? born[l] : 0;   // ... and start here
  const uint64_t goff = v.offsets[l];                  // global index of local 0 at generation start
  const uint64_t id_hi = (static_cast<uint64_t>(gen + 1) << 56) | (static_cast<uint64_t>(l) << 40);
  // The state of the parent at local index j: z0 + j * GOLDEN (the key's
  // fields do not overlap: global indices stay below 2^48).
  const uint64_t z0 = seed + ((static_cast<uint64_t>(gen) << 48) + goff + 1) * kSpawnGolden;
  uint32_t nb = v.nbuckets[l];
  for (uint32_t i = t; i < nb; i += NT) s_tab[i] = bk[i];
  __syncthreads();

  uint64_t base = s, cap = bucket_first(nb, v.log2B);
  uint32_t par = 0;
  bool stop = false;
  for (uint64_t c0 = first; c0 < s && !stop; c0 += kPass, par ^= 1u) {
    // The warp's parents: j0 + 32 p + lane.  Mostly all in one bucket.
    const uint64_t j0 = c0 + w * (32 * P);
    uint32_t jb;
    uint64_t joff;
    bucket_of(j0, v.log2B, jb, joff);
    const uint64_t left = j0 < s ? s - j0 : 0;                 // parents from j0 on
    const uint32_t have = left < 32 * P ? static_cast<uint32_t>(left) : 32u * P;
    const bool one = joff + have <= bucket_len(jb, v.log2B);
    const uint2* src = have && one ? reinterpret_cast<const uint2*>(s_tab[jb] + joff * 16 + 8) : nullptr;
    if (have && !one) {   // across buckets: pos and vel through shared memory
#pragma unroll 1
      for (uint32_t i = lane; i < have; i += 32) {
        uint32_t bb;
        uint64_t off;
        bucket_of(j0 + i, v.log2B, bb, off);
        my_pv[i] = *reinterpret_cast<const uint2*>(s_tab[bb] + off * 16 + 8);
      }
    }
    uint2 pv[P];
#pragma unroll
    for (int p = 0; p < P; ++p) {
      const uint32_t i = 32 * p + lane;
      pv[p] = make_uint2(0, 0);
      if (i < have) pv[p] = one ? __ldcs(src + 2 * i) : my_pv[i];
    }
    __syncwarp();   // my_pv is read before it is filled again
    uint64_t z = z0 + (j0 + lane) * kSpawnGolden;
    uint32_t pk[KP], inc[KP];
#pragma unroll
    for (int j2 = 0; j2 < KP; ++j2) {
      uint32_t c[2];
#pragma unroll
      for (int h = 0; h < 2; ++h, z += 32 * kSpawnGolden) {
        const uint32_t n = trailing_ones(spawn_mix(z));
        c[h] = 32u * (2 * j2 + h) + lane < have ? n : 0u;
      }
      pk[j2] = c[0] | (c[1] << 16);
      inc[j2] = warp_scan_packed(pk[j2]);
    }
    // The warp's children, and the parents that have some in order.
    uint32_t run = 0, heads = 0;   // children, parents with children of the earlier rounds
#pragma unroll
    for (int j2 = 0; j2 < KP; ++j2) {
      const uint32_t ex = inc[j2] - pk[j2];
      const uint32_t wt = __shfl_sync(0xffffffffu, inc[j2], 31);
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const uint32_t c = (pk[j2] >> (16 * h)) & 0xFFFFu;
        const uint32_t m = __ballot_sync(0xffffffffu, c != 0);
        if (c) my_pv[heads + __popc(m & (upto >> 1))] = pv[2 * j2 + h];
        my_ce[32 * (2 * j2 + h) + lane] = (c << 16) | ((ex >> (16 * h)) & 0xFFFFu);
        heads += __popc(m);
        run += (wt >> (16 * h)) & 0xFFFFu;
      }
    }
    if (lane == 0) s_wt[par][w] = run;
    __syncthreads();

    // Where the warp's run starts, and the pass's children.
    uint32_t woff, total;
    if constexpr (NW == 4) {
      const uint4 y = *reinterpret_cast<const uint4*>(s_wt[par]);
      woff = (w > 0 ? y.x : 0u) + (w > 1 ? y.y : 0u) + (w > 2 ? y.z : 0u);
      total = y.x + y.y + y.z + y.w;
    } else {
      const uint32_t y = lane < NW ? s_wt[par][lane] : 0u;
      const uint32_t yi = warp_scan_packed(y);
      woff = __shfl_sync(0xffffffffu, yi - y, w);
      total = __shfl_sync(0xffffffffu, yi, 31);
    }
    uint32_t commit = total;
    if (base + total > cap) {   // the same in every thread
      if (w == 0) {
        const uint32_t got = grow_buckets_warp(v, l, nb, buckets_for(base + total, v.log2B));
        if (lane == 0) {
          v.nbuckets[l] = got;
          s_nb = got;
        }
      }
      __syncthreads();          // synchronize(): the buckets exist before any write
      const uint32_t got = s_nb;
      for (uint32_t i = nb + t; i < got; i += NT) s_tab[i] = bk[i];
      nb = got;
      cap = bucket_first(nb, v.log2B);
      if (base + total > cap) {   // keep the groups of parents whose children fit
        commit = 0;
        uint32_t upto_w = 0;
        for (uint32_t i = 0; i < static_cast<uint32_t>(NW); ++i) {
          upto_w += s_wt[par][i];
          if ((i + 1) * (32 * P) % kSpawnGroup == 0 && base + upto_w <= cap) commit = upto_w;
        }
        stop = true;
        if (t == 0) latch_error(v.status, GGA_ERR_POOL_EXHAUSTED);
      }
      __syncthreads();          // the table is filled; s_nb and s_wt are read
    }

    // The children.  A pass mostly is kept whole and stays in one bucket:
    // then a child's address is the pass's plus 16 bytes per place.
    uint32_t cb;
    uint64_t coff;
    bucket_of(base, v.log2B, cb, coff);
    const bool flat = commit == total && coff + total <= bucket_len(cb, v.log2B);
    const uint64_t id0 = id_hi | base;   // + the child's place in the pass (ids stay below 2^40 per LFVector)
    uint32_t q0 = woff, head0 = 0;       // the round's first child, its first parent with children
    auto children = [&](auto store) {
#pragma unroll 1
      for (int p = 0; p < P; ++p) {
        const uint32_t ce = my_ce[32 * p + lane], c = ce >> 16, ex = ce & 0xFFFFu;
        const uint32_t n = __shfl_sync(0xffffffffu, ex + c, 31);
        uint32_t at = c ? ex : ~0u;      // the parent's first child, from the window's start; 32 and more: not in it
        for (uint32_t q = lane; q < n + lane; q += 32, at -= 32) {
          const uint32_t m = __reduce_or_sync(0xffffffffu, at < 32u ? 1u << at : 0u);
          if (q < n) store(q0 + q, my_pv[head0 + __popc(m & upto) - 1]);
          head0 += __popc(m);
        }
        q0 += n;
      }
    };
    if (flat) {
      uint4* const dst = reinterpret_cast<uint4*>(total ? s_tab[cb] + coff * 16 : 0);
      children([&](uint32_t q, uint2 x) {
        const uint64_t id = id0 + q;
        __stcs(dst + q, make_uint4(static_cast<uint32_t>(id), static_cast<uint32_t>(id >> 32), x.x, x.y));
      });
    } else {
      children([&](uint32_t q, uint2 x) {
        if (q >= commit) return;
        uint32_t bb;
        uint64_t off;
        bucket_of(base + q, v.log2B, bb, off);
        const uint64_t id = id0 + q;
        __stcs(reinterpret_cast<uint4*>(s_tab[bb]) + off,
               make_uint4(static_cast<uint32_t>(id), static_cast<uint32_t>(id >> 32), x.x, x.y));
      });
    }
    base += commit;
    // The next pass writes my_pv and my_ce after this, and s_wt of this parity only
    // two passes later, behind a barrier every thread reaches past its reads.
    __syncwarp();
  }
  if (t == 0) {
    v.sizes[l] = base;
    if (only_newborn) born[l] = s;
  }
}

// An LFVector that a small block would be too long with: its rounds follow one another, and the others' blocks leave the SMs
// idle meanwhile.  (Half of 2^20 records in one of 1024 LFVectors, 4
// generations: 23.0 ms by its block of 128 threads, 7.9 by one of 1024.)
// From the offsets, which stay those of the generation's start.
constexpr uint64_t kSpawnLarge = 16384;
__device__ __forceinline__ bool spawn_large(const ArrayView& v, uint64_t l) {
  const uint64_t size = v.offsets[l + 1] - v.offsets[l];
  return size > kSpawnLarge && size / 4 > v.offsets[v.L] / v.L;
}

// One block per LFVector; with small blocks, those that are not large.
template <int NT, int MINB>
__global__ void __launch_bounds__(NT, MINB) spawn_kernel(const __grid_constant__ ArrayView v, uint32_t gen,
                                                         uint64_t seed, int only_newborn, uint64_t* born) {
  if (NT < 512 && spawn_large(v, blockIdx.x)) return;   // spawn_finish_kernel's
  spawn_lfv<NT>(v, blockIdx.x, gen, seed, only_newborn, born);
}

// After spawn_kernel: the large ones -- every block looks through its share of
// the LFVectors (at most a quarter are large, usually none) -- and, by the last
// block to finish, what ends every insertion (finalize_kernel).  A kernel of
// its own for the large ones was 5 us more per generation.
__global__ void __launch_bounds__(1024, 1) spawn_finish_kernel(const __grid_constant__ ArrayView v, uint32_t gen,
                                                               uint64_t seed, int only_newborn, uint64_t* born,
                                                               uint32_t* done) {
  __shared__ uint32_t s_large[1024];
  __shared__ uint32_t s_n;
  for (uint64_t l0 = blockIdx.x; l0 < v.L; l0 += static_cast<uint64_t>(gridDim.x) * 1024) {   // block-uniform
    if (threadIdx.x == 0) s_n = 0;
    __syncthreads();
    const uint64_t l = l0 + static_cast<uint64_t>(gridDim.x) * threadIdx.x;
    if (l < v.L && spawn_large(v, l)) s_large[atomicAdd(&s_n, 1u)] = static_cast<uint32_t>(l);
    __syncthreads();
    const uint32_t n = s_n;
    for (uint32_t i = 0; i < n; ++i) {
      spawn_lfv<1024>(v, s_large[i], gen, seed, only_newborn, born);
      __syncthreads();
    }
    __syncthreads();   // s_n and s_large are read
  }
  __shared__ FinalizeShared s_fin;
  __shared__ int s_last;
  if (threadIdx.x == 0) {
    __threadfence();
    s_last = atomicAdd(done, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  ring_fixup_class(v.pool, threadIdx.x);
  finalize_block(v, nullptr, nullptr, nullptr, 1, s_fin);
  if (threadIdx.x == 0) *done = 0;
}

// One streaming pass over flattened records: pos += vel.
__global__ void __launch_bounds__(256) work_pass_kernel(uint4* __restrict__ rec, uint64_t n) {
  const uint64_t stride = static_cast<uint64_t>(gridDim.x) * blockDim.x;
  constexpr int U = 4;
  for (uint64_t i0 = static_cast<uint64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i0 < n; i0 += stride * U) {
    uint4 r[U];
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (i0 + u * stride < n) r[u] = __ldcs(rec + i0 + u * stride);
#pragma unroll
    for (int u = 0; u < U; ++u) {
      if (i0 + u * stride < n) {
        r[u].z = __float_as_uint(__fadd_rn(__uint_as_float(r[u].z), __uint_as_float(r[u].w)));
        __stcs(rec + i0 + u * stride, r[u]);
      }
    }
  }
}

}  // namespace

template <int NT>
constexpr int spawn_smem() { return NT * kSpawnP * static_cast<int>(sizeof(uint2) + sizeof(uint32_t)); }

template <int NT, int MINB>
static int launch_spawn(const ArrayView& v, uint32_t gen, uint64_t seed, int only_newborn, uint64_t* born,
                        uint32_t* done, int sms, cudaStream_t st) {
  auto kern = spawn_kernel<NT, MINB>;
  if (spawn_smem<NT>() > 32768) cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, spawn_smem<NT>());
  kern<<<v.L, NT, spawn_smem<NT>(), st>>>(v, gen, seed, only_newborn, born);
  if (NT >= 512) return cudaGetLastError() == cudaSuccess ? launch_finalize(v, st) : GGA_ERR_CUDA;
  cudaFuncSetAttribute(spawn_finish_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, spawn_smem<1024>());
  spawn_finish_kernel<<<sms, 1024, spawn_smem<1024>(), st>>>(v, gen, seed, only_newborn, born, done);
  return cudaGetLastError() == cudaSuccess ? GGA_OK : GGA_ERR_CUDA;
}

int launch_twophase_spawn(const ArrayView& v, uint32_t gen, uint64_t seed, int only_newborn, uint64_t* born,
                          uint32_t* done, cudaStream_t st) {
  // The children's order and values depend on parent indices only, so the
  // block size is free, whatever T is: the smallest whose blocks still fill
  // the SMs (about 1024 threads each).  Small blocks wait less at their
  // barriers and leave no wave half empty: 1024 LFVectors are 1024 resident
  // blocks of 128 threads, but seven waves of one 1024-thread block per SM.
  // They leave LFVectors far above the average to blocks of 1024.
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return GGA_ERR_CUDA;
  const uint32_t per_sm = v.L / static_cast<uint32_t>(sms);
  if (per_sm >= 4) return launch_spawn<128, 8>(v, gen, seed, only_newborn, born, done, sms, st);
  if (per_sm >= 2) return launch_spawn<256, 4>(v, gen, seed, only_newborn, born, done, sms, st);
  if (per_sm >= 1) return launch_spawn<512, 2>(v, gen, seed, only_newborn, born, done, sms, st);
  return launch_spawn<1024, 1>(v, gen, seed, only_newborn, born, done, sms, st);
}

int launch_twophase_work(void* records, uint64_t n, uint32_t passes, int num_sms, cudaStream_t st) {
  if (n == 0) return GGA_OK;
  int per_sm = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, work_pass_kernel, 256, 0) != cudaSuccess ||
      per_sm < 1)
    per_sm = 1;
  const uint64_t want = (n + 255) / 256;
  const uint64_t wave = static_cast<uint64_t>(num_sms) * per_sm;
  const unsigned grid = static_cast<unsigned>(want < wave ? want : wave);
  for (uint32_t p = 0; p < passes; ++p)
    work_pass_kernel<<<grid, 256, 0, st>>>(static_cast<uint4*>(records), n);
  return cudaGetLastError() == cudaSuccess ? GGA_OK : GGA_ERR_CUDA;
}

}  // namespace gga
