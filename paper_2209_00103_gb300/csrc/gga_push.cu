// gga_push.cu -- the device API's own entry points: the view a user kernel
// pushes through, the commit that follows such a kernel, the generated
// insertion written as a user kernel would write it (Algorithm 1 as the
// paper states it: one block per LFVector, one push per round, through the
// device API's BlockPusher), and pushes of values read from device memory
// (RoundsPusher, several rounds per push).
#include <algorithm>
#include <cmath>

#include "gga_core.cuh"
#include "gga_device.cuh"
#include "gga_gen.cuh"

namespace gga {

// Block l draws round r's counts and values exactly as gga_insert_generated
// does (SplitMix64 on ((r << 32) | l*T + t)), and appends them with one push
// per round through a BlockPusher on LFVector l.  A round that does not fit
// ends the block's rounds (the rounds that fit are kept, as in every
// insertion).
//
// A round is a scan, a barrier and the writes of about T elements, so the
// kernel is bound by the instructions around the elements and by the wait at
// the barrier.  A thread plays kPushSlots consecutive threads of the
// LFVector: one scan and one share of the barrier serve four of them, a
// block of T = 512 has four warps, and all 1024 blocks of the paper-shaped
// workload are resident at once; the push is assembled in shared memory and
// leaves as one 128-bit store per thread behind the next push's barrier.
// Measured on GB300 for 1024 LFVectors x 512 threads x 512 rounds, int32:
// 0.87 ms against 2.27 ms with one thread per LFVector thread (blocks of
// 512, two per SM) storing its own elements.
// Up to T = 128 a thread plays one: a block of a few lanes would otherwise do
// four threads' work in each (1500 LFVectors x 32 threads x 100 rounds with
// geometric counts, clear and flatten included: 225 us with four, 139 with one).
constexpr int kPushSlots = 4;
constexpr uint32_t kPushSlotsMinT = 129;

// Shared memory for the stage's two halves.  Wanted: a push at the counts' mean
// and eight standard deviations of its sum (a larger push stores straight to
// the buckets), for mean 1 and variance 2 at least.  Where that would keep
// blocks off the SM, as many blocks as hold 2.5 deviations stay resident and
// share its memory: 2^24 Poisson draws of mean 6 into 16-byte elements at T =
// 512: 569 us with two blocks per SM, 845 with one that has room for all.
// (Stage for mean one, larger pushes by the threads' own stores, int32 at T =
// 512, mean 3 and 6: 280 and 646 us; now 155 and 258.)
constexpr uint32_t kSmBytes = 233472, kPushOwnBytes = 6144;   // an SM's shared memory; a block's beside the stage

uint32_t push_stage_bytes(uint32_t T, uint32_t E, uint32_t nt, const GenParams& g) {
  double mean = 1, var = 2;
  if (g.dist == GGA_DIST_POISSON) {
    double sq = 0;   // of c^2 = sum over k < c of 2 k + 1 (ascending thresholds; a bound of the kind for others)
    for (uint32_t k = 0; k < g.nthr; ++k) sq += (2.0 * k + 1.0) * (1.0 - g.thr[k] / 4294967296.0);
    mean = std::max(mean, static_cast<double>(g.mean));
    var = std::max(var, sq - static_cast<double>(g.mean) * g.mean);
  }
  const double sd = std::sqrt(T * var), vec = 16.0 / E;
  const double want = 2 * E * (T * mean + 8 * sd + 2 * vec), least = 2 * E * (T * mean + 2.5 * sd + 2 * vec);
  const uint32_t blocks = std::min(1024 / nt, static_cast<uint32_t>(kSmBytes / (least + kPushOwnBytes)));   // by registers
  if (blocks == 0) return 0;
  return static_cast<uint32_t>(std::min(want, static_cast<double>(kSmBytes / blocks - kPushOwnBytes))) / 32 * 32;
}

template <int E, int DIST, int S>
__global__ void __launch_bounds__(S == 1 ? 128 : 1024 / S, S == 1 ? 8 : 4) push_generated_kernel(const ArrayView* view,
                                                                              const __grid_constant__ GenParams g,
                                                                              uint32_t R, uint32_t T,
                                                                              uint32_t stage_bytes) {
  typedef typename Elem<E>::T V;
  typedef typename std::conditional<E == 4, uint32_t, uint64_t>::type W;   // a 4-byte element keeps the low 32 bits
  extern __shared__ uint4 s_stage[];
  __shared__ PushShared sh;
  __shared__ ThresholdTable s_thr;
  const uint32_t l = blockIdx.x, t = S * threadIdx.x;
  const uint64_t g0 = static_cast<uint64_t>(l) * T + t;
  const bool tabled = DIST == GGA_DIST_POISSON && g.thr_sorted;
  if (tabled) s_thr.fill(g, threadIdx.x, blockDim.x);   // the pusher's first barrier follows
  RoundDraws draws[S];
#pragma unroll
  for (int i = 0; i < S; ++i) draws[i] = RoundDraws(g.seed, g0 + i);
  BlockPusher<V> pusher(view, l, sh, s_stage, stage_bytes);
  const W va = static_cast<W>(g.va), vb = static_cast<W>(g.vb), vc = static_cast<W>(g.vc);
  W vr = va * static_cast<W>(g0) + vb * static_cast<W>(g.round0);
#pragma unroll 1
  for (uint32_t i = 0; i < R; ++i, vr += vb) {
    const uint64_t r = static_cast<uint64_t>(g.round0) + i;
    uint32_t c[S], sum = 0;
#pragma unroll
    for (int q = 0; q < S; ++q) {
      // Drawn unconditionally and masked (no branch around every draw).
      if (tabled) c[q] = s_thr.count(g.nthr, splitmix_mix_hi(draws[q].state(r)));
      else c[q] = gen_count_state<false, DIST>(g, draws[q].state(r));
      if (t + q >= T) c[q] = 0;
      sum += c[q];
    }
    const bool ok = pusher.template push_run<S * 63>(sum, [&](auto put) {   // counts stay below 64
      uint32_t k = 0;
#pragma unroll
      for (int q = 0; q < S; ++q) {
        W x = vr + va * static_cast<W>(q);
        if (max_count<DIST>() == 1 || max_count<DIST>() == 2) {
          if constexpr (decltype(put)::kOneStore) {
            store_shared_if<E>(put.at + k, gen_value<E>(x), c[q] > 0);
            if (max_count<DIST>() == 2) store_shared_if<E>(put.at + k + 1, gen_value<E>(x + vc), c[q] > 1);
          } else {
            if (c[q] > 0) put(k, gen_value<E>(x));
            if (max_count<DIST>() == 2 && c[q] > 1) put(k + 1, gen_value<E>(x + vc));
          }
        } else {
          for (uint32_t m = 0; m < c[q]; ++m, x += vc) put(k + m, gen_value<E>(x));
        }
        k += c[q];
      }
    });
    if (!ok) break;
  }
  pusher.flush();
}

template <int E>
void launch_push_generated_as(const ArrayView& v, const ArrayView* dview, const GenParams& g, uint32_t rounds,
                              cudaStream_t st) {
  const uint32_t slots = v.T >= kPushSlotsMinT ? kPushSlots : 1;
  const uint32_t nt = ((v.T + slots - 1) / slots + 31) / 32 * 32;
  const uint32_t smem = push_stage_bytes(v.T, E, nt, g);
#define GGA_PUSH(D)                                                                                         \
  do {                                                                                                      \
    auto kern = slots == 1 ? push_generated_kernel<E, D, 1> : push_generated_kernel<E, D, kPushSlots>;      \
    if (smem > 32768u)   /* with the count table the block's shared memory may pass 48 KB; the limit is the \
                            kernel's: other threads launch it for arrays of other shapes */                 \
      cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmBytes - kPushOwnBytes);    \
    kern<<<v.L, nt, smem, st>>>(dview, g, rounds, v.T, smem);                                               \
  } while (0)
  switch (g.dist) {
    case GGA_DIST_BERNOULLI: GGA_PUSH(GGA_DIST_BERNOULLI); break;
    case GGA_DIST_UNIFORM3: GGA_PUSH(GGA_DIST_UNIFORM3); break;
    case GGA_DIST_GEOMETRIC: GGA_PUSH(GGA_DIST_GEOMETRIC); break;
    default: GGA_PUSH(GGA_DIST_POISSON); break;
  }
#undef GGA_PUSH
}

int launch_push_generated(const ArrayView& v, const ArrayView* dview, const gga_gen_spec& spec, uint32_t rounds,
                          cudaStream_t st) {
  const GenParams g = make_gen_params(spec);
  if (v.E == 4) launch_push_generated_as<4>(v, dview, g, rounds, st);
  else if (v.E == 8) launch_push_generated_as<8>(v, dview, g, rounds, st);
  else launch_push_generated_as<16>(v, dview, g, rounds, st);
  if (cudaGetLastError() != cudaSuccess) return GGA_ERR_CUDA;
  return launch_finalize(v, st);
}

// Memory-sourced pushes through the device API: block l appends, per
// thread slot t and round r, counts[r][l][t] copies of inputs[r][l][t],
// K rounds per push of a gga::RoundsPusher (staged, 128-bit stores).  A
// thread plays S consecutive slots S t, ..., S t + S - 1 and pushes their
// counts together (its elements are slot S t's copies, then S t + 1's, ...,
// which is their order in the LFVector): one scan slot and one share of
// every barrier then serve S slots, and the blocks (512 / S threads for
// T = 512) are small enough for all 1024 of the paper-shaped workload to
// be resident at once.  The kernel streams counts and inputs in and the
// elements out; its rate is that of the bytes it keeps in flight.  With
// WIDE (T a multiple of S, both buffers 16-byte aligned) a thread's S counts
// and S inputs of a round are 128-bit loads, and a round's loads for the next
// push are issued as soon as this push has staged the round, so they are in
// flight during its barrier and write-out without a register more.  A push
// that does not fit ends the block's rounds.
// Measured on GB300 for the paper-shaped workload (1024 x 512, 512 rounds,
// int32): one slot per thread, K = 8, 2 blocks per SM: 1.42 ms (with the
// loads prefetched into shared memory by cp.async: 1.52 ms); S = 2, K = 4,
// 4 per SM: 0.98 ms; S = 4, K = 2, 8 per SM: 0.90 ms; S = 4, K = 4, 8 per
// SM: 0.84 ms, 0.80 with the write-out's bucket math per bucket; with one
// cursor for all pushes, the wide early loads and predicated stores 0.56 ms
// (a conditional per store: 0.64; a loop per slot: 0.81).
template <int S, typename V, bool WIDE>
__device__ __forceinline__ void load_slots(V (&x)[S], const V* __restrict__ p, uint32_t have) {
  constexpr uint32_t kWord = S * sizeof(V) >= 16 ? 16 : S * sizeof(V);   // bytes of a load
  if constexpr (WIDE && kWord == 16) {
    constexpr uint32_t kPer = 16 / sizeof(V);
#pragma unroll
    for (int i = 0; i < S; i += kPer) {
      uint4 w = make_uint4(0, 0, 0, 0);
      if (have) w = __ldcs(reinterpret_cast<const uint4*>(p + i));
      if constexpr (sizeof(V) == 16) {
        x[i] = w;
      } else if constexpr (sizeof(V) == 8) {
        x[i] = w.x | static_cast<V>(w.y) << 32;
        x[i + 1] = w.z | static_cast<V>(w.w) << 32;
      } else {
        x[i] = w.x;
        x[i + 1] = w.y;
        x[i + 2] = w.z;
        x[i + 3] = w.w;
      }
    }
  } else if constexpr (WIDE && sizeof(V) == 4 && S == 2) {
    uint2 w = make_uint2(0, 0);
    if (have) w = __ldcs(reinterpret_cast<const uint2*>(p));
    x[0] = w.x;
    x[1] = w.y;
  } else {
#pragma unroll
    for (int i = 0; i < S; ++i) {
      x[i] = V();
      if (static_cast<uint32_t>(i) < have) x[i] = __ldcs(p + i);
    }
  }
}

template <int E, int K, int S, int MINB, bool WIDE>
__global__ void __launch_bounds__(512 / S, MINB) push_expand_s_kernel(const ArrayView* view,
                                                                  const uint32_t* __restrict__ counts,
                                                                  const typename Elem<E>::T* __restrict__ inputs,
                                                                  uint32_t R, uint32_t L, uint32_t T,
                                                                  uint32_t stage_bytes) {
  typedef typename Elem<E>::T V;
  extern __shared__ uint4 s_stage[];
  __shared__ RoundsShared<K> s_rounds;
  const uint32_t l = blockIdx.x, t = S * threadIdx.x;
  const uint32_t mine = t < T ? (T - t < S ? T - t : S) : 0u;   // slots this thread plays
  const uint64_t at0 = static_cast<uint64_t>(l) * T + t, row = static_cast<uint64_t>(L) * T;
  uint32_t cs[K][S];
  V x[K][S];
  auto load = [&](int k, uint32_t r) {
    const uint64_t at = at0 + r * row;
    const uint32_t have = r < R ? mine : 0u;
    load_slots<S, uint32_t, WIDE>(cs[k], counts + at, have);
    load_slots<S, V, WIDE>(x[k], inputs + at, have);
  };
#pragma unroll
  for (int k = 0; k < K; ++k) load(k, k);
  RoundsPusher<V, K> pusher(view, l, s_rounds, s_stage, stage_bytes);
#pragma unroll 1
  for (uint32_t r0 = 0; r0 < R; r0 += K) {
    uint32_t c[K], any = 0;
#pragma unroll
    for (int k = 0; k < K; ++k) {
      c[k] = 0;
#pragma unroll
      for (int i = 0; i < S; ++i) {
        c[k] += cs[k][i];
        any |= cs[k][i];
      }
    }
    if (S > 1 && any >= (1u << 30)) {   // sums that pass 32 bits: the thread pushes nothing in that round
#pragma unroll
      for (int k = 0; k < K; ++k) {
        uint64_t sum = 0;
#pragma unroll
        for (int i = 0; i < S; ++i) sum += cs[k][i];
        if (sum >> 32) {
          c[k] = 0;
#pragma unroll
          for (int i = 0; i < S; ++i) cs[k][i] = 0;
          latch_error(view->status, GGA_ERR_INVALID);
        }
      }
    }
    const uint32_t done = pusher.push_run(c, [&](uint32_t kr, auto put) {
      // Two copies by predicated stores, the third and later ones (rare at
      // about one copy per slot) by a loop only the threads that have some enter.
      constexpr uint32_t kFlat = decltype(put)::kOneStore ? 2 : 0;
      uint32_t m = 0, most = 0;
#pragma unroll
      for (int i = 0; i < S; ++i) {
        const uint32_t n = cs[kr][i];
        if constexpr (kFlat > 0) {
          store_shared_if<E>(put.at + m, x[kr][i], n > 0);
          store_shared_if<E>(put.at + m + 1, x[kr][i], n > 1);
        }
        m += n;
        most = max(most, n);
      }
      if (most > kFlat) {
        m = 0;
#pragma unroll
        for (int i = 0; i < S; ++i) {
          for (uint32_t j = kFlat; j < cs[kr][i]; ++j) put(m + j, x[kr][i]);
          m += cs[kr][i];
        }
      }
      load(static_cast<int>(kr), r0 + K + kr);
    });
    if (done < static_cast<uint32_t>(K)) break;
  }
}

template <int E, int K, int S, int MINB, bool WIDE>
int launch_expand_as(const ArrayView& v, const ArrayView* dview, const uint32_t* counts, const void* inputs,
                     uint32_t rounds, cudaStream_t st) {
  const uint32_t NTS = ((v.T + S - 1) / S + 31) / 32 * 32;
  // Stage: twice a call's elements at one per slot of 512 (larger calls go
  // unstaged; with 28 KB a block instead of 16 the loads in flight lack L1, and
  // the paper-shaped workload takes 0.75 ms instead of 0.56).
  const size_t smem = static_cast<size_t>(K) * 512u * E * 2u;
  auto kern = push_expand_s_kernel<E, K, S, MINB, WIDE>;
  cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
  kern<<<v.L, NTS, smem, st>>>(dview, counts, static_cast<const typename Elem<E>::T*>(inputs), rounds, v.L, v.T,
                               static_cast<uint32_t>(smem));
  if (cudaGetLastError() != cudaSuccess) return GGA_ERR_CUDA;
  return launch_finalize(v, st);
}

template <int E, int K, int S, int MINB>
int launch_expand_s(const ArrayView& v, const ArrayView* dview, const uint32_t* counts, const void* inputs,
                    uint32_t rounds, cudaStream_t st) {
  // Every row of T counts and inputs then starts on a 16-byte boundary (8
  // for two counts), and a thread plays all of its slots or none.
  const bool wide = S > 1 && v.T % S == 0 &&
                    ((reinterpret_cast<uintptr_t>(counts) | reinterpret_cast<uintptr_t>(inputs)) & 15) == 0;
  return wide ? launch_expand_as<E, K, S, MINB, true>(v, dview, counts, inputs, rounds, st)
              : launch_expand_as<E, K, S, MINB, false>(v, dview, counts, inputs, rounds, st);
}

int launch_push_expand(const ArrayView& v, const ArrayView* dview, const uint32_t* counts, const void* inputs,
                       uint32_t rounds, cudaStream_t st) {
  if (v.T > 512) return GGA_ERR_INVALID;
  // Few LFVectors: the time is a block's chain of pushes, which more threads
  // with one slot each shorten (20 LFVectors x 512 x 200 rounds, int32: 249 us
  // with four slots, 160 with one, clear and flatten included).
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return GGA_ERR_CUDA;
  if (v.L <= static_cast<uint32_t>(sms)) {
    if (v.E == 4) return launch_expand_as<4, 4, 1, 2, false>(v, dview, counts, inputs, rounds, st);
    if (v.E == 8) return launch_expand_as<8, 2, 1, 2, false>(v, dview, counts, inputs, rounds, st);
    return launch_expand_as<16, 2, 1, 2, false>(v, dview, counts, inputs, rounds, st);
  }
  if (v.E == 4) return launch_expand_s<4, 4, 4, 7>(v, dview, counts, inputs, rounds, st);
  if (v.E == 8) return launch_expand_s<8, 2, 4, 7>(v, dview, counts, inputs, rounds, st);
  return launch_expand_s<16, 2, 2, 4>(v, dview, counts, inputs, rounds, st);
}

}  // namespace gga

extern "C" {

int gga_device_view(gga_handle h, const void** view_dev) {
  if (!h || !view_dev) return GGA_ERR_INVALID;
  *view_dev = gga::handle_dview(h);
  return *view_dev ? GGA_OK : GGA_ERR_INVALID;
}

int gga_device_commit(gga_handle h, void* stream) {
  gga::ArrayView v;
  if (!gga::handle_parts(h, &v, nullptr, nullptr, nullptr)) return GGA_ERR_INVALID;
  return gga::launch_finalize(v, static_cast<cudaStream_t>(stream));
}

int gga_push_expand(gga_handle h, const uint32_t* counts_dev, const void* inputs_dev, uint32_t rounds,
                    void* stream) {
  gga::ArrayView v;
  if (!h || !gga::handle_parts(h, &v, nullptr, nullptr, nullptr)) return GGA_ERR_INVALID;
  if (rounds == 0) return GGA_OK;
  if (!counts_dev || !inputs_dev || v.T > 512) return GGA_ERR_INVALID;
  if ((reinterpret_cast<uintptr_t>(counts_dev) & 3) != 0 || (reinterpret_cast<uintptr_t>(inputs_dev) % v.E) != 0)
    return GGA_ERR_INVALID;
  return gga::launch_push_expand(v, gga::handle_dview(h), counts_dev, inputs_dev, rounds,
                                 static_cast<cudaStream_t>(stream));
}

int gga_push_generated(gga_handle h, const gga_gen_spec* spec, uint32_t rounds, void* stream) {
  gga::ArrayView v;
  if (!h || !spec || !gga::handle_parts(h, &v, nullptr, nullptr, nullptr)) return GGA_ERR_INVALID;
  if (spec->dist > GGA_DIST_POISSON || spec->n_thresholds > GGA_MAX_THRESHOLDS) return GGA_ERR_INVALID;
  if (spec->dist == GGA_DIST_POISSON && spec->n_thresholds == 0) return GGA_ERR_INVALID;
  if (rounds == 0) return GGA_OK;
  return gga::launch_push_generated(v, gga::handle_dview(h), *spec, rounds, static_cast<cudaStream_t>(stream));
}

}  // extern "C"
