// gga_gen.cuh -- device helpers shared by the insertion kernels: the
// counter-based draws of the generated workloads, and the block-wide
// finalize (prefix sum of LFVector sizes, Sec. IV; work lists).
#pragma once

#include <type_traits>

#include "gga_core.cuh"

namespace gga {

struct GenParams {
  uint64_t seed, va, vb, vc;
  uint32_t dist, nthr, round0;
  uint32_t thr_sorted;   // 1: thr[0..nthr) ascending (set on the host)
  float mean;            // of a draw's count
  uint32_t thr[GGA_MAX_THRESHOLDS];
};

// SplitMix64 (Steele, Lea and Flood, 2014): output number key+1 of the
// stream seeded with `seed`.  The generator's state after key+1 steps is
// seed + (key+1) * GOLDEN (a Weyl sequence); the output is that state
// passed through the mixing function below.
constexpr uint64_t kGolden = 0x9E3779B97F4A7C15ull;

__device__ __forceinline__ uint64_t splitmix_mix(uint64_t z) {
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

// The high 32 bits of splitmix_mix(z): the final xor-shift by 31 changes
// the high word only by its own top bit, so the last step stays in 32 bits.
__device__ __forceinline__ uint32_t splitmix_mix_hi(uint64_t z) {
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  const uint32_t h = static_cast<uint32_t>(z >> 32);
  return h ^ (h >> 31);
}

__device__ __forceinline__ uint64_t splitmix(uint64_t seed, uint64_t key) {
  return splitmix_mix(seed + (key + 1) * kGolden);
}

// The draws of one thread over consecutive rounds, for keys
// (round << 32) | gid.  Write gid = gh * 2^32 + gl (gl < 2^32); the key's
// high word is then uint32(round) | gh and its low word gl, so the state is
//   seed + (gl + 1) * GOLDEN + ((hi_word * GOLDEN) mod 2^32) * 2^32,
// where only the last term depends on the round: one 32-bit multiply and
// one 32-bit add into the state's high word per draw, instead of a 64-bit
// multiply.  Equal to splitmix(seed, (round << 32) | gid) for every gid.
struct RoundDraws {
  uint64_t base;   // seed + (gl + 1) * GOLDEN
  uint32_t gh;     // gid >> 32
  __device__ __forceinline__ RoundDraws() : base(0), gh(0) {}
  __device__ __forceinline__ RoundDraws(uint64_t seed, uint64_t gid)
      : base(seed + ((gid & 0xFFFFFFFFull) + 1ull) * kGolden), gh(static_cast<uint32_t>(gid >> 32)) {}
  __device__ __forceinline__ uint64_t state(uint64_t round) const {
    const uint32_t hw = (static_cast<uint32_t>(round) | gh) * static_cast<uint32_t>(kGolden);
    return base + (static_cast<uint64_t>(hw) << 32);
  }
};

// Count of one draw from the mixed state z.  DIST >= 0 fixes the
// distribution at compile time (GGA_DIST_*), -1 reads g.dist.  Every
// distribution but the geometric one uses only the high word of the draw.
// SEARCH: g lives in shared memory, where a binary search over ascending
// thresholds costs a few indexed loads; for kernel parameters (constant bank)
// the unrolled count reads each threshold as an operand instead, and an indexed
// read would copy the parameters to local memory.  (The pass loops take ascending
// thresholds through a ThresholdTable, and come here with others.)
template <bool SEARCH = false, int DIST = -1>
__device__ __forceinline__ uint32_t gen_count_state(const GenParams& g, uint64_t z) {
  const uint32_t dist = DIST >= 0 ? static_cast<uint32_t>(DIST) : g.dist;
  if (dist == GGA_DIST_GEOMETRIC) {
    const uint64_t inv = ~splitmix_mix(z);
    return inv == 0 ? 63u : min(63u, static_cast<uint32_t>(__ffsll(static_cast<long long>(inv)) - 1));
  }
  const uint32_t u = splitmix_mix_hi(z);
  if (dist == GGA_DIST_BERNOULLI) return u >> 31;
  if (dist == GGA_DIST_UNIFORM3) return __umulhi(u, 3u);
  // c = #{k < nthr : u >= thr[k]}.  Ascending thresholds make that set a prefix,
  // whose length a binary search finds in five steps; other tables are counted.
  uint32_t c = 0;
  if (SEARCH && g.thr_sorted) {
#pragma unroll
    for (uint32_t step = 16; step > 0; step >>= 1)
      if (c + step <= g.nthr && u >= g.thr[c + step - 1]) c += step;
  } else {
#pragma unroll
    for (uint32_t k = 0; k < GGA_MAX_THRESHOLDS; ++k) c += (k < g.nthr) & (u >= g.thr[k]);
  }
  return c;
}

template <int E>
__device__ __forceinline__ typename Elem<E>::T gen_value(uint64_t v);
template <>
__device__ __forceinline__ uint32_t gen_value<4>(uint64_t v) { return static_cast<uint32_t>(v); }
template <>
__device__ __forceinline__ unsigned long long gen_value<8>(uint64_t v) { return v; }
template <>
__device__ __forceinline__ uint4 gen_value<16>(uint64_t v) {
  const float x = static_cast<float>(static_cast<uint32_t>(v & 0xFFFFull));
  const float y = static_cast<float>(static_cast<uint32_t>((v >> 16) & 0xFFFFull));
  return make_uint4(static_cast<uint32_t>(v), static_cast<uint32_t>(v >> 32), __float_as_uint(x), __float_as_uint(y));
}


inline GenParams make_gen_params(const gga_gen_spec& spec) {
  GenParams g;
  g.seed = spec.seed;
  g.va = spec.va;
  g.vb = spec.vb;
  g.vc = spec.vc;
  g.dist = spec.dist;
  g.nthr = spec.n_thresholds;
  g.round0 = spec.round0;
  g.thr_sorted = 1;
  for (int i = 0; i < GGA_MAX_THRESHOLDS; ++i) g.thr[i] = spec.thresholds[i];
  for (uint32_t i = 1; i < spec.n_thresholds && i < GGA_MAX_THRESHOLDS; ++i)
    if (g.thr[i] < g.thr[i - 1]) g.thr_sorted = 0;
  g.mean = g.dist == GGA_DIST_BERNOULLI ? 0.5f : 1.0f;
  if (g.dist == GGA_DIST_POISSON) {
    double m = 0;
    for (uint32_t k = 0; k < g.nthr; ++k) m += 1.0 - g.thr[k] / 4294967296.0;
    g.mean = static_cast<float>(m);
  }
  return g;
}

// ---------------------------------------------------------------------------
// Finalize: prefix sum of sizes, flatten/rw_b chunk prefix, copy chunk prefix.
// Run by one block (any multiple of 32 threads, 64 <= threads <= 1024).

__device__ __forceinline__ uint64_t block_excl_scan_u64(uint64_t x, uint64_t* s_warp, uint64_t& total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const uint64_t inc = warp_incl_scan(x);
  if (lane == 31) s_warp[warp] = inc;
  __syncthreads();
  if (warp == 0) {
    const uint64_t w = lane < nw ? s_warp[lane] : 0;
    const uint64_t wi = warp_incl_scan(w);
    if (lane < nw) s_warp[lane] = wi - w;
    if (lane == 31) s_warp[32] = wi;
  }
  __syncthreads();
  const uint64_t res = s_warp[warp] + inc - x;
  total = s_warp[32];
  __syncthreads();
  return res;
}

// Prefix sums of the LFVector sizes (offsets), of their 16 KB chunks
// (fl_prefix) and, if cp_prefix is given, of the insertion's copy chunks.
// The step is bound by latency (one block, a few KB): every thread takes up
// to kFinItems consecutive LFVectors, so 1024 LFVectors are one sweep of 256
// threads, the three sums go through one pass of warp scans, and every warp
// combines the warp totals by itself: one barrier per sweep (two when
// another sweep follows) against nine.  finalize_kernel at 1024 LFVectors on
// GB300: 9.5-12.2 us before this and the parallel fix-up, 4.3-4.7 us after.
constexpr int kFinItems = 4;
struct FinalizeShared {
  uint64_t warp[3][32];
};

__device__ inline void finalize_block(const ArrayView& v, const uint64_t* ins_base, const uint64_t* ins_len,
                               uint64_t* cp_prefix, uint32_t copy_chunk_elems, FinalizeShared& sh) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const int sums = cp_prefix ? 3 : 2;
  uint64_t run[3] = {0, 0, 0};
  uint32_t l0 = 0;
  while (l0 < v.L) {
    const uint32_t left = v.L - l0;
    const uint32_t per = min(static_cast<uint32_t>(kFinItems), (left + blockDim.x - 1) / blockDim.x);
    const uint32_t lt = l0 + threadIdx.x * per;   // this thread's LFVectors: lt .. lt + per - 1
    uint64_t x[3][kFinItems];
    uint64_t s[3] = {0, 0, 0};
#pragma unroll
    for (int i = 0; i < kFinItems; ++i) {
      const uint32_t l = lt + i;
      x[0][i] = x[1][i] = x[2][i] = 0;
      if (static_cast<uint32_t>(i) < per && l < v.L) {
        x[0][i] = __ldcg(v.sizes + l);
        if (cp_prefix) {
          const uint64_t b0 = __ldcg(ins_base + l), n = __ldcg(ins_len + l);
          x[2][i] = n ? (b0 + n - 1) / copy_chunk_elems - b0 / copy_chunk_elems + 1 : 0;
        }
      }
    }
#pragma unroll
    for (int i = 0; i < kFinItems; ++i) {
      x[1][i] = bucket_chunks(x[0][i], v.log2B, v.E);
#pragma unroll
      for (int q = 0; q < 3; ++q) s[q] += x[q][i];
    }
    uint64_t inc[3];
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      inc[q] = q < sums ? warp_incl_scan(s[q]) : 0;
      if (lane == 31) sh.warp[q][warp] = inc[q];
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      if (q >= sums) break;
      const uint64_t y = lane < nw ? sh.warp[q][lane] : 0;
      const uint64_t yi = warp_incl_scan(y);
      uint64_t at = run[q] + __shfl_sync(0xffffffffu, yi - y, warp) + inc[q] - s[q];
      run[q] += __shfl_sync(0xffffffffu, yi, 31);
      uint64_t* out = q == 0 ? v.offsets : (q == 1 ? v.fl_prefix : cp_prefix);
#pragma unroll
      for (int i = 0; i < kFinItems; ++i) {
        if (static_cast<uint32_t>(i) < per && lt + i < v.L) out[lt + i] = at;
        at += x[q][i];
      }
    }
    l0 += per * blockDim.x < left ? per * blockDim.x : left;
    if (l0 < v.L) __syncthreads();   // the warp totals are read before the next sweep writes them
  }
  if (threadIdx.x == 0) {
    v.offsets[v.L] = run[0];
    v.fl_prefix[v.L] = run[1];
    if (cp_prefix) cp_prefix[v.L] = run[2];
  }
}


// ---------------------------------------------------------------------------
// Growth of one LFVector by rounds of in-thread insertions (the in-kernel
// push_back of Algorithm 1, positions from Sec. III-B's block prefix sum),
// K rounds per pass.  Shared by the generated insertion (one block per
// LFVector, a fixed number of rounds) and the batched growth (a persistent
// block per item, rounds until the LFVector's target).
//
// Per pass every thread draws its counts for K rounds (virtual threads
// t = t0 * kv + i, kv = ceil(T / blockDim) <= KV <= 4), the per-thread round
// sums are scanned two rounds per 32-bit word (sums < 2^16 per block: counts
// are below 64 and blockDim * KV * 63 < 2^16), warp 0 scans the warp totals and its
// lane 0 makes one size reservation for the pass -- clipped at `target`,
// and, if the pool cannot hold the buckets it reaches, cut back to the
// longest prefix of whole rounds that fits -- and takes the buckets
// (Algorithm 2); then (synchronize) the values go to a shared-memory stage
// at their positions and the block streams the stage to the buckets with
// aligned 128-bit stores (marked passes in as many parts as it takes, others SP
// rounds at a time; where those do not fit, straight to the buckets).  Elements past the target are the ones a round-by-round
// growth would clip (positions are round-major).  The LFVector's bucket
// table is kept in shared memory, so the write-out finds a bucket's
// address without a global load.

__device__ __forceinline__ uint32_t warp_incl_scan_u32(uint32_t v) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t n = __shfl_up_sync(0xffffffffu, v, o);
    if (lane >= o) v += n;
  }
  return v;
}

// Largest count a distribution draws (0 when it has no small bound).
template <int DIST>
__host__ __device__ constexpr uint32_t max_count() {
  return DIST == GGA_DIST_BERNOULLI ? 1u : (DIST == GGA_DIST_UNIFORM3 ? 2u : 0u);
}

// Threshold counts (ascending thresholds) per interval of 2^23 draws, in
// shared memory: entry i is {c_i, next_i}, c_i = #{k : thr[k] <= i * 2^23}
// and next_i the threshold after those if it lies inside the interval (else
// 2^32 - 1).  A draw u of interval i counts c_i + (u >= next_i): one table
// load and no branch, unless u reaches `second`, the least value at which
// that could be wrong (the second threshold inside some interval, or
// 2^32 - 1), where the thresholds are stepped over.  (Poisson(1): thr[6], one
// draw in 12,000; with 256 intervals it is thr[5], one in 1,700, and a warp
// of eight draws per thread takes the slow way every seventh time.)
struct ThresholdTable {
  static constexpr uint32_t kShift = 23, kEntries = 1u << (32 - kShift);
  uint32_t thr[GGA_MAX_THRESHOLDS];
  uint2 tab[kEntries];
  uint32_t second;

  // Fill from ascending g.thr[0 .. nthr) (every thread of the block; a
  // barrier must follow).
  __device__ __forceinline__ void fill(const GenParams& g, uint32_t t, uint32_t nt) {
    for (uint32_t i = t; i < GGA_MAX_THRESHOLDS; i += nt) thr[i] = g.thr[i];
    for (uint32_t i = t; i < kEntries; i += nt) {
      uint32_t c = 0;
      for (uint32_t k = 0; k < g.nthr; ++k) c += g.thr[k] <= (i << kShift) ? 1u : 0u;
      tab[i] = make_uint2(c, c < g.nthr && g.thr[c] >> kShift == i ? g.thr[c] : ~0u);
    }
    if (t == 0) {
      second = ~0u;
      for (uint32_t k = g.nthr; k-- > 1;)
        if (g.thr[k] >> kShift == g.thr[k - 1] >> kShift && (g.thr[k - 1] & ((1u << kShift) - 1u)) != 0)
          second = g.thr[k];
    }
  }

  // The count of a draw with high word u < second.
  __device__ __forceinline__ uint32_t first_count(uint32_t u) const {
    const uint2 e = tab[u >> kShift];
    return e.x + (u >= e.y ? 1u : 0u);
  }

  // #{k < nthr : u >= thr[k]} for the high word u of any draw.
  __device__ __forceinline__ uint32_t count(uint32_t nthr, uint32_t u) const {
    uint32_t c = first_count(u);   // (loaded whatever u is: no branch before it)
    if (u >= second) c = slow_count(nthr, u);
    return c;
  }

  __device__ __forceinline__ uint32_t slow_count(uint32_t nthr, uint32_t u) const {
    uint32_t c = 0;
    while (c < nthr && u >= thr[c]) ++c;
    return c;
  }
};

constexpr int kMaxCluster = 8;

struct GenShared {
  uint32_t wt[4][32];         // packed warp prefixes (K / 2 <= 4 words)
  uint32_t rb[9];             // pass-relative start of every round (K <= 8)
  uint64_t base;              // LFVector size before the pass
  uint32_t commit, nb;
  int stop;                   // 1: pool exhausted, 2: target reached
  uint64_t tab[kMaxBuckets];  // the LFVector's bucket table (copy)
  ThresholdTable thr;
  // Clusters only, written by the peers: the blocks' pass totals (by pass
  // parity) and the allocated buckets after a growth.
  uint32_t peer_total[2][kMaxCluster];
  uint32_t peer_nb;
  uint32_t rounds;            // rounds the cluster's next pass takes
};

// Rounds a cluster's pass takes: its C K, or as many as the `rem` elements up
// to the target should need (a draw's mean and four deviations of their sum;
// if they do not suffice, another pass follows).  Blocks with none of them
// draw nothing.  (Without it the last pass draws half its rounds for nothing,
// an eighth of what a chain of 16 single passes draws.)
__device__ __forceinline__ uint32_t pass_rounds(uint64_t rem, float per_round, uint32_t most) {
  const float r = static_cast<float>(rem);
  const float n = (r + 4.0f * sqrtf(r)) / per_round + 1.0f;   // (a mean of zero: inf)
  return n < static_cast<float>(most) ? static_cast<uint32_t>(n) : most;
}

// Thread-block cluster operations (the blocks of a cluster are co-resident,
// so their barrier always completes).
__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}

__device__ __forceinline__ void cluster_barrier() {
  __syncwarp();
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// Store x to block `rank`'s copy of this block's shared variable *p.
__device__ __forceinline__ void cluster_store(uint32_t* p, uint32_t rank, uint32_t x) {
  uint32_t a;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(smem_u32(p)), "r"(rank));
  asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(a), "r"(x) : "memory");
}

// *p = x in shared memory if `cond`, as a predicated store.  (As an `if` the
// generated insertion of 4-byte uniform counts took 53.5 instructions per
// draw against 49.9, 80 us against 72 for 2^25 draws on GB300.)
template <int E>
__device__ __forceinline__ void store_shared_if(typename Elem<E>::T* p, typename Elem<E>::T x, bool cond) {
  const uint32_t a = smem_u32(p), c = cond ? 1u : 0u;
  if constexpr (E == 4) {
    asm volatile("{.reg .pred q; setp.ne.u32 q, %2, 0; @q st.shared.u32 [%0], %1;}" ::"r"(a), "r"(x), "r"(c) : "memory");
  } else if constexpr (E == 8) {
    asm volatile("{.reg .pred q; setp.ne.u32 q, %2, 0; @q st.shared.u64 [%0], %1;}" ::"r"(a), "l"(x), "r"(c) : "memory");
  } else {
    asm volatile("{.reg .pred q; setp.ne.u32 q, %5, 0; @q st.shared.v4.u32 [%0], {%1, %2, %3, %4};}" ::"r"(a), "r"(x.x),
                 "r"(x.y), "r"(x.z), "r"(x.w), "r"(c)
                 : "memory");
  }
}

// Marks.  A thread whose counts have no small bound would store its elements
// one by one in a loop that runs as often as the largest count of its warp,
// most lanes idle, and compute every value there.  Such a pass stages one
// 32-bit mark per non-empty draw instead, at its first element's place:
// (word + 1) << 13 | (round of the pass << 10) | (virtual thread), word being
// the mark's index in the stage.  Marks grow with the place, so the draw an
// element belongs to is the largest mark at or before it: a running maximum,
// which the write-out takes with a warp scan and from which every lane computes
// its own elements' values.  Words with no mark hold zero.  Measured on GB300
// for 2^25 draws (1024 LFVectors x 512 threads), elements stored in loops / by
// marks: geometric counts 219 / 117 us (4 bytes), 378 / 133 (8), 337 / 157
// (16); Poisson 216 / 125, 278 / 139, 296 / 161.
//
// A pass of more elements than the stage holds (counts with a mean above the
// one it is sized for) is written in parts, one stage after another: each has
// the marks of its own stretch and of the kMarkHalo places before it, as a draw
// has at most 63 elements.
constexpr uint32_t kMarkBits = 13;   // 3 of the round, 10 of the virtual thread
constexpr uint32_t kMarkHalo = 64;   // words before a part's first element
constexpr uint32_t kMarkMaxStage = (1u << (32 - kMarkBits)) - kMarkHalo - 2u;
// Consecutive elements of a lane in a step of the write-out: as many as its
// 128-bit stores still cover whole 32-byte sectors with.  (Four records a
// lane: 197 us against 161 for 2^25 draws on GB300.)
constexpr uint32_t mark_group(int E) { return E == 16 ? 2 : 4; }

// Writes n marked elements (places shv .. shv + n - 1, position base at shv, shv
// = base mod mark_group(E); place i's mark is word kMarkHalo + i) to their
// buckets; all threads of the block, after a barrier that follows the marks.
// Element m of draw (k, vt) is v0 + va * vt + vb * k + vc * m.  A warp
// takes a contiguous span of each bucket's part, a lane mark_group(E)
// consecutive elements at a time.
template <int E, typename V>
__device__ __forceinline__ void marks_to_buckets(const uint64_t* tab, uint32_t log2B, uint64_t base, uint32_t n,
                                                 uint32_t shv, const uint32_t* words, V v0, V va, V vb, V vc,
                                                 uint32_t t, uint32_t nt) {
  typedef typename Elem<E>::T T;
  constexpr uint32_t G = mark_group(E);
  const uint32_t lane = t & 31, warp = t >> 5, nw = nt >> 5;
  const uint64_t gbeg = base - shv;
  const uint32_t end = n + shv;
  const uint32_t* const marks = words + kMarkHalo;
  for (uint32_t s0 = 0; s0 < end;) {       // block-uniform: the part in one bucket
    uint32_t bb;
    uint64_t off;
    bucket_of(gbeg + s0, log2B, bb, off);
    const uint64_t room = bucket_len(bb, log2B) - off;
    const uint32_t s1 = room < end - s0 ? s0 + static_cast<uint32_t>(room) : end;
    T* const dst = reinterpret_cast<T*>(tab[bb] + off * sizeof(T));   // element s0's place
    const uint32_t steps = (s1 - s0 + 32 * G - 1) / (32 * G), per = (steps + nw - 1) / nw;
    uint32_t c = s0 + warp * per * (32 * G);
    const uint32_t cend = min(s1, c + per * (32 * G));
    // The last mark before the span: a draw has at most 63 elements, so it
    // lies within the 64 places before (or there is none: the run's start).
    uint32_t carry = 0;
    if (c < cend) {
#pragma unroll
      for (uint32_t back = 0; back < kMarkHalo; back += 32) {
        const uint32_t w = words[c + (kMarkHalo - 1) - back - lane];
        if (carry == 0) carry = __reduce_max_sync(0xffffffffu, w);
      }
    }
    for (; c < cend; c += 32 * G) {        // warp-uniform
      const uint32_t si = c + lane * G;
      uint32_t w[G];
      if constexpr (G == 4) {
        const uint4 x = *reinterpret_cast<const uint4*>(marks + si);
        w[0] = x.x; w[1] = x.y; w[2] = x.z; w[3] = x.w;
      } else {
        const uint2 x = *reinterpret_cast<const uint2*>(marks + si);
        w[0] = x.x; w[1] = x.y;
      }
#pragma unroll
      for (uint32_t e = 1; e < G; ++e) w[e] = max(w[e], w[e - 1]);
      uint32_t inc = w[G - 1];
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) inc = max(inc, __shfl_up_sync(0xffffffffu, inc, o));   // own value below lane o
      uint32_t ex = __shfl_up_sync(0xffffffffu, inc, 1);
      if (lane == 0) ex = 0;
      ex = max(ex, carry);
      carry = max(carry, __shfl_sync(0xffffffffu, inc, 31));
      if (si >= s1) continue;
      union {
        T e[G];
        uint4 q[sizeof(T) * G / 16];
      } x;
#pragma unroll
      for (uint32_t e = 0; e < G; ++e) {
        const uint32_t m = max(w[e], ex);
        x.e[e] = gen_value<E>(v0 + va * static_cast<V>(m & 1023u) + vb * static_cast<V>((m >> 10) & 7u) +
                              vc * static_cast<V>(si + e + (kMarkHalo + 1) - (m >> kMarkBits)));
      }
      T* const p = dst + (si - s0);
      if (si >= shv && si + G <= s1) {
#pragma unroll
        for (uint32_t i = 0; i < sizeof(T) * G / 16; ++i) __stcs(reinterpret_cast<uint4*>(p) + i, x.q[i]);
      } else {
#pragma unroll
        for (uint32_t e = 0; e < G; ++e)
          if (si + e >= shv && si + e < s1) p[e] = x.e[e];
      }
    }
    s0 = s1;
  }
}

// Zero for marks[0 .. n), by all threads of the block.
__device__ __forceinline__ void clear_marks(uint4* marks4, uint32_t n, uint32_t t, uint32_t nt) {
  for (uint32_t i = t; i < (n + 3) / 4; i += nt) marks4[i] = make_uint4(0, 0, 0, 0);
}

// Returns the number of rounds it drew; *done is set when the LFVector
// reached `target` or the pool ran out.  Every thread of the block calls
// it.  DIST as for gen_count_state (-1: g.dist at run time).
//
// C > 1: the C blocks of a cluster grow the LFVector together, block q of a
// pass drawing its rounds q K .. q K + K - 1 of the pass's C K (the last pass
// takes fewer: pass_rounds).  The blocks
// store their totals into one another's shared memory, one cluster barrier
// takes the place of the pass's second block barrier, and every block then
// knows where its run starts and whether the pass stays inside the allocated
// buckets; only when it does not, block 0 allocates behind a second cluster
// barrier.  Draws, positions, clipping and the rounds kept when the pool
// runs out are those of one block drawing the same rounds one after another.
template <int E, int K, int KV, int DIST = -1, int C = 1, int SP = K, bool SKIP = false>
__device__ uint32_t grow_passes(const ArrayView& v, const GenParams& g, uint32_t l, uint32_t R, uint64_t target,
                                GenShared& sh, uint4* stage4, uint32_t cap, bool* done) {
  typedef typename Elem<E>::T T;
  constexpr uint32_t VEC = 16 / E;
  constexpr int KP = K / 2;
  static_assert(K % 2 == 0 && K <= 8, "K rounds per pass: even, at most 8");
  static_assert(KV == 1 || KV == 4, "a round's counts in one word");
  T* stage = reinterpret_cast<T*>(stage4);
  const uint32_t t0 = threadIdx.x, NT = blockDim.x;
  const int lane = t0 & 31, warp = t0 >> 5, nwarps = NT >> 5;
  const uint32_t kv = KV == 1 ? 1u : (v.T + NT - 1) / NT;
  const uint64_t tfirst = static_cast<uint64_t>(t0) * kv;        // first virtual thread
  const uint32_t nvt = tfirst < v.T ? min(kv, v.T - static_cast<uint32_t>(tfirst)) : 0u;   // virtual threads played
  const uint32_t played = nvt >= 4 ? ~0u : (1u << (8 * nvt)) - 1u;   // a byte of ones per virtual thread
  const uint64_t gfirst = static_cast<uint64_t>(l) * v.T + tfirst;
  const uint64_t* bk = v.buckets + static_cast<uint64_t>(l) * kMaxBuckets;
  RoundDraws dv[KV];   // virtual threads gfirst, ..., gfirst + KV - 1
#pragma unroll
  for (int i = 0; i < KV; ++i) dv[i] = RoundDraws(g.seed, gfirst + i);
  if (t0 == 0) {
    sh.base = v.sizes[l];
    sh.nb = v.nbuckets[l];
    sh.stop = sh.base >= target ? 2 : 0;
    if constexpr (C > 1) sh.rounds = pass_rounds(target - sh.base, g.mean * static_cast<float>(v.T), C * K);
  }
  {
    const uint32_t nb0 = v.nbuckets[l];
    for (uint32_t i = t0; i < nb0; i += NT) sh.tab[i] = bk[i];
  }
  const bool tabled = DIST == GGA_DIST_POISSON && g.thr_sorted;   // uniform
  if (tabled) sh.thr.fill(g, t0, NT);
  __syncthreads();
  const uint32_t rank = C > 1 ? cluster_rank() : 0u;
  uint32_t par = 0;
  // Counts without a small bound are staged as marks (buckets must hold a
  // lane's group); `dirty` marks of the last pass are still set.
  constexpr bool kMarks = !(DIST >= 0 && max_count<DIST>() > 0 && max_count<DIST>() <= 2);
  constexpr uint32_t kGroup = mark_group(E);
  uint32_t* const words = reinterpret_cast<uint32_t*>(stage4);
  // Elements a part holds: whole groups, beside the halo and the 32 groups that a
  // warp's last step of the write-out reads past the end.
  const uint32_t part =
      v.B < kGroup ? 0u : min(cap * static_cast<uint32_t>(E / 4) - kMarkHalo - 32 * kGroup, kMarkMaxStage) & ~(kGroup - 1u);
  uint32_t dirty = 0;
  if (kMarks) clear_marks(stage4, cap * (E / 4), t0, NT);   // (the pass's barriers come before the first mark)
  uint32_t r0 = 0;   // the pass's first round
  while (r0 < R && sh.stop == 0) {
    const uint32_t rb0 = r0 + rank * K;   // this block's first round of the pass
    const uint32_t rend = C > 1 ? r0 + min(R - r0, sh.rounds) : R;   // rounds before this one are drawn
    const uint32_t kk = rb0 < rend ? min(static_cast<uint32_t>(K), rend - rb0) : 0u;
    // exw: the thread's offsets in its warp, two rounds per word; cw: its
    // counts, one byte each (round k, virtual thread i at byte k * KV + i).
    constexpr int KC = (K * KV + 3) / 4;
    uint32_t exw[KP], cw[KC];
#pragma unroll
    for (int q = 0; q < KC; ++q) cw[q] = 0;
    auto count_of = [&](uint32_t k, uint32_t i) { return (cw[(k * KV + i) / 4] >> (8 * ((k * KV + i) % 4))) & 0xFFu; };
    // G rounds at a time, virtual thread by virtual thread: all its draws of the
    // G rounds are made, and masked a round at a time (a branch or a test around
    // every draw costs more than the draws of the threads and rounds past the
    // end).  kSkip: virtual threads that no thread of the block plays are left
    // out, for a test per virtual thread and all rounds together (SKIP: batches,
    // whose blocks are not sized by T and whose g lives in shared memory).  Elsewhere bounded counts take two
    // rounds at a time (paper-shaped workload, flatten included: 837 us, with the
    // test 845, with the test and two rounds 855).
    constexpr bool kSkip = SKIP || kMarks;
    constexpr int G = KV == 1 || !kSkip ? 2 : K;
#pragma unroll
    for (int k0 = 0; k0 < K; k0 += G) {
      uint32_t w[G];   // a round's counts, one byte per virtual thread
#pragma unroll
      for (int h = 0; h < G; ++h) w[h] = 0;
      const uint64_t r1 = static_cast<uint64_t>(g.round0) + rb0 + k0;
#pragma unroll
      for (int i = 0; i < KV; ++i) {
        if (kSkip && ((i > 0 && static_cast<uint32_t>(i) >= kv) || (C > 1 && kk == 0))) break;   // block-uniform
        uint32_t top = 0;
#pragma unroll
        for (int h = 0; h < G; ++h) {
          uint32_t ci;
          if (DIST == GGA_DIST_POISSON && tabled) {
            const uint32_t u = splitmix_mix_hi(dv[i].state(r1 + h));
            top = max(top, u);
            ci = sh.thr.first_count(u);
          } else {
            ci = gen_count_state<SKIP, DIST>(g, dv[i].state(r1 + h));
          }
          w[h] |= ci << (8 * i);
        }
        if (DIST == GGA_DIST_POISSON && tabled && top >= sh.thr.second) {
          // A draw among the thresholds the table does not tell apart: the
          // virtual thread's draws again, threshold by threshold.
          uint64_t all = 0;
#pragma unroll 1
          for (uint32_t h = 0; h < G; ++h)
            all |= static_cast<uint64_t>(sh.thr.slow_count(g.nthr, splitmix_mix_hi(dv[i].state(r1 + h)))) << (8 * h);
#pragma unroll
          for (int h = 0; h < G; ++h)
            w[h] = (w[h] & ~(0xFFu << (8 * i))) | (static_cast<uint32_t>(all >> (8 * h)) & 0xFFu) << (8 * i);
        }
      }
#pragma unroll
      for (int j2 = 0; j2 < G / 2; ++j2) {
        uint32_t pk = 0;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const uint32_t k = k0 + 2 * j2 + h, x = w[2 * j2 + h] & (k < kk ? played : 0u);
          cw[k * KV / 4] |= x << (8 * (k * KV % 4));
          pk |= (KV == 1 ? x : __dp4a(x, 0x01010101u, 0u)) << (16 * h);
        }
        const uint32_t inc = warp_incl_scan_u32(pk);
        exw[k0 / 2 + j2] = inc - pk;
        if (lane == 31) sh.wt[k0 / 2 + j2][warp] = inc;
      }
    }
    __syncthreads();
    if (kMarks) clear_marks(stage4, dirty, t0, NT);   // the last pass's write-out is over
    if (warp == 0) {
      uint32_t rb = 0;
#pragma unroll
      for (int j = 0; j < KP; ++j) {
        const uint32_t w = lane < nwarps ? sh.wt[j][lane] : 0u;
        const uint32_t wi = warp_incl_scan_u32(w);
        if (lane < nwarps) sh.wt[j][lane] = wi - w;
        const uint32_t tot = __shfl_sync(0xffffffffu, wi, 31);
        if (lane == 0) {
          sh.rb[2 * j] = rb;
          rb += tot & 0xFFFFu;
          sh.rb[2 * j + 1] = rb;
          rb += tot >> 16;
        }
      }
      if constexpr (C > 1) {
        if (lane == 0) sh.rb[K] = rb;
        rb = __shfl_sync(0xffffffffu, rb, 0);
        if (lane < C) cluster_store(&sh.peer_total[par][rank], lane, rb);
      } else if (lane == 0) {
        sh.rb[K] = rb;
        const uint64_t base = sh.base;
        const uint64_t rem = target - base;   // > 0 while the loop runs
        uint32_t commit = rb < rem ? rb : static_cast<uint32_t>(rem);
        if (commit > 0) {
          const uint32_t nb = sh.nb;
          const uint32_t need = buckets_for(base + commit, v.log2B);
          if (need > nb) {
            const uint32_t got = grow_buckets(v, l, nb, need);
            for (uint32_t i = nb; i < got; ++i) sh.tab[i] = bk[i];
            sh.nb = got;
            v.nbuckets[l] = got;
            if (got < need) {
              const uint64_t capg = bucket_first(got, v.log2B);
              int kf = 0;
              while (kf < K && base + sh.rb[kf + 1] <= capg) ++kf;
              if (sh.rb[kf] < commit) commit = sh.rb[kf];
              sh.stop = 1;
              latch_error(v.status, GGA_ERR_POOL_EXHAUSTED);
            }
          }
        }
        if (sh.stop == 0 && base + commit >= target) sh.stop = 2;
        sh.commit = commit;
        v.sizes[l] = base + commit;
      }
    }
    uint64_t base;     // position of this block's first element of the pass
    uint32_t commit;   // elements of this block the pass keeps
    uint64_t next;     // the LFVector's size after the pass
    if constexpr (C > 1) {
      cluster_barrier();   // every block's total is here; this block's scan too
      const uint64_t size = sh.base, rem = target - size;
      uint32_t pre = 0, sum = 0;
#pragma unroll
      for (uint32_t q = 0; q < C; ++q) {
        const uint32_t tq = sh.peer_total[par][q];
        if (q < rank) pre += tq;
        sum += tq;
      }
      par ^= 1u;
      const uint32_t kept = sum < rem ? sum : static_cast<uint32_t>(rem);
      const uint32_t mine = sh.rb[K];
      commit = pre >= kept ? 0u : min(mine, kept - pre);
      base = size + pre;
      next = size + kept;
      const uint32_t nb = sh.nb;
      const uint32_t need = kept ? buckets_for(next, v.log2B) : 0u;
      bool full = false;
      if (need > nb) {   // the same in every thread of the cluster
        if (rank == 0 && t0 == 0) {
          const uint32_t got = grow_buckets(v, l, nb, need);
          v.nbuckets[l] = got;
          for (uint32_t q = 0; q < C; ++q) cluster_store(&sh.peer_nb, q, got);
        }
        cluster_barrier();   // synchronize(): the buckets exist before any write
        const uint32_t got = sh.peer_nb;
        for (uint32_t i = nb + t0; i < got; i += NT) sh.tab[i] = __ldcg(bk + i);
        full = got < need;
        if (full) {          // keep the longest prefix of whole rounds that fits
          const uint64_t capg = bucket_first(got, v.log2B);
          uint32_t kf = 0;
          while (kf < static_cast<uint32_t>(K) && base + sh.rb[kf + 1] <= capg) ++kf;
          commit = base > capg ? 0u : min(commit, sh.rb[kf]);
          if (t0 == 0) {
            if (commit) atomicMax(reinterpret_cast<unsigned long long*>(v.sizes + l), base + commit);
            if (rank == 0) latch_error(v.status, GGA_ERR_POOL_EXHAUSTED);
          }
        }
        __syncthreads();     // the table is filled, and every thread has read sh.nb
        if (t0 == 0) sh.nb = got;
      }
      if (t0 == 0) {         // read by the others after the stage's barrier
        if (rank == 0 && !full) v.sizes[l] = next;
        sh.stop = full ? 1 : (next >= target ? 2 : 0);
        sh.rounds = pass_rounds(target - next, g.mean * static_cast<float>(v.T), C * K);
      }
    } else {
      __syncthreads();   // synchronize(): the buckets exist before any write
      base = sh.base;
      commit = sh.commit;
      next = base + commit;
    }
    const bool marked = kMarks && part > 0;
    // Fast path (block-uniform): the whole pass is kept and staged, SP rounds at
    // a time, so no element needs the clipping test or the bucket math.
    bool whole = !kMarks && commit == sh.rb[K];
#pragma unroll
    for (int k = 0; k < K; k += SP) whole = whole && sh.rb[k + SP] - sh.rb[k] + VEC - 1 <= cap;
    typedef typename std::conditional<E == 4, uint32_t, uint64_t>::type V;
    if (marked) {
      // Place (stage index) = pass position + shv.
      const uint32_t shv = static_cast<uint32_t>(base & (kGroup - 1));
      const uint32_t end = commit + shv, most = sh.rb[K] + shv;
      // More than one part: the thread's offsets and counts in local memory, so
      // that no register holds them over the write-out of a part.
      uint32_t lex[KP], lcw[KC];
      if (most <= part) {
#pragma unroll
        for (int j = 0; j < KP; ++j) {
          const uint32_t ex = sh.wt[j][warp] + exw[j];
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const uint32_t k = 2 * j + h;
            uint32_t at = sh.rb[k] + ((ex >> (16 * h)) & 0xFFFFu) + shv + kMarkHalo;
#pragma unroll
            for (int i = 0; i < KV; ++i) {
              if (i > 0 && static_cast<uint32_t>(i) >= kv) break;
              const uint32_t c = count_of(k, i);
              if (c) words[at] = ((at + 1) << kMarkBits) + ((k << 10) + static_cast<uint32_t>(tfirst) + i);
              at += c;
            }
          }
        }
      } else {
#pragma unroll
        for (int j = 0; j < KP; ++j) lex[j] = sh.wt[j][warp] + exw[j];
#pragma unroll
        for (int q = 0; q < KC; ++q) lcw[q] = cw[q];
      }
      for (uint32_t lo = 0;;) {   // one part after another, mostly one
        if (most > part) {
#pragma unroll 1
          for (uint32_t k = 0; k < K && sh.rb[k] + shv < lo + part; ++k) {
            if (sh.rb[k + 1] + shv + kMarkHalo <= lo) continue;   // block-uniform, as the loop's end: rounds of this part
            const uint32_t w = lcw[k * KV / 4] >> (8 * (k * KV % 4));
            uint32_t at = sh.rb[k] + ((lex[k / 2] >> (16 * (k % 2))) & 0xFFFFu) + shv + kMarkHalo - lo;
#pragma unroll
            for (int i = 0; i < KV; ++i) {
              const uint32_t c = (w >> (8 * i)) & 0xFFu;
              if (c && at < part + kMarkHalo)
                words[at] = ((at + 1) << kMarkBits) + ((k << 10) + static_cast<uint32_t>(tfirst) + i);
              at += c;
            }
          }
        }
        __syncthreads();
        const uint32_t at0 = lo ? 0u : shv;
        if (commit)
          marks_to_buckets<E, V>(sh.tab, v.log2B, base - shv + lo + at0, min(part, end - lo) - at0, at0, words,
                                 static_cast<V>(g.va * (static_cast<uint64_t>(l) * v.T) +
                                                g.vb * (static_cast<uint64_t>(g.round0) + rb0)),
                                 static_cast<V>(g.va), static_cast<V>(g.vb), static_cast<V>(g.vc), t0, NT);
        lo += part;
        if (lo >= end) break;
        __syncthreads();   // the part is written out
        clear_marks(stage4, kMarkHalo + part, t0, NT);
        __syncthreads();
      }
      dirty = kMarkHalo + min(most, part);
    } else {
      // Element m of virtual thread i in round k: va * gid + vb * round + vc * m
      // (a 4-byte element keeps the low 32 bits, which 32-bit arithmetic gives
      // exactly).
      // The value parameters in registers: g may live in shared memory, where
      // the stage stores below could alias it and force a reload per element.
      const V va = static_cast<V>(g.va), vb = static_cast<V>(g.vb), vc = static_cast<V>(g.vc);
      const V vr = va * static_cast<V>(gfirst) + vb * static_cast<V>(static_cast<uint64_t>(g.round0) + rb0);
      if (whole) {
#pragma unroll
        for (int k0 = 0; k0 < K; k0 += SP) {
          const uint32_t first = sh.rb[k0], n = sh.rb[k0 + SP] - first;
          const uint32_t at = static_cast<uint32_t>(base + first) & (VEC - 1);
          if (k0 > 0) __syncthreads();   // the part before is written out
#pragma unroll
          for (int k = k0; k < k0 + SP; ++k) {
            const uint32_t ex = sh.wt[k / 2][warp] + exw[k / 2];
            T* st = stage + (sh.rb[k] - first + at + ((ex >> (16 * (k % 2))) & 0xFFFFu));
            const V v0 = vr + vb * static_cast<V>(k);
#pragma unroll
            for (int i = 0; i < KV; ++i) {
              const uint32_t c = count_of(k, i);
              V val = v0 + va * static_cast<V>(i);
              // At most two elements: predicated stores, no loop.
              store_shared_if<E>(st, gen_value<E>(val), c > 0);
              if (max_count<DIST>() > 1) store_shared_if<E>(st + 1, gen_value<E>(val + vc), c > 1);
              st += c;
            }
          }
          __syncthreads();
          if (n) stage_to_buckets<T>(sh.tab, v.log2B, v.B, base + first, n, at, stage4, t0, NT);
        }
      } else {
        // A clipped pass, or one that does not fit: SP rounds after SP rounds,
        // element by element, straight to the buckets where they do not fit.
        uint32_t lex[KP], lcw[KC];
#pragma unroll
        for (int j = 0; j < KP; ++j) lex[j] = sh.wt[j][warp] + exw[j];
#pragma unroll
        for (int q = 0; q < KC; ++q) lcw[q] = cw[q];
        dirty = 0;
        uint32_t k = 0;
#pragma unroll 1
        do {
          const uint32_t first = sh.rb[k], n = first < commit ? min(sh.rb[k + SP], commit) - first : 0u;
          const uint32_t at = static_cast<uint32_t>(base + first) & (VEC - 1);
          const bool staged = n + at <= cap;
          if (k > 0) __syncthreads();   // the part before is written out
#pragma unroll 1
          for (const uint32_t kend = k + SP; k < kend; ++k) {
            uint32_t q = sh.rb[k] - first + ((lex[k / 2] >> (16 * (k % 2))) & 0xFFFFu);
#pragma unroll 1
            for (uint32_t i = 0; i < kv; ++i) {
              const uint32_t c = (lcw[(k * KV + i) / 4] >> (8 * ((k * KV + i) % 4))) & 0xFFu;
              V val = vr + va * static_cast<V>(i) + vb * static_cast<V>(k);
              for (uint32_t m = 0; m < c; ++m, ++q, val += vc) {
                if (q >= n) continue;
                if (staged) {
                  stage[q + at] = gen_value<E>(val);
                } else {
                  uint32_t bb;
                  uint64_t off;
                  bucket_of(base + first + q, v.log2B, bb, off);
                  reinterpret_cast<T*>(sh.tab[bb])[off] = gen_value<E>(val);
                }
              }
            }
          }
          __syncthreads();
          if (staged && n) {
            stage_to_buckets<T>(sh.tab, v.log2B, v.B, base + first, n, at, stage4, t0, NT);
            dirty = max(dirty, (n + at) * static_cast<uint32_t>(E / 4));
          }
        } while (k < K && sh.rb[k] < commit);
      }
    }
    // No barrier here: the next pass writes the stage, sh.wt, sh.rb and
    // sh.commit only after its first two barriers, which every thread reaches
    // after finishing this pass; sh.base is written by thread 0 and read by
    // thread 0 (the leader) before the next pass's second barrier and by the
    // others after it; sh.stop was set before this pass's second barrier;
    // sh.tab only gains entries past those this pass reads.
    if (t0 == 0) sh.base = next;
    if constexpr (C > 1) r0 = rend;
    else r0 = R - r0 > static_cast<uint32_t>(K) ? r0 + K : R;
  }
  *done = sh.stop != 0;
  __syncthreads();   // the caller may reuse the stage and sh
  return r0;
}

}  // namespace gga
