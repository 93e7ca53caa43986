// aggregate.cu — decompress and sum n workers' sparse vectors (the exchange
// step of Algorithm 1, Delta_bar = (1/n) sum_i Delta_i, without the 1/n).
//
// Deterministic by construction: the dense range [0, d) is cut into tiles of
// kAggTile coordinates; one CTA owns a tile in shared memory, starts it at
// +0.0f and adds worker 0's pairs, then worker 1's, ..., with a CTA barrier
// between workers. Within one worker the indices are distinct (the lists are
// strictly ascending), so no two threads add to the same slot at once, and
// every coordinate receives its contributions in ascending worker order —
// the same fp32 sum as the plain sequential loop.
//
// Kernel 1 finds where each worker's sorted list crosses each tile boundary
// (not needed when the messages come with their tile indexes); kernel 2 does
// the reduction and writes each dense tile once with 16-byte stores: a CTA per
// tile as above, or for a plain sum of up to 32 workers over many tiles one
// warp per tile (agg_stream_kernel), where worker order needs no barriers.
// Traffic: 8 B per pair read + 4 B per coordinate written (+ the small offsets
// table).
//
// The same reduction can instead end in the model update that follows the
// exchange (sparse_aggregate_apply): Delta' = alpha * s rounded once, then
// x <- x - Delta' (Algorithm 1), or m <- fmaf(mu, m, Delta') and
// x <- fmaf(-lr, Delta' + m, x) (the Appendix's EF SGD with momentum by
// gradient compression). The dense sum then never reaches memory: 8 B per
// coordinate (read and write x), 16 B with momentum, instead of writing the
// sum and a second pass that reads it back.
#include <algorithm>
#include <cstddef>

#include "agg_rule.h"
#include "internal.h"
#include "tma.cuh"

namespace efs {
namespace {

// The lists, passed as kernel parameters: 768 bytes for up to 32 workers, 6 KB
// for more (a launch copies its parameters: an exchange of 4 lists took the
// host 5.3 us with the large form).
constexpr uint32_t kFewWorkers = 32;
template <uint32_t kCap>
struct AggPtrs {
  const uint32_t* idx[kCap];
  const float* val[kCap];
  const uint32_t* tiles[kCap];  // the lists' tile indexes, when the caller has them
};

// off[i * (tiles + 1) + t] = number of entries of list i below t * kAggTile;
// off[i * (tiles + 1) + tiles] = counts[i]. Grid: blockIdx.y = list, x over
// the tiles + 1 entries. Two ways to the same numbers (agg_rule.h):
//  - scattered, when this list holds up to kScatterPerTile entries a tile, or
//    the lists at most kScatterEntries together, and this one at least
//    (tiles + 1) / 16: entry p (p = 0..count, count standing for the end) owns
//    the tiles t with list[p - 1] < t * kAggTile <= list[p] and writes p
//    there. A thread reads 4 consecutive entries and the one before them,
//    nothing waits for anything else; a run of more than 8 tiles is written by
//    the whole warp;
//  - otherwise one binary search per tile (14-23 dependent loads, but
//    independent of the lists' length).
// Either way every entry lies in [0, count]; a list that is not strictly
// ascending is latched as bad input (scatter) and may leave entries the
// reduction clamps to the list. A strictly ascending list below d has at most
// d entries: a larger count is latched, and nothing past d entries is read.
template <uint32_t kCap>
__global__ void __launch_bounds__(kThreads)
    agg_offsets_kernel(AggPtrs<kCap> p, const uint32_t* __restrict__ counts, uint32_t n,
                       uint32_t d, uint32_t tiles, uint32_t* __restrict__ off,
                       uint32_t* __restrict__ error) {
  griddep_wait();                // the lists and counts come from the kernels before
  griddep_launch_dependents();    // the reduction may be scheduled (it waits for this grid)
  const uint32_t per = tiles + 1;
  const uint32_t i = blockIdx.y;
  const uint32_t stride = gridDim.x * kThreads;  // >= per
  const int lane = threadIdx.x & 31;
  uint32_t all = 0;  // entries of all lists
  for (uint32_t q = lane; q < n; q += 32) all += scatter_share(counts[q]);
  all = warp_sum(all);
  const uint32_t cnt = min(counts[i], d);
  if (counts[i] > d && blockIdx.x == 0 && threadIdx.x == 0) atomicOr(error, kDevErrBadInput);
  const uint32_t* x = p.idx[i];
  uint32_t* o = off + static_cast<uint64_t>(i) * per;
  if (!scatter_offsets(cnt, all, per)) {
    // an equal run of the tiles for every CTA: the grid is as wide as the
    // scatter wants it, and with 256 searches in each of the first CTAs, which
    // tend to share SMs, those SMs' loads took 20 us more (16 lists of 20 % over
    // 2,728 tiles, update 190.8 us a call, this way 163)
    const uint32_t run = (per + gridDim.x - 1) / gridDim.x;  // at most kThreads
    const uint32_t t = blockIdx.x * run + threadIdx.x;
    if (threadIdx.x >= run || t >= per) return;
    uint32_t result = cnt;
    if (t < tiles) {
      const uint64_t target = static_cast<uint64_t>(t) * kAggTile;
      uint32_t lo = 0, hi = cnt;
      while (lo < hi) {
        const uint32_t mid = lo + (hi - lo) / 2;
        if (static_cast<uint64_t>(__ldg(x + mid)) < target)
          lo = mid + 1;
        else
          hi = mid;
      }
      result = lo;
    }
    o[t] = result;
    return;
  }
  bool bad = false;
  const bool vec = (reinterpret_cast<uintptr_t>(x) & 15u) == 0;
  const uint32_t quads = cnt / 4 + 1;  // positions 0..cnt
#pragma unroll 1
  for (uint32_t g0 = blockIdx.x * kThreads + (threadIdx.x & ~31u); g0 < quads; g0 += stride) {
    const uint32_t p0 = (g0 + lane) * 4;
    uint32_t v[5];  // the entry before p0, then entries p0 .. p0 + 3
    v[0] = p0 > 0 && p0 <= cnt ? __ldg(x + p0 - 1) : 0u;
    if (vec && p0 + 4 <= cnt) {
      const uint4 w = __ldg(reinterpret_cast<const uint4*>(x + p0));
      v[1] = w.x, v[2] = w.y, v[3] = w.z, v[4] = w.w;
    } else {
#pragma unroll
      for (int u = 0; u < 4; ++u) v[1 + u] = p0 + u < cnt ? __ldg(x + p0 + u) : 0u;
    }
    bool far = false;
    uint32_t t_lo[4], t_hi[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const uint32_t pos = p0 + u;
      t_lo[u] = pos == 0 ? 0u : min(v[u] / kAggTile + 1u, per);
      t_hi[u] = pos == cnt ? tiles : min(v[u + 1] / kAggTile, tiles - 1u);
      if (pos > cnt) t_lo[u] = t_hi[u] + 1;  // nothing
      if (pos > 0 && pos < cnt && v[u] >= v[u + 1]) bad = true;  // not strictly ascending
      if (t_lo[u] > t_hi[u]) continue;  // a shared tile (or malformed): nothing
      if (t_hi[u] - t_lo[u] < 8)
        for (uint32_t t = t_lo[u]; t <= t_hi[u]; ++t) o[t] = pos;
      else
        far = true;
    }
    if (!__any_sync(0xffffffffu, far)) continue;
#pragma unroll
    for (int u = 0; u < 4; ++u) {  // longer runs: the whole warp writes them, one after another
      uint32_t m = __ballot_sync(0xffffffffu, t_lo[u] <= t_hi[u] && t_hi[u] - t_lo[u] >= 8);
      while (m) {
        const int l = __ffs(m) - 1;
        m &= m - 1;
        const uint32_t a = __shfl_sync(0xffffffffu, t_lo[u], l);
        const uint32_t b = __shfl_sync(0xffffffffu, t_hi[u], l);
        const uint32_t pos = __shfl_sync(0xffffffffu, p0 + u, l);
        for (uint32_t t = a + lane; t <= b; t += 32) o[t] = pos;
      }
    }
  }
  if (bad) atomicOr(error, kDevErrBadInput);
}

// What the reduction does with a finished tile.
enum AggMode { kAggDense = 0, kAggSgd = 1, kAggMomentum = 2 };
struct AggOut {
  float* out;  // kAggDense: the sum; otherwise x, updated in place
  float* m;    // kAggMomentum: the momentum, updated in place
  float alpha, mu, lr;
};

template <int kMode>
__device__ __forceinline__ void apply_update(const AggOut& o, float s, float& x, float& m) {
  const float delta = __fmul_rn(o.alpha, s);
  if constexpr (kMode == kAggSgd) {
    x = __fsub_rn(x, delta);
  } else {
    m = __fmaf_rn(o.mu, m, delta);
    x = __fmaf_rn(-o.lr, __fadd_rn(delta, m), x);
  }
}

// 4-byte asynchronous copy global -> shared (no register staging).
__device__ __forceinline__ void cp_async_4(void* dst, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(
                   static_cast<uint32_t>(__cvta_generic_to_shared(dst))),
               "l"(src)
               : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() {
  asm volatile("cp.async.wait_all;" ::: "memory");
}

// Bulk prefetch of [p, p + bytes) into L2 (16-byte aligned, bytes % 16 == 0).
__device__ __forceinline__ void prefetch_l2_bulk(const void* p, uint32_t bytes) {
  asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(bytes) : "memory");
}

// kSearch: without offsets or tile indexes, for few tiles (kAggSearchTiles). A
// kernel of its own: with a run-time choice the check of the runs' order in
// the adding loop cost the others too (64 lists of 140 K pairs, d = 138.4 M, 655
// -> 685 us). It checks a stage at once: 64 lists of 1 %, d = 3.7 M, update,
// take 67.1 us without the check, 70.2 this way, 74.3 with it in the loop that
// adds worker by worker.
template <bool kVec, int kMode, uint32_t kCap, bool kSearch>
__global__ void __launch_bounds__(kThreads)
    agg_reduce_kernel(AggPtrs<kCap> p, uint32_t n, uint32_t d, uint32_t tiles,
                      const uint32_t* __restrict__ off, const uint32_t* __restrict__ counts,
                      AggOut o, uint32_t* __restrict__ error) {
  __shared__ __align__(16) float acc[kAggTile];
  __shared__ uint32_t s_lo[kCap], s_pre[kCap + 1];
  __shared__ uint32_t st_idx[kAggStage];
  __shared__ float st_val[kAggStage];
  const uint32_t t = blockIdx.x;
  const int lane = threadIdx.x & 31;
  const uint64_t j0 = static_cast<uint64_t>(t) * kAggTile;
  for (int q = threadIdx.x; q < kAggTile / 4; q += kThreads)
    reinterpret_cast<float4*>(acc)[q] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
  if constexpr (kMode != kAggDense) {
    // the tile's x (and m), read by the epilogue, on their way to L2 while
    // the pairs are gathered (a prefetch: no data moves into the CTA)
    if (kVec && threadIdx.x == 0 && j0 + kAggTile <= d) {
      prefetch_l2_bulk(o.out + j0, kAggTile * sizeof(float));
      if constexpr (kMode == kAggMomentum) prefetch_l2_bulk(o.m + j0, kAggTile * sizeof(float));
    }
  }
  griddep_wait();  // the offsets (and everything before them) are complete
  griddep_launch_dependents();  // the next kernel waits for this grid before its reads
  bool bad = false;
  if constexpr (kSearch) {
    // two threads per list search its run's ends. The last tile's run ends
    // with the list, so that indexes past every tile are in it, to be skipped
    // and latched.
    for (uint32_t q0 = 0; q0 < 2 * n; q0 += kThreads) {
      const uint32_t q = q0 + threadIdx.x, i = q >> 1;
      uint32_t at = 0;
      if (i < n) {
        const uint64_t target = (static_cast<uint64_t>(t) + (q & 1u)) * kAggTile;
        const uint32_t* x = p.idx[i];
        uint32_t hi = min(counts[i], d);  // a strictly ascending list holds no more
        bad |= counts[i] > d;
        if (t == tiles - 1 && (q & 1u)) at = hi;
        while (at < hi) {
          const uint32_t mid = at + (hi - at) / 2;
          if (static_cast<uint64_t>(__ldg(x + mid)) < target)
            at = mid + 1;
          else
            hi = mid;
        }
      }
      const uint32_t end = __shfl_down_sync(0xffffffffu, at, 1);
      if (i < n && !(q & 1u)) {
        s_lo[i] = at;
        s_pre[i + 1] = end > at ? end - at : 0u;
      }
    }
  } else {
    for (uint32_t i = threadIdx.x; i < n; i += kThreads) {
      // the list's range in this tile: from the offsets kernel, or from the
      // caller's tile index, clamped to the list (never out of bounds)
      const uint32_t* r = off ? off + static_cast<uint64_t>(i) * (tiles + 1) : p.tiles[i];
      const uint32_t cnt = counts[i];
      uint32_t lo = min(r[t], cnt), hi = min(r[t + 1], cnt);
      s_lo[i] = lo;
      s_pre[i + 1] = hi > lo ? hi - lo : 0u;  // this tile's pairs of worker i
    }
  }
  __syncthreads();
  if (threadIdx.x < 32) {  // s_pre: the tile's pairs of the workers before each one
    uint32_t carry = 0;
    for (uint32_t i0 = 0; i0 < n; i0 += 32) {
      const uint32_t i = i0 + lane;
      uint32_t v = i < n ? s_pre[i + 1] : 0u;
#pragma unroll
      for (int o2 = 1; o2 < 32; o2 <<= 1) {
        const uint32_t x = __shfl_up_sync(0xffffffffu, v, o2);
        if (lane >= o2) v += x;
      }
      if (i < n) s_pre[i + 1] = carry + v;
      carry += __shfl_sync(0xffffffffu, v, 31);
    }
    if (lane == 0) s_pre[0] = 0;
  }
  __syncthreads();
  const uint32_t total = s_pre[n];
  // The tile's pairs of all workers, in worker order, a stage at a time:
  // every copy of a stage is in flight at once (one round trip), then the
  // stage is added worker by worker, with a barrier between workers so that
  // each coordinate receives its contributions in worker order.
  for (uint32_t b0 = 0; b0 < total; b0 += kAggStage) {
    const uint32_t bn = total - b0 < kAggStage ? total - b0 : kAggStage;
    uint32_t inner = 0;  // kSearch: bit per pair of the thread: not a run's first
    uint32_t before = 0;  // thread 0: the index before the stage's first, of the same run
    {
      uint32_t i = 0, bit = 1;
      for (uint32_t q = threadIdx.x; q < bn; q += kThreads) {
        const uint32_t gp = b0 + q;
        while (s_pre[i + 1] <= gp) ++i;
        const uint32_t src = s_lo[i] + (gp - s_pre[i]);
        cp_async_4(st_idx + q, p.idx[i] + src);
        cp_async_4(st_val + q, p.val[i] + src);
        if constexpr (kSearch) {
          if (gp > s_pre[i]) {
            inner |= bit;
            if (q == 0) before = __ldg(p.idx[i] + src - 1);
          }
          bit <<= 1;
        }
      }
    }
    cp_async_wait_all();
    __syncthreads();
    if constexpr (kSearch) {
      // nothing else has looked at the lists: a run must ascend. (The index
      // before a run's first is below j0, or the search had gone on.)
#pragma unroll
      for (uint32_t u = 0; u < kAggStage / kThreads; ++u) {
        const uint32_t q = u * kThreads + threadIdx.x;
        const uint32_t prev = q > 0 ? st_idx[q - 1] : before;
        bad |= ((inner >> u) & 1u) && prev >= st_idx[q];
      }
    }
    uint32_t i = 0;
    while (s_pre[i + 1] <= b0) ++i;  // the stage's first worker (uniform)
    for (; i < n && s_pre[i] < b0 + bn; ++i) {
      const uint32_t a = (s_pre[i] > b0 ? s_pre[i] : b0) - b0;
      const uint32_t z = (s_pre[i + 1] < b0 + bn ? s_pre[i + 1] : b0 + bn) - b0;
      if (a >= z) continue;  // uniform: no pairs of worker i here
      for (uint32_t q = a + threadIdx.x; q < z; q += kThreads) {
        const uint32_t j = st_idx[q];
        const uint64_t r = static_cast<uint64_t>(j) - j0;  // wraps when j < j0
        if (r < kAggTile && j < d)
          acc[r] += st_val[q];
        else
          bad = true;  // unsorted or out-of-range input: skipped, latched
      }
      __syncthreads();
    }
  }
  if (bad) atomicOr(error, kDevErrBadInput);
  if (kVec && j0 + kAggTile <= d) {
    float4* out = reinterpret_cast<float4*>(o.out + j0);
    float4* mom = kMode == kAggMomentum ? reinterpret_cast<float4*>(o.m + j0) : nullptr;
    for (int q = threadIdx.x; q < kAggTile / 4; q += kThreads) {
      const float4 sv = reinterpret_cast<const float4*>(acc)[q];
      if constexpr (kMode == kAggDense) {
        out[q] = sv;
      } else {
        float4 xv = out[q];
        float4 mv = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        if constexpr (kMode == kAggMomentum) mv = mom[q];
        apply_update<kMode>(o, sv.x, xv.x, mv.x);
        apply_update<kMode>(o, sv.y, xv.y, mv.y);
        apply_update<kMode>(o, sv.z, xv.z, mv.z);
        apply_update<kMode>(o, sv.w, xv.w, mv.w);
        out[q] = xv;
        if constexpr (kMode == kAggMomentum) mom[q] = mv;
      }
    }
  } else {
    for (int q = threadIdx.x; q < kAggTile; q += kThreads) {
      if (j0 + q >= d) continue;
      if constexpr (kMode == kAggDense) {
        o.out[j0 + q] = acc[q];
      } else {
        float xv = o.out[j0 + q], mv = 0.0f;
        if constexpr (kMode == kAggMomentum) mv = o.m[j0 + q];
        apply_update<kMode>(o, acc[q], xv, mv);
        o.out[j0 + q] = xv;
        if constexpr (kMode == kAggMomentum) o.m[j0 + q] = mv;
      }
    }
  }
}

// ---------------------------------------------- the dense sum, many tiles
// One warp per CTA, persistent, a tile at a time: the warp keeps the tile's
// sum in shared memory and adds worker 0's pairs, then worker 1's, ... — a
// single warp needs no barrier between workers —, while the next pairs are on
// their way. Lane i holds worker i's list: it fetches the offsets of its next
// run a tile ahead and copies the run's aligned 16-byte windows of indices
// and values with one bulk copy each into a stage of kAggPairs pairs (a tile
// whose runs need more takes several stages; the windows are laid out in
// worker order). A lane then takes 4 consecutive pairs at a time (two
// 16-byte reads), so that 128 pairs cost about 45 instructions.
//
// Why: with a CTA of 8 warps per tile (agg_reduce_kernel) the reduction was
// bound by instructions, not by memory: 8,200 warp instructions a tile of
// 1,640 pairs (issue slots 77 % busy, DRAM at 27 %), most of them the loops
// and barriers around a few pairs per warp and worker. Here the same tile
// takes about 1,500, and what bounds it is the latency of the shared-memory
// reads of 8 warps an SM (16 KB of sums each), or DRAM once tiles hold many
// pairs. Measured on a GB300, us an exchange, before -> after: 8 workers'
// hard-threshold messages at 5 % of d = 138.4 M, with tile indexes, 262 ->
// 164 (6.1 TB/s, 91 % of the copy rate); 16 workers' Top-k messages at 1 % of
// d = 25.6 M, 51.8 -> 49.2. Stages of 448, 544, 768, 896 and 1,792 pairs:
// 175, 171, 183, 169 and 192 on the first, 61, 52, 62, 56 and 55 on the
// second. Copies by cp.async instead of bulk copies (more instructions of the
// one warp): 194-236 and 62-66.
constexpr uint32_t kAggPairs = 640;   // pairs a stage holds
constexpr int kAggStages = 2;          // one being added, one on its way
// From this many tiles on (6 per SM): with fewer, warps would be left without
// a tile while others take two, and a CTA of 8 warps finishes a tile sooner.
constexpr uint32_t kAggMinTiles = 912;

struct AggStream {  // shared memory of a CTA
  float acc[kAggTile + 32];  // the tile's sum; one unused slot per lane
  uint32_t idx[kAggStages][kAggPairs];
  float val[kAggStages][kAggPairs];
  uint32_t run[kAggStages][32];  // worker's first pair in the stage | pairs << 16
  uint32_t tile[kAggStages], last[kAggStages];
  uint64_t bar[kAggStages];
};
static_assert(offsetof(AggStream, idx) % 16 == 0 && offsetof(AggStream, val) % 16 == 0 &&
                  offsetof(AggStream, bar) % 8 == 0 && kAggPairs % 4 == 0,
              "bulk copies");

template <bool kVec>
__global__ void __launch_bounds__(32)
    agg_stream_kernel(AggPtrs<kFewWorkers> p, uint32_t n, uint32_t d, uint32_t tiles,
                      const uint32_t* __restrict__ off, const uint32_t* __restrict__ counts,
                      float* __restrict__ out, uint32_t* __restrict__ error,
                      uint64_t wait_limit_ns) {
  extern __shared__ __align__(128) unsigned char smem[];
  AggStream& sm = *reinterpret_cast<AggStream*>(smem);
  const uint32_t lane = threadIdx.x;
  if (lane == 0) {
    for (int s = 0; s < kAggStages; ++s) mbar_init(&sm.bar[s], 1);
    mbar_init_fence();
  }
  for (uint32_t q = lane; q < kAggTile / 4; q += 32)
    reinterpret_cast<float4*>(sm.acc)[q] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
  __syncwarp();
  griddep_wait();  // the lists and offsets (and everything before them) are complete
  griddep_launch_dependents();
  const bool has = lane < n;
  const uint32_t* const li = has ? p.idx[lane] : nullptr;
  const float* const lv = has ? p.val[lane] : nullptr;
  const uint32_t* const r =
      !has ? nullptr : off ? off + static_cast<uint64_t>(lane) * (tiles + 1) : p.tiles[lane];
  const uint32_t count = has ? counts[lane] : 0u;
  const bool bulk =
      ((reinterpret_cast<uintptr_t>(li) | reinterpret_cast<uintptr_t>(lv)) & 15u) == 0;
  const uint64_t policy = l2_evict_normal_policy();
  bool bad = false;

  // the tile whose pairs are copied next: this lane's run [lo, lo + cnt), its
  // place `base` in the tile's sequence of windows, and the sequence's
  // length; and the offsets read for the tile after it
  uint32_t next = blockIdx.x, lo = 0, cnt = 0, base = 0, total = 0, b0 = 0;
  uint32_t r0 = 0, r1 = 0;
  auto fetch = [&](uint32_t t) {
    if (has && t < tiles) {
      r0 = __ldg(r + t);
      r1 = __ldg(r + t + 1);
    }
  };
  auto enter = [&]() {  // tile `next`, whose offsets were fetched
    lo = min(r0, count);
    const uint32_t hi = min(r1, count);  // never past the list
    cnt = hi > lo ? hi - lo : 0u;
    if (cnt > kAggTile) {  // more than a tile can hold: not a tile's run
      cnt = kAggTile;
      bad = true;
    }
    const uint32_t len = cnt ? ((lo & 3u) + cnt + 3u) & ~3u : 0u;
    uint32_t incl = len;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t x = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= static_cast<uint32_t>(o)) incl += x;
    }
    base = incl - len;
    total = __shfl_sync(0xffffffffu, incl, 31);
    b0 = 0;
    fetch(next + gridDim.x);
  };
  fetch(next);
  if (next < tiles) enter();

  // copies the next pairs into stage s; false when there are no more tiles
  auto issue = [&](uint32_t s) -> bool {
    if (next >= tiles) return false;
    const uint32_t head = base + (lo & 3u);
    const uint32_t y0 = max(head, b0), y1 = min(head + cnt, b0 + kAggPairs);
    const bool some = y1 > y0;
    const uint32_t x0 = (y0 & ~3u) - b0, x1 = ((y1 + 3u) & ~3u) - b0;  // in the stage
    sm.run[s][lane] = some ? (y0 - b0) | ((y1 - y0) << 16) : 0u;
    const uint32_t src = (lo & ~3u) + (b0 + x0 - base);  // list position of x0
    const uint32_t bytes = some && bulk ? (x1 - x0) * 4u : 0u;
    const uint32_t tx = 2u * warp_sum(bytes);
    if (lane == 0) {
      sm.tile[s] = next;
      sm.last[s] = b0 + kAggPairs >= total ? 1u : 0u;
      mbar_arrive_expect_tx(&sm.bar[s], tx);
    }
    __syncwarp();
    if (bytes) {
      tma_load_1d(&sm.idx[s][x0], li + src, bytes, &sm.bar[s], policy);
      tma_load_1d(&sm.val[s][x0], lv + src, bytes, &sm.bar[s], policy);
    }
    uint32_t plain = __ballot_sync(0xffffffffu, some && !bulk);
    if (plain) {  // lists that are not 16-byte aligned: by plain loads
      while (plain) {
        const int q = __ffs(plain) - 1;
        plain &= plain - 1;
        const uint32_t run = sm.run[s][q];
        const uint32_t a = run & 0xffffu, z = a + (run >> 16);
        const uint32_t at = __shfl_sync(0xffffffffu, src + (y0 & 3u), q);
        const uint32_t* qi = p.idx[q];
        const float* qv = p.val[q];
        for (uint32_t x = a + lane; x < z; x += 32) {
          sm.idx[s][x] = __ldg(qi + at + (x - a));
          sm.val[s][x] = __ldg(qv + at + (x - a));
        }
      }
      // these writes before the stage's next bulk copies
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      __syncwarp();
    }
    if (b0 + kAggPairs >= total) {
      next += gridDim.x;
      if (next < tiles) enter();
    } else {
      b0 += kAggPairs;
    }
    return true;
  };

  bool more = true;
  uint32_t issued = 0, done = 0;
  while (true) {
    while (more && issued - done < static_cast<uint32_t>(kAggStages)) {
      more = issue(issued % kAggStages);
      if (more) ++issued;
    }
    if (done == issued) break;
    const uint32_t s = done % kAggStages;
    if (!__all_sync(0xffffffffu, mbar_wait(&sm.bar[s], (done / kAggStages) & 1u, wait_limit_ns))) {
      if (lane == 0) atomicOr(error, kDevErrTimeout);
      break;
    }
    const uint32_t tile = sm.tile[s];
    const uint64_t j0 = static_cast<uint64_t>(tile) * kAggTile;
    const uint32_t room = static_cast<uint32_t>(min(d - j0, static_cast<uint64_t>(kAggTile)));
    const uint32_t my_run = sm.run[s][lane];
    uint32_t live = __ballot_sync(0xffffffffu, my_run >> 16);
    // the stage's pairs, 128 at a time, worker by worker: (first, end) of the
    // worker's run and this lane's 4 pairs from x on, read one step ahead
    struct Quad {
      uint4 j;
      float4 v;
      uint32_t x, first, len;
    };
    uint32_t q_first = 0, q_end = 0, q_x = 0;
    auto read = [&](Quad& c) -> bool {
      if (q_x >= q_end) {
        if (!live) return false;
        const uint32_t run = __shfl_sync(0xffffffffu, my_run, __ffs(live) - 1);
        live &= live - 1;
        q_first = run & 0xffffu;
        q_end = q_first + (run >> 16);
        q_x = q_first & ~3u;
      }
      c.x = q_x + 4 * lane;
      c.first = q_first;
      c.len = q_end - q_first;
      if (c.x < q_end) {
        c.j = *reinterpret_cast<const uint4*>(&sm.idx[s][c.x]);
        c.v = *reinterpret_cast<const float4*>(&sm.val[s][c.x]);
      }
      q_x += 128;
      return true;
    };
    auto add = [&](const Quad& c) {
      const uint32_t j[4] = {c.j.x, c.j.y, c.j.z, c.j.w};
      const float v[4] = {c.v.x, c.v.y, c.v.z, c.v.w};
      uint32_t at[4];
      float sum[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const bool in_run = c.x + u - c.first < c.len;  // wraps before the run
        const uint32_t rel = j[u] - static_cast<uint32_t>(j0);
        // unsorted or out-of-range input: skipped, latched
        const bool ok = in_run && rel < room;
        bad |= in_run != ok;
        at[u] = ok ? rel : kAggTile + lane;
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) sum[u] = sm.acc[at[u]];
#pragma unroll
      for (int u = 0; u < 4; ++u) sm.acc[at[u]] = sum[u] + v[u];
      __syncwarp();
    };
    Quad a, b;
    bool have = read(a);
    while (have) {
      const bool have_b = read(b);
      add(a);
      if (!have_b) break;
      have = read(a);
      add(b);
    }
    if (sm.last[s]) {  // the tile is complete: write it, and zero the sum again
      float4* acc4 = reinterpret_cast<float4*>(sm.acc);
      if (kVec && room == kAggTile) {
        float4* o4 = reinterpret_cast<float4*>(out + j0);
#pragma unroll 8
        for (uint32_t q = lane; q < kAggTile / 4; q += 32) {
          o4[q] = acc4[q];
          acc4[q] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        }
      } else {
        for (uint32_t q = lane; q < kAggTile; q += 32) {
          if (q < room) out[j0 + q] = sm.acc[q];
          sm.acc[q] = 0.0f;
        }
      }
    }
    __syncwarp();
    ++done;
  }
  // no copy may land after the CTA exits (only after a wait ran out)
  for (; done < issued; ++done)
    mbar_wait(&sm.bar[done % kAggStages], (done / kAggStages) & 1u, wait_limit_ns);
  if (bad) atomicOr(error, kDevErrBadInput);
}

template <int kMode, uint32_t kCap, bool kSearch>
const void* reduce_kernel(bool vec) {
  return vec ? reinterpret_cast<const void*>(&agg_reduce_kernel<true, kMode, kCap, kSearch>)
             : reinterpret_cast<const void*>(&agg_reduce_kernel<false, kMode, kCap, kSearch>);
}

template <int kMode, uint32_t kCap>
cudaError_t launch_reduce(bool vec, AggPtrs<kCap>& p, uint32_t n, uint32_t d, uint32_t tiles,
                          const uint32_t* off, const uint32_t* counts, AggOut o, Workspace& ws) {
  uint32_t* error = ws.u32(kOffError);
  void* params[] = {&p, &n, &d, &tiles, &off, &counts, &o, &error};
  const bool search = !off && !p.tiles[0];
  const void* fn = search ? reduce_kernel<kMode, kCap, true>(vec)
                          : reduce_kernel<kMode, kCap, false>(vec);
  return launch_pdl(fn, tiles, kThreads, 0, ws.stream, params, false);
}

// Each list's position at every tile boundary, for lists without tile indexes.
template <uint32_t kCap>
cudaError_t launch_offsets(AggPtrs<kCap>& p, const uint32_t* counts, uint32_t n, uint32_t d,
                           uint32_t tiles, uint32_t* off, Workspace& ws) {
  // a thread per tile for the searches; for the scatter about 8 CTAs per SM
  // in all, but no more than 16 entries a tile would occupy
  const uint32_t per_tile = (tiles + 1 + kThreads - 1) / kThreads;
  const uint32_t wide = std::min((1216 + n - 1) / n, (tiles / kThreads + 1) * 16);
  const dim3 grid(std::max(per_tile, wide), n);
  uint32_t* error = ws.u32(kOffError);
  void* params[] = {&p, &counts, &n, &d, &tiles, &off, &error};
  const cudaError_t err = launch_pdl(reinterpret_cast<const void*>(&agg_offsets_kernel<kCap>),
                                     grid, kThreads, 0, ws.stream, params, false);
  count_launch();
  return err;
}

// Up to this many tiles the reduction finds its runs itself instead of reading
// them from the offsets kernel: its CTAs are resident at once (8 per SM), so
// the searches of all tiles run side by side, and a launch is saved. Measured
// on a GB300, us a call from Python, offsets kernel -> searched in place: 4
// lists of 10 %, d = 100,000, update 12.7 -> 11.5, d = 2.4 M 30.3 -> 25.6; 16
// lists of 1 %, d = 3.7 M (904 tiles), sum 25.6 -> 23.8. The sum over more tiles
// (agg_stream_kernel) needs the offsets.
constexpr uint32_t kAggSearchTiles = kAggMinTiles - 1;

template <uint32_t kCap>
cudaError_t launch_common(uint32_t n, const uint32_t* const* idx, const float* const* val,
                          const uint32_t* const* tile_index, const uint32_t* counts, uint32_t d,
                          const AggOut& o, int mode, Workspace& ws, int agg_stream_slots) {
  AggPtrs<kCap> p;
  for (uint32_t i = 0; i < n; ++i) {
    p.idx[i] = idx[i];
    p.val[i] = val[i];
    p.tiles[i] = tile_index ? tile_index[i] : nullptr;
  }
  uint32_t tiles = agg_tiles_for(d);
  cudaError_t err = cudaSuccess;
  uint32_t* off = nullptr;
  if (!tile_index && tiles > kAggSearchTiles) {  // locate each list's tile boundaries first
    off = ws.offsets();
    err = launch_offsets(p, counts, n, d, tiles, off, ws);
    if (err != cudaSuccess) return err;
  }
  const bool vec = reinterpret_cast<uintptr_t>(o.out) % 16 == 0 &&
                   reinterpret_cast<uintptr_t>(o.m) % 16 == 0;
  if (mode == kAggDense) {
    if constexpr (kCap == kFewWorkers) {
      if (tiles >= kAggMinTiles && agg_stream_slots > 0) {
        float* out = o.out;
        uint32_t* error = ws.u32(kOffError);
        uint64_t limit = wait_limit_ns();
        void* params[] = {&p, &n, &d, &tiles, &off, &counts, &out, &error, &limit};
        const void* fn = vec ? reinterpret_cast<const void*>(&agg_stream_kernel<true>)
                             : reinterpret_cast<const void*>(&agg_stream_kernel<false>);
        err = launch_pdl(fn, std::min(tiles, static_cast<uint32_t>(agg_stream_slots)), 32,
                         sizeof(AggStream), ws.stream, params, false);
        count_launch();
        return err;
      }
    }
    err = launch_reduce<kAggDense>(vec, p, n, d, tiles, off, counts, o, ws);
  } else if (mode == kAggSgd) {
    err = launch_reduce<kAggSgd>(vec, p, n, d, tiles, off, counts, o, ws);
  } else {
    err = launch_reduce<kAggMomentum>(vec, p, n, d, tiles, off, counts, o, ws);
  }
  count_launch();
  return err;
}

cudaError_t launch_any(uint32_t n, const uint32_t* const* idx, const float* const* val,
                       const uint32_t* const* tiles, const uint32_t* counts, uint32_t d,
                       const AggOut& o, int mode, Workspace& ws, int agg_stream_slots) {
  return n <= kFewWorkers ? launch_common<kFewWorkers>(n, idx, val, tiles, counts, d, o, mode, ws,
                                                       agg_stream_slots)
                          : launch_common<kMaxWorkers>(n, idx, val, tiles, counts, d, o, mode, ws,
                                                       agg_stream_slots);
}

template <uint32_t kCap, bool kSearch>
void prefer_shared() {
  for (bool vec : {false, true})
    for (const void* f :
         {reduce_kernel<kAggDense, kCap, kSearch>(vec), reduce_kernel<kAggSgd, kCap, kSearch>(vec),
          reduce_kernel<kAggMomentum, kCap, kSearch>(vec)})
      cudaFuncSetAttribute(f, cudaFuncAttributePreferredSharedMemoryCarveout,
                           cudaSharedmemCarveoutMaxShared);
}
}  // namespace

void aggregate_init_device(DeviceInfo& info) {
  const void* streams[] = {reinterpret_cast<const void*>(&agg_stream_kernel<true>),
                           reinterpret_cast<const void*>(&agg_stream_kernel<false>)};
  int per_sm = 0;
  for (const void* f : streams) {
    int b = 0;
    cudaFuncSetAttribute(f, cudaFuncAttributePreferredSharedMemoryCarveout,
                         cudaSharedmemCarveoutMaxShared);
    if (cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, sizeof(AggStream)) !=
            cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, f, 32, sizeof(AggStream)) != cudaSuccess)
      b = 0;
    per_sm = f == streams[0] || b < per_sm ? b : per_sm;
  }
  info.agg_stream_slots = per_sm * info.sm_count;
  prefer_shared<kFewWorkers, false>();
  prefer_shared<kFewWorkers, true>();
  prefer_shared<kMaxWorkers, false>();
  prefer_shared<kMaxWorkers, true>();
  cudaGetLastError();
}

cudaError_t launch_aggregate(uint32_t n, const uint32_t* const* idx, const float* const* val,
                             const uint32_t* const* tiles, const uint32_t* counts, uint32_t d,
                             float* dense_out, Workspace& ws, const DeviceInfo& dev) {
  return launch_any(n, idx, val, tiles, counts, d,
                       AggOut{dense_out, nullptr, 1.0f, 0.0f, 0.0f}, kAggDense, ws,
                       dev.agg_stream_slots);
}

cudaError_t launch_aggregate_apply(uint32_t n, const uint32_t* const* idx,
                                   const float* const* val, const uint32_t* const* tiles,
                                   const uint32_t* counts, uint32_t d, float alpha, float* x,
                                   float* m, float mu, float lr, Workspace& ws) {
  return launch_any(n, idx, val, tiles, counts, d, AggOut{x, m, alpha, mu, lr},
                       m ? kAggMomentum : kAggSgd, ws, 0);
}

cudaError_t launch_list_tiles(const uint32_t* idx, const uint32_t* count, uint32_t d,
                              uint32_t* tiles_out, Workspace& ws) {
  AggPtrs<kFewWorkers> p;
  p.idx[0] = idx;
  return launch_offsets(p, count, 1, d, agg_tiles_for(d), tiles_out, ws);
}

}  // namespace efs
