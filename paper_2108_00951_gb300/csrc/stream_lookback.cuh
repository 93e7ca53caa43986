// stream_lookback.cuh — ordered stream compaction at memory speed with
// dynamically claimed work: persistent CTAs (one per SM) take groups of
// tiles from a global counter, stream them through a TMA-fed ring, and place
// each group's selected pairs straight from shared memory once a decoupled
// look-back has given the group its output position.
//
// Why dynamic groups: on this GPU the DRAM bandwidth a single SM receives
// varies from call to call by about +-15 % (the same SM is among the fastest
// in one call and the slowest in the next), so any partition fixed at launch
// leaves the memory system partly idle while the slowest CTAs finish.
// Claiming small groups balances that automatically, and because a group
// only ever waits for groups claimed before it (held by CTAs that are
// already running), progress does not depend on which CTAs are resident.
//
// Roles (warps of a CTA), which hand groups to one another through a ring of
// entries with three mbarriers each (counted, ready, free):
//  - 16 compute warps. Warp w owns the 256-coordinate segment [w*256,
//    (w+1)*256) of every tile (the element layout of stream_compact.cuh). A
//    group's two tiles arrive in consecutive ring stages; the warp computes
//    each tile's values and selection bits and releases its stage at once,
//    then, once for the group: the positions of its selected pairs (one warp
//    scan of the four units' counts), the pairs appended to its own circular
//    buffer in shared memory — or, for a segment that finds no room, to the
//    segment's slot in global memory —, and for each segment a word with its
//    count and place in the group's entry; its arrival on "counted" is all
//    that the others need of it.
//  - a producer warp: lane 1 claims groups, up to kLbClaimAhead ahead; lane 0
//    takes a claimed group when an entry is free and issues the bulk copies
//    (cp.async.bulk, completing on the stage's "full" mbarrier) of its tiles
//    as ring stages are released; after the last group, an end marker.
//  - an aggregate warp publishes each counted group's total.
//  - a look-back warp: for each counted group of the CTA in claim order, the
//    decoupled look-back over the published group totals (Merrill & Garland,
//    the routine of the one-tile-per-CTA kernel), the inclusive total
//    published, then the output position of each of the group's segments in
//    (tile, warp) order, which is coordinate order; arrives on "ready".
//  - kLbPlaceWarps placer warps: for each ready group, placer p copies the
//    segments p, p + kLbPlaceWarps, ... (a warp's lanes on consecutive pairs,
//    so loads and stores are coalesced) from the buffers or slots to the
//    output; the last to finish a group hands the buffers' space back and
//    frees the entry.
// A warp that waits is suspended on an mbarrier and issues next to nothing:
// the compute warps, whose instruction chain bounds the kernel, have the
// issue slots. Measured on a GB300, us a call, against the same roles with
// polled words, a counter that the compute warps increment, and a barrier of
// all placers twice a group: VGG-16-shaped fp32 262.8 -> 248.2 (100 % of the
// copy rate), bf16 g 235.3 -> 219.0 (95 %), at 25 % sent 335 -> 325;
// ResNet-50-shaped at 22 % sent 94.4 -> 84.7, with a bf16 g 89.8 -> 78.7;
// LSTM-shaped 65.6 -> 65.1. Eight placers that each serve two compute warps
// and poll: 268, 255, 359, 106, 102 and 69.
//
// Deadlock freedom. Take the lowest group m that is claimed but whose
// aggregate is not published. Groups below m have published aggregates, so
// the look-back (and then the placement) of every group below m completes,
// which frees every entry and buffer space they hold. The CTA holding m waits
// for nothing else: a compute warp never waits for buffer space (a segment
// without room goes to its slot), the producer waits only for entries of
// older groups of its own CTA and for its ring, the ring's stages are
// released by the compute warps as soon as they have read them, and the
// aggregate warp never waits for a look-back. So m is published and the
// argument repeats; no wait depends on which CTAs are
// resident. Every wait is nevertheless bounded in time; one that runs out
// latches kDevErrTimeout, and the CTA stops (after its bulk copies have
// landed).
//
// Traffic: the op's own bytes plus 8 bytes per selected pair, written once,
// plus 16 bytes per pair that goes through a slot; 8 bytes of look-back
// status per group. The error norm (when la.err_out is set) follows
// stream_compact.cuh's rule per coordinate; each group's share (its warps'
// float-float shares in warp order) is stored per group, and the last CTA to
// finish adds the groups' shares in group order, so the value does not
// depend on which CTA took which group.
#pragma once

#include "internal.h"
#include "stream_compact.cuh"

namespace efs {

constexpr int kLbProducerWarp = kSWarps;       // 16
constexpr int kLbScanWarp = kSWarps + 1;       // 17
constexpr int kLbAggWarp = kSWarps + 2;        // 18
constexpr int kLbPlaceWarp = kSWarps + 3;      // 19: the first placer warp
constexpr int kLbPlaceWarps = 12;  // with 8, calls that send a quarter of a vector take 6 % longer
constexpr int kLbThreads = 32 * (kSWarps + 3 + kLbPlaceWarps);  // 992
static_assert(kLbThreads <= 1024, "one CTA of at most 1024 threads");
constexpr uint32_t kLbGroupTiles = 2;          // tiles per claimed group (the placement
                                               // assumes 2: 32 segments, one per lane)
constexpr uint32_t kLbGroupSegs = kLbGroupTiles * kSWarps;
constexpr uint32_t kLbClaimAhead = 2;          // groups claimed before the producer needs them
// Groups of a CTA in flight or pending. More entries let streaming run ahead
// of the look-back; in dense calls they also let it run ahead of the placers,
// whose buffers then overflow into the slots. Measured with 8, 10, 12, 16 and 24, us a
// call: VGG-16-shaped 262.0, 252.7, 248.2, 249.6, 252.0; with 5, 6, 7, 8 and 10 on the
// shallow ring: ResNet-50-shaped at 22 % sent 82.2, 81.1, 84.7, 86.3, 87.0;
// VGG-16-shaped at 25 % sent 365, 335, 325, 319, 322.
constexpr int kLbManyEntries = 12, kLbFewEntries = 7;
constexpr uint32_t kLbStageEnd = 0xffffffffu;
constexpr uint32_t kLbSuspendNs = 1000;        // a suspended wait re-checks its flag and limit this often
constexpr uint32_t kLbSegsPerLane = kLbGroupSegs / 32;  // segments per lane in the offset scan
static_assert(kLbGroupSegs % 32 == 0 && kLbSegsPerLane <= 2, "segments per look-back lane");

// One group of a CTA, from the producer taking it until its pairs are placed.
struct LbEntry {
  uint32_t seg[kLbGroupSegs];  // segment (q, w) at q * 16 + w: its pairs and where they are
  uint32_t off[kLbGroupSegs];  // output position of each segment's first pair
  FF err[kSWarps];             // the warps' shares of ||e'||^2 in this group
  uint32_t group;              // group index
  uint32_t ntiles;             // tiles of the group (the last may have fewer); 0: no more groups
  uint32_t placed;             // placers done with it
  uint32_t pad;
};
// A segment's word: its pairs (at most 256), whether they are in its global
// slot, and else the position of the first in its warp's buffer.
__device__ __forceinline__ uint32_t lb_seg(uint32_t count, bool slot, uint32_t first) {
  return count | (slot ? 0x8000u : 0u) | (first << 16);
}
__device__ __forceinline__ uint32_t lb_seg_count(uint32_t seg) { return seg & 0x1ffu; }
__device__ __forceinline__ bool lb_seg_slot(uint32_t seg) { return (seg & 0x8000u) != 0; }
__device__ __forceinline__ uint32_t lb_seg_first(uint32_t seg) { return seg >> 16; }

template <class Op, int kStages, int kEntries>
struct LbLayout {
  static constexpr uint32_t kRing = kStages * Op::kStageBytes;
  // pair buffer per compute warp: what is left of 227 KB (less 2 KB of static
  // shared memory), in whole warps of pairs
  static constexpr uint32_t kEntryBytes = kEntries * sizeof(LbEntry);
  static constexpr uint32_t kBudget = 227u * 1024u - 2048u;
  static constexpr uint32_t kFifo = ((kBudget - kRing - kEntryBytes) / (kSWarps * 8u)) / 32u * 32u;
  // (a segment that finds no room goes to its global slot, so nothing waits
  // for buffer space; a buffer smaller than a segment would only spill more)
  static_assert(kFifo >= kSWarpElems, "a whole segment fits a warp's buffer");
  static constexpr uint32_t kOffEntries = kRing + kSWarps * kFifo * 8u;
  static constexpr uint32_t kSmem = kOffEntries + kEntryBytes;  // dynamic shared memory
};

struct LbArgs {
  uint32_t* claim;      // groups handed out so far, zero at the call's start
  uint32_t* claim_next; // the next call's counter, zeroed here (null: a captured call's)
  uint32_t* tile_base;  // optional [num_tiles + 1]: output position of each tile's first pair,
                        // and the total (untruncated), or null
  double* err_out;      // optional: sum of a^2 over the coordinates whose residual is final
                        // here (not selected, not deferred), or null
  FF* err_parts;        // [groups] the groups' shares of it (used when err_out is set)
  uint32_t* err_count;  // [2] groups resolved, CTAs finished (zero between calls)
  uint2* slot;          // [num_tiles * 16 * 256] a segment's pairs (index, value bits) when its
                        // warp's buffer is full: segment (tile, warp) at (tile * 16 + warp) * 256
  uint32_t* density_out;  // optional (host-mapped): the call's pair count * 65536 / d, a hint
                          // the host reads for later calls' choice of ring depth, or null
};

__device__ __forceinline__ uint32_t vld(const uint32_t& x) {
  return *reinterpret_cast<const volatile uint32_t*>(&x);
}
__device__ __forceinline__ void vst(uint32_t& x, uint32_t v) {
  *reinterpret_cast<volatile uint32_t*>(&x) = v;
}

// The arguments of a launch on a workspace (the groups' shares of ||e'||^2 use
// the per-tile count area, 16 words a tile). The two counters rely on every
// launch running in the order it was made. A captured one may run later or
// never: it takes a third, zeroed by a node of its own graph, and leaves the
// order of the two as it is.
inline cudaError_t lb_args(Workspace& ws, uint32_t* tile_base, double* err_out,
                           uint32_t* density_out, LbArgs* la) {
  uint32_t* const claims = ws.u32(kOffGroupClaim);
  cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
  cudaError_t err = cudaStreamIsCapturing(ws.stream, &capture);
  if (err != cudaSuccess) return err;
  *la = LbArgs{nullptr, nullptr, tile_base, err_out, reinterpret_cast<FF*>(ws.counts()),
               ws.u32(kOffGroupErr), ws.stage_pairs(), density_out};
  if (capture == cudaStreamCaptureStatusNone) {
    const uint32_t parity = ws.group_calls++ & 1u;
    la->claim = claims + parity;
    la->claim_next = claims + (parity ^ 1u);
  } else {
    la->claim = ws.u32(kOffGroupCaptured);
    err = cudaMemsetAsync(la->claim, 0, sizeof(uint32_t), ws.stream);
  }
  return err;
}

// Bounded spin of one thread until pred() holds; false (and the CTA's failed
// flag set, the timeout latched) when the limit passes, false at once when
// another thread of the CTA has failed.
template <class Pred>
__device__ __forceinline__ bool lb_spin(Pred pred, uint32_t* s_failed, const ScanCtx& ctx) {
  if (pred()) return true;
  const uint64_t t0 = global_timer_ns();
  for (uint32_t it = 0;; ++it) {
    if (pred()) return true;
    if (vld(*s_failed)) return false;
    if (it > (1u << 26) || global_timer_ns() - t0 > ctx.wait_limit_ns) {
      vst(*s_failed, 1u);
      atomicOr(ctx.error, kDevErrTimeout);
      return false;
    }
    __nanosleep(64);
  }
}

// Bounded wait for an mbarrier phase, giving up when the CTA has failed.
__device__ __forceinline__ bool lb_mbar_wait(uint64_t* bar, uint32_t parity, uint32_t* s_failed,
                                             const ScanCtx& ctx) {
  if (mbar_try_wait(bar, parity)) return true;
  const uint64_t t0 = global_timer_ns();
  for (uint32_t it = 0;; ++it) {
    if (mbar_try_wait_for(bar, parity, kLbSuspendNs)) return true;
    if (vld(*s_failed)) return false;
    if (it > (1u << 26) || global_timer_ns() - t0 > ctx.wait_limit_ns) {
      vst(*s_failed, 1u);
      atomicOr(ctx.error, kDevErrTimeout);
      return false;
    }
  }
}

// The barriers of an entry complete one phase per group that uses it.
template <int kEntries>
__device__ __forceinline__ uint32_t lb_parity(uint32_t seq) {
  return (seq / kEntries) & 1u;
}

// x[j] for a run-time j without an indexed (local-memory) access.
__device__ __forceinline__ float lb_pick(const float (&x)[4], int j) {
  const float lo = (j & 1) ? x[1] : x[0];
  const float hi = (j & 1) ? x[3] : x[2];
  return (j & 2) ? hi : lo;
}

// The test hook withholds a tile; here the group holding it never publishes.
__device__ __forceinline__ bool lb_withheld(const ScanCtx& ctx, uint32_t group) {
  return ctx.withheld_tile >= 0 &&
         static_cast<int64_t>(group) == ctx.withheld_tile / static_cast<int64_t>(kLbGroupTiles);
}

template <class Op, int kStages, int kEntries>
__global__ void __launch_bounds__(kLbThreads, 1)
    lookback_stream_kernel(Op op, uint32_t* __restrict__ idx_out,
                           float* __restrict__ val_out, uint32_t* __restrict__ count_out,
                           uint32_t cap, ScanCtx ctx, LbArgs la) {
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ __align__(8) uint64_t s_full[kStages];
  __shared__ __align__(8) uint64_t s_empty[kStages];
  __shared__ uint32_t s_stage_tile[kStages];  // tile of the stage's current use, or the end
  __shared__ uint32_t s_stage_slot[kStages];  // its group's entry
  __shared__ __align__(8) uint64_t s_counted[kEntries];  // every segment's word is there
  __shared__ __align__(8) uint64_t s_ready[kEntries];    // so are the output positions
  __shared__ __align__(8) uint64_t s_free[kEntries];     // every pair is placed, the total published
  __shared__ uint32_t s_failed;               // a wait of this CTA ran out
  __shared__ uint32_t s_resolved;             // groups the look-back warp resolved
  __shared__ uint32_t s_freed[kSWarps];       // pairs of each compute warp placed so far
  __shared__ uint32_t s_cq[kLbClaimAhead];    // groups claimed ahead, with the queue counts
  __shared__ uint32_t s_cq_tail, s_cq_head;
  __shared__ uint32_t s_last;                 // this CTA finished last
  __shared__ FF s_err_sum[32];
  using L = LbLayout<Op, kStages, kEntries>;
  uint2* const f_pair = reinterpret_cast<uint2*>(smem + L::kRing);  // (index, value bits)
  LbEntry* const ent = reinterpret_cast<LbEntry*>(smem + L::kOffEntries);

  const uint32_t T = ctx.num_tiles;
  const uint32_t G = (T + kLbGroupTiles - 1) / kLbGroupTiles;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;

  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(&s_full[s], 1);
      mbar_init(&s_empty[s], kSWarps);
    }
    for (uint32_t s = 0; s < kEntries; ++s) {
      mbar_init(&s_counted[s], kSWarps);
      mbar_init(&s_ready[s], 1);
      mbar_init(&s_free[s], 2);  // the aggregate warp and the last placer
    }
    mbar_init_fence();
    s_failed = 0;
    s_resolved = 0;
    s_cq_tail = 0;
    s_cq_head = 0;
  }
  if (threadIdx.x < kSWarps) s_freed[threadIdx.x] = 0;
  __syncthreads();
  // A dependent launch starts while the previous kernel's last groups are
  // placed, a phase that leaves DRAM mostly idle: pull the first groups that
  // will be claimed (two for every CTA, whichever takes them) toward L2
  // meanwhile. A prefetch is not a read of the data: L2 is the point of
  // coherence, so the previous kernel's writes still land before the bulk
  // copies read these lines. Whole tiles only.
  if (threadIdx.x == 0 && Op::kPrefetchTiles > 0) {
    for (uint32_t r = 0; r < 2; ++r)
      for (uint32_t j = 0; j < kLbGroupTiles; ++j) {
        const uint32_t t = (blockIdx.x + r * gridDim.x) * kLbGroupTiles + j;
        if (op.full(t)) op.prefetch(t);
      }
  }
  // The first claims too are made before the wait: this call's counter was
  // left at zero by the call before on this workspace (each zeroes the other
  // of two, whose user is complete by then, before it lets the next start); a
  // captured call's by the memset before it.
  const bool claimer = warp == kLbProducerWarp && lane == 1;
  uint32_t claimed = 0;  // claimer: groups claimed so far, and whether that was all
  bool last_claim = false;
  if (claimer) {
    for (; claimed < kLbClaimAhead && !last_claim; ++claimed) {
      const uint32_t g = atomicAdd(la.claim, 1u);
      s_cq[claimed] = g;
      last_claim = g >= G;
    }
    __threadfence_block();
    vst(s_cq_tail, claimed);
  }
  // everything the previous kernels on the stream wrote is read only after this
  griddep_wait();
  op.prologue();
  const uint64_t aux = op.initial_aux();  // uniform

  if (warp == kLbProducerWarp) {
    if (claimer) {
      // ---------------------------------------------------- claimer
      // Claims groups up to kLbClaimAhead ahead of the producer, so that a
      // claim's round trip never stalls the producer's refills (a fence or
      // an mbarrier arrival of the producer would wait for it).
      while (!last_claim) {
        if (!lb_spin([&] { return claimed - vld(s_cq_head) < kLbClaimAhead; }, &s_failed, ctx))
          break;
        const uint32_t g = atomicAdd(la.claim, 1u);
        s_cq[claimed % kLbClaimAhead] = g;
        __threadfence_block();
        vst(s_cq_tail, ++claimed);
        last_claim = g >= G;
      }
    }
    // ------------------------------------------------------ producer
    if (lane == 0) {
      const uint64_t policy = l2_evict_normal_policy();
      uint32_t r = 0, seq = 0;
      bool ok = true;
      if (blockIdx.x == 0 && la.claim_next) {
        *la.claim_next = 0;
        __threadfence();  // before this thread lets the next kernel be scheduled
      }
      // the stage of use r is free once its previous use was released
      auto stage_free = [&](int s) {
        return r < static_cast<uint32_t>(kStages) ||
               lb_mbar_wait(&s_empty[s], ((r / kStages) - 1) & 1u, &s_failed, ctx);
      };
      uint32_t cq_head = 0;
      while (ok) {
        const uint32_t slot = seq % kEntries;
        LbEntry& en = ent[slot];
        if (seq >= kEntries &&
            !lb_mbar_wait(&s_free[slot], lb_parity<kEntries>(seq) ^ 1u, &s_failed, ctx)) {
          ok = false;
          break;
        }
        if (!lb_spin([&] { return vld(s_cq_tail) > cq_head; }, &s_failed, ctx)) {
          ok = false;
          break;
        }
        __threadfence_block();  // the claimed number after the count
        const uint32_t g = vld(s_cq[cq_head % kLbClaimAhead]);
        vst(s_cq_head, ++cq_head);
        const uint32_t nt = g < G ? min(kLbGroupTiles, T - g * kLbGroupTiles) : 0u;
        en.group = g;
        en.ntiles = nt;
        en.placed = 0;
        // the group's stages; none left: one that ends the compute warps, whose
        // arrivals carry the entry's end mark (ntiles == 0) to the other roles
        for (uint32_t q = 0; q < (nt ? nt : 1u); ++q, ++r) {
          const int s = static_cast<int>(r % kStages);
          if (!stage_free(s)) {
            ok = false;
            break;
          }
          const uint32_t t = g * kLbGroupTiles + q;
          s_stage_tile[s] = nt ? t : kLbStageEnd;
          s_stage_slot[s] = slot;
          if (nt && op.full(t))
            op.fill(smem + s * Op::kStageBytes, t, &s_full[s], policy);
          else
            mbar_arrive(&s_full[s]);  // a partial tile is read from global memory
        }
        ++seq;
        if (!nt) break;
      }
      griddep_launch_dependents();  // this CTA reads nothing more: the next kernel may be scheduled
      // no copy may land after the CTA exits: wait for the last use of every
      // stage (a completed phase reports complete at once)
      for (uint32_t q = r > static_cast<uint32_t>(kStages) ? r - kStages : 0; q < r; ++q)
        if (!mbar_wait(&s_full[q % kStages], (q / kStages) & 1u, ctx.wait_limit_ns))
          atomicOr(ctx.error, kDevErrTimeout);
    }
  } else if (warp == kLbScanWarp) {
    // ------------------------------------------------------ look-back
    bool ended = false;  // at the end mark, and not at a wait that ran out
    for (uint32_t seq = 0;; ++seq) {
      const uint32_t slot = seq % kEntries;
      LbEntry& en = ent[slot];
      const bool counted = lb_mbar_wait(&s_counted[slot], lb_parity<kEntries>(seq), &s_failed, ctx);
      if (!__all_sync(0xffffffffu, counted)) break;
      const uint32_t g = en.group, nt = en.ntiles;
      if (nt == 0) {  // no more groups: the placers end too
        if (lane == 0) mbar_arrive(&s_ready[slot]);
        ended = true;
        break;
      }
      // segment positions in (tile, warp) order: lane l holds segments
      // l * kLbSegsPerLane onwards
      const uint32_t nseg = nt * kSWarps;
      uint32_t cs[kLbSegsPerLane], mine = 0;
#pragma unroll
      for (uint32_t i = 0; i < kLbSegsPerLane; ++i) {
        const uint32_t sg = lane * kLbSegsPerLane + i;
        cs[i] = sg < nseg ? lb_seg_count(en.seg[sg]) : 0u;
        mine += cs[i];
      }
      uint32_t incl = mine;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t v = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += v;
      }
      const uint32_t total = __shfl_sync(0xffffffffu, incl, 31);
      bool timed_out = false;
      const uint32_t excl = lookback_exclusive(ctx, g, timed_out);
      if (timed_out) {
        if (lane == 0) {
          vst(s_failed, 1u);
          atomicOr(ctx.error, kDevErrTimeout);
        }
        break;
      }
      if (lane == 0 && !lb_withheld(ctx, g))
        st_relaxed_u64(ctx.status + g, pack_status(ctx.epoch, kFlagPrefix, excl + total));
      const uint32_t first = excl + incl - mine;
      uint32_t run = first;
#pragma unroll
      for (uint32_t i = 0; i < kLbSegsPerLane; ++i) {
        en.off[lane * kLbSegsPerLane + i] = run;
        run += cs[i];
      }
      // a tile's first segment is segment q * 16, the first of lane q * 16 / kLbSegsPerLane
      const uint32_t tile_first =
          __shfl_sync(0xffffffffu, first, (lane * (kSWarps / kLbSegsPerLane)) & 31);
      if (la.tile_base && static_cast<uint32_t>(lane) < nt)
        la.tile_base[g * kLbGroupTiles + lane] = tile_first;
      if (lane == 0) {
        if (g == G - 1) {
          const uint32_t end = excl + total;
          *count_out = end < cap ? end : cap;
          if (la.tile_base) la.tile_base[T] = end;
          if (la.density_out)
            *la.density_out =
                static_cast<uint32_t>((static_cast<uint64_t>(end) << 16) / (op.end - op.shift()));
        }
        if (la.err_out) {
          FF s{0.0f, 0.0f};
          for (int w = 0; w < kSWarps; ++w) s = ff_add(s, en.err[w]);
          la.err_parts[g] = s;
        }
      }
      __syncwarp();
      if (lane == 0) {
        mbar_arrive(&s_ready[slot]);
        ++s_resolved;
      }
    }
    // The last group's CTA writes the call's count, unless one of its waits
    // runs out (or every CTA stops before that group is claimed). A CTA that
    // stops says 0 instead: what reads the message next takes its length from
    // that word, which may hold anything before the call. Where the count is
    // written too, either of the two may stay; the call has failed.
    if constexpr (!Op::kKeepPairs)
      if (!ended && lane == 0) *count_out = 0;
  } else if (warp == kLbAggWarp) {
    // ------------------------------------------------------ aggregates
    // Publishes each group's total as soon as its segments are counted (the
    // look-back warp may still be waiting for an earlier group's neighbours).
    for (uint32_t seq = 0;; ++seq) {
      const uint32_t slot = seq % kEntries;
      const bool counted = lb_mbar_wait(&s_counted[slot], lb_parity<kEntries>(seq), &s_failed, ctx);
      if (!__all_sync(0xffffffffu, counted)) break;
      const LbEntry& en = ent[slot];
      const uint32_t g = en.group, nseg = en.ntiles * kSWarps;
      if (nseg == 0) break;
      uint32_t part = 0;
#pragma unroll
      for (uint32_t i = 0; i < kLbSegsPerLane; ++i) {
        const uint32_t sg = lane + 32 * i;
        part += sg < nseg ? lb_seg_count(en.seg[sg]) : 0u;
      }
      const uint32_t agg = warp_sum(part);
      if (lane == 0) {
        // max: the look-back warp may have published the group's prefix, whose
        // flag is the larger one
        if (!lb_withheld(ctx, g))
          atomicMax(reinterpret_cast<unsigned long long*>(ctx.status + g),
                    static_cast<unsigned long long>(pack_status(ctx.epoch, kFlagAggregate, agg)));
        mbar_arrive(&s_free[slot]);  // done with the entry
      }
    }
  } else if (warp >= kLbPlaceWarp) {
    // ------------------------------------------------------ placement
    // For each group in claim order, once its positions are there: placer p
    // copies the segments l = p, p + kLbPlaceWarps, ...: a segment's pairs are
    // consecutive in its source and in the output, so the warp's lanes take
    // consecutive pairs (coalesced loads and stores). No placer waits for
    // another. The last to finish a group hands the buffers' space back and
    // frees the entry: every placer goes through the groups in order, so all
    // earlier groups' pairs are placed by then.
    const int pw = warp - kLbPlaceWarp;
    const uint64_t keep_policy = Op::kKeepPairs ? l2_evict_last_policy() : 0ull;
    bool overflow = false;
    for (uint32_t seq = 0;; ++seq) {
      const uint32_t slot = seq % kEntries;
      LbEntry& en = ent[slot];
      const bool ready = lb_mbar_wait(&s_ready[slot], lb_parity<kEntries>(seq), &s_failed, ctx);
      if (!__all_sync(0xffffffffu, ready)) break;
      const uint32_t nt = en.ntiles;
      if (nt == 0) break;
      const uint32_t nseg = nt * kSWarps;
      // lane l describes segment l (l < nseg)
      const uint32_t seg = static_cast<uint32_t>(lane) < nseg ? en.seg[lane] : 0u;
      const uint32_t dst = en.off[lane];
      for (int l = pw; l < static_cast<int>(nseg); l += kLbPlaceWarps) {
        const uint32_t sl = __shfl_sync(0xffffffffu, seg, l);
        const uint32_t dl = __shfl_sync(0xffffffffu, dst, l);
        const uint32_t cl = lb_seg_count(sl), first = lb_seg_first(sl);
        const bool slotted = lb_seg_slot(sl);
        const uint32_t fbase = static_cast<uint32_t>(l & (kSWarps - 1)) * L::kFifo;
        const size_t sbase =
            (static_cast<size_t>(en.group * kLbGroupTiles) * kSWarps + l) * kSWarpElems;
        for (uint32_t k = lane; k < cl; k += 32) {
          uint2 x;
          if (slotted) {
            x = la.slot[sbase + k];  // written by a warp of this CTA (ordered by the barriers)
          } else {
            uint32_t b = first + k;
            if (b >= L::kFifo) b -= L::kFifo;
            x = f_pair[fbase + b];
          }
          const uint32_t pos = dl + k;
          if (pos < cap) {
            if constexpr (Op::kKeepPairs) {
              st_pair_policy(idx_out + pos, val_out + pos, x.x, __uint_as_float(x.y), keep_policy);
            } else {
              idx_out[pos] = x.x;
              val_out[pos] = __uint_as_float(x.y);
            }
          } else {
            overflow = true;
          }
        }
      }
      __syncwarp();  // every lane has read its pairs and the entry
      uint32_t before = 0;
      if (lane == 0) {
        __threadfence_block();
        before = atomicAdd(&en.placed, 1u);
      }
      before = __shfl_sync(0xffffffffu, before, 0);
      if (before == kLbPlaceWarps - 1) {
        __threadfence_block();  // the other placers' reads, before the space is handed back
        const uint32_t in_buffer = lb_seg_slot(seg) ? 0u : lb_seg_count(seg);
        const uint32_t both = in_buffer + __shfl_down_sync(0xffffffffu, in_buffer, kSWarps);
        if (lane < kSWarps) atomicAdd(&s_freed[lane], both);
        __syncwarp();
        if (lane == 0) mbar_arrive(&s_free[slot]);
      }
    }
    if (__any_sync(0xffffffffu, overflow) && lane == 0) atomicOr(ctx.error, kDevErrOverflow);
  } else {
    // ------------------------------------------------------ compute warps
    uint2* const my_pair = f_pair + warp * L::kFifo;
    uint32_t tail = 0;      // next buffer position this warp writes
    uint32_t appended = 0;  // pairs appended so far (the placer counts the freed ones)
    FF warp_err{0.0f, 0.0f};  // lane 0: share of ||e'||^2 in the current group

    // A group's tiles arrive in consecutive ring uses; each tile is computed
    // and its stage released at once, and the group's bookkeeping (positions,
    // buffer, counts, arrival) is done once for both tiles.
    auto compute_tile = [&](int s, uint32_t t, float (&a)[kSUnits][4],
                            uint32_t (&sel)[kSUnits]) {
      if (op.full(t)) {
        op.tile_smem(smem + s * Op::kStageBytes, t, warp, lane, a, sel, aux);
      } else {
        op.tile_global(t, warp, lane, a, sel, aux);
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(&s_empty[s]);  // this warp is done with the stage
      if (la.err_out) {
        float sq = 0.0f;
#pragma unroll
        for (int v = 0; v < kSUnits; ++v)
#pragma unroll
          for (int j = 0; j < 4; ++j)
            if (!((sel[v] >> j) & 0x11u)) sq = __fmaf_rn(a[v][j], a[v][j], sq);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
        if (lane == 0) warp_err = ff_add(warp_err, FF{sq, 0.0f});
      }
    };
    static_assert(kSUnits == 2 && kLbGroupTiles == 2, "four units of a group packed in one scan");
    for (uint32_t r = 0;;) {
      int s = static_cast<int>(r % kStages);
      bool arrived = lb_mbar_wait(&s_full[s], (r / kStages) & 1u, &s_failed, ctx);
      if (!__all_sync(0xffffffffu, arrived)) break;
      const uint32_t t0 = s_stage_tile[s];
      const uint32_t slot = s_stage_slot[s];
      if (t0 == kLbStageEnd) {
        if (lane == 0) mbar_arrive(&s_counted[slot]);  // the end mark, for the other roles
        break;
      }
      LbEntry& en = ent[slot];
      const uint32_t nt = en.ntiles;
      float a[kLbGroupTiles][kSUnits][4];
      uint32_t sel[kLbGroupTiles][kSUnits] = {{0u, 0u}, {0u, 0u}};
      compute_tile(s, t0, a[0], sel[0]);
      ++r;
      if (nt == 2) {
        s = static_cast<int>(r % kStages);
        arrived = lb_mbar_wait(&s_full[s], (r / kStages) & 1u, &s_failed, ctx);
        if (!__all_sync(0xffffffffu, arrived)) break;
        compute_tile(s, t0 + 1, a[1], sel[1]);
        ++r;
      }
      // positions in coordinate order: one warp scan of the four units'
      // per-lane counts (at most 4 each, 128 a warp) packed in bytes
      const uint32_t cnt4 = __popc(sel[0][0] & 0xfu) | (__popc(sel[0][1] & 0xfu) << 8) |
                            (__popc(sel[1][0] & 0xfu) << 16) | (__popc(sel[1][1] & 0xfu) << 24);
      uint32_t incl4 = cnt4;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t x = __shfl_up_sync(0xffffffffu, incl4, o);
        if (lane >= o) incl4 += x;
      }
      const uint32_t all4 = __shfl_sync(0xffffffffu, incl4, 31);
      const uint32_t excl4 = incl4 - cnt4;
      const uint32_t u0 = all4 & 0xffu, u1 = (all4 >> 8) & 0xffu;
      const uint32_t u2 = (all4 >> 16) & 0xffu, u3 = all4 >> 24;
      const uint32_t seg_total[kLbGroupTiles] = {u0 + u1, u2 + u3};
      // each unit's first position within its tile's segment
      const uint32_t off[kLbGroupTiles][kSUnits] = {
          {excl4 & 0xffu, u0 + ((excl4 >> 8) & 0xffu)},
          {(excl4 >> 16) & 0xffu, u2 + (excl4 >> 24)}};
      // each segment's pairs go to the warp's buffer when it has room (the
      // placer frees it group by group), else to the segment's global slot;
      // bit q of to_slot: segment q goes to its slot
      uint32_t to_slot = 0;
      if ((seg_total[0] | seg_total[1]) && lane == 0) {
        const uint32_t held = appended - vld(s_freed[warp]);
        if (held + seg_total[0] > L::kFifo) to_slot |= 1u;
        const uint32_t held1 = held + ((to_slot & 1u) ? 0u : seg_total[0]);
        if (held1 + seg_total[1] > L::kFifo) to_slot |= 2u;
        if (to_slot != 3u) __threadfence_block();  // the buffer writes after the placer's reads
      }
      to_slot = __shfl_sync(0xffffffffu, to_slot, 0);
      __syncwarp();
      const uint32_t buf_total = ((to_slot & 1u) ? 0u : seg_total[0]) +
                                 ((to_slot & 2u) ? 0u : seg_total[1]);
      // each lane writes its selected pairs in coordinate order, one set
      // selection bit at a time (at a few percent density most lanes have
      // none, and the warp takes as many rounds as its fullest lane)
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const uint32_t t = t0 + q;
        const uint32_t first_elem =
            static_cast<uint32_t>(stream_element_index(t, warp, 0, lane, 0)) - op.shift();
        if ((to_slot >> q) & 1u) {
          const size_t sb = (static_cast<size_t>(t) * kSWarps + warp) * kSWarpElems;
#pragma unroll
          for (int v = 0; v < kSUnits; ++v) {
            uint32_t p = off[q][v];
            for (uint32_t bits = sel[q][v] & 0xfu; bits; bits &= bits - 1, ++p) {
              const int j = __ffs(bits) - 1;
              la.slot[sb + p] =
                  make_uint2(first_elem + v * 128 + j, __float_as_uint(lb_pick(a[q][v], j)));
            }
          }
        } else {
#pragma unroll
          for (int v = 0; v < kSUnits; ++v) {
            uint32_t p = tail + ((q && !(to_slot & 1u)) ? seg_total[0] : 0u) + off[q][v];
            if (p >= L::kFifo) p -= L::kFifo;
            for (uint32_t bits = sel[q][v] & 0xfu; bits; bits &= bits - 1) {
              const int j = __ffs(bits) - 1;
              my_pair[p] =
                  make_uint2(first_elem + v * 128 + j, __float_as_uint(lb_pick(a[q][v], j)));
              if (++p == L::kFifo) p = 0;
            }
          }
        }
      }
      __syncwarp();  // every lane's pairs before the arrival
      if (lane == 0) {
        en.seg[warp] = lb_seg(seg_total[0], to_slot & 1u, tail);
        uint32_t first1 = tail + ((to_slot & 1u) ? 0u : seg_total[0]);
        if (first1 >= L::kFifo) first1 -= L::kFifo;
        if (nt == 2) en.seg[kSWarps + warp] = lb_seg(seg_total[1], to_slot & 2u, first1);
        if (la.err_out) {
          en.err[warp] = warp_err;
          warp_err = FF{0.0f, 0.0f};
        }
        mbar_arrive(&s_counted[slot]);  // releases the pairs and the words
      }
      tail += buf_total;
      if (tail >= L::kFifo) tail -= L::kFifo;
      appended += buf_total;
    }
  }

  if (!la.err_out) return;
  // every CTA counts itself finished, with its resolved groups; the last one
  // adds the groups' error shares when every group was resolved
  __syncthreads();
  if (threadIdx.x == 0) {
    atomicAdd(la.err_count, s_resolved);
    __threadfence();
    s_last = atomicAdd(la.err_count + 1, 1u) == gridDim.x - 1 ? 1u : 0u;
    if (s_last) {
      __threadfence();
      s_resolved = atomicAdd(la.err_count, 0u);
      la.err_count[0] = 0;
      la.err_count[1] = 0;
    }
  }
  __syncthreads();
  if (s_last) {
    __threadfence();
    const bool ok = s_resolved == G;
    const FF err = sum_parts_ff(la.err_parts, ok ? G : 0u, s_err_sum);
    if (threadIdx.x == 0) *la.err_out = ok ? ff_to_double(err) : err_invalid();
  }
}

}  // namespace efs
