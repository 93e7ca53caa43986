// ht.cu — the fused error-feedback + hard-threshold + compaction kernel.
//
// One pass over the d coordinates performs, per coordinate j (Algorithm 1
// with the hard-threshold sparsifier of Sec. 1 / Sec. 4.2):
//   a_j  = fmaf(gamma, g_j, e_j)                 corrected update p = e + gamma g
//   s_j  = (|a_j| >= lambda) and (a_j != 0)      j in S_lambda(a)
//   e_j <- s_j ? +0 : a_j                        error update e <- p - C(p)
// and writes the selected (j, a_j) pairs in ascending j through the ordered
// compaction. HBM traffic per coordinate is the algorithmic minimum: read g
// (4 B, or 2 B for bf16) and e (4 B), write e (4 B); plus 8 B per sent pair.
#include <algorithm>

#include "compact.cuh"
#include "internal.h"
#include "stream_lookback.cuh"

namespace efs {
namespace {

__device__ __forceinline__ uint32_t in_support(float a, float lambda) {
  return (fabsf(a) >= lambda && a != 0.0f) ? 1u : 0u;
}

// One tile per CTA with the decoupled look-back of compact.cuh: the
// allocation-free entry's kernel (its scratch is one status word per tile).
template <bool kVec>
__global__ void __launch_bounds__(kThreads)
    ht_kernel(const float* __restrict__ g, float* __restrict__ e, float gamma, float lambda,
              uint32_t d, uint32_t* __restrict__ idx_out, float* __restrict__ val_out,
              uint32_t* __restrict__ count_out, ScanCtx ctx) {
  // The tile comes from the dispenser, in the order CTAs start, so every
  // lower tile this CTA's look-back waits for is held by a running CTA.
  __shared__ uint32_t s_tile;
  if (threadIdx.x == 0) s_tile = atomicAdd(ctx.tile_claim, 1u);
  __syncthreads();
  const uint32_t tile = s_tile;
  if (tile >= ctx.num_tiles) {
    // the dispenser did not start at zero (an earlier launch was cut short):
    // touch nothing, report it, and still count this CTA as finished
    if (threadIdx.x == 0) {
      atomicOr(ctx.error, kDevErrTimeout);
      if (atomicAdd(ctx.tile_claim + 1, 1u) == gridDim.x - 1) {
        ctx.tile_claim[0] = 0;
        ctx.tile_claim[1] = 0;
      }
    }
    return;
  }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint64_t first = element_index(tile, warp, 0, lane, 0);

  float a[kUnits][4];
  uint32_t sel[kUnits];
  const bool full_tile = static_cast<uint64_t>(tile + 1) * kTileElems <= d;

  if (kVec && full_tile) {
    GradVec<float> gv[kUnits];
    float4 ev[kUnits];
#pragma unroll
    for (int v = 0; v < kUnits; ++v) {  // all loads in flight before any use
      gv[v].load(g + first + v * 128);
      ev[v] = ld_stream_f4(e + first + v * 128);
    }
#pragma unroll
    for (int v = 0; v < kUnits; ++v) {
      a[v][0] = __fmaf_rn(gamma, gv[v][0], ev[v].x);
      a[v][1] = __fmaf_rn(gamma, gv[v][1], ev[v].y);
      a[v][2] = __fmaf_rn(gamma, gv[v][2], ev[v].z);
      a[v][3] = __fmaf_rn(gamma, gv[v][3], ev[v].w);
      sel[v] = in_support(a[v][0], lambda) | (in_support(a[v][1], lambda) << 1) |
               (in_support(a[v][2], lambda) << 2) | (in_support(a[v][3], lambda) << 3);
      const float4 r = make_float4((sel[v] & 1u) ? 0.0f : a[v][0], (sel[v] & 2u) ? 0.0f : a[v][1],
                                   (sel[v] & 4u) ? 0.0f : a[v][2], (sel[v] & 8u) ? 0.0f : a[v][3]);
      st_stream_f4(e + first + v * 128, r);
    }
  } else {
#pragma unroll
    for (int v = 0; v < kUnits; ++v) {
      sel[v] = 0;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const uint64_t i = first + v * 128 + j;
        a[v][j] = 0.0f;
        if (i < d) {
          const float x = __fmaf_rn(gamma, grad_scalar(g, i), e[i]);
          const uint32_t s = in_support(x, lambda);
          a[v][j] = x;
          sel[v] |= s << j;
          e[i] = s ? 0.0f : x;
        }
      }
    }
  }
  compact_tile(ctx, tile, sel, a, idx_out, val_out, count_out, d);
  if (threadIdx.x == 0) {
    // every CTA took its tile before it counts itself finished; the last one
    // leaves the dispenser at zero for the next launch
    __threadfence();
    if (atomicAdd(ctx.tile_claim + 1, 1u) == gridDim.x - 1) {
      ctx.tile_claim[0] = 0;
      ctx.tile_claim[1] = 0;
    }
  }
}

// The hard-threshold step as a streaming-compaction op: a stage holds a
// tile of g followed by the same tile of e; the residual is written to e from
// registers with streaming stores.
template <typename GT, bool kAny>
struct HtOp : StreamIn<GT, kAny> {
  float gamma, lambda;
  static constexpr uint32_t kWarpStagePairs = 768;  // on-chip staged pairs per compute warp
  static constexpr bool kKeepPairs = false;  // the message: read by the exchange, much later
  // the chunk's first tiles of g and e toward L2 before the wait for the
  // previous kernel (its tail leaves DRAM mostly idle)
  static constexpr uint32_t kPrefetchTiles = 8;
  __device__ void prologue() const {}
  __device__ uint64_t initial_aux() const { return 0; }

  __device__ __forceinline__ void tile_smem(const unsigned char* stage, uint32_t t, int warp,
                                            int lane, float (&a)[kSUnits][4],
                                            uint32_t (&sel)[kSUnits], uint64_t) const {
    const int local = warp * kSWarpElems + lane * 4;
    float* eg = this->e + stream_element_index(t, warp, 0, lane, 0);
    // with lambda > 0, |a| >= lambda already excludes a == 0 (and NaN): one
    // comparison a coordinate; lambda == 0 keeps the a != 0 test
    const bool pos = lambda > 0.0f;
#pragma unroll
    for (int v = 0; v < kSUnits; ++v) {
      this->accumulate(stage, local + v * 128, gamma, a[v]);
      bool s[4];
#pragma unroll
      for (int j = 0; j < 4; ++j)
        s[j] = pos ? fabsf(a[v][j]) >= lambda : in_support(a[v][j], lambda) != 0u;
      sel[v] = (s[0] ? 1u : 0u) | (s[1] ? 2u : 0u) | (s[2] ? 4u : 0u) | (s[3] ? 8u : 0u);
      st_stream_f4(eg + v * 128, make_float4(s[0] ? 0.0f : a[v][0], s[1] ? 0.0f : a[v][1],
                                             s[2] ? 0.0f : a[v][2], s[3] ? 0.0f : a[v][3]));
    }
  }

  __device__ __forceinline__ void tile_global(uint32_t t, int warp, int lane,
                                              float (&a)[kSUnits][4],
                                              uint32_t (&sel)[kSUnits], uint64_t) const {
    const uint64_t first = stream_element_index(t, warp, 0, lane, 0);
#pragma unroll
    for (int v = 0; v < kSUnits; ++v) {
      sel[v] = 0;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const uint64_t i = first + v * 128 + j;
        a[v][j] = 0.0f;
        if (this->valid(i)) {
          const float x = this->accumulate_at(i, gamma);
          const uint32_t sj = in_support(x, lambda);
          a[v][j] = x;
          sel[v] |= sj << j;
          this->e[i] = sj ? 0.0f : x;
        }
      }
    }
  }
};

// ring stages: 4 of 32 KB (fp32 g); bf16 g makes a stage 24 KB, and a fifth
// stage keeps about as many bytes in flight within the same shared memory
template <typename GT>
constexpr int kHtStages = sizeof(GT) == 2 ? 5 : 4;

// group entries: the shallow ring is the dense calls'
template <typename GT, int kStages>
constexpr int kHtEntries = kStages < kHtStages<GT> ? kLbFewEntries : kLbManyEntries;

template <typename GT, bool kAny, int kStages = kHtStages<GT>>
using HtGroupKernel = LbLayout<HtOp<GT, kAny>, kStages, kHtEntries<GT, kStages>>;
template <typename GT, bool kAny>
using HtChunkKernel = StreamLayout<HtOp<GT, kAny>, kHtStages<GT>>;

// Streaming hard-threshold over dynamically claimed groups of tiles: one CTA
// per SM. A group waits only for groups claimed before it, held by running
// CTAs, so the launch needs no co-residency. Programmatic: it may start while
// the previous kernel on the stream finishes (the kernel waits for it before
// its first read). kStages: the ring depth (one stage fewer for dense calls,
// whose pair buffers then take the freed shared memory).
template <int kStages, typename GT, bool kAny>
cudaError_t launch_groups(const StreamIn<GT, kAny>& in, float gamma, float lambda, uint32_t d,
                          uint32_t* idx_out, float* val_out, uint32_t* count_out, double* err_out,
                          uint32_t* tiles_out, Workspace& ws, const DeviceInfo& dev,
                          const ScanCtx& ctx, int per_sm) {
  HtOp<GT, kAny> op{in, gamma, lambda};
  const uint32_t tiles = ctx.num_tiles;
  const uint32_t groups = (tiles + kLbGroupTiles - 1) / kLbGroupTiles;
  const uint32_t slots = static_cast<uint32_t>(per_sm * dev.sm_count);
  const uint32_t grid = groups < slots ? groups : slots;
  uint32_t cap = d;
  ScanCtx c = ctx;
  LbArgs la;
  cudaError_t err = lb_args(ws, tiles_out, err_out, ws.density_dev, &la);
  if (err != cudaSuccess) return err;
  void* params[] = {&op, &idx_out, &val_out, &count_out, &cap, &c, &la};
  err = launch_pdl(
      reinterpret_cast<const void*>(
          &lookback_stream_kernel<HtOp<GT, kAny>, kStages, kHtEntries<GT, kStages>>),
      grid, kLbThreads, HtGroupKernel<GT, kAny, kStages>::kSmem, ws.stream, params, false);
  count_launch();
  ws.ht_part_ready = false;  // the chunk kernel's boundaries are not written by this kernel
  return err;
}

// Streaming hard-threshold over static chunks (stream_compact.cuh): one CTA
// per SM, CTA c waiting only on the chunk totals of lower-numbered CTAs. The
// grid fits the device at once and CTAs are dispatched in index order, so
// those CTAs are running; if other work holds SMs long enough that one cannot
// start, the bounded wait ends the call with EF_ERR_TIMEOUT (never a hang or a
// wrong result). Balanced chunks: the previous call of this size wrote this
// call's chunk boundaries from its chunk totals (dense regions get fewer
// tiles); any boundaries partition the tiles, so the result never depends on
// them.
template <typename GT, bool kAny>
cudaError_t launch_chunks(const StreamIn<GT, kAny>& in, float gamma, float lambda, uint32_t d,
                          uint32_t* idx_out, float* val_out, uint32_t* count_out, double* err_out,
                          uint32_t* tiles_out, Workspace& ws, const DeviceInfo& dev,
                          const ScanCtx& ctx, int per_sm) {
  HtOp<GT, kAny> op{in, gamma, lambda};
  const uint32_t tiles = ctx.num_tiles;
  uint32_t slots = static_cast<uint32_t>(per_sm * dev.sm_count);
  if (slots > kMaxChunks) slots = kMaxChunks;
  const uint32_t grid = tiles < slots ? tiles : slots;
  uint32_t cap = d;
  ScanCtx c = ctx;
  StreamArgs sa{ws.stage_idx(), ws.stage_val(), ws.counts(), ws.ht_chunks(ws.ht_seq), tiles_out,
                err_out, ws.errparts()};
  const uint32_t seq = ws.ht_seq;
  const bool same = seq > 0 && ws.ht_last_tiles == tiles && ws.ht_last_grid == grid;
  // (a call that returns ||e'||^2 uses equal chunks: the norm's summation
  // order follows the chunks, and it is reproducible for an input)
  sa.part_in = same && ws.ht_part_ready && !err_out ? ws.ht_part(seq) : nullptr;
  sa.prev_sums = same ? ws.ht_chunks(seq + 1) : nullptr;   // the other parity: seq - 1
  sa.prev_part = same && ws.ht_prev_balanced ? ws.ht_part(seq + 2) : nullptr;  // seq - 1
  sa.prev_epoch = ws.ht_last_epoch;
  sa.part_out = ws.ht_part(seq + 1);
  sa.density_out = ws.density_dev;
  void* params[] = {&op, &idx_out, &val_out, &count_out, &cap, &c, &sa};
  const cudaError_t err = launch_pdl(
      reinterpret_cast<const void*>(&stream_compact_kernel<HtOp<GT, kAny>, kHtStages<GT>>), grid,
      kStreamThreads, HtChunkKernel<GT, kAny>::kSmem, ws.stream, params, false);
  count_launch();
  ws.ht_prev_balanced = sa.part_in != nullptr;
  ws.ht_part_ready = err == cudaSuccess;
  ws.ht_last_tiles = tiles;
  ws.ht_last_grid = grid;
  ws.ht_last_epoch = c.epoch;
  ++ws.ht_seq;
  return err;
}

template <bool kAny, typename GT>
cudaError_t launch_typed(const GT* g, float* e, float gamma, float lambda, uint32_t d,
                         uint32_t* idx_out, float* val_out, uint32_t* count_out, double* err_out,
                         uint32_t* tiles_out, Workspace& ws, const DeviceInfo& dev) {
  const StreamIn<GT, kAny> in = stream_in<GT, kAny>(g, e, d);
  const uint32_t tiles = tiles_for(in.end);
  const ScanCtx ctx = next_scan_ctx(ws, tiles);
  // the kernels' tile index is that of positions: with a shift, the message's
  // comes from its list instead
  uint32_t* kernel_tiles = in.shift_ == 0 ? tiles_out : nullptr;
  const int per_group = sizeof(GT) == 4 ? dev.ht_group_per_sm_f32 : dev.ht_group_per_sm_bf16;
  const int per_dense = sizeof(GT) == 4 ? dev.ht_dense_per_sm_f32 : dev.ht_dense_per_sm_bf16;
  const int per_chunk = sizeof(GT) == 4 ? dev.ht_stream_per_sm_f32 : dev.ht_stream_per_sm_bf16;
  cudaError_t err = cudaErrorInvalidConfiguration;
  const int mode = stream_kernel_mode();
  const bool dense_hint = mode == 0 && ws.density_host &&
                          *static_cast<volatile uint32_t*>(ws.density_host) >= kDenseRingHint;
  // (a norm's summation order is the kernel's: with one, the size alone decides)
  const bool groups =
      per_group > 0 && (use_group_kernel(tiles) ||
                        (dense_hint && tiles >= kDenseGroupMinTiles && !err_out));
  const bool dense = groups && per_dense > 0 && (mode == 3 || dense_hint);
  if (dense)
    err = launch_groups<kHtStages<GT> - 1>(in, gamma, lambda, d, idx_out, val_out, count_out,
                                               err_out, kernel_tiles, ws, dev, ctx, per_dense);
  else if (groups)
    err = launch_groups<kHtStages<GT>>(in, gamma, lambda, d, idx_out, val_out, count_out,
                                           err_out, kernel_tiles, ws, dev, ctx, per_group);
  else if (per_chunk > 0)
    err = launch_chunks(in, gamma, lambda, d, idx_out, val_out, count_out, err_out, kernel_tiles,
                        ws, dev, ctx, per_chunk);
  if (err == cudaSuccess && tiles_out && !kernel_tiles)
    err = launch_list_tiles(idx_out, count_out, d, tiles_out, ws);
  return err;
}

template <typename GT, typename Layout>
int blocks_per_sm(const void* fn, int threads) {
  int n = 0;
  if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, Layout::kSmem) !=
          cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, fn, threads, Layout::kSmem) != cudaSuccess)
    n = 0;
  cudaGetLastError();
  return n;
}

template <typename GT, bool kAny, int kStages>
int group_blocks() {
  return blocks_per_sm<GT, HtGroupKernel<GT, kAny, kStages>>(
      reinterpret_cast<const void*>(
          &lookback_stream_kernel<HtOp<GT, kAny>, kStages, kHtEntries<GT, kStages>>),
      kLbThreads);
}
template <typename GT, int kStages>
int group_blocks_per_sm() {
  return std::min(group_blocks<GT, false, kStages>(), group_blocks<GT, true, kStages>());
}
template <typename GT, bool kAny>
int chunk_blocks() {
  return blocks_per_sm<GT, HtChunkKernel<GT, kAny>>(
      reinterpret_cast<const void*>(&stream_compact_kernel<HtOp<GT, kAny>, kHtStages<GT>>),
      kStreamThreads);
}
template <typename GT>
int chunk_blocks_per_sm() {
  return std::min(chunk_blocks<GT, false>(), chunk_blocks<GT, true>());
}

}  // namespace

void ht_init_device(DeviceInfo& info) {
  info.ht_stream_per_sm_f32 = chunk_blocks_per_sm<float>();
  info.ht_stream_per_sm_bf16 = chunk_blocks_per_sm<uint16_t>();
  info.ht_group_per_sm_f32 = group_blocks_per_sm<float, kHtStages<float>>();
  info.ht_group_per_sm_bf16 = group_blocks_per_sm<uint16_t, kHtStages<uint16_t>>();
  info.ht_dense_per_sm_f32 = group_blocks_per_sm<float, kHtStages<float> - 1>();
  info.ht_dense_per_sm_bf16 = group_blocks_per_sm<uint16_t, kHtStages<uint16_t> - 1>();
}

// Launch the look-back kernel over caller-provided scratch (the tile-status
// words and the error word named by ctx); used by the allocation-free entry.
cudaError_t launch_hard_threshold_lookback(const float* g, float* e, float gamma, float lambda,
                                           uint32_t d, uint32_t* idx_out, float* val_out,
                                           uint32_t* count_out, const ScanCtx& ctx,
                                           cudaStream_t stream) {
  const uint32_t tiles = tiles_for(d);
  const bool vec = reinterpret_cast<uintptr_t>(g) % 16 == 0 &&
                   reinterpret_cast<uintptr_t>(e) % 16 == 0;
  if (vec)
    ht_kernel<true><<<tiles, kThreads, 0, stream>>>(g, e, gamma, lambda, d, idx_out,
                                                           val_out, count_out, ctx);
  else
    ht_kernel<false><<<tiles, kThreads, 0, stream>>>(g, e, gamma, lambda, d, idx_out,
                                                            val_out, count_out, ctx);
  count_launch();
  return cudaGetLastError();
}

cudaError_t launch_hard_threshold(const void* g, bool g_bf16, float* e, float gamma,
                                  float lambda, uint32_t d, uint32_t* idx_out, float* val_out,
                                  uint32_t* count_out, double* err_out, uint32_t* tiles_out,
                                  Workspace& ws, const DeviceInfo& dev) {
  auto run = [&](auto* gt) {
    return positions(gt, e).any()
               ? launch_typed<true>(gt, e, gamma, lambda, d, idx_out, val_out, count_out, err_out,
                                    tiles_out, ws, dev)
               : launch_typed<false>(gt, e, gamma, lambda, d, idx_out, val_out, count_out,
                                     err_out, tiles_out, ws, dev);
  };
  return g_bf16 ? run(static_cast<const uint16_t*>(g)) : run(static_cast<const float*>(g));
}

}  // namespace efs
