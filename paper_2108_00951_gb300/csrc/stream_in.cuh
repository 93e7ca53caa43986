// stream_in.cuh — the inputs of a streaming pass: g and e at any element
// alignment, read tile by tile through 16-byte aligned bulk copies.
//
// The streaming kernels work on positions p = j + shift of the coordinates
// j in [0, d). shift (0..3, with a bf16 g 0..7) is what makes e + j 16-byte
// aligned at every p that is a multiple of 4, so a tile is a whole number of
// aligned 16-byte words of e whatever e's base: rows of an [n, d] matrix with
// an odd d, or a tensor's slice of a flat buffer, stream like an aligned
// vector. Position 0 (at most 7 coordinates before the vector) and the end
// fall into partial tiles, which are read and written coordinate by
// coordinate; every full tile lies inside the vector.
//
// g is aligned by the same shift when g and e start at the same place of
// their 16-byte words (rows or slices cut alike); otherwise its tile starts
// g_sub elements into a word. The copy then takes one more word, and the
// reading threads pick their four values out of two words in shared memory.
// Such a copy reads up to 15 bytes before or after the tile's part of g, of
// aligned 16-byte words that also hold elements of it (so never of another
// page), and nothing uses them.
//
// Both are compiled out of the aligned case's kernels (kAny false): the
// run-time choice in the tile loop cost them 1 to 3 % (ResNet-18-shaped
// iteration 255.4 -> 258.4 us, VGG-16-shaped bf16 call 236.0 -> 242.6 us).
//
// A gradient cut unlike its error memory costs its second word a read: d =
// 11.2 M, us a call aligned, g and e shifted alike, shifted unlike: hard-threshold
// at 36 % sent 30.4, 30.4, 31.5 (bf16 g 29.0, 29.0, 30.0), Top-k at 1 % 56.1,
// 57.1, 58.4; at 28.9 M all three within 2 % of one another.
//
// Measured on a GB300 (LSTM-shaped vector, d = 28.9 M, 3 % sent, us per call):
// rows 1..3 of [4, d] matrices (12, 8 and 4 bytes past a word) 280 with the
// one-tile-per-CTA kernel that misaligned vectors used before, 66 for row 0;
// four such workers' calls and their exchange went from 991 to 337 (and to 290
// with what the exchange and the claimed-group kernel gained since).
#pragma once

#include "gradient.cuh"
#include "tma.cuh"

namespace efs {

template <typename GT, bool kAny>
struct StreamIn {
  const GT* g;      // 16-byte aligned; position p is at g[p + sub()]
  float* e;         // 16-byte aligned; position p is at e[p]
  uint64_t end;     // positions [shift(), end) are the coordinates
  uint32_t n_full;  // full tiles: the first ones, or those after tile 0 with a shift
  uint32_t shift_, sub_;  // read by kAny kernels only (0 otherwise)
  static constexpr uint32_t kGBytes = kTileElems * sizeof(GT);
  static constexpr uint32_t kEBytes = kTileElems * sizeof(float);
  // a stage: a tile of e, then of g, then room for one more word of g; a
  // whole number of 128-byte lines, so that every copy fills whole lines
  static constexpr uint32_t kStageBytes = kEBytes + kGBytes + (kAny ? 128 : 0);

  __device__ __forceinline__ uint32_t shift() const { return kAny ? shift_ : 0u; }
  __device__ __forceinline__ uint32_t sub() const { return kAny ? sub_ : 0u; }
  // the tile's positions are all coordinates
  __device__ __forceinline__ bool full(uint32_t t) const {
    return kAny ? t - (shift_ ? 1u : 0u) < n_full : t < n_full;
  }
  __device__ __forceinline__ bool valid(uint64_t p) const {
    return (!kAny || p >= shift_) && p < end;
  }
  __device__ __forceinline__ void prefetch(uint32_t t) const {
    prefetch_l2_1d(g + static_cast<size_t>(t) * kTileElems, kGBytes);
    prefetch_l2_1d(e + static_cast<size_t>(t) * kTileElems, kEBytes);
  }
  // bulk copies of a full tile into a stage, completing on bar
  __device__ __forceinline__ void fill(unsigned char* stage, uint32_t t, uint64_t* bar,
                                       uint64_t policy) const {
    const uint32_t gb = sub() ? kGBytes + 16u : kGBytes;
    mbar_arrive_expect_tx(bar, gb + kEBytes);
    tma_load_1d(stage + kEBytes, g + static_cast<size_t>(t) * kTileElems, gb, bar, policy);
    tma_load_1d(stage, e + static_cast<size_t>(t) * kTileElems, kEBytes, bar, policy);
  }
  // a of the 4 positions from `local` (a multiple of 4) of a staged tile
  __device__ __forceinline__ void accumulate(const unsigned char* stage, int local, float gamma,
                                             float (&a)[4]) const {
    const GT* gs = reinterpret_cast<const GT*>(stage + kEBytes);
    const float4 ev = *reinterpret_cast<const float4*>(stage + local * sizeof(float));
    GradVec<GT> gv;
    if (sub() == 0)
      gv.load_aligned(gs + local);
    else
      gv.load_at(gs + local, sub());
    a[0] = __fmaf_rn(gamma, gv[0], ev.x);
    a[1] = __fmaf_rn(gamma, gv[1], ev.y);
    a[2] = __fmaf_rn(gamma, gv[2], ev.z);
    a[3] = __fmaf_rn(gamma, gv[3], ev.w);
  }
  // a of position p, straight from memory
  __device__ __forceinline__ float accumulate_at(uint64_t p, float gamma) const {
    return __fmaf_rn(gamma, grad_scalar(g, p + sub()), e[p]);
  }
  // a of the 4 positions from p (a multiple of 4, all of them coordinates),
  // straight from memory through the read-only path (the samplings)
  __device__ __forceinline__ void load4(uint64_t p, GradVec<GT>& gv, float4& ev) const {
    if (sub() == 0)
      gv.load_readonly(g + p);
    else
      gv.load_scalars(g + p + sub());
    ev = __ldg(reinterpret_cast<const float4*>(e + p));
  }
};

// The positions of a call (host).
struct Positions {
  uint32_t shift, sub;
  bool any() const { return shift != 0 || sub != 0; }
  uint64_t end(uint32_t d) const { return static_cast<uint64_t>(d) + shift; }
};
template <typename GT>
Positions positions(const GT* g, const float* e) {
  constexpr uint32_t kWord = 16 / sizeof(GT);  // elements of g per 16-byte word
  const uint32_t ge = static_cast<uint32_t>(reinterpret_cast<uintptr_t>(g) / sizeof(GT) % kWord);
  uint32_t shift = static_cast<uint32_t>(reinterpret_cast<uintptr_t>(e) / sizeof(float) % 4);
  // with a bf16 g two shifts align e; take the one that aligns g, if any does
  if (kWord == 8 && ge == shift + 4) shift += 4;
  return Positions{shift, (ge + kWord - shift) % kWord};
}
template <typename GT, bool kAny>
StreamIn<GT, kAny> stream_in(const GT* g, float* e, uint32_t d) {
  const Positions p = positions(g, e);
  const uint32_t whole = static_cast<uint32_t>(p.end(d) / kTileElems);
  const uint32_t first = p.shift ? 1u : 0u;
  return StreamIn<GT, kAny>{g - p.shift - p.sub, e - p.shift, p.end(d),
                            whole > first ? whole - first : 0u, p.shift, p.sub};
}

}  // namespace efs
