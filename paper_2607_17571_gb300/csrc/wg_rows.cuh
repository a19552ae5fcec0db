// wg_rows.cuh -- adjacency units and the expansion of vertex lists into bit sets,
// shared by the row-by-row fixpoints (wg_kern_rows.cu, wg_kern_sg.cu).
#pragma once
#include "wg_device.cuh"

namespace wg {

// Adjacency in units of 16 bytes (U = 8 16-bit or 4 32-bit ranks).  Each vertex
// has a record {degree (16 bits saturate), its first U-1 neighbours}: one load
// gives most vertices' whole adjacency.  Its further neighbours lie in units from
// (off[v] + (U-1) v + U-1) / U: room for every vertex before it without a scan.
// Unused places repeat the vertex's last neighbour (setting a bit twice is
// harmless).
template <typename IdT> struct Unit { static constexpr uint32_t n = 16 / sizeof(IdT); };
template <typename IdT>
__device__ __forceinline__ uint32_t unit_start(uint32_t off, uint32_t v) {
  constexpr uint32_t U = Unit<IdT>::n;
  return (off + (U - 1) * (v + 1)) / U;
}
__device__ __forceinline__ void set_bit(uint32_t* n, uint32_t byte_off, uint32_t z) {
  atomicOr((uint32_t*)((char*)n + byte_off), __funnelshift_l(0u, 1u, z));  // 1 << (z & 31)
}
// The bits of the two 16-bit ranks, or the 32-bit rank, in a word.
__device__ __forceinline__ void set_part(uint32_t* n, uint32_t v, uint16_t) {
  set_bit(n, (v >> 3) & 0x1FFCu, v);
  set_bit(n, (v >> 19) & 0x1FFCu, v >> 16);
}
__device__ __forceinline__ void set_part(uint32_t* n, uint32_t v, uint32_t) {
  set_bit(n, (v >> 3) & ~3u, v);
}
// A vertex's record: its degree, and the bits of its neighbours there (pairs by
// the lane's own degree: the shared atomics, not the tests, are the scarce part).
template <typename IdT> struct Rec;
template <> struct Rec<uint16_t> {
  uint4 a;
  __device__ __forceinline__ void load(const void* rec, uint32_t v) { a = __ldg((const uint4*)rec + v); }
  __device__ __forceinline__ uint32_t deg() const { return a.x & 0xFFFFu; }
  __device__ __forceinline__ void set(uint32_t* n, uint32_t deg) const {
    set_bit(n, (a.x >> 19) & 0x1FFCu, a.x >> 16);
    if (deg > 1) set_part(n, a.y, uint16_t());
    if (deg > 3) set_part(n, a.z, uint16_t());
    if (deg > 5) set_part(n, a.w, uint16_t());
  }
};
template <> struct Rec<uint32_t> {
  uint4 a;
  __device__ __forceinline__ void load(const void* rec, uint32_t v) { a = __ldg((const uint4*)rec + v); }
  __device__ __forceinline__ uint32_t deg() const { return a.x; }
  __device__ __forceinline__ void set(uint32_t* n, uint32_t deg) const {
    set_part(n, a.y, uint32_t());
    if (deg > 1) { set_part(n, a.z, uint32_t()); set_part(n, a.w, uint32_t()); }
  }
};

__device__ __forceinline__ uint32_t warp_incl_scan(uint32_t v, uint32_t lane) {
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, v, o);
    if (lane >= (uint32_t)o) v += y;
  }
  return v;
}

// The bits of the neighbours of a warp's vertices (lane: vertex v with record r of
// degree deg, 0: none) into the bit set N (shared memory): the records' own, then
// the vertices' units as one strip, 32 units per step, a lane finding its unit's
// vertex from the bit mask of the strip's first units.  strip: 32 words of the
// warp.  Returns the degree of the lane's vertex.
template <typename IdT>
__device__ __forceinline__ uint32_t expand_strip(const RowInst& I, uint32_t v, uint32_t deg,
                                                 const Rec<IdT>& r, uint32_t* N, uint32_t* strip) {
  constexpr uint32_t U = Unit<IdT>::n, kRecIds = U - 1;
  const uint32_t lane = threadIdx.x & 31, upto = 0xFFFFFFFFu >> (31 - lane);
  uint32_t us = 0;
  if (deg) {
    uint32_t o = 0, o1 = 0;
    if (deg > kRecIds) {
      o = __ldg(I.off + v);
      o1 = __ldg(I.off + v + 1);
    }
    r.set(N, deg);
    if (deg > kRecIds) {
      deg = o1 - o;
      us = unit_start<IdT>(o, v);
    }
  }
  const uint32_t more = deg > kRecIds ? (deg - kRecIds + U - 1) / U : 0u;  // units
  const uint32_t has = __ballot_sync(0xffffffffu, more > 0);
  if (!has) return deg;
  const uint32_t in = warp_incl_scan(more, lane);
  const uint32_t tot = __shfl_sync(0xffffffffu, in, 31), st = in - more;
  if (more) strip[__popc(has & upto) - 1] = us - st;
  __syncwarp();
  uint32_t prev = 0;  // vertices whose units begin before this step
  for (uint32_t e0 = 0; e0 < tot; e0 += 32) {
    const uint32_t sh = st - e0, e = e0 + lane;
    const uint32_t m = __reduce_or_sync(0xffffffffu, more && sh < 32u ? 1u << sh : 0u);
    const uint32_t t = strip[prev + __popc(m & upto) - 1];
    prev += __popc(m);
    if (e < tot) {
      const uint4 u = __ldg((const uint4*)I.units + (t + e));
      set_part(N, u.x, IdT());
      set_part(N, u.y, IdT());
      set_part(N, u.z, IdT());
      set_part(N, u.w, IdT());
    }
  }
  __syncwarp();
  return deg;
}

// The bits of the neighbours of the vertices l[b..n), l[b + step..n), ..., 32 at
// most each, every one with neighbours.  One warp; returns the sum of the degrees
// of the lane's vertices.  kAhead: the next 32 records are loaded before the bits
// of these are set (same-generation rows, few warps per SM: 1.35 -> 1.32 ms; TC rows
// gain nothing and R-MAT 2^17 / 400k loses 1%).
template <typename IdT, bool kAhead>
__device__ __forceinline__ uint32_t expand_vertices(const RowInst& I, const IdT* l, uint32_t b,
                                                    uint32_t n, uint32_t step, uint32_t* N,
                                                    uint32_t* strip) {
  const uint32_t lane = threadIdx.x & 31;
  uint32_t sum = 0, v = 0;
  Rec<IdT> r;
  auto load = [&](uint32_t at) {
    r.a = uint4{0, 0, 0, 0};
    if (at + lane < n) {
      v = l[at + lane];
      r.load(I.rec, v);
    }
  };
  if (kAhead) load(b);
  for (; b < n; b += step) {
    if (!kAhead) load(b);
    const uint32_t v0 = v;
    const Rec<IdT> r0 = r;
    if (kAhead) load(b + step);
    sum += expand_strip<IdT>(I, v0, r0.deg(), r0, N, strip);
  }
  return sum;
}

// The set bits of a row's mask (at most 32 words) as an ordered list; returns
// their number.  One warp.
__device__ __forceinline__ uint32_t list_pieces(uint32_t m, uint16_t* to) {
  const uint32_t lane = threadIdx.x & 31, c = __popc(m), sum = warp_incl_scan(c, lane);
  for (uint32_t at = sum - c; m; m &= m - 1) to[at++] = (uint16_t)(lane * 32 + __ffs(m) - 1);
  return __shfl_sync(0xffffffffu, sum, 31);
}

}  // namespace wg
