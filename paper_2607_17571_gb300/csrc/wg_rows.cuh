// wg_rows.cuh -- adjacency units and the expansion of vertex lists into bit sets,
// shared by the row-by-row fixpoints (wg_kern_rows.cu, wg_kern_sg.cu).
#pragma once
#include "wg_device.cuh"

namespace wg {

// Adjacency in units of 16 bytes (8 16-bit or 4 32-bit ranks).  Each vertex has
// a 32-byte record (one sector): {first further unit, degree, -, -} and its
// first unit, so one access gives most vertices' whole adjacency.  Its further
// units start at (off[v] + (U-1) v + U-1) / U: room for every vertex before it
// without a scan.  A unit's unused places repeat the vertex's last neighbour
// (setting a bit twice is harmless), so no place needs a test.
template <typename IdT> struct Unit { static constexpr uint32_t n = 16 / sizeof(IdT); };
template <typename IdT>
__device__ __forceinline__ uint32_t unit_start(uint32_t off, uint32_t v) {
  constexpr uint32_t U = Unit<IdT>::n;
  return (off + (U - 1) * (v + 1)) / U;
}
// The bits of places [2p, 2p + 2) of a unit (16-bit ranks) or place p (32-bit).
__device__ __forceinline__ void set_bit(uint32_t* n, uint32_t byte_off, uint32_t z) {
  atomicOr((uint32_t*)((char*)n + byte_off), __funnelshift_l(0u, 1u, z));  // 1 << (z & 31)
}
__device__ __forceinline__ void set_part(uint32_t* n, uint32_t v, uint16_t) {
  set_bit(n, (v >> 3) & 0x1FFCu, v);
  set_bit(n, (v >> 19) & 0x1FFCu, v >> 16);
}
__device__ __forceinline__ void set_part(uint32_t* n, uint32_t v, uint32_t) {
  set_bit(n, (v >> 3) & ~3u, v);
}

__device__ __forceinline__ uint32_t warp_incl_scan(uint32_t v, uint32_t lane) {
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, v, o);
    if (lane >= (uint32_t)o) v += y;
  }
  return v;
}

// The bits of the neighbours of vertices l[0..n), 1 <= n <= 32, each with at
// least one, into the bit set N (shared memory): one warp, each lane its vertex's
// record, then the vertices' further units as one strip, 32 units per step, a
// lane finding its unit's vertex from the bit mask of the strip's first units.
// strip: 32 words of the warp.  Returns the degree of the lane's vertex.
template <typename IdT>
__device__ __forceinline__ uint32_t expand_vertices(const RowInst& I, const IdT* l, uint32_t n,
                                                    uint32_t* N, uint32_t* strip) {
  constexpr uint32_t U = Unit<IdT>::n, P = U / 4;  // places in a unit, and in a word of one
  const uint32_t lane = threadIdx.x & 31, upto = 0xFFFFFFFFu >> (31 - lane);
  uint32_t us = 0, deg = 0;
  uint4 u = {0, 0, 0, 0};
  if (lane < n) {
    const uint4* r = (const uint4*)I.rec + 2 * (size_t)l[lane];
    const uint2 t = __ldg((const uint2*)r);
    u = __ldg(r + 1);
    us = t.x;
    deg = t.y;
  }
  const uint32_t most = __reduce_max_sync(0xffffffffu, deg);
  if (lane < n) {
    set_part(N, u.x, IdT());
    if (most > P) set_part(N, u.y, IdT());
    if (most > 2 * P) set_part(N, u.z, IdT());
    if (most > 3 * P) set_part(N, u.w, IdT());
  }
  if (most <= U) return deg;
  const uint32_t more = deg > U ? (deg - 1) / U : 0u;  // further units
  const uint32_t has = __ballot_sync(0xffffffffu, more > 0);
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
      u = __ldg((const uint4*)I.units + (t + e));
      set_part(N, u.x, IdT());
      set_part(N, u.y, IdT());
      set_part(N, u.z, IdT());
      set_part(N, u.w, IdT());
    }
  }
  __syncwarp();
  return deg;
}

// The set bits of a row's mask (at most 32 words) as an ordered list; returns
// their number.  One warp.
__device__ __forceinline__ uint32_t list_pieces(uint32_t m, uint16_t* to) {
  const uint32_t lane = threadIdx.x & 31, c = __popc(m), sum = warp_incl_scan(c, lane);
  for (uint32_t at = sum - c; m; m &= m - 1) to[at++] = (uint16_t)(lane * 32 + __ffs(m) - 1);
  return __shfl_sync(0xffffffffu, sum, 31);
}

}  // namespace wg
