// wg_kern_tri.cu -- triangle counting by set intersection (sm_103a).
//
// triangle(a,b,c) <- E(a,b), E(b,c), E(c,a): the count is the sum over the
// edges (a,b) of |Out(b) /\ In(a)|.  A CTA takes one vertex and keeps one of
// its two neighbour sets as a bit set over all vertices in shared memory; each
// edge is counted at the end whose set is the larger, walking the smaller list
// of the two: sum over edges of min(deg Out(b), deg In(a)) bit tests instead of
// a binary search per two-path.  In(v) is the transpose, built per call with
// one atomic per edge (its lists need no order).
//
// Bound by the latency of the gathered lists (L2) and issue slots.  Undirected
// R-MAT 2^16 / 800k edges, 2.9e8 two-paths: 0.24 ms (0.18 of it k_tri_count),
// against 15.1 ms with the join and a binary search per two-path.
#include "wg_device.cuh"
#include "wg_launch.h"

namespace wg {

// In-degrees, and the number of two-paths (a,b,c).
template <typename K>
__global__ void __launch_bounds__(kThreads) k_tri_degrees(const K* E, uint32_t ne, uint32_t w,
                                                          TriJob J) {
  const K mask = (K)(((K)1 << w) - 1);
  unsigned long long paths = 0;
  for (uint32_t i = blockIdx.x * kThreads + threadIdx.x; i < ne; i += gridDim.x * kThreads) {
    const uint32_t b = (uint32_t)(E[i] & mask);
    atomicAdd(J.ideg + b, 1u);
    paths += J.off[b + 1] - J.off[b];
  }
  for (int o = 16; o > 0; o >>= 1) paths += __shfl_xor_sync(0xffffffffu, paths, o);
  if ((threadIdx.x & 31) == 0 && paths) atomicAdd(&J.ctl->paths, paths);
}

// Room for every in-list, in any order (one atomic per warp), and the tasks:
// vertex v's edges from both ends, chunk neighbours a task, so that a hub's
// are spread over the chip (one task per vertex and end: 1.06 ms, the hubs
// ending last; the bit set is built once per task, sum of d^2 / chunk atomics).
__global__ void __launch_bounds__(kThreads) k_tri_rooms(TriJob J) {
  const uint32_t v = blockIdx.x * kThreads + threadIdx.x, lane = threadIdx.x & 31;
  const uint32_t d = v < J.nv ? J.ideg[v] : 0u;
  uint32_t in = d;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, in, o);
    if (lane >= (uint32_t)o) in += y;
  }
  uint32_t at = 0;
  if (lane == 31 && in) at = atomicAdd(&J.ctl->room, in);
  at = __shfl_sync(0xffffffffu, at, 31) + in - d;
  if (v >= J.nv) return;
  J.ioff[v] = at;
  J.ifill[v] = at;
  const uint32_t od = J.off[v + 1] - J.off[v];
  if (!d || !od) return;  // one of its sets is empty
  const uint32_t n0 = (od + J.chunk - 1) / J.chunk, n1 = (d + J.chunk - 1) / J.chunk;
  uint2* task = J.task + atomicAdd(&J.ctl->tasks, n0 + n1);
  for (uint32_t i = 0; i < n0; ++i) *task++ = uint2{v, 2 * i};
  for (uint32_t i = 0; i < n1; ++i) *task++ = uint2{v, 2 * i + 1};
}

template <typename K>
__global__ void __launch_bounds__(kThreads) k_tri_transpose(const K* E, uint32_t ne, uint32_t w,
                                                            TriJob J) {
  const K mask = (K)(((K)1 << w) - 1);
  for (uint32_t i = blockIdx.x * kThreads + threadIdx.x; i < ne; i += gridDim.x * kThreads) {
    const K k = E[i];
    J.iadj[atomicAdd(J.ifill + (uint32_t)(k & mask), 1u)] = (uint32_t)(k >> w);
  }
}

// Task {v, 2 i + odd}: even: the set is In(v), lists Out(b) of the i-th chunk of
// Out(v); odd: the set is Out(v), lists In(a) of the i-th chunk of In(v).  An
// edge whose two lists are equally long belongs to the even task.  Four steps
// of 32 list elements are in flight per warp.
__global__ void __launch_bounds__(1024, 1) k_tri_count(TriJob J) {
  extern __shared__ uint32_t bits[];  // [words] | per warp 32 list starts
  __shared__ uint32_t s_t[2];
  const uint32_t tid = threadIdx.x, T = blockDim.x, lane = tid & 31, warp = tid >> 5;
  uint32_t* strip = bits + J.words + warp * 32;
  const uint32_t upto = 0xFFFFFFFFu >> (31 - lane);
  unsigned long long hits = 0;
  for (uint32_t i = tid; i < J.words; i += T) bits[i] = 0;
  if (tid == 0) s_t[0] = atomicAdd(&J.ctl->next, 1u);
  __syncthreads();
  for (uint32_t p = 0;; p ^= 1) {
    const uint32_t t = s_t[p];
    if (t >= J.ctl->tasks) break;
    uint32_t next = 0;
    if (tid == 0) next = atomicAdd(&J.ctl->next, 1u);
    const uint2 task = J.task[t];
    const uint32_t v = task.x, odd = task.y & 1u;
    const uint32_t oo = J.off[v], od = J.off[v + 1] - oo, io = J.ioff[v], id = J.ideg[v];
    const uint32_t* ladj = odd ? J.iadj : J.adj;  // neighbours and their lists
    const uint32_t* sadj = odd ? J.adj : J.iadj;  // the set
    uint32_t no = odd ? io : oo, nd = odd ? id : od;
    const uint32_t so = odd ? oo : io, sd = odd ? od : id;
    const uint32_t top = odd ? sd - 1 : sd;       // longest list walked here
    no += (task.y >> 1) * J.chunk;
    nd = min(J.chunk, nd - (task.y >> 1) * J.chunk);
    for (uint32_t i = tid; i < sd; i += T) {
      const uint32_t z = sadj[so + i];
      atomicOr(bits + (z >> 5), 1u << (z & 31));
    }
    __syncthreads();
    uint32_t mine = 0;
    for (uint32_t b = warp * 32; b < nd; b += T) {
      const uint32_t i = b + lane;
      uint32_t lo = 0, len = 0;
      if (i < nd) {
        const uint32_t y = ladj[no + i];
        if (odd) {
          lo = J.ioff[y];
          len = J.ideg[y];
        } else {
          lo = J.off[y];
          len = J.off[y + 1] - lo;
        }
        if (len > top) len = 0;
      }
      const uint32_t has = __ballot_sync(0xffffffffu, len > 0);
      if (!has) continue;
      uint32_t in = len;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, in, o);
        if (lane >= (uint32_t)o) in += y;
      }
      const uint32_t tot = __shfl_sync(0xffffffffu, in, 31), st = in - len;
      if (len) strip[__popc(has & upto) - 1] = lo - st;
      __syncwarp();
      uint32_t prev = 0;  // lists that begin before this step
      for (uint32_t e0 = 0; e0 < tot; e0 += 128) {
        uint32_t z[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const uint32_t s0 = e0 + 32 * k, sh = st - s0, e = s0 + lane;
          const uint32_t m = __reduce_or_sync(0xffffffffu, len && sh < 32u ? 1u << sh : 0u);
          const uint32_t at = strip[prev + __popc(m & upto) - 1];
          prev += __popc(m);
          z[k] = e < tot ? __ldg(ladj + (at + e)) : 0xFFFFFFFFu;
        }
#pragma unroll
        for (int k = 0; k < 4; ++k)
          if (z[k] != 0xFFFFFFFFu) mine += bits[z[k] >> 5] >> (z[k] & 31) & 1u;
      }
      __syncwarp();
    }
    hits += mine;
    __syncthreads();
    for (uint32_t i = tid; i < sd; i += T) bits[sadj[so + i] >> 5] = 0;
    if (tid == 0) s_t[p ^ 1] = next;
    __syncthreads();
  }
  for (int o = 16; o > 0; o >>= 1) hits += __shfl_xor_sync(0xffffffffu, hits, o);
  if (lane == 0 && hits) atomicAdd(&J.ctl->hits, hits);
}

// Threads per CTA: about 32 warps an SM, split over as many CTAs as the bit
// sets leave room for (most tasks are short, and a CTA waits for its slowest
// warp three times per task).
static uint32_t tri_threads(uint32_t words) {
  const uint32_t ctas = min(16u, (uint32_t)kTriSmem / (words * 4 + 2048));
  return ctas >= 16 ? 64u : ctas >= 8 ? 128u : ctas >= 4 ? 256u : ctas >= 2 ? 512u : 1024u;
}
template <typename K>
void launch_tri(const K* E, uint32_t ne, uint32_t w, const TriJob& job, int sms, cudaStream_t s) {
  const int grid = sms * 8;
  TriJob J = job;
  const uint32_t t = tri_threads(J.words), smem = J.words * 4 + t * 4;
  J.chunk = t;  // (a batch of 32 neighbours per warp)
  k_tri_degrees<K><<<grid, kThreads, 0, s>>>(E, ne, w, J);
  k_tri_rooms<<<(J.nv + kThreads - 1) / kThreads, kThreads, 0, s>>>(J);
  k_tri_transpose<K><<<grid, kThreads, 0, s>>>(E, ne, w, J);
  cudaFuncSetAttribute(k_tri_count, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kTriSmem);
  int occ = 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_tri_count, (int)t, smem);
  k_tri_count<<<sms * max(1, occ), t, smem, s>>>(J);
}
template void launch_tri<uint32_t>(const uint32_t*, uint32_t, uint32_t, const TriJob&, int, cudaStream_t);
template void launch_tri<unsigned long long>(const unsigned long long*, uint32_t, uint32_t,
                                             const TriJob&, int, cudaStream_t);

}  // namespace wg
