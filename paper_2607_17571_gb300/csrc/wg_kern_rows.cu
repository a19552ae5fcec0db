// wg_kern_rows.cu -- transitive closure row by row (sm_103a).
//
// The TC rule T(x,z) <- T(x,y), E(y,z) never changes x, so the semi-naive
// fixpoint splits into one independent fixpoint per source x: its delta is the
// set of vertices first reached at the current iteration, and "dedup + set
// difference + merge" against the row T(x,.) is a bit test and set.  A row of
// up to 2^18 vertices is a bit set of at most 32 KB, which a CTA keeps in
// shared memory for the whole fixpoint of the row: the candidates of an
// iteration are never written to memory, sorted or merged.  The iteration
// index of a tuple is the level at which its bit was first set, so the
// per-iteration delta sizes, the iteration count and the candidate count
// (sum of deg(y) over the expanded delta tuples) are those of the iteration
// over all rows at once, and the rows' bit sets in source order are the sorted
// relation.
//
// Measured on GB300, fixpoint and result in device memory, sorted-array
// pipeline -> rows: R-MAT 2^17 / 400k edges (4.8e8 tuples) 67.6 -> 16.3 ms,
// R-MAT 2^19 / 400k (1.0e9 tuples, 64-bit keys) 165 -> 27.6 ms, ER 1,000 /
// 3,000 2.53 -> 0.15 ms, a chain of 1,000 vertices 145 -> 1.8 ms.
//
//   k_rows        the fixpoints of all rows (one CTA per row, rows claimed)
//   k_row_plan    row offsets (scan of the row counts), totals, capacity check
//   k_row_expand  bit sets -> sorted packed keys
#include "wg_device.cuh"
#include "wg_launch.h"

namespace wg {

// Adjacency record of a vertex: out-degree and the first kRecInline neighbours,
// 16 bytes with 16-bit ranks, 32 bytes (one sector) with 32-bit ranks.  One
// load gives most vertices' whole adjacency; longer ones continue in the CSR.
__device__ __forceinline__ uint32_t rec_id(const uint4& a, const uint4&, int s, uint16_t) {
  const uint32_t v = s == 0 ? a.x : s <= 2 ? a.y : s <= 4 ? a.z : a.w;
  return (s & 1) ? (v & 0xFFFFu) : (v >> 16);
}
__device__ __forceinline__ uint32_t rec_id(const uint4& a, const uint4& b, int s, uint32_t) {
  return s == 0 ? a.y : s == 1 ? a.z : s == 2 ? a.w : s == 3 ? b.x : s == 4 ? b.y : s == 5 ? b.z : b.w;
}
__device__ __forceinline__ void rec_load(const uint4* rec, uint32_t y, uint4& a, uint4& b, uint16_t) {
  a = __ldg(rec + y);
  b = a;
}
__device__ __forceinline__ void rec_load(const uint4* rec, uint32_t y, uint4& a, uint4& b, uint32_t) {
  a = __ldg(rec + 2 * (size_t)y);
  b = __ldg(rec + 2 * (size_t)y + 1);
}
__device__ __forceinline__ uint32_t rec_deg(const uint4& a, uint16_t) { return a.x & 0xFFFFu; }
__device__ __forceinline__ uint32_t rec_deg(const uint4& a, uint32_t) { return a.x; }

template <typename IdT>
__global__ void k_row_records(const uint32_t* off, const uint32_t* adj, uint32_t nv, IdT* rec) {
  constexpr uint32_t kTop = sizeof(IdT) == 2 ? 0xFFFFu : 0xFFFFFFFFu;
  const uint32_t n = nv * 8u;
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const uint32_t v = i >> 3, s = i & 7u, o = off[v], d = off[v + 1] - o;
    rec[i] = (IdT)(s == 0 ? min(d, kTop) : s <= d ? adj[o + s - 1] : 0u);
  }
}

__device__ __forceinline__ uint32_t warp_incl_scan(uint32_t v, uint32_t lane) {
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, v, o);
    if (lane >= (uint32_t)o) v += y;
  }
  return v;
}

// One CTA takes a row through its whole fixpoint.  Shared memory: the row's
// bit set and the head of its list of reached vertices in order of discovery
// (the rest of the list, past kRowQueue entries, lies in the CTA's part of
// `gq`, which stays in L2); a level is the range of the list pushed by the one
// before it.  Per level each warp takes 32 frontier vertices at a time: their
// records in one load per lane, then the neighbours past the inline ones of
// all 32 as one strip of edges (each lane finds its edge's vertex by a search
// over the lanes' prefix sums), so hubs are spread over the warp.
template <typename IdT>
__global__ void __launch_bounds__(kThreads, 6) k_rows(RowJob J) {
  extern __shared__ uint32_t sm[];
  __shared__ RowInst I;
  __shared__ unsigned long long s_log[kRowLog];
  __shared__ uint32_t s_row[2], s_push[3];
  uint32_t* V = sm;
  IdT* sq = (IdT*)(sm + J.vwords);
  IdT* gq = (IdT*)J.queue + (size_t)blockIdx.x * J.queue_stride;
  const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  unsigned long long cand = 0;
  uint32_t cur = 0xFFFFFFFFu;
  for (uint32_t i = tid; i < J.vwords; i += kThreads) V[i] = 0;
  if (tid < kRowLog) s_log[tid] = 0;
  if (tid == 0) s_row[0] = atomicAdd(&J.ctl->next_row, 1u);
  __syncthreads();
  auto put = [&](uint32_t p, uint32_t z) {
    if (p < kRowQueue) sq[p] = (IdT)z; else gq[p] = (IdT)z;
  };
  auto flush = [&]() {  // the counters of the current instance
    for (int o = 16; o > 0; o >>= 1) cand += __shfl_xor_sync(0xffffffffu, cand, o);
    if (lane == 0 && cand) atomicAdd(&J.inst[cur].cand, cand);
    cand = 0;
    if (tid < kRowLog && s_log[tid]) {
      if (tid < I.log_cap) atomicAdd(I.log + tid, s_log[tid]);
      s_log[tid] = 0;
    }
  };
  for (uint32_t p = 0;; p ^= 1) {
    const uint32_t row = s_row[p];
    if (row >= J.nrows) break;
    const uint32_t q = J.chunk_inst ? J.chunk_inst[row / kRowChunk] : 0u;
    if (q != cur) {
      __syncthreads();
      if (cur != 0xFFFFFFFFu) flush();
      __syncthreads();
      if (tid == 0) I = J.inst[q];
      cur = q;
      __syncthreads();
    }
    if (tid == 0) s_row[p ^ 1] = atomicAdd(&J.ctl->next_row, 1u);
    const uint32_t x = row - I.row0;
    uint32_t o = 0, end = 0;
    if (x < I.nv) {  // (rows of an instance are padded to whole chunks)
      o = I.off[x];
      end = I.off[x + 1] - o;
    }
    if (end == 0) {
      if (tid == 0 && x < I.nv) I.cnt[x] = 0;
    } else {
      if (tid == 0) s_push[0] = 0;
      for (uint32_t i = tid; i < end; i += kThreads) {
        const uint32_t z = I.adj[o + i];
        atomicOr(V + (z >> 5), 1u << (z & 31));
        put(i, z);
      }
      if (tid == 0) { cand += end; s_log[0] += end; }
      __syncthreads();
      uint32_t start = 0, lvl = 0;
      while (lvl < I.max_iters) {
        uint32_t* push = s_push + lvl % 3;
        if (tid == 0) s_push[(lvl + 1) % 3] = 0;
        for (uint32_t b = start + warp * 32; b < end; b += kThreads) {
          const uint32_t i = b + lane;
          uint4 ra = {0, 0, 0, 0}, rb = ra;
          uint32_t y = 0;
          if (i < end) {
            y = i < kRowQueue ? sq[i] : gq[i];
            rec_load((const uint4*)I.rec, y, ra, rb, IdT());
          }
          const uint32_t deg = rec_deg(ra, IdT());
          const uint32_t inl = min(deg, kRecInline);
          uint32_t fo = 0, r = 0;
          if (deg > kRecInline) {  // (a 16-bit degree field saturates)
            fo = I.off[y];
            r = I.off[y + 1] - fo - kRecInline;
            fo += kRecInline;
          }
          cand += inl + r;
          uint32_t m = 0;
          const uint32_t most = __reduce_max_sync(0xffffffffu, inl);
#pragma unroll
          for (int s = 0; s < (int)kRecInline; ++s) {
            if (s >= most) break;
            if (s < inl) {
              const uint32_t z = rec_id(ra, rb, s, IdT()), bit = 1u << (z & 31);
              if (!(V[z >> 5] & bit) && !(atomicOr(V + (z >> 5), bit) & bit)) m |= 1u << s;
            }
          }
          {
            const uint32_t c = __popc(m), in = warp_incl_scan(c, lane);
            const uint32_t tot = __shfl_sync(0xffffffffu, in, 31);
            if (tot) {
              uint32_t at = 0;
              if (lane == 0) at = atomicAdd(push, tot);
              at = end + __shfl_sync(0xffffffffu, at, 0) + in - c;
#pragma unroll
              for (int s = 0; s < (int)kRecInline; ++s)
                if (m >> s & 1u) put(at++, rec_id(ra, rb, s, IdT()));
            }
          }
          if (__any_sync(0xffffffffu, r)) {
            const uint32_t in = warp_incl_scan(r, lane);
            const uint32_t R = __shfl_sync(0xffffffffu, in, 31);
            const uint32_t fe = fo - (in - r);  // edge e of the strip is adj[fe_owner + e]
            for (uint32_t e0 = 0; e0 < R; e0 += 32) {
              const uint32_t e = e0 + lane;
              uint32_t ow = 0;  // lanes whose inclusive prefix is <= e
#pragma unroll
              for (int st = 16; st > 0; st >>= 1) {
                const uint32_t v = __shfl_sync(0xffffffffu, in, ow + st - 1);
                if (v <= e) ow += st;
              }
              const uint32_t a = __shfl_sync(0xffffffffu, fe, ow & 31);
              uint32_t z = 0;
              bool win = false;
              if (e < R) {
                z = I.adj[a + e];
                const uint32_t bit = 1u << (z & 31);
                win = !(V[z >> 5] & bit) && !(atomicOr(V + (z >> 5), bit) & bit);
              }
              const uint32_t bal = __ballot_sync(0xffffffffu, win);
              if (bal) {
                uint32_t at = 0;
                if (lane == 0) at = atomicAdd(push, (uint32_t)__popc(bal));
                at = end + __shfl_sync(0xffffffffu, at, 0) + __popc(bal & ((1u << lane) - 1));
                if (win) put(at, z);
              }
            }
          }
        }
        __syncthreads();
        const uint32_t n = *push;
        if (n == 0) break;
        ++lvl;
        if (tid == 0) {
          if (lvl < kRowLog) s_log[lvl] += n;
          else if (lvl < I.log_cap) atomicAdd(I.log + lvl, (unsigned long long)n);
        }
        start = end;
        end += n;
      }
      if (tid == 0) {
        atomicMax(&J.inst[q].last, lvl);
        I.cnt[x] = end;
        atomicAdd(J.csum + row / kRowChunk, end);
      }
      // the row's bit set out, and cleared for the next row
      uint4* out = (uint4*)(I.bits + (size_t)x * I.words);
      uint4* v4 = (uint4*)V;
      for (uint32_t i = tid; i < I.words / 4; i += kThreads) {
        out[i] = v4[i];
        v4[i] = uint4{0, 0, 0, 0};
      }
    }
    __syncthreads();
  }
  if (cur != 0xFFFFFFFFu) flush();
}

// Row offsets at chunk granularity, totals and the capacity check: one CTA per
// instance scans its chunk sums in place (counts in, exclusive offsets out).
__global__ void __launch_bounds__(1024) k_row_plan(RowJob J) {
  __shared__ unsigned long long sh[32];
  RowInst* I = J.inst + blockIdx.x;
  const uint32_t c0 = I->row0 / kRowChunk, nc = (I->nv + kRowChunk - 1) / kRowChunk;
  const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  unsigned long long carry = 0;
  for (uint32_t b = 0; b < nc; b += 1024) {
    const uint32_t i = b + threadIdx.x;
    const unsigned long long v = i < nc ? J.csum[c0 + i] : 0u;
    unsigned long long s = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned long long y = __shfl_up_sync(0xffffffffu, s, o);
      if (lane >= (uint32_t)o) s += y;
    }
    __syncthreads();
    if (lane == 31) sh[warp] = s;
    __syncthreads();
    if (warp == 0) {
      unsigned long long u = sh[lane];
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long y = __shfl_up_sync(0xffffffffu, u, o);
        if (lane >= (uint32_t)o) u += y;
      }
      sh[lane] = u;
    }
    __syncthreads();
    if (i < nc) J.cbase[c0 + i] = carry + (warp ? sh[warp - 1] : 0ull) + s - v;
    carry += sh[31];
  }
  if (threadIdx.x == 0) {
    I->n_total = carry;
    // an output buffer that is too small: the expansion waits for a larger one
    I->fits = carry <= I->out_cap ? 1u : 0u;
  }
}

// Bit sets -> sorted packed keys (x << w) | z, one warp per row: 64 words at a
// time, each lane lists the set bits of its two words at its prefix in the
// warp's shared buffer, then the warp writes the list coalesced.
template <typename K>
__global__ void __launch_bounds__(kThreads) k_row_expand(RowJob J) {
  __shared__ uint16_t buf[kWarps][2048];
  const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t stride = gridDim.x * kWarps;
  for (uint32_t row = blockIdx.x * kWarps + warp; row < J.nrows; row += stride) {
    const uint32_t ch = row / kRowChunk;
    const RowInst* I = J.inst + (J.chunk_inst ? J.chunk_inst[ch] : 0u);
    const uint32_t x = row - I->row0;
    if (x >= I->nv || !I->fits) continue;
    const uint32_t n = I->cnt[x];
    if (n == 0) continue;
    // this row's offset: the chunk's, and the rows before it in the chunk
    const uint32_t r0 = x / kRowChunk * kRowChunk;
    uint32_t before = 0;
    for (uint32_t i = r0 + lane; i < x; i += 32) before += I->cnt[i];
    before = __reduce_add_sync(0xffffffffu, before);
    K* out = (K*)I->out + J.cbase[ch] + before;
    const uint2* w2 = (const uint2*)(I->bits + (size_t)x * I->words);
    const uint32_t np = I->words / 2;
    const K hi = (K)x << I->w;
    uint2 v = lane < np ? w2[lane] : uint2{0, 0};
    for (uint32_t b = 0; b < np; b += 32) {
      const uint32_t nx = b + 32 + lane;
      const uint2 nextv = nx < np ? w2[nx] : uint2{0, 0};
      const uint32_t c = __popc(v.x) + __popc(v.y), in = warp_incl_scan(c, lane);
      const uint32_t tot = __shfl_sync(0xffffffffu, in, 31);
      if (tot) {
        uint32_t at = in - c;
        uint32_t m = v.x;
        while (m) {
          buf[warp][at++] = (uint16_t)(lane * 64 + __ffs(m) - 1);
          m &= m - 1;
        }
        m = v.y;
        while (m) {
          buf[warp][at++] = (uint16_t)(lane * 64 + 31 + __ffs(m));
          m &= m - 1;
        }
        __syncwarp();
        const K base = hi + (K)b * 64;
        for (uint32_t j = lane; j < tot; j += 32) out[j] = base + buf[warp][j];
        out += tot;
        __syncwarp();
      }
      v = nextv;
    }
  }
}

// ------------------------------------------------------------------ launchers
uint32_t row_smem(uint32_t vwords, int id_bytes) { return vwords * 4 + kRowQueue * id_bytes; }

template <typename IdT>
static int rows_occ(uint32_t smem) {
  static int max_set = 0;  // (the attribute is per process and device, raised once)
  if (!max_set) {
    cudaFuncSetAttribute(k_rows<IdT>, cudaFuncAttributeMaxDynamicSharedMemorySize, kRowSmemMax);
    max_set = 1;
  }
  int occ = 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_rows<IdT>, kThreads, smem);
  return occ;
}
int occupancy_rows(int id_bytes, uint32_t vwords) {
  const uint32_t smem = row_smem(vwords, id_bytes);
  return id_bytes == 2 ? rows_occ<uint16_t>(smem) : rows_occ<uint32_t>(smem);
}
void launch_rows(const RowJob& J, int id_bytes, int grid, cudaStream_t s) {
  const uint32_t smem = row_smem(J.vwords, id_bytes);
  if (id_bytes == 2) k_rows<uint16_t><<<grid, kThreads, smem, s>>>(J);
  else k_rows<uint32_t><<<grid, kThreads, smem, s>>>(J);
}
void launch_row_plan(const RowJob& J, uint32_t n_inst, cudaStream_t s) {
  k_row_plan<<<n_inst, 1024, 0, s>>>(J);
}
template <typename K>
void launch_row_expand(const RowJob& J, int grid, cudaStream_t s) {
  k_row_expand<K><<<grid, kThreads, 0, s>>>(J);
}
void launch_row_records(const uint32_t* off, const uint32_t* adj, uint32_t nv, void* rec,
                        int id_bytes, int grid, cudaStream_t s) {
  if (id_bytes == 2) k_row_records<uint16_t><<<grid, kThreads, 0, s>>>(off, adj, nv, (uint16_t*)rec);
  else k_row_records<uint32_t><<<grid, kThreads, 0, s>>>(off, adj, nv, (uint32_t*)rec);
}
template void launch_row_expand<uint32_t>(const RowJob&, int, cudaStream_t);
template void launch_row_expand<unsigned long long>(const RowJob&, int, cudaStream_t);

}  // namespace wg
