// wg_kern_sg.cu -- same-generation over rows of bit sets (sm_103a).
//
// sg(x,y) <- E(a,x), sg(a,b), E(b,y): all tuples (x,.) of one iteration come from
// the delta rows of x's parents, and every child x of a receives the same set
// S_a = union of the children of b over delta(a,.).  So an iteration takes each
// row a with a non-empty delta once: S_a is built in shared memory from the
// delta's vertices (as in k_rows), and each child's row drops what it has and
// keeps the rest as its next delta -- deg(a) passes over the non-zero 128-bit
// pieces of S_a instead of deg(a) * deg(b) candidates per tuple written, sorted
// and merged.  Iteration k gives delta^k exactly (base: delta^-1(p) = {p}, the
// child's own bit left out), so sizes, iteration count and the candidate count
// (sum of deg(a) deg(b)) are those of the sorted-array pipeline.
//
// Rows live in HBM / L2: the relation F and two deltas (read and written in
// turn).  A bit per piece says which are valid, so rows are neither cleared nor
// scanned: only the masks are.  A row of one parent is written by one CTA per
// iteration with plain stores; rows of several parents (cleared before) take
// atomics.  One cooperative launch runs every iteration of all its instances,
// a barrier over the grid between two.
//
// A row of more than kSgSlice children is several items, each with its own S_a: with
// one item per row a hub's children (|S_a| / 128 pieces each) were one CTA's work
// while the grid waited, at the barrier's limit even a timeout.  Stars of 4,000 /
// 10,000 / 40,000 children, whole call: one item 1.45 / 9.7 / 154 ms (sorted-array
// pipeline 0.94 / 5.0 / 73), slices of 1,024 0.49 / 1.24 / 5.5, of 512 0.29 / 0.73 / 3.6,
// of 256 0.20 / 0.47 / 2.6; R-MAT 2^12 / 9,000 0.82, 0.80, 0.80, 0.70.
//
// Bound by the latency of an item's steps (delta pieces, records, row pieces) and
// the barriers between them (ncu: 24% of the issue slots, DRAM 1%), so CTAs are
// small: 256 / 128 / 64 / 32 threads 1.71 / 1.05 / 0.86 / 0.88 ms on the forest of
// 60,000 vertices (7.5e7 tuples, 12 iterations; 0.83 since records are loaded
// ahead); whole call 6.5 ms on the sorted-array pipeline, 1.3-1.4 here.
#include "wg_device.cuh"
#include "wg_launch.h"
#include "wg_rows.cuh"

namespace wg {

__device__ __forceinline__ uint32_t popc4(const uint4& v) {
  return __popc(v.x) + __popc(v.y) + __popc(v.z) + __popc(v.w);
}
__device__ __forceinline__ bool any4(const uint4& v) { return (v.x | v.y | v.z | v.w) != 0; }
__device__ __forceinline__ uint32_t sg_slices(uint32_t deg) {
  return (deg + kSgSlice - 1) / kSgSlice;
}
constexpr uint32_t kNone = 0xFFFFFFFFu;
__device__ __forceinline__ bool bit_of(const uint32_t* s, uint32_t i) {
  return s[i >> 5] >> (i & 31) & 1u;
}

// Clears the rows of vertices with several parents (their pieces are all valid), and
// lists the slices of every row past its first for iteration 0, which takes all rows.
__global__ void __launch_bounds__(kThreads) k_sg_init(SgJob J) {
  const uint32_t lane = threadIdx.x & 31;
  for (uint32_t r = (blockIdx.x * kThreads + threadIdx.x) / 32; r < J.rows.nrows;
       r += gridDim.x * kWarps) {
    const uint32_t q = J.rows.chunk_inst ? J.rows.chunk_inst[r / kRowChunk] : 0u;
    const RowInst& I = J.rows.inst[q];
    const uint32_t x = r - I.row0;
    if (x >= I.nv) continue;
    const uint32_t more = sg_slices(I.off[x + 1] - I.off[x]) - 1;
    if (more != 0 && more != kNone) {
      uint32_t at = 0;
      if (lane == 0) at = atomicAdd(&J.ctl->count[0], more);
      at = __shfl_sync(0xffffffffu, at, 0);
      for (uint32_t i = lane; i < more; i += 32) J.list[0][at + i] = uint2{r, i + 1};
    }
    if (!bit_of(I.mp, x)) continue;
    const SgInst& G = J.sg[q];
    const uint32_t quads = I.words / 4;
    const size_t at = (size_t)x * quads;
    const uint4 z = {0, 0, 0, 0};
    for (uint32_t w = lane; w < quads; w += 32) {
      ((uint4*)I.bits)[at + w] = z;
      G.d[0][at + w] = z;
      G.d[1][at + w] = z;
    }
    for (uint32_t w = lane; w < G.mw; w += 32)
      G.fm[(size_t)x * G.mw + w] =
          w + 1 < G.mw || quads % 32 == 0 ? 0xFFFFFFFFu : (1u << quads % 32) - 1;
  }
}

// The barrier between two iterations: every CTA of the grid is resident
// (cooperative launch).  Bounded: a CTA that waits too long records the timeout
// and every CTA returns.
__device__ __forceinline__ bool sg_barrier(SgCtl* c, uint32_t target) {
  __shared__ uint32_t s_ok;
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    atomicAdd(&c->arrived, 1u);
    uint32_t spins = 0, ok = 1;
    while (!sg_arrived(*(volatile uint32_t*)&c->arrived, target)) {
      if (++spins > kSgSpinLimit || *(volatile uint32_t*)&c->error) {
        atomicExch(&c->error, DEV_TIMEOUT);
        ok = 0;
        break;
      }
      __nanosleep(64);
    }
    __threadfence();
    s_ok = ok;
  }
  __syncthreads();
  return s_ok != 0;
}

template <typename IdT>
__global__ void __launch_bounds__(kSgThreads, 16) k_sg(SgJob J) {
  constexpr uint32_t kW = kSgThreads / 32;
  extern __shared__ uint4 S4[];
  __shared__ RowInst I;
  __shared__ SgInst G;
  __shared__ uint2 s_item[2];                                // {row, slice of its children}
  __shared__ uint32_t s_nq, s_nz, s_last, s_kids[kSgSlice / 32];  // children with new tuples
  const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  uint32_t* S = (uint32_t*)S4;
  uint32_t* strip = S + J.rows.vwords + warp * 32;
  uint16_t* nzl = (uint16_t*)(S + J.rows.vwords + kW * 32);  // non-zero pieces of S
  uint16_t* vql = nzl + J.rows.vwords / 4;                   // valid pieces of the delta row
  IdT* list = (IdT*)(vql + J.rows.vwords / 4) + warp * kSgList;
  for (uint32_t i = tid; i < J.rows.vwords / 4; i += kSgThreads) S4[i] = uint4{0, 0, 0, 0};
  if (tid == 0) s_nz = 0;
  if (tid < kSgSlice / 32) s_kids[tid] = 0;
  unsigned long long cand = 0, got = 0;
  uint32_t cur = 0xFFFFFFFFu;
  SgCtl* ctl = J.ctl;
  bool hubs = false;  // some row has several slices
  for (uint32_t k = 0;; ++k) {
    auto flush = [&]() {  // the counters of the current instance and iteration
      for (int o = 16; o > 0; o >>= 1) {
        cand += __shfl_xor_sync(0xffffffffu, cand, o);
        got += __shfl_xor_sync(0xffffffffu, got, o);
      }
      if (lane == 0) {
        if (cand) atomicAdd(&J.rows.inst[cur].cand, cand);
        if (got) {
          if (k < I.log_cap) atomicAdd(I.log + k, got);
          atomicMax(&J.rows.inst[cur].last, k);
        }
      }
      cand = got = 0;
    };
    const uint32_t in = k & 1, out = in ^ 1u;
    const uint32_t first = k == 0 ? J.rows.nrows : 0u;  // (all rows, before what is listed)
    const uint32_t n = first + __ldcg(&ctl->count[k % 3]);
    if (k == 0) hubs = n > first;
    uint32_t* const next_n = &ctl->count[(k + 1) % 3];
    if (blockIdx.x == 0 && tid == 0) {  // (the slots no CTA uses in this iteration)
      ctl->count[(k + 2) % 3] = 0;
      ctl->next[(k + 2) % 3] = 0;
    }
    const uint2* const listed = in ? J.list[1] : J.list[0];
    uint2* const to_list = in ? J.list[0] : J.list[1];
    auto item_of = [&](uint32_t i) {
      return i >= n ? uint2{kNone, 0} : i < first ? uint2{i, 0} : __ldcg(listed + (i - first));
    };
    if (tid == 0) s_item[0] = item_of(atomicAdd(&ctl->next[k % 3], 1u));
    __syncthreads();
    for (uint32_t p = 0;; p ^= 1) {
      const uint32_t row = s_item[p].x, c0 = s_item[p].y * kSgSlice;
      if (row == kNone) break;
      const uint32_t q = J.rows.chunk_inst ? J.rows.chunk_inst[row / kRowChunk] : 0u;
      if (q != cur) {
        if (cur != 0xFFFFFFFFu) flush();
        __syncthreads();
        if (tid == 0) { I = J.rows.inst[q]; G = J.sg[q]; }
        cur = q;
        __syncthreads();
      }
      // the next item, claimed here and stored at the end: nothing waits for it
      uint32_t next = 0;
      if (tid == 0) next = atomicAdd(&ctl->next[k % 3], 1u);
      const uint32_t a = row - I.row0, quads = I.words / 4;
      uint32_t o = 0, deg = 0;
      if (a < I.nv) {
        o = I.off[a];
        deg = I.off[a + 1] - o;
      }
      if (deg == 0) {
        if (tid == 0) s_item[p ^ 1] = item_of(next);
        __syncthreads();
        continue;
      }
      const uint32_t* adj = I.adj + o;
      const uint32_t kids = min(deg - c0, kSgSlice), slices = sg_slices(deg);
      if (k == 0) {
        for (uint32_t i = tid; i < deg; i += kSgThreads) {
          const uint32_t z = adj[i];
          atomicOr(S + (z >> 5), 1u << (z & 31));
        }
        if (tid == 0) cand += (unsigned long long)kids * (deg - 1);
      } else {
        if (warp == 0) {  // valid pieces of the delta row (at most 32 mask words)
          uint32_t m = 0;
          uint32_t* dm = G.dm[in] + (size_t)a * G.mw + lane;
          if (lane < G.mw && (m = __ldcg(dm)) != 0 && slices == 1) *dm = 0;
          const uint32_t valid = list_pieces(m, vql);
          if (lane == 0) s_nq = valid;
        }
        __syncthreads();
        const uint32_t nq = s_nq;
        const bool many = bit_of(I.mp, a);
        uint32_t dsum = 0;
        for (uint32_t g = warp * 8; g < nq; g += kW * 8) {
          uint4 v = {0, 0, 0, 0};
          uint32_t w = 0;
          if (lane < 8 && g + lane < nq) {
            w = vql[g + lane];
            uint4* p = G.d[in] + (size_t)a * quads + w;
            v = __ldcg(p);
            if (many && slices == 1) *p = uint4{0, 0, 0, 0};
            const uint4 ns = __ldg((const uint4*)I.ns + w);
            v.x &= ns.x; v.y &= ns.y; v.z &= ns.z; v.w &= ns.w;
          }
          const uint32_t c = popc4(v), sum = warp_incl_scan(c, lane);
          const uint32_t len = __shfl_sync(0xffffffffu, sum, 31);
          uint32_t at = sum - c;
          auto put = [&](uint32_t m, uint32_t base) {
            for (; m; m &= m - 1) list[at++] = (IdT)(base + __ffs(m) - 1);
          };
          put(v.x, w * 128); put(v.y, w * 128 + 32); put(v.z, w * 128 + 64); put(v.w, w * 128 + 96);
          __syncwarp();
          dsum += expand_vertices<IdT, true>(I, list, 0, len, 32, S, strip);
          __syncwarp();
        }
        cand += (unsigned long long)dsum * kids;
        if (slices > 1) {  // the last of the row's items to have read the delta clears it
          __syncthreads();
          if (tid == 0) {
            __threadfence();
            s_last = atomicAdd(G.done + a, 1u) == slices - 1;
            if (s_last) G.done[a] = 0;
          }
          __syncthreads();
          if (s_last) {
            for (uint32_t i = tid; i < G.mw; i += kSgThreads) G.dm[in][(size_t)a * G.mw + i] = 0;
            for (uint32_t i = tid; many && i < nq; i += kSgThreads)
              G.d[in][(size_t)a * quads + vql[i]] = uint4{0, 0, 0, 0};
          }
        }
      }
      __syncthreads();
      for (uint32_t w0 = warp * 32; w0 < quads; w0 += kSgThreads) {
        const uint32_t w = w0 + lane;
        const bool some = w < quads && any4(S4[w]);
        const uint32_t m = __ballot_sync(0xffffffffu, some);
        if (!m) continue;
        uint32_t at = 0;
        if (lane == 0) at = atomicAdd(&s_nz, (uint32_t)__popc(m));
        at = __shfl_sync(0xffffffffu, at, 0) + __popc(m & ((1u << lane) - 1));
        if (some) nzl[at] = (uint16_t)w;
      }
      __syncthreads();
      const uint32_t nz = s_nz, more = k < I.max_iters ? 1u : 0u;
      uint2 item;
      if (tid == 0) item = item_of(next);
      for (uint32_t i = tid; i < nz * kids; i += kSgThreads) {
        const uint32_t c = i / nz, w = nzl[i - c * nz], x = __ldg(adj + c0 + c);
        uint4 s = S4[w];
        if (k == 0 && w == x >> 7) {  // (x, x) is not in the base
          const uint32_t keep = ~(1u << (x & 31)), p = x >> 5 & 3;
          s.x &= p == 0 ? keep : ~0u;
          s.y &= p == 1 ? keep : ~0u;
          s.z &= p == 2 ? keep : ~0u;
          s.w &= p == 3 ? keep : ~0u;
        }
        const size_t at = (size_t)x * quads + w, mat = (size_t)x * G.mw + (w >> 5);
        const uint32_t bit = 1u << (w & 31);
        const bool on = more && bit_of(I.ns, x);  // x's delta joins something
        uint4* F = (uint4*)I.bits + at;
        uint4 d = s;
        if (!bit_of(I.mp, x)) {
          uint4 old = __ldcg(F);  // (beside the mask, not after it: unused if not valid)
          const bool old_valid = (__ldcg(G.fm + mat) & bit) != 0;
          if (!old_valid) old = uint4{0, 0, 0, 0};
          d.x &= ~old.x; d.y &= ~old.y; d.z &= ~old.z; d.w &= ~old.w;
          if (!any4(d)) continue;
          *F = uint4{old.x | d.x, old.y | d.y, old.z | d.z, old.w | d.w};
          if (!old_valid) atomicOr(G.fm + mat, bit);
          if (on) G.d[out][at] = d;
        } else {
          uint32_t* f = (uint32_t*)F;
          if (s.x) d.x &= ~atomicOr(f, s.x);
          if (s.y) d.y &= ~atomicOr(f + 1, s.y);
          if (s.z) d.z &= ~atomicOr(f + 2, s.z);
          if (s.w) d.w &= ~atomicOr(f + 3, s.w);
          if (!any4(d)) continue;
          if (on) {
            uint32_t* e = (uint32_t*)(G.d[out] + at);
            if (d.x) atomicOr(e, d.x);
            if (d.y) atomicOr(e + 1, d.y);
            if (d.z) atomicOr(e + 2, d.z);
            if (d.w) atomicOr(e + 3, d.w);
          }
        }
        got += popc4(d);
        if (on) {
          atomicOr(G.dm[out] + mat, bit);
          atomicOr(s_kids + (c >> 5), 1u << (c & 31));
        }
      }
      __syncthreads();
      // list the children with new tuples: a child of one parent only here, so
      // without asking; one of several once per iteration
      for (uint32_t c = tid; c < kids; c += kSgThreads) {
        if (!(s_kids[c >> 5] >> (c & 31) & 1u)) continue;
        const uint32_t x = __ldg(adj + c0 + c);
        uint32_t s = 1;
        if (hubs) s = sg_slices(__ldg(I.off + x + 1) - __ldg(I.off + x));
        if (bit_of(I.mp, x) && atomicExch(G.act + x, k + 1) == k + 1) continue;
        if (s == 1) {
          to_list[atomicAdd(next_n, 1u)] = uint2{I.row0 + x, 0};
          continue;
        }
        uint2* to = to_list + atomicAdd(next_n, s);
        for (uint32_t i = 0; i < s; ++i) to[i] = uint2{I.row0 + x, i};
      }
      for (uint32_t i = tid; i < nz; i += kSgThreads) S4[nzl[i]] = uint4{0, 0, 0, 0};
      if (tid == 0) { s_nz = 0; s_item[p ^ 1] = item; }
      __syncthreads();  // (every read of s_kids is done)
      if (tid < kSgSlice / 32) s_kids[tid] = 0;
    }
    if (cur != 0xFFFFFFFFu) flush();
    if (!sg_barrier(ctl, (k + 1) * gridDim.x)) return;
    if (__ldcg(next_n) == 0) return;
  }
}

// Tuples of every row, and of every chunk of rows.
__global__ void __launch_bounds__(kThreads) k_sg_count(SgJob J) {
  __shared__ uint16_t s_list[kWarps][kSgMaxVertices / 128];
  const uint32_t lane = threadIdx.x & 31;
  uint16_t* list = s_list[threadIdx.x >> 5];
  for (uint32_t r = (blockIdx.x * kThreads + threadIdx.x) / 32; r < J.rows.nrows;
       r += gridDim.x * kWarps) {
    const uint32_t q = J.rows.chunk_inst ? J.rows.chunk_inst[r / kRowChunk] : 0u;
    const RowInst& I = J.rows.inst[q];
    const uint32_t x = r - I.row0;
    if (x >= I.nv) continue;
    const SgInst& G = J.sg[q];
    const uint32_t quads = I.words / 4;
    const uint4* F = (const uint4*)I.bits + (size_t)x * quads;
    uint32_t c = 0;
    const uint32_t n = list_pieces(lane < G.mw ? G.fm[(size_t)x * G.mw + lane] : 0u, list);
    __syncwarp();
    for (uint32_t i = lane; i < n; i += 32) c += popc4(F[list[i]]);
    c = __reduce_add_sync(0xffffffffu, c);
    if (lane == 0) {
      I.cnt[x] = c;
      if (c) atomicAdd(J.rows.csum + r / kRowChunk, c);
    }
  }
}

static uint32_t sg_smem(uint32_t vwords, int id_bytes) {
  constexpr uint32_t kW = kSgThreads / 32;
  return vwords * 4 + kW * 32 * 4 + vwords / 4 * 2 * 2 + kW * kSgList * id_bytes;
}
static void* sg_kernel(int id_bytes) {
  return id_bytes == 2 ? (void*)k_sg<uint16_t> : (void*)k_sg<uint32_t>;
}
int occupancy_sg(int id_bytes, uint32_t vwords) {
  const uint32_t smem = sg_smem(vwords, id_bytes);
  if (smem > 48 * 1024)
    cudaFuncSetAttribute(sg_kernel(id_bytes), cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  int occ = 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, sg_kernel(id_bytes), kSgThreads, smem);
  return occ;
}
cudaError_t launch_sg(const SgJob& job, int id_bytes, int grid, int sms, cudaStream_t s) {
  SgJob J = job;
  k_sg_init<<<sms * 8, kThreads, 0, s>>>(J);
  void* args[] = {&J};
  const cudaError_t e = cudaLaunchCooperativeKernel(sg_kernel(id_bytes), dim3(grid), dim3(kSgThreads),
                                                    args, sg_smem(J.rows.vwords, id_bytes), s);
  if (e != cudaSuccess) return e;
  k_sg_count<<<sms * 8, kThreads, 0, s>>>(J);
  return cudaGetLastError();
}

}  // namespace wg
