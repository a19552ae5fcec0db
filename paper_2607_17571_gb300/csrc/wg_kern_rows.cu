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
// pipeline -> rows: R-MAT 2^17 / 400k edges (4.8e8 tuples) 68.0 -> 5.35 ms (k_rows
// 3.50), R-MAT 2^19 / 400k (1.0e9 tuples, 64-bit keys) 164 -> 12.6 ms (7.69), ER
// 1,000 / 3,000 2.55 -> 0.10 ms, a chain of 1,000 vertices 147 -> 0.72 ms.
//
//   k_rows        the fixpoints of all rows (one CTA per row, rows claimed)
//   k_row_plan    row offsets (scan of the row counts), totals, capacity check
//   k_row_expand  bit sets -> sorted packed keys
#include "wg_device.cuh"
#include "wg_launch.h"
#include "wg_rows.cuh"

namespace wg {

// The vertex records, the bit set of vertices with out-edges, and the further
// units of a relation (edges in source order, the source of edge i is E[i] >> w);
// the bit set mp of the vertices with several parents.
template <typename K, typename IdT>
__global__ void __launch_bounds__(kThreads) k_row_layout(const K* E, uint32_t ne, uint32_t w,
                                                         const uint32_t* off, const uint32_t* adj,
                                                         uint32_t nv, IdT* rec, uint32_t* ns,
                                                         uint32_t words, IdT* units, uint32_t* mp) {
  constexpr uint32_t U = Unit<IdT>::n, kRecIds = U - 1, kTop = sizeof(IdT) == 2 ? 0xFFFFu : 0xFFFFFFFFu;
  const uint32_t stride = gridDim.x * kThreads, t = blockIdx.x * kThreads + threadIdx.x;
  for (uint32_t v = t; v < words * 32; v += stride) {
    uint32_t d = 0;
    if (v < nv) {
      d = off[v + 1] - off[v];
      rec[U * (size_t)v] = (IdT)min(d, kTop);
    }
    const uint32_t m = __ballot_sync(0xffffffffu, d > 0);
    if ((v & 31) == 0) ns[v >> 5] = m;
  }
  for (uint32_t i = t; i < ne; i += stride) {
    const uint32_t x = (uint32_t)(E[i] >> w), o = off[x], j = i - o, z = adj[i];
    const uint32_t bit = 1u << (z & 31);  // (mp: several parents; after it: at least one)
    if (atomicOr(mp + words + (z >> 5), bit) & bit) atomicOr(mp + (z >> 5), bit);
    IdT* to = j < kRecIds ? rec + U * (size_t)x + 1 + j
                          : units + (size_t)unit_start<IdT>(o, x) * U + (j - kRecIds);
    *to = (IdT)z;
    if (i + 1 == off[x + 1]) {
      const uint32_t room = j < kRecIds ? kRecIds - 1 - j : U - 1 - (j - kRecIds) % U;
      for (uint32_t r = 0; r < room; ++r) *++to = (IdT)z;
    }
  }
}

// Two-paths from every source (scratch `paths`, nv zeros): out[0] their maximum,
// out[1] their sum (zero before).  The edges are in source order, so most warps add
// once.
template <typename K>
__global__ void __launch_bounds__(kThreads) k_row_paths(const K* E, uint32_t ne, uint32_t w,
                                                        const uint32_t* off, const uint32_t* adj,
                                                        uint32_t* paths, unsigned long long* out) {
  const uint32_t stride = gridDim.x * kThreads, lane = threadIdx.x & 31;
  unsigned long long sum = 0;
  uint32_t top = 0;
  for (uint32_t i0 = (blockIdx.x * kThreads + threadIdx.x) & ~31u; i0 < ne; i0 += stride) {
    const uint32_t i = min(i0 + lane, ne - 1);
    const uint32_t x = (uint32_t)(E[i] >> w), z = adj[i];
    uint32_t d = i0 + lane < ne ? off[z + 1] - off[z] : 0u;
    sum += d;
    const bool same = __all_sync(0xffffffffu, x == __shfl_sync(0xffffffffu, x, 0));
    if (same) {
      d = __reduce_add_sync(0xffffffffu, d);
      if (lane) d = 0;
    }
    if (d) top = max(top, atomicAdd(paths + x, d) + d);
  }
  top = __reduce_max_sync(0xffffffffu, top);
  for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
  if (lane == 0) {
    atomicMax(out, (unsigned long long)top);
    atomicAdd(out + 1, sum);
  }
}

template <int T>
__device__ __forceinline__ void cta_sync() {
  if (T == 32) __syncwarp();
  else __syncthreads();
}

// One CTA takes a row through its whole fixpoint.  Shared memory: the row's bit
// set S and the candidates' bit set N of the next iteration.
// An iteration: the threads take 128 bits of N at a time, drop what S has, merge
// the rest (the delta) into S and list the delta's vertices that have out-edges
// (on the R-MAT workloads 4 to 5 in 10 have none); the warps then expand the
// list 32 vertices at a time: each lane its vertex's record, then the vertices'
// units as one strip, 32 units per step, a lane finding its unit's
// vertex from the bit mask of the strip's first units.  Setting a bit in the
// next N needs no answer, so a candidate costs one shared atomic and no list of
// winners is kept; scanning N costs words / 128 lane steps per iteration.  Two
// barriers per iteration; a delta of more than row_list(T) such vertices takes
// several rounds, the bits not yet listed waiting in the row's place in `bits`.
//
// kDry: a sample of the listed rows, of which only levels and tuples are counted
// (deep rows of wide relations go to the sorted-array pipeline, see rows_deep).
//
// Bound by the L1 / shared pipe, issue slots and barriers (ncu on R-MAT 2^15 / 100k,
// 324 us: pipe 76%, issue 62%, DRAM 0.05%; on ER 16,384 / 34,000 82% and 68%).
// What it measured on R-MAT 2^17 / 400k, whole call: winners of each
// bit listed by an answering atomic, records of 7 neighbours and single edges
// past them 16.1 ms; candidate bits without an answer, edges in 16-byte units,
// a list per warp (one barrier, but it waited for the warp with the most to
// expand) 8.3; one list per CTA 7.5; one N instead of two, no test per place 7.0; vertex
// records of 16 bytes 5.35.  With one warp (T = 32) an iteration is a chain of
// dependent instructions: a chain of 1,000 vertices took 1.09 ms with the counts in
// shared memory and one global atomic per iteration past its log, 1.02 with 32
// iterations' counts to an atomic, 0.84 with the list's length and the delta's size
// in registers, 0.72 without scan and barriers where no lane has two new vertices.
template <typename IdT, int T, int kMin, bool kDry = false>
__global__ void __launch_bounds__(T, kMin) k_rows(RowJob J) {
  constexpr uint32_t kW = T / 32, kList = row_list(T);
  constexpr bool kOne = kW == 1;  // one warp: counts stay in registers
  extern __shared__ uint4 sm4[];
  __shared__ RowInst I;
  __shared__ unsigned long long s_log[kRowLog];
  __shared__ uint32_t s_row[2], s_cnt[2], s_len[2];
  uint32_t* S = (uint32_t*)sm4;
  uint32_t* N = S + J.vwords;
  const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  uint32_t* strip = N + J.vwords + warp * 32;
  IdT* list = (IdT*)(N + J.vwords + kW * 32);
  unsigned long long cand = 0;
  uint32_t cur = 0xFFFFFFFFu;
  for (uint32_t i = tid; i < 2 * J.vwords; i += T) S[i] = 0;
  for (uint32_t i = tid; i < kRowLog; i += T) s_log[i] = 0;
  if (tid == 0) s_row[0] = atomicAdd(&J.ctl->next_row, 1u);
  __syncthreads();
  auto flush = [&]() {  // the counters of the current instance
    if (kDry) return;
    for (int o = 16; o > 0; o >>= 1) cand += __shfl_xor_sync(0xffffffffu, cand, o);
    if (lane == 0 && cand) atomicAdd(&J.inst[cur].cand, cand);
    cand = 0;
    for (uint32_t i = tid; i < kRowLog; i += T) {
      if (s_log[i] && i < I.log_cap) atomicAdd(I.log + i, s_log[i]);
      s_log[i] = 0;
    }
  };
  // listed rows (k_rows_small's leftovers): their bit sets lie in list order
  const uint32_t n_list = J.rows ? J.inst->n_big : J.nrows;
  const uint32_t nrows = kDry ? min(J.sample, n_list) : n_list;
  // no room, or a sample is wanted: the host sees to it and launches again
  if (J.rows && (nrows > J.slots || nrows > J.few)) return;
  for (uint32_t p = 0;; p ^= 1) {
    const uint32_t at_row = s_row[p];
    if (at_row >= nrows) break;
    // (a sample is spread over the list: neighbours are alike)
    const uint32_t at_list = kDry ? (uint32_t)(at_row * 4294967291ull % n_list) : at_row;
    const uint32_t row = J.rows ? J.rows[at_list] : at_row;
    const uint32_t q = J.chunk_inst ? J.chunk_inst[row / kRowChunk] : 0u;
    if (q != cur) {
      __syncthreads();
      if (cur != 0xFFFFFFFFu) flush();
      __syncthreads();
      if (tid == 0) I = J.inst[q];
      cur = q;
      __syncthreads();
    }
    // the next row, claimed here and stored at the end: nothing waits for it
    uint32_t next = 0;
    if (tid == 0) next = atomicAdd(&J.ctl->next_row, 1u);
    const uint32_t x = row - I.row0;
    uint32_t o = 0, deg = 0;
    if (x < I.nv) {  // (rows of an instance are padded to whole chunks)
      o = I.off[x];
      deg = I.off[x + 1] - o;
    }
    if (deg == 0) {
      if (tid == 0 && x < I.nv) I.cnt[x] = 0;
    } else {
      const uint32_t words = I.words, quads = words / 4;
      if (tid == 0) { s_cnt[0] = 0; s_len[0] = 0; cand += deg; }
      for (uint32_t i = tid; i < deg; i += T) {
        const uint32_t z = I.adj[o + i];
        atomicOr(N + (z >> 5), 1u << (z & 31));
      }
      __syncthreads();
      uint32_t lvl = 0, total = 0, turn = 0;
      // iterations past the log in shared memory: warp 0's lanes hold 32 of them
      uint32_t held = 0;
      auto log_held = [&](uint32_t first) {
        if (held && !kDry && first + lane < I.log_cap) atomicAdd(I.log + first + lane, (unsigned long long)held);
        held = 0;
      };
      uint4* const n4 = (uint4*)N;
      uint4* const out = (uint4*)(I.bits + (size_t)(J.rows ? at_row : x) * words);
      for (;; ++lvl) {
        uint32_t listed = 0, cnt = 0, wait = 0;  // wait: this thread's steps with bits not yet listed
        for (uint32_t round = 0;; ++round, turn ^= 1) {
          if (!kOne && tid == 0) s_len[turn ^ 1] = 0;
          uint32_t got = 0, len = 0;
          uint4 nd = {0, 0, 0, 0};
          if (round == 0 && tid < quads) nd = n4[tid];
          for (uint32_t g = warp * 32, step = 1; g < quads; g += T, step <<= 1) {
            const uint32_t w = g + lane;
            uint4 d = nd;
            if (round == 0) {
              nd = w + T < quads ? n4[w + T] : uint4{0, 0, 0, 0};
              if (d.x | d.y | d.z | d.w) {
                n4[w] = uint4{0, 0, 0, 0};
                const uint4 s = sm4[w], ns = __ldg((const uint4*)I.ns + w);
                d.x &= ~s.x; d.y &= ~s.y; d.z &= ~s.z; d.w &= ~s.w;
                sm4[w] = uint4{s.x | d.x, s.y | d.y, s.z | d.z, s.w | d.w};
                got += __popc(d.x) + __popc(d.y) + __popc(d.z) + __popc(d.w);
                d.x &= ns.x; d.y &= ns.y; d.z &= ns.z; d.w &= ns.w;
                if (lvl >= I.max_iters) d = uint4{0, 0, 0, 0};
              }
            } else if (wait & step) {
              d = out[w];
            }
            const uint32_t any = d.x | d.y | d.z | d.w;
            const uint32_t has = __ballot_sync(0xffffffffu, any != 0);
            if (!has) continue;
            const uint32_t c = __popc(d.x) + __popc(d.y) + __popc(d.z) + __popc(d.w);
            if (kOne && round == 0 && len + 32 <= kList && !__any_sync(0xffffffffu, c > 1)) {
              // at most one vertex a lane (a deep relation's deltas): no scan
              if (any)
                list[len + __popc(has & ((1u << lane) - 1))] =
                    (IdT)(w * 128 + (d.x ? 0 : d.y ? 32 : d.z ? 64 : 96) + __ffs(any) - 1);
              len += __popc(has);
              continue;
            }
            const uint32_t in = warp_incl_scan(c, lane);
            uint32_t at = 0;
            if (kOne) at = len, len += __shfl_sync(0xffffffffu, in, 31);
            else if (lane == 31) at = atomicAdd(s_len + turn, in);
            if (!kOne) at = __shfl_sync(0xffffffffu, at, 31);
            at += in - c;
            auto put = [&](uint32_t& m, uint32_t base) {
              while (m && at < kList) {
                list[at++] = (IdT)(base + __ffs(m) - 1);
                m &= m - 1;
              }
            };
            put(d.x, w * 128); put(d.y, w * 128 + 32); put(d.z, w * 128 + 64); put(d.w, w * 128 + 96);
            wait &= ~step;
            if (d.x | d.y | d.z | d.w) {
              out[w] = d;
              wait |= step;
            }
          }
          got = __reduce_add_sync(0xffffffffu, got);
          if (!kOne && lane == 0 && got) atomicAdd(s_cnt + (lvl & 1), got);
          cnt += got;  // (kOne)
          cta_sync<T>();
          if (!kOne) len = s_len[turn];
          const uint32_t n = min(len, kList);
          if (!kOne && round == 0 && tid == 0) s_cnt[~lvl & 1] = 0;
          listed |= len;
          if (len == 0) break;
          cand += expand_vertices<IdT, false>(I, list, warp * 32, n, T, N, strip);
          cta_sync<T>();
          if (len <= kList) break;
        }
        const uint32_t n = kOne ? cnt : s_cnt[lvl & 1];
        if (n == 0) break;
        total += n;
        if (lvl < kRowLog) {
          if (tid == 0) s_log[lvl] += n;
        } else if (warp == 0) {
          if (lane == (lvl & 31)) held = n;
          if ((lvl & 31) == 31) log_held(lvl & ~31u);
        }
        if (listed == 0) { ++lvl; break; }  // nothing of this delta joins any edge
        turn ^= 1;
      }
      if (warp == 0 && lvl > kRowLog) log_held((lvl - 1) & ~31u);
      if (kDry) {
        if (tid == 0) {
          atomicMax(&J.ctl->deepest, lvl);
          atomicAdd(&J.ctl->levels, (unsigned long long)lvl);
          atomicAdd(&J.ctl->tuples, (unsigned long long)total);
        }
      } else if (tid == 0) {  // (the delta of iteration lvl - 1 was the last that is not empty)
        atomicMax(&J.inst[q].last, lvl - 1);
        I.cnt[x] = total;
        atomicAdd(J.csum + row / kRowChunk, total);
      }
      // the row's bit set out, and cleared for the next row
      for (uint32_t i = tid; i < quads; i += T) {
        out[i] = sm4[i];
        sm4[i] = uint4{0, 0, 0, 0};
      }
    }
    if (tid == 0) s_row[p ^ 1] = next;
    __syncthreads();
  }
  if (cur != 0xFFFFFFFFu) flush();
}

// Rows of at most kSmallRow tuples, for relations whose bit sets are wide (one
// instance, 32-bit ranks): one warp per row, the reached vertices in a hash set
// and a list in shared memory, the sorted list out to small + row * kSmallRow.  A row
// that turns out longer is listed for k_rows.  Without it a sparse relation pays
// a bit set per row to hold a few vertices: ER 400,000 vertices / 360,000 edges,
// 335,000 rows of 9 tuples on average against bit sets of 42 KB, 15.5 ms on the
// sorted-array pipeline, 1.03 ms here (0.39 this kernel, 0.38 k_rows).  Bound by
// the latency of the gathered CSR entries.
__global__ void __launch_bounds__(kThreads) k_rows_small(RowJob J) {
  constexpr uint32_t kSlots = 2 * kSmallRow, kNone = 0xFFFFFFFFu;
  static_assert(kSlots >= kSmallRow + 64 && (kSlots & (kSlots - 1)) == 0, "the probes must end");
  __shared__ uint32_t s_hash[kWarps][kSlots], s_list[kWarps][kSmallRow], s_end[kWarps][kSmallRow + 1];
  __shared__ unsigned long long s_log[kRowLog];
  const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  uint32_t* hash = s_hash[warp];
  uint32_t* list = s_list[warp];
  uint32_t* ends = s_end[warp];  // list length after each level
  const RowInst& I = *J.inst;
  const uint32_t* off = I.off;
  const uint32_t* adj = I.adj;
  const uint32_t nv = I.nv, max_iters = I.max_iters;
  for (uint32_t i = tid; i < kRowLog; i += kThreads) s_log[i] = 0;
  for (uint32_t i = lane; i < kSlots; i += 32) hash[i] = kNone;
  __syncthreads();
  unsigned long long cand = 0;
  uint32_t last = 0;
  for (uint32_t x = blockIdx.x * kWarps + warp; x < nv; x += gridDim.x * kWarps) {
    const uint32_t o = off[x], deg = off[x + 1] - o;
    if (deg == 0) {
      if (lane == 0) I.cnt[x] = 0;
      continue;
    }
    uint32_t n = 0, lvl = 0, mine = lane == 0 ? deg : 0;
    // adds the lanes' vertices z that are new to the list; false when it is full
    auto add = [&](uint32_t z, bool valid) {
      bool fresh = false;
      if (valid) {
        uint32_t h = (z * 2654435761u) >> 16 & (kSlots - 1);
        for (;;) {  // (at most kSmallRow + 32 of the slots are taken)
          const uint32_t old = atomicCAS(hash + h, kNone, z);
          if (old == kNone) { fresh = true; break; }
          if (old == z) break;
          h = (h + 1) & (kSlots - 1);
        }
      }
      const uint32_t m = __ballot_sync(0xffffffffu, fresh);
      const uint32_t at = n + __popc(m & ((1u << lane) - 1));
      n += __popc(m);
      if (n > kSmallRow) return false;
      if (fresh) list[at] = z;
      return true;
    };
    bool fits = deg <= kSmallRow;
    for (uint32_t i = 0; i < deg && fits; i += 32) fits = add(i + lane < deg ? adj[o + i + lane] : 0u, i + lane < deg);
    uint32_t start = 0;
    while (fits) {
      __syncwarp();
      if (lane == 0) ends[lvl] = n;
      const uint32_t end = n;
      if (lvl >= max_iters) { ++lvl; break; }
      for (uint32_t b = start; b < end && fits; b += 32) {
        uint32_t fo = 0, d = 0;
        if (b + lane < end) {
          const uint32_t y = list[b + lane];
          fo = off[y];
          d = off[y + 1] - fo;
        }
        const uint32_t in = warp_incl_scan(d, lane), tot = __shfl_sync(0xffffffffu, in, 31);
        mine += d;
        const uint32_t fe = fo - (in - d);  // edge e of the strip is adj[fe of its vertex + e]
        for (uint32_t e0 = 0; e0 < tot && fits; e0 += 32) {
          const uint32_t e = e0 + lane;
          uint32_t ow = 0;  // lanes whose edges all come before e
#pragma unroll
          for (int st = 16; st > 0; st >>= 1) {
            const uint32_t v = __shfl_sync(0xffffffffu, in, ow + st - 1);
            if (v <= e) ow += st;
          }
          const uint32_t a = __shfl_sync(0xffffffffu, fe, ow & 31);
          fits = add(e < tot ? adj[a + e] : 0u, e < tot);
        }
      }
      ++lvl;
      if (n == end) break;  // an empty delta
      start = end;
    }
    if (fits) {
      // the list in order: each lane ranks its vertices against all
      __syncwarp();
      uint32_t* to = J.small + (size_t)x * kSmallRow;
      for (uint32_t i = lane; i < n; i += 32) {
        const uint32_t v = list[i];
        uint32_t r = 0;
        for (uint32_t j = 0; j < n; ++j) r += list[j] < v;
        to[r] = v;
      }
      cand += mine;
      last = max(last, lvl - 1);
      for (uint32_t l = lane; l < lvl; l += 32) {
        const unsigned long long c = ends[l] - (l ? ends[l - 1] : 0u);
        if (l < kRowLog) atomicAdd(s_log + l, c);
        else if (l < I.log_cap) atomicAdd(I.log + l, c);
      }
      if (lane == 0) {
        I.cnt[x] = n;
        atomicAdd(J.csum + x / kRowChunk, n);
      }
    } else if (lane == 0) {
      J.rows[atomicAdd(&J.inst->n_big, 1u)] = x;
    }
    __syncwarp();
    for (uint32_t i = lane; i < kSlots; i += 32) hash[i] = kNone;
    __syncwarp();
  }
  for (int o = 16; o > 0; o >>= 1) cand += __shfl_xor_sync(0xffffffffu, cand, o);
  if (lane == 0) {
    if (cand) atomicAdd(&J.inst->cand, cand);
    atomicMax(&J.inst->last, last);
  }
  __syncthreads();
  for (uint32_t i = tid; i < kRowLog; i += kThreads)
    if (s_log[i] && i < I.log_cap) atomicAdd(I.log + i, s_log[i]);
}

// Small rows -> sorted packed keys: a warp takes 32 rows.
template <typename K>
__global__ void __launch_bounds__(kThreads) k_row_expand_small(RowJob J) {
  const uint32_t lane = threadIdx.x & 31;
  const RowInst& I = *J.inst;
  if (!I.fits) return;
  for (uint32_t r = (blockIdx.x * kThreads + threadIdx.x) & ~31u; r < I.nv; r += gridDim.x * kThreads) {
    const uint32_t r0 = r / kRowChunk * kRowChunk;
    uint32_t before = 0;
    for (uint32_t i = r0 + lane; i < r; i += 32) before += I.cnt[i];
    before = __reduce_add_sync(0xffffffffu, before);
    const uint32_t c = r + lane < I.nv ? I.cnt[r + lane] : 0u, in = warp_incl_scan(c, lane);
    K* out = (K*)I.out + J.cbase[r / kRowChunk] + before;
    for (uint32_t k = 0; k < 32; ++k) {
      const uint32_t n = __shfl_sync(0xffffffffu, c, k), at = __shfl_sync(0xffffffffu, in, k) - n;
      if (n > kSmallRow) continue;
      for (uint32_t i = lane; i < n; i += 32)
        out[at + i] = ((K)(r + k) << I.w) | J.small[(size_t)(r + k) * kSmallRow + i];
    }
  }
}

// The start of a single query: its instance, from the launch's arguments, and the
// cleared scratch (one launch in place of two small copies and a memset).
__global__ void __launch_bounds__(kThreads) k_row_begin(RowJob J, RowInst I, SgInst G, uint4* clear,
                                                        size_t n) {
  const size_t t = (size_t)blockIdx.x * kThreads + threadIdx.x;
  if (t == 0) {
    *J.inst = I;
    if (J.sg) *(SgInst*)J.sg = G;
  }
  for (size_t i = t; i < n; i += (size_t)gridDim.x * kThreads) clear[i] = uint4{0, 0, 0, 0};
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
    I->fits = carry <= I->out_cap && !(J.rows && (J.sample || I->n_big > min(J.slots, J.few))) ? 1u : 0u;
    if (RowReport* r = J.report) {
      r->n_total = carry;
      r->cand = I->cand;
      r->last = I->last;
      r->fits = I->fits;
      r->n_big = I->n_big;
      r->error = J.sg_ctl ? J.sg_ctl->error : 0u;
      if (J.sample) {
        r->levels = J.ctl->levels;
        r->tuples = J.ctl->tuples;
        r->deepest = J.ctl->deepest;
      }
    }
  }
  if (J.report && threadIdx.x < kRowLog)
    J.report->log[threadIdx.x] = threadIdx.x < I->log_cap ? I->log[threadIdx.x] : 0ull;
}

// Bit sets -> sorted packed keys (x << w) | z, one warp per row: 64 words at a
// time, each lane lists the set bits of its two words at its prefix in the
// warp's shared buffer, then the warp writes the list coalesced.  kMasked
// (same-generation): of each row the 128-bit pieces marked valid only, 16 at a
// time; a step that is a quarter full is written a word at a time by the whole
// warp (unmasked rows of low-degree graphs, 2/3 full, lose 5% by that).
// 7.5e7 same-generation tuples, rows of nearly full pieces: 0.31 -> 0.18 ms with
// the padding and the word steps (ncu had the buffer's bank conflicts at 87% of
// the L1 pipe).
template <typename K, bool kMasked>
__global__ void __launch_bounds__(kThreads) k_row_expand(RowJob J) {
  __shared__ uint16_t s_buf[kWarps][2048 + 64], s_list[kMasked ? kWarps : 1][kMasked ? kSgMaxVertices / 128 : 1];
  const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t below = (1u << lane) - 1;
  constexpr uint32_t kDense = 512;  // of 2,048 bits
  // (valid pieces are often nearly full, so lanes list some 64 places apart: two
  // places of padding spread the banks; unmasked rows are sparser, and it costs
  // them more than it saves: 0.62 against 0.56 ms for 4.8e8 tuples)
  auto pad = [](uint32_t at) { return kMasked ? at + (at >> 6) * 2 : at; };
  uint16_t* buf = s_buf[warp];
  uint16_t* list = s_list[kMasked ? warp : 0];
  const uint32_t stride = gridDim.x * kWarps, nrows = J.rows ? J.inst->n_big : J.nrows;
  for (uint32_t i = blockIdx.x * kWarps + warp; i < nrows; i += stride) {
    const uint32_t row = J.rows ? J.rows[i] : i;
    const uint32_t ch = row / kRowChunk;
    const uint32_t q = J.chunk_inst ? J.chunk_inst[ch] : 0u;
    const RowInst* I = J.inst + q;
    const uint32_t x = row - I->row0;
    if (x >= I->nv || !I->fits) continue;
    const uint32_t n = I->cnt[x];
    if (n == 0) continue;
    // this row's offset: the chunk's, and the rows before it in the chunk
    const uint32_t r0 = x / kRowChunk * kRowChunk;
    uint32_t before = 0;
    for (uint32_t r = r0 + lane; r < x; r += 32) before += I->cnt[r];
    before = __reduce_add_sync(0xffffffffu, before);
    K* out = (K*)I->out + J.cbase[ch] + before;
    const uint2* w2 = (const uint2*)(I->bits + (size_t)(J.rows ? i : x) * I->words);
    uint32_t np = I->words / 2;  // pairs of words to list
    if (kMasked) {
      const SgInst* G = J.sg + q;
      np = 2 * list_pieces(lane < G->mw ? G->fm[(size_t)x * G->mw + lane] : 0u, list);
      __syncwarp();
    }
    // the place in the row of the p-th pair listed
    auto place = [&](uint32_t p) { return kMasked ? 2u * list[p >> 1] + (p & 1u) : p; };
    const K hi = (K)x << I->w;
    uint2 v = lane < np ? w2[place(lane)] : uint2{0, 0};
    for (uint32_t b = 0; b < np; b += 32) {
      const uint32_t nx = b + 32 + lane;
      const uint2 nextv = nx < np ? w2[place(nx)] : uint2{0, 0};
      const uint32_t c = __popc(v.x) + __popc(v.y), in = warp_incl_scan(c, lane);
      const uint32_t tot = __shfl_sync(0xffffffffu, in, 31);
      if (kMasked && tot >= kDense) {
        // dense: the warp takes a word at a time, a lane per bit
        uint32_t off = 0;
        for (uint32_t j = 0; j < 64; ++j) {
          const uint32_t m = __shfl_sync(0xffffffffu, j & 1 ? v.y : v.x, j >> 1);
          if (m >> lane & 1u)
            out[off + __popc(m & below)] = hi + (K)place(b + (j >> 1)) * 64 + ((j & 1u) * 32 + lane);
          off += __popc(m);
        }
        out += tot;
      } else if (tot) {
        auto put = [&](uint32_t at, uint32_t m, uint32_t base) {
          for (; m; m &= m - 1, ++at) buf[pad(at)] = (uint16_t)(base + __ffs(m) - 1);
        };
        put(in - c, v.x, lane * 64);
        put(in - __popc(v.y), v.y, lane * 64 + 32);
        __syncwarp();
        for (uint32_t j = lane; j < tot; j += 32) {
          const uint32_t t = buf[pad(j)];
          out[j] = kMasked ? hi + (K)place(b + (t >> 6)) * 64 + (t & 63u) : hi + (K)b * 64 + t;
        }
        out += tot;
        __syncwarp();
      }
      v = nextv;
    }
    if (kMasked) __syncwarp();
  }
}

// ------------------------------------------------------------------ launchers
static uint32_t row_smem(uint32_t vwords, int id_bytes, int threads) {
  return 2 * vwords * 4 + (threads / 32) * 32 * 4 + row_list(threads) * id_bytes;
}
// Threads per CTA: a CTA waits twice per iteration for its slowest warp, so the
// smaller the better while its bit sets leave room for enough CTAs per SM.
// Whole calls, 32 / 64 / 128 / 256 / 512 threads: chain of 1,000 (32 words) 0.72 /
// 1.18 / 1.17 / 2.1 / 2.4 ms; the 64-query batch (up to 512) 12.3 / 12.3 / 13.1 ms;
// R-MAT 2^15 / 100k (750) - / 537 / 510 us; R-MAT 2^17 / 400k (1,900) - / 7.3 / 7.0 /
// 7.2 / 8.4 ms and 2^19 / 400k (3,900 words) - / 22.7 / 16.8 / 15.2 / 16.9 ms (both
// before the 16-byte records).  From 131,072 vertices two CTAs of 512 share an SM
// while their bit sets allow (k_rows on ER 400,000 / 360,000: 0.95 against 1.48 ms
// with one of 1,024).
static int row_threads(uint32_t vwords) {
  return vwords <= 128    ? 32
         : vwords <= 512  ? 64
         : vwords <= 2048 ? 128
         : vwords <= 4096 ? 256
         : vwords <= 12800 ? 512
                           : 1024;
}

// Time of one candidate in a row that has its CTA to itself and the others idle:
// one hub of 500 to 5,000 children with the same 1,000 to 60,000 children each.
double row_candidate_ns(uint32_t vwords) {
  const int t = row_threads(vwords);
  return t == 32 ? 1.08 : t == 64 ? 0.68 : t <= 256 ? 0.57 : t == 512 ? 0.27 : 0.17;
}

template <typename F>
static auto rows_kernel(uint32_t vwords, int id_bytes, F f) {
  const int t = row_threads(vwords);
  if (id_bytes == 2)  // (at most 2,048 words)
    return t == 32   ? f(k_rows<uint16_t, 32, 32>)
           : t == 64 ? f(k_rows<uint16_t, 64, 20>)
                     : f(k_rows<uint16_t, 128, 10>);
  return t == 256   ? f(k_rows<uint32_t, 256, 5>)  // (more than 2,048)
         : t == 512 ? f(k_rows<uint32_t, 512, 2>)
                    : f(k_rows<uint32_t, 1024, 1>);
}
int occupancy_rows(int id_bytes, uint32_t vwords) {
  const int t = row_threads(vwords);
  const uint32_t smem = row_smem(vwords, id_bytes, t);
  return rows_kernel(vwords, id_bytes, [&](auto k) {
    if (smem > 48 * 1024)
      cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kRowSmemMax);
    int occ = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k, t, smem);
    return occ;
  });
}
void launch_rows(const RowJob& J, int id_bytes, int grid, cudaStream_t s) {
  const int t = row_threads(J.vwords);
  const uint32_t smem = row_smem(J.vwords, id_bytes, t);
  if (J.sample) {  // (more than 2^18 vertices)
    auto k = t == 512 ? k_rows<uint32_t, 512, 2, true> : k_rows<uint32_t, 1024, 1, true>;
    cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kRowSmemMax);
    k<<<grid, t, smem, s>>>(J);
    return;
  }
  rows_kernel(J.vwords, id_bytes, [&](auto k) {
    k<<<grid, t, smem, s>>>(J);
    return 0;
  });
}
void launch_row_plan(const RowJob& J, uint32_t n_inst, cudaStream_t s) {
  k_row_plan<<<n_inst, 1024, 0, s>>>(J);
}
void launch_row_begin(const RowJob& J, const RowInst& I, const SgInst& G, void* clear,
                      size_t bytes, int sms, cudaStream_t s) {
  const size_t n = bytes / 16, ctas = (n + kThreads - 1) / kThreads;
  k_row_begin<<<(int)min(max(ctas, (size_t)1), (size_t)sms * 8), kThreads, 0, s>>>(J, I, G,
                                                                                 (uint4*)clear, n);
}
void launch_rows_small(const RowJob& J, int grid, cudaStream_t s) {
  k_rows_small<<<grid, kThreads, 0, s>>>(J);
}
template <typename K>
void launch_row_expand(const RowJob& J, int grid, cudaStream_t s) {
  if (J.rows) k_row_expand_small<K><<<grid, kThreads, 0, s>>>(J);
  if (J.sg) k_row_expand<K, true><<<grid, kThreads, 0, s>>>(J);
  else k_row_expand<K, false><<<grid, kThreads, 0, s>>>(J);
}
template <typename K>
void launch_row_paths(const K* E, uint32_t ne, uint32_t w, const uint32_t* off, const uint32_t* adj,
                      uint32_t* paths, unsigned long long* out, int grid, cudaStream_t s) {
  k_row_paths<K><<<grid, kThreads, 0, s>>>(E, ne, w, off, adj, paths, out);
}
template void launch_row_paths<uint32_t>(const uint32_t*, uint32_t, uint32_t, const uint32_t*,
                                         const uint32_t*, uint32_t*, unsigned long long*, int,
                                         cudaStream_t);
template void launch_row_paths<unsigned long long>(const unsigned long long*, uint32_t, uint32_t,
                                                   const uint32_t*, const uint32_t*, uint32_t*,
                                                   unsigned long long*, int, cudaStream_t);
size_t row_units(uint64_t ne, uint32_t nv, int id_bytes) {
  const uint64_t U = 16 / id_bytes;
  return (size_t)((ne + (U - 1) * ((uint64_t)nv + 1)) / U + 1);
}
template <typename K>
void launch_row_layout(const K* E, uint32_t ne, uint32_t w, const uint32_t* off,
                       const uint32_t* adj, uint32_t nv, void* rec, uint32_t* ns, uint32_t words,
                       void* units, uint32_t* mp, int id_bytes, int grid, cudaStream_t s) {
  cudaMemsetAsync(mp, 0, (size_t)words * 8, s);
  if (id_bytes == 2)
    k_row_layout<K, uint16_t><<<grid, kThreads, 0, s>>>(E, ne, w, off, adj, nv, (uint16_t*)rec, ns,
                                                        words, (uint16_t*)units, mp);
  else
    k_row_layout<K, uint32_t><<<grid, kThreads, 0, s>>>(E, ne, w, off, adj, nv, (uint32_t*)rec, ns,
                                                        words, (uint32_t*)units, mp);
}
template void launch_row_expand<uint32_t>(const RowJob&, int, cudaStream_t);
template void launch_row_expand<unsigned long long>(const RowJob&, int, cudaStream_t);
template void launch_row_layout<uint32_t>(const uint32_t*, uint32_t, uint32_t, const uint32_t*,
                                          const uint32_t*, uint32_t, void*, uint32_t*, uint32_t,
                                          void*, uint32_t*, int, int, cudaStream_t);
template void launch_row_layout<unsigned long long>(const unsigned long long*, uint32_t, uint32_t,
                                                    const uint32_t*, const uint32_t*, uint32_t,
                                                    void*, uint32_t*, uint32_t, void*, uint32_t*,
                                                    int, int, cudaStream_t);

}  // namespace wg
