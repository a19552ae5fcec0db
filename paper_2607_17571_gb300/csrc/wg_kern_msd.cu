// wg_kern_msd.cu -- radix sort of a large array by its top digit first (sm_103a).
//
// The lookback passes (k_sort_pass) read and write every key once per 7 or 8 bits
// and must keep their order from the second pass on.  Here one pass partitions
// the keys by their top B bits -- in any order within a bin, so it needs neither
// stable ranks nor a lookback: each tile counts its bins in shared memory and
// reserves its places with one global atomic per bin -- and then a CTA sorts each
// bin, which fits its shared memory, on the remaining bits: three sweeps over HBM
// in all (count, partition, bins) whatever the key width.  Keys whose top bits are
// skewed (a bin over kMsdCap keys) go to the lookback passes: a sample finds most
// of them in a few microseconds, the exact count the rest.
//
// 2^24 uniform 64-bit keys on 34 bits: whole call 276 us (1,054 with the lookback
// passes' five; 399 with the partition's keys written from where they were read, 652
// with the bins also sorted by three LSD passes, both with two read-backs); 48 bits
// 276, 1,227, 396 and 864.  Bound by shared memory: one counting atomic and two
// staged moves a key and kernel.
#include "wg_device.cuh"
#include "wg_launch.h"

namespace wg {

template <typename K>
__device__ __forceinline__ uint32_t msd_bin(const MsdJob& J, K k) {
  return (uint32_t)(k >> (J.bits - J.top)) & ((1u << J.top) - 1);
}

// A sample of the keys: are 2^8 (or fewer) bins of the top bits about even?  Clears
// the bins' counts too.
template <typename K>
__global__ void __launch_bounds__(1024) k_msd_probe(MsdJob J) {
  constexpr uint32_t kSample = 4096;
  __shared__ uint32_t cnt[256], s_max;
  const K* in = (const K*)J.in;
  const uint32_t t = threadIdx.x, coarse = min(J.top, 8u);
  if (t < 256) cnt[t] = 0;
  if (t == 0) s_max = 0;
  for (uint32_t i = t; i < 1u << J.top; i += 1024) J.cnt[i] = 0;
  __syncthreads();
  const uint32_t step = J.n / kSample;  // (at least 1: n >= kMsdMin)
#pragma unroll
  for (uint32_t i = t; i < kSample; i += 1024)
    atomicAdd(cnt + (msd_bin(J, in[(size_t)i * step]) >> (J.top - coarse)), 1u);
  __syncthreads();
  if (t < 256) atomicMax(&s_max, cnt[t]);
  __syncthreads();
  if (t == 0) {
    // twice the even share and some: a fuller bin would rarely fit
    const uint32_t ok = s_max <= 2 * (kSample >> coarse) + 16 ? 1u : 0u;
    J.state->ok = ok;
    J.state->next = 0;
    if (!ok) *J.report = 0;
  }
}

// Keys per bin.
template <typename K>
__global__ void __launch_bounds__(1024) k_msd_count(MsdJob J) {
  extern __shared__ uint32_t cnt[];
  const uint32_t nb = 1u << J.top;
  if (!J.state->ok) return;
  for (uint32_t i = threadIdx.x; i < nb; i += 1024) cnt[i] = 0;
  __syncthreads();
  const K* in = (const K*)J.in;
  for (uint32_t t = blockIdx.x * kMsdTile; t < J.n; t += gridDim.x * kMsdTile) {
    K k[16];
#pragma unroll
    for (int e = 0; e < 16; ++e) {
      const uint32_t i = t + threadIdx.x + e * 1024;
      k[e] = i < J.n ? __ldcs(in + i) : (K)0;
    }
#pragma unroll
    for (int e = 0; e < 16; ++e)
      if (t + threadIdx.x + e * 1024 < J.n) atomicAdd(cnt + msd_bin(J, k[e]), 1u);
  }
  __syncthreads();
  for (uint32_t i = threadIdx.x; i < nb; i += 1024)
    if (cnt[i]) atomicAdd(J.cnt + i, cnt[i]);
}

// Bin offsets, and whether every bin fits.
__global__ void __launch_bounds__(1024) k_msd_plan(MsdJob J) {
  __shared__ uint32_t sh[32], s_max;
  const uint32_t nb = 1u << J.top, t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const uint32_t per = (nb + 1023) / 1024, b0 = t * per;
  if (!J.state->ok) return;
  if (t == 0) s_max = 0;
  __syncthreads();
  uint32_t sum = 0, top = 0;
  for (uint32_t i = b0; i < min(b0 + per, nb); ++i) {
    const uint32_t c = J.cnt[i];
    sum += c;
    top = max(top, c);
  }
  atomicMax(&s_max, top);
  uint32_t in = sum;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, in, o);
    if (lane >= (uint32_t)o) in += y;
  }
  if (lane == 31) sh[warp] = in;
  __syncthreads();
  uint32_t before = in - sum;
  for (uint32_t w = 0; w < warp; ++w) before += sh[w];
  for (uint32_t i = b0; i < min(b0 + per, nb); ++i) {
    J.off[i] = before;
    J.cur[i] = before;
    before += J.cnt[i];
  }
  if (t == 0) {
    J.state->ok = *J.report = s_max <= kMsdCap ? 1u : 0u;
  }
}

// Keys to their bins, in any order.  A tile is put in bin order in shared memory
// first, so that a bin's keys (4 on average at 2^12 bins) leave as one run; the
// next tile's loads are in flight meanwhile.
template <typename K>
__global__ void __launch_bounds__(1024) k_msd_partition(MsdJob J) {
  extern __shared__ __align__(16) unsigned long long smem_part[];  // [kMsdTile] keys | [bins]
  __shared__ uint32_t s_sum[32];
  K* buf = (K*)smem_part;
  uint32_t* cnt = (uint32_t*)(buf + kMsdTile);  // keys of the bin; first place in buf | keys << 16; to out
  static_assert(kMsdTile < 1u << 16, "a place and a count share a word");
  const uint32_t nb = 1u << J.top, t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const uint32_t per = (nb + 1023) / 1024;
  const K* in = (const K*)J.in;
  K* out = (K*)J.tmp;
  K k[16];
  auto load = [&](size_t tile) {
#pragma unroll
    for (int e = 0; e < 16; ++e) {
      const size_t i = tile + t + e * 1024;
      k[e] = i < J.n ? __ldcs(in + i) : (K)0;
    }
  };
  size_t tile = (size_t)blockIdx.x * kMsdTile;
  load(tile);
  for (; tile < J.n; tile += (size_t)gridDim.x * kMsdTile) {
    const uint32_t m = (uint32_t)min((size_t)kMsdTile, J.n - tile);
    for (uint32_t i = t; i < nb; i += 1024) cnt[i] = 0;
    __syncthreads();
    uint32_t rank[8];  // two 16-bit ranks each
#pragma unroll
    for (int e = 0; e < 16; ++e) {
      uint32_t r = 0;
      if (t + e * 1024 < m) r = atomicAdd(cnt + msd_bin(J, k[e]), 1u);
      rank[e >> 1] = e & 1 ? rank[e >> 1] | r << 16 : r;
    }
    __syncthreads();
    const uint32_t b0 = min(t * per, nb), b1 = min(b0 + per, nb);
    uint32_t sum = 0;
    for (uint32_t i = b0; i < b1; ++i) sum += cnt[i];
    uint32_t inc = sum;
#pragma unroll
    for (int q = 1; q < 32; q <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, inc, q);
      if (lane >= (uint32_t)q) inc += y;
    }
    if (lane == 31) s_sum[warp] = inc;
    __syncthreads();
    const uint32_t ws = s_sum[lane];
    uint32_t at = __reduce_add_sync(0xffffffffu, lane < warp ? ws : 0u) + inc - sum;
    for (uint32_t i = b0; i < b1; ++i) {
      const uint32_t c = cnt[i];
      cnt[i] = at | c << 16;
      at += c;
    }
    __syncthreads();
#pragma unroll
    for (int e = 0; e < 16; ++e)
      if (t + e * 1024 < m)
        buf[(cnt[msd_bin(J, k[e])] & 0xFFFFu) + (rank[e >> 1] >> (e & 1 ? 16 : 0) & 0xFFFFu)] = k[e];
    load(tile + (size_t)gridDim.x * kMsdTile);
    __syncthreads();
    for (uint32_t i = t; i < nb; i += 1024) {
      const uint32_t v = cnt[i], c = v >> 16;
      if (c) cnt[i] = atomicAdd(J.cur + i, c) - (v & 0xFFFFu);
    }
    __syncthreads();
#pragma unroll
    for (int e = 0; e < 16; ++e) {
      const uint32_t i = t + e * 1024;
      if (i < m) {
        const K key = buf[i];
        out[cnt[msd_bin(J, key)] + i] = key;
      }
    }
    __syncthreads();
  }
}

// Each bin sorted on the bits below its own, in shared memory.  Equal keys are
// alike, so no order has to be kept: the next kMsdFine bits split the bin into
// about as many buckets as it has keys (one shared atomic per key), and a key's
// place in its bucket is the number of smaller ones, found by comparing.  A bin
// whose buckets would take more than about eight comparisons per key, or that has
// one of more than 64, goes through LSD passes of at most 8 bits instead (a warp
// ranks its consecutive keys with match_any).
template <typename K>
__global__ void __launch_bounds__(kMsdThreads, sizeof(K) == 4 ? 3 : 2) k_msd_bins(MsdJob J) {
  extern __shared__ __align__(16) unsigned long long smem_bins[];  // [kMsdCap] keys | [warps][256] counters
  constexpr uint32_t kW = kMsdThreads / 32, kItems = kMsdCap / kMsdThreads;
  __shared__ uint32_t s_sum[kW], s_bin, s_cost;
  K* buf = (K*)smem_bins;
  uint32_t* cnt = (uint32_t*)(buf + kMsdCap);
  const uint32_t t = threadIdx.x, lane = t & 31, warp = t >> 5, below = (1u << lane) - 1;
  uint32_t* mine = cnt + warp * 256;
  const uint32_t low = J.bits - J.top, passes = (low + 7) / 8, dbits = passes ? (low + passes - 1) / passes : 0;
  const uint32_t mask = (1u << dbits) - 1;
  constexpr uint32_t kFine = 1u << kMsdFine, kPer = kFine / kMsdThreads;
  static_assert(kFine <= kW * 256 && kPer % 4 == 0, "the buckets' counters take the passes' room");
  const uint32_t fshift = low > kMsdFine ? low - kMsdFine : 0;  // (low >= 1)
  const uint32_t fmask = (1u << min(low, kMsdFine)) - 1;
  const K* in = (const K*)J.tmp;
  K* out = (K*)J.out;
  for (;;) {
    if (t == 0) {
      s_bin = atomicAdd(&J.state->next, 1u);
      s_cost = 0;
    }
    for (uint32_t i = t; i < kFine / 4; i += kMsdThreads) ((uint4*)cnt)[i] = uint4{0, 0, 0, 0};
    __syncthreads();
    const uint32_t b = s_bin;
    if (b >= 1u << J.top) return;
    const uint32_t o = J.off[b], m = J.cnt[b];
    if (m == 0) {
      __syncthreads();
      continue;
    }
    // warp w holds keys [w * run, (w + 1) * run) of the bin, 32 at a time
    const uint32_t items = (m + kMsdThreads - 1) / kMsdThreads, run = items * 32, w0 = warp * run;
    K k[kItems];
#pragma unroll
    for (uint32_t e = 0; e < kItems; ++e) {
      if (e >= items) break;
      const uint32_t i = w0 + e * 32 + lane;
      k[e] = i < m ? __ldcs(in + o + i) : (K)0;
    }
    uint32_t rank[kItems / 2];  // two 16-bit ranks within the digit each
    uint32_t cost = 0;
#pragma unroll
    for (uint32_t e = 0; e < kItems; ++e) {
      if (e >= items) break;
      uint32_t r = 0;
      if (w0 + e * 32 + lane < m) r = atomicAdd(cnt + ((uint32_t)(k[e] >> fshift) & fmask), 1u);
      cost += r < 64 ? r : 4 * kMsdCap;
      rank[e >> 1] = e & 1 ? rank[e >> 1] | r << 16 : r;
    }
    cost = __reduce_add_sync(0xffffffffu, cost);
    if (lane == 0 && cost) atomicAdd(&s_cost, cost);
    __syncthreads();
    const bool fine = !fshift || s_cost <= 4 * m;  // (twice s_cost comparisons)
    if (fine) {
      uint32_t c[kPer], sum = 0;
#pragma unroll
      for (uint32_t i = 0; i < kPer; i += 4) *(uint4*)(c + i) = *(const uint4*)(cnt + t * kPer + i);
#pragma unroll
      for (uint32_t i = 0; i < kPer; ++i) {
        const uint32_t v = c[i];
        c[i] = sum;
        sum += v;
      }
      uint32_t inc = sum;
#pragma unroll
      for (int q = 1; q < 32; q <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, inc, q);
        if (lane >= (uint32_t)q) inc += y;
      }
      if (lane == 31) s_sum[warp] = inc;
      __syncthreads();
      uint32_t ws = lane < kW ? s_sum[lane] : 0u;
      ws = lane < warp ? ws : 0u;
      const uint32_t base = __reduce_add_sync(0xffffffffu, ws) + inc - sum;
#pragma unroll
      for (uint32_t i = 0; i < kPer; ++i) c[i] += base;
#pragma unroll
      for (uint32_t i = 0; i < kPer; i += 4) *(uint4*)(cnt + t * kPer + i) = *(const uint4*)(c + i);
      __syncthreads();
#pragma unroll
      for (uint32_t e = 0; e < kItems; ++e) {
        if (e >= items) break;
        if (w0 + e * 32 + lane < m)
          buf[cnt[(uint32_t)(k[e] >> fshift) & fmask] + (rank[e >> 1] >> (e & 1 ? 16 : 0) & 0xFFFFu)] = k[e];
      }
      __syncthreads();
      for (uint32_t i = t; i < m; i += kMsdThreads) {
        const K key = buf[i];
        uint32_t at = i;
        if (fshift) {
          const uint32_t d = (uint32_t)(key >> fshift) & fmask;
          const uint32_t j0 = cnt[d], j1 = d < kFine - 1 ? cnt[d + 1] : m;
          at = j0;
          for (uint32_t j = j0; j < j1; ++j) {
            const K other = buf[j];
            at += other < key || (other == key && j < i);
          }
        }
        out[o + at] = key;
      }
      __syncthreads();
      continue;
    }
    for (uint32_t p = 0; p < passes; ++p) {
      const uint32_t shift = p * dbits;
      for (uint32_t i = lane; i < 256; i += 32) mine[i] = 0;
      __syncwarp();
#pragma unroll
      for (uint32_t e = 0; e < kItems; ++e) {
        if (e >= items) break;
        const bool on = w0 + e * 32 + lane < m;
        const uint32_t d = on ? (uint32_t)(k[e] >> shift) & mask : 256u;
        const uint32_t same = __match_any_sync(0xffffffffu, d);
        const uint32_t before = on ? mine[d] : 0u;
        __syncwarp();
        if (on && !(same & below)) mine[d] = before + __popc(same);
        __syncwarp();
        const uint32_t r = before + __popc(same & below);
        rank[e >> 1] = e & 1 ? rank[e >> 1] | r << 16 : r;
      }
      __syncthreads();
      // each digit's places: before it all smaller digits, then the warps in order
      if (t < 256) {
        uint32_t sum = 0;
#pragma unroll
        for (uint32_t w = 0; w < kW; ++w) {
          const uint32_t c = cnt[w * 256 + t];
          cnt[w * 256 + t] = sum;
          sum += c;
        }
        uint32_t inc = sum;
#pragma unroll
        for (int q = 1; q < 32; q <<= 1) {
          const uint32_t y = __shfl_up_sync(0xffffffffu, inc, q);
          if (lane >= (uint32_t)q) inc += y;
        }
        if (lane == 31) s_sum[warp] = inc;
        asm volatile("bar.sync 1, 256;" ::: "memory");
        uint32_t base = inc - sum;
        for (uint32_t w = 0; w < warp; ++w) base += s_sum[w];
#pragma unroll
        for (uint32_t w = 0; w < kW; ++w) cnt[w * 256 + t] += base;
      }
      __syncthreads();
#pragma unroll
      for (uint32_t e = 0; e < kItems; ++e) {
        if (e >= items) break;
        if (w0 + e * 32 + lane < m) {
          const uint32_t d = (uint32_t)(k[e] >> shift) & mask;
          buf[mine[d] + (rank[e >> 1] >> (e & 1 ? 16 : 0) & 0xFFFFu)] = k[e];
        }
      }
      __syncthreads();
      if (p + 1 < passes) {
#pragma unroll
        for (uint32_t e = 0; e < kItems; ++e) {
          if (e >= items) break;
          const uint32_t i = w0 + e * 32 + lane;
          if (i < m) k[e] = buf[i];
        }
        __syncthreads();
      }
    }
    for (uint32_t i = t; i < m; i += kMsdThreads) out[o + i] = buf[i];
    __syncthreads();
  }
}

// Step 0: the sample, then count and plan (state->ok: the bins fit); 1: the sort.
// The caller waits for the report between them; a skewed array skips the count.
template <typename K>
void launch_msd_sort(const MsdJob& J, int step, int sms, cudaStream_t s) {
  const uint32_t nb = 1u << J.top;
  if (step == 0) {
    k_msd_probe<K><<<1, 1024, 0, s>>>(J);
    cudaFuncSetAttribute(k_msd_count<K>, cudaFuncAttributeMaxDynamicSharedMemorySize, 4 << kMsdTopMax);
    k_msd_count<K><<<sms, 1024, nb * 4, s>>>(J);
    k_msd_plan<<<1, 1024, 0, s>>>(J);
  } else {
    const uint32_t bins = kMsdCap * sizeof(K) + kMsdThreads / 32 * 256 * 4;
    const uint32_t part = kMsdTile * sizeof(K);  // (and the bins' words: at most 192 KB)
    cudaFuncSetAttribute(k_msd_partition<K>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)(part + (4 << kMsdTopMax)));
    cudaFuncSetAttribute(k_msd_bins<K>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bins);
    int occ = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_msd_bins<K>, kMsdThreads, bins);
    k_msd_partition<K><<<sms, 1024, part + nb * 4, s>>>(J);
    k_msd_bins<K><<<sms * max(1, occ), kMsdThreads, bins, s>>>(J);
  }
}
template void launch_msd_sort<uint32_t>(const MsdJob&, int, int, cudaStream_t);
template void launch_msd_sort<unsigned long long>(const MsdJob&, int, int, cudaStream_t);

}  // namespace wg
