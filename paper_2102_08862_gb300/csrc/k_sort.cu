// k_sort.cu -- A0 ingest for input that is not sorted: order the clusters by
// (sector, row, time, pad, input index) and keep the permutation, so that every
// later stage sees the same sorted frame as for sorted input and the results map
// back to the caller's order.
//
//   1. k_sort_count: each CTA counts the (sector, row) keys of a contiguous chunk of
//      the input in shared memory (invalid keys go to the last bin) and reserves its
//      part of every bin with one atomic; the last CTA to finish scans the bins;
//   2. k_sort_scatter: each CTA moves its chunk's (time, pad, index) into the bins,
//      positions from shared-memory counters (order inside a bin is arbitrary);
//   3. k_sort_bins: one CTA orders a bin in shared memory.  Its clusters go into
//      about one time bucket each (a counting sort), then each finds its place among
//      its bucket's few by comparing (time, pad, index), which is unique, so the
//      result does not depend on step 2's order.  A bin whose clusters crowd a bucket
//      is sorted by a bitonic network instead.
// A bin holds at most kSegCap clusters (more -> TPC_ERR_CAPACITY; pass sorted
// input then).  The call goes on after that error, so a larger bin is filled too, with
// an order of its own (fill_refused_bin).
//
// What bounds it: memory traffic, 4 B in per cluster for the count, 12 B in and 16 B
// scattered out, 16 B in and 16 B out for the bins (0.06 ms for 6.2 M clusters at the
// measured copy rate); the scatter's 16-byte records each touch a memory sector of
// their own, which takes twice that share.  On a shuffled 2 ms frame (6.2 M clusters,
// one GPU, CUDA events): count 0.020, scatter 0.126, bins 0.089 ms, 0.26 in all with
// the two kernels that find no bin of their size.  An earlier form took 1.52 ms: one
// global atomic per cluster to count and one to scatter (0.19 + 0.13), then a bitonic
// network over every bin, padded to a power of two, one CTA per SM, with the fields
// gathered from the input (1.20).
#include "tpc_dev.cuh"
#include "tpc_internal.h"

namespace tpc {

namespace {
constexpr int kSegCap = 16384;
constexpr int kBins = kNKeys + 1;     // the last one holds invalid keys
constexpr int kBinStride = 5504;
constexpr int kChunkThreads = 1024;
constexpr uint32_t kChunkMin = 8192;  // clusters of a chunk at least
constexpr int kChunksMax = 304;       // two per SM
constexpr int kCrowd = 64;            // a bucket with more clusters is not ranked by comparing all of them

__device__ __forceinline__ uint32_t ord_bits(float f) {
  uint32_t b = __float_as_uint(f);
  if ((b << 1) == 0) b = 0;  // -0.0 and +0.0 compare equal
  return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}
__device__ __forceinline__ float ord_value(uint32_t o) {
  return __uint_as_float((o & 0x80000000u) ? (o & 0x7fffffffu) : ~o);
}
__device__ __forceinline__ uint64_t ord_key(float2 v) { return ((uint64_t)ord_bits(v.x) << 32) | ord_bits(v.y); }

struct SortScratch {
  int32_t *count;    // [kBins] clusters of each bin, then the lists' lengths at [kBins], [kBins + 1]
  int32_t *offset;   // [kBins + 1]
  int32_t *list[2];  // bins too large for the small and for the middle kernel
  int32_t *base;     // [chunks][kBins] where each chunk's part of a bin begins in it
};

__host__ __device__ inline SortScratch carve(void *p) {
  SortScratch s;
  s.count = static_cast<int32_t *>(p);
  s.offset = s.count + kBinStride;
  s.list[0] = s.count + 2 * kBinStride;
  s.list[1] = s.count + 3 * kBinStride;
  s.base = s.count + 4 * kBinStride;
  return s;
}

inline uint32_t sort_chunks(uint32_t n) {
  const uint32_t c = (n + kChunkMin - 1) / kChunkMin;
  return c < 1u ? 1u : c > (uint32_t)kChunksMax ? (uint32_t)kChunksMax : c;
}

__device__ __forceinline__ int bin_of(int sector, int row) {
  return sector >= kNSect || row >= kNRows ? kNKeys : sector * kNRows + row;
}

// Bin classes by size: a CTA of THREADS threads holds up to CAP clusters, EACH of
// them per thread, and BUCKETS counters.
template <int CAP, int BUCKETS>
struct BinSmem {
  float2 v[CAP];  // (time, pad)
  uint32_t idx[CAP];
  int32_t bucket[BUCKETS + 1];
  uint32_t warp[32], warp2[32];
  int crowded;
};
constexpr int kCapSmall = 2048, kCapMid = 8192;
using BinSmall = BinSmem<kCapSmall, 2048>;  // 33 KB: 6 CTAs of 256 threads per SM
using BinMid = BinSmem<kCapMid, 2048>;      // 107 KB: 2 of 1024
using BinLarge = BinSmem<kSegCap, 8192>;    // 225 KB
static_assert(sizeof(BinLarge) <= 232448, "shared memory of one CTA");
}  // namespace

__global__ void __launch_bounds__(kChunkThreads) k_sort_count(Args a, const uint16_t *__restrict__ sector,
                                                              const uint16_t *__restrict__ row, SortScratch s,
                                                              uint32_t chunk) {
  pdl_begin();
  __shared__ int32_t h[kBins];
  __shared__ uint32_t s_warp[kChunkThreads / 32];
  __shared__ bool s_last;
  for (int k = threadIdx.x; k < kBins; k += kChunkThreads) h[k] = 0;
  __syncthreads();
  const uint32_t i0 = blockIdx.x * chunk, i1 = min(a.n, i0 + chunk);
#pragma unroll 4
  for (uint32_t i = i0 + threadIdx.x; i < i1; i += kChunkThreads) atomicAdd(&h[bin_of(sector[i], row[i])], 1);
  __syncthreads();
  if (threadIdx.x == 0 && h[kNKeys] > 0) raise(a.ctr, kErrInput);
  int32_t *base = s.base + (size_t)blockIdx.x * kBinStride;
  for (int k = threadIdx.x; k < kBins; k += kChunkThreads)
    if (h[k] > 0) base[k] = atomicAdd(&s.count[k], h[k]);
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) s_last = atomicAdd(&a.ctr[kCtrSortDone], 1u) == gridDim.x - 1;
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  // the last CTA: the bins' offsets, and the lists of the larger ones
  constexpr int kPer = (kBins + kChunkThreads - 1) / kChunkThreads;
  int32_t c[kPer];
  uint32_t sum = 0, total;
#pragma unroll
  for (int q = 0; q < kPer; ++q) {
    const int k = (int)threadIdx.x * kPer + q;
    c[q] = k < kBins ? __ldcg(s.count + k) : 0;
    sum += (uint32_t)c[q];
  }
  int32_t run = (int32_t)block_exclusive_scan<kChunkThreads>(sum, s_warp, &total);
#pragma unroll
  for (int q = 0; q < kPer; ++q) {
    const int k = (int)threadIdx.x * kPer + q;
    if (k < kBins) {
      s.offset[k] = run;
      if (c[q] > kCapSmall) {
        const int m = c[q] > kCapMid ? 1 : 0;
        s.list[m][atomicAdd(&s.count[kBins + m], 1)] = k;
      }
    }
    run += c[q];
  }
  if (threadIdx.x == 0) s.offset[kBins] = (int32_t)total;
}

__global__ void __launch_bounds__(kChunkThreads) k_sort_scatter(Args a, const uint16_t *__restrict__ sector,
                                                                const uint16_t *__restrict__ row,
                                                                const float *__restrict__ pad,
                                                                const float *__restrict__ time, SortScratch s,
                                                                uint32_t chunk, float4 *__restrict__ rec) {
  pdl_begin();
  __shared__ int32_t cur[kBins];
  const int32_t *base = s.base + (size_t)blockIdx.x * kBinStride;
  for (int k = threadIdx.x; k < kBins; k += kChunkThreads) cur[k] = s.offset[k] + base[k];  // (unused where the chunk has none)
  __syncthreads();
  const uint32_t i0 = blockIdx.x * chunk, i1 = min(a.n, i0 + chunk);
#pragma unroll 4
  for (uint32_t i = i0 + threadIdx.x; i < i1; i += kChunkThreads) {
    const float t = time[i], p = pad[i];
    const int pos = atomicAdd(&cur[bin_of(sector[i], row[i])], 1);
    rec[pos] = make_float4(t, p, __uint_as_float(i), 0.0f);
  }
}

// one bin of cnt clusters, cnt <= CAP
template <int CAP, int BUCKETS, int THREADS>
__device__ __forceinline__ void sort_bin(BinSmem<CAP, BUCKETS> &sm, const float4 *__restrict__ rec, int bin, int b,
                                         int cnt, const uint16_t *__restrict__ sector,
                                         const uint16_t *__restrict__ row, uint16_t *__restrict__ s_sector,
                                         uint16_t *__restrict__ s_row, float *__restrict__ s_pad,
                                         float *__restrict__ s_time, int32_t *__restrict__ perm) {
  constexpr int kEach = CAP / THREADS;
  static_assert(CAP % THREADS == 0 && BUCKETS % THREADS == 0, "whole rounds");
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  float4 v[kEach];
  uint32_t lo = ~0u, hi = 0;
#pragma unroll
  for (int e = 0; e < kEach; ++e) {
    const int q = tid + e * THREADS;
    if (q < cnt) {
      v[e] = __ldcs(rec + b + q);
      const uint32_t o = ord_bits(v[e].x);
      lo = min(lo, o);
      hi = max(hi, o);
    }
  }
  for (int q = tid; q < BUCKETS; q += THREADS) sm.bucket[q] = 0;
  lo = __reduce_min_sync(0xffffffffu, lo);
  hi = __reduce_max_sync(0xffffffffu, hi);
  if (lane == 0) {
    sm.warp[w] = lo;
    sm.warp2[w] = hi;
  }
  if (tid == 0) sm.crowded = 0;
  __syncthreads();
  lo = __reduce_min_sync(0xffffffffu, lane < THREADS / 32 ? sm.warp[lane] : ~0u);
  hi = __reduce_max_sync(0xffffffffu, lane < THREADS / 32 ? sm.warp2[lane] : 0u);
  // buckets of equal width over the bin's time span, monotone in the time; about
  // one cluster each (values that are not finite all go to bucket 0)
  const float t0 = ord_value(lo);
  const int nb = min(BUCKETS, max(cnt, 1));
  const float scale = hi > lo ? (float)nb / (ord_value(hi) - t0) : 0.0f;
  const auto bucket_of = [&](float t) { return min(max(__float2int_rz((t - t0) * scale), 0), nb - 1); };
  int slot[kEach];
#pragma unroll
  for (int e = 0; e < kEach; ++e)
    if (tid + e * THREADS < cnt) {
      const int k = bucket_of(v[e].x);
      const int r = atomicAdd(&sm.bucket[k], 1);
      if (r == kCrowd) sm.crowded = 1;
      slot[e] = (k << 16) | r;  // (r <= 16383)
    }
  __syncthreads();
  if (!sm.crowded) {
    {  // exclusive scan of the bucket counts, BUCKETS / THREADS consecutive ones per thread
      constexpr int kPer = BUCKETS / THREADS;
      int32_t c[kPer];
      uint32_t sum = 0, total;
#pragma unroll
      for (int q = 0; q < kPer; ++q) {
        c[q] = sm.bucket[tid * kPer + q];
        sum += (uint32_t)c[q];
      }
      int32_t run = (int32_t)block_exclusive_scan<THREADS>(sum, sm.warp, &total);
#pragma unroll
      for (int q = 0; q < kPer; ++q) {
        sm.bucket[tid * kPer + q] = run;
        run += c[q];
      }
      if (tid == 0) sm.bucket[BUCKETS] = cnt;
    }
    __syncthreads();
#pragma unroll
    for (int e = 0; e < kEach; ++e)
      if (tid + e * THREADS < cnt) {
        const int q = sm.bucket[slot[e] >> 16] + (slot[e] & 0xffff);
        sm.v[q] = make_float2(v[e].x, v[e].y);
        sm.idx[q] = __float_as_uint(v[e].z);
      }
    __syncthreads();
  } else {  // many equal or unevenly spread times: bitonic network over the whole bin
    int n2 = 1;
    while (n2 < cnt) n2 <<= 1;
#pragma unroll
    for (int e = 0; e < kEach; ++e) {
      const int q = tid + e * THREADS;
      if (q < cnt) {
        sm.v[q] = make_float2(v[e].x, v[e].y);
        sm.idx[q] = __float_as_uint(v[e].z);
      }
    }
    __syncthreads();
    // entries at and past cnt count as larger than any other
    for (int k = 2; k <= n2; k <<= 1) {
      for (int j = k >> 1; j > 0; j >>= 1) {
        // the first step of a merge compares mirrored entries, so that every
        // comparison puts the smaller entry first and the padding never moves
        for (int t = tid; t < n2 / 2; t += THREADS) {
          const int i = j == k >> 1 ? (t / j) * k + (t & (j - 1)) : 2 * t - (t & (j - 1));
          const int l = j == k >> 1 ? (t / j) * k + k - 1 - (t & (j - 1)) : i + j;
          if (l < cnt) {
            const float2 vi = sm.v[i], vl = sm.v[l];
            const uint32_t ii = sm.idx[i], il = sm.idx[l];
            const uint64_t ki = ord_key(vi), kl = ord_key(vl);
            if (ki > kl || (ki == kl && ii > il)) {
              sm.v[i] = vl;
              sm.v[l] = vi;
              sm.idx[i] = il;
              sm.idx[l] = ii;
            }
          }
        }
        __syncthreads();
      }
    }
  }
  // each cluster's place among its bucket's, and the sorted copies
  for (int q = tid; q < cnt; q += THREADS) {
    const float2 x = sm.v[q];
    const uint32_t i = sm.idx[q];
    int p = q;
    if (!sm.crowded) {
      const int k = bucket_of(x.x), o = sm.bucket[k], end = sm.bucket[k + 1];
      if (end - o > 1) {
        const uint64_t key = ord_key(x);
        p = o;
        for (int m = o; m < end; ++m) {
          const uint64_t other = ord_key(sm.v[m]);
          p += other < key || (other == key && sm.idx[m] < i);
        }
      }
    }
    p += b;
    perm[p] = (int32_t)i;
    s_pad[p] = x.y;
    s_time[p] = x.x;
    s_sector[p] = bin < kNKeys ? (uint16_t)(bin / kNRows) : sector[i];
    s_row[p] = bin < kNKeys ? (uint16_t)(bin % kNRows) : row[i];
  }
}

// A bin too large to sort: its clusters in the order of the records, so that the
// permutation stays one (the later stages store through it), at coordinates that pass
// the order check and cost the later stages little whatever the bin's size: times
// spread over the whole validated range, pads beyond any window of the rows next to it.
__device__ __forceinline__ void fill_refused_bin(const float4 *__restrict__ rec, int bin, int b, int cnt,
                                                 const uint16_t *__restrict__ sector,
                                                 const uint16_t *__restrict__ row, uint16_t *__restrict__ s_sector,
                                                 uint16_t *__restrict__ s_row, float *__restrict__ s_pad,
                                                 float *__restrict__ s_time, int32_t *__restrict__ perm) {
  const float pad = bin & 1 ? 1000.0f : -1000.0f;  // (neighbouring rows: 2000 pads of 4 mm or more, wy < 4.2 m)
  const float step = 196608.0f / (float)cnt;
  for (int q = (int)threadIdx.x; q < cnt; q += (int)blockDim.x) {
    const uint32_t i = __float_as_uint(rec[b + q].z);
    perm[b + q] = (int32_t)i;
    s_pad[b + q] = pad;
    s_time[b + q] = fminf(fmaf((float)q, step, -65536.0f), 131072.0f);
    s_sector[b + q] = bin < kNKeys ? (uint16_t)(bin / kNRows) : sector[i];
    s_row[b + q] = bin < kNKeys ? (uint16_t)(bin % kNRows) : row[i];
  }
}

// Every bin of up to kCapSmall clusters has a CTA of the small kernel; the larger
// ones are taken from the lists by the middle and the large kernel's few CTAs.
template <int CAP, int BUCKETS, int THREADS>
__global__ void __launch_bounds__(THREADS) k_sort_bins(Args a, const float4 *__restrict__ rec,
                                                       const uint16_t *__restrict__ sector,
                                                       const uint16_t *__restrict__ row, uint16_t *s_sector,
                                                       uint16_t *s_row, float *s_pad, float *s_time, int32_t *perm,
                                                       SortScratch s) {
  pdl_begin();
  extern __shared__ __align__(16) unsigned char smraw[];
  auto &sm = *reinterpret_cast<BinSmem<CAP, BUCKETS> *>(smraw);
  if constexpr (CAP == kCapSmall) {
    const int bin = blockIdx.x, b = s.offset[bin], cnt = s.offset[bin + 1] - b;
    if (cnt <= 0 || cnt > CAP) return;
    sort_bin<CAP, BUCKETS, THREADS>(sm, rec, bin, b, cnt, sector, row, s_sector, s_row, s_pad, s_time, perm);
  } else {
    constexpr int m = CAP == kCapMid ? 0 : 1;
    const int nlist = s.count[kBins + m];
    for (int e = blockIdx.x; e < nlist; e += gridDim.x) {
      const int bin = s.list[m][e], b = s.offset[bin], cnt = s.offset[bin + 1] - b;
      if (cnt > CAP) {
        if (threadIdx.x == 0) raise(a.ctr, kErrSortCap);
        fill_refused_bin(rec, bin, b, cnt, sector, row, s_sector, s_row, s_pad, s_time, perm);
        continue;
      }
      sort_bin<CAP, BUCKETS, THREADS>(sm, rec, bin, b, cnt, sector, row, s_sector, s_row, s_pad, s_time, perm);
      __syncthreads();  // the shared memory is reused for the next bin
    }
  }
}

size_t sort_scratch_bytes(uint32_t max_n) { return (size_t)(4 + sort_chunks(max_n)) * kBinStride * sizeof(int32_t); }

int launch_sort(const Args &a, const uint16_t *sector, const uint16_t *row, const float *pad, const float *time,
                uint16_t *s_sector, uint16_t *s_row, float *s_pad, float *s_time, int32_t *perm, void *scratch,
                size_t scratch_bytes, void *records, size_t records_bytes, int sms, cudaStream_t st) {
  const auto small = k_sort_bins<kCapSmall, 2048, 256>;
  const auto mid = k_sort_bins<kCapMid, 2048, 1024>;
  const auto large = k_sort_bins<kSegCap, 8192, 1024>;
  static bool configured[64] = {};  // per device: the attribute is a per-device property
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return -1;
  if (dev < 0 || dev >= 64 || !configured[dev]) {
    const auto opt_in = [](auto k, size_t bytes) {
      return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes) == cudaSuccess;
    };
    if (!opt_in(small, sizeof(BinSmall)) || !opt_in(mid, sizeof(BinMid)) || !opt_in(large, sizeof(BinLarge)))
      return -1;
    if (dev >= 0 && dev < 64) configured[dev] = true;
  }
  if (scratch_bytes < sort_scratch_bytes(a.n) || records_bytes < (size_t)a.n * sizeof(float4)) return -1;
  SortScratch s = carve(scratch);
  if (cudaMemsetAsync(s.count, 0, kBinStride * sizeof(int32_t), st) != cudaSuccess) return -1;
  if (a.n == 0) return 1;
  const uint32_t chunks = sort_chunks(a.n), chunk = (a.n + chunks - 1) / chunks;
  float4 *rec = static_cast<float4 *>(records);
  launch_pdl(k_sort_count, chunks, kChunkThreads, 0, st, a.n, a, sector, row, s, chunk);
  launch_pdl(k_sort_scatter, chunks, kChunkThreads, 0, st, a.n, a, sector, row, pad, time, s, chunk, rec);
  launch_pdl(small, (uint32_t)kBins, 256, sizeof(BinSmall), st, a.n, a, rec, sector, row, s_sector, s_row, s_pad, s_time,
             perm, s);
  launch_pdl(mid, 2u * (uint32_t)sms, 1024, sizeof(BinMid), st, a.n, a, rec, sector, row, s_sector, s_row, s_pad, s_time, perm,
             s);
  launch_pdl(large, (uint32_t)sms, 1024, sizeof(BinLarge), st, a.n, a, rec, sector, row, s_sector, s_row, s_pad, s_time, perm,
             s);
  return 6;
}

// ------------------------------------------------------------ inspection
__global__ void k_debug_order(const int32_t *perm, uint32_t n, int32_t *order) {
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
    order[i] = perm ? perm[i] : (int32_t)i;
}

void launch_debug_order(const int32_t *perm, uint32_t n, int32_t *order, cudaStream_t st) {
  k_debug_order<<<1024, 256, 0, st>>>(perm, n, order);
}

}  // namespace tpc
