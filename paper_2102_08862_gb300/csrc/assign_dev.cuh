// assign_dev.cuh -- the cluster -> track assignment after the chain walk, as a device
// function: run by its own kernel (k_links.cu), behind the fit's blocks (k_fit.cu) and
// inside the persistent kernel.
#pragma once
#include "tpc_dev.cuh"

namespace tpc {

constexpr int kAssignCap = 12288;  // clusters of a row built in shared memory at once (48 KB)
// CTAs that take the (sector, row)s in turn: 4 per SM by shared memory (48 KB each)
inline uint32_t assign_blocks(const Args &a, int sms) {
  const uint32_t cap = (uint32_t)sms * 4u, keys = (uint32_t)a.nkeys;
  return keys < cap ? (keys ? keys : 1u) : cap;
}

// cluster_track of one (sector, row) per CTA step.  The sector's tracks have
// contiguous ids (start order is sector-major); each one that crosses row r has its
// member there at chain step r - first row.  A thread takes 8 consecutive tracks:
// one 16-byte load of their (first row, length) words, then their chain loads,
// issued together.  With a shared-memory buffer (kCap entries) the row is built
// there (-1, then the ids) and written out coalesced, in chunks of kCap clusters
// for longer rows: the global memory sees whole lines only.  Without one (kCap =
// 0, inside the persistent kernel, whose occupancy the buffer would cut) the row
// is filled with -1 in global memory and the ids are stored over it while its
// lines are in L2.
constexpr int kAssignBatch = 3;  // groups of 8 tracks a thread loads per round
template <int kCap>
__device__ __forceinline__ void stage_assign(const Args &a, uint32_t bid, uint32_t nblk, int32_t *buf) {
  const size_t stride = a.track_list_cap;
  const uint32_t nl = listed(a, kCtrTracks, a.track_list_cap);
  for (uint32_t key = bid; key < (uint32_t)a.nkeys; key += nblk) {
    const int rb = a.row_begin[key], re = a.row_begin[key + 1];
    const uint32_t sec = key / kNRows;
    const int r = (int)(key - sec * kNRows);
    const uint32_t t0 = a.sec_first[sec];
    const uint32_t t1 = t0 == ~0u ? t0 : min(nl, t0 + a.sec_cnt[sec]);
    const int chunk = kCap > 0 ? kCap : (re > rb ? re - rb : 1);
    for (int base = rb; base < re; base += chunk) {
      const int end = min(re, base + chunk);
      if (kCap > 0) {
        for (int i = (int)threadIdx.x; i < end - base; i += blockDim.x) buf[i] = -1;
      } else {
        for (int i = base + (int)threadIdx.x; i < end; i += blockDim.x) a.cluster_track[caller_index(a, i)] = -1;
      }
      __syncthreads();  // the fill before the ids, for every thread of the CTA
      if (t0 < t1) {
        // kAssignBatch groups of 8 track ids per thread and round: their (first row,
        // length) words are loaded together, then all their chain loads, so that a
        // round costs two memory latencies whatever its size
        const uint32_t a0 = t0 & ~7u;  // 8-aligned groups of track ids (trk_rl is 16-byte aligned)
        const uint32_t span = 8u * blockDim.x;
        for (uint32_t g0 = a0 + 8u * threadIdx.x; g0 < t1; g0 += kAssignBatch * span) {
          uint4 w[kAssignBatch];
#pragma unroll
          for (int b = 0; b < kAssignBatch; ++b) {
            const uint32_t g = g0 + (uint32_t)b * span;
            w[b] = g < t1 ? *reinterpret_cast<const uint4 *>(a.trk_rl + g) : make_uint4(0u, 0u, 0u, 0u);
          }
          int32_t c[kAssignBatch][8];
#pragma unroll
          for (int b = 0; b < kAssignBatch; ++b) {
            const uint32_t g = g0 + (uint32_t)b * span;
            const uint32_t wv[4] = {w[b].x, w[b].y, w[b].z, w[b].w};
#pragma unroll
            for (int e = 0; e < 8; ++e) {
              const uint32_t t = g + (uint32_t)e;
              const uint32_t rl = (wv[e >> 1] >> (16 * (e & 1))) & 0xffffu;
              const int m = r - (int)(rl & 0xffu), len = (int)(rl >> 8);
              c[b][e] = (t >= t0 && t < t1 && m >= 0 && m < len) ? a.chain[(size_t)m * stride + t] : -1;
            }
          }
#pragma unroll
          for (int b = 0; b < kAssignBatch; ++b)
#pragma unroll
            for (int e = 0; e < 8; ++e) {
              const int32_t ce = c[b][e];
              if (ce >= base && ce < end) {
                const int32_t t = (int32_t)(g0 + (uint32_t)b * span + (uint32_t)e);
                if (kCap > 0) buf[ce - base] = t;
                else a.cluster_track[caller_index(a, ce)] = t;
              }
            }
        }
      }
      __syncthreads();
      if (kCap > 0) {
        for (int i = (int)threadIdx.x; i < end - base; i += blockDim.x) a.cluster_track[caller_index(a, base + i)] = buf[i];
        __syncthreads();  // buf is refilled by the next chunk or key
      }
    }
  }
}

}  // namespace tpc
