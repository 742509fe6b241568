// k_links.cu -- A2 link cleaning (mutual links), A3 start-hit compaction and
// A4 chain membership.
//
// The CA tracker the paper builds on (Sec. 1) keeps a link only when both
// clusters chose each other; the mutual links form disjoint vertical chains, one
// cluster per row.  A chain starts at a cluster with a mutual up link and no
// mutual down link; chains of at least n_min clusters become tracks, numbered in
// the order of their start cluster.
//
// GB300 design.  k_links streams the link array, stores each mutual up link as a
// 16-bit index inside row r+1 (a 32M-cluster frame's links then take 64 MB and stay in
// L2 for the walk) and marks the start hits in a bit mask; k_start_list compacts them
// in cluster order with a block scan plus a decoupled look-back across tiles.  k_walk
// gives each start hit one thread: it
// follows the chain n_min - 1 links to decide whether it is a track, takes its
// track id from a second ordered compaction, then walks the whole chain writing
// the chain's cluster positions as [step][track], so the fit reads them coalesced
// with no pointer chasing, and records each track's first row and length and
// each sector's range of track ids.  k_assign then writes cluster_track one
// (sector, row) at a time: a CTA builds the row in shared memory (-1, then the
// id of every track of the sector that crosses the row, at its member there) and
// writes it out coalesced.  Written from the walk (or the fit), the 4-byte stores
// landed on scattered rows, each a separate L2 transaction that partly filled a
// 32-byte sector the memory read back before writing: 0.21 of the walk's 0.38 ms
// on the 10 ms frame, or 0.12 ms of the fit's time.
#include "assign_dev.cuh"
#include "tpc_dev.cuh"
#include "tpc_internal.h"

namespace tpc {

namespace {
constexpr int kThreads = 256;
constexpr int kLinkTile = kLinkTileN;  // clusters per tile of the hit removal
constexpr uint16_t kNone16 = 0xffff;

}  // namespace

// A2 + A3: mup[i] = up[i] if down[up[i]] = i; start(i) = no mutual down, a mutual up,
// as a bit mask over the clusters.  A step of a CTA takes kLinkStep clusters; thread t
// holds clusters t, t + 256, ... of it, so that a warp's loads, and its gathers of the
// partners' links (the partners of neighbours in time are neighbours too), touch a few
// lines each.  Steps share nothing and need no barrier, so that the dependent loads
// (link, partners' links) of 64 warps overlap.
// What bounds it: the latency of those two loads and the instructions between them (63
// % of the issue slots); 2.7 TB/s of DRAM traffic.  An earlier form gave a thread 8
// consecutive clusters (every lane of a gather met a line of its own) and compacted the
// start hits in the same pass: 0.27 ms on the 10 ms frame, 0.061 on 2 ms.  With
// coalesced gathers alone it took 0.25: the barriers around each tile's look-back were
// what its warps waited for.  Now 0.125 and 0.042 with the start list.
constexpr int kLinkItems = 4;
constexpr int kLinkStep = kThreads * kLinkItems;
__device__ __forceinline__ void stage_links(const Args &a, uint32_t bid, uint32_t nblk) {
  const int32_t *rb = a.row_begin;
  const int nkeys = a.nkeys;
  const uint32_t n = a.n, steps = (n + kLinkStep - 1) / kLinkStep;
  const uint64_t keep = l2_keep_policy();
  const int lane = threadIdx.x & 31;
  bool bad = false;
  for (uint32_t step = bid; step < steps; step += nblk) {
    const int i0 = (int)(step * kLinkStep + threadIdx.x);
    // all loads first: the thread's links, then the partner links they point to
    int2 l[kLinkItems];
#pragma unroll
    for (int q = 0; q < kLinkItems; ++q)
      l[q] = i0 + q * kThreads < (int)n ? __ldcs(a.link + i0 + q * kThreads) : make_int2(-1, -1);
    int32_t pu[kLinkItems], pd[kLinkItems];  // up partner's down link, down partner's up link
#pragma unroll
    for (int q = 0; q < kLinkItems; ++q) {
      pu[q] = l[q].y >= 0 ? a.link[l[q].y].x : -2;
      pd[q] = l[q].x >= 0 ? a.link[l[q].x].y : -2;
    }
    // the key of the step's first cluster, while the loads are under way: the last one
    // with rb[key] <= i (a warp's 32 probes per round)
    int key = 0;
    {
      const int first = (int)(step * kLinkStep);
      for (int span = nkeys; span > 1;) {
        const int w = (span + 31) >> 5, k = key + (lane + 1) * w;
        const int c = __popc(__ballot_sync(0xffffffffu, k < key + span && rb[min(k, nkeys)] <= first));
        key += c * w;
        span = min(w, span - c * w);
      }
    }
#pragma unroll
    for (int q = 0; q < kLinkItems; ++q) {
      const int i = i0 + q * kThreads;
      uint16_t m16 = kNone16;
      const int32_t mup = pu[q] == i ? l[q].y : -1;
      const bool mdn = pd[q] == i;
      if (i < (int)n) {
        // its key, from the previous cluster's, in steps of growing size
        for (int g = 1; key + 1 < nkeys && i >= rb[key + 1];) {
          if (key + g < nkeys && i >= rb[key + g]) {
            key += g;
            g <<= 1;
          } else {
            g = 1;
          }
        }
        if (mup >= 0) {
          const int d = mup - rb[key + 1];
          if (d < 0 || d >= kNone16) bad = true; else m16 = (uint16_t)d;
        }
        st_keep_u16(a.mup16 + i, m16, keep);
      }
      const uint32_t bits = __ballot_sync(0xffffffffu, i < (int)n && mup >= 0 && !mdn);
      if (lane == 0 && i < (int)n) a.start_bits[i >> 5] = bits;
    }
  }
  if (bad) raise(a.ctr, kErrRowCap | kErrRowLost);
}

// The set bits of a mask over the clusters in cluster order (the start hits; the
// followed tracks' first clusters): each thread of a tile takes kListWords words of the
// mask (a tile is kListTileN clusters); positions come from a block scan and a
// decoupled look-back across tiles taken in order from a counter.  The start mask is
// 1/64 of the links' bytes, so the look-back chain is short.
constexpr int kListWords = 4;
constexpr int kListTileN = 32 * kListWords * kThreads;
static_assert(kListTileN >= kLinkTileN, "look-back words");
__device__ __forceinline__ void stage_bit_list(const Args &a, int32_t *__restrict__ out, uint32_t cap,
                                               int tile_counter, int total_counter) {
  __shared__ uint32_t s_tile, s_prefix;
  __shared__ uint32_t s_warp[kThreads / 32];
  const uint32_t n = a.n, words = (n + 31) / 32, n_tiles = (n + kListTileN - 1) / kListTileN;
  for (;;) {
    if (threadIdx.x == 0) s_tile = atomicAdd(&a.ctr[tile_counter], 1u);
    __syncthreads();
    const uint32_t tile = s_tile;
    if (tile >= n_tiles) break;
    const uint32_t w0 = (tile * kThreads + threadIdx.x) * kListWords;
    uint32_t bits[kListWords], count = 0, total;
    if (w0 + kListWords <= words) {
      const uint4 v = *reinterpret_cast<const uint4 *>(a.start_bits + w0);
      bits[0] = v.x, bits[1] = v.y, bits[2] = v.z, bits[3] = v.w;
    } else {
#pragma unroll
      for (int q = 0; q < kListWords; ++q) bits[q] = w0 + q < words ? a.start_bits[w0 + q] : 0u;
    }
#pragma unroll
    for (int q = 0; q < kListWords; ++q) count += (uint32_t)__popc(bits[q]);
    const uint32_t excl = block_exclusive_scan<kThreads>(count, s_warp, &total);
    if (threadIdx.x < 32) {
      const uint32_t pre = lookback_exclusive(a.lb_links, tile, total, a.ctr, a.spin_limit);
      if (threadIdx.x == 0) {
        s_prefix = pre;
        if (tile == n_tiles - 1) a.ctr[total_counter] = pre + total;
      }
    }
    __syncthreads();
    uint32_t pos = s_prefix + excl;
#pragma unroll
    for (int q = 0; q < kListWords; ++q)
      for (uint32_t b = bits[q]; b; b &= b - 1u, ++pos)
        if (pos < cap) out[pos] = (int32_t)(32u * (w0 + q)) + __ffs((int)b) - 1;
    __syncthreads();
  }
}
__device__ __forceinline__ void stage_start_list(const Args &a) {
  stage_bit_list(a, a.starts, a.starts_cap, kCtrTileLinks, kCtrStarts);
}

// A4: one start hit per thread (kWalkChains; walking two or four chains per
// thread interleaved was slower: more threads hide the pointer chase better).
// Chains that reach n_min clusters become tracks (ids in start order); their
// clusters are recorded in the chain buffer; cluster_track comes from k_assign.
template <bool kSmemRb>
__device__ __forceinline__ void stage_walk(const Args &a, uint32_t bid) {
  __shared__ int32_t s_rb[kSmemRb ? kNKeys + 1 : 1];
  __shared__ uint32_t s_tile, s_prefix;
  __shared__ uint32_t s_warp[kThreads / 32];
  const uint32_t ns = min(a.ctr[kCtrStarts], a.starts_cap);
  __shared__ bool s_gone;  // the start list's wait gave up: no chains (thread 0's; in shared memory for its register)
  if (threadIdx.x == 0) {
    s_gone = timed_out(a);
    if (s_gone && bid == 0 && a.n_tracks_out) *a.n_tracks_out = 0;
  }
  const uint32_t n_tiles = (ns + kWalkTileN - 1) / kWalkTileN;
  if (n_tiles == 0) {
    if (bid == 0 && threadIdx.x == 0) {
      a.ctr[kCtrTracks] = 0;
      if (a.n_tracks_out) *a.n_tracks_out = 0;
    }
    return;
  }
  const int32_t *rb = a.row_begin;
  if constexpr (kSmemRb) {
    for (int k = threadIdx.x; k <= a.nkeys; k += kThreads) s_rb[k] = a.row_begin[k];
    rb = s_rb;  // (read behind the first barrier of the loop)
  }
  const int n_min = a.n_min;
  const size_t stride = a.track_list_cap;
  const uint64_t keep = l2_keep_policy();
  // one link step of a chain: (c, key) -> next cluster, or c = -1 at the end
  auto next = [&](int &c, int &key) {
    const uint16_t m = ld_keep_u16(a.mup16 + c, keep);
    if (m == kNone16) {
      c = -1;
    } else {
      c = rb[key + 1] + m;
      ++key;
    }
  };
  constexpr int C = kWalkChains;
  for (;;) {
    if (threadIdx.x == 0) s_tile = s_gone ? ~0u : atomicAdd(&a.ctr[kCtrTileKeep], 1u);
    __syncthreads();
    const uint32_t tile = s_tile;
    if (tile >= n_tiles) break;
    const uint32_t j = tile * kWalkTileN + C * threadIdx.x;
    int2 st[C];
    int c[C], kk[C], len[C];
#pragma unroll
    for (int q = 0; q < C; ++q) {
      st[q] = make_int2(-1, 0);
      if (j + q < ns) {
        const int32_t i = a.starts[j + q];
        st[q] = make_int2(i, key_at<kSmemRb>(a, rb, i));
      }
      c[q] = st[q].x;
      kk[q] = st[q].y;
      len[q] = c[q] >= 0;
    }
    // walk at most n_min - 1 links of every chain, interleaved (C loads in flight)
    for (int s = 1; s < n_min; ++s) {
      bool any = false;
#pragma unroll
      for (int q = 0; q < C; ++q)
        if (c[q] >= 0) {
          next(c[q], kk[q]);
          len[q] += c[q] >= 0;
          any = true;
        }
      if (!any) break;
    }
    bool kept[C];
    uint32_t nkept = 0;
#pragma unroll
    for (int q = 0; q < C; ++q) {
      kept[q] = len[q] >= n_min;
      nkept += kept[q];
    }
    uint32_t total;
    const uint32_t excl = block_exclusive_scan<kThreads>(nkept, s_warp, &total);
    if (threadIdx.x < 32) {
      const uint32_t pre = lookback_exclusive(a.lb_keep, tile, total, a.ctr, a.spin_limit);
      if (threadIdx.x == 0) s_prefix = pre;
    }
    __syncthreads();
    uint32_t id[C];
    bool w[C];
    {
      uint32_t nx = s_prefix + excl;
#pragma unroll
      for (int q = 0; q < C; ++q) {
        id[q] = nx;
        nx += kept[q];
        if (kept[q] && id[q] >= a.track_list_cap) raise(a.ctr, kErrCapacity);
        w[q] = kept[q] && id[q] < a.track_list_cap;
        // second walk: the members of tracks go to the chain buffer (the
        // assignment pass gives every cluster its cluster_track entry)
        c[q] = w[q] ? st[q].x : -1;
        kk[q] = st[q].y;
      }
    }
    for (int m = 0; m < kNRows; ++m) {
      bool any = false;
#pragma unroll
      for (int q = 0; q < C; ++q)
        if (c[q] >= 0) {
          any = true;
          __stcs(a.chain + (size_t)m * stride + id[q], c[q]);
          if (m + 1 < kNRows) next(c[q], kk[q]); else c[q] = -1;
          if (c[q] < 0) a.trk_len[id[q]] = m + 1;
        }
      if (!any) break;
    }
#pragma unroll
    for (int q = 0; q < C; ++q) {
      const int key = st[q].y, sec = w[q] ? key / kNRows : -1;
      if (w[q]) {
        a.trk_key[id[q]] = key;
        a.trk_rl[id[q]] = (uint16_t)((key - sec * kNRows) | (a.trk_len[id[q]] << 8));
      }
      // the sector's id range: one atomic pair per warp and sector (a warp's tracks
      // are consecutive, so the lowest lane of a group holds the group's first id);
      // one pair per track put ~12 k atomics on each of 36 addresses on the 10 ms frame
      const unsigned grp = __match_any_sync(0xffffffffu, sec);
      if (w[q] && (threadIdx.x & 31) == __ffs(grp) - 1) {
        atomicMin(&a.sec_first[sec], id[q]);
        atomicAdd(&a.sec_cnt[sec], (uint32_t)__popc(grp));
      }
    }
    if (tile == n_tiles - 1 && threadIdx.x == 0) {
      const uint32_t nt = s_prefix + total;
      a.ctr[kCtrTracks] = nt;
      if (a.n_tracks_out) *a.n_tracks_out = nt;
      if (a.track_capacity > 0 && nt > a.track_capacity) raise(a.ctr, kErrCapacity);
    }
    __syncthreads();
  }
}

// Up to one tile of the list (32768 clusters) its own launch, or its own barrier of the
// persistent kernel, would cost more than the list itself: 0.186 against 0.175 ms for a
// frame of 7600 clusters.
__host__ __device__ inline bool one_tile_list(uint32_t n) { return n <= (uint32_t)kListTileN; }

// The start list by the last CTA to finish its share of the links
__device__ __forceinline__ void stage_last_list(const Args &a, uint32_t nblk) {
  __shared__ bool s_last;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) s_last = atomicAdd(&a.ctr[kCtrLinksDone], 1u) == nblk - 1;
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  stage_start_list(a);
}

#ifndef TPC_STAGES_ONLY
// with_list: the last CTA to finish makes the start list too
__global__ void __launch_bounds__(kThreads, 8) k_links(Args a, int with_list) {
  pdl_begin();
  stage_links(a, blockIdx.x, gridDim.x);
  if (with_list) stage_last_list(a, gridDim.x);
}
__global__ void __launch_bounds__(kThreads) k_start_list(Args a) {
  pdl_begin();
  stage_start_list(a);
}
__global__ void __launch_bounds__(kThreads) k_first_list(Args a) {
  pdl_begin();
  stage_bit_list(a, a.starts, a.starts_cap, kCtrFirstTile, kCtrFirsts);
}
template <bool kSmemRb>
__global__ void __launch_bounds__(kThreads) k_walk(Args a) {
  stage_walk<kSmemRb>(a, blockIdx.x);
}
__global__ void __launch_bounds__(kThreads) k_assign(Args a) {
  extern __shared__ int32_t assign_buf[];
  stage_assign<kAssignCap>(a, blockIdx.x, gridDim.x, assign_buf);
}

// Hit removal: the clusters attached to a track, in caller order.  k_compact_count
// counts the kept ones of every 2048-cluster tile (4 B per cluster), its last CTA turns
// the counts into offsets; k_compact then copies each tile on its own: a warp holds 256
// consecutive clusters, 32 at a time, so that loads are coalesced and the kept ones of a
// round go to consecutive places.  No tile waits for another.
// The counter of the finished CTAs is zero between calls: the last CTA puts it back, so
// that a small call needs no memset (24 us with one and a full launch gap before the
// copies, 7600 clusters, host and device; 22.9 so; 22.4 in one pass).
// What bounds it: memory, 4 + 16 B per cluster and 16 per kept one.  16.8 M clusters,
// 90 % kept: 0.125 ms (k_compact 0.086, 5.8 TB/s).  An ordered compaction in one pass
// (each tile's fields loaded once a look-back had told its place, staged in shared
// memory) took 0.183 ms.
__global__ void __launch_bounds__(kThreads) k_compact_count(uint32_t n, const int32_t *__restrict__ ct, int vec,
                                                            uint32_t *__restrict__ offset, uint32_t *o_count,
                                                            uint32_t *ctr) {
  pdl_begin();
  __shared__ uint32_t s_warp[kThreads / 32];
  __shared__ bool s_last;
  const uint32_t n_tiles = (n + kLinkTile - 1) / kLinkTile;
  const uint32_t lane = threadIdx.x & 31;
  for (uint32_t tile = blockIdx.x * (kThreads / 32) + (threadIdx.x >> 5); tile < n_tiles;
       tile += gridDim.x * (kThreads / 32)) {  // a tile per warp
    const uint32_t i0 = tile * kLinkTile;
    uint32_t c = 0;
    if (vec && i0 + kLinkTile <= n) {
      const int4 *p = reinterpret_cast<const int4 *>(ct + i0) + lane;
#pragma unroll 8
      for (int q = 0; q < kLinkTile / 128; ++q) {
        const int4 x = p[32 * q];
        c += (x.x >= 0) + (x.y >= 0) + (x.z >= 0) + (x.w >= 0);
      }
    } else {
      for (uint32_t i = i0 + lane; i < min(n, i0 + kLinkTile); i += 32) c += ct[i] >= 0;
    }
    c = __reduce_add_sync(0xffffffffu, c);
    if (lane == 0) offset[tile] = c;
  }
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) s_last = atomicAdd(&ctr[kCtrCompactTile], 1u) == gridDim.x - 1;
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  // exclusive scan: each thread's tiles in turn, kScan read at a time
  constexpr uint32_t kScan = 32;
  const uint32_t per = (n_tiles + kThreads - 1) / kThreads;
  const uint32_t t0 = min(n_tiles, threadIdx.x * per), t1 = min(n_tiles, t0 + per);
  uint32_t sum = 0, total;
  for (uint32_t t = t0; t < t1; t += kScan) {
    uint32_t v[kScan];
#pragma unroll
    for (uint32_t u = 0; u < kScan; ++u) v[u] = t + u < t1 ? __ldcg(offset + t + u) : 0u;
#pragma unroll
    for (uint32_t u = 0; u < kScan; ++u) sum += v[u];
  }
  uint32_t run = block_exclusive_scan<kThreads>(sum, s_warp, &total);
  for (uint32_t t = t0; t < t1; t += kScan) {
    uint32_t v[kScan];
#pragma unroll
    for (uint32_t u = 0; u < kScan; ++u) v[u] = t + u < t1 ? __ldcg(offset + t + u) : 0u;
#pragma unroll
    for (uint32_t u = 0; u < kScan; ++u) {
      if (t + u < t1) offset[t + u] = run;
      run += v[u];
    }
  }
  if (threadIdx.x == 0) {
    *o_count = total;
    ctr[kCtrCompactTile] = 0;  // (all CTAs have counted: the next call finds it as this one did)
  }
}

__global__ void __launch_bounds__(kThreads) k_compact(uint32_t n, const uint16_t *__restrict__ sector,
                                                      const uint16_t *__restrict__ row, const float *__restrict__ pad,
                                                      const float *__restrict__ time, const int32_t *__restrict__ ct,
                                                      const uint32_t *__restrict__ offset,
                                                      uint16_t *__restrict__ o_sector, uint16_t *__restrict__ o_row,
                                                      float *__restrict__ o_pad, float *__restrict__ o_time,
                                                      int32_t *__restrict__ o_track) {
  pdl_begin();
  constexpr int kWarps = kThreads / 32, kRounds = kLinkTile / kThreads;
  __shared__ uint32_t s_cnt[kWarps];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t i0 = blockIdx.x * kLinkTile + (uint32_t)warp * (kRounds * 32u) + (uint32_t)lane;
  int32_t t[kRounds];
  uint16_t sec[kRounds], rw[kRounds];
  float p[kRounds], tm[kRounds];
#pragma unroll
  for (int q = 0; q < kRounds; ++q) {
    const uint32_t i = i0 + 32u * (uint32_t)q;
    t[q] = -1;
    if (i < n) {
      t[q] = __ldcs(ct + i);
      sec[q] = __ldcs(sector + i);
      rw[q] = __ldcs(row + i);
      p[q] = __ldcs(pad + i);
      tm[q] = __ldcs(time + i);
    }
  }
  uint32_t mask[kRounds], mine = 0;
#pragma unroll
  for (int q = 0; q < kRounds; ++q) {
    mask[q] = __ballot_sync(0xffffffffu, t[q] >= 0);
    mine += (uint32_t)__popc(mask[q]);
  }
  if (lane == 0) s_cnt[warp] = mine;
  __syncthreads();
  uint32_t pos = offset[blockIdx.x];
#pragma unroll
  for (int w = 0; w < kWarps; ++w)
    if (w < warp) pos += s_cnt[w];
  const uint32_t below = (1u << lane) - 1u;
#pragma unroll
  for (int q = 0; q < kRounds; ++q) {
    if (t[q] >= 0) {
      const uint32_t o = pos + (uint32_t)__popc(mask[q] & below);
      o_sector[o] = sec[q];
      o_row[o] = rw[q];
      o_pad[o] = p[q];
      o_time[o] = tm[q];
      if (o_track) o_track[o] = t[q];
    }
    pos += (uint32_t)__popc(mask[q]);
  }
}

void launch_compact(const Args &a, const uint16_t *sector, const uint16_t *row, const float *pad, const float *time,
                    const int32_t *ct, uint16_t *o_sector, uint16_t *o_row, float *o_pad, float *o_time,
                    int32_t *o_track, uint32_t *o_count, int sms, cudaStream_t st) {
  const uint32_t tiles = (a.n + kLinkTile - 1) / kLinkTile, cap = (uint32_t)sms * 8u;
  uint32_t *offset = reinterpret_cast<uint32_t *>(a.lb_links);  // (a word per tile; no look-back here)
  const uint32_t blocks = (tiles + kThreads / 32 - 1) / (kThreads / 32);
  k_compact_count<<<blocks < cap ? (blocks ? blocks : 1u) : cap, kThreads, 0, st>>>(
      a.n, ct, ((uintptr_t)ct & 15) == 0 ? 1 : 0, offset, o_count, a.ctr);
  if (tiles > 0)
    launch_pdl(k_compact, tiles, kThreads, 0, st, a.n, a.n, sector, row, pad, time, ct, offset, o_sector, o_row, o_pad,
               o_time, o_track);
}

// inspection: the mutual up link as a sorted position, and the start flag
__global__ void k_debug_links(Args a, int32_t *mup, uint8_t *is_start) {
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < a.n; i += gridDim.x * blockDim.x) {
    const int key = (int)a.sector[i] * kNRows + a.row[i];
    const uint16_t m = a.mup16[i];
    const int32_t up = (m == kNone16 || key + 1 > a.nkeys) ? -1 : a.row_begin[key + 1] + m;
    if (mup) mup[i] = up;
    if (is_start) {
      const int dn = a.link[i].x;
      const bool mdn = dn >= 0 && a.link[dn].y == (int32_t)i;
      is_start[i] = (uint8_t)(!mdn && up >= 0);
    }
  }
}

bool links_with_list(uint32_t n) { return one_tile_list(n); }

void launch_links(const Args &a, int sms, cudaStream_t st) {
  const uint32_t steps = (a.n + kLinkStep - 1) / kLinkStep, cap = (uint32_t)sms * 8u;
  const bool with_list = links_with_list(a.n);
  launch_pdl(k_links, steps < cap ? (steps ? steps : 1u) : cap, kThreads, 0, st, a.n, a, with_list ? 1 : 0);
  if (with_list) return;
  const uint32_t tiles = (a.n + kListTileN - 1) / kListTileN;
  launch_pdl(k_start_list, tiles < cap ? tiles : cap, kThreads, 0, st, a.n, a);
}

void launch_first_list(const Args &a, int sms, cudaStream_t st) {
  const uint32_t tiles = (a.n + kListTileN - 1) / kListTileN, cap = (uint32_t)sms * 8u;
  k_first_list<<<tiles < cap ? (tiles ? tiles : 1u) : cap, kThreads, 0, st>>>(a);
}

void launch_walk(const Args &a, int sms, cudaStream_t st) {
  if (a.nkeys <= kNKeys) k_walk<true><<<sms * 8, kThreads, 0, st>>>(a);
  else k_walk<false><<<sms * 8, kThreads, 0, st>>>(a);
}

void launch_assign(const Args &a, int sms, cudaStream_t st) {
  k_assign<<<assign_blocks(a, sms), kThreads, kAssignCap * 4, st>>>(a);
}

int assign_prepare() {
  return cudaFuncSetAttribute(k_assign, cudaFuncAttributeMaxDynamicSharedMemorySize, kAssignCap * 4) == cudaSuccess &&
                 fit_assign_prepare() == 0
             ? 0
             : -1;
}

// Failure path of the bounded waits: tile 1 of a look-back whose tile 0 never
// publishes (one warp).  The wait gives up after spin_limit polls, records
// kErrTimeout and finishes with a zero prefix.
__global__ void k_debug_wait(uint64_t *lb, uint32_t *ctr, uint32_t spin_limit) {
  const uint32_t pre = lookback_exclusive(lb, 1u, 1u, ctr, spin_limit);
  if (threadIdx.x == 0) ctr[kCtrStarts] = pre;
}

void launch_debug_wait(uint64_t *lb, uint32_t *ctr, uint32_t spin_limit, cudaStream_t st) {
  k_debug_wait<<<1, 32, 0, st>>>(lb, ctr, spin_limit);
}

void launch_debug_links(const Args &a, int32_t *mup, uint8_t *is_start, cudaStream_t st) {
  k_debug_links<<<1024, 256, 0, st>>>(a, mup, is_start);
}

#endif  // TPC_STAGES_ONLY

}  // namespace tpc
