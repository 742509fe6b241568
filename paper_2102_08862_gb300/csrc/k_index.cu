// k_index.cu -- A0 ingest of the sorted clusters in one pass: validation,
// quantisation and the (sector, row) index row_begin[] with the neighbour kernel's
// tile table.
//
// The paper processes a whole ~10 ms time frame at once, held in GPU memory
// (Sec. 1); clusters arrive sorted by row and time from the clusteriser, so every
// (sector, row) begins where the key of a cluster differs from its predecessor's, which
// the validation compares anyway: the pass records those clusters, and its last CTA
// turns them into the tables.
#include "tpc_dev.cuh"
#include "tpc_internal.h"

namespace tpc {

// One block: row_begin from the recorded first clusters (key_first: index + 1, 0 for a
// key without clusters; a key begins where the next one present does), the largest row
// and the first neighbour tile of every row.  Each thread owns a contiguous block of
// keys, read at L2 (ld.cg: other blocks wrote them) kBatch at a time, so that one round
// trip serves a whole frame's 22 keys per thread; block-wide scans join the blocks.
// With unsorted input (an error) the minima keep row_begin monotone and inside [0, n].
// The first key begins at 0 whatever it holds: clusters in front of the first one with a
// valid key (an error too) lie in its row, so that every cluster is in a row and gets its
// links written.
__device__ __forceinline__ void stage_row_index_table(const Args &a) {
  constexpr int kBatch = 24;
  __shared__ int32_t s_min[256];
  __shared__ uint32_t s_warp[8];
  __shared__ int s_max[8];
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  for (int q = tid; q < a.nsect; q += 256) {  // the walk's per-sector track ranges
    a.sec_first[q] = ~0u;
    a.sec_cnt[q] = 0u;
  }
  const int nkeys = a.nkeys, tile = a.nb_tile;
  const int per = (nkeys + 255) / 256, k0 = min(nkeys, tid * per), k1 = min(nkeys, k0 + per);
  const int32_t n = (int32_t)a.n;
  if (tid == 0) a.key_first[0] = 1u;  // (its keys are read by this thread alone)
  // first present cluster of this thread's keys, then of all keys behind them
  int32_t mine = n;
  for (int k = k0; k < k1; k += kBatch) {
    uint32_t v[kBatch];
#pragma unroll
    for (int u = 0; u < kBatch; ++u) v[u] = k + u < k1 ? __ldcg(a.key_first + k + u) : 0u;
#pragma unroll
    for (int u = 0; u < kBatch; ++u)
      if (v[u]) mine = min(mine, (int32_t)v[u] - 1);
  }
  int32_t x = mine;
  for (int o = 1; o < 32; o <<= 1) x = min(x, __shfl_down_sync(0xffffffffu, x, o));  // (past lane 31: its own value)
  if (lane == 0) s_min[w] = x;
  __syncthreads();
  int32_t next = __shfl_down_sync(0xffffffffu, x, 1);
  if (lane == 31) next = n;
  for (int q = w + 1; q < 8; ++q) next = min(next, s_min[q]);
  // row_begin of this thread's keys, from the last one back, and its tiles
  int mx = 0, ntile = 0;
  int32_t run = next;
  for (int ke = k1; ke > k0; ke -= kBatch) {
    uint32_t v[kBatch];
#pragma unroll
    for (int u = 0; u < kBatch; ++u) v[u] = ke - 1 - u >= k0 ? __ldcg(a.key_first + ke - 1 - u) : 0u;
#pragma unroll
    for (int u = 0; u < kBatch; ++u)
      if (ke - 1 - u >= k0) {
        const int32_t begin = v[u] ? min(run, (int32_t)v[u] - 1) : run;
        const int c = run - begin;
        a.row_begin[ke - 1 - u] = begin;
        mx = max(mx, c);
        ntile += (c + tile - 1) / tile;
        run = begin;
      }
  }
  mx = __reduce_max_sync(0xffffffffu, mx);
  if (lane == 0) s_max[w] = mx;
  uint32_t total;
  uint32_t off = block_exclusive_scan<256>((uint32_t)ntile, s_warp, &total);
  int32_t b = run;  // row_begin[k0] (written above by this thread, as are its other keys)
  for (int k = k0; k < k1; ++k) {
    const int32_t e = k + 1 < k1 ? a.row_begin[k + 1] : next;
    a.tile_off[k] = (int32_t)off;
    off += (uint32_t)((e - b + tile - 1) / tile);
    b = e;
  }
  if (tid == 0) {
    a.row_begin[nkeys] = n;
    a.tile_off[nkeys] = (int32_t)total;
    a.ctr[kCtrTiles] = total;
    if (total > a.tile_cap) raise(a.ctr, kErrInternal);
    int m = 0;
    for (int q = 0; q < 8; ++q) m = max(m, s_max[q]);
    a.ctr[kCtrMaxRow] = (uint32_t)m;
    if (m > 65534) raise(a.ctr, kErrRowCap);  // row-local links are 16-bit
  }
}

// A0 validation and quantisation, one pass over the sorted clusters: every
// cluster must have sector < nsect, row < 152, a pad and a time inside the
// validated range, and follow its predecessor in (sector, row, time, pad) order;
// anything else raises kErrInput (the cluster then gets the coordinates of pad
// 0, time 0 so that later stages stay in range).  The pass writes each cluster's
// fixed-point (t_q, y_q) = (rint(64 time), (rint(64 pad) - 32 (npads - 1)) *
// pitch_um) once, so that the neighbour, window and claim kernels read 8
// quantised bytes per cluster instead of converting the same clusters again
// for every tile whose windows hold them.  A thread takes 8 consecutive clusters
// with 16-byte loads (arrays on a 16-byte boundary; otherwise, and for the
// tail, one cluster per thread); the predecessor of its first cluster comes
// from the lane below (a shuffle) or, for lane 0, from global memory.
struct QCheck {
  int kp;
  float tp, pp;
  bool bad;
  __device__ __forceinline__ void step(const Args &a, uint32_t i, int key, float t, float p) {
    if (i > 0 && !(kp < key || (kp == key && (tp < t || (tp == t && pp <= p))))) bad = true;
    if ((i == 0 || kp != key) && key < a.nkeys) a.key_first[key] = i + 1u;  // its (sector, row) begins here
    kp = key;
    tp = t;
    pp = p;
  }
};
__device__ __forceinline__ int2 quant_checked(int sec, int row, float p, float t, int nsect, bool &bad) {
  if (sec >= nsect || row >= kNRows) bad = true;
  if (!pad_ok(p) || !time_ok(t)) {
    bad = true;
    p = 0.0f;
    t = 0.0f;
  }
  return make_int2(q64(t), y_quant(p, min(row, kNRows - 1)));
}

__device__ __forceinline__ void stage_quantize(const Args &a, int vec, uint32_t bid, uint32_t nblk) {
  const uint32_t n = a.n;
  const int lane = threadIdx.x & 31;
  const int nsect = a.nsect;
  QCheck ck;
  ck.bad = false;
  const uint32_t nvec = vec ? n / 256u * 256u : 0u;  // clusters handled 8 per thread (whole warps of 256)
  const uint32_t stride = nblk * blockDim.x;
  for (uint32_t w0 = (bid * blockDim.x + (threadIdx.x & ~31u)) * 8u; w0 < nvec; w0 += stride * 8u) {
    const uint32_t i0 = w0 + (uint32_t)lane * 8u;
    const uint4 sv = *reinterpret_cast<const uint4 *>(a.sector + i0);
    const uint4 rv = *reinterpret_cast<const uint4 *>(a.row + i0);
    const float4 p0 = *reinterpret_cast<const float4 *>(a.pad + i0), p1 = *reinterpret_cast<const float4 *>(a.pad + i0 + 4);
    const float4 t0 = *reinterpret_cast<const float4 *>(a.time + i0), t1 = *reinterpret_cast<const float4 *>(a.time + i0 + 4);
    const uint32_t sw[4] = {sv.x, sv.y, sv.z, sv.w}, rw[4] = {rv.x, rv.y, rv.z, rv.w};
    const float pv[8] = {p0.x, p0.y, p0.z, p0.w, p1.x, p1.y, p1.z, p1.w};
    const float tv[8] = {t0.x, t0.y, t0.z, t0.w, t1.x, t1.y, t1.z, t1.w};
    // the predecessor of the first cluster: the last one of the lane below
    const int klast = (int)(sw[3] >> 16) * kNRows + (int)(rw[3] >> 16);
    ck.kp = __shfl_up_sync(0xffffffffu, klast, 1);
    ck.tp = __shfl_up_sync(0xffffffffu, tv[7], 1);
    ck.pp = __shfl_up_sync(0xffffffffu, pv[7], 1);
    if (lane == 0 && i0 > 0) {
      ck.kp = (int)a.sector[i0 - 1] * kNRows + a.row[i0 - 1];
      ck.tp = a.time[i0 - 1];
      ck.pp = a.pad[i0 - 1];
    }
    int2 q[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      const int sec = (int)((sw[e >> 1] >> (16 * (e & 1))) & 0xffffu), row = (int)((rw[e >> 1] >> (16 * (e & 1))) & 0xffffu);
      const int key = sec * kNRows + row;
      ck.step(a, i0 + e, key, tv[e], pv[e]);
      q[e] = quant_checked(sec, row, pv[e], tv[e], nsect, ck.bad);
    }
    int4 *dst = reinterpret_cast<int4 *>(a.tq + i0);
#pragma unroll
    for (int e = 0; e < 4; ++e) dst[e] = make_int4(q[2 * e].x, q[2 * e].y, q[2 * e + 1].x, q[2 * e + 1].y);
  }
  for (uint32_t i = nvec + bid * blockDim.x + threadIdx.x; i < n; i += stride) {  // the rest
    const int sec = a.sector[i], row = a.row[i];
    const float p = a.pad[i], t = a.time[i];
    if (i > 0) {
      ck.kp = (int)a.sector[i - 1] * kNRows + a.row[i - 1];
      ck.tp = a.time[i - 1];
      ck.pp = a.pad[i - 1];
    }
    ck.step(a, i, sec * kNRows + row, t, p);
    a.tq[i] = quant_checked(sec, row, p, t, nsect, ck.bad);
  }
  if (ck.bad) raise(a.ctr, kErrInput);
}

#ifndef TPC_STAGES_ONLY
// The last CTA to finish builds the tables: with a pass of its own (a binary search per
// key, then the same table) the ingest of a 0.9 M frame took 18 us more.
__global__ void __launch_bounds__(256) k_quantize(Args a, int vec) {
  pdl_begin();
  stage_quantize(a, vec, blockIdx.x, gridDim.x);
  __shared__ bool s_last;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) s_last = atomicAdd(&a.ctr[kCtrIndexDone], 1u) == gridDim.x - 1;
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  stage_row_index_table(a);
}

void launch_quantize(const Args &a, int sms, cudaStream_t st) {
  const bool vec = ((((uintptr_t)a.pad | (uintptr_t)a.time | (uintptr_t)a.sector | (uintptr_t)a.row) & 15) == 0);
  const uint32_t blocks = (a.n / 8 + 255) / 256 + 1;
  const uint32_t cap = (uint32_t)sms * 8u;
  launch_pdl(k_quantize, blocks < cap ? blocks : cap, 256, 0, st, a.n, a, vec ? 1 : 0);
}

// The neighbour kernels' fixed-point conversion, element by element (tests of
// the quantisation contract).
__global__ void __launch_bounds__(256) k_debug_quantize(const float *__restrict__ v, uint32_t n, int32_t *q) {
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) q[i] = q64(v[i]);
}

void launch_debug_quantize(const float *v, uint32_t n, int32_t *q, cudaStream_t st) {
  const uint32_t blocks = (n + 255) / 256;
  k_debug_quantize<<<blocks < 8192u ? blocks : 8192u, 256, 0, st>>>(v, n, q);
}

#endif  // TPC_STAGES_ONLY

}  // namespace tpc
