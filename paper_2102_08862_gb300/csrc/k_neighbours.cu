// k_neighbours.cu -- A1 neighbour finding (cellular-automaton seeding) and the
// edge-row claims of A2.
//
// The paper's tracker seeds in native coordinates with the drift time standing in
// for z (Sec. 1).  For every cluster i of pad row r = 1..150 the kernel picks the
// pair (j in row r-1, k in row r+1) of the same sector whose straight-line midpoint
// residual (y_j + y_k - 2 y_i)^2 + (z_j + z_k - 2 z_i)^2 is smallest, with
// |y_j - y_i|, |y_k - y_i| <= wy and |t_j - t_i|, |t_k - t_i| <= wt, and accepts it
// when the residual is <= cost_max; ties go to the smaller row-local j, then k.
// All of it is integer arithmetic in 1/64 um units, so results are exact.
//
// GB300 design: the ingest pass has validated every cluster and written its
// quantised (t, y) once into an 8-byte array, sorted like the clusters.  Every
// (sector, row) is cut into tiles of nb_tile clusters; the tile-window kernel
// finds, for each tile, the clusters of rows r-1 and r+1 whose time lies within
// wt of the tile's time span (binary searches, all tiles in parallel).  The
// neighbour kernel gives each tile one CTA: the bulk-copy (TMA) engine copies the
// tile and both windows from the quantised array into shared memory, completion
// on an mbarrier; then each warp links 32 consecutive clusters at a time, a cluster
// per lane.  A tile whose windows are larger than the staging buffers is cut into parts;
// windows that are still larger are read from global memory with the same arithmetic.
//
// What bounds it: instruction issue (79 % of the slots) and the integer pipe, which
// takes half of them at half rate; DRAM traffic is 14 of the 16 bytes a cluster
// needs, at a tenth of the bandwidth.  Warp instructions per 32 clusters (16.8 M
// clusters, plain): staging 45, searches 66, scan 150, scoring and output 165.  In an
// earlier form each thread linked a run of two clusters (a search by galloping,
// pointers moved forward, divergent scans that pushed candidates into 16-bit shift
// registers): 700.  Stage times, earlier -> now: 0.71 -> 0.43 ms plain and 0.81 -> 0.48
// ms pruned on the 10 ms frame (32 M clusters), 0.154 -> 0.092 ms plain on 2 ms.
#include "mlp_dev.cuh"
#include "tpc_dev.cuh"
#include "tpc_internal.h"

namespace tpc {

namespace {

constexpr int kMaxCand = 4;  // candidates per neighbour row kept in registers (windows read from global memory)

// Pruned mode: the tile's ambiguous clusters (two pairs or more under the cut) go
// to the tile's own region: for each one its candidates as two masks, and the place
// of its pairs among the region's kPruneRegionRows rows (a shared-memory counter
// reserves both, so no global atomic is taken); the rescoring enumerates the pairs.
// (Written out here as 48-byte rows they cost 160 warp instructions per 32 clusters,
// as masks 70.)  Clusters with more than kPruneMaxPairs such pairs, or that do not
// fit, go to the global list.
constexpr int kPruneMaxPairs = 32;
struct NbQueue {
  uint32_t count;       // records << 16 | rows, also of those that did not fit
  uint32_t end;         // the count before the first that did not fit
  unsigned warps_done;  // the last warp to finish publishes the region's count
};
template <bool kPrune> struct NbExtra {};
template <> struct NbExtra<true> { NbQueue q; };

// first e in [lo, hi) with tq[e].x >= x
__device__ __forceinline__ int tq_lower_bound(const int2 *tq, int lo, int hi, int x) {
  while (lo < hi) {
    const int mid = (int)(((unsigned)lo + (unsigned)hi) >> 1);
    if (tq[mid].x < x) lo = mid + 1; else hi = mid;
  }
  return lo;
}


// Pruned mode: append a cluster with >= 2 pairs under the cost cut to the list
// the classifier rescores: its position, the first entries of its windows and its
// (sector, row), which is its tile's (pruned mode has a CTA per tile).  The lanes that
// append together share one atomic.
__device__ __forceinline__ void amb_push(const Args &a, int i, int j0, int k0) {
  const int4 e = make_int4(i, j0, k0, a.tile_win[2 * blockIdx.x].x);
  const unsigned m = __activemask();
  const int lane = threadIdx.x & 31, leader = __ffs(m) - 1;
  uint32_t base = 0;
  if (lane == leader) base = atomicAdd(&a.ctr[kCtrAmb], (uint32_t)__popc(m));
  base = __shfl_sync(m, base, leader);
  const uint32_t slot = base + (uint32_t)__popc(m & ((1u << lane) - 1u));
  if (slot < a.amb_cap) a.amb[slot] = e; else raise(a.ctr, kErrInternal);
}

// first e in [0, n) with t(e) >= x, searched outwards from `guess` (galloping)
template <class T>
__device__ __forceinline__ int gallop_lower_bound(T t, int n, int x, int guess) {
  int lo, hi;  // answer in [lo, hi]
  guess = min(max(guess, 0), n);
  if (guess < n && t(guess) < x) {
    lo = guess + 1;
    int step = 1;
    hi = lo;
    while (hi < n && t(hi) < x) {
      lo = hi + 1;
      hi = min(n, hi + step);
      step <<= 1;
    }
  } else {
    hi = guess;
    int step = 1;
    lo = hi;
    while (lo > 0 && t(lo - 1) >= x) {
      hi = lo - 1;
      lo = max(0, lo - step);
      step <<= 1;
    }
  }
  while (lo < hi) {
    const int mid = (int)(((unsigned)lo + (unsigned)hi) >> 1);
    if (t(mid) < x) lo = mid + 1; else hi = mid;
  }
  return lo;
}

// Link the contiguous run [li0, li1) of a tile of cnt clusters.  C(i), P(j), N(k)
// return quantised (t, y) of the tile's clusters and of the windows of rows r-1
// (np entries) and r+1 (nn entries).  Links are written as sorted positions
// (window base + window-local index).
template <bool kPrune, class CT, class PT, class NT_>
__device__ __noinline__ void link_run(const Args &a, int li0, int li1, int cnt, CT C, PT P, int np, NT_ N, int nn,
                                         int wy, int wt, int64_t cost_max, int2 *out, int base_p, int base_n,
                                         int base_c) {
  if (li0 >= li1) return;
  auto tp = [&](int j) { return P(j).x; };
  auto tn = [&](int k) { return N(k).x; };
  const int t0 = C(li0).x;
  int jlo = gallop_lower_bound(tp, np, t0 - wt, (int)((long long)li0 * np / cnt));
  int klo = gallop_lower_bound(tn, nn, t0 - wt, (int)((long long)li0 * nn / cnt));
  for (int li = li0; li < li1; ++li) {
    const int2 ci = C(li);
    const int32_t ti = ci.x, yi = ci.y;
    while (jlo < np && tp(jlo) < ti - wt) ++jlo;
    while (klo < nn && tn(klo) < ti - wt) ++klo;
    int nj = 0, nk = 0;
    int cj0 = 0, cj1 = 0, cj2 = 0, cj3 = 0, ck0 = 0, ck1 = 0, ck2 = 0, ck3 = 0;
    for (int j = jlo; j < np; ++j) {
      const int2 e = P(j);
      if (e.x - ti > wt) break;
      if (abs(e.y - yi) > wy) continue;
      if (nj == 0) cj0 = j;
      else if (nj == 1) cj1 = j;
      else if (nj == 2) cj2 = j;
      else if (nj == 3) cj3 = j;
      ++nj;
    }
    if (nj > 0) {
      for (int k = klo; k < nn; ++k) {
        const int2 e = N(k);
        if (e.x - ti > wt) break;
        if (abs(e.y - yi) > wy) continue;
        if (nk == 0) ck0 = k;
        else if (nk == 1) ck1 = k;
        else if (nk == 2) ck2 = k;
        else if (nk == 3) ck3 = k;
        ++nk;
      }
    }
    int64_t best = INT64_MAX;
    int bj = -1, bk = -1, nc = 0;
    if (nj <= kMaxCand && nk <= kMaxCand) {
      const int cj[4] = {cj0, cj1, cj2, cj3}, ck[4] = {ck0, ck1, ck2, ck3};
#pragma unroll
      for (int x = 0; x < kMaxCand; ++x) {
        if (x >= nj) break;
        const int2 ej = P(cj[x]);
        const int32_t dyj = ej.y - yi, dtj = ej.x - ti;
#pragma unroll
        for (int z = 0; z < kMaxCand; ++z) {
          if (z >= nk) break;
          const int2 ek = N(ck[z]);
          const int64_t c = triplet_cost(dyj, ek.y - yi, dtj, ek.x - ti);
          if (kPrune) nc += (c <= cost_max);
          if (c < best) {
            best = c;
            bj = cj[x];
            bk = ck[z];
          }
        }
      }
    } else {  // crowded windows: score every pair in window order
      for (int j = jlo; j < np; ++j) {
        const int2 ej = P(j);
        const int32_t dtj = ej.x - ti;
        if (dtj > wt) break;
        const int32_t dyj = ej.y - yi;
        if (abs(dyj) > wy) continue;
        for (int k = klo; k < nn; ++k) {
          const int2 ek = N(k);
          const int32_t dtk = ek.x - ti;
          if (dtk > wt) break;
          const int32_t dyk = ek.y - yi;
          if (abs(dyk) > wy) continue;
          const int64_t c = triplet_cost(dyj, dyk, dtj, dtk);
          if (kPrune) nc += (c <= cost_max);
          if (c < best) {
            best = c;
            bj = j;
            bk = k;
          }
        }
      }
    }
    out[li] = (bj >= 0 && best <= cost_max) ? make_int2(base_p + bj, base_n + bk) : make_int2(-1, -1);
    if (kPrune && nc >= 2) amb_push(a, base_c + li, base_p + jlo, base_n + klo);
  }
}

// The same linking for staged windows, on shared-memory arrays of (t, y).  Lane l
// of a warp takes cluster l of 32 consecutive ones, so the lanes' windows nearly
// coincide and the warp stays converged: a binary search of fixed depth over
// each window (CAP entries, kNbEnd behind the last real one) finds the first
// entry in time, then both windows are scanned together, one entry of each row
// per step, until both have passed the window's end.  An entry inside the pad
// window too sets a bit; the pairs of set bits are scored afterwards in (j, k)
// order, so that a strict comparison of the cost keeps the smaller j, then the
// smaller k, of equal costs.  |dy| <= wy is one unsigned compare:
// (unsigned)(dy + wy) <= 2 wy.
//
// A cluster whose time window holds more than 31 entries of a row (dense
// instances; a mask has 32 bits) scores each j's pairs directly, over the entries of
// row r+1 with |d2z| <= sqrt(cost_max), found by one more binary search.
//
// Measured beside it: a table of time buckets per row instead of the searches (the
// buckets' slack costs more scan steps than the searches cost: 0.123 against 0.117 ms
// on 2 ms); 64-bit pointers (0.117 against 0.107).  Entries are addressed by their
// 32-bit shared-memory address (as bytes), so that a step costs no 64-bit arithmetic.
__device__ __forceinline__ uint32_t smem_addr(const void *p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ int2 lds_entry(uint32_t addr) {
  int2 v;
  asm volatile("ld.shared.v2.b32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(addr));
  return v;
}
template <int OFF>
__device__ __forceinline__ int lds_time(uint32_t addr) {
  int v;
  asm volatile("ld.shared.b32 %0, [%1 + %2];" : "=r"(v) : "r"(addr), "n"(OFF));
  return v;
}
// address of the first of CAP sorted entries from e with t >= x
template <int S>
__device__ __forceinline__ uint32_t nb_lower_bound(uint32_t e, int x) {
  if (lds_time<8 * (S - 1)>(e) < x) e += 8u * S;
  if constexpr (S > 1) return nb_lower_bound<S / 2>(e, x);
  else return e;
}
// both windows' lower bounds, their steps alternating
template <int S>
__device__ __forceinline__ void nb_lower_bounds(uint32_t &p, uint32_t &n, int x) {
  const int tp = lds_time<8 * (S - 1)>(p), tn = lds_time<8 * (S - 1)>(n);
  if (tp < x) p += 8u * S;
  if (tn < x) n += 8u * S;
  if constexpr (S > 1) nb_lower_bounds<S / 2>(p, n, x);
}

template <bool kPrune, int THREADS, int CAP>
__device__ __forceinline__ void link_tile_smem(const Args &a, int cnt, const int2 *__restrict__ sc,
                                               const int2 *__restrict__ sp, int np, const int2 *__restrict__ sn,
                                               int nn, int wy, int wt, int64_t cost_max, int2 *out, int base_p,
                                               int base_n, int base_c, NbQueue *q, PruneRec *region) {
  const uint32_t wy2 = 2u * (uint32_t)wy;
  const uint64_t cut = (uint64_t)cost_max + 1u;
  const uint32_t ac = smem_addr(sc), ap = smem_addr(sp), an = smem_addr(sn);
  for (int li = threadIdx.x; li < cnt; li += THREADS) {
    const int2 ci = lds_entry(ac + 8u * (uint32_t)li);
    const int32_t ti = ci.x, yi = ci.y, tlo = ti - wt, thi = ti + wt, ylo = yi - wy, yhi = yi + wy;
    uint32_t jlo = ap, klo = an;
    nb_lower_bounds<CAP / 2>(jlo, klo, tlo);
    // Two entries of each row per step.  thi - t, y - ylo and yhi - y are all
    // nonnegative for an entry inside both windows, so the sign bit of their OR is
    // shifted into the row's mask.
    uint32_t mj = 0, mk = 0;
    uint32_t pj = jlo, pk = klo;
    const uint32_t pstop = jlo + 32 * 8;
    int tj, tk;
    do {
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int2 ej = lds_entry(pj + 8 * h), ek = lds_entry(pk + 8 * h);
        tj = thi - ej.x;
        tk = thi - ek.x;
        mj = __funnelshift_l((uint32_t)(tj | (ej.y - ylo) | (yhi - ej.y)), mj, 1);
        mk = __funnelshift_l((uint32_t)(tk | (ek.y - ylo) | (yhi - ek.y)), mk, 1);
      }
      pj += 16;
      pk += 16;
    } while ((tj & tk) >= 0 && pj != pstop);
    const bool wide = (tj & tk) >= 0;
    {  // bit 31 - m set: entry m from jlo (klo) lies in both windows
      const int c = 32 - (int)((pj - jlo) >> 3);
      mj = ~mj << c;
      mk = ~mk << c;
    }
    uint64_t best = cut;
    uint32_t bj = 0, bk = 0;  // its pair, as entries from jlo and klo
    int nc = 0;  // (pruned) pairs under the cut
    // cost of the pair with kinks (d2y, d2z); smaller than the best so far: kept
    auto score = [&](int32_t d2y, int32_t d2z, uint32_t j, uint32_t k) {
      const uint64_t c = (uint64_t)((int64_t)d2y * d2y) + (uint64_t)((int64_t)d2z * d2z);
      if (kPrune) nc += c < cut;
      if (c < best) {
        best = c;
        bj = j;
        bk = k;
      }
    };
    // the pairs of a cluster with a wide window, in (j, k) order
    const int rz = a.cost_rmax / kUmPerBin;  // |d2z| <= sqrt(cost_max)  <=>  |tj + tk - 2 ti| <= rz
    const uint32_t pend = ap + 8u * (uint32_t)np, nend = an + 8u * (uint32_t)nn;
    auto wide_pairs = [&](auto f) {
      for (uint32_t j = jlo; j < pend; j += 8) {
        const int2 ej = lds_entry(j);
        if (ej.x > thi) break;
        if ((uint32_t)(ej.y - ylo) > wy2) continue;
        const int t2 = 2 * ti - ej.x, k1 = min(thi, t2 + rz);
        for (uint32_t k = nb_lower_bound<CAP / 2>(an, max(tlo, t2 - rz)); k < nend; k += 8) {
          const int2 ek = lds_entry(k);
          if (ek.x > k1) break;
          if ((uint32_t)(ek.y - ylo) <= wy2) f((j - jlo) >> 3, (k - klo) >> 3, ej, ek);
        }
      }
    };
    // the first entry of a mask; the mask without it
    auto first = [](uint32_t m) { return (uint32_t)__clz((int)m); };
    auto rest = [](uint32_t m, uint32_t z) { return m & (0x7fffffffu >> z); };
    if (!wide) {
      if (mj != 0 && mk != 0) {
        // the first two candidates of row r+1 stay in registers over the j loop
        const uint32_t z0 = first(mk), mk1 = rest(mk, z0);
        const uint32_t z1 = mk1 ? first(mk1) : z0, mk2 = rest(mk1, z1);
        const int2 e0 = lds_entry(klo + 8u * z0), e1 = lds_entry(klo + 8u * z1);
        const int32_t y0 = e0.y - yi, x0 = (e0.x - ti) * kUmPerBin;
        const int32_t y1 = e1.y - yi, x1 = (e1.x - ti) * kUmPerBin;
        uint32_t m = mj;
        do {
          const uint32_t x = first(m);
          m = rest(m, x);
          const int2 ej = lds_entry(jlo + 8u * x);
          const int32_t dy = ej.y - yi, dz = (ej.x - ti) * kUmPerBin;
          score(dy + y0, dz + x0, x, z0);
          if (!kPrune || mk1) score(dy + y1, dz + x1, x, z1);  // (plain: a repeated pair changes nothing)
          for (uint32_t r = mk2, z; r; r = rest(r, z)) {
            z = first(r);
            const int2 ek = lds_entry(klo + 8u * z);
            score(dy + ek.y - yi, dz + (ek.x - ti) * kUmPerBin, x, z);
          }
        } while (m);
      }
    } else {
      wide_pairs([&](uint32_t j, uint32_t k, int2 ej, int2 ek) {
        score(ej.y + ek.y - 2 * yi, (ej.x + ek.x - 2 * ti) * kUmPerBin, j, k);
      });
    }
    const int j0 = base_p + (int)((jlo - ap) >> 3), k0 = base_n + (int)((klo - an) >> 3);
    out[li] = best < cut ? make_int2(j0 + (int)bj, k0 + (int)bk) : make_int2(-1, -1);
    if (kPrune && nc >= 2) {
      // The tile's region takes the cluster's masks; its pairs get the rows behind
      // those of the clusters before it.  A wide cluster takes a record for each pair,
      // so that the rescoring never scans a window.  The count holds
      // (records, rows), and reservations that fit form a prefix of it; a cluster
      // that does not fit goes to the list.
      uint32_t old = kPruneRegionRows;
      if (nc <= kPruneMaxPairs) old = atomicAdd(&q->count, ((wide ? (uint32_t)nc : 1u) << 16) + (uint32_t)nc);
      int row = (int)(old & 0xffffu);
      if (row + nc <= kPruneRegionRows) {
        int4 *rec = reinterpret_cast<int4 *>(region + (old >> 16));
        int nj = __popc(mj), nk = __popc(mk);
        if (!wide) {
          rec[0] = make_int4(base_c + li, j0, k0, row | (nc << 16));
          rec[1] = make_int4((int)mj, (int)mk, nj | (nk << 16), 0);
        } else {
          nj = nk = 0;
          int2 e;
          for (uint32_t j = jlo; j < pend && (e = lds_entry(j)).x <= thi; j += 8) nj += (uint32_t)(e.y - ylo) <= wy2;
          for (uint32_t k = klo; k < nend && (e = lds_entry(k)).x <= thi; k += 8) nk += (uint32_t)(e.y - ylo) <= wy2;
          const int one = (int)0x80000000u;
          wide_pairs([&](uint32_t j, uint32_t k, int2 ej, int2 ek) {
            if ((uint64_t)triplet_cost(ej.y - yi, ek.y - yi, ej.x - ti, ek.x - ti) >= cut) return;
            rec[0] = make_int4(base_c + li, j0 + (int)j, k0 + (int)k, row++ | (1 << 16));
            rec[1] = make_int4(one, one, nj | (nk << 16), 0);
            rec += 2;
          });
        }
      } else {
        if (nc <= kPruneMaxPairs && row <= kPruneRegionRows) q->end = old;  // the first that does not fit
        amb_push(a, base_c + li, j0, k0);
      }
    }
  }
}

// ------------------------------------------------------- bulk-copy staging
// The tile and both windows are copied from the quantised cluster array into
// shared memory by the bulk-copy (TMA) engine: cp.async.bulk with completion on
// an mbarrier, in 16-byte granules (two 8-byte entries), so a range [lo, hi) is
// copied from lo & ~1 to (hi + 1) & ~1 (the array is padded past n).
__device__ __forceinline__ void mbar_init1(uint64_t *bar) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(bar)) : "memory");
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void mbar_expect(uint64_t *bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ bool mbar_try(uint64_t *bar, uint32_t parity) {
  uint32_t done;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(done)
      : "r"(smem_addr(bar)), "r"(parity)
      : "memory");
  return done != 0;
}
__device__ __forceinline__ void bulk_g2s(void *dst, const void *src, uint32_t bytes, uint64_t *bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                   smem_addr(dst)),
               "l"(src), "r"(bytes), "r"(smem_addr(bar))
               : "memory");
}

// shared memory of one neighbour CTA: the quantised tile and windows, each with
// a granule offset of 0 or 1 entry in front.  A window holds at most CAP - 1
// entries; kNbEnd behind them up to CAP (the searches' depth) and for the
// 32 steps a scan may go on.
constexpr int kNbPad = 32;
constexpr int kNbEnd = 1 << 30;  // later than any cluster, and far from overflow
template <int TILE, int CAP>
struct __align__(16) NbSmem {
  int2 c[TILE + 2];
  int2 p[CAP + 2 + kNbPad];
  int2 n[CAP + 2 + kNbPad];
  uint64_t bar;
};

}  // namespace

// ------------------------------------------------------------ tile windows
// A tile with a range of more than win_cap entries (the neighbour kernel's staging
// buffers) is cut into parts, which become tiles behind the others: halved until every
// part's ranges fit, down to kNbPart clusters.  The neighbour kernel's grid has as many
// places as tiles could be needed for any division into rows, and the parts take those
// that this frame leaves free (one per row is there for a row's last tile, so half of the
// rows' number on average); a tile that finds none stays whole.  1 M clusters of one
// sector at 160 and 200 times the usual density, tile 768, a call: whole tiles, read from
// global memory, 48 and 90 ms; parts 6.7 and 8.3; windows of up to 1279 entries, which an
// earlier form staged, 22 and 33.  Parts linked one after the other by the tile's own CTA
// took 6.7 and 8.7, but the loop cost the usual tiles 1 to 5 %.
constexpr int kNbPart = 128;
// Tile t, clusters [ta, tb) of `key`, whose ranges do not fit: its parts' entries.  Out
// of line, so that the usual tile's search keeps its registers.
static __device__ __noinline__ void split_tile(const Args &a, int win_cap, uint32_t t, int key, int ta, int tb) {
  const int pb = a.row_begin[key - 1], nb = a.row_begin[key + 1], ne = a.row_begin[key + 2], pe = a.row_begin[key];
  auto windows = [&](int c0, int c1) {
    const int t0 = a.tq[c0].x - a.wt, t1 = a.tq[c1 - 1].x + a.wt + 1;
    int4 w;
    w.x = tq_lower_bound(a.tq, pb, pe, t0);
    w.y = tq_lower_bound(a.tq, w.x, pe, t1);
    w.z = tq_lower_bound(a.tq, nb, ne, t0);
    w.w = tq_lower_bound(a.tq, w.z, ne, t1);
    return w;
  };
  int len = tb - ta;
  for (bool ok = false; !ok && len > kNbPart;) {
    len = max(kNbPart, (len + 1) / 2);
    ok = true;
    for (int c = ta; ok && c < tb; c += len) {
      const int4 w = windows(c, min(tb, c + len));
      ok = w.y - w.x <= win_cap && w.w - w.z <= win_cap;
    }
  }
  const uint32_t places = min(a.n / (uint32_t)a.nb_tile + (uint32_t)a.nkeys + 1u, a.tile_cap);
  const uint32_t extra = (uint32_t)((tb - ta - 1) / len);
  uint32_t slot = a.ctr[kCtrTiles], seen;
  for (;; slot = seen) {
    if (slot + extra > places) {
      len = tb - ta;
      break;
    }
    seen = atomicCAS(&a.ctr[kCtrTiles], slot, slot + extra);
    if (seen == slot) break;
  }
  for (int c = ta; c < tb; c += len) {
    const int end = min(tb, c + len);
    const uint32_t e = c == ta ? t : slot++;
    a.tile_win[2 * e] = make_int4(key, c, end, 0);
    a.tile_win[2 * e + 1] = windows(c, end);
  }
}

// One thread per tile: the tile's cluster range and the ranges of rows r-1 and
// r+1 whose t_q lies in [t_first - wt, t_last + wt].
__device__ __forceinline__ void stage_tile_windows(const Args &a, int win_cap, uint32_t bid, uint32_t nblk) {
  const uint32_t ntiles = min((uint32_t)a.tile_off[a.nkeys], a.tile_cap);
  for (uint32_t t = bid * blockDim.x + threadIdx.x; t < ntiles; t += nblk * blockDim.x) {
    // key = last (sector, row) whose first tile is <= t
    int lo = 0, hi = a.nkeys;
    while (hi - lo > 1) {
      const int mid = (lo + hi) >> 1;
      if (a.tile_off[mid] <= (int)t) lo = mid; else hi = mid;
    }
    const int key = lo, r = key % kNRows;
    const int rb = a.row_begin[key], re = a.row_begin[key + 1];
    const int ta = rb + ((int)t - a.tile_off[key]) * a.nb_tile;
    const int tb = min(re, ta + a.nb_tile);
    int4 win = make_int4(0, 0, 0, 0);
    if (r >= 1 && r <= kNRows - 2 && tb > ta) {
      const int t0 = a.tq[ta].x, t1 = a.tq[tb - 1].x;
      const int pb = a.row_begin[key - 1], pe = rb, nb = re, ne = a.row_begin[key + 2];
      // the four lower bounds (first e in [lo, hi) with t_q(e) >= x) advance together
      // and quarter their ranges, so that twelve loads are in flight at once and the
      // dependent round trips are half those of halving; a finished search keeps
      // loading its own position (< n: the array is padded) and ignores it
      int lo[4] = {pb, pb, nb, nb}, hi[4] = {pe, pe, ne, ne};
      const int x[4] = {t0 - a.wt, t1 + a.wt + 1, t0 - a.wt, t1 + a.wt + 1};
      for (;;) {
        bool more = false;
        int m[4][3], tm[4][3];
#pragma unroll
        for (int s = 0; s < 4; ++s) {
          const int len = max(hi[s] - lo[s], 0);  // (probes lo <= m0 <= m1 <= m2 < hi)
          m[s][0] = lo[s] + (len >> 2);
          m[s][1] = lo[s] + (len >> 1);
          m[s][2] = lo[s] + (len >> 1) + (len >> 2);
#pragma unroll
          for (int p = 0; p < 3; ++p) tm[s][p] = a.tq[m[s][p]].x;
        }
#pragma unroll
        for (int s = 0; s < 4; ++s)
          if (lo[s] < hi[s]) {
            if (tm[s][1] < x[s]) {
              if (tm[s][2] < x[s]) lo[s] = m[s][2] + 1;
              else lo[s] = m[s][1] + 1, hi[s] = m[s][2];
            } else {
              if (tm[s][0] < x[s]) lo[s] = m[s][0] + 1, hi[s] = m[s][1];
              else hi[s] = m[s][0];
            }
            more |= lo[s] < hi[s];
          }
        if (!more) break;
      }
      win = make_int4(lo[0], max(lo[1], lo[0]), lo[2], max(lo[3], lo[2]));  // (max: only with unsorted input)
      if (max(win.y - win.x, win.w - win.z) > win_cap && tb - ta > kNbPart) {
        split_tile(a, win_cap, t, key, ta, tb);
        continue;
      }
    }
    a.tile_win[2 * t] = make_int4(key, ta, max(ta, tb), 0);
    a.tile_win[2 * t + 1] = win;
  }
}

// ------------------------------------------------------------ neighbours
// One CTA per tile: one thread issues the bulk copies of the tile and its two
// windows, every thread waits on the mbarrier (bounded) and writes its share of the
// entries behind the windows, then the warps link.  CTAs of 128 threads (4 or 6
// passes of 32 clusters per warp spread the per-warp cost of the staging over more
// clusters than the 2 or 3 of 256 threads: 0.100 -> 0.092 ms on 2 ms, 0.66 -> 0.48
// pruned on 10 ms with the region records), 9 or 10 of them per SM by shared memory,
// which leaves 48 registers a thread; the 1024-cluster tile's 41 KB take 256 threads.
// (A persistent, double-buffered form of an earlier version measured 35-45 % slower:
// its per-tile barrier holds every warp until the tile's slowest one.)
// The work of one tile (t < the number of tiles).  `phase` is the parity of the
// CTA's mbarrier phase to wait for; `init` is set until the CTA has initialised
// its mbarrier (edge-row tiles do not use it).
template <bool kPrune, int TILE, int CAP, int THREADS>
__device__ __forceinline__ void nb_tile(const Args &a, int win_cap, uint32_t t, uint32_t &phase, bool &init) {
  static_assert((CAP & (CAP - 1)) == 0 && THREADS % 32 == 0, "the searches halve CAP");
  __shared__ NbSmem<TILE, CAP> sm;
  __shared__ NbExtra<kPrune> ex;
  const int4 h = a.tile_win[2 * t], w = a.tile_win[2 * t + 1];
  const int key = h.x, ta = h.y, cnt = h.z - h.y;
  const int r = key % kNRows;
  const int tid = threadIdx.x, NT = blockDim.x;
  if (r == 0 || r == kNRows - 1) {  // edge rows: no A1 links (claims come later)
    if (kPrune && tid == 0) a.q_count[t] = 0;
    for (int e = tid; e < cnt; e += NT) a.link[ta + e] = make_int2(-1, -1);
    return;
  }
  const int np = w.y - w.x, nn = w.w - w.z;
  const bool staged = np <= win_cap && nn <= win_cap;
  // granule-aligned copies: tile [ta & ~1, (ta + cnt + 1) & ~1), windows likewise
  const int c0 = ta & ~1, p0 = w.x & ~1, n0 = w.z & ~1;
  NbQueue *q = nullptr;
  if constexpr (kPrune) {
    q = &ex.q;
    if (tid == 0) q->count = q->end = 0, q->warps_done = 0;
  }
  if (init && tid == 0) mbar_init1(&sm.bar);
  __syncthreads();  // the barrier is initialised; the buffers' previous readers are done
  init = false;
  if (tid == 0) {
    // generic-proxy reads of the previous tile are ordered before the copies' writes
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    const uint32_t bc = 8u * (uint32_t)(((ta + cnt + 1) & ~1) - c0);
    const uint32_t bp = staged ? 8u * (uint32_t)(((w.y + 1) & ~1) - p0) : 0u;
    const uint32_t bn = staged ? 8u * (uint32_t)(((w.w + 1) & ~1) - n0) : 0u;
    mbar_expect(&sm.bar, bc + bp + bn);
    if (bc) bulk_g2s(sm.c, a.tq + c0, bc, &sm.bar);
    if (bp) bulk_g2s(sm.p, a.tq + p0, bp, &sm.bar);
    if (bn) bulk_g2s(sm.n, a.tq + n0, bn, &sm.bar);
  }
  // bounded wait for the copies; if any thread gives up, the CTA records a
  // timeout, waits once more (bounded) for copies still in flight and gives the tile
  // no links (the decision is taken by the whole CTA at one barrier).  The limit is
  // not the handle's: a CTA must not end with copies into its shared memory in flight.
  bool ok = true;
  const uint32_t ph = phase;
  phase ^= 1u;
  for (uint32_t it = 0; !mbar_try(&sm.bar, ph); ++it) {  // try_wait suspends the thread for a while itself
    if (it >= kSpinLimit) {
      ok = false;
      break;
    }
  }
  const int2 *sc = sm.c + (ta - c0);
  int2 *s_p = sm.p + (w.x - p0), *s_n = sm.n + (w.z - n0);
  if (ok && staged) {  // behind the windows (the copies are done)
    const int2 end = make_int2(kNbEnd, 0);
    for (int e = np + tid; e < CAP + kNbPad; e += THREADS) s_p[e] = end;
    for (int e = nn + tid; e < CAP + kNbPad; e += THREADS) s_n[e] = end;
  }
  if (__syncthreads_or(!ok)) {
    if (tid == 0) raise(a.ctr, kErrTimeout);
    if (!ok)
      for (uint32_t it = 0; it < kSpinLimit && !mbar_try(&sm.bar, ph); ++it) {
      }
    if (kPrune && tid == 0) a.q_count[t] = 0;
    for (int e = tid; e < cnt; e += NT) a.link[ta + e] = make_int2(-1, -1);
    return;
  }
  if (staged) {
    link_tile_smem<kPrune, THREADS, CAP>(a, cnt, sc, s_p, np, s_n, nn, a.wy, a.wt, a.cost_max, a.link + ta, w.x, w.z,
                                         ta, q, a.q_rec + (size_t)t * kPruneRegionRows);
  } else {
    const int2 *tq = a.tq;
    const int pb = w.x, nb = w.z;
    const int K = (cnt + NT - 1) / NT, li0 = tid * K, li1 = min(cnt, li0 + K);
    link_run<kPrune>(
        a, li0, li1, cnt, [&](int i) { return sc[i]; }, [&](int j) { return tq[pb + j]; }, np,
        [&](int k) { return tq[nb + k]; }, nn, a.wy, a.wt, a.cost_max, a.link + ta, w.x, w.z, ta);
  }
  if constexpr (kPrune) {  // records and rows of this tile's region, published by the last warp to finish
    __syncwarp();
    if ((tid & 31) == 0) {
      __threadfence_block();
      if (atomicAdd(&q->warps_done, 1u) == (unsigned)(THREADS / 32 - 1)) {
        const uint32_t c = atomicAdd(&q->count, 0u);
        a.q_count[t] = (int32_t)((c & 0xffffu) <= kPruneRegionRows ? c : atomicAdd(&q->end, 0u));
      }
    }
  }
}

#ifndef TPC_STAGES_ONLY
template <bool kPrune, int TILE, int CAP, int THREADS>
__global__ void __launch_bounds__(THREADS, THREADS == 128 ? 10 : 5)
    k_neighbours(Args a, int win_cap) {
  pdl_begin();
  const uint32_t t = blockIdx.x;
  if (t >= min(a.ctr[kCtrTiles], a.tile_cap)) return;
  uint32_t phase = 0;
  bool init = true;
  nb_tile<kPrune, TILE, CAP, THREADS>(a, win_cap, t, phase, init);
}
#endif

// all tiles t = bid, bid + nblk, ... in one CTA (the persistent kernel); a tile
// whose copies timed out records the error and the CTA goes on (its results are
// not valid then, and the call reports TPC_ERR_TIMEOUT)
template <bool kPrune, int TILE, int CAP, int THREADS>
__device__ __forceinline__ void stage_neighbours(const Args &a, int win_cap, uint32_t bid, uint32_t nblk) {
  const uint32_t ntiles = min(a.ctr[kCtrTiles], a.tile_cap);
  uint32_t phase = 0;
  bool init = true;
  for (uint32_t t = bid; t < ntiles; t += nblk) {
    nb_tile<kPrune, TILE, CAP, THREADS>(a, win_cap, t, phase, init);
    __syncthreads();  // the staged buffers are free for the next tile
  }
}

// ------------------------------------------------------------- edge-row claims
// A row-0 cluster j takes as up link the row-1 cluster i with down[i] = j of
// smallest (cost_i, i); a row-151 cluster k takes as down link the row-150
// cluster i with up[i] = k of smallest (cost_i, i).  The claimants lie inside
// j's (k's) time window, so the kernel scans that window of the adjacent row and
// recomputes each claimant's triplet cost exactly.
constexpr int kClaimBlocks = 32;  // blocks per edge row
__device__ __forceinline__ void edge_claims_block(const Args &a, int e, int x) {
  const int s = e >> 1;
  const bool top = (e & 1) != 0;
  const int r = top ? kNRows - 1 : 0, rn = top ? kNRows - 2 : 1;
  const int rb = a.row_begin[s * kNRows + r], re = a.row_begin[s * kNRows + r + 1];
  const int nb = a.row_begin[s * kNRows + rn], ne = a.row_begin[s * kNRows + rn + 1];
  for (int j = rb + x * (int)blockDim.x + (int)threadIdx.x; j < re; j += kClaimBlocks * (int)blockDim.x) {
    const int2 qj = a.tq[j];
    const int32_t tj = qj.x, yj = qj.y;
    const int lo = tq_lower_bound(a.tq, nb, ne, tj - a.wt);
    int64_t best = INT64_MAX;
    int bi = -1;
    for (int i = lo; i < ne; ++i) {
      const int2 qi = a.tq[i];
      const int32_t ti = qi.x;
      if (ti - tj > a.wt) break;
      const int2 l = a.link[i];
      if ((top ? l.y : l.x) != j) continue;
      const int o = top ? l.x : l.y;  // far end of i's triplet
      const int2 qo = a.tq[o];
      const int32_t yi = qi.y, yo = qo.y, to = qo.x;
      const int64_t c = triplet_cost(yj - yi, yo - yi, tj - ti, to - ti);
      if (c < best) {
        best = c;
        bi = i;
      }
    }
    if (bi >= 0) {
      if (top) a.link[j].x = bi; else a.link[j].y = bi;
    }
  }
}

__device__ __forceinline__ void stage_edge_claims(const Args &a, uint32_t bid, uint32_t nblk) {
  const uint32_t nb = (uint32_t)kClaimBlocks * 2u * (uint32_t)a.nsect;
  for (uint32_t b = bid; b < nb; b += nblk) edge_claims_block(a, (int)(b / kClaimBlocks), (int)(b % kClaimBlocks));
}

#ifndef TPC_STAGES_ONLY
__global__ void __launch_bounds__(256) k_tile_windows(Args a, int win_cap) {
  pdl_begin();
  stage_tile_windows(a, win_cap, blockIdx.x, gridDim.x);
}
__global__ void __launch_bounds__(256) k_edge_claims(Args a) {
  pdl_begin();
  edge_claims_block(a, (int)blockIdx.x / kClaimBlocks, (int)blockIdx.x % kClaimBlocks);
}

// ------------------------------------------------------------------ launchers
// entries of a staged window: the variant's capacity, or row_cap if that is smaller
static int nb_win_cap(const Args &a, int row_cap) {
  const int cap = (a.nb_tile == 1024 ? 2048 : 1024) - 1;
  return row_cap > 0 && row_cap < cap ? row_cap : cap;
}

void launch_tile_windows(const Args &a, int row_cap, cudaStream_t st) {
  const uint32_t tiles = neighbour_tiles_max(a.n, a.nkeys, a.nb_tile);
  launch_pdl(k_tile_windows, (tiles + 255) / 256, 256, 0, st, a.n, a, nb_win_cap(a, row_cap));
}

template <int TILE, int CAP, int THREADS>
static void launch_nb(const Args &a, int row_cap, cudaStream_t st, bool prune) {
  const uint32_t grid = neighbour_tiles_max(a.n, a.nkeys, TILE);
  launch_pdl(prune ? k_neighbours<true, TILE, CAP, THREADS> : k_neighbours<false, TILE, CAP, THREADS>, grid, THREADS, 0, st,
             a.n, a, nb_win_cap(a, row_cap));
}

void launch_neighbours(const Args &a, int row_cap, int sms, cudaStream_t st, bool prune) {
  (void)sms;
  if (a.nb_tile == 512) launch_nb<512, 1024, 128>(a, row_cap, st, prune);
  else if (a.nb_tile == 1024) launch_nb<1024, 2048, 256>(a, row_cap, st, prune);
  else launch_nb<768, 1024, 128>(a, row_cap, st, prune);
}

void launch_edge_claims(const Args &a, cudaStream_t st) {
  launch_pdl(k_edge_claims, (uint32_t)(kClaimBlocks * 2 * a.nsect), 256, 0, st, a.n, a);
}
#endif  // TPC_STAGES_ONLY

}  // namespace tpc
