// Parts of the shared-scan kernel (scan_tc.cu): the order in which a CTA takes its row blocks,
// and the streaming select behind the scan (Eq. 6 / Eq. 7) -- survivor queues between the warps
// that produce scores and one append warp per row, the row histogram that keeps the running
// threshold, the row's candidate segment, and the final exact selection, which finisher warps
// take one block behind the scan (a row has two segments, used by alternate blocks).
#pragma once
#include "kernels.h"
#include "ptx.cuh"
#include "segselect.cuh"

namespace pivot {
namespace scan {

constexpr int TILE_KEYS = 128;
constexpr int KS_SLOTS = 8;       // key-scale ring: deeper than (key stages + accumulator buffers)

// Block sequence of one CTA: blocks sorted longest-first are dealt in snake order.
struct BlockIter {
  int n_blocks, G, cta, round;
  __device__ BlockIter(int nb, int g, int c) : n_blocks(nb), G(g), cta(c), round(0) {}
  __device__ int next() {   // block index, or -1
    const int pos = (round & 1) ? (G - 1 - cta) : cta;
    const long long d = (long long)round * G + pos;
    ++round;
    if (d >= n_blocks) return -1;
    return n_blocks - 1 - (int)d;
  }
};

// What the roles of a CTA need to know about one of its row blocks.  The thread that loads the keys, several tiles ahead
// of everybody else, looks it up and leaves it in a small ring in shared memory: a block's descriptors are chains of
// global loads, and looked up by every role at the start of its block they left the tensor core idle for some three
// tiles' time, a seventh of a block of a dozen tiles.  (The producer's whole warp fetching the gates as well, a block
// ahead, starved the key ring: packed batch +4 %, dense 16K +14 %.)
constexpr int kBlockSlots = 4;
template <int NROWS>
struct BlockInfo {
  int b;                      // block index, -1: no more blocks
  int ntiles, k_row0;         // key tiles (of its longest live row), first key-tensor row of its sequence
  int n_vis[NROWS], K[NROWS]; // 0: no such row, or nothing to select
  const float* w[NROWS];      // gates and their scales (K > 0)
  const float* qscale[NROWS];
};
template <int NROWS>
struct BlockRing {
  BlockInfo<NROWS> info[kBlockSlots];
  uint64_t full[kBlockSlots], empty[kBlockSlots];
};

// The consumers' side: block number n's info, nullptr at the end (or if the wait ran out).  Every consumer warp
// arrives on empty[slot] once it needs it no more.  next_block: one thread; next_block_warp: a whole warp, whose
// lanes agree on the outcome.
template <int NROWS>
__device__ __forceinline__ const BlockInfo<NROWS>* next_block(BlockRing<NROWS>& ring, uint32_t n, volatile int* abort_flag) {
  const int slot = n % kBlockSlots;
  const bool ok = ptx::mbar_wait(&ring.full[slot], (n / kBlockSlots) & 1, abort_flag, 32);
  return ok && ring.info[slot].b >= 0 ? &ring.info[slot] : nullptr;
}
template <int NROWS>
__device__ __forceinline__ const BlockInfo<NROWS>* next_block_warp(BlockRing<NROWS>& ring, uint32_t n, volatile int* abort_flag) {
  const BlockInfo<NROWS>* const f = next_block(ring, n, abort_flag);
  return __all_sync(0xffffffffu, f != nullptr) ? f : nullptr;
}

// One of a block's effective gates (fl32(w * qscale)), as the two loads that it takes: a row that selects nothing has
// gates of 0, proxies no scale.
struct GateLoad { float w, qscale; };
template <int NROWS>
__device__ __forceinline__ GateLoad load_gate(const BlockInfo<NROWS>& f, int r, int j) {
  GateLoad g{0.f, 1.f};
  if (f.K[r] > 0) {
    g.w = f.w[r][j];
    if (f.qscale[r]) g.qscale = f.qscale[r][j];
  }
  return g;
}

// Shared-memory state of the streaming select of a block of NROWS rows.
template <int NROWS, int QD>
struct SelectCtrl {
  alignas(16) uint32_t rhist[NROWS][kSelBins];      // per row: histogram of every score appended so far
  uint64_t sc_full[QD], sc_empty[QD];   // survivor queues: score warps -> append warps
  alignas(16) unsigned long long q[QD][NROWS][4][32];   // [tile % QD][row][lane quarter]: packed entries
  alignas(16) uint32_t qn[QD][NROWS][4];                // their counts
  // published append threshold of each row, (block sequence number << 32) | key: only grows
  // within a block; a reader that is already in the next block sees a stale tag and takes 0
  volatile unsigned long long thr[NROWS];
  // End of a block: what the row's finisher needs (the append warp moves on to the next block
  // and the row's other segment at once).  Two slots, used by alternate blocks like the segments.
  struct FinRow {
    int b;                              // the block, -1: no more
    int cnt;                            // entries held in the row's segment
    int base;                           // the row histogram's anchor
    int bsel;                           // boundary bin of the exact histogram, -1 = everything is wanted
    uint32_t need_b, pop;               // entries wanted from that bin, and its population
  } fin[NROWS][2];
  uint64_t fin_full[NROWS][2], fin_done[NROWS][2];   // append warp -> finisher -> append warp
  int abort_code;                       // device status to report besides a timed-out wait
  SegSelSmem sel[NROWS];                // the row's append warp (segment overflow) or its finisher
};

// The threshold the score warps of block sequence number `seq` compare row r's scores with.
template <int NROWS, int QD>
__device__ __forceinline__ uint32_t row_threshold(const SelectCtrl<NROWS, QD>& s, int r, uint32_t seq) {
  const unsigned long long t = s.thr[r];
  return (uint32_t)(t >> 32) == seq ? (uint32_t)t : 0u;
}

// Row r's segment for the block with sequence number seq.
template <int NROWS>
__device__ __forceinline__ entry_t* row_segment(const ScanScratch& sc, int r, uint32_t seq) {
  return sc.cand64 + (((size_t)blockIdx.x * NROWS + r) * 2 + (seq & 1u)) * sc.cap;
}

// A score warp leaves the survivors of its 32 keys of rows r0 .. r0 + NR - 1 in the tile's queue: each row's
// compacted by one vote, the counts beside them (lane i stores row r0 + i's).  `take` must already include the
// causal cut and the threshold test.  No branches.
template <int NR, int NROWS, int QD>
__device__ __forceinline__ void push_survivors(SelectCtrl<NROWS, QD>& s, int qb, int r0, int lq, int lane, const bool (&take)[NR],
                                               const uint32_t (&key)[NR], int s_key) {
  const uint32_t lt = (1u << lane) - 1u;
  const uint32_t q = ptx::smem_u32(&s.q[qb][r0][lq][0]);
  uint32_t n = 0;
#pragma unroll
  for (int i = 0; i < NR; ++i) {
    const uint32_t m = __ballot_sync(0xffffffffu, take[i]);
    ptx::st_shared_if(q + i * (4 * 32 * 8) + __popc(m & lt) * 8, (uint64_t)make_entry(key[i], s_key), take[i]);
    n = lane == i ? (uint32_t)__popc(m) : n;
  }
  ptx::st_shared_if(ptx::smem_u32(&s.qn[qb][r0][lq]) + (lane < NR ? lane : 0) * 16, n, lane < NR);
}

// Score key -> histogram bin: 256 bins per octave (8 mantissa bits), 2048 bins anchored two
// octaves above the row's first-tile maximum; keys outside land in the end bins.
__device__ __forceinline__ int select_bin(uint32_t key, int base) {
  const int b = (int)(key >> 15) - base;
  return b < 0 ? 0 : (b > kSelBins - 1 ? kSelBins - 1 : b);
}

// Smallest key of a bin: the end bins take everything beyond them (key 0 stands for "no entry").
// (bins the boundary asks for lie above 0 and at most at kSelBins, so the top bin's end is the largest key)
__device__ __forceinline__ uint32_t select_bin_lo(int bin, int base) {
  if (bin <= 0) return 1u;
  return bin >= kSelBins || bin + base > 0x1ffff ? 0xffffffffu : (uint32_t)(bin + base) << 15;
}

// The append warps' rare steps, out of their loop: a row's segment without what lies at or below a threshold (returns
// what is left), and its K best alone (returns the key of the last; more than K entries).
static __device__ __noinline__ int drop_below(entry_t* seg, int cnt, int lane, uint32_t thr) {
  return seg_filter_inplace(seg, cnt, lane, [thr](entry_t x) { return entry_key(x) > thr; });
}
static __device__ __noinline__ uint32_t compact_to_best(const Team& tm, SegSelSmem& sel, entry_t* seg, int cnt, int K) {
  entry_t cut;
  (void)seg_compact<false>(tm, sel, Seg{seg, cnt}, K, &cut);
  return entry_key(cut);
}

// The append warp of row r (one warp, all blocks of this CTA): counts the survivors of every tile
// in the row histogram, moves them to the row's segment in the L2-resident scratch and keeps the
// row's threshold fresh -- alone, without barriers.  At the end of a block it reads the boundary
// bin off the (then exact) histogram, hands the segment to the row's finisher and goes on with
// the next block in the row's other segment.
template <int NROWS, int QD>
__device__ __noinline__ void append_role(SelectCtrl<NROWS, QD>& s, int r, int lane, const Team& tm,
                                            BlockRing<NROWS>& ring, const ScanScratch& sc, volatile int* abort_flag) {
  SegSelSmem& sel = s.sel[r];
  const int CAP = sc.cap;                        // entries of this row's candidate segment
  uint32_t* const rhist = s.rhist[r];
  // Lower bound on the K-th best score seen so far, read off the row histogram: the largest
  // bin edge with at least K scores at or above it.  Returned as a key threshold t such that
  // only keys > t can still belong to the top K.
  auto hist_threshold = [&](int K, int base) -> uint32_t {
    uint32_t b, need_in, pop;
    if (!warp_hist_boundary(rhist, (uint32_t)K, lane, &b, &need_in, &pop)) return 0u;
    return b > 0 ? (((uint32_t)((int)b + base)) << 15) - 1u : 0u;
  };
  // The threshold is refreshed every CHK tiles, more often while it still moves fast (the K-th best of t tiles lets
  // K / (128 t) of the next one through).  A tile adds at most TILE_KEYS entries, so a segment that has room for the
  // tiles until the next refresh never overflows.
  const int CHK = CAP / (2 * TILE_KEYS) < kThresholdRefreshTiles ? (CAP / (2 * TILE_KEYS) > 0 ? CAP / (2 * TILE_KEYS) : 1) : kThresholdRefreshTiles;
  const int headroom = TILE_KEYS * CHK;
  uint32_t it = 0, seq = 0;
  while (const BlockInfo<NROWS>* const info = next_block_warp(ring, seq, abort_flag)) {
    const int b = info->b, ntiles = info->ntiles, K = info->K[r];
    __syncwarp();
    if (lane == 0) ptx::mbar_arrive(&ring.empty[seq % kBlockSlots]);
    int cnt = 0, base = 0;
    uint32_t thr = 0;
#pragma unroll 4
    for (int i = lane; i < kSelBins / 4; i += 32) reinterpret_cast<uint4*>(rhist)[i] = make_uint4(0, 0, 0, 0);
    if (lane == 0) s.thr[r] = (unsigned long long)seq << 32;
    // this block's segment was the block's before last: its finisher must be through with it
    const int fb = seq & 1;
    (void)ptx::mbar_wait(&s.fin_done[r][fb], ((seq >> 1) & 1) ^ 1, abort_flag, 64);
    entry_t* const seg = row_segment<NROWS>(sc, r, seq);
    bool sel_mine = seq == 0;                    // the finisher of the previous block may still use `sel`
    __syncwarp();
    // tiles until the next refresh; the first when the segment holds a quarter more than K
    int due = (K + K / 4 + TILE_KEYS - 1) / TILE_KEYS;
    due = due < kRefreshMin ? kRefreshMin : due;
    due = due < CAP / (2 * TILE_KEYS) ? due : CHK;
    for (int t = 0; t < ntiles; ++t, ++it) {
      if (due-- == 0) {
        int next = t / 2 < kRefreshMin ? kRefreshMin : t / 2;
        next = next < CHK ? next : CHK;
        const int left = ntiles - t;
        if (left <= kRefreshLast && cnt + TILE_KEYS * left <= CAP) {
          next = left;                             // too few tiles left to gain by it
        } else if (K > 0) {
          const uint32_t th = hist_threshold(K, base);
          thr = th > thr ? th : thr;
          if (cnt + TILE_KEYS * (next < kLeastRoomTiles ? next : kLeastRoomTiles) > CAP) {
            // Nearly full: drop what fell below the threshold; if that is not enough (ties, adversarial
            // order) compact exactly to the K best.  What goes lies below every bin the final boundary can
            // be in, so the histogram stays exact for what the selection looks at.
            const uint32_t tcur = thr;
            cnt = drop_below(seg, cnt, lane, tcur);
            if (cnt + headroom > CAP && cnt > K) {
              if (!sel_mine) {                     // (rare path: waiting here costs nothing that matters)
                (void)ptx::mbar_wait(&s.fin_done[r][fb ^ 1], ((seq - 1) >> 1) & 1, abort_flag, 64);
                sel_mine = true;
              }
              const uint32_t cut = compact_to_best(tm, sel, seg, cnt, K);
              cnt = K;
              thr = cut > thr ? cut : thr;
            }
          }
          const int room = (CAP - cnt) / TILE_KEYS;
          next = next < room ? next : room;
          if (lane == 0) s.thr[r] = ((unsigned long long)seq << 32) | thr;
        }
        due = next - 1;
      }
      const int sb = it % QD;
      (void)ptx::mbar_wait(&s.sc_full[sb], (it / QD) & 1, abort_flag);
      const uint4 n4 = *reinterpret_cast<const uint4*>(&s.qn[sb][r][0]);
      const uint32_t total = n4.x + n4.y + n4.z + n4.w;
      // Every entry that reaches the segment is counted: the ones the score warps dropped were
      // at or below a valid threshold and can never reach a bin edge the threshold could still
      // move to, so the counts that matter stay exact.
      auto take = [&](entry_t x, bool on, int p) {
        if (on && p < CAP) {                     // (CHK leaves room for every tile until the next check)
          atomicAdd(&rhist[select_bin(entry_key(x), base)], 1u);
          seg[p] = x;
        }
      };
      if (t > 0 && total <= 32) {
        // All of the tile's survivors in one step, a lane each: once the threshold has settled a tile
        // leaves some twenty, and the step's cost is its instruction count, not the entries.
        const uint32_t c1 = n4.x, c2 = c1 + n4.y, c3 = c2 + n4.z;
        const uint32_t l = (uint32_t)lane;
        const uint32_t j = (l >= c1 ? 1u : 0u) + (l >= c2 ? 1u : 0u) + (l >= c3 ? 1u : 0u);
        const uint32_t first = l >= c3 ? c3 : l >= c2 ? c2 : l >= c1 ? c1 : 0u;
        const bool on = l < total;
        const entry_t x = on ? s.q[sb][r][j][l - first] : kPadEntry;
        __syncwarp();
        if (lane == 0) ptx::mbar_arrive(&s.sc_empty[sb]);
        if (K <= 0) continue;                    // a dead row still takes part in the handshake
        take(x, on, cnt + lane);
      } else {
        const uint32_t nq[4] = {n4.x, n4.y, n4.z, n4.w};
        entry_t e[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) e[j] = (uint32_t)lane < nq[j] ? s.q[sb][r][j][lane] : kPadEntry;
        __syncwarp();
        if (lane == 0) ptx::mbar_arrive(&s.sc_empty[sb]);
        if (K <= 0) continue;
        if (t == 0) {          // anchor the histogram range on the first tile's maximum
          uint32_t mx = 0;
#pragma unroll
          for (int j = 0; j < 4; ++j) mx = entry_key(e[j]) > mx ? entry_key(e[j]) : mx;
          mx = __reduce_max_sync(0xffffffffu, mx);
          const int top = (int)(mx >> 15) + 512 - (kSelBins - 1);
          base = top > 0 ? top : 0;
        }
        int p = cnt + lane;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          take(e[j], (uint32_t)lane < nq[j], p);
          p += (int)nq[j];
        }
      }
      cnt += (int)total;
      if (cnt > CAP) { cnt = CAP; s.abort_code = DEV_CAND_OVERFLOW; }
    }
    // ---- end of the block: the histogram is exact for everything the segment still holds; read
    //      the boundary bin off it and hand the row to its finisher
    uint32_t bb = 0, need_b = 0, pop = 0;
    const bool found = K > 0 && warp_hist_boundary(rhist, (uint32_t)K, lane, &bb, &need_b, &pop);
    if (lane == 0) {
      typename SelectCtrl<NROWS, QD>::FinRow& f = s.fin[r][fb];
      f.b = b; f.cnt = cnt; f.base = base; f.bsel = found ? (int)bb : -1; f.need_b = need_b; f.pop = pop;
    }
    __threadfence_block();
    __syncwarp();
    if (lane == 0) ptx::mbar_arrive(&s.fin_full[r][fb]);
    ++seq;
  }
  // no more blocks (or a wait ran out)
  (void)ptx::mbar_wait(&s.fin_done[r][seq & 1], ((seq >> 1) & 1) ^ 1, abort_flag, 64);
  if (lane == 0) {
    s.fin[r][seq & 1].b = -1;
    ptx::mbar_arrive(&s.fin_full[r][seq & 1]);
  }
}

// A finisher warp: the final exact selection of rows r0 .. r0 + nr - 1 of every block of this CTA,
// one block behind the scan.  The append warp has counted every entry the segment holds, so its
// boundary bin is exact and one sweep over the segment suffices (a boundary bin too crowded to
// rank takes the general way).  Pads the row with -1 and copies it to the other members of a
// Reuse group.
template <int NROWS, int QD>
__device__ __noinline__ void finisher_role(SelectCtrl<NROWS, QD>& s, int r0, int nr, int lane,
                                              const RowDesc* rows, int n_rows, const ScanScratch& sc,
                                              volatile int* abort_flag) {
  for (uint32_t seq = 0;; ++seq) {
    const int fb = seq & 1;
    for (int r = r0; r < r0 + nr; ++r) {
      if (!__all_sync(0xffffffffu, ptx::mbar_wait(&s.fin_full[r][fb], (seq >> 1) & 1, abort_flag, 64))) return;
      const int b = s.fin[r][fb].b;
      if (b < 0) return;
      const int ri = b * NROWS + r;
      const typename SelectCtrl<NROWS, QD>::FinRow f = s.fin[r][fb];
      const StagedSeg staged(s.sel[r], row_segment<NROWS>(sc, r, seq), f.cnt);
      staged.start(lane);
      const RowDesc rd = rows[ri < n_rows ? ri : n_rows - 1];
      const int K = ri < n_rows ? rd.K : 0;
      if (K > 0) {
        const int rbase = f.base;
        auto bin_lo = [rbase](int bin) { return select_bin_lo(bin, rbase); };
        const int n_valid = warp_seg_topk_binned(s.sel[r], staged, bin_lo, f.bsel, f.need_b, f.pop, rd.out, rd.out_score, K,
                                                 lane);
        for (int i = n_valid + lane; i < K; i += 32) {
          rd.out[i] = -1;
          if (rd.out_score) rd.out_score[i] = -INFINITY;
        }
        __syncwarp();
        if (rd.out_rows > 1) {
          constexpr int U = 16;               // one load for all copies, sixteen in flight
          for (int i0 = 0; i0 < K; i0 += 32 * U) {
            int32_t v[U];
#pragma unroll
            for (int u = 0; u < U; ++u) v[u] = i0 + u * 32 + lane < K ? rd.out[i0 + u * 32 + lane] : 0;
            for (int rr = 1; rr < rd.out_rows; ++rr) {
              int32_t* const o = rd.out + (size_t)rr * rd.out_stride + i0 + lane;
#pragma unroll
              for (int u = 0; u < U; ++u)
                if (i0 + u * 32 + lane < K) o[u * 32] = v[u];
            }
          }
          if (rd.out_score)
            for (int rr = 1; rr < rd.out_rows; ++rr)
              for (int i = lane; i < K; i += 32) rd.out_score[(size_t)rr * rd.out_stride + i] = rd.out_score[i];
        }
      }
      __syncwarp();
      if (lane == 0) ptx::mbar_arrive(&s.fin_done[r][fb]);
    }
  }
}

}  // namespace scan
}  // namespace pivot
