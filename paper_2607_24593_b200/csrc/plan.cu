// Planner kernels: turn a call's geometry into row descriptors (one per scan row) and group
// descriptors (one per Refine group).  Grouping follows Eq. 2 (prefill) and Eq. 3 (decode);
// the short-group guardrail of Algorithm 1 decides which rows are dense.
#include "kernels.h"
#include "plan.cuh"
#include "proxy_math.cuh"
#include "ptx.cuh"

namespace pivot {

namespace {

constexpr int kPrepThreads = 256;
constexpr int kPrepSlots = 32;        // scan-row slots per planning block

// Which request holds entry i of a concatenated numbering (`first` = the request's own start in it).
template <int PrefillReq::*FIRST>
__device__ __forceinline__ int find_req(const PrefillPlan& p, int i) {
  int r = 0;
  while (r + 1 < p.n_req && i >= p.req[r + 1].*FIRST) ++r;
  return r;
}

// Position of a request's j-th scan row: the dense rows come first, then one row per proxy group.
__device__ __forceinline__ int row_pos(const PrefillReq& q, int g, int j) {
  return j < q.n_dense ? q.dense_begin + j : (q.first_group + j - q.n_dense) * g;
}

// Blocks (of four scan rows) of a request whose first row sits at a position below `pos`.
__device__ __forceinline__ int blocks_below(const PrefillReq& q, int g, int pos) {
  int n = min(max(pos - q.dense_begin, 0), q.n_dense);
  const int p0 = q.first_group * g;
  if (pos > p0) n += min((pos - p0 + g - 1) / g, q.n_proxy);
  return (n + 3) / 4;
}

// A row that selects everything it sees: the planner writes it.
struct FillRow { int32_t* out; int n_vis, K, out_rows, out_stride; };

}  // namespace

// One launch prepares a prefill call.  Blocks [0, proxy_blocks) form the proxies (Eq. 4), a warp per unit of
// four (e4m3) or two (bf16) heads; each of the others plans kPrepSlots scan rows and writes the rows among
// them that have no choice.  The two parts are independent, so the planner's few microseconds of
// dependent loads and descriptor stores run beside the proxies' HBM stream instead of in a launch of their
// own (proxies and plan in separate launches: 10.5 + 10.2 us of a 2048-token bf16 request, now one of 10.4).
//
// Scan-row order: rows by ascending prefix, in blocks of four rows that share a key stream (the scan deals
// blocks from the last, longest one down).  One request: slot i is its i-th row.  Several requests: each is
// padded to whole blocks, and a block's place is its rank among the blocks of all requests by the position of
// its first row -- counted in closed form, every request's positions being an ascending sequence -- so that
// the deal stays longest-first over the whole batch.
//
// A row with no more visible keys than it has to select (every row below k of a dense request) selects them
// all: its positions are written here and the scan skips it.
template <int DT>
__global__ void __launch_bounds__(kPrepThreads)
prepare_prefill_kernel(const __grid_constant__ PrefillPlan p, RowDesc* rows, GroupDesc* groups, int proxy_blocks) {
  ptx::grid_launch_dependents();         // the scan may set itself up meanwhile (it waits before it reads)
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (blockIdx.x == 0 && threadIdx.x < 2 && p.status) p.status[threadIdx.x] = 0;
  if ((int)blockIdx.x < proxy_blocks) {
    constexpr int WPG = proxy_units_per_group<DT>();
    const long long wid = (long long)blockIdx.x * (kPrepThreads / 32) + warp;
    const int pr = (int)(wid / WPG);
    if (pr >= p.n_proxy) return;
    const PrefillReq& q = p.req[find_req<&PrefillReq::proxy0>(p, pr)];
    const int t0 = (q.first_group + pr - q.proxy0) * p.g;
    proxy_build_unit<DT>(p.q, p.qscale, p.w, p.proxy_q, p.proxy_w, q.tok0 + t0, min(p.g, q.L - t0), pr, (int)(wid % WPG),
                         p.pool, lane);
    return;
  }
  __shared__ FillRow fill[kPrepSlots];
  const int i = ((int)blockIdx.x - proxy_blocks) * kPrepSlots + (int)threadIdx.x;
  if (threadIdx.x < kPrepSlots) fill[threadIdx.x].K = 0;
  if (threadIdx.x < kPrepSlots && i < p.n_slots) {
    const int ri = find_req<&PrefillReq::slot0>(p, i);
    const PrefillReq& q = p.req[ri];
    const int j = i - q.slot0;                       // row of the request
    const int jb = j >> 2;
    int slot = i;
    if (p.n_req > 1) {
      const int pos = row_pos(q, p.g, jb * 4);
      int rank = 0;
      for (int o = 0; o < p.n_req; ++o) rank += blocks_below(p.req[o], p.g, o < ri ? pos + 1 : pos);
      slot = rank * 4 + (j & 3);
    }
    const size_t qrow = (size_t)kHeads * kDim * (DT == DT_FP8 ? 1 : 2);
    RowDesc r;
    r.kbase = (const char*)p.kc + (size_t)q.tok0 * (p.k_stride > 0 ? (size_t)p.k_stride : kDim * (DT == DT_FP8 ? 1 : 2));
    r.kscale = p.kscale ? p.kscale + q.tok0 : nullptr;
    r.k_row0 = q.tok0;
    if (j < q.n_dense) {
      const int t = q.dense_begin + j;      // query row (= position) of this dense row
      const size_t row = (size_t)q.tok0 + t;
      r.q = (const char*)p.q + row * qrow;
      r.w = p.w + row * kHeads;
      r.qscale = p.qscale ? p.qscale + row * kHeads : nullptr;
      r.n_vis = t + 1;
      r.K = p.k;
      r.out = p.out + row * p.k;
      r.out_score = p.out_score ? p.out_score + row * p.k : nullptr;
      r.out_rows = 1;
      r.out_stride = p.k;
      r.q_map = 0; r.q_row = (int)row;
    } else if (j < q.n_dense + q.n_proxy) {
      const int lp = j - q.n_dense;         // proxy of the request
      const int pr = q.proxy0 + lp;         // ... and of the call
      const int t0 = (q.first_group + lp) * p.g;
      const int m = min(p.g, q.L - t0);
      const size_t row = (size_t)q.tok0 + t0;
      r.q = (const char*)p.proxy_q + (size_t)pr * qrow;
      r.w = p.proxy_w + (size_t)pr * kHeads;
      r.qscale = nullptr;
      // With a local window the proxy ranks s <= t0 - W only (Appendix B); the window itself is
      // appended to the candidate set below.
      r.n_vis = p.W > 0 ? max(t0 - p.W + 1, 0) : t0 + 1;
      r.q_map = 1; r.q_row = pr;
      if (p.mode == 0) {   // Reuse: the proxy top-k goes to every member (Eq. 6)
        r.K = p.k;
        r.out = p.out + row * p.k;
        r.out_score = p.out_score ? p.out_score + row * p.k : nullptr;
        r.out_rows = m;
        r.out_stride = p.k;
      } else {             // Refine: top-c candidate set (Eq. 7)
        const int w_g = p.W > 0 ? p.W + m - 1 : 0;      // slots reserved for the window union
        r.K = p.c - w_g;
        r.out = p.cand + (size_t)pr * p.c;
        for (int s0 = 0; s0 < w_g; ++s0) {              // t0-W+1 .. t0+m-1, ascending
          const int s = t0 - p.W + 1 + s0;
          p.cand[(size_t)pr * p.c + (p.c - w_g) + s0] = s >= 0 ? s : -1;
          if (p.cand_score) p.cand_score[(size_t)pr * p.c + (p.c - w_g) + s0] = __int_as_float(0x7fc00000);
        }
        r.out_score = p.cand_score ? p.cand_score + (size_t)pr * p.c : nullptr;
        r.out_rows = 1;
        r.out_stride = p.c;
        GroupDesc gd;
        gd.q = (const char*)p.q + row * qrow;
        gd.w = p.w + row * kHeads;
        gd.qscale = p.qscale ? p.qscale + row * kHeads : nullptr;
        gd.kbase = r.kbase;
        gd.kscale = r.kscale;
        gd.k_stride = p.k_stride;
        gd.cand = r.out;
        gd.n_cand = p.W > 0 ? p.c : min(p.c, r.n_vis);   // with a window every slot is read (pads are skipped)
        gd.m = m;
        gd.K = p.k;
        gd.first_pos = t0;
        gd.pos_max = t0 + m - 1;
        gd.q_row = (int)row;
        gd.out = p.out + row * p.k;
        gd.out_score = p.out_score ? p.out_score + row * p.k : nullptr;
        gd.out_stride = p.k;
        gd.ent_out = nullptr; gd.ent_stride = 0; gd.slot0 = 0;
        const int chunks = (p.g + kMembersPerDesc - 1) / kMembersPerDesc;
        put_group_chunks(groups + (size_t)pr * chunks, gd, p.g, p.dtype);
      }
    } else {
      // Padding of the request's last block: never live.  Its queries are still multiplied (the head sum of FP8 runs
      // over the block's four rows at once, with zero gates for this one, and zero times NaN is NaN), so they are
      // those of the block's last live row: any other row's may not have been written yet, or not be numbers.
      r.q = p.q; r.w = p.w; r.qscale = p.qscale;
      r.n_vis = 0; r.K = 0;
      r.out = nullptr; r.out_score = nullptr; r.out_rows = 0; r.out_stride = 0;
      r.q_map = q.n_proxy > 0 ? 1 : 0;
      r.q_row = q.n_proxy > 0 ? q.proxy0 + q.n_proxy - 1 : q.tok0 + q.dense_begin + q.n_dense - 1;
    }
    if (p.split > 1) {
      // The block's key tiles in p.split equal runs, each a block of its own; what the parts select goes to the
      // merge.  (The runs are the block's, so that its four rows keep sharing one key stream.)
      const int last = row_pos(q, p.g, min(jb * 4 + 3, q.n_proxy - 1));
      const int tiles = (max(p.W > 0 ? last - p.W + 1 : last + 1, 0) + 127) / 128;
      const RowDesc whole = r;
      const int pr = q.proxy0 + j;
      for (int h = 0; h < p.split; ++h) {
        const int lo = (int)((long long)tiles * h / p.split) * 128, hi = (int)((long long)tiles * (h + 1) / p.split) * 128;
        r.k_row0 = whole.k_row0 + lo;
        r.n_vis = min(max(whole.n_vis - lo, 0), hi - lo);
        if (whole.K > 0) {
          r.out = p.part_pos + ((size_t)pr * p.split + h) * whole.K;
          r.out_score = p.part_score + ((size_t)pr * p.split + h) * whole.K;
          r.out_rows = 1;
        }
        rows[(jb * p.split + h) * 4 + (j & 3)] = r;
      }
      if (whole.K > 0)
        p.merges[pr] = MergeRow{p.part_pos + (size_t)pr * p.split * whole.K, p.part_score + (size_t)pr * p.split * whole.K,
                                p.split, tiles, whole.K, whole.out, whole.out_score, whole.out_rows, whole.out_stride};
    } else {         // (a split call has no rows without a choice)
      if (p.skip_trivial && r.K > 0 && r.n_vis <= r.K && !r.out_score) {
        fill[threadIdx.x] = FillRow{r.out, r.n_vis, r.K, r.out_rows, r.out_stride};
        r.K = 0;
      }
      rows[slot] = r;
    }
  }
  __syncthreads();
  for (int s = warp; s < kPrepSlots; s += kPrepThreads / 32) {
    const FillRow f = fill[s];
    for (int rr = 0; rr < f.out_rows && f.K > 0; ++rr)
      for (int e = lane; e < f.K; e += 32) f.out[(size_t)rr * f.out_stride + e] = e < f.n_vis ? e : -1;
  }
}

cudaError_t launch_prepare_prefill(const PrefillPlan& p, RowDesc* rows, GroupDesc* groups, cudaStream_t st) {
  const int units = p.dtype == DT_FP8 ? proxy_units_per_group<DT_FP8>() : proxy_units_per_group<DT_BF16>();
  const long long warps = (long long)p.n_proxy * units;
  const int proxy_blocks = (int)((warps + kPrepThreads / 32 - 1) / (kPrepThreads / 32));
  const int plan_blocks = (p.n_slots + kPrepSlots - 1) / kPrepSlots;
  if (proxy_blocks + plan_blocks <= 0) return cudaSuccess;
  if (p.dtype == DT_FP8)
    prepare_prefill_kernel<DT_FP8><<<proxy_blocks + plan_blocks, kPrepThreads, 0, st>>>(p, rows, groups, proxy_blocks);
  else
    prepare_prefill_kernel<DT_BF16><<<proxy_blocks + plan_blocks, kPrepThreads, 0, st>>>(p, rows, groups, proxy_blocks);
  ++launch_counter();
  return cudaGetLastError();
}

__global__ void plan_decode_kernel(DecodePlan p, RowDesc* rows, GroupDesc* groups) {
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= p.B) return;
  if (!plan_decode_sequence(p, b, rows, groups)) fill_decode_rows_empty(p, b, 0, 1);
  if (p.raw_q) raw_query_gates(p, b, 0, 1);
}

void launch_plan_decode(const DecodePlan& p, RowDesc* rows, GroupDesc* groups, cudaStream_t st) {
  plan_decode_kernel<<<(p.B + 127) / 128, 128, 0, st>>>(p, rows, groups);
  ++launch_counter();
}

}  // namespace pivot
