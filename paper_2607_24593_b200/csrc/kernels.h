// Host-callable launchers of the library's kernels (internal header).
#pragma once
#include <utility>
#include <cuda_runtime.h>
#include <stdint.h>

#include "common.cuh"

namespace pivot {

constexpr int kMembersPerDesc = 4;
inline int group_chunks(int g) { return (g + kMembersPerDesc - 1) / kMembersPerDesc; }

// One group's fine step (Eq. 8-9): m members re-score the candidate list.
struct GroupDesc {
  const void* q;        // first member [m, H, d] codes, members contiguous
  const float* w;       // [m, H]
  const float* qscale;  // [m, H] or nullptr
  const void* kbase;
  const float* kscale;
  int k_stride = 0;     // bytes between key rows (0: dense)
  const int32_t* cand;  // candidate key positions, valid entries first
  int n_cand;           // valid candidates (0: group is skipped)
  int m;                // members (at most kMembersPerDesc per descriptor)
  int K;                // entries to select per member
  int first_pos;        // position of the first member (slot i sits at first_pos + i)
  int q_row;            // row of the first member inside the raw query tensor (units of H x d)
  int32_t* out;         // [m, out_stride]
  float* out_score;     // optional
  int out_stride;
  // Chunked mode (decode): when ent_out is set the kernel does not select; member r's packed
  // entries go to ent_out[r * ent_stride + slot0 + slot] for a later top-k over the whole list.
  unsigned long long* ent_out;
  int ent_stride;
  int slot0;
  // Paged key cache (decode): kbase / kscale are the page pool and key position s lives in pool
  // row pages[s / 128] * 128 + s % 128; pages == nullptr means one contiguous cache.
  const int32_t* pages = nullptr;
  int n_pages = 0;      // pages in the pool (entries outside [0, n_pages) are treated as holes)
  // Per-query window slots (decode form of Appendix B): the member at position t takes a slot
  // only if t - win_span < position <= t.  The default never excludes anything below t.
  int win_span = 1 << 30;
  // Largest key position a candidate of this group may name (the group's last member); the
  // gather drops anything beyond it and reports DEV_BOUNDS.
  int pos_max = 0x7fffffff;
};

constexpr int kDecodeWinMax = 512;      // most window slots (W + g - 1) of a decode step

constexpr int kDecodeCandChunk = 512;   // candidates per re-score work item in decode

// One query's re-scored candidates (packed entries) awaiting the final top-k.
struct EntryList {
  const unsigned long long* list;
  int n;
  int K;
  int32_t* out;
  float* out_score;
};

// One request of a prefill-shaped call: where it lies in the packed tensors and which of its rows are indexed.
struct PrefillReq {
  int tok0;         // first token (query row = key row) of the request in the packed tensors
  int L;            // its tokens
  int dense_begin;  // first densely scored row of this call (positions are relative to the request)
  int n_dense;      // rows dense_begin .. dense_begin+n_dense-1 are scored densely (guarded groups or dense control)
  int first_group;  // first group taking the proxy path
  int n_proxy;      // groups on the proxy path
  int slot0;        // scan-row slots of the requests before it
  int proxy0;       // proxies of the requests before it
};
constexpr int kMaxPlanReqs = 64;

// One scan row whose prefix was scanned in parts: the top-K of every part, of which merge_parts takes the top-K.
struct MergeRow {
  const int32_t* pos;   // [parts, K] inside the part, which starts at key tile tiles * part / parts; -1: empty
  const float* score;   // [parts, K]
  int parts, tiles, K;
  int32_t* out; float* out_score;
  int out_rows, out_stride;
};
constexpr int kMaxMerge = 16384;      // entries (parts x K) merge_parts takes per row

// Geometry of a prefill-shaped call (by value to the planner kernel).
struct PrefillPlan {
  const void* q; const float* w; const float* qscale;   // raw per-query operands
  const void* kc; const float* kscale;                  // key cache
  int k_stride = 0;                                     // bytes between key rows (0: dense)
  void* proxy_q; float* proxy_w;                        // [nP, H, d], [nP, H]
  int32_t* cand; float* cand_score;                     // [nP, c] (Refine)
  int32_t* out; float* out_score;                       // [tokens, k]
  int g, c, k, mode, dtype;
  int pool = 0;
  int W = 0;            // local window (Appendix B); 0 = off
  bool skip_trivial = true;   // rows that select all they see are written by the planner instead of scanned
  int* status = nullptr;      // status word and row counter: cleared by the planner (nullptr: left as they are)
  int n_slots = 0;      // scan-row slots: the rows of all requests, each request padded to whole blocks of four if there are several
  int n_proxy = 0;      // proxies of all requests
  int n_req = 0;
  // split > 1 (one request, no dense rows): every block of scan rows becomes `split` blocks over consecutive parts
  // of the prefix, n_slots (a multiple of four) counts the rows before that
  int split = 1;
  int32_t* part_pos = nullptr; float* part_score = nullptr;     // [n_proxy, split, K]
  MergeRow* merges = nullptr;                                   // [n_proxy]
  PrefillReq req[kMaxPlanReqs];
};

struct DecodePlan {
  const void* q; const float* w; const float* qscale;   // [B, g, H, d] ...
  const void* kc; const float* kscale;                  // [B, Lmax, d], [B, Lmax]
  int k_stride = 0;                                     // bytes between key rows (0: dense)
  const int32_t* pos0;
  void* proxy_q; float* proxy_w;                        // [B, H, d], [B, H]
  int32_t* cand; float* cand_score;                     // [B, c]
  int32_t* out; float* out_score;                       // [B, g, k]
  int B, Lmax, g, c, k, mode, dtype, guard_len;
  const int32_t* block_table = nullptr;                 // paged cache: [B, Lmax / 128] pool pages
  int n_pages = 0;
  int W = 0;                                            // per-query local window (Appendix B, decode form)
  int* status = nullptr;                                // device status word (a bad pos0 is reported there)
  // Dense control (Eq. 1 per query): every query of the step is planned as a sequence of its own
  // with one member.  kv_share consecutive plan slots then share one key cache: slot b reads cache
  // b / kv_share and sits at position pos0[b / kv_share] + b % kv_share.  raw_q: the scan rows
  // are the raw queries themselves (no proxy is built); the planner leaves their effective gates
  // fl32(w * qscale) in proxy_w.
  int kv_share = 1;
  bool raw_q = false;
};

#ifndef PIVOT_CHK
#define PIVOT_CHK 32
#endif
constexpr int kThresholdRefreshTiles = PIVOT_CHK;   // the scan's append warps re-read their rows' thresholds off the histograms this often
// ... sooner while a threshold still moves fast: first when a row has seen 5/4 K keys, then after half as many tiles as it has
// seen, kRefreshMin at least; not with kRefreshLast or fewer tiles left of its block (a refresh takes some two tiles' time:
// without this 12 packed requests took 3 % longer); and as soon as the segment's room asks for it, which is thinned
// out only when that is less than kLeastRoomTiles.  Against a refresh every 32 tiles, with room kept for as many (and the boundary
// read of that time), us, medians of calls timed in turn: 16K tokens, K = 512 480 -> 425 (runs of one side within 2 %); dense 5001
// tokens, K = 512 193.6 -> 175.7 (0.2 %); dense 32001, K = 1024 5816 -> 5228 (3.5 %).  After a quarter as many tiles instead of half: 1 .. 3 % slower.
constexpr int kRefreshMin = 4, kRefreshLast = 12, kLeastRoomTiles = 8;

struct ScanScratch {
  uint32_t* cand_key;   // [n_cta][2][cap]   (CUDA-core kernels: separate key / index arrays)
  int32_t* cand_idx;    // [n_cta][2][cap]
  unsigned long long* cand64;   // the same memory seen as packed 64-bit entries (tensor-core kernels)
  int cap;
  int n_cta;
  int* status;
  int* counter;         // dynamic row scheduler
  uint32_t* rkeys = nullptr;   // re-score: [SMs][2][4][rslots] score keys between the tile loop and the select warps
  int rslots = 0;              // ... slots per row: the candidate budget rounded up to whole 128-key tiles
};

void launch_proxy_build(const void* q, const float* qscale, const float* w, void* proxy_q,
                        float* proxy_w, int rows, int g, int first_group, int n_proxy, int dtype,
                        int pool, cudaStream_t st);
// One kernel prepares a prefill call: proxies (Eq. 4), row and group descriptors, rows without a choice.
cudaError_t launch_prepare_prefill(const PrefillPlan& p, RowDesc* rows, GroupDesc* groups, cudaStream_t st);
void launch_plan_decode(const DecodePlan& p, RowDesc* rows, GroupDesc* groups, cudaStream_t st);
// Decode proxies need the guard test on device (pos0 lives there): rows of guarded sequences
// get K = 0 and are skipped.
void launch_scan_simt(const RowDesc* rows, int n_rows, int dtype, const ScanScratch& s, cudaStream_t st);
void launch_refine_simt(const GroupDesc* groups, int n_groups, int dtype, const ScanScratch& s, cudaStream_t st);

// Operand tensors of a tensor-core scan, for the TMA tensor maps.
struct ScanOperands {
  const void* kc; long long k_rows;        // key cache [k_rows, d]
  const float* kscale;                     // [k_rows] (FP8) or nullptr
  const void* q; int q_rows;               // raw queries [q_rows, H, d]
  const void* proxy_q; int proxy_rows;     // proxies [proxy_rows, H, d]
  int dtype;
  int k_stride = 0;                        // bytes between key rows (0: dense)
};
// rows_per_block consecutive scan rows share one key stream (4 in prefill, 1 in decode).
// fp32_head_sum: keep the gate-weighted head sum in fp32 FMAs even where the tensor-core form
// (FP8, four rows per block) is available.  mean_keys: keys that a scan row sees on average; up to
// kShortBlockKeys (48 tiles) every row has a finisher of its own.  us, two -> four finisher warps, medians of calls timed in turn (runs
// of one side within 0.3 % below 20 tiles, 2 % below 35, 3 .. 5 % above), by the mean: 12 tiles, 12 packed requests 431 -> 407, dense
// K = 256 73.1 -> 66.4, K = 1024 72.6 -> 64.6; 20 tiles, 5003 tokens 157 -> 149, 7K 316 -> 299, dense K = 512 159.8 -> 156.5; 23 tiles,
// 8K 394 -> 378, dense K = 256 and 1024 no change, K = 2048 220 -> 209; 31 .. 43 tiles, requests with dense rows and proxies 12K
// c = 4096 722 -> 699, c = 1024 423 -> 409, c = 8192 850 -> 849, 16K 1095 -> 1075; but dense requests, whose blocks are all
// alike, 35 tiles 444 -> 458 (K = 256), 470 -> 480 (1024), 462 -> 468 (2048), 420 -> 421 (4096), 47 tiles 2 .. 5 % slower for
// the same four budgets; 55 tiles and more, 16K K = 512 412 -> 416, dense 2 .. 5 % slower for every budget.  (When the bound was chosen the dense
// requests of 35 .. 47 tiles gained 0 .. 6 % from it, more for larger budgets: two finishers have become faster since.)
constexpr long long kShortBlockKeys = 6144;
cudaError_t launch_scan_tc(const ScanOperands& op, const RowDesc* rows, int n_rows, int rows_per_block,
                           const ScanScratch& s, int sms, cudaStream_t st, bool fp32_head_sum = false,
                           bool overlap_prev = false, long long mean_keys = 1ll << 40);

cudaError_t launch_refine_tc(const void* q, int q_rows, int dtype, const GroupDesc* groups, int n_groups,
                             const ScanScratch& s, int sms, cudaStream_t st, bool fp32_head_sum = false,
                             bool chunked = false, int max_cand = 0, bool overlap_prev = false);

cudaError_t launch_merge_parts(const MergeRow* rows, int n_rows, int n_max, cudaStream_t st);

// Decode fast path: key-tile-split scan -> per-sequence select -> chunked re-score -> top-k.
struct DecodeFast {
  DecodePlan plan;            // the call's geometry: the prepare kernel plans the sequences itself
  int pool = 0;               // proxy aggregation (the prepare kernel builds the proxies)
  RowDesc* prox;              // [B + B * g] row slots; [0, B) = proxy rows (K = 0: guarded sequence, skipped)
  GroupDesc* groups;          // [B * group_chunks(g)]
  const void* kc; const float* kscale; const void* q; const void* proxy_q;
  int B, Lmax, g, c, k, mode, dtype, sms;
  long long k_rows;           // rows of the key tensor (B * Lmax, or pool pages * 128 when paged)
  int k_stride = 0;           // bytes between key rows (0: dense)
  int W = 0;                  // per-query local window (Appendix B, decode form); Refine only
  bool skip_scan = false;     // the candidate sets come from the caller: no scan, no top-c select
  void* scratch;              // decode_fast_bytes(...) bytes
  ScanScratch scratch_tc;     // candidate scratch of the re-score kernel
  int* status;
  cudaEvent_t ev_scan_begin, ev_scan_end;   // optional: recorded around the scan kernel
  cudaEvent_t ev_select_end = nullptr;      // ... and behind the per-sequence select
};
size_t decode_fast_bytes(int B, int Lmax, int g, int c);
cudaError_t launch_decode_fast(const DecodeFast& d, cudaStream_t st);

long long& launch_counter();
// Top-K of the union of n_seg candidate lists (see pivot_merge_topk); entries = scratch for n_seg * seg_len packed entries.
cudaError_t launch_merge_topk(const float* scores, const int32_t* idx, int n_seg, int seg_len, const int32_t* seg_offset,
                              unsigned long long* entries, int K, int32_t* out_idx, float* out_scores, cudaStream_t st);

// Diagnostic: a kernel whose bounded waits run out after limit_ns (see debug_probe.cu).
cudaError_t launch_wait_expiry_probe(int* status, unsigned long long limit_ns, cudaStream_t st);
// Diagnostic: tensor-pipe / tensor-memory / hand-over timings of one SM (see debug_probe.cu); out = 256 slots.
cudaError_t launch_mma_model_probe(long long* out, cudaStream_t st);
// Diagnostic: rate at which all SMs together can pull the scan's 16 KB key tiles out of L2.
cudaError_t launch_key_stream_probe(const void* keys, int n_keys, int ctas, int tiles, int stages, int mode, long long* out,
                                    cudaStream_t st);

// The opt-in to more than 48 KB of dynamic shared memory is an attribute of (function, device):
// remembered per device, so that a process driving several GPUs sets it on each of them.
constexpr int kMaxDevices = 64;
template <typename Kern>
inline cudaError_t opt_in_dynamic_smem(Kern kern, size_t bytes, bool (&done)[kMaxDevices]) {
  int dev = -1;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const bool tracked = dev >= 0 && dev < kMaxDevices;
  if (tracked && done[dev]) return cudaSuccess;
  e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  if (e == cudaSuccess && tracked) done[dev] = true;
  return e;
}

// Launch with programmatic stream serialisation (`overlap`): the kernel may start before its
// predecessor in the stream has finished and must call ptx::grid_dependency_wait() before it
// touches anything the predecessor writes or reads.  cluster > 1: thread-block clusters of that many
// blocks along x.
template <typename... KArgs, typename... Args>
inline cudaError_t launch_clusters(int cluster, void (*kern)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                                   bool overlap, Args&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  int n = 0;
  if (overlap) {
    attr[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[n++].val.programmaticStreamSerializationAllowed = 1;
  }
  if (cluster > 1) {
    attr[n].id = cudaLaunchAttributeClusterDimension;
    attr[n].val.clusterDim.x = (unsigned)cluster;
    attr[n].val.clusterDim.y = 1;
    attr[n++].val.clusterDim.z = 1;
  }
  cfg.attrs = attr;
  cfg.numAttrs = n;
  return cudaLaunchKernelEx(&cfg, kern, KArgs(std::forward<Args>(args))...);
}
template <typename... KArgs, typename... Args>
inline cudaError_t launch_kernel(void (*kern)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, bool overlap,
                                 Args&&... args) {
  return launch_clusters(1, kern, grid, block, smem, st, overlap, std::forward<Args>(args)...);
}

}  // namespace pivot
