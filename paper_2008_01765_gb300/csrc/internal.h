// Internal interfaces between the host orchestration (api.cu) and the kernel files.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

#include "bos.h"
#include "common.cuh"

namespace bos {

constexpr int kModeFirst = 1;
constexpr int kModeLast = 2;

struct PassArgs {
  const void* in;           // FIRST: input records
  const void* in_rec;       // otherwise: slot records of the previous array
  const uint32_t* in_tag;   // otherwise: slot tags of the previous array
  void* out_rec;            // not LAST: slot records of the next array
  uint32_t* out_tag;        // not LAST: slot tags of the next array
  void* out0;               // LAST: output records
  void* out1;               // LAST: alternate output (sort scratch), see out_sel
  uint32_t out_sel;         // LAST: 1 = write out1 when an odd number of radix passes will run
  uint32_t skip_publish;    // debug: subproblem 0 of the LAST pass never publishes
  uint64_t n, B;
  uint32_t Z, L, i, k, attempt, ticket_slot;
  uint64_t seed;
  Ctrl* ctrl;
  unsigned long long* status;  // LAST: look-back words, one per subproblem
  uint32_t buf_in_rec, buf_in_tag, buf_out_rec, buf_out_tag;  // trace buffer ids
  Trace trace;
  const uint16_t* ord;      // LAST (persistent kernel): in-bin permutation table, B*Z slot indexes
  uint64_t bucket0;         // global index of local bucket 0 (a shard's buckets; 0 otherwise): the
                            // first pass's groups and the in-bin permutation keys use global indexes
  const uint32_t* load;     // LAST (orp_last.cu): [B] reals per final bucket, counted ahead of the pass;
                            // status[q] then holds the inclusive prefix of the subproblems' reals
};

// In-bin permutation table (perm_table.cu): row b < B lists final bucket b's slots in the order
// of the Section 3.2 keys of (b, attempt, seed), ord[b*Z + rank] = slot. With the LAST pass's
// input tags (tag != null; levels i..i+k-1 of L) a row holds the bucket's m real slots, then
// 0xFFFF, m counted first into load[b] by a kernel of its own; without them, all Z slots. Z a
// multiple of 32, <= 4096; k <= 12.
struct PermTableArgs {
  uint64_t bucket0;      // global index of local bucket 0 (the keys use global bucket indexes)
  uint16_t* ord;
  const uint32_t* tag;
  uint32_t* load;        // [B] reals per final bucket (workspace), written and read here
  uint64_t B;
  uint32_t Z, attempt, i, k, L, buf_tag;
  uint64_t seed;
  Trace trace;
  // prefix of the loads over the LAST subproblems (null: not wanted): status[q] = inclusive prefix of
  // the reals of subproblems 0..q (decoupled look-back; zeroed words, a zeroed ticket)
  unsigned long long* status;
  uint32_t* ticket;
  Ctrl* ctrl;
  uint32_t skip_publish;  // debug: subproblem 0 never publishes
};
cudaError_t launch_perm_table(const PermTableArgs& a, cudaStream_t st, bool trace);

uint32_t orp_smem_bytes(int R, uint32_t Z, uint32_t k, bool last);

// One launch of the one-CTA-per-subproblem pass over many arrays (batched ORP).
struct BatchPass {
  const PassArgs* args;   // device: one entry per array in this launch
  const uint64_t* first;  // device: running sum of subproblem counts, narr + 1 entries
  uint32_t narr;
  uint64_t nblocks;       // = first[narr]
  uint32_t* ticket;       // device: zeroed counter (LAST passes)
};
cudaError_t launch_orp_pass_batched(const BatchPass& bp, int mode, uint32_t smem, cudaStream_t st, int R,
                                    bool trace);
cudaError_t launch_orp_pass(const PassArgs& a, int mode, uint64_t grid, cudaStream_t st, int R,
                            bool trace);

// Persistent, cluster-wide ORP pass (orp_fast.cu); Z must be a multiple of 32.
uint32_t orp_fast_smem_bytes(int R, uint32_t Z, uint32_t k, uint32_t C, bool last);
// Co-resident clusters (C > 1) or CTAs per SM (C = 1) of that configuration; 0 = cannot run.
int orp_fast_occupancy(int R, int mode, uint32_t Z, uint32_t k, uint32_t C);
cudaError_t launch_orp_fast(const PassArgs& a, int mode, uint32_t C, uint32_t max_clusters, cudaStream_t st,
                            int R, bool trace);

// Batched forms of the streaming, table and packed-tile kernels: one CTA per unit, a unit being
// subproblem y of array x of the launch's argument list.
struct StreamLayout {  // shared memory of the streaming pass (orp_stream.cu)
  uint32_t ring_rec, ring_tag, list, stage, stage_bytes, zero, cf, acc, tail, done, misc, total;
  uint32_t stages, lub;  // batches in flight; log2 of the input buckets (groups) per batch
};
struct LastLayout {  // shared memory of the packed-tile last pass (orp_last.cu)
  uint32_t stage, stage_bytes, cnt, base, fill, misc, total;
  uint32_t cap, stages, lub, stride;  // tile records, stages, log2 buckets per batch, u16 per row of counts
};
struct BatchStream {
  PassArgs a;
  StreamLayout lay;
};
struct BatchLast {
  PassArgs a;
  LastLayout lay;
};
StreamLayout orp_stream_layout(int R, uint32_t Z, uint32_t k, bool first);
LastLayout orp_last_layout(int R, uint32_t Z, uint32_t k);
cudaError_t launch_orp_stream_batched(const BatchStream* args, const uint2* units, uint32_t nunits, uint32_t smem,
                                      bool first, cudaStream_t st, int R, bool trace);
cudaError_t launch_orp_last_batched(const BatchLast* args, const uint2* units, uint32_t nunits, uint32_t smem,
                                    cudaStream_t st, int R, bool trace);
// final loads with their prefix (units in array order, taken by ticket), and the table rows
cudaError_t launch_perm_table_batched(const BatchLast* args, const uint2* units, uint32_t nunits, uint32_t max_k,
                                      uint32_t max_Z, uint32_t* ticket, cudaStream_t st, bool trace);

// Streaming first / middle ORP pass (orp_stream.cu): one CTA per subproblem, input buckets
// through a TMA ring, output chunks write-combined in shared memory; Z a multiple of 32, <= 2048.
// Most levels a streaming pass holds in smem_limit bytes (0: the kernel cannot take this Z).
uint32_t orp_stream_max_k(int R, uint32_t Z, bool first, uint32_t smem_limit);
inline uint32_t orp_stream_min_k() { return 5; }  // of a caller-given k; automatic plans go down to 4
double orp_stream_sub_us(uint32_t Z, uint32_t k, bool first, double fill);  // planner: one subproblem on one SM
cudaError_t launch_orp_stream(const PassArgs& a, bool first, cudaStream_t st, int R, bool trace);

// LAST pass with known final loads and table (orp_last.cu): a.load, a.status and a.ord filled by
// launch_perm_table. Z a multiple of 32, <= 2048; k <= orp_last_max_k.
uint32_t orp_last_max_k(int R, uint32_t Z);  // 0: the kernel cannot take this Z
double orp_last_sub_us(int R, uint32_t Z, uint32_t k, double fill);  // planner: one subproblem on one SM
cudaError_t launch_orp_last(const PassArgs& a, cudaStream_t st, int R, bool trace);

// The ORP with O(1) client storage (oblivious.cu, Section 4.1): bitonic-sort MergeSplits, one
// launch per level, bitonic in-bin permutations, a scan of the loads and the strip.
struct ObliviousArgs {
  const void* in;        // n input records
  void* out0;            // n output records
  void* out1;            // alternate output (sort scratch); used when out_sel and an odd number of
  uint32_t out_sel;      // radix passes will run (as the fused LAST pass chooses)
  void* rec[2];          // slot record arrays (B*Z each), used in turn
  uint32_t* tag[2];      // slot tag arrays
  uint32_t* load;        // [B] reals per final bucket
  uint32_t* off;         // [B] output offsets inside scan blocks
  uint32_t* part;        // [B / 4096 + 1] scan block offsets
  uint64_t n, B;
  uint32_t Z, L, attempt;
  uint64_t seed;
  Ctrl* ctrl;
  Trace trace;
};
uint32_t oblivious_smem_bytes(int R, uint32_t Z);
cudaError_t launch_oblivious_orp(const ObliviousArgs& a, int R, cudaStream_t st, bool trace);

// Stable merge sort by key (mergesort.cu): runs of 4096 sorted in shared memory, then merge
// passes that double the run width. The result lands in buf0; the block-sorted runs are written
// to buf0 when merge_passes(n) is even and to buf1 when it is odd, so `in` may be that buffer.
// hooks (optional) bracket the block sort (stage 0) and each merge pass (stage 1) with the algorithmic
// bytes.
struct MergeHooks {
  int (*begin)(cudaStream_t st, int stage, double bytes);
  void (*end)(int slot, cudaStream_t st);
};
uint32_t merge_passes(uint64_t n);
cudaError_t launch_merge_sort(const void* in, void* buf0, void* buf1, uint64_t n, int R, cudaStream_t st,
                              const MergeHooks& hooks);

// LSD radix sort (radix.cu)
struct RadixArgs {
  const void* in;                 // histogram source (any order of the same multiset)
  void* buf0;                     // final output
  void* buf1;                     // scratch of n records
  uint64_t n;
  uint32_t* hist;                 // [digits][256]
  unsigned long long* dbase;      // [digits][256] exclusive digit offsets
  unsigned long long* status;     // [tiles][256] look-back words
  Ctrl* ctrl;
  uint32_t ticket_base;
};
uint64_t radix_tiles(uint64_t n, int R);

// Hybrid radix sort (sort_hybrid.cu): MSD partitions on the top one or two digits, then an on-chip
// sort of every range of groups; falls back to the LSD passes (ctrl->sort_mode = 0) when a group
// exceeds Local<R>::kCap records. stage: 0 histogram (hist and joint), 1 plan, 2 partition by the
// top varying digit, 3 partition by the next one inside every bucket, 4 the on-chip sort.
constexpr uint32_t kSortClasses = 6;
// What the plan kernel tells the host (mapped pinned memory): the host launches only the passes and the
// range classes that the plan calls for. seq is written last.
struct HostPlan {
  uint32_t seq, mode, live, list[kSortClasses];
};
struct HybridArgs {
  const void* in;                   // histogram source (the ORP's input: the same multiset of keys)
  void* buf0;                       // final output
  void* buf1;                       // scratch of n records
  uint64_t n;
  uint32_t* hist;                   // [digits][256] digit counts (shared with the LSD path)
  unsigned long long* dbase;        // [digits][256] exclusive digit offsets (written by the plan)
  uint32_t* joint;                  // [65536] counts of the top two digits
  unsigned long long* gstart;       // [65537] group starts
  uint32_t* rlist;                  // [65537] first group of every range
  unsigned long long* first;        // [257] partition tiles before every top-digit bucket
  uint32_t* meta;                   // [11] mode, top varying digit, next varying digit, ranges left over,
                                    // starts of the six range classes' lists in ridx and their end
  uint32_t* ridx;                   // [65536] the ranges, class by class
  unsigned long long* status;       // look-back words for radix_tiles(n) + 256 tiles
  unsigned char* scratch;           // hybrid_spill_bytes(n, R): one spill buffer per on-chip-sort CTA
  uint32_t local_ctas;              // = hybrid_local_ctas(n, R)
  HostPlan* host;                   // null: the plan stays on the device
  uint32_t host_seq;
  Ctrl* ctrl;
};
uint32_t hybrid_local_ctas(uint64_t n, int R);
size_t hybrid_spill_bytes(uint64_t n, int R);
// list (stage 4): ranges of every class (their launches are left out where there are none).
cudaError_t launch_hybrid(const HybridArgs& a, int R, int stage, const uint32_t* list, cudaStream_t st);
// Radix stages over many arrays in one launch (batched sort).
struct BatchRadix {
  const RadixArgs* args;  // device: one entry per array
  const uint64_t* first;  // device: running sum of tiles (kTile records each), narr + 1 entries
  uint32_t narr;
  uint64_t nblocks;       // = first[narr]
  uint32_t* ticket;       // device: the digit passes' tickets (zeroed)
  uint32_t* lsd;          // device: the digits that some array's LSD passes take (zeroed; set by the plans)
};
// stage 0 = histograms, 1 = the digit passes
cudaError_t launch_radix_batched(const BatchRadix& br, int R, int stage, cudaStream_t st);
// Batched hybrid sort (sort_hybrid.cu): every array's plan (digit offsets, its mode: kBatchOnChip, 2 or 0,
// its ranges in the lists of classes 0..4), the partition of the arrays in mode 2, then one launch per
// class. The ORP's last pass writes the output buffer in either mode (both count as even).
constexpr uint32_t kBatchOnChip = 4;  // the array is one range, sorted in place
struct BatchSort {
  BatchRadix br;
  uint4* list;        // [kSortClasses - 1][cap] ranges: array, first record, records, sorted in place
  uint32_t cap;
  uint32_t P;         // records of a range of packed groups, at most
  uint64_t max_n;     // records of the largest array: classes beyond its size are not launched
  uint32_t* count;    // [kSortClasses - 1] ranges listed (zeroed), then [kSortClasses - 1] taken (zeroed)
  uint32_t* ticket;   // partition tiles (zeroed)
};
uint32_t batch_sort_ranges(uint64_t n, int R);  // most ranges of an array of n records
uint32_t batch_sort_cap(int R);                     // arrays above it may be left to the LSD passes
uint32_t batch_sort_pack(uint64_t records, int R);  // P for a batch of that many records
// stage 0: plans; 1: partition; 2: the range classes
cudaError_t launch_batch_sort(const BatchSort& bs, int R, int stage, cudaStream_t st);
cudaError_t launch_radix_hist(const RadixArgs& a, int R, cudaStream_t st);
cudaError_t launch_radix_prep(const RadixArgs& a, int R, cudaStream_t st);
cudaError_t launch_radix_pass(const RadixArgs& a, int R, uint32_t digit, cudaStream_t st);

// Bucket ORP with a caller-chosen workspace (api.cu); workspace bytes of the ORP alone.
size_t orp_workspace_bytes(uint64_t n, const bos_params* p);
bos_status orp_with_workspace(const void* d_in, void* d_out, uint64_t n, const bos_params* p,
                              void* d_ws, size_t ws_bytes, void* stream, bos_info* info);

// Bitonic comparator (bitonic.cu)
cudaError_t launch_bitonic(const void* in, void* out, uint64_t n, int R, cudaStream_t st);

}  // namespace bos
