// Streaming bucket ORP pass (sm_103a): the first pass and the middle passes of a fused plan.
//
// A pass applies k butterfly levels of Algorithm 3.1 (levels i..i+k-1): subproblem
// q = G*2^i + t reads the input buckets G*2^(i+k) + s*2^i + t (s < 2^k) and writes the contiguous
// output buckets q*2^k + u, each real going to u = label bits [L-1-i .. L-i-k], stable by (s, slot),
// then dummies (the MergeSplit order of the butterfly; Figure 1).
//
// The persistent-cluster kernel (orp_fast.cu) holds all 2^k output buckets on chip, which caps k
// by shared memory. This kernel streams instead: one CTA takes a whole subproblem and reads its
// input in order, in batches of one, two or four input buckets (groups of the input in the first
// pass) brought in by TMA bulk copies, about 1024 reals each. Every output bucket owns a ring of
// kRingSlots / 2^k slots in shared memory; a real is appended to its bucket's ring at its stable
// rank, and whenever a ring holds a whole chunk of kChunk slots the chunk leaves for HBM (coalesced
// 16-byte stores). At the end of the subproblem every bucket's last partial chunk is padded with
// dummies and its remaining chunks are written as dummies. So shared memory bounds the rings, not
// the subproblem, and one pass applies up to 8 levels with no cluster.
//
// Obliviousness (Section 3.1): reads are whole input buckets (or the whole input range of the
// groups); writes are whole chunks of kChunk slots, and every chunk of every output bucket is
// written exactly once. The multiset of addresses is therefore a function of (n, Z, k, pass) alone;
// only the order in which chunks leave depends on the labels, as in every GPU schedule here.
//
// One batch, two block barriers; sixteen warps work, a seventeenth issues the copies and counts:
//   A  every real draws a place in its bucket's list (shared-memory atomic, which also returns the
//      bucket's fill) and leaves its slot index there; unused places are above every index;
//   -- barrier; the batch is redone in smaller rounds if a list ran out of places (see below)
//   B  a real's stable rank is the number of listed indexes below its own: the list is read eight
//      words at a time (one 16-byte load) and compared two words per subtraction. The record goes
//      to its ring slot; a real that completes a chunk enters the chunk in the done list;
//   -- barrier; the batch's stage is free, the next TMA copies into it
//   C  the completed chunks leave, eight lanes to a chunk. C of a batch runs in the same barrier
//      interval as A of the next one (lists, counts and fills are double-buffered).
// Half of a middle pass's slots are dummies, at the end of every bucket, so a thread's slots are
// taken half a bucket apart: every warp gets about the same rows of reals. The dummies that a pass
// writes, half of its output, leave as bulk stores from a block of dummies in shared memory, spread
// by the last warp over the batches of the next subproblem: all CTAs end their subproblems at the
// same time, and written there the dummies took 95,000 cycles of write bandwidth while nothing was
// read, 750 per batch.
//
// What bounds it: latency between the barriers and shared-memory wavefronts (random 16-byte
// accesses): about 4800 cycles per batch, where the copy bandwidth alone would allow 3800 in a
// middle pass. n = 2^29 16-byte records, Z = 1024, k = 8: first pass 14.6 -> 8.25 ms (3643 GB/s),
// middle pass 15.9 -> 8.05 ms (5338 GB/s) against the kernel before it (1024 threads, three
// barriers, lists compared entry by entry, level counters by eight of the working warps: 1500
// cycles of each batch). Spilled registers cost as much as all of that gained: the layout is a
// kernel parameter (constant memory), and each step is written out once.
//
// A list holds kListWords / 2^k places. At about 1024 reals a batch it overflows about once in
// thousands of batches; then the batch is redone in smaller rounds: halved while a round would
// overflow, 16 slots at the least, which always fit (16 <= kListWords / 2^k, and a ring holds
// kChunk - 1 leftover slots and a full list).
//
// Overflow (MergeSplit receives more than Z reals, Lemma 3.2): the level-(i+l) buckets of the
// subproblem (l = 1..k-1) gather 2^l consecutive input buckets and the digits with a common l-bit
// prefix; per-batch digit counts are folded into one counter per (level, prefix) and checked at the
// end of each block. A batch of four input buckets holds two level-1 blocks, which are counted on
// their own (middle pass; two groups of the first pass hold at most Z records). The final level is
// the bucket's fill.
#include "common.cuh"
#include "internal.h"

namespace bos {
namespace {

constexpr int kST = 512;            // worker threads; one more warp issues the copies and checks the levels
constexpr int kSW = kST / 32;
constexpr int kSThreads = kST + 32;
constexpr uint32_t kChunk = 8;          // slots per HBM write (128 B of 16-byte records)
constexpr uint32_t kRingSlots = 6144;   // ring slots of all output buckets together (24 each at k = 8)
constexpr uint32_t kListWords = 4096;   // list places of all output buckets together (16 each at k = 8):
                                        // 0x8000 | slot index, or 0xFFFF when unused
constexpr uint32_t kBatchSlots = 2048;  // most slots per batch of a middle pass (four per thread)
constexpr uint32_t kBatchRecs = 1024;   // most records per batch of the first pass (two per thread)
constexpr uint32_t kWhole = 2 * kBatchSlots;  // round size of a batch's first round: all of it, and above every
                                              // size of a redone round (doubled only while below the batch's)
constexpr uint32_t kSub = 16;           // slots per round when a batch is redone
constexpr uint32_t kDone = (kBatchSlots + 256 * 7) / 8;  // most chunks a batch completes
constexpr uint32_t kAcc = 11;           // level counters per lane of the last warp
constexpr uint32_t kZeroRecs = 4096, kZeroTags = 512;  // bytes of dummies in shared memory (bulk stores)
constexpr uint32_t kMaxZ = 2048;
constexpr uint32_t kMinK = 4, kMaxK = 8;
static_assert(kSub <= (kListWords >> kMaxK), "the smallest round always fits the lists");
static_assert((kListWords >> kMaxK) + kChunk - 1 <= (kRingSlots >> kMaxK), "a full list fits a ring");
static_assert((kListWords >> kMinK) + kChunk - 1 <= (kRingSlots >> kMinK), "a full list fits a ring");

inline uint32_t st_align(uint32_t x, uint32_t a) { return (x + a - 1) / a * a; }

inline StreamLayout stream_layout(int R, uint32_t Z, uint32_t k, bool first) {
  const uint32_t D = 1u << k;
  StreamLayout l{};
  // one, two or four input buckets (groups of at most Z / 2 records) per batch
  const uint32_t per = first ? Z / 2 : Z, most = first ? kBatchRecs : kBatchSlots;
  l.lub = per * 4 <= most ? 2u : per * 2 <= most ? 1u : 0u;
  const uint32_t ub = 1u << l.lub;
  l.stages = first ? 3u : 2u;
  uint32_t off = 0;
  l.ring_rec = off;
  off += kRingSlots * R;
  l.ring_tag = off;
  off += kRingSlots * 4;
  l.list = off;
  off += 2 * kListWords * 2;
  // first pass: the batch's records plus one of alignment; middle pass: its tags, then its records
  l.stage_bytes = first ? st_align((ub * (Z / 2) + 2) * R, 128) : st_align(ub * Z * (4 + R), 128);
  l.stage = st_align(off, 128);
  off = l.stage + l.stages * l.stage_bytes;
  l.zero = off;
  off += kZeroRecs + kZeroTags;
  l.cf = off;
  off += 2 * D * 4;
  l.acc = off;
  off += kAcc * 32 * 4;
  l.tail = off;
  off += D * 2;
  l.done = off;
  off += kDone * 2;
  l.misc = st_align(off, 16);
  off = l.misc + 80;
  l.total = off;
  return l;
}

// Subproblems q0, q0 + qstep, .. (mysub of them) of one array.
template <int R, bool FIRST, bool TRACE>
__device__ __forceinline__ void orp_stream_body(const PassArgs& a, const StreamLayout& lay, const uint64_t q0,
                                                const uint32_t mysub, const uint32_t qstep) {
  using Rec = typename RecT<R>::T;
  constexpr uint32_t kItems = (FIRST ? kBatchRecs : kBatchSlots) / kST;  // slots per thread per batch
  extern __shared__ __align__(128) unsigned char smem[];
  const uint32_t Z = a.Z, k = a.k, D = 1u << k, L = a.L, i = a.i;
  const uint32_t shift = L - i - k;
  Rec* ring_rec = reinterpret_cast<Rec*>(smem + lay.ring_rec);
  uint32_t* ring_tag = reinterpret_cast<uint32_t*>(smem + lay.ring_tag);
  uint16_t* list = reinterpret_cast<uint16_t*>(smem + lay.list);  // [2][cap / 8][D][8]
  uint32_t* cf = reinterpret_cast<uint32_t*>(smem + lay.cf);  // [2][D] reals before the batch << 12 | reals of the batch
  uint16_t* done = reinterpret_cast<uint16_t*>(smem + lay.done);  // completed chunks: bucket << 8 | chunk
  uint16_t* tail = reinterpret_cast<uint16_t*>(smem + lay.tail);  // [D] first slot of the last subproblem's dummy chunks
  unsigned long long* bars = reinterpret_cast<unsigned long long*>(smem + lay.misc);  // [lay.stages]
  uint32_t* lv1 = reinterpret_cast<uint32_t*>(smem + lay.misc + 32);  // [2][4] level 1 of a batch of four buckets
  uint32_t* ndone = reinterpret_cast<uint32_t*>(smem + lay.misc + 64);  // [2] completed chunks of the batch

  const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const bool worker = warp < kSW;
  const uint32_t ring = kRingSlots >> k, cap = kListWords >> k;
  const uint32_t third = 11 - k;  // ring = 3 << third
  const uint32_t lub = lay.lub, ub = 1u << lub, NB = D >> lub;  // batches per subproblem
  const uint32_t nst = lay.stages;
  const uint32_t nbatch = mysub * NB;
  const Rec* in_first = reinterpret_cast<const Rec*>(a.in);
  const Rec* in_rec = reinterpret_cast<const Rec*>(a.in_rec);

  // Clears the lists and the chunk count of buffer b (a barrier must follow).
  auto clear_lists = [&](uint32_t b) {
    if (tid < kListWords / 8)
      reinterpret_cast<uint4*>(list + b * kListWords)[tid] = make_uint4(~0u, ~0u, ~0u, ~0u);
    if (tid == 0) ndone[b] = 0;
  };
  static_assert(kListWords <= 8 * kST, "one 16-byte store per thread clears the lists");
  clear_lists(0);
  clear_lists(1);
  if (tid < D) cf[tid] = cf[D + tid] = 0;
  if (tid < 8) lv1[tid] = 0;
  for (uint32_t x = tid; x < kZeroRecs / 16; x += kSThreads)
    reinterpret_cast<uint4*>(smem + lay.zero)[x] = make_uint4(0, 0, 0, 0);
  if (tid < kZeroTags / 16)
    reinterpret_cast<uint4*>(smem + lay.zero + kZeroRecs)[tid] = make_uint4(kDummy, kDummy, kDummy, kDummy);
  fence_proxy_async();  // the bulk stores read the dummies
  if (tid == 0) {
    for (uint32_t s = 0; s < nst; ++s) mbar_init(smem_u32(bars + s), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();

  // first pass: batch s of subproblem q = groups q*D + s*ub .. + ub - 1 (B = 2^L)
  auto first_range = [&](uint64_t q, uint32_t s, uint64_t& lo, uint64_t& hi) {
    const uint64_t g0 = a.bucket0 + q * D + ((uint64_t)s << lub);
    lo = (g0 * a.n) >> L;
    hi = ((g0 + ub) * a.n) >> L;
  };
  // Input records [lo, hi) of a first-pass batch sit at stage index soff + (record - lo); the
  // bulk copy takes [lo2, hi2), the largest sub-range whose global and shared addresses are both
  // 16-byte aligned (d_in is only guaranteed rec_bytes alignment).
  const uint32_t in_odd = R == 8 ? (uint32_t)((reinterpret_cast<uintptr_t>(a.in) >> 3) & 1u) : 0u;
  auto first_bulk = [&](uint64_t lo, uint64_t hi, uint64_t& lo2, uint64_t& hi2, uint32_t& soff) {
    if (R == 8) {
      lo2 = lo + ((lo + in_odd) & 1u);  // (d_in + 8 * lo2) is a multiple of 16
      hi2 = hi - ((hi + in_odd) & 1u);
      soff = (uint32_t)((lo2 - lo) & 1u);  // so that lo2's stage index is even
    } else {
      lo2 = lo;
      hi2 = hi;
      soff = 0;
    }
  };
  auto in_bucket = [&](uint64_t q, uint32_t s) -> uint64_t {
    const uint64_t t = q & ((1ull << i) - 1), G = q >> i;
    return (G << (i + k)) + ((uint64_t)s << i) + t;
  };
  // TMA of batch s of subproblem q into stage st (one thread of the last warp)
  auto issue = [&](uint64_t q, uint32_t s, uint32_t st) {
    const uint32_t bar = smem_u32(bars + st);
    const uint32_t dst = smem_u32(smem + lay.stage + st * lay.stage_bytes);
    if constexpr (FIRST) {
      uint64_t lo, hi;
      first_range(q, s, lo, hi);
      // a bulk copy starts and ends on 16-byte addresses: 8-byte records at the odd ends are
      // loaded by a thread
      uint64_t lo2, hi2;
      uint32_t soff;
      first_bulk(lo, hi, lo2, hi2, soff);
      const uint32_t bytes = hi2 > lo2 ? (uint32_t)((hi2 - lo2) * R) : 0u;
      mbar_expect_tx(bar, bytes);
      if (bytes) tma_load(dst + (uint32_t)((lo2 - lo + soff) * R), in_first + lo2, bytes, bar);
      trace_log<TRACE>(a.trace, kRead, kBufIn, (uint32_t)((hi - lo) * R), lo * R);
    } else {
      mbar_expect_tx(bar, ub * Z * (4 + R));
      for (uint32_t b = 0; b < ub; ++b) {
        const uint64_t bk = in_bucket(q, (s << lub) + b);
        tma_load(dst + b * Z * 4, a.in_tag + bk * Z, Z * 4, bar);
        tma_load(dst + ub * Z * 4 + b * Z * R, in_rec + bk * Z, Z * R, bar);
        trace_log<TRACE>(a.trace, kRead, a.buf_in_tag, Z * 4, bk * Z * 4);
        trace_log<TRACE>(a.trace, kRead, a.buf_in_rec, Z * R, bk * Z * R);
      }
    }
  };
  // f mod ring (f < 2^19, so f >> third < 2^16 and the multiply-shift divides by three exactly)
  auto ring_pos = [&](uint32_t f) -> uint32_t { return f - ring * (((f >> third) * 0xAAABu) >> 17); };

  // C: writes the chunks that the batch of buffer b completed, eight lanes to a chunk; the loads of
  // two chunks are in flight together.
  auto drain = [&](uint32_t b, Rec* orec, uint32_t* otag) {
    const uint32_t jj = lane & 7, n = worker ? ndone[b] : 0u;
    for (uint32_t x0 = tid >> 3; x0 < n; x0 += 2 * (kST / 8)) {
      uint32_t o[2], tg[2];
      Rec rc[2];
#pragma unroll
      for (uint32_t y = 0; y < 2; ++y) {
        const uint32_t x = x0 + y * (kST / 8);
        if (x < n) {
          const uint32_t e = done[x], u = e >> 8, c = e & 255u;
          const uint32_t pos = u * ring + ring_pos(c * kChunk) + jj;
          o[y] = u * Z + c * kChunk + jj;
          rc[y] = ring_rec[pos];
          tg[y] = ring_tag[pos];
        }
      }
#pragma unroll
      for (uint32_t y = 0; y < 2; ++y) {
        if (x0 + y * (kST / 8) < n) {
          orec[o[y]] = rc[y];
          otag[o[y]] = tg[y];
          if (jj == 0) {
            trace_log<TRACE>(a.trace, kWrite, a.buf_out_rec, kChunk * R, (uint64_t)((char*)(orec + o[y]) - (char*)a.out_rec));
            trace_log<TRACE>(a.trace, kWrite, a.buf_out_tag, kChunk * 4, (uint64_t)((char*)(otag + o[y]) - (char*)a.out_tag));
          }
        }
      }
    }
  };
  // Level counters (the last warp): lane l holds the sums over the digits 8l .. 8l + 7, so groups of
  // 2, 4 and 8 digits are summed in the lane, wider ones (held by all their lanes) by shuffles.
  // Level l = k - g: groups of 2^g digits; its blocks end after every 2^l input buckets, so levels
  // lub..e end with batch s.
  uint32_t* acc = reinterpret_cast<uint32_t*>(smem + lay.acc) + lane;  // [kAcc][32]
  if (!worker)
    for (uint32_t y = 0; y < kAcc; ++y) acc[y * 32] = 0;
  auto levels = [&](uint32_t b) {
    uint32_t v[8];
    const uint4* w = reinterpret_cast<const uint4*>(cf + b * D) + lane * 2;
    const uint4 none = make_uint4(0, 0, 0, 0), w0 = lane * 8 < D ? w[0] : none, w1 = lane * 8 < D ? w[1] : none;
    v[0] = w0.x & 4095u, v[1] = w0.y & 4095u, v[2] = w0.z & 4095u, v[3] = w0.w & 4095u;
    v[4] = w1.x & 4095u, v[5] = w1.y & 4095u, v[6] = w1.z & 4095u, v[7] = w1.w & 4095u;
#pragma unroll
    for (uint32_t y = 0; y < 4; ++y) acc[y * 32] += v[y] = v[2 * y] + v[2 * y + 1];
#pragma unroll
    for (uint32_t y = 0; y < 2; ++y) acc[(4 + y) * 32] += v[y] = v[2 * y] + v[2 * y + 1];
    acc[6 * 32] += v[0] += v[1];
#pragma unroll
    for (uint32_t y = 0; y < 4; ++y) {
      v[0] += __shfl_xor_sync(0xFFFFFFFFu, v[0], 1u << y);
      acc[(7 + y) * 32] += v[0];
    }
  };
  auto check = [&](uint32_t s) {
    const uint32_t e = __ffs(~s) - 1 + lub;
#pragma unroll
    for (uint32_t y = 0; y < kAcc; ++y) {
      const uint32_t gsz = y < 4 ? 1u : y < 6 ? 2u : y - 3;
      if (gsz >= k || k - gsz > e) continue;
      if (acc[y * 32] > Z && (lub < 2 || k - gsz > 1)) atomicExch(&a.ctrl->overflow, 1u);
      acc[y * 32] = 0;
    }
  };
  auto check1 = [&](uint32_t b) {  // level 1 of a batch of four buckets (a barrier after append comes first)
    if (!FIRST && lub == 2 && lane < 4) {
      if (lv1[b * 4 + lane] > Z) atomicExch(&a.ctrl->overflow, 1u);
      lv1[b * 4 + lane] = 0;
    }
  };

  if (tid == kST)  // the first nst batches (NB >= nst)
    for (uint32_t x = 0; x < nst && x < nbatch; ++x) issue(q0, x, x);

  // The dummy chunks of subproblem qq's buckets s*ub .. s*ub + ub - 1 (the last warp): bulk stores of
  // dummies from shared memory, to the records or the tags. They are issued with batch s of the
  // CTA's next subproblem, so the dummies, half of what a pass writes, leave evenly instead of in a
  // burst at a subproblem's end.
  auto write_tail = [&](uint64_t qq, uint32_t s, bool recs) {
    const uint32_t blk = recs ? kZeroRecs / R : kZeroTags / 4;  // slots per bulk store
    const uint32_t per = 32u >> lub, u = (s << lub) + lane / per;
    const uint64_t ob = (qq * D + u) * Z;
    for (uint32_t x = tail[u] + (lane & (per - 1)) * blk; x < Z; x += per * blk) {
      const uint32_t m = Z - x < blk ? Z - x : blk;
      if (recs)
        tma_store(reinterpret_cast<Rec*>(a.out_rec) + ob + x, smem_u32(smem + lay.zero), m * R);
      else
        tma_store(a.out_tag + ob + x, smem_u32(smem + lay.zero + kZeroRecs), m * 4);
      if (TRACE)
        for (uint32_t y = 0; y < m; y += kChunk)
          trace_log<TRACE>(a.trace, kWrite, recs ? a.buf_out_rec : a.buf_out_tag, kChunk * (recs ? R : 4),
                           (ob + x + y) * (recs ? R : 4));
    }
    tma_store_commit();
  };

  // One iteration per round: a round is a whole batch, or a part of one while a batch is redone.
  uint64_t q = q0;
  uint32_t g = 0, s = 0, st = 0, par = 0;  // batch g is batch s of subproblem q; its stage and the stage's parity
  uint32_t pb = 0;      // the round's buffer of lists, counts and fills
  uint32_t rlo = 0, sz = kWhole;  // the round's first slot and size
  bool pend = false;    // the previous round (buffer pb ^ 1) has not been drained yet
  Rec* orec = reinterpret_cast<Rec*>(a.out_rec) + q * D * Z;  // the subproblem's output buckets
  uint32_t* otag = a.out_tag + q * D * Z;
  while (nbatch) {
    if (pend) drain(pb ^ 1, orec, otag);
    if (s == NB) {
      // ---- end of the subproblem: the last partial chunk of every bucket padded with dummies; the
      // final loads are checked against Z ----
      for (uint32_t u = tid >> 3; u < D; u += kSThreads / 8) {
        const uint32_t f = cf[pb * D + u] >> 12, jj = lane & 7;
        uint32_t d = f / kChunk * kChunk;
        if (d < f && f < Z) {
          const bool real = d + jj < f;
          const uint32_t pos = u * ring + ring_pos(d) + jj, o = u * Z + d + jj;
          orec[o] = real ? ring_rec[pos] : RecT<R>::zero();
          otag[o] = real ? ring_tag[pos] : kDummy;
          if (jj == 0) {
            trace_log<TRACE>(a.trace, kWrite, a.buf_out_rec, kChunk * R, (uint64_t)((char*)(orec + o) - (char*)a.out_rec));
            trace_log<TRACE>(a.trace, kWrite, a.buf_out_tag, kChunk * 4, (uint64_t)((char*)(otag + o) - (char*)a.out_tag));
          }
          d += kChunk;
        }
        if (jj == 0) {
          if (f > Z) atomicExch(&a.ctrl->overflow, 1u);
          tail[u] = (uint16_t)(d < Z ? d : Z);
        }
      }
      __syncthreads();
      if (g == nbatch) break;
      if (tid < D) cf[tid] = cf[D + tid] = 0;
      clear_lists(pb ^ 1);
      pend = false;
      s = 0;
      q += qstep;
      orec += (uint64_t)qstep * D * Z;
      otag += (uint64_t)qstep * D * Z;
      __syncthreads();
    }
    unsigned char* stg = smem + lay.stage + st * lay.stage_bytes;
    const uint32_t* stag = reinterpret_cast<const uint32_t*>(stg);
    Rec* srec = reinterpret_cast<Rec*>(FIRST ? stg : stg + ub * Z * 4);
    uint32_t* cfp = cf + pb * D;
    uint16_t* listp = list + pb * kListWords;
    uint64_t lo = 0;
    uint32_t nslot = ub * Z, soff = 0;
    if constexpr (FIRST) {
      uint64_t hi;
      first_range(q, s, lo, hi);
      nslot = (uint32_t)(hi - lo);
      if (R == 8) {
        uint64_t lo2, hi2;
        first_bulk(lo, hi, lo2, hi2, soff);
        if (tid == kST - 1) {  // the records the bulk copy leaves out (odd ends)
          if (hi2 <= lo2) {  // at most two records, no bulk part
            for (uint32_t x = 0; x < nslot; ++x) srec[soff + x] = in_first[lo + x];
          } else {
            if (lo2 > lo) srec[soff] = in_first[lo];
            if (hi2 < hi) srec[soff + nslot - 1] = in_first[hi - 1];
          }
        }
      }
    } else {
      if (worker) mbar_wait(smem_u32(bars + st), par, a.ctrl);
    }
    const uint32_t rhi = rlo + sz < nslot ? rlo + sz : nslot;

    // item j of a thread: slot rlo + slot_of(j). In a middle pass the rows are shifted by half a
    // bucket from item to item (and a little more after every kSW rows), so that the rows of reals
    // at the front of the buckets, and the last, partly filled one of each, spread over the warps.
    auto slot_of = [&](uint32_t j) -> uint32_t {
      const uint32_t half = j * (Z / 64);
      return FIRST ? j * kST + tid : j * kST + ((((warp - half - 3 * (half / kSW)) & (kSW - 1)) << 5) | lane);
    };
    auto digit = [&](uint32_t tg) -> uint32_t { return (tg >> shift) & (D - 1); };
    uint32_t itg[kItems], ifl[kItems];  // tag, fill of its bucket before the round

    // ---- A: every real draws a place in its bucket's list; full: a list ran out of places ----
    bool full = false;
    if (worker) {
#pragma unroll
      for (uint32_t j = 0; j < kItems; ++j) {
        const uint32_t x = rlo + slot_of(j);
        itg[j] = kDummy;
        if (x < rhi) {
          if constexpr (FIRST)
            itg[j] = label_of(lo + x, a.seed, a.attempt, L);
          else
            itg[j] = stag[x];
        }
      }
#pragma unroll
      for (uint32_t j = 0; j < kItems; ++j)  // the atomics of a thread's items are in flight together
        if (itg[j] != kDummy) ifl[j] = atomicAdd(&cfp[digit(itg[j])], 1u);
#pragma unroll
      for (uint32_t j = 0; j < kItems; ++j)
        if (itg[j] != kDummy) {
          const uint32_t at = ifl[j] & 4095u;
          ifl[j] >>= 12;
          if (at < cap)
            listp[((at >> 3) * D + digit(itg[j])) * 8 + (at & 7)] = (uint16_t)(0x8000u | (rlo + slot_of(j)));
          else
            full = true;
        }
    } else if (g >= NB && sz == kWhole) {  // once per batch: a redone round never has this size
      write_tail(q - qstep, s, false);
    }
    if (__syncthreads_or(full)) {
      // a list ran out of places: again with half the slots (kSub at the least, which always fit)
      clear_lists(0);
      clear_lists(1);
      if (tid < D) cfp[tid] &= ~4095u;
      pend = false;  // the previous round was drained before the barrier
      sz = (rhi - rlo) / 2 > kSub ? (rhi - rlo) / 2 : kSub;
      __syncthreads();
      continue;
    }

    // ---- B: stable ranks, records into the rings, the completed chunks into the done list ----
    if constexpr (FIRST) mbar_wait(smem_u32(bars + st), par, a.ctrl);
    clear_lists(pb ^ 1);  // the previous round's: it was drained before the barrier
    if (worker) {
      if (tid < D) cf[(pb ^ 1) * D + tid] = ((cfp[tid] >> 12) + (cfp[tid] & 4095u)) << 12;
#pragma unroll
      for (uint32_t j = 0; j < kItems; ++j) {
        const uint32_t x = rlo + slot_of(j), u = digit(itg[j]);
        const bool real = itg[j] != kDummy;
        if (!__any_sync(0xFFFFFFFFu, real)) continue;  // a row of dummies
        if (!FIRST && lub == 2) {  // level 1 of a batch of four buckets: two blocks of two buckets
          const uint32_t cls = real ? (x >= 2 * Z ? 2u : 0u) + (u >> (k - 1)) : 4u;
#pragma unroll
          for (uint32_t y = 0; y < 4; ++y) {
            const uint32_t m = __ballot_sync(0xFFFFFFFFu, cls == y);
            if (lane == y && m) atomicAdd(&lv1[(g & 1) * 4 + y], __popc(m));
          }
        }
        bool last = false;  // this real completes a chunk
        uint32_t p = 0;
        if (real) {
          const uint32_t f = ifl[j], xx = x * 0x10001u;
          auto below = [&](const uint4& v) -> uint32_t {  // a half of v - xx has its top bit set iff its index >= x
            const uint32_t m = ((v.x - xx) & 0x80008000u) | (((v.y - xx) & 0x80008000u) >> 1) |
                               (((v.z - xx) & 0x80008000u) >> 2) | (((v.w - xx) & 0x80008000u) >> 3);
            return 8u - __popc(m);
          };
          const uint4* lp = reinterpret_cast<const uint4*>(listp) + u;
          const Rec rc = srec[soff + x];
          uint4 w = lp[0];
          uint32_t r = below(w);
#pragma unroll 1
          for (uint32_t e = 8; w.w < 0xFFFF0000u && e < cap; e += 8) {  // the eight places are all used
            w = *(lp += D);
            r += below(w);
          }
          p = f + r;
          last = (p & (kChunk - 1)) == kChunk - 1 && p < Z;  // at or past Z: the bucket overflowed
          uint32_t pos = ring_pos(f) + r;
          pos = u * ring + (pos >= ring ? pos - ring : pos);
          ring_rec[pos] = rc;
          ring_tag[pos] = itg[j];
        }
        const uint32_t m = __ballot_sync(0xFFFFFFFFu, last);
        if (m) {
          uint32_t at = 0;
          if (lane == 0) at = atomicAdd(&ndone[pb], __popc(m));
          at = __shfl_sync(0xFFFFFFFFu, at, 0) + __popc(m & lanemask_lt());
          if (last) done[at] = (uint16_t)(u << 8 | p / kChunk);
        }
      }
    } else {
      levels(pb);
      if (rhi == nslot) {
        check(s);
        if (g >= NB) write_tail(q - qstep, s, true);
      }
    }
    __syncthreads();
    pend = true;
    pb ^= 1;
    if (rhi < nslot) {  // the batch's next round, twice as large
      rlo = rhi;
      sz *= 2;
      continue;
    }
    // ---- the batch is done: its stage is free ----
    if (!worker) {
      if (lane == 0 && g + nst < nbatch) {
        const bool wrap = s + nst >= NB;
        issue(wrap ? q + qstep : q, wrap ? s + nst - NB : s + nst, st);
      }
      check1(g & 1);
    }
    ++g;
    ++s;
    rlo = 0;
    sz = kWhole;
    if (++st == nst) {
      st = 0;
      par ^= 1u;
    }
  }
  if (nbatch) {  // the last subproblem's dummies: all warps
    for (uint32_t x = warp; x < NB; x += kSThreads / 32) {
      write_tail(q, x, true);
      write_tail(q, x, false);
    }
    tma_store_wait_all();
  }
}

template <int R, bool FIRST, bool TRACE>
__global__ void __launch_bounds__(kSThreads, 1) orp_stream_kernel(const __grid_constant__ PassArgs a,
                                                                  const __grid_constant__ StreamLayout lay) {
  const uint64_t nsub = a.B >> a.k;
  if (blockIdx.x < nsub)
    orp_stream_body<R, FIRST, TRACE>(a, lay, blockIdx.x, (uint32_t)((nsub - 1 - blockIdx.x) / gridDim.x) + 1, gridDim.x);
}

// Many arrays: one CTA per unit.
template <int R, bool FIRST, bool TRACE>
__global__ void __launch_bounds__(kSThreads, 1) orp_stream_batched_kernel(const BatchStream* args, const uint2* units) {
  __shared__ BatchStream sa;
  const uint2 un = units[blockIdx.x];
  for (uint32_t x = threadIdx.x; x < sizeof(BatchStream) / 4; x += kSThreads)
    reinterpret_cast<uint32_t*>(&sa)[x] = reinterpret_cast<const uint32_t*>(args + un.x)[x];
  __syncthreads();
  orp_stream_body<R, FIRST, TRACE>(sa.a, sa.lay, un.y, 1, 1);
}

template <int R, bool FIRST, bool TRACE>
cudaError_t stream_batched(const BatchStream* args, const uint2* units, uint32_t nunits, uint32_t smem, cudaStream_t st) {
  auto kern = orp_stream_batched_kernel<R, FIRST, TRACE>;
  const cudaError_t e = set_smem_optin(kern);
  if (e != cudaSuccess) return e;
  kern<<<nunits, kSThreads, smem, st>>>(args, units);
  return cudaGetLastError();
}


template <int R, bool FIRST, bool TRACE>
cudaError_t stream_launch(const PassArgs& a, cudaStream_t st) {
  const StreamLayout lay = stream_layout(R, a.Z, a.k, FIRST);
  const uint32_t smem = lay.total;
  auto kern = orp_stream_kernel<R, FIRST, TRACE>;
  cudaError_t e = set_smem_optin(kern);
  if (e != cudaSuccess) return e;
  int per_sm = 0, sms = 0, dev = 0;
  if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kSThreads, smem)) != cudaSuccess) return e;
  if (per_sm <= 0) return cudaErrorInvalidConfiguration;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
  if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
  const uint64_t nsub = a.B >> a.k;
  uint64_t grid = (uint64_t)per_sm * sms;
  if (grid > nsub) grid = nsub;
  if (grid == 0) return cudaSuccess;
  kern<<<(unsigned)grid, kSThreads, smem, st>>>(a, lay);
  return cudaGetLastError();
}

}  // namespace

uint32_t orp_stream_max_k(int R, uint32_t Z, bool first, uint32_t smem_limit) {
  if (Z % 32 != 0 || Z > kMaxZ) return 0;
  uint32_t best = 0;
  for (uint32_t k = kMinK; k <= kMaxK; ++k)
    if (stream_layout(R, Z, k, first).total <= smem_limit) best = k;
  return best;
}

// Microseconds of one subproblem on one SM (fill: reals per slot): about 2.4 per batch of 1024 reals
// (n = 2^29, Z = 1024, k = 8: 128 batches in 300 us), 2.2 per batch of half as many (n = 2^20, Z = 512).
double orp_stream_sub_us(uint32_t Z, uint32_t k, bool first, double fill) {
  const uint32_t per = first ? Z / 2 : Z, most = first ? kBatchRecs : kBatchSlots;
  const uint32_t ub = per * 4 <= most ? 4u : per * 2 <= most ? 2u : 1u;
  return (double)(1u << k) / ub * (1.9 + 0.5 * ub * fill * Z / 1024.0) + 2.0;
}

StreamLayout orp_stream_layout(int R, uint32_t Z, uint32_t k, bool first) { return stream_layout(R, Z, k, first); }

cudaError_t launch_orp_stream_batched(const BatchStream* args, const uint2* units, uint32_t nunits, uint32_t smem,
                                      bool first, cudaStream_t st, int R, bool trace) {
  if (nunits == 0) return cudaSuccess;
  if (R == 8) {
    if (first) return trace ? stream_batched<8, true, true>(args, units, nunits, smem, st)
                            : stream_batched<8, true, false>(args, units, nunits, smem, st);
    return trace ? stream_batched<8, false, true>(args, units, nunits, smem, st)
                 : stream_batched<8, false, false>(args, units, nunits, smem, st);
  }
  if (first) return trace ? stream_batched<16, true, true>(args, units, nunits, smem, st)
                          : stream_batched<16, true, false>(args, units, nunits, smem, st);
  return trace ? stream_batched<16, false, true>(args, units, nunits, smem, st)
               : stream_batched<16, false, false>(args, units, nunits, smem, st);
}

cudaError_t launch_orp_stream(const PassArgs& a, bool first, cudaStream_t st, int R, bool trace) {
  if (a.k < kMinK || a.k > kMaxK || a.Z % 32 != 0 || a.Z > kMaxZ || a.i + a.k > a.L)
    return cudaErrorInvalidValue;
  if (R == 8) {
    if (first) return trace ? stream_launch<8, true, true>(a, st) : stream_launch<8, true, false>(a, st);
    return trace ? stream_launch<8, false, true>(a, st) : stream_launch<8, false, false>(a, st);
  }
  if (first) return trace ? stream_launch<16, true, true>(a, st) : stream_launch<16, true, false>(a, st);
  return trace ? stream_launch<16, false, true>(a, st) : stream_launch<16, false, false>(a, st);
}

}  // namespace bos
