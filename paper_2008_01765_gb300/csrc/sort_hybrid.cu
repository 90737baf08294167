// Hybrid radix sort of the ORP's output (Section 3.3: after the ORP, any non-oblivious sort). Its
// result is the stable sort by key of the ORP output, the same as the LSD radix sort's; it moves
// the records over HBM fewer times when the keys spread over the top digits.
//
//   1. histogram: one read of the keys gives the counts of every 8-bit digit and of the top two
//      digits together (65536 groups);
//   2. plan (one CTA): mode 1 when all n records fit one CTA's on-chip sort (kCap records); mode 2
//      when every value of the most significant varying digit dA holds at most kCap records;
//      mode 3 when dA and dB (the next varying digit) are the key's top two digits and every
//      (dA, dB) group holds at most kCap; otherwise mode 0, and the LSD passes run instead.
//      Consecutive groups are packed into ranges of whole groups, listed by size class;
//   3. modes 2, 3: a stable partition of the whole array by dA (the onesweep tile of the LSD pass);
//   4. mode 3: a stable partition by dB inside every dA bucket (tiles per bucket, the look-back
//      stopping at the bucket's first tile);
//   5. every range is sorted on chip by (key, position): a range of at most 256 records by one warp in
//      registers, a larger one by a CTA sized for it (bin_sort_kernel: its records in shared memory,
//      binned by key and ranked inside the bins); a range whose keys crowd a bin by
//      local_sort_kernel (partition, warp sorts or LSD passes).
// The partitions are stable and a range holds whole groups in key order, so sorting every range
// by key sorts the array; ties keep the ORP's order. HBM passes: the mode's count (1 to 3) plus
// the histogram, against 1 + the live digits for the LSD sort.
#include "common.cuh"
#include "internal.h"
#include "radix_tile.cuh"

namespace bos {

namespace {

constexpr int kJThreads = 1024;          // histogram CTA (one per SM: its shared memory holds the groups)
constexpr uint32_t kGroups = 65536;      // top two digits
constexpr int kPlanThreads = 1024;
constexpr int kLThreads = 512;           // local sort CTA
constexpr int kLWarps = kLThreads / 32;
constexpr uint32_t kLocalMaxCtas = 192;  // spill buffers in the workspace (one per CTA)
constexpr uint32_t kTagMsd1 = 12, kTagMsd2 = 13;
constexpr uint32_t kTicketMsd1 = 10, kTicketMsd2 = 11, kTicketLocal = 12;
constexpr uint32_t kWarpMax = 256;        // largest sub-bucket one warp sorts in registers (local_sort_kernel)
constexpr int kSThreads = 256;            // warp-per-range kernel
constexpr uint32_t kTicketClass = 13;     // .. 18: one per range class
// Range classes by size, each with its own list and launch: 0 one warp per range (registers); 1..4 the
// bin sort with the records in shared memory, 128 to 1024 threads (8, 4, 2 and 1 CTAs per SM); 5 the bin
// sort with the keys in shared memory (1024 threads).
constexpr uint32_t kClasses = kSortClasses, kMidClass = 3;
static_assert(kClasses == 6, "Bin<R, 0..5>");
constexpr uint32_t kFull = 20;            // a range with a fuller bin is sorted by LSD passes

constexpr uint32_t kMetaLeft = 3, kMetaList = 4;  // meta words: ranges left over; list starts [kClasses + 1]
template <int R, int CLS> struct Bin;
template <int R> struct Bin<R, 0> { static constexpr uint32_t kMax = 256; };
template <int R> struct Bin<R, 1> { static constexpr uint32_t kMax = 1056, kBits = 11; static constexpr int kT = 128, kCtas = 8; };
template <int R> struct Bin<R, 2> { static constexpr uint32_t kMax = 2112, kBits = 12; static constexpr int kT = 256, kCtas = 4; };
template <> struct Bin<16, 3> { static constexpr uint32_t kMax = 4352, kBits = 13; static constexpr int kT = 512, kCtas = 2; };
template <> struct Bin<8, 3> { static constexpr uint32_t kMax = 6656, kBits = 13; static constexpr int kT = 512, kCtas = 2; };
template <> struct Bin<16, 4> { static constexpr uint32_t kMax = 9216, kBits = 13; static constexpr int kT = 1024, kCtas = 1; };
template <> struct Bin<8, 4> { static constexpr uint32_t kMax = 14848, kBits = 13; static constexpr int kT = 1024, kCtas = 1; };

template <int R> struct Local;
template <> struct Local<16> { static constexpr uint32_t kCap = 19456; };  // 10 B per record on chip
template <> struct Local<8> { static constexpr uint32_t kCap = 28672; };   // 6 B per record on chip
template <int R> struct Bin<R, 5> { static constexpr uint32_t kMax = Local<R>::kCap, kBits = 13; static constexpr int kT = 1024, kCtas = 1; };

__host__ __device__ constexpr uint32_t al16(uint32_t x) { return (x + 15u) & ~15u; }

// Shared memory of the local sort: keys [kCap], positions (u16) [kCap], two per-warp digit count
// tables [2][kLWarps][257], the count scan's scratch [512 + 8], the key AND/OR of every warp, misc
// [4], the sub-bucket starts [257].
template <int R>
__host__ __device__ constexpr uint32_t local_smem_bytes() {
  using Key = typename RecT<R>::Key;
  return al16(Local<R>::kCap * (uint32_t)(sizeof(Key) + 2)) + 2 * kLWarps * 257 * 4 + (512 + 8) * 4 +
         2 * kLWarps * (uint32_t)sizeof(Key) + 16 + 257 * 4;
}
static_assert(local_smem_bytes<16>() <= 232448 - 1024, "local sort shared memory");
static_assert(local_smem_bytes<8>() <= 232448 - 1024, "local sort shared memory");

template <int R>
__device__ __forceinline__ typename RecT<R>::T* sort_buf(const HybridArgs& a, uint32_t passes, uint32_t j) {
  // buffer chain of the sort: X_passes = output, alternating backwards (X_0 is the ORP's target)
  return reinterpret_cast<typename RecT<R>::T*>(((passes - j) & 1u) ? a.buf1 : a.buf0);
}

// Key of record p (its first key_bytes bytes, little-endian), read without the payload.
template <int R>
__device__ __forceinline__ typename RecT<R>::Key load_key(const typename RecT<R>::T* p) {
  return *reinterpret_cast<const typename RecT<R>::Key*>(p);
}

// ---- 1. histogram ---------------------------------------------------------------------------

// The group counters are 16 bits, two to a shared-memory word; an increment that takes one to
// 2^15 moves 2^15 to the group's global counter, so a half never carries into its neighbour.
template <int R>
__device__ __forceinline__ void count_key(typename RecT<R>::Key key, uint32_t* h, uint32_t* jp, uint32_t* joint) {
  constexpr int D = RecT<R>::kDigits;
#pragma unroll
  for (int d = 0; d < D; ++d) atomicAdd(&h[d * 256 + (uint32_t)((key >> (8 * d)) & 255u)], 1u);
  const uint32_t g = (uint32_t)(key >> (8 * (D - 2))) & 0xFFFFu;
  const uint32_t sh = (g & 1u) << 4;
  const uint32_t old = atomicAdd(&jp[g >> 1], 1u << sh);
  if (((old >> sh) & 0xFFFFu) == 0x7FFFu) {
    atomicSub(&jp[g >> 1], 0x8000u << sh);
    atomicAdd(joint + g, 0x8000u);
  }
}

template <int R>
__global__ void __launch_bounds__(kJThreads, 1) hybrid_hist_kernel(HybridArgs a) {
  using Rec = typename RecT<R>::T;
  using Key = typename RecT<R>::Key;
  constexpr int D = RecT<R>::kDigits;
  extern __shared__ __align__(16) uint32_t hsm[];
  uint32_t* h = hsm;             // [D][256]
  uint32_t* jp = hsm + D * 256;  // [kGroups / 2]
  for (uint32_t x = threadIdx.x; x < D * 256 + kGroups / 2; x += kJThreads) hsm[x] = 0;
  __syncthreads();
  const Rec* in = reinterpret_cast<const Rec*>(a.in);
  const uint64_t step = (uint64_t)gridDim.x * kJThreads;
  uint64_t idx = (uint64_t)blockIdx.x * kJThreads + threadIdx.x;
  for (; idx + 3 * step < a.n; idx += 4 * step) {  // four loads in flight per thread
    Key k[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) k[u] = load_key<R>(in + idx + u * step);
#pragma unroll
    for (int u = 0; u < 4; ++u) count_key<R>(k[u], h, jp, a.joint);
  }
  for (; idx < a.n; idx += step) count_key<R>(load_key<R>(in + idx), h, jp, a.joint);
  __syncthreads();
  for (uint32_t x = threadIdx.x; x < D * 256; x += kJThreads)
    if (h[x]) atomicAdd(a.hist + x, h[x]);
  for (uint32_t w = threadIdx.x; w < kGroups / 2; w += kJThreads) {
    const uint32_t v = jp[w];
    if (v & 0xFFFFu) atomicAdd(a.joint + 2 * w, v & 0xFFFFu);
    if (v >> 16) atomicAdd(a.joint + 2 * w + 1, v >> 16);
  }
}

// ---- 2. plan --------------------------------------------------------------------------------

// Exclusive scan of one value per thread over the CTA (kPlanThreads threads); *total gets the sum.
__device__ __forceinline__ unsigned long long plan_scan(unsigned long long v, unsigned long long* s_w,
                                                        unsigned long long* total) {
  const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
  unsigned long long incl = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned long long y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
    if (lane >= (uint32_t)o) incl += y;
  }
  if (lane == 31) s_w[warp] = incl;
  __syncthreads();
  if (warp == 0) {
    unsigned long long t = s_w[lane];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned long long y = __shfl_up_sync(0xFFFFFFFFu, t, o);
      if (lane >= (uint32_t)o) t += y;
    }
    s_w[lane] = t;
  }
  __syncthreads();
  const unsigned long long ex = incl - v + (warp ? s_w[warp - 1] : 0ull);
  *total = s_w[31];
  __syncthreads();
  return ex;
}

// The plan for the host, which launches only the kernels that it calls for: the words, then the
// sequence number the host waits for.
__device__ void publish_plan(HostPlan* h, uint32_t seq, uint32_t mode, uint32_t live, const uint32_t* list) {
  if (!h) return;
  volatile HostPlan* v = h;
  v->mode = mode;
  v->live = live;
  for (uint32_t y = 0; y < kClasses; ++y) v->list[y] = list ? list[y] : 0u;
  __threadfence_system();
  v->seq = seq;
}

template <int R>
__global__ void __launch_bounds__(kPlanThreads) sort_plan_kernel(HybridArgs a) {
  constexpr int D = RecT<R>::kDigits;
  constexpr uint32_t kCap = Local<R>::kCap;
  __shared__ uint32_t s_max[8], s_jmax, s_live, s_mode, s_dA, s_dB;
  __shared__ uint32_t s_list[kClasses];
  __shared__ unsigned long long s_w[32];
  const uint32_t tid = threadIdx.x;
  if (tid < 8) s_max[tid] = 0;
  if (tid == 0) s_jmax = s_live = 0;
  __syncthreads();
  // every digit's exclusive offsets, its fullest value, and whether it varies (1024 threads: four
  // digits at a time, eight warps each)
  for (uint32_t x0 = 0; x0 < D * 256; x0 += kPlanThreads) {
    const uint32_t x = x0 + tid, lane = tid & 31u, warp = tid >> 5;
    const uint32_t c = a.hist[x];
    uint32_t incl = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
      if (lane >= (uint32_t)o) incl += y;
    }
    if (lane == 31) s_w[warp] = incl;
    const uint32_t mx = __reduce_max_sync(0xFFFFFFFFu, c);
    if (lane == 0) atomicMax(&s_max[x >> 8], mx);
    __syncthreads();
    uint32_t before = 0;
    for (uint32_t w = warp & ~7u; w < warp; ++w) before += (uint32_t)s_w[w];
    a.dbase[x] = before + incl - c;
    __syncthreads();
  }
  if (tid < D && (uint64_t)s_max[tid] < a.n) atomicOr(&s_live, 1u << tid);
  uint32_t jm = 0;
  for (uint32_t x = tid; x < kGroups; x += kPlanThreads) jm = a.joint[x] > jm ? a.joint[x] : jm;
  atomicMax(&s_jmax, jm);
  __syncthreads();
  if (tid == 0) {
    int dA = -1, dB = -1;
    for (int d = D - 1; d >= 0; --d)
      if ((uint64_t)s_max[d] < a.n) {  // some key differs in digit d
        if (dA < 0) dA = d;
        else if (dB < 0) dB = d;
      }
    uint32_t mode = 0;
    if (a.n >= 2 && dA >= 0) {
      if (a.n <= kCap) mode = 1;
      else if (s_max[dA] <= kCap) mode = 2;
      else if (dA == D - 1 && dB == D - 2 && s_jmax <= kCap) mode = 3;
    }
    s_mode = mode;
    s_dA = dA < 0 ? 0u : (uint32_t)dA;
    s_dB = dB < 0 ? 0u : (uint32_t)dB;
    a.meta[0] = mode;
    a.meta[1] = s_dA;
    a.meta[2] = s_dB;
    a.ctrl->radix_live = s_live;
  }
  __syncthreads();
  const uint32_t mode = s_mode, dA = s_dA;
  if (mode == 0) {
    if (tid == 0) {
      a.ctrl->sort_mode = 0;
      publish_plan(a.host, a.host_seq, 0, s_live, nullptr);
    }
    return;
  }
  // groups: the whole array (mode 1), the values of dA (mode 2), the (dA, dB) pairs (mode 3)
  const uint32_t G = mode == 1 ? 1u : mode == 2 ? 256u : kGroups;
  const uint64_t gmax = mode == 1 ? a.n : mode == 2 ? s_max[dA] : s_jmax;
  auto count = [&](uint32_t g) -> uint64_t {
    return mode == 1 ? a.n : mode == 2 ? (uint64_t)a.hist[dA * 256 + g] : (uint64_t)a.joint[g];
  };
  // Ranges of whole groups. Groups that are large for a packed range get one each (with the empty
  // groups after it); smaller ones are packed: a range is a run of consecutive groups whose starts
  // fall in one window of S records (at most S - 1 + gmax <= P records). P gives every SM two ranges
  // where n allows it, within the sizes of classes 1 to 3.
  const uint32_t want = (uint32_t)(a.n / 304);
  constexpr uint32_t kPmin = Bin<R, 1>::kMax, kPmax = Bin<R, kMidClass>::kMax;
  const uint32_t P = want < kPmin ? kPmin : want < kPmax ? want : kPmax;
  const bool single = gmax * 3 > P;
  const uint32_t S = single ? 1u : P - (uint32_t)gmax + 1u;
  auto starts = [&](uint32_t g, uint64_t gs) -> bool {  // gs < 2^31
    if (g == 0) return true;
    if (single) return count(g) > 0;
    return (uint32_t)gs / S != (uint32_t)(gs - count(g - 1)) / S;
  };
  // Warp w takes the groups (later the ranges) [w per, (w + 1) per), 32 consecutive ones at a time: two
  // passes over the groups (sums and range counts need the sums of the warps before), two over the
  // ranges, every access coalesced. (One thread per 64 groups, as before: 0.37 ms in mode 3.)
  const uint32_t lane = tid & 31u, warp = tid >> 5;
  constexpr uint32_t kPW = kPlanThreads / 32;
  const uint32_t per = ((G + kPW - 1) / kPW + 31u) & ~31u;
  const uint32_t g0 = warp * per < G ? warp * per : G, g1 = g0 + per < G ? g0 + per : G;
  unsigned long long sum = 0, total = 0;
#pragma unroll 4
  for (uint32_t g = g0 + lane; g < g1; g += 32) sum += count(g);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xFFFFFFFFu, sum, o);
  const unsigned long long ex = __shfl_sync(0xFFFFFFFFu, plan_scan(lane == 0 ? sum : 0ull, s_w, &total), 0);
  unsigned long long run = ex;
  uint32_t nr = 0;
  auto walk = [&](auto&& each) {  // each(group, its start, is it a range's first group, lanes that are)
    run = ex;
    for (uint32_t b = g0; b < g1; b += 32) {
      const uint32_t g = b + lane;
      const uint32_t c = g < g1 ? (uint32_t)count(g) : 0u;
      uint32_t incl = c;  // 32 groups of at most kCap records: 32 bits
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
        if (lane >= (uint32_t)o) incl += y;
      }
      const unsigned long long gs = run + incl - c;
      const bool st = g < g1 && starts(g, gs);
      each(g, gs, st, __ballot_sync(0xFFFFFFFFu, st));
      run += __shfl_sync(0xFFFFFFFFu, incl, 31);
    }
  };
  walk([&](uint32_t g, unsigned long long gs, bool, uint32_t firsts) {
    if (g < g1) a.gstart[g] = gs;
    nr += __popc(firsts);
  });
  if (tid == 0) a.gstart[G] = total;
  unsigned long long nranges = 0;
  uint32_t rx = (uint32_t)__shfl_sync(0xFFFFFFFFu, plan_scan(lane == 0 ? nr : 0ull, s_w, &nranges), 0);
  walk([&](uint32_t g, unsigned long long, bool st, uint32_t firsts) {
    if (st) a.rlist[rx + __popc(firsts & lanemask_lt())] = g;
    rx += __popc(firsts);
  });
  if (tid == 0) a.rlist[nranges] = G;
  __syncthreads();  // the range list and the group starts are written
  {  // the ranges by class, one list after the other
    const uint32_t NR = (uint32_t)nranges, rper = ((NR + kPW - 1) / kPW + 31u) & ~31u;
    const uint32_t r0 = warp * rper < NR ? warp * rper : NR, r1 = r0 + rper < NR ? r0 + rper : NR;
    auto cls = [&](uint32_t r) -> uint32_t {
      const unsigned long long m = a.gstart[a.rlist[r + 1]] - a.gstart[a.rlist[r]];
      return m <= Bin<R, 0>::kMax ? 0u : m <= Bin<R, 1>::kMax ? 1u : m <= Bin<R, 2>::kMax ? 2u
             : m <= Bin<R, 3>::kMax ? 3u : m <= Bin<R, 4>::kMax ? 4u : 5u;
    };
    uint32_t nc[kClasses] = {0, 0, 0, 0, 0, 0}, at[kClasses], list = 0;
#pragma unroll 4
    for (uint32_t r = r0 + lane; r < r1; r += 32) {
      const uint32_t c = cls(r);
#pragma unroll
      for (uint32_t y = 0; y < kClasses; ++y) nc[y] += c == y ? 1u : 0u;
    }
#pragma unroll
    for (uint32_t y = 0; y < kClasses; ++y) {
      unsigned long long tot = 0;
      const uint32_t w = __reduce_add_sync(0xFFFFFFFFu, nc[y]);
      at[y] = list + (uint32_t)__shfl_sync(0xFFFFFFFFu, plan_scan(lane == 0 ? w : 0ull, s_w, &tot), 0);
      if (tid == 0) {
        a.meta[kMetaList + y] = list;
        s_list[y] = (uint32_t)tot;
      }
      list += (uint32_t)tot;
    }
    if (tid == 0) {
      a.meta[kMetaList + kClasses] = list;
      a.meta[kMetaLeft] = 0;  // ranges left to local_sort_kernel, listed in a.joint (dead after the plan)
    }
#pragma unroll 2
    for (uint32_t b = r0; b < r1; b += 32) {
      const uint32_t r = b + lane, c = r < r1 ? cls(r) : kClasses;
#pragma unroll
      for (uint32_t y = 0; y < kClasses; ++y) {
        const uint32_t m = __ballot_sync(0xFFFFFFFFu, c == y);
        if (c == y) a.ridx[at[y] + __popc(m & lanemask_lt())] = r;
        at[y] += __popc(m);
      }
    }
  }
  if (mode == 3) {  // MSD2 tiles: every dA bucket is cut into tiles of its own
    const uint64_t tb = tid < 256 ? ((uint64_t)a.hist[dA * 256 + tid] + kTile - 1) / kTile : 0ull;
    unsigned long long ttot = 0;
    const unsigned long long tx = plan_scan(tb, s_w, &ttot);
    if (tid < 256) a.first[tid] = tx;
    if (tid == 0) a.first[256] = ttot;
  }
  __syncthreads();
  if (tid == 0) {
    a.ctrl->sort_mode = mode;
    publish_plan(a.host, a.host_seq, mode, s_live, s_list);
  }
}

// ---- 3, 4. MSD partitions ---------------------------------------------------------------------
// Persistent, like the LSD pass: CTAs take tiles by ticket, so a launch whose mode does not run
// it (the host did not learn the mode in time) costs one early return per CTA.

template <int R>
__global__ void __launch_bounds__(kTileThreads, 2) msd1_kernel(HybridArgs a) {
  const uint32_t mode = a.ctrl->sort_mode;
  if (mode < 2) return;
  __shared__ unsigned long long t_s;
  const uint32_t dA = a.meta[1];
  const uint64_t tiles = (a.n + kTile - 1) / kTile;
  while (true) {
    if (threadIdx.x == 0) t_s = atomicAdd(&a.ctrl->tickets[kTicketMsd1], 1u);
    __syncthreads();
    const unsigned long long t = t_s;
    if (t >= tiles) break;
    radix_tile<R>(sort_buf<R>(a, mode, 0), sort_buf<R>(a, mode, 1), a.n, t, 8 * dA, kTagMsd1, a.status,
                  a.dbase + dA * 256, a.n, a.ctrl);
    __syncthreads();
  }
}

template <int R>
__global__ void __launch_bounds__(kTileThreads, 2) msd2_kernel(HybridArgs a) {
  if (a.ctrl->sort_mode != 3) return;
  __shared__ unsigned long long t_s;
  __shared__ uint32_t b_s;
  const uint32_t dA = a.meta[1], dB = a.meta[2];
  const unsigned long long tiles = a.first[256];
  while (true) {
    if (threadIdx.x == 0) {
      const unsigned long long t = atomicAdd(&a.ctrl->tickets[kTicketMsd2], 1u);
      uint32_t lo = 0, hi = 256;  // the dA bucket of tile t: the last b with first[b] <= t
      while (hi - lo > 1) {
        const uint32_t mid = (lo + hi) >> 1;
        if (a.first[mid] <= t) lo = mid; else hi = mid;
      }
      t_s = t;
      b_s = lo;
    }
    __syncthreads();
    const unsigned long long t = t_s;
    if (t >= tiles) break;
    const uint32_t b = b_s;
    const uint64_t lo = a.dbase[dA * 256 + b];
    const uint64_t nb = a.hist[dA * 256 + b];
    // group (b, v) starts at gstart[b * 256 + v]: the absolute base of digit value v in this bucket
    radix_tile<R>(sort_buf<R>(a, 3, 1) + lo, sort_buf<R>(a, 3, 2), nb, t - a.first[b], 8 * dB, kTagMsd2,
                  a.status + a.first[b] * 256, a.gstart + b * 256, a.n, a.ctrl);
    __syncthreads();
  }
}

// ---- 5. on-chip sort of every range ----------------------------------------------------------

// Per-warp counts -> per-warp output starts, in place: wc[w][v] becomes the position of warp w's
// first item with digit value v (all items of smaller values first, then those of earlier warps).
__device__ __forceinline__ void local_scan(uint32_t* wc, uint32_t* half, uint32_t* wsum) {
  const uint32_t tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5;
  const uint32_t v = tid & 255u, h = tid >> 8;  // thread (h, v) covers warps 8h .. 8h+7
  uint32_t s = 0;
#pragma unroll
  for (int j = 0; j < 8; ++j) s += wc[(h * 8 + j) * 257 + v];
  half[h * 256 + v] = s;
  __syncthreads();
  const uint32_t tot = half[v] + half[256 + v];
  uint32_t incl = tot;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
    if (lane >= (uint32_t)o) incl += y;
  }
  if (h == 0 && lane == 31) wsum[warp] = incl;
  __syncthreads();
  uint32_t run = incl - tot + (h ? half[v] : 0u);
  for (uint32_t w = 0; w < (warp & 7u); ++w) run += wsum[w];
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const uint32_t x = wc[(h * 8 + j) * 257 + v];
    wc[(h * 8 + j) * 257 + v] = run;
    run += x;
  }
  __syncthreads();
}

// Ascending bitonic sort of the s <= 32 * EPL words at base, in registers: lane l holds elements
// l * EPL .. l * EPL + EPL - 1, so the stages with partner distance below EPL stay in registers.
// Positions past s hold the largest word, which no entry equals (entries are distinct).
template <typename W, int EPL>
__device__ __forceinline__ void warp_sort(W* base, uint32_t s, uint32_t lane) {
  W v[EPL];
#pragma unroll
  for (int r = 0; r < EPL; ++r) {
    const uint32_t e = lane * EPL + r;
    v[r] = e < s ? base[e] : ~W(0);
  }
#pragma unroll
  for (int kk = 2; kk <= 32 * EPL; kk <<= 1) {
#pragma unroll
    for (int j = kk >> 1; j > 0; j >>= 1) {
      if (j < EPL) {  // partners in the same lane: elements r and r ^ j
#pragma unroll
        for (int r = 0; r < EPL; ++r) {
          if ((r & j) == 0) {
            const bool up = ((lane * EPL + (uint32_t)r) & (uint32_t)kk) == 0;
            const W x = v[r], y = v[r | j];
            const bool sw = (y < x) == up;
            v[r] = sw ? y : x;
            v[r | j] = sw ? x : y;
          }
        }
      } else {  // partners in lane ^ (j / EPL), same r
        const uint32_t lj = (uint32_t)j / EPL;
#pragma unroll
        for (int r = 0; r < EPL; ++r) {
          const W o = __shfl_xor_sync(0xFFFFFFFFu, v[r], lj);
          const bool up = ((lane * EPL + (uint32_t)r) & (uint32_t)kk) == 0;
          const bool keep_min = ((lane & lj) == 0) == up;
          if ((o < v[r]) == keep_min) v[r] = o;
        }
      }
    }
  }
#pragma unroll
  for (int r = 0; r < EPL; ++r) {
    const uint32_t e = lane * EPL + r;
    if (e < s) base[e] = v[r];
  }
}

// Lanes of the warp with this lane's digit value (0..255, or 256 = no item). A full row of the
// warp has no empty lane, so eight ballots decide it.
__device__ __forceinline__ uint32_t row_peers(uint32_t dg, bool full) {
  return full ? ballot_peers(dg, 8) : ballot_peers(dg, 9);
}

// Per-warp counts of digit d of the keys at positions [wlo, whi) (shared-memory atomics on the warp's
// own counters: counts need no ranks).
template <int R>
__device__ __forceinline__ void local_count(const typename RecT<R>::T* in, uint32_t* wc, uint32_t d, uint32_t wlo,
                                            uint32_t whi, uint32_t lane, uint32_t warp) {
  for (uint32_t b = wlo; b < whi; b += 32) {
    const uint32_t j = b + lane;
    const bool valid = j < whi;
    if (valid) atomicAdd(&wc[warp * 257 + (uint32_t)((load_key<R>(in + j) >> (8 * d)) & 255u)], 1u);
  }
}

// One range of at most kCap records, sorted by key (stable). Fast form: one stable partition of
// the range by its most significant varying digit dC into shared memory, each entry packed as
// (key bits below dC, position) in one key-sized word, then every sub-bucket (at most 256
// entries) sorted by a warp in registers; the packed words are distinct, so that order is the
// stable one. Otherwise (the packed word would not fit, or a sub-bucket is larger): LSD passes
// over the varying digits, alternating between shared memory and the CTA's spill buffers.
template <int R>
__global__ void __launch_bounds__(kLThreads, 1) local_sort_kernel(HybridArgs a) {
  using Rec = typename RecT<R>::T;
  using Key = typename RecT<R>::Key;
  constexpr int D = RecT<R>::kDigits;
  constexpr uint32_t kCap = Local<R>::kCap;
  constexpr uint32_t kU = 8;  // rows of a warp whose loads are in flight together
  const uint32_t mode = a.ctrl->sort_mode;
  if (mode == 0) return;
  extern __shared__ __align__(16) unsigned char lsm[];
  Key* SK = reinterpret_cast<Key*>(lsm);
  uint16_t* SI = reinterpret_cast<uint16_t*>(lsm + kCap * sizeof(Key));
  uint32_t* WC = reinterpret_cast<uint32_t*>(lsm + al16(kCap * (uint32_t)(sizeof(Key) + 2)));
  uint32_t* half = WC + 2 * kLWarps * 257;
  uint32_t* wsum = half + 512;
  Key* red = reinterpret_cast<Key*>(wsum + 8);
  uint32_t* misc = reinterpret_cast<uint32_t*>(red + 2 * kLWarps);
  uint32_t* sub = misc + 4;
  // this CTA's spill buffers: the even LSD passes write them (they stay in L2 for the next pass)
  Key* GK = reinterpret_cast<Key*>(a.scratch + (size_t)blockIdx.x * kCap * (sizeof(Key) + 2));
  uint16_t* GI = reinterpret_cast<uint16_t*>(GK + kCap);
  const Rec* src = sort_buf<R>(a, mode, mode - 1);
  Rec* dst = sort_buf<R>(a, mode, mode);
  const uint32_t tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5;
  const uint32_t lt_mask = lanemask_lt();
  const uint32_t nbig = a.meta[kMetaLeft];  // this kernel's ranges: those the bin sort left (a bin too full)
  // the digit read 1 counts: the top varying digit of a one-group range under this mode
  const uint32_t dspec = mode == 3 ? D - 3 : mode == 2 ? D - 2 : D - 1;

  while (true) {
    if (tid == 0) misc[0] = atomicAdd(&a.ctrl->tickets[kTicketLocal], 1u);
    __syncthreads();
    const uint32_t ti = misc[0];
    if (ti >= nbig) break;
    const uint32_t r = a.joint[ti];
    const uint64_t lo = a.gstart[a.rlist[r]];
    const uint64_t m64 = a.gstart[a.rlist[r + 1]] - lo;
    if (m64 == 0 || m64 > kCap) {  // empty; or more than the plan allows (never: the counts bound it)
      if (m64 > kCap && tid == 0) atomicExch(&a.ctrl->bad, 1u);
      __syncthreads();
      continue;
    }
    const uint32_t m = (uint32_t)m64;
    const Rec* in = src + lo;
    Rec* out = dst + lo;
    // warp w orders the positions [w c, (w+1) c) of the current order, c a multiple of 32
    const uint32_t c = ((m + kLWarps - 1) / kLWarps + 31u) & ~31u;
    const uint32_t cmagic = 0xFFFFFFFFu / c + 1u;  // __umulhi(pos, cmagic) = pos / c for pos < 2^16
    const uint32_t wlo = warp * c < m ? warp * c : m, whi = wlo + c < m ? wlo + c : m;
    uint32_t* wc = WC;
    uint32_t* wn = WC + kLWarps * 257;
    for (uint32_t x = tid; x < kLWarps * 257; x += kLThreads) wc[x] = 0;
    __syncthreads();
    // read 1: the key AND / OR over the range, and each warp's counts of digit dspec
    Key kand = ~Key(0), kor = Key(0);
    for (uint32_t b0 = wlo; b0 < whi; b0 += 32 * kU) {
      Key kk[kU];
#pragma unroll
      for (uint32_t u = 0; u < kU; ++u) {
        const uint32_t j = b0 + u * 32 + lane;
        kk[u] = j < whi ? load_key<R>(in + j) : Key(0);
      }
#pragma unroll
      for (uint32_t u = 0; u < kU; ++u) {
        if (b0 + u * 32 >= whi) break;
        const uint32_t j = b0 + u * 32 + lane;
        const bool valid = j < whi;
        if (valid) {
          kand &= kk[u];
          kor |= kk[u];
        }
        // counts only (no ranks): one shared-memory atomic per key on the warp's own counters
        if (valid) atomicAdd(&wc[warp * 257 + (uint32_t)((kk[u] >> (8 * dspec)) & 255u)], 1u);
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      kand &= __shfl_xor_sync(0xFFFFFFFFu, kand, o);
      kor |= __shfl_xor_sync(0xFFFFFFFFu, kor, o);
    }
    if (lane == 0) {
      red[warp] = kand;
      red[kLWarps + warp] = kor;
    }
    __syncthreads();
    Key band = ~Key(0), bor = Key(0);
    for (int w = 0; w < kLWarps; ++w) {
      band &= red[w];
      bor |= red[kLWarps + w];
    }
    const Key vary = band ^ bor;
    uint32_t vm = 0;  // digits that vary inside the range
#pragma unroll
    for (int d = 0; d < D; ++d)
      if ((vary >> (8 * d)) & 255u) vm |= 1u << d;
    if (vm == 0) {  // every key equal: the range is already in order
      for (uint32_t j0 = tid; j0 < m; j0 += 4 * kLThreads) {
        Rec v[4];
#pragma unroll
        for (uint32_t u = 0; u < 4; ++u)
          if (j0 + u * kLThreads < m) v[u] = in[j0 + u * kLThreads];
#pragma unroll
        for (uint32_t u = 0; u < 4; ++u)
          if (j0 + u * kLThreads < m) out[j0 + u * kLThreads] = v[u];
      }
      __syncthreads();
      continue;
    }
    uint32_t counted = dspec;  // the digit wc holds counts of
    const uint32_t dC = 31u - (uint32_t)__clz(vm);
    bool fast = 8 * dC + 16 <= 8 * sizeof(Key);
    if (fast) {
      if (dC != counted) {
        for (uint32_t x = tid; x < kLWarps * 257; x += kLThreads) wc[x] = 0;
        __syncthreads();
        local_count<R>(in, wc, dC, wlo, whi, lane, warp);
        __syncthreads();
        counted = dC;
      }
      local_scan(wc, half, wsum);
      // sub-bucket v = [sub[v], sub[v + 1]): warp 0's start of digit value v
      if (tid < 256) sub[tid] = wc[tid];
      if (tid == 0) sub[256] = m;
      const uint32_t tot = tid < 256 ? half[tid] + half[256 + tid] : 0u;
      fast = !__syncthreads_or(tot > kWarpMax);
      counted = 0xFFFFFFFFu;  // wc now holds starts, not counts
    }
    if (fast) {
      // stable partition by dC from the records (the shared keys are overwritten by the packed
      // words): word = (key bits below dC) << 16 | position
      const Key low = (Key)((((unsigned long long)1) << (8 * dC)) - 1ull);
      for (uint32_t b0 = wlo; b0 < whi; b0 += 32 * kU) {
        Key kk[kU];
#pragma unroll
        for (uint32_t u = 0; u < kU; ++u) {
          const uint32_t j = b0 + u * 32 + lane;
          kk[u] = j < whi ? load_key<R>(in + j) : Key(0);
        }
#pragma unroll
        for (uint32_t u = 0; u < kU; ++u) {
          if (b0 + u * 32 >= whi) break;
          const uint32_t j = b0 + u * 32 + lane;
          const bool valid = j < whi;
          const uint32_t dg = valid ? (uint32_t)((kk[u] >> (8 * dC)) & 255u) : 256u;
          const uint32_t peers = row_peers(dg, b0 + u * 32 + 32 <= whi);
          const uint32_t lt = __popc(peers & lt_mask);
          const uint32_t base = wc[warp * 257 + dg];
          __syncwarp();
          if (valid && lt == 0) wc[warp * 257 + dg] = base + __popc(peers);
          __syncwarp();
          if (valid) SK[base + lt] = ((kk[u] & low) << 16) | (Key)j;
        }
      }
      if (tid == 0) misc[1] = 0;
      __syncthreads();
      while (true) {  // warps take sub-buckets as they free up (their sizes differ)
        uint32_t v = 0;
        if (lane == 0) v = atomicAdd(&misc[1], 1u);
        v = __shfl_sync(0xFFFFFFFFu, v, 0);
        if (v >= 256) break;
        const uint32_t s0 = sub[v], sz = sub[v + 1] - s0;
        if (sz <= 1) continue;
        if (sz <= 32) warp_sort<Key, 1>(SK + s0, sz, lane);
        else if (sz <= 64) warp_sort<Key, 2>(SK + s0, sz, lane);
        else if (sz <= 128) warp_sort<Key, 4>(SK + s0, sz, lane);
        else warp_sort<Key, 8>(SK + s0, sz, lane);
      }
      __syncthreads();
      for (uint32_t j0 = tid; j0 < m; j0 += 4 * kLThreads) {
        Rec v[4];
#pragma unroll
        for (uint32_t u = 0; u < 4; ++u)
          if (j0 + u * kLThreads < m) v[u] = in[(uint32_t)(SK[j0 + u * kLThreads] & 0xFFFFu)];
#pragma unroll
        for (uint32_t u = 0; u < 4; ++u)
          if (j0 + u * kLThreads < m) out[j0 + u * kLThreads] = v[u];
      }
      __syncthreads();
      continue;
    }
    // LSD passes over the varying digits. Pass q moves (key, position) from the shared buffers to
    // the spill buffers (q even) or back (q odd), stably by digit d, and counts the next digit for
    // the warp that will read each position.
    for (uint32_t j = tid; j < m; j += kLThreads) {  // keys and positions into shared memory
      SK[j] = load_key<R>(in + j);
      SI[j] = (uint16_t)j;
    }
    uint32_t d = (uint32_t)__ffs(vm) - 1;
    vm &= vm - 1;
    if (d != counted) {
      for (uint32_t x = tid; x < kLWarps * 257; x += kLThreads) wc[x] = 0;
      __syncthreads();
      local_count<R>(in, wc, d, wlo, whi, lane, warp);
    }
    __syncthreads();
    uint32_t q = 0;
    while (true) {
      const bool more = vm != 0;
      const uint32_t dn = more ? (uint32_t)__ffs(vm) - 1 : 0u;
      local_scan(wc, half, wsum);
      if (more) {
        for (uint32_t x = tid; x < kLWarps * 257; x += kLThreads) wn[x] = 0;
        __syncthreads();
      }
      const Key* sk = (q & 1u) ? GK : SK;
      const uint16_t* si = (q & 1u) ? GI : SI;
      Key* dk = (q & 1u) ? SK : GK;
      uint16_t* di = (q & 1u) ? SI : GI;
      for (uint32_t b0 = wlo; b0 < whi; b0 += 32 * kU) {
        Key kk[kU];
        uint32_t ii[kU];
#pragma unroll
        for (uint32_t u = 0; u < kU; ++u) {
          const uint32_t j = b0 + u * 32 + lane;
          kk[u] = j < whi ? sk[j] : Key(0);
          ii[u] = j < whi ? si[j] : 0u;
        }
#pragma unroll
        for (uint32_t u = 0; u < kU; ++u) {
          if (b0 + u * 32 >= whi) break;
          const bool valid = b0 + u * 32 + lane < whi;
          const uint32_t dg = valid ? (uint32_t)((kk[u] >> (8 * d)) & 255u) : 256u;
          const uint32_t peers = row_peers(dg, b0 + u * 32 + 32 <= whi);
          const uint32_t lt = __popc(peers & lt_mask);
          const uint32_t base = wc[warp * 257 + dg];
          __syncwarp();
          if (valid && lt == 0) wc[warp * 257 + dg] = base + __popc(peers);
          __syncwarp();
          if (valid) {
            const uint32_t pos = base + lt;
            dk[pos] = kk[u];
            di[pos] = (uint16_t)ii[u];
            if (more)
              atomicAdd(&wn[__umulhi(pos, cmagic) * 257 + (uint32_t)((kk[u] >> (8 * dn)) & 255u)], 1u);
          }
        }
      }
      __syncthreads();
      ++q;
      if (!more) break;
      uint32_t* t = wc;
      wc = wn;
      wn = t;
      d = dn;
      vm &= vm - 1;
    }
    // gather the records in key order: the last pass (q - 1) wrote the spill buffers when q - 1
    // is even, the shared ones when it is odd
    const uint16_t* fi = ((q - 1) & 1u) ? SI : GI;
    for (uint32_t j0 = tid; j0 < m; j0 += 4 * kLThreads) {
      Rec v[4];
#pragma unroll
      for (uint32_t u = 0; u < 4; ++u)
        if (j0 + u * kLThreads < m) v[u] = in[fi[j0 + u * kLThreads]];
#pragma unroll
      for (uint32_t u = 0; u < 4; ++u)
        if (j0 + u * kLThreads < m) out[j0 + u * kLThreads] = v[u];
    }
    __syncthreads();
  }
}

// The ranges of classes 1..5: one CTA per range. The range is split by key, evenly between its smallest
// and its largest one, into about as many bins as it has records: counts, a scan, and a scatter of (position, next
// 32 key bits) into bin order by shared-memory atomics (any order inside a bin). Then every record
// finds its rank among its bin's few members by (key, position), which is the stable order: 32 bits
// decide almost every comparison, the whole keys the rest. Keys spread evenly over the bins give
// at most about a dozen to a bin; a range with more than kFull in one (few distinct keys, clusters) is
// ordered by LSD passes over the varying digits instead, positions moving between two arrays in
// shared memory (class 5 has no room for them: such a range is left to local_sort_kernel).
// n = 2^29 16-byte records (8192 per range): 6.43 ms, 14.9 ms for local_sort_kernel, which read a range
// three times and sorted sub-buckets with bitonic networks; 40,000,001 records (packed ranges of about
// 3600): 0.52 ms against 2.19 for one warp per group; n = 2^27 (2048 per range): 1.56 ms, 1.96 without
// the class of 256 threads.
// Bound by shared-memory wavefronts and the latency between a range's barriers.
// Classes 1..4 hold the records in shared memory (one bulk copy in, gathered from there on the way
// out; the CTA's next range is prefetched into L2 meanwhile), so each record is read and written once.
// Class 5 holds the keys and gathers the records from a second read of the range.
template <int R, int CLS>
struct BinSmem {
  using Key = typename RecT<R>::Key;
  using B = Bin<R, CLS>;
  static constexpr bool kRecs = CLS < 5;
  static constexpr uint32_t kItem = kRecs ? (uint32_t)R : (uint32_t)sizeof(Key);
  static constexpr uint32_t bins = al16(B::kMax * kItem + (kRecs && R == 8 ? 8 : 0));
  static constexpr uint32_t rem = bins + (2u << B::kBits);
  static constexpr uint32_t pl = rem + (kRecs ? al16(B::kMax * 4) : 0u);
  static constexpr uint32_t wsum = pl + al16(B::kMax * 2);
  static constexpr uint32_t total = wsum + 32 * 4 + 48;
};

// BATCH: the ranges of many arrays (bs.list); else one array's, listed by its plan.
template <int R, int CLS, bool BATCH>
__global__ void __launch_bounds__(Bin<R, CLS>::kT, Bin<R, CLS>::kCtas) bin_sort_kernel(HybridArgs a, BatchSort bs) {
  using Rec = typename RecT<R>::T;
  using Key = typename RecT<R>::Key;
  using L = BinSmem<R, CLS>;
  constexpr uint32_t T = Bin<R, CLS>::kT, kMax = Bin<R, CLS>::kMax, kBits = Bin<R, CLS>::kBits;
  constexpr uint32_t kItems = (kMax + T - 1) / T;
  constexpr uint32_t kU = 4;  // loads in flight per thread
  constexpr bool kRecs = L::kRecs;
  static_assert(kRecs || !BATCH, "a batch's plans list no ranges of class 5");
  uint32_t mode = 0, l0 = 0, nlist = 0;
  if constexpr (BATCH) {
    nlist = bs.count[CLS];
  } else {
    mode = a.ctrl->sort_mode;
    if (mode == 0) return;
    l0 = a.meta[kMetaList + CLS];
    nlist = a.meta[kMetaList + CLS + 1] - l0;
  }
  if (blockIdx.x >= nlist) return;
  extern __shared__ __align__(16) unsigned char bsm[];
  Rec* SR = reinterpret_cast<Rec*>(bsm);                          // [kMax] records (classes 1..4)
  Key* SK = reinterpret_cast<Key*>(bsm);                          // [kMax] keys (class 5)
  uint32_t* bins = reinterpret_cast<uint32_t*>(bsm + L::bins);    // [2^kBits / 2]: 16 bits each
  uint32_t* rem = reinterpret_cast<uint32_t*>(bsm + L::rem);      // [kMax] next key bits in bin order (classes 1..4)
  uint16_t* pl = reinterpret_cast<uint16_t*>(bsm + L::pl);        // [kMax] positions in bin order
  uint32_t* wsum = reinterpret_cast<uint32_t*>(bsm + L::wsum);    // [32]
  unsigned long long* red = reinterpret_cast<unsigned long long*>(wsum + 32);  // smallest and largest key
  unsigned long long* bar = red + 2;
  uint32_t* next = reinterpret_cast<uint32_t*>(red + 3);  // the CTA's next range
  // range t: its records, their place in the sort's output, their count, its array's control block
  auto range = [&](uint32_t t, const Rec*& in, Rec*& out, uint64_t& m, Ctrl*& ctrl) {
    if constexpr (BATCH) {
      const uint4 e = bs.list[CLS * bs.cap + t];
      const RadixArgs& ra = bs.br.args[e.x];
      in = reinterpret_cast<const Rec*>(e.w ? ra.buf0 : ra.buf1) + e.y;  // in place, or from the scratch buffer
      out = reinterpret_cast<Rec*>(ra.buf0) + e.y;
      m = e.z;
      ctrl = ra.ctrl;
    } else {
      const uint32_t r = a.ridx[l0 + t];
      const uint64_t lo = a.gstart[a.rlist[r]];
      in = sort_buf<R>(a, mode, mode - 1) + lo;
      out = sort_buf<R>(a, mode, mode) + lo;
      m = a.gstart[a.rlist[r + 1]] - lo;
      ctrl = a.ctrl;
    }
  };
  uint32_t* ticket;
  if constexpr (BATCH)
    ticket = bs.count + (kClasses - 1) + CLS;
  else
    ticket = &a.ctrl->tickets[kTicketClass + CLS];
  const uint32_t tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5;
  if (kRecs && tid == 0) {
    mbar_init(smem_u32(bar), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  uint32_t ti = blockIdx.x, parity = 0;  // the first range is the block's own, later ones come by ticket

  while (true) {
    const Rec* in;
    Rec* out;
    uint64_t m64;
    Ctrl* ctrl;
    range(ti, in, out, m64, ctrl);
    const bool fits = m64 > 0 && m64 <= kMax;  // always: the plan lists only this class's sizes
    const uint32_t m = fits ? (uint32_t)m64 : 0u;
    // 8-byte records on an odd address start one slot into the array, so that the bulk copy's both
    // ends are 16-byte aligned; the records at the odd ends are copied by threads
    const uint32_t odd = kRecs && R == 8 ? (uint32_t)((reinterpret_cast<uintptr_t>(in) >> 3) & 1u) : 0u;
    const uint32_t c0 = odd < m ? odd : m, c1 = R == 8 ? c0 + ((m - c0) & ~1u) : m;  // bulk part [c0, c1)
    if (tid == 0) {
      if (kRecs) {
        mbar_expect_tx(smem_u32(bar), (c1 - c0) * R);
        if (c1 > c0) tma_load(smem_u32(SR + odd + c0), in + c0, (c1 - c0) * R, smem_u32(bar));
      }
      if (!fits) atomicExch(&ctrl->bad, 1u);
      red[0] = ~0ull;
      red[1] = 0;
      *next = gridDim.x + atomicAdd(ticket, 1u);
    }
    const uint32_t lg = m > 1 ? 32u - (uint32_t)__clz(m - 1) : 0u, nb = lg < kBits ? (lg > 6 ? lg : 6u) : kBits;
    for (uint32_t x = tid; x < (1u << nb) / 8; x += T) reinterpret_cast<uint4*>(bins)[x] = make_uint4(0, 0, 0, 0);
    if (kRecs && R == 8) {
      if (tid == 32 && c0 > 0) SR[odd] = in[0];
      if (tid == 33 && c1 < m) SR[odd + c1] = in[c1];
    }
    __syncthreads();
    const uint32_t tn = *next;
    if (kRecs && tid == 0 && tn < nlist) {  // the next range on its way to L2
      const Rec* in2;
      Rec* out2;
      uint64_t m2;
      Ctrl* ctrl2;
      range(tn, in2, out2, m2, ctrl2);
      const uintptr_t p0 = (reinterpret_cast<uintptr_t>(in2) + 15) & ~(uintptr_t)15;
      const uintptr_t p1 = reinterpret_cast<uintptr_t>(in2 + m2) & ~(uintptr_t)15;
      const uint32_t nby = p1 > p0 ? (uint32_t)(p1 - p0) : 0u;
      if (nby) asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p0), "r"(nby) : "memory");
    }
    // ---- the smallest and the largest key ----
    auto key_at = [&](uint32_t j) -> Key { return kRecs ? load_key<R>(SR + odd + j) : SK[j]; };
    if (kRecs) mbar_wait(smem_u32(bar), parity, ctrl);
    parity ^= 1u;
    Key kmin = ~Key(0), kmax = Key(0);
    for (uint32_t j0 = tid; j0 < m; j0 += kU * T) {
      Key kk[kU];
#pragma unroll
      for (uint32_t u = 0; u < kU; ++u)
        if (j0 + u * T < m) kk[u] = kRecs ? key_at(j0 + u * T) : load_key<R>(in + j0 + u * T);
#pragma unroll
      for (uint32_t u = 0; u < kU; ++u)
        if (j0 + u * T < m) {
          if (!kRecs) SK[j0 + u * T] = kk[u];
          kmin = kk[u] < kmin ? kk[u] : kmin;
          kmax = kk[u] > kmax ? kk[u] : kmax;
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const Key x = __shfl_xor_sync(0xFFFFFFFFu, kmin, o), y = __shfl_xor_sync(0xFFFFFFFFu, kmax, o);
      kmin = x < kmin ? x : kmin;
      kmax = y > kmax ? y : kmax;
    }
    if (lane == 0) {
      atomicMin(&red[0], (unsigned long long)kmin);
      atomicMax(&red[1], (unsigned long long)kmax);
    }
    __syncthreads();
    kmin = (Key)red[0];
    kmax = (Key)red[1];
    if (m < 2 || kmin == kmax) {  // every key equal: the range is already in order
      for (uint32_t j = tid; j < m; j += T) out[j] = kRecs ? SR[odd + j] : in[j];
    } else {
      const uint32_t top = 64u - (uint32_t)__clzll((long long)(unsigned long long)(Key)(kmax - kmin));
      const uint32_t sh = top > nb ? top - nb : 0u;
      auto bin_of = [&](Key k) -> uint32_t { return (uint32_t)((Key)(k - kmin) >> sh); };
      // the 32 bits below the bin's (all of them when sh <= 32)
      auto rest_of = [&](Key k) -> uint32_t {
        const unsigned long long d = (Key)(k - kmin);
        return sh >= 32 ? (uint32_t)(d >> (sh - 32)) : sh ? (uint32_t)d << (32 - sh) : 0u;
      };
      // ---- counts, starts ----
#pragma unroll 4
      for (uint32_t j = tid; j < m; j += T) {
        const uint32_t b = bin_of(key_at(j));
        atomicAdd(&bins[b >> 1], 1u << ((b & 1u) * 16));
      }
      __syncthreads();
      bool crowded;
      {
        constexpr uint32_t kPer = ((1u << kBits) / 2 + T - 1) / T;  // words per thread, consecutive
        const uint32_t W = (1u << nb) / 2, w0 = tid * kPer;
        uint32_t w[kPer], sum = 0, big = 0;
        if constexpr (kPer % 4 == 0) {
#pragma unroll
          for (uint32_t x = 0; x < kPer; x += 4) {
            const uint4 v = w0 + x < W ? reinterpret_cast<const uint4*>(bins)[(w0 + x) / 4] : make_uint4(0, 0, 0, 0);
            w[x] = v.x, w[x + 1] = v.y, w[x + 2] = v.z, w[x + 3] = v.w;
          }
        } else {
#pragma unroll
          for (uint32_t x = 0; x < kPer; ++x) w[x] = w0 + x < W ? bins[w0 + x] : 0u;
        }
#pragma unroll
        for (uint32_t x = 0; x < kPer; ++x) {
          sum += (w[x] & 0xFFFFu) + (w[x] >> 16);
          big |= ((w[x] & 0xFFFFu) > kFull || (w[x] >> 16) > kFull) ? 1u : 0u;
        }
        uint32_t incl = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
          if (lane >= (uint32_t)o) incl += y;
        }
        if (lane == 31) wsum[warp] = incl;
        crowded = __syncthreads_or(big);
        uint32_t run = __reduce_add_sync(0xFFFFFFFFu, lane < warp ? wsum[lane] : 0u) + incl - sum;
#pragma unroll
        for (uint32_t x = 0; x < kPer; ++x) {
          const uint32_t c = w[x];
          w[x] = run | (run + (c & 0xFFFFu)) << 16;
          run += (c & 0xFFFFu) + (c >> 16);
        }
        if constexpr (kPer % 4 == 0) {
#pragma unroll
          for (uint32_t x = 0; x < kPer; x += 4)
            if (w0 + x < W) reinterpret_cast<uint4*>(bins)[(w0 + x) / 4] = make_uint4(w[x], w[x + 1], w[x + 2], w[x + 3]);
        } else {
#pragma unroll
          for (uint32_t x = 0; x < kPer; ++x)
            if (w0 + x < W) bins[w0 + x] = w[x];
        }
      }
      const uint16_t* order = pl;  // positions in key order
      if (crowded && !kRecs) {  // the other kernel's range
        if (tid == 0) a.joint[atomicAdd(&a.meta[kMetaLeft], 1u)] = a.ridx[l0 + ti];
        order = nullptr;
      } else if (crowded) {
        // ---- LSD passes. Warp w owns the positions [w c, (w + 1) c) of the current order; its counts
        // of the 256 digit values, later its next places, are 16-bit words in the bins' memory ----
        constexpr uint32_t W = T / 32;
        uint16_t* cur = pl;
        uint16_t* nxt = reinterpret_cast<uint16_t*>(rem);
        const uint32_t c = ((m + W - 1) / W + 31u) & ~31u;
        const uint32_t wlo = warp * c < m ? warp * c : m, whi = wlo + c < m ? wlo + c : m;
        for (uint32_t j = tid; j < m; j += T) cur[j] = (uint16_t)j;
        for (uint32_t d = 0; d * 8 < top; ++d) {
          auto digit = [&](uint32_t j) -> uint32_t { return (uint32_t)((Key)(key_at(j) - kmin) >> (8 * d)) & 255u; };
          __syncthreads();
          for (uint32_t x = tid; x < W * 128; x += T) bins[x] = 0;
          __syncthreads();
          for (uint32_t q = wlo + lane; q < whi; q += 32) {
            const uint32_t v = digit(cur[q]);
            atomicAdd(&bins[warp * 128 + v / 2], 1u << ((v & 1u) * 16));
          }
          __syncthreads();
          uint32_t tot = 0, incl = 0, same = 0;  // thread t < 128: the digit values 2t and 2t + 1, packed
          if (tid < 128) {
            for (uint32_t w = 0; w < W; ++w) tot += bins[w * 128 + tid];
            same = (tot & 0xFFFFu) == m || (tot >> 16) == m ? 1u : 0u;
            incl = (tot & 0xFFFFu) + (tot >> 16);
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
              const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
              if (lane >= (uint32_t)o) incl += y;
            }
            if (lane == 31) wsum[warp] = incl;
          }
          if (__syncthreads_or(same)) continue;  // one value: the pass would change nothing
          if (tid < 128) {
            uint32_t run = incl - (tot & 0xFFFFu) - (tot >> 16);
            for (uint32_t w = 0; w < warp; ++w) run += wsum[w];
            run |= (run + (tot & 0xFFFFu)) << 16;
            for (uint32_t w = 0; w < W; ++w) {
              const uint32_t x = bins[w * 128 + tid];
              bins[w * 128 + tid] = run;
              run += x;
            }
          }
          __syncthreads();
          uint16_t* place = reinterpret_cast<uint16_t*>(bins) + warp * 256;
          for (uint32_t b = wlo; b < whi; b += 32) {
            const bool valid = b + lane < whi;
            const uint32_t j = valid ? cur[b + lane] : 0u, v = valid ? digit(j) : 256u;
            const uint32_t peers = row_peers(v, b + 32 <= whi);
            const uint32_t lt = __popc(peers & lanemask_lt());
            const uint32_t base = valid ? place[v] : 0u;
            __syncwarp();
            if (valid && lt == 0) place[v] = (uint16_t)(base + __popc(peers));
            __syncwarp();
            if (valid) nxt[base + lt] = (uint16_t)j;
          }
          uint16_t* t = cur;
          cur = nxt;
          nxt = t;
        }
        __syncthreads();
        order = cur;
      } else {
        __syncthreads();
        // ---- positions (and rests) into bin order; a bin's start becomes its end ----
        uint32_t it[kItems];  // place in bin order << 16 | bin
#pragma unroll
        for (uint32_t i = 0; i < kItems; ++i) {
          const uint32_t j = tid + i * T;
          if (j < m) {
            const Key k = key_at(j);
            const uint32_t b = bin_of(k), hs = (b & 1u) * 16;
            const uint32_t p = (atomicAdd(&bins[b >> 1], 1u << hs) >> hs) & 0xFFFFu;
            pl[p] = (uint16_t)j;
            if (kRecs) rem[p] = rest_of(k);
            it[i] = p << 16 | b;
          }
        }
        __syncthreads();
        // ---- every record's rank in its bin ----
#pragma unroll
        for (uint32_t i = 0; i < kItems; ++i) {
          const uint32_t j = tid + i * T;
          if (j < m) {
            const uint32_t b = it[i] & 0xFFFFu, p = it[i] >> 16;
            const uint32_t e = (bins[b >> 1] >> ((b & 1u) * 16)) & 0xFFFFu;
            const uint32_t s = b ? (bins[(b - 1) >> 1] >> (((b - 1) & 1u) * 16)) & 0xFFFFu : 0u;
            uint32_t rank = s;
            if (kRecs) {
              const uint32_t mine = rem[p];
              for (uint32_t q = s; q < e; ++q) {
                const uint32_t x = rem[q];
                rank += x < mine ? 1u : 0u;
                if (x == mine && q != p) {  // equal so far: the whole keys, then the positions
                  const uint32_t j2 = pl[q];
                  const Key k = key_at(j), k2 = key_at(j2);
                  rank += (k2 < k || (k2 == k && j2 < j)) ? 1u : 0u;
                }
              }
            } else {
              const Key k = key_at(j);
              for (uint32_t q = s; q < e; ++q) {
                const uint32_t j2 = pl[q];
                const Key k2 = key_at(j2);
                rank += (k2 < k || (k2 == k && j2 < j)) ? 1u : 0u;
              }
            }
            it[i] = rank;
          }
        }
        __syncthreads();
#pragma unroll
        for (uint32_t i = 0; i < kItems; ++i)
          if (tid + i * T < m) pl[it[i]] = (uint16_t)(tid + i * T);
        __syncthreads();
      }
      if (order) {  // ---- the records in key order ----
        for (uint32_t j0 = tid; j0 < m; j0 += kU * T) {
          Rec v[kU];
#pragma unroll
          for (uint32_t u = 0; u < kU; ++u)
            if (j0 + u * T < m) v[u] = kRecs ? SR[odd + order[j0 + u * T]] : in[order[j0 + u * T]];
#pragma unroll
          for (uint32_t u = 0; u < kU; ++u)
            if (j0 + u * T < m) out[j0 + u * T] = v[u];
        }
      }
    }
    ti = tn;
    if (ti >= nlist) break;
    __syncthreads();  // the arrays are free
  }
}

template <int R, int CLS>
cudaError_t launch_bins(const HybridArgs& a, uint32_t count, int sms, cudaStream_t st) {
  if (count == 0) return cudaSuccess;
  auto kern = bin_sort_kernel<R, CLS, false>;
  static_assert(Bin<R, CLS>::kCtas * (BinSmem<R, CLS>::total + 1024) <= 233472, "the CTAs of this class fit an SM");
  const cudaError_t e = set_smem_optin(kern);
  if (e != cudaSuccess) return e;
  const uint32_t grid = (uint32_t)(sms * Bin<R, CLS>::kCtas);
  kern<<<grid < count ? grid : count, Bin<R, CLS>::kT, BinSmem<R, CLS>::total, st>>>(a, BatchSort{});
  return cudaGetLastError();
}

// Ascending bitonic sort of (key, position) pairs in registers, the same network as warp_sort:
// lane l holds elements l * EPL .. l * EPL + EPL - 1. Positions are distinct; padding is the
// largest pair. The stage loops stay rolled (one body per partner distance below EPL and one for
// the distances across lanes), so the code of every size fits the instruction cache.
template <typename Key>
__device__ __forceinline__ bool pair_less(Key ka, uint32_t xa, Key kb, uint32_t xb) {
  return ka < kb || (ka == kb && xa < xb);
}

template <typename Key, int EPL, int J>
__device__ __forceinline__ void pair_stage_lane(Key (&k)[EPL], uint32_t (&x)[EPL], uint32_t lane, uint32_t kk) {
  if constexpr (J < EPL) {
#pragma unroll
    for (int r = 0; r < EPL; ++r) {
      if ((r & J) == 0) {
        const bool up = ((lane * EPL + (uint32_t)r) & kk) == 0;
        const bool sw = pair_less(k[r | J], x[r | J], k[r], x[r]) == up;
        const Key tk = k[r];
        const uint32_t tx = x[r];
        k[r] = sw ? k[r | J] : k[r];
        x[r] = sw ? x[r | J] : x[r];
        k[r | J] = sw ? tk : k[r | J];
        x[r | J] = sw ? tx : x[r | J];
      }
    }
  }
}

template <typename Key, int EPL>
__device__ __forceinline__ void pair_stage_cross(Key (&k)[EPL], uint32_t (&x)[EPL], uint32_t lane, uint32_t kk,
                                                 uint32_t lj) {
#pragma unroll
  for (int r = 0; r < EPL; ++r) {
    const Key ok = __shfl_xor_sync(0xFFFFFFFFu, k[r], lj);
    const uint32_t ox = __shfl_xor_sync(0xFFFFFFFFu, x[r], lj);
    const bool up = ((lane * EPL + (uint32_t)r) & kk) == 0;
    const bool keep_min = ((lane & lj) == 0) == up;
    if (pair_less(ok, ox, k[r], x[r]) == keep_min) {
      k[r] = ok;
      x[r] = ox;
    }
  }
}

template <typename Key, int EPL>
__device__ __forceinline__ void warp_sort_pairs(Key (&k)[EPL], uint32_t (&x)[EPL], uint32_t lane) {
#pragma unroll 1
  for (uint32_t kk = 2; kk <= 32u * EPL; kk <<= 1) {
#pragma unroll 1
    for (uint32_t j = kk >> 1; j > 0; j >>= 1) {
      if (j >= (uint32_t)EPL) pair_stage_cross<Key, EPL>(k, x, lane, kk, j / EPL);
      else if (j == 1) pair_stage_lane<Key, EPL, 1>(k, x, lane, kk);
      else if (j == 2) pair_stage_lane<Key, EPL, 2>(k, x, lane, kk);
      else pair_stage_lane<Key, EPL, 4>(k, x, lane, kk);
    }
  }
}

// One range of m <= 32 * EPL records sorted by one warp: keys and positions into registers (in
// any arrangement: the network sorts them all), sorted, the order through shared memory, then the
// records gathered into place with coalesced writes.
template <int R, int EPL>
__device__ __forceinline__ void small_range(const typename RecT<R>::T* in, typename RecT<R>::T* out, uint32_t m,
                                            uint16_t* sidx, uint32_t lane) {
  using Key = typename RecT<R>::Key;
  Key k[EPL];
  uint32_t x[EPL];
#pragma unroll
  for (int r = 0; r < EPL; ++r) {
    const uint32_t e = (uint32_t)r * 32 + lane;
    k[r] = e < m ? load_key<R>(in + e) : ~Key(0);
    x[r] = e < m ? e : 0xFFFFFFFFu;
  }
  warp_sort_pairs<Key, EPL>(k, x, lane);
#pragma unroll
  for (int r = 0; r < EPL; ++r) {
    const uint32_t e = lane * EPL + (uint32_t)r;
    if (e < m) sidx[e] = (uint16_t)x[r];
  }
  __syncwarp();
  typename RecT<R>::T v[EPL];  // all read before the first is written: out may be in
#pragma unroll
  for (int r = 0; r < EPL; ++r)
    if ((uint32_t)r * 32 + lane < m) v[r] = in[sidx[r * 32 + lane]];
  __syncwarp();
#pragma unroll
  for (int r = 0; r < EPL; ++r)
    if ((uint32_t)r * 32 + lane < m) out[r * 32 + lane] = v[r];
  __syncwarp();
}

// The ranges of class 0 (many small groups), a warp each, taken by ticket; no block-wide barrier.
template <int R>
__device__ __forceinline__ void small_sort(const typename RecT<R>::T* in, typename RecT<R>::T* out, uint32_t m,
                                           uint16_t* sidx, uint32_t lane) {
  if (m == 0) return;
  if (m <= 32) small_range<R, 1>(in, out, m, sidx, lane);
  else if (m <= 64) small_range<R, 2>(in, out, m, sidx, lane);
  else if (m <= 128) small_range<R, 4>(in, out, m, sidx, lane);
  else small_range<R, 8>(in, out, m, sidx, lane);
}

template <int R>
__global__ void __launch_bounds__(kSThreads) local_small_kernel(HybridArgs a) {
  using Rec = typename RecT<R>::T;
  constexpr uint32_t kMax = Bin<R, 0>::kMax;
  const uint32_t mode = a.ctrl->sort_mode;
  if (mode == 0) return;
  __shared__ uint16_t sidx[kSThreads / 32][kMax];
  const Rec* src = sort_buf<R>(a, mode, mode - 1);
  Rec* dst = sort_buf<R>(a, mode, mode);
  const uint32_t lane = threadIdx.x & 31u, w = threadIdx.x >> 5;
  const uint32_t l0 = a.meta[kMetaList], nlist = a.meta[kMetaList + 1] - l0;
  while (true) {
    uint32_t t = 0;
    if (lane == 0) t = atomicAdd(&a.ctrl->tickets[kTicketClass], 1u);
    t = __shfl_sync(0xFFFFFFFFu, t, 0);
    if (t >= nlist) break;
    const uint32_t r = a.ridx[l0 + t];
    const uint64_t lo = a.gstart[a.rlist[r]];
    const uint64_t m64 = a.gstart[a.rlist[r + 1]] - lo;
    if (m64 > kMax) {  // never: the plan lists only small ranges here
      if (lane == 0) atomicExch(&a.ctrl->bad, 1u);
      continue;
    }
    small_sort<R>(src + lo, dst + lo, (uint32_t)m64, sidx[w], lane);
  }
}

// ---- batched: the plans, the partition and the ranges of many arrays --------------------------

// One CTA per array: the digit offsets, the live digits and the mode (kBatchOnChip: the array is one
// range; 2: one partition by the top varying digit; 0: LSD passes), and the ranges into the lists of
// their classes. Four digits at a time, eight warps each.
template <int R>
__global__ void __launch_bounds__(1024) batch_plan_kernel(BatchSort bs) {
  constexpr uint32_t D = RecT<R>::kDigits, kCap = Bin<R, kClasses - 2>::kMax, kOne = Bin<R, 2>::kMax;
  __shared__ uint32_t s_w[32], s_max[8], s_start[257], s_cnt[256], s_first[256];
  const RadixArgs& a = bs.br.args[blockIdx.x];
  const uint32_t tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5, n = (uint32_t)a.n;
  if (tid < 8) s_max[tid] = 0;
  __syncthreads();
  for (uint32_t x = tid; x < D * 256; x += 1024) {
    const uint32_t mx = __reduce_max_sync(0xFFFFFFFFu, a.hist[x]);
    if (lane == 0) atomicMax(&s_max[x >> 8], mx);
  }
  __syncthreads();
  uint32_t live = 0;
  for (uint32_t d = 0; d < D; ++d) live |= s_max[d] < n ? 1u << d : 0u;  // some key differs in digit d
  const uint32_t dA = live ? 31u - (uint32_t)__clz(live) : 0u;
  for (uint32_t x = tid; x < D * 256; x += 1024) {
    const uint32_t c = a.hist[x];
    uint32_t incl = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
      if (lane >= (uint32_t)o) incl += y;
    }
    if (lane == 31) s_w[warp] = incl;
    __syncthreads();
    uint32_t ex = incl - c;
    for (uint32_t w = warp & ~7u; w < warp; ++w) ex += s_w[w];
    a.dbase[x] = ex;
    if (x >> 8 == dA) {
      s_start[x & 255u] = ex;
      s_cnt[x & 255u] = c;
    }
    __syncthreads();
  }
  const uint32_t maxA = s_max[dA];
  const uint32_t mode = n < 2 || !live ? 0u : n <= kOne ? kBatchOnChip : maxA <= kCap ? 2u : 0u;
  if (tid == 0) {
    s_start[256] = n;
    a.ctrl->radix_live = live;
    a.ctrl->sort_mode = mode;
    if (mode == 0 && live) atomicOr(bs.br.lsd, live);
  }
  if (mode == 0) return;
  auto list = [&](uint32_t lo, uint32_t m, uint32_t in_place) {
    const uint32_t c = m <= Bin<R, 0>::kMax ? 0u : m <= Bin<R, 1>::kMax ? 1u : m <= Bin<R, 2>::kMax ? 2u
                       : m <= Bin<R, 3>::kMax ? 3u : 4u;
    bs.list[c * bs.cap + atomicAdd(&bs.count[c], 1u)] = make_uint4(blockIdx.x, lo, m, in_place);
  };
  if (mode == kBatchOnChip) {
    if (tid == 0) list(0, n, 1);
    return;
  }
  __syncthreads();
  const bool single = maxA * 3 > bs.P;
  const uint32_t S = single ? 1u : bs.P - maxA + 1u, v = tid & 255u, g = s_start[v];
  const bool first = v == 0 || (single ? s_cnt[v] > 0 : g / S != (g - s_cnt[v - 1]) / S);
  if (tid < 256) s_first[v] = first ? 1u : 0u;
  __syncthreads();
  if (tid < 256 && first) {
    uint32_t e = v + 1;
    while (e < 256 && !s_first[e]) ++e;
    const uint32_t m = s_start[e] - g;
    if (m) list(g, m, 0);
  }
}

// The partition of the arrays in mode 2 (the top varying digit); tiles by ticket, in array order.
template <int R>
__global__ void __launch_bounds__(kTileThreads, 2) batch_msd_kernel(BatchSort bs) {
  __shared__ unsigned long long t_s;
  __shared__ uint32_t j_s;
  while (true) {
    if (threadIdx.x == 0) {
      const uint64_t t = atomicAdd(bs.ticket, 1u);
      uint32_t lo = 0, hi = bs.br.narr;
      while (t < bs.br.nblocks && hi - lo > 1) {
        const uint32_t mid = (lo + hi) >> 1;
        if (bs.br.first[mid] <= t) lo = mid; else hi = mid;
      }
      j_s = t < bs.br.nblocks ? lo : 0xFFFFFFFFu;
      t_s = t - bs.br.first[lo];
    }
    __syncthreads();
    if (j_s == 0xFFFFFFFFu) break;
    const RadixArgs& a = bs.br.args[j_s];
    if (a.ctrl->sort_mode == 2) {
      const uint32_t dA = 31u - (uint32_t)__clz(a.ctrl->radix_live);
      radix_tile<R>(reinterpret_cast<const typename RecT<R>::T*>(a.buf0), reinterpret_cast<typename RecT<R>::T*>(a.buf1), a.n,
                    t_s, 8 * dA, kTagMsd1, a.status, a.dbase + dA * 256, a.n, a.ctrl);
    }
    __syncthreads();
  }
}

template <int R>
__global__ void __launch_bounds__(kSThreads) batch_small_kernel(BatchSort bs) {
  using Rec = typename RecT<R>::T;
  __shared__ uint16_t sidx[kSThreads / 32][Bin<R, 0>::kMax];
  const uint32_t lane = threadIdx.x & 31u, w = threadIdx.x >> 5, nlist = bs.count[0];
  while (true) {
    uint32_t t = 0;
    if (lane == 0) t = atomicAdd(bs.count + kClasses - 1, 1u);
    t = __shfl_sync(0xFFFFFFFFu, t, 0);
    if (t >= nlist) break;
    const uint4 e = bs.list[t];
    const RadixArgs& a = bs.br.args[e.x];
    small_sort<R>(reinterpret_cast<const Rec*>(e.w ? a.buf0 : a.buf1) + e.y, reinterpret_cast<Rec*>(a.buf0) + e.y, e.z, sidx[w], lane);
  }
}

template <int R, int CLS>
cudaError_t batch_bins(const BatchSort& bs, int sms, cudaStream_t st) {
  auto kern = bin_sort_kernel<R, CLS, true>;
  const cudaError_t e = set_smem_optin(kern);
  if (e != cudaSuccess) return e;
  const uint32_t grid = (uint32_t)(sms * Bin<R, CLS>::kCtas);
  kern<<<grid < bs.cap ? grid : bs.cap, Bin<R, CLS>::kT, BinSmem<R, CLS>::total, st>>>(HybridArgs{}, bs);
  return cudaGetLastError();
}

int device_sms() {
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return 0;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 0;
  return sms;
}

template <int R>
cudaError_t launch_r(const HybridArgs& a, int stage, const uint32_t* list, cudaStream_t st) {
  constexpr int D = RecT<R>::kDigits;
  cudaError_t e = cudaSuccess;
  const int sms = device_sms();
  if (sms <= 0) return cudaErrorInvalidDevice;
  switch (stage) {
    case 0: {
      const uint32_t smem = (D * 256 + kGroups / 2) * 4;
      if ((e = cudaFuncSetAttribute(hybrid_hist_kernel<R>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) !=
          cudaSuccess)
        return e;
      const uint64_t need = (a.n + kJThreads - 1) / kJThreads;
      const unsigned grid = (unsigned)(need < (uint64_t)sms ? (need ? need : 1) : (uint64_t)sms);
      hybrid_hist_kernel<R><<<grid, kJThreads, smem, st>>>(a);
      break;
    }
    case 1:
      sort_plan_kernel<R><<<1, kPlanThreads, 0, st>>>(a);
      break;
    case 2:
    case 3: {
      const uint32_t smem = radix_tile_smem<R>();
      const uint64_t tiles = radix_tiles(a.n, R) + (stage == 3 ? 256u : 0u);  // upper bound for stage 3
      const unsigned grid = (unsigned)(tiles < 2ull * sms ? tiles : 2ull * sms);  // two CTAs per SM
      if (stage == 2) {
        if ((e = set_smem_optin(msd1_kernel<R>)) != cudaSuccess) return e;
        msd1_kernel<R><<<grid, kTileThreads, smem, st>>>(a);
      } else {
        if ((e = set_smem_optin(msd2_kernel<R>)) != cudaSuccess) return e;
        msd2_kernel<R><<<grid, kTileThreads, smem, st>>>(a);
      }
      break;
    }
    default: {
      if (list[0]) {
        // rounded up without a sum: the count is all ones when the host does not know it
        const uint32_t need = (list[0] - 1) / (kSThreads / 32) + 1, most = (uint32_t)sms * 8;
        local_small_kernel<R><<<need < most ? need : most, kSThreads, 0, st>>>(a);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
      }
      if ((e = launch_bins<R, 1>(a, list[1], sms, st)) != cudaSuccess) return e;
      if ((e = launch_bins<R, 2>(a, list[2], sms, st)) != cudaSuccess) return e;
      if ((e = launch_bins<R, 3>(a, list[3], sms, st)) != cudaSuccess) return e;
      if ((e = launch_bins<R, 4>(a, list[4], sms, st)) != cudaSuccess) return e;
      if (list[5] == 0) break;
      if ((e = launch_bins<R, 5>(a, list[5], sms, st)) != cudaSuccess) return e;
      // only class 5 leaves ranges over
      const uint32_t smem = local_smem_bytes<R>();
      if ((e = cudaFuncSetAttribute(local_sort_kernel<R>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) !=
          cudaSuccess)
        return e;
      const unsigned grid = a.local_ctas < (uint32_t)sms ? a.local_ctas : (unsigned)sms;
      local_sort_kernel<R><<<grid, kLThreads, smem, st>>>(a);
      break;
    }
  }
  return cudaGetLastError();
}

template <int R>
cudaError_t batch_sort_r(const BatchSort& bs, int stage, cudaStream_t st) {
  const int sms = device_sms();
  if (sms <= 0) return cudaErrorInvalidDevice;
  cudaError_t e = cudaSuccess;
  if (stage == 0) {
    batch_plan_kernel<R><<<bs.br.narr, 1024, 0, st>>>(bs);
  } else if (stage == 1) {
    if ((e = set_smem_optin(batch_msd_kernel<R>)) != cudaSuccess) return e;
    const uint64_t grid = bs.br.nblocks < 2ull * sms ? bs.br.nblocks : 2ull * sms;  // two CTAs per SM
    batch_msd_kernel<R><<<(unsigned)grid, kTileThreads, radix_tile_smem<R>(), st>>>(bs);
  } else {
    batch_small_kernel<R><<<(unsigned)sms * 4, kSThreads, 0, st>>>(bs);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    if (bs.max_n > Bin<R, 0>::kMax && (e = batch_bins<R, 1>(bs, sms, st)) != cudaSuccess) return e;
    if (bs.max_n > Bin<R, 1>::kMax && (e = batch_bins<R, 2>(bs, sms, st)) != cudaSuccess) return e;
    if (bs.max_n > Bin<R, 2>::kMax && (e = batch_bins<R, 3>(bs, sms, st)) != cudaSuccess) return e;
    if (bs.max_n > Bin<R, 3>::kMax && (e = batch_bins<R, 4>(bs, sms, st)) != cudaSuccess) return e;
  }
  return cudaGetLastError();
}

}  // namespace

uint32_t batch_sort_ranges(uint64_t n, int) { return n <= Bin<16, 2>::kMax ? 1u : 256u; }
static_assert(Bin<16, 2>::kMax == Bin<8, 2>::kMax, "one rule for both widths");

// Ranges of class 1 (eight CTAs per SM) while the batch gives every SM few of them, then of class 3.
uint32_t batch_sort_pack(uint64_t records, int R) {
  if (records < (4u << 20)) return Bin<16, 1>::kMax;
  return R == 8 ? Bin<8, kMidClass>::kMax : Bin<16, kMidClass>::kMax;
}

cudaError_t launch_batch_sort(const BatchSort& bs, int R, int stage, cudaStream_t st) {
  if (bs.br.narr == 0 || bs.br.nblocks == 0) return cudaSuccess;
  return R == 8 ? batch_sort_r<8>(bs, stage, st) : batch_sort_r<16>(bs, stage, st);
}

uint32_t hybrid_local_ctas(uint64_t n, int R) {
  const uint64_t cap = R == 8 ? Local<8>::kCap : Local<16>::kCap;
  const uint64_t want = (n + cap / 2 - 1) / (cap / 2);
  return (uint32_t)(want < 1 ? 1 : want > kLocalMaxCtas ? kLocalMaxCtas : want);
}

size_t hybrid_spill_bytes(uint64_t n, int R) {
  const size_t per = R == 8 ? (size_t)Local<8>::kCap * 6 : (size_t)Local<16>::kCap * 10;
  return per * hybrid_local_ctas(n, R);
}

uint32_t batch_sort_cap(int R) { return R == 8 ? Bin<8, kClasses - 2>::kMax : Bin<16, kClasses - 2>::kMax; }

cudaError_t launch_hybrid(const HybridArgs& a, int R, int stage, const uint32_t* list, cudaStream_t st) {
  if (a.n == 0) return cudaSuccess;
  return R == 8 ? launch_r<8>(a, stage, list, st) : launch_r<16>(a, stage, list, st);
}

}  // namespace bos
