// One tile of a stable scatter by one 8-bit digit (onesweep organisation), shared by the LSD
// radix sort (radix.cu) and the MSD partition passes of the hybrid sort (sort_hybrid.cu).
#pragma once
#include "common.cuh"

namespace bos {
namespace rtile {

constexpr int kThreads = 512;
constexpr int kWarps = kThreads / 32;
constexpr int kItems = 8;
constexpr uint32_t kTile = kThreads * kItems;

constexpr int kLook = 256;                      // look-back threads, one per digit value
constexpr int kTileThreads = kThreads + kLook;  // of the kernels that run radix_tile

template <int ID, int N>
__device__ __forceinline__ void bar_sync() {
  asm volatile("bar.sync %0, %1;" ::"n"(ID), "n"(N) : "memory");
}
template <int ID, int N>
__device__ __forceinline__ void bar_arrive() {
  asm volatile("bar.arrive %0, %1;" ::"n"(ID), "n"(N) : "memory");
}

// Look-back of one digit value at tile `tile` >= 1 (count `own`), `st` its status words (256 apart per
// tile). A word that is not inclusive yet holds the tile's own count (bits 0..15) and, once its owner
// has summed it, the count of the tile and its seven predecessors (bits 16..31, valid with kHas8). So
// seven words give the first seven predecessors, and every further word stands for eight tiles: about
// 15 words are read for the 80 to 140 tiles that have no inclusive word yet at n = 2^29 (a load takes
// 1300 cycles under the pass's own traffic). Words that are missing are waited for one by one: loading
// all of them anew together put 13 % on the pass.
constexpr unsigned long long kHas8 = 1ull << 32;

__device__ __forceinline__ unsigned long long wait_count(const unsigned long long* p, unsigned long long v,
                                                         bool need8, uint32_t tag, Ctrl* ctrl) {
  uint32_t spins = 0;
  while (!((v >> 62) != 0 && ((v >> 56) & 63u) == tag && (!need8 || (v & (kStIncl | kHas8))))) {
    if (++spins > kSpinLimit) {
      atomicExch(&ctrl->timeout, 1u);
      return kStIncl;  // gives up: the result is not valid
    }
    if (spins > 16) __nanosleep(32);
    v = ld_status(p);
  }
  return v;
}

__device__ __forceinline__ unsigned long long lookback_by8(unsigned long long* st, uint64_t tile, uint32_t own,
                                                           uint32_t tag, Ctrl* ctrl) {
  unsigned long long w[8];
  unsigned long long prefix = 0;
  {
    const uint32_t m = tile < 7 ? (uint32_t)tile : 7u;
    const unsigned long long* p = st + (tile - 1) * 256;
#pragma unroll
    for (int x = 0; x < 7; ++x) w[x] = x < m ? ld_status(p - x * 256) : 0ull;
#pragma unroll
    for (int x = 0; x < 7; ++x) {
      if (x >= m) return prefix;  // the first tiles
      const unsigned long long v = wait_count(p - x * 256, w[x], false, tag, ctrl);
      if (v & kStIncl) return prefix + (v & kStValue);
      prefix += v & 0xFFFFu;
    }
  }
  if (tile == 7) return prefix;
  st_status(st + tile * 256, st_word(kStAgg, tag, own | (prefix + own) << 16 | kHas8));
  // the next word stands for tiles j-7 .. j; tiles 0 .. 7 only ever get an inclusive one: the walk ends there
  for (uint64_t j = tile - 8;; j -= 64) {
    const uint32_t m = j < 56 ? (uint32_t)(j >> 3) + 1 : 8u;
    const unsigned long long* p = st + j * 256;
#pragma unroll
    for (int x = 0; x < 8; ++x) w[x] = x < m ? ld_status(p - x * 2048) : 0ull;
#pragma unroll
    for (int x = 0; x < 8; ++x) {
      if (x >= m) break;
      const unsigned long long v = wait_count(p - x * 2048, w[x], true, tag, ctrl);
      if (v & kStIncl) return prefix + (v & kStValue);
      prefix += (v >> 16) & 0xFFFFu;
    }
    if (j < 64) return prefix;
  }
}

// One tile (kTile records) of a stable scatter by one 8-bit digit (the whole CTA, kTileThreads).
//   src, n        the records of the segment being sorted (tile t covers [t*kTile, ...))
//   dst, dbase    output: records with digit value v go to dst[dbase[v] + rank among them];
//                 nout bounds the output (a position at or past it is never written)
//   status        the segment's look-back words, 256 per tile, tile 0 first
// Ranking is stable: warp-contiguous positions, lane-striped per item, ranked item by item with
// per-warp counters. 512 threads rank; 256 more publish the tile's counts before that and walk the
// decoupled look-back over the segment's preceding tiles meanwhile. The records stay where cp.async puts
// them and only their places are put in digit order, so that 768 threads at 40 registers fit twice.
// Bound by the latency of its phases, two CTAs an SM (load 3100 cycles, count 1700, rank 4300, places
// 2300, rest of the look-back 3400, write 3500 at n = 2^28; issue slots 47 %, shared memory 51 %, HBM
// 45 %). Two partitions at n = 2^29 of 16 B: 9.75 ms (3.5 TB/s), 10.3 with the look-back (6000 cycles)
// after the ranking in the same threads; eight LSD passes at 2^24: 1290 us against 1400.
// No gain: the next tile prefetched to L2, a look-back that starts after the ranking.
template <int R>
__device__ __forceinline__ void radix_tile(const typename RecT<R>::T* src, typename RecT<R>::T* dst, uint64_t n,
                                           uint64_t tile, uint32_t shift, uint32_t tag, unsigned long long* status,
                                           const unsigned long long* dbase, uint64_t nout, Ctrl* ctrl) {
  using Rec = typename RecT<R>::T;
  extern __shared__ __align__(16) unsigned char smem[];
  Rec* rec = reinterpret_cast<Rec*>(smem);                                               // [kTile]
  unsigned long long* gstart = reinterpret_cast<unsigned long long*>(rec + kTile);       // [256]
  uint32_t* wcnt = reinterpret_cast<uint32_t*>(gstart + 256);                            // [kWarps][257]
  uint32_t* lstart = wcnt + kWarps * 257;                                                // [257]
  uint32_t* cnt = lstart + 257;                                                          // [256]
  uint32_t* half0 = cnt + 256;                                                           // [256]
  uint32_t* wsum = half0 + 256;                                                          // [8]
  uint16_t* sidx = reinterpret_cast<uint16_t*>(wsum + 8);                                // [kTile]

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint64_t t0 = tile * kTile;
  const uint32_t left = n - t0 < kTile ? (uint32_t)(n - t0) : kTile;
  const uint32_t p0 = warp * 32 * kItems + lane;  // this thread's items: p0 + 32 it
  if (tid < kThreads) {
    const Rec* s = src + t0;
#pragma unroll
    for (int it = 0; it < kItems; ++it)
      if (p0 + it * 32 < left) cp_async<sizeof(Rec)>(rec + p0 + it * 32, s + p0 + it * 32);
    for (int x = tid; x < kWarps * 257; x += kThreads) wcnt[x] = 0;
  } else {
    cnt[tid - kThreads] = 0;
  }
  __syncthreads();
  if (tid < kThreads) {
    asm volatile("cp.async.wait_all;" ::: "memory");
    uint32_t dr[kItems];  // digit (bits 0..8, 256 = none) | rank inside the warp << 9
#pragma unroll
    for (int it = 0; it < kItems; ++it) {
      dr[it] = 256;
      if (p0 + it * 32 < left) {
        dr[it] = (uint32_t)(RecT<R>::key(rec[p0 + it * 32]) >> shift) & 255u;
        atomicAdd(&cnt[dr[it]], 1u);
      }
    }
    bar_sync<4, kTileThreads>();  // the tile's counts
    const uint32_t lt_mask = lanemask_lt();
    const bool full = left == kTile;  // every item present: eight ballots decide a digit
#pragma unroll
    for (int it = 0; it < kItems; ++it) {
      const uint32_t d = dr[it];
      const uint32_t peers = full ? ballot_peers(d, 8) : ballot_peers(d, 9);  // 9 bits: 256 = no item
      const uint32_t lt = __popc(peers & lt_mask);
      const uint32_t r = wcnt[warp * 257 + d] + lt;
      __syncwarp();
      if (lt == 0) wcnt[warp * 257 + d] = r + __popc(peers);
      __syncwarp();
      dr[it] = d | (r << 9);
    }
    bar_sync<3, kTileThreads>();  // all warps' counts, and lstart
    // Thread (h, v), v = tid & 255, turns wcnt[w][v] of the warps w = 8h .. 8h+7 into the tile-local
    // start of warp w's items with digit v.
    const uint32_t v = tid & 255u, h = tid >> 8;
    uint32_t run = lstart[v];
    if (h == 0) {
      uint32_t s = 0;
#pragma unroll
      for (int j = 0; j < 8; ++j) s += wcnt[j * 257 + v];
      half0[v] = s;
    }
    bar_sync<1, kThreads>();
    if (h) run += half0[v];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const uint32_t x = wcnt[(h * 8 + j) * 257 + v];
      wcnt[(h * 8 + j) * 257 + v] = run;
      run += x;
    }
    bar_sync<1, kThreads>();
    // the tile in digit order, as places
#pragma unroll
    for (int it = 0; it < kItems; ++it) {
      const uint32_t d = dr[it] & 511u;
      if (d < 256) sidx[wcnt[warp * 257 + d] + (dr[it] >> 9)] = (uint16_t)(p0 + it * 32);
    }
  } else {
    bar_sync<4, kTileThreads>();
    const uint32_t v = tid - kThreads, w = v >> 5;
    const uint32_t total_v = cnt[v];
    st_status(status + tile * 256 + v, st_word(tile == 0 ? kStIncl : kStAgg, tag, total_v));
    uint32_t incl = total_v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
      if (lane >= o) incl += y;
    }
    if (lane == 31) wsum[w] = incl;
    bar_sync<2, kLook>();
    uint32_t excl = incl - total_v;
    for (uint32_t x = 0; x < w; ++x) excl += wsum[x];
    lstart[v] = excl;
    bar_arrive<3, kTileThreads>();
    // global offset of the digit value
    unsigned long long pre = 0;
    if (tile > 0) {
      pre = lookback_by8(status + v, tile, total_v, tag, ctrl);
      st_status(status + tile * 256 + v, st_word(kStIncl, tag, pre + total_v));
    }
    gstart[v] = dbase[v] + pre - excl;  // output index of the tile's place j with digit v: gstart[v] + j
  }
  __syncthreads();
#pragma unroll 2
  for (uint32_t j = tid; j < left; j += kTileThreads) {
    const Rec r = rec[sidx[j]];
    const uint32_t dv = (uint32_t)(RecT<R>::key(r) >> shift) & 255u;
    const uint64_t pos = gstart[dv] + j;
    if (pos < nout) dst[pos] = r;
  }
}

template <int R>
inline uint32_t radix_tile_smem() {
  using Rec = typename RecT<R>::T;
  return kTile * sizeof(Rec) + 256 * 8 + (kWarps * 257 + 257 + 512 + 8) * 4 + kTile * 2;
}

}  // namespace rtile
using namespace rtile;
}  // namespace bos
