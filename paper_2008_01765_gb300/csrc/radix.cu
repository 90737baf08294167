// Stable LSD radix sort on the record key (the non-oblivious sort of Section 3.3), sm_103a.
//
// Onesweep organisation: one histogram pass gives the counts of all 8-bit digits at once; each
// digit then takes one pass that ranks a tile of records stably per digit (one ballot per digit
// bit + per-warp counters), finds the tile's global offset per digit by decoupled look-back over
// the tiles in ticket order, puts the records' places in digit order and writes the tile out in runs.
// A digit on which every key agrees is skipped (the pass would be the identity); the buffers
// alternate so that the last pass that runs writes the final output.
#include "common.cuh"
#include "internal.h"
#include "radix_tile.cuh"

namespace bos {

namespace {

constexpr int kHistCtas = 4 * 152;

// Counts of every 8-bit digit of the keys in records [lo, hi), added to a.hist.
template <int R>
__device__ __forceinline__ void radix_hist_body(const RadixArgs& a, uint64_t lo, uint64_t hi, uint64_t step) {
  using Rec = typename RecT<R>::T;
  constexpr int D = RecT<R>::kDigits;
  __shared__ uint32_t h[D][256];
  for (int x = threadIdx.x; x < D * 256; x += kThreads) (&h[0][0])[x] = 0;
  __syncthreads();
  const Rec* in = reinterpret_cast<const Rec*>(a.in);
  for (uint64_t idx = lo + threadIdx.x; idx < hi; idx += step) {
    const auto key = RecT<R>::key(in[idx]);
#pragma unroll
    for (int d = 0; d < D; ++d) atomicAdd(&h[d][(key >> (8 * d)) & 255u], 1u);
  }
  __syncthreads();
  for (int x = threadIdx.x; x < D * 256; x += kThreads) {
    const uint32_t c = (&h[0][0])[x];
    if (c) atomicAdd(a.hist + x, c);
  }
}

template <int R>
__global__ void __launch_bounds__(kThreads) radix_hist_kernel(RadixArgs a) {
  // grid-stride over the whole array: block b handles b*kThreads + j*gridDim*kThreads + tid
  const uint64_t step = (uint64_t)gridDim.x * kThreads;
  radix_hist_body<R>(a, (uint64_t)blockIdx.x * kThreads, a.n, step);
}

// Batched: block b counts chunk b - first[j] (kTile records) of array j.
template <int R>
__global__ void __launch_bounds__(kThreads) radix_hist_batched_kernel(BatchRadix br) {
  __shared__ uint32_t j_s;
  __shared__ unsigned long long c_s;
  if (threadIdx.x == 0) {
    uint32_t lo = 0, hi = br.narr;
    while (hi - lo > 1) {
      const uint32_t mid = (lo + hi) >> 1;
      if (br.first[mid] <= blockIdx.x) lo = mid; else hi = mid;
    }
    j_s = lo;
    c_s = blockIdx.x - br.first[lo];
  }
  __syncthreads();
  const RadixArgs& a = br.args[j_s];
  const uint64_t lo = c_s * kTile, hi = lo + kTile < a.n ? lo + kTile : a.n;
  radix_hist_body<R>(a, lo, hi, kThreads);
}

// Per digit: exclusive offsets of the 256 digit values, and whether the digit is live.
__global__ void __launch_bounds__(256) radix_prep_kernel(RadixArgs a) {
  const int d = blockIdx.x;
  __shared__ uint32_t s[256];
  __shared__ uint32_t any_full;
  const int v = threadIdx.x;
  const uint32_t c = a.hist[d * 256 + v];
  s[v] = c;
  if (v == 0) any_full = 0;
  __syncthreads();
  if ((uint64_t)c == a.n) any_full = 1;
  // inclusive scan (Hillis-Steele)
  for (int o = 1; o < 256; o <<= 1) {
    const uint32_t y = v >= o ? s[v - o] : 0;
    __syncthreads();
    s[v] += y;
    __syncthreads();
  }
  a.dbase[d * 256 + v] = s[v] - c;
  if (v == 0 && !any_full) atomicOr(&a.ctrl->radix_live, 1u << d);
}

// One tile of one live digit of the LSD chain (the whole CTA).
template <int R>
__device__ __forceinline__ void radix_pass_body(const RadixArgs& a, uint32_t digit, uint64_t tile) {
  using Rec = typename RecT<R>::T;
  const uint32_t live = a.ctrl->radix_live;
  // Buffer chain: X_nlive = buf0 (output); X_j alternates backwards. This pass maps X_c -> X_c+1.
  const uint32_t nlive = __popc(live);
  const uint32_t c = __popc(live & ((1u << digit) - 1));
  auto X = [&](uint32_t j) -> Rec* {
    return reinterpret_cast<Rec*>(((nlive - j) & 1) ? a.buf1 : a.buf0);
  };
  radix_tile<R>(X(c), X(c + 1), a.n, tile, 8 * digit, digit + 1, a.status, a.dbase + digit * 256, a.n, a.ctrl);
}

template <int R>
// Persistent: CTAs take tiles by ticket until none is left (tiles start in ticket order, so every
// look-back waits only on tiles already taken by running CTAs).
__global__ void __launch_bounds__(kTileThreads, 2) radix_pass_kernel(RadixArgs a, uint32_t digit) {
  __shared__ unsigned long long t_s;
  // a constant digit is skipped; so is every LSD pass when the hybrid sort runs instead
  if (!((a.ctrl->radix_live >> digit) & 1u) || a.ctrl->sort_mode) return;
  const uint64_t tiles = (a.n + kTile - 1) / kTile;
  while (true) {
    if (threadIdx.x == 0) t_s = atomicAdd(&a.ctrl->tickets[a.ticket_base + digit], 1u);
    __syncthreads();
    const unsigned long long t = t_s;
    if (t >= tiles) break;
    radix_pass_body<R>(a, digit, t);
    __syncthreads();
  }
}

// Batched: every digit pass of the arrays whose plans leave their keys to the LSD sort (br.lsd: the digits
// any of them takes), in one launch that returns at once when there is none: eight launches that did so
// took 34 us of a batch of 64 small arrays. Tickets run over the digits, then over all tiles of all
// arrays, so inside every array the tiles start in order (the look-back stops at the array's tile 0). A
// tile of an array's later digit waits until all its tiles of the digit before are written: their tickets
// are lower, so running CTAs hold them and the wait ends. Arrays that another sort takes (sort_mode) and
// constant digits are passed over.
constexpr uint32_t kTicketDone = 57;  // ctrl word: tiles an array has written

template <int R>
__global__ void __launch_bounds__(kTileThreads, 2) radix_pass_batched_kernel(BatchRadix br) {
  __shared__ unsigned long long t_s;
  __shared__ uint32_t j_s, d_s;
  const uint32_t lsd = *br.lsd;
  if (!lsd) return;
  while (true) {
    if (threadIdx.x == 0) {
      const uint32_t t = atomicAdd(br.ticket, 1u), x = t / (uint32_t)br.nblocks, tile = t % (uint32_t)br.nblocks;
      uint32_t left = lsd;
      for (uint32_t y = 0; y < x && left; ++y) left &= left - 1;  // the x-th digit, if there is one
      uint32_t lo = 0, hi = br.narr;
      while (hi - lo > 1) {
        const uint32_t mid = (lo + hi) >> 1;
        if (br.first[mid] <= tile) lo = mid; else hi = mid;
      }
      j_s = left ? lo : 0xFFFFFFFFu;
      d_s = left ? (uint32_t)__ffs(left) - 1u : 0u;
      t_s = tile - br.first[lo];
    }
    __syncthreads();
    if (j_s == 0xFFFFFFFFu) break;
    const RadixArgs& a = br.args[j_s];
    const uint32_t digit = d_s, live = a.ctrl->radix_live;
    if (((live >> digit) & 1u) && !a.ctrl->sort_mode) {
      uint32_t* done = &a.ctrl->tickets[kTicketDone];
      const uint32_t before = __popc(live & ((1u << digit) - 1)) * (uint32_t)((a.n + kTile - 1) / kTile);
      if (before) {
        if (threadIdx.x == 0) {
          uint32_t spins = 0, v;
          while (true) {
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(done) : "memory");
            if (v >= before) break;
            if (++spins > kSpinLimit) {
              atomicExch(&a.ctrl->timeout, 1u);  // gives up: the result is not valid
              break;
            }
            if (spins > 16) __nanosleep(64);
          }
        }
        __syncthreads();
        __threadfence();  // no line of an earlier digit is left in L1
      }
      radix_pass_body<R>(a, digit, t_s);
      __syncthreads();
      if (threadIdx.x == 0) {
        __threadfence();
        atomicAdd(done, 1u);
      }
    }
    __syncthreads();
  }
}

template <int R>
uint32_t pass_smem() {
  return radix_tile_smem<R>();
}

}  // namespace

uint64_t radix_tiles(uint64_t n, int) { return (n + kTile - 1) / kTile; }

cudaError_t launch_radix_hist(const RadixArgs& a, int R, cudaStream_t st) {
  const uint64_t need = (a.n + kThreads - 1) / kThreads;
  const unsigned grid = (unsigned)(need < (uint64_t)kHistCtas ? (need ? need : 1) : kHistCtas);
  if (R == 8)
    radix_hist_kernel<8><<<grid, kThreads, 0, st>>>(a);
  else
    radix_hist_kernel<16><<<grid, kThreads, 0, st>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_radix_batched(const BatchRadix& br, int R, int stage, cudaStream_t st) {
  if (br.narr == 0) return cudaSuccess;
  if (stage == 0) {  // histograms: one block per chunk of kTile records
    if (br.nblocks == 0) return cudaSuccess;
    if (R == 8)
      radix_hist_batched_kernel<8><<<(unsigned)br.nblocks, kThreads, 0, st>>>(br);
    else
      radix_hist_batched_kernel<16><<<(unsigned)br.nblocks, kThreads, 0, st>>>(br);
  } else {  // the digit passes
    if (br.nblocks == 0) return cudaSuccess;
    int dev = 0, sms = 0;
    cudaError_t e0 = cudaGetDevice(&dev);
    if (e0 == cudaSuccess) e0 = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e0 != cudaSuccess) return e0;
    const unsigned grid = (unsigned)(br.nblocks < 2ull * sms ? br.nblocks : 2ull * sms);  // two CTAs per SM
    if (R == 8) {
      const uint32_t sm = pass_smem<8>();
      cudaError_t e = set_smem_optin(radix_pass_batched_kernel<8>);
      if (e != cudaSuccess) return e;
      radix_pass_batched_kernel<8><<<grid, kTileThreads, sm, st>>>(br);
    } else {
      const uint32_t sm = pass_smem<16>();
      cudaError_t e = set_smem_optin(radix_pass_batched_kernel<16>);
      if (e != cudaSuccess) return e;
      radix_pass_batched_kernel<16><<<grid, kTileThreads, sm, st>>>(br);
    }
  }
  return cudaGetLastError();
}

cudaError_t launch_radix_prep(const RadixArgs& a, int R, cudaStream_t st) {
  radix_prep_kernel<<<R == 8 ? RecT<8>::kDigits : RecT<16>::kDigits, 256, 0, st>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_radix_pass(const RadixArgs& a, int R, uint32_t digit, cudaStream_t st) {
  const uint64_t tiles = radix_tiles(a.n, R);
  if (tiles == 0) return cudaSuccess;
  int dev = 0, sms = 0;
  cudaError_t e0 = cudaGetDevice(&dev);
  if (e0 == cudaSuccess) e0 = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e0 != cudaSuccess) return e0;
  const unsigned grid = (unsigned)(tiles < 2ull * sms ? tiles : 2ull * sms);  // two CTAs per SM
  if (R == 8) {
    const uint32_t sm = pass_smem<8>();
    cudaError_t e = set_smem_optin(radix_pass_kernel<8>);
    if (e != cudaSuccess) return e;
    radix_pass_kernel<8><<<grid, kTileThreads, sm, st>>>(a, digit);
  } else {
    const uint32_t sm = pass_smem<16>();
    cudaError_t e = set_smem_optin(radix_pass_kernel<16>);
    if (e != cudaSuccess) return e;
    radix_pass_kernel<16><<<grid, kTileThreads, sm, st>>>(a, digit);
  }
  return cudaGetLastError();
}

}  // namespace bos
