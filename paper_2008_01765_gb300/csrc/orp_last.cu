// Last ORP pass with known final loads (sm_103a): the last k <= 5 butterfly levels, the in-bin
// permutation (Section 3.2) and the strip, streaming its input.
//
// Subproblem q = G*2^i + t reads the input buckets G*2^(i+k) + s*2^i + t (s < 2^k) and produces the
// final buckets q*2^k + u, u = the label's low k bits, stable by (s, slot). perm_table.cu has counted
// every final bucket's reals and found every subproblem's output offset ahead of this pass, so a real
// of bucket u with stable rank s has its place in a packed tile at once: tile[base[u] + s], base = the
// exclusive prefix of the loads. The tile holds the subproblem's reals only (half of its slots), so
// one CTA takes 2^k buckets where the cluster kernel (orp_fast.cu) needs up to four, and no
// look-back, tag tile or filter is left. The finished tile is gathered in table order into one
// contiguous run of the output.
//
// A batch is one, two or four input buckets (at most 2048 slots), brought in by TMA bulk copies:
//   A  every row of 32 slots is ranked by ballots (k + 1 of them: at most 32 digits); lane d stores
//      the row's count of digit d;
//   -- barrier; one warp per digit scans its column over the rows and adds the bucket's fill;
//   -- barrier; B: the records go to the tile. A of the next batch follows without a barrier.
// Counts and offsets come from the digits alone; every global address depends on (n, Z, k) and the
// final loads (Lemma 3.3). Overflow (MergeSplit: more than Z reals) is checked for every level from the
// column totals, as in the other pass kernels.
//
// What bounds it: latency (ranking and scan, about 1400 cycles per input bucket of 1024 slots in
// batches of two, where the copy bandwidth would allow 1500 for all it moves) and the copy-out, which
// does not overlap the batches. n = 2^29 16-byte records, Z = 1024, k = 4: 9.44 ms (12.1 with the
// cluster kernel, C = 2); n = 2^26, k = 3: 0.96 ms (4196 GB/s) against 3.15 for the cluster kernel at
// k = 1, which the planner gave it; 2^24, Z = 512, k = 4: 0.28 ms (1.56).
//
// A subproblem with more reals than the tile (the planner leaves 2.5 standard deviations) is run in
// parts, each a run of its final buckets that fits, reading its input once per part.
#include <cmath>

#include "common.cuh"
#include "internal.h"

namespace bos {
namespace {

constexpr int kLT = 512;             // worker threads; one more warp issues the copies and checks the levels
constexpr int kLW = kLT / 32;
constexpr int kLThreads = kLT + 32;
constexpr uint32_t kBatchSlots = 2048;
constexpr uint32_t kItems = kBatchSlots / kLT;
constexpr uint32_t kRows = kBatchSlots / 32;
constexpr uint32_t kMaxK = 5;        // one lane per digit
constexpr uint32_t kMaxStages = 4;
constexpr uint32_t kSmemLimit = 232448 - 1024;

inline uint32_t l_align(uint32_t x, uint32_t a) { return (x + a - 1) / a * a; }

inline uint32_t isqrt_up(uint32_t x) {  // the smallest r with r * r >= x
  uint32_t r = (uint32_t)std::sqrt((double)x);
  while (r * r < x) ++r;
  return r;
}

// cap = 0: this k does not fit.
LastLayout last_layout(int R, uint32_t Z, uint32_t k) {
  const uint32_t D = 1u << k, mean = D * Z / 2, dev = isqrt_up(mean);
  LastLayout l{};
  l.stride = D + 2;
  const uint32_t fixed = 2 * kRows * l.stride * 2 + 2 * (D + 1) * 4 + D * 4 + 128 + 256;
  // as many buckets per batch as leave three stages beside the tile, two or four stages deep
  for (int lub = 2; lub >= 0; --lub) {
    if ((1u << lub) > D || (Z << lub) > kBatchSlots) continue;
    const uint32_t sb = l_align((Z << lub) * (4 + R), 128);
    for (uint32_t st = kMaxStages; st >= (lub ? 3u : 2u); --st) {
      if (st > (D >> lub)) continue;
      if (fixed + st * sb >= kSmemLimit) continue;
      const uint32_t room = (kSmemLimit - fixed - st * sb) / R / 16 * 16;
      if (room < mean + 5 * dev / 2 || room < Z) continue;
      const uint32_t want = l_align(mean + 6 * dev, 16) > Z ? l_align(mean + 6 * dev, 16) : l_align(Z, 16);
      l.cap = want < room ? want : room;
      l.stages = st;
      l.lub = (uint32_t)lub;
      l.stage_bytes = sb;
      uint32_t off = l_align(l.cap * R, 128);
      l.stage = off;
      off += st * sb;
      l.cnt = off;
      off += 2 * kRows * l.stride * 2;
      l.base = l_align(off, 16);
      off = l.base + 2 * (D + 1) * 4;
      l.fill = off;
      off += D * 4;
      l.misc = l_align(off, 16);
      l.total = l.misc + 96;
      return l;
    }
  }
  return l;
}

// Subproblems q0, q0 + qstep, .. below nsub of one array.
template <int R, int K, bool TRACE>
__device__ __forceinline__ void orp_last_body(const PassArgs& a, const LastLayout& lay, const uint64_t q0,
                                              const uint64_t nsub, const uint32_t qstep) {
  using Rec = typename RecT<R>::T;
  extern __shared__ __align__(128) unsigned char smem[];
  constexpr uint32_t k = K, D = 1u << k;
  const uint32_t Z = a.Z, i = a.i;
  const uint32_t shift = a.L - i - k;
  Rec* tile = reinterpret_cast<Rec*>(smem);                         // [cap]
  uint16_t* cnt = reinterpret_cast<uint16_t*>(smem + lay.cnt);      // [2][kRows][stride] counts, then offsets
  uint32_t* base = reinterpret_cast<uint32_t*>(smem + lay.base);    // [2][D + 1] prefix of the loads, per subproblem parity
  uint32_t* fill = reinterpret_cast<uint32_t*>(smem + lay.fill);    // [D] reals seen per final bucket
  unsigned long long* bars = reinterpret_cast<unsigned long long*>(smem + lay.misc);           // [stages]

  const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const bool worker = warp < kLW;
  const uint32_t lub = lay.lub, ub = 1u << lub, NB = D >> lub, nst = lay.stages;
  const uint32_t nslot = ub * Z, nrow = nslot / 32;
  const Rec* in_rec = reinterpret_cast<const Rec*>(a.in_rec);

  if (tid < D) fill[tid] = 0;
  if (tid == 0) {
    for (uint32_t s = 0; s < nst; ++s) mbar_init(smem_u32(bars + s), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();

  // TMA of batch s of subproblem q into stage st (one thread of the last warp)
  auto issue = [&](uint64_t q, uint32_t s, uint32_t st) {
    const uint32_t bar = smem_u32(bars + st);
    const uint32_t dst = smem_u32(smem + lay.stage + st * lay.stage_bytes);
    const uint64_t t = q & ((1ull << i) - 1), G = q >> i;
    mbar_expect_tx(bar, ub * Z * (4 + R));
    for (uint32_t b = 0; b < ub; ++b) {
      const uint64_t bk = (G << (i + k)) + ((uint64_t)((s << lub) + b) << i) + t;
      tma_load(dst + b * Z * 4, a.in_tag + bk * Z, Z * 4, bar);
      tma_load(dst + ub * Z * 4 + b * Z * R, in_rec + bk * Z, Z * R, bar);
      trace_log<TRACE>(a.trace, kRead, a.buf_in_tag, Z * 4, bk * Z * 4);
      trace_log<TRACE>(a.trace, kRead, a.buf_in_rec, Z * R, bk * Z * R);
    }
  };
  // The last warp: prefix of subproblem q's loads into base[par]; its table rows on their way to L2.
  auto fetch_loads = [&](uint64_t q, uint32_t par) {
    const uint32_t m = lane < D ? min(a.load[q * D + lane], Z) : 0u;
    uint32_t incl = m;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
      if (lane >= (uint32_t)o) incl += y;
    }
    uint32_t* b = base + par * (D + 1);
    if (lane < D) b[lane + 1] = incl;
    if (lane == 0) {
      b[0] = 0;
      const uint64_t row = q * D * (uint64_t)Z;
      asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(a.ord + row), "r"(D * Z * 2) : "memory");
      trace_log<TRACE>(a.trace, kRead, kBufPerm, D * Z * 2, row * 2);
    }
  };

  // A pass over a subproblem's input serves the part [u0, u1) of its final buckets. The next pass is
  // another part of the same subproblem (rare) or the CTA's next subproblem; `ahead` batches, counted
  // from the current pass's first, have been requested, nst of them in flight (nst <= NB).
  uint64_t q = q0;
  if (q >= nsub) return;  // (the grid never exceeds nsub)
  uint32_t sp = 0;              // subproblem parity
  uint32_t st = 0, ph = 0;      // stage and parity of the next batch
  uint32_t cb = 0;              // count buffer of the next batch
  uint32_t u0 = 0, u1 = 0;
  uint32_t ahead = nst;
  if (!worker) {
    fetch_loads(q, 0);
    if (lane == 0)
      for (uint32_t x = 0; x < nst; ++x) issue(q, x, x);
  }
  __syncthreads();

  while (true) {
    const uint32_t* bs = base + sp * (D + 1);
    // the part: as many final buckets as fit the tile (all of them but for rare subproblems)
    u1 = D;
    while (bs[u1] - bs[u0] > lay.cap) --u1;
    const bool ends = u1 == D;  // the subproblem's last part
    const uint64_t qn = ends ? q + qstep : q;  // the next pass's subproblem
    uint32_t a1 = 0, a2 = 0, a3 = 0, a4 = 0;  // the last warp: reals per group of 2, 4, 8, 16 digits

    uint32_t dr[kItems];  // digit | rank inside the row << 8; 0xFFFFFFFF: dummy
    for (uint32_t s = 0; s <= NB; ++s) {
      const uint32_t pst = st == 0 ? nst - 1 : st - 1;
      if (worker && s > 0) {
        // ---- B: the previous batch's records into the tile ----
        const Rec* srec = reinterpret_cast<const Rec*>(smem + lay.stage + pst * lay.stage_bytes + ub * Z * 4);
        const uint16_t* c = cnt + (cb ^ 1) * kRows * lay.stride;
#pragma unroll
        for (uint32_t j = 0; j < kItems; ++j) {
          const uint32_t r = j * kLW + ((warp - j * (Z / 64)) & (kLW - 1));
          if (dr[j] != 0xFFFFFFFFu) {
            const uint32_t u = dr[j] & 255u, slot = c[r * lay.stride + u] + (dr[j] >> 8);
            if (u >= u0 && u < u1 && slot < bs[u + 1] - bs[u])  // (more: the bucket overflowed)
              tile[bs[u] - bs[u0] + slot] = srec[r * 32 + lane];
          }
        }
      }
      if (s == NB) break;
      // ---- A: rank every row of the batch ----
      if (worker) {
        mbar_wait(smem_u32(bars + st), ph, a.ctrl);
        const uint32_t* stag = reinterpret_cast<const uint32_t*>(smem + lay.stage + st * lay.stage_bytes);
        uint16_t* c = cnt + cb * kRows * lay.stride;
#pragma unroll
        for (uint32_t j = 0; j < kItems; ++j) {
          const uint32_t r = j * kLW + ((warp - j * (Z / 64)) & (kLW - 1));
          dr[j] = 0xFFFFFFFFu;
          if (r < nrow) {
            const uint32_t tg = stag[r * 32 + lane];
            const bool real = tg != kDummy;
            uint32_t peers = __ballot_sync(0xFFFFFFFFu, real), mine = peers;
            if (peers) {
              const uint32_t u = (tg >> shift) & (D - 1);
#pragma unroll
              for (uint32_t b = 0; b < k; ++b) {
                const uint32_t bal = __ballot_sync(0xFFFFFFFFu, (u >> b) & 1u);
                peers &= (u >> b) & 1u ? bal : ~bal;
                mine &= (lane >> b) & 1u ? bal : ~bal;
              }
              if (real) dr[j] = u | __popc(peers & lanemask_lt()) << 8;
            }
            if (lane < D) c[r * lay.stride + lane] = (uint16_t)__popc(mine);
          }
        }
      }
      __syncthreads();  // S1: the counts are whole; the previous batch's stage is free
      if (worker) {
        // ---- scan: warp w takes digits w and w + 16; lanes are rows ----
        uint16_t* c = cnt + cb * kRows * lay.stride;
        for (uint32_t d = warp; d < D; d += kLW) {
          const uint32_t f = fill[d];
          const uint32_t v0 = lane < nrow ? c[lane * lay.stride + d] : 0u;
          const uint32_t v1 = lane + 32 < nrow ? c[(lane + 32) * lay.stride + d] : 0u;
          uint32_t x0 = v0, x1 = v1;
#pragma unroll
          for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y0 = __shfl_up_sync(0xFFFFFFFFu, x0, o), y1 = __shfl_up_sync(0xFFFFFFFFu, x1, o);
            if (lane >= (uint32_t)o) {
              x0 += y0;
              x1 += y1;
            }
          }
          const uint32_t t0 = __shfl_sync(0xFFFFFFFFu, x0, 31);
          x0 += f - v0;
          x1 += f + t0 - v1;
          if (lane < nrow) c[lane * lay.stride + d] = (uint16_t)x0;
          if (lane + 32 < nrow) c[(lane + 32) * lay.stride + d] = (uint16_t)x1;
          if (lane == 31) fill[d] = x1 + v1;
        }
      }
      if (s > 0) {  // the previous batch's stage takes batch `ahead`, of this pass or of the next subproblem
        if (ahead < NB) {
          if (tid == kLT) issue(q, ahead, pst);
          ++ahead;
        } else if (ends) {
          if (tid == kLT && qn < nsub) issue(qn, ahead - NB, pst);
          ++ahead;
        }
      }
      __syncthreads();  // S2: the offsets are whole
      if (!worker) {
        // ---- overflow: level l = 1..k-1 buckets gather 2^l input buckets and the digits with a
        // common l-bit prefix; the batch's counts are the growth of the fills ----
        const uint16_t* c = cnt + cb * kRows * lay.stride;
        const uint32_t f = lane < D ? fill[lane] : 0u;
        uint32_t v = lane < D ? (f - c[lane]) & 0xFFFFu : 0u;  // row 0's offset is the fill before the batch
        if (lub == 2 && k > 1) {  // level 1 of a batch of four buckets: its two blocks
          uint32_t lo = lane < D ? (c[(2 * Z / 32) * lay.stride + lane] - c[lane]) & 0xFFFFu : 0u, hi = v - lo;
          for (uint32_t b = 0; b + 1 < k; ++b) {
            lo += __shfl_xor_sync(0xFFFFFFFFu, lo, 1u << b);
            hi += __shfl_xor_sync(0xFFFFFFFFu, hi, 1u << b);
          }
          if (lo > Z || hi > Z) atomicExch(&a.ctrl->overflow, 1u);
        }
        const uint32_t e = __ffs(~s) - 1 + lub;  // levels lub..e end with this batch
        auto level = [&](uint32_t gsz, uint32_t& acc) {
          if (gsz >= k) return;
          v += __shfl_xor_sync(0xFFFFFFFFu, v, 1u << (gsz - 1));
          acc += v;
          const uint32_t l = k - gsz;
          if (l <= e) {
            if (acc > Z && (lub < 2 || l > 1)) atomicExch(&a.ctrl->overflow, 1u);
            acc = 0;
          }
        };
        level(1, a1);
        level(2, a2);
        level(3, a3);
        level(4, a4);
        if (s == NB - 1) {
          if (f > Z) atomicExch(&a.ctrl->overflow, 1u);
          if (ends && qn < nsub) fetch_loads(qn, sp ^ 1);  // the next subproblem's
        }
      }
      cb ^= 1;
      if (++st == nst) {
        st = 0;
        ph ^= 1u;
      }
    }
    __syncthreads();  // the tile is whole; the stages are free; the fills are checked
    // ---- the tile leaves in table order, one contiguous run; the next pass's copies start ----
    if (tid < D) fill[tid] = 0;
    ahead = ends ? ahead - NB : 0;
    if (!worker) {
      if (lane == 0 && qn < nsub)
        for (uint32_t x = ahead; x < nst; ++x) issue(qn, x, (st + x) % nst);
    } else {
      Rec* out = reinterpret_cast<Rec*>(a.out0);
      if (a.out_sel && sort_passes_odd(a.ctrl)) out = reinterpret_cast<Rec*>(a.out1);
      const uint32_t out_buf = (out == reinterpret_cast<Rec*>(a.out0)) ? kBufOut : kBufTmp;
      const uint64_t gofs = (q ? a.status[q - 1] & kStValue : 0ull) + bs[u0];
      // a warp takes a bucket's row (a part of one when there are fewer buckets than warps), kU groups
      // of 32 entries in flight
      constexpr uint32_t kU = 4, kWpb = kLW > D ? kLW / D : 1u;
      for (uint32_t u = warp / kWpb; u < D; u += kLW / kWpb) {
        if (u < u0 || u >= u1) continue;
        const uint32_t b = bs[u] - bs[u0];
        const uint64_t pos = gofs + b;
        uint32_t m = bs[u + 1] - bs[u];
        if (pos + m > a.n) m = pos < a.n ? (uint32_t)(a.n - pos) : 0u;  // only after an overflow
        const uint16_t* row = a.ord + (q * D + u) * Z;
        const Rec* tb = tile + b;
        Rec* ob = out + pos;
        for (uint32_t j0 = warp % kWpb * 32 + lane; j0 < m; j0 += kU * kWpb * 32) {
          uint32_t e[kU];
          Rec rc[kU];
#pragma unroll
          for (uint32_t y = 0; y < kU; ++y) e[y] = j0 + y * kWpb * 32 < m ? row[j0 + y * kWpb * 32] : 0u;
#pragma unroll
          for (uint32_t y = 0; y < kU; ++y) rc[y] = tb[e[y]];
#pragma unroll
          for (uint32_t y = 0; y < kU; ++y)
            if (j0 + y * kWpb * 32 < m) {
              ob[j0 + y * kWpb * 32] = rc[y];
              trace_log<TRACE>(a.trace, kWrite, out_buf, R, (pos + j0 + y * kWpb * 32) * R);
            }
        }
      }
    }
    if (ends) {
      q = qn;
      sp ^= 1;
      u0 = 0;
    } else {
      u0 = u1;
    }
    ahead = nst;
    __syncthreads();  // the tile and the fills are free
    if (q >= nsub) break;
  }
}

template <int R, int K, bool TRACE>
__global__ void __launch_bounds__(kLThreads, 1) orp_last_kernel(const __grid_constant__ PassArgs a,
                                                                const __grid_constant__ LastLayout lay) {
  orp_last_body<R, K, TRACE>(a, lay, blockIdx.x, a.B >> K, gridDim.x);
}

// Many arrays: one CTA per unit, whatever its levels (one launch: a batch of small arrays has few
// subproblems of each level count).
template <int R, bool TRACE>
__global__ void __launch_bounds__(kLThreads, 1) orp_last_batched_kernel(const BatchLast* args, const uint2* units) {
  __shared__ BatchLast sa;
  const uint2 un = units[blockIdx.x];
  for (uint32_t x = threadIdx.x; x < sizeof(BatchLast) / 4; x += kLThreads)
    reinterpret_cast<uint32_t*>(&sa)[x] = reinterpret_cast<const uint32_t*>(args + un.x)[x];
  __syncthreads();
  const uint64_t q = un.y;
  switch (sa.a.k) {
    case 1: orp_last_body<R, 1, TRACE>(sa.a, sa.lay, q, q + 1, 1); break;
    case 2: orp_last_body<R, 2, TRACE>(sa.a, sa.lay, q, q + 1, 1); break;
    case 3: orp_last_body<R, 3, TRACE>(sa.a, sa.lay, q, q + 1, 1); break;
    case 4: orp_last_body<R, 4, TRACE>(sa.a, sa.lay, q, q + 1, 1); break;
    default: orp_last_body<R, 5, TRACE>(sa.a, sa.lay, q, q + 1, 1); break;
  }
}

template <int R, bool TRACE>
cudaError_t last_batched(const BatchLast* args, const uint2* units, uint32_t nunits, uint32_t smem, cudaStream_t st) {
  auto kern = orp_last_batched_kernel<R, TRACE>;
  const cudaError_t e = set_smem_optin(kern);
  if (e != cudaSuccess) return e;
  kern<<<nunits, kLThreads, smem, st>>>(args, units);
  return cudaGetLastError();
}

template <int R, int K, bool TRACE>
cudaError_t last_launch(const PassArgs& a, cudaStream_t st) {
  const LastLayout lay = last_layout(R, a.Z, a.k);
  auto kern = orp_last_kernel<R, K, TRACE>;
  cudaError_t e = set_smem_optin(kern);
  if (e != cudaSuccess) return e;
  int per_sm = 0, sms = 0, dev = 0;
  if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kLThreads, lay.total)) != cudaSuccess) return e;
  if (per_sm <= 0) return cudaErrorInvalidConfiguration;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
  if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
  const uint64_t nsub = a.B >> a.k;
  uint64_t grid = (uint64_t)per_sm * sms;
  if (grid > nsub) grid = nsub;
  kern<<<(unsigned)grid, kLThreads, lay.total, st>>>(a, lay);
  return cudaGetLastError();
}

template <int R, bool TRACE>
cudaError_t last_k(const PassArgs& a, cudaStream_t st) {
  switch (a.k) {
    case 1: return last_launch<R, 1, TRACE>(a, st);
    case 2: return last_launch<R, 2, TRACE>(a, st);
    case 3: return last_launch<R, 3, TRACE>(a, st);
    case 4: return last_launch<R, 4, TRACE>(a, st);
    default: return last_launch<R, 5, TRACE>(a, st);
  }
}

}  // namespace

// Microseconds of one subproblem on one SM (fill: reals per slot). Measured: n = 2^26 16-byte records,
// Z = 1024, k = 3 (four batches of two buckets): 8.9 us; k = 4 (sixteen of one): 21.9; n = 2^24, Z = 512,
// k = 4 (four batches of four buckets): 10.4, k = 5 (sixteen of two): 27.
double orp_last_sub_us(int R, uint32_t Z, uint32_t k, double fill) {
  const LastLayout l = last_layout(R, Z, k);
  const double slots = (double)(Z << l.lub);
  return (double)((1u << k) >> l.lub) * (0.5 + 0.6 * slots / 1024.0) + 0.7 + 0.00045 * R / 16 * fill * Z * (1u << k);
}

uint32_t orp_last_max_k(int R, uint32_t Z) {
  if (Z % 32 != 0 || Z > kBatchSlots) return 0;
  uint32_t best = 0;
  for (uint32_t k = 1; k <= kMaxK; ++k)
    if (last_layout(R, Z, k).cap) best = k;
  return best;
}

LastLayout orp_last_layout(int R, uint32_t Z, uint32_t k) { return last_layout(R, Z, k); }

cudaError_t launch_orp_last_batched(const BatchLast* args, const uint2* units, uint32_t nunits, uint32_t smem,
                                    cudaStream_t st, int R, bool trace) {
  if (nunits == 0) return cudaSuccess;
  if (R == 8) return trace ? last_batched<8, true>(args, units, nunits, smem, st)
                           : last_batched<8, false>(args, units, nunits, smem, st);
  return trace ? last_batched<16, true>(args, units, nunits, smem, st)
               : last_batched<16, false>(args, units, nunits, smem, st);
}

cudaError_t launch_orp_last(const PassArgs& a, cudaStream_t st, int R, bool trace) {
  if (a.k == 0 || a.k > orp_last_max_k(R, a.Z) || a.i + a.k > a.L || !a.load || !a.ord || !a.status)
    return cudaErrorInvalidValue;
  if (R == 8) return trace ? last_k<8, true>(a, st) : last_k<8, false>(a, st);
  return trace ? last_k<16, true>(a, st) : last_k<16, false>(a, st);
}

}  // namespace bos
