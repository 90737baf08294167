// In-bin permutation table of the fused LAST pass (Section 3.2), sm_103a.
//
// Final bucket b ends the butterfly with its m reals at slots 0..m-1 in stable order. Slot s has
// the key r(b, s) = (w0 << 32 | w1) of Philox(b*Z + s, attempt, stream 1), and the reals leave
// the bucket ordered by (r, s). The keys depend on neither the data nor the routing, so this
// kernel sorts each final bucket's slots by (r, s) ahead of the LAST pass, at full occupancy,
// and the LAST pass only filters its rows.
//
// Row b of the table lists slots in key order, Z entries of u16. The LAST pass keeps the entries
// below m; dropping the others keeps their relative order, so either of two rows serves:
//   * reals only (the pass has input tags): final_load_kernel reads the LAST pass's input tags and
//     counts m for every final bucket exactly as the LAST pass will (the label digit of every
//     real); the table kernel sorts slots 0..m-1 and pads the row with 0xFFFF;
//   * all slots (a single pass that draws the labels itself): slots 0..Z-1 sorted.
// One warp sorts one final bucket with no block-wide barrier: it draws the keys, counts the top 9
// bits of w0 into 512 bins of its own (16 bits each), scans them, places each slot in its bin, and
// puts each slot at its bin's start plus its rank among the bin's few members (compared by
// (w0, w1, s)).
// Bound by issue (63 % of the cycles) at 24 warps per SM, which the 9 KB of a warp allow. n = 2^24,
// Z = 1024: 150 us (167 with 256 bins). Fewer warps with the keys in bin order (12 KB each) took a third
// longer, keys in registers (32 unrolled rows) missed the instruction cache and took 204 us.
#include "common.cuh"
#include "internal.h"

namespace bos {

namespace {

constexpr int kPBins = 512;        // bins: top 9 bits of w0
constexpr int kShift = 23;
constexpr int kPWords = kPBins / 2;  // two 16-bit bins per word
constexpr uint32_t kMaxK = 12;     // final buckets per LAST subproblem: at most 2^12

// Slot s3 sorts before slot s2 (same bucket, base = b*Z, equal w0): smaller w1, or equal w1 and
// s3 < s2. Rare (equal 32-bit words), so out of line.
__device__ __noinline__ bool tie_less(uint64_t base, uint32_t s3, uint32_t s2, uint32_t attempt, uint64_t seed) {
  const uint32_t l2 = philox_at(base + s2, attempt, 1, seed).w1;
  const uint32_t l3 = philox_at(base + s3, attempt, 1, seed).w1;
  return (l3 < l2) || (l3 == l2 && s3 < s2);
}

// warps per CTA and shared memory: per warp Z keys (u32), Z placed slots and Z row entries (u16),
// 512 bins
__host__ __device__ inline uint32_t table_warps(uint32_t Z) { return Z <= 1024 ? 8u : (Z <= 2048 ? 4u : 2u); }
__host__ __device__ inline uint32_t warp_bytes(uint32_t Z) { return Z * 8 + kPWords * 4; }
uint32_t table_smem(uint32_t Z) { return table_warps(Z) * warp_bytes(Z); }

constexpr int kLT = 256;     // threads of the load-count kernel
constexpr int kLUnroll = 8;  // 16-byte tag loads in flight per thread

// load[q*D + u] = reals of LAST subproblem q whose routing digit is u, for every subproblem q:
// the reals of its input buckets s*2^i + t (s < D, q = G*2^i + t) with label bits [shift, shift+k)
// equal to u, as the LAST pass counts them. With a.status, the subproblems are taken by ticket and
// status[q] gets the inclusive prefix of their reals (loads above Z, an overflow, count as Z).
template <bool TRACE>
__device__ __forceinline__ void final_load_unit(const PermTableArgs& a, uint64_t q) {
  extern __shared__ __align__(16) unsigned char smem[];
  uint32_t* mcnt = reinterpret_cast<uint32_t*>(smem);
  const uint32_t Z = a.Z, D = 1u << a.k, cpb = Z / 4;  // 16-byte chunks per input bucket
  const uint32_t shift = a.L - a.i - a.k;
  const int tid = threadIdx.x;
  for (uint32_t x = tid; x < D; x += kLT) mcnt[x] = 0;
  __syncthreads();
  const uint64_t t = q & ((1ull << a.i) - 1), G = q >> a.i;
  if (TRACE && tid == 0)
    for (uint32_t s = 0; s < D; ++s)
      trace_log<TRACE>(a.trace, kRead, a.buf_tag, Z * 4, ((G << (a.i + a.k)) + ((uint64_t)s << a.i) + t) * Z * 4);
  const uint32_t nchunk = D * cpb;
  for (uint32_t c0 = tid; c0 < nchunk; c0 += kLT * kLUnroll) {
    uint4 v[kLUnroll];
#pragma unroll
    for (int e = 0; e < kLUnroll; ++e) {
      const uint32_t c = c0 + e * kLT;
      v[e] = make_uint4(kDummy, kDummy, kDummy, kDummy);
      if (c < nchunk) {
        const uint32_t s = c / cpb, off = c - s * cpb;
        const uint64_t gb = (G << (a.i + a.k)) + ((uint64_t)s << a.i) + t;
        v[e] = reinterpret_cast<const uint4*>(a.tag + gb * Z)[off];  // Z multiple of 32: aligned
      }
    }
#pragma unroll
    for (int e = 0; e < kLUnroll; ++e) {
      const uint32_t w[4] = {v[e].x, v[e].y, v[e].z, v[e].w};
#pragma unroll
      for (int f = 0; f < 4; ++f)
        if (w[f] != kDummy) atomicAdd(&mcnt[(w[f] >> shift) & (D - 1)], 1u);
    }
  }
  __syncthreads();
  for (uint32_t x = tid; x < D; x += kLT) a.load[q * D + x] = mcnt[x];
  if (a.status && tid < 32) {
    uint32_t total = 0;
    for (uint32_t x = tid; x < D; x += 32) total += min(mcnt[x], Z);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) total += __shfl_xor_sync(0xFFFFFFFFu, total, o);
    if (tid == 0) {
      if (q == 0) {
        if (!a.skip_publish) st_status(a.status, st_word(kStIncl, 0, total));
      } else {
        st_status(a.status + q, st_word(kStAgg, 0, total));
        const unsigned long long pre = lookback_window<8>(a.status, q, 1, 0, a.ctrl);
        st_status(a.status + q, st_word(kStIncl, 0, pre + total));
      }
    }
  }
}

template <bool TRACE>
__global__ void __launch_bounds__(kLT) final_load_kernel(PermTableArgs a) {
  __shared__ uint32_t q_s;
  const uint64_t units = a.B >> a.k;
  uint64_t q = blockIdx.x;
  while (true) {
    if (a.status) {
      if (threadIdx.x == 0) q_s = atomicAdd(a.ticket, 1u);
      __syncthreads();
      q = q_s;
    }
    if (q >= units) break;
    final_load_unit<TRACE>(a, q);
    __syncthreads();  // the counts are cleared for the next subproblem
    q += gridDim.x;
  }
}

// The table's arguments of a batch's array.
__device__ __forceinline__ PermTableArgs table_args(const PassArgs& p) {
  PermTableArgs a{};
  a.bucket0 = p.bucket0;
  a.ord = const_cast<uint16_t*>(p.ord);
  a.tag = p.in_tag;
  a.load = const_cast<uint32_t*>(p.load);
  a.B = p.B;
  a.Z = p.Z;
  a.attempt = p.attempt;
  a.i = p.i;
  a.k = p.k;
  a.L = p.L;
  a.buf_tag = p.buf_in_tag;
  a.seed = p.seed;
  a.trace = p.trace;
  a.status = p.status;
  a.ctrl = p.ctrl;
  return a;
}

// Many arrays: units by ticket, in array order, so that every look-back predecessor has started.
template <bool TRACE>
__global__ void __launch_bounds__(kLT) final_load_batched_kernel(const BatchLast* args, const uint2* units, uint32_t nunits,
                                                                 uint32_t* ticket) {
  __shared__ uint32_t t_s;
  while (true) {
    if (threadIdx.x == 0) t_s = atomicAdd(ticket, 1u);
    __syncthreads();
    const uint32_t t = t_s;
    if (t >= nunits) break;
    const uint2 un = units[t];
    final_load_unit<TRACE>(table_args(args[un.x].a), un.y);
    __syncthreads();
  }
}

// The row of final bucket b, sorted by one warp in its shared memory at wbase.
template <bool TRACE>
__device__ __forceinline__ void table_row(const PermTableArgs& a, uint64_t b, unsigned char* wbase) {
  const uint32_t Z = a.Z;
  const int lane = threadIdx.x & 31;
  uint32_t* key = reinterpret_cast<uint32_t*>(wbase);               // [Z] w0 of each slot
  uint32_t* bins = key + Z;                                         // [kPWords] starts, then ends
  uint16_t* placed = reinterpret_cast<uint16_t*>(bins + kPWords);   // [Z] slots grouped by bin
  uint16_t* row = placed + Z;                                       // [Z] the sorted row
  const bool tagged = a.tag != nullptr;

  {
    const uint64_t base = (a.bucket0 + b) * Z;  // the keys' counters use the global bucket
    const uint32_t m = tagged ? min(a.load[b], Z) : Z;
    for (int x = lane; x < kPWords; x += 32) bins[x] = 0;
    __syncwarp();
    // keys and bin counts (four independent Philox chains per lane per step)
    for (uint32_t s0 = lane; s0 < m; s0 += 128) {
      uint32_t w[4];
#pragma unroll
      for (int c = 0; c < 4; ++c) w[c] = s0 + c * 32 < m ? philox_at(base + s0 + c * 32, a.attempt, 1, a.seed).w0 : 0u;
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const uint32_t s = s0 + c * 32;
        if (s < m) {
          key[s] = w[c];
          atomicAdd(&bins[w[c] >> (kShift + 1)], 1u << (((w[c] >> kShift) & 1u) * 16));
        }
      }
    }
    __syncwarp();
    {  // exclusive scan of the bins: eight consecutive words (sixteen bins) per lane
      uint32_t v[kPWords / 32], sum = 0;
#pragma unroll
      for (int e = 0; e < kPWords / 32; ++e) {
        v[e] = bins[lane * (kPWords / 32) + e];
        sum += v[e];  // packed: both halves stay below 2^16
      }
      sum = (sum & 0xFFFFu) + (sum >> 16);
      uint32_t incl = sum;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
        if (lane >= o) incl += y;
      }
      uint32_t run = incl - sum;
#pragma unroll
      for (int e = 0; e < kPWords / 32; ++e) {
        bins[lane * (kPWords / 32) + e] = run | (run + (v[e] & 0xFFFFu)) << 16;
        run += (v[e] & 0xFFFFu) + (v[e] >> 16);
      }
    }
    __syncwarp();
    // slots grouped by bin (any order inside a bin); bins[] becomes each bin's end. Four slots
    // per lane per step: independent chains.
    for (uint32_t s0 = lane; s0 < m; s0 += 128) {
      uint32_t p[4];
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const uint32_t s = s0 + c * 32;
        const uint32_t b = s < m ? key[s] >> kShift : 0u, h = (b & 1u) * 16;
        p[c] = s < m ? (atomicAdd(&bins[b >> 1], 1u << h) >> h) & 0xFFFFu : 0u;
      }
#pragma unroll
      for (int c = 0; c < 4; ++c)
        if (s0 + c * 32 < m) placed[p[c]] = (uint16_t)(s0 + c * 32);
    }
    __syncwarp();
    // each slot's final place: its bin's start plus the members of the bin that sort before it
    for (uint32_t s0 = lane; s0 < m; s0 += 128) {
      uint32_t ks[4], start[4], end[4], rank[4];
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const uint32_t s = s0 + c * 32;
        ks[c] = s < m ? key[s] : 0u;
        const uint32_t bin = ks[c] >> kShift;
        const uint16_t* ends = reinterpret_cast<const uint16_t*>(bins);
        start[c] = s < m && bin ? ends[bin - 1] : 0u;
        end[c] = s < m ? ends[bin] : 0u;
        rank[c] = 0;
      }
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const uint32_t s = s0 + c * 32;
        for (uint32_t e = start[c]; e < end[c]; ++e) {
          const uint32_t o = placed[e], ko = key[o];
          rank[c] += (ko < ks[c] || (ko == ks[c] && o != s && tie_less(base, o, s, a.attempt, a.seed))) ? 1u : 0u;
        }
      }
#pragma unroll
      for (int c = 0; c < 4; ++c)
        if (s0 + c * 32 < m) row[start[c] + rank[c]] = (uint16_t)(s0 + c * 32);
    }
    for (uint32_t s = m + lane; s < Z; s += 32) row[s] = 0xFFFFu;  // no real at these ranks
    __syncwarp();
    // Z is a multiple of 32: the bucket's row is whole 16-byte words, 16-byte aligned
    uint4* dst = reinterpret_cast<uint4*>(a.ord + b * Z);
    const uint4* src = reinterpret_cast<const uint4*>(row);
    for (uint32_t x = lane; x < Z / 8; x += 32) dst[x] = src[x];
    if (lane == 0) trace_log<TRACE>(a.trace, kWrite, kBufPerm, Z * 2, b * Z * 2);
    __syncwarp();  // the warp's next bucket reuses its arrays
  }
}

template <bool TRACE>
__global__ void __launch_bounds__(256, 3) perm_table_kernel(PermTableArgs a) {
  extern __shared__ __align__(16) unsigned char smem[];
  const uint32_t W = table_warps(a.Z), warp = threadIdx.x >> 5;
  for (uint64_t b = (uint64_t)blockIdx.x * W + warp; b < a.B; b += (uint64_t)gridDim.x * W)
    table_row<TRACE>(a, b, smem + warp * warp_bytes(a.Z));
}

// Many arrays: a CTA per unit (the final buckets of one LAST subproblem).
template <bool TRACE>
__global__ void __launch_bounds__(256, 3) perm_table_batched_kernel(const BatchLast* args, const uint2* units, uint32_t stride) {
  extern __shared__ __align__(16) unsigned char smem[];
  const uint2 un = units[blockIdx.x];
  const PermTableArgs a = table_args(args[un.x].a);
  const uint32_t D = 1u << a.k, W = blockDim.x >> 5, warp = threadIdx.x >> 5;
  for (uint32_t u = warp; u < D; u += W) table_row<TRACE>(a, (uint64_t)un.y * D + u, smem + warp * stride);
}

}  // namespace

template <bool TRACE>
cudaError_t perm_table_launch(const PermTableArgs& a, cudaStream_t st) {
  int dev = 0, sms = 0, occ = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  if (a.tag) {  // final loads first
    const uint32_t D = 1u << a.k;
    const uint32_t sm = D * 4;
    if ((e = set_smem_optin(final_load_kernel<TRACE>)) != cudaSuccess) return e;
    if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, final_load_kernel<TRACE>, kLT, sm)) != cudaSuccess)
      return e;
    const uint64_t units = a.B >> a.k, want = (uint64_t)sms * (occ > 0 ? occ : 1);
    final_load_kernel<TRACE><<<(unsigned)(units < want ? units : want), kLT, sm, st>>>(a);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  const uint32_t sm = table_smem(a.Z), W = table_warps(a.Z);
  if ((e = set_smem_optin(perm_table_kernel<TRACE>)) != cudaSuccess) return e;
  if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, perm_table_kernel<TRACE>, W * 32, sm)) != cudaSuccess)
    return e;
  const uint64_t need = (a.B + W - 1) / W, want = (uint64_t)sms * (occ > 0 ? occ : 1);
  perm_table_kernel<TRACE><<<(unsigned)(need < want ? need : want), W * 32, sm, st>>>(a);
  return cudaGetLastError();
}

template <bool TRACE>
static cudaError_t table_batched(const BatchLast* args, const uint2* units, uint32_t nunits, uint32_t max_k, uint32_t max_Z,
                                 uint32_t* ticket, cudaStream_t st) {
  int dev = 0, sms = 0, occ = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  const uint32_t sl = (1u << max_k) * 4;
  if ((e = set_smem_optin(final_load_batched_kernel<TRACE>)) != cudaSuccess) return e;
  if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, final_load_batched_kernel<TRACE>, kLT, sl)) != cudaSuccess)
    return e;
  const uint32_t want = (uint32_t)sms * (occ > 0 ? occ : 1);
  final_load_batched_kernel<TRACE><<<nunits < want ? nunits : want, kLT, sl, st>>>(args, units, nunits, ticket);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  const uint32_t W = table_warps(max_Z), stride = warp_bytes(max_Z);
  if ((e = set_smem_optin(perm_table_batched_kernel<TRACE>)) != cudaSuccess) return e;
  perm_table_batched_kernel<TRACE><<<nunits, W * 32, W * stride, st>>>(args, units, stride);
  return cudaGetLastError();
}

cudaError_t launch_perm_table_batched(const BatchLast* args, const uint2* units, uint32_t nunits, uint32_t max_k,
                                      uint32_t max_Z, uint32_t* ticket, cudaStream_t st, bool trace) {
  if (nunits == 0) return cudaSuccess;
  return trace ? table_batched<true>(args, units, nunits, max_k, max_Z, ticket, st)
               : table_batched<false>(args, units, nunits, max_k, max_Z, ticket, st);
}

cudaError_t launch_perm_table(const PermTableArgs& a, cudaStream_t st, bool trace) {
  if (a.B == 0) return cudaSuccess;
  if (a.Z % 32 != 0 || a.Z > 4096 || (a.tag && (a.k > kMaxK || !a.load))) return cudaErrorInvalidValue;
  return trace ? perm_table_launch<true>(a, st) : perm_table_launch<false>(a, st);
}

}  // namespace bos
