// Stable merge sort by key, sm_103a: the comparison-based sort that Section 3.3 composes with the
// ORP (any non-oblivious comparison sort after the permutation gives an oblivious sort; its
// accesses depend only on the relative order of the keys, which the ORP has made random).
//
// Block sort: a CTA sorts a tile of kBT records by (key, place): eight per thread in registers by
// adjacent exchanges, then rounds of pairwise merges of sorted runs in shared memory; the records
// follow once, by the sorted places.
// Merge passes: runs of width w become runs of 2w. Two warps of a chunk's CTA find how many of the
// outputs before the chunk's two ends come from the left run (merge path: a search on the diagonal, 32
// probes a step); the CTA loads its two input ranges, merges places in shared memory and writes the
// chunk. Equal keys always take the left run first, so the sort is stable: equal keys keep the order
// they had after the ORP.
#include "common.cuh"
#include "internal.h"

namespace bos {

namespace {

constexpr int kMT = 256;               // threads per CTA of a merge pass
constexpr int kMI = 8;                 // records per thread
constexpr uint32_t kMC = kMT * kMI;    // merge chunk (2048 records); runs are at least kMC long
constexpr int kBThreads = 512;         // threads per CTA of the block sort
constexpr uint32_t kBT = kBThreads * kMI;  // block-sorted run (4096 records)

// Merge path: of the first d outputs of the stable merge of A[0..na) and B[0..nb) (A first on
// equal keys), how many come from A. key(x): key at place x; A starts at place a, B at place b.
template <typename K>
__device__ __forceinline__ uint32_t merge_split(K key, uint32_t a, uint32_t na, uint32_t b, uint32_t nb, uint32_t d) {
  uint32_t lo = d > nb ? d - nb : 0u, hi = d < na ? d : na;
  while (lo < hi) {
    const uint32_t mid = (lo + hi) >> 1;
    if (!(key(b + d - 1 - mid) < key(a + mid)))  // A[mid] goes before B[d-1-mid]
      lo = mid + 1;
    else
      hi = mid;
  }
  return lo;
}

// The same by a warp, in device memory: 32 probes a step, so 5 steps where one thread takes 21.
template <int R>
__device__ __forceinline__ uint32_t merge_split_warp(const typename RecT<R>::T* A, uint32_t na,
                                                     const typename RecT<R>::T* B, uint32_t nb, uint32_t d) {
  const uint32_t lane = threadIdx.x & 31u;
  uint32_t lo = d > nb ? d - nb : 0u, hi = d < na ? d : na;
  while (lo < hi) {
    const uint32_t q = (hi - lo + 31) / 32;
    const uint32_t mid = lo + lane * q + q - 1;
    bool before = false;
    if (mid < hi) before = !(RecT<R>::key(B[d - 1 - mid]) < RecT<R>::key(A[mid]));
    const uint32_t c = __popc(__ballot_sync(0xFFFFFFFFu, before));  // monotone: the first c probes
    lo += c * q;
    hi = lo + q - 1 < hi ? lo + q - 1 : hi;
  }
  return lo;
}

// Places of the next `cnt` outputs of the stable merge from places i (of [i, ia)) and j (of [j, jb)), two to
// a word, and their keys if KEYS.
template <bool KEYS, typename Key, typename K>
__device__ __forceinline__ void merge_run(K key, uint32_t i, uint32_t ia, uint32_t j, uint32_t jb, uint32_t cnt,
                                          uint32_t (&p)[kMI / 2], Key (&k)[kMI]) {
  Key ka = i < ia ? key(i) : 0, kb = j < jb ? key(j) : 0;
#pragma unroll
  for (int x = 0; x < kMI; ++x) {
    if ((uint32_t)x < cnt) {
      const bool takeA = j >= jb || (i < ia && !(kb < ka));
      const uint32_t pl = takeA ? i : j;
      p[x / 2] = (x & 1) ? p[x / 2] | pl << 16 : pl;
      if (KEYS) k[x] = takeA ? ka : kb;
      if (takeA) {
        if (++i < ia) ka = key(i);
      } else {
        if (++j < jb) kb = key(j);
      }
    }
  }
}

// Place x of the block sort's arrays: one word of padding for every eight, since the threads of a warp
// stand eight places apart.
__device__ __forceinline__ uint32_t pad8(uint32_t x) { return x + (x >> 3); }

// In place allowed (in == out). Bound by the shared-memory rounds (nine, each a search and a merge of
// eight). Keys and 16-bit places move instead of records, without the conflicts of rows 128 B apart: 133 us
// for 2^22 16-byte records with runs of 4096, where sorting records gave 305 us with runs of 2048. Runs of
// 2048 take 113 us and one more pass, runs of 8192 (one CTA an SM) 183 us and one less.
template <int R>
__global__ void __launch_bounds__(kBThreads, 2) merge_block_kernel(const typename RecT<R>::T* in, typename RecT<R>::T* out,
                                                                uint64_t n) {
  using Rec = typename RecT<R>::T;
  using Key = typename RecT<R>::Key;
  extern __shared__ __align__(16) unsigned char smem[];
  Key* keys = reinterpret_cast<Key*>(smem);                                   // [pad8(kBT)]
  uint16_t* place = reinterpret_cast<uint16_t*>(keys + kBT + kBT / 8);        // [pad8(kBT)]
  const uint32_t tid = threadIdx.x;
  const uint64_t t0 = (uint64_t)blockIdx.x * kBT;
  const uint32_t cnt = (uint32_t)(n - t0 < kBT ? n - t0 : kBT);
#pragma unroll
  for (int x = 0; x < kMI; ++x) {
    const uint32_t y = tid + x * kBThreads;
    if (y < cnt) keys[pad8(y)] = RecT<R>::key(in[t0 + y]);
  }
  __syncthreads();
  const uint32_t o = tid * kMI;
  const uint32_t m = o < cnt ? (cnt - o < (uint32_t)kMI ? cnt - o : (uint32_t)kMI) : 0u;
  Key k[kMI];
  uint32_t p[kMI];
#pragma unroll
  for (int x = 0; x < kMI; ++x) {
    p[x] = o + x;
    k[x] = (uint32_t)x < m ? keys[pad8(o) + x] : 0;
  }
  // odd-even transposition: exchanging only strictly out-of-order neighbours keeps it stable
#pragma unroll
  for (int r = 0; r < kMI; ++r) {
#pragma unroll
    for (int x = r & 1; x + 1 < kMI; x += 2) {
      if ((uint32_t)(x + 1) < m && k[x + 1] < k[x]) {
        const Key t = k[x];
        k[x] = k[x + 1];
        k[x + 1] = t;
        const uint32_t u = p[x];
        p[x] = p[x + 1];
        p[x + 1] = u;
      }
    }
  }
#pragma unroll
  for (int x = 0; x < kMI; ++x)
    if ((uint32_t)x < m) {
      keys[pad8(o) + x] = k[x];
      place[pad8(o) + x] = (uint16_t)p[x];
    }
  __syncthreads();
  for (uint32_t w = kMI; w < kBT && w < cnt; w <<= 1) {  // runs of w -> runs of 2w
    uint32_t q[kMI / 2];
    if (m) {
      const uint32_t pb = o / (2 * w) * (2 * w), b0 = pb + w;
      const uint32_t na = cnt - pb < w ? cnt - pb : w;
      const uint32_t nb = b0 < cnt ? (cnt - b0 < w ? cnt - b0 : w) : 0u;
      const uint32_t d = o - pb;
      auto key = [&](uint32_t x) { return keys[pad8(x)]; };
      const uint32_t i = merge_split(key, pb, na, b0, nb, d);
      merge_run<true>(key, pb + i, pb + na, b0 + d - i, b0 + nb, m, q, k);
#pragma unroll
      for (int x = 0; x < kMI; ++x)
        if ((uint32_t)x < m) p[x] = place[pad8((x & 1) ? q[x / 2] >> 16 : q[x / 2] & 0xFFFFu)];
    }
    __syncthreads();  // every read of this round is done
#pragma unroll
    for (int x = 0; x < kMI; ++x)
      if ((uint32_t)x < m) {
        keys[pad8(o) + x] = k[x];
        place[pad8(o) + x] = (uint16_t)p[x];
      }
    __syncthreads();
  }
  Rec v[kMI];
#pragma unroll
  for (int x = 0; x < kMI; ++x) {
    const uint32_t y = tid + x * kBThreads;
    if (y < cnt) v[x] = in[t0 + place[pad8(y)]];
  }
  __syncthreads();  // every record is read before the first is written
#pragma unroll
  for (int x = 0; x < kMI; ++x) {
    const uint32_t y = tid + x * kBThreads;
    if (y < cnt) out[t0 + y] = v[x];
  }
}

// Bound by latency: search, load, search in shared memory, eight dependent steps, copy-out. Only places
// move in the merge (each step reads one key), so five CTAs fit an SM where three did. 37 us a pass of 2^22
// 16-byte records (3.6 TB/s); 73 us with records merged into a second buffer, two key reads a step and the
// ends found by a kernel before it. Six CTAs at 40 registers: 39 us, chunks of 1024 or 4096: 45 or 41 us.
// One chunk of one merge pass (runs of w >= kMC, so a chunk lies inside one pair of runs).
template <int R>
__global__ void __launch_bounds__(kMT, 5) merge_pass_kernel(const typename RecT<R>::T* in, typename RecT<R>::T* out,
                                                         uint64_t n, uint64_t w) {
  using Rec = typename RecT<R>::T;
  using Key = typename RecT<R>::Key;
  extern __shared__ __align__(16) unsigned char smem[];
  Rec* src = reinterpret_cast<Rec*>(smem);                      // [kMC] the chunk's two input ranges
  uint16_t* place = reinterpret_cast<uint16_t*>(src + kMC);     // [kMC] places of the merged chunk
  __shared__ uint32_t split[2];
  const uint32_t tid = threadIdx.x, warp = tid >> 5;
  const uint64_t o0 = (uint64_t)blockIdx.x * kMC, o1 = o0 + kMC < n ? o0 + kMC : n;
  const uint64_t pb = o0 / (2 * w) * (2 * w), b0 = pb + w;
  const uint32_t na = (uint32_t)(n - pb < w ? n - pb : w);
  const uint32_t nb = (uint32_t)(b0 < n ? (n - b0 < w ? n - b0 : w) : 0u);
  if (warp < 2) {
    const uint32_t i = merge_split_warp<R>(in + pb, na, in + b0, nb, (uint32_t)((warp ? o1 : o0) - pb));
    if ((tid & 31u) == 0) split[warp] = i;
  }
  __syncthreads();
  const uint32_t cnt = (uint32_t)(o1 - o0), la = split[1] - split[0], lb = cnt - la;
  const Rec* A = in + pb + split[0];
  const Rec* B = in + b0 + ((uint32_t)(o0 - pb) - split[0]);
#pragma unroll
  for (int x = 0; x < kMI; ++x) {
    const uint32_t y = tid + x * kMT;
    if (y < cnt) cp_async<sizeof(Rec)>(src + y, y < la ? A + y : B + (y - la));
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
  __syncthreads();
  const uint32_t o = tid * kMI;
  if (o < cnt) {
    const uint32_t m = cnt - o < (uint32_t)kMI ? cnt - o : (uint32_t)kMI;
    auto key = [&](uint32_t x) { return RecT<R>::key(src[x]); };
    const uint32_t i = merge_split(key, 0, la, la, lb, o);
    uint32_t q[kMI / 2] = {0, 0, 0, 0};
    Key k[kMI];
    merge_run<false>(key, i, la, la + o - i, cnt, m, q, k);
    *reinterpret_cast<uint4*>(place + o) = make_uint4(q[0], q[1], q[2], q[3]);  // a ragged end fits: o + 8 <= kMC
  }
  __syncthreads();
  for (uint32_t x = tid; x < cnt; x += kMT) out[o0 + x] = src[place[x]];
}

template <int R>
cudaError_t merge_sort_r(const void* in, void* buf0, void* buf1, uint64_t n, cudaStream_t st,
                         const MergeHooks& hooks) {
  using Rec = typename RecT<R>::T;
  const uint32_t passes = merge_passes(n);
  // the block-sorted runs go where an even number of merge passes leaves the result in buf0
  Rec* cur = reinterpret_cast<Rec*>((passes & 1) ? buf1 : buf0);
  Rec* oth = reinterpret_cast<Rec*>((passes & 1) ? buf0 : buf1);
  cudaError_t e = cudaSuccess;
  {
    const uint64_t grid = (n + kBT - 1) / kBT;
    const int ev = hooks.begin ? hooks.begin(st, 0, 2.0 * n * R) : -1;
    if ((e = set_smem_optin(merge_block_kernel<R>)) != cudaSuccess) return e;
    const uint32_t smem = (kBT + kBT / 8) * (sizeof(typename RecT<R>::Key) + 2);
    merge_block_kernel<R><<<(unsigned)grid, kBThreads, smem, st>>>(reinterpret_cast<const Rec*>(in), cur, n);
    if (hooks.end) hooks.end(ev, st);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  if ((e = set_smem_optin(merge_pass_kernel<R>)) != cudaSuccess) return e;
  const uint64_t nchunks = (n + kMC - 1) / kMC;
  for (uint64_t w = kBT; w < n; w <<= 1) {
    const int ev = hooks.begin ? hooks.begin(st, 1, 2.0 * n * R) : -1;
    merge_pass_kernel<R><<<(unsigned)nchunks, kMT, kMC * (sizeof(Rec) + 2), st>>>(cur, oth, n, w);
    if (hooks.end) hooks.end(ev, st);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    Rec* t = cur;
    cur = oth;
    oth = t;
  }
  return cudaSuccess;
}

}  // namespace

uint32_t merge_passes(uint64_t n) {
  uint32_t p = 0;
  for (uint64_t w = kBT; w < n; w <<= 1) ++p;
  return p;
}

cudaError_t launch_merge_sort(const void* in, void* buf0, void* buf1, uint64_t n, int R, cudaStream_t st,
                              const MergeHooks& hooks) {
  if (n == 0) return cudaSuccess;
  return R == 8 ? merge_sort_r<8>(in, buf0, buf1, n, st, hooks)
                : merge_sort_r<16>(in, buf0, buf1, n, st, hooks);
}

}  // namespace bos
