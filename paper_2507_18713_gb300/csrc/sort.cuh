// sort.cuh -- stable LSD radix sort of (64-bit key, 32-bit value) pairs, 8 bits
// per pass, used by the tile rasteriser and the device scene build.
#pragma once

#include <cuda_runtime.h>

#include "scan.cuh"

namespace salf_sort {

constexpr int kSortThreads = 256;
constexpr int kSortItems = 4;      // items per thread (8 and 16: 3 us more per 1.2M-pair sort, 2: 17)
constexpr int kSortTile = kSortThreads * kSortItems;
constexpr int kRadixBits = 8;
constexpr int kRadix = 1 << kRadixBits;

// LSD radix sort of the pairs, 8 bits per pass.  A block owns kSortTile
// consecutive items, a warp a run of kSortItems x 32 of them (round r, lane l
// holds item 32 r + l of the run), so the order of (warp, round, lane) is the
// input order and the scatter below keeps it among equal digits (stable).
// Per pass: counts, their scan (one block per digit), scatter.

// Digit counts of each block's items (hist[digit * nblk + block]).
static __global__ void __launch_bounds__(kSortThreads) k_radix_hist(const unsigned long long* __restrict__ keys,
                                                             long long n, int shift,
                                                             unsigned* __restrict__ hist, int nblk) {
  __shared__ unsigned h[kRadix];
  for (int d = threadIdx.x; d < kRadix; d += kSortThreads) h[d] = 0;
  __syncthreads();
  const long long base = (long long)blockIdx.x * kSortTile;
#pragma unroll
  for (int r = 0; r < kSortItems; ++r) {
    const long long i = base + (long long)r * kSortThreads + threadIdx.x;
    if (i < n) atomicAdd(&h[(unsigned)(keys[i] >> shift) & (kRadix - 1)], 1u);
  }
  __syncthreads();
  for (int d = threadIdx.x; d < kRadix; d += kSortThreads) hist[d * nblk + blockIdx.x] = h[d];
}

// Per digit (blockIdx.x): exclusive scan of its blocks' counts, and its total.
static __global__ void __launch_bounds__(kSortThreads) k_radix_scan(const unsigned* __restrict__ hist,
                                                                    int nblk,
                                                                    unsigned* __restrict__ hoff,
                                                                    unsigned* __restrict__ total) {
  const unsigned* in = hist + (long long)blockIdx.x * nblk;
  unsigned* out = hoff + (long long)blockIdx.x * nblk;
  unsigned run = 0;
  for (int b0 = 0; b0 < nblk; b0 += kSortThreads) {
    const int b = b0 + (int)threadIdx.x;
    const unsigned c = b < nblk ? in[b] : 0u;
    unsigned sum;
    const unsigned before = salf_scan::block_exclusive_scan<unsigned>(c, &sum);
    if (b < nblk) out[b] = run + before;
    run += sum;
  }
  if (threadIdx.x == 0) total[blockIdx.x] = run;
}

// Stable scatter: item goes to (items of smaller digits) + scanned count[digit]
// [block] + (items of this block before it with the same digit).  Lanes with
// equal digits are ranked by a match, rounds and warps by counts in shared
// memory: three block barriers per tile instead of five per round.  Bound by the
// scattered writes (12 us a pass for 1.2M pairs, as before; the scan of the counts
// took three kernels and 8 us a pass, now one and 3).
static __global__ void __launch_bounds__(kSortThreads) k_radix_scatter(
    const unsigned long long* __restrict__ kin, const unsigned* __restrict__ vin,
    unsigned long long* __restrict__ kout, unsigned* __restrict__ vout, long long n, int shift,
    const unsigned* __restrict__ hoff, const unsigned* __restrict__ total, int nblk) {
  constexpr int kWarps = kSortThreads / 32;
  static_assert(kRadix == kSortThreads, "one thread per digit");
  __shared__ unsigned s_cnt[kWarps][kRadix];  // counts, then first positions
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  for (int k = threadIdx.x; k < kWarps * kRadix; k += kSortThreads) (&s_cnt[0][0])[k] = 0;
  unsigned all;
  const unsigned first = salf_scan::block_exclusive_scan<unsigned>(total[threadIdx.x], &all) +
                         hoff[(long long)threadIdx.x * nblk + blockIdx.x];
  // (the scan's barriers also order the zeroing above)
  const long long base = (long long)blockIdx.x * kSortTile + wid * (kSortItems * 32) + lane;
  unsigned long long key[kSortItems];
  unsigned val[kSortItems], rank[kSortItems];
#pragma unroll
  for (int r = 0; r < kSortItems; ++r) {
    const bool ok = base + 32 * r < n;
    key[r] = ok ? kin[base + 32 * r] : 0ull;
    val[r] = ok ? vin[base + 32 * r] : 0u;
  }
#pragma unroll
  for (int r = 0; r < kSortItems; ++r) {
    const bool ok = base + 32 * r < n;
    const unsigned d = ok ? (unsigned)(key[r] >> shift) & (kRadix - 1) : (unsigned)kRadix;
    const unsigned peers = __match_any_sync(0xffffffffu, d);
    const int leader = __ffs(peers) - 1;
    unsigned old = 0;
    if (ok && lane == leader) {
      old = s_cnt[wid][d];
      s_cnt[wid][d] = old + __popc(peers);
    }
    rank[r] = __shfl_sync(0xffffffffu, old, leader) + __popc(peers & ((1u << lane) - 1u));
    __syncwarp();
  }
  __syncthreads();
  unsigned run = first;
#pragma unroll
  for (int w = 0; w < kWarps; ++w) {
    const unsigned c = s_cnt[w][threadIdx.x];
    s_cnt[w][threadIdx.x] = run;
    run += c;
  }
  __syncthreads();
#pragma unroll
  for (int r = 0; r < kSortItems; ++r) {
    if (base + 32 * r >= n) break;
    const unsigned pos = s_cnt[wid][(unsigned)(key[r] >> shift) & (kRadix - 1)] + rank[r];
    kout[pos] = key[r];
    vout[pos] = val[r];
  }
}

// Workspace of radix_sort_pairs for n pairs: the histogram and its scan.
inline long long radix_hist_elems(long long n) {
  const long long nblk = (n + kSortTile - 1) / kSortTile;
  return (long long)kRadix * (nblk > 0 ? nblk : 1);
}

// Sorts (ka, va) by the low `bits` bits of the keys, ping-ponging with (kb,
// vb); returns through *keys / *vals the buffers that hold the result.  hist
// and hoff hold radix_hist_elems(n) elements, htmp kRadix.
inline cudaError_t radix_sort_pairs(unsigned long long* ka, unsigned* va, unsigned long long* kb,
                                    unsigned* vb, long long n, int bits, unsigned* hist,
                                    unsigned* hoff, unsigned* htmp, cudaStream_t st,
                                    int* launches, unsigned long long** keys, unsigned** vals) {
  const long long nblk = (n + kSortTile - 1) / kSortTile;
  const int passes = (bits + kRadixBits - 1) / kRadixBits;
  unsigned long long *ki = ka, *ko = kb;
  unsigned *vi = va, *vo = vb;
  for (int pass = 0; pass < passes && n > 0; ++pass) {
    const int shift = kRadixBits * pass;
    k_radix_hist<<<(unsigned)nblk, kSortThreads, 0, st>>>(ki, n, shift, hist, (int)nblk);
    k_radix_scan<<<kRadix, kSortThreads, 0, st>>>(hist, (int)nblk, hoff, htmp);
    k_radix_scatter<<<(unsigned)nblk, kSortThreads, 0, st>>>(ki, vi, ko, vo, n, shift, hoff, htmp,
                                                             (int)nblk);
    *launches += 3;
    unsigned long long* tk = ki;
    ki = ko;
    ko = tk;
    unsigned* tv = vi;
    vi = vo;
    vo = tv;
  }
  *keys = ki;
  *vals = vi;
  return cudaGetLastError();
}

}  // namespace salf_sort
