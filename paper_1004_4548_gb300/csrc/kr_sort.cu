// Term ordering (Sec. 3.1: the factors are sorted by ascending code so that
// the output is written in order and each block of output codes meets a
// contiguous range of each factor, the property behind the disjoint output
// intervals of Sec. 4).  Three sorts, chosen per operand by the host:
//  * bitmap: keys are distinct and their range fits an on-chip bitmap; the
//    rank of a key is the number of set bits below it (one pass, O(n + range/32));
//  * bitonic: (key << idx_bits | index) words, n <= 16384: tiles sorted by a
//    bitonic network in the shared memory of a cluster's CTAs, and ranked
//    against one another;
//  * radix: device-wide LSD radix sort of (key, payload) pairs, 8-bit digits,
//    also used for the hash-path output.
// Plus a single-CTA exclusive scan used by the compaction and the radix sort.
#include <cooperative_groups.h>

#include "kr_internal.cuh"
#include "kr_plan.h"

namespace kr {

namespace cg = cooperative_groups;

// ---------------------------------------------------------------------------
// block-wide exclusive scan of int64 values held one per thread
// ---------------------------------------------------------------------------
template <int NT>
__device__ __forceinline__ int64_t block_exclusive_scan(int64_t v, int64_t* total) {
  __shared__ int64_t warp_sums[NT / 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int64_t x = v;
  for (int o = 1; o < 32; o <<= 1) {
    int64_t y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) warp_sums[warp] = x;
  __syncthreads();
  if (warp == 0) {
    int64_t s = lane < NT / 32 ? warp_sums[lane] : 0;
    for (int o = 1; o < 32; o <<= 1) {
      int64_t y = __shfl_up_sync(0xffffffffu, s, o);
      if (lane >= o) s += y;
    }
    if (lane < NT / 32) warp_sums[lane] = s;
  }
  __syncthreads();
  int64_t base = warp > 0 ? warp_sums[warp - 1] : 0;
  if (total) *total = warp_sums[NT / 32 - 1];
  __syncthreads();
  return base + x - v;
}

// ---------------------------------------------------------------------------
// single-CTA exclusive scan of d[0, n); d[n] is not touched; *total = sum
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(1024) k_scan_exclusive(int64_t* __restrict__ d, int64_t n,
                                                         int64_t* __restrict__ total) {
  const int64_t per = (n + blockDim.x - 1) / blockDim.x;
  const int64_t a = min(n, per * threadIdx.x), b = min(n, a + per);
  int64_t s = 0;
  for (int64_t i = a; i < b; ++i) s += d[i];
  int64_t tot;
  int64_t run = block_exclusive_scan<1024>(s, &tot);
  for (int64_t i = a; i < b; ++i) {
    int64_t x = d[i];
    d[i] = run;
    run += x;
  }
  if (threadIdx.x == 0 && total) *total = tot;
}

// ---------------------------------------------------------------------------
// multi-CTA exclusive scan for long arrays: block sums, a scan of the sums,
// then each block scanned with its offset.  scratch: scan_scratch_entries(n).
// ---------------------------------------------------------------------------
constexpr int SC_THREADS = 1024;
constexpr int SC_ITEMS = 8;
constexpr int64_t SC_BLOCK = (int64_t)SC_THREADS * SC_ITEMS;
constexpr int64_t SC_ONE_CTA_MAX = 65536;

int64_t scan_scratch_entries(int64_t n) { return (n + SC_BLOCK - 1) / SC_BLOCK + 1; }

__global__ void __launch_bounds__(SC_THREADS) k_scan_sums(const int64_t* __restrict__ d, int64_t n,
                                                          int64_t* __restrict__ sums) {
  const int64_t b0 = blockIdx.x * SC_BLOCK;
  int64_t s = 0;
#pragma unroll
  for (int r = 0; r < SC_ITEMS; ++r) {
    const int64_t i = b0 + (int64_t)r * SC_THREADS + threadIdx.x;
    if (i < n) s += d[i];
  }
  int64_t tot;
  block_exclusive_scan<SC_THREADS>(s, &tot);
  if (threadIdx.x == 0) sums[blockIdx.x] = tot;
}

__global__ void __launch_bounds__(SC_THREADS) k_scan_blocks(int64_t* __restrict__ d, int64_t n,
                                                            const int64_t* __restrict__ sums) {
  // each thread scans SC_ITEMS consecutive values
  const int64_t i0 = blockIdx.x * SC_BLOCK + (int64_t)threadIdx.x * SC_ITEMS;
  int64_t v[SC_ITEMS];
  int64_t s = 0;
#pragma unroll
  for (int r = 0; r < SC_ITEMS; ++r) {
    v[r] = i0 + r < n ? d[i0 + r] : 0;
    s += v[r];
  }
  int64_t run = sums[blockIdx.x] + block_exclusive_scan<SC_THREADS>(s, nullptr);
#pragma unroll
  for (int r = 0; r < SC_ITEMS; ++r) {
    if (i0 + r < n) d[i0 + r] = run;
    run += v[r];
  }
}

cudaError_t launch_scan_exclusive(int64_t* d, int64_t n, int64_t* dtotal, int64_t* scratch, cudaStream_t s) {
  if (n <= SC_ONE_CTA_MAX || !scratch) {
    k_scan_exclusive<<<1, 1024, 0, s>>>(d, n, dtotal);
    return cudaGetLastError();
  }
  const int64_t nb = (n + SC_BLOCK - 1) / SC_BLOCK;
  k_scan_sums<<<(unsigned)nb, SC_THREADS, 0, s>>>(d, n, scratch);
  k_scan_exclusive<<<1, 1024, 0, s>>>(scratch, nb, dtotal);   // offsets of the blocks, and the total
  k_scan_blocks<<<(unsigned)nb, SC_THREADS, 0, s>>>(d, n, scratch);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// bitmap rank sort (one CTA per operand).  Shared memory: the bitmap (32-bit
// words, padded to groups of 32 words) and, per 8 words, the number of set
// bits before them, so the rank of a key costs at most 8 popcounts.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(1024) k_bitmap_sort(Prod* __restrict__ prods,
                                                      const OpRef* __restrict__ ops) {
  extern __shared__ uint32_t sm[];
  const OpRef r = ops[blockIdx.x];
  Prod& P = prods[r.prod];
  Operand& O = r.which ? P.g : P.f;
  const int64_t nwords = (O.key_range + 31) >> 5;
  const int64_t ngroups = (nwords + 31) >> 5;
  const int64_t nw = ngroups * 32;       // padded bitmap words
  const int64_t n8 = nw >> 3;            // 8-word blocks
  uint32_t* bits = sm;
  uint32_t* pre8 = sm + nw;
  for (int64_t w = threadIdx.x; w < nw; w += blockDim.x) bits[w] = 0;
  __syncthreads();
  uint32_t dup = 0;
  for (int64_t i = threadIdx.x; i < O.n; i += blockDim.x) {
    const uint64_t key = O.skey[i];
    const uint32_t bit = 1u << (key & 31);
    const uint32_t old = atomicOr(&bits[key >> 5], bit);
    if (old & bit) dup = 1;
  }
  __syncthreads();
  // set bits per 8-word block, each thread over a contiguous range of blocks,
  // then an exclusive scan over the threads
  const int64_t per = (n8 + blockDim.x - 1) / blockDim.x;
  const int64_t ba = min(n8, per * threadIdx.x), bb = min(n8, ba + per);
  int64_t s = 0;
  for (int64_t b = ba; b < bb; ++b) {
    const uint4 lo = *(const uint4*)&bits[8 * b];
    const uint4 hi = *(const uint4*)&bits[8 * b + 4];
    const uint32_t c = __popc(lo.x) + __popc(lo.y) + __popc(lo.z) + __popc(lo.w) +
                       __popc(hi.x) + __popc(hi.y) + __popc(hi.z) + __popc(hi.w);
    pre8[b] = c;
    s += c;
  }
  int64_t run = block_exclusive_scan<1024>(s, nullptr);
  for (int64_t b = ba; b < bb; ++b) {
    const uint32_t c = pre8[b];
    pre8[b] = (uint32_t)run;
    run += c;
  }
  __syncthreads();
  for (int64_t i = threadIdx.x; i < O.n; i += blockDim.x) {
    const uint64_t key = O.skey[i];
    const int64_t w = (int64_t)(key >> 5);
    uint32_t rank = pre8[w >> 3];
    for (int64_t x = w & ~(int64_t)7; x < w; ++x) rank += __popc(bits[x]);
    rank += __popc(bits[w] & ((1u << (key & 31)) - 1u));
    if (rank >= O.n) { dup = 1; continue; }
    O.skey2[rank] = key;
    O.sidx2[rank] = (uint64_t)i;
  }
  if (__any_sync(0xffffffffu, dup) && (threadIdx.x & 31) == 0) atomicOr(&P.status, ST_DUP);
}

// ---------------------------------------------------------------------------
// sort of n <= 16384 distinct packed words: the cluster's CTAs sort a tile each
// in shared memory, and a word's rank is its place in its tile plus the numbers
// of smaller words in the others, found through distributed shared memory.
//
// Bound by the chain of barriers (and of remote loads in the searches), so the
// tiles are small: 45 to 66 steps of one or two pairs a thread, those within a
// warp's 64 words without a CTA barrier, then 10 to 12 search steps over all
// the other tiles at once.  One CTA sorting the whole operand took 78 to 91
// steps of up to 8 pairs (both operands of 6188 terms: 93 -> 32 us, 2311 and 1507
// terms: 48 -> 20 us).  Up to BS_MIN terms a cluster has nothing to share.
// ---------------------------------------------------------------------------
constexpr int BS_THREADS = 512;
constexpr int BS_CTAS = 8;                         // the portable cluster size
constexpr int BS_TILE = BITONIC_MAX_N / BS_CTAS;   // words of a tile at most (16 KB)
constexpr int BS_MIN = 512;                        // words that one CTA sorts alone: a pair or less a thread

template <int CTAS>
__global__ void __cluster_dims__(CTAS, 1, 1) __launch_bounds__(BS_THREADS)
    k_bitonic_sort(Prod* __restrict__ prods, const OpRef* __restrict__ ops) {
  __shared__ uint64_t sk[BS_TILE];
  const int rank = (int)(blockIdx.x % CTAS);
  const OpRef r = ops[blockIdx.x / CTAS];
  Prod& P = prods[r.prod];
  Operand& O = r.which ? P.g : P.f;
  const int n = (int)O.n;
  const int tile = max((n + CTAS - 1) / CTAS, BS_MIN);
  const int lo = min(rank * tile, n), m = min(tile, n - lo);
  for (int i = threadIdx.x; i < m; i += BS_THREADS) sk[i] = O.skey[lo + i];
  __syncthreads();
  // all merges ascending: a place at or above m holds no word and is never
  // compared, so padding to a power of two needs no storage
  auto order = [&](int i, int j) {
    if (j < m) {
      const uint64_t a = sk[i], b = sk[j];
      if (a > b) { sk[i] = b; sk[j] = a; }
    }
  };
  // 32 pairs in sequence lie in 64 words in sequence where the words of a pair
  // are that near, and a warp has the same pairs in every such step
  auto barrier = [](bool own, bool next_own) {
    if (own && next_own) __syncwarp(); else __syncthreads();
  };
  for (int lg = 1; (1 << (lg - 1)) < m; ++lg) {
    const int size = 1 << lg, half = size >> 1;
    int pairs = half;
    while (2 * pairs < m) pairs <<= 1;
    // merge two ascending runs: compare i with its mirror in the block of `size`
    for (int p = threadIdx.x; p < pairs; p += BS_THREADS) {
      const int blk = (p >> (lg - 1)) << lg, off = p & (half - 1);
      order(blk + off, blk + size - 1 - off);
    }
    barrier(size <= 64, true);   // (the step after it spans size / 4, or is the mirror of 4)
    for (int ls = lg - 2; ls >= 0; --ls) {
      const int stride = 1 << ls;
      for (int p = threadIdx.x; p < pairs; p += BS_THREADS) {
        const int i = ((p >> ls) << (ls + 1)) + (p & (stride - 1));
        order(i, i + stride);
      }
      barrier(stride <= 32, ls > 0 ? stride <= 64 : size <= 32);
    }
  }
  __syncthreads();
  if (CTAS == 1 || n <= tile) {   // (uniform over the cluster: the others have no words)
    for (int i = threadIdx.x; i < m; i += BS_THREADS) O.skey[lo + i] = sk[i];
    return;
  }
  cg::cluster_group cl = cg::this_cluster();
  cl.sync();   // every tile is sorted; and every word of O.skey is read before any is written
  const uint64_t* peer[CTAS];
  int len[CTAS];
#pragma unroll
  for (int c = 0; c < CTAS; ++c) {
    peer[c] = cl.map_shared_rank(sk, c);
    len[c] = c == rank ? 0 : max(0, min(tile, n - c * tile));
  }
  int top = 1;
  while (2 * top <= tile) top <<= 1;
  for (int i = threadIdx.x; i < m; i += BS_THREADS) {
    const uint64_t x = sk[i];
    int below[CTAS];
#pragma unroll
    for (int c = 0; c < CTAS; ++c) below[c] = 0;
    for (int step = top; step > 0; step >>= 1) {
#pragma unroll
      for (int c = 0; c < CTAS; ++c) {
        const int t = below[c] + step;
        if (t <= len[c] && peer[c][t - 1] < x) below[c] = t;
      }
    }
    int at = i;
#pragma unroll
    for (int c = 0; c < CTAS; ++c) at += below[c];
    O.skey[at] = x;
  }
  cl.sync();   // no CTA leaves while its tile is searched
}

cudaError_t launch_sort_bitmap(Prod* dprods, const OpRef* dops, int nops, size_t smem, cudaStream_t s) {
  if (nops <= 0) return cudaSuccess;
  cudaError_t e = raise_smem_limit((const void*)k_bitmap_sort, (size_t)smem);
  if (e != cudaSuccess) return e;
  k_bitmap_sort<<<nops, 1024, smem, s>>>(dprods, dops);
  return cudaGetLastError();
}

cudaError_t launch_sort_bitonic(Prod* dprods, const OpRef* dops, int nops, int64_t max_n, cudaStream_t s) {
  if (nops <= 0) return cudaSuccess;
  if (max_n <= BS_MIN) k_bitonic_sort<1><<<nops, BS_THREADS, 0, s>>>(dprods, dops);
  else k_bitonic_sort<BS_CTAS><<<(unsigned)nops * BS_CTAS, BS_THREADS, 0, s>>>(dprods, dops);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// device-wide LSD radix sort, 8-bit digits, stable
// counts layout: counts[digit * ntiles + tile]
// ---------------------------------------------------------------------------
constexpr int RS_THREADS = 256;
constexpr int RS_ITEMS = RADIX_TILE / RS_THREADS;   // 16 rounds of 256 elements

__global__ void __launch_bounds__(RS_THREADS) k_rs_hist(const uint64_t* __restrict__ key, int64_t n,
                                                        int shift, int64_t ntiles,
                                                        int64_t* __restrict__ counts) {
  __shared__ uint32_t h[256];
  for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    h[threadIdx.x] = 0;
    __syncthreads();
    const int64_t base = tile * RADIX_TILE;
    for (int r = 0; r < RS_ITEMS; ++r) {
      const int64_t i = base + r * RS_THREADS + threadIdx.x;
      if (i < n) atomicAdd(&h[(key[i] >> shift) & 255], 1u);
    }
    __syncthreads();
    counts[(int64_t)threadIdx.x * ntiles + tile] = h[threadIdx.x];
    __syncthreads();
  }
}

__global__ void __launch_bounds__(RS_THREADS) k_rs_scatter(const uint64_t* __restrict__ key,
                                                           const uint64_t* __restrict__ val, int64_t n,
                                                           int shift, int64_t ntiles,
                                                           const int64_t* __restrict__ offs,
                                                           uint64_t* __restrict__ key_out,
                                                           uint64_t* __restrict__ val_out) {
  constexpr int NW = RS_THREADS / 32;
  __shared__ int64_t base[256];
  __shared__ uint32_t wcount[NW][256];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t lt = (1u << lane) - 1u;
  for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    base[threadIdx.x] = offs[(int64_t)threadIdx.x * ntiles + tile];
    const int64_t t0 = tile * RADIX_TILE;
    for (int r = 0; r < RS_ITEMS; ++r) {
      for (int d = lane; d < 256; d += 32) wcount[warp][d] = 0;
      __syncthreads();
      const int64_t i = t0 + r * RS_THREADS + threadIdx.x;
      const bool ok = i < n;
      uint64_t k = 0, v = 0;
      int d = 256;
      if (ok) { k = key[i]; v = val[i]; d = (int)((k >> shift) & 255); }
      const uint32_t peers = __match_any_sync(0xffffffffu, d);
      const uint32_t rank = __popc(peers & lt);
      if (ok && rank == 0) wcount[warp][d] = __popc(peers);
      __syncthreads();
      {
        // per digit: exclusive offsets over the warps, advance the tile base
        const int dd = threadIdx.x;
        int64_t run = 0;
        for (int w = 0; w < NW; ++w) {
          uint32_t c = wcount[w][dd];
          wcount[w][dd] = (uint32_t)run;
          run += c;
        }
        // base[dd] is read below by every thread; advance after the reads
        __syncthreads();
        if (ok) {
          const int64_t pos = base[d] + wcount[warp][d] + rank;
          key_out[pos] = k;
          val_out[pos] = v;
        }
        __syncthreads();
        base[dd] += run;
      }
      __syncthreads();
    }
  }
}

int64_t radix_scan_entries(int64_t n) {
  const int64_t e = 256 * ((n + RADIX_TILE - 1) / RADIX_TILE);
  return e + 1 + scan_scratch_entries(e);   // digit counts, their total, the scan's block sums
}

cudaError_t radix_sort_pairs(uint64_t* key, uint64_t* val, uint64_t* key_tmp, uint64_t* val_tmp,
                             int64_t n, int bits, int64_t* dscan, cudaStream_t s,
                             bool* result_in_tmp) {
  *result_in_tmp = false;
  if (n <= 1 || bits <= 0) return cudaSuccess;
  const int64_t ntiles = (n + RADIX_TILE - 1) / RADIX_TILE;
  const int grid = (int)(ntiles < 152 * 8 ? ntiles : 152 * 8);
  uint64_t *ki = key, *vi = val, *ko = key_tmp, *vo = val_tmp;
  for (int shift = 0; shift < bits; shift += 8) {
    k_rs_hist<<<grid, RS_THREADS, 0, s>>>(ki, n, shift, ntiles, dscan);
    cudaError_t e = launch_scan_exclusive(dscan, 256 * ntiles, dscan + 256 * ntiles, dscan + 256 * ntiles + 1, s);
    if (e != cudaSuccess) return e;
    k_rs_scatter<<<grid, RS_THREADS, 0, s>>>(ki, vi, n, shift, ntiles, dscan, ko, vo);
    uint64_t* t = ki; ki = ko; ko = t;
    t = vi; vi = vo; vo = t;
    *result_in_tmp = !*result_in_tmp;
  }
  return cudaGetLastError();
}

}  // namespace kr
