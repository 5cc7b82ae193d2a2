// Windowed accumulation of highly sparse products (Sec. 3.2's hash table, kept
// on chip; the disjoint output intervals of Sec. 4 across CTAs).
//
// A table of the whole product in device memory costs a random
// read-modify-write of HBM or L2 per term pair, clearing, compacting and then
// ordering it.  Here the output key range is cut into windows of about equal
// work, one CTA forms every pair of a window, accumulates it in a small table
// in shared memory and orders the window's terms there.  Nothing is cleared,
// compacted or ordered in device memory.  A window's terms go to the next free
// stretch of a raw array (no CTA waits for another), and one pass puts the
// stretches together in key order: the decode of a single product, or a copy.
//
// Measured on GB300 (whole calls): 6188 x 6188 terms of the weighted sparse
// structure 1.90 -> 1.05 ms, 2311 x 1507 random float64 terms over 2.8e11 keys
// 12.7 -> 0.42 ms (its ordering alone took 11.9), a Poisson product of 5003 x
// 3989 terms (37 M output terms) 6.5 -> 2.0 ms, 20000 x 20000 (597 M terms) 64.5
// -> 43.5 ms.  The window kernel is bound by instruction issue (62% of the issue
// slots; 2 CTAs of 512 threads per SM, 110 KB of shared memory each): forming,
// adding and ordering a pair takes about 20 warp instructions (640 for a row of
// 32), and the walk over the terms that have no partner in a window adds to it.
//
// Pairs of a window.  One factor (the shorter, "A") is walked, the other ("B")
// is searched: for a term a of A the partners that land in [lo, hi) are the
// contiguous range [lower_bound(lo - a), lower_bound(hi - a)) of B's ascending
// codes, found through a bucket index.  A polynomial product is one such
// convolution.  A Poisson product is four per result kind: with the signed
// code u = t Wp + p of a term and v = -t Wp + p of its mirror image (t the
// trig code, p the polynomial code), the keys of the sum terms are uA + uB,
// those of the difference terms uA + vB where tA >= tB and vA + uB where
// tA < tB.  B's lists hold the v codes of its terms (t > 0) followed by the u
// codes, ascending; a term with t = 0 is held twice (its sum and difference
// terms fall on the same key).  Both classes are restricted to the keys that
// are theirs by the window's lower end (key >= 0, or >= Wp where T = 0 is
// excluded: a sine of zero, or a difference already counted).
//
// Windows.  Sampled pairs give a histogram of the output keys; the cuts put
// about `pt` pairs in a window.  The cuts only balance the work: a window whose
// terms do not fit its table is halved and done in pieces, and a window of at
// most SLOTS keys is addressed directly, without a hash, and always fits.
// Another sample estimates the terms per pair by region of the key range
// (k_win_dup).  Where pairs share keys a CTA takes a run of windows through one
// table (a mean over the whole product instead let a third of the runs of the
// weighted product overflow, which doubled its time); where they do not, a
// window's pairs are ordered as a list, without a table, and several windows'
// pairs are formed in one walk if a window has few of them per term walked
// (one walk per window: 1.3 against 0.95 ms on the 5003 x 3989 terms).
#include <algorithm>
#include <cstring>
#include <type_traits>

#include "kr_internal.cuh"

namespace kr {

constexpr int WT = 512;                // threads per CTA
constexpr int WNW = WT / 32;
constexpr int WSUBS = 8;               // convolutions of a window at most
constexpr int WST = WIN_STAGE_MAX;     // windows of a staged run at most
// pairs of a window that is ordered as a list: 10 (32-bit offsets) or 5 per thread
template <int SLOTS>
__host__ __device__ constexpr int win_list_cap() { return SLOTS * 5 / 8; }
// pairs that the staging area takes of a window (more than a list: two lists)
template <int SLOTS>
__host__ __device__ constexpr int win_stage_cap() { return SLOTS * 15 / 16; }
constexpr int WLONG = 192;             // long ranges put aside per window at most
constexpr uint32_t WLONG_MIN = 64;     // pairs from which a range is long
constexpr uint32_t WLONG_SEG = 256;    // pairs of a long range per turn of a warp
constexpr int WNB = 4096;              // buckets of the window's ordering
constexpr int WSPLIT = 256;            // buckets where the keys cluster: sampled splitters
constexpr uint32_t WCROWD = 24;        // keys of a bucket that count as clustered
constexpr int WIN_PROBES = 48;         // probes before a window counts as full (at about 0.8 of its slots)
constexpr unsigned WFULL = 0xffffffffu;

// ---------------------------------------------------------------------------
// lists of a Poisson product: see above
// ---------------------------------------------------------------------------
__device__ __forceinline__ int64_t first_sine(const Operand& O) {
  int64_t lo = 0, hi = O.n;
  while (lo < hi) {
    const int64_t mid = (lo + hi) >> 1;
    if (O.kind[mid] < 1) lo = mid + 1; else hi = mid;
  }
  return lo;
}

// first index in [s0, s1) whose trig code is >= t
__device__ __forceinline__ int64_t trig_bound(const Operand& O, int64_t s0, int64_t s1, int64_t t) {
  return s0 + lower_bound_i64(O.tcode + s0, s1 - s0, t);
}

// the least code of the B list of block [s0, s1): the mirror image of its
// first term of the largest multiplier code
__device__ __forceinline__ int64_t list_base(const Operand& O, int64_t s0, int64_t s1, int64_t Wp) {
  if (s1 <= s0) return 0;
  const int64_t t = O.tcode[s1 - 1];
  const int64_t a = trig_bound(O, s0, s1, t);
  return -t * Wp + O.code[a];
}

__global__ void __launch_bounds__(256) k_win_lists(const Prod* __restrict__ prods,
                                                   const int32_t* __restrict__ wprods) {
  const Prod& P = prods[wprods[blockIdx.y]];
  if (P.nt == 0 || P.status) return;
  const Operand& A = P.win.swap ? P.g : P.f;
  const Operand& B = P.win.swap ? P.f : P.g;
  const int64_t Wp = P.Wp;
  const int64_t total = A.n + B.n;
  const int64_t nca = first_sine(A), ncb = first_sine(B);
  const int64_t base0 = list_base(B, 0, ncb, Wp), base1 = list_base(B, ncb, B.n, Wp);
  for (int64_t x = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; x < total;
       x += (int64_t)gridDim.x * blockDim.x) {
    const bool isA = x < A.n;
    const Operand& O = isA ? A : B;
    const int64_t q = isA ? x : x - A.n;
    const int64_t nc = isA ? nca : ncb;
    const bool sine = q >= nc;
    const int64_t s0 = sine ? nc : 0, s1 = sine ? O.n : nc;
    const int64_t t = O.tcode[q], p = O.code[q];
    const double c = ((const double*)O.coef)[q];
    const int64_t a = trig_bound(O, s0, s1, t), b = trig_bound(O, s0, s1, t + 1);
    const int64_t u = t * Wp + p, v = -t * Wp + p;
    if (isA) {
      const int64_t vp = s0 + (s1 - b) + (q - a);
      P.win.acode[q] = u;
      P.win.acode[A.n + vp] = v;
      P.win.acoef[vp] = c;
    } else {
      int64_t* code = P.win.bcode + 2 * s0;
      double* coef = P.win.bcoef + 2 * s0;
      const int64_t base = sine ? base1 : base0;
      const int64_t N = s1 - s0, pos = q - s0;
      if (t > 0) {
        const int64_t vp = (s1 - b) + (q - a);
        code[vp] = v - base;
        coef[vp] = c;
        code[N + pos] = u - base;
        coef[N + pos] = c;
      } else {   // t == 0: the first z terms of the block, twice
        const int64_t z = b - s0;
        const int64_t at = N - z + 2 * pos;
        code[at] = code[at + 1] = p - base;
        coef[at] = coef[at + 1] = c;
      }
    }
  }
}

// Bucket index of every searched list and, by one thread per list, the list's
// and the product's descriptors.  The buckets of a wide gap (a far term's, all
// 65536 of them) are written by the whole warp.
__global__ void __launch_bounds__(256) k_win_index(const Prod* __restrict__ prods,
                                                   const int32_t* __restrict__ wprods) {
  const Prod& P = prods[wprods[blockIdx.y >> 1]];
  const int which = blockIdx.y & 1;   // list: 0 = the polynomial's or the cosines', 1 = the sines'
  if (P.status || (P.nt == 0 && which)) return;
  const Operand& A = P.win.swap ? P.g : P.f;
  const Operand& B = P.win.swap ? P.f : P.g;
  WinDesc& D = *P.win.desc;
  WinList L;
  int64_t z = 0, s0 = 0, s1 = 0;
  L.idx = P.win.idx + which * (P.win.idx_cap + 2);
  if (P.nt == 0) {
    L.code = B.code;
    L.coef = B.coef;
    L.n = B.nkeep;
    L.base = 0;
    L.nv = 0;
  } else {
    const int64_t nc = first_sine(B);
    s0 = which ? nc : 0;
    s1 = which ? B.n : nc;
    z = trig_bound(B, s0, s1, 1) - s0;
    L.code = P.win.bcode + 2 * s0;
    L.coef = P.win.bcoef + 2 * s0;
    L.n = 2 * (s1 - s0);
    L.base = list_base(B, s0, s1, P.Wp);
    L.nv = (s1 - s0) - z;
  }
  L.span = L.n > 0 ? L.code[L.n - 1] : 0;
  int sh = 0;
  while ((L.span >> sh) + 1 > P.win.idx_cap) ++sh;
  L.shift = sh;
  L.nidx = (L.span >> sh) + 1;
  int32_t* idx = (int32_t*)L.idx;
  const int lane = threadIdx.x & 31;
  for (int64_t j0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x - lane; j0 <= L.n;
       j0 += (int64_t)gridDim.x * blockDim.x) {
    const int64_t j = j0 + lane;
    int blo = 1, bhi = 0;   // (at most 65536 buckets)
    if (j <= L.n) {
      blo = j == 0 ? 0 : (int)max((L.code[j - 1] >> sh) + 1, (int64_t)0);
      bhi = j == L.n ? (int)L.nidx : (int)min(L.code[j] >> sh, L.nidx);
    }
    unsigned wide = __ballot_sync(WFULL, bhi - blo >= 32);
    if (bhi - blo < 32)
      for (int b = blo; b <= bhi; ++b) idx[b] = (int32_t)j;
    for (; wide; wide &= wide - 1) {
      const int src = __ffs(wide) - 1;
      const int lo = __shfl_sync(WFULL, blo, src), hi = __shfl_sync(WFULL, bhi, src);
      for (int b = lo + lane; b <= hi; b += 32) idx[b] = (int32_t)(j0 + src);
    }
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    D.L[which] = L;
    if (which == 0) {
      D.nca = P.nt ? first_sine(A) : A.nkeep;
      D.na = P.nt ? A.n : A.nkeep;
    }
  }
}

// ---------------------------------------------------------------------------
// window cuts
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint32_t hash32(uint64_t x) { return (uint32_t)(mix64(x) >> 32); }

// Histogram of the output keys of `samples` term pairs (all of them when
// samples is the number of pairs; else stratified over A, B's term by a
// counter-based hash).  A warp adds up the hits of its first lane's bin until that
// changes: where one bin takes nearly all samples, the adds of 5.4 million one by one
// took 4.3 ms.
__global__ void __launch_bounds__(256) k_win_hist(const Prod* __restrict__ prods,
                                                  const int32_t* __restrict__ wprods) {
  const Prod& P = prods[wprods[blockIdx.y]];
  if (P.status) return;
  const Operand& F = P.win.swap ? P.g : P.f;
  const Operand& G = P.win.swap ? P.f : P.g;
  const int64_t nf = F.nkeep, ng = G.nkeep;
  if (nf <= 0 || ng <= 0) return;
  const int64_t S = P.win.samples;
  const bool all = S >= F.n * G.n;
  const int64_t T2Wp = P.T2 * P.Wp;
  const int sh = P.win.bin_shift;
  const uint64_t K0 = (uint64_t)P.klo, K = (uint64_t)P.kspan;
  const int64_t last = P.win.nbins - 1;
  const int lane = threadIdx.x & 31;
  int cur = -1;   // the bin being added up (of the whole warp), and its hits
  uint32_t hits = 0;
  auto flush = [&]() {
    if (lane == 0 && cur >= 0) atomicAdd(&P.win.hist[cur], hits);
  };
  auto hit = [&](bool act, int64_t key) {   // by whole warps
    const uint64_t k = (uint64_t)key - K0;
    act = act && k < K;
    const int bin = act ? (int)min((int64_t)(k >> sh), last) : -1, first = __shfl_sync(WFULL, bin, 0);
    if (act && bin != first) atomicAdd(&P.win.hist[bin], 1u);
    if (first != cur) {
      flush();
      cur = first;
      hits = 0;
    }
    hits += (uint32_t)__popc(__ballot_sync(WFULL, bin == first));
  };
  for (int64_t u0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x - lane; u0 < S;
       u0 += (int64_t)gridDim.x * blockDim.x) {
    const int64_t u = u0 + lane;
    bool act = u < S;
    int64_t i = 0, j = 0;
    if (all) {
      i = u / G.n;
      j = u - i * G.n;
      act = act && i < nf && j < ng;
      if (!act) i = j = 0;
    } else if (act) {
      i = (int64_t)((uint64_t)u * (uint64_t)nf / (uint64_t)S);   // samples < 2^32, terms < 2^31
      j = (int64_t)(((uint64_t)hash32((uint64_t)u + 1ull) * (uint64_t)ng) >> 32);
    }
    const int64_t pc = F.code[i] + G.code[j];
    if (P.nt == 0) {
      hit(act, pc);
      continue;
    }
    const int kd = F.kind[i] ^ G.kind[j];
    const int64_t ts = F.tcode[i] + G.tcode[j];
    int64_t td = F.tcode[i] - G.tcode[j];
    if (td < 0) td = -td;
    hit(act, kd * T2Wp + ts * P.Wp + pc);
    hit(act && !(td == 0 && kd), kd * T2Wp + td * P.Wp + pc);
  }
  flush();
}

// One CTA per product: the windows' starts, from the histogram.  The last CTA
// to finish turns the products' window counts into offsets.
//
// A bin's windows lie as if its samples were spread evenly, which is wrong by at
// most the bin's own windows.  Where a bin holds more of them than a CTA's share
// of all (a cluster in a range that a few far terms made wide: 1820 terms of a
// simplex and one monomial of degree 10^9, squared, lie in one bin of 6601), the
// cuts are quantiles of sampled keys instead, found by sorting the sample here.
// With the bins alone one CTA formed most of the pairs, halving its windows again
// and again: 18.7 ms for those 3.3 M pairs, now 0.37 (a table in device memory
// 0.69); 583 ms for 9 M pairs of 3.8 M keys, now 0.90 (1.47).  Keys so close that
// not even quantiles divide them (25 M pairs on 10000 keys) are left to the table,
// which adds them from all CTAs at once.
constexpr int WC_THREADS = 1024;
constexpr int WC_SORT = 16 * WC_THREADS;  // sampled keys at most (128 KB)
__host__ __device__ inline int wc_sort_size(int64_t windows) {   // a power of two
  int n = 2 * WC_THREADS;
  while (n < WC_SORT && n < 4 * windows) n <<= 1;
  return n;
}
constexpr int64_t WC_CROWD = 8;          // windows in a bin that are few in any case
constexpr int64_t WC_DIRECT = 512;       // windows' pairs on the keys of one directly addressed window at most:
                                         // an update takes about 0.3 ns there, a table's call 0.5 ms at least

// The key, relative to klo, of sample u of n term pairs (-1: outside the range).
__device__ __forceinline__ int64_t wc_sample(const Prod& P, int64_t u, int64_t n) {
  const Operand& F = P.win.swap ? P.g : P.f;
  const Operand& G = P.win.swap ? P.f : P.g;
  const int64_t i = u * F.nkeep / n;
  // multiples of the golden ratio: spread over G evenly for any number of samples
  const int64_t j = (int64_t)(((uint64_t)((uint32_t)u * 2654435769u) * (uint64_t)G.nkeep) >> 32);
  int64_t key = F.code[i] + G.code[j];
  if (P.nt) {
    const int kd = F.kind[i] ^ G.kind[j];
    int64_t T = F.tcode[i] + ((hash32((uint64_t)u + 77ull) & 1u) ? G.tcode[j] : -G.tcode[j]);
    if (T < 0) T = -T;
    if (T == 0 && kd) return -1;
    key += kd * (P.T2 * P.Wp) + T * P.Wp;
  }
  key -= P.klo;
  return key >= 0 && key < P.kspan ? key : -1;
}

// Sorts the CTA's words, E a thread in sequence (v[e] is word E t + e), by a
// bitonic network: strides below E within the thread, below 32 E by shuffles, the
// others through shared memory k.  (Every step through shared memory took 400 us for
// 16384 words.)
template <int E>
__device__ __forceinline__ void wc_sort(uint64_t (&v)[E], uint64_t* k) {
  const int tid = threadIdx.x;
  constexpr int N = E * WC_THREADS;
  for (int size = 2; size <= N; size <<= 1) {
    for (int stride = size >> 1; stride >= E; stride >>= 1) {
      const int far = stride / E;   // the partner's distance in threads
      const bool low = (((tid * E) & size) == 0) == ((tid & far) == 0);   // keeps the smaller word
      if (far >= 32) {
#pragma unroll
        for (int e = 0; e < E; ++e) k[e * WC_THREADS + tid] = v[e];
        __syncthreads();
      }
#pragma unroll
      for (int e = 0; e < E; ++e) {
        const uint64_t o = far >= 32 ? k[e * WC_THREADS + (tid ^ far)] : __shfl_xor_sync(WFULL, v[e], far);
        v[e] = (o < v[e]) == low ? o : v[e];
      }
      if (far >= 32) __syncthreads();
    }
#pragma unroll
    for (int stride = E / 2; stride > 0; stride >>= 1)
      if (stride < size) {
#pragma unroll
        for (int e = 0; e < E; ++e)
          if (!(e & stride)) {
            const uint64_t a = v[e], b = v[e | stride];
            const bool swap = (a > b) == (((tid * E + e) & size) == 0);
            v[e] = swap ? b : a;
            v[e | stride] = swap ? a : b;
          }
      }
  }
}

// E * WC_THREADS sampled keys into k, ascending; returns how many lie in range (the first ones).
template <int E>
__device__ __noinline__ int wc_sorted_sample(const Prod& P, uint64_t* k) {
  uint64_t v[E];
  int valid = 0;
#pragma unroll
  for (int e = 0; e < E; ++e) {   // (in any order)
    const int64_t x = wc_sample(P, e * WC_THREADS + threadIdx.x, E * WC_THREADS);
    v[e] = (uint64_t)x;   // (-1 sorts last)
    valid += x >= 0;
  }
  __shared__ int s_valid;
  if (threadIdx.x == 0) s_valid = 0;
  __syncthreads();
  valid = __reduce_add_sync(WFULL, valid);
  if ((threadIdx.x & 31) == 0) atomicAdd(&s_valid, valid);
  wc_sort<E>(v, k);
#pragma unroll
  for (int e = 0; e < E; ++e) k[threadIdx.x * E + e] = v[e];
  __syncthreads();
  return s_valid;
}

__device__ __forceinline__ int64_t wc_scan(int64_t v, int64_t* total, int64_t* ws) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int64_t x = v;
  for (int o = 1; o < 32; o <<= 1) {
    const int64_t y = __shfl_up_sync(WFULL, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) ws[warp] = x;
  __syncthreads();
  if (warp == 0) {
    int64_t s = ws[lane];
    for (int o = 1; o < 32; o <<= 1) {
      const int64_t y = __shfl_up_sync(WFULL, s, o);
      if (lane >= o) s += y;
    }
    ws[lane] = s;
  }
  __syncthreads();
  const int64_t base = warp ? ws[warp - 1] : 0;
  *total = ws[WC_THREADS / 32 - 1];
  __syncthreads();
  return base + x - v;
}

// Records a product's number of runs; the last CTA to finish turns them into
// offsets.  By one CTA per product.
__device__ __forceinline__ void win_prefix(int64_t nrun, int nwp, int64_t* rprefix, unsigned int* done, int64_t* ws,
                                           unsigned int* s_last) {
  if (threadIdx.x == 0) {
    rprefix[blockIdx.x + 1] = nrun;
    __threadfence();
    *s_last = atomicAdd(done, 1u) == gridDim.x - 1 ? 1u : 0u;
  }
  __syncthreads();
  if (!*s_last) return;
  __threadfence();
  int64_t run = 0;
  for (int p0 = 0; p0 < nwp; p0 += WC_THREADS) {
    const int p = p0 + threadIdx.x;
    const int64_t v = p < nwp ? __ldcg(&rprefix[p + 1]) : 0;
    int64_t tot;
    const int64_t e = wc_scan(v, &tot, ws);
    if (p < nwp) rprefix[p + 1] = run + e + v;
    run += tot;
  }
  if (threadIdx.x == 0) {
    rprefix[0] = 0;
    *done = 0;
  }
}

// Estimated terms per pair around window w of nw.
__device__ __forceinline__ float win_distinct(const WinDesc& D, int64_t w, int64_t nw) {
  const int r = (int)(w * WIN_REGIONS / nw);
  const float n = D.rn[r];
  return n >= 4.0f ? D.rs[r] / n : 1.0f;
}

__global__ void __launch_bounds__(WC_THREADS) k_win_cut(Prod* __restrict__ prods,
                                                        const int32_t* __restrict__ wprods, int nwp,
                                                        int64_t* __restrict__ rprefix, int64_t slots, int64_t ctas,
                                                        unsigned int* __restrict__ done) {
  extern __shared__ __align__(8) uint32_t hs[];   // the histogram, one word of padding per 32 bins; or sampled keys
  __shared__ int64_t ws[WC_THREADS / 32];
  __shared__ unsigned int s_last, s_top;
  Prod& P = prods[wprods[blockIdx.x]];
  int64_t nw = 1;
  if (P.status == 0) {
    const int nb = (int)P.win.nbins;
    uint32_t top = 0;
    if (threadIdx.x == 0) s_top = 0;
    for (int i = threadIdx.x; i < nb; i += WC_THREADS) {
      const uint32_t x = P.win.hist[i];
      hs[i + (i >> 5)] = x;
      top = max(top, x);
    }
    __syncthreads();
    top = __reduce_max_sync(WFULL, top);
    if ((threadIdx.x & 31) == 0) atomicMax(&s_top, top);   // (read after the scan's barriers)
    // inclusive prefix sums in place
    const int per = (nb + WC_THREADS - 1) / WC_THREADS;
    const int a = min(nb, per * (int)threadIdx.x), b = min(nb, a + per);
    int64_t s = 0;
    for (int i = a; i < b; ++i) s += hs[i + (i >> 5)];
    int64_t tot;
    uint32_t c = (uint32_t)wc_scan(s, &tot, ws);
    for (int i = a; i < b; ++i) hs[i + (i >> 5)] = c += hs[i + (i >> 5)];
    __syncthreads();
    // window k starts where k * spw samples lie before it, placed inside its
    // bin as if the bin's samples were spread evenly, at a multiple of an eighth
    // of `slots` keys from the bin's start (bins are at least `slots` wide):
    // windows that would start at the same key are one
    int64_t spw = max((int64_t)1, (tot + P.win.nw - 1) / max((int64_t)1, P.win.nw));
    int64_t nk = max((int64_t)1, (tot + spw - 1) / spw);
    const float binw = (float)(int64_t(1) << P.win.bin_shift);
    // more than a CTA's share (and a quarter: the 6188 x 6188 weighted product, 34 of 9539
    // windows in a bin at a share of 31, is cut well by its bins) in windows wider than a
    // table, or many times that in narrow ones, which are addressed directly and never
    // halved (a bin of the sums of two simplexes: the sample alone would cost a call of
    // 0.5 ms 30 us)
    const int64_t few = spw * max(WC_CROWD, 5 * nk / (4 * ctas)), many = spw * max(WC_DIRECT, 16 * nk / ctas);
    bool crowded = false;
    if ((int64_t)s_top > few) {   // uniform
      for (int i = a; i < b; ++i) {
        const int64_t x = (int64_t)(hs[i + (i >> 5)] - (i ? hs[(i - 1) + ((i - 1) >> 5)] : 0u));
        crowded |= x > many || (x > few && x / spw < (int64_t(1) << P.win.bin_shift) / slots);
      }
      crowded = __syncthreads_or(crowded);
    }
    const uint64_t* const ks = (const uint64_t*)hs;
    int64_t nv = 0;   // sampled keys
    if (crowded) {
      __syncthreads();   // the histogram has been read
      const int n = wc_sort_size(P.win.nw);
      uint64_t* const k = (uint64_t*)hs;
      nv = n == 2 * WC_THREADS ? wc_sorted_sample<2>(P, k) : n == 4 * WC_THREADS ? wc_sorted_sample<4>(P, k)
         : n == 8 * WC_THREADS ? wc_sorted_sample<8>(P, k) : wc_sorted_sample<16>(P, k);
      nk = P.win.nw + P.win.nw / 15;   // (the cap is 3 nw + 16)
      spw = 1;   // (Win::before counts windows)
      tot = nk;
    }
    auto start_of = [&](int64_t k) -> int64_t {   // relative to klo
      if (k <= 0) return 0;
      if (crowded) {
        // the share y of the windows, 1 / 16 of them spread over the range and the
        // others over the samples: no window is wider than 16 of the mean, so that a
        // wide gap is not left to one CTA (32-bit offsets walk it in steps of 2^32:
        // 113 M pairs beside a far term of degree 10^7, 3.5 -> 1.9 ms)
        const float y = (float)k / (float)nk, a = 0.9375f / (float)nv, b = 0.0625f / (float)P.kspan;
        auto upto = [&](int i) -> float { return a * (float)(i + 1) + b * (float)(int64_t)ks[i]; };
        int i = 0, top = (int)nv;   // the first sample past the share
        while (i < top) {
          const int mid = (i + top) >> 1;
          if (upto(mid) > y) top = mid; else i = mid + 1;
        }
        const int64_t lo = i > 0 ? (int64_t)ks[i - 1] : 0, hi = i < (int)nv ? (int64_t)ks[i] : P.kspan;
        const float ylo = i > 0 ? upto(i - 1) : 0.0f, yhi = i < (int)nv ? upto(i) : 1.0f;
        const float part = fminf(fmaxf((y - ylo) / fmaxf(yhi - ylo, 1e-30f), 0.0f), 1.0f);
        return (lo + min((int64_t)(part * (float)(hi - lo)), hi - lo)) & ~(slots / 8 - 1);
      }
      const uint32_t want = (uint32_t)(k * spw);
      int lo = 0, hi = nb - 1;   // the first bin whose prefix exceeds it
      while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (hs[mid + (mid >> 5)] > want) hi = mid; else lo = mid + 1;
      }
      const uint32_t c0 = lo ? hs[(lo - 1) + ((lo - 1) >> 5)] : 0u;
      const uint32_t x = hs[lo + (lo >> 5)] - c0;
      const int64_t off = (int64_t)(__fdividef((float)(want - c0), (float)max(x, 1u)) * binw) & ~(slots / 8 - 1);
      return ((int64_t)lo << P.win.bin_shift) + min(off, (int64_t(1) << P.win.bin_shift) - slots / 8);
    };
    int64_t at = 0;
    for (int64_t k0 = 0; k0 < nk; k0 += WC_THREADS) {
      const int64_t k = k0 + threadIdx.x;
      int64_t st = 0;
      bool keep = false;
      if (k < nk) {
        st = start_of(k);
        keep = k == 0 || (st > start_of(k - 1) && st < P.kspan);
      }
      int64_t all;
      const int64_t q = at + wc_scan(keep ? 1 : 0, &all, ws);
      if (keep && q < P.win.cap) {
        P.win.start[q] = P.klo + st;
        P.win.before[q] = (uint32_t)(k * spw);
      }
      at += all;
    }
    nw = min(at, P.win.cap);
    if (threadIdx.x == 0) {   // the cap + 1 entries hold the end
      P.win.start[nw] = P.klo + P.kspan;
      P.win.before[nw] = (uint32_t)tot;
      P.win.desc->total = (float)tot;
      P.win.desc->nw = nw;
    }
    if (!P.win.merge)
      for (int64_t q = threadIdx.x; q <= nw; q += WC_THREADS) P.win.run[q] = (int32_t)q;
    if (crowded) {   // windows that would start at the same key are one: too many pairs for a CTA?
      __syncthreads();
      uint32_t most = 0;
      for (int64_t q = threadIdx.x; q < nw; q += WC_THREADS) most = max(most, P.win.before[q + 1] - P.win.before[q]);
      if ((int64_t)most > max(WC_DIRECT, 16 * nk / ctas)) atomicOr(&P.status, ST_WINDOW);
    }
  }
  if (done) win_prefix(nw, nwp, rprefix, done, ws, &s_last);
}
// Groups the windows of a merging product into runs, each of about one table's
// terms (estimated) and at most 8 windows' pairs, or of Win::stage windows to
// stage; short ones at the end, so that the CTAs finish together.
__global__ void __launch_bounds__(WC_THREADS) k_win_runs(const Prod* __restrict__ prods,
                                                         const int32_t* __restrict__ wprods, int nwp,
                                                         int64_t* __restrict__ rprefix, int64_t slots, int64_t ctas,
                                                         unsigned int* __restrict__ done) {
  __shared__ int64_t ws[WC_THREADS / 32];
  __shared__ unsigned int s_last;
  const Prod& P = prods[wprods[blockIdx.x]];
  int64_t nrun = 1;
  if (P.status == 0) {
    const WinDesc& D = *P.win.desc;
    const int64_t nw = D.nw;
    nrun = nw;
    if (P.win.merge) {
      const float per = P.win.updates / fmaxf(D.total, 1.0f);   // pairs per sample
      int64_t before = 0, at = 0;
      auto weight = [&](int64_t i) -> int64_t {   // in 1 / 65536 of a run
        const float r = win_distinct(D, i, nw);
        const float left = (float)(nw - i) / (float)(2 * ctas);
        float w;
        if (P.win.stage && r > 0.5f) {
          w = 1.0f / fminf((float)P.win.stage, fmaxf(left, 1.0f));
        } else {
          const float pairs = per * (float)(P.win.before[i + 1] - P.win.before[i]);
          w = fmaxf(pairs * r / (0.4f * (float)slots), pairs / (8.0f * (float)P.win.pt));
          w = fmaxf(w, 1.0f / fminf(16.0f, fmaxf(left, 1.0f)));
        }
        return (int64_t)(fminf(w, 4.0f) * 65536.0f) + 1;
      };
      for (int64_t i0 = 0; i0 < nw; i0 += WC_THREADS) {
        const int64_t i = i0 + threadIdx.x;
        const int64_t w = i < nw ? weight(i) : 0;
        int64_t all, runs;
        const int64_t s = before + wc_scan(w, &all, ws);   // before this window
        const int64_t prev = i > 0 && i < nw ? s - weight(i - 1) : 0;
        const bool first = i < nw && (i == 0 || (s >> 16) != (prev >> 16));
        const int64_t q = at + wc_scan(first ? 1 : 0, &runs, ws);
        if (first) P.win.run[q] = (int32_t)i;
        before += all;
        at += runs;
      }
      if (threadIdx.x == 0) P.win.run[at] = (int32_t)nw;
      nrun = at;
    }
  }
  win_prefix(nrun, nwp, rprefix, done, ws, &s_last);
}

// ---------------------------------------------------------------------------
// the window kernel
// ---------------------------------------------------------------------------
template <typename KT>
struct WinKey;
template <>
struct WinKey<uint32_t> {
  static __device__ __forceinline__ uint32_t cas(uint32_t* p, uint32_t v) { return atomicCAS(p, 0u, v); }
  static __device__ __forceinline__ uint32_t home(uint32_t off, int bits) {
    // two multiplicative rounds: one alone sends the arithmetic progressions
    // of a product's codes to a few slots for some strides
    uint32_t h = off * 2654435769u;
    h ^= h >> 15;
    return (h * 2246822519u) >> (32 - bits);
  }
};
template <>
struct WinKey<uint64_t> {
  static __device__ __forceinline__ uint64_t cas(uint64_t* p, uint64_t v) {
    return atomicCAS((unsigned long long*)p, 0ull, (unsigned long long)v);
  }
  static __device__ __forceinline__ uint32_t home(uint64_t off, int bits) {
    uint64_t h = off * 0x9e3779b97f4a7c15ull;
    h ^= h >> 32;
    return (uint32_t)((h * 0xd6e8feb86659fd93ull) >> (64 - bits));
  }
};

template <int N>
struct Log2 { static constexpr int v = 1 + Log2<N / 2>::v; };
template <>
struct Log2<1> { static constexpr int v = 0; };

// Shared memory of a window: the table (keys, values), then a region that
// holds the warps' entries while pairs are formed and the bucket counts while
// the window is ordered.
template <typename KT, int SLOTS>
struct WinSmem {
  uint64_t val[SLOTS];   // float64 sums, or int64 sums as low words [0, SLOTS) and high words
  KT key[SLOTS];         // offset in the window + 1 (0: empty); then the keys by bucket
  union {
    struct {
      uint64_t c[32];    // the A term's coefficient
      KT a[32];          // its part of the offset
      int32_t jb[32];    // B index of a pair: jb + pair number
    } e[WNW];
    uint32_t cnt[WNB / 2];      // two 16-bit bucket counts a word
    struct {
      uint32_t n[WSPLIT];       // clustered keys: counts between splitters
      KT s[WSPLIT];             // ascending splitters
    } g;
  } u;
  // ranges put aside: coefficient, offset, first partner, pairs (then the
  // segments up to and with this range's), convolution
  uint64_t lc[WLONG];
  KT la[WLONG];
  int32_t ll[WLONG];
  uint32_t ln[WLONG];
  int32_t lseg[WLONG];
  uint8_t ls[WLONG];
};

// One convolution of a window: the A terms [i0, i0 + n) against list L.
struct WinSub {
  const int64_t* a;
  const uint64_t* ca;
  int64_t i0, n;
  int64_t xlo, xhi;      // B codes b with xlo <= a + b < xhi
  int64_t off0;          // offset in the window = a + b + off0
  uint64_t sv, su;       // sign flips of the list's difference and sum entries
  int32_t list;
};

struct WinShared {
  int64_t t, m, excl;
  int full, big, next, nsub, nlong;
  int cnt[WNW];
  int ws[2][WNW];
  int first[WSUBS + 1];  // chunks before each convolution
  WinSub sub[WSUBS];
  int fill[WST];         // staged run: pairs of each window
  uint64_t bnd[WST];     // and the first offset of the one after it
};

// Block-wide exclusive scan of one value per thread; ws: two alternating rows.
__device__ __forceinline__ int win_scan(int v, int (*ws)[WNW], int& row) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(WFULL, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) ws[row][warp] = x;
  __syncthreads();
  const int base = __reduce_add_sync(WFULL, lane < warp ? ws[row][lane & (WNW - 1)] : 0);
  row ^= 1;   // the next scan writes the other row: no barrier after the reads
  return base + x - v;
}

template <typename T>
__device__ __forceinline__ uint64_t win_mul(uint64_t a, uint64_t b) {
  if constexpr (std::is_same<T, double>::value)
    return (uint64_t)__double_as_longlong(__longlong_as_double((long long)a) * __longlong_as_double((long long)b));
  else
    return a * b;
}

// Adds v to the table entry of offset `off`.  False: no slot within the probes.
template <typename T, typename KT, int SLOTS>
__device__ __forceinline__ bool win_add(WinSmem<KT, SLOTS>& sm, KT off, uint64_t v, bool direct) {
  constexpr int BITS = Log2<SLOTS>::v;
  uint32_t slot;
  if (direct) {
    slot = (uint32_t)off & (SLOTS - 1);
  } else {
    slot = WinKey<KT>::home(off, BITS);
    const KT me = off + 1;
    int probe = 0;
    for (; probe < WIN_PROBES; ++probe) {
      const KT old = WinKey<KT>::cas(&sm.key[slot], me);
      if (old == 0 || old == me) break;
      slot = (slot + 1) & (SLOTS - 1);
    }
    if (probe == WIN_PROBES) return false;
  }
  if constexpr (std::is_same<T, double>::value)
    atomicAdd((double*)&sm.val[slot], __longlong_as_double((long long)v));
  else
    smem_acc_split64((uint32_t)__cvta_generic_to_shared(sm.val) + 4u * slot, 4u * SLOTS, v);
  return true;
}

// The convolutions that reach keys [B, E) of the product, offsets relative to
// B; the chunks of 32 A terms of all of them are numbered for the warps.
__device__ __forceinline__ void win_subs(WinShared& sh, const Prod& P, const WinDesc& D, int64_t B, int64_t E) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int ns = P.nt ? WSUBS : 1;
  if (warp < ns) {
    const Operand& A = P.win.swap ? P.g : P.f;
    constexpr uint64_t NEG = 1ull << 63;
    WinSub S;
    int64_t lo = B, hi = E, kb = 0, na = D.na;
    S.sv = S.su = 0;
    S.list = 0;
    S.a = A.code;
    S.ca = (const uint64_t*)A.coef;
    if (P.nt) {
      const int64_t half = P.T2 * P.Wp;
      const int kd = warp >> 2, ka = (warp >> 1) & 1, mirror = warp & 1;
      kb = kd * half;
      hi = min(E - kb, half);
      lo = max(B - kb, (mirror || kd) ? P.Wp : (int64_t)0);
      S.list = ka ^ kd;
      const int64_t a0 = ka ? D.nca : 0;
      na = ka ? D.na - D.nca : D.nca;
      // signs: the sum of two sines is negated; a difference of a cosine and a
      // sine takes the sign of which factor is the sine and which multiplier is larger
      S.su = mirror ? ((kd && ka) ? NEG : 0ull) : ((ka & S.list) ? NEG : 0ull);
      S.sv = (!ka && S.list) ? NEG : 0ull;
      S.a = P.win.acode + (mirror ? D.na : 0) + a0;
      S.ca = mirror ? (const uint64_t*)P.win.acoef + a0 : (const uint64_t*)A.coef + a0;
    }
    const WinList& L = D.L[S.list];
    S.xlo = lo - L.base;
    S.xhi = hi - L.base;
    S.off0 = L.base + kb - B;
    int64_t i0 = 0, i1 = 0;
    if (lo < hi && na > 0 && L.n > 0) warp_lower_bound2(S.a, na, S.xlo - L.span, S.xhi, &i0, &i1);
    S.i0 = i0;
    S.n = i1 - i0;
    if (lane == 0) sh.sub[warp] = S;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    int c = 0;
    for (int s = 0; s < ns; ++s) {
      sh.first[s] = c;
      c += (int)((max(sh.sub[s].n, (int64_t)0) + 31) >> 5);
    }
    sh.first[ns] = c;
    sh.nsub = ns;
    sh.next = 0;
    sh.full = 0;
    sh.nlong = 0;
  }
  __syncthreads();
}

// Forms the pairs of the listed convolutions.  Every warp takes 32 A terms at
// a time: each lane finds its term's range of partners, the ranges are laid
// end to end by a warp scan, and the warp walks that row of pairs 32 at a
// time, so that short ranges still fill the lanes.  Long ranges are put aside in a
// list of the CTA's and then shared out among the warps in segments, so that no
// warp is left with the pairs of a few long ranges.
template <typename T, typename KT, int SLOTS, typename Sink>
__device__ __forceinline__ void win_form(WinSmem<KT, SLOTS>& sm, WinShared& sh, const WinDesc& D, Sink sink) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  auto& ent = sm.u.e[warp];
  const int nsub = sh.nsub, nchunks = sh.first[nsub];
  for (;;) {
    int c = 0;
    if (lane == 0) c = *(volatile int*)&sh.full ? nchunks : atomicAdd(&sh.next, 1);
    c = __shfl_sync(WFULL, c, 0);
    if (c >= nchunks) break;
    int s = 0;
    while (s + 1 < nsub && sh.first[s + 1] <= c) ++s;
    const WinSub& S = sh.sub[s];
    const WinList& L = D.L[S.list];
    const int64_t* __restrict__ bcode = L.code;
    const uint64_t* __restrict__ bcoef = (const uint64_t*)L.coef;
    const int64_t nv = L.nv;
    const int64_t i = (int64_t)(c - sh.first[s]) * 32 + lane;
    int32_t l = 0;
    uint32_t cnt = 0;
    int64_t av = 0;
    uint64_t ca = 0;
    if (i < S.n) {
      av = S.a[S.i0 + i];
      ca = S.ca[S.i0 + i];
      int64_t x, y;
      g_lower_bound2(bcode, L.n, L.idx, L.nidx, L.shift, S.xlo - av, S.xhi - av, &x, &y);
      l = (int32_t)x;
      cnt = (uint32_t)(y - x);
      if (cnt >= WLONG_MIN) {
        const int k = atomicAdd(&sh.nlong, 1);
        if (k < WLONG) {
          sm.lc[k] = ca;
          sm.la[k] = (KT)(av + S.off0);
          sm.ll[k] = l;
          sm.ln[k] = cnt;
          sm.ls[k] = (uint8_t)s;
          cnt = 0;
        }
      }
    }
    uint32_t at = cnt;   // pairs up to and with this lane's (below 2^26)
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(WFULL, at, o);
      if (lane >= o) at += y;
    }
    const uint32_t total = __shfl_sync(WFULL, at, 31);
    at -= cnt;
    const unsigned some = __ballot_sync(WFULL, cnt > 0);
    if (cnt > 0) {
      const int e = __popc(some & ((1u << lane) - 1u));
      ent.c[e] = ca;
      ent.a[e] = (KT)(av + S.off0);
      ent.jb[e] = (int32_t)((uint32_t)l - at);
    }
    __syncwarp();
    const uint64_t sv = S.sv, su = S.su;
    for (uint32_t p0 = 0; p0 < total; p0 += 32) {
      // the entry of each pair: that of the row's first pair, plus the ones
      // that start after it
      const unsigned heads =
          __reduce_or_sync(WFULL, cnt > 0 && at > p0 && at - p0 < 32u ? 1u << (at - p0) : 0u);
      const int e0 = __popc(__ballot_sync(WFULL, cnt > 0 && at <= p0)) - 1;
      const uint32_t p = p0 + lane;
      uint64_t v = 0;
      KT off = 0;
      const bool act = p < total;
      if (act) {
        const int e = (e0 + __popc(heads & ((2u << lane) - 1u))) & 31;
        const uint32_t j = min((uint32_t)ent.jb[e] + p, (uint32_t)(L.n - 1));
        off = ent.a[e] + (KT)bcode[j];
        v = win_mul<T>(ent.c[e], bcoef[j]);
        if constexpr (std::is_same<T, double>::value) v ^= (int64_t)j < nv ? sv : su;
      }
      sink(act, off, v);
    }
    __syncwarp();
  }
  __syncthreads();
  const int nl = min(sh.nlong, WLONG);
  if (nl == 0) return;   // uniform
  if (warp == 0) {   // segments up to and with each long range
    int run = 0;
    for (int k0 = 0; k0 < nl; k0 += 32) {
      const int k = k0 + lane;
      int x = k < nl ? (int)((sm.ln[k] + WLONG_SEG - 1) / WLONG_SEG) : 0;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(WFULL, x, o);
        if (lane >= o) x += y;
      }
      if (k < nl) sm.lseg[k] = run + x;
      run += __shfl_sync(WFULL, x, 31);
    }
    if (lane == 0) sh.next = 0;
  }
  __syncthreads();
  const int nseg = sm.lseg[nl - 1];
  for (;;) {
    int c = 0;
    if (lane == 0) c = *(volatile int*)&sh.full ? nseg : atomicAdd(&sh.next, 1);
    c = __shfl_sync(WFULL, c, 0);
    if (c >= nseg) break;
    int lo = 0, hi = nl - 1;   // the range of segment c
    while (lo < hi) {
      const int mid = (lo + hi) >> 1;
      if (sm.lseg[mid] <= c) lo = mid + 1; else hi = mid;
    }
    const WinSub& S = sh.sub[sm.ls[lo]];
    const WinList& L = D.L[S.list];
    const int64_t* __restrict__ bcode = L.code;
    const uint64_t* __restrict__ bcoef = (const uint64_t*)L.coef;
    const uint32_t q0 = (uint32_t)(c - (lo ? sm.lseg[lo - 1] : 0)) * WLONG_SEG;
    const uint32_t q1 = min(sm.ln[lo], q0 + WLONG_SEG);
    const uint64_t ca = sm.lc[lo];
    const KT a = sm.la[lo];
    const uint32_t j0 = (uint32_t)sm.ll[lo];
    for (uint32_t q = q0; q < q1; q += 32) {
      const bool act = q + lane < q1;
      KT off = 0;
      uint64_t v = 0;
      if (act) {
        const uint32_t j = min(j0 + q + lane, (uint32_t)(L.n - 1));
        off = a + (KT)bcode[j];
        v = win_mul<T>(ca, bcoef[j]);
        if constexpr (std::is_same<T, double>::value) v ^= (int64_t)j < L.nv ? S.sv : S.su;
      }
      sink(act, off, v);
    }
  }
}

template <typename T, typename KT, int SLOTS>
__device__ __forceinline__ uint64_t win_value(const WinSmem<KT, SLOTS>& sm, int slot) {
  if constexpr (std::is_same<T, double>::value) {
    return sm.val[slot];
  } else {
    const uint32_t* w = (const uint32_t*)sm.val;
    return ((uint64_t)w[SLOTS + slot] << 32) | (uint64_t)w[slot];
  }
}

template <typename T>
__device__ __forceinline__ bool win_live(uint64_t v) {
  return std::is_same<T, double>::value ? (v << 1) != 0 : v != 0;
}

template <typename KT, int SLOTS>
__device__ __forceinline__ void win_clear(WinSmem<KT, SLOTS>& sm, bool direct) {
  const uint4 zero = make_uint4(0, 0, 0, 0);
  uint4* v = (uint4*)sm.val;
  for (int i = threadIdx.x; i < SLOTS / 2; i += WT) v[i] = zero;
  if (!direct) {
    uint4* k = (uint4*)sm.key;
    for (int i = threadIdx.x; i < (int)(SLOTS * sizeof(KT) / 16); i += WT) k[i] = zero;
  }
}

// Clustered keys: splitters from a sample, one key of each of the first WSPLIT
// threads (~0: it has none; the threads' keys are in no order), sorted by
// counting.  The counts between splitters are cleared.
template <typename KT, int SLOTS>
__device__ __noinline__ void win_splitters(WinSmem<KT, SLOTS>& sm, KT mine) {
  const int tid = threadIdx.x;
  if (tid < WSPLIT) sm.key[tid] = mine;
  __syncthreads();   // (the counts by high bits have been read)
  if (tid < WSPLIT) {
    int rank = 0;
    for (int x = 0; x < WSPLIT; ++x) {
      const KT y = sm.key[x];
      rank += y < mine || (y == mine && x < tid) ? 1 : 0;
    }
    sm.u.g.s[rank] = mine;
    sm.u.g.n[tid] = 0;
  }
  __syncthreads();
}

// Bucket b: the keys in (splitter b - 1, splitter b]; the last takes the rest.
template <typename KT, int SLOTS>
__device__ __forceinline__ int win_between(const WinSmem<KT, SLOTS>& sm, KT x) {
  int lo = 0;
#pragma unroll
  for (int step = WSPLIT / 2; step > 0; step >>= 1) lo += sm.u.g.s[lo + step - 1] < x ? step : 0;
  return lo;
}

// The terms of a directly addressed table (lim slots), in order: place(n)
// gives the position of the first (called by every thread), write(position,
// offset, value) takes each.
template <typename T, typename KT, int SLOTS, typename Place, typename Write>
__device__ __forceinline__ int win_emit_direct(WinSmem<KT, SLOTS>& sm, WinShared& sh, int lim, Place place,
                                               Write write) {
  // slot order is key order: each warp a contiguous part, 32 slots a row
  constexpr int PART = SLOTS / WNW;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int c = 0;
  for (int r = 0; r < PART / 32; ++r) {
    const int s = warp * PART + 32 * r + lane;
    c += __popc(__ballot_sync(WFULL, s < lim && win_live<T>(win_value<T, KT, SLOTS>(sm, s))));
  }
  if (lane == 0) sh.cnt[warp] = c;
  __syncthreads();
  const int part = lane < WNW ? sh.cnt[lane] : 0;
  const int n = __reduce_add_sync(WFULL, part), mine = __reduce_add_sync(WFULL, lane < warp ? part : 0);
  int64_t pos = place(n) + mine;
  for (int r = 0; r < PART / 32; ++r) {
    const int s = warp * PART + 32 * r + lane;
    const uint64_t v = s < lim ? win_value<T, KT, SLOTS>(sm, s) : 0ull;
    const bool lv = s < lim && win_live<T>(v);
    const unsigned b = __ballot_sync(WFULL, lv);
    if (lv) write(pos + __popc(b & ((1u << lane) - 1u)), (KT)s, v);
    pos += __popc(b);
  }
  return n;
}

// The same for a hashed table of keys in [k0, k0 + lim): the live keys are
// counted into buckets by their high bits, then ranked inside their bucket by
// comparison (keys are distinct).  Where some bucket holds many keys (codes
// cluster at every scale) the buckets lie between sampled keys instead, which
// bounds them by the sample's spacing whatever the distribution.
template <typename T, typename KT, int SLOTS, typename Place, typename Write>
__device__ __forceinline__ int win_emit_hash(WinSmem<KT, SLOTS>& sm, WinShared& sh, int& row, KT k0, KT lim,
                                             Place place, Write write) {
  constexpr int PER = SLOTS / WT;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  KT k[PER];
  unsigned lv = 0;
#pragma unroll
  for (int q = 0; q < PER; ++q) {
    const int s = tid + q * WT;
    k[q] = sm.key[s];
    if (k[q] != 0 && win_live<T>(win_value<T, KT, SLOTS>(sm, s))) lv |= 1u << q;
    k[q] -= 1;
  }
  {
    const int c = __reduce_add_sync(WFULL, __popc(lv));
    if (lane == 0) sh.cnt[warp] = c;
  }
  for (int i = tid; i < WNB / 2; i += WT) sm.u.cnt[i] = 0;
  if (tid == 0) sh.big = 0;
  __syncthreads();   // every key is in registers, the counts are clear
  const int n = __reduce_add_sync(WFULL, lane < WNW ? sh.cnt[lane] : 0);
  int shf = 0;
  while (((lim - 1) >> shf) >= (KT)WNB) ++shf;
  auto bucket = [&](KT x) -> int { return (int)((x - k0) >> shf) & (WNB - 1); };
#pragma unroll
  for (int q = 0; q < PER; ++q)
    if (lv & (1u << q)) {
      const int b = bucket(k[q]);
      atomicAdd(&sm.u.cnt[b >> 1], 1u << (16 * (b & 1)));
    }
  __syncthreads();
  {
    constexpr int W = WNB / 2 / WT;   // words per thread
    uint32_t c[W];
    int s = 0;
#pragma unroll
    for (int i = 0; i < W; ++i) {
      c[i] = sm.u.cnt[tid * W + i];
      s += (int)((c[i] & 0xffffu) + (c[i] >> 16));
      if ((c[i] & 0xffffu) > WCROWD || (c[i] >> 16) > WCROWD) sh.big = 1;
    }
    uint32_t run = (uint32_t)win_scan(s, sh.ws, row);
#pragma unroll
    for (int i = 0; i < W; ++i) {
      const uint32_t a = c[i] & 0xffffu, b = c[i] >> 16;
      sm.u.cnt[tid * W + i] = run | ((run + a) << 16);
      run += a + b;
    }
  }
  __syncthreads();
  if (sh.big == 0) {   // uniform
#pragma unroll
    for (int q = 0; q < PER; ++q)
      if (lv & (1u << q)) {
        const int b = bucket(k[q]);
        const uint32_t old = atomicAdd(&sm.u.cnt[b >> 1], 1u << (16 * (b & 1)));
        sm.key[(old >> (16 * (b & 1))) & (SLOTS - 1)] = k[q];
      }
    __syncthreads();   // the keys by bucket are written, each count is its bucket's end
    const int64_t pos = place(n);
#pragma unroll
    for (int q = 0; q < PER; ++q)
      if (lv & (1u << q)) {
        const int b = bucket(k[q]);
        const int e = (int)((sm.u.cnt[b >> 1] >> (16 * (b & 1))) & 0xffffu);
        int rank = b ? (int)((sm.u.cnt[(b - 1) >> 1] >> (16 * ((b - 1) & 1))) & 0xffffu) : 0;
        for (int x = rank; x < e; ++x) rank += sm.key[x] < k[q] ? 1 : 0;
        write(pos + rank, k[q], win_value<T, KT, SLOTS>(sm, tid + q * WT));
      }
    return n;
  }
  KT mine = ~(KT)0;
#pragma unroll
  for (int q = PER - 1; q >= 0; --q)
    if (lv & (1u << q)) mine = k[q];
  win_splitters<KT, SLOTS>(sm, mine);
  auto between = [&](KT x) -> int { return win_between<KT, SLOTS>(sm, x); };
#pragma unroll
  for (int q = 0; q < PER; ++q)
    if (lv & (1u << q)) atomicAdd(&sm.u.g.n[between(k[q])], 1u);
  __syncthreads();
  {
    const int c = tid < WSPLIT ? (int)sm.u.g.n[tid] : 0;
    const int at = win_scan(c, sh.ws, row);
    if (tid < WSPLIT) sm.u.g.n[tid] = (uint32_t)at;
  }
  __syncthreads();
#pragma unroll
  for (int q = 0; q < PER; ++q)
    if (lv & (1u << q)) sm.key[atomicAdd(&sm.u.g.n[between(k[q])], 1u) & (SLOTS - 1)] = k[q];
  __syncthreads();
  const int64_t pos = place(n);
#pragma unroll
  for (int q = 0; q < PER; ++q)
    if (lv & (1u << q)) {
      const int b = between(k[q]);
      const int e = (int)sm.u.g.n[b];
      int rank = b ? (int)sm.u.g.n[b - 1] : 0;
      for (int x = rank; x < e; ++x) rank += sm.key[x] < k[q] ? 1 : 0;
      write(pos + rank, k[q], win_value<T, KT, SLOTS>(sm, tid + q * WT));
    }
  return n;
}

// The same for a window whose pairs are a list (n of at most win_list_cap, in
// global memory or in the table's own space), where most pairs have a key of their own: the pairs are ordered as
// the keys of a table are, equal keys next to each other, and each run of
// equal keys becomes one term.  Without the table a pair costs no probing, and
// the rows are full.  Returns -1 where the keys cluster, or many are equal (the
// table's case): nothing has been placed.
template <typename T, typename KT, int SLOTS, typename Place, typename Write>
__device__ __forceinline__ int win_emit_list(WinSmem<KT, SLOTS>& sm, WinShared& sh, int& row, KT k0, KT lim, int n,
                                             const KT* so, const uint64_t* sv, Place place, Write write) {
  constexpr int ROWS = win_list_cap<SLOTS>() / WT;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  KT k[ROWS];
  uint64_t v[ROWS];
#pragma unroll
  for (int q = 0; q < ROWS; ++q) {
    k[q] = 0;
    v[q] = 0;
    if (tid + q * WT < n) {
      k[q] = so[tid + q * WT];
      v[q] = sv[tid + q * WT];
    }
  }
  for (int i = tid; i < WNB / 2; i += WT) sm.u.cnt[i] = 0;
  if (tid == 0) sh.big = 0;
  __syncthreads();   // every pair is in registers, the counts are clear
  int shf = 0;
  while (((lim - 1) >> shf) >= (KT)WNB) ++shf;
  auto bucket = [&](KT x) -> int { return (int)((x - k0) >> shf) & (WNB - 1); };
#pragma unroll
  for (int q = 0; q < ROWS; ++q)
    if (tid + q * WT < n) {
      const int b = bucket(k[q]);
      atomicAdd(&sm.u.cnt[b >> 1], 1u << (16 * (b & 1)));
    }
  __syncthreads();
  {
    constexpr int W = WNB / 2 / WT;   // words per thread
    uint32_t c[W];
    int s = 0, work = 0;
#pragma unroll
    for (int i = 0; i < W; ++i) {
      c[i] = sm.u.cnt[tid * W + i];
      const int a = (int)(c[i] & 0xffffu), b = (int)(c[i] >> 16);
      s += a + b;
      work += a * a + b * b;   // comparisons of the ranking
    }
    work = __reduce_add_sync(WFULL, work);
    if (lane == 0) atomicAdd(&sh.big, work);
    uint32_t run = (uint32_t)win_scan(s, sh.ws, row);
#pragma unroll
    for (int i = 0; i < W; ++i) {
      const uint32_t a = c[i] & 0xffffu, b = c[i] >> 16;
      sm.u.cnt[tid * W + i] = run | ((run + a) << 16);
      run += a + b;
    }
  }
  __syncthreads();
  if (sh.big > (int)WCROWD * n) return -1;   // uniform
  uint32_t at[(ROWS + 1) / 2] = {};   // places, then ranks, 16 bits each
  auto get = [&](int q) -> int { return (int)((at[q >> 1] >> (16 * (q & 1))) & 0xffffu); };
  auto set = [&](int q, int x) {
    at[q >> 1] = (at[q >> 1] & (0xffff0000u >> (16 * (q & 1)))) | ((uint32_t)x << (16 * (q & 1)));
  };
  // rank among the keys [s, e) of the bucket, equal ones in the order of their places
  auto rank_of = [&](int q, int s, int e) {
    const int mine = get(q);
    int rank = s;
    for (int x = s; x < e; ++x) {
      const KT y = sm.key[x];
      rank += y < k[q] || (y == k[q] && x < mine) ? 1 : 0;
    }
    set(q, rank);
  };
#pragma unroll
  for (int q = 0; q < ROWS; ++q)
    if (tid + q * WT < n) {
      const int b = bucket(k[q]);
      const uint32_t old = atomicAdd(&sm.u.cnt[b >> 1], 1u << (16 * (b & 1)));
      const int p = (int)((old >> (16 * (b & 1))) & (SLOTS - 1));
      sm.key[p] = k[q];
      set(q, p);
    }
  __syncthreads();   // the keys by bucket are written, each count is its bucket's end
#pragma unroll
  for (int q = 0; q < ROWS; ++q)
    if (tid + q * WT < n) {
      const int b = bucket(k[q]);
      rank_of(q, b ? (int)((sm.u.cnt[(b - 1) >> 1] >> (16 * ((b - 1) & 1))) & 0xffffu) : 0,
              (int)((sm.u.cnt[b >> 1] >> (16 * (b & 1))) & 0xffffu));
    }
  __syncthreads();   // the buckets have been read
#pragma unroll
  for (int q = 0; q < ROWS; ++q)
    if (tid + q * WT < n) {
      const int r = get(q) & (SLOTS - 1);
      sm.key[r] = k[q];
      sm.val[r] = v[q];
    }
  __syncthreads();
  // each warp a contiguous part: the first pair of every key adds up the others
  unsigned lv = 0;
  int c = 0;
#pragma unroll
  for (int q = 0; q < ROWS; ++q) {
    const int i = (warp * ROWS + q) * 32 + lane;
    bool live = false;
    if (i < n) {
      k[q] = sm.key[i];
      if (i == 0 || sm.key[i - 1] != k[q]) {
        v[q] = sm.val[i];
        for (int x = i + 1; x < n && sm.key[x] == k[q]; ++x) {
          if constexpr (std::is_same<T, double>::value)
            v[q] = (uint64_t)__double_as_longlong(__longlong_as_double((long long)v[q]) +
                                                  __longlong_as_double((long long)sm.val[x]));
          else
            v[q] += sm.val[x];
        }
        live = win_live<T>(v[q]);
      }
    }
    const unsigned b = __ballot_sync(WFULL, live);
    if (live) lv |= 1u << q;
    c += __popc(b);
  }
  if (lane == 0) sh.cnt[warp] = c;
  __syncthreads();
  const int part = lane < WNW ? sh.cnt[lane] : 0;
  const int total = __reduce_add_sync(WFULL, part), mine = __reduce_add_sync(WFULL, lane < warp ? part : 0);
  int64_t pos = place(total) + mine;
#pragma unroll
  for (int q = 0; q < ROWS; ++q) {
    const bool live = (lv >> q) & 1u;
    const unsigned b = __ballot_sync(WFULL, live);
    if (live) write(pos + __popc(b & ((1u << lane) - 1u)), k[q], v[q]);
    pos += __popc(b);
  }
  return total;
}

// m base windows of one product, from wfirst on, by the whole CTA; t: the
// first's number.  The terms of a piece go to a stretch of the raw arrays (no
// CTA waits for another); the run keeps its pieces as a list, in key order,
// for the copy that puts the product together.
template <typename KT, int SLOTS>
struct WinBlock {
  WinSmem<KT, SLOTS> sm;
  WinShared sh;
};

// The CTA's shared memory (named here and not passed, so that functions that
// are not inlined still address it as shared memory).
template <typename KT, int SLOTS>
__device__ __forceinline__ WinBlock<KT, SLOTS>& win_block() {
  extern __shared__ __align__(16) unsigned char win_raw[];
  return *(WinBlock<KT, SLOTS>*)win_raw;
}

template <typename T, typename KT, int SLOTS>
struct WinRun {
  Prod& P;
  const WinOut& O;
  int64_t t, m, out;
  int32_t last;   // thread 0: the run's newest piece
  int row;        // of the block scans' scratch

  // a stretch of n terms (none without terms); by every thread
  __device__ __forceinline__ int64_t place(int n) {
    auto& sh = win_block<KT, SLOTS>().sh;
    if (threadIdx.x == 0) {
      const int64_t pos = (int64_t)atomicAdd(&O.used[0], (unsigned long long)n);
      const int64_t s = n > 0 ? (int64_t)atomicAdd(&O.used[1], 1ull) : -1;
      if (pos + n > O.cap) atomicOr(&P.status, ST_OUTCAP);
      if (s < 0) {
      } else if (s < O.nseg) {
        O.seg[s] = WinSeg{pos, n, -1};
        if (last < 0) O.head[t] = (int32_t)s + 1; else O.seg[last].next = (int32_t)s;
        last = (int32_t)s;
      } else {
        atomicOr(&P.status, ST_WINDOW);
      }
      sh.excl = pos;
    }
    __syncthreads();
    return sh.excl;
  }

  // writes a term to its place
  __device__ __forceinline__ auto writer(int64_t key0) {
    uint64_t* const key = O.key;
    uint64_t* const val = O.val;
    const int64_t cap = O.cap;
    return [key, val, cap, key0](int64_t pos, KT off, uint64_t v) {
      if ((uint64_t)pos < (uint64_t)cap) {
        key[pos] = (uint64_t)key0 + (uint64_t)off;
        val[pos] = v;
      }
    };
  }

  // n pairs with keys [key0 + k0, key0 + k0 + lim) as a list; false: not done
  __device__ __forceinline__ bool list(int64_t key0, KT k0, KT lim, int n, const KT* so, const uint64_t* sv) {
    auto& sm = win_block<KT, SLOTS>().sm;
    auto& sh = win_block<KT, SLOTS>().sh;
    const int c = win_emit_list<T, KT, SLOTS>(sm, sh, row, k0, lim, n, so, sv,
                                              [&](int x) -> int64_t { return place(x); }, writer(key0));
    __syncthreads();   // the table's space is free
    if (c >= 0) out += c;
    return c >= 0;
  }

  // keys [cur, stop) through the table, in pieces that fit it; given their n
  // pairs as a list (n >= 0; offsets from key cur - delta), from there
  __device__ __forceinline__ void pieces(const WinDesc& D, int64_t cur, int64_t stop, int n, KT delta, const KT* so,
                                         const uint64_t* sv) {
    auto& sm = win_block<KT, SLOTS>().sm;
    auto& sh = win_block<KT, SLOTS>().sh;
    constexpr int64_t MAXLIM = sizeof(KT) == 4 ? (int64_t)0xfffffff0ll : INT64_MAX;
    int64_t end = stop;
    while (cur < stop) {
      const int64_t E = (end - cur) > MAXLIM ? cur + MAXLIM : end;
      const bool direct = E - cur <= SLOTS;
      win_clear<KT, SLOTS>(sm, direct);
      if (n >= 0) {
        if (threadIdx.x == 0) sh.full = 0;
        __syncthreads();
        for (int i = threadIdx.x; i < n; i += WT)
          if (!win_add<T, KT, SLOTS>(sm, so[i] - delta, sv[i], direct)) *(volatile int*)&sh.full = 1;
      } else {
        win_subs(sh, P, D, cur, E);   // (barriers: the table is clear)
        win_form<T, KT, SLOTS>(sm, sh, D, [&](bool act, KT off, uint64_t v) {
          // (a full table answers slowly: no more pairs after the first failure)
          if (act && !*(volatile int*)&sh.full && !win_add<T, KT, SLOTS>(sm, off, v, direct))
            *(volatile int*)&sh.full = 1;
        });
      }
      __syncthreads();
      if (sh.full) {   // halve the piece (a piece of at most SLOTS keys never fills up)
        end = cur + (E - cur) / 2;
        n = -1;
        __syncthreads();   // every thread has seen the flag
        continue;
      }
      auto at = [&](int n) -> int64_t { return place(n); };
      auto write = writer(cur - P.klo);
      if (direct) out += win_emit_direct<T, KT, SLOTS>(sm, sh, (int)(E - cur), at, write);
      else out += win_emit_hash<T, KT, SLOTS>(sm, sh, row, (KT)0, (KT)(E - cur), at, write);
      __syncthreads();   // the table is cleared for the next piece or window
      cur = E;
      end = stop;
    }
  }

  // The pairs of all m windows, formed in one walk and put down by window in
  // the CTA's staging area (which L2 holds).
  __device__ __forceinline__ void stage(const WinDesc& D, const int64_t* start, KT* soff, uint64_t* sval) {
    constexpr int CAP = win_stage_cap<SLOTS>();
    auto& sm = win_block<KT, SLOTS>().sm;
    auto& sh = win_block<KT, SLOTS>().sh;
    const int64_t W0 = start[0];
    if (threadIdx.x < WST) {
      sh.fill[threadIdx.x] = 0;
      const int64_t w = threadIdx.x + 1;
      sh.bnd[threadIdx.x] = w < m ? (uint64_t)(start[w] - W0) : ~0ull;
    }
    win_subs(sh, P, D, W0, start[m]);   // (barriers)
    const int top = 1 << (31 - __clz((int)m));   // steps of the search over m windows
    win_form<T, KT, SLOTS>(sm, sh, D, [&](bool act, KT off, uint64_t v) {
      int w = 0;
      for (int step = top; step > 0; step >>= 1) w += w + step < (int)m && sh.bnd[w + step - 1] <= (uint64_t)off ? step : 0;
      if (act) {
        const int at = atomicAdd(&sh.fill[w], 1);
        if (at < CAP) {
          soff[w * CAP + at] = off;
          sval[w * CAP + at] = v;
        }
      }
    });
    __syncthreads();
  }

  // The pairs of one window as a list in the table's space; returns their
  // number (the list holds win_list_cap of them).
  __device__ __forceinline__ int form_list(const WinDesc& D, int64_t W0, int64_t W1) {
    constexpr int CAP = win_list_cap<SLOTS>();
    auto& sm = win_block<KT, SLOTS>().sm;
    auto& sh = win_block<KT, SLOTS>().sh;
    const int lane = threadIdx.x & 31;
    if (threadIdx.x == 0) sh.fill[0] = 0;
    win_subs(sh, P, D, W0, W1);   // (barriers)
    win_form<T, KT, SLOTS>(sm, sh, D, [&](bool act, KT off, uint64_t v) {
      const unsigned b = __ballot_sync(WFULL, act);
      int at = 0;
      if (lane == 0) at = atomicAdd(&sh.fill[0], __popc(b));
      at = __shfl_sync(WFULL, at, 0) + __popc(b & ((1u << lane) - 1u));
      if (act && at < CAP) {
        sm.key[at] = off;
        sm.val[at] = v;
      }
      if (act && at >= CAP) *(volatile int*)&sh.full = 1;   // no use in going on
    });
    __syncthreads();
    return sh.fill[0];
  }

  // The run.  Where most pairs have a key of their own (estimated) a window is
  // ordered as a list of its pairs, and where its pairs are also few against
  // the terms walked for it, the run's windows are formed in one walk first;
  // windows that do not fit a list, and all others, go through the table.
  __device__ __forceinline__ void run(int64_t wfirst, KT* soff, uint64_t* sval) {
    constexpr int CAP = win_list_cap<SLOTS>(), SCAP = win_stage_cap<SLOTS>();
    auto& sm = win_block<KT, SLOTS>().sm;
    auto& sh = win_block<KT, SLOTS>().sh;
    const WinDesc& D = *P.win.desc;
    const int64_t* start = P.win.start + wfirst;
    const bool narrow = sizeof(KT) == 8 || start[m] - start[0] <= (int64_t)0xfffffff0ll;   // offsets fit
    const bool sparse = narrow && P.win.merge && win_distinct(D, wfirst, D.nw) > 0.5f;
    // (the staging area holds Win::stage windows, at most WST; a run that starts where keys
    // are distinct may go on into a region where they are not, whose windows are
    // weighed otherwise)
    const bool staged = sparse && m > 1 && m <= min(P.win.stage, WST);
    const bool listed = sparse && m == 1 && start[1] - start[0] > SLOTS;
    if (staged) stage(D, start, soff, sval);
    const int parts = staged ? (int)m : 1;
    for (int w = 0; w < parts; ++w) {
      int n = staged ? sh.fill[w] : listed ? form_list(D, start[0], start[1]) : CAP + 1;
      const bool kept = staged && n <= SCAP;   // the window's pairs are in the staging area
      const int halves = kept && n > CAP ? 2 : 1;
      const int64_t w0 = start[w], w1 = staged ? start[w + 1] : start[m];
      for (int h = 0; h < halves; ++h) {
        const int64_t a = w0 + (w1 - w0) / halves * h, b = h + 1 < halves ? w0 + (w1 - w0) / halves : w1;
        const KT k0 = (KT)(a - start[0]), lim = (KT)(b - a);
        const KT* so = staged ? soff + w * SCAP : sm.key;
        const uint64_t* sv = staged ? sval + w * SCAP : sm.val;
        int c = n;
        if (halves == 2) {   // half of the pairs, into the table's space
          if (threadIdx.x == 0) sh.nlong = 0;
          __syncthreads();
          for (int i = threadIdx.x; i < n; i += WT) {
            const KT off = so[i];
            if (off - k0 < lim) {
              const int at = atomicAdd(&sh.nlong, 1);
              if (at < CAP) {
                sm.key[at] = off;
                sm.val[at] = sv[i];
              }
            }
          }
          __syncthreads();
          c = sh.nlong;
        }
        const bool in_table = halves == 2 || !staged;
        const bool done = c <= CAP && list(start[0] - P.klo, k0, lim, c, in_table ? sm.key : so, in_table ? sm.val : sv);
        if (!done) pieces(D, a, b, kept && halves == 1 ? n : -1, k0, so, sv);   // uniform
      }
    }
    if (threadIdx.x == 0) {
      O.count[t] = out;
      atomicAdd((unsigned long long*)&P.nout, (unsigned long long)out);
    }
  }
};

template <typename KT, int SLOTS>
__host__ __device__ constexpr size_t win_staging_bytes() {   // per window
  return (size_t)win_stage_cap<SLOTS>() * (sizeof(KT) + 8);
}

// Persistent: CTAs take runs of windows in order from a ticket.
template <typename KT, int SLOTS>
__global__ void __launch_bounds__(WT, 2) k_window(Prod* __restrict__ prods, const int32_t* __restrict__ wprods,
                                                  const int64_t* __restrict__ rprefix, int nwp,
                                                  unsigned long long* __restrict__ ticket, const WinOut O,
                                                  unsigned char* staging, int stage_max) {
  WinShared& sh = win_block<KT, SLOTS>().sh;
  const int64_t nrun = rprefix[nwp];
  uint64_t* sval = (uint64_t*)(staging + (size_t)blockIdx.x * stage_max * win_staging_bytes<KT, SLOTS>());
  KT* soff = (KT*)(sval + (size_t)stage_max * win_stage_cap<SLOTS>());
  for (;;) {
    if (threadIdx.x == 0) sh.t = (int64_t)atomicAdd(ticket, 1ull);
    __syncthreads();
    const int64_t t = sh.t;
    if (t >= nrun) break;
    int lo = 0, hi = nwp - 1;
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (rprefix[mid] <= t) lo = mid; else hi = mid - 1;
    }
    Prod& P = prods[wprods[lo]];
    if (threadIdx.x == 0) sh.full = *(volatile uint32_t*)&P.status != 0;
    __syncthreads();
    const bool failed = sh.full != 0;
    __syncthreads();
    if (!failed) {   // (a failed product has no terms; the flag is read once for the CTA)
      const int64_t w = P.win.run[t - rprefix[lo]], m = P.win.run[t - rprefix[lo] + 1] - w;
      if (P.f64) {
        WinRun<double, KT, SLOTS> r{P, O, t, m, 0, -1, 0};
        r.run(w, soff, sval);
      } else {
        WinRun<int64_t, KT, SLOTS> r{P, O, t, m, 0, -1, 0};
        r.run(w, soff, sval);
      }
    }
    __syncthreads();
  }
}

// Puts the products together: the terms of run t (windows in product and key
// order) go from their stretches to the position that the counts of the runs
// before it give.  Terms: what becomes of a term at its position.  base: where
// the first run's terms go (null: 0); *total: the position after the last
// run's (null: not wanted).  before: the scanned counts, or null (few windows):
// each CTA adds them up.  The CTAs of a column of the grid share its runs'
// stretches: two of them, since runs differ in length (1 to 8 a column are within 2 %).
constexpr int WIN_PUT_TERMS = 4;   // terms of a thread at once, 256 apart: loads in flight
template <typename Terms>
__device__ __forceinline__ void win_put(Prod* prods, const int32_t* wprods, const int64_t* rprefix, int nwp,
                                        const WinOut& O, const int64_t* before, const int64_t* base_ptr,
                                        int64_t* total, Terms terms) {
  __shared__ int64_t ws[8];
  const int tid = threadIdx.x, lane = tid & 31;
  const int64_t nrun = rprefix[nwp];
  const int64_t base = base_ptr ? *base_ptr : 0;
  for (int64_t t = blockIdx.x; t <= nrun; t += gridDim.x) {
    const int64_t n = t < nrun ? O.count[t] : 0;
    int lo = 0, hi = nwp - 1;
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (rprefix[mid] <= t) lo = mid; else hi = mid - 1;
    }
    const bool first = t < nrun && rprefix[lo] == t;   // of product lo
    if (n == 0 && !first && t < nrun) continue;   // uniform
    int64_t pos;
    if (before) {
      pos = t < nrun ? before[t] : before[nrun - 1] + O.count[nrun - 1];
    } else {
      int64_t s = 0;
      for (int64_t x = tid; x < t; x += 256) s += O.count[x];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(WFULL, s, o);
      if (lane == 0) ws[tid >> 5] = s;
      __syncthreads();
      pos = 0;
      for (int w = 0; w < 8; ++w) pos += ws[w];
      __syncthreads();
    }
    pos += base;
    if (t == nrun) {
      if (tid == 0 && blockIdx.y == 0 && total) *total = pos;
      break;
    }
    if (first && tid == 0 && blockIdx.y == 0) prods[wprods[lo]].out_start = pos;
    for (int32_t s = O.head[t] - 1; s >= 0 && n > 0;) {
      const WinSeg g = O.seg[s];
      const int64_t m = min((int64_t)g.n, O.cap - g.pos);
      constexpr int U = WIN_PUT_TERMS;
      for (int64_t i0 = tid + 256 * U * (int64_t)blockIdx.y; i0 < m; i0 += 256 * U * (int64_t)gridDim.y) {
        const int cnt = (int)min((int64_t)U, (m - i0 + 255) >> 8);
        uint64_t k[U], v[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
          k[u] = v[u] = 0;
          if (u < cnt) {
            k[u] = __ldcs(O.key + g.pos + i0 + 256 * u);
            v[u] = __ldcs(O.val + g.pos + i0 + 256 * u);
          }
        }
        terms(pos + i0, cnt, k, v);
      }
      pos += g.n;
      s = g.next;
    }
  }
}

__global__ void __launch_bounds__(256) k_win_copy(Prod* __restrict__ prods, const int32_t* __restrict__ wprods,
                                                  const int64_t* __restrict__ rprefix, int nwp, const WinOut O,
                                                  const int64_t* __restrict__ before,
                                                  const int64_t* __restrict__ base_ptr, int64_t* __restrict__ total,
                                                  int64_t cap, uint64_t* __restrict__ okey,
                                                  uint64_t* __restrict__ oval) {
  win_put(prods, wprods, rprefix, nwp, O, before, base_ptr, total, [&](int64_t q, int cnt, const uint64_t* key, const uint64_t* val) {
#pragma unroll
    for (int u = 0; u < WIN_PUT_TERMS; ++u, q += 256)
      if (u < cnt && q < cap) {
        okey[q] = key[u];
        oval[q] = val[u];
      }
  });
}

// decode_digits of a thread's terms, 256 places apart (cnt of them): a digit's
// divisor is fetched and its row's address formed once for all of them.  At
// 37 million Poisson terms of seven digits 252 M warp instructions against 354 M
// for a term at a time, 0.52 against 0.60 ms.
__device__ __forceinline__ void decode_digits_put(const Divisor* div, const int32_t* lo, int n, uint64_t* x,
                                                  int cnt, int32_t* __restrict__ p, int64_t ld) {
  constexpr int U = WIN_PUT_TERMS;
  for (int k = 0; k < n; ++k, p += ld) {
    const int32_t l = lo[k];
    uint32_t m[U];
    if (k + 1 < n) {
      const Divisor v = div[k];
      uint64_t high = 0;
#pragma unroll
      for (int u = 0; u < U; ++u) high |= x[u];
      if (high >> 32) {
#pragma unroll
        for (int u = 0; u < U; ++u) {
          int64_t r;
          x[u] = (uint64_t)divmod((int64_t)x[u], v, &r);
          m[u] = (uint32_t)r;
        }
      } else {
        const uint32_t d = (uint32_t)v.d;   // widths are below 2^31
#pragma unroll
        for (int u = 0; u < U; ++u) {
          uint32_t q = __umulhi((uint32_t)x[u], v.r32);
          m[u] = (uint32_t)x[u] - q * d;
          if (m[u] >= d) { ++q; m[u] -= d; }
          x[u] = q;
        }
      }
    } else {
#pragma unroll
      for (int u = 0; u < U; ++u) m[u] = (uint32_t)x[u];   // (below the last width)
    }
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (u < cnt) p[256 * u] = (int32_t)m[u] + l;
  }
}

// The same for a single product, its terms decoded straight into the caller's
// arrays: no copy and no second pass.  Bound by its writes (1.43 GB in columns of
// 4 bytes, 0.76 GB read: 4.2 TB/s) at 37 million Poisson terms: 0.52 ms, against
// 0.34 + 0.44 ms for a copy and a decode of it with plain divisions.  Nothing is
// written when the product does not fit the arrays.
template <bool SERIES>
__global__ void __launch_bounds__(256) k_win_decode(Prod* __restrict__ prods, const int32_t* __restrict__ wprods,
                                                    const int64_t* __restrict__ rprefix, const WinOut O,
                                                    const int64_t* __restrict__ before, const SeriesOut D) {
  __shared__ Prod s_prod;
  const Prod& P = shared_prod(&prods[wprods[0]], &s_prod);
  if (P.status || P.nout > D.cap) return;   // uniform
  win_put(prods, wprods, rprefix, 1, O, before, nullptr, nullptr, [&](int64_t q, int cnt, const uint64_t* key, const uint64_t* val) {
    constexpr int U = WIN_PUT_TERMS;
    uint64_t pc[U], tc[U];
    const int64_t per_kind = P.T2 * P.Wp;
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int64_t code = (int64_t)key[u] + P.klo;   // keys are relative to the key window
      if (u < cnt) {
        if (D.codes) D.codes[q + 256 * u] = code;
        D.coef[q + 256 * u] = val[u];
      }
      pc[u] = (uint64_t)code;
      if (SERIES) {
        const int64_t kd = code >= per_kind ? 1 : 0;   // keys lie below 2 * per_kind
        int64_t r;
        tc[u] = (uint64_t)(divmod(code - kd * per_kind, P.divWp, &r) + (P.T2 - 1));   // T2 - 1 = sum_k c_k R_k
        pc[u] = (uint64_t)r;
        if (u < cnt && D.kind) D.kind[q + 256 * u] = (uint8_t)kd;
      }
    }
    if (D.exps && !P.graded) {
      decode_digits_put(P.div, P.omin, P.np, pc, cnt, D.exps + q, D.cap);
    } else if (D.exps) {
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (u < cnt) decode_poly_part(P, (int64_t)pc[u], D.exps, D.cap, q + 256 * u);
    }
    if (SERIES && D.trig) decode_digits_put(P.div + P.np, P.omin + P.np, P.nt, tc, cnt, D.trig + q, D.cap);
  });
}

// How many pairs share a key, by region of the product's windows: the mean of
// 1 / (pairs with the key of a random pair) is the number of terms per pair.
// One CTA per sampled pair, which searches the partners of every A term that
// give the same key.
constexpr int WIN_DUP_SAMPLES = 32 * WIN_REGIONS;

__global__ void __launch_bounds__(256) k_win_dup(const Prod* __restrict__ prods, const int32_t* __restrict__ wprods) {
  const Prod& P = prods[wprods[0]];
  if (P.status || !P.win.merge) return;   // uniform
  WinDesc& D = *P.win.desc;
  const Operand& A = P.win.swap ? P.g : P.f;
  const Operand& B = P.win.swap ? P.f : P.g;
  if (A.nkeep <= 0 || B.nkeep <= 0) return;
  const int64_t half = P.T2 * P.Wp;
  // the sampled pair's key (every thread forms the same)
  const uint64_t u = 2ull * blockIdx.x + 1ull;
  const int64_t i = (int64_t)(((uint64_t)hash32(u) * (uint64_t)A.nkeep) >> 32);
  const int64_t j = (int64_t)(((uint64_t)hash32(u + 1000000007ull) * (uint64_t)B.nkeep) >> 32);
  int64_t key = A.code[i] + B.code[j];
  int kd = 0;
  if (P.nt) {
    kd = A.kind[i] ^ B.kind[j];
    int64_t T = A.tcode[i] + ((hash32(u + 77ull) & 1u) ? B.tcode[j] : -B.tcode[j]);
    if (T < 0) T = -T;
    if (T == 0 && kd) return;
    key += T * P.Wp;
  }
  const int64_t full = key + kd * half;
  if (full < P.klo || full >= P.klo + P.kspan) return;
  int count = 0;
  if (P.nt == 0) {
    const WinList& L = D.L[0];
    for (int64_t x = threadIdx.x; x < D.na; x += blockDim.x) {
      int64_t l, h;
      g_lower_bound2(L.code, L.n, L.idx, L.nidx, L.shift, key - A.code[x], key - A.code[x] + 1, &l, &h);
      count += (int)(h - l);
    }
  } else {
    for (int64_t x = threadIdx.x; x < 2 * D.na; x += blockDim.x) {
      const bool mirror = x >= D.na;
      const int64_t q = mirror ? x - D.na : x;
      if (mirror && key < P.Wp) continue;
      const WinList& L = D.L[(q >= D.nca ? 1 : 0) ^ kd];
      if (L.n <= 0) continue;
      const int64_t want = key - P.win.acode[x] - L.base;
      int64_t l, h;
      g_lower_bound2(L.code, L.n, L.idx, L.nidx, L.shift, want, want + 1, &l, &h);
      count += (int)(h - l);
    }
  }
  __shared__ int s_count;
  if (threadIdx.x == 0) s_count = 0;
  __syncthreads();
  count = __reduce_add_sync(WFULL, count);
  if ((threadIdx.x & 31) == 0) atomicAdd(&s_count, count);
  __syncthreads();
  if (threadIdx.x == 0) {
    const int64_t nw = D.nw;
    const int64_t w = max((int64_t)0, lower_bound_i64(P.win.start, nw, full + 1) - 1);   // the key's window
    const int r = (int)(w * WIN_REGIONS / nw);
    atomicAdd(&D.rs[r], 1.0f / (float)max(1, s_count));
    atomicAdd(&D.rn[r], 1.0f);
  }
}

cudaError_t launch_win_plan(Prod* dprods, const int32_t* dwprods, int nwp, bool poisson, const int* merging, int merge,
                            int64_t max_terms, int64_t max_samples, int64_t max_bins, int64_t max_windows, int64_t* drprefix,
                            int64_t slots, int64_t ctas,
                            unsigned int* ddone, cudaStream_t s) {
  if (nwp <= 0) return cudaSuccess;
  auto gx = [](int64_t n, int64_t most) {
    const int64_t g = (n + 255) / 256;
    return (unsigned)(g < 1 ? 1 : (g > most ? most : g));
  };
  if (poisson) k_win_lists<<<dim3(gx(max_terms, 64), nwp), 256, 0, s>>>(dprods, dwprods);
  k_win_index<<<dim3(gx(2 * max_terms, 64), 2 * nwp), 256, 0, s>>>(dprods, dwprods);
  const int64_t most = nwp > 64 ? 32 : 2048 / nwp;
  k_win_hist<<<dim3(gx(max_samples, most), nwp), 256, 0, s>>>(dprods, dwprods);
  const size_t smem = std::max((size_t)(max_bins + max_bins / 32 + 1) * 4, (size_t)wc_sort_size(max_windows) * 8);
  cudaError_t e = raise_smem_limit((const void*)k_win_cut, smem);
  if (e != cudaSuccess) return e;
  k_win_cut<<<nwp, WC_THREADS, smem, s>>>(dprods, dwprods, nwp, drprefix, slots, ctas, merge ? nullptr : ddone);
  if (merge) {
    for (int i = 0; i < merge; ++i) k_win_dup<<<WIN_DUP_SAMPLES, 256, 0, s>>>(dprods, dwprods + merging[i]);
    k_win_runs<<<nwp, WC_THREADS, 0, s>>>(dprods, dwprods, nwp, drprefix, slots, ctas, ddone);
  }
  return cudaGetLastError();
}

template <typename KT, int SLOTS>
static cudaError_t launch_window_t(Prod* dprods, const int32_t* dwprods, const int64_t* drprefix, int nwp,
                                   int64_t* dticket, const WinOut& out, unsigned char* staging, int stage_max, int sms,
                                   cudaStream_t s) {
  const size_t smem = sizeof(WinBlock<KT, SLOTS>);
  auto* fn = k_window<KT, SLOTS>;
  cudaError_t e = raise_smem_limit((const void*)fn, smem);
  if (e != cudaSuccess) return e;
  int per = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, fn, WT, smem) != cudaSuccess || per < 1) {
    cudaGetLastError();
    per = 1;
  }
  if (per > WIN_CTAS_PER_SM) per = WIN_CTAS_PER_SM;   // the staging areas
  fn<<<(unsigned)(sms * per), WT, smem, s>>>(dprods, dwprods, drprefix, nwp, (unsigned long long*)dticket, out,
                                             staging, stage_max);
  return cudaGetLastError();
}

size_t win_staging(int stage_max, int sms) {
  return (size_t)sms * WIN_CTAS_PER_SM * stage_max *
         std::max(win_staging_bytes<uint32_t, WIN_SLOTS_32>(), win_staging_bytes<uint64_t, WIN_SLOTS_64>());
}

cudaError_t launch_window(Prod* dprods, const WinLaunch& L, int64_t* dticket, unsigned char* staging, int stage_max,
                          int sms, cudaStream_t s, int* launches) {
  if (L.nwp <= 0) return cudaSuccess;
  cudaError_t e =
      L.kind == WIN_32
          ? launch_window_t<uint32_t, WIN_SLOTS_32>(dprods, L.prods, L.rprefix, L.nwp, dticket, L.out, staging, stage_max,
                                                    sms, s)
          : launch_window_t<uint64_t, WIN_SLOTS_64>(dprods, L.prods, L.rprefix, L.nwp, dticket, L.out, staging, stage_max,
                                                    sms, s);
  if (e != cudaSuccess) return e;
  *launches += 1;
  if (win_scanned(L)) {
    e = cudaMemcpyAsync(L.before, L.out.count, sizeof(int64_t) * (size_t)L.max_windows, cudaMemcpyDeviceToDevice, s);
    if (e == cudaSuccess) e = launch_scan_exclusive(L.before, L.max_windows, nullptr, L.scan, s);
    *launches += 1;
  }
  return e;
}

constexpr int WIN_PUT_PARTS = 2;
static dim3 put_grid(const WinLaunch& L, int sms) {
  return dim3((unsigned)std::min<int64_t>(L.max_windows + 1, 8 * (int64_t)sms), WIN_PUT_PARTS);
}

cudaError_t launch_win_copy(Prod* dprods, const WinLaunch& L, const int64_t* dbase, int64_t* dtotal, int64_t cap,
                            uint64_t* okey, uint64_t* oval, int sms, cudaStream_t s) {
  if (L.nwp <= 0) return cudaSuccess;
  k_win_copy<<<put_grid(L, sms), 256, 0, s>>>(dprods, L.prods, L.rprefix, L.nwp, L.out,
                                              win_scanned(L) ? L.before : nullptr, dbase, dtotal, cap, okey, oval);
  return cudaGetLastError();
}

cudaError_t launch_win_decode(Prod* dprods, const WinLaunch& L, bool series, const SeriesOut& out, int sms,
                              cudaStream_t s) {
  auto* fn = series ? k_win_decode<true> : k_win_decode<false>;
  fn<<<put_grid(L, sms), 256, 0, s>>>(dprods, L.prods, L.rprefix, L.out, win_scanned(L) ? L.before : nullptr, out);
  return cudaGetLastError();
}

}  // namespace kr
