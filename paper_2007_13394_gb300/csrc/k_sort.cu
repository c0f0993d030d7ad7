// Stable counting sort of particles into 16^3-cell tiles of the mesh.
//
// key = tile * 8 + face class (see pm.h, pm_sort).  The order is a stable
// least-significant-digit radix sort of (key, incoming index) with 7- to 9-bit digits (two
// 9-bit passes cover the 18-bit keys of a 512^3 mesh).  Each CTA owns one contiguous chunk of
// whole 4096-key tiles, at most three CTAs an SM, so a pass is: digit counts per chunk (made by
// the key kernel for the first pass), a scan of them over the chunks, and a scatter in which the
// CTA walks its tiles with its own running digit positions -- nothing waits for another CTA.
// In a tile, warp w ranks 512 contiguous keys in 16 rounds of 32 (ballots for the rank inside
// a round, warp-private digit counters across rounds), one block scan over (digit, warp) gives
// staging offsets, and the keys go out through shared memory in coalesced runs.  A bucket's
// start is a binary search in the sorted keys, done by the gather.
//
// The scatter is bound by instruction issue and by latency inside a tile (SM 60 %, DRAM 21 to 27 %
// of peak at 512^3).  us a pass (counts, scan and scatter), 19 M particles, 9 bits: 28 + 3 + 137
// (with a warp match per round, 4096-key blocks and a three-launch scan: 42 + 15 + 215); the key
// kernel, which no longer counts buckets with global atomics, 103 -> 56.
//
// Near-sorted re-sort (pm_step): the state is in the order of the last step's sort,
// bucket starts bprev, and most particles keep their key.  A stayer (same key, inside
// its old key's range) keeps its relative order; movers are compacted in index order
// and radix-sorted alone.  Old ranges are ordered by key, so among the particles of new
// key B those with index below bprev[B] are exactly the movers from lower keys, those
// inside B's old range are B's stayers, the rest came from higher keys: bucket B is
// [lower movers | stayers | higher movers], which is the stable order.  The result is
// the same permutation as the radix sort from scratch.  A particle outside its old key's
// range (a state not in bprev's order) makes every particle a mover, in index order: then it
// is the radix sort from scratch.  That choice and the number of movers stay on the device:
// the kernels take their ranges from there, and the host never waits.
#include <cuda_runtime.h>

#include <algorithm>

#include "pm_internal.cuh"

namespace pmnu {

namespace {

constexpr int kRadixThreads = 256;
constexpr int kRadixRounds = 16;
constexpr int kRadixTile = kRadixThreads * kRadixRounds;  // 4096 keys per tile
constexpr int kRadixWarps = kRadixThreads / 32;
constexpr int kCountThreads = 512;
constexpr int kCountUnroll = 4;

// Number of movers of a near-sorted re-sort (every particle when the state was not in
// bprev's order), from the device: flags of k_kick_drift_keys<true>, scans in bstart3.
// Counts that are not those of n particles give more than n: err is set (by the caller that has it).
__device__ __forceinline__ int64_t movers_of(const uint32_t* flags, const uint32_t* bstart3, long long nb1, int64_t n,
                                             int* err = nullptr) {
  if (*flags & 1u) return n;
  const int64_t m = scan_difference(bstart3[2 * nb1], bstart3[3 * nb1 - 1]);
  if (m > n && err) atomicOr(err, 1);
  return m > n ? n : m;
}

// ------------------------------------------------------------------ scan
__device__ __forceinline__ uint32_t block_exclusive_scan(uint32_t v, uint32_t* warp_sums,
                                                         uint32_t* total) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  uint32_t x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) warp_sums[w] = x;
  __syncthreads();
  if (w == 0) {
    const int nw = blockDim.x >> 5;
    uint32_t s = lane < nw ? warp_sums[lane] : 0u;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      uint32_t y = __shfl_up_sync(0xffffffffu, s, o);
      if (lane >= o) s += y;
    }
    if (lane < nw) warp_sums[lane] = s;  // inclusive warp prefix
  }
  __syncthreads();
  uint32_t before = (w > 0 ? warp_sums[w - 1] : 0u) + (x - v);
  if (total) *total = warp_sums[(blockDim.x >> 5) - 1];
  return before;
}

// Exclusive scan without a wait between CTAs: a launch sums the tiles of kScanTile words, the next
// one scans each tile behind the sum of the tiles before it, which every CTA adds up itself.  Up to
// kScanFew tiles (meshes of 128^3 or less) the second launch alone, its CTAs adding up the words
// before their tile: a launch costs more than they do.  (One launch whose tiles look back at their
// predecessors' sums, with a bounded wait for them, left the starts unordered when the wait ran
// out, and the paint reads its particles between two starts.)
constexpr int kScanThreads = 512;
constexpr int kScanItems = 8;
constexpr int kScanFew = 8;

__global__ void __launch_bounds__(kScanThreads) k_scan_sums(const uint32_t* in, long long n,
                                                            uint32_t* __restrict__ sums) {
  pdl_begin();
  __shared__ uint32_t ws[32];
  const long long base = (long long)blockIdx.x * kScanTile + threadIdx.x;
  uint32_t s = 0, total;
#pragma unroll
  for (int k = 0; k < kScanItems; ++k) s += base + k * kScanThreads < n ? in[base + k * kScanThreads] : 0u;
  block_exclusive_scan(s, ws, &total);
  if (threadIdx.x == 0) sums[blockIdx.x] = total;
}

// sums null: few tiles
__global__ void __launch_bounds__(kScanThreads) k_scan(const uint32_t* in, long long n,
                                                       const uint32_t* sums, uint32_t* __restrict__ out) {
  pdl_begin();
  __shared__ uint32_t ws[32], wb[32];
  const int t = threadIdx.x;
  const long long base = (long long)blockIdx.x * kScanTile + (long long)t * kScanItems;
  uint32_t v[kScanItems], s = 0;
#pragma unroll
  for (int k = 0; k < kScanItems; ++k) {
    v[k] = (base + k < n) ? in[base + k] : 0u;
    s += v[k];
  }
  const uint32_t* const prev = sums ? sums : in;
  const int nprev = sums ? blockIdx.x : blockIdx.x * kScanTile;
  uint32_t b = 0, before;
#pragma unroll 8
  for (int i = t; i < nprev; i += kScanThreads) b += prev[i];
  block_exclusive_scan(b, wb, &before);
  uint32_t run = block_exclusive_scan(s, ws, nullptr) + before;
#pragma unroll
  for (int k = 0; k < kScanItems; ++k) {
    if (base + k < n) out[base + k] = run;
    run += v[k];
  }
}
static_assert(kScanThreads * kScanItems == kScanTile, "scan tile");

// ------------------------------------------------------------------ keys and digit counts
// CTA c of C owns the particles [chunk_lo, chunk_hi): whole tiles, the same in every kernel of a pass.
__device__ __forceinline__ void chunk_of(int64_t n, int64_t& lo, int64_t& hi) {
  const int64_t tiles = (n + kRadixTile - 1) / kRadixTile, per = (tiles + gridDim.x - 1) / gridDim.x * kRadixTile;
  lo = (int64_t)blockIdx.x * per;
  if (lo > n) lo = n;
  hi = lo + per < n ? lo + per : n;
}

// h[digit] += 1: neighbouring lanes often hold the same digit (nearly sorted particles), so
// the first lane of a run adds its length.  Lanes without a particle pass 0xffffffff.
__device__ __forceinline__ void count_digit(uint32_t d, uint32_t* h) {
  const int lane = threadIdx.x & 31;
  const uint32_t prev = __shfl_up_sync(0xffffffffu, d, 1);
  const bool head = lane == 0 || prev != d;
  const unsigned heads = __ballot_sync(0xffffffffu, head);
  if (head && d != 0xffffffffu) {
    const unsigned next = heads & ~((2u << lane) - 1u);  // heads above this lane (lane 31: none)
    atomicAdd(h + d, (uint32_t)((next ? __ffs(next) - 1 : 32) - lane));
  }
}

// Keys of the particles and the chunk's counts of the first digit, hist[d C + c].
template <int BITS>
__global__ void __launch_bounds__(kCountThreads) k_keys(const uint32_t* u, int64_t n, int shift, int ntl,
                                                        uint32_t* __restrict__ keys, uint32_t* __restrict__ hist) {
  pdl_begin();
  constexpr int DIG = 1 << BITS;
  __shared__ uint32_t h[DIG];
  for (int i = threadIdx.x; i < DIG; i += kCountThreads) h[i] = 0;
  __syncthreads();
  int64_t lo, hi;
  chunk_of(n, lo, hi);
  for (int64_t base = lo; base < hi; base += kCountThreads * kCountUnroll) {
    uint32_t ux[kCountUnroll], uy[kCountUnroll], uz[kCountUnroll];
#pragma unroll
    for (int k = 0; k < kCountUnroll; ++k) {
      const int64_t i = base + k * kCountThreads + threadIdx.x;
      if (i < hi) {
        ux[k] = u[i];
        uy[k] = u[n + i];
        uz[k] = u[2 * n + i];
      }
    }
#pragma unroll
    for (int k = 0; k < kCountUnroll; ++k) {
      const int64_t i = base + k * kCountThreads + threadIdx.x;
      uint32_t d = 0xffffffffu;
      if (i < hi) {
        const uint32_t key = tile_key(ux[k], uy[k], uz[k], shift, ntl);
        keys[i] = key;
        d = key & (DIG - 1);
      }
      count_digit(d, h);
    }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < DIG; i += kCountThreads) hist[(size_t)i * gridDim.x + blockIdx.x] = h[i];
}

// A digit's counts of existing keys: n of them, or (flags set) the movers of a re-sort.
template <int BITS>
__global__ void __launch_bounds__(kCountThreads) k_digits(const uint32_t* keys, int64_t n, int shift,
                                                          uint32_t* __restrict__ hist,
                                                          const uint32_t* flags,
                                                          const uint32_t* bstart3, long long nb1) {
  pdl_begin();
  constexpr int DIG = 1 << BITS;
  __shared__ uint32_t h[DIG];
  for (int i = threadIdx.x; i < DIG; i += kCountThreads) h[i] = 0;
  if (flags) n = movers_of(flags, bstart3, nb1, n);
  __syncthreads();
  int64_t lo, hi;
  chunk_of(n, lo, hi);
  for (int64_t base = lo; base < hi; base += kCountThreads * kCountUnroll) {
    uint32_t key[kCountUnroll];
#pragma unroll
    for (int k = 0; k < kCountUnroll; ++k) {
      const int64_t i = base + k * kCountThreads + threadIdx.x;
      key[k] = i < hi ? keys[i] : 0u;
    }
#pragma unroll
    for (int k = 0; k < kCountUnroll; ++k)
      count_digit(base + k * kCountThreads + threadIdx.x < hi ? (key[k] >> shift) & (DIG - 1) : 0xffffffffu, h);
  }
  __syncthreads();
  for (int i = threadIdx.x; i < DIG; i += kCountThreads) hist[(size_t)i * gridDim.x + blockIdx.x] = h[i];
}

// Exclusive scan of each digit's counts over the C chunks, in place; totals[d].  A warp a digit.
__global__ void __launch_bounds__(256) k_chunk_scan(uint32_t* __restrict__ hist, int C, int digits,
                                                    uint32_t* __restrict__ totals) {
  pdl_begin();
  const int d = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (d >= digits) return;
  uint32_t* const h = hist + (size_t)d * C;
  uint32_t run = 0;
  for (int c0 = 0; c0 < C; c0 += 128) {  // four words a lane
    uint32_t v[4], s = 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int c = c0 + lane * 4 + k;
      v[k] = c < C ? h[c] : 0u;
      s += v[k];
    }
    uint32_t x = s;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += y;
    }
    uint32_t at = run + x - s;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int c = c0 + lane * 4 + k;
      if (c < C) h[c] = at;
      at += v[k];
    }
    run += __shfl_sync(0xffffffffu, x, 31);
  }
  if (lane == 0) totals[d] = run;
}

// ------------------------------------------------------------------ radix scatter
// One stable pass over (key, value) pairs (vin null: the value is the index), see the top of
// the file: hist holds the chunks' exclusive counts per digit and totals every digit's count, or
// (RAW, few chunks: a launch costs more than the sums) the counts themselves.
template <int BITS, bool RAW>
__global__ void __launch_bounds__(kRadixThreads, 3) k_radix_scatter(
    const uint32_t* kin, const uint32_t* vin, int64_t n, int shift,
    const uint32_t* hist, const uint32_t* totals, uint32_t* __restrict__ kout,
    uint32_t* __restrict__ vout, const uint32_t* flags, const uint32_t* bstart3,
    long long nb1) {
  pdl_begin();
  constexpr int DIG = 1 << BITS, PER = DIG > kRadixThreads ? DIG / kRadixThreads : 1;
  constexpr uint32_t MASK = DIG - 1;
  constexpr int KPW = kRadixTile / kRadixWarps;  // keys per warp
  constexpr int RPW = KPW / 32;                  // rounds per warp
  extern __shared__ uint32_t stage_kv[];  // keys then values of the tile, in digit order
  uint32_t* const sk = stage_kv;
  uint32_t* const sv = stage_kv + kRadixTile;
  __shared__ uint32_t wcnt[kRadixWarps][DIG];  // per-warp digit counts, then staging offsets
  __shared__ uint32_t delta[DIG];              // global minus staging position of the tile's run of a digit
  __shared__ uint32_t ws[32];
  const int t = threadIdx.x, lane = t & 31, w = t >> 5;
  if (flags) n = movers_of(flags, bstart3, nb1, n);
  int64_t lo, hi;
  chunk_of(n, lo, hi);
  if (lo >= hi) return;
  const bool owner = t * PER < DIG;  // this thread's digits: t PER + q
  uint32_t next[PER];                // where the chunk's next key of a digit goes
  {
    uint32_t c[PER], sum = 0;
#pragma unroll
    for (int q = 0; q < PER; ++q) {
      c[q] = 0u;
      next[q] = 0u;
      if (owner) {
        const uint32_t* const h = hist + (size_t)(t * PER + q) * gridDim.x;
        if constexpr (RAW) {
#pragma unroll 8
          for (int k = 0; k < (int)gridDim.x; ++k) {
            const uint32_t v = h[k];
            c[q] += v;
            if (k < (int)blockIdx.x) next[q] += v;
          }
        } else {
          c[q] = totals[t * PER + q];
          next[q] = h[blockIdx.x];
        }
      }
      sum += c[q];
    }
    uint32_t ex = block_exclusive_scan(sum, ws, nullptr);
#pragma unroll
    for (int q = 0; q < PER; ++q) {
      next[q] += ex;
      ex += c[q];
    }
  }
  const unsigned lt = (1u << lane) - 1u;
  for (int64_t base = lo; base < hi; base += kRadixTile) {
    // 1. ranks inside the warp's digit runs
    uint32_t key[RPW], val[RPW], rk[RPW / 2];  // ranks are below 512: two to a word
#pragma unroll
    for (int r = 0; r < RPW; ++r) {
      const int64_t i = base + w * KPW + r * 32 + lane;
      key[r] = i < hi ? kin[i] : 0u;
      val[r] = i < hi ? (vin ? vin[i] : (uint32_t)i) : 0u;
    }
    __syncthreads();  // the previous tile's shared memory is read
    for (int i = t; i < kRadixWarps * DIG; i += kRadixThreads) (&wcnt[0][0])[i] = 0;
    __syncthreads();
#pragma unroll
    for (int r = 0; r < RPW; ++r) {
      const bool ok = base + w * KPW + r * 32 + lane < hi;
      const uint32_t d = (key[r] >> shift) & MASK;
      unsigned peers = __ballot_sync(0xffffffffu, ok);
#pragma unroll
      for (int b = 0; b < BITS; ++b) {
        const unsigned m = __ballot_sync(0xffffffffu, (d >> b) & 1u);
        peers &= ((d >> b) & 1u) ? m : ~m;
      }
      const uint32_t below = (uint32_t)__popc(peers & lt);
      const uint32_t c0 = ok ? wcnt[w][d] : 0u;  // every peer reads the count before this round
      if (r & 1) rk[r / 2] |= (c0 + below) << 16; else rk[r / 2] = c0 + below;
      __syncwarp();
      if (ok && below == 0) wcnt[w][d] = c0 + (uint32_t)__popc(peers);
      __syncwarp();
    }
    __syncthreads();
    // 2. digit totals -> tile-exclusive digit starts -> per-warp staging offsets
    {
      uint32_t c[PER], sum = 0;
#pragma unroll
      for (int q = 0; q < PER; ++q) {
        uint32_t tot = 0;
        if (owner) {
#pragma unroll
          for (int ww = 0; ww < kRadixWarps; ++ww) tot += wcnt[ww][t * PER + q];
        }
        c[q] = tot;
        sum += tot;
      }
      uint32_t ex = block_exclusive_scan(sum, ws, nullptr);
      if (owner) {
#pragma unroll
        for (int q = 0; q < PER; ++q) {
          const int d = t * PER + q;
          uint32_t run = ex;
#pragma unroll
          for (int ww = 0; ww < kRadixWarps; ++ww) {
            const uint32_t cw = wcnt[ww][d];
            wcnt[ww][d] = run;
            run += cw;
          }
          delta[d] = next[q] - ex;
          next[q] += c[q];
          ex += c[q];
        }
      }
    }
    __syncthreads();
    // 3. stage in digit order
#pragma unroll
    for (int r = 0; r < RPW; ++r) {
      if (base + w * KPW + r * 32 + lane < hi) {
        const uint32_t pos = wcnt[w][(key[r] >> shift) & MASK] + ((r & 1) ? rk[r / 2] >> 16 : rk[r / 2] & 0xffffu);
        sk[pos] = key[r];
        sv[pos] = val[r];
      }
    }
    __syncthreads();
    // 4. coalesced runs to the digit's global position
    const int cnt = (int)((hi - base) < kRadixTile ? (hi - base) : kRadixTile);
    for (int j = t; j < cnt; j += kRadixThreads) {
      const uint32_t k = sk[j];
      const uint32_t dst = delta[(k >> shift) & MASK] + (uint32_t)j;
      kout[dst] = k;
      vout[dst] = sv[j];
    }
  }
}

// ------------------------------------------------------------------ gather
// A particle's words in registers: every load is issued before the first store (the compiler keeps
// loads of plain const pointers behind earlier stores).
struct Particle {
  uint32_t u[3], id;
  float p[3];
};
__device__ __forceinline__ Particle load_particle(const uint32_t* u, const float* p, const uint32_t* id, int64_t n,
                                                  uint32_t i) {
  Particle q;
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    q.u[d] = u[d * n + i];
    q.p[d] = p ? p[d * n + i] : 0.0f;
  }
  q.id = id ? id[i] : i;
  return q;
}
__device__ __forceinline__ void store_particle(const Particle& q, int64_t n, int64_t k, uint32_t* __restrict__ us,
                                               float* __restrict__ ps, uint32_t* __restrict__ ids) {
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    us[d * n + k] = q.u[d];
    if (ps) ps[d * n + k] = q.p[d];
  }
  ids[k] = q.id;
}

// Records of the particles [i0, n) for the gather, in the sort's free buffers: (u, id), or
// (u, id, p) when there are momenta.  Neutrinos (the input's tail in canonical order) stream
// freely, so their order says nothing about their place: gathered array by array, each costs four
// or seven scattered sectors, from a record one or two.  Written through shared memory, whole lines.
// A state that a step has left is in tile order, and its tail gathers whole lines already: the
// records would only add their own traffic.  So every CTA looks at the same 256 places of the
// permutation, and none is packed (flag 0) where the input's neighbours mostly stay neighbours.
constexpr int kPackThreads = 256;
constexpr int kPackCtas = 8 * 152;
__global__ void __launch_bounds__(kPackThreads) k_pack(const uint32_t* u, const float* p, const uint32_t* id, int64_t n,
                                                       int64_t i0, const uint32_t* perm, uint32_t* __restrict__ rec,
                                                       uint32_t* __restrict__ flag) {
  pdl_begin();
  __shared__ uint32_t sh[7 * kPackThreads], seen[kPackThreads / 32];
  const int W = p ? 7 : 4, t = threadIdx.x;
  const int64_t k = t * (n - 1) / kPackThreads;
  const uint32_t at = perm[k], next = perm[k + 1];
  // samples in the tail, and (from bit 16) those whose successor comes next
  uint32_t c = (int64_t)at < i0 ? 0u : (next == at + 1 ? 0x10001u : 1u);
  c = __reduce_add_sync(0xffffffffu, c);
  if ((t & 31) == 0) seen[t >> 5] = c;
  __syncthreads();
  c = 0;
#pragma unroll
  for (int w = 0; w < kPackThreads / 32; ++w) c += seen[w];
  const bool pack = 3 * (c & 0xffffu) > 4 * (c >> 16);  // runs shorter than four on average
  if (blockIdx.x == 0 && t == 0) *flag = pack ? 1u : 0u;
  if (!pack) return;
  for (int64_t first = i0 + (int64_t)blockIdx.x * kPackThreads; first < n; first += (int64_t)gridDim.x * kPackThreads) {
    const int64_t i = first + t;
    if (i < n) {
      sh[t * W] = u[i];
      sh[t * W + 1] = u[n + i];
      sh[t * W + 2] = u[2 * n + i];
      sh[t * W + 3] = id ? id[i] : (uint32_t)i;
      if (p) {
#pragma unroll
        for (int d = 0; d < 3; ++d) sh[t * W + 4 + d] = __float_as_uint(p[d * n + i]);
      }
    }
    __syncthreads();
    const int words = (int)((n - first < kPackThreads ? n - first : kPackThreads) * W);
    uint32_t* const out = rec + (size_t)(first - i0) * W;
    for (int q = t; q < words; q += kPackThreads) out[q] = sh[q];
    __syncthreads();
  }
}

// The first nbb CTAs find the bucket starts in the sorted keys (bstart[k] = number of keys
// below k; nb1 of them), the others gather the particles (from index i0 on from rec if there is a
// flag and it is set).
__global__ void k_gather(const uint32_t* u, const float* p,
                         const uint32_t* id, int64_t n,
                         const uint32_t* perm, uint32_t* __restrict__ us,
                         float* __restrict__ ps, uint32_t* __restrict__ ids, const uint32_t* skeys,
                         long long nb1, unsigned nbb, uint32_t* __restrict__ bstart,
                         const uint32_t* rec, int64_t i0, const uint32_t* flag) {
  pdl_begin();
  if (blockIdx.x < nbb) {
    const long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= nb1) return;
    uint32_t lo = 0, len = (uint32_t)n;
    while (len > 0) {
      const uint32_t h = len >> 1;
      if ((long long)skeys[lo + h] < k) {
        lo += h + 1;
        len -= h + 1;
      } else {
        len = h;
      }
    }
    bstart[k] = lo;
    return;
  }
  int64_t k = (int64_t)(blockIdx.x - nbb) * blockDim.x + threadIdx.x;
  if (k >= n) return;
  const uint32_t i = perm[k];
  if (flag && (int64_t)i >= i0 && *flag) {
    const uint32_t* const r = rec + (size_t)(i - i0) * (p ? 7 : 4);
    Particle q = {{r[0], r[1], r[2]}, r[3], {0.f, 0.f, 0.f}};
    if (p) {
#pragma unroll
      for (int d = 0; d < 3; ++d) q.p[d] = __uint_as_float(r[4 + d]);
    }
    store_particle(q, n, k, us, p ? ps : nullptr, ids);
  } else {
    store_particle(load_particle(u, p, id, n, i), n, k, us, p ? ps : nullptr, ids);
  }
}

// ------------------------------------------------------------------ near-sorted re-sort
// One CTA per old tile O: walks O's range [bprev[8 O], bprev[8 O + 8]) in chunks of the
// block size, in index order.  With stage, a mover's position, momentum and id also go to a
// 32-byte record at its list position (the placement then reads one sector a mover
// instead of seven scattered words), and mv holds that position.  A block scan of the mover flags gives every particle the
// number of movers of its own old key before it (mrank); a stayer goes to
// bstart[B] + low[B] + (i - bprev[B]) - mrank, a mover's (new key, index) to its old
// key's slot of the mover list, mstart3[ko] - base3 + mrank (movers in index order).  With
// flag bit 1 every particle is a mover at its own index.  stage_room: the movers' records
// that the staging area holds (more movers: none is staged).
template <int NT>
__global__ void __launch_bounds__(NT) k_resort_old_tiles(
    const uint32_t* u, const float* p, const uint32_t* id, int64_t n,
    const uint32_t* keys, const uint32_t* bprev, const uint32_t* bstart3,
    long long nb1, const uint32_t* low, uint32_t* __restrict__ us, float* __restrict__ ps,
    uint32_t* __restrict__ ids, uint32_t* __restrict__ mk, uint32_t* __restrict__ mv,
    const uint32_t* flags, int* __restrict__ err, uint4* __restrict__ stage, int64_t stage_room) {
  pdl_begin();
  constexpr int W = NT / 32;
  __shared__ uint32_t cls_lo[9];   // bprev[8 O + c]
  __shared__ uint32_t cls_m0[8];   // movers of the tile before class c's first particle
  __shared__ uint32_t wsum[W];
  const int t = threadIdx.x, lane = t & 31, w = t >> 5;
  const uint32_t O = blockIdx.x;
  if (*flags & 1u) {
    for (int64_t i = (int64_t)O * NT + t; i < n; i += (int64_t)gridDim.x * NT) {
      mk[i] = keys[i];
      mv[i] = (uint32_t)i;
    }
    return;
  }
  const int64_t nm = movers_of(flags, bstart3, nb1, n);
  if (nm > stage_room) stage = nullptr;
  // (bprev may be of more particles: a captured step replayed after another call has sorted into
  // its array, the state's n being the first of those in order)
  if (t < 9) cls_lo[t] = min(bprev[8 * O + t], (uint32_t)n);
  __syncthreads();
  const uint32_t lo = cls_lo[0], hi = cls_lo[8];
  if (lo == hi) return;
  const uint32_t base3 = bstart3[2 * nb1];  // n + all stayers: offset of the third scan
  const unsigned lt = (1u << lane) - 1u;
  uint32_t run = 0;  // movers of the tile before this chunk
  for (uint32_t chunk = lo; chunk < hi; chunk += NT) {
    const uint32_t i = chunk + t;
    const bool ok = i < hi;
    uint32_t kn = 0, c = 0;
    uint32_t pu[3] = {0u, 0u, 0u}, pid = 0u;
    float pp[3] = {0.f, 0.f, 0.f};
    if (ok) {  // the particle's data is loaded before the block scan, not after it
      kn = keys[i];
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        pu[d] = u[d * n + i];
        if (p) pp[d] = p[d * n + i];
      }
      pid = id ? id[i] : i;
#pragma unroll
      for (int k = 1; k < 8; ++k) c += i >= cls_lo[k] ? 1u : 0u;
    }
    const uint32_t ko = 8 * O + c;
    const bool mover = ok && kn != ko;
    // where the particle's run starts: B's stayers, or old key ko's slot of the mover list
    const uint32_t run0 = !ok ? 0u : (mover ? bstart3[2 * nb1 + ko] - base3 : bstart3[ko] + low[ko]);
    const unsigned bal = __ballot_sync(0xffffffffu, mover);
    if (lane == 0) wsum[w] = (uint32_t)__popc(bal);
    __syncthreads();
    uint32_t before = run, total = 0;
#pragma unroll
    for (int ww = 0; ww < W; ++ww) {
      before += ww < w ? wsum[ww] : 0u;
      total += wsum[ww];
    }
    const uint32_t mex = before + (uint32_t)__popc(bal & lt);  // movers of the tile before i
    if (ok && i == cls_lo[c]) cls_m0[c] = mex;                   // class c starts here
    __syncthreads();
    if (ok) {
      const uint32_t mrank = mex - cls_m0[c];
      if (!mover) {
        const uint32_t dst = run0 + (i - cls_lo[c]) - mrank;
        if (dst < (uint64_t)n) {
#pragma unroll
          for (int d = 0; d < 3; ++d) {
            us[d * n + dst] = pu[d];
            if (p) ps[d * n + dst] = pp[d];
          }
          ids[dst] = pid;
        } else {
          atomicOr(err, 1);  // inconsistent counts: never written out of range
        }
      } else {
        const uint32_t pos = run0 + mrank;
        if (pos < (uint64_t)nm) {
          mk[pos] = kn;
          if (stage) {  // the mover's 28 bytes as one 32-byte record at its list position
            mv[pos] = pos;
            stage[2 * (size_t)pos] = make_uint4(pu[0], pu[1], pu[2], pid);
            stage[2 * (size_t)pos + 1] = make_uint4(__float_as_uint(pp[0]), __float_as_uint(pp[1]),
                                                    __float_as_uint(pp[2]), 0u);
          } else {
            mv[pos] = i;
          }
        } else {
          atomicOr(err, 1);
        }
      }
    }
    run += total;
    __syncthreads();  // wsum is rewritten by the next chunk
  }
}

// Mover r of new key B in the movers' stable order: destination bstart[B] + r, behind B's
// stayers when it came from a higher key (r >= low[B]).  The movers of keys below B
// number bstart[B] - sstart[B], sstart = the stayers' scan (bstart3's second third
// minus n).
__device__ __forceinline__ void place_mover(int64_t j, bool all, const uint32_t* mk,
                                            const uint32_t* mv, int64_t nm,
                                            const uint32_t* u, const float* p,
                                            const uint32_t* id, int64_t n,
                                            const uint32_t* bstart3, long long nb1, long long nbuckets,
                                            const uint32_t* low, uint32_t* __restrict__ us,
                                            float* __restrict__ ps, uint32_t* __restrict__ ids,
                                            int* __restrict__ err, const uint4* stage) {
  const uint32_t B = mk[j], i = mv[j];
  if (B >= (uint64_t)nbuckets || i >= (uint64_t)(stage ? nm : n)) {
    atomicOr(err, 1);
    return;
  }
  int64_t dst = j;
  if (!all) {
    const uint32_t s0 = bstart3[nb1 + B], s1 = bstart3[nb1 + B + 1], b0 = bstart3[B], lo = low[B];
    const uint32_t r = (uint32_t)j - (b0 - (s0 - (uint32_t)n));
    dst = b0 + r + (r >= lo ? s1 - s0 : 0u);
    if (dst >= n) {
      atomicOr(err, 1);
      return;
    }
  }
  if (stage) {  // one 32-byte record (i: its position in the mover list)
    const uint4 a = stage[2 * (size_t)i], b = stage[2 * (size_t)i + 1];
    const Particle q = {{a.x, a.y, a.z}, a.w, {__uint_as_float(b.x), __uint_as_float(b.y), __uint_as_float(b.z)}};
    store_particle(q, n, dst, us, p ? ps : nullptr, ids);
  } else {
    // scattered words, one array after the other: all seven loads at once spread wider than the
    // caches hold (35 M particles at 256^3, two steps: 491 us, 692 with all loads first)
#pragma unroll
    for (int d = 0; d < 3; ++d) us[d * n + dst] = u[d * n + i];
    if (p) {
#pragma unroll
      for (int d = 0; d < 3; ++d) ps[d * n + dst] = p[d * n + i];
    }
    ids[dst] = id ? id[i] : i;
  }
}

// With flag bit 1 the movers are all particles: mover j goes to slot j.  Counts the re-sort in
// stats (near-sorted, from scratch, movers of the last near-sorted one).
__global__ void k_place_movers(const uint32_t* mk, const uint32_t* mv,
                               const uint32_t* u, const float* p,
                               const uint32_t* id, int64_t n, const uint32_t* bstart3,
                               long long nb1, long long nbuckets, const uint32_t* low,
                               uint32_t* __restrict__ us, float* __restrict__ ps, uint32_t* __restrict__ ids,
                               const uint32_t* flags, int* __restrict__ err,
                               const uint4* stage, int64_t stage_room, long long* __restrict__ stats) {
  pdl_begin();
  const bool all = (*flags & 1u) != 0u;
  const int64_t nm = movers_of(flags, bstart3, nb1, n, err);
  if (all || nm > stage_room) stage = nullptr;
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    stats[all ? 1 : 0] += 1;
    if (!all) stats[2] = nm;
  }
  for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < nm; j += (int64_t)gridDim.x * blockDim.x)
    place_mover(j, all, mk, mv, nm, u, p, id, n, bstart3, nb1, nbuckets, low, us, ps, ids, err, stage);
}

// the chunks of a sort of up to n keys: as many as tiles, at most kMaxChunks
unsigned chunks_of(int64_t n) {
  return (unsigned)std::min<int64_t>(kMaxChunks, std::max<int64_t>(1, (n + kRadixTile - 1) / kRadixTile));
}

// up to 32 chunks (131 k keys) the scatter adds up the counts itself
bool raw_counts(int64_t n) { return chunks_of(n) <= 32; }

template <int BITS>
void launch_scatter(pm_ctx* c, const uint32_t* kin, const uint32_t* vin, int64_t n, int shift, uint32_t* kout,
                    uint32_t* vout, const uint32_t* flags, cudaStream_t s) {
  const size_t dyn = 2 * kRadixTile * sizeof(uint32_t);
  const bool raw = raw_counts(n);
  auto kern = raw ? k_radix_scatter<BITS, true> : k_radix_scatter<BITS, false>;
  static DeviceOnce once[2];
  allow_smem(once[raw], (const void*)kern, dyn);
  pdl_launch(kern, chunks_of(n), kRadixThreads, dyn, s, kin, vin, n, shift, c->hist, c->digit_totals, kout, vout, flags,
                                                c->bstart, c->nbuckets + 1);
}

// LSD radix passes over n (key, value) pairs in buffer pair 0 (values absent: the incoming
// index), pair 1 the other buffers; flags: only the movers of a re-sort.  counted: hist holds
// the first digit's chunk counts already.  Returns which pair holds the result.
template <int BITS>
int passes_of(pm_ctx* c, uint32_t* const kb[2], uint32_t* const vb[2], bool index_vals, bool counted, int64_t n,
              const uint32_t* flags, cudaStream_t s) {
  const unsigned C = chunks_of(n);
  int cur = 0;
  for (int pass = 0; pass < c->radix_passes; ++pass) {
    const int shift = BITS * pass;
    if (!counted || pass > 0) {
      LaunchScope L(c, s, K_RADIX_HIST);
      pdl_launch(k_digits<BITS>, C, kCountThreads, 0, s, kb[cur], n, shift, c->hist, flags, c->bstart, c->nbuckets + 1);
    }
    if (!raw_counts(n)) {
      LaunchScope L(c, s, K_SCAN);
      pdl_launch(k_chunk_scan, (1 << BITS) / 8, 256, 0, s, c->hist, (int)C, 1 << BITS, c->digit_totals);
    }
    LaunchScope L(c, s, K_RADIX_SCATTER);
    launch_scatter<BITS>(c, kb[cur], (pass == 0 && index_vals) ? nullptr : vb[cur], n, shift, kb[cur ^ 1], vb[cur ^ 1],
                         flags, s);
    cur ^= 1;
  }
  return cur;
}

int radix_passes(pm_ctx* c, uint32_t* const kb[2], uint32_t* const vb[2], bool index_vals, bool counted, int64_t n,
                 const uint32_t* flags, cudaStream_t s) {
  if (c->radix_bits == 9) return passes_of<9>(c, kb, vb, index_vals, counted, n, flags, s);
  if (c->radix_bits == 8) return passes_of<8>(c, kb, vb, index_vals, counted, n, flags, s);
  return passes_of<7>(c, kb, vb, index_vals, counted, n, flags, s);
}

void sort_keys0(pm_ctx* c, bool counted, int64_t n, cudaStream_t s) {  // keys[0] -> keys[0], vals[0]
  uint32_t* const kb[2] = {c->keys[0], c->keys[1]};
  uint32_t* const vb[2] = {c->vals[0], c->vals[1]};
  if (radix_passes(c, kb, vb, true, counted, n, nullptr, s) != 0) {  // keep the result in keys[0] / vals[0]
    std::swap(c->keys[0], c->keys[1]);
    std::swap(c->vals[0], c->vals[1]);
  }
}

}  // namespace

int sort_by_keys(pm_ctx* c, int64_t n, cudaStream_t s) {
  if (n > 0) sort_keys0(c, false, n, s);
  return PM_OK;
}

int sort_particles(pm_ctx* c, const uint32_t* u, int64_t n, cudaStream_t s) {
  if (n == 0) {  // no gather will run: every bucket is empty
    PM_CUDA_TRY(cudaMemsetAsync(c->bstart, 0, sizeof(uint32_t) * (c->nbuckets + 1), s));
    return PM_OK;
  }
  {
    LaunchScope L(c, s, K_KEYS);
    const int shift = 32 - c->g.logn;
    auto kern = c->radix_bits == 9 ? k_keys<9> : (c->radix_bits == 8 ? k_keys<8> : k_keys<7>);
    pdl_launch(kern, chunks_of(n), kCountThreads, 0, s, u, n, shift, c->ntl, c->keys[0], c->hist);
  }
  sort_keys0(c, true, n, s);
  return PM_OK;
}

void gather_sorted(pm_ctx* c, const uint32_t* u, const float* p, const uint32_t* id, int64_t n,
                   const uint32_t* perm, cudaStream_t s) {
  if (n == 0) return;
  // The neutrinos through records where scattered sectors are what the gather costs: from 2^21 of
  // them on with momenta, 2^22 without (fewer stay in the second-level cache), if they fit the free
  // half of the sort's buffers (16 bytes a particle of the capacity); the kernel leaves out those in
  // tile order.  us without / with records, 4 and 7 words a particle: 0.9 M of 17.7 M neutrinos
  // 144 / 159 and 230 / 242, 2.3 M of 19 M 183 / 184 and 318 / 285, 18 M of 35 M 1005 / 525 and
  // 2073 / 818; the last in tile order 235 / 340 and 324 / 475 if they were packed.
  const int64_t i0 = std::min<int64_t>(n, c->mt.n_cdm);
  uint32_t* const rec = c->keys[0] == c->sortbuf ? c->rs_k2 : c->sortbuf;
  const int64_t rec_bytes = (n - i0) * (p ? 28 : 16);
  const uint32_t* flag = nullptr;
  if (n - i0 >= (p ? 1 << 21 : 1 << 22) && rec_bytes <= 16 * std::max<int64_t>(c->n_max, 1)) {
    LaunchScope L(c, s, K_GATHER);
    const unsigned grid = (unsigned)std::min<int64_t>(kPackCtas, (n - i0 + kPackThreads - 1) / kPackThreads);
    pdl_launch(k_pack, grid, kPackThreads, 0, s, u, p, id, n, i0, perm, rec, c->pack_flag);
    flag = c->pack_flag;
  }
  LaunchScope L(c, s, K_GATHER);
  const unsigned nbb = (unsigned)((c->nbuckets + 1 + 255) / 256);
  pdl_launch(k_gather, nbb + (unsigned)((n + 255) / 256), 256, 0, s, u, p, id, n, perm, c->us, c->ps, c->ids, c->keys[0],
                                                            c->nbuckets + 1, nbb, c->bstart, rec, i0, flag);
}

int clear_resort(pm_ctx* c, cudaStream_t s) {
  PM_CUDA_TRY(cudaMemsetAsync(c->counts, 0, sizeof(uint32_t) * c->clear_words, s));
  return PM_OK;
}

int resort_near_sorted(pm_ctx* c, const uint32_t* u, const float* p, const uint32_t* id, int64_t n,
                       cudaStream_t s) {
  const long long nb1 = c->nbuckets + 1;
  {  // bucket starts, stayers' and old keys' movers' starts in one scan
    const unsigned tiles = (unsigned)((3 * nb1 + kScanTile - 1) / kScanTile);
    const bool few = tiles <= kScanFew;
    if (!few) {
      LaunchScope L(c, s, K_SCAN);
      pdl_launch(k_scan_sums, tiles, kScanThreads, 0, s, c->counts, 3 * nb1, c->scan_sums);
    }
    LaunchScope L(c, s, K_SCAN);
    pdl_launch(k_scan, tiles, kScanThreads, 0, s, c->counts, 3 * nb1, few ? nullptr : c->scan_sums, c->bstart);
  }
  // the movers' records go to the second mesh, free during a step, when they fit (32 bytes a
  // mover: up to 2^30 movers at 2048^3); else the placement gathers from the state itself
  uint4* const stage = reinterpret_cast<uint4*>(c->meshB);
  const int64_t room = (int64_t)(c->g.elems() * sizeof(float2) / 32);
  {
    LaunchScope L(c, s, K_RESORT_PLACE);
    const int threads = tile_threads(c);
    auto kern = threads == 1024 ? k_resort_old_tiles<1024> : (threads == 512 ? k_resort_old_tiles<512> : k_resort_old_tiles<256>);
    pdl_launch(kern, (unsigned)((long long)c->nt * c->nt * c->nt), threads, 0, s, 
        u, p, id, n, c->keys[0], c->bprev, c->bstart, nb1, c->rs_low, c->us, c->ps, c->ids, c->keys[1], c->vals[1],
        c->rs_dev, c->err_dev, stage, room);
  }
  uint32_t* const kb[2] = {c->keys[1], c->rs_k2};
  uint32_t* const vb[2] = {c->vals[1], c->rs_v2};
  const int r = radix_passes(c, kb, vb, false, false, n, c->rs_dev, s);
  LaunchScope L(c, s, K_RESORT_MISC);
  if (c->place_ctas == 0) {  // grid-stride: the CTAs that fill the GPU once
    int per_sm = 0, sms = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_place_movers, 256, 0);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, c->device);
    c->place_ctas = (unsigned)(std::max(per_sm, 1) * std::max(sms, 1));
  }
  pdl_launch(k_place_movers, (unsigned)std::min<int64_t>(c->place_ctas, (n + 255) / 256), 256, 0, s, 
      kb[r], vb[r], u, p, id, n, c->bstart, nb1, c->nbuckets, c->rs_low, c->us, c->ps, c->ids, c->rs_dev, c->err_dev,
      stage, room, c->rs_stats);
  return PM_OK;
}

}  // namespace pmnu
