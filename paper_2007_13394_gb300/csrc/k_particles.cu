// Particle <-> mesh kernels: deterministic tile paint, CIC readout fused with the
// kick (of force meshes, or of the potential with the 4-point gradient applied in
// shared memory), the first kick fused with the drift and the next sort keys.
//
// Paint (CIC of rho / rho_bar): one CTA per 16^3 tile.  The tile's own particles
// are the bucket range [bstart[8 t], bstart[8 t + 8]); a particle on the tile's
// high face layer (class bits) also reaches the neighbouring tile, which reads
// exactly those classes of its seven low-side neighbours.  Each (particle,
// corner) pair is therefore counted by the one CTA that owns the corner cell.
// Contributions are accumulated in shared memory as fixed-point integers: integer
// addition is associative, so the result does not depend on thread scheduling, and
// no float atomics are used.  Mass paints use 2^-24 resolution: each contribution
// q < 2^31 goes to a 32-bit accumulator with one atomic add, whose returned old value
// shows when the sum wrapped past 2^32, and then a second word counts the carry
// (value = carry 2^32 + low word: exact, whatever the order).  A wrap needs a cell of
// 256 mean cell masses, so nearly every corner costs one 32-bit shared atomic (those
// run ~4x faster than 64-bit ones, and the 32-bit conversions of the write-out avoid
// the narrow FP64 pipe that 64-bit float <-> integer conversions use).  Masses of 128
// or more and the signed weights of the adjoint are 64-bit integers in the same two words
// (resolution 2^-24 for masses, so both forms give the same bits; 2^-32 for weights): the
// low word is added with a 32-bit atomic and the high word only when it changes, which for
// weights is when a cell's sum crosses a multiple of 2^32.
#include <cuda_runtime.h>

#include <algorithm>

#include "pm_internal.cuh"

namespace pmnu {

namespace {

constexpr int kPaintThreads = 256;
constexpr float kFixW = 4294967296.0f;              // 2^32: signed weights
constexpr float kUnfixW = 2.3283064365386963e-10f;  // 2^-32
constexpr float kFixM = 16777216.0f;                // 2^24: masses
constexpr float kUnfixM = 5.9604644775390625e-08f;  // 2^-24

// The 14 bucket runs a tile reads, as (neighbour offset o, first class, end class):
// its own tile (all classes), then for each low-side neighbour o the classes that
// contain every bit of o, merged where they are contiguous.
__constant__ int8_t c_runs[14][3] = {{0, 0, 8}, {4, 4, 8}, {2, 2, 4}, {2, 6, 8}, {1, 1, 2},
                                     {1, 3, 4}, {1, 5, 6}, {1, 7, 8}, {6, 6, 8}, {5, 5, 6},
                                     {5, 7, 8}, {3, 3, 4}, {3, 7, 8}, {7, 7, 8}};

// Shared accumulator layout: cell (x, y, z) of the tile at x * kSx + y * kSy + z.  With
// kSy = 18 and kSx = 292 (4 and 2 modulo 16) the 8 CIC corners of one particle land in
// 8 distinct 8-byte bank pairs.
constexpr int kSy = 18, kSx = 292;
constexpr int kAccWords = kTile * kSx;
// fast paint: wrap bitmap words, event list capacity, and the whole shared area in words
// (low words, bitmap, event count, 16-bit events, rounded up to whole 16-byte groups)
constexpr int kWrapBits = (kAccWords + 31) / 32;
constexpr unsigned int kWraps = 1024;
constexpr int kFastWords = ((kAccWords + kWrapBits + 1 + kWraps / 2) + 3) / 4 * 4;

// Records that the fast paint's low word ad wrapped: its bit in the bitmap and an event in
// the list (layout of paint_tile); false when the list is full.  Out of line: rarely taken,
// and it keeps the paint's inner loop at fewer registers.
__device__ __noinline__ bool record_wrap(unsigned int* accw, unsigned int ad) {
  atomicOr(accw + kAccWords + (ad >> 5), 1u << (ad & 31));
  const unsigned int e = atomicAdd(accw + kAccWords + kWrapBits, 1u);
  if (e >= kWraps) return false;
  reinterpret_cast<unsigned short*>(accw + kAccWords + kWrapBits + 1)[e] = (unsigned short)ad;
  return true;
}

// __float2ll_rn without the narrow FP64 pipe: below 2^31 the 32-bit conversion (same rounding),
// above it the value is an integer already (24-bit mantissa), so shift the mantissa.
__device__ __forceinline__ long long fixed64(float x) {
  if (fabsf(x) < 2147483648.0f) return (long long)__float2int_rn(x);
  if (!(fabsf(x) < 9.0e18f)) return __float2ll_rn(x);  // saturation, NaN
  const uint32_t bits = __float_as_uint(x);
  const long long m = (long long)(unsigned long long)((bits & 0x7fffffu) | 0x800000u) << (((bits >> 23) & 255u) - 150u);
  return (bits >> 31) ? -m : m;
}

// 64-bit sum in two 32-bit words: lo += low word of q, hi += high word + carry (only if not 0)
__device__ __forceinline__ void add64(unsigned int* lo, unsigned int* hi, long long q) {
  const unsigned int ql = (unsigned int)q, old = atomicAdd(lo, ql);
  const unsigned int h = (unsigned int)(q >> 32) + (old + ql < old ? 1u : 0u);
  if (h) atomicAdd(hi, h);
}

// __ll2float_rn of the two-word sum; the usual cases (|value| < 2^32) by 32-bit conversions
__device__ __forceinline__ float float64w(unsigned int hi, unsigned int lo) {
  if (hi == 0u) return __uint2float_rn(lo);
  if (hi == 0xffffffffu && lo != 0u) return -__uint2float_rn(0u - lo);
  return __ll2float_rn((long long)(((unsigned long long)hi << 32) | (unsigned long long)lo));
}

// A tile whose list of wraps overflowed, painted again by its CTA: half of its x planes at a
// time in two words a cell, which fit where the low words of the whole tile were.  Out of line:
// rare, and the main form keeps its 32 registers.  Every thread of the CTA calls it.
template <int NT>
__device__ __noinline__ void paint_halves(uint32_t tile, unsigned int* __restrict__ accw,
                                          const uint32_t* __restrict__ run_lo, const uint32_t* __restrict__ run_pre,
                                          const uint32_t* us, const uint32_t* ids, int64_t n,
                                          float* __restrict__ mesh, const MassTable& mt, int species, int nm, int shift,
                                          int ntl, int row_pitch) {
  constexpr int HX = kTile / 2, WORDS = HX * kSx;
  const int t = threadIdx.x, nt = 1 << ntl;
  const int ox = (int)(tile >> (2 * ntl)) * kTile, oy = (int)((tile >> ntl) & (nt - 1)) * kTile,
            oz = (int)(tile & (nt - 1)) * kTile;
  const float fscale = 1.0f / (float)(1u << shift);
  const uint32_t fmask = (1u << shift) - 1u, total = run_pre[14];
  for (int x0 = 0; x0 < kTile; x0 += HX) {
    __syncthreads();  // the accumulators are free
    for (int i = t; i < 2 * WORDS; i += NT) accw[i] = 0;
    __syncthreads();
    int r = 0;
    for (uint32_t v = t; v < total; v += NT) {
      while (v >= run_pre[r + 1]) ++r;
      const uint32_t k = run_lo[r] + (v - run_pre[r]);
      const uint32_t q[3] = {us[k], us[n + k], us[2 * n + k]};
      bool bad = false;  // reported by the first pass
      const float m = id_mass(mt, ids[k], species, &bad);
      if (m == 0.0f) continue;
      int l[3] = {(int)(q[0] >> shift) - ox, (int)(q[1] >> shift) - oy, (int)(q[2] >> shift) - oz};
#pragma unroll
      for (int d = 0; d < 3; ++d) {  // periodic wrap relative to the tile origin
        if (l[d] > nm / 2) l[d] -= nm;
        if (l[d] < -nm / 2) l[d] += nm;
      }
      const float fx = (float)(q[0] & fmask) * fscale, fy = (float)(q[1] & fmask) * fscale,
                  fz = (float)(q[2] & fmask) * fscale;
      for (int corner = 0; corner < 8; ++corner) {
        const int bx = corner >> 2, by = (corner >> 1) & 1, bz = corner & 1;
        const int x = l[0] + bx - x0, y = l[1] + by, z = l[2] + bz;
        if ((unsigned)x >= (unsigned)HX || (unsigned)y >= (unsigned)kTile || (unsigned)z >= (unsigned)kTile) continue;
        const float wc = (bx ? fx : 1.0f - fx) * (by ? fy : 1.0f - fy) * (bz ? fz : 1.0f - fz);
        const unsigned int qv = __float2uint_rn(wc * m * kFixM);  // < 2^31: masses below 128
        unsigned int* const lo = accw + x * kSx + y * kSy + z;
        const unsigned int old = atomicAdd(lo, qv);
        if (old + qv < old) atomicAdd(lo + WORDS, 1u);
      }
    }
    __syncthreads();
    for (int q = t; q < HX * kTile * kTile; q += NT) {
      const int x = q / (kTile * kTile), y = (q / kTile) % kTile, z = q % kTile;
      const int a = x * kSx + y * kSy + z;
      mesh[((size_t)(ox + x0 + x) * nm + (oy + y)) * (size_t)row_pitch + oz + z] = float64w(accw[WORDS + a], accw[a]) * kUnfixM;
    }
  }
}

// Paint of one tile.  FAST: 32-bit low words only (half the shared memory of the two-word form:
// zeroed, and read at the write-out, once per cell).  A low word that wraps past 2^32 (the
// cell passes another 256 mean cell masses) is recorded as an event -- the cell's bit in a
// bitmap, its index in a list of up to kWraps events -- and at the write-out a cell whose
// bit is set counts its events in the list: value = events 2^32 + low word.  A tile with
// more events than the list holds is painted again (paint_halves).  Every form sums the same
// exact integers, so all give the same floats.  Else two words a cell and NW = 0 (masses), or NW = 1 or 3 signed
// weights a particle (wts[j n + k]), weight j painted onto mesh j (mesh, mesh1, mesh2).
template <bool FAST, int NW, int NT>
__device__ __forceinline__ void paint_tile(
    uint32_t tile, unsigned int* __restrict__ accw, uint32_t* __restrict__ run_lo, uint32_t* __restrict__ run_pre,
    const uint32_t* us, const uint32_t* ids, int64_t n,
    const uint32_t* bstart, float* __restrict__ mesh, const MassTable& mt, int species, int nm,
    int shift, int ntl, int row_pitch, int* __restrict__ err, const float* wts,
    float* __restrict__ mesh1 = nullptr, float* __restrict__ mesh2 = nullptr) {
  constexpr int NA = NW > 1 ? NW : 1;  // meshes painted
  // FAST: low words, then the wrap bitmap, the event count and the event list.  Else per
  // mesh the low words, then the high words.
  unsigned int* const acc_lo = accw;
  volatile unsigned int* const wbits = accw + kAccWords;          // FAST: kWrapBits words
  unsigned int* const wcount = accw + kAccWords + kWrapBits;       // FAST: one word
  volatile unsigned short* const wlist = reinterpret_cast<unsigned short*>(accw + kAccWords + kWrapBits + 1);
  const int t = threadIdx.x;
  if constexpr (FAST) {
    for (int i = t; i < (kAccWords + kWrapBits + 1) / 4 + 1; i += NT)
      reinterpret_cast<uint4*>(accw)[i] = make_uint4(0, 0, 0, 0);
  } else {
    static_assert(kAccWords % 2 == 0, "whole 16-byte groups");
    for (int i = t; i < NA * kAccWords / 2; i += NT) reinterpret_cast<uint4*>(accw)[i] = make_uint4(0, 0, 0, 0);
  }
  const int nt = 1 << ntl;
  const int tx = tile >> (2 * ntl), ty = (tile >> ntl) & (nt - 1), tz = tile & (nt - 1);
  if (t < 32) {  // one warp resolves the 14 runs and their prefix
    uint32_t lo = 0, len = 0;
    if (t < 14) {
      const int o = c_runs[t][0];
      const int ox = (o >> 2) & 1, oy = (o >> 1) & 1, oz = o & 1;
      const uint32_t nb = ((uint32_t)((tx - ox) & (nt - 1)) << (2 * ntl)) |
                          ((uint32_t)((ty - oy) & (nt - 1)) << ntl) | (uint32_t)((tz - oz) & (nt - 1));
      lo = bstart[nb * 8 + c_runs[t][1]];
      len = bstart[nb * 8 + c_runs[t][2]] - lo;
    }
    uint32_t x = len;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      uint32_t y = __shfl_up_sync(0xffffffffu, x, d);
      if (t >= d) x += y;
    }
    if (t < 14) {
      run_lo[t] = lo;
      run_pre[t + 1] = x;
    }
    if (t == 0) run_pre[0] = 0;
  }
  __syncthreads();
  const float fscale = 1.0f / (float)(1u << shift);
  const uint32_t fmask = (1u << shift) - 1u;
  const uint32_t total = run_pre[14];
  // One particle per thread (coalesced loads in bucket order), its 8 corners added by
  // the same thread.
  const int ox = tx * kTile, oy = ty * kTile, oz = tz * kTile;
  bool bad = false, wrap = false;
  int r = 0;
  // the particle of iteration v + NT is loaded while v's corners are added
  auto locate = [&](uint32_t v) {
    while (v >= run_pre[r + 1]) ++r;  // v only grows, so the run index only grows
    return run_lo[r] + (v - run_pre[r]);
  };
  uint32_t qid = 0, qu0 = 0, qu1 = 0, qu2 = 0;
  float qw[NA];
  auto load = [&](uint32_t k) {
    if constexpr (NW > 0) {
#pragma unroll
      for (int j = 0; j < NW; ++j) qw[j] = wts[(int64_t)j * n + k];
    } else {
      qid = ids[k];
    }
    qu0 = us[k];
    qu1 = us[n + k];
    qu2 = us[2 * n + k];
  };
  if ((uint32_t)t < total) load(locate(t));
  for (uint32_t v = t; v < total; v += NT) {
    const uint32_t u0 = qu0, u1 = qu1, u2 = qu2, idv = qid;
    float m[NA];  // mass, or the signed weights
#pragma unroll
    for (int j = 0; j < NA; ++j) m[j] = NW > 0 ? qw[j] : 0.0f;
    const uint32_t vn = v + NT;
    if (vn < total) load(locate(vn));
    if constexpr (NW == 0) m[0] = id_mass(mt, idv, species, &bad);
    if constexpr (NW <= 1) {
      if (m[0] == 0.0f) continue;
    }
    int l[3] = {(int)(u0 >> shift) - ox, (int)(u1 >> shift) - oy, (int)(u2 >> shift) - oz};
    int lo_ok = 0;  // bit d: lower corner inside along d; bit 3 + d: upper inside
#pragma unroll
    for (int d = 0; d < 3; ++d) {  // periodic wrap relative to the tile origin
      if (l[d] > nm / 2) l[d] -= nm;
      if (l[d] < -nm / 2) l[d] += nm;
      if (l[d] >= 0 && l[d] < kTile) lo_ok |= 1 << d;
      if (l[d] + 1 >= 0 && l[d] + 1 < kTile) lo_ok |= 8 << d;
    }
    const int cell = l[0] * kSx + l[1] * kSy + l[2];
    const float fx = (float)(u0 & fmask) * fscale, fy = (float)(u1 & fmask) * fscale,
                fz = (float)(u2 & fmask) * fscale;
#pragma unroll
    for (int corner = 0; corner < 8; ++corner) {
      const int bx = corner >> 2, by = (corner >> 1) & 1, bz = corner & 1;
      const bool inside = ((lo_ok >> (bx ? 3 : 0)) & 1) && ((lo_ok >> (by ? 4 : 1)) & 1) &&
                          ((lo_ok >> (bz ? 5 : 2)) & 1);
      if (inside) {
        const int ad = cell + bx * kSx + by * kSy + bz;
        const float wc = (bx ? fx : 1.0f - fx) * (by ? fy : 1.0f - fy) * (bz ? fz : 1.0f - fz);
        if constexpr (FAST) {
          const unsigned int q = __float2uint_rn(wc * m[0] * kFixM);  // < 2^31: masses below 128
          const unsigned int old = atomicAdd(&acc_lo[ad], q);
          if (old + q < old && !record_wrap(accw, ad)) wrap = true;  // the low word wrapped; a full list
        } else {
#pragma unroll
          for (int j = 0; j < NA; ++j) {
            unsigned int* const w = acc_lo + j * 2 * kAccWords + ad;
            add64(w, w + kAccWords, fixed64(wc * m[j] * (NW > 0 ? kFixW : kFixM)));
          }
        }
      }
    }
  }
  if (bad) atomicOr(err, 1);
  if constexpr (FAST) {
    // the barrier's vote tells every thread whether the event list overflowed
    if (__syncthreads_or(wrap ? 1 : 0)) {
      paint_halves<NT>(tile, accw, run_lo, run_pre, us, ids, n, mesh, mt, species, nm, shift, ntl, row_pitch);
      return;
    }
  } else {
    __syncthreads();
  }
  // FAST: whether any low word of the tile wrapped (else the write-out reads low words only)
  bool any_wrap = false;
  if constexpr (FAST) any_wrap = *(volatile unsigned int*)wcount != 0u;
  // write the tile: 256 rows of 16 floats, as float4
#pragma unroll
  for (int j = 0; j < NA; ++j) {
    float* const mj = j == 0 ? mesh : (j == 1 ? mesh1 : mesh2);
    for (int q = t; q < kTile * kTile * kTile / 4; q += NT) {
      int row = q >> 2, z4 = (q & 3) * 4;
      int lx = row >> 4, ly = row & 15;
      const int a0 = lx * kSx + ly * kSy + z4;
      float fv[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const unsigned int ad = a0 + e, lo = acc_lo[j * 2 * kAccWords + ad];
        if constexpr (FAST) {
          if (any_wrap && ((wbits[ad >> 5] >> (ad & 31)) & 1u)) {  // the cell wrapped: count its events
            const unsigned int ne = *(volatile unsigned int*)wcount;
            unsigned int hi = 0;
            for (unsigned int k = 0; k < ne; ++k) hi += wlist[k] == ad ? 1u : 0u;
            fv[e] = __ull2float_rn(((unsigned long long)hi << 32) + (unsigned long long)lo);
          } else {
            fv[e] = __uint2float_rn(lo);
          }
        } else {
          fv[e] = float64w(acc_lo[(j * 2 + 1) * kAccWords + ad], lo);
        }
      }
      const float un = NW > 0 ? kUnfixW : kUnfixM;
      float4 v = make_float4(fv[0] * un, fv[1] * un, fv[2] * un, fv[3] * un);
      size_t off = ((size_t)(ox + lx) * nm + (oy + ly)) * (size_t)row_pitch + oz + z4;
      *reinterpret_cast<float4*>(mj + off) = v;
    }
  }
}

// One CTA per tile.  FAST: the 32-bit form with wrap events (masses below 128); else the
// two-word form, with NW signed weights instead of masses when NW > 0.
template <bool FAST, int NW, int NT>
__global__ void __launch_bounds__(NT, FAST ? 2048 / NT : 1) k_paint_tiles(
    const uint32_t* us, const uint32_t* ids, int64_t n,
    const uint32_t* bstart, float* __restrict__ mesh, const __grid_constant__ MassTable mt, int species,
    int nm, int shift, int ntl, int row_pitch, int* __restrict__ err, const float* wts) {
  pdl_begin();
  __shared__ __align__(16) unsigned int accw[FAST ? kFastWords : 2 * kAccWords];
  __shared__ uint32_t run_lo[14], run_pre[15];
  paint_tile<FAST, NW, NT>(blockIdx.x, accw, run_lo, run_pre, us, ids, n, bstart, mesh, mt, species, nm,
                                      shift, ntl, row_pitch, err, wts);
}

// Three signed weights a particle onto three meshes in one pass over the particles: positions,
// corners and weights of the corners once instead of three times.  The 109 KB of sums leave two
// CTAs an SM, of 512 threads so that 32 warps hide the atomics' latency.
constexpr int kPaint3Threads = 512;
constexpr size_t kPaint3Smem = sizeof(unsigned int) * 3 * 2 * kAccWords;
__global__ void __launch_bounds__(kPaint3Threads, 2) k_paint_weights3(
    const uint32_t* us, int64_t n, const uint32_t* bstart, float* __restrict__ m0,
    float* __restrict__ m1, float* __restrict__ m2, int nm, int shift, int ntl, int row_pitch, int* __restrict__ err,
    const float* wts) {
  pdl_begin();
  extern __shared__ __align__(16) unsigned int accw3[];
  __shared__ uint32_t run_lo[14], run_pre[15];
  const MassTable none{};
  paint_tile<false, 3, kPaint3Threads>(blockIdx.x, accw3, run_lo, run_pre, us, nullptr, n, bstart, m0, none, 0, nm,
                                       shift, ntl, row_pitch, err, wts, m1, m2);
}

// CIC readout of one real mesh component fused with the kick p_j += K F_j.
__global__ void k_readout_kick(const uint32_t* us, const float* ps,
                               const uint32_t* ids, int64_t n,
                               const float* mesh, int nm, int shift, int row_pitch,
                               int comp, float K, float* __restrict__ p_out,
                               float* __restrict__ f_out, uint32_t* __restrict__ u_out,
                               uint32_t* __restrict__ id_out, const uint32_t* perm) {
  pdl_begin();
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const uint32_t ux = us[i], uy = us[n + i], uz = us[2 * n + i];
  const float fscale = 1.0f / (float)(1u << shift);
  const uint32_t fmask = (1u << shift) - 1u;
  const int cx = ux >> shift, cy = uy >> shift, cz = uz >> shift;
  const int cx1 = (cx + 1) & (nm - 1), cy1 = (cy + 1) & (nm - 1), cz1 = (cz + 1) & (nm - 1);
  const float fx = (float)(ux & fmask) * fscale, fy = (float)(uy & fmask) * fscale,
              fz = (float)(uz & fmask) * fscale;
  const size_t r00 = ((size_t)cx * nm + cy) * row_pitch, r01 = ((size_t)cx * nm + cy1) * row_pitch;
  const size_t r10 = ((size_t)cx1 * nm + cy) * row_pitch, r11 = ((size_t)cx1 * nm + cy1) * row_pitch;
  const float v000 = mesh[r00 + cz], v001 = mesh[r00 + cz1];
  const float v010 = mesh[r01 + cz], v011 = mesh[r01 + cz1];
  const float v100 = mesh[r10 + cz], v101 = mesh[r10 + cz1];
  const float v110 = mesh[r11 + cz], v111 = mesh[r11 + cz1];
  const float gx = 1.0f - fx, gy = 1.0f - fy, gz = 1.0f - fz;
  const float F = gx * (gy * (gz * v000 + fz * v001) + fy * (gz * v010 + fz * v011)) +
                  fx * (gy * (gz * v100 + fz * v101) + fy * (gz * v110 + fz * v111));
  if (perm) {  // stage-level readout / force in the caller's order
    uint32_t j = perm[i];
    f_out[(int64_t)comp * n + j] = F;
    return;
  }
  if (p_out) p_out[(int64_t)comp * n + i] = __fmaf_rn(K, F, ps[(int64_t)comp * n + i]);
  if (f_out) f_out[(int64_t)comp * n + i] = F;
  if (u_out) {
    u_out[i] = ux;
    u_out[n + i] = uy;
    u_out[2 * n + i] = uz;
    id_out[i] = ids[i];
  }
}

// CIC readout of all three force meshes at once, fused with the kick p += K F.
__global__ void k_readout3_kick(const uint32_t* us, const float* ps,
                                const uint32_t* ids, int64_t n,
                                const float* mx, const float* my,
                                const float* mz, int nm, int shift, int row_pitch,
                                float K, float* __restrict__ p_out, float* __restrict__ f_out,
                                uint32_t* __restrict__ u_out, uint32_t* __restrict__ id_out,
                                const uint32_t* perm) {
  pdl_begin();
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const uint32_t ux = us[i], uy = us[n + i], uz = us[2 * n + i];
  const float fscale = 1.0f / (float)(1u << shift);
  const uint32_t fmask = (1u << shift) - 1u;
  const int cx = ux >> shift, cy = uy >> shift, cz = uz >> shift;
  const int cx1 = (cx + 1) & (nm - 1), cy1 = (cy + 1) & (nm - 1), cz1 = (cz + 1) & (nm - 1);
  const float fx = (float)(ux & fmask) * fscale, fy = (float)(uy & fmask) * fscale,
              fz = (float)(uz & fmask) * fscale;
  const float gx = 1.0f - fx, gy = 1.0f - fy, gz = 1.0f - fz;
  const size_t r00 = ((size_t)cx * nm + cy) * row_pitch, r01 = ((size_t)cx * nm + cy1) * row_pitch;
  const size_t r10 = ((size_t)cx1 * nm + cy) * row_pitch, r11 = ((size_t)cx1 * nm + cy1) * row_pitch;
  const float w000 = gx * gy * gz, w001 = gx * gy * fz, w010 = gx * fy * gz, w011 = gx * fy * fz;
  const float w100 = fx * gy * gz, w101 = fx * gy * fz, w110 = fx * fy * gz, w111 = fx * fy * fz;
  const float* m[3] = {mx, my, mz};
  float F[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const float* g = m[d];
    F[d] = w000 * g[r00 + cz] + w001 * g[r00 + cz1] + w010 * g[r01 + cz] +
           w011 * g[r01 + cz1] + w100 * g[r10 + cz] + w101 * g[r10 + cz1] +
           w110 * g[r11 + cz] + w111 * g[r11 + cz1];
  }
  if (perm) {  // force in the caller's order
    const uint32_t j = perm[i];
#pragma unroll
    for (int d = 0; d < 3; ++d) f_out[(int64_t)d * n + j] = F[d];
    return;
  }
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    if (p_out) p_out[(int64_t)d * n + i] = __fmaf_rn(K, F[d], ps[(int64_t)d * n + i]);
    if (f_out) f_out[(int64_t)d * n + i] = F[d];
  }
  if (u_out) {
    u_out[i] = ux;
    u_out[n + i] = uy;
    u_out[2 * n + i] = uz;
    id_out[i] = ids[i];
  }
}

// Force from the potential mesh with the 4-point gradient in real space, fused with
// the kick.  The finite-difference gradient [8 (phi(x+H) - phi(x-H)) - (phi(x+2H) -
// phi(x-2H))] / (12 H) has exactly the transfer function i D(k) of the k-space kernel
// (0 on the Nyquist index), so this equals the CIC readout of IFFT(-i D(k_j) phi_k)
// while the mesh side needs one inverse transform instead of three.
//
// One CTA per 16^3 tile.  The tile's potential with a halo of 2 cells below and 3
// above along x and y, and of 4 below and 3 above along z (so that every z row splits
// into 16-byte aligned chunks, also where it wraps), is staged in shared memory with
// asynchronous 16-byte copies (21 x 21 x 24 floats).  Each thread then takes particles
// of the tile's bucket range [bstart[8 t], bstart[8 t + 8]), all of whose cells lie
// in the tile, and gathers the 56 potential values its 8 CIC corners' stencils touch;
// the first particle's position is loaded while the copies are in flight, the next
// one's while the current one is computed.  Differences of neighbouring values are
// formed first, so FP32 rounding scales with the gradient, not with the potential.
// A particle outside its tile (a bucket range that does not match the positions)
// sets the error word's invalid-input bit.
// The next step's first half kick and drift, fused into the readout that ends a step
// (pm_run): p = (ps + K2 F) + K1' F, u' = u + rne(Delta' p 2^32 / L), in the operations
// and order of the unfused path (readout, then k_kick_drift_keys), so the state is
// bit-identical.  Writes the new key and the near-sorted re-sort's counts (the
// particle's old key is its current bucket, so it is in range by construction).
__device__ __forceinline__ uint32_t drift_fixed(uint32_t u, float dscale, float p) {
  const float x = dscale * p;
  const uint32_t step = fabsf(x) < 2147483648.0f ? (uint32_t)__float2int_rn(x)
                                                 : (uint32_t)(unsigned long long)__float2ll_rn(x);
  return u + step;
}

// Counts for the near-sorted re-sort, by the lanes of act: all particles by new key kn, stayers
// (new key = old key) by new key, movers by old key, movers from a lower key by new key.  The
// lanes hold consecutive particles of the state; those in range of their old key ko (in) have
// old keys that never decrease from lane to lane, so stayers and movers are counted per run
// of equal old keys with ballots, and only the movers' new keys need a match over the lanes.
__device__ __forceinline__ void count_resort(unsigned act, uint32_t kn, uint32_t ko, bool in, uint32_t* __restrict__ cnt3,
                                             long long nb1, uint32_t* __restrict__ low) {
  const int lane = threadIdx.x & 31;
  const bool stay = in && kn == ko;
  const unsigned below = act & ((1u << lane) - 1u);
  const int prev = below ? 31 - __clz(below) : lane;  // the nearest active lane below
  const uint32_t run_key = in ? ko : 0xffffffffu;
  const uint32_t prev_key = __shfl_sync(act, run_key, prev);
  const bool head = prev == lane || prev_key != run_key;
  const unsigned heads = __ballot_sync(act, head);
  const unsigned stays = __ballot_sync(act, stay);
  const unsigned lows = __ballot_sync(act, in && ko < kn);
  if (head && in) {
    const unsigned after = heads & ~((2u << lane) - 1u);  // heads above this lane (lane 31: none)
    const unsigned upto = after ? (1u << (__ffs(after) - 1)) - 1u : 0xffffffffu;
    const unsigned run = act & upto & ~((1u << lane) - 1u);
    const uint32_t ns = (uint32_t)__popc(run & stays), nmv = (uint32_t)__popc(run & ~stays);
    if (ns) {
      atomicAdd(cnt3 + ko, ns);
      atomicAdd(cnt3 + nb1 + ko, ns);
    }
    if (nmv) atomicAdd(cnt3 + 2 * nb1 + ko, nmv);
  }
  if (!stay) {
    const unsigned peers = __match_any_sync(act & ~stays, kn);
    if (lane == __ffs(peers) - 1) {
      atomicAdd(cnt3 + kn, (uint32_t)__popc(peers));
      const uint32_t nl = (uint32_t)__popc(peers & lows);
      if (nl) atomicAdd(low + kn, nl);
    }
  }
}

__device__ __forceinline__ void drift_next(const DriftNext& dn, const float (&F)[3], const float (&pv)[3],
                                           float K2, int64_t n, uint32_t i, uint32_t ux, uint32_t uy, uint32_t uz,
                                           int shift, int ntl, float* __restrict__ p_out, float* __restrict__ f_out,
                                           uint32_t* __restrict__ u_out) {
  uint32_t uu[3] = {ux, uy, uz};
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const float p1 = __fmaf_rn(K2, F[d], pv[d]);
    const float p2 = __fmaf_rn(dn.K1, F[d], p1);
    p_out[(int64_t)d * n + i] = p2;
    if (f_out) f_out[(int64_t)d * n + i] = F[d];
    uu[d] = drift_fixed(uu[d], dn.dscale, p2);
    u_out[(int64_t)d * n + i] = uu[d];
  }
  const uint32_t kn = tile_key(uu[0], uu[1], uu[2], shift, ntl);
  const uint32_t ko = tile_key(ux, uy, uz, shift, ntl);
  dn.keys[i] = kn;
  count_resort(__activemask(), kn, ko, true, dn.cnt3, dn.nb1, dn.low);
}

constexpr int kSpanXY = kTile + 5;                 // cells -2 .. 18 along x and y
constexpr int kSpanZ = kTile + 8;                  // cells -4 .. 19 along z
constexpr int kChunksZ = kSpanZ / 4;               // 16-byte chunks per staged z row
constexpr int kStageChunks = kSpanXY * kSpanXY * kChunksZ;
constexpr int kFd4SY = kSpanZ, kFd4SX = kSpanXY * kSpanZ;
constexpr int kNodeThreads = 512;
constexpr int kNodesMin = 1500;    // mean particles a tile from which the node form is taken
constexpr int kNodes = kTile + 1;  // corner nodes of a tile per axis
constexpr size_t kFd4Smem = sizeof(float) * kSpanXY * kFd4SX;
constexpr size_t kNodeSmem = kFd4Smem + sizeof(float) * 3 * kNodes * kNodes * kNodes;

__device__ __forceinline__ void cp_async16(void* smem_dst, const void* gmem_src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(smem_dst)),
               "l"(gmem_src)
               : "memory");
}

// The tile's potential with its halo into sp, by asynchronous copies of one group.  Chunk k of
// staged row (x, y) holds cells oz - 4 + 4k .. oz - 1 + 4k (mod N): contiguous and 16-byte aligned
// because N, oz and the row pitch are multiples of 4 floats.
template <int NT>
__device__ __forceinline__ void stage_potential(float* sp, const float* phi, int ox, int oy, int oz, int nm,
                                                int row_pitch) {
  const int wrap = nm - 1;
  for (int c = threadIdx.x; c < kStageChunks; c += NT) {
    const int x = c / (kSpanXY * kChunksZ), r = c - x * (kSpanXY * kChunksZ);
    const int y = r / kChunksZ, k = r - y * kChunksZ;
    const int gx = (ox + x - 2) & wrap, gy = (oy + y - 2) & wrap, gz = (oz - 4 + 4 * k) & wrap;
    cp_async16(sp + x * kFd4SX + y * kFd4SY + 4 * k, phi + ((size_t)gx * nm + gy) * (size_t)row_pitch + gz);
  }
  asm volatile("cp.async.commit_group;" ::: "memory");
}

// NODES = false: each particle gathers the 56 potential values of its 8 corners' stencils
// (207 shared-memory wavefronts a warp: random cells, about 3.7 conflicts a gather).  NODES =
// true: the CTA first computes the force at the tile's 17^3 corner nodes (2500 wavefronts, free
// of conflicts), then each particle gathers 8 x 3 values (89 wavefronts a warp).  us a launch of
// 4096 tiles, gathering / nodes, by mean particles a tile: 500 63 / 104, 1000 113 / 131, 1500
// 162 / 157, 2000 211 / 184, 4000 411 / 292, 8000 806 / 494.
// The gathering form runs five CTAs an SM (48 registers; at 60 to 104 it holds four to two: 4.65
// to 6.2 ms against 4.1 on the late steps of 152 M particles at 1024^3).
template <bool DRIFT, bool NODES, int NT>
__global__ void __launch_bounds__(NT, NODES ? 2 : (NT == 256 ? 5 : 1024 / NT)) k_readout_fd4_kick(
    const uint32_t* us, const float* ps, const uint32_t* ids,
    int64_t n, const uint32_t* bstart, const float* phi, int nm, int shift,
    int ntl, int row_pitch, float inv12h, float K, float* __restrict__ p_out, float* __restrict__ f_out,
    uint32_t* __restrict__ u_out, uint32_t* __restrict__ id_out, const uint32_t* perm,
    int* __restrict__ err, DriftNext dn) {
  pdl_begin();
  extern __shared__ __align__(16) float sp[];  // the potential, then (NODES) the nodes' forces
  float* const nodes = sp + kSpanXY * kFd4SX;
  const int t = threadIdx.x;
  const uint32_t tile = blockIdx.x;
  const uint32_t lo = bstart[8 * tile], hi = bstart[8 * tile + 8];
  if (lo == hi) return;
  const int nt = 1 << ntl;
  const int ox = (int)(tile >> (2 * ntl)) * kTile, oy = (int)((tile >> ntl) & (nt - 1)) * kTile,
            oz = (int)(tile & (nt - 1)) * kTile;
  stage_potential<NT>(sp, phi, ox, oy, oz, nm, row_pitch);
  // a particle's position, momentum and id are loaded one iteration ahead
  const bool kick = ps != nullptr && perm == nullptr;
  auto load = [&](uint32_t j, uint32_t (&uq)[3], float (&pq)[3], uint32_t& idq) {
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      uq[d] = us[(int64_t)d * n + j];
      pq[d] = kick ? ps[(int64_t)d * n + j] : 0.0f;
    }
    idq = id_out ? ids[j] : 0u;
  };
  uint32_t i = lo + t;
  uint32_t cu[3] = {0u, 0u, 0u}, cid = 0u;
  float cp[3] = {0.f, 0.f, 0.f};
  if (i < hi) load(i, cu, cp, cid);
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncthreads();
  if constexpr (NODES) {
    for (int c = t; c < kNodes * kNodes * kNodes; c += NT) {
      const int x = c / (kNodes * kNodes), r = c - x * (kNodes * kNodes), y = r / kNodes, z = r - y * kNodes;
      const float* const q = sp + (x + 2) * kFd4SX + (y + 2) * kFd4SY + (z + 4);
      auto st = [q](int S) { return 8.0f * (q[S] - q[-S]) - (q[2 * S] - q[-2 * S]); };
      nodes[3 * c] = -inv12h * st(kFd4SX);
      nodes[3 * c + 1] = -inv12h * st(kFd4SY);
      nodes[3 * c + 2] = -inv12h * st(1);
    }
    __syncthreads();
  }
  const float fscale = 1.0f / (float)(1u << shift);
  const uint32_t fmask = (1u << shift) - 1u;
  bool bad = false, nonfinite = false;
  for (; i < hi; i += NT) {
    const uint32_t inext = i + NT;
    uint32_t nu[3] = {0u, 0u, 0u}, nid = 0u;
    float np[3] = {0.f, 0.f, 0.f};
    if (inext < hi) load(inext, nu, np, nid);
    const uint32_t ux = cu[0], uy = cu[1], uz = cu[2];
    const int lx = (int)(ux >> shift) - ox, ly = (int)(uy >> shift) - oy, lz = (int)(uz >> shift) - oz;
    if ((unsigned)lx < (unsigned)kTile && (unsigned)ly < (unsigned)kTile && (unsigned)lz < (unsigned)kTile) {
      const float fx = (float)(ux & fmask) * fscale, fy = (float)(uy & fmask) * fscale,
                  fz = (float)(uz & fmask) * fscale;
      const float gx = 1.0f - fx, gy = 1.0f - fy, gz = 1.0f - fz;
      float F[3];
      if constexpr (NODES) {
        const float* const q = nodes + 3 * ((lx * kNodes + ly) * kNodes + lz);
        constexpr int Y = 3 * kNodes, X = 3 * kNodes * kNodes;
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          const float* const v = q + d;
          F[d] = gx * (gy * (gz * v[0] + fz * v[3]) + fy * (gz * v[Y] + fz * v[Y + 3])) +
                 fx * (gy * (gz * v[X] + fz * v[X + 3]) + fy * (gz * v[X + Y] + fz * v[X + Y + 3]));
        }
      } else {
        const float* q = sp + (lx + 2) * kFd4SX + (ly + 2) * kFd4SY + (lz + 4);  // phi at the particle's cell
        // stencil sum of one axis at the two corners 0 (weight g) and 1 (weight f) of a
        // line through q0 with stride S: g (8 (p1 - m1) - (p2 - m2)) + f (8 (p2 - p0) - (p3 - m1))
        auto axis_sum = [](const float* q0, int S, float g, float f) {
          const float m2 = q0[-2 * S], m1 = q0[-S], p0 = q0[0], p1 = q0[S], p2 = q0[2 * S], p3 = q0[3 * S];
          return g * (8.0f * (p1 - m1) - (p2 - m2)) + f * (8.0f * (p2 - p0) - (p3 - m1));
        };
        float Fx = 0.0f, Fy = 0.0f, Fz = 0.0f;
#pragma unroll
        for (int a = 0; a < 2; ++a) {
#pragma unroll
          for (int b = 0; b < 2; ++b) {
            // x lines at (y, z) = (b, a); y lines at (x, z) = (b, a); z lines at (x, y) = (b, a)
            Fx = fmaf((b ? fy : gy) * (a ? fz : gz), axis_sum(q + b * kFd4SY + a, kFd4SX, gx, fx), Fx);
            Fy = fmaf((b ? fx : gx) * (a ? fz : gz), axis_sum(q + b * kFd4SX + a, kFd4SY, gy, fy), Fy);
            Fz = fmaf((b ? fx : gx) * (a ? fy : gy), axis_sum(q + b * kFd4SX + a * kFd4SY, 1, gz, fz), Fz);
          }
        }
        F[0] = -inv12h * Fx;
        F[1] = -inv12h * Fy;
        F[2] = -inv12h * Fz;
      }
      // a NaN or infinity in the force or the incoming momentum poisons the sum
      if (!isfinite(F[0] + F[1] + F[2] + cp[0] + cp[1] + cp[2])) nonfinite = true;
      if (perm) {  // force in the caller's order
        const uint32_t j = perm[i];
#pragma unroll
        for (int d = 0; d < 3; ++d) f_out[(int64_t)d * n + j] = F[d];
      } else if constexpr (DRIFT) {
        drift_next(dn, F, cp, K, n, i, ux, uy, uz, shift, ntl, p_out, f_out, u_out);
        id_out[i] = cid;
      } else {
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          if (p_out) p_out[(int64_t)d * n + i] = __fmaf_rn(K, F[d], cp[d]);
          if (f_out) f_out[(int64_t)d * n + i] = F[d];
        }
        if (u_out) {
          u_out[i] = ux;
          u_out[n + i] = uy;
          u_out[2 * n + i] = uz;
          id_out[i] = cid;
        }
      }
    } else {
      bad = true;
    }
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      cu[d] = nu[d];
      cp[d] = np[d];
    }
    cid = nid;
  }
  if (bad) atomicOr(err, 1);
  if (nonfinite) atomicOr(err, 4);
}

// First half kick with the cached force, drift in fixed point, next sort key.
// RESORT (the state is in the tile order of the last step, whose bucket starts are
// bprev): also classify each particle for the near-sorted re-sort of k_sort.cu.  A
// stayer keeps its key ko; every other particle is a mover.  Counts (cnt3 holds three
// arrays of nbuckets + 1): cnt3[0][kn] all particles of new key kn, cnt3[1][kn]
// stayers, cnt3[2][ko] movers out of old key ko; low[kn] movers from a lower old key.
// Flag bit 1: a particle outside its old key's range [bprev[ko], bprev[ko + 1]) (the
// state is not in bprev's order: every particle is then sorted as a mover).
template <bool RESORT>
__global__ void k_kick_drift_keys(uint32_t* __restrict__ u, float* __restrict__ p,
                                  const float* f, int64_t n, float K1, float dscale,
                                  int shift, int ntl, uint32_t* __restrict__ keys,
                                  uint32_t* __restrict__ cnt3, long long nb1, const uint32_t* bprev,
                                  uint32_t* __restrict__ low, uint32_t* __restrict__ flags, int* __restrict__ err) {
  pdl_begin();
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const unsigned act = __ballot_sync(0xffffffffu, i < n);
  if (i >= n) return;
  uint32_t uu[3], u0[3];
  float pv[3], chk = 0.0f;  // a NaN or infinity in p or f poisons the sum
#pragma unroll
  for (int d = 0; d < 3; ++d) {  // every load before the first store
    pv[d] = __fmaf_rn(K1, f[d * n + i], p[d * n + i]);
    u0[d] = u[d * n + i];
  }
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    chk += pv[d];
    p[d * n + i] = pv[d];
    // u += rne(Delta p 2^32 / L), modulo 2^32; the 32-bit conversion (same rounding)
    // whenever the step fits, the 64-bit one (FP64 pipe) only for steps of 2^31 or more
    uu[d] = drift_fixed(u0[d], dscale, pv[d]);
    u[d * n + i] = uu[d];
  }
  const uint32_t key = tile_key(uu[0], uu[1], uu[2], shift, ntl);
  keys[i] = key;
  if (!isfinite(chk)) atomicOr(err, 4);
  if constexpr (RESORT) {
    const uint32_t k0 = tile_key(u0[0], u0[1], u0[2], shift, ntl);
    const bool in = (uint32_t)i >= bprev[k0] && (uint32_t)i < bprev[k0 + 1];
    count_resort(act, key, k0, in, cnt3, nb1, low);
    const unsigned out = __ballot_sync(act, !in);
    if (out && (int)(threadIdx.x & 31) == __ffs(out) - 1) atomicOr(flags, 1u);
  }
}

__global__ void k_repack_real(const float* src, int sp, float* __restrict__ dst,
                              int dp, int nm) {
  pdl_begin();
  long long row = blockIdx.x;
  for (int z = threadIdx.x; z < nm; z += blockDim.x) dst[row * dp + z] = src[row * sp + z];
}

__global__ void k_repack_complex(const float2* src, int sp, float2* __restrict__ dst,
                                 int dp, int ncols) {
  pdl_begin();
  long long row = blockIdx.x;
  for (int z = threadIdx.x; z < ncols; z += blockDim.x) dst[row * dp + z] = src[row * sp + z];
}

}  // namespace

void paint_tiles(pm_ctx* c, const uint32_t* us, const uint32_t* ids, int64_t n, int species,
                 float* mesh, int row_pitch, cudaStream_t s, const float* weights) {
  unsigned grid = (unsigned)(c->nt * c->nt * c->nt);
  float mmax = 0.0f;  // largest particle mass of the painted species
  if (species & PM_SPECIES_CDM) mmax = std::max(mmax, c->mt.m_cdm);
  if (species & PM_SPECIES_NU)
    for (int i = 0; i < c->mt.nshell && i < kMaxShell; ++i) mmax = std::max(mmax, c->mt.m_nu[i]);
  LaunchScope L(c, s, K_PAINT);
  // masses below 128: w 2^24 < 2^31, so every contribution fits the 32-bit form
  int threads = kPaintThreads;
  auto kern = k_paint_tiles<false, 1, kPaintThreads>;
  if (!weights) {
    kern = k_paint_tiles<false, 0, kPaintThreads>;
    if (mmax < 128.0f) {
      threads = tile_threads(c);
      kern = threads == 1024 ? k_paint_tiles<true, 0, 1024>
                             : (threads == 512 ? k_paint_tiles<true, 0, 512> : k_paint_tiles<true, 0, 256>);
    }
  }
  pdl_launch(kern, grid, threads, 0, s, us, ids, n, c->bstart, mesh, c->mt, species, c->g.n, 32 - c->g.logn, c->ntl,
                                      row_pitch, c->err_dev, weights);
}

void paint_weights3(pm_ctx* c, const uint32_t* us, int64_t n, const float* weights, float* m0, float* m1, float* m2,
                    int row_pitch, cudaStream_t s) {
  static DeviceOnce once;
  allow_smem(once, (const void*)k_paint_weights3, kPaint3Smem);
  LaunchScope L(c, s, K_PAINT);
  pdl_launch(k_paint_weights3, (unsigned)(c->nt * c->nt * c->nt), kPaint3Threads, kPaint3Smem, s, 
      us, n, c->bstart, m0, m1, m2, c->g.n, 32 - c->g.logn, c->ntl, row_pitch, c->err_dev, weights);
}

void readout_kick(pm_ctx* c, const uint32_t* us, const float* ps, const uint32_t* ids, int64_t n,
                  const float* mesh, int row_pitch, int comp, float K, float* p_out, float* f_out,
                  uint32_t* u_out, uint32_t* id_out, const uint32_t* perm_scatter,
                  cudaStream_t s) {
  if (n == 0) return;
  LaunchScope L(c, s, K_READOUT_KICK);
  pdl_launch(k_readout_kick, (unsigned)((n + 255) / 256), 256, 0, s, 
      us, ps, ids, n, mesh, c->g.n, 32 - c->g.logn, row_pitch, comp, K, p_out, f_out, u_out,
      id_out, perm_scatter);
}

void readout3_kick(pm_ctx* c, const uint32_t* us, const float* ps, const uint32_t* ids, int64_t n,
                   const float* mx, const float* my, const float* mz, int row_pitch, float K,
                   float* p_out, float* f_out, uint32_t* u_out, uint32_t* id_out,
                   const uint32_t* perm_scatter, cudaStream_t s) {
  if (n == 0) return;
  LaunchScope L(c, s, K_READOUT3_KICK);
  pdl_launch(k_readout3_kick, (unsigned)((n + 255) / 256), 256, 0, s, 
      us, ps, ids, n, mx, my, mz, c->g.n, 32 - c->g.logn, row_pitch, K, p_out, f_out, u_out, id_out,
      perm_scatter);
}

void readout_fd4_kick(pm_ctx* c, const uint32_t* us, const float* ps, const uint32_t* ids, int64_t n,
                      const float* phi, int row_pitch, float K, float* p_out, float* f_out,
                      uint32_t* u_out, uint32_t* id_out, const uint32_t* perm_scatter, cudaStream_t s,
                      const DriftNext* dn) {
  if (n == 0) return;
  LaunchScope L(c, s, K_READOUT_FD4_KICK);
  const float inv12h = (float)((double)c->g.n / (12.0 * c->cfg.box));
  const unsigned grid = (unsigned)(c->nt * c->nt * c->nt);
  // Forces at the nodes first where tiles are full: see the kernel for both sides, measured with 4096
  // tiles (256^3).  Meshes below keep the gathering form at any filling for the sake of their bits,
  // not of speed: the node form was not measured there.
  const bool nodes = c->g.n >= 256 && n >= (int64_t)kNodesMin * grid;
  const bool few = !nodes && tile_threads(c) == 1024;  // (at 128^3 five CTAs of 256 hold more warps than two of 512)
  const int threads = nodes ? kNodeThreads : (few ? 1024 : 256);
  const int v = nodes ? 2 : (few ? 1 : 0);
  decltype(&k_readout_fd4_kick<false, false, 256>) const kerns[2][3] = {
      {k_readout_fd4_kick<false, false, 256>, k_readout_fd4_kick<false, false, 1024>,
       k_readout_fd4_kick<false, true, kNodeThreads>},
      {k_readout_fd4_kick<true, false, 256>, k_readout_fd4_kick<true, false, 1024>,
       k_readout_fd4_kick<true, true, kNodeThreads>}};
  const auto kern = kerns[dn != nullptr][v];
  const size_t smem = nodes ? kNodeSmem : kFd4Smem;
  static DeviceOnce once[2][3];
  allow_smem(once[dn != nullptr][v], (const void*)kern, smem);
  pdl_launch(kern, grid, threads, smem, s, us, ps, ids, n, c->bstart, phi, c->g.n, 32 - c->g.logn,
                                                             c->ntl, row_pitch, inv12h, K, p_out, f_out, u_out, id_out,
                                                             dn ? nullptr : perm_scatter, c->err_dev,
                                                             dn ? *dn : DriftNext{});
}

void kick_drift_keys(pm_ctx* c, uint32_t* u, float* p, const float* f, int64_t n, float K1,
                     float dscale, cudaStream_t s, bool resort) {
  const long long nb1 = c->nbuckets + 1;
  if (resort) clear_resort(c, s);
  if (n == 0) return;
  LaunchScope L(c, s, K_KICK_DRIFT_KEYS);
  const unsigned grid = (unsigned)((n + 255) / 256);
  if (resort)
    pdl_launch(k_kick_drift_keys<true>, grid, 256, 0, s, u, p, f, n, K1, dscale, 32 - c->g.logn, c->ntl, c->keys[0],
                                                  c->counts, nb1, c->bprev, c->rs_low, c->rs_dev, c->err_dev);
  else
    pdl_launch(k_kick_drift_keys<false>, grid, 256, 0, s, u, p, f, n, K1, dscale, 32 - c->g.logn, c->ntl, c->keys[0],
                                                   c->counts, nb1, nullptr, nullptr, nullptr, c->err_dev);
}

void repack_real(pm_ctx* c, const Geom& g, const float* src, int sp, float* dst, int dp,
                 cudaStream_t s) {
  LaunchScope L(c, s, K_REPACK);
  pdl_launch(k_repack_real, (unsigned)g.rows(), 256, 0, s, src, sp, dst, dp, g.n);
}

void repack_complex(pm_ctx* c, const Geom& g, const float2* src, int sp, float2* dst, int dp,
                    cudaStream_t s) {
  LaunchScope L(c, s, K_REPACK);
  pdl_launch(k_repack_complex, (unsigned)g.rows(), 256, 0, s, src, sp, dst, dp, g.n / 2 + 1);
}

}  // namespace pmnu
