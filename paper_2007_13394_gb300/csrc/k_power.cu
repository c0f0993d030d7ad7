// Binned (cross) power spectrum of two half-spectrum meshes.
//
// P_ab(k) = (V / N^6) Re(delta_a delta_b^*) / W(k)^2 per mode, W the CIC window, each
// species mesh divided by its own mean (read from its k = 0 mode);
// bins of width k_F from k_F / 2: mode n (integer wavevector) falls in bin b when
// (b + 1/2)^2 <= |n|^2 < (b + 3/2)^2, decided exactly in integers.  Modes with
// 0 < n_z < N/2 count twice (Hermitian partners not stored).
//
// What bounds the binning is the FP64 pipe (about two operations a clock and SM) when every
// mode converts, takes a square root and adds three FP64 shared atomics: 3.15 ms at 512^3
// where the two spectra take 0.16 ms to read.  So:
// * The up to eight rows (+-n_x, +-n_y) and (+-n_y, +-n_x) share |n|, the window and the bin: a
//   warp takes all of them at once, adds their products error-free in pairs of FP32 (value and
//   rounding error), and converts one sum for eight modes to FP64.
// * Along a row the bin never decreases, so the lanes of one bin are neighbours: a segmented
//   warp sum leaves one addition per bin, into bins private to the warp -- no atomics, and a
//   fixed order: the spectrum is reproducible bit for bit.
// * Mode counts and sum |n| do not depend on the data: r2(t), the number of (n_x, n_y) with
//   n_x^2 + n_y^2 = t, is counted in integers, and bin b sums c(s) and c(s) sqrt(s) over its
//   2 (b + 1) values s = |n|^2 with c(s) = sum_{n_z} r2(s - n_z^2): one square root per s.
// Measured: the binning of a cross spectrum at 512^3, 256 bins, 3146 -> 143 us (two spectra of
// 540 MB: 7.5 TB/s), the counts and sums 47 -> 54 us; the spectrum's gradient at 256^3 (which needs
// the counts only, so no binning pass) 1.13 -> 0.51 ms a call.
#include <cuda_runtime.h>

#include <algorithm>

#include "pm_internal.cuh"

namespace pmnu {

namespace {

constexpr int kPowThreads = 256;
constexpr int kPowWarps = kPowThreads / 32;
constexpr int kMaxBins = 2048;
constexpr int kMaxRows = 608;  // CTAs of the binning pass (rows of partial sums), four an SM

__device__ __forceinline__ int bin_of(int n2) {
  int b = (int)floorf(sqrtf((float)n2) - 0.5f);
  if (b < 0) b = 0;
  while ((b + 1) * (b + 1) + (b + 1) < n2) ++b;   // n2 > (b+1)^2 + (b+1): next bin
  while (b > 0 && b * b + b >= n2) --b;            // n2 <= b^2 + b: previous bin
  return b;
}

// (a, b) of unit w in the triangle 0 <= b <= a <= N/2: the rows with {|n_x|, |n_y|} = {a, b}
__device__ __forceinline__ void unit_ab(int w, int& a, int& b) {
  a = (int)((sqrtf(8.0f * (float)w + 1.0f) - 1.0f) * 0.5f);
  while (a * (a + 1) / 2 > w) --a;
  while ((a + 1) * (a + 2) / 2 <= w) ++a;
  b = w - a * (a + 1) / 2;
}

// rows of the unit: multiplicity of |n| = i along an axis is 1 at 0 and N/2, else 2
__device__ __forceinline__ int axis_mult(int i, int nm) { return (i == 0 || i == nm / 2) ? 1 : 2; }

// r2[t] += the unit's (n_x, n_y) pairs, t = a^2 + b^2 (t <= tmax only)
__device__ __forceinline__ void count_unit(int a, int b, int nm, int tmax, uint32_t* r2) {
  const int t = a * a + b * b;
  if (t <= tmax) atomicAdd(r2 + t, (uint32_t)(axis_mult(a, nm) * axis_mult(b, nm) * (a != b ? 2 : 1)));
}

__global__ void k_power_counts(int nm, int units, int tmax, uint32_t* __restrict__ r2) {
  pdl_begin();
  const int w = blockIdx.x * blockDim.x + threadIdx.x;
  if (w >= units) return;
  int a, b;
  unit_ab(w, a, b);
  count_unit(a, b, nm, tmax, r2);
}

// Sums of Re(da db^*) mult / W^2 (unscaled) by bin, one row of nbins a CTA; also fills r2.
// A warp walks its units; for each, its lanes walk n_z, so every load covers 256 contiguous bytes.
template <bool CROSS>
__global__ void __launch_bounds__(kPowThreads) k_power_bin(const float2* da,
                                                           const float2* db, int nm,
                                                           int pc, int nbins, int units, int tmax,
                                                           const float* __restrict__ winv,
                                                           double* __restrict__ partial,
                                                           uint32_t* __restrict__ r2) {
  pdl_begin();
  extern __shared__ double sh[];  // nbins per warp
  for (int i = threadIdx.x; i < kPowWarps * nbins; i += kPowThreads) sh[i] = 0.0;
  __syncthreads();
  const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5, half = nm / 2;
  double* const mine = sh + wp * nbins;
  for (int w = blockIdx.x * kPowWarps + wp; w < units; w += gridDim.x * kPowWarps) {
    int a, b;
    unit_ab(w, a, b);
    const int p2 = a * a + b * b;
    if (p2 > tmax) continue;  // beyond the last bin
    if (lane == 0) count_unit(a, b, nm, tmax, r2);
    // row r of the unit: bit 0 mirrors a, bit 1 mirrors b, bit 2 swaps them
    const int ra = axis_mult(a, nm) - 1, rb = axis_mult(b, nm) - 1, rs = a != b ? 1 : 0;
    const float wab = __ldg(winv + a) * __ldg(winv + b);
    for (int z0 = 0; z0 <= half; z0 += 32) {
      const int kz = z0 + lane, n2 = p2 + kz * kz;
      const int bin = (kz <= half && n2 > 0) ? min(bin_of(n2), nbins) : (n2 > 0 ? nbins : 0);
      if (__shfl_sync(0xffffffffu, bin, 0) >= nbins) break;  // the bins only grow along the row
      float s = 0.0f, e = 0.0f;  // sum of the rows' products and its rounding error
      if (bin < nbins && n2 > 0) {
        float2 va[8], vb[8];
#pragma unroll
        for (int r = 0; r < 8; ++r) {
          const bool on = (!(r & 1) || ra) && (!(r & 2) || rb) && (!(r & 4) || rs);
          const int ia = (r & 1) ? nm - a : a, ib = (r & 2) ? nm - b : b;
          const size_t idx = ((size_t)((r & 4) ? ib : ia) * nm + ((r & 4) ? ia : ib)) * pc + kz;
          va[r] = on ? da[idx] : make_float2(0.f, 0.f);
          if constexpr (CROSS) vb[r] = on ? db[idx] : make_float2(0.f, 0.f);
        }
#pragma unroll
        for (int r = 0; r < 8; ++r) {
          const float2 y = CROSS ? vb[r] : va[r];
          const float re = va[r].x * y.x + va[r].y * y.y;
          const float t = s + re, d = t - s;  // Knuth's two-sum
          e += (s - (t - d)) + (re - d);
          s = t;
        }
      }
      const float f = wab * __ldg(winv + min(kz, half)) * ((kz == 0 || kz == half) ? 1.0f : 2.0f);
      const float p = s * f;
      double v = (double)p;
      if (isfinite(p)) v += (double)(fmaf(s, f, -p) + e * f);
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {  // sum of the lanes above of the same bin
        const double y = __shfl_down_sync(0xffffffffu, v, o);
        const int by = __shfl_down_sync(0xffffffffu, bin, o);
        if (lane + o < 32 && by == bin) v += y;
      }
      const int below = __shfl_up_sync(0xffffffffu, bin, 1);
      if (bin < nbins && (lane == 0 || below != bin)) mine[bin] += v;  // one lane a bin
      __syncwarp();
    }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < nbins; i += kPowThreads) {
    double t = 0.0;
    for (int q = 0; q < kPowWarps; ++q) t += sh[q * nbins + i];
    partial[(size_t)blockIdx.x * nbins + i] = t;
  }
}

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  return v;
}

// One CTA per bin: out = {mode counts, sum |k|, sum P} (nbins each).  The bin's s = |n|^2 run
// over b^2 + b < s <= (b + 1)^2 + (b + 1); a lane takes one of them and walks n_z.  With no
// partial rows (nrows = 0) only the counts and sum |k|.
constexpr int kRedThreads = 1024;
__global__ void __launch_bounds__(kRedThreads) k_power_reduce(const double* partial, int nrows, int nbins,
                                                              int nm, const uint32_t* r2, double kf,
                                                              float norm, const float2* da,
                                                              const float2* db, double* __restrict__ out) {
  pdl_begin();
  constexpr int W = kRedThreads / 32;
  __shared__ double red[3][W];
  const int b = blockIdx.x, lane = threadIdx.x & 31, w = threadIdx.x >> 5, half = nm / 2;
  const int slo = b * b + b + 1, shi = min((b + 1) * (b + 1) + (b + 1), 3 * half * half);
  double cnt = 0.0, ks = 0.0, ps = 0.0;
  // groups of 32 values of s; with fewer groups than warps, each is split over n_z (c(s) and
  // c(s) sqrt(s) add up)
  const int groups = (shi - slo + 32) / 32, split = shi < slo ? 1 : max(1, W / groups);
  for (int q = w; q < groups * split; q += W) {
    const int s = slo + 32 * (q % groups) + lane;
    uint32_t c = 0;  // below 2^32: at most the modes of one bin
    if (s <= shi) {
#pragma unroll 8
      for (int kz = q / groups; kz <= half; kz += split) {
        const int t = s - kz * kz;
        if (t < 0) break;
        if (t <= 2 * half * half) c += r2[t] * ((kz == 0 || kz == half) ? 1u : 2u);
      }
    }
    cnt += (double)c;
    if (c) ks += (double)c * sqrt((double)s);
  }
  cnt = warp_sum(cnt);
  ks = warp_sum(ks);
  for (int r = threadIdx.x; r < nrows; r += kRedThreads) ps += partial[(size_t)r * nbins + b];
  ps = warp_sum(ps);
  if (lane == 0) {
    red[0][w] = cnt;
    red[1][w] = ks;
    red[2][w] = ps;
  }
  __syncthreads();
  if (threadIdx.x != 0) return;
  double t[3] = {0.0, 0.0, 0.0};
  for (int q = 0; q < W; ++q)
    for (int d = 0; d < 3; ++d) t[d] += red[d][q];
  out[b] = t[0];
  out[nbins + b] = kf * t[1];
  if (nrows == 0) return;
  // delta_s = rho_s / mean_s: the k = 0 mode holds N^3 mean_s
  const float nn3 = (float)nm * (float)nm * (float)nm;
  const float ma = da[0].x / nn3, mb = db[0].x / nn3;
  const float scale = (ma != 0.0f && mb != 0.0f) ? norm / (ma * mb) : 0.0f;
  out[2 * nbins + b] = scale != 0.0f ? (double)scale * t[2] : 0.0;
}

// cw[b] = 2 dL_dP[b] V / (N^6 rho_bar^2 N_b), the weights of k_power_weight (0 for empty bins)
__global__ void k_power_cw(const double* counts, const double* dL, int nbins, double vol,
                           double n3, const float2* d, float* __restrict__ cw) {
  pdl_begin();
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= nbins) return;
  const double rho_bar = (double)d[0].x / n3, nb = counts[b];
  cw[b] = (rho_bar != 0.0 && nb > 0.0) ? (float)(2.0 * dL[b] * vol / (n3 * n3 * rho_bar * rho_bar * nb)) : 0.0f;
}

// d *= cw[b(n)] / W(k)^2 on the half spectrum (0 at k = 0 and beyond the last bin): the
// k-space cotangent of a binned auto-spectrum.  A warp takes one row (n_x, n_y).
__global__ void __launch_bounds__(kPowThreads) k_power_weight(float2* __restrict__ d, int nm, int pc, int nbins,
                                                              const float* __restrict__ winv,
                                                              const float* cw) {
  pdl_begin();
  const int lane = threadIdx.x & 31;
  const long long row = (long long)blockIdx.x * kPowWarps + (threadIdx.x >> 5);  // x N + y, N^2 rows in all
  const int x = (int)(row / nm), y = (int)(row % nm);
  const int nx = x < nm / 2 ? x : x - nm, ny = y < nm / 2 ? y : y - nm;
  const float wxy = __ldg(winv + x) * __ldg(winv + y);
  float2* const rp = d + row * pc;
  for (int kz = lane; kz <= nm / 2; kz += 32) {
    const int n2 = nx * nx + ny * ny + kz * kz;
    float w = 0.0f;
    if (n2 > 0) {
      const int b = bin_of(n2);
      if (b < nbins) w = cw[b] * wxy * __ldg(winv + kz);
    }
    rp[kz] = cscale(rp[kz], w);
  }
}

// Scratch: pk_partial holds N x 2 x 2048 doubles; partial rows (at most N, of nbins) come
// first, r2 (N^2 / 2 + 1 words) and the copy of dL_dP from N x 2048 doubles on.
struct PowerPlan {
  int units, tmax, rows;
  uint32_t* r2;
  double* dL;
};

PowerPlan power_plan(pm_ctx* c, int nbins) {
  const int N = c->g.n, half = N / 2;
  PowerPlan p;
  p.units = (half + 1) * (half + 2) / 2;
  p.tmax = (int)std::min<long long>(2LL * half * half, (long long)nbins * nbins + nbins);
  p.rows = std::min({N, kMaxRows, (p.units + kPowWarps - 1) / kPowWarps});
  p.dL = c->pk_partial + (size_t)N * kMaxBins;
  p.r2 = reinterpret_cast<uint32_t*>(p.dL + kMaxBins);
  return p;
}

}  // namespace

// Cotangent mesh of sum_b dL_dP[b] P_b (auto-spectrum of the half spectrum in meshA, in
// place): meshA <- c_k F_k, c_k = 2 dL_dP[b] V / (N^6 rho_bar^2 W_k^2 N_b).  dL_dP (host) is
// read before the call returns; the mode counts N_b need no pass over the mesh.
int power_weight(pm_ctx* c, int nbins, const double* dL_dP, cudaStream_t s) {
  if (nbins < 1 || nbins > kMaxBins) return PM_EINVAL;
  if (!c->pk_w && ctx_alloc_n(c, &c->pk_w, kMaxBins) != PM_OK) return PM_ENOMEM;
  const Geom& g = c->g;
  const PowerPlan p = power_plan(c, nbins);
  const double n3 = (double)g.n * g.n * g.n, kf = 2.0 * 3.14159265358979323846 / c->cfg.box;
  // from pageable memory: staged before the copy call returns
  PM_CUDA_TRY(cudaMemcpyAsync(p.dL, dL_dP, sizeof(double) * nbins, cudaMemcpyHostToDevice, s));
  PM_CUDA_TRY(cudaMemsetAsync(p.r2, 0, sizeof(uint32_t) * (p.tmax + 1), s));
  {
    LaunchScope L(c, s, K_POWER_BIN);
    pdl_launch(k_power_counts, (p.units + 255) / 256, 256, 0, s, g.n, p.units, p.tmax, p.r2);
  }
  {
    LaunchScope L(c, s, K_POWER_REDUCE);
    pdl_launch(k_power_reduce, nbins, kRedThreads, 0, s, nullptr, 0, nbins, g.n, p.r2, kf, 0.0f, nullptr, nullptr, c->pk_final);
  }
  {
    LaunchScope L(c, s, K_POWER_REDUCE);
    pdl_launch(k_power_cw, (nbins + 255) / 256, 256, 0, s, c->pk_final, p.dL, nbins, c->cfg.box * c->cfg.box * c->cfg.box, n3,
                                                   c->meshA, c->pk_w);
  }
  LaunchScope L(c, s, K_POWER_BIN);
  pdl_launch(k_power_weight, (unsigned)(g.rows() / kPowWarps), kPowThreads, 0, s, c->meshA, g.n, g.pc, nbins, c->winv, c->pk_w);
  return PM_OK;
}

int power_bin(pm_ctx* c, const float2* da, const float2* db, int nbins, double* k_out,
              double* P_out, int64_t* nmodes_out, cudaStream_t s) {
  if (nbins < 1 || nbins > kMaxBins) return PM_EINVAL;
  const Geom& g = c->g;
  const double nn = (double)g.n;
  const float norm = (float)(c->cfg.box * c->cfg.box * c->cfg.box / (nn * nn * nn * nn * nn * nn));
  const double kf = 2.0 * 3.14159265358979323846 / c->cfg.box;
  const PowerPlan p = power_plan(c, nbins);
  const size_t smem = sizeof(double) * kPowWarps * nbins;
  auto kern = da == db ? k_power_bin<false> : k_power_bin<true>;
  static DeviceOnce once[2];
  allow_smem(once[da == db], (const void*)kern, sizeof(double) * kPowWarps * kMaxBins);
  PM_CUDA_TRY(cudaMemsetAsync(p.r2, 0, sizeof(uint32_t) * (p.tmax + 1), s));
  {
    LaunchScope L(c, s, K_POWER_BIN);
    pdl_launch(kern, p.rows, kPowThreads, smem, s, da, db, g.n, g.pc, nbins, p.units, p.tmax, c->winv, c->pk_partial, p.r2);
  }
  {
    LaunchScope L(c, s, K_POWER_REDUCE);
    pdl_launch(k_power_reduce, nbins, kRedThreads, 0, s, c->pk_partial, p.rows, nbins, g.n, p.r2, kf, norm, da, db,
                                                 c->pk_final);
  }
  std::vector<double> h(3 * nbins);
  PM_CUDA_TRY(cudaMemcpyAsync(h.data(), c->pk_final, sizeof(double) * 3 * nbins,
                              cudaMemcpyDeviceToHost, s));
  PM_CUDA_TRY(cudaStreamSynchronize(s));
  for (int b = 0; b < nbins; ++b) {
    double cnt = h[b];
    nmodes_out[b] = (int64_t)cnt;
    k_out[b] = cnt > 0 ? h[nbins + b] / cnt : 0.0;
    P_out[b] = cnt > 0 ? h[2 * nbins + b] / cnt : 0.0;
  }
  return PM_OK;
}

}  // namespace pmnu
