// Adjoint (vector-Jacobian products) of the particle-mesh step, for gradients of a
// final-field loss with respect to the initial modes (reconstruction).
//
// * CIC readout gradient: d/dx sum_c W(x - c) M(c), with dw/dx = -+1/H per axis.
// * Paint transpose = readout; readout transpose = paint of per-particle weights
//   (the deterministic tile paint with signed weights).
// * Force VJP for a cotangent lambda_F (F_j = R[G_j rho], G_j real with an odd
//   kernel so G_j^T = -G_j):
//     dL/dx_i = sum_j lambda_F,ij grad R[G_j rho](x_i) + m_i grad R[B](x_i),
//     B_k = sum_j i D(k_j) g(k) FFT(paint(lambda_F,j))_k, D the gradient kernel.
//   With the 4-point kernel both terms run on one potential mesh each: G_j rho = -S_j phi,
//   and B = G * (sum_j S_j paint(lambda_F,j)).  With the learned factor the first term keeps
//   its three force meshes (the stencil of an FP32 potential would carry seven times their
//   rounding error), and the factor's gradient needs only the spectra of rho and of the
//   divergence (k_vjp_combine).
// * KDK step VJP (p_h = p0 + K1 F(x0), x1 = x0 + Delta p_h, p1 = p_h + K2 F(x1)).
// * Zel'dovich IC transpose: s_j = T_j omega with T_j = IFFT diag(S_j) FFT, so
//   dL/domega = IFFT(sum_j conj(S_j) FFT(lambda_s,j)), neutrino sites with the
//   conjugate phase.
// Cotangent arrays at the C-ABI are indexed by canonical particle id.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <vector>

#include "pm_internal.cuh"

namespace pmnu {

namespace {

// out[d][perm[i]] (+)= sum_j a_j(i) d/dx_d R[M_j](x_i) for the sorted particle i.
// a_j(i) = wts[j * n + i] when wts is set, else the particle's mass.
__global__ void k_readout_grad(const uint32_t* us, const uint32_t* ids,
                               int64_t n, const float* m0, const float* m1,
                               const float* m2, int nmesh_used, int nm, int shift,
                               int row_pitch, float inv_h, const float* wts, MassTable mt,
                               const uint32_t* perm, float* __restrict__ out,
                               int accumulate, int species) {
  pdl_begin();
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
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
  const float* ms[3] = {m0, m1, m2};
  bool bad = false;
  const float mass = wts ? 0.0f : id_mass(mt, ids[i], species, &bad);
  float o[3] = {0.f, 0.f, 0.f};
  for (int j = 0; j < nmesh_used; ++j) {
    const float* M = ms[j];
    const float a = wts ? wts[(int64_t)j * n + i] : mass;
    if (a == 0.0f) continue;
    const float v000 = M[r00 + cz], v001 = M[r00 + cz1];
    const float v010 = M[r01 + cz], v011 = M[r01 + cz1];
    const float v100 = M[r10 + cz], v101 = M[r10 + cz1];
    const float v110 = M[r11 + cz], v111 = M[r11 + cz1];
    // d/dx: (x1 plane - x0 plane) weighted in y, z; likewise for y and z
    const float dX = gy * (gz * (v100 - v000) + fz * (v101 - v001)) +
                     fy * (gz * (v110 - v010) + fz * (v111 - v011));
    const float dY = gx * (gz * (v010 - v000) + fz * (v011 - v001)) +
                     fx * (gz * (v110 - v100) + fz * (v111 - v101));
    const float dZ = gx * (gy * (v001 - v000) + fy * (v011 - v010)) +
                     fx * (gy * (v101 - v100) + fy * (v111 - v110));
    o[0] += a * dX;
    o[1] += a * dY;
    o[2] += a * dZ;
  }
  const int64_t dst = perm ? (int64_t)perm[i] : i;
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const float v = o[d] * inv_h;
    if (accumulate)
      out[(int64_t)d * n + dst] += v;
    else
      out[(int64_t)d * n + dst] = v;
  }
}

// B_k (+)= i D(k_j) g(k) m(k) A_k on the half spectrum (padded pitch pc), the transpose
// of -G_j (D the gradient kernel); m = 1 without the learned factor.  With rho (the
// density's half spectrum) it also bins d <lambda_F, F> / d m(k) =
// Re[(-i D(k_j)) g rho_k conj(A_k)] (twice for 0 < k_z < N/2) by s = |n|^2 into gbin.
__global__ void k_adj_combine(const float2* a, float2* __restrict__ b, int nm, int pc,
                              const float* __restrict__ ksq, const float* __restrict__ winv,
                              const float* __restrict__ kvec0, float gcoef, int comp, int accumulate,
                              const float* mtab, const float2* rho,
                              double* __restrict__ gbin) {
  pdl_begin();
  const int x = blockIdx.x / nm, y = blockIdx.x % nm;
  const int nx = x < nm / 2 ? x : x - nm, ny = y < nm / 2 ? y : y - nm;
  for (int kz = threadIdx.x; kz <= nm / 2; kz += blockDim.x) {
    const size_t idx = ((size_t)x * nm + y) * pc + kz;
    const int sidx = nx * nx + ny * ny + kz * kz;
    const float k2 = ksq[x] + ksq[y] + ksq[kz];
    float g = gcoef * winv[x] * winv[y] * winv[kz] / k2;
    if (k2 == 0.0f) g = 0.0f;
    const float kj = comp == 0 ? kvec0[x] : (comp == 1 ? kvec0[y] : kvec0[kz]);
    const float2 v = a[idx];
    if (rho) {
      const float2 r = rho[idx];
      const float mult = (kz > 0 && kz < nm / 2) ? 2.0f : 1.0f;
      const float q = mult * kj * g * (r.y * v.x - r.x * v.y);
      if (q != 0.0f) atomicAdd(gbin + sidx, (double)q);
    }
    const float s = kj * (mtab ? g * mtab[sidx] : g);
    const float2 r = make_float2(-s * v.y, s * v.x);  // i s v
    if (accumulate) {
      float2 o = b[idx];
      b[idx] = make_float2(o.x + r.x, o.y + r.y);
    } else {
      b[idx] = r;
    }
  }
}

// ---- one-mesh force VJP (4-point kernel): the forward force is F_j = -S_j phi with S_j
// the 4-point stencil along axis j (transfer function i D(k_j)), so
//   term 1: sum_j lambda_j grad R[F_j] from the potential staged per tile, and
//   term 2: B = G * (sum_j S_j paint(lambda_j)) (IFFT[g sum_j i D(k_j) FFT(paint_j)]).
constexpr int kVjpSpanXY = kTile + 5;  // cells -2 .. 18 along x and y
constexpr int kVjpSpanZ = kTile + 8;   // cells -4 .. 19 along z (16-byte aligned rows)
constexpr int kVjpChunksZ = kVjpSpanZ / 4;
constexpr int kVjpStage = kVjpSpanXY * kVjpSpanXY * kVjpChunksZ;
constexpr int kVjpSY = kVjpSpanZ, kVjpSX = kVjpSpanXY * kVjpSpanZ;

__device__ __forceinline__ void vjp_cp_async16(void* smem_dst, const void* gmem_src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(smem_dst)),
               "l"(gmem_src)
               : "memory");
}

// Both terms of the force VJP in one pass over the sorted particles, one CTA per tile:
//   out[d][perm[i]] = sum_j lambda_j(i) d/dx_d R[F_j](x_i) + m_i d/dx_d R[B](x_i),  F_j = -S_j phi.
// The tile's potential with the stencil halo is staged like the forward readout's, B with the
// halo of the CIC corners; F_j at the particle's 8 corners comes from 56 values of phi, then
// the CIC weight derivatives.  Bound by the shared-memory pipe (56 + 8 random gathers a
// particle); a separate pass over B gathered 8 values from global memory and updated the
// gradient a second time (step_vjp at 256^3: 124 us a force).
constexpr long long kStagedMin = 200;                  // mean particles a tile, see readout_grad
constexpr int kVjpSpanB = kTile + 1;                   // cells 0 .. 16 along x and y
constexpr int kVjpSpanBZ = kTile + 4;                  // cells 0 .. 19 along z
constexpr int kVjpStageB = kVjpSpanB * kVjpSpanB * (kVjpSpanBZ / 4);
constexpr int kVjpBSY = kVjpSpanBZ, kVjpBSX = kVjpSpanB * kVjpSpanBZ;
constexpr size_t kVjpSmem = sizeof(float) * (kVjpSpanXY * kVjpSX + kVjpSpanB * kVjpBSX);

template <int NT>
__global__ void __launch_bounds__(NT) k_force_vjp_readout(
    const uint32_t* us, const uint32_t* ids, int64_t n, const uint32_t* bstart,
    const float* phi, const float* B, int nm, int shift, int ntl, int row_pitch,
    float inv12h, float inv_h, const float* lam, MassTable mt, const uint32_t* perm,
    float* __restrict__ out, int* __restrict__ err) {
  pdl_begin();
  extern __shared__ __align__(16) float sp[];
  float* const sb = sp + kVjpSpanXY * kVjpSX;
  const int t = threadIdx.x;
  const uint32_t tile = blockIdx.x;
  const uint32_t lo = bstart[8 * tile], hi = bstart[8 * tile + 8];
  if (lo == hi) return;
  const int nt = 1 << ntl;
  const int ox = (int)(tile >> (2 * ntl)) * kTile, oy = (int)((tile >> ntl) & (nt - 1)) * kTile,
            oz = (int)(tile & (nt - 1)) * kTile;
  const int wrap = nm - 1;
  for (int c = t; c < kVjpStage; c += NT) {
    const int x = c / (kVjpSpanXY * kVjpChunksZ), r = c - x * (kVjpSpanXY * kVjpChunksZ);
    const int y = r / kVjpChunksZ, k = r - y * kVjpChunksZ;
    const int gx = (ox + x - 2) & wrap, gy = (oy + y - 2) & wrap, gz = (oz - 4 + 4 * k) & wrap;
    vjp_cp_async16(sp + x * kVjpSX + y * kVjpSY + 4 * k, phi + ((size_t)gx * nm + gy) * (size_t)row_pitch + gz);
  }
  for (int c = t; c < kVjpStageB; c += NT) {
    const int x = c / (kVjpSpanB * (kVjpSpanBZ / 4)), r = c - x * (kVjpSpanB * (kVjpSpanBZ / 4));
    const int y = r / (kVjpSpanBZ / 4), k = r - y * (kVjpSpanBZ / 4);
    const int gx = (ox + x) & wrap, gy = (oy + y) & wrap, gz = (oz + 4 * k) & wrap;
    vjp_cp_async16(sb + x * kVjpBSX + y * kVjpBSY + 4 * k, B + ((size_t)gx * nm + gy) * (size_t)row_pitch + gz);
  }
  asm volatile("cp.async.commit_group;" ::: "memory");
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncthreads();
  const float fscale = 1.0f / (float)(1u << shift);
  const uint32_t fmask = (1u << shift) - 1u;
  bool bad = false;
  for (uint32_t i = lo + t; i < hi; i += NT) {
    const uint32_t ux = us[i], uy = us[n + i], uz = us[2 * n + i];
    const int lx = (int)(ux >> shift) - ox, ly = (int)(uy >> shift) - oy, lz = (int)(uz >> shift) - oz;
    if ((unsigned)lx >= (unsigned)kTile || (unsigned)ly >= (unsigned)kTile || (unsigned)lz >= (unsigned)kTile) {
      bad = true;
      continue;
    }
    const float fx = (float)(ux & fmask) * fscale, fy = (float)(uy & fmask) * fscale,
                fz = (float)(uz & fmask) * fscale;
    const float gx = 1.0f - fx, gy = 1.0f - fy, gz = 1.0f - fz;
    // CIC derivative of corner values v[a][b][c]
    auto grad = [&](const float (*v)[2][2], float& dX, float& dY, float& dZ) {
      dX = gy * (gz * (v[1][0][0] - v[0][0][0]) + fz * (v[1][0][1] - v[0][0][1])) +
           fy * (gz * (v[1][1][0] - v[0][1][0]) + fz * (v[1][1][1] - v[0][1][1]));
      dY = gx * (gz * (v[0][1][0] - v[0][0][0]) + fz * (v[0][1][1] - v[0][0][1])) +
           fx * (gz * (v[1][1][0] - v[1][0][0]) + fz * (v[1][1][1] - v[1][0][1]));
      dZ = gx * (gy * (v[0][0][1] - v[0][0][0]) + fy * (v[0][1][1] - v[0][1][0])) +
           fx * (gy * (v[1][0][1] - v[1][0][0]) + fy * (v[1][1][1] - v[1][1][0]));
    };
    const float* q = sp + (lx + 2) * kVjpSX + (ly + 2) * kVjpSY + (lz + 4);
    // F_j at corner (a, b, c) of the cell, Fj[a][b][c] = -S_j phi / ... (scaled below)
    float Fx[2][2][2], Fy[2][2][2], Fz[2][2][2];
    auto line = [](const float* q0, int S, float& c0, float& c1) {  // stencil sums at corners 0, 1
      const float m2 = q0[-2 * S], m1 = q0[-S], p0 = q0[0], p1 = q0[S], p2 = q0[2 * S], p3 = q0[3 * S];
      c0 = 8.0f * (p1 - m1) - (p2 - m2);
      c1 = 8.0f * (p2 - p0) - (p3 - m1);
    };
#pragma unroll
    for (int a = 0; a < 2; ++a) {
#pragma unroll
      for (int b = 0; b < 2; ++b) {
        line(q + a * kVjpSY + b, kVjpSX, Fx[0][a][b], Fx[1][a][b]);  // x line at (y, z) = (a, b)
        line(q + a * kVjpSX + b, kVjpSY, Fy[a][0][b], Fy[a][1][b]);  // y line at (x, z) = (a, b)
        line(q + a * kVjpSX + b * kVjpSY, 1, Fz[a][b][0], Fz[a][b][1]);  // z line at (x, y) = (a, b)
      }
    }
    float o[3] = {0.f, 0.f, 0.f};
    const float (*Fs[3])[2][2] = {Fx, Fy, Fz};
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      float dX, dY, dZ;
      grad(Fs[j], dX, dY, dZ);
      const float lj = lam[(int64_t)j * n + i];
      o[0] += lj * dX;
      o[1] += lj * dY;
      o[2] += lj * dZ;
    }
    const float* qb = sb + lx * kVjpBSX + ly * kVjpBSY + lz;
    float vb[2][2][2], bX, bY, bZ;
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
      for (int b = 0; b < 2; ++b)
#pragma unroll
        for (int c = 0; c < 2; ++c) vb[a][b][c] = qb[a * kVjpBSX + b * kVjpBSY + c];
    grad(vb, bX, bY, bZ);
    const float m = id_mass(mt, ids[i], PM_SPECIES_ALL, &bad) * inv_h;
    const int64_t dst = perm ? (int64_t)perm[i] : (int64_t)i;
    const float scale = -inv12h * inv_h;  // F_j = -(stencil sum) / (12 H); d/dx: 1 / H
    out[dst] = fmaf(scale, o[0], m * bX);
    out[n + dst] = fmaf(scale, o[1], m * bY);
    out[2 * n + dst] = fmaf(scale, o[2], m * bZ);
  }
  if (bad) atomicOr(err, 1);
}

// One mesh's or three meshes' worth of the VJP, staged per tile like B above (the learned path):
// NM = 1: m_i d/dx_d R[B](x_i), m_i the mass if the species is selected, to out[d][perm[i]] or
// (perm null) in sorted order to tmp[d][i]; NM = 3: out[d][perm[i]] = tmp[d][i] + sum_j lambda_j(i)
// d/dx_d R[F_j](x_i).  Staging replaces 8 NM scattered global reads a particle.
template <int NM, int NT>
__global__ void __launch_bounds__(NT) k_vjp_readout(
    const uint32_t* us, const uint32_t* ids, int64_t n, const uint32_t* bstart,
    const float* m0, const float* m1, const float* m2, int nm, int shift,
    int ntl, int row_pitch, float inv_h, const float* lam, MassTable mt,
    const uint32_t* perm, float* __restrict__ tmp, float* __restrict__ out, int species,
    int* __restrict__ err) {
  pdl_begin();
  extern __shared__ __align__(16) float sb[];
  const int t = threadIdx.x;
  const uint32_t tile = blockIdx.x;
  const uint32_t lo = bstart[8 * tile], hi = bstart[8 * tile + 8];
  if (lo == hi) return;
  const int nt = 1 << ntl;
  const int ox = (int)(tile >> (2 * ntl)) * kTile, oy = (int)((tile >> ntl) & (nt - 1)) * kTile,
            oz = (int)(tile & (nt - 1)) * kTile;
  const int wrap = nm - 1;
#pragma unroll
  for (int j = 0; j < NM; ++j) {
    const float* const M = j == 0 ? m0 : (j == 1 ? m1 : m2);
    float* const dst = sb + j * kVjpSpanB * kVjpBSX;
    for (int c = t; c < kVjpStageB; c += NT) {
      const int x = c / (kVjpSpanB * (kVjpSpanBZ / 4)), r = c - x * (kVjpSpanB * (kVjpSpanBZ / 4));
      const int y = r / (kVjpSpanBZ / 4), k = r - y * (kVjpSpanBZ / 4);
      const int gx = (ox + x) & wrap, gy = (oy + y) & wrap, gz = (oz + 4 * k) & wrap;
      vjp_cp_async16(dst + x * kVjpBSX + y * kVjpBSY + 4 * k, M + ((size_t)gx * nm + gy) * (size_t)row_pitch + gz);
    }
  }
  asm volatile("cp.async.commit_group;" ::: "memory");
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncthreads();
  const float fscale = 1.0f / (float)(1u << shift);
  const uint32_t fmask = (1u << shift) - 1u;
  bool bad = false;
  for (uint32_t i = lo + t; i < hi; i += NT) {
    const uint32_t ux = us[i], uy = us[n + i], uz = us[2 * n + i];
    const int lx = (int)(ux >> shift) - ox, ly = (int)(uy >> shift) - oy, lz = (int)(uz >> shift) - oz;
    if ((unsigned)lx >= (unsigned)kTile || (unsigned)ly >= (unsigned)kTile || (unsigned)lz >= (unsigned)kTile) {
      bad = true;
      continue;
    }
    const float fx = (float)(ux & fmask) * fscale, fy = (float)(uy & fmask) * fscale,
                fz = (float)(uz & fmask) * fscale;
    const float gx = 1.0f - fx, gy = 1.0f - fy, gz = 1.0f - fz;
    float o[3] = {0.f, 0.f, 0.f};
#pragma unroll
    for (int j = 0; j < NM; ++j) {
      const float a = NM == 1 ? id_mass(mt, ids[i], species, &bad) : lam[(int64_t)j * n + i];
      const float* const q = sb + j * kVjpSpanB * kVjpBSX + lx * kVjpBSX + ly * kVjpBSY + lz;
      const float v000 = q[0], v001 = q[1], v010 = q[kVjpBSY], v011 = q[kVjpBSY + 1];
      const float v100 = q[kVjpBSX], v101 = q[kVjpBSX + 1], v110 = q[kVjpBSX + kVjpBSY],
                  v111 = q[kVjpBSX + kVjpBSY + 1];
      const float dX = gy * (gz * (v100 - v000) + fz * (v101 - v001)) +
                       fy * (gz * (v110 - v010) + fz * (v111 - v011));
      const float dY = gx * (gz * (v010 - v000) + fz * (v011 - v001)) +
                       fx * (gz * (v110 - v100) + fz * (v111 - v101));
      const float dZ = gx * (gy * (v001 - v000) + fy * (v011 - v010)) +
                       fx * (gy * (v101 - v100) + fy * (v111 - v110));
      if (NM == 3 || a != 0.0f) {  // a masked species takes nothing from the mesh, whatever it holds
        o[0] += a * dX;
        o[1] += a * dY;
        o[2] += a * dZ;
      }
    }
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      const int64_t k = (int64_t)d * n + i;
      if constexpr (NM == 1) {
        if (perm)
          out[(int64_t)d * n + perm[i]] = o[d] * inv_h;
        else
          tmp[k] = o[d] * inv_h;
      } else {
        out[(int64_t)d * n + perm[i]] = fmaf(o[d], inv_h, tmp[k]);
      }
    }
  }
  if (bad) atomicOr(err, 1);
}

// C <- S_x A + S_y B + S_z C on real meshes (row pitch rp): the divergence of the painted
// cotangents with the 4-point stencil, periodic, in place on the third.  A thread takes four
// cells along z and walks kDivSteps planes along x with the five A values it needs in
// registers; its CTA holds whole rows of C, read before any is written.  One pass over the
// three meshes: three single-axis passes that add into one mesh took 307 us at 256^3.
constexpr int kDivThreads = 256;
constexpr int kDivSteps = 8;
__global__ void __launch_bounds__(kDivThreads) k_stencil_div(const float* A, const float* B,
                                                             float* C, int nm, int rp, float inv12h) {
  pdl_begin();
  const int quads = nm / 4, rows = kDivThreads / quads;  // rows of z quads a CTA (nm <= 1024)
  const int q = threadIdx.x % quads, z = 4 * q, w = nm - 1;
  const int y = (blockIdx.x % (nm / rows)) * rows + threadIdx.x / quads;
  const int x0 = (blockIdx.x / (nm / rows)) * kDivSteps;
  auto at = [&](const float* M, int x, int yy, int zz) -> float4 {
    return *reinterpret_cast<const float4*>(M + ((size_t)(x & w) * nm + (yy & w)) * rp + (zz & w));
  };
  float4 a[5];  // A at x - 2 .. x + 2
#pragma unroll
  for (int k = 0; k < 4; ++k) a[k + 1] = at(A, x0 - 2 + k, y, z);
  for (int s = 0; s < kDivSteps; ++s) {
    const int x = x0 + s;
#pragma unroll
    for (int k = 0; k < 4; ++k) a[k] = a[k + 1];
    a[4] = at(A, x + 2, y, z);
    const float4 b0 = at(B, x, y - 2, z), b1 = at(B, x, y - 1, z), b3 = at(B, x, y + 1, z), b4 = at(B, x, y + 2, z);
    const float4 c0 = at(C, x, y, z - 4), c1 = at(C, x, y, z), c2 = at(C, x, y, z + 4);
    auto st = [](float m2, float m1, float p1, float p2) { return 8.0f * (p1 - m1) - (p2 - m2); };
    float4 r;
    r.x = st(a[0].x, a[1].x, a[3].x, a[4].x) + st(b0.x, b1.x, b3.x, b4.x) + st(c0.z, c0.w, c1.y, c1.z);
    r.y = st(a[0].y, a[1].y, a[3].y, a[4].y) + st(b0.y, b1.y, b3.y, b4.y) + st(c0.w, c1.x, c1.z, c1.w);
    r.z = st(a[0].z, a[1].z, a[3].z, a[4].z) + st(b0.z, b1.z, b3.z, b4.z) + st(c1.x, c1.y, c1.w, c2.x);
    r.w = st(a[0].w, a[1].w, a[3].w, a[4].w) + st(b0.w, b1.w, b3.w, b4.w) + st(c1.y, c1.z, c2.x, c2.y);
    __syncthreads();  // the row's C values are read
    *reinterpret_cast<float4*>(C + ((size_t)x * nm + y) * rp + z) =
        make_float4(inv12h * r.x, inv12h * r.y, inv12h * r.z, inv12h * r.w);
  }
}

// The same divergence from the three half spectra, C <- i (D_x A + D_y B + D_z C): the learned
// path's form.  The factor's gradient weighs the largest scales by 1 / k^2, and there the
// transform of the real-space divergence has lost digits to its smallest scales.
__global__ void __launch_bounds__(256) k_spectrum_div(const float2* A, const float2* B,
                                                      float2* __restrict__ C, int nm, int pc,
                                                      const float* __restrict__ kvec0) {
  pdl_begin();
  const long long row = (long long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);  // x N + y: a warp a row
  const float kx = __ldg(kvec0 + row / nm), ky = __ldg(kvec0 + row % nm);
  for (int kz = threadIdx.x & 31; kz <= nm / 2; kz += 32) {
    const size_t i = (size_t)row * pc + kz;
    const float kq = __ldg(kvec0 + kz);
    const float2 a = A[i], b = B[i], c = C[i];
    C[i] = make_float2(-(kx * a.y + ky * b.y + kq * c.y), kx * a.x + ky * b.x + kq * c.x);
  }
}

// The learned factor's part of the force VJP between the transforms: rho (the density's half
// spectrum) and C = FFT(sum_j S_j paint(lambda_j)) become the spectra of the two potentials,
// rho <- g m rho, C <- g m C, and d <lambda_F, F> / d m(k) = g Re[rho_k conj(C_k)] (twice for
// 0 < k_z < N/2) is added to gbin by s = |n|^2.  The rows (+-n_x, +-n_y), (+-n_y, +-n_x) share
// g, m and s: a warp takes all of them, its lanes walk k_z, and one FP64 atomic serves eight
// modes (their products added error-free in FP32 pairs).
__global__ void __launch_bounds__(256) k_vjp_combine(float2* __restrict__ rho, float2* __restrict__ C, int nm, int pc,
                                                     int units, const float* __restrict__ ksq,
                                                     const float* __restrict__ winv, float gcoef,
                                                     const float* mtab, double* __restrict__ gbin) {
  pdl_begin();
  const int wu = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), lane = threadIdx.x & 31, half = nm / 2;
  if (wu >= units) return;
  int a = (int)((sqrtf(8.0f * (float)wu + 1.0f) - 1.0f) * 0.5f);  // (a, b), 0 <= b <= a <= N/2
  while (a * (a + 1) / 2 > wu) --a;
  while ((a + 1) * (a + 2) / 2 <= wu) ++a;
  const int b = wu - a * (a + 1) / 2;
  const bool ra = a != 0 && a != half, rb = b != 0 && b != half, rs = a != b;
  const float kab = ksq[a] + ksq[b], wab = winv[a] * winv[b];
  for (int kz = lane; kz <= half; kz += 32) {
    const int s = a * a + b * b + kz * kz;
    const float k2 = kab + ksq[kz];
    const float g = k2 == 0.0f ? 0.0f : gcoef * wab * winv[kz] / k2;
    const float gm = g * mtab[s];
    float sum = 0.0f, e = 0.0f;
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      if (((r & 1) && !ra) || ((r & 2) && !rb) || ((r & 4) && !rs)) continue;
      const int ia = (r & 1) ? nm - a : a, ib = (r & 2) ? nm - b : b;
      const size_t idx = ((size_t)((r & 4) ? ib : ia) * nm + ((r & 4) ? ia : ib)) * pc + kz;
      const float2 v = rho[idx], c = C[idx];
      const float p = v.x * c.x + v.y * c.y;
      const float t = sum + p, d = t - sum;  // Knuth's two-sum
      e += (sum - (t - d)) + (p - d);
      sum = t;
      rho[idx] = cscale(v, gm);
      C[idx] = cscale(c, gm);
    }
    const float q = ((kz > 0 && kz < half) ? 2.0f : 1.0f) * g;
    if (q != 0.0f) atomicAdd(gbin + s, (double)q * ((double)sum + (isfinite(sum) ? (double)e : 0.0)));
  }
}

// B (+)= S_j A on real meshes (row pitch rp): the 4-point stencil along axis j, periodic.
__global__ void k_stencil_axis(const float* A, float* __restrict__ B, int nm, int rp, int axis,
                               float inv12h, int accumulate) {
  pdl_begin();
  const int x = blockIdx.x / nm, y = blockIdx.x % nm;
  const int w = nm - 1;
  const size_t row = ((size_t)x * nm + y) * rp;
  for (int z = threadIdx.x; z < nm; z += blockDim.x) {
    auto at = [&](int o) -> float {  // A at offset o along the axis
      if (axis == 0) return A[((size_t)((x + o) & w) * nm + y) * rp + z];
      if (axis == 1) return A[((size_t)x * nm + ((y + o) & w)) * rp + z];
      return A[row + ((z + o) & w)];
    };
    const float v = inv12h * (8.0f * (at(1) - at(-1)) - (at(2) - at(-2)));
    B[row + z] = accumulate ? B[row + z] + v : v;
  }
}

// Start of a step's VJP, in state order: the cotangents by id, the drifted positions
// u1 = u0 + rne(Delta (p0 + K1 f0) 2^32 / L) and the force cotangent K2 lambda_p of x1.
__global__ void k_vjp_begin(const float* lx1, const float* lp1,
                            const uint32_t* id, const uint32_t* u0,
                            const float* p0, const float* f0, int64_t n, float K1,
                            float dscale, float K2, float* __restrict__ Lx, float* __restrict__ Lp,
                            float* __restrict__ lamF, uint32_t* __restrict__ u1) {
  pdl_begin();
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int64_t j = (int64_t)id[i];
  float lx[3], lp[3], ph[3];  // every load before the first store
  uint32_t uq[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    lx[d] = lx1[d * n + j];
    lp[d] = lp1[d * n + j];
    ph[d] = p0[d * n + i] + K1 * f0[d * n + i];
    uq[d] = u0[d * n + i];
  }
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    Lx[d * n + i] = lx[d];
    Lp[d * n + i] = lp[d];
    lamF[d * n + i] = K2 * lp[d];
    u1[d * n + i] = uq[d] + (uint32_t)(unsigned long long)__float2ll_rn(dscale * ph[d]);
  }
}

// Between the two force VJPs, over 3n: Lx += g, Lp += Delta Lx, lamF = K1 Lp.
__global__ void k_vjp_middle(const float* g, int64_t m, float delta, float K1, float* __restrict__ Lx,
                             float* __restrict__ Lp, float* __restrict__ lamF) {
  pdl_begin();
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= m) return;
  const float x = Lx[i] + g[i], p = fmaf(delta, x, Lp[i]);
  Lx[i] = x;
  Lp[i] = p;
  lamF[i] = K1 * p;
}

// End: lx0 = Lx + g and lp0 = Lp in canonical order.
__global__ void k_vjp_end(const float* g, const float* Lx, const float* Lp,
                          const uint32_t* id, int64_t n, float* __restrict__ lx0,
                          float* __restrict__ lp0) {
  pdl_begin();
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int64_t j = (int64_t)id[i];
  float x[3], p[3];  // every load before the first store
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    x[d] = Lx[d * n + i] + g[d * n + i];
    p[d] = Lp[d * n + i];
  }
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    lx0[d * n + j] = x[d];
    lp0[d * n + j] = p[d];
  }
}

// gather weights into the sorted order: ws[k] = w[perm[k]]
__global__ void k_gather_weights(const float* w, const uint32_t* perm, int64_t n,
                                 float* __restrict__ ws) {
  pdl_begin();
  const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k < n) ws[k] = w[perm[k]];
}

// IC transpose: lattice mesh (padded real, nc) of lambda_s for CDM nodes (canonical order)
__global__ void k_icadj_cdm(const float* lx, const float* lp, int nc,
                            int rp, int comp, float D0, float gp0, int64_t n_total,
                            float* __restrict__ mesh) {
  pdl_begin();
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t ncell = (int64_t)nc * nc * nc;
  if (i >= ncell) return;
  const int ix = (int)(i / ((int64_t)nc * nc)), iy = (int)((i / nc) % nc), iz = (int)(i % nc);
  mesh[((size_t)ix * nc + iy) * rp + iz] =
      D0 * lx[comp * n_total + i] + gp0 * lp[comp * n_total + i];
}

// neutrino sites: sum of lambda_s over the site's shell x direction particles
__global__ void k_icadj_nu(const float* lx, const float* lp, int nc,
                           int rp, int comp, float D0, float gp0, int nsites, int stride, int j0,
                           int per_site, int64_t n_offset, int64_t n_total, float* __restrict__ mesh) {
  pdl_begin();
  const int64_t site = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t nsite3 = (int64_t)nsites * nsites * nsites;
  if (site >= nsite3) return;
  float s = 0.f;
  for (int q = 0; q < per_site; ++q) {
    const int64_t i = n_offset + site * per_site + q;
    s += D0 * lx[comp * n_total + i] + gp0 * lp[comp * n_total + i];
  }
  const int sx = (int)(site / ((int64_t)nsites * nsites)), sy = (int)((site / nsites) % nsites),
            sz = (int)(site % nsites);
  const int ix = (j0 + stride * sx) % nc, iy = (j0 + stride * sy) % nc, iz = (j0 + stride * sz) % nc;
  mesh[((size_t)ix * nc + iy) * rp + iz] = s;
}

// K (+)= conj(S_j) A_k with S_j = i f e^{i theta}, f = amp(|n|^2) n_j / |n|^2 (the forward
// ZA multiplier of k_ic_za), theta = pi (n_x + n_y + n_z) / nc for shifted sites.
__global__ void k_icadj_kspace(const float2* a, float2* __restrict__ kacc, int nc, int pc,
                               const float* __restrict__ amp, int comp, int phase_shift,
                               int accumulate) {
  pdl_begin();
  const int x = blockIdx.x / nc, y = blockIdx.x % nc;
  const int nx = x < nc / 2 ? x : x - nc, ny = y < nc / 2 ? y : y - nc;
  for (int kz = threadIdx.x; kz <= nc / 2; kz += blockDim.x) {
    const size_t idx = ((size_t)x * nc + y) * pc + kz;
    const long long n2 = (long long)nx * nx + (long long)ny * ny + (long long)kz * kz;
    float2 r = make_float2(0.f, 0.f);
    const bool nyq = (x == nc / 2) || (y == nc / 2) || (kz == nc / 2);
    if (n2 > 0 && !nyq) {
      const int nj = comp == 0 ? nx : (comp == 1 ? ny : kz);
      const float f = __ldg(amp + n2) * (float)nj / (float)n2;
      float2 cs = make_float2(0.f, -f);  // conj(i f) = -i f
      if (phase_shift) {
        float sn, co;
        sincospif((float)(nx + ny + kz) / (float)nc, &sn, &co);
        cs = cmul(cs, make_float2(co, -sn));  // conj(e^{i theta})
      }
      r = cmul(cs, a[idx]);
    }
    if (accumulate) {
      const float2 o = kacc[idx];
      kacc[idx] = make_float2(o.x + r.x, o.y + r.y);
    } else {
      kacc[idx] = r;
    }
  }
}

int ensure_adj(pm_ctx* c, int64_t n) {
  if (n <= c->adj_cap) return PM_OK;
  ctx_free(c, c->adj);
  c->adj = nullptr;
  c->adj_cap = 0;
  if (ctx_alloc_n(c, &c->adj, 8 * 3 * (size_t)std::max<int64_t>(n, 1)) != PM_OK) return PM_ENOMEM;
  c->adj_cap = n;
  return PM_OK;
}

unsigned blocks(int64_t n) { return (unsigned)((n + 255) / 256); }

// Threads a tile of the staged VJP readouts: 512 where tiles are full (us a launch of the
// potentials' readout, 256 / 512 threads: 2000 a tile at 128^3 71 / 60, at 256^3 310 / 293; 580 a
// tile 35 / 36 and 126 / 139).
int vjp_threads(const pm_ctx* c, int64_t n) { return n >= 1000LL * c->nt * c->nt * c->nt ? 512 : 256; }

}  // namespace

int gather_weights(pm_ctx* c, const float* w, int64_t n, float* w_sorted, cudaStream_t s) {
  if (n == 0) return PM_OK;
  LaunchScope L(c, s, K_ADJOINT);
  pdl_launch(k_gather_weights, blocks(n), 256, 0, s, w, c->vals[0], n, w_sorted);
  return PM_OK;
}

// Readout gradient of up to three padded meshes at the sorted scratch particles
void readout_grad(pm_ctx* c, int64_t n, const float* const* meshes, int nmeshes, int row_pitch,
                  const float* wts_sorted, const uint32_t* perm, float* out, bool accumulate,
                  cudaStream_t s, int species) {
  if (n == 0) return;
  LaunchScope L(c, s, K_ADJOINT);
  const float inv_h = (float)(c->g.n / c->cfg.box);
  const long long tiles = (long long)c->nt * c->nt * c->nt;
  // one mesh and the particles' masses: staged per tile where the tiles hold enough particles to
  // pay for it, and the mesh takes 16-byte copies (rows are whole 16-byte groups).  us, gathered /
  // staged, by mean particles a tile: 256^3 128 21 / 23, 256 36 / 32, 580 75 / 55; 512^3 128
  // 150 / 169, 256 257 / 228, 580 576 / 456.
  if (nmeshes == 1 && !wts_sorted && !accumulate && perm && (reinterpret_cast<uintptr_t>(meshes[0]) & 15) == 0 &&
      n >= kStagedMin * tiles) {
    const int threads = vjp_threads(c, n);
    auto kern = threads == 512 ? k_vjp_readout<1, 512> : k_vjp_readout<1, 256>;
    pdl_launch(kern, (unsigned)tiles, threads, sizeof(float) * kVjpSpanB * kVjpBSX, s, c->us, c->ids, n, c->bstart,
               meshes[0], nullptr, nullptr, c->g.n, 32 - c->g.logn, c->ntl, row_pitch, inv_h, nullptr, c->mt, perm,
               nullptr, out, species, c->err_dev);
    return;
  }
  pdl_launch(k_readout_grad, blocks(n), 256, 0, s, c->us, c->ids, n, meshes[0], nmeshes > 1 ? meshes[1] : nullptr,
                                           nmeshes > 2 ? meshes[2] : nullptr, nmeshes, c->g.n,
                                           32 - c->g.logn, row_pitch, inv_h, wts_sorted, c->mt, perm,
                                           out, accumulate ? 1 : 0, species);
}

// Force VJP: u (any order, with id), cotangent lam_f[3n] in the same order -> grad[3n].
// With the learned factor (evaluated at scale factor a) it also accumulates
// d <lam_f, F> / d theta; that needs the third mesh, which holds rho_k meanwhile.
int force_vjp(pm_ctx* c, const uint32_t* u, const uint32_t* id, int64_t n, const float* lam_f,
              double a, float* grad, cudaStream_t s) {
  if (n == 0) return PM_OK;
  const bool learned = c->mlp_on;
  if (learned && !c->meshC) return PM_EINVAL;
  int rc = ensure_adj(c, n);
  if (rc != PM_OK) return rc;
  rc = sort_particles(c, u, n, s);
  if (rc != PM_OK) return rc;
  // the cotangents travel with the particles, where the momenta of a step do
  gather_sorted(c, u, lam_f, id, n, c->vals[0], s);
  const float* lam_s = c->ps;  // sorted cotangent, 3n
  float* realA = reinterpret_cast<float*>(c->meshA);
  float* realB = reinterpret_cast<float*>(c->meshB);
  const int rp = 2 * c->g.pc;
  if ((c->cfg.flags & (PM_FLAG_SPECTRAL_KERNEL | PM_FLAG_KSPACE_GRADIENT)) == 0) {
    // two potentials, phi in realA and B in pot (see k_force_vjp_readout)
    const float inv12h = (float)((double)c->g.n / (12.0 * c->cfg.box));
    const float inv_h = (float)(c->g.n / c->cfg.box);
    float2* const pot = c->meshC ? c->meshC : c->meshB;
    float* const realP = reinterpret_cast<float*>(pot);
    if (c->meshC) {
      paint_weights3(c, c->us, n, lam_s, realA, realB, realP, rp, s);
      if (learned) {
        fft_forward(c, c->g, c->meshA, c->meshA, 0, s);
        fft_forward(c, c->g, c->meshB, c->meshB, 0, s);
        fft_forward(c, c->g, pot, pot, 0, s);
      }
      LaunchScope L(c, s, K_ADJOINT);
      const int rows = kDivThreads / (c->g.n / 4);
      if (learned)
        pdl_launch(k_spectrum_div, (unsigned)(c->g.rows() / 8), 256, 0, s, c->meshA, c->meshB, pot, c->g.n, c->g.pc, c->kvec0);
      else
        pdl_launch(k_stencil_div, (unsigned)(c->g.n / rows * (c->g.n / kDivSteps)), kDivThreads, 0, s, 
            realA, realB, realP, c->g.n, rp, inv12h);
    } else {  // two meshes: one component at a time
      for (int j = 0; j < 3; ++j) {
        paint_tiles(c, c->us, c->ids, n, PM_SPECIES_ALL, realA, rp, s, lam_s + (int64_t)j * n);
        LaunchScope L(c, s, K_ADJOINT);
        pdl_launch(k_stencil_axis, (unsigned)(c->g.n * c->g.n), 256, 0, s, realA, realP, c->g.n, rp, j, inv12h, j > 0);
      }
    }
    paint_tiles(c, c->us, c->ids, n, PM_SPECIES_ALL, realA, rp, s);
    if (learned) {
      mlp_table(c, a, s);
      fft_forward(c, c->g, c->meshA, c->meshA, 0, s);
      {
        LaunchScope L(c, s, K_ADJOINT);
        const double nn = (double)c->g.n;
        const int units = (c->g.n / 2 + 1) * (c->g.n / 2 + 2) / 2;
        pdl_launch(k_vjp_combine, (units + 7) / 8, 256, 0, s, c->meshA, pot, c->g.n, c->g.pc, units, c->ksq, c->wforce,
                                                      (float)(-1.5 * c->cosmo.omega_m0 / (nn * nn * nn)), c->mlp_tab,
                                                      c->mlp_gbin);
      }
      fft_inverse_plain(c, c->g, pot, s);  // B
      const size_t sm1 = sizeof(float) * kVjpSpanB * kVjpBSX;
      const int threads = vjp_threads(c, n);
      auto read1 = threads == 512 ? k_vjp_readout<1, 512> : k_vjp_readout<1, 256>;
      auto read3 = threads == 512 ? k_vjp_readout<3, 512> : k_vjp_readout<3, 256>;
      static DeviceOnce once3[2];
      allow_smem(once3[threads == 512], (const void*)read3, 3 * sm1);
      const unsigned tiles = (unsigned)(c->nt * c->nt * c->nt);
      float* const tmp = c->adj + 6 * 3 * n;  // the second term, sorted order
      {
        LaunchScope L(c, s, K_ADJOINT);
        pdl_launch(read1, tiles, threads, sm1, s, c->us, c->ids, n, c->bstart, realP, nullptr, nullptr, c->g.n, 32 - c->g.logn,
                                          c->ntl, rp, inv_h, nullptr, c->mt, nullptr, tmp, nullptr, PM_SPECIES_ALL,
                   c->err_dev);
      }
      // F_y, F_z into the other meshes, F_x in place over phi_k
      fft_inverse_component(c, c->g, c->meshA, c->meshB, 1, s);
      fft_inverse_component(c, c->g, c->meshA, pot, 2, s);
      fft_inverse_component(c, c->g, c->meshA, c->meshA, 0, s);
      {
        LaunchScope L(c, s, K_ADJOINT);
        pdl_launch(read3, tiles, threads, 3 * sm1, s, c->us, c->ids, n, c->bstart, realA, realB, realP, c->g.n, 32 - c->g.logn,
                                              c->ntl, rp, inv_h, lam_s, c->mt, c->vals[0], tmp, grad, PM_SPECIES_ALL,
                   c->err_dev);
      }
      mlp_backward(c, a, s);
      return cudaGetLastError() == cudaSuccess ? PM_OK : PM_ECUDA;
    }
    fft_potential(c, c->g, c->meshA, s);
    fft_potential(c, c->g, pot, s);
    const int threads = vjp_threads(c, n);
    auto kern = threads == 512 ? k_force_vjp_readout<512> : k_force_vjp_readout<256>;
    static DeviceOnce once[2];
    allow_smem(once[threads == 512], (const void*)kern, kVjpSmem);
    {
      LaunchScope L(c, s, K_ADJOINT);
      pdl_launch(kern, (unsigned)(c->nt * c->nt * c->nt), threads, kVjpSmem, s, 
          c->us, c->ids, n, c->bstart, realA, realP, c->g.n, 32 - c->g.logn, c->ntl, rp, inv12h, inv_h, lam_s, c->mt,
          c->vals[0], grad, c->err_dev);
    }
    return cudaGetLastError() == cudaSuccess ? PM_OK : PM_ECUDA;
  }
  // term 1: sum_j lambda_j grad R[G_j rho]
  paint_tiles(c, c->us, c->ids, n, PM_SPECIES_ALL, realA, rp, s);
  if (learned) {
    mlp_table(c, a, s);
    fft_forward(c, c->g, c->meshA, c->meshC, 0, s);  // rho_k, kept for the factor's gradient
    mlp_green_apply(c, c->meshC, c->meshB, s);
  } else {
    fft_forward(c, c->g, c->meshA, c->meshB, 1, s);
  }
  for (int j = 0; j < 3; ++j) {
    fft_inverse_component(c, c->g, c->meshB, c->meshA, j, s);
    const float* m[1] = {realA};
    readout_grad(c, n, m, 1, rp, lam_s + (int64_t)j * n, c->vals[0], grad, j > 0, s);
  }
  // term 2: m_i grad R[B], B_k = sum_j i D(k_j) g FFT(paint(lambda_j))
  const double nn = (double)c->g.n;
  const float gcoef = (float)(-1.5 * c->cosmo.omega_m0 / (nn * nn * nn));
  for (int j = 0; j < 3; ++j) {
    paint_tiles(c, c->us, c->ids, n, PM_SPECIES_ALL, realA, rp, s, lam_s + (int64_t)j * n);
    fft_forward(c, c->g, c->meshA, c->meshA, 0, s);
    LaunchScope L(c, s, K_ADJOINT);
    pdl_launch(k_adj_combine, (unsigned)(c->g.n * c->g.n), 128, 0, s, 
        c->meshA, c->meshB, c->g.n, c->g.pc, c->ksq, c->wforce, c->kvec0, gcoef, j, j > 0,
        learned ? c->mlp_tab : nullptr, learned ? c->meshC : nullptr, c->mlp_gbin);
  }
  fft_inverse_plain(c, c->g, c->meshB, s);
  const float* m[1] = {realB};
  readout_grad(c, n, m, 1, rp, nullptr, c->vals[0], grad, true, s);
  if (learned) mlp_backward(c, a, s);
  return cudaGetLastError() == cudaSuccess ? PM_OK : PM_ECUDA;
}

int step_vjp(pm_ctx* c, const pm_state* st, double a0, double ah, double a1, const float* lx1,
             const float* lp1, float* lx0, float* lp0, cudaStream_t s) {
  const int64_t n = st->n;
  if (n == 0) return PM_OK;
  int rc = ensure_adj(c, n);
  if (rc != PM_OK) return rc;
  double k[3];
  c->cosmo.coeffs(a0, ah, a1, k);
  const int64_t m3 = 3 * n;
  float* Lx = c->adj;             // lambda_x in state order
  float* Lp = c->adj + m3;        // lambda_p in state order
  float* lamF = c->adj + 2 * m3;
  float* g = c->adj + 3 * m3;
  uint32_t* u1 = reinterpret_cast<uint32_t*>(c->adj + 4 * m3);
  {  // lambda_F of x1: K2 lambda_p1
    LaunchScope L(c, s, K_ADJOINT);
    pdl_launch(k_vjp_begin, blocks(n), 256, 0, s, lx1, lp1, st->id, st->u, st->p, st->f, n, (float)k[0],
                                          (float)(k[1] * 4294967296.0 / c->cfg.box), (float)k[2], Lx, Lp, lamF, u1);
  }
  rc = force_vjp(c, u1, st->id, n, lamF, a1, g, s);
  if (rc != PM_OK) return rc;
  {  // lambda_x1' = lambda_x1 + F_vjp(x1), lambda_ph = lambda_p1 + Delta lambda_x1', lambda_F of x0: K1 lambda_ph
    LaunchScope L(c, s, K_ADJOINT);
    pdl_launch(k_vjp_middle, blocks(m3), 256, 0, s, g, m3, (float)k[1], (float)k[0], Lx, Lp, lamF);
  }
  rc = force_vjp(c, st->u, st->id, n, lamF, a0, g, s);
  if (rc != PM_OK) return rc;
  {  // lambda_x0 = lambda_x1' + F_vjp(x0)
    LaunchScope L(c, s, K_ADJOINT);
    pdl_launch(k_vjp_end, blocks(n), 256, 0, s, g, Lx, Lp, st->id, n, lx0, lp0);
  }
  return cudaGetLastError() == cudaSuccess ? PM_OK : PM_ECUDA;
}

int ic_vjp(pm_ctx* c, const float* lx, const float* lp, double a0, double k_fs, float* grad_noise,
           cudaStream_t s) {
  const pm_config& cf = c->cfg;
  const int nc = cf.nc;
  if (nc < 32 || (nc & (nc - 1)) || nc > c->g.n) return PM_EINVAL;
  if (!c->ic_amp || k_fs != c->ic_kfs) return PM_EINVAL;  // pm_ic with the same k_fs first
  Geom gi;
  gi.n = nc;
  gi.logn = 0;
  while ((1 << gi.logn) < nc) ++gi.logn;
  gi.pc = nc / 2 + 2;
  const int64_t n_cdm = (int64_t)nc * nc * nc;
  const int ndir = 2 * cf.nfib + 1;
  const int64_t n_nu = cf.nsites > 0 ? (int64_t)cf.nsites * cf.nsites * cf.nsites * cf.nshell * ndir : 0;
  const int64_t n = n_cdm + n_nu;
  const float D0 = (float)c->cosmo.D(a0), gp0 = (float)c->cosmo.gp(a0);
  const int stride = cf.nsites > 0 ? nc / cf.nsites : 1;
  const bool even = (stride % 2) == 0;
  const int j0 = even ? stride / 2 : (stride + 1) / 2;
  float* realA = reinterpret_cast<float*>(c->meshA);
  const int rp = 2 * gi.pc;
  bool first = true;
  for (int species = 0; species < 2; ++species) {
    if (species == 1 && n_nu == 0) break;
    for (int comp = 0; comp < 3; ++comp) {
      PM_CUDA_TRY(cudaMemsetAsync(c->meshA, 0, sizeof(float2) * gi.elems(), s));
      {
        LaunchScope L(c, s, K_ADJOINT);
        if (species == 0)
          pdl_launch(k_icadj_cdm, blocks(n_cdm), 256, 0, s, lx, lp, nc, rp, comp, D0, gp0, n, realA);
        else
          pdl_launch(k_icadj_nu, blocks((int64_t)cf.nsites * cf.nsites * cf.nsites), 256, 0, s, 
              lx, lp, nc, rp, comp, D0, gp0, cf.nsites, stride, j0, cf.nshell * ndir, n_cdm, n, realA);
      }
      fft_forward(c, gi, c->meshA, c->meshA, 0, s);
      LaunchScope L(c, s, K_ADJOINT);
      pdl_launch(k_icadj_kspace, (unsigned)(nc * nc), 128, 0, s, c->meshA, c->meshB, nc, gi.pc,
                                                         species == 0 ? c->ic_amp : c->ic_amp_nu, comp,
                                                         species == 1 && even ? 1 : 0, first ? 0 : 1);
      first = false;
    }
  }
  fft_inverse_plain(c, gi, c->meshB, s);
  repack_real(c, gi, reinterpret_cast<float*>(c->meshB), rp, grad_noise, nc, s);
  return cudaGetLastError() == cudaSuccess ? PM_OK : PM_ECUDA;
}

}  // namespace pmnu
