// The two direct-sum estimators of Sec. 4, "sum-gal" and "sum-grid", on the GPU.
//
// Both evaluate Eq. (4) with A_n(k) = sum_p s_p w_p (k_hat . r_hat_p)^n e^{-i k.x_p} at
// every half-grid mode k = k_F m of the binning, for n = 0, 2, 4 (and 6), then the
// shell means of Eqs. (6)-(8):
//   sum-gal   the points are the galaxies (s = +1) and randoms (s = -alpha), r_p the
//             point's own line of sight: no mesh, no window, no aliasing, and any
//             k lattice (k_F m with |m| below n_mesh / 2 of the configuration, which
//             need not be an FFT size);
//   sum-grid  the points are the nodes of a plan's assigned mesh(es), weight F,
//             r = node - observer as in the FFT path: its exact DFT, which the FFT
//             path reproduces mode by mode.
// One more complex sum per mode, with the top hat Theta(|mu| <= 1/2) in place of the
// Legendre weight, gives the wedges by their definition (Sec. 5, Eqs. 14-15).
//
// Layout: one thread per group of SG_GROUP modes with neighbouring m_z, their complex
// sums in registers; points stream through shared memory in chunks that every thread
// reads as broadcasts.  Positions are 32-bit fixed-point fractions of the box,
// u = (x - box_min) / L, so the phase k.x = 2 pi m.u is taken mod one turn exactly by
// integer multiply-adds.  The group's middle mode takes sine and cosine of its phase
// (cis_minus: beyond the angle's float rounding), the others multiply by the point's
// e^{-2 pi i j u_z}, j = +-1, +-2, formed once per point in FP64.  Every term of A_0 and of the
// top-hat sum goes into a compensated float sum (add_comp); of A_2, A_4, .. SG_BLOCK terms
// are added in float first.  CTAs that split the points add their sums into FP64 per-mode
// accumulators, and a second kernel forms the shell sums in FP64.
//
// What bounds the mode kernel: the FP32 pipes and issue, about 30 instructions per mode and
// point at l_max = 4, the sums in packed pairs (105 with one sincospif and six scalar
// compensated adds per mode and point).  The sums carry (m . r_hat)^n, normalised in FP64
// afterwards: with k_hat in float its rounding was common to all points.  Against FP64, over
// 10 to 40 catalogues and lattices of 20 to 64: P_2 and P_4 are off by 0.3 to 0.5 times what
// one sincospif and one compensated add per term give, P_0 and the wedges by 0.8 to 1.1 times
// (with the angles rounded to float and A_0 summed in blocks 1.2 to 2.0 times): 4.7e-8 rms a
// term, 7.2e-8 then.
// 68 000 modes of a 64^3 lattice, 120 000 points: 26.9 -> 9.8 ms a call.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <string>
#include <vector>

#include "fft.cuh"
#include "ys_internal.h"

namespace ys {
namespace {

constexpr int SG_THREADS = 128;
constexpr int SG_CHUNK = 256;  // points per shared-memory chunk
constexpr int SG_SPLIT_MIN = 128;  // points per thread at least
constexpr int SG_GROUP = 5;    // modes per thread (neighbouring m_z)
constexpr int SG_BLOCK = 4;    // points per block of plain sums

// Components of the per-mode sums: A_0, A_2, A_4, A_6 and the top-hat sum B_perp.
enum { C_A0 = 0, C_A2 = 1, C_A4 = 2, C_A6 = 3, C_BP = 4, C_COUNT = 5 };

struct __align__(16) SgPoint {
  uint32_t u[3];  // position as a fraction of the box, 2^-32 units
  float sw;       // signed weight
  float rh[3];    // r_hat (0 at r = 0)
  float pad;
  float2 w1, w2;  // e^{-2 pi i u_z}, e^{-4 pi i u_z}
};

struct SgMode {
  short m[3];     // integer frequency
  short bin;      // shell
  float w;        // Hermitian weight (1 or 2)
};

// Up to SG_GROUP modes (m_x, m_y, m_z .. m_z + count - 1), entries first .. of the mode list.
struct SgGroup {
  short mx, my, mz, count;
  int first;
};

// s += v with the rounding error added to c, both components (Fast2Sum: exact where |s| >= |v|,
// else off by an ulp of v at most; over a walk of 64 to 1024 terms that leaves 3e-9 to 5e-9 of
// a term per term, a tenth of the terms' own rounding, for 4 instructions instead of 7).
__device__ __forceinline__ void add_comp(float2& s, float2& c, float2 v) {
  const float2 t = cadd(s, v);
  c = cadd(c, csub(v, csub(t, s)));
  s = t;
}

// FP64 catalogue sums of Eqs. (1) and (3) (the same slots as the assignment's).
__global__ void k_sg_sums(const float* __restrict__ w, const float* __restrict__ nbar, int64_t n, int is_ran,
                          double* __restrict__ sums) {
  double s1 = 0.0, s2 = 0.0, s3 = 0.0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const double v = w ? (double)w[i] : 1.0;
    s1 += v;
    s2 += v * v;
    if (is_ran && nbar) s3 += v * v * (double)nbar[i];
  }
  for (int o = 16; o > 0; o >>= 1) {
    s1 += __shfl_xor_sync(0xffffffffu, s1, o);
    s2 += __shfl_xor_sync(0xffffffffu, s2, o);
    s3 += __shfl_xor_sync(0xffffffffu, s3, o);
  }
  if ((threadIdx.x & 31) == 0) {
    if (is_ran) {
      atomicAdd(&sums[SUM_WR], s1);
      atomicAdd(&sums[SUM_WR2], s2);
      atomicAdd(&sums[SUM_WR2N], s3);
    } else {
      atomicAdd(&sums[SUM_WG], s1);
      atomicAdd(&sums[SUM_WG2], s2);
    }
  }
}

__device__ __forceinline__ uint32_t to_fixed(double u) {
  u -= floor(u);  // one period of the box (the sums are periodic in x with period L)
  return (uint32_t)(uint64_t)(u * 4294967296.0);
}

__device__ __forceinline__ void unit3(double x, double y, double z, float (&o)[3]) {
  const double r = sqrt(x * x + y * y + z * z);
  const double inv = r > 0.0 ? 1.0 / r : 0.0;
  o[0] = (float)(x * inv);
  o[1] = (float)(y * inv);
  o[2] = (float)(z * inv);
}

// w e^{-2 pi i turn}, turn in units of 2^-32.  The angle's leading 24 bits are exact in float;
// the rest, at most 1.9e-7, is applied to first order (an angle rounded to float is off by up
// to 9.4e-8, more than all other roundings of the result).
__device__ __forceinline__ float2 cis_minus(uint32_t turn, float w) {
  const uint32_t hi = (turn + 128u) & ~255u;
  float sn, cs;
  sincospif((float)(int32_t)hi * 4.656612873077393e-10f, &sn, &cs);  // angle / pi in [-1, 1)
  const float d = w * ((float)(int32_t)(turn - hi) * 1.4629180792671596e-9f);  // pi 2^-31
  return make_float2(fmaf(w, cs, -d * sn), -fmaf(w, sn, d * cs));
}

// e^{-2 pi i turn} within 0.75 ulp (2.07e-8 rms; correct rounding 2.06e-8): the points' rotations,
// which four of a group's five modes share.  The angle t + e is reduced to [-pi/4, pi/4] in
// integers, then the Taylor series to t^11 and t^10 with the leading terms' rounding carried
// (FP64 sincospi took 0.2 ms for 1.2e6 points).
__device__ __forceinline__ float2 cis_minus_exact(uint32_t turn) {
  const uint32_t q = (turn + (1u << 29)) >> 30;  // quadrant, 0 .. 4
  const int r = (int)(turn - (q << 30)), rh = (r + 32) & ~63;
  const float pi_h = 1.4629180792671596e-9f, pi_l = (float)(1.4629180792671596e-9 - (double)pi_h);  // pi 2^-31
  const float x = (float)rh, t = __fmul_rn(x, pi_h);
  const float e = fmaf(x, pi_l, fmaf((float)(r - rh), pi_h, fmaf(x, pi_h, -t)));
  const float z = __fmul_rn(t, t), ez = fmaf(t, t, -z);
  float ps = fmaf(z, -1.f / 39916800.f, 1.f / 362880.f);
  ps = fmaf(z, fmaf(z, fmaf(z, ps, -1.f / 5040.f), 1.f / 120.f), -1.f / 6.f);
  const float sn = t + fmaf(__fmul_rn(t, z), ps, fmaf(__fmul_rn(e, z), -0.5f, e));
  float pc = fmaf(z, -1.f / 3628800.f, 1.f / 40320.f);
  pc = fmaf(z, fmaf(z, pc, -1.f / 720.f), 1.f / 24.f);
  const float a = fmaf(z, -0.5f, 1.f), b = fmaf(z, -0.5f, 1.f - a);  // a + b = 1 - z / 2
  const float cs = a + fmaf(__fmul_rn(z, z), pc, fmaf(e, -sn, fmaf(ez, -0.5f, b)));
  const float c = (q & 1u) ? sn : cs, s = (q & 1u) ? cs : sn;
  return make_float2(((q + 1u) & 2u) ? -c : c, (q & 2u) ? s : -s);
}

// Catalogue particles as points: galaxies +w, randoms -alpha w.
__global__ void k_sg_points_cat(const float* __restrict__ x, const float* __restrict__ y,
                                const float* __restrict__ z, const float* __restrict__ w, int64_t n, int is_ran,
                                const double* __restrict__ sums, double alpha_cfg, double bx, double by, double bz,
                                double inv_len, double ox, double oy, double oz, SgPoint* __restrict__ out) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  double sgn = 1.0;
  if (is_ran) sgn = -(alpha_cfg >= 0.0 ? alpha_cfg : sums[SUM_WG] / sums[SUM_WR]);
  const double px = x[i], py = y[i], pz = z[i];
  SgPoint q;
  q.u[0] = to_fixed((px - bx) * inv_len);
  q.u[1] = to_fixed((py - by) * inv_len);
  q.u[2] = to_fixed((pz - bz) * inv_len);
  q.sw = (float)(sgn * (w ? (double)w[i] : 1.0));
  unit3(px - ox, py - oy, pz - oz, q.rh);
  q.pad = 0.f;
  q.w1 = cis_minus_exact(q.u[2]);
  q.w2 = cis_minus_exact(2u * q.u[2]);
  out[i] = q;
}

// Mesh nodes [first, first + count) of mesh j with F != 0 as points (compacted with a
// counter).  Node i of mesh j sits at box_min + (i + j/2) H; scale multiplies F (1/2
// for each of two interlaced meshes).
__global__ void k_sg_points_mesh(const float* __restrict__ mesh, int n, int j, int64_t first, int64_t count_nodes,
                                 double rel_x0, double rel_y0, double rel_z0, double H, float scale,
                                 unsigned* __restrict__ count, SgPoint* __restrict__ out) {
  const int64_t idx = first + (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= first + count_nodes) return;
  const float f = mesh[idx];
  if (f == 0.f) return;
  const int iz = (int)(idx % n), iy = (int)((idx / n) % n), ix = (int)(idx / ((int64_t)n * n));
  const double s = 0.5 * j;
  SgPoint q;
  const double inv_n = 1.0 / n;
  q.u[0] = to_fixed((ix + s) * inv_n);
  q.u[1] = to_fixed((iy + s) * inv_n);
  q.u[2] = to_fixed((iz + s) * inv_n);
  q.sw = f * scale;
  unit3(rel_x0 + (ix + s) * H, rel_y0 + (iy + s) * H, rel_z0 + (iz + s) * H, q.rh);
  q.pad = 0.f;
  q.w1 = cis_minus_exact(q.u[2]);
  q.w2 = cis_minus_exact(2u * q.u[2]);
  out[atomicAdd(count, 1u)] = q;
}

// Per-mode sums over the points of this CTA's split (blockIdx.y); FP64 atomics into
// acc[C_COUNT][nmodes] (interleaved re, im).
template <int ELL, bool WEDGE, bool SLICED>
__global__ void __launch_bounds__(SG_THREADS) k_sg_modes(const SgGroup* __restrict__ groups, int ngroups, int nmodes,
                                                          const SgPoint* __restrict__ pts,
                                                          const unsigned* __restrict__ npts_dev, int64_t npts_host,
                                                          int splits, int slices, double* __restrict__ acc) {
  __shared__ SgPoint s_pts[SG_CHUNK];
  // SLICED, at most half as many groups as threads: each group gets `slices` threads, which
  // share out the points of a chunk in blocks (an 8^3 lattice has 41 groups; 1.2e6 points took
  // 1.2 to 1.9 ms a call with one thread each, 0.9 to 1.5 ms with one mode per thread, 0.8 to
  // 1.3 ms so).
  const int width = SLICED ? ngroups : SG_THREADS, slice = SLICED ? threadIdx.x / width : 0;
  const int gi = blockIdx.x * width + threadIdx.x - slice * width;
  const bool active = gi < ngroups && (!SLICED || slice < slices);
  const int64_t npts = npts_dev ? (int64_t)*npts_dev : npts_host;
  const int64_t per = (npts + splits - 1) / splits;
  const int64_t p_lo = std::min<int64_t>(npts, per * blockIdx.y), p_hi = std::min<int64_t>(npts, p_lo + per);
  SgGroup g{};
  if (active) g = groups[gi];
  const int mid = g.mz + SG_GROUP / 2;
  // The sums carry (m . r_hat)^n: the mode's 1 / |m|^n is applied in FP64 (k_sg_shells).  In
  // float m is scaled by 2^-sh, |m| <= 2^sh over the group, so that no power leaves the range
  // of the weights.
  const int mz_far = max(abs((int)g.mz), abs((int)g.mz + SG_GROUP - 1));
  const int sh = (33 - __clz(g.mx * g.mx + g.my * g.my + mz_far * mz_far)) / 2;
  const float unit = __int_as_float((127 - sh) << 23);
  const float fx = g.mx * unit, fy = g.my * unit;
  // The top hat, which jumps at |mu| = 1/2, takes mu from k_hat's components.
  [[maybe_unused]] float kh[WEDGE ? SG_GROUP : 1][3];
  if constexpr (WEDGE) {
#pragma unroll
    for (int j = 0; j < SG_GROUP; ++j) {
      const int mz = g.mz + j, n2 = g.mx * g.mx + g.my * g.my + mz * mz;
      const double inv = n2 > 0 ? 1.0 / sqrt((double)n2) : 0.0;
      kh[j][0] = (float)(g.mx * inv);
      kh[j][1] = (float)(g.my * inv);
      kh[j][2] = (float)(mz * inv);
    }
  }
  constexpr int NM = ELL >= 6 ? 4 : ELL / 2 + 1;  // A_0, A_2, ..
  constexpr int NC = NM + (WEDGE ? 1 : 0);
  float2 S[SG_GROUP][NC], C[SG_GROUP][NC];
#pragma unroll
  for (int j = 0; j < SG_GROUP; ++j)
#pragma unroll
    for (int c = 0; c < NC; ++c) S[j][c] = C[j][c] = make_float2(0.f, 0.f);
  for (int64_t base = p_lo; base < p_hi; base += SG_CHUNK) {
    const int cnt = (int)std::min<int64_t>(SG_CHUNK, p_hi - base);
    __syncthreads();
    // points past the end carry no weight
    for (int i = threadIdx.x; i < SG_CHUNK; i += SG_THREADS) s_pts[i] = i < cnt ? pts[base + i] : SgPoint{};
    __syncthreads();
    if (!active) continue;
#pragma unroll 1
    for (int i = slice * SG_BLOCK; i < cnt; i += SLICED ? slices * SG_BLOCK : SG_BLOCK) {
      float2 e[SG_BLOCK];  // s w e^{-i k.x} of the middle mode
      float d[SG_BLOCK];   // (m_x r_hat_x + m_y r_hat_y) 2^-sh
#pragma unroll
      for (int b = 0; b < SG_BLOCK; ++b) {
        const SgPoint& q = s_pts[i + b];
        // one turn = 2^32: the phase m.u mod 1 is exact in wrapping integer arithmetic
        e[b] = cis_minus((uint32_t)(int)g.mx * q.u[0] + (uint32_t)(int)g.my * q.u[1] + (uint32_t)mid * q.u[2], q.sw);
        d[b] = fmaf(fx, q.rh[0], fy * q.rh[1]);
      }
#pragma unroll
      for (int j = 0; j < SG_GROUP; ++j) {
        [[maybe_unused]] float2 p[NM];  // the block's plain sums of A_2, A_4, ..
#pragma unroll
        for (int b = 0; b < SG_BLOCK; ++b) {
          const SgPoint& q = s_pts[i + b];
          const int o = j - SG_GROUP / 2;
          float2 t = e[b];
          if (o != 0) {
            const float2 w = (o == 1 || o == -1) ? q.w1 : q.w2;
            t = cmul(t, o > 0 ? w : make_float2(w.x, -w.y));
          }
          add_comp(S[j][0], C[j][0], t);
          if constexpr (NM > 1) {
            const float md = fmaf((float)(g.mz + j) * unit, q.rh[2], d[b]), md2 = md * md;  // m . r_hat 2^-sh
            float f = md2;
#pragma unroll
            for (int c = 1; c < NM; ++c) {
              const float2 ff = make_float2(f, f);
              p[c] = b == 0 ? __fmul2_rn(ff, t) : __ffma2_rn(ff, t, p[c]);
              f *= md2;
            }
          }
          if constexpr (WEDGE) {
            const float mu = fmaf(kh[j][0], q.rh[0], fmaf(kh[j][1], q.rh[1], kh[j][2] * q.rh[2]));
            const bool in = fabsf(mu) <= 0.5f;
            add_comp(S[j][NC - 1], C[j][NC - 1], make_float2(in ? t.x : 0.f, in ? t.y : 0.f));
          }
        }
#pragma unroll
        for (int c = 1; c < NM; ++c) add_comp(S[j][c], C[j][c], p[c]);
      }
    }
  }
  if (!SLICED && !active) return;
  // the slices of a group meet in shared memory: FP64 atomics on one address are served one
  // after another
  [[maybe_unused]] double2* red = reinterpret_cast<double2*>(s_pts);
  static_assert(sizeof(s_pts) >= sizeof(double2) * SG_THREADS, "slices' sums");
#pragma unroll
  for (int j = 0; j < SG_GROUP; ++j) {
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      double2 v = make_double2((double)S[j][c].x + (double)C[j][c].x, (double)S[j][c].y + (double)C[j][c].y);
      if constexpr (SLICED) {
        __syncthreads();
        red[threadIdx.x] = v;
        __syncthreads();
        if (slice == 0)
          for (int q = 1; q < slices; ++q) {
            const double2 o = red[threadIdx.x + q * width];
            v.x += o.x;
            v.y += o.y;
          }
      }
      if (!active || slice > 0 || j >= g.count) continue;
      const int comp = (WEDGE && c == NC - 1) ? C_BP : c;
      double* a = acc + ((size_t)comp * nmodes + g.first + j) * 2;
      const double back = c < NM ? __longlong_as_double((1023ll + 2 * c * sh) << 52) : 1.0;  // 2^(2 c sh)
      atomicAdd(a, v.x * back);
      atomicAdd(a + 1, v.y * back);
    }
  }
}

// Shell sums in FP64: slot s = Re A_0 A_{2s}^* for s < nmain and, with wedge, slot 4 =
// Re A_0 B_perp^*, weighted; the window is divided out of every A (invw per axis, 1
// without it).
__global__ void k_sg_shells(const SgMode* __restrict__ modes, int nmodes, const double* __restrict__ acc,
                            const float* __restrict__ invw, int n, int nmain, int wedge, int nbins,
                            double* __restrict__ shell_acc) {
  const int mi = blockIdx.x * blockDim.x + threadIdx.x;
  if (mi >= nmodes) return;
  const SgMode md = modes[mi];
  double cw = 1.0;
  if (invw) {
    for (int a = 0; a < 3; ++a) {
      const int idx = md.m[a] < 0 ? md.m[a] + n : md.m[a];
      cw *= (double)invw[idx];
    }
  }
  const double* a0 = acc + (size_t)mi * 2;
  const double r0 = a0[0] * cw, i0 = a0[1] * cw;
  const double inv_n2 = 1.0 / (double)(md.m[0] * md.m[0] + md.m[1] * md.m[1] + md.m[2] * md.m[2]);
  double norm = 1.0;  // 1 / |m|^(2 s)
  for (int s = 0; s < nmain + (wedge ? 1 : 0); ++s) {
    const int comp = s < nmain ? s : C_BP;
    const int slot = s < nmain ? s : 4;
    const double* as = acc + ((size_t)comp * nmodes + mi) * 2;
    const double v = md.w * (s < nmain ? norm : 1.0) * (r0 * as[0] * cw + i0 * as[1] * cw);
    atomicAdd(&shell_acc[(size_t)slot * nbins + md.bin], v);
    norm *= inv_n2;
  }
}

// Result row (plan layout) and the wedges from the shell sums.
__global__ void k_sg_finalize(const double* __restrict__ sacc, const double* __restrict__ shell,
                              const double* __restrict__ sums, double alpha_cfg, int nbins, int ell, int wedges,
                              double* __restrict__ res, double* __restrict__ wout) {
  const double alpha = alpha_cfg >= 0.0 ? alpha_cfg : sums[SUM_WG] / sums[SUM_WR];
  const double I = alpha * sums[SUM_WR2N];
  const double S = sums[SUM_WG2] + alpha * alpha * sums[SUM_WR2];
  const double nan = __longlong_as_double(0x7ff8000000000000ULL);
  for (int b = threadIdx.x; b < nbins; b += blockDim.x) {
    const double nm = shell[b];
    double km = nan, p0 = nan, p2 = nan, p4 = nan, p6 = nan, pp = nan, pq = nan;
    if (nm > 0.0) {
      km = shell[nbins + b] / nm;
      const double m0 = sacc[b] / nm, m2 = sacc[nbins + b] / nm, m4 = sacc[2 * nbins + b] / nm;
      p0 = (m0 - S) / I;  // Eqs. (6)-(8)
      if (ell >= 2) p2 = 2.5 / I * (3.0 * m2 - m0);
      if (ell >= 4) p4 = 1.125 / I * (35.0 * m4 - 30.0 * m2 + 3.0 * m0);
      if (ell >= 6) p6 = 0.8125 / I * (231.0 * sacc[3 * nbins + b] / nm - 315.0 * m4 + 105.0 * m2 - 5.0 * m0);
      if (wedges) {  // Eqs. 14-15: the top hats normalised by 1 / (1/2), shot noise S/I
        const double mp = sacc[4 * nbins + b] / nm;
        pp = 2.0 / I * mp - S / I;
        pq = 2.0 / I * (m0 - mp) - S / I;
      }
    }
    res[b] = km;
    res[nbins + b] = nm;
    res[2 * nbins + b] = p0;
    res[3 * nbins + b] = p2;
    res[4 * nbins + b] = p4;
    if (ell >= 6) res[5 * nbins + 5 + b] = p6;
    if (wedges) {
      wout[b] = pp;
      wout[nbins + b] = pq;
    }
  }
  if (threadIdx.x == 0) {
    res[5 * nbins + 0] = alpha;
    res[5 * nbins + 1] = I;
    res[5 * nbins + 2] = S / I;
    res[5 * nbins + 3] = 0.0;
    res[5 * nbins + 4] = 0.0;
  }
}

struct ModeTable {
  std::vector<SgMode> modes;
  std::vector<SgGroup> groups;
  size_t mode_bytes() const { return sizeof(SgMode) * modes.size(); }
  size_t group_bytes() const { return sizeof(SgGroup) * groups.size(); }
  std::vector<double> shell;  // [2][nbins]: mode count, sum |k|
};

// Half-grid modes of an n^3 lattice (m_x, m_y in [-n/2, n/2), m_z in [0, n/2]; weight 2
// for 0 < m_z < n/2) with 0 < |k| < k_F n / 2 that fall in a shell.
ModeTable build_modes(const ys_config& c) {
  ModeTable t;
  const int n = c.n_mesh;
  const double kf = 2.0 * M_PI / c.box_len, knyq = kf * n / 2.0;
  const double kmax = std::min(knyq, c.k_min + c.dk * c.n_bins);
  const int mr = std::min(n / 2, (int)std::ceil(kmax / kf) + 1);
  t.shell.assign(2 * (size_t)c.n_bins, 0.0);
  // shell (-1: none) and |k| of every |m|^2 up to the largest that can fall in one
  const int n2_max = mr * mr;
  std::vector<int> shell(n2_max + 1, -1);
  std::vector<double> k_of(n2_max + 1, 0.0);
  for (int n2 = 1; n2 <= n2_max; ++n2) {
    const double km = kf * std::sqrt((double)n2);
    if (!(km < knyq)) continue;
    const double b = std::floor((km - c.k_min) / c.dk);
    if (!(b >= 0 && b < c.n_bins)) continue;
    shell[n2] = (int)b;
    k_of[n2] = km;
  }
  const int hi = std::min(mr, n / 2 - 1);  // m_x, m_y in [-n/2, n/2)
  for (int mx = -mr; mx <= hi; ++mx)
    for (int my = -mr; my <= hi; ++my) {
      const int xy2 = mx * mx + my * my;
      for (int mz = 0; mz <= mr && xy2 + mz * mz <= n2_max; ++mz) {
        const int n2 = xy2 + mz * mz;
        if (shell[n2] < 0) continue;
        SgMode md;
        md.m[0] = (short)mx;
        md.m[1] = (short)my;
        md.m[2] = (short)mz;
        md.bin = (short)shell[n2];
        md.w = (mz > 0 && mz < n / 2) ? 2.f : 1.f;
        // modes of one (m_x, m_y) with consecutive m_z share a group
        SgGroup* g = t.groups.empty() ? nullptr : &t.groups.back();
        if (g && g->mx == mx && g->my == my && g->mz + g->count == mz && g->count < SG_GROUP) {
          ++g->count;
        } else {
          t.groups.push_back({(short)mx, (short)my, (short)mz, 1, (int)t.modes.size()});
        }
        t.modes.push_back(md);
        t.shell[(size_t)md.bin] += md.w;
        t.shell[(size_t)c.n_bins + (size_t)md.bin] += md.w * k_of[n2];
      }
    }
  return t;
}

// Device buffers of one direct-sum call, freed on every return path.
struct Scratch {
  std::vector<void*> ptrs;
  template <class T>
  cudaError_t get(T*& p, size_t count) {
    void* raw = nullptr;
    cudaError_t e = cudaMalloc(&raw, std::max<size_t>(1, count) * sizeof(T));
    if (!e) {
      ptrs.push_back(raw);
      p = static_cast<T*>(raw);
    }
    return e;
  }
  ~Scratch() {
    for (void* q : ptrs) cudaFree(q);
  }
};

ys_status fail(cudaError_t e) {
  g_last_cuda_error = cudaGetErrorString(e);
  return e == cudaErrorMemoryAllocation ? YS_ERR_OOM : YS_ERR_CUDA;
}

// The mode and group lists on the device, in one piece.
cudaError_t upload(const ModeTable& mt, Scratch& sc, cudaStream_t st, SgMode*& d_modes, SgGroup*& d_groups) {
  static_assert(alignof(SgGroup) <= alignof(SgMode), "groups follow the modes");
  unsigned char* raw = nullptr;
  cudaError_t e = sc.get(raw, mt.mode_bytes() + mt.group_bytes());
  if (e) return e;
  d_modes = reinterpret_cast<SgMode*>(raw);
  d_groups = reinterpret_cast<SgGroup*>(raw + mt.mode_bytes());
  if (mt.modes.empty()) return cudaSuccess;
  e = cudaMemcpyAsync(d_modes, mt.modes.data(), mt.mode_bytes(), cudaMemcpyHostToDevice, st);
  return e ? e : cudaMemcpyAsync(d_groups, mt.groups.data(), mt.group_bytes(), cudaMemcpyHostToDevice, st);
}

// The modes' groups on the device.
struct ModeGroups {
  const SgGroup* groups;
  int ngroups, nmodes;
};

template <int ELL, bool WEDGE>
cudaError_t launch_modes(const ModeGroups& mg, const SgPoint* pts, const unsigned* npts_dev,
                         int64_t npts_host, double* acc, cudaStream_t st) {
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (!e) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e) return e;
  const int mblocks = (mg.ngroups + SG_THREADS - 1) / SG_THREADS;
  const int slices = std::max(1, SG_THREADS / mg.ngroups);
  // split the points so that the grid fills the GPU a few times over, with SG_SPLIT_MIN points
  // per thread at least (npts_host bounds *npts_dev)
  const int64_t want = ((int64_t)sms * 16 + mblocks - 1) / mblocks;
  const int splits = (int)std::max<int64_t>(1, std::min(want, (npts_host + SG_SPLIT_MIN * slices - 1) / (SG_SPLIT_MIN * slices)));
  dim3 grid(mblocks, splits);
  auto kern = slices > 1 ? k_sg_modes<ELL, WEDGE, true> : k_sg_modes<ELL, WEDGE, false>;
  kern<<<grid, SG_THREADS, 0, st>>>(mg.groups, mg.ngroups, mg.nmodes, pts, npts_dev, npts_host, splits, slices, acc);
  return cudaGetLastError();
}

cudaError_t run_modes(int ell, bool wedge, const ModeGroups& mg, const SgPoint* pts,
                      const unsigned* npts_dev, int64_t npts_host, double* acc, cudaStream_t st) {
  switch (ell * 2 + (wedge ? 1 : 0)) {
    case 0: return launch_modes<0, false>(mg, pts, npts_dev, npts_host, acc, st);
    case 1: return launch_modes<0, true>(mg, pts, npts_dev, npts_host, acc, st);
    case 4: return launch_modes<2, false>(mg, pts, npts_dev, npts_host, acc, st);
    case 5: return launch_modes<2, true>(mg, pts, npts_dev, npts_host, acc, st);
    case 8: return launch_modes<4, false>(mg, pts, npts_dev, npts_host, acc, st);
    case 9: return launch_modes<4, true>(mg, pts, npts_dev, npts_host, acc, st);
    case 12: return launch_modes<6, false>(mg, pts, npts_dev, npts_host, acc, st);
    default: return launch_modes<6, true>(mg, pts, npts_dev, npts_host, acc, st);
  }
}

// Shells, finalize and copies shared by both estimators.
ys_status finish(const ModeTable& mt, const SgMode* d_modes, const double* d_acc, const float* d_invw, int n,
                 const double* d_sums, double alpha_cfg, int nbins, int ell, bool wedge, double* d_out,
                 double* d_wedges, Scratch& sc, cudaStream_t st) {
  const int nmodes = (int)mt.modes.size();
  const int nmain = ell >= 6 ? 4 : ell / 2 + 1;
  const int slots_alloc = 5;
  double *d_sacc = nullptr, *d_shell = nullptr;
  cudaError_t e;
  if ((e = sc.get(d_sacc, (size_t)slots_alloc * nbins)) || (e = sc.get(d_shell, mt.shell.size()))) return fail(e);
  if ((e = cudaMemsetAsync(d_sacc, 0, sizeof(double) * slots_alloc * nbins, st))) return fail(e);
  if ((e = cudaMemcpyAsync(d_shell, mt.shell.data(), sizeof(double) * mt.shell.size(), cudaMemcpyHostToDevice, st)))
    return fail(e);
  if (nmodes > 0) {
    // slots 0..3 = mu^0..mu^6; the top-hat sum goes to slot 4 whatever l_max is
    k_sg_shells<<<(nmodes + 255) / 256, 256, 0, st>>>(d_modes, nmodes, d_acc, d_invw, n, nmain, wedge ? 1 : 0,
                                                      nbins, d_sacc);
    if ((e = cudaGetLastError())) return fail(e);
  }
  k_sg_finalize<<<1, 256, 0, st>>>(d_sacc, d_shell, d_sums, alpha_cfg, nbins, ell, wedge ? 1 : 0, d_out, d_wedges);
  if ((e = cudaGetLastError())) return fail(e);
  if ((e = cudaStreamSynchronize(st))) return fail(e);
  return YS_OK;
}

}  // namespace
}  // namespace ys

using namespace ys;

extern "C" ys_status ys_sum_gal(const ys_config* cfg, const ys_catalog* gal, const ys_catalog* ran, double* d_out,
                                double* d_wedges) {
  if (!cfg || !gal || !ran || !d_out) return YS_ERR_ARG;
  const ys_config& c = *cfg;
  if (c.n_mesh < 4 || c.n_mesh > 16384 || (c.n_mesh & 1)) return YS_ERR_ARG;
  if (!(c.box_len > 0) || !std::isfinite(c.box_len)) return YS_ERR_ARG;
  if (c.ell_max != 0 && c.ell_max != 2 && c.ell_max != 4 && c.ell_max != 6) return YS_ERR_ARG;
  if (c.n_bins <= 0 || c.n_bins > 4096 || !(c.dk > 0) || !(c.k_min >= 0)) return YS_ERR_ARG;
  for (const ys_catalog* k : {gal, ran})
    if (k->n < 0 || (k->n > 0 && (!k->x || !k->y || !k->z))) return YS_ERR_ARG;
  cudaStream_t st = static_cast<cudaStream_t>(c.stream);
  const ModeTable mt = build_modes(c);
  const int nmodes = (int)mt.modes.size();
  const bool wedge = d_wedges != nullptr;
  Scratch sc;
  SgMode* d_modes = nullptr;
  SgGroup* d_groups = nullptr;
  double *d_acc = nullptr, *d_sums = nullptr;
  SgPoint* d_pts = nullptr;
  const int64_t npts = gal->n + ran->n;
  cudaError_t e;
  if ((e = upload(mt, sc, st, d_modes, d_groups)) || (e = sc.get(d_acc, (size_t)C_COUNT * 2 * std::max(1, nmodes))) ||
      (e = sc.get(d_sums, (size_t)SUM_COUNT)) || (e = sc.get(d_pts, (size_t)std::max<int64_t>(1, npts))))
    return fail(e);
  const ModeGroups mg{d_groups, (int)mt.groups.size(), nmodes};
  if ((e = cudaMemsetAsync(d_acc, 0, sizeof(double) * C_COUNT * 2 * std::max(1, nmodes), st)) ||
      (e = cudaMemsetAsync(d_sums, 0, sizeof(double) * SUM_COUNT, st)))
    return fail(e);
  const ys_catalog* cats[2] = {gal, ran};
  for (int k = 0; k < 2; ++k)
    if (cats[k]->n > 0) {
      const unsigned blocks = (unsigned)std::min<int64_t>(1024, (cats[k]->n + 255) / 256);
      k_sg_sums<<<blocks, 256, 0, st>>>(cats[k]->w, cats[k]->nbar, cats[k]->n, k, d_sums);
      if ((e = cudaGetLastError())) return fail(e);
    }
  int64_t off = 0;
  for (int k = 0; k < 2; ++k) {
    const ys_catalog& q = *cats[k];
    if (q.n > 0) {
      k_sg_points_cat<<<(unsigned)((q.n + 255) / 256), 256, 0, st>>>(
          q.x, q.y, q.z, q.w, q.n, k, d_sums, c.alpha, c.box_min[0], c.box_min[1], c.box_min[2], 1.0 / c.box_len,
          c.observer[0], c.observer[1], c.observer[2], d_pts + off);
      if ((e = cudaGetLastError())) return fail(e);
    }
    off += q.n;
  }
  if (nmodes > 0 && npts > 0 && (e = run_modes(c.ell_max, wedge, mg, d_pts, nullptr, npts, d_acc, st)))
    return fail(e);
  return finish(mt, d_modes, d_acc, nullptr, c.n_mesh, d_sums, c.alpha, c.n_bins, c.ell_max, wedge, d_out, d_wedges,
                sc, st);
}

extern "C" ys_status ys_sum_grid(ys_plan* plan, double* d_out, double* d_wedges) {
  if (!plan || !d_out) return YS_ERR_ARG;
  Plan& p = plan->p;
  if (!p.assigned) return YS_ERR_STATE;
  const ys_config& c = p.cfg;
  cudaStream_t st = p.stream;
  const ModeTable mt = build_modes(c);
  const int nmodes = (int)mt.modes.size();
  const bool wedge = d_wedges != nullptr;
  const int64_t n3 = (int64_t)p.n * p.n * p.n;
  // the nodes go through in chunks of at most 2 GB of points, each added into the FP64
  // per-mode sums
  const int64_t chunk = std::min<int64_t>(n3, ((int64_t)2 << 30) / (int64_t)sizeof(SgPoint));
  Scratch sc;
  SgMode* d_modes = nullptr;
  SgGroup* d_groups = nullptr;
  double* d_acc = nullptr;
  SgPoint* d_pts = nullptr;
  unsigned* d_count = nullptr;
  cudaError_t e;
  if ((e = upload(mt, sc, st, d_modes, d_groups)) || (e = sc.get(d_acc, (size_t)C_COUNT * 2 * std::max(1, nmodes))) ||
      (e = sc.get(d_pts, (size_t)chunk)) || (e = sc.get(d_count, 1)))
    return fail(e);
  const ModeGroups mg{d_groups, (int)mt.groups.size(), nmodes};
  if ((e = cudaMemsetAsync(d_acc, 0, sizeof(double) * C_COUNT * 2 * std::max(1, nmodes), st))) return fail(e);
  // The interlaced pair is averaged: each mesh's nodes carry F / 2.
  const float scale = p.m == 2 ? 0.5f : 1.f;
  for (int j = 0; j < p.m; ++j)
    for (int64_t first = 0; first < n3 && nmodes > 0; first += chunk) {
      const int64_t cnt = std::min(chunk, n3 - first);
      if ((e = cudaMemsetAsync(d_count, 0, sizeof(unsigned), st))) return fail(e);
      k_sg_points_mesh<<<(unsigned)((cnt + 255) / 256), 256, 0, st>>>(
          p.d_mesh + j * n3, p.n, j, first, cnt, c.box_min[0] - c.observer[0], c.box_min[1] - c.observer[1],
          c.box_min[2] - c.observer[2], p.H, scale, d_count, d_pts);
      if ((e = cudaGetLastError())) return fail(e);
      if ((e = run_modes(c.ell_max, wedge, mg, d_pts, d_count, cnt, d_acc, st))) return fail(e);
    }
  return finish(mt, d_modes, d_acc, c.compensate ? p.d_invw : nullptr, p.n, p.d_sums, c.alpha, c.n_bins, c.ell_max,
                wedge, d_out, d_wedges, sc, st);
}
