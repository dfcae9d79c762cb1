// Steps 2-4 of the estimator (Sec. 3, Eqs. 5-13): the line-of-sight weighted fields,
// their 3D FFTs, the k-space combination into A_0, A_2, A_4, the Legendre products
// of Eqs. (6)-(8) and the |k|-shell sums.
//
// Data flow per mesh (x-major mesh F[ix][iy][iz]):
//  k_yz (persistent, ticketed work list; see the block comment above YZParams)
//     row item     one x-plane, R rows: the source fields F, F / |r|^d and F Z / |r|^d
//                  transformed along z (real lines in pairs), split into half spectra
//                  (k_z < nzc) and written to a ring slot laid out [k_z][source][y].
//     column item  KC k_z columns of one plane: sources times X^a Y^b are the basis fields,
//                  transformed along y, folded with k_y, k_z polynomial weights into
//                  the groups G_{n,p} (power p of k_x; GroupTable); only the pencils
//                  (k_y, k_z) with k_y^2 + k_z^2 < n2_hi are written, layout
//                  [mesh][group][pencil block][x][pencil].
//  k_x_combine  P pencils per CTA, tiles loaded by TMA: FFT along x of every group of
//             every mesh, interlacing phase and window compensation per mode, A_0
//             and k^n A_n = sum_p k_x^p G_{n,p}, then w |A_0|^2, w Re A_0 A_2^*,
//             w Re A_0 A_4^* (and w Re A_0 A_6^* for l_max = 6, the same
//             decomposition one order up) summed per shell: per-warp float bins, each with a
//             companion bin that collects the exact rounding error of every add
//             (so the pair carries the sum to ~2^-48), folded into the FP64 global
//             accumulators once per CTA.
//  k_finalize   alpha, I, S and Eqs. (6)-(8) per shell.
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>

#include <cstdint>

#include "fft.cuh"
#include "ys_internal.h"

namespace ys {

#include "group_table.inc"

// Source fields and basis fields.  A basis field is F times r_hat_x^a r_hat_y^b
// r_hat_z^c of degree d = a + b + c in {2, 4, 6} (c <= 1), or F itself, or F without the
// node at r = 0 (F').  With r = (X, Y, Z) from the observer and X, Y fixed along a
// z-line, the field is X^a Y^b times the source field h_{c,d} = F Z^c / |r|^d: the
// factor passes through the z transform, so only the sources (F and, per degree,
// c = 0 and 1: 5 real lines instead of 16 for l_max = 4) are transformed along z, and
// the y stage multiplies their spectra by X^a Y^b before its own transforms.
//   source 0: F;  sources 1 + 2 u, 2 + 2 u: F / |r|^d and F Z / |r|^d, d = 2 u + 2.
// F' needs no line of its own: it differs from F at one node at most, whose
// transform is a phase (see column_fold).
//
// Ranges.  r is held in units of a power of two near the largest |r| component (the
// monomials have degree 0, so the unit cancels exactly).  The sources of one row are
// scaled by rho^(d - c) and X, Y divided by rho, rho = max(2^floor(log2 |X|),
// 2^floor(log2 |Y|)), at least 2^-90.  With rho within a factor of two of the row's
// distance from the z axis through the observer, both sources of a degree, which share
// a complex line, and the factors (X / rho)^a (Y / rho)^b are O(F) and O(1): neither
// source's rounding shows in the other's field (one rho per x-plane instead lost 3.5
// bits next to the observer's planes), and nothing overflows next to the observer.
// (|r| / rho)^2 is at least 1 except at r = 0, the one node without a line-of-sight weight
// (its components are 0, see YZ_EXP_MIN); it is cut at 2^125, where the sources are at most
// 2^-35 F, so that rows much nearer the axis than 2^-62 stay finite.
// Line l of a column item: basis field 0 (l = 0) or l + 1 (F' is left out); its source
// field and the exponents of X and Y.
template <int ELL>
struct YLines {
  static constexpr int NL = ELL == 0 ? 1 : GroupTable<ELL>::NB - 1;
  unsigned char src[NL], a[NL], b[NL];
  constexpr YLines() : src(), a(), b() {
    for (int l = 0; l < NL; ++l) {
      const int beta = l == 0 ? 0 : l + 1;
      const int d = GroupTable<ELL>::mono_c(beta, 3);
      src[l] = (unsigned char)(d == 0 ? 0 : d - 1 + GroupTable<ELL>::mono_c(beta, 2));
      a[l] = (unsigned char)GroupTable<ELL>::mono_c(beta, 0);
      b[l] = (unsigned char)GroupTable<ELL>::mono_c(beta, 1);
    }
  }
};
template <int ELL> __constant__ constexpr YLines<ELL> kYLines{};

// ---------------------------------------------------------------------------
// y,z stage: one persistent kernel over a ticketed work list.
//
// Planes p = 0 .. m N - 1 (mesh j = p / N, x index p % N).  Per plane there are NZ
// "row items" (R rows of the plane: the source fields, their transforms along z and the
// split into half spectra for k_z < nzc, written to a ring slot) and NY "column items"
// (KC k_z columns: the basis fields' transforms along y, the k_y, k_z polynomial fold
// into the k_x-power groups, written for the pencils of those columns).  Tickets are
// handed out in steps: step t = row items of plane t, then column items of plane t - D.
// Row items of plane p reuse ring slot p mod S once the column items of plane p - S are
// done; column items of plane p start once its row items are done.  Both waits are on
// per-plane completion counters (release / acquire), bounded in time; a CTA only
// ever waits on items claimed before its own, so the list cannot deadlock.
//
// What bounds it: instruction issue (512^3, l_max = 4: about half of the slots, 16 warps
// per SM at 128 registers; shared memory 57 % busy).  The interlaced pair at 512^3 took
// 12.1 ms when every basis field was transformed along z (16 real lines per row instead of
// 5) with radix-8 stages, 6.5 ms with source fields and line transforms, 5.7 ms with two
// barriers per item and the radix-2 twiddles left to the readers; l_max = 6 30.8, 13.9,
// 11.8 ms; 1024^3 87, 40, 35 ms; 256^3 interlaced 1.76, 1.19, 0.97 ms.
// ---------------------------------------------------------------------------

struct YZParams {
  const float* mesh;     // [m][N][N][N]
  const float2* rel;     // [m][2][N] x, y of node - observer v, and 2^-floor(log2 |v|) (2^90 for v = 0)
  const float* relz;     // [m][N] z of node - observer
  const float2* tw;      // [TWN] twiddles of the line transforms (LineFft<N>)
  float2* ring;          // [S][nzc][NF][N]
  float2* gout;          // [m][NG][ngb][N][gw] (GROUP_BLOCK)
  const int* col_off;    // [nzc + 1]
  int* done_z;           // [m N]
  int* done_y;           // [m N]
  int* ticket;           // [1]
  int* err;              // [1]
  int nzc, gw, ngb, m, S, D;
  int org[2][3];         // node at r = 0 of each mesh (x < 0: none)
  long long spin_limit;  // ns
  int skip_plane;        // >= 0: that plane's row items withhold their completion (test hook)
};

// Several catalogues of one configuration ("lanes", each with its own mesh, ring,
// counters, error flag and grouped output) in one launch: the ticket queue runs
// through lane 0's items, then lane 1's, and so on (end[l] = items of lanes 0..l).
// Items of different lanes never wait on each other, so the argument above holds
// lane by lane.  A single plan is the one-lane case.
struct YZMulti {
  YZParams lane[YZ_MAX_LANES];
  int end[YZ_MAX_LANES];
  int nlanes;
  int* ticket;
};


__device__ __forceinline__ int ld_acquire(const int* p) {
  int v;
  asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// Thread 0 waits until *addr >= target; false (and the error flag set) on timeout
// or when another CTA has already failed.
__device__ __forceinline__ unsigned long long globaltimer_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// Thread 0 waits until *addr >= target, for at most limit_ns nanoseconds; false (and
// the error flag set) on timeout, or when another CTA has already failed.
__device__ __forceinline__ bool wait_geq(const int* addr, int target, int* err, long long limit_ns) {
  const unsigned long long t0 = globaltimer_ns();
  long long it = 0;
  while (ld_acquire(addr) < target) {
    if ((++it & 31) == 0) {
      if (*reinterpret_cast<volatile int*>(err)) return false;
      if ((long long)(globaltimer_ns() - t0) > limit_ns) {
        atomicExch(err, 1);
        return false;
      }
    }
    __nanosleep(128);
  }
  return true;
}


template <int N, int ELL>
struct YZ {
  using L = LineFft<N>;
  static constexpr int NG = GroupTable<ELL>::NG;
  static constexpr int ND = ELL / 2;             // degrees 2, 4, 6: one complex line (c = 0, 1) per row each
  static constexpr int NF = 1 + 2 * ND;          // source fields
  static constexpr int NL = YLines<ELL>::NL;     // y lines per column
  static constexpr int TPL = L::TPL, LINE = L::LINE, R1 = L::R1;
  // 512 threads where a column's lines leave room for one CTA per SM only
  static constexpr int THREADS = (size_t)NL * LINE * sizeof(float2) > 100 * 1024 || N >= 768 ? 512 : 256;
  static constexpr int GROUPS = THREADS / TPL;   // lines transformed at once
  // Rows per row item: a line per thread group, at least 8 rows (64-byte runs in the
  // ring); half of that for l_max = 6 where the item's lines would take too much.
  static constexpr int R0 = ELL == 0 ? 2 * GROUPS : (N <= 256 ? (ELL == 6 ? GROUPS / 2 : GROUPS) : 8);
  static constexpr int R = R0 > N ? N : (N % R0 ? 8 : R0);
  // With twice as many groups as rows, half of the groups take the upper degrees and F.
  // (The half of a group is decided by its line, and the halves skip each other's transforms.)
  static constexpr bool SPLIT = ND > 1 && GROUPS >= 2 * R && warps_on_one_side<TPL>(GROUPS, R);
  static constexpr int DSPLIT = SPLIT ? (ND + 1) / 2 : ND;  // degrees of the first half
  static constexpr int RLINES = R * ND + R / 2;  // the F lines hold two rows each
  // Columns per column item: as many as the thread groups transform at once.
  static constexpr int kc() {
    int k = 1;
    while (2 * k * NL <= GROUPS && k < 16) k *= 2;
    return k;
  }
  static constexpr int KC = kc();
  static constexpr int CLINES = NL * KC;
  static constexpr int LPG = (CLINES + GROUPS - 1) / GROUPS;  // lines per thread group
  // whether the last warp has less to transform than the others in a column item
  static constexpr bool SLACK = TPL >= 32 && GROUPS * LPG > CLINES;
  static constexpr int LINES = (RLINES > CLINES ? RLINES : CLINES) * LINE;  // elements of the line buffers
  static constexpr int TWN = L::TWN;                                         // and of the twiddles
  static constexpr size_t smem = sizeof(float2) * (LINES + TWN);
  static_assert(N % R == 0, "rows per item must divide N");
  // Resident CTAs per SM the register budget is set for: two of 256 threads when their
  // shared memory fits the SM (228 KB, less 1 KB reserved per CTA), else one.
  static constexpr int MIN_BLOCKS = THREADS == 256 && 2 * (smem + 1024 + 64) <= 228 * 1024 ? 2 : 1;
};

// 1/x for a normal x > 0: the hardware approximation refined by one Newton-Raphson
// step, y' = y + y (1 - x y), which leaves it within about an ulp (the correctly
// rounded reciprocal costs a long instruction sequence per node).
__device__ __forceinline__ float recip_nr(float x) {
  const float y = __fdividef(1.f, x);
  return fmaf(y, fmaf(-x, y, 1.f), y);
}

// Row item: the source fields of R rows of one x-plane, transformed along z.  Each
// degree's two real fields (c = 0, 1) go through one complex line; F goes through
// half a line per row (rows 2 p and 2 p + 1 as real and imaginary part).  All lines of
// the item stay in shared memory, so one barrier separates the transforms from the
// split into half spectra, which writes runs of R rows to the ring slot
// [k_z][source][y].
// before_mid() is called by every thread between the transforms and the barrier before the
// split (it elects the threads that claim and wait); false after that barrier: give up.
template <int N, int ELL, class Mid>
__device__ __forceinline__ bool row_item(float2* S, const float2* tws, const float* __restrict__ plane, float2 X,
                                         const float2* __restrict__ rely, const float* __restrict__ relz, int row0,
                                         float2* __restrict__ zslot, int nzc, Mid&& before_mid, const int& ok_flag) {
  using Y = YZ<N, ELL>;
  using L = typename Y::L;
  constexpr int R = Y::R, LINE = L::LINE, R1 = L::R1, TPL = L::TPL, GROUPS = Y::GROUPS, ND = Y::ND, NF = Y::NF;
  const int t = threadIdx.x % TPL, g = line_of_group<TPL>(threadIdx.x / TPL);
  float2 tw[R1 - 1];
  load_twiddles<N>(tw, tws, t);
  const float2* wE = tws + L::TW2;
  if constexpr (ND > 0) {
#pragma unroll 1
    for (int r0 = 0; r0 < R; r0 += GROUPS) {
      const bool upper = Y::SPLIT && g >= R;
      const int r = r0 + g - (upper ? R : 0);
      const bool ok = R % GROUPS == 0 || r < R;
      if (TPL >= 32 && !ok) break;
      float f[R1], i2[R1], irho = 1.f;
      if (ok) {
        const float2 Yc = rely[row0 + r];
        irho = fminf(X.y, Yc.y);  // a power of two: every product with it is exact
        const float xs = X.x * irho, ys = Yc.x * irho, xy2 = fmaf(xs, xs, ys * ys);
        const float* frow = plane + (size_t)(row0 + r) * N + t;
#pragma unroll
        for (int k = 0; k < R1; ++k) f[k] = frow[k * TPL];
#pragma unroll
        for (int k = 0; k < R1; ++k) {
          const float zs = relz[t + k * TPL] * irho, r2 = fmaf(zs, zs, xy2);  // (|r| / rho)^2
          i2[k] = r2 > 0.f ? recip_nr(fminf(r2, 0x1p125f)) : 0.f;
          f[k] *= 0.5f;  // for line_halves
        }
      }
#pragma unroll
      for (int d = 0; d < ND; ++d) {
        float2 v[R1];
        if (ok) {
#pragma unroll
          for (int k = 0; k < R1; ++k) {
            f[k] *= i2[k];
            v[k] = make_float2(f[k], f[k] * (relz[t + k * TPL] * irho));
          }
        }
        if (Y::SPLIT && (d >= Y::DSPLIT) != upper) continue;
        line_fft<N>(v, S + (d * R + r) * LINE, t, tw, wE, ok);
      }
    }
  }
#pragma unroll 1
  for (int p0 = 0; p0 < R / 2; p0 += GROUPS) {
    const int p = p0 + g - (Y::SPLIT ? R : 0);
    const bool ok = p >= 0 && p < R / 2;
    if (TPL >= 32 && !ok) break;
    float2 v[R1];
    if (ok) {
      const float* frow = plane + (size_t)(row0 + 2 * p) * N + t;
#pragma unroll
      for (int k = 0; k < R1; ++k) v[k] = make_float2(0.5f * frow[k * TPL], 0.5f * frow[N + k * TPL]);
    }
    line_fft<N>(v, S + (ND * R + p) * LINE, t, tw, wE, ok);
  }
  before_mid();
  __syncthreads();
  if (!ok_flag) return false;
  // Two real lines per complex line: their half spectra.
  if constexpr (ND > 0) {
    constexpr int RL = R < 16 ? R : 16, KS = Y::THREADS / RL;
#pragma unroll 1
    for (int rb = 0; rb < R; rb += RL) {
      const int r = rb + threadIdx.x % RL;
#pragma unroll 1
      for (int d = 0; d < ND; ++d) {
        const float2* line = S + (d * R + r) * LINE;
        float2* out = zslot + (size_t)(1 + 2 * d) * N + row0 + r;
        for (int i = threadIdx.x / RL; i < L::HALF_ITEMS; i += KS)
          line_halves<N>(line, wE, i, nzc, [&](int kz, float2 A, float2 B) {
            float2* o = out + (size_t)kz * NF * N;
            o[0] = A;
            o[N] = B;
          });
      }
    }
  }
  {
    constexpr int PL = R / 2 < 16 ? R / 2 : 16, KS = Y::THREADS / PL;
#pragma unroll 1
    for (int pb = 0; pb < R / 2; pb += PL) {
      const int p = pb + threadIdx.x % PL;
      const float2* line = S + (ND * R + p) * LINE;
      float2* out = zslot + row0 + 2 * p;
      for (int i = threadIdx.x / PL; i < L::HALF_ITEMS; i += KS)
        line_halves<N>(line, wE, i, nzc, [&](int kz, float2 A, float2 B) {
          *reinterpret_cast<float4*>(out + (size_t)kz * NF * N) = make_float4(A.x, A.y, B.x, B.y);
        });
    }
  }
  return true;
}

// Fold of one column (k_z): the y transforms of the basis fields at k_y become the
// k_x-power groups, written for the column's pencils.  The column's lines start at S.
// F' at the plane of the node at r = 0 (org): the transform of F less that node's
// value times its phase.
template <int N, int ELL>
__device__ __forceinline__ void column_fold(const float2* S, const float2* wE, int kz, const int* __restrict__ col_off,
                                            float2* __restrict__ gout, int j, int ix, int gw, int ngb, const int* org,
                                            const float* __restrict__ mesh, int tid, int nthr) {
  using Y = YZ<N, ELL>;
  using L = typename Y::L;
  constexpr int NG = Y::NG, NL = Y::NL, LINE = L::LINE, M = N / L::E2;
  [[maybe_unused]] constexpr bool HOLD = NL <= 15;  // both halves of every line in registers
  const int p0 = col_off[kz];
  const int cnt = col_off[kz + 1] - p0;
  const int kymax = (cnt - 1) / 2;
  const size_t gstep = (size_t)ngb * N * gw;  // between groups
  float2* g0 = gout + j * NG * gstep + (size_t)ix * gw;
  const bool at_org = ELL > 0 && ix == org[0];
  float f0 = 0.f;
  if (at_org) f0 = mesh[((size_t)ix * N + org[1]) * N + org[2]];
  // line(l): the transform of the column's line l at k_y
  auto emit = [&](auto&& line, int ky) {
    const float2 F0 = line(0);
    float2 Fp = F0;
    if (at_org) {
      const int turn = (((ky * org[1] + kz * org[2]) % N) + N) % N;
      float sn, cs;
      sincospif((float)(2 * turn) / (float)N, &sn, &cs);
      Fp = make_float2(fmaf(-f0, cs, Fp.x), fmaf(f0, sn, Fp.y));
    }
    float2 gr[NG];
    GroupTable<ELL>::combine([&](int f) { return f == 0 ? F0 : (f == 1 ? Fp : line(f - 1)); }, (float)ky, (float)kz, gr);
    const int pen = p0 + kymax + ky;
    float2* gp = g0 + (size_t)(pen / GROUP_BLOCK) * N * gw + pen % GROUP_BLOCK;
#pragma unroll
    for (int gi = 0; gi < NG; ++gi) gp[gi * gstep] = gr[gi];
  };
  if constexpr (L::E2 == 1) {
    // Lanes start at a multiple of 16 of the line position (k_y = -kymax sits at
    // N - kymax), so each half-warp reads 16 consecutive, 16-aligned frequencies.
    const int lead = (N - kymax) & 15;
    for (int q = tid - lead; q < cnt; q += nthr) {
      if (q < 0) continue;
      const int ky = q - kymax;
      const float2* sp = S + L::slot(ky < 0 ? ky + N : ky);
      emit([&](int l) { return sp[l * LINE]; }, ky);
    }
  } else if constexpr (L::E2 == 2) {
    // slots of kappa hold the halves of k_y = kappa and kappa - N/2
    for (int kap = tid; kap < M; kap += nthr) {
      const bool up = kap <= kymax, dn = M - kap <= kymax;
      if (!up && !dn) continue;
      const float2* sp = S + L::slot(kap);
      const float2 w = wE[kap / L::R1];
      if constexpr (HOLD) {
        float2 Ta[NL], Tb[NL];
#pragma unroll
        for (int l = 0; l < NL; ++l) {
          const float4 q = *reinterpret_cast<const float4*>(sp + l * LINE);
          const float2 x = make_float2(q.x, q.y), y = cmul(make_float2(q.z, q.w), w);
          Ta[l] = cadd(x, y);
          Tb[l] = csub(x, y);
        }
        if (up) emit([&](int l) { return Ta[l]; }, kap);
        if (dn) emit([&](int l) { return Tb[l]; }, kap - M);
      } else {
#pragma unroll 1
        for (int half = 0; half < 2; ++half) {
          if (half ? !dn : !up) continue;
          const float2 sg = half ? make_float2(-1.f, -1.f) : make_float2(1.f, 1.f);
          emit([&](int l) {
            const float4 q = *reinterpret_cast<const float4*>(sp + l * LINE);
            return __ffma2_rn(cmul(make_float2(q.z, q.w), w), sg, make_float2(q.x, q.y));
          }, kap - half * M);
        }
      }
    }
  } else {
    // four quarters: unit (kappa, odd) gives k_y = kappa + odd M and kappa + (odd - 2) M
    for (int u = tid; u < 2 * M; u += nthr) {
      const int odd = u >= M ? 1 : 0, kap = u - odd * M;
      const int kya = kap + odd * M, kyb = kap + (odd - 2) * M;
      const bool up = kya <= kymax, dn = -kyb <= kymax;
      if (!up && !dn) continue;
      const float2* sp = S + L::slot(kap);
      float2 Ta[NL], Tb[NL];
#pragma unroll
      for (int l = 0; l < NL; ++l) {
        const float4 q0 = *reinterpret_cast<const float4*>(sp + l * LINE);
        const float4 q1 = *reinterpret_cast<const float4*>(sp + l * LINE + 2);
        const float2 x0 = make_float2(q0.x, q0.y), x1 = make_float2(q0.z, q0.w);
        const float2 x2 = make_float2(q1.x, q1.y), x3 = make_float2(q1.z, q1.w);
        if (odd) {
          const float2 s = csub(x0, x2), d = csub(x1, x3);
          Ta[l] = add_mi(s, d);
          Tb[l] = sub_mi(s, d);
        } else {
          const float2 s = cadd(x0, x2), d = cadd(x1, x3);
          Ta[l] = cadd(s, d);
          Tb[l] = csub(s, d);
        }
      }
      if (up) emit([&](int l) { return Ta[l]; }, kya);
      if (dn) emit([&](int l) { return Tb[l]; }, kyb);
    }
  }
}

// Column item: the y transforms of KC columns (k_z) of one plane.  A thread group
// loads a source line, multiplies it by (X / rho)^a (Y / rho)^b and transforms it, LPG
// lines in turn.  The exponents are uniform over the group, so the tests on their bits
// skip whole unrolled loops where a group is a warp or more.
template <int N, int ELL, class Mid>
__device__ __forceinline__ void column_item(float2* S, const float2* tws, const float2* __restrict__ zslot, int kz0,
                                            const YZParams& prm, int j, int ix, Mid&& before_mid) {
  using Y = YZ<N, ELL>;
  using L = typename Y::L;
  constexpr int LINE = L::LINE, R1 = L::R1, TPL = L::TPL, NF = Y::NF, NL = Y::NL, KC = Y::KC, LPG = Y::LPG;
  const int t = threadIdx.x % TPL, g = line_of_group<TPL>(threadIdx.x / TPL);
  const int ncol = min(KC, prm.nzc - kz0);
  const float2* __restrict__ rel = prm.rel + (size_t)j * 2 * N;
  const float2* __restrict__ rely = rel + N + t;
  const float2 X = rel[ix];
  {
    float2 tw[R1 - 1];
    load_twiddles<N>(tw, tws, t);
    const float2* wE = tws + L::TW2;
#pragma unroll 1
    for (int i = 0; i < LPG; ++i) {
      const int l = g * LPG + i, c = l / NL, ln = l - c * NL;
      const bool ok = c < ncol;
      if (TPL >= 32 && !ok) break;
      float2 v[R1];
      if (ok) {
        const float2* zl = zslot + ((size_t)(kz0 + c) * NF + kYLines<ELL>.src[ln]) * N + t;
#pragma unroll
        for (int k = 0; k < R1; ++k) v[k] = __ldcg(zl + k * TPL);
        if constexpr (ELL > 0) {
          const int ea = kYLines<ELL>.a[ln], eb = kYLines<ELL>.b[ln];
          if (ea | eb) {
            float2 u[R1];  // (X, Y) / rho, then its squares and fourth powers
            float K[R1];
#pragma unroll
            for (int k = 0; k < R1; ++k) {
              const float2 Yc = rely[k * TPL];
              const float irho = fminf(X.y, Yc.y);
              u[k] = __fmul2_rn(make_float2(X.x, Yc.x), make_float2(irho, irho));
              K[k] = (ea & 1) ? u[k].x : 1.f;
            }
            if (eb & 1) {
#pragma unroll
              for (int k = 0; k < R1; ++k) K[k] *= u[k].y;
            }
            if ((ea | eb) > 1) {
#pragma unroll
              for (int k = 0; k < R1; ++k) {
                u[k] = __fmul2_rn(u[k], u[k]);
                if (ea & 2) K[k] *= u[k].x;
                if (eb & 2) K[k] *= u[k].y;
              }
            }
            if (ELL >= 4 && (ea | eb) > 3) {
#pragma unroll
              for (int k = 0; k < R1; ++k) {
                u[k] = __fmul2_rn(u[k], u[k]);
                if (ea & 4) K[k] *= u[k].x;
                if (eb & 4) K[k] *= u[k].y;
              }
            }
#pragma unroll
            for (int k = 0; k < R1; ++k) v[k] = __fmul2_rn(v[k], make_float2(K[k], K[k]));
          }
        }
      }
      line_fft<N>(v, S + l * LINE, t, tw, wE, ok);
    }
  }
  if constexpr (Y::SLACK) before_mid();
  __syncthreads();  // every ring load is done, every line transformed
  if constexpr (!Y::SLACK) before_mid();
  // The ring lines of these columns are dead once read: drop them from L2 without a
  // write-back (the slot is rewritten only after this item's completion is
  // released).  A column is NF * N * 8 bytes, a whole number of 128-byte lines.
  {
    const float2* dead = zslot + (size_t)kz0 * NF * N;
    for (int c = threadIdx.x; c < ncol * (NF * N / 16); c += Y::THREADS)
      asm volatile("discard.global.L2 [%0], 128;" ::"l"(dead + c * 16) : "memory");
  }
  constexpr int NTHR = Y::THREADS / KC;
  const int c = threadIdx.x / NTHR;
  if (c < ncol)
    column_fold<N, ELL>(S + c * NL * LINE, tws + L::TW2, kz0 + c, prm.col_off, prm.gout, j, ix, prm.gw, prm.ngb, prm.org[j],
                        prm.mesh + (size_t)j * N * N * N, threadIdx.x % NTHR, NTHR);
}

// What a CTA does next: one item of the list, decoded from its ticket by one thread.
struct YZItem {
  int lane;   // -1: the list is at its end
  int plane;  // of the row or column item; -1: nothing to do (the list's ragged ends)
  int sub;    // row item index (< NZ), or NZ + column item index
  int ready;  // the items it depends on were done when it was claimed
};

// The completion counter that item `it` waits on, and its target; nullptr: none.
template <int N, int ELL>
__device__ __forceinline__ const int* yz_dependency(const YZMulti& pm, const YZItem& it, int& target) {
  using Y = YZ<N, ELL>;
  if (it.lane < 0 || it.plane < 0) return nullptr;
  const YZParams& prm = pm.lane[it.lane];
  if (it.sub >= N / Y::R) {  // column item: the plane's row items
    target = N / Y::R;
    return prm.done_z + it.plane;
  }
  if (it.plane < prm.S) return nullptr;  // row item: the column items of the ring slot's last plane
  target = (prm.nzc + Y::KC - 1) / Y::KC;
  return prm.done_y + (it.plane - prm.S);
}

// Decodes a ticket and looks once whether its dependency is met.
template <int N, int ELL>
__device__ __forceinline__ YZItem yz_decode(const YZMulti& pm, int ticket) {
  using Y = YZ<N, ELL>;
  constexpr int NZ = N / Y::R;
  YZItem it{-1, -1, 0, 0};
  if (ticket >= pm.end[pm.nlanes - 1]) return it;
  int l = 0;
  while (ticket >= pm.end[l]) ++l;
  const YZParams& prm = pm.lane[l];
  const int item = ticket - (l > 0 ? pm.end[l - 1] : 0);
  const int per_step = NZ + (prm.nzc + Y::KC - 1) / Y::KC;
  const int step = item / per_step;
  it.lane = l;
  it.sub = item - step * per_step;
  it.plane = it.sub < NZ ? (step < prm.m * N ? step : -1) : step - prm.D;
  if (it.plane < 0) it.plane = -1;
  int target = 0;
  const int* dep = yz_dependency<N, ELL>(pm, it, target);
  it.ready = dep == nullptr || ld_acquire(dep) >= target;
  return it;
}

// Completion of an item: the CTA is past a barrier after its last writes, and thread 0's
// release-add orders them (it is cumulative over the barrier).
__device__ __forceinline__ void signal_release(int* counter) {
  asm volatile("red.release.gpu.global.add.s32 [%0], 1;" ::"l"(counter) : "memory");
}

// One thread of the last warp, which has the least to transform, claims the next ticket
// when its own transforms of the item are done (of a column item without SLACK: after the
// middle barrier; the fold leaves the last warp idle first): the atomic's round trip, the
// decoding and one look at the next item's dependency (~1400 cycles) overlap the other
// warps' work, and the barrier that ends the item publishes the result.  Usually the dependency is met and the
// next item starts without another barrier: two per item (five with a wait, a completion
// and a hand-over barrier each).  A row item needs its ring slot only for the split, so
// there a wait delays the middle barrier only.  Claiming a whole item ahead delayed the
// items waiting on it too much.  Items wait only on items of earlier tickets, so the list
// cannot deadlock; a CTA signals its item before it waits for the next one's dependency.
template <int N, int ELL>
__global__ void __launch_bounds__(YZ<N, ELL>::THREADS, YZ<N, ELL>::MIN_BLOCKS) k_yz(const __grid_constant__ YZMulti pm) {
  using Y = YZ<N, ELL>;
  constexpr int R = Y::R, NZ = N / R;
  constexpr int CLAIM = Y::THREADS - 32, WAIT = Y::THREADS - 64;  // the claiming and the waiting thread
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ YZItem s_item[2];  // this item and the next
  __shared__ int s_ok;
  float2* work = reinterpret_cast<float2*>(smem_raw);
  // Twiddles of the line transforms (same N: the same for every lane).
  float2* tws = work + Y::LINES;
  for (int k = threadIdx.x; k < Y::TWN; k += Y::THREADS) tws[k] = pm.lane[0].tw[k];
  const size_t n3 = (size_t)N * N * N;
  if (threadIdx.x == CLAIM) s_item[0] = yz_decode<N, ELL>(pm, atomicAdd(pm.ticket, 1));
  if (threadIdx.x == 0) s_ok = 1;
  __syncthreads();
  for (int turn = 0;; turn ^= 1) {
    const YZItem it = s_item[turn];
    if (it.lane < 0) break;
    const YZParams& prm = pm.lane[it.lane];
    const bool row = it.sub < NZ;
    auto wait = [&]() {
      int target = 0;
      const int* dep = yz_dependency<N, ELL>(pm, it, target);
      if (!wait_geq(dep, target, prm.err, prm.spin_limit)) s_ok = 0;
    };
    if (!it.ready && !row) {
      if (threadIdx.x == WAIT) wait();
      __syncthreads();
      if (!s_ok) break;
    }
    auto before_mid = [&]() {
      if (threadIdx.x == CLAIM) s_item[turn ^ 1] = yz_decode<N, ELL>(pm, atomicAdd(pm.ticket, 1));
      if (threadIdx.x == WAIT && !it.ready && row) wait();
    };
    int* done = nullptr;
    const int p = it.plane, j = p / N, ix = p - j * N;
    if (p >= 0) {
      float2* slot = prm.ring + (size_t)(p % prm.S) * Y::NF * prm.nzc * N;
      const float* plane = prm.mesh + j * n3 + (size_t)ix * N * N;
      if (row) {
        // L2 prefetch of the next plane's rows, about one grid of tickets ahead
        if (p + 1 < prm.m * N && threadIdx.x < R * N / 32)
          asm volatile("prefetch.global.L2 [%0];" ::"l"(plane + (size_t)N * N + (size_t)it.sub * R * N +
                                                        threadIdx.x * 32));  // one 128-byte line each
        const float2* rel = prm.rel + (size_t)j * 2 * N;
        if (!row_item<N, ELL>(work, tws, plane, rel[ix], rel + N, prm.relz + (size_t)j * N, it.sub * R, slot, prm.nzc,
                              before_mid, s_ok))
          break;
        if (p != prm.skip_plane) done = prm.done_z + p;  // (withheld: its column items wait until their limit)
      } else {
        column_item<N, ELL>(work, tws, slot, (it.sub - NZ) * Y::KC, prm, j, ix, before_mid);
        done = prm.done_y + p;
      }
    } else {
      before_mid();
    }
    __syncthreads();  // every thread is past this item, and the next one is published
    if (threadIdx.x == 0 && done) signal_release(done);
  }
}


// The x stage of several lanes (catalogues of one configuration, as for k_yz) in one
// launch: grid (blocks per lane, lanes); the tables (pencils, twiddles, window, phases,
// shell lookup) are the configuration's and the same for every lane.
struct XMulti {
  CUtensorMap map[YZ_MAX_LANES];
  double* acc[YZ_MAX_LANES];
  int* err[YZ_MAX_LANES];
  int nlanes;
};

// First group of multipole slot s (groups: A_0 | l = 2, powers 0..2 of k_x | l = 4,
// powers 0..4 | l = 6, powers 0..6): s^2; its last is s^2 + 2 s.
//
// Group transformed at tile position q of a pencil block: the powers of k_x of each
// multipole come highest first, so that they are summed by Horner's rule.
__host__ __device__ constexpr int group_slot(int g) { return g == 0 ? 0 : (g <= 3 ? 1 : (g <= 8 ? 2 : 3)); }
__host__ __device__ constexpr int tile_group(int q) {
  const int s = group_slot(q);
  return 2 * s * s + 2 * s - q;
}

// Whether the x stage carries the rounding errors of the Horner sums of each multipole
// (see k_x_combine): always for l_max = 6, and for l_max = 2, 4 except at 256^3 and
// 512^3, where the x stage is held to 80 registers for three CTAs per SM and the extra
// error terms would spill (shells there hold many modes, and the plain sums meet the
// parity bar with a wide margin).  The rule goes by the mesh size alone, so that a plan's
// accuracy does not depend on the tile size the autotuner picks.
template <int N, int ELL>
__host__ __device__ constexpr bool x_horner() { return ELL == 6 || (ELL >= 2 && N != 256 && N != 512); }

// ---------------------------------------------------------------------------
// x stage: FFT along x of every (mesh, group) tile of P pencils, fed by TMA.
// The grouped y,z transforms are a 2D tensor [m NG ngb N rows][gw pencils] of
// float2; one tile (all N rows x P pencils) arrives by BOXES 2D bulk-tensor copies
// in a shared buffer (mbarrier completion).  Its first FFT stage moves it to the work
// buffer, and the copy of a later tile overlaps the other stages, which run in
// place there.  The last FFT stage stays in registers: each thread owns E modes (one
// pencil, E values of k_x) for the whole pencil block.
//
// Per multipole and mesh the powers of k_x are summed by Horner's rule, one FMA per
// component and tile; the interlacing phase, the window and the mean over the two meshes
// are common to all powers and applied once, when the multipole is complete.  A_0 waits
// in shared memory for the other multipoles.  The per-mode terms of the shell sums go to
// compensated per-warp float bins in shared memory, folded into the FP64 accumulators
// when the CTA ends.
// ---------------------------------------------------------------------------

__device__ __forceinline__ unsigned smem_u32(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(unsigned long long* bar, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(unsigned long long* bar, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}

__device__ __forceinline__ void tma_load_2d(void* dst, const CUtensorMap* map, int x, int y,
                                            unsigned long long* bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(
          smem_u32(dst)),
      "l"(map), "r"(x), "r"(y), "r"(smem_u32(bar))
      : "memory");
}

// Wait for an mbarrier phase (by parity) for at most limit_ns nanoseconds; false on timeout.
__device__ __forceinline__ bool mbar_wait(unsigned long long* bar, unsigned parity, long long limit_ns) {
  unsigned long long t0 = 0;
  for (;;) {
    unsigned ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    if (ok) return true;
    const unsigned long long t = globaltimer_ns();
    if (t0 == 0) t0 = t;
    else if ((long long)(t - t0) > limit_ns) return false;
  }
}

// Exact rounding error (a + b) - fl(a + b) of a float add (Knuth's TwoSum).
// The shell bins use it with shared-memory atomics: the atomic returns the value it
// added to, so the stored sum is fl(old + v), and two_sum_err(old, v) is the exact
// error of that add whatever other threads add before or after; it goes into a
// companion bin.  Summed over every add, sum + companion equals the exact sum up to
// the companion's own rounding, a relative ~2^-24 of the errors themselves: the pair
// accumulates like FP64 on the FP32 pipes (FP64 arithmetic on this GPU runs at a
// small fraction of FP32).  The atomic flushes a subnormal sum to zero; that changes
// the error by less than 2^-126.
__device__ __forceinline__ float two_sum_err(float a, float b) {
  const float s = a + b;
  const float bb = s - a;
  return (a - (s - bb)) + (b - bb);
}

// The same for both components of a complex sum s = a + b.
__device__ __forceinline__ float2 two_sum_err2(float2 a, float2 b, float2 s) {
  const float2 bb = csub(s, a);
  return cadd(csub(a, csub(s, bb)), csub(b, bb));
}

template <int N, int ELL, int M, int PX = k3_pencils(N)>
struct XCombine {
  static constexpr int P = PX;  // pencils per CTA
  static constexpr int E = fft_elems(N);
  static constexpr int TPL = N / E;
  static constexpr int THREADS = P * TPL;
  static constexpr int NW = THREADS / 32;
  static constexpr int NG = GroupTable<ELL>::NG;
  // shell-sum slots: |A_0|^2, Re A_0 A_2^*, Re A_0 A_4^* (and Re A_0 A_6^* for l = 6)
  static constexpr int SLOTS = ELL / 2 + 1;
  static constexpr int TILES = NG * M;
  static constexpr int BOX_ROWS = x_box_rows(N);
  static constexpr int BOXES = N / BOX_ROWS;
  static_assert(BOXES * BOX_ROWS == N, "boxes must tile the x axis");
  static constexpr unsigned TILE_BYTES = (unsigned)(N * P * sizeof(float2));
  static constexpr int STAGES = fft_nstages(N);
  // tile buffers: one where several CTAs per SM hide the copies, more for small meshes,
  // whose few CTAs would wait for each (128^3 49.2 -> 46.5 us, 32^3 20.4 -> 19.6 us)
  static constexpr int NBUF = N <= 128 ? 4 : 1;
  static constexpr int WK_ELEMS = lf_elems<N, P>();
  static constexpr int RL = fft_radix(N, STAGES - 1);  // last radix
  // resident CTAs per SM the register budget is set for (3 x 256 threads at 256^3, 512^3;
  // 2 where the sums' errors are carried)
  static constexpr int MIN_BLOCKS = THREADS != 256 || E != 8 ? 1 : (x_horner<N, ELL>() ? 2 : 3);
  static_assert(THREADS % 32 == 0, "threads");
  // nwb copies of the compensated float shell bins: a sum and an error term per shell
  // and slot.  With nwb = NW c (c copies per warp) the lanes of pencil p add into copy
  // p mod c of their warp's: the run-reduced sums of different pencils, which often fall
  // in one shell, then never meet in one instruction (same-address shared atomics are
  // served one after another); with fewer copies warp w adds into copy w mod nwb.
  static size_t smem(int nbins, int nwb) {
    size_t b = NBUF * (size_t)TILE_BYTES + sizeof(float2) * WK_ELEMS;  // tile buffers and work buffer
    if (ELL > 0) b += TILE_BYTES;                       // A_0
    b += sizeof(float2) * 2 * N + sizeof(float) * N;    // twiddles, phases, windows
    b += sizeof(float) * 2 * nwb * SLOTS * nbins;       // float bins and their error terms
    return b;
  }
};

template <int N, int ELL, int M, int PX>
__global__ void __launch_bounds__(XCombine<N, ELL, M, PX>::THREADS, XCombine<N, ELL, M, PX>::MIN_BLOCKS)
k_x_combine(const __grid_constant__ XMulti pm, int np_pad, int ngb, const short2* __restrict__ pencil,
            const float2* __restrict__ tw_g, const float* __restrict__ invw_g, const float2* __restrict__ phase_g,
            const short* __restrict__ lut, int n2_hi, int nbins, int nwb) {
  // lane blockIdx.y: its grouped transforms (tensor map), shell accumulators, error flag
  const CUtensorMap* gmap = &pm.map[blockIdx.y];
  using XC = XCombine<N, ELL, M, PX>;
  constexpr int P = XC::P, E = XC::E, TPL = XC::TPL, TILES = XC::TILES, RL = XC::RL, SLOTS = XC::SLOTS;
  constexpr int THREADS = XC::THREADS;
  constexpr bool COMP = x_horner<N, ELL>();
  extern __shared__ __align__(128) float2 smem_x[];
  __shared__ __align__(8) unsigned long long bar[XC::NBUF];
  __shared__ int s_fail;
  float2* T = smem_x;
  constexpr int NBUF = XC::NBUF;
  float2* Wk = T + NBUF * N * P;
  float2* sA0 = Wk + XC::WK_ELEMS;
  float2* tw = sA0 + (ELL > 0 ? N * P : 0);
  float2* phs = tw + N;
  float* invw = reinterpret_cast<float*>(phs + N);
  float* wbin = invw + N;                    // [nwb][SLOTS][nbins] sums
  float* wcmp = wbin + nwb * SLOTS * nbins;  // [nwb][SLOTS][nbins] their rounding errors
  const int tid = threadIdx.x, warp = tid >> 5;
  for (int k = tid; k < N; k += THREADS) {
    tw[k] = tw_g[k];
    phs[k] = phase_g[k];
    invw[k] = invw_g[k];
  }
  for (int k = tid; k < 2 * nwb * SLOTS * nbins; k += THREADS) wbin[k] = 0.f;
  if (tid == 0) {
    for (int b = 0; b < NBUF; ++b) mbar_init(&bar[b], 1);
    s_fail = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  const int npb = np_pad / P;
  const int mine = blockIdx.x < npb ? (npb - 1 - blockIdx.x) / gridDim.x + 1 : 0;
  const int total = mine * TILES;
  auto issue = [&](int s) {  // thread 0: the copy of tile s
    const int k = s / TILES, t = s - k * TILES;
    const int gi = tile_group(t / M), mj = t % M;
    const int pen = (blockIdx.x + k * gridDim.x) * P;  // a block of P pencils lies in one pencil block
    const int row = ((mj * XC::NG + gi) * ngb + pen / GROUP_BLOCK) * N;
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    unsigned long long* bs = &bar[s % NBUF];
    float2* dst = T + (s % NBUF) * N * P;
    mbar_expect_tx(bs, XC::TILE_BYTES);
#pragma unroll
    for (int bx = 0; bx < XC::BOXES; ++bx)
      tma_load_2d(dst + bx * XC::BOX_ROWS * P, gmap, pen % GROUP_BLOCK * 2, row + bx * XC::BOX_ROWS, bs);
  };
  if (tid == 0)
    for (int q = 0; q < NBUF && q < total; ++q) issue(q);
  const int p = tid % P, tl = tid / P;
  const float m0 = (float)tl;
  // mode e of this thread: k_x = tl + koff(e), as a signed frequency tl + koff(e) - N past N / 2
  auto koff = [](int e) { return (e / RL) * TPL + (e % RL) * (N / RL); };
  auto msign = [&](int e) { return koff(e) < N / 2 ? koff(e) : koff(e) - N; };
  const int copy = nwb >= XC::NW ? warp * (nwb / XC::NW) + p % (nwb / XC::NW) : warp % nwb;
  float* wb0 = wbin + copy * SLOTS * nbins;
  const int cmp_off = nwb * SLOTS * nbins;
  int s = 0;
  bool failed = false;
  for (int k = 0; k < mine && !failed; ++k) {
    const short2 pc = pencil[(blockIdx.x + k * gridDim.x) * P + p];
    const int ky = pc.x, kz = pc.y;  // kz < 0: a padding pencil, no shell
    const int iyk = ky < 0 ? ky + N : ky, kzc = kz < 0 ? 0 : kz;
    const int kyz2 = ky * ky + kz * kz;
    const float cf_pen = invw[iyk] * invw[kzc] * (M == 2 ? 0.5f : 1.f);
    const float2 ph_pen = cmul(phs[iyk], phs[kzc]);
    const float wgt = kz == 0 ? 1.f : 2.f;
    unsigned keys[(E + 1) / 2];  // shells of this thread's modes (16 bits each; 0xffff: none)
#pragma unroll
    for (int e = 0; e < E; ++e) {
      const int mx = tl + msign(e), n2 = mx * mx + kyz2;
      const unsigned key = (kz >= 0 && n2 < n2_hi) ? (unsigned short)lut[n2] : 0xffffu;
      if (e & 1) keys[e / 2] |= key << 16;
      else keys[e / 2] = key;
    }
#pragma unroll 1
    for (int slot = 0; slot < SLOTS && !failed; ++slot) {
      float2 H[M][E];               // Horner sums of each mesh
      float2 C[COMP ? M : 1][COMP ? E : 1];  // and their rounding errors
#pragma unroll
      for (int mj = 0; mj < M; ++mj)
#pragma unroll
        for (int e = 0; e < E; ++e) {
          H[mj][e] = make_float2(0.f, 0.f);
          if constexpr (COMP) C[mj][e] = make_float2(0.f, 0.f);
        }
#pragma unroll 1
      for (int q = 0; q <= 2 * slot && !failed; ++q) {
#pragma unroll
        for (int mj = 0; mj < M; ++mj) {
          float2 v[E];
          if (!mbar_wait(&bar[s % NBUF], (s / NBUF) & 1, 1000000000LL)) s_fail = 1;  // 1 s
          lf_first_stage<N, P>(T + (s % NBUF) * N * P, Wk, p, tl);
          __syncthreads();
          if (s_fail) {
            failed = true;
            break;
          }
          if (tid == 0 && s + NBUF < total) issue(s + NBUF);
          LfMiddle<N, P, 1>::run(Wk, p, tl, tw);
          lf_last_stage<N, P>(Wk, p, tl, tw, v);  // (a barrier after its loads)
          ++s;
#pragma unroll
          for (int e = 0; e < E; ++e) {
            const float m = m0 + (float)msign(e);
            if constexpr (COMP) {
              // every step error-free: the product by the integer m is split exactly with
              // an FMA and the add with TwoSum, and both errors go to C
              const float2 mm = make_float2(m, m);
              const float2 pr = __fmul2_rn(H[mj][e], mm);
              const float2 er = __ffma2_rn(H[mj][e], mm, make_float2(-pr.x, -pr.y));
              H[mj][e] = cadd(pr, v[e]);
              C[mj][e] = cadd(__ffma2_rn(C[mj][e], mm, er), two_sum_err2(pr, v[e], H[mj][e]));
            } else {
              H[mj][e].x = fmaf(H[mj][e].x, m, v[e].x);
              H[mj][e].y = fmaf(H[mj][e].y, m, v[e].y);
            }
          }
        }
      }
      if (failed) break;
      // The lanes of one pencil (lane = p + P j, j < 32 / P) hold neighbouring k_x and
      // mostly share a shell: each run of equal shells (cut wherever neighbouring lanes
      // differ) is first summed across its lanes by a segmented suffix scan with
      // compensated adds, and only the run's first lane adds it to the bins.
      const int jl = (tid & 31) / P;
      constexpr int LG = 32 / P;
      float* wb = wb0 + slot * nbins;
#pragma unroll
      for (int e = 0; e < E; ++e) {
        const int kx = tl + koff(e);
        float2 A = H[0][e];
        if constexpr (COMP) A = cadd(A, C[0][e]);
        if constexpr (M == 2) {
          float2 B = H[M - 1][e];
          if constexpr (COMP) B = cadd(B, C[M - 1][e]);
          B = cmul(B, cmul(phs[kx], ph_pen));
          A = cadd(A, B);
        }
        const float c = cf_pen * invw[kx];
        A = make_float2(c * A.x, c * A.y);
        float val;
        if (slot == 0) {
          if (ELL > 0) sA0[e * THREADS + tid] = A;
          val = wgt * (A.x * A.x + A.y * A.y);
        } else {
          const float2 a0 = sA0[e * THREADS + tid];
          const int mx = tl + msign(e);
          const float inv = 1.f / (float)(mx * mx + kyz2);
          const float ik = slot == 1 ? inv : (slot == 2 ? inv * inv : inv * inv * inv);  // 1 / k^(2 slot)
          val = wgt * ik * (a0.x * A.x + a0.y * A.y);
        }
        const unsigned key = (e & 1) ? keys[e / 2] >> 16 : keys[e / 2] & 0xffffu;
        if (__all_sync(0xffffffffu, key == 0xffffu)) continue;  // no lane's mode is in a shell
        const unsigned key_next = __shfl_down_sync(0xffffffffu, key, P);
        const unsigned key_prev = __shfl_up_sync(0xffffffffu, key, P);
        int end = (jl == LG - 1 || key_next != key) ? 1 : 0;  // this lane's run stops here
        float cmp = 0.f;
#pragma unroll
        for (int d = P; d < 32; d <<= 1) {
          const float vn = __shfl_down_sync(0xffffffffu, val, d);
          const float cn = __shfl_down_sync(0xffffffffu, cmp, d);
          const int en = __shfl_down_sync(0xffffffffu, end, d);
          if (!end) {  // the run reaches lane + d, inside this pencil's lanes
            cmp += cn + two_sum_err(val, vn);
            val += vn;
            end = en;
          }
        }
        if (key != 0xffffu && (jl == 0 || key_prev != key)) {
          const float old = atomicAdd(wb + key, val);
          const float err = cmp + two_sum_err(old, val);
          if (err != 0.f) atomicAdd(wb + cmp_off + key, err);
        }
      }
    }
  }
  if (failed) {
    if (tid == 0) {
      atomicExch(pm.err[blockIdx.y], 2);
      // Copies s .. s + NBUF - 1 are the last ones issued: wait for each by its own phase
      // parity before the CTA's shared memory is released (bounded; every earlier copy
      // has completed).
      for (int q = s; q < s + NBUF && q < total; ++q) mbar_wait(&bar[q % NBUF], (q / NBUF) & 1, 100000000LL);
    }
    return;
  }
  __syncthreads();
  // FP64 fold of every warp copy's sum and error term, once per CTA.
  double* __restrict__ acc = pm.acc[blockIdx.y];
  for (int b = tid; b < SLOTS * nbins; b += THREADS) {
    double v = 0.0;
    for (int w = 0; w < nwb; ++w) v += (double)wbin[w * SLOTS * nbins + b] + (double)wcmp[w * SLOTS * nbins + b];
    if (v != 0.0) atomicAdd(&acc[b], v);
  }
}

}  // namespace ys
