// Shared-memory complex FFTs for the mesh transforms (forward, e^{-2 pi i j k / N}).
//
// The method (Sec. 3) places no condition on the FFT algorithm.  N is 2^a or 3 * 2^a, and
// results come out in natural order.
//   y,z stage: lines walked by consecutive threads, 16 (12) elements per thread, two
//     large radices and a small last one done by the reader (LineFft, below).
//   x stage: interleaved lines, a Stockham autosort transform with 8 (12) elements per
//     thread: radix-8 stages, then one radix-4 or radix-2; for 3 * 2^a a radix-12 stage,
//     then radix-4 stages and an optional radix-2.  The data go through shared memory
//     between stages.
// Twiddles come from tables computed in FP64 on the host and rounded to float.
#pragma once
#include <cuda_runtime.h>

#include <type_traits>

namespace ys {

__host__ __device__ constexpr bool is_pow2(int n) { return n > 0 && (n & (n - 1)) == 0; }

// Elements per thread of the x stage's interleaved lines.
__host__ __device__ constexpr int fft_elems(int n) { return is_pow2(n) ? 8 : 12; }

// Barrier over the TPL consecutive threads that own one line: the warp when the
// line fits in it, else a named barrier (ids 1..15) shared by those threads only.
template <int TPL>
__device__ __forceinline__ void line_group_sync() {
  if constexpr (TPL <= 32) {
    __syncwarp();
  } else {
    asm volatile("bar.sync %0, %1;" ::"r"(1 + (int)(threadIdx.x / TPL)), "r"(TPL) : "memory");
  }
}

// Radix of stage s of the x stage's transform, and the number of stages.
__host__ __device__ constexpr int fft_radix(int n, int stage) {
  int m = n, big = 8;
  if (!is_pow2(n)) {
    if (stage == 0) return 12;
    m = n / 12;
    big = 4;
    --stage;
  }
  for (; m >= big; m /= big, --stage)
    if (stage == 0) return big;
  return m;
}

__host__ __device__ constexpr int fft_nstages(int n) {
  int s = 0;
  for (int m = n; m > 1; ++s) m /= fft_radix(n, s);
  return s;
}

__host__ __device__ constexpr int fft_ns_before(int n, int stage) {
  int ns = 1;
  for (int s = 0; s < stage; ++s) ns *= fft_radix(n, s);
  return ns;
}

__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
  return make_float2(fmaf(a.x, b.x, -a.y * b.y), fmaf(a.x, b.y, a.y * b.x));
}
// Complex sums and differences use the packed two-lane float instructions of
// sm_100-class GPUs (one instruction for both components).  a - b is formed as
// fma(b, -1, a), whose product is exact, so it rounds exactly as a - b does.
__device__ __forceinline__ float2 cadd(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 csub(float2 a, float2 b) { return __ffma2_rn(b, make_float2(-1.f, -1.f), a); }
__device__ __forceinline__ float2 cswap(float2 a) { return make_float2(a.y, a.x); }
// a + (-i) t and a - (-i) t
__device__ __forceinline__ float2 add_mi(float2 a, float2 t) { return __ffma2_rn(cswap(t), make_float2(1.f, -1.f), a); }
__device__ __forceinline__ float2 sub_mi(float2 a, float2 t) { return __ffma2_rn(cswap(t), make_float2(-1.f, 1.f), a); }
// a + s t for a real s given as (s, s)
__device__ __forceinline__ float2 cfma(float2 t, float2 s, float2 a) { return __ffma2_rn(t, s, a); }

template <int R> struct Dft;

template <> struct Dft<2> {
  __device__ static __forceinline__ void run(float2* v) {
    const float2 a = v[0], b = v[1];
    v[0] = cadd(a, b);
    v[1] = csub(a, b);
  }
};

template <> struct Dft<3> {
  __device__ static __forceinline__ void run(float2* v) {
    // w = e^{-2 pi i / 3} = -1/2 - i sqrt(3)/2
    const float s3 = 0.866025403784438647f;
    const float2 a = v[0], b = v[1], c = v[2];
    const float2 t1 = cadd(b, c);
    const float2 t2 = cfma(t1, make_float2(-0.5f, -0.5f), a);
    const float2 d = csub(b, c);
    // t2 +/- (-i sqrt3/2) d
    v[0] = cadd(a, t1);
    v[1] = cfma(cswap(d), make_float2(s3, -s3), t2);
    v[2] = cfma(cswap(d), make_float2(-s3, s3), t2);
  }
};

template <> struct Dft<4> {
  __device__ static __forceinline__ void run(float2* v) {
    const float2 a = v[0], b = v[1], c = v[2], d = v[3];
    const float2 s0 = cadd(a, c), s1 = csub(a, c);
    const float2 s2 = cadd(b, d), t = csub(b, d);
    v[0] = cadd(s0, s2);
    v[2] = csub(s0, s2);
    v[1] = add_mi(s1, t);
    v[3] = sub_mi(s1, t);
  }
};

template <> struct Dft<8> {
  __device__ static __forceinline__ void run(float2* v) {
    // even / odd split into two DFT-4s, then w8^k = e^{-i pi k / 4}.
    const float h = 0.707106781186547524f;
    float2 e[4] = {v[0], v[2], v[4], v[6]};
    float2 o[4] = {v[1], v[3], v[5], v[7]};
    Dft<4>::run(e);
    Dft<4>::run(o);
    // w8 o1 = h u1 with u1 = (o1.x + o1.y, o1.y - o1.x); w8^3 o3 = -h u3 with
    // u3 = (o3.x - o3.y, o3.y + o3.x); w8^2 o2 = -i o2.
    const float2 u1 = add_mi(o[1], o[1]);
    const float2 u3 = sub_mi(o[3], o[3]);
    v[0] = cadd(e[0], o[0]);
    v[4] = csub(e[0], o[0]);
    v[1] = cfma(u1, make_float2(h, h), e[1]);
    v[5] = cfma(u1, make_float2(-h, -h), e[1]);
    v[2] = add_mi(e[2], o[2]);
    v[6] = sub_mi(e[2], o[2]);
    v[3] = cfma(u3, make_float2(-h, -h), e[3]);
    v[7] = cfma(u3, make_float2(h, h), e[3]);
  }
};

// 16 = 4 x 4: DFT-4 over the inputs 4 a + b for each b, twiddles w16^(b k1), DFT-4 over b.
//
// LONG, for lines whose second radix is 16 too: cos(pi / 8) rounded up.  The nearest float makes
// |c1 - i s1| 2.9e-8 short, which with h (1.7e-8 short) biases every mode the same way: over a
// line of 256 (512) the mean gain was 2.7e-8 (3.4e-8) short, 2.1e-8 (2.4e-8) with radix-8 stages,
// and P_0 1.4e-7 (1.6e-7) low.  One float up it is 2.7e-8 long and cancels h: mean gains 1e-9 and
// 6e-9 short, P_0 4e-8 and 5e-8 low.  Lines with one radix-16 stage gain nothing (their gain is
// that of radix 8) and would take the larger phase error, 1.8e-8 instead of 0.5e-8: P_2 of a
// 32^3 mesh was off by 1.1 times as much.
template <bool LONG>
struct Dft16 {
  __device__ static __forceinline__ void run(float2* v) {
    const float h = 0.707106781186547524f, s1 = 0.382683432365089772f;
    const float c1 = LONG ? 0.92387956380844116f : 0.923879532511286756f;
    float2 t[4][4];  // [k1][b]
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      float2 u[4] = {v[b], v[4 + b], v[8 + b], v[12 + b]};
      Dft<4>::run(u);
#pragma unroll
      for (int k = 0; k < 4; ++k) t[k][b] = u[k];
    }
    t[1][1] = cmul(t[1][1], make_float2(c1, -s1));
    t[1][3] = cmul(t[1][3], make_float2(s1, -c1));
    t[3][1] = cmul(t[3][1], make_float2(s1, -c1));
    t[3][3] = cmul(t[3][3], make_float2(-c1, s1));
    t[1][2] = __fmul2_rn(add_mi(t[1][2], t[1][2]), make_float2(h, h));    // w16^2 = h (1 - i)
    t[2][1] = __fmul2_rn(add_mi(t[2][1], t[2][1]), make_float2(h, h));
    t[2][3] = __fmul2_rn(sub_mi(t[2][3], t[2][3]), make_float2(-h, -h));  // w16^6 = -h (1 + i)
    t[3][2] = __fmul2_rn(sub_mi(t[3][2], t[3][2]), make_float2(-h, -h));
    t[2][2] = make_float2(t[2][2].y, -t[2][2].x);                         // w16^4 = -i
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      Dft<4>::run(t[k]);
#pragma unroll
      for (int q = 0; q < 4; ++q) v[k + 4 * q] = t[k][q];
    }
  }
};

// 12 = 3 x 4 with coprime factors: inputs (4 a + 3 b) mod 12, outputs (4 k + 9 q) mod 12,
// no twiddles (the prime-factor mapping).
template <> struct Dft<12> {
  __device__ static __forceinline__ void run(float2* v) {
    float2 t[3][4];
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      float2 u[3] = {v[(3 * b) % 12], v[(4 + 3 * b) % 12], v[(8 + 3 * b) % 12]};
      Dft<3>::run(u);
#pragma unroll
      for (int k = 0; k < 3; ++k) t[k][b] = u[k];
    }
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      Dft<4>::run(t[k]);
#pragma unroll
      for (int q = 0; q < 4; ++q) v[(4 * k + 9 * q) % 12] = t[k][q];
    }
  }
};

template <> struct Dft<1> {
  __device__ static __forceinline__ void run(float2*) {}
};

// ---------------------------------------------------------------------------
// Line transforms of the y,z stage: one line of N complex elements by TPL consecutive
// threads with R1 = 16 (12) elements each, N = R1 R2 E2.
//   1. Thread t holds x[t + TPL r] and does one radix-R1 butterfly in registers,
//      multiplies by exp(-2 pi i t k1 / N) and stores element (k1, t) at k1 P + t.
//   2. Butterfly (k1, e), e < E2, takes (k1, e + E2 s), s < R2, through a radix-R2
//      butterfly, multiplies by exp(-2 pi i e q / (R2 E2)) (E2 = 4) and puts the results
//      back where its inputs were.
//   3. The reader does the last radix E2 (1, 2 or 4) on the E2 neighbouring elements
//      of a slot: frequency kappa + (N / E2) h, kappa = k1 + R1 q, is
//      sum_e exp(-2 pi i e h / E2) element[slot(kappa) + e], the second element of an
//      E2 = 2 slot times exp(-2 pi i q / (2 R2)) (in step 2 half of the lanes would idle).
// A line thus crosses shared memory twice (three times with radix-8 stages of 8
// elements per thread at N = 512), and its twiddles stay in registers.  The pitch P
// and the line length LINE keep every access conflict-free: the E2 elements of a slot
// are adjacent and a warp's k1 step through the banks by E2 (steps 1 and 2), and
// LINE is odd in units of a slot's (at most 16-byte) load, for readers that go across lines.
// ---------------------------------------------------------------------------
template <int N>
struct LineFft {
  static constexpr bool P2 = is_pow2(N);
  static constexpr int R1 = P2 ? 16 : 12;
  static constexpr int E2 = P2 ? (N > 256 ? N / 256 : 1) : (N > 192 ? N / 192 : 1);
  static constexpr int R2 = N / (R1 * E2);
  static constexpr int TPL = N / R1;
  static constexpr int UNITS = R1 * E2;                  // butterflies of step 2
  static constexpr int NB2 = (UNITS + TPL - 1) / TPL;    // and per thread
  static constexpr int P = E2 == 1 ? (TPL | 1) : TPL + E2;
  static constexpr int LINE = E2 == 1 ? ((R1 * P) | 1) : R1 * P + (6 - (R1 * P) % 4) % 4;
  static constexpr int M = N / E2;
  static constexpr int HALF_ITEMS = E2 == 1 ? N / 2 : M / 2;  // items of line_halves
  // Twiddle table: exp(-2 pi i t k / N) at (k - 1) TPL + t, 1 <= k < R1, then for E2 = 2
  // exp(-2 pi i q / (2 R2)) at q, for E2 = 4 exp(-2 pi i e q / (4 R2)) at 17 e + q.
  static constexpr int TW2 = (R1 - 1) * TPL;
  static constexpr int TWN = TW2 + (E2 == 4 ? 4 * 17 : (E2 == 2 ? R2 : 0));
  static_assert(R1 * R2 * E2 == N && TPL * R1 == N, "factors");
  __host__ __device__ static constexpr int slot(int kappa) { return (kappa % R1) * P + (kappa / R1) * E2; }
};

// Line handled by thread group g.  Where several groups share a half-warp, their lines
// are TPL apart, so that the groups' elements fall on different banks (LINE is odd).
template <int TPL>
__host__ __device__ constexpr int line_of_group(int g) {
  if constexpr (TPL >= 16) {
    return g;
  } else {
    constexpr int G = 16 / TPL;
    return (g % G) * TPL + (g / G) % TPL + (g / 16) * 16;
  }
}

// Whether in each warp of `groups` thread groups all lines lie below r, or all from r on: a
// branch on the line is then uniform over every barrier of line_group_sync.
template <int TPL>
__host__ __device__ constexpr bool warps_on_one_side(int groups, int r) {
  constexpr int PER = TPL >= 32 ? 1 : 32 / TPL;  // groups per warp
  for (int g = 0; g < groups; ++g)
    if ((line_of_group<TPL>(g) >= r) != (line_of_group<TPL>(g / PER * PER) >= r)) return false;
  return true;
}

// The twiddles of thread t of a line, from the table.
template <int N>
__device__ __forceinline__ void load_twiddles(float2 (&tw)[LineFft<N>::R1 - 1], const float2* table, int t) {
#pragma unroll
  for (int k = 0; k < LineFft<N>::R1 - 1; ++k) tw[k] = table[k * LineFft<N>::TPL + t];
}

// Steps 1 and 2 for the line at `line`; v: the thread's R1 elements.  Every thread of a
// warp calls this (ok: whether its line exists); tw: exp(-2 pi i t k / N), k = 1..R1 - 1;
// wE: the table's part from TW2.
template <int N>
__device__ __forceinline__ void line_fft(float2 (&v)[LineFft<N>::R1], float2* line, int t,
                                         const float2 (&tw)[LineFft<N>::R1 - 1], const float2* wE, bool ok) {
  using L = LineFft<N>;
  constexpr int R1 = L::R1, R2 = L::R2, E2 = L::E2, P = L::P, TPL = L::TPL;
  using First = std::conditional_t<R1 == 16, Dft16<R2 == 16>, Dft<R1>>;
  using Second = std::conditional_t<R2 == 16, Dft16<true>, Dft<R2>>;
  if (ok) {
    First::run(v);
    line[t] = v[0];
#pragma unroll
    for (int k = 1; k < R1; ++k) line[k * P + t] = cmul(v[k], tw[k - 1]);
  }
  line_group_sync<TPL>();
  if constexpr (R2 > 1) {
#pragma unroll
    for (int i = 0; i < L::NB2; ++i) {
      const int u = t + i * TPL;
      if (ok && (L::UNITS % TPL == 0 || u < L::UNITS)) {
        const int e = u % E2;
        float2* q = line + (u / E2) * P + e;
        float2 b[R2];
#pragma unroll
        for (int s = 0; s < R2; ++s) b[s] = q[E2 * s];
        Second::run(b);
        if constexpr (E2 == 4) {
#pragma unroll
          for (int s = 1; s < R2; ++s) b[s] = cmul(b[s], wE[17 * e + s]);
        }
#pragma unroll
        for (int s = 0; s < R2; ++s) q[E2 * s] = b[s];
      }
    }
  }
}

// The two half spectra of a line that holds real lines (a + i b) / 2: emit(k, A_k, B_k) for
// the k < nk of item i (0 <= i < HALF_ITEMS covers every k < N / 2 once).  With
// C_k the line's transform, A_k = C_k + C_{N-k}^*, B_k = (C_k - C_{N-k}^*) / i.
template <int N, class Emit>
__device__ __forceinline__ void line_halves(const float2* line, const float2* wE, int i, int nk, Emit&& emit) {
  using L = LineFft<N>;
  constexpr int M = L::M;
  auto out = [&](int k, float2 c, float2 m) {
    if (k < nk) {
      const float2 s = __ffma2_rn(m, make_float2(1.f, -1.f), c), d = __ffma2_rn(m, make_float2(-1.f, 1.f), c);
      emit(k, s, make_float2(d.y, -d.x));
    }
  };
  if constexpr (L::E2 == 1) {
    if (i >= nk) return;
    const float2 c = line[L::slot(i)];
    out(i, c, i ? line[L::slot(N - i)] : c);
  } else {
    // kappa = i and M - i (M / 2 for i = 0) hold each other's mirror frequencies
    const int k0 = i, k1 = i ? M - i : M / 2;
    if (L::E2 == 2 && k0 >= nk && k1 >= nk) return;
    const float4* s0 = reinterpret_cast<const float4*>(line + L::slot(k0));
    const float4* s1 = reinterpret_cast<const float4*>(line + L::slot(k1));
    const float4 p = s0[0], q = s1[0];
    float2 p0 = make_float2(p.x, p.y), p1 = make_float2(p.z, p.w);
    float2 q0 = make_float2(q.x, q.y), q1 = make_float2(q.z, q.w);
    if constexpr (L::E2 == 2) {
      p1 = cmul(p1, wE[k0 / L::R1]);
      q1 = cmul(q1, wE[k1 / L::R1]);
      const float2 a0 = cadd(p0, p1), a1 = csub(p0, p1), b0 = cadd(q0, q1), b1 = csub(q0, q1);
      out(k0, a0, i ? b1 : a0);
      out(k1, b0, i ? a1 : b1);
    } else {
      const float4 pp = s0[1], qq = s1[1];
      float2 a[4] = {p0, p1, make_float2(pp.x, pp.y), make_float2(pp.z, pp.w)};
      float2 b[4] = {q0, q1, make_float2(qq.x, qq.y), make_float2(qq.z, qq.w)};
      Dft<4>::run(a);
      Dft<4>::run(b);
      out(k0, a[0], i ? b[3] : a[0]);
      out(k0 + M, a[1], i ? b[2] : a[3]);
      out(k1, b[0], i ? a[3] : b[3]);
      out(k1 + M, b[1], i ? a[2] : b[2]);
    }
  }
}

// Twiddles are stored stage by stage: for stage s >= 1 (N_s = fft_ns_before(N, s)
// elements already combined, radix R_s), entry k (R_s - 1) + r - 1 of the stage's
// block is exp(-2 pi i r k / (N_s R_s)), k < N_s, 1 <= r < R_s.  A butterfly then
// reads its R_s - 1 twiddles from one base address.  The blocks fill N - R_0 < N
// entries in all.
__host__ __device__ constexpr int fft_tw_offset(int n, int stage) {
  int off = 0;
  for (int s = 1; s < stage; ++s) off += fft_ns_before(n, s) * (fft_radix(n, s) - 1);
  return off;
}

// ---------------------------------------------------------------------------
// x stage: P interleaved lines, element i of line p at (i + pad) P + p, thread
// (p, tl = tid / P) with E elements of line p.  Where the first radix is 8, one element
// of padding follows every 8, so that the first stage's stores, 8 elements apart
// across a warp, land on distinct bank pairs.
// ---------------------------------------------------------------------------
template <int N>
__host__ __device__ constexpr bool lf_padded() { return fft_radix(N, 0) == 8; }
template <int N, int P>
__host__ __device__ constexpr int lf_elems() { return (lf_padded<N>() ? N + N / 8 : N) * P; }
// Offset of element i; separable (pos(a + c) = pos(a) + pos(c)) for c a multiple of 8.
template <int N, int P>
__host__ __device__ constexpr int lf_pos(int i) { return (lf_padded<N>() ? i + (i >> 3) : i) * P; }

// First stage (no twiddles): from the unpadded tile src into the work buffer dst.
template <int N, int P>
__device__ __forceinline__ void lf_first_stage(const float2* src, float2* dst, int p, int tl) {
  constexpr int R = fft_radix(N, 0), E = fft_elems(N), TPL = N / E, STRIDE = N / R;
  const float2* s = src + tl * P + p;
  float2* d = dst + lf_pos<N, P>(R * tl) + p;
  float2 v[E];
#pragma unroll
  for (int q = 0; q < E / R; ++q)
#pragma unroll
    for (int r = 0; r < R; ++r) v[q * R + r] = s[(q * TPL + r * STRIDE) * P];
#pragma unroll
  for (int q = 0; q < E / R; ++q) {
    Dft<R>::run(&v[q * R]);
#pragma unroll
    for (int r = 0; r < R; ++r) d[lf_pos<N, P>(R * q * TPL) + r * P] = v[q * R + r];  // R | 8 or no pad
  }
}

// The inputs of stage S of the thread's butterflies.
template <int N, int P, int S>
__device__ __forceinline__ void lf_load(const float2* buf, int p, int tl, float2 (&v)[fft_elems(N)]) {
  constexpr int R = fft_radix(N, S), E = fft_elems(N), TPL = N / E, STRIDE = N / R;
  constexpr bool SEP = !lf_padded<N>() || (TPL % 8 == 0 && STRIDE % 8 == 0);
  const float2* s = buf + (SEP ? lf_pos<N, P>(tl) : 0) + p;
#pragma unroll
  for (int q = 0; q < E / R; ++q)
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int c = q * TPL + r * STRIDE;
      v[q * R + r] = s[SEP ? lf_pos<N, P>(c) : lf_pos<N, P>(tl + c)];
    }
}

// Twiddles and butterflies of stage S on the loaded inputs.
template <int N, int S>
__device__ __forceinline__ void lf_butterflies(float2 (&v)[fft_elems(N)], int tl, const float2* tw) {
  constexpr int R = fft_radix(N, S), E = fft_elems(N), TPL = N / E, NS = fft_ns_before(N, S);
#pragma unroll
  for (int q = 0; q < E / R; ++q) {
    const float2* tk = tw + fft_tw_offset(N, S) + ((tl + q * TPL) % NS) * (R - 1);
#pragma unroll
    for (int r = 1; r < R; ++r) v[q * R + r] = cmul(v[q * R + r], tk[r - 1]);
    Dft<R>::run(&v[q * R]);
  }
}

// Stages S .. last - 1 in place, two CTA barriers each.
template <int N, int P, int S, bool Done = (S >= fft_nstages(N) - 1)>
struct LfMiddle {
  __device__ static __forceinline__ void run(float2* buf, int p, int tl, const float2* tw) {
    constexpr int R = fft_radix(N, S), E = fft_elems(N), TPL = N / E, NS = fft_ns_before(N, S);
    static_assert(!lf_padded<N>() || NS % 8 == 0, "separable stores");
    float2 v[E];
    lf_load<N, P, S>(buf, p, tl, v);
    lf_butterflies<N, S>(v, tl, tw);
    __syncthreads();
#pragma unroll
    for (int q = 0; q < E / R; ++q) {
      const int j = tl + q * TPL, outb = (j / NS) * NS * R + j % NS;
      float2* d = buf + lf_pos<N, P>(outb) + p;
#pragma unroll
      for (int r = 0; r < R; ++r) d[lf_pos<N, P>(r * NS)] = v[q * R + r];
    }
    __syncthreads();
    LfMiddle<N, P, S + 1>::run(buf, p, tl, tw);
  }
};
template <int N, int P, int S>
struct LfMiddle<N, P, S, true> {
  __device__ static __forceinline__ void run(float2*, int, int, const float2*) {}
};

// Last stage into registers: v[q R + r] is frequency tl + q TPL + r N / R.  The CTA is
// past its loads when this returns.
template <int N, int P>
__device__ __forceinline__ void lf_last_stage(const float2* buf, int p, int tl, const float2* tw,
                                              float2 (&v)[fft_elems(N)]) {
  constexpr int S = fft_nstages(N) - 1;
  lf_load<N, P, S>(buf, p, tl, v);
  __syncthreads();
  lf_butterflies<N, S>(v, tl, tw);
}

}  // namespace ys
