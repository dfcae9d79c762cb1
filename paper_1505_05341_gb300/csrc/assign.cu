// Step 1 of the estimator: F = w (n - alpha n_s) on the mesh (Eq. 1; Sec. 4 assigns
// galaxies and randoms to a cubic mesh by CIC), plus the FP64 catalogue sums behind
// alpha, the normalisation I and the shot noise S (Eqs. 1 and 3).
//
// GB300 design: particles arrive in random order, and a direct global atomic
// deposit onto a 0.5-1 GB mesh would miss L2 on almost every update.  Instead a
// counting sort groups particles by mesh tile (16 x 16 x 16 nodes by default, both
// meshes of an interlaced pair held together), and one CTA per tile accumulates its
// nodes in shared memory with integer shared-memory atomics (exact fixed-point sums),
// then writes the tile with coalesced plain stores.  A particle whose stencil crosses tile borders is listed once per
// tile it touches (at most 8), so tiles never write each other's nodes: no global
// atomics on the mesh and no zero-fill pass.
//
//   k_particles : cell index per particle, compensated sums, per-tile counts
//   k_scan      : exclusive scan of the counts
//   k_bin_agg / k_bin : one 16-byte record (position, signed weight) per tile touched;
//                 records whose stencils lie inside one tile fill its list from the
//                 front, the others from the back, so the deposit walks the interior
//                 ones without per-node range checks
//                 (the deposit locates the particle again: 20-byte records with the
//                 cell index cost two partial L2 sector writes each)
//   k_deposit   : per-tile shared-memory deposit and store
//
// Both catalogues go through one launch of each pass (Cats).
//
// Sub-cell offsets are formed against a host-built FP64 table of node positions
// split into float (hi, lo) pairs, so d = u - floor(u) keeps ~1e-7 accuracy even
// where u = (x - box_min)/H itself is only good to ~1e-5 in float.
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "ys_internal.h"

namespace ys {
namespace {

constexpr int THREADS = 256;

// Galaxies and randoms of one launch: blocks [0, blocks0) take the galaxies, the others
// the randoms.
struct Cats {
  const float* x[2];
  const float* y[2];
  const float* z[2];
  const float* w[2];
  const float* nbar[2];
  int64_t n[2];
  int blocks0;
};

// This block's catalogue (0 galaxies, 1 randoms), its place among that catalogue's
// blocks and their number.
__device__ __forceinline__ int block_catalogue(const Cats& c, int& bid, int& nblk) {
  const int k = (int)blockIdx.x >= c.blocks0;
  bid = blockIdx.x - (k ? c.blocks0 : 0);
  nblk = k ? gridDim.x - c.blocks0 : c.blocks0;
  return k;
}

// a + b and its rounding error (TwoSum, error-free).
__device__ __forceinline__ float two_sum(float a, float b, float& err) {
  const float t = a + b, bb = t - a;
  err = (a - (t - bb)) + (b - bb);
  return t;
}

// Sums of w, w^2 and w^2 nbar over this thread's particles: float sums s, and in c the exact
// rounding errors of every addition and product.
struct ThreadSums {
  float s[3] = {0.f, 0.f, 0.f}, c[3] = {0.f, 0.f, 0.f};
  __device__ __forceinline__ float add(int k, float v) {
    float err;
    s[k] = two_sum(s[k], v, err);
    return err;
  }
  // (__fmul_rn: a product contracted into the addition would not be the one whose error is taken)
  __device__ __forceinline__ void particle(float w, const float* nbar, float nb) {
    c[0] += add(0, w);
    const float p = __fmul_rn(w, w), e = fmaf(w, w, -p);
    c[1] += add(1, p) + e;
    if (nbar) {
      const float q = __fmul_rn(p, nb);
      c[2] += add(2, q) + fmaf(e, nb, fmaf(p, nb, -q));
    }
  }
};

// Adds the block's sums (and its count of particles outside the box) to the catalogue
// sums.  The lanes of a warp meet in expansions of three floats (~2^-70, below an FP64
// addition's rounding; an FP64 shuffle tree of three sums took 15 x 16 cycles of the SM per
// warp), scaled by 2^-10 where 32 of the sums might overflow; the warps meet in FP64, and
// each CTA makes one FP64 atomic per sum: per-warp atomics on the three addresses alone
// took ~30 us per catalogue.  FKP-weighted catalogues of 6e6 to 3e7 particles: alpha, I and
// S / I are within 5e-15 of FP64 sums (4e-11 to 8e-11 with Kahan sums, which round every term).
template <int NT>
__device__ __forceinline__ void block_sums(ThreadSums& ts, unsigned bad, int is_ran, double* __restrict__ sums) {
  __shared__ float4 red[3][NT / 32];  // sum, its two tails, scale
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    if (!is_ran && k == 2) break;
    float s = ts.s[k], c = ts.c[k], e = 0.f, scale = 1.f;
    if (__any_sync(0xffffffffu, !(fabsf(s) < 0x1p120f))) {
      scale = 1024.f;
      s *= 0x1p-10f;
      c *= 0x1p-10f;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      float e1, e2, e3;
      const float s2 = __shfl_xor_sync(0xffffffffu, s, o), c2 = __shfl_xor_sync(0xffffffffu, c, o);
      e += __shfl_xor_sync(0xffffffffu, e, o);
      s = two_sum(s, s2, e1);
      c = two_sum(c, c2, e2);
      c = two_sum(c, e1, e3);
      e += e2 + e3;
    }
    if (lane == 0) red[k][wid] = make_float4(s, c, e, scale);
  }
  const int nbad = __syncthreads_or(bad != 0);
  if (nbad) {
    unsigned tot = bad;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) tot += __shfl_xor_sync(0xffffffffu, tot, o);
    if (lane == 0 && tot) atomicAdd(&sums[SUM_BAD], (double)tot);
  }
  if (wid == 0) {
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      if (!is_ran && k == 2) break;
      const float4 r = lane < NT / 32 ? red[k][lane] : make_float4(0.f, 0.f, 0.f, 1.f);
      double v = ((double)r.x + ((double)r.y + (double)r.z)) * (double)r.w;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1)
        if (o < NT / 32) v += __shfl_xor_sync(0xffffffffu, v, o);
      const int slot = is_ran ? (k == 0 ? SUM_WR : (k == 1 ? SUM_WR2 : SUM_WR2N)) : (k == 0 ? SUM_WG : SUM_WG2);
      if (lane == 0) atomicAdd(&sums[slot], v);
    }
  }
}

// Cell index i and offset d in [0, 1) of coordinate x along one axis.  Returns
// false (and a periodically wrapped in-range cell) when x lies outside the box.
__device__ __forceinline__ bool locate(float x, int axis, const Geom& g, const float2* __restrict__ nodes,
                                       int& i_out, float& d_out) {
  const int n = g.n;
  const float u0 = (x - g.bmin[axis]) * g.inv_h;
  int i = max(-1, min(n, __float2int_rd(u0)));  // (the conversion saturates; NaN gives 0)
  const float2* nd = nodes + axis * (n + 3) + 1;  // nd[i] for i in [-1, n + 1]
  float2 nv = nd[i];
  float d = ((x - nv.x) - nv.y) * g.inv_h;
  // One-cell correction of the float guess (rarely needed); a particle within rounding
  // of a node can land on d = 1.0f (or a hair below 0) after it, so d is clamped into
  // [0, 1): the stencils are continuous across the node, so either side gives the same mesh.
  if (d < 0.f) {
    i = max(i - 1, -1);
    nv = nd[i];
    d = fminf(((x - nv.x) - nv.y) * g.inv_h, 0.99999994f);
  } else if (d >= 1.f) {
    i = min(i + 1, n);
    nv = nd[i];
    d = fmaxf(((x - nv.x) - nv.y) * g.inv_h, 0.f);
  }
  d = fminf(fmaxf(d, 0.f), 0.99999994f);
  const bool ok = (unsigned)i < (unsigned)n && u0 == u0;
  if (!ok) {
    const bool finite = isfinite(u0);
    const float uw = finite ? u0 - floorf(u0 / (float)n) * (float)n : 0.f;
    int iw = (int)floorf(uw);
    iw = max(0, min(n - 1, iw));
    i = iw;
    d = fminf(fmaxf(uw - (float)iw, 0.f), 0.99999994f);
  }
  i_out = i;
  d_out = d;
  return ok;
}

// Stencil of one axis: up to KIND nodes and weights, for mesh 1 (nodes at i) and
// mesh 2 (nodes at i + 1/2, i.e. coordinate u - 1/2).
template <int KIND>
__device__ __forceinline__ void stencil(int i, float d, bool second, int& first, float (&w)[3]) {
  if (KIND == 1) {  // NGP
    first = second ? i : i + (d >= 0.5f ? 1 : 0);
    w[0] = 1.f;
  } else if (KIND == 2) {  // CIC
    int i2 = i;
    float d2 = d;
    if (second) {
      if (d >= 0.5f) { d2 = d - 0.5f; } else { i2 = i - 1; d2 = d + 0.5f; }
    }
    first = i2;
    w[0] = 1.f - d2;
    w[1] = d2;
  } else {  // TSC
    int c;
    float dd;
    if (second) { c = i; dd = d - 0.5f; }
    else if (d >= 0.5f) { c = i + 1; dd = d - 1.f; }
    else { c = i; dd = d; }
    first = c - 1;
    const float a = 0.5f - dd, b = 0.5f + dd;
    w[0] = 0.5f * a * a;
    w[1] = 0.75f - dd * dd;
    w[2] = 0.5f * b * b;
  }
}

// Inclusive node range [lo, hi] covered by the stencils of the M meshes.
template <int KIND, int M>
__device__ __forceinline__ void node_range(int i, float d, int& lo, int& hi) {
  float w[3];
  int f1;
  stencil<KIND>(i, d, false, f1, w);
  lo = f1;
  hi = f1 + KIND - 1;
  if (M == 2) {
    int f2;
    stencil<KIND>(i, d, true, f2, w);
    lo = min(lo, f2);
    hi = max(hi, f2 + KIND - 1);
  }
}

__device__ __forceinline__ int wrapn(int v, int n) { return v < 0 ? v + n : (v >= n ? v - n : v); }

// Tiles a particle's stencils touch, one or two per axis: first, and first plus any sum of
// dx, dy, dz; inner when the stencils lie inside one tile without periodic wrap.
struct Touched {
  int first, dx, dy, dz;  // dx, dy, dz: 0 where the axis has one tile only
  bool inner, ok;         // ok: the particle is inside the box
  // f(tile) for every tile but the first
  template <class F>
  __device__ __forceinline__ void others(F&& f) const {
    const int all = (dx ? 1 : 0) | (dy ? 2 : 0) | (dz ? 4 : 0);
    for (int m = all; m; m = (m - 1) & all)  // the non-empty subsets of the axes with two tiles
      f(first + ((m & 1) ? dx : 0) + ((m & 2) ? dy : 0) + ((m & 4) ? dz : 0));
  }
};

template <int KIND, int M>
__device__ __forceinline__ Touched touched_tiles(float x, float y, float z, const Geom& g,
                                                 const float2* __restrict__ nodes) {
  int ci[3], t0[3], d[3];
  float cd[3];
  Touched r;
  r.ok = locate(x, 0, g, nodes, ci[0], cd[0]);
  r.ok &= locate(y, 1, g, nodes, ci[1], cd[1]);
  r.ok &= locate(z, 2, g, nodes, ci[2], cd[2]);
  r.inner = true;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    int lo, hi;
    node_range<KIND, M>(ci[a], cd[a], lo, hi);
    t0[a] = wrapn(lo, g.n) >> g.tshift[a];
    d[a] = (wrapn(hi, g.n) >> g.tshift[a]) - t0[a];
    r.inner = r.inner && d[a] == 0 && lo >= 0 && hi < g.n;
  }
  r.first = (t0[0] * g.tiles[1] + t0[1]) * g.tiles[2] + t0[2];
  r.dx = d[0] * g.tiles[1] * g.tiles[2];
  r.dy = d[1] * g.tiles[2];
  r.dz = d[2];
  return r;
}

// What the binning pass needs of a particle's tiles, kept by the counting pass in 32 bits:
// the first tile (16 bits), two bits per axis (0: one tile, 1: the next one too, 2: the
// first one of the axis too, across the periodic edge), and the inner flag.
__device__ __forceinline__ unsigned pack_touched(const Touched& t) {
  auto step = [](int d) { return d == 0 ? 0u : (d > 0 ? 1u : 2u); };
  return (unsigned)t.first | step(t.dx) << 16 | step(t.dy) << 18 | step(t.dz) << 20 | (t.inner ? 1u << 22 : 0u);
}
__device__ __forceinline__ Touched unpack_touched(unsigned c, const Geom& g) {
  Touched t;
  auto delta = [](unsigned s, int stride, int tiles) { return s == 0u ? 0 : (s == 1u ? stride : -(tiles - 1) * stride); };
  t.first = (int)(c & 0xffffu);
  t.dx = delta(c >> 16 & 3u, g.tiles[1] * g.tiles[2], g.tiles[0]);
  t.dy = delta(c >> 18 & 3u, g.tiles[2], g.tiles[1]);
  t.dz = delta(c >> 20 & 3u, 1, g.tiles[2]);
  t.inner = (c >> 22 & 1u) != 0u;
  t.ok = true;
  return t;
}

// Counting pass.  codes: where the aggregated binning pass finds each particle's tiles
// (galaxies first, then randoms; nullptr: it locates them again).  HIST: the tile counts go to a histogram in shared memory (ntiles
// counters), added to the global counts once per CTA at the end -- a few CTAs per SM and
// a grid-stride loop, instead of one global atomic per (particle, tile) on counters that
// every SM contends for.
template <int KIND, int M, bool HIST, int NT>
__global__ void __launch_bounds__(NT)
k_particles(const __grid_constant__ Cats cats, Geom g, const float2* __restrict__ nodes,
            unsigned* __restrict__ tile_count, double* __restrict__ sums, int ntiles, unsigned* __restrict__ codes) {
  extern __shared__ unsigned s_hist[];
  if (HIST) {
    for (int t = threadIdx.x; t < ntiles; t += NT) s_hist[t] = 0u;
    __syncthreads();
  }
  int bid, nblk;
  const int is_ran = block_catalogue(cats, bid, nblk);
  const float* __restrict__ px = cats.x[is_ran];
  const float* __restrict__ py = cats.y[is_ran];
  const float* __restrict__ pz = cats.z[is_ran];
  const float* __restrict__ pw = cats.w[is_ran];
  const float* __restrict__ pnbar = is_ran ? cats.nbar[1] : nullptr;
  const int64_t n = cats.n[is_ran];
  if (codes && is_ran) codes += cats.n[0];
  ThreadSums ts;
  unsigned bad = 0;
  const int64_t stride = (int64_t)nblk * NT;
  // Two particles per iteration (the same order as one per iteration): their loads are issued
  // together, so that the latencies overlap.
  constexpr int U = 2;
  for (int64_t base = (int64_t)bid * NT + threadIdx.x; base < n; base += U * stride) {
    float xs[U], ys[U], zs[U], ws[U], nbs[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int64_t i = base + u * stride < n ? base + u * stride : base;
      xs[u] = px[i];
      ys[u] = py[i];
      zs[u] = pz[i];
      ws[u] = pw ? pw[i] : 1.f;
      nbs[u] = pnbar ? pnbar[i] : 0.f;
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      if (base + u * stride >= n) break;
      const float x = xs[u], y = ys[u], z = zs[u], w = ws[u];
      const Touched tt = touched_tiles<KIND, M>(x, y, z, g, nodes);
      bad += tt.ok ? 0u : 1u;
      if (codes) codes[base + u * stride] = pack_touched(tt);
      ts.particle(w, pnbar, nbs[u]);
      auto count = [&](int tile) {
        if constexpr (HIST) atomicAdd(&s_hist[tile], 1u);
        else atomicAdd(&tile_count[tile], 1u);
      };
      count(tt.first);
      if (!tt.inner) tt.others(count);
    }
  }
  if (HIST) {
    __syncthreads();
    for (int t = threadIdx.x; t < ntiles; t += NT)
      if (s_hist[t]) atomicAdd(&tile_count[t], s_hist[t]);
  }
  block_sums<NT>(ts, bad, is_ran, sums);
}

// Signed weight factor of a catalogue: 1 for galaxies, -alpha for randoms.
__device__ __forceinline__ float catalogue_scale(int is_ran, double alpha_cfg, const double* __restrict__ sums) {
  return is_ran ? (float)(-(alpha_cfg >= 0.0 ? alpha_cfg : sums[SUM_WG] / sums[SUM_WR])) : 1.f;
}

// Binning pass: one 16-byte record (position, signed weight) per tile a particle's
// stencils touch; records whose stencils lie inside one tile (no periodic wrap) fill
// the tile's list from the front (cursor tile_cur), the others from the back (the
// tile's remaining count tile_left, from off[tile]).
//
// Few tiles (k_bin_agg, up to BIN_AGG_TILES): a CTA counts the records of a chunk of
// particles per tile in shared memory, reserves each tile's range with one global
// atomic, and hands out the slots from shared-memory cursors.  One global atomic per
// record serialises on the tiles' cursors when there are few of them: 6.6e6 particles
// on the 512 tiles of a 128^3 mesh took 790 us, 151 us now.  CODES: the tiles come from the
// counting pass (4 bytes per particle instead of two locates; counting and binning
// together 333 -> 298 us on the 256^3 cone, 243 -> 236 at 128^3).
// Many tiles (k_bin): a chunk would hold about one record per tile, so each record takes
// its own global atomic; each thread takes U particles per iteration, whose loads and
// first-tile cursor atomics are independent, so that their latencies overlap.
constexpr int BIN_AGG_TILES = 4096;
constexpr int BIN_AGG_NT = 512;

template <int KIND, int M, bool CODES>
__global__ void __launch_bounds__(BIN_AGG_NT)
k_bin_agg(const __grid_constant__ Cats cats, int per_thread, Geom g, const float2* __restrict__ nodes,
          const unsigned* __restrict__ codes, int ntiles,
          const unsigned* __restrict__ off, unsigned* __restrict__ tile_left, unsigned* __restrict__ tile_cur,
          float4* __restrict__ rec, const double* __restrict__ sums, double alpha_cfg) {
  extern __shared__ unsigned s_cur[];  // [2][ntiles]: interior, border
  for (int t = threadIdx.x; t < 2 * ntiles; t += BIN_AGG_NT) s_cur[t] = 0u;
  int bid, nblk;
  const int is_ran = block_catalogue(cats, bid, nblk);
  const float* __restrict__ px = cats.x[is_ran];
  const float* __restrict__ py = cats.y[is_ran];
  const float* __restrict__ pz = cats.z[is_ran];
  const float* __restrict__ pw = cats.w[is_ran];
  const int64_t first = (int64_t)bid * BIN_AGG_NT * per_thread;
  px += first;
  py += first;
  pz += first;
  if (pw) pw += first;
  if (CODES) codes += first + (is_ran ? cats.n[0] : 0);
  const int last = (int)min(cats.n[is_ran] - first, (int64_t)BIN_AGG_NT * per_thread);
  __syncthreads();
#pragma unroll 2
  for (int i = threadIdx.x; i < last; i += BIN_AGG_NT) {
    const Touched tt = CODES ? unpack_touched(codes[i], g) : touched_tiles<KIND, M>(px[i], py[i], pz[i], g, nodes);
    unsigned* cnt = s_cur + (tt.inner ? 0 : ntiles);
    atomicAdd(cnt + tt.first, 1u);
    if (!tt.inner) tt.others([&](int tile) { atomicAdd(cnt + tile, 1u); });
  }
  __syncthreads();
  for (int t = threadIdx.x; t < ntiles; t += BIN_AGG_NT) {
    const unsigned f = s_cur[t], b = s_cur[ntiles + t];
    if (f) s_cur[t] = atomicAdd(&tile_cur[t], f);
    if (b) s_cur[ntiles + t] = off[t] + atomicSub(&tile_left[t], b) - b;
  }
  __syncthreads();
  const float wscale = catalogue_scale(is_ran, alpha_cfg, sums);
#pragma unroll 2
  for (int i = threadIdx.x; i < last; i += BIN_AGG_NT) {
    const float4 q = make_float4(px[i], py[i], pz[i], (pw ? pw[i] : 1.f) * wscale);
    const Touched tt = CODES ? unpack_touched(codes[i], g) : touched_tiles<KIND, M>(q.x, q.y, q.z, g, nodes);
    unsigned* cur = s_cur + (tt.inner ? 0 : ntiles);
    rec[atomicAdd(cur + tt.first, 1u)] = q;
    if (!tt.inner) tt.others([&](int tile) { rec[atomicAdd(cur + tile, 1u)] = q; });
  }
}

template <int KIND, int M, int U>
__global__ void __launch_bounds__(THREADS)
k_bin(const __grid_constant__ Cats cats, Geom g, const float2* __restrict__ nodes, const unsigned* __restrict__ off,
      unsigned* __restrict__ tile_left, unsigned* __restrict__ tile_cur, float4* __restrict__ rec,
      const double* __restrict__ sums, double alpha_cfg) {
  int bid, nblk;
  const int is_ran = block_catalogue(cats, bid, nblk);
  const float* __restrict__ px = cats.x[is_ran];
  const float* __restrict__ py = cats.y[is_ran];
  const float* __restrict__ pz = cats.z[is_ran];
  const float* __restrict__ pw = cats.w[is_ran];
  const int64_t n = cats.n[is_ran];
  const float wscale = catalogue_scale(is_ran, alpha_cfg, sums);
  const int64_t stride = (int64_t)nblk * blockDim.x;
  for (int64_t base = (int64_t)bid * blockDim.x + threadIdx.x; base < n; base += U * stride) {
    float4 q[U];
    Touched tt[U];
    bool valid[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int64_t idx = base + u * stride;
      valid[u] = idx < n;
      const int64_t i = valid[u] ? idx : base;
      q[u] = make_float4(px[i], py[i], pz[i], (pw ? pw[i] : 1.f) * wscale);
    }
#pragma unroll
    for (int u = 0; u < U; ++u) tt[u] = touched_tiles<KIND, M>(q[u].x, q[u].y, q[u].z, g, nodes);
    unsigned slot[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      if (!valid[u]) continue;
      const int tile = tt[u].first;
      slot[u] = tt[u].inner ? atomicAdd(&tile_cur[tile], 1u) : off[tile] + atomicSub(&tile_left[tile], 1u) - 1u;
    }
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (valid[u]) rec[slot[u]] = q[u];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      if (!valid[u] || tt[u].inner) continue;
      tt[u].others([&](int tile) { rec[off[tile] + atomicSub(&tile_left[tile], 1u) - 1u] = q[u]; });
    }
  }
}

// Exclusive scan of the tile counts into off and the front cursors cur, one CTA per 1024
// tiles.  Each CTA sums all counts before its own (at most 1 MB, from L2) instead of
// waiting for the CTAs before it: 32768 tiles 102 -> 8 us, 262144 tiles 785 -> 16 us
// against one CTA for all.
__global__ void __launch_bounds__(1024)
k_scan(const unsigned* __restrict__ count, int ntiles, unsigned* __restrict__ off, unsigned* __restrict__ cur) {
  __shared__ unsigned part[33];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const uint4* c4 = reinterpret_cast<const uint4*>(count);
  unsigned before = 0;
#pragma unroll 4
  for (int i = threadIdx.x; i < (int)blockIdx.x * 256; i += 1024) {
    const uint4 v = c4[i];
    before += v.x + v.y + v.z + v.w;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) before += __shfl_xor_sync(0xffffffffu, before, o);
  if (lane == 0) part[wid] = before;
  __syncthreads();
  if (wid == 0) {
    unsigned v = part[lane];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (lane == 0) part[32] = v;
  }
  __syncthreads();
  const unsigned base = part[32];
  __syncthreads();
  const int i = blockIdx.x * 1024 + threadIdx.x;
  const unsigned c = i < ntiles ? count[i] : 0u;
  unsigned incl = c;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned v = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += v;
  }
  if (lane == 31) part[wid] = incl;
  __syncthreads();
  if (wid == 0) {
    unsigned v = part[lane];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned u = __shfl_up_sync(0xffffffffu, v, o);
      if (lane >= o) v += u;
    }
    part[lane] = v;
  }
  __syncthreads();
  const unsigned excl = base + (wid > 0 ? part[wid - 1] : 0u) + incl - c;
  if (i < ntiles) {
    off[i] = excl;
    cur[i] = excl;
    if (i == ntiles - 1) off[ntiles] = excl + c;
  }
}

// Extents of a tile: TD^3 nodes known at compile time, or the launch's (TD = 0).
template <int TD>
struct TileDims {
  int d[3];
  __device__ __forceinline__ explicit TileDims(const Geom& g) : d{g.tdim[0], g.tdim[1], g.tdim[2]} {}
  __device__ __forceinline__ int operator[](int a) const { return TD > 0 ? TD : d[a]; }
  __device__ __forceinline__ int volume() const { return TD > 0 ? TD * TD * TD : d[0] * d[1] * d[2]; }
};

// Stencil walk of one record: add(k, wxy, wz) for every node of the record's stencil,
// k the node's index in the tile's (mesh, x, y, z) order and its weight the product
// wxy * wz (wxy = wq W_x W_y, wz = W_z).  A node outside this tile goes to `trash`
// (a per-lane word past the tile that is never read): in a warp of 32 records nearly
// every stencil node is inside for some lane, so branching per node saves no adds
// and costs a divergent branch each.
template <int KIND, int M, class Dims, class Add>
__device__ __forceinline__ void deposit_record(const float4& q, float wq, const Geom& g,
                                               const float2* __restrict__ nodes, const int (&o)[3],
                                               const Dims& td, int trash, Add&& add) {
  const int tvol = td.volume();
  const int n = g.n;
  int ci[3];
  float cd[3];  // the cell and offset the binning pass found (same arithmetic)
  locate(q.x, 0, g, nodes, ci[0], cd[0]);
  locate(q.y, 1, g, nodes, ci[1], cd[1]);
  locate(q.z, 2, g, nodes, ci[2], cd[2]);
#pragma unroll
  for (int mj = 0; mj < M; ++mj) {
    int loc[3][3];
    float wt[3][3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      int first;
      stencil<KIND>(ci[a], cd[a], mj == 1, first, wt[a]);
#pragma unroll
      for (int s = 0; s < KIND; ++s) {
        const int l = wrapn(first + s - o[a], n);  // first + s in [-1, n + 1]; o[a] in [0, n)
        loc[a][s] = (l >= 0 && l < td[a]) ? l : -1;
      }
    }
#pragma unroll
    for (int a = 0; a < KIND; ++a) {
#pragma unroll
      for (int bb = 0; bb < KIND; ++bb) {
        const float wxy = wq * wt[0][a] * wt[1][bb];
        const bool in_row = loc[0][a] >= 0 && loc[1][bb] >= 0;
        const int row = mj * tvol + (loc[0][a] * td[1] + loc[1][bb]) * td[2];
#pragma unroll
        for (int c = 0; c < KIND; ++c) add(in_row && loc[2][c] >= 0 ? row + loc[2][c] : trash, wxy, wt[2][c]);
      }
    }
  }
}

// Stencil walk of an interior record (every node of both stencils inside this tile,
// no periodic wrap): the same weights and node order as deposit_record, without the
// per-node range checks, and with the nodes of one (x, y) row at fixed offsets.
template <int KIND, int M, class Dims, class Add>
__device__ __forceinline__ void deposit_inner(const float4& q, float wq, const Geom& g,
                                              const float2* __restrict__ nodes, const int (&o)[3],
                                              const Dims& td, Add&& add) {
  const int tvol = td.volume();
  int ci[3];
  float cd[3];
  locate(q.x, 0, g, nodes, ci[0], cd[0]);
  locate(q.y, 1, g, nodes, ci[1], cd[1]);
  locate(q.z, 2, g, nodes, ci[2], cd[2]);
#pragma unroll
  for (int mj = 0; mj < M; ++mj) {
    int first[3];
    float wt[3][3];
#pragma unroll
    for (int a = 0; a < 3; ++a) stencil<KIND>(ci[a], cd[a], mj == 1, first[a], wt[a]);
    const int base = mj * tvol + ((first[0] - o[0]) * td[1] + (first[1] - o[1])) * td[2] + (first[2] - o[2]);
#pragma unroll
    for (int a = 0; a < KIND; ++a)
#pragma unroll
      for (int bb = 0; bb < KIND; ++bb) {
        const float wxy = wq * wt[0][a] * wt[1][bb];
        const int row = base + (a * td[1] + bb) * td[2];
#pragma unroll
        for (int c = 0; c < KIND; ++c) add(row + c, wxy, wt[2][c]);
      }
  }
}

// Per-tile deposit.  FIXED (the tile fits twice in shared memory): the node sums are
// kept in fixed point, as two int32 words per node, because shared-memory integer
// atomics are several times faster than float ones and integer sums are exact.
//
// Fixed point.  A node value v is stored as V = v 2^s (units of 2^-s), split into
// hi 2^sb + lo with |lo| <= 2^(sb-1); hi and lo are summed in separate int32 arrays.
// With n < 2^30 records in the tile and w_m the largest |w| among them:
//   sb = min(22, floor(31 - log2 n))  => n 2^(sb-1) <= 2^30: the lo sums cannot
//                                        overflow;
//   s  = floor(min(30 + sb - log2(n w_m), 21 + sb - log2 w_m))
//      => |V| <= 2^(21+sb) for one stencil weight (|W| <= 1), which the rounding
//         below needs, and sum |V| <= 2^(30+sb), so the hi sums stay below
//         2^30 + n/2 < 2^31.  (A float log2 off in its last bits moves these bounds by
//         a factor 1 + 1e-6, well inside the slack.)
// One stencil weight V = wxy wz 2^s (wxy already carries 2^s, an exact power-of-two
// scaling) is split without conversion instructions: fma(wxy, wz, K) with
// K = 1.5 2^(23+sb) rounds V to a multiple of 2^sb, and the bit pattern of the
// result minus that of K is V / 2^sb rounded (hi); fma(wxy, wz, -(t - K)) is the
// remainder to one float rounding, and adding 1.5 2^23 rounds it to an integer (lo).
// Each stencil weight is thus quantised to 2^-s (2^-37 of the largest weight for a
// tile of ~3000 records; 2^-17 of it for one of a million, still far finer than
// float sums, which drop every weight below half an ulp of a large node) and the sums
// are exact, so the mesh is the same bit for bit whatever order the records arrive
// in.  A tile with a non-finite weight (or 2^30 or more records) is summed in float
// instead, so that a NaN reaches exactly the nodes it touches.
//
// rmesh (shared randoms): the kept random mesh sum_ran w W, written as
// F = (galaxy deposit) - alpha rmesh, with alpha from the catalogue sums.
//
// MULTI: a cluster of CTAs shares one tile (deposit_cluster gives its size), where there
// are too few tiles to fill the GPU: each CTA deposits its share of the records into its
// own copy, and each sums its share of the nodes over the cluster's copies (integers:
// the same bits whatever the split) before storing them.
//
// TD: the tile's side when it is a cube known at compile time (16, the default tile), so
// that a record's nodes and both words of a sum are at constant offsets; 0 otherwise.
// 512^3 survey, TSC interlaced: 4.41 ms with tile indices by division and run-time extents,
// 4.18 with shifts, 4.08 with constant extents; 1024^3 CIC 2.83, 2.29, 1.84 ms.  Bound by
// shared memory (89 % busy, 69 % of its wavefronts are bank conflicts of 32 random nodes).
template <int KIND, int M, bool FIXED, bool MULTI, int TD>
__global__ void __launch_bounds__(THREADS, 3)
k_deposit(Geom g, const float2* __restrict__ nodes, const unsigned* __restrict__ off,
          const unsigned* __restrict__ split, const float4* __restrict__ rec, float* __restrict__ mesh,
          const float* __restrict__ rmesh, const double* __restrict__ sums, double alpha_cfg) {
  extern __shared__ float s_tile[];
  __shared__ float s_wmax[THREADS / 32];
  __shared__ float s_part;  // this CTA's largest |w|, NaN if a weight is not finite
  namespace cg = cooperative_groups;
  [[maybe_unused]] cg::cluster_group cluster = cg::this_cluster();
  const unsigned cl = MULTI ? cluster.num_blocks() : 1u, rank = MULTI ? cluster.block_rank() : 0u;
  const int n = g.n;
  const TileDims<TD> td(g);
  const int tdx = td[0], tdy = td[1], tdz = td[2], tvol = td.volume();
  const int tile = blockIdx.x / cl;
  const unsigned tid = rank * THREADS + threadIdx.x, step = cl * THREADS;  // over the tile's records
  const int tz = tile % g.tiles[2];
  const int ty = (tile / g.tiles[2]) % g.tiles[1];
  const int tx = tile / (g.tiles[2] * g.tiles[1]);
  const int o[3] = {tx * tdx, ty * tdy, tz * tdz};
  const unsigned b = off[tile], e = off[tile + 1];
  const unsigned mid = split[tile];  // records [b, mid) are interior, [mid, e) cross a border
  const unsigned nrec = e - b;
  bool fixed = false;
  int sb = 0, sc = 0;  // split bits and scale exponent s
  // Layout: M tvol node words + 32 trash words, twice when FIXED (hi, then lo).
  const int words = M * tvol + 32;
  const int trash = M * tvol + (threadIdx.x & 31);
  if (FIXED) {
    for (int k = threadIdx.x; k < 2 * words; k += blockDim.x) s_tile[k] = 0.f;
    const float* wrec = reinterpret_cast<const float*>(rec) + 3;
    float wm = 0.f;
    bool bad = false;
    for (unsigned r = b + tid; r < e; r += step) {
      const float w = wrec[(size_t)r * 4];
      bad |= !isfinite(w);
      wm = fmaxf(wm, fabsf(w));
    }
#pragma unroll
    for (int k = 16; k > 0; k >>= 1) wm = fmaxf(wm, __shfl_xor_sync(0xffffffffu, wm, k));
    if ((threadIdx.x & 31) == 0) s_wmax[threadIdx.x >> 5] = wm;
    bad = __syncthreads_or(bad);  // also orders s_wmax and the zero fill
#pragma unroll
    for (int k = 0; k < THREADS / 32; ++k) wm = fmaxf(wm, s_wmax[k]);
    if constexpr (MULTI) {  // over the cluster
      if (threadIdx.x == 0) s_part = bad ? __int_as_float(0x7fc00000) : wm;
      cluster.sync();
      for (unsigned q = 0; q < cl; ++q) {
        const float v = *cluster.map_shared_rank(&s_part, q);
        bad |= isnan(v);
        wm = fmaxf(wm, v);
      }
    }
    fixed = !bad && nrec < (1u << 30);
    if (fixed && nrec > 0) {
      const float ln = log2f((float)nrec), lw = log2f(wm);
      sb = min(22, (int)floorf(31.f - ln));
      // s <= 100 only loses resolution; weights beyond ~2^100 (s < -100) sum in float
      const float sf = wm > 0.f ? floorf(fminf(30.f + sb - ln - lw, 21.f + sb - lw)) : 0.f;
      fixed = sf >= -100.f;
      sc = (int)fminf(100.f, fmaxf(sf, -100.f));
    }
  } else {
    for (int k = threadIdx.x; k < M * tvol; k += blockDim.x) s_tile[k] = 0.f;
    __syncthreads();
  }
  if (fixed) {
    int* s_hi = reinterpret_cast<int*>(s_tile);
    int* s_lo = s_hi + words;
    const float scale = __int_as_float((127 + sc) << 23);            // 2^s
    const int kbits = ((127 + 23 + sb) << 23) | 0x400000;            // 1.5 2^(23+sb)
    const float kh = __int_as_float(kbits);
    auto add = [&](int k, float wxy, float wz) {
      const float t = __fmaf_rn(wxy, wz, kh);
      const float lf = __fmaf_rn(wxy, wz, -__fsub_rn(t, kh));
      atomicAdd(s_hi + k, __float_as_int(t) - kbits);
      atomicAdd(s_lo + k, __float_as_int(__fadd_rn(lf, 12582912.f)) - 0x4B400000);  // + 1.5 2^23
    };
    for (unsigned r = b + tid; r < mid; r += step) {
      const float4 q = rec[r];
      deposit_inner<KIND, M>(q, q.w * scale, g, nodes, o, td, add);
    }
    for (unsigned r = mid + tid; r < e; r += step) {
      const float4 q = rec[r];
      deposit_record<KIND, M>(q, q.w * scale, g, nodes, o, td, trash, add);
    }
  } else {
    auto add = [&](int k, float wxy, float wz) { atomicAdd(s_tile + k, wxy * wz); };
    for (unsigned r = b + tid; r < mid; r += step) {
      const float4 q = rec[r];
      deposit_inner<KIND, M>(q, q.w, g, nodes, o, td, add);
    }
    for (unsigned r = mid + tid; r < e; r += step) {
      const float4 q = rec[r];
      deposit_record<KIND, M>(q, q.w, g, nodes, o, td, trash, add);
    }
  }
  if constexpr (MULTI) cluster.sync();
  else __syncthreads();
  const size_t n3 = (size_t)n * n * n;
  const float ran_scale =
      rmesh ? (float)(-(alpha_cfg >= 0.0 ? alpha_cfg : sums[SUM_WG] / sums[SUM_WR])) : 0.f;
  // hi 2^sb + lo in units of 2^-s, in float: each int32 rounds to float once and the
  // fma once more (within one ulp of the exact sum, and the same bits on every run)
  const float unscale = __int_as_float((127 - sc) << 23);       // 2^-s
  const float hscale = __int_as_float((127 + sb - sc) << 23);   // 2^(sb-s)
  int* s_hi = reinterpret_cast<int*>(s_tile);
  const int shz = g.tshift[2], shy = g.tshift[1], shv = shz + shy + g.tshift[0];
  for (int k = tid; k < M * tvol; k += step) {
    const int mj = k >> shv;
    const int lz = k & (tdz - 1);
    const int ly = (k >> shz) & (tdy - 1);
    const int lx = (k >> (shz + shy)) & (tdx - 1);
    const size_t at = mj * n3 + ((size_t)(o[0] + lx) * n + (o[1] + ly)) * n + (o[2] + lz);
    float v;
    if constexpr (MULTI) {
      if (fixed) {
        int hi = 0, lo = 0;
        for (unsigned q = 0; q < cl; ++q) {
          const int* part = cluster.map_shared_rank(s_hi, q);
          hi += part[k];
          lo += part[words + k];
        }
        v = __fmaf_rn(__int2float_rn(hi), hscale, __int2float_rn(lo) * unscale);
      } else {
        v = 0.f;
        for (unsigned q = 0; q < cl; ++q) v += cluster.map_shared_rank(s_tile, q)[k];
      }
    } else {
      v = fixed ? __fmaf_rn(__int2float_rn(s_hi[k]), hscale, __int2float_rn(s_hi[words + k]) * unscale) : s_tile[k];
    }
    mesh[at] = rmesh ? fmaf(ran_scale, rmesh[at], v) : v;
  }
  if constexpr (MULTI) cluster.sync();  // every copy stays until the last CTA has read it
}

// FP64 sums of a random catalogue (sum w, sum w^2, sum w^2 nbar) for the kept copy.
__global__ void k_ran_sums(const float* __restrict__ w, const float* __restrict__ nbar, int64_t n,
                           double* __restrict__ out) {
  double s[3] = {0.0, 0.0, 0.0};
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const double v = w ? (double)w[i] : 1.0;
    s[0] += v;
    s[1] += v * v;
    if (nbar) s[2] += v * v * (double)nbar[i];
  }
  for (int k = 0; k < 3; ++k) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s[k] += __shfl_xor_sync(0xffffffffu, s[k], o);
    if ((threadIdx.x & 31) == 0) atomicAdd(&out[k], s[k]);
  }
}

// Catalogue sums of Eqs. (1) and (3) without the counting pass: four CTAs per SM with eight
// particles in flight per thread (with eight CTAs and four the meeting of the threads, twice
// as much, takes 1 us longer).
__global__ void __launch_bounds__(THREADS)
k_sums(const __grid_constant__ Cats cats, double* __restrict__ sums) {
  int bid, nblk;
  const int is_ran = block_catalogue(cats, bid, nblk);
  const float* __restrict__ pw = cats.w[is_ran];
  const float* __restrict__ pnbar = is_ran ? cats.nbar[1] : nullptr;
  const int64_t n = cats.n[is_ran];
  ThreadSums ts;
  const int64_t stride = (int64_t)nblk * THREADS;
  constexpr int U = 8;  // particles per iteration, whose loads are issued together
  for (int64_t base = (int64_t)bid * THREADS + threadIdx.x; base < n; base += U * stride) {
    float w[U], nb[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int64_t i = min(base + u * stride, n - 1);
      w[u] = pw ? pw[i] : 1.f;
      nb[u] = pnbar ? pnbar[i] : 0.f;
    }
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (base + u * stride < n) ts.particle(w[u], pnbar, nb[u]);
  }
  block_sums<THREADS>(ts, 0u, is_ran, sums);
}

// ---------------------------------------------------------------------------
// Direct assignment for meshes that stay resident in L2 (m N^3 floats of at most
// 64 MB, half of it): one pass over each catalogue adds every stencil weight
// into the zeroed mesh with global float reductions, served in L2.  The catalogue
// sums come first (the randoms carry -alpha w), so particles are read twice in all
// (4-12 bytes, then 16) instead of the sort's count, bin and deposit passes.
// ---------------------------------------------------------------------------

// row[z[c]] += wxy wz[c] for the KIND consecutive nodes z[0] .. of a mesh row (n a
// multiple of 4 nodes, periodic).  The reductions are bound by L2 operations, not bytes, so
// the nodes of one aligned group of four go in one 16-byte reduction (zeros elsewhere):
// a CIC pair takes 1.25 operations instead of 2 on average, TSC 1.5 instead of 3.
// 6.6e6 particles, CIC, 128^3: 260 -> 170 us.
template <int KIND>
__device__ __forceinline__ void add_row(float* row, const int (&z)[3], float wxy, const float (&wz)[3]) {
  if constexpr (KIND == 1) {
    atomicAdd(row + z[0], wxy * wz[0]);
  } else {
    float v[KIND];
#pragma unroll
    for (int c = 0; c < KIND; ++c) v[c] = wxy * wz[c];
    const int q0 = z[0] >> 2, q1 = z[KIND - 1] >> 2, at = z[0] & 3;  // groups of the first and last node
    float g[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      g[k] = 0.f;
#pragma unroll
      for (int c = 0; c < KIND; ++c)
        if (at + c == k) g[k] = v[c];
    }
    atomicAdd(reinterpret_cast<float4*>(row) + q0, make_float4(g[0], g[1], g[2], g[3]));
    if (q1 != q0) {
      // the nodes past the group: the last one, or the last two of three
      if (KIND == 3 && at == 3) atomicAdd(reinterpret_cast<float4*>(row) + q1, make_float4(v[1], v[KIND - 1], 0.f, 0.f));
      else atomicAdd(row + z[KIND - 1], v[KIND - 1]);
    }
  }
}

template <int KIND, int M>
__global__ void __launch_bounds__(THREADS)
k_direct(const __grid_constant__ Cats cats, Geom g, const float2* __restrict__ nodes, double* __restrict__ sums,
         double alpha_cfg, float* __restrict__ mesh) {
  int bid, nblk;
  const int is_ran = block_catalogue(cats, bid, nblk);
  const float* __restrict__ px = cats.x[is_ran];
  const float* __restrict__ py = cats.y[is_ran];
  const float* __restrict__ pz = cats.z[is_ran];
  const float* __restrict__ pw = cats.w[is_ran];
  const int64_t n = cats.n[is_ran];
  const float wscale = catalogue_scale(is_ran, alpha_cfg, sums);
  const int nn = g.n;
  const size_t n3 = (size_t)nn * nn * nn;
  unsigned bad = 0;
  const int64_t stride = (int64_t)nblk * blockDim.x;
  for (int64_t idx = (int64_t)bid * blockDim.x + threadIdx.x; idx < n; idx += stride) {
    const float x = px[idx], y = py[idx], z = pz[idx];
    const float w = (pw ? pw[idx] : 1.f) * wscale;
    int ci[3];
    float cd[3];
    bool ok = locate(x, 0, g, nodes, ci[0], cd[0]);
    ok &= locate(y, 1, g, nodes, ci[1], cd[1]);
    ok &= locate(z, 2, g, nodes, ci[2], cd[2]);
    bad += ok ? 0u : 1u;
#pragma unroll
    for (int mj = 0; mj < M; ++mj) {
      int node[3][3];
      float wt[3][3];
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        int first;
        stencil<KIND>(ci[a], cd[a], mj == 1, first, wt[a]);
#pragma unroll
        for (int s = 0; s < KIND; ++s) node[a][s] = wrapn(first + s, nn);
      }
      float* mm = mesh + mj * n3;
#pragma unroll
      for (int a = 0; a < KIND; ++a)
#pragma unroll
        for (int b = 0; b < KIND; ++b) {
          const float wxy = w * wt[0][a] * wt[1][b];
          float* row = mm + ((size_t)node[0][a] * nn + node[1][b]) * nn;
          add_row<KIND>(row, node[2], wxy, wt[2]);
        }
    }
  }
  unsigned tot = bad;  // particles outside the box
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) tot += __shfl_xor_sync(0xffffffffu, tot, o);
  if ((threadIdx.x & 31) == 0 && tot) atomicAdd(&sums[SUM_BAD], (double)tot);
}

// The two catalogues of a launch of `grid` blocks, shared out by their particle counts
// (at least one block each).
Cats make_cats(const ys_catalog& gal, const ys_catalog& ran, int& grid) {
  Cats c{};
  const ys_catalog* k[2] = {&gal, &ran};
  for (int i = 0; i < 2; ++i) {
    c.x[i] = k[i]->x;
    c.y[i] = k[i]->y;
    c.z[i] = k[i]->z;
    c.w[i] = k[i]->w;
    c.nbar[i] = k[i]->nbar;
    c.n[i] = k[i]->n;
  }
  const double total = (double)gal.n + (double)ran.n;
  if (gal.n > 0 && ran.n > 0) {
    grid = std::max(grid, 2);
    c.blocks0 = std::min(grid - 1, std::max(1, (int)(grid * (gal.n / total) + 0.5)));
  } else {
    grid = std::max(grid, 1);
    c.blocks0 = gal.n > 0 ? grid : 0;
  }
  return c;
}

int blocks_for(int64_t n, int per_block, int most) {
  return (int)std::max<int64_t>(1, std::min<int64_t>((n + per_block - 1) / per_block, most));
}

template <int KIND, int M>
cudaError_t run_direct(Plan& p, const ys_catalog& gal, const ys_catalog& ran) {
  cudaStream_t st = p.stream;
  cudaError_t err;
  const size_t n3 = (size_t)p.n * p.n * p.n;
  if ((err = cudaMemsetAsync(p.d_sums, 0, sizeof(double) * SUM_COUNT, st))) return err;
  if ((err = cudaMemsetAsync(p.d_mesh, 0, sizeof(float) * p.m * n3, st))) return err;
  int dev = 0, sms = 0;
  if ((err = cudaGetDevice(&dev)) || (err = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)))
    return err;
  const int64_t total = gal.n + ran.n;
  if (total == 0) return cudaSuccess;
  {
    int grid = blocks_for(total, 8 * THREADS, sms * 4);
    const Cats cats = make_cats(gal, ran, grid);
    LaunchScope ls(p, 0);
    k_sums<<<grid, THREADS, 0, st>>>(cats, p.d_sums);
    if ((err = cudaGetLastError())) return err;
  }
  int grid = blocks_for(total, THREADS, sms * 8);
  const Cats cats = make_cats(gal, ran, grid);
  LaunchScope ls(p, 3);
  k_direct<KIND, M><<<grid, THREADS, 0, st>>>(cats, p.geom, p.d_nodes, p.d_sums, p.cfg.alpha, p.d_mesh);
  return cudaGetLastError();
}

// The counting pass with NT threads per CTA.
template <int KIND, int M, int NT>
cudaError_t run_count(Plan& p, const ys_catalog& gal, const ys_catalog& ran, int sms) {
  cudaError_t err;
  const int64_t total = gal.n + ran.n;
  // shared-memory histograms while the tile counters fit (a few CTAs per SM)
  const size_t hist_bytes = sizeof(unsigned) * (size_t)p.ntiles;
  const bool hist = hist_bytes <= 160u * 1024u;
  auto kern = hist ? k_particles<KIND, M, true, NT> : k_particles<KIND, M, false, NT>;
  const size_t smem = hist ? hist_bytes : 0;
  int per = 0;
  if (hist && (err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem))) return err;
  if ((err = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kern, NT, smem))) return err;
  int grid = blocks_for(total, NT, std::max(1, per) * sms);
  const Cats cats = make_cats(gal, ran, grid);
  LaunchScope ls(p, 0);
  kern<<<grid, NT, smem, p.stream>>>(cats, p.geom, p.d_nodes, p.d_tile_count, p.d_sums, p.ntiles,
                                       p.ntiles <= BIN_AGG_TILES ? p.d_codes : nullptr);
  return cudaGetLastError();
}

// CTAs per tile of the deposit: doubled (up to 8) while there are fewer than five per SM
// and a CTA would still get 256 records.  Times in us with 1, 2, 4 and 8 CTAs per tile, on
// 152 SMs, CIC, 6.6e6 particles: 64 tiles 491, 368, 204, 189 (8 taken); 216 tiles 175, 140, 130,
// 168 (4); 512 tiles 142, 153, 153, 210 (2; TSC interlaced 532, 481, 491, 577); 1728 tiles 104,
// 176, 234, 416 (1).  6e5 particles: 64 tiles 40, 35, 25, 34; 216 tiles 21, 23, 31, 58; 512
// tiles 23, 38, 52, 108: so few records would want half of what the rule takes.
int deposit_cluster(int ntiles, int64_t particles, int sms) {
  int cl = 1;
  while (cl < 8 && (int64_t)ntiles * cl < 5 * sms && particles / ((int64_t)ntiles * 2 * cl) >= 256) cl *= 2;
  return cl;
}

// rmesh != nullptr (shared randoms): ran is empty, the random sums come from rsums
// (sum w, sum w^2, sum w^2 nbar) and the deposit subtracts alpha rmesh.
template <int KIND, int M>
cudaError_t run_assign(Plan& p, const ys_catalog& gal, const ys_catalog& ran, const float* rmesh = nullptr,
                       const double* rsums = nullptr) {
  cudaStream_t st = p.stream;
  cudaError_t err;
  if ((err = cudaMemsetAsync(p.d_tile_count, 0, sizeof(unsigned) * p.ntiles, st)) != cudaSuccess) return err;
  if ((err = cudaMemsetAsync(p.d_sums, 0, sizeof(double) * SUM_COUNT, st)) != cudaSuccess) return err;
  if (rsums && (err = cudaMemcpyAsync(p.d_sums + SUM_WR, rsums, sizeof(double) * 3, cudaMemcpyDeviceToDevice, st)))
    return err;
  int dev = 0, sms = 0;
  if ((err = cudaGetDevice(&dev)) || (err = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)))
    return err;
  const int64_t total = gal.n + ran.n;
  // CTAs of 1024 threads share one histogram; a catalogue that would leave most of them
  // idle takes CTAs of 256 (shorter sums at their end)
  if (total > 0 && (err = total >= (int64_t)sms * 1024 ? run_count<KIND, M, 1024>(p, gal, ran, sms)
                                                       : run_count<KIND, M, 256>(p, gal, ran, sms)))
    return err;
  {
    LaunchScope ls(p, 1);
    k_scan<<<(p.ntiles + 1023) / 1024, 1024, 0, st>>>(p.d_tile_count, p.ntiles, p.d_tile_off, p.d_tile_cur);
    if ((err = cudaGetLastError()) != cudaSuccess) return err;
  }
  if (total > 0 && p.ntiles <= BIN_AGG_TILES) {
    // chunks of up to 16 particles per thread, in whole waves of three CTAs per SM
    const int64_t wave = (int64_t)BIN_AGG_NT * sms * 3, waves = (total + 16 * wave - 1) / (16 * wave);
    const int per_thread = (int)((total + wave * waves - 1) / (wave * waves));
    const int chunk = BIN_AGG_NT * per_thread;
    int grid = 1;
    Cats cats = make_cats(gal, ran, grid);
    cats.blocks0 = (int)((gal.n + chunk - 1) / chunk);
    grid = cats.blocks0 + (int)((ran.n + chunk - 1) / chunk);
    const size_t smem = 2 * sizeof(unsigned) * (size_t)p.ntiles;
    LaunchScope ls(p, 2);
    auto bin = p.d_codes ? k_bin_agg<KIND, M, true> : k_bin_agg<KIND, M, false>;
    bin<<<grid, BIN_AGG_NT, smem, st>>>(cats, per_thread, p.geom, p.d_nodes, p.d_codes, p.ntiles, p.d_tile_off,
                                        p.d_tile_count, p.d_tile_cur, p.d_rec, p.d_sums, p.cfg.alpha);
    if ((err = cudaGetLastError()) != cudaSuccess) return err;
  } else if (total > 0) {
    constexpr int U = 2;
    int grid = blocks_for(total, U * THREADS, sms * 16);
    const Cats cats = make_cats(gal, ran, grid);
    LaunchScope ls(p, 2);
    k_bin<KIND, M, U><<<grid, THREADS, 0, st>>>(cats, p.geom, p.d_nodes, p.d_tile_off, p.d_tile_count, p.d_tile_cur,
                                                p.d_rec, p.d_sums, p.cfg.alpha);
    if ((err = cudaGetLastError()) != cudaSuccess) return err;
  }
  const int tvol = p.geom.tdim[0] * p.geom.tdim[1] * p.geom.tdim[2];
  int optin = 0;
  if ((err = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev))) return err;
  // fixed-point sums need two words per node; a tile that cannot hold them sums in float
  const size_t words = (size_t)M * tvol + 32;  // nodes and one trash word per lane
  const size_t smem_fixed = 2 * sizeof(float) * words;
  const bool fixed = smem_fixed + 64 <= (size_t)optin;
  const size_t smem = fixed ? smem_fixed : sizeof(float) * words;
  const int cl = deposit_cluster(p.ntiles, total, sms);
  const bool cube16 = p.geom.tdim[0] == 16 && p.geom.tdim[1] == 16 && p.geom.tdim[2] == 16;
  auto kern = cube16 ? (cl > 1 ? k_deposit<KIND, M, true, true, 16> : k_deposit<KIND, M, true, false, 16>)
              : fixed ? (cl > 1 ? k_deposit<KIND, M, true, true, 0> : k_deposit<KIND, M, true, false, 0>)
                      : (cl > 1 ? k_deposit<KIND, M, false, true, 0> : k_deposit<KIND, M, false, false, 0>);
  if ((err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) != cudaSuccess)
    return err;
  LaunchScope ls(p, 3);
  cudaLaunchConfig_t cfg{};
  cudaLaunchAttribute attr{};
  cfg.gridDim = dim3((unsigned)p.ntiles * cl);
  cfg.blockDim = dim3(THREADS);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  if (cl > 1) {
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = (unsigned)cl;
    attr.val.clusterDim.y = 1;
    attr.val.clusterDim.z = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
  }
  return cudaLaunchKernelEx(&cfg, kern, p.geom, (const float2*)p.d_nodes, (const unsigned*)p.d_tile_off,
                            (const unsigned*)p.d_tile_cur, (const float4*)p.d_rec, p.d_mesh, rmesh,
                            (const double*)p.d_sums, p.cfg.alpha);
}

}  // namespace

cudaError_t launch_assign(Plan& p, const ys_catalog& gal, const ys_catalog& ran, const float* rmesh,
                          const double* rsums) {
  const int key = p.kind * 2 + (p.m - 1);
  if (p.direct_assign && !rmesh) {
    switch (key) {
      case 2: return run_direct<1, 1>(p, gal, ran);
      case 3: return run_direct<1, 2>(p, gal, ran);
      case 4: return run_direct<2, 1>(p, gal, ran);
      case 5: return run_direct<2, 2>(p, gal, ran);
      case 6: return run_direct<3, 1>(p, gal, ran);
      case 7: return run_direct<3, 2>(p, gal, ran);
      default: return cudaErrorInvalidValue;
    }
  }
  switch (key) {
    case 2: return run_assign<1, 1>(p, gal, ran, rmesh, rsums);
    case 3: return run_assign<1, 2>(p, gal, ran, rmesh, rsums);
    case 4: return run_assign<2, 1>(p, gal, ran, rmesh, rsums);
    case 5: return run_assign<2, 2>(p, gal, ran, rmesh, rsums);
    case 6: return run_assign<3, 1>(p, gal, ran, rmesh, rsums);
    case 7: return run_assign<3, 2>(p, gal, ran, rmesh, rsums);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_random_sums(Plan& p, const ys_catalog& ran, double* out) {
  cudaError_t e = cudaMemsetAsync(out, 0, sizeof(double) * 3, p.stream);
  if (e || ran.n == 0) return e;
  const int blocks = blocks_for(ran.n, THREADS, 152 * 8);
  k_ran_sums<<<blocks, THREADS, 0, p.stream>>>(ran.w, ran.nbar, ran.n, out);
  return cudaGetLastError();
}

}  // namespace ys
