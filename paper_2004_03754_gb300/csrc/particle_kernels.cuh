// particle_kernels.cuh -- the tiled particle kernel and the straggler kernel of
// libpic with their launchers, as templates over the field type; particles_f32.cu,
// particles_f64.cu and particles_dfl.cu instantiate one field type each (parallel
// compilation).
//
// Particles are binned by tile (a box of cells).  The Faraday pass has formed the
// time-centred B^n = B^{n-1/2} - (dt/2) d_E x E^n (Eq. (7) in its half-step form)
// over the grid.  One CTA owns one tile: it stages E^n and B^n of the tile plus
// a guard in shared memory and runs every particle of the bin through
//   gather (App. A, quadratic B-spline at each component's staggered node)
//   -> push (Boris, Higuera-Cary or analytic, FP64; next to FP32 fields the parts of
//      it that lose nothing by it in FP32 pairs, pair_push.cuh)
//   -> x^{n+1} = x^n + dt u/gamma (FP64)
//   -> Esirkepov deposit (Sec. 3.3) into a shared-memory current window (int32
//      fixed point),
// then adds the window into the global current once.  Bins are rebuilt every
// few steps; a particle that has drifted out of its tile's window takes the
// global-memory path of straggler_kernel instead, so correctness never depends
// on the rebinning interval.
#pragma once
#include <math.h>

#include <type_traits>

#include "common.cuh"
#include "field_tile.cuh"
#include "particle_core.cuh"

namespace pic {

namespace {

// 16-byte (N = 16) or single-value copies into shared memory, in flight until
// stage_wait
template <int N>
__device__ __forceinline__ void stage_copy(void* dst, const void* src) {
  if constexpr (N == 16)   // (8 bytes: two FP32 columns)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_addr(dst)), "l"(src) : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(smem_addr(dst)), "l"(src), "n"(N) : "memory");
}
__device__ __forceinline__ void stage_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// The rows (l2, l3) of a window in chunks: f(o, j, k, c) for every chunk -- o its
// offset in a component of the window, (j, k) its x2, x3 grid indices, c its x1 grid
// column -- spread over the CTA's threads.  A chunk is C values (16 bytes, or one
// value where grid rows don't start on 16-byte boundaries); the thread's chunk
// advances by the same step each time, so no division runs in the loop but the one
// by W2 (3D).  All three components share the index arithmetic.
template <int C, int NDIM, class F>
__device__ __forceinline__ void for_window_chunks(const int* W, const int* wlo, const GridArgs& g,
                                                  F&& f) {
  const int cpr = W[0] / C, rows = W[1] * W[2];
  const int dr = (int)blockDim.x / cpr, dc = (int)blockDim.x - dr * cpr;
  int row = (int)threadIdx.x / cpr, ch = (int)threadIdx.x - row * cpr;
  while (row < rows) {
    const int l3 = NDIM == 3 ? row / W[1] : 0, l2 = NDIM == 3 ? row - l3 * W[1] : row;
    f(row * W[0] + ch * C, pwrap(wlo[1] + l2, g.n[1]), NDIM == 3 ? pwrap(wlo[2] + l3, g.n[2]) : 0,
      pwrap(wlo[0] + ch * C, g.n[0]));
    row += dr;
    ch += dc;
    if (ch >= cpr) {
      ch -= cpr;
      ++row;
    }
  }
}

// p[0..3] += v[0..3], one 16-byte reduction
__device__ __forceinline__ void red_add4(float* p, const float* v) {
  asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(p), "f"(v[0]), "f"(v[1]), "f"(v[2]),
               "f"(v[3])
               : "memory");
}

// cell of a coordinate in cells and the fraction in the field precision (exact, rounded
// once; no FP64 conversion)
template <typename T>
__device__ __forceinline__ int cell_split(double c, T& f) {
  if constexpr (std::is_same<T, float>::value) {
    return floor_split(c, f);
  } else {
    double frac;
    const int k = floor_split(c, frac);
    f = to_prec<T>(frac);
    return k;
  }
}

// threads 0 .. NDIM+3 ask L2 for one particle array each over [c0, c1) (bulk
// prefetch: 16-byte aligned start and size, so the range is cut to even indices)
template <int NDIM>
__device__ __forceinline__ void prefetch_chunk(const PartPtrs& p, int64_t c0, int64_t c1) {
  const int t = threadIdx.x;
  if (t >= NDIM + 4) return;
  const int64_t s0 = c0 & ~1LL, e0 = c1 & ~1LL;
  if (e0 <= s0) return;
  const int c = t - NDIM;   // constant indices only: the pointer arrays stay in the parameter bank
  const double* arr = t < NDIM ? (t == 0 ? p.x[0] : (t == 1 ? p.x[1] : p.x[2]))
                               : (c == 0 ? p.u[0] : (c == 1 ? p.u[1] : (c == 2 ? p.u[2] : p.w)));
  if ((reinterpret_cast<uintptr_t>(arr) & 15u) != 0) return;   // a hint only: skip if unaligned
  asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(arr + s0),
               "r"((unsigned)((e0 - s0) * 8)) : "memory");
}

// Threads per CTA and CTAs per SM of the tile kernel, with the tile shapes of
// choose_particle_tiles.  Measured, steps and their read-back: 3D FP32, 84 M electrons,
// two analytic steps 2 x 512 threads 42.8 ms (a thread per particle of a tile at 2 per
// cell; 3 x 256 44.6, 2 x 384 47.8); 3D FP64, four steps on 301x60x44, one CTA of 384 on
// 8x8x8 cells 11.6 ms (512 threads 11.8, 2 x 256 on 8x8x4 12.0); 3D compensated (8x8x4,
// 103 KB of windows), four Boris steps of 96^3 at 2 per cell and of 301x60x44 at 1,
// 2 x 384 5.27 and 3.13 ms (1 x 384 6.71 and 4.49, 1 x 512 6.18 and 4.35, 2 x 256 5.45 and
// 3.49, 2 x 320 5.27 and 3.12, but analytic 8.75 against 8.04); 2D FP32, ten Boris steps of
// 29 M electrons, 3 x 256 at 80 registers 20.0 ms (2 x 384 20.4, 4 x 256 at 64, which spill,
// 20.7; 2 x 256 22.9; 1 x 512 24.0).
template <typename T, int NDIM>
struct TileCfg {
  static constexpr bool F = sizeof(T) == 4, C = is_dfl<T>::value;
  static constexpr int threads = NDIM == 3 ? (F ? 512 : 384) : 256;
  static constexpr int ctas = NDIM == 3 ? (F || C ? 2 : 1) : (F ? 3 : 2);
};

// The time-centred B^n is read from a global array formed once per step; E^n and
// B^n are staged over the particle window by asynchronous 16-byte copies, the
// current is accumulated in a shared-memory window (in int32 fixed point, FixAcc /
// FixAcc64) and added into the global current once, 16 bytes at a time for FP32.
// In 3D a tile holds few particles per window node (512 particles at 2 per cell, 924
// nodes of E, B and 1872 of the current), so the window's handling counts as much as
// the particles': copied and flushed value by value it took half the kernel's
// instructions (84 M electrons, two steps and their read-back 62.8 -> 38.7 ms; 2D,
// 29 M electrons, ten steps 23.7 -> 19.1 ms; both with a cheaper, less accurate push
// than now, 42.8 and 20.0 ms).
template <typename T, int NDIM, int PUSH, bool GAIN>
__global__ void __launch_bounds__(TileCfg<T, NDIM>::threads, TileCfg<T, NDIM>::ctas)
    particle_kernel(FieldPtrs<T> f, BbarPtrs<T> bg, PartPtrs p, GridArgs g, StencilArgs<T> s,
                    PartTile t, PartArgs a, BinBufs bins) {
  using D = typename DepositOf<T>::type;
  constexpr int V = VecOf<T>::V;
  // current window: FP32 deposits as two int32 fixed-point sums (FixAcc), FP64
  // deposits as three (FixAcc64)
  constexpr bool F64 = std::is_same<D, double>::value;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ unsigned long long wmax_warp[32];
  T* sm = reinterpret_cast<T*>(smem_raw);
  // CTAs beyond the tiles take the further shares of crowded tiles
  unsigned tile = blockIdx.x;
  int part = 0;
  if (tile >= t.ntiles) {
    const unsigned x = tile - (unsigned)t.ntiles;
    if (x >= (unsigned)bins.share.counts[0]) return;
    const TileShare sh = bins.share.list[x];
    tile = (unsigned)sh.tile;
    part = sh.part;
  }
  const int64_t tbeg = bins.start[tile], tend = bins.start[tile + 1];
  if (tbeg == tend) return;
  int64_t pbeg = tbeg, pend = tend;
  // (in shared memory: read again after the particle loop, no registers held across it)
  __shared__ int s_parts, s_slot;
  if (threadIdx.x == 0) s_parts = 1;
  if (bins.share.chunk > 0 && tend - tbeg > *bins.share.line) {
    const int parts = (int)((tend - tbeg + bins.share.chunk - 1) / bins.share.chunk);
    const int64_t per = (tend - tbeg + parts - 1) / parts;
    pbeg = min(tend, tbeg + part * per);
    pend = min(tend, pbeg + per);
    if (threadIdx.x == 0) {
      s_parts = parts;
      s_slot = bins.share.slot[tile];
    }
  }
  prefetch_chunk<NDIM>(p, pbeg, min(pend, pbeg + (int64_t)blockDim.x));
  int tc[3];
  {
    const unsigned r = tile / (unsigned)t.nt[0];
    tc[0] = (int)(tile - r * (unsigned)t.nt[0]);
    tc[2] = NDIM == 3 ? (int)(r / (unsigned)t.nt[1]) : 0;
    tc[1] = (int)(r - (unsigned)tc[2] * (unsigned)t.nt[1]);
  }
  const int n1 = g.n[0], n2 = g.n[1];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarp = blockDim.x >> 5;
  // two windows (common.cuh): E, B over the particles' gather, the current over
  // their deposit; g - 3 cells of drift are allowed on both sides
  int We[3], elo[3], W[3], wlo[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const WindowAxis ew = d < NDIM ? eb_window(d, t.t[d], t.g[d]) : WindowAxis{0, 1};
    const WindowAxis jw = d < NDIM ? j_window(d, t.t[d], t.g[d], V) : WindowAxis{0, 1};
    We[d] = ew.w;
    W[d] = jw.w;
    elo[d] = d < NDIM ? tc[d] * t.t[d] - ew.lo : 0;
    wlo[d] = d < NDIM ? tc[d] * t.t[d] - jw.lo : 0;
  }
  const int nE = We[0] * We[1] * We[2], nW = W[0] * W[1] * W[2];
  T* sE = sm;                 // [3][We3][We2][We1]
  T* sB = sE + 3 * nE;        // [3][We3][We2][We1], the time-centred B
  int* sJh = reinterpret_cast<int*>(smem_raw + ((size_t)nE * 6 * sizeof(T) + 15) / 16 * 16);
  int* sJl = sJh + 3 * nW;    // current: [3][W3][W2][W1] per limb, hi first
  int* sJc = sJl + 3 * nW;    // FP64: the third limb
  // rows on 2-column and on 16-byte boundaries
  const bool pairs = (n1 & 1) == 0, vec = n1 % V == 0;

  auto stage = [&](auto C) {
    constexpr int c = decltype(C)::value;
    for_window_chunks<c, NDIM>(We, elo, g, [&](int o, int j, int k, int i) {
      const int64_t r = ((int64_t)k * n2 + j) * n1 + i;
      stage_copy<c * (int)sizeof(T)>(sE + o, f.e[0] + r);
      stage_copy<c * (int)sizeof(T)>(sE + nE + o, f.e[1] + r);
      stage_copy<c * (int)sizeof(T)>(sE + 2 * nE + o, f.e[2] + r);
      stage_copy<c * (int)sizeof(T)>(sB + o, bg.b[0] + r);
      stage_copy<c * (int)sizeof(T)>(sB + nE + o, bg.b[1] + r);
      stage_copy<c * (int)sizeof(T)>(sB + 2 * nE + o, bg.b[2] + r);
    });
  };
  if (pairs) stage(std::integral_constant<int, 2>{});
  else stage(std::integral_constant<int, 1>{});
  {
    // largest |w| of the tile (non-negative doubles order as their bit patterns)
    unsigned long long wm = 0ull;
    for (int64_t q = tbeg + threadIdx.x; q < tend; q += blockDim.x)
      wm = max(wm, (unsigned long long)__double_as_longlong(p.w[q]) & 0x7fffffffffffffffull);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) wm = max(wm, __shfl_xor_sync(0xffffffffu, wm, o));
    if (lane == 0) wmax_warp[warp] = wm;
  }
  // (the width is a multiple of V, so the limbs are whole 8- or 16-byte words)
  for (int q = threadIdx.x * 4; q < (F64 ? 9 : 6) * nW; q += blockDim.x * 4) {
    if (q + 4 <= (F64 ? 9 : 6) * nW) *reinterpret_cast<int4*>(sJh + q) = make_int4(0, 0, 0, 0);
    else *reinterpret_cast<int2*>(sJh + q) = make_int2(0, 0);
  }
  stage_wait();
  __syncthreads();
  float S = 1.0f, L = 1.0f;
  int eS = 0, l64 = 0;
  bool finite;
  {
    unsigned long long wm = 0ull;
    for (int k = 0; k < nwarp; ++k) wm = max(wm, wmax_warp[k]);
    // |contribution| <= |w|: a J_d term is -w (dx_d/dt) times a difference of the
    // cumulative shape weights before and after the move (at most |delta_d| in
    // magnitude: the node sums of the quadratic spline have slope <= 1) times a
    // time-averaged shape weight (<= 1), so at most |w| |v_d| < |w|; the 2D
    // out-of-plane term is w v3 times a path-averaged weight product (<= 1)
    finite = wm < 0x7ff0000000000000ull;
    if constexpr (F64) fix64_scales(tend - tbeg, __longlong_as_double((long long)wm), eS, l64);
    else fix_scales(tend - tbeg, narrow_signed(__longlong_as_double((long long)wm)) * 1.001f, S, L);
  }

  // views indexed by the current window's node
  SmemView<T> ve[3], vb[3];
  const int eoff = ((elo[2] - wlo[2]) * We[1] + (elo[1] - wlo[1])) * We[0] + (elo[0] - wlo[0]);
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    ve[c] = SmemView<T>{sE + c * nE - eoff, We[0], We[0] * We[1], 0};
    vb[c] = SmemView<T>{sB + c * nE - eoff, We[0], We[0] * We[1], 0};
  }
  using Acc = typename std::conditional<F64, FixAcc64, FixAcc>::type;
  Acc acc[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    if constexpr (F64)
      acc[c] = FixAcc64{sJh + c * nW, sJl + c * nW, sJc + c * nW, W[0], W[0] * W[1], eS, l64};
    else acc[c] = FixAcc{sJh + c * nW, sJl + c * nW, W[0], W[0] * W[1], S, L};
  }
  const float invS = 1.0f / S, invSL = 1.0f / (S * L);   // powers of two: exact
  // FP64 limb weights 2^-eS, 2^-(eS + l), 2^-(eS + 2l), from the exponent bits; with an
  // infinite or NaN weight in the tile the integers mean nothing and its current is NaN
  auto pow2 = [](int e) { return __longlong_as_double((long long)(uint64_t)(1023 + e) << 52); };
  const double i0 = F64 ? (finite ? pow2(-eS) : __longlong_as_double(0x7ff8000000000000ll)) : 0.0,
               i1 = F64 ? pow2(-eS - l64) : 0.0, i2 = F64 ? pow2(-eS - 2 * l64) : 0.0;
  // value of window node q of component c
  auto jval = [&](int c, int q) -> D {
    if constexpr (F64) return fix64_decode(sJh[c * nW + q], sJl[c * nW + q], sJc[c * nW + q], i0, i1, i2);
    else return fix_decode(sJh[c * nW + q], sJl[c * nW + q], invS, invSL);
  };
  // window-local cell index: periodic unwrap limits [ulo, uhi) (the grid's period
  // centred on the tile with its drift) and the cells a particle may be in
  int ulo[3], uhi[3], lmin[3], lmax[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const int tile0 = d < NDIM ? tc[d] * t.t[d] - wlo[d] : 0, dr = d < NDIM ? t.g[d] - 3 : 0;
    lmin[d] = tile0 - dr;
    lmax[d] = tile0 + (d < NDIM ? t.t[d] : 1) - 1 + dr;
    ulo[d] = lmin[d] + (lmax[d] - lmin[d] + 1 - g.n[d]) / 2;
    uhi[d] = ulo[d] + g.n[d];
  }
  for (int64_t q = pbeg + threadIdx.x; q < pend; q += blockDim.x) {
    {
      const int64_t c0 = q - threadIdx.x + blockDim.x;
      if (c0 < pend) prefetch_chunk<NDIM>(p, c0, min(pend, c0 + (int64_t)blockDim.x));
    }
    int li[3], gc[3];
    T fr[3];
    bool inside = true;
#pragma unroll
    for (int d = 0; d < NDIM; ++d) {
      gc[d] = cell_split(p.x[d][q] * g.inv_dx[d], fr[d]);
      int l = gc[d] - wlo[d];
      if (l < ulo[d]) l += g.n[d];
      else if (l >= uhi[d]) l -= g.n[d];
      li[d] = l;
      inside = inside && l >= lmin[d] && l <= lmax[d];
    }
    if (!inside) {
      const unsigned long long slot = atomicAdd(bins.strag_count, 1ull);
      bins.strag[slot] = q;
      continue;
    }
    advance_particle<T, NDIM, PUSH, GAIN>(ve, vb, acc, p, q, li, fr, gc, g, a, bins.err);
  }
  __syncthreads();
  if (s_parts > 1) {
    // add this share's integers to the tile's; the last share takes the sum
    __shared__ int last;
    int* scr = bins.share.scratch + (size_t)s_slot * bins.share.words;
    const int words = (F64 ? 9 : 6) * nW;
    for (int q = threadIdx.x; q < words; q += blockDim.x)
      if (sJh[q] != 0) atomicAdd(scr + 4 + q, sJh[q]);
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(scr, 1) == s_parts - 1;
    __syncthreads();
    if (!last) return;
    __threadfence();
    for (int q = threadIdx.x; q < words; q += blockDim.x) {
      sJh[q] = __ldcg(scr + 4 + q);
      scr[4 + q] = 0;   // for the next step
    }
    if (threadIdx.x == 0) scr[0] = 0;
    __syncthreads();
  }
  auto flush = [&](auto C) {
    constexpr int c = decltype(C)::value;
    for_window_chunks<c, NDIM>(W, wlo, g, [&](int o, int j, int k, int i) {
      const int64_t r = ((int64_t)k * n2 + j) * n1 + i;
#pragma unroll
      for (int m = 0; m < 3; ++m) {
        T* dst = (m == 0 ? f.j[0] : (m == 1 ? f.j[1] : f.j[2])) + r;
        D v[c];
        bool any = false;
#pragma unroll
        for (int e = 0; e < c; ++e) {
          v[e] = jval(m, o + e);
          any = any || v[e] != (D)0;
        }
        if (!any) continue;
        if constexpr (c == 4 && std::is_same<T, float>::value) {
          red_add4(dst, v);
        } else {
#pragma unroll
          for (int e = 0; e < c; ++e)
            if (v[e] != (D)0) atomic_acc(dst + e, v[e]);
        }
      }
    });
  };
  const int n3 = NDIM == 3 ? g.n[2] : 1;
  if (W[0] > n1 || W[1] > n2 || W[2] > n3) {
    // the window wraps onto itself: one thread per grid node sums its window nodes,
    // in a fixed order
    const int m0 = min(W[0], n1), m1 = min(W[1], n2), m2 = min(W[2], n3);
    for (int q = threadIdx.x; q < m0 * m1 * m2; q += blockDim.x) {
      const int r = q / m0, i0 = q - r * m0, k0 = r / m1, j0 = r - k0 * m1;
      const int64_t o = ((int64_t)pwrap(wlo[2] + k0, n3) * n2 + pwrap(wlo[1] + j0, n2)) * n1 +
                        pwrap(wlo[0] + i0, n1);
#pragma unroll
      for (int m = 0; m < 3; ++m) {
        D v = 0;
        for (int k = k0; k < W[2]; k += n3)
          for (int j = j0; j < W[1]; j += n2)
            for (int i = i0; i < W[0]; i += n1) v += jval(m, (k * W[1] + j) * W[0] + i);
        if (v != (D)0) atomic_acc((m == 0 ? f.j[0] : (m == 1 ? f.j[1] : f.j[2])) + o, v);
      }
    }
  } else if (vec) {
    flush(std::integral_constant<int, V>{});
  } else {
    flush(std::integral_constant<int, 1>{});
  }
}

// Particles that left their tile's window: the whole update through global
// memory, with the time-centred B from bg.
template <typename T, int NDIM, bool GAIN>
__global__ void straggler_kernel(FieldPtrs<T> f, BbarPtrs<T> bg, PartPtrs p, GridArgs g,
                                 StencilArgs<T> s, PartArgs a, BinBufs bins) {
  (void)s;
  const unsigned long long cnt = *bins.strag_count;
  const int n1 = g.n[0], n2 = g.n[1], n3 = (NDIM == 3) ? g.n[2] : 1;
  GlobView<T> ve[3], vb[3];
  GlobAcc<T> acc[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    ve[c] = GlobView<T>{f.e[c], n1, n2, n3, n1};
    vb[c] = GlobView<T>{bg.b[c], n1, n2, n3, n1};
    acc[c] = GlobAcc<T>{f.j[c], n1, n2, n3, n1};
  }
  for (unsigned long long i = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; i < cnt;
       i += (unsigned long long)gridDim.x * blockDim.x) {
    const int64_t q = bins.strag[i];
    int li[3];
    T fr[3];
#pragma unroll
    for (int d = 0; d < NDIM; ++d) {
      li[d] = cell_split(p.x[d][q] * g.inv_dx[d], fr[d]);
    }
    advance_particle<T, NDIM, -1, GAIN>(ve, vb, acc, p, q, li, fr, li, g, a, bins.err);
  }
}

// Few particles: a warp each, straight from global memory.  The lanes copy the
// particle's 4^NDIM nodes of E and the time-centred B into shared memory, lane 0
// advances it from there and deposits into global memory.  No windows, no bins: a
// tile's window costs the same for one particle as for hundreds.
template <typename T, int NDIM, bool GAIN>
__global__ void __launch_bounds__(128) sparse_kernel(FieldPtrs<T> f, BbarPtrs<T> bg, PartPtrs p,
                                                     GridArgs g, PartArgs a, unsigned* err) {
  constexpr int NODES = NDIM == 3 ? 64 : 16;
  __shared__ T sm[4][6 * NODES];
  const int lane = threadIdx.x & 31;
  T* buf = sm[threadIdx.x >> 5];
  const int n1 = g.n[0], n2 = g.n[1], n3 = NDIM == 3 ? g.n[2] : 1;
  for (int64_t q = blockIdx.x * 4ll + (threadIdx.x >> 5); q < a.np; q += gridDim.x * 4ll) {
    int gc[3] = {0, 0, 0};
    T fr[3];
#pragma unroll
    for (int d = 0; d < NDIM; ++d) {
      gc[d] = cell_split(p.x[d][q] * g.inv_dx[d], fr[d]);
    }
    const int o3 = NDIM == 3 ? gc[2] - 1 : 0;
    for (int m = lane; m < NODES; m += 32) {
      const int64_t r = ((int64_t)wrap_index(o3 + (m >> 4), n3) * n2 + wrap_index(gc[1] - 1 + ((m >> 2) & 3), n2)) *
                            n1 + wrap_index(gc[0] - 1 + (m & 3), n1);
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        buf[c * NODES + m] = f.e[c][r];
        buf[(3 + c) * NODES + m] = bg.b[c][r];
      }
    }
    __syncwarp();
    if (lane == 0) {
      SmemView<T> ve[3], vb[3];
      OffsetAcc<T> acc[3];
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        ve[c] = SmemView<T>{buf + c * NODES, 4, 16, 0};
        vb[c] = SmemView<T>{buf + (3 + c) * NODES, 4, 16, 0};
        acc[c] = OffsetAcc<T>{GlobAcc<T>{f.j[c], n1, n2, n3, n1}, gc[0] - 1, gc[1] - 1, o3};
      }
      const int li[3] = {1, 1, NDIM == 3 ? 1 : 0};
      advance_particle<T, NDIM, -1, GAIN>(ve, vb, acc, p, q, li, fr, gc, g, a, err);
    }
    __syncwarp();
  }
}

}  // namespace

template <typename T, int NDIM>
void launch_sparse_nd(const FieldPtrs<T>& f, const BbarPtrs<T>& bg, const PartPtrs& p,
                      const GridArgs& g, const PartArgs& a, unsigned* err, cudaStream_t st) {
  const unsigned nb = (unsigned)((a.np + 3) / 4);
  if (p.wl) sparse_kernel<T, NDIM, true><<<nb, 128, 0, st>>>(f, bg, p, g, a, err);
  else sparse_kernel<T, NDIM, false><<<nb, 128, 0, st>>>(f, bg, p, g, a, err);
}

// one CTA per particle tile
template <typename T, class K>
cudaError_t launch_tiles(K kern, const FieldPtrs<T>& f, const BbarPtrs<T>& bg, const PartPtrs& p,
                         const GridArgs& g, const StencilArgs<T>& s, const PartTile& t,
                         const PartArgs& a, const BinBufs& b, size_t smem, int threads, cudaStream_t st) {
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  const unsigned extra = b.share.chunk > 0 ? (unsigned)b.share.most : 0u;
  kern<<<(unsigned)t.ntiles + extra, threads, smem, st>>>(f, bg, p, g, s, t, a, b);
  return cudaGetLastError();
}

// the tile kernel instance of the context's pusher
template <typename T, int NDIM, bool GAIN>
cudaError_t launch_pushers(const FieldPtrs<T>& f, const BbarPtrs<T>& bg, const PartPtrs& p,
                           const GridArgs& g, const StencilArgs<T>& s, const PartTile& t,
                           const PartArgs& a, const BinBufs& b, size_t smem, cudaStream_t st) {
  constexpr int threads = TileCfg<T, NDIM>::threads;
  if (a.pusher == PIC_ANALYTIC)
    return launch_tiles(particle_kernel<T, NDIM, PIC_ANALYTIC, GAIN>, f, bg, p, g, s, t, a, b, smem,
                        threads, st);
  if (a.pusher == PIC_HC)
    return launch_tiles(particle_kernel<T, NDIM, PIC_HC, GAIN>, f, bg, p, g, s, t, a, b, smem,
                        threads, st);
  return launch_tiles(particle_kernel<T, NDIM, PIC_BORIS, GAIN>, f, bg, p, g, s, t, a, b, smem,
                      threads, st);
}

template <typename T>
cudaError_t launch_particle_step(const FieldPtrs<T>& f, const BbarPtrs<T>& bg, const PartPtrs& p,
                                 const GridArgs& g, const StencilArgs<T>& s, const PartTile& t,
                                 const PartArgs& a, const BinBufs& b, cudaStream_t st) {
  const size_t smem = particle_smem_bytes(g.ndim, sizeof(T), t, s.M);
  cudaError_t e;
  if constexpr (std::is_same<T, double>::value) {
    if (particles_sparse(true, a.np)) {
      if (g.ndim == 3) launch_sparse_nd<T, 3>(f, bg, p, g, a, b.err, st);
      else launch_sparse_nd<T, 2>(f, bg, p, g, a, b.err, st);
      return cudaGetLastError();
    }
  }
  if (g.ndim == 3)
    e = p.wl ? launch_pushers<T, 3, true>(f, bg, p, g, s, t, a, b, smem, st)
             : launch_pushers<T, 3, false>(f, bg, p, g, s, t, a, b, smem, st);
  else
    e = p.wl ? launch_pushers<T, 2, true>(f, bg, p, g, s, t, a, b, smem, st)
             : launch_pushers<T, 2, false>(f, bg, p, g, s, t, a, b, smem, st);
  return e;
}

template <typename T, int NDIM>
void launch_straggler_nd(const FieldPtrs<T>& f, const BbarPtrs<T>& bg, const PartPtrs& p,
                         const GridArgs& g, const StencilArgs<T>& s, const PartArgs& a,
                         const BinBufs& b, cudaStream_t st) {
  if (p.wl) straggler_kernel<T, NDIM, true><<<152, 128, 0, st>>>(f, bg, p, g, s, a, b);
  else straggler_kernel<T, NDIM, false><<<152, 128, 0, st>>>(f, bg, p, g, s, a, b);
}

template <typename T>
cudaError_t launch_straggler_step(const FieldPtrs<T>& f, const BbarPtrs<T>& bg, const PartPtrs& p,
                                  const GridArgs& g, const StencilArgs<T>& s, const PartArgs& a,
                                  const BinBufs& b, int64_t max_count, cudaStream_t st) {
  (void)max_count;
  if (g.ndim == 3) launch_straggler_nd<T, 3>(f, bg, p, g, s, a, b, st);
  else launch_straggler_nd<T, 2>(f, bg, p, g, s, a, b, st);
  return cudaGetLastError();
}

#define PIC_PARTICLE_INST(T)                                                                  \
  template cudaError_t launch_particle_step<T>(const FieldPtrs<T>&, const BbarPtrs<T>&,       \
                                               const PartPtrs&, const GridArgs&,              \
                                               const StencilArgs<T>&, const PartTile&,        \
                                               const PartArgs&, const BinBufs&, cudaStream_t); \
  template cudaError_t launch_straggler_step<T>(const FieldPtrs<T>&, const BbarPtrs<T>&,       \
                                                const PartPtrs&, const GridArgs&,              \
                                                const StencilArgs<T>&, const PartArgs&,        \
                                                const BinBufs&, int64_t, cudaStream_t);

}  // namespace pic
