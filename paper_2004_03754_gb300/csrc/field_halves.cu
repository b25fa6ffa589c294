// field_halves.cu -- the field step as two row passes with the particles between:
//   Faraday  B^{n+1/2} = B^{n-1/2} - dt d_E x E^n     (Eq. (1), App. B Eq. (B.1))
//            with the time-centred B^n = B^{n-1/2} - (dt/2) d_E x E^n (Eq. (7)) from
//            the same curl, and the current cleared for the deposit;
//   Ampere   E^{n+1} = E^n + dt (d_B x B^{n+1/2} - J)  (Eq. (1), App. B Eq. (B.2)).
//
// Why two passes: a step with particles needs the time-centred B before the push
// anyway.  Formed by a pass of its own it took the curl of E twice (of the six
// wide x1 stencils per cell of an FP64 step two were that pass's), and the fused
// Faraday + Ampere kernels recompute B over the x1 reach of the Ampere stencil and
// one row per item on top.  Here each stencil is evaluated once per cell.  HBM
// traffic is the same: 12 + 12 values per cell (15 with the cleared current)
// against 9 + 15 (and the current's memset).
//
// Split of the work: one CTA per x1 segment of one row, V = 16/sizeof(T) outputs
// per thread; the two rows an x1 stencil runs over are staged in shared memory
// with its reach.  A segment's groups start on 16-byte boundaries of the array,
// whatever the row length (a row of n1 % V != 0 starts at a different offset each
// time, so its first and last group are partial), hence 16-byte loads and stores
// everywhere but at the row ends and in the x2/x3 neighbours of such rows.
// The operations on each value and their order are the fused kernels' (the same bits).
//
// Bound: FP64 and compensated fields by the FP64 and FP32 pipes (FP64 4096x1024 in
// vacuum 1174 us per step for 144 FP64 operations per cell, 82 % of the pipe; fused
// 1457), FP32 by HBM or, on small grids, by latency.  Per step with particles,
// against fused kernel + time-centred B pass + memsets: FP64 512x128 with one electron
// 128 -> 44 us (all kernels), FP64 2048x512 583 -> 309, compensated 282 -> 64 us, FP32
// 1501x389 (rows off 16 bytes, CTA tiles before) 72 -> 15 us.
#include <algorithm>
#include <initializer_list>

#include "common.cuh"
#include "field_tile.cuh"

namespace pic {

namespace {

// V values at columns c .. c+V-1 of the row at p (column 0), one 16-byte load when
// the group is whole and aligned; columns outside [0, n1) give zero
template <typename T>
__device__ __forceinline__ void ld_group(T* r, const T* p, int c, bool whole, int n1) {
  constexpr int V = VecOf<T>::V;
  const T* q = p + c;
  if (whole && (reinterpret_cast<uintptr_t>(q) & 15u) == 0) {
    vld_global<false>(r, q);
  } else {
#pragma unroll
    for (int v = 0; v < V; ++v) r[v] = (unsigned)(c + v) < (unsigned)n1 ? q[v] : (T)0;
  }
}
template <typename T>
__device__ __forceinline__ void st_group(T* p, const T* r, int c, bool whole, int n1) {
  constexpr int V = VecOf<T>::V;
  T* q = p + c;
  if (whole) {
    vst(q, r);
  } else {
#pragma unroll
    for (int v = 0; v < V; ++v)
      if ((unsigned)(c + v) < (unsigned)n1) q[v] = r[v];
  }
}

// W values (a multiple of V) of two periodic rows from column c0 into shared
// memory; c0 lies on a 16-byte boundary of the rows' arrays
template <typename T>
__device__ __forceinline__ void stage_rows(T* d0, T* d1, const T* r0, const T* r1, int c0, int W,
                                           int n1) {
  constexpr int V = VecOf<T>::V;
  for (int l = threadIdx.x * V; l < W; l += blockDim.x * V) {
    const int c = c0 + l;
    T a[V], b[V];
    if (c >= 0 && c + V <= n1) {
      vld_global<false>(a, r0 + c);
      vld_global<false>(b, r1 + c);
    } else {
#pragma unroll
      for (int v = 0; v < V; ++v) {
        const int w = pwrap(c + v, n1);
        a[v] = r0[w];
        b[v] = r1[w];
      }
    }
    vst(d0 + l, a);
    vst(d1 + l, b);
  }
}

// the CTA's segment: row (j, k), base offset of the row, first column of the
// segment (on a 16-byte boundary) and of the thread's group
struct Segment {
  int j, k, c0, c;
  int64_t r0;
};
template <typename T>
__device__ __forceinline__ Segment segment(int n1, int n2, int nseg) {
  constexpr int V = VecOf<T>::V;
  Segment s;
  const int seg = blockIdx.x % nseg;
  const int64_t row = blockIdx.x / nseg;
  s.j = (int)(row % n2);
  s.k = (int)(row / n2);
  s.r0 = row * n1;
  s.c0 = seg * (int)blockDim.x * V - (int)(s.r0 % V);
  s.c = s.c0 + (int)threadIdx.x * V;
  return s;
}

// BBAR: also the time-centred B into bg and zeros into f.j
template <typename T, int NDIM, int MT, bool BBAR>
__global__ void __launch_bounds__(256) faraday_rows_kernel(FieldPtrs<T> f, FieldPtrs<T> o,
                                                           BbarPtrs<T> bg, GridArgs g,
                                                           StencilArgs<T> s, int nseg,
                                                           unsigned long long* strag_count) {
  constexpr int V = VecOf<T>::V;
  constexpr Reach RC(MT, V);
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int n1 = g.n[0], n2 = g.n[1], n3 = (NDIM == 3) ? g.n[2] : 1;
  const Segment S = segment<T>(n1, n2, nseg);
  if (BBAR && blockIdx.x == 0 && threadIdx.x == 0) *strag_count = 0ull;
  const int WL = (int)blockDim.x * V - V + RC.LE;
  T* s2 = reinterpret_cast<T*>(smem_raw);   // E2 row from column c0 - DE
  T* s3 = s2 + ceil_to(WL, V);              // E3 row
  const bool any = S.c + V > 0 && S.c < n1, whole = S.c >= 0 && S.c + V <= n1;
  const int64_t rj = ((int64_t)S.k * n2 + (S.j + 1 == n2 ? 0 : S.j + 1)) * n1;
  const int64_t rk = NDIM == 3 ? ((int64_t)(S.k + 1 == n3 ? 0 : S.k + 1) * n2 + S.j) * n1 : 0;
  T e1[V], e1j[V], e3j[V], e1k[V], e2k[V], b1[V], b2[V], b3[V];
  if (any) {   // in flight while the rows are staged
    ld_group(e1, f.e[0] + S.r0, S.c, whole, n1);
    ld_group(e1j, f.e[0] + rj, S.c, whole, n1);
    ld_group(e3j, f.e[2] + rj, S.c, whole, n1);
    if (NDIM == 3) {
      ld_group(e1k, f.e[0] + rk, S.c, whole, n1);
      ld_group(e2k, f.e[1] + rk, S.c, whole, n1);
    }
    ld_group(b1, f.b[0] + S.r0, S.c, whole, n1);
    ld_group(b2, f.b[1] + S.r0, S.c, whole, n1);
    ld_group(b3, f.b[2] + S.r0, S.c, whole, n1);
  }
  stage_rows(s2, s3, f.e[1] + S.r0, f.e[2] + S.r0, S.c0 - RC.DE, WL, n1);
  __syncthreads();
  if (!any) return;
  const int col = threadIdx.x * V;
  T dE3[V], dE2[V], e2[V], e3[V];
  x1_stencil<T, V, MT, RC.DE, RC.LE, 1>(dE3, s3 + col, s.kE);
  x1_stencil<T, V, MT, RC.DE, RC.LE, 1>(dE2, s2 + col, s.kE);
  vld(e2, s2 + col + RC.DE);
  vld(e3, s3 + col + RC.DE);
  T o1[V], o2[V], o3[V];
#pragma unroll
  for (int v = 0; v < V; ++v) {
    const T d2E3 = s.y2 * (e3j[v] - e3[v]);
    const T d2E1 = s.y2 * (e1j[v] - e1[v]);
    T d3E2 = 0, d3E1 = 0;
    if (NDIM == 3) {
      d3E2 = s.y3 * (e2k[v] - e2[v]);
      d3E1 = s.y3 * (e1k[v] - e1[v]);
    }
    o1[v] = b1[v] - (T)0.5 * (d2E3 - d3E2);
    o2[v] = b2[v] - (T)0.5 * (d3E1 - dE3[v]);
    o3[v] = b3[v] - (T)0.5 * (dE2[v] - d2E1);
    b1[v] -= d2E3 - d3E2;   // B1 -= dt (d2 E3 - d3 E2)
    b2[v] -= d3E1 - dE3[v];
    b3[v] -= dE2[v] - d2E1;
  }
  st_group(o.b[0] + S.r0, b1, S.c, whole, n1);
  st_group(o.b[1] + S.r0, b2, S.c, whole, n1);
  st_group(o.b[2] + S.r0, b3, S.c, whole, n1);
  if constexpr (BBAR) {
    st_group(bg.b[0] + S.r0, o1, S.c, whole, n1);
    st_group(bg.b[1] + S.r0, o2, S.c, whole, n1);
    st_group(bg.b[2] + S.r0, o3, S.c, whole, n1);
    const T z[V] = {};
    st_group(f.j[0] + S.r0, z, S.c, whole, n1);
    st_group(f.j[1] + S.r0, z, S.c, whole, n1);
    st_group(f.j[2] + S.r0, z, S.c, whole, n1);
  }
}

// E^{n+1} into o.e from f.e, f.j and B^{n+1/2} in o.b
template <typename T, int NDIM, int MT>
__global__ void __launch_bounds__(256) ampere_rows_kernel(FieldPtrs<T> f, FieldPtrs<T> o,
                                                          GridArgs g, StencilArgs<T> s, int nseg) {
  constexpr int V = VecOf<T>::V;
  constexpr Reach RC(MT, V);
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int n1 = g.n[0], n2 = g.n[1], n3 = (NDIM == 3) ? g.n[2] : 1;
  const T dt = (T)g.dt;
  const Segment S = segment<T>(n1, n2, nseg);
  const int WL = (int)blockDim.x * V - V + RC.LB;
  T* s2 = reinterpret_cast<T*>(smem_raw);   // B2 row from column c0 - DB
  T* s3 = s2 + ceil_to(WL, V);              // B3 row
  const bool any = S.c + V > 0 && S.c < n1, whole = S.c >= 0 && S.c + V <= n1;
  const int64_t rj = ((int64_t)S.k * n2 + (S.j == 0 ? n2 - 1 : S.j - 1)) * n1;
  const int64_t rk = NDIM == 3 ? ((int64_t)(S.k == 0 ? n3 - 1 : S.k - 1) * n2 + S.j) * n1 : 0;
  T b1[V], b1m[V], b3m[V], b1k[V], b2k[V], e1[V], e2[V], e3[V], j1[V], j2[V], j3[V];
  if (any) {
    ld_group(b1, o.b[0] + S.r0, S.c, whole, n1);
    ld_group(b1m, o.b[0] + rj, S.c, whole, n1);
    ld_group(b3m, o.b[2] + rj, S.c, whole, n1);
    if (NDIM == 3) {
      ld_group(b1k, o.b[0] + rk, S.c, whole, n1);
      ld_group(b2k, o.b[1] + rk, S.c, whole, n1);
    }
    ld_group(e1, f.e[0] + S.r0, S.c, whole, n1);
    ld_group(e2, f.e[1] + S.r0, S.c, whole, n1);
    ld_group(e3, f.e[2] + S.r0, S.c, whole, n1);
    if (f.j[0]) {
      ld_group(j1, f.j[0] + S.r0, S.c, whole, n1);
      ld_group(j2, f.j[1] + S.r0, S.c, whole, n1);
      ld_group(j3, f.j[2] + S.r0, S.c, whole, n1);
    } else {
#pragma unroll
      for (int v = 0; v < V; ++v) j1[v] = j2[v] = j3[v] = (T)0;
    }
  }
  stage_rows(s2, s3, o.b[1] + S.r0, o.b[2] + S.r0, S.c0 - RC.DB, WL, n1);
  __syncthreads();
  if (!any) return;
  const int col = threadIdx.x * V;
  T dB3[V], dB2[V], b2[V], b3[V];
  x1_stencil<T, V, MT, RC.DB, RC.LB, 0>(dB3, s3 + col, s.kB);
  x1_stencil<T, V, MT, RC.DB, RC.LB, 0>(dB2, s2 + col, s.kB);
  vld(b2, s2 + col + RC.DB);
  vld(b3, s3 + col + RC.DB);
#pragma unroll
  for (int v = 0; v < V; ++v) {
    const T d2B3 = s.y2 * (b3[v] - b3m[v]);
    const T d2B1 = s.y2 * (b1[v] - b1m[v]);
    T d3B2 = 0, d3B1 = 0;
    if (NDIM == 3) {
      d3B2 = s.y3 * (b2[v] - b2k[v]);
      d3B1 = s.y3 * (b1[v] - b1k[v]);
    }
    e1[v] = e1[v] + ((d2B3 - d3B2) - dt * j1[v]);
    e2[v] = e2[v] + ((d3B1 - dB3[v]) - dt * j2[v]);
    e3[v] = e3[v] + ((dB2[v] - d2B1) - dt * j3[v]);
  }
  st_group(o.e[0] + S.r0, e1, S.c, whole, n1);
  st_group(o.e[1] + S.r0, e2, S.c, whole, n1);
  st_group(o.e[2] + S.r0, e3, S.c, whole, n1);
}

// threads per CTA: 256, halved while a row's groups would leave half of them idle or
// the grid has fewer than about eight CTAs per SM (small grids are spread thinner,
// down to one warp: the FP64 stencils of a row are bound by the SM's FP64 rate)
template <typename T>
int segment_threads(const GridArgs& g, int* nseg) {
  constexpr int V = VecOf<T>::V;
  const int64_t rows = g.ncell / g.n[0];
  const int groups = g.n[0] % V == 0 ? g.n[0] / V : (g.n[0] + 2 * V - 2) / V;   // with the offset
  int t = 256;
  while (t > 32 && (2 * groups <= t || (groups + t - 1) / t * rows < 152 * 8)) t /= 2;
  *nseg = (groups + t - 1) / t;
  return t;
}

template <typename T, int NDIM, int MT>
cudaError_t faraday_mt(const FieldPtrs<T>& f, const FieldPtrs<T>& o, const BbarPtrs<T>* bg,
                       const GridArgs& g, const StencilArgs<T>& s, unsigned long long* strag,
                       cudaStream_t st) {
  constexpr int V = VecOf<T>::V;
  constexpr Reach RC(MT, V);
  int nseg;
  const int t = segment_threads<T>(g, &nseg);
  const size_t smem = 2 * (size_t)ceil_to(t * V - V + RC.LE, V) * sizeof(T);
  const unsigned nb = (unsigned)(nseg * (g.ncell / g.n[0]));
  if (bg)
    faraday_rows_kernel<T, NDIM, MT, true><<<nb, t, smem, st>>>(f, o, *bg, g, s, nseg, strag);
  else
    faraday_rows_kernel<T, NDIM, MT, false><<<nb, t, smem, st>>>(f, o, BbarPtrs<T>{}, g, s, nseg, strag);
  return cudaGetLastError();
}
template <typename T, int NDIM, int MT>
cudaError_t ampere_mt(const FieldPtrs<T>& f, const FieldPtrs<T>& o, const GridArgs& g,
                      const StencilArgs<T>& s, cudaStream_t st) {
  constexpr int V = VecOf<T>::V;
  constexpr Reach RC(MT, V);
  int nseg;
  const int t = segment_threads<T>(g, &nseg);
  const size_t smem = 2 * (size_t)ceil_to(t * V - V + RC.LB, V) * sizeof(T);
  const unsigned nb = (unsigned)(nseg * (g.ncell / g.n[0]));
  ampere_rows_kernel<T, NDIM, MT><<<nb, t, smem, st>>>(f, o, g, s, nseg);
  return cudaGetLastError();
}

// every array that is given starts on a 16-byte boundary
template <typename T>
bool on_16(const FieldPtrs<T>& f, const FieldPtrs<T>& o, const BbarPtrs<T>* bg) {
  uintptr_t any = 0;
  for (int c = 0; c < 3; ++c) {
    for (const T* p : {f.e[c], f.b[c], f.j[c], o.e[c], o.b[c]}) any |= reinterpret_cast<uintptr_t>(p);
    if (bg) any |= reinterpret_cast<uintptr_t>(bg->b[c]);
  }
  return (any & 15u) == 0;
}

}  // namespace

template <typename T>
cudaError_t launch_faraday(const FieldPtrs<T>& f, const FieldPtrs<T>& o, const BbarPtrs<T>* bg,
                           const GridArgs& g, const StencilArgs<T>& s, unsigned long long* strag,
                           cudaStream_t st) {
  if (!on_16(f, o, bg)) return cudaErrorInvalidValue;
  const int mt = stencil_mt(s.M);
  if (g.ndim == 3)
    return mt == 8    ? faraday_mt<T, 3, 8>(f, o, bg, g, s, strag, st)
           : mt == 16 ? faraday_mt<T, 3, 16>(f, o, bg, g, s, strag, st)
                      : faraday_mt<T, 3, 32>(f, o, bg, g, s, strag, st);
  return mt == 8    ? faraday_mt<T, 2, 8>(f, o, bg, g, s, strag, st)
         : mt == 16 ? faraday_mt<T, 2, 16>(f, o, bg, g, s, strag, st)
                    : faraday_mt<T, 2, 32>(f, o, bg, g, s, strag, st);
}

template <typename T>
cudaError_t launch_ampere(const FieldPtrs<T>& f, const FieldPtrs<T>& o, const GridArgs& g,
                          const StencilArgs<T>& s, cudaStream_t st) {
  if (!on_16(f, o, static_cast<const BbarPtrs<T>*>(nullptr))) return cudaErrorInvalidValue;
  const int mt = stencil_mt(s.M);
  if (g.ndim == 3)
    return mt == 8    ? ampere_mt<T, 3, 8>(f, o, g, s, st)
           : mt == 16 ? ampere_mt<T, 3, 16>(f, o, g, s, st)
                      : ampere_mt<T, 3, 32>(f, o, g, s, st);
  return mt == 8    ? ampere_mt<T, 2, 8>(f, o, g, s, st)
         : mt == 16 ? ampere_mt<T, 2, 16>(f, o, g, s, st)
                    : ampere_mt<T, 2, 32>(f, o, g, s, st);
}

#define PIC_HALVES_INST(T)                                                                     \
  template cudaError_t launch_faraday<T>(const FieldPtrs<T>&, const FieldPtrs<T>&,             \
                                         const BbarPtrs<T>*, const GridArgs&,                  \
                                         const StencilArgs<T>&, unsigned long long*,           \
                                         cudaStream_t);                                        \
  template cudaError_t launch_ampere<T>(const FieldPtrs<T>&, const FieldPtrs<T>&,              \
                                        const GridArgs&, const StencilArgs<T>&, cudaStream_t);
PIC_HALVES_INST(double)
PIC_HALVES_INST(float)
PIC_HALVES_INST(dfl)
#undef PIC_HALVES_INST

}  // namespace pic
