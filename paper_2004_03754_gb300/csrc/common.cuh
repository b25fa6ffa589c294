// common.cuh -- shared device/host definitions of libpic (GB300, sm_103a).
//
// Layout of a context in HBM (all arrays separate allocations, 256-byte aligned):
//   fields   E1 E2 E3 B1 B2 B3 J1 J2 J3   n1*n2*n3 values of T (double or float), x1 fastest
//   particles x1 x2 [x3] u1 u2 u3 w (double) + id (int64), two copies (ping-pong for re-binning)
//   bins     per-tile counts and starts (int64), per-particle tile key and slot (int32)
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "march_layout.cuh"
#include "pic.h"
#include "push_const.h"

namespace pic {

template <typename T>
struct FieldPtrs {
  T* e[3];
  T* b[3];  // B^{n-1/2}
  T* j[3];
};

// time-centred B^n arrays (formed once per step before the particles)
template <typename T>
struct BbarPtrs {
  T* b[3];
};

struct PartPtrs {
  double* x[3];
  double* u[3];
  double* w;
  int64_t* id;
  // energy-gain integrals of Sec. 4.2 per particle (W_LWFA, W_DLA); null when
  // the diagnostic is off
  double* wl;
  double* wd;
};

struct GridArgs {
  int ndim;
  int n[3];
  double dx[3];
  double inv_dx[3];
  double len[3];
  double dx_dt[3];   // dx_d / dt (Esirkepov running-sum factor)
  double dt;
  int64_t ncell;
};

// Stencil coefficients pre-multiplied by dt/dx1 (full step) in the field's type.
template <typename T>
struct StencilArgs {
  int M;
  T kE[PIC_MAX_M];   // dt * C^E_j / dx1
  T kB[PIC_MAX_M];   // dt * C^B_j / dx1
  T y2, y3;          // dt/dx2, dt/dx3 (Yee)
};

// Device error word bits (latched, read back by pic_sync / pic_read_*).
enum : unsigned {
  ERRBIT_MOVE = 1u,          // a particle moved a full cell or more in one step
  ERRBIT_ANALYTIC = 2u,      // the analytic pusher's proper-time iteration did not converge
  ERRBIT_NONFINITE = 4u,     // a non-finite momentum or position was produced
  ERRBIT_POSITION = 8u,      // a loaded particle position lies outside the box
  ERRBIT_TIMEOUT = 16u,      // a bounded wait (grid barrier, staging copy) ran out
};

__host__ __device__ inline int wrap_index(int i, int n) {
  int r = i % n;
  return r < 0 ? r + n : r;
}

// ---------------------------------------------------------------------------
// Launch helpers implemented in fields.cu / particles.cu (host side).
// ---------------------------------------------------------------------------
// Field tile shape and CTA size (threads 0 = 256); staging 0 = asynchronous bulk
// copies where the grid allows them (persistent kernels), 1 = synchronous loads
// only.  2D grids with bulk copies stream rows per warp instead: strips of sw x1
// columns and `rows` rows per work item, `warps` per CTA, a ring of `stages` rows.
struct FieldTile {
  int t[3];
  int threads;
  int staging;
  int sw, rows, warps, stages;
};

// Reads E^n, B^{n-1/2}, J from f; writes E^{n+1}, B^{n+1/2} into out.e / out.b.
// A staging wait that runs out latches ERRBIT_TIMEOUT in *err.
template <typename T>
cudaError_t launch_field_step(const FieldPtrs<T>& f, const FieldPtrs<T>& out, const GridArgs& g,
                              const StencilArgs<T>& s, const FieldTile& tile, unsigned* err,
                              cudaStream_t st);

// The field step as two passes (field_halves.cu): Faraday of f into out.b -- with
// bg (nullable) also the time-centred B into bg, zeros into f.j and into
// *strag_count -- and Ampere of f.e and out.b into out.e with the current f.j (null
// pointers: none).  Every array starts on a 16-byte boundary (the rows are loaded and
// stored 16 bytes at a time from there); cudaErrorInvalidValue otherwise.
template <typename T>
cudaError_t launch_faraday(const FieldPtrs<T>& f, const FieldPtrs<T>& out, const BbarPtrs<T>* bg,
                           const GridArgs& g, const StencilArgs<T>& s,
                           unsigned long long* strag_count, cudaStream_t st);
template <typename T>
cudaError_t launch_ampere(const FieldPtrs<T>& f, const FieldPtrs<T>& out, const GridArgs& g,
                          const StencilArgs<T>& s, cudaStream_t st);

// Field states E1 E2 E3 B1 B2 B3 of ncell values each, one after another in one
// allocation: every component starts on a 256-byte boundary, also where ncell is odd.
template <typename T>
struct FieldStates {
  T* base;
  int64_t pitch;
  static int64_t pitch_of(int64_t ncell) { return (ncell + 31) / 32 * 32; }
  T* at(int64_t state, int comp) const { return base + (state * 6 + comp) * pitch; }
};

template <typename T>
cudaError_t launch_bbar(const FieldPtrs<T>& f, const GridArgs& g, const StencilArgs<T>& s,
                        double* out, int comp, cudaStream_t st);

// path: 0 automatic, 1 whole rows in place, 2 row segments, 3 global memory
template <typename T>
cudaError_t launch_correct_j1(T* j1, T* tmp, const GridArgs& g, const T* taps, int lo, int count,
                              int path, cudaStream_t st);

template <typename T>
cudaError_t launch_convert_in(T* dst, const double* src, int64_t n, cudaStream_t st);
template <typename T>
cudaError_t launch_convert_out(double* dst, const T* src, int64_t n, cudaStream_t st);

template <typename T>
cudaError_t launch_laser_expand(const FieldPtrs<T>& f, const GridArgs& g, const double* eprof,
                                const double* bprof, double w0, double x2c, double x3c,
                                cudaStream_t st);

// Windows of a particle tile along axis d: `t` cells with `lo` nodes below and `hi`
// above; along x1 widened so that it starts and ends on multiples of A columns (pad:
// the columns added below).  E and B are staged over a particle's gather (one node
// below its cell, two above, plus the drift g - 3), the current is accumulated over
// its deposit (two below, three above).
struct WindowAxis {
  int lo, w;   // nodes below the tile, with the padding; width
};
__host__ __device__ inline WindowAxis window_axis(int d, int t, int lo, int hi, int A) {
  const int l = d == 0 ? (lo + A - 1) / A * A : lo;
  const int w = l + t + hi;
  return WindowAxis{l, d == 0 ? (w + A - 1) / A * A : w};
}
__host__ __device__ inline WindowAxis eb_window(int d, int t, int g) {
  return window_axis(d, t, g - 2, g - 1, 2);
}
__host__ __device__ inline WindowAxis j_window(int d, int t, int g, int V) {
  return window_axis(d, t, g - 1, g, V);
}

struct PartTile {
  int t[3];      // tile size in cells
  int g[3];      // guard cells of the staged window
  int nt[3];     // tiles per axis
  int64_t ntiles;
};

struct PartArgs {
  double qm;
  int pusher;
  int64_t np;
  PushConst push{};   // of the push next to FP32 fields (zeros: its FP64 form)
};
inline PartArgs part_args(double qm, double dt, int pusher, int64_t np) {
  return PartArgs{qm, pusher, np, push_const(qm, dt)};
}

// Few enough particles to take a warp each instead of tiles (FP64 fields; FP32 currents
// keep their windows, whose sums are rounded once): 512x128 cells with one electron, 20
// steps 0.889 -> 0.731 ms; the adjoint of 64 electrons, 1024x256, 74.6 -> 67.8 ms.  256
// warps, two per SM, end before a tile has staged its window.  Their currents meet in
// FP64 atomics on the grid, in any order: electrons that share nodes leave last-bit
// differences from run to run, as electrons of neighbouring tiles always did; within
// one tile's integer window there were none.
__host__ __device__ inline bool particles_sparse(bool f64, int64_t np) { return f64 && np <= 256; }

// Crowded tiles: a tile of more than `line` particles is shared by several CTAs of up to
// `chunk` each (its time would otherwise bound the whole step: an electron sheet in front
// of a strong pulse put 12 times the mean into one tile).  Each share runs in a current
// window of its own, on the scales of the whole tile; the windows' integers are added up
// in `scratch` and the last CTA to arrive flushes the sum, so the current does not depend
// on the split.  The list is made with the tile counts of each re-binning.
// A share is a quarter of what an SM gets of all particles: four tiles of that size are
// resident on an SM at least in part, so a smaller one does not stand out; and never
// under 1024 particles, where staging the windows again costs what the split gives.
// 2D compensated, 1.5 M electrons behind a pulse of a0 = 100, particle kernel per
// step: largest tile 3.2 k particles 0.75 -> 0.79 ms, 9.4 k 1.18 -> 0.89, 12 k
// 1.39 -> 0.94; with no crowded tile 1.58 -> 1.56 (29.4 M electrons, mixed) and
// 2.16 -> 2.16 ms (6.3 M, FP64).
// The line (share_line) is a share, but at least half more than the mean of the occupied
// tiles: where few tiles hold a uniform plasma, every one of them is larger than a share
// and splitting them all only adds windows (1024x256 in 512 tiles, 4 electrons per cell,
// eight steps: mixed 1.49 -> 1.05 ms, compensated 3.28 -> 2.61, FP64 5.19 -> 4.62 with the
// tiles whole; 48^3, 8 per cell, four steps 1.66 -> 1.33).  Past what an SM gets of all
// particles a tile is always split: there are fewer tiles than SMs, or one is a sheet
// (256x128 in 64 tiles, 8 per cell, 0.53 ms split and 0.61 whole).
__host__ __device__ inline int64_t share_line(int64_t particles, int64_t occupied, int64_t chunk) {
  const int64_t half_more = occupied > 0 ? (3 * particles + 2 * occupied - 1) / (2 * occupied) : 0;
  const int64_t sm = (particles + 151) / 152;
  const int64_t line = half_more < sm ? half_more : sm;
  return line > chunk ? line : chunk;
}
struct TileShare {
  int tile, part, slot;
};
struct TileShares {
  int64_t chunk;      // particles per share; 0: no list
  int64_t ntiles;
  int* counts;        // [0] shares beyond the first of their tiles, [1] crowded tiles,
                      // [2] occupied tiles while they are counted
  int64_t* line;      // most particles of a tile that is not shared
  TileShare* list;    // the former
  int* slot;          // ntiles: index of a crowded tile
  int* scratch;       // per crowded tile: arrival count (16 bytes), then the window's integers
  int words;          // ints per crowded tile
  int most;           // upper bound of both counts: particles / chunk
  int cap;            // the most that list and scratch hold
};

struct BinBufs {
  int64_t* count;     // ntiles + 1 (the last bin holds particles being dropped)
  int64_t* start;     // ntiles + 2
  int* key;           // np
  int* slot;          // np
  int64_t* strag;     // np (indices of particles that take the global path)
  unsigned long long* strag_count;
  unsigned* err;
  int64_t* part;      // bin_scan_chunks(ntiles + 1): chunk sums of the scan
  TileShares share{};
};

// chunks of the tile-count scan for n counts (the size of BinBufs::part)
int64_t bin_scan_chunks(int64_t n);


// kill_col >= 0: particles in x1 column kill_col are binned past the last tile
// (dropped by the caller); the count array holds ntiles + 1 bins
cudaError_t launch_bin_count(const PartPtrs& p, const GridArgs& g, const PartTile& t,
                             const BinBufs& b, int64_t np, cudaStream_t st, int kill_col = -1);
cudaError_t launch_bin_scan(const BinBufs& b, int64_t ntiles, cudaStream_t st);
cudaError_t launch_bin_scatter(const PartPtrs& src, const PartPtrs& dst, const GridArgs& g,
                               const BinBufs& b, int64_t np, cudaStream_t st);

template <typename T>
cudaError_t launch_particle_step(const FieldPtrs<T>& f, const BbarPtrs<T>& bg, const PartPtrs& p,
                                 const GridArgs& g, const StencilArgs<T>& s, const PartTile& t,
                                 const PartArgs& a, const BinBufs& b, cudaStream_t st);

template <typename T>
cudaError_t launch_straggler_step(const FieldPtrs<T>& f, const BbarPtrs<T>& bg, const PartPtrs& p,
                                  const GridArgs& g, const StencilArgs<T>& s, const PartArgs& a,
                                  const BinBufs& b, int64_t max_count, cudaStream_t st);

// copy particles back in their original order; positions on the box edge are
// mapped into [0, len)
cudaError_t launch_unpermute(const PartPtrs& p, int ndim, int64_t np, double* x, double* u,
                             double* w, const double* len, cudaStream_t st);

// After particles were dropped: the kept ones (positions 0..kept-1, ids among
// 0..np_old-1) get ids 0..kept-1 in their old id order.  tmp: 2 np_old + 1 +
// bin_scan_chunks(np_old) values.
cudaError_t launch_renumber(int64_t* id, int64_t np_old, int64_t kept, int64_t* tmp,
                            cudaStream_t st);

// W_LWFA then W_DLA of every particle, in load order, into out (2 np values)
cudaError_t launch_unpermute_gain(const PartPtrs& p, int64_t np, double* out, cudaStream_t st);

// ints of one tile's current window
int particle_window_ints(int ndim, bool f64, size_t tsize, const PartTile& t);

size_t particle_smem_bytes(int ndim, size_t tsize, const PartTile& t, int M);

}  // namespace pic
