// cl_internal.cuh -- types shared by the translation units of libcellmap.
//
// Data layout in device memory (one cl_list):
//   xs[n]        float4  cell-sorted particles: (x, y, z) FP32 relative to the
//                        CENTRE of the particle's own cell, w = original index
//                        (int bits). 2D sets z = 0.
//   cellc[n]     uint32  packed cell coordinates of each sorted particle:
//                        cx | cy << 10 | cz << 20 (at most 1023 cells per axis)
//   cell_start[ncells+1] prefix sum of the per-cell counts: particles of cell
//                        c occupy xs[cell_start[c] .. cell_start[c+1]). Cells
//                        are linearised x-fastest, c = cx + nx (cy + ny cz),
//                        so a row of cells along x is one contiguous range.
// The displacement from particle i (cell ci) to particle j in the neighbour
// cell reached by the integer offset o (wrapped periodically) is
//   r = (xs_j + S_o) - xs_i,   S_o = sum_k (o_k / n_k) H_k,
// because the centre of cell ci + o, unwrapped, is the centre of the wrapped
// cell plus the lattice translation. S_o depends on o only, so one FP32 shift
// per stencil entry serves every cell (Sec. 2.6 replicates ghost particles to
// the same end; this build stores no ghosts).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>

#include "cellmap.h"

namespace clk {

// Launch parameters worked out once per device (occupancy, opt-in shared
// memory, which cudaFuncSetAttribute sets for the current device only): one
// slot per device, 0 until known. Devices past the table are not cached.
constexpr int kCacheDevices = 64;
struct DevCache {
  std::atomic<int> v[kCacheDevices];
  int get(int dev) const { return dev >= 0 && dev < kCacheDevices ? v[dev].load(std::memory_order_relaxed) : 0; }
  void put(int dev, int x) {
    if (dev >= 0 && dev < kCacheDevices) v[dev].store(x, std::memory_order_relaxed);
  }
};

constexpr int kMaxOff = 768;      // stencil entries (9^3 = 729 plus margin)
constexpr int kMaxRows2 = 9;      // rows of a 2D stencil, and cells of a row (reach <= 4)
constexpr int kMaxAxis = 1023;    // cells per axis (10-bit packing)
constexpr int kMaxBins = 4096;    // histogram bins (shared-memory histogram)
// Windowed cells of kOctMin to kOctCap particles are ordered by the octant of
// their particles' local coordinates (sign of x, y, z), and within it by the
// octants of that, by the 3D half-shell sweep when it builds its work lists, so
// that consecutive particles form compact groups.
constexpr int kOctMin = 65;
constexpr int kOctCap = 2048;

// One neighbour-cell offset of the stencil.
struct Off {
  int dx, dy, dz;     // o_k mod n_k, in [0, n_k)
  float sx, sy, sz;   // Cartesian shift S_o (FP32 of an FP64 value)
};

// Box geometry after preparation (host and device copies).
struct Geo {
  int dim;
  int n[3];           // cells per axis (1 for unused axes)
  long long ncells;
  double h[9];        // lattice rows, 3x3 (2D padded with identity z)
  double hinv[9];     // H^-1, 3x3
  double m[9];        // M = H^-1 diag(n): t = x M is the position in cell units
  double w[3];        // distances between opposite faces
  float g[9];         // cell edge vectors G_k = H_k / n_k (rows), FP32
  int ortho;          // 1 when H is diagonal
  double rc;
  int lcell;
};

// Device-side error latch bits.
constexpr int kErrNonFinite = 1;

// Stand-in coordinates for a particle whose input position is not finite (and
// for the element past the last one in the shifted-pair arrays): far outside
// any box, unique per index and at least 1e12 apart from each other, finite,
// so that every distance test against them fails without producing NaN.
__device__ __forceinline__ float4 sentinel_pos(int i) {
  const float big = 1e15f, step = 1.0f / 1024.0f;
  return make_float4(big * (1.0f + (float)(i & 1023) * step), big * (1.0f + (float)((i >> 10) & 1023) * step),
                     big * (1.0f + (float)((i >> 20) & 1023) * step), 0.0f);
}

// Launch arguments of the sweep kernels (passed as one __grid_constant__ parameter).
struct SweepArgs {
  const float4* xs;
  const unsigned* cellc;
  const int* cell_start;
  int n;
  int nx, ny, nz;
  float rc2, irc, irc2;
  // Half-widths of one cell's Cartesian bounding box, padded by 1e-3 rc (3D
  // packed per-particle sweep: a neighbour cell whose box lies at least rc
  // from the particle is skipped); 0 turns the test off.
  float ex, ey, ez;
  // 2D: the stencil as rows of cells (row_sweep): row r covers the offsets
  // rows2[r].ox0 .. ox1 at oy, whose stencil entries are idx2[e0 ..]. nrow2 = 0
  // when not given.
  struct Row2 {
    signed char ox0, ox1, oy;
    unsigned char e0;
  };
  int nrow2;
  Row2 rows2[kMaxRows2];
  unsigned char idx2[kMaxRows2 * kMaxRows2];
  int noff;             // entries in off[]; off[0] is the own cell
  Off off[kMaxOff];
};

// Host helpers implemented in cl_geom.cu.
int prepare_geometry(const cl_box* box, Geo* geo);
// Builds the half-shell (half = 1) or full stencil; returns the entry count or a
// negative error.
int build_stencil(const Geo& geo, int half, Off* out, int cap);
// Both at once; opk_* (optional) receive each entry's unwrapped offset packed
// as bytes: (ox & 255) | (oy & 255) << 8 | (oz & 255) << 16.
int build_stencils(const Geo& geo, int cap, Off* half, int* opk_half, int* nhalf, Off* full, int* opk_full, int* nfull);
// Fills A's rows of cells from a 2D stencil of noff entries (opk as above);
// leaves nrow2 = 0 when the entries do not form such rows.
void fill_rows2(const int* opk, int noff, SweepArgs* A);
// Half-widths of one cell's Cartesian bounding box (sum over the cell edge
// vectors of |G_k,a| / 2 per axis a), each padded by 1e-3 rc.
void cell_halfwidths(const Geo& geo, float* e);

}  // namespace clk

namespace clk {

// Stream-ordered device memory of the library (cl_mem.cu): a pool per device
// that keeps at most kPoolKeep bytes of freed memory for later calls.
bool capturing(cudaStream_t s);  // work on s is being recorded into a graph
int mem_alloc(void** p, size_t bytes, cudaStream_t s);
void mem_free(void* p, cudaStream_t s);
constexpr unsigned long long kPoolKeep = 256ull << 20;
// After frees on s: freed memory beyond kPoolKeep goes back to the device now.
// Waits for s when the pool holds more than that.
void mem_settle(cudaStream_t s);
// Pieces of one block, 256-byte aligned: with base null only their total is
// counted.
struct Carver {
  char* base;
  size_t used = 0;
  template <class T>
  void take(T** p, size_t count) {
    *p = base ? reinterpret_cast<T*>(base + used) : nullptr;
    used += ((count ? count : 1) * sizeof(T) + 255) & ~(size_t)255;
  }
};

// Buffers of one binning pipeline (cl_build.cu).
struct BuildBufs {
  const double* pos;
  int n;
  int* slot;    // per original particle: position inside its cell
  float4* xl;   // per original particle: centred local coordinate, w = packed cell (cx | cy << 10 | cz << 20)
  int* counts;
  bool counts_zeroed = false;  // the caller has zeroed counts
  int* cell_start;
  int* tile_sum;
  int* meta;  // [0] error latch, [1] non-empty cells, [2] max occupancy
  float4* xs;
  unsigned* cellc;
};
int scan_tiles_for(long long ncells);
int launch_build(const Geo& g, const BuildBufs& b, cudaStream_t s);
// Orders the particles of the listed cells (ncells_listed of them, read on the
// device) with kOctMin..kOctCap particles by octant; slots follow.
// (hx, hy, hz: half-widths of a cell's bounding box).
int launch_octsort(const int* cells, const int* ncells_listed, const int* cell_start, float hx, float hy, float hz,
                   float4* xs, int* slot, cudaStream_t s);
// Prefix sum of the per-cell counts into cell_start; meta[1], meta[2] (zeroed
// by the caller): non-empty cells, largest count.
int launch_scan_cells(const int* counts, long long ncells, int* tile_sum, int* meta, int* cell_start, cudaStream_t s);
// Moves xl[i] (w = packed cell) to its place in cell order (w = i) and writes
// the packed cells along the sorted array.
int launch_cell_order(int n, int nx, int ny, long long ncells, const int* slot, const float4* xl,
                      const int* cell_start, float4* xs, unsigned* cellc, cudaStream_t s);
int launch_scan64(const int* counts, long long n, long long* tile_sum, long long* start, cudaStream_t s);

// Sweeps and reductions (cl_sweep.cu).
int sweep_partials_needed(int n);
int launch_count(const SweepArgs& A, int dim, unsigned long long* out, cudaStream_t s);
int launch_scalar(const SweepArgs& A, int dim, int kind, double* partials, double* sums, double* out,
                  cudaStream_t s);
int launch_hist(const SweepArgs& A, int dim, int nbins, float rmax, unsigned long long* hist, cudaStream_t s);
// The same three sweeps (3D) over the particles of the cells with flag != 0
// only (the cells a neighbourhood sweep left), adding to out / hist without
// zeroing them; the sum 1/r kind writes blocks_for(n) partials and no final
// reduction.
int launch_count_flagged(const SweepArgs& A, const unsigned char* flag, unsigned long long* out, cudaStream_t s);
int launch_suminvr_flagged(const SweepArgs& A, const unsigned char* flag, double* partials, cudaStream_t s);
int launch_hist_flagged(const SweepArgs& A, const unsigned char* flag, int nbins, float rmax,
                        unsigned long long* hist, cudaStream_t s);
int flagged_blocks(int n);
int launch_force(const SweepArgs& A, int dim, int mode, const double* hinv, float* forces, double* grad,
                 const double* gE, const double* pos, double* partials, double* sums, double* energy,
                 double* virial, double* gradbox, cudaStream_t s);
int launch_candidates(const SweepArgs& A, long long ncells, unsigned long long* out, cudaStream_t s);
// Sums per-CTA partials[nblocks][nv] and writes the caller's outputs. final_mode:
// 0 sum 1/r, 1 energy, 2 forward forces (energy + virial), 3 backward, 4 energy
// and backward (partials S6, X9, E).
int launch_scale(const double* g, const double* in, double* out, long long count, cudaStream_t s);
int finish_reduction(int final_mode, int dim, const double* hinv, int nblocks, int nv, const double* partials,
                     double* sums, double* scalar, double* virial, double* gradbox, const double* gE,
                     cudaStream_t s);

// Neighbourhood sweep of the 3D shifted-force energy (cl_hood.cu).
constexpr int kWorkWords = 16;
struct HoodArgs {
  int opk[2][kMaxOff];  // unwrapped stencil offsets (see build_stencil): [0] full, [1] half stencil
  // rows of the half stencil (entries 1..: runs of consecutive ox with one
  // (oy, oz)) as (ox0, ox1, oy, oz); nrows_half of them, 0 when more than 128
  signed char rows_half[128][4];
  int nrows_half;
  double g[9];        // cell edge vectors G_k = H_k / n_k (rows), FP64
  float gf[9];        // the same, FP32
  float rc;
  float hd;           // largest distance of a cell point from the cell centre
  float eps;          // rounding margin of the staging radius
  int rawcap;         // particles in the half neighbourhood up to which a cell takes the fast path
  int smallcap;       // particles of a cell and its half neighbourhood up to which one warp takes it
  int split;          // CTAs sharing a listed cell's home particles (home-major scalar sweeps)
  int ncells;
  int* work;          // [0], [1], [4], [5] work counters of the listed, small, whole and dense cells, [2..3] candidates
                      // (zeroed by the launcher); [6] list length, [7] dense cells, [8] small cells (at the end
                      // of list, backwards), [9] whole cells (at the end of dense, backwards; written by k_hood_list)
  int* list;          // cells the neighbourhood sweep takes (ncells capacity)
  unsigned long long* cand;  // candidate pairs evaluated (work[2..3] of the same buffer), zeroed by the launcher
  unsigned char* flag;       // per cell: 1 per-particle companion sweep, 2 dense-cell sweep
  int* dense;                // cells of the dense-cell sweep (ncells capacity)
  int* ndense;               // their number (work[7])
  float hrow[9];             // lattice rows H (FP32): lattice image T maps to the shift T.H
  float4* hforce;            // half-shell path: per sorted particle, accumulated force (n entries)
  const float4* xl;          // per original particle: local coordinate, w = packed cell (binning output)
  const int* slot;           // per original particle: position inside its cell
  int half;                  // 1 when the half-shell path is tried for this launch
  // scalar reductions of the staged half-shell sweep (launch_hood_scalar)
  unsigned long long* count;  // pair count, added to
  unsigned long long* hist;   // nbins counts of r in [0, rmax), added to
  int nbins;
  float rmax, hscale;         // hscale = nbins / rmax
  float hxlim;                // min(nbins, rc hscale): bin coordinate limit of counted pairs
  int hcopies, hstride;       // shared-memory copies of the histogram (a power of two) and their stride
};
int fill_hood_args(const Geo& geo, const int* opk_full, int noff_full, const int* opk_half, int noff_half,
                   HoodArgs* H);
size_t hood_smem_bytes();
// mode 0: energy, forces, virial; 1: backward; 2: energy (half shell, A = half
// stencil); 3: energy and the backward outputs.
// partials_cap: doubles available in partials (sweep_partials_needed).
// lists_half (host, may be null): 1 when the list buffers (list, dense, flag,
// work[6..9]) hold the half-shell work lists of the current cell list; they
// are then reused, and the flag is set after a half-shell launch and cleared
// by any other.
// Ahalf (modes 0, 1, 3; may be null): the half stencil, for the half-shell
// path, taken when both stencils fit the kernels' table (H.hforce must then
// hold n entries); the full-shell kernels take the launch otherwise.
bool half_path_applies(const SweepArgs& A, const SweepArgs* Ahalf, const HoodArgs& H, int mode);
int launch_hood(const SweepArgs& A, const SweepArgs* Ahalf, const HoodArgs& H, int* work, int mode, const double* hinv, float* forces,
                double* grad, const double* gE, const double* pos, double* partials, long long partials_cap,
                double* sums, double* energy, double* virial, double* gradbox, cudaStream_t s,
                int* lists_half = nullptr);

// Count (kind 0), sum 1/r (1), distance histogram (2) or shifted-force
// energy (3) over the half stencil (A = half stencil, 3D): the staged sweeps
// (home-major for the fast-path cells, the windowed half-shell sweep for the
// others), or, when the stencil does not fit the kernels' table, the staged
// sweep for the cells that fit it and the per-particle sweep for the rest
// (the energy then returns CL_ERR_UNSUPPORTED: launch_hood's mode 2 takes it).
// The outputs (count: 1 value, scalar_out: 1 value, hist: nbins values) are
// overwritten.
bool hood_half_fits(const SweepArgs& A);
int launch_hood_scalar(const SweepArgs& A, const HoodArgs& H, int* work, int kind, unsigned long long* count,
                       double* partials, long long partials_cap, double* sums, double* scalar_out, int nbins,
                       float rmax, unsigned long long* hist, cudaStream_t s, int* lists_half = nullptr);

// Two sets (cl_cross.cu). The query points of set B, binned on set A's grid.
struct Queries {
  const float4* q;        // coordinate relative to the cell centre, w = query index (int bits)
  const unsigned* cell;   // packed cell
  long long nb;
};
// Workspace of the query binning: the prepared arrays and, when the queries
// are sorted by cell (queries_sorted), the counting sort's.
struct QueryBufs {
  float4* q;        // nb
  unsigned* cell;   // nb
  float4* raw;      // nb, sorted only
  int* slot;        // nb, sorted only
  int* counts;      // ncells, sorted only
  int* start;       // ncells + 1, sorted only
  int* tiles;       // scan_tiles_for(ncells), sorted only
  int* meta;        // 4, sorted only
};
bool queries_sorted(long long n, long long nb, long long ncells);
int launch_query_bin(const SweepArgs& A, const Geo& g, const double* posb, long long nb, const QueryBufs& b, int* err,
                     Queries* out, cudaStream_t s);
// The sweeps (off: the full stencil in device memory). Count: per query (count
// may be null) and their sum (total may be null). Fill: segments of the list at
// start, each sorted by a; those longer than kMaxSegment are listed in longs
// for launch_sort_long. knn: per query the k nearest.
int launch_cross_count(const SweepArgs& A, const Off* off, const Queries& Q, int* count, unsigned long long* total,
                       cudaStream_t s);
int launch_cross_fill(const SweepArgs& A, const Off* off, const Queries& Q, const int* count, const long long* start,
                      int* pa, int* pb, float* pd, int* longs, int* nlong, cudaStream_t s);
int launch_cross_knn(const SweepArgs& A, const Off* off, const Queries& Q, int k, int* out_a, float* out_d,
                     cudaStream_t s);
// The k closest of nb per-query lists of k (each ascending, -1 past its end);
// part_d, part_id: topk_parts(nb, k) * k entries of workspace.
long long topk_parts(long long nb, int k);
int launch_topk_merge(const int* la, const float* ld, long long nb, int k, float* part_d, long long* part_id, int* oa,
                      int* ob, float* od, int* found, cudaStream_t s);

// Mapped functions over the list (cl_pairfns.cu). The list's internals, from
// cl_api.cu: hforce is free scratch of n float4 between sweeps, zero before
// and after every call that uses it.
struct ListParts {
  const SweepArgs* half;
  const SweepArgs* full;
  double* partials;
  double* sums;
  float4* hforce;  // null in 2D
  double rc;
};
void list_parts(const cl_list* cl, ListParts* p);

// Neighbour list (cl_pairs.cu). count[n] (int: one particle's pairs), start[n+1]
// (64-bit scan of count: the list may pass 2^31 pairs), tiles, meta:
// workspace; outputs pair_i/j/d of capacity entries.
constexpr int kMaxSegment = 1024;  // segments up to this length are sorted by one warp in shared memory
// Workspace and plan of the two passes, the same for both.
struct PairLists {
  float ball2;          // squared radius about a cell's centre that holds the cell's neighbours
  int cap;              // staged entries per cell (32..3072)
  double expect;        // particles expected in that ball
  bool images;          // the stencil reaches some cell twice: two images of a particle may be staged
  int* last;            // ncells: largest original index per cell
  unsigned char* flag;  // ncells: 1 for the cells of fcells
  int* fcells;          // ncells: cells whose neighbourhood passes cap
  int* mid;             // ncells: sparse grids' cells that take the general staging
  int* ctr;             // [0] long segments, [1] fcells, [2] mid: their numbers
  int* count;           // n
};
// Count pass of the pair list: per-cell staged sweep, then the per-particle
// sweep for the cells it flags. Writes everything L points to.
int launch_pairs_count(const SweepArgs& A, const Off* off, int dim, const PairLists& L, cudaStream_t s);
// Sorts each listed segment [start[a], start[a] + count[a]), a = longs[q], q <
// *nlong, of pj (carrying pd) by pj.
int launch_sort_long(const int* longs, const int* nlong, const int* count, const long long* start, int* pj, float* pd,
                     cudaStream_t s);
// Fill pass: the same two sweeps, each segment sorted by j and written.
// longs (n ints): workspace for segments longer than kMaxSegment.
int launch_pairs_fill(const SweepArgs& A, const Off* off, int dim, const PairLists& L, const long long* start, int* pi,
                      int* pj, float* pd, int* longs, cudaStream_t s);

}  // namespace clk
