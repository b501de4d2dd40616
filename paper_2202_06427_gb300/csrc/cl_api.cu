// cl_api.cu -- the extern "C" boundary (cellmap.h): handle lifecycle,
// argument checks, and dispatch of the binning, sweep and reduction kernels.
#include <algorithm>
#include <cmath>
#include <cstdlib>
#include <cstring>
#include <memory>
#include <new>

#include "cl_internal.cuh"

struct cl_list {
  clk::Geo geo;
  cl_box box;  // the box geo was prepared from
  int device;
  int n;
  const double* pos;
  long long ncells_alloc;  // cells the per-cell arrays have room for
  // device workspace: blocks of the library's pool, and the arrays in them
  void* block;        // per particle and fixed
  void* cell_block;   // per cell
  void* pair_block;   // neighbour list, on its first call
  int* slot;
  float4* xl;
  float4* xs;
  unsigned* cellc;
  int* counts;
  int* cell_start;
  unsigned char* hflag;  // per cell: 1 when a staged sweep (neighbourhood or pair list) leaves it to a per-particle sweep
  int* hlist;            // cells the neighbourhood sweep takes
  int* hdense;           // cells the dense-cell sweep takes
  int* tile_sum;
  int* meta;
  double* partials;
  double* sums;
  int* work;  // work counters of the persistent neighbourhood sweeps
  float4* hforce;  // per sorted particle: forces accumulated by the half-shell sweep (kept zero between launches)
  int last_half;   // the last 3D energy/force sweep took the half-shell path
  int lists_half;  // hlist / hdense / work[6..9] hold the half-shell work lists of the current cell list
  int replayed;    // a graph may bin into this list: its cell contents change without a call (kept_lists)
  int lists_none;
  unsigned long long* u64;
  // neighbour-list workspace, allocated on the first CL_RED_PAIRLIST call
  int* pl_count;
  long long* pl_start;  // 64-bit: a list may pass 2^31 pairs
  long long* pl_tiles;
  int* pl_meta;
  int* pl_long;  // particles whose segments are sorted by the long-segment pass
  // device copies of the stencils (for sweeps compiled outside the library)
  clk::Off* d_off_half;
  clk::Off* d_off_full;
  // stencils (host copies of the sweep arguments)
  clk::SweepArgs* half;
  clk::SweepArgs* full;
  clk::HoodArgs* hood;  // 3D neighbourhood sweep arguments
  size_t bytes;
};

namespace {

// The list's per-particle and fixed-size arrays in one block: with base null
// their size. Those from `zero_from` on (zero_bytes) start as zeros.
size_t carve_list(cl_list* c, char* base, int dim, char** zero_from, size_t* zero_bytes) {
  clk::Carver v{base};
  const size_t n = (size_t)c->n;
  v.take(&c->slot, n);
  v.take(&c->xl, n);
  v.take(&c->xs, n);
  v.take(&c->cellc, n);
  v.take(&c->partials, (size_t)clk::sweep_partials_needed(c->n));
  v.take(&c->work, clk::kWorkWords);  // see HoodArgs
  v.take(&c->u64, 8);
  v.take(&c->d_off_half, 2 * (size_t)clk::kMaxOff);  // both stencils, one after the other
  const size_t at = v.used;
  v.take(&c->meta, 4);
  v.take(&c->sums, 32);  // [31]: the final reduction's completion counter, zero between launches
  if (dim == 3) v.take(&c->hforce, n);
  *zero_from = base + at;
  *zero_bytes = v.used - at;
  return v.used;
}

struct Cells {
  int *counts, *cell_start, *tile_sum, *hlist, *hdense;
  unsigned char* hflag;
};

size_t carve_cells(Cells* p, char* base, long long ncells) {
  clk::Carver v{base};
  v.take(&p->counts, (size_t)ncells);
  v.take(&p->cell_start, (size_t)ncells + 1);
  v.take(&p->tile_sum, (size_t)clk::scan_tiles_for(ncells));
  v.take(&p->hlist, (size_t)ncells);
  v.take(&p->hdense, (size_t)ncells);
  v.take(&p->hflag, (size_t)ncells);
  return v.used;
}

// Gives the list's memory back; no work on it may be in flight.
void free_all(cl_list* c) {
  clk::mem_free(c->block, nullptr);
  clk::mem_free(c->cell_block, nullptr);
  clk::mem_free(c->pair_block, nullptr);
  delete c->half;
  delete c->full;
  delete c->hood;
}

// Makes block (of carve_cells' size for ncells cells) the list's per-cell arrays.
// The old block may still be in use on another stream, so it is given back after
// a device synchronisation.
void adopt_cells(cl_list* c, void* block, long long ncells, cudaStream_t s) {
  if (c->cell_block) {
    Cells old;
    c->bytes -= carve_cells(&old, nullptr, c->ncells_alloc);
    if (!clk::capturing(s)) cudaDeviceSynchronize();
    clk::mem_free(c->cell_block, s);  // (under capture cudaFree, which waits itself)
    clk::mem_settle(s);
  }
  Cells p;
  c->bytes += carve_cells(&p, (char*)block, ncells);
  c->cell_block = block;
  c->counts = p.counts;
  c->cell_start = p.cell_start;
  c->tile_sum = p.tile_sum;
  c->hlist = p.hlist;
  c->hdense = p.hdense;
  c->hflag = p.hflag;
  c->ncells_alloc = ncells;
}

// Partials (doubles) available to the neighbourhood sweep and its per-particle companion.
long long hood_cap(const cl_list* c) { return clk::sweep_partials_needed(c->n); }

// Count, sum 1/r and the histogram take the staged neighbourhood sweep when
// the cells hold enough particles on average to pay for staging the half
// neighbourhood once per cell (measured: 23 per cell on the 1M lattice runs
// the count in 0.57 ms staged against 0.75 ms per particle), else one thread
// per particle over the stencil.
constexpr double kStagedMinOccupancy = 16.0;
bool scalar_staged(const cl_list* c) {
  return c->geo.dim == 3 && c->n > 0 && (double)c->n >= kStagedMinOccupancy * (double)c->geo.ncells;
}

// 2D sweeps go by rows of cells (row_sweep) up to this mean occupancy, above it
// cell by cell: rows keep a warp's lanes together where cells hold a few
// particles, but read each candidate's cell as well. Rows against cells, count
// and forces at two cells per cutoff: 400,000 particles 0.93 and 0.85 at one per
// cell, 0.95 and 0.92 at 4, 1.09 and 1.04 at 8, 1.52 and 1.32 at 32; 4M 0.81 and
// 0.80 at 4, 0.97 and 0.95 at 8; 20,000, whose sweep ends with its slowest warps,
// 0.98 and 0.97 at one, 1.07 and 1.09 at 4, 1.58 and 1.60 at 32.
double rows_max_occupancy(long long n) { return n >= 152 * 2048 ? 8.0 : 3.0; }

void fill_sweep_args(cl_list* c, clk::SweepArgs* A) {
  A->xs = c->xs;
  A->cellc = c->cellc;
  A->cell_start = c->cell_start;
  A->n = c->n;
  A->nx = c->geo.n[0];
  A->ny = c->geo.n[1];
  A->nz = c->geo.n[2];
  A->rc2 = (float)(c->geo.rc * c->geo.rc);
  A->irc = (float)(1.0 / c->geo.rc);
  A->irc2 = (float)(1.0 / (c->geo.rc * c->geo.rc));
  float e[3];
  clk::cell_halfwidths(c->geo, e);
  A->ex = e[0];
  A->ey = e[1];
  A->ez = e[2];
}

bool same_box(const cl_box& a, const cl_box& b) {
  if (a.dim != b.dim || a.lcell != b.lcell || !(a.cutoff == b.cutoff)) return false;
  for (int k = 0; k < a.dim * a.dim; ++k)
    if (!(a.h[k] == b.h[k])) return false;
  return true;
}

int set_geometry(cl_list* c, const cl_box* box, cudaStream_t s) {
  clk::Geo g;
  int e = clk::prepare_geometry(box, &g);
  if (e) return e;
  struct Host {
    clk::Off off[2 * clk::kMaxOff];
    int opk_half[clk::kMaxOff], opk_full[clk::kMaxOff];
  };
  std::unique_ptr<Host> t(new (std::nothrow) Host);
  if (!t) return CL_ERR_OOM;
  int nh = 0, nf = 0;
  if ((e = clk::build_stencils(g, clk::kMaxOff, t->off, t->opk_half, &nh, t->off + clk::kMaxOff, t->opk_full, &nf)))
    return e;
  // A larger grid than the block has room for needs a new one. One of less than a
  // quarter of a large block (2^20 cells: 18 MB) gives the surplus back, if it
  // can: the old block serves as well. The list is unchanged until nothing can
  // fail.
  void* block = nullptr;
  const bool grows = g.ncells > c->ncells_alloc;
  if (grows || (c->ncells_alloc > (1 << 20) && g.ncells < c->ncells_alloc / 4)) {
    Cells p;
    e = clk::mem_alloc(&block, carve_cells(&p, nullptr, g.ncells), s);
    if (e && grows) return e;
  }
  std::memmove(t->off + nh, t->off + clk::kMaxOff, sizeof(clk::Off) * nf);  // one after the other: one copy
  // pageable source: staged before the call returns, where a captured copy would
  // read it when the graph runs
  const size_t bytes = sizeof(clk::Off) * (nh + nf);
  if ((clk::capturing(s) ? cudaMemcpy(c->d_off_half, t->off, bytes, cudaMemcpyHostToDevice)
                         : cudaMemcpyAsync(c->d_off_half, t->off, bytes, cudaMemcpyHostToDevice, s)) != cudaSuccess) {
    clk::mem_free(block, s);
    return CL_ERR_CUDA;
  }
  if (block) adopt_cells(c, block, g.ncells, s);
  c->d_off_full = c->d_off_half + nh;
  std::memcpy(c->half->off, t->off, sizeof(clk::Off) * nh);
  std::memcpy(c->full->off, t->off + nh, sizeof(clk::Off) * nf);
  std::memset(c->hood, 0, sizeof(*c->hood));
  if (g.dim == 3) clk::fill_hood_args(g, t->opk_full, nf, t->opk_half, nh, c->hood);
  c->hood->flag = c->hflag;
  c->hood->list = c->hlist;
  c->hood->dense = c->hdense;
  c->hood->hforce = c->hforce;
  c->hood->xl = c->xl;
  c->hood->slot = c->slot;
  c->half->noff = nh;
  c->full->noff = nf;
  c->half->nrow2 = c->full->nrow2 = 0;
  if (g.dim == 2 && (double)c->n < rows_max_occupancy(c->n) * (double)g.ncells) {
    clk::fill_rows2(t->opk_half, nh, c->half);
    clk::fill_rows2(t->opk_full, nf, c->full);
  }
  c->geo = g;
  c->box = *box;
  fill_sweep_args(c, c->half);
  fill_sweep_args(c, c->full);
  return CL_OK;
}

int run_build(cl_list* c, cudaStream_t s) {
  clk::BuildBufs b;
  b.pos = c->pos;
  b.n = c->n;
  b.slot = c->slot;
  c->lists_half = 0;  // new cell contents: the sweeps' work lists are rebuilt
  if (clk::capturing(s)) c->replayed = 1;
  b.xl = c->xl;
  b.counts = c->counts;
  b.cell_start = c->cell_start;
  b.tile_sum = c->tile_sum;
  b.meta = c->meta;
  b.xs = c->xs;
  b.cellc = c->cellc;
  return clk::launch_build(c->geo, b, s);
}

// The flag that tells a sweep whether the work lists are there. A captured sweep
// makes its own, for the cell contents it is replayed on, and lists of contents that
// a graph may replace are made at every sweep: the sweeps' buffers are sized by the
// lists, which must be those of the cells they meet.
int* kept_lists(cl_list* c, cudaStream_t s) {
  if (!c->replayed && !clk::capturing(s)) return &c->lists_half;
  c->lists_none = 0;
  return &c->lists_none;
}

// Squared radius about a cell's centre that holds every particle within rc of
// a point of the cell: (rc + half the longest cell diagonal + a margin)^2.
float pairs_ball2(const clk::Geo& g) {
  double hd = 0.0;
  for (int corner = 0; corner < (1 << g.dim); ++corner) {
    double v[3] = {0, 0, 0};
    for (int k = 0; k < g.dim; ++k) {
      const double sg = ((corner >> k) & 1) ? 0.5 : -0.5;
      for (int a = 0; a < g.dim; ++a) v[a] += sg * g.h[k * 3 + a] / g.n[k];
    }
    hd = std::max(hd, std::sqrt(v[0] * v[0] + v[1] * v[1] + v[2] * v[2]));
  }
  const double r = g.rc + hd * (1.0 + 1e-6) + 1e-4 * (g.rc + hd);
  return (float)(r * r);
}

// Particles the pair list's staging ball holds at the box's mean density.
double pairs_expected(const clk::Geo& g, long long n, float ball2) {
  double vol = 1.0;
  if (g.dim == 3)
    vol = std::fabs(g.h[0] * (g.h[4] * g.h[8] - g.h[5] * g.h[7]) - g.h[1] * (g.h[3] * g.h[8] - g.h[5] * g.h[6]) +
                    g.h[2] * (g.h[3] * g.h[7] - g.h[4] * g.h[6]));
  else
    vol = std::fabs(g.h[0] * g.h[4] - g.h[1] * g.h[3]);
  const double r = std::sqrt((double)ball2);
  const double ball = g.dim == 3 ? 4.18879020478639 * r * r * r : 3.14159265358979 * r * r;
  return (vol > 0 ? (double)n / vol : 0.0) * ball;
}

// The stencil holds a cell twice: it reaches m_k cells each way along an axis of
// fewer than 2 m_k + 1 (the reach of build_stencils).
bool stencil_wraps(const clk::Geo& g) {
  for (int k = 0; k < g.dim; ++k)
    if (g.n[k] < 2 * (int)std::ceil(g.rc * g.n[k] / g.w[k]) + 1) return true;
  return false;
}

// Staged entries per cell: that with 30 % to spare, in steps of 128 (1,024 to
// 3,072). Denser cells overflow and take the per-particle path.
int pairs_stage_cap(double expect) {
  const int cap = (int)std::ceil((expect * 1.3 + 64.0) / 128.0) * 128;
  return std::min(3072, std::max(1024, cap));
}

// Neighbour list: count pass, scan, one synchronisation to learn the total,
// fill pass (each segment sorted as it is written).
int map_pairlist(cl_list* c, cl_result* r, cudaStream_t s) {
  if (!r->npairs || r->capacity < 0) return CL_ERR_INVALID_ARG;
  for (int k = 0; k < c->geo.dim; ++k)
    if (!(2.0 * c->geo.rc <= c->geo.w[k])) return CL_ERR_CUTOFF_TOO_LARGE;  // unique images only
  int e;
  if (!c->pair_block) {
    const size_t n = (size_t)c->n;
    auto carve = [&](char* base) {
      clk::Carver v{base};
      v.take(&c->pl_count, n);
      v.take(&c->pl_start, n + 1);
      v.take(&c->pl_tiles, (size_t)clk::scan_tiles_for(c->n));
      v.take(&c->pl_meta, 8);
      v.take(&c->pl_long, n);
      return v.used;
    };
    const size_t bytes = carve(nullptr);
    if ((e = clk::mem_alloc(&c->pair_block, bytes, s))) return e;
    carve((char*)c->pair_block);
    c->bytes += bytes;
  }
  const int dim = c->geo.dim;
  // the cells' buffers are shared with the binning (counts) and with the
  // neighbourhood sweep, which rewrite them on every launch
  clk::PairLists L;
  L.ball2 = pairs_ball2(c->geo);
  L.expect = pairs_expected(c->geo, c->n, L.ball2);
  L.cap = pairs_stage_cap(L.expect);
  L.images = stencil_wraps(c->geo);
  L.last = c->hdense;
  L.flag = c->hflag;
  L.fcells = c->hlist;
  L.mid = c->counts;
  L.ctr = c->pl_meta;
  L.count = c->pl_count;
  c->lists_half = 0;  // the pair list's passes use the list buffers
  if ((e = clk::launch_pairs_count(*c->full, c->d_off_full, dim, L, s))) return e;
  if ((e = clk::launch_scan64(c->pl_count, c->n, c->pl_tiles, c->pl_start, s))) return e;
  long long total = 0;
  if (cudaMemcpyAsync(&total, c->pl_start + c->n, sizeof(long long), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
      cudaStreamSynchronize(s) != cudaSuccess)
    return CL_ERR_CUDA;
  *r->npairs = total;
  if ((e = cl_pairlist_fits(total, r->capacity))) return e;
  if (total == 0) return CL_OK;
  if (!r->pair_i || !r->pair_j || !r->pair_d) return CL_ERR_INVALID_ARG;
  return clk::launch_pairs_fill(*c->full, c->d_off_full, dim, L, c->pl_start, r->pair_i, r->pair_j, r->pair_d, c->pl_long,
                                s);
}

}  // namespace

namespace clk {
void list_parts(const cl_list* cl, ListParts* p) {
  cl_list* c = const_cast<cl_list*>(cl);
  p->half = c->half;
  p->full = c->full;
  p->partials = c->partials;
  p->sums = c->sums;
  p->hforce = c->hforce;
  p->rc = c->geo.rc;
}
}  // namespace clk

extern "C" {

int cl_pairlist_fits(long long npairs, long long capacity) {
  if (npairs < 0) return CL_ERR_INVALID_ARG;  // a total read back from the 64-bit scan is never negative
  return npairs > capacity ? CL_ERR_CAPACITY : CL_OK;
}

const char* cl_error_string(int code) {
  switch (code) {
    case CL_OK: return "ok";
    case CL_ERR_INVALID_ARG: return "invalid argument";
    case CL_ERR_INVALID_BOX: return "singular or non-finite box matrix";
    case CL_ERR_CUTOFF_TOO_LARGE: return "cutoff too large for the box";
    case CL_ERR_NONFINITE: return "non-finite position";
    case CL_ERR_OOM: return "device out of memory";
    case CL_ERR_CAPACITY: return "pair list capacity exceeded";
    case CL_ERR_TIMEOUT: return "device wait timed out";
    case CL_ERR_CUDA: return "CUDA runtime error";
    case CL_ERR_UNSUPPORTED: return "grid or stencil beyond library limits";
    default: return "unknown error";
  }
}

int cl_box_info(const cl_box* box, long long* grid, double* widths, long long* stencil) {
  if (!box) return CL_ERR_INVALID_ARG;
  clk::Geo g;
  int e = clk::prepare_geometry(box, &g);
  if (e) return e;
  clk::Off* tmp = new (std::nothrow) clk::Off[clk::kMaxOff];
  if (!tmp) return CL_ERR_OOM;
  int nh = clk::build_stencil(g, 1, tmp, clk::kMaxOff);
  int nf = clk::build_stencil(g, 0, tmp, clk::kMaxOff);
  delete[] tmp;
  if (nh < 0) return nh;
  if (nf < 0) return nf;
  for (int k = 0; k < 3; ++k) {
    if (grid) grid[k] = g.n[k];
    if (widths) widths[k] = k < g.dim ? g.w[k] : 0.0;
  }
  if (stencil) {
    stencil[0] = nh;
    stencil[1] = nf;
  }
  return CL_OK;
}

int cl_build(const double* pos_dev, long long n, const cl_box* box, void* stream, cl_list** out) {
  if (!out || !box || n < 0 || n >= 2147483647LL || (n > 0 && !pos_dev)) return CL_ERR_INVALID_ARG;
  *out = nullptr;
  cl_list* c = new (std::nothrow) cl_list;
  if (!c) return CL_ERR_OOM;
  std::memset(c, 0, sizeof(*c));
  c->half = new (std::nothrow) clk::SweepArgs;
  c->full = new (std::nothrow) clk::SweepArgs;
  c->hood = new (std::nothrow) clk::HoodArgs;
  if (!c->half || !c->full || !c->hood) {
    free_all(c);
    delete c;
    return CL_ERR_OOM;
  }
  std::memset(c->half, 0, sizeof(clk::SweepArgs));
  std::memset(c->full, 0, sizeof(clk::SweepArgs));
  c->n = (int)n;
  c->pos = pos_dev;
  c->ncells_alloc = -1;
  cudaStream_t s = (cudaStream_t)stream;
  int e = cudaGetDevice(&c->device) == cudaSuccess ? CL_OK : CL_ERR_CUDA;
  char* zero = nullptr;
  size_t zero_bytes = 0;
  c->bytes = carve_list(c, nullptr, box->dim, &zero, &zero_bytes);
  if (!e) e = clk::mem_alloc(&c->block, c->bytes, s);
  if (!e) {
    carve_list(c, (char*)c->block, box->dim, &zero, &zero_bytes);
    if (cudaMemsetAsync(zero, 0, zero_bytes, s) != cudaSuccess) e = CL_ERR_CUDA;
  }
  if (!e) e = set_geometry(c, box, s);
  if (!e) e = run_build(c, s);
  if (e) {
    if (!clk::capturing(s)) cudaStreamSynchronize(s);
    free_all(c);
    delete c;
    return e;
  }
  *out = c;
  return CL_OK;
}

int cl_update(cl_list* c, const double* pos_dev, const cl_box* box, void* stream) {
  if (!c || (c->n > 0 && !pos_dev)) return CL_ERR_INVALID_ARG;
  // an unchanged box keeps its grid, stencils and buffers (a differentiable
  // step passes its box every time)
  if (box && !same_box(*box, c->box)) {
    int e = set_geometry(c, box, (cudaStream_t)stream);
    if (e) return e;
  }
  c->pos = pos_dev;
  return run_build(c, (cudaStream_t)stream);
}

int cl_map(const cl_list* cc, cl_reduction red, const cl_params* params, cl_result* r, void* stream) {
  if (!cc || !r) return CL_ERR_INVALID_ARG;
  cl_list* c = const_cast<cl_list*>(cc);
  cudaStream_t s = (cudaStream_t)stream;
  const int dim = c->geo.dim;
  switch (red) {
    case CL_RED_COUNT:
      if (!r->count) return CL_ERR_INVALID_ARG;
      if (scalar_staged(c))
        return clk::launch_hood_scalar(*c->half, *c->hood, c->work, 0, r->count, c->partials, hood_cap(c), c->sums,
                                       nullptr, 0, 0.f, nullptr, s, kept_lists(c, s));
      return clk::launch_count(*c->half, dim, r->count, s);
    case CL_RED_SUM_INV_R:
      if (!r->sum_inv_r) return CL_ERR_INVALID_ARG;
      if (scalar_staged(c))
        return clk::launch_hood_scalar(*c->half, *c->hood, c->work, 1, nullptr, c->partials, hood_cap(c), c->sums,
                                       r->sum_inv_r, 0, 0.f, nullptr, s, kept_lists(c, s));
      return clk::launch_scalar(*c->half, dim, 0, c->partials, c->sums, r->sum_inv_r, s);
    case CL_RED_SF_ENERGY:
      if (!r->energy) return CL_ERR_INVALID_ARG;
      if (dim == 3 && c->n > 0 && clk::hood_half_fits(*c->half))
        return clk::launch_hood_scalar(*c->half, *c->hood, c->work, 3, nullptr, c->partials, hood_cap(c), c->sums,
                                       r->energy, 0, 0.f, nullptr, s, kept_lists(c, s));
      if (dim == 3 && c->n > 0)
        return clk::launch_hood(*c->half, nullptr, *c->hood, c->work, 2, c->geo.hinv, nullptr, nullptr, nullptr, nullptr,
                                c->partials, hood_cap(c), c->sums, r->energy, nullptr, nullptr, s, kept_lists(c, s));
      return clk::launch_scalar(*c->half, dim, 1, c->partials, c->sums, r->energy, s);
    case CL_RED_SF_ENERGY_FORCES_VIRIAL:
      if (!r->forces && c->n > 0) return CL_ERR_INVALID_ARG;
      if (dim == 3 && c->n > 0) {
        c->last_half = clk::half_path_applies(*c->full, c->half, *c->hood, 0) ? 1 : 0;
        return clk::launch_hood(*c->full, c->half, *c->hood, c->work, 0, c->geo.hinv, r->forces, nullptr, nullptr, nullptr,
                                c->partials, hood_cap(c), c->sums, r->energy, r->virial, nullptr, s, kept_lists(c, s));
      }
      return clk::launch_force(*c->full, dim, 0, c->geo.hinv, r->forces, nullptr, nullptr, nullptr, c->partials,
                               c->sums, r->energy, r->virial, nullptr, s);
    case CL_RED_HIST: {
      if (!params || !r->hist || params->nbins < 1 || params->nbins > clk::kMaxBins) return CL_ERR_INVALID_ARG;
      double rmax = params->rmax > 0 ? params->rmax : c->geo.rc;
      if (scalar_staged(c))
        return clk::launch_hood_scalar(*c->half, *c->hood, c->work, 2, nullptr, c->partials, hood_cap(c), c->sums,
                                       nullptr, params->nbins, (float)rmax, r->hist, s, kept_lists(c, s));
      return clk::launch_hist(*c->half, dim, params->nbins, (float)rmax, r->hist, s);
    }
    case CL_RED_PAIRLIST:
      return map_pairlist(c, r, s);
    default:
      return CL_ERR_INVALID_ARG;
  }
}

int cl_backward(const cl_list* cc, const double* grad_energy_dev, double* grad_pos_dev, double* grad_box_dev,
                double* virial_dev, void* stream) {
  if (!cc || !grad_energy_dev || (cc->n > 0 && !grad_pos_dev)) return CL_ERR_INVALID_ARG;
  cl_list* c = const_cast<cl_list*>(cc);
  cudaStream_t s = (cudaStream_t)stream;
  if (c->geo.dim == 3 && c->n > 0) {
    c->last_half = clk::half_path_applies(*c->full, c->half, *c->hood, 1) ? 1 : 0;
    return clk::launch_hood(*c->full, c->half, *c->hood, c->work, 1, c->geo.hinv, nullptr, grad_pos_dev, grad_energy_dev,
                            c->pos, c->partials, hood_cap(c), c->sums, nullptr, virial_dev, grad_box_dev,
                            s, kept_lists(c, s));
  }
  return clk::launch_force(*c->full, c->geo.dim, 1, c->geo.hinv, nullptr, grad_pos_dev, grad_energy_dev, c->pos,
                           c->partials, c->sums, nullptr, virial_dev, grad_box_dev, s);
}

int cl_energy_grad(const cl_list* cc, const double* scale_dev, double* energy_dev, double* grad_pos_dev,
                   double* grad_box_dev, double* virial_dev, void* stream) {
  if (!cc || !scale_dev || !energy_dev || (cc->n > 0 && !grad_pos_dev)) return CL_ERR_INVALID_ARG;
  cl_list* c = const_cast<cl_list*>(cc);
  cudaStream_t s = (cudaStream_t)stream;
  if (c->geo.dim == 3 && c->n > 0) {
    c->last_half = clk::half_path_applies(*c->full, c->half, *c->hood, 3) ? 1 : 0;
    return clk::launch_hood(*c->full, c->half, *c->hood, c->work, 3, c->geo.hinv, nullptr, grad_pos_dev, scale_dev, c->pos,
                            c->partials, hood_cap(c), c->sums, energy_dev, virial_dev, grad_box_dev, s,
                            kept_lists(c, s));
  }
  // 2D (and the empty list): the energy sweep, then the backward sweep
  int e = clk::launch_scalar(*c->half, c->geo.dim, 1, c->partials, c->sums, energy_dev, s);
  if (e) return e;
  return clk::launch_force(*c->full, c->geo.dim, 1, c->geo.hinv, nullptr, grad_pos_dev, scale_dev, c->pos,
                           c->partials, c->sums, nullptr, virial_dev, grad_box_dev, s);
}

int cl_scale(const double* scale_dev, const double* in_dev, double* out_dev, long long count, void* stream) {
  if (count < 0 || (count > 0 && (!scale_dev || !in_dev || !out_dev))) return CL_ERR_INVALID_ARG;
  return clk::launch_scale(scale_dev, in_dev, out_dev, count, (cudaStream_t)stream);
}

// ---- two sets: queries of set B against the cell list of set A
namespace {

int check_query(const cl_list* c, const double* posb, long long nb) {
  if (!c || nb < 0 || nb >= 2147483647LL || (nb > 0 && !posb)) return CL_ERR_INVALID_ARG;
  return CL_OK;
}

// Workspace of one two-set call: pieces of one block of the library's pool.
struct QueryWs {
  clk::QueryBufs bin{};
  int* count = nullptr;
  long long* start = nullptr;  // nb + 1 offsets (64-bit), then the error latch
  long long* tiles = nullptr;
  int* meta = nullptr;
  int* err = nullptr;
  int* longs = nullptr;
  int* knn_a = nullptr;
  float* knn_d = nullptr;
  float* part_d = nullptr;
  long long* part_id = nullptr;

  QueryWs(cl_list* list, cudaStream_t stream) : c(list), s(stream) {}
  ~QueryWs() {
    clk::mem_free(base, s);
    if (bytes > clk::kPoolKeep) clk::mem_settle(s);
  }
  // list: the arrays of the cross list; k > 0: those of the global k closest.
  int open(long long nb, bool list, int k) {
    const size_t need = carve(nullptr, nb, list, k);
    if (int e = clk::mem_alloc(&base, need, s)) return e;
    bytes = need;
    carve((char*)base, nb, list, k);
    return cudaMemsetAsync(err, 0, sizeof(long long), s) == cudaSuccess ? CL_OK : CL_ERR_CUDA;
  }

 private:
  size_t carve(char* at, long long nb, bool list, int k) {
    clk::Carver v{at};
    const size_t n = nb > 0 ? (size_t)nb : 1;
    const long long nc = c->geo.ncells;
    v.take(&bin.q, n);
    v.take(&bin.cell, n);
    if (clk::queries_sorted(c->n, nb, nc)) {
      v.take(&bin.raw, n);
      v.take(&bin.slot, n);
      v.take(&bin.counts, (size_t)nc);
      v.take(&bin.start, (size_t)nc + 1);
      v.take(&bin.tiles, (size_t)clk::scan_tiles_for(nc));
      v.take(&bin.meta, 4);
    }
    if (list) {
      v.take(&count, n);
      v.take(&tiles, (size_t)clk::scan_tiles_for((long long)n));
      v.take(&meta, 4);
      v.take(&longs, n);
    }
    v.take(&start, list ? n + 2 : 1);
    err = reinterpret_cast<int*>(start + (list ? n + 1 : 0));
    if (k > 0) {
      const size_t parts = (size_t)clk::topk_parts((long long)n, k);
      v.take(&knn_a, n * k);
      v.take(&knn_d, n * k);
      v.take(&part_d, parts * k);
      v.take(&part_id, parts * k);
    }
    return v.used;
  }
  cl_list* c;
  cudaStream_t s;
  void* base = nullptr;
  size_t bytes = 0;
};

int read_err(const int* err_dev, cudaStream_t s) {
  int v = 0;
  if (cudaMemcpyAsync(&v, err_dev, sizeof(int), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
      cudaStreamSynchronize(s) != cudaSuccess)
    return CL_ERR_CUDA;
  return v ? CL_ERR_NONFINITE : CL_OK;
}

}  // namespace

int cl_cross_count(const cl_list* cc, const double* posb_dev, long long nb, unsigned long long* count_dev,
                   void* stream) {
  int e = check_query(cc, posb_dev, nb);
  if (e || !count_dev) return e ? e : CL_ERR_INVALID_ARG;
  cl_list* c = const_cast<cl_list*>(cc);
  cudaStream_t s = (cudaStream_t)stream;
  if (cudaMemsetAsync(count_dev, 0, sizeof(unsigned long long), s) != cudaSuccess) return CL_ERR_CUDA;
  QueryWs w(c, s);
  clk::Queries q;
  if ((e = w.open(nb, false, 0)) || (e = clk::launch_query_bin(*c->full, c->geo, posb_dev, nb, w.bin, w.err, &q, s)) ||
      (e = clk::launch_cross_count(*c->full, c->d_off_full, q, nullptr, count_dev, s)))
    return e;
  return read_err(w.err, s);
}

int cl_cross_pairlist(const cl_list* cc, const double* posb_dev, long long nb, long long capacity, int* pa_dev,
                      int* pb_dev, float* pd_dev, long long* npairs, void* stream) {
  int e = check_query(cc, posb_dev, nb);
  if (e || !npairs || capacity < 0) return e ? e : CL_ERR_INVALID_ARG;
  cl_list* c = const_cast<cl_list*>(cc);
  for (int k = 0; k < c->geo.dim; ++k)
    if (!(2.0 * c->geo.rc <= c->geo.w[k])) return CL_ERR_CUTOFF_TOO_LARGE;  // unique images only
  cudaStream_t s = (cudaStream_t)stream;
  *npairs = 0;
  if (nb == 0) return CL_OK;
  QueryWs w(c, s);
  clk::Queries q;
  if ((e = w.open(nb, true, 0)) || (e = clk::launch_query_bin(*c->full, c->geo, posb_dev, nb, w.bin, w.err, &q, s)) ||
      (e = clk::launch_cross_count(*c->full, c->d_off_full, q, w.count, nullptr, s)) ||
      (e = clk::launch_scan64(w.count, nb, w.tiles, w.start, s)))
    return e;
  long long back[2] = {0, 0};  // the total and, after it, the error latch
  if (cudaMemcpyAsync(back, w.start + nb, sizeof(back), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
      cudaStreamSynchronize(s) != cudaSuccess)
    return CL_ERR_CUDA;
  if (back[1]) return CL_ERR_NONFINITE;
  const long long total = back[0];
  *npairs = total;
  if ((e = cl_pairlist_fits(total, capacity))) return e;
  if (total == 0) return CL_OK;
  if (!pa_dev || !pb_dev || !pd_dev) return CL_ERR_INVALID_ARG;
  if ((e = clk::launch_cross_fill(*c->full, c->d_off_full, q, w.count, w.start, pa_dev, pb_dev, pd_dev, w.longs,
                                  w.meta + 3, s)))
    return e;
  return cudaStreamSynchronize(s) == cudaSuccess ? CL_OK : CL_ERR_CUDA;
}

int cl_cross_knn(const cl_list* cc, const double* posb_dev, long long nb, int k, int* knn_a_dev, float* knn_d_dev,
                 void* stream) {
  int e = check_query(cc, posb_dev, nb);
  if (e || k < 1 || k > CL_KNN_MAX || (nb > 0 && (!knn_a_dev || !knn_d_dev))) return e ? e : CL_ERR_INVALID_ARG;
  cl_list* c = const_cast<cl_list*>(cc);
  cudaStream_t s = (cudaStream_t)stream;
  if (nb == 0) return CL_OK;
  QueryWs w(c, s);
  clk::Queries q;
  if ((e = w.open(nb, false, 0)) || (e = clk::launch_query_bin(*c->full, c->geo, posb_dev, nb, w.bin, w.err, &q, s)) ||
      (e = clk::launch_cross_knn(*c->full, c->d_off_full, q, k, knn_a_dev, knn_d_dev, s)))
    return e;
  return read_err(w.err, s);
}

int cl_cross_topk(const cl_list* cc, const double* posb_dev, long long nb, int k, int* a_dev, int* b_dev,
                  float* d_dev, long long* nfound, void* stream) {
  int e = check_query(cc, posb_dev, nb);
  if (e || k < 1 || k > CL_KNN_MAX || !a_dev || !b_dev || !d_dev || !nfound) return e ? e : CL_ERR_INVALID_ARG;
  cl_list* c = const_cast<cl_list*>(cc);
  cudaStream_t s = (cudaStream_t)stream;
  *nfound = 0;
  QueryWs w(c, s);
  clk::Queries q;
  // err[0]: the error latch, err[1]: the number found
  if ((e = w.open(nb, false, k)) || (e = clk::launch_query_bin(*c->full, c->geo, posb_dev, nb, w.bin, w.err, &q, s)) ||
      (e = clk::launch_cross_knn(*c->full, c->d_off_full, q, k, w.knn_a, w.knn_d, s)) ||
      (e = clk::launch_topk_merge(w.knn_a, w.knn_d, nb, k, w.part_d, w.part_id, a_dev, b_dev, d_dev, w.err + 1, s)))
    return e;
  int back[2] = {0, 0};
  if (cudaMemcpyAsync(back, w.err, sizeof(back), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
      cudaStreamSynchronize(s) != cudaSuccess)
    return CL_ERR_CUDA;
  if (back[0]) return CL_ERR_NONFINITE;
  *nfound = back[1];
  return CL_OK;
}

int cl_query(const cl_list* c, int what, long long* value, void* stream) {
  if (!c || !value) return CL_ERR_INVALID_ARG;
  cudaStream_t s = (cudaStream_t)stream;
  switch (what) {
    case CL_INFO_N: *value = c->n; return CL_OK;
    case CL_INFO_DIM: *value = c->geo.dim; return CL_OK;
    case CL_INFO_GRID_X: *value = c->geo.n[0]; return CL_OK;
    case CL_INFO_GRID_Y: *value = c->geo.n[1]; return CL_OK;
    case CL_INFO_GRID_Z: *value = c->geo.n[2]; return CL_OK;
    case CL_INFO_NCELLS: *value = c->geo.ncells; return CL_OK;
    case CL_INFO_BYTES: *value = (long long)c->bytes; return CL_OK;
    case CL_INFO_STENCIL_HALF: *value = c->half->noff; return CL_OK;
    case CL_INFO_STENCIL_FULL: *value = c->full->noff; return CL_OK;
    case CL_INFO_WORK_TILES: *value = (c->n + 255) / 256; return CL_OK;
    case CL_INFO_NONEMPTY:
    case CL_INFO_MAX_OCCUPANCY: {
      int m[3];
      if (cudaStreamSynchronize(s) != cudaSuccess) return CL_ERR_CUDA;
      if (cudaMemcpy(m, c->meta, sizeof(m), cudaMemcpyDeviceToHost) != cudaSuccess) return CL_ERR_CUDA;
      *value = what == CL_INFO_NONEMPTY ? m[1] : m[2];
      return CL_OK;
    }
    case CL_INFO_SWEEP_HALF:
      *value = c->last_half;
      return CL_OK;
    case CL_INFO_SWEEP_CANDIDATES: {
      unsigned long long v = 0;
      if (cudaMemcpyAsync(&v, c->work + 2, sizeof(v), cudaMemcpyDeviceToHost, s) != cudaSuccess) return CL_ERR_CUDA;
      if (cudaStreamSynchronize(s) != cudaSuccess) return CL_ERR_CUDA;
      *value = (long long)v;
      return CL_OK;
    }
    case CL_INFO_CANDIDATES: {
      int e = clk::launch_candidates(*c->half, c->geo.ncells, c->u64, s);
      if (e) return e;
      unsigned long long v = 0;
      if (cudaMemcpyAsync(&v, c->u64, sizeof(v), cudaMemcpyDeviceToHost, s) != cudaSuccess) return CL_ERR_CUDA;
      if (cudaStreamSynchronize(s) != cudaSuccess) return CL_ERR_CUDA;
      *value = (long long)v;
      return CL_OK;
    }
    default: return CL_ERR_INVALID_ARG;
  }
}

int cl_get_view(const cl_list* c, cl_view* v) {
  if (!c || !v) return CL_ERR_INVALID_ARG;
  static_assert(sizeof(cl_offset) == sizeof(clk::Off), "public and internal stencil entries differ");
  v->dim = c->geo.dim;
  v->n = c->n;
  v->nx = c->geo.n[0];
  v->ny = c->geo.n[1];
  v->nz = c->geo.n[2];
  v->cutoff = (float)c->geo.rc;
  v->xs = c->xs;
  v->cellc = c->cellc;
  v->cell_start = c->cell_start;
  v->off_half = reinterpret_cast<const cl_offset*>(c->d_off_half);
  v->noff_half = c->half->noff;
  v->off_full = reinterpret_cast<const cl_offset*>(c->d_off_full);
  v->noff_full = c->full->noff;
  return CL_OK;
}

int cl_status(cl_list* c, void* stream) {
  if (!c) return CL_ERR_INVALID_ARG;
  cudaStream_t s = (cudaStream_t)stream;
  int flag = 0;
  if (cudaStreamSynchronize(s) != cudaSuccess) return CL_ERR_CUDA;
  if (cudaMemcpy(&flag, c->meta, sizeof(int), cudaMemcpyDeviceToHost) != cudaSuccess) return CL_ERR_CUDA;
  if (flag) {
    int zero = 0;
    if (cudaMemcpy(c->meta, &zero, sizeof(int), cudaMemcpyHostToDevice) != cudaSuccess) return CL_ERR_CUDA;
  }
  return (flag & clk::kErrNonFinite) ? CL_ERR_NONFINITE : CL_OK;
}

void cl_free(cl_list* c) {
  if (!c) return;
  int dev = -1;
  const bool other = cudaGetDevice(&dev) == cudaSuccess && dev != c->device;
  if (other) cudaSetDevice(c->device);
  cudaDeviceSynchronize();  // what earlier calls freed beyond kPoolKeep goes back here
  free_all(c);
  if (c->bytes > clk::kPoolKeep / 16) clk::mem_settle(nullptr);
  if (other) cudaSetDevice(dev);
  delete c;
}

}  // extern "C"
