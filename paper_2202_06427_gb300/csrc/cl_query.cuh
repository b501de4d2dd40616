// cl_query.cuh -- one warp about one point: the device pieces of the two-set
// sweeps (cl_cross.cu) and of the pair list's cells that overflow their staging
// (cl_pairs.cu). The warp's lanes test the stencil's cells 32 at a time (the
// cell's bounding box against the cutoff, as in sweep_particle2), the kept ones
// are compacted in shared memory, and groups of G lanes run over them. The
// displacement to a particle is x + (S_o - p).
#pragma once

#include <cfloat>

#include "cl_sweep.cuh"

namespace clk {

struct CrossArgs {
  const float4* xs;
  const int* cell_start;
  const Off* off;  // device memory
  int noff;
  int nx, ny, nz;
  float rc2;
  float ex, ey, ez;  // padded half-widths of a cell's bounding box; cull: use them
  bool cull;
};

// A warp's stencil cells under way: shift minus the query (w: squared distance
// of the query to the cell's bounding box) and range of sorted particles.
struct WarpCells {
  float4 s[32];
  int2 j[32];
};

// Stencil to shared memory: (S_x, S_y, S_z, dx | dy << 10 | dz << 20).
// NEAR: in order of |S|, so that the nearest cells come first.
template <bool NEAR>
__device__ __forceinline__ void load_stencil(const CrossArgs& A, float4* stab, float* key) {
  for (int k = threadIdx.x; k < A.noff; k += blockDim.x) {
    const Off o = A.off[k];
    const float4 e = make_float4(o.sx, o.sy, o.sz,
                                 __uint_as_float((unsigned)o.dx | ((unsigned)o.dy << 10) | ((unsigned)o.dz << 20)));
    if (NEAR) key[k] = fmaf(o.sx, o.sx, fmaf(o.sy, o.sy, o.sz * o.sz));
    else stab[k] = e;
  }
  if (NEAR) {
    __syncthreads();
    for (int k = threadIdx.x; k < A.noff; k += blockDim.x) {
      const float v = key[k];
      int r = 0;  // entries before k in the order (|S|^2, k)
      for (int t = 0; t < A.noff; ++t) r += (key[t] < v || (key[t] == v && t < k)) ? 1 : 0;
      const Off o = A.off[k];
      stab[r] = make_float4(o.sx, o.sy, o.sz,
                            __uint_as_float((unsigned)o.dx | ((unsigned)o.dy << 10) | ((unsigned)o.dz << 20)));
    }
  }
  __syncthreads();
}

// Entries k0 + lane of the stencil about the query's cell: the non-empty cells
// within sqrt(lim) of the query (all of them without culling) go to W; returns
// their number. The squared box distance is taken FLT_MIN low, which changes it at
// 0 only: such a cell stays in when lim is 0, the k-th distance of a query on k
// points of the set, as a smaller index may tie there (beyond 0 the boxes'
// padding excludes a tie).
__device__ __forceinline__ int query_cells(const CrossArgs& A, const float4* stab, WarpCells& W, int k0, int lane,
                                           unsigned cc, const float4& p, float lim) {
  const int k = k0 + lane;
  bool keep = false;
  float4 e = make_float4(0.f, 0.f, 0.f, 0.f);
  int2 r = make_int2(0, 0);
  if (k < A.noff) {
    e = stab[k];
    const unsigned d = __float_as_uint(e.w);
    const float bx = fmaxf(fabsf(p.x - e.x) - A.ex, 0.f), by = fmaxf(fabsf(p.y - e.y) - A.ey, 0.f),
                bz = fmaxf(fabsf(p.z - e.z) - A.ez, 0.f);
    e.w = fmaf(bx, bx, fmaf(by, by, fmaf(bz, bz, -FLT_MIN)));
    if (!A.cull) e.w = -FLT_MIN;
    if (e.w < lim) {
      int x2 = (int)(cc & 1023u) + (int)(d & 1023u);
      x2 -= (x2 >= A.nx) ? A.nx : 0;
      int y2 = (int)((cc >> 10) & 1023u) + (int)((d >> 10) & 1023u);
      y2 -= (y2 >= A.ny) ? A.ny : 0;
      int z2 = (int)(cc >> 20) + (int)(d >> 20);
      z2 -= (z2 >= A.nz) ? A.nz : 0;
      const int c = x2 + A.nx * (y2 + A.ny * z2);
      r.x = __ldg(A.cell_start + c);
      r.y = __ldg(A.cell_start + c + 1);
      keep = r.y > r.x;
    }
  }
  const unsigned m = __ballot_sync(0xffffffffu, keep);
  __syncwarp();
  if (keep) {
    const int at = __popc(m & ((1u << lane) - 1u));
    W.s[at] = make_float4(e.x - p.x, e.y - p.y, e.z - p.z, e.w);
    W.j[at] = r;
  }
  __syncwarp();
  return __popc(m);
}

__device__ __forceinline__ float query_d2(const float4& q, const float4& s) {
  const float dx = q.x + s.x, dy = q.y + s.y, dz = q.z + s.z;
  return fmaf(dx, dx, fmaf(dy, dy, dz * dz));
}

// Particles within the cutoff of the point with an index above imin, this
// lane's share.
template <int G>
__device__ __forceinline__ unsigned query_count(const CrossArgs& A, const float4* stab, WarpCells& W, unsigned cc,
                                                const float4& p, int imin) {
  const int lane = threadIdx.x & 31;
  unsigned n = 0;
  for (int k0 = 0; k0 < A.noff; k0 += 32) {
    const int nk = query_cells(A, stab, W, k0, lane, cc, p, A.rc2);
    for (int i = lane / G; i < nk; i += 32 / G) {
      const float4 s = W.s[i];
      const int2 r = W.j[i];
#pragma unroll 2
      for (int j = r.x + lane % G; j < r.y; j += G) {
        const float4 q = __ldg(&A.xs[j]);
        n += query_d2(q, s) < A.rc2 && __float_as_int(q.w) > imin ? 1u : 0u;
      }
    }
  }
  return n;
}

// Calls f(e, a, d2) for every particle a > imin within the cutoff, e = 0, 1, ..
// over the warp; returns their number.
template <int G, class F>
__device__ __forceinline__ int query_hits(const CrossArgs& A, const float4* stab, WarpCells& W, unsigned cc,
                                          const float4& p, int imin, F&& f) {
  const int lane = threadIdx.x & 31;
  const unsigned lt = (1u << lane) - 1u;
  int L = 0;
  for (int k0 = 0; k0 < A.noff; k0 += 32) {
    const int nk = query_cells(A, stab, W, k0, lane, cc, p, A.rc2);
    for (int i0 = 0; i0 < nk; i0 += 32 / G) {
      const int i = i0 + lane / G;
      float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
      int j = 0, j1 = 0;
      if (i < nk) {
        s = W.s[i];
        const int2 r = W.j[i];
        j = r.x + lane % G;
        j1 = r.y;
      }
      while (__any_sync(0xffffffffu, j < j1)) {
        int a[2];
        float d2[2];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          a[u] = -1;
          d2[u] = FLT_MAX;
          if (j + u * G < j1) {
            const float4 q = __ldg(&A.xs[j + u * G]);
            a[u] = __float_as_int(q.w);
            d2[u] = query_d2(q, s);
          }
        }
        j += 2 * G;
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          const bool hit = d2[u] < A.rc2 && a[u] > imin;
          const unsigned m = __ballot_sync(0xffffffffu, hit);
          if (hit) f(L + __popc(m & lt), a[u], d2[u]);
          L += __popc(m);
        }
      }
    }
  }
  return L;
}

inline CrossArgs cross_args(const SweepArgs& A, const Off* off) {
  CrossArgs C;
  C.xs = A.xs;
  C.cell_start = A.cell_start;
  C.off = off;
  C.noff = A.noff;
  C.nx = A.nx;
  C.ny = A.ny;
  C.nz = A.nz;
  C.rc2 = A.rc2;
  C.ex = A.ex;
  C.ey = A.ey;
  C.ez = A.ez;
  // The padding of the box test covers the FP32 rounding of the coordinates
  // while cells are not thousands of cutoffs wide (capped grids).
  const float rc = sqrtf(A.rc2);
  C.cull = A.ex > 0.f && A.ex < 512.f * rc && A.ey < 512.f * rc && A.ez < 512.f * rc;
  return C;
}

// Lanes per cell: a group's last pass over a cell is partly empty, so small
// cells want small groups.
inline int group_lanes(const SweepArgs& A) {
  const double occ = (double)A.n / ((double)A.nx * A.ny * A.nz);
  return occ < 3.0 ? 2 : (occ < 8.0 ? 4 : 8);
}

}  // namespace clk
