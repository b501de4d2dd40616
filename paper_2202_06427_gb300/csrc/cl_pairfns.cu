// cl_pairfns.cu -- C entry points for the mapped functions of the paper's
// examples (Code 5, 6, 7, 10).
//
// In 3D the Lennard-Jones energy and forces, the mass-weighted sum and the
// velocity histogram run on sweeps of their own below, one thread per
// cell-sorted particle like the ready-made device functors of
// cellmap_pairfns.cuh, and add each particle's terms in the functors' order, so
// that their FP32 sums round alike. 2D, the Lennard-Jones energy alone and the mass
// sum of sparse lists run the functors on the compile-time hook of
// cellmap_functor.cuh, as a user's own would. (The half-shell sweep of cl_hood.cu does Lennard-Jones forces in half
// the functor's time, 0.74 against 1.57 ms at 500,000 particles, but its
// energy, summed pair by pair instead of per particle from both ends, differs
// from the functor's by 5e-9; it was left out.)
#include "cellmap_pairfns.cuh"
#include "cl_sweep.cuh"

namespace clk {
namespace {

// A particle's data in cell order: (x, y, z, mass), or its velocity.
__global__ void __launch_bounds__(256) k_sorted_mass(const float4* __restrict__ xs, int n,
                                                     const float* __restrict__ mass, float4* __restrict__ out) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= n) return;
  float4 v = xs[p];
  v.w = __ldg(mass + __float_as_int(v.w));
  out[p] = v;
}

__global__ void __launch_bounds__(256) k_sorted_velocity(const float4* __restrict__ xs, int n,
                                                         const float* __restrict__ vel, float4* __restrict__ out) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= n) return;
  const float* v = vel + (size_t)__float_as_int(xs[p].w) * 3;
  out[p] = make_float4(__ldg(v), __ldg(v + 1), __ldg(v + 2), 0.f);
}

// Sum of m_i m_j / r, one thread per sorted particle, two candidates per step
// in packed FP32 (scan_pairs with the masses in w). Against the functor, which
// loads m_j from the caller's array for every pair (long-scoreboard stalls 16
// per issue, 893 us at 500,000 particles in random order), the candidate's one
// 16-byte load brings its mass.
__device__ __forceinline__ void mass_scan(const float4* __restrict__ xm, int j0, int j1, float sx, float sy, float sz,
                                          float mi, float rc2, float& s) {
  const float2 s2x = f2(sx), s2y = f2(sy), s2z = f2(sz);
#pragma unroll 2
  for (int j = j0; j < j1; j += 2) {
    const float4 a = __ldg(&xm[j]);
    const float4 b = __ldg(&xm[min(j + 1, j1 - 1)]);
    const float2 dx = __fadd2_rn(make_float2(a.x, b.x), s2x);
    const float2 dy = __fadd2_rn(make_float2(a.y, b.y), s2y);
    const float2 dz = __fadd2_rn(make_float2(a.z, b.z), s2z);
    const float2 d2 = __ffma2_rn(dx, dx, __ffma2_rn(dy, dy, __fmul2_rn(dz, dz)));
    // one after the other into one sum, as the functor adds them; selects
    // instead of branches (a warp's step nearly always has a pair)
    const float t0 = fmaf(mi * a.w, rsqrtf(d2.x), s);
    s = d2.x < rc2 ? t0 : s;
    const float t1 = fmaf(mi * b.w, rsqrtf(d2.y), s);
    s = d2.y < rc2 && j + 1 < j1 ? t1 : s;
  }
}

__global__ void __launch_bounds__(256) k_sweep_mass(const __grid_constant__ SweepArgs A, const float4* __restrict__ xm,
                                                    float rc2, double* __restrict__ partials) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  float sum = 0.f;
  if (p < A.n) {
    const float4 pi = xm[p];
    const unsigned cc = A.cellc[p];
    const int cx = (int)(cc & 1023u), cy = (int)((cc >> 10) & 1023u), cz = (int)(cc >> 20);
    mass_scan(xm, p + 1, A.cell_start[cx + A.nx * (cy + A.ny * cz) + 1], -pi.x, -pi.y, -pi.z, pi.w, rc2, sum);
    for (int k = 1; k < A.noff; ++k) {
      const Off& o = A.off[k];
      const float bx = fmaxf(fabsf(pi.x - o.sx) - A.ex, 0.f), by = fmaxf(fabsf(pi.y - o.sy) - A.ey, 0.f),
                  bz = fmaxf(fabsf(pi.z - o.sz) - A.ez, 0.f);
      if (fmaf(bx, bx, fmaf(by, by, bz * bz)) >= rc2) continue;  // the whole cell is beyond the cutoff
      const int c = stencil_cell(A, k, cx, cy, cz);
      mass_scan(xm, A.cell_start[c], A.cell_start[c + 1], o.sx - pi.x, o.sy - pi.y, o.sz - pi.z, pi.w, rc2, sum);
    }
  }
  double v[1] = {(double)sum};
  block_sum_store<1>(v, partials + blockIdx.x);
}

// Pairwise-velocity histogram, one thread per sorted particle: per candidate
// the distance as the functor computes it (q - (x_i - S_o), so the same pairs
// fall in the same bins), two at a time in packed FP32; velocities in cell
// order, so a warp's loads fall together; the thread's bins (sum of |v_i - v_j|
// and count) in a shared-memory column of its own, where the functor kept them
// in local memory (20 KB of L1 per 256 threads and bins array), gathered every
// v_j from the caller's array (long-scoreboard stalls 11 per issue) and ended
// with a 32-step FP64 shuffle sum per warp and bin.
__global__ void k_sweep_velocity(const __grid_constant__ SweepArgs A, const float4* __restrict__ vs, float rc2,
                                 float inv_binstep, int nbins, unsigned long long* __restrict__ counts,
                                 double* __restrict__ vsum) {
  extern __shared__ float2 bins[];  // [bin][thread]: (sum, count bits)
  const int T = blockDim.x, t = threadIdx.x;
  for (int b = 0; b < nbins; ++b) bins[b * T + t] = make_float2(0.f, 0.f);
  const int p = blockIdx.x * T + t;
  if (p < A.n) {
    const float4 pi = A.xs[p], vi = vs[p];
    const unsigned cc = A.cellc[p];
    const int cx = (int)(cc & 1023u), cy = (int)((cc >> 10) & 1023u), cz = (int)(cc >> 20);
    auto pair = [&](float d2, int j) {
      // 1-based bin k = ceil(r / binstep), from the low mantissa bits of the
      // quotient + 2^23 rounded up (no conversion on the special-function unit);
      // d2 = 0 gives NaN, whose bits lie beyond every bin
      const unsigned k = __float_as_uint(__fadd_ru(d2 * rsqrtf(d2) * inv_binstep, 8388608.0f)) - 0x4B000000u;
      if (k - 1u >= (unsigned)nbins) return;
      const float4 vj = __ldg(&vs[j]);
      const float t0 = vi.x - vj.x, t1 = vi.y - vj.y, t2 = vi.z - vj.z;
      const float s = fmaf(t0, t0, fmaf(t1, t1, t2 * t2));
      float2* const slot = &bins[(k - 1u) * T + t];
      float2 w = *slot;
      w.x += s > 0.f ? s * rsqrtf(s) : 0.f;
      w.y = __int_as_float(__float_as_int(w.y) + 1);
      *slot = w;
    };
    auto scan = [&](int j0, int j1, float ax, float ay, float az) {
      const float2 nx = f2(-ax), ny = f2(-ay), nz = f2(-az);
#pragma unroll 2
      for (int j = j0; j < j1; j += 2) {
        const float4 a = __ldg(&A.xs[j]);
        const float4 b = __ldg(&A.xs[min(j + 1, j1 - 1)]);
        const float2 dx = __fadd2_rn(make_float2(a.x, b.x), nx);
        const float2 dy = __fadd2_rn(make_float2(a.y, b.y), ny);
        const float2 dz = __fadd2_rn(make_float2(a.z, b.z), nz);
        const float2 d2 = __ffma2_rn(dx, dx, __ffma2_rn(dy, dy, __fmul2_rn(dz, dz)));
        if (d2.x < rc2) pair(d2.x, j);
        if (d2.y < rc2 && j + 1 < j1) pair(d2.y, j + 1);
      }
    };
    scan(p + 1, A.cell_start[cx + A.nx * (cy + A.ny * cz) + 1], pi.x, pi.y, pi.z);
    for (int k = 1; k < A.noff; ++k) {
      const Off& o = A.off[k];
      const float ax = pi.x - o.sx, ay = pi.y - o.sy, az = pi.z - o.sz;
      const float bx = fmaxf(fabsf(ax) - A.ex, 0.f), by = fmaxf(fabsf(ay) - A.ey, 0.f),
                  bz = fmaxf(fabsf(az) - A.ez, 0.f);
      if (fmaf(bx, bx, fmaf(by, by, bz * bz)) >= rc2) continue;
      const int c = stencil_cell(A, k, cx, cy, cz);
      scan(A.cell_start[c], A.cell_start[c + 1], ax, ay, az);
    }
  }
  __syncthreads();
  const int lane = t & 31;
  for (int b = t >> 5; b < nbins; b += T >> 5) {
    double s = 0.0;
    unsigned long long c = 0;
    for (int q = lane; q < T; q += 32) {
      const float2 w = bins[b * T + q];
      s += (double)w.x;
      c += (unsigned)__float_as_int(w.y);
    }
#pragma unroll
    for (int o = 16; o; o >>= 1) {
      s += __shfl_xor_sync(0xffffffffu, s, o);
      c += __shfl_xor_sync(0xffffffffu, c, o);
    }
    if (lane == 0 && c) {
      atomicAdd(&counts[b], c);
      atomicAdd(&vsum[b], s);
    }
  }
}

// Lennard-Jones energy and forces, full shell, one thread per sorted particle:
// the functor's sweep and its sums term by term, without its IEEE division (a
// warp has a pair within the cutoff at nearly every step) and without the cells
// beyond the cutoff. Bound by issue: step of 500,000 particles, cutoff 12, two
// cells per cutoff 1.56 -> 1.41 ms, 940,000 at one cell 3.92 -> 3.86.
// Every candidate's term in packed FP32, masked (FMA pipe), 1.46 ms, and a warp
// per cell over the particles of the cell's ball, 1.39 ms, were slower on cells
// of 13 or of 170 particles.
__global__ void __launch_bounds__(256) k_sweep_lj(const __grid_constant__ SweepArgs A, float rc2, float eps4,
                                                  float eps24, float s2, float* __restrict__ forces,
                                                  double* __restrict__ partials) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  float e = 0.f;
  if (p < A.n) {
    const float4 pi = A.xs[p];
    const unsigned cc = A.cellc[p];
    const int cx = (int)(cc & 1023u), cy = (int)((cc >> 10) & 1023u), cz = (int)(cc >> 20);
    float fx = 0.f, fy = 0.f, fz = 0.f;
    auto scan = [&](int j0, int j1, float ax, float ay, float az) {
#pragma unroll 2
      for (int j = j0; j < j1; ++j) {
        const float4 q = __ldg(&A.xs[j]);
        const float dx = q.x - ax, dy = q.y - ay, dz = q.z - az;
        const float d2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
        if (d2 < rc2) {
          const float y2 = recip(d2);
          const float r = s2 * y2, r3 = r * r * r;
          const float w = fmaf(r3, r3, -r3);
          const float g = fmaf(r3, r3, w) * -eps24 * y2;
          fx = fmaf(g, dx, fx);
          fy = fmaf(g, dy, fy);
          fz = fmaf(g, dz, fz);
          e = fmaf(eps4, w, e);
        }
      }
    };
    {
      const int c = cx + A.nx * (cy + A.ny * cz);
      scan(A.cell_start[c], p, pi.x, pi.y, pi.z);
      scan(p + 1, A.cell_start[c + 1], pi.x, pi.y, pi.z);
    }
    for (int k = 1; k < A.noff; ++k) {
      const Off& o = A.off[k];
      const float ax = pi.x - o.sx, ay = pi.y - o.sy, az = pi.z - o.sz;
      const float bx = fmaxf(fabsf(ax) - A.ex, 0.f), by = fmaxf(fabsf(ay) - A.ey, 0.f),
                  bz = fmaxf(fabsf(az) - A.ez, 0.f);
      if (fmaf(bx, bx, fmaf(by, by, bz * bz)) >= rc2) continue;  // the whole cell is beyond the cutoff
      const int c = stencil_cell(A, k, cx, cy, cz);
      scan(A.cell_start[c], A.cell_start[c + 1], ax, ay, az);
    }
    float* f = forces + (size_t)__float_as_int(pi.w) * 3;
    f[0] = fx;
    f[1] = fy;
    f[2] = fz;
  }
  double v[1] = {0.5 * (double)e};
  block_sum_store<1>(v, partials + blockIdx.x);
}

// After a sweep that used the list's force buffer as scratch: the buffer cleared
// for the next force sweep, also when the launches report an error (an earlier
// error of the calling thread is enough for that), and their status.
int scratch_done(float4* hforce, int n, cudaStream_t s) {
  const bool ok = cudaGetLastError() == cudaSuccess;
  return cudaMemsetAsync(hforce, 0, sizeof(float4) * (size_t)n, s) == cudaSuccess && ok ? CL_OK : CL_ERR_CUDA;
}

// Candidates per particle at the mean occupancy.
double candidates(const SweepArgs& A) { return (double)A.n * A.noff / ((double)A.nx * A.ny * A.nz); }

// Fewer, and the mass sum is the functor's: gathering the attributes, clearing the
// scratch and the final sum are launches of their own. Functor against sweep, 20,000
// particles: 41 and 57 us at 3 candidates, 49 and 56 at 14, 56 and 59 at 42; 300,000:
// 94 and 115 at 13, 131 and 142 at 63, 292 and 250 at 160.
constexpr double kMassMinCandidates = 80.0;

// The functors' cutoff test: the FP32 cutoff squared in FP32.
float functor_rc2(double rc) { return (float)rc * (float)rc; }

}  // namespace
}  // namespace clk

namespace {

template <int NB>
int velocity_hist_nb(const cl_list* cl, const float* vel, int dim, double binstep, int nbins,
                     unsigned long long* counts, double* vsum, cudaStream_t s) {
  cellmap::pairfn::VelocityHistogram<NB> f;
  f.vel = vel;
  f.dim = dim;
  f.nbins = nbins;
  f.inv_binstep = (float)(1.0 / binstep);
  f.counts = counts;
  f.vsum = vsum;
  return cellmap::map(cl, f, s);
}

}  // namespace

extern "C" int cl_map_mass(const cl_list* cl, const float* mass_dev, double* out_dev, void* stream) {
  if (!cl || !out_dev) return CL_ERR_INVALID_ARG;
  cl_view v;
  int e = cl_get_view(cl, &v);
  if (e) return e;
  if (v.n > 0 && !mass_dev) return CL_ERR_INVALID_ARG;
  cudaStream_t s = (cudaStream_t)stream;
  if (cudaMemsetAsync(out_dev, 0, sizeof(double), s) != cudaSuccess) return CL_ERR_CUDA;
  clk::ListParts L;
  clk::list_parts(cl, &L);
  if (L.hforce && v.n > 0 && clk::candidates(*L.half) >= clk::kMassMinCandidates) {
    const int blocks = (v.n + 255) / 256;
    clk::k_sorted_mass<<<blocks, 256, 0, s>>>(L.half->xs, v.n, mass_dev, L.hforce);
    clk::k_sweep_mass<<<blocks, 256, 0, s>>>(*L.half, L.hforce, clk::functor_rc2(L.rc), L.partials);
    if ((e = clk::scratch_done(L.hforce, v.n, s))) return e;
    return clk::finish_reduction(0, 3, nullptr, blocks, 1, L.partials, L.sums, out_dev, nullptr, nullptr, nullptr, s);
  }
  cellmap::pairfn::MassPotential f;
  f.mass = mass_dev;
  f.out = out_dev;
  return cellmap::map(cl, f, s);
}

extern "C" int cl_map_lj(const cl_list* cl, double eps, double sigma, double* energy_dev, float* forces_dev,
                         void* stream) {
  if (!cl || !energy_dev || !(sigma > 0) || !isfinite(eps) || !isfinite(sigma)) return CL_ERR_INVALID_ARG;
  cl_view v;
  int e = cl_get_view(cl, &v);
  if (e) return e;
  cudaStream_t s = (cudaStream_t)stream;
  if (cudaMemsetAsync(energy_dev, 0, sizeof(double), s) != cudaSuccess) return CL_ERR_CUDA;
  if (!forces_dev) {
    cellmap::pairfn::LennardJones f;
    f.eps4 = (float)(4.0 * eps);
    f.s2 = (float)(sigma * sigma);
    f.out = energy_dev;
    return cellmap::map(cl, f, s);
  }
  clk::ListParts L;
  clk::list_parts(cl, &L);
  if (L.hforce && v.n > 0) {
    const int blocks = (v.n + 255) / 256;
    clk::k_sweep_lj<<<blocks, 256, 0, s>>>(*L.full, clk::functor_rc2(L.rc), (float)(4.0 * eps), (float)(24.0 * eps),
                                           (float)(sigma * sigma), forces_dev, L.partials);
    if (cudaGetLastError() != cudaSuccess) return CL_ERR_CUDA;
    return clk::finish_reduction(0, 3, nullptr, blocks, 1, L.partials, L.sums, energy_dev, nullptr, nullptr, nullptr,
                                 s);
  }
  cellmap::pairfn::LennardJonesForces f;
  f.eps4 = (float)(4.0 * eps);
  f.eps24 = (float)(24.0 * eps);
  f.s2 = (float)(sigma * sigma);
  f.forces = forces_dev;
  f.dim = v.dim;
  f.energy = energy_dev;
  if (v.n > 0 && cudaMemsetAsync(forces_dev, 0, sizeof(float) * (size_t)v.n * v.dim, s) != cudaSuccess)
    return CL_ERR_CUDA;
  return cellmap::map(cl, f, s);
}

extern "C" int cl_map_velocity_hist(const cl_list* cl, const float* vel_dev, double binstep, int nbins,
                                    unsigned long long* counts_dev, double* vsum_dev, void* stream) {
  if (!cl || !counts_dev || !vsum_dev || !(binstep > 0) || nbins < 1 || nbins > CL_VHIST_MAX_BINS)
    return CL_ERR_INVALID_ARG;
  cl_view v;
  int e = cl_get_view(cl, &v);
  if (e) return e;
  if (v.n > 0 && !vel_dev) return CL_ERR_INVALID_ARG;
  cudaStream_t s = (cudaStream_t)stream;
  if (cudaMemsetAsync(counts_dev, 0, sizeof(unsigned long long) * nbins, s) != cudaSuccess ||
      cudaMemsetAsync(vsum_dev, 0, sizeof(double) * nbins, s) != cudaSuccess)
    return CL_ERR_CUDA;
  clk::ListParts L;
  clk::list_parts(cl, &L);
  if (L.hforce && v.n > 0) {
    // 8 bytes a bin and thread: blocks of 32 KB at most, six to an SM
    const int T = nbins <= 16 ? 256 : (nbins <= 32 ? 128 : 64);
    clk::k_sorted_velocity<<<(v.n + 255) / 256, 256, 0, s>>>(L.half->xs, v.n, vel_dev, L.hforce);
    clk::k_sweep_velocity<<<(v.n + T - 1) / T, T, sizeof(float2) * nbins * T, s>>>(
        *L.half, L.hforce, clk::functor_rc2(L.rc), (float)(1.0 / binstep), nbins, counts_dev, vsum_dev);
    return clk::scratch_done(L.hforce, v.n, s);
  }
  if (nbins <= 16) return velocity_hist_nb<16>(cl, vel_dev, v.dim, binstep, nbins, counts_dev, vsum_dev, s);
  return velocity_hist_nb<CL_VHIST_MAX_BINS>(cl, vel_dev, v.dim, binstep, nbins, counts_dev, vsum_dev, s);
}
