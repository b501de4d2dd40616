// cl_cross.cu -- pairs between two sets of particles (Sec. 3.2, Code 8: a cell
// list of x and a second set y; Sec. 4.1: neighbour lists between two sets).
// The cell list is the one of set A (cl_build); every particle b of set B is
// binned on A's grid (FP64 wrap and cell, FP32 coordinate relative to the cell
// centre) and sweeps the FULL stencil of its cell, the displacement to a being
// (xs_a + S_o) - x_b as in the one-set sweep. Every (a, b) pair-image within
// the cutoff is visited once; there is no a < b rule.
//
//   k_query_bin      cell and local coordinate of each query point
//   (cell order)     the queries counting-sorted by cell, when they are many
//   k_cross_count    per-b counts (and their sum), one warp per query
//   k_cross_fill     (a, b, r) of b's segment of the list, sorted by a
//   k_cross_knn      per b the k nearest a within the cutoff (k <= 32)
//   k_topk_part, k_topk_last  the k smallest over all per-b lists
//
// A warp takes one query: its lanes test the stencil's cells 32 at a time
// (the cell's bounding box against the cutoff, as in sweep_particle2), the
// kept ones are compacted in shared memory, and groups of G lanes run over
// them, G chosen by the mean occupancy so that a group's passes are mostly
// full. One thread per query in input order, the form before this one, was
// bound by its serial chain of uncoalesced loads and wrote each segment with
// one lane's stores.
#include <algorithm>
#include <cfloat>
#include <climits>
#include <cmath>

#include "cl_query.cuh"
#include "cl_sort.cuh"

namespace clk {
namespace {

constexpr int kKnnMax = CL_KNN_MAX;
constexpr int kCrossWarps = 8;
constexpr int kFillWarps = 4;  // 8.4 KB of segment per warp: five CTAs of four warps fit an SM, two of eight

struct QueryArgs {
  const double* pos;  // (nb, dim) FP64
  long long nb;
  int nx, ny, nz;
  double m[9];        // t = x M (cell units)
  float g[9];         // cell edge vectors (rows)
};

// Packed cell and centred FP32 coordinate of every query point; a point that
// is not finite is parked in cell 0 at its sentinel position, where every
// distance test against it fails. With counts the point also takes its slot
// in its cell (q then holds the packed cell in w, for the reordering).
template <int DIM, bool ORTHO>
__global__ void __launch_bounds__(256) k_query_bin(const __grid_constant__ QueryArgs Q, float4* __restrict__ q,
                                                   unsigned* __restrict__ cell, int* __restrict__ counts,
                                                   int* __restrict__ slot, int* __restrict__ err) {
  const long long b = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (b >= Q.nb) return;
  double x[DIM];
  bool finite = true;
#pragma unroll
  for (int k = 0; k < DIM; ++k) {
    x[k] = Q.pos[b * DIM + k];
    finite = finite && isfinite(x[k]);
  }
  const int nk[3] = {Q.nx, Q.ny, Q.nz};
  int c[3] = {0, 0, 0};
  float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
  if (finite) {
    float u[DIM];
#pragma unroll
    for (int k = 0; k < DIM; ++k) {
      double t;
      if (ORTHO) {
        t = x[k] * Q.m[k * 3 + k];
      } else {
        t = 0.0;
#pragma unroll
        for (int p = 0; p < DIM; ++p) t = fma(x[p], Q.m[p * 3 + k], t);
      }
      const double f = floor(t);
      long long ci = (long long)f;
      if (ci < 0 || ci >= nk[k]) {
        ci %= nk[k];
        if (ci < 0) ci += nk[k];
      }
      c[k] = (int)ci;
      u[k] = (float)(t - f) - 0.5f;
    }
#pragma unroll
    for (int k = 0; k < DIM; ++k) {
      o.x = fmaf(u[k], Q.g[k * 3 + 0], o.x);
      o.y = fmaf(u[k], Q.g[k * 3 + 1], o.y);
      o.z = fmaf(u[k], Q.g[k * 3 + 2], o.z);
    }
  } else {
    o = sentinel_pos((int)b);
    atomicOr(err, kErrNonFinite);
  }
  const unsigned pc = (unsigned)c[0] | ((unsigned)c[1] << 10) | ((unsigned)c[2] << 20);
  if (counts) {
    o.w = __uint_as_float(pc);
    slot[b] = atomicAdd(&counts[c[0] + Q.nx * (c[1] + Q.ny * c[2])], 1);
  } else {
    o.w = __int_as_float((int)b);
    cell[b] = pc;
  }
  q[b] = o;
}

template <int G>
__global__ void __launch_bounds__(32 * kCrossWarps) k_cross_count(const __grid_constant__ CrossArgs A,
                                                                  const Queries Q, int* __restrict__ count,
                                                                  unsigned long long* __restrict__ total) {
  extern __shared__ float4 stab[];
  __shared__ WarpCells cells[kCrossWarps];
  load_stencil<false>(A, stab, nullptr);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  WarpCells& W = cells[warp];
  unsigned long long sum = 0;
  for (long long b = blockIdx.x * (long long)kCrossWarps + warp; b < Q.nb; b += (long long)gridDim.x * kCrossWarps) {
    const float4 p = Q.q[b];
    const unsigned cc = Q.cell[b];
    unsigned n = query_count<G>(A, stab, W, cc, p, -1);
    n = __reduce_add_sync(0xffffffffu, n);
    if (count && lane == 0) count[__float_as_int(p.w)] = (int)n;
    sum += n;
  }
  if (total && lane == 0 && sum) atomicAdd(total, sum);
}

// The kept pairs of a query are compacted into the warp's shared-memory
// segment and sorted by a. WIDE false (set A has fewer than 2^22 particles):
// the key is a << 10 | slot, one word, and the distances stay in place; WIDE:
// (a, distance) pairs. A segment longer than kMaxSegment is written unsorted
// and listed in longs.
template <int G, bool WIDE>
__global__ void __launch_bounds__(32 * kFillWarps, 5) k_cross_fill(const __grid_constant__ CrossArgs A,
                                                                    const Queries Q, const int* __restrict__ count,
                                                                    const long long* __restrict__ start,
                                                                    int* __restrict__ pa, int* __restrict__ pb,
                                                                    float* __restrict__ pd, int* __restrict__ longs,
                                                                    int* __restrict__ nlong) {
  extern __shared__ float4 stab[];
  __shared__ WarpCells cells[kFillWarps];
  float* seg = reinterpret_cast<float*>(stab + A.noff);
  load_stencil<false>(A, stab, nullptr);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  WarpCells& W = cells[warp];
  float* V = seg + (size_t)warp * 2 * kSegPad;
  unsigned* K = reinterpret_cast<unsigned*>(V + kSegPad);
  for (long long t = blockIdx.x * (long long)kFillWarps + warp; t < Q.nb; t += (long long)gridDim.x * kFillWarps) {
    const float4 p = Q.q[t];
    const unsigned cc = Q.cell[t];
    const int b = __float_as_int(p.w);
    const int cnt = __ldg(count + b);
    if (cnt == 0) continue;
    const long long base = __ldg(start + b);
    const bool big = cnt > kMaxSegment;
    const int L = query_hits<G>(A, stab, W, cc, p, -1, [&](int e, int a, float d2) {
      if (e >= cnt) return;
      if (big) {
        pa[base + e] = a;
        pb[base + e] = b;
        pd[base + e] = sqrtf(d2);
      } else {
        K[seg_at(e)] = WIDE ? (unsigned)a : ((unsigned)a << 10) | (unsigned)e;
        V[seg_at(e)] = d2;
      }
    });
    __syncwarp();
    if (big) {
      if (lane == 0) longs[atomicAdd(nlong, 1)] = b;
      continue;
    }
    const int nw = min(L, cnt);
    if (WIDE) sort_segment(reinterpret_cast<int*>(K), V, nw, lane);
    else sort_keys(K, nw, lane);
    for (int i = lane; i < nw; i += 32) {
      const unsigned key = K[seg_at(i)];
      pa[base + i] = WIDE ? (int)key : (int)(key >> 10);
      pb[base + i] = b;
      pd[base + i] = sqrtf(V[WIDE ? seg_at(i) : seg_at((int)(key & 1023u))]);
    }
    __syncwarp();
  }
}

template <class ID>
__device__ __forceinline__ bool nearer(float d, ID i, float e, ID j) {
  return d < e || (d == e && i < j);
}

// One compare-exchange of a lane with its partner, `up` when it keeps the nearer.
template <class ID>
__device__ __forceinline__ void nearer_exchange(float& d, ID& i, int mask, bool up) {
  const float e = __shfl_xor_sync(0xffffffffu, d, mask);
  const ID j = __shfl_xor_sync(0xffffffffu, i, mask);
  const bool take = nearer(e, j, d, i) == up && !(e == d && j == i);
  d = take ? e : d;
  i = take ? j : i;
}

// A warp's running best k of (distance, id), ascending, entry l in lane l
// (the lanes past k hold what was pushed out): offers the lanes' candidates
// (ok ones) and keeps the k smallest. A few candidates are inserted one by
// one; more than kBulk, as in the first steps, when nearly every lane has one,
// are sorted across the warp and merged with the list at once (25 against 190
// instructions: 8 nearest and 5 closest of 60,000 queries 449 -> 418 us).
constexpr int kBulk = 6;

template <class ID>
__device__ __forceinline__ void best_offer(float& bd, ID& bi, float& kd, ID& ki, int k, bool ok, float d, ID id,
                                           float none_d, ID none_i) {
  const int lane = threadIdx.x & 31;
  ok = ok && nearer(d, id, kd, ki);
  unsigned m = __ballot_sync(0xffffffffu, ok);
  // The nearest alone: two warp minima. Sorting and merging lost to the one thread
  // per query that came before (100,000 queries in 2D, 28 candidates each, against a
  // million particles: 79 us then, 131 so, 84 now).
  if (k == 1 && __popc(m) > 1) {
    d = ok ? d : none_d;
    id = ok ? id : none_i;
    if (sizeof(ID) == 4) {  // squared distances are not negative: their bits order like them
      const unsigned b = __reduce_min_sync(0xffffffffu, __float_as_uint(d));
      id = __reduce_min_sync(0xffffffffu, __float_as_uint(d) == b ? (int)id : INT_MAX);
      d = __uint_as_float(b);
    } else {
#pragma unroll
      for (int st = 16; st > 0; st >>= 1) nearer_exchange(d, id, st, true);
    }
    kd = bd = d;
    ki = bi = id;
    return;
  }
  if (__popc(m) > kBulk) {
    d = ok ? d : none_d;
    id = ok ? id : none_i;
#pragma unroll
    for (int size = 2; size <= 32; size <<= 1)
#pragma unroll
      for (int st = size >> 1; st > 0; st >>= 1)
        nearer_exchange(d, id, st, ((lane & st) == 0) == ((lane & size) == 0 || size == 32));
    // the 32 nearest of both lists: entry l against the other's 31 - l, a
    // bitonic sequence, merged in five steps
    const float rd = __shfl_sync(0xffffffffu, d, 31 - lane);
    const ID ri = __shfl_sync(0xffffffffu, id, 31 - lane);
    const bool take = nearer(rd, ri, bd, bi);
    bd = take ? rd : bd;
    bi = take ? ri : bi;
#pragma unroll
    for (int st = 16; st > 0; st >>= 1) nearer_exchange(bd, bi, st, (lane & st) == 0);
    kd = __shfl_sync(0xffffffffu, bd, k - 1);
    ki = __shfl_sync(0xffffffffu, bi, k - 1);
    return;
  }
  while (m) {
    const int src = __ffs(m) - 1;
    m &= m - 1;
    const float cd = __shfl_sync(0xffffffffu, d, src);
    const ID ci = __shfl_sync(0xffffffffu, id, src);
    if (!nearer(cd, ci, kd, ki)) continue;  // uniform: a better one came in since
    const bool before = lane < k && !nearer(cd, ci, bd, bi);
    const int at = __popc(__ballot_sync(0xffffffffu, before));
    const float ud = __shfl_up_sync(0xffffffffu, bd, 1);
    const ID ui = __shfl_up_sync(0xffffffffu, bi, 1);
    if (lane > at) {
      bd = ud;
      bi = ui;
    } else if (lane == at) {
      bd = cd;
      bi = ci;
    }
    kd = __shfl_sync(0xffffffffu, bd, k - 1);
    ki = __shfl_sync(0xffffffffu, bi, k - 1);
  }
}

// Per query b: the k nearest a within the cutoff, ascending by distance (ties:
// smaller a first); empty slots hold a = -1, r = +inf. The stencil's cells are
// visited nearest first and a cell beyond the k-th distance found so far is
// skipped, so a query tests the particles of about the ball of its k-th
// neighbour and not of the cutoff's.
template <int G>
__global__ void __launch_bounds__(32 * kCrossWarps) k_cross_knn(const __grid_constant__ CrossArgs A, const Queries Q,
                                                                int k, int* __restrict__ out_a,
                                                                float* __restrict__ out_d) {
  extern __shared__ float4 stab[];
  __shared__ WarpCells cells[kCrossWarps];
  load_stencil<true>(A, stab, reinterpret_cast<float*>(stab + A.noff));
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  WarpCells& W = cells[warp];
  for (long long t = blockIdx.x * (long long)kCrossWarps + warp; t < Q.nb; t += (long long)gridDim.x * kCrossWarps) {
    const float4 p = Q.q[t];
    const unsigned cc = Q.cell[t];
    float bd = FLT_MAX, kd = FLT_MAX;
    int ba = INT_MAX, ka = INT_MAX;
    for (int k0 = 0; k0 < A.noff; k0 += 32) {
      const int nk = query_cells(A, stab, W, k0, lane, cc, p, fminf(A.rc2, kd));
      for (int i0 = 0; i0 < nk; i0 += 32 / G) {
        const int i = i0 + lane / G;
        float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
        int j = 0, j1 = 0;
        if (i < nk) {
          s = W.s[i];
          const int2 r = W.j[i];
          j = r.x + lane % G;
          j1 = s.w < kd ? r.y : 0;
        }
        while (__any_sync(0xffffffffu, j < j1)) {
          int a = 0;
          float d2 = FLT_MAX;
          if (j < j1) {
            const float4 q = __ldg(&A.xs[j]);
            a = __float_as_int(q.w);
            d2 = query_d2(q, s);
          }
          j += G;
          best_offer(bd, ba, kd, ka, k, d2 < A.rc2, d2, a, FLT_MAX, INT_MAX);
        }
      }
    }
    if (lane < k) {
      const long long o = (long long)__float_as_int(p.w) * k + lane;
      const bool have = bd < FLT_MAX;
      out_a[o] = have ? ba : -1;
      out_d[o] = have ? sqrtf(bd) : INFINITY;
    }
  }
}

// The k smallest (r, id), id = b * k + q, over nb per-query lists of k: each
// warp keeps the best of its share, the last kernel the best of theirs. (One
// CTA sorting 1,024 candidates at a time took 5.0 ms for 60,000 lists of 5.)
constexpr int kTopkWarps = 8;

__global__ void __launch_bounds__(32 * kTopkWarps) k_topk_part(const int* __restrict__ la, const float* __restrict__ ld,
                                                               long long total, long long share, int k,
                                                               float* __restrict__ part_d,
                                                               long long* __restrict__ part_id) {
  const int lane = threadIdx.x & 31;
  const long long w = blockIdx.x * (long long)kTopkWarps + (threadIdx.x >> 5);
  const long long e1 = min(total, (w + 1) * share);
  float bd = INFINITY, kd = INFINITY;
  long long bi = LLONG_MAX, ki = LLONG_MAX;
  for (long long e0 = w * share; e0 < e1; e0 += 32) {
    const long long e = e0 + lane;
    const bool ok = e < e1 && la[e] >= 0;
    best_offer(bd, bi, kd, ki, k, ok, ok ? ld[e] : INFINITY, e, INFINITY, LLONG_MAX);
  }
  if (lane < k) {
    part_d[w * k + lane] = bd;
    part_id[w * k + lane] = bi;
  }
}

__global__ void __launch_bounds__(1024) k_topk_last(const int* __restrict__ la, const float* __restrict__ part_d,
                                                    const long long* __restrict__ part_id, long long m, int k,
                                                    int* __restrict__ oa, int* __restrict__ ob, float* __restrict__ od,
                                                    int* __restrict__ found) {
  __shared__ float sd[32 * kKnnMax];
  __shared__ long long sid[32 * kKnnMax];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float bd = INFINITY, kd = INFINITY;
  long long bi = LLONG_MAX, ki = LLONG_MAX;
  for (long long e0 = warp * 32LL; e0 < m; e0 += 1024) {
    const long long e = e0 + lane;
    const long long id = e < m ? part_id[e] : LLONG_MAX;
    best_offer(bd, bi, kd, ki, k, id != LLONG_MAX, e < m ? part_d[e] : INFINITY, id, INFINITY, LLONG_MAX);
  }
  if (lane < k) {
    sd[warp * k + lane] = bd;
    sid[warp * k + lane] = bi;
  }
  __syncthreads();
  if (warp) return;
  bd = kd = INFINITY;
  bi = ki = LLONG_MAX;
  for (int e = lane; e < 32 * k; e += 32)
    best_offer(bd, bi, kd, ki, k, sid[e] != LLONG_MAX, sd[e], sid[e], INFINITY, LLONG_MAX);
  const bool ok = lane < k && bi != LLONG_MAX;
  if (lane < k) {
    oa[lane] = ok ? la[bi] : -1;
    ob[lane] = ok ? (int)(bi / k) : -1;
    od[lane] = ok ? bd : INFINITY;
  }
  const unsigned have = __ballot_sync(0xffffffffu, ok);
  if (lane == 0) *found = __popc(have);
}

// CTAs of one wave of the kernel for nb queries. The kernel's shared-memory limit
// is raised once per device, to what its largest stencil takes: a limit set to
// each call's own size could be lowered by another thread's smaller grid between
// this call's set and its launch, which then failed. ready: the kernel's own.
template <class K>
int cross_grid(K kernel, DevCache& ready, int warps, size_t most, size_t smem, long long nb) {
  int dev = 0, sms = 0, per = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return 0;
  if (!ready.get(dev)) {
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most) != cudaSuccess) return 0;
    ready.put(dev, 1);
  }
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kernel, 32 * warps, smem) != cudaSuccess || per < 1)
    return 0;
  const long long want = (nb + warps - 1) / warps;
  return (int)(want < (long long)sms * per ? want : (long long)sms * per);
}

constexpr size_t count_smem(int noff) { return (size_t)noff * sizeof(float4); }
constexpr size_t fill_smem(int noff) {
  return (size_t)noff * sizeof(float4) + (size_t)kFillWarps * 2 * kSegPad * sizeof(float);
}
constexpr size_t knn_smem(int noff) { return (size_t)noff * (sizeof(float4) + sizeof(float)); }

template <int G>
int run_count(const CrossArgs& C, const Queries& Q, int* count, unsigned long long* total, cudaStream_t s) {
  static DevCache ready;
  const size_t smem = count_smem(C.noff);
  const int grid = cross_grid(k_cross_count<G>, ready, kCrossWarps, count_smem(kMaxOff), smem, Q.nb);
  if (grid < 1) return CL_ERR_CUDA;
  k_cross_count<G><<<grid, 32 * kCrossWarps, smem, s>>>(C, Q, count, total);
  return cudaGetLastError() == cudaSuccess ? CL_OK : CL_ERR_CUDA;
}

template <int G, bool WIDE>
int run_fill(const CrossArgs& C, const Queries& Q, const int* count, const long long* start, int* pa, int* pb,
             float* pd, int* longs, int* nlong, cudaStream_t s) {
  static DevCache ready;
  const size_t smem = fill_smem(C.noff);
  const int grid = cross_grid(k_cross_fill<G, WIDE>, ready, kFillWarps, fill_smem(kMaxOff), smem, Q.nb);
  if (grid < 1) return CL_ERR_CUDA;
  k_cross_fill<G, WIDE><<<grid, 32 * kFillWarps, smem, s>>>(C, Q, count, start, pa, pb, pd, longs, nlong);
  return cudaGetLastError() == cudaSuccess ? CL_OK : CL_ERR_CUDA;
}

template <int G>
int run_knn(const CrossArgs& C, const Queries& Q, int k, int* out_a, float* out_d, cudaStream_t s) {
  static DevCache ready;
  const size_t smem = knn_smem(C.noff);
  const int grid = cross_grid(k_cross_knn<G>, ready, kCrossWarps, knn_smem(kMaxOff), smem, Q.nb);
  if (grid < 1) return CL_ERR_CUDA;
  k_cross_knn<G><<<grid, 32 * kCrossWarps, smem, s>>>(C, Q, k, out_a, out_d);
  return cudaGetLastError() == cudaSuccess ? CL_OK : CL_ERR_CUDA;
}

}  // namespace

// Queries are sorted by cell, in five more launches and a pass over the cell
// counts, when set A's coordinates (16 B each) pass most of the L2, so that
// neighbouring warps share what they read from DRAM, and the queries are at least
// a quarter as many as the cells. Sorted against in input order, random queries:
// 8M particles, 200,000 queries count 657 against 778 us, list 10.3 / 10.9 ms;
// 1M queries list 8.8 / 10.3 ms. Of a set in L2: 1M, 100,000 queries count 371 /
// 348 us, list 1,965 / 1,909, nearest 307 / 296; 1M, 21,000 list 595 / 539; 2D 4M,
// 1M queries list 1,887 / 1,837.
bool queries_sorted(long long n, long long nb, long long ncells) {
  return n >= (6 << 20) && nb >= 2048 && nb * 4 >= ncells;
}

int launch_query_bin(const SweepArgs& A, const Geo& g, const double* posb, long long nb, const QueryBufs& b, int* err,
                     Queries* out, cudaStream_t s) {
  out->q = b.q;
  out->cell = b.cell;
  out->nb = nb;
  if (nb <= 0) return CL_OK;
  QueryArgs Q;
  Q.pos = posb;
  Q.nb = nb;
  Q.nx = A.nx;
  Q.ny = A.ny;
  Q.nz = A.nz;
  for (int q = 0; q < 9; ++q) {
    Q.m[q] = g.m[q];
    Q.g[q] = g.g[q];
  }
  const bool sorted = queries_sorted(A.n, nb, g.ncells);
  int* counts = sorted ? b.counts : nullptr;
  if (sorted && (cudaMemsetAsync(b.counts, 0, sizeof(int) * g.ncells, s) != cudaSuccess ||
                 cudaMemsetAsync(b.meta, 0, sizeof(int) * 4, s) != cudaSuccess))
    return CL_ERR_CUDA;
  const unsigned blocks = (unsigned)((nb + 255) / 256);
  float4* q = sorted ? b.raw : b.q;
  if (g.dim == 3) {
    if (g.ortho) k_query_bin<3, true><<<blocks, 256, 0, s>>>(Q, q, b.cell, counts, b.slot, err);
    else k_query_bin<3, false><<<blocks, 256, 0, s>>>(Q, q, b.cell, counts, b.slot, err);
  } else {
    if (g.ortho) k_query_bin<2, true><<<blocks, 256, 0, s>>>(Q, q, b.cell, counts, b.slot, err);
    else k_query_bin<2, false><<<blocks, 256, 0, s>>>(Q, q, b.cell, counts, b.slot, err);
  }
  if (cudaGetLastError() != cudaSuccess) return CL_ERR_CUDA;
  if (!sorted) return CL_OK;
  const int e = launch_scan_cells(b.counts, g.ncells, b.tiles, b.meta, b.start, s);
  return e ? e : launch_cell_order((int)nb, A.nx, A.ny, g.ncells, b.slot, b.raw, b.start, b.q, b.cell, s);
}

int launch_cross_count(const SweepArgs& A, const Off* off, const Queries& Q, int* count, unsigned long long* total,
                       cudaStream_t s) {
  if (Q.nb <= 0) return CL_OK;
  const CrossArgs C = cross_args(A, off);
  switch (group_lanes(A)) {
    case 2: return run_count<2>(C, Q, count, total, s);
    case 4: return run_count<4>(C, Q, count, total, s);
    default: return run_count<8>(C, Q, count, total, s);
  }
}

int launch_cross_fill(const SweepArgs& A, const Off* off, const Queries& Q, const int* count, const long long* start,
                      int* pa, int* pb, float* pd, int* longs, int* nlong, cudaStream_t s) {
  if (Q.nb <= 0) return CL_OK;
  if (cudaMemsetAsync(nlong, 0, sizeof(int), s) != cudaSuccess) return CL_ERR_CUDA;
  const CrossArgs C = cross_args(A, off);
  int e;
  if (A.n >= (1 << 22)) {
    e = run_fill<8, true>(C, Q, count, start, pa, pb, pd, longs, nlong, s);
  } else {
    switch (group_lanes(A)) {
      case 2: e = run_fill<2, false>(C, Q, count, start, pa, pb, pd, longs, nlong, s); break;
      case 4: e = run_fill<4, false>(C, Q, count, start, pa, pb, pd, longs, nlong, s); break;
      default: e = run_fill<8, false>(C, Q, count, start, pa, pb, pd, longs, nlong, s); break;
    }
  }
  return e ? e : launch_sort_long(longs, nlong, count, start, pa, pd, s);
}

int launch_cross_knn(const SweepArgs& A, const Off* off, const Queries& Q, int k, int* out_a, float* out_d,
                     cudaStream_t s) {
  if (Q.nb <= 0) return CL_OK;
  const CrossArgs C = cross_args(A, off);
  switch (group_lanes(A)) {
    case 2: return run_knn<2>(C, Q, k, out_a, out_d, s);
    case 4: return run_knn<4>(C, Q, k, out_a, out_d, s);
    default: return run_knn<8>(C, Q, k, out_a, out_d, s);
  }
}

// A warp's share is at least 256 candidates (its first ones all enter its list,
// one at a time), and at most 1,216 warps, one wave, share the lists.
static long long topk_share(long long nb, int k) {
  const long long total = nb * k;
  const long long share = (total + 1215) / 1216;
  return (std::max<long long>(share, 256) + 31) / 32 * 32;
}

long long topk_parts(long long nb, int k) {
  const long long share = topk_share(nb, k), w = (nb * k + share - 1) / share;
  return (std::max<long long>(w, 1) + kTopkWarps - 1) / kTopkWarps * kTopkWarps;
}

int launch_topk_merge(const int* la, const float* ld, long long nb, int k, float* part_d, long long* part_id, int* oa,
                      int* ob, float* od, int* found, cudaStream_t s) {
  const long long parts = topk_parts(nb, k);
  k_topk_part<<<(unsigned)(parts / kTopkWarps), 32 * kTopkWarps, 0, s>>>(la, ld, nb * k, topk_share(nb, k), k, part_d,
                                                                         part_id);
  k_topk_last<<<1, 1024, 0, s>>>(la, part_d, part_id, parts * k, k, oa, ob, od, found);
  return cudaGetLastError() == cudaSuccess ? CL_OK : CL_ERR_CUDA;
}

}  // namespace clk
