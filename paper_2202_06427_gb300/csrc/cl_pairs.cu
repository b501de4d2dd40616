// cl_pairs.cu -- the i<j neighbour list (Sec. 4.1: "the lists of pairs of
// particles within a cutoff"), sorted by (i, j), with the FP32 distance.
//
//   k_cell_last    the largest original index of each cell
//   k_pairs_sparse the two passes below with a warp per cell, on grids whose
//                  cells have few neighbours; the cells it leaves go on to
//   k_pairs_cell<COUNT>  one CTA per cell stages the cell's neighbourhood
//                  (the particles of its full stencil that lie within
//                  rc + half a cell diagonal of its centre and whose index is
//                  above the smallest of the cell's own) in shared memory;
//                  one warp per home particle sweeps it and counts the pairs
//                  with j > i (original indices), so every pair is counted
//                  once, by its smaller index, without atomics. A cell whose
//                  neighbourhood does not fit is flagged and listed.
//   (scan)         exclusive prefix sum of the counts in original order:
//                  segment of i = [start[i], start[i] + count[i])
//   k_pairs_cell<FILL>   the same staging, then the staged list's original
//                  indices are sorted (stage_sort), so each particle's pairs with
//                  j > i come out of a suffix of that order in ascending j and
//                  are written in order with coalesced stores
//   k_pairs_count / k_pairs_fill
//                  the listed cells' particles, one warp per particle
//                  straight from the sorted arrays; a
//                  segment longer than kMaxSegment is written unsorted and
//                  listed for k_pairs_sort_long
//   k_pairs_sort_long  one CTA per listed segment, in place in global memory
//
// Each particle's count and fill run the same arithmetic in the same kernel
// family, so the fill keeps exactly count[i] pairs (the write is clamped to
// count[i] all the same). The sweep visits the pair-images of a particle; the
// list is only defined when each pair has at most one image within rc
// (rc <= w_min / 2), which the host checks before launching.
#include <algorithm>
#include <climits>

#include "cl_query.cuh"
#include "cl_sort.cuh"

namespace clk {


// The particles of the listed cells (cells[0, *ncells)), a warp each: the pairs
// with j > i by the per-point sweep of cl_query.cuh. (One thread per particle
// for the count and a warp walking every stencil cell, with the segment
// sorted as (key, value) pairs, for the fill: a list of 230,000 particles at
// one cell per cutoff, whose cells all overflow, took 13.2 ms with its build
// and histogram; now 4.5.)
constexpr int kFillWarps = 4;

template <int G>
__global__ void __launch_bounds__(32 * kFillWarps) k_pairs_count(const __grid_constant__ CrossArgs A,
                                                                 const unsigned* __restrict__ cellc,
                                                                 const int* __restrict__ cells,
                                                                 const int* __restrict__ ncells,
                                                                 int* __restrict__ count) {
  extern __shared__ float4 stab[];
  __shared__ WarpCells work[kFillWarps];
  const int m = *ncells;
  if ((int)blockIdx.x >= m) return;
  load_stencil<false>(A, stab, nullptr);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int q = blockIdx.x; q < m; q += gridDim.x) {
    const int c = cells[q], p1 = A.cell_start[c + 1];
    for (int p = A.cell_start[c] + warp; p < p1; p += kFillWarps) {
      const float4 x = A.xs[p];
      const int i = __float_as_int(x.w);
      const unsigned n = __reduce_add_sync(0xffffffffu, query_count<G>(A, stab, work[warp], cellc[p], x, i));
      if (lane == 0) count[i] = (int)n;
    }
  }
}

// A segment of at most kMaxSegment pairs is sorted in the warp's shared memory
// (WIDE false, fewer than 2^22 particles: by the one-word key j << 10 | slot),
// a longer one written unsorted and listed in longs.
template <int G, bool WIDE>
__global__ void __launch_bounds__(32 * kFillWarps, 5) k_pairs_fill(const __grid_constant__ CrossArgs A,
                                                                   const unsigned* __restrict__ cellc,
                                                                   const int* __restrict__ cells,
                                                                   const int* __restrict__ ncells,
                                                                   const int* __restrict__ count,
                                                                   const long long* __restrict__ start,
                                                                   int* __restrict__ pi_out, int* __restrict__ pj_out,
                                                                   float* __restrict__ pd_out, int* __restrict__ longs,
                                                                   int* __restrict__ nlong) {
  extern __shared__ float4 stab[];
  __shared__ WarpCells work[kFillWarps];
  const int m = *ncells;
  if ((int)blockIdx.x >= m) return;
  load_stencil<false>(A, stab, nullptr);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float* V = reinterpret_cast<float*>(stab + A.noff) + (size_t)warp * 2 * kSegPad;
  unsigned* K = reinterpret_cast<unsigned*>(V + kSegPad);
  for (int q = blockIdx.x; q < m; q += gridDim.x) {
    const int c = cells[q], p1 = A.cell_start[c + 1];
    for (int p = A.cell_start[c] + warp; p < p1; p += kFillWarps) {
      const float4 x = A.xs[p];
      const int i = __float_as_int(x.w), cnt = __ldg(count + i);
      if (cnt == 0) continue;
      const long long base = __ldg(start + i);
      const bool big = cnt > kMaxSegment;
      const int L = query_hits<G>(A, stab, work[warp], cellc[p], x, i, [&](int e, int j, float d2) {
        if (e >= cnt) return;
        if (big) {
          pi_out[base + e] = i;
          pj_out[base + e] = j;
          pd_out[base + e] = d2 * rsqrt_nr(d2);
        } else {
          K[seg_at(e)] = WIDE ? (unsigned)j : ((unsigned)j << 10) | (unsigned)e;
          V[seg_at(e)] = d2;
        }
      });
      __syncwarp();
      if (big) {
        if (lane == 0) longs[atomicAdd(nlong, 1)] = i;
        continue;
      }
      const int nw = min(L, cnt);
      if (WIDE) sort_segment(reinterpret_cast<int*>(K), V, nw, lane);
      else sort_keys(K, nw, lane);
      for (int t = lane; t < nw; t += 32) {
        const unsigned key = K[seg_at(t)];
        const float d2 = V[WIDE ? seg_at(t) : seg_at((int)(key & 1023u))];
        pi_out[base + t] = i;
        pj_out[base + t] = WIDE ? (int)key : (int)(key >> 10);
        pd_out[base + t] = d2 * rsqrt_nr(d2);
      }
      __syncwarp();
    }
  }
}

// One CTA per listed segment (grid-stride over the *nlong entries): the
// segment sorted by j in place in global memory by a bitonic network whose
// compare-exchanges all put the smaller key first (each merge opens with the
// mirrored pairing i <-> size - 1 - i of its block), padded to a power of two
// with virtual +inf keys past the end, which never move.
__global__ void __launch_bounds__(1024) k_pairs_sort_long(const int* __restrict__ longs,
                                                         const int* __restrict__ nlong,
                                                         const int* __restrict__ count,
                                                         const long long* __restrict__ start, int* __restrict__ pj,
                                                         float* __restrict__ pd) {
  const int m = *nlong;
  for (int q = blockIdx.x; q < m; q += gridDim.x) {
    const int a = longs[q];
    const int L = count[a];
    int* K = pj + start[a];
    float* V = pd + start[a];
    int P = 2;
    while (P < L) P <<= 1;
    for (int size = 2; size <= P; size <<= 1) {
      for (int stride = size >> 1; stride > 0; stride >>= 1) {
        for (int t = threadIdx.x; t < (P >> 1); t += blockDim.x) {
          int lo, hi;
          if (stride == (size >> 1)) {
            const int blk = t / stride, off = t - blk * stride;
            lo = blk * size + off;
            hi = blk * size + size - 1 - off;
          } else {
            lo = ((t & ~(stride - 1)) << 1) | (t & (stride - 1));
            hi = lo + stride;
          }
          if (hi < L) {
            const int ka = K[lo], kb = K[hi];
            if (ka > kb) {
              K[lo] = kb;
              K[hi] = ka;
              const float va = V[lo];
              V[lo] = V[hi];
              V[hi] = va;
            }
          }
        }
        __syncthreads();
      }
    }
  }
}

// Shared pieces of the per-cell sweeps. A warp takes the stencil 32 entries
// at a time, one per lane: each lane finds its neighbour cell's particle
// range, a warp scan lays the ranges end to end, and the warp walks the
// concatenation 32 candidates per step (a shuffle binary search finds each
// candidate's entry), so the lanes stay busy however small the cells are.
constexpr int kStageMax = 3072;  // largest staged neighbourhood of one cell (the launch picks its capacity)

// Stencil entry k (a lane's; none from A.noff on) of cell (cx, cy, cz): the
// lane's range [j0, j0 + len) of sorted particles, its shift and, over the warp,
// the exclusive offsets of the ranges laid end to end and their total. A cell
// whose largest original index (last) is not above amin is left out.
struct Chunk {
  int j0, len, excl, total;
  float sx, sy, sz;
};

template <int DIM>
__device__ __forceinline__ Chunk chunk_ranges(const SweepArgs& A, const float4* stab, const int* __restrict__ last,
                                              int amin, int k, int cx, int cy, int cz) {
  const int lane = threadIdx.x & 31;
  Chunk ch;
  ch.j0 = 0;
  ch.len = 0;
  ch.sx = ch.sy = ch.sz = 0.f;
  if (k < A.noff) {
    const float4 e = stab[k];
    const unsigned d = __float_as_uint(e.w);
    int x2 = cx + (int)(d & 1023u);
    x2 -= (x2 >= A.nx) ? A.nx : 0;
    int y2 = cy + (int)((d >> 10) & 1023u);
    y2 -= (y2 >= A.ny) ? A.ny : 0;
    int z2 = 0;
    if (DIM == 3) {
      z2 = cz + (int)(d >> 20);
      z2 -= (z2 >= A.nz) ? A.nz : 0;
    }
    const int c = x2 + A.nx * (y2 + A.ny * z2);
    ch.j0 = __ldg(A.cell_start + c);
    ch.len = __ldg(last + c) > amin ? __ldg(A.cell_start + c + 1) - ch.j0 : 0;
    ch.sx = e.x;
    ch.sy = e.y;
    ch.sz = e.z;
  }
  int inc = ch.len;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int u = __shfl_up_sync(0xffffffffu, inc, o);
    inc += lane >= o ? u : 0;
  }
  ch.total = __shfl_sync(0xffffffffu, inc, 31);
  ch.excl = inc - ch.len;
  return ch;
}

// Candidate t of the chunk: its sorted index and the shift of its entry.
__device__ __forceinline__ int chunk_candidate(const Chunk& ch, int t, float& ax, float& ay, float& az) {
  int l = 0;  // last entry whose range starts at or before t
#pragma unroll
  for (int b = 16; b >= 1; b >>= 1) {
    const int u = __shfl_sync(0xffffffffu, ch.excl, l + b);
    l += (u <= t) ? b : 0;
  }
  ax = __shfl_sync(0xffffffffu, ch.sx, l);
  ay = __shfl_sync(0xffffffffu, ch.sy, l);
  az = __shfl_sync(0xffffffffu, ch.sz, l);
  return __shfl_sync(0xffffffffu, ch.j0, l) + (t - __shfl_sync(0xffffffffu, ch.excl, l));
}

__device__ __forceinline__ void stencil_to_smem(const SweepArgs& A, float4* stab) {
  for (int k = threadIdx.x; k < A.noff; k += blockDim.x) {
    const Off& o = A.off[k];
    stab[k] = make_float4(o.sx, o.sy, o.sz,
                          __uint_as_float((unsigned)o.dx | ((unsigned)o.dy << 10) | ((unsigned)o.dz << 20)));
  }
}

// Stable LSD radix sort (8-bit digits) of the staged list's original indices,
// the whole CTA (W warps) taking part: the slots 0..S-1 into st are sorted by
// the key jo - kmin (of `bits` bits), read through the slot (no key array, so
// that five CTAs fit per SM). Each warp ranks a fixed span of positions in
// order with __match_any_sync, and the (digit, warp) offsets come from one
// exclusive scan per pass, so equal digits keep their order. Returns the buffer
// that holds the sorted slots.
template <int W>
__device__ __noinline__ void stage_radix(const float4* st, int S, int bits, int kmin, unsigned short* s0,
                                         unsigned short* s1, unsigned short* cnt, int* scal,
                                         unsigned short*& slots) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const unsigned lt = (1u << lane) - 1u;
  __syncthreads();  // every warp has read the buckets' starts
  for (int i = threadIdx.x; i < S; i += blockDim.x) s0[i] = (unsigned short)i;
  __syncthreads();
  const int span = (((S + W - 1) / W) + 31) & ~31;
  const int b0 = min(S, warp * span), b1 = min(S, b0 + span);
  for (int sh = 0; sh < bits; sh += 8) {
    for (int i = threadIdx.x; i < 256 * W; i += blockDim.x) cnt[i] = 0;
    __syncthreads();
    for (int r = b0; r < b1; r += 32) {
      const int i = r + lane;
      const bool ok = i < b1;
      const int d = ok ? (int)(((unsigned)(__float_as_int(st[s0[i]].w) - kmin) >> sh) & 255u) : 256 + lane;
      const unsigned peers = __match_any_sync(0xffffffffu, d);
      if (ok && lane == __ffs(peers) - 1) cnt[d * W + warp] += (unsigned short)__popc(peers);
      __syncwarp();
    }
    __syncthreads();
    {  // exclusive scan of cnt in (digit, warp) order; 8 entries per thread
      const int per = 256 * W / blockDim.x;
      int loc = 0;
      for (int e = 0; e < per; ++e) loc += cnt[threadIdx.x * per + e];
      int inc = loc;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int u = __shfl_up_sync(0xffffffffu, inc, o);
        inc += lane >= o ? u : 0;
      }
      if (lane == 31) scal[4 + warp] = inc;
      __syncthreads();
      int off = inc - loc;
      for (int w = 0; w < warp; ++w) off += scal[4 + w];
      for (int e = 0; e < per; ++e) {
        const int v = cnt[threadIdx.x * per + e];
        cnt[threadIdx.x * per + e] = (unsigned short)off;
        off += v;
      }
    }
    __syncthreads();
    for (int r = b0; r < b1; r += 32) {
      const int i = r + lane;
      const bool ok = i < b1;
      const unsigned key = ok ? (unsigned)(__float_as_int(st[s0[i]].w) - kmin) : 0u;
      const int d = ok ? (int)((key >> sh) & 255u) : 256 + lane;
      const unsigned peers = __match_any_sync(0xffffffffu, d);
      const int base = ok ? cnt[d * W + warp] : 0;
      __syncwarp();
      if (ok) {
        if (lane == __ffs(peers) - 1) cnt[d * W + warp] = (unsigned short)(base + __popc(peers));
        const int pos = base + __popc(peers & lt);
        s1[pos] = s0[i];
      }
      __syncwarp();
    }
    __syncthreads();
    unsigned short* ts = s0;
    s0 = s1;
    s1 = ts;
  }
  slots = s0;
}

constexpr int kBuckets = 1024;
constexpr int kBucketMost = 48;  // a fuller bucket sends the cell to the radix sort

// Orders the staged list's slots 0..S-1 (into st) by original index, the whole
// CTA (W warps) taking part; scal[1], scal[2]: the smallest and largest index.
// Returns the sorted slots (one of s0, s1) and kmin, the smallest index.
//
// The indices are spread over kBuckets equal parts of their range by a counting
// sort whose slots come from shared-memory atomics, then each entry finds its
// place within its bucket by counting the smaller ones. On an input in random
// order a bucket holds about one entry; on one that follows space the entries
// are runs of a few consecutive indices, a run or two to a bucket. Six barriers
// against thirteen for the radix sort's three passes. A cell whose fullest
// bucket passes kBucketMost (indices in a few tight clumps) takes the radix
// sort.
//
// IMAGES: two images of a particle may be staged (PairLists), one at most within
// the cutoff. Each needs a place of its own, so an entry also counts the equal
// ones before it: a variant of its own, because doing so always took a list of
// 2.1e8 pairs with a histogram from 4.12 to 4.22 ms (a branch on it 4.16).
template <int W, bool IMAGES>
__device__ __forceinline__ void stage_sort(const float4* st, int S, unsigned short* s0, unsigned short* s1, int* cnt,
                                           int* scal, unsigned short*& slots, int& kmin) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  constexpr int T = 32 * W, per = kBuckets / T;
  if (tid == 0) {
    scal[1] = INT_MAX;
    scal[2] = 0;
    scal[3] = 0;
  }
#pragma unroll
  for (int e = 0; e < per; ++e) cnt[tid + T * e] = 0;
  __syncthreads();
  int lo = INT_MAX, hi = 0;
  for (int i = tid; i < S; i += T) {
    const int jo = __float_as_int(st[i].w);
    lo = min(lo, jo);
    hi = max(hi, jo);
  }
  lo = __reduce_min_sync(0xffffffffu, lo);
  hi = __reduce_max_sync(0xffffffffu, hi);
  if (lane == 0) {
    atomicMin(scal + 1, lo);
    atomicMax(scal + 2, hi);
  }
  __syncthreads();
  kmin = scal[1];
  if (S == 0) {
    slots = s0;
    return;
  }
  const unsigned range = (unsigned)(scal[2] - kmin);
  const int bits = range ? 32 - __clz(range) : 0;
  const int sh = max(0, bits - 10);  // range >> sh < kBuckets
  for (int i = tid; i < S; i += T)
    s0[i] = (unsigned short)atomicAdd(&cnt[(unsigned)(__float_as_int(st[i].w) - kmin) >> sh], 1);
  __syncthreads();
  {  // exclusive scan of the buckets, per of them per thread
    int v[per], loc = 0, most = 0;
#pragma unroll
    for (int e = 0; e < per; ++e) {
      v[e] = cnt[tid * per + e];
      loc += v[e];
      most = max(most, v[e]);
    }
    most = __reduce_max_sync(0xffffffffu, most);
    int inc = loc;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int u = __shfl_up_sync(0xffffffffu, inc, o);
      inc += lane >= o ? u : 0;
    }
    if (lane == 31) scal[4 + warp] = inc;
    if (lane == 0 && most > kBucketMost) scal[3] = 1;
    __syncthreads();
    int off = inc - loc;
    for (int w = 0; w < warp; ++w) off += scal[4 + w];
#pragma unroll
    for (int e = 0; e < per; ++e) {
      cnt[tid * per + e] = off;
      off += v[e];
    }
  }
  __syncthreads();
  if (scal[3]) {
    stage_radix<W>(st, S, bits, kmin, s0, s1, reinterpret_cast<unsigned short*>(cnt), scal, slots);
    return;
  }
  for (int i = tid; i < S; i += T)
    s1[cnt[(unsigned)(__float_as_int(st[i].w) - kmin) >> sh] + s0[i]] = (unsigned short)i;
  __syncthreads();
  for (int p = tid; p < S; p += T) {
    const int i = s1[p];
    const int jo = __float_as_int(st[i].w);
    const unsigned b = (unsigned)(jo - kmin) >> sh;
    const int b0 = cnt[b], b1 = b + 1 < (unsigned)kBuckets ? cnt[b + 1] : S;
    int r = b0;
    for (int q = b0; q < b1; ++q) r += __float_as_int(st[s1[q]].w) < jo + (IMAGES && q < p ? 1 : 0) ? 1 : 0;
    s0[r] = (unsigned short)i;
  }
  __syncthreads();
  slots = s0;
}

// Squared distances of a staged entry q to two home particles (nx, ny, nz:
// their negated coordinates), both in packed FP32: per lane the same rounding
// as fmaf(dx, dx, fmaf(dy, dy, dz * dz)) with dx = q.x - x. The count and the
// fill pass both decide j within rc from this one expression.
template <int DIM>
__device__ __forceinline__ float2 pair_d2(const float4& q, float2 nx, float2 ny, float2 nz, float2& dx, float2& dy,
                                          float2& dz) {
  dx = __fadd2_rn(make_float2(q.x, q.x), nx);
  dy = __fadd2_rn(make_float2(q.y, q.y), ny);
  if (DIM == 3) {
    dz = __fadd2_rn(make_float2(q.z, q.z), nz);
    return __ffma2_rn(dx, dx, __ffma2_rn(dy, dy, __fmul2_rn(dz, dz)));
  }
  dz = make_float2(0.f, 0.f);
  return __ffma2_rn(dx, dx, __fmul2_rn(dy, dy));
}

// Largest original index of each cell's particles (-1: none), kLastLanes lanes
// to a cell, and the list's counters cleared. A cell's staging leaves out the
// cells whose largest index is not above the smallest of its own: on an input
// whose order follows space about half of the stencil (list of 2.1e8 pairs of a
// million particles with a histogram 4.55 -> 4.28 ms); in random order the
// launch is all it adds.
constexpr int kLastLanes = 8;

__global__ void __launch_bounds__(256) k_cell_last(long long ncells, const int* __restrict__ cell_start,
                                                   const float4* __restrict__ xs, int* __restrict__ last,
                                                   int* __restrict__ ctr) {
  const long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x, c = t / kLastLanes;
  if (t < 3) ctr[t] = 0;
  const int sub = (int)(t % kLastLanes);
  int m = -1;
  if (c < ncells)
    for (int p = cell_start[c] + sub, p1 = cell_start[c + 1]; p < p1; p += kLastLanes)
      m = max(m, __float_as_int(__ldg(&xs[p].w)));
#pragma unroll
  for (int o = kLastLanes / 2; o; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
  if (c < ncells && sub == 0) last[c] = m;
}

// U steps of a warp's staging, 32 candidates of ch each from t0 on: the
// particles, shifted to the cell's frame, and the lanes (m) that hold one within
// sqrt(ball2) of the cell's centre and of an index above amin.
template <int U>
struct StagedSteps {
  float4 q[U];
  unsigned m[U];
  int total;
};

template <int DIM, int U>
__device__ __forceinline__ StagedSteps<U> staged_steps(const SweepArgs& A, const Chunk& ch, int t0, float ball2,
                                                       int amin) {
  const int lane = threadIdx.x & 31;
  StagedSteps<U> r;
  float ax[U], ay[U], az[U];
#pragma unroll
  for (int u = 0; u < U; ++u) {
    const int t = t0 + 32 * u + lane;
    const int j = chunk_candidate(ch, t, ax[u], ay[u], az[u]);
    r.q[u] = make_float4(0.f, 0.f, 0.f, __int_as_float(-1));  // beyond the end: not above amin
    if (t < ch.total) r.q[u] = __ldg(&A.xs[j]);
  }
  r.total = 0;
#pragma unroll
  for (int u = 0; u < U; ++u) {
    float4& q = r.q[u];
    q.x += ax[u];
    q.y += ay[u];
    q.z = DIM == 3 ? q.z + az[u] : 0.f;
    r.m[u] = __ballot_sync(0xffffffffu, fmaf(q.x, q.x, fmaf(q.y, q.y, q.z * q.z)) < ball2 && __float_as_int(q.w) > amin);
    r.total += __popc(r.m[u]);
  }
  return r;
}

// Appends them to the list st of cap entries from entry base on.
template <int U>
__device__ __forceinline__ void append_steps(const StagedSteps<U>& r, int base, int cap, float4* st) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int u = 0; u < U; ++u) {
    if (r.m[u] >> lane & 1u) {
      const int e = base + __popc(r.m[u] & ((1u << lane) - 1u));
      if (e < cap) st[e] = r.q[u];
    }
    base += __popc(r.m[u]);
  }
}

template <int DIM, int U>
__device__ __forceinline__ void stage_steps(const SweepArgs& A, const Chunk& ch, int t0, float ball2, int amin, int cap,
                                            float4* st, int* nst) {
  const StagedSteps<U> r = staged_steps<DIM, U>(A, ch, t0, ball2, amin);
  int base = 0;
  if ((threadIdx.x & 31) == 0 && r.total) base = atomicAdd(nst, r.total);
  append_steps(r, __shfl_sync(0xffffffffu, base, 0), cap, st);
}

// Home particles p and p + 1 (the second if below h1) against the S staged
// entries, a warp; both share each staged load. The pairs with j > i are
// counted; the distance of each (particle, candidate) is computed as in the fill
// pass.
template <int DIM>
__device__ __forceinline__ void count_two(const SweepArgs& A, int p, int h1, const float4* st, int S,
                                          int* __restrict__ count) {
  const int lane = threadIdx.x & 31;
  const bool two = p + 1 < h1;
  const float4 pa = A.xs[p];
  const float4 pb = two ? A.xs[p + 1] : pa;
  const int a0 = __float_as_int(pa.w), a1 = two ? __float_as_int(pb.w) : INT_MAX;
  const float2 nx = make_float2(-pa.x, -pb.x), ny = make_float2(-pa.y, -pb.y),
               nz = make_float2(-pa.z, -pb.z);
  int L0 = 0, L1 = 0;  // per lane, summed over the warp at the end
#pragma unroll 2
  for (int t = lane; t < S; t += 32) {
    const float4 q = st[t];
    const int jo = __float_as_int(q.w);
    float2 dx, dy, dz;
    const float2 d2 = pair_d2<DIM>(q, nx, ny, nz, dx, dy, dz);
    L0 += (jo > a0 && d2.x < A.rc2) ? 1 : 0;
    L1 += (jo > a1 && d2.y < A.rc2) ? 1 : 0;
  }
  L0 = __reduce_add_sync(0xffffffffu, L0);
  L1 = __reduce_add_sync(0xffffffffu, L1);
  if (lane == 0) {
    count[a0] = L0;
    if (two) count[a1] = L1;
  }
}

// The same two particles' segments of the list, from the staged entries in
// order of their indices (at(t): entry t; kmin: the smallest index). The sweep
// starts at the earlier of their suffixes (entries before a particle's own
// suffix fail j > i) and each particle's kept pairs are written in order from
// its own ballot.
template <int DIM, class At>
__device__ __forceinline__ void fill_two(const SweepArgs& A, int p, int h1, At at, int S, int kmin,
                                         const int* __restrict__ count, const long long* __restrict__ start,
                                         int* __restrict__ pi_out, int* __restrict__ pj_out,
                                         float* __restrict__ pd_out) {
  const int lane = threadIdx.x & 31;
  const unsigned lt = (1u << lane) - 1u;
  const bool two = p + 1 < h1;
  const float4 pa = A.xs[p];
  const float4 pb = two ? A.xs[p + 1] : pa;
  const int a0 = __float_as_int(pa.w), a1 = two ? __float_as_int(pb.w) : INT_MAX;
  int f0 = 0, f1 = S;  // first position (in index order) with index > a0, a1
  {
    const unsigned ka = a0 >= kmin ? (unsigned)(a0 - kmin) : 0u;
    int lo = 0, hi = S;
    while (a0 >= kmin && lo < hi) {
      const int mid = (lo + hi) >> 1;
      if ((unsigned)(__float_as_int(at(mid).w) - kmin) > ka) hi = mid;
      else lo = mid + 1;
    }
    f0 = a0 >= kmin ? lo : 0;
  }
  if (two) {
    const unsigned kb = a1 >= kmin ? (unsigned)(a1 - kmin) : 0u;
    int lo = 0, hi = S;
    while (a1 >= kmin && lo < hi) {
      const int mid = (lo + hi) >> 1;
      if ((unsigned)(__float_as_int(at(mid).w) - kmin) > kb) hi = mid;
      else lo = mid + 1;
    }
    f1 = a1 >= kmin ? lo : 0;
  }
  const int c0 = __ldg(count + a0), c1 = two ? __ldg(count + a1) : 0;
  const long long b0 = __ldg(start + a0), b1 = two ? __ldg(start + a1) : 0;
  const float2 nx = make_float2(-pa.x, -pb.x), ny = make_float2(-pa.y, -pb.y),
               nz = make_float2(-pa.z, -pb.z);
  int L0 = 0, L1 = 0;
#pragma unroll 2
  for (int t0 = min(f0, f1); t0 < S; t0 += 32) {
    const int t = t0 + lane;
    bool k0 = false, k1 = false;
    int jo = 0;
    float d20 = 0.f, d21 = 0.f;
    if (t < S) {
      const float4 q = at(t);
      jo = __float_as_int(q.w);
      float2 dx, dy, dz;
      const float2 d2 = pair_d2<DIM>(q, nx, ny, nz, dx, dy, dz);
      d20 = d2.x;
      d21 = d2.y;
      k0 = jo > a0 && d20 < A.rc2;
      k1 = jo > a1 && d21 < A.rc2;
    }
    const unsigned m0 = __ballot_sync(0xffffffffu, k0), m1 = __ballot_sync(0xffffffffu, k1);
    if (k0) {
      const int e = L0 + __popc(m0 & lt);
      if (e < c0) {
        pi_out[b0 + e] = a0;
        pj_out[b0 + e] = jo;
        pd_out[b0 + e] = d20 * rsqrt_nr(d20);
      }
    }
    if (k1) {
      const int e = L1 + __popc(m1 & lt);
      if (e < c1) {
        pi_out[b1 + e] = a1;
        pj_out[b1 + e] = jo;
        pd_out[b1 + e] = d21 * rsqrt_nr(d21);
      }
    }
    L0 += __popc(m0);
    L1 += __popc(m1);
  }
}

// Sparse grids (at most kSparse particles expected in a staging ball): a warp
// per cell, no barrier; the staged entries, up to kSparseCap, are ordered by
// counting the smaller indices of each. Latency-bound: 2D lists with their
// builds took, with a CTA of eight warps per cell of one particle, 525 us at
// 57,000 particles and 371 at 31,000; 190 and 178 so. Cells that do not fit are
// listed (cells) for k_pairs_cell in both passes. kSparse: those two lists expect
// 25 in a ball, 2D lists at other cell sizes up to 40; denser grids keep the CTA.
// So do large stencils about few particles, where the list takes as long as one
// warp needs for its cell's entries: 3D at 0.1 per cell, 613 entries, 646 us by
// warps and 275 by CTAs for 5,000 particles, 716 and 634 for 20,000, 875 and 1,067
// for 40,000; 311 entries 318 and 224 for 5,000, 340 and 306 for 10,000, 385 and
// 487 for 20,000; 125 entries 117 and 121 for 2,000.
constexpr int kSparse = 64, kSparseCap = 160, kSparseWarps = 4;
static_assert((kMaxOff + 2 * kSparseWarps * kSparseCap) * sizeof(float4) <= 48 * 1024, "the default shared memory");

template <int DIM, bool FILL>
__global__ void __launch_bounds__(32 * kSparseWarps) k_pairs_sparse(const __grid_constant__ SweepArgs A, float ball2,
                                                                    const int* __restrict__ last,
                                                                    int* __restrict__ cells, int* __restrict__ nlisted,
                                                                    int* __restrict__ count,
                                                                    const long long* __restrict__ start,
                                                                    int* __restrict__ pi_out, int* __restrict__ pj_out,
                                                                    float* __restrict__ pd_out) {
  extern __shared__ float4 smem[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float4* stab = smem;
  float4* st = stab + A.noff + warp * kSparseCap * (FILL ? 2 : 1);
  stencil_to_smem(A, stab);
  __syncthreads();
  const int ncells = A.nx * A.ny * A.nz;
  for (int c = blockIdx.x * kSparseWarps + warp; c < ncells; c += gridDim.x * kSparseWarps) {
    const int h0 = __ldg(A.cell_start + c), h1 = __ldg(A.cell_start + c + 1);
    if (h1 == h0) continue;
    const int cx = c % A.nx, cy = (c / A.nx) % A.ny, cz = c / (A.nx * A.ny);
    int amin = INT_MAX;  // as in k_pairs_cell
    for (int p = h0 + lane; p < h1; p += 32) amin = min(amin, __float_as_int(__ldg(&A.xs[p].w)));
    amin = __reduce_min_sync(0xffffffffu, amin);
    __syncwarp();  // the cell before is done with
    int S = 0;
    for (int k0 = 0; k0 < A.noff; k0 += 32) {
      const Chunk ch = chunk_ranges<DIM>(A, stab, last, amin, k0 + lane, cx, cy, cz);
      for (int t0 = 0; t0 < ch.total; t0 += 32) {
        const StagedSteps<1> q = staged_steps<DIM, 1>(A, ch, t0, ball2, amin);
        append_steps(q, S, kSparseCap, st);
        S += q.total;
      }
    }
    __syncwarp();
    if (S > kSparseCap) {
      if (!FILL && lane == 0) cells[atomicAdd(nlisted, 1)] = c;
      continue;
    }
    if (!FILL) {
      for (int p = h0; p < h1; p += 2) count_two<DIM>(A, p, h1, st, S, count);
    } else {
      float4* so = st + kSparseCap;
      int kmin = INT_MAX;
      for (int e = lane; e < S; e += 32) {
        const int v = __float_as_int(st[e].w);
        int r = 0;
        for (int f = 0; f < S; ++f) {
          const int w = __float_as_int(st[f].w);
          r += (w < v || (w == v && f < e)) ? 1 : 0;  // equal: two images, at most one within the cutoff
        }
        so[r] = st[e];
        kmin = min(kmin, v);
      }
      kmin = __reduce_min_sync(0xffffffffu, kmin);
      __syncwarp();
      for (int p = h0; p < h1; p += 2)
        fill_two<DIM>(A, p, h1, [&](int t) { return so[t]; }, S, kmin, count, start, pi_out, pj_out, pd_out);
    }
  }
}

// One CTA of W warps per cell (grid-stride over the cells). The stencil
// entries are shared among the warps 32 at a time; each warp appends the
// particles of its entries that lie within sqrt(ball2) of the cell centre,
// shifted to the cell's frame (x_j + s_o), to the staged list. Then warp w
// sweeps home particles w, w + W, ... against it (distance (x_j + s_o) - x_i).
// Particles whose original index is not above the smallest of the cell's own
// are not staged: no pair with j > i of this cell needs them.
// COUNT: count[a] = pairs with j > a; a cell whose list does not fit gets
// flag 1 (else 0) and is listed in fcells. FILL: flagged cells are skipped; the staged list is ordered
// by original index (stage_sort), so a particle's pairs with
// j > a come from a suffix of that order in ascending j and are written in
// order, coalesced, as the ballot finds them.
// With cells, the *nlisted cells of that list only. IMAGES: see stage_sort.
template <int DIM, bool FILL, bool IMAGES>
__global__ void __launch_bounds__(256, FILL ? 5 : 6) k_pairs_cell(const __grid_constant__ SweepArgs A,
                                                                               float ball2, int cap,
                                                                               const int* __restrict__ cells,
                                                                               const int* __restrict__ nlisted,
                                                                               const int* __restrict__ last,
                                                                               unsigned char* __restrict__ flag,
                                                                               int* __restrict__ fcells,
                                                                               int* __restrict__ nfcells,
                                                                               int* __restrict__ count,
                                                                               const long long* __restrict__ start,
                                                                               int* __restrict__ pi_out,
                                                                               int* __restrict__ pj_out,
                                                                               float* __restrict__ pd_out) {
  constexpr int W = 8;
  extern __shared__ float4 smem[];
  float4* st = smem;           // staged neighbourhood: (x, y, z in the cell's frame, original index)
  float4* stab = st + cap;     // stencil: (s_x, s_y, s_z, dx | dy << 10 | dz << 20)
  int* scal = reinterpret_cast<int*>(stab + A.noff);  // [0] staged count, [1..2] index range, [4..] warp sums
  int* cnt = scal + 16;  // FILL: bucket (or radix) counters and slots
  unsigned short* rs0 = reinterpret_cast<unsigned short*>(cnt + kBuckets);
  unsigned short* rs1 = rs0 + cap;
  const int m = cells ? *nlisted : A.nx * A.ny * A.nz;
  if ((int)blockIdx.x >= m) return;
  stencil_to_smem(A, stab);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int q = blockIdx.x; q < m; q += gridDim.x) {
    const int c = cells ? cells[q] : q;
    const int h0 = __ldg(A.cell_start + c), h1 = __ldg(A.cell_start + c + 1);
    if (h1 == h0) continue;
    if (FILL && flag[c]) continue;
    const int cx = c % A.nx, cy = (c / A.nx) % A.ny, cz = c / (A.nx * A.ny);
    if (threadIdx.x == 0) scal[0] = 0;
    // the smallest original index among the cell's particles (each warp on
    // its own): a staged particle of index <= amin pairs with none of them
    // under j > i, so neither pass stages it
    int amin = INT_MAX;
    for (int p = h0 + lane; p < h1; p += 32) amin = min(amin, __float_as_int(__ldg(&A.xs[p].w)));
    amin = __reduce_min_sync(0xffffffffu, amin);
    __syncthreads();
    // the stencil dealt to the warps entry by entry: of an input whose order
    // follows space, the cells left out are one side of the stencil
    for (int k0 = warp; k0 < A.noff; k0 += 32 * W) {
      const Chunk ch = chunk_ranges<DIM>(A, stab, last, amin, k0 + W * lane, cx, cy, cz);
      // pairs of steps: two loads in flight per lane, one reservation for both
      // (the list and histogram above 4.28 -> 4.13 ms)
      int t0 = 0;
      for (; t0 + 32 < ch.total; t0 += 64) stage_steps<DIM, 2>(A, ch, t0, ball2, amin, cap, st, scal);
      if (t0 < ch.total) stage_steps<DIM, 1>(A, ch, t0, ball2, amin, cap, st, scal);
    }
    __syncthreads();
    const int S = scal[0];
    if (S <= cap) {
      unsigned short* slots = rs0;
      int kmin = 0;
      if (FILL) stage_sort<W, IMAGES>(st, S, rs0, rs1, cnt, scal, slots, kmin);
      if (!FILL) {
        for (int p = h0 + 2 * warp; p < h1; p += 2 * W) count_two<DIM>(A, p, h1, st, S, count);
      }
      if (FILL)
        for (int p = h0 + 2 * warp; p < h1; p += 2 * W)
          fill_two<DIM>(A, p, h1, [&](int t) { return st[(int)slots[t]]; }, S, kmin, count, start, pi_out, pj_out, pd_out);
    }
    if (!FILL && threadIdx.x == 0) {
      flag[c] = S > cap ? 1 : 0;
      if (S > cap) fcells[atomicAdd(nfcells, 1)] = c;
    }
    __syncthreads();
  }
}

size_t pairs_cell_smem(int noff, bool fill, int cap) {
  const size_t head = (size_t)(cap + noff) * sizeof(float4) + 16 * sizeof(int);
  static_assert(kBuckets * sizeof(int) >= 256 * 8 * sizeof(unsigned short), "the radix counters fit");
  return fill ? head + kBuckets * sizeof(int) + 2 * (size_t)cap * sizeof(unsigned short) : head;
}

// The grids of k_pairs_sparse (measured at kSparse).
static bool by_warps(const SweepArgs& A, const PairLists& L) {
  return L.expect <= kSparse && (A.noff <= 160 || A.n >= 40 * A.noff);
}

// The staged passes: k_pairs_sparse for sparse grids and k_pairs_cell for the
// cells it lists, k_pairs_cell alone otherwise.
template <int DIM, bool FILL, bool IMAGES>
static int launch_cell(const SweepArgs& A, const PairLists& L, const long long* start, int* pi, int* pj, float* pd,
                       cudaStream_t s) {
  static DevCache ready;  // shared-memory limit raised on this device
  if (L.cap < 32 || L.cap > kStageMax) return CL_ERR_INVALID_ARG;
  int dev = 0, sms = 0, per = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return CL_ERR_CUDA;
  if (!ready.get(dev)) {
    if (cudaFuncSetAttribute(k_pairs_cell<DIM, FILL, IMAGES>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)pairs_cell_smem(kMaxOff, FILL, kStageMax)) != cudaSuccess)
      return CL_ERR_CUDA;
    ready.put(dev, 1);
  }
  const size_t smem = pairs_cell_smem(A.noff, FILL, L.cap);
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_pairs_cell<DIM, FILL, IMAGES>, 256, smem) !=
          cudaSuccess ||
      per < 1)
    return CL_ERR_CUDA;
  long long blocks = (long long)sms * per;
  const long long ncells = (long long)A.nx * A.ny * A.nz;
  if (blocks > ncells) blocks = ncells;
  const bool sparse = by_warps(A, L);
  if (sparse) {
    const size_t sm = sizeof(float4) * (size_t)(A.noff + kSparseWarps * kSparseCap * (FILL ? 2 : 1));
    const long long sb = std::min<long long>((ncells + kSparseWarps - 1) / kSparseWarps, (long long)sms * 64);
    k_pairs_sparse<DIM, FILL><<<(int)sb, 32 * kSparseWarps, sm, s>>>(A, L.ball2, L.last, L.mid, L.ctr + 2, L.count,
                                                                    start, pi, pj, pd);
  }
  k_pairs_cell<DIM, FILL, IMAGES><<<(int)blocks, 256, smem, s>>>(A, L.ball2, L.cap, sparse ? L.mid : nullptr,
                                                                L.ctr + 2, L.last, L.flag, L.fcells, L.ctr + 1,
                                                                L.count, start, pi, pj, pd);
  return cudaGetLastError() == cudaSuccess ? CL_OK : CL_ERR_CUDA;
}

int launch_pairs_count(const SweepArgs& A, const Off* off, int dim, const PairLists& L, cudaStream_t s) {
  if (A.n <= 0) return CL_OK;
  const long long ncells = (long long)A.nx * A.ny * A.nz;
  k_cell_last<<<(unsigned)((ncells * kLastLanes + 255) / 256), 256, 0, s>>>(ncells, A.cell_start, A.xs, L.last, L.ctr);
  const int e = dim == 3 ? launch_cell<3, false, false>(A, L, nullptr, nullptr, nullptr, nullptr, s)
                         : launch_cell<2, false, false>(A, L, nullptr, nullptr, nullptr, nullptr, s);
  if (e) return e;
  const CrossArgs C = cross_args(A, off);
  const size_t dyn = (size_t)C.noff * sizeof(float4);
  const int* nf = L.ctr + 1;
  switch (group_lanes(A)) {
    case 2: k_pairs_count<2><<<152 * 8, 32 * kFillWarps, dyn, s>>>(C, A.cellc, L.fcells, nf, L.count); break;
    case 4: k_pairs_count<4><<<152 * 8, 32 * kFillWarps, dyn, s>>>(C, A.cellc, L.fcells, nf, L.count); break;
    default: k_pairs_count<8><<<152 * 8, 32 * kFillWarps, dyn, s>>>(C, A.cellc, L.fcells, nf, L.count); break;
  }
  return cudaGetLastError() == cudaSuccess ? CL_OK : CL_ERR_CUDA;
}

template <int G, bool WIDE>
static int launch_fill_listed(const CrossArgs& C, const unsigned* cellc, const int* fcells, const int* nfcells,
                              const int* count, const long long* start, int* pi, int* pj, float* pd, int* longs,
                              int* nlong, cudaStream_t s) {
  static DevCache ready;  // shared-memory limit raised on this device
  const size_t seg = (size_t)kFillWarps * 2 * kSegPad * sizeof(float);
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return CL_ERR_CUDA;
  if (!ready.get(dev)) {
    if (cudaFuncSetAttribute(k_pairs_fill<G, WIDE>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)(seg + kMaxOff * sizeof(float4))) != cudaSuccess)
      return CL_ERR_CUDA;
    ready.put(dev, 1);
  }
  k_pairs_fill<G, WIDE><<<152 * 5, 32 * kFillWarps, seg + (size_t)C.noff * sizeof(float4), s>>>(
      C, cellc, fcells, nfcells, count, start, pi, pj, pd, longs, nlong);
  return cudaGetLastError() == cudaSuccess ? CL_OK : CL_ERR_CUDA;
}

int launch_sort_long(const int* longs, const int* nlong, const int* count, const long long* start, int* pj,
                            float* pd, cudaStream_t s) {
  k_pairs_sort_long<<<152, 1024, 0, s>>>(longs, nlong, count, start, pj, pd);
  return cudaGetLastError() == cudaSuccess ? CL_OK : CL_ERR_CUDA;
}

int launch_pairs_fill(const SweepArgs& A, const Off* off, int dim, const PairLists& L, const long long* start, int* pi,
                      int* pj, float* pd, int* longs, cudaStream_t s) {
  if (A.n <= 0) return CL_OK;
  int e;
  if (dim == 3)
    e = L.images ? launch_cell<3, true, true>(A, L, start, pi, pj, pd, s)
                 : launch_cell<3, true, false>(A, L, start, pi, pj, pd, s);
  else
    e = L.images ? launch_cell<2, true, true>(A, L, start, pi, pj, pd, s)
                 : launch_cell<2, true, false>(A, L, start, pi, pj, pd, s);
  if (e) return e;
  const CrossArgs C = cross_args(A, off);
  const int g = group_lanes(A);
  int *nf = L.ctr + 1, *nlong = L.ctr;
  int f;
  if (A.n >= (1 << 22))
    f = launch_fill_listed<8, true>(C, A.cellc, L.fcells, nf, L.count, start, pi, pj, pd, longs, nlong, s);
  else if (g == 2)
    f = launch_fill_listed<2, false>(C, A.cellc, L.fcells, nf, L.count, start, pi, pj, pd, longs, nlong, s);
  else if (g == 4)
    f = launch_fill_listed<4, false>(C, A.cellc, L.fcells, nf, L.count, start, pi, pj, pd, longs, nlong, s);
  else
    f = launch_fill_listed<8, false>(C, A.cellc, L.fcells, nf, L.count, start, pi, pj, pd, longs, nlong, s);
  if (f) return f;
  return launch_sort_long(longs, nlong, L.count, start, pj, pd, s);
}

}  // namespace clk
