// cl_sort.cuh -- sorting of one warp's segment of (index, value) pairs, shared
// by the one-set and the two-set neighbour lists.
#pragma once

#include <limits.h>

#include "cl_internal.cuh"

namespace clk {

constexpr int kSegPad = kMaxSegment + kMaxSegment / 32;

// Segment buffer index with one pad word per 32: conflict-free both for lane i
// at i (coalesced order) and for lane l at l * E + e (blocked order, E <= 32).
__device__ __forceinline__ int seg_at(int i) { return i + (i >> 5); }

// Bitonic sort, ascending by key, of 32 E elements held E per lane in blocked
// order (element lane * E + e). Pairs closer than E apart are in one lane's
// registers; farther ones are exchanged with a shuffle.
template <int E>
__device__ __forceinline__ void sort_blocked(int (&k)[E], float (&v)[E], int lane) {
#pragma unroll
  for (int size = 2; size <= 32 * E; size <<= 1) {
#pragma unroll
    for (int stride = size >> 1; stride > 0; stride >>= 1) {
      if (stride >= E) {
        const int ls = stride / E;
        const bool lower = (lane & ls) == 0;
#pragma unroll
        for (int e = 0; e < E; ++e) {
          const bool up = ((lane * E + e) & size) == 0;
          const int ok = __shfl_xor_sync(0xffffffffu, k[e], ls);
          const float ov = __shfl_xor_sync(0xffffffffu, v[e], ls);
          const bool take = (lower == up) ? (ok < k[e]) : (ok > k[e]);
          k[e] = take ? ok : k[e];
          v[e] = take ? ov : v[e];
        }
      } else {
#pragma unroll
        for (int e = 0; e < E; ++e) {
          if ((e & stride) == 0) {
            const int f = e | stride;
            const bool up = ((lane * E + e) & size) == 0;
            const bool sw = up ? (k[e] > k[f]) : (k[e] < k[f]);
            const int tk = k[e];
            const float tv = v[e];
            k[e] = sw ? k[f] : k[e];
            v[e] = sw ? v[f] : v[e];
            k[f] = sw ? tk : k[f];
            v[f] = sw ? tv : v[f];
          }
        }
      }
    }
  }
}

template <int E>
__device__ __forceinline__ void sort_segment_regs(int* K, float* V, int L, int lane) {
  int k[E];
  float v[E];
#pragma unroll
  for (int e = 0; e < E; ++e) {
    const int i = lane * E + e;
    k[e] = i < L ? K[seg_at(i)] : INT_MAX;
    v[e] = i < L ? V[seg_at(i)] : 0.f;
  }
  sort_blocked<E>(k, v, lane);
  __syncwarp();
#pragma unroll
  for (int e = 0; e < E; ++e) {
    const int i = lane * E + e;
    if (i < L) {
      K[seg_at(i)] = k[e];
      V[seg_at(i)] = v[e];
    }
  }
  __syncwarp();
}

// Segments longer than 16 per lane: the same network in shared memory.
__device__ __forceinline__ void sort_segment_smem(int* K, float* V, int L, int lane) {
  int P = 32;
  while (P < L) P <<= 1;
  for (int i = L + lane; i < P; i += 32) {
    K[seg_at(i)] = INT_MAX;
    V[seg_at(i)] = 0.f;
  }
  __syncwarp();
  for (int size = 2; size <= P; size <<= 1) {
    for (int stride = size >> 1; stride > 0; stride >>= 1) {
      for (int t = lane; t < (P >> 1); t += 32) {
        const int lo = 2 * stride * (t / stride) + (t % stride);
        const int hi = lo + stride;
        const bool up = (lo & size) == 0;
        const int ka = K[seg_at(lo)], kb = K[seg_at(hi)];
        if ((ka > kb) == up) {
          K[seg_at(lo)] = kb;
          K[seg_at(hi)] = ka;
          const float va = V[seg_at(lo)];
          V[seg_at(lo)] = V[seg_at(hi)];
          V[seg_at(hi)] = va;
        }
      }
      __syncwarp();
    }
  }
}

// Sorts the warp's segment of nw <= kMaxSegment pairs by key, in place.
__device__ __forceinline__ void sort_segment(int* K, float* V, int nw, int lane) {
  if (nw <= 1) {
  } else if (nw <= 32) {
    sort_segment_regs<1>(K, V, nw, lane);
  } else if (nw <= 64) {
    sort_segment_regs<2>(K, V, nw, lane);
  } else if (nw <= 128) {
    sort_segment_regs<4>(K, V, nw, lane);
  } else if (nw <= 256) {
    sort_segment_regs<8>(K, V, nw, lane);
  } else if (nw <= 512) {
    sort_segment_regs<16>(K, V, nw, lane);
  } else {
    sort_segment_smem(K, V, nw, lane);
  }
}

// Compare-exchange: the smaller key to a.
__device__ __forceinline__ void key_cas(unsigned& a, unsigned& b) {
  const unsigned lo = min(a, b);
  b = max(a, b);
  a = lo;
}

// Ascending sort of 32 E one-word keys, E per lane in blocked order: the
// merging network whose compare-exchanges all put the smaller key first (each
// merge opens with the mirrored pairing i <-> size - 1 - i), so a
// compare-exchange is one min and one max, with no direction to select.
template <int E>
__device__ __forceinline__ void sort_keys_blocked(unsigned (&k)[E], int lane) {
#pragma unroll
  for (int size = 2; size <= E; size <<= 1) {
#pragma unroll
    for (int e = 0; e < E; ++e)
      if (e < (e ^ (size - 1))) key_cas(k[e], k[e ^ (size - 1)]);
#pragma unroll
    for (int stride = size >> 2; stride > 0; stride >>= 1) {
#pragma unroll
      for (int e = 0; e < E; ++e)
        if ((e & stride) == 0) key_cas(k[e], k[e | stride]);
    }
  }
#pragma unroll 1  // rolled: unrolled, the 512- and 1,024-key networks overflow the instruction cache
  for (int lanes = 2; lanes <= 32; lanes <<= 1) {
    const bool low = (lane & (lanes >> 1)) == 0;
#pragma unroll
    for (int e = 0; e < (E + 1) / 2; ++e) {
      const int f = E - 1 - e;
      const unsigned a = __shfl_xor_sync(0xffffffffu, k[f], lanes - 1);
      const unsigned b = __shfl_xor_sync(0xffffffffu, k[e], lanes - 1);
      k[e] = low ? min(k[e], a) : max(k[e], a);
      if (f != e) k[f] = low ? min(k[f], b) : max(k[f], b);
    }
#pragma unroll 1
    for (int ls = lanes >> 2; ls > 0; ls >>= 1) {
      const bool lo = (lane & ls) == 0;
#pragma unroll
      for (int e = 0; e < E; ++e) {
        const unsigned o = __shfl_xor_sync(0xffffffffu, k[e], ls);
        k[e] = lo ? min(k[e], o) : max(k[e], o);
      }
    }
#pragma unroll
    for (int stride = E >> 1; stride > 0; stride >>= 1) {
#pragma unroll
      for (int e = 0; e < E; ++e)
        if ((e & stride) == 0) key_cas(k[e], k[e | stride]);
    }
  }
}

template <int E>
__device__ __forceinline__ void sort_keys_regs(unsigned* K, int L, int lane) {
  unsigned k[E];
#pragma unroll
  for (int e = 0; e < E; ++e) {
    const int i = lane * E + e;
    k[e] = i < L ? K[seg_at(i)] : 0xffffffffu;
  }
  sort_keys_blocked<E>(k, lane);
  __syncwarp();
#pragma unroll
  for (int e = 0; e < E; ++e) {
    const int i = lane * E + e;
    if (i < L) K[seg_at(i)] = k[e];
  }
  __syncwarp();
}

// Sorts the warp's segment of nw <= kMaxSegment one-word keys, in place. All
// keys are below 2^32 - 1 (the padding).
__device__ __forceinline__ void sort_keys(unsigned* K, int nw, int lane) {
  if (nw <= 1) {
  } else if (nw <= 32) {
    sort_keys_regs<1>(K, nw, lane);
  } else if (nw <= 64) {
    sort_keys_regs<2>(K, nw, lane);
  } else if (nw <= 128) {
    sort_keys_regs<4>(K, nw, lane);
  } else if (nw <= 256) {
    sort_keys_regs<8>(K, nw, lane);
  } else if (nw <= 512) {
    sort_keys_regs<16>(K, nw, lane);
  } else {
    sort_keys_regs<32>(K, nw, lane);
  }
}

}  // namespace clk
