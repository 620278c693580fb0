// Gridding lists of a block of grid rows, as the host lays them out, and the
// sum of one lane's taps for a frame pair (sm_103a).
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

#include "epic_fft.cuh"

namespace epic {
namespace {

// One row block's lists: header (slices, byte offsets of the cells and of
// the entries), slices (first entry, taps), cells (place in the block; 0xffff
// = none), entries (byte offset of E'_a, weight bits), entry k of a slice's 32
// lanes contiguous.
struct BlockLists {
  int nslice, cells, ents, unused;
};

// Slice of a warp in its k-th turn among `warps`: the slices are sorted by
// length, so every other turn runs backwards.
__device__ __forceinline__ int slice_of(int k, int warp, int warps) {
  return k * warps + (k & 1 ? warps - 1 - warp : warp);
}

// sum of w E'_a over the n entries e[0], e[32], ... of a lane's list.
__device__ __forceinline__ fft::Cf2 sum_taps(const uint2* __restrict__ e, int n, const fft::Cf2* Es) {
  fft::Cf2 sum{0ull, 0ull};
#pragma unroll 2
  for (int k = 0; k < n; ++k) {
    const uint2 en = e[k * 32];
    const fft::Cf2 x = *reinterpret_cast<const fft::Cf2*>(reinterpret_cast<const unsigned char*>(Es) + en.x);
    const fft::f32x2 w = fft::f2_splat(__uint_as_float(en.y));
    sum.re = fft::f2_fma(w, x.re, sum.re);
    sum.im = fft::f2_fma(w, x.im, sum.im);
  }
  return sum;
}

}  // namespace
}  // namespace epic
