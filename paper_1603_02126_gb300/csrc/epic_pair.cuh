// Shared parts of the frame-pair kernels that keep a whole frame pair on one SM
// (imaging and its adjoint, sm_103a): launch geometry, a channel's tables,
// gridding.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

#include "epic_fft.cuh"
#include "epic_internal.h"
#include "epic_lists.cuh"
#include "epic_residue.cuh"

namespace epic {
namespace {

using fft::Cf2;

// Frame pairs per FP32 partial gradient, and most per partial image (FP64
// across).
constexpr int kPairRun = 128;

template <int N> struct PCfg;
template <> struct PCfg<16>  { static constexpr int BT = 32,  PER_SM = 8; };
template <> struct PCfg<32>  { static constexpr int BT = 64,  PER_SM = 8; };
template <> struct PCfg<64>  { static constexpr int BT = 256, PER_SM = 2; };
template <> struct PCfg<128> { static constexpr int BT = 512, PER_SM = 1; };

template <int N>
struct PGeo {
  static constexpr int BT = PCfg<N>::BT;
  static constexpr int NR = N / 16;                  // residues = lanes per transform
  static constexpr int TASKS = N * NR;               // column tasks
  static constexpr int ROUNDS = TASKS < BT ? 1 : TASKS / BT;
  static_assert(TASKS < BT || TASKS % BT == 0, "column tasks must fill the CTA");
};

// Gridding of one frame pair: slices of 32 cells, one cell per lane.
template <int BT>
__device__ __forceinline__ void grid_pair(const int* __restrict__ cell, const int2* __restrict__ slice,
                                          const uint2* __restrict__ ent, int nslice, const Cf2* Es, Cf2* grid) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int k = 0; k * (BT / 32) < nslice; ++k) {
    const int sl = slice_of(k, warp, BT / 32);
    if (sl >= nslice) break;
    const int2 s = slice[sl];
    const int at = cell[sl * 32 + lane];
    const Cf2 sum = sum_taps(ent + s.x + lane, s.y, Es);
    if (at >= 0) grid[at] = sum;
  }
}

// Bring the voltages of frame pair p of channel c into L1.
template <int FMT, int BT>
__device__ __forceinline__ void prefetch_pair(const ImageArgs& A, long long p, int c) {
  constexpr int esz = FMT == 0 ? 1 : 8;
  const size_t bytes = static_cast<size_t>(A.n_ant) * esz;
#pragma unroll
  for (int f = 0; f < 2; ++f)
    if (2 * p + f < A.n_time) {
      const uintptr_t b0 = reinterpret_cast<uintptr_t>(A.volt) +
                           (static_cast<size_t>(2 * p + f) * A.n_chan + c) * bytes;
      for (uintptr_t q = (b0 & ~static_cast<uintptr_t>(127)) + static_cast<uintptr_t>(threadIdx.x) * 128; q < b0 + bytes;
           q += BT * 128)
        asm volatile("prefetch.global.L1 [%0];" ::"l"(q));
    }
}

// A channel's tables and geometry, its tap lists in shared memory (TS) or
// read through L1.
struct Chan {
  int R, R4, W4, nslice;
  const int2* slice;
  const int* cell;
  const uint2* ent;
  float vs;
  float2 pph;
  const float2* wg;
};

template <bool TS>
__device__ __forceinline__ Chan channel(const ImageArgs& A, int c, const int2* sslice, const int* scell,
                                        const uint2* sent) {
  Chan q;
  const int4 wn = __ldg(A.win4 + c);                       // (y0, rows, x0, cols)
  q.R = wn.y;
  q.R4 = (wn.y + 3) & ~3;
  q.W4 = (wn.w + 3) & ~3;
  const int sb = __ldg(A.psbase + c), eb = __ldg(A.pebase + c);
  q.nslice = __ldg(A.psbase + c + 1) - sb;
  q.slice = TS ? sslice : A.pslice + sb;
  q.cell = TS ? scell : A.pcell + static_cast<size_t>(sb) * 32;
  q.ent = TS ? sent : A.pent + eb;
  q.vs = A.vscale ? __ldg(A.vscale + c) : 1.0f;
  q.pph = A.do_cal ? __ldg(A.pixph + c) : make_float2(1.f, 0.f);
  q.wg = A.wgain + static_cast<size_t>(c) * A.n_ant;
  return q;
}

template <int BT>
__device__ __forceinline__ void load_lists(const ImageArgs& A, int c, int2* sslice, int* scell, uint2* sent) {
  const int sb = __ldg(A.psbase + c), eb = __ldg(A.pebase + c);
  const int ns = __ldg(A.psbase + c + 1) - sb, ne = __ldg(A.pebase + c + 1) - eb;
  for (int i = threadIdx.x; i < ns; i += BT) sslice[i] = __ldg(A.pslice + sb + i);
  for (int i = threadIdx.x; i < ns * 32; i += BT) scell[i] = __ldg(A.pcell + static_cast<size_t>(sb) * 32 + i);
  for (int i = threadIdx.x; i < ne; i += BT) sent[i] = __ldg(A.pent + eb + i);
}

}  // namespace
}  // namespace epic
