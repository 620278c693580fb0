// Transforms of frame pairs by residue tasks, shared by the frame-pair
// imaging kernels (sm_103a).
//
// Every value is the same sample of two consecutive frames as one FP32 pair
// (fft::Cf2).  A 1-D transform of length N = P NR of an input with L occupied
// entries is NR independent tasks, one per output residue r: with
// n = n' + P q and k = NR m + r,
//   X[NR m + r] = sum_n' e^{2 pi i m n' / P} ( e^{2 pi i r n' / N}
//                 sum_q x[n' + P q] e^{2 pi i r q / NR} ),
// a sum over the L / P occupied blocks, P - 1 twiddles and one P-point DFT in
// registers, for any L.  The tasks of a transform read the same L inputs
// (shared-memory broadcasts: the NR lanes of one transform are neighbours)
// and exchange nothing.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

#include "epic_fft.cuh"

namespace epic {
namespace {

// y[j] += x[j] a for four complex pairs and one complex factor a given as
// splats; consecutive instructions share the factor's operand.
__device__ __forceinline__ void cmadd4(fft::Cf2* y, const fft::Cf2* __restrict__ x, fft::f32x2 ar, fft::f32x2 ai,
                                       fft::f32x2 nai) {
  using fft::Cf2;
  using fft::f2_fma;
  Cf2 v[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) v[j] = x[j];
#pragma unroll
  for (int j = 0; j < 4; ++j) y[j].re = f2_fma(v[j].re, ar, y[j].re);
#pragma unroll
  for (int j = 0; j < 4; ++j) y[j].im = f2_fma(v[j].im, ar, y[j].im);
#pragma unroll
  for (int j = 0; j < 4; ++j) y[j].re = f2_fma(v[j].im, nai, y[j].re);
#pragma unroll
  for (int j = 0; j < 4; ++j) y[j].im = f2_fma(v[j].re, ai, y[j].im);
}

// Task r of a transform of src[0 .. len4), len4 a multiple of 4 and uniform
// over the warp: y[m] = X[NR m + r].  tw: [P][NR] e^{2 pi i r n' / N};
// wq: [..][NR] e^{2 pi i r q / NR}.
template <int P, int NR>
__device__ __forceinline__ void dft_task(const fft::Cf2* __restrict__ src, int len4, int r, const float2* tw,
                                         const float2* wq, fft::Cf2 (&y)[P]) {
  using fft::Cf2;
  using fft::f2_fma;
  using fft::f2_splat;
  using fft::f32x2;
#pragma unroll
  for (int b = 0; b < P / 4; ++b) {
    if (4 * b < len4) {
#pragma unroll
      for (int j = 4 * b; j < 4 * b + 4; ++j) y[j] = src[j];
    } else {
#pragma unroll
      for (int j = 4 * b; j < 4 * b + 4; ++j) y[j] = Cf2{0ull, 0ull};
    }
  }
  for (int q = 1; P * q < len4; ++q) {
    const float2 a = wq[q * NR + r];
    const f32x2 ar = f2_splat(a.x), ai = f2_splat(a.y), nai = f2_splat(-a.y);
    const Cf2* s = src + P * q;
    const int left = len4 - P * q;
#pragma unroll
    for (int b = 0; b < P / 4; ++b)
      if (4 * b < left) cmadd4(&y[4 * b], s + 4 * b, ar, ai, nai);
  }
  if constexpr (NR > 1) {
#pragma unroll
    for (int j = 1; j < P; ++j) {
      const float2 t = tw[j * NR + r];
      const f32x2 c = f2_splat(t.x), s = f2_splat(t.y), ns = f2_splat(-t.y);
      const Cf2 v = y[j];
      y[j].re = f2_fma(v.im, ns, fft::f2_mul(v.re, c));
      y[j].im = f2_fma(v.re, s, fft::f2_mul(v.im, c));
    }
  }
  fft::Dft<P>::run(y);
}

// The tables tw [P][NR] and wq [NR][NR] (rounded up to n entries each) of
// dft_task from e^{2 pi i m / n}, by `threads` threads.
template <int N, int NR>
__device__ __forceinline__ void residue_tables(const float2* __restrict__ twid, float2* tw, float2* wq, int threads) {
  for (int i = threadIdx.x; i < N; i += threads) {
    const int n = i / NR, r = i % NR;
    tw[i] = twid[(n * r) & (N - 1)];
    wq[i] = twid[(N / NR * n * r) & (N - 1)];
  }
}

// |E|^2 of the outputs of a column task, both frames, into the running sums
// (one rounding of a sum per pair).
template <int P>
__device__ __forceinline__ void square_add(const fft::Cf2 (&y)[P], float (&acc)[P]) {
#pragma unroll
  for (int m = 0; m < P; ++m) {
    const float2 re = fft::f2_unpack(y[m].re), im = fft::f2_unpack(y[m].im);
    acc[m] += fmaf(re.x, re.x, fmaf(im.x, im.x, fmaf(re.y, re.y, im.y * im.y)));
  }
}

// Output slot `slot` of both frames times the phase ph (p1: may be null).
template <int P>
__device__ __forceinline__ void store_pixel(const fft::Cf2 (&y)[P], int slot, float2 ph, float2* p0, float2* p1) {
#pragma unroll
  for (int m = 0; m < P; ++m)
    if (m == slot) {
      const float2 re = fft::f2_unpack(y[m].re), im = fft::f2_unpack(y[m].im);
      *p0 = fft::cmul(make_float2(re.x, im.x), ph);
      if (p1) *p1 = fft::cmul(make_float2(re.y, im.y), ph);
    }
}

// Scaled voltage of the 4-bit sample in the low byte of b.
__device__ __forceinline__ float2 unpack_ci4(unsigned b, float vs) {
  const int re = static_cast<int>(b << 24) >> 28;
  const int im = static_cast<int>(b << 28) >> 28;
  return make_float2(static_cast<float>(re) * vs, static_cast<float>(im) * vs);
}

template <int FMT>
__device__ __forceinline__ float2 pair_volt(const void* volt, size_t idx, float vs) {
  if constexpr (FMT == 0) {
    return unpack_ci4(__ldg(static_cast<const unsigned char*>(volt) + idx), vs);
  } else {
    const float2 e = __ldg(static_cast<const float2*>(volt) + idx);
    return make_float2(e.x * vs, e.y * vs);
  }
}

// The share of one CTA in the cost of a list of work: `parts` equal parts of
// every channel, `pairs` frame pairs of each, cost[c + 1] - cost[c] per pair
// and part.  Positions [lo, hi) of the list; consecutive CTAs' shares meet.
struct Share {
  long long lo, hi, pairs;
  const int* cost;                                   // prefix sums, from any start
  int parts, start;
  __device__ __forceinline__ Share(const int* cost_prefix, int n_chan, int n_parts, long long n_pairs)
      : pairs(n_pairs), cost(cost_prefix), parts(n_parts), start(__ldg(cost_prefix)) {
    const long long total = static_cast<long long>(__ldg(cost + n_chan) - start) * parts * pairs, g = gridDim.x, b = blockIdx.x;
    lo = total / g * b + total % g * b / g;
    hi = total / g * (b + 1) + total % g * (b + 1) / g;
  }
  __device__ __forceinline__ long long weight(int v) const {
    const int c = v / parts;
    return __ldg(cost + c + 1) - __ldg(cost + c);
  }
  // position of part v = c * parts + part (v may be one past the last)
  __device__ __forceinline__ long long before(int v) const {
    const int c = v / parts, i = v - c * parts;
    const long long w = static_cast<long long>(__ldg(cost + c) - start) * parts + (i ? weight(v) * i : 0);
    return w * pairs;
  }
  // first pair of part v at or after position pos
  __device__ __forceinline__ long long pair_at(long long pos, int v) const {
    const long long w = weight(v);
    const long long p = (pos - before(v) + w - 1) / w;
    return p < 0 ? 0 : (p > pairs ? pairs : p);
  }
  // the first part that reaches past lo, of n parts
  __device__ __forceinline__ int first(int n) const {
    int a = 0, b = n;                                // before(a) <= lo < before(b)
    while (b - a > 1) {
      const int m = (a + b) / 2;
      if (before(m) <= lo) a = m;
      else b = m;
    }
    return a;
  }
};

}  // namespace
}  // namespace epic
