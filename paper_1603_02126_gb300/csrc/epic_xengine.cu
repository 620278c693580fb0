// Visibility-based comparison path of the noise-trend study (Sec. 4): an
// X-engine forming every antenna pair's visibility from the same voltage
// stream EPICal uses, and the Eq. 21 gain solve on those visibilities.
//
//   xengine      V[c][a][b] += (s_c^2 / T) sum_t E_a(t) conj(E_b(t)) per channel, a
//                [Na x T] by [T x Na] complex product, tiled 64 x 64 per CTA
//                (4 x 4 outputs per thread, FP32 in registers, upper-triangle
//                tiles only, the lower triangle written as the conjugate).
//                For 4-bit input every product and partial sum is an integer
//                below 2^24, so the FP32 sums are exact.
//   model_vis    V^M[c][a][b] = sum_s S_s e_a(s) conj(e_b(s)), e_a(s) =
//                e^{-2 pi i u_a . s}, FP64 from host phasors, kept in FP32.
//   stefcal      Eq. 21 by alternating least squares with every other iterate
//                averaged (StEFCal): a cluster of CTAs per channel, iterated
//                in the kernel until max_a |g_new - g| <= tol max_a |g_new| or
//                max_iter.
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <algorithm>

#include "epic_internal.h"
#include "epic_smem.cuh"
#include "epic_sum.cuh"

namespace epic {
namespace {

constexpr int kXT = 64;          // antennas per tile side
constexpr int kXK = 32;          // time samples per staged chunk
constexpr int kXThreads = 256;   // 16 x 16 threads, 4 x 4 outputs each
constexpr int kXSeg = 32768;     // samples per FP32 segment (exact for 4-bit input)

__device__ __forceinline__ float2 xload(const void* volt, int fmt, size_t idx) {
  if (fmt == 0) {
    const unsigned b = __ldg(static_cast<const unsigned char*>(volt) + idx);
    const int re = static_cast<int>(b << 24) >> 28;
    const int im = static_cast<int>(b << 28) >> 28;
    return make_float2(static_cast<float>(re), static_cast<float>(im));
  }
  return __ldg(static_cast<const float2*>(volt) + idx);
}

// blockIdx.x: channel * tile pairs + pair (upper triangle, row-major);
// blockIdx.y: time segment.
__global__ void __launch_bounds__(kXThreads) xengine_kernel(const XengineArgs A) {
  __shared__ __align__(16) float2 ea[kXK][kXT];
  __shared__ __align__(16) float2 eb[kXK][kXT];
  const int nb = (A.n_ant + kXT - 1) / kXT;
  const int pairs = nb * (nb + 1) / 2;
  const int c = blockIdx.x / pairs;
  int pr = blockIdx.x - c * pairs;
  int bi = 0;
  while (pr >= nb - bi) {                // (bi, bj) with bi <= bj
    pr -= nb - bi;
    ++bi;
  }
  const int bj = bi + pr;
  const int C = A.n_chan, Na = A.n_ant;
  const long long tb = static_cast<long long>(blockIdx.y) * kXSeg;
  const long long te = tb + kXSeg < A.n_time ? tb + kXSeg : A.n_time;
  const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
  float2 acc[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = make_float2(0.f, 0.f);
  for (long long t0 = tb; t0 < te; t0 += kXK) {
    __syncthreads();
    for (int i = threadIdx.x; i < kXK * kXT; i += kXThreads) {
      const int tt = i / kXT, k = i % kXT;
      const long long t = t0 + tt;
      const int a = bi * kXT + k, b = bj * kXT + k;
      const size_t row = (static_cast<size_t>(t) * C + c) * Na;
      ea[tt][k] = (t < te && a < Na) ? xload(A.volt, A.input_fmt, row + a) : make_float2(0.f, 0.f);
      eb[tt][k] = (t < te && b < Na) ? xload(A.volt, A.input_fmt, row + b) : make_float2(0.f, 0.f);
    }
    __syncthreads();
#pragma unroll 4
    for (int tt = 0; tt < kXK; ++tt) {
      float2 x[4], y[4];
      const float4 x01 = *reinterpret_cast<const float4*>(&ea[tt][ty * 4]);
      const float4 x23 = *reinterpret_cast<const float4*>(&ea[tt][ty * 4 + 2]);
      const float4 y01 = *reinterpret_cast<const float4*>(&eb[tt][tx * 4]);
      const float4 y23 = *reinterpret_cast<const float4*>(&eb[tt][tx * 4 + 2]);
      x[0] = make_float2(x01.x, x01.y); x[1] = make_float2(x01.z, x01.w);
      x[2] = make_float2(x23.x, x23.y); x[3] = make_float2(x23.z, x23.w);
      y[0] = make_float2(y01.x, y01.y); y[1] = make_float2(y01.z, y01.w);
      y[2] = make_float2(y23.x, y23.y); y[3] = make_float2(y23.z, y23.w);
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          // E_a conj(E_b)
          acc[i][j].x = fmaf(x[i].x, y[j].x, fmaf(x[i].y, y[j].y, acc[i][j].x));
          acc[i][j].y = fmaf(x[i].y, y[j].x, fmaf(-x[i].x, y[j].y, acc[i][j].y));
        }
    }
  }
  const float vs = A.vscale ? __ldg(A.vscale + c) : 1.0f;
  const double scale = static_cast<double>(vs) * static_cast<double>(vs) * A.scale;
  double2* V = A.vis + static_cast<size_t>(c) * Na * Na;
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int a = bi * kXT + ty * 4 + i, b = bj * kXT + tx * 4 + j;
      if (a >= Na || b >= Na) continue;
      if (bi == bj && b < a) continue;             // diagonal tile: upper half and the diagonal
      const double re = static_cast<double>(acc[i][j].x) * scale;
      const double im = static_cast<double>(acc[i][j].y) * scale;
      atomicAdd(&V[static_cast<size_t>(a) * Na + b].x, re);
      atomicAdd(&V[static_cast<size_t>(a) * Na + b].y, im);
      if (a != b) {
        atomicAdd(&V[static_cast<size_t>(b) * Na + a].x, re);
        atomicAdd(&V[static_cast<size_t>(b) * Na + a].y, -im);
      }
    }
}

// V^M[c][a][b] = sum_s S_s ph[c][s][a] conj(ph[c][s][b]) in FP64, stored
// rounded to FP32 for the solver; one thread per pair.
__global__ void model_vis_kernel(int n_chan, int n_ant, int n_src, const double2* __restrict__ ph,
                                 const double* __restrict__ flux, float2* __restrict__ vm) {
  const long long n = static_cast<long long>(n_chan) * n_ant * n_ant;
  const long long i = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x;
  if (i >= n) return;
  const int b = static_cast<int>(i % n_ant);
  const int a = static_cast<int>((i / n_ant) % n_ant);
  const int c = static_cast<int>(i / (static_cast<long long>(n_ant) * n_ant));
  double re = 0.0, im = 0.0;
  for (int s = 0; s < n_src; ++s) {
    const double2 pa = ph[(static_cast<size_t>(c) * n_src + s) * n_ant + a];
    const double2 pb = ph[(static_cast<size_t>(c) * n_src + s) * n_ant + b];
    const double S = flux[s];
    re += S * (pa.x * pb.x + pa.y * pb.y);
    im += S * (pa.y * pb.x - pa.x * pb.y);
  }
  vm[i] = make_float2(static_cast<float>(re), static_cast<float>(im));
}

constexpr int kSThreads = 1024;
constexpr double kStefcalMinTol = 1e-6;   // smallest stopping tolerance with FP32 pair products

// Pair terms of the solve, once per call: W_ab = V_ab conj(M_ab) and |M_ab|^2
// in FP32, M the model times a power of two that keeps its square in range
// (a model in SI units is near 1e-26).  For the pairs that are left out
// (autos, flagged antennas, baselines below the cut) and in the padding of a
// row W is 0 and |M|^2 is -0, which adds nothing and tells them apart.
__global__ void __launch_bounds__(128) pair_terms_kernel(const StefcalArgs A, const double2* __restrict__ vis) {
  const int Na = A.n_ant, ld = A.ld;
  const long long row = blockIdx.x;                          // channel * Na + antenna
  const int c = static_cast<int>(row / Na), a = static_cast<int>(row - static_cast<long long>(c) * Na);
  const double mb2 = A.min_baseline * A.min_baseline;
  const bool live = !A.flags[a];
  for (int b = threadIdx.x; b < ld; b += 128) {
    float2 w = make_float2(0.f, 0.f);
    float m2 = -0.f;
    bool use = live && b < Na && b != a && !A.flags[b];
    if (use && mb2 > 0.0) {
      const double2 ua = A.uv[row], ub = A.uv[static_cast<size_t>(c) * Na + b];
      const double dx = ua.x - ub.x, dy = ua.y - ub.y;
      use = !(dx * dx + dy * dy < mb2);
    }
    if (use) {
      float2 m = A.vm[row * Na + b];
      m = make_float2(m.x * A.vm_scale, m.y * A.vm_scale);
      const double2 v = vis[row * Na + b];
      const float vr = static_cast<float>(v.x), vi = static_cast<float>(v.y);
      w = make_float2(fmaf(vr, m.x, vi * m.y), fmaf(vi, m.x, -vr * m.y));
      m2 = fmaf(m.x, m.x, m.y * m.y);
    }
    A.w[row * ld + b] = w;
    A.m2[row * ld + b] = m2;
  }
}

// Size of a gain, as a number that orders as it: the bits of its larger part;
// kNotFinite where it is not finite.
constexpr unsigned kNotFinite = 0x7f800000u;
__device__ __forceinline__ unsigned size_of(float2 f) {
  const unsigned m = __float_as_uint(fmaxf(fabsf(f.x), fabsf(f.y)));
  return isfinite(f.x) && isfinite(f.y) ? m : kNotFinite;
}

// Power of two for gains of largest size m: 1 between 2^-20 and 2^20 (and for
// 0), else one that brings large gains near 2^-16 and small ones near 2^16, so
// that their squares stay in FP32's range and their products with W too, for
// visibilities (of order |g|^2) from 2^-120 to 2^120.
__device__ __forceinline__ float gain_scale(unsigned m) {
  const int k = static_cast<int>(m >> 23) - 127;
  if (m == 0u || (k >= -20 && k <= 20)) return 1.f;
  return ldexpf(1.f, k > 0 ? -k - 16 : -k + 16 > 120 ? 120 : -k + 16);
}

// A sum as hi + lo (FP32 each).
struct Sum2 {
  float hi, lo;
  __device__ __forceinline__ void add(float h, float l) {
    lo += l;
    add_kept(hi, lo, h);
  }
};

// Largest of the values so far (non-negative doubles order as their bits; NaN
// is passed over).
__device__ __forceinline__ void raise(unsigned long long* most, double v) {
  if (v >= 0.0) atomicMax(most, static_cast<unsigned long long>(__double_as_longlong(v)));
}

// Sums over the warp of three values of four rows: lane 8 j ends with row j's.
__device__ __forceinline__ void sum_rows(const float (&v)[4][3], Sum2 (&out)[3]) {
  const int lane = threadIdx.x & 31;
  Sum2 h[2][3];
#pragma unroll
  for (int k = 0; k < 3; ++k)
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const float keep = lane & 16 ? v[2 + i][k] : v[i][k], send = lane & 16 ? v[i][k] : v[2 + i][k];
      h[i][k] = Sum2{keep, 0.f};
      h[i][k].add(__shfl_xor_sync(0xffffffffu, send, 16), 0.f);
    }
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const Sum2 keep = lane & 8 ? h[1][k] : h[0][k], send = lane & 8 ? h[0][k] : h[1][k];
    out[k] = keep;
    out[k].add(__shfl_xor_sync(0xffffffffu, send.hi, 8), __shfl_xor_sync(0xffffffffu, send.lo, 8));
#pragma unroll
    for (int o = 4; o > 0; o >>= 1)
      out[k].add(__shfl_xor_sync(0xffffffffu, out[k].hi, o), __shfl_xor_sync(0xffffffffu, out[k].lo, o));
  }
}

// Eq. 21 by alternating least squares: g_a <- sum_b W_ab g_b / sum_b |V^M_ab|^2
// |g_b|^2, every other iterate averaged.  A cluster of CTAs per channel, each
// with a block of antenna rows; a warp sums four rows at a time (FP32
// products, two-float sums across the lanes: this GPU's FP64 rate is 1/73 of
// its FP32 rate, and the FP64 lane reductions took a third of an iteration),
// one thread per antenna divides, averages and tests in FP64 and writes the
// new gain, rounded to FP32, into every CTA's shared memory; one cluster
// barrier per iteration.  Gains far from 1 (|g|^2 alone would leave FP32's
// range) are multiplied by a power of two before an iteration uses them.
//
// What bounds it: W and |V^M|^2 (12 bytes a pair) come through L2 once per
// iteration, the division and a cluster barrier follow in series.
__global__ void __launch_bounds__(kSThreads) stefcal_kernel(const StefcalArgs A) {
  namespace cg = cooperative_groups;
  cg::cluster_group cluster = cg::this_cluster();
  extern __shared__ __align__(16) unsigned char ssm[];
  const int Na = A.n_ant, ld = A.ld, rows = A.rows;
  float2* gf = reinterpret_cast<float2*>(ssm);               // [2][ld] gains as FP32 (flagged and padding: 0)
  float* g2 = reinterpret_cast<float*>(gf + 2 * ld);         // [2][ld] |g|^2
  double2* g = reinterpret_cast<double2*>(g2 + 2 * ld);      // [rows] own gains
  float* sums = reinterpret_cast<float*>(g + rows);          // [rows][6] (hi, lo) of Re, Im, denominator
  __shared__ unsigned long long most[2][2];                  // by parity: largest |change|^2, |g|^2 of this CTA
  __shared__ unsigned long long all[2][2][8];                // the same of every CTA of the cluster
  __shared__ unsigned size[2], sizes[2][8];                  // likewise the largest size of the gains in use
  __shared__ unsigned finite;                                // the same of the finite ones
  const int cl = static_cast<int>(cluster.num_blocks()), q = static_cast<int>(cluster.block_rank());
  const int c = blockIdx.x / cl;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int a0 = q * rows, na = Na - a0 < rows ? (Na - a0 > 0 ? Na - a0 : 0) : rows;   // own antennas
  const float2* W = A.w + static_cast<size_t>(c) * Na * ld;
  const float* M = A.m2 + static_cast<size_t>(c) * Na * ld;
  double2* gio = A.gains + static_cast<size_t>(c) * Na;
  if (threadIdx.x < 2) size[threadIdx.x] = 0u;
  __syncthreads();
  for (int a = threadIdx.x; a < ld; a += kSThreads) {
    const double2 v = a < Na ? gio[a] : make_double2(0.0, 0.0);
    const bool live = a < Na && !A.flags[a];
    const float2 f = live ? make_float2(static_cast<float>(v.x), static_cast<float>(v.y)) : make_float2(0.f, 0.f);
    gf[a] = f;
    gf[ld + a] = make_float2(0.f, 0.f);
    g2[a] = fmaf(f.x, f.x, f.y * f.y);
    g2[ld + a] = 0.f;
    atomicMax(&size[1], size_of(f));
    if (a >= a0 && a < a0 + na) g[a - a0] = v;
  }
  if (threadIdx.x < 4) most[threadIdx.x >> 1][threadIdx.x & 1] = 0ull;
  cluster.sync();                                            // every CTA is resident and has read the gains
  const double tol = fmax(A.tol, kStefcalMinTol), tol2 = tol * tol;
  unsigned u = size[1];                                      // of the whole start, in every CTA
  int it = 0;
  for (; it < A.max_iter;) {
    const int cur = it & 1, nxt = cur ^ 1;
    // a gain in use that is not finite reaches the pairs it is part of, but
    // not, as 0 times it, those that are left out
    const bool skip = u == kNotFinite;                       // of the whole cluster, as t
    if (skip) {
      if (threadIdx.x == 0) finite = 0u;
      __syncthreads();
      for (int a = threadIdx.x; a < ld; a += kSThreads) {
        const unsigned m = size_of(gf[cur * ld + a]);
        if (m != kNotFinite) atomicMax(&finite, m);
      }
      __syncthreads();
      u = finite;
    }
    const float t = gain_scale(u);
    if (t != 1.f) {
      for (int a = threadIdx.x; a < ld; a += kSThreads) {
        const float2 f = make_float2(gf[cur * ld + a].x * t, gf[cur * ld + a].y * t);
        gf[cur * ld + a] = f;
        g2[cur * ld + a] = fmaf(f.x, f.x, f.y * f.y);
      }
      __syncthreads();
    }
    const float4* gp = reinterpret_cast<const float4*>(gf + cur * ld);
    const float4* hp = reinterpret_cast<const float4*>(g2 + cur * ld);
    for (int r = 4 * warp; r < na; r += 4 * (kSThreads / 32)) {
      float v[4][3];
#pragma unroll
      for (int i = 0; i < 4; ++i) v[i][0] = v[i][1] = v[i][2] = 0.f;
      for (int b = lane; 4 * b < ld; b += 32) {              // antennas 4 b .. 4 b + 3
        const float4 x0 = gp[2 * b], x1 = gp[2 * b + 1], y = hp[b];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int row = a0 + (r + i < na ? r + i : r);
          const float4* wp = reinterpret_cast<const float4*>(W + static_cast<size_t>(row) * ld);
          const float4 w0 = __ldg(wp + 2 * b), w1 = __ldg(wp + 2 * b + 1);
          const float4 m = __ldg(reinterpret_cast<const float4*>(M + static_cast<size_t>(row) * ld) + b);
          if (skip) {
            const float wr[4] = {w0.x, w0.z, w1.x, w1.z}, wi[4] = {w0.y, w0.w, w1.y, w1.w}, mm[4] = {m.x, m.y, m.z, m.w};
            const float xr[4] = {x0.x, x0.z, x1.x, x1.z}, xi[4] = {x0.y, x0.w, x1.y, x1.w}, yy[4] = {y.x, y.y, y.z, y.w};
#pragma unroll
            for (int j = 0; j < 4; ++j)
              if (!signbit(mm[j])) {
                v[i][0] = fmaf(wr[j], xr[j], fmaf(-wi[j], xi[j], v[i][0]));
                v[i][1] = fmaf(wr[j], xi[j], fmaf(wi[j], xr[j], v[i][1]));
                v[i][2] = fmaf(mm[j], yy[j], v[i][2]);
              }
            continue;
          }
          v[i][0] = fmaf(w0.x, x0.x, fmaf(-w0.y, x0.y, v[i][0]));
          v[i][1] = fmaf(w0.x, x0.y, fmaf(w0.y, x0.x, v[i][1]));
          v[i][0] = fmaf(w0.z, x0.z, fmaf(-w0.w, x0.w, v[i][0]));
          v[i][1] = fmaf(w0.z, x0.w, fmaf(w0.w, x0.z, v[i][1]));
          v[i][0] = fmaf(w1.x, x1.x, fmaf(-w1.y, x1.y, v[i][0]));
          v[i][1] = fmaf(w1.x, x1.y, fmaf(w1.y, x1.x, v[i][1]));
          v[i][0] = fmaf(w1.z, x1.z, fmaf(-w1.w, x1.w, v[i][0]));
          v[i][1] = fmaf(w1.z, x1.w, fmaf(w1.w, x1.z, v[i][1]));
          v[i][2] = fmaf(m.x, y.x, fmaf(m.y, y.y, fmaf(m.z, y.z, fmaf(m.w, y.w, v[i][2]))));
        }
      }
      Sum2 sum[3];
      sum_rows(v, sum);
      const int row = r + (lane >> 3);
      if ((lane & 7) == 0 && row < na) {
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          sums[row * 6 + 2 * k] = sum[k].hi;
          sums[row * 6 + 2 * k + 1] = sum[k].lo;
        }
      }
    }
    __syncthreads();
    for (int r = threadIdx.x; r < na; r += kSThreads) {
      const float* s = sums + 6 * r;
      const double den = static_cast<double>(s[4]) + static_cast<double>(s[5]);
      const double2 o = g[r];
      double2 x = o;
      if (den > 0.0) {
        x.x = (static_cast<double>(s[0]) + static_cast<double>(s[1])) / den;
        x.y = (static_cast<double>(s[2]) + static_cast<double>(s[3])) / den;
        if (t != 1.f || A.vm_scale != 1.f) {                 // the sums were those of s V^M and t g
          const double st = static_cast<double>(A.vm_scale) * static_cast<double>(t);
          x.x *= st;
          x.y *= st;
        }
      }
      if (it & 1) x = make_double2(0.5 * (x.x + o.x), 0.5 * (x.y + o.y));
      const double dx = x.x - o.x, dy = x.y - o.y;
      g[r] = x;
      raise(&most[cur][0], dx * dx + dy * dy);
      raise(&most[cur][1], x.x * x.x + x.y * x.y);
      if (!A.flags[a0 + r]) {
        const float2 f = make_float2(static_cast<float>(x.x), static_cast<float>(x.y));
        const float h = fmaf(f.x, f.x, f.y * f.y);
        atomicMax(&size[cur], size_of(f));
        for (int d = 0; d < cl; ++d) {
          cluster.map_shared_rank(gf, d)[nxt * ld + a0 + r] = f;
          cluster.map_shared_rank(g2, d)[nxt * ld + a0 + r] = h;
        }
      }
    }
    __syncthreads();
    if (threadIdx.x < cl) {
      unsigned long long(*dst)[2][8] = cluster.map_shared_rank(all, static_cast<int>(threadIdx.x));
      dst[cur][0][q] = most[cur][0];
      dst[cur][1][q] = most[cur][1];
      cluster.map_shared_rank(sizes, static_cast<int>(threadIdx.x))[cur][q] = size[cur];
    }
    if (threadIdx.x < 2) most[nxt][threadIdx.x] = 0ull;
    if (threadIdx.x == 2) size[nxt] = 0u;
    cluster.sync();
    ++it;
    unsigned long long d = 0, m = 0;
    u = 0;
    for (int k = 0; k < cl; ++k) {
      d = all[cur][0][k] > d ? all[cur][0][k] : d;
      m = all[cur][1][k] > m ? all[cur][1][k] : m;
      u = sizes[cur][k] > u ? sizes[cur][k] : u;
    }
    // FP32 pair products: changes below ~1e-6 are rounding, not progress
    if (__longlong_as_double(static_cast<long long>(d)) <= tol2 * __longlong_as_double(static_cast<long long>(m))) break;
  }
  for (int r = threadIdx.x; r < na; r += kSThreads) gio[a0 + r] = g[r];
  if (threadIdx.x == 0 && q == 0 && A.iters) A.iters[c] = it;
}

// CTAs per channel: as many as fill the GPU, up to 8 (a portable cluster),
// and as many as the gains' shared memory needs; rows per CTA a multiple of 4.
size_t stefcal_smem(int ld, int rows) {
  return static_cast<size_t>(2 * ld) * (sizeof(float2) + sizeof(float)) +
         static_cast<size_t>(rows) * (sizeof(double2) + 6 * sizeof(float));
}

}  // namespace

cudaError_t launch_xengine(const XengineArgs& a, cudaStream_t s) {
  const int nb = (a.n_ant + kXT - 1) / kXT;
  const int pairs = nb * (nb + 1) / 2;
  const long long segs = (a.n_time + kXSeg - 1) / kXSeg;
  dim3 grid(static_cast<unsigned>(a.n_chan * pairs), static_cast<unsigned>(segs));
  xengine_kernel<<<grid, kXThreads, 0, s>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_model_vis(int n_chan, int n_ant, int n_src, const double2* ph, const double* flux,
                             float2* vm, cudaStream_t s) {
  const long long n = static_cast<long long>(n_chan) * n_ant * n_ant;
  model_vis_kernel<<<static_cast<unsigned>((n + 255) / 256), 256, 0, s>>>(n_chan, n_ant, n_src, ph, flux, vm);
  return cudaGetLastError();
}

int stefcal_ld(int n_ant) { return (n_ant + 3) & ~3; }

// 64 channels x 256 antennas, 50 sources: 0.118 ms and 0.030 for the pair
// terms (two CTAs a channel), 1.2 ms with one CTA a channel and FP64 lane
// reductions.
cudaError_t launch_stefcal(const StefcalArgs& args, const double2* vis64, int sms, cudaStream_t s) {
  StefcalArgs a = args;
  a.ld = stefcal_ld(a.n_ant);
  int cl = 1;
  while (cl < 8 && (a.n_chan * 2 * cl <= sms && a.n_ant > 32 * cl)) cl *= 2;
  auto rows_of = [&](int k) { return ((a.n_ant + k - 1) / k + 3) & ~3; };
  while (cl < 8 && stefcal_smem(a.ld, rows_of(cl)) > 220 * 1024) cl *= 2;
  a.rows = rows_of(cl);
  const size_t smem = stefcal_smem(a.ld, a.rows);
  pair_terms_kernel<<<static_cast<unsigned>(a.n_chan * a.n_ant), 128, 0, s>>>(a, vis64);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  e = allow_smem(stefcal_kernel);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(static_cast<unsigned>(a.n_chan * cl));
  cfg.blockDim = dim3(kSThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = static_cast<unsigned>(cl);
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, stefcal_kernel, a);
}

}  // namespace epic
