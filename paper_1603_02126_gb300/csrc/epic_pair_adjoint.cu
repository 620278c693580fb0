// Frame-pair adjoint of the fused imaging kernel (differentiation form, FP32,
// N = 16..128, sm_103a): the gradient of a loss on the time-averaged image
// with respect to the conjugate gain multipliers,
//   dL/dconj(w_a) = (1/T) sum_t conj(E_a(t)) sum_j W'_a(j) [F^H (R . X(t))]_j,
// R = dL/dI, X the raw transform of frame t's folded grid, F^H the conjugate
// transform, every frame recomputed.  Two frames go through all four
// transforms as FP32 pairs, with the image kernel's geometry, tap lists and
// shared memory; the grid is in window coordinates (the window's phase of X
// and its conjugate in F^H cancel).
//
// The conjugate transforms are the transposes of the residue tasks: lane r of
// the NR lanes of one transform has the values k = NR m + r, takes their
// 16-point DFT over m and the twiddle e^{2 pi i r n' / N} in registers, and the
// sum over r with e^{2 pi i r q / NR} for every q of the window is a transform
// across the lanes by shuffles: each step but the last keeps, in the lower
// lanes, the sums (even q) and, in the upper, the twiddled differences (odd
// q); the last step shares the 16 n' between the two lanes and gives q and
// q + NR / 2.  (As conj(F^H y) = F conj(y), values are conjugated once, at
// the product with R.)
//
// Four phases per frame pair, a CTA barrier after each:
//   rows       grid -> spectra; E' of the next pair;
//   columns    spectra -> X, times R (registers), back into the column's
//              window rows in place; the next pair is gridded;
//   rows back  row spectra -> window cells, in place;
//   degrid     the K x K taps of every antenna, times conj(E_a).
//
// What bounds it: latency between the four barriers with 16 warps (issue 46 %,
// FP32 pipe 43 %, short scoreboards of the shuffles and loads first).  256
// antennas, 16 channels, 128 x 128, 4096 samples: 4.3 ms against 4.8 for one
// frame per FP32 value with exchanges through shared memory; without the
// permuted places the 16-byte stores of a transform's lanes fell into one
// bank (0.59 against 0.58 ms for 8192 frames), without unrolled taps 0.58
// against 0.56.
#include "epic_pair.cuh"
#include "epic_smem.cuh"

namespace epic {
namespace {

using fft::cmul;
using fft::f2_add;
using fft::f2_fma;
using fft::f2_mul;
using fft::f2_pack;
using fft::f2_splat;
using fft::f2_sub;
using fft::f2_unpack;
using fft::f32x2;

__device__ __forceinline__ Cf2 shfl_xor2(const Cf2& v, int m) {
  return Cf2{__shfl_xor_sync(fft::kFull, v.re, m), __shfl_xor_sync(fft::kFull, v.im, m)};
}

// Steps M = NR, NR / 2, ... 4 of the transform across the lanes.
template <int M, int NR>
__device__ __forceinline__ void lane_steps(Cf2 (&z)[16], int r, const float2* wq) {
  if constexpr (M > 2) {
    const bool hi = (r & (M / 2)) != 0;
    // e^{2 pi i r' / M} for the differences, r' = r mod M / 2; 1 for the sums
    const float2 t = hi ? wq[(NR / M) * NR + (r & (M / 2 - 1))] : make_float2(1.f, 0.f);
    const f32x2 sg = f2_splat(hi ? -1.f : 1.f), c = f2_splat(t.x), s = f2_splat(t.y), ns = f2_splat(-t.y);
#pragma unroll
    for (int j = 0; j < 16; ++j) {
      const Cf2 o = shfl_xor2(z[j], M / 2);
      const f32x2 re = f2_fma(z[j].re, sg, o.re), im = f2_fma(z[j].im, sg, o.im);
      z[j].re = f2_fma(im, ns, f2_mul(re, c));
      z[j].im = f2_fma(re, s, f2_mul(im, c));
    }
    lane_steps<M / 2, NR>(z, r, wq);
  }
}

// Block q of the window that lane r holds after the steps: bit reversal of
// the lane's bits above the last.
template <int NR>
__device__ __forceinline__ int lane_block(int r) {
  int q = 0;
#pragma unroll
  for (int m = NR / 2, b = 1; m > 1; m /= 2, b *= 2)
    if (r & m) q += b;
  return q;
}

// Place of window row or column n between the phases of the way back: the
// lanes of a transform store n = j mod 8 together, so the low bits are
// exchanged by the block of 8 (a permutation inside each block).
__device__ __forceinline__ int place(int n) { return n ^ ((n >> 3) & 7); }

// Conjugate transform of a task's values z[m] = y[NR m + r] (already
// conjugated) to dst[place(n) * stride], n < len, of all lanes together.
// live: this lane's transform exists (dead lanes take part in the shuffles).
template <int NR>
__device__ __forceinline__ void inverse_task(Cf2 (&z)[16], int r, const float2* tw, const float2* wq, Cf2* dst,
                                             int stride, int len, bool live) {
  fft::Dft<16>::run(z);
  if constexpr (NR == 1) {
    if (live)
#pragma unroll
      for (int j = 0; j < 16; ++j)
        if (j < len) dst[place(j) * stride] = z[j];
  } else {
#pragma unroll
    for (int j = 1; j < 16; ++j) {
      const float2 t = tw[j * NR + r];
      const f32x2 c = f2_splat(t.x), s = f2_splat(t.y), ns = f2_splat(-t.y);
      const Cf2 v = z[j];
      z[j].re = f2_fma(v.im, ns, f2_mul(v.re, c));
      z[j].im = f2_fma(v.re, s, f2_mul(v.im, c));
    }
    lane_steps<NR, NR>(z, r, wq);
    // last step: lane bit 0 keeps n' = 0..7 or 8..15
    const bool hi = (r & 1) != 0;
    const int q = lane_block<NR>(r), n0 = 16 * q + (hi ? 8 : 0), n1 = n0 + 8 * NR;   // blocks q and q + NR / 2
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const Cf2 keep = hi ? z[j + 8] : z[j], send = hi ? z[j] : z[j + 8];
      const Cf2 o = shfl_xor2(send, 1);
      if (live) {
        if (n0 + j < len) dst[place(n0 + j) * stride] = Cf2{f2_add(keep.re, o.re), f2_add(keep.im, o.im)};
        if (n1 + j < len)
          dst[place(n1 + j) * stride] = hi ? Cf2{f2_sub(o.re, keep.re), f2_sub(o.im, keep.im)}
                                      : Cf2{f2_sub(keep.re, o.re), f2_sub(keep.im, o.im)};
      }
    }
  }
}

// sum over the K x K taps of w T at window column x, row y (KC: K at compile
// time, all loads in flight; 0: any K).
template <int KC>
__device__ __forceinline__ Cf2 degrid(const float* __restrict__ wa, int K, const Cf2* T, int rs, int x, int y) {
  Cf2 s{0ull, 0ull};
  if constexpr (KC > 0) {
    float w[KC * KC];
#pragma unroll
    for (int i = 0; i < KC * KC; ++i) w[i] = __ldg(wa + i);
#pragma unroll
    for (int dx = 0; dx < KC; ++dx)
#pragma unroll
      for (int dy = 0; dy < KC; ++dy) {
        const f32x2 v = f2_splat(w[dy * KC + dx]);
        const Cf2 b = T[place(x + dx) * rs + place(y + dy)];
        s.re = f2_fma(v, b.re, s.re);
        s.im = f2_fma(v, b.im, s.im);
      }
  } else {
    for (int dx = 0; dx < K; ++dx)
      for (int dy = 0; dy < K; ++dy) {
        const f32x2 v = f2_splat(__ldg(wa + dy * K + dx));
        const Cf2 b = T[place(x + dx) * rs + place(y + dy)];
        s.re = f2_fma(v, b.re, s.re);
        s.im = f2_fma(v, b.im, s.im);
      }
  }
  return s;
}

template <int N, int FMT, int MAXA, bool TS>
__global__ void __launch_bounds__(PCfg<N>::BT, PCfg<N>::PER_SM) epic_adjoint_pair(const ImageArgs A, const double* dldi,
                                                                                 double2* dldw) {
  using G = PGeo<N>;
  constexpr int BT = G::BT, NR = G::NR, TASKS = G::TASKS, ROUNDS = G::ROUNDS;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int rs = A.rs, gs = A.gs, Na = A.n_ant;
  Cf2* Tt = reinterpret_cast<Cf2*>(smem_raw);              // [N][rs] spectra, transposed; then window cells
  Cf2* grid = Tt + N * rs;                                 // [rows_alloc][gs]
  Cf2* Es = grid + A.rows_alloc * gs;                      // [Na + 1] E' (entry Na is zero)
  float2* tw = reinterpret_cast<float2*>(Es + Na + 1);     // [16][NR]
  float2* wq = tw + N;                                     // [16][NR]
  int2* sslice = reinterpret_cast<int2*>(wq + N + 2);      // [max_slices] (TS)
  uint2* sent = reinterpret_cast<uint2*>(sslice + A.max_slices);   // [max_ent] (TS)
  int* scell = reinterpret_cast<int*>(sent + A.max_ent);   // [max_slices * 32] (TS)

  const int tid = threadIdx.x;
  const int aw = (BT - 32 - (tid & ~31)) + (tid & 31);     // antenna of this thread: the last warps first
  residue_tables<N, NR>(A.twid, tw, wq, BT);
  if (tid == 0) Es[Na] = Cf2{0ull, 0ull};

  const long long T = A.n_time;
  const int C = A.n_chan, K = A.support, KK = K * K;
  const Share share(A.pcost, C, 1, (T + 1) / 2);
  int cur = -1;
  for (int c = share.first(C); c < C && share.before(c) < share.hi; ++c) {
    const long long p_lo = share.pair_at(share.lo, c), p_hi = share.pair_at(share.hi, c);
    const Chan ch = channel<TS>(A, c, sslice, scell, sent);
    const int x0 = __ldg(A.win4 + c).z, pad = ch.R4 - ch.R;
    const int* cell0 = A.cell0 + static_cast<size_t>(c) * Na;   // window row * N + absolute column of tap (0, 0)
    const float* wts = A.wts + static_cast<size_t>(c) * Na * KK;
    // E' of pair p (a missing second frame is zero)
    auto form_e = [&](long long p) {
#pragma unroll
      for (int i = 0; i < MAXA; ++i) {
        const int a = aw + BT * i;
        if (a < Na) {
          const size_t idx = (static_cast<size_t>(2 * p) * C + c) * Na + a;
          const float2 w = __ldg(ch.wg + a);
          const float2 e0 = cmul(pair_volt<FMT>(A.volt, idx, ch.vs), w);
          float2 e1 = make_float2(0.f, 0.f);
          if (2 * p + 1 < T) e1 = cmul(pair_volt<FMT>(A.volt, idx + static_cast<size_t>(C) * Na, ch.vs), w);
          Es[a] = Cf2{f2_pack(e0.x, e1.x), f2_pack(e0.y, e1.y)};
        }
      }
    };
    // R of this thread's pixels, in the column tasks' output order
    float rk[ROUNDS][16];
    if (p_lo < p_hi) {
      const double* rimg = dldi + static_cast<size_t>(c) * N * N;
#pragma unroll
      for (int i = 0; i < ROUNDS; ++i) {
        const int task = tid + BT * i;
#pragma unroll
        for (int m = 0; m < 16; ++m)
          rk[i][m] = TASKS >= BT || task < TASKS
                         ? static_cast<float>(__ldg(rimg + (NR * m + task % NR) * N + task / NR))
                         : 0.f;
      }
    }
    for (long long pa = p_lo; pa < p_hi; pa += kPairRun) {
      const long long pb = pa + kPairRun < p_hi ? pa + kPairRun : p_hi;
      __syncthreads();                                     // the previous run's shared memory is free
      if (cur != c) {
        if (TS) load_lists<BT>(A, c, sslice, scell, sent);
        for (int i = tid; i < A.rows_alloc * gs; i += BT) grid[i] = Cf2{0ull, 0ull};   // cells without taps stay zero
        for (int i = tid; i < N * pad; i += BT) Tt[(i / pad) * rs + ch.R + i % pad] = Cf2{0ull, 0ull};
        cur = c;
      }
      float2 gac[MAXA];
#pragma unroll
      for (int i = 0; i < MAXA; ++i) gac[i] = make_float2(0.f, 0.f);
      form_e(pa);
      __syncthreads();
      grid_pair<BT>(ch.cell, ch.slice, ch.ent, ch.nslice, Es, grid);
      __syncthreads();
      for (long long p = pa; p < pb; ++p) {
        if (p + 2 < pb) prefetch_pair<FMT, BT>(A, p + 2, c);
        // ---- rows ----
        for (int task = tid; task < ch.R * NR; task += BT) {
          const int row = task / NR, r = task % NR;
          Cf2 y[16];
          dft_task<16, NR>(grid + row * gs, ch.W4, r, tw, wq, y);
#pragma unroll
          for (int m = 0; m < 16; ++m) Tt[(NR * m + r) * rs + row] = y[m];
        }
        if (p + 1 < pb) form_e(p + 1);
        __syncthreads();
        // ---- columns, times R, back into the window rows ----
#pragma unroll
        for (int i = 0; i < ROUNDS; ++i) {
          const int task = tid + BT * i;
          const bool live = TASKS >= BT || task < TASKS;
          const int kx = live ? task / NR : 0, r = task % NR;
          Cf2* col = Tt + kx * rs;
          Cf2 y[16];
          dft_task<16, NR>(col, ch.R4, r, tw, wq, y);
#pragma unroll
          for (int m = 0; m < 16; ++m) {                   // conj(R X)
            y[m].re = f2_mul(y[m].re, f2_splat(rk[i][m]));
            y[m].im = f2_mul(y[m].im, f2_splat(-rk[i][m]));
          }
          __syncwarp();                                    // every lane has read the column
          inverse_task<NR>(y, r, tw, wq, col, 1, ch.R, live);
        }
        if (p + 1 < pb) grid_pair<BT>(ch.cell, ch.slice, ch.ent, ch.nslice, Es, grid);
        __syncthreads();
        // ---- rows back to window cells: T[place(x)][place(row)] ----
        for (int t0 = 0; t0 < ch.R * NR; t0 += BT) {
          const int task = t0 + tid;
          if (t0 + (tid & ~31) >= ch.R * NR) break;        // whole warps
          const bool live = task < ch.R * NR;
          const int row = live ? task / NR : 0, r = task % NR;
          Cf2 y[16];
#pragma unroll
          for (int m = 0; m < 16; ++m) y[m] = Tt[(NR * m + r) * rs + place(row)];
          __syncwarp();                                    // every lane has read the row
          inverse_task<NR>(y, r, tw, wq, Tt + place(row), rs, ch.W4, live);
        }
        __syncthreads();
        // ---- degrid: Y_a = conj(sum of w T), conj(E_a) Y_a ----
#pragma unroll
        for (int i = 0; i < MAXA; ++i) {
          const int a = aw + BT * i;
          const int c0 = a < Na ? __ldg(cell0 + a) : -1;
          if (c0 >= 0) {
            const size_t idx = (static_cast<size_t>(2 * p) * C + c) * Na + a;
            const float2 e0 = pair_volt<FMT>(A.volt, idx, ch.vs);
            float2 e1 = make_float2(0.f, 0.f);
            if (2 * p + 1 < T) e1 = pair_volt<FMT>(A.volt, idx + static_cast<size_t>(C) * Na, ch.vs);
            const float* wa = wts + static_cast<size_t>(a) * KK;
            const int x = (c0 & (N - 1)) - x0, y = c0 / N;
            const Cf2 s = K == 3 ? degrid<3>(wa, 3, Tt, rs, x, y) : degrid<0>(wa, K, Tt, rs, x, y);
            const float2 sr = f2_unpack(s.re), si = f2_unpack(s.im);
            gac[i].x += e0.x * sr.x - e0.y * si.x + (e1.x * sr.y - e1.y * si.y);
            gac[i].y -= e0.x * si.x + e0.y * sr.x + (e1.x * si.y + e1.y * sr.y);
          }
        }
        // the columns read rows R .. R4 - 1 as zeros; the way back may have
        // left window rows there (place stays inside a block of 8)
        __syncthreads();
        for (int i = tid; i < N * pad; i += BT) Tt[(i / pad) * rs + ch.R + i % pad] = Cf2{0ull, 0ull};
      }
#pragma unroll
      for (int i = 0; i < MAXA; ++i) {
        const int a = aw + BT * i;
        if (a < Na && __ldg(cell0 + a) >= 0) {
          const size_t o = static_cast<size_t>(c) * Na + a;
          atomicAdd(&dldw[o].x, static_cast<double>(gac[i].x) * A.img_scale);
          atomicAdd(&dldw[o].y, static_cast<double>(gac[i].y) * A.img_scale);
        }
      }
    }
  }
}

using AdjKernel = void (*)(const ImageArgs, const double*, double2*);

template <int N, int FMT>
AdjKernel adj_nf(bool many, bool table) {
  if (many) return table ? epic_adjoint_pair<N, FMT, kPairMaxAnt, true> : epic_adjoint_pair<N, FMT, kPairMaxAnt, false>;
  return table ? epic_adjoint_pair<N, FMT, 1, true> : epic_adjoint_pair<N, FMT, 1, false>;
}

template <int N>
cudaError_t adj_launch(const ImageArgs& a, const double* dldi, double2* dldw, cudaStream_t s) {
  constexpr int BT = PCfg<N>::BT;
  const AdjKernel k = a.input_fmt ? adj_nf<N, 1>(a.n_ant > BT, a.gsmem != 0) : adj_nf<N, 0>(a.n_ant > BT, a.gsmem != 0);
  const cudaError_t e = allow_smem(k);
  if (e != cudaSuccess) return e;
  k<<<a.grid, BT, a.smem, s>>>(a, dldi, dldw);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_adjoint_pair(int n, const ImageArgs& a, const double* dldi, double2* dldw, cudaStream_t s) {
  switch (n) {
    case 16: return adj_launch<16>(a, dldi, dldw, s);
    case 32: return adj_launch<32>(a, dldi, dldw, s);
    case 64: return adj_launch<64>(a, dldi, dldw, s);
    case 128: return adj_launch<128>(a, dldi, dldw, s);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace epic
