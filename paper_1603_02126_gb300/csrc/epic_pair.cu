// Frame-pair forms of the fused imaging kernel (sm_103a, N = 16..128): two
// consecutive frames of one channel go through gain correction, gridding,
// both transforms and the square together, each value of the two frames one
// FP32 pair (fft::Cf2), so that every add and multiply of both frames is one
// packed instruction and every weight, twiddle and list entry is read once
// for both.
//
// The transforms are residue tasks (epic_residue.cuh) of 16 outputs.
//
// One persistent launch images a batch.  Every CTA takes an equal share of
// the estimated cost of the (channel, frame pair) list, so that no last wave
// is left and an image block is flushed once per channel and share.  Shared
// memory holds the grid of a frame pair, its row spectra and E' = E / g.
// Gridding (Eq. 9) gives each lane one grid cell, the cells sorted by their
// number of taps so that the 32 lanes of a slice run equally long.
//
// What bounds it: no unit is full (64 channels x 4096 4-bit samples of 256
// antennas, 128 x 128: issue slots 51 %, FP32 pipe 51 %, shared-memory pipe
// 46 %); 16 warps wait in turn for the FP32 pipe and for the shared-memory
// loads and dependent steps of their tasks (stalls per issue: wait 1.5, not
// selected 1.3, math throttle 1.3, barrier 1.1, short scoreboard 1.1).  A
// packed instruction takes two cycles (the scalar rate) and three with three
// distinct operands; one transform task of 40 inputs takes 252 SM cycles with
// 16 warps resident (DFT 75, twiddles 37, square 20, the rest the input sum and
// its loads), 42 tasks per pair of the 256-antenna station: three quarters of
// the time.  64 channels x 10^4 samples: 15.3 ms against 19.2 for one frame per
// FP32 value with an exchange through shared memory (63 % of the issue slots,
// 42 % of the FP32 pipe); 128 samples 0.264 against 0.363 ms; 248 antennas,
// 64 x 64, 15 channels, 1023 complex64 samples 0.310 against 0.425; 32 antennas,
// 32 x 32, 2000 samples 37.4 against 53.1 us (with the update).
#include "epic_fft.cuh"
#include "epic_internal.h"
#include "epic_pair.cuh"
#include "epic_smem.cuh"

#include <cstdint>

namespace epic {
namespace {

using fft::cmul;
using fft::f2_pack;

// Multiple-pixel EPICal: the calibration pixels among a thread's outputs
// (slot mask, index of its first tap) of frame pair p.
__device__ __forceinline__ void store_taps(const ImageArgs& A, const Cf2 (&y)[16], int entry, long long p, int c) {
  const uint2 tb = __ldg(A.ptab + entry);
  if (!tb.x) return;
  float2* d0 = A.ptap + (static_cast<size_t>(2 * p) * A.n_chan + c) * A.npix;
  float2* d1 = 2 * p + 1 < A.n_time ? d0 + static_cast<size_t>(A.n_chan) * A.npix : nullptr;
  const float2* ph = A.pph + static_cast<size_t>(c) * A.npix;
#pragma unroll
  for (int m = 0; m < 16; ++m)
    if ((tb.x >> m) & 1u) {
      const int pi = static_cast<int>(tb.y) + __popc(tb.x & ((1u << m) - 1u));
      store_pixel(y, m, __ldg(ph + pi), d0 + pi, d1 ? d1 + pi : nullptr);
    }
}

// One antenna's EPICal sums over a run of pairs (FP32; FP64 across).
struct Corr {
  float2 k;
  float p;
  __device__ __forceinline__ void add(float2 e, float2 q) {
    k.x += e.x * q.x + e.y * q.y;
    k.y += e.y * q.x - e.x * q.y;
    p += e.x * e.x + e.y * e.y;
  }
  __device__ __forceinline__ void flush(const ImageArgs& A, int c, int a) {
    const size_t o = static_cast<size_t>(c) * A.n_ant + a;
    if (__ldg(A.cellf + o) >= 0) {
      atomicAdd(&A.kacc[o].x, static_cast<double>(k.x));
      atomicAdd(&A.kacc[o].y, static_cast<double>(k.y));
      atomicAdd(A.pacc + o, static_cast<double>(p));
    }
    k = make_float2(0.f, 0.f);
    p = 0.f;
  }
};

// Two phases per frame pair, a CTA barrier after each:
//   rows      tasks (grid row, r): grid -> spectra; the last warps also
//             correlate the previous pair with the calibrator pixel (Eqs. 12,
//             15) and form E' of the next pair (Eq. 8);
//   columns   tasks (column kx, r): spectra -> |E|^2 in registers (Eq. 10),
//             calibrator pixel stored; then the next pair is gridded.
// LONG: runs of kPairRun pairs known at compile time (15.25 against 15.4 ms for
// 64 channels x 10^4 samples), the correlation flushed with the image; else
// A.run pairs per partial image and A.corr_mask + 1 per partial correlation.
template <int N, int FMT, int MAXA, bool TS, bool LONG>
__global__ void __launch_bounds__(PCfg<N>::BT, PCfg<N>::PER_SM) epic_image_pair(const ImageArgs A) {
  using G = PGeo<N>;
  constexpr int BT = G::BT, NR = G::NR, TASKS = G::TASKS, ROUNDS = G::ROUNDS;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int rs = A.rs, gs = A.gs, Na = A.n_ant;
  Cf2* Tt = reinterpret_cast<Cf2*>(smem_raw);              // [N][rs] row spectra, transposed
  Cf2* grid = Tt + N * rs;                                 // [rows_alloc][gs]
  Cf2* Es = grid + A.rows_alloc * gs;                      // [Na + 1] E' (entry Na is zero)
  float2* tw = reinterpret_cast<float2*>(Es + Na + 1);     // [16][NR]
  float2* wq = tw + N;                                     // [16][NR]
  float2* pixs = wq + N;                                   // [2] calibrator pixel of the pair
  int2* sslice = reinterpret_cast<int2*>(pixs + 2);        // [max_slices] (TS)
  uint2* sent = reinterpret_cast<uint2*>(sslice + A.max_slices);   // [max_ent] (TS)
  int* scell = reinterpret_cast<int*>(sent + A.max_ent);   // [max_slices * 32] (TS)

  const int tid = threadIdx.x;
  const int aw = (BT - 32 - (tid & ~31)) + (tid & 31);     // antenna of this thread: the last warps first
  residue_tables<N, NR>(A.twid, tw, wq, BT);
  if (tid == 0) Es[Na] = Cf2{0ull, 0ull};

  const long long T = A.n_time;
  const int C = A.n_chan;
  const Share share(A.pcost, A.n_chan, 1, (A.n_time + 1) / 2);
  int cur = -1;
  for (int c = share.first(C); c < C && share.before(c) < share.hi; ++c) {
    const long long p_lo = share.pair_at(share.lo, c), p_hi = share.pair_at(share.hi, c);
    const Chan ch = channel<TS>(A, c, sslice, scell, sent);
    for (long long pa = p_lo; pa < p_hi; pa += LONG ? kPairRun : A.run) {
      const long long pe = pa + (LONG ? kPairRun : A.run), pb = pe < p_hi ? pe : p_hi;
      __syncthreads();                                     // the previous run's shared memory is free
      if (cur != c) {
        if (TS) load_lists<BT>(A, c, sslice, scell, sent);
        for (int i = tid; i < A.rows_alloc * gs; i += BT) grid[i] = Cf2{0ull, 0ull};   // cells without taps stay zero
        const int pad = ch.R4 - ch.R;
        for (int i = tid; i < N * pad; i += BT) Tt[(i / pad) * rs + ch.R + i % pad] = Cf2{0ull, 0ull};
        cur = c;
      }
      Corr corr[MAXA];
      unsigned hist[MAXA];                                 // 4-bit voltages of the last two pairs, 16 bits each
#pragma unroll
      for (int i = 0; i < MAXA; ++i) {
        corr[i] = Corr{make_float2(0.f, 0.f), 0.f};
        hist[i] = 0;
      }
      // E' of pair p (a missing second frame is zero)
      auto form_e = [&](long long p) {
#pragma unroll
        for (int i = 0; i < MAXA; ++i) {
          const int a = aw + BT * i;
          hist[i] <<= 16;
          if (a < Na && p < pb) {
            const size_t idx = (static_cast<size_t>(2 * p) * C + c) * Na + a, next = static_cast<size_t>(C) * Na;
            const bool two = 2 * p + 1 < T;
            const float2 w = __ldg(ch.wg + a);
            float2 v0, v1 = make_float2(0.f, 0.f);
            if (FMT == 0) {
              const unsigned char* v = static_cast<const unsigned char*>(A.volt) + idx;
              const unsigned b = __ldg(v) | (two ? static_cast<unsigned>(__ldg(v + next)) << 8 : 0u);
              hist[i] |= b;
              v0 = unpack_ci4(b, ch.vs);
              v1 = unpack_ci4(b >> 8, ch.vs);
            } else {
              v0 = pair_volt<FMT>(A.volt, idx, ch.vs);
              if (two) v1 = pair_volt<FMT>(A.volt, idx + next, ch.vs);
            }
            const float2 e0 = cmul(v0, w), e1 = cmul(v1, w);
            Es[a] = Cf2{f2_pack(e0.x, e1.x), f2_pack(e0.y, e1.y)};
          }
        }
      };
      // correlation of pair p, the last but one formed, with the calibrator
      // pixel (Eqs. 12, 15); a missing second frame adds zero
      auto correlate = [&](long long p) {
#pragma unroll
        for (int i = 0; i < MAXA; ++i) {
          const int a = aw + BT * i;
          if (a < Na) {
#pragma unroll
            for (int f = 0; f < 2; ++f) {
              if (FMT == 0)
                corr[i].add(unpack_ci4(hist[i] >> (16 + 8 * f), ch.vs), pixs[f]);
              else if (2 * p + f < T)
                corr[i].add(pair_volt<FMT>(A.volt, (static_cast<size_t>(2 * p + f) * C + c) * Na + a, ch.vs), pixs[f]);
            }
          }
        }
      };
      auto flush_corr = [&]() {
#pragma unroll
        for (int i = 0; i < MAXA; ++i)
          if (aw + BT * i < Na) corr[i].flush(A, c, aw + BT * i);
      };
      float acc[ROUNDS][16];
#pragma unroll
      for (int i = 0; i < ROUNDS; ++i)
#pragma unroll
        for (int m = 0; m < 16; ++m) acc[i][m] = 0.f;

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
        if (A.do_cal && p > pa) {
          correlate(p - 1);
          if (!LONG && (p & A.corr_mask) == 0) flush_corr();
        }
        form_e(p + 1);
        __syncthreads();
        // ---- columns ----
#pragma unroll
        for (int i = 0; i < ROUNDS; ++i) {
          const int task = tid + BT * i;
          if (TASKS >= BT || task < TASKS) {
            const int kx = task / NR, r = task % NR;
            Cf2 y[16];
            dft_task<16, NR>(Tt + kx * rs, ch.R4, r, tw, wq, y);
            square_add(y, acc[i]);
            if (A.do_cal && kx == A.k0x && r == A.k0y % NR) store_pixel(y, A.k0y / NR, ch.pph, pixs, pixs + 1);
            if (A.npix) store_taps(A, y, task, p, c);
          }
        }
        if (p + 1 < pb) grid_pair<BT>(ch.cell, ch.slice, ch.ent, ch.nslice, Es, grid);
        __syncthreads();
      }
      if (A.do_cal) correlate(pb - 1);

      // flush the run's partial sums (FP32 over the run, FP64 across)
      double* img = A.image + static_cast<size_t>(c) * N * N;
#pragma unroll
      for (int i = 0; i < ROUNDS; ++i) {
        const int task = tid + BT * i;
        if (TASKS >= BT || task < TASKS) {
          const int kx = task / NR, r = task % NR;
#pragma unroll
          for (int m = 0; m < 16; ++m)
            atomicAdd(img + (NR * m + r) * N + kx, static_cast<double>(acc[i][m]) * A.img_scale);
        }
      }
      if (A.do_cal) flush_corr();
    }
  }
}

using PairKernel = void (*)(const ImageArgs);

template <int N, int FMT, bool LONG>
PairKernel pair_kernel_nfl(bool many, bool table) {
  if (many)
    return table ? epic_image_pair<N, FMT, kPairMaxAnt, true, LONG> : epic_image_pair<N, FMT, kPairMaxAnt, false, LONG>;
  return table ? epic_image_pair<N, FMT, 1, true, LONG> : epic_image_pair<N, FMT, 1, false, LONG>;
}

template <int N>
PairKernel pair_kernel_n(int fmt, bool many, bool table, bool run) {
  if (run) return fmt ? pair_kernel_nfl<N, 1, true>(many, table) : pair_kernel_nfl<N, 0, true>(many, table);
  return fmt ? pair_kernel_nfl<N, 1, false>(many, table) : pair_kernel_nfl<N, 0, false>(many, table);
}

// run: partial images of kPairRun pairs.
PairKernel pair_kernel(int n, int fmt, bool many, bool table, bool run) {
  switch (n) {
    case 16: return pair_kernel_n<16>(fmt, many, table, run);
    case 32: return pair_kernel_n<32>(fmt, many, table, run);
    case 64: return pair_kernel_n<64>(fmt, many, table, run);
    case 128: return pair_kernel_n<128>(fmt, many, table, run);
    default: return nullptr;
  }
}

}  // namespace

int pair_threads(int n) {
  switch (n) {
    case 16: return PCfg<16>::BT;
    case 32: return PCfg<32>::BT;
    case 64: return PCfg<64>::BT;
    case 128: return PCfg<128>::BT;
    default: return 0;
  }
}

int pair_col_rounds(int n) {
  const int bt = pair_threads(n);
  if (!bt) return 0;
  const int tasks = n * n / 16;
  return tasks < bt ? 1 : tasks / bt;
}

bool pair_pixel_owner(int n, int kx, int ky, PixelOwner* out) {
  const int bt = pair_threads(n);
  if (!bt || kx < 0 || ky < 0 || kx >= n || ky >= n) return false;
  const int nr = n / 16, task = kx * nr + ky % nr;
  out->round = task / bt;
  out->thread = task % bt;
  out->slot = ky / nr;
  return true;
}

// Row stride of the spectra: room for the rows rounded up to 4 (to 8 for the
// adjoint, whose way back permutes blocks of 8), and a
// stride that keeps the row phase's stores free of bank conflicts (a quarter
// warp stores NR columns of 8 / NR neighbouring rows, 16 bytes each).
int pair_rs(int n, int rows, bool adjoint) {
  const int nr = n / 16;
  int rs = adjoint ? (rows + 7) & ~7 : (rows + 3) & ~3;
  const int step = 8 / nr;                       // rows per quarter warp
  while (!(nr == 1 || (rs % step == 0 && (rs / step) % 2 == 1))) ++rs;
  return rs;
}

size_t pair_smem_bytes(int n, int n_ant, int rows, int gs, int max_slices, int max_ent, bool adjoint) {
  const size_t cells = static_cast<size_t>(n) * pair_rs(n, rows, adjoint) + static_cast<size_t>(rows) * gs + n_ant + 1;
  return cells * 16 + (2 * static_cast<size_t>(n) + 2) * sizeof(float2) +
         static_cast<size_t>(max_slices) * (sizeof(int2) + 32 * sizeof(int)) +
         static_cast<size_t>(max_ent) * sizeof(uint2);
}

cudaError_t pair_prepare(int n, int n_ant, bool table, size_t smem, int* ctas_per_sm) {
  const int bt = pair_threads(n);
  cudaError_t e = cudaSuccess;
  for (int k = 0; k < 4 && e == cudaSuccess; ++k) e = allow_smem(pair_kernel(n, k & 1, n_ant > bt, table, k > 1));
  if (e != cudaSuccess) return e;
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(ctas_per_sm, pair_kernel(n, 0, n_ant > bt, table, false), bt, smem);
}

cudaError_t launch_pair(int n, const ImageArgs& a, cudaStream_t s) {
  const int bt = pair_threads(n);
  const PairKernel k = pair_kernel(n, a.input_fmt, a.n_ant > bt, a.gsmem != 0, a.run == kPairRun);
  if (!k) return cudaErrorInvalidValue;
  k<<<a.grid, bt, a.smem, s>>>(a);
  return cudaGetLastError();
}

}  // namespace epic
