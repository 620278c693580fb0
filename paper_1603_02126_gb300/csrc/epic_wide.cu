// Frame-pair form of the plain FP32 path for N = 256 and 512, and of N = 128
// where the footprint does not fit one SM (sm_103a): the row spectra of a
// batch of frames go through HBM, two frames per FP32 pair.
//
//   wide_rows    per (channel, frame pair): E' = E / g (Eq. 8) of every
//                antenna into shared memory, then by blocks of RB grid rows
//                the gridding (Eq. 9) into shared memory and the row
//                transforms (residue tasks of 32 outputs), written transposed
//                to spec[pair][c][kx][row];
//   wide_cols    per (channel, block of NCOL columns, range of pairs): the
//                next pair's block arrives by one bulk copy while the current
//                one is transformed (Eq. 10); |E|^2 stays in registers, the
//                calibrator pixel is stored per frame.
// The correlation kernel of the plain path follows.
//
// What bounds it: latency with the 8 warps per SM that 32-output tasks leave
// (255 registers), the FP32 pipe at 65 % in the column kernel (packed
// instructions take two cycles, three with distinct operands), at 27 % in the
// row kernel, whose loads and gridding share the shared-memory pipe (51 %).
// 8192 frames of 1024 antennas, 256 x 256: rows 0.47, columns 0.55 ms, HBM 2.7
// and 2.6 TB/s.  16-output tasks would need twice the loads; three CTAs per SM
// (168 registers) were slower in the row kernel (17.0 against 16.6 ms).  4096
// samples of 32 channels: 16.8 ms against 38.2 for the one-frame kernels; 2048
// antennas, 512 x 512, 128 complex64 samples of 256 channels 24.0 against 53.3;
// 200 antennas on 76 of 128 grid rows, 16 channels, 2000 samples 1.34 against
// 1.57 for the one-frame fused kernel.
//
// Gridding: one lane per grid cell; the cells of a row block sorted by their
// number of taps in slices of 32 (empty cells last, stored as zeros, since
// the block buffer is used again), the lists of a block one contiguous piece
// of memory that is copied to shared memory a block ahead.
#include "epic_bulk.cuh"
#include "epic_fft.cuh"
#include "epic_internal.h"
#include "epic_lists.cuh"
#include "epic_residue.cuh"
#include "epic_smem.cuh"

#include <cstdint>

namespace epic {
namespace {

using fft::Cf2;
using fft::cmul;
using fft::f2_pack;

constexpr int kWBT = 128;          // threads of the row kernel; two CTAs per SM (255 registers each)
constexpr int kWP = 32;            // outputs per task

template <int N>
struct WGeo {
  static constexpr int NR = N / kWP;                 // residues
  static constexpr int RB = kWBT / NR;               // grid rows per block
  static constexpr int CT = N == 128 ? 64 : 128;     // threads of the column kernel, 256 per SM
  static constexpr int NCOL = CT / NR;               // columns per block
  static constexpr int CB = N / NCOL;                // column blocks
};

// Column stride of a channel's spectra: its rows rounded up to 4, and 4 mod 8
// so that the two columns of neighbouring quarter warps lie in different
// shared-memory banks.
__host__ __device__ inline int wide_stride(int rows) {
  const int r4 = (rows + 3) & ~3;
  return r4 % 8 ? r4 : r4 + 4;
}

__device__ __forceinline__ void grid_block(const unsigned char* lists, const Cf2* Es, Cf2* grid) {
  const BlockLists hd = *reinterpret_cast<const BlockLists*>(lists);
  const int2* slice = reinterpret_cast<const int2*>(lists + sizeof(BlockLists));
  const uint16_t* cell = reinterpret_cast<const uint16_t*>(lists + hd.cells);
  const uint2* ent = reinterpret_cast<const uint2*>(lists + hd.ents);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int k = 0; k * (kWBT / 32) < hd.nslice; ++k) {
    const int sl = slice_of(k, warp, kWBT / 32);
    if (sl >= hd.nslice) break;
    const int2 s = slice[sl];
    const unsigned at = cell[sl * 32 + lane];
    const Cf2 sum = sum_taps(ent + s.x + lane, s.y, Es);
    if (at != 0xffffu) grid[at] = sum;
  }
}

template <int N, int FMT>
__global__ void __launch_bounds__(kWBT, 2) wide_rows_kernel(const WideArgs W, long long t0, int nt) {
  using G = WGeo<N>;
  constexpr int NR = G::NR, RB = G::RB;
  const UnfusedArgs& A = W.u;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  const int Na = A.n_ant, C = A.n_chan, gs = W.gs, tid = threadIdx.x;
  unsigned char* lists = smem_raw;                           // [2][max_lists] of the current and the next block
  Cf2* grid = reinterpret_cast<Cf2*>(lists + 2 * static_cast<size_t>(W.max_lists));   // [RB][gs]
  Cf2* Es = grid + RB * gs;                                  // [Na + 1] E' (entry Na is zero)
  float2* tw = reinterpret_cast<float2*>(Es + Na + 1);       // [32][NR]
  float2* wq = tw + N;                                       // [NR][NR]
  __shared__ uint64_t bars[2];
  __shared__ int abort_flag;
  residue_tables<N, NR>(A.twid, tw, wq, kWBT);
  if (tid == 0) {
    Es[Na] = Cf2{0ull, 0ull};
    mbar_init_one(bars, 2);
    abort_flag = 0;
  }
  __syncthreads();

  const long long P = (nt + 1) / 2;
  // E' of pair p of channel c (a missing second frame is zero)
  auto form_e = [&](int c, long long p) {
    const float vs = A.vscale ? __ldg(A.vscale + c) : 1.0f;
    const float2* wg = A.wgain + static_cast<size_t>(c) * Na;
    const size_t i0 = (static_cast<size_t>(t0 + 2 * p) * C + c) * Na;
    const bool two = 2 * p + 1 < nt;
#pragma unroll 4
    for (int a = tid; a < Na; a += kWBT) {
      const float2 w = __ldg(wg + a);
      const float2 e0 = cmul(pair_volt<FMT>(A.volt, i0 + a, vs), w);
      float2 e1 = make_float2(0.f, 0.f);
      if (two) e1 = cmul(pair_volt<FMT>(A.volt, i0 + static_cast<size_t>(C) * Na + a, vs), w);
      Es[a] = Cf2{f2_pack(e0.x, e1.x), f2_pack(e0.y, e1.y)};
    }
  };
  auto load_lists = [&](int c, int b, int slot) {
    const int2 at = __ldg(W.lists_at + c * W.nb_max + b);    // (offset, bytes) / 16
    bulk_load(smem_addr(lists + static_cast<size_t>(slot) * W.max_lists), W.lists + static_cast<size_t>(at.x) * 16,
              static_cast<uint32_t>(at.y) * 16u, smem_addr(bars + slot));
  };

  // This CTA's share: row blocks [k_lo, k_hi) of each channel it reaches,
  // block k = pair * blocks per pair + row block, cost[c + 1] - cost[c] per
  // pair and the blocks of a channel equal parts of it.
  const int* cost = W.row_cost;
  const int c_end = W.c0 + W.nc;
  const long long base = __ldg(cost + W.c0);
  const long long total = (__ldg(cost + c_end) - base) * P, g = gridDim.x, bid = blockIdx.x;
  const long long lo = total / g * bid + total % g * bid / g;
  const long long hi = total / g * (bid + 1) + total % g * (bid + 1) / g;
  auto blocks_of = [&](int c) { return (__ldg(W.win4 + c).y + RB - 1) / RB; };
  auto block_at = [&](long long pos, int c, int nb) {        // first block of channel c at or after position pos
    const long long w = __ldg(cost + c + 1) - __ldg(cost + c), off = pos - (__ldg(cost + c) - base) * P;
    const long long k = off <= 0 ? 0 : (off * nb + w - 1) / w;
    return k > P * nb ? P * nb : k;
  };

  const int lane = tid & 31, warp = tid >> 5;
  // a warp transforms 8 rows x 4 residues: its loads have two addresses per
  // quarter warp, its 16-byte stores whole 128-byte runs of a column
  const int lrow = warp / (NR / 4) * 8 + (lane >> 2), r = warp % (NR / 4) * 4 + (lane & 3);
  unsigned it = 0;                                           // row blocks so far: lists slot it & 1
  bool first = true;
  for (int c = W.c0; c < c_end; ++c) {
    if ((__ldg(cost + c + 1) - base) * P <= lo) continue;
    if ((__ldg(cost + c) - base) * P >= hi) break;
    const int nb = blocks_of(c);
    const long long k_lo = block_at(lo, c, nb), k_hi = block_at(hi, c, nb);
    if (k_lo >= k_hi) continue;
    const int4 wn = __ldg(W.win4 + c);                       // (y0, rows, x0, cols)
    const int R = wn.y, R4 = (R + 3) & ~3, W4 = (wn.w + 3) & ~3, S = wide_stride(R);
    if (first) {
      if (tid == 0) load_lists(c, static_cast<int>(k_lo % nb), 0);
      form_e(c, k_lo / nb);
      first = false;
    }
    // the columns past this channel's window, read as zeros by the tasks
    for (int i = tid; i < RB * (W4 - wn.w); i += kWBT) grid[i / (W4 - wn.w) * gs + wn.w + i % (W4 - wn.w)] = Cf2{0ull, 0ull};
    // the next channel of this share, for what is fetched ahead
    const bool more = c + 1 < c_end && block_at(hi, c + 1, blocks_of(c + 1)) > 0;
    __syncthreads();
    long long p = k_lo / nb;
    int b = static_cast<int>(k_lo - p * nb);
    for (long long k = k_lo; k < k_hi; ++k, ++it) {
      const int slot = it & 1;
      const bool last = b + 1 == nb;                         // of the pair
      if (tid == 0) {                                        // the other slot was read out two barriers ago
        if (k + 1 < k_hi) load_lists(c, last ? 0 : b + 1, slot ^ 1);
        else if (more) load_lists(c + 1, 0, slot ^ 1);
      }
      if (!mbar_wait_bounded(smem_addr(bars + slot), (it >> 1) & 1u)) {
        abort_flag = 1;
        atomicExch(A.err, 1);
      } else {
        grid_block(lists + static_cast<size_t>(slot) * W.max_lists, Es, grid);
      }
      __syncthreads();
      if (*reinterpret_cast<volatile int*>(&abort_flag)) {
        // let the copy in flight land (bounded) before the CTA exits
        if (tid == 0 && (k + 1 < k_hi || more)) mbar_wait_bounded(smem_addr(bars + (slot ^ 1)), ((it + 1) >> 1) & 1u);
        return;
      }
      const int row = b * RB + lrow;
      if (row < R4) {
        Cf2 y[kWP];
        if (row < R) {
          dft_task<kWP, NR>(grid + lrow * gs, W4, r, tw, wq, y);
        } else {
#pragma unroll
          for (int m = 0; m < kWP; ++m) y[m] = Cf2{0ull, 0ull};
        }
        Cf2* dst = reinterpret_cast<Cf2*>(A.spec) + (static_cast<size_t>(p) * W.nc + (c - W.c0)) * N * A.rs +
                   static_cast<size_t>(r) * S + row;
#pragma unroll
        for (int m = 0; m < kWP; ++m) dst[static_cast<size_t>(NR * m) * S] = y[m];
      }
      // after the pair's last gridding the next pair's E' takes its place
      if (k + 1 < k_hi) {
        if (last) form_e(c, p + 1);
      } else if (more) {
        form_e(c + 1, 0);
      }
      if (last) {
        b = 0;
        ++p;
      } else {
        ++b;
      }
      __syncthreads();
    }
  }
}

template <int N>
__global__ void __launch_bounds__(WGeo<N>::CT, 256 / WGeo<N>::CT) wide_cols_kernel(const WideArgs W, int nt) {
  using G = WGeo<N>;
  constexpr int NR = G::NR, NCOL = G::NCOL, CB = G::CB;
  const UnfusedArgs& A = W.u;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  const int C = A.n_chan, rs = A.rs, tid = threadIdx.x;
  Cf2* slots = reinterpret_cast<Cf2*>(smem_raw);             // [2][NCOL][rs]
  float2* tw = reinterpret_cast<float2*>(slots + 2 * NCOL * rs);   // [32][NR]
  float2* wq = tw + N;                                       // [NR][NR]
  __shared__ uint64_t bars[2];
  __shared__ int abort_flag;
  residue_tables<N, NR>(A.twid, tw, wq, G::CT);
  if (tid == 0) {
    mbar_init_one(bars, 2);
    abort_flag = 0;
  }
  __syncthreads();

  const long long P = (nt + 1) / 2;
  // parts (channel, column block) of the channels [c0, c0 + nc)
  const Share share(W.col_cost + W.c0, W.nc, CB, P);
  const int j = tid / NR, r = tid % NR;                      // column of the block, output residue
  unsigned it = 0;                                           // blocks transformed so far: slot it & 1
  for (int v = share.first(W.nc * CB); v < W.nc * CB && share.before(v) < share.hi; ++v) {
    const int c = W.c0 + v / CB, kx = v % CB * NCOL + j;
    const long long p_lo = share.pair_at(share.lo, v), p_hi = share.pair_at(share.hi, v);
    if (p_lo >= p_hi) continue;
    const int R = __ldg(W.win4 + c).y, R4 = (R + 3) & ~3, S = wide_stride(R);
    const size_t stride = static_cast<size_t>(W.nc) * N * rs;   // spectra of one pair
    const Cf2* src = reinterpret_cast<const Cf2*>(A.spec) + static_cast<size_t>(c - W.c0) * N * rs +
                     static_cast<size_t>(kx - j) * S;
    const uint32_t bytes = static_cast<uint32_t>(NCOL * S) * 16u;
    auto load = [&](long long p, int slot) {
      bulk_load(smem_addr(slots + static_cast<size_t>(slot) * NCOL * rs), src + static_cast<size_t>(p) * stride, bytes,
                smem_addr(bars + slot));
    };
    const bool pix = A.do_cal && kx == A.k0x && r == A.k0y % NR;
    if (tid == 0) load(p_lo, it & 1);                        // both slots are free here
    for (long long pa = p_lo; pa < p_hi; pa += W.run) {
      const long long pb = pa + W.run < p_hi ? pa + W.run : p_hi;
      float acc[kWP];
#pragma unroll
      for (int m = 0; m < kWP; ++m) acc[m] = 0.f;
      for (long long p = pa; p < pb; ++p, ++it) {
        const int slot = it & 1;
        if (tid == 0 && p + 1 < p_hi) load(p + 1, slot ^ 1); // read out before the last barrier
        if (!mbar_wait_bounded(smem_addr(bars + slot), (it >> 1) & 1u)) {
          abort_flag = 1;
          atomicExch(A.err, 1);
        } else {
          Cf2 y[kWP];
          dft_task<kWP, NR>(slots + static_cast<size_t>(slot) * NCOL * rs + j * S, R4, r, tw, wq, y);
          square_add(y, acc);
          if (pix) {
            float2* q = A.pix + static_cast<size_t>(2 * p) * C + c;
            store_pixel(y, A.k0y / NR, __ldg(A.pixph + c), q, 2 * p + 1 < nt ? q + C : nullptr);
          }
        }
        __syncthreads();
        if (*reinterpret_cast<volatile int*>(&abort_flag)) {
          // let the copy in flight land (bounded) before the CTA exits
          if (tid == 0 && p + 1 < p_hi) mbar_wait_bounded(smem_addr(bars + (slot ^ 1)), ((it + 1) >> 1) & 1u);
          return;
        }
      }
      double* img = A.image + static_cast<size_t>(c) * N * N + kx;
#pragma unroll
      for (int m = 0; m < kWP; ++m)
        atomicAdd(img + static_cast<size_t>(NR * m + r) * N, static_cast<double>(acc[m]) * A.img_scale);
    }
  }
}

template <int N>
size_t rows_smem(const WideArgs& w) {
  return 2 * static_cast<size_t>(w.max_lists) +
         (static_cast<size_t>(WGeo<N>::RB) * w.gs + w.u.n_ant + 1) * sizeof(Cf2) + 2 * N * sizeof(float2);
}

template <int N>
size_t cols_smem(const WideArgs& w) {
  return 2 * static_cast<size_t>(WGeo<N>::NCOL) * w.u.rs * sizeof(Cf2) + 2 * N * sizeof(float2);
}

template <int N>
cudaError_t prepare_n(const WideArgs& w, int fmt, int* rows_per_sm, int* cols_per_sm) {
  int dev = 0, most = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (e != cudaSuccess) return e;
  *rows_per_sm = *cols_per_sm = 0;
  const int room = most - 256;                               // static shared memory beside the dynamic
  if (rows_smem<N>(w) > static_cast<size_t>(room) || cols_smem<N>(w) > static_cast<size_t>(room)) return cudaSuccess;
  auto rk = fmt ? wide_rows_kernel<N, 1> : wide_rows_kernel<N, 0>;
  e = allow_smem(rk);
  if (e == cudaSuccess) e = allow_smem(wide_cols_kernel<N>);
  if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(rows_per_sm, rk, kWBT, rows_smem<N>(w));
  if (e == cudaSuccess)
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(cols_per_sm, wide_cols_kernel<N>,
                                                      WGeo<N>::CT, cols_smem<N>(w));
  return e;
}

template <int N>
cudaError_t launch_n(const WideArgs& w, long long t0, int nt, cudaStream_t s) {
  const long long pairs = static_cast<long long>((nt + 1) / 2) * w.nc;
  if (w.u.input_fmt) wide_rows_kernel<N, 1><<<w.rows_grid, kWBT, rows_smem<N>(w), s>>>(w, t0, nt);
  else wide_rows_kernel<N, 0><<<w.rows_grid, kWBT, rows_smem<N>(w), s>>>(w, t0, nt);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  const long long cu = pairs * WGeo<N>::CB;
  const long long cg = cu < w.cols_ctas ? cu : w.cols_ctas;
  wide_cols_kernel<N><<<static_cast<unsigned>(cg), WGeo<N>::CT, cols_smem<N>(w), s>>>(w, nt);
  return cudaGetLastError();
}

}  // namespace

bool wide_supported(int n) { return n == 128 || n == 256 || n == 512; }

int wide_row_block(int n) { return n == 128 ? WGeo<128>::RB : n == 256 ? WGeo<256>::RB : n == 512 ? WGeo<512>::RB : 0; }

cudaError_t wide_prepare(const WideArgs& w, int fmt, int* rows_per_sm, int* cols_per_sm) {
  switch (w.u.grid_n) {
    case 128: return prepare_n<128>(w, fmt, rows_per_sm, cols_per_sm);
    case 256: return prepare_n<256>(w, fmt, rows_per_sm, cols_per_sm);
    case 512: return prepare_n<512>(w, fmt, rows_per_sm, cols_per_sm);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_wide_batch(const WideArgs& w, long long t0, int nt, cudaStream_t s) {
  switch (w.u.grid_n) {
    case 128: return launch_n<128>(w, t0, nt, s);
    case 256: return launch_n<256>(w, t0, nt, s);
    case 512: return launch_n<512>(w, t0, nt, s);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace epic
