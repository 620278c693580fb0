// Host arithmetic of the frame-pair forms' batches and shares (no CUDA).
#pragma once

#include <algorithm>
#include <cstddef>
#include <vector>

namespace epic {

// Batch of the wide frame-pair form: samples per batch and channels per
// launch.  All samples that fit with every channel, or kWideTime of them with
// fewer channels (an image block is added to once per batch and share).  The
// whole scratch budget is used: a launch costs its start and its tail, and
// batches that stay in L2 were slower (1024 antennas, 256 x 256: 48 MB 29.5,
// 200 MB 20.7, 512 MB 17.9, 2 GB 16.6 ms).
struct WideBatch {
  long long nt = 0;              // even: the kernels take the samples in pairs
  int nc = 0;
  size_t spec_n = 0, need = 0;   // float2 of the spectra, of the whole scratch
};

// C channels of N columns of rs rows, a budget of at least one frame pair of
// one channel, at most tune_nt samples (0: no such limit).
inline WideBatch wide_batch(int C, int N, int rs, size_t budget, int tune_nt, long long n_time) {
  constexpr long long kWideTime = 256;
  const size_t chan_t = static_cast<size_t>(N) * rs * 8;   // bytes of one sample of one channel
  const auto even_up = [](long long v) { return (v + 1) / 2 * 2; };
  const auto even_down = [](long long v) { return v / 2 * 2; };
  WideBatch b;
  b.nt = std::min(even_up(n_time),
                  std::max<long long>(kWideTime, even_down(static_cast<long long>(budget / (chan_t * C)))));
  if (tune_nt > 0) b.nt = std::max<long long>(2, std::min(b.nt, even_down(tune_nt)));
  b.nt = std::max<long long>(2, std::min(b.nt, even_down(static_cast<long long>(budget / chan_t))));
  const long long fit = static_cast<long long>(budget / (chan_t * static_cast<size_t>(b.nt)));
  const int most = static_cast<int>(std::max<long long>(1, std::min<long long>(fit, C)));
  const int groups = (C + most - 1) / most;
  b.nc = (C + groups - 1) / groups;
  b.spec_n = static_cast<size_t>(b.nt) * b.nc * N * rs;
  b.need = b.spec_n + static_cast<size_t>(b.nt) * C;
  return b;
}

// float2 of a scratch that every call of a plan fits, whatever its n_time.
inline size_t wide_scratch(int C, int N, int rs, size_t budget) {
  const size_t frames = budget / (static_cast<size_t>(N) * rs * 8);
  const long long nt = wide_batch(C, N, rs, budget, 0, 1LL << 40).nt;
  return frames * N * rs + static_cast<size_t>(nt) * C;
}

// [n + 1] prefix sums of the costs by which CTAs share the channels, scaled
// down together where their sum would not fit.
inline std::vector<int> cost_prefix(const std::vector<long long>& cost) {
  const auto sum_of = [&](int shift) {
    long long s = 0;
    for (long long c : cost) s += std::max(1LL, c >> shift);
    return s;
  };
  int shift = 0;
  while (sum_of(shift) > (1LL << 30) && shift < 40) ++shift;
  std::vector<int> out{0};
  for (long long c : cost) out.push_back(out.back() + static_cast<int>(std::max(1LL, c >> shift)));
  return out;
}

}  // namespace epic
