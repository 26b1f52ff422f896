// lj_teams.cuh -- team-size variants and per-team shared-memory carving,
// shared by the kernel translation units.
#pragma once
#include <type_traits>
#include <cuda_runtime.h>
#include "lj_device.cuh"

namespace ljd {

// Team size T and atom slots per thread A for clusters of up to max_n atoms.
// Thread `rank` owns atoms rank + a*T, a < A.
template <class F>
__host__ cudaError_t dispatch_team(int max_n, F&& f) {
  using std::integral_constant;
  if (max_n <= 32) return f(integral_constant<int, 32>{}, integral_constant<int, 1>{});
  if (max_n <= 64) return f(integral_constant<int, 32>{}, integral_constant<int, 2>{});
  if (max_n <= 128) return f(integral_constant<int, 64>{}, integral_constant<int, 2>{});
  if (max_n <= 256) return f(integral_constant<int, 128>{}, integral_constant<int, 2>{});
  if (max_n <= 512) return f(integral_constant<int, 256>{}, integral_constant<int, 2>{});
  if (max_n <= 1024) return f(integral_constant<int, 512>{}, integral_constant<int, 2>{});
  return cudaErrorInvalidValue;
}

__host__ __device__ constexpr int cta_threads_for(int T) { return T < 128 ? 128 : T; }

__host__ __device__ constexpr size_t align16(size_t b) { return (b + 15) & ~size_t(15); }

// How FP64 and double-float evaluations take every pair once, by the largest
// cluster of the launch, and the team's buffer for it:
//   up to kHalfMaxN atoms    half pairs, 24 bytes per pair;
//   up to kTileMinN          mixed precision: ring, 24 bytes per atom and shift of a
//                            chunk (4,096 clusters of 13..150 atoms: 17.1 ms, 19.1 with
//                            one-sided rows, which evaluate every pair twice; 3
//                            to 8 atom blocks leave warps idle in a tile round).
//                            FP64 path: no buffer, one-sided rows -- its results hang
//                            on the order of the sums (tri_pairs, lj_device.cuh);
//                            a ring takes 65.6 instead of 94.4 ms (Basin Hopping, 11
//                            walkers x 8, 5 steps, 77 atoms) but ends 8% of the
//                            trials with another status;
//   above                    32 x 32 tiles, 24 bytes per atom.
constexpr int kHalfMaxN = 64;
constexpr int kTileMinN = 256;
enum PairLayout : int { LAYOUT_HALF = 0, LAYOUT_TILES = 1, LAYOUT_RING = 2 };
__host__ __device__ constexpr int pair_layout(int max_n) {
  return max_n <= kHalfMaxN ? LAYOUT_HALF : max_n <= kTileMinN ? LAYOUT_RING : LAYOUT_TILES;
}
__host__ __device__ constexpr bool pair_buffer(int max_n, bool mixed) {
  return mixed || pair_layout(max_n) != LAYOUT_RING;
}
// Shared memory of a CTA that leaves room for a second one on the SM.
constexpr size_t kSmemTwo = 113 * 1024;

// Shifts of a ring chunk: the history of up to 256 atoms (m = 10, FP32) stays on
// chip beside it.  L-BFGS with a longer one (m > 27 up to 128 atoms, m > 13 above): as
// many shifts, but two at least, as leave it within kSmemTwo, where HIST_CHIP keeps it
// (1,024 x 128 atoms, m = 31, without allocation: 6.7 ms, 9.4 with the history in the
// fixed scratch, 8.1 before the ring).  The number belongs to the sizes and not
// to the place, since the order of the sums follows it.
__host__ __device__ constexpr int ring_shifts(int max_n, int m = 0) {
  const int most = max_n <= 128 ? 8 : 4, slots = max_n <= 128 ? 128 : 256;
  const long long left = (long long)kSmemTwo - 1024 - 32LL * max_n - 24LL * m * slots;
  const long long fit = left / (24LL * max_n);
  return fit >= most || fit < 2 ? most : (int)fit;
}

__host__ __device__ constexpr size_t half_bytes(int max_n, bool half, int ks) {
  return !half ? 0
         : align16((size_t)24 * (pair_layout(max_n) == LAYOUT_HALF   ? max_n * (max_n - 1) / 2
                                 : pair_layout(max_n) == LAYOUT_RING ? max_n * ks
                                                                     : max_n));
}

// per-team shared bytes: positions (32-byte records; the FP32 phase uses the
// first half of the same buffer), the optional half-pair buffer, the optional
// L-BFGS history (hist_bytes > 0: kept on chip instead of in the workspace),
// cross-warp reduction scratch (double-buffered), one word
template <int T>
__host__ __device__ constexpr size_t team_smem_bytes(int max_n, bool half, size_t hist_bytes,
                                                             int ks) {
  return align16((size_t)max_n * sizeof(PosD)) + half_bytes(max_n, half, ks) + align16(hist_bytes) +
         (T > 32 ? 2 * 8 * (T / 32) * sizeof(double) : 0) + 16;
}

template <int T>
__device__ __forceinline__ void carve_team(unsigned char* base, int max_n, bool half,
                                           size_t hist_bytes, int ks, void*& pos, void*& hbuf,
                                           void*& hist, double*& red, long long*& word) {
  pos = base;
  unsigned char* p = base + align16((size_t)max_n * sizeof(PosD));
  const size_t hb = half_bytes(max_n, half, ks);
  hbuf = hb ? static_cast<void*>(p) : nullptr;
  p += hb;
  hist = hist_bytes ? static_cast<void*>(p) : nullptr;
  p += align16(hist_bytes);
  red = reinterpret_cast<double*>(p);
  p += (T > 32 ? 2 * 8 * (T / 32) * sizeof(double) : 0);
  word = reinterpret_cast<long long*>(p);
}

// What a kernel is allowed to ask for: the most a CTA can have (227 KB), set
// once and for all its launches -- the buckets of one call share kernels, and a
// smaller value set for one would refuse the launch of another.
constexpr int kSmemMax = 227 * 1024;

// History goes on chip when a CTA's shared memory stays within this budget.
constexpr size_t kSmemBudget = 100 * 1024;

}  // namespace ljd
