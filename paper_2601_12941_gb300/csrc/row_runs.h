// Where the prefilter's runs of 64 gray levels are read from: the mirror at the image's sides and the
// words of unaligned rows. Plain C++, so that the host can check it for any geometry.
#pragma once

#include <stdint.h>

#ifdef __CUDACC__
#define DIC_RUN_FN __host__ __device__ __forceinline__
#else
#define DIC_RUN_FN inline
#endif

namespace dic {

// Whole-sample mirror of k into [0, n), n >= 2. NEAR: k lies at most n - 1 outside, one
// reflection away (without a branch; for the 64-element runs and 28 halo rows: n >= 192), and n at most
// 2^30 (both sides of such an image are long, no memory holds a longer one). Otherwise any k > -2^31:
// the period 2 (n - 1) of a side above 2^30 does not fit an int, hence unsigned.
constexpr int kPfNear = 192;
template <bool NEAR>
DIC_RUN_FN int mirror_k(int k, int n) {
  const int m = k < 0 ? -k : k;                 // the mirror is even
  if constexpr (NEAR) {
    const int v = 2 * (n - 1) - m;
    return m < v ? m : v;
  } else {
    const unsigned period = 2u * (static_cast<unsigned>(n) - 1u), u = static_cast<unsigned>(m) % period;
    return static_cast<int>(u < period - u ? u : period - u);
  }
}

// A run of 64 elements of `bytes` bytes at columns xa .. xa + 63 of row y, inside the image, whose
// first byte lies `shift` bytes behind a 4-byte boundary, read as aligned words: the last word
// then holds 4 - shift bytes behind the run. They lie inside the buffer, whose last byte is that of the
// last pixel, in every row but the last, and there when the run ends that far before the row.
DIC_RUN_FN bool words_inside(int xa, int y, int W, int H, int bytes, unsigned shift) {
  return shift == 0 || y + 1 < H || static_cast<int64_t>(W - 64 - xa) * bytes >= static_cast<int64_t>(4 - shift);
}

}  // namespace dic
