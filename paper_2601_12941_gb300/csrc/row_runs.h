// Where the prefilter's runs of 64 gray levels are read from. Plain C++, so that the host
// can check it for any geometry.
#pragma once

#include <stdint.h>

#ifdef __CUDACC__
#define DIC_RUN_FN __host__ __device__ __forceinline__
#else
#define DIC_RUN_FN inline
#endif

namespace dic {

// A run of 64 elements of `bytes` bytes at columns xa .. xa + 63 of row y, inside the image, whose
// first byte lies `shift` bytes behind a 4-byte boundary, read as aligned words: the last word
// then holds 4 - shift bytes behind the run. They lie inside the buffer, whose last byte is that of the
// last pixel, in every row but the last, and there when the run ends that far before the row.
DIC_RUN_FN bool words_inside(int xa, int y, int W, int H, int bytes, unsigned shift) {
  return shift == 0 || y + 1 < H || static_cast<int64_t>(W - 64 - xa) * bytes >= static_cast<int64_t>(4 - shift);
}

}  // namespace dic
