// Index arithmetic of the warm-start network that host code can check.
#pragma once

#include <stddef.h>

#ifdef __CUDACC__
#define FIRLS_HD __host__ __device__
#else
#define FIRLS_HD
#endif

namespace firls {

// First value of pixel (y, x) of an n x n image with `channels` values a pixel.
// 64 bits: one image of more than 8192^2 pixels has more than 2^31 values at 32
// channels, and fits the device (33 GB of activations at 8320^2).  The pixel's number
// itself has 32 (an image of 2^32 pixels would need 2 TB).
FIRLS_HD inline size_t cnn_pixel(int y, int x, int n, int channels) {
  return (size_t)((unsigned)y * (unsigned)n + (unsigned)x) * (size_t)channels;
}

}  // namespace firls
