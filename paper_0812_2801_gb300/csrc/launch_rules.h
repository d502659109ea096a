// How launches are divided over the GPU: plain functions of sizes, kept free
// of CUDA so that the host compiler can check them over their whole range.
#pragma once
#include <algorithm>

constexpr int kSMs = 152;   // GB300: two dies of 76

// Row chunks of the overlap products G = X^H Y (n3 rows, m columns; k_gram),
// one CTA per chunk and 16 x 16 tile of G: enough for 16 CTAs per SM, of at
// least 96 rows each (three of the kernel's rounds).  n3 / 4096 chunks alone,
// at most 64, left 3 CTAs on 24^3 with 9 states: 1.23 ms per product.
// Never fewer than those, though: each entry is summed in one FP64 chain per
// chunk, and many tiles (above 96 states on 96^3) must not make the chains longer.
inline int emd_gram_chunks(int n3, int m) {
  const int tiles = ((m + 15) / 16) * ((m + 15) / 16);
  const int fill = std::min((16 * kSMs + tiles - 1) / tiles, n3 / 96);
  return std::max({1, fill, std::min(64, n3 / 4096)});
}
