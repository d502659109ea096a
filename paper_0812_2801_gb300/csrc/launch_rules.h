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
// Measured per FP64 product on 96^3, n3 / 4096 / filling / the larger: 9 states
// 3.92 / 1.00 / 1.00 ms, 64 states 24.4 / 23.4 / 23.4 ms, 138 states 120 / 116 /
// 115 ms, 200 states 247 / 244 / 237 ms; an entry's error over n3 at 138 states
// 2.5e-16 / 1.4e-15 / 1.3e-16.
inline int emd_gram_chunks(int n3, int m) {
  const int tiles = ((m + 15) / 16) * ((m + 15) / 16);
  const int fill = std::min((16 * kSMs + tiles - 1) / tiles, n3 / 96);
  return std::max({1, fill, std::min(64, n3 / 4096)});
}

// Planes per z-chunk of a marching stage launch with `cols` CTAs per layer of
// chunks: the split with the smallest estimated time.  A chunk of zc planes
// costs zc planes, its 2M halo planes at `halo` of one each, and `fill` planes
// to fill its ring; CTAs are dealt to the SMs in rounds, and one CTA alone on an
// SM runs at about 0.7 of the speed of two.  A finer split has to be 2 % better.
//   complex64 stage: halo planes are restaged and re-stencilled in full, halo =
//     1, fill = 2.  At least 304 CTAs or 16 planes per chunk, the rule before,
//     gave 108 CTAs of 24 planes with their halo on 16 orbitals of 48^3, this
//     one 144 of 20 (5.96 -> 5.44 ms a run, with the reductions).
//   double-float stage: they only feed the z direction (80 of 302 packed FP32
//     instructions), halo = 0.3, fill = 0.
inline int emd_zchunk(int n, int half_order, int cols, double halo, int fill) {
  int best = n;
  double cost = 1e300;
  for (int nz = 1; nz <= n / 4; ++nz) {
    const int zc = (n + nz - 1) / nz, ctas = cols * ((n + zc - 1) / zc);
    const double load = (ctas + kSMs - 1) / kSMs;
    const double t = std::max(load, 1.4) * (zc + halo * 2 * half_order + fill);
    if (t < 0.98 * cost) {
      cost = t;
      best = zc;
    }
  }
  return best;
}

// CTAs of 256 threads per (projector, orbital block) of the atom-major gathers:
// one when the pairs fill the GPU, else 2, 4 or 8 that share the atom's
// entries.  Aims at 12 CTAs per SM and at least one full round of the loop (1024
// entries; about half of a table's capacity, a cube around the sphere, is used)
// per CTA.  With a split, pairs x split stays below kGatherMaxCtas.
constexpr int kGatherMaxCtas = kSMs * 12 * 2;
inline int emd_gather_split(int pairs, int cap) {
  int s = 1;
  while (s < 8 && pairs * s < kGatherMaxCtas / 2 && cap / 2 >= 1024 * 2 * s) s *= 2;
  return s;
}
