// The plan of a line transform: how the factors, the shared-memory layout and
// the threads of fft2.cu follow from the grid size.  Free of CUDA types, so
// that the host compiler can check it for every size.
#pragma once
#include <atomic>
#include <cstddef>
#include <cstdint>
#include <mutex>
#include "launch_rules.h"
#ifdef __CUDACC__
#define EMD_HD __host__ __device__ __forceinline__
#else
#define EMD_HD inline
#endif

// A line transform of n = r[0] r[1] .. r[ns-1] points, ns >= 2.  One step
// turns a block of R m values x[j + m t] into R blocks of m: block k holds
// w_{Rm}^{jk} sum_t w_R^{tk} x[j + m t] and is the transform of length m that
// gives the frequencies k, k + R, ...; so a step reads and writes the same
// places, and the last one leaves X[k_1 + r_1 (k_2 + r_2 (...))].  Line l's
// first-step blocks start at l ls + k_1 (m_1 | 1) (odd strides: no conflicts).
constexpr int kFftSteps = 4;
// t / d for t d < 2^32 by one multiplication (an integer division is ~30
// instructions, and a step of a small grid is only ~150)
struct FastDiv {
  unsigned mul, d;
};
EMD_HD FastDiv fast_div(unsigned d) {
  FastDiv f;
  f.d = d;
  f.mul = d > 1 ? 0xffffffffu / d + 1u : 0u;
  return f;
}
EMD_HD int operator/(int t, const FastDiv &f) {
#ifdef __CUDA_ARCH__
  return f.d == 1 ? t : (int)__umulhi((unsigned)t, f.mul);
#else
  return f.d == 1 ? t : (int)((uint64_t)(unsigned)t * f.mul >> 32);
#endif
}
struct FftLine {
  int n, ns;              // grid edge and line length; steps
  int r[kFftSteps];       // factors
  int m[kFftSteps];       // block length after the step
  FastDiv by_n, by_nh;    // nh: n / 2 + 1
  FastDiv by_r[kFftSteps], by_m[kFftSteps], by_blocks;   // by_blocks: n / r[ns - 1]
  int lsh;                // 2^lsh lines per CTA
  int ls;                 // shared-memory stride of a line
  int threads;            // per CTA
};

// block offset of frequency index kk = k_1 + r_1 (k_2 + ..) after `steps` steps
EMD_HD int block_at(const FftLine &p, int kk, int steps) {
  if (steps == 1) return kk * (p.m[0] | 1);
  int q = kk / p.by_r[0];
  int off = (kk - q * p.r[0]) * (p.m[0] | 1);
  for (int s = 1; s + 1 < steps; ++s) {
    const int t = q / p.by_r[s];
    off += (q - t * p.r[s]) * p.m[s];
    q = t;
  }
  return off + q * p.m[steps - 1];
}

constexpr int kFftMaxN = 1024;
constexpr size_t kFftMaxShared = 200 * 1024;
// roots | exchange array | lines in natural order, 16 bytes a value
inline size_t fft_shared_bytes(const FftLine &p) {
  return (p.n + ((size_t)(p.ls + (p.n | 1)) << p.lsh)) * 16;
}

// about the FP64 instructions of a butterfly, and its R - 1 twiddle products
inline int butterfly_cost(int R) {
  static const int dft[17] = {0, 0, 4, 14, 16, 36, 44, 66, 64, 100, 92, 150, 108, 210, 156, 170, 160};
  return dft[R] + 4 * (R - 1);
}

// the cheapest way to write n as 2 to 4 factors of at most 16, in ascending
// order: a step costs its instructions times 64 cycles times the warps per
// scheduler (at least one), and about 1500 cycles for its exchange
inline void best_factors(FftLine &p, int nlines, int ns, int at, int left, int lo, int *r, double c,
                         double &best) {
  if (at == ns - 1) {
    if (left > 16 || left < lo) return;
    r[at] = left;
    const double w = (double)nlines * (p.n / left) / 32.0 / (4.0 * kSMs);
    c += (w > 1.0 ? w : 1.0) * (butterfly_cost(left) - 4 * (left - 1)) * 64.0;
    if (c >= best) return;
    best = c;
    p.ns = ns;
    for (int s = 0; s < ns; ++s) p.r[s] = r[s];
    return;
  }
  for (int f = lo; f <= 16; ++f) {
    if (left % f) continue;
    const double w = (double)nlines * (p.n / f) / 32.0 / (4.0 * kSMs);
    r[at] = f;
    best_factors(p, nlines, ns, at + 1, left / f, f, r,
                 c + 1500.0 + (w > 1.0 ? w : 1.0) * butterfly_cost(f) * 64.0, best);
  }
}

// false: n is not a product of four factors of at most 16
inline bool line_plan(FftLine &p, int n) {
  const int nlines = n * (n / 2 + 1);
  p.n = n;
  p.ns = 0;
  int r[kFftSteps];
  double best = 1e300;
  for (int ns = 2; ns <= kFftSteps; ++ns) best_factors(p, nlines, ns, 0, n, 1, r, 0.0, best);
  if (!p.ns) return false;
  int m = n;
  for (int s = 0; s < p.ns; ++s) {
    p.m[s] = m /= p.r[s];
    p.by_r[s] = fast_div(p.r[s]);
    p.by_m[s] = fast_div(p.m[s]);
  }
  p.by_n = fast_div(n);
  p.by_nh = fast_div(n / 2 + 1);
  p.by_blocks = fast_div(n / p.r[p.ns - 1]);
  p.ls = (p.r[0] * (p.m[0] | 1)) | 1;
  // 8 lines: transposed writes of 128 bytes; 4 where that takes too much
  // shared memory (n above ~740)
  p.lsh = 3;
  if (fft_shared_bytes(p) > kFftMaxShared) p.lsh = 2;
  const int most = (n / p.r[0]) << p.lsh;              // threads of the widest step
  p.threads = most >= 256 ? 256 : (most + 31) / 32 * 32;
  return true;
}

// The plan of grid size n, nullptr if there is none; worked out once per size
// and kept in static storage (the solve that allocates nothing uses it too).
static inline const FftLine *fft_plan(int n) {
  enum : unsigned char { kUnknown, kNone, kReady };
  static FftLine plans[kFftMaxN + 1];
  static std::atomic<unsigned char> state[kFftMaxN + 1];
  static std::mutex mu;
  if (n < 2 || n > kFftMaxN) return nullptr;
  unsigned char st = state[n].load(std::memory_order_acquire);
  if (st == kUnknown) {
    std::lock_guard<std::mutex> lk(mu);
    st = state[n].load(std::memory_order_relaxed);
    if (st == kUnknown) {
      st = line_plan(plans[n], n) ? kReady : kNone;
      state[n].store(st, std::memory_order_release);
    }
  }
  return st == kReady ? &plans[n] : nullptr;
}
