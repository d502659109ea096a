// Test driver for the line plans (fft_plan.h).
//   plans     -> one line per n = 2 .. 1024 that has a plan: n, lines per CTA,
//                shared bytes, threads, factors
//   layout    -> the first inconsistency of any plan, or "ok"
//   fft n     -> largest error of a line transform done by the plan's steps
//                with direct butterflies, against a direct sum
//   allocs    -> heap allocations made by asking for every plan
#include <algorithm>
#include <cmath>
#include <complex>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <new>
#include <vector>
#include "fft_plan.h"

static long g_allocs = 0;
void *operator new(size_t n) {
  ++g_allocs;
  if (void *p = std::malloc(n)) return p;
  throw std::bad_alloc();
}
void operator delete(void *p) noexcept { std::free(p); }
void operator delete(void *p, size_t) noexcept { std::free(p); }

static bool div_ok(const FastDiv &f, int below) {
  for (int t = 0; t < below; ++t)
    if (t / f != t / (int)f.d) return false;
  return true;
}

static const char *layout(const FftLine &p) {
  const int n = p.n, nh = n / 2 + 1;
  if (p.ns < 2 || p.ns > kFftSteps) return "steps";
  int prod = 1;
  for (int s = 0; s < p.ns; ++s) {
    if (p.r[s] < 1 || p.r[s] > 16) return "factor";
    prod *= p.r[s];
    if (p.m[s] != n / prod) return "block length";
  }
  if (prod != n) return "product";
  if (fft_shared_bytes(p) > kFftMaxShared) return "shared memory";
  if (p.threads < 32 || p.threads > 256 || p.threads % 32) return "threads";
  if (!div_ok(p.by_n, std::max(n << p.lsh, n * nh)) || !div_ok(p.by_nh, std::max(nh << p.lsh, n * nh)))
    return "division by n or n / 2 + 1";
  int groups = 1;
  for (int s = 0; s + 1 < p.ns; ++s) {
    const int m = p.m[s], st = s ? m : m | 1;
    if (!div_ok(p.by_m[s], (groups * m) << p.lsh) || !div_ok(p.by_r[s], n)) return "division";
    std::vector<char> seen(p.ls, 0);           // a step's values lie apart, within the line
    for (int g = 0; g < groups; ++g)
      for (int j = 0; j < m; ++j)
        for (int k = 0; k < p.r[s]; ++k) {
          const int at = (s ? block_at(p, g, s) : 0) + j + k * st;
          if (at < 0 || at >= p.ls || seen[at]++) return "step's places";
        }
    groups *= p.r[s];
  }
  if ((int)p.by_blocks.d != groups) return "blocks";
  std::vector<char> seen(p.ls, 0);
  for (int k = 0; k < groups; ++k)
    for (int j = 0; j < p.r[p.ns - 1]; ++j) {
      const int at = block_at(p, k, p.ns - 1) + j;
      if (at < 0 || at >= p.ls || seen[at]++) return "last step's places";
    }
  return nullptr;
}

typedef std::complex<double> C;
static C root(long num, long den) { return std::polar(1.0, -2.0 * M_PI * (double)(num % den) / den); }
static double fft_error(const FftLine &p) {
  const int n = p.n;
  std::vector<C> x(n), ex(p.ls), X(n);
  for (int i = 0; i < n; ++i) x[i] = C(std::sin(1.0 + 3.7 * i), std::cos(0.3 * i * i));
  int groups = 1;
  for (int s = 0; s < p.ns; ++s) {
    const int m = p.m[s], R = p.r[s], st = s ? m : m | 1;
    const bool last = s == p.ns - 1;
    for (int g = 0; g < groups; ++g)
      for (int j = 0; j < m; ++j) {
        const int at = (s ? block_at(p, g, s) : 0) + j;
        std::vector<C> v(R);
        for (int r = 0; r < R; ++r) v[r] = s ? ex[at + r * m] : x[j + r * m];
        for (int k = 0; k < R; ++k) {
          C y = 0.0;
          for (int r = 0; r < R; ++r) y += v[r] * root((long)r * k, R);
          if (last) X[g + groups * k] = y;
          else ex[at + k * st] = y * root((long)groups * j * k, n);
        }
      }
    groups *= R;
  }
  double worst = 0.0;
  for (int k = 0; k < n; ++k) {
    C y = 0.0;
    for (int i = 0; i < n; ++i) y += x[i] * root((long)i * k, n);
    worst = std::max(worst, std::abs(y - X[k]));
  }
  return worst / std::sqrt((double)n);
}

int main(int argc, char **argv) {
  if (argc < 2) return 2;
  if (!std::strcmp(argv[1], "allocs")) {
    const long before = g_allocs;
    for (int n = -1; n <= kFftMaxN + 1; ++n) fft_plan(n);
    std::printf("%ld\n", g_allocs - before);
  } else if (!std::strcmp(argv[1], "plans")) {
    for (int n = 2; n <= kFftMaxN; ++n)
      if (const FftLine *p = fft_plan(n)) {
        std::printf("%d %d %zu %d", n, 1 << p->lsh, fft_shared_bytes(*p), p->threads);
        for (int s = 0; s < p->ns; ++s) std::printf(" %d", p->r[s]);
        std::printf("\n");
      }
  } else if (!std::strcmp(argv[1], "layout")) {
    for (int n = 2; n <= kFftMaxN; ++n)
      if (const FftLine *p = fft_plan(n))
        if (const char *what = layout(*p)) {
          std::printf("%d: %s\n", n, what);
          return 0;
        }
    std::printf("ok\n");
  } else if (!std::strcmp(argv[1], "fft") && argc == 3) {
    const FftLine *p = fft_plan(std::atoi(argv[2]));
    if (!p) return 2;
    std::printf("%g\n", fft_error(*p));
  } else {
    return 2;
  }
  return 0;
}
