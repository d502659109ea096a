// Spectral multiplication on periodic grids in five passes: the transforms of
// the Hartree and ionic electrostatics (eq. E_KS, eq. ionicpotential; a
// periodic spectral solve stands in for the paper's finite-system solver) and
// of Kerker's preconditioner.
//
// What bounds it: GB300's FP64 rate.  One FP64 warp instruction occupies a
// quarter of an SM (a scheduler's FP64 lanes) for 64 cycles, so a pass costs
// (FP64 instructions of a thread) x 64 cycles x (warps per scheduler), and on
// small grids, which do not fill the 608 schedulers, what counts is the length
// of one thread's chain.  So
//  * a line's transform is two to four register butterflies of at most 16
//    points with exchanges through shared memory between them.  The factors
//    are chosen by that cost: few large butterflies (fewest instructions) on
//    large grids, more small ones (short chains) on small grids;
//  * the butterflies' own twiddles are constants, prime butterflies use the
//    real symmetric form (half the multiplications of the direct sum), and
//    those of coprime factors need no twiddles between them;
//  * the forward z transform, the spectral factor and the inverse z transform
//    are one pass: the spectrum along z never leaves the SM;
//  * two real lines run as one complex line and only kx <= n / 2 is kept.
// Measured: emd_poisson_static on 48^3 92 -> 51 us a call (seven passes of one
// exchange per radix 2, 3, 4 or 5 on complex data before); the five passes
// alone, 48^3 45 us, 64^3 63 us, 96^3 148 us, 120^3 311 us, 160^3 687 us.
// Every pass reads lines that are contiguous and writes 64-byte pieces or
// longer of the layout whose next axis is contiguous.
//   X    x, real -> complex       [z][y][x]    -> [kx][z][y]
//   Y    y                        [kx][z][y]   -> [ky][kx][z]
//   Z    z, factor, inverse z     [ky][kx][z]  -> [kx][z][ky]
//   YINV inverse y                [kx][z][ky]  -> [z][y][kx]
//   XINV inverse x, complex -> real [z][y][kx] -> [z][y][x]
// Inverse transforms run the forward butterflies with real and imaginary
// parts exchanged on the way in and out.
//
// Accuracy: a solve is off by about three roundings (2-norm), most of them of
// the additions: 3.5e-16 on average over 20 grids of 16^3 to 64^3, 3.7e-16 with
// the complex transforms, 4.2e-16 with lines of n / 2 complex values.  What
// keeps it there: pairs of real lines average the errors of Z_k and Z_{n-k} (a
// line as n / 2 complex values adds those of its untangling), coprime
// butterflies have no twiddles to round, and sqrt(3) / 2 and sqrt(1/2) come with
// their low parts, since the rounding of a constant that every line meets
// scales the whole result (27^3: by 2.5e-16).
#include "emd_internal.cuh"
#include "fft_plan.h"

namespace {

__device__ __forceinline__ double2 cadd(double2 a, double2 b) {
  return make_double2(a.x + b.x, a.y + b.y);
}
__device__ __forceinline__ double2 csub(double2 a, double2 b) {
  return make_double2(a.x - b.x, a.y - b.y);
}
__device__ __forceinline__ double2 cmul(double2 a, double2 b) {
  return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
__device__ __forceinline__ double2 cswap(double2 a) { return make_double2(a.y, a.x); }

// (cos, sin)(2 pi k / R); with k known at compile time the table folds away
template <int R> __device__ __forceinline__ double2 circle(int k) {
  if (R == 3) {
    const double c[3] = {
        1.0, -0.5, -0.5};
    const double s[3] = {
        0.0, 0.8660254037844386, -0.8660254037844386};
    return make_double2(c[k], s[k]);
  }
  if (R == 5) {
    const double c[5] = {
        1.0, 0.30901699437494745, -0.8090169943749475, -0.8090169943749475,
        0.30901699437494745};
    const double s[5] = {
        0.0, 0.9510565162951535, 0.5877852522924731, -0.5877852522924731,
        -0.9510565162951535};
    return make_double2(c[k], s[k]);
  }
  if (R == 6) {
    const double c[6] = {
        1.0, 0.5, -0.5, -1.0, -0.5, 0.5};
    const double s[6] = {
        0.0, 0.8660254037844386, 0.8660254037844386, 0.0, -0.8660254037844386,
        -0.8660254037844386};
    return make_double2(c[k], s[k]);
  }
  if (R == 7) {
    const double c[7] = {
        1.0, 0.6234898018587335, -0.2225209339563144, -0.9009688679024191,
        -0.9009688679024191, -0.2225209339563144, 0.6234898018587335};
    const double s[7] = {
        0.0, 0.7818314824680298, 0.9749279121818236, 0.4338837391175581,
        -0.4338837391175581, -0.9749279121818236, -0.7818314824680298};
    return make_double2(c[k], s[k]);
  }
  if (R == 8) {
    const double c[8] = {
        1.0, 0.7071067811865476, 0.0, -0.7071067811865476, -1.0, -0.7071067811865476, 0.0,
        0.7071067811865476};
    const double s[8] = {
        0.0, 0.7071067811865476, 1.0, 0.7071067811865476, 0.0, -0.7071067811865476, -1.0,
        -0.7071067811865476};
    return make_double2(c[k], s[k]);
  }
  if (R == 9) {
    const double c[9] = {
        1.0, 0.766044443118978, 0.17364817766693036, -0.5, -0.9396926207859084,
        -0.9396926207859084, -0.5, 0.17364817766693036, 0.766044443118978};
    const double s[9] = {
        0.0, 0.6427876096865394, 0.984807753012208, 0.8660254037844386, 0.3420201433256687,
        -0.3420201433256687, -0.8660254037844386, -0.984807753012208, -0.6427876096865394};
    return make_double2(c[k], s[k]);
  }
  if (R == 10) {
    const double c[10] = {
        1.0, 0.8090169943749475, 0.30901699437494745, -0.30901699437494745,
        -0.8090169943749475, -1.0, -0.8090169943749475, -0.30901699437494745,
        0.30901699437494745, 0.8090169943749475};
    const double s[10] = {
        0.0, 0.5877852522924731, 0.9510565162951535, 0.9510565162951535, 0.5877852522924731,
        0.0, -0.5877852522924731, -0.9510565162951535, -0.9510565162951535,
        -0.5877852522924731};
    return make_double2(c[k], s[k]);
  }
  if (R == 11) {
    const double c[11] = {
        1.0, 0.8412535328311812, 0.41541501300188644, -0.14231483827328514,
        -0.6548607339452851, -0.9594929736144974, -0.9594929736144974, -0.6548607339452851,
        -0.14231483827328514, 0.41541501300188644, 0.8412535328311812};
    const double s[11] = {
        0.0, 0.5406408174555976, 0.9096319953545183, 0.9898214418809327, 0.7557495743542583,
        0.28173255684142967, -0.28173255684142967, -0.7557495743542583, -0.9898214418809327,
        -0.9096319953545183, -0.5406408174555976};
    return make_double2(c[k], s[k]);
  }
  if (R == 12) {
    const double c[12] = {
        1.0, 0.8660254037844386, 0.5, 0.0, -0.5, -0.8660254037844386, -1.0,
        -0.8660254037844386, -0.5, 0.0, 0.5, 0.8660254037844386};
    const double s[12] = {
        0.0, 0.5, 0.8660254037844386, 1.0, 0.8660254037844386, 0.5, 0.0, -0.5,
        -0.8660254037844386, -1.0, -0.8660254037844386, -0.5};
    return make_double2(c[k], s[k]);
  }
  if (R == 13) {
    const double c[13] = {
        1.0, 0.8854560256532099, 0.5680647467311558, 0.12053668025532305,
        -0.3546048870425356, -0.7485107481711011, -0.970941817426052, -0.970941817426052,
        -0.7485107481711011, -0.3546048870425356, 0.12053668025532305, 0.5680647467311558,
        0.8854560256532099};
    const double s[13] = {
        0.0, 0.46472317204376856, 0.8229838658936564, 0.992708874098054, 0.9350162426854148,
        0.6631226582407952, 0.23931566428755777, -0.23931566428755777, -0.6631226582407952,
        -0.9350162426854148, -0.992708874098054, -0.8229838658936564, -0.46472317204376856};
    return make_double2(c[k], s[k]);
  }
  if (R == 14) {
    const double c[14] = {
        1.0, 0.9009688679024191, 0.6234898018587335, 0.2225209339563144,
        -0.2225209339563144, -0.6234898018587335, -0.9009688679024191, -1.0,
        -0.9009688679024191, -0.6234898018587335, -0.2225209339563144, 0.2225209339563144,
        0.6234898018587335, 0.9009688679024191};
    const double s[14] = {
        0.0, 0.4338837391175581, 0.7818314824680298, 0.9749279121818236, 0.9749279121818236,
        0.7818314824680298, 0.4338837391175581, 0.0, -0.4338837391175581,
        -0.7818314824680298, -0.9749279121818236, -0.9749279121818236, -0.7818314824680298,
        -0.4338837391175581};
    return make_double2(c[k], s[k]);
  }
  if (R == 15) {
    const double c[15] = {
        1.0, 0.9135454576426009, 0.6691306063588582, 0.30901699437494745,
        -0.10452846326765347, -0.5, -0.8090169943749475, -0.9781476007338057,
        -0.9781476007338057, -0.8090169943749475, -0.5, -0.10452846326765347,
        0.30901699437494745, 0.6691306063588582, 0.9135454576426009};
    const double s[15] = {
        0.0, 0.4067366430758002, 0.7431448254773942, 0.9510565162951535, 0.9945218953682733,
        0.8660254037844386, 0.5877852522924731, 0.20791169081775934, -0.20791169081775934,
        -0.5877852522924731, -0.8660254037844386, -0.9945218953682733, -0.9510565162951535,
        -0.7431448254773942, -0.4067366430758002};
    return make_double2(c[k], s[k]);
  }
  if (R == 16) {
    const double c[16] = {
        1.0, 0.9238795325112867, 0.7071067811865476, 0.3826834323650898, 0.0,
        -0.3826834323650898, -0.7071067811865476, -0.9238795325112867, -1.0,
        -0.9238795325112867, -0.7071067811865476, -0.3826834323650898, 0.0,
        0.3826834323650898, 0.7071067811865476, 0.9238795325112867};
    const double s[16] = {
        0.0, 0.3826834323650898, 0.7071067811865476, 0.9238795325112867, 1.0,
        0.9238795325112867, 0.7071067811865476, 0.3826834323650898, 0.0,
        -0.3826834323650898, -0.7071067811865476, -0.9238795325112867, -1.0,
        -0.9238795325112867, -0.7071067811865476, -0.3826834323650898};
    return make_double2(c[k], s[k]);
  }
  return make_double2(1.0, 0.0);
}

// ---- forward DFTs of R points in registers ----------------------------------
// odd primes: y_j = a_j - i b_j, y_{R-j} = a_j + i b_j with a_j = x_0 + sum_k
// cos(2 pi j k / R) (x_k + x_{R-k}), b_j = sum_k sin(2 pi j k / R) (x_k - x_{R-k})
template <int R> struct Dft {
  static __device__ __forceinline__ void run(double2 (&v)[R]) {
    constexpr int H = (R - 1) / 2;
    double2 t[H], d[H];
    double2 s0 = v[0];
#pragma unroll
    for (int k = 1; k <= H; ++k) {
      t[k - 1] = cadd(v[k], v[R - k]);
      d[k - 1] = csub(v[k], v[R - k]);
      s0 = cadd(s0, t[k - 1]);
    }
    const double2 x0 = v[0];
    v[0] = s0;
#pragma unroll
    for (int j = 1; j <= H; ++j) {
      double2 a = x0, b = make_double2(0.0, 0.0);
#pragma unroll
      for (int k = 1; k <= H; ++k) {
        const double2 w = circle<R>(j * k % R);
        a.x = fma(w.x, t[k - 1].x, a.x);
        a.y = fma(w.x, t[k - 1].y, a.y);
        b.x = fma(w.y, d[k - 1].x, b.x);
        b.y = fma(w.y, d[k - 1].y, b.y);
      }
      v[j] = make_double2(a.x + b.y, a.y - b.x);
      v[R - j] = make_double2(a.x - b.y, a.y + b.x);
    }
  }
};
template <> struct Dft<1> {
  static __device__ __forceinline__ void run(double2 (&)[1]) {}
};
template <> struct Dft<2> {
  static __device__ __forceinline__ void run(double2 (&v)[2]) {
    const double2 a = v[0];
    v[0] = cadd(a, v[1]);
    v[1] = csub(a, v[1]);
  }
};
// sqrt(3) / 2 to twice the precision
template <> struct Dft<3> {
  static __device__ __forceinline__ void run(double2 (&v)[3]) {
    constexpr double hi = 0.8660254037844386, lo = 5.017542110902451e-17;
    const double2 t = cadd(v[1], v[2]), d = csub(v[1], v[2]);
    const double2 a = make_double2(fma(-0.5, t.x, v[0].x), fma(-0.5, t.y, v[0].y));
    v[0] = cadd(v[0], t);
    v[1] = make_double2(fma(hi, d.y, fma(lo, d.y, a.x)), fma(-hi, d.x, fma(-lo, d.x, a.y)));
    v[2] = make_double2(fma(-hi, d.y, fma(-lo, d.y, a.x)), fma(hi, d.x, fma(lo, d.x, a.y)));
  }
};
template <> struct Dft<4> {
  static __device__ __forceinline__ void run(double2 (&v)[4]) {
    const double2 a = cadd(v[0], v[2]), b = csub(v[0], v[2]);
    const double2 c = cadd(v[1], v[3]), d = csub(v[1], v[3]);
    v[0] = cadd(a, c);
    v[2] = csub(a, c);
    v[1] = make_double2(b.x + d.y, b.y - d.x);   // b - i d
    v[3] = make_double2(b.x - d.y, b.y + d.x);
  }
};
// v (c - i s) for a constant (c, s); 1, -1, i and -i need no multiplication,
// and the diagonals take sqrt(1/2) to twice the precision
__device__ __forceinline__ double2 ctwiddle(double2 v, double2 w) {
  if (w.y == 0.0) return w.x > 0.0 ? v : make_double2(-v.x, -v.y);
  if (w.x == 0.0) return w.y > 0.0 ? make_double2(v.y, -v.x) : make_double2(-v.y, v.x);
  if (w.x == w.y || w.x == -w.y) {
    constexpr double hi = 0.7071067811865476, lo = -4.833646656726457e-17;
    const double sx = w.x > 0.0 ? 1.0 : -1.0, sy = w.y > 0.0 ? 1.0 : -1.0;
    const double a = sx * v.x + sy * v.y, b = sx * v.y - sy * v.x;
    return make_double2(fma(hi, a, lo * a), fma(hi, b, lo * b));
  }
  return cmul(v, make_double2(w.x, -w.y));
}
// composite R = A B: B transforms of A points, constant twiddles, A of B points
template <int A, int B> struct DftAB {
  static __device__ __forceinline__ void run(double2 (&v)[A * B]) {
    constexpr int R = A * B;
    double2 u[B][A];
#pragma unroll
    for (int j = 0; j < B; ++j) {
#pragma unroll
      for (int r = 0; r < A; ++r) u[j][r] = v[j + B * r];
      Dft<A>::run(u[j]);
#pragma unroll
      for (int k = 1; k < A; ++k)
        if (j > 0) u[j][k] = ctwiddle(u[j][k], circle<R>(j * k % R));
    }
#pragma unroll
    for (int k = 0; k < A; ++k) {
      double2 w[B];
#pragma unroll
      for (int j = 0; j < B; ++j) w[j] = u[j][k];
      Dft<B>::run(w);
#pragma unroll
      for (int q = 0; q < B; ++q) v[k + A * q] = w[q];
    }
  }
};
// R = A B with A and B coprime: n = (B j + A i) mod R and k = the number that
// is k_1 mod A and k_2 mod B (Good 1958, Thomas 1963): no twiddles between
// the B transforms of A points and the A of B points
template <int A, int B> struct DftCoprime {
  static __host__ __device__ constexpr int crt(int k1, int k2) {
    int k = k2;
    while (k % A != k1) k += B;
    return k;
  }
  static __device__ __forceinline__ void run(double2 (&v)[A * B]) {
    constexpr int R = A * B;
    double2 u[B][A];
#pragma unroll
    for (int i = 0; i < B; ++i) {
#pragma unroll
      for (int j = 0; j < A; ++j) u[i][j] = v[(B * j + A * i) % R];
      Dft<A>::run(u[i]);
    }
#pragma unroll
    for (int k = 0; k < A; ++k) {
      double2 w[B];
#pragma unroll
      for (int i = 0; i < B; ++i) w[i] = u[i][k];
      Dft<B>::run(w);
#pragma unroll
      for (int q = 0; q < B; ++q) v[crt(k, q)] = w[q];
    }
  }
};
template <> struct Dft<6> : DftCoprime<2, 3> {};
template <> struct Dft<8> : DftAB<2, 4> {};
template <> struct Dft<9> : DftAB<3, 3> {};
template <> struct Dft<10> : DftCoprime<2, 5> {};
template <> struct Dft<12> : DftCoprime<3, 4> {};
template <> struct Dft<14> : DftCoprime<2, 7> {};
template <> struct Dft<15> : DftCoprime<3, 5> {};
template <> struct Dft<16> : DftAB<4, 4> {};

#define EMD_FFT_SWITCH(R, CALL)                                                     \
  switch (R) {                                                                      \
    case 1: CALL(1); break;                                                         \
    case 2: CALL(2); break;                                                         \
    case 3: CALL(3); break;                                                         \
    case 4: CALL(4); break;                                                         \
    case 5: CALL(5); break;                                                         \
    case 6: CALL(6); break;                                                         \
    case 7: CALL(7); break;                                                         \
    case 8: CALL(8); break;                                                         \
    case 9: CALL(9); break;                                                         \
    case 10: CALL(10); break;                                                       \
    case 11: CALL(11); break;                                                       \
    case 12: CALL(12); break;                                                       \
    case 13: CALL(13); break;                                                       \
    case 14: CALL(14); break;                                                       \
    case 15: CALL(15); break;                                                       \
    case 16: CALL(16); break;                                                       \
  }

// The five passes are one kernel: the butterflies of 1 to 16 points are nearly
// all of its code, and the first solve of a process waits until the code is on
// the GPU (48^3: 0.7 ms for 0.5 MB; five kernels with a copy per transform were
// 4 MB and took 14 ms).
//   X    real -> complex.  Two real lines a, b run as one complex line Z of a
//        + i b; 2 A_k = Z_k + conj Z_{n-k}, 2 i B_k = Z_k - conj Z_{n-k}, k <=
//        n / 2: twice the spectrum.
//   Y    lines (kx, z) along y
//   Z    lines (kx, ky) along z: forward, times the factor of the integer s =
//        mx^2 + my^2 + mz^2 (|G|^2 = (2 pi / L)^2 s), inverse.  kappa < 0: the
//        Poisson kernel c / s, 0 at s = 0 (inv_s[s] = 1 / s, inv_s[0] = 0);
//        else Kerker's c s / (s + kappa), c at s = 0.
//   YINV lines (z, kx) along ky
//   XINV two Hermitian lines A, B as one: Z_k = A_k + i B_k, Z_{n-k} = conj A_k
//        + i conj B_k; the imaginary parts that rounding left at k = 0 and n /
//        2 are dropped.
enum FftPass { FFT_X, FFT_Y, FFT_Z, FFT_YINV, FFT_XINV };

// Shared memory of a CTA: roots | exchange array | lines in natural
// order (line l, element i at l (n | 1) + i).
struct FftCta {
  FftPass pass;
  int l0, nlines;               // first line; lines of the pass
  const double2 *in;
  double2 *out;
  const FftLine *p;
  double2 *roots, *ex, *nat;
  bool from_nat, to_nat, swap_in, swap_out;    // this transform's ends
  // where line l of the CTA starts; its elements are contiguous
  __device__ __forceinline__ const double2 *source(int l) const {
    const int n = p->n, nh = (int)p->by_nh.d;
    if (from_nat) return nat + l * (n | 1);
    int line = min(l0 + l, nlines - 1);
    if (pass == FFT_Z) {
      const int kx = line / p->by_n;
      line = (line - kx * n) * nh + kx;
    } else if (pass == FFT_YINV) {
      const int z = line / p->by_nh;
      line = (line - z * nh) * n + z;
    }
    return in + (size_t)line * n;
  }
  // where its frequency 0 goes (nullptr: no such line), and the step to the next
  __device__ __forceinline__ double2 *target(int l, size_t &step) const {
    const int n = p->n, nh = (int)p->by_nh.d, line = l0 + l;
    step = 1;
    if (to_nat) return nat + l * (n | 1);
    if (line >= nlines) return nullptr;
    if (pass == FFT_Y) {
      step = nlines;
      return out + line;
    }
    if (pass == FFT_Z) {
      const int kx = line / p->by_n, ky = line - kx * n;
      step = n;
      return out + (size_t)kx * n * n + ky;
    }
    const int z = line / p->by_nh, kx = line - z * nh;
    step = nh;
    return out + (size_t)z * n * nh + kx;
  }
};

// step s but the last, into the exchange array; groups = product of the
// factors before it.  The first reads the lines' source, the others what
// they overwrite.
template <int R> __device__ __forceinline__ void step(const FftCta &f, int s, int groups) {
  const FftLine &p = *f.p;
  const int m = p.m[s], st = s ? m : m | 1;
  for (int t = threadIdx.x; t < (groups * m) << p.lsh; t += blockDim.x) {
    const int b = t / p.by_m[s], j = t - b * m, l = b & ((1 << p.lsh) - 1), g = b >> p.lsh;
    double2 *e = f.ex + l * p.ls + (s ? block_at(p, g, s) : 0) + j;
    const double2 *x = s ? e : f.source(l) + j;
    double2 v[R];
#pragma unroll
    for (int r = 0; r < R; ++r) v[r] = x[r * m];
    if (!s && f.swap_in) {
#pragma unroll
      for (int r = 0; r < R; ++r) v[r] = cswap(v[r]);
    }
    Dft<R>::run(v);
    const double2 *w = f.roots;
    e[0] = v[0];
#pragma unroll
    for (int k = 1; k < R; ++k) {
      w += groups * j;                     // root j k groups
      e[k * st] = cmul(v[k], *w);
    }
  }
}
// the last step, to the lines' target; neighbouring threads take neighbouring lines
template <int R> __device__ __forceinline__ void last(const FftCta &f) {
  const FftLine &p = *f.p;
  const int per = (int)p.by_blocks.d;
  for (int t = threadIdx.x; t < per << p.lsh; t += blockDim.x) {
    const int l = t & ((1 << p.lsh) - 1), k = t >> p.lsh;
    const double2 *e = f.ex + l * p.ls + block_at(p, k, p.ns - 1);
    double2 v[R];
#pragma unroll
    for (int j = 0; j < R; ++j) v[j] = e[j];
    Dft<R>::run(v);
    size_t next;
    double2 *o = f.target(l, next);
    if (!o) continue;
    o += k * next;
    next *= per;
    if (f.swap_out) {
#pragma unroll
      for (int q = 0; q < R; ++q) v[q] = cswap(v[q]);
    }
#pragma unroll
    for (int q = 0; q < R; ++q) o[q * next] = v[q];
  }
}

__device__ __forceinline__ void line_fft(const FftCta &f) {
  const FftLine &p = *f.p;
  int groups = 1;
  for (int s = 0; s < p.ns - 1; ++s) {
#define EMD_STEP(R) step<R>(f, s, groups)
    EMD_FFT_SWITCH(p.r[s], EMD_STEP)
    groups *= p.r[s];
    __syncthreads();
  }
#define EMD_LAST(R) last<R>(f)
  EMD_FFT_SWITCH(p.r[p.ns - 1], EMD_LAST)
}

__global__ void __launch_bounds__(256)
k_fft(FftPass pass, const void *__restrict__ vin, void *__restrict__ vout,
      const __grid_constant__ FftLine p, double c, double kappa,
      const double *__restrict__ inv_s, const double2 *__restrict__ roots) {
  extern __shared__ __align__(16) unsigned char sm[];
  const int n = p.n, nh = n / 2 + 1, stride = n | 1;
  const bool real = pass == FFT_X || pass == FFT_XINV;       // two lines as one
  FftCta f;
  f.pass = pass;
  f.nlines = n * (real ? n : nh);
  f.l0 = blockIdx.x << (p.lsh + real);
  f.in = static_cast<const double2 *>(vin);
  f.out = static_cast<double2 *>(vout);
  f.p = &p;
  f.roots = reinterpret_cast<double2 *>(sm);
  f.ex = f.roots + n;
  f.nat = f.ex + (p.ls << p.lsh);
  f.from_nat = real;
  f.to_nat = real || pass == FFT_Z;
  f.swap_in = pass == FFT_YINV;
  f.swap_out = pass == FFT_YINV;
  for (int t = threadIdx.x; t < n; t += blockDim.x) f.roots[t] = __ldg(roots + t);
  if (pass == FFT_X) {
    const double *x = static_cast<const double *>(vin);
#pragma unroll 4
    for (int t = threadIdx.x; t < n << p.lsh; t += blockDim.x) {
      const int l = t / p.by_n, i = t - l * n;
      // 8-byte loads: a caller's grid may start on any 8-byte boundary
      const int a = min(f.l0 + 2 * l, f.nlines - 1), b = min(a + 1, f.nlines - 1);
      f.nat[l * stride + i] =
          make_double2(__ldg(x + (size_t)a * n + i), __ldg(x + (size_t)b * n + i));
    }
  } else if (pass == FFT_XINV) {
#pragma unroll 4
    for (int t = threadIdx.x; t < nh << p.lsh; t += blockDim.x) {
      const int l = t / p.by_nh, k = t - l * nh;
      const int la = min(f.l0 + 2 * l, f.nlines - 1), lb = min(la + 1, f.nlines - 1);
      const double2 a = __ldg(f.in + (size_t)la * nh + k), b = __ldg(f.in + (size_t)lb * nh + k);
      double2 *z = f.nat + l * stride;
      // exchanged: inverse
      if (k == 0 || 2 * k == n) {
        z[k] = make_double2(b.x, a.x);
      } else {
        z[k] = make_double2(a.y + b.x, a.x - b.y);
        z[n - k] = make_double2(b.x - a.y, a.x + b.y);
      }
    }
  }
  __syncthreads();
  for (int half = pass == FFT_Z ? 0 : 1;; ++half) {
    line_fft(f);
    if (half) break;
    __syncthreads();
#pragma unroll 4
    for (int t = threadIdx.x; t < n << p.lsh; t += blockDim.x) {
      const int l = t / p.by_n, k = t - l * n, line = min(f.l0 + l, f.nlines - 1);
      const int kx = line / p.by_n, ky = line - kx * n;
      const int my = 2 * ky < n ? ky : ky - n, mz = 2 * k < n ? k : k - n;
      const int s = kx * kx + my * my + mz * mz;
      double g;
      if (kappa < 0.0)
        g = c * __ldg(inv_s + s);
      else
        g = s == 0 ? c : c * (double)s / ((double)s + kappa);
      double2 *v = f.nat + l * stride + k;
      *v = make_double2(g * v->y, g * v->x);                   // exchanged: inverse
    }
    f.from_nat = true;
    f.to_nat = false;
    f.swap_out = true;
    __syncthreads();
  }
  if (pass == FFT_X) {
    __syncthreads();
    for (int t = threadIdx.x; t < nh << p.lsh; t += blockDim.x) {
      const int k = t >> p.lsh, l = t & ((1 << p.lsh) - 1), a = f.l0 + 2 * l;
      const double2 zk = f.nat[l * stride + k], zr = f.nat[l * stride + (k ? n - k : 0)];
      double2 *o = f.out + (size_t)k * f.nlines + a;
      if (a < f.nlines) o[0] = make_double2(zk.x + zr.x, zk.y - zr.y);
      if (a + 1 < f.nlines) o[1] = make_double2(zk.y + zr.y, zr.x - zk.x);
    }
  } else if (pass == FFT_XINV) {
    __syncthreads();
    double *x = static_cast<double *>(vout);
    for (int t = threadIdx.x; t < n << p.lsh; t += blockDim.x) {
      const int l = t / p.by_n, i = t - l * n, a = f.l0 + 2 * l;
      const double2 v = f.nat[l * stride + i];
      if (a < f.nlines) x[(size_t)a * n + i] = v.y;
      if (a + 1 < f.nlines) x[(size_t)(a + 1) * n + i] = v.x;
    }
  }
}

// Grids above ~170 points need more than 48 KB of shared memory: asked for once
// per device (again for devices past the 64th, which changes nothing).
void allow_large_shared() {
  static std::atomic<bool> done[64];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return;     // the launch will fail and say so
  if (dev < 64 && done[dev].load(std::memory_order_acquire)) return;
  if (cudaFuncSetAttribute(k_fft, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)kFftMaxShared) == cudaSuccess && dev < 64)
    done[dev].store(true, std::memory_order_release);
}

}  // namespace

bool emd_fft2_ok(int n) { return fft_plan(n) != nullptr; }

// out = the inverse transform of the spectral factor times the transform of
// the real grid `in`.  in is read by the first pass only, so out may alias it;
// wa, wb: n^2 (n / 2 + 1) values each; roots: exp(-2 pi i t / n), t < n.
void emd_fft2_multiply(int n, const double *in, double *out, double2 *wa, double2 *wb,
                       const double2 *roots, double c, double kappa, const double *inv_s,
                       cudaStream_t st) {
  const int nh = n / 2 + 1;                       // (n + 1) / 2 for odd n
  const FftLine &p = *fft_plan(n);
  const int per = 1 << p.lsh;
  const int bx = (n * n + 2 * per - 1) / (2 * per), by = (nh * n + per - 1) / per;
  const size_t sm = fft_shared_bytes(p);
  if (sm > 49152) allow_large_shared();
  auto pass = [&](FftPass which, const void *src, void *dst, double scale) {
    const int blocks = which == FFT_X || which == FFT_XINV ? bx : by;
    k_fft<<<blocks, p.threads, sm, st>>>(which, src, dst, p, scale, kappa, inv_s, roots);
  };
  pass(FFT_X, in, wa, 0.0);
  pass(FFT_Y, wa, wb, 0.0);
  pass(FFT_Z, wb, wa, 0.5 * c);                   // the x pass leaves twice the spectrum
  pass(FFT_YINV, wa, wb, 0.0);
  pass(FFT_XINV, wb, out, 0.0);
}
