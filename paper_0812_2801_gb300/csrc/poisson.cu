// Hartree/ionic electrostatics by a periodic spectral Poisson solve, the
// Perdew-Zunger LDA, the effective potential of each AETRS half and
// deterministic grid reductions.
//
// Paper: the Hartree term of E_KS (eq. E_KS) and the ionic potential
// (eq. ionicpotential) are electrostatic potentials; the paper's finite
// systems use an interpolating-scaling-function Poisson solver (Sec. 5), the
// periodic boxes here solve nabla^2 v = -4 pi n in Fourier space with the
// G = 0 component set to zero.  XC: Perdew-Zunger LDA (Sec. 5), adiabatic
// (instantaneous density, Sec. 4.1).  H(t+dt) of AETRS uses a v_Hxc
// extrapolated from previous steps (Sec. 5.1, eq. aetrs).
//
// The transforms are in fft2.cu; here are their tables of roots, kept per grid
// size, and the entry point that allocates nothing.
#include <cmath>
#include <mutex>
#include <vector>
#include "emd_internal.cuh"

namespace {

// exp(-2 pi i num / den) evaluated in extended precision on the host.
double2 unit_root(long num, long den) {
  const long double PI_L = 3.141592653589793238462643383279502884L;
  const long double ang = -2.0L * PI_L * (long double)num / (long double)den;
  return make_double2((double)cosl(ang), (double)sinl(ang));
}

// Perdew-Zunger LDA (unpolarised): eps_xc, v_xc; vhxc = v_h + v_xc.
__global__ void k_lda(int n3, const double *rho, const double *vh,
                      double *eps, double *vxc, double *vhxc) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n3) return;
  const double r = rho[i];
  double e = 0.0, v = 0.0;
  if (r >= 1e-30) {
    // one root: with c = r^(-1/3), (3 r / pi)^(1/3) = c1 r c^2 and r_s = c2 c
    // (FP64 instructions are the cost; a cube root and three divisions took
    // 17 us on 48^3 and 192 us on 120^3)
    const double rc = rcbrt(r);
    const double ex = -0.75 * (0.98474502184269654115 * (r * rc * rc));   // (3/pi)^(1/3)
    const double vx = (4.0 / 3.0) * ex;
    const double rs = 0.62035049089940001667 * rc;                        // (3/(4 pi))^(1/3)
    double ec, vc;
    if (rs >= 1.0) {
      using namespace pz81;
      const double s = sqrt(rs);
      const double iq = 1.0 / (1.0 + b1 * s + b2 * rs);
      ec = gam * iq;
      vc = ec * (1.0 + (7.0 / 6.0) * b1 * s + (4.0 / 3.0) * b2 * rs) * iq;
    } else {
      using namespace pz81;
      const double lx = log(rs);
      ec = A * lx + B + C * rs * lx + D * rs;
      vc = A * lx + (B - A / 3.0) + (2.0 / 3.0) * C * rs * lx +
           ((2.0 * D - C) / 3.0) * rs;
    }
    e = ex + ec;
    v = vx + vc;
  }
  eps[i] = e;
  vxc[i] = v;
  vhxc[i] = vh[i] + v;
}

// v_eff = v_loc + extrapolated v_Hxc + field * (z - L/2).
__global__ void k_veff(int n, double h, double L, const double *vloc,
                       const double *h0, const double *h1, const double *h2,
                       int hist_len, double field, double *ve, float *vef,
                       float4 *vdiag, double w0, float2 *vsplit, double dvs, double dv0) {
  const int n3 = n * n * n;
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n3) return;
  double x;
  if (hist_len <= 1)
    x = h0[i];
  else if (hist_len == 2)
    x = 2.0 * h0[i] - h1[i];
  else
    x = 3.0 * h0[i] - 3.0 * h1[i] + h2[i];
  double v = vloc[i] + x;
  if (field != 0.0) {
    const int z = i / (n * n);
    v += field * (z * h - 0.5 * L);
  }
  ve[i] = v;
  if (vef) vef[i] = (float)v;
  if (vsplit) vsplit[i] = df_split(__fma_rn(dvs, v, dv0));
  if (vdiag) {
    const float d = (float)(w0 + v);
    vdiag[i] = make_float4(d, d, d, d);
  }
}

// partial[b] = sum over block b of (a - c)(b + d) (c, d optional).
__global__ void __launch_bounds__(256)
k_dot4(int n, const double *a, const double *b, const double *c,
       const double *d, double *part) {
  __shared__ double red[8];
  double acc[1] = {0.0};
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += gridDim.x * blockDim.x) {
    const double x = c ? a[i] - c[i] : a[i];
    const double y = b ? (d ? b[i] + d[i] : b[i]) : 1.0;
    acc[0] += x * y;
  }
  emd_block_sum<1>(acc, red);
  if (threadIdx.x == 0) part[blockIdx.x] = acc[0];
}

__global__ void __launch_bounds__(256)
k_sum(const double *part, int n, double *out) {
  __shared__ double red[8];
  double acc[1] = {0.0};
  for (int i = threadIdx.x; i < n; i += blockDim.x) acc[0] += part[i];
  emd_block_sum<1>(acc, red);
  if (threadIdx.x == 0) *out = acc[0];
}

// Tables of a grid size, one per (device, grid size), created on first use and
// kept for the life of the process.
struct PlanCache {
  int dev = -1, n = -1;
  double2 *roots = nullptr;  // exp(-2 pi i t / n), t < n
  double *inv_s = nullptr;   // 1 / s for s = 0 .. 3 (n/2)^2, inv_s[0] = 0
};
std::mutex g_plan_mu;
std::vector<PlanCache *> g_plans;

const PlanCache *get_plan(int n) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return nullptr;
  std::lock_guard<std::mutex> lk(g_plan_mu);
  for (PlanCache *c : g_plans)
    if (c->n == n && c->dev == dev) return c;
  if (!emd_fft2_ok(n)) return nullptr;
  std::vector<double2> w(n);
  for (int t = 0; t < n; ++t) w[t] = unit_root(t, n);
  const int smax = 3 * (n / 2) * (n / 2);
  std::vector<double> inv(smax + 1);
  inv[0] = 0.0;
  for (int q = 1; q <= smax; ++q) inv[q] = 1.0 / (double)q;
  PlanCache *c = new PlanCache();
  c->n = n;
  c->dev = dev;
  if (cudaMalloc(&c->roots, w.size() * sizeof(double2)) != cudaSuccess ||
      cudaMemcpy(c->roots, w.data(), w.size() * sizeof(double2), cudaMemcpyHostToDevice) !=
          cudaSuccess ||
      cudaMalloc(&c->inv_s, inv.size() * sizeof(double)) != cudaSuccess ||
      cudaMemcpy(c->inv_s, inv.data(), inv.size() * sizeof(double), cudaMemcpyHostToDevice) !=
          cudaSuccess) {
    if (c->roots) cudaFree(c->roots);
    if (c->inv_s) cudaFree(c->inv_s);
    delete c;
    return nullptr;
  }
  g_plans.push_back(c);
  return c;
}

}  // namespace

void emd_fft_plan_check(int n, int *ok) { *ok = emd_fft2_ok(n); }

int emd_fft_prepare(int n) { return get_plan(n) == nullptr; }

namespace {

// v = the inverse transform of factor(s) times the transform of the real grid
// `charge` (kappa < 0: Poisson's c / s, else Kerker's c s / (s + kappa); c
// includes the 1/N^3 of the inverse); v may alias `charge`
void spectral_multiply(const GridInfo &g, const double *charge, double *v, double2 *wa,
                       double2 *wb, double c, double kappa, cudaStream_t st) {
  const PlanCache *pc = get_plan(g.n);
  emd_note_launches(5);
  emd_fft2_multiply(g.n, charge, v, wa, wb, pc->roots, c, kappa, pc->inv_s, st);
}

}  // namespace

// 4 pi / ((2 pi / L)^2 N^3) with L = n h, rounded once
static double poisson_scale(int n, double h) {
  const long double PI_L = 3.141592653589793238462643383279502884L;
  return (double)((long double)h * h / (PI_L * n));
}

void emd_launch_poisson(const GridInfo &g, const double *charge, double *v,
                        double2 *wa, double2 *wb, cudaStream_t st) {
  spectral_multiply(g, charge, v, wa, wb, poisson_scale(g.n, g.h), -1.0, st);
}

void emd_launch_kerker(const GridInfo &g, double q0, const double *r, double *out,
                       double2 *wa, double2 *wb, cudaStream_t st) {
  const double k = q0 * g.L / (2.0 * M_PI);
  spectral_multiply(g, r, out, wa, wb, 1.0 / (double)g.n3, k * k, st);
}

void emd_launch_lda(int n3, const double *rho, const double *v_h,
                    double *eps_xc, double *v_xc, double *vhxc,
                    cudaStream_t st) {
  emd_note_launches(1);
  k_lda<<<(n3 + 255) / 256, 256, 0, st>>>(n3, rho, v_h, eps_xc, v_xc, vhxc);
}

void emd_launch_veff(const GridInfo &g, const double *v_loc,
                     const double *const *hist, int hist_len, double field,
                     double *v_eff, float *v_eff_f, cudaStream_t st,
                     float4 *v_diag, double w0, float2 *v_split, double dv_scale,
                     double dv_shift) {
  emd_note_launches(1);
  k_veff<<<(g.n3 + 255) / 256, 256, 0, st>>>(
      g.n, g.h, g.L, v_loc, hist[0], hist_len > 1 ? hist[1] : hist[0],
      hist_len > 2 ? hist[2] : hist[0], hist_len, field, v_eff, v_eff_f, v_diag, w0,
      v_split, dv_scale, dv_shift);
}

void emd_launch_dot_partials(int n3, const double *a, const double *b,
                             const double *c, const double *d,
                             double *partials, int nblocks, cudaStream_t st) {
  emd_note_launches(1);
  k_dot4<<<nblocks, 256, 0, st>>>(n3, a, b, c, d, partials);
}

void emd_launch_sum(const double *partials, int n, double *out,
                    cudaStream_t st) {
  emd_note_launches(1);
  k_sum<<<1, 256, 0, st>>>(partials, n, out);
}

// ===========================================================================
// Poisson solve that allocates nothing (emd_poisson_static).
//
// For callers that cannot allocate device memory: code that runs while a
// CUDA graph is being captured (cudaMalloc is not capturable), applications
// whose device memory is owned by another allocator or a fixed budget, and
// latency-critical loops where cudaMalloc/cudaFree would synchronise the
// device.  The FFT work arrays and the table of roots live in one file-scope
// __device__ array of fixed size, present on every GPU that loads the
// library until the process exits.
// ===========================================================================
namespace {

constexpr int kStaticMaxN = 64;                       // largest grid edge
constexpr size_t kStaticN3 = (size_t)kStaticMaxN * kStaticMaxN * kStaticMaxN;
constexpr int kStaticMaxS = 3 * (kStaticMaxN / 2) * (kStaticMaxN / 2);
// [0, N^3): work a, [N^3, 2 N^3): work b, then the roots, then 1 / s
__device__ __align__(256) double2 g_static_scratch[2 * kStaticN3 + kStaticMaxN +
                                                   kStaticMaxS / 2 + 1];

constexpr int kMaxDevices = 64;
std::mutex g_static_mu;
double2 *g_static_ptr[kMaxDevices] = {};

// Device address of g_static_scratch on the current device (set-up on the
// first call per device).  In host code the symbol is only a stand-in.
cudaError_t static_scratch(double2 **out) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lk(g_static_mu);
  if (!g_static_ptr[dev]) {
    void *p = nullptr;
    e = cudaGetSymbolAddress(&p, g_static_scratch);
    if (e != cudaSuccess) return e;
    g_static_ptr[dev] = static_cast<double2 *>(p);
  }
  *out = g_static_ptr[dev];
  return cudaSuccess;
}

// roots: exp(-2 pi i t / n), t < n; inv_s[s] = 1 / s, s = 1 .. smax, 0 at 0.
// An angle is brought to its octant in integers first: the rounding of -2 t /
// n as an argument near 2 would turn the root by up to 3.5e-16.
__global__ void k_fill_tables(int n, double2 *roots, int smax, double *inv_s) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t < n) {
    const int o = 8 * t / n;                                  // octant
    const int num = o & 1 ? (o + 1) * n - 8 * t : 8 * t - o * n;
    double sn, cs;                                            // 0 .. pi / 4
    sincospi((double)num / (double)(4 * n), &sn, &cs);
    const bool swap = (o + 1) & 2;                            // octants 1, 2, 5, 6
    const double x = swap ? sn : cs, y = swap ? cs : sn;
    roots[t] = make_double2(o >= 2 && o < 6 ? -x : x, o < 4 ? -y : y);
  }
  if (t <= smax) inv_s[t] = t ? 1.0 / (double)t : 0.0;
}

}  // namespace

extern "C" int emd_poisson_static(int n, double h, const double *charge,
                                  double *v, void *cuda_stream) {
  if (!charge || !v || !(h > 0.0) || n < 2)
    return emd_set_error(EMD_EINVAL, "emd_poisson_static: NULL pointer, h <= 0 or n < 2");
  if (n > kStaticMaxN)
    return emd_set_error(EMD_EINVAL, "emd_poisson_static: n exceeds the static "
                                     "scratch limit of 64 points per axis");
  if (!emd_fft2_ok(n))
    return emd_set_error(EMD_EINVAL, "emd_poisson_static: n has a prime factor above 13");
  double2 *base = nullptr;
  if (static_scratch(&base) != cudaSuccess)
    return emd_set_error(EMD_ECUDA, "emd_poisson_static: cudaGetSymbolAddress of "
                                    "the static scratch failed");
  double2 *wa = base, *wb = base + kStaticN3, *tab = base + 2 * kStaticN3;
  cudaStream_t st = (cudaStream_t)cuda_stream;
  double *inv_s = reinterpret_cast<double *>(tab + kStaticMaxN);
  const int smax = 3 * (n / 2) * (n / 2);
  k_fill_tables<<<smax / 64 + 1, 64, 0, st>>>(n, tab, smax, inv_s);
  emd_fft2_multiply(n, charge, v, wa, wb, tab, poisson_scale(n, h), -1.0, inv_s, st);
  if (cudaGetLastError() != cudaSuccess)
    return emd_set_error(EMD_ECUDA, "emd_poisson_static: kernel launch failed");
  return emd_set_error(EMD_OK, "");
}
