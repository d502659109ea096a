// FP64 Horner stage in double-float arithmetic (complex128 orbitals, bo = 2):
// u_out = psi0 + (-i a) H u_in, H = -1/2 nabla^2_FD + v_eff + sum_P h_P |p_P><p_P|
// (eq. new_EoM_a; the nested Taylor-4 polynomial of Sec. 5.1, four stages per
// exponential).
//
// GB300 issues one FP64 warp instruction per 16 SM cycles, and the plain FP64
// stage spends ~59 FP64 instructions per update.  Here every value is split
// into two floats, x = hi + lo (hi: the top 24 significand bits, lo: the rest
// rounded to 24 bits; 48 bits in all), by integer operations on its bits, and
// the stencil runs on the FP32 pipes: products by the integer FD numerators
// num_k (exact in FP32) through TwoProduct with an FMA, sums through Knuth's
// TwoSum, the rounding errors gathered in the low word.  The accumulated K =
// dv u + sum_k num_k S_k, dv = 3 num_0 - 2 h^2 den v_eff, gives H u = -K / (2
// h^2 den) + V_nl u; only the conversion of H u back to double and the Taylor
// update use FP64 instructions (four per update).
//
// What bounds it: FP32 issue.  An update at order 8 takes 302 packed FP32x2
// instructions of two issue cycles each; everything else is kept small:
//  * u_2, u_3, u_4 live between the stages as split values (16 bytes, like the
//    complex128 ones), and the last stage leaves its result in both forms, so
//    a value is split once, by the thread that computed it, instead of by each
//    of the three tiles that stage it and each of the atoms that project it.
//    The splits are those that the readers would have made: the results keep
//    their bits.
//  * Planes zi that lie in the z halo of the chunk only feed the z direction:
//    they skip the x/y shells and stage no x/y halo.
//  * The z direction accumulates in a register line of 2M+1 outputs per
//    point; three planes are unrolled, so the line moves by three slots once
//    per three planes and each ring slot is a compile-time constant.  Not at
//    order 8 with several projectors per atom: there the two more slots and the
//    epilogue in three copies crowd out the record loads (96^3, 9 projectors
//    per atom, 32 orbitals: 3.89 ms per launch unrolled, 3.05 one plane at a
//    time; order 6: 2.88 and 2.85, 4 projectors 1.46 either way).
//  * Projector entries past a warp's longest list are skipped.
// Each thread owns one orbital of one point of a 16 x 8 tile and marches
// through z; 256 threads, 128 registers, two CTAs per SM, so that one CTA
// computes while the other waits at its barrier.  Planes arrive by cp.async
// two ahead in a ring of three.
// Measured on 96^3 x 128 orbitals, order 8: 4.06 ms per launch before (one CTA
// of 512 threads, every staged value split by its tile), 2.85-2.90 ms with
// split input, 3.46 ms with complex128 input (568 instead of 707 instructions
// per update, FP32 pipe 59 % busy).  32^3 x 16, order 4: 60 -> 22 us.
#include "emd_internal.cuh"

namespace {

struct DFWeights {
  float num[EMD_MAX_HALF_ORDER + 1];   // FD numerators, exact in FP32
  float sk_hi, sk_lo;                  // -1 / (2 h^2 den) as double-float
  double dvs, dv0;                     // dv = dv0 + dvs v_eff
};

template <int M> struct DFTile {
  static constexpr int BO = 2;
  static constexpr int TX = 16, TY = 8;         // points per tile
  static constexpr int NT = TX * TY * BO;       // threads: (row, point, orbital)
  static constexpr int SW = TX + 2 * M, SH = TY + 2 * M;
  static constexpr int NCH = SH * SW * BO;      // complex values per staged plane
  static constexpr int CPT = (NCH + NT - 1) / NT;
  static constexpr int NV = TX * TY;            // tile points
  static constexpr int NS = 2 * M + 1;          // register line
  // ring slot (3, cp.async, two planes ahead): plane | diagonal of the tile
  // points | records and psi0 of the output plane completed by it
  static constexpr int RU = NCH * 16, RV = NV * 8, RQ = NV * 48, RP = NV * BO * 16;
  static constexpr int RSLOT = RU + RV + RQ + RP;
  // complex128 input only: split slot (2), plane | diagonal
  static constexpr int DSLOT = NCH * 16 + NV * 8;
};

// MP: several projectors per atom (the pre-split records past the first four
// are read with four in flight); a separate instantiation keeps the
// s-projector kernel's registers as they were.  IN / OUT: u_in / u_out as
// split values (float4) instead of complex128; IN reads the split diagonal dv.
// OUT = 2: complex128, and the split values over psi0: a point of psi0 is
// staged by the CTA that writes it, two planes before it writes it, and by no
// other, so the next exponential's first stage reads split values without a
// further orbital set.  psi0 is therefore neither const nor restrict.
template <int M, bool HCS, bool MP, bool IN, int OUT>
__global__ void __launch_bounds__(256, 2)
k_stage_df(const void *__restrict__ u_in, double2 *psi0,
           void *__restrict__ u_out, const double *__restrict__ v_eff,
           const float2 *__restrict__ dv, const int4 *__restrict__ pt4d,
           const int *__restrict__ pt_J, const double *__restrict__ pt_p,
           const int4 *__restrict__ pt_rec, const double2 *__restrict__ hc, int n, int ntx,
           int zc, int n_orb_pad, int n_proj, double a, int apply_only, DFWeights W) {
  typedef DFTile<M> Z;
  constexpr int BO = Z::BO, NS = Z::NS, SW = Z::SW, NT = Z::NT;
  constexpr int PH = MP && M == 4 ? 1 : 3;     // planes unrolled
  extern __shared__ __align__(16) unsigned char smraw[];
  unsigned char *dfbase = smraw + 3 * Z::RSLOT;
  float4 *hcs = reinterpret_cast<float4 *>(dfbase + (IN ? 0 : 2 * Z::DSLOT));
  const int tid = threadIdx.x;
  const int j = tid % BO, xl = tid / BO % Z::TX, yl = tid / (BO * Z::TX);
  const int tx0 = (blockIdx.x % ntx) * Z::TX, ty0 = (blockIdx.x / ntx) * Z::TY;
  const int z0 = blockIdx.y * zc;
  const int total = min(zc, n - z0) + 2 * M;
  const int n2 = n * n;
  const size_t n3 = (size_t)n2 * n;
  const size_t boff = (size_t)blockIdx.z * n3 * BO;
  const float4 *ub = static_cast<const float4 *>(u_in) + boff;   // 16-byte elements
  const double2 *pb = psi0 + boff;
  const int x = tx0 + xl, y = ty0 + yl;
  const bool valid = x < n && y < n;
  const size_t pxy = (size_t)min(y, n - 1) * n + min(x, n - 1);

  // staging map of the plane values: source index within a plane, -1 = none;
  // bit i of own: value i belongs to the tile itself (not its x/y halo)
  int src[Z::CPT];
  unsigned own = 0;
#pragma unroll
  for (int i = 0; i < Z::CPT; ++i) {
    const int q = tid + i * NT;
    src[i] = -1;
    if (q < Z::NCH) {
      const int jj = q % BO, pnt = q / BO;
      const int c = pnt % SW, rr = pnt / SW;
      const int xx = (tx0 - M + c + 2 * n) % n;
      const int yy = (ty0 - M + rr + 2 * n) % n;
      src[i] = (yy * n + xx) * BO + jj;
      if (c >= M && c < M + Z::TX && rr >= M && rr < M + Z::TY) own |= 1u << i;
    }
  }
  // tile point of this thread in the per-point stagings (diagonal, records)
  const int vp = tid < Z::NV ? min(ty0 + tid / Z::TX, n - 1) * n + min(tx0 + tid % Z::TX, n - 1)
                             : -1;
  if (HCS) {
    for (int i = tid; i < n_proj * BO; i += NT)
      hcs[i] = df_split2(hc[(size_t)(i / BO) * n_orb_pad + (size_t)blockIdx.z * BO + i % BO]);
  }
  const unsigned sm0 = (unsigned)__cvta_generic_to_shared(smraw);
  auto inner = [&](int zi) { return zi >= M && zi < total - M; };

  auto issue = [&](int zi) {
    const unsigned base = sm0 + (zi % 3) * Z::RSLOT;
    const bool in = inner(zi);
    int zz = z0 - M + zi;
    zz += zz < 0 ? n : 0;
    zz -= zz >= n ? n : 0;
    const size_t poff = (size_t)zz * n2;
    const float4 *up = ub + poff * BO;
#pragma unroll
    for (int i = 0; i < Z::CPT; ++i)
      if (src[i] >= 0 && (in || (own >> i & 1u)))
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(base + (tid + i * NT) * 16),
                     "l"(up + src[i]) : "memory");
    if (vp >= 0) {
      if (in)
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(base + Z::RU + tid * 8),
                     "l"((IN ? reinterpret_cast<const double *>(dv) : v_eff) + poff + vp) : "memory");
      if (zi >= 2 * M) {
        const size_t po = (size_t)(z0 + zi - 2 * M) * n2 + vp;
#pragma unroll
        for (int k = 0; k < 3; ++k)
          asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(
                           base + Z::RU + Z::RV + (tid * 3 + k) * 16),
                       "l"(pt4d + po * 3 + k) : "memory");
        if (!apply_only) {
#pragma unroll
          for (int jj = 0; jj < BO; ++jj)
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(
                             base + Z::RU + Z::RV + Z::RQ + (tid * BO + jj) * 16),
                         "l"(pb + po * BO + jj) : "memory");
        }
      }
    }
    cp_async_commit();
  };
  // complex128 input: split the raw plane zi into double-float slot zi & 1
  auto convert = [&](int zi) {
    const unsigned char *raw = smraw + (zi % 3) * Z::RSLOT;
    unsigned char *dst = dfbase + (zi & 1) * Z::DSLOT;
    const double2 *R = reinterpret_cast<const double2 *>(raw);
    float4 *D = reinterpret_cast<float4 *>(dst);
    const bool in = inner(zi);
#pragma unroll
    for (int i = 0; i < Z::CPT; ++i)
      if (src[i] >= 0 && (in || (own >> i & 1u))) D[tid + i * NT] = df_split2(R[tid + i * NT]);
    if (in && vp >= 0)
      reinterpret_cast<float2 *>(dst + Z::RU)[tid] =
          df_split(__fma_rn(W.dvs, reinterpret_cast<const double *>(raw + Z::RU)[tid], W.dv0));
  };

  // at phase ph of a group of PH planes, [s + ph]: output plane zi - M + s,
  // K as hi = (re, im), lo = (re, im)
  float2 ah[NS + PH - 1], al[NS + PH - 1];
#pragma unroll
  for (int s = 0; s < NS + PH - 1; ++s) ah[s] = al[s] = make_float2(0.f, 0.f);
  const int ci = ((yl + M) * SW + xl + M) * BO + j;        // centre, float4 index
  const int pt = yl * Z::TX + xl;                          // tile point index
  const char *hcj = reinterpret_cast<const char *>(hcs + j);
  const double2 *hcg = hc + (size_t)blockIdx.z * BO + j;

  issue(0);
  if (total > 1) issue(1);
  if (!IN) {
    if (total > 1) cp_async_wait<1>();
    else cp_async_wait<0>();
    __syncthreads();
    convert(0);
  }
  for (int zg = 0; zg < total; zg += PH) {
#pragma unroll
    for (int ph = 0; ph < PH; ++ph) {
      const int zi = zg + ph;
      if (zi >= total) break;
      // IN: planes zi and zi + 1 are in flight, wait for zi.  Else raw plane
      // zi + 1 (issued one iteration ago) is the only group in flight.
      if (IN && zi + 1 < total) cp_async_wait<1>();
      else cp_async_wait<0>();
      // one barrier: the copies (and the split of plane zi, made in the last
      // iteration) are visible, and every thread has finished iteration zi - 1,
      // so the slots of zi + 2 and of the split of zi + 1 are free
      __syncthreads();
      if (zi + 2 < total) issue(zi + 2);
      if (!IN && zi + 1 < total) convert(zi + 1);
      const unsigned char *raw = smraw + (PH == 3 ? ph : zi % 3) * Z::RSLOT;
      const unsigned char *base = IN ? raw : dfbase + (zi & 1) * Z::DSLOT;
      const float4 *P = reinterpret_cast<const float4 *>(base) + ci;
      const float4 c = P[0];
      const float2 ch = f4hi(c), cl = f4lo(c);
      if (inner(zi)) {                         // own plane: dv u + the x/y shells
        const float2 d = reinterpret_cast<const float2 *>(base + Z::RU)[pt];
        dfp_add_prod(ah[M + ph], al[M + ph], d.x, d.y, ch, cl);
#pragma unroll
        for (int k = 1; k <= M; ++k) {
          const float4 v1 = P[k * BO], v2 = P[-k * BO], v3 = P[k * SW * BO], v4 = P[-k * SW * BO];
          float2 sh = f4hi(v1), sl = f4lo(v1);
          dfp_add(sh, sl, f4hi(v2), f4lo(v2));
          dfp_add(sh, sl, f4hi(v3), f4lo(v3));
          dfp_add(sh, sl, f4hi(v4), f4lo(v4));
          const float2 w2 = make_float2(W.num[k], W.num[k]);
          float2 p, pe;
          dfp_two_prod(w2, sh, p, pe);
          dfp_add(ah[M + ph], al[M + ph], p, __ffma2_rn(w2, sl, pe));
        }
      }
      // z-direction: this plane is neighbour k of output planes zi +- k
      // (planes before the chunk's first output leave the line unstored);
      // zi + M enters the line here
#pragma unroll
      for (int k = 1; k <= M; ++k) {
        const float2 w2 = make_float2(W.num[k], W.num[k]);
        float2 p, pe;
        dfp_two_prod(w2, ch, p, pe);
        const float2 q = __ffma2_rn(w2, cl, pe);
        if (k == M) {
          ah[M + k + ph] = p;
          al[M + k + ph] = q;
        } else {
          dfp_add(ah[M + k + ph], al[M + k + ph], p, q);
        }
        dfp_add(ah[M - k + ph], al[M - k + ph], p, q);
      }
      if (zi >= 2 * M) {   // output plane z0 + zi - 2M is complete in slot 0
        const int4 *Q = reinterpret_cast<const int4 *>(raw + Z::RU + Z::RV) + pt * 3;
        const int4 q0 = Q[0], q1 = Q[1], q2 = Q[2];
        float2 hh = make_float2(0.f, 0.f), hl = make_float2(0.f, 0.f);
        dfp_add_prod(hh, hl, W.sk_hi, W.sk_lo, ah[ph], al[ph]);
        // four entries (unused ones have p = 0 and add exactly zero)
        const int cnt = q0.x >> 16;
        const int Je[4] = {q0.x & 0xffff, q0.y, q0.z, q0.w};
        const float ep[4] = {__int_as_float(q1.x), __int_as_float(q1.z), __int_as_float(q2.x),
                             __int_as_float(q2.z)};
        const float el[4] = {__int_as_float(q1.y), __int_as_float(q1.w), __int_as_float(q2.y),
                             __int_as_float(q2.w)};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          if (!__any_sync(0xffffffffu, cnt > e)) break;
          const float4 h4 = HCS ? *reinterpret_cast<const float4 *>(hcj + Je[e] * (BO * 16))
                                : df_split2(hcg[(size_t)Je[e] * n_orb_pad]);
          dfp_add_prod(hh, hl, ep[e], el[e], f4hi(h4), f4lo(h4));
        }
        const size_t po = (size_t)(z0 + zi - 2 * M) * n2 + pxy;
        if (cnt > 4) {
          if (MP) {
            // several projectors per atom: pre-split 16-byte records, four in
            // flight, summed into four independent pairs (combined in a fixed
            // order) so that the TwoSum chains overlap
            float2 xh[4], xs[4];
#pragma unroll
            for (int v = 0; v < 4; ++v) xh[v] = xs[v] = make_float2(0.f, 0.f);
            for (int e = 4; e < cnt; e += 4) {
              int4 q[4];
#pragma unroll
              for (int v = 0; v < 4; ++v)
                q[v] = e + v < cnt ? __ldg(pt_rec + (size_t)(e + v) * n3 + po)
                                   : make_int4(0, 0, 0, 0);
#pragma unroll
              for (int v = 0; v < 4; ++v) {
                const float4 h4 = HCS ? *reinterpret_cast<const float4 *>(hcj + q[v].x * (BO * 16))
                                      : df_split2(hcg[(size_t)q[v].x * n_orb_pad]);
                dfp_add_prod(xh[v], xs[v], __int_as_float(q[v].y), __int_as_float(q[v].z),
                             f4hi(h4), f4lo(h4));
              }
            }
#pragma unroll
            for (int v = 0; v < 4; ++v) dfp_add(hh, hl, xh[v], xs[v]);
          } else {
            for (int e = 4; e < cnt; ++e) {
              const int J = pt_J[(size_t)e * n3 + po];
              const float2 pv = df_split(pt_p[(size_t)e * n3 + po]);
              const float4 h4 = HCS ? *reinterpret_cast<const float4 *>(hcj + J * (BO * 16))
                                    : df_split2(hcg[(size_t)J * n_orb_pad]);
              dfp_add_prod(hh, hl, pv.x, pv.y, f4hi(h4), f4lo(h4));
            }
          }
        }
        const double Hr = __dadd_rn(df_widen(hh.x), df_widen(hl.x));
        const double Hi = __dadd_rn(df_widen(hh.y), df_widen(hl.y));
        double2 out;
        if (apply_only) {
          out = make_double2(Hr, Hi);
        } else {
          const double2 sv =
              reinterpret_cast<const double2 *>(raw + Z::RU + Z::RV + Z::RQ)[pt * BO + j];
          out.x = __fma_rn(a, Hi, sv.x);
          out.y = __fma_rn(-a, Hr, sv.y);
        }
        if (valid) {
          const size_t o = boff + po * BO + j;
          if (OUT == 1) static_cast<float4 *>(u_out)[o] = df_split2(out);
          else static_cast<double2 *>(u_out)[o] = out;
          if (OUT == 2) reinterpret_cast<float4 *>(psi0)[o] = df_split2(out);
        }
      }
    }
    // the next group's planes find output zi - M + s in slot s again
#pragma unroll
    for (int s = 0; s + PH < NS + PH - 1; ++s) {
      ah[s] = ah[s + PH];
      al[s] = al[s + PH];
    }
  }
}

template <int M, bool HCS, bool MP, bool IN, int OUT>
void stage_df_tt(const OrbLayout &o, const StageArgs &a, cudaStream_t st) {
  typedef DFTile<M> Z;
  const int fixed = 3 * Z::RSLOT + (IN ? 0 : 2 * Z::DSLOT);
  static bool attr_done = false;
  if (!attr_done) {
    cudaFuncSetAttribute(k_stage_df<M, HCS, MP, IN, OUT>,
                         cudaFuncAttributeMaxDynamicSharedMemorySize, fixed + 32768);
    attr_done = true;
  }
  const int ntx = (o.n + Z::TX - 1) / Z::TX, nty = (o.n + Z::TY - 1) / Z::TY;
  const int cols = ntx * nty * o.n_blk;
  const int zc = o.zchunk > 0 ? std::min(o.zchunk, o.n)
                              : emd_zchunk(o.n, o.half_order, cols, 0.3, 0);
  DFWeights W;
  for (int k = 0; k <= EMD_MAX_HALF_ORDER; ++k) W.num[k] = (float)o.num[k];
  const double sk = -1.0 / (2.0 * o.h * o.h * o.den);
  W.sk_hi = (float)sk;
  W.sk_lo = (float)(sk - (double)W.sk_hi);
  W.dvs = o.dv_scale();
  W.dv0 = o.dv_shift();
  const int smem = fixed + (HCS ? o.n_proj * Z::BO * (int)sizeof(float4) : 0);
  dim3 grid(ntx * nty, (o.n + zc - 1) / zc, o.n_blk);
  k_stage_df<M, HCS, MP, IN, OUT><<<grid, Z::NT, smem, st>>>(
      a.u_in, (double2 *)const_cast<void *>(a.psi0), a.u_out, (const double *)a.v_eff,
      (const float2 *)a.v_diag, a.tab->pt4d, a.tab->pt_J, a.tab->pt_p, a.tab->pt_rec,
      (const double2 *)a.hc, o.n, ntx, zc, o.n_orb_pad, o.n_proj, a.a, a.apply_only, W);
}

template <int M, bool MP, bool HCS>
void stage_df_t(const OrbLayout &o, const StageArgs &a, cudaStream_t st) {
  if (a.in_split && a.out_split == 2) stage_df_tt<M, HCS, MP, true, 2>(o, a, st);
  else if (a.in_split) stage_df_tt<M, HCS, MP, true, 1>(o, a, st);
  else if (a.out_split) stage_df_tt<M, HCS, MP, false, 1>(o, a, st);
  else stage_df_tt<M, HCS, MP, false, 0>(o, a, st);
}

template <int M>
void stage_df_m(const OrbLayout &o, const StageArgs &a, cudaStream_t st) {
  // h c of every projector as split pairs in shared memory, up to 32 KB (1024
  // projectors); more read it from global memory.  Both take split sets: with
  // complex128 sets above 1024 (216 atoms of 9 projectors, 96^3, 64 orbitals,
  // order 8) a step took 77.8 ms, 76.9 before the split sets, 73.8 now.
  const bool hcs = o.n_proj * 2 * (int)sizeof(float4) <= 32768;
  if (a.tab->pt_rec) {
    if (hcs) stage_df_t<M, true, true>(o, a, st);
    else stage_df_t<M, true, false>(o, a, st);
  } else {
    if (hcs) stage_df_t<M, false, true>(o, a, st);
    else stage_df_t<M, false, false>(o, a, st);
  }
}

}  // namespace

void emd_launch_stage_df(const OrbLayout &o, const StageArgs &a, cudaStream_t st) {
  switch (o.half_order) {
    case 1: stage_df_m<1>(o, a, st); break;
    case 2: stage_df_m<2>(o, a, st); break;
    case 3: stage_df_m<3>(o, a, st); break;
    case 4: stage_df_m<4>(o, a, st); break;
  }
}
