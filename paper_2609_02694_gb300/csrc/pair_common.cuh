// pair_common.cuh -- pair interaction of the real-space part (Eqs. F_i, G_short, LJ) shared
// by the cell-list kernel and the random batch list kernel.
#pragma once
#include <cuda_fp16.h>

#include <cmath>

#include "f32x2.cuh"
#include "rbe_internal.cuh"

namespace rbe {

constexpr int kPairWarps = 1;  // one-warp blocks: a finished warp frees its slot at once

struct PairArgs {
  PairSet set;
  Grid grid;
  PairConst pc;
  // single-type LJ coefficients (as in LJTable)
  float ljA, ljB, ljA12, ljB6;
  double ljAd, ljBd, ljA12d, ljB6d;
  const LJTable *table;  // device copy, multi-type only
  float *F;
  double *Fd;
  int64_t Fstride;   // N of the force arrays (SoA stride)
  int accumulate;    // add to F instead of overwriting
  double *epart;     // per-block partials (NQ_PAIR doubles each)
  int32_t *nbr;      // per-particle neighbour counts (sorted order of the set), nullable
  // Coarse-test frame: coordinates relative to the group leader are a valid minimum
  // image only while (distance of a member from the leader) + r_c < L/2 on every axis.
  // A group spans at most `smax` cells in x (one cell in y and z); boxes too small for
  // even one cell use the wrapping variant, which folds every difference into [-L/2, L/2).
  int smax;
  int trim;           // cut each row's run to the group's x-reach (rows are sorted by x)
  float L[3], invL[3];
  int comp;  // compensated (Kahan) Coulomb energy and virial sums
  // Packed half-precision candidate test: frame coordinates scaled by scale16 = 8 / r_c
  // (the cutoff maps to 8), compared with thr16 = 66.5 > 64 + the worst rounding of the
  // test (2.06 for |coordinate| < 64 scaled units, which smax16 guarantees). No true
  // neighbour is rejected; the exact decision is taken again when the pair is evaluated.
  float scale16;
  int smax16;
  // The work of a tile of 32 particles shared by nsplit one-warp blocks (small systems): block
  // part p sums every candidate chunk of its share into part p of Fpart ([nsplit][3][N]), which
  // pair_sum_kernel adds up in order. nsplit 1: straight to F.
  int nsplit;
  double *Fpart;
  int64_t wfix[2];       // 2^48 / cells in y and z (rounded down): a cell's width
  // FP64 form: r^2 and force factors in grid units of x: h_d / h_x, the band around r_c^2, (h_y /
  // h_x)^2, (h_z / h_x)^2, h_d / h_x^2, h_x, 1 / h_x, h_x^-6, and the single-type LJ coefficients times
  // h_x^-12 and h_x^-6
  float gh[3], glo, ghi;
  double ry, rz, fs[3], hx, ihx, ih6, A12s, B6s;
  int cubic;
  // Verlet-list build (the cell kernel's BUILD variant): pc's cutoff fields then hold
  // r_list = r_c + skin, and every j != i with r_ij^2 <= r_list^2 (1 + 1e-5) in FP32 is
  // appended to i's list: warp-interleaved, entry t of the particle in slot i at
  // list[((i / 32) * K + t) * 32 + i % 32].
  int32_t *list, *len;
  int K;
  const int32_t *gate;   // build only when *gate != 0
  int32_t *maxlen;       // longest list (atomic max)
  int *err;
};

// Fold a coordinate difference into [-L/2, L/2) (only the small-box variants use it).
__device__ __forceinline__ float fold(float d, float L, float invL) {
  return mad(-L, rintf(d * invL), d);
}

template <typename real>
struct PairAcc {
  real fx, fy, fz, ulj, wlj, uc, wc;
  real cuc, cwc;  // Kahan compensations of uc, wc (compensated form)
  int nbr;
};

template <typename real>
__device__ __forceinline__ void kahan_add(real &s, real &c, real x) {
  const real y = x - c;
  const real t = s + y;
  c = (t - s) - y;
  s = t;
}

__device__ __forceinline__ float rcp_approx(float x) {
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float min3(float a, float b, float c) {
  float r;
  asm("min.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}
__device__ __forceinline__ float max3(float a, float b, float c) {
  float r;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}
// erfc(sqrt(alpha) r) and exp(-alpha r^2) of a packed pair, r <= r_c, by the handle's fit
// (f.ok). The exponent's rounding and alpha log2(e)'s low part go into a linear correction, so
// the exponential is as close as the unit's 2^x (2 ulp). A third of erfcf and expf's
// instructions: the Coulomb pair terms were two thirds of a charged pair.
__device__ __forceinline__ float ex2_approx(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ void erfc_exp2(const ErfcFit &f, f32x2 r, f32x2 r2, f32x2 &er,
                                          f32x2 &ex) {
  const f32x2 t = fma2(r, pk(f.ts), pk(-1.f));
  f32x2 p = pk(f.c[kErfcDeg]);
#pragma unroll
  for (int k = kErfcDeg - 1; k >= 0; --k) p = fma2(p, t, pk(f.c[k]));
  const f32x2 nea = pk(-f.ea), arg = mul2(r2, pk(f.ea));
  const f32x2 d = fma2(r2, pk(-f.ea_lo), fma2(r2, nea, arg));
  const f32x2 e = pk(ex2_approx(-arg.x), ex2_approx(-arg.y));
  ex = fma2(e, mul2(d, pk(0.693147181f)), e);
  er = mul2(ex, p);
}

// One value of each.
__device__ __forceinline__ void erfc_exp1(const ErfcFit &f, float r, float r2, float &er, float &ex) {
  const float t = fmaf(r, f.ts, -1.f);
  float p = f.c[kErfcDeg];
#pragma unroll
  for (int k = kErfcDeg - 1; k >= 0; --k) p = fmaf(p, t, f.c[k]);
  const float arg = r2 * f.ea, d = fmaf(r2, -f.ea_lo, fmaf(r2, -f.ea, arg)), e = ex2_approx(-arg);
  ex = fmaf(e, d * 0.693147181f, e);
  er = ex * p;
}

// Squared distance of the exact cutoff decision (the oracle's definition): dx_d =
// (int32)(s_i - s_j) * (L_d / 2^32) and r2 = dx^2 + dy^2 + dz^2 in FP64, no FMA.
__device__ __forceinline__ double exact_r2(const PairConst &pc, int dsx, int dsy, int dsz) {
  const double ex = __dmul_rn(i2d(dsx), pc.hd[0]);
  const double ey = __dmul_rn(i2d(dsy), pc.hd[1]);
  const double ez = __dmul_rn(i2d(dsz), pc.hd[2]);
  return __dadd_rn(__dadd_rn(__dmul_rn(ex, ex), __dmul_rn(ey, ey)), __dmul_rn(ez, ez));
}

// LJ terms of one pair from 1/r^2 (types ti, tj): force factor gl (F_i = gl (r_i - r_j)),
// energy u = A r^-12 - B r^-6 and virial w = gl r^2 = r^-6 (12 A r^-6 - 6 B). With
// 1/r^2 = 0 all three are exact zeros.
template <typename real, bool MULTI>
__device__ __forceinline__ void lj_terms(const PairArgs &a, const LJTable *tab, int ti, int tj,
                                         real ir2, real &gl, real &u, real &w) {
  real A, B, A12, B6;
  if (MULTI) {
    const int pt = ti * tab->nt + tj;
    if (sizeof(real) == 8) { A = (real)tab->Ad[pt]; B = (real)tab->Bd[pt]; A12 = (real)tab->A12d[pt]; B6 = (real)tab->B6d[pt]; }
    else { A = (real)tab->A[pt]; B = (real)tab->B[pt]; A12 = (real)tab->A12[pt]; B6 = (real)tab->B6[pt]; }
  } else {
    if (sizeof(real) == 8) { A = (real)a.ljAd; B = (real)a.ljBd; A12 = (real)a.ljA12d; B6 = (real)a.ljB6d; }
    else { A = (real)a.ljA; B = (real)a.ljB; A12 = (real)a.ljA12; B6 = (real)a.ljB6; }
  }
  const real ir6 = ir2 * ir2 * ir2;
  w = ir6 * mad(A12, ir6, -B6);
  gl = w * ir2;
  u = ir6 * mad(A, ir6, -B);
}

// Pair force, energies and virial of one pair that is inside the cutoff (Eqs. F_i, G_short, LJ),
// added to acc: the FP64 form's random batch list.
template <bool COUL, bool MULTI>
__device__ __forceinline__ void pair_force_v(const PairArgs &a, const LJTable *tab, double dx,
                                             double dy, double dz, double r2, double qi, int ti,
                                             double qj, int tj, PairAcc<double> &acc) {
  const PairConst &pc = a.pc;
  double g, u, w;
  lj_terms<double, MULTI>(a, tab, ti, tj, 1.0 / r2, g, u, w);
  acc.ulj += u;
  acc.wlj += w;
  if (COUL) {
    const double qq = qi * qj;
    if (qq != 0.0) {
      const double r = sqrt(r2), rinv = 1.0 / r;
      const double erfcv = erfc(pc.sqrt_alpha_d * r), expv = exp(-pc.alpha_d * r2);
      const double Cqq = pc.C_d * qq, rinv2 = rinv * rinv;
      const double gc =
          Cqq * mad(erfcv * rinv, rinv2, pc.two_sqrt_alpha_over_sqrt_pi_d * expv * rinv2);
      g += gc;
      acc.uc = mad(Cqq * erfcv, rinv, acc.uc);
      acc.wc = mad(gc, r2, acc.wc);
    }
  }
  acc.fx = mad(g, dx, acc.fx);
  acc.fy = mad(g, dy, acc.fy);
  acc.fz = mad(g, dz, acc.fz);
}

// Branch-light evaluation for the cell-list kernel: `act` says whether this lane holds a
// candidate pair at all (idle lanes compute a masked dummy). The cutoff decision is exact:
// FP32 outside the +-1e-5 band around r_c^2, the oracle's FP64 expression inside it (a
// rare, divergent branch). A zero displacement (the particle itself; r^2 = 0 exactly when the
// integer displacement is 0) is never a pair. Rejected and idle lanes evaluate with 1/r^2 = 0,
// which makes every LJ term an exact zero, so no early return diverges the warp.
template <bool LJ, bool COUL, bool MULTI, bool CUBIC>
__device__ __forceinline__ void pair_eval_masked(const PairArgs &a, const LJTable *tab,
                                                 bool act, int dsx, int dsy, int dsz, float qi,
                                                 int ti, float qj, int tj,
                                                 PairAcc<float> &acc) {
  const PairConst &pc = a.pc;
  const float dx = (float)dsx * pc.h[0], dy = (float)dsy * pc.h[1], dz = (float)dsz * pc.h[2];
  const float r2 = mad(dx, dx, mad(dy, dy, dz * dz));
  bool inside = act && r2 < pc.rc2_lo && r2 > 0.f;
  const bool band = act && r2 >= pc.rc2_lo && r2 <= pc.rc2_hi;
  if (band) inside = exact_r2(pc, dsx, dsy, dsz) <= pc.rc2d;
  acc.nbr += inside ? 1 : 0;
  // off the pair: 1/r^2 = 0 exactly (the fast quotient is documented to return 0 for divisors
  // between 2^126 and 2^128)
  const float r2s = inside ? r2 : 1e38f;
  float g = 0.f;
  if (LJ) {
    const float ir2 = __fdividef(1.0f, r2s);  // fast reciprocal (2 ulp)
    float gl, u, w;
    lj_terms<float, MULTI>(a, tab, ti, tj, ir2, gl, u, w);
    g += gl;
    acc.ulj += u;
    acc.wlj += w;
  }
  if (COUL) {
    const float qq = qi * qj;
    if (inside && qq != 0.f) {
      const float rinv = rsqrtf(r2);  // 1/r and r from one reciprocal square root
      const float r = r2 * rinv;
      const float erfcv = erfcf(pc.sqrt_alpha * r);
      const float expv = expf(-pc.alpha * r2);
      const float Cqq = pc.C * qq;
      const float rinv2 = rinv * rinv;
      const float gc = Cqq * mad(erfcv * rinv, rinv2, pc.two_sqrt_alpha_over_sqrt_pi * expv * rinv2);
      g += gc;
      if (a.comp) {
        kahan_add(acc.uc, acc.cuc, Cqq * erfcv * rinv);
        kahan_add(acc.wc, acc.cwc, gc * r2);
      } else {
        acc.uc = mad(Cqq * erfcv, rinv, acc.uc);
        acc.wc = mad(gc, r2, acc.wc);
      }
    }
  }
  acc.fx = mad(g, dx, acc.fx);
  acc.fy = mad(g, dy, acc.fy);
  acc.fz = mad(g, dz, acc.fz);
}

// The FP64 form's evaluation. FP64 runs at 1/64 of the FP32 rate, so its operations are what it
// costs: 19 a pair in a cubic box (21 otherwise), where scaled displacements, a division, FP64
// cutoff tests and conversions took about 40 (65,536 particles, 10% charged: 2,888 -> 1,692 us
// with the ring and split of k_pair.cu). The cutoff is decided in FP32 from the exact displacement,
// in the +-1e-5 band by the oracle's FP64 expression. r^2 and the force sums stay in grid units
// of x (the integer displacement converts exactly; the caller scales the sums by fs). 1/r^2 is
// an FP32 reciprocal refined by one third-order Householder step, y (1 + e + e^2) with
// e = 1 - r^2 y (|e| < 2^-21: the error left is below 2^-62), the Coulomb 1/r likewise,
// y (1 + e/2 + 3 e^2 / 8). acc.ulj and acc.wlj hold sum r^-12 and sum r^-6 in grid units for one
// LJ type, U and W for several.
// (CUBIC: the three edges are equal. A kernel of its own: as a branch its other side's FP64
// instructions were issued with a false predicate and still took the pipe.)
template <bool LJ, bool COUL, bool MULTI, bool CUBIC>
__device__ __forceinline__ void pair_eval_masked(const PairArgs &a, const LJTable *tab,
                                                 bool act, int dsx, int dsy, int dsz, double qi,
                                                 int ti, double qj, int tj,
                                                 PairAcc<double> &acc) {
  const PairConst &pc = a.pc;
  const float ex = (float)dsx * a.gh[0], ey = (float)dsy * a.gh[1], ez = (float)dsz * a.gh[2];
  const float Rf = fmaf(ex, ex, fmaf(ey, ey, ez * ez));
  bool inside = act && Rf < a.glo && Rf > 0.f;
  if (act && Rf >= a.glo && Rf <= a.ghi) inside = exact_r2(pc, dsx, dsy, dsz) <= pc.rc2d;
  acc.nbr += inside ? 1 : 0;
  const double Dx = i2d(dsx), Dy = i2d(dsy), Dz = i2d(dsz);
  const double R = CUBIC ? fma(Dz, Dz, fma(Dy, Dy, Dx * Dx))
                         : fma(Dz * Dz, a.rz, fma(Dy * Dy, a.ry, Dx * Dx));
  // (off the pair y = 0: every term below is an exact zero)
  const double y = f2d(inside ? rcp_approx(Rf) : 0.f);
  const double e = fma(-R, y, 1.0);
  const double iR = fma(y, fma(e, e, e), y);
  double w = 0.0;
  if (LJ) {
    const double i6 = iR * iR * iR;
    if (MULTI) {
      const int pt = ti * tab->nt + tj;
      const double ir6 = i6 * a.ih6;
      w = ir6 * fma(tab->A12d[pt], ir6, -tab->B6d[pt]);
      acc.ulj = fma(ir6, fma(tab->Ad[pt], ir6, -tab->Bd[pt]), acc.ulj);
      acc.wlj += w;
    } else {
      w = i6 * fma(a.A12s, i6, -a.B6s);
      acc.ulj = fma(i6, i6, acc.ulj);
      acc.wlj += i6;
    }
  }
  if (COUL) {
    const double qq = qi * qj;
    if (inside && qq != 0.0) {
      const double z = f2d(rsqrtf(Rf)), ez_ = fma(-(R * z), z, 1.0);
      const double zr = fma(z, ez_ * fma(ez_, 0.375, 0.5), z);  // 1 / r in grid units
      const double r = R * zr * a.hx;
      const double erfcv = erfc(pc.sqrt_alpha_d * r), expv = exp(-pc.alpha_d * (r * r));
      const double Cqq = pc.C_d * qq, u = Cqq * erfcv * (zr * a.ihx);
      const double wc = fma(Cqq * pc.two_sqrt_alpha_over_sqrt_pi_d, expv, u);
      acc.uc += u;
      acc.wc += wc;
      w += wc;
    }
  }
  const double g = w * iR;
  acc.fx = fma(g, Dx, acc.fx);
  acc.fy = fma(g, Dy, acc.fy);
  acc.fz = fma(g, Dz, acc.fz);
}

// What the FP64 evaluation needs beside PairArgs' other fields. The powers of h_x are formed as
// unevaluated sums of two doubles and divided out with one correction, so that each constant is
// its true value rounded about once: an error here would be in every pair, sevenfold in the force.
inline void set_grid_units(const Ctx &c, PairArgs &a) {
  const double hx = c.pc.hd[0];
  struct DD { double h, l; };
  auto mul = [](DD x, DD y) {
    const double p = x.h * y.h;
    return DD{p, std::fma(x.h, y.h, -p) + (x.h * y.l + x.l * y.h)};
  };
  auto div = [](double v, DD y) {
    const double q = v / y.h;
    return q + (std::fma(-q, y.h, v) - q * y.l) / y.h;
  };
  const DD p1{hx, 0.0}, p2 = mul(p1, p1), p6 = mul(mul(p2, p2), p2), p12 = mul(p6, p6);
  a.ry = (c.pc.hd[1] / hx) * (c.pc.hd[1] / hx);
  a.rz = (c.pc.hd[2] / hx) * (c.pc.hd[2] / hx);
  for (int d = 0; d < 3; ++d) a.fs[d] = div(c.pc.hd[d], p2);
  for (int d = 0; d < 3; ++d) a.gh[d] = (float)(c.pc.hd[d] / hx);
  a.glo = (float)(c.pc.rc2d / (hx * hx) * (1.0 - 1e-5));
  a.ghi = (float)(c.pc.rc2d / (hx * hx) * (1.0 + 1e-5));
  a.hx = hx;
  a.ihx = 1.0 / hx;
  a.ih6 = div(1.0, p6);
  a.A12s = div(c.lj.A12d[0], p12);
  a.B6s = div(c.lj.B6d[0], p6);
  a.cubic = c.pc.hd[0] == c.pc.hd[1] && c.pc.hd[1] == c.pc.hd[2];
}
// U and W of one LJ type from the FP64 sums in grid units.
__device__ __forceinline__ void grid_energies(const PairArgs &a, double s12, double s6, double &u,
                                              double &w) {
  const double p = a.A12s * s12, q = a.B6s * s6;
  u = p / 12.0 - q / 6.0;
  w = p - q;
}

}  // namespace rbe
