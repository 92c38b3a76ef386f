// k_coul.cu -- real-space Coulomb forces among the charged particles (Eqs. F_i, G_short):
//
//   F_i += sum_{j charged, j != i, r_ij <= r_c} C q_i q_j G(r) (r_i - r_j),
//   G(r) = erfc(sqrt(alpha) r) / r^3 + 2 sqrt(alpha / pi) exp(-alpha r^2) / r^2,
//
// the pass that follows the LJ pass when a minority of the particles carries charge. The
// charged subset is dilute (about one particle per cell of r_c / 2 at 10% charged), so a
// thread per particle would spend most of its time testing candidates its neighbours in the
// warp need and it does not. Here a warp serves one charged particle i:
//  1. Stencil: one lane per row (dy, dz) of cells finds the x-cells of the row within r_c of
//     i (a row farther than r_c is skipped), as at most two runs of the subset's
//     cell-ordered particles; a warp scan flattens the runs into one candidate list.
//  2. Test: 32 candidates at a time, one per lane, from their packed (s, q) records: the
//     exact minimum-image integer displacement, the cutoff decided in FP32 outside a band
//     around r_c^2 and by the oracle's FP64 expression inside it (in the FP64 form too: the
//     band covers FP32's rounding of the exact integer displacement). Hits are compacted
//     (ballot) into a small per-warp buffer in shared memory.
//  3. Evaluate: whenever 32 hits are buffered (and once at the end) every lane evaluates one
//     of them (erfc, exp and a reciprocal square root), so the expensive terms run on full
//     warps. A warp sum gives F_i, added to the force of i's slot in the full set: to F after
//     a pass that wrote F, or to the cluster kernel's 64-bit fixed-point sums (three integer
//     atomics per particle, whose sums do not depend on their order).
// Each pair is evaluated from both sides, so the forces are reproducible run to run; the
// energy and virial partials take half of the per-i sums.
#include <climits>
#include <cmath>

#include "pair_common.cuh"

namespace rbe {

constexpr int kCoulWarps = 4;     // warps (charged particles) per block
constexpr int kCoulBuf = 64;      // buffered hits per warp (at most 31 pending + 32 new)
constexpr int kCoulMaxRows = 49;  // (2R+1)^2 stencil rows for R <= 3

struct CoulArgs {
  const uint4 *s4;            // charged subset, sorted: (s_x, s_y, s_z, q bits)
  const double *qd;           // FP64 charges of the subset (FP64 form)
  const int32_t *cell_start;  // the subset's cell starts (ncell + 1)
  const int32_t *map;         // subset slot -> slot of the full sorted set
  int64_t nq;
  Grid grid;
  PairConst pc;
  float *F;
  double *Fd;
  int64_t Fstride;
  double *epart;              // per-block partials (NQ_PAIR doubles)
  int comp;                   // Kahan-compensated energy and virial sums
  float reach2;               // r_c^2 widened: rows and cells farther than this are skipped
  long long *facc;            // nullable: 3 x N fixed-point force sums of the full set (then
  float fscale;               //   F is not written), their scale (FP32 forms)
  double fscale_d;            //   (FP64 form)
  int *err;                   //   (a sum out of range sets ERRBIT_NONFINITE)
  ErfcFit fit;
};

int64_t coul_blocks(int64_t nq) { return (nq + kCoulWarps - 1) / kCoulWarps; }

template <typename real>
__device__ __forceinline__ void coul_body(const CoulArgs a, int bx, int) {
  constexpr bool F64 = sizeof(real) == 8;
  constexpr unsigned FULL = 0xffffffffu;
  // hits: displacement and charge (FP32 forms), or integer displacement and index
  __shared__ int4 buf[kCoulWarps][kCoulBuf];
  __shared__ int32_t seg_off[kCoulWarps][2 * kCoulMaxRows];
  __shared__ int32_t seg_pre[kCoulWarps][2 * kCoulMaxRows];
  __shared__ double wred[kCoulWarps][2];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const PairConst &pc = a.pc;
  const int64_t i = (int64_t)bx * kCoulWarps + wid;
  real fx = (real)0, fy = (real)0, fz = (real)0;
  real uc = (real)0, wc = (real)0, cuc = (real)0, cwc = (real)0;
  if (i < a.nq) {
    const uint4 pi = a.s4[i];
    const real qi = F64 ? (real)a.qd[i] : (real)__uint_as_float(pi.w);
    const int n0 = a.grid.n[0], n1 = a.grid.n[1], n2 = a.grid.n[2];
    const int R1 = a.grid.R[1], R2 = a.grid.R[2];
    const int cy = cell_of(pi.y, n1), cz = cell_of(pi.z, n2);
    const int ny = 2 * R1 + 1, nrows = ny * (2 * R2 + 1);
    // t / ny as (t m) >> 8, m = ceil(256 / ny): exact for t < 64 and ny in {1, 3, 5, 7}
    const int mny = (256 + ny - 1) / ny;
    // i's y and z in cell units, and the cell widths
    const float fyc = (float)pi.y * ((float)n1 * 2.3283064365386963e-10f);
    const float fzc = (float)pi.z * ((float)n2 * 2.3283064365386963e-10f);
    const float wy = pc.h[1] * (4294967296.0f / (float)n1), wz = pc.h[2] * (4294967296.0f / (float)n2);
    int carry = 0, nseg = 0;
    for (int rb = 0; rb < nrows; rb += 32) {
      const int t = rb + lane;
      int b0 = 0, l0 = 0, b1 = 0, l1 = 0;
      if (t < nrows) {
        const int tq = (t * mny) >> 8;
        const int dz = tq - R2, dy = t - tq * ny - R1;
        // distance of i from the row's cells in y and z, in cell widths (i's position in cell
        // units is within about 1e-5 cells in FP32; the distance is shrunk by 1e-3 cells)
        const float ey = fmaxf(0.f, fmaxf((float)(cy + dy) - fyc, fyc - (float)(cy + dy + 1)) - 1e-3f);
        const float ez = fmaxf(0.f, fmaxf((float)(cz + dz) - fzc, fzc - (float)(cz + dz + 1)) - 1e-3f);
        const float dyl = ey * wy, dzl = ez * wz;
        const float rx2 = mad(-dzl, dzl, mad(-dyl, dyl, a.reach2));
        if (rx2 > 0.f) {
          // periodic row indices (|dy| <= R1 < n1, |dz| <= R2 < n2)
          int ryw = cy + dy, rzw = cz + dz;
          ryw += ryw < 0 ? n1 : 0;
          ryw -= ryw >= n1 ? n1 : 0;
          rzw += rzw < 0 ? n2 : 0;
          rzw -= rzw >= n2 ? n2 : 0;
          const int64_t rowbase = (int64_t)n0 * (ryw + (int64_t)n1 * rzw);
          // x-cells within reach: one run, or two where the reach passes an end of the box
          const uint32_t reach = (uint32_t)(sqrtf(rx2) * (1.0f + 1e-5f) / pc.h[0]) + 4u;
          const uint32_t xl = pi.x - reach, xr = pi.x + reach;
          const bool wl = xl > pi.x, wr = xr < pi.x;
          int sa0 = cell_of(xl, n0), sb0 = cell_of(xr, n0), sb1 = -1;
          if (wl || wr) {
            if ((wl && wr) || sb0 + 1 >= sa0) sa0 = 0;  // (the whole row)
            else sb1 = sb0;                             // and from the row's start
            sb0 = n0 - 1;
          }
          b0 = a.cell_start[rowbase + sa0];
          l0 = a.cell_start[rowbase + sb0 + 1] - b0;
          if (sb1 >= 0) {
            b1 = a.cell_start[rowbase];
            l1 = a.cell_start[rowbase + sb1 + 1] - b1;
          }
        }
      }
      const int tot = l0 + l1;
      int incl = tot;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(FULL, incl, o);
        if (lane >= o) incl += v;
      }
      // the runs that hold candidates, in order: offset in the list, and first particle minus it
      const int excl = carry + incl - tot;
      const unsigned m0 = __ballot_sync(FULL, l0 > 0), m1 = __ballot_sync(FULL, l1 > 0);
      const unsigned below = (1u << lane) - 1u;
      int k = nseg + __popc(m0 & below) + __popc(m1 & below);
      if (l0 > 0) {
        seg_pre[wid][k] = excl;
        seg_off[wid][k++] = b0 - excl;
      }
      if (l1 > 0) {
        seg_pre[wid][k] = excl + l0;
        seg_off[wid][k] = b1 - excl - l0;
      }
      nseg += __popc(m0) + __popc(m1);
      carry += __shfl_sync(FULL, incl, 31);
    }
    __syncwarp();
    const int T = carry;
    // Buffered hits [0, n), one per lane, in the FP32 forms.
    auto evaluate32 = [&](int n) {
      if (lane >= n) return;
      const int4 e = buf[wid][lane];
      const float dx = __int_as_float(e.x), dy = __int_as_float(e.y), dz = __int_as_float(e.z);
      const float r2 = mad(dx, dx, mad(dy, dy, dz * dz)), rinv = rsqrtf(r2), r = r2 * rinv;
      float er, ex;
      if (a.fit.ok) {
        erfc_exp1(a.fit, r, r2, er, ex);
      } else {
        er = erfcf(pc.sqrt_alpha * r);
        ex = expf(-pc.alpha * r2);
      }
      const float Cqq = pc.C * (float)qi * __int_as_float(e.w), rinv2 = rinv * rinv;
      const float gc = Cqq * mad(er * rinv, rinv2, pc.two_sqrt_alpha_over_sqrt_pi * ex * rinv2);
      fx = mad((real)gc, (real)dx, fx); fy = mad((real)gc, (real)dy, fy); fz = mad((real)gc, (real)dz, fz);
      if (a.comp) {
        kahan_add(uc, cuc, (real)(Cqq * er * rinv));
        kahan_add(wc, cwc, (real)(gc * r2));
      } else {
        uc = mad((real)(Cqq * er), (real)rinv, uc);
        wc = mad((real)gc, (real)r2, wc);
      }
    };
    // FP64 form: one per lane.
    auto evaluate64 = [&](int n) {
      if (lane < n) {
        const int4 e = buf[wid][lane];
        const double dx = i2d(e.x) * pc.hd[0], dy = i2d(e.y) * pc.hd[1], dz = i2d(e.z) * pc.hd[2];
        const double r2 = mad(dx, dx, mad(dy, dy, dz * dz));
        // 1/r from an FP32 start by one third-order Householder step (as in the pair kernel)
        const float ex = (float)e.x * pc.h[0], ey = (float)e.y * pc.h[1], ez = (float)e.z * pc.h[2];
        const double z = f2d(rsqrtf(fmaf(ex, ex, fmaf(ey, ey, ez * ez))));
        const double c = fma(-(r2 * z), z, 1.0);
        const double rinv = fma(z, c * fma(c, 0.375, 0.5), z), r = r2 * rinv;
        const double erfcv = erfc(pc.sqrt_alpha_d * r), expv = exp(-pc.alpha_d * r2);
        const double Cqq = pc.C_d * (double)qi * a.qd[e.w], rinv2 = rinv * rinv;
        const double gc =
            Cqq * mad(erfcv * rinv, rinv2, pc.two_sqrt_alpha_over_sqrt_pi_d * expv * rinv2);
        fx = mad((real)gc, (real)dx, fx); fy = mad((real)gc, (real)dy, fy); fz = mad((real)gc, (real)dz, fz);
        uc = mad((real)(Cqq * erfcv), (real)rinv, uc);
        wc = mad((real)gc, (real)r2, wc);
      }
    };
    auto evaluate = [&](int n) {
      if constexpr (F64) evaluate64(n); else evaluate32(n);
    };
    int nb = 0;      // buffered hits (warp-uniform)
    int before = 0;  // runs that start before the 32 candidates
    for (int base = 0; base < T; base += 32) {
      const int cc = base + lane;
      bool hit = false;
      int4 rec = make_int4(0, 0, 0, 0);
      // a bit for each run that starts among these candidates; cc's run is the last one at or
      // before it
      unsigned starts = 0u;
      for (int k = lane; k < nseg; k += 32) {
        const unsigned d = (unsigned)(seg_pre[wid][k] - base);
        starts |= d < 32u ? 1u << d : 0u;
      }
      starts = __reduce_or_sync(FULL, starts);
      const int run = before + __popc(starts & (0xffffffffu >> (31 - lane))) - 1;
      before += __popc(starts);
      if (cc < T) {
        const int64_t j = cc + seg_off[wid][run];
        if (j != i) {
          const uint4 pj = a.s4[j];
          const int dsx = (int)(pi.x - pj.x), dsy = (int)(pi.y - pj.y), dsz = (int)(pi.z - pj.z);
          const float ex = (float)dsx * pc.h[0], ey = (float)dsy * pc.h[1],
                      ez = (float)dsz * pc.h[2];
          const float r2 = mad(ex, ex, mad(ey, ey, ez * ez));
          hit = r2 < pc.rc2_lo;
          if (r2 >= pc.rc2_lo && r2 <= pc.rc2_hi) hit = exact_r2(pc, dsx, dsy, dsz) <= pc.rc2d;
          rec = F64 ? make_int4(dsx, dsy, dsz, (int)j)
                    : make_int4(__float_as_int(ex), __float_as_int(ey), __float_as_int(ez), (int)pj.w);
        }
      }
      const unsigned hm = __ballot_sync(FULL, hit);
      if (hit) buf[wid][nb + __popc(hm & ((1u << lane) - 1u))] = rec;
      nb += __popc(hm);
      __syncwarp();
      if (nb >= 32) {
        evaluate(32);
        const int4 keep = lane + 32 < nb ? buf[wid][lane + 32] : make_int4(0, 0, 0, 0);
        __syncwarp();
        if (lane + 32 < nb) buf[wid][lane] = keep;
        nb -= 32;
        __syncwarp();
      }
    }
    evaluate(nb);
    fx = warp_sum(fx); fy = warp_sum(fy); fz = warp_sum(fz);
    if (a.facc) {  // one component per lane (every lane holds the sums)
      if (lane < 3) {
        const real sc = F64 ? (real)a.fscale_d : (real)a.fscale;
        fx_add_i32(a.facc + lane * a.Fstride + a.map[i], lane == 0 ? fx : (lane == 1 ? fy : fz),
                   sc, a.err);
      }
    } else if (lane == 0) {
      const int64_t o = a.map[i];
      const int64_t S = a.Fstride;
      if (F64) {
        a.Fd[o] += (double)fx; a.Fd[S + o] += (double)fy; a.Fd[2 * S + o] += (double)fz;
      } else {
        a.F[o] += (float)fx; a.F[S + o] += (float)fy; a.F[2 * S + o] += (float)fz;
      }
    }
  }
  // block partials of the Coulomb energy and virial (halves of the per-i sums)
  const double us = F64 ? (double)uc : f2d((float)uc) - f2d((float)cuc);
  const double ws = F64 ? (double)wc : f2d((float)wc) - f2d((float)cwc);
  const double uw = warp_sum2(us, ws, lane);
  if (lane < 2) wred[wid][lane] = uw;
  __syncthreads();
  if (threadIdx.x < NQ_PAIR) {
    double s = 0.0;
    if (threadIdx.x == Q_UREAL || threadIdx.x == Q_WREAL)
      for (int k = 0; k < kCoulWarps; ++k) s += wred[k][threadIdx.x == Q_UREAL ? 0 : 1];
    a.epart[(int64_t)bx * NQ_PAIR + threadIdx.x] = 0.5 * s;
  }
}

// (12 blocks of 4 warps in the FP32 forms, 40 registers without spills; 16 run as fast with spills,
// 10 slower: the pass is bound by issue and by the latency of each warp's dependent loads. Two hits
// a lane as a packed pair took 48 registers and 154 us where one takes 121. 104,858 charged of
// 2^20: 135 us with a binary search for a candidate's run and erfcf and expf, 122 so; 400,000 of
// 4,000,001: 481 -> 433. 8 in the
// FP64 form, whose registers would spill.)
template <typename real>
__global__ void __launch_bounds__(kCoulWarps * 32, sizeof(real) == 8 ? 8 : 12)
    coul_kernel(const CoulArgs a) {
  coul_body<real>(a, (int)blockIdx.x, (int)gridDim.x);
}


cudaError_t launch_coulomb_subset(Ctx &c, const uint4 *s4, bool into_facc) {
  CoulArgs a;
  a.s4 = s4;
  a.qd = c.cqd;
  a.cell_start = c.ccell_start;
  a.map = c.cmap;
  a.nq = c.Nq;
  a.grid = c.grid;
  a.pc = c.pc;  // the default +-1e-5 band covers an r^2 from exact integer displacements
  a.F = c.F; a.Fd = c.Fd; a.Fstride = c.N;
  a.epart = c.epart + c.off_coul;
  a.comp = c.precision == RBE_FP32_COMP;
  const double rr = c.rc * (1.0 + 1e-5) + 8.0 * std::ldexp(1.0, -24) * std::max(c.box[0], std::max(c.box[1], c.box[2]));
  a.reach2 = (float)(rr * rr);
  a.facc = into_facc ? c.facc : nullptr;
  a.fscale = (float)kFixScale32;
  a.fscale_d = kFixScale64;
  a.err = c.err;
  a.fit = c.fit;
  const dim3 g((unsigned)c.n_coul_blk), b(kCoulWarps * 32);  // every slot of the partial range
  // (per replica in a batch, like the other pair kernels)
  if (c.precision == RBE_FP64)
    return dispatch(c, coul_kernel<double>, nullptr, g, b, 0, a, true);
  return dispatch(c, coul_kernel<float>, nullptr, g, b, 0, a, true);
}

}  // namespace rbe
