// k_cpair.cu -- real-space pair forces over clusters of particles, each pair evaluated once
// (Newton's third law), for the cell-list real space (Eqs. F_i, G_short, LJ):
//
//   F_i += sum_{j != i, r_ij <= r_c} (C q_i q_j G(r) + G_LJ(r)) (r_i - r_j),   F_j -= the same.
//
// Clusters. Particles are sorted by (cell, s_x, id) with cells of r_c / sub, so each row of
// cells (c_y, c_z) holds its particles in ascending s_x. A cluster is 8 consecutive
// particles of a row (the last cluster of a row may hold fewer) and a super-cluster is up
// to NC consecutive clusters of a row: one warp's work. Global cluster indices run over the
// rows in order (cl_base per row), and so do the super-clusters (sc_base per row).
//
// Half list. The cluster pair (I, J) is evaluated once, by the super-cluster that holds I,
// when I <= J (global index) and the bounding boxes of I and J are within r_c of each
// other. Every particle pair within r_c lies in one such pair of clusters, or inside one
// cluster (I = J: then only particle a with particle b > a of the cluster).
//
// Lanes. Lane (h, a) = (lane / 8, lane % 8) holds the forces on particle a of every i-cluster
// of the super-cluster (its coordinates come from shared memory) and particles h and h + 4 of
// the j-cluster being visited, so one visit evaluates the 8 x 8 pairs of every i-cluster the
// visit's mask names, two per lane: in the FP32 forms as one packed pair. The reaction on j is
// summed over the 8 lanes that share h by shuffles, once per visit, and added to j's force.
//
// Forces are summed in 64-bit fixed point by integer atomics. Integer sums do not depend on
// their order, so the forces are the same run to run; a final pass converts them to
// floating point. Energies and virials are per-block partial sums, as in the other kernels.
//
// Frame. A super-cluster's coordinates are the exact integer offsets of its particles from
// the centre of its bounding box, converted to FP32 (kept as integers in the FP64 form). A
// visited j particle's x is converted the same way; its y and z are the frame coordinates of
// its cluster's box corner plus its FP32 offsets from that corner, stored per step in the
// cluster's eight record slots (a cluster lies in one cell in y and z, so the offsets are
// small and never wrap; a cluster across the frame's edge counts from the side in reach; the
// one extra rounding widens the band below).
// The difference of two offsets is the minimum-image displacement of a pair within r_c as
// long as the super-cluster's extent plus 2 r_c stays below L on every axis: the host
// checks y and z (a cell width), the kernel splits a super-cluster whose x extent is
// larger into groups of clusters that fit, down to single particles. The cutoff decision is exact: FP32 outside a
// band around r_c^2 that covers the rounding of the frame coordinates, and the oracle's
// FP64 expression of the integer displacement inside it (a rare branch per visit whose
// pairs are added by atomics); the FP64 form always takes the FP64 expression.
#include <climits>
#include <cmath>

#include "f32x2.cuh"
#include "pair_common.cuh"

namespace rbe {

constexpr int kClSize = 8;              // particles per cluster
constexpr int kCpMaxRows = 49;          // (2R+1)^2 stencil rows for R <= 3
constexpr int kCpMaxSeg = 2 * kCpMaxRows;
constexpr int kCpMaxWarps = 4;          // FP32 forms: warps a block,
constexpr int kCpWarpsLJ = 28, kCpWarpsCoul = 20;  // and resident warps an SM

struct ClusterArgs {
  PairSet set;                 // full sorted set
  Grid grid;
  PairConst pc;
  float ljA12, ljB6;
  double ljAd, ljBd, ljA12d, ljB6d;
  const LJTable *table;        // device copy, multi-type only
  const int32_t *cl_base;      // nrows + 1: first global cluster of each row
  const int32_t *sc_base;      // nrows + 1: first super-cluster of each row
  const int4 *sc_info;         // per super-cluster: row, first cluster and particle, counts
  const uint4 *cl_lo, *cl_hi;  // per cluster: (min s_x, s_y, s_z, first particle), (max..., count)
  const uint4 *jrec;           // FP32 forms: 8 slots per cluster (s_x, y and z offsets from the
                               // box corner as FP32 bits, q bits); empty slots y = -3e18
  int nrows;
  long long *facc;             // 3 x N fixed-point forces (x block, y, z)
  int64_t N;
  float fscale;                // fixed-point scale (FP32 forms)
  double fscale_d;             // (FP64 form)
  double *epart;               // per-block partials (NQ_PAIR doubles)
  int32_t *nbr;                // neighbour counts (sorted order, zeroed before), nullable
  int comp;                    // Kahan sums for the Coulomb energy and virial
  uint32_t xlim;               // largest x extent of a cluster group the frame allows
  float bb2;                   // bounding-box test: squared gap <= bb2 (r_c^2, widened)
  float rc2_mid, rc2_half;     // band test: |r^2 - rc2_mid| <= rc2_half covers [rc2_lo, rc2_hi]
  int *err;
  int64_t nslots;              // the pass's energy partial slots (at least the grid)
  int nsplit;                  // FP32 forms: blocks a super-cluster
  int64_t wfix[2];             // 2^48 / cells in y and z (rounded down): a cell's width
  ErfcFit fit;                 // FP32 forms
};

// ---------------------------------------------------------------------------------------
// Per-step cluster tables

struct RowsArgs {
  const int32_t *cell_start;
  int n0, nrows, nc_sc;
  int32_t *cl_base, *sc_base;
};
struct BoundsArgs {
  const uint32_t *sx, *sy, *sz;
  const float *qf;
  const int32_t *cell_start;
  int n0, nrows;
  const int32_t *cl_base;
  int64_t cap;
  uint4 *lo, *hi;
  uint4 *jrec;                 // nullable (FP64 form)
  float hy, hz;                // length of one fractional unit in y and z
  const int32_t *sc_base;
  int nc_sc;
  int4 *sc_info;               // (row, first cluster, first particle, clusters | particles << 8)
};
struct FinishArgs {
  long long *facc;
  void *F;                 // float or double forces, by the kernel's type
  int64_t n3;
  float sh, sl;
  double inv_scale;
  int per;                 // sums a block (a multiple of 512, at most 512 kFinishPairs)
};

// One block: clusters and super-clusters of every row, as exclusive prefix sums.
__device__ __forceinline__ void cluster_rows_body(const RowsArgs &a, int, int) {
  __shared__ int2 ws[32];
  const int32_t *__restrict__ cell_start = a.cell_start;
  const int n0 = a.n0, nrows = a.nrows, nc_sc = a.nc_sc;
  int32_t *__restrict__ cl_base = a.cl_base;
  int32_t *__restrict__ sc_base = a.sc_base;
  const unsigned FULL = 0xffffffffu;
  const int t = threadIdx.x, ln = t & 31;
  const int per = (nrows + 1023) / 1024;
  const int r0 = min(nrows, t * per), r1 = min(nrows, r0 + per);
  int cl = 0, sc = 0;
  for (int r = r0; r < r1; ++r) {
    const int n = cell_start[(int64_t)(r + 1) * n0] - cell_start[(int64_t)r * n0];
    const int k = (n + kClSize - 1) / kClSize;
    cl += k;
    sc += (k + nc_sc - 1) / nc_sc;
  }
  int icl = cl, isc = sc;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int u = __shfl_up_sync(FULL, icl, o), v = __shfl_up_sync(FULL, isc, o);
    if (ln >= o) { icl += u; isc += v; }
  }
  if (ln == 31) ws[t >> 5] = make_int2(icl, isc);
  __syncthreads();
  if (t < 32) {
    const int2 v = ws[t];
    int u = v.x, w = v.y;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int p = __shfl_up_sync(FULL, u, o), q = __shfl_up_sync(FULL, w, o);
      if (ln >= o) { u += p; w += q; }
    }
    ws[t] = make_int2(u - v.x, w - v.y);
  }
  __syncthreads();
  int bc = ws[t >> 5].x + icl - cl, bs = ws[t >> 5].y + isc - sc;
  for (int r = r0; r < r1; ++r) {
    const int n = cell_start[(int64_t)(r + 1) * n0] - cell_start[(int64_t)r * n0];
    const int k = (n + kClSize - 1) / kClSize;
    cl_base[r] = bc;
    sc_base[r] = bs;
    bc += k;
    bs += (k + nc_sc - 1) / nc_sc;
  }
  if (t == 1023) {
    cl_base[nrows] = bc;
    sc_base[nrows] = bs;
  }
}
RBE_BATCHED_KERNEL(__launch_bounds__(1024), cluster_rows_kernel, RowsArgs, cluster_rows_body)

// Largest r in [0, nrows) with base[r] <= g (base is non-decreasing; g < base[nrows]).
__device__ __forceinline__ int row_of(const int32_t *__restrict__ base, int nrows, int g) {
  int lo = 0, hi = nrows - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (base[mid] <= g) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}

// Bounding box (integer fractional coordinates), first particle and count of every cluster,
// and its j records: slot k holds particle k's s_x, its y and z offsets from the box's low
// corner in length units (FP32 bits) and its charge bits; a slot past the cluster's count
// holds y = -3e18, beyond the reach of any i particle. Eight threads per cluster, one per
// slot, with the box reduced over the eight by shuffles.
static_assert(kClSize == 8, "eight threads per cluster");
__device__ __forceinline__ void cluster_bounds_body(const BoundsArgs &a, int bx, int) {
  const int32_t *__restrict__ cell_start = a.cell_start;
  const int32_t *__restrict__ cl_base = a.cl_base;
  const int n0 = a.n0, nrows = a.nrows;
  const int64_t t = (int64_t)bx * blockDim.x + threadIdx.x;
  const int64_t g = t >> 3;
  const int k = (int)(t & 7);
  // (the same for the eight threads of a cluster, which exit together)
  if (g >= a.cap || g >= cl_base[nrows]) return;
  const unsigned gm = 0xffu << (threadIdx.x & 24);
  const int r = row_of(cl_base, nrows, (int)g);
  const int ps = cell_start[(int64_t)r * n0], pe = cell_start[(int64_t)(r + 1) * n0];
  const int b = ps + (int)(g - cl_base[r]) * kClSize;
  const int n = min(kClSize, pe - b);
  const bool v = k < n;
  uint32_t x = 0u, y = 0u, z = 0u;
  float q = 0.f;
  if (v) {
    x = a.sx[b + k]; y = a.sy[b + k]; z = a.sz[b + k];
    q = a.qf[b + k];
  }
  uint32_t x0 = v ? x : 0xffffffffu, y0 = v ? y : 0xffffffffu, z0 = v ? z : 0xffffffffu;
  uint32_t x1 = x, y1 = y, z1 = z;
#pragma unroll
  for (int o = 1; o < 8; o <<= 1) {
    x0 = min(x0, __shfl_xor_sync(gm, x0, o)); x1 = max(x1, __shfl_xor_sync(gm, x1, o));
    y0 = min(y0, __shfl_xor_sync(gm, y0, o)); y1 = max(y1, __shfl_xor_sync(gm, y1, o));
    z0 = min(z0, __shfl_xor_sync(gm, z0, o)); z1 = max(z1, __shfl_xor_sync(gm, z1, o));
  }
  if (k == 0) {
    a.lo[g] = make_uint4(x0, y0, z0, (uint32_t)b);
    a.hi[g] = make_uint4(x1, y1, z1, (uint32_t)n);
    const int kc = (int)(g - cl_base[r]);  // the row's cluster; each super-cluster's first one
    if (kc % a.nc_sc == 0) {               // writes its record
      const int ncl = min(a.nc_sc, cl_base[r + 1] - (int)g), npt = min(a.nc_sc * kClSize, pe - b);
      a.sc_info[a.sc_base[r] + kc / a.nc_sc] = make_int4(r, (int)g, b, ncl | (npt << 8));
    }
  }
  if (a.jrec)
    a.jrec[t] = v ? make_uint4(x, __float_as_uint((float)(int)(y - y0) * a.hy),
                               __float_as_uint((float)(int)(z - z0) * a.hz), __float_as_uint(q))
                  : make_uint4(0u, __float_as_uint(-3e18f), 0u, 0u);
}
RBE_BATCHED_KERNEL(__launch_bounds__(256), cluster_bounds_kernel, BoundsArgs, cluster_bounds_body)

// F = fixed-point sums / scale (overwriting), and the sums cleared for the next pass. The
// 64-bit sum converts as its two 32-bit halves (a 64-bit integer conversion is slow here):
// v = hi 2^32 + lo with hi signed and lo unsigned; FP32 forms take the FP32 factors
// sh = 2^32 / scale and sl = 1 / scale (no FP64 work per element), the FP64 form the FP64 ones.
// The pass waits on the latency of loads from sums that atomics have just written, so a thread has up
// to eight 16-byte loads in flight: 12,000,003 sums, 512 / 1,024 / 2,048 / 4,096 a block: 159 / 115 / 67 /
// 46 us, an 8-byte pair of floats a store; cold 120 -> 32 (it moves 240 MB). Fewer a block in a small box, to spread over the SMs.
constexpr int kFinishPairs = 8;  // pairs of sums a thread, at most
template <typename real> struct Pair2 { using type = float2; };
template <> struct Pair2<double> { using type = double2; };
template <typename real>
__device__ __forceinline__ real fx_value(long long v, const FinishArgs &a) {
  const int hi = (int)(v >> 32);
  const unsigned lo = (unsigned)(v & 0xffffffffll);
  if (sizeof(real) == 8) return (real)(((double)hi * 4294967296.0 + (double)lo) * a.inv_scale);
  return (real)fmaf((float)hi, a.sh, (float)lo * a.sl);
}

template <typename real>
__device__ __forceinline__ void cpair_finalize_body(const FinishArgs &a, int bx, int) {
  using real2 = typename Pair2<real>::type;
  // (facc and F start 256-byte aligned and b0 is even: pairs)
  const int64_t b0 = (int64_t)bx * a.per, b1 = min(b0 + a.per, a.n3);
  const int np = (int)((b1 - b0) >> 1);
  longlong2 *p = reinterpret_cast<longlong2 *>(a.facc + b0);
  real2 *f = reinterpret_cast<real2 *>(static_cast<real *>(a.F) + b0);
  longlong2 v[kFinishPairs];
#pragma unroll
  for (int k = 0; k < kFinishPairs; ++k) {
    const int t = threadIdx.x + 256 * k;
    if (t < np) v[k] = p[t];
  }
#pragma unroll
  for (int k = 0; k < kFinishPairs; ++k) {
    const int t = threadIdx.x + 256 * k;
    if (t < np) {
      p[t] = make_longlong2(0, 0);
      real2 o;
      o.x = fx_value<real>(v[k].x, a);
      o.y = fx_value<real>(v[k].y, a);
      f[t] = o;
    }
  }
  if (((b1 - b0) & 1) && threadIdx.x == 0) {  // the last sum of an odd number
    const long long w = a.facc[b1 - 1];
    a.facc[b1 - 1] = 0;
    static_cast<real *>(a.F)[b1 - 1] = fx_value<real>(w, a);
  }
}
template <typename real>
__global__ void __launch_bounds__(256) cpair_finalize_kernel(const FinishArgs a) {
  cpair_finalize_body<real>(a, (int)blockIdx.x, (int)gridDim.x);
}
template <typename real>
__global__ void __launch_bounds__(256)
    cpair_finalize_kernel_b(const FinishArgs *__restrict__ t, const int32_t *__restrict__ pre,
                            int nrep) {
  const BatchIdx q = batch_locate(pre, nrep);
  cpair_finalize_body<real>(t[q.r], q.bx, q.nbx);
}

// ---------------------------------------------------------------------------------------
// Pair evaluation

struct CpAcc {
  double u0, u1;  // single type: sum r^-12, sum r^-6; several types: U_LJ, W_LJ
  double uc, wc;  // Coulomb energy and virial
};

// FP64 form: LJ and Coulomb terms of one pair at squared distance r2 inside the cutoff
// (1/r^2 = 0 and qq = 0 give exact zeros); returns the force factor g (F_i += g (r_i - r_j)).
template <bool COUL, bool MULTI>
__device__ __forceinline__ double cp_terms(const ClusterArgs &a, bool in, double r2, double ir2,
                                           double qi, double qj, int ti, int tj, CpAcc &acc) {
  double g;
  const double ir6 = ir2 * ir2 * ir2;
  if (MULTI) {
    const LJTable *tab = a.table;
    const int pt = ti * tab->nt + tj;
    const double w = ir6 * mad(tab->A12d[pt], ir6, -tab->B6d[pt]);
    g = w * ir2;
    acc.u0 = mad(ir6, mad(tab->Ad[pt], ir6, -tab->Bd[pt]), acc.u0);
    acc.u1 += w;
  } else {
    g = ir6 * ir2 * mad(a.ljA12d, ir6, -a.ljB6d);
    acc.u0 = mad(ir6, ir6, acc.u0);
    acc.u1 += ir6;
  }
  if (COUL) {
    const double qq = qi * qj;
    if (in && qq != 0.0) {
      const PairConst &pc = a.pc;
      const double r = sqrt(r2), rinv = 1.0 / r;
      const double erfcv = erfc(pc.sqrt_alpha_d * r);
      const double expv = exp(-pc.alpha_d * r2);
      const double Cqq = pc.C_d * qq;
      const double rinv2 = rinv * rinv;
      const double gc = Cqq * mad(erfcv * rinv, rinv2, pc.two_sqrt_alpha_over_sqrt_pi_d * expv * rinv2);
      g += gc;
      acc.uc = mad(Cqq * erfcv, rinv, acc.uc);
      acc.wc = mad(gc, r2, acc.wc);
    }
  }
  return g;
}

// Candidate j-clusters of a group of i-clusters with box [lo, hi] and frame centre (rx, ry, rz)
// in row (cy, cz), by one warp: for each stencil row (dy, dz), the clusters holding the row's
// particles within the group's x-reach (one lane per row; a row wraps into at most two parts),
// from cluster jmin on; a warp scan gives their offsets. Writes the runs (first cluster, offset;
// the total last) to seg_beg / seg_pre and returns the total.
__device__ __forceinline__ int cp_segments(const ClusterArgs &a, int lane, int cy, int cz,
                                           uint32_t rx, uint32_t ry, uint32_t rz, uint32_t xlo,
                                           uint32_t xhi, uint32_t ylo, uint32_t yhi, uint32_t zlo,
                                           uint32_t zhi, int jmin, int32_t *seg_beg,
                                           int32_t *seg_pre) {
  constexpr unsigned FULL = 0xffffffffu;
  const PairConst &pc = a.pc;
  const int n0 = a.grid.n[0], n1 = a.grid.n[1], n2 = a.grid.n[2];
  const int R1 = a.grid.R[1], R2 = a.grid.R[2];
  const int ny = 2 * R1 + 1, nrst = ny * (2 * R2 + 1);
  const int gxlo = (int)(xlo - rx), gxhi = (int)(xhi - rx);
  const int gylo = (int)(ylo - ry), gyhi = (int)(yhi - ry);
  const int gzlo = (int)(zlo - rz), gzhi = (int)(zhi - rz);
  int carry = 0;
  for (int rb = 0; rb < nrst; rb += 32) {
    const int t = rb + lane;
    int b0 = 0, l0 = 0, b1 = 0, l1 = 0;
    if (t < nrst) {
      const int dz = t / ny - R2, dy = t % ny - R1;
      const int ryw = ((cy + dy) % n1 + n1) % n1, rzw = ((cz + dz) % n2 + n2) % n2;
      const int r2i = ryw + n1 * rzw;
      const int qs = a.set.cell_start[(int64_t)r2i * n0];
      const int qe = a.set.cell_start[(int64_t)(r2i + 1) * n0];
      if (qe > qs) {
        // the row's y and z extent in frame units (unwrapped; cell edges from the width in
        // 2^-16 units, within 2 units up to 2^16 cells, widened by 4 or more), its distance from
        // the group's box, and the x-reach that is left
        const int my = 4 + (n1 >> 16), mz = 4 + (n2 >> 16);
        const int64_t y0 = (((int64_t)(cy + dy) * a.wfix[0]) >> 16) - (int64_t)ry - my;
        const int64_t y1 = (((int64_t)(cy + dy + 1) * a.wfix[0]) >> 16) - (int64_t)ry + my;
        const int64_t z0 = (((int64_t)(cz + dz) * a.wfix[1]) >> 16) - (int64_t)rz - mz;
        const int64_t z1 = (((int64_t)(cz + dz + 1) * a.wfix[1]) >> 16) - (int64_t)rz + mz;
        const int64_t ey = max((int64_t)0, max(y0 - gyhi, (int64_t)gylo - y1));
        const int64_t ez = max((int64_t)0, max(z0 - gzhi, (int64_t)gzlo - z1));
        const float dyl = (float)ey * pc.h[1], dzl = (float)ez * pc.h[2];
        const float rx2 = a.bb2 - dyl * dyl - dzl * dzl;
        if (rx2 > 0.f) {
          const int64_t reach = (int64_t)(sqrtf(rx2) * (1.0f + 1e-5f) / pc.h[0]) + 4;
          const int64_t X0 = (int64_t)rx + gxlo - reach, X1 = (int64_t)rx + gxhi + reach;
          const int64_t W = (int64_t)1 << 32;
          // the particles of the row's cells from key k0 to key k1 (whole cells: the box test
          // rejects the clusters past the reach; a search of the row by x would cost its chain of
          // dependent loads at every block's start)
          auto cell_beg = [&](int64_t key) {
            return a.set.cell_start[(int64_t)r2i * n0 + (int)((key * n0) >> 32)];
          };
          auto cell_end = [&](int64_t key) {
            return a.set.cell_start[(int64_t)r2i * n0 + (int)((key * n0) >> 32) + 1];
          };
          int uH = qs, vH = qs, uL = qs, vL = qs;  // particle ranges: high part, low part
          if (X1 - X0 + 1 >= W) { uL = qs; vL = qe; }
          else if (X0 < 0) { uH = cell_beg(X0 + W); vH = qe; uL = qs; vL = cell_end(X1); }
          else if (X1 >= W) { uH = cell_beg(X0); vH = qe; uL = qs; vL = cell_end(X1 - W); }
          else { uL = cell_beg(X0); vL = cell_end(X1); }
          // to cluster ranges of the row (merged when both parts reach one cluster)
          int kL0 = 0, kL1 = -1, kH0 = 0, kH1 = -1;
          if (vL > uL) { kL0 = (uL - qs) / kClSize; kL1 = (vL - 1 - qs) / kClSize; }
          if (vH > uH) { kH0 = (uH - qs) / kClSize; kH1 = (vH - 1 - qs) / kClSize; }
          if (kL1 >= kL0 && kH1 >= kH0 && kL1 >= kH0 - 1) { kL1 = max(kL1, kH1); kH1 = kH0 - 1; }
          const int base = a.cl_base[r2i];
          if (kL1 >= kL0) {
            const int j0 = max(base + kL0, jmin), j1 = base + kL1;
            if (j1 >= j0) { b0 = j0; l0 = j1 - j0 + 1; }
          }
          if (kH1 >= kH0) {
            const int j0 = max(base + kH0, jmin), j1 = base + kH1;
            if (j1 >= j0) { b1 = j0; l1 = j1 - j0 + 1; }
          }
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
    const int excl = carry + incl - tot;
    if (t < nrst) {
      seg_beg[2 * t] = b0;
      seg_pre[2 * t] = excl;
      seg_beg[2 * t + 1] = b1;
      seg_pre[2 * t + 1] = excl + l0;
    }
    carry += __shfl_sync(FULL, incl, 31);
  }
  if (lane == 0) seg_pre[2 * nrst] = carry;
  return carry;
}

// ---------------------------------------------------------------------------------------
// The FP32 forms' kernel. A super-cluster's visits are shared by `nsplit` blocks of blockDim.y
// warps: warp number w of the W = nsplit * blockDim.y takes every W-th candidate, so the warps
// of a super-cluster carry equal shares. (cpair_shape gives the split and its reason.)
//
// What bounds it: instruction issue and, in the pair loop, latency. A lane's two j particles are
// a packed pair of FP32 values (f32x2.cuh), so the 8 x 8 pairs of an i-cluster cost a warp about
// 33 instructions (49 with scalar pairs); the reaction of a visit is reduced while the next
// visit's j records load; a block's start reads its super-cluster from one record and its
// stencil rows by cell. On 2^20 particles the LJ pass went from 0.99e9 to 0.89e9 instructions
// and from 1,101 to 955 us (issue 75% of the slots, FMA pipe 48%). Per visit (3.3e6 of them):
// the pair loop about 120 instructions, its branches 24, the loads and conversions 38, the
// reaction 31.

// 1.0 where a < b, else 0.0
__device__ __forceinline__ float lt_one(float a, float b) {
  float r;
  asm("set.lt.f32.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
  return r;
}

struct CpAcc2 {
  f32x2 u0, u1;            // one type: the virial and sum r^-6; several: sum 12 A r^-12, sum -6 B r^-6
  f32x2 uc, wc, cuc, cwc;  // Coulomb energy and virial (Kahan compensations)
};

// FP32 forms: terms of one pair inside the cutoff that the exact decision admitted (lj: 12 A and
// -6 B), added to the first half of the sums; returns the force factor.
template <bool COUL, bool MULTI>
__device__ __forceinline__ float cp_band_terms(const ClusterArgs &a, float r2, float qi, float qj,
                                               float2 lj, CpAcc2 &acc) {
  const float ir2 = rcp_approx(r2), ir6 = ir2 * ir2 * ir2, t = fmaf(lj.x, ir6, lj.y);
  float g = MULTI ? ir6 * t * ir2 : ir6 * ir2 * t;
  acc.u0 = add2(acc.u0, pk(MULTI ? lj.x * ir6 * ir6 : ir6 * t, 0.f));
  acc.u1 = add2(acc.u1, pk(MULTI ? lj.y * ir6 : ir6, 0.f));
  if (COUL) {
    const PairConst &pc = a.pc;
    const float Cqq = pc.C * qi * qj, rinv = rsqrtf(r2), r = r2 * rinv;
    const float u = Cqq * erfcf(pc.sqrt_alpha * r) * rinv;
    const float gc = fmaf(Cqq * pc.two_sqrt_alpha_over_sqrt_pi, expf(-pc.alpha * r2), u) * ir2;
    g += gc;
    acc.uc = add2(acc.uc, pk(u, 0.f));
    acc.wc = add2(acc.wc, pk(gc * r2, 0.f));
  }
  return g;
}

// COUL: 0 none, 1 with the erfcx fit (ErfcFit), 2 with erfcf and expf
template <int COUL, bool MULTI, bool COUNT>
__device__ __forceinline__ void cpair32_body(const ClusterArgs &a, int bx, int nbx) {
  constexpr int NC = 8;                    // clusters per super-cluster
  constexpr int NP = NC * kClSize;         // particles per super-cluster
  constexpr unsigned FULL = 0xffffffffu;
  __shared__ uint4 si[NP];                 // s_x, s_y, s_z, charge bits
  __shared__ int32_t sti[MULTI ? NP : 1];
  __shared__ float4 ibl[NC];               // i-cluster boxes in frame coordinates: -hi x, lo x,
  __shared__ float2 ibz[NC];               // -hi y, lo y; -hi z, lo z
  // the group's i particles in frame coordinates (x, y, z, charge); slots outside the group hold
  // a point no j reaches
  __shared__ float4 sif[NP];
  __shared__ float2 stab[MULTI ? kMaxTypes * kMaxTypes : 1];  // (12 A, -6 B) per type pair
  __shared__ int32_t seg_beg[kCpMaxSeg], seg_pre[kCpMaxSeg + 1];
  __shared__ int T_s;
  __shared__ double wred[kCpMaxWarps][NQ_PAIR];
  // candidates a warp visits: (J, mask | count << 8, first particle, -corner y), -corner z
  extern __shared__ uint4 rec_dyn[];
  const int lane = threadIdx.x, wid = threadIdx.y, W = blockDim.y, a8 = lane & 7, hh = lane >> 3;
  const int tid = wid * 32 + lane, nthr = W * 32;
  uint4 *const rec = rec_dyn + wid * 32;
  float *const recz = reinterpret_cast<float *>(rec_dyn + W * 32) + wid * 32;
  const int w = bx / a.nsplit, part = (bx - w * a.nsplit) * W + wid, nparts = a.nsplit * W;
  const PairConst &pc = a.pc;
  const int64_t N = a.N;
  // this lane's j particles of a visited cluster, and where it adds their reaction (lanes with
  // bits 1 and 2 of a8 set add nothing)
  const bool b0 = a8 & 1, b1 = a8 & 2, b2 = a8 & 4;
  const int ja = hh + (b0 ? 4 : 0), jb_ = hh + (b0 ? 0 : 4);
  const int rslot = b1 && b2 ? INT_MAX : ja;
  long long *const fdst = a.facc + (int64_t)(b2 ? 2 : (b1 ? 1 : 0)) * N + ja;
  CpAcc2 acc;
  acc.u0 = acc.u1 = acc.uc = acc.wc = acc.cuc = acc.cwc = pk(0.f);
  const int nrows = a.nrows;
  if (w < a.sc_base[nrows]) {
    const int4 info = a.sc_info[w];
    const int g0 = info.y, nc = info.w & 0xff, p0 = info.z, np = info.w >> 8;
    const int cy = info.x % a.grid.n[1], cz = info.x / a.grid.n[1];
    // (slots past the particles hold type 0 and no charge: masked lanes still look up the
    // LJ table by type before their result is zeroed)
    for (int t = tid; t < NP; t += nthr) {
      uint4 v = make_uint4(0u, 0u, 0u, 0u);
      int ty = 0;
      if (t < np) {
        const int p = p0 + t;
        v = make_uint4(a.set.sx[p], a.set.sy[p], a.set.sz[p],
                       COUL ? __float_as_uint(a.set.qf[p]) : 0u);
        if (MULTI) ty = a.set.type[p];
      }
      si[t] = v;
      if (MULTI) sti[t] = ty;
    }
    const int nt = MULTI ? a.table->nt : 1;
    if (MULTI)
      for (int t = tid; t < nt * nt; t += nthr) stab[t] = make_float2(a.table->A12[t], -a.table->B6[t]);
    __syncthreads();
    // Groups of consecutive clusters whose x extent the frame allows (normally one group).
    // A single cluster wider than that is taken one particle at a time (asub), as a group
    // of one point.
    int cb = 0, asub = -1;
    while (cb < nc) {
      int ce = cb + 1;
      if (asub < 0) {
        const uint32_t xfirst = si[kClSize * cb].x;
        while (ce < nc && si[min(np, kClSize * (ce + 1)) - 1].x - xfirst <= a.xlim) ++ce;
        if (si[min(np, kClSize * ce) - 1].x - xfirst > a.xlim) asub = 0;
      }
      const int q0 = asub < 0 ? kClSize * cb : kClSize * cb + asub;
      const int q1 = asub < 0 ? min(np, kClSize * ce) : q0 + 1;
      // group box and frame centre (no wrap inside a row: x ascending, y and z in one cell)
      uint32_t ylo = 0xffffffffu, yhi = 0u, zlo = 0xffffffffu, zhi = 0u;
      for (int t = q0 + lane; t < q1; t += 32) {
        const uint4 v = si[t];
        ylo = min(ylo, v.y); yhi = max(yhi, v.y);
        zlo = min(zlo, v.z); zhi = max(zhi, v.z);
      }
      ylo = __reduce_min_sync(FULL, ylo); yhi = __reduce_max_sync(FULL, yhi);
      zlo = __reduce_min_sync(FULL, zlo); zhi = __reduce_max_sync(FULL, zhi);
      const uint32_t xlo = si[q0].x, xhi = si[q1 - 1].x;
      const uint32_t rx = xlo + ((xhi - xlo) >> 1), ry = ylo + ((yhi - ylo) >> 1),
                     rz = zlo + ((zhi - zlo) >> 1);
      for (int t = tid; t < NP; t += nthr) {
        const int c = t / kClSize, a_ = t % kClSize;
        const bool v = c >= cb && c < ce && t < np && (asub < 0 || a_ == asub);
        const uint4 s = si[t];
        const float x = v ? (float)(int)(s.x - rx) * pc.h[0] : 3e18f;
        const float y = v ? (float)(int)(s.y - ry) * pc.h[1] : 3e18f;
        const float z = v ? (float)(int)(s.z - rz) * pc.h[2] : 3e18f;
        const float q = v && COUL ? __uint_as_float(s.w) : 0.f;
        sif[t] = make_float4(x, y, z, q);
      }
      if (wid == 0) {
        // i-cluster boxes in the frame (lanes cb..ce-1)
        if (lane < NC) {
          float4 lo4 = make_float4(3e18f, 3e18f, 3e18f, 0.f), hi4 = make_float4(3e18f, 3e18f, 3e18f, 0.f);
          if (lane >= cb && lane < ce) {
            uint4 l, u;
            if (asub < 0) { l = a.cl_lo[g0 + lane]; u = a.cl_hi[g0 + lane]; }
            else { l = u = si[q0]; }  // the one particle of a point group
            lo4 = make_float4((float)(int)(l.x - rx) * pc.h[0], (float)(int)(l.y - ry) * pc.h[1],
                              (float)(int)(l.z - rz) * pc.h[2], 0.f);
            hi4 = make_float4((float)(int)(u.x - rx) * pc.h[0], (float)(int)(u.y - ry) * pc.h[1],
                              (float)(int)(u.z - rz) * pc.h[2], 0.f);
          }
          ibl[lane] = make_float4(-hi4.x, lo4.x, -hi4.y, lo4.y);
          ibz[lane] = make_float2(-hi4.z, lo4.z);
        }
        const int T0 = cp_segments(a, lane, cy, cz, rx, ry, rz, xlo, xhi, ylo, yhi, zlo, zhi, g0 + cb,
                                   seg_beg, seg_pre);
        if (lane == 0) T_s = T0;
      }
      __syncthreads();
      const int T = T_s;
      const int nseg = 2 * (2 * a.grid.R[1] + 1) * (2 * a.grid.R[2] + 1);
      // forces on particle a8 of each i-cluster
      float fxi[NC], fyi[NC], fzi[NC];
      int cnti[NC];
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        fxi[c] = fyi[c] = fzi[c] = 0.f;
        cnti[c] = 0;
      }
      // Minus the reaction on the j-cluster visited last (particles ja, jb of the cluster), its
      // first particle and count. It is summed and added at the next visit, while that visit's
      // j records load: over the 8 lanes sharing h, first with lane a8 xor 1, which holds the
      // same two particles in the other order (each keeps its first one's sums: no selection),
      // then x or y (the lane's bit 1 tells which) and z with lanes a8 xor 2 and xor 4. Every
      // sum is the tree ((v_a + v_a^1) + (v_a^2 + v_a^3)) + (...). (The scale's sign turns it.)
      f32x2 fxj = pk(0.f), fyj = pk(0.f), fzj = pk(0.f);
      int pvb = 0, pvn = 0;
      auto reaction = [&]() {
        const float x0 = fxj.x + __shfl_xor_sync(FULL, fxj.y, 1);
        const float y0 = fyj.x + __shfl_xor_sync(FULL, fyj.y, 1);
        float z0 = fzj.x + __shfl_xor_sync(FULL, fzj.y, 1);
        float u = (b1 ? y0 : x0) + __shfl_xor_sync(FULL, b1 ? x0 : y0, 2);
        z0 += __shfl_xor_sync(FULL, z0, 2);
        u += __shfl_xor_sync(FULL, u, 4);
        z0 += __shfl_xor_sync(FULL, z0, 4);
        if (rslot < pvn) fx_add(fdst + pvb, b2 ? z0 : u, -a.fscale, a.err);
      };
      // This warp's candidates in chunks of 32, one per lane: the box test against every
      // i-cluster of the group gives a mask, the candidates with a mask are compacted into the
      // warp's records, and the warp visits them.
      for (int base = part; base < T; base += 32 * nparts) {
        const int cc = base + lane * nparts;
        uint32_t msk = 0u;
        int J = 0, jb = 0, jn = 0;
        float cy0 = 0.f, cz0 = 0.f;  // the candidate box's low corner in y and z (frame)
        if (cc < T) {
          int s = 0, e = nseg;       // the candidate's run: the last one starting at or before it
          while (e - s > 1) {
            const int mid = (s + e) >> 1;
            if (seg_pre[mid] <= cc) s = mid; else e = mid;
          }
          J = seg_beg[s] + (cc - seg_pre[s]);
          const uint4 l = a.cl_lo[J], u = a.cl_hi[J];
          jb = (int)l.w;
          jn = (int)u.w;
          const float jx0 = (float)(int)(l.x - rx) * pc.h[0];
          const float jy0 = (float)(int)(l.y - ry) * pc.h[1];
          const float jz0 = (float)(int)(l.z - rz) * pc.h[2];
          cy0 = jy0;
          cz0 = jz0;
          const float jx1 = (float)(int)(u.x - rx) * pc.h[0];
          const float jy1 = (float)(int)(u.y - ry) * pc.h[1];
          const float jz1 = (float)(int)(u.z - rz) * pc.h[2];
          // a box that reaches past L/2 from the frame centre wraps (its ends swap sides): its
          // distance is then that of the nearer of its two pieces
          const bool wx = jx0 > jx1, wy = jy0 > jy1, wz = jz0 > jz1;
          const f32x2 px = pk(jx0, -jx1), py = pk(jy0, -jy1), pz = pk(jz0, -jz1);
          if (!(wx || wy || wz)) {
#pragma unroll
            for (int c = 0; c < NC; ++c) {
              const float4 bxy = ibl[c];
              const f32x2 ex = add2(px, pk(bxy.x, bxy.y)), ey = add2(py, pk(bxy.z, bxy.w));
              const f32x2 ez = add2(pz, ibz[c]);
              const float gx = max3(0.f, ex.x, ex.y), gy = max3(0.f, ey.x, ey.y),
                          gz = max3(0.f, ez.x, ez.y);
              msk |= fmaf(gx, gx, fmaf(gy, gy, gz * gz)) <= a.bb2 ? (1u << c) : 0u;
            }
          } else {
            // (a box that straddles the frame's edge in y or z by its lower piece, nearer the
            // group: its corner counts from below, so that corner plus offset stays in reach)
            if (wy && (float)(int)(ylo - ry) * pc.h[1] - jy1 < jy0 - (float)(int)(yhi - ry) * pc.h[1])
              cy0 = jy0 - 4294967296.f * pc.h[1];
            if (wz && (float)(int)(zlo - rz) * pc.h[2] - jz1 < jz0 - (float)(int)(zhi - rz) * pc.h[2])
              cz0 = jz0 - 4294967296.f * pc.h[2];
            for (int c = 0; c < NC; ++c) {
              const float4 bxy = ibl[c];
              const float2 bz = ibz[c];
              const float ax = jx0 + bxy.x, bx_ = bxy.y - jx1;
              const float ay = jy0 + bxy.z, by_ = bxy.w - jy1;
              const float az = jz0 + bz.x, bz_ = bz.y - jz1;
              const float gx = fmaxf(0.f, wx ? fminf(ax, bx_) : fmaxf(ax, bx_));
              const float gy = fmaxf(0.f, wy ? fminf(ay, by_) : fmaxf(ay, by_));
              const float gz = fmaxf(0.f, wz ? fminf(az, bz_) : fmaxf(az, bz_));
              msk |= fmaf(gx, gx, fmaf(gy, gy, gz * gz)) <= a.bb2 ? (1u << c) : 0u;
            }
          }
          // the group's clusters at or before J (a pair of clusters is taken once)
          const int last = min(ce - 1, J - g0);
          msk &= (2u << last) - (1u << cb);
        }
        const unsigned vis = __ballot_sync(FULL, msk != 0u);
        if (msk) {
          const int k = __popc(vis & ((1u << lane) - 1u));
          rec[k] = make_uint4((uint32_t)J, msk | ((uint32_t)jn << 8), (uint32_t)jb,
                              __float_as_uint(-cy0));
          recz[k] = -cz0;
        }
        __syncwarp();
        const int nv = __popc(vis);
        for (int v = 0; v < nv; ++v) {
          const uint4 rc4 = rec[v];
          const float ncz = recz[v];
          const int Jv = (int)rc4.x, vb = (int)rc4.z, vn = (int)(rc4.y >> 8);
          const uint32_t M = rc4.y & 0xffu;
          const float ncy = __uint_as_float(rc4.w);
          const int cdiag = Jv - g0;  // the visited cluster's place in the super-cluster
          // This lane's j particles, ja and jb of the cluster, as negated coordinates: x from
          // the exact integer offset from the frame centre, y and z from the cluster's corner
          // plus the record's offsets (an empty slot's offset of -3e18 puts it out of reach).
          const uint4 *jr = a.jrec + ((int64_t)Jv << 3);
          const uint4 pj0 = __ldg(jr + ja), pj1 = __ldg(jr + jb_);
          reaction();
          const f32x2 nx = pk((float)(int)(rx - pj0.x) * pc.h[0], (float)(int)(rx - pj1.x) * pc.h[0]);
          const f32x2 ny = pk(ncy - __uint_as_float(pj0.y), ncy - __uint_as_float(pj1.y));
          const f32x2 nz = pk(ncz - __uint_as_float(pj0.z), ncz - __uint_as_float(pj1.z));
          f32x2 qjC = pk(0.f);
          if (COUL) qjC = mul2(pk(__uint_as_float(pj0.w), __uint_as_float(pj1.w)), pk(pc.C));
          int tj0 = 0, tj1 = 0;
          if (MULTI) {
            tj0 = ja < vn ? a.set.type[vb + ja] : 0;
            tj1 = jb_ < vn ? a.set.type[vb + jb_] : 0;
          }
          fxj = fyj = fzj = pk(0.f);
          int cntj0 = 0, cntj1 = 0;
          float bmin = 3e38f;  // smallest |r^2 - r_c^2| of the visit (band test)
          // Force factors of an i particle with this lane's two j particles, their displacements,
          // and the force on j. (ok0, ok1: the pair counts, for a cluster with itself)
          auto pairs = [&](f32x2 xi, f32x2 yi, f32x2 zi, f32x2 qi, int ti, bool self, bool ok0,
                           bool ok1, f32x2 &dx, f32x2 &dy, f32x2 &dz, bool &in0, bool &in1) -> f32x2 {
            dx = add2(xi, nx);
            dy = add2(yi, ny);
            dz = add2(zi, nz);
            f32x2 r2 = fma2(dx, dx, fma2(dy, dy, mul2(dz, dz)));
            float ra = r2.x, rb = r2.y;
            const f32x2 bd = add2(r2, pk(-a.rc2_mid));
            bmin = min3(bmin, fabsf(bd.x), fabsf(bd.y));
            if (self) {
              ra = ok0 ? ra : 3e37f;
              rb = ok1 ? rb : 3e37f;
            }
            in0 = ra < pc.rc2_lo;
            in1 = rb < pc.rc2_lo;
            const f32x2 m = pk(lt_one(ra, pc.rc2_lo), lt_one(rb, pc.rc2_lo));
            const f32x2 ir2 = mul2(pk(rcp_approx(ra), rcp_approx(rb)), m);
            const f32x2 ir6 = mul2(mul2(ir2, ir2), ir2);
            f32x2 g;
            if (MULTI) {
              const float2 t0 = stab[ti * nt + tj0], t1 = stab[ti * nt + tj1];
              const f32x2 A = pk(t0.x, t1.x), B = pk(t0.y, t1.y);
              g = mul2(mul2(ir6, fma2(A, ir6, B)), ir2);  // (r^-8 alone leaves FP32 sooner)
              acc.u0 = fma2(mul2(A, ir6), ir6, acc.u0);
              acc.u1 = fma2(B, ir6, acc.u1);
            } else {
              // (12 A stays in the factor: forces in units of 12 A would leave FP32's range in
              // large units of length, at 340 pm say, and were no faster)
              const f32x2 t = fma2(pk(a.ljA12), ir6, pk(-a.ljB6));
              g = mul2(mul2(ir6, ir2), t);
              acc.u0 = fma2(ir6, t, acc.u0);
              acc.u1 = add2(acc.u1, ir6);
            }
            if (COUL) {
              const f32x2 qq = mul2(qi, qjC);
              const float ca = fminf(ra, pc.rc2_hi), cbb = fminf(rb, pc.rc2_hi);
              const f32x2 r2c = pk(ca, cbb);
              const f32x2 rinv = pk(rsqrtf(ca), rsqrtf(cbb));
              const f32x2 rr = mul2(r2c, rinv);
              f32x2 er, ex;
              if (COUL == 1) {
                erfc_exp2(a.fit, rr, r2c, er, ex);
              } else {
                er = pk(erfcf(pc.sqrt_alpha * rr.x), erfcf(pc.sqrt_alpha * rr.y));
                ex = pk(expf(-pc.alpha * ca), expf(-pc.alpha * cbb));
              }
              const f32x2 u = mul2(mul2(qq, er), mul2(rinv, m));
              const f32x2 ts = pk(pc.two_sqrt_alpha_over_sqrt_pi);
              const f32x2 gc = mul2(fma2(mul2(qq, ts), ex, u), ir2);
              g = add2(g, gc);
              if (a.comp) {
                kahan_add2(acc.uc, acc.cuc, u);
                kahan_add2(acc.wc, acc.cwc, mul2(gc, r2c));
              } else {
                acc.uc = add2(acc.uc, u);
                acc.wc = fma2(gc, r2c, acc.wc);
              }
            }
            fxj = fma2(g, dx, fxj);
            fyj = fma2(g, dy, fyj);
            fzj = fma2(g, dz, fzj);
            if (COUNT) {
              cntj0 += in0 ? 1 : 0;
              cntj1 += in1 ? 1 : 0;
            }
            return g;
          };
          // The visited cluster may be one of the super-cluster's own (cdiag): its pairs with
          // itself count once (particle a8 with a later one). They are taken here, with the i
          // particle's force added by atomics, so that the loop below carries no exclusion.
          uint32_t Mh = M;
          if (cdiag >= 0 && cdiag < NC && ((M >> cdiag) & 1u)) {
            Mh &= ~(1u << cdiag);
            const int t = kClSize * cdiag + a8;
            const bool vd = t < np && (asub < 0 || a8 == asub);
            const float4 pi = sif[t];
            f32x2 dx, dy, dz;
            bool in0, in1;
            const f32x2 g = pairs(pk(pi.x), pk(pi.y), pk(pi.z), pk(pi.w), MULTI ? sti[t] : 0, true, vd && a8 < ja,
                                  vd && a8 < jb_, dx, dy, dz, in0, in1);
            float fdx = fmaf(g.y, dx.y, g.x * dx.x), fdy = fmaf(g.y, dy.y, g.x * dy.x),
                  fdz = fmaf(g.y, dz.y, g.x * dz.x);
            fdx += __shfl_xor_sync(FULL, fdx, 8); fdx += __shfl_xor_sync(FULL, fdx, 16);
            fdy += __shfl_xor_sync(FULL, fdy, 8); fdy += __shfl_xor_sync(FULL, fdy, 16);
            fdz += __shfl_xor_sync(FULL, fdz, 8); fdz += __shfl_xor_sync(FULL, fdz, 16);
            if (vd && hh < 3)
              fx_add(a.facc + (int64_t)hh * N + p0 + t, hh == 0 ? fdx : (hh == 1 ? fdy : fdz),
                     a.fscale, a.err);
            if (COUNT) {
              int cd = (in0 ? 1 : 0) + (in1 ? 1 : 0);
              cd += __shfl_xor_sync(FULL, cd, 8);
              cd += __shfl_xor_sync(FULL, cd, 16);
              if (vd && hh == 3 && cd) atomicAdd(a.nbr + p0 + t, cd);
            }
          }
#pragma unroll
          for (int c = 0; c < NC; ++c) {
            if ((Mh >> c) & 1u) {
              const int t = kClSize * c + a8;
              const float4 pi = sif[t];
              f32x2 dx, dy, dz;
              bool in0, in1;
              const f32x2 g = pairs(pk(pi.x), pk(pi.y), pk(pi.z), pk(pi.w), MULTI ? sti[t] : 0, false, true, true,
                                    dx, dy, dz, in0, in1);
              fxi[c] = fmaf(g.y, dx.y, fmaf(g.x, dx.x, fxi[c]));
              fyi[c] = fmaf(g.y, dy.y, fmaf(g.x, dy.x, fyi[c]));
              fzi[c] = fmaf(g.y, dz.y, fmaf(g.x, dz.x, fzi[c]));
              if (COUNT) cnti[c] += (in0 ? 1 : 0) + (in1 ? 1 : 0);
            }
          }
          // Band pairs: the exact decision; a pair inside is added by atomics.
          if (__any_sync(FULL, bmin <= a.rc2_half)) {
            for (int c = cb; c < ce; ++c) {
              if (!((M >> c) & 1u)) continue;
              const int t = kClSize * c + a8;
              if (t >= np || (asub >= 0 && a8 != asub)) continue;
              const uint4 s = si[t];
              const float x0 = sif[t].x, y0 = sif[t].y, z0 = sif[t].z;
              for (int k = 0; k < 2; ++k) {
                const int j = k ? jb_ : ja;
                if (!(j < vn) || !(c != cdiag || a8 < j)) continue;
                const float dx = x0 + (k ? nx.y : nx.x), dy = y0 + (k ? ny.y : ny.x),
                            dz = z0 + (k ? nz.y : nz.x);
                const float r2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
                if (!(r2 >= pc.rc2_lo && r2 <= pc.rc2_hi)) continue;
                const int pj = vb + j;
                const int dsx = (int)(s.x - a.set.sx[pj]), dsy = (int)(s.y - a.set.sy[pj]),
                          dsz = (int)(s.z - a.set.sz[pj]);
                if (!(exact_r2(pc, dsx, dsy, dsz) <= pc.rc2d)) continue;
                const float g = cp_band_terms<COUL != 0, MULTI>(
                    a, r2, COUL ? __uint_as_float(s.w) : 0.f, COUL ? a.set.qf[pj] : 0.f,
                    MULTI ? stab[sti[t] * nt + (k ? tj1 : tj0)] : make_float2(a.ljA12, -a.ljB6), acc);
                const int pi = p0 + t;
                fx_add(a.facc + pi, g * dx, a.fscale, a.err);
                fx_add(a.facc + N + pi, g * dy, a.fscale, a.err);
                fx_add(a.facc + 2 * N + pi, g * dz, a.fscale, a.err);
                fx_add(a.facc + pj, -g * dx, a.fscale, a.err);
                fx_add(a.facc + N + pj, -g * dy, a.fscale, a.err);
                fx_add(a.facc + 2 * N + pj, -g * dz, a.fscale, a.err);
                if (COUNT) { atomicAdd(a.nbr + pi, 1); atomicAdd(a.nbr + pj, 1); }
              }
            }
          }
          if (COUNT) {
            const unsigned gm = 0xffu << (8 * hh);
            const int c0 = __reduce_add_sync(gm, b0 ? cntj1 : cntj0);
            const int c1 = __reduce_add_sync(gm, b0 ? cntj0 : cntj1);
            if (a8 == 0) {
              if (hh < vn && c0) atomicAdd(a.nbr + vb + hh, c0);
              if (hh + 4 < vn && c1) atomicAdd(a.nbr + vb + hh + 4, c1);
            }
          }
          pvb = vb;
          pvn = vn;
        }
        __syncwarp();
      }
      reaction();
      // i forces: sum over the four lanes sharing a8, then lane (h, a8) adds clusters c with
      // c % 4 == h
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        float fx = fxi[c], fy = fyi[c], fz = fzi[c];
        fx += __shfl_xor_sync(FULL, fx, 8); fx += __shfl_xor_sync(FULL, fx, 16);
        fy += __shfl_xor_sync(FULL, fy, 8); fy += __shfl_xor_sync(FULL, fy, 16);
        fz += __shfl_xor_sync(FULL, fz, 8); fz += __shfl_xor_sync(FULL, fz, 16);
        if (COUNT) {
          cnti[c] += __shfl_xor_sync(FULL, cnti[c], 8);
          cnti[c] += __shfl_xor_sync(FULL, cnti[c], 16);
        }
        const int t = kClSize * c + a8;
        if ((c & 3) == hh && c >= cb && c < ce && t < np && (asub < 0 || a8 == asub)) {
          const int64_t pi = p0 + t;
          fx_add(a.facc + pi, fx, a.fscale, a.err);
          fx_add(a.facc + N + pi, fy, a.fscale, a.err);
          fx_add(a.facc + 2 * N + pi, fz, a.fscale, a.err);
          if (COUNT && cnti[c]) atomicAdd(a.nbr + pi, cnti[c]);
        }
      }
      __syncthreads();  // (the group's shared arrays are free for the next one)
      if (asub < 0) {
        cb = ce;
      } else if (++asub >= min(kClSize, np - kClSize * cb)) {
        asub = -1;
        ++cb;
      }
    }
  }
  // Block partials of the energies and virials (each pair counted once). FP64 runs at 1/64 of the
  // FP32 rate, and in a small box all warps end together: the sums are converted by integer
  // operations and reduced as a list, and the LJ units enter once a block (3,000 charged
  // particles: FP64 pipe 29% of the pass, 44.6 -> 43.2 us; list 4 x 5 additions a warp before, 6 now).
  const double e0 = f2d(acc.u0.x) + f2d(acc.u0.y), e1 = f2d(acc.u1.x) + f2d(acc.u1.y);
  double s;  // lane k: sum k of u0, u1 and with Coulomb terms energy and virial
  if (COUL) {
    const double e[4] = {
        e0, e1, (f2d(acc.uc.x) - f2d(acc.cuc.x)) + (f2d(acc.uc.y) - f2d(acc.cuc.y)),
        (f2d(acc.wc.x) - f2d(acc.cwc.x)) + (f2d(acc.wc.y) - f2d(acc.cwc.y))};
    s = warp_sum4(e, lane);
  } else {
    s = warp_sum2(e0, e1, lane);
  }
  constexpr int NS = COUL ? 4 : 2;
  if (W > 1) {
    if (lane < NS) wred[wid][lane] = s;
    __syncthreads();
    if (wid == 0) {
      s = 0.0;
      for (int k = 0; k < W; ++k) s += wred[k][lane % NS];
    }
  }
  if (wid == 0) {
    const double u0 = __shfl_sync(FULL, s, 0), u1 = __shfl_sync(FULL, s, 1);
    const double uc = COUL ? __shfl_sync(FULL, s, 2) : 0.0, wc = COUL ? __shfl_sync(FULL, s, 3) : 0.0;
    if (lane == 0) {
      double *out = a.epart + (int64_t)bx * NQ_PAIR;
      // (one type: u0 = 12 A s12 - 6 B s6 and u1 = s6, so A s12 - B s6 = (u0 - 6 B s6) / 12)
      out[Q_ULJ] = MULTI ? u0 / 12.0 + u1 / 6.0 : (u0 - (double)a.ljB6 * u1) / 12.0;
      out[Q_WLJ] = MULTI ? u0 + u1 : u0;
      out[Q_UREAL] = uc;
      out[Q_WREAL] = wc;
    }
  }
  // the pass's partial slots past the grid (the range is sized for the per-particle kernel,
  // the grid for the super-clusters) hold zeros
  for (int64_t z = (int64_t)bx + nbx; z < a.nslots; z += nbx)
    if (tid < NQ_PAIR) a.epart[z * NQ_PAIR + tid] = 0.0;
}

// (Register caps: 72 for the LJ pass, 28 warps an SM at 60 spilled bytes; 80 without spills
// ran 2% slower, 96 8% slower. 96 with Coulomb terms, 20 warps; 128 ran 10% slower.)
template <int COUL, bool MULTI, bool COUNT>
__global__ void __launch_bounds__(32 * kCpMaxWarps,
                                  (COUL ? kCpWarpsCoul : kCpWarpsLJ) / kCpMaxWarps)
    cpair32_kernel(const ClusterArgs a) {
  cpair32_body<COUL, MULTI, COUNT>(a, (int)blockIdx.x, (int)gridDim.x);
}

// ---------------------------------------------------------------------------------------
// The FP64 form's kernel: one warp per super-cluster.

template <bool COUL, bool MULTI, bool COUNT>
__device__ __forceinline__ void cpair64_body(const ClusterArgs &a, int bx, int nbx) {
  using real = double;
  constexpr int NC = 4;                    // clusters per super-cluster
  constexpr int NP = NC * kClSize;         // particles per super-cluster
  constexpr unsigned FULL = 0xffffffffu;
  __shared__ uint4 si[NP];                 // s_x, s_y, s_z
  __shared__ int32_t sti[MULTI ? NP : 1];
  __shared__ float4 ibl[NC], ibh[NC];      // i-cluster boxes in frame coordinates
  __shared__ int32_t seg_beg[kCpMaxSeg], seg_pre[kCpMaxSeg + 1];
  const int lane = threadIdx.x, a8 = lane & 7, hh = lane >> 3;
  const int w = bx;
  const PairConst &pc = a.pc;
  const int64_t N = a.N;
  CpAcc acc;
  acc.u0 = acc.u1 = acc.uc = acc.wc = 0.0;
  const int nrows = a.nrows;
  if (w < a.sc_base[nrows]) {
    const int4 info = a.sc_info[w];
    const int g0 = info.y, nc = info.w & 0xff, p0 = info.z, np = info.w >> 8;
    const int cy = info.x % a.grid.n[1], cz = info.x / a.grid.n[1];
    // (slots past the particles hold type 0 and no charge: masked lanes still look up the
    // LJ table by type before their result is zeroed)
    for (int t = lane; t < NP; t += 32) {
      uint4 v = make_uint4(0u, 0u, 0u, 0u);
      int ty = 0;
      if (t < np) {
        const int p = p0 + t;
        v = make_uint4(a.set.sx[p], a.set.sy[p], a.set.sz[p], 0u);
        if (MULTI) ty = a.set.type[p];
      }
      si[t] = v;
      if (MULTI) sti[t] = ty;
    }
    __syncwarp();
    // Groups of consecutive clusters whose x extent the frame allows (normally one group).
    // A single cluster wider than that is taken one particle at a time (asub), as a group
    // of one point.
    int cb = 0, asub = -1;
    while (cb < nc) {
      int ce = cb + 1;
      if (asub < 0) {
        const uint32_t xfirst = si[kClSize * cb].x;
        while (ce < nc && si[min(np, kClSize * (ce + 1)) - 1].x - xfirst <= a.xlim) ++ce;
        if (si[min(np, kClSize * ce) - 1].x - xfirst > a.xlim) asub = 0;
      }
      const int q0 = asub < 0 ? kClSize * cb : kClSize * cb + asub;
      const int q1 = asub < 0 ? min(np, kClSize * ce) : q0 + 1;
      // group box and frame centre (no wrap inside a row: x ascending, y and z in one cell)
      uint32_t ylo = 0xffffffffu, yhi = 0u, zlo = 0xffffffffu, zhi = 0u;
      for (int t = q0 + lane; t < q1; t += 32) {
        const uint4 v = si[t];
        ylo = min(ylo, v.y); yhi = max(yhi, v.y);
        zlo = min(zlo, v.z); zhi = max(zhi, v.z);
      }
      ylo = __reduce_min_sync(FULL, ylo); yhi = __reduce_max_sync(FULL, yhi);
      zlo = __reduce_min_sync(FULL, zlo); zhi = __reduce_max_sync(FULL, zhi);
      const uint32_t xlo = si[q0].x, xhi = si[q1 - 1].x;
      const uint32_t rx = xlo + ((xhi - xlo) >> 1), ry = ylo + ((yhi - ylo) >> 1),
                     rz = zlo + ((zhi - zlo) >> 1);
      // i particles of this lane: particle a8 of each cluster of the group
      real fxi[NC], fyi[NC], fzi[NC], qi[NC];
      int oxi[NC], oyi[NC], ozi[NC], ti[NC], cnti[NC];
      bool vi[NC];
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        const int t = kClSize * c + a8;
        const bool v = c >= cb && c < ce && t < np && (asub < 0 || a8 == asub);
        vi[c] = v;
        const uint4 s = si[t];
        oxi[c] = (int)(s.x - rx); oyi[c] = (int)(s.y - ry); ozi[c] = (int)(s.z - rz);
        qi[c] = COUL && v ? a.set.qd[p0 + t] : 0.0;
        ti[c] = MULTI ? sti[t] : 0;
        fxi[c] = fyi[c] = fzi[c] = (real)0;
        cnti[c] = 0;
      }
      // i-cluster boxes in the frame (lanes cb..ce-1)
      if (lane < NC) {
        float4 lo4 = make_float4(3e18f, 3e18f, 3e18f, 0.f), hi4 = make_float4(3e18f, 3e18f, 3e18f, 0.f);
        if (lane >= cb && lane < ce) {
          uint4 l, u;
          if (asub < 0) { l = a.cl_lo[g0 + lane]; u = a.cl_hi[g0 + lane]; }
          else { l = u = si[q0]; }  // the one particle of a point group
          lo4 = make_float4((float)(int)(l.x - rx) * pc.h[0], (float)(int)(l.y - ry) * pc.h[1],
                            (float)(int)(l.z - rz) * pc.h[2], 0.f);
          hi4 = make_float4((float)(int)(u.x - rx) * pc.h[0], (float)(int)(u.y - ry) * pc.h[1],
                            (float)(int)(u.z - rz) * pc.h[2], 0.f);
        }
        ibl[lane] = lo4;
        ibh[lane] = hi4;
      }
      const int T = cp_segments(a, lane, cy, cz, rx, ry, rz, xlo, xhi, ylo, yhi, zlo, zhi, g0 + cb,
                                seg_beg, seg_pre);
      __syncwarp();
      // Candidates in chunks of 32, one per lane: the box test against every i-cluster of
      // the group gives a mask; the warp then visits each candidate with a mask.
      int sg = 0;
      for (int base = 0; base < T; base += 32) {
        const int cc = base + lane;
        int s = sg, J = 0, jb = 0, jn = 0;
        uint32_t msk = 0u;
        if (cc < T) {
          while (seg_pre[s + 1] <= cc) ++s;
          J = seg_beg[s] + (cc - seg_pre[s]);
          const uint4 l = a.cl_lo[J], u = a.cl_hi[J];
          jb = (int)l.w;
          jn = (int)u.w;
          const float jx0 = (float)(int)(l.x - rx) * pc.h[0];
          const float jy0 = (float)(int)(l.y - ry) * pc.h[1];
          const float jz0 = (float)(int)(l.z - rz) * pc.h[2];
          const float jx1 = (float)(int)(u.x - rx) * pc.h[0];
          const float jy1 = (float)(int)(u.y - ry) * pc.h[1];
          const float jz1 = (float)(int)(u.z - rz) * pc.h[2];
          // a box that reaches past L/2 from the frame centre wraps (its ends swap sides): its
          // distance is then that of the nearer of its two pieces
          const bool wx = jx0 > jx1, wy = jy0 > jy1, wz = jz0 > jz1;
#pragma unroll
          for (int c = 0; c < NC; ++c) {
            const float4 lo4 = ibl[c], hi4 = ibh[c];
            const float ax = jx0 - hi4.x, bx = lo4.x - jx1;
            const float ay = jy0 - hi4.y, by = lo4.y - jy1;
            const float az = jz0 - hi4.z, bz = lo4.z - jz1;
            const float gx = fmaxf(0.f, wx ? fminf(ax, bx) : fmaxf(ax, bx));
            const float gy = fmaxf(0.f, wy ? fminf(ay, by) : fmaxf(ay, by));
            const float gz = fmaxf(0.f, wz ? fminf(az, bz) : fmaxf(az, bz));
            const bool hit = c >= cb && c < ce && J >= g0 + c &&
                             fmaf(gx, gx, fmaf(gy, gy, gz * gz)) <= a.bb2;
            msk |= hit ? (1u << c) : 0u;
          }
        }
        sg = __shfl_sync(FULL, s, 31);
        unsigned vis = __ballot_sync(FULL, msk != 0u);
        while (vis) {
          const int t0 = __ffs(vis) - 1;
          vis &= vis - 1u;
          const int Jv = __shfl_sync(FULL, J, t0);
          const uint32_t M = __shfl_sync(FULL, msk, t0);
          const int vb = __shfl_sync(FULL, jb, t0), vn = __shfl_sync(FULL, jn, t0);
          const int cdiag = Jv - g0;  // the visited cluster's place in the super-cluster
          // This lane's j particles, h and h + 4 of the cluster: exact integer offsets from the
          // frame centre.
          real qj[2], fxj[2], fyj[2], fzj[2];
          int oxj[2], oyj[2], ozj[2], tj[2], cntj[2];
          bool vj[2];
#pragma unroll
          for (int k = 0; k < 2; ++k) {
            const int t = hh + 4 * k;
            vj[k] = t < vn;
            const int p = vb + (vj[k] ? t : 0);
            oxj[k] = (int)(a.set.sx[p] - rx);
            oyj[k] = (int)(a.set.sy[p] - ry);
            ozj[k] = (int)(a.set.sz[p] - rz);
            qj[k] = COUL ? a.set.qd[p] : 0.0;
            tj[k] = MULTI ? a.set.type[p] : 0;
            fxj[k] = fyj[k] = fzj[k] = (real)0;
            cntj[k] = 0;
          }
          // Pair force of i (integer offsets) with this lane's j particle k, when `ok`; adds the
          // reaction to j and returns the force factor and displacement.
          auto pair_one = [&](bool ok, int oxi_, int oyi_, int ozi_, real qi_, int ti_, int k,
                              real &dx, real &dy, real &dz, bool &in) -> real {
            // the offsets' difference (mod 2^32) is the exact minimum-image displacement
            const int dsx = (int)((uint32_t)oxi_ - (uint32_t)oxj[k]);
            const int dsy = (int)((uint32_t)oyi_ - (uint32_t)oyj[k]);
            const int dsz = (int)((uint32_t)ozi_ - (uint32_t)ozj[k]);
            dx = __dmul_rn((double)dsx, pc.hd[0]);
            dy = __dmul_rn((double)dsy, pc.hd[1]);
            dz = __dmul_rn((double)dsz, pc.hd[2]);
            const real r2 = __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)),
                                      __dmul_rn(dz, dz));
            in = ok && vj[k] && r2 <= pc.rc2d;
            const real ir2 = in ? 1.0 / r2 : 0.0;
            const real g = cp_terms<COUL, MULTI>(a, in, r2, ir2, qi_, qj[k], ti_, tj[k], acc);
            fxj[k] = mad(-g, dx, fxj[k]); fyj[k] = mad(-g, dy, fyj[k]); fzj[k] = mad(-g, dz, fzj[k]);
            if (COUNT) cntj[k] += in ? 1 : 0;
            return g;
          };
          // The visited cluster may be one of the super-cluster's own (cdiag): its pairs with
          // itself count once (particle a8 with particle h + 4k > a8). They are taken here, with
          // the i particle read from shared memory and its force added by atomics, so that the
          // loop below carries no exclusion.
          uint32_t Mh = M;
          if (cdiag >= 0 && cdiag < NC && ((M >> cdiag) & 1u)) {
            Mh &= ~(1u << cdiag);
            const int t = kClSize * cdiag + a8;
            const bool vd = t < np && (asub < 0 || a8 == asub);
            const uint4 sd = si[t];
            const int ox = (int)(sd.x - rx), oy = (int)(sd.y - ry), oz = (int)(sd.z - rz);
            const real qd = COUL && vd ? a.set.qd[p0 + t] : 0.0;
            const int td = MULTI ? sti[t] : 0;
            real fdx = (real)0, fdy = (real)0, fdz = (real)0;
            int cd = 0;
#pragma unroll
            for (int k = 0; k < 2; ++k) {
              real dx, dy, dz;
              bool in;
              const real g = pair_one(vd && a8 < hh + 4 * k, ox, oy, oz, qd, td, k, dx, dy, dz, in);
              fdx = mad(g, dx, fdx); fdy = mad(g, dy, fdy); fdz = mad(g, dz, fdz);
              if (COUNT) cd += in ? 1 : 0;
            }
            fdx += __shfl_xor_sync(FULL, fdx, 8); fdx += __shfl_xor_sync(FULL, fdx, 16);
            fdy += __shfl_xor_sync(FULL, fdy, 8); fdy += __shfl_xor_sync(FULL, fdy, 16);
            fdz += __shfl_xor_sync(FULL, fdz, 8); fdz += __shfl_xor_sync(FULL, fdz, 16);
            if (COUNT) {
              cd += __shfl_xor_sync(FULL, cd, 8);
              cd += __shfl_xor_sync(FULL, cd, 16);
            }
            if (vd && hh < 3) {
              const real v = hh == 0 ? fdx : (hh == 1 ? fdy : fdz);
              fx_add(a.facc + (int64_t)hh * N + p0 + t, v, a.fscale_d, a.err);
            }
            if (COUNT && vd && hh == 3 && cd) atomicAdd(a.nbr + p0 + t, cd);
          }
#pragma unroll
          for (int c = 0; c < NC; ++c) {
            if ((Mh >> c) & 1u) {
#pragma unroll
              for (int k = 0; k < 2; ++k) {
                real dx, dy, dz;
                bool in;
                const real g = pair_one(vi[c], oxi[c], oyi[c], ozi[c], qi[c], ti[c], k, dx, dy, dz, in);
                fxi[c] = mad(g, dx, fxi[c]); fyi[c] = mad(g, dy, fyi[c]); fzi[c] = mad(g, dz, fzi[c]);
                if (COUNT) cnti[c] += in ? 1 : 0;
              }
            }
          }
          // Reaction on the visited cluster, reduce-scattered over the 8 lanes sharing h: of
          // the slots (fx, fy, fz of particle h, then of particle h + 4, then two zeros) lane
          // a8 ends with the sum of slot a8 over the 8 lanes and adds it (slots 0-5). The
          // exchange with lane a8 xor m (m = 1, 2, 4) pairs the slots that differ in bit m: a
          // lane keeps the one whose bit matches its own and adds its partner's copy of it,
          // so each sum is formed as the tree ((v_a + v_a^1) + (v_a^2 + v_a^3)) + (...) of a
          // full butterfly, with a third of its shuffles.
          {
            const bool b0 = a8 & 1, b1 = a8 & 2, b2 = a8 & 4;
            // xor 1: slot pairs (0, 1), (2, 3), (4, 5); w[p] holds slot 2p + b0 ((6, 7): zero)
            real w[3];
            {
              const real s0[3] = {fxj[0], fzj[0], fyj[1]}, s1[3] = {fyj[0], fxj[1], fzj[1]};
#pragma unroll
              for (int p = 0; p < 3; ++p)
                w[p] = (b0 ? s1[p] : s0[p]) + __shfl_xor_sync(FULL, b0 ? s0[p] : s1[p], 1);
            }
            // xor 2: (w0, w1) and (w2, 0); u[q] holds slot 4q + 2 b1 + b0
            const real u0 = (b1 ? w[1] : w[0]) + __shfl_xor_sync(FULL, b1 ? w[0] : w[1], 2);
            const real u1 = (b1 ? (real)0 : w[2]) + __shfl_xor_sync(FULL, b1 ? w[2] : (real)0, 2);
            // xor 4: slot a8
            const real v = (b2 ? u1 : u0) + __shfl_xor_sync(FULL, b2 ? u0 : u1, 4);
            if (a8 < 6) {
              const int k = a8 / 3, d = a8 - 3 * k;
              if (vj[k]) {
                fx_add(a.facc + (int64_t)d * N + vb + hh + 4 * k, v, a.fscale_d, a.err);
              }
            }
          }
          if (COUNT) {
            const unsigned gm = 0xffu << (8 * hh);
            const int c0 = __reduce_add_sync(gm, cntj[0]);
            const int c1 = __reduce_add_sync(gm, cntj[1]);
            if (a8 == 0) {
              if (vj[0] && c0) atomicAdd(a.nbr + vb + hh, c0);
              if (vj[1] && c1) atomicAdd(a.nbr + vb + hh + 4, c1);
            }
          }
        }
      }
      // i forces: sum over the four lanes sharing a8, then lane (h, a8) adds clusters c with
      // c % 4 == h
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        fxi[c] += __shfl_xor_sync(FULL, fxi[c], 8); fxi[c] += __shfl_xor_sync(FULL, fxi[c], 16);
        fyi[c] += __shfl_xor_sync(FULL, fyi[c], 8); fyi[c] += __shfl_xor_sync(FULL, fyi[c], 16);
        fzi[c] += __shfl_xor_sync(FULL, fzi[c], 8); fzi[c] += __shfl_xor_sync(FULL, fzi[c], 16);
        if (COUNT) {
          cnti[c] += __shfl_xor_sync(FULL, cnti[c], 8);
          cnti[c] += __shfl_xor_sync(FULL, cnti[c], 16);
        }
        const int t = kClSize * c + a8;
        if ((c & 3) == hh && vi[c]) {
          const int64_t pi = p0 + t;
          fx_add(a.facc + pi, fxi[c], a.fscale_d, a.err);
          fx_add(a.facc + N + pi, fyi[c], a.fscale_d, a.err);
          fx_add(a.facc + 2 * N + pi, fzi[c], a.fscale_d, a.err);
          if (COUNT && cnti[c]) atomicAdd(a.nbr + pi, cnti[c]);
        }
      }
      __syncwarp();
      if (asub < 0) {
        cb = ce;
      } else if (++asub >= min(kClSize, np - kClSize * cb)) {
        asub = -1;
        ++cb;
      }
    }
  }
  // block partials of the energies and virials (each pair counted once)
  double ulj = acc.u0, wlj = acc.u1;
  if (!MULTI) {
    ulj = a.ljAd * acc.u0 - a.ljBd * acc.u1;
    wlj = 12.0 * a.ljAd * acc.u0 - 6.0 * a.ljBd * acc.u1;
  }
  const double v[NQ_PAIR] = {acc.uc, ulj, acc.wc, wlj};
  const double s = warp_sum4(v, lane);
  if (lane < NQ_PAIR) a.epart[(int64_t)bx * NQ_PAIR + lane] = s;
  // the pass's partial slots past the grid (the range is sized for the per-particle kernel,
  // the grid for the super-clusters) hold zeros
  for (int64_t z = (int64_t)bx + nbx; z < a.nslots; z += nbx)
    if (lane < NQ_PAIR) a.epart[z * NQ_PAIR + lane] = 0.0;
}

template <bool COUL, bool MULTI, bool COUNT>
__global__ void __launch_bounds__(32, COUL ? 8 : 12) cpair64_kernel(const ClusterArgs a) {
  cpair64_body<COUL, MULTI, COUNT>(a, (int)blockIdx.x, (int)gridDim.x);
}

// ---------------------------------------------------------------------------------------
// Host side

int cpair_nc(const Ctx &c) { return c.precision == RBE_FP64 ? 4 : 8; }

// Upper bound of the super-clusters of N particles in the rows of the grid.
static int64_t cpair_super_bound(const Ctx &c) {
  const int64_t nrows = (int64_t)c.grid.n[1] * c.grid.n[2];
  return c.N / (kClSize * cpair_nc(c)) + nrows + 1;
}
// FP32 forms: warps a block (they share the block's start: the super-cluster's particles and
// stencil) and blocks a super-cluster. A super-cluster alone is a chain of some 200 visits, so
// a box with fewer super-clusters than the GPU holds warps (28 an SM, 20 with Coulomb terms)
// leaves SMs idle behind that chain: four warps a block, then as many blocks (at most 8) as
// fill it. With enough super-clusters two warps a block are best: half the starts, and blocks
// short enough for an even end. Pair phase, us, at (warps, blocks):
//   3,000 charged (83 super-clusters):  (1,1) 529, (4,1) 150, (4,2) 86, (4,4) 55, (4,8) 43
//   50,002 charged, two types (1,006):  (1,1) 412, (2,1) 240, (4,1) 141, (4,2) 148, (4,4) 211
//   1,048,576, 10% charged (18,234):    (1,1) 983, (2,1) 957, (4,1) 986, (4,2) 1,137
static void cpair_shape(const Ctx &c, int *warps, int *nsplit) {
  *warps = *nsplit = 1;
  if (c.precision == RBE_FP64) return;
  const int64_t n = cpair_super_bound(c);
  const int64_t fill = (int64_t)c.sms * (c.Nq * 2 > c.N ? kCpWarpsCoul : kCpWarpsLJ);
  *warps = n >= fill ? 2 : kCpMaxWarps;
  *nsplit = (int)std::min<int64_t>(8, std::max<int64_t>(1, fill / (kCpMaxWarps * n)));
}
int64_t cpair_blocks_bound(const Ctx &c) {
  int warps, nsplit;
  cpair_shape(c, &warps, &nsplit);
  return cpair_super_bound(c) * nsplit;
}
int64_t cpair_clusters_bound(const Ctx &c) {
  const int64_t nrows = (int64_t)c.grid.n[1] * c.grid.n[2];
  return c.N / kClSize + nrows + 1;
}

// The cluster kernel applies when a super-cluster's frame is a valid minimum image for y
// and z (one cell width plus 2 r_c below L) and a group of at least one typical cluster
// fits in x, with a stencil of at most 3 cells.
bool cpair_usable(const Ctx &c) {
  if (c.rbl || !c.pair_cluster) return false;
  for (int d = 1; d < 3; ++d) {
    if (c.grid.R[d] > 3) return false;
    const double w = c.box[d] / c.grid.n[d];
    if (!(w + 2.0 * c.rc < c.box[d] * (1.0 - 1e-9))) return false;
  }
  // room in x for at least a few cells' worth of a group
  return c.box[0] - 2.0 * c.rc > 2.0 * c.box[0] / c.grid.n[0];
}

cudaError_t launch_cluster_rows(Ctx &c) {
  const RowsArgs ra{c.cell_start, c.grid.n[0], c.grid.n[1] * c.grid.n[2], cpair_nc(c), c.cl_base,
                    c.sc_base};
  return dispatch(c, cluster_rows_kernel, cluster_rows_kernel_b, dim3(1), dim3(1024), 0, ra);
}

cudaError_t launch_cluster_bounds(Ctx &c) {
  const int b = c.cur;
  const int nrows = c.grid.n[1] * c.grid.n[2];
  const int64_t ccap = cpair_clusters_bound(c);
  const BoundsArgs ba{c.s[b], c.s[b] + c.N, c.s[b] + 2 * c.N, c.qf[b], c.cell_start, c.grid.n[0],
                      nrows, c.cl_base, ccap, c.cl_lo, c.cl_hi, c.cjrec, c.pc.h[1], c.pc.h[2],
                      c.sc_base, cpair_nc(c), c.sc_info};
  return dispatch(c, cluster_bounds_kernel, cluster_bounds_kernel_b,
                  dim3((unsigned)((kClSize * ccap + 255) / 256)), dim3(256), 0, ba);
}

// The pair pass itself (the tables of the two passes above must be current); its forces stay
// in the fixed-point sums, which the Coulomb pass and the k-space gather add to before
// launch_cluster_finish converts them.
cudaError_t launch_cluster_pair(Ctx &c, bool coul, bool multi, bool want_counts) {
  const int b = c.cur;
  const int nrows = c.grid.n[1] * c.grid.n[2];
  ClusterArgs a;
  a.set.sx = c.s[b]; a.set.sy = c.s[b] + c.N; a.set.sz = c.s[b] + 2 * c.N;
  a.set.qf = c.qf[b]; a.set.qd = c.qd[b]; a.set.type = c.type[b];
  a.set.cell_start = c.cell_start; a.set.map = nullptr; a.set.n = c.N;
  a.grid = c.grid;
  a.pc = c.pc;
  a.ljA12 = c.lj.A12[0]; a.ljB6 = c.lj.B6[0];
  a.ljAd = c.lj.Ad[0]; a.ljBd = c.lj.Bd[0]; a.ljA12d = c.lj.A12d[0]; a.ljB6d = c.lj.B6d[0];
  a.table = reinterpret_cast<const LJTable *>(c.lj_dev);
  a.cl_base = c.cl_base; a.sc_base = c.sc_base; a.sc_info = c.sc_info; a.cl_lo = c.cl_lo; a.cl_hi = c.cl_hi;
  a.jrec = c.cjrec;
  a.nrows = nrows;
  a.facc = c.facc;
  a.N = c.N;
  for (int d = 0; d < 2; ++d) a.wfix[d] = ((int64_t)1 << 48) / c.grid.n[d + 1];
  a.fscale = (float)kFixScale32;
  a.fscale_d = kFixScale64;
  a.epart = c.epart + c.off_pair;
  a.nbr = want_counts ? c.nbr : nullptr;
  a.comp = c.precision == RBE_FP32_COMP;
  {
    // x extent of a group: (extent + 2 r_c) < L, in fractional units, with margin
    const double lim = (c.box[0] - 2.0 * c.rc) / c.box[0] * kTwo32 * (1.0 - 1e-7) - 16.0;
    a.xlim = (uint32_t)std::max(0.0, std::min(lim, 4294967295.0));
    // frame coordinates within L/2 on every axis: the exact-decision band for that extent.
    // A j particle's y and z add one more rounding (corner plus offset: within 3u |y| + 4u w
    // for a cell width w, against the 2u |y| the band assumes per coordinate); extents
    // raised by 2 r_c + 2 w cover it, as |y| <= L/2.
    double X[3];
    for (int d = 0; d < 3; ++d) X[d] = 0.5 * c.box[d];
    for (int d = 1; d < 3; ++d) X[d] += 2.0 * c.rc + 2.0 * c.box[d] / c.grid.n[d];
    const double band = frame_band(X, c.rc, c.box, false);
    a.pc.rc2_lo = (float)(c.rc * c.rc * (1.0 - band));
    a.pc.rc2_hi = (float)(c.rc * c.rc * (1.0 + band));
    // band test |r^2 - mid| <= half: half reaches past both FP32 edges by a few ulps (the
    // edges are rounded to FP32; the difference r^2 - mid is exact near mid)
    a.rc2_mid = (float)(c.rc * c.rc);
    const double mid = a.rc2_mid, ulp = std::nextafter((float)mid, 3e38f) - (float)mid;
    a.rc2_half = (float)(std::max((double)a.pc.rc2_hi - mid, mid - (double)a.pc.rc2_lo) + 4.0 * ulp);
    // box test: squared gap of FP32 frame boxes (each bound within 2u L/2, the gap within
    // u L more), widened so that no pair within r_c is lost
    const double u = std::ldexp(1.0, -24);
    double e = 0.0;
    for (int d = 0; d < 3; ++d) e = std::max(e, 3.0 * u * c.box[d]);
    const double rr = c.rc * (1.0 + 1e-5) + 2.0 * e;
    a.bb2 = (float)(rr * rr);
  }
  a.err = c.err;
  if (want_counts) {
    const cudaError_t e = fill_zero(c, c.nbr, c.N);
    if (e != cudaSuccess) return e;
  }
  // a block per possible super-cluster (blocks past the last one, and each block for the
  // slots past the grid, write zeros to the pass's partial range)
  a.nslots = c.n_pair_blk;
  int warps;
  cpair_shape(c, &warps, &a.nsplit);
  const dim3 g((unsigned)cpair_blocks_bound(c)), bl(32, warps);
  const size_t shm = (size_t)warps * 32 * (sizeof(uint4) + sizeof(float));
  const bool fp64 = c.precision == RBE_FP64;
  a.fit = c.fit;
  cudaError_t e;
  // (per replica in a batch)
#define RBE_CP_LAUNCH(CO, MU)                                                               \
  e = want_counts ? dispatch(c, cpair32_kernel<CO, MU, true>, nullptr, g, bl, shm, a, true) \
                  : dispatch(c, cpair32_kernel<CO, MU, false>, nullptr, g, bl, shm, a, true)
#define RBE_CP_LAUNCH64(CO, MU)                                                           \
  e = want_counts ? dispatch(c, cpair64_kernel<CO, MU, true>, nullptr, g, bl, 0, a, true) \
                  : dispatch(c, cpair64_kernel<CO, MU, false>, nullptr, g, bl, 0, a, true)
  if (fp64) {
    if (coul) { if (multi) RBE_CP_LAUNCH64(true, true); else RBE_CP_LAUNCH64(true, false); }
    else { if (multi) RBE_CP_LAUNCH64(false, true); else RBE_CP_LAUNCH64(false, false); }
  } else if (coul && c.fit.ok) {
    if (multi) RBE_CP_LAUNCH(1, true); else RBE_CP_LAUNCH(1, false);
  } else if (coul) {
    if (multi) RBE_CP_LAUNCH(2, true); else RBE_CP_LAUNCH(2, false);
  } else {
    if (multi) RBE_CP_LAUNCH(0, true); else RBE_CP_LAUNCH(0, false);
  }
#undef RBE_CP_LAUNCH64
#undef RBE_CP_LAUNCH
  return e;
}

// F = the fixed-point sums / scale, and the sums cleared for the next step.
cudaError_t launch_cluster_finish(Ctx &c) {
  const bool fp64 = c.precision == RBE_FP64;
  const int64_t n3 = 3 * c.N;
  // (per replica in a batch too: it joins the pair kernel, the Coulomb pass and the gather in
  // one run of per-replica launches, one fork and join per step)
  const int per = (int)std::min<int64_t>(
      512 * kFinishPairs, std::max<int64_t>(512, n3 / ((int64_t)4 * c.sms) / 512 * 512));
  const dim3 fg((unsigned)((n3 + per - 1) / per)), fb(256);
  if (fp64) {
    const FinishArgs f{c.facc, c.Fd, n3, 0.f, 0.f, 1.0 / kFixScale64, per};
    return dispatch(c, cpair_finalize_kernel<double>, cpair_finalize_kernel_b<double>, fg, fb, 0, f,
                    true);
  }
  const FinishArgs f{c.facc, c.F, n3, (float)(4294967296.0 / kFixScale32),
                     (float)(1.0 / kFixScale32), 0.0, per};
  return dispatch(c, cpair_finalize_kernel<float>, cpair_finalize_kernel_b<float>, fg, fb, 0, f,
                  true);
}

}  // namespace rbe
