// k_integrate.cu -- velocity Verlet on the fixed-point grid, energy totals, and the
// gathers that translate between cell-sorted storage and caller id order.
//
// Velocity Verlet (the time integrator of Sec. 2.1):
//   v += (F/m)(dt/2) kappa;  s += rint(v dt 2^32 / L)  (FP64 increment, wraps mod 2^32)
//   ... forces at the new positions ...;  v += (F/m)(dt/2) kappa
// Every kernel here is a single streaming pass (HBM-bound) except the totals, which sum
// the per-block partials of all force kernels in a fixed order (latency-bound).
#include <cmath>

#include "rbe_internal.cuh"

namespace rbe {

int64_t rbl_compact_count(int64_t nblk);

// g_d = dt 2^32 / L_d (FP64, from the host): the fixed-point increment is rint(v g_d), in
// FP64 in the FP64 form. The FP32 forms round the FP32 product (off by at most one grid unit
// of L / 2^32 where the FP64 rounding would differ); FP64 runs at 1/64 of the FP32 rate on
// this GPU, and this pass would otherwise be bound by it instead of by memory.
template <typename V, typename FT>
struct KickDriftArgs {
  V *v;
  const FT *F;
  const float *invm;
  uint32_t *s;
  int64_t N;
  double hdk, gx, gy, gz;
  int *err;
  const double *scale;
  uint64_t *step;  // the step counter, advanced by the first thread (the sampler reads it next)
};

// Solo and batched kernels of a body templated on the velocity and force types.
#define RBE_VF_KERNELS(LB, NAME, ARGS, BODY)                                                   \
  template <typename V, typename FT>                                                         \
  __global__ void LB NAME(const ARGS<V, FT> a) {                                              \
    BODY<V, FT>(a, (int)blockIdx.x, (int)gridDim.x);                                          \
  }                                                                                          \
  template <typename V, typename FT>                                                         \
  __global__ void LB NAME##_b(const ARGS<V, FT> *__restrict__ t,                              \
                              const int32_t *__restrict__ pre, int nrep) {                    \
    const BatchIdx q = batch_locate(pre, nrep);                                               \
    BODY<V, FT>(t[q.r], q.bx, q.nbx);                                                         \
  }

template <typename V, typename FT>
__device__ __forceinline__ void kick_drift_body(const KickDriftArgs<V, FT> &a, int bx, int) {
  const int64_t i = (int64_t)bx * blockDim.x + threadIdx.x;
  const int64_t N = a.N;
  if (i == 0) *a.step += 1;
  if (i >= N) return;
  V *__restrict__ v = a.v;
  const FT *__restrict__ F = a.F;
  uint32_t *__restrict__ s = a.s;
  const double *scale = a.scale;
  const double hdk = a.hdk;
  const double g[3] = {a.gx, a.gy, a.gz};
  const float *__restrict__ invm = a.invm;
  const V im = (V)invm[i];
  const V sc = scale ? (V)*scale : (V)1;  // Nose-Hoover start-of-step scaling
  bool bad = false;
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    V vv = v[d * N + i] * sc + (V)F[d * N + i] * im * (V)hdk;
    v[d * N + i] = vv;
    int st;
    if (sizeof(V) == 8) {
      const double inc = (double)vv * g[d];
      bad |= !isfinite(inc) || fabs(inc) > 2.0e9;
      st = bad ? 0 : __double2int_rn(inc);
    } else {
      const float inc = (float)vv * (float)g[d];
      bad |= !isfinite(inc) || fabsf(inc) > 2.0e9f;
      st = bad ? 0 : __float2int_rn(inc);
    }
    s[d * N + i] += (uint32_t)st;
  }
  if (bad) atomicOr(a.err, ERRBIT_NONFINITE);
}
RBE_VF_KERNELS(__launch_bounds__(256), kick_drift_kernel, KickDriftArgs, kick_drift_body)

// The FP32 forms with N a multiple of 4: four consecutive particles a thread in 16-byte
// accesses (the arrays start 256-byte aligned, and d N keeps each axis block aligned), each
// with kick_drift_body's arithmetic in the same order.
__device__ __forceinline__ void kick_drift4_body(const KickDriftArgs<float, float> &a, int bx, int) {
  const int64_t q = (int64_t)bx * blockDim.x + threadIdx.x;
  const int64_t N = a.N;
  if (q == 0) *a.step += 1;
  const int64_t i = 4 * q;
  if (i >= N) return;
  const float4 im = *reinterpret_cast<const float4 *>(a.invm + i);
  const float sc = a.scale ? (float)*a.scale : 1.f;  // Nose-Hoover start-of-step scaling
  const float hdk = (float)a.hdk;
  const double g[3] = {a.gx, a.gy, a.gz};
  bool bad0 = false, bad1 = false, bad2 = false, bad3 = false;
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    float4 *vp = reinterpret_cast<float4 *>(a.v + d * N + i);
    uint4 *sp = reinterpret_cast<uint4 *>(a.s + d * N + i);
    float4 v = *vp;
    const float4 f = *reinterpret_cast<const float4 *>(a.F + d * N + i);
    uint4 sv = *sp;
    const float gd = (float)g[d];
    auto one = [&](float &vv, float ff, float imm, uint32_t &ss, bool &bad) {
      vv = vv * sc + ff * imm * hdk;
      const float inc = vv * gd;
      bad |= !isfinite(inc) || fabsf(inc) > 2.0e9f;
      const int st = bad ? 0 : __float2int_rn(inc);
      ss += (uint32_t)st;
    };
    one(v.x, f.x, im.x, sv.x, bad0);
    one(v.y, f.y, im.y, sv.y, bad1);
    one(v.z, f.z, im.z, sv.z, bad2);
    one(v.w, f.w, im.w, sv.w, bad3);
    *vp = v;
    *sp = sv;
  }
  if (bad0 || bad1 || bad2 || bad3) atomicOr(a.err, ERRBIT_NONFINITE);
}
using KickDriftArgsF = KickDriftArgs<float, float>;
RBE_BATCHED_KERNEL(__launch_bounds__(256), kick_drift4_kernel, KickDriftArgsF, kick_drift4_body)

template <typename V, typename FT>
struct KickArgs {
  V *v;
  const FT *F;
  const float *invm;
  int64_t N;
  double hdk, inv_kappa;
  int do_kick;
  double *ke_part;
};

// Particles a block of the kick kernels, four consecutive ones a thread. The kinetic energy's terms
// are summed in FP64: a thread's four, then the warp's, then the warps' in order, the same in the
// scalar and the 16-byte kernel, so their partials agree bit for bit. (One particle a thread and
// a 256-term tree left the pass waiting on memory and barriers: the kinetic energy of 4,000,001
// particles by the scalar kernel 76 -> 30 us, and the totals over a quarter of the partials
// 30 -> 14 us.)
constexpr int kKickThreads = 256;

__device__ __forceinline__ void kick_reduce(const double (&ke)[4], double *out) {
  __shared__ double sh[kKickThreads / 32];
  const double s = warp_sum((ke[0] + ke[1]) + (ke[2] + ke[3]));
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < kKickThreads / 32; ++w) t += sh[w];
    *out = t;
  }
}

template <typename V, typename FT>
__device__ __forceinline__ void kick_body(const KickArgs<V, FT> &a, int bx, int) {
  V *__restrict__ v = a.v;
  const FT *__restrict__ F = a.F;
  const float *__restrict__ invm = a.invm;
  const int64_t N = a.N;
  const int64_t i0 = 4 * ((int64_t)bx * kKickThreads + threadIdx.x);
  V vv[4][3];
  float im[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const int64_t i = min(i0 + j, N - 1);
    im[j] = invm[i];
#pragma unroll
    for (int d = 0; d < 3; ++d) vv[j][d] = v[d * N + i];
  }
  if (a.do_kick) {
    FT f[4][3];
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int d = 0; d < 3; ++d) f[j][d] = F[d * N + min(i0 + j, N - 1)];
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        vv[j][d] += (V)f[j][d] * (V)im[j] * (V)a.hdk;
        if (i0 + j < N) v[d * N + i0 + j] = vv[j][d];
      }
  }
  double ke[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    V v2 = (V)0;
#pragma unroll
    for (int d = 0; d < 3; ++d) v2 += vv[j][d] * vv[j][d];
    // 1/2 m v^2 / kappa, m = 1 / (1/m): FP64 in the FP64 form; the FP32 forms form each
    // particle's term in FP32 and sum the terms in FP64
    if (i0 + j >= N) ke[j] = 0.0;
    else if (sizeof(V) == 8) ke[j] = 0.5 * (double)v2 / (double)im[j] * a.inv_kappa;
    else ke[j] = f2d(0.5f * (float)v2 * __frcp_rn(im[j]) * (float)a.inv_kappa);
  }
  kick_reduce(ke, a.ke_part + bx);
}
RBE_VF_KERNELS(__launch_bounds__(kKickThreads), kick_kernel, KickArgs, kick_body)

// The FP32 forms with N a multiple of 4: the same in 16-byte accesses.
__device__ __forceinline__ void kick4_body(const KickArgs<float, float> &a, int bx, int) {
  const int64_t N = a.N;
  const int64_t i = 4 * ((int64_t)bx * kKickThreads + threadIdx.x);
  const float hdk = (float)a.hdk, ik = (float)a.inv_kappa;
  double ke[4] = {0.0, 0.0, 0.0, 0.0};
  if (i < N) {  // (all four, N being a multiple of 4)
    const float4 im = *reinterpret_cast<const float4 *>(a.invm + i);
    float v2[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      float4 *vp = reinterpret_cast<float4 *>(a.v + d * N + i);
      float4 vv = *vp;
      if (a.do_kick) {
        const float4 f = *reinterpret_cast<const float4 *>(a.F + d * N + i);
        vv.x += f.x * im.x * hdk;
        vv.y += f.y * im.y * hdk;
        vv.z += f.z * im.z * hdk;
        vv.w += f.w * im.w * hdk;
        *vp = vv;
      }
      v2[0] += vv.x * vv.x;
      v2[1] += vv.y * vv.y;
      v2[2] += vv.z * vv.z;
      v2[3] += vv.w * vv.w;
    }
    ke[0] = f2d(0.5f * v2[0] * __frcp_rn(im.x) * ik);
    ke[1] = f2d(0.5f * v2[1] * __frcp_rn(im.y) * ik);
    ke[2] = f2d(0.5f * v2[2] * __frcp_rn(im.z) * ik);
    ke[3] = f2d(0.5f * v2[3] * __frcp_rn(im.w) * ik);
  }
  kick_reduce(ke, a.ke_part + bx);
}
using KickArgsF = KickArgs<float, float>;
RBE_BATCHED_KERNEL(__launch_bounds__(kKickThreads), kick4_kernel, KickArgsF, kick4_body)

// Nose-Hoover half steps (chain of one): from 2K = 2 sum(kinetic partials) the end-of-step
// half (mode 0) gives the velocity scale s_end and the start-of-next-step half gives
// s_start, applied by the next kick-drift; mode 1 only does the start half (first step).
struct ThermoArgs {
  const double *ke_part;
  int64_t n;
  double Nf, kT, Q, dt;
  double *th;
  int mode;
  double *ke;  // mode 0: the step's kinetic energy
};

__device__ __forceinline__ void thermostat_body(const ThermoArgs &a, int, int) {
  __shared__ double sh[8];
  const double *__restrict__ ke_part = a.ke_part;
  const int64_t n = a.n;
  const double Nf = a.Nf, kT = a.kT, Q = a.Q, dt = a.dt;
  double *__restrict__ th = a.th;
  const int mode = a.mode;
  double acc = 0.0;
#pragma unroll 4
  for (int64_t b = threadIdx.x; b < n; b += blockDim.x) acc += ke_part[b];
  acc = warp_sum(acc);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x != 0) return;
  double K2 = 2.0 * (((sh[0] + sh[1]) + (sh[2] + sh[3])) + ((sh[4] + sh[5]) + (sh[6] + sh[7])));
  double xi = th[0], eta = th[1], s_end = 1.0;
  if (mode == 0) {
    xi += 0.25 * dt * (K2 - Nf * kT) / Q;
    s_end = exp(-xi * 0.5 * dt);
    K2 *= s_end * s_end;
    eta += xi * 0.5 * dt;
    xi += 0.25 * dt * (K2 - Nf * kT) / Q;
  }
  th[3] = 0.5 * K2;
  if (mode == 0) *a.ke = 0.5 * K2;
  th[4] = s_end;
  th[5] = xi;   // state at the end of the step (reported)
  th[6] = eta;
  xi += 0.25 * dt * (K2 - Nf * kT) / Q;
  const double s_start = exp(-xi * 0.5 * dt);
  K2 *= s_start * s_start;
  eta += xi * 0.5 * dt;
  xi += 0.25 * dt * (K2 - Nf * kT) / Q;
  th[0] = xi;
  th[1] = eta;
  th[2] = s_start;
}
RBE_BATCHED_KERNEL(__launch_bounds__(256), thermostat_kernel, ThermoArgs, thermostat_body)

template <typename V, typename FT>
struct ScaleArgs {
  V *v;
  int64_t N;
  const double *scale;
};
template <typename V, typename FT>
__device__ __forceinline__ void scale_v_body(const ScaleArgs<V, FT> &a, int bx, int) {
  const int64_t k = (int64_t)bx * blockDim.x + threadIdx.x;
  if (k >= 3 * a.N) return;
  a.v[k] *= (V)*a.scale;
}
RBE_VF_KERNELS(__launch_bounds__(256), scale_v_kernel, ScaleArgs, scale_v_body)

struct TotalsArgs {
  const double *ke_override;
  const double *pair, *coul, *rbl, *ke, *emode;
  int64_t n_pair, n_coul, n_rbl, n_ke;
  int P;
  double U_self;
  double *scal;
  int parts;  // 1: energies and virials, 2: kinetic energy
};

// Fixed-order reduction of every partial into the scalars (ACC = float for the plain
// FP32 form, double otherwise). One block of kTotalsThreads: strided per-thread sums (four
// partials in flight per thread), then warp shuffles, then the warp sums in order. Four
// warps: the warp reductions of the FP64 sums dominate on one SM (FP64 runs at 1/64 of the FP32
// rate), and they scale with the warps, the strided sums do not. (Seven sums as a list, 9 additions a
// warp instead of 35, and the kinetic energy apart from the rest, on the step's other branch:
// a step of 3,000 charged particles 74 -> 71 us, of 100,000 ions with a Verlet list 85 -> 79.)
constexpr int kTotalsThreads = 128;
constexpr int64_t kTotalsDirect = 1024;  // partials of a pass it reads without a compaction

template <typename ACC>
__device__ __forceinline__ void totals_body(const TotalsArgs &a, int, int) {
  constexpr int NV = 8;  // ureal ulj wreal wlj uk wk ke, none
  constexpr int NW = kTotalsThreads / 32;
  __shared__ ACC sh[NV][NW];
  ACC acc[NV];
  for (int k = 0; k < NV; ++k) acc[k] = (ACC)0;
  const double *srcs[3] = {a.pair, a.coul, a.rbl};
  const bool en = a.parts & 1, kin = a.parts & 2;
  const int64_t ns[3] = {en ? a.n_pair : 0, en ? a.n_coul : 0, en ? a.n_rbl : 0};
  const int64_t n_ke = kin ? a.n_ke : 0;
  for (int r = 0; r < 3; ++r) {
#pragma unroll 4
    for (int64_t b = threadIdx.x; b < ns[r]; b += blockDim.x)
      for (int k = 0; k < NQ_PAIR; ++k) acc[k] += (ACC)srcs[r][b * NQ_PAIR + k];
  }
  for (int l = threadIdx.x; l < (en ? a.P : 0); l += blockDim.x) {
    acc[4] += (ACC)a.emode[2 * l];
    acc[5] += (ACC)a.emode[2 * l + 1];
  }
#pragma unroll 4
  for (int64_t b = threadIdx.x; b < n_ke; b += blockDim.x) acc[6] += (ACC)a.ke[b];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const ACC v = warp_sum8(acc, lane);
  if (lane < NV) sh[lane][wid] = v;
  __syncthreads();
  if (threadIdx.x < NV) {
    ACC t = (ACC)0;
    for (int w = 0; w < NW; ++w) t += sh[threadIdx.x][w];
    sh[threadIdx.x][0] = t;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    const double ur = (double)sh[Q_UREAL][0], ul = (double)sh[Q_ULJ][0];
    const double wr = (double)sh[Q_WREAL][0], wl = (double)sh[Q_WLJ][0];
    const double uk = (double)sh[4][0], wk = (double)sh[5][0];
    if (kin) a.scal[S_KE] = a.ke_override ? *a.ke_override : (double)sh[6][0];
    if (!en) return;
    a.scal[S_UREAL] = ur;
    a.scal[S_ULJ] = ul;
    a.scal[S_UK] = uk;
    a.scal[S_USELF] = a.U_self;
    a.scal[S_UTOT] = ur + ul + uk - a.U_self;
    a.scal[S_WREAL] = wr;
    a.scal[S_WLJ] = wl;
    a.scal[S_WK] = wk;
    a.scal[S_WTOT] = wr + wl + wk;
  }
}
template <typename ACC>
__global__ void __launch_bounds__(kTotalsThreads) totals_kernel(const TotalsArgs a) {
  totals_body<ACC>(a, (int)blockIdx.x, (int)gridDim.x);
}
template <typename ACC>
__global__ void __launch_bounds__(kTotalsThreads)
    totals_kernel_b(const TotalsArgs *__restrict__ t, const int32_t *__restrict__ pre, int nrep) {
  const BatchIdx q = batch_locate(pre, nrep);
  totals_body<ACC>(t[q.r], q.bx, q.nbx);
}

// Results in particle order, in device or pinned host memory; err_out and scal_out (nullable, pinned):
// the error flags and the totals, for the host that waits for the results (a copy less: an evaluation
// of 3,000 particles 113 -> 108 us, of 50,002 237 -> 231).
template <typename FT, typename OT>
__global__ void scatter_forces_kernel(const FT *__restrict__ F, const int32_t *__restrict__ id,
                                      int64_t N, OT *__restrict__ out, const int *err,
                                      int *err_out, const double *scal, double *scal_out) {
  const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k == 0 && err_out) *err_out = *err;
  if (k < S_COUNT && scal_out) scal_out[k] = scal[k];
  if (k >= N) return;
  const int64_t o = (int64_t)id[k] * 3;
  out[o] = (OT)F[k];
  out[o + 1] = (OT)F[N + k];
  out[o + 2] = (OT)F[2 * N + k];
}

template <typename V>
__global__ void scatter_state_kernel(const uint32_t *__restrict__ s, const V *__restrict__ v,
                                     const int32_t *__restrict__ id, int64_t N, double hx,
                                     double hy, double hz, double *pos, double *vel, uint32_t *frac,
                                     const int *err, int *err_out) {
  const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k == 0 && err_out) *err_out = *err;
  if (k >= N) return;
  const int64_t o = (int64_t)id[k] * 3;
  const uint32_t x = s[k], y = s[N + k], z = s[2 * N + k];
  if (pos) {
    pos[o] = (double)x * hx;
    pos[o + 1] = (double)y * hy;
    pos[o + 2] = (double)z * hz;
  }
  if (vel) {
    vel[o] = (double)v[k];
    vel[o + 1] = (double)v[N + k];
    vel[o + 2] = (double)v[2 * N + k];
  }
  if (frac) {
    frac[o] = x;
    frac[o + 1] = y;
    frac[o + 2] = z;
  }
}

// A position's fractional coordinate s = rint(fl(r / L) 2^32) mod 2^32 (fl: rounded to double).
// For 0 <= r < L it is formed in integers, since FP64 runs at 1/64 of the FP32 rate: with r = M
// 2^(e - 63) (M the 64-bit left-aligned significand) and K = floor(2^sh / L) in [2^63, 2^64), the
// high half of M K shifted right by n = sh - 64 - e is r / L in 2^-63 units, short by less than 4.
// fl moves the quotient by at most 2^10 of those units, so s rounds as in the FP64 expression
// unless the fraction of s (31 bits) is within 2^12 of one half: those (one in 260,000) and all
// other positions take that expression. The pass is bound by its 144 MB at 4,000,001 particles (309 us
// with the FP64 expression throughout, 32 us so; a divide is some 20 FP64 instructions).
__device__ __forceinline__ uint32_t quantise_f64(double r, double L) {
  const double f = __dmul_rn(__ddiv_rn(r, L), kTwo32);
  const double fm = f - kTwo32 * floor(f / kTwo32);  // wrap into [0, 2^32)
  return (uint32_t)(unsigned long long)__double2ll_rn(fm);
}
__device__ __forceinline__ uint32_t quantise_pos(double r, double L, unsigned long long K, int sh) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(r);
  if (b == 0ull) return 0u;
  const int e = (int)(b >> 52) - 1023;  // (a negative r: e >= 1025)
  const int n = sh - 64 - e;
  if (n < 0 || n > 63 || e < -1000) return quantise_f64(r, L);
  const unsigned long long M = (b << 11) | 0x8000000000000000ull;
  const unsigned long long F = __umul64hi(M, K) >> n;  // (2^63 and more: r >= L)
  const uint32_t frac = (uint32_t)F & 0x7fffffffu;
  if ((F >> 63) || frac - 0x3ffff000u < 0x2000u) return quantise_f64(r, L);
  return (uint32_t)(F >> 31) + (frac >> 30);
}

struct PosScale {
  double L[3];
  unsigned long long K[3];
  int sh[3];
};
__global__ void __launch_bounds__(256)
    set_positions_kernel(const double *__restrict__ pos, const int32_t *__restrict__ id, int64_t N,
                         const PosScale p, uint32_t *__restrict__ s) {
  const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= N) return;
  const int64_t o = (int64_t)id[k] * 3;
  const double r[3] = {pos[o], pos[o + 1], pos[o + 2]};
#pragma unroll
  for (int d = 0; d < 3; ++d) s[d * N + k] = quantise_pos(r[d], p.L[d], p.K[d], p.sh[d]);
}

// Checkpoint load: state given in id order (row-major per particle) into the sorted slots.
template <typename V>
__global__ void gather_state_kernel(const uint32_t *__restrict__ s_id, const double *__restrict__ v_id,
                                    const int32_t *__restrict__ id, int64_t N,
                                    uint32_t *__restrict__ s, V *__restrict__ v) {
  const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= N) return;
  const int64_t o = (int64_t)id[k] * 3;
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    s[d * N + k] = s_id[o + d];
    v[d * N + k] = (V)v_id[o + d];
  }
}

__global__ void scatter_int_kernel(const int32_t *__restrict__ src, const int32_t *__restrict__ id,
                                   int64_t N, int width, int32_t *__restrict__ dst) {
  const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= N) return;
  const int64_t o = (int64_t)id[k] * width;
  for (int w = 0; w < width; ++w) dst[o + w] = src[k * width + w];
}

static inline unsigned nblk(int64_t n, int t) { return (unsigned)((n + t - 1) / t); }

// First half-kick and drift, with the step counter's advance (alone when there are no
// particles).
cudaError_t launch_kick_drift(Ctx &c) {
  const int b = c.cur;
  const double hdk = 0.5 * c.dt * c.kappa;
  if (c.N == 0) return launch_step_advance(c);
  const double *scale = c.nvt ? c.thermo + 2 : nullptr;
  const double gx = c.dt * kTwo32 / c.box[0], gy = c.dt * kTwo32 / c.box[1],
               gz = c.dt * kTwo32 / c.box[2];
  const dim3 g(nblk(c.N, 256)), t(256);
  if (c.precision == RBE_FP64) {
    const KickDriftArgs<double, double> a{c.vd[b], c.Fd, c.invm[b], c.s[b], c.N, hdk, gx, gy, gz,
                                          c.err, scale, c.step_dev};
    return dispatch(c, kick_drift_kernel<double, double>, kick_drift_kernel_b<double, double>, g,
                    t, 0, a);
  }
  const KickDriftArgs<float, float> a{c.vf[b], c.F, c.invm[b], c.s[b], c.N, hdk, gx, gy, gz,
                                      c.err, scale, c.step_dev};
  // (a batch keeps the one-particle kernel: the same results, and replicas of any N share a
  //  class)
  if (c.N % 4 == 0 && !c.rec)
    return dispatch(c, kick_drift4_kernel, kick_drift4_kernel_b, dim3(nblk(c.N / 4, 256)), t, 0,
                    a);
  return dispatch(c, kick_drift_kernel<float, float>, kick_drift_kernel_b<float, float>, g, t, 0,
                  a);
}

cudaError_t launch_thermostat(Ctx &c, int mode) {
  const int b = c.cur;
  const ThermoArgs ta{c.epart + c.off_ke, c.n_ke_blk, c.Nf, c.kB * c.T0, c.Qnh, c.dt, c.thermo,
                      mode, c.scal + S_KE};
  cudaError_t e = dispatch(c, thermostat_kernel, thermostat_kernel_b, dim3(1), dim3(256), 0, ta);
  if (e != cudaSuccess || mode != 0) return e;
  const dim3 g(nblk(3 * c.N, 256)), t(256);
  if (c.precision == RBE_FP64) {
    const ScaleArgs<double, double> a{c.vd[b], c.N, c.thermo + 4};
    return dispatch(c, scale_v_kernel<double, double>, scale_v_kernel_b<double, double>, g, t, 0, a);
  }
  const ScaleArgs<float, float> a{c.vf[b], c.N, c.thermo + 4};
  return dispatch(c, scale_v_kernel<float, float>, scale_v_kernel_b<float, float>, g, t, 0, a);
}

static cudaError_t kick_impl(Ctx &c, int do_kick) {
  const int b = c.cur;
  const double hdk = 0.5 * c.dt * c.kappa;
  if (c.N == 0) return cudaSuccess;
  const dim3 g(nblk(c.N, 4 * kKickThreads)), t(kKickThreads);
  if (c.precision == RBE_FP64) {
    const KickArgs<double, double> a{c.vd[b], c.Fd, c.invm[b], c.N, hdk, 1.0 / c.kappa, do_kick,
                                     c.epart + c.off_ke};
    return dispatch(c, kick_kernel<double, double>, kick_kernel_b<double, double>, g, t, 0, a);
  }
  const KickArgs<float, float> a{c.vf[b], c.F, c.invm[b], c.N, hdk, 1.0 / c.kappa, do_kick,
                                 c.epart + c.off_ke};
  // (a batch keeps the scalar accesses, four particles a thread as here: the same results, and
  //  replicas of any N share a class)
  if (c.N % 4 == 0 && !c.rec) return dispatch(c, kick4_kernel, kick4_kernel_b, g, t, 0, a);
  return dispatch(c, kick_kernel<float, float>, kick_kernel_b<float, float>, g, t, 0, a);
}

cudaError_t launch_kick(Ctx &c) { return kick_impl(c, 1); }
cudaError_t launch_kinetic(Ctx &c) { return kick_impl(c, 0); }

// Block partials of a pair pass ([nblk][NQ_PAIR]) summed over fixed contiguous ranges in a
// fixed order into [gridDim.x][NQ_PAIR]: the FP64 adds are spread over many SMs (one SM's
// FP64 rate is low) before the one-block totals.
struct CompactArgs {       // two passes' partials: blocks [0, nc0) the first, the rest the second
  const double *in[2];
  int64_t nblk[2], per[2];
  double *out[2];
  int nc0;
};

__device__ __forceinline__ void partials_compact_body(const CompactArgs &a, int bx, int) {
  __shared__ double sh[NQ_PAIR][8];
  const int w = bx >= a.nc0 ? 1 : 0;
  if (w) bx -= a.nc0;
  const double *__restrict__ in = a.in[w];
  const int64_t nblk = a.nblk[w], per = a.per[w];
  const int64_t b0 = (int64_t)bx * per, b1 = min(nblk, b0 + per);
  double acc[NQ_PAIR];
#pragma unroll
  for (int k = 0; k < NQ_PAIR; ++k) acc[k] = 0.0;
  for (int64_t b = b0 + threadIdx.x; b < b1; b += blockDim.x)
#pragma unroll
    for (int k = 0; k < NQ_PAIR; ++k) acc[k] += in[b * NQ_PAIR + k];
  const int lane = threadIdx.x & 31;
  const double v[8] = {acc[0], acc[1], acc[2], acc[3], 0.0, 0.0, 0.0, 0.0};
  const double s = warp_sum8(v, lane);
  if (lane < NQ_PAIR) sh[lane][threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x < NQ_PAIR) {
    double t = 0.0;
    for (int k = 0; k < 8; ++k) t += sh[threadIdx.x][k];
    a.out[w][(int64_t)bx * NQ_PAIR + threadIdx.x] = t;
  }
}
RBE_BATCHED_KERNEL(__launch_bounds__(256), partials_compact_kernel, CompactArgs,
                   partials_compact_body)

// Blocks of the compaction of nblk partials (0: few enough for the totals to read themselves);
// one for each 256 partials, at most kCompactMax.
int64_t partials_compact_count(int64_t nblk) {
  return nblk <= kTotalsDirect ? 0 : std::min<int64_t>((nblk + 255) / 256, kCompactMax);
}

// Pair and Coulomb-pass partials, compacted where there are many, by one launch for both (recorded
// without blocks too, so that boxes of any size share a batch's class).
cudaError_t launch_totals_compact(Ctx &c) {
  const int64_t n[2] = {c.n_pair_blk, c.n_coul_blk};
  const double *part[2] = {c.epart + c.off_pair, c.epart + c.off_coul};
  const int64_t nc[2] = {partials_compact_count(n[0]), partials_compact_count(n[1])};
  CompactArgs ca{};
  for (int w = 0; w < 2; ++w) {
    ca.in[w] = part[w];
    ca.nblk[w] = n[w];
    ca.per[w] = nc[w] ? (n[w] + nc[w] - 1) / nc[w] : 0;
    ca.out[w] = c.ecomp + w * kCompactMax * NQ_PAIR;
  }
  ca.nc0 = (int)nc[0];
  return dispatch(c, partials_compact_kernel, partials_compact_kernel_b,
                  dim3((unsigned)(nc[0] + nc[1])), dim3(256), 0, ca);
}

// The totals; the pair passes' partials must be compacted.
cudaError_t launch_totals(Ctx &c, int parts) {
  TotalsArgs a;
  const int64_t n[2] = {c.n_pair_blk, c.n_coul_blk};
  const double *part[2] = {c.epart + c.off_pair, c.epart + c.off_coul};
  const int64_t nc[2] = {partials_compact_count(n[0]), partials_compact_count(n[1])};
  a.pair = nc[0] ? c.ecomp : part[0]; a.n_pair = nc[0] ? nc[0] : n[0];
  a.coul = nc[1] ? c.ecomp + kCompactMax * NQ_PAIR : part[1]; a.n_coul = nc[1] ? nc[1] : n[1];
  // RBL partials: the compacted ones (rbl_compact_kernel runs after the RBL kernel)
  a.rbl = c.rbl ? c.rbl_cpart : c.epart + c.off_rbl;
  a.n_rbl = c.rbl ? rbl_compact_count(c.n_rbl_blk) : 0;
  a.ke = c.epart + c.off_ke; a.n_ke = c.n_ke_blk;
  a.emode = c.emode; a.P = c.P;
  a.U_self = c.U_self;
  a.scal = c.scal;
  a.parts = parts;
  a.ke_override = c.nvt ? c.thermo + 3 : nullptr;
  if (c.precision == RBE_FP32)
    return dispatch(c, totals_kernel<float>, totals_kernel_b<float>, dim3(1), dim3(kTotalsThreads),
                    0, a);
  return dispatch(c, totals_kernel<double>, totals_kernel_b<double>, dim3(1),
                  dim3(kTotalsThreads), 0, a);
}

cudaError_t launch_scatter_forces(Ctx &c, bool to_double, float *outf, int *err_out,
                                  double *scal_out) {
  const int b = c.cur;
  if (c.N == 0) return cudaSuccess;
  if (!outf) outf = c.outf;
  const unsigned g = nblk(c.N, 256);
  const int32_t *id = c.id[b];
  if (c.precision == RBE_FP64) {
    if (to_double) scatter_forces_kernel<double, double><<<g, 256, 0, c.stream>>>(c.Fd, id, c.N, c.outd, c.err, err_out, c.scal, scal_out);
    else scatter_forces_kernel<double, float><<<g, 256, 0, c.stream>>>(c.Fd, id, c.N, outf, c.err, err_out, c.scal, scal_out);
  } else {
    if (to_double) scatter_forces_kernel<float, double><<<g, 256, 0, c.stream>>>(c.F, id, c.N, c.outd, c.err, err_out, c.scal, scal_out);
    else scatter_forces_kernel<float, float><<<g, 256, 0, c.stream>>>(c.F, id, c.N, outf, c.err, err_out, c.scal, scal_out);
  }
  return cudaGetLastError();
}

cudaError_t launch_scatter_state(Ctx &c, double *pos, double *vel, uint32_t *frac, int *err_out) {
  const int b = c.cur;
  if (c.N == 0) return cudaSuccess;
  const double hx = c.box[0] / kTwo32, hy = c.box[1] / kTwo32, hz = c.box[2] / kTwo32;
  const unsigned g = nblk(c.N, 256);
  if (c.precision == RBE_FP64)
    scatter_state_kernel<double><<<g, 256, 0, c.stream>>>(c.s[b], c.vd[b], c.id[b], c.N, hx, hy, hz, pos, vel, frac, c.err, err_out);
  else
    scatter_state_kernel<float><<<g, 256, 0, c.stream>>>(c.s[b], c.vf[b], c.id[b], c.N, hx, hy, hz, pos, vel, frac, c.err, err_out);
  return cudaGetLastError();
}

// K = floor(2^sh / L) in [2^63, 2^64) by long division of powers of two by L's significand.
static unsigned long long inverse_bits(double L, int *sh) {
  int e = 0;
  const double m = std::frexp(L, &e);                              // L = m 2^e, m in [1/2, 1)
  const unsigned long long D = (unsigned long long)std::ldexp(m, 53);  // L = D 2^(e - 53)
  // K = floor(2^k / D), k the largest with K < 2^64: k = 116 (D in [2^52, 2^53)), or 115 for a
  // power of two (2^116 / 2^52 = 2^64)
  const int k = D == (1ull << 52) ? 115 : 116;
  unsigned long long q = 0, r = 0;
  for (int i = k; i >= 0; --i) {
    r = 2 * r + (i == k ? 1ull : 0ull);
    q = 2 * q + (r >= D ? 1ull : 0ull);
    if (r >= D) r -= D;
  }
  *sh = k + e - 53;  // 1 / L = 2^(53 - e) / D
  return q;
}

cudaError_t launch_set_positions(Ctx &c, const double *pos) {
  const int b = c.cur;
  if (c.N == 0) return cudaSuccess;
  PosScale p;
  for (int d = 0; d < 3; ++d) {
    p.L[d] = c.box[d];
    p.K[d] = inverse_bits(c.box[d], &p.sh[d]);
  }
  set_positions_kernel<<<nblk(c.N, 256), 256, 0, c.stream>>>(pos, c.id[b], c.N, p, c.s[b]);
  return cudaGetLastError();
}

cudaError_t launch_gather_state(Ctx &c, const uint32_t *s_id, const double *v_id) {
  const int b = c.cur;
  if (c.N == 0) return cudaSuccess;
  if (c.precision == RBE_FP64)
    gather_state_kernel<double><<<nblk(c.N, 256), 256, 0, c.stream>>>(s_id, v_id, c.id[b], c.N, c.s[b], c.vd[b]);
  else
    gather_state_kernel<float><<<nblk(c.N, 256), 256, 0, c.stream>>>(s_id, v_id, c.id[b], c.N, c.s[b], c.vf[b]);
  return cudaGetLastError();
}

void zero_partials_tail(Ctx &c, int64_t off, int64_t written, int64_t capacity) {
  if (written >= capacity) return;
  fill_zero(c, c.epart + off + written * NQ_PAIR, 2 * (capacity - written) * NQ_PAIR);
}

cudaError_t launch_scatter_int(Ctx &c, const int32_t *src_sorted, int32_t *dst_id, int width) {
  const int b = c.cur;
  if (c.N == 0) return cudaSuccess;
  scatter_int_kernel<<<nblk(c.N, 256), 256, 0, c.stream>>>(src_sorted, c.id[b], c.N, width, dst_id);
  return cudaGetLastError();
}

}  // namespace rbe
