// k_kspace.cu -- structure factor and k-space force gather of the RBE estimator.
//
// rho(k_l) = sum_j q_j exp(i k_l . r_j)           (Eq. U_Coul_Fourier, charged particles only)
// F_i = -q_i sum_l c_l k_l (Im rho_l cos t_il - Re rho_l sin t_il),  c_l = 4 pi C S / (P V k_l^2)
//                                                  (Eq. F_long_RBE with the sign of Eq. F_i)
// U = sum_l (c_l / 2) |rho_l|^2,  W = sum_l (c_l / 2) |rho_l|^2 (1 - k_l^2 / 2 alpha)
//
// Phases are exact: on the 2^-32 grid k_l . r_j / 2 pi = sum_d m_d s_d / 2^32 (mod 1), an
// integer multiply-add in wrapping uint32 arithmetic. Only the final angle is rounded
// (2^-23 turns in the FP32 forms).
//
// The paper's pipeline is sampling -> local accumulation -> global reduction ->
// force application (Sec. 2.3.1). On one GPU its AllReduce of 2P values becomes a grid
// reduction. Each block writes compensated FP32 partials of its particle tile for a
// contiguous slice of modes (one thread per mode, particles broadcast from shared memory,
// no atomics). A combine kernel then sums the partials in FP64 in a fixed order, so the
// result is reproducible run to run. In the FP32 forms both passes are bound by FMA and issue slots
// (three integer multiply-adds, a sine and a cosine, five to nine further operations a particle
// and mode), so they take two phases a step, on packed pairs where those are not the slower form.
#include "f32x2.cuh"
#include "rbe_internal.cuh"

namespace rbe {

struct SfArgs {
  const uint32_t *cs;
  const float *cqf;
  const double *cqd;
  int64_t Nq;
  const int4 *m;
  int P, tile;
  int slices;  // tiles a block (P <= 256; otherwise 1 and blockIdx.y counts the modes' blocks)
  double *part;
};
struct CombineArgs {
  const double *part;
  int nblk, P;
  const double4_16a *kcd;
  double alpha;
  double2 *rho;
  float2 *abf;
  double2 *abd;
  double *emode;
};
struct GatherArgs {
  const uint32_t *cs;
  const float *cqf;
  const double *cqd;
  int64_t Nq;
  const int4 *m;
  const float4 *kcf;
  const double4_16a *kcd;
  const float2 *abf;
  const double2 *abd;
  int P, slices;           // the modes shared by `slices` threads a particle
  const int32_t *cmap;
  void *fk;                // 3 x Nq forces in charged order (of the form's type), or, with facc,
  int64_t N;
  long long *facc;         // nullable: add to these 3 x N fixed-point sums instead
  float fscale;            // (their scale in the FP32 forms,
  double fscale_d;         //  and in the FP64 form)
  int *err;
};

// Solo and batched kernels of a body templated on MODE.
#define RBE_MODE_KERNELS(LB, NAME, ARGS, BODY)                                                 \
  template <int MODE>                                                                        \
  __global__ void LB NAME(const ARGS a) { BODY<MODE>(a, (int)blockIdx.x, (int)gridDim.x); }   \
  template <int MODE>                                                                        \
  __global__ void LB NAME##_b(const ARGS *__restrict__ t, const int32_t *__restrict__ pre,   \
                              int nrep) {                                                     \
    const BatchIdx q = batch_locate(pre, nrep);                                               \
    BODY<MODE>(t[q.r], q.bx, q.nbx);                                                          \
  }

// sin and cos of a phase ph / 2^32 turns in FP64. The phase is exact, so its reduction to the
// nearest quarter turn is integer arithmetic, and Taylor polynomials to x^15 and x^16 on
// |x| <= pi / 4 leave less than 7e-17 relative: 19 FP64 operations, where sincos() of the angle
// took about three times as many (the FP64 form's k-space passes are bound by the FP64 pipe).
__device__ __forceinline__ void sincos_phase(uint32_t ph, double &sn, double &co) {
  const uint32_t q = (ph + 0x20000000u) >> 30;
  const double x = i2d((int)(ph - (q << 30))) * (2.0 * kPi / kTwo32);
  const double t = x * x;
  double s = -1.0 / 1307674368000.0;
  s = fma(s, t, 1.0 / 6227020800.0);
  s = fma(s, t, -1.0 / 39916800.0);
  s = fma(s, t, 1.0 / 362880.0);
  s = fma(s, t, -1.0 / 5040.0);
  s = fma(s, t, 1.0 / 120.0);
  s = fma(s, t, -1.0 / 6.0);
  s = fma(x * t, s, x);
  double c = 1.0 / 20922789888000.0;
  c = fma(c, t, -1.0 / 87178291200.0);
  c = fma(c, t, 1.0 / 479001600.0);
  c = fma(c, t, -1.0 / 3628800.0);
  c = fma(c, t, 1.0 / 40320.0);
  c = fma(c, t, -1.0 / 720.0);
  c = fma(c, t, 1.0 / 24.0);
  c = fma(c, t, -0.5);
  c = fma(c, t, 1.0);
  // quarter turns: (s, c), (c, -s), (-s, -c), (-c, s)
  const double a = q & 1u ? c : s, b = q & 1u ? s : c;
  sn = __hiloint2double(__double2hiint(a) ^ (int)((q & 2u) << 30), __double2loint(a));
  co = __hiloint2double(__double2hiint(b) ^ (int)(((q + 1u) & 2u) << 30), __double2loint(b));
}

// A phase plus a bias, which rides on the multiply-adds.
__device__ __forceinline__ uint32_t phase_add(int4 m, uint32_t x, uint32_t y, uint32_t z,
                                              uint32_t bias) {
  return (uint32_t)m.x * x + ((uint32_t)m.y * y + ((uint32_t)m.z * z + bias));
}
// The angles of two phases with kTurnBias added: the values of phase_to_radians, the exponent of
// 2^23 set by the shift.
constexpr uint32_t kTurnBias = 0x80000100u;
__device__ __forceinline__ f32x2 turns_to_radians(uint32_t pa, uint32_t pb) {
  const f32x2 f = pk(__uint_as_float(__funnelshift_r(pa, 150u, 9)),  // 2^23 + (p >> 9)
                     __uint_as_float(__funnelshift_r(pb, 150u, 9)));
  return mul2(add2(f, pk(-12582912.0f)), pk((float)(2.0 * kPi / 8388608.0)));
}
// The angles of two phases with kHalfBias added, from the middle of their half turn: 2^-24 turns,
// twice as fine; bit 31 tells the second half turn, where sine and cosine change sign.
constexpr uint32_t kHalfBias = 0x40000080u;
__device__ __forceinline__ f32x2 half_turns_to_radians(uint32_t pa, uint32_t pb) {
  const f32x2 f = pk(__uint_as_float(((pa >> 8) & 0x7fffffu) | 0x4b000000u),
                     __uint_as_float(((pb >> 8) & 0x7fffffu) | 0x4b000000u));
  return mul2(add2(f, pk(-12582912.0f)), pk((float)(kPi / 8388608.0)));
}

// MODE: 0 = FP32 with Kahan-compensated per-thread sums, 1 = plain FP32, 2 = FP64.
// MODE 0 compensates the sum of two particles' terms at once. That alone would leave rho 0.5% less
// exact (2.77e-7 against 64 bits for 200,000 ions); the finer phases more than make up for it
// (1.98e-7). 1,400,000 ions, P = 200: 198 us with one particle a step and every term compensated
// by itself, 184 on full warps (see sf_launch), 172 so.
template <int MODE>
__device__ __forceinline__ void sf_body(const SfArgs &a, int bx, int) {
  extern __shared__ uint4 smem[];  // tile particles (an even number) a slice
  uint4 *sh = smem;
  const uint32_t *__restrict__ cs = a.cs;
  const float *__restrict__ cqf = a.cqf;
  const double *__restrict__ cqd = a.cqd;
  const int64_t Nq = a.Nq;
  const int P = a.P, tile = a.tile;
  const int64_t b0 = (int64_t)bx * a.slices * tile;
  const int nb = (int)min((int64_t)tile * a.slices, Nq - b0);
  double *shq = reinterpret_cast<double *>(sh + tile);
  for (int k = threadIdx.x; k < nb; k += blockDim.x) {
    sh[k] = make_uint4(cs[b0 + k], cs[Nq + b0 + k], cs[2 * Nq + b0 + k],
                       __float_as_uint(cqf[b0 + k]));
    if (MODE == 2) shq[k] = cqd[b0 + k];
  }
  if (MODE != 2 && (nb & 1) && threadIdx.x == 0) sh[nb] = make_uint4(0u, 0u, 0u, 0u);  // no charge
  __syncthreads();
  int l = blockIdx.y * blockDim.x + threadIdx.x, slice = 0;
  if (MODE != 2 && a.slices > 1) {
    slice = l / P;
    l -= slice * P;
    sh += slice * tile;
  }
  const int np = min(tile, nb - slice * tile);
  if (l >= P || slice >= a.slices || np <= 0) return;
  const int4 mm = a.m[l];
  double *out = a.part + (((int64_t)bx * a.slices + slice) * P + l) * 2;
  if (MODE == 2) {
    double re = 0.0, im = 0.0;
    for (int k = 0; k < np; ++k) {
      const uint4 e = sh[k];
      double sn, co;
      sincos_phase(phase_u32(mm, e.x, e.y, e.z), sn, co);
      re = mad(shq[k], co, re);
      im = mad(shq[k], sn, im);
    }
    out[0] = re;
    out[1] = im;
  } else {
    f32x2 sum = pk(0.f), low = pk(0.f);  // (Re, Im) and what their additions dropped
    const f32x2 m1 = pk(-1.f);
    if (MODE == 0) {
#pragma unroll 2
      for (int k = 0; k < np; k += 2) {
        const uint4 e = sh[k], g = sh[k + 1];
        const uint32_t pa = phase_add(mm, e.x, e.y, e.z, kHalfBias),
                       pb = phase_add(mm, g.x, g.y, g.z, kHalfBias);
        const f32x2 w = half_turns_to_radians(pa, pb);
        f32x2 ea, eb;
        __sincosf(w.x, &ea.y, &ea.x);
        __sincosf(w.y, &eb.y, &eb.x);
        // the second half turn's sign, on the charge
        const f32x2 qa = pk(__uint_as_float(e.w ^ (pa & 0x80000000u))),
                    qb = pk(__uint_as_float(g.w ^ (pb & 0x80000000u)));
        // Kahan summation of the pair's terms
        const f32x2 y = fma2(qb, eb, fma2(qa, ea, low)), t = add2(sum, y);
        low = fma2(fma2(sum, m1, t), m1, y);
        sum = t;
      }
    } else {
#pragma unroll 8
      for (int k = 0; k < np; k += 2) {
        const uint4 e = sh[k], g = sh[k + 1];
        const f32x2 w = turns_to_radians(phase_add(mm, e.x, e.y, e.z, kTurnBias),
                                         phase_add(mm, g.x, g.y, g.z, kTurnBias));
        f32x2 ea, eb;
        __sincosf(w.x, &ea.y, &ea.x);
        __sincosf(w.y, &eb.y, &eb.x);
        sum = fma2(pk(__uint_as_float(g.w)), eb, fma2(pk(__uint_as_float(e.w)), ea, sum));
      }
    }
    out[0] = f2d(sum.x) + f2d(low.x);
    out[1] = f2d(sum.y) + f2d(low.y);
  }
}
RBE_MODE_KERNELS(__launch_bounds__(MODE == 2 ? 256 : 1024), sf_kernel, SfArgs, sf_body)

// One block per mode: sum the block partials in a fixed order, then derive the per-mode
// energy, virial and the gather coefficients (c Im rho, c Re rho).
template <int MODE>
__device__ __forceinline__ void sf_combine_body(const CombineArgs &a, int bx, int) {
  __shared__ double sre[128], sim[128];
  __shared__ float fre[128], fim[128];
  const double *__restrict__ part = a.part;
  const int nblk = a.nblk, P = a.P;
  const int l = bx;
  if (MODE == 1) {
    float re = 0.f, im = 0.f;
    for (int b = threadIdx.x; b < nblk; b += blockDim.x) {
      re += (float)part[((int64_t)b * P + l) * 2];
      im += (float)part[((int64_t)b * P + l) * 2 + 1];
    }
    fre[threadIdx.x] = re;
    fim[threadIdx.x] = im;
    __syncthreads();
    for (int s = 64; s > 0; s >>= 1) {
      if (threadIdx.x < s) {
        fre[threadIdx.x] += fre[threadIdx.x + s];
        fim[threadIdx.x] += fim[threadIdx.x + s];
      }
      __syncthreads();
    }
    if (threadIdx.x == 0) { sre[0] = fre[0]; sim[0] = fim[0]; }
  } else {
    double re = 0.0, im = 0.0;
    for (int b = threadIdx.x; b < nblk; b += blockDim.x) {
      re += part[((int64_t)b * P + l) * 2];
      im += part[((int64_t)b * P + l) * 2 + 1];
    }
    sre[threadIdx.x] = re;
    sim[threadIdx.x] = im;
    __syncthreads();
    for (int s = 64; s > 0; s >>= 1) {
      if (threadIdx.x < s) {
        sre[threadIdx.x] += sre[threadIdx.x + s];
        sim[threadIdx.x] += sim[threadIdx.x + s];
      }
      __syncthreads();
    }
  }
  if (threadIdx.x == 0) {
    const double re = sre[0], im = sim[0];
    const double4_16a kc = a.kcd[l];
    const double k2 = kc.x * kc.x + kc.y * kc.y + kc.z * kc.z;
    const double E = 0.5 * kc.w * (re * re + im * im);
    a.rho[l] = make_double2(re, im);
    a.emode[2 * l] = E;
    a.emode[2 * l + 1] = E * (1.0 - k2 / (2.0 * a.alpha));
    a.abf[l] = make_float2((float)(kc.w * im), (float)(kc.w * re));
    a.abd[l] = make_double2(kc.w * im, kc.w * re);
  }
}
RBE_MODE_KERNELS(__launch_bounds__(128), sf_combine_kernel, CombineArgs, sf_combine_body)

constexpr int kGatherThreads = 256;
constexpr int kGatherChunk = 256;

template <int MODE> struct GatherReal { using type = float; };
template <> struct GatherReal<2> { using type = double; };

// FP32 forms: a thread takes the modes in pairs, whose data lie side by side in shared memory (two
// 16-byte loads a mode instead of three): 1,400,000 charged, P = 200: 176 -> 156 us; 400,000, P = 500:
// 137 -> 121 us.
template <int MODE>
__device__ __forceinline__ void gather_body(const GatherArgs &a, int bx, int) {
  const uint32_t *__restrict__ cs = a.cs;
  const int64_t Nq = a.Nq, N = a.N;
  const int P = a.P;
  const int4 *__restrict__ m = a.m;
  const float4 *__restrict__ kcf = a.kcf;
  const double4_16a *__restrict__ kcd = a.kcd;
  const float2 *__restrict__ abf = a.abf;
  const double2 *__restrict__ abd = a.abd;
  __shared__ int4 sm[MODE == 2 ? kGatherChunk : 1];
  __shared__ float4 skp[MODE == 2 ? 1 : kGatherChunk * 2];  // 4 a pair of modes
  __shared__ double4_16a skd[MODE == 2 ? kGatherChunk : 1];
  __shared__ double2 sabd[MODE == 2 ? kGatherChunk : 1];
  const int nper = kGatherThreads / a.slices;  // particles a block (a multiple of 32)
  const int slice = threadIdx.x / nper, ip = threadIdx.x - slice * nper;
  const int64_t i = (int64_t)bx * nper + ip;
  const bool valid = i < Nq;
  const uint32_t sx = valid ? cs[i] : 0u, sy = valid ? cs[Nq + i] : 0u,
                 sz = valid ? cs[2 * Nq + i] : 0u;
  f32x2 gx = pk(0.f), gy = pk(0.f), gz = pk(0.f);  // over the even and the odd modes
  double dx = 0.0, dy = 0.0, dz = 0.0;
  for (int l0 = 0; l0 < P; l0 += kGatherChunk) {
    const int nl = min(kGatherChunk, P - l0);
    __syncthreads();
    if (MODE == 2) {
      for (int t = threadIdx.x; t < nl; t += blockDim.x) {
        sm[t] = m[l0 + t];
        skd[t] = kcd[l0 + t];
        sabd[t] = abd[l0 + t];
      }
    } else {  // a pair of modes: (m.x, m.y) (m.z, A) (B, kx) (ky, kz) of both, side by side
      for (int h = threadIdx.x; 2 * h < nl; h += blockDim.x) {
        const int ta = l0 + 2 * h;
        const bool two = 2 * h + 1 < nl;
        const int4 ma = m[ta], mb = two ? m[ta + 1] : make_int4(0, 0, 0, 0);
        const float4 ka = kcf[ta], kb = two ? kcf[ta + 1] : make_float4(0.f, 0.f, 0.f, 0.f);
        const float2 ca = abf[ta], cb = two ? abf[ta + 1] : make_float2(0.f, 0.f);
        float2 *o = reinterpret_cast<float2 *>(skp) + 8 * h;
        o[0] = pk(__int_as_float(ma.x), __int_as_float(mb.x));
        o[1] = pk(__int_as_float(ma.y), __int_as_float(mb.y));
        o[2] = pk(__int_as_float(ma.z), __int_as_float(mb.z));
        o[3] = pk(ca.x, cb.x);
        o[4] = pk(-ca.y, -cb.y);
        o[5] = pk(ka.x, kb.x);
        o[6] = pk(ka.y, kb.y);
        o[7] = pk(ka.z, kb.z);
      }
    }
    __syncthreads();
    const int nt = MODE == 2 ? nl : (nl + 1) / 2;
    const int t0 = nt * slice / a.slices, t1 = nt * (slice + 1) / a.slices;
    if (MODE == 2) {
      for (int t = t0; t < t1; ++t) {
        double sn, co;
        sincos_phase(phase_u32(sm[t], sx, sy, sz), sn, co);
        const double g = mad(sabd[t].x, co, -(sabd[t].y * sn));
        dx = mad(g, skd[t].x, dx);
        dy = mad(g, skd[t].y, dy);
        dz = mad(g, skd[t].z, dz);
      }
    } else {
#pragma unroll 2
      for (int t = t0; t < t1; ++t) {
        const float4 u = skp[4 * t], v = skp[4 * t + 1], b = skp[4 * t + 2], k = skp[4 * t + 3];
        const int4 ma = make_int4(__float_as_int(u.x), __float_as_int(u.z), __float_as_int(v.x), 0);
        const int4 mb = make_int4(__float_as_int(u.y), __float_as_int(u.w), __float_as_int(v.y), 0);
        const f32x2 w = turns_to_radians(phase_add(ma, sx, sy, sz, kTurnBias),
                                         phase_add(mb, sx, sy, sz, kTurnBias));
        f32x2 sn, co;
        __sincosf(w.x, &sn.x, &co.x);
        __sincosf(w.y, &sn.y, &co.y);
        const f32x2 g = fma2(pk(v.z, v.w), co, mul2(pk(b.x, b.y), sn));
        gx = fma2(g, pk(b.z, b.w), gx);
        gy = fma2(g, pk(k.x, k.y), gy);
        gz = fma2(g, pk(k.z, k.w), gz);
      }
    }
  }
  float fx = gx.x + gx.y, fy = gy.x + gy.y, fz = gz.x + gz.y;
  if (a.slices > 1) {  // the slices' sums, added up in order
    using real = typename GatherReal<MODE>::type;
    __shared__ real part[3][kGatherThreads];
    const int t = threadIdx.x;
    part[0][t] = MODE == 2 ? (real)dx : (real)fx;
    part[1][t] = MODE == 2 ? (real)dy : (real)fy;
    part[2][t] = MODE == 2 ? (real)dz : (real)fz;
    __syncthreads();
    if (slice) return;
    real s[3];
    for (int d = 0; d < 3; ++d) {
      s[d] = part[d][ip];
      for (int k = 1; k < a.slices; ++k) s[d] += part[d][k * nper + ip];
    }
    if (MODE == 2) { dx = (double)s[0]; dy = (double)s[1]; dz = (double)s[2]; }
    else { fx = (float)s[0]; fy = (float)s[1]; fz = (float)s[2]; }
  }
  if (!valid) return;
  if (a.facc) {
    const int64_t p = a.cmap[i];  // into the cluster kernel's fixed-point sums (integer atomics)
    if (MODE == 2) {
      const double q = a.cqd[i];
      fx_add(a.facc + p, -q * dx, a.fscale_d, a.err);
      fx_add(a.facc + N + p, -q * dy, a.fscale_d, a.err);
      fx_add(a.facc + 2 * N + p, -q * dz, a.fscale_d, a.err);
    } else {
      const float q = a.cqf[i];
      fx_add_i32(a.facc + p, -q * fx, a.fscale, a.err);
      fx_add_i32(a.facc + N + p, -q * fy, a.fscale, a.err);
      fx_add_i32(a.facc + 2 * N + p, -q * fz, a.fscale, a.err);
    }
  } else if (MODE == 2) {
    double *__restrict__ fk = static_cast<double *>(a.fk);
    const double q = a.cqd[i];
    fk[i] = -q * dx;
    fk[Nq + i] = -q * dy;
    fk[2 * Nq + i] = -q * dz;
  } else {
    float *__restrict__ fk = static_cast<float *>(a.fk);
    const float q = a.cqf[i];
    fk[i] = -q * fx;
    fk[Nq + i] = -q * fy;
    fk[2 * Nq + i] = -q * fz;
  }
}
RBE_MODE_KERNELS(__launch_bounds__(kGatherThreads, 1), gather_kernel, GatherArgs, gather_body)

// F += the k-space forces of the charged particles (gather_kernel without fixed-point sums), so
// that the gather can run beside the pass that writes F.
struct KAddArgs {
  const void *fk;
  const int32_t *cmap;
  void *F;
  int64_t Nq, N;
  int fp64;
};
__device__ __forceinline__ void kspace_add_body(const KAddArgs &a, int bx, int) {
  const int64_t i = (int64_t)bx * blockDim.x + threadIdx.x;
  if (i >= a.Nq) return;
  const int64_t p = a.cmap[i];
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    if (a.fp64)
      static_cast<double *>(a.F)[d * a.N + p] += static_cast<const double *>(a.fk)[d * a.Nq + i];
    else
      static_cast<float *>(a.F)[d * a.N + p] += static_cast<const float *>(a.fk)[d * a.Nq + i];
  }
}
RBE_BATCHED_KERNEL(__launch_bounds__(256), kspace_add_kernel, KAddArgs, kspace_add_body)

template <int MODE>
static cudaError_t sf_launch(Ctx &c, dim3 grid, size_t shm) {
  // Of P = 200 modes' seven warps one has 8 of its 32 lanes at work. Where the tiles are long and
  // give every SM four, a block takes up to four of them and lays its threads over modes and tiles
  // (P = 200: 25 full warps for four; 1,400,000 charged: a step 1,105 -> 1,086 us). Shorter ones keep
  // small blocks, which find room beside those of the other graph branch (100,000 charged, Verlet
  // list: a step 87 us, 114 with blocks of four tiles).
  int k = 1;
  if (MODE != 2 && c.P <= 256 && c.sf_tile >= 256 && c.sf_nblk_p >= 4 * c.sms) {
    auto full = [&](int n) { return (double)(c.P * n) / ((c.P * n + 31) / 32); };
    for (int n = 2; n <= 4; ++n)
      if (n * shm <= 48 * 1024 && full(n) > 1.01 * full(k)) k = n;
  }
  const SfArgs a{c.cs, c.cqf, c.cqd, c.Nq, c.m, c.P, c.sf_tile, k, c.sf_part};
  const dim3 block((unsigned)(k > 1 ? (k * c.P + 31) / 32 * 32 : c.sf_mb));
  grid.x = (grid.x + k - 1) / k;
  cudaError_t e = dispatch(c, sf_kernel<MODE>, sf_kernel_b<MODE>, grid, block, k * shm, a);
  if (e != cudaSuccess) return e;
  const CombineArgs b{c.sf_part, c.sf_nblk_p, c.P, c.kcd, c.alpha, c.rho, c.abf, c.abd, c.emode};
  return dispatch(c, sf_combine_kernel<MODE>, sf_combine_kernel_b<MODE>, dim3(c.P), dim3(128),
                  0, b);
}

cudaError_t launch_structure_factor(Ctx &c) {
  if (c.Nq == 0) return cudaSuccess;
  const dim3 grid((unsigned)c.sf_nblk_p, (unsigned)c.sf_nblk_m);
  const size_t shm = (size_t)c.sf_tile * (sizeof(uint4) + (c.precision == RBE_FP64 ? 8 : 0));
  switch (c.precision) {
    case RBE_FP32_COMP: return sf_launch<0>(c, grid, shm);
    case RBE_FP32: return sf_launch<1>(c, grid, shm);
    default: return sf_launch<2>(c, grid, shm);
  }
}

cudaError_t launch_kspace_gather(Ctx &c, bool into_facc) {
  if (c.Nq == 0) return cudaSuccess;
  // threads a particle, each with its slice of the modes: one, and twice as many (up to 8) while
  // the blocks would not give every SM four (FP64 form, 6,554 charged, P = 200: 446 -> 172 us with
  // 32-thread blocks, 94 with eight slices, at the FP64 pipe's rate).
  int slices = 1;
  while (slices < 8 && c.Nq * slices < (int64_t)4 * c.sms * kGatherThreads) slices *= 2;
  const int nper = kGatherThreads / slices;
  const unsigned blocks = (unsigned)((c.Nq + nper - 1) / nper);
  const GatherArgs a{c.cs, c.cqf, c.cqd, c.Nq, c.m, c.kcf, c.kcd, c.abf, c.abd, c.P, slices, c.cmap,
                     c.fk, c.N, into_facc ? c.facc : nullptr, (float)kFixScale32,
                     kFixScale64, c.err};
  // (into the fixed-point sums it runs per replica in a batch, within the pair pass's run)
  if (c.precision == RBE_FP64)
    return dispatch(c, gather_kernel<2>, gather_kernel_b<2>, dim3(blocks), dim3(kGatherThreads),
                    0, a, into_facc);
  return dispatch(c, gather_kernel<0>, gather_kernel_b<0>, dim3(blocks), dim3(kGatherThreads), 0,
                  a, into_facc);
}

cudaError_t launch_kspace_add(Ctx &c) {
  if (c.Nq == 0) return cudaSuccess;
  const bool fp64 = c.precision == RBE_FP64;
  const KAddArgs a{c.fk, c.cmap, fp64 ? (void *)c.Fd : (void *)c.F, c.Nq, c.N, fp64 ? 1 : 0};
  return dispatch(c, kspace_add_kernel, kspace_add_kernel_b, dim3((unsigned)((c.Nq + 255) / 256)),
                  dim3(256), 0, a);
}

}  // namespace rbe
