// Effective potential and the density-dependent energy terms (Sec. 2.1 /
// Sec. 2.3): E_ext = h^3 sum Vext rho, E_H (variational form), E_xc =
// h^3 sum rho eps_xc(rho), and V_eff = Vext + vH + v_xc with
// v_xc = d(rho eps_xc)/d rho.  LDA = Slater exchange, optionally with the
// Perdew-Zunger (1981) correlation of the unpolarised electron gas.
#include <algorithm>

#include "ks_device.cuh"

namespace ks {

// Perdew-Zunger parameters (hartree): gamma, beta1, beta2, A, B as
// published; C and D from continuity of eps_c and d eps_c / d r_s at r_s = 1
// (the published 0.0020 and -0.0116 are these rounded; rounded, they leave a
// 3.2e-5 Ha jump that makes the energy discontinuous).
constexpr double kPzGamma = -0.1423, kPzBeta1 = 1.0529, kPzBeta2 = 0.3334;
constexpr double kPzA = 0.0311, kPzB = -0.048;
constexpr double kPzDen1 = 1.0 + kPzBeta1 + kPzBeta2;
constexpr double kPzD = kPzGamma / kPzDen1 - kPzB;
constexpr double kPzC = -kPzGamma * (0.5 * kPzBeta1 + kPzBeta2) / (kPzDen1 * kPzDen1) - kPzA - kPzD;

// Elementary functions of the FP64 potential.  On GB300 every FP64 warp
// instruction holds the pipe for 16 clocks and the kernel is bound by it, so
// each function is a single-precision start (relative error e ~ 1e-7) and one
// third-order step of the binomial series, which leaves e^3 ~ 1e-21, below
// FP64 rounding: with e = 1 - rho z^3, (1 - e)^(-1/3) = 1 + e/3 + 2 e^2/9 + ...
// With library log, rsqrt and division and two Newton steps per cube root
// (taken twice in the orbital-free model) the kernel took 200 us at 105^3.
// rho^(-1/3) for rho >= 1e-30 (six FP64 instructions; two Newton steps took ten)
__device__ __forceinline__ double inv_cbrt(double rho) {
  const double z = (double)rcbrtf((float)rho);
  const double e = fma(-rho, z * z * z, 1.0);
  return fma(z, e * fma(2.0 / 9.0, e, 1.0 / 3.0), z);
}

// x^(-1/2): e = 1 - x y^2, (1 - e)^(-1/2) = 1 + e/2 + 3 e^2/8 + ...
__device__ __forceinline__ double inv_sqrt(double x) {
  const double y = (double)rsqrtf((float)x);
  const double e = fma(-x, y * y, 1.0);
  return fma(y, e * fma(0.375, e, 0.5), y);
}

// 1 / x: e = 1 - x y, (1 - e)^(-1) = 1 + e + e^2 + ...
__device__ __forceinline__ double inv_of(double x) {
  const double y = (double)__frcp_rn((float)x);
  const double e = fma(-x, y, 1.0);
  return fma(y, fma(e, e, e), y);
}

// ln x: x = 2^k m with m in [sqrt(1/2), sqrt(2)), and the area-tangent series
// ln m = 2 (s + s^3/3 + s^5/5 + ...), s = (m - 1)/(m + 1), |s| <= 0.1716: the
// terms through s^21 leave 2 s^23/23 < 3e-19.  Its roundings leave 3.5 unit
// roundoffs (the library's log about two); in v_xc, where the exchange term is tens
// of times larger, nothing of it is left: within 5.0 unit roundoffs of 128-bit values
// over rho = 1e-30 .. 1e12, against 7.7 with the library functions.  -inf at 0: r_s
// of a density beyond the FP32 range, whose start of rho^(-1/3) is 0, must not pass
// for a number.
__device__ __forceinline__ double ln_series(double x) {
  const long long bits = __double_as_longlong(x);
  // exponent of x / sqrt(1/2), by its high word (sqrt(1/2) = 0x3fe6a09e...)
  const int hi = (int)(bits >> 32);
  const int k = (hi - 0x3fe6a09e) >> 20;
  const double m = __longlong_as_double(bits - ((long long)k << 52));
  const double s = (m - 1.0) * inv_of(m + 1.0);
  const double q = s * s;
  double t = 1.0 / 21.0;
  t = fma(t, q, 1.0 / 19.0);
  t = fma(t, q, 1.0 / 17.0);
  t = fma(t, q, 1.0 / 15.0);
  t = fma(t, q, 1.0 / 13.0);
  t = fma(t, q, 1.0 / 11.0);
  t = fma(t, q, 1.0 / 9.0);
  t = fma(t, q, 1.0 / 7.0);
  t = fma(t, q, 0.2);
  t = fma(t, q, 1.0 / 3.0);
  const double s2 = s + s;
  if (bits <= 0) return __longlong_as_double(0xfff0000000000000ll);
  return fma((double)k, 0.69314718055994530942, fma(s2 * q, t, s2));
}

// eps_xc and v_xc = d(rho eps_xc)/d rho at one point, in precision R
// (FP64; FP32 for the mixed-precision phase, whose orbitals carry FP32
// rounding already; the energy sums stay FP64 in both).
//   Slater: eps_x = -(3/4) (3/pi)^(1/3) rho^(1/3), v_x = (4/3) eps_x;
//   PZ81 (r_s = (3 / (4 pi rho))^(1/3)): eps_c = gamma / (1 + beta1 sqrt(r_s)
//   + beta2 r_s) for r_s >= 1, A ln r_s + B + C r_s ln r_s + D r_s below;
//   v_c = eps_c - (r_s / 3) d eps_c / d r_s.
// z: rho^(-1/3) where rho >= 1e-30, for the Thomas-Fermi term.
template <typename R>
__device__ __forceinline__ void lda_point(double rho_d, int xc, R &eps, R &v, R &z) {
  z = 0;
  if (!(rho_d >= 1e-30)) {
    eps = 0;
    v = 0;
    return;
  }
  const R c = (R)0.98474502184269654;              // (3/pi)^(1/3)
  const R crs = (R)0.62035049089940001;            // (3/(4 pi))^(1/3)
  const R rho = (R)rho_d;
  if constexpr (sizeof(R) == 8) z = inv_cbrt(rho_d);
  else z = rcbrtf(rho);
  const R r13 = rho * z * z;                       // rho^(1/3)
  eps = (R)-0.75 * c * r13;
  v = -c * r13;
  if (xc == KS_XC_SLATER_PZ81) {
    const R rs = crs * z;
    R ec, dec;
    if (rs >= (R)1) {
      R irs;                                       // 1 / sqrt(r_s)
      if constexpr (sizeof(R) == 8) irs = inv_sqrt(rs);
      else irs = rsqrtf(rs);
      const R srs = rs * irs;
      R iden;
      if constexpr (sizeof(R) == 8)
        iden = inv_of((R)1 + (R)kPzBeta1 * srs + (R)kPzBeta2 * rs);
      else iden = (R)1 / ((R)1 + (R)kPzBeta1 * srs + (R)kPzBeta2 * rs);
      ec = (R)kPzGamma * iden;
      dec = -(R)kPzGamma * ((R)(0.5 * kPzBeta1) * irs + (R)kPzBeta2) * (iden * iden);
    } else {
      R lrs;
      if constexpr (sizeof(R) == 8) lrs = ln_series(rs);
      else lrs = logf(rs);
      ec = (R)kPzA * lrs + (R)kPzB + (R)kPzC * rs * lrs + (R)kPzD * rs;
      // A / r_s = A rho^(1/3) / crs
      dec = (R)kPzA * (r13 * (R)(1.0 / 0.62035049089940001)) + (R)kPzC * (lrs + (R)1) + (R)kPzD;
    }
    eps += ec;
    if constexpr (sizeof(R) == 8) v += ec - (rs * (R)(1.0 / 3.0)) * dec;
    else v += ec - (rs / (R)3) * dec;
  }
}

// Thomas-Fermi kinetic energy per unit volume C_TF rho^(5/3) and its
// derivative v_TF = (5/3) C_TF rho^(2/3) (the T_TF term of Eq. TFW), both 0
// below the density floor; ctf = C_TF and vtf = (5/3) C_TF in precision R.
template <typename R>
__device__ __forceinline__ void tf_point(double rho_d, R z, R ctf, R vtf, R &e, R &v) {
  if (!(rho_d >= 1e-30)) {
    e = 0;
    v = 0;
    return;
  }
  const R rho = (R)rho_d;
  const R r23 = rho * z;                           // rho^(2/3)
  v = vtf * r23;
  e = ctf * rho * r23;
}

// Channels of the block partials: 0 = E_ext, 1 = E_H, 2 = E_xc, 3 = E_TF (0
// unless ctf != 0, the orbital-free model, with v_TF added to V_eff).  Block
// vb of vnb (grid-stride over the n nodes); the last block to finish sums
// the partials in block order.
template <typename R>
__device__ __forceinline__ void potential_body(long long n, double h3, int xc, int with_h,
                                               double ctf,
                                               const double *__restrict__ rho,
                                               const double *__restrict__ vext,
                                               const double *__restrict__ vH,
                                               const double *__restrict__ r,
                                               double *__restrict__ veff, double *__restrict__ part,
                                               double *__restrict__ out, unsigned int *counter,
                                               int vb, int vnb) {
  __shared__ double smem[4 * 33];
  const double inv8pi = 1.0 / (8.0 * M_PI);
  const R ctf_r = (R)ctf, vtf_r = (R)(ctf * (5.0 / 3.0));
  double e_ext = 0.0, e_h = 0.0, e_xc = 0.0, e_tf = 0.0;
  for (long long k = (long long)vb * blockDim.x + threadIdx.x; k < n;
       k += (long long)vnb * blockDim.x) {
    const double rk = rho[k], ve = vext[k];
    R eps_r, vxc_r, z_r;
    lda_point<R>(rk, xc, eps_r, vxc_r, z_r);
    const double eps = (double)eps_r;
    double v = ve + (double)vxc_r;
    e_ext = fma(h3 * ve, rk, e_ext);
    e_xc = fma(h3 * rk, eps, e_xc);
    if (with_h) {
      const double vh = vH[k];
      v += vh;
      e_h += 0.5 * h3 * vh * rk + vh * r[k] * inv8pi;
    }
    if (ctf != 0.0) {
      R etf_r, vtf_p;
      tf_point<R>(rk, z_r, ctf_r, vtf_r, etf_r, vtf_p);
      v += (double)vtf_p;
      e_tf = fma(h3, (double)etf_r, e_tf);
    }
    veff[k] = v;
  }
  double s[4] = {e_ext, e_h, e_xc, e_tf};
  block_sum_n<4>(s, smem);
  if (threadIdx.x == 0)
#pragma unroll
    for (int c = 0; c < 4; ++c) part[c * vnb + vb] = s[c];
  grid_reduce_tail<4>(part, vnb, out, 1.0, counter, smem);
}

template <typename R>
__global__ void potential_kernel(long long n, double h3, int xc, int with_h, double ctf,
                                 const double *__restrict__ rho, const double *__restrict__ vext,
                                 const double *__restrict__ vH, const double *__restrict__ r,
                                 double *__restrict__ veff, double *__restrict__ part,
                                 double *__restrict__ out, unsigned int *counter) {
  potential_body<R>(n, h3, xc, with_h, ctf, rho, vext, vH, r, veff, part, out, counter,
                    blockIdx.x, gridDim.x);
}

// Batched: job j takes pot_nb blocks.
template <typename R>
__global__ void potential_batch_kernel(const BJob *__restrict__ jobs, const int *__restrict__ start,
                                       int J, const unsigned char *__restrict__ active) {
  const int j = batch_job_of(start, J, blockIdx.x);
  if (!active[j]) return;
  const BJob &b = jobs[j];
  potential_body<R>(b.n, b.h3, b.xc, 1, 0.0, b.rho, b.vext, b.vH, b.cg_r, b.veff, b.partials,
                    b.scal + SC_EEXT, b.red_counter, blockIdx.x - start[j], b.pot_nb);
}

ks_status batch_potential(Batch &B, bool fp32_xc) {
  const int nb = B.total(BM_POTENTIAL);
  if (nb == 0) return KS_OK;
  {
    ProfScope ps_(B.stream, KP_POTENTIAL);
    if (fp32_xc)
      potential_batch_kernel<float><<<nb, kThreads, 0, B.stream>>>(B.jobs_dev, B.map(BM_POTENTIAL),
                                                                   B.J, B.active_dev);
    else
      potential_batch_kernel<double><<<nb, kThreads, 0, B.stream>>>(
          B.jobs_dev, B.map(BM_POTENTIAL), B.J, B.active_dev);
  }
  KS_CUDA_TRY(cudaGetLastError());
  return KS_OK;
}

// out[c] = scale * sum_{b < nb} part[c * nb + b], one block per channel, in
// a fixed order.
__global__ void reduce_kernel(const double *__restrict__ part, int nb, double scale,
                              double *__restrict__ out) {
  __shared__ double smem[33];
  const double s = block_sum_array(part + (long long)blockIdx.x * nb, nb, smem);
  if (threadIdx.x == 0) out[blockIdx.x] = scale * s;
}

int reduce_blocks(const Problem &P, long long work) {
  long long nb = (work + kThreads - 1) / kThreads;
  const long long cap = 8LL * P.sms;
  if (nb > cap) nb = cap;
  if (nb < 1) nb = 1;
  return (int)nb;
}

ks_status launch_reduce(Problem &P, const double *partials, int nchan, int nb, double *out,
                        double scale) {
  {
    ProfScope ps_(P.stream, KP_REDUCE);
    reduce_kernel<<<nchan, kThreads, 0, P.stream>>>(partials, nb, scale, out);
  }
  KS_CUDA_TRY(cudaGetLastError());
  return KS_OK;
}

ks_status launch_potential(Problem &P, const double *rho, const double *vH, const double *r,
                           double *veff, bool with_hartree, bool fp32_xc) {
  // at most two blocks per SM: a block ends in four FP64 sums, as much work for
  // the FP64 pipe as a third of a node per thread, and the last one sums all
  // blocks' partials.  Up to eight blocks per SM against two: FP64 step_potential
  // at 64^3 93 / 85 us, at 128^3 400 / 387, at 200^3 1388 / 1376, even below 48^3;
  // the FP32 form in a minimisation, 64^3 53 / 43 us per launch, 96^3 121 / 108
  const int nb = std::min(reduce_blocks(P, P.n), 2 * P.sms);
  const double h3 = P.h * P.h * P.h;
  {
    ProfScope ps_(P.stream, KP_POTENTIAL, 40.0 * P.n, 40.0 * P.n);
    if (fp32_xc)
      potential_kernel<float><<<nb, kThreads, 0, P.stream>>>(
          P.n, h3, P.xc, with_hartree ? 1 : 0, P.ctf, rho, P.vext, vH, r, veff, P.partials,
          P.scal + SC_EEXT, P.red_counter);
    else
      potential_kernel<double><<<nb, kThreads, 0, P.stream>>>(
          P.n, h3, P.xc, with_hartree ? 1 : 0, P.ctf, rho, P.vext, vH, r, veff, P.partials,
          P.scal + SC_EEXT, P.red_counter);
  }
  KS_CUDA_TRY(cudaGetLastError());
  return KS_OK;
}

}  // namespace ks
