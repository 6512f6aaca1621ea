// Radial and angular distance factors of the FP64 path, one thread per pair: the primitive-
// basis coefficients b_alpha(r) (Eq. 04 from the erf seed, the buffer zone of Sec. III.B as a
// second Gaussian, the closed-form Gaussian row) and w_l ilexp_l(r) (Sec. III.C), with d/dr for
// the adjoint.  The forward and adjoint pair kernels read them back.
//
// FP64 instructions bound the FP64 path (about two lanes per SM and clock), and a warp
// instruction costs the same whatever its active lanes.  Inside the warp-per-atom kernels this
// work ran on batches of 32 pairs of one atom (78 pairs fill 81 % of three batches) and, for
// small systems, as one long chain per warp.  Here every warp is full, the batch spreads over
// all SMs, and three warps share one group of 32 pairs: the integral over [0, r_soft], the one
// over the buffer zone with the Gaussian row, and the ilexp factors.  ilexp_l comes from a
// downward recurrence started high enough above l_max (2 instructions per step) instead of two
// power series with a division per term, and its derivative from ilexp_(l+1) instead of dual
// numbers.
//
// W = S^-1/2 amplifies rounding differences between the alphas of one pair by sqrt(cond S) (7e5
// at n_max = 8, 4e7 at 10).  For n_max, l_max <= 8 and a constant sigma_r the constants of the
// two Gaussians are hoisted, the seeds come from erfcx and the derivatives are analytic (dJ_k/dc
// by parts, one operation per k, against eight of the dual recursion); otherwise the operations
// and their order are those of soapmath.cuh, so that results above n_max = 8 keep their bits.
// 1000 atoms, 77,642 pairs, n = l = 8: forward kernel 725 us before; now 140 us here (with the
// derivatives) and 186 us in the forward kernel; adjoint kernel 1545 -> 466 us.
#include <algorithm>
#include <cmath>

#include "internal.h"
#include "soapmath.cuh"

namespace {

constexpr int RAD_WARPS = 3;
constexpr double FOUR_PI = 12.566370614359172;

__constant__ double odd_number[64] = {
    1,  3,  5,  7,  9,  11, 13, 15, 17, 19, 21, 23, 25, 27,  29,  31,  33,  35,  37,  39,  41,  43,
    45, 47, 49, 51, 53, 55, 57, 59, 61, 63, 65, 67, 69, 71,  73,  75,  77,  79,  81,  83,  85,  87,
    89, 91, 93, 95, 97, 99, 101, 103, 105, 107, 109, 111, 113, 115, 117, 119, 121, 123, 125, 127};

// e^-z i_l(z) for l = 0..LT, z > 0:
//   z >= 30: upward recursion from the closed forms of l = 0, 1 (error below 1e-14 to l = 13);
//   z < 1e-3: leading terms of the power series (the next is below 1e-18);
//   else: i_(l-1) = i_(l+1) + (2l+1)/z i_l downwards from l = LT + 9 + 0.7 z, where the ratio of
//   neighbouring orders has dropped enough that the start value no longer matters, normalised
//   by l = 0.  Error below 1e-15 relative for LT = 6..13 over the range.
template <int LT> __device__ __forceinline__ void ilexp_orders(double z, double* il) {
  const double w = 1.0 / z;
  if (z >= 30.0) {
    const double e2 = exp(-2.0 * z);
    il[0] = -expm1(-2.0 * z) * (0.5 * w);
    il[1] = ((z - 1.0) + e2 * (z + 1.0)) * (0.5 * w * w);
#pragma unroll
    for (int l = 2; l <= LT; ++l) il[l] = il[l - 2] - (double)(2 * l - 1) * w * il[l - 1];
  } else if (z < 1e-3) {
    double t = exp(-z);
    const double h = 0.5 * z * z;
#pragma unroll
    for (int l = 0; l <= LT; ++l) {
      if (l > 0) t *= z / (2.0 * l + 1.0);
      il[l] = t * (1.0 + h / (2.0 * l + 3.0) * (1.0 + h / (2.0 * (2.0 * l + 5.0))));
    }
  } else {
    double hi = 0.0, lo = 1.0;
    for (int l = LT + 9 + (int)(0.7 * z); l > LT; --l) {
      const double nx = fma(odd_number[l] * w, lo, hi);
      hi = lo;
      lo = nx;
    }
#pragma unroll
    for (int l = LT; l >= 1; --l) {
      il[l] = lo;
      const double nx = fma((double)(2 * l + 1) * w, lo, hi);
      hi = lo;
      lo = nx;
    }
    const double s = -expm1(-2.0 * z) * (0.5 * w) / lo;
    il[0] = lo * s;
#pragma unroll
    for (int l = 1; l <= LT; ++l) il[l] *= s;
  }
}

// Gaussian of fixed width on [a, b] with the constants of its recursion (Eq. 04)
struct FixedGauss {
  double a, b, isw, seed, i2, eps, bcoef, irc, ta, tb;
  void set(double w, double lo, double hi, double rc) {
    a = lo;
    b = hi;
    isw = 1.0 / (std::sqrt(2.0) * w);
    seed = std::sqrt(0.5 * M_PI) * w;
    i2 = 1.0 / (2.0 * w * w);
    eps = (w * w) / (rc * rc);
    bcoef = (w * w) / rc;
    irc = 1.0 / rc;
    ta = 1.0 - lo / rc;
    tb = 1.0 - hi / rc;
  }
  // J_k = int_a^b (1 - r/rc)^k exp(-(r - c)^2 / (2 w^2)) dr, k = 0..K, and with DC dJ_k/dc.
  // The erf difference of the seed in terms of erfc(|t|) = erfcx(|t|) exp(-t^2), whose
  // exponentials are the boundary terms of the recursion: no branch on the signs, and neither
  // a second exponential nor a division of erf and erfc.
  template <int K, bool DC> __device__ __forceinline__ void integrals(double c, double* J, double* dJ) const {
    const double la = (a - c) * isw, lb = (b - c) * isw;
    double ga = exp(-la * la), gb = exp(-lb * lb);
    const double ea = erfcx(fabs(la)) * ga, eb = erfcx(fabs(lb)) * gb;
    J[0] = seed * (la >= 0.0 ? ea - eb : (lb <= 0.0 ? eb - ea : 2.0 - ea - eb));
    const double beta = 1.0 - c * irc;
    if constexpr (DC) dJ[0] = ga - gb;
    J[1] = fma(beta, J[0], bcoef * (gb - ga));
#pragma unroll
    for (int k = 1; k <= K; ++k) {
      ga *= ta;
      gb *= tb;
      const double d = ga - gb;  // t_a^k g_a - t_b^k g_b
      if constexpr (DC) dJ[k] = fma(-(double)k * irc, J[k - 1], d);
      if (k < K) J[k + 1] = fma((double)k * eps, J[k - 1], fma(beta, J[k], -bcoef * d));
    }
  }
};

// Constants of the fast path (sigma_r = sigma_0r for every pair), formed on the host.
struct FastConst {
  FixedGauss core, buf;   // [0, r_soft] with sigma_r, [r_soft, r_cut] with the product Gaussian
  double mu1, mu0, i2cb;  // centre mu1 r + mu0 of the product Gaussian, 1/2 of its width^-2 in r
  double i2g, dxg, kg;    // Gaussian row: kg exp(-i2g r^2) (1 + erf(dxg r))
  double inv_norm[SG_MAX_NMAX];
  explicit FastConst(const DevParams& p) {
    const double w = p.s0r, rs = std::min(p.rs, p.rc);
    const double tau = rs < p.rc ? (p.rc - rs) / p.nf : 1.0, s2 = 1.0 / (1.0 / (w * w) + 1.0 / (tau * tau));
    core.set(w, 0.0, rs, p.rc);
    buf.set(std::sqrt(s2), rs, p.rc, p.rc);
    mu1 = s2 / (w * w);
    mu0 = s2 * rs / (tau * tau);
    i2cb = 1.0 / (2.0 * (w * w + tau * tau));
    i2g = 1.0 / (4.0 * w * w);
    dxg = 1.0 / (2.0 * w);
    kg = std::pow(M_PI, 0.25) * std::sqrt(0.5 * w);
    for (int n = 0; n < SG_MAX_NMAX; ++n) inv_norm[n] = 1.0 / std::sqrt(p.rc / (2.0 * (n + 1) + 5.0));
  }
};

// MODE 0: values; 1: values and derivatives by forward-mode duals, both with the operations of
// soapmath.cuh.  FAST (sigma_r constant, n_max and l_max <= 8): MODE 2 values and derivatives,
// 3 values, with the constants of both Gaussians hoisted and analytic derivatives.
template <int NC, int LC, int MODE>
__global__ void __launch_bounds__(RAD_WARPS * 32) pair_radial_kernel(const PairRadialArgs a, const FastConst fc) {
  pdl_begin();
  using D = Dual<double>;
  constexpr bool FAST = MODE >= 2, DERIV = MODE == 1 || MODE == 2;
  constexpr int K = NC + 1;  // J_0 .. J_K
  auto KI = [](int n) constexpr { return n + 3 <= K ? n + 3 : K; };  // J index of alpha = n + 1
  __shared__ double jb[K + 1][32], djb[DERIV ? K + 1 : 1][32], gr[DERIV ? 2 : 1][32], cbs[DERIV ? 2 : 1][32];
  const int role = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int p0 = a.seg_offs[a.atom0 * a.nsp], p1 = a.seg_offs[a.atom1 * a.nsp];
  const DevParams& p = a.p;
  const double rs = p.rs < p.rc ? p.rs : p.rc;
  const bool buffer = rs < p.rc;
  const double tau = buffer ? (p.rc - rs) / p.nf : 1.0;
  for (int base = p0 + blockIdx.x * 32; base < p1; base += gridDim.x * 32) {
    const int pidx = base + lane;
    const bool valid = pidx < p1;
    double r = 1.0;
    if (valid) {
      const double w = a.pair_r[a.pair_idx ? a.pair_idx[pidx] : pidx].w;
      if (w >= 0.0) r = w;  // |r| < 0 marks a pair beyond r_cut in a list built with a skin
    }
    double* out = a.rad + (pidx - p0);
    double* od = out + (a.nmax + a.lmax + 1) * a.stride;
    // role 0: the integral over [0, r_soft] and the amplitude, before and after the barrier
    double J[K + 1], dJ[DERIV ? K + 1 : 1];
    double amp = 0.0, damp = 0.0;
    if (role == 2) {
      const double sp = p.s0p + p.ap * r;
      double* ov = out + a.nmax * a.stride;
      double il[LC + 2];
      if constexpr (MODE == 0 && NC > 8) {
        // (above n_max = 8 a last-bit change of a_lm moves the rounding of c_alpha, which W
        // amplifies past 1e-9: the original operations)
        ilexp_all<double, LC>(r * r / (sp * sp), il);
      } else {
        const double isp = 1.0 / sp, x = r * isp, z = x * x;
        constexpr int LT = DERIV ? LC + 1 : LC;
        ilexp_orders<LT>(z, il);
        if constexpr (DERIV) {
          const double dz = 2.0 * x * isp * (1.0 - x * p.ap), iz = 1.0 / z;
          double* odl = od + a.nmax * a.stride;
#pragma unroll
          for (int l = 0; l <= LC; ++l)
            if (l <= a.lmax && valid)
              odl[l * a.stride] = FOUR_PI * (p.eq08 ? (2.0 * l + 1.0) : 1.0) * dz *
                                  (il[l + 1] + ((double)l * iz - 1.0) * il[l]);
        }
      }
#pragma unroll
      for (int l = 0; l <= LC; ++l)
        if (l <= a.lmax && valid) ov[l * a.stride] = il[l] * (p.eq08 ? (2.0 * l + 1.0) : 1.0) * FOUR_PI;
    } else if constexpr (FAST) {
      if (role == 1) {
        if (buffer) {
          const double cb = exp(-(r - rs) * (r - rs) * fc.i2cb), dcb = -2.0 * (r - rs) * fc.i2cb * cb;
          double Jb[K + 1], dJb[DERIV ? K + 1 : 1];
          fc.buf.integrals<K, DERIV>(fma(fc.mu1, r, fc.mu0), Jb, dJb);
#pragma unroll
          for (int k = 3; k <= K; ++k) {
            jb[k][lane] = cb * Jb[k];
            if constexpr (DERIV) djb[k][lane] = fma(dcb, Jb[k], cb * fc.mu1 * dJb[k]);
          }
        }
        const double x = fc.dxg * r, ex = exp(-x * x);  // = exp(-r^2 / (2 s*^2)): both exponents r^2 / (4 sigma^2)
        const double g = fc.kg * ex, fx = 2.0 - erfcx(x) * ex;  // 1 + erf(x)
        gr[0][lane] = g * fx;
        if constexpr (DERIV) gr[1][lane] = g * fma(-2.0 * r * fc.i2g, fx, SG_TWO_OVER_SQRTPI * ex * fc.dxg);
      } else {
        const double sp = p.s0p + p.ap * r, x = r / p.rc;
        const double poly = (1.0 - x) * (1.0 - x) * (1.0 + 2.0 * x), isp = 1.0 / sp, iv = isp * isp / p.s0r;
        const double pw = p.amp_a == 1.0 ? poly : (p.amp_a == 0.0 ? 1.0 : pow(poly, p.amp_a));
        amp = pw * iv;
        if constexpr (DERIV) {
          const double dpoly = -6.0 * x * (1.0 - x) / p.rc;
          const double dpw = p.amp_a == 1.0 ? dpoly
                             : (p.amp_a == 0.0 || poly == 0.0) ? 0.0 : p.amp_a * pow(poly, p.amp_a - 1.0) * dpoly;
          damp = dpw * iv - amp * (2.0 * p.ap * isp);
        }
        fc.core.integrals<K, DERIV>(r, J, dJ);
      }
    } else if (role == 1) {
      if constexpr (MODE == 1) {
        const D rd(r, 1.0), sr = p.s0r + p.ar * rd;
        if (buffer) {
          const D s2 = 1.0 / (1.0 / (sr * sr) + 1.0 / (tau * tau));
          const D mu = s2 * (rd / (sr * sr) + rs / (tau * tau));
          const D cb = s_exp(-(rd - rs) * (rd - rs) / (2.0 * (sr * sr + tau * tau)));
          D Jd[K + 1];
#pragma unroll
          for (int k = 0; k <= K; ++k) Jd[k] = D(0.0);
          radial_integrals_add<D, K>(mu, s_sqrt(s2), rs, p.rc, p.rc, D(1.0), Jd);
#pragma unroll
          for (int k = 0; k <= K; ++k) {
            jb[k][lane] = Jd[k].v;
            djb[k][lane] = Jd[k].d;
          }
          cbs[0][lane] = cb.v;
          cbs[1][lane] = cb.d;
        }
        const D g = gaussian_row(rd, sr, p.s0r);
        gr[0][lane] = g.v;
        gr[1][lane] = g.d;
      } else {
        const double sr = p.s0r + p.ar * r;
        if (buffer) {
          const double s2 = 1.0 / (1.0 / (sr * sr) + 1.0 / (tau * tau));
          const double mu = s2 * (r / (sr * sr) + rs / (tau * tau));
          double Jd[K + 1];
#pragma unroll
          for (int k = 0; k <= K; ++k) Jd[k] = 0.0;
          radial_integrals_add<double, K>(mu, sqrt(s2), rs, p.rc, p.rc, 1.0, Jd);
#pragma unroll
          for (int k = 0; k <= K; ++k) jb[k][lane] = Jd[k];
          cbs[0][lane] = exp(-(r - rs) * (r - rs) / (2.0 * (sr * sr + tau * tau)));
        }
        gr[0][lane] = gaussian_row(r, sr, p.s0r);
      }
    } else {
      if constexpr (MODE == 1) {
        const D rd(r, 1.0), sr = p.s0r + p.ar * rd, sp = p.s0p + p.ap * rd, x = rd / p.rc;
        const D poly = (1.0 - x) * (1.0 - x) * (1.0 + 2.0 * x);
        const D da = ((p.amp_a == 0.0) ? D(1.0) : s_pow(poly, p.amp_a)) / (sr * sp * sp);
        amp = da.v;
        damp = da.d;
        D Jd[K + 1];
#pragma unroll
        for (int k = 0; k <= K; ++k) Jd[k] = D(0.0);
        radial_integrals_add<D, K>(rd, sr, 0.0, rs, p.rc, D(1.0), Jd);
#pragma unroll
        for (int k = 0; k <= K; ++k) {
          J[k] = Jd[k].v;
          dJ[k] = Jd[k].d;
        }
      } else {
        const double sr = p.s0r + p.ar * r, sp = p.s0p + p.ap * r, x = r / p.rc;
        const double poly = (1.0 - x) * (1.0 - x) * (1.0 + 2.0 * x);
        amp = ((p.amp_a == 0.0) ? 1.0 : pow(poly, p.amp_a)) / (sr * sp * sp);
#pragma unroll
        for (int k = 0; k <= K; ++k) J[k] = 0.0;
        radial_integrals_add<double, K>(r, sr, 0.0, rs, p.rc, 1.0, J);
      }
    }
    __syncthreads();
    if (role == 0 && valid) {
      const double cb = !FAST && buffer ? cbs[0][lane] : 0.0;
#pragma unroll
      for (int n = 0; n < NC; ++n) {
        if (n >= a.nmax) break;
        const int k = KI(n);
        double v, d = 0.0;
        if (n + 1 == a.nmax) {
          v = amp * gr[0][lane];
          if constexpr (DERIV) d = damp * gr[0][lane] + amp * gr[1][lane];
        } else if constexpr (FAST) {
          const double jt = buffer ? J[k] + jb[k][lane] : J[k];
          v = amp * jt * fc.inv_norm[n];
          if constexpr (DERIV) d = (damp * jt + amp * (buffer ? dJ[k] + djb[k][lane] : dJ[k])) * fc.inv_norm[n];
        } else {
          v = amp * (buffer ? fma(cb, jb[k][lane], J[k]) : J[k]) / a.norm[n];
          if constexpr (DERIV) {
            D jd(J[k], dJ[k]);
            if (buffer) jd = jd + D(cb, cbs[1][lane]) * D(jb[k][lane], djb[k][lane]);
            d = (D(amp, damp) * jd).d / a.norm[n];
          }
        }
        out[n * a.stride] = v;
        if constexpr (DERIV) od[n * a.stride] = d;
      }
    }
    __syncthreads();
  }
}

template <int NC, int LC>
cudaError_t launch(const PairRadialArgs& a, bool deriv, cudaStream_t st) {
  const FastConst fc(a.p);
  const long long need = std::max(1LL, (a.max_pairs + 31) / 32);
  const int grid = (int)std::min<long long>(need, (long long)sg_sm_count() * 64);
  if constexpr (NC <= 8) {
    if (a.p.ar == 0.0) {
      if (deriv) sg_launch(pair_radial_kernel<NC, LC, 2>, grid, RAD_WARPS * 32, 0, st, a, fc);
      else sg_launch(pair_radial_kernel<NC, LC, 3>, grid, RAD_WARPS * 32, 0, st, a, fc);
      ++sg_kernel_launches;
      return cudaGetLastError();
    }
  }
  if (deriv) sg_launch(pair_radial_kernel<NC, LC, 1>, grid, RAD_WARPS * 32, 0, st, a, fc);
  else sg_launch(pair_radial_kernel<NC, LC, 0>, grid, RAD_WARPS * 32, 0, st, a, fc);
  ++sg_kernel_launches;
  return cudaGetLastError();
}

}  // namespace

bool sg_pair_radial_one_pass(const DevParams& p, int cls) { return cls <= 1 && p.ar == 0.0; }

cudaError_t sg_pair_radial(const PairRadialArgs& a, int cls, bool deriv, cudaStream_t st) {
  if (a.atom1 <= a.atom0) return cudaSuccess;
  switch (cls) {
    case 0: return launch<6, 6>(a, deriv, st);
    case 1: return launch<8, 8>(a, deriv, st);
    case 2: return launch<10, 10>(a, deriv, st);
    default: return launch<12, 12>(a, deriv, st);
  }
}
