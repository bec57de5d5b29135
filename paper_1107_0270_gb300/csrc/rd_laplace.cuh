// FP64 pair quantities from their Laplace transforms, one warp per pair.
//
// In units a = D = 1 and with w = sqrt(s), the transforms in time of the paper's Green's functions
// are products of modified Bessel functions.  With the boundary at R = 1, orders n (2D: K_n, I_n;
// 3D: the modified spherical functions k_n) and the Wronskian taken out,
//   ref - abs : K_n(wR) K_n(wR0) / (K_n(w) (-K_n'(w)))      (up to a factor w)
//   ref - rad : h K_0(wR) K_0(wR0) / (K_1(w) (w K_1(w) + h K_0(w)))        (2D, n = 0)
//   free - abs: w (I_0(w) / K_0(w)) K_0(wR) K_0(wR0)                       (2D, n = 0)
// and the value at time tau is a constant times Re int e^{tau w^2} (...) d xi along w = c - i xi,
// xi in [0, inf).  Every factor behaves like e^{-w u}, u = R + R0 - 2, so on the line
// c = u / 2 tau the integrand is e^{-tau xi^2} times a slowly varying function: no oscillation and
// nothing cancels, which the same integrals on the real axis of x = i w (the paper's form) do
// within e^{-u^2/4 tau}.  The midpoint rule with 32 nodes, one per lane, converges to rounding
// there: the spacing h = sqrt(39.5/tau)/32 leaves e^{-2 pi d/h} with d the distance to the branch
// point w = 0, and the line is kept at d >= 1.25/sqrt(tau) (at contact that costs a factor e^{1.25^2}
// of rounding).  The functions of the third kind grow upward in n, so their three-term recurrence is
// run upward from n = 0, 1 without stored arrays.
//
// Why this form: the real-axis quadrature took 300-900 nodes with six Bessel sequences each (a
// downward and an upward one for three arguments).  On GB300's FP64 pipe (two lanes per SM) that
// was 2-4 ms of one SM per direction, and 1328 nodes of four to ten Bessel calls per 2D
// probability or CDF value.  Here a direction in 3D is about 1500 warp instructions.
#pragma once

#include "rd_angle.cuh"
#include "rd_gf2d.cuh"
#include "rd_internal.cuh"

namespace rd {

#define RD_HD __host__ __device__ __forceinline__

struct cplx {
  double re, im;
};
RD_HD cplx cx(double re, double im) { return cplx{re, im}; }
RD_HD cplx operator+(cplx a, cplx b) { return cplx{a.re + b.re, a.im + b.im}; }
RD_HD cplx operator-(cplx a, cplx b) { return cplx{a.re - b.re, a.im - b.im}; }
RD_HD cplx operator*(cplx a, cplx b) { return cplx{a.re * b.re - a.im * b.im, a.re * b.im + a.im * b.re}; }
RD_HD cplx operator*(double s, cplx a) { return cplx{s * a.re, s * a.im}; }
RD_HD cplx crcp(cplx a) {
  const double q = 1.0 / (a.re * a.re + a.im * a.im);
  return cplx{a.re * q, -a.im * q};
}
// Re(a / b)
RD_HD double re_quot(cplx a, cplx b) { return (a.re * b.re + a.im * b.im) / (b.re * b.re + b.im * b.im); }

// Rational coefficients of the recurrences (filled at compile time).
constexpr int kLapMiller = 72;                 // largest order of the K_0, K_1 recurrence below
struct LapTab {
  double r[kLapMiller + 1];                    // n / (n - 1/2)^2
  double leg_a[kAngNMax + 1], leg_b[kAngNMax + 1];   // (2n+1)/(n+1), n/(n+1)
  double ik[kAngNMax + 1], ih[25];             // 1/k, H_k
};
constexpr LapTab make_lap_tab() {
  LapTab t{};
  for (int n = 1; n <= kLapMiller; ++n) t.r[n] = 4.0 * n / ((2.0 * n - 1.0) * (2.0 * n - 1.0));
  for (int n = 0; n <= kAngNMax; ++n) {
    t.leg_a[n] = (2.0 * n + 1.0) / (n + 1.0);
    t.leg_b[n] = n / (n + 1.0);
  }
  for (int k = 1; k <= kAngNMax; ++k) t.ik[k] = 1.0 / k;
  for (int k = 1; k < 25; ++k) t.ih[k] = t.ih[k - 1] + 1.0 / k;
  return t;
}
static __constant__ LapTab c_lap = make_lap_tab();
#ifdef __CUDA_ARCH__
#define RD_LAP c_lap
#else
static constexpr LapTab h_lap = make_lap_tab();
#define RD_LAP h_lap
#endif

// e^x K_0(x) and e^x K_1(x) for Re x > 0.  Where |x| + Re x < 5 the ascending series (Abramowitz &
// Stegun 9.6.11, 9.6.13); elsewhere Temme's backward recurrence (J. Comput. Phys. 19 (1975) 324) with
// the terms of its normalising sum as the unknowns, u_n = C_n z_n:
//   u_{n-1} = n / (n - 1/2)^2 [2 (n + x) u_n - (n + 1) u_{n+1}],
//   e^x K_0 = sqrt(pi / 2x) u_0 / sum u_n,  K_1 = K_0 (x + 1/2 - u_1 / u_0) / x,
// started 12 + 280 / (|x| + Re x) orders up (both forms checked against 30-digit values: relative
// error below 2e-14 for |x| in 0.3..60 and any phase in the right half plane).
RD_HD void k01_scaled(cplx x, cplx& k0, cplx& k1) {
  const double ax = sqrt(x.re * x.re + x.im * x.im), key = ax + x.re;
  const cplx ix = crcp(x);
  if (key < 5.0) {
    const cplx z = 0.25 * (x * x);
    const cplx L = cx(log(0.5 * ax) + 0.57721566490153286061, atan2(x.im, x.re));   // ln(x/2) + Euler's gamma
    cplx t = cx(1.0, 0.0), i0 = t, i1 = t, s0 = cx(0.0, 0.0), s1 = t;
#pragma unroll 1
    for (int k = 1; k < 24; ++k) {
      const double a = RD_LAP.ik[k], b = RD_LAP.ik[k + 1];
      t = (a * a) * (t * z);                   // z^k / k!^2
      const cplx t1 = b * t;                   // z^k / (k! (k+1)!)
      i0 = i0 + t;
      i1 = i1 + t1;
      s0 = s0 + RD_LAP.ih[k] * t;
      s1 = s1 + (RD_LAP.ih[k] + RD_LAP.ih[k + 1]) * t1;
      if (fabs(t.re) + fabs(t.im) < 1e-18) break;
    }
    const cplx hx = 0.5 * x;
    const cplx a0 = s0 - L * i0, a1 = ix + L * (hx * i1) - 0.5 * (hx * s1);
    double sn, cs;
#ifdef __CUDA_ARCH__
    sincos(x.im, &sn, &cs);
#else
    sn = sin(x.im);
    cs = cos(x.im);
#endif
    const double e = exp(x.re);
    const cplx ex = cx(e * cs, e * sn);
    k0 = ex * a0;
    k1 = ex * a1;
    return;
  }
  int n = 12 + (int)(280.0 / key);
  if (n > kLapMiller) n = kLapMiller;
  cplx up = cx(0.0, 0.0), u = cx(1e-150, 0.0), sum = u;
  double n1 = n + 1.0;
  cplx b = cx(2.0 * (n + x.re), 2.0 * x.im);
#pragma unroll 1
  for (; n >= 1; --n) {
    const cplx v = RD_LAP.r[n] * (b * u - n1 * up);
    up = u;
    u = v;
    sum = sum + v;
    b.re -= 2.0;
    n1 -= 1.0;
  }
  // sqrt(pi / 2x): principal root (Re x > 0)
  const cplx q = (0.5 * kPi) * ix;
  const double aq = sqrt(q.re * q.re + q.im * q.im);
  const double sr = sqrt(0.5 * (aq + q.re));
  const cplx root = cx(sr, 0.5 * q.im / sr);
  const cplx iu = crcp(u);
  k0 = root * u * crcp(sum);
  k1 = k0 * ((cx(x.re + 0.5, x.im) - up * iu) * ix);
}

// e^{-x} I_0(x) for Re x > 0 (k0, k1 as from k01_scaled).  From Re x = 20 on the asymptotic series
// (Abramowitz & Stegun 9.7.1): the part it leaves out is e^{-2 Re x} < 5e-18 of it, and |x| >= 20 needs 27
// terms at most (checked against 40-digit values: below 1e-15).  Elsewhere from the Wronskian,
// I_0 = 1 / (x (K_1 + (I_1/I_0) K_0)), with the ratio from the downward recurrence of the minimal
// solution I_n, 24 + 1.5 |x| orders: at most 180 on the line below, where |x| <= 5.2 Re x, but thousands
// at small tau, where |x| grows like u / 2 tau (absorbing 2D system of 3000 particles, tau = 1e-5:
// 0.80 ms a step with the recurrence alone, 0.068 with the series).
RD_HD cplx i0_scaled(cplx x, cplx k0, cplx k1) {
  if (x.re >= 20.0) {
    const double q8 = 0.125 / (x.re * x.re + x.im * x.im);
    const cplx i8 = cx(x.re * q8, -x.im * q8);                    // 1 / 8x
    cplx t = cx(1.0, 0.0), sum = t;
#pragma unroll 1
    for (int k = 1; k < 40; ++k) {
      t = ((2.0 * k - 1.0) * (2.0 * k - 1.0) * RD_LAP.ik[k]) * (t * i8);
      sum = sum + t;
      if (fabs(t.re) + fabs(t.im) < 1e-17) break;
    }
    const cplx q = (4.0 / kPi) * i8;                              // 1 / 2 pi x: principal root
    const double sr = sqrt(0.5 * (sqrt(q.re * q.re + q.im * q.im) + q.re));
    return cx(sr, 0.5 * q.im / sr) * sum;
  }
  const cplx ix = crcp(x);
  const double ax = sqrt(x.re * x.re + x.im * x.im);
  cplx jp = cx(0.0, 0.0), j = cx(1e-100, 0.0);
#pragma unroll 1
  for (int n = 24 + (int)(1.5 * ax); n >= 1; --n) {
    const cplx jm = jp + (2.0 * n) * (ix * j);
    jp = j;
    j = jm;
    if (fabs(j.re) + fabs(j.im) > 1e100) {
      j = 1e-100 * j;
      jp = 1e-100 * jp;
    }
  }
  return ix * crcp(k1 + (jp * crcp(j)) * k0);
}

// Lane k's node of the line for the separation sum u = R + R0 - 2: w = c - i xi and the weight
// e^{tau (w - u/2tau)^2} (the integral over xi is h times the sum; the constant e^{-u^2/4tau} of
// e^{tau w^2 - u w} is left out).
struct LapNode {
  cplx w, wt;
  double h;
};
RD_HD LapNode lap_node(double u, double tau, int lane) {
  const double s = sqrt(tau), c0 = u / (2.0 * tau);
  const double d = fmax(0.0, 1.25 - s * c0) / s;
  LapNode k;
  k.h = sqrt(39.5) / (32.0 * s);
  const double xi = (lane + 0.5) * k.h;
  k.w = cx(c0 + d, -xi);
  const double e = exp(tau * (d - xi) * (d + xi)), ph = -2.0 * tau * d * xi;
  k.wt = cx(e * cos(ph), e * sin(ph));
  return k;
}

// ------------------------------------------------------------------------------------------------
// Partial-wave coefficients of the conditional angle
// ------------------------------------------------------------------------------------------------
// The sequences K_n, K_{n+1} (scaled) of one lane's node at the arguments w, R w, R0 w; the weight
// is folded into the R0 sequence.  step() returns the node's share of D_n and moves on to n + 1.
struct LapAng {
  cplx am;                      // K_{n-1} at w (n = 0: its continuation)
  cplx a, a1, b, b1, q, q1;     // K_n, K_{n+1} at w, R w, R0 w
  cplx iw, cw, cr, cq;          // 1/w; (2n+1)/z (3D) or 2n/z (2D) of K_{n+1}'s recurrence, per argument
  cplx dw, dr, dq;              // 2/z
  RD_HD void start(int dim, const LapNode& k, double R, double R0) {
    const cplx w = k.w, wr = R * w, wq = R0 * w;
    iw = crcp(w);
    const cplx ir = (1.0 / R) * iw, iq = (1.0 / R0) * iw;
    if (dim == 3) {
      a = iw; b = ir; q = iq;                                         // e^z k_0 = 1/z
      am = cx(0.0, 0.0);
      a1 = iw * (cx(1.0, 0.0) + iw); b1 = ir * (cx(1.0, 0.0) + ir); q1 = iq * (cx(1.0, 0.0) + iq);
      cw = iw; cr = ir; cq = iq;
    } else {
      k01_scaled(w, a, a1);
      k01_scaled(wr, b, b1);
      k01_scaled(wq, q, q1);
      am = a1;
      cw = cr = cq = cx(0.0, 0.0);
    }
    q = q * k.wt;
    q1 = q1 * k.wt;
    dw = 2.0 * iw; dr = 2.0 * ir; dq = 2.0 * iq;
  }
  // dn = n.  The derivative as the recurrence gives it, -(2n+1) k_n' = n k_{n-1} + (n+1) k_{n+1} (3D),
  // -2 K_n' = K_{n-1} + K_{n+1} (2D): the share comes out divided by 2n + 1 (3D) or by 2.
  RD_HD double step(bool d3, double dn) {
    const cplx kd = d3 ? dn * am + (dn + 1.0) * a1 : am + a1;
    const double c = re_quot(b * q, a * kd);
    cw = cw + dw; cr = cr + dr; cq = cq + dq;
    am = a;
    cplx t = am + cw * a1; a = a1; a1 = t;
    t = b + cr * b1; b = b1; b1 = t;
    t = q + cq * q1; q = q1; q1 = t;
    if (fabs(a.re) + fabs(a.im) > 1e60) {      // all three scaled alike: the quotient does not change
      am = 1e-60 * am; a = 1e-60 * a; a1 = 1e-60 * a1; b = 1e-60 * b; b1 = 1e-60 * b1; q = 1e-60 * q; q1 = 1e-60 * q1;
    }
    return c;
  }
};

// Orders that matter: beyond 9 sqrt(kappa) + 9 the coefficients are below 1e-17 of D_0 (largest for
// pairs at contact, where the law is closest to the free propagator's; checked for kappa 0.06..53).
RD_HD int lap_ang_terms(double kappa, int n_law) {
  const int n = (int)ceil(9.0 * sqrt(kappa) + 9.0);
  return n < n_law ? n : n_law;
}

// D_n / D_0 of the law at (R, R0, tau), n = 0 .. N, into Dn (shared memory of this warp, kAngNMax
// entries).  Returns the last order worth summing.  Warp-collective.
__device__ __forceinline__ int lap_ang_coeffs_warp(int dim, double R, double R0, double tau, int N, double* Dn) {
  const int lane = threadIdx.x & 31;
  const bool d3 = dim == 3;
  const LapNode k = lap_node(fmax(R + R0 - 2.0, 0.0), tau, lane);
  LapAng A;
  A.start(dim, k, R, R0);
  double dn = 0.0, c0 = 0.0;
  int last = 0, small = 0;
#pragma unroll 1
  for (int n = 0; n <= N; ++n) {
    const double c = warp_sum(A.step(d3, dn));
    dn += 1.0;
    if (n == 0) c0 = c;
    if (lane == 0) Dn[n] = c;
    last = n;
    small = fabs(c) < 1e-20 * fabs(c0) ? small + 1 : 0;
    if (small == 2) break;
  }
  __syncwarp();
  const double inv = 1.0 / c0;
  for (int n = lane; n <= last; n += 32) Dn[n] *= d3 ? (2 * n + 1) * inv : inv;
  __syncwarp();
  return last;
}

// CDF (and density) of the angle at this lane's own v from the coefficients (lanes may differ in v).
__device__ __forceinline__ void lap_ang_cdf(int dim, const double* Dn, int N, double v, double& F, double& f) {
  double acc = 0.0, den = 0.0;
  if (dim == 3) {
    double pm1 = 1.0, p = v;
#pragma unroll 1
    for (int n = 1; n <= N; ++n) {
      const double d = Dn[n];
      const double pp1 = c_lap.leg_a[n] * v * p - c_lap.leg_b[n] * pm1;
      acc += d * (pp1 - pm1);
      den += (2.0 * n + 1.0) * d * p;
      pm1 = p;
      p = pp1;
    }
    F = 0.5 * (1.0 + v) + 0.5 * acc;
    f = 0.5 * (1.0 + den);
    return;
  }
  double s1, c1;
  sincos(v, &s1, &c1);
  double sn = s1, cn = c1;
#pragma unroll 1
  for (int n = 1; n <= N; ++n) {
    const double d = Dn[n];
    acc += d * (sn * c_lap.ik[n]);
    den += d * cn;
    const double t = sn * c1 + cn * s1;
    cn = cn * c1 - sn * s1;
    sn = t;
  }
  F = (v + 2.0 * acc) * (1.0 / kPi);
  f = (1.0 + 2.0 * den) * (1.0 / kPi);
}

// The same in FP32 from the same coefficients (the starting point of the FP64 solution).
__device__ __forceinline__ void lap_ang_cdf_f(bool d3, const double* Dn, int N, float v, float& F, float& f) {
  float acc = 0.0f, den = 0.0f;
  if (d3) {
    float pm1 = 1.0f, p = v;
#pragma unroll 1
    for (int n = 1; n <= N; ++n) {
      const float d = (float)Dn[n];
      const float pp1 = (float)c_lap.leg_a[n] * v * p - (float)c_lap.leg_b[n] * pm1;
      acc += d * (pp1 - pm1);
      den += (2.0f * n + 1.0f) * d * p;
      pm1 = p;
      p = pp1;
    }
    F = 0.5f * (1.0f + v) + 0.5f * acc;
    f = 0.5f * (1.0f + den);
    return;
  }
  float s1, c1;
  sincosf(v, &s1, &c1);
  float sn = s1, cn = c1;
#pragma unroll 1
  for (int n = 1; n <= N; ++n) {
    const float d = (float)Dn[n];
    acc += d * (sn * (float)c_lap.ik[n]);
    den += d * cn;
    const float t = sn * c1 + cn * s1;
    cn = cn * c1 - sn * s1;
    sn = t;
  }
  F = (v + 2.0f * acc) * (float)(1.0 / kPi);
  f = (1.0f + 2.0f * den) * (float)(1.0 / kPi);
}

// Angle of the new separation to the start separation at CDF value U (3D its cosine in [-1, 1], 2D the
// angle in [0, pi]) from the full propagator.  NaN if the law needs more than kAngNMax - 1 partial
// waves.  Warp-collective, identical arguments in every lane; Dn: kAngNMax doubles of shared memory.
// Three rounds of 32 trial points in FP32 come within 1e-4 of the range, Newton steps in FP64 inside a
// bracket finish (the CDF is monotonic); an FP64 evaluation costs a warp about 8000 cycles.
__device__ __noinline__ double lap_ang_sample_warp(int dim, double U, double R, double R0, double tau, double* Dn) {
  const double kappa = R * R0 / (2.0 * tau);
  const int n_law = ang_terms(kappa);
  if (n_law > kAngNMax - 1) return NAN;
  __syncwarp();                                   // the previous pair's readers are done with Dn
  const int N = lap_ang_coeffs_warp(dim, R, R0, tau, lap_ang_terms(kappa, n_law), Dn);
  const int lane = threadIdx.x & 31;
  const float Uf = (float)U;
  float lof = dim == 3 ? -1.0f : 0.0f, hif = dim == 3 ? 1.0f : (float)kPi, Ff, ff;
#pragma unroll 1
  for (int round = 0; round < 3; ++round) {
    const float st = (hif - lof) * (1.0f / 33.0f);
    lap_ang_cdf_f(dim == 3, Dn, N, lof + (lane + 1) * st, Ff, ff);
    const int below = __popc(__ballot_sync(0xFFFFFFFFu, Ff < Uf));
    const float nlo = lof + below * st;
    hif = below < 32 ? lof + (below + 1) * st : hif;
    lof = nlo;
  }
  float vf = 0.5f * (lof + hif);
  lap_ang_cdf_f(dim == 3, Dn, N, vf, Ff, ff);
  if (ff > 0.0f) vf = fminf(fmaxf(vf - (Ff - Uf) / ff, lof), hif);
  double lo = dim == 3 ? -1.0 : 0.0, hi = dim == 3 ? 1.0 : kPi, F, f;
  double v = fmin(fmax((double)vf, lo), hi);
#pragma unroll 1
  for (int it = 0; it < 80; ++it) {
    lap_ang_cdf(dim, Dn, N, v, F, f);
    if (F < U)
      lo = v;
    else
      hi = v;
    double vn = f > 0.0 ? v - (F - U) / f : lo - 1.0;
    const bool inside = vn >= lo && vn <= hi;
    if (!inside) vn = 0.5 * (lo + hi);
    const double step = fabs(vn - v);
    v = vn;
    if (step <= (inside ? 4e-16 : 1e-16)) break;
    // quadratic convergence: a step below 1e-9 leaves an error below rounding
    if (inside && step <= 1e-9 * fmin(1.0, f)) break;
  }
  return v;
}

// ------------------------------------------------------------------------------------------------
// 2D radial quantities (n = 0)
// ------------------------------------------------------------------------------------------------
// Eq. (bayes1D) in 2D: p_enc = e^{-(R-1)(R0-1)/tau} (4 tau/pi) h Sum Re[wt w I0/K0 K0(wR) K0(wR0)]
// / I0e(R R0/2tau), all functions scaled.  Warp-collective.
__device__ __noinline__ double lap_p_enc2_warp(double R, double R0, double tau) {
  if (R <= 1.0 || R0 <= 1.0) return 1.0;
  const LapNode k = lap_node(R + R0 - 2.0, tau, threadIdx.x & 31);
  cplx a, a1, b, b1, q, q1;
  k01_scaled(k.w, a, a1);
  k01_scaled(R * k.w, b, b1);
  k01_scaled(R0 * k.w, q, q1);
  const cplx i0 = i0_scaled(k.w, a, a1);
  const double S = k.h * warp_sum(re_quot(k.wt * (k.w * (i0 * (b * q))), a));
  const double p = exp(-(R - 1.0) * (R0 - 1.0) / tau) * (4.0 * tau / kPi) * S / i0e_d(R * R0 / (2.0 * tau));
  return p < 0.0 ? 0.0 : (p > 1.0 ? 1.0 : p);
}

// FP32 value that the FP64 step's encounter draw must lie below for the pair to need its exact p_enc,
// from the contact distances d = R - 1 > 0 and d0 = R0 - 1 computed in FP32.
// 3D: the FP32 closed form.  2D: a closed upper bound: u(R) = sqrt(R) g obeys the 1D diffusion equation
// plus the growth term u / 4R^2, so g_abs is at least the 1D absorbing kernel over sqrt(R R0),
//   1 - p_enc >= (1 - e^{-d d0/tau}) / m,  m = sqrt(2 pi z) e^{-z} I0(z), z = R R0/2tau.
// Margin: with e = 2^-24, the squared length, the root, the contact radius and its reciprocal leave
// each distance within 6e (1 + d) of its value, so the exponent x = d d0 / tau is within
// 6e ((d + d0)/tau + 2x) and p <= e^{-x} within that times p, which grows like 1/sqrt(tau): at
// tau = 1e-7 up to 1e-3.  The first part of the margin is 5e-7 (d + d0)/tau (6e = 3.6e-7); the 1e-4 are
// far above the rest: 2x e^{-x} 6e < 3e-7 and a few e of the factors (in 2D also where m < 1, since
// x e^{-x}/m <= (1 - e^{-x})/m <= 1, and (d + d0)/(tau m) < 12 there).
__device__ __forceinline__ float p_enc_screen(int dim, float d, float d0, float inv_tau) {
  if (d0 <= 0.0f) return 2.0f;
  const float margin = 1e-4f + 5e-7f * (d + d0) * inv_tau;
  if (dim == 3) return p_enc3_f(d, d0, inv_tau) + margin;
  const float z = (1.0f + d) * (1.0f + d0) * 0.5f * inv_tau;
  const float m = z < 40.0f ? sqrtf(6.2831853f * z) * expf(-z) * cyl_bessel_i0f(z)
                            : 1.0f + 0.125f / z + 0.0703125f / (z * z) + 0.0732422f / (z * z * z);
  return 1.0f + expm1f(-d * d0 * inv_tau) / m + margin;
}

// Eq. (psurv_radII) in 2D.  Warp-collective.
__device__ __noinline__ double lap_p_reac2_warp(double R, double R0, double tau, double h) {
  R = fmax(R, 1.0);
  R0 = fmax(R0, 1.0);
  const LapNode k = lap_node(R + R0 - 2.0, tau, threadIdx.x & 31);
  cplx a, a1, b, b1, q, q1;
  k01_scaled(k.w, a, a1);
  k01_scaled(R * k.w, b, b1);
  k01_scaled(R0 * k.w, q, q1);
  const cplx num = k.wt * (b * q);
  const double sn = h * warp_sum(re_quot(num, a1 * (k.w * a1 + h * a)));
  const double sd = warp_sum(re_quot(num, a * a1));
  const double p = sn / sd;
  return p < 0.0 ? 0.0 : (p > 1.0 ? 1.0 : p);
}

// New separation R' >= 1 of an encountered 2D pair at tail fraction U of the radial law: the tail
// beyond 1 + V is, with R K_1(wR)/w the antiderivative of R K_0(wR),
//   T(V) = Sum Re[wt R' K_1(wR') K_0(wR0) / (w K_0 K_1)] e^{-u^2/4tau} over the same at V = 0 (where
// K_1 cancels), and -dT/dV has R' K_0(wR') in the place of R' K_1(wR')/w.  Newton on ln T inside a
// bracket; the line is that of the current V and kept while V moves less than half a sqrt(tau).
// Warp-collective.
__device__ __noinline__ double lap_resample2_warp(double U, double R0, double tau, double v_seed) {
  if (R0 < 1.0) R0 = 1.0;
  const double s = sqrt(tau), w0 = R0 - 1.0;
  const int lane = threadIdx.x & 31;
  double ln_tot;
  {
    const LapNode k = lap_node(w0, tau, lane);
    cplx a, a1, q, q1;
    k01_scaled(k.w, a, a1);
    k01_scaled(R0 * k.w, q, q1);
    ln_tot = log(warp_sum(re_quot(k.wt * q, k.w * a))) - w0 * w0 / (4.0 * tau);
  }
  const double target = log(U) + ln_tot;
  double lo = 0.0, hi = R0 + 13.0 * s, V = fmin(fmax(v_seed, 0.0), hi);
  double v_line = -1.0;
  LapNode k{};
  cplx f{};                    // wt K_0(wR0) / (K_0(w) K_1(w)) on the current line
#pragma unroll 1
  for (int it = 0; it < 100; ++it) {
    const double R = 1.0 + V;
    if (v_line < 0.0 || fabs(V - v_line) > 0.5 * s) {
      v_line = V;
      k = lap_node(V + w0, tau, lane);
      cplx a, a1, q, q1;
      k01_scaled(k.w, a, a1);
      k01_scaled(R0 * k.w, q, q1);
      f = (k.wt * q) * crcp(a * a1);
    }
    // off the line's own V the factor e^{-w (V - v_line)} is explicit
    const double dv = V - v_line;
    const double e = exp(-k.w.re * dv);
    double sn, cs;
    sincos(-k.w.im * dv, &sn, &cs);
    cplx b, b1;
    k01_scaled(R * k.w, b, b1);
    const cplx g = cx(e * cs, e * sn) * f;
    const double den = R * warp_sum((g * b).re);
    const double tail = R * warp_sum((g * (b1 * crcp(k.w))).re);
    const double u = v_line + w0;
    const double y = log(tail) - u * u / (4.0 * tau) - target;     // ln T - ln U, falls with V
    if (y > 0.0)
      lo = V;
    else
      hi = V;
    double Vn = tail > 0.0 && den > 0.0 ? V + y * tail / den : -1.0;
    // (a step that rounds to the bracket's end has converged)
    const bool inside = Vn >= lo && Vn <= hi;
    if (!inside) Vn = 0.5 * (lo + hi);
    const double step = fabs(Vn - V);
    V = Vn;
    if (inside && step <= 1e-9 * fmax(V, s)) break;
    if (hi - lo <= 4e-16 * fmax(hi, s)) break;
  }
  return 1.0 + V;
}

}  // namespace rd
