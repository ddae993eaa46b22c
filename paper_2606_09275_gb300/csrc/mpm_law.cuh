// Hencky / return-map law shared by the assembly and the adjoint kernels
// (Sec. 2.2; model 3, the CPT material's Willam-Warnke cone, Sec. 6.4):
// principal-space return in Kirchhoff stress, 3x3 symmetric
// eigen-decomposition, divided difference of the logarithm.
#pragma once
#include "mpm_internal.cuh"

namespace mpm {

struct Law {
  int model;
  double nu, eta, xi, etab;
  double cmu, clm;  // Lame constants per unit E: 1 / (2 (1 + nu)), nu / ((1 + nu) (1 - 2 nu))
  double ecc;  // model 3: tensile / compressive meridian radius, (3 - sin phi)/(3 + sin phi)
};

// Willam-Warnke deviatoric section (Sec. 6.4): r(theta) by the elliptic
// interpolation r = (4 a c^2 + b^2)/(2 a c + b sqrt(4 a c^2 + 5 e^2 - 4 e)),
// c = cos(theta), a = 1 - e^2, b = 2 e - 1 (theta the Lode angle, 0 on the
// tensile meridian where r = 1/e, pi/3 on the compressive one where r = 1),
// and dr/dzeta for zeta = cos(3 theta); at the compressive meridian the limit
// 4 a / (6 b^2 (2 c + 1)) of dr/dc over dzeta/dc is taken
__device__ inline double ww_section(double zeta, double e, double* drdz) {
  zeta = fmin(fmax(zeta, -1.0), 1.0);
  double c = cos(acos(zeta) / 3.0);
  double a = 1.0 - e * e, b = 2.0 * e - 1.0;
  double w = sqrt(4.0 * a * c * c + 5.0 * e * e - 4.0 * e);
  double N = 4.0 * a * c * c + b * b, D = 2.0 * a * c + b * w;
  double dN = 8.0 * a * c, dD = 2.0 * a + 4.0 * a * b * c / w;
  double rc = (dN * D - N * dD) / (D * D);
  double q = 4.0 * c * c - 1.0;
  *drdz = fabs(q) > 1e-5 ? rc / (3.0 * q) : 4.0 * a / (6.0 * b * b * (2.0 * c + 1.0));
  return N / D;
}

// one Jacobi rotation in the plane (P, Q_) of the symmetric A = diag(d) plus
// the off-diagonal a (a[0] = A01, a[1] = A02, a[2] = A12), columns of Q along
template <int P, int Q_, class T>
__device__ inline void jacobi_rotate(T* d, T* a, T* Q) {
  constexpr int O = 3 - P - Q_, PQ = P + Q_ - 1, OP = O + P - 1, OQ = O + Q_ - 1;
  T apq = a[PQ];
  if (apq == (T)0) return;
  // tan of the rotation angle, smaller root of t^2 + (h / apq) t - 1 = 0
  T h = d[Q_] - d[P], th = (T)0.5 * h / apq;
  T t = fabs(th) > (sizeof(T) == 8 ? (T)1e150 : (T)1e18) ? (T)0.5 / th
                                                          : copysign((T)1, th) / (fabs(th) + sqrt(th * th + (T)1));
  T cs = rsqrt(t * t + (T)1), sn = t * cs;
  d[P] -= t * apq;
  d[Q_] += t * apq;
  a[PQ] = (T)0;
  T aop = a[OP], aoq = a[OQ];
  a[OP] = cs * aop - sn * aoq;
  a[OQ] = sn * aop + cs * aoq;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    T qp = Q[3 * k + P], qq = Q[3 * k + Q_];
    Q[3 * k + P] = cs * qp - sn * qq;
    Q[3 * k + Q_] = sn * qp + cs * qq;
  }
}

// the same rotation for |apq / h| <= 1e-4, without its two square roots and
// one of its divisions: t = apq / h up to t^3 (what stays of apq is 1e-8 of
// it, for the next sweep), c = 1 - t^2 / 2 and s = t c up to t^4 (1e-16)
template <int P, int Q_>
__device__ inline void jacobi_nudge(double* d, double* a, double* Q, double t) {
  constexpr int O = 3 - P - Q_, PQ = P + Q_ - 1, OP = O + P - 1, OQ = O + Q_ - 1;
  double apq = a[PQ], t2 = t * t;
  double cs = fma(-0.5, t2, 1.0), sn = t * cs;
  d[P] = fma(-t, apq, d[P]);
  d[Q_] = fma(t, apq, d[Q_]);
  a[PQ] = -apq * t2;
  double aop = a[OP], aoq = a[OQ];
  a[OP] = fma(cs, aop, -sn * aoq);
  a[OQ] = fma(sn, aop, cs * aoq);
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    double qp = Q[3 * k + P], qq = Q[3 * k + Q_];
    Q[3 * k + P] = fma(cs, qp, -sn * qq);
    Q[3 * k + Q_] = fma(sn, qp, cs * qq);
  }
}

template <int P, int Q_>
__device__ inline void jacobi_step(double* d, double* a, double* Q) {
  constexpr int PQ = P + Q_ - 1;
  double h = d[Q_] - d[P], t = a[PQ] == 0.0 ? 0.0 : a[PQ] / h;
  if (fabs(t) <= 1e-4)
    jacobi_nudge<P, Q_>(d, a, Q, t);
  else
    jacobi_rotate<P, Q_>(d, a, Q);
}

// quaternion q <- q (x) the rotation that jacobi_rotate<P, Q_> applies to the
// columns (by its angle about the third axis), on FP32; A as there
template <int P, int Q_>
__device__ inline void jacobi_seed(float* d, float* a, float* q) {
  constexpr int O = 3 - P - Q_, PQ = P + Q_ - 1, OP = O + P - 1, OQ = O + Q_ - 1;
  float apq = a[PQ];
  float h = d[Q_] - d[P];
  if (fabsf(apq) <= 1e-9f * (fabsf(d[P]) + fabsf(d[Q_]))) return;
  float th = 0.5f * h / apq;
  float t = copysignf(1.f, th) / (fabsf(th) + sqrtf(th * th + 1.f));
  if (!(t == t) || fabsf(th) > 1e18f) t = 0.f;
  float cs = rsqrtf(t * t + 1.f), sn = t * cs;
  d[P] -= t * apq;
  d[Q_] += t * apq;
  a[PQ] = 0.f;
  float aop = a[OP], aoq = a[OQ];
  a[OP] = cs * aop - sn * aoq;
  a[OQ] = sn * aop + cs * aoq;
  // half angle; the rotation's sense about axis O is negative but for (0, 2)
  float ch = sqrtf(0.5f * (1.f + cs)), sh = (O == 1 ? 0.5f : -0.5f) * sn / ch;
  float w = q[0], x = q[1], y = q[2], z = q[3];
  if (O == 0) {
    q[0] = w * ch - x * sh, q[1] = w * sh + x * ch, q[2] = y * ch + z * sh, q[3] = z * ch - y * sh;
  } else if (O == 1) {
    q[0] = w * ch - y * sh, q[1] = x * ch - z * sh, q[2] = w * sh + y * ch, q[3] = x * sh + z * ch;
  } else {
    q[0] = w * ch - z * sh, q[1] = x * ch + y * sh, q[2] = y * ch - x * sh, q[3] = w * sh + z * ch;
  }
}

// symmetric 3x3 eigen-decomposition; columns of Q are the eigenvectors
// (Q[3*i + a] = component i of vector a).  Cyclic Jacobi rotations, as many
// sweeps as it takes, but started from the eigenvectors of the deviator that
// FP32 Jacobi sweeps find (as a quaternion, so that the FP64 start is
// orthonormal to rounding): FP64 instructions are the cost of the point
// kernels here (16 SM cycles each, against a quarter for FP32), and from the
// start two sweeps of three small rotations (32 instructions) finish, where
// the identity takes four of full ones (65).  A million matrices of strains of
// 1e-2: 1.40 ms from the identity, 0.65 ms so, with smaller errors
// (|Q^T Q - I| 2.2e-16 in the mean against 3.3e-16); of nearly equal
// eigenvalues, which FP32 cannot tell apart, 1.00 and 1.03 ms.
__device__ inline void jacobi3(double* A, double* lam, double* Q) {
  double m = (A[0] + A[4] + A[8]) * (1.0 / 3.0);
  double d[3] = {A[0] - m, A[4] - m, A[8] - m}, a[3] = {A[1], A[2], A[5]};
  auto done = [&] {
    double off = fma(a[0], a[0], fma(a[1], a[1], a[2] * a[2]));
    double on = fma(d[0], d[0], fma(d[1], d[1], fma(d[2], d[2], 3.0 * m * m)));
    return off == 0.0 || off <= 1e-36 * on;
  };
  if (done()) {
#pragma unroll
    for (int i = 0; i < 9; ++i) Q[i] = i % 4 == 0 ? 1.0 : 0.0;
    lam[0] = A[0];
    lam[1] = A[4];
    lam[2] = A[8];
    return;
  }
  float df[3], af[3], q[4] = {1.f, 0.f, 0.f, 0.f}, big = 0.f;
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    df[i] = (float)d[i];
    af[i] = (float)a[i];
    big = fmaxf(big, fmaxf(fabsf(df[i]), fabsf(af[i])));
  }
  if (big > 1e-30f && big < 1e30f) {
    float sc = 1.f / big;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      df[i] *= sc;
      af[i] *= sc;
    }
    for (int sweep = 0; sweep < 6; ++sweep) {
      if (fabsf(af[0]) + fabsf(af[1]) + fabsf(af[2]) < 1e-9f) break;
      jacobi_seed<0, 1>(df, af, q);
      jacobi_seed<0, 2>(df, af, q);
      jacobi_seed<1, 2>(df, af, q);
    }
  }
  double w = q[0], x = q[1], y = q[2], z = q[3];
  // 2 / |q|^2 for |q|^2 = 1 + e, e some 1e-6
  double e = fma(w, w, fma(x, x, fma(y, y, fma(z, z, -1.0))));
  double k = fma(fma(fma(-2.0, e, 2.0), e, -2.0), e, 2.0);
  double xs = k * x, ys = k * y, zs = k * z;
  double xx = x * xs, yy = y * ys, zz = z * zs, xy = x * ys, xz = x * zs, yz = y * zs;
  Q[0] = 1.0 - (yy + zz); Q[1] = fma(-w, zs, xy); Q[2] = fma(w, ys, xz);
  Q[3] = fma(w, zs, xy); Q[4] = 1.0 - (xx + zz); Q[5] = fma(-w, xs, yz);
  Q[6] = fma(-w, ys, xz); Q[7] = fma(w, xs, yz); Q[8] = 1.0 - (xx + yy);
  // Q^T (A - m I) Q
  double T[9];
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    T[j] = fma(d[0], Q[j], fma(a[0], Q[3 + j], a[1] * Q[6 + j]));
    T[3 + j] = fma(a[0], Q[j], fma(d[1], Q[3 + j], a[2] * Q[6 + j]));
    T[6 + j] = fma(a[1], Q[j], fma(a[2], Q[3 + j], d[2] * Q[6 + j]));
  }
  auto qt = [&](int i, int j) { return fma(Q[i], T[j], fma(Q[3 + i], T[3 + j], Q[6 + i] * T[6 + j])); };
  d[0] = qt(0, 0); d[1] = qt(1, 1); d[2] = qt(2, 2);
  a[0] = qt(0, 1); a[1] = qt(0, 2); a[2] = qt(1, 2);
  for (int sweep = 0; sweep < 40; ++sweep) {
    if (done()) break;
    jacobi_step<0, 1>(d, a, Q);
    jacobi_step<0, 2>(d, a, Q);
    jacobi_step<1, 2>(d, a, Q);
  }
#pragma unroll
  for (int i = 0; i < 3; ++i) lam[i] = m + d[i];
}

// log(1 + x) / x for |x| <= 1/16 by its Taylor series (the first term left
// out is x^14 / 15, below 1e-18)
__device__ inline double log1p_over(double x) {
  double s = -1.0 / 14.0;
  s = fma(s, x, 1.0 / 13.0);
  s = fma(s, x, -1.0 / 12.0);
  s = fma(s, x, 1.0 / 11.0);
  s = fma(s, x, -1.0 / 10.0);
  s = fma(s, x, 1.0 / 9.0);
  s = fma(s, x, -1.0 / 8.0);
  s = fma(s, x, 1.0 / 7.0);
  s = fma(s, x, -1.0 / 6.0);
  s = fma(s, x, 1.0 / 5.0);
  s = fma(s, x, -1.0 / 4.0);
  s = fma(s, x, 1.0 / 3.0);
  s = fma(s, x, -1.0 / 2.0);
  return fma(s, x, 1.0);
}

// natural logarithm, half the instructions near 1, where the stretches of a
// load step are
__device__ inline double log_stretch(double v) {
  double x = v - 1.0;
  return fabs(x) <= 0.0625 ? x * log1p_over(x) : log(v);
}

// divided difference of the logarithm: (ln a - ln b)/(a - b), 1/b in the limit
__device__ inline double ln_divdiff(double a, double b) {
  double ib = 1.0 / b, x = (a - b) * ib;
  return fabs(x) <= 0.0625 ? log1p_over(x) * ib : log1p(x) / (a - b);
}

// principal-space return: trial strains e -> tau_a, tangent d_ab = dtau_a/deps_b,
// shear ratio g = (tau_a - tau_b)/(eps_a - eps_b); Hencky moduli from E, nu
__device__ inline void principal_return(const Law& L, double E, double ys, const double* e, double* ta,
                                 double* dd, double* gr) {
  const double third = 1.0 / 3.0;
  double mu = E * L.cmu;
  double lm = E * L.clm;
  double kb = lm + 2.0 * third * mu;
  double tr = e[0] + e[1] + e[2], em = tr * third;
  double dev[3] = {e[0] - em, e[1] - em, e[2] - em};
  double dn = sqrt(dev[0] * dev[0] + dev[1] * dev[1] + dev[2] * dev[2]);
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    ta[a] = kb * tr + 2.0 * mu * dev[a];
#pragma unroll
    for (int b = 0; b < 3; ++b) dd[3 * a + b] = lm + (a == b ? 2.0 * mu : 0.0);
  }
  *gr = 2.0 * mu;
  if (L.model == 1) {
    // von Mises: q = sqrt(3/2)|s|, radial return onto q = ys
    double q = 1.224744871391589 * 2.0 * mu * dn;
    if (q <= ys) return;
    double fac = ys / q, g = 2.0 * mu * fac;
    double n0 = dev[0] / dn, n1 = dev[1] / dn, n2 = dev[2] / dn;
    double nn[3] = {n0, n1, n2};
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      ta[a] = kb * tr + g * dev[a];
#pragma unroll
      for (int b = 0; b < 3; ++b) dd[3 * a + b] = kb + g * ((a == b ? 1.0 : 0.0) - 1.0 / 3.0 - nn[a] * nn[b]);
    }
    *gr = g;
  } else if (L.model == 2 || L.model == 3) {
    // Drucker-Prager cone: f = sqrt(J2) r + eta p - xi c with r = 1 (model 2)
    // or the Willam-Warnke section r(theta) (model 3); potential sqrt(J2) +
    // etab p, circular, so the return is radial in the deviatoric plane and
    // keeps theta: f(dg) = (sqrt(J2) - G dg) r + eta (p - K etab dg) - xi c
    double G = mu, pm = kb * tr;
    double sj = 1.4142135623730951 * G * dn;
    double r = 1.0, drz = 0.0, dz[3] = {0.0, 0.0, 0.0};
    if (L.model == 3 && dn > 0.0) {
      // zeta = cos(3 theta) = 3 sqrt6 e1 e2 e3 / |e|^3 of the trial deviator
      double pr = dev[0] * dev[1] * dev[2], dn3 = dn * dn * dn;
      double zeta = 7.348469228349534 * pr / dn3;
      r = ww_section(zeta, L.ecc, &drz);
      if (zeta > -1.0 && zeta < 1.0) {
        double mm[3] = {dev[1] * dev[2], dev[0] * dev[2], dev[0] * dev[1]};
        double M3 = (mm[0] + mm[1] + mm[2]) / 3.0;
#pragma unroll
        for (int b = 0; b < 3; ++b)
          dz[b] = 7.348469228349534 * ((mm[b] - M3) / dn3 - 3.0 * pr * dev[b] / (dn3 * dn * dn));
      }
    }
    double f = sj * r + L.eta * pm - L.xi * ys;
    if (f <= 0.0) return;
    double den = G * r + kb * L.eta * L.etab;
    double dg = f / den;
    if (sj - G * dg >= 0.0 && dn > 0.0) {
      double ratio = 1.0 - G * dg / sj;
      double pn = pm - kb * L.etab * dg;
      double nn[3] = {dev[0] / dn, dev[1] / dn, dev[2] / dn};
      double ddg[3];
#pragma unroll
      for (int b = 0; b < 3; ++b)
        ddg[b] = (1.4142135623730951 * G * nn[b] * r + (sj - G * dg) * drz * dz[b] + L.eta * kb) / den;
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        ta[a] = pn + 2.0 * G * ratio * dev[a];
#pragma unroll
        for (int b = 0; b < 3; ++b) {
          double pd = (a == b ? 1.0 : 0.0) - 1.0 / 3.0;
          dd[3 * a + b] = 2.0 * G * pd -
                          1.4142135623730951 * G * (nn[a] * ddg[b] + dg * (pd - nn[a] * nn[b]) / dn) +
                          kb * (1.0 - L.etab * ddg[b]);
        }
      }
      *gr = 2.0 * G * ratio;
    } else {
      double pa = L.xi * ys / L.eta;
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        ta[a] = pa;
#pragma unroll
        for (int b = 0; b < 3; ++b) dd[3 * a + b] = 0.0;
      }
      *gr = 0.0;
    }
  }
}

inline Law make_law(const mpm_material& mat) {
  Law L{};
  L.model = mat.model;
  L.nu = mat.nu;
  L.cmu = 1.0 / (2.0 * (1.0 + mat.nu));
  L.clm = mat.nu / ((1.0 + mat.nu) * (1.0 - 2.0 * mat.nu));
  double sp = sin(mat.phi), ss = sin(mat.psi);
  L.eta = 6.0 * sp / (sqrt(3.0) * (3.0 - sp));
  L.xi = 6.0 * cos(mat.phi) / (sqrt(3.0) * (3.0 - sp));
  L.etab = 6.0 * ss / (sqrt(3.0) * (3.0 - ss));
  L.ecc = (3.0 - sp) / (3.0 + sp);
  return L;
}

}  // namespace mpm
