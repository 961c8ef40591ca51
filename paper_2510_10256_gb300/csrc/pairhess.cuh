// pairhess.cuh -- barrier gradient and PSD-projected Hessian of one active
// pair in closed form.
//
// Let d = |r| be the distance of a point-edge, point-triangle-face or
// line-line pair, r the vector between the closest points, n = r / d,
// beta = kappa b''(y) >= 0 and lam = -kappa b'(y) >= 0 (the barrier falls and
// is convex below its width).  Writing d as the minimum over the closest-point
// parameters and expanding to second order (the parameters' first-order change
// eliminated), with a = sum_q c_q dx_q the displacement of r at fixed
// parameters, c the closest-point weights,
//   grad d . dx = n . a,
//   dx^T (hess d) dx = -d |K^T y|^2 - 2 (K^T y) . a_par        (face, line-line)
//   dx^T (hess d) dx = a_3^2 / d - d (s y)^2 - 2 (s y) a_1     (point-edge)
// where a_par is a's part in the plane of the two edge vectors (a_1: along the
// edge, a_3: across edge and n), y the coordinates of the points' motion along
// n in a basis of the zero-sum weights, and K (2x2; s for one edge) takes y to
// the dual edge vectors.  So on the few motions that matter -- c / |c| along
// the plane's axes, the basis of zero-sum weights along n -- the Hessian of
// the barrier is, with mu = |c| and m = the coordinates of c,
//   T = [[0, lam mu K^T], [lam mu K, lam d K K^T + beta m m^T]],
// zero on every other motion (the a_3^2 term is -lam a_3^2 / d: negative, so
// its projection is zero).  K's singular values s_1 >= s_2 > 0 turn T into two
// 2x2 blocks and a zero, diagonalisable by hand, plus the rank-one beta m m^T:
// T has exactly as many negative eigenvalues as K has columns, each the only
// root of a secular equation between two known poles, and its eigenvector is
// rational in the root.  The projection is T - sum (negative eigenpairs).
//
// This replaces an iterative 9x9 (3x3 for point-edge) eigenproblem per pair.
// The Hessian stage is bound by the FP64 pipe (one warp instruction per 16
// cycles and SM at best, a 64th of the FP32 rate): the roots are found in FP32 by
// an iteration whose model has the equation's poles, and polished to FP64 by
// two Newton steps whose slopes come from FP32.  All poles, gaps and sums are
// formed from terms of one sign, so the roots and every component of the
// eigenvectors are accurate to a few ulp, however the pair is graded.
//
// Measured on GB300, the Hessian kernels of one pass (from the derivatives and
// an FP32 + FP64 Jacobi eigenproblem per pair, three kernels and their queues
// in memory, to one kernel): pleated 256x256 sheet (862k active pairs, 153k of
// them face / line-line) 5.56 -> 0.98 ms; 64 rod scenes (1.01M active, 243k)
// 7.11 -> 1.36 ms; two 12x12 layers (9.6k, 577) 0.67 -> 0.09 ms, where one
// thread's chain of Jacobi sweeps had set the time.  Against 40-digit results
// the largest error of a face / line-line block, relative to its largest
// entry, is 3 to 10 times below the eigenproblem's for edges at angles of
// 0.1 to 1e-7 (1e-14 against 6e-14 at 0.01; both grow as 1 / angle), and
// point-edge blocks stay at 1e-15 down to gaps of 1e-6 of the edge.
#pragma once
#include "common.cuh"

namespace cbh {

#ifdef __CUDA_ARCH__
__device__ __forceinline__ double hd_rsqrt(double v) { return rsqrt(v); }
#else
inline double hd_rsqrt(double v) { return 1.0 / sqrt(v); }
#endif

// 1 / v for v within FP32 range: the FP32 reciprocal refined by two Newton
// steps (relative error squared each time)
__host__ __device__ __forceinline__ double rcp_refined(double v) {
  double r = (double)(1.f / (float)v);
  r = fma(r, fma(-v, r, 1.0), r);
  return fma(r, fma(-v, r, 1.0), r);
}

// Bounds of the odds x the FP32 root finders return.  An eigenvector whose
// root lies closer to a pole than this is that pole's axis to FP64 rounding.
constexpr float ODDS_LO = 1e-30f, ODDS_HI = 1e30f;

// The next odds of a root between two poles: the model c + S (1 + x) - B (1 + 1/x)
// = 0 (S, B > 0), else the middle (in the exponent) of the bracket.
__host__ __device__ __forceinline__ float next_odds(float c, float S, float B, float lo, float hi) {
  float m = c + S - B;
  const float sc = 1.f / fmaxf(fabsf(m), fmaxf(S, B));
  m *= sc;
  S *= sc;
  B *= sc;
  const float D = sqrtf(m * m + 4.f * S * B);
  float x = m > 0.f ? 2.f * B / (m + D) : (D - m) / (2.f * S);
  if (!(x > lo && x < hi)) x = sqrtf(lo) * sqrtf(hi);
  return fminf(fmaxf(x, ODDS_LO), ODDS_HI);
}

constexpr int ODDS_ITERS = 40;        // a bound; a handful suffice away from extreme gradings
constexpr float ODDS_TOL = 2e-5f;     // squared twice by the FP64 steps

// The scaled problem of a face / line-line pair (unit lam mu s_1): blocks
// [[0, 1], [1, e1]] and rho [[0, 1], [1, e1 rho]] with eigenvalues -v_i < 0 < p_i,
// g = v_1 - v_2, and the rank-one coefficients b_i.
struct Secular {
  double v1, p1, v2, p2, g, b1, b2, b3;
};

// F(v) = 1 + b3/v + b1 v/((v - v1)(v + p1)) + b2 v/((v - v2)(v + p2)) vanishes
// once in (v2, v1) and once in (0, v2).  Root B: v = v1 - t = v2 + u, t + u = g,
// odds x = t / u.  Root A: t = v2 - v, odds x = v / t.
__host__ __device__ __forceinline__ float odds_b(float v1, float p1, float v2, float p2, float g, float b1, float b2,
                                                 float b3) {
  float lo = ODDS_LO, hi = ODDS_HI, x = 1.f;
  for (int it = 0; it < ODDS_ITERS; ++it) {
    const float u = g / (1.f + x), t = u * x, v = x < 1.f ? v1 - t : v2 + u;
    const float i1 = 1.f / (v + p1), i2 = 1.f / (v + p2), iv = 1.f / v;
    // b / g first: t and u may be far below b in exponent
    const float w = 1.f + x, g1 = (b1 / g) * v * i1 * (w / x), g2 = (b2 / g) * v * i2 * w;
    const float f = 1.f + b3 * iv + g2 - g1;
    if (f < 0.f) lo = x;
    else hi = x;
    const float e1 = t * p1 * iv * i1, e2 = u * p2 * iv * i2, B = b3 * iv * u * iv;
    const float xn = next_odds(1.f + b3 * iv - B + g2 * e2 + g1 * e1, (g2 * (1.f - e2) + B) / w, g1 * (1.f + e1) * x / w,
                               lo, hi);
    const float dx = fabsf(xn - x);
    x = xn;
    if (dx <= ODDS_TOL * x) break;
  }
  return x;
}
__host__ __device__ __forceinline__ float odds_a(float v1, float p1, float v2, float p2, float g, float b1, float b2,
                                                 float b3) {
  float lo = ODDS_LO, hi = ODDS_HI, x = 1.f;
  for (int it = 0; it < ODDS_ITERS; ++it) {
    const float t = v2 / (1.f + x), v = t * x;
    const float i1 = 1.f / (v + p1), i2 = 1.f / (v + p2), iv = 1.f / v, ig = 1.f / (g + t);
    const float g1 = b1 * v * i1 * ig, g2 = b2 * i2 * x;
    const float f = 1.f + b3 * iv - g1 - g2;
    if (f > 0.f) lo = x;
    else hi = x;
    const float e1 = t * p1 * iv * i1, e2 = t * p2 * iv * i2;
    const float c = 1.f + g2 * e2 + g1 * (e1 - g * ig), S = (g2 * (1.f + e2) + g1 * (e1 + t * ig)) / (1.f + x);
    const float xn = next_odds(-c, S, b3 / v2, lo, hi);
    const float dx = fabsf(xn - x);
    x = xn;
    if (dx <= ODDS_TOL * x) break;
  }
  return x;
}

// One damped Newton step on the odds in the exponent, f / (df / dln x) in FP32
__host__ __device__ __forceinline__ double odds_step(double x, double f, float df) {
  const float s = (float)f / df;
  return fma(x, -(double)fminf(fmaxf(s, -0.5f), 0.5f), x);
}

// The two negative eigenvalues' magnitudes and the eigenvectors' components
// (x1, x2, y1, y2, y3), unnormalised, for the coefficients q of the rank-one term.
__host__ __device__ __forceinline__ void secular_vectors(const Secular& s, double rho, const double (&q)[3],
                                                         double (&nu)[2], double (&V)[2][5]) {
  const float v1 = (float)s.v1, p1 = (float)s.p1, v2 = (float)s.v2, p2 = (float)s.p2, g = (float)s.g;
  const float b1 = (float)s.b1, b2 = (float)s.b2, b3 = (float)s.b3;
  {
    double x = (double)odds_b(v1, p1, v2, p2, g, b1, b2, b3);
    double r1 = 0.0, r2 = 0.0, v = 0.0, iv = 0.0;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const double iw = rcp_refined(1.0 + x), u = s.g * iw, t = u * x;
      v = x < 1.0 ? s.v1 - t : s.v2 + u;
      r1 = 1.0 / (t * (v + s.p1));
      r2 = 1.0 / (u * (v + s.p2));
      iv = rcp_refined(v);
      if (k == 2) break;
      const double g1 = s.b1 * v * r1, g2 = s.b2 * v * r2, f = 1.0 + s.b3 * iv + (g2 - g1);
      const float tf = (float)t, uf = (float)u, vf = (float)v, ivf = (float)iv;
      const float e1 = tf * p1 * ivf / (vf + p1), e2 = uf * p2 * ivf / (vf + p2);
      // dF/dln x = (t u / g) (g1'/... ): every term positive
      const float df = (float)g1 * (1.f + e1) * (uf / g) + ((float)g2 * (1.f - e2) + b3 * ivf * ivf * uf) * (tf / g);
      x = odds_step(x, f, df);
    }
    nu[0] = v;
    V[0][0] = q[0] * r1;
    V[0][1] = -rho * q[1] * r2;
    V[0][2] = -q[0] * v * r1;
    V[0][3] = q[1] * v * r2;
    V[0][4] = q[2] * iv;
  }
  {
    double x = (double)odds_a(v1, p1, v2, p2, g, b1, b2, b3);
    double r1 = 0.0, r2 = 0.0, v = 0.0, iv = 0.0;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const double t = s.v2 * rcp_refined(1.0 + x), w = s.g + t;
      v = t * x;
      r1 = 1.0 / (w * (v + s.p1));
      r2 = 1.0 / (t * (v + s.p2));
      iv = 1.0 / v;
      if (k == 2) break;
      const double g1 = s.b1 * v * r1, g2 = s.b2 * v * r2, f = (1.0 + s.b3 * iv) - (g1 + g2);
      const float tf = (float)t, vf = (float)v, ivf = (float)iv, fr = tf / (float)w;
      const float e1 = tf * p1 * ivf / (vf + p1), e2 = tf * p2 * ivf / (vf + p2);
      const float df = -(b3 * ivf * (tf / v2) + ((float)g1 * (e1 + fr) + (float)g2 * (1.f + e2)) * (vf / v2));
      x = odds_step(x, f, df);
    }
    nu[1] = v;
    V[1][0] = q[0] * r1;
    V[1][1] = rho * q[1] * r2;
    V[1][2] = -q[0] * v * r1;
    V[1][3] = -q[1] * v * r2;
    V[1][4] = q[2] * iv;
  }
}

// half of the angle of the unit vector (c, s): cosine and sine, cosine >= 0
__host__ __device__ __forceinline__ void half_angle(double c, double s, double& ch, double& sh) {
  const double a = 0.5 + 0.5 * fabs(c), ia = hd_rsqrt(a), ra = a * ia, rs = 0.5 * s * ia;
  ch = c >= 0.0 ? ra : fabs(rs);
  sh = c >= 0.0 ? rs : (s >= 0.0 ? ra : -ra);
}

// A projected pair Hessian as its blocks need it: block (q1, q2) is
//   c_q1 c_q2 M0 + (c_q1 h_q2 + sig_q1q2 n) n^T + n (c_q2 h_q1)^T.
struct PlaneBlocks {
  double n[3];      // unit normal, from the second primitive's side to the first's (r = d n)
  double c[4];      // closest-point weights: r = sum_q c_q x_q
  double M0[6];     // xx xy xz yy yz zz
  double h[4][3];
  double sig[10];   // 00 01 02 03 11 12 13 22 23 33
};

// w, u, v: the pair's difference vectors (face: p - t0, t1 - t0, t2 - t0; line-line: b0 - a0, a1 - a0, b1 - b0).
// beta = kappa b'', lam = -kappa b', d the distance.
__host__ __device__ __forceinline__ void plane_blocks(bool ee, const double (&w)[3], const double (&u)[3],
                                                      const double (&v)[3], double d, double beta, double lam,
                                                      PlaneBlocks& P) {
  double n[3] = {u[1] * v[2] - u[2] * v[1], u[2] * v[0] - u[0] * v[2], u[0] * v[1] - u[1] * v[0]};
  const double N = n[0] * n[0] + n[1] * n[1] + n[2] * n[2], in = hd_rsqrt(N), iN = in * in;
  const double uu = u[0] * u[0] + u[1] * u[1] + u[2] * u[2], iu = hd_rsqrt(uu);
  const double uv = u[0] * v[0] + u[1] * v[1] + u[2] * v[2];
  // r = w - s u - t v
  const double s = ((w[1] * v[2] - w[2] * v[1]) * n[0] + (w[2] * v[0] - w[0] * v[2]) * n[1] +
                    (w[0] * v[1] - w[1] * v[0]) * n[2]) * iN;
  const double t = ((u[1] * w[2] - u[2] * w[1]) * n[0] + (u[2] * w[0] - u[0] * w[2]) * n[1] +
                    (u[0] * w[1] - u[1] * w[0]) * n[2]) * iN;
  const double sg = w[0] * n[0] + w[1] * n[1] + w[2] * n[2] >= 0.0 ? in : -in;
  double f1[3], f2[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) f1[k] = u[k] * iu;
  f2[0] = (n[1] * f1[2] - n[2] * f1[1]) * in;
  f2[1] = (n[2] * f1[0] - n[0] * f1[2]) * in;
  f2[2] = (n[0] * f1[1] - n[1] * f1[0]) * in;
#pragma unroll
  for (int k = 0; k < 3; ++k) P.n[k] = n[k] * sg;
  // K = [[k11, k12], [0, k22]] in (f1, f2): the dual edge vectors u* = (1/|u|, -(u.v)/(|u| |n|)), v* = (0, |u|/|n|)
  // in an orthonormal basis of the weights of u and v, and c's coordinates in that basis and its complement
  constexpr double r2 = 1.41421356237309504880, ir2 = 0.70710678118654752440, r32 = 1.22474487139158904910,
                   ir6 = 0.40824829046386301637, f3 = 1.15470053837925152902, ir12 = 0.28867513459481288225;
  const double ul = uu * iu, us2 = -uv * iu * in, vs2 = ul * in;
  const double k11 = r2 * iu, k12 = ee ? r2 * us2 : fma(r2, us2, ir2 * vs2), k22 = (ee ? r2 : r32) * vs2;
  const double m1 = ee ? (1.0 - 2.0 * s) * ir2 : (1.0 - 2.0 * s - t) * ir2;
  const double m2 = ee ? -(1.0 + 2.0 * t) * ir2 : (1.0 - 3.0 * t) * ir6;
  const double m3 = ee ? -1.0 : f3;
  P.c[0] = ee ? s - 1.0 : 1.0;
  P.c[1] = ee ? -s : s + t - 1.0;
  P.c[2] = ee ? 1.0 + t : -s;
  P.c[3] = -t;
  // K = Rot(phi) diag(s1, s2) Rot(theta) with s1 = Q + R, s2 = Q - R = k11 k22 / s1
  const double E = 0.5 * (k11 + k22), F = 0.5 * (k11 - k22), H = 0.5 * k12;  // (c + b)/2 = H, (c - b)/2 = -H
  const double QQ = E * E + H * H, RR = F * F + H * H, iQ = hd_rsqrt(QQ);
  const double iR = RR > 0.0 ? hd_rsqrt(RR) : 0.0;
  const double Qm = QQ * iQ, Rm = RR * iR, s1 = Qm + Rm;
  const double is1 = 1.0 / s1, rho = k11 * k22 * is1 * is1;
  const double del = fmax(2.0 * Rm * is1, 1e-15);  // 1 - rho, held off zero (an exact double pole) at rounding level
  const double ca1 = RR > 0.0 ? F * iR : 1.0, sa1 = H * iR, ca2 = E * iQ, sa2 = -H * iQ;
  double cph, sph, cth, sth;
  half_angle(ca2 * ca1 - sa2 * sa1, sa2 * ca1 + ca2 * sa1, cph, sph);   // phi = (a2 + a1) / 2
  half_angle(ca2 * ca1 + sa2 * sa1, sa2 * ca1 - ca2 * sa1, cth, sth);   // theta = (a2 - a1) / 2
  // the half angles are each known up to pi: K = Rot(phi) S Rot(theta) fixes the sign of the product
  {
    const double k = cph * cth - rho * sph * sth;  // K11 / s1
    if ((fabs(k) > 1e-3 && k < 0.0) || (fabs(k) <= 1e-3 && (-cph * sth - rho * sph * cth) * k12 < 0.0)) {
      cth = -cth;
      sth = -sth;
    }
  }
  const double mu2 = m1 * m1 + m2 * m2 + m3 * m3, imu = hd_rsqrt(mu2), mu = mu2 * imu;
  const double Lam = lam * mu * s1, iL = 1.0 / Lam, e1 = d * s1 * imu, e2 = e1 * rho;
  Secular S;
  double q[3] = {cph * m1 + sph * m2, cph * m2 - sph * m1, m3};
#pragma unroll
  for (int k = 0; k < 2; ++k)  // off zero at rounding level: a decoupled axis would sit on its pole
    if (fabs(q[k]) < 1e-15) q[k] = q[k] < 0.0 ? -1e-15 : 1e-15;
  const double sq1 = sqrt(fma(e1, e1, 4.0)), sq2 = sqrt(fma(e2, e2, 4.0));
  const double hp1 = 0.5 * (sq1 + e1), hp2 = 0.5 * (sq2 + e2), n1 = 1.0 / hp1, n2 = 1.0 / hp2;
  S.v1 = n1;
  S.p1 = hp1;
  S.v2 = rho * n2;
  S.p2 = rho * hp2;
  S.g = del * (n1 + n2) * (n1 + n2) / (e1 + e2 + 2.0 * (n1 + n2));
  const double bs = beta * iL;
  S.b1 = bs * q[0] * q[0];
  S.b2 = bs * q[1] * q[1];
  S.b3 = bs * q[2] * q[2];
  double nu[2], V[2][5];
  secular_vectors(S, rho, q, nu, V);
  // T+ = T + sum nu v v^T / |v|^2, scaled by Lam; order x1 x2 y1 y2 y3
  double T[15] = {0.0, 0.0, Lam, 0.0, 0.0,  0.0, 0.0, Lam * rho, 0.0,  Lam * e1 + beta * q[0] * q[0],
                  beta * q[0] * q[1], beta * q[0] * q[2],  Lam * e2 * rho + beta * q[1] * q[1], beta * q[1] * q[2],
                  beta * q[2] * q[2]};
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    const double vv = V[k][0] * V[k][0] + V[k][1] * V[k][1] + V[k][2] * V[k][2] + V[k][3] * V[k][3] + V[k][4] * V[k][4];
    const double sc = Lam * nu[k] / vv;
    int e = 0;
#pragma unroll
    for (int i = 0; i < 5; ++i) {
      const double wi = sc * V[k][i];
#pragma unroll
      for (int j = i; j < 5; ++j) T[e++] += wi * V[k][j];
    }
  }
  // the rotated axes, the in-plane ones over mu (c takes the place of c / mu)
  double F1[3], F2[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    F1[k] = (cth * f1[k] - sth * f2[k]) * imu;
    F2[k] = (sth * f1[k] + cth * f2[k]) * imu;
  }
  {
    int e = 0;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      const double a = T[0] * F1[i] + T[1] * F2[i], b = T[1] * F1[i] + T[5] * F2[i];
#pragma unroll
      for (int j = i; j < 3; ++j) P.M0[e++] = a * F1[j] + b * F2[j];
    }
  }
  // weights of the basis at the four points, rotated
  double k[4][3];
  {
    const double a1[4] = {ee ? -ir2 : 0.0, ee ? ir2 : -ir2, ee ? 0.0 : ir2, 0.0};
    const double a2[4] = {0.0, ee ? 0.0 : -ir6, ee ? -ir2 : -ir6, ee ? ir2 : 2.0 * ir6};
    const double a3[4] = {ee ? 0.5 : 3.0 * ir12, ee ? 0.5 : -ir12, ee ? -0.5 : -ir12, ee ? -0.5 : -ir12};
#pragma unroll
    for (int p = 0; p < 4; ++p) {
      k[p][0] = cph * a1[p] + sph * a2[p];
      k[p][1] = cph * a2[p] - sph * a1[p];
      k[p][2] = a3[p];
    }
  }
  double G[3][3];
  {
    const double X1[3] = {T[2], T[3], T[4]}, X2[3] = {T[6], T[7], T[8]};
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int j = 0; j < 3; ++j) G[i][j] = X1[i] * F1[j] + X2[i] * F2[j];
  }
  const double Sy[3][3] = {{T[9], T[10], T[11]}, {T[10], T[12], T[13]}, {T[11], T[13], T[14]}};
  double W[4][3];
#pragma unroll
  for (int p = 0; p < 4; ++p)
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      P.h[p][j] = k[p][0] * G[0][j] + k[p][1] * G[1][j] + k[p][2] * G[2][j];
      W[p][j] = k[p][0] * Sy[0][j] + k[p][1] * Sy[1][j] + k[p][2] * Sy[2][j];
    }
  int e = 0;
#pragma unroll
  for (int p = 0; p < 4; ++p)
#pragma unroll
    for (int r = p; r < 4; ++r) P.sig[e++] = W[p][0] * k[r][0] + W[p][1] * k[r][1] + W[p][2] * k[r][2];
}

// block (p, r), p <= r, row-major
__host__ __device__ __forceinline__ void plane_block(const PlaneBlocks& P, int p, int r, double (&blk)[9]) {
  const int e = p * 4 - (p * (p - 1)) / 2 + (r - p);
  const double a = P.c[p] * P.c[r];
  const int s6[9] = {0, 1, 2, 1, 3, 4, 2, 4, 5};
  double l[3], m[3];
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    l[i] = P.c[p] * P.h[r][i] + P.sig[e] * P.n[i];
    m[i] = P.c[r] * P.h[p][i];
  }
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j)  // a diagonal block is symmetric: its lower triangle is copied
      blk[3 * i + j] = p == r && j < i ? blk[3 * j + i] : a * P.M0[s6[3 * i + j]] + l[i] * P.n[j] + P.n[i] * m[j];
}

// Point-edge pair: q off the edge e0 e1, w = q - e0, u = e1 - e0; points in the order q, e0, e1.  Block (p, r) is
// e1 (al e1 + be n)^T + n (ga e1 + sig n)^T with e1 the edge's direction.
struct EdgeBlocks {
  double n[3], e[3];
  double c[3];      // 1, -(1 - t), -t
  double A;         // coefficient of c_p c_r e1 e1^T
  double h[3];      // block (p, r) takes c_p h_r e1 n^T and c_r h_p n e1^T
  double sig[6];    // 00 01 02 11 12 22
};

// n, e1, t = w.u / |u|^2 and 1/|u| from the caller (frame of w and u)
__host__ __device__ __forceinline__ void edge_blocks(double t, double iu, double d, double beta, double lam,
                                                     EdgeBlocks& P) {
  constexpr double r2 = 1.41421356237309504880, ir2 = 0.70710678118654752440, r32 = 1.22474487139158904910,
                   ir6 = 0.40824829046386301637;
  P.c[0] = 1.0;
  P.c[1] = t - 1.0;
  P.c[2] = -t;
  // basis of the zero-sum weights: b1 = (0, -1, 1) / sqrt 2 (the edge's), b2 = (2, -1, -1) / sqrt 6
  const double m1 = (1.0 - 2.0 * t) * ir2, m2 = r32;
  const double mu2 = m1 * m1 + m2 * m2, imu = hd_rsqrt(mu2), mu = mu2 * imu;
  const double s = r2 * iu, p = lam * mu * s, a = d * s * imu;  // T / p = [[0, 1, 0], [1, a + B1, c], [0, c, B2]]
  const double ip = 1.0 / p, bs = beta * ip, B1 = bs * m1 * m1, B2 = bs * m2 * m2, B12 = bs * m1 * m2;
  // the negative eigenvalue -v: v^2 + a v + B1 v^2 / (B2 + v) = 1, convex and increasing in v > 0.  Newton from
  // above (the root without B1), in FP32, then two steps to FP64.
  const float af = (float)a, B1f = (float)B1, B2f = (float)B2;
  float vf = 2.f / (af + sqrtf(af * af + 4.f));
  for (int it = 0; it < 12; ++it) {
    const float ib = 1.f / (B2f + vf), x = vf * ib, f = vf * (vf + af + B1f * x) - 1.f;
    const float df = 2.f * vf + af + B1f * x * (2.f - x), st = f / df;
    vf -= st;
    if (!(fabsf(st) > 1e-6f * vf)) break;
  }
  double v = (double)vf, ib = 0.0;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    ib = 1.0 / (B2 + v);
    if (k == 2) break;
    const double x = v * ib, f = fma(v, v + a + B1 * x, -1.0);
    const float xf = (float)x, df = 2.f * (float)v + af + B1f * xf * (2.f - xf);
    v -= (double)((float)f / df);
  }
  // eigenvector (-1/v, 1, -B12 / (B2 + v)); T+ = T + v y y^T / |y|^2, each entry a sum or product of one sign
  const double y0 = -1.0 / v, y2 = -B12 * ib, y02 = y0 * y0, y22 = y2 * y2;
  const double in = 1.0 / (y02 + 1.0 + y22), sc = v * in;
  const double T00 = p * sc * y02, T01 = p * in * (y02 + y22), T02 = p * sc * y0 * y2;
  const double T11 = p * (a + B1 + sc), T12 = p * (B12 * (1.0 - sc * ib)), T22 = p * (B2 + sc * y22);
  P.A = T00 * imu * imu;
  // weights at the three points: b1 = (0, -ir2, ir2), b2 = (2, -1, -1) ir6
  const double g1 = T01 * ir2 * imu, g2 = T02 * ir6 * imu;
  P.h[0] = 2.0 * g2;
  P.h[1] = -g1 - g2;
  P.h[2] = g1 - g2;
  const double S11 = 0.5 * T11, S12 = ir2 * ir6 * T12, S22 = (1.0 / 6.0) * T22;
  P.sig[0] = 4.0 * S22;
  P.sig[1] = -2.0 * (S12 + S22);
  P.sig[2] = 2.0 * (S12 - S22);
  P.sig[3] = S11 + 2.0 * S12 + S22;
  P.sig[4] = S22 - S11;
  P.sig[5] = S11 - 2.0 * S12 + S22;
}

// block (p, r), p <= r, row-major
__host__ __device__ __forceinline__ void edge_block(const EdgeBlocks& P, int p, int r, double (&blk)[9]) {
  const int k = p * 3 - (p * (p - 1)) / 2 + (r - p);
  const double al = P.A * P.c[p] * P.c[r], be = P.c[p] * P.h[r], ga = P.c[r] * P.h[p];
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    const double x = al * P.e[j] + be * P.n[j], y = ga * P.e[j] + P.sig[k] * P.n[j];
#pragma unroll
    for (int i = 0; i < 3; ++i)
      if (p != r || i <= j) blk[3 * i + j] = P.e[i] * x + P.n[i] * y;
  }
  if (p == r) {  // symmetric
    blk[3] = blk[1];
    blk[6] = blk[2];
    blk[7] = blk[5];
  }
}

}  // namespace cbh
