// Boundary-integral terms: the Nystrom matrix of the 2-D Helmholtz double-layer
// operator of the scattering-pole problem (Sec. 4.2), formed entry by entry on
// the device, and the Bessel functions of complex argument it needs.
//
// K(kappa) phi(x) = 2 int_C d/dnu(y) Phi(x, y) phi(y) ds(y), Phi = (i/4) H_0^(1)(kappa |x - y|).
// With the curve x(t) sampled at t_j = 2 pi j / n (n = 2 n'), n(t) = (x2', -x1'),
// r = |x(t_i) - x(t_j)| and q = n(t_j).(x(t_i) - x(t_j)), Kress's rule for kernels
// with a logarithmic singularity (R. Kress, Linear Integral Equations, Sec. 12.3)
// gives the matrix entry
//   K_ij = h L_ij + (R_m - h log(4 sin^2(pi m / n))) L1_ij,   m = (i - j) mod n, h = 2 pi / n,
//   L  = (i kappa / 2) q H_1^(1)(kappa r) / r,   L1 = -(kappa / (2 pi)) q J_1(kappa r) / r,
//   K_jj = h n(t_j).x''(t_j) / (2 pi |x'(t_j)|^2),
//   R_m = -(2 pi / n') sum_{k=1}^{n'-1} cos(k m pi / n') / k - (pi / n'^2) cos(m pi).
// The host folds R_m - h log(4 sin^2(pi m / n)) into one table of n values.
//
// Everything here is plain arithmetic on double2 and compiles for the host too.
#pragma once

#include <cuda_runtime.h>
#include <math.h>

#if defined(__CUDACC__)
#define BIE_HD __host__ __device__ __forceinline__
// the entry is a call: inlined into the assembly loops it would raise their register
// pressure on every path, also where a problem has no boundary-integral term
#define BIE_ENTRY static __host__ __device__ __noinline__
#else
#define BIE_HD inline
#define BIE_ENTRY inline
#endif

namespace bie {

constexpr double kPi = 3.14159265358979323846;
constexpr double kEulerGamma = 0.57721566490153286061;
constexpr double kSeriesMax = 6.0;   // |w| at or below: ascending series
constexpr double kMillerMax = 13.0;  // at or below: backward recurrence; above: Hankel's expansion
constexpr int kMillerTop = 46;       // J_46(w) is below 1e-20 of the largest J_k for |w| <= 13
constexpr int kSeriesTerms = 32, kAsymTerms = 64;

// The series' coefficients, made at compile time and read from the constant cache:
//   cj[k] = 1 / (k! (k+1)!),  cs[k] = (psi(k+1) + psi(k+2)) / (k! (k+1)!) with
//   psi(k+1) + psi(k+2) = 2 (H_k - gamma) + 1/(k+1),
//   nm[2k+1] = (-1)^k (2k+1) / (k (k+1))  (Neumann's series),
//   ak[k] = prod_{j=1..k} (4 - (2j-1)^2) / (8 j)  (Hankel's a_k for order 1).
struct SeriesTables {
  double cj[kSeriesTerms];
  double cs[kSeriesTerms];
  double nm[kMillerTop + 1];
  double ak[kAsymTerms];
};
constexpr SeriesTables make_series_tables() {
  SeriesTables T{};
  double Hk = 0.0, f = 1.0;
  T.cj[0] = 1.0;
  T.cs[0] = 1.0 - 2.0 * kEulerGamma;
  for (int k = 1; k < kSeriesTerms; ++k) {
    f /= (double)k * (double)(k + 1);
    Hk += 1.0 / (double)k;
    T.cj[k] = f;
    T.cs[k] = f * (2.0 * (Hk - kEulerGamma) + 1.0 / (double)(k + 1));
  }
  for (int k = 1; 2 * k + 1 <= kMillerTop; ++k)
    T.nm[2 * k + 1] = ((k & 1) ? -1.0 : 1.0) * (double)(2 * k + 1) / ((double)k * (double)(k + 1));
  double a = 1.0;
  T.ak[0] = 1.0;
  for (int k = 1; k < kAsymTerms; ++k) {
    a *= (4.0 - (double)(2 * k - 1) * (double)(2 * k - 1)) / (8.0 * (double)k);
    T.ak[k] = a;
  }
  return T;
}
#if defined(__CUDACC__)
static __constant__ SeriesTables kSeriesDev = make_series_tables();
#endif
static const SeriesTables kSeriesHost = make_series_tables();
#if defined(__CUDA_ARCH__)
#define BIE_TABLES kSeriesDev
#else
#define BIE_TABLES kSeriesHost
#endif

BIE_HD double2 cm(double2 a, double2 b) { return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x); }
BIE_HD double2 ca(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
BIE_HD double2 cs(double2 a, double s) { return make_double2(a.x * s, a.y * s); }
BIE_HD double2 ci(double2 a) { return make_double2(-a.y, a.x); }  // i a
BIE_HD double2 crec(double2 b) {                                    // 1 / b (Smith's scaling)
  if (fabs(b.x) >= fabs(b.y)) {
    const double t = b.y / b.x, d = b.x + b.y * t;
    return make_double2(1.0 / d, -t / d);
  }
  const double t = b.x / b.y, d = b.x * t + b.y;
  return make_double2(t / d, -1.0 / d);
}

// What the entries of one wave number kappa share.
struct Wave {
  double2 kappa, inv;   // kappa, 1 / kappa
  double2 lg;           // log(kappa / 2)
  double2 pref;         // sqrt(2 / (pi kappa))
  double mod;           // |kappa|
};
BIE_HD Wave wave_of(double2 kappa) {
  Wave W;
  W.kappa = kappa;
  W.inv = crec(kappa);
  W.mod = hypot(kappa.x, kappa.y);
  const double arg = atan2(kappa.y, kappa.x);
  W.lg = make_double2(log(0.5 * W.mod), arg);
  double s, c;
  sincos(-0.5 * arg, &s, &c);
  const double m = sqrt(2.0 / (kPi * W.mod));
  W.pref = make_double2(m * c, m * s);
  return W;
}

// J_1(w) and H_1^(1)(w), w = kappa r, for Re w > 0; ri = 1 / r, lr = log r.
//  |w| <= 6: the ascending series J_1(w) = sum_k (-1)^k (w/2)^{2k+1} / (k! (k+1)!) and
//    Y_1(w) = -2 / (pi w) + (2/pi) log(w/2) J_1(w)
//             - (1/pi) sum_k (psi(k+1) + psi(k+2)) (-1)^k (w/2)^{2k+1} / (k! (k+1)!)
//    (DLMF 10.2.2 and 10.8.1; psi(k+1) = -gamma + H_k with H_k the harmonic number),
//    H_1^(1) = J_1 + i Y_1 (DLMF 10.4.3). Both sums are polynomials in -(w/2)^2 with real
//    coefficients, by Horner's rule, 8 FP64 operations per term (a term with a running
//    product and a stopping test took about 20, and FP64 bounds the assembly). The number
//    of terms, ceil(5.9 + 3 |w| - 0.095 |w|^2), leaves out less than 1e-17 of the largest
//    term; each entry takes its own, so that its value does not depend on the entries that
//    share its warp. Near the real axis the sums cancel to e^{-|w|} of their largest term, which sets the range.
//  6 < |w| <= 13: J_k by the backward recurrence J_{k-1} = (2k / w) J_k - J_{k+1} (DLMF
//    3.6(iii)) from k = 46, scaled by e^{+-iw} = J_0 + 2 sum_k (+-i)^k J_k (DLMF 10.12.1; the
//    sign that makes the left side large), and Y_1 by Neumann's series (Abramowitz & Stegun
//    9.1.88): Y_1 = -2 J_0 / (pi w) + (2/pi) ((log(w/2) + gamma - 1) J_1
//    - sum_k (-1)^k (2k+1) / (k (k+1)) J_{2k+1}).
//  |w| > 13: Hankel's expansions (DLMF 10.17.5, 10.17.6)
//    H_1^(1,2)(w) ~ sqrt(2 / (pi w)) e^{+-i (w - 3 pi / 4)} sum_k (+-i)^k a_k / w^k,
//    a_k = prod_{j=1..k} (4 - (2j - 1)^2) / (k! 8^k), truncated before the smallest term
//    grows again, and J_1 = (H_1^(1) + H_1^(2)) / 2 (DLMF 10.4.4).
BIE_HD void j1_h1(const Wave& W, double r, double ri, double lr, double2* J, double2* H) {
  const SeriesTables& TB = BIE_TABLES;
  const double2 w = cs(W.kappa, r);
  const double aw = W.mod * r;
  const double2 iw = cs(W.inv, ri);
  if (aw <= kSeriesMax) {
    const double2 h = cs(w, 0.5);
    const double2 u = make_double2(h.y * h.y - h.x * h.x, -2.0 * h.x * h.y);  // -(w/2)^2
    const float fw = (float)aw;
    int k = (int)ceilf(5.9f + fw * (3.0f - 0.095f * fw)) - 1;
    double2 p = make_double2(TB.cj[k], 0.0), q = make_double2(TB.cs[k], 0.0);
    for (--k; k >= 0; --k) {
      const double px = fma(p.x, u.x, fma(-p.y, u.y, TB.cj[k])), qx = fma(q.x, u.x, fma(-q.y, u.y, TB.cs[k]));
      p.y = fma(p.x, u.y, p.y * u.x);
      q.y = fma(q.x, u.y, q.y * u.x);
      p.x = px;
      q.x = qx;
    }
    const double2 Js = cm(h, p), S = cm(h, q);
    const double2 lg = make_double2(W.lg.x + lr, W.lg.y);  // log(w/2)
    const double2 lj = cm(lg, Js);
    const double2 Y = make_double2((2.0 / kPi) * (lj.x - iw.x) - (1.0 / kPi) * S.x,
                                   (2.0 / kPi) * (lj.y - iw.y) - (1.0 / kPi) * S.y);
    *J = Js;
    *H = ca(Js, ci(Y));
    return;
  }
  if (aw <= kMillerMax) {
    const double sg = w.y <= 0.0 ? 1.0 : -1.0;
    double2 up = make_double2(0.0, 0.0), cur = make_double2(1e-30, 0.0);  // J_{k+1}, J_k up to a factor
    double2 sum = up, nm = up, j1 = up;  // sum_k (+-i)^k J_k, Neumann's series
    for (int k = kMillerTop; k >= 1; --k) {
      switch (k & 3) {  // (sg i)^k
        case 0: sum.x += cur.x; sum.y += cur.y; break;
        case 1: sum.x -= sg * cur.y; sum.y += sg * cur.x; break;
        case 2: sum.x -= cur.x; sum.y -= cur.y; break;
        default: sum.x += sg * cur.y; sum.y -= sg * cur.x; break;
      }
      if ((k & 1) && k > 1) {
        nm.x = fma(TB.nm[k], cur.x, nm.x);
        nm.y = fma(TB.nm[k], cur.y, nm.y);
      }
      if (k == 1) j1 = cur;
      const double2 f = cs(iw, 2.0 * (double)k);
      const double2 dn = make_double2(fma(f.x, cur.x, fma(-f.y, cur.y, -up.x)),
                                      fma(f.x, cur.y, fma(f.y, cur.x, -up.y)));
      up = cur;
      cur = dn;
    }
    sum = make_double2(fma(2.0, sum.x, cur.x), fma(2.0, sum.y, cur.y));
    double so, co;
    sincos(sg * w.x, &so, &co);
    const double em = exp(-sg * w.y);
    const double2 scale = cm(make_double2(em * co, em * so), crec(sum));
    const double2 J0 = cm(cur, scale), Js = cm(j1, scale), S = cm(nm, scale);
    const double2 lg = make_double2(W.lg.x + lr + (kEulerGamma - 1.0), W.lg.y);
    const double2 lj = cm(lg, Js), jw = cm(iw, J0);
    const double2 Y = cs(make_double2(lj.x - S.x - jw.x, lj.y - S.y - jw.y), 2.0 / kPi);
    *J = Js;
    *H = ca(Js, ci(Y));
    return;
  }
  double2 p = make_double2(1.0, 0.0);   // 1 / w^k
  double2 s1 = p, s2 = p;               // sums with (+i)^k and (-i)^k
  double prev = 1.0;
  for (int k = 1; k < kAsymTerms; ++k) {
    p = cm(p, iw);
    const double2 tk = cs(p, TB.ak[k]);
    const double mag = fabs(tk.x) + fabs(tk.y);
    if (mag > prev) break;  // past the smallest term
    // (+i)^k tk and (-i)^k tk
    double2 t1, t2;
    switch (k & 3) {
      case 0: t1 = tk; t2 = tk; break;
      case 1: t1 = ci(tk); t2 = make_double2(tk.y, -tk.x); break;
      case 2: t1 = make_double2(-tk.x, -tk.y); t2 = t1; break;
      default: t1 = make_double2(tk.y, -tk.x); t2 = ci(tk); break;
    }
    s1 = ca(s1, t1);
    s2 = ca(s2, t2);
    prev = mag;
    if (mag < 1e-17) break;
  }
  const double2 pref = cs(W.pref, sqrt(ri));
  double so, co;
  sincos(w.x - 0.75 * kPi, &so, &co);
  const double eu = exp(-w.y), ed = exp(w.y);
  const double2 e1 = make_double2(eu * co, eu * so);   // e^{+i (w - 3 pi / 4)}
  const double2 e2 = make_double2(ed * co, -ed * so);  // e^{-i (w - 3 pi / 4)}
  const double2 h1 = cm(pref, cm(e1, s1));
  const double2 h2 = cm(pref, cm(e2, s2));
  *H = h1;
  *J = cs(ca(h1, h2), 0.5);
}
BIE_HD void j1_h1(double2 w, double2* J, double2* H) { j1_h1(wave_of(w), 1.0, 1.0, 0.0, J, H); }

// Entries (i, j) and (j, i), i != j, of K_n(kappa). They share r and with it the Bessel
// values, and differ in the normal: K_ij = (n(t_j).(x_i - x_j) / r) F, K_ji =
// (n(t_i).(x_j - x_i) / r) F with F = kappa ((i h / 2) H_1 - (G[5 n + m] / 2 pi) J_1).
// G: the device geometry of the term (n >= 4, even),
//   G[5 j + 0..4] = x1, x2, n1 = x2', n2 = -x1', d = n.x'' / (2 pi |x'|^2) at t_j,
//   G[5 n + m]    = R_m - (2 pi / n) log(4 sin^2(pi m / n))  (m = 1..n-1; m = 0 unused),
//   G[6 n]        = 1 when the sampled curve is invariant under the shift j -> j + 1 (a
//                   circle), so that K_n is circulant: K_ij = K_{(i-j) mod n, 0}; else 0.
BIE_ENTRY void dlp_pair(const double* G, int n, int i, int j, const Wave& W, double2* Kij, double2* Kji) {
  const double h = 2.0 * kPi / (double)n;
  const double* pi_ = G + 5 * (size_t)i;
  const double* pj = G + 5 * (size_t)j;
  const double ex = pi_[0] - pj[0], ey = pi_[1] - pj[1];
  const double rr = ex * ex + ey * ey;
#if defined(__CUDA_ARCH__)
  const double ri = rsqrt(rr);
  double r = rr * ri;
  r = fma(0.5 * ri, fma(-r, r, rr), r);  // one Newton step: the rounding of ri stays out of r
#else
  const double r = sqrt(rr), ri = 1.0 / r;
#endif
  double2 J1, H1;
  j1_h1(W, r, ri, log(r), &J1, &H1);
  const int m = i > j ? i - j : i - j + n;
  const double wj = G[5 * (size_t)n + m] * (1.0 / (2.0 * kPi)), wh = 0.5 * h;
  const double2 F = cm(W.kappa, make_double2(-wh * H1.y - wj * J1.x, wh * H1.x - wj * J1.y));
  *Kij = cs(F, (pj[2] * ex + pj[3] * ey) * ri);
  *Kji = cs(F, -(pi_[2] * ex + pi_[3] * ey) * ri);
}
// A diagonal entry.
BIE_HD double2 dlp_diagonal(const double* G, int n, int j) {
  return make_double2(2.0 * kPi / (double)n * G[5 * (size_t)j + 4], 0.0);
}
// Entry (i, j) alone.
BIE_HD double2 dlp_entry(const double* G, int n, int i, int j, const Wave& W) {
  if (i == j) return dlp_diagonal(G, n, j);
  double2 a, b;
  dlp_pair(G, n, i, j, W, &a, &b);
  return a;
}
BIE_HD double2 dlp_entry(const double* G, int n, int i, int j, double2 kappa) {
  return dlp_entry(G, n, i, j, wave_of(kappa));
}

// Pair number p of the n (n/2) - n/2 pairs {i, j}, i != j: column j and row j + d mod n with
// d = 1 + p / n, so that consecutive p share d (and nearly r). False past the last one.
BIE_HD bool pair_of(int n, int p, int* i, int* j) {
  const int d = 1 + p / n;
  *j = p - (d - 1) * n;
  if (d > n / 2 || (d == n / 2 && *j >= n / 2)) return false;
  *i = *j + d < n ? *j + d : *j + d - n;
  return true;
}

constexpr int kCirculantMaxN = 8192;  // the shift-invariance test is O(n^2)

// Host: the device geometry G (6 n + 1 doubles) of a curve given by its samples
// s = [x1 | x2 | x1' | x2' | x1'' | x2''] (six rows of n values at t_j = 2 pi j / n).
// Returns false when n is odd or below 4, a sample is not finite, x'(t_j) = 0, or
// two sample points coincide.
inline bool build_geometry(const double* s, int n, double* G) {
  if (n < 4 || (n & 1)) return false;
  for (int j = 0; j < n; ++j) {
    const double x1 = s[j], x2 = s[n + j], d1 = s[2 * n + j], d2 = s[3 * n + j];
    const double dd1 = s[4 * n + j], dd2 = s[5 * n + j];
    const double sp2 = d1 * d1 + d2 * d2;
    if (!(isfinite(x1) && isfinite(x2) && isfinite(d1) && isfinite(d2) && isfinite(dd1) && isfinite(dd2)) ||
        !(sp2 > 0.0))
      return false;
    G[5 * j + 0] = x1;
    G[5 * j + 1] = x2;
    G[5 * j + 2] = d2;
    G[5 * j + 3] = -d1;
    G[5 * j + 4] = (d2 * dd1 - d1 * dd2) / (2.0 * kPi * sp2);
  }
  for (int i = 0; i < n; ++i)
    for (int j = i + 1; j < n; ++j)
      if (s[i] == s[j] && s[n + i] == s[n + j]) return false;
  const int np = n / 2;
  const double h = 2.0 * kPi / (double)n;
  // cos(k m pi / n') through the index k m mod 2 n'
  double* ct = new double[2 * np];
  for (int q = 0; q < 2 * np; ++q) ct[q] = cos(kPi * (double)q / (double)np);
  G[5 * (size_t)n] = 0.0;
  for (int m = 1; m < n; ++m) {
    double R = -(kPi / ((double)np * (double)np)) * ((m & 1) ? -1.0 : 1.0);
    double acc = 0.0;
    for (int k = 1; k < np; ++k) acc += ct[(int)(((long long)k * m) % (2 * np))] / (double)k;
    R -= (2.0 * kPi / (double)np) * acc;
    const double sn = sin(kPi * (double)m / (double)n);
    G[5 * (size_t)n + m] = R - h * log(4.0 * sn * sn);
  }
  delete[] ct;
  // circulant when every entry's geometry (r, n(t_j).(x_i - x_j), and the diagonal term)
  // depends on i - j only, to a few rounding units of the curve's size
  bool circ = n <= kCirculantMaxN;
  double scale = 0.0, dmax = 0.0;
  for (int j = 0; j < n; ++j) {
    scale = fmax(scale, fmax(fabs(G[5 * j]), fabs(G[5 * j + 1])));
    scale = fmax(scale, fmax(fabs(G[5 * j + 2]), fabs(G[5 * j + 3])));
    dmax = fmax(dmax, fabs(G[5 * j + 4]));
  }
  const double tol = 8e-15 * scale, tq = 8e-15 * scale * scale;
  for (int j = 1; j < n && circ; ++j) circ = fabs(G[5 * j + 4] - G[4]) <= 8e-15 * dmax;
  for (int m = 1; m < n && circ; ++m) {
    const double ex0 = G[5 * m] - G[0], ey0 = G[5 * m + 1] - G[1];
    const double r0 = hypot(ex0, ey0), q0 = G[2] * ex0 + G[3] * ey0;
    for (int j = 1; j < n; ++j) {
      const int i = (j + m) % n;
      const double ex = G[5 * i] - G[5 * j], ey = G[5 * i + 1] - G[5 * j + 1];
      if (fabs(hypot(ex, ey) - r0) > tol || fabs(G[5 * j + 2] * ex + G[5 * j + 3] * ey - q0) > tq) {
        circ = false;
        break;
      }
    }
  }
  G[6 * (size_t)n] = circ ? 1.0 : 0.0;
  return true;
}

}  // namespace bie
