// The pair model of one listed pair (FP64 arithmetic).  Branches (contact,
// Coulomb slip, gap clamp, taper ends) are taken on the values; the adjoint's
// hand-written reverse (dss_adjoint.cu) differentiates the same functions.
//
// Contact: Eq. 4-5 (linear spring-dashpot normal force, tangential spring
// with the stretch carried between steps, Coulomb rescale of the stretch).
// Lubrication: App. A (Eq. A2, A3 with the coefficient functions of Eq. A6,
// A7 and the 6 pi eta0 prefactor) in the simple shear of Sec. II; with a
// taper width w > 0 the lubrication force and torques are scaled by
// s = t^2 (3 - 2t), t = clamp((delta_ij - d) / (w delta_ij), 0, 1) (an
// extension that makes the cutoff differentiable; w = 0 is the hard cutoff).
//
// The lubrication functions in closed form.  With S = a_i + a_j, h = a_i a_j / S
// and b = a_i a_j / S^2 the coefficients of Eq. A7 of a pair are
//   XA = 2 X h b,             YA = (4/15) Y b (2 S - 3 h),
//   YBi = -(2/15) Y b a_i (3 a_i + S),  YBj likewise,
//   YCi = (8/15) Y h a_i^2,   YCj likewise,   YCx = (2/15) Y h a_i a_j,
//   XG = S XA,  YG = (S/2) YA,  YHi = -(S/2) YBi,  YHj = -(S/2) YBj
// (each follows from the rational functions of a_j / a_i by factoring; for
// instance 4 a^2 + 5 a b + b^2 = (4 a + b)(a + b)).  The strain terms therefore
// fold into the relative velocity G = V_i - V_j - (S/2) 2E.n:
//   F   = -6 pi eta0 (XA (n.G) n + YA (G - (n.G) n) + n x (YBi W_i + YBj W_j)),
//   T_i =  6 pi eta0 (YBi n x G - tang(YCi W_i + YCx W_j)),  T_j likewise,
// two fifths of the operations of the separate resistance functions.  With it,
// one reciprocal for three, the tangent projection taken once, comparisons on
// bit patterns and the stresslet from r (x) F and r x F^L, the FP64 pair kernel
// (85% of the FP64 pipe's rate before, 81% after) went from 274 to 189 us on
// 267k pairs (the step of 100k spheres 355 -> 266 us).
#pragma once

#include "dss_internal.cuh"

// ---------------------------------------------------------------- vectors
template <typename T>
struct Vec3 {
  T x, y, z;
};
template <typename T>
__device__ __forceinline__ Vec3<T> mk3(T a, T b, T c) { return Vec3<T>{a, b, c}; }
template <typename T>
__device__ __forceinline__ Vec3<T> operator+(const Vec3<T>& a, const Vec3<T>& b) {
  return mk3<T>(a.x + b.x, a.y + b.y, a.z + b.z);
}
template <typename T>
__device__ __forceinline__ Vec3<T> operator-(const Vec3<T>& a, const Vec3<T>& b) {
  return mk3<T>(a.x - b.x, a.y - b.y, a.z - b.z);
}
template <typename T, typename S>
__device__ __forceinline__ Vec3<T> operator*(const S& s, const Vec3<T>& a) {
  return mk3<T>(s * a.x, s * a.y, s * a.z);
}
template <typename T>
__device__ __forceinline__ T dot(const Vec3<T>& a, const Vec3<T>& b) {
  return a.x * b.x + a.y * b.y + a.z * b.z;
}
template <typename T>
__device__ __forceinline__ Vec3<T> cross(const Vec3<T>& a, const Vec3<T>& b) {
  return mk3<T>(a.y * b.z - a.z * b.y, a.z * b.x - a.x * b.z, a.x * b.y - a.y * b.x);
}
template <typename T>
__device__ __forceinline__ Vec3<T> tang(const Vec3<T>& n, const Vec3<T>& v) {
  return v - dot(n, v) * n;
}

// a / b from r = 1/b rounded: the quotient estimate a r corrected by its exact
// remainder (Markstein): the rounded quotient, three operations instead of a
// division's ten on GB300's narrow FP64 pipe.
__device__ __forceinline__ double div_by(double a, double b, double r) {
  const double q = a * r;
  return fma(fma(-q, b, a), r, q);
}

// 1/r, 1/S and X = 1/(gap + eps) = S/num of a pair (num: S (max(2 d / S, 0) +
// eps)) from one reciprocal: a division costs about ten instructions of the
// FP64 pipe.  The roundings of the products are taken out of 1/r and X again, so
// that both are within a rounding and a half of the quotients.
struct PairRecips {
  double ir, iS, X;
};
__device__ __forceinline__ PairRecips pair_recips(double rr, double S, double num) {
  const double p = rr * S, inv = 1.0 / (p * num);
  const double rnum = inv * p, q = inv * num;
  PairRecips o;
  o.iS = q * rr;
  o.ir = q * S;
  o.ir = fma(o.ir, fma(-o.ir, rr, 1.0), o.ir);
  o.X = S * rnum;
  o.X = fma(fma(-o.X, num, S), rnum, o.X);
  return o;
}

// Outputs: force on i (F = Fc + Fl), torques on i and j, the lubrication part
// of the force (its stresslet is sym(r (x) Fl), that of the rest, contact and
// electro-chemical, r (x) F), the new stretch (i -> j orientation) and the new
// rolling stretch (App. B; orientation-free).
struct PairModelOut {
  Vec3<double> F, Ti, Tj, Fl, xi, xr;
  int contact;
};

// r = x_j(image) - x_i, rr = |r|; Vi, Vj velocities relative to U_inf at each
// centre; Wi, Wj angular velocities relative to Omega_inf at each centre;
// du = u_j(image) - u_i (absolute); wi, wj absolute angular velocities; xo
// stretch (i -> j); ro rolling stretch (used when k_r > 0); rate the shear
// rate whose strain acts on the pair's lubrication (gdot, or in the wave of
// Eq. 17 the mean of the two centres' local rates).
template <bool EXT>
__device__ __forceinline__ PairModelOut pair_model(const Geo& g, double gn, Vec3<double> r, double rr, double ai,
                                                   double aj, Vec3<double> Vi, Vec3<double> Vj, Vec3<double> Wi,
                                                   Vec3<double> Wj, Vec3<double> du, Vec3<double> wi,
                                                   Vec3<double> wj, Vec3<double> xo, Vec3<double> ro, double rate) {
  using V = Vec3<double>;
  PairModelOut o;
  const double S = ai + aj, d = rr - S;
  o.contact = __double2hiint(d) < 0;   // (rr - S is never -0)
  const double num = fma(g.eps, S, o.contact ? 0.0 : 2.0 * d);   // S (max(2 d / S, 0) + eps)
  const PairRecips q = pair_recips(rr, S, num);
  const double iS = q.iS, X = q.X;
  const V n = q.ir * r;
  // ---- contact, Eq. 4-5
  V Fc = mk3<double>(0.0, 0.0, 0.0);
  o.xi = o.xr = o.Ti = o.Tj = Fc;
  if (o.contact) {
    const double fn = g.kn * d + gn * dot(n, du);
    // the projection onto the tangent plane is linear: old stretch and
    // increment together
    V xs = tang(n, xo + g.dt * (du - cross(ai * wi + aj * wj, n)));
    const double cap = g.mu_kt * fabs(fn), xm2 = dot(xs, xs);
    if (xm2 > cap * cap) xs = (cap * rsqrt(xm2)) * xs;
    const V Ft = g.kt * xs;
    Fc = fn * n + Ft;
    const V nxf = cross(n, Ft);
    o.Ti = ai * nxf;
    o.Tj = aj * nxf;
    o.xi = xs;
    // rolling resistance, App. B: the procedure of Eq. 5 on the rolling
    // velocity abar (n x w_i - n x w_j) with k_r; torques only
    if (EXT && g.k_r > 0.0) {
      const double abar = 2.0 * ai * aj * iS;
      V xr = tang(n, ro) + (g.dt * abar) * cross(n, wi - wj);
      const double capr = g.mu * fabs(fn) / g.k_r, xrm2 = dot(xr, xr);
      if (xrm2 > capr * capr) xr = (capr * rsqrt(xrm2)) * xr;
      const V Tr = abar * cross(n, g.k_r * xr);
      o.Ti = o.Ti + Tr;
      o.Tj = o.Tj - Tr;
      o.xr = xr;
    }
  }
  // ---- electro-chemical forces, Eq. 6-7 (central; stresslet r (x) F like contact)
  bool lub_on = true;
  if (g.de > 0.0) {
    const double abar = 2.0 * ai * aj * iS;
    double m = 0.0;
    if (g.f_er > 0.0 && d < 20.0 * g.lambda_d)
      m = m - (g.f_er * (abar / g.a0)) * (d >= 0.0 ? exp(-d / g.lambda_d) : 1.0);
    if (g.hamaker > 0.0 && d < 4.0 * g.a0) {
      const double eps = g.vdw_eps * abar;
      const double dp = d >= 0.0 ? d : 0.0;
      m = m + (g.hamaker * abar) / (12.0 * (dp * dp + eps * eps));
    }
    Fc = Fc + m * n;
    // lubrication only within its own cutoff: the listing predicate with the
    // lubrication range, in the same operations as the neighbour test
    const double r2 = __dadd_rn(__dadd_rn(__dmul_rn(r.x, r.x), __dmul_rn(r.y, r.y)), __dmul_rn(r.z, r.z));
    const double dl = g.mode == 1 ? __dmul_rn(g.delta, g.a0) : __dmul_rn(__dmul_rn(g.delta, __dadd_rn(ai, aj)), 0.5);
    const double sl = __dadd_rn(__dadd_rn(ai, aj), dl);
    lub_on = r2 < __dmul_rn(sl, sl);
  }
  // ---- lubrication, App. A, for the pairs within its range (every listed
  // pair unless electro-chemical forces widen the list)
  o.Fl = mk3<double>(0.0, 0.0, 0.0);
  o.F = Fc;
  if (lub_on) {
    const double Y = -log(num * iS);
    const double AB = ai * aj, h = AB * iS, b = h * iS;
    const double xa = ((2.0 * g.k6) * X) * (h * b);
    const double y2 = ((2.0 / 15.0) * g.k6) * Y, yb = y2 * b, yh = y2 * h;
    const double ya = (2.0 * yb) * (2.0 * S - 3.0 * h);
    const double ybi = -(yb * ai) * (3.0 * ai + S), ybj = -(yb * aj) * (3.0 * aj + S);
    const double yci = (4.0 * yh) * (ai * ai), ycj = (4.0 * yh) * (aj * aj), ycx = yh * AB;
    // 2 E.n = rate (n_y, n_x, 0)
    const double e = 0.5 * S * rate;
    const V G = mk3<double>((Vi.x - Vj.x) - e * n.y, (Vi.y - Vj.y) - e * n.x, Vi.z - Vj.z);
    const double nG = dot(n, G);
    const V nW = cross(n, ybi * Wi + ybj * Wj), nxG = cross(n, G);
    const double fn = (ya - xa) * nG;
    V Fl = mk3<double>(fn * n.x - ya * G.x - nW.x, fn * n.y - ya * G.y - nW.y, fn * n.z - ya * G.z - nW.z);
    V Tli = ybi * nxG - tang(n, yci * Wi + ycx * Wj);
    V Tlj = ybj * nxG - tang(n, ycx * Wi + ycj * Wj);
    if (g.taper > 0.0) {
      const double dl = g.mode == 1 ? g.delta * g.a0 : g.delta * (0.5 * S);
      const double t = (dl - d) / (g.taper * dl);
      if (t < 1.0) {
        const double s = t > 0.0 ? t * t * (3.0 - 2.0 * t) : 0.0;
        Fl = s * Fl;
        Tli = s * Tli;
        Tlj = s * Tlj;
      }
    }
    o.Fl = Fl;
    o.F = Fc + Fl;
    o.Ti = o.Ti + Tli;
    o.Tj = o.Tj + Tlj;
  }
  return o;
}
