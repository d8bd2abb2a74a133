// The double form's interface levels and edge solution (the single form's are
// iface_unit and edge_unit in stage.cuh).
//
// On this GPU the FP64 pipe has two lanes per SM, so every kernel of the
// double form runs at 89-92% of it and its time is its count of FP64
// operations (library calls in pipe slots: exp 15, erf 45, erfc 62, expm1 19,
// a/b 8, sqrt 8, 1/x 5, rsqrt 5). The formulation here is the one with the
// fewest (measured with 501 k triangles, 753 k edges): 1211 -> 777 per edge,
// layer and point (k_edge<double> 6595 -> 4274 us) and 341 -> 274 per edge and
// layer (k_iface<double> 954 -> 763 us), then, with the sides' values kept by
// k_iface and the results rotated once per edge, 633 (k_edge<double> 582 -> 496
// us at 65,522 triangles):
//   - face-frame evaluation: the derivatives are formed along n and t at
//     once, a mirrored side through the frame that its cell sees;
//   - half-space moments split into a full-space and a boundary part, and the
//     equilibrium's two sides summed before its moments are taken;
//   - the fit's weights in closed form, where most parts cancel;
//   - one reciprocal root per side in place of three divisions and two roots,
//     and the error function by its series where its argument is small.
// Every operation is rounded as written (Rn), so that the kernels which form
// the same value get the same bits whatever code surrounds them.
#pragma once
#include "stage.cuh"

namespace gks2l {

using D64 = Rn<double>;

// erf(z)/2 for |z| <= 1/2 by the Maclaurin series 1/sqrt(pi) sum_n (-1)^n
// z^(2n+1) / (n! (2n+1)); the first term left out is below 2^-58 of the sum.
// Larger arguments take the library's: normal Froude numbers above 0.5 (z = U /
// sqrt(G h)), and in the blend U_n^l + U_n^r above 1 (z is half their sum).
constexpr int kErfTerms = 13;
struct ErfSeries {
  double c[kErfTerms];
  constexpr ErfSeries() : c() {
    double f = 1;
    for (int n = 0; n < kErfTerms; n++) {
      if (n > 0) f *= n;
      c[n] = (n % 2 ? -1.0 : 1.0) * 0.56418958354775628694807945156077 / (f * (2 * n + 1));
    }
  }
};
// |x| <= 1/2 by the bits, off the FP64 pipe
__host__ __device__ __forceinline__ bool within_half(double x) {
  return (dbits(x) & 0x7fffffffffffffffll) <= 0x3fe0000000000000ll;
}
__host__ __device__ __forceinline__ double half_erf(double z) {
  constexpr ErfSeries S;
  if (!within_half(z)) return 0.5 * erf(z);
  const double y = D64::mul(z, z);
  double s = S.c[kErfTerms - 1];
#pragma unroll
  for (int n = kErfTerms - 2; n >= 0; n--) s = D64::fma(s, y, S.c[n]);
  return D64::mul(z, s);
}
__host__ __device__ __forceinline__ double half_erfc(double x) {
  if (!within_half(x)) return 0.5 * erfc(x);
  return D64::sub(0.5, half_erf(x));
}

// Taylor monomials of degree 1..3 at (x, y): m[1..9]. Their x- and
// y-derivatives are the lower ones again: d/dx of m[1], m[3], m[4], m[6],
// m[7], m[8] is 1, m[1], m[2], m[3], m[4], m[5], and d/dy of m[2], m[4],
// m[5], m[7], m[8], m[9] is 1, m[1], m[2], m[3], m[4], m[5].
__host__ __device__ __forceinline__ void monos64(double x, double y, double m[10]) {
  using O = D64;
  m[1] = x;
  m[2] = y;
  m[3] = O::mul(0.5, O::mul(x, x));
  m[4] = O::mul(x, y);
  m[5] = O::mul(0.5, O::mul(y, y));
  m[6] = O::mul(1.0 / 3.0, O::mul(x, m[3]));
  m[7] = O::mul(m[3], y);
  m[8] = O::mul(x, m[5]);
  m[9] = O::mul(1.0 / 3.0, O::mul(y, m[5]));
}
// a polynomial's value (cf[10] the cell average) and its x- and y-derivatives
__host__ __device__ __forceinline__ double poly_val64(const double *cf, const double m[10]) {
  double a = cf[0];
  for (int k = 1; k < 10; k++) a = D64::fma(cf[k], m[k], a);
  return D64::add(cf[10], a);
}
__host__ __device__ __forceinline__ void poly_grad64(const double *cf, const double m[10], double &gx, double &gy) {
  using O = D64;
  gx = O::fma(cf[4], m[2], O::fma(cf[3], m[1], cf[1]));
  gy = O::fma(cf[5], m[2], O::fma(cf[4], m[1], cf[2]));
  for (int k = 3; k < 6; k++) {
    gx = O::fma(cf[k + 3], m[k], gx);
    gy = O::fma(cf[k + 4], m[k], gy);
  }
}

// The normal n and tangent (-n1, n0) of an edge as seen in the frame of a side
// whose cell appears through transform xf (the image of a vector v is M v, so
// its component along n is v . M^T n): fr = (n, t). Only a wall's mirrored
// side has a transform.
__host__ __device__ __forceinline__ void face_frame(const Dev &d, double n0, double n1, int xf, double fr[4]) {
  using O = D64;
  fr[0] = n0; fr[1] = n1; fr[2] = -n1; fr[3] = n0;
  if (xf != 0) {
    const double *M = d.xf + 4 * xf;
    fr[0] = O::fma(M[0], n0, O::mul(M[2], n1));
    fr[1] = O::fma(M[1], n0, O::mul(M[3], n1));
    fr[2] = O::fma(M[2], n0, -O::mul(M[0], n1));
    fr[3] = O::fma(M[3], n0, -O::mul(M[1], n1));
  }
}

// Blended level deviation at one point (Sec. 2.3): d^r + xi (d^l - d^r) with
// xi = erfc((U_n^l + U_n^r)/2)/2.
__host__ __device__ __forceinline__ double blend64(double dl, double ul, double dr, double ur) {
  using O = D64;
  return O::fma(half_erfc(O::mul(0.5, O::add(ul, ur))), O::sub(dl, dr), dr);
}

// One side's values at a point: the level deviation, the velocity along n and
// t and the depth's inverse root
struct Point64 {
  double d, U, V, r;
};
__host__ __device__ __forceinline__ Point64 point64(const double *w, const double m[10], const double fr[4],
                                                    double href) {
  using O = D64;
  Point64 v;
  v.d = poly_val64(w, m);
  v.r = r_rsqrt(O::add(href, v.d));
  const double ih = O::mul(v.r, v.r), mx = poly_val64(w + 12, m), my = poly_val64(w + 24, m);
  v.U = O::mul(O::fma(mx, fr[0], O::mul(my, fr[1])), ih);
  v.V = O::mul(O::fma(mx, fr[2], O::mul(my, fr[3])), ih);
  return v;
}

// iface_unit in the double form, by two lanes, one per side (sd): each hands
// the other its values at one point and blends at the other, and the two
// layers' lanes form one point's monomials each and exchange. The sides' values
// are kept for the edge solution (write), which would form them again.
#ifdef __CUDACC__
__device__ __forceinline__ double iface_unit64(const Dev &d, int e, int ell, int sd, bool write) {
  using O = D64;
  const EdgeIds g = edge_ids(d, e);
  double x[2][2], n[2], fr[4], w[NREC], m[2][10], lev[2], un[2];
  for (int q = 0; q < 2; q++) load_n<double, 2>((const double *)d.exi + ((size_t)q * d.ne + e) * 4 + 2 * sd, x[q]);
  load_n<double, 2>((const double *)d.en + 2 * (size_t)e, n);
  face_frame(d, n[0], n[1], sd == 0 ? 0 : g.xf, fr);
  load_rec<double, NREC>(d, ell, sd == 0 ? g.L : g.R, w);
  {
    double mine[10];
    monos64(ell == 0 ? x[0][0] : x[1][0], ell == 0 ? x[0][1] : x[1][1], mine);
    for (int k = 1; k < 10; k++) {
      const double theirs = __shfl_xor_sync(0xffffffffu, mine[k], 2);
      m[0][k] = ell == 0 ? mine[k] : theirs;
      m[1][k] = ell == 0 ? theirs : mine[k];
    }
  }
  for (int q = 0; q < 2; q++) {
    const Point64 v = point64(w, m[q], fr, ref_depth<double>(d, ell, e, q));
    const double t[4] = {v.d, v.U, v.V, v.r};
    if (write) store_n<double, 4>(d.ept + ((((size_t)e * 2 + ell) * 2 + q) * 2 + sd) * 4, t);
    lev[q] = v.d;
    un[q] = v.U;
  }
  const double ml = sd == 0 ? lev[0] : lev[1], mu = sd == 0 ? un[0] : un[1];
  const double tl = __shfl_xor_sync(0xffffffffu, sd == 0 ? lev[1] : lev[0], 1);
  const double tu = __shfl_xor_sync(0xffffffffu, sd == 0 ? un[1] : un[0], 1);
  const double b = sd == 0 ? blend64(ml, mu, tl, tu) : blend64(tl, tu, ml, mu);
  return O::mul(0.5, O::add(b, __shfl_xor_sync(0xffffffffu, b, 1)));
}
#endif

// Edge-point side data for one layer, deviations, in the face's frame (n, t).
struct Side64 {
  double d;              // level deviation at the point (eta1 - R1 or h2 - R2)
  double h, r, ih;       // depth at the point (href + d), its inverse root and its inverse
  double U, V;           // velocity along n and t
  double dn[3], dt[3];   // derivatives along n and t of (depth, m_n, m_t)
  double lev[2];         // derivatives along n and t of the level
  double oth[2];         // the same of the other layer's level
};

// derivatives along n and t of the level polynomial cf, from the frame scaled by 1/h_s
__host__ __device__ __forceinline__ void level_dirs(const double *cf, const double m[10], const double fs[4],
                                                    double lev[2]) {
  using O = D64;
  double gx, gy;
  poly_grad64(cf, m, gx, gy);
  lev[0] = O::fma(gx, fs[0], O::mul(gy, fs[1]));
  lev[1] = O::fma(gx, fs[2], O::mul(gy, fs[3]));
}

// One side of an edge point: cell c's reconstruction of layer ell at the point
// of m, in the frame fr as that cell sees it; href is the depth of the
// reference level at the point. OTHER: also the other layer's level
// derivatives from its record (otherwise the caller takes them from the lane
// that forms them as its own). have: the side's values from k_iface, or null.
template <bool OTHER>
__host__ __device__ __forceinline__ void side64(const Dev &d, int ell, int c, int xf, const double fr[4],
                                                const double m[10], double href, const double *have, Side64 &s) {
  using O = D64;
  double w[NREC];
  load_rec<double, NREC>(d, ell, c, w);
  const double ih = w[11];
  double fs[4] = {O::mul(fr[0], ih), O::mul(fr[1], ih), 0, 0};
  fs[2] = -fs[1];
  fs[3] = fs[0];
  if (xf != 0) {
    fs[2] = O::mul(fr[2], ih);
    fs[3] = O::mul(fr[3], ih);
  }
  Point64 v;
  if (have) {
    double t[4];
    load_n<double, 4>(have, t);
    v = {t[0], t[1], t[2], t[3]};
  } else {
    v = point64(w, m, fr, href);
  }
  s.d = v.d;
  s.h = O::add(href, v.d);
  s.r = v.r;
  s.ih = O::mul(v.r, v.r);
  s.U = v.U;
  s.V = v.V;
  level_dirs(w, m, fs, s.lev);
  // the depth is the level less the bottom in the lower layer (its slots 1, 2
  // carry grad B)
  s.dn[0] = s.lev[0];
  s.dt[0] = s.lev[1];
  if (ell == 0) {
    s.dn[0] = O::fma(-w[23], fr[0], O::fma(-w[35], fr[1], s.dn[0]));
    s.dt[0] = O::fma(-w[23], fr[2], O::fma(-w[35], fr[3], s.dt[0]));
  }
  double xx, xy, yx, yy;
  poly_grad64(w + 12, m, xx, xy);
  poly_grad64(w + 24, m, yx, yy);
  for (int k = 0; k < 2; k++) {
    double *o = k == 0 ? s.dn : s.dt;
    const double px = O::fma(xx, fs[2 * k], O::mul(xy, fs[2 * k + 1]));
    const double py = O::fma(yx, fs[2 * k], O::mul(yy, fs[2 * k + 1]));
    o[1] = O::fma(px, fr[0], O::mul(py, fr[1]));
    o[2] = O::fma(px, fr[2], O::mul(py, fr[3]));
  }
  s.oth[0] = s.oth[1] = 0;
  if (OTHER) {
    double wo[12];
    load_rec<double, 12>(d, 1 - ell, c, wo);
    level_dirs(wo, m, fs, s.oth);
  }
}

// plane gradient (Sec. 2.3) of the blended level `which` for cell c, along n
// and t of the frame fr
__host__ __device__ __forceinline__ void plane_dirs(const Dev &d, int c, int which, const double fr[4],
                                                    double out[2]) {
  using O = D64;
  double g[2];
  plane_grad<double>(d, c, which, g);
  out[0] = O::fma(g[0], fr[0], O::mul(g[1], fr[1]));
  out[1] = O::fma(g[0], fr[2], O::mul(g[1], fr[3]));
}

// Slope + force kernel of one side on a Maxwellian base (U, V, th = G h / 2),
// written as a polynomial in c = u - U and multiplied by h th, which leaves
// only the base's velocity in it: the exact derivative of ln g along n and t,
//   gu c_u + gv c_v + puu c_u^2 + puv c_u c_v + pvv c_v^2,
// plus the force term, whose cubic part combines into |c|^2 (bu c_u + bv c_v),
// b = D / 2 with D = grad h - grad Phi / G (local frame).
struct Kern64 {
  double gu, gv, puu, puv, pvv, bu, bv;
};
__host__ __device__ __forceinline__ Kern64 make_kern64(double U, double V, const double dn[3], const double dt[3],
                                                       const double D[2]) {
  using O = D64;
  const double an = O::fma(-U, dn[0], dn[1]), at = O::fma(-U, dt[0], dt[1]);
  const double bn = O::fma(-V, dn[0], dn[2]), bt = O::fma(-V, dt[0], dt[2]);
  const double ah = O::mul(0.5, O::fma(U, dn[0], O::mul(V, dt[0])));
  Kern64 K;
  K.gu = O::fma(U, an, O::mul(V, at));
  K.gv = O::fma(U, bn, O::mul(V, bt));
  K.puu = O::add(ah, an);
  K.pvv = O::add(ah, bt);
  K.puv = O::add(bn, at);
  K.bu = O::mul(0.5, D[0]);
  K.bv = O::mul(0.5, D[1]);
  return K;
}

// Moments of a kernel on its base, h <.> (h cancels the kernel's scaling).
// On a half line sgn u > 0 every central moment <c^k> is a_k m + b_k e with
// m = <1> the half line's share, e = sgn E its boundary density (E =
// e^{-lam U^2} / (2 sqrt(pi lam)), lam = 1 / (2 th)), a = (1, 0, th, 0,
// 3 th^2, 0) and b = (0, 1, -U, 2 th + U^2, ...): a moment of the kernel is
// its full-space value times m plus a boundary part times e. In the raw
// moments with u, u^2 and u v the boundary parts lose all but a few terms,
// the weight u vanishing at u = 0.
struct Full64 {   // full space: <1>, <c_u>, <c_v>, <c_u^2>, <c_u c_v>
  double t00, t10, t01, t20, t11;
};
__host__ __device__ __forceinline__ Full64 full_moments(const Kern64 &K, double th) {
  using O = D64;
  const double th4 = O::mul(4.0, th);
  Full64 f;
  f.t00 = O::add(K.puu, K.pvv);
  f.t10 = O::fma(th4, K.bu, K.gu);
  f.t01 = O::fma(th4, K.bv, K.gv);
  f.t20 = O::mul(th, O::fma(3.0, K.puu, K.pvv));
  f.t11 = O::mul(th, K.puv);
  return f;
}
struct Bound64 {  // boundary parts of <1>, <u>, <c_v>, and of <u c_v>
  double b0, b1, b2, b5;
};
__host__ __device__ __forceinline__ Bound64 bound_moments(const Kern64 &K, double U, double th, double ith) {
  using O = D64;
  Bound64 b;
  const double q = O::fma(U, U, O::mul(3.0, th));
  b.b0 = O::mul(ith, O::fma(K.bu, q, O::fma(-U, K.puu, K.gu)));
  b.b1 = O::fma(-U, K.bu, O::fma(2.0, K.puu, K.pvv));
  b.b2 = O::fma(-U, K.bv, K.puv);
  b.b5 = O::fma(O::mul(5.0, th), K.bv, K.gv);
  return b;
}
// raw moments of one side's kernel over its half line: 1, u, v, u^2, u v
__host__ __device__ __forceinline__ void side_moments(const Kern64 &K, double U, double V, double th, double ith,
                                                      double m, double e, double o[5]) {
  using O = D64;
  const Full64 f = full_moments(K, th);
  const Bound64 b = bound_moments(K, U, th, ith);
  o[0] = O::fma(m, f.t00, O::mul(e, b.b0));
  o[1] = O::fma(m, O::fma(U, f.t00, f.t10), O::mul(e, b.b1));
  o[2] = O::fma(V, o[0], O::fma(m, f.t01, O::mul(e, b.b2)));
  const double u2 = O::fma(U, O::fma(U, f.t00, O::add(f.t10, f.t10)), f.t20);
  const double b4 = O::fma(U, f.t00, O::fma(2.0, K.gu, O::mul(O::mul(10.0, th), K.bu)));
  o[3] = O::fma(m, u2, O::mul(e, b4));
  o[4] = O::fma(V, o[1], O::fma(m, O::fma(U, f.t01, f.t11), O::mul(e, b.b5)));
}

// e^{-z^2}, sqrt(h), half the error function and E of a Maxwellian, with z =
// sqrt(lam) U; r the depth's inverse root
struct Maxw64 {
  double x, s, e0, E;
};
__host__ __device__ __forceinline__ Maxw64 maxwellian(const Par &p, double h, double r, double U) {
  using O = D64;
  Maxw64 m;
  const double z = O::mul(U, O::mul(r, p.rg));
  m.x = r_exp<double>(-O::mul(z, z));
  m.s = O::mul(h, r);
  m.e0 = half_erf(z);
  m.E = O::mul(O::mul(p.cphi, m.s), m.x);
  return m;
}

// gks_layer in the double form. The solution is a combination of five parts:
// C1 (equilibrium), C2 (its slopes), C3 (its time derivative, by
// compatibility), C4 (free transport) and C5 (its slopes). So are its time
// integrals over [0, delta] and [0, delta/2] and the value and time derivative
// at the stage start that reproduce both, with weights kv_i and kd_i: with
// s = tau/delta, x = 1/(2 s), eh = e^{-x}, em = 1 - eh
//   kv4 = s em (2 + em),  kv1 = 1 - kv4,  kv3 = -tau kv1,
//   kv5 = tau (eh (2 - eh) - kv4),  kv2 = kv3 - kv5,
//   kd1 = -kd4 = 4 s em^2 / delta,  kd3 = 1 - 4 (s em)^2,
//   kd5 = 4 s em (s em - eh),  kd2 = kd3 - 1 - kd5,
// so only C1, C4 - C1, C2 + C3 and C5 - C2 enter, and C4 - C1 and C2 + C3
// vanish for 1, u and v (conservation and the compatibility condition).
__host__ __device__ inline void gks_layer64(const Par &p, double href, const Side64 &l, const Side64 &r,
                                            const double Dl[2], const double Dr[2], double dt, double idt, double F[3],
                                            double Ft[3], double W[3], double Wt[3]) {
  using O = D64;
  const double g = p.g, hg = 0.5 * p.g;
  const double hl = l.h, hr = r.h, Ul = l.U, Ur = r.U;
  const double dlr = O::sub(l.d, r.d);                  // h_l - h_r, exact at rest
  const double thl = O::mul(hg, hl), thr = O::mul(hg, hr);
  const Maxw64 L = maxwellian(p, hl, l.r, Ul), Q = maxwellian(p, hr, r.r, Ur);
  const double ml = O::add(0.5, L.e0), mr = O::sub(0.5, Q.e0);       // <1> over the half lines
  const double nl = O::fma(Ul, ml, L.E), nr = O::fma(Ur, mr, -Q.E);  // <u>
  // W-bar: the t = 0 interface state; h_b = (h_l + h_r)/2, h-bar = h_b + hdev
  const double db = O::mul(0.5, O::add(l.d, r.d));      // h_b - href
  const double hb = O::add(href, db);
  const double hdev = O::fma(hl, L.e0, -O::mul(hr, Q.e0));
  // h_l E_l - h_r E_r with h E = sqrt(G/(4 pi)) h^{3/2} e^{-z^2}, written
  // through h_l - h_r so that it vanishes exactly for equal depths and velocities
  const double dphi = O::mul(O::mul(dlr, O::fma(L.s, Q.s, O::add(hl, hr))), 1 / O::add(L.s, Q.s));
  const double ediff = O::mul(p.cphi, O::fma(O::mul(hl, L.s), O::sub(L.x, Q.x), O::mul(dphi, Q.x)));
  const double wl = O::mul(hl, ml), wr = O::mul(hr, mr);
  const double mbn = O::add(O::fma(wl, Ul, O::mul(wr, Ur)), ediff);
  const double mbt = O::fma(wl, l.V, O::mul(wr, r.V));
  const double hbR = O::add(hb, hdev), rb = r_rsqrt(hbR), ihb = O::mul(rb, rb);
  const double Ub = O::mul(mbn, ihb), Vb = O::mul(mbt, ihb);
  const double thb = O::mul(hg, hbR), ithb = O::mul(p.ig2, ihb);
  const Maxw64 B = maxwellian(p, hbR, rb, Ub);
  const double mb = O::add(0.5, B.e0);
  // C2: the left kernel over u > 0 and the right one over u < 0 on the same
  // base are the kernel of the mixed slopes in full space plus the boundary
  // part of the difference. a: raw moments with 1, u, v, u^2, u v; s4, s5:
  // C2 + C3 for u^2 and u v, central moments
  double a[5], s4, s5;
  {
    double xn[3], xt[3], xd[2], yn[3], yt[3], yd[2];
    for (int i = 0; i < 3; i++) {
      xn[i] = O::sub(l.dn[i], r.dn[i]);
      xt[i] = O::sub(l.dt[i], r.dt[i]);
      yn[i] = O::fma(mb, xn[i], r.dn[i]);
      yt[i] = O::fma(mb, xt[i], r.dt[i]);
    }
    for (int i = 0; i < 2; i++) {
      xd[i] = O::sub(Dl[i], Dr[i]);
      yd[i] = O::fma(mb, xd[i], Dr[i]);
    }
    const Kern64 ky = make_kern64(Ub, Vb, yn, yt, yd), kx = make_kern64(Ub, Vb, xn, xt, xd);
    const Full64 f = full_moments(ky, thb);
    const Bound64 b = bound_moments(kx, Ub, thb, ithb);
    a[0] = O::fma(B.E, b.b0, f.t00);
    a[1] = O::fma(B.E, b.b1, O::fma(Ub, f.t00, f.t10));
    a[2] = O::fma(Vb, a[0], O::fma(B.E, b.b2, f.t01));
    const double t = O::fma(4.0, O::mul(thb, kx.bu), O::mul(Ub, O::fma(Ub, b.b0, -O::add(kx.puu, kx.pvv))));
    s4 = O::fma(B.E, t, O::mul(thb, O::sub(ky.puu, ky.pvv)));
    s5 = O::fma(B.E, O::fma(-Ub, b.b2, b.b5), f.t11);
    a[3] = O::add(s4, O::fma(2.0, O::mul(Ub, a[1]), O::mul(O::fma(-Ub, Ub, O::add(thb, thb)), a[0])));
    a[4] = O::add(s5, O::fma(Vb, a[1], O::mul(Ub, O::fma(-Vb, a[0], a[2]))));
  }
  // C5 - C2: each side's kernel on its own base and half line
  double ol[5], qr[5], e[5];
  side_moments(make_kern64(Ul, l.V, l.dn, l.dt, Dl), Ul, l.V, thl, O::mul(p.ig2, l.ih), ml, L.E, ol);
  side_moments(make_kern64(Ur, r.V, r.dn, r.dt, Dr), Ur, r.V, thr, O::mul(p.ig2, r.ih), mr, -Q.E, qr);
  for (int i = 0; i < 5; i++) e[i] = O::sub(O::add(ol[i], qr[i]), a[i]);
  // C1 (full-space moments of g-bar) and C4 (g^l, g^r on their half spaces)
  // for u^2 and u v, deviations from the base G h_b^2 / 2
  const double c14 = O::fma(mbn, Ub, O::mul(O::mul(g, hdev), O::fma(0.5, hdev, hb)));
  const double c15 = O::mul(mbn, Vb);
  const double c44 = O::fma(hl, O::fma(Ul, nl, O::mul(thl, L.e0)),
                            O::fma(hr, O::fma(Ur, nr, -O::mul(thr, Q.e0)), O::mul(0.125 * g, O::mul(dlr, dlr))));
  const double c45 = O::fma(O::mul(hl, l.V), nl, O::mul(O::mul(hr, r.V), nr));
  const double x4 = O::sub(c44, c14), x5 = O::sub(c45, c15);
  // collision time (Sec. 4): tau = eps dt + eps_num |(hl^2 - hr^2)/(hl^2 + hr^2)| dt,
  // with one reciprocal for s = tau/dt = v/u and 1/s
  const double u = O::fma(hl, hl, O::mul(hr, hr));
  const double v = O::fma(p.eps_num, r_abs<double>(O::mul(dlr, O::add(hl, hr))), O::mul(p.eps, u));
  const double iuv = 1 / O::mul(u, v);
  const double s = O::mul(v, O::mul(v, iuv)), tau = O::mul(s, dt);
  const double em = -r_expm1<double>(O::mul(-0.5, O::mul(u, O::mul(u, iuv)))), eh = O::sub(1.0, em);
  const double sem = O::mul(s, em), sem4 = O::mul(4.0, sem);
  const double kv4 = O::mul(sem, O::add(2.0, em)), kv3 = O::mul(tau, O::sub(kv4, 1.0));
  const double kv5 = O::mul(tau, O::fma(eh, O::sub(2.0, eh), -kv4));
  const double kd1 = O::mul(O::mul(sem4, em), idt), kd3 = O::fma(-sem4, sem, 1.0), kd5 = O::mul(sem4, O::sub(sem, eh));
  // bases relative to the reference: h_b - href and G (h_b^2 - href^2) / 2
  W[0] = O::add(db, O::fma(kv5, e[0], hdev));
  W[1] = O::fma(kv5, e[1], mbn);
  W[2] = O::fma(kv5, e[2], mbt);
  for (int i = 0; i < 3; i++) Wt[i] = O::fma(kd5, e[i], -a[i]);
  F[0] = W[1];
  F[1] = O::fma(O::mul(hg, db), O::add(hb, href), O::fma(kv5, e[3], O::fma(kv3, s4, O::fma(kv4, x4, c14))));
  F[2] = O::fma(kv5, e[4], O::fma(kv3, s5, O::fma(kv4, x5, c15)));
  Ft[0] = Wt[1];
  Ft[1] = O::fma(kd5, e[3], O::fma(kd3, s4, O::fma(-kd1, x4, -a[3])));
  Ft[2] = O::fma(kd5, e[4], O::fma(kd3, s5, O::fma(-kd1, x5, -a[4])));
}

// edge_unit in the double form (see there for the modes). The two lanes of an
// edge's layer form one side's plane gradients each, and with PAIRED the two
// layers' lanes one side's monomials each, and exchange: shuffles cost the
// FP64 pipe nothing. HAVE: k_iface has left the sides' values. The vectors of
// out stay in the face's frame.
template <bool FUSED, bool PAIRED, bool POS, bool HAVE>
__host__ __device__ inline bool edge_unit64(const Dev &d, const Par &p, int e, int ell, int q, double out[12],
                                            double *blend, double *own) {
  using O = D64;
  const EdgeIds g = edge_ids(d, e);
  const int cL = g.L, cR = g.R, xf = g.xf, in = g.inst;
  double x[4], n[2];
  load_n<double, 4>((const double *)d.exi + ((size_t)q * d.ne + e) * 4, x);
  load_n<double, 2>((const double *)d.en + 2 * (size_t)e, n);
  // both stages fit the value and time derivative at their start from the
  // time integrals over dt and dt/2 (reading R20)
  const double dt = ((const double *)d.dtR)[in], idt = ((const double *)d.dtR)[d.ninst + in];
  const double href = ref_depth<double>(d, ell, e, q);
  const double n0 = n[0], n1 = n[1];
  double fr[2][4], m[2][10];
  face_frame(d, n0, n1, 0, fr[0]);
  face_frame(d, n0, n1, xf, fr[1]);
#ifdef __CUDA_ARCH__
  constexpr bool SH = PAIRED;
#else
  constexpr bool SH = false;
#endif
  if (!SH) {
    monos64(x[0], x[1], m[0]);
    monos64(x[2], x[3], m[1]);
  }
#ifdef __CUDA_ARCH__
  if (SH) {
    double mine[10];
    monos64(ell == 0 ? x[0] : x[2], ell == 0 ? x[1] : x[3], mine);
#pragma unroll
    for (int k = 1; k < 10; k++) {
      const double theirs = __shfl_xor_sync(0xffffffffu, mine[k], 2);
      m[0][k] = ell == 0 ? mine[k] : theirs;
      m[1][k] = ell == 0 ? theirs : mine[k];
    }
  }
#endif
  Side64 s[2];
  const double *have = HAVE ? d.ept + (((size_t)e * 2 + ell) * 2 + q) * 8 : nullptr;
  side64<!SH>(d, ell, cL, 0, fr[0], m[0], href, have, s[0]);
  side64<!SH>(d, ell, cR, xf, fr[1], m[1], href, HAVE ? have + 4 : nullptr, s[1]);
#ifdef __CUDA_ARCH__
  if (SH) {
    for (int sd = 0; sd < 2; sd++)
      for (int k = 0; k < 2; k++) s[sd].oth[k] = __shfl_xor_sync(0xffffffffu, s[sd].lev[k], 2);
  }
#endif
  // blended derivative of the other layer's level and the well-balance vector
  // D = grad h - grad Phi / G = grad(level) + c (w grad(other) + (1 - w) grad P1)
  const int oth = 1 - ell;  // hc / omg index of the other layer: 0 = eta1, 1 = h2
  const double *om = (const double *)d.omg;
  double w = om[oth * d.cs + cL] < om[oth * d.cs + cR] ? om[oth * d.cs + cL] : om[oth * d.cs + cR];
  w = w < 0 ? 0 : (w > 1 ? 1 : w);
  double pl[2][2] = {{0, 0}, {0, 0}};
  if (!FUSED) {
#ifdef __CUDA_ARCH__
    double mine[2], fq[4];
    for (int k = 0; k < 4; k++) fq[k] = q == 0 ? fr[0][k] : fr[1][k];
    plane_dirs(d, q == 0 ? cL : cR, oth, fq, mine);
    for (int k = 0; k < 2; k++) {
      const double theirs = __shfl_xor_sync(0xffffffffu, mine[k], 1);
      pl[0][k] = q == 0 ? mine[k] : theirs;
      pl[1][k] = q == 0 ? theirs : mine[k];
    }
#else
    plane_dirs(d, cL, oth, fr[0], pl[0]);
    plane_dirs(d, cR, oth, fr[1], pl[1]);
#endif
  }
  const double cf = ell == 0 ? p.chi : 1.0, w1 = O::sub(1.0, w);
  double D[2][2];
  for (int sd = 0; sd < 2; sd++)
    for (int k = 0; k < 2; k++)
      D[sd][k] = O::fma(cf, FUSED ? s[sd].oth[k] : O::fma(w, s[sd].oth[k], O::mul(w1, pl[sd][k])), s[sd].lev[k]);
  if (FUSED) *blend = blend64(s[0].d, s[0].U, s[1].d, s[1].U);
  if (POS) {
    const int N = d.cs;
    const bool fl[2] = {d.pos_flag[ell * N + cL] != 0, d.pos_flag[ell * N + cR] != 0};
    if (fl[0] || fl[1]) {
      const double *hb = (const double *)d.pos_hbar;
      double un[2], ut[2];
      for (int sd = 0; sd < 2; sd++) {
        const int c = sd == 0 ? cL : cR;
        const double *mq = dq_at<double>(d, ell == 0 ? 2 : 1, c);
        const double mx = mq[0], my = mq[1], ihb = 1 / hb[ell * N + c];
        un[sd] = O::mul(O::fma(mx, fr[sd][0], O::mul(my, fr[sd][1])), ihb);
        ut[sd] = O::mul(O::fma(mx, fr[sd][2], O::mul(my, fr[sd][3])), ihb);
      }
      const double ulo = un[0] < un[1] ? un[0] : un[1], uhi = un[0] < un[1] ? un[1] : un[0];
      const double tlo = ut[0] < ut[1] ? ut[0] : ut[1], thi = ut[0] < ut[1] ? ut[1] : ut[0];
      for (int sd = 0; sd < 2; sd++) {
        if (!fl[sd]) continue;
        s[sd].U = s[sd].U < ulo ? ulo : (s[sd].U > uhi ? uhi : s[sd].U);
        s[sd].V = s[sd].V < tlo ? tlo : (s[sd].V > thi ? thi : s[sd].V);
      }
    }
  }
  // each side's own level at the point: the interlayer source's values (R16)
  if (own) {
    own[0] = s[0].d;
    own[1] = s[1].d;
  }
  if (FUSED && w < 1) return false;
  gks_layer64(p, href, s[0], s[1], D[0], D[1], dt, idt, out, out + 3, out + 6, out + 9);   // F, F_t, W, W_t
  return true;
}

// The mean over an edge's two points of (F, F_t) or (W, W_t) from the points'
// sum in the face's frame, in the global frame
__host__ __device__ __forceinline__ void mean64(const Dev &d, int e, const double sum[6], double avg[6]) {
  using O = D64;
  double n[2];
  load_n<double, 2>((const double *)d.en + 2 * (size_t)e, n);
  const double h0 = O::mul(0.5, n[0]), h1 = O::mul(0.5, n[1]);
  for (int k = 0; k < 6; k += 3) {
    avg[k] = O::mul(0.5, sum[k]);
    avg[k + 1] = O::fma(sum[k + 1], h0, -O::mul(sum[k + 2], h1));
    avg[k + 2] = O::fma(sum[k + 1], h1, O::mul(sum[k + 2], h0));
  }
}

}  // namespace gks2l
