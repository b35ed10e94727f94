// su2_kick.cuh -- the kick of one site of the doublet models (SU(2) x U(1) doublet,
// and with FULL the lphi4SU2U1 model's singlet and U(1)-charged scalar), shared by the
// two passes: each plaquette formed once and its values carried along z.
//
// A thread marches up in z.  Each plaquette is formed once per site (xy, xz, yz at n) and serves the
// staples of its links at n directly (P and P^dag); along z it also serves the
// two links it reaches from below, rotated by a link,
//     m(L_iz(n)) = m(U_z^dag(n-z) P_iz(n-z)^dag U_z(n-z)),
// which the thread forms at plane z - 1 and carries to plane z in registers.
// The lower staples across x and y are formed directly at each site (handing
// them on between lanes would leave the tile's edge column to one lane of a
// warp, which costs the whole warp the work).  The same goes for the compact
// U(1) plaquette sines and the backward hops W_i^dag(n-i) psi(n-i): carried
// along z, direct across x and y.  In the FP32 passes that need no gauge energies the
// seven U(1) plaquette sines are evaluated two at a time and the six plaquette products and
// four lower staples are formed two at a time, in the packed two-lane FP32 form,
// each lane rounded as the single evaluation (trig2.cuh, Q2 below).
//
// What a pass sums (RED): 0 nothing; 1 the Friedmann kicks' sums; 2 a full measurement;
// SU2_RED_ALPHA1 the Friedmann kicks' sums at alpha = 1, where the gauge fields' energies
// enter with alpha - 1 = 0 and are not formed.
#pragma once

#include "su2_common.cuh"
#include "trig2.cuh"

namespace clg {

namespace {

template <typename T>
struct V3 {
  T x, y, z;
};

// vector part (a b)_{x,y,z} of a quaternion product
template <typename T>
__device__ __forceinline__ V3<T> qvec(const Q4<T>& a, const Q4<T>& b) {
  V3<T> r;
  r.x = fmaT(a.y, b.z, fmaT(-a.z, b.y, fmaT(b.w, a.x, a.w * b.x)));
  r.y = fmaT(a.z, b.x, fmaT(-a.x, b.z, fmaT(b.w, a.y, a.w * b.y)));
  r.z = fmaT(a.x, b.y, fmaT(-a.y, b.x, fmaT(b.w, a.z, a.w * b.z)));
  return r;
}
// scalar part (a b)_w
template <typename T>
__device__ __forceinline__ T qsca(const Q4<T>& a, const Q4<T>& b) {
  return fmaT(-a.z, b.z, fmaT(-a.y, b.y, fmaT(-a.x, b.x, a.w * b.w)));
}
// vector part of U^dag (v.s) U for a unit quaternion U = (u0, u): the rotation
// of v by U^dag,  v + 2 (u x t - u0 t),  t = u x v
template <typename T>
__device__ __forceinline__ V3<T> rotc(const Q4<T>& u, const V3<T>& v) {
  const T tx = fmaT(u.y, v.z, -u.z * v.y), ty = fmaT(u.z, v.x, -u.x * v.z), tz = fmaT(u.x, v.y, -u.y * v.x);
  const T wx = fmaT(u.y, tz, -u.z * ty), wy = fmaT(u.z, tx, -u.x * tz), wz = fmaT(u.x, ty, -u.y * tx);
  V3<T> r;
  r.x = fmaT(T(2), fmaT(-u.w, tx, wx), v.x);
  r.y = fmaT(T(2), fmaT(-u.w, ty, wy), v.y);
  r.z = fmaT(T(2), fmaT(-u.w, tz, wz), v.z);
  return r;
}
template <typename T>
__device__ __forceinline__ V3<T> neg(const V3<T>& v) {
  V3<T> r;
  r.x = -v.x;
  r.y = -v.y;
  r.z = -v.z;
  return r;
}

// Two independent quaternion products at once (FP32, the packed two-lane form):
// lane 0 and lane 1 of every component are the two products, each lane rounded
// exactly as qmul / qvec round one product (a conjugated operand enters by exact
// sign changes, (-a)(-b) = ab), so the pass's results are the same bits.
struct Q2 {
  float2 w, x, y, z;
};
struct P3 {
  float2 x, y, z;
};
__device__ __forceinline__ Q2 q2(const Q4<float>& a, const Q4<float>& b) {
  return Q2{make_float2(a.w, b.w), make_float2(a.x, b.x), make_float2(a.y, b.y), make_float2(a.z, b.z)};
}
__device__ __forceinline__ float2 ng(float2 v) { return make_float2(-v.x, -v.y); }
__device__ __forceinline__ Q4<float> lane_of(const Q2& a, int l) {
  return l ? Q4<float>{a.w.y, a.x.y, a.y.y, a.z.y} : Q4<float>{a.w.x, a.x.x, a.y.x, a.z.x};
}
__device__ __forceinline__ V3<float> lane_of(const P3& a, int l) {
  return l ? V3<float>{a.x.y, a.y.y, a.z.y} : V3<float>{a.x.x, a.y.x, a.z.x};
}
// a b (qmul)
__device__ __forceinline__ Q2 qmul2(const Q2& a, const Q2& b) {
  Q2 r;
  r.w = __ffma2_rn(ng(a.z), b.z, __ffma2_rn(ng(a.y), b.y, __ffma2_rn(ng(a.x), b.x, __fmul2_rn(a.w, b.w))));
  r.x = __ffma2_rn(a.y, b.z, __ffma2_rn(ng(a.z), b.y, __ffma2_rn(b.w, a.x, __fmul2_rn(a.w, b.x))));
  r.y = __ffma2_rn(a.z, b.x, __ffma2_rn(ng(a.x), b.z, __ffma2_rn(b.w, a.y, __fmul2_rn(a.w, b.y))));
  r.z = __ffma2_rn(a.x, b.y, __ffma2_rn(ng(a.y), b.x, __ffma2_rn(b.w, a.z, __fmul2_rn(a.w, b.z))));
  return r;
}
// a b^dag (qmul(a, qconj(b)))
__device__ __forceinline__ Q2 qmul2_cb(const Q2& a, const Q2& b) {
  Q2 r;
  r.w = __ffma2_rn(a.z, b.z, __ffma2_rn(a.y, b.y, __ffma2_rn(a.x, b.x, __fmul2_rn(a.w, b.w))));
  r.x = __ffma2_rn(ng(a.y), b.z, __ffma2_rn(a.z, b.y, __ffma2_rn(b.w, a.x, __fmul2_rn(ng(a.w), b.x))));
  r.y = __ffma2_rn(ng(a.z), b.x, __ffma2_rn(a.x, b.z, __ffma2_rn(b.w, a.y, __fmul2_rn(ng(a.w), b.y))));
  r.z = __ffma2_rn(ng(a.x), b.y, __ffma2_rn(a.y, b.x, __ffma2_rn(b.w, a.z, __fmul2_rn(ng(a.w), b.z))));
  return r;
}
// vector part of a b (qvec)
__device__ __forceinline__ P3 qvec2(const Q2& a, const Q2& b) {
  P3 r;
  r.x = __ffma2_rn(a.y, b.z, __ffma2_rn(ng(a.z), b.y, __ffma2_rn(b.w, a.x, __fmul2_rn(a.w, b.x))));
  r.y = __ffma2_rn(a.z, b.x, __ffma2_rn(ng(a.x), b.z, __ffma2_rn(b.w, a.y, __fmul2_rn(a.w, b.y))));
  r.z = __ffma2_rn(a.x, b.y, __ffma2_rn(ng(a.y), b.x, __ffma2_rn(b.w, a.z, __fmul2_rn(a.w, b.z))));
  return r;
}
// vector part of a b^dag (qvec(a, qconj(b)))
__device__ __forceinline__ P3 qvec2_cb(const Q2& a, const Q2& b) {
  const Q2 r = qmul2_cb(a, b);
  return P3{r.x, r.y, r.z};
}

// Coefficients of a pass in the storage precision: kicks (doublet Laplacian, potential,
// U(1) current and curl, SU(2) current and plaquettes, vphi's current), phases per A_i,
// potential constants.
template <typename T>
struct Su2Coef {
  T A1, A3, AJA, ACA, AJB, AMB, gd, v2, lam, lam2, qG, qH, gdc, AJC;
};
// A pass's coefficients in shared memory, and its drift: of the fields, of the links, and
// half the SU(2) links' drift angle per momentum.
template <typename T>
struct Su2Pass {
  Su2Coef<T> k;
  T cd, cdA, hB;
};
// By one whole warp: lane l forms value l as a product of up to five numbers over a product
// of up to four (in every warp of a CTA and one value after the other they were 89 FP64
// operations a thread, 12 of the 165 us of a 128^3 pass without sums).
template <typename T>
__device__ __noinline__ void su2_coefficients(const LatConst& L, const LatScalars* SC, double ck, double cd,
                                              double cdA, int lane, Su2Pass<T>* out) {
  static_assert(sizeof(Su2Pass<T>) == 17 * sizeof(T), "the values by lane");
  const double ap1 = __ldcg(&SC->apow1), apm1 = __ldcg(&SC->apowm1), ap3 = __ldcg(&SC->apow3);
  const double dx = L.dx, gQ = L.gQ, gQB = L.gQB;
  double n0 = 1.0, n1 = 1.0, n2 = 1.0, n3 = 1.0, n4 = 1.0, d0 = 1.0, d1 = 1.0, d2 = 1.0, d3 = 1.0;
  switch (lane) {
    case 0: n0 = ck; n1 = ap1; n2 = L.inv_dx2; break;
    case 1: n0 = ck; n1 = ap3; break;
    case 2: n0 = ck; n1 = ap1; n2 = L.fo2; n3 = gQ; d0 = dx; break;
    case 3: n0 = -ck; n1 = apm1; d0 = gQ; d1 = d2 = d3 = dx; break;
    case 4: n0 = ck; n1 = ap1; n2 = L.fo2; n3 = gQB; d0 = 2.0; d1 = dx; break;
    case 5: n0 = -2.0; n1 = ck; n2 = apm1; d0 = gQB; d1 = d2 = d3 = dx; break;
    case 6: n0 = gQ; n1 = dx; break;
    case 7: n0 = n1 = L.v; break;
    case 8: n0 = L.lam; break;
    case 9: n0 = 2.0; n1 = L.lam; break;
    case 10: n0 = L.qG; break;
    case 11: n0 = L.qH; break;
    case 12: n0 = L.Qc; n1 = gQ; n2 = dx; break;
    case 13: n0 = ck; n1 = ap1; n2 = L.fo2; n3 = L.Qc; n4 = gQ; d0 = dx; break;
    case 14: n0 = cd; break;
    case 15: n0 = cdA; break;
    case 16: n0 = 0.5; n1 = gQB; n2 = dx; n3 = cdA; break;
    default: break;
  }
  const double num = n0 * n1 * n2 * n3 * n4, den = d0 * d1 * d2 * d3;
  // without a U(1) charge the links' plaquettes do not act (value 3)
  const double v = lane == 3 && gQ == 0.0 ? 0.0 : num / den;
  if (lane < 17) reinterpret_cast<T*>(out)[lane] = (T)v;
}

// Carried along z from the plane below: U(1) plaquette sines xz and yz at n - z, the lower
// staples m(L_xz(n)), m(L_yz(n)), the backward hop W_z^dag(n-z) psi(n-z), and (FULL)
// phi_s(n - z) and vphi's backward hop along z.
template <typename T>
struct Su2Carry {
  T sxz, syz, s, w0, w1;
  V3<T> xz, yz;
  Q4<T> bz;
};

// at: the site's neighbourhood, values of plane p (0 its own, 1 the one above) at offset
// (dx, dy): at.f the doublet, at.u(p, i, ..) link i, at.a(p, i, ..) A_i, at.x(p, k, ..) phi_s and
// vphi's components; at.mom(array) the site's momenta.

// The carries for a plane from the plane below it (p = 0 here) and itself (p = 1).
template <typename T, bool FULL, class At>
__device__ __forceinline__ void su2_carry(const At& at, const Su2Coef<T>& cf, Su2Carry<T>& k) {
  const T ax = at.a(0, 0, 0, 0), ay = at.a(0, 1, 0, 0), az = at.a(0, 2, 0, 0);
  k.sxz = sin_rn(cf.gd * ((ax + at.a(0, 2, 1, 0)) - (at.a(1, 0, 0, 0) + az)));
  k.syz = sin_rn(cf.gd * ((ay + at.a(0, 2, 0, 1)) - (at.a(1, 1, 0, 0) + az)));
  const Q4<T> Ux = at.u(0, 0, 0, 0), Uy = at.u(0, 1, 0, 0), Uz = at.u(0, 2, 0, 0);
  const V3<T> pxz = qvec(qmul(Ux, at.u(0, 2, 1, 0)), qconj(qmul(Uz, at.u(1, 0, 0, 0))));
  const V3<T> pyz = qvec(qmul(Uy, at.u(0, 2, 0, 1)), qconj(qmul(Uz, at.u(1, 1, 0, 0))));
  k.xz = neg(rotc(Uz, pxz));
  k.yz = neg(rotc(Uz, pyz));
  T s, c;
  sincos_t(cf.gd * az, s, c);
  k.bz = udmul(Uz, at.f(0, 0, 0));
  phase(k.bz, c, -s);
  if constexpr (FULL) {
    k.s = at.x(0, 0, 0, 0);
    const T b0 = at.x(0, 1, 0, 0), b1 = at.x(0, 2, 0, 0);
    sincos_t(cf.gdc * az, s, c);
    k.w0 = c * b0 - s * b1;
    k.w1 = c * b1 + s * b0;
  }
}

template <typename T>
struct Su2Site {
  T pn[4], fc[4], pns, pnc0, pnc1, xs0, xc0, xc1;   // kicked momenta, fields
  T s_g, s_pA, s_pB, s_mA, s_mB, s_gs, s_gc;        // sums of the site
  T r2, dd, c2v;                                    // |Phi|^2, |Phi|^2 - v^2, |vphi|^2
};

// The kick of one site; mid() is called once half way, link(i, U_i, A_i, pi_A,i, pi_B,i) with
// the kicked momenta of each direction's link.
template <typename T, int RED, bool FULL, class At, class Mid, class Link>
__device__ __forceinline__ void su2_kick(const At& at, const Su2Coef<T>& cf, Su2Carry<T>& k, Su2Site<T>& o, Mid mid,
                                         Link link) {
  constexpr bool GS = RED == 1 || RED == 2;  // the gauge fields' sums
  const Q4<T> psi = at.f(0, 0, 0);
  const T ax = at.a(0, 0, 0, 0), ay = at.a(0, 1, 0, 0), az = at.a(0, 2, 0, 0);

  // ---- compact U(1) plaquettes: sines at n, at n - x and n - y (direct), at n - z (carried) ----
  const T txy = cf.gd * ((ax + at.a(0, 1, 1, 0)) - (at.a(0, 0, 0, 1) + ay));
  const T txz = cf.gd * ((ax + at.a(0, 2, 1, 0)) - (at.a(1, 0, 0, 0) + az));
  const T tyz = cf.gd * ((ay + at.a(0, 2, 0, 1)) - (at.a(1, 1, 0, 0) + az));
  const T axm = at.a(0, 0, -1, 0);
  // the seven sines in one block (FP32: two at a time, one range check)
  const T ts[7] = {txy, txz, tyz, cf.gd * ((axm + ay) - (at.a(0, 0, -1, 1) + at.a(0, 1, -1, 0))),
                   cf.gd * ((axm + az) - (at.a(1, 0, -1, 0) + at.a(0, 2, -1, 0))),
                   cf.gd * ((at.a(0, 0, 0, -1) + at.a(0, 1, 1, -1)) - (ax + at.a(0, 1, 0, -1))),
                   cf.gd * ((at.a(0, 1, 0, -1) + az) - (at.a(1, 1, 0, -1) + at.a(0, 2, 0, -1)))};
  T sn[7];
  sin_many(ts, sn);
  const T sxy = sn[0], sxz = sn[1], syz = sn[2], sxy_xm = sn[3], sxz_xm = sn[4], sxy_ym = sn[5], syz_ym = sn[6];
  const T Cc[3] = {(sxy - sxy_ym) + (sxz - k.sxz), (sxy_xm - sxy) + (syz - k.syz),
                   (sxz_xm - sxz) + (syz_ym - syz)};
  k.sxz = sxz;
  k.syz = syz;
  T s_mA = T(0);
  if constexpr (GS) {
    const T h1 = sin_t(T(0.5) * txy), h2 = sin_t(T(0.5) * txz), h3 = sin_t(T(0.5) * tyz);
    s_mA = T(2) * (h1 * h1 + h2 * h2 + h3 * h3);
  }

  // ---- SU(2): the three plaquettes at n and the force vectors m(U_i S_i) ----
  const Q4<T> Ux = at.u(0, 0, 0, 0), Uy = at.u(0, 1, 0, 0), Uz = at.u(0, 2, 0, 0);
  V3<T> M[3];
  T s_mB = T(0);
  {
    V3<T> pxy, pxz, pyz, ryx, rzx, mxy, mzy;
    if constexpr (sizeof(T) == 4 && !GS) {
      // the step passes (FP32): products paired lane-wise, the same bits as below
      const Q2 UyUz = q2(Uy, Uz);
      const Q2 A = qmul2(q2(Ux, Ux), q2(at.u(0, 1, 1, 0), at.u(0, 2, 1, 0)));  // Axy, Axz
      const Q2 B = qmul2(UyUz, q2(at.u(0, 0, 0, 1), at.u(1, 0, 0, 0)));             // Bxy, Bxz (unconjugated)
      const Q2 Cp = qmul2(UyUz, q2(at.u(0, 2, 0, 1), at.u(1, 1, 0, 0)));    // Ayz, Byz (unconjugated)
      const P3 pp = qvec2_cb(A, B);
      pxy = lane_of(pp, 0);
      pxz = lane_of(pp, 1);
      pyz = qvec(lane_of(Cp, 0), qconj(lane_of(Cp, 1)));
      // lower staples in the x planes (of U_y, U_z) and in the y planes (of U_x, U_z)
      const Q4<T> uxm = at.u(0, 0, -1, 0), uym = at.u(0, 1, 0, -1);
      const Q2 ix = qmul2(q2(at.u(0, 1, -1, 0), at.u(0, 2, -1, 0)), q2(at.u(0, 0, -1, 1), at.u(1, 0, -1, 0)));
      const P3 rr = qvec2(qmul2_cb(UyUz, ix), q2(uxm, uxm));
      const Q2 iy = qmul2(q2(at.u(0, 0, 0, -1), at.u(0, 2, 0, -1)), q2(at.u(0, 1, 1, -1), at.u(1, 1, 0, -1)));
      const P3 mm = qvec2(qmul2_cb(q2(Ux, Uz), iy), q2(uym, uym));
      ryx = lane_of(rr, 0);
      rzx = lane_of(rr, 1);
      mxy = lane_of(mm, 0);
      mzy = lane_of(mm, 1);
    } else {
      const Q4<T> Axy = qmul(Ux, at.u(0, 1, 1, 0)), Bxy = qconj(qmul(Uy, at.u(0, 0, 0, 1)));
      const Q4<T> Axz = qmul(Ux, at.u(0, 2, 1, 0)), Bxz = qconj(qmul(Uz, at.u(1, 0, 0, 0)));
      const Q4<T> Ayz = qmul(Uy, at.u(0, 2, 0, 1)), Byz = qconj(qmul(Uz, at.u(1, 1, 0, 0)));
      pxy = qvec(Axy, Bxy);
      pxz = qvec(Axz, Bxz);
      pyz = qvec(Ayz, Byz);
      if constexpr (GS) {
        s_mB = (pxy.x * pxy.x + pxy.y * pxy.y + pxy.z * pxy.z) / (T(1) + qsca(Axy, Bxy)) +
               (pxz.x * pxz.x + pxz.y * pxz.y + pxz.z * pxz.z) / (T(1) + qsca(Axz, Bxz)) +
               (pyz.x * pyz.x + pyz.y * pyz.y + pyz.z * pyz.z) / (T(1) + qsca(Ayz, Byz));
      }
      // lower staples of U_y(n), U_z(n) in the x planes, directly
      const Q4<T> uxm = at.u(0, 0, -1, 0);
      ryx = qvec(qmul(Uy, qconj(qmul(at.u(0, 1, -1, 0), at.u(0, 0, -1, 1)))), uxm);
      rzx = qvec(qmul(Uz, qconj(qmul(at.u(0, 2, -1, 0), at.u(1, 0, -1, 0)))), uxm);
      // lower staples of U_x(n), U_z(n) in the y planes, directly
      const Q4<T> uym = at.u(0, 1, 0, -1);
      mxy = qvec(qmul(Ux, qconj(qmul(at.u(0, 0, 0, -1), at.u(0, 1, 1, -1)))), uym);
      mzy = qvec(qmul(Uz, qconj(qmul(at.u(0, 2, 0, -1), at.u(1, 1, 0, -1)))), uym);
    }
    M[0].x = (pxy.x + pxz.x) + (mxy.x + k.xz.x);
    M[0].y = (pxy.y + pxz.y) + (mxy.y + k.xz.y);
    M[0].z = (pxy.z + pxz.z) + (mxy.z + k.xz.z);
    M[1].x = (pyz.x - pxy.x) + (ryx.x + k.yz.x);
    M[1].y = (pyz.y - pxy.y) + (ryx.y + k.yz.y);
    M[1].z = (pyz.z - pxy.z) + (ryx.z + k.yz.z);
    M[2].x = (rzx.x + mzy.x) - (pxz.x + pyz.x);
    M[2].y = (rzx.y + mzy.y) - (pxz.y + pyz.y);
    M[2].z = (rzx.z + mzy.z) - (pxz.z + pyz.z);
    // for plane z + 1: its lower staples of U_x, U_y in the z planes
    k.xz = neg(rotc(Uz, pxz));
    k.yz = neg(rotc(Uz, pyz));
  }
  mid();

  // ---- hops, currents, link kicks and link drifts, direction by direction ----
  // A direction's two hops are added to each other before they join the sum: one rounding at
  // twice the field's size each, and the sum passes through -4 and -2 times the field (hop by
  // hop it was rounded at every multiple from -5 up, and a step's error grew: FP32 64^3, 5 VV2
  // steps, pi 1.3 %, pi_s 1.1 %, vphi's momentum 4 %).
  Q4<T> D;
  T s_g = T(0), s_pA = T(0), s_pB = T(0);
  // FULL: singlet Laplacian and vphi's covariant Laplacian, their gradient sums
  T xs0 = T(0), xc0 = T(0), xc1 = T(0), Ls = T(0), Dv0 = T(0), Dv1 = T(0), s_gs = T(0), s_gc = T(0);
  if constexpr (FULL) {
    xs0 = at.x(0, 0, 0, 0);
    xc0 = at.x(0, 1, 0, 0);
    xc1 = at.x(0, 2, 0, 0);
  }
  const T av[3] = {ax, ay, az};
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    const Q4<T> Ui = i == 0 ? Ux : (i == 1 ? Uy : Uz);
    const Q4<T> fn = i == 0 ? at.f(0, 1, 0) : (i == 1 ? at.f(0, 0, 1) : at.f(1, 0, 0));
    T si, ci;
    sincos_t(cf.gd * av[i], si, ci);
    Q4<T> chi = umul(Ui, fn);
    phase(chi, ci, si);
    // the backward hop W_i^dag(n-i) psi(n-i): across x and y directly; along z the
    // thread's own W_z^dag(n) psi(n) is carried to plane z + 1
    Q4<T> b;
    if (i < 2) {
      T s, c;
      sincos_t(cf.gd * (i == 0 ? axm : at.a(0, 1, 0, -1)), s, c);
      b = i == 0 ? udmul(at.u(0, 0, -1, 0), at.f(0, -1, 0)) : udmul(at.u(0, 1, 0, -1), at.f(0, 0, -1));
      phase(b, c, -s);
    } else {
      b = k.bz;
      k.bz = udmul(Ui, psi);
      phase(k.bz, ci, -si);
    }
    qadd(b, chi);
    if (i == 0) {
      D.w = fmaT(T(-6), psi.w, b.w);
      D.x = fmaT(T(-6), psi.x, b.x);
      D.y = fmaT(T(-6), psi.y, b.y);
      D.z = fmaT(T(-6), psi.z, b.z);
    } else {
      qadd(D, b);
    }
    // psi = (p, q) = (w + i x, y + i z), chi = (c1, c2)
    const T ImA = fmaT(psi.w, chi.x, fmaT(-psi.x, chi.w, fmaT(psi.y, chi.z, -psi.z * chi.y)));  // Im psi^dag chi
    const T Im1 = fmaT(psi.w, chi.z, fmaT(-psi.x, chi.y, fmaT(psi.y, chi.x, -psi.z * chi.w)));  // Im psi^dag s1 chi
    const T Im2 = fmaT(psi.y, chi.w, fmaT(psi.z, chi.x, fmaT(-psi.w, chi.y, -psi.x * chi.z)));  // Im psi^dag s2 chi
    const T Im3 = fmaT(psi.w, chi.x, fmaT(-psi.x, chi.w, fmaT(-psi.y, chi.z, psi.z * chi.y)));  // Im psi^dag s3 chi
    if constexpr (RED > 0) {
      const T e0 = chi.w - psi.w, e1 = chi.x - psi.x, e2 = chi.y - psi.y, e3 = chi.z - psi.z;
      s_g += (e0 * e0 + e1 * e1) + (e2 * e2 + e3 * e3);
    }
    T pnA = at.mom(SPA + i) + (cf.AJA * ImA + cf.ACA * Cc[i]);
    if constexpr (FULL) {
      // singlet: neighbours along i (the one below in z carried)
      const T sfw = i == 0 ? at.x(0, 0, 1, 0) : (i == 1 ? at.x(0, 0, 0, 1) : at.x(1, 0, 0, 0));
      const T sbw = i == 0 ? at.x(0, 0, -1, 0) : (i == 1 ? at.x(0, 0, 0, -1) : k.s);
      Ls = i == 0 ? fmaT(T(-6), xs0, sfw + sbw) : Ls + (sfw + sbw);
      if (i == 2) k.s = xs0;
      // vphi: forward hop Vc_i(n) vphi(n+i), Vc = exp(-i Qc gQ dx A)
      const T y0v = i == 0 ? at.x(0, 1, 1, 0) : (i == 1 ? at.x(0, 1, 0, 1) : at.x(1, 1, 0, 0));
      const T y1v = i == 0 ? at.x(0, 2, 1, 0) : (i == 1 ? at.x(0, 2, 0, 1) : at.x(1, 2, 0, 0));
      T sc2, cc;
      sincos_t(cf.gdc * av[i], sc2, cc);
      const T u0 = cc * y0v + sc2 * y1v, u1 = cc * y1v - sc2 * y0v;
      // backward hop Vc_i^*(n-i) vphi(n-i): across x and y directly; along z the
      // thread's own Vc_z^*(n) vphi(n) is carried to plane z + 1
      T w0, w1;
      if (i < 2) {
        const T b0 = i == 0 ? at.x(0, 1, -1, 0) : at.x(0, 1, 0, -1);
        const T b1 = i == 0 ? at.x(0, 2, -1, 0) : at.x(0, 2, 0, -1);
        T sb, cb;
        sincos_t(cf.gdc * (i == 0 ? axm : at.a(0, 1, 0, -1)), sb, cb);
        w0 = cb * b0 - sb * b1;
        w1 = cb * b1 + sb * b0;
      } else {
        w0 = k.w0;
        w1 = k.w1;
        k.w0 = cc * xc0 - sc2 * xc1;
        k.w1 = cc * xc1 + sc2 * xc0;
      }
      Dv0 = i == 0 ? fmaT(T(-6), xc0, u0 + w0) : Dv0 + (u0 + w0);
      Dv1 = i == 0 ? fmaT(T(-6), xc1, u1 + w1) : Dv1 + (u1 + w1);
      pnA += cf.AJC * (xc0 * u1 - xc1 * u0);
      if constexpr (RED > 0) {
        const T gs = sfw - xs0, g0 = u0 - xc0, g1 = u1 - xc1;
        s_gs += gs * gs;
        s_gc += g0 * g0 + g1 * g1;
      }
    }
    const T Ims[3] = {Im1, Im2, Im3};
    const T Ms[3] = {M[i].x, M[i].y, M[i].z};
    T pnB[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) pnB[a] = at.mom(SPB + 3 * i + a) + (cf.AJB * Ims[a] + cf.AMB * Ms[a]);
    if constexpr (GS) {
      s_pA += pnA * pnA;
      s_pB += pnB[0] * pnB[0] + pnB[1] * pnB[1] + pnB[2] * pnB[2];
    }
    link(i, Ui, av[i], pnA, pnB);
  }
  // ---- doublet kick and drift ----
  const T r2 = T(0.5) * ((psi.w * psi.w + psi.x * psi.x) + (psi.y * psi.y + psi.z * psi.z));
  const T dd = r2 - cf.v2;
  T gp = cf.lam2 * dd;
  T c2v = T(0);  // FULL: |vphi|^2
  if constexpr (FULL) {
    c2v = T(0.5) * (xc0 * xc0 + xc1 * xc1);
    gp += cf.qG * xs0 * xs0 + T(2) * cf.qH * c2v;
  }
  T pn[4];
  const T Dc[4] = {D.w, D.x, D.y, D.z};
  const T fc[4] = {psi.w, psi.x, psi.y, psi.z};
#pragma unroll
  for (int c2 = 0; c2 < 4; ++c2) pn[c2] = at.mom(SP + c2) + (cf.A1 * Dc[c2] - cf.A3 * gp * fc[c2]);
  T pns = T(0), pnc0 = T(0), pnc1 = T(0);
  if constexpr (FULL) {
    pns = at.mom(SPS) + (cf.A1 * Ls - cf.A3 * (T(2) * cf.qG * r2) * xs0);
    pnc0 = at.mom(SPC) + (cf.A1 * Dv0 - cf.A3 * (T(2) * cf.qH * r2) * xc0);
    pnc1 = at.mom(SPC + 1) + (cf.A1 * Dv1 - cf.A3 * (T(2) * cf.qH * r2) * xc1);
  }
#pragma unroll
  for (int c2 = 0; c2 < 4; ++c2) {
    o.pn[c2] = pn[c2];
    o.fc[c2] = fc[c2];
  }
  o.pns = pns;
  o.pnc0 = pnc0;
  o.pnc1 = pnc1;
  o.xs0 = xs0;
  o.xc0 = xc0;
  o.xc1 = xc1;
  o.s_g = s_g;
  o.s_pA = s_pA;
  o.s_pB = s_pB;
  o.s_mA = s_mA;
  o.s_mB = s_mB;
  o.s_gs = s_gs;
  o.s_gc = s_gc;
  o.r2 = r2;
  o.dd = dd;
  o.c2v = c2v;
}

// The site's sums into the accumulators of a pass of measurement level RED.
template <typename T, int RED, bool FULL, int NACC>
__device__ __forceinline__ void su2_sums(const Su2Coef<T>& cf, const Su2Site<T>& o, Acc<T> (&acc)[NACC],
                                         float& nonfinite) {
  if constexpr (RED == 1 || RED == SU2_RED_ALPHA1) {
    T spi = (o.pn[0] * o.pn[0] + o.pn[1] * o.pn[1]) + (o.pn[2] * o.pn[2] + o.pn[3] * o.pn[3]);
    T sg = o.s_g, sv = cf.lam * o.dd * o.dd;
    if constexpr (FULL) {  // the Friedmann kicks take the totals
      spi += o.pns * o.pns + (o.pnc0 * o.pnc0 + o.pnc1 * o.pnc1);
      sg += o.s_gs + o.s_gc;
      sv += cf.qG * o.r2 * o.xs0 * o.xs0 + T(2) * cf.qH * o.r2 * o.c2v;
    }
    acc[0].add(spi);
    if constexpr (RED == 1) {
      acc[1].add(o.s_pA + o.s_pB);
      acc[2].add(sg);
      acc[3].add(o.s_mA);
      acc[4].add(o.s_mB);
      acc[5].add(sv);
    } else {
      acc[1].add(sg);
      acc[2].add(sv);
    }
  } else if constexpr (RED == 2) {
#pragma unroll
    for (int c2 = 0; c2 < 4; ++c2) {
      acc[c2].add(o.pn[c2] * o.pn[c2]);
      acc[10 + c2].add(o.fc[c2]);
      acc[14 + c2].add(o.fc[c2] * o.fc[c2]);
      acc[18 + c2].add(o.pn[c2]);
      if (!isfinite(o.pn[c2])) nonfinite += 1.f;
    }
    acc[4].add(o.s_pA);
    acc[5].add(o.s_pB);
    acc[6].add(o.s_g);
    acc[7].add(o.s_mA);
    acc[8].add(o.s_mB);
    acc[9].add(cf.lam * o.dd * o.dd);
    if (!isfinite(o.s_pA) || !isfinite(o.s_pB)) nonfinite += 1.f;
    if constexpr (FULL) {  // per species: singlet, vphi
      acc[23].add(o.pns * o.pns);
      acc[24].add(o.pnc0 * o.pnc0 + o.pnc1 * o.pnc1);
      acc[25].add(o.s_gs);
      acc[26].add(o.s_gc);
      acc[27].add(cf.qG * o.r2 * o.xs0 * o.xs0);
      acc[28].add(T(2) * cf.qH * o.r2 * o.c2v);
      if (!isfinite(o.pns) || !isfinite(o.pnc0) || !isfinite(o.pnc1)) nonfinite += 1.f;
    }
  }
}

}  // namespace

}  // namespace clg
