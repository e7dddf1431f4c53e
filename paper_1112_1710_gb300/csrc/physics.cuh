// physics.cuh -- point functions of the ideal-MHD patch advance on the GPU,
// templated on the arithmetic type R (double or float).
//
// The scheme (the paper names only "the hyperbolic advance of each grid",
// Sec. 2.3, consuming n_ghost ghost layers per step):
//   primitive PLM reconstruction with a van Leer / minmod / MC limiter,
//   a conservative Hancock half-step predictor, a CT half-step predictor for
//   the face-normal field, the HLLD Riemann solver of Miyoshi & Kusano (2005,
//   JCP 208:315) and Gardiner & Stone (2005, JCP 205:509) edge EMFs.
// Every expression is written in one fixed evaluation order; the FP64
// translation unit is compiled with --fmad=false so that no multiply-add is
// contracted and results are reproducible bit for bit.
#pragma once

#include <cstdint>

#include "int64div.cuh"

namespace mhd {

// Arithmetic of each type.  FP64 divisions, square roots, sign tests and
// scalings by powers of two run on the integer pipe (int64div.cuh): the FP64
// pipe bounds every FP64 stage and the integer pipe idles.  The results have
// the bits of the FP64 instructions.  div2: (a + a) / b.  flip: -x where c.
// degen: relative threshold of the HLLD single-star degeneracy test.  It must
// sit well above the rounding of rho (S - u)(S - S_M) - Bn^2 in the arithmetic
// type: 1e-12 in FP64 (about 4500 ulp), 1e-5 in FP32 (about 80 ulp); an FP32
// test at 1e-12 never fires, and a denominator that is rounding noise then
// divides the transverse velocity and field.
template <typename R> struct Tr;
template <> struct Tr<double> {
  __device__ static __forceinline__ double abs(double x) { return fabs(x); }
  __device__ static __forceinline__ double sqrt_(double x) { return i64::sqrt_rn(x); }
  __device__ static __forceinline__ double div(double a, double b) { return i64::div(a, b); }
  __device__ static __forceinline__ double div2(double a, double b) { return i64::div_scaled<1>(a, b); }
  __device__ static __forceinline__ double half(double x) { return i64::scale<-1>(x); }
  __device__ static __forceinline__ double quarter(double x) { return i64::scale<-2>(x); }
  __device__ static __forceinline__ double times2(double x) { return i64::scale<1>(x); }
  __device__ static __forceinline__ double times4(double x) { return i64::scale<2>(x); }
  __device__ static __forceinline__ bool pos(double x) { return i64::pos(x); }
  __device__ static __forceinline__ bool neg(double x) { return i64::neg(x); }
  __device__ static __forceinline__ bool ge0(double x) { return i64::ge0(x); }
  __device__ static __forceinline__ bool abs_gt(double x, double t) { return i64::abs_gt(x, t); }
  __device__ static __forceinline__ bool less_mag(double a, double b) { return i64::less_mag(a, b); }
  __device__ static __forceinline__ bool nan(double x) { return i64::nan(x); }
  __device__ static __forceinline__ bool special(double x) { return i64::special(x); }
  __device__ static __forceinline__ bool any_special(double a, double b, double c) { return i64::any_special(a, b, c); }
  __device__ static __forceinline__ double undef() { return i64::value(0x7ff8000000000000ull); }
  __device__ static __forceinline__ double degen() { return 1e-12; }
  // |den| <= degen max(a1 a2, b); the exponents settle it almost always
  __device__ static __forceinline__ bool degenerate(double den, double a1, double a2, double b) {
    return !i64::clearly_above(den, a1, a2, b) && fabs(den) <= degen() * ((a1 * a2 > b) ? a1 * a2 : b);
  }
};
template <> struct Tr<float> {
  __device__ static __forceinline__ float abs(float x) { return fabsf(x); }
  __device__ static __forceinline__ float sqrt_(float x) { return sqrtf(x); }
  __device__ static __forceinline__ float rsqrt_(float x) { return rsqrtf(x); }
  __device__ static __forceinline__ float div(float a, float b) { return a / b; }
  __device__ static __forceinline__ float div2(float a, float b) { return (a + a) / b; }
  __device__ static __forceinline__ float half(float x) { return 0.5f * x; }
  __device__ static __forceinline__ float quarter(float x) { return 0.25f * x; }
  __device__ static __forceinline__ float times2(float x) { return 2.0f * x; }
  __device__ static __forceinline__ float times4(float x) { return 4.0f * x; }
  __device__ static __forceinline__ bool pos(float x) { return x > 0.0f; }
  __device__ static __forceinline__ bool neg(float x) { return x < 0.0f; }
  __device__ static __forceinline__ bool less_mag(float a, float b) { return fabsf(a) < fabsf(b); }
  __device__ static __forceinline__ float degen() { return 1e-5f; }
};
template <typename R> __device__ __forceinline__ R flip(R x, bool c) { return c ? -x : x; }

template <typename R> __device__ __forceinline__ R rmin(R a, R b) { return (a < b) ? a : b; }
template <typename R> __device__ __forceinline__ R rmax(R a, R b) { return (a > b) ? a : b; }

// Limited slope of the backward difference a and forward difference b;
// a*b <= 0 gives zero.
template <typename R> __device__ __forceinline__ R limiter(int lim, R a, R b) {
  R ab = a * b;
  if (!Tr<R>::pos(ab)) return R(0);
  if (lim == 1) return Tr<R>::less_mag(a, b) ? a : b;
  if (lim == 2) {
    const R ma = Tr<R>::abs(a), mb = Tr<R>::abs(b);
    const R t = Tr<R>::times2(Tr<R>::less_mag(a, b) ? ma : mb), h = Tr<R>::half(Tr<R>::abs(a + b));
    return flip(Tr<R>::less_mag(t, h) ? t : h, Tr<R>::neg(a));
  }
  return Tr<R>::div2(ab, a + b);
}

// Half the limited slope (what the face values add and subtract): the van
// Leer form is one quotient, a b / (a + b).
template <typename R> __device__ __forceinline__ R half_slope(int lim, R a, R b) {
  if (lim != 0) return Tr<R>::half(limiter(lim, a, b));
  const R ab = a * b;
  return Tr<R>::pos(ab) ? Tr<R>::div(ab, a + b) : R(0);
}

// conserved (rho, M, E, Bc) -> primitive (rho, v, p, Bc)
template <typename R> __device__ __forceinline__ void cons2prim(const R* u, R gm1, R* w) {
  R rho = u[0];
  R ir = Tr<R>::div(R(1), rho);
  R vx = u[1] * ir, vy = u[2] * ir, vz = u[3] * ir;
  R ke = Tr<R>::half(rho) * (vx * vx + vy * vy + vz * vz);
  R me = Tr<R>::half(u[5] * u[5] + u[6] * u[6] + u[7] * u[7]);
  w[0] = rho; w[1] = vx; w[2] = vy; w[3] = vz;
  w[4] = gm1 * (u[4] - ke - me);
  w[5] = u[5]; w[6] = u[6]; w[7] = u[7];
}

template <typename R> __device__ __forceinline__ void prim2cons(const R* w, R igm1, R* u) {
  R rho = w[0];
  R ke = Tr<R>::half(rho) * (w[1] * w[1] + w[2] * w[2] + w[3] * w[3]);
  R me = Tr<R>::half(w[5] * w[5] + w[6] * w[6] + w[7] * w[7]);
  u[0] = rho;
  u[1] = rho * w[1]; u[2] = rho * w[2]; u[3] = rho * w[3];
  u[4] = w[4] * igm1 + ke + me;
  u[5] = w[5]; u[6] = w[6]; u[7] = w[7];
}

// Fast magnetosonic speed: c_f^2 = ((a^2+b^2) + sqrt((a^2+b^2)^2 - 4 a^2 b_n^2))/2.
template <typename R>
__device__ __forceinline__ R fast_speed(R rho, R p, R bn, R bt1, R bt2, R gamma) {
  R ir = Tr<R>::div(R(1), rho);
  R a2 = gamma * p * ir;
  R b2 = (bn * bn + bt1 * bt1 + bt2 * bt2) * ir;
  R bn2 = bn * bn * ir;
  R s = a2 + b2;
  R d = s * s - Tr<R>::times4(a2) * bn2;
  if (Tr<R>::neg(d)) d = R(0);
  return Tr<R>::sqrt_(Tr<R>::half(s + Tr<R>::sqrt_(d)));
}

// Ideal-MHD flux along the normal of a rotated primitive state
// (rho, vn, vt1, vt2, p, -, bt1, bt2) with normal field bn; rotated output,
// f[5] (normal-B flux) is zero.
template <typename R> __device__ __forceinline__ void flux_rot(const R* r, R bn, R igm1, R* f) {
  R rho = r[0], vn = r[1], vt1 = r[2], vt2 = r[3], p = r[4];
  R bt1 = r[6], bt2 = r[7];
  R pm = Tr<R>::half(bn * bn + bt1 * bt1 + bt2 * bt2);
  R pt = p + pm;
  R ke = Tr<R>::half(rho) * (vn * vn + vt1 * vt1 + vt2 * vt2);
  R e = p * igm1 + ke + pm;
  R vb = vn * bn + vt1 * bt1 + vt2 * bt2;
  R mn_ = rho * vn;
  f[0] = mn_;
  f[1] = mn_ * vn + pt - bn * bn;
  f[2] = mn_ * vt1 - bn * bt1;
  f[3] = mn_ * vt2 - bn * bt2;
  f[4] = (e + pt) * vn - bn * vb;
  f[5] = R(0);
  f[6] = bt1 * vn - bn * vt1;
  f[7] = bt2 * vn - bn * vt2;
}

// rotation helpers: axis d -> (n, t1, t2) = (d, d+1, d+2) mod 3
template <typename R> __device__ __forceinline__ void rot_in(int d, const R* w, R* r) {
  const int t1 = (d + 1) % 3, t2 = (d + 2) % 3;
  r[0] = w[0]; r[1] = w[1 + d]; r[2] = w[1 + t1]; r[3] = w[1 + t2];
  r[4] = w[4]; r[5] = w[5 + d]; r[6] = w[5 + t1]; r[7] = w[5 + t2];
}
template <typename R> __device__ __forceinline__ void rot_out(int d, const R* fr, R* f) {
  const int t1 = (d + 1) % 3, t2 = (d + 2) % 3;
  f[0] = fr[0]; f[1 + d] = fr[1]; f[1 + t1] = fr[2]; f[1 + t2] = fr[3];
  f[4] = fr[4]; f[5 + d] = fr[5]; f[5 + t1] = fr[6]; f[5 + t2] = fr[7];
}

// Physical flux along axis d of an xyz primitive state (own B_d as normal).
template <typename R> __device__ __forceinline__ void flux_xyz(int d, const R* w, R igm1, R* f) {
  R r[8], fr[8];
  rot_in(d, w, r);
  flux_rot(r, r[5], igm1, fr);
  rot_out(d, fr, f);
}

// The conserved state u of an xyz primitive state and its physical flux f
// along axis d.  FR: the flux from the conserved values (momenta, energy and
// magnetic pressure computed once for both); else the expressions of
// prim2cons and flux_xyz, whose sums run in different orders.
template <bool FR, typename R> __device__ __forceinline__ void cons_flux(int d, const R* w, R igm1, R* u, R* f) {
  if constexpr (FR) {
    const R mx = w[0] * w[1], my = w[0] * w[2], mz = w[0] * w[3];
    const R me = Tr<R>::half(w[5] * w[5] + w[6] * w[6] + w[7] * w[7]);
    u[0] = w[0];
    u[1] = mx; u[2] = my; u[3] = mz;
    u[4] = w[4] * igm1 + Tr<R>::half(mx * w[1] + my * w[2] + mz * w[3]) + me;
    u[5] = w[5]; u[6] = w[6]; u[7] = w[7];
    const R pt = w[4] + me, vn = w[1 + d], bn = w[5 + d], mn = u[1 + d];
    const R vb = w[1] * w[5] + w[2] * w[6] + w[3] * w[7];
    f[0] = mn;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      f[1 + c] = mn * w[1 + c] - bn * w[5 + c];
      f[5 + c] = c == d ? R(0) : w[5 + c] * vn - bn * w[1 + c];
    }
    f[1 + d] = f[1 + d] + pt;
    f[4] = (u[4] + pt) * vn - bn * vb;
  } else {
    prim2cons(w, igm1, u);
    flux_xyz(d, w, igm1, f);
  }
}

// a / b, or a * ib with ib = 1 / b computed once for several quotients (the
// reciprocal form of the FP32 and the contracted FP64 builds; the parity
// build divides, as the oracle does)
template <bool FR, typename R> __device__ __forceinline__ R qdiv(R a, R b, R ib) {
  if constexpr (FR) return a * ib;
  else return Tr<R>::div(a, b);
}
template <bool FR, typename R> __device__ __forceinline__ R recip(R b) {
  if constexpr (FR) return Tr<R>::div(R(1), b);
  else return R(0);
}

// FP32 HLLD: hlld_side's formulas in the reciprocal form, with every region's
// flux from F* = F + S (U* - U), which the contracted FP64 build replaces by the
// star state's own.  The staged kernels and the fused pass take the same
// bits from it, so where an expression can be contracted in more than one way, and
// the code around it could change the compiler's choice, the multiply-adds are
// written out: the first product fused, the second rounded (dot3: for d = 2 the
// other way round; U* - U of the momenta: by region).  Energies and fluxes
// for the interface's side only, the single-star flux shared with the double-star
// region: 128^3 k_flux 115 -> 113 us, a step 363 -> 359.
__device__ __forceinline__ float dot3(int d, float u, float bn, float v, float by, float w, float bz) {
  return __fmaf_rn(w, bz, d == 2 ? __fmaf_rn(v, by, __fmul_rn(u, bn)) : __fmaf_rn(u, bn, __fmul_rn(v, by)));
}
__device__ __forceinline__ void hlld32(int d, const float* L, const float* Rr, float bn, float gamma, float igm1,
                                       float eps_up, float* f, float* upw) {
  using R = float;
  R rl = L[0], ul = L[1], vl = L[2], wl_ = L[3], pl = L[4], byl = L[6], bzl = L[7];
  R rr = Rr[0], ur = Rr[1], vr = Rr[2], wr_ = Rr[3], pr = Rr[4], byr = Rr[6], bzr = Rr[7];

  R pml = R(0.5) * (bn * bn + byl * byl + bzl * bzl);
  R pmr = R(0.5) * (bn * bn + byr * byr + bzr * bzr);
  R ptl = pl + pml, ptr = pr + pmr;

  R cfl = fast_speed(rl, pl, bn, byl, bzl, gamma);
  R cfr = fast_speed(rr, pr, bn, byr, bzr, gamma);
  R cmax = rmax(cfl, cfr);
  R sl = rmin(ul, ur) - cmax;
  R sr = rmax(ul, ur) + cmax;

  if (sl >= R(0)) {
    flux_rot(L, bn, igm1, f);
    *upw = R(1);
    return;
  }
  if (sr < R(0)) {
    flux_rot(Rr, bn, igm1, f);
    *upw = R(-1);
    return;
  }

  R sdl = sl - ul, sdr = sr - ur;
  R rsl = sdl * rl, rsr = sdr * rr;
  R dd = rsr - rsl;
  const R idd = R(1) / dd;
  R sm = ((rsr * ur - rsl * ul) - (ptr - ptl)) * idd;
  R pts = __fmaf_rn(__fmul_rn(rsl, rsr), ur - ul, __fmaf_rn(rsr, ptl, -__fmul_rn(rsl, ptr))) * idd;
  R tie = eps_up * (sr - sl);
  *upw = (sm > tie) ? R(1) : ((sm < -tie) ? R(-1) : R(0));

  R sml = sl - sm, smr = sr - sm;
  const R isml = R(1) / sml, ismr = R(1) / smr;
  R rls = rsl * isml, rrs = rsr * ismr;
  R bn2 = bn * bn;
  R vls, wls, byls, bzls;
  R denl = rsl * sml - bn2;
  if (Tr<R>::abs(denl) <= Tr<R>::degen() * rmax(rsl * sdl, bn2)) {
    vls = vl; wls = wl_; byls = byl; bzls = bzl;
  } else {
    // numerator of fb = den + rho (S - u)(S_M - u): fb = 1 + rho (S - u) t
    // with t = (S_M - u) / den, exactly 1 where S_M = u
    const R t = (sm - ul) * (R(1) / denl);
    const R fv = bn * t, fb = R(1) + rsl * t;
    vls = vl - byl * fv; wls = wl_ - bzl * fv;
    byls = byl * fb; bzls = bzl * fb;
  }
  R vrs, wrs, byrs, bzrs;
  R denr = rsr * smr - bn2;
  if (Tr<R>::abs(denr) <= Tr<R>::degen() * rmax(rsr * sdr, bn2)) {
    vrs = vr; wrs = wr_; byrs = byr; bzrs = bzr;
  } else {
    // numerator of fb = den + rho (S - u)(S_M - u): fb = 1 + rho (S - u) t
    // with t = (S_M - u) / den, exactly 1 where S_M = u
    const R t = (sm - ur) * (R(1) / denr);
    const R fv = bn * t, fb = R(1) + rsr * t;
    vrs = vr - byr * fv; wrs = wr_ - bzr * fv;
    byrs = byr * fb; bzrs = bzr * fb;
  }

  // the interface lies in the half of the fan on S_M's side (see hlld_side)
  const bool left = (sm >= R(0));
  const R rho = left ? rl : rr, u = left ? ul : ur, v = left ? vl : vr, w = left ? wl_ : wr_;
  const R p = left ? pl : pr, by = left ? byl : byr, bz = left ? bzl : bzr;
  const R pm = left ? pml : pmr, pt = left ? ptl : ptr;
  const R S = left ? sl : sr, sd = left ? sdl : sdr;
  const R rs = left ? rls : rrs, vs = left ? vls : vrs, ws = left ? wls : wrs;
  const R bys = left ? byls : byrs, bzs = left ? bzls : bzrs;
  const R e = __fmaf_rn(p, igm1, __fmul_rn(R(0.5) * rho, dot3(0, u, u, v, v, w, w))) + pm;
  const R vb = dot3(0, u, bn, v, by, w, bz);
  const R vbs = dot3(d, sm, bn, vs, bys, ws, bzs);
  const R es = __fmul_rn(__fmaf_rn(bn, vb - vbs, __fmaf_rn(pts, sm, __fmaf_rn(sd, e, -__fmul_rn(pt, u)))),
                         left ? isml : ismr);

  const R isl = Tr<R>::rsqrt_(rls), isr = Tr<R>::rsqrt_(rrs);
  const R sqrl = rls * isl, sqrr = rrs * isr;
  const R ab = Tr<R>::abs(bn);
  const R Ss = __fmaf_rn(left ? -ab : ab, left ? isl : isr, sm);

  // single-star region: F* = F_outer + S_outer (U* - U_outer)
  const R mn = rho * u;
  const R fo[8] = {mn, mn * u + pt - bn * bn, mn * v - bn * by, mn * w - bn * bz, (e + pt) * u - bn * vb, R(0),
                   by * u - bn * v, bz * u - bn * w};
  const R u0[8] = {rho, mn, __fmul_rn(rho, v), __fmul_rn(rho, w), e, bn, by, bz};
  const R us[8] = {rs, rs * sm, rs * vs, rs * ws, es, bn, bys, bzs};
#pragma unroll
  for (int q = 0; q < 8; ++q) f[q] = __fmaf_rn(S, us[q] - u0[q], fo[q]);
  if (left ? Ss >= R(0) : Ss < R(0)) {
    f[1] = __fmaf_rn(S, __fmaf_rn(rs, sm, -u0[1]), fo[1]);
    f[2] = __fmaf_rn(S, __fmaf_rn(rs, vs, -u0[2]), fo[2]);
    f[3] = __fmaf_rn(S, __fmaf_rn(rs, ws, -u0[3]), fo[3]);
    return;
  }
  f[1] = __fmaf_rn(S, __fmaf_rn(-rho, u, us[1]), fo[1]);
  f[2] = __fmaf_rn(S, __fmaf_rn(-rho, v, us[2]), fo[2]);
  f[3] = __fmaf_rn(S, __fmaf_rn(-rho, w, us[3]), fo[3]);

  // double-star region: F** = F* + S* (U** - U*)
  R sgn = (bn >= R(0)) ? R(1) : R(-1);
  R ssum = sqrl + sqrr;
  const R iss = R(1) / ssum;
  R vss = ((sqrl * vls + sqrr * vrs) + sgn * (byrs - byls)) * iss;
  R wss = ((sqrl * wls + sqrr * wrs) + sgn * (bzrs - bzls)) * iss;
  R byss = ((sqrl * byrs + sqrr * byls) + sgn * (sqrl * sqrr) * (vrs - vls)) * iss;
  R bzss = ((sqrl * bzrs + sqrr * bzls) + sgn * (sqrl * sqrr) * (wrs - wls)) * iss;
  R vbss = dot3(d, sm, bn, vss, byss, wss, bzss);
  const R ess = __fmaf_rn(__fmul_rn(left ? -sqrl : sqrr, vbs - vbss), sgn, es);
  const R uss[8] = {rs, rs * sm, rs * vss, rs * wss, ess, bn, byss, bzss};
#pragma unroll
  for (int q = 0; q < 8; ++q) f[q] = f[q] + Ss * (uss[q] - us[q]);
}

// HLLD flux (Miyoshi & Kusano 2005) between rotated primitive states L (lower
// side) and R_ (upper side) with interface normal field bn.  Wave speeds
// S_L = min(u_L,u_R) - max(cf), S_R = max(u_L,u_R) + max(cf); S_M, p_T* from
// MK05 eqs. (38), (41); star states eqs. (43)-(48) with a degenerate branch
// (|rho(S-u)(S-S_M) - Bn^2| <= degen max(rho(S-u)^2, Bn^2), degen 1e-12 in
// FP64 and 1e-5 in FP32, keeps the outer
// transverse v, B); Alfven speeds S* = S_M -/+ |Bn|/sqrt(rho*); double-star
// states eqs. (59)-(63); left-closed region selection.  f gets the rotated
// flux (f[5], the normal-B component, is 0); *upw, where up is set (the
// upwinded EMF average), the upwind side of the contact (+1, -1, or 0 when
// |S_M| <= eps_up (S_R - S_L)), else 0.
// The interface lies in the half of the fan on S_M's side (S_M >= 0: left):
// a star region left of the contact needs S*_L <= S_M, one right of it
// S_M <= S*_R.  So the energies, the Alfven speed and the flux are computed
// for that side alone, from operands selected first, with the expressions
// (and in the parity build the bits) they would have on either side; only the
// transverse star states, which the double-star states mix, are computed for
// both.
// FR: quotients with a common denominator multiply by its reciprocal (8
// divisions per face instead of 16), and the single-star field factor
// is written as 1 + rho (S - u)(S_M - u)/den, which is exactly 1 where
// S_M = u (a plain reciprocal would turn x/x into x (1/x), off by an ulp,
// and give a 2D problem a z-field of rounding noise).
template <typename R, bool FR = false>
__device__ __forceinline__ void hlld_side(const R* L, const R* Rr, R bn, R gamma, R igm1, R eps_up, bool up,
                                     R* f, R* upw) {
  using T = Tr<R>;
  R rl = L[0], ul = L[1], vl = L[2], wl_ = L[3], pl = L[4], byl = L[6], bzl = L[7];
  R rr = Rr[0], ur = Rr[1], vr = Rr[2], wr_ = Rr[3], pr = Rr[4], byr = Rr[6], bzr = Rr[7];

  R cfl = fast_speed(rl, pl, bn, byl, bzl, gamma);
  R cfr = fast_speed(rr, pr, bn, byr, bzr, gamma);
  // max(cfl, cfr), min(ul, ur) and max(ul, ur), as a > b ? a : b and a < b ? a : b
  // (a NaN in a gives b)
  const bool ulo = ul < ur;
  R cmax = T::less_mag(cfr, cfl) ? cfl : cfr, umax = ulo ? ur : ul;
  if (T::any_special(cfl, ul, ur)) {
    if (T::nan(cfl)) cmax = cfr;
    if (T::nan(ul) || T::nan(ur)) umax = ur;
  }
  R sl = (ulo ? ul : ur) - cmax;
  R sr = umax + cmax;

  if (T::ge0(sl)) {
    flux_rot(L, bn, igm1, f);
    *upw = R(1);
    return;
  }
  if (T::neg(sr)) {
    flux_rot(Rr, bn, igm1, f);
    *upw = R(-1);
    return;
  }

  R pml = T::half(bn * bn + byl * byl + bzl * bzl);
  R pmr = T::half(bn * bn + byr * byr + bzr * bzr);
  R ptl = pl + pml, ptr = pr + pmr;
  R sdl = sl - ul, sdr = sr - ur;
  R rsl = sdl * rl, rsr = sdr * rr;
  R dd = rsr - rsl;
  const R idd = recip<FR>(dd);
  R sm = qdiv<FR>((rsr * ur - rsl * ul) - (ptr - ptl), dd, idd);
  *upw = R(0);
  if (up && T::abs_gt(sm, eps_up * (sr - sl))) *upw = T::neg(sm) ? R(-1) : R(1);

  R sml = sl - sm, smr = sr - sm;
  const R isml = recip<FR>(sml), ismr = recip<FR>(smr);
  R rls = qdiv<FR>(rsl, sml, isml), rrs = qdiv<FR>(rsr, smr, ismr);
  R bn2 = bn * bn;
  R vls, wls, byls, bzls;
  R denl = rsl * sml - bn2;
  const bool dgl = T::degenerate(denl, rsl, sdl, bn2);
  if (dgl) {
    vls = vl; wls = wl_; byls = byl; bzls = bzl;
  } else {
    R fv, fb;
    if constexpr (FR) {
      // numerator of fb = den + rho (S - u)(S_M - u): fb = 1 + rho (S - u) t
      // with t = (S_M - u) / den, exactly 1 where S_M = u
      const R t = (sm - ul) * recip<FR>(denl);
      fv = bn * t;
      fb = R(1) + rsl * t;
    } else {
      fv = T::div(bn * (sm - ul), denl);
      fb = T::div(rsl * sdl - bn2, denl);
    }
    vls = vl - byl * fv; wls = wl_ - bzl * fv;
    byls = byl * fb; bzls = bzl * fb;
  }
  R vrs, wrs, byrs, bzrs;
  R denr = rsr * smr - bn2;
  const bool dgr = T::degenerate(denr, rsr, sdr, bn2);
  if (dgr) {
    vrs = vr; wrs = wr_; byrs = byr; bzrs = bzr;
  } else {
    R fv, fb;
    if constexpr (FR) {
      const R t = (sm - ur) * recip<FR>(denr);
      fv = bn * t;
      fb = R(1) + rsr * t;
    } else {
      fv = T::div(bn * (sm - ur), denr);
      fb = T::div(rsr * sdr - bn2, denr);
    }
    vrs = vr - byr * fv; wrs = wr_ - bzr * fv;
    byrs = byr * fb; bzrs = bzr * fb;
  }

  // the side of the contact the interface lies on
  const bool left = T::ge0(sm);
  const R rho = left ? rl : rr, u = left ? ul : ur, v = left ? vl : vr, w = left ? wl_ : wr_;
  const R p = left ? pl : pr, by = left ? byl : byr, bz = left ? bzl : bzr;
  const R pm = left ? pml : pmr, pt = left ? ptl : ptr;
  // p_T*: MK05 eq. (41), or FR eq. (23) on the selected side, p_T + rho (S - u)
  // (S_M - u), which is exactly p_T in a uniform state
  R pts;
  if constexpr (FR) pts = pt + (left ? rsl : rsr) * (sm - u);
  else pts = T::div((rsr * ptl - rsl * ptr) + rsl * rsr * (ur - ul), dd);
  const R S = left ? sl : sr, sd = left ? sdl : sdr, sS = left ? sml : smr, isS = left ? isml : ismr;
  const R rs = left ? rls : rrs, vs = left ? vls : vrs, ws = left ? wls : wrs;
  const R bys = left ? byls : byrs, bzs = left ? bzls : bzrs;
  const R e = p * igm1 + T::half(rho) * (u * u + v * v + w * w) + pm;
  const R vb = u * bn + v * by + w * bz;
  const R vbs = sm * bn + vs * bys + ws * bzs;
  const R es = qdiv<FR>(((sd * e - pt * u) + pts * sm) + bn * (vb - vbs), sS, isS);

  const R sqrl = T::sqrt_(rls), sqrr = T::sqrt_(rrs);
  const R ab = T::div(T::abs(bn), left ? sqrl : sqrr);
  const R Ss = left ? sm - ab : sm + ab;

  const R mxs = rs * sm;
  const bool bneg = !T::ge0(bn);
  const bool single = left ? T::ge0(Ss) : T::neg(Ss);
  if constexpr (FR) {
    // F* = F + S (U* - U) and F** = F* + S* (U** - U*) are the physical fluxes
    // of the star states (pressure p_T*, normal velocity S_M), the jumps being
    // the Rankine-Hugoniot conditions that define those states: one flux of
    // the state the interface lies in, 14 operations instead of 42.  A
    // degenerate outer state kept its transverse field, whose induction flux
    // then moves with the outer velocity.
    R vF = vs, wF = ws, byF = bys, bzF = bzs, eF = es, vbF = vbs;
    if (!single) {
      // the double-star state as changes from the side's star state, which
      // vanish exactly in a uniform state: dv = (sqrt(rho*) of the other side
      // times the velocity jump, plus the field jump) / sum, dB = sqrt(rho*) dv
      const R iss = recip<FR>(sqrl + sqrr), so = left ? sqrr : sqrl, ss = left ? sqrl : sqrr;
      const R dv = (flip(so * (vrs - vls), !left) + flip(byrs - byls, bneg)) * iss;
      const R dw = (flip(so * (wrs - wls), !left) + flip(bzrs - bzls, bneg)) * iss;
      vF = vs + dv;
      wF = ws + dw;
      byF = bys + flip(ss * dv, left == bneg);
      bzF = bzs + flip(ss * dw, left == bneg);
      vbF = sm * bn + vF * byF + wF * bzF;
      eF = es + flip(ss * (vbs - vbF), left != bneg);
    }
    f[0] = mxs;
    f[1] = mxs * sm + (pts - bn2);
    f[2] = mxs * vF - bn * byF;
    f[3] = mxs * wF - bn * bzF;
    f[4] = (eF + pts) * sm - bn * vbF;
    f[5] = R(0);
    f[6] = byF * sm - bn * vF;
    f[7] = bzF * sm - bn * wF;
    if (left ? dgl : dgr) {
      f[6] = f[6] + bys * (u - sm);
      f[7] = f[7] + bzs * (u - sm);
    }
    if (!single && T::special(Ss)) {  // (a state with rho <= 0)
#pragma unroll
      for (int q = 0; q < 8; ++q) f[q] = T::undef();
    }
    return;
  }
  // outer flux and conserved states; single-star region: F* = F + S (U* - U)
  const R mx = rho * u, my = rho * v, mz = rho * w;
  const R mys = rs * vs, mzs = rs * ws;
  f[0] = mx + S * (rs - rho);
  f[1] = (mx * u + pt - bn2) + S * (mxs - mx);
  f[2] = (mx * v - bn * by) + S * (mys - my);
  f[3] = (mx * w - bn * bz) + S * (mzs - mz);
  f[4] = ((e + pt) * u - bn * vb) + S * (es - e);
  f[5] = R(0);
  f[6] = (by * u - bn * v) + S * (bys - by);
  f[7] = (bz * u - bn * w) + S * (bzs - bz);
  if (single) return;

  // double-star region: F** = F* + S* (U** - U*); rho and S_M are U*'s, whose
  // zero jumps still carry what is not finite
  if (T::any_special(Ss, rs, mxs)) {
    if (T::special(Ss) || T::special(rs)) f[0] = T::undef();
    if (T::special(Ss) || T::special(mxs)) f[1] = T::undef();
  }
  R ssum = sqrl + sqrr;
  R vss = T::div((sqrl * vls + sqrr * vrs) + flip(byrs - byls, bneg), ssum);
  R wss = T::div((sqrl * wls + sqrr * wrs) + flip(bzrs - bzls, bneg), ssum);
  const R sq2 = flip(sqrl * sqrr, bneg);
  R byss = T::div((sqrl * byrs + sqrr * byls) + sq2 * (vrs - vls), ssum);
  R bzss = T::div((sqrl * bzrs + sqrr * bzls) + sq2 * (wrs - wls), ssum);
  R vbss = sm * bn + vss * byss + wss * bzss;
  const R ess = es + flip((left ? sqrl : sqrr) * (vbs - vbss), left != bneg);
  f[2] = f[2] + Ss * (rs * vss - mys);
  f[3] = f[3] + Ss * (rs * wss - mzs);
  f[4] = f[4] + Ss * (ess - es);
  f[6] = f[6] + Ss * (byss - bys);
  f[7] = f[7] + Ss * (bzss - bzs);
}

// HLLD flux of an axis-d face.
template <typename R, bool FR = false>
__device__ __forceinline__ void hlld(int d, const R* L, const R* Rr, R bn, R gamma, R igm1, R eps_up, bool up, R* f,
                                     R* upw) {
  if constexpr (sizeof(R) == 4) hlld32(d, L, Rr, bn, gamma, igm1, eps_up, f, upw);
  else hlld_side<R, FR>(L, Rr, bn, gamma, igm1, eps_up, up, f, upw);
}

}  // namespace mhd
