// The central screen of the fast policy (1D): which interface fluxes are the plain sixth-order
// central flux of the physical flux f, proven in FP32 without any FP64 projection.
//
// A restricted reconstruction (Eq. (be_res)) is linear: with theta = 0 it is the central scheme C
// (Eq. (fh_6)), with theta = 1 it is C -/+ Delta^5 q / 60 (Eq. (fh_5)) on the + / - side.  C is the
// same on both sides, so with the splitting v+- = (l.f +- alpha l.u) / 2 (Eq. (flux_split_lf)) an
// interface whose six reconstructions are all restricted with theta = 0 has
//     F_s = C v+ + C v- = l_s . C f,   h = R F = R L C f = C f :
// alpha and the eigenvectors drop out, and three components of C f replace Roe's average, the
// projections, the reconstructions and the back-projection (about 300 FP64 instructions per
// interface).  The choice of theta does not matter either where |Delta^5 v| / 60 is below the
// rounding of the projected flux itself.
//
// The FP64 pipe issues one warp instruction per 64 clocks, an FP32 or integer instruction takes
// one, so the decisions are screened in FP32 from FP32 pairs (47 bits) of the FP64 cell
// differences of f and u; every quantity carries an error bound, and an interface for which any of
// the six reconstructions is not proven takes the FP64 path (projections, theta, weights).
// Every operation is an explicit rounded intrinsic: all kernels take the same decisions.
//
// Measured (1D, GB300): FP64 thread instructions per cell and stage 364 -> about 60 where the data are
// smooth; a run of 999,983 cells 18.0 -> 4.5 ms for 8 steps, a batch of 12.0 M cells in problems of
// 256 to 65536 cells 103.6 -> 29.0 ms for 4 steps, 600 problems of 64 to 1024 cells (a third of
// the interfaces listed) 14.3 -> 12.6 ms for 20 steps.  Error of L against extended precision:
// as before or smaller (smooth data 5.5e-14 -> 1.5e-14 rms at 5000 cells; C f rounds less).
#pragma once

#include "wt_device.cuh"

namespace wt {

__device__ __forceinline__ float fadd(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float fsub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float fmul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float ffma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
// hardware reciprocal and reciprocal square root (within 2^-22 relative)
__device__ __forceinline__ float frcp_hw(float x) {
  float r;
  asm("rcp.approx.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ float frsqrt_hw(float x) {
  float r;
  asm("rsqrt.approx.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

// A double as the float of its leading 24 bits, truncated: within 2^-23 |x|; magnitudes below
// 2^-126 come out below 2^-125, those of 2^128 and above (and NaN) as inf or NaN.  Integer
// pipe only (a conversion instruction costs as much as an FP64 operation).
__device__ __forceinline__ float f32_trunc(double x) {
  const int hi = __double2hiint(x), lo = __double2loint(x);
  const int m = min(max(hi & 0x7fffffff, 0x38000000), 0x47f00000) - 0x38000000;
  return __int_as_float((int)__funnelshift_l((unsigned)lo, (unsigned)m, 3) | (hi & 0x80000000));
}

// x as h + l: h the truncation above, l the remaining 29 bits truncated to 23, so |x - h - l| <
// 2^-46 |x| (below 2^-100 the tail may be lost: within 2^-125)
__device__ __forceinline__ float2 f32_pair(double x) {
  const int hi = __double2hiint(x), lo = __double2loint(x);
  const int sg = hi & 0x80000000;
  const int m = min(max(hi & 0x7fffffff, 0x38000000), 0x47f00000) - 0x38000000;
  const int t = (int)__funnelshift_l((unsigned)lo, (unsigned)m, 3);
  const int base = max((t & 0x7f800000) - (23 << 23), 0);
  const float tail = fsub(__int_as_float(base | (int)(((unsigned)lo << 3) >> 9)), __int_as_float(base));
  return make_float2(__int_as_float(t | sg), __int_as_float(__float_as_int(tail) ^ sg));
}

// the same with a nonzero high part for every x other than zero
__device__ __forceinline__ float2 f32_pair_nz(double x) {
  float2 p = f32_pair(x);
  const unsigned any = ((unsigned)__double2hiint(x) << 1) | (unsigned)__double2loint(x);
  if (p.x == 0.0f && any != 0u) p.x = 0x1p-126f;
  return p;
}

// whether eps and alpha_R (as floats) are in the screen's range: the thresholds of Eq. (be_res) are then
// normal floats
__device__ __forceinline__ bool screen_constants(float eps, float aR) { return fmul(aR, eps) > 1e-30f && eps > 0x1p-120f; }

// a - b of FP32 pairs: the high parts' difference and its exact rounding error, plus the low
// parts' (not renormalised; the low part's own roundings stay below 2^-46 of the largest input)
__device__ __forceinline__ float2 pair_sub(float2 a, float2 b) {
  const float s = fsub(a.x, b.x);
  const float bb = fsub(s, a.x);
  const float e = fsub(fsub(a.x, fsub(s, bb)), fadd(b.x, bb));
  return make_float2(s, fadd(fsub(a.y, b.y), e));
}

// From the five cell differences d_0..d_4 of one component over a stencil: the centre third
// difference (x), the two fourth differences (y, z) and the fifth (w), each within 2^-23 of itself
// plus 2^-41 max |d_k| (1-norm 16 of the fifth difference's coefficients, 2^-46 per input)
__device__ __forceinline__ float4 high_differences(const float2* d) {
  const float2 s0 = pair_sub(d[1], d[0]), s1 = pair_sub(d[2], d[1]), s2 = pair_sub(d[3], d[2]),
               s3 = pair_sub(d[4], d[3]);
  const float2 t0 = pair_sub(s1, s0), t1 = pair_sub(s2, s1), t2 = pair_sub(s3, s2);
  const float2 v0 = pair_sub(t1, t0), v1 = pair_sub(t2, t1);
  return make_float4(fadd(t1.x, t1.y), fadd(v0.x, v0.y), fadd(v1.x, v1.y),
                     fadd(fsub(v1.x, v0.x), fsub(v1.y, v0.y)));
}

// Roe's average in FP32 and the error bounds of the projections it enters.
//   u   within E = 2^-22 U + 2^-20 |ua - ub| of Roe's mean velocity, U = max(|ua|, |ub|)
//   b1 = (gamma - 1) / c^2 and ic = 1 / c within `rel` of theirs
//   q   E / U + 2.25 * 2^-23, rounded up: the projection's input (truncation, 2^-23) and rounding
//       errors per unit of its majorants (proj_bound)
//   thr 60 * 2^-53 rho (|u| + c): a side's |Delta^5 v| below this moves F_s by less than 2^-53
//       rho (|u| + c), the rounding of the products of l.f alone
//   ok  false where the bounds do not hold (vacuum, c^2 lost to cancellation, out of range)
struct Roe32 {
  float u, U, ic, b1, q, rel, thr;
  bool ok;
};
__device__ __forceinline__ Roe32 roe32(double ra_, double ua_, double Ha_, double rb_, double ub_, double Hb_,
                                       float gm1) {
  Roe32 r;
  const float ra = f32_trunc(ra_), rb = f32_trunc(rb_), ua = f32_trunc(ua_), ub = f32_trunc(ub_);
  const float Ha = f32_trunc(Ha_), Hb = f32_trunc(Hb_);
  const float sa = fmul(ra, frsqrt_hw(ra)), sb = fmul(rb, frsqrt_hw(rb));
  // the weights' difference: the mean is symmetric in the two cells bit for bit
  const float hw = fmul(fmul(0.5f, fsub(sa, sb)), frcp_hw(fadd(sa, sb)));
  const float du = fsub(ua, ub);
  r.u = ffma(hw, du, fmul(0.5f, fadd(ua, ub)));
  const float H = ffma(hw, fsub(Ha, Hb), fmul(0.5f, fadd(Ha, Hb)));
  r.U = fmaxf(fabsf(ua), fabsf(ub));
  const float he = ffma(fmul(-0.5f, r.u), r.u, H);  // H - u^2 / 2 = c^2 / (gamma - 1)
  const float big = ffma(r.U, r.U, fmaxf(fabsf(Ha), fabsf(Hb)));
  const float c2 = fmul(gm1, he);
  r.ic = frsqrt_hw(c2);
  r.b1 = fmul(gm1, fmul(r.ic, r.ic));
  r.rel = ffma(0x1p-19f, fmul(big, r.b1), 0x1p-20f);
  r.q = ffma(0x1p-20f, fmul(fabsf(du), frcp_hw(fadd(r.U, 1e-30f))), 0x1.8p-21f);
  const float speed = ffma(c2, r.ic, fabsf(r.u));
  r.thr = fmul(fmul(60.0f * 0x1p-53f, fminf(ra, rb)), speed);
  r.ok = ra > 0x1p-60f && rb > 0x1p-60f && ra < 0x1p60f && rb < 0x1p60f && fmul(he, 32.0f) >= big && big < 0x1p60f &&
         big > 0x1p-60f;
  return r;
}

// The left eigenvectors applied to x: with w1 = x1 - u x0 and w2 = x2 - u x1 + u^2 x0 / 2,
//   2 l_0.x = b1 w2 - w1 / c,  l_1.x = x0 - b1 w2,  2 l_2.x = b1 w2 + w1 / c.
// Returns (j, k) = (w1 / c, b1 w2).  The form keeps the cancellation in a wave of another field
// in w1, w2, whose errors are below q N1 and q N2 (N1 = |x1| + U |x0|, N2 = |x2| + U N1: d w2 /
// d u = -w1), while the errors of b1 and 1 / c are relative to k and j.
__device__ __forceinline__ float2 project32(const Roe32& r, float x0, float x1, float x2) {
  const float w1 = ffma(-r.u, x0, x1);
  const float w2 = ffma(fmul(-0.5f, r.u), fadd(x1, w1), x2);
  return make_float2(fmul(r.ic, w1), fmul(r.b1, w2));
}
// (N1 / c, b1 N2)
__device__ __forceinline__ float2 proj_bound(const Roe32& r, float x0, float x1, float x2) {
  const float n1 = ffma(r.U, fabsf(x0), fabsf(x1));
  return make_float2(fmul(r.ic, n1), fmul(r.b1, ffma(r.U, n1, fabsf(x2))));
}
// Field s's projection from (j, k) and x0: 2 l_0.x, l_1.x, 2 l_2.x
__device__ __forceinline__ float field32(int s, float2 jk, float x0) {
  return s == 1 ? fsub(x0, jk.y) : fadd(jk.y, s == 0 ? -jk.x : jk.x);
}
// Its error, from the bounds nb of the vector, |j|, |k| and |x0|
__device__ __forceinline__ float field_err(int s, const Roe32& r, float2 nb, float aj, float ak, float ax0) {
  return s == 1 ? ffma(r.rel, ak, ffma(r.q, nb.y, fmul(0x1p-22f, ax0)))
                : ffma(r.rel, fadd(aj, ak), fmul(r.q, fadd(nb.x, nb.y)));
}

// The least value of the largest cell difference of a component in the error bounds.  The pairs lose what
// lies below 2^-125, 2^-121 in a fifth difference, whatever the differences' own size: with this
// floor the pairs' error 2^-40 max |d| covers it too.  (Cold or thin gas, rho c^3 below 2^-74:
// there the loss is above 60 * 2^-53 rho c after the product with b1 = (gamma - 1) / c^2.)
constexpr float kLow32 = 0x1p-80f;

// The projections of one array (f or u) over an interface's stencil, before the field is chosen:
// d[c] the high parts of component c's five differences, h[c] its high differences.  [0..4]
// the cell differences, [5..8] third, fourth, fourth, fifth.
struct Proj32 {
  float2 jk[9];
  float x0[9];
  float2 nb[5];   // proj_bound of the largest |d| ([0]) and of [5..8]
  float jm, km, xm;  // max |j|, |k|, |x0| over the cell differences
};
__device__ __forceinline__ void project_stencil(const Roe32& r, const float (*d)[5], const float4* h, Proj32& p) {
  p.jm = p.km = 0.0f;
  p.xm = kLow32;
  float m1 = kLow32, m2 = kLow32;
#pragma unroll
  for (int k = 0; k < 5; ++k) {
    p.jk[k] = project32(r, d[0][k], d[1][k], d[2][k]);
    p.x0[k] = d[0][k];
    p.jm = fmaxf(p.jm, fabsf(p.jk[k].x));
    p.km = fmaxf(p.km, fabsf(p.jk[k].y));
    p.xm = fmaxf(p.xm, fabsf(d[0][k]));
    m1 = fmaxf(m1, fabsf(d[1][k]));
    m2 = fmaxf(m2, fabsf(d[2][k]));
  }
  p.nb[0] = proj_bound(r, p.xm, m1, m2);
  const float x[4][3] = {{h[0].x, h[1].x, h[2].x}, {h[0].y, h[1].y, h[2].y}, {h[0].z, h[1].z, h[2].z},
                         {h[0].w, h[1].w, h[2].w}};
#pragma unroll
  for (int v = 0; v < 4; ++v) {
    p.jk[5 + v] = project32(r, x[v][0], x[v][1], x[v][2]);
    p.x0[5 + v] = x[v][0];
    p.nb[1 + v] = proj_bound(r, x[v][0], x[v][1], x[v][2]);
  }
}
// Field s's projections and their error bounds
__device__ __forceinline__ void take_field(int s, const Roe32& r, const Proj32& p, float* a, float* ea) {
#pragma unroll
  for (int k = 0; k < 9; ++k) a[k] = field32(s, p.jk[k], p.x0[k]);
  ea[0] = field_err(s, r, p.nb[0], p.jm, p.km, p.xm);
  // the pairs' own error, 2^-41 of the largest cell differences
  const float pe = fmul(0x1p-40f, s == 1 ? fadd(p.xm, p.nb[0].y) : fadd(p.nb[0].x, p.nb[0].y));
#pragma unroll
  for (int v = 0; v < 4; ++v)
    ea[1 + v] = fadd(pe, field_err(s, r, p.nb[1 + v], fabsf(p.jk[5 + v].x), fabsf(p.jk[5 + v].y), fabsf(p.x0[5 + v])));
}

// One field of one interface.  a, b: the projections of the differences of f and of u: [0..4] the
// cell differences, [5] third, [6], [7] fourth, [8] fifth; ea, eb: their error bounds ([0] for all
// five cell differences, [1..4] for [5..8]).  al: alpha_s.  The sides' stencil differences are (a
// +- al b) times kappa (1/4 for the acoustic fields, 1/2 for the others); epsk = eps / kappa^2,
// thrk = thr / kappa.  Returns 0 if some decision is left to FP64; else 1, plus 2 where the +
// side has theta = 1, plus 4 where the - side has (0 where theta does not matter).
//   beta_k: with each difference within eta and S their maximum, the indicators move by at most 54
//   S eta + 27 eta^2 (the worst: beta_3, forms of 1-norm 8 and 3), and their FP32 roundings by
//   2^-16 S^2; the test is that of Eq. (be_res), max beta <= alpha_R (eps + min beta), with the
//   indicators moved against it.
//   theta = 0: tau6's upper bound is below tau5's lower bound (Eqs. (tau_5), (tau_6), (tau_we6));
//   theta = 1: the other way round.  TH1 = false: only theta = 0 is proven (else 0).  The 2D sweeps take
//   both verdicts (with the reduction of phase E's maxima by warps: 2048 x 2048 vortices 18.8 ->
//   17.5 ms, 120 x 360 Rayleigh-Taylor 13.8 -> 11.6 ms); in the 1D Euler tiles the second one's
//   registers cost more than it saves (batch of 1024 problems 29.0 -> 30.0 .. 32.9 ms).
template <bool TH1 = true>
__device__ __forceinline__ int prove_field(const float* a, const float* b, const float* ea, const float* eb, float al,
                                            float epsk, float alpha_R, float thrk, int sides = 3) {
  constexpr float F1312 = 13.0f / 12.0f, F1348 = 13.0f / 48.0f;
  int verdict = 1;
  bool ok = true;
  float bm = fmaxf(fmaxf(fmaxf(fabsf(b[0]), fabsf(b[1])), fmaxf(fabsf(b[2]), fabsf(b[3]))), fabsf(b[4]));
  const float eta = ffma(al, ffma(0x1p-21f, bm, eb[0]), ea[0]);
  float ehi[4];
#pragma unroll
  for (int v = 0; v < 4; ++v) ehi[v] = ffma(al, ffma(0x1p-21f, fabsf(b[5 + v]), eb[1 + v]), ea[1 + v]);
#pragma unroll
  for (int side = 0; side < 2; ++side) {
    if (!((sides >> side) & 1)) continue;  // (a side known to vanish)
    const float sa = side ? -al : al;
    float d[5];
#pragma unroll
    for (int k = 0; k < 5; ++k) {
      const int p = side ? 4 - k : k;  // the - side reads the stencil mirrored
      d[k] = ffma(sa, b[p], a[p]);
    }
    const float s0 = fsub(d[1], d[0]), s1 = fsub(d[2], d[1]), s2 = fsub(d[3], d[2]), s3 = fsub(d[4], d[3]);
    const float e0 = fadd(s0, d[1]), g3 = ffma(3.0f, s2, -s3), e3 = fsub(s3, d[3]), dd = fmul(d[2], d[2]);
    const float b0 = ffma(fmul(F1312, s0), s0, fmul(e0, e0));
    const float b1 = ffma(fmul(F1312, s1), s1, dd);
    const float b2 = ffma(fmul(F1312, s2), s2, dd);
    const float b3 = ffma(fmul(F1348, g3), g3, fmul(e3, e3));
    const float S = fmaxf(fmaxf(fmaxf(fabsf(d[0]), fabsf(d[1])), fmaxf(fabsf(d[2]), fabsf(d[3]))), fabsf(d[4]));
    const float del = ffma(fmul(54.0f, S), eta, ffma(fmul(27.0f, eta), eta, fmul(fmul(0x1p-16f, S), S)));
    const float bmax = fmaxf(fmaxf(b0, b1), fmaxf(b2, b3)), bmin = fminf(fminf(b0, b1), fminf(b2, b3));
    const bool restricted =
        fadd(bmax, del) < fmul(fmul(alpha_R, fadd(epsk, fsub(bmin, del))), 1.0f - 0x1p-18f);
    const int y = side ? 7 : 6, z = side ? 6 : 7;  // the side's own fourth difference, the other
    const float t3 = fabsf(ffma(sa, b[5], a[5]));
    const float ty = ffma(sa, b[y], a[y]), tz = ffma(sa, b[z], a[z]);
    const float a5 = fabsf(ffma(sa, b[8], a[8])), a6 = fabsf(fadd(ty, tz)), e6 = fadd(ehi[1], ehi[2]);
    const float t5 = fadd(a5, ehi[3]), hi6 = fadd(a6, e6);
    const float lo3 = fmaxf(fsub(t3, ehi[0]), 0.0f), lo4 = fmaxf(fsub(fabsf(ty), ehi[y - 5]), 0.0f);
    const float tau5lo = ffma(fmul(F1312, lo4), lo4, fmul(lo3, lo3));
    const float tau6hi = ffma(fmul(F1312, t5), t5, fmul(0.25f, fmul(hi6, hi6)));
    const bool theta0 = fmul(tau6hi, 1.0f + 0x1p-18f) < tau5lo && tau5lo > 0x1p-100f;
    ok = ok && restricted;
    if (!TH1) {
      ok = ok && (theta0 || t5 <= thrk);
    } else if (!(theta0 || t5 <= thrk)) {  // (few stencils: not evaluated for the others)
      const float hi3 = fadd(t3, ehi[0]), hi4 = fadd(fabsf(ty), ehi[y - 5]);
      const float lo5 = fmaxf(fsub(a5, ehi[3]), 0.0f), lo6 = fmaxf(fsub(a6, e6), 0.0f);
      const float tau5hi = ffma(fmul(F1312, hi4), hi4, fmul(hi3, hi3));
      // (halved before the square: a bound that overflows must be one whose value does)
      const float hl6 = fmul(0.5f, lo6), tau6lo = ffma(fmul(F1312, lo5), lo5, fmul(hl6, hl6));
      ok = ok && fmul(tau5hi, 1.0f + 0x1p-18f) < tau6lo && tau6lo > 0x1p-100f;
      verdict |= side ? 4 : 2;
    }
  }
  return ok ? verdict : 0;
}
constexpr int kAllCentral = 1 | 1 << 3 | 1 << 6;  // the verdicts of three fields, three bits each
constexpr int kAllCentral2D = kAllCentral | 1 << 9;

// the fifth difference from the five cell differences, antisymmetric for mirrored data
__device__ __forceinline__ double fifth_difference(double d0, double d1, double d2, double d3, double d4) {
  return fma(6.0, d2, fma(-4.0, __dadd_rn(d1, d3), __dadd_rn(d0, d4)));
}
// the same from the six cell values
__device__ __forceinline__ double fifth_difference_q(double q0, double q1, double q2, double q3, double q4, double q5) {
  return fma(10.0, __dsub_rn(q3, q2), fma(-5.0, __dsub_rn(q4, q1), __dsub_rn(q5, q0)));
}
// F_s of a field whose decisions the screen has taken: C v+ + C v- less the theta = 1 sides' Delta^5 v / 60
// (the mirrored side's with the other sign), from c = l.(C f), a = l.(Delta^5 f), b = l.(Delta^5 u)
// with l scaled by 1/2
__device__ __forceinline__ double decided_field(int verdict, double c, double a, double b, double al) {
  const double tp = verdict & 2 ? 1.0 : 0.0, tm = verdict & 4 ? 1.0 : 0.0;
  const double w = fma(al * (tp + tm), b, (tp - tm) * a);
  return fma(-1.0 / 60.0, w, 2.0 * c);
}

// ---- 2D (Sec. 4.3): normal velocity u and tangential velocity t of a sweep.  Projections with w1 = xn - u
// x0, wt = xt - t x0, w2 = xE - u (xn + w1) / 2 - t (xt + wt) / 2; the shear field is wt itself, the
// others are those of 1D.
struct Roe32Shear {
  Roe32 r;
  float t, T;
};
__device__ __forceinline__ Roe32Shear roe32_2d(double ra_, double na_, double ta_, double Ha_, double rb_, double nb_,
                                               double tb_, double Hb_, float gm1) {
  Roe32Shear o;
  Roe32& r = o.r;
  const float ra = f32_trunc(ra_), rb = f32_trunc(rb_), ua = f32_trunc(na_), ub = f32_trunc(nb_);
  const float ta = f32_trunc(ta_), tb = f32_trunc(tb_), Ha = f32_trunc(Ha_), Hb = f32_trunc(Hb_);
  const float sa = fmul(ra, frsqrt_hw(ra)), sb = fmul(rb, frsqrt_hw(rb));
  const float hw = fmul(fmul(0.5f, fsub(sa, sb)), frcp_hw(fadd(sa, sb)));
  const float du = fsub(ua, ub), dt = fsub(ta, tb);
  r.u = ffma(hw, du, fmul(0.5f, fadd(ua, ub)));
  o.t = ffma(hw, dt, fmul(0.5f, fadd(ta, tb)));
  const float H = ffma(hw, fsub(Ha, Hb), fmul(0.5f, fadd(Ha, Hb)));
  r.U = fmaxf(fabsf(ua), fabsf(ub));
  o.T = fmaxf(fabsf(ta), fabsf(tb));
  const float he = ffma(-0.5f, fadd(fmul(r.u, r.u), fmul(o.t, o.t)), H);
  const float big = fadd(fadd(fmul(r.U, r.U), fmul(o.T, o.T)), fmaxf(fabsf(Ha), fabsf(Hb)));
  const float c2 = fmul(gm1, he);
  r.ic = frsqrt_hw(c2);
  r.b1 = fmul(gm1, fmul(r.ic, r.ic));
  r.rel = ffma(0x1p-19f, fmul(big, r.b1), 0x1p-20f);
  // (one more product and sum than in 1D: 2.75 * 2^-23 beside E / U, still below 1.5 * 2^-21)
  r.q = ffma(0x1p-20f, fmaxf(fmul(fabsf(du), frcp_hw(fadd(r.U, 1e-30f))), fmul(fabsf(dt), frcp_hw(fadd(o.T, 1e-30f)))),
             0x1.8p-21f);
  r.thr = fmul(fmul(60.0f * 0x1p-53f, fminf(ra, rb)), ffma(c2, r.ic, fabsf(r.u)));
  r.ok = ra > 0x1p-60f && rb > 0x1p-60f && ra < 0x1p60f && rb < 0x1p60f && fmul(he, 32.0f) >= big && big < 0x1p60f &&
         big > 0x1p-60f;
  return o;
}
// fields 0..3 (u - c, u, shear, u + c) of one array (f or u), as take_field: a field's projections and errors
struct Proj32Shear {
  float2 jk[9];
  float x0[9], wt[9];
  float2 nb[5];
  float nt[5];
  float jm, km, xm, tm;
};
__device__ __forceinline__ void project_stencil_2d(const Roe32Shear& o, const float (*d)[5], const float4* h,
                                                   Proj32Shear& p) {
  const Roe32& r = o.r;
  p.jm = p.km = p.xm = p.tm = 0.0f;
  // (no floor for tangential momenta that are equal throughout, f32_pair_nz: a sweep along a stream has a
  // shear field of zeros and a threshold of zero, and takes the central flux)
  float mx[4] = {kLow32, kLow32, 0.0f, kLow32};
#pragma unroll
  for (int v = 0; v < 9; ++v) {
    float x[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) x[c] = v < 5 ? d[c][v < 5 ? v : 0] : (v == 5 ? h[c].x : (v == 6 ? h[c].y : (v == 7 ? h[c].z : h[c].w)));
    const float w1 = ffma(-r.u, x[0], x[1]), wt = ffma(-o.t, x[0], x[2]);
    const float w2 = ffma(fmul(-0.5f, o.t), fadd(x[2], wt), ffma(fmul(-0.5f, r.u), fadd(x[1], w1), x[3]));
    p.jk[v] = make_float2(fmul(r.ic, w1), fmul(r.b1, w2));
    p.x0[v] = x[0];
    p.wt[v] = wt;
    if (v < 5) {
      p.jm = fmaxf(p.jm, fabsf(p.jk[v].x));
      p.km = fmaxf(p.km, fabsf(p.jk[v].y));
#pragma unroll
      for (int c = 0; c < 4; ++c) mx[c] = fmaxf(mx[c], fabsf(x[c]));
    }
    if (v >= 4) {  // the bounds of the largest cell difference, then of the high differences
      const int b = v - 4;
      if (b == 0) {
        p.xm = mx[0];
        if (mx[2] > 0.0f) mx[2] = fmaxf(mx[2], kLow32);
      }
      const float y0 = b == 0 ? mx[0] : fabsf(x[0]), y1 = b == 0 ? mx[1] : fabsf(x[1]),
                  y2 = b == 0 ? mx[2] : fabsf(x[2]), y3 = b == 0 ? mx[3] : fabsf(x[3]);
      const float n1 = ffma(r.U, y0, y1), nt = ffma(o.T, y0, y2);
      p.nb[b] = make_float2(fmul(r.ic, n1), fmul(r.b1, ffma(o.T, nt, ffma(r.U, n1, y3))));
      p.nt[b] = nt;
    }
  }
}
__device__ __forceinline__ void take_field_2d(int s, const Roe32Shear& o, const Proj32Shear& p, float* a, float* ea) {
  const Roe32& r = o.r;
  const int s1 = s == 3 ? 2 : s;  // the 1D field's number (s != 2)
#pragma unroll
  for (int k = 0; k < 9; ++k) a[k] = s == 2 ? p.wt[k] : field32(s1, p.jk[k], p.x0[k]);
  ea[0] = s == 2 ? fmul(r.q, p.nt[0]) : field_err(s1, r, p.nb[0], p.jm, p.km, p.xm);
  const float pe = fmul(0x1p-40f, s == 2 ? p.nt[0] : (s == 1 ? fadd(p.xm, p.nb[0].y) : fadd(p.nb[0].x, p.nb[0].y)));
#pragma unroll
  for (int v = 0; v < 4; ++v)
    ea[1 + v] = fadd(pe, s == 2 ? fmul(r.q, p.nt[1 + v])
                                : field_err(s1, r, p.nb[1 + v], fabsf(p.jk[5 + v].x), fabsf(p.jk[5 + v].y),
                                            fabsf(p.x0[5 + v])));
}

// the sixth-order central value (Eq. (fh_6)) from the two centre values and the outer four
// differences d_0, d_1, d_3, d_4: (q2 + q3) / 2 + (7 (d1 - d3) - (d0 - d4)) / 60, the same value
// for mirrored data
__device__ __forceinline__ double central_value(double q2, double q3, double d0, double d1, double d3, double d4) {
  const double x = fma(7.0 / 60.0, __dsub_rn(d1, d3), __dmul_rn(-1.0 / 60.0, __dsub_rn(d0, d4)));
  return fma(0.5, __dadd_rn(q2, q3), x);
}

}  // namespace wt
