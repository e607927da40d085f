// qs_grad.cuh -- device side of the adjoint of the beam phase-space
// integration, shared by the single-shot (qs_scatter_grad) and batched
// (qs_scatter_grad_batch) kernels: the discretised phase integration with
// two tangents (ln a_eff, 1/gamma0), or seven for the per-cell focus
// (every cell's amplitude depends on the geometry in its own way), a
// sample's decode and focus with the derivatives of ln a_eff, the sample's
// share of the upstream gradient and the chain rule to the 8 parameters, and
// the fixed-order reductions.
//
// Paper: Amaro & Vranic, "QScatter", arXiv 2308.09348 -- Eqs. 2, 3, 6, 8 and
// the reconstruction use of Sec. 6.
#pragma once

#include "qscatter.h"
#include "qs_device.cuh"

namespace qs {

constexpr int kNumGrad = QS_NUM_GRAD;

// ---- the phase integration with tangents --------------------------------
// The value recursion of qs_device (same cells, same midpoint prediction,
// same frozen-rate variance step) with first derivatives, written for one
// number type X: float2 (two samples, packed FP32: the path that is used) or
// double.  Every operation below is one FMA-pipe instruction per sample, and
// their number bounds the kernels, so the derivatives are arranged in
// logarithmic form.  With the field of a cell scaled by 1 + e (e = d ln A of
// a parameter; e = 0 for 1/gamma0), dum the state 1/mu - 1/gamma0 predicted
// at the midpoint and a dash its derivative,
//   rho = d ln chi = e - mu dum'   (for u0 = 1/gamma0: -mu (1 + dum'))
// is the only way in which a parameter enters the rates, so the derivatives
// of the rates are formed once per cell (X, Y, Zh, Ch below) and every
// tangent costs six to nine operations:
//   hlam/2 = L = n2 (s/2),            n2 = -2 hK mu,  s = 2g + chi g'
//   d L    = e L + X rho,             X = L + n2 (chi s'/2)
//   hD2    = bD h,                    bD = n2 mu^2 chi,  h = -(C55/2) h2
//   d hD2  = -e hD2 + Y rho,          Y = bD (4 h + chi h')
//   V_new  = V + hr (1 + L),          hr = 2 L V + hD2
//   d V    -> (1 + 2 L (1 + L)) dV + rho Zh + 2 e Ch,
//   Zh = (1 + L)(2 V X + Y) + hr X,   Ch = 2 L V (1/2 + L) - hD2/2.
// V is carried as W = 2V, g as gph = g/2, chi g' as m = chi g'/2.
// The two-tangent recursion takes 78 operations per cell this way, 103 with
// each derivative expanded by itself: 2^22 samples x 512 cells 6.59 -> 5.02
// ms.  Seven tangents, packed over two samples: 22.5 -> 9.8 ms; two tangents
// of the cycle-resolved model, packed and from the monomial tables: 10.4 ->
// 4.8 ms.
__device__ __forceinline__ float2 xmul(float2 a, float2 b) { return mul2(a, b); }
__device__ __forceinline__ float2 xfma(float2 a, float2 b, float2 c) { return fma2(a, b, c); }
__device__ __forceinline__ float2 xadd(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 xrcp(float2 a) { return rcpx2(a); }
__device__ __forceinline__ float2 xneg(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ double xmul(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ double xfma(double a, double b, double c) { return __fma_rn(a, b, c); }
__device__ __forceinline__ double xadd(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ double xrcp(double a) { return rcp_d(a); }
__device__ __forceinline__ double xneg(double a) { return -a; }
template <typename X> __device__ __forceinline__ X xset(double c);
template <> __device__ __forceinline__ float2 xset<float2>(double c) { return f2((float)c); }
template <> __device__ __forceinline__ double xset<double>(double c) { return c; }
// A launch constant in the path's type.
#define QS_XV(X, field) xset_pv<X>(p.field, p.f.field)
template <typename X> __device__ __forceinline__ X xset_pv(double d, float f);
template <> __device__ __forceinline__ float2 xset_pv<float2>(double, float f) { return f2(f); }
template <> __device__ __forceinline__ double xset_pv<double>(double d, float) { return d; }

// Table entry of cell j: G, and G^2 or (per-cell focus) the path shift s_j.
template <bool FOC>
__device__ __forceinline__ void tab_x(const Params&, const float4* t, int j, float2& G, float2& b) {
  const float4 e = t[j];
  G = make_float2(e.x, e.y);
  b = make_float2(e.z, e.w);
}
template <bool FOC>
__device__ __forceinline__ void tab_x(const Params& p, const double* t, int j, double& G, double& b) {
  G = t[j];
  b = FOC ? cell_shift(p, j) : G * G;
}

// The rates' factors at chi: gph = g/2, m = chi g'/2, sx = chi s'/2 with s =
// 2g + chi g' (chi s' = 3 chi g' + chi^2 g''), h = -(C55/2) h2 and hx =
// chi dh/dchi -- closed forms of the fits, or (VAR & kVarCycle) their means
// over the laser cycle.
template <typename X> struct Factors { X gph, m, sx, h, hx; };

// FP64: from the closed forms' derivatives.
template <int VAR>
__device__ __forceinline__ void factors(const Params& p, const float4* __restrict__, double chi,
                                        Factors<double>& o) {
  double g, chig1, chis1, h2, chih1;                   // g, chi g', chi s', h2, chi h2'
  if constexpr ((VAR & kVarCycle) != 0) {
    double s, dG, dS, dH;
    cycle_factors_d(p.cyc_gl, chi, g, s, h2, &dG, &dS, &dH);
    chig1 = chi * dG;
    chis1 = chi * dS;
    chih1 = chi * dH;
  } else {
    //   g'  = -(2/3) g B'/B,  g'' = (10/9) g (B'/B)^2 - (2/3) g B''/B,
    //   B'  = 4.8 ln(1+1.7chi) + 4.8 + 3.36/(1+1.7chi) + 4.88 chi,
    //   B'' = 8.16/(1+1.7chi) - 5.712/(1+1.7chi)^2 + 4.88,
    //   h2 = g R, R = N/D (the rational second-moment fit), R' = (N' - R D')/D
    const double x1 = fma(1.7, chi, 1.0), L1 = log_d(x1), r1 = rcp_d(x1);
    const double B = fma(fma(4.8, chi, 4.8), L1, fma(2.44 * chi, chi, 1.0));
    const double t = icbrt_d(B);
    g = t * t;
    const double ci = chi * (t * g);                   // chi / B
    const double q = ci * fma(4.8, L1, fma(3.36, r1, fma(4.88, chi, 4.8)));      // chi B'/B
    const double b2 = ci * chi * fma(fma(-5.712, r1, 8.16), r1, 4.88);           // chi^2 B''/B
    chig1 = (-2.0 / 3.0) * g * q;
    chis1 = fma(3.0, chig1, g * fma((10.0 / 9.0) * q, q, (-2.0 / 3.0) * b2));
    const double D = fma(fma(fma(kHB3, chi, kHB2), chi, kHB1), chi, 1.0), iD = rcp_d(D);
    const double R = fma(fma(kHA2, chi, kHA1), chi, 1.0) * iD;
    const double Np = fma(2.0 * kHA2, chi, kHA1);
    const double Dp = fma(fma(3.0 * kHB3, chi, 2.0 * kHB2), chi, kHB1);
    h2 = g * R;
    chih1 = fma(chig1, R, g * (fma(-R, Dp, Np) * (chi * iD)));
  }
  o.gph = 0.5 * g;
  o.m = 0.5 * chig1;
  o.sx = 0.5 * chis1;
  o.h = (-0.5 * kC55) * h2;
  o.hx = (-0.5 * kC55) * chih1;
}

// FP32, two samples.  Cycle means: the monomial tables A of the forward
// lookup (per interval c0..c3 of G, then of H), value, first and half the
// second derivative in t by synthetic division; with k = dt/d ln chi =
// chi / (DU (chi + chi_s)), DU = du ln2 (so dk/d ln chi = k (1 - k DU)),
//   chi G' = G_t k,  chi^2 G'' = k^2 (G_tt - DU G_t),  chi H' = H_t k.
__device__ __forceinline__ void cycle_eval(const float4 c, float t, float& v, float& d1,
                                           float& hd2) {
  const float b2 = __fmaf_rn(c.w, t, c.z), b1 = __fmaf_rn(b2, t, c.y);
  const float e2 = __fmaf_rn(c.w, t, b2);
  v = __fmaf_rn(b1, t, c.x);
  d1 = __fmaf_rn(e2, t, b1);
  hd2 = __fmaf_rn(c.w, t, e2);
}
template <int VAR>
__device__ __forceinline__ void factors(const Params&, const float4* __restrict__ A, float2 chi,
                                        Factors<float2>& o) {
  if constexpr ((VAR & kVarCycle) != 0) {
    constexpr float kS = (float)(kCycN - 1) - 1e-3f;
    constexpr double DU = kCycDu * 0.69314718055994530942;
    const float2 u = lg2x2(fma2(chi, f2((float)(1.0 / kCycChiS)), f2(1.f)));
    const float sa = (float)(1.0 / (kCycDu * kS));
    const float2 sx = make_float2(fma_sat(u.x, sa, 0.f), fma_sat(u.y, sa, 0.f));
    const float2 xm = __fadd2_rn(fma2(sx, f2(kS), f2(-0.5f)), f2(12582912.f));
    const int i0 = __float_as_int(xm.x) - 0x4B400000, i1 = __float_as_int(xm.y) - 0x4B400000;
    const float2 t = fma2(sx, f2(kS), fma2(xm, f2(-1.f), f2(12582912.f)));
    const float2 k = mul2(chi, rcpx2(mul2(f2((float)DU), __fadd2_rn(chi, f2((float)kCycChiS)))));
    float2 G, Gt, Gh, H, Ht, Hh;
    cycle_eval(A[i0], t.x, G.x, Gt.x, Gh.x);
    cycle_eval(A[i1], t.y, G.y, Gt.y, Gh.y);
    cycle_eval(A[kCycN + i0], t.x, H.x, Ht.x, Hh.x);
    cycle_eval(A[kCycN + i1], t.y, H.y, Ht.y, Hh.y);
    const float2 k2 = mul2(k, k);
    o.gph = mul2(f2(0.5f), G);
    o.m = mul2(mul2(f2(0.5f), Gt), k);
    o.sx = fma2(f2(3.f), o.m, mul2(k2, fma2(f2((float)(-0.5 * DU)), Gt, Gh)));
    o.h = mul2(f2((float)(-0.5 * kC55)), H);
    o.hx = mul2(mul2(f2((float)(-0.5 * kC55)), Ht), k);
  } else {
    // In xh = sqrt(2.44) chi, t = B^(-1/3)/sqrt2 (so t^2 = g/2 and chi/B =
    // (2 sqrt2/sqrt2.44) xh t gph); q = -(2/3) chi B'/B, so m = gph q and
    // chi^2 g''/2 = gph ((5/2) q^2 - (2/3) chi^2 B''/B).
    constexpr double kap = 1.5620499351813308;         // sqrt(2.44)
    constexpr double kk = -(2.0 / 3.0) * 2.8284271247461901 / kap;
    constexpr double ln2 = 0.69314718055994530942;
    const float2 ONE = f2(1.f);
    const float2 xh = mul2(f2((float)kap), chi);
    const float2 l1 = lg2x2(fma2(f2(1.7f), chi, ONE));
    const float2 B = fma2(fma2(f2((float)(4.8 * ln2 / kap)), xh, f2((float)(4.8 * ln2))), l1,
                          fma2(xh, xh, ONE));
    const float2 t = ex2x2(fma2(lg2x2(B), f2(-1.f / 3.f), f2(-0.5f)));
    const float2 r1 = ex2x2(make_float2(-l1.x, -l1.y));              // 1/(1+1.7 chi)
    o.gph = mul2(t, t);
    const float2 ci = mul2(xh, mul2(t, o.gph));
    const float2 q = mul2(ci, fma2(f2((float)(kk * 4.8 * ln2)), l1,
                                   fma2(f2((float)(kk * 4.88 / kap)), xh,
                                        fma2(f2((float)(kk * 3.36)), r1, f2((float)(kk * 4.8))))));
    const float2 b2 = mul2(mul2(ci, xh), fma2(fma2(f2((float)(-kk / kap * 5.712)), r1,
                                                   f2((float)(kk / kap * 8.16))), r1,
                                              f2((float)(kk / kap * 4.88))));
    o.m = mul2(o.gph, q);
    o.sx = mul2(o.gph, fma2(q, fma2(f2(2.5f), q, f2(3.f)), b2));
    // R = -C55 N/D, R' from N' and -D' (all in xh)
    constexpr double a1 = -kC55 * kHA1 / kap, a2 = -kC55 * kHA2 / (kap * kap);
    constexpr double d1 = kHB1 / kap, d2 = kHB2 / (kap * kap), d3 = kHB3 / (kap * kap * kap);
    const float2 iD = rcpx2(fma2(fma2(fma2(f2((float)d3), xh, f2((float)d2)), xh, f2((float)d1)),
                                 xh, ONE));
    const float2 R = mul2(fma2(fma2(f2((float)a2), xh, f2((float)a1)), xh, f2((float)-kC55)), iD);
    const float2 nDp = fma2(fma2(f2((float)(-3.0 * d3)), xh, f2((float)(-2.0 * d2))), xh,
                            f2((float)-d1));
    const float2 xR = mul2(fma2(R, nDp, fma2(f2((float)(2.0 * a2)), xh, f2((float)a1))),
                           mul2(xh, iD));
    o.h = mul2(o.gph, R);
    o.hx = fma2(o.m, R, mul2(o.gph, xR));
  }
}

// Value state, and what a cell hands to its tangents.
template <typename X> struct CellState { X du, W, gph; };
template <typename X> struct CellOut { X m, gph, hK2, H, Zh, Ch; };

// The second half of a cell: value update and the tangents' coefficients,
// from the midpoint (hK, nmu = -mu, chi).
template <typename X, int VAR>
__device__ __forceinline__ void cell_update(const Params& p, const float4* __restrict__ cA, X hK,
                                            X nmu, X chi, CellState<X>& st, CellOut<X>& o) {
  Factors<X> F;
  factors<VAR>(p, cA, chi, F);
  const X ONE = xset<X>(1.0);
  o.m = F.m;
  o.gph = F.gph;
  o.hK2 = xadd(hK, hK);
  const X sh = xfma(xset<X>(2.0), F.gph, F.m);
  const X n2 = xmul(o.hK2, nmu);
  const X L = xmul(n2, sh), Xc = xmul(n2, xadd(sh, F.sx));
  const X bD = xmul(xmul(n2, xmul(nmu, nmu)), chi);
  const X hD2 = xmul(bD, F.h), Y = xmul(bD, xfma(xset<X>(4.0), F.h, F.hx));
  const X fac = xadd(L, ONE), fac2 = xadd(fac, fac);
  const X LW = xmul(L, st.W), hr = xadd(LW, hD2);
  o.Zh = xfma(fac, xfma(Xc, st.W, Y), xmul(hr, Xc));
  o.Ch = xfma(LW, xadd(L, xset<X>(0.5)), xmul(xset<X>(-0.5), hD2));
  o.H = xfma(fac2, L, ONE);
  st.W = xfma(hr, fac2, st.W);
  st.du = xfma(o.hK2, F.gph, st.du);
  st.gph = F.gph;
}

// Result of the two-tangent integration: the state and V, their derivatives
// with respect to ln a_eff, and du + u0 and V with respect to u0 = 1/gamma0
// (u: d(1/mu)/du0).
template <typename T> struct QfpTan { T du, V, du_l, V_l, u, V_u; };

// The model whose every cell sees a_eff (variant 0, cycle-resolved chi): the
// tangents of the field's logarithm l and of u0.  The l tangent is carried for
// e = 1/2, i.e. with respect to 2 ln a (then hK' = hK).
template <typename X, int VAR, typename TT>
__device__ __forceinline__ void qfp_tangent(const Params& p, const TT* __restrict__ tab, X a, X ig0,
                                            X& du_o, X& V_o, X& du_l, X& V_l, X& u_o, X& V_u,
                                            const float4* __restrict__ cA) {
  const X hcK = xmul(QS_XV(X, h), QS_XV(X, cK));
  const X c1 = xmul(xmul(hcK, a), a), nca = xneg(xmul(QS_XV(X, cchi), a));
  const X ZERO = xset<X>(0.0), HALF = xset<X>(0.5);
  CellState<X> st{ZERO, ZERO, HALF};
  // tangents of du and V, and of the previous cell's hK g/2 over hK
  X du_a = ZERO, V_a = ZERO, pa = HALF, du_g = ZERO, V_g = ZERO, pg = ZERO;
  const int N = p.n_phase;
  for (int j = 0; j < N; ++j) {
    X G, G2;
    tab_x<false>(p, tab, j, G, G2);
    const X hK = xmul(c1, G2);
    const X nmu = xrcp(xneg(xadd(xfma(hK, st.gph, st.du), ig0)));
    const X chi = xmul(xmul(nca, G), nmu);
    const X ra = xfma(nmu, xfma(hK, pa, du_a), HALF);
    const X rg = xfma(nmu, xfma(hK, pg, du_g), nmu);
    CellOut<X> o;
    cell_update<X, VAR>(p, cA, hK, nmu, chi, st, o);
    pa = xfma(o.m, ra, o.gph);
    pg = xmul(o.m, rg);
    du_a = xfma(o.hK2, pa, du_a);
    du_g = xfma(o.hK2, pg, du_g);
    V_a = xfma(o.H, V_a, xfma(ra, o.Zh, o.Ch));
    V_g = xfma(o.H, V_g, xmul(rg, o.Zh));
  }
  const X TWO = xset<X>(2.0);
  du_o = st.du;
  V_o = xmul(HALF, st.W);
  du_l = xmul(TWO, du_a);
  V_l = xmul(TWO, V_a);
  u_o = xadd(xset<X>(1.0), du_g);
  V_u = V_g;
}

// Upstream gradient, reduced to the per-sample coefficients it needs (in
// the path's arithmetic type).
template <typename T>
struct Seeds {
  T invW, mean, spread, dxr, dyr;             // forward moments
  T gM, gSp, gDx, gDy, gA, gG0;               // effective dL/d(mean, spread, div_x, div_y, a, g0)
};

// A sample's decode and focus with the derivatives of ln a (rows a1-a3).
template <typename T>
struct GFront {
  T w, xi3, xi4, xi5, gamma0, a, a_over_a0;
  T dla_w0, dla_dx, dla_dy, dla_thx, dla_thy, dla_del, thx, thy;
  T zq, xs, ys, ct, w0;        // crossing geometry (per-cell focus)
  bool ok, clamped;
};

template <typename T>
__device__ __forceinline__ void grad_front(const Params& p, int64_t i, T w0, GFront<T>& f) {
  const T xi0 = load_t<T>(p.xi[0], i, p.dtype), xi1 = load_t<T>(p.xi[1], i, p.dtype);
  const T xi2 = load_t<T>(p.xi[2], i, p.dtype);
  f.xi3 = load_t<T>(p.xi[3], i, p.dtype);
  f.xi4 = load_t<T>(p.xi[4], i, p.dtype);
  f.xi5 = load_t<T>(p.xi[5], i, p.dtype);
  f.w = p.weighted ? load_t<T>(p.w, i, p.dtype) : (T)1;
  f.ok = f.w >= (T)0 && isfinite(f.w);
  const T x = QS_PV(T, bdx) + QS_PV(T, sx) * xi0;
  const T y = QS_PV(T, bdy) + QS_PV(T, sy) * xi1;
  const T z = QS_PV(T, sz) * xi2;
  T gamma0 = p.flat ? QS_PV(T, glo) + QS_PV(T, gspan) * f.xi3
                    : QS_PV(T, gmean) * ((T)1 + QS_PV(T, spread) * f.xi3);
  f.clamped = gamma0 < (T)1;
  if (f.clamped) gamma0 = (T)1;
  f.gamma0 = gamma0;
  const T thx = QS_PV(T, div) * f.xi4, thy = QS_PV(T, div) * f.xi5;
  f.thx = thx;
  f.thy = thy;
  const T cdel = QS_PV(T, c_delay);
  const T ct = (T)0.5 * (z + cdel);
  const T zs = (T)0.5 * (z - cdel);
  const T xs = x + thx * ct - QS_PV(T, ldx);
  const T ys = y + thy * ct - QS_PV(T, ldy);
  const T rho2 = xs * xs + ys * ys;
  const T izR = QS_PV(T, inv_zR), iw2 = QS_PV(T, inv_w0sq);
  const T zq = zs * izR;
  const T q = (T)1 + zq * zq;
  const T rq = M<T>::rcp(q);
  const T E = rho2 * iw2 * rq;                         // a = a0 q^-1/2 exp(-E)
  if constexpr (sizeof(T) == 4)
    f.a_over_a0 = M<T>::rsqrt(q) * M<T>::ex2(-(T)1.4426950408889634074 * E);
  else
    f.a_over_a0 = M<T>::rsqrt(q) * (T)exp(-(double)E);
  f.a = QS_PV(T, a0) * f.a_over_a0;
  // d ln a / d(parameter)
  const T k2 = (T)2 * iw2 * rq;                        // 2 / (W0^2 q)
  f.dla_dx = k2 * xs;
  f.dla_dy = k2 * ys;
  f.dla_thx = -k2 * xs * ct;
  f.dla_thy = -k2 * ys * ct;
  const T cc = (T)0.299792458;
  const T dq_del = -cc * zq * izR;                     // dq/d delay
  const T drho_del = cc * (xs * thx + ys * thy);       // d rho^2 / d delay
  f.dla_del = (E - (T)0.5) * dq_del * rq - drho_del * iw2 * rq;
  const T dq_w0 = (T)-4 * zq * zq / w0;                // dq/dW0 (z_R ~ W0^2)
  f.dla_w0 = (T)-0.5 * dq_w0 * rq + E * ((T)2 / w0 + dq_w0 * rq);
  f.zq = zq;
  f.xs = xs;
  f.ys = ys;
  f.ct = ct;
  f.w0 = w0;
}

// Per-cell focus (QS_VARIANT_CELL_FOCUS): the local amplitude a_j of a cell
// at shift s along the path (Eq. 2 at z* - s, xs + theta_x s, ys + theta_y s)
// and e_k = d ln a_j / d(parameter), from
//   ln a_j = ln a0 - (1/2) ln q_j - E_j,  q_j = 1 + zq_j^2,  E_j = rho_j^2/(W0^2 q_j):
//   W0    (E - 1/2) q'/q + 2E/W0 with q' = -4 zq_j^2/W0 (z_R ~ W0^2)
//         = (2/W0) (E - zq^2 (2E - 1)/q)
//         (as (2/W0) (1 - E + (2E - 1)/q), one operation more, it cancels for a
//         spot wide against the beam: E and zq^2 small, FP32 relative error
//         per sample 3e-3 for W0 = 40 um and a beam of 0.1 um)
//   dx    2 x_j/(W0^2 q_j),  dy the same with y_j
//   delay (E - 1/2) q'/q - rho'/(W0^2 q) with q' = -c zq_j/z_R,
//         rho' = c (x_j theta_x + y_j theta_y) (the crossing moves by c/2)
//         = -c ((2E - 1) zq/(2 z_R q) + div P)
//   div   -2 (x_j xi4 + y_j xi5)(ct + s)/(W0^2 q_j) = -2 P (ct + s)
// with P = (x_j xi4 + y_j xi5)/(W0^2 q_j).  The tangents are linear in e_k,
// so the cells carry e[1..5] without the constant factors (2/W0, 2, 2, -c,
// -2), which the result takes once; e[0] = 1 (ln a0).
template <typename X> struct FocPath { X zq, xs, ys, thx, thy, xi4, xi5, ct; };
__device__ __forceinline__ float2 xrsqrt(float2 a) { return rsqrtx2(a); }
__device__ __forceinline__ double xrsqrt(double a) { return rsqrt_d(a); }
__device__ __forceinline__ float2 xexpn(float2 E) {
  return ex2x2(mul2(f2(-1.4426950408889634074f), E));
}
__device__ __forceinline__ double xexpn(double E) { return exp(-E); }

constexpr int kNE = 5;         // e[1..5]: W0, dx, dy, delay, div
template <typename X>
__device__ __forceinline__ X cell_amp(const Params& p, const FocPath<X>& f, X s, X (&e)[kNE]) {
  const X ONE = xset<X>(1.0);
  const X izR = QS_XV(X, inv_zR);
  const X zq = xfma(s, xneg(izR), f.zq);
  const X rs = xrsqrt(xfma(zq, zq, ONE)), rq = xmul(rs, rs);
  const X xj = xfma(f.thx, s, f.xs), yj = xfma(f.thy, s, f.ys);
  const X kq = xmul(QS_XV(X, inv_w0sq), rq);
  const X E = xmul(xfma(xj, xj, xmul(yj, yj)), kq);
  const X Fq = xmul(xfma(xset<X>(2.0), E, xset<X>(-1.0)), rq);           // (2E - 1)/q
  const X zF = xmul(zq, Fq);
  e[0] = xfma(xneg(zq), zF, E);
  e[1] = xmul(kq, xj);
  e[2] = xmul(kq, yj);
  const X P = xfma(e[1], f.xi4, xmul(e[2], f.xi5));
  e[3] = xfma(xmul(xset<X>(0.5), izR), zF, xmul(QS_XV(X, div), P));
  e[4] = xmul(P, xadd(f.ct, s));
  return xmul(xmul(QS_XV(X, a0), rs), xexpn(E));
}

// Tangents of the per-cell-focus model: ln a0, the five of cell_amp (without
// their constant factors) and u0 = 1/gamma0 (du_t[6] is d(1/mu)/du0); for
// the classical model Eq. 3's exponent summed cell by cell.
constexpr int kNT = 7;
template <typename X> struct FocTanX { X du, V, du_t[kNT], V_t[kNT]; };
template <typename T> struct FocTan { T du, V, du_t[kNT], V_t[kNT]; };

template <typename X, bool QFP, int VAR, typename TT>
__device__ __forceinline__ void focus_tangent(const Params& p, const TT* __restrict__ tab,
                                              const FocPath<X>& f, X ig0, FocTanX<X>& o,
                                              const float4* __restrict__ cA) {
  const X hcK = xmul(QS_XV(X, h), QS_XV(X, cK)), ncchi = xneg(QS_XV(X, cchi));
  const X ZERO = xset<X>(0.0), HALF = xset<X>(0.5);
  const int N = p.n_phase;
  X du_t[kNT], V_t[kNT], q_t[kNT];
#pragma unroll
  for (int k = 0; k < kNT; ++k) du_t[k] = V_t[k] = q_t[k] = ZERO;
  CellState<X> st{ZERO, ZERO, HALF};
  q_t[0] = HALF;                               // ln a0: carried for e = 1/2 (see qfp_tangent)
#pragma unroll 1
  for (int j = 0; j < N; ++j) {
    X G, s, e[kNE];
    tab_x<true>(p, tab, j, G, s);
    const X A = xmul(cell_amp<X>(p, f, s, e), G);
    const X hK = xmul(xmul(hcK, A), A);
    if constexpr (!QFP) {
      st.du = xadd(st.du, hK);
#pragma unroll
      for (int k = 0; k < kNE; ++k) du_t[k + 1] = xfma(hK, e[k], du_t[k + 1]);
    } else {
      const X nmu = xrcp(xneg(xadd(xfma(hK, st.gph, st.du), ig0)));
      const X chi = xmul(xmul(ncchi, A), nmu);
      const X g2 = xadd(st.gph, st.gph);
      X r[kNT];
      r[0] = xfma(nmu, xfma(hK, q_t[0], du_t[0]), HALF);
#pragma unroll
      for (int k = 0; k < kNE; ++k)
        r[k + 1] = xfma(nmu, xfma(hK, xfma(e[k], g2, q_t[k + 1]), du_t[k + 1]), e[k]);
      r[6] = xfma(nmu, xfma(hK, q_t[6], du_t[6]), nmu);
      CellOut<X> c;
      cell_update<X, VAR>(p, cA, hK, nmu, chi, st, c);
      const X g2n = xadd(c.gph, c.gph), Ch2 = xadd(c.Ch, c.Ch);
      q_t[0] = xfma(c.m, r[0], c.gph);
      du_t[0] = xfma(c.hK2, q_t[0], du_t[0]);
      V_t[0] = xfma(c.H, V_t[0], xfma(r[0], c.Zh, c.Ch));
#pragma unroll
      for (int k = 1; k <= kNE; ++k) {
        q_t[k] = xmul(c.m, r[k]);
        du_t[k] = xfma(c.hK2, xfma(e[k - 1], g2n, q_t[k]), du_t[k]);
        V_t[k] = xfma(c.H, V_t[k], xfma(r[k], c.Zh, xmul(e[k - 1], Ch2)));
      }
      q_t[6] = xmul(c.m, r[6]);
      du_t[6] = xfma(c.hK2, q_t[6], du_t[6]);
      V_t[6] = xfma(c.H, V_t[6], xmul(r[6], c.Zh));
    }
  }
  o.du = st.du;
  o.V = xmul(HALF, st.W);
  const X TWO = xset<X>(2.0);
  if constexpr (!QFP) {
    // dhK = 2 hK e_k; 1/gamma_f = 1/gamma0 + sum hK
    o.du_t[0] = xmul(TWO, st.du);
#pragma unroll
    for (int k = 1; k <= kNE; ++k) o.du_t[k] = xmul(TWO, du_t[k]);
    o.du_t[6] = xset<X>(1.0);
#pragma unroll
    for (int k = 0; k < kNT; ++k) o.V_t[k] = ZERO;
  } else {
#pragma unroll
    for (int k = 0; k < kNT; ++k) {
      o.du_t[k] = du_t[k];
      o.V_t[k] = V_t[k];
    }
    o.du_t[0] = xmul(TWO, du_t[0]);
    o.V_t[0] = xmul(TWO, V_t[0]);
    o.du_t[6] = xadd(xset<X>(1.0), du_t[6]);
  }
}

// Per-thread gradient partials: FP64 sums (FP64 path), compensated FP32
// sums (FP32 path).
template <typename T> struct GAcc;
template <> struct GAcc<double> {
  double s[kNumGrad];
  __device__ __forceinline__ void init() {
    for (int k = 0; k < kNumGrad; ++k) s[k] = 0.0;
  }
  __device__ __forceinline__ void add(int k, double x) { s[k] += x; }
  __device__ __forceinline__ double get(int k) const { return s[k]; }
};
template <> struct GAcc<float> {
  float s[kNumGrad], c[kNumGrad];
  __device__ __forceinline__ void init() {
    for (int k = 0; k < kNumGrad; ++k) s[k] = c[k] = 0.f;
  }
  __device__ __forceinline__ void add(int k, float x) { kahan(s[k], c[k], x); }
  __device__ __forceinline__ double get(int k) const { return (double)s[k] - (double)c[k]; }
};

// dL/d(the sample's outputs) from the upstream gradient (adjoint of rows
// a8-a9 and of the smoothed spectrum), and through Eq. 8 (theta_e = kappa_s
// a sqrt(V) / mu^2, a the crossing a_eff): the sample's share of dL/d mu,
// dL/d V, dL/d a_eff (directly), dL/d gamma0 (directly) and dL/d theta_x0,
// theta_y0.  False if the sample's result is not finite (it then adds
// nothing, as the forward excluded it).
template <typename T>
struct GOut {
  T g_mu, g_V, g_a, g_g0, g_thx, g_thy;
};

template <typename T, bool QFP, typename S>
__device__ __forceinline__ bool sample_upstream(const Params& p, const Seeds<T>& sd,
                                                const S* __restrict__ dLdS, int64_t i,
                                                const GFront<T>& f, T mu, T V, GOut<T>& go) {
  const T a = f.a;
  if (!isfinite(mu) || !isfinite(V)) return false;
  // outputs of the sample (row a6)
  T theta_e = 0, gout = mu, sv = 0;
  const T xi7 = QFP ? load_t<T>(p.xi[7], i, p.dtype) : (T)0;
  if (QFP && V > (T)0) {
    sv = sqrt(V);
    theta_e = QS_PV(T, kappa_s) * a * sv / (mu * mu);
    gout = mu + sv * xi7;
  }
  // sample's share of dL/d(outputs)
  const T wn = f.w * sd.invW;
  T g_out = 0;                                          // dL/d gamma_out
  if (dLdS != nullptr) {
    const T tt = (gout - QS_PV(T, lo)) * QS_PV(T, inv_w);
    if (tt > (T)-1e9 && tt < (T)1e9) {
      int k0, k1;
      T c;
      if constexpr (sizeof(T) == 4) {
        smooth_range_f32(p, tt, &k0, &k1);
        c = p.f.smooth_c;
      } else {
        smooth_range(p, tt, &k0, &k1);
        c = p.smooth_c;
      }
      const T tf = tt - (T)k0;
      for (int k = k0; k <= k1; ++k) {
        const T d = (T)(k - k0) + (T)0.5 - tf;
        T e;
        if constexpr (sizeof(T) == 4) e = M<float>::ex2(-(d * d) * c);
        else e = exp2(-d * d * c);
        g_out += (T)dLdS[k] * e * d;
      }
      const T sg = QS_PV(T, smooth_sigma);
      g_out *= f.w * QS_PV(T, smooth_pref) * QS_PV(T, inv_w) / (sg * sg);
    }
  }
  T g_mu = sd.gM * wn + g_out;
  if (sd.spread > (T)0) g_mu += sd.gSp * wn * (mu - sd.mean) / sd.spread;
  T g_V = (sd.spread > (T)0 ? sd.gSp * wn * (T)0.5 / sd.spread : (T)0);
  if (QFP && V > (T)0) g_V += g_out * xi7 * (T)0.5 / sv;
  const T g_te = sd.gDx * wn * theta_e * sd.dxr;
  go.g_thx = sd.gDx * wn * f.thx * sd.dxr;
  go.g_thy = sd.gDy * wn * f.thy * sd.dyr;
  T g_a = sd.gA * wn;
  go.g_g0 = sd.gG0 * wn;
  // theta_e = kappa_s a sqrt(V) / mu^2
  if (QFP && V > (T)0) {
    const T ks = QS_PV(T, kappa_s);
    g_a += g_te * ks * sv / (mu * mu);
    g_V += g_te * ks * a * (T)0.5 / (sv * mu * mu);
    g_mu += g_te * ((T)-2 * theta_e / mu);
  }
  go.g_mu = g_mu;
  go.g_V = g_V;
  go.g_a = g_a;
  return true;
}

// The sample's outputs, its share of dL/d(outputs) and the chain rule to the
// parameters (rows a4-a6), for the model whose phase integration sees a_eff
// in every cell (variant 0, cycle-resolved chi): (mu, V) = F(ln a_eff,
// 1/gamma0), and ln a_eff carries the parameters' dependence.
template <typename T, bool QFP, typename S>
__device__ __forceinline__ void grad_back(const Params& p, const Seeds<T>& sd,
                                          const S* __restrict__ dLdS, int64_t i,
                                          const GFront<T>& f, const QfpTan<T>& o, GAcc<T>& acc) {
  const T g0 = f.gamma0, a = f.a, ig0 = (T)1 / g0;
  T mu, V = 0, mu_l, mu_g, V_l = 0, V_g = 0;            // d/d ln a, d/d gamma0
  if (!QFP) {
    mu = g0 / ((T)1 + QS_PV(T, cRR) * g0 * a * a);
    mu_l = -mu * mu * (T)2 * QS_PV(T, cRR) * a * a;
    mu_g = mu * mu * ig0 * ig0;
  } else {
    mu = g0 / ((T)1 + g0 * o.du);
    mu_l = -mu * mu * o.du_l;
    mu_g = mu * mu * ig0 * ig0 * o.u;
    V = o.V;
    V_l = o.V_l;
    V_g = -ig0 * ig0 * o.V_u;
  }
  GOut<T> go;
  if (!sample_upstream<T, QFP, S>(p, sd, dLdS, i, f, mu, V, go)) return;
  const T ga = go.g_a * a + go.g_mu * mu_l + go.g_V * V_l;     // dL/d ln a
  const T g_g0 = go.g_g0 + go.g_mu * mu_g + go.g_V * V_g;
  // chain to the parameters
  const T a0v = QS_PV(T, a0);
  acc.add(QS_G_A0, a0v > (T)0 ? ga / a0v : (T)0);
  acc.add(QS_G_W0, ga * f.dla_w0);
  acc.add(QS_G_DX, ga * f.dla_dx);
  acc.add(QS_G_DY, ga * f.dla_dy);
  acc.add(QS_G_DELAY, ga * f.dla_del);
  if (!p.flat && !f.clamped) {
    acc.add(QS_G_GAMMA, g_g0 * ((T)1 + QS_PV(T, spread) * f.xi3));
    acc.add(QS_G_SPREAD, g_g0 * QS_PV(T, gmean) * f.xi3);
  }
  acc.add(QS_G_DIV, (go.g_thx + ga * f.dla_thx) * f.xi4 + (go.g_thy + ga * f.dla_thy) * f.xi5);
}

// The same for the per-cell focus: mu and V depend on the parameters through
// every cell's a_j (the seven tangents of focus_tangent, their constant
// factors taken here), while a_eff at the crossing still enters Eq. 8 and
// the a_eff moment directly.
template <typename T, bool QFP, typename S>
__device__ __forceinline__ void grad_back_focus(const Params& p, const Seeds<T>& sd,
                                                const S* __restrict__ dLdS, int64_t i,
                                                const GFront<T>& f, const FocTan<T>& o,
                                                GAcc<T>& acc) {
  const T g0 = f.gamma0, a = f.a, ig0 = (T)1 / g0;
  const T mu = g0 / ((T)1 + g0 * o.du);
  const T m2 = mu * mu;
  const T V = QFP ? o.V : (T)0;
  GOut<T> go;
  if (!sample_upstream<T, QFP, S>(p, sd, dLdS, i, f, mu, V, go)) return;
  // d(mu, V)/d theta_k through the cells (k: ln a0, W0, dx, dy, delay, div)
  T gk[6];
#pragma unroll
  for (int k = 0; k < 6; ++k) gk[k] = go.g_mu * (-m2 * o.du_t[k]) + (QFP ? go.g_V * o.V_t[k] : (T)0);
  const T g_g0 = go.g_g0 + ig0 * ig0 * (go.g_mu * m2 * o.du_t[6] -
                                        (QFP ? go.g_V * o.V_t[6] : (T)0));
  const T ga = go.g_a * a;                              // direct dL/d ln a_eff
  const T a0v = QS_PV(T, a0), cc = (T)0.299792458;
  acc.add(QS_G_A0, a0v > (T)0 ? (ga + gk[0]) / a0v : (T)0);
  acc.add(QS_G_W0, ga * f.dla_w0 + (T)2 * gk[1] / f.w0);
  acc.add(QS_G_DX, ga * f.dla_dx + (T)2 * gk[2]);
  acc.add(QS_G_DY, ga * f.dla_dy + (T)2 * gk[3]);
  acc.add(QS_G_DELAY, ga * f.dla_del - cc * gk[4]);
  if (!p.flat && !f.clamped) {
    acc.add(QS_G_GAMMA, g_g0 * ((T)1 + QS_PV(T, spread) * f.xi3));
    acc.add(QS_G_SPREAD, g_g0 * QS_PV(T, gmean) * f.xi3);
  }
  acc.add(QS_G_DIV, (go.g_thx + ga * f.dla_thx) * f.xi4 + (go.g_thy + ga * f.dla_thy) * f.xi5 -
                        (T)2 * gk[5]);
}

// Upstream coefficients from the forward moments and dL/d(moments):
// rel_spread = spread/mean and div = sqrt(div_x^2 + div_y^2) folded into
// mean, spread, div_x, div_y.  Formed once (a dozen FP64 divisions), written
// as kSeeds doubles, rounded to the path's type by those who read them.
constexpr int kSeeds = 11;
__device__ __forceinline__ void write_seeds(const qs_moments* __restrict__ mom,
                                            const double* __restrict__ dLdm, double* o) {
  const double W = mom->W, mean = mom->mean, spread = mom->spread;
  const double Dx = mom->div_x, Dy = mom->div_y, D = mom->div;
  const double d1 = dLdm[1], d2 = dLdm[2], d3 = dLdm[3], d4 = dLdm[4], d5 = dLdm[5],
               d6 = dLdm[6];
  o[0] = W > 0.0 ? 1.0 / W : 0.0;
  o[1] = mean;
  o[2] = spread;
  o[3] = Dx > 0.0 ? 1.0 / Dx : 0.0;
  o[4] = Dy > 0.0 ? 1.0 / Dy : 0.0;
  o[5] = d1 - (mean != 0.0 ? d3 * spread / (mean * mean) : 0.0);
  o[6] = d2 + (mean != 0.0 ? d3 / mean : 0.0);
  o[7] = d4 + (D > 0.0 ? d6 * Dx / D : 0.0);
  o[8] = d5 + (D > 0.0 ? d6 * Dy / D : 0.0);
  o[9] = dLdm[7];
  o[10] = dLdm[11];
}
template <typename T>
__device__ __forceinline__ Seeds<T> load_seeds(const double* o) {
  return Seeds<T>{(T)o[0], (T)o[1], (T)o[2], (T)o[3], (T)o[4], (T)o[5],
                  (T)o[6], (T)o[7], (T)o[8], (T)o[9], (T)o[10]};
}

// The index of a sample as a value the compiler knows nothing about: what is
// loaded and decoded from it after the cell loop is then loaded and decoded
// again, instead of being held in registers across the loop.
__device__ __forceinline__ int64_t fresh(int64_t i) {
  asm volatile("" : "+l"(i));
  return i;
}

// One pair of samples (FP32; i1 == i0: one sample) through the integration
// with tangents and the chain rule.
template <bool QFP, typename S, int VAR>
__device__ __forceinline__ void grad_pair(const Params& p, const float4* __restrict__ tab,
                                          const Seeds<float>& sd, const S* dS, float w0,
                                          GAcc<float>& acc, int64_t i0, int64_t i1,
                                          const float4* __restrict__ cA) {
  GFront<float> f0, f1;
  grad_front<float>(p, i0, w0, f0);
  grad_front<float>(p, i1, w0, f1);
  const float2 ig0 = make_float2(__frcp_rn(f0.gamma0), __frcp_rn(f1.gamma0));
  if constexpr ((VAR & kVarCell) != 0) {
    const FocPath<float2> fp{make_float2(f0.zq, f1.zq),   make_float2(f0.xs, f1.xs),
                             make_float2(f0.ys, f1.ys),   make_float2(f0.thx, f1.thx),
                             make_float2(f0.thy, f1.thy), make_float2(f0.xi4, f1.xi4),
                             make_float2(f0.xi5, f1.xi5), make_float2(f0.ct, f1.ct)};
    FocTanX<float2> x;
    focus_tangent<float2, QFP, VAR>(p, tab, fp, ig0, x, cA);
    FocTan<float> o;
    auto lane = [&](bool y) {
      o.du = y ? x.du.y : x.du.x;
      o.V = y ? x.V.y : x.V.x;
#pragma unroll
      for (int k = 0; k < kNT; ++k) {
        o.du_t[k] = y ? x.du_t[k].y : x.du_t[k].x;
        o.V_t[k] = y ? x.V_t[k].y : x.V_t[k].x;
      }
    };
    lane(false);
    i0 = fresh(i0);
    grad_front<float>(p, i0, w0, f0);
    if (f0.ok) grad_back_focus<float, QFP, S>(p, sd, dS, i0, f0, o, acc);
    if (i1 != i0) {
      lane(true);
      i1 = fresh(i1);
      grad_front<float>(p, i1, w0, f1);
      if (f1.ok) grad_back_focus<float, QFP, S>(p, sd, dS, i1, f1, o, acc);
    }
  } else {
    float2 du{}, V{}, du_l{}, V_l{}, u{}, V_u{};
    if constexpr (QFP)
      qfp_tangent<float2, VAR>(p, tab, make_float2(f0.a, f1.a), ig0, du, V, du_l, V_l, u, V_u, cA);
    i0 = fresh(i0);
    grad_front<float>(p, i0, w0, f0);
    if (f0.ok)
      grad_back<float, QFP, S>(p, sd, dS, i0, f0,
                               QfpTan<float>{du.x, V.x, du_l.x, V_l.x, u.x, V_u.x}, acc);
    if (i1 != i0) {
      i1 = fresh(i1);
      grad_front<float>(p, i1, w0, f1);
      if (f1.ok)
        grad_back<float, QFP, S>(p, sd, dS, i1, f1,
                                 QfpTan<float>{du.y, V.y, du_l.y, V_l.y, u.y, V_u.y}, acc);
    }
  }
}

// Samples [begin, end) of one launch's samples, thread `tid` of `nthr`: the
// FP32 models with phase cells take two samples per thread through the
// packed tangent integration (begin even), the other paths one.
template <typename T, bool QFP, typename S, int VAR = 0>
__device__ __forceinline__ void grad_range(const Params& p,
                                           const typename Tab<T>::type* __restrict__ tab,
                                           const Seeds<T>& sd, const S* dS, T w0, GAcc<T>& acc,
                                           int64_t begin, int64_t end, int64_t tid,
                                           int64_t nthr, const float4* __restrict__ cA = nullptr) {
  if constexpr (sizeof(T) == 4 && (QFP || (VAR & kVarCell))) {
    for (int64_t k = begin / 2 + tid; 2 * k < end; k += nthr)
      grad_pair<QFP, S, VAR>(p, tab, sd, dS, w0, acc, 2 * k, (2 * k + 1 < end) ? 2 * k + 1 : 2 * k,
                             cA);
  } else {
    for (int64_t i = begin + tid; i < end; i += nthr) {
      GFront<T> f;
      grad_front<T>(p, i, w0, f);
      if (!f.ok) continue;
      if constexpr ((VAR & kVarCell) != 0) {
        const FocPath<T> fp{f.zq, f.xs, f.ys, f.thx, f.thy, f.xi4, f.xi5, f.ct};
        FocTanX<T> x;
        focus_tangent<T, QFP, VAR>(p, tab, fp, (T)1 / f.gamma0, x, cA);
        FocTan<T> o;
        o.du = x.du;
        o.V = x.V;
#pragma unroll
        for (int k = 0; k < kNT; ++k) {
          o.du_t[k] = x.du_t[k];
          o.V_t[k] = x.V_t[k];
        }
        grad_back_focus<T, QFP, S>(p, sd, dS, i, f, o, acc);
      } else {
        QfpTan<T> o{};
        if constexpr (QFP)
          qfp_tangent<T, VAR>(p, tab, f.a, (T)1 / f.gamma0, o.du, o.V, o.du_l, o.V_l, o.u, o.V_u,
                              cA);
        grad_back<T, QFP, S>(p, sd, dS, i, f, o, acc);
      }
    }
  }
}

// Registers per thread of the adjoint kernels and, from them, the block size
// when the caller leaves it open (FP32: one CTA that fills the register
// file; CTAs that share an SM are served oldest first and finish far apart).
// 2^22 samples x 512 cells, us, for the registers tried (warps per SM):
//   two tangents      72 (28) 5004, 80 (24) 4985, 96 (20) 5050, 128 (16) 5022
//   cycle-resolved    80 (24) 5061, 96 (20) 4813, 104 (16) 4956
//   seven tangents    112 (16) 9822, 128 (16) 9827, 168 (12) 9530
// The two-tangent kernel takes 16 warps: the same rate, and a CTA's step of
// 1024 samples divides the batched adjoint's tiles.  Seven tangents take 128
// (2^17 samples: 416 us against 427 with 168).
constexpr int grad_regs(bool f64, int var) {
  return f64 ? (var ? 255 : 128) : ((var & kVarCell) ? 128 : (var ? 96 : 128));
}
constexpr int grad_block(bool f64, int var) {
  return f64 ? 256 : ((65536 / (grad_regs(f64, var) * 32)) & ~3) * 32;
}

// Fixed-order block reduction of the per-thread gradient partials into
// out[0..kNumGrad): one warp tree for the eight sums together, then warps in
// order.  red holds (blockDim.x / 32) * kNumGrad doubles; the caller
// synchronises before red is reused.
template <typename T>
__device__ __forceinline__ void grad_block_reduce(const GAcc<T>& acc, double* red, double* out) {
  static_assert(kNumGrad == 8, "warp_sum8 carries eight fields");
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  double f[8];
#pragma unroll
  for (int k = 0; k < 8; ++k) f[k] = acc.get(k);
  const double v = warp_sum8(f);
  if ((lane & 3) == 0)
    red[warp * kNumGrad + 4 * ((lane >> 4) & 1) + 2 * ((lane >> 3) & 1) + ((lane >> 2) & 1)] = v;
  __syncthreads();
  if (threadIdx.x < kNumGrad) {
    double s = 0.0;
    for (int wv = 0; wv < (int)(blockDim.x >> 5); ++wv) s += red[wv * kNumGrad + threadIdx.x];
    out[threadIdx.x] = s;
  }
}

}  // namespace qs
