// FP32 physics with two values per float2: the packed FP32x2 instructions of
// sm_100+ (__ffma2_rn, __fadd2_rn, __fmul2_rn) work on two primitive variables of
// a cell (limited face states) or on the two sides of a face (Riemann flux).
// The fused FP32 kernels are bound by instruction issue, so whatever can be
// packed is; selects, minima, roots and reciprocals are per lane.  Formulas,
// region rules and thresholds are those of physics.cuh; only the grouping of
// operations differs (FP32 rounding level).
#pragma once

#include "physics.cuh"

namespace amrvac {

__device__ __forceinline__ float2 sp2(float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
// a - b as one packed FMA with -1 (exact: one rounding)
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __ffma2_rn(b, sp2(-1.f), a); }
__device__ __forceinline__ float2 neg2(float2 a) { return mul2(a, sp2(-1.f)); }
__device__ __forceinline__ float2 rcp2(float2 a) { return make_float2(1.f / a.x, 1.f / a.y); }
__device__ __forceinline__ float2 sqrt2(float2 a) { return make_float2(sqrtf(a.x), sqrtf(a.y)); }
__device__ __forceinline__ float2 min2(float2 a, float2 b) {
  return make_float2(fminf(a.x, b.x), fminf(a.y, b.y));
}
__device__ __forceinline__ float2 max2(float2 a, float2 b) {
  return make_float2(fmaxf(a.x, b.x), fmaxf(a.y, b.y));
}
__device__ __forceinline__ float2 abs2(float2 a) { return make_float2(fabsf(a.x), fabsf(a.y)); }
__device__ __forceinline__ float2 sel2(bool px, bool py, float2 a, float2 b) {
  return make_float2(px ? a.x : b.x, py ? a.y : b.y);
}

// ---------------------------------------------------------------- limiters

// parameters of the runtime symmetric limiters, slope = sgn(dp) min(beta mn,
// c1 mx + c2 mn) with mn, mx the smaller and larger of |dm|, |dp|: superbee
// (2, 1, 0), woodward (2, 1/2, 1/2), mcbeta (1.4, 1/2, 1/2)
struct SymLim {
  float beta, c1, c2;
};
__device__ __forceinline__ SymLim sym_lim(int lim) {
  if (lim == AMRVAC_LIM_SUPERBEE) return {2.f, 1.f, 0.f};
  return {lim == AMRVAC_LIM_WOODWARD ? 2.f : 1.4f, 0.5f, 0.5f};
}

// Increments of two variables with cell values b and neighbours a (i-1) and c
// (i+1): the face values are b - lo at i-1/2 and b + hi at i+1/2, from one slope
// evaluation.
// LIM: MINMOD, VANLEER, KOREN; -1 the symmetric family by sl; -3 albada, cada3
// or venk by the runtime value lim.
template <int LIM>
__device__ __forceinline__ void cell_increments2(float2 a, float2 b, float2 c, int lim, SymLim sl,
                                                 float2& lo, float2& hi) {
  const float2 dm = sub2(b, a), dp = sub2(c, b);
  if constexpr (LIM == -3) {
    if (lim == AMRVAC_LIM_CADA3) {
      hi = make_float2(cada3_half(dm.x, dp.x), cada3_half(dm.y, dp.y));
      lo = make_float2(cada3_half(dp.x, dm.x), cada3_half(dp.y, dm.y));
      return;
    }
    if (lim == AMRVAC_LIM_VENK) {
      lo = hi = make_float2(venk_increment(a.x, b.x, c.x), venk_increment(a.y, b.y, c.y));
      return;
    }
  }
  const float2 prod = mul2(dm, dp);
  const bool px = prod.x > 0.f, py = prod.y > 0.f;
  if constexpr (LIM == AMRVAC_LIM_KOREN) {
    // halves: min(|dm|, |dp|, (|dm| + 2 |dp|)/6) towards i+1/2, mirrored to i-1/2
    const float2 am = abs2(dm), ap = abs2(dp), m = min2(am, ap);
    const float2 k6 = sp2(1.f / 6.f);
    const float2 h = min2(m, mul2(fma2(sp2(2.f), ap, am), k6));
    const float2 l = min2(m, mul2(fma2(sp2(2.f), am, ap), k6));
    hi = make_float2(px ? copysignf(h.x, dp.x) : 0.f, py ? copysignf(h.y, dp.y) : 0.f);
    lo = make_float2(px ? copysignf(l.x, dp.x) : 0.f, py ? copysignf(l.y, dp.y) : 0.f);
  } else {
    float2 s;
    if constexpr (LIM == AMRVAC_LIM_VANLEER) {
      s = mul2(prod, rcp2(sub2(c, a)));  // dm dp / (dm + dp): half the slope
    } else if constexpr (LIM == -3) {    // albada
      const float2 den = fma2(dm, dm, mul2(dp, dp));
      s = mul2(mul2(prod, mul2(sp2(0.5f), add2(dm, dp))), rcp2(den));
    } else {
      const float2 am = abs2(dm), ap = abs2(dp);
      const float2 mn = min2(am, ap);
      float2 g;
      if constexpr (LIM == AMRVAC_LIM_MINMOD) g = mul2(sp2(0.5f), mn);
      else g = min2(mul2(sp2(0.5f * sl.beta), mn),
                    fma2(sp2(0.5f * sl.c1), max2(am, ap), mul2(sp2(0.5f * sl.c2), mn)));
      s = make_float2(copysignf(g.x, dp.x), copysignf(g.y, dp.y));
    }
    lo = hi = sel2(px, py, s, sp2(0.f));
  }
}

// local component c of a y face -> primitive variable (normal y, tangential
// (z, x)); an x face uses the identity
__device__ __forceinline__ constexpr int yface_var(int c) {
  return c == 1 ? 2 : c == 2 ? 3 : c == 3 ? 1 : c == 5 ? 6 : c == 6 ? 7 : c == 7 ? 5 : c;
}

// ---------------------------------------------------------------- Riemann
// one face, its left and right states in the lanes

// squares of the fast speeds of both sides; bt = B_t^2, bx2 = B_n^2
__device__ __forceinline__ float2 fast2(float g, float2 rho, float2 p, float2 bt, float bx2) {
  float2 ir = rcp2(rho);
  float2 a2 = mul2(mul2(sp2(g), p), ir);
  float2 bt2 = mul2(bt, ir);
  float2 bb = mul2(add2(sp2(bx2), bt), ir);
  float2 dd = sub2(a2, bb);
  float2 sq = sqrt2(fma2(dd, dd, mul2(mul2(sp2(4.f), a2), bt2)));
  return mul2(sp2(0.5f), add2(add2(a2, bb), sq));
}

// local frame pairs: rho, u, v, w, p, by, bz (x = left, y = right); bx shared
struct Side2 {
  float2 rho, u, v, w, p, by, bz;
};

// total pressure and total energy of both sides; bt = B_t^2 of both sides
__device__ __forceinline__ void pt_e2(const Side2& q, float bx2, float ig1, float2& pt,
                                      float2& e, float2& bt) {
  bt = fma2(q.bz, q.bz, mul2(q.by, q.by));
  float2 b2 = add2(bt, sp2(bx2));
  pt = fma2(b2, sp2(0.5f), q.p);
  float2 uu = fma2(q.w, q.w, fma2(q.v, q.v, mul2(q.u, q.u)));
  e = fma2(q.p, sp2(ig1), fma2(mul2(sp2(0.5f), q.rho), uu, mul2(sp2(0.5f), b2)));
}

// physical flux and conserved state of one side (scalar)
__device__ __forceinline__ void side_flux(float rho, float u, float v, float w, float by,
                                          float bz, float bx, float pt, float e, float* U,
                                          float* F) {
  float mu = rho * u;
  U[0] = rho;
  U[1] = mu;
  U[2] = rho * v;
  U[3] = rho * w;
  U[4] = e;
  U[5] = bx;
  U[6] = by;
  U[7] = bz;
  F[0] = mu;
  F[1] = mu * u + pt - bx * bx;
  F[2] = mu * v - bx * by;
  F[3] = mu * w - bx * bz;
  F[4] = (e + pt) * u - bx * (u * bx + v * by + w * bz);
  F[5] = 0.f;
  F[6] = by * u - bx * v;
  F[7] = bz * u - bx * w;
}

__device__ __forceinline__ void hll_pair(float g, float ig1, const Side2& q, float bx, float* f) {
  const float bx2 = bx * bx;
  float2 pt, e, bt;
  pt_e2(q, bx2, ig1, pt, e, bt);
  float2 cf = sqrt2(fast2(g, q.rho, q.p, bt, bx2));
  float sl = fminf(q.u.x - cf.x, q.u.y - cf.y);
  float sr = fmaxf(q.u.x + cf.x, q.u.y + cf.y);
  float UL[8], FL[8], UR[8], FR[8];
  side_flux(q.rho.x, q.u.x, q.v.x, q.w.x, q.by.x, q.bz.x, bx, pt.x, e.x, UL, FL);
  side_flux(q.rho.y, q.u.y, q.v.y, q.w.y, q.by.y, q.bz.y, bx, pt.y, e.y, UR, FR);
  const float inv = 1.f / (sr - sl);
  const float2 srsl = make_float2(sr, -sl);
  const float slsr = sl * sr;
#pragma unroll
  for (int c = 0; c < 8; c += 2) {
    // (sr FL - sl FR + sl sr (UR - UL)) / (sr - sl) for components c, c+1
    float2 fl = make_float2(FL[c], FL[c + 1]), fr = make_float2(FR[c], FR[c + 1]);
    float2 ul = make_float2(UL[c], UL[c + 1]), ur = make_float2(UR[c], UR[c + 1]);
    float2 t = fma2(sp2(srsl.x), fl, mul2(sp2(srsl.y), fr));
    t = mul2(fma2(sp2(slsr), sub2(ur, ul), t), sp2(inv));
    f[c] = sl >= 0.f ? FL[c] : (sr <= 0.f ? FR[c] : t.x);
    f[c + 1] = sl >= 0.f ? FL[c + 1] : (sr <= 0.f ? FR[c + 1] : t.y);
  }
}

// TVD Lax-Friedrichs with both sides' physical fluxes in packed lanes
__device__ __forceinline__ void tvdlf_pair(float g, float ig1, const Side2& q, float bx,
                                           float* f) {
  const float bx2 = bx * bx;
  float2 pt, e, bt;
  pt_e2(q, bx2, ig1, pt, e, bt);
  const float2 cf = sqrt2(fast2(g, q.rho, q.p, bt, bx2));
  const float cmax = fmaxf(fabsf(q.u.x) + cf.x, fabsf(q.u.y) + cf.y);
  float UL[8], FL[8], UR[8], FR[8];
  side_flux(q.rho.x, q.u.x, q.v.x, q.w.x, q.by.x, q.bz.x, bx, pt.x, e.x, UL, FL);
  side_flux(q.rho.y, q.u.y, q.v.y, q.w.y, q.by.y, q.bz.y, bx, pt.y, e.y, UR, FR);
#pragma unroll
  for (int c = 0; c < 8; c += 2) {
    const float2 fl = make_float2(FL[c], FL[c + 1]), fr = make_float2(FR[c], FR[c + 1]);
    const float2 ul = make_float2(UL[c], UL[c + 1]), ur = make_float2(UR[c], UR[c + 1]);
    const float2 t = fma2(sp2(-0.5f * cmax), sub2(ur, ul), mul2(sp2(0.5f), add2(fl, fr)));
    f[c] = t.x;
    f[c + 1] = t.y;
  }
}

// HLLD (MK05).  Up to the single-star states the two sides share the lanes; from
// there on the lanes are the tangential components (v, w) and (By, Bz) of one
// side: the degeneracy selects write that layout, so that no register has to be
// moved to change it.
__device__ __forceinline__ void hlld_pair(float g, float ig1, const Side2& q, float bx, float* f) {
  const float bx2 = bx * bx;
  const float2 bxp = sp2(bx), bx2p = sp2(bx2);
  const float2 bt = fma2(q.bz, q.bz, mul2(q.by, q.by));
  const float2 b2 = add2(bt, bx2p);
  const float2 hb = mul2(b2, sp2(0.5f));
  const float2 pt = add2(q.p, hb);
  const float2 uu = fma2(q.w, q.w, fma2(q.v, q.v, mul2(q.u, q.u)));
  const float2 e = fma2(q.p, sp2(ig1), fma2(mul2(sp2(0.5f), q.rho), uu, hb));
  // fast speeds (see local_fast2); one root for both sides: the larger square
  const float2 ir = rcp2(q.rho);
  const float2 a2 = mul2(mul2(sp2(g), q.p), ir), bb = mul2(b2, ir);
  const float2 dd = sub2(a2, bb);
  const float2 rad = fma2(dd, dd, mul2(mul2(sp2(4.f), a2), mul2(bt, ir)));
  const float2 cf2 = add2(add2(a2, bb), sqrt2(rad));
  const float cmax = sqrtf(0.5f * fmaxf(cf2.x, cf2.y));
  const float sl = fminf(q.u.x, q.u.y) - cmax;
  const float sr = fmaxf(q.u.x, q.u.y) + cmax;
  const float2 S = make_float2(sl, sr);
  const float2 su = sub2(S, q.u);              // (S_L - u_L, S_R - u_R)
  const float2 A = mul2(su, q.rho);            // rho (S - u)
  const float iden = 1.f / (A.y - A.x);
  const float sm = ((A.y * q.u.y + pt.x) - (A.x * q.u.x + pt.y)) * iden;
  const float pts = ((A.y * pt.x - A.x * pt.y) + A.x * A.y * (q.u.y - q.u.x)) * iden;
  const float psm = pts * sm, sbx = sm * bx;
  // single-star states of both sides
  const float2 smp = sp2(sm);
  const float2 ssm = sub2(S, smp);             // S - S_M
  const float2 isd = rcp2(ssm);
  const float2 rs = mul2(A, isd);
  const float2 big = mul2(A, ssm);
  const float2 den = sub2(big, bx2p);
  const float2 iden2 = rcp2(den);
  const float2 ntv = mul2(mul2(bxp, sub2(q.u, smp)), iden2);
  const float2 tb = mul2(sub2(mul2(A, su), bx2p), iden2);
  const float2 vs = fma2(q.by, ntv, q.v), ws = fma2(q.bz, ntv, q.w);
  const float2 bys = mul2(q.by, tb), bzs = mul2(q.bz, tb);
  const float eps = Num<float>::hlld_eps;
  const bool dl = fabsf(den.x) <= eps * fmaxf(fabsf(big.x), bx2);
  const bool dr = fabsf(den.y) <= eps * fmaxf(fabsf(big.y), bx2);
  const float2 VL = make_float2(dl ? q.v.x : vs.x, dl ? q.w.x : ws.x);
  const float2 VR = make_float2(dr ? q.v.y : vs.y, dr ? q.w.y : ws.y);
  const float2 BL = make_float2(dl ? q.by.x : bys.x, dl ? q.bz.x : bzs.x);
  const float2 BR = make_float2(dr ? q.by.y : bys.y, dr ? q.bz.y : bzs.y);
  const float2 vb = fma2(q.w, q.bz, fma2(q.v, q.by, mul2(q.u, bxp)));
  const float2 vbl = mul2(VL, BL), vbr = mul2(VR, BR);
  const float2 vbs = make_float2(sbx + (vbl.x + vbl.y), sbx + (vbr.x + vbr.y));
  const float2 t = sub2(mul2(su, e), mul2(pt, q.u));
  const float2 es = mul2(fma2(bxp, sub2(vb, vbs), add2(t, sp2(psm))), isd);
  // double-star states (averages of the two sides)
  const float isl = rsqrtf(rs.x), isr = rsqrtf(rs.y);  // 1/sqrt(rho*)
  const float sql = rs.x * isl, sqr = rs.y * isr;
  const float abx = fabsf(bx);
  const float ssl = sm - abx * isl, ssr = sm + abx * isr;
  const float sb = bx == 0.f ? 0.f : copysignf(1.f, bx);
  const float issum = 1.f / (sql + sqr);
  const float wl = sql * issum, wr = sqr * issum;
  const float2 wlp = sp2(wl), wrp = sp2(wr);
  const float2 VSS = fma2(sub2(BR, BL), sp2(sb * issum), fma2(wrp, VR, mul2(wlp, VL)));
  const float2 BSS = fma2(sub2(VR, VL), sp2(sql * wr * sb), fma2(wrp, BL, mul2(wlp, BR)));
  const float2 vbd = mul2(VSS, BSS);
  const float vbss = sbx + (vbd.x + vbd.y);
  // region containing x/t = 0 (same tie rules as the scalar solver)
  const bool left = sm >= 0.f;
  const bool outer = left ? (sl > 0.f) : (sr < 0.f);
  const bool single = left ? (ssl >= 0.f) : !(ssr >= 0.f);
  // the upwind side of S_M
  const float rho = left ? q.rho.x : q.rho.y, u = left ? q.u.x : q.u.y;
  const float pu = left ? pt.x : pt.y, eu = left ? e.x : e.y;
  const float r = left ? rs.x : rs.y, eS = left ? es.x : es.y, vbS = left ? vbs.x : vbs.y;
  const float vbu = left ? vb.x : vb.y, sq = left ? -sql : sqr;
  const float c1 = left ? sl : sr, c2 = left ? ssl : ssr;
  const float2 V = make_float2(left ? q.v.x : q.v.y, left ? q.w.x : q.w.y);
  const float2 B = make_float2(left ? q.by.x : q.by.y, left ? q.bz.x : q.bz.y);
  const float2 VS = make_float2(left ? VL.x : VR.x, left ? VL.y : VR.y);
  const float2 BS = make_float2(left ? BL.x : BR.x, left ? BL.y : BR.y);
  // F + c1 (U* - U) + c2 (U** - U*); the double star keeps rho* and S_M, and
  // e** - e* = -/+ sqrt(rho*) (v*.B* - v**.B**) sgn(Bx)
  const float mu = rho * u;
  const float F1 = mu * u + (pu - bx2), F4 = (eu + pu) * u - bx * vbu;
  const float2 F23 = sub2(mul2(sp2(mu), V), mul2(bxp, B));
  const float2 F67 = sub2(mul2(sp2(u), B), mul2(bxp, V));
  const float2 c1p = sp2(c1);
  const float2 fs23 = fma2(c1p, sub2(mul2(sp2(r), VS), mul2(sp2(rho), V)), F23);
  const float2 fs67 = fma2(c1p, sub2(BS, B), F67);
  const float fs4 = F4 + c1 * (eS - eu);
  const float fss4 = fs4 + c2 * ((sq * sb) * (vbS - vbss));
  const float2 fss23 = fma2(sp2(c2 * r), sub2(VSS, VS), fs23);
  const float2 fss67 = fma2(sp2(c2), sub2(BSS, BS), fs67);
  f[0] = outer ? mu : mu + c1 * (r - rho);
  f[1] = outer ? F1 : F1 + c1 * (r * sm - mu);
  f[2] = outer ? F23.x : (single ? fs23.x : fss23.x);
  f[3] = outer ? F23.y : (single ? fs23.y : fss23.y);
  f[4] = outer ? F4 : (single ? fs4 : fss4);
  f[5] = 0.f;
  f[6] = outer ? F67.x : (single ? fs67.x : fss67.x);
  f[7] = outer ? F67.y : (single ? fs67.y : fss67.y);
}

// constants of a face flux: gamma, 1/(gamma - 1), c_h, 1/(2 c_h)
struct FaceConst2 {
  float g, ig1, ch, hich;
  int glm;
};
__device__ __forceinline__ FaceConst2 face_const2(float g, float ch, int glm) {
  return {g, 1.f / (g - 1.f), ch, 0.5f / ch, glm};
}

// glm solve and Riemann flux along D from the face states w[v] = (left, right)
template <int D, int FLUX>
__device__ __forceinline__ void face_flux2(const float2* w, const FaceConst2& fc, float* f) {
  constexpr int t1 = D == 2 ? 0 : D + 1, t2 = D == 0 ? 2 : D - 1;
  const float bnl = w[5 + D].x, bnr = w[5 + D].y;
  float bns = 0.5f * (bnl + bnr), psis = 0.f, fpsi = 0.f;
  if (fc.glm) {
    bns = fmaf(w[8].x - w[8].y, fc.hich, bns);
    psis = fmaf(bnl - bnr, 0.5f * fc.ch, 0.5f * (w[8].x + w[8].y));
    fpsi = fc.ch * fc.ch * bns;
  }
  const Side2 q = {w[0], w[1 + D], w[1 + t1], w[1 + t2], w[4], w[5 + t1], w[5 + t2]};
  float fl[8];
  if constexpr (FLUX == AMRVAC_FLUX_HLL) {
    hll_pair(fc.g, fc.ig1, q, bns, fl);
  } else if constexpr (FLUX == AMRVAC_FLUX_HLLD) {
    hlld_pair(fc.g, fc.ig1, q, bns, fl);
  } else if constexpr (FLUX == AMRVAC_FLUX_TVDLF) {
    tvdlf_pair(fc.g, fc.ig1, q, bns, fl);
  } else {
    // HLLC: the scalar three-wave solver on the unpacked face states
    const float ql[8] = {q.rho.x, q.u.x, q.v.x, q.w.x, q.p.x, bns, q.by.x, q.bz.x};
    const float qr[8] = {q.rho.y, q.u.y, q.v.y, q.w.y, q.p.y, bns, q.by.y, q.bz.y};
    hllc_local<float>(fc.g, fc.ig1, ql, qr, bns, fl);
  }
  f[0] = fl[0];
  f[1 + D] = fl[1];
  f[1 + t1] = fl[2];
  f[1 + t2] = fl[3];
  f[4] = fl[4];
  f[5 + D] = psis;
  f[5 + t1] = fl[6];
  f[5 + t2] = fl[7];
  f[8] = fpsi;
}

// a face state is not positive (or NaN): the face takes the cell values
__device__ __forceinline__ bool not_positive2(const float2* w) {
  return !(w[0].x > 0.f) || !(w[4].x > 0.f) || !(w[0].y > 0.f) || !(w[4].y > 0.f);
}

// ---------------------------------------------------------------- Riemann, two faces
// lane x the x face of a cell and lane y its y face, each in its local frame
// (normal velocity and field first): every operation is packed, and the solver's
// latency is paid once for both faces

struct Prim2 {
  float2 rho, u, v, w, p, by, bz;
};

// squares of the fast speeds (cancellation-free form) from rho, p, B_t^2, B_n^2
__device__ __forceinline__ float2 fast_xy(float g, float2 rho, float2 p, float2 bt, float2 bx2) {
  const float2 ir = rcp2(rho);
  const float2 a2 = mul2(mul2(sp2(g), p), ir);
  const float2 bt2 = mul2(bt, ir);
  const float2 bb = mul2(add2(bx2, bt), ir);
  const float2 dd = sub2(a2, bb);
  const float2 sq = sqrt2(fma2(dd, dd, mul2(mul2(sp2(4.f), a2), bt2)));
  return mul2(sp2(0.5f), add2(add2(a2, bb), sq));
}

// B_t^2, total pressure and total energy
__device__ __forceinline__ void pt_e_xy(const Prim2& q, float2 bx2, float ig1, float2& bt,
                                      float2& pt, float2& e) {
  bt = fma2(q.bz, q.bz, mul2(q.by, q.by));
  const float2 b2 = add2(bt, bx2);
  pt = fma2(b2, sp2(0.5f), q.p);
  const float2 uu = fma2(q.w, q.w, fma2(q.v, q.v, mul2(q.u, q.u)));
  e = fma2(q.p, sp2(ig1), fma2(mul2(sp2(0.5f), q.rho), uu, mul2(sp2(0.5f), b2)));
}

// conserved state and physical flux (component 5, the normal field, is left to
// the glm solve)
__device__ __forceinline__ void state_flux2(const Prim2& q, float2 bx, float2 bx2, float2 pt,
                                            float2 e, float2* U, float2* F) {
  const float2 mu = mul2(q.rho, q.u), nbx = neg2(bx);
  const float2 vb = fma2(q.w, q.bz, fma2(q.v, q.by, mul2(q.u, bx)));
  U[0] = q.rho;
  U[1] = mu;
  U[2] = mul2(q.rho, q.v);
  U[3] = mul2(q.rho, q.w);
  U[4] = e;
  U[5] = bx;
  U[6] = q.by;
  U[7] = q.bz;
  F[0] = mu;
  F[1] = fma2(mu, q.u, sub2(pt, bx2));
  F[2] = fma2(mu, q.v, mul2(nbx, q.by));
  F[3] = fma2(mu, q.w, mul2(nbx, q.bz));
  F[4] = fma2(add2(e, pt), q.u, mul2(nbx, vb));
  F[5] = sp2(0.f);
  F[6] = fma2(q.by, q.u, mul2(nbx, q.v));
  F[7] = fma2(q.bz, q.u, mul2(nbx, q.w));
}

// HLL and TVD Lax-Friedrichs
template <int FLUX>
__device__ __forceinline__ void hll2(float g, float ig1, const Prim2& L, const Prim2& R,
                                     float2 bx, float2* f) {
  const float2 bx2 = mul2(bx, bx);
  float2 btL, ptL, eL, btR, ptR, eR, UL[8], FL[8], UR[8], FR[8];
  pt_e_xy(L, bx2, ig1, btL, ptL, eL);
  pt_e_xy(R, bx2, ig1, btR, ptR, eR);
  const float2 cL = sqrt2(fast_xy(g, L.rho, L.p, btL, bx2));
  const float2 cR = sqrt2(fast_xy(g, R.rho, R.p, btR, bx2));
  state_flux2(L, bx, bx2, ptL, eL, UL, FL);
  state_flux2(R, bx, bx2, ptR, eR, UR, FR);
  if (FLUX == AMRVAC_FLUX_TVDLF) {
    const float2 c = mul2(sp2(-0.5f), max2(add2(abs2(L.u), cL), add2(abs2(R.u), cR)));
#pragma unroll
    for (int k = 0; k < 8; k++)
      f[k] = fma2(c, sub2(UR[k], UL[k]), mul2(sp2(0.5f), add2(FL[k], FR[k])));
    return;
  }
  const float2 sl = min2(sub2(L.u, cL), sub2(R.u, cR)), sr = max2(add2(L.u, cL), add2(R.u, cR));
  const float2 inv = rcp2(sub2(sr, sl)), nsl = neg2(sl), slsr = mul2(sl, sr);
  const bool lx = sl.x >= 0.f, ly = sl.y >= 0.f, rx = sr.x <= 0.f, ry = sr.y <= 0.f;
#pragma unroll
  for (int k = 0; k < 8; k++) {
    if (k == 5) continue;
    const float2 t = fma2(sr, FL[k], mul2(nsl, FR[k]));
    const float2 m = mul2(fma2(slsr, sub2(UR[k], UL[k]), t), inv);
    f[k] = sel2(lx, ly, FL[k], sel2(rx, ry, FR[k], m));
  }
  f[5] = sp2(0.f);
}

// HLLC (see hllc_local)
__device__ __forceinline__ void hllc2(float g, float ig1, const Prim2& L, const Prim2& R,
                                      float2 bx, float2* f) {
  const float2 bx2 = mul2(bx, bx);
  float2 btL, ptL, eL, btR, ptR, eR, UL[8], FL[8], UR[8], FR[8];
  pt_e_xy(L, bx2, ig1, btL, ptL, eL);
  pt_e_xy(R, bx2, ig1, btR, ptR, eR);
  const float2 cL = sqrt2(fast_xy(g, L.rho, L.p, btL, bx2));
  const float2 cR = sqrt2(fast_xy(g, R.rho, R.p, btR, bx2));
  state_flux2(L, bx, bx2, ptL, eL, UL, FL);
  state_flux2(R, bx, bx2, ptR, eR, UR, FR);
  const float2 sl = min2(sub2(L.u, cL), sub2(R.u, cR)), sr = max2(add2(L.u, cL), add2(R.u, cR));
  const float2 inv = rcp2(sub2(sr, sl)), nsl = neg2(sl);
  float2 uh[8];
#pragma unroll
  for (int k = 0; k < 8; k++)
    uh[k] = mul2(add2(fma2(sr, UR[k], mul2(nsl, UL[k])), sub2(FL[k], FR[k])), inv);
  const float2 ih = rcp2(uh[0]);
  const float2 sm = mul2(uh[1], ih), vy = mul2(uh[2], ih), vz = mul2(uh[3], ih);
  const float2 by = uh[6], bz = uh[7];
  const float2 pts =
      fma2(mul2(L.rho, sub2(sl, L.u)), sub2(sm, L.u), ptL);
  const float2 vbs = fma2(vz, bz, fma2(vy, by, mul2(sm, bx)));
  const bool lx = sm.x >= 0.f, ly = sm.y >= 0.f;
  const Prim2 q = {sel2(lx, ly, L.rho, R.rho), sel2(lx, ly, L.u, R.u), sel2(lx, ly, L.v, R.v),
                   sel2(lx, ly, L.w, R.w),     sel2(lx, ly, L.p, R.p), sel2(lx, ly, L.by, R.by),
                   sel2(lx, ly, L.bz, R.bz)};
  const float2 S = sel2(lx, ly, sl, sr), pt = sel2(lx, ly, ptL, ptR), e = sel2(lx, ly, eL, eR);
  const float2 su = sub2(S, q.u), isd = rcp2(sub2(S, sm));
  const float2 vb = fma2(q.w, q.bz, fma2(q.v, q.by, mul2(q.u, bx)));
  const float2 nbx = neg2(bx);
  float2 Us[8];
  const float2 ru = mul2(q.rho, su);
  Us[0] = mul2(ru, isd);
  Us[1] = mul2(Us[0], sm);
  Us[2] = mul2(fma2(ru, q.v, mul2(nbx, sub2(by, q.by))), isd);
  Us[3] = mul2(fma2(ru, q.w, mul2(nbx, sub2(bz, q.bz))), isd);
  Us[4] = mul2(fma2(nbx, sub2(vbs, vb), fma2(pts, sm, sub2(mul2(e, su), mul2(pt, q.u)))), isd);
  Us[6] = by;
  Us[7] = bz;
  const bool olx = sl.x >= 0.f, oly = sl.y >= 0.f, orx = sr.x <= 0.f, ory = sr.y <= 0.f;
#pragma unroll
  for (int k = 0; k < 8; k++) {
    if (k == 5) continue;
    const float2 U = sel2(lx, ly, UL[k], UR[k]), F = sel2(lx, ly, FL[k], FR[k]);
    const float2 m = fma2(S, sub2(Us[k], U), F);
    f[k] = sel2(olx, oly, FL[k], sel2(orx, ory, FR[k], m));
  }
  f[5] = sp2(0.f);
}

// single-star state of one side (MK05 eqs. 43-48)
struct Star2 {
  float2 rs, vs, ws, bys, bzs, es, vbs;
};

__device__ __forceinline__ Star2 hlld_star2(const Prim2& q, float2 S, float2 su, float2 A,
                                            float2 pt, float2 e, float2 sm, float2 psm,
                                            float2 sbx, float2 bx, float2 bx2) {
  Star2 r;
  const float2 ssm = sub2(S, sm);
  const float2 isd = rcp2(ssm);
  r.rs = mul2(A, isd);
  const float2 big = mul2(A, ssm);
  const float2 den = sub2(big, bx2);
  const float2 iden = rcp2(den);
  const float2 ntv = mul2(mul2(bx, sub2(q.u, sm)), iden);
  const float2 tb = mul2(sub2(mul2(A, su), bx2), iden);
  const float eps = Num<float>::hlld_eps;
  const bool dgx = fabsf(den.x) <= eps * fmaxf(fabsf(big.x), bx2.x);
  const bool dgy = fabsf(den.y) <= eps * fmaxf(fabsf(big.y), bx2.y);
  r.vs = sel2(dgx, dgy, q.v, fma2(q.by, ntv, q.v));
  r.ws = sel2(dgx, dgy, q.w, fma2(q.bz, ntv, q.w));
  r.bys = sel2(dgx, dgy, q.by, mul2(q.by, tb));
  r.bzs = sel2(dgx, dgy, q.bz, mul2(q.bz, tb));
  const float2 vb = fma2(q.w, q.bz, fma2(q.v, q.by, mul2(q.u, bx)));
  r.vbs = fma2(r.ws, r.bzs, fma2(r.vs, r.bys, sbx));
  float2 t = sub2(mul2(su, e), mul2(pt, q.u));
  t = fma2(bx, sub2(vb, r.vbs), add2(psm, t));
  r.es = mul2(t, isd);
  return r;
}

// HLLD (MK05)
__device__ __forceinline__ void hlld2(float g, float ig1, const Prim2& L, const Prim2& R,
                                      float2 bx, float2* f) {
  const float2 bx2 = mul2(bx, bx);
  float2 btL, ptL, eL, btR, ptR, eR;
  pt_e_xy(L, bx2, ig1, btL, ptL, eL);
  pt_e_xy(R, bx2, ig1, btR, ptR, eR);
  // one root for both sides: the larger of the squared fast speeds
  const float2 cmax =
      sqrt2(max2(fast_xy(g, L.rho, L.p, btL, bx2), fast_xy(g, R.rho, R.p, btR, bx2)));
  const float2 sl = sub2(min2(L.u, R.u), cmax), sr = add2(max2(L.u, R.u), cmax);
  const float2 suL = sub2(sl, L.u), suR = sub2(sr, R.u);
  const float2 AL = mul2(suL, L.rho), AR = mul2(suR, R.rho);
  const float2 iden = rcp2(sub2(AR, AL));
  // S_M and p_T* from the HLL-averaged normal momentum (MK05 eqs. 38, 41)
  const float2 sm = mul2(sub2(fma2(AR, R.u, ptL), fma2(AL, L.u, ptR)), iden);
  const float2 pts =
      mul2(fma2(mul2(AL, AR), sub2(R.u, L.u), sub2(mul2(AR, ptL), mul2(AL, ptR))), iden);
  const float2 psm = mul2(pts, sm), sbx = mul2(sm, bx);
  const Star2 SL = hlld_star2(L, sl, suL, AL, ptL, eL, sm, psm, sbx, bx, bx2);
  const Star2 SR = hlld_star2(R, sr, suR, AR, ptR, eR, sm, psm, sbx, bx, bx2);
  // double-star states (MK05 eqs. 59-63)
  const float2 isqL = make_float2(rsqrtf(SL.rs.x), rsqrtf(SL.rs.y));
  const float2 isqR = make_float2(rsqrtf(SR.rs.x), rsqrtf(SR.rs.y));
  const float2 sqrL = mul2(SL.rs, isqL), sqrR = mul2(SR.rs, isqR);
  const float2 abx = abs2(bx);
  const float2 ssl = sub2(sm, mul2(abx, isqL)), ssr = fma2(abx, isqR, sm);
  const float2 sb = make_float2(bx.x == 0.f ? 0.f : copysignf(1.f, bx.x),
                                bx.y == 0.f ? 0.f : copysignf(1.f, bx.y));
  const float2 issum = rcp2(add2(sqrL, sqrR));
  const float2 wL = mul2(sqrL, issum), wR = mul2(sqrR, issum), wS = mul2(sb, issum);
  const float2 wQ = mul2(mul2(sqrL, wR), sb);
  const float2 vss = fma2(sub2(SR.bys, SL.bys), wS, fma2(wR, SR.vs, mul2(wL, SL.vs)));
  const float2 wss = fma2(sub2(SR.bzs, SL.bzs), wS, fma2(wR, SR.ws, mul2(wL, SL.ws)));
  const float2 byss = fma2(sub2(SR.vs, SL.vs), wQ, fma2(wL, SR.bys, mul2(wR, SL.bys)));
  const float2 bzss = fma2(sub2(SR.ws, SL.ws), wQ, fma2(wL, SR.bzs, mul2(wR, SL.bzs)));
  const float2 vbss = fma2(wss, bzss, fma2(vss, byss, sbx));
  // fan region containing x/t = 0, per face (ties as in the scalar solver)
  const bool lx = sm.x >= 0.f, ly = sm.y >= 0.f;
  const bool ox = lx ? (sl.x > 0.f) : (sr.x < 0.f), oy = ly ? (sl.y > 0.f) : (sr.y < 0.f);
  const bool sx = lx ? (ssl.x >= 0.f) : !(ssr.x >= 0.f);
  const bool sy = ly ? (ssl.y >= 0.f) : !(ssr.y >= 0.f);
  // the upwind side of S_M
  const Prim2 q = {sel2(lx, ly, L.rho, R.rho), sel2(lx, ly, L.u, R.u), sel2(lx, ly, L.v, R.v),
                   sel2(lx, ly, L.w, R.w),     sp2(0.f),               sel2(lx, ly, L.by, R.by),
                   sel2(lx, ly, L.bz, R.bz)};
  const float2 pt = sel2(lx, ly, ptL, ptR), e = sel2(lx, ly, eL, eR);
  const float2 rs = sel2(lx, ly, SL.rs, SR.rs), vs = sel2(lx, ly, SL.vs, SR.vs);
  const float2 ws = sel2(lx, ly, SL.ws, SR.ws), bys = sel2(lx, ly, SL.bys, SR.bys);
  const float2 bzs = sel2(lx, ly, SL.bzs, SR.bzs), es = sel2(lx, ly, SL.es, SR.es);
  const float2 vbs = sel2(lx, ly, SL.vbs, SR.vbs);
  const float2 sq = sel2(lx, ly, neg2(sqrL), sqrR);
  const float2 c1 = sel2(lx, ly, sl, sr), c2 = sel2(lx, ly, ssl, ssr);
  float2 U[8], F[8];
  state_flux2(q, bx, bx2, pt, e, U, F);
  // flux F + c1 (U* - U) + c2 (U** - U*): the double star keeps rho* and S_M,
  // and e** - e* = -/+ sqrt(rho*) (v*.B* - v**.B**) sgn(Bx)
  const float2 c2r = mul2(c2, rs);
  const float2 US[8] = {rs, mul2(rs, sm), mul2(rs, vs), mul2(rs, ws), es, bx, bys, bzs};
  const float2 de = mul2(mul2(sq, sb), sub2(vbs, vbss));
#pragma unroll
  for (int c = 0; c < 8; c++) {
    if (c == 5) {
      f[c] = sp2(0.f);
      continue;
    }
    const float2 fs = fma2(c1, sub2(US[c], U[c]), F[c]);
    float2 fss = fs;
    if (c == 2) fss = fma2(c2r, sub2(vss, vs), fs);
    if (c == 3) fss = fma2(c2r, sub2(wss, ws), fs);
    if (c == 4) fss = fma2(c2, de, fs);
    if (c == 6) fss = fma2(c2, sub2(byss, bys), fs);
    if (c == 7) fss = fma2(c2, sub2(bzss, bzs), fs);
    f[c] = sel2(ox, oy, F[c], c < 2 ? fs : sel2(sx, sy, fs, fss));
  }
}

// fluxes of an x face (lane x) and a y face (lane y) from their left and right
// states in the local frames (component c of lane y is variable yface_var(c));
// component 5 is the flux of the normal field
template <int FLUX>
__device__ __forceinline__ void face_flux_xy(const float2* wl, const float2* wr,
                                             const FaceConst2& fc, float2* f) {
  const float2 bnl = wl[5], bnr = wr[5];
  float2 bns = mul2(sp2(0.5f), add2(bnl, bnr)), psis = sp2(0.f), fpsi = sp2(0.f);
  if (fc.glm) {
    bns = fma2(sub2(wl[8], wr[8]), sp2(fc.hich), bns);
    psis = fma2(sub2(bnl, bnr), sp2(0.5f * fc.ch), mul2(sp2(0.5f), add2(wl[8], wr[8])));
    fpsi = mul2(sp2(fc.ch * fc.ch), bns);
  }
  const Prim2 L = {wl[0], wl[1], wl[2], wl[3], wl[4], wl[6], wl[7]};
  const Prim2 R = {wr[0], wr[1], wr[2], wr[3], wr[4], wr[6], wr[7]};
  if constexpr (FLUX == AMRVAC_FLUX_HLLD) hlld2(fc.g, fc.ig1, L, R, bns, f);
  else if constexpr (FLUX == AMRVAC_FLUX_HLLC) hllc2(fc.g, fc.ig1, L, R, bns, f);
  else hll2<FLUX>(fc.g, fc.ig1, L, R, bns, f);
  f[5] = psis;
  f[8] = fpsi;
}

// ---------------------------------------------------------------- five points
// Both states of a face from its six cells (lane x: the left state, from cells
// 0 .. 4; lane y: the right state, the mirrored stencil 5 .. 1), as increments
// to the cell value next to the face: with s1 .. s4 the differences along the
// stencil every formula of physics.cuh becomes free of the cell value itself
// (and exact on constant data).  Minima and selects are per lane.
__device__ __forceinline__ float minmod_f(float a, float b) {
  return fmaxf(fminf(a, b), 0.f) + fminf(fmaxf(a, b), 0.f);
}
__device__ __forceinline__ float minmod4_f(float w, float x, float y, float z) {
  return fmaxf(fminf(fminf(w, x), fminf(y, z)), 0.f) + fminf(fmaxf(fmaxf(w, x), fmaxf(y, z)), 0.f);
}

// the limited part of mp5 (one lane): q = the fifth-order increment
__device__ __forceinline__ float mp5_clip(float q, float s1, float s2, float s3, float s4) {
  const float djm = s2 - s1, dj = s3 - s2, djp = s4 - s3;
  const float dp = minmod4_f(4.f * dj - djp, 4.f * djp - dj, dj, djp);
  const float dm = minmod4_f(4.f * dj - djm, 4.f * djm - dj, dj, djm);
  const float ul = 4.f * s2, md = 0.5f * s3 - 0.5f * dp, lc = 0.5f * s2 + (4.f / 3.f) * dm;
  const float lo = fmaxf(fminf(fminf(0.f, s3), md), fminf(fminf(0.f, ul), lc));
  const float hi = fminf(fmaxf(fmaxf(0.f, s3), md), fmaxf(fmaxf(0.f, ul), lc));
  return q + minmod_f(lo - q, hi - q);
}

template <int LIM>
__device__ __forceinline__ float2 recon5_pair(const float* c, float lam) {
  if constexpr (LIM == AMRVAC_LIM_WENOZP5) {
    // weights from a near-cancellation: the explicitly rounded scalar form
    return make_float2(weno5_face(2, c[0], c[1], c[2], c[3], c[4], lam),
                       weno5_face(2, c[5], c[4], c[3], c[2], c[1], lam));
  } else {
    const float2 C = make_float2(c[2], c[3]);
    const float d0 = c[1] - c[0], d1 = c[2] - c[1], d2 = c[3] - c[2], d3 = c[4] - c[3],
                d4 = c[5] - c[4];
    const float2 s1 = make_float2(d0, -d4), s2 = make_float2(d1, -d3), s3 = make_float2(d2, -d2),
                 s4 = make_float2(d3, -d1);
    if constexpr (LIM == AMRVAC_LIM_MP5) {
      // (2 a - 13 b + 47 c + 27 d - 3 e)/60 - c
      float2 q = fma2(sp2(-2.f / 60.f), s1, mul2(sp2(11.f / 60.f), s2));
      q = fma2(sp2(24.f / 60.f), s3, fma2(sp2(-3.f / 60.f), s4, q));
      // kept where it lies between c and c + minmod(s3, 4 s2)
      const float mx = minmod_f(s3.x, 4.f * s2.x), my = minmod_f(s3.y, 4.f * s2.y);
      const bool kx = q.x * (q.x - mx) <= 0.f, ky = q.y * (q.y - my) <= 0.f;
      if (!kx) q.x = mp5_clip(q.x, s1.x, s2.x, s3.x, s4.x);
      if (!ky) q.y = mp5_clip(q.y, s1.y, s2.y, s3.y, s4.y);
      return add2(C, q);
    } else {
      const float2 t0 = sub2(s2, s1), u0 = fma2(sp2(3.f), s2, neg2(s1));
      const float2 t1 = sub2(s3, s2), u1 = add2(s2, s3);
      const float2 t2 = sub2(s4, s3), u2 = fma2(sp2(-3.f), s3, s4);
      const float2 k13 = sp2(13.f / 12.f), k14 = sp2(0.25f);
      const float2 b0 = fma2(mul2(k13, t0), t0, mul2(mul2(k14, u0), u0));
      const float2 b1 = fma2(mul2(k13, t1), t1, mul2(mul2(k14, u1), u1));
      const float2 b2 = fma2(mul2(k13, t2), t2, mul2(mul2(k14, u2), u2));
      const float2 q0 = mul2(fma2(sp2(5.f), s2, mul2(sp2(-2.f), s1)), sp2(1.f / 6.f));
      const float2 q1 = mul2(fma2(sp2(2.f), s3, s2), sp2(1.f / 6.f));
      const float2 q2 = mul2(fma2(sp2(4.f), s3, neg2(s4)), sp2(1.f / 6.f));
      float2 a0, a1, a2;
      if constexpr (LIM == AMRVAC_LIM_WENOZ5) {
        // scaled weights (see weno5_face): a_k = d_k (bm + bm/(b_k + eps) tau)/(bm + tau)
        const float2 eps = sp2(1e-36f), tau = abs2(sub2(b0, b2));
        const float2 bm = add2(min2(min2(b0, b1), b2), eps);
        // (in this order: bm tau alone may underflow)
        const float2 iden = rcp2(add2(bm, tau));
        a0 = mul2(sp2(0.1f), mul2(fma2(mul2(bm, rcp2(add2(b0, eps))), tau, bm), iden));
        a1 = mul2(sp2(0.6f), mul2(fma2(mul2(bm, rcp2(add2(b1, eps))), tau, bm), iden));
        a2 = mul2(sp2(0.3f), mul2(fma2(mul2(bm, rcp2(add2(b2, eps))), tau, bm), iden));
      } else {
        const float2 eps = sp2(1e-6f);
        const float2 e0 = rcp2(add2(b0, eps)), e1 = rcp2(add2(b1, eps)), e2 = rcp2(add2(b2, eps));
        a0 = mul2(mul2(sp2(0.1f), e0), e0);
        a1 = mul2(mul2(sp2(0.6f), e1), e1);
        a2 = mul2(mul2(sp2(0.3f), e2), e2);
      }
      const float2 num = fma2(a2, q2, fma2(a1, q1, mul2(a0, q0)));
      return fma2(num, rcp2(add2(add2(a0, a1), a2)), C);
    }
  }
}

// Face flux along D with the five-point limiter LIM (lam the wenozp5 lambda):
// st(v, t) for the six cells f-3 .. f+2 around the face f-1/2
template <int D, int LIM, int FLUX, class Acc>
__device__ __forceinline__ void stencil_flux5_f2(Acc st, float lam, const FaceConst2& fc,
                                                 float* f) {
  float2 w[NV];
#pragma unroll
  for (int v = 0; v < NV; v++) {
    const float c[6] = {st(v, 0), st(v, 1), st(v, 2), st(v, 3), st(v, 4), st(v, 5)};
    w[v] = recon5_pair<LIM>(c, lam);
  }
  if (not_positive2(w)) {
#pragma unroll
    for (int v = 0; v < NV; v++) w[v] = make_float2(st(v, 2), st(v, 3));
  }
  face_flux2<D, FLUX>(w, fc, f);
}

}  // namespace amrvac
