// FP32 face solvers of the flux pass on packed (left, right) pairs.
//
// The flux pass is bound by instruction issue, and a Riemann solver does the
// same arithmetic for the left and the right state: the pair is the packed
// operand (pair.cuh) from the reconstruction to the choice of the region; only
// that choice and the double-star states are scalar.
//
// The formulas are those of common.cuh's scalar solvers, which FP64, the
// unfused path and the learned flux's fallback use.  Every rounding is written
// out (which product of a sum enters a fused multiply-add, and which is
// rounded by itself), so that a face's flux does not depend on what the
// compiler fuses in one instantiation and not in the next: shocks and limiters
// amplify a last-bit difference, and results stay comparable bit for bit
// across tile shapes, block layouts and versions of the kernel around them.
// MHD = false drops every field term (a product with zero) with the same bits.
#pragma once
#include "pair.cuh"

namespace aeth {

__device__ __forceinline__ float rmul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float radd(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float rsub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float rfma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
// A product that a sum takes in rounded: as two scalar multiplications (a packed
// one is fused into the packed sum that follows, whatever its rounding says).
__device__ __forceinline__ float2 mul_apart(float2 a, float2 b) {
  return make_float2(rmul(a.x, b.x), rmul(a.y, b.y));
}
__device__ __forceinline__ float pick(bool left, float2 a) { return left ? a.x : a.y; }

// Conserved vector, physical flux, total pressure and fast speed of the pair;
// W = (rho, vn, vt1, vt2, p, Bt1, Bt2).  g: gamma (ISO: cs^2); igm1 =
// 1 / (gamma - 1) (the pressure is divided by gamma - 1 as one product).
template <bool MHD, bool ISO>
struct SidePair {
  float2 nrho, nun;                    // -rho, -vn
  float2 e, vv;                        // total energy, |v|^2
  float2 f0, f1, f2, f3, f4, f5, f6;   // physical flux (f0 = rho vn)
  float2 f1t;                          // f1 before the subtraction of bn^2
  float2 pt, vb, cf;

  __device__ __forceinline__ SidePair(float g, float igm1, const float2* W, float bn, float bn2) {
    const float2 rho = W[0], un = W[1], v1 = W[2], v2 = W[3], b1 = W[5], b2 = W[6];
    nrho = make_float2(-rho.x, -rho.y);
    nun = make_float2(-un.x, -un.y);
    const float2 ir = make_float2(recip(rho.x), recip(rho.y));
    const float2 p = ISO ? splat(g) * rho : W[4];
    const float2 a2 = (ISO ? p : splat(g) * p) * ir;
    f0 = rho * un;
    if constexpr (MHD) {
      const float2 B = splat(bn), nB = splat(-bn);
      const float2 bb = fma2(b2, b2, fma2(b1, b1, splat(bn2)));
      if constexpr (ISO) pt = fma2(splat(g), rho, splat(0.5f) * bb);
      else pt = fma2(splat(0.5f), bb, p);
      f1t = fma2(f0, un, pt);
      f1 = f1t - splat(bn2);
      f2 = fma2(f0, v1, nB * b1);
      f3 = fma2(f0, v2, nB * b2);
      f5 = fma2(b1, un, nB * v1);
      f6 = fma2(b2, un, nB * v2);
      const float2 s = fma2(bb, ir, a2);
      const float2 disc = fma2(s, s, (((splat(-4.0f) * a2) * B) * B) * ir);
      cf = speed(s, disc);
      if constexpr (!ISO) {
        vb = fma2(v2, b2, fma2(un, B, v1 * b1));
        vv = fma2(v2, v2, fma2(un, un, v1 * v1));
        e = fma2(splat(0.5f), bb, fma2(splat(0.5f) * rho, vv, p * splat(igm1)));
        f4 = fma2(e + pt, un, nB * vb);
      }
    } else {
      pt = p;
      f1 = f1t = fma2(f0, un, pt);
      f2 = f0 * v1;
      f3 = f0 * v2;
      cf = speed(a2, a2 * a2);
      if constexpr (!ISO) {
        vv = fma2(v2, v2, fma2(un, un, v1 * v1));
        e = fma2(splat(0.5f) * rho, vv, p * splat(igm1));
        f4 = (e + pt) * un;
      }
    }
  }
  static __device__ __forceinline__ float2 speed(float2 s, float2 disc) {
    const float2 r = make_float2(sqrtf(fmaxf(disc.x, 0.0f)), sqrtf(fmaxf(disc.y, 0.0f)));
    const float2 h = splat(0.5f) * (s + r);
    return make_float2(sqrtf(h.x), sqrtf(h.y));
  }
};

// HLLD (hlld_s of common.cuh; LD: LHLLD); MHD = false: HLLC / LHLLC.  SPLIT decides
// one rounding of the right side.  The left normal momentum flux subtracts bn^2
// rounded; the right one does the same with SPLIT, and without it subtracts the
// unrounded square in one multiply-add.  So without SPLIT the solver is mirror
// symmetric up to that last bit only.  Both forms are what the scalar solver's compiled
// text rounded to (SPLIT: z faces of donor states), kept so that results stay
// comparable bit for bit.
template <bool LD, bool MHD, bool SPLIT>
__device__ __forceinline__ void hlld2(float gamma, float igm1, const float2* W, float bn, float* f) {
  const float bn2 = rmul(bn, bn);
  const SidePair<MHD, false> P(gamma, igm1, W, bn, bn2);
  const float2 rho = W[0], un = W[1], v1 = W[2], v2 = W[3], b1 = W[5], b2 = W[6];
  const float cmax = fmaxf(P.cf.x, P.cf.y);
  const float2 S = make_float2(rsub(fminf(un.x, un.y), cmax), radd(fmaxf(un.x, un.y), cmax));
  if constexpr (!MHD) f[5] = f[6] = 0.0f;
  if (S.x > 0.0f || S.y < 0.0f) {   // supersonic: the upwind side's flux
    const bool l = S.x > 0.0f;
    f[0] = pick(l, P.f0); f[1] = pick(l, P.f1); f[2] = pick(l, P.f2); f[3] = pick(l, P.f3);
    f[4] = pick(l, P.f4);
    if constexpr (MHD) { f[5] = pick(l, P.f5); f[6] = pick(l, P.f6); }
    return;
  }
  const float2 su = S - un, m = su * rho;
  const float iden = recip(rsub(m.y, m.x));
  const float sm = rmul(radd(rsub(rfma(m.y, un.y, rmul(m.x, P.nun.x)), P.pt.y), P.pt.x), iden);
  const float t5 = rmul(rmul(rmul(rho.x, rho.y), su.y), su.x), du = rsub(un.y, un.x);
  const float x = rfma(m.y, P.pt.x, -rmul(m.x, P.pt.y));
  const float pts = rmul(LD ? radd(rmul(t5, du), x) : rfma(t5, du, x), iden);
  const float2 ss = S - splat(sm), iss = make_float2(recip(ss.x), recip(ss.y));
  const float2 rs = m * iss;
  // star energy, without the field's work in hydro
  const float2 ea = fma2(su, P.e, P.pt * P.nun), eb = splat(rmul(pts, sm)) + ea;
  float pd = 0.0f;   // LHLLD: the change of the pressure dissipation
  if constexpr (LD) {
    const float phi = fminf(1.0f, rmul(fmaxf(sqrtf(P.vv.x), sqrtf(P.vv.y)), recip(cmax)));
    pd = rmul(rsub(phi, 1.0f), rmul(rmul(t5, du), iden));
  }
  // F* = F + S (U* - U) of both sides
  const float2 g0 = fma2(S, rs - rho, P.f0);
  const float2 d1 = fma2(rs, splat(sm), rho * P.nun);
  if constexpr (!MHD) {
    const float2 es = mul_apart(eb, iss);
    const float2 g1 = fma2(S, d1, P.f1);
    const float2 g2 = fma2(S, fma2(P.nrho, v1, rs * v1), P.f2);
    const float2 g3 = fma2(S, fma2(P.nrho, v2, rs * v2), P.f3);
    const float2 g4 = fma2(S, es - P.e, P.f4);
    const bool l = sm >= 0.0f;
    f[0] = pick(l, g0);
    f[1] = LD ? radd(pick(l, g1), pd) : pick(l, g1);
    f[2] = pick(l, g2);
    f[3] = pick(l, g3);
    f[4] = LD ? rfma(pd, sm, pick(l, g4)) : pick(l, g4);
  } else {
    const float2 nbn2 = splat(-bn2);
    const float2 dd = fma2(m, ss, nbn2), idd = make_float2(recip(dd.x), recip(dd.y));
    float2 nfv = (splat(bn) * (un - splat(sm))) * idd;   // -(transverse velocity factor)
    float2 fb = fma2(m, su, nbn2) * idd;
    const float lim = rmul(Eps<float>::hlld, pts);
    if (fabsf(dd.x) < lim) { nfv.x = 0.0f; fb.x = 1.0f; }
    if (fabsf(dd.y) < lim) { nfv.y = 0.0f; fb.y = 1.0f; }
    const float2 v1s = fma2(b1, nfv, v1), v2s = fma2(b2, nfv, v2), b1s = b1 * fb, b2s = b2 * fb;
    const float smb = rmul(sm, bn);
    const float2 vbs = fma2(v2s, b2s, fma2(v1s, b1s, splat(smb)));
    const float2 es = fma2(splat(bn), P.vb - vbs, eb) * iss;
    const float2 q = make_float2(rsqrtf(rs.x), rsqrtf(rs.y)), sq = rs * q;
    const float abn = fabsf(bn);
    const bool degen = rmul(0.5f, bn2) < lim;
    const float ssl = degen ? sm : rfma(-abn, q.x, sm);
    const float ssr = degen ? sm : rfma(abn, q.y, sm);
    const float2 f1 = make_float2(P.f1.x, SPLIT ? P.f1.y : rfma(-bn, bn, P.f1t.y));
    const float2 g1 = fma2(S, d1, f1);
    const float2 g2 = fma2(S, fma2(P.nrho, v1, rs * v1s), P.f2);
    const float2 g3 = fma2(S, fma2(P.nrho, v2, rs * v2s), P.f3);
    const float2 g4 = fma2(S, es - P.e, P.f4);
    const float2 g5 = fma2(S, b1s - b1, P.f5), g6 = fma2(S, b2s - b2, P.f6);
    // region 1 (*L), 2 (**L), 3 (**R), 4 (*R)
    const bool star_l = ssl >= 0.0f, left = star_l || sm >= 0.0f;
    const bool dbl = !star_l && (left || ssr >= 0.0f);
    f[0] = pick(left, g0);
    f[1] = LD ? radd(pick(left, g1), pd) : pick(left, g1);
    float h2 = pick(left, g2), h3 = pick(left, g3);
    float h4 = LD ? rfma(pd, sm, pick(left, g4)) : pick(left, g4);
    float h5 = pick(left, g5), h6 = pick(left, g6);
    if (dbl) {
      // double-star states: shared velocity and field, sqrt(rho*) weighted
      const float sgn = bn > 0.0f ? 1.0f : (bn < 0.0f ? -1.0f : 0.0f);
      const float inv = recip(radd(sq.x, sq.y)), qq = rmul(sq.x, sq.y);
      const float v1ss = rmul(rfma(rsub(b1s.y, b1s.x), sgn, rfma(sq.x, v1s.x, rmul(sq.y, v1s.y))), inv);
      const float v2ss = rmul(rfma(rsub(b2s.y, b2s.x), sgn, rfma(sq.x, v2s.x, rmul(sq.y, v2s.y))), inv);
      const float b1ss = rmul(rfma(rmul(qq, rsub(v1s.y, v1s.x)), sgn,
                                   rfma(sq.x, b1s.y, rmul(sq.y, b1s.x))), inv);
      const float b2ss = rmul(rfma(rmul(qq, rsub(v2s.y, v2s.x)), sgn,
                                   rfma(sq.x, b2s.y, rmul(sq.y, b2s.x))), inv);
      const float vbss = rfma(v2ss, b2ss, rfma(v1ss, b1ss, smb));
      const float r = pick(left, rs), st = left ? ssl : ssr, ese = pick(left, es);
      const float w = left ? -sq.x : sq.y;
      const float ess = rfma(rmul(w, rsub(pick(left, vbs), vbss)), sgn, ese);
      // F** = F* + S* (U** - U*); rho** = rho* and u** = S_M
      h2 = rfma(st, rfma(r, v1ss, -rmul(r, pick(left, v1s))), h2);
      h3 = rfma(st, rfma(r, v2ss, -rmul(r, pick(left, v2s))), h3);
      h4 = rfma(st, rsub(ess, ese), h4);
      h5 = rfma(st, rsub(b1ss, pick(left, b1s)), h5);
      h6 = rfma(st, rsub(b2ss, pick(left, b2s)), h6);
    }
    f[2] = h2; f[3] = h3; f[4] = h4; f[5] = h5; f[6] = h6;
  }
}

// Isothermal HLLD (hlld_iso of common.cuh), g = cs^2.  SPLIT: the right side's
// induction fluxes are differences of two rounded products, the left side's (and
// without SPLIT both) one multiply-add of a rounded product: again the last bit in
// which the two sides differ.
template <bool MHD, bool SPLIT>
__device__ __forceinline__ void hlld_iso2(float g, const float2* W, float bn, float* f) {
  const float bn2 = rmul(bn, bn);
  SidePair<MHD, true> P(g, 0.0f, W, bn, bn2);
  const float2 rho = W[0], un = W[1], v1 = W[2], v2 = W[3], b1 = W[5], b2 = W[6];
  if constexpr (MHD && SPLIT) {
    P.f5.y = rsub(rmul(b1.y, un.y), rmul(bn, v1.y));
    P.f6.y = rsub(rmul(b2.y, un.y), rmul(bn, v2.y));
  }
  const float cm = fmaxf(P.cf.x, P.cf.y);
  const float2 S = make_float2(rsub(fminf(un.x, un.y), cm), radd(fmaxf(un.x, un.y), cm));
  f[4] = f[5] = f[6] = 0.0f;
  if (S.x >= 0.0f || S.y <= 0.0f) {
    const bool l = S.x >= 0.0f;
    f[0] = pick(l, P.f0); f[1] = pick(l, P.f1); f[2] = pick(l, P.f2); f[3] = pick(l, P.f3);
    if constexpr (MHD) { f[5] = pick(l, P.f5); f[6] = pick(l, P.f6); }
    return;
  }
  const float idn = recip(rsub(S.y, S.x)), ssp = rmul(S.x, S.y), df = rsub(P.f0.y, P.f0.x);
  const float rs = rmul(rsub(rfma(S.y, rho.y, -rmul(S.x, rho.x)), df), idn);
  const float fm = rmul(rfma(ssp, rsub(rho.y, rho.x), rfma(S.y, P.f0.x, -rmul(S.x, P.f0.y))), idn);
  f[0] = fm;
  f[1] = rmul(rfma(ssp, df, rfma(S.y, P.f1.x, -rmul(S.x, P.f1.y))), idn);
  const float us = rmul(fm, recip(rs));
  const float2 rs2 = splat(rs);
  if constexpr (!MHD) {   // no Alfven waves: the side the flow comes from
    const bool l = !(us < 0.0f);
    f[2] = pick(l, fma2(S, fma2(rs2, v1, P.nrho * v1), P.f2));
    f[3] = pick(l, fma2(S, fma2(rs2, v2, P.nrho * v2), P.f3));
  } else {
    const float sq = sqrtf(rs), isq = recip(sq), al = rmul(fabsf(bn), isq);
    const float ssl = rsub(us, al), ssr = radd(us, al);
    // transverse star states across the fast waves
    const float2 su = S - un, m = rho * su;
    const float2 den = fma2(m, S - splat(us), splat(-bn2));
    const float2 id = make_float2(recip(den.x), recip(den.y));
    float2 nfv = (splat(bn) * (un - splat(us))) * id, fb = (mul_apart(m, su) - splat(bn2)) * id;
    const float2 lim = splat(Eps<float>::hlld) * fma2(m, su, splat(bn2));
    if (!(fabsf(den.x) >= lim.x)) { nfv.x = 0.0f; fb.x = 1.0f; }
    if (!(fabsf(den.y) >= lim.y)) { nfv.y = 0.0f; fb.y = 1.0f; }
    const float2 v1s = fma2(b1, nfv, v1), v2s = fma2(b2, nfv, v2), b1s = b1 * fb, b2s = b2 * fb;
    const float2 g2 = fma2(S, fma2(rs2, v1s, P.nrho * v1), P.f2);
    const float2 g3 = fma2(S, fma2(rs2, v2s, P.nrho * v2), P.f3);
    const float2 g5 = fma2(S, b1s - b1, P.f5), g6 = fma2(S, b2s - b2, P.f6);
    const bool l = !(ssl < 0.0f && ssr <= 0.0f);
    float h2 = pick(l, g2), h3 = pick(l, g3), h5 = pick(l, g5), h6 = pick(l, g6);
    if (ssl < 0.0f && ssr > 0.0f) {
      // central state between the Alfven waves (equal densities both sides)
      const float sgn = bn > 0.0f ? 1.0f : (bn < 0.0f ? -1.0f : 0.0f), hs = rmul(0.5f, sq);
      auto cv = [&](float2 v, float2 b) {
        return rfma(0.5f, radd(v.x, v.y), rmul(rmul(rmul(0.5f, rsub(b.y, b.x)), sgn), isq));
      };
      auto cb = [&](float2 v, float2 b) {
        return rfma(0.5f, radd(b.x, b.y), rmul(rmul(hs, rsub(v.y, v.x)), sgn));
      };
      h2 = rfma(ssl, rfma(rs, cv(v1s, b1s), -rmul(rs, v1s.x)), h2);
      h3 = rfma(ssl, rfma(rs, cv(v2s, b2s), -rmul(rs, v2s.x)), h3);
      h5 = rfma(ssl, rsub(cb(v1s, b1s), b1s.x), h5);
      h6 = rfma(ssl, rsub(cb(v2s, b2s), b2s.x), h6);
    }
    f[2] = h2; f[3] = h3; f[5] = h5; f[6] = h6;
  }
}

// HLLE (hlle of common.cuh): sides on pairs, the average scalar.  Smooth 256^3 in
// eight linked blocks, RK2: flux pass 943 -> 923 us
// (the stores and the staged halo weigh more there than the solver), step 3588 -> 3540.
template <bool MHD>
__device__ __forceinline__ void hlle2(float gamma, float igm1, const float2* W, float bn, float* f) {
  const float bn2 = rmul(bn, bn);
  const SidePair<MHD, false> P(gamma, igm1, W, bn, bn2);
  const float2 rho = W[0], un = W[1];
  // the energy as this solver's text is contracted: the pressure's product fused
  float2 e = fma2(W[4], splat(igm1), splat(0.5f) * rho * P.vv), f4;
  if constexpr (MHD) {
    const float2 bb = fma2(W[6], W[6], fma2(W[5], W[5], splat(bn2)));
    e = fma2(splat(0.5f), bb, e);
    f4 = fma2(e + P.pt, un, splat(-bn) * P.vb);
  } else {
    f4 = (e + P.pt) * un;
  }
  const float cm = fmaxf(P.cf.x, P.cf.y);
  const float bm = fminf(rsub(fminf(un.x, un.y), cm), 0.0f);
  const float bp = fmaxf(radd(fmaxf(un.x, un.y), cm), 0.0f);
  const float inv = recip(rsub(bp, bm)), bb = rmul(bp, bm);
  auto average = [&](float2 fx, float du) {
    return rmul(rfma(bb, du, rfma(bp, fx.x, -rmul(bm, fx.y))), inv);
  };
  f[0] = average(P.f0, rsub(rho.y, rho.x));
  f[1] = average(P.f1, rsub(P.f0.y, P.f0.x));
  f[2] = average(P.f2, rfma(rho.y, W[2].y, -rmul(rho.x, W[2].x)));
  f[3] = average(P.f3, rfma(rho.y, W[3].y, -rmul(rho.x, W[3].x)));
  f[4] = average(f4, rsub(e.y, e.x));
  if constexpr (MHD) {
    f[5] = average(P.f5, rsub(W[5].y, W[5].x));
    f[6] = average(P.f6, rsub(W[6].y, W[6].x));
  } else {
    f[5] = f[6] = 0.0f;
  }
}

}  // namespace aeth
