// FP32 face solvers and PLM reconstruction of the flux pass on packed pairs.
//
// The flux pass is bound by instruction issue (no pipe near its peak, other
// warps ready when one waits), and sm_103a executes two FP32 additions,
// multiplications or FMAs of a lane in one packed instruction (f32x2).  A
// Riemann solver does the same arithmetic for the left and the right state,
// so the pair (left, right) is the packed operand from the reconstruction to
// the choice of the region; only that choice and the double-star states are
// scalar.  Reciprocals are the hardware approximation (1 ulp) and one
// multiplication, where the division operator scales its operands first.
//
// Measured with the scalar solvers (division and square-root operators, one
// 4-byte shared load a value) before and these after, us per launch of the
// PLM corrector: see k_flux3.
//
// The formulas are those of common.cuh's scalar solvers, which FP64, the
// unfused path and the learned flux's fallback use; MHD = false drops every
// field term, which the scalar solvers carry as zeros.
#pragma once
#include "common.cuh"

namespace aeth {

__device__ __forceinline__ float2 splat(float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 operator+(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 operator*(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 operator-(float2 a, float2 b) {
  float2 r;
  asm("{\n\t.reg .b64 x, y, z;\n\tmov.b64 x, {%2, %3};\n\tmov.b64 y, {%4, %5};\n\t"
      "sub.rn.ftz.f32x2 z, x, y;\n\tmov.b64 {%0, %1}, z;\n\t}"
      : "=f"(r.x), "=f"(r.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return r;
}

__device__ __forceinline__ float rcp_(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ float sqrt_(float x) {
  float r;
  asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ float2 rcp2(float2 a) { return make_float2(rcp_(a.x), rcp_(a.y)); }
__device__ __forceinline__ float2 sqrt2(float2 a) { return make_float2(sqrt_(a.x), sqrt_(a.y)); }

// Half the van Leer slope of two variables at once: dm dp / (dm + dp) where
// the differences have one sign, else 0.
__device__ __forceinline__ float2 plm_half2(float2 dm, float2 dp) {
  const float2 q = dm * dp, r = rcp2(dm + dp);
  const float2 t = q * r;
  return make_float2(q.x > 0.0f ? t.x : 0.0f, q.y > 0.0f ? t.y : 0.0f);
}

// One side pair: conserved vector and physical flux of (left, right), total
// pressure and fast speed.  W = (rho, vn, vt1, vt2, p, Bt1, Bt2).
template <bool MHD, bool ISO>
struct SidePair {
  float2 u2, u3, e;                     // rho vt1, rho vt2, total energy
  float2 f0, f1, f2, f3, f4, f5, f6;    // physical flux (f0 = rho vn)
  float2 pt, vb, cf;

  // g: gamma (ISO: the sound speed squared); igm1 = 1 / (gamma - 1)
  __device__ __forceinline__ SidePair(float g, float igm1, const float2* W, float bn, float bn2) {
    const float2 rho = W[0], un = W[1], v1 = W[2], v2 = W[3], b1 = W[5], b2 = W[6];
    const float2 ir = rcp2(rho), B = splat(bn), nB = splat(-bn);
    const float2 p = ISO ? splat(g) * rho : W[4];
    f0 = rho * un;
    u2 = rho * v1;
    u3 = rho * v2;
    if constexpr (MHD) {
      const float2 bb = fma2(b2, b2, fma2(b1, b1, splat(bn2)));
      pt = fma2(bb, splat(0.5f), p);
      f1 = fma2(f0, un, pt - splat(bn2));
      f2 = fma2(u2, un, nB * b1);
      f3 = fma2(u3, un, nB * b2);
      f5 = fma2(b1, un, nB * v1);
      f6 = fma2(b2, un, nB * v2);
      const float2 a2 = ISO ? splat(g) : p * (splat(g) * ir);
      const float2 s = fma2(bb, ir, a2);
      const float2 disc = fma2(s, s, (a2 * ir) * splat(-4.0f * bn2));
      const float2 root = sqrt2(make_float2(fmaxf(disc.x, 0.0f), fmaxf(disc.y, 0.0f)));
      cf = sqrt2((s + root) * splat(0.5f));
      if constexpr (!ISO) {
        vb = fma2(v2, b2, fma2(v1, b1, un * B));
        const float2 k = fma2(u3, v2, fma2(u2, v1, f0 * un));
        e = fma2(p, splat(igm1), (k + bb) * splat(0.5f));
        f4 = fma2(e + pt, un, nB * vb);
      }
    } else {
      pt = p;
      f1 = fma2(f0, un, pt);
      f2 = u2 * un;
      f3 = u3 * un;
      if constexpr (ISO) {
        cf = splat(sqrt_(g));
      } else {
        cf = sqrt2(p * (splat(g) * ir));
        const float2 k = fma2(u3, v2, fma2(u2, v1, f0 * un));
        e = fma2(p, splat(igm1), k * splat(0.5f));
        f4 = (e + pt) * un;
      }
    }
  }
};

// HLLD (hlld_s of common.cuh; LD: LHLLD).  MHD = false: HLLC / LHLLC.
template <bool LD, bool MHD>
__device__ __forceinline__ void hlld2(float gamma, float igm1, const float2* W, float bn, float* f) {
  const float bn2 = bn * bn;
  const SidePair<MHD, false> P(gamma, igm1, W, bn, bn2);
  const float2 rho = W[0], un = W[1], v1 = W[2], v2 = W[3], b1 = W[5], b2 = W[6];
  const float cmax = fmaxf(P.cf.x, P.cf.y);
  const float2 S = make_float2(fminf(un.x, un.y) - cmax, fmaxf(un.x, un.y) + cmax);
  if constexpr (!MHD) f[5] = f[6] = 0.0f;
  if (S.x > 0.0f || S.y < 0.0f) {   // supersonic: the upwind side's flux
    const bool l = S.x > 0.0f;
    f[0] = l ? P.f0.x : P.f0.y;
    f[1] = l ? P.f1.x : P.f1.y;
    f[2] = l ? P.f2.x : P.f2.y;
    f[3] = l ? P.f3.x : P.f3.y;
    f[4] = l ? P.f4.x : P.f4.y;
    if constexpr (MHD) {
      f[5] = l ? P.f5.x : P.f5.y;
      f[6] = l ? P.f6.x : P.f6.y;
    }
    return;
  }
  const float2 su = S - un, m = rho * su;
  const float iden = rcp_(m.y - m.x);
  const float sm = (fmaf(m.y, un.y, -m.x * un.x) + (P.pt.x - P.pt.y)) * iden;
  const float du = un.y - un.x, mm = m.x * m.y;
  const float pts = fmaf(mm, du, fmaf(m.y, P.pt.x, -m.x * P.pt.y)) * iden;
  const float2 sm2 = splat(sm), ss = S - sm2, iss = rcp2(ss);
  const float2 rs = m * iss;
  float ld1 = 0.0f;   // LHLLD: the change of the pressure dissipation
  if constexpr (LD) {
    const float2 vm = sqrt2(fma2(v2, v2, fma2(v1, v1, un * un)));
    const float phi = fminf(1.0f, fmaxf(vm.x, vm.y) * rcp_(cmax));
    ld1 = (phi - 1.0f) * (mm * du * iden);
  }
  if constexpr (!MHD) {
    // one star state a side, transverse velocities unchanged
    const float2 es = (fma2(su, P.e, splat(pts * sm)) - P.pt * un) * iss;
    const float2 dr = rs - rho;
    const float2 g0 = fma2(S, dr, P.f0), g1 = fma2(S, rs * sm2 - P.f0, P.f1);
    const float2 sd = S * dr;
    const float2 g2 = fma2(sd, v1, P.f2), g3 = fma2(sd, v2, P.f3), g4 = fma2(S, es - P.e, P.f4);
    const bool l = sm >= 0.0f;
    f[0] = l ? g0.x : g0.y;
    f[1] = (l ? g1.x : g1.y) + ld1;
    f[2] = l ? g2.x : g2.y;
    f[3] = l ? g3.x : g3.y;
    f[4] = fmaf(ld1, sm, l ? g4.x : g4.y);
    return;
  } else {
    const float2 dd = fma2(m, ss, splat(-bn2)), idd = rcp2(dd);
    const float2 bni = splat(bn) * idd;
    float2 nfv = bni * (un - sm2);                       // -(transverse velocity factor)
    float2 fb = fma2(m, su, splat(-bn2)) * idd;
    const float lim = Eps<float>::hlld * pts;
    if (fabsf(dd.x) < lim) { nfv.x = 0.0f; fb.x = 1.0f; }
    if (fabsf(dd.y) < lim) { nfv.y = 0.0f; fb.y = 1.0f; }
    const float2 v1s = fma2(b1, nfv, v1), v2s = fma2(b2, nfv, v2), b1s = b1 * fb, b2s = b2 * fb;
    const float2 vbs = fma2(v2s, b2s, fma2(v1s, b1s, splat(sm * bn)));
    const float2 es = fma2(splat(bn), P.vb - vbs, fma2(su, P.e, splat(pts * sm)) - P.pt * un) * iss;
    const float2 q = make_float2(rsqrtf(rs.x), rsqrtf(rs.y)), sq = rs * q;
    const float abn = fabsf(bn);
    const bool degen = 0.5f * bn2 < lim;
    const float ssl = degen ? sm : fmaf(-abn, q.x, sm);
    const float ssr = degen ? sm : fmaf(abn, q.y, sm);
    // F* = F + S (U* - U) of both sides
    const float2 rv1 = rs * v1s, rv2 = rs * v2s;
    const float2 g0 = fma2(S, rs - rho, P.f0);
    const float2 g1 = fma2(S, rs * sm2 - P.f0, P.f1);
    const float2 g2 = fma2(S, rv1 - P.u2, P.f2), g3 = fma2(S, rv2 - P.u3, P.f3);
    const float2 g4 = fma2(S, es - P.e, P.f4);
    const float2 g5 = fma2(S, b1s - b1, P.f5), g6 = fma2(S, b2s - b2, P.f6);
    // region 1 (*L), 2 (**L), 3 (**R), 4 (*R)
    const bool star_l = ssl >= 0.0f, left = star_l || sm >= 0.0f;
    const bool dbl = !star_l && (left || ssr >= 0.0f);
    f[0] = left ? g0.x : g0.y;
    f[1] = (left ? g1.x : g1.y) + ld1;
    float h2 = left ? g2.x : g2.y, h3 = left ? g3.x : g3.y;
    float h4 = fmaf(ld1, sm, left ? g4.x : g4.y);
    float h5 = left ? g5.x : g5.y, h6 = left ? g6.x : g6.y;
    if (dbl) {
      // double-star states: shared velocity and field, sqrt(rho*) weighted
      const float sgn = bn > 0.0f ? 1.0f : (bn < 0.0f ? -1.0f : 0.0f);
      const float inv = rcp_(sq.x + sq.y), si = sgn * inv, qq = sq.x * sq.y * si;
      const float wl = sq.x * inv, wr = sq.y * inv;
      const float v1ss = fmaf(wl, v1s.x, fmaf(wr, v1s.y, (b1s.y - b1s.x) * si));
      const float v2ss = fmaf(wl, v2s.x, fmaf(wr, v2s.y, (b2s.y - b2s.x) * si));
      const float b1ss = fmaf(wl, b1s.y, fmaf(wr, b1s.x, (v1s.y - v1s.x) * qq));
      const float b2ss = fmaf(wl, b2s.y, fmaf(wr, b2s.x, (v2s.y - v2s.x) * qq));
      const float vbss = fmaf(v2ss, b2ss, fmaf(v1ss, b1ss, sm * bn));
      const float r = left ? rs.x : rs.y, st = left ? ssl : ssr;
      const float w = (left ? -sgn : sgn) * (left ? sq.x : sq.y);
      const float d1 = v1ss - (left ? v1s.x : v1s.y), d2 = v2ss - (left ? v2s.x : v2s.y);
      // F** = F* + S* (U** - U*); rho** = rho* and u** = S_M
      h2 = fmaf(st * r, d1, h2);
      h3 = fmaf(st * r, d2, h3);
      h4 = fmaf(st * w, (left ? vbs.x : vbs.y) - vbss, h4);
      h5 = fmaf(st, b1ss - (left ? b1s.x : b1s.y), h5);
      h6 = fmaf(st, b2ss - (left ? b2s.x : b2s.y), h6);
    }
    f[2] = h2; f[3] = h3; f[4] = h4; f[5] = h5; f[6] = h6;
  }
}

// HLLE (hlle of common.cuh) and the isothermal HLLE (g = cs^2, no energy):
// F = (b+ F_L - b- F_R + b+ b- (U_R - U_L)) / (b+ - b-) as two packed
// products a component and one sum of the halves.
template <bool MHD, bool ISO>
__device__ __forceinline__ void hlle2(float g, float igm1, const float2* W, float bn, float* f) {
  const SidePair<MHD, ISO> P(g, igm1, W, bn, bn * bn);
  const float2 un = W[1];
  const float cm = fmaxf(P.cf.x, P.cf.y);
  const float bm = fminf(fminf(un.x, un.y) - cm, 0.0f), bp = fmaxf(fmaxf(un.x, un.y) + cm, 0.0f);
  const float inv = rcp_(bp - bm), c = bp * bm * inv;
  const float2 wf = make_float2(bp * inv, -bm * inv), wu = make_float2(-c, c);
  auto mix = [&](float2 fx, float2 u) {
    const float2 t = fma2(wu, u, wf * fx);
    return t.x + t.y;
  };
  f[0] = mix(P.f0, W[0]);
  f[1] = mix(P.f1, P.f0);
  f[2] = mix(P.f2, P.u2);
  f[3] = mix(P.f3, P.u3);
  f[4] = 0.0f;
  if constexpr (!ISO) f[4] = mix(P.f4, P.e);
  f[5] = f[6] = 0.0f;
  if constexpr (MHD) {
    f[5] = mix(P.f5, W[5]);
    f[6] = mix(P.f6, W[6]);
  }
}

// Isothermal HLLD (hlld_iso of common.cuh), g = cs^2.
template <bool MHD>
__device__ __forceinline__ void hlld_iso2(float g, const float2* W, float bn, float* f) {
  const float bn2 = bn * bn;
  const SidePair<MHD, true> P(g, 0.0f, W, bn, bn2);
  const float2 rho = W[0], un = W[1], v1 = W[2], v2 = W[3], b1 = W[5], b2 = W[6];
  const float cm = fmaxf(P.cf.x, P.cf.y);
  const float2 S = make_float2(fminf(un.x, un.y) - cm, fmaxf(un.x, un.y) + cm);
  f[4] = f[5] = f[6] = 0.0f;
  if (S.x >= 0.0f || S.y <= 0.0f) {
    const bool l = S.x >= 0.0f;
    f[0] = l ? P.f0.x : P.f0.y;
    f[1] = l ? P.f1.x : P.f1.y;
    f[2] = l ? P.f2.x : P.f2.y;
    f[3] = l ? P.f3.x : P.f3.y;
    if constexpr (MHD) {
      f[5] = l ? P.f5.x : P.f5.y;
      f[6] = l ? P.f6.x : P.f6.y;
    }
    return;
  }
  const float idn = rcp_(S.y - S.x), ssp = S.x * S.y;
  const float rs = (fmaf(S.y, rho.y, -S.x * rho.x) - (P.f0.y - P.f0.x)) * idn;
  const float fm = fmaf(ssp, rho.y - rho.x, fmaf(S.y, P.f0.x, -S.x * P.f0.y)) * idn;
  f[0] = fm;
  f[1] = fmaf(ssp, P.f0.y - P.f0.x, fmaf(S.y, P.f1.x, -S.x * P.f1.y)) * idn;
  const float us = fm * rcp_(rs);
  const float iq = rsqrtf(rs), sq = rs * iq, al = fabsf(bn) * iq;
  const float ssl = us - al, ssr = us + al;
  // transverse star states across the fast waves
  const float2 su = S - un, m = rho * su, msu = m * su;
  float2 v1s = v1, v2s = v2, b1s = b1, b2s = b2;
  if constexpr (MHD) {
    const float2 den = fma2(m, S - splat(us), splat(-bn2)), id = rcp2(den);
    float2 nfv = (splat(bn) * id) * (un - splat(us)), fb = (msu - splat(bn2)) * id;
    const float2 lim = (msu + splat(bn2)) * splat(Eps<float>::hlld);
    if (!(fabsf(den.x) >= lim.x)) { nfv.x = 0.0f; fb.x = 1.0f; }
    if (!(fabsf(den.y) >= lim.y)) { nfv.y = 0.0f; fb.y = 1.0f; }
    v1s = fma2(b1, nfv, v1);
    v2s = fma2(b2, nfv, v2);
    b1s = b1 * fb;
    b2s = b2 * fb;
  }
  const float2 rs2 = splat(rs);
  const float2 g2 = fma2(S, rs2 * v1s - P.u2, P.f2);
  const float2 g3 = fma2(S, rs2 * v2s - P.u3, P.f3);
  const bool right = ssl < 0.0f && ssr <= 0.0f, central = ssl < 0.0f && ssr > 0.0f;
  float h2 = right ? g2.y : g2.x, h3 = right ? g3.y : g3.x, h5 = 0.0f, h6 = 0.0f;
  if constexpr (MHD) {
    const float2 g5 = fma2(S, b1s - b1, P.f5), g6 = fma2(S, b2s - b2, P.f6);
    h5 = right ? g5.y : g5.x;
    h6 = right ? g6.y : g6.x;
  }
  if (central) {
    // central state between the Alfven waves (equal densities both sides)
    const float sgn = bn > 0.0f ? 1.0f : (bn < 0.0f ? -1.0f : 0.0f);
    const float hv = 0.5f * sgn * iq, hb = 0.5f * sgn * sq, sr = ssl * rs;
    float c1 = 0.5f * (v1s.y - v1s.x), c2 = 0.5f * (v2s.y - v2s.x);   // v** - v*_L
    if constexpr (MHD) {
      const float k1 = fmaf(hb, v1s.y - v1s.x, 0.5f * (b1s.y - b1s.x));   // B** - B*_L
      const float k2 = fmaf(hb, v2s.y - v2s.x, 0.5f * (b2s.y - b2s.x));
      c1 = fmaf(hv, b1s.y - b1s.x, c1);
      c2 = fmaf(hv, b2s.y - b2s.x, c2);
      h5 = fmaf(ssl, k1, h5);
      h6 = fmaf(ssl, k2, h6);
    }
    h2 = fmaf(sr, c1, h2);
    h3 = fmaf(sr, c2, h3);
  }
  f[2] = h2; f[3] = h3; f[5] = h5; f[6] = h6;
}

}  // namespace aeth
