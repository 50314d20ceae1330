// Multifluid dust (Sec. 2.2, Eqs. 6-7) with the IMEX2P integrator (Sec. 2.6).
//
// Per stage: ghost fill; the fused hydro-gas flux pass (HLLD at B = 0); the
// pressureless Rusanov fluxes of every species (FP32: one pass that leaves their
// divergence; FP64: a flux pass per direction); then one fused kernel that forms
// the explicit stage combination and solves the implicit drag of every cell in
// closed form (arrowhead system, O(N) per velocity component), by default
// (aeth_config.drag_precision) in FP64 or, under FP32 transport, FP32 pairs.
//
// The stage combinations run in the working precision.  GB300 executes an FP64
// operation at 1/64 of the FP32 rate, and the solve's ~215 operations and ~65
// conversions a cell made the update 68% of the step, so FP32 transport solves
// in FP32 pairs (dfloat.cuh, about 48 bits: the same FP32 results but for rare
// last bits; error against FP64 of 10 steps unchanged, 1.4e-7).  128^3, 8
// species: the update 1751 -> 458 / 565 us a launch (now 400 / 504 on the
// divergence, 1.0 and 1.4 GB: bound by memory latency at 16 warps an SM and the
// pairs' serial sums), the step 5169 -> 2504 us; 61 x 100 x 37, 3 species,
// per-species precision: 395 -> 273 us a step.  The FP64 solve stays
// for FP64 transport, the constant-coefficient law, and cells or constants
// outside the pairs' range.
//
// IMEX2P with implicit weight g = 1 + 1/sqrt 2 and explicit weight
// d = 1 - 1/(2g) in two registers (A, B):
//   stage 2: X = U^n + g dt L(U^n), W = U^n + d dt L(U^n), U2 = drag_h(X),
//            B <- U2, A <- W + (1-g)/g (U2 - X)          [(U2-X)/g = dt R(U2)]
//   stage 3: Y = A + (1-d) dt L(U2), A <- drag_h(Y)      (h = g dt)
#include <type_traits>

#include "dfloat.cuh"
#include "ghost.cuh"
#include "pair.cuh"
#include "runtime.hpp"

namespace aeth {

template <typename R>
void launch_fill(const BlockPtrs<R>& P, R* const* arrs, int nv, cudaStream_t st);
template <typename R, bool P64>
void hydro_flux_pass(aeth_ctx* c, int block, int recon, int src);

// z depth of the update's CTAs: 1 (128 threads; 2 or 3 CTAs per SM at its
// 160-180 registers) measured 6-9% faster than 2 (256 threads, one CTA)
#ifndef AETH_DUST_BZ
#define AETH_DUST_BZ 1
#endif

constexpr double kImexG = 1.0 + 0.70710678118654752440;
constexpr double kImexD = 1.0 - 1.0 / (2.0 * kImexG);

// ------------------------------------------------------------------------
// Rusanov fluxes of every species, and their divergence
// ------------------------------------------------------------------------

// Flux across a D-face from its states (rho, v1, v2, v3).
template <int D, typename R>
__device__ __forceinline__ void dust_flux(const R* wl, const R* wr, R* f) {
  const R vnl = wl[1 + D], vnr = wr[1 + D];
  const R sp = fmax(fabs(vnl), fabs(vnr));
  const R ul[4] = {wl[0], wl[0] * wl[1], wl[0] * wl[2], wl[0] * wl[3]};
  const R ur[4] = {wr[0], wr[0] * wr[1], wr[0] * wr[2], wr[0] * wr[3]};
#pragma unroll
  for (int q = 0; q < 4; ++q)
    f[q] = R(0.5) * (ul[q] * vnl + ur[q] * vnr) - R(0.5) * sp * (ur[q] - ul[q]);
}

// The same in FP32, and the PPM and PPM5 face states, with every rounding written
// out: the two cells of a face compute its flux each for itself, and what the compiler
// fuses in one place and not in the other would give a face two fluxes (what leaves
// one cell would not be what enters the next).
template <int D>
__device__ __forceinline__ void dust_flux(const float* wl, const float* wr, float* f) {
  const float vl = wl[1 + D], vr = wr[1 + D];
  const float hs = -0.5f * fmaxf(fabsf(vl), fabsf(vr));
  float ml[3], mr[3];
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    ml[q] = __fmul_rn(wl[0], wl[1 + q]);
    mr[q] = __fmul_rn(wr[0], wr[1 + q]);
  }
  f[0] = __fmaf_rn(0.5f, __fadd_rn(ml[D], mr[D]), __fmul_rn(hs, __fsub_rn(wr[0], wl[0])));
#pragma unroll
  for (int q = 0; q < 3; ++q)
    f[1 + q] = __fmaf_rn(0.5f, __fmaf_rn(ml[q], vl, __fmul_rn(mr[q], vr)),
                         __fmul_rn(hs, __fsub_rn(mr[q], ml[q])));
}
// ppm_iface, ppm5_left, ppm5_right (clipped) and ppm_limit of common.cuh
__device__ __forceinline__ float dust_iface(const float* s) {
  const float x = __fadd_rn(s[1], s[2]), y = __fadd_rn(s[0], s[3]);
  return clip_pair(__fmaf_rn((float)(7.0 / 12.0), x, -__fmul_rn((float)(1.0 / 12.0), y)), s[1], s[2]);
}
__device__ __forceinline__ float dust_left(const float* q) {
  float a = __fmaf_rn(27.0f, q[1], __fmul_rn(-3.0f, q[0]));
  a = __fmaf_rn(2.0f, q[4], __fmaf_rn(-13.0f, q[3], __fmaf_rn(47.0f, q[2], a)));
  return clip_pair(__fmul_rn(a, (float)(1.0 / 60.0)), q[1], q[2]);
}
__device__ __forceinline__ float dust_right(const float* q) {
  float a = __fmaf_rn(-13.0f, q[1], __fmul_rn(2.0f, q[0]));
  a = __fmaf_rn(-3.0f, q[4], __fmaf_rn(27.0f, q[3], __fmaf_rn(47.0f, q[2], a)));
  return clip_pair(__fmul_rn(a, (float)(1.0 / 60.0)), q[2], q[3]);
}
__device__ __forceinline__ void dust_limit(float w, float& l, float& r) {
  if (__fmul_rn(__fsub_rn(r, w), __fsub_rn(w, l)) <= 0.0f) {
    l = r = w;
    return;
  }
  const float d = __fsub_rn(r, l), q = __fmul_rn(d, __fmaf_rn(-0.5f, __fadd_rn(l, r), w));
  const float d2 = __fmul_rn(__fmul_rn(d, d), (float)(1.0 / 6.0));
  if (q > d2) l = __fmaf_rn(3.0f, w, -__fmul_rn(2.0f, r));
  else if (-d2 > q) r = __fmaf_rn(3.0f, w, -__fmul_rn(2.0f, l));
}
// Face states of one variable, as recon_face.
template <int RECON>
__device__ __forceinline__ void dust_states(const float* s, float& wl, float& wr) {
  if constexpr (RECON < 2) {
    recon_face<RECON>(s, wl, wr);
  } else {
    float l1, r1, l2, r2;
    if constexpr (RECON == 2) {
      l1 = dust_iface(s);
      r1 = l2 = dust_iface(s + 1);
      r2 = dust_iface(s + 2);
    } else {
      l1 = dust_left(s);
      r1 = dust_right(s);
      l2 = dust_left(s + 1);
      r2 = dust_right(s + 1);
    }
    dust_limit(s[2], l1, r1);
    dust_limit(s[3], l2, r2);
    wl = r1;
    wr = l2;
  }
}
template <int RECON>
__device__ __forceinline__ void dust_states(const double* s, double& wl, double& wr) {
  recon_face<RECON>(s, wl, wr);
}

// Flux across the D-face between cells w[2] and w[3] of a line of cells.
template <int RECON, int D, typename R>
__device__ __forceinline__ void dust_face(const R (*w)[4], R* f) {
  R wl[4], wr[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    R s[6];
#pragma unroll
    for (int t = 0; t < 6; ++t) s[t] = w[t][q];
    dust_states<RECON>(s, wl[q], wr[q]);
  }
  dust_flux<D>(wl, wr, f);
}

// FP64: the fluxes of all species across the lower D-face of each cell.  The
// FP64 pipe bounds these passes, so each face is computed once and its flux goes
// through memory: with every x and y face computed by both of its cells (the FP32
// pass below) a PLM step of 96^3 with 4 species took 17901 us against 15035, and 61 x 100 x 37
// with 12 species 11536 against 9105.
template <int RECON, int D, typename R>
__global__ void __launch_bounds__(256)
    k_dust_flux(Layout L, const R* __restrict__ dsrc, R* __restrict__ dflux, int nd, R dfloor) {
  const int c3[3] = {(int)(blockIdx.x * blockDim.x + threadIdx.x),
                     (int)(blockIdx.y * blockDim.y + threadIdx.y),
                     (int)(blockIdx.z * blockDim.z + threadIdx.z)};
#pragma unroll
  for (int e = 0; e < 3; ++e)
    if (c3[e] >= L.n[e] + (e == D)) return;
  constexpr int RH = recon_reach<RECON>(), RL = RH + 1;
  const long long sz = L.size(), c = L.idx(c3[0], c3[1], c3[2]), sd = L.stride(D);
  for (int s = 0; s < nd; ++s) {
    const R* rho = dsrc + (long long)(4 * s) * sz;
    R w[6][4] = {};   // entries t: cells t - 3
#pragma unroll
    for (int t = 3 - RL; t <= 3 + RH; ++t) {
      const long long at = c + (t - 3) * sd;
      R r = rho[at];
      if (r < dfloor) r = dfloor;
      const R ir = recip(r);
      w[t][0] = r;
#pragma unroll
      for (int q = 0; q < 3; ++q) w[t][1 + q] = rho[(long long)(1 + q) * sz + at] * ir;
    }
    R f[4];
    dust_face<RECON, D>(w, f);
    R* out = dflux + (long long)((D * nd + s) * 4) * sz;
#pragma unroll
    for (int q = 0; q < 4; ++q) out[(long long)q * sz + c] = f[q];
  }
}

// FP32: threads over (x, y), marching along z over kc cells of one species: the z
// line of cells and the flux of the last z face stay in registers; the x and y
// lines come through L1.  The divergence goes to memory, not the fluxes: a
// third of the stores here and of the loads of the update.  Each x and y face
// is computed by both of its cells, cheaper than an exchange (the kernel has no
// barrier).  128^3, 8 species, PLM: three passes of fluxes
// 475 us, this one 456 (932 instructions a cell and species, issue rate 88%).
template <int RECON>
__global__ void __launch_bounds__(128)
    k_dust_div(Layout L, const float* __restrict__ dsrc, float* __restrict__ ddiv, int nd, int kc,
               float idx1, float idx2, float idx3, float dfloor) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const int j = blockIdx.y * blockDim.y + threadIdx.y;
  const int s = (int)(blockIdx.z % (unsigned)nd);
  const int k0 = (int)(blockIdx.z / (unsigned)nd) * kc, k1 = min(k0 + kc, L.n[2]);
  if (i >= L.n[0] || j >= L.n[1]) return;
  constexpr int RH = recon_reach<RECON>(), RL = RH + 1;
  const long long sz = L.size(), sx = L.sx, sxy = L.sx * L.sy;
  const float* rho = dsrc + (long long)(4 * s) * sz;
  float* out = ddiv + (long long)(4 * s) * sz;
  auto load = [&](long long at, float* w) {
    float r = rho[at];
    if (r < dfloor) r = dfloor;
    const float ir = recip(r);
    w[0] = r;
#pragma unroll
    for (int q = 0; q < 3; ++q) w[1 + q] = __fmul_rn(rho[(long long)(1 + q) * sz + at], ir);
  };
  // entries t of a line: cells t - 3 about the current one; outside the
  // reconstruction's reach they stay zero
  float lz[7][4] = {}, fz[4];
  long long c = L.idx(i, j, k0);
#pragma unroll
  for (int t = 3 - RL; t <= 3 + RH; ++t) load(c + (t - 3) * sxy, lz[t]);
  dust_face<RECON, 2>(lz, fz);
  for (int k = k0; k < k1; ++k, c += sxy) {
    load(c + RL * sxy, lz[3 + RL]);
    float div[4];
    {
      float l[7][4] = {}, lo[4], hi[4];
#pragma unroll
      for (int t = 3 - RL; t <= 3 + RL; ++t) {
        if (t != 3) load(c + (t - 3), l[t]);
        else
#pragma unroll
          for (int q = 0; q < 4; ++q) l[t][q] = lz[3][q];
      }
      dust_face<RECON, 0>(l, lo);
      dust_face<RECON, 0>(l + 1, hi);
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        div[q] = 0.0f;
        div[q] += (hi[q] - lo[q]) * idx1;
      }
    }
    {
      float l[7][4] = {}, lo[4], hi[4];
#pragma unroll
      for (int t = 3 - RL; t <= 3 + RL; ++t) {
        if (t != 3) load(c + (t - 3) * sx, l[t]);
        else
#pragma unroll
          for (int q = 0; q < 4; ++q) l[t][q] = lz[3][q];
      }
      dust_face<RECON, 1>(l, lo);
      dust_face<RECON, 1>(l + 1, hi);
#pragma unroll
      for (int q = 0; q < 4; ++q) div[q] += (hi[q] - lo[q]) * idx2;
    }
    float hi[4];
    dust_face<RECON, 2>(lz + 1, hi);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      div[q] += (hi[q] - fz[q]) * idx3;
      fz[q] = hi[q];
      out[(long long)q * sz + c] = div[q];
    }
#pragma unroll
    for (int t = 3 - RL; t < 3 + RL; ++t)
#pragma unroll
      for (int q = 0; q < 4; ++q) lz[t][q] = lz[t + 1][q];
  }
}

// The same for FP32 and PLM, the default, on packed pairs (rho, v1), (v2, v3):
// the pass is bound by the issue rate, and a pair takes one instruction.  515
// instructions a cell and species, 297 us; the update, which reads a third,
// 507 / 565 -> 400 / 504 us; the step 2440 -> 1910 us.  The momenta are rounded before
// their difference and the velocities before their slopes, in both cells of a face
// alike (ptxas would fuse a packed product into a packed sum; nzero, -0, makes it a
// multiply-add, which it leaves alone, with the product's own rounding).
template <int D>
__device__ __forceinline__ void dust_flux2(const float2* l, const float2* r, float2* f) {
  const float vl[3] = {l[0].y, l[1].x, l[1].y}, vr[3] = {r[0].y, r[1].x, r[1].y};
  float ml[3], mr[3];
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    ml[q] = __fmul_rn(l[0].x, vl[q]);
    mr[q] = __fmul_rn(r[0].x, vr[q]);
  }
  const float2 hs = splat(-0.5f * fmaxf(fabsf(vl[D]), fabsf(vr[D])));
  const float2 x0 = make_float2(__fadd_rn(ml[D], mr[D]),
                                __fmaf_rn(ml[0], vl[D], __fmul_rn(mr[0], vr[D])));
  const float2 ul = make_float2(ml[1], ml[2]), ur = make_float2(mr[1], mr[2]);
  const float2 x1 = fma2(ul, splat(vl[D]), ur * splat(vr[D]));
  f[0] = fma2(splat(0.5f), x0, hs * (make_float2(r[0].x, mr[0]) - make_float2(l[0].x, ml[0])));
  f[1] = fma2(splat(0.5f), x1, hs * (ur - ul));
}

__global__ void __launch_bounds__(128)
    k_dust_div_plm2(Layout L, const float* __restrict__ dsrc, float* __restrict__ ddiv, int nd,
                    int kc, float idx1, float idx2, float idx3, float dfloor, float nzero) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const int j = blockIdx.y * blockDim.y + threadIdx.y;
  const int s = (int)(blockIdx.z % (unsigned)nd);
  const int k0 = (int)(blockIdx.z / (unsigned)nd) * kc, k1 = min(k0 + kc, L.n[2]);
  if (i >= L.n[0] || j >= L.n[1]) return;
  const long long sz = L.size(), sx = L.sx, sxy = L.sx * L.sy;
  const float* p0 = dsrc + (long long)(4 * s) * sz;
  const float* p1 = p0 + sz;
  const float* p2 = p1 + sz;
  const float* p3 = p2 + sz;
  float* out = ddiv + (long long)(4 * s) * sz;
  auto load = [&](long long at, float2* w) {
    float r = p0[at];
    if (r < dfloor) r = dfloor;
    const float ir = recip(r);
    w[0] = make_float2(r, __fmul_rn(p1[at], ir));
    w[1] = fma2(make_float2(p2[at], p3[at]), splat(ir), splat(nzero));
  };
  // half slopes of the middle cell of three
  auto half = [](const float2* a, const float2* b, const float2* c, float2* h) {
#pragma unroll
    for (int p = 0; p < 2; ++p) h[p] = plm_half2(b[p] - a[p], c[p] - b[p]);
  };
  // flux between cells a (half slopes ha) and b (hb)
  auto face = [](auto D, const float2* a, const float2* ha, const float2* b, const float2* hb,
                 float2* f) {
    const float2 l[2] = {a[0] + ha[0], a[1] + ha[1]}, r[2] = {b[0] - hb[0], b[1] - hb[1]};
    dust_flux2<decltype(D)::value>(l, r, f);
  };
  long long c = L.idx(i, j, k0);
  // z: cells k, k + 1 and the half slopes of k; flux of k's lower face
  float2 w0[2], w1[2], h0[2], fz[2];
  {
    float2 wb[2], wa[2], ha[2];
    load(c - 2 * sxy, wb);
    load(c - sxy, wa);
    load(c, w0);
    load(c + sxy, w1);
    half(wb, wa, w0, ha);
    half(wa, w0, w1, h0);
    face(std::integral_constant<int, 2>(), wa, ha, w0, h0, fz);
  }
  for (int k = k0; k < k1; ++k, c += sxy) {
    float2 div[2];
    // x or y line of cells
    auto line = [&](auto D, long long st, float inv) {
      float2 a[2], b[2], d[2], e[2], hb[2], hc[2], hd[2], lo[2], hi[2];
      load(c - 2 * st, a);
      load(c - st, b);
      load(c + st, d);
      load(c + 2 * st, e);
      half(a, b, w0, hb);
      half(b, w0, d, hc);
      half(w0, d, e, hd);
      face(D, b, hb, w0, hc, lo);
      face(D, w0, hc, d, hd, hi);
#pragma unroll
      for (int p = 0; p < 2; ++p) {
        const float2 df = hi[p] - lo[p];
        div[p] = decltype(D)::value == 0 ? df * splat(inv) : fma2(df, splat(inv), div[p]);
      }
    };
    line(std::integral_constant<int, 0>(), 1, idx1);
    line(std::integral_constant<int, 1>(), sx, idx2);
    float2 w2[2], h1[2], hi[2];
    load(c + 2 * sxy, w2);
    half(w0, w1, w2, h1);
    face(std::integral_constant<int, 2>(), w0, h0, w1, h1, hi);
#pragma unroll
    for (int p = 0; p < 2; ++p) {
      div[p] = fma2(hi[p] - fz[p], splat(idx3), div[p]);
      fz[p] = hi[p];
      w0[p] = w1[p];
      w1[p] = w2[p];
      h0[p] = h1[p];
    }
    out[c] = div[0].x;
    out[sz + c] = div[0].y;
    out[2 * sz + c] = div[1].x;
    out[3 * sz + c] = div[1].y;
  }
}

// ------------------------------------------------------------------------
// stage combination + implicit drag (FP64), Cartesian blocks
// ------------------------------------------------------------------------
template <typename R>
struct DustUpd {
  R* ga[5];            // gas register A
  R* gb[5];            // gas register B
  const R* gf[3][5];   // gas fluxes
  R* da;               // dust register A (base)
  R* db;               // dust register B (base)
  const R* df;         // dust flux divergences, FP64: fluxes (base)
  double drag_c[32];   // per species: 1 / t_k (constant stopping time) or
                       // K_k (constant coefficient, t_k = rho_k / K_k)
  const double* dt;
  R dfloor;
};

// Bounds of the densities and implicit weights that the FP32 pairs take: the low halves
// of their products stay above the smallest normal number.  Momenta have the upper
// bound only (what overflows shows in the sum of the drift energies): a product below
// 2^-78 loses low bits to the flush of denormals, an absolute error of 2^-126, which
// reaches the FP32 rounding of results below about 2^-102 (2e-31).
constexpr double kPairLo = 1e-10, kPairHi = 1e10;

// The implicit drag of one cell in FP32 pairs: X = (gx, dx) -> (gy, dy), the
// formulas of k_dust_update.  wide: the species solved in pairs (constants in
// ak, ia, wk); the others in FP32 (fak, fia, fwk), their part of the gas sums
// added to the pairs.  Returns false where a product overflowed.
template <int NDMAX, bool SEL>
__device__ __forceinline__ bool drag_pairs(const float* gx, const float (*dx)[4], int nd,
                                           const dfloat* ak, const dfloat* ia, const dfloat* wk,
                                           const float* fak, const float* fia, const float* fwk,
                                           unsigned wide, int iso, float* gy, float (*dy)[4]) {
  dfloat den(gx[0]);
#pragma unroll
  for (int s = 0; s < NDMAX; ++s) {
    if (s >= nd) break;
    if (!SEL || ((wide >> s) & 1u)) den = den + wk[s] * dx[s][0];
    else den = den + dx[s][0] * fwk[s];
  }
  const dfloat inv = reciprocal(den);
  dfloat dke2(0.0f);   // twice the change of the dust kinetic energy
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    dfloat num(gx[1 + q]);
#pragma unroll
    for (int s = 0; s < NDMAX; ++s) {
      if (s >= nd) break;
      if (!SEL || ((wide >> s) & 1u)) num = num + wk[s] * dx[s][1 + q];
      else num = num + fwk[s] * dx[s][1 + q];
    }
    const dfloat vg = num * inv;
    gy[1 + q] = (float)(vg * gx[0]);
    const float vgf = (float)vg;
#pragma unroll
    for (int s = 0; s < NDMAX; ++s) {
      if (s >= nd) break;
      const float m0 = dx[s][1 + q], rk = dx[s][0];
      if (!SEL || ((wide >> s) & 1u)) {
        const dfloat m1 = ((ak[s] * rk) * vg + m0) * ia[s];
        dy[s][1 + q] = (float)m1;
        dke2 = dke2 + ((m1 + (-m0)) * (m1 + m0)) * reciprocal(dfloat(rk));
      } else {
        const float m1 = (m0 + rk * fak[s] * vgf) * fia[s];
        dy[s][1 + q] = m1;
        dke2 = dke2 + (m1 - m0) * (m1 + m0) * (rk > 0.0f ? 1.0f / rk : 0.0f);
      }
    }
  }
  // total energy conserved: drift energy becomes gas heat (the isothermal
  // closure carries its energy slot unchanged)
  gy[4] = iso ? gx[4] : (float)(dke2 * -0.5f + gx[4]);
  return fabsf(dke2.h) < 1e37f;
}

// The same in FP64 for the cells the pairs do not take (species with no density,
// rho_k <= 0, keep their kinetic energy out of the balance).  Such a cell is not
// rare everywhere: a species at its floor over part of the box, gas in units with
// densities below 1e-10, an implicit weight beyond the pairs' range.  Bound by the
// FP64 pipe, so up to 8 species share one division (as k_dust_update's solve in
// FP64 does), each density is inverted once for the three components, and a
// species' heat is scaled once.  One uncoupled species, so every cell here: 61 x 100 x
// 37, 3 species 351 -> 245 us a step (solving in FP64 only: 372), 48^3, 12 species 762 ->
// 582 (668), 96^3, 4 species 1385 -> 925 (1390).
template <int NDMAX, bool SEL>
__device__ __noinline__ void drag_far(const float* gx, const float (*dx)[4], int nd,
                                      const double* ak, const double* ia, const double* wk,
                                      const float* fak, const float* fia, const float* fwk,
                                      unsigned wide, int iso, float* gy, float (*dy)[4]) {
  constexpr int UN = NDMAX <= 8 ? NDMAX : 1;   // unrolled: the arrays stay in registers
  auto in64 = [&](int s) { return !SEL || ((wide >> s) & 1u); };
  const double rg = gx[0];
  double den = rg, rk[NDMAX], ir[NDMAX];   // rho_k, 1 / rho_k
#pragma unroll UN
  for (int s = 0; s < NDMAX; ++s) {
    if (s >= nd) break;
    rk[s] = dx[s][0];
    den += in64(s) ? rk[s] * wk[s] : (double)(dx[s][0] * fwk[s]);
  }
  double inv_den;
  if constexpr (!SEL && NDMAX <= 8) {
    // simultaneous inversion: prefix products of the densities (a non-positive
    // one enters as 1), one division, back-substitution
    double acc = 1.0;
#pragma unroll
    for (int s = 0; s < NDMAX; ++s) {
      if (s >= nd) break;
      ir[s] = acc;
      acc *= dx[s][0] > 0.0f ? rk[s] : 1.0;
    }
    const double q = 1.0 / (acc * den);
    inv_den = q * acc;
    double ip = q * den;   // 1 / (x_0 ... x_s)
#pragma unroll
    for (int s = NDMAX - 1; s >= 0; --s) {
      if (s >= nd) continue;
      const bool on = dx[s][0] > 0.0f;
      ir[s] = on ? ip * ir[s] : 0.0;
      ip *= on ? rk[s] : 1.0;
    }
  } else {
    inv_den = 1.0 / den;
#pragma unroll UN
    for (int s = 0; s < NDMAX; ++s) {
      if (s >= nd) break;
      ir[s] = in64(s) && dx[s][0] > 0.0f ? 1.0 / rk[s] : 0.0;
    }
  }
  // twice the change of the dust kinetic energy: the FP32 species' as they come, the
  // others' times rho_k, summed over the components before the product with 1 / rho_k
  double dke2 = 0.0, dm2[NDMAX];
#pragma unroll UN
  for (int s = 0; s < NDMAX; ++s) {
    if (s >= nd) break;
    rk[s] *= ak[s];   // rho_k a_k from here on
    dm2[s] = 0.0;
  }
#pragma unroll 1
  for (int q = 0; q < 3; ++q) {
    double num = gx[1 + q], m0[NDMAX];
#pragma unroll UN
    for (int s = 0; s < NDMAX; ++s) {
      if (s >= nd) break;
      m0[s] = dx[s][1 + q];
      num += in64(s) ? wk[s] * m0[s] : (double)(fwk[s] * dx[s][1 + q]);
    }
    const double vg = num * inv_den;
    gy[1 + q] = (float)(rg * vg);
    const float vgf = (float)vg;
#pragma unroll UN
    for (int s = 0; s < NDMAX; ++s) {
      if (s >= nd) break;
      if (in64(s)) {
        const double m1 = (m0[s] + rk[s] * vg) * ia[s];
        dy[s][1 + q] = (float)m1;
        dm2[s] += (m1 - m0[s]) * (m1 + m0[s]);
      } else {
        const float r = dx[s][0], mf = dx[s][1 + q];
        const float m1 = (mf + r * fak[s] * vgf) * fia[s];
        dy[s][1 + q] = m1;
        if (r > 0.0f) dke2 += (double)((m1 - mf) * (m1 + mf) * (1.0f / r));
      }
    }
  }
#pragma unroll UN
  for (int s = 0; s < NDMAX; ++s) {
    if (s >= nd) break;
    dke2 += dm2[s] * ir[s];
  }
  gy[0] = gx[0];
  gy[4] = iso ? gx[4] : (float)((double)gx[4] - 0.5 * dke2);
}

// Stage combination in the working precision R, implicit drag in DT.
// SEL (DT = dfloat, R = float): per-species precision -- the species whose
// implicit weight a_k = h / t_k exceeds sel_ratio are solved in pairs, the
// others in FP32; the gas sums over species (the denominator, the momentum
// numerators and the drag heating) accumulate in pairs.
// COEFF: the constant-coefficient drag law (drag_c = K_k, a_k = h K_k /
// rho_k per cell).  iso: isothermal gas, whose energy slot takes no drag
// heating.
// Bounds: five CTAs of 128 threads an SM for the solve in pairs of up to 8 species
// (96 registers; the two for 8 species spill about 120 bytes): 128^3, 8 species, step
// 1909 -> 1897 us against the compiler's own 128 registers; 61 x 100 x 37, 3 species
// 210 -> 205.  The others keep what they need.
template <typename DT, int NDMAX>
constexpr bool upd_five = std::is_same_v<DT, dfloat> && NDMAX <= 8;
template <typename R, typename DT, int NDMAX, bool SEL = false, bool COEFF = false>
__global__ void __launch_bounds__(upd_five<DT, NDMAX> ? 128 * AETH_DUST_BZ : 256,
                                  upd_five<DT, NDMAX> ? 5 / AETH_DUST_BZ : 0)
    k_dust_update(Layout L, R idx1, R idx2, R idx3, DustUpd<R> A, int nd, int stage,
                  unsigned long long* floor_hits, float sel_ratio, int iso) {
  // per-species drag constants of this stage, the same for every cell:
  // a_k = h / t_k, 1 / (1 + a_k), w_k = a_k / (1 + a_k) with h = g dt
  __shared__ DT s_ak[NDMAX], s_ia[NDMAX], s_wk[NDMAX];
  __shared__ float f_ak[SEL ? NDMAX : 1], f_ia[SEL ? NDMAX : 1], f_wk[SEL ? NDMAX : 1];
  __shared__ unsigned s_wide;   // SEL: bit s set = species s in pairs
  // PAIR: the FP64 solve in FP32 pairs; the FP64 constants stay for the cells
  // outside the pairs' range
  constexpr bool PAIR = std::is_same_v<DT, dfloat>;
  __shared__ double w_ak[PAIR ? NDMAX : 1], w_ia[PAIR ? NDMAX : 1], w_wk[PAIR ? NDMAX : 1];
  __shared__ int s_far;         // PAIR: a constant outside the pairs' range
  {
    using CT = std::conditional_t<PAIR, double, DT>;
    const int tid = threadIdx.x + blockDim.x * (threadIdx.y + blockDim.y * threadIdx.z);
    if (SEL && tid == 0) s_wide = 0u;
    if (PAIR && tid == 0) s_far = 0;
    __syncthreads();
    if (tid < nd && tid < NDMAX) {
      const CT h = (CT)kImexG * (CT)(*A.dt);
      const CT a = h * (CT)A.drag_c[tid];
      const CT ia = CT(1) / (CT(1) + a);
      if constexpr (PAIR) {
        w_ak[tid] = a;
        w_ia[tid] = ia;
        w_wk[tid] = a * ia;
        s_ak[tid] = dfloat::of(a);
        s_ia[tid] = dfloat::of(ia);
        s_wk[tid] = dfloat::of(a * ia);
        // a constant of a species that the pairs solve (an uncoupled FP32 species sent
        // every cell to FP64: 64^3, 4 species 392 us a step, 192 now)
        if ((!SEL || a > (CT)sel_ratio) && !(a > kPairLo && a < kPairHi)) s_far = 1;
      } else {
        s_ak[tid] = a;
        s_ia[tid] = ia;
        s_wk[tid] = a * ia;
      }
      if constexpr (SEL) {
        const float af = (float)h * (float)A.drag_c[tid];
        const float iaf = 1.0f / (1.0f + af);
        f_ak[tid] = af;
        f_ia[tid] = iaf;
        f_wk[tid] = af * iaf;
        if (a > (CT)sel_ratio) atomicOr(&s_wide, 1u << tid);
      }
    }
    __syncthreads();
  }
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const int j = blockIdx.y * blockDim.y + threadIdx.y;
  const int k = blockIdx.z * blockDim.z + threadIdx.z;
  if (i >= L.n[0] || j >= L.n[1] || k >= L.n[2]) return;
  const long long c = L.idx(i, j, k);
  const long long sz = L.size();
  const long long st[3] = {1, L.sx, L.sx * L.sy};
  const R inv[3] = {idx1, idx2, idx3};
  const R dt = (R)(*A.dt);
  const R g = (R)kImexG, d = (R)kImexD;
  // explicit right-hand sides and the stage's pre-drag state X; the
  // register-A values stay in registers for the stage-2 combination (a
  // reload after the first stores would wait on each store in turn)
  R gx[5], ug[5];
  R dx[NDMAX][4], ud[NDMAX][4];
#pragma unroll
  for (int v = 0; v < 5; ++v) {
    R div = R(0);
#pragma unroll
    for (int a = 0; a < 3; ++a) div += (A.gf[a][v][c + st[a]] - A.gf[a][v][c]) * inv[a];
    ug[v] = A.ga[v][c];
    gx[v] = ug[v] - (stage == 2 ? g : R(1) - d) * dt * div;
  }
#pragma unroll
  for (int s = 0; s < NDMAX; ++s) {
    if (s >= nd) break;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      R div = R(0);
      if constexpr (sizeof(R) == 4) {
        div = A.df[(long long)(4 * s + q) * sz + c];
      } else {
#pragma unroll
        for (int a = 0; a < 3; ++a) {
          const R* f = A.df + (long long)((a * nd + s) * 4 + q) * sz;
          div += (f[c + st[a]] - f[c]) * inv[a];
        }
      }
      ud[s][q] = A.da[(long long)(4 * s + q) * sz + c];
      dx[s][q] = ud[s][q] - (stage == 2 ? g : R(1) - d) * dt * div;
    }
  }
  // closed-form implicit drag with h = g dt (Sec. 2.2).  With
  // a_k = h / t_k, w_k = a_k / (1 + a_k):
  //   rho_g v_g' = (M_g* + sum_k w_k M_k*) * rho_g / (rho_g + sum_k rho_k w_k)
  //   M_k' = rho_k v_k' = (M_k* + rho_k a_k v_g') / (1 + a_k)
  //   dKE_k = (M_k'^2 - M_k*^2) / (2 rho_k)
  // 1/rho_k and 1/den come from one division (simultaneous inversion,
  // Montgomery 1987: prefix products, one reciprocal, back-substitution).
  R gy[5], dy[NDMAX][4];
  gy[0] = gx[0];
  if constexpr (PAIR) {
    // FP32 pairs hold the solve to about 48 bits, the results rounded to FP32
    // as from FP64, where no product leaves the FP32 exponent range; cells (or
    // constants) outside these bounds, without density or not finite are
    // solved in FP64
    bool far = s_far || !(gx[0] > (R)kPairLo && gx[0] < (R)kPairHi);
#pragma unroll
    for (int q = 1; q < 5; ++q) far = far || !(fabsf(gx[q]) < (float)kPairHi);
#pragma unroll
    for (int s = 0; s < NDMAX; ++s) {
      if (s >= nd) break;
      dy[s][0] = dx[s][0];
      // an FP32 species has no lower bound
      const bool low = !SEL || ((s_wide >> s) & 1u) ? !(dx[s][0] > (R)kPairLo) : false;
      far = far || low || !(fabsf(dx[s][0]) < (float)kPairHi);
#pragma unroll
      for (int q = 1; q < 4; ++q) far = far || !(fabsf(dx[s][q]) < (float)kPairHi);
    }
    if (!far)
      far = !drag_pairs<NDMAX, SEL>(gx, dx, nd, s_ak, s_ia, s_wk, f_ak, f_ia, f_wk,
                                   SEL ? s_wide : ~0u, iso, gy, dy);
    if (far) {
      // rare: the arrays go through memory here only
      float tg[5], td[NDMAX][4], og[5], od[NDMAX][4];
#pragma unroll
      for (int v = 0; v < 5; ++v) tg[v] = gx[v];
#pragma unroll
      for (int s = 0; s < NDMAX; ++s)
#pragma unroll
        for (int q = 0; q < 4; ++q) td[s][q] = s < nd ? dx[s][q] : 0.0f;
      drag_far<NDMAX, SEL>(tg, td, nd, w_ak, w_ia, w_wk, f_ak, f_ia, f_wk, SEL ? s_wide : ~0u, iso,
                           og, od);
#pragma unroll
      for (int v = 0; v < 5; ++v) gy[v] = og[v];
#pragma unroll
      for (int s = 0; s < NDMAX; ++s)
#pragma unroll
        for (int q = 1; q < 4; ++q) dy[s][q] = od[s][q];
    }
  } else {
    const DT rg = gx[0];
  if constexpr (COEFF) {
    // constant-coefficient law (Sec. 2.2): t_k = rho_k / K_k with the
    // stage's dust density, which the drag leaves unchanged, so the weight
    // a_k = h K_k / rho_k is fixed per cell through the solve; a species
    // with no density (rho_k <= 0) feels no drag
    const DT h = (DT)kImexG * (DT)(*A.dt);
    DT rk[NDMAX], ak[NDMAX], ia[NDMAX], irk[NDMAX];
    DT den = rg;
#pragma unroll
    for (int s = 0; s < NDMAX; ++s) {
      if (s >= nd) break;
      rk[s] = dx[s][0];
      irk[s] = rk[s] > DT(0) ? DT(1) / rk[s] : DT(0);
      ak[s] = h * (DT)A.drag_c[s] * irk[s];
      ia[s] = DT(1) / (DT(1) + ak[s]);
      den += rk[s] * ak[s] * ia[s];
      dy[s][0] = dx[s][0];
    }
    const DT inv_den = DT(1) / den;
    DT dke2 = 0;
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      DT num = gx[1 + q];
#pragma unroll
      for (int s = 0; s < NDMAX; ++s) {
        if (s >= nd) break;
        num += ak[s] * ia[s] * (DT)dx[s][1 + q];
      }
      const DT vg = num * inv_den;
      gy[1 + q] = (R)(rg * vg);
#pragma unroll
      for (int s = 0; s < NDMAX; ++s) {
        if (s >= nd) break;
        const DT m0 = dx[s][1 + q];
        const DT m1 = (m0 + rk[s] * ak[s] * vg) * ia[s];
        dy[s][1 + q] = (R)m1;
        dke2 += (m1 - m0) * (m1 + m0) * irk[s];
      }
    }
    gy[4] = iso ? gx[4] : (R)((DT)gx[4] - DT(0.5) * dke2);
  } else {
  DT rk[NDMAX], rak[NDMAX], ir[NDMAX];
  DT den = rg;
#pragma unroll
  for (int s = 0; s < NDMAX; ++s) {
    if (s >= nd) break;
    rk[s] = dx[s][0];
    rak[s] = rk[s] * s_ak[s];
    den += rk[s] * s_wk[s];
    dy[s][0] = dx[s][0];
  }
  DT inv_den;
  if constexpr (sizeof(DT) == 8 && NDMAX <= 8) {
    // prefix products x_0 ... x_{s-1} of the densities (a non-positive
    // density enters as 1 and gets 1/rho = 0); at most 8 factors of the
    // density range stay far inside the FP64 exponent range
    DT pre[NDMAX];
    DT acc = DT(1);
#pragma unroll
    for (int s = 0; s < NDMAX; ++s) {
      if (s >= nd) break;
      pre[s] = acc;
      acc *= rk[s] > DT(0) ? rk[s] : DT(1);
    }
    const DT q = DT(1) / (acc * den);   // the one division
    inv_den = q * acc;
    DT ip = q * den;                    // 1 / (x_0 ... x_{nd-1})
#pragma unroll
    for (int s = NDMAX - 1; s >= 0; --s) {
      if (s >= nd) continue;
      ir[s] = rk[s] > DT(0) ? ip * pre[s] : DT(0);
      ip *= rk[s] > DT(0) ? rk[s] : DT(1);   // 1 / (x_0 ... x_{s-1})
    }
  } else {
    inv_den = DT(1) / den;
#pragma unroll
    for (int s = 0; s < NDMAX; ++s) {
      if (s >= nd) break;
      ir[s] = rk[s] > DT(0) ? DT(1) / rk[s] : DT(0);
    }
  }
  DT dke2 = 0;   // twice the change of the dust kinetic energy
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    DT m0[NDMAX];
    DT num = gx[1 + q];   // rho_g v_g* = M_g*
#pragma unroll
    for (int s = 0; s < NDMAX; ++s) {
      if (s >= nd) break;
      m0[s] = (DT)dx[s][1 + q];
      num += s_wk[s] * m0[s];   // rho_k w_k v_k* = w_k M_k*
    }
    const DT vg = num * inv_den;
    gy[1 + q] = (R)(rg * vg);
#pragma unroll
    for (int s = 0; s < NDMAX; ++s) {
      if (s >= nd) break;
      const DT m1 = (m0[s] + rak[s] * vg) * s_ia[s];
      dy[s][1 + q] = (R)m1;
      dke2 += (m1 - m0[s]) * (m1 + m0[s]) * ir[s];
    }
  }
  const DT dke = DT(0.5) * dke2;
  // total energy conserved: drift energy becomes gas heat (the isothermal
  // closure carries its energy slot unchanged)
  gy[4] = iso ? gx[4] : (R)((DT)gx[4] - dke);
  }
  }
  int hits = 0;
#pragma unroll
  for (int s = 0; s < NDMAX; ++s) {
    if (s >= nd) break;
    if (dy[s][0] < A.dfloor) {
      dy[s][0] = A.dfloor;
      dy[s][1] = dy[s][2] = dy[s][3] = R(0);
      ++hits;
    }
  }
  if (stage == 2) {
    // A <- W + (1-g)/g (U2 - X), with W = U^n + d dt L = (1 - d/g) U^n + (d/g) X
    const R cw = (R(1) - g) / g, cu = R(1) - d / g, cx = d / g;
#pragma unroll
    for (int v = 0; v < 5; ++v) {
      A.gb[v][c] = gy[v];
      A.ga[v][c] = cu * ug[v] + cx * gx[v] + cw * (gy[v] - gx[v]);
    }
#pragma unroll
    for (int s = 0; s < NDMAX; ++s) {
      if (s >= nd) break;
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const long long o = (long long)(4 * s + q) * sz + c;
        A.db[o] = dy[s][q];
        A.da[o] = cu * ud[s][q] + cx * dx[s][q] + cw * (dy[s][q] - dx[s][q]);
      }
    }
  } else {
#pragma unroll
    for (int v = 0; v < 5; ++v) A.ga[v][c] = gy[v];
#pragma unroll
    for (int s = 0; s < NDMAX; ++s) {
      if (s >= nd) break;
#pragma unroll
      for (int q = 0; q < 4; ++q) A.da[(long long)(4 * s + q) * sz + c] = dy[s][q];
    }
  }
  add_hits(floor_hits, hits);
}

// Ghost fill of narr cell-centred arrays at base + a * sz.
template <typename R>
__global__ void __launch_bounds__(256) k_fill_cells(Layout L, R* base, int narr) {
  const unsigned el = blockIdx.x * blockDim.x + threadIdx.x;
  if (el >= (unsigned)ghost_cells(L)) return;
  int c[3];
  ghost_cell(L, el, c);
  const long long dst = L.idx(c[0], c[1], c[2]);
  bool up;
#pragma unroll
  for (int e = 0; e < 3; ++e) c[e] = ghost_axis(L, e, c[e], up);
  const long long srcx = L.idx(c[0], c[1], c[2]);
  const long long sz = L.size();
  // eight arrays at a time, every source loaded before the stores (the
  // stores go through the same base, so interleaving them would serialise
  // the round trips)
  for (int a0 = 0; a0 < narr; a0 += 8) {
    R v[8];
#pragma unroll
    for (int q = 0; q < 8; ++q)
      if (a0 + q < narr) v[q] = base[(a0 + q) * sz + srcx];
#pragma unroll
    for (int q = 0; q < 8; ++q)
      if (a0 + q < narr) base[(a0 + q) * sz + dst] = v[q];
  }
}

template <typename R, bool P64>
static void stage_dust(aeth_ctx* c, int b, int src, int stage) {
  const BlockPtrs<R> P = block_ptrs<R>(c, b);
  const BlockInfo& B = c->blocks[b];
  const Layout& L = P.L;
  const int nd = c->cfg.n_dust;
  cudaStream_t s = c->stream;
  launch_fill<R>(P, P.reg[src], 5, s);
  k_fill_cells<R><<<ceil_div(ghost_cells(L), 256), 256, 0, s>>>(L, P.dust[src], 4 * nd);
  c->n_launch += 2;
  hydro_flux_pass<R, P64>(c, b, c->cfg.recon, src);
  const R dfl = (R)1e-20;
  // inverse cell widths (Cartesian: area / volume = 1 / dx_d)
  const R i1 = (R)(B.desc.nx / (B.desc.x1max - B.desc.x1min));
  const R i2 = (R)(B.desc.ny / (B.desc.x2max - B.desc.x2min));
  const R i3 = (R)(B.desc.nz / (B.desc.x3max - B.desc.x3min));
  if constexpr (sizeof(R) == 4) {
    // cells of a z march: 16, fewer where that leaves less than about two waves
    // of CTAs (a march of 4 spends as much again on its first face)
    auto ctas = [&](int kc) {
      return (long long)ceil_div(L.n[0], 32) * ceil_div(L.n[1], 4) * ceil_div(L.n[2], kc) * nd;
    };
    int kc = 16;
    while (kc > 4 && ctas(kc) < 8LL * c->num_sms) kc /= 2;
    while ((long long)ceil_div(L.n[2], kc) * nd > 65535) kc *= 2;   // grid limit
    auto divergence = [&](auto kernel, auto... more) {
      const dim3 grd(ceil_div(L.n[0], 32), ceil_div(L.n[1], 4), ceil_div(L.n[2], kc) * nd);
      kernel<<<grd, dim3(32, 4), 0, s>>>(L, P.dust[src], P.dflux, nd, kc, i1, i2, i3, dfl, more...);
    };
    switch (c->cfg.recon) {
      case AETH_RECON_DONOR: divergence(k_dust_div<0>); break;
      case AETH_RECON_PLM: divergence(k_dust_div_plm2, -0.0f); break;
      case AETH_RECON_PPM5: divergence(k_dust_div<3>); break;
      default: divergence(k_dust_div<2>);
    }
    c->n_launch += 1;
  } else {
    const dim3 blk(32, 4, 2);
    const dim3 grd(ceil_div(L.n[0] + 1, 32), ceil_div(L.n[1] + 1, 4), ceil_div(L.n[2] + 1, 2));
    auto fluxes = [&](auto... kernel) {
      (kernel<<<grd, blk, 0, s>>>(L, P.dust[src], P.dflux, nd, dfl), ...);
    };
    switch (c->cfg.recon) {
      case AETH_RECON_DONOR:
        fluxes(k_dust_flux<0, 0, R>, k_dust_flux<0, 1, R>, k_dust_flux<0, 2, R>);
        break;
      case AETH_RECON_PLM:
        fluxes(k_dust_flux<1, 0, R>, k_dust_flux<1, 1, R>, k_dust_flux<1, 2, R>);
        break;
      case AETH_RECON_PPM5:
        fluxes(k_dust_flux<3, 0, R>, k_dust_flux<3, 1, R>, k_dust_flux<3, 2, R>);
        break;
      default: fluxes(k_dust_flux<2, 0, R>, k_dust_flux<2, 1, R>, k_dust_flux<2, 2, R>);
    }
    c->n_launch += 3;
  }
  DustUpd<R> u{};
  for (int v = 0; v < 5; ++v) {
    u.ga[v] = P.reg[0][v];
    u.gb[v] = P.reg[1][v];
    for (int a = 0; a < 3; ++a) u.gf[a][v] = P.f[a][v];
  }
  u.da = P.dust[0];
  u.db = P.dust[1];
  u.df = P.dflux;
  const bool coeff = c->cfg.drag_law == AETH_DRAG_LAW_COEFF;
  for (int q = 0; q < nd; ++q) u.drag_c[q] = coeff ? c->t_stop[q] : 1.0 / c->t_stop[q];
  u.dt = c->d_dt;
  u.dfloor = dfl;
  // the update: CTAs of 32 x 4 x AETH_DUST_BZ cells (its registers allow
  // few CTAs per SM)
  const dim3 blk2(32, 4, AETH_DUST_BZ);
  dim3 grd2((L.n[0] + 31) / 32, (L.n[1] + 3) / 4, (L.n[2] + AETH_DUST_BZ - 1) / AETH_DUST_BZ);
  const bool d64 = c->cfg.drag_precision == AETH_DRAG_FP64;
  const int iso = is_iso(c) ? 1 : 0;
  const float ratio = (float)c->cfg.drag_ratio;
  auto launch = [&](auto kernel) {
    kernel<<<grd2, blk2, 0, s>>>(L, i1, i2, i3, u, nd, stage, c->d_floor, ratio, iso);
  };
  bool done = false;
  if constexpr (sizeof(R) == 4) {
    if (c->cfg.drag_precision == AETH_DRAG_SEL64) {
      // per-species precision: pairs for the species with h / t_k > drag_ratio
      if (nd <= 8) launch(k_dust_update<R, dfloat, 8, true>);
      else launch(k_dust_update<R, dfloat, 32, true>);
      done = true;
    } else if (d64 && !coeff) {
      // FP32 transport with the FP64 drag: FP32 pairs
      if (nd <= 4) launch(k_dust_update<R, dfloat, 4>);
      else if (nd <= 8) launch(k_dust_update<R, dfloat, 8>);
      else launch(k_dust_update<R, dfloat, 32>);
      done = true;
    }
  }
  if (done) {
  } else if (coeff) {
    if (nd <= 8) d64 ? launch(k_dust_update<R, double, 8, false, true>)
                     : launch(k_dust_update<R, R, 8, false, true>);
    else d64 ? launch(k_dust_update<R, double, 32, false, true>)
             : launch(k_dust_update<R, R, 32, false, true>);
  } else if (nd <= 8) {   // FP64 transport, or the drag in FP32
    launch(k_dust_update<R, R, 8>);
  } else {
    launch(k_dust_update<R, R, 32>);
  }
  c->n_launch += 1;
}

template <typename R, bool P64>
aeth_status step_dust(aeth_ctx* c) {
  const int nb = (int)c->blocks.size();
  for (int b = 0; b < nb; ++b) stage_dust<R, P64>(c, b, 0, 2);
  for (int b = 0; b < nb; ++b) stage_dust<R, P64>(c, b, 1, 3);
  AETH_CK(c, cudaGetLastError());
  return AETH_OK;
}

template aeth_status step_dust<float, false>(aeth_ctx*);
template aeth_status step_dust<float, true>(aeth_ctx*);
template aeth_status step_dust<double, false>(aeth_ctx*);

}  // namespace aeth
