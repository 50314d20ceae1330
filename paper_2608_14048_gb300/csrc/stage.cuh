// Per-cell helpers shared by the stage kernels (fused flux pass, learned
// flux): primitive recovery and stencil reconstruction.
#pragma once
#include "runtime.hpp"

namespace aeth {

// Primitive variables (Eq. 5 with the floors of Sec. 2.1) from the conserved
// values u = (rho, M1, M2, M3, E) and the cell-centred field b:
// w = (rho, v1, v2, v3, p, Bc1, Bc2, Bc3).  Returns the number of floors hit.
// ISO: isothermal closure, p = gm1 * rho with gm1 holding cs^2 (the energy
// entry is not used and no pressure floor applies).
template <typename R, bool P64, bool ISO>
__device__ __forceinline__ int prim_values(float p64_ratio, const R* u, const R* b, R gm1,
                                           R rho_floor, R p_floor, R* w) {
  int hits = 0;
  R rho = u[0];
  if (rho < rho_floor) { rho = rho_floor; ++hits; }
  const R ir = recip(rho);
  const R v1 = u[1] * ir, v2 = u[2] * ir, v3 = u[3] * ir;
  R pr;
  if (ISO) {
    pr = gm1 * rho;
  } else if (P64) {
    // FP64 subtraction of Eq. 5 in every cell, or (p64_ratio > 0) only where
    // the FP32 one would cancel: kinetic + magnetic > ratio x internal
    bool wide = true;
    if (p64_ratio > 0.0f) {
      const R ke = R(0.5) * rho * (v1 * v1 + v2 * v2 + v3 * v3);
      const R me = R(0.5) * (b[0] * b[0] + b[1] * b[1] + b[2] * b[2]);
      const R ei = u[4] - ke - me;
      wide = ke + me > (R)p64_ratio * ei;
      pr = gm1 * ei;
    }
    if (wide) {
      const double m1 = u[1], m2 = u[2], m3 = u[3];
      const double ke = 0.5 * (m1 * m1 + m2 * m2 + m3 * m3) / (double)rho;
      const double me = 0.5 * ((double)b[0] * b[0] + (double)b[1] * b[1] + (double)b[2] * b[2]);
      pr = (R)((double)gm1 * ((double)u[4] - ke - me));
    }
  } else {
    pr = gm1 * (u[4] - R(0.5) * rho * (v1 * v1 + v2 * v2 + v3 * v3) -
                R(0.5) * (b[0] * b[0] + b[1] * b[1] + b[2] * b[2]));
  }
  if (!ISO && pr < p_floor) { pr = p_floor; ++hits; }
  w[0] = rho; w[1] = v1; w[2] = v2; w[3] = v3; w[4] = pr; w[5] = b[0]; w[6] = b[1]; w[7] = b[2];
  return hits;
}

// Dual energy (Sec. 2.8): the same with the pressure from the entropy S where
// the internal energy from E is below alpha_switch times the kinetic plus
// magnetic energy, else from E; sp = S / rho, the specific entropy the faces
// reconstruct.
template <typename R>
__device__ __forceinline__ int prim_values_dual(const R* u, const R* b, R S, R gm1, R rho_floor,
                                                R p_floor, R alpha_switch, R* w, R& sp) {
  int hits = 0;
  R rho = u[0];
  if (rho < rho_floor) { rho = rho_floor; ++hits; }
  const R ir = recip(rho);
  const R v1 = u[1] * ir, v2 = u[2] * ir, v3 = u[3] * ir;
  // the internal energy in the same arithmetic as prim_values, so that a run
  // whose cells all trust E reproduces the plain run bit for bit
  const R ke = R(0.5) * rho * (v1 * v1 + v2 * v2 + v3 * v3);
  const R me = R(0.5) * (b[0] * b[0] + b[1] * b[1] + b[2] * b[2]);
  const R eint = u[4] - ke - me;
  R pr = eint < alpha_switch * (ke + me) ? S * pow(rho, gm1) : gm1 * eint;
  if (pr < p_floor) { pr = p_floor; ++hits; }
  w[0] = rho; w[1] = v1; w[2] = v2; w[3] = v3; w[4] = pr; w[5] = b[0]; w[6] = b[1]; w[7] = b[2];
  sp = S * ir;
  return hits;
}

// Conserved values and cell-centred field of cell c of the state arrays u.
template <typename R, bool MHD, typename Arr>
__device__ __forceinline__ void load_cell(long long sx, long long plane, const Arr& u, long long c,
                                          bool energy, R* x, R* b) {
#pragma unroll
  for (int v = 0; v < 4; ++v) x[v] = u.p[v][c];
  x[4] = energy ? u.p[4][c] : R(0);
  b[0] = b[1] = b[2] = R(0);
  if (MHD) {
    b[0] = R(0.5) * (u.p[5][c] + u.p[5][c + 1]);
    b[1] = R(0.5) * (u.p[6][c] + u.p[6][c + sx]);
    b[2] = R(0.5) * (u.p[7][c] + u.p[7][c + plane]);
  }
}

// Primitives of cell c of the state arrays u.
template <typename R, bool P64, bool MHD, bool ISO = false>
__device__ __forceinline__ int prim_cell(const Layout& L, const ConstArr8<R>& u, long long c,
                                         R gm1, R rho_floor, R p_floor, R* w) {
  R x[5], b[3];
  load_cell<R, MHD>(L.sx, L.sx * L.sy, u, c, !ISO, x, b);
  return prim_values<R, P64, ISO>(L.p64_ratio, x, b, gm1, rho_floor, p_floor, w);
}

// Same, with the 8 state arrays at base + v * pitch.
template <typename R, bool P64, bool MHD, bool ISO = false>
__device__ __forceinline__ int prim_cell_s(const Layout& L, const R* __restrict__ base,
                                           long long pitch, long long c, R gm1, R rho_floor,
                                           R p_floor, R* w) {
  ConstArr8<R> u;
#pragma unroll
  for (int v = 0; v < NVAR; ++v) u.p[v] = base + v * pitch;
  return prim_cell<R, P64, MHD, ISO>(L, u, c, gm1, rho_floor, p_floor, w);
}

// Reconstruct face states of one variable from a stencil with stride.
template <int RECON, typename R, typename Get>
__device__ __forceinline__ void recon_var(Get get, R& wl, R& wr) {
  constexpr int RH = recon_reach<RECON>(), RL = RH + 1;
  R s[6];
#pragma unroll
  for (int t = 0; t < 6; ++t) {
    const int off = t - 3;   // cell offset from the face's right cell
    s[t] = (off >= -RL && off <= RH) ? get(off) : R(0);
  }
  recon_face<RECON>(s, wl, wr);
}

}  // namespace aeth
