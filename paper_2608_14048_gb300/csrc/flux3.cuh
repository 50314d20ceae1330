// Flux pass of the fused stage (Sec. 2.4): conserved->primitive,
// reconstruction and the Riemann solver for all three face directions of
// every cell in one sweep.  A CTA owns a TX x TY column tile and marches
// along z: each x-y plane of primitives (with the reconstruction halo) is
// staged in a ring of shared-memory planes for the x- and y-faces, while
// every thread keeps the z-stencil of its own column in a register queue
// for the z-faces, filled from the ring.
// Each face is solved exactly once.  Outputs: hydro fluxes, face EMFs (the
// transverse induction fluxes) and the cell-centred reference EMF of the
// upwind CT scheme.
//
// The kernel template lives here so that its instantiations (one per
// Riemann solver family) compile in separate translation units.
#pragma once
#include "riemann2.cuh"
#include "runtime.hpp"
#include "stage.cuh"

namespace aeth {

// resident CTAs per SM requested for the FP32 flux pass with donor or PLM
// reconstruction, in 256-thread units (register budget 65536 / (256 *
// FLUX_MINB) per thread: 3, 85 registers, measured 1.3% faster at 256^3
// than 2 with 106 registers); the PPM and PPM5 stencils keep 2 (at 85
// registers they spill about 250 bytes per thread); FP64 takes the whole
// register file.  A 128-thread tile counts half.
#ifndef AETH_FLUX_MINB
#define AETH_FLUX_MINB 3
#endif
// the same for the 128-thread 2-D tiles, in CTAs: 5 (the PLM corrector at
// 96 registers with a 20-byte spill) measured 1% faster at 256^3 than 6
// (80 registers, 160 bytes spilled); PPM keeps 4
#ifndef AETH_FLUX_MINB_2D
#define AETH_FLUX_MINB_2D 5
#endif
#ifndef AETH_FLUX_MINB_2D_PPM
#define AETH_FLUX_MINB_2D_PPM 4
#endif
template <typename R, int RECON>
__host__ __device__ constexpr int flux_minb(int txt) {
  return txt == 0 ? (sizeof(R) == 4 ? (RECON >= 2 ? 2 : AETH_FLUX_MINB) : 1)
                  : (sizeof(R) == 4 ? (RECON >= 2 ? AETH_FLUX_MINB_2D_PPM : AETH_FLUX_MINB_2D) : 2);
}

// a compile-time direction as an argument
template <int V>
struct Int {
  static constexpr int value = V;
};

__host__ __device__ __forceinline__ int ceil_div_d(int a, int b) { return (a + b - 1) / b; }

// Shared-memory plane (one variable, tile + halo) of a band tile (TXT = 0,
// see band_rows): the largest (rows + halo) x (width + halo) over the
// widths a band tile takes, so that its stride is a compile-time constant.
__host__ __device__ constexpr int band_smem(int halo) {
  int m = 0;
  for (int w = 3; w <= FLUX_BAND_WMAX; ++w) {
    const int a = (band_rows(w - 2) + halo) * (w + halo);
    m = a > m ? a : m;
  }
  return m;
}

// Cells of one staged plane of a flux tile TXT wide (0: band), rounded up to
// a multiple of 4 so that every plane of quads starts on a 16-byte boundary
// whatever the number of words staged per cell.
template <int RECON>
__host__ __device__ constexpr int flux_plane(int txt) {
  const int n = txt ? (txt + 2 * recon_reach<RECON>() + 1) * (FLUX_NT / txt + 2 * recon_reach<RECON>() + 1)
                    : band_smem(2 * recon_reach<RECON>() + 1);
  return (n + 3) / 4 * 4;
}

// Planes in the shared-memory ring of a 2-D flux tile: the z-queue takes
// plane k + RH while the x- and y-faces read plane k, and the next plane is
// staged while slower warps still read plane k - 1.  Band tiles stage one
// plane at a time (two barriers per plane, the z queue from memory): on the
// small blocks they serve, the ring's larger shared-memory footprint cost
// more in L1 hits than its one barrier per plane saved.
template <int RECON>
__host__ __device__ constexpr int flux_ring(int txt) { return txt ? recon_reach<RECON>() + 2 : 1; }

// Solver families 3 and 4 are the isothermal ones.
constexpr bool iso_solver(int solver) { return solver == 3 || solver == 4; }

// Riemann solver family SOLVER (numbering of k_flux3 below) on one face, the
// states as 7 values a side (FP64) or as packed pairs (FP32).
template <int SOLVER, bool MHD>
__device__ __forceinline__ void solve_face(double g, double, const double* wl, const double* wr,
                                           double bn, double* fx) {
  if constexpr (SOLVER == 2) hlle(g, wl, wr, bn, fx);
  else if constexpr (SOLVER == 3) hlld_iso(g, wl, wr, bn, fx);
  else if constexpr (SOLVER == 4) hlle_iso(g, wl, wr, bn, fx);
  else if constexpr (SOLVER == 5) hlld<true>(g, wl, wr, bn, fx);
  else hlld(g, wl, wr, bn, fx);
}
template <int SOLVER, bool MHD>
__device__ __forceinline__ void solve_face(float g, float igm1, const float* wl, const float* wr,
                                           float bn, float* fx) {
  float2 W[7];
#pragma unroll
  for (int v = 0; v < 7; ++v) W[v] = make_float2(wl[v], wr[v]);
  if constexpr (SOLVER == 2) hlle2<MHD, false>(g, igm1, W, bn, fx);
  else if constexpr (SOLVER == 3) hlld_iso2<MHD>(g * g, W, bn, fx);
  else if constexpr (SOLVER == 4) hlle2<MHD, true>(g * g, igm1, W, bn, fx);
  else if constexpr (SOLVER == 5) hlld2<true, MHD>(g, igm1, W, bn, fx);
  else hlld2<false, MHD>(g, igm1, W, bn, fx);
}

// Four staged values of a cell (16-byte shared accesses in FP32).
template <typename R>
struct Quad {
  R v[4];
};
__device__ __forceinline__ Quad<float> ld_quad(const float* p) {
  const float4 t = *reinterpret_cast<const float4*>(p);
  return {{t.x, t.y, t.z, t.w}};
}
__device__ __forceinline__ Quad<double> ld_quad(const double* p) {
  const double2 a = *reinterpret_cast<const double2*>(p), b = *reinterpret_cast<const double2*>(p + 2);
  return {{a.x, a.y, b.x, b.y}};
}
__device__ __forceinline__ void st_quad(float* p, float a, float b, float c, float d) {
  *reinterpret_cast<float4*>(p) = make_float4(a, b, c, d);
}
__device__ __forceinline__ void st_quad(double* p, double a, double b, double c, double d) {
  *reinterpret_cast<double2*>(p) = make_double2(a, b);
  *reinterpret_cast<double2*>(p + 2) = make_double2(c, d);
}

// Half the van Leer slopes of four variables of a cell (PLM).
__device__ __forceinline__ Quad<float> plm_half(const Quad<float>& m, const Quad<float>& c,
                                                const Quad<float>& p) {
  Quad<float> t;
#pragma unroll
  for (int q = 0; q < 4; q += 2) {
    const float2 x = make_float2(c.v[q], c.v[q + 1]);
    const float2 h = plm_half2(x - make_float2(m.v[q], m.v[q + 1]), make_float2(p.v[q], p.v[q + 1]) - x);
    t.v[q] = h.x;
    t.v[q + 1] = h.y;
  }
  return t;
}
__device__ __forceinline__ Quad<double> plm_half(const Quad<double>& m, const Quad<double>& c,
                                                 const Quad<double>& p) {
  Quad<double> t;
#pragma unroll
  for (int q = 0; q < 4; ++q) t.v[q] = 0.5 * vl_slope(m.v[q], c.v[q], p.v[q]);
  return t;
}

// Face states of four variables from c[0 .. RL + RH] = cells f - RL .. f + RH.
template <int RECON, typename R>
__device__ __forceinline__ void recon_quad(const Quad<R>* c, R* wl, R* wr) {
  constexpr int RH = recon_reach<RECON>(), RL = RH + 1;
  if constexpr (RECON == 1) {
    const Quad<R> a = plm_half(c[0], c[1], c[2]), b = plm_half(c[1], c[2], c[3]);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      wl[q] = c[1].v[q] + a.v[q];
      wr[q] = c[2].v[q] - b.v[q];
    }
  } else {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      R s[6];
#pragma unroll
      for (int t = 0; t < 6; ++t) s[t] = (t - 3 >= -RL && t - 3 <= RH) ? c[t - 3 + RL].v[q] : R(0);
      recon_face<RECON>(s, wl[q], wr[q]);
    }
  }
}

// Staged planes of one variable plane set: (rho, v1, v2, v3) and (p, Bc1,
// Bc2, Bc3) as quads, hydro the pressure alone; with DUAL also S / rho.
template <bool MHD, bool DUAL>
__host__ __device__ constexpr int flux_words() { return (MHD ? 8 : 5) + (DUAL ? 1 : 0); }

// Store the outputs of one face of direction D.  Scratch arrays sit at
// sb + slot * pitch: E_ref 0..2, fluxes 8 + 5 D + v, face EMFs 23 + 2 D + q.
template <int D, bool MHD, typename R>
__device__ __forceinline__ void store_face(R* __restrict__ sb, long long pitch, long long fc,
                                           const R* fx) {
  constexpr int T1 = (D + 1) % 3, T2 = (D + 2) % 3;
  R* f = sb + (8 + 5 * D) * pitch + fc;
  f[0] = fx[0];
  f[(1 + D) * pitch] = fx[1];
  f[(1 + T1) * pitch] = fx[2];
  f[(1 + T2) * pitch] = fx[3];
  f[4 * pitch] = fx[4];
  if constexpr (MHD) {   // hydro reads no face EMF
    R* e = sb + (23 + 2 * D) * pitch + fc;
    e[0] = fx[6];        // E_t1 =  F(B_t2)
    e[pitch] = -fx[5];   // E_t2 = -F(B_t1)
  }
}

// ------------------------------------------------------------------------
// 1. flux pass.  Persistent: CTAs stride over the tiles of all blocks.
//    FP32 solves on packed (left, right) pairs (riemann2.cuh), staged cells
//    are two quads (one 16-byte shared access each, where eight 4-byte ones
//    were), the z slopes of a cell are formed once, and hydro carries no
//    field terms and writes no face EMFs.  A step (VL2, PLM, HLLD, 256^3
//    MHD): 3944 -> 3562 us; 128^3 isothermal MHD 576 -> 499 us; 128^3 hydro
//    LHLLC RK2 510 -> 342 us (32 x 4 tiles).
//    AETH_FLUX_MINB CTAs per SM in FP32; FP64 takes the full register file.
// ------------------------------------------------------------------------
// SOLVER 0: HLLD; 2: HLLE; 1: write the face states (wl, wr, bn) for the
// learned flux instead of solving; 3: isothermal HLLD; 4: isothermal HLLE;
// 5: the low-dissipation HLLD (LHLLD).  For the isothermal solvers the
// `gamma` argument carries the sound speed cs, the primitive pressure is
// cs^2 rho and is not reconstructed (the isothermal fluxes take the
// pressure from the reconstructed density).
// DUAL: dual energy (Sec. 2.8): the pressure of an untrusted internal energy
// (below alpha_switch x kinetic + magnetic) comes from the entropy, and each
// face also gets the entropy flux, its mass flux times the reconstructed
// specific entropy S/rho of the upwind side, in scratch slot 3 + D.
// TXT: the tile's x width (32 or 16; y width NT / TXT), or 0 for a band
// tile: whole rows of the block (x from -1 to n_x), band_rows(n_x) of them,
// so that a block narrower than the 2-D tile keeps its lanes busy.
// Dynamic shared memory: flux_ring<RECON>(TXT) x NW planes of
// flux_plane<RECON>(TXT) values.
template <typename R, bool P64, int RECON, bool MHD, typename Src, int SOLVER = 0,
          bool DUAL = false, int TXT = FLUX_TX>
__global__ void __launch_bounds__(flux_threads(TXT), (flux_minb<R, RECON>(TXT)))
    k_flux3(Src S, int t0, int t1, int src, R gamma, R rho_floor, R p_floor, int kchunk,
            unsigned long long* floor_hits, R alpha_switch) {
  constexpr bool BAND = TXT == 0;
  constexpr int NT = flux_threads(TXT);
  constexpr int TX = BAND ? 1 : TXT, TY = NT / TX;
  constexpr int RH = recon_reach<RECON>(), RL = RH + 1;
  constexpr int WX = TX + RL + RH, WY = TY + RL + RH;
  constexpr int QN = RL + RH + 1;
  constexpr int NB = flux_ring<RECON>(TXT);
  constexpr bool RING = NB > 1;
  constexpr bool PLM = RECON == 1;
  constexpr int NW = flux_words<MHD, DUAL>();   // staged values of a cell
  extern __shared__ __align__(16) unsigned char flux_smem[];
  R* __restrict__ sw = reinterpret_cast<R*>(flux_smem);
  constexpr int SN = flux_plane<RECON>(TXT);   // cells of one staged plane
  static_assert(SN % 4 == 0, "quads of every plane slot start on 16 bytes");
  // staging slots of a thread: cells threadIdx.x + n NT of the plane
  constexpr int NS = (SN + NT - 1) / NT;
  constexpr bool ISO = iso_solver(SOLVER);
  const R gm1 = ISO ? gamma * gamma : gamma - R(1);   // cs^2 for ISO
  const R igm1 = ISO ? R(0) : R(1) / gm1;
  int hits = 0;
  // half 0 / 1 of plane slot b at cell s; the entropy plane
  auto quad = [&](int b, int half, int s) -> R* { return sw + b * (NW * SN) + half * (4 * SN) + 4 * s; };
  auto fetch = [&](int b, int half, int s) -> Quad<R> {
    if constexpr (!MHD) {
      if (half == 1) return {{sw[b * (NW * SN) + 4 * SN + s], R(0), R(0), R(0)}};
    }
    return ld_quad(quad(b, half, s));
  };
  auto sent = [&](int b, int s) -> R& { return sw[b * (NW * SN) + (NW - 1) * SN + s]; };

  for (int t = t0 + (int)blockIdx.x; t < t1; t += gridDim.x) {
    int loc;
    const BlockPtrs<R>& P = S.get(t, loc);
    const Layout L = P.L;
    const R* __restrict__ ub = P.reg[src][0];   // state arrays at ub + v * pitch
    const R* __restrict__ eb = P.ent[src];       // entropy (DUAL)
    R* __restrict__ sb = P.w[0];                 // scratch arrays at sb + slot * pitch
    const long long pitch = P.pitch;
    const int nx = L.n[0], ny = L.n[1], nz = L.n[2];
    int i0, j0, bz, tx, ty, wxr, wyr;
    if constexpr (BAND) {
      const int W = nx + 2, br = band_rows(nx);
      const int nb = ceil_div_d(ny + 2, br);
      bz = loc / nb;
      i0 = -1;
      j0 = -1 + (loc % nb) * br;
      tx = (int)threadIdx.x % W;
      ty = (int)threadIdx.x / W;   // >= br: an idle thread of the band
      wxr = W + RL + RH;
      wyr = br + RL + RH;
    } else {
      const int ntx = ceil_div_d(nx + 2, TX), nty = ceil_div_d(ny + 2, TY);
      const int bx = loc % ntx, by = (loc / ntx) % nty;
      bz = loc / (ntx * nty);
      i0 = -1 + bx * TX;
      j0 = -1 + by * TY;
      tx = (int)threadIdx.x % TX;
      ty = (int)threadIdx.x / TX;
      wxr = WX;
      wyr = WY;
    }
    const int i = i0 + tx, j = j0 + ty;
    const int k0 = -1 + bz * kchunk;
    const int k1 = min(nz, k0 + kchunk - 1);
    const bool active =
        i <= nx && j <= ny && (!BAND || ty < band_rows(nx));

    // primitives of cell cc (+ specific entropy sp with DUAL); returns floor hits
    auto prim_at = [&](long long cc, R* w, R& sp) -> int {
      if constexpr (DUAL) {
        return prim_cell_dual<R, MHD>(L, ub, pitch, eb, cc, gm1, rho_floor, p_floor, alpha_switch,
                                      w, sp);
      } else {
        sp = R(0);
        return prim_cell_s<R, P64, MHD, ISO>(L, ub, pitch, cc, gm1, rho_floor, p_floor, w);
      }
    };
    const int sx = tx + RL, sy = ty + RL, so = sy * wxr + sx;   // own cell in a plane
    // the thread's staging cells: offset in a plane of the state arrays, or
    // < 0 outside the primitive range (the same for every plane of the tile)
    long long soff[NS];
#pragma unroll
    for (int n = 0; n < NS; ++n) {
      const int s = (int)threadIdx.x + n * NT;
      const int ci = i0 - RL + s % wxr, cj = j0 - RL + s / wxr;
      soff[n] = s < wxr * wyr && ci < nx + L.g && cj < ny + L.g && ci >= -L.g && cj >= -L.g
                    ? (long long)(cj + L.g) * L.sx + ci + OX : -1;
    }
    // own column: both halves and S/rho of plane kk, from memory or a ring slot
    auto own_mem = [&](int kk, Quad<R>* h, R& sp) {
      R w[8];
      sp = R(1);
      if (active && in_prim_range(L, i, j, kk)) {
        prim_at(L.idx(i, j, kk), w, sp);
      } else {
        w[0] = R(1); w[1] = w[2] = w[3] = R(0); w[4] = R(1); w[5] = w[6] = w[7] = R(0);
      }
      h[0] = {{w[0], w[1], w[2], w[3]}};
      h[1] = {{w[4], w[5], w[6], w[7]}};
    };
    auto own_ring = [&](int b, Quad<R>* h, R& sp) {
      h[0] = fetch(b, 0, so);
      h[1] = fetch(b, 1, so);
      if constexpr (DUAL) sp = sent(b, so);
    };
    // stage plane kk (tile + halo) into ring slot b
    auto stage = [&](int kk, int b) {
      const bool kin = kk >= -L.g && kk < nz + L.g;
      const long long base = (long long)(kk + L.g) * L.sx * L.sy;
#pragma unroll
      for (int n = 0; n < NS; ++n) {
        const int s = (int)threadIdx.x + n * NT;
        if (s >= wxr * wyr) break;
        R w[8], sp = R(1);
        if (kin && soff[n] >= 0) {
          const int h = prim_at(base + soff[n], w, sp);
          if (kk <= k1) hits += h;   // the planes above the chunk are the next one's
        } else {
          w[0] = R(1); w[1] = w[2] = w[3] = R(0); w[4] = R(1); w[5] = w[6] = w[7] = R(0);
        }
        st_quad(quad(b, 0, s), w[0], w[1], w[2], w[3]);
        if constexpr (MHD) st_quad(quad(b, 1, s), w[4], w[5], w[6], w[7]);
        else sw[b * (NW * SN) + 4 * SN + s] = w[4];
        if constexpr (DUAL) sent(b, s) = sp;
      }
    };
    // the z stencil of the own column.  PLM: the cells k - 1, k and k + 1 and
    // the upper-edge values of cell k - 1, carried from the previous plane,
    // so that each cell's slope is formed once; else cells k - RL .. k + RH.
    constexpr int ZN = PLM ? 3 : QN;
    Quad<R> zq[ZN][2], hi[2];
    R zs[ZN], his = R(0);
    (void)hi; (void)his;
    // the previous tile's last plane is read until every warp is past here
    __syncthreads();
    if constexpr (RING) {
      if constexpr (PLM) {
#pragma unroll
        for (int s = 0; s < 2; ++s) own_mem(k0 - 2 + s, zq[s], zs[s]);
      } else {
#pragma unroll
        for (int s = 0; s < RL; ++s) own_mem(k0 - RL + s, zq[s], zs[s]);
      }
#pragma unroll
      for (int m = 0; m < RH; ++m) stage(k0 + m, m);
    } else {
      // band tiles: every plane of the z stencil from memory
      if constexpr (PLM) {
        own_mem(k0 - 2, zq[0], zs[0]);
        own_mem(k0 - 1, zq[1], zs[1]);
        own_mem(k0, zq[2], zs[2]);
      } else {
#pragma unroll
        for (int s = 0; s < QN - 1; ++s) own_mem(k0 - RL + s, zq[s + 1], zs[s + 1]);
      }
    }
    auto z_advance = [&]() {
#pragma unroll
      for (int s = 0; s < ZN - 1; ++s) {
        zq[s][0] = zq[s + 1][0];
        zq[s][1] = zq[s + 1][1];
        if constexpr (DUAL) zs[s] = zs[s + 1];
      }
    };
    // PLM: upper-edge values of the middle cell of zq
    auto z_edge = [&]() {
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const Quad<R> t = plm_half(zq[0][h], zq[1][h], zq[2][h]);
#pragma unroll
        for (int q = 0; q < 4; ++q) hi[h].v[q] = zq[1][h].v[q] + t.v[q];
      }
      if constexpr (DUAL) his = zs[1] + R(0.5) * vl_slope(zs[0], zs[1], zs[2]);
    };
    for (int k = k0; k <= k1; ++k) {
      int bk = 0;
      if constexpr (RING) {
        // plane k + RH goes to ring slot (k - k0 + RH) % NB, which last held
        // plane k - 2, read by no warp past the previous barrier: one
        // barrier per plane, and each warp stages the next plane as soon as
        // its faces are done
        const int m = k - k0;
        const int bq = (m + RH) % NB;
        bk = m % NB;
        stage(k + RH, bq);
        __syncthreads();
        if (m == 0) {
          if constexpr (PLM) {
            own_ring(0, zq[2], zs[2]);
            z_edge();
            z_advance();
            own_ring(bq, zq[2], zs[2]);
          } else {
#pragma unroll
            for (int s = 0; s <= RH; ++s) own_ring(s, zq[RL + s], zs[RL + s]);
          }
        } else {
          z_advance();
          own_ring(bq, zq[ZN - 1], zs[ZN - 1]);
        }
      } else {
        // one staged plane, the z stencil from memory
        if (k > k0) __syncthreads();
        stage(k, 0);
        if constexpr (PLM) {
          if (k == k0) z_edge();
        }
        z_advance();
        own_mem(k + RH, zq[ZN - 1], zs[ZN - 1]);
        __syncthreads();
      }
      if (!active) continue;

      // the faces of plane k from ring slot bk (x, y, E_ref) and the z stencil
      const long long fc = L.idx(i, j, k);
      R l8[8], r8[8];   // face states (rho, v1, v2, v3, p, B1, B2, B3)
      R sl = R(0), sr = R(0);
      // solve and store the face of direction D from l8, r8 (sl, sr)
      auto face = [&](auto dir) {
        constexpr int D = decltype(dir)::value;
        constexpr int T1 = (D + 1) % 3, T2 = (D + 2) % 3;
        constexpr int slot[7] = {0, 1 + D, 1 + T1, 1 + T2, 4, 5 + T1, 5 + T2};
        R wl[7], wr[7], fx[7];
#pragma unroll
        for (int v = 0; v < 7; ++v) {
          const bool zero = (!MHD && v >= 5) || (ISO && v == 4);
          wl[v] = zero ? R(0) : l8[slot[v]];
          wr[v] = zero ? R(0) : r8[slot[v]];
        }
        const R bn = MHD ? ub[(5 + D) * pitch + fc] : R(0);
        if constexpr (SOLVER != 1) {
          solve_face<SOLVER, MHD>(gamma, igm1, wl, wr, bn, fx);
          store_face<D, MHD>(sb, pitch, fc, fx);
          if constexpr (DUAL) sb[(3 + D) * pitch + fc] = fx[0] >= R(0) ? fx[0] * sl : fx[0] * sr;
        } else {
          R* fs = P.fstate + (D * 15) * pitch + fc;
#pragma unroll
          for (int v = 0; v < 7; ++v) { fs[v * pitch] = wl[v]; fs[(7 + v) * pitch] = wr[v]; }
          fs[14 * pitch] = bn;
        }
      };
      // states of the lower face along a staged axis (cell stride ds)
      auto plane_states = [&](int ds) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          Quad<R> c[QN];
#pragma unroll
          for (int q = 0; q < QN; ++q) c[q] = fetch(bk, h, so + (q - RL) * ds);
          recon_quad<RECON>(c, l8 + 4 * h, r8 + 4 * h);
        }
        if constexpr (DUAL) recon_var<RECON>([&](int off) { return sent(bk, so + off * ds); }, sl, sr);
      };
      if (i >= 0) {
        plane_states(1);
        face(Int<0>{});
      }
      if (j >= 0) {
        plane_states(wxr);
        face(Int<1>{});
      }
      if constexpr (PLM) {
        // lower-edge values of cell k, and its upper-edge values for face k + 1
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const Quad<R> t = plm_half(zq[0][h], zq[1][h], zq[2][h]);
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            l8[4 * h + q] = hi[h].v[q];
            r8[4 * h + q] = zq[1][h].v[q] - t.v[q];
            hi[h].v[q] = zq[1][h].v[q] + t.v[q];
          }
        }
        if constexpr (DUAL) {
          const R t = R(0.5) * vl_slope(zs[0], zs[1], zs[2]);
          sl = his;
          sr = zs[1] - t;
          his = zs[1] + t;
        }
      } else {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          Quad<R> c[QN];
#pragma unroll
          for (int q = 0; q < QN; ++q) c[q] = zq[q][h];
          recon_quad<RECON>(c, l8 + 4 * h, r8 + 4 * h);
        }
        if constexpr (DUAL) recon_var<RECON>([&](int off) { return zs[off + RL]; }, sl, sr);
      }
      if (k >= 0) face(Int<2>{});
      // ---- cell-centred reference EMF, E = -v x B
      if constexpr (MHD) {
        const Quad<R> a = zq[PLM ? 1 : RL][0], b = zq[PLM ? 1 : RL][1];
        sb[fc] = -(a.v[2] * b.v[3] - a.v[3] * b.v[2]);
        sb[pitch + fc] = -(a.v[3] * b.v[1] - a.v[1] * b.v[3]);
        sb[2 * pitch + fc] = -(a.v[1] * b.v[2] - a.v[2] * b.v[1]);
      }
    }
  }
  if (hits) atomicAdd(floor_hits, (unsigned long long)hits);
}

// ------------------------------------------------------------------------
// host side
// ------------------------------------------------------------------------
struct TileRange {
  int t0, t1;
};

static TileRange range_of(const aeth_ctx* c, int kind, int block) {
  const int nb = (int)c->blocks.size();
  const int* p = c->h_prefix.data() + kind * (nb + 1);
  if (block < 0) return {0, p[nb]};
  return {p[block], p[block + 1]};
}

template <typename R>
static const BlockPtrs<R>* dtab(const aeth_ctx* c) {
  return (const BlockPtrs<R>*)c->d_tab;
}

static const int* dpre(const aeth_ctx* c, int kind) {
  return c->d_prefix + kind * ((int)c->blocks.size() + 1);
}

// Launch a pass either from the device table (several blocks) or with the
// block's pointers in the kernel parameters (one block).
template <typename R, typename F>
static void with_src(aeth_ctx* c, int kind, int block, F launch) {
  const int nb = (int)c->blocks.size();
  if (nb == 1 || block >= 0) {
    const int b = block >= 0 ? block : 0;
    const TileRange r = range_of(c, kind, b);
    launch(ParamSrc<R>{block_ptrs<R>(c, b), r.t0}, r);
  } else {
    launch(TableSrc<R>{dtab<R>(c), dpre(c, kind), nb, c->d_tmap[kind]}, range_of(c, kind, -1));
  }
}

template <typename R, bool P64, int RECON, bool MHD, int SOLVER, bool DUAL>
static void launch_flux3(aeth_ctx* c, int src, int block) {

  constexpr int NW = flux_words<MHD, DUAL>();
  with_src<R>(c, PK_FLUX, block, [&](auto S, TileRange r) {
    // tx: the tile width the kernel was built for (0: band tiles)
    auto go = [&](auto kernel, int tx) {
      const int per_sm = flux_minb<R, RECON>(tx);
      const int grid = std::max(1, std::min(r.t1 - r.t0, c->num_sms * per_sm));
      const int bytes = flux_ring<RECON>(tx) * NW * flux_plane<RECON>(tx) * (int)sizeof(R);
      // above the 48 KB default (FP64, PPM rings, bands); a plain attribute
      // call, also legal while a graph is being captured
      if (bytes > 48 * 1024)
        cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
      kernel<<<grid, flux_threads(tx), bytes, c->stream>>>(
          S, r.t0, r.t1, src, (R)(iso_solver(SOLVER) ? c->cfg.cs_iso : c->cfg.gamma),
          (R)c->cfg.rho_floor, (R)c->cfg.p_floor, c->kchunk, c->d_floor,
          (R)c->cfg.alpha_switch);
    };
    // the 16-wide tile is built for the FP32 solver passes (the contexts
    // whose tiles the autotuner may switch: tile_shape_tunable)
    if constexpr (sizeof(R) == 4 && !DUAL && SOLVER != 1) {
      if (c->flux_tx == 16) {
        go(k_flux3<R, P64, RECON, MHD, decltype(S), SOLVER, DUAL, 16>, 16);
        return;
      }
      if (c->flux_tx == 0) {
        go(k_flux3<R, P64, RECON, MHD, decltype(S), SOLVER, DUAL, 0>, 0);
        return;
      }
    }
    go(k_flux3<R, P64, RECON, MHD, decltype(S), SOLVER, DUAL, 32>, 32);
  });
  c->n_launch += 1;
}

// One flux pass with the solver family SOLVER and the reconstruction of the
// context (explicitly instantiated per family in flux_*.cu; DUAL in
// flux_dual_*.cu).
template <typename R, bool P64, bool MHD, int SOLVER, bool DUAL = false>
void flux_pass_solver(aeth_ctx* c, int recon, int src, int block);

template <typename R, bool P64, bool MHD, int SOLVER, bool DUAL>
void flux_pass_solver_impl(aeth_ctx* c, int recon, int src, int block) {
  if (recon == AETH_RECON_DONOR) launch_flux3<R, P64, 0, MHD, SOLVER, DUAL>(c, src, block);
  else if (recon == AETH_RECON_PLM) launch_flux3<R, P64, 1, MHD, SOLVER, DUAL>(c, src, block);
  else if (recon == AETH_RECON_PPM5) launch_flux3<R, P64, 3, MHD, SOLVER, DUAL>(c, src, block);
  else launch_flux3<R, P64, 2, MHD, SOLVER, DUAL>(c, src, block);
}

}  // namespace aeth
