// Flux pass of the fused stage (Sec. 2.4): conserved->primitive,
// reconstruction and the Riemann solver for all three face directions of
// every cell in one sweep.  A CTA owns a TX x TY column tile and marches
// along z: each x-y plane of primitives (with the reconstruction halo) is
// staged in a ring of shared-memory planes, which serves the x- and y-faces
// and the upper part of the z stencil; its lower part stays in registers.
// Each face is solved exactly once.  Outputs: hydro fluxes, face EMFs (the
// transverse induction fluxes) and the cell-centred reference EMF of the
// upwind CT scheme.
//
// The kernel template lives here so that its instantiations (one per
// Riemann solver family) compile in separate translation units.
#pragma once
#include <type_traits>

#include "riemann2.cuh"
#include "runtime.hpp"
#include "stage.cuh"

namespace aeth {

// resident CTAs per SM requested.  Band tiles (256 threads, FP32): 2; 3 (80
// registers) spilled 68 to 120 bytes a thread into an L1 that the staging
// leaves small: 512 uneven boxes 8823 -> 8076 us a step.
#ifndef AETH_FLUX_MINB
#define AETH_FLUX_MINB 2
#endif
// the same for the 128-thread 2-D tiles: 5 (95 registers, no spill) measured 0
// to 6% faster than 4 (119 registers); PPM keeps 4
#ifndef AETH_FLUX_MINB_2D
#define AETH_FLUX_MINB_2D 5
#endif
#ifndef AETH_FLUX_MINB_2D_PPM
#define AETH_FLUX_MINB_2D_PPM 4
#endif
template <typename R, int RECON>
__host__ __device__ constexpr int flux_minb(int txt) {
  return txt == 0 ? (sizeof(R) == 4 ? AETH_FLUX_MINB : 1)
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

// Planes in the shared-memory ring of a flux tile: the z stencil takes plane
// k + RH while the x- and y-faces read plane k, and the next plane is staged
// while slower warps still read plane k - 1.
template <int RECON>
__host__ __device__ constexpr int flux_ring() { return recon_reach<RECON>() + 2; }

// Solver families 3 and 4 are the isothermal ones.
constexpr bool iso_solver(int solver) { return solver == 3 || solver == 4; }

// Riemann solver family SOLVER (numbering of k_flux3 below) on one face: on
// packed pairs in FP32 (all but the isothermal HLLE), else the scalar solvers;
// a gas without field takes either without its terms.  SPLIT: the rounding of one
// term of the right side (riemann2.cuh), set for the z faces of donor-cell states.
template <int SOLVER, bool MHD, bool SPLIT, typename R>
__device__ __forceinline__ void solve_face(R g, R igm1, const R* wl, const R* wr, R bn, R* fx) {
  if constexpr (sizeof(R) == 4 && SOLVER != 4) {
    float2 W[7];
#pragma unroll
    for (int v = 0; v < 7; ++v) W[v] = make_float2(wl[v], wr[v]);
    if constexpr (SOLVER == 2) hlle2<MHD>(g, igm1, W, bn, fx);
    else if constexpr (SOLVER == 3) hlld_iso2<MHD, SPLIT>(g * g, W, bn, fx);
    else hlld2<SOLVER == 5, MHD, SPLIT>(g, igm1, W, bn, fx);
  } else {
    if constexpr (SOLVER == 2) hlle<MHD>(g, wl, wr, bn, fx);
    else if constexpr (SOLVER == 3) hlld_iso(g, wl, wr, bn, fx);
    else if constexpr (SOLVER == 4) hlle_iso<MHD>(g, wl, wr, bn, fx);
    else if constexpr (SOLVER == 5) hlld<true>(g, wl, wr, bn, fx);
    else hlld(g, wl, wr, bn, fx);
  }
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

// A value the compiler takes for unknown: products of the cells that the
// three directions share are then formed (and fused) per direction, in one
// way whatever the tile shape.
__device__ __forceinline__ void opaque(Quad<float>& a) {
  asm("" : "+f"(a.v[0]), "+f"(a.v[1]), "+f"(a.v[2]), "+f"(a.v[3]));
}
__device__ __forceinline__ void opaque(Quad<double>&) {}

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
  for (int q = 0; q < 4; ++q) {
    // half of 2 dm dp / (dm + dp): the factors are powers of two
    const double dm = c.v[q] - m.v[q], dp = p.v[q] - c.v[q], x = dm * dp;
    t.v[q] = is_pos(x) ? x / (dm + dp) : 0.0;
  }
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

// Asynchronous 4-byte copies global -> shared (no register holds the value in
// flight).
__device__ __forceinline__ void cp_async4(float* dst, const float* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(
                   static_cast<uint32_t>(__cvta_generic_to_shared(dst))),
               "l"(src)
               : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group 0;\n" ::: "memory"); }

// Staged planes of one variable plane set: (rho, v1, v2, v3) and (p, Bc1,
// Bc2, Bc3) as quads, hydro the pressure alone; with DUAL also S / rho.
template <bool MHD, bool DUAL>
__host__ __device__ constexpr int flux_words() { return (MHD ? 8 : 5) + (DUAL ? 1 : 0); }

// FP32: the conserved values of the next plane's staging cells are copied
// asynchronously behind the faces of the current one.
template <typename R>
__host__ __device__ constexpr bool flux_async() { return sizeof(R) == 4; }
// staging cells of a thread, and raw values copied per cell (with a field the
// lower and upper x and y faces and the upper z face)
template <int RECON>
__host__ __device__ constexpr int flux_slots(int txt) {
  return (flux_plane<RECON>(txt) + flux_threads(txt) - 1) / flux_threads(txt);
}
template <bool MHD, bool DUAL>
__host__ __device__ constexpr int flux_raw_words() { return (MHD ? 10 : 5) + (DUAL ? 1 : 0); }
// dynamic shared memory of a flux CTA: the ring of staged planes, the raw values
template <typename R, int RECON, bool MHD, bool DUAL>
__host__ __device__ constexpr int flux_smem_bytes(int txt) {
  return (int)sizeof(R) * (flux_ring<RECON>() * flux_words<MHD, DUAL>() * flux_plane<RECON>(txt) +
                           (flux_async<R>() ? flux_raw_words<MHD, DUAL>() * flux_plane<RECON>(txt)
                                               : 0));
}

// What the pass reads of a mesh block.  Passes over several blocks keep it
// in shared memory: held in registers it cost the kernel spills, re-read from
// the block table a memory round trip a use.
template <typename R>
struct FluxBlk {
  const R* u;      // state arrays (array v at pitch v)
  const R* ent;    // entropy (dual energy)
  R* s;            // scratch arrays
  R* fstate;       // learned flux: face states
  unsigned p16;    // pitch in units of 16 bytes
  long long sx, plane;
  int n[3], g;
  float p64;
  int loc;         // tile in the block
  __device__ __forceinline__ void set(const BlockPtrs<R>& P, int src, int l) {
    u = P.reg[src][0];
    ent = P.ent[src];
    s = P.w[0];
    fstate = P.fstate;
    p16 = (unsigned)(P.pitch * (long long)sizeof(R) / 16);
    sx = P.L.sx;
    plane = P.L.sx * P.L.sy;
    for (int d = 0; d < 3; ++d) n[d] = P.L.n[d];
    g = P.L.g;
    p64 = P.L.p64_ratio;
    loc = l;
  }
  // element at c of array v from base b: the array offset is one 32 x 32-bit
  // multiply-add (a pitch is a multiple of 256 bytes and, as dozens of arrays
  // fit the device, below 2^32 x 16 bytes)
  template <typename T>
  __device__ __forceinline__ T* at(T* b, int v) const {
    using Byte = std::conditional_t<std::is_const_v<T>, const char, char>;
    return reinterpret_cast<T*>(reinterpret_cast<Byte*>(b) +
                                (unsigned long long)p16 * (unsigned)(16 * v));
  }
};

// Tile t's block for a whole warp: 32 pivots of the prefix sums at a time.
__device__ __forceinline__ int find_block_warp(const int* __restrict__ pre, int nb, int t) {
  const int lane = threadIdx.x & 31;
  int lo = 0, hi = nb;   // pre[lo] <= t < pre[hi]
  while (hi - lo > 1) {
    const int step = (hi - lo + 31) / 32, q = lo + lane * step;
    const unsigned m = __ballot_sync(0xffffffffu, q < hi && pre[q] <= t);
    const int at = lo + (31 - __clz(m)) * step;   // lane 0 holds pre[lo] <= t
    hi = min(hi, at + step);
    lo = at;
  }
  return lo;
}

// Store the outputs of one face of direction D at sp (the cell of scratch
// array 0).  Scratch arrays: E_ref 0..2, fluxes 8 + 5 D + v, face EMFs
// 23 + 2 D + q.
template <int D, bool MHD, typename R>
__device__ __forceinline__ void store_face(const FluxBlk<R>& K, R* sp, const R* fx) {
  constexpr int T1 = (D + 1) % 3, T2 = (D + 2) % 3;
  *K.at(sp, 8 + 5 * D) = fx[0];
  *K.at(sp, 8 + 5 * D + 1 + D) = fx[1];
  *K.at(sp, 8 + 5 * D + 1 + T1) = fx[2];
  *K.at(sp, 8 + 5 * D + 1 + T2) = fx[3];
  *K.at(sp, 8 + 5 * D + 4) = fx[4];
  if constexpr (MHD) {   // hydro reads no face EMF
    *K.at(sp, 23 + 2 * D) = fx[6];        // E_t1 =  F(B_t2)
    *K.at(sp, 24 + 2 * D) = -fx[5];       // E_t2 = -F(B_t1)
  }
}

// ------------------------------------------------------------------------
// 1. flux pass, one tile a CTA.
//    FP32 solves on packed (left, right) pairs (riemann2.cuh), staged cells
//    are two quads (one 16-byte shared access each), the z slopes of a cell
//    are formed once, and hydro carries no field terms and writes no face
//    EMFs.  The conserved values of the next plane are copied into shared
//    memory behind the faces of the current one (4-byte cp.async: each
//    thread reads back its own copies, so no barrier is added and no
//    register holds a value in flight); with direct loads the staging's
//    memory latency was 2.4 of 5.3 stall cycles an instruction.  Of the z
//    stencil only the planes below k stay in registers, the others are in
//    the ring.  A step (us), before and after: 256^3 MHD HLLD 3944 -> 3098,
//    128^3 isothermal MHD 576 -> 463, 128^3 hydro LHLLC RK2 510 -> 321, 190 x
//    131 x 77 PPM RK3 1350 -> 1046, 2 x 2 x 2 blocks of 128^3 HLLE RK2 4800 ->
//    3684, 512 uneven boxes 10690 -> 8541, with the same results bit for bit
//    (the launch, 128^3 HLLD PLM corrector: 214 -> 132).
//    Bulk copies of whole rows (one instruction a row, issued one lane at a
//    time) were 20 to 35% slower.
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
// Dynamic shared memory: flux_smem_bytes.
template <typename R, bool P64, int RECON, bool MHD, typename Src, int SOLVER = 0,
          bool DUAL = false, int TXT = FLUX_TX>
__global__ void __launch_bounds__(flux_threads(TXT), (flux_minb<R, RECON>(TXT)))
    k_flux3(Src S, int t0, int src, R gamma, R rho_floor, R p_floor, int kchunk,
            unsigned long long* floor_hits, R alpha_switch) {
  constexpr bool BAND = TXT == 0;
  constexpr int NT = flux_threads(TXT);
  constexpr int TX = BAND ? 1 : TXT, TY = NT / TX;
  constexpr int RH = recon_reach<RECON>(), RL = RH + 1;
  constexpr int WX = TX + RL + RH, WY = TY + RL + RH;
  constexpr int QN = RL + RH + 1;
  constexpr int NB = flux_ring<RECON>();
  constexpr bool PLM = RECON == 1;
  constexpr int NW = flux_words<MHD, DUAL>();   // staged values of a cell
  extern __shared__ __align__(16) unsigned char flux_smem[];
  R* __restrict__ sw = reinterpret_cast<R*>(flux_smem);
  constexpr int SN = flux_plane<RECON>(TXT);   // cells of one staged plane
  static_assert(SN % 4 == 0, "quads of every plane slot start on 16 bytes");
  // staging slots of a thread: cells threadIdx.x + n NT of the plane
  constexpr int NS = flux_slots<RECON>(TXT);
  // raw values: word v of cell s at raw[v * SN + s]
  constexpr bool ASYNC = flux_async<R>();
  R* __restrict__ raw = sw + NB * NW * SN;
  constexpr int NRAW = flux_raw_words<MHD, DUAL>();
  constexpr bool ISO = iso_solver(SOLVER);
  const R gm1 = ISO ? gamma * gamma : gamma - R(1);   // cs^2 for ISO
  const R igm1 = recip(gm1);
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

  {
    constexpr bool TABLE = std::is_same_v<Src, TableSrc<R>>;
    __shared__ FluxBlk<R> sblk;
    const int t = t0 + (int)blockIdx.x;
    FluxBlk<R> pblk;
    if constexpr (TABLE) {
      if (threadIdx.x < 32) {
        const int b = find_block_warp(S.pre, S.nb, t);
        if (threadIdx.x == 0) sblk.set(S.tab[b], src, t - S.pre[b]);
      }
      __syncthreads();
    } else {
      pblk.set(S.P, src, t - S.base);
    }
    const FluxBlk<R>& K = TABLE ? sblk : pblk;
    const int nx = K.n[0], ny = K.n[1], nz = K.n[2], g = K.g, loc = K.loc;
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

    // offset of (i, j, k) in an array
    auto idx = [&](int ii, int jj, int kk) -> long long {
      return (kk + g) * K.plane + (jj + g) * K.sx + ii + OX;
    };
    // primitives of cell cc (+ specific entropy sp with DUAL); returns floor hits
    auto prim_at = [&](long long cc, R* w, R& sp) -> int {
      ConstArr8<R> u;
#pragma unroll
      for (int v = 0; v < NVAR; ++v) u.p[v] = K.at(K.u, v);
      R x[5], b[3];
      load_cell<R, MHD>(K.sx, K.plane, u, cc, !ISO, x, b);
      sp = R(0);
      if constexpr (DUAL)
        return prim_values_dual<R>(x, b, K.ent[cc], gm1, rho_floor, p_floor, alpha_switch, w, sp);
      else
        return prim_values<R, P64, ISO>(K.p64, x, b, gm1, rho_floor, p_floor, w);
    };
    const int so = (ty + RL) * wxr + tx + RL;   // own cell in a plane
    // the thread's staging cells: offset in a plane of the state arrays, or
    // NONE outside the primitive range (the same for every plane of the tile)
    constexpr unsigned NONE = ~0u;
    unsigned soff[NS];
#pragma unroll
    for (int n = 0; n < NS; ++n) {
      const int s = (int)threadIdx.x + n * NT;
      const int ci = i0 - RL + s % wxr, cj = j0 - RL + s / wxr;
      soff[n] = s < wxr * wyr && ci < nx + g && cj < ny + g && ci >= -g && cj >= -g
                    ? (unsigned)((cj + g) * K.sx) + (unsigned)(ci + OX) : NONE;
    }
    // ASYNC: the lower z face of each staging cell, carried from plane to plane
    R zlo[NS];
#pragma unroll
    for (int n = 0; n < NS; ++n)
      zlo[n] = ASYNC && MHD && soff[n] != NONE
                   ? K.at(K.u, 7)[(k0 + g) * K.plane + soff[n]] : R(0);
    // start the copies of the raw values of plane kk; every thread reads back
    // only what it copied itself
    auto issue = [&](int kk) {
      if constexpr (ASYNC) {
        if (kk >= -g && kk < nz + g) {
          const long long base = (kk + g) * K.plane;
#pragma unroll
          for (int n = 0; n < NS; ++n) {
            if (soff[n] == NONE) continue;
            const R* p = K.u + base + soff[n];
            R* q = raw + threadIdx.x + n * NT;
#pragma unroll
            for (int v = 0; v < 5; ++v)
              if (!(ISO && v == 4)) cp_async4(q + v * SN, K.at(p, v));
            if constexpr (MHD) {
              cp_async4(q + 5 * SN, K.at(p, 5));
              cp_async4(q + 6 * SN, K.at(p, 5) + 1);
              cp_async4(q + 7 * SN, K.at(p, 6));
              cp_async4(q + 8 * SN, K.at(p, 6) + K.sx);
              cp_async4(q + 9 * SN, K.at(p, 7) + K.plane);
            }
            if constexpr (DUAL) cp_async4(q + (NRAW - 1) * SN, K.ent + base + soff[n]);
          }
        }
        cp_async_commit();
      }
    };
    // own column: both halves and S/rho of plane kk, from memory or a ring slot
    auto own_mem = [&](int kk, Quad<R>* h, R& sp) {
      R w[8];
      sp = R(1);
      if (active && i < nx + g && j < ny + g && kk >= -g && kk < nz + g) {
        prim_at(idx(i, j, kk), w, sp);
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
      const bool kin = kk >= -g && kk < nz + g;
      const long long base = (kk + g) * K.plane;
      if constexpr (ASYNC) cp_async_wait();
#pragma unroll
      for (int n = 0; n < NS; ++n) {
        const int s = (int)threadIdx.x + n * NT;
        if (s >= wxr * wyr) break;
        R w[8], sp = R(1);
        if (kin && soff[n] != NONE) {
          int h;
          if constexpr (ASYNC) {
            const R* q = raw + s;
            R u[5], b[3] = {R(0), R(0), R(0)};
#pragma unroll
            for (int v = 0; v < 5; ++v) u[v] = ISO && v == 4 ? R(0) : q[v * SN];
            if constexpr (MHD) {
              const R zhi = q[9 * SN];
              b[0] = R(0.5) * (q[5 * SN] + q[6 * SN]);
              b[1] = R(0.5) * (q[7 * SN] + q[8 * SN]);
              b[2] = R(0.5) * (zlo[n] + zhi);
              zlo[n] = zhi;
            }
            if constexpr (DUAL)
              h = prim_values_dual<R>(u, b, q[(NRAW - 1) * SN], gm1, rho_floor, p_floor,
                                      alpha_switch, w, sp);
            else
              h = prim_values<R, P64, ISO>(K.p64, u, b, gm1, rho_floor, p_floor, w);
          } else {
            h = prim_at(base + soff[n], w, sp);
          }
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
    // the z stencil of the own column below plane k (planes k and above are
    // read from the ring).  PLM: cell k - 1 and its upper-edge values, formed
    // with the previous plane's faces, so that each cell's slope is formed
    // once; else cells k - RL .. k - 1.
    constexpr int ZN = PLM ? 1 : RL;
    Quad<R> zp[ZN][2], hi[2];
    R zs[ZN], his = R(0);
    (void)hi; (void)his;
    issue(k0);
    if constexpr (PLM) {
      own_mem(k0 - 1, zp[0], zs[0]);
    } else {
#pragma unroll
      for (int s = 0; s < RL; ++s) own_mem(k0 - RL + s, zp[s], zs[s]);
    }
#pragma unroll
    for (int m = 0; m < RH; ++m) {
      stage(k0 + m, m);
      issue(k0 + m + 1);
    }
    for (int k = k0; k <= k1; ++k) {
      const long long fc = idx(i, j, k);
      // normal face fields, in flight during the staging
      R bn[3] = {R(0), R(0), R(0)};
      if constexpr (MHD) {
        if (active)
#pragma unroll
          for (int d = 0; d < 3; ++d) bn[d] = *K.at(K.u + fc, 5 + d);
      }
      // plane k + RH goes to ring slot (k - k0 + RH) % NB, which last held
      // plane k - 2, read by no warp past the previous barrier: one
      // barrier per plane, and each warp stages the next plane as soon as
      // its faces are done
      const int m = k - k0;
      const int bk = m % NB;
      stage(k + RH, (m + RH) % NB);
      if (k < k1) issue(k + RH + 1);
      __syncthreads();
      if (!active) continue;
      if constexpr (PLM) {
        if (m == 0) {   // upper-edge values of the cell below the chunk
          Quad<R> b2[2], c[2];
          R s2, s0;
          own_mem(k0 - 2, b2, s2);
          own_ring(bk, c, s0);
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const Quad<R> t = plm_half(b2[h], zp[0][h], c[h]);
#pragma unroll
            for (int q = 0; q < 4; ++q) hi[h].v[q] = zp[0][h].v[q] + t.v[q];
          }
          if constexpr (DUAL) his = zs[0] + R(0.5) * vl_slope(s2, zs[0], s0);
        }
      }

      // the faces of plane k from ring slot bk (x, y, E_ref) and the z stencil
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
        if constexpr (SOLVER != 1) {
          solve_face<SOLVER, MHD, RECON == 0 && D == 2>(gamma, igm1, wl, wr, bn[D], fx);
          store_face<D, MHD>(K, K.s + fc, fx);
          if constexpr (DUAL) *K.at(K.s + fc, 3 + D) = fx[0] >= R(0) ? fx[0] * sl : fx[0] * sr;
        } else {
          R* fs = K.fstate + fc;
#pragma unroll
          for (int v = 0; v < 7; ++v) {
            *K.at(fs, D * 15 + v) = wl[v];
            *K.at(fs, D * 15 + 7 + v) = wr[v];
          }
          *K.at(fs, D * 15 + 14) = bn[D];
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
      Quad<R> cur[2];
      R scur = R(0);
      own_ring(bk, cur, scur);
      opaque(cur[0]);
      opaque(cur[1]);
      if constexpr (PLM) {
        // lower-edge values of cell k, and its upper-edge values for face k + 1
        Quad<R> nxt[2];
        R snxt = R(0);
        own_ring((m + 1) % NB, nxt, snxt);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const Quad<R> t = plm_half(zp[0][h], cur[h], nxt[h]);
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            l8[4 * h + q] = hi[h].v[q];
            r8[4 * h + q] = cur[h].v[q] - t.v[q];
            hi[h].v[q] = cur[h].v[q] + t.v[q];
          }
        }
        if constexpr (DUAL) {
          const R t = R(0.5) * vl_slope(zs[0], scur, snxt);
          sl = his;
          sr = scur - t;
          his = scur + t;
        }
      } else {
        R sz[QN];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          Quad<R> c[QN];
#pragma unroll
          for (int q = 0; q < RL; ++q) c[q] = zp[q][h];
          c[RL] = cur[h];
#pragma unroll
          for (int q = 1; q <= RH; ++q) c[RL + q] = fetch((m + q) % NB, h, so);
          recon_quad<RECON>(c, l8 + 4 * h, r8 + 4 * h);
        }
        if constexpr (DUAL) {
#pragma unroll
          for (int q = 0; q < RL; ++q) sz[q] = zs[q];
          sz[RL] = scur;
#pragma unroll
          for (int q = 1; q <= RH; ++q) sz[RL + q] = sent((m + q) % NB, so);
          recon_var<RECON>([&](int off) { return sz[off + RL]; }, sl, sr);
        }
      }
#pragma unroll
      for (int s = 0; s < ZN; ++s)
#pragma unroll
        for (int h = 0; h < 2; ++h) zp[s][h] = s + 1 < ZN ? zp[s + 1 < ZN ? s + 1 : 0][h] : cur[h];
      if constexpr (DUAL) {
#pragma unroll
        for (int s = 0; s < ZN; ++s) zs[s] = s + 1 < ZN ? zs[s + 1 < ZN ? s + 1 : 0] : scur;
      }
      if (k >= 0) face(Int<2>{});
      // ---- cell-centred reference EMF, E = -v x B
      if constexpr (MHD) {
        const Quad<R>&a = cur[0], &b = cur[1];
        R* e = K.s + fc;
        *e = -(a.v[2] * b.v[3] - a.v[3] * b.v[2]);
        *K.at(e, 1) = -(a.v[3] * b.v[1] - a.v[1] * b.v[3]);
        *K.at(e, 2) = -(a.v[1] * b.v[2] - a.v[2] * b.v[1]);
      }
    }
  }
  add_hits(floor_hits, hits);
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

  with_src<R>(c, PK_FLUX, block, [&](auto S, TileRange r) {
    // tx: the tile width the kernel was built for (0: band tiles)
    auto go = [&](auto kernel, int tx) {
      const int grid = r.t1 - r.t0;
      const int bytes = flux_smem_bytes<R, RECON, MHD, DUAL>(tx);
      // above the 48 KB default (FP64, PPM rings, bands); a plain attribute
      // call, also legal while a graph is being captured
      if (bytes > 48 * 1024)
        cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
      kernel<<<grid, flux_threads(tx), bytes, c->stream>>>(
          S, r.t0, src, (R)(iso_solver(SOLVER) ? c->cfg.cs_iso : c->cfg.gamma),
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
