// FP64 residual of one implicit Euler step on the finest grid, with or
// without its Jacobian (Eqs. 1-5 integrated over each cell; the discrete
// equations of henry_device.cuh). Used by the time loop (k_residual in its
// multigrid layout), the adjoint and henry_residual_jacobian (natural layout).
//
// What bounds it: GB300's FP64 pipe. One FP64 warp instruction (arithmetic,
// comparison or conversion alike) costs about 18 cycles of an SM, so the
// floor of a launch is its FP64 instructions per cell, and a kernel that
// leaves SMs without a warp loses proportionally. Hence:
//  * every face is evaluated once: a thread owns C neighbouring columns and
//    walks R rows; faces between its own columns stay in registers, the face
//    to the next lane's column is passed by shuffle, the north face becomes
//    the next row's south face. Only a tile's first row (south) and, on
//    grids of several tiles in x, its first column (west; all rows of it
//    in one pass, a row per lane) are evaluated twice;
//  * the unit of scheduling is one warp (a block of 32 threads, no barrier,
//    no shared memory), so a small batch spreads over all SMs: 16 samples of
//    64x32 cells are 128 to 256 blocks, where a 256-thread tile per sample
//    kept 16 SMs busy. Tall tiles, which a large batch wants, may be shared by
//    the warps of a block (SPLIT);
//  * the densities and rho c are formed once per cell; upwinding tests the
//    sign bit of the flux (integer pipe); the FP32 Jacobian takes its face
//    constants from FP32 copies instead of converting them.
// Every rounding is written out (fma, one product and sum at a time), so that
// a solve's iterates do not depend on how the compiler contracts expressions
// for a tile's first or last column.
// Per cell: 34 FP64 instructions for the residual, + 2 conversions with FP32
// multigrid.
#pragma once

#include <type_traits>

#include "common.cuh"
#include "henry_device.cuh"

// (included by kernels.cuh, which defines kJP and store_operator)

namespace henry {

// Derivatives of a face's fluxes (mass m, salt s): with respect to p_L mp
// and sp (to p_U their negatives), to c_L and c_U the others.
template <typename T>
struct FaceJ {
  T mp, sp, mLc, mUc, sLc, sUc;
};

// A cell's values: pressure, mass fraction, density, rho c.
struct CellV {
  double p, c, r, rc;
};

__device__ __forceinline__ void cell_values(const Phys& P, CellV& v) {
  v.r = fma(P.drho, v.c, P.rho0);
  v.rc = v.r * v.c;
}

// One face from L to U, residual only: t = A K_f / (mu d), dh = A phi_f D /
// (2 d), hdg = (drho / 2) g d (vertical faces); a face's mean density and its
// gravity term share c_L + c_U. The upwind side is the sign bit of q (a zero
// flux of either sign carries nothing).
template <bool VERT>
__device__ __forceinline__ void res_face(const Phys& P, const CellV& L, const CellV& U, double t,
                                         double dh, double hdg, double& q, double& Fm, double& Fs) {
  const double sc = L.c + U.c;
  const double rs = fma(P.drho, sc, 2.0 * P.rho0);   // rho_L + rho_U
  const double dp = U.p - L.p;
  q = -t * (VERT ? fma(hdg, sc, dp) : dp);
  const bool up = __double2hiint(q) >= 0;
  Fm = q * (up ? L.r : U.r);
  Fs = fma(q, up ? L.rc : U.rc, -(dh * rs) * (U.c - L.c));
}

// q >= 0 (either zero included) without an FP64 instruction.
__device__ __forceinline__ bool not_negative(double q) {
  const int hi = __double2hiint(q);
  return hi >= 0 || ((hi << 1) | __double2loint(q)) == 0;
}

// The same face with its derivatives in the multigrid type T, formed from
// few converted values (on GB300 a conversion costs an FP64 slot): t_, h_ =
// (T)dh, cL, cU. dp = p_U - p_L; gd = g d of a vertical face.
template <typename T, bool VERT>
__device__ __forceinline__ void jac_face(const Phys& P, const CellV& L, const CellV& U, double dp,
                                         double t, double dh, double gd, T t_, T h_, T cL, T cU,
                                         double& q, double& Fm, double& Fs, FaceJ<T>& f) {
  constexpr bool D = sizeof(T) == 8;
  const double dc = U.c - L.c;
  q = VERT ? -t * fma((0.5 * P.drho) * (L.c + U.c), gd, dp) : -t * dp;
  const bool up = not_negative(q);
  const double rup = up ? L.r : U.r;
  Fm = q * rup;
  Fs = fma(q, up ? L.rc : U.rc, -(dh * (L.r + U.r)) * dc);
  const T q_ = (T)q, dr = (T)P.drho, r0 = (T)P.rho0;
  const T rL = D ? (T)L.r : fma(dr, cL, r0), rU = D ? (T)U.r : fma(dr, cU, r0);
  const T ru = up ? rL : rU;
  const T rcu = D ? (T)(up ? L.rc : U.rc) : (up ? rL * cL : rU * cU);
  const T sm = rL + rU;
  const T dct = D ? (T)dc : cU - cL;
  f.mp = t_ * ru;
  f.sp = t_ * rcu;
  const T qd = q_ * dr;
  const T qw = q_ * fma(dr, up ? cL : cU, ru);   // d(rho c)/dc of the upwind cell
  f.mLc = up ? qd : (T)0;
  f.mUc = up ? (T)0 : qd;
  // diffusion: d(-dco rbar dc)/dc from rbar (common), from dc (+, -)
  f.sLc = fma(h_, sm, fma(-h_ * dr, dct, up ? qw : (T)0));
  f.sUc = fma(-h_, sm, fma(-h_ * dr, dct, up ? (T)0 : qw));
  if (VERT) {
    const T s_ = -t_ * (T)gd * (T)0.5 * dr;       // dq/dc_L = dq/dc_U
    f.mLc = fma(s_, ru, f.mLc);
    f.mUc = fma(s_, ru, f.mUc);
    f.sLc = fma(s_, rcu, f.sLc);
    f.sUc = fma(s_, rcu, f.sUc);
  }
}

// C consecutive doubles; V: both the base and the column are even (16-byte
// aligned).
template <int C, bool V>
__device__ __forceinline__ void ld_row(double (&v)[C], const double* __restrict__ a) {
  if (V && C >= 2) {
#pragma unroll
    for (int k = 0; k + 1 < C; k += 2) {
      const double2 w = *reinterpret_cast<const double2*>(a + k);
      v[k] = w.x;
      v[k + 1] = w.y;
    }
  } else {
#pragma unroll
    for (int k = 0; k < C; ++k) v[k] = a[k];
  }
}

template <int C>
__device__ __forceinline__ void st_row(double* __restrict__ a, const double (&v)[C]) {
  if (C >= 2) {
#pragma unroll
    for (int k = 0; k + 1 < C; k += 2) *reinterpret_cast<double2*>(a + k) = make_double2(v[k], v[k + 1]);
  } else {
    a[0] = v[0];
  }
}

// Harmonic-mean face constants from the two cells' K and phi (OWN).
__device__ __forceinline__ void own_face(double ck, double cd, double k1, double f1, double k2,
                                         double f2, double& t, double& d) {
  t = (ck * k1) * (k2 * (1.0 / (k1 + k2)));
  d = (cd * f1) * (f2 * (1.0 / (f1 + f2)));
}

// T: multigrid type. C: columns per thread (nx a multiple of C). J: with
// the Jacobian. NAT: natural layout, R [B][2][ncell] and J [B][20][ncell]
// in FP64 (henry_residual_jacobian, the adjoint); else the row-scaled
// operator, b = -Dinv R and x = 0 in the colour-split layout. The solver's
// residual-only form takes the old time level's storage terms as arrays.
// OWN: full pressure, face constants and storage from phi and K. V: vector
// loads (nx even and every array 16-byte aligned). SPLIT: tl.split warps share
// a tile. Grid (tiles of a sample, B), 32 threads (times tl.split).
//
// Registers: a warp's registers come from its scheduler's 16,384, so 128 per
// thread keep 4 warps per scheduler, 168 keep 3 and 255 keep 2; the bounds
// below take the step that the kernel reaches without spilling.
constexpr int res_min_blocks(int C, bool J, bool own) { return J ? 8 : (own ? 12 : C == 4 ? 8 : 16); }
constexpr int kResSplitSlots = 152 * res_min_blocks(4, false, false);   // warps resident

template <typename T, int C, bool J, bool NAT, bool OWN, bool V, bool SPLIT = false, bool F32 = true>
__global__ void __launch_bounds__(SPLIT ? 32 * kResSplit : 32, res_min_blocks(C, J, OWN) / (SPLIT ? kResSplit : 1))
k_residual(unsigned long long* ctr, Phys P, Geom G, double vtau, ResTile tl, ResArgs A,
           T* __restrict__ Jm, T* __restrict__ bvec, T* __restrict__ xvec) {
  HENRY_COUNT_LAUNCH(ctr);
  constexpr bool PRE = !J && !NAT;                           // mo, so given
  constexpr bool TF = J && sizeof(T) == 4 && F32;            // face constants in FP32 given
  const int b = blockIdx.y;
  if (A.active && !A.active[b]) return;
  if (A.refresh && !A.refresh[b]) return;
  const int nx = G.nx, ny = G.ny, ncell = G.ncell(), half = G.half();
  const int lane = threadIdx.x & 31;
  const int grp = lane / tl.lpr, col = lane - grp * tl.lpr;
  const int by = blockIdx.x / tl.ntx, bx = blockIdx.x - by * tl.ntx;
  const int i0 = (bx * tl.lpr + col) * C;
  // SPLIT: rows per band, this warp's first band and rows
  const int h = SPLIT ? tl.R / kResSplit : 1, band0 = SPLIT ? (threadIdx.x >> 5) * (kResSplit / tl.split) : 0;
  const int rows = SPLIT ? tl.R / tl.split : tl.R;
  const int j0 = (by * tl.gpw + grp) * tl.R + band0 * h;
  const bool thr = grp < tl.gpw && i0 < nx;
  const bool last = i0 + C >= nx;                            // owns the right side
  const bool edge = thr && !last && col == tl.lpr - 1;       // east neighbour in the next tile
  const int64_t o = (int64_t)b * ncell + i0;                 // this thread's first column, row 0
  const double hd = 0.5 * P.drho, gdy = P.g * G.hy, hdg = hd * P.g * G.hy;
  const double wp = P.rho0 * P.g;                            // OWN: p' = p - wp (Ly - y)
  const double ckx = 2.0 * G.hy / (P.mu * G.hx), cdx = G.hy * P.D / G.hx;
  const double cky = 2.0 * G.hx / (P.mu * G.hy), cdy = G.hx * P.D / G.hy;
  const double dcoL = 2.0 * G.hy * P.D / G.hx;               // boundary diffusion per unit phi
  CellV me[C];
  T ct[C];                               // J: c in the multigrid type
  double Kme[C], fme[C];                 // OWN: K and phi of the row
  double FmS[C], FsS[C];                 // south faces
  FaceJ<T> jS[C];
#pragma unroll
  for (int k = 0; k < C; ++k) {
    FmS[k] = FsS[k] = 0.0;
    me[k].p = me[k].c = me[k].r = me[k].rc = 0.0;
    ct[k] = (T)0;
    Kme[k] = fme[k] = 1.0;
  }
  auto load_cells = [&](CellV (&v)[C], int j) {
    double a[C], d[C];
    ld_row<C, V>(a, A.p + o + (int64_t)j * nx);
    ld_row<C, V>(d, A.c + o + (int64_t)j * nx);
    const double w = OWN ? wp * (P.Ly - (j + 0.5) * G.hy) : 0.0;
#pragma unroll
    for (int k = 0; k < C; ++k) {
      v[k].p = OWN ? a[k] - w : a[k];
      v[k].c = d[k];
      cell_values(P, v[k]);
    }
  };
  // one face: f.x, f.y are (t, 2 dh) in FP32 (TF)
  auto face = [&](auto vert, const CellV& L, const CellV& U, double dp, double t, double dh, float fx,
                  float fy, T cL, T cU, double& q, double& Fm, double& Fs, FaceJ<T>& f) {
    constexpr bool VT = decltype(vert)::value;
    if constexpr (J)
      jac_face<T, VT>(P, L, U, dp, t, dh, gdy, TF ? (T)fx : (T)t, TF ? (T)0.5f * (T)fy : (T)dh, cL, cU, q, Fm, Fs, f);
    else
      res_face<VT>(P, L, U, t, dh, hdg, q, Fm, Fs);
  };
  using Hor = std::integral_constant<bool, false>;
  using Ver = std::integral_constant<bool, true>;
  if (thr && j0 < ny) {
    load_cells(me, j0);
    if (J) {
#pragma unroll
      for (int k = 0; k < C; ++k) ct[k] = (T)me[k].c;
    }
    if (OWN) {
      ld_row<C, V>(Kme, A.K + o + (int64_t)j0 * nx);
      ld_row<C, V>(fme, A.phi + o + (int64_t)j0 * nx);
    }
    if (j0 > 0) {                        // south faces of the first row
      const int64_t is = o + (int64_t)(j0 - 1) * nx;
      CellV S[C];
      double tv[C], dv[C];
      load_cells(S, j0 - 1);
      if (OWN) {
        double Ks[C], fs[C];
        ld_row<C, V>(Ks, A.K + is);
        ld_row<C, V>(fs, A.phi + is);
#pragma unroll
        for (int k = 0; k < C; ++k) own_face(cky, cdy, Ks[k], fs[k], Kme[k], fme[k], tv[k], dv[k]);
      } else {
        ld_row<C, V>(tv, A.ty + is);
        ld_row<C, V>(dv, A.dy + is);
      }
#pragma unroll
      for (int k = 0; k < C; ++k) {
        float4 f = {};
        if (TF) f = A.tf[is + k];
        double q;
        face(Ver{}, S[k], me[k], me[k].p - S[k].p, tv[k], dv[k], f.z, f.w, J ? (T)S[k].c : (T)0, ct[k], q, FmS[k], FsS[k], jS[k]);
      }
    }
  }
  __shared__ double band_sum[SPLIT ? kResSplit : 1][32];
  double v = 0.0;
  double w0 = 0.0, w1 = 0.0, edgeP = 0.0;
  FaceJ<T> wJ{};
#pragma unroll 1
  for (int r = 0; r < rows; ++r) {
    const int j = j0 + r;
    const bool cv = thr && j < ny;
    const int64_t id = o + (int64_t)j * nx;
    // boundary data of the next lpr rows, one row per lane of the group (a
    // single lane would cost the FP64 pipe as much for every row): the
    // seawater pressure right of the last column, the inflow and the
    // boundary conductance left of the first one, or the west face of a
    // tile's first column
    const int rl = r % tl.lpr;
    if (rl == 0) {
      const int jw = j0 + r + col;
      if (grp < tl.gpw && r + col < rows && jw < ny) {
        if (bx == tl.ntx - 1) {
          edgeP = P.Ly - (jw + 0.5) * G.hy;
          if (!J) edgeP = P.drho * P.g * edgeP;
        }
        // the tile's first column in row jw, by the form that compiles to the shorter launch
        // (FP32 Jacobian, 1024x512 x 16, us: 951 so, 993 by the other; FP64, 32x16 x 1024: 200, 189)
        const int64_t e = TF ? (int64_t)b * ncell + (int64_t)jw * nx + bx * tl.lpr * C
                             : o - col * C + (int64_t)jw * nx;
        if (bx == 0) {
          w0 = A.qin[(int64_t)b * ny + jw];
          w1 = dcoL * A.phi[e];
        } else {
          CellV W, Q;
          W.p = A.p[e - 1];
          Q.p = A.p[e];
          if (OWN) {
            const double w = wp * (P.Ly - (jw + 0.5) * G.hy);
            W.p -= w;
            Q.p -= w;
          }
          W.c = A.c[e - 1];
          Q.c = A.c[e];
          cell_values(P, W);
          cell_values(P, Q);
          double t, d, q;
          if (OWN) own_face(ckx, cdx, A.K[e - 1], A.phi[e - 1], A.K[e], A.phi[e], t, d);
          else { t = A.tx[e - 1]; d = A.dx[e - 1]; }
          float4 f = {};
          if (TF) f = A.tf[e - 1];
          face(Hor{}, W, Q, Q.p - W.p, t, d, f.x, f.y, J ? (T)W.c : (T)0, J ? (T)Q.c : (T)0, q, w0, w1, wJ);
        }
      }
    }
    const int src = grp * tl.lpr + rl;   // the lane that holds this row's boundary data
    // east neighbour of the last own column: the next lane's first column,
    // the next tile's from memory, or the seawater values at the right side
    // (reduced hydrostatic pressure, c = 1)
    CellV E;
    E.p = __shfl_down_sync(0xffffffffu, me[0].p, 1);
    E.c = __shfl_down_sync(0xffffffffu, me[0].c, 1);
    E.r = __shfl_down_sync(0xffffffffu, me[0].r, 1);
    E.rc = __shfl_down_sync(0xffffffffu, me[0].rc, 1);
    T ctE = (T)0;
    if (J) ctE = __shfl_down_sync(0xffffffffu, ct[0], 1);
    double KE = 1.0, fE = 1.0;
    if (OWN) {
      KE = __shfl_down_sync(0xffffffffu, Kme[0], 1);
      fE = __shfl_down_sync(0xffffffffu, fme[0], 1);
    }
    if (cv && edge) {
      E.p = A.p[id + C];
      if (OWN) E.p -= wp * (P.Ly - (j + 0.5) * G.hy);
      E.c = A.c[id + C];
      cell_values(P, E);
      if (J) ctE = (T)E.c;
      if (OWN) {
        KE = A.K[id + C];
        fE = A.phi[id + C];
      }
    }
    const double pb = __shfl_sync(0xffffffffu, edgeP, src);
    if (last) {
      E.p = pb;
      E.c = 1.0;
      E.r = E.rc = P.rho0 + P.drho;
      ctE = (T)1;
    }
    double qE[C], FmE[C], FsE[C], qN[C], FmN[C], FsN[C];
    FaceJ<T> jE[C], jN[C];
    CellV N[C];
    T ctN[C];
    double ph[C], a0[C], a1[C], a2[C];
#pragma unroll
    for (int k = 0; k < C; ++k) {
      qE[k] = FmE[k] = FsE[k] = qN[k] = FmN[k] = FsN[k] = 0.0;
      N[k].p = N[k].c = N[k].r = N[k].rc = 0.0;
      ctN[k] = (T)0;
      jE[k] = FaceJ<T>{};
      jN[k] = FaceJ<T>{};
    }
    if (cv) {
      double txv[C], dxv[C], tyv[C], dyv[C], KN[C], fN[C];
      const bool hn = j < ny - 1;
      if (!OWN) {
        ld_row<C, V>(txv, A.tx + id);
        ld_row<C, V>(dxv, A.dx + id);
        ld_row<C, V>(a0, A.vt + id);
      }
      if (PRE) {
        ld_row<C, V>(a1, A.mo + id);
        ld_row<C, V>(a2, A.so + id);
      } else {
        ld_row<C, V>(a1, A.c_old + id);
      }
      if (OWN) {
#pragma unroll
        for (int k = 0; k < C; ++k) ph[k] = fme[k];
      }
      if (hn) {
        load_cells(N, j + 1);
        if (J) {
#pragma unroll
          for (int k = 0; k < C; ++k) ctN[k] = (T)N[k].c;
        }
        if (OWN) {
          ld_row<C, V>(KN, A.K + id + nx);
          ld_row<C, V>(fN, A.phi + id + nx);
        } else {
          ld_row<C, V>(tyv, A.ty + id);
          ld_row<C, V>(dyv, A.dy + id);
        }
      }
      if (OWN) {
#pragma unroll
        for (int k = 0; k < C; ++k) {
          const int kn = k + 1 < C ? k + 1 : 0;
          const double k2 = k + 1 < C ? Kme[kn] : KE, f2 = k + 1 < C ? fme[kn] : fE;
          if (k == C - 1 && last) {      // the right side's coefficients
            txv[k] = ckx * Kme[k];
            dxv[k] = cdx * fme[k];
          } else {
            own_face(ckx, cdx, Kme[k], fme[k], k2, f2, txv[k], dxv[k]);
          }
          if (hn) own_face(cky, cdy, Kme[k], fme[k], KN[k], fN[k], tyv[k], dyv[k]);
        }
      }
#pragma unroll
      for (int k = 0; k < C; ++k) {
        const int kn = k + 1 < C ? k + 1 : 0;
        float4 f = {};
        if (TF) f = A.tf[id + k];
        const CellV& U = k + 1 < C ? me[kn] : E;
        // (right side: one rounding of the seawater pressure less the cell's)
        const double dp = k == C - 1 && last ? fma(P.drho * P.g, pb, -me[k].p) : U.p - me[k].p;
        face(Hor{}, me[k], U, dp, txv[k], dxv[k], f.x, f.y, ct[k],
             k + 1 < C ? ct[kn] : ctE, qE[k], FmE[k], FsE[k], jE[k]);
        if (J && k == C - 1 && last) {
          // right side: derivatives with respect to the cell, formed in FP64
          const double c = me[k].c, rho = me[k].r, rho1 = P.rho0 + P.drho;
          const double q = qE[k], tR = txv[k], dco = dxv[k] + dxv[k];
          const bool up = not_negative(q);
          const double rup = up ? rho : rho1, rcup = up ? rho * c : rho1, rb = 0.5 * (rho + rho1);
          jE[k].mp = (T)(tR * rup);
          jE[k].mLc = (T)(up ? q * P.drho : 0.0);
          jE[k].sp = (T)(tR * rcup);
          const double s = fma(-(dxv[k] * P.drho), 1.0 - c, up ? q * fma(P.drho, c, rho) : 0.0);
          jE[k].sLc = (T)__dadd_rn(s, __dmul_rn(dco, rb));
        }
        if (hn)
          face(Ver{}, me[k], N[k], N[k].p - me[k].p, tyv[k], dyv[k], f.z, f.w, ct[k], ctN[k], qN[k], FmN[k], FsN[k], jN[k]);
      }
      if (OWN) {
#pragma unroll
        for (int k = 0; k < C; ++k) {
          Kme[k] = KN[k];
          fme[k] = fN[k];
        }
      }
    }
    // west face of the first own column: the previous lane's last east face;
    // a tile's first column takes it from the lane that evaluated it
    double FmW = __shfl_up_sync(0xffffffffu, FmE[C - 1], 1);
    double FsW = __shfl_up_sync(0xffffffffu, FsE[C - 1], 1);
    FaceJ<T> jW{};
    if (J) {
      jW.mp = __shfl_up_sync(0xffffffffu, jE[C - 1].mp, 1);
      jW.sp = __shfl_up_sync(0xffffffffu, jE[C - 1].sp, 1);
      jW.mLc = __shfl_up_sync(0xffffffffu, jE[C - 1].mLc, 1);
      jW.mUc = __shfl_up_sync(0xffffffffu, jE[C - 1].mUc, 1);
      jW.sLc = __shfl_up_sync(0xffffffffu, jE[C - 1].sLc, 1);
      jW.sUc = __shfl_up_sync(0xffffffffu, jE[C - 1].sUc, 1);
    }
    const double l0 = __shfl_sync(0xffffffffu, w0, src), l1 = __shfl_sync(0xffffffffu, w1, src);
    if (col == 0) {
      FmW = bx > 0 ? l0 : 0.0;
      FsW = bx > 0 ? l1 : 0.0;
    }
    if (J && bx > 0) {
      FaceJ<T> g;
      g.mp = __shfl_sync(0xffffffffu, wJ.mp, src);
      g.sp = __shfl_sync(0xffffffffu, wJ.sp, src);
      g.mLc = __shfl_sync(0xffffffffu, wJ.mLc, src);
      g.mUc = __shfl_sync(0xffffffffu, wJ.mUc, src);
      g.sLc = __shfl_sync(0xffffffffu, wJ.sLc, src);
      g.sUc = __shfl_sync(0xffffffffu, wJ.sUc, src);
      if (col == 0) jW = g;
    }
    if (cv) {
      double Rp[C], Rc[C];
      T bp[C], bc[C];
#pragma unroll
      for (int k = 0; k < C; ++k) {
        const int kw = k ? k - 1 : 0;
        const double fmw = k ? FmE[kw] : FmW, fsw = k ? FsE[kw] : FsW;
        const double vt = OWN ? vtau * ph[k] : a0[k];
        double rp, rc;
        if (PRE) {
          const double a = vt * me[k].r;
          rp = (a - a1[k]) + FmE[k] + FmN[k] - fmw - FmS[k];
          rc = fma(a, me[k].c, -a2[k]) + FsE[k] + FsN[k] - fsw - FsS[k];
        } else {
          const double ro = fma(P.drho, a1[k], P.rho0);
          rp = fma(vt, me[k].r - ro, FmE[k]) + FmN[k] - fmw - FmS[k];
          rc = fma(vt, fma(me[k].r, me[k].c, -__dmul_rn(ro, a1[k])), FsE[k]) + FsN[k] - fsw - FsS[k];
        }
        const bool left = k == 0 && i0 == 0;
        if (left) {   // fresh-water inflow, diffusion to c = 0 at hx/2
          rp = fma(-(G.hy * P.rho0), l0, rp);
          rc = fma((0.5 * l1) * (me[0].r + P.rho0), me[0].c, rc);
        }
        T Jc[20];
        if (J) {
          const FaceJ<T>& w = k ? jE[kw] : jW;
          const FaceJ<T>& e = jE[k];
          const bool hw = !left, he = !(k == C - 1 && last), hn = j < ny - 1, hs = j > 0;
          const T z = (T)0;
          Jc[0] = Jc[2] = z;
          Jc[1] = (T)__dmul_rn(vt, P.drho);
          const double w3 = fma(P.drho, me[k].c, me[k].r);
          Jc[3] = (T)__dmul_rn(vt, w3);
          if (hw) { Jc[0] += w.mp; Jc[1] -= w.mUc; Jc[2] += w.sp; Jc[3] -= w.sUc; }
          else {
            const double t = fma(0.5 * P.drho, me[k].c, 0.5 * (me[k].r + P.rho0));
            if (sizeof(T) == 8) Jc[3] = (T)fma(l1, t, (double)Jc[3]);
            else Jc[3] += (T)(l1 * t);
          }
          Jc[0] += e.mp; Jc[1] += e.mLc; Jc[2] += e.sp; Jc[3] += e.sLc;
          if (hs) { Jc[0] += jS[k].mp; Jc[1] -= jS[k].mUc; Jc[2] += jS[k].sp; Jc[3] -= jS[k].sUc; }
          if (hn) { Jc[0] += jN[k].mp; Jc[1] += jN[k].mLc; Jc[2] += jN[k].sp; Jc[3] += jN[k].sLc; }
          Jc[4] = hw ? -w.mp : z; Jc[5] = hw ? -w.mLc : z;
          Jc[6] = hw ? -w.sp : z; Jc[7] = hw ? -w.sLc : z;
          Jc[8] = he ? -e.mp : z; Jc[9] = he ? e.mUc : z;
          Jc[10] = he ? -e.sp : z; Jc[11] = he ? e.sUc : z;
          Jc[12] = hs ? -jS[k].mp : z; Jc[13] = hs ? -jS[k].mLc : z;
          Jc[14] = hs ? -jS[k].sp : z; Jc[15] = hs ? -jS[k].sLc : z;
          Jc[16] = hn ? -jN[k].mp : z; Jc[17] = hn ? jN[k].mUc : z;
          Jc[18] = hn ? -jN[k].sp : z; Jc[19] = hn ? jN[k].sUc : z;
        }
        Rp[k] = rp;
        Rc[k] = rc;
        v = fma(rp, rp, fma(rc, rc, v));
        if (NAT) {
          if (J) {
            T* Jn = Jm + (int64_t)b * 20 * ncell + (int64_t)j * nx + i0 + k;
#pragma unroll
            for (int m = 0; m < 20; ++m) Jn[(int64_t)m * ncell] = Jc[m];
          }
        } else {
          const int cs = cs_pos(i0 + k, j, nx, half);
          T* Jb = Jm + (int64_t)b * kJP * ncell + cs;
          T d[4];   // Dinv of the operator the multigrid will use
          if (J) {
            store_operator<T>(Jb, ncell, Jc, d);
          } else {
#pragma unroll
            for (int m = 0; m < 4; ++m) d[m] = Jb[(int64_t)m * ncell];
          }
          const T mp = (T)(-rp), mc = (T)(-rc);
          bp[k] = d[0] * mp + d[1] * mc;
          bc[k] = d[2] * mp + d[3] * mc;
        }
      }
      if (NAT) {
        double* Rn = (double*)bvec + (int64_t)b * 2 * ncell + (int64_t)j * nx + i0;
#pragma unroll
        for (int k = 0; k < C; ++k) {
          Rn[k] = Rp[k];
          Rn[ncell + k] = Rc[k];
        }
      } else {
        const int64_t ob = (int64_t)b * 2 * ncell;
#pragma unroll
        for (int k = 0; k < C; ++k) {
          const int cs = cs_pos(i0 + k, j, nx, half);
          bvec[ob + cs] = bp[k];
          bvec[ob + ncell + cs] = bc[k];
          const bool red = A.guess && cs < half;
          xvec[ob + cs] = red ? bp[k] : (T)0;
          xvec[ob + ncell + cs] = red ? bc[k] : (T)0;
        }
        if (J) {
          st_row<C>(A.qx + id, qE);
          st_row<C>(A.qy + id, qN);
        }
      }
    }
#pragma unroll
    for (int k = 0; k < C; ++k) {
      me[k] = N[k];
      FmS[k] = FmN[k];
      FsS[k] = FsN[k];
      if (J) {
        ct[k] = ctN[k];
        jS[k] = jN[k];
      }
    }
    if (SPLIT && (r + 1) % h == 0) {
      band_sum[band0 + r / h][lane] = v;
      v = 0.0;
    }
  }
  if (SPLIT) {   // the tile's sum, in the order of its bands
    __syncthreads();
    if (threadIdx.x >= 32) return;
    v = band_sum[0][lane];
#pragma unroll
    for (int m = 1; m < kResSplit; ++m) v += band_sum[m][lane];
  }
  if (A.partial) {
#pragma unroll
    for (int s = 16; s > 0; s >>= 1) v += __shfl_down_sync(0xffffffffu, v, s);
    if (lane == 0) A.partial[(int64_t)b * gridDim.x + blockIdx.x] = v;
  }
}

static __global__ void k_scale(int64_t n, double f, double* __restrict__ v) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) v[i] *= f;
}

// Face fluxes of the state (p, c), as the residual-only form evaluates them
// (which does not store them: only a rebuild reads them): qx of the east faces,
// the right side in the last column, qy of the north faces. For diagnostics.
static __global__ void k_face_fluxes(Phys P, Geom G, int B, const double* __restrict__ p,
                                     const double* __restrict__ c, const double* __restrict__ tx,
                                     const double* __restrict__ ty, double* __restrict__ qx,
                                     double* __restrict__ qy) {
  const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= (int64_t)B * G.ncell()) return;
  const int cell = (int)(idx % G.ncell()), j = cell / G.nx, i = cell - j * G.nx;
  auto value = [&](int64_t at) {
    CellV v = {p[at], c[at], 0.0, 0.0};
    cell_values(P, v);
    return v;
  };
  const CellV L = value(idx);
  const double hd = 0.5 * P.drho, hdg = hd * P.g * G.hy;
  double q, m, s;
  if (i < G.nx - 1) {
    res_face<false>(P, L, value(idx + 1), tx[idx], 0.0, 0.0, q, m, s);
  } else {
    const double h = P.Ly - (j + 0.5) * G.hy;
    const CellV sea = {P.drho * P.g * h, 1.0, P.rho0 + P.drho, P.rho0 + P.drho};
    res_face<false>(P, L, sea, tx[idx], 0.0, 0.0, q, m, s);
  }
  qx[idx] = q;
  q = 0.0;
  if (j < G.ny - 1) res_face<true>(P, L, value(idx + G.nx), ty[idx], 0.0, hdg, q, m, s);
  qy[idx] = q;
}

}  // namespace henry
