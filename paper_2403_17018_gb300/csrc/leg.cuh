#pragma once
// One leg of a V-cycle on a large FP32 level in a single launch: the two
// pre-sweeps with the restricted residual (k_leg<false>), or the
// prolongation with the two post-sweeps (k_leg<true>).
//
// On large levels a half-sweep is bound by HBM: it reads half of the operator
// (the 16 off-diagonal planes of one colour), and a leg reads every plane
// twice. Here a warp walks up a strip of columns and runs all four
// half-sweeps of the leg on the way, each one row behind the one before it,
// so that an operator row is read once and stays in registers for its second
// use. In the colour-split layout lane k's red and black cell of row j are
// columns 2k and 2k + 1, a vertical neighbour is the same lane's, and a
// horizontal one is the same lane's or the next lane's: two shuffles an
// update and no barrier. Rows come through shared memory, three ahead of the
// one in use, each lane copying what it reads itself (loads one row ahead
// into registers: 197 us where this takes 181). Strips overlap by the four
// columns (two lanes) that four half-sweeps reach, chunks of rows by three
// below and three above; the overlap is computed twice, from the same values
// in the same order, so the results are bitwise those of one launch per
// operation. 1024x512 cells x 16: 181 us a leg, 4.6 TB/s of the 0.84 GB it
// needs; the four or five launches that it replaces took 260 us. FP64 levels
// keep the launches per operation: their sweeps are bound by the FP64 pipe.
#include "kernels.cuh"

namespace henry {
namespace {

constexpr int kLegWarps = 4;           // warps per block: neighbouring strips
constexpr int kLegBlocks = 2;          // blocks per SM (about 200 registers a thread)
constexpr int kLegSlots = 152 * kLegBlocks;
constexpr int kLegSets = 4;            // rows in flight: three ahead of the one in use
constexpr int kLegVals = 46;           // values per lane and row
constexpr int kLegSmem = kLegWarps * kLegSets * kLegVals * 32 * (int)sizeof(float);

struct LegTile {
  int own, off, ntx;   // lanes that own their cells, the first of them, strips
  int rows, nty;       // rows per chunk (even), chunks
  int64_t steps;       // rows that a block slot walks
  int blocks() const { return (ntx * nty + kLegWarps - 1) / kLegWarps; }
};

// Strips of at most 28 lanes' cells (32 where one holds the grid's width);
// the number of chunks that leaves the fewest rows per block slot.
inline LegTile make_leg_tile(const Geom& G, int B) {
  LegTile t;
  const int hx2 = G.nx / 2;
  t.ntx = hx2 <= 32 ? 1 : (hx2 + 27) / 28;
  t.off = t.ntx == 1 ? 0 : 2;
  t.own = (hx2 + t.ntx - 1) / t.ntx;
  int64_t best = -1;
  for (int n = 1; n <= (G.ny + 3) / 4; ++n) {
    const int rows = ((G.ny + n - 1) / n + 1) & ~1, nty = (G.ny + rows - 1) / rows;
    const int64_t blocks = (int64_t)(t.ntx * nty + kLegWarps - 1) / kLegWarps * B;
    const int64_t cost = (blocks + kLegSlots - 1) / kLegSlots * (rows + 6);
    if (best < 0 || cost < best) {
      t.steps = best = cost;
      t.rows = rows;
      t.nty = nty;
    }
  }
  return t;
}

// Whether the legs are worth it: a step takes 1.2 to 1.4 us and the launches
// per operation take 33 us a leg per million cells, so that the line lies at
// 42,500 cells a step. Measured per leg, one launch against four or five:
// 1024x512 x 16 181 us against 260, 512x256 x 16 63 against 72, 128x64 x 256
// (70 steps) 85 against 76, 256x128 x 16 23 against 20.
inline bool leg_pays(const Geom& G, int B, const LegTile& t) {
  return (int64_t)G.ncell() * B >= 42500 * t.steps;
}

// Copies of four bytes into this lane's own place in shared memory: no other
// lane reads it, so that waiting for the copies is all the order it needs.
__device__ __forceinline__ void leg_copy(float* dst, const float* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((unsigned)__cvta_generic_to_shared(dst)),
               "l"(src));
}
__device__ __forceinline__ void leg_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void leg_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// A is the colour swept first (black down: the guess has had its first red
// half-sweep; red up), O the other one. Step s runs: A on row s, O on row
// s - 1, A again on row s - 2, and on row s - 3 O again (up) or its residual,
// restricted (down). Rings of four rows hold the operators, right-hand sides
// and iterates. Grid (blocks, B), kLegSmem bytes of shared memory.
template <bool UP>
__global__ void __launch_bounds__(32 * kLegWarps, kLegBlocks)
k_leg(unsigned long long* ctr, Geom Gf, Geom Gc, LegTile tl, const int* __restrict__ active,
      const float* __restrict__ J, const float* __restrict__ bvec, const float* __restrict__ xin,
      float* __restrict__ xout, const float* __restrict__ xcin, const float* __restrict__ Jc,
      float* __restrict__ bc, float* __restrict__ xc) {
  HENRY_COUNT_LAUNCH(ctr);
  using T = float;
  extern __shared__ float leg_sh[];
  const int b = blockIdx.y;
  if (!active[b]) return;
  constexpr int A = UP ? 0 : 1, O = 1 - A;
  const unsigned all = 0xffffffffu;
  const int nx = Gf.nx, ny = Gf.ny, hx2 = nx >> 1, half = Gf.half(), ncell = Gf.ncell();
  const int ncc = Gc.ncell(), hc = Gc.half();
  const int lane = threadIdx.x & 31;
  const int w = blockIdx.x * kLegWarps + (threadIdx.x >> 5);
  const int by = w / tl.ntx, bx = w - by * tl.ntx;
  if (by >= tl.nty) return;   // a whole warp; no barrier below
  const int pos = bx * tl.own - tl.off + lane;
  const int kk = pos < 0 ? 0 : (pos < hx2 ? pos : hx2 - 1);   // loads stay in the grid
  const bool mine = lane >= tl.off && lane < tl.off + tl.own && pos < hx2;
  const bool hasW = pos > 0, hasE = pos < hx2 - 1;
  const int j0 = by * tl.rows, j1 = min(j0 + tl.rows, ny);
  const int64_t oJ = (int64_t)b * kJP * ncell + kk, o2 = (int64_t)b * 2 * ncell + kk;
  const T* JA = J + oJ + 4 * (int64_t)ncell + A * half;
  const T* JO = J + oJ + 4 * (int64_t)ncell + O * half;
  const T* bA = bvec + o2 + A * half;
  const T* bO = bvec + o2 + O * half;
  const T* xO = xin + o2 + O * half;
  T* yA = xout + o2 + A * half;
  T* yO = xout + o2 + O * half;
  const T* xcb = UP ? xcin + (int64_t)b * 2 * ncc : nullptr;
  const T* Dc = UP ? nullptr : Jc + (int64_t)b * kJP * ncc;
  T* bcb = UP ? nullptr : bc + (int64_t)b * 2 * ncc;
  T* xcd = UP ? nullptr : xc + (int64_t)b * 2 * ncc;
  // the place has the source's alignment (on widths of whole lines): a copy
  // shifted within its 128 bytes takes six passes over shared memory, not two
  T* sets = leg_sh + (threadIdx.x >> 5) * kLegSets * kLegVals * 32 + (pos & 31);

  T cA[4][16] = {}, cO[4][16] = {}, rA[4][2] = {}, rO[4][2] = {}, vA[4][2] = {}, vO[4][2] = {};
  T ep = 0, ec = 0;
  auto in = [&](int row) { return row < 0 ? 0 : (row < ny ? row : ny - 1); };
  // the values at the coarse cells that prolong_value reads for row r's O cell
  auto coarse = [&](int r, int (&q)[4]) {
    const int Jr = r >> 1;
    int I2 = kk + ((r & 1) ? -1 : 1), J2 = Jr + ((r & 1) ? 1 : -1);
    I2 = I2 < 0 ? 0 : (I2 >= Gc.nx ? Gc.nx - 1 : I2);
    J2 = J2 < 0 ? 0 : (J2 >= Gc.ny ? Gc.ny - 1 : J2);
    q[0] = cs_pos(kk, Jr, Gc.nx, hc), q[1] = cs_pos(I2, Jr, Gc.nx, hc);
    q[2] = cs_pos(kk, J2, Gc.nx, hc), q[3] = cs_pos(I2, J2, Gc.nx, hc);
  };
  // value v[m] of O's start (up: corrected) from x and four coarse values
  auto corrected = [&](T x, T x0, T x1, T x2, T x3) {
    const T w0 = (T)0.5625, w1 = (T)0.1875, w3 = (T)0.0625;
    return x + fma(w3, x3, fma(w0, x0, w1 * (x1 + x2)));
  };
  auto first = [&](int row, T (&v)[2]) {
    const int r = in(row);
    v[0] = xO[r * hx2];
    v[1] = xO[r * hx2 + ncell];
    if (UP) {
      int q[4];
      coarse(r, q);
#pragma unroll
      for (int m = 0; m < 2; ++m) {
        const T* x = xcb + m * ncc;
        v[m] = corrected(v[m], x[q[0]], x[q[1]], x[q[2]], x[q[3]]);
      }
    }
  };
  // what step s reads: A's operators and right-hand side on row s, O's on row
  // s - 1, O's start on row s + 1; down, D of row s - 3 and (its odd rows) the
  // coarse cell's blocks
  auto issue = [&](int s, int slot, bool odd) {
    T* d = sets + slot * kLegVals * 32;
    const T* p = JA + in(s) * hx2;
#pragma unroll
    for (int m = 0; m < 16; ++m) leg_copy(d + m * 32, p + (int64_t)m * ncell);
    p = JO + in(s - 1) * hx2;
#pragma unroll
    for (int m = 0; m < 16; ++m) leg_copy(d + (16 + m) * 32, p + (int64_t)m * ncell);
    p = bA + in(s) * hx2;
    leg_copy(d + 32 * 32, p), leg_copy(d + 33 * 32, p + ncell);
    p = bO + in(s - 1) * hx2;
    leg_copy(d + 34 * 32, p), leg_copy(d + 35 * 32, p + ncell);
    const int r1 = in(s + 1);
    p = xO + r1 * hx2;
    leg_copy(d + 36 * 32, p), leg_copy(d + 37 * 32, p + ncell);
    if (UP) {
      int q[4];
      coarse(r1, q);
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        leg_copy(d + (38 + m) * 32, xcb + q[m]);
        leg_copy(d + (42 + m) * 32, xcb + ncc + q[m]);
      }
    } else {
      const int r3 = in(s - 3);
      p = JO + r3 * hx2 + (int64_t)16 * ncell;
#pragma unroll
      for (int m = 0; m < 4; ++m) leg_copy(d + (38 + m) * 32, p + (int64_t)m * ncell);
      if (odd) {
        p = Dc + cs_pos(kk, r3 >> 1, Gc.nx, hc);
#pragma unroll
        for (int m = 0; m < 4; ++m) leg_copy(d + (42 + m) * 32, p + (int64_t)m * ncc);
      }
    }
  };
  // gs_point's operations on a cell of `row` whose missing horizontal
  // neighbour is the next lane's (east) or that of the lane before
  auto update = [&](bool east, int row, const T (&c)[16], T& rp, T& rc, const T (&own)[2],
                    const T (&S)[2], const T (&N)[2]) {
    const T op = east ? __shfl_down_sync(all, own[0], 1) : __shfl_up_sync(all, own[0], 1);
    const T oc = east ? __shfl_down_sync(all, own[1], 1) : __shfl_up_sync(all, own[1], 1);
    auto sub = [&](int m, T vp, T vc) {
      rp -= c[m] * vp;
      rp -= c[m + 1] * vc;
      rc -= c[m + 2] * vp;
      rc -= c[m + 3] * vc;
    };
    if (east) {
      sub(0, own[0], own[1]);
      if (hasE) sub(4, op, oc);
    } else {
      if (hasW) sub(0, op, oc);
      sub(4, own[0], own[1]);
    }
    if (row > 0) sub(8, S[0], S[1]);
    if (row < ny - 1) sub(12, N[0], N[1]);
  };

  const int s0 = j0 - 3;   // odd: row s0 + u is odd for even u
  const int steps = j1 - j0 + 6;
#pragma unroll
  for (int u = 0; u < kLegSets - 1; ++u) {
    issue(s0 + u, u, (u & 1) != 0);
    leg_commit();
  }
  first(s0 - 1, vO[3]);
  first(s0, vO[0]);
  for (int base = 0; base < steps; base += 4) {
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int s = s0 + base + u;
      const int e0 = u & 3, e1 = (u + 3) & 3, e2 = (u + 2) & 3, e3 = (u + 1) & 3;   // rows s, s-1, ..
      if (base + u + 3 < steps) issue(s + 3, e1, (u & 1) == 0);   // the slot of step s - 1
      leg_commit();
      leg_wait<kLegSets - 1>();
      const T* d = sets + e0 * kLegVals * 32;
      const T oldO[2] = {vO[e3][0], vO[e3][1]}, oldA[2] = {vA[e0][0], vA[e0][1]};   // rows s-3, s-4
#pragma unroll
      for (int m = 0; m < 16; ++m) {
        cA[e0][m] = d[m * 32];
        cO[e1][m] = d[(16 + m) * 32];
      }
#pragma unroll
      for (int m = 0; m < 2; ++m) {
        rA[e0][m] = d[(32 + m) * 32];
        rO[e1][m] = d[(34 + m) * 32];
        vO[e3][m] = d[(36 + m) * 32];   // row s + 1
        const T* x = d + (38 + 4 * m) * 32;
        if (UP) vO[e3][m] = corrected(vO[e3][m], x[0], x[32], x[64], x[96]);
      }
      // the colour's cell of an even row lies in column 2k (red) or 2k + 1
      const bool evenrow = (u & 1) != 0;   // of rows s and s - 2
      const bool eastA = evenrow == (A == 1), eastO = !evenrow == (O == 1);
      T rp, rc;
      rp = rA[e0][0], rc = rA[e0][1];
      update(eastA, s, cA[e0], rp, rc, vO[e0], vO[e1], vO[e3]);
      vA[e0][0] = rp, vA[e0][1] = rc;
      rp = rO[e1][0], rc = rO[e1][1];
      update(eastO, s - 1, cO[e1], rp, rc, vA[e1], vA[e2], vA[e0]);
      vO[e1][0] = rp, vO[e1][1] = rc;
      if (!UP && mine && s - 1 >= j0 && s - 1 < j1) {
        yO[(s - 1) * hx2] = rp;
        yO[ncell + (s - 1) * hx2] = rc;
      }
      rp = rA[e2][0], rc = rA[e2][1];
      update(eastA, s - 2, cA[e2], rp, rc, vO[e2], oldO, vO[e1]);
      vA[e2][0] = rp, vA[e2][1] = rc;
      if (mine && s - 2 >= j0 && s - 2 < j1) {
        yA[(s - 2) * hx2] = rp;
        yA[ncell + (s - 2) * hx2] = rc;
      }
      const int r = s - 3;
      rp = rO[e3][0], rc = rO[e3][1];
      if (!UP) {
        rp -= oldO[0];
        rc -= oldO[1];
      }
      update(eastO, r, cO[e3], rp, rc, vA[e3], oldA, vA[e2]);
      if (UP) {
        if (mine && r >= j0 && r < j1) {
          yO[r * hx2] = rp;
          yO[ncell + r * hx2] = rc;
        }
      } else {
        const T* D = d + 38 * 32;
        const T tp = fma(D[0], rp, D[32] * rc), tc = fma(D[64], rp, D[96] * rc);
        if (!evenrow) {          // r even: child 0 of its coarse cell; child 3 is the next row's
          ep = tp;
          ec = tc;
        } else if (mine && r >= j0 && r < j1) {
          const int Jr = r >> 1;
          const T sp = ep + tp, sc = ec + tc;
          const T* dc = d + 42 * 32;
          const T zp = fma(dc[0], sp, dc[32] * sc), zc = fma(dc[64], sp, dc[96] * sc);
          const int q = cs_pos(pos, Jr, Gc.nx, hc);
          const bool red = ((pos + Jr) & 1) == 0;
          bcb[q] = zp;
          bcb[ncc + q] = zc;
          xcd[q] = red ? zp : (T)0;      // the coarse guess after its first red half-sweep
          xcd[ncc + q] = red ? zc : (T)0;
        }
      }
      asm volatile("" ::: "memory");   // this set is read before its slot is written again
    }
  }
  leg_wait<0>();
}

}  // namespace
}  // namespace henry
