// Constants and helpers shared by all kernels of libhenry.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace henry {

constexpr int kNQ = 22;
constexpr int kStatusMaxit = 1;
constexpr int kStatusNonfinite = 2;
constexpr int kStatusBadInput = 4;
constexpr int kStatusStall = 8;      // a bounded wait for an asynchronous copy gave up
constexpr int kBlock = 256;
constexpr int kMaxCoarseUnknowns = 64;

#define HENRY_COUNT_LAUNCH(ctr)                                                        \
  do {                                                                                 \
    if (ctr && blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0 &&               \
        threadIdx.y == 0)                                                              \
      atomicAdd((unsigned long long*)(ctr), 1ULL);                                     \
  } while (0)

// ---------------------------------------------------------------------------
// One-dimensional bulk copies from global to shared memory by the TMA unit
// (cp.async.bulk), completing on an mbarrier in shared memory. A copy needs
// both addresses and its size to be multiples of 16 bytes (bulk_ok); callers
// copy anything else with plain loads. Waits are bounded by the global
// timer so that a copy that never lands cannot hang the block.
// ---------------------------------------------------------------------------
constexpr unsigned long long kBulkWaitNs = 200000000ull;   // 0.2 s

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ bool bulk_ok(const void* dst, const void* src, size_t bytes) {
  return bytes > 0 && ((((uintptr_t)dst) | ((uintptr_t)src) | (uintptr_t)bytes) & 15) == 0;
}

__device__ __forceinline__ void mbar_init(uint64_t* bar, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

// One arrival that also raises the barrier's expected transaction bytes.
__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t* bar, unsigned bytes) {
  asm volatile(
      "{\n .reg .b64 st;\n mbarrier.arrive.expect_tx.shared::cta.b64 st, [%0], %1;\n}" ::"r"(
          smem_u32(bar)),
      "r"(bytes)
      : "memory");
}

__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, unsigned bytes, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
          smem_u32(dst)),
      "l"(src), "r"(bytes), "r"(smem_u32(bar))
      : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, unsigned parity) {
  uint32_t done;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
      " selp.u32 %0, 1, 0, p;\n}"
      : "=r"(done)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return done != 0;
}

__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// Wait for phase `parity` of the barrier; false when kBulkWaitNs passed first.
__device__ __forceinline__ bool mbar_wait_bounded(uint64_t* bar, unsigned parity) {
  const unsigned long long t0 = global_ns();
  while (!mbar_try_wait(bar, parity))
    if (global_ns() - t0 > kBulkWaitNs) return false;
  return true;
}

// Stage the runs that runs(f) enumerates as f(destination in shared memory,
// source in global memory, bytes; every size a multiple of 4) with the
// whole block: one thread issues a TMA bulk copy for each 16-byte aligned
// run, all threads copy the others with plain loads; bar is an mbarrier in
// shared memory. Returns true once everything has landed. When a copy does
// not land within the bounded wait, sets kStatusStall in status[b], gives
// the copies in flight one more bounded wait and returns false (uniformly
// over the block: the caller returns; a block of a cluster first agrees
// with the others, see cluster_stage).
template <typename Runs>
__device__ __forceinline__ bool stage_runs(uint64_t* bar, Runs runs, int* status, int b) {
  unsigned tx = 0;
  runs([&](void* d, const void* src, unsigned bytes) { tx += bulk_ok(d, src, bytes) ? bytes : 0u; });
  if (threadIdx.x == 0 && tx > 0) {
    mbar_init(bar, 1);
    mbar_arrive_expect_tx(bar, tx);
    runs([&](void* d, const void* src, unsigned bytes) {
      if (bulk_ok(d, src, bytes)) bulk_g2s(d, src, bytes, bar);
    });
  }
  runs([&](void* d, const void* src, unsigned bytes) {
    if (bulk_ok(d, src, bytes)) return;
    uint32_t* dw = (uint32_t*)d;
    const uint32_t* sw = (const uint32_t*)src;
    for (unsigned e = threadIdx.x; e < bytes / 4; e += blockDim.x) dw[e] = sw[e];
  });
  __syncthreads();              // the barrier is initialised before anyone waits on it
  if (tx > 0 && !__syncthreads_and(mbar_wait_bounded(bar, 0))) {
    if (threadIdx.x == 0) status[b] |= kStatusStall;
    mbar_wait_bounded(bar, 0);
    return false;
  }
  return true;
}

// Block sum of a double, result valid in thread 0. Fixed order.
__device__ __forceinline__ double block_sum(double v, double* sh) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  __syncthreads();
  if (l == 0) sh[w] = v;
  __syncthreads();
  double s = 0.0;
  if (threadIdx.x == 0)
    for (int k = 0; k < (int)(blockDim.x >> 5); ++k) s += sh[k];
  return s;
}

// Tiling of k_residual (residual.cuh): lpr lanes share a row of a warp (C
// columns each), gpw row groups per warp, R rows per group; ntx x nty tiles
// cover a sample, a warp each, or `split` warps that share the rows.
struct ResTile {
  int lpr, gpw, R, ntx, nty, split;
  __host__ __device__ int tiles() const { return ntx * nty; }
};

constexpr int kResSplit = 4;   // bands of rows, and most warps, of a tile that warps may share

// rows 0 selects the tile height from the grid alone (never from the batch:
// the partial sums that decide convergence keep their order whatever the
// batch is). A tile evaluates its south faces again, so tall tiles do less
// work; short ones give a small batch more warps. Measured (us), residual
// only: 32x16 cells x 1 sample 12 with 2 rows of 2 columns, 18 (2 rows) and 29
// (4 rows) of 4 columns; x 1024 samples 57, 61, 49; 128x64 x 64 61 with 2 rows,
// 47 with 4, 57 with 8; 512x256 x 16 194 with 8, 166 with 16; 1024x512 x 16 661
// with 8, 717 with 16. With the Jacobian (FP32): 32x16 x 1 16 with 2 rows, 27
// with 4; 128x64 x 64 94 with 2, 89 with 4, 80 with 8, but x 16 25, 29, 47;
// 1024x512 x 16 978 with 8, 967 with 16.
//
// The lanes per row are those whose warps do the least work, counted in FP64
// instructions, which cost a warp the same however many lanes are active: per
// row and column 34 (with the Jacobian about 90), per group of rows the south
// faces again, per lpr rows the west face of a tile's first column. On widths
// that are a multiple of 32 C columns those are all 32. Residual only (FP32),
// us: 80x24 cells x 1024 322 with tiles of 32 and 8 lanes, 212 with five of 8;
// 192x160 x 256 852 with 32 and 16, 660 with three of 16.
__host__ inline ResTile make_res_tile(int nx, int ny, int C, int rows, bool jac) {
  const int lanes = (nx + C - 1) / C, cell = jac ? 90 : 34, face = jac ? 35 : 13;
  const int64_t ncell = (int64_t)nx * ny;
  if (rows <= 0)
    rows = jac ? (ncell <= 4096 ? 2 : (ncell <= 65536 ? 4 : (ncell <= 262144 ? 8 : 16)))
               : (ncell <= 4096 ? 2 : (ncell <= 65536 ? 4 : (ncell <= 262144 ? 16 : 8)));
  ResTile best = {};
  int64_t least = -1;
  for (int lpr = lanes < 32 ? lanes : 32; lpr >= 1; --lpr) {
    ResTile t = {};
    t.lpr = lpr;
    t.gpw = 32 / lpr;
    const int all = (ny + t.gpw - 1) / t.gpw;   // rows per group if a tile covered the height
    t.R = rows < all ? rows : all;
    t.ntx = (lanes + lpr - 1) / lpr;
    t.nty = (all + t.R - 1) / t.R;
    t.split = 1;
    const int64_t cost = (int64_t)t.tiles() * (t.R * C * cell + C * face +
                                               (t.ntx > 1 ? (t.R + lpr - 1) / lpr * face : 0));
    if (least < 0 || cost < least) {
      least = cost;
      best = t;
    }
  }
  return best;
}

// Warps that share a tile of B samples' grids, where the kernel allows it
// (its sum goes over kResSplit bands of rows either way, so that the batch
// leaves it as it is): those whose waves over `slots` resident warps take the
// fewest rows, a third of a row more for the south faces. Residual only, FP64,
// 512x256 cells, us with a warp per tile / so: x 1 102 / 34 (four), x 4 102 / 57
// (four), x 8 124 / 105 (two), x 16 175 / 175 (one), x 64 743 / 693 (two).
__host__ inline ResTile split_res_tile(ResTile t, int B, int slots) {
  int64_t least = -1;
  for (int s = 1; s <= kResSplit && t.R % kResSplit == 0; s *= 2) {
    const int64_t waves = ((int64_t)t.tiles() * B * s + slots - 1) / slots, cost = waves * (3 * t.R / s + 1);
    if (least < 0 || cost < least) {
      least = cost;
      t.split = s;
    }
  }
  return t;
}

// Inputs of k_residual.
struct ResArgs {
  const double* p;        // [B][ncell] reduced pressure (full pressure with OWN)
  const double* c;
  const double* c_old;    // old time level (otherwise)
  const double* phi;
  const double* K;        // OWN only
  const double* tx;       // face constants (without OWN), dx and dy halves; the
  const double* dx;       //   last column's east slots hold the right side's
  const double* ty;
  const double* dy;
  const float4* tf;       // (tx, dx, ty, dy), not halved (FP32 Jacobian)
  const double* qin;      // [B][ny]
  const double* vt;       // V phi / tau (without OWN); (V phi / tau) rho_old and
  const double* mo;       //   (V phi / tau) rho_old c_old (solver's residual)
  const double* so;
  const int* active;      // [B] or null
  const int* refresh;     // [B] or null: samples to skip
  double* partial;        // [B][warps] sums of R_p^2 + R_c^2, or null
  double* qx;             // face fluxes (WANT_J of the multigrid layout), or null
  double* qy;
  int guess;              // the guess xvec: 0, or with b on the red cells (its first half-sweep)
};

}  // namespace henry
