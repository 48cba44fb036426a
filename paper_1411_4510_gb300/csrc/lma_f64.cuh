// Right-looking blocked Cholesky of ONE FP64 matrix with appended rows, on
// 16 x 16 tiles: Sigma_SS (with identity rows appended, giving L^-T) and
// I + A of the global summary (identity rows and y appended, giving L_C^-T
// and L_C^-1 y).
//
// FP64 arithmetic is scarce on this part (under two FP64 FMAs per clock per
// SM, about 65 cycles of latency each), so the factorisation is a chain of
// small latency-bound steps.  Per column panel kp one launch does
//   * every trailing tile (i, j), kp < j <= i: solve L_ik = T_ik inv(L_kk)^T
//     and L_jk the same way in the CTA, then A_ij -= L_ik L_jk^T;  the CTA
//     of tile (kp + 1, kp + 1) then factorises it (the next diagonal factor);
//   * the in-place solve L_ik = T_ik inv(L_kk)^T of every tile of panel
//     kp - 1, deferred by one launch because the trailing update of panel
//     kp - 1 read T there; nobody reads column kp - 1 any more.
// A last launch (kp = npan) solves panel npan - 1.  The result is the
// factor L (zeros above the diagonal in the diagonal tiles), the appended
// rows (L^-1 Y)^T and the inverse diagonal tiles in dinv.
//
// Layout: row-major, leading dimension ld = npad (the padded order, a
// multiple of 16; padding rows/columns of the matrix hold the identity);
// rows [npad, rows) are appended rows.  The first nid appended rows are
// identity rows e_q^T: row tile e of them stays zero in every column panel
// k < e and is skipped there.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "lma_kernels.cuh"

namespace lma {
namespace f64 {

constexpr int TS = 16;     // tile order
constexpr int NTH = 64;    // threads per CTA (4 TS, as diag_factor needs)

// True when row tile i (appended row tile e = i - npan) holds only identity
// rows that are still zero in column panel k.
__device__ __forceinline__ bool zero_identity_tile(int i, int npan, int k, int nid) {
  const int e = i - npan;
  return e > k && (e + 1) * TS <= nid;
}

// Loads a TS x TS tile (rows >= rows read as zero).
__device__ __forceinline__ void load_tile(double (*dst)[TS + 1], const double* buf, int64_t ld, int r0, int c0,
                                          int rows) {
  for (int q = threadIdx.x; q < TS * TS; q += NTH) {
    const int r = q / TS, c = q % TS;
    dst[r][c] = (r0 + r < rows) ? buf[(int64_t)(r0 + r) * ld + c0 + c] : 0.0;
  }
}

// out = T X^T for a TS x TS tile (X = inv(L_kk), lower); thread t computes
// row t / 4, columns (t mod 4) + 4 q.
__device__ __forceinline__ void solve_tile(double (*out)[TS + 1], const double (*T)[TS + 1],
                                           const double (*X)[TS + 1]) {
  const int r = threadIdx.x >> 2, p = threadIdx.x & 3;
  double acc[TS / 4] = {};
#pragma unroll
  for (int k = 0; k < TS; ++k) {
    const double a = T[r][k];
#pragma unroll
    for (int q = 0; q < TS / 4; ++q) acc[q] = fma(a, X[p + 4 * q][k], acc[q]);
  }
#pragma unroll
  for (int q = 0; q < TS / 4; ++q) out[r][p + 4 * q] = acc[q];
}

// Factor of diagonal tile kp (the first panel; later diagonal tiles are
// factorised inside k_f64_panel).
__global__ void __launch_bounds__(NTH) k_f64_potrf(double* __restrict__ buf, int64_t ld, int kp,
                                                   double* __restrict__ dinv, int* __restrict__ info) {
  grid_dep_wait();
  grid_dep_launch();
  __shared__ double D[TS][TS + 1];
  double* A = buf + (int64_t)kp * TS * ld + kp * TS;
  load_tile(D, A, ld, 0, 0, TS);
  diag_factor<double, TS>(D, A, ld, dinv + (int64_t)kp * TS * TS, info, kp * TS);
}

// One launch per column panel kp (see the file comment).  Block order:
// [0, t1) matrix tiles (kp < j <= i < npan, block 0 = (kp + 1, kp + 1)),
// [t1, t2) appended-row tiles (i >= npan, kp < j < npan),
// [t2, t2 + nrt - kp) deferred solves of row tiles kp .. nrt - 1 of panel kp - 1.
__global__ void __launch_bounds__(NTH) k_f64_panel(double* __restrict__ buf, int64_t ld, int rows, int npan, int kp,
                                                   int nid, double* __restrict__ dinv, int* __restrict__ info) {
  grid_dep_wait();
  grid_dep_launch();
  const int nrt = (rows + TS - 1) / TS, napp = nrt - npan;
  const int m = npan - kp - 1;  // trailing panels (may be <= 0)
  const int t1 = m > 0 ? m * (m + 1) / 2 : 0;
  const int t2 = t1 + (m > 0 ? napp * m : 0);
  __shared__ double Ti[TS][TS + 1], Tj[TS][TS + 1], X[TS][TS + 1];
  __shared__ double Li[TS][TS + 1], Lj[TS][TS + 1];
  const int b = blockIdx.x;
  if (b >= t2) {  // deferred solve of tile (i, kp - 1)
    const int i = kp + (b - t2), k = kp - 1;
    if (k < 0 || zero_identity_tile(i, npan, k, nid)) return;
    load_tile(Ti, buf, ld, i * TS, k * TS, rows);
    load_tile(X, dinv + (int64_t)k * TS * TS, TS, 0, 0, TS);
    __syncthreads();
    solve_tile(Li, Ti, X);
    __syncthreads();
    for (int q = threadIdx.x; q < TS * TS; q += NTH) {
      const int r = q / TS, c = q % TS;
      if (i * TS + r < rows) buf[(int64_t)(i * TS + r) * ld + k * TS + c] = Li[r][c];
    }
    return;
  }
  int i, j;
  if (b < t1) {
    int I = (int)((sqrtf(8.f * (float)b + 1.f) - 1.f) * 0.5f);
    while (I * (I + 1) / 2 > b) --I;
    while ((I + 1) * (I + 2) / 2 <= b) ++I;
    i = kp + 1 + I;
    j = kp + 1 + (b - I * (I + 1) / 2);
  } else {
    const int q = b - t1;
    i = npan + q / m;
    j = kp + 1 + q % m;
  }
  const int r0 = i * TS, c0 = j * TS, k0 = kp * TS;
  if (zero_identity_tile(i, npan, kp, nid)) return;
  load_tile(Ti, buf, ld, r0, k0, rows);
  load_tile(X, dinv + (int64_t)kp * TS * TS, TS, 0, 0, TS);
  if (i != j) load_tile(Tj, buf, ld, c0, k0, rows);
  __syncthreads();
  solve_tile(Li, Ti, X);
  if (i != j) solve_tile(Lj, Tj, X);
  __syncthreads();
  const double(*LJ)[TS + 1] = (i != j) ? Lj : Li;
  const int r = threadIdx.x >> 2, p = threadIdx.x & 3;
  double acc[TS / 4] = {};
#pragma unroll
  for (int k = 0; k < TS; ++k) {
    const double a = Li[r][k];
#pragma unroll
    for (int q = 0; q < TS / 4; ++q) acc[q] = fma(a, LJ[p + 4 * q][k], acc[q]);
  }
  double* A = buf + (int64_t)r0 * ld + c0;
  if (b != 0) {
    if (r0 + r < rows)
#pragma unroll
      for (int q = 0; q < TS / 4; ++q) A[(int64_t)r * ld + p + 4 * q] -= acc[q];
    return;
  }
  // tile (kp + 1, kp + 1): update into shared memory, factorise, store
#pragma unroll
  for (int q = 0; q < TS / 4; ++q) Tj[r][p + 4 * q] = A[(int64_t)r * ld + p + 4 * q] - acc[q];
  diag_factor<double, TS>(Tj, A, ld, dinv + (int64_t)(kp + 1) * TS * TS, info, c0);
}

// Two-phase variant (two launches per column panel, no repeated solves):
// k_f64_solve2 solves every tile of panel kp below the diagonal in place,
// L_ik = T_ik inv(L_kk)^T (identity-row tiles that are still zero are
// skipped); k_f64_update2 then applies A_ij -= L_ik L_jk^T to every trailing
// tile (kp < j <= i < npan, and the appended-row tiles i >= npan, kp < j <
// npan) from the solved tiles, and its CTA 0 (tile (kp + 1, kp + 1))
// factorises that diagonal tile.  Each trailing tile thus does one product
// instead of two solves and a product, which pays at large orders.
__global__ void __launch_bounds__(NTH) k_f64_solve2(double* __restrict__ buf, int64_t ld, int rows, int npan, int kp,
                                                    int nid, const double* __restrict__ dinv) {
  grid_dep_wait();
  grid_dep_launch();
  const int i = kp + 1 + blockIdx.x;
  if (zero_identity_tile(i, npan, kp, nid)) return;
  __shared__ double Ti[TS][TS + 1], X[TS][TS + 1], Li[TS][TS + 1];
  load_tile(Ti, buf, ld, i * TS, kp * TS, rows);
  load_tile(X, dinv + (int64_t)kp * TS * TS, TS, 0, 0, TS);
  __syncthreads();
  solve_tile(Li, Ti, X);
  __syncthreads();
  for (int q = threadIdx.x; q < TS * TS; q += NTH) {
    const int r = q / TS, c = q % TS;
    if (i * TS + r < rows) buf[(int64_t)(i * TS + r) * ld + kp * TS + c] = Li[r][c];
  }
}

__global__ void __launch_bounds__(NTH) k_f64_update2(double* __restrict__ buf, int64_t ld, int rows, int npan,
                                                     int kp, int nid, double* __restrict__ dinv,
                                                     int* __restrict__ info) {
  grid_dep_wait();
  grid_dep_launch();
  const int napp = (rows + TS - 1) / TS - npan;
  const int m = npan - kp - 1;
  const int t1 = m * (m + 1) / 2;
  const int b = blockIdx.x;
  int i, j;
  if (b < t1) {
    int I = (int)((sqrtf(8.f * (float)b + 1.f) - 1.f) * 0.5f);
    while (I * (I + 1) / 2 > b) --I;
    while ((I + 1) * (I + 2) / 2 <= b) ++I;
    i = kp + 1 + I;
    j = kp + 1 + (b - I * (I + 1) / 2);
  } else {
    const int q = b - t1;
    if (q >= napp * m) return;
    i = npan + q / m;
    j = kp + 1 + q % m;
  }
  if (zero_identity_tile(i, npan, kp, nid)) return;
  __shared__ double Li[TS][TS + 1], Lj[TS][TS + 1], Tj[TS][TS + 1];
  const int r0 = i * TS, c0 = j * TS, k0 = kp * TS;
  load_tile(Li, buf, ld, r0, k0, rows);
  if (i != j) load_tile(Lj, buf, ld, c0, k0, rows);
  __syncthreads();
  const double(*LJ)[TS + 1] = (i != j) ? Lj : Li;
  const int r = threadIdx.x >> 2, p = threadIdx.x & 3;
  double acc[TS / 4] = {};
#pragma unroll
  for (int k = 0; k < TS; ++k) {
    const double a = Li[r][k];
#pragma unroll
    for (int qq = 0; qq < TS / 4; ++qq) acc[qq] = fma(a, LJ[p + 4 * qq][k], acc[qq]);
  }
  double* A = buf + (int64_t)r0 * ld + c0;
  if (b != 0) {
    if (r0 + r < rows)
#pragma unroll
      for (int qq = 0; qq < TS / 4; ++qq) A[(int64_t)r * ld + p + 4 * qq] -= acc[qq];
    return;
  }
#pragma unroll
  for (int qq = 0; qq < TS / 4; ++qq) Tj[r][p + 4 * qq] = A[(int64_t)r * ld + p + 4 * qq] - acc[qq];
  diag_factor<double, TS>(Tj, A, ld, dinv + (int64_t)(kp + 1) * TS * TS, info, c0);
}

// ---------------------------------------------------------------------------
// Persistent form: the whole right-looking factorisation in ONE cooperative
// launch (all CTAs resident), the launch boundaries of the two-phase form
// replaced by grid barriers.  At order 512 the two-phase form is 64 launches
// of a few microseconds of work each, so launch latency, not the FP64 pipe,
// set its time.  Per column panel kp:
//   solve phase   every tile (i, kp), i > kp, becomes T_ik inv(L_kk)^T;
//   barrier;
//   update phase  A_ij -= L_ik L_jk^T over the trailing tiles, CTA 0 taking
//                 tile (kp + 1, kp + 1) first and factorising it;
//   barrier.
// Tiles are dealt to CTAs round-robin.  Data written by other CTAs during
// the launch is read with ld.global.cg (L2), never through L1.

constexpr uint32_t kBarrierSpin = 1u << 22;  // polls before a grid barrier gives up

// Grid-wide barrier: *bar (zero before the launch) counts arrivals, barrier
// number g completes at g * gridDim.x.  Gives up after kBarrierSpin polls or
// once another CTA gave up (*err != 0), setting *err; returns false then.
__device__ __forceinline__ bool grid_barrier(unsigned* bar, unsigned& gen, int* err) {
  __shared__ int ok;
  __syncthreads();
  if (threadIdx.x == 0) {
    const unsigned target = ++gen * gridDim.x;
    __threadfence();
    atomicAdd(bar, 1u);
    int good = 1;
    for (uint32_t it = 0;; ++it) {
      unsigned v;
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(bar) : "memory");
      if (v >= target) break;
      if (it >= kBarrierSpin || ((it & 1023u) == 1023u && *(volatile int*)err)) {
        good = 0;
        atomicExch(err, 1);
        break;
      }
    }
    __threadfence();
    ok = good;
  }
  __syncthreads();
  return ok != 0;
}

// load_tile through L2 (the tile may have been written by another CTA).
__device__ __forceinline__ void load_tile_cg(double (*dst)[TS + 1], const double* buf, int64_t ld, int r0, int c0,
                                             int rows) {
  for (int q = threadIdx.x; q < TS * TS; q += NTH) {
    const int r = q / TS, c = q % TS;
    dst[r][c] = (r0 + r < rows) ? __ldcg(buf + (int64_t)(r0 + r) * ld + c0 + c) : 0.0;
  }
}

__global__ void __launch_bounds__(NTH) k_f64_coop(double* buf, int64_t ld, int rows, int npan, int nid,
                                                  double* dinv, int* info, unsigned* bar, int* err) {
  __shared__ double Ti[TS][TS + 1], X[TS][TS + 1], Li[TS][TS + 1], Lj[TS][TS + 1];
  const int G = gridDim.x, nrt = (rows + TS - 1) / TS, napp = nrt - npan;
  const int r = threadIdx.x >> 2, p = threadIdx.x & 3;
  unsigned gen = 0;
  if (blockIdx.x == 0) {
    load_tile_cg(Ti, buf, ld, 0, 0, rows);
    diag_factor<double, TS>(Ti, buf, ld, dinv, info, 0);
  }
  if (!grid_barrier(bar, gen, err)) return;
  for (int kp = 0; kp < npan; ++kp) {
    // solve phase
    for (int t = blockIdx.x; t < nrt - kp - 1; t += G) {
      const int i = kp + 1 + t;
      if (zero_identity_tile(i, npan, kp, nid)) continue;
      load_tile_cg(Ti, buf, ld, i * TS, kp * TS, rows);
      load_tile_cg(X, dinv + (int64_t)kp * TS * TS, TS, 0, 0, TS);
      __syncthreads();
      solve_tile(Li, Ti, X);
      __syncthreads();
      for (int q = threadIdx.x; q < TS * TS; q += NTH) {
        const int rr = q / TS, c = q % TS;
        if (i * TS + rr < rows) buf[(int64_t)(i * TS + rr) * ld + kp * TS + c] = Li[rr][c];
      }
      __syncthreads();
    }
    const int m = npan - kp - 1;
    if (m <= 0) break;
    if (!grid_barrier(bar, gen, err)) return;
    // update phase
    const int t1 = m * (m + 1) / 2, total = t1 + napp * m;
    for (int b = blockIdx.x; b < total; b += G) {
      int i, j;
      if (b < t1) {
        int I = (int)((sqrtf(8.f * (float)b + 1.f) - 1.f) * 0.5f);
        while (I * (I + 1) / 2 > b) --I;
        while ((I + 1) * (I + 2) / 2 <= b) ++I;
        i = kp + 1 + I;
        j = kp + 1 + (b - I * (I + 1) / 2);
      } else {
        const int q = b - t1;
        i = npan + q / m;
        j = kp + 1 + q % m;
      }
      if (zero_identity_tile(i, npan, kp, nid)) continue;
      const int r0 = i * TS, c0 = j * TS, k0 = kp * TS;
      load_tile_cg(Li, buf, ld, r0, k0, rows);
      if (i != j) load_tile_cg(Lj, buf, ld, c0, k0, rows);
      __syncthreads();
      const double(*LJ)[TS + 1] = (i != j) ? Lj : Li;
      double acc[TS / 4] = {};
#pragma unroll
      for (int k = 0; k < TS; ++k) {
        const double a = Li[r][k];
#pragma unroll
        for (int qq = 0; qq < TS / 4; ++qq) acc[qq] = fma(a, LJ[p + 4 * qq][k], acc[qq]);
      }
      double* A = buf + (int64_t)r0 * ld + c0;
      if (b != 0) {
        if (r0 + r < rows)
#pragma unroll
          for (int qq = 0; qq < TS / 4; ++qq) {
            double* a = A + (int64_t)r * ld + p + 4 * qq;
            *a = __ldcg(a) - acc[qq];
          }
      } else {
#pragma unroll
        for (int qq = 0; qq < TS / 4; ++qq) Ti[r][p + 4 * qq] = __ldcg(A + (int64_t)r * ld + p + 4 * qq) - acc[qq];
        diag_factor<double, TS>(Ti, A, ld, dinv + (int64_t)(kp + 1) * TS * TS, info, c0);
      }
      __syncthreads();
    }
    if (!grid_barrier(bar, gen, err)) return;
  }
}

// ---------------------------------------------------------------------------
// Dataflow form (one cooperative launch, at most one CTA per SM).  What bounds
// it: each of the SM's four schedulers takes one FP64 warp instruction per 64
// clocks, whatever the number of active lanes, and a warp's next one waits for
// it even when independent (measured: 64.6 clocks an FMA at 1 warp, 16.1 at 4 and
// more).  So a serial step costs 64 clocks per FP64 instruction of its warp, and
// work has to be spread over warps of all four schedulers.  The factorisation's
// chain is 16 columns per panel, each a reciprocal square root (357 clocks), two
// products and an FMA.  Hence three roles:
//   * CTA 0, the chain, alone on its SM: warp 0 (alone on its scheduler) runs the
//     pivot columns of diagonal tile k and applies each to the next column only;
//     warps 1-3 apply it to the columns after that and hand them back in time, and
//     warps 13-15 build the tile's inverse behind it.  Then all solve (k + 1, k),
//     apply it to (k + 1, k + 1) and go on: no global round trip between two panels,
//     and the fences that publish a panel are warp 12's, which no barrier of the
//     others waits for.
//   * CTAs 1 .. nband, the band, four warps (one per scheduler) each: row i's tiles
//     (i, i - 2), (i, i - 1) and (i, i).  When panel i - 2 is there, such a group solves
//     the first, applies it to the other two and hands them to the chain, all without
//     a round trip of its own; it shares its SM with nobody, as the chain waits for it
//     16 columns later.
//   * every group of four warps of the other CTAs owns whole tiles (i, j): it applies
//     A_ij -= L_ik L_jk^T for k = 0 .. j - 1 as those tiles become final, solves
//     against inv(L_jj) and publishes the tile.
// prog[i] counts the final tiles of row tile i (they become final in column
// order), xprog the published inverses; both are polled in L2.  The bulk's tiles
// are listed column by column, a group takes its tiles in list order and a band CTA
// its rows in ascending order; a bulk tile of column j waits for the chain's panels
// and the band's rows up to j only, those for bulk tiles of lower columns, so with
// all CTAs resident every wait ends.  Identity-row tiles that stay zero are left
// out, and so are the padding panels.  The operations on each element and their
// order are those of a plain tile loop (k ascending, one FMA per term).
//
// Order 512 with 512 identity rows: 0.82 ms -> 0.26 (before: one 64-thread CTA
// per tile, per-tile flags, a CTA barrier per column of the diagonal tile); order
// 1,024: 1.92 -> 0.76; order 2,048: 7.1 -> 5.5 (the FP64 pipe alone: 5).

constexpr int FW = 16;          // warps per CTA
constexpr int FTH = 32 * FW;    // threads per CTA
constexpr int FG = FW / 4;      // groups per CTA
constexpr int FP = TS + 2;      // row pitch of a group's tiles (16-byte aligned, conflict-free)
constexpr int CSTR = 32;        // prog counters lie 128 bytes apart

struct alignas(16) FlowBulk {   // per group (its rows are read 16 bytes at a time)
  double a[TS][FP], b[TS][FP];
  unsigned have;
};
struct alignas(16) FlowBand {
  double li[TS][FP], l1[TS][FP], l2[TS][FP];
  unsigned have;
};
constexpr int kBand = 16;       // band CTAs at most: 16 rows ahead of the chain
struct FlowChain {
  double D[TS][TS + 1], X[TS][TS + 1], T[TS][TS + 1], A[TS][TS + 1], Ls[TS][TS + 1], Lt[TS][TS + 1];
  // slots (one set per panel): column j of the diagonal tile times 1 / pivot, and as it is; column j up to date
  // but for column j - 1; reciprocal square root of pivot j
  double cola[TS][TS], colc[TS][TS], next[TS][TS], rj[TS];
  int bad;
};
union alignas(16) FlowSmem {
  FlowBulk g[FG];
  FlowBand b;
  FlowChain c;
  __device__ FlowSmem() {}
};

__device__ __forceinline__ unsigned ld_acq(const unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_rel(unsigned* p, unsigned v) {
  asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ void bar_arrive(int id, int threads) {
  asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(threads) : "memory");
}
__device__ __forceinline__ void bar_sync(int id, int threads) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}

// One thread waits until *f >= want; false on timeout or once another CTA gave up.
__device__ __forceinline__ bool wait_count(const unsigned* f, unsigned want, int* err) {
  for (uint32_t it = 0;; ++it) {
    if (ld_acq(f) >= want) return true;
    if (it >= kBarrierSpin || ((it & 255u) == 255u && *(volatile int*)err)) {
      atomicExch(err, 1);
      return false;
    }
  }
}

// A warp waits until both counters reach `want`; returns the smaller one (0: gave up).
__device__ __forceinline__ unsigned wait_rows(const unsigned* fi, const unsigned* fj, unsigned want, int* err) {
  const int lane = threadIdx.x & 31;
  for (uint32_t it = 0;; ++it) {
    unsigned v = 0xffffffffu;
    if (lane == 0) v = ld_acq(fi);
    if (lane == 1) v = ld_acq(fj);
    const unsigned m = min(__shfl_sync(0xffffffffu, v, 0), __shfl_sync(0xffffffffu, v, 1));
    if (m >= want) return m;
    int stop = 0;
    if (lane == 0 && (it >= kBarrierSpin || ((it & 255u) == 255u && *(volatile int*)err))) {
      atomicExch(err, 1);
      stop = 1;
    }
    if (__shfl_sync(0xffffffffu, stop, 0)) return 0;
    __nanosleep(40);
  }
}

// Values handed from warp to warp inside the chain CTA announce themselves: a slot holds kEmpty (a NaN whose
// payload no arithmetic gives) until its value is written, so neither a fence nor a flag lies between a store
// and its use (a fence and a flag cost about 300 clocks a column, an mbarrier more).
constexpr unsigned long long kEmpty = 0xFFFFFFFFFFFFFFF1ull;
__device__ __forceinline__ double take_slot(const double* p, volatile int* bad) {
  const volatile unsigned long long* q = reinterpret_cast<const volatile unsigned long long*>(p);
  unsigned long long v = *q;
  for (uint32_t it = 0; v == kEmpty; ++it) {
    if (it >= kBarrierSpin) {
      *bad = 1;
      break;
    }
    v = *q;
  }
  return __longlong_as_double((long long)v);
}
__device__ __forceinline__ void put_slot(double* p, double v) { *reinterpret_cast<volatile double*>(p) = v; }

// First row of row tile i (matrix tiles i < npan, then the appended rows from row ld on).
__device__ __forceinline__ int flow_row0(int i, int npan, int64_t ld) {
  return i < npan ? i * TS : (int)ld + (i - npan) * TS;
}

// Row and column of element e of a lower triangle listed row by row.
__device__ __forceinline__ void tri_element(int e, int& r, int& c) {
  r = (int)((sqrtf(8.f * (float)e + 1.f) - 1.f) * 0.5f);
  while (r * (r + 1) / 2 > e) --r;
  while ((r + 1) * (r + 2) / 2 <= e) ++r;
  c = e - r * (r + 1) / 2;
}

// The chain CTA.  hsub[k] / hdiag[k] (0 or 1): tile (k + 1, k) / (k, k) handed over with every panel below k /
// k - 1 applied.  Returns false in every thread once a wait has given up.  c.bad is cleared by the caller ahead of the
// first call and stays set from then on: the publishing warp may read it a panel later than the others.
__device__ bool flow_chain(FlowChain& c, double* buf, int64_t ld, int npan, double* dinv, int* info, unsigned* prog,
                           unsigned* xprog, const unsigned* hsub, const unsigned* hdiag, int* err) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int r = lane & 15, h = lane >> 4;
  volatile int* bad = &c.bad;
  if (tid < TS * TS) {
    const int rr = tid / TS, cc = tid % TS;
    c.D[rr][cc] = cc <= rr ? __ldcg(buf + (int64_t)rr * ld + cc) : 0.0;
  }
  auto clear_slots = [&](int q) {  // q < 256
    const double e = __longlong_as_double((long long)kEmpty);
    c.cola[q / TS][q % TS] = c.colc[q / TS][q % TS] = c.next[q / TS][q % TS] = e;
    if (q < TS) c.rj[q] = e;
  };
  if (tid >= FTH - TS * TS) clear_slots(tid - (FTH - TS * TS));
  int er = 0, ec = 0;  // this thread's element of the (k + 1, k + 1) update
  if (tid < 128) tri_element(tid, er, ec);
  double tcorner = 0.0;  // warp 4, lanes 0-7: element (15, 8 + lane) before that update
  constexpr int MT = FTH - 32;  // threads at the barriers of the chain (all but the publishing warp)
  __syncthreads();
  if (warp == 12) {  // publishes: inv(L_kk) and L_kk after stage A, (k + 1, k) after the solve
    // Barrier ids alternate with the panel: when the others arrive for panel k, this warp is past panel k - 2,
    // since their panel k - 1 needed bulk tiles that needed xprog >= k - 1.
    for (int k = 0; k < npan; ++k) {
      bar_sync(6 + 2 * (k & 1), FTH);
      if (*bad) return false;
      if (lane == 0) {
        __threadfence();
        st_rel(xprog, (unsigned)(k + 1));
      }
      __syncwarp();
      if (k + 1 == npan) return true;
      bar_sync(7 + 2 * (k & 1), FTH);
      if (lane == 0) {
        __threadfence();
        st_rel(prog + (int64_t)(k + 1) * CSTR, (unsigned)(k + 1));
      }
      __syncwarp();
    }
    return true;
  }
  for (int k = 0; k < npan; ++k) {
    const bool more = k + 1 < npan;
    const int k0 = k * TS, r1 = k0 + TS;
    if (warp == 0) {
      double cur = c.D[r][0];
#pragma unroll
      for (int j = 0; j < TS; ++j) {
        double piv = __shfl_sync(0xffffffffu, cur, j);
        const double cvn = __shfl_sync(0xffffffffu, cur, j < TS - 1 ? j + 1 : j);
        double lr = cur;
        const long long bits = __double_as_longlong(piv);
        if (!(bits > 0 && bits <= 0x7FF0000000000000LL)) {  // not (piv > 0)
          if (lane == 0 && *info == 0) *info = k0 + j + 1;
          piv = 1.0;
          if (r == j) lr = 1.0;
        }
        const double rj = rsqrt(piv);
        const double l = lr * rj;
        double nx = 0.0;
        if (j + 1 < TS) {
          nx = j + 1 >= 2 ? take_slot(&c.next[j + 1][r], bad) : c.D[r][1];
        }
        const double a = l * rj;
        nx = fma(-a, cvn, nx);
        if (h == 0) {
          put_slot(&c.cola[j][r], a);
          put_slot(&c.colc[j][r], cur);
          c.Lt[r][j] = r >= j ? l : 0.0;
          if (r == 0) put_slot(&c.rj[j], rj);
        }
        cur = nx;
      }
    } else if (warp < 4) {
      // columns 3 m + warp - 1 of the diagonal tile, m = 2 s + h
      double v[3];
#pragma unroll
      for (int s = 0; s < 3; ++s) {
        const int col = 3 * (2 * s + h) + warp - 1;
        v[s] = col <= r ? c.D[r][col] : 0.0;
      }
#pragma unroll
      for (int j = 0; j < TS - 2; ++j) {
        const double a = take_slot(&c.cola[j][r], bad);
        const int m = (j + 2) / 3;  // column j + 2 is slot m >> 1, half m & 1 of warp (j + 2) % 3 + 1
#pragma unroll
        for (int s0 = 0; s0 < 3; ++s0) {
          const int s = s0 == 0 ? (m >> 1) : (s0 <= (m >> 1) ? s0 - 1 : s0);  // column j + 2's slot first
          if (s < (m >> 1)) continue;                                          // its columns are final
          const int col = 3 * (2 * s + h) + warp - 1;
          if (col >= j + 2 && col < TS) v[s] = fma(-a, take_slot(&c.colc[j][col], bad), v[s]);
          if (s0 == 0 && warp - 1 == (j + 2) % 3 && h == (m & 1) && (r < 15 || j + 2 < 8))
            put_slot(&c.next[j + 2][r], v[s]);
        }
      }
    } else if (warp == 4) {
      // elements (15, 8 + lane), first the (k, k) update (the others' is done before the barrier), then the columns
      if (lane < 8) {
        double t = k > 0 ? tcorner : c.D[15][8 + lane];
        if (k > 0)
#pragma unroll
          for (int kk = 0; kk < TS; ++kk) t = fma(-c.Ls[15][kk], c.Ls[8 + lane][kk], t);
#pragma unroll
        for (int j = 0; j < TS - 2; ++j) {
          const double a = take_slot(&c.cola[j][15], bad);
          if (8 + lane >= j + 2) t = fma(-a, take_slot(&c.colc[j][8 + lane], bad), t);
          if (8 + lane == j + 2) put_slot(&c.next[j + 2][15], t);
        }
      }
      __syncwarp();
    } else if (warp >= 13) {
      // inverse: x[r][c] -= a_r x[j][c] for r > j, rows scaled at the end; column pairs q = warp - 13 + 3 s
      double x[3];
#pragma unroll
      for (int s = 0; s < 3; ++s) x[s] = (2 * (warp - 13 + 3 * s) + h == r) ? 1.0 : 0.0;
#pragma unroll
      for (int j = 0; j < TS - 1; ++j) {
        const double a = take_slot(&c.cola[j][r], bad);
#pragma unroll
        for (int s = 0; s < 3; ++s)
          if (2 * (warp - 13 + 3 * s) <= j) {
            const double xv = __shfl_sync(0xffffffffu, x[s], j + 16 * h);
            if (r > j) x[s] = fma(-a, xv, x[s]);
          }
      }
      const double rj = take_slot(&c.rj[r], bad);
      double* Dv = dinv + (int64_t)k * TS * TS;
#pragma unroll
      for (int s = 0; s < 3; ++s) {
        const int cc = 2 * (warp - 13 + 3 * s) + h;
        if (cc >= TS) break;
        x[s] *= rj;
        c.X[r][cc] = x[s];
        Dv[r * TS + cc] = x[s];
      }
    } else if (more && warp >= 8 && warp < 10) {
      // tile (k + 1, k) with every panel below k applied, the lower half of (k + 1, k + 1) with those below k too
      if (k >= 1) {
        int ok = 1;
        if (lane == 0) ok = wait_count(warp == 8 ? hsub + k : hdiag + k + 1, 1u, err) ? 1 : 0;
        if (!__shfl_sync(0xffffffffu, ok, 0)) *bad = 1;
      }
      double(*dst)[TS + 1] = warp == 8 ? c.T : c.A;
      const double* src = buf + (int64_t)(r1 + r) * ld + (warp == 8 ? k0 : r1) + h;
#pragma unroll
      for (int q = 0; q < TS / 2; ++q) dst[r][2 * q + h] = __ldcg(src + 2 * q);
    }
    bar_sync(0, MT);
    bar_arrive(6 + 2 * (k & 1), FTH);
    if (tid < TS * TS) buf[(int64_t)(k0 + tid / TS) * ld + k0 + tid % TS] = c.Lt[tid / TS][tid % TS];  // read after the kernel
    if (*bad) {
      if (tid == 0) atomicExch(err, 1);
      return false;
    }
    if (!more) break;
    if (warp < 8) {  // solve L = T inv(L_kk)^T: a column pair per warp (inv(L_kk) is lower), even over the schedulers
      const int pr = warp < 4 ? 7 - warp : warp - 4, cc = 2 * pr + h;
      double o = 0.0;
#pragma unroll
      for (int q = 0; q < TS; ++q)
        if (q < 2 * pr + 2) o = fma(c.T[r][q], c.X[cc][q], o);
      c.Ls[r][cc] = o;
      buf[(int64_t)(r1 + r) * ld + k0 + cc] = o;
    }
    if (warp >= 8) {
      const int u = (warp < 12 ? warp - 8 : warp - 9) * 32 + lane;  // 224 threads
      clear_slots(u);
      if (u < 32) clear_slots(u + 224);
    }
    bar_sync(0, MT);
    bar_arrive(7 + 2 * (k & 1), FTH);
    if (tid < 128) {
      double t = c.A[er][ec];
#pragma unroll
      for (int kk = 0; kk < TS; ++kk) t = fma(-c.Ls[er][kk], c.Ls[ec][kk], t);
      c.D[er][ec] = t;
    }
    if (warp == 4 && lane < 8) tcorner = c.A[15][8 + lane];
    bar_sync(0, MT);
  }
  return true;
}

// A band CTA: rows first, first + step, ... < npan.  Threads 0-127 compute, warp 4 publishes.
__device__ void flow_band(FlowBand& w, double* buf, int64_t ld, int npan, const double* dinv, int first, int step,
                          unsigned* prog, const unsigned* xprog, unsigned* hsub, unsigned* hdiag, int* err) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  volatile unsigned* shared_have = &w.have;
  // barriers 5, 6, 7: the row's three tiles are written (the next row's solve needs the chain to have taken this
  // row's, so the publishing warp is never a row behind)
  if (warp >= 4) {
    if (warp > 4) return;
    for (int i = first; i < npan; i += step) {
      unsigned* const out[3] = {prog + (int64_t)i * CSTR, hsub + i - 1, hdiag + i};
      for (int q = 0; q < 3; ++q) {
        bar_sync(5 + q, 160);
        if (!*shared_have) return;
        if (lane == 0) {
          __threadfence();
          st_rel(out[q], q == 0 ? (unsigned)(i - 1) : 1u);
        }
        __syncwarp();
      }
    }
    return;
  }
  const int r = lane & 15, h = lane >> 4;
  const int c0 = 2 * warp + h, c1 = 2 * (7 - warp) + h;     // this thread's elements: row r, columns c0 and c1
  const int lrow = threadIdx.x >> 3, lc = 2 * (threadIdx.x & 7);
  auto sync = [&] { bar_sync(1, 128); };
  auto give_up = [&] {  // (uniform) the publishing warp leaves too
    bar_arrive(5, 160);
  };
  auto load = [&](int row, int col) {
    return __ldcg(reinterpret_cast<const double2*>(buf + (int64_t)(row * TS + lrow) * ld + col * TS + lc));
  };
  auto stash = [&](double (*dst)[FP], double2 g) { *reinterpret_cast<double2*>(&dst[lrow][lc]) = g; };
  // x0, x1 -= the products of rows r of a and c0, c1 of b
  auto apply = [&](double& x0, double& x1, const double (*a)[FP], const double (*b)[FP]) {
#pragma unroll
    for (int kk = 0; kk < TS; kk += 2) {
      const double2 u = *reinterpret_cast<const double2*>(&a[r][kk]);
      const double2 v0 = *reinterpret_cast<const double2*>(&b[c0][kk]);
      const double2 v1 = *reinterpret_cast<const double2*>(&b[c1][kk]);
      x0 = fma(-u.x, v0.x, x0);
      x1 = fma(-u.x, v1.x, x1);
      x0 = fma(-u.y, v0.y, x0);
      x1 = fma(-u.y, v1.y, x1);
    }
  };
  if (threadIdx.x == 0) *shared_have = 1u;
  for (int i = first; i < npan; i += step) {
    double p0, p1, t0, t1, a0, a1;  // tiles (i, i - 2), (i, i - 1), (i, i)
    const double* row = buf + (int64_t)(i * TS + r) * ld + (i - 2) * TS;
    p0 = __ldcg(row + c0);
    p1 = __ldcg(row + c1);
    t0 = __ldcg(row + TS + c0);
    t1 = __ldcg(row + TS + c1);
    a0 = __ldcg(row + 2 * TS + c0);
    a1 = __ldcg(row + 2 * TS + c1);
    unsigned have = 0;
    for (int k = 0; k + 2 < i; ++k) {
      if (have < (unsigned)(k + 1)) {
        sync();
        if (warp == 0) {
          const unsigned m = wait_rows(prog + (int64_t)i * CSTR, prog + (int64_t)(i - 1) * CSTR, (unsigned)(k + 1), err);
          const unsigned m2 = m ? wait_rows(prog + (int64_t)(i - 2) * CSTR, prog + (int64_t)(i - 2) * CSTR,
                                            (unsigned)(k + 1), err) : 0u;
          if (lane == 0) *shared_have = min(m, m2);
        }
        sync();
        have = *shared_have;
        if (!have) return give_up();
      }
      const double2 gi = load(i, k), g1 = load(i - 1, k), g2 = load(i - 2, k);
      sync();
      stash(w.li, gi);
      stash(w.l1, g1);
      stash(w.l2, g2);
      sync();
      apply(p0, p1, w.li, w.l2);
      apply(t0, t1, w.li, w.l1);
      apply(a0, a1, w.li, w.li);
    }
    // panel i - 2: (i, i - 2) solved against its diagonal tile's inverse ...
    sync();
    w.li[r][c0] = p0;
    w.li[r][c1] = p1;
    if (threadIdx.x == 0) *shared_have = wait_count(xprog, (unsigned)(i - 1), err) ? 1u : 0u;
    sync();
    if (!*shared_have) return give_up();
    stash(w.l2, __ldcg(reinterpret_cast<const double2*>(dinv + (int64_t)(i - 2) * TS * TS + lrow * TS + lc)));
    sync();
    double o0 = 0.0, o1 = 0.0;
#pragma unroll
    for (int kk = 0; kk < TS; ++kk) {
      const double u = w.li[r][kk];
      if (kk < 2 * warp + 2) o0 = fma(u, w.l2[c0][kk], o0);
      if (kk < 16 - 2 * warp) o1 = fma(u, w.l2[c1][kk], o1);
    }
    double* out = buf + (int64_t)(i * TS + r) * ld + (i - 2) * TS;
    out[c0] = o0;
    out[c1] = o1;
    bar_arrive(5, 160);
    sync();
    w.li[r][c0] = o0;
    w.li[r][c1] = o1;
    // ... and applied to (i, i - 1), with the chain's (i - 1, i - 2), and to (i, i)
    if (threadIdx.x == 0)
      *shared_have = wait_count(prog + (int64_t)(i - 1) * CSTR, (unsigned)(i - 1), err) ? 1u : 0u;
    sync();
    if (!*shared_have) {
      bar_arrive(6, 160);
      return;
    }
    stash(w.l1, load(i - 1, i - 2));
    sync();
    apply(t0, t1, w.li, w.l1);
    out[TS + c0] = t0;
    out[TS + c1] = t1;
    bar_arrive(6, 160);
    apply(a0, a1, w.li, w.li);
    out[2 * TS + c0] = a0;
    out[2 * TS + c1] = a1;
    bar_arrive(7, 160);
  }
}

// One matrix of a factorisation, as the bulk sees it.
struct FlowMat {
  double* buf;
  const double* dinv;
  unsigned* cnt;  // zeroed counters: prog (nrt x CSTR), xprog (CSTR), hsub (npan), hdiag (npan)
  int64_t ld;
  int rows, npan, nrt, nid;
};

// A group's tiles t = first, first + step, ... < ntiles; tile(t, m, i, j) gives the matrix and the tile.  HAND: the
// list holds tiles (j + 1, j) and (j, j) too; they get the panels below j and j - 1 and are handed to the chain.
template <bool HAND, class Tile>
__device__ void flow_bulk(FlowBulk& w, int bar, int ntiles, int first, int step, Tile tile, int* err) {
  const int lane = threadIdx.x & 31, gw = (threadIdx.x >> 5) & 3, gt = threadIdx.x & 127;
  const int r = lane & 15, h = lane >> 4;
  const int c0 = 2 * gw + h, c1 = 2 * (7 - gw) + h;  // this thread's elements: row r, columns c0 and c1
  const int lrow = gt >> 3, lc = 2 * (gt & 7);       // its two values of a tile to load or store
  volatile unsigned* shared_have = &w.have;
  auto sync = [&] { bar_sync(bar, 128); };
  for (int t = first; t < ntiles; t += step) {
    FlowMat m;
    int i, j;
    tile(t, m, i, j);
    unsigned* prog = m.cnt;
    unsigned* xprog = m.cnt + (int64_t)m.nrt * CSTR;
    const bool app = i >= m.npan;
    const int ri = flow_row0(i, m.npan, m.ld), rj = j * TS;
    const int k0 = (app && (i - m.npan + 1) * TS <= m.nid) ? i - m.npan : 0;  // identity rows: zero before column i - npan
    const bool handed = HAND && !app && i <= j + 1;
    const int kend = HAND && i == j ? j - 1 : j;
    const bool li = ri + lrow < m.rows;
    double* pi = m.buf + (int64_t)(ri + lrow) * m.ld + lc;
    const double* pj = m.buf + (int64_t)(rj + lrow) * m.ld + lc;
    const double2 zero = make_double2(0.0, 0.0);
    double2 ga = zero, gb = zero;
    auto load = [&](int k) {
      if (li) ga = __ldcg(reinterpret_cast<const double2*>(pi + k * TS));
      gb = __ldcg(reinterpret_cast<const double2*>(pj + k * TS));
    };
    auto stash = [&](double (*dst)[FP], double2 g) { *reinterpret_cast<double2*>(&dst[lrow][lc]) = g; };
    const double2 gc = li ? __ldcg(reinterpret_cast<const double2*>(pi + j * TS)) : zero;
    sync();
    stash(w.a, gc);
    sync();
    double a0 = w.a[r][c0], a1 = w.a[r][c1];
    const unsigned *fi = prog + (int64_t)i * CSTR, *fj = prog + (int64_t)j * CSTR;
    unsigned have = 0;
    bool ahead = false;  // ga / gb hold panel k already
    for (int k = k0; k < kend; ++k) {
      if (!ahead) {
        if (have < (unsigned)(k + 1)) {
          if (gw == 0) {
            const unsigned v = wait_rows(fi, fj, (unsigned)(k + 1), err);
            if (lane == 0) *shared_have = v;
          }
          sync();
          have = *shared_have;
          if (!have) return;
        }
        load(k);
      }
      sync();
      stash(w.a, ga);
      stash(w.b, gb);
      sync();
      ahead = k + 1 < kend && have >= (unsigned)(k + 2);
      if (ahead) load(k + 1);
#pragma unroll
      for (int kk = 0; kk < TS; kk += 2) {
        const double2 a = *reinterpret_cast<const double2*>(&w.a[r][kk]);
        const double2 b0 = *reinterpret_cast<const double2*>(&w.b[c0][kk]);
        const double2 b1 = *reinterpret_cast<const double2*>(&w.b[c1][kk]);
        a0 = fma(-a.x, b0.x, a0);
        a1 = fma(-a.x, b1.x, a1);
        a0 = fma(-a.y, b0.y, a0);
        a1 = fma(-a.y, b1.y, a1);
      }
    }
    if (!handed && gt == 0) *shared_have = wait_count(xprog, (unsigned)(j + 1), err) ? 1u : 0u;
    sync();
    w.a[r][c0] = a0;
    w.a[r][c1] = a1;
    if (!handed) {
      if (!*shared_have) return;
      stash(w.b, __ldcg(reinterpret_cast<const double2*>(m.dinv + (int64_t)j * TS * TS + lrow * TS + lc)));
      sync();
      // out = T inv(L_jj)^T; inv(L_jj) is lower, so columns c <= 2 p + 1 end at k = 2 p + 1
      double o0 = 0.0, o1 = 0.0;
#pragma unroll
      for (int kk = 0; kk < TS; ++kk) {
        const double u = w.a[r][kk];
        if (kk < 2 * gw + 2) o0 = fma(u, w.b[c0][kk], o0);
        if (kk < 16 - 2 * gw) o1 = fma(u, w.b[c1][kk], o1);
      }
      sync();
      w.a[r][c0] = o0;
      w.a[r][c1] = o1;
    }
    sync();
    if (li) *reinterpret_cast<double2*>(pi + j * TS) = *reinterpret_cast<const double2*>(&w.a[lrow][lc]);
    sync();
    if (gt == 0) {
      __threadfence();
      if (!handed)
        st_rel(prog + (int64_t)i * CSTR, (unsigned)(j + 1));
      else
        st_rel(xprog + CSTR + (i == j ? m.npan : 0) + j, 1u);
    }
  }
}

// cnt: zeroed counters: prog (nrt x CSTR), xprog (CSTR), hsub (npan), hdiag (npan).  Block 0 is the chain, then
// nband band CTAs, then the bulk.
__global__ void __launch_bounds__(FTH, 1) k_f64_flow(double* buf, int64_t ld, int rows, int npan, int nrt, int nid,
                                                     double* dinv, int* info, const int2* __restrict__ tiles,
                                                     int ntiles, int nband, unsigned* cnt, int* err) {
  __shared__ FlowSmem sm;
  unsigned* prog = cnt;
  unsigned* xprog = cnt + (int64_t)nrt * CSTR;
  unsigned* hsub = xprog + CSTR;
  unsigned* hdiag = hsub + npan;
  const int g = threadIdx.x >> 7, b = (int)blockIdx.x - 1 - nband, nb = (int)gridDim.x - 1 - nband;
  if (blockIdx.x == 0) {
    if (threadIdx.x == 0) sm.c.bad = 0;
    flow_chain(sm.c, buf, ld, npan, dinv, info, prog, xprog, hsub, hdiag, err);
  } else if (b < 0)
    flow_band(sm.b, buf, ld, npan, dinv, 1 + (int)blockIdx.x, nband, prog, xprog, hsub, hdiag, err);
  else
    flow_bulk<false>(
        sm.g[g], 1 + g, ntiles, g * nb + b, nb * FG,
        [&](int t, FlowMat& m, int& i, int& j) {
          i = tiles[t].x;
          j = tiles[t].y;
          m = FlowMat{buf, dinv, cnt, ld, rows, npan, nrt, nid};
        },
        err);
}

// The same for many matrices at once (the FP64 form's windows): one launch
// factorises `nwin` windows and solves their extra rows.  Block c < nchain is the
// chain of windows c, c + nchain, ...; the other CTAs' groups take the tiles of all
// windows (list: window, i, j; round by round of nchain windows, then column by
// column, see k_f64_tiles), among them (j + 1, j) and (j + 1, j + 1) up
// to the panel that the chain applies itself.  The FP64 pipe bounds it once there are enough windows: a group's warp
// keeps two of its four 64-clock slots a 16-column step busy.  dv16: 16 x 16
// inverse diagonal tiles (npan per window from its dv on), cnt: FlowMat counters.
//
// 16 windows of 250 points with 65 extra rows: 0.21 ms against 17.2 of 64-wide panel
// launches, a window at a time, before; 20 windows of 500 with 201: 1.9 against 63.7.
struct FlowWin {
  int64_t base, dv, cnt;
  int ld, rows, npan, nrt;
};

// The bulk's tile list.  Column j of a window (npan panels, nrt row tiles) has flow_column() tiles: ahead of the others
// what the chain's panel j needs, (j + 1, j) and (j + 1, j + 1), handed over (no wait is for a tile later in the list;
// panel 0 finds it in the original matrix), then (i, j) for i >= j + 2 and the appended rows.
__host__ __device__ inline int flow_handed(int npan, int j) { return j > 0 && j + 1 < npan ? 2 : 0; }
__host__ __device__ inline int flow_first(int npan, int j) { return j + 2 < npan ? j + 2 : npan; }
__host__ __device__ inline int flow_column(int npan, int nrt, int j) {
  return flow_handed(npan, j) + nrt - flow_first(npan, j);
}
// Tiles of columns 0 .. j - 1, j <= npan.
__host__ __device__ inline int64_t flow_columns(int npan, int nrt, int j) {
  const int64_t c = j, handed = j - 1 < npan - 2 ? j - 1 : npan - 2;
  return c * nrt - (c * (c - 1) / 2 + 2 * c - (j == npan ? 1 : 0)) + 2 * (handed > 0 ? handed : 0);
}
// Tiles of window v (described by f) ahead of column j of window w: rounds of nchain windows, then columns, then windows.
__host__ __device__ inline int64_t flow_ahead(const FlowWin& f, int v, int w, int j, int nchain) {
  if (v / nchain != w / nchain) return v < w ? flow_columns(f.npan, f.nrt, f.npan) : 0;
  if (j >= f.npan) return flow_columns(f.npan, f.nrt, f.npan);
  return flow_columns(f.npan, f.nrt, j) + (v < w ? flow_column(f.npan, f.nrt, j) : 0);
}
// Tile q of column j of window w.
__host__ __device__ inline int4 flow_tile(int npan, int w, int j, int q) {
  const int h = flow_handed(npan, j);
  return q < h ? make_int4(w, j + 1, j + q, 0) : make_int4(w, flow_first(npan, j) + q - h, j, 0);
}

// Writes the list: one CTA per window, a warp per column.  Made on the host and uploaded it was 16 bytes of page-locked
// memory a tile (385 KB for a window of 2,000 points with 2,049 extra rows).
__global__ void __launch_bounds__(256) k_f64_tiles(const FlowWin* __restrict__ wins, int nwin, int nchain,
                                                   int4* __restrict__ tiles) {
  grid_dep_wait();
  grid_dep_launch();
  const int w = blockIdx.x, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const FlowWin f = wins[w];
  for (int j = warp; j < f.npan; j += 8) {
    int64_t at = 0;
    for (int v = lane; v < nwin; v += 32) at += flow_ahead(wins[v], v, w, j, nchain);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) at += __shfl_xor_sync(0xffffffffu, at, o);
    for (int q = lane; q < flow_column(f.npan, f.nrt, j); q += 32) tiles[at + q] = flow_tile(f.npan, w, j, q);
  }
}

__global__ void __launch_bounds__(FTH, 1) k_f64_windows(const FlowWin* __restrict__ wins, int nwin, int nchain,
                                                        double* buf, double* dv16, int* info,
                                                        const int4* __restrict__ tiles, int ntiles, unsigned* cnt,
                                                        int* err) {
  __shared__ FlowSmem sm;
  const int g = threadIdx.x >> 7, b = (int)blockIdx.x - nchain, nb = (int)gridDim.x - nchain;
  if (b < 0) {
    if (threadIdx.x == 0) sm.c.bad = 0;
    for (int w = blockIdx.x; w < nwin; w += nchain) {
      const FlowWin f = wins[w];
      unsigned* prog = cnt + f.cnt;
      unsigned* xprog = prog + (int64_t)f.nrt * CSTR;
      // no further window once a wait gave up: a warp still in this one would meet the others at another barrier
      if (!flow_chain(sm.c, buf + f.base, f.ld, f.npan, dv16 + f.dv, info + w, prog, xprog, xprog + CSTR,
                      xprog + CSTR + f.npan, err))
        return;
    }
    return;
  }
  flow_bulk<true>(
      sm.g[g], 1 + g, ntiles, g * nb + b, nb * FG,
      [&](int t, FlowMat& m, int& i, int& j) {
        const int4 it = tiles[t];
        const FlowWin f = wins[it.x];
        i = it.y;
        j = it.z;
        m = FlowMat{buf + f.base, dv16 + f.dv, cnt + f.cnt, f.ld, f.rows, f.npan, f.nrt, 0};
      },
      err);
}

// Forward solve of the FP64 form's prediction right-hand sides by the stored
// factors: CTA (pair, 16 test rows; four warps, one per scheduler) sweeps the
// window's 16-column panels left to right, P_j = (P_j - sum_{k<j} P_k L_jk^T) inv(L_jj)^T,
// with the operations of a row of k_f64_windows in the same order, so that a
// test row has the bits it would have as an extra row of the window.  Bounded by the
// FP64 pipe, 2,048 clocks a tile product; 64-row CTAs left most SMs without one
// (31 pairs of C1: 20.5 ms one pair a launch, 0.20 now).
__global__ void __launch_bounds__(128) k_f64_psweep(const Pair* __restrict__ pairs, const int2* __restrict__ items,
                                                    const Win* __restrict__ wins, const double* __restrict__ buf,
                                                    const double* __restrict__ dv16, double* P) {
  grid_dep_wait();
  grid_dep_launch();
  __shared__ __align__(16) double ta[TS][FP], tb[TS][FP];
  const int2 it = items[blockIdx.x];
  const Pair pr = pairs[it.x];
  const Win w = wins[pr.win];
  const int npan = (w.n + TS - 1) / TS, u0 = it.y * TS;
  const int lane = threadIdx.x & 31, gw = threadIdx.x >> 5;
  const int r = lane & 15, h = lane >> 4, c0 = 2 * gw + h, c1 = 2 * (7 - gw) + h;
  const int lrow = threadIdx.x >> 3, lc = 2 * (threadIdx.x & 7);
  const bool live = u0 + lrow < pr.nu;
  const double2 zero = make_double2(0.0, 0.0);
  double* pi = P + pr.pbase + (int64_t)(u0 + lrow) * w.npad + lc;
  auto stash = [&](double (*dst)[FP], double2 g) { *reinterpret_cast<double2*>(&dst[lrow][lc]) = g; };
  for (int j = 0; j < npan; ++j) {
    const double* pj = buf + w.base + (int64_t)(j * TS + lrow) * w.npad + lc;
    double2 ga = live ? __ldcg(reinterpret_cast<const double2*>(pi + j * TS)) : zero;
    __syncthreads();
    stash(ta, ga);
    __syncthreads();
    double a0 = ta[r][c0], a1 = ta[r][c1];
    double2 gb = zero;
    auto load = [&](int k) {
      ga = live ? __ldcg(reinterpret_cast<const double2*>(pi + k * TS)) : zero;
      gb = *reinterpret_cast<const double2*>(pj + k * TS);
    };
    if (j > 0) load(0);
    for (int k = 0; k < j; ++k) {
      __syncthreads();
      stash(ta, ga);
      stash(tb, gb);
      __syncthreads();
      if (k + 1 < j) load(k + 1);
#pragma unroll
      for (int kk = 0; kk < TS; kk += 2) {
        const double2 a = *reinterpret_cast<const double2*>(&ta[r][kk]);
        const double2 b0 = *reinterpret_cast<const double2*>(&tb[c0][kk]);
        const double2 b1 = *reinterpret_cast<const double2*>(&tb[c1][kk]);
        a0 = fma(-a.x, b0.x, a0);
        a1 = fma(-a.x, b1.x, a1);
        a0 = fma(-a.y, b0.y, a0);
        a1 = fma(-a.y, b1.y, a1);
      }
    }
    __syncthreads();
    ta[r][c0] = a0;
    ta[r][c1] = a1;
    stash(tb, *reinterpret_cast<const double2*>(dv16 + w.dinv / 4 + (int64_t)j * TS * TS + lrow * TS + lc));
    __syncthreads();
    double o0 = 0.0, o1 = 0.0;
#pragma unroll
    for (int kk = 0; kk < TS; ++kk) {
      const double u = ta[r][kk];
      if (kk < 2 * gw + 2) o0 = fma(u, tb[c0][kk], o0);
      if (kk < 16 - 2 * gw) o1 = fma(u, tb[c1][kk], o1);
    }
    __syncthreads();
    ta[r][c0] = o0;
    ta[r][c1] = o1;
    __syncthreads();
    if (live) *reinterpret_cast<double2*>(pi + j * TS) = *reinterpret_cast<const double2*>(&ta[lrow][lc]);
  }
}

// inv(L_kk) of every 64 x 64 diagonal block from its 16 x 16 diagonal tiles' inverses (those past npan are the
// identity): X_ij = -X_ii sum_{j <= k < i} L_ik X_kj, block diagonal by block diagonal.  Grid: x = block, y = window.
__global__ void __launch_bounds__(256) k_f64_dinv64(const Win* __restrict__ wins, const FlowWin* __restrict__ fw,
                                                    const double* __restrict__ buf, const double* __restrict__ dv16,
                                                    double* __restrict__ dinv) {
  grid_dep_wait();
  grid_dep_launch();
  const Win w = wins[blockIdx.y];
  const FlowWin f = fw[blockIdx.y];
  const int kp = blockIdx.x;
  if (kp * TB >= w.npad) return;
  __shared__ double X[4][4][TS][TS + 1], Lt[TS][TS + 1], S[TS][TS + 1];
  const int r = threadIdx.x >> 4, c = threadIdx.x & 15;
  const double* A = buf + w.base + (int64_t)kp * TB * w.npad + kp * TB;
  for (int i = 0; i < 4; ++i) {
    const int t = 4 * kp + i;
    X[i][i][r][c] = t < f.npan ? dv16[f.dv + (int64_t)t * TS * TS + r * TS + c] : (r == c ? 1.0 : 0.0);
    for (int j = i + 1; j < 4; ++j) X[i][j][r][c] = 0.0;
  }
  for (int d = 1; d < 4; ++d)
    for (int j = 0; j + d < 4; ++j) {
      const int i = j + d;
      double acc = 0.0;
      for (int k = j; k < i; ++k) {
        __syncthreads();
        Lt[r][c] = 4 * kp + i < f.npan ? A[(int64_t)(i * TS + r) * w.npad + k * TS + c] : 0.0;
        __syncthreads();
#pragma unroll
        for (int q = 0; q < TS; ++q) acc = fma(Lt[r][q], X[k][j][q][c], acc);
      }
      S[r][c] = acc;
      __syncthreads();
      acc = 0.0;
#pragma unroll
      for (int q = 0; q < TS; ++q) acc = fma(-X[i][i][r][q], S[q][c], acc);
      X[i][j][r][c] = acc;
    }
  __syncthreads();
  double* Dv = dinv + w.dinv + (int64_t)kp * TB * TB;
  for (int e = threadIdx.x; e < TB * TB; e += 256) {
    const int er = e / TB, ec = e % TB;
    Dv[e] = X[er >> 4][ec >> 4][er & 15][ec & 15];
  }
}

}  // namespace f64
}  // namespace lma
