// Prediction on the tensor cores (mixed form): the forward solve of the test
// rows by the stored window factors and the accumulation of h.
//
// Both take the window's matrix (factor rows, or the solved rows X_{1+k}) as the
// 128-row operand and the test rows as the N columns of the product, N = 16, 64 or
// 128 with the number of test rows: with the test rows as the 128-row operand a
// handful of them cost as much as 128.  A test row's result does not depend on the
// arrangement: each element's products enter its accumulator in the same order (P_hi
// L_hi, P_hi L_lo, P_lo L_hi per 8 values of K, K ascending).
#pragma once
#include <type_traits>

#include "lma_tc.cuh"

namespace lma {
namespace tc {

// 12 kind::tf32 MMAs of a 32-wide chunk: D[128 x N] (+)= A B^T with B's halves taken in the order hi, hi, lo.
template <int N>
__device__ __forceinline__ void mma_chunk_ba(uint32_t d, TcStage<N>& S, bool first) {
  const uint32_t idesc = idesc_tf32(128, N);
  const uint32_t ah = smem_addr(S.a_hi), al = smem_addr(S.a_lo), bh = smem_addr(S.b_hi), bl = smem_addr(S.b_lo);
#pragma unroll
  for (int ks = 0; ks < 4; ++ks) {
    const uint32_t o = ks * 32;
    mma_tf32(d, sdesc_sw128(ah + o), sdesc_sw128(bh + o), idesc, (first && ks == 0) ? 0u : 1u);
    mma_tf32(d, sdesc_sw128(al + o), sdesc_sw128(bh + o), idesc, 1u);
    mma_tf32(d, sdesc_sw128(ah + o), sdesc_sw128(bl + o), idesc, 1u);
  }
}

// Bounded wait by lane 0, the result shared with the warp; raises the abort flag on a timeout.
__device__ __forceinline__ bool wait_warp(uint64_t* bar, uint32_t parity, volatile int* abort_flag) {
  int ok = 1;
  if ((threadIdx.x & 31) == 0) ok = mbar_wait(bar, parity) ? 1 : 0;
  ok = __shfl_sync(0xffffffffu, ok, 0);
  if (!ok) *abort_flag = 1;
  return ok != 0 && !*abort_flag;
}

constexpr int kPsProducers = 8;
constexpr int kPsThreads = 32 * (kPsProducers + 1);
constexpr int ps_stages(int n) { return n == 128 ? 3 : 4; }
template <int N>
struct PsSmem {
  TcStage<N> st[ps_stages(N)];
  uint64_t full[4], empty[4], done, rows, fin;
  uint32_t tmem;
  int abort;
};

}  // namespace tc

// Forward solve of one window's test rows (CTA: window rows [N it.y, + N) of pair it.x, which holds every test row
// of the window): the window's columns left to right in groups of two 64-wide panels a, b,
//   D = L[a b, 0:k0] P[:, 0:k0]^T,  P_a = (P_a - D_a) inv(L_aa)^T,  D += L[a b, a] P_a^T,  P_b = (P_b - D_b) inv(L_bb)^T.
// What bounds it: the window's factor is read once, 5 to 8 MB a CTA, and 20 panels follow one another.  Eight
// producer warps keep two or three 32-wide chunks of the factor in flight in registers across panel boundaries, split them
// into TF32 hi/lo and fill a ring of stages; one warp issues the MMAs; the producers also turn the accumulators of a
// panel into the next product's operand (tensor memory lane = factor column = K, so that a warp's stores fill rows).
//
// 64 test points against a C2 model: 0.70 -> 0.31 ms (before: a CTA per pair of test block and window, one chunk
// in flight between CTA barriers); 32,768 against N = 65,536: 1.99 -> 1.52.
template <int N>
__global__ void __launch_bounds__(tc::kPsThreads, 1) k_pred_sweep_tc(const Pair* __restrict__ pairs,
                                                                     const int2* __restrict__ items,
                                                                     const Win* __restrict__ wins,
                                                                     const float* __restrict__ buf,
                                                                     const float* __restrict__ dinv, float* P,
                                                                     int* __restrict__ err) {
  grid_dep_wait();
  grid_dep_launch();
  using namespace tc;
  constexpr int NS = ps_stages(N), NA = 4, NBV = N >= 32 ? N / 32 : 1, PF = N == 16 ? 3 : 2;
  constexpr uint32_t TCOL = 2 * N < 32 ? 32 : 2 * N;
  extern __shared__ __align__(16) unsigned char smraw[];
  PsSmem<N>& sm = *reinterpret_cast<PsSmem<N>*>((reinterpret_cast<uintptr_t>(smraw) + 1023) & ~uintptr_t(1023));
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int2 it = items[blockIdx.x];
  const Pair pr = pairs[it.x];
  const Win w = wins[pr.win];
  const int64_t ld = w.npad;
  const int u0 = it.y * N, nu = min(N, pr.nu - u0), npad = w.npad, ngroups = (npad + 127) / 128;
  const float* L = buf + w.base;
  const float* Dv = dinv + w.dinv;
  float* Pu = P + pr.pbase + (int64_t)u0 * ld;
  if (tid == 0) {
    for (int s = 0; s < NS; ++s) {
      mbar_init(&sm.full[s], kPsProducers);
      mbar_init(&sm.empty[s], 1);
    }
    mbar_init(&sm.done, 1);
    mbar_init(&sm.rows, kPsProducers);
    mbar_init(&sm.fin, 1);
    sm.abort = 0;
    mbar_fence_init();
  }
  if (warp == kPsProducers) tmem_alloc(&sm.tmem, TCOL);
  fence_before_sync();
  __syncthreads();
  fence_after_sync();
  const uint32_t tmem = sm.tmem;
  volatile int* abort_flag = &sm.abort;
  // chunks of group g: 4 g of the factor's columns before it, then per panel the solve (2) and, for a group of two
  // panels, the first panel's columns in between (2)
  auto two = [&](int g) { return npad - 128 * g >= 128; };
  auto count = [&](int g) { return 4 * g + (two(g) ? 6 : 2); };

  if (warp < kPsProducers) {
    const int ar = tid >> 3, ac = (tid & 7) * 4;  // rows ar + 32 j, columns ac .. ac + 3 of a chunk
    const int q = warp & 3, half = warp >> 2;
    // Fetches load unconditionally, from addresses clamped into the window: rows and columns past an end feed only
    // accumulator lanes and columns that nobody reads, and a load under a condition makes the next instructions wait
    // for it (1,200 clocks a chunk).
    float4 ra[PF][NA], rb[PF][NBV];
    auto load_b = [&](int i, float4 (&b)[NBV]) {
#pragma unroll
      for (int j = 0; j < NBV; ++j)
        b[j] = *reinterpret_cast<const float4*>(Pu + min(ar + 32 * j, nu - 1) * ld + 32 * i + ac);
    };
    int pg = 0, pi = 0;  // chunk to fetch next
    auto fetch = [&](float4 (&a)[NA], float4 (&b)[NBV]) {
      const int k0 = 128 * pg, e = pi - 4 * pg, kind = e < 0 ? 0 : e / 2 + 1;
      const bool fac = (kind & 1) == 0;  // a factor chunk, or a piece of the inverted diagonal blocks
      const float* src = fac ? L + (kind == 0 ? 32 * pi : k0 + 32 * (e - 2)) : Dv + 32 * (e & 1);
      const int64_t pitch = fac ? ld : TB;
#pragma unroll
      for (int j = 0; j < NA; ++j)
        a[j] = *reinterpret_cast<const float4*>(src + min(k0 + ar + 32 * j, npad - 1) * pitch + ac);
      // test rows of columns that are final by now (group 1's are loaded when they are used)
      load_b(kind == 0 && pg > 1 ? pi : 0, b);
      const bool wrap = pi + 1 == count(pg);
      if (pg < ngroups - 1 || !wrap) {  // stays at the last chunk
        pi = wrap ? 0 : pi + 1;
        pg += wrap ? 1 : 0;
      }
    };
#pragma unroll
    for (int p = 0; p < PF; ++p) fetch(ra[p], rb[p]);
    int g = 0, i = 0, C = 0, nd = 0, nr = 0;
    auto wait_done = [&]() -> bool {
      const bool ok = wait_warp(&sm.done, nd & 1, abort_flag);
      ++nd;
      fence_after_sync();
      return ok;
    };
    // This lane's factor column k0 + 32 q + lane of test rows [half N/2, + N/2): T = P - D (D: accumulator present)
    // into the stage (the rows of P eight ahead), or the solved row from the second accumulator into P and, with a
    // stage, into that.
    auto stage_t = [&](TcStage<N>& S, int k0, bool have_d) {
      const float* col = Pu + k0 + 32 * q + lane;
      float nx[8];
      auto rows8 = [&](int c0) {
#pragma unroll
        for (int e = 0; e < 8; ++e) nx[e] = col[min(c0 + e, nu - 1) * ld];
      };
      rows8(half * (N / 2));
#pragma unroll 1
      for (int c0 = half * (N / 2); c0 < (half + 1) * (N / 2); c0 += 8) {
        float t[8], d[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) t[e] = nx[e];
        rows8(c0 + 8);
        if (have_d) {
          tmem_ld8(tmem + ((uint32_t)(q * 32) << 16) + c0, d);
#pragma unroll
          for (int e = 0; e < 8; ++e) t[e] -= d[e];
        }
#pragma unroll
        for (int e = 0; e < 8; ++e) store_split1(S.b_hi, S.b_lo, c0 + e, lane, t[e]);
      }
    };
    auto solved = [&](TcStage<N>* S, int k0) {
      float* col = Pu + k0 + 32 * q + lane;
#pragma unroll 1
      for (int c0 = half * (N / 2); c0 < (half + 1) * (N / 2); c0 += 8) {
        float d[8];
        tmem_ld8(tmem + N + ((uint32_t)(q * 32) << 16) + c0, d);
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          if (c0 + e < nu) col[(c0 + e) * ld] = d[e];
          if (S) store_split1(S->b_hi, S->b_lo, c0 + e, lane, d[e]);
        }
      }
    };
    auto step = [&](auto PI) -> bool {
      constexpr int p = decltype(PI)::value;
      if (g >= ngroups) return false;
      const int s = C % NS, k0 = 128 * g;
      const int e = i - 4 * g, kind = e < 0 ? 0 : e / 2 + 1, c = e & 1;
      if (C >= NS && !wait_warp(&sm.empty[s], (C / NS - 1) & 1, abort_flag)) return false;
      TcStage<N>& S = sm.st[s];
      // before the first fetch of the group's columns just solved (PF chunks ahead; in place for group 1): every
      // warp's rows are written
      if (kind == 0 && nr < g && i + PF >= 4 * (g - 1)) {
        if (!wait_warp(&sm.rows, nr & 1, abort_flag)) return false;
        ++nr;
      }
      if (kind > 0 && c == 0 && (kind > 1 || g > 0) && !wait_done()) return false;
      if (kind == 0) {
        if (g == 1) load_b(i, rb[p]);
#pragma unroll
        for (int j = 0; j < NBV; ++j)
          if (ar + 32 * j < N) store_split4(S.b_hi, S.b_lo, ar + 32 * j, ac, rb[p][j]);
      } else if (kind == 1) {
        if (q == c) stage_t(S, k0, g > 0);
      } else if (kind == 2) {
        if (q == c) solved(&S, k0);
      } else {
        if (q == 2 + c) stage_t(S, k0, true);
      }
#pragma unroll
      for (int j = 0; j < NA; ++j) store_split4(S.a_hi, S.a_lo, ar + 32 * j, ac, ra[p][j]);
      fence_async_smem();
      fence_before_sync();
      __syncwarp();
      if (lane == 0) mbar_arrive(&sm.full[s]);
      fetch(ra[p], rb[p]);  // after the arrival, which releases the warp's earlier accesses, loads among them
      ++C;
      if (++i == count(g)) {  // the group's last panel: its rows are final now
        if (!wait_done()) return false;
        if (q >= (two(g) ? 2 : 0) && q < (two(g) ? 4 : 2)) solved(nullptr, k0);
        fence_before_sync();
        __syncwarp();
        if (lane == 0) mbar_arrive(&sm.rows);
        i = 0;
        ++g;
      }
      return true;
    };
    while (step(std::integral_constant<int, 0>{}) && step(std::integral_constant<int, 1>{}) &&
           (PF == 2 || step(std::integral_constant<int, PF - 1>{}))) {
    }
  } else {
    int C = 0;
    for (int g = 0; g < ngroups && !*abort_flag; ++g)
      for (int i = 0; i < count(g); ++i, ++C) {
        const int s = C % NS, e = i - 4 * g, kind = e < 0 ? 0 : e / 2 + 1, c = e & 1;
        if (!wait_warp(&sm.full[s], (C / NS) & 1, abort_flag)) break;
        fence_after_sync();
        if (lane == 0) {
          const bool first = kind == 0 ? i == 0 : (c == 0 && (kind != 2 || g == 0));
          mma_chunk_ba<N>(tmem + ((kind & 1) ? N : 0), sm.st[s], first);
          mma_commit(&sm.empty[s]);
          if (kind == 0 ? e == -1 : c == 1) mma_commit(&sm.done);
        }
        __syncwarp();
      }
    if (lane == 0) mma_commit(&sm.fin);  // arrives once every MMA issued above has completed
    __syncwarp();
  }
  const bool okf = mbar_wait(&sm.fin, 0);
  if ((!okf || *abort_flag) && tid == 0) atomicExch(err, 1);
  fence_before_sync();
  __syncthreads();
  if (warp == kPsProducers) tmem_dealloc(tmem, TCOL);
}

namespace tc {

// 8 producer warps, 1 MMA warp, then the drain warps (a lane quarter x 32 or 16 test rows each).
constexpr int pa_drain(int n) { return n == 16 ? 4 : 8; }
constexpr int pa_threads(int n) { return 32 * (kPsProducers + 1 + pa_drain(n)); }
template <int N>
struct PaSmem {
  TcStage<N> st[4];
  uint64_t full[4], empty[4], pfull[4], pfree[4], fin;
  uint32_t tmem;
  int abort;
};

}  // namespace tc

// One (window, N test rows, 128 support coordinates) item of the h accumulation: which window pair (all test rows of
// the window, those of its own block first), row tile, coordinate tile; own = test rows of the window's own block,
// hrow = the window's first partial row.
struct AccItem {
  int pair, ut, kt, own;
  int64_t hrow;
};

// hw[(hrow + r) s + k] = sum over the kept columns c of P[r][c] X_{1+k}[c]: block columns [nB, n) for every test row,
// then the blanket columns [0, nB) for the rows of the window's own block.  Pairs of 32-wide chunks accumulate in
// tensor memory and are added with TwoSum into (hi, lo), which go to the FP32 partial (k_pred_hsum adds a test
// point's partials in window order).  Persistent, one CTA per SM over the items: producers run two or three chunks ahead in
// registers, across items, the drain warps take a pair's accumulator (one of four) while the next ones fill.
// Bounded by the split stores to shared memory (about 900 clocks a chunk at N = 64).
//
// Before, 16 warps loaded, split and drained with one chunk in flight, a CTA per item: 41 ms at C4 (10 % of DRAM), 0.23
// for 64 points against a C2 model; now 27 and 0.10.
template <int N>
__global__ void __launch_bounds__(tc::pa_threads(N), 1) k_pred_accum_win(const Pair* __restrict__ pairs,
                                                                         const AccItem* __restrict__ items, int nitems,
                                                                         const Win* __restrict__ wins,
                                                                         const float* __restrict__ buf,
                                                                         const float* __restrict__ P, int s,
                                                                         float* __restrict__ hw,
                                                                         int* __restrict__ err) {
  grid_dep_wait();
  grid_dep_launch();
  using namespace tc;
  constexpr int NS = 4, NSLOT = 4, NA = 4, NBV = N >= 32 ? N / 32 : 1, PF = N == 16 ? 3 : 2, ND = pa_drain(N);
  constexpr int NC = N / (ND / 4);  // test rows per drain thread
  constexpr uint32_t TCOL = NSLOT * N;
  extern __shared__ __align__(16) unsigned char smraw[];
  PaSmem<N>& sm = *reinterpret_cast<PaSmem<N>*>((reinterpret_cast<uintptr_t>(smraw) + 1023) & ~uintptr_t(1023));
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (tid == 0) {
    for (int k = 0; k < 4; ++k) {
      mbar_init(&sm.full[k], kPsProducers);
      mbar_init(&sm.empty[k], 1);
      mbar_init(&sm.pfull[k], 1);
      mbar_init(&sm.pfree[k], ND);
    }
    mbar_init(&sm.fin, 1);
    sm.abort = 0;
    mbar_fence_init();
  }
  if (warp == kPsProducers) tmem_alloc(&sm.tmem, TCOL);
  fence_before_sync();
  __syncthreads();
  fence_after_sync();
  const uint32_t tmem = sm.tmem;
  volatile int* abort_flag = &sm.abort;
  // chunks of an item: first the block columns from nB rounded down to 4 on, then the blanket's
  auto chunks = [&](const AccItem& it, const Win& w, int& n1, int& n2) {
    n1 = (w.n - (w.nB & ~3) + 31) / 32;
    n2 = it.ut * N < it.own ? (w.nB + 31) / 32 : 0;
  };

  if (warp < kPsProducers) {
    const int ar = tid >> 3, ac = (tid & 7) * 4;
    const float4 z4 = make_float4(0.f, 0.f, 0.f, 0.f);
    float4 ra[PF][NA], rb[PF][NBV];
    // the item being fetched
    int item = blockIdx.x, pc = 0, n1 = 0, n2 = 0, ld = 0, nB = 0, n = 0, rows = 0, own = 0, klim = 0;
    const float *E = nullptr, *Pr = nullptr;
    auto open = [&] {
      const AccItem it = items[item];
      const Pair pr = pairs[it.pair];
      const Win w = wins[pr.win];
      chunks(it, w, n1, n2);
      ld = w.npad;
      nB = w.nB;
      n = w.n;
      rows = min(N, pr.nu - it.ut * N);
      own = min(N, it.own - it.ut * N);
      klim = s - it.kt * 128;
      E = buf + w.base + (int64_t)(w.npad + 1 + it.kt * 128) * w.npad;
      Pr = P + pr.pbase + (int64_t)it.ut * N * w.npad;
    };
    // Fetches load unconditionally, from addresses clamped into the window; values outside [kbeg, kend) and test rows
    // past `lim` are masked when they are stored (a mask or a condition at the load waits for each load in turn: 6,500
    // clocks a chunk).
    int mk[PF], mb[PF], me[PF], ml[PF];
    auto masked = [&](float4 v, int kk, int kbeg, int kend) -> float4 {
      if (kk < kbeg || kk + 4 > kend) {
        v.x = (kk >= kbeg && kk < kend) ? v.x : 0.f;
        v.y = (kk + 1 >= kbeg && kk + 1 < kend) ? v.y : 0.f;
        v.z = (kk + 2 >= kbeg && kk + 2 < kend) ? v.z : 0.f;
        v.w = (kk + 3 >= kbeg && kk + 3 < kend) ? v.w : 0.f;
      }
      return v;
    };
    auto fetch = [&](float4 (&a)[NA], float4 (&b)[NBV], int& kk, int& kbeg, int& kend, int& lim) {
      const bool blk = pc < n1;
      lim = blk ? rows : own;
      kbeg = blk ? nB : 0;
      kend = blk ? n : nB;
      kk = blk ? (nB & ~3) + 32 * pc + ac : 32 * (pc - n1) + ac;
      const int kc = min(kk, ld - 4);
#pragma unroll
      for (int j = 0; j < NA; ++j)
        a[j] = *reinterpret_cast<const float4*>(E + (int64_t)min(ar + 32 * j, klim - 1) * ld + kc);
#pragma unroll
      for (int j = 0; j < NBV; ++j)
        b[j] = *reinterpret_cast<const float4*>(Pr + (int64_t)min(ar + 32 * j, rows - 1) * ld + kc);
      if (++pc == n1 + n2) {
        pc = 0;
        if (item + (int)gridDim.x < nitems) {  // stays at the last item
          item += gridDim.x;
          open();
        }
      }
    };
    // chunks of this CTA in all
    int total = 0;
    for (int t = blockIdx.x; t < nitems; t += gridDim.x) {
      const AccItem it = items[t];
      int a, b;
      chunks(it, wins[pairs[it.pair].win], a, b);
      total += a + b;
    }
    open();
#pragma unroll
    for (int p = 0; p < PF; ++p) fetch(ra[p], rb[p], mk[p], mb[p], me[p], ml[p]);
    int C = 0;
    auto step = [&](auto PI) -> bool {
      constexpr int p = decltype(PI)::value;
      if (C >= total) return false;
      const int st = C % NS;
      if (C >= NS && !wait_warp(&sm.empty[st], (C / NS - 1) & 1, abort_flag)) return false;
      TcStage<N>& S = sm.st[st];
#pragma unroll
      for (int j = 0; j < NA; ++j)
        store_split4(S.a_hi, S.a_lo, ar + 32 * j, ac, masked(ra[p][j], mk[p], mb[p], me[p]));
#pragma unroll
      for (int j = 0; j < NBV; ++j)
        if (ar + 32 * j < N)
          store_split4(S.b_hi, S.b_lo, ar + 32 * j, ac,
                       ar + 32 * j < ml[p] ? masked(rb[p][j], mk[p], mb[p], me[p]) : z4);
      fence_async_smem();
      __syncwarp();
      if (lane == 0) mbar_arrive(&sm.full[st]);
      fetch(ra[p], rb[p], mk[p], mb[p], me[p], ml[p]);
      ++C;
      return true;
    };
    while (step(std::integral_constant<int, 0>{}) && step(std::integral_constant<int, 1>{}) &&
           (PF == 2 || step(std::integral_constant<int, PF - 1>{}))) {
    }
  } else if (warp == kPsProducers) {
    int C = 0, G = 0;  // chunks, pairs issued
    for (int t = blockIdx.x; t < nitems && !*abort_flag; t += gridDim.x) {
      const AccItem it = items[t];
      int n1, n2;
      chunks(it, wins[pairs[it.pair].win], n1, n2);
      for (int c = 0; c < n1 + n2; ++c, ++C) {
        const int e = c < n1 ? c : c - n1, ne = c < n1 ? n1 : n2, slot = G % NSLOT, st = C % NS;
        if ((e & 1) == 0 && G >= NSLOT && !wait_warp(&sm.pfree[slot], (G / NSLOT - 1) & 1, abort_flag)) break;
        if (!wait_warp(&sm.full[st], (C / NS) & 1, abort_flag)) break;
        fence_after_sync();
        if (lane == 0) {
          mma_chunk_ba<N>(tmem + N * slot, sm.st[st], (e & 1) == 0);
          mma_commit(&sm.empty[st]);
          if ((e & 1) == 1 || e == ne - 1) mma_commit(&sm.pfull[slot]);
        }
        __syncwarp();
        if ((e & 1) == 1 || e == ne - 1) ++G;
      }
    }
    if (lane == 0) mma_commit(&sm.fin);  // arrives once every MMA issued above has completed
    __syncwarp();
  } else {
    const int q = warp & 3, part = (warp - kPsProducers - 1) >> 2;
    const uint32_t tl = tmem + ((uint32_t)(q * 32) << 16) + part * NC;
    int G = 0;
    for (int t = blockIdx.x; t < nitems && !*abort_flag; t += gridDim.x) {
      const AccItem it = items[t];
      const Pair pr = pairs[it.pair];
      int n1, n2;
      chunks(it, wins[pr.win], n1, n2);
      float hi[NC], lo[NC];
#pragma unroll
      for (int j = 0; j < NC; ++j) hi[j] = lo[j] = 0.f;
      const int np = (n1 + 1) / 2 + (n2 + 1) / 2;
      bool ok = true;
      for (int k = 0; k < np; ++k, ++G) {
        const int slot = G % NSLOT;
        if (!wait_warp(&sm.pfull[slot], (G / NSLOT) & 1, abort_flag)) {
          ok = false;
          break;
        }
        fence_after_sync();
#pragma unroll
        for (int c0 = 0; c0 < NC; c0 += 8) {
          float v[8];
          tmem_ld8(tl + N * slot + c0, v);
#pragma unroll
          for (int j = 0; j < 8; ++j) two_sum(hi[c0 + j], lo[c0 + j], v[j]);
        }
        fence_before_sync();
        __syncwarp();
        if (lane == 0) mbar_arrive(&sm.pfree[slot]);
      }
      if (!ok) break;
      const int k = it.kt * 128 + q * 32 + lane, r0 = it.ut * N + part * NC;
      if (k < s) {
        float* dst = hw + (it.hrow + r0) * (int64_t)s + k;
#pragma unroll
        for (int j = 0; j < NC; ++j)
          if (r0 + j < pr.nu) dst[(int64_t)j * s] = hi[j] + lo[j];
      }
    }
  }
  const bool okf = mbar_wait(&sm.fin, 0);
  if ((!okf || *abort_flag) && tid == 0) atomicExch(err, 1);
  fence_before_sync();
  __syncthreads();
  if (warp == kPsProducers) tmem_dealloc(tmem, TCOL);
}

}  // namespace lma
