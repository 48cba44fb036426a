// Kernels of the hand-written adjoint of the LMA log-likelihood.
//
// Forward (whitened support coordinates, Vt = Sigma_DS L_SS^-T, C = I + A):
//   loglik = -1/2 (quad - y^T C^-1 y) - 1/2 (sum_m log|R_W| - log|R_B| + log|C|) - N/2 log 2 pi
// with, per window W = D_m u D^B_m and blanket B = D^B_m (Lemma 1):
//   quad, y, A = sum_m  Y_W^T R_W^-1 Y_W - Y_B^T R_B^-1 Y_B,   Y = [r | Vt].
// Reverse sweep, beta = C^-1 y, e = r - Vt beta, Lc = chol(C),
// Y-hat = [e | Vt Lc^-T], Phi_X = R_X^-1 Y-hat_X:
//   G_m   = 1/2 [Phi_W Phi_W^T - pad(Phi_B Phi_B^T) - (R_W^-1 - pad R_B^-1)]
//   Vt-bar += (Phi_W - pad Phi_B)[:,0] beta^T - (Phi_W - pad Phi_B)[:,1:] Lc^-1 - 2 G_m Vt_W
//   theta-bar += <G_m, dK_W/dtheta> + 2 sigma_n^2 tr G_m
// then K_DS-bar = Vt-bar L_SS^-1, L_SS-bar = -L_SS^-T Vt-bar^T Vt and the
// Cholesky adjoint back to Sigma_SS.  With the window factor L (blanket first,
// R_W = L L^T) every R^-1 product is a backward solve with L:
//   Phi_W = L^-T [L^-1 Y-hat],  pad Phi_B = L^-T [L^-1 Y-hat with block rows zeroed],
//   R_W^-1 - pad R_B^-1 = T T^T with T = L^-T [0; I_b].
#pragma once
#include "lma_kernels.cuh"

namespace lma {

// Backward right-hand sides of window w, stored as rows (length npad):
//   [0, s]        L^-1 Y-hat   (row 0 = L^-1 e, rows 1+i = (L^-1 Vt Lc^-T)[:, i])
//   [s+1, 2s+1]   the same with the block-part columns [nB, n) zeroed
//   [2s+2, ...)   unit rows e_{nB+t}, t < b
struct GWin {
  int64_t q;    // element offset of the RHS rows
  int64_t g;    // element offset of this window's G (npad x npad)
  int64_t gv;   // element offset of G^T-product rows (s x npad)
  int nrows;    // 2(s+1) + b
  int pad_;
};

// One past the last column that right-hand-side rows [lo, hi] of a window (see GWin) reach: the zeroed copies end
// at the blanket, unit row t at column nB + t, and a backward solve fills columns to the left only.
__device__ __forceinline__ int rhs_columns(const Win& w, int s, int lo, int hi) {
  if (lo <= s) return w.n;
  if (hi <= 2 * s + 1) return w.nB;
  return w.nB + (hi - (2 * s + 2)) + 1;
}

// rows 1+i and s+2+i: sum_{k<=i} Lc^-1[i][k] X_{1+k}[c]  (LcT[k][i] = Lc^-1[i][k])
template <typename T>
__global__ void __launch_bounds__(NT) k_grad_rhs(const Win* __restrict__ wins, const GWin* __restrict__ gw,
                                                 const T* __restrict__ buf, const T* __restrict__ LcT, int s,
                                                 T* __restrict__ Q) {
  grid_dep_wait();
  grid_dep_launch();
  const Win w = wins[blockIdx.z];
  const GWin g = gw[blockIdx.z];
  const int c0 = blockIdx.x * TB, i0 = blockIdx.y * TB;
  if (c0 >= w.npad || i0 >= s) return;
  __shared__ GemmSmem<T> sm;
  const T* X = buf + w.base + (int64_t)w.npad * w.npad;  // extra rows of the forward sweep
  const int64_t ld = w.npad;
  const int K = min(s, i0 + TB);
  T acc[4][4] = {};
  auto fa = [&](int r, int k) -> T { return (i0 + r < s) ? LcT[(int64_t)k * s + i0 + r] : T(0); };
  auto fb = [&](int r, int k) -> T { return X[(int64_t)(1 + k) * ld + c0 + r]; };
  tile_mma<T, false, false>(acc, K, sm, fa, fb);
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  T* Qw = Q + g.q;
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      int i = i0 + ty + 16 * a, c = c0 + tx + 16 * b;
      if (i >= s) continue;
      T v = (c < w.n) ? acc[a][b] : T(0);
      Qw[(int64_t)(1 + i) * ld + c] = v;
      Qw[(int64_t)(s + 2 + i) * ld + c] = (c >= w.nB) ? T(0) : v;
    }
}

// rows 0, s+1 (from L^-1 e) and the unit rows
template <typename T>
__global__ void k_grad_rhs_fill(const Win* __restrict__ wins, const GWin* __restrict__ gw,
                                const T* __restrict__ ew, int s, T* __restrict__ Q) {
  grid_dep_wait();
  grid_dep_launch();
  const Win w = wins[blockIdx.y];
  const GWin g = gw[blockIdx.y];
  T* Qw = Q + g.q;
  const int ld = w.npad;
  const int b = w.n - w.nB;
  const int64_t total = (int64_t)(2 + b) * ld;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
    int r = (int)(e / ld), c = (int)(e % ld);
    if (r == 0) {
      Qw[c] = (c < w.n) ? ew[w.ew + c] : T(0);
    } else if (r == 1) {
      Qw[(int64_t)(s + 1) * ld + c] = (c < w.nB) ? ew[w.ew + c] : T(0);
    } else {
      int t = r - 2;
      Qw[(int64_t)(2 * s + 2 + t) * ld + c] = (c == w.nB + t) ? T(1) : T(0);
    }
  }
}

// Backward sweep: each RHS row q becomes x with x L = q (x = (L^-T q^T)^T),
// column panels from the last to the first (items: x = window, y = row tile).
template <typename T>
__global__ void __launch_bounds__(NT) k_bwd_sweep(const int2* __restrict__ items, const Win* __restrict__ wins,
                                                  const GWin* __restrict__ gw, const T* __restrict__ buf,
                                                  const T* __restrict__ dinv, int s, T* __restrict__ Q) {
  grid_dep_wait();
  grid_dep_launch();
  const int2 it = items[blockIdx.x];
  const Win w = wins[it.x];
  const GWin g = gw[it.x];
  const int u0 = it.y * TB;
  extern __shared__ __align__(16) unsigned char smraw[];
  CholSmem<T>& sm = *reinterpret_cast<CholSmem<T>*>(smraw);
  const T* L = buf + w.base;
  const int64_t ld = w.npad;
  T* Qw = Q + g.q;
  const int nr = g.nrows;
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  const int npan = (rhs_columns(w, s, u0, min(u0 + TB, nr) - 1) + TB - 1) / TB;  // zero to the right of these
  for (int kp = npan - 1; kp >= 0; --kp) {
    const int k0 = kp * TB;
    const int t0 = k0 + TB;
    T acc[4][4] = {};
    auto fa = [&](int r, int k) -> T { return (u0 + r < nr) ? Qw[(int64_t)(u0 + r) * ld + t0 + k] : T(0); };
    auto fb = [&](int r, int k) -> T { return L[(int64_t)(t0 + k) * ld + k0 + r]; };
    tile_mma<T, true, false>(acc, npan * TB - t0, sm.g, fa, fb);
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
      for (int b = 0; b < 4; ++b) {
        int r = ty + 16 * a, c = tx + 16 * b;
        sm.D[r][c] = (u0 + r < nr) ? Qw[(int64_t)(u0 + r) * ld + k0 + c] - acc[a][b] : T(0);
      }
    const T* Dv = dinv + w.dinv + (int64_t)kp * TB * TB;
    for (int q = threadIdx.x; q < TB * TB; q += NT) sm.X[q / TB][q % TB] = Dv[q];
    __syncthreads();
    T o[4][4] = {};
    for (int j = 0; j < TB; ++j) {
      T a4[4], b4[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        a4[q] = sm.D[ty + 16 * q][j];
        b4[q] = sm.X[j][tx + 16 * q];
      }
#pragma unroll
      for (int p = 0; p < 4; ++p)
#pragma unroll
        for (int q = 0; q < 4; ++q) o[p][q] = fma(a4[p], b4[q], o[p][q]);
    }
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
      for (int b = 0; b < 4; ++b) {
        int r = ty + 16 * a;
        if (u0 + r < nr) Qw[(int64_t)(u0 + r) * ld + k0 + tx + 16 * b] = o[a][b];
      }
    __syncthreads();
  }
}

// G_m tiles (lower, items: x = window, y = tile index) with the covariance
// derivative contraction fused in.  partial[blockIdx.x][0..d-1] log-length-scale
// terms, [d] log sigma_s, [d+1] log sigma_n.
template <typename T>
__global__ void __launch_bounds__(NT) k_grad_G(const int2* __restrict__ items, const Win* __restrict__ wins,
                                               const GWin* __restrict__ gw, const T* __restrict__ Q,
                                               const T* __restrict__ xs, int d, int s, double ss2, double sn2,
                                               T* __restrict__ Gbuf, double* __restrict__ partial) {
  grid_dep_wait();
  grid_dep_launch();
  const int2 it = items[blockIdx.x];
  const Win w = wins[it.x];
  const GWin g = gw[it.x];
  int I, J;
  tri_index(it.y, I, J);
  const int r0 = I * TB, c0 = J * TB;
  __shared__ GemmSmem<T> sm;
  __shared__ T xr[TB][MAXD + 1];
  __shared__ T xc[TB][MAXD + 1];
  __shared__ double red[NT];
  for (int e = threadIdx.x; e < TB * d; e += NT) {
    int r = e / d, q = e % d;
    xr[r][q] = (r0 + r < w.n) ? xs[(w.g_end - 1 - (r0 + r)) * d + q] : T(0);
    xc[r][q] = (c0 + r < w.n) ? xs[(w.g_end - 1 - (c0 + r)) * d + q] : T(0);
  }
  const T* Qw = Q + g.q;
  const int64_t ld = w.npad;
  const int b = w.n - w.nB;
  T acc[4][4] = {};
  {
    auto fa = [&](int r, int k) -> T { return Qw[(int64_t)k * ld + r0 + r]; };
    auto fb = [&](int r, int k) -> T { return Qw[(int64_t)k * ld + c0 + r]; };
    tile_mma<T, false, false>(acc, s + 1, sm, fa, fb);
  }
  if (r0 < w.nB) {  // the zeroed copies have no columns past the blanket
    const T* P = Qw + (int64_t)(s + 1) * ld;
    auto fa = [&](int r, int k) -> T { return P[(int64_t)k * ld + r0 + r]; };
    auto fb = [&](int r, int k) -> T { return -P[(int64_t)k * ld + c0 + r]; };
    tile_mma<T, false, false>(acc, s + 1, sm, fa, fb);
  }
  const int t0 = max(0, r0 - w.nB) / KS * KS;  // unit rows before it end left of this tile's rows
  if (t0 < b) {
    const T* P = Qw + (int64_t)(2 * s + 2 + t0) * ld;
    auto fa = [&](int r, int k) -> T { return P[(int64_t)k * ld + r0 + r]; };
    auto fb = [&](int r, int k) -> T { return -P[(int64_t)k * ld + c0 + r]; };
    tile_mma<T, false, false>(acc, b - t0, sm, fa, fb);
  }
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  const double wgt = (I == J) ? 1.0 : 2.0;
  double gl[MAXD];
  for (int q = 0; q < d; ++q) gl[q] = 0.0;
  double gsig = 0.0, gnoise = 0.0;
  T* G = Gbuf + g.g;
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int bb = 0; bb < 4; ++bb) {
      int r = ty + 16 * a, c = tx + 16 * bb;
      int gi = r0 + r, gj = c0 + c;
      T v = T(0.5) * acc[a][bb];
      if (gi < w.n && gj < w.n) {
        double d2 = 0.0;
        for (int q = 0; q < d; ++q) {
          double t = (double)xr[r][q] - (double)xc[c][q];
          d2 += t * t;
        }
        double kg = (double)v * ss2 * exp(-0.5 * d2) * wgt;
        for (int q = 0; q < d; ++q) {
          double t = (double)xr[r][q] - (double)xc[c][q];
          gl[q] += kg * t * t;
        }
        gsig += 2.0 * kg;
        if (gi == gj) gnoise += 2.0 * sn2 * (double)v;
      } else {
        v = T(0);
      }
      G[(int64_t)gi * ld + gj] = v;
      if (I != J) G[(int64_t)gj * ld + gi] = v;
    }
  // block reduction of d+2 values
  double* P = partial + (int64_t)blockIdx.x * (d + 2);
  for (int q = 0; q < d + 2; ++q) {
    double v = (q < d) ? gl[q] : (q == d ? gsig : gnoise);
    red[threadIdx.x] = v;
    __syncthreads();
    for (int o = NT / 2; o > 0; o >>= 1) {
      if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
      __syncthreads();
    }
    if (threadIdx.x == 0) P[q] = red[0];
    __syncthreads();
  }
}

// GVt_w[k][i] = sum_j Vt[g(j)][k] G[j][i]   (grid: npad tiles, s tiles, windows)
template <typename T>
__global__ void __launch_bounds__(NT) k_grad_gv(const Win* __restrict__ wins, const GWin* __restrict__ gw,
                                                const T* __restrict__ Gbuf, const T* __restrict__ Vt, int s,
                                                T* __restrict__ GV) {
  grid_dep_wait();
  grid_dep_launch();
  const Win w = wins[blockIdx.z];
  const GWin g = gw[blockIdx.z];
  const int c0 = blockIdx.x * TB, k0 = blockIdx.y * TB;
  if (c0 >= w.npad || k0 >= s) return;
  __shared__ GemmSmem<T> sm;
  const T* G = Gbuf + g.g;
  const int64_t ld = w.npad;
  T acc[4][4] = {};
  auto fa = [&](int r, int j) -> T { return (k0 + r < s && j < w.n) ? Vt[(w.g_end - 1 - j) * s + k0 + r] : T(0); };
  auto fb = [&](int r, int j) -> T { return G[(int64_t)j * ld + c0 + r]; };
  tile_mma<T, false, false>(acc, w.n, sm, fa, fb);
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  T* O = GV + g.gv;
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      int k = k0 + ty + 16 * a, c = c0 + tx + 16 * b;
      if (k < s) O[(int64_t)k * ld + c] = acc[a][b];
    }
}

// Gather the per-window contributions onto training rows (fixed window order):
//   PsiT[k][p] = sum_{m: p in W_m} (Phi_W - pad Phi_B)[k][i_m(p)]     k in [0, s]
//   GVT[k][p]  = sum_{m: p in W_m} GVt_m[k][i_m(p)]                   k in [0, s)
// over the windows of the gradient only: window of block m is wins[m - w0],
// taken when m - w0 is in [k_lo, k_hi), its backward layout gw[m - w0 - k_lo].
// (grid: x over rows p, y over k in [0, 2s+1))
template <typename T>
__global__ void k_grad_gather(const Win* __restrict__ wins, const GWin* __restrict__ gw,
                              const int64_t* __restrict__ bptr, int M, int B, int64_t n, int s,
                              const T* __restrict__ Q, const T* __restrict__ GV, T* __restrict__ PsiT,
                              T* __restrict__ GVT, int w0, int k_lo, int k_hi) {
  grid_dep_wait();
  grid_dep_launch();
  const int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int k = blockIdx.y;
  if (p >= n) return;
  int lo = 0, hi = M;  // block of row p: bptr[j] <= p < bptr[j+1]
  while (hi - lo > 1) {
    int mid = (lo + hi) >> 1;
    if (bptr[mid] <= p) lo = mid;
    else hi = mid;
  }
  const int j = lo;
  double acc = 0.0;
  for (int m = max(0, j - B); m <= j; ++m) {
    const int wi = m - w0;  // window index in the model
    if (wi < k_lo || wi >= k_hi) continue;
    const Win w = wins[wi];
    const GWin g = gw[wi - k_lo];
    const int i = (int)(w.g_end - 1 - p);
    if (k <= s) {
      const T* Qw = Q + g.q;
      acc += (double)Qw[(int64_t)k * w.npad + i] - (double)Qw[(int64_t)(s + 1 + k) * w.npad + i];
    } else {
      acc += (double)GV[g.gv + (int64_t)(k - s - 1) * w.npad + i];
    }
  }
  if (k <= s) PsiT[(int64_t)k * n + p] = (T)acc;
  else GVT[(int64_t)(k - s - 1) * n + p] = (T)acc;
}

// VbT[k][p] = beta_k Psi_e[p] - sum_{j>=k} Lc^-1[j][k] Psi_{1+j}[p] - 2 GVT[k][p]
template <typename T>
__global__ void __launch_bounds__(NT) k_grad_vbar(const T* __restrict__ PsiT, const T* __restrict__ GVT,
                                                  const T* __restrict__ LcT, const double* __restrict__ beta,
                                                  int64_t n, int s, T* __restrict__ VbT) {
  grid_dep_wait();
  grid_dep_launch();
  __shared__ GemmSmem<T> sm;
  const int k0 = blockIdx.y * TB;
  const int64_t p0 = (int64_t)blockIdx.x * TB;
  const int K = s - k0;
  T acc[4][4] = {};
  auto fa = [&](int r, int jj) -> T { return (k0 + r < s) ? LcT[(int64_t)(k0 + r) * s + k0 + jj] : T(0); };
  auto fb = [&](int r, int jj) -> T { return (p0 + r < n) ? PsiT[(int64_t)(1 + k0 + jj) * n + p0 + r] : T(0); };
  tile_mma<T, true, false>(acc, K, sm, fa, fb);
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      int k = k0 + ty + 16 * a;
      int64_t p = p0 + tx + 16 * b;
      if (k < s && p < n)
        VbT[(int64_t)k * n + p] = (T)(beta[k] * (double)PsiT[p]) - acc[a][b] - T(2) * GVT[(int64_t)k * n + p];
    }
}

// K_DS-bar^T[k][p] = sum_{i>=k} (L_SS^-1)[i][k] VbT[i][p]  (ET[k][i] = L_SS^-1[i][k]),
// contracted on the fly with dK_DS/dtheta (no storage).
template <typename T>
__global__ void __launch_bounds__(NT) k_grad_kds(const T* __restrict__ VbT, const T* __restrict__ ET,
                                                 const T* __restrict__ xs, const T* __restrict__ ss, int d,
                                                 int64_t n, int s, double ss2, double* __restrict__ partial) {
  grid_dep_wait();
  grid_dep_launch();
  __shared__ GemmSmem<T> sm;
  __shared__ T xp[TB][MAXD + 1];
  __shared__ T xk[TB][MAXD + 1];
  __shared__ double red[NT];
  const int k0 = blockIdx.y * TB;
  const int64_t p0 = (int64_t)blockIdx.x * TB;
  for (int e = threadIdx.x; e < TB * d; e += NT) {
    int r = e / d, q = e % d;
    xk[r][q] = (k0 + r < s) ? ss[(int64_t)(k0 + r) * d + q] : T(0);
    xp[r][q] = (p0 + r < n) ? xs[(p0 + r) * d + q] : T(0);
  }
  const int K = s - k0;
  T acc[4][4] = {};
  auto fa = [&](int r, int ii) -> T { return (k0 + r < s) ? ET[(int64_t)(k0 + r) * s + k0 + ii] : T(0); };
  auto fb = [&](int r, int ii) -> T { return (p0 + r < n) ? VbT[(int64_t)(k0 + ii) * n + p0 + r] : T(0); };
  tile_mma<T, true, false>(acc, K, sm, fa, fb);
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  double gl[MAXD];
  for (int q = 0; q < d; ++q) gl[q] = 0.0;
  double gsig = 0.0;
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      int kr = ty + 16 * a, pc = tx + 16 * b;
      if (k0 + kr < s && p0 + pc < n) {
        double d2 = 0.0;
        for (int q = 0; q < d; ++q) {
          double t = (double)xk[kr][q] - (double)xp[pc][q];
          d2 += t * t;
        }
        double kg = (double)acc[a][b] * ss2 * exp(-0.5 * d2);
        for (int q = 0; q < d; ++q) {
          double t = (double)xk[kr][q] - (double)xp[pc][q];
          gl[q] += kg * t * t;
        }
        gsig += 2.0 * kg;
      }
    }
  double* P = partial + ((int64_t)blockIdx.y * gridDim.x + blockIdx.x) * (d + 2);
  for (int q = 0; q < d + 1; ++q) {
    red[threadIdx.x] = (q < d) ? gl[q] : gsig;
    __syncthreads();
    for (int o = NT / 2; o > 0; o >>= 1) {
      if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
      __syncthreads();
    }
    if (threadIdx.x == 0) P[q] = red[0];
    __syncthreads();
  }
  if (threadIdx.x == 0) P[d + 1] = 0.0;
}

// Rows [q0, q0 + K) of the pieces that the sum over points of M1 is cut into: `nch` chunks of `chunk` rows, each
// in pieces of `len` rows (the last ones shorter).
struct Pieces {
  int64_t n, chunk, len;
  int per;  // pieces per chunk
  __device__ __forceinline__ int get(int piece, int64_t& q0) const {
    const int64_t pb = (piece / per) * chunk;
    q0 = pb + (piece % per) * len;
    const int64_t e = min(min(n, pb + chunk), q0 + len);
    return e > q0 ? (int)(e - q0) : 0;
  }
};

// M1 = Vt-bar^T Vt (s x s): each piece is summed in T, the pieces of slice z = blockIdx.z in FP64 into its partial.
template <typename T>
__global__ void __launch_bounds__(NT) k_grad_m1(const T* __restrict__ VbT, const T* __restrict__ Vt, int64_t n,
                                                int s, Pieces pc, int npieces, int per_slice,
                                                double* __restrict__ partial) {
  grid_dep_wait();
  grid_dep_launch();
  __shared__ GemmSmem<T> sm;
  const int i0 = blockIdx.y * TB, j0 = blockIdx.x * TB;
  double accd[4][4] = {};
  for (int p = blockIdx.z * per_slice; p < min(npieces, (int)(blockIdx.z + 1) * per_slice); ++p) {
    int64_t q0;
    const int K = pc.get(p, q0);
    T acc[4][4] = {};
    auto fa = [&](int r, int k) -> T { return (i0 + r < s) ? VbT[(int64_t)(i0 + r) * n + q0 + k] : T(0); };
    auto fb = [&](int r, int k) -> T { return (j0 + r < s) ? Vt[(q0 + k) * s + j0 + r] : T(0); };
    tile_mma<T, true, false>(acc, K, sm, fa, fb);
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
      for (int b = 0; b < 4; ++b) accd[a][b] += (double)acc[a][b];
  }
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  double* P = partial + (int64_t)blockIdx.z * s * s;
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      int i = i0 + ty + 16 * a, j = j0 + tx + 16 * b;
      if (i < s && j < s) P[(int64_t)i * s + j] = accd[a][b];
    }
}

// ---------------------------------------------------------------------------
// FP32 forms of the N x s products with 128 x 128 tiles and 8 x 8 values a thread
// (the 64 x 64 tiles above read shared memory for every second FMA: 11-15 TFLOP/s at
// N = 65,536, s = 1,024, M1 12.3 ms and Vt-bar 4.6; these 33-37, 3.7 and 2.1 ms).
// One FMA per term, k ascending, as there.

constexpr int GK = 8;  // K step
struct Smem128 {
  float a[2][GK][132], b[2][GK][132];
};

// Four consecutive floats at p, at most lim of them valid (the rest zero).
__device__ __forceinline__ float4 grad_load4(const float* p, int lim) {
  if (lim >= 4 && (reinterpret_cast<uintptr_t>(p) & 15u) == 0) return *reinterpret_cast<const float4*>(p);
  return make_float4(lim > 0 ? p[0] : 0.f, lim > 1 ? p[1] : 0.f, lim > 2 ? p[2] : 0.f, lim > 3 ? p[3] : 0.f);
}

// acc[x][y] += sum_{k<K} A[r][k] B[k][c] for r = 4 ty + 64 (x / 4) + x % 4, c = 4 tx + 64 (y / 4) + y % 4 (256
// threads, tx = tid % 16, ty = tid / 16); A: mlim rows of lda, B: rows of ldb with nlim columns.
__device__ __forceinline__ void mma128(float (&acc)[8][8], Smem128& sm, const float* A, int64_t lda, int64_t mlim,
                                       const float* B, int64_t ldb, int64_t nlim, int K) {
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  const int ar = tid >> 1, ak = (tid & 1) * 4, br = tid >> 5, bc = (tid & 31) * 4;
  const int blim = (int)min((int64_t)4, max((int64_t)0, nlim - bc));
  float4 a, b;
  auto load = [&](int k0) {
    a = ar < mlim ? grad_load4(A + (int64_t)ar * lda + k0 + ak, min(4, K - k0 - ak)) : make_float4(0.f, 0.f, 0.f, 0.f);
    b = k0 + br < K ? grad_load4(B + (int64_t)(k0 + br) * ldb + bc, blim) : make_float4(0.f, 0.f, 0.f, 0.f);
  };
  auto stash = [&](int s) {
    sm.a[s][ak][ar] = a.x;
    sm.a[s][ak + 1][ar] = a.y;
    sm.a[s][ak + 2][ar] = a.z;
    sm.a[s][ak + 3][ar] = a.w;
    *reinterpret_cast<float4*>(&sm.b[s][br][bc]) = b;
  };
  if (K <= 0) return;
  load(0);
  __syncthreads();
  stash(0);
  __syncthreads();
  int cur = 0;
  for (int k0 = 0; k0 < K; k0 += GK) {
    const bool more = k0 + GK < K;
    if (more) load(k0 + GK);
#pragma unroll
    for (int kk = 0; kk < GK; ++kk) {
      const float4 a0 = *reinterpret_cast<const float4*>(&sm.a[cur][kk][4 * ty]);
      const float4 a1 = *reinterpret_cast<const float4*>(&sm.a[cur][kk][64 + 4 * ty]);
      const float4 b0 = *reinterpret_cast<const float4*>(&sm.b[cur][kk][4 * tx]);
      const float4 b1 = *reinterpret_cast<const float4*>(&sm.b[cur][kk][64 + 4 * tx]);
      const float ra[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
      const float rb[8] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
#pragma unroll
      for (int x = 0; x < 8; ++x)
#pragma unroll
        for (int y = 0; y < 8; ++y) acc[x][y] = fmaf(ra[x], rb[y], acc[x][y]);
    }
    if (more) {
      stash(cur ^ 1);
      __syncthreads();
      cur ^= 1;
    }
  }
}
__device__ __forceinline__ int row128(int x) { return 4 * (int)(threadIdx.x >> 4) + 64 * (x >> 2) + (x & 3); }
__device__ __forceinline__ int col128(int y) { return 4 * (int)(threadIdx.x & 15) + 64 * (y >> 2) + (y & 3); }

__global__ void __launch_bounds__(256) k_grad_m1_128(const float* __restrict__ VbT, const float* __restrict__ Vt,
                                                     int64_t n, int s, Pieces pc, int npieces, int per_slice,
                                                     double* __restrict__ partial) {
  grid_dep_wait();
  grid_dep_launch();
  __shared__ __align__(16) Smem128 sm;
  const int i0 = blockIdx.y * 128, j0 = blockIdx.x * 128;
  double* P = partial + (int64_t)blockIdx.z * s * s;
  bool first = true;
  for (int p = blockIdx.z * per_slice; p < min(npieces, (int)(blockIdx.z + 1) * per_slice); ++p) {
    int64_t q0;
    const int K = pc.get(p, q0);
    float acc[8][8];
#pragma unroll
    for (int x = 0; x < 8; ++x)
#pragma unroll
      for (int y = 0; y < 8; ++y) acc[x][y] = 0.f;
    mma128(acc, sm, VbT + (int64_t)i0 * n + q0, n, s - i0, Vt + q0 * s + j0, s, s - j0, K);
#pragma unroll
    for (int x = 0; x < 8; ++x)
#pragma unroll
      for (int y = 0; y < 8; ++y) {
        const int i = i0 + row128(x), j = j0 + col128(y);
        if (i < s && j < s) {
          double* o = P + (int64_t)i * s + j;  // the slice's FP64 sum stays in the partial (no room in registers)
          *o = first ? (double)acc[x][y] : *o + (double)acc[x][y];
        }
      }
    first = false;
  }
}

// k_grad_vbar with 128 x 128 tiles (grid: x over points, y over support coordinates).
__global__ void __launch_bounds__(256) k_grad_vbar_128(const float* __restrict__ PsiT, const float* __restrict__ GVT,
                                                       const float* __restrict__ LcT, const double* __restrict__ beta,
                                                       int64_t n, int s, float* __restrict__ VbT) {
  grid_dep_wait();
  grid_dep_launch();
  __shared__ __align__(16) Smem128 sm;
  const int k0 = blockIdx.y * 128;
  const int64_t p0 = (int64_t)blockIdx.x * 128;
  float acc[8][8];
#pragma unroll
  for (int x = 0; x < 8; ++x)
#pragma unroll
    for (int y = 0; y < 8; ++y) acc[x][y] = 0.f;
  mma128(acc, sm, LcT + (int64_t)k0 * s + k0, s, s - k0, PsiT + (int64_t)(1 + k0) * n + p0, n, n - p0, s - k0);
#pragma unroll
  for (int x = 0; x < 8; ++x)
#pragma unroll
    for (int y = 0; y < 8; ++y) {
      const int k = k0 + row128(x);
      const int64_t p = p0 + col128(y);
      if (k < s && p < n)
        VbT[(int64_t)k * n + p] = (float)(beta[k] * (double)PsiT[p]) - acc[x][y] - 2.f * GVT[(int64_t)k * n + p];
    }
}

// k_grad_kds in FP32 on tiles of TS2 x TS2 (128 or, for small problems, 64): the product is parked in shared memory,
// then a thread takes one point and every (256 / TS2)-th support coordinate for the covariance terms, which are FP64 as
// there (a float difference or exponential would lose what cancels in the sums; a pair at any distance gives 0 x finite).
// D: d rounded up to 8 or MAXD, the bound of the unrolled loops.  The FP64 terms bound it (4 instructions a dimension,
// about 20 for exp, one per 64 clocks and scheduler): 8.4 ms at N = 65,536, s = 1,024, d = 8 (9.0 with one CTA per SM,
// whose product and terms do not overlap), against 12.8 of k_grad_kds.
template <int TS2, int D>
__global__ void __launch_bounds__(256, 2) k_grad_kds_f32(const float* __restrict__ VbT, const float* __restrict__ ET,
                                                      const float* __restrict__ xs, const float* __restrict__ ss, int d,
                                                      int64_t n, int s, double ss2, double* __restrict__ partial) {
  grid_dep_wait();
  grid_dep_launch();
  extern __shared__ __align__(16) unsigned char smraw[];
  float* prod = reinterpret_cast<float*>(smraw);                            // [TS2][TS2 + 1]
  double(*xk)[D] = reinterpret_cast<double(*)[D]>(prod + TS2 * (TS2 + 4));  // [TS2][D]
  __shared__ double red[8][D + 1];
  const int k0 = blockIdx.y * TS2;
  const int64_t p0 = (int64_t)blockIdx.x * TS2;
  for (int e = threadIdx.x; e < TS2 * D; e += 256) {
    const int r = e / D, q = e % D;
    xk[r][q] = (k0 + r < s && q < d) ? (double)ss[(int64_t)(k0 + r) * d + q] : 0.0;
  }
  if constexpr (TS2 == 128) {
    Smem128& sm = *reinterpret_cast<Smem128*>(smraw);
    float acc[8][8];
#pragma unroll
    for (int x = 0; x < 8; ++x)
#pragma unroll
      for (int y = 0; y < 8; ++y) acc[x][y] = 0.f;
    mma128(acc, sm, ET + (int64_t)k0 * s + k0, s, s - k0, VbT + (int64_t)k0 * n + p0, n, n - p0, s - k0);
    __syncthreads();
#pragma unroll
    for (int x = 0; x < 8; ++x)
#pragma unroll
      for (int y = 0; y < 8; ++y) prod[row128(x) * (TS2 + 1) + col128(y)] = acc[x][y];
  } else {
    GemmSmem<float>& sm = *reinterpret_cast<GemmSmem<float>*>(smraw);
    float acc[4][4] = {};
    auto fa = [&](int r, int ii) -> float { return (k0 + r < s) ? ET[(int64_t)(k0 + r) * s + k0 + ii] : 0.f; };
    auto fb = [&](int r, int ii) -> float { return (p0 + r < n) ? VbT[(int64_t)(k0 + ii) * n + p0 + r] : 0.f; };
    tile_mma<float, true, false>(acc, s - k0, sm, fa, fb);
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
      for (int b = 0; b < 4; ++b) prod[(ty + 16 * a) * (TS2 + 1) + tx + 16 * b] = acc[a][b];
  }
  __syncthreads();
  const int pc = threadIdx.x % TS2;
  const int64_t p = p0 + pc;
  double xp[D], gl[D], gs = 0.0;
#pragma unroll
  for (int q = 0; q < D; ++q) {
    xp[q] = (p < n && q < d) ? (double)xs[p * d + q] : 0.0;
    gl[q] = 0.0;
  }
  if (p < n)
    for (int kr = threadIdx.x / TS2; kr < min(TS2, s - k0); kr += 256 / TS2) {
      double d2 = 0.0;
#pragma unroll
      for (int q = 0; q < D; ++q)
        if (q < d) {
          const double t = xk[kr][q] - xp[q];
          d2 += t * t;
        }
      const double kg = (double)prod[kr * (TS2 + 1) + pc] * exp(-0.5 * d2);
      gs += kg;
#pragma unroll
      for (int q = 0; q < D; ++q)
        if (q < d) {
          const double t = xk[kr][q] - xp[q];
          gl[q] += kg * t * t;
        }
    }
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
  for (int q = 0; q < D + 1; ++q)
    if (q < d || q == D) {
      double v = q < D ? gl[q < D ? q : 0] : gs;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
      if (lane == 0) red[warp][q] = v;
    }
  __syncthreads();
  double* P = partial + ((int64_t)blockIdx.y * gridDim.x + blockIdx.x) * (d + 2);
  if (threadIdx.x <= d) {
    const int q = threadIdx.x < d ? threadIdx.x : D;
    double v = 0.0;
    for (int k = 0; k < 8; ++k) v += red[k][q];
    P[threadIdx.x] = v * (threadIdx.x < d ? ss2 : 2.0 * ss2);
  }
  if (threadIdx.x == d + 1) P[d + 1] = 0.0;
}

__global__ void k_sum_chunks(const double* __restrict__ partial, int nchunk, int64_t len, double* __restrict__ out) {
  grid_dep_wait();
  grid_dep_launch();
  int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (e >= len) return;
  double v = 0.0;
  for (int c = 0; c < nchunk; ++c) v += partial[(int64_t)c * len + e];
  out[e] = v;
}

// Dense FP64 product C = alpha op(A) op(B) (s x s, row-major, leading dims lda/ldb/ldc) of triangular operands.
// SHAPE says which terms and results are zero: bit 0: op(A)[i][k] = 0 for k < i; bit 1: op(A)[i][k] = 0 for k > i;
// bit 2: op(B)[k][j] = 0 for k < j; bit 3: only C's lower triangle is wanted (the rest is left).  TILE x TILE results
// a CTA of 256 threads: 16 where 32 would leave SMs without a tile (FP64: 16 K clocks a 64-wide tile and K, which
// made the four products of s = 100 130 us each on four CTAs).
template <bool TA, bool TBm, int SHAPE, int TILE>
__global__ void __launch_bounds__(256) k_dgemm(const double* __restrict__ A, int64_t lda, const double* __restrict__ Bm,
                                               int64_t ldb, double* __restrict__ C, int64_t ldc, int s, double alpha) {
  grid_dep_wait();
  grid_dep_launch();
  constexpr int KT = 16, R = TILE / 16;
  __shared__ double sa[KT][TILE + 1], sb[KT][TILE + 1];
  const int i0 = blockIdx.y * TILE, j0 = blockIdx.x * TILE;
  if ((SHAPE & 8) && j0 > i0 + TILE - 1) return;
  int kb = 0, ke = s;
  if (SHAPE & 1) kb = max(kb, i0);
  if (SHAPE & 4) kb = max(kb, j0);
  if (SHAPE & 2) ke = min(ke, i0 + TILE);
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  double acc[R][R] = {};
  for (int k0 = kb; k0 < ke; k0 += KT) {
    for (int e = threadIdx.x; e < TILE * KT; e += 256) {
      const int ra = TA ? e % TILE : e / KT, ka = TA ? e / TILE : e % KT;
      sa[ka][ra] = (i0 + ra < s && k0 + ka < ke)
                       ? (TA ? A[(int64_t)(k0 + ka) * lda + i0 + ra] : A[(int64_t)(i0 + ra) * lda + k0 + ka])
                       : 0.0;
      const int rb = TBm ? e / KT : e % TILE, kq = TBm ? e % KT : e / TILE;
      sb[kq][rb] = (j0 + rb < s && k0 + kq < ke)
                       ? (TBm ? Bm[(int64_t)(j0 + rb) * ldb + k0 + kq] : Bm[(int64_t)(k0 + kq) * ldb + j0 + rb])
                       : 0.0;
    }
    __syncthreads();
#pragma unroll
    for (int kk = 0; kk < KT; ++kk) {
      double a[R], b[R];
#pragma unroll
      for (int q = 0; q < R; ++q) {
        a[q] = sa[kk][ty + 16 * q];
        b[q] = sb[kk][tx + 16 * q];
      }
#pragma unroll
      for (int p = 0; p < R; ++p)
#pragma unroll
        for (int q = 0; q < R; ++q) acc[p][q] = fma(a[p], b[q], acc[p][q]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int p = 0; p < R; ++p)
#pragma unroll
    for (int q = 0; q < R; ++q) {
      const int i = i0 + ty + 16 * p, j = j0 + tx + 16 * q;
      if (i < s && j < s) C[(int64_t)i * ldc + j] = alpha * acc[p][q];
    }
}

// Phi(X): lower triangle with halved diagonal, in place (s x s, ld s)
static __global__ void k_phi(double* __restrict__ X, int s) {
  grid_dep_wait();
  grid_dep_launch();
  int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (e >= (int64_t)s * s) return;
  int i = (int)(e / s), j = (int)(e % s);
  if (j > i) X[e] = 0.0;
  else if (j == i) X[e] *= 0.5;
}

// after k_phi on a copy of L: restore the diagonal halved by k_phi (x2)
static __global__ void k_tril_fix(double* __restrict__ X, int s) {
  grid_dep_wait();
  grid_dep_launch();
  int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (e >= (int64_t)s * s) return;
  int i = (int)(e / s), j = (int)(e % s);
  if (i == j) X[e] *= 2.0;
}

// <Sigma-bar_SS, dK_SS/dtheta> (jitter held fixed); one CTA row-chunk per block
static __global__ void k_grad_kss(const double* __restrict__ Sb, const double* __restrict__ ss, int s, int d,
                                  double ss2, double* __restrict__ partial) {
  grid_dep_wait();
  grid_dep_launch();
  __shared__ double red[NT];
  double gl[MAXD];
  for (int q = 0; q < d; ++q) gl[q] = 0.0;
  double gsig = 0.0;
  const int i = blockIdx.x;
  for (int j = threadIdx.x; j < s; j += NT) {
    double d2 = 0.0;
    for (int q = 0; q < d; ++q) {
      double t = ss[(int64_t)i * d + q] - ss[(int64_t)j * d + q];
      d2 += t * t;
    }
    double kg = Sb[(int64_t)i * s + j] * ss2 * exp(-0.5 * d2);
    for (int q = 0; q < d; ++q) {
      double t = ss[(int64_t)i * d + q] - ss[(int64_t)j * d + q];
      gl[q] += kg * t * t;
    }
    gsig += 2.0 * kg;
  }
  double* P = partial + (int64_t)i * (d + 2);
  for (int q = 0; q < d + 1; ++q) {
    red[threadIdx.x] = (q < d) ? gl[q] : gsig;
    __syncthreads();
    for (int o = NT / 2; o > 0; o >>= 1) {
      if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
      __syncthreads();
    }
    if (threadIdx.x == 0) P[q] = red[0];
    __syncthreads();
  }
  if (threadIdx.x == 0) P[d + 1] = 0.0;
}

}  // namespace lma
