"""The sums of the predictions have FP64's accuracy and range: kernels against exact sums of crafted rows.

A lane's sum of any crafted row but the random one is exact in FP64, five adds across the warp follow: within 5 x 2^-53
of the terms' magnitudes.  Random terms: each lane adds n / 32 of them, (n / 32 + 5) 2^-53.  20,000 terms are more than
the kernels add in floats."""
import math

import numpy as np
import pytest

from _native import compile_program, run_program

pytestmark = pytest.mark.gpu

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include <vector>
#include "lma_kernels.cuh"
#include "lma_tc.cuh"
using namespace lma;
#define CK(x) do { cudaError_t e_ = (x); if (e_ != cudaSuccess) { printf("%s\n", cudaGetErrorString(e_)); return 1; } } while (0)
template <typename T> T* up(const std::vector<T>& v) {
  T* p = nullptr;
  if (cudaMalloc((void**)&p, sizeof(T) * v.size()) != cudaSuccess) exit(1);
  if (cudaMemcpy(p, v.data(), sizeof(T) * v.size(), cudaMemcpyHostToDevice) != cudaSuccess) exit(1);
  return p;
}
template <typename T> void show(const char* name, const T* d, size_t n) {
  std::vector<T> h(n);
  cudaMemcpy(h.data(), d, sizeof(T) * n, cudaMemcpyDeviceToHost);
  printf("%s", name);
  for (T x : h) printf(" %.17g", (double)x);
  printf("\n");
}
int main(int argc, char** argv) {
  const int n = atoi(argv[2]), rows = atoi(argv[3]);
  FILE* f = fopen(argv[1], "rb");
  std::vector<float> P((size_t)rows * n), E((size_t)rows * n), H(4 * rows);
  std::vector<double> beta(n);
  if (!f || fread(P.data(), 4, P.size(), f) != P.size() || fread(E.data(), 4, E.size(), f) != E.size() ||
      fread(beta.data(), 8, beta.size(), f) != beta.size() || fread(H.data(), 4, H.size(), f) != H.size())
    return 2;
  // one window and one pair per row, so that every row has its own L^-1 e
  std::vector<Pair> pairs(rows);
  std::vector<Win> wins(rows);
  std::vector<int4> items;
  for (int r = 0; r < rows; ++r) {
    Pair p{};
    p.pbase = (int64_t)r * n;
    p.win = r;
    p.u0 = r;
    p.nu = 1;
    p.c1 = n;
    pairs[r] = p;
    Win w{};
    w.n = w.npad = n;
    w.ew = (int64_t)r * n;
    wins[r] = w;
    items.push_back(make_int4(r, 1, 0, 0));
  }
  float *Pd = up(P), *Ed = up(E), *Hd = up(H);
  double* bd = up(beta);
  float4* bs = up(std::vector<float4>(n));
  k_split_beta<<<(n + 255) / 256, 256>>>(bd, n, bs);
  Pair* pd = up(pairs);
  Win* wd = up(wins);
  int4* id = up(items);
  std::vector<double> zero(rows, 0.0);
  double *t1 = up(zero), *t2 = up(zero), *q = up(zero), *mean = up(zero), *var = up(zero), *z = up(zero);
  const int nb = (rows * 32 + 255) / 256;
  k_pred_t12<float><<<nb, 256>>>(pd, id, rows, wd, Pd, Ed, t1, t2);
  k_row_sqnorm<<<nb, 256>>>(Pd, rows, n, q);
  k_pred_final<float><<<nb, 256>>>(Pd, rows, n, bd, bs, z, z, z, 1, 0.0, 0.0, mean, var);
  // hsum: three partial rows and Vu, one column, one test block
  std::vector<int4> tb{make_int4(0, 3, 0, rows)};
  std::vector<int64_t> prow{0, rows, 2 * (int64_t)rows};
  float* h = up(std::vector<float>(rows, 0.f));
  k_pred_hsum<<<dim3((rows + 255) / 256, 1), 256>>>(up(tb), up(prow), Hd, Hd + 3 * rows, 1, h);
  CK(cudaDeviceSynchronize());
  show("t1", t1, rows);
  show("t2", t2, rows);
  show("sq", q, rows);
  show("mean", mean, rows);
  show("var", var, rows);
  show("h", h, rows);
  return 0;
}
"""


def _rows(N):
    i = np.arange(N) // 32  # a lane's i-th term
    tail = np.where(i == 0, 1.0, np.where(i == 1, 2.0 ** -13, 2.0 ** -26))
    inf = tail.copy()
    inf[77] = np.inf
    nan = tail.copy()
    nan[5] = np.nan
    rng = np.random.default_rng(3)
    ones = np.ones(N)
    P = [tail,                                        # many terms far below the first two
         ones * 2.0 ** -60 * (1 + 2.0 ** -20),        # the products' low halves underflow a float
         ones * 2.0 ** -90,                           # the products underflow a float
         ones * 2.0 ** 100,                           # ... overflow it
         inf, nan, np.zeros(N), rng.standard_normal(N)]
    E = [tail, ones * 2.0 ** -60 * (1 + 2.0 ** -21), ones * 2.0 ** -90, ones * 2.0 ** 100, ones, ones, ones,
         rng.standard_normal(N)]
    return np.array(P, dtype=np.float32), np.array(E, dtype=np.float32)


def _agree(got, terms, rel):
    if np.isnan(terms).any():
        return math.isnan(got)
    if np.isinf(terms).any():
        return got == np.inf
    return abs(got - math.fsum(terms)) <= rel * math.fsum(np.abs(terms))


@pytest.mark.parametrize("N, beta7", [(4096, 1.0), (4096, 1e300), (4096, 1e-40 / 3), (20000, 1.0)])
def test_sums_have_fp64_accuracy_and_range(tmp_path, N, beta7):
    P, E = _rows(N)
    rows = len(P)
    beta = np.full(N, 1 + 2.0 ** -25 + 2.0 ** -52)  # three floats, but for one
    beta[7] = beta7
    # partial rows a, b, c and Vu of one column each: h = a + b + c - Vu, rounded once
    H = np.zeros((4, rows), dtype=np.float32)
    H[:, 0] = 1, 2.0 ** -24, 2.0 ** -50, 0             # above the tie: rounds up
    H[:, 1] = 1, 2.0 ** -24, -2.0 ** -50, 0            # below it: rounds down
    H[:, 2] = 3e38, 3e38, -3e38, 1e38                  # a partial sum overflows a float
    H[:, 3] = np.inf, 1, 2, 3
    H[:, 4] = 1, -1, 2.0 ** -140, 0
    H[:, 5] = 1, 2.0 ** -24, 0, 0                      # the tie itself: to even
    H[:, 6] = 2.0 ** 30, 1, -2.0 ** 30, 2.0 ** -23
    H[:, 7] = np.nan, 1, 1, 1
    data = tmp_path / "in.bin"
    data.write_bytes(P.tobytes() + E.tobytes() + beta.tobytes() + H.tobytes())
    out = run_program(compile_program(PROGRAM, tmp_path), data, N, rows)
    got = {ln.split()[0]: [float(x) for x in ln.split()[1:]] for ln in out.splitlines()}
    P64, E64 = P.astype(np.float64), E.astype(np.float64)
    wrong = []
    with np.errstate(all="ignore"):
        for r in range(rows):
            rel = (N / 32 + 5) * 2.0 ** -53 if r == rows - 1 else 5 * 2.0 ** -53
            for name, terms in (("t1", P64[r] * E64[r]), ("t2", P64[r] ** 2), ("sq", P64[r] ** 2)):
                if not _agree(got[name][r], terms, rel):
                    wrong.append((name, r, got[name][r], math.fsum(terms) if np.isfinite(terms).all() else None))
            # the mean's products are rounded once each (FMA accumulation): the general bound
            if not _agree(got["mean"][r], P64[r] * beta, (N / 32 + 6) * 2.0 ** -53):
                wrong.append(("mean", r, got["mean"][r]))
            if not _agree(-got["var"][r], P64[r] ** 2, rel):
                wrong.append(("var", r, got["var"][r]))
            h64 = H[:, r].astype(np.float64)
            want = np.float32(((h64[0] + h64[1]) + h64[2]) - h64[3])
            if not (np.float32(got["h"][r]) == want or (np.isnan(want) and math.isnan(got["h"][r]))):
                wrong.append(("h", r, got["h"][r], want))
    assert not wrong, wrong
