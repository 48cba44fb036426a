"""The FP64 window factorisation when a wait runs out: the kernel ends with its error word set.

The chain CTA of three windows runs alone, without the CTAs that would hand it the tiles of its third panel, so its
waits give up (after a second or two) in the first window; it takes up no further one."""
import pytest

from _native import compile_program, run_program

pytestmark = pytest.mark.gpu

PROGRAM = r"""
#include <cstdio>
#include <vector>
#include "lma_f64.cuh"
using namespace lma;
using namespace lma::f64;
#define CK(x) do { cudaError_t e_ = (x); if (e_ != cudaSuccess) { printf("%s\n", cudaGetErrorString(e_)); return 1; } } while (0)
int main() {
  constexpr int NW = 3, LD = 64, NPAN = 4, CNT = (NPAN + 1) * CSTR + 2 * NPAN;
  std::vector<double> h((size_t)NW * LD * LD, 0.0);
  std::vector<FlowWin> fw(NW);
  for (int w = 0; w < NW; ++w) {
    for (int i = 0; i < LD; ++i) h[((size_t)w * LD + i) * LD + i] = 4.0;
    fw[w] = FlowWin{(int64_t)w * LD * LD, (int64_t)w * NPAN * TS * TS, (int64_t)w * CNT, LD, LD, NPAN, NPAN};
  }
  double *buf, *dv;
  FlowWin* fd;
  int *info, *err;
  unsigned* cnt;
  CK(cudaMalloc((void**)&buf, sizeof(double) * h.size()));
  CK(cudaMalloc((void**)&dv, sizeof(double) * NW * NPAN * TS * TS));
  CK(cudaMalloc((void**)&fd, sizeof(FlowWin) * NW));
  CK(cudaMalloc((void**)&info, sizeof(int) * NW));
  CK(cudaMalloc((void**)&err, sizeof(int)));
  CK(cudaMalloc((void**)&cnt, sizeof(unsigned) * NW * CNT));
  CK(cudaMemcpy(buf, h.data(), sizeof(double) * h.size(), cudaMemcpyHostToDevice));
  CK(cudaMemcpy(fd, fw.data(), sizeof(FlowWin) * NW, cudaMemcpyHostToDevice));
  CK(cudaMemset(info, 0, sizeof(int) * NW));
  CK(cudaMemset(err, 0, sizeof(int)));
  CK(cudaMemset(cnt, 0, sizeof(unsigned) * NW * CNT));
  k_f64_windows<<<1, FTH>>>(fd, NW, 1, buf, dv, info, nullptr, 0, cnt, err);
  CK(cudaGetLastError());
  CK(cudaDeviceSynchronize());
  int e = 0;
  std::vector<unsigned> c(NW * CNT);
  CK(cudaMemcpy(&e, err, sizeof(int), cudaMemcpyDeviceToHost));
  CK(cudaMemcpy(h.data(), buf, sizeof(double) * h.size(), cudaMemcpyDeviceToHost));
  CK(cudaMemcpy(c.data(), cnt, sizeof(unsigned) * NW * CNT, cudaMemcpyDeviceToHost));
  // the error word, the inverses published in each window, the first pivot of each window
  printf("%d", e);
  for (int w = 0; w < NW; ++w) printf(" %u", c[w * CNT + NPAN * CSTR]);
  for (int w = 0; w < NW; ++w) printf(" %g", h[(size_t)w * LD * LD]);
  printf("\n");
  return 0;
}
"""


def test_window_factorisation_ends_when_a_wait_runs_out(tmp_path):
    out = run_program(compile_program(PROGRAM, tmp_path), timeout=60).split()
    err, published, pivots = int(out[0]), [int(x) for x in out[1:4]], [float(x) for x in out[4:]]
    assert err == 1
    assert published == [1, 0, 0]      # panel 0 of the first window; panel 1 waits for a tile that nobody hands over
    assert pivots == [2.0, 4.0, 4.0]   # the other windows are left as they were
