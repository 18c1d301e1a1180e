// chol_trapezoid on the CPU, its warps in a chosen order between barriers.
#include "chol_device.cuh"

// W: kb x (kb + nx) rows (leading dimension kb + nx), overwritten by the
// factor's rows, the diagonal in dg.  Returns the row that broke down, -1, or
// -2 if the block fell apart at a barrier.
template <int T>
static int run(const int* order, int kb, int nx, double* W, double* dg) {
  const int us = kb + nx;
  std::vector<double> rows(8 * us);
  std::vector<unsigned short> tab(kb * us);
  int broken = 0, ret = -1;
  const std::vector<int> warps(order, order + T / 32);
  const bool whole = device_on_cpu::run_block(T, warps, [&] {
    const int r = cqr::chol_trapezoid<T>(W, us, kb, nx, rows.data(), us, dg, tab.data(), &broken);
    if (threadIdx.x == 0) ret = r;
  });
  return whole ? ret : -2;
}

extern "C" int trapezoid(int T, const int* order, int kb, int nx, double* W, double* dg) {
  return T == 256 ? run<256>(order, kb, nx, W, dg) : run<512>(order, kb, nx, W, dg);
}
