#include "ozaki_value.cuh"

extern "C" void group_values(int n, const long long* g0, const long long* g1, const int* exy, double* out) {
  for (int i = 0; i < n; ++i) out[i] = cqr::group_value(g0[i], g1[i], exy[i]);
}
