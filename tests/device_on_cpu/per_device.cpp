// What the library remembers per device, with a device chosen by the test.
#include "cqr_common.cuh"

static int device = 0;
extern "C" cudaError_t cudaGetDevice(int* d) {
  *d = device;
  return cudaSuccess;
}

// How often an opt-in guarded as in the library is made when the current
// device goes through devices[0 .. n).
extern "C" int opt_ins(const int* devices, int n) {
  cqr::PerDevice<bool> done;
  int made = 0;
  for (int i = 0; i < n; ++i) {
    device = devices[i];
    if (bool& set = done.here(); !set) {
      ++made;
      set = true;
    }
  }
  return made;
}
