// The plane access of the kernels compiled for the host.
#define __device__
#define __forceinline__ inline
#include "../paper_1910_13515_gb300/csrc/plane.cuh"

// Byte offset of element `index` of a plane (of doubles, or of floats) from the plane's start.
extern "C" unsigned long long plane_offset(int doubles, int index) {
  if (doubles) {
    double* p = reinterpret_cast<double*>(1ull << 40);
    return reinterpret_cast<unsigned long long>(&lbm39::at(p, index)) - (1ull << 40);
  }
  float* p = reinterpret_cast<float*>(1ull << 40);
  return reinterpret_cast<unsigned long long>(&lbm39::at(p, index)) - (1ull << 40);
}
