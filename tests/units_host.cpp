// More entry points to the host build of the device arithmetic.
#include "fixed_host.cpp"

extern "C" void fx_floor58(const double* v, int top, long long* out, long long n) {
  for (long long i = 0; i < n; ++i) out[i] = (long long)fx::floor58(v[i], top);
}
