// More entry points to the host build of the device arithmetic.
#include "fixed_host.cpp"

extern "C" void fx_floor58(const double* v, int top, long long* out, long long n) {
  for (long long i = 0; i < n; ++i) out[i] = (long long)fx::floor58(v[i], top);
}

// The multipliers of the Gaussian start, with the fixed-point exponential and with CUDA's (here the
// host's) exp.  Returns 0 where the former gives the state up.
extern "C" int fx_gaussian(const double* u, double T, double* fixed, double* fp64) {
  double ws[WS_DOUBLES] = {0};
  fx::load_table();
  const int ok = gaussian_guess_fx<1>(u[0], u[1], u[2], T, WS<1>{ws});
  for (int k = 0; k < NM; ++k) fixed[k] = ws[WS_LAM + k];
  gaussian_guess<1>(u[0], u[1], u[2], T, WS<1>{fp64});
  return ok;
}
