// The bit arithmetic of the kernels (csrc/bits.cuh) behind a C interface, for tests on the host.
#include "bits.cuh"

extern "C" {

void host_rcp(long n, const double* d, double* out) {
  for (long i = 0; i < n; ++i) out[i] = mto::newton_rcp(d[i]);
}

void host_fixed56(long n, const unsigned long long* bits, int ex, unsigned long long* out) {
  for (long i = 0; i < n; ++i) out[i] = mto::fixed56(bits[i], ex);
}

void host_levels(long n, const long long* H, const long long* L, const int* ex, unsigned long long* out) {
  for (long i = 0; i < n; ++i) out[i] = mto::levels_to_double(H[i], L[i], ex[i]);
}

void host_split(long n, const unsigned long long* bits, float* hi, float* lo) {
  for (long i = 0; i < n; ++i) mto::split_pair(bits[i], hi[i], lo[i]);
}
}
