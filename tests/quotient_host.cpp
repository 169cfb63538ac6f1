// Host build of quotient.cuh for the unit tests.
#include "../paper_2606_10030_gb300/csrc/quotient.cuh"

extern "C" void quotients(const uint64_t* b, const uint32_t* c, int64_t n, uint64_t* out, uint8_t* ok) {
  for (int64_t i = 0; i < n; ++i) ok[i] = agg::quotient_bits(b[i], c[i], &out[i]) ? 1 : 0;
}
extern "C" void conversions(const int64_t* v, int64_t n, uint64_t* out) {
  for (int64_t i = 0; i < n; ++i) out[i] = agg::float64_bits_of(v[i]);
}
