// fp_bits.cuh compiled for the host, with the device's bit intrinsics written out, and loops over arrays.
#include <stdint.h>
#include <string.h>

#define __device__
#define __forceinline__ inline

static inline unsigned __float_as_uint(float x) {
  unsigned u;
  memcpy(&u, &x, 4);
  return u;
}
static inline float __uint_as_float(unsigned u) {
  float x;
  memcpy(&x, &u, 4);
  return x;
}
static inline uint64_t bits64(double x) {
  uint64_t u;
  memcpy(&u, &x, 8);
  return u;
}
static inline int __double2hiint(double x) { return (int)(bits64(x) >> 32); }
static inline int __double2loint(double x) { return (int)(uint32_t)bits64(x); }
static inline double __hiloint2double(int hi, int lo) {
  const uint64_t u = (uint64_t)(uint32_t)hi << 32 | (uint32_t)lo;
  double x;
  memcpy(&x, &u, 8);
  return x;
}
static inline unsigned __funnelshift_l(unsigned lo, unsigned hi, unsigned shift) {
  const unsigned s = shift & 31;
  return s ? hi << s | lo >> (32 - s) : hi;
}

#include "fp_bits.cuh"

extern "C" {
void widen_all(const float *x, double *y, long long n) {
  for (long long i = 0; i < n; i++) y[i] = ibfsa::widen(x[i]);
}
void narrow_all(const double *x, float *y, long long n) {
  for (long long i = 0; i < n; i++) y[i] = ibfsa::narrow(x[i]);
}
void low_precision_all(const double *x, float *y, long long n) {
  for (long long i = 0; i < n; i++) y[i] = ibfsa::low_precision(x[i]);
}
}
