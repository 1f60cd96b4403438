// Square root, reciprocal, quotient and reciprocal root of the mass-spring kernels (spring_math.cuh) on
// the GPU against FP64: every float that a squared length (1e-30 and up) or a guarded length (1e-4 to
// the root of the largest float) can be, and 2^28 quotients of both signs.  Prints for each the largest
// error in ulps of the result and the number of results that CUDA's own correctly rounded function
// (for the reciprocal root: rsqrtf) does not give.
#include <cmath>
#include <cstdio>
#include <cstring>

#include "../../paper_1910_00935_gb300/csrc/spring_math.cuh"

struct Worst {
  unsigned long long err[4];  // ulps in units of 2^-32
  unsigned long long differ[4];
};

__device__ double ulps(float got, double want) {
  int e;
  frexp(want, &e);  // want = m 2^e, 0.5 <= |m| < 1: an ulp is 2^(e - 24)
  return fabs((double)got - want) * ldexp(1.0, 24 - e);
}
__device__ void note(Worst& w, int k, float got, double want, float cuda) {
  const unsigned long long u = (unsigned long long)(ulps(got, want) * 4294967296.0);
  if (u > w.err[k]) w.err[k] = u;
  w.differ[k] += got != cuda;
}
__device__ unsigned hash(unsigned x) {
  x ^= x >> 16;
  x *= 0x7feb352du;
  x ^= x >> 15;
  x *= 0x846ca68bu;
  return x ^ (x >> 16);
}
// a float of random mantissa with an exponent in [lo, hi]
__device__ float draw(unsigned h, unsigned g, int lo, int hi) {
  return ldexpf(1.0f + (float)(h & 0x7fffff) * 0x1p-23f, lo + (int)(g % (unsigned)(hi - lo + 1)));
}

__global__ void check(unsigned sq_lo, unsigned sq_hi, unsigned len_lo, unsigned len_hi, Worst* out) {
  Worst w = {};
  const unsigned step = gridDim.x * blockDim.x, first = blockIdx.x * blockDim.x + threadIdx.x;
  for (unsigned long long b = sq_lo + (unsigned long long)first; b <= sq_hi; b += step) {
    const float x = __uint_as_float((unsigned)b), r = ms_rsqrt(x);
    note(w, 0, ms_sqrt(x, r), sqrt((double)x), __fsqrt_rn(x));
    note(w, 3, r, 1.0 / sqrt((double)x), rsqrtf(x));
  }
  for (unsigned long long b = len_lo + (unsigned long long)first; b <= len_hi; b += step) {
    const float x = __uint_as_float((unsigned)b);
    note(w, 1, ms_rcp(x), 1.0 / (double)x, __frcp_rn(x));
  }
  for (unsigned k = first; k < 1u << 28; k += step) {
    const unsigned a = hash(4 * k + 1), b = hash(4 * k + 2), c = hash(4 * k + 3);
    // lengths 2^-13 .. 2^64, numerators 2^-30 .. 2^101 (results and residuals are then normal)
    const float den = draw(a, c & 0xffff, -13, 63);
    float num = draw(b, c >> 16, -30, 100);
    if (a >> 31) num = -num;
    note(w, 2, ms_div(num, den), (double)num / (double)den, __fdiv_rn(num, den));
  }
  for (int k = 0; k < 4; ++k) {
    atomicMax(&out->err[k], w.err[k]);
    atomicAdd(&out->differ[k], w.differ[k]);
  }
}

static unsigned bits(float x) {
  unsigned b;
  std::memcpy(&b, &x, 4);
  return b;
}

int main() {
  Worst* out;
  if (cudaMallocManaged(&out, sizeof(Worst)) != cudaSuccess) return 1;
  std::memset(out, 0, sizeof(Worst));
  check<<<152 * 8, 256>>>(bits(1e-30f), bits(FLT_MAX), bits(1e-4f), bits(1.8446743e19f), out);
  if (cudaDeviceSynchronize() != cudaSuccess) return 2;
  const char* name[4] = {"sqrt", "rcp", "div", "rsqrt"};
  for (int k = 0; k < 4; ++k) std::printf("%s %.9f %llu\n", name[k], (double)out->err[k] / 4294967296.0, out->differ[k]);
  return 0;
}
