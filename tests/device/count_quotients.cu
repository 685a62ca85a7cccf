// The reciprocals and quotients of counts (ccc_metric.cuh) against CUDA's
// correctly rounded ones and against the exact values in double precision.
//
// Prints, one number per line:
//   reciprocals of the whole numbers below 2^24 that differ from __frcp_rn;
//   reciprocals of the single-precision whole numbers from 2^24 to 2^31 that differ
//     (sums of the tallies of several cohorts);
//   quotients x / d checked, and those that differ from __fdiv_rn;
//   the largest relative error of a quotient, in units of 2^-24.
// Quotients: every x <= d for d <= 2,048; for 2^17 larger d (the first and last
// 1,024 of every octave, the rest spread) the 64 x next to 0 and d, 128 spread
// over the range, and for each the numerator d - gamma x of a JOINT factor, for
// gamma = 2/3 and 1.
#include <cstdint>
#include <cstdio>

#include "ccc.h"
#include "ccc_dev.cuh"
#include "ccc_metric.cuh"

using namespace ccc;

struct Found {
  unsigned long long rcp, rcp_large, quotients, differ, worst;
};

__device__ void quotient(float x, float d, float inv, Found &f) {
  const float q = div_count(x, d, inv);
  const float2 q2 = div_count(make_float2(x, x), d, inv);
  ++f.quotients;
  f.differ += q != __fdiv_rn(x, d);
  const double e = static_cast<double>(x) / static_cast<double>(d);
  double r = x == 0.f ? (q == 0.f ? 0.0 : 1e9) : fabs(static_cast<double>(q) - e) / e * 0x1p24;
  if (q2.x != q || q2.y != q) r = 1e9;  // the two-wide form is the same operation
  const unsigned long long bits = __double_as_longlong(r);  // ordered as the value: r >= 0
  if (bits > f.worst) f.worst = bits;
}

__device__ void quotients(float x, float d, float inv, Found &f) {
  quotient(x, d, inv, f);
  quotient(__fmaf_rn(-static_cast<float>(2.0 / 3.0), x, d), d, inv, f);
  quotient(__fmaf_rn(-1.f, x, d), d, inv, f);
}

__global__ void check(Found *out) {
  const uint32_t t = blockIdx.x * blockDim.x + threadIdx.x, n = gridDim.x * blockDim.x;
  Found f = {};
  for (uint32_t d = 1 + t; d < (1u << 24); d += n) {
    const float x = static_cast<float>(d);
    f.rcp += rcp_count(x) != __frcp_rn(x);
  }
  for (uint32_t b = __float_as_uint(0x1p24f) + t; b <= __float_as_uint(0x1p31f); b += n) {
    const float x = __uint_as_float(b);
    f.rcp_large += rcp_count(x) != __frcp_rn(x);
  }
  for (uint32_t k = t; k < 2048u * 2049u; k += n) {
    const uint32_t d = k / 2049u + 1, x = k % 2049u;
    if (x > d) continue;
    quotients(static_cast<float>(x), static_cast<float>(d), rcp_count(static_cast<float>(d)), f);
  }
  for (uint32_t k = t; k < (1u << 17); k += n) {
    uint32_t d;
    if (k < 13u * 2048u) {  // octaves 2^11 .. 2^24
      const uint32_t o = 11 + k / 2048u, r = k % 2048u;
      d = r < 1024u ? (1u << o) + r : (2u << o) - (r - 1023u);
    } else {
      uint64_t h = k * 0x9E3779B97F4A7C15ull;
      h ^= h >> 29;
      d = 2048u + static_cast<uint32_t>(h * 0xBF58476D1CE4E5B9ull >> 40) % ((1u << 24) - 2048u);
    }
    const float df = static_cast<float>(d), inv = rcp_count(df);
    for (uint32_t x = 0; x < 64u; ++x) {
      quotients(static_cast<float>(x), df, inv, f);
      quotients(static_cast<float>(d - x), df, inv, f);
    }
    uint64_t h = d * 0x94D049BB133111EBull + 1;
    for (int s = 0; s < 128; ++s) {
      h = h * 6364136223846793005ull + 1442695040888963407ull;
      quotients(static_cast<float>(static_cast<uint32_t>(h >> 33) % (d + 1)), df, inv, f);
    }
  }
  atomicAdd(&out->rcp, f.rcp);
  atomicAdd(&out->rcp_large, f.rcp_large);
  atomicAdd(&out->quotients, f.quotients);
  atomicAdd(&out->differ, f.differ);
  atomicMax(&out->worst, f.worst);
}

int main() {
  Found *d, h;
  if (cudaMalloc(&d, sizeof h) != cudaSuccess || cudaMemset(d, 0, sizeof h) != cudaSuccess) return 1;
  check<<<152 * 8, 256>>>(d);
  if (cudaMemcpy(&h, d, sizeof h, cudaMemcpyDeviceToHost) != cudaSuccess) return 1;
  double worst;
  static_assert(sizeof worst == sizeof h.worst, "the bits of a double");
  __builtin_memcpy(&worst, &h.worst, sizeof worst);
  std::printf("%llu\n%llu\n%llu\n%llu\n%.10f\n", h.rcp, h.rcp_large, h.quotients, h.differ, worst);
}
