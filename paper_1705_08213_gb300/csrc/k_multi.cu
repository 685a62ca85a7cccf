// 2-way CCC of markers with s allele states on the tcgen05 tensor cores.
//
// Sec. 7 item 2 extends CCC from biallelic SNPs to markers with any number of
// states: a pair of markers gets an s x s table.  Written with the state set
// S = {0..s-1}, Eqs. 1-3 keep their form, and the tally table is again a block
// of a Gram product (Sec. 3.1): with s count rows rho_i(a) per SNP,
// r_ij^{ab} = sum_q rho_{i,q}(a) rho_{j,q}(b) is entry (row(i,a), row(j,b)) of
// R R^T.  Counts 0, 1, 2 are exact in e4m3 and every sum stays an integer
// below 2^24, so the FP32 accumulation of kind::f8f6f4 is exact.
//
// Operand rows.  The rows of a SNP must sit in one 32-lane quarter of the
// accumulator so that the epilogue can sum a pair's table with warp shuffles:
// a quarter (32 rows) holds PW = floor(32 / s) SNPs, SNP i at rows
// 32 (i / PW) + s (i % PW) + a; the 32 - s PW rows left over are zero.  A
// 256-row block then holds 8 PW SNPs, on both sides of the product, and the
// SM-pair pipeline of the biallelic kernel (tc_pipeline_pair.cuh: 256 x 256
// tiles, cta_group::2) walks the upper triangle of those blocks.
//
// Epilogue: the thread of accumulator lane (i, a) holds r_ij^{ab} for every
// column (j, b) of its chunk.  n_ij comes from a shuffle sum over the s lanes
// of SNP i; the CCC values (Eq. 3, PERSNP or JOINT normalisation) use the same
// single-precision operations, in the same order, as the biallelic epilogue,
// so s = 2 reproduces the biallelic results bit for bit.
#include "k_multi.cuh"

namespace ccc {
namespace {

// Bytes of a 4-entry word whose low (high) nibble equals state a: 0x01 per byte.
__device__ __forceinline__ uint32_t nibble_eq(uint32_t nib, uint32_t a) {
  const uint32_t t = nib ^ (a * 0x01010101u);  // bytes 0..15, zero where equal
  return (~((t | 0x80808080u) - 0x01010101u) & 0x80808080u) >> 7;
}

// Bytes whose nibble is >= s (the entry is missing): 0x01 per byte.
__device__ __forceinline__ uint32_t nibble_ge(uint32_t nib, uint32_t s) {
  return (((nib | 0x80808080u) - s * 0x01010101u) & 0x80808080u) >> 7;
}

// Bytes q < n_f of the 4-entry word starting at entry q0: 0x01 per byte.
__device__ __forceinline__ uint32_t valid_bytes(int64_t q0, int64_t n_f) {
  const int64_t k = n_f - q0;
  if (k >= 4) return 0x01010101u;
  if (k <= 0) return 0u;
  return 0x01010101u & ((1u << (8 * k)) - 1u);
}

// ---------------------------------------------------------------- per-SNP counts
//
// One warp per SNP: s_i^a = sum_q rho_{i,q}(a) (Eq. 1 numerators), n_i, and the
// PERSNP factors 1 - gamma s_i^a / (2 n_i) rounded once to fp32 (the formula of
// the biallelic counts kernel).  Templated on the number of states S.
template <int S>
__global__ void __launch_bounds__(256) k_multi_counts(const uint8_t *__restrict__ geno, int64_t n_f,
                                                      int64_t n_v, int64_t ld,
                                                      int32_t *__restrict__ counts,
                                                      float *__restrict__ w, double gamma) {
  constexpr int s = S;
  const int lane = threadIdx.x & 31;
  const int64_t i = static_cast<int64_t>(blockIdx.x) * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (i >= n_v) return;
  const uint8_t *row = geno + i * ld;
  uint32_t c[S];
#pragma unroll
  for (int a = 0; a < S; ++a) c[a] = 0;
  uint32_t n = 0;
  const uint32_t us = static_cast<uint32_t>(s);
  auto count16 = [&](int64_t q0, const uint4 &v) {
    const uint32_t words[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const uint32_t lo = words[k] & 0x0F0F0F0Fu, hi = (words[k] >> 4) & 0x0F0F0F0Fu;
      const uint32_t present =
          valid_bytes(q0 + 4 * k, n_f) & ~(nibble_ge(lo, us) | nibble_ge(hi, us));
      n += __popc(present);
#pragma unroll
      for (int a = 0; a < S; ++a)
        c[a] += __popc(nibble_eq(lo, a) & present) + __popc(nibble_eq(hi, a) & present);
    }
  };
  // Four 16-byte loads in flight per lane, then the remainder one at a time.
  int64_t q0 = 16 * static_cast<int64_t>(lane);
  for (; q0 + 3 * 16 * 32 < n_f; q0 += 4 * 16 * 32) {
    uint4 v[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) v[u] = *reinterpret_cast<const uint4 *>(row + q0 + u * 16 * 32);
#pragma unroll
    for (int u = 0; u < 4; ++u) count16(q0 + u * 16 * 32, v[u]);
  }
  for (; q0 < n_f; q0 += 16 * 32) count16(q0, *reinterpret_cast<const uint4 *>(row + q0));
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    n += __shfl_xor_sync(0xffffffffu, n, o);
#pragma unroll
    for (int a = 0; a < S; ++a) c[a] += __shfl_xor_sync(0xffffffffu, c[a], o);
  }
  if (lane == 0) {
#pragma unroll
    for (int a = 0; a < S; ++a) {
      if (counts) counts[i * (s + 1) + a] = static_cast<int32_t>(c[a]);
      if (w) {
        const double f = n > 0 ? static_cast<double>(c[a]) / (2.0 * static_cast<double>(n)) : 0.0;
        w[i * s + a] = static_cast<float>(1.0 - gamma * f);
      }
    }
    if (counts) counts[i * (s + 1) + s] = static_cast<int32_t>(n);
  }
}

// PERSNP factors from an int32[n_v][s + 1] counts array (same formula).
__global__ void k_multi_factors(const int32_t *__restrict__ counts, int64_t n_v, int s,
                                float *__restrict__ w, double gamma) {
  const int64_t t = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (t >= n_v * s) return;
  const int64_t i = t / s;
  const int a = static_cast<int>(t - i * s);
  const double n = counts[i * (s + 1) + s];
  const double f = n > 0 ? counts[i * (s + 1) + a] / (2.0 * n) : 0.0;
  w[t] = static_cast<float>(1.0 - gamma * f);
}

// ---------------------------------------------------------------- operand rows
//
// One thread per (32-row quarter, 16 individuals): the quarter's PW SNPs each
// give s rows of 16 e4m3 counts (0x00, 0x38 = 1, 0x40 = 2); the rows past
// s PW, SNPs past n_v and individuals past n_f are zero.
__global__ void __launch_bounds__(256) k_multi_unpack(const uint8_t *__restrict__ geno, int64_t n_f,
                                                      int64_t n_v, int64_t ld, int s,
                                                      uint8_t *__restrict__ op, int64_t kpad,
                                                      int64_t n_quarters) {
  const int64_t chunks = kpad / 16;
  const int64_t total = n_quarters * chunks;
  const int pw = snps_per_quarter(s);
  const uint32_t us = static_cast<uint32_t>(s);
  for (int64_t t = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; t < total;
       t += static_cast<int64_t>(gridDim.x) * blockDim.x) {
    const int64_t g = t / chunks;
    const int64_t c = t - g * chunks;
    const int64_t q0 = 16 * c;
    uint8_t *dst = op + (32 * g) * kpad + q0;
    int r = 0;
    for (int u = 0; u < pw; ++u) {
      const int64_t i = g * pw + u;
      uint32_t words[4] = {0u, 0u, 0u, 0u};
      if (i < n_v && q0 < n_f) {
        const uint4 v = *reinterpret_cast<const uint4 *>(geno + i * ld + q0);
        words[0] = v.x;
        words[1] = v.y;
        words[2] = v.z;
        words[3] = v.w;
      }
      uint32_t lo[4], hi[4], present[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        lo[k] = words[k] & 0x0F0F0F0Fu;
        hi[k] = (words[k] >> 4) & 0x0F0F0F0Fu;
        present[k] = (i < n_v ? valid_bytes(q0 + 4 * k, n_f) : 0u) &
                     ~(nibble_ge(lo[k], us) | nibble_ge(hi[k], us));
      }
      for (int a = 0; a < s; ++a, ++r) {
        uint32_t e[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const uint32_t fx = nibble_eq(lo[k], a) & present[k];
          const uint32_t fy = nibble_eq(hi[k], a) & present[k];
          e[k] = (fx ^ fy) * 0x38u | (fx & fy) * 0x40u;  // count 1 -> 0x38, 2 -> 0x40
        }
        *reinterpret_cast<uint4 *>(dst + r * kpad) = make_uint4(e[0], e[1], e[2], e[3]);
      }
    }
    for (; r < 32; ++r) *reinterpret_cast<uint4 *>(dst + r * kpad) = make_uint4(0u, 0u, 0u, 0u);
  }
}

// FP4 (e2m1) operand rows: as k_multi_unpack with each count 0, 1, 2 stored
// as the nibble 0x0, 0x2, 0x4, two entries per byte (entry q in the low nibble
// of byte q / 2 for even q), rows of kpad / 2 bytes (kpad a multiple of 256);
// and, when w is set, the marker's PERSNP factors (the formula of
// k_multi_counts) from the same read.  One 128-thread block per marker (markers
// past n_v give zero rows, a quarter's last marker also its rows past S PW), or,
// without w, per marker and part of part_chunks 32-individual chunks of its row; a
// thread 32 individuals at a time, eight of them per step:
//   the low and high nibbles of eight entries are packed into one word each (x, y);
//   an entry with x >= S or y >= S gets nibble 15 in both;
//   per state a, a byte permutation with the nibbles as selectors looks up 2
//   where the nibble equals a (prmt itself: a selector above 7 gives a byte's
//   sign, here 0; __byte_perm takes three bits of it only), the sum
//   of both is the count's code, and the bytes are packed back to nibbles.
// About 12 operations per state and eight entries (40 when every byte was compared).
// GB300, 10,000 x 16,384, S = 4: counts 118 us and unpack 156 us -> 100 us (4.9 TB/s).
__device__ __forceinline__ uint32_t pack_nibbles(uint32_t b0, uint32_t b1) {
  return __byte_perm(b0 | (b0 >> 4), b1 | (b1 >> 4), 0x6420);
}

__device__ __forceinline__ uint32_t lookup_nibbles(uint32_t lo, uint32_t hi, uint32_t sel) {
  uint32_t r;
  asm("prmt.b32 %0, %1, %2, %3;" : "=r"(r) : "r"(lo), "r"(hi), "r"(sel));
  return r;
}

template <int S>
__global__ void __launch_bounds__(128) k_multi_unpack_e2m1(const uint8_t *__restrict__ geno,
                                                           int64_t n_f, int64_t n_v, int64_t ld,
                                                           uint8_t *__restrict__ op, int64_t kpad,
                                                           float *__restrict__ w, double gamma,
                                                           int part_chunks) {
  constexpr int PW = snps_per_quarter(S);
  const int64_t i = blockIdx.x;
  const int u = static_cast<int>(i % PW);
  const int64_t row_bytes = kpad / 2;
  uint8_t *const rows = op + (32 * (i / PW) + S * u) * row_bytes;
  const uint8_t *const src = geno + i * ld;
  const int begin = static_cast<int>(blockIdx.y) * part_chunks;
  const int end = min(static_cast<int>(kpad / 32), begin + part_chunks);
  const int zeros = u == PW - 1 ? 32 - S * PW : 0;
  uint32_t c[S] = {}, n = 0;
  for (int ch = begin + threadIdx.x; ch < end; ch += 128) {
    const int64_t q0 = 32 * static_cast<int64_t>(ch);
    uint8_t *const dst = rows + 16 * ch;
    uint32_t in[8] = {};
    if (i < n_v && q0 < n_f) {
      const uint4 v0 = __ldg(reinterpret_cast<const uint4 *>(src + q0));
      in[0] = v0.x, in[1] = v0.y, in[2] = v0.z, in[3] = v0.w;
      if (q0 + 16 < n_f) {  // the row holds ld >= n_f bytes, ld a multiple of 16
        const uint4 v1 = __ldg(reinterpret_cast<const uint4 *>(src + q0 + 16));
        in[4] = v1.x, in[5] = v1.y, in[6] = v1.z, in[7] = v1.w;
      }
    }
    uint32_t out[S][4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      uint32_t x = pack_nibbles(in[2 * e] & 0x0F0F0F0Fu, in[2 * e + 1] & 0x0F0F0F0Fu);
      uint32_t y = pack_nibbles((in[2 * e] >> 4) & 0x0F0F0F0Fu, (in[2 * e + 1] >> 4) & 0x0F0F0F0Fu);
      // Bit 3 of a nibble: it is at least S (or 8).
      const uint32_t add = (8u - S) * 0x11111111u;
      uint32_t ge = (x | y | ((x & 0x77777777u) + add) | ((y & 0x77777777u) + add)) & 0x88888888u;
      const int64_t left = i < n_v ? n_f - q0 - 8 * e : 0;
      if (left < 8) ge |= left > 0 ? 0x88888888u << (4 * left) : 0x88888888u;
      const uint32_t gone = (ge << 1) - (ge >> 3);  // nibble 15 per missing entry
      x |= gone;
      y |= gone;
      n += 8 - __popc(ge);
#pragma unroll
      for (int a = 0; a < S; ++a) {
        const uint32_t lo = a < 4 ? 2u << (8 * a) : 0u, hi = a < 4 ? 0u : 2u << (8 * (a - 4));
        const uint32_t b0 = lookup_nibbles(lo, hi, x) + lookup_nibbles(lo, hi, y);
        const uint32_t b1 = lookup_nibbles(lo, hi, x >> 16) + lookup_nibbles(lo, hi, y >> 16);
        out[a][e] = pack_nibbles(b0, b1);
        c[a] += __popc(out[a][e]) + __popc(out[a][e] & 0x44444444u);
      }
    }
#pragma unroll
    for (int a = 0; a < S; ++a)
      *reinterpret_cast<uint4 *>(dst + a * row_bytes) =
          make_uint4(out[a][0], out[a][1], out[a][2], out[a][3]);
    for (int r = 0; r < zeros; ++r)
      *reinterpret_cast<uint4 *>(dst + (S + r) * row_bytes) = make_uint4(0u, 0u, 0u, 0u);
  }
  if (w == nullptr || i >= n_v) return;  // the whole block
  __shared__ uint32_t part[4][S + 1];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    n += __shfl_xor_sync(0xffffffffu, n, o);
#pragma unroll
    for (int a = 0; a < S; ++a) c[a] += __shfl_xor_sync(0xffffffffu, c[a], o);
  }
  if ((threadIdx.x & 31) == 0) {
    part[threadIdx.x >> 5][S] = n;
#pragma unroll
    for (int a = 0; a < S; ++a) part[threadIdx.x >> 5][a] = c[a];
  }
  __syncthreads();
  if (threadIdx.x < S) {
    const int a = threadIdx.x;
    const uint32_t total = part[0][S] + part[1][S] + part[2][S] + part[3][S];
    const uint32_t sum = part[0][a] + part[1][a] + part[2][a] + part[3][a];
    const double f = total > 0 ? static_cast<double>(sum) / (2.0 * static_cast<double>(total)) : 0.0;
    w[i * S + a] = static_cast<float>(1.0 - gamma * f);
  }
}

// ---------------------------------------------------------------- CCC from stored tallies

// One thread per pair: Eq. 3 over the pair's s x s table, the same operations
// as the tally kernel's epilogue.
__global__ void k_metric2_multi(const int32_t *__restrict__ tally, const float *__restrict__ w,
                                int64_t n_v, int s, float gamma, int32_t norm,
                                float *__restrict__ ccc) {
  const int64_t npairs = n_v * (n_v - 1) / 2;
  const int ss = s * s;
  for (int64_t p = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; p < npairs;
       p += static_cast<int64_t>(gridDim.x) * blockDim.x) {
    // Row i of pair p: the largest i with pair_index(i, i + 1) <= p.
    int64_t i = static_cast<int64_t>(
        (2.0 * n_v - 1.0 - sqrt((2.0 * n_v - 1.0) * (2.0 * n_v - 1.0) - 8.0 * static_cast<double>(p))) / 2.0);
    if (i < 0) i = 0;
    while (i > 0 && i * (2 * n_v - i - 1) / 2 > p) --i;
    while ((i + 1) * (2 * n_v - i - 2) / 2 <= p) ++i;
    const int64_t j = p - i * (2 * n_v - i - 1) / 2 + i + 1;
    const int32_t *t = tally + p * ss;
    float *out = ccc + p * ss;
    int32_t n4 = 0;
    for (int x = 0; x < ss; ++x) n4 += t[x];
    if (n4 == 0) {
      for (int x = 0; x < ss; ++x) out[x] = 0.f;
      continue;
    }
    const float d = static_cast<float>(n4);
    const float inv = rcp_count(d);
    for (int a = 0; a < s; ++a) {
      float wi;
      if (norm == CCC_NORM_PERSNP) {
        wi = w[i * s + a];
      } else {
        int32_t rs = 0;
        for (int b = 0; b < s; ++b) rs += t[a * s + b];
        wi = joint_factor(static_cast<float>(rs), d, inv, gamma);
      }
      for (int b = 0; b < s; ++b) {
        const float r = static_cast<float>(t[a * s + b]);
        if (norm == CCC_NORM_PERSNP) {
          out[a * s + b] = __fmul_rn(__fmul_rn(__fmul_rn(r, inv), wi), w[j * s + b]);
        } else {
          int32_t cs = 0;
          for (int x = 0; x < s; ++x) cs += t[x * s + b];
          out[a * s + b] = __fmul_rn(__fmul_rn(div_count(r, d, inv), wi),
                                     joint_factor(static_cast<float>(cs), d, inv, gamma));
        }
      }
    }
  }
}

}  // namespace

int64_t multi_rows_pad(int64_t n_v, int s) {
  const int64_t quarters = (n_v + snps_per_quarter(s) - 1) / snps_per_quarter(s);
  return (32 * quarters + 255) / 256 * 256;
}

int launch_multi_counts(const uint8_t *geno, int64_t n_f, int64_t n_v, int64_t ld, int s,
                        int32_t *counts, float *w, double gamma, cudaStream_t st) {
  if (n_v < 1) return CCC_OK;
  const unsigned blocks = static_cast<unsigned>((n_v + 7) / 8);
  switch (s) {
#define CCC_MULTI_COUNTS(S)                                                                   \
  case S:                                                                                    \
    k_multi_counts<S><<<blocks, 256, 0, st>>>(geno, n_f, n_v, ld, counts, w, gamma);       \
    break;
    CCC_MULTI_COUNTS(2) CCC_MULTI_COUNTS(3) CCC_MULTI_COUNTS(4) CCC_MULTI_COUNTS(5)
    CCC_MULTI_COUNTS(6) CCC_MULTI_COUNTS(7) CCC_MULTI_COUNTS(8) CCC_MULTI_COUNTS(9)
    CCC_MULTI_COUNTS(10) CCC_MULTI_COUNTS(11) CCC_MULTI_COUNTS(12) CCC_MULTI_COUNTS(13)
    CCC_MULTI_COUNTS(14) CCC_MULTI_COUNTS(15)
#undef CCC_MULTI_COUNTS
    default:
      return CCC_EINVAL;
  }
  return note_launch();
}

int launch_multi_factors(const int32_t *counts, int64_t n_v, int s, float *w, double gamma,
                         cudaStream_t st) {
  const int64_t n = n_v * s;
  if (n < 1) return CCC_OK;
  k_multi_factors<<<static_cast<unsigned>((n + 255) / 256), 256, 0, st>>>(counts, n_v, s, w, gamma);
  return note_launch();
}

int launch_multi_unpack(const uint8_t *geno, int64_t n_f, int64_t n_v, int64_t ld, int s,
                        uint8_t *op, int64_t kpad, int64_t rows_pad, cudaStream_t st, bool fp4,
                        float *w, double gamma) {
  const int64_t quarters = rows_pad / 32;
  if (fp4) {
    if (kpad % 256 != 0 || s < 2 || s > 8) return CCC_EINVAL;
    const int64_t markers = quarters * snps_per_quarter(s);
    if (markers < 1) return CCC_OK;
    if (markers > 0x7FFFFFFFLL) return CCC_ERANGE;
    // Without factors (tallies alone, JOINT) nothing is summed over a row, so few
    // markers' rows are cut into parts of whole 4,096-individual steps, 16 blocks
    // per SM in all.  GB300, us per call, a block per row / in parts (the call
    // with factors, always a block per row): 100 x 1,000,000, s = 2: 1391 / 1219
    // (1390), s = 8: 1565 / 1293 (1564); 40 x 300,000, s = 8: 476 / 382 (474);
    // 300 x 16,384, s = 4: 41 / 39; 8 or 32 blocks per SM within 1%.
    const int64_t chunks = kpad / 32, steps = (chunks + 127) / 128;
    const int64_t want = w == nullptr ? (152 * 16 + markers - 1) / markers : 1;
    const int64_t part_steps = (steps + want - 1) / want;
    const int part_chunks = static_cast<int>(128 * part_steps);
    const dim3 grid(static_cast<unsigned>(markers),
                    static_cast<unsigned>((steps + part_steps - 1) / part_steps), 1);
    auto go = [&](auto kernel) {
      kernel<<<grid, 128, 0, st>>>(geno, n_f, n_v, ld, op, kpad, w, gamma, part_chunks);
      return note_launch();
    };
    switch (s) {
      case 2: return go(k_multi_unpack_e2m1<2>);
      case 3: return go(k_multi_unpack_e2m1<3>);
      case 4: return go(k_multi_unpack_e2m1<4>);
      case 5: return go(k_multi_unpack_e2m1<5>);
      case 6: return go(k_multi_unpack_e2m1<6>);
      case 7: return go(k_multi_unpack_e2m1<7>);
      default: return go(k_multi_unpack_e2m1<8>);
    }
  }
  if (w != nullptr) {
    const int rc = launch_multi_counts(geno, n_f, n_v, ld, s, nullptr, w, gamma, st);
    if (rc != CCC_OK) return rc;
  }
  const int64_t total = quarters * (kpad / 16);
  if (total < 1) return CCC_OK;
  const int64_t blocks = (total + 255) / 256 < 152 * 16 ? (total + 255) / 256 : 152 * 16;
  k_multi_unpack<<<static_cast<unsigned>(blocks), 256, 0, st>>>(geno, n_f, n_v, ld, s, op, kpad,
                                                               quarters);
  return note_launch();
}

int launch_tally2_multi(int s, int64_t n_v, const float *w, int32_t *tally, float *out_ccc,
                        int32_t *status, float gamma, int32_t norm, int32_t group, const uint8_t *op,
                        int64_t rows_pad, int64_t kpad, int num_sms, cudaStream_t st,
                        int64_t i_begin, int64_t i_end, int64_t pair0, int split, bool fp4) {
  if (n_v < 2) return CCC_OK;
  if (fp4) {
    // e2m1 rows of kpad / 2 bytes; 256 x 192 tiles, no K split; s <= 8.
    if (split > 1 || s > 8 || kpad % 256 != 0) return CCC_EINVAL;
    MultiMaps maps;
    if (!tc::make_operand_map(&maps.m[0], op, rows_pad, kpad / 2, tcp::BMH) ||
        !tc::make_operand_map(&maps.m[1], op, rows_pad, kpad / 2, kMultiRectNB / 2))
      return CCC_ECUDA;
    MultiArgs a4{n_v, w, tally, out_ccc, status, gamma, norm, i_begin, i_end, pair0};
    a4.out_len = checked_out_len(pairs_in_rows(n_v, i_begin, i_end));
    const int nkb4 = static_cast<int>((kpad / 2) / tcp::BK);
    switch (s) {
      case 2: return launch_tally2_multi_fp4_s<2>(maps, a4, group, nkb4, num_sms, st);
      case 3: return launch_tally2_multi_fp4_s<3>(maps, a4, group, nkb4, num_sms, st);
      case 4: return launch_tally2_multi_fp4_s<4>(maps, a4, group, nkb4, num_sms, st);
      case 5: return launch_tally2_multi_fp4_s<5>(maps, a4, group, nkb4, num_sms, st);
      case 6: return launch_tally2_multi_fp4_s<6>(maps, a4, group, nkb4, num_sms, st);
      case 7: return launch_tally2_multi_fp4_s<7>(maps, a4, group, nkb4, num_sms, st);
      case 8: return launch_tally2_multi_fp4_s<8>(maps, a4, group, nkb4, num_sms, st);
      default: return CCC_EINVAL;
    }
  }
  if (s > 8) return launch_tally2_multi_wide(s, n_v, w, tally, out_ccc, status, gamma, norm, group,
                                             op, rows_pad, kpad, num_sms, st, i_begin, i_end, pair0,
                                             split);
  CUtensorMap tm;
  if (!tc::make_operand_map(&tm, op, rows_pad, kpad, tcp::BMH)) return CCC_ECUDA;
  MultiArgs a{n_v, w, tally, out_ccc, status, gamma, norm, i_begin, i_end, pair0};
  a.out_len = checked_out_len(pairs_in_rows(n_v, i_begin, i_end));
  // 256-row blocks holding a SNP (rows_pad has exactly these).
  const int64_t nB = rows_pad / 256;
  const int nkb = static_cast<int>(kpad / tcp::BK);
  if (split > 1) {
    switch (s) {
      case 2: return launch_tally2_multi_split_s<2>(tm, a, nB, group, nkb, split, num_sms, st);
      case 3: return launch_tally2_multi_split_s<3>(tm, a, nB, group, nkb, split, num_sms, st);
      case 4: return launch_tally2_multi_split_s<4>(tm, a, nB, group, nkb, split, num_sms, st);
      case 5: return launch_tally2_multi_split_s<5>(tm, a, nB, group, nkb, split, num_sms, st);
      case 6: return launch_tally2_multi_split_s<6>(tm, a, nB, group, nkb, split, num_sms, st);
      case 7: return launch_tally2_multi_split_s<7>(tm, a, nB, group, nkb, split, num_sms, st);
      case 8: return launch_tally2_multi_split_s<8>(tm, a, nB, group, nkb, split, num_sms, st);
      default: return CCC_EINVAL;
    }
  }
  switch (s) {
    case 2: return launch_tally2_multi_s<2>(tm, a, nB, group, nkb, num_sms, st);
    case 3: return launch_tally2_multi_s<3>(tm, a, nB, group, nkb, num_sms, st);
    case 4: return launch_tally2_multi_s<4>(tm, a, nB, group, nkb, num_sms, st);
    case 5: return launch_tally2_multi_s<5>(tm, a, nB, group, nkb, num_sms, st);
    case 6: return launch_tally2_multi_s<6>(tm, a, nB, group, nkb, num_sms, st);
    case 7: return launch_tally2_multi_s<7>(tm, a, nB, group, nkb, num_sms, st);
    case 8: return launch_tally2_multi_s<8>(tm, a, nB, group, nkb, num_sms, st);
    default: return CCC_EINVAL;
  }
}

int launch_metric2_multi(const int32_t *tally, const float *w, int64_t n_v, int s, float gamma,
                         int32_t norm, float *out_ccc, cudaStream_t st) {
  const int64_t npairs = n_v * (n_v - 1) / 2;
  if (npairs < 1) return CCC_OK;
  const int64_t blocks = (npairs + 255) / 256 < 152 * 32 ? (npairs + 255) / 256 : 152 * 32;
  k_metric2_multi<<<static_cast<unsigned>(blocks), 256, 0, st>>>(tally, w, n_v, s, gamma, norm,
                                                                 out_ccc);
  return note_launch();
}

}  // namespace ccc
