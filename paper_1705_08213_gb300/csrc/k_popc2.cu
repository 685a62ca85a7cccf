// 2-way tallies by bitwise AND + population count on the CUDA cores: the plain
// form of Sec. 3.1, where every 2-bit entry is handled by word-wide bitwise
// operations and counted with a hardware population count.
//
// Each SNP is held as three bit planes per 64 entries (built by k_planes as
// P1 = first copy of allele 1, P2 = second copy, M = present; a hom 1 entry has
// both copies): H = P1 ^ P2 (het), A = P2 (hom 1), M.  With rho_1 = H + 2 A and
// rho_0 = 2M - rho_1:
//   r11 = sum_q rho_1,i rho_1,j = |Hi&Hj| + 2 (|Hi&Aj| + |Ai&Hj|) + 4 |Ai&Aj|
//   X   = sum_q rho_1,i m_j     = |Hi&Mj| + 2 |Ai&Mj|
//   Y   = sum_q m_i rho_1,j     = |Mi&Hj| + 2 |Mi&Aj|
//   Z   = sum_q m_i m_j         = |Mi&Mj|
//   r10 = 2X - r11,  r01 = 2Y - r11,  r00 = 4Z - 2X - 2Y + r11.
// Hi&Aj and Ai&Hj exclude each other, so one population count takes both.
//
// The population count runs at a quarter of the rate of the bitwise operations
// and is what bounds this form, so the products are not counted one by one:
// carry-save adders (sum x^y^z, carry majority, two 3-input operations each)
// add words of equal weight into a running word per weight, and only the
// carries out of the highest running word are counted (Harley and Seal).  Per
// four words and pair: 11 adders and 21 counts instead of 32 counts, which is
// where counts (84 cycles of an SM per 32 pairs) and bitwise operations (about
// 73) take about as long; three adders more for X, counted at weight 4 as r11
// is, took the registers of the second block per SM (6.0 ms).  GB300, 4,096 x
// 16,384: 8.23 -> 5.47 ms per call.
//
// Block tile: 32 x 32 SNPs of the upper triangle (J >= I), 256 threads, each
// thread 2 x 2 pairs (running words and counts take 16 registers per pair); the planes
// of both sides are staged in shared memory 8 words (512 entries) at a time.  A
// K split (gridDim.y parts) gives each block a range of words; since the four
// tallies are linear in the four sums, the parts add their partial tallies into
// the zeroed output with integer reductions, and the CCC values follow from the
// summed tallies (k_metric2).
#include "ccc_dev.cuh"
#include "ccc_launch.h"
#include "ccc_metric.cuh"
#include "popc_tiles.cuh"

namespace ccc {
namespace {

constexpr int TS = 32;       // SNPs per tile side
constexpr int KC = 8;        // 64-entry words per stage
constexpr int THREADS = 256;
constexpr int LDS = TS + 1;  // padded row (u64) against bank conflicts

// Planes H, A, M of 32 SNPs x KC words, 2 halves of 16 bytes per word.
__device__ __forceinline__ void load_stage(const uint64_t *__restrict__ planes, int64_t w64,
                                           int64_t kend, int64_t n_v, int64_t snp0, int64_t k0,
                                           uint64_t (*s)[KC][LDS]) {
#pragma unroll
  for (int l = threadIdx.x; l < TS * KC * 2; l += THREADS) {
    const int half = l & 1;
    const int word = (l >> 1) % KC;
    const int snp = (l >> 1) / KC;
    const int64_t i = snp0 + snp;
    const int64_t k = k0 + word;
    uint4 v = make_uint4(0u, 0u, 0u, 0u);
    if (i < n_v && k < kend) v = __ldg(reinterpret_cast<const uint4 *>(planes + (i * w64 + k) * 4) + half);
    const uint64_t lo = (static_cast<uint64_t>(v.y) << 32) | v.x;
    const uint64_t hi = (static_cast<uint64_t>(v.w) << 32) | v.z;
    if (half == 0) {
      s[0][word][snp] = lo ^ hi;
      s[1][word][snp] = hi;
    } else {
      s[2][word][snp] = lo;
    }
  }
}

__device__ __forceinline__ uint64_t sum3(uint64_t a, uint64_t b, uint64_t c) { return a ^ b ^ c; }
__device__ __forceinline__ uint32_t maj3(uint32_t a, uint32_t b, uint32_t c) {
  uint32_t r;
  asm("lop3.b32 %0, %1, %2, %3, 0xE8;" : "=r"(r) : "r"(a), "r"(b), "r"(c));
  return r;
}

// Carry-save adder: run takes the sum bits of run + a + b, the carries are returned.
__device__ __forceinline__ uint64_t csa(uint64_t &run, uint64_t a, uint64_t b) {
  const uint32_t lo = maj3(static_cast<uint32_t>(run), static_cast<uint32_t>(a), static_cast<uint32_t>(b));
  const uint32_t hi = maj3(static_cast<uint32_t>(run >> 32), static_cast<uint32_t>(a >> 32),
                           static_cast<uint32_t>(b >> 32));
  run = sum3(run, a, b);
  return (static_cast<uint64_t>(hi) << 32) | lo;
}

// One SNP's planes of a word.
struct Word {
  uint64_t h, a, m;
};

// The four sums of a pair: running words by weight, counts by weight.
struct PairSums {
  uint64_t r1 = 0, r2 = 0;          // r11, weights 1 and 2
  uint64_t x1 = 0, y1 = 0, z1 = 0;  // X, Y, Z
  uint32_t r4 = 0, x2 = 0, y2 = 0, z2 = 0;  // counts of weight 4, 2, 2, 2
  uint64_t rc;  // r11's weight-2 carry of the first two words of four

  // Words 2 half and 2 half + 1 of a group of four.
  __device__ __forceinline__ void add(int half, const Word &i0, const Word &j0, const Word &i1,
                                      const Word &j1) {
    const uint64_t c = csa(r1, i0.h & j0.h, i1.h & j1.h);
    r4 += __popcll(csa(r2, (i0.h & j0.a) | (i0.a & j0.h), (i1.h & j1.a) | (i1.a & j1.h)));
    r4 += __popcll(i0.a & j0.a) + __popcll(i1.a & j1.a);
    if (half == 0)
      rc = c;
    else
      r4 += __popcll(csa(r2, rc, c));
    x2 += __popcll(csa(x1, i0.h & j0.m, i1.h & j1.m));
    x2 += __popcll(i0.a & j0.m) + __popcll(i1.a & j1.m);
    y2 += __popcll(csa(y1, i0.m & j0.h, i1.m & j1.h));
    y2 += __popcll(i0.m & j0.a) + __popcll(i1.m & j1.a);
    z2 += __popcll(csa(z1, i0.m & j0.m, i1.m & j1.m));
  }
  __device__ __forceinline__ int32_t r11() const { return __popcll(r1) + 2 * __popcll(r2) + 4 * r4; }
  __device__ __forceinline__ int32_t x() const { return __popcll(x1) + 2 * x2; }
  __device__ __forceinline__ int32_t y() const { return __popcll(y1) + 2 * y2; }
  __device__ __forceinline__ int32_t z() const { return __popcll(z1) + 2 * z2; }
};

__global__ void __launch_bounds__(THREADS, 2)
    k_tally2_popc(const uint64_t *__restrict__ planes, int64_t w64, const Tally2Args args,
                  int64_t nB, int64_t t0, int64_t part_words) {
  __shared__ uint64_t sI[3][KC][LDS];
  __shared__ uint64_t sJ[3][KC][LDS];
  int64_t I, J;
  PopcTri{nB}.coords(t0 + blockIdx.x, I, J);
  const int64_t n_v = args.n_v;
  const int tx = threadIdx.x & 15;
  const int ty = threadIdx.x >> 4;
  PairSums acc[2][2];

  const int64_t kbeg = static_cast<int64_t>(blockIdx.y) * part_words;
  const int64_t kend = kbeg + part_words < w64 ? kbeg + part_words : w64;
  for (int64_t k0 = kbeg; k0 < kend; k0 += KC) {
    load_stage(planes, w64, kend, n_v, I * TS, k0, sI);
    load_stage(planes, w64, kend, n_v, J * TS, k0, sJ);
    __syncthreads();
#pragma unroll
    for (int k = 0; k < KC; k += 2) {
      Word wi[2][2], wj[2][2];  // [SNP][word]
#pragma unroll
      for (int x = 0; x < 2; ++x)
#pragma unroll
        for (int w = 0; w < 2; ++w) {
          wi[x][w] = Word{sI[0][k + w][ty + 16 * x], sI[1][k + w][ty + 16 * x], sI[2][k + w][ty + 16 * x]};
          wj[x][w] = Word{sJ[0][k + w][tx + 16 * x], sJ[1][k + w][tx + 16 * x], sJ[2][k + w][tx + 16 * x]};
        }
#pragma unroll
      for (int x = 0; x < 2; ++x)
#pragma unroll
        for (int y = 0; y < 2; ++y)
          acc[x][y].add((k >> 1) & 1, wi[x][0], wj[y][0], wi[x][1], wj[y][1]);
    }
    __syncthreads();
  }

#pragma unroll
  for (int x = 0; x < 2; ++x) {
    const int64_t i = I * TS + ty + 16 * x;
    if (i >= n_v || i < args.i_begin || i >= args.i_end) continue;
    const bool filter = args.hits != nullptr;
    const bool partial = gridDim.y > 1;  // K split: partial tallies, no CCC here
    const bool want_ccc = !partial && (filter || args.ccc != nullptr);
    float wi0 = 1.f, wi1 = 1.f;
    if (want_ccc && args.norm == CCC_NORM_PERSNP) {
      wi0 = __ldg(args.w + 2 * i);
      wi1 = __ldg(args.w + 2 * i + 1);
    }
    const int64_t row_base = i * (2 * n_v - i - 1) / 2 - i - 1 - args.pair0;
#pragma unroll
    for (int y = 0; y < 2; ++y) {
      const int64_t j = J * TS + tx + 16 * y;
      if (!(i < j && j < n_v)) continue;
      const int32_t r11 = acc[x][y].r11(), X = acc[x][y].x(), Y = acc[x][y].y(), Z = acc[x][y].z();
      const int32_t r10 = 2 * X - r11;
      const int32_t r01 = 2 * Y - r11;
      const int32_t r00 = 4 * Z - 2 * X - 2 * Y + r11;
      const int64_t pidx = row_base + j;
      if (!filter && !CCC_IN_BOUNDS(pidx, args.out_len, args.status)) continue;
      if (partial) {
        int32_t *t = args.tally + 4 * pidx;
        if (r00 != 0) atomicAdd(t + 0, r00);
        if (r01 != 0) atomicAdd(t + 1, r01);
        if (r10 != 0) atomicAdd(t + 2, r10);
        if (r11 != 0) atomicAdd(t + 3, r11);
        continue;
      }
      if (!filter) reinterpret_cast<int4 *>(args.tally)[pidx] = make_int4(r00, r01, r10, r11);
      if (want_ccc) {
        float wj0 = 1.f, wj1 = 1.f;
        if (args.norm == CCC_NORM_PERSNP) {
          const float2 wj = __ldg(reinterpret_cast<const float2 *>(args.w) + j);
          wj0 = wj.x;
          wj1 = wj.y;
        }
        const float4 cv =
            ccc2_values(r00, r01, r10, r11, wi0, wi1, wj0, wj1, args.norm, args.gamma);
        if (filter)
          filter_pair(args.hits, args.n_hits, args.cap, args.threshold, i, j, r00, r01, r10, r11,
                      cv);
        else
          reinterpret_cast<float4 *>(args.ccc)[pidx] = cv;
      }
    }
  }
}

// CCC values from stored tallies: one block per row i, threads over j > i.
__global__ void k_metric2(const int32_t *__restrict__ tally, const float *__restrict__ w,
                          int64_t n_v, float gamma, int32_t norm, float *__restrict__ ccc) {
  for (int64_t i = blockIdx.x; i < n_v; i += gridDim.x) {
    const int64_t row_base = i * (2 * n_v - i - 1) / 2 - i - 1;
    float wi0 = 1.f, wi1 = 1.f;
    if (norm == CCC_NORM_PERSNP) {
      wi0 = __ldg(w + 2 * i);
      wi1 = __ldg(w + 2 * i + 1);
    }
    for (int64_t j = i + 1 + threadIdx.x; j < n_v; j += blockDim.x) {
      const int4 r = __ldg(reinterpret_cast<const int4 *>(tally) + row_base + j);
      float wj0 = 1.f, wj1 = 1.f;
      if (norm == CCC_NORM_PERSNP) {
        const float2 wj = __ldg(reinterpret_cast<const float2 *>(w) + j);
        wj0 = wj.x;
        wj1 = wj.y;
      }
      reinterpret_cast<float4 *>(ccc)[row_base + j] =
          ccc2_values(r.x, r.y, r.z, r.w, wi0, wi1, wj0, wj1, norm, gamma);
    }
  }
}

}  // namespace

int64_t popc2_tiles(int64_t n_v) {
  const int64_t nB = (n_v + TS - 1) / TS;
  return nB * (nB + 1) / 2;
}

int launch_tally2_popc(const Tally2Args &a, const uint64_t *planes, int64_t w64, cudaStream_t s,
                       int split) {
  const int64_t nB = (a.n_v + TS - 1) / TS;
  int64_t t0;
  const int64_t tiles = PopcTri::in_rows(a.n_v, a.i_begin, a.i_end, TS, &t0);
  if (tiles <= 0) return CCC_OK;
  if (!popc_in_range(a.n_v, a.i_begin, a.i_end)) return CCC_ERANGE;
  // Parts of whole KC-word stages; split > 1 only with a.tally zeroed, no
  // thresholded output and the CCC values formed afterwards.
  const int64_t stages = (w64 + KC - 1) / KC;
  if (split < 1 || split > 65535 || (split > 1 && a.hits != nullptr)) return CCC_EINVAL;
  if (split > stages) split = static_cast<int>(stages);
  const int64_t part_words = (stages + split - 1) / split * KC;
  const int parts = static_cast<int>((w64 + part_words - 1) / part_words);
  return popc_launches(t0, tiles, [&](int64_t first, int64_t count) {
    const dim3 grid(static_cast<unsigned>(count), static_cast<unsigned>(parts > 0 ? parts : 1), 1);
    k_tally2_popc<<<grid, THREADS, 0, s>>>(planes, w64, a, nB, first, parts > 1 ? part_words : w64);
    return note_launch();
  });
}

int launch_metric2(const int32_t *tally, const float *w, int64_t n_v, float gamma, int32_t norm,
                   float *ccc, cudaStream_t s) {
  const int64_t blocks = n_v < 65536 ? n_v : 65536;
  if (blocks <= 0) return CCC_OK;
  k_metric2<<<static_cast<unsigned>(blocks), 256, 0, s>>>(tally, w, n_v, gamma, norm, ccc);
  return note_launch();
}

}  // namespace ccc
