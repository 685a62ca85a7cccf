// The multi-allelic 2-way tally kernel (k_multi.cu describes the method and
// the operand layout), templated on the number of states s.  k_multi.cu
// instantiates s = 2..8 and k_multi_wide.cu s = 9..15.
#pragma once

#include "ccc_launch.h"
#include "ccc_metric.cuh"
#include "tc_pipeline.cuh"
#include "tc_pipeline_pair.cuh"
#include "tc_sched.cuh"

#include <type_traits>

namespace ccc {
namespace {

constexpr int kMultiEpiWarps = 8;
constexpr int kMultiThreads = 64 + 32 * kMultiEpiWarps;

__host__ __device__ constexpr int snps_per_quarter(int s) { return 32 / s; }

struct MultiArgs {
  int64_t n_v;
  const float *w;   // [n_v][s] PERSNP factors, or null
  int32_t *tally;   // [npairs][s*s]
  float *ccc;       // [npairs][s*s], or null
  int32_t *status;
  float gamma;
  int32_t norm;
  // Row range of a phase: only pairs with i_begin <= i < i_end, stored at
  // pair_index(i, j) - pair0.
  int64_t i_begin, i_end, pair0;
  // Pairs the tally / ccc arrays hold (checked builds test every store index).
  int64_t out_len = int64_t(1) << 62;
};

// s consecutive values from registers to global memory (streaming stores).
template <int S>
__device__ __forceinline__ void store_row(int32_t *dst, const int32_t (&v)[S]) {
  if constexpr (S % 4 == 0) {
#pragma unroll
    for (int b = 0; b < S; b += 4)
      __stcs(reinterpret_cast<int4 *>(dst + b), make_int4(v[b], v[b + 1], v[b + 2], v[b + 3]));
  } else if constexpr (S % 2 == 0) {
#pragma unroll
    for (int b = 0; b < S; b += 2) __stcs(reinterpret_cast<int2 *>(dst + b), make_int2(v[b], v[b + 1]));
  } else {
#pragma unroll
    for (int b = 0; b < S; ++b) __stcs(dst + b, v[b]);
  }
}

template <int S>
__device__ __forceinline__ void store_row(float *dst, const float (&v)[S]) {
  if constexpr (S % 4 == 0) {
#pragma unroll
    for (int b = 0; b < S; b += 4)
      __stcs(reinterpret_cast<float4 *>(dst + b), make_float4(v[b], v[b + 1], v[b + 2], v[b + 3]));
  } else if constexpr (S % 2 == 0) {
#pragma unroll
    for (int b = 0; b < S; b += 2)
      __stcs(reinterpret_cast<float2 *>(dst + b), make_float2(v[b], v[b + 1]));
  } else {
#pragma unroll
    for (int b = 0; b < S; ++b) __stcs(dst + b, v[b]);
  }
}

// B blocks of NBQ quarters (32 operand rows each): 8 for the 256 x 256 e4m3
// tiles (TriSchedPair), 6 for the 256 x 192 FP4 tiles (RectSchedT; two
// 192-column accumulators and the scale factors fit the 512 TMEM columns).
constexpr int kMultiRectQ = 6;
constexpr int kMultiRectNB = 32 * kMultiRectQ;

template <int S, int NBQ = 8>
struct EpiMultiT {
  using Params = MultiArgs;
  static constexpr int PW = snps_per_quarter(S);
  static constexpr int CHUNKS = NBQ / 2;  // of a warp
  // FP4 tiles with S = 2 or odd S, e4m3 tiles with odd S, 10 or 14 (S = 2
  // does not fit beside their operand stages): the outputs leave through shared memory
  // (put_chunk).  Otherwise (direct) a lane stores its own row of the table in
  // pieces of 16 bytes (S = 4, 8, 12) or 8 (S = 6), which make up runs of S^2 words
  // anyway; the stage's traffic then costs more than it saves, because it
  // competes with the MMAs' operand reads.  GB300, us per call, direct / staged:
  //   S = 4, 10,000 x 16,384: 4536 / 4751; 3,000 x 4,000: 159 / 217
  //   S = 8, 2,000 x 8,000: 460 / 447; 3,000 x 2,000, JOINT: 668 / 824
  //   S = 6, 3,000 x 4,000: 487 / 461; 3,000 x 1,500, JOINT: 455 / 551
  // e4m3, JOINT, the sums over columns bound S > 7 at short K and the stage costs a
  // little there (S = 9, 2,000 x 1,500: 711 / 719; S = 11, 1,500 x 1,500: 657 / 761),
  // but at long K direct stores delay the operand loads (S = 11, 1,500 x 16,384:
  // 2744 / 2463; S = 13, 1,200 x 16,384: 1965 / 1661; S = 10, 1,500 x 1,500: 392 /
  // 423, x 16,384: 1266 / 1190; S = 15, 1,200 x 16,384: 2291 / 1738).
  // The rule goes by S alone.  Against direct stores with IEEE divisions every S gains
  // from the two together (S = 11, JOINT, 1,500 x 1,500: 1267 -> 761), but for e4m3 tiles
  // with S = 6 or 8, PERSNP, around 4,000 individuals (2,500 x 4,000: 426 -> 434, 638 ->
  // 649): the values come faster there and bunch the direct stores.
  // Loading all of a warp's chunks and releasing the accumulator before the first
  // is stored was slower for every S (S = 4, 10,000 x 16,384: 4601; S = 3, 3,000 x
  // 4,000: 175 for 168).
  static constexpr bool STAGED = NBQ == kMultiRectQ ? S == 2 || S % 2 == 1 : S % 2 == 1 || S == 10 || S == 14;
  // A marker i's words of one chunk, RUN = PW S^2, start RUN_LD words apart:
  // RUN_LD = S^2 (mod 32), so that the rows that the lanes (u, a) write at
  // u RUN_LD + a S fall on different banks (S = 3 on e4m3 tiles, 10, 15: as near to it as fits).
  static constexpr int SS = S * S;
  static constexpr int RUN = PW * SS;
  static constexpr int RUN_LD =
      NBQ == 8 && S == 3 ? 91 : S == 10 ? 308 : S == 15 ? 464 : SS % 32 + (RUN - SS % 32 + 31) / 32 * 32;
  static constexpr int W = S % 2 == 0 ? 4 : 1;  // words a lane stores
  static constexpr int NV = RUN / W;
  static constexpr int LPR = NV <= 16 ? 16 : 32;  // lanes of a run
  static constexpr int OUT_WORDS = STAGED ? (PW * RUN_LD + 3) / 4 * 4 : 0;
  // Behind them, the PERSNP factors w_j of the warp's NBQ / 2 quarters of markers.
  static constexpr int STAGE_BYTES_PER_WARP = (OUT_WORDS + CHUNKS * 32) * 4;
  using Sched = std::conditional_t<NBQ == 8, TriSchedPair,
                                   RectSchedT<8 * PW, NBQ * PW, 32 * NBQ>>;

  // The warps of column half h (c0 = h NC) take the chunks of 32 columns
  // [h NBQ / 2, (h + 1) NBQ / 2); chunk c is B quarter NBQ J + c.
  template <int NC>
  __device__ __forceinline__ static tcp::NoEarly early(const Params &, const Sched &, bool, int, int, int, int) {
    return {};
  }
  template <int NC, bool PRELOAD = false>
  __device__ static void tile(const Params &args, const Sched &sc, int rank, int quarter,
                              int lane, uint32_t t_base, uint32_t release_cluster_bar, int c0,
                              float *stage, tcp::NoEarly, int) {
    static_assert(!PRELOAD, "s-state tiles run on the two-accumulator pipeline");
    static_assert(NBQ % 2 == 0, "two column halves");
    const int cb = (c0 / NC) * CHUNKS;
    const int ce = cb + CHUNKS;
    float *const wstage = stage + OUT_WORDS;
    const int u = lane / S;
    const int a = lane - u * S;
    const int64_t n_v = args.n_v;
    // Accumulator lane = A row (i, a) of CTA `rank`'s 128 rows.
    const int64_t i = ((2 * static_cast<int64_t>(sc.I) + rank) * 4 + quarter) * PW + u;
    const bool row_ok = u < PW && i < n_v;
    const bool want_ccc = args.ccc != nullptr;
    const bool persnp = args.norm == CCC_NORM_PERSNP;
    float wi = 1.f;
    if (want_ccc && persnp && row_ok) wi = __ldg(args.w + i * S + a);
    const int64_t row_base = i * (2 * n_v - i - 1) / 2 - i - 1;  // pair index = row_base + j
    const int src0 = (u < PW ? u : 0) * S;                        // first lane of SNP i
    // w_j of the warp's markers jw0 .. (NBQ / 2 quarters), staged once per tile; every lane
    // then reads the same address (a broadcast) instead of its own global load per pair.
    const int64_t jw0 = (NBQ * static_cast<int64_t>(sc.J) + cb) * PW;
    if (want_ccc && persnp) {
      __syncwarp();  // the previous tile's reads are done
      for (int k = lane; k < CHUNKS * PW * S; k += 32) {
        const int64_t e = jw0 * S + k;
        wstage[k] = e < n_v * S ? __ldg(args.w + e) : 1.f;
      }
      __syncwarp();
    }
    // Row a of the table of (i, j0 + jl) as counts; the sums that its value needs.
    struct Sums {
      int32_t n4, rs, col[S];
    };
    auto row = [&](const uint32_t *v, int (&r)[S]) {
#pragma unroll
      for (int b = 0; b < S; ++b) r[b] = __float2int_rn(__uint_as_float(v[b]));
    };
    auto sums = [&](const int (&r)[S]) {
      Sums m;
      m.rs = 0;
#pragma unroll
      for (int b = 0; b < S; ++b) m.rs += r[b];
      // 4 n_ij = sum over the pair's table: the row sums of SNP i's s lanes.
      m.n4 = 0;
#pragma unroll
      for (int k = 0; k < S; ++k) m.n4 += __shfl_sync(0xffffffffu, m.rs, src0 + k);
      if (want_ccc && !persnp) {
#pragma unroll
        for (int b = 0; b < S; ++b) {
          m.col[b] = 0;
#pragma unroll
          for (int k = 0; k < S; ++k) m.col[b] += __shfl_sync(0xffffffffu, r[b], src0 + k);
        }
      }
      return m;
    };
    auto values = [&](const int (&r)[S], const Sums &m, const float *wjs, float (&cv)[S]) {
      const float d = m.n4 == 0 ? 1.f : static_cast<float>(m.n4);
      const float inv = rcp_count(d);
      if (persnp) {
#pragma unroll
        for (int b = 0; b < S; ++b)
          cv[b] = __fmul_rn(__fmul_rn(__fmul_rn(static_cast<float>(r[b]), inv), wi), wjs[b]);
      } else {
        const float wia = joint_factor(static_cast<float>(m.rs), d, inv, args.gamma);
#pragma unroll
        for (int b = 0; b < S; ++b) {
          const float wjb = joint_factor(static_cast<float>(m.col[b]), d, inv, args.gamma);
          cv[b] = __fmul_rn(__fmul_rn(div_count(static_cast<float>(r[b]), d, inv), wia), wjb);
        }
      }
    };
    // Each lane stores its own row of the chunk's tables.
    auto direct = [&](const uint32_t *v, int c) {
      // Column chunk c = 32 rows of the B block: its quarter c.
      const int64_t j0 = (NBQ * static_cast<int64_t>(sc.J) + c) * PW;
#pragma unroll
      for (int jl = 0; jl < PW; ++jl) {
        const int64_t j = j0 + jl;
        int r[S];
        row(v + jl * S, r);
        const Sums m = sums(r);
        if (!(row_ok && i < j && j < n_v && i >= args.i_begin && i < args.i_end)) continue;
        if (!CCC_IN_BOUNDS(row_base + j - args.pair0, args.out_len, args.status)) continue;
        const int64_t base = (row_base + j - args.pair0) * SS + a * S;
        store_row<S>(args.tally + base, r);
        if (!want_ccc) continue;
        float cv[S];
        values(r, m, wstage + ((c - cb) * PW + jl) * S, cv);
        store_row<S>(args.ccc + base, cv);
      }
    };
    auto staged = [&](const uint32_t *v, int c) {
      const int64_t i0 = i - u;
      const int64_t j0 = (NBQ * static_cast<int64_t>(sc.J) + c) * PW;
      __syncwarp();  // the previous reads of the stage are done
#pragma unroll
      for (int jl = 0; jl < PW; ++jl) {
        int r[S];
        row(v + jl * S, r);
        if (u < PW) put_row(reinterpret_cast<int *>(stage) + u * RUN_LD + jl * SS + a * S, r);
      }
      __syncwarp();
      put_chunk(args, i0, j0, lane, reinterpret_cast<const int *>(stage), args.tally);
      if (!want_ccc) return;
      __syncwarp();
#pragma unroll
      for (int jl = 0; jl < PW; ++jl) {
        int r[S];
        row(v + jl * S, r);
        const Sums m = sums(r);
        float cv[S];
        values(r, m, wstage + ((c - cb) * PW + jl) * S, cv);
        if (u < PW) put_row(stage + u * RUN_LD + jl * SS + a * S, cv);
      }
      __syncwarp();
      put_chunk(args, i0, j0, lane, stage, args.ccc);
    };
    for (int c = cb; c < ce; ++c) {
      uint32_t v[32];
      tmem_ld_32x32b_x32(t_base + c * 32, v);
      tmem_ld_wait();
      if (c == ce - 1) {
        tc_fence_before();
        mbar_arrive_cluster(release_cluster_bar);
      }
      if constexpr (STAGED)
        staged(v, c);
      else
        direct(v, c);
    }
  }

  // s consecutive words into the stage, as wide as their alignment allows.
  template <typename T>
  __device__ __forceinline__ static void put_row(T *dst, const T (&v)[S]) {
    constexpr int R = S % 2 == 0 ? 2 : 1;
    struct alignas(4 * R) Vec {
      T x[R];
    };
#pragma unroll
    for (int b = 0; b < S; b += R) {
      Vec t;
#pragma unroll
      for (int q = 0; q < R; ++q) t.x[q] = v[b + q];
      *reinterpret_cast<Vec *>(dst + b) = t;
    }
  }

  // One chunk of one array from the stage to global memory.  For each of the
  // warp's markers i the words of the pairs (i, j0 .. j0 + PW - 1) are contiguous
  // there, so the lanes store them side by side: 16 bytes each for even S (a
  // pair's S^2 words are then whole 16-byte units), words for odd S.  When each
  // lane stored its own row of the table, an instruction wrote 32 pieces of at
  // most 8 bytes in as many 128-byte lines as the warp has markers.
  // GB300, 3,000 markers, us per call, direct -> staged:
  //   4,000 individuals:  S = 2: 98 -> 85, 3: 235 -> 168, 5 (JOINT): 504 -> 426, 7: 979 -> 674
  //   16,384 individuals: S = 2: 174 -> 171, 3: 340 -> 338, 5: 977 -> 880, 7: 1984 -> 1744
  // e4m3, 4,096 individuals: 2,000 markers, S = 9: 1035 -> 628; 1,500, S = 11: 1029 -> 719;
  //   1,200, S = 13: 922 -> 487, S = 14: 706 -> 493, S = 15: 1487 -> 533; 4,000, S = 3: 461 -> 322
  template <typename T>
  __device__ __forceinline__ static void put_chunk(const MultiArgs &args, int64_t i0, int64_t j0,
                                                   int lane, const T *stage, T *out) {
    static_assert(PW % (32 / LPR) == 0 && (W == 1 || RUN_LD % 4 == 0), "whole runs and units");
    struct alignas(4 * W) Vec {
      T x[W];
    };
    const int64_t n_v = args.n_v;
    const int el = (lane & (LPR - 1)) * W;
    const int hi = n_v - j0 < PW ? static_cast<int>(n_v - j0) : PW;  // j < n_v
#pragma unroll 2
    for (int ul = LPR == 32 ? 0 : lane / LPR; ul < PW; ul += 32 / LPR) {
      const int64_t i = i0 + ul;
      const bool ok = i < n_v && i >= args.i_begin && i < args.i_end;
      const int64_t pair = i * (2 * n_v - i - 1) / 2 - i - 1 + j0 - args.pair0;  // (i, j0)
      // i < j: words from e0 on.
      const int e0 = i < j0 ? 0 : i - j0 < PW ? static_cast<int>(i + 1 - j0) * SS : RUN;
      const int e1 = ok ? hi * SS : 0;
      T *const dst = out + pair * SS;
      const T *const src = stage + ul * RUN_LD;
#pragma unroll
      for (int k = 0; k < (NV + LPR - 1) / LPR; ++k) {
        const int e = el + k * LPR * W;
        if (e >= e0 && e < e1 && CCC_IN_BOUNDS(pair + e / SS, args.out_len, args.status)) {
          const Vec t = *reinterpret_cast<const Vec *>(src + e);
          if constexpr (W == 4)
            stcs4(dst + e, t.x);
          else
            __stcs(dst + e, t.x[0]);
        }
      }
    }
  }
  __device__ __forceinline__ static void stcs4(int *dst, const int (&x)[4]) {
    __stcs(reinterpret_cast<int4 *>(dst), make_int4(x[0], x[1], x[2], x[3]));
  }
  __device__ __forceinline__ static void stcs4(float *dst, const float (&x)[4]) {
    __stcs(reinterpret_cast<float4 *>(dst), make_float4(x[0], x[1], x[2], x[3]));
  }
};

// Partial tallies of one K part (K split): each accumulator element is added
// into the zeroed tally array with an integer reduction.
template <int S>
struct EpiMultiSplit {
  using Params = MultiArgs;
  static constexpr int PW = snps_per_quarter(S);
  static constexpr int STAGE_BYTES_PER_WARP = 0;

  template <int NC>
  __device__ __forceinline__ static tcp::NoEarly early(const Params &, const SplitSchedPair &, bool, int, int, int, int) {
    return {};
  }
  template <int NC, bool PRELOAD = false>
  __device__ static void tile(const Params &args, const SplitSchedPair &sc, int rank, int quarter,
                              int lane, uint32_t t_base, uint32_t release_cluster_bar, int c0,
                              float *, tcp::NoEarly, int) {
    static_assert(!PRELOAD, "s-state tiles run on the two-accumulator pipeline");
    const int u = lane / S;
    const int a = lane - u * S;
    const int64_t n_v = args.n_v;
    const int64_t i = ((2 * static_cast<int64_t>(sc.I) + rank) * 4 + quarter) * PW + u;
    const bool row_ok = u < PW && i < n_v && i >= args.i_begin && i < args.i_end;
    const int64_t row_base = i * (2 * n_v - i - 1) / 2 - i - 1 - args.pair0;
    for (int c = c0; c < c0 + NC; ++c) {
      uint32_t v[32];
      tmem_ld_32x32b_x32(t_base + c * 32, v);
      tmem_ld_wait();
      if (c == c0 + NC - 1) {
        tc_fence_before();
        mbar_arrive_cluster(release_cluster_bar);
      }
      const int64_t j0 = ((2 * static_cast<int64_t>(sc.J) + (c >> 2)) * 4 + (c & 3)) * PW;
#pragma unroll
      for (int jl = 0; jl < PW; ++jl) {
        const int64_t j = j0 + jl;
        if (!(row_ok && i < j && j < n_v)) continue;
        if (!CCC_IN_BOUNDS(row_base + j, args.out_len, args.status)) continue;
        int32_t *dst = args.tally + (row_base + j) * (S * S) + a * S;
#pragma unroll
        for (int b = 0; b < S; ++b) {
          const int32_t r = __float2int_rn(__uint_as_float(v[jl * S + b]));
          if (r != 0) atomicAdd(dst + b, r);
        }
      }
    }
  }
};

template <int S>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kMultiThreads, 1)
    k_tally2_multi_split(const __grid_constant__ CUtensorMap tm, const MultiArgs args,
                         SplitSchedPair::Params sp, int nkb) {
  tcp::persistent_gemm_pair<SplitSchedPair, EpiMultiSplit<S>, kMultiEpiWarps>(&tm, sp, args, nkb,
                                                                               args.status);
}

template <int S>
using EpiMulti = EpiMultiT<S, 8>;

template <int S>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kMultiThreads, 1)
    k_tally2_multi(const __grid_constant__ CUtensorMap tm, const MultiArgs args,
                   TriSched::Params sp, int nkb) {
  tcp::persistent_gemm_pair<TriSchedPair, EpiMulti<S>, kMultiEpiWarps>(&tm, sp, args, nkb, args.status);
}

// FP4 (e2m1) operands: 256 x 192 tiles on SM pairs, two accumulators
// (tcp::persistent_gemm_pair with NB = 192); A through maps.m[0] (box 128 rows),
// B through maps.m[1] (box 96 rows).
struct MultiMaps {
  CUtensorMap m[2];
};

template <int S>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kMultiThreads, 1)
    k_tally2_multi_fp4(const __grid_constant__ MultiMaps maps, const MultiArgs args,
                       TriSched::Params sp, int nkb) {
  using Epi = EpiMultiT<S, kMultiRectQ>;
  tcp::persistent_gemm_pair<typename Epi::Sched, Epi, kMultiEpiWarps, false, true, kMultiRectNB>(
      maps.m, sp, args, nkb, args.status);
}

template <int S>
constexpr size_t multi_fp4_smem() {
  return tcp::smem_bytes_nb(kMultiRectNB, kMultiEpiWarps, EpiMultiT<S, kMultiRectQ>::STAGE_BYTES_PER_WARP);
}
template <int S>
constexpr size_t multi_smem() {
  static_assert(tcp::smem_bytes(kMultiEpiWarps, EpiMultiT<S, 8>::STAGE_BYTES_PER_WARP) <= 232448,
                "dynamic shared memory limit");
  return tcp::smem_bytes(kMultiEpiWarps, EpiMultiT<S, 8>::STAGE_BYTES_PER_WARP);
}

// Persistent grid size for a pair kernel of kMultiThreads threads.
template <typename K>
int multi_max_clusters(K kernel, int num_sms) {
  if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           static_cast<int>(tcp::SMEM_BYTES)) != cudaSuccess)
    return 0;
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeClusterDimension;
  attr.val.clusterDim.x = 2;
  attr.val.clusterDim.y = 1;
  attr.val.clusterDim.z = 1;
  cfg.gridDim = dim3(static_cast<unsigned>(num_sms), 1, 1);
  cfg.blockDim = dim3(kMultiThreads, 1, 1);
  cfg.dynamicSmemBytes = tcp::SMEM_BYTES;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  int n = 0;
  if (cudaOccupancyMaxActiveClusters(&n, kernel, &cfg) != cudaSuccess || n < 1) return 0;
  return n < num_sms / 2 ? n : num_sms / 2;
}

// K-split launch over the whole triangle of nB row blocks (split <= nkb).
template <int S>
int launch_tally2_multi_split_s(const CUtensorMap &tm, const MultiArgs &a, int64_t nB, int group,
                                int nkb, int split, int num_sms, cudaStream_t s) {
  static int max_clusters_dev[kMaxDevices] = {};
  const int dev_c = current_device();
  if (dev_c < 0) return CCC_ECUDA;
  int &max_clusters = max_clusters_dev[dev_c];
  if (max_clusters == 0) max_clusters = multi_max_clusters(k_tally2_multi_split<S>, num_sms);
  if (max_clusters == 0) return CCC_ECUDA;
  if (split < 1 || split > nkb) return CCC_EINVAL;
  SplitSchedPair::Params sp;
  sp.tri.nI = static_cast<int>(nB);
  sp.tri.nJ = sp.tri.nI;
  sp.tri.group = group > 0 ? group : 8;
  sp.tri.shift = 0;
  sp.tri.I0 = 0;
  sp.tri.I1 = sp.tri.nI;
  sp.split = split;
  sp.nkb = nkb;
  sp.tiles = nB * (nB + 1) / 2;
  const int64_t units = sp.tiles * split;
  if (units == 0) return CCC_OK;
  const int64_t clusters = units < max_clusters ? units : max_clusters;
  k_tally2_multi_split<S><<<static_cast<unsigned>(2 * clusters), kMultiThreads, tcp::SMEM_BYTES,
                            s>>>(tm, a, sp, nkb);
  return note_launch();
}

// FP4 launch over the rows [i_begin, i_end) (nI row blocks of 8 PW markers,
// nJ column blocks of 6 PW).
template <int S>
int launch_tally2_multi_fp4_s(const MultiMaps &maps, const MultiArgs &a, int group, int nkb,
                              int num_sms, cudaStream_t s) {
  using Epi = EpiMultiT<S, kMultiRectQ>;
  constexpr int64_t pi = 8 * static_cast<int64_t>(snps_per_quarter(S));
  constexpr int64_t pj = kMultiRectQ * static_cast<int64_t>(snps_per_quarter(S));
  TriSched::Params sp;
  sp.nI = static_cast<int>((a.n_v + pi - 1) / pi);
  sp.nJ = static_cast<int>((a.n_v + pj - 1) / pj);
  // Default tile order: groups of 32 column blocks (GB300, s = 4, 10,000 x
  // 16,384, per call: 4.81 ms against 4.86 with 16, 4.95 with 8, 4.84 with 64).
  sp.group = group > 0 ? group : 32;
  sp.shift = 0;
  sp.I0 = static_cast<int>(a.i_begin / pi);
  const int64_t iend = a.i_end < a.n_v ? a.i_end : a.n_v;
  sp.I1 = static_cast<int>((iend + pi - 1) / pi < sp.nI ? (iend + pi - 1) / pi : sp.nI);
  const int64_t tiles = rect_tiles<typename Epi::Sched>(sp.nI, sp.nJ, sp.I0, sp.I1);
  if (tiles <= 0) return CCC_OK;
  static int max_clusters_dev[kMaxDevices] = {};
  const int dev_c = current_device();
  if (dev_c < 0) return CCC_ECUDA;
  int &max_clusters = max_clusters_dev[dev_c];
  if (max_clusters == 0) {
    if (cudaFuncSetAttribute(k_tally2_multi_fp4<S>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             static_cast<int>(multi_fp4_smem<S>())) != cudaSuccess)
      return CCC_ECUDA;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = 2;
    attr.val.clusterDim.y = 1;
    attr.val.clusterDim.z = 1;
    cfg.gridDim = dim3(static_cast<unsigned>(num_sms), 1, 1);
    cfg.blockDim = dim3(kMultiThreads, 1, 1);
    cfg.dynamicSmemBytes = multi_fp4_smem<S>();
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, k_tally2_multi_fp4<S>, &cfg) != cudaSuccess || n < 1)
      return CCC_ECUDA;
    max_clusters = n < num_sms / 2 ? n : num_sms / 2;
  }
  const int64_t clusters = tiles < max_clusters ? tiles : max_clusters;
  k_tally2_multi_fp4<S><<<static_cast<unsigned>(2 * clusters), kMultiThreads, multi_fp4_smem<S>(),
                          s>>>(maps, a, sp, nkb);
  return note_launch();
}

template <int S>
int launch_tally2_multi_s(const CUtensorMap &tm, const MultiArgs &a, int64_t nB, int group, int nkb,
                          int num_sms, cudaStream_t s) {
  // Row blocks of 8 PW markers holding rows [i_begin, i_end).
  const int64_t per_block = 8 * static_cast<int64_t>(snps_per_quarter(S));
  const int64_t I0 = a.i_begin / per_block;
  const int64_t I1 = (a.i_end < a.n_v ? a.i_end : a.n_v) + per_block - 1;
  TriSched::Params sp;
  sp.nI = static_cast<int>(nB);
  sp.nJ = sp.nI;
  sp.group = group > 0 ? group : 8;
  sp.shift = 0;
  sp.I0 = static_cast<int>(I0);
  sp.I1 = static_cast<int>(I1 / per_block < nB ? I1 / per_block : nB);
  // Tiles of rows [I0, I1): sum of nB - I.
  const int64_t rows = sp.I1 > sp.I0 ? sp.I1 - sp.I0 : 0;
  const int64_t tiles = rows * nB - (static_cast<int64_t>(sp.I0) + sp.I1 - 1) * rows / 2;
  if (tiles <= 0) return CCC_OK;
  static int max_clusters_dev[kMaxDevices] = {};
  const int dev_c = current_device();
  if (dev_c < 0) return CCC_ECUDA;
  int &max_clusters = max_clusters_dev[dev_c];
  if (max_clusters == 0) {
    if (cudaFuncSetAttribute(k_tally2_multi<S>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             static_cast<int>(multi_smem<S>())) != cudaSuccess)
      return CCC_ECUDA;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = 2;
    attr.val.clusterDim.y = 1;
    attr.val.clusterDim.z = 1;
    cfg.gridDim = dim3(static_cast<unsigned>(num_sms), 1, 1);
    cfg.blockDim = dim3(kMultiThreads, 1, 1);
    cfg.dynamicSmemBytes = multi_smem<S>();
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, k_tally2_multi<S>, &cfg) != cudaSuccess || n < 1)
      return CCC_ECUDA;
    max_clusters = n < num_sms / 2 ? n : num_sms / 2;
  }
  const int64_t clusters = tiles < max_clusters ? tiles : max_clusters;
  k_tally2_multi<S><<<static_cast<unsigned>(2 * clusters), kMultiThreads, multi_smem<S>(), s>>>(tm, a, sp,
                                                                                          nkb);
  return note_launch();
}

}  // namespace
}  // namespace ccc
