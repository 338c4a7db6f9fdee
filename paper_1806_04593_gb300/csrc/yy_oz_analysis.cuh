// k_oz_analysis: the azimuthal stage of the float64 analysis by the Ozaki
// scheme.
//
//   F[row][t] = sum_k (rho w)[row][k] az[k][t]     rows (shell, theta row), t = 0 .. 2 l_max
//
// The cells are folded about the middle of the row first (k_rhow_ozaki): with
// E, O the sum and difference of a cell and its mirror, cos slots take E and sin slots
// O over half the columns, so the contraction is two of half the length and half
// the slots each (class 0: E with the cos slots, class 1: O with the sin
// slots, BN = 32 orders up to l_max 31, 64 up to 63).  Both operands are written as
// FormOzaki's six bf16 digit slices (ozaki_prepare_analysis).  Up to 292 cells a class is
// one fill whose level sums stay exact in fp32 (below 2^24); longer rows take two or
// three, which the epilogue adds in integers (ozaki_accumulate) before the one rounding to
// float64.  1-degree grid, 550 zones, l_max 25: 105 us (129 without the fold, with all 64
// slots over 320 columns); 300 zones of a 1-degree polar grid: 80 (92); 61 x 185 cells,
// 317 zones, l_max 40: 67 (93 in the general pair kernel, slots in tiles of 32).  The
// digits are read at 3.7 TB/s and the tensor cores are busy for half of the time: 387 row
// tiles on 76 pairs are six rounds of which the last is nearly empty.
//
// Schedule: each stage of a four-stage ring (three for BN = 64) holds one 32-wide K
// block of both operands: the six digit slices of 128 density rows (48 KiB) and three
// slices of the class's BN table rows (6 or 12 KiB) -- the even slices in the
// even CTA, the odd ones in the odd CTA, at the same offsets.  The table is
// re-read from L2 for every row tile.
//
// Two digit products per MMA: an MMA of N = 2 BN takes the first half of its B columns
// from the even CTA and the other half from the odd one, so with A = density slice s
// and the table slot holding slices u (even CTA) and u + 1 (odd CTA) it adds
// the products (s, u) and (s, u + 1) into the accumulators of levels s + u
// and s + u + 1, which lie side by side (level L at TMEM column BN L of its set).  The
// 26 products of levels <= 6 take 14 MMAs per 16-wide K step
// instead of 26 (two of them also add a level-7 product into a spare
// accumulator that is never read).  Since one MMA starts two accumulators that
// other MMAs continue, the MMAs always accumulate and the epilogue clears the
// accumulators (TMEM stores of zeros) after reading each fill, and once
// before the first.  Eight levels of 32 columns leave TMEM room for a set per class:
// while the epilogue reads one class's fill, the MMAs of the other run (103 us against
// 109 with one set).  With BN = 64 the classes take turns in the one set.
//   warp 0  lane 0: TMA producer
//   warp 1  TMEM allocation; in the even CTA lane 0 issues MMAs and commits
//   warps 2-17: epilogue, 8 or 16 orders x 32 rows each, results stored straight
//               from registers
// Every wait is bounded (~2 s): on expiry the device error word gets
// YY_DEVERR_TIMEOUT and the CTA winds down, releasing TMEM.
#pragma once

namespace yy {

constexpr int kOzAnSlotA = kPairRows * kRowBytes;                    // 8 KiB
constexpr int kOzAnStageA = FormOzaki::kPA * kOzAnSlotA;             // 48 KiB
constexpr int kOzAnLevels = FormOzaki::kAccs + 1;                    // levels 0..6 and the spare level 7
// BN: slots of a class, 32 or 64 (l_max up to 31, up to 63)
template <int BN>
struct OzAn {
  static constexpr int kSets = kPairTmemCols / (kOzAnLevels * BN);   // accumulator sets: 2 or 1
  static constexpr int kStages = BN == 32 ? 4 : 3;
  static constexpr int kSlotB = BN * kRowBytes;                      // one table slice of a class
  static constexpr int kStage = kOzAnStageA + FormOzaki::kPB / 2 * kSlotB;   // 54 or 60 KiB
  static constexpr int kSmem = 1024 + kStages * kStage + 512;
  static_assert(kSmem <= kSmemLimit && kSets >= 1 && kSlotB % 512 == 0, "k_oz_analysis tiles");
};
static_assert(FormOzaki::kPA == 6 && FormOzaki::kPB == 6, "k_oz_analysis pairs slices u, u + 1 of six");

// The paired products of one K step: density slice s with table slices
// u, u + 1 (u = 0, 2, 4), for s + u <= 6; 14 pairs cover the 26 products of
// levels <= 6 (and (2, 5), (4, 3) of level 7).
__host__ __device__ constexpr int oz_an_pairs() { return 14; }
__host__ __device__ constexpr int oz_an_s(int i) { return i < 6 ? i : (i < 11 ? i - 6 : i - 11); }
__host__ __device__ constexpr int oz_an_u(int i) { return i < 6 ? 0 : (i < 11 ? 2 : 4); }

struct OzAnalysisArgs {
  int cells, cell_tiles;        // valid density rows; tiles of 256 rows (pairs of 128)
  int cols;                     // valid slots (2 l_max + 1)
  int width;                    // columns of a class, a multiple of 16
  int kb_class, kb_fill;        // K blocks of a class; those of an accumulator fill
  int a_rows, b_rows;           // rows of one slice in the stacked operands
  long long ldo;                // output row stride (doubles)
  double *out;                  // [cells][ldo]
  const int *cell_exp;          // per row: power of two of a unit level-6 sum
  int *err;
};

struct OzAnalysisMaps {
  CUtensorMap a, b;             // density digits (box 32 x 128), table digits (box 32 x BN)
};

template <int BN>
__global__ void __launch_bounds__(kThreads, 1)
k_oz_analysis(const __grid_constant__ OzAnalysisMaps maps, const __grid_constant__ OzAnalysisArgs a) {
  pdl_wait();
  typedef FormOzaki F;
  static_assert(kRowBytes == 64, "two K steps of 16 per block");
  typedef OzAn<BN> P;
  constexpr int S = P::kStages;

  extern __shared__ uint8_t smem_raw[];
  uint8_t *smem = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint8_t *ring = smem;                                      // [stage]{[slice][128 rows][64 B], [slice][BN slots][64 B]}
  uint64_t *bars = (uint64_t *)(ring + S * P::kStage);
  uint64_t *full = bars, *empty = full + S;
  uint64_t *tfull = empty + S, *tempty = tfull + 2;          // per accumulator set; tempty counted in the even CTA
  uint32_t *tmem_slot = (uint32_t *)(tempty + 2);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rank = (int)cluster_rank();
  const int pair = (int)blockIdx.x >> 1, n_pairs = (int)gridDim.x >> 1;
  const int total = a.cell_tiles;
  const int fills = (a.kb_class + a.kb_fill - 1) / a.kb_fill;

  if (threadIdx.x == 0) {
    for (int s = 0; s < S; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int q = 0; q < 2; ++q) {
      mbar_init(&tfull[q], 1);
      mbar_init(&tempty[q], 2 * kEpiWarps);
    }
    fence_barrier_init();
  }
  if (warp == 1) {
    tmem_alloc_pair(tmem_slot, kPairTmemCols);
    tc_fence_before();
  }
  __syncthreads();
  cluster_sync();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;

  if (warp == 0) {
    if (lane == 0) {
      const uint32_t tx = 2u * (uint32_t)P::kStage;
      int gk = 0, s = 0;
      uint32_t ph = 0;
      bool ok = true;
      for (int t = pair; t < total && ok; t += n_pairs) {
        const int arow = (2 * t + rank) * kPairRows;
        for (int i = 0; i < 2 * a.kb_class; ++i, ++gk) {   // the sums' K blocks, then the differences'
          if (gk >= S && !mbar_wait(&empty[s], ph ^ 1, a.err)) {
            ok = false;
            break;
          }
          const int q = i >= a.kb_class ? 1 : 0, kb = i - q * a.kb_class;
          if (rank == 0) mbar_expect_tx(&full[s], tx);
          const uint32_t fbar = mapa_rank(smem_u32(&full[s]), 0);
          uint8_t *st = ring + s * P::kStage;
#pragma unroll
          for (int p = 0; p < F::kPA; ++p)
            tma_load_2d_pair(&maps.a, smem_u32(st + p * kOzAnSlotA), fbar, q * a.width + kb * 32, p * a.a_rows + arow);
          // this CTA's three table slices (rank, rank + 2, rank + 4), the class's slots
#pragma unroll
          for (int p = 0; p < F::kPB / 2; ++p)
            tma_load_2d_pair(&maps.b, smem_u32(st + kOzAnStageA + p * P::kSlotB), fbar, kb * 32,
                             (2 * p + rank) * a.b_rows + q * BN);
          if (++s == S) {
            s = 0;
            ph ^= 1;
          }
        }
      }
      if (ok)
        for (int i = max(0, gk - S); i < gk; ++i)
          if (!mbar_wait(&empty[i % S], (i / S) & 1, a.err)) break;
    }
  } else if (warp == 1) {
    if (rank == 0 && lane == 0) {
      const uint32_t idesc = instr_desc_pair<F>(2 * BN);
      int turn = 0, s = 0;   // turn: fills of either class
      uint32_t ph = 0;
      bool ok = true;
      for (int t = pair; t < total && ok; t += n_pairs, turn += fills) {
        for (int f = 0; f < 2 * fills && ok; ++f) {   // the sums' fills, then the differences'
          const int q = f >= fills ? 1 : 0, fq = f - q * fills, c0 = fq * a.kb_fill;
          // the epilogue has read the set's previous fill out of the accumulators
          // and cleared them (or cleared them before the first)
          if (!mbar_wait_cluster(&tempty[q % P::kSets], (uint32_t)((P::kSets == 2 ? turn + fq : 2 * turn + f) & 1), a.err)) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint32_t dq0 = tmem_base + (uint32_t)(q % P::kSets * kOzAnLevels * BN);
          const int n = min(a.kb_fill, a.kb_class - c0);
          for (int i = 0; i < n; ++i) {
            if (!mbar_wait_cluster(&full[s], ph, a.err)) {
              ok = false;
              break;
            }
            tc_fence_after();
            const uint32_t sa = smem_u32(ring + s * P::kStage);
            const uint32_t sb = sa + kOzAnStageA;
            // an MMA takes about as long as forming two descriptors from addresses:
            // their low words are one addition each here
            const uint32_t da0 = (uint32_t)smem_desc(sa), db0 = (uint32_t)smem_desc(sb);
            constexpr uint64_t kHigh = (1ull << 46 | 4ull << 61 | (uint64_t)(512 >> 4) << 32);
            auto step = [&](int kk) {
#pragma unroll
              for (int m = 0; m < oz_an_pairs(); ++m) {
                const int s_a = oz_an_s(m), u = oz_an_u(m);
                mma_pair<F>(dq0 + (uint32_t)((s_a + u) * BN), kHigh | (da0 + (uint32_t)((s_a * kOzAnSlotA + kk * 32) >> 4)),
                            kHigh | (db0 + (uint32_t)(((u / 2) * P::kSlotB + kk * 32) >> 4)), idesc, 1u);
              }
            };
            step(0);
            if (32 * (c0 + i) + 16 < a.width) step(1);   // else: the next class, or past the row
            mma_commit_pair(&empty[s]);
            if (++s == S) {
              s = 0;
              ph ^= 1;
            }
          }
          if (ok) mma_commit_pair(&tfull[q % P::kSets]);
        }
      }
    }
  } else {
    // epilogue: lane quarter `quarter` (32 rows), orders m0 .. m0 + NC - 1
    constexpr int NC = BN / (kEpiWarps / 4), G = NC / 8;   // 8 or 16, in groups of 8
    const int quarter = warp & 3;
    const int m0 = ((warp - 2) >> 2) * NC;
    const uint32_t tempty_even = mapa_rank(smem_u32(tempty), 0);
    const uint32_t tbase = tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)m0;
    // clear this warp's columns of the set's level accumulators, then release them
    auto clear_levels = [&](int set) {
#pragma unroll
      for (int L = 0; L < kOzAnLevels; ++L)
#pragma unroll
        for (int g = 0; g < G; ++g) tmem_zero8(tbase + (uint32_t)((set * kOzAnLevels + L) * BN + 8 * g));
      tmem_wait_st();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive_cluster_relaxed(tempty_even + (uint32_t)(set * sizeof(uint64_t)));
    };
#pragma unroll
    for (int set = 0; set < P::kSets; ++set) clear_levels(set);
    int turn = 0;   // fills of either class
    bool ok = true;
    for (int t = pair; t < total && ok; t += n_pairs, turn += fills) {
      const int cell = (2 * t + rank) * kPairRows + quarter * 32 + lane;
      const bool cell_ok = cell < a.cells;
      const int ce = cell_ok ? a.cell_exp[cell] : 0;
      // slot 2 m - 1 = cos, 2 m = sin of order m; slot 0 = cos of order 0
      const int t0 = 2 * m0;
      double *o = a.out + (size_t)cell * a.ldo + t0;
      double c[8];   // kSets == 2: the cos slots, until the sin slots are there
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        long long hi[G][8];
        float lo[G][8];
#pragma unroll
        for (int g = 0; g < G; ++g)
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            hi[g][j] = 0;
            lo[g][j] = 0.0f;
          }
        for (int f = 0; f < fills; ++f) {
          const int n = P::kSets == 2 ? turn + f : 2 * turn + q * fills + f;
          if (!mbar_wait_cluster(&tfull[q % P::kSets], (uint32_t)(n & 1), a.err)) {
            ok = false;
            break;
          }
          tc_fence_after();
#pragma unroll
          for (int g = 0; g < G; ++g)
            ozaki_accumulate(tbase + (uint32_t)(q % P::kSets * kOzAnLevels * BN + 8 * g), BN, hi[g], lo[g]);
          clear_levels(q % P::kSets);
        }
        if (!ok) break;
        if constexpr (P::kSets == 2) {
          double v[8];
          ozaki_finish(hi[0], lo[0], ce, v);
          if (q == 0) {
#pragma unroll
            for (int j = 0; j < 8; ++j) c[j] = v[j];
          } else if (cell_ok) {
            if (m0 == 0)
              v[0] = c[0];
            else if (t0 - 1 < a.cols)
              o[-1] = c[0];
            if ((a.ldo & 1) == 0 && t0 + 14 < a.cols) {
#pragma unroll
              for (int j = 0; j < 7; ++j) *reinterpret_cast<double2 *>(o + 2 * j) = make_double2(v[j], c[j + 1]);
              o[14] = v[7];
            } else {
#pragma unroll
              for (int j = 0; j < 8; ++j) {
                if (t0 + 2 * j < a.cols) o[2 * j] = v[j];
                if (j < 7 && t0 + 2 * j + 1 < a.cols) o[2 * j + 1] = c[j + 1];
              }
            }
          }
        } else {
#pragma unroll
          for (int g = 0; g < G; ++g) {
            double v[8];
            ozaki_finish(hi[g], lo[g], ce, v);
#pragma unroll
            for (int j = 0; j < 8; ++j) {
              const int m = m0 + 8 * g + j, slot = m == 0 ? 0 : q == 0 ? 2 * m - 1 : 2 * m;
              if (cell_ok && slot < a.cols && (m > 0 || q == 0)) o[slot - t0] = v[j];
            }
          }
        }
      }
    }
  }
  __syncthreads();
  cluster_sync();   // no CTA leaves while its peer may still reach its barriers or TMEM
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc_pair(tmem_base, kPairTmemCols);
  }
}

}  // namespace yy
