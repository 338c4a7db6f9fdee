// k_oz_synth: the azimuthal stage of the float64 synthesis by the Ozaki
// scheme, over half of the longitudes.
//
//   out[row][k] = sum_t G[row][t] trig[t][k]     rows (shell, theta row), k = phi_k
//
// for up to four fields (Phi, g_r, g_theta, g_phi).  The cells mirror about
// phi = 0 (phi = pi on the polar grid): with C the sum over the cos slots and S
// over the sin slots, cell +phi is C + S and cell -phi is C - S, so the
// contractions run over half of the longitudes with half of the slots each.
//
// Digits (FormOzSynth): x = sum_s a_s 2^(-10 (s + 1)), five balanced base-1024
// digits |a_s| <= 512 (528 for one of G's), exact in fp16; rows of G scaled to |x| <= 1/2, the trig
// table to |y| <= 1/4.  The products of digit levels L = s + t
// <= 4 are kept, the dropped ones add up to below 2^-50 of the scales.  A class
// (the cos or sin slots; above l_max 31 those of even and of odd m apart) has at
// most 32 slots, and a level sum S_L of L <= 2 stays below 2^24 (528 times the sum of
// the trig digits, checked on the host) and accumulates exactly in fp32.  Level 4
// enters the accumulator of level 3 first, its trig digits scaled
// by 2^-10 (still exact in fp16): S_4 2^-10 is exact in fp32, and what the additions
// of level 3 round off it is some 2^-3 of a level-3 unit.  Level 3 itself is not
// checked: were all of its products of one sign and every digit of G at its largest, it
// could reach 1.15 2^24, where an addition rounds to 2 units.  So four
// accumulators hold a class, and
//   V = S_0 2^30 + S_1 2^20 + S_2 2^10 + round(S_3 + S_4 2^-10)
// is the class's sum in level-3 units, 2^-50 of the two rows' scales.  V_C + V_S
// and V_C - V_S are exact integers, at most (2 l_max + 1) 2^47 (below 2^53 up to
// l_max 31), and give the two cells' float64.
// (Six base-256 digits in bf16 with the whole row in one class: seven accumulators
// per cell, 26 products over 64 slots and all longitudes, 511 us on the 1-degree
// grid at l_max 25 with the gradient; this form 348; 180 x 360 polar grid of 300 zones: 377 and 260; l_max 40 on 61 x
// 185 cells, 317 zones: 412 and 217.)
//
// Schedule: a CTA pair (cluster of two, cta_group::2, M = 256 rows) takes a
// cell tile of 256 rows of one field, loads its G digits once and runs every tile
// of N = 48 columns against it, a class at a time: the class's trig digits (13.5
// KiB per CTA) come through a ring, its 30 MMAs fill the four accumulators of one
// of two TMEM buffers while the epilogue reads the other.  The G digits of a class
// are replaced as soon as its last MMAs of the cell tile are done, under the
// other class's; L2 is asked for them a cell tile ahead.
//   warp 0  lane 0: TMA producer (G tiles per class, the trig ring)
//   warp 1  TMEM allocation; in the even CTA lane 0 issues MMAs and commits
//   warps 2-13: epilogue, 16 columns x 32 rows each (lane quarter, column
//               group), values staged in shared memory 8 columns at a time so
//               that each store instruction writes 64-byte row runs
// Every wait is bounded (~2 s): on expiry the device error word gets
// YY_DEVERR_TIMEOUT and the CTA winds down, releasing TMEM.
#pragma once

namespace yy {

struct FormOzSynth {
  typedef __half elem;
  static constexpr int kKind = KIND_F16, kElem = 2;
  static constexpr int kSlices = 5;             // digits of G
  // trig slices: digits 0..3, then digits 0..4 scaled by 2^-10 (level 4)
  static constexpr int kTrig = 9, kTrigScaled = 4;
  static constexpr int kClassSlots = 32;        // slots of a class: one 64-byte swizzle row
};

constexpr int kOzBN = 48;                       // columns per tile (N of the MMA)
constexpr int kOzLevels = 4;                    // accumulators of a class
constexpr int kOzEpiWarps = 12;                 // lane quarters x column groups of 16
constexpr int kOzEpiCols = kOzBN / (kOzEpiWarps / 4);
constexpr int kOzThreads = 64 + 32 * kOzEpiWarps;
constexpr int kOzSlotA = kPairRows * kRowBytes;                      // one slice of a class: 8 KiB
constexpr int kOzSlotB = (kOzBN / 2) * kRowBytes;                    // 1.5 KiB
constexpr int kOzClassA = FormOzSynth::kSlices * kOzSlotA;           // 40 KiB
constexpr int kOzStageB = FormOzSynth::kTrig * kOzSlotB;             // 13.5 KiB
constexpr int kOzEpiPad = 8 + 2;                                     // staged row: 8 values + 2 pad
constexpr int kOzEpiWarpBytes = 32 * kOzEpiPad * 8 + 32 * 8;         // values + row pointers
template <int NCLS>
__host__ __device__ constexpr int oz_stages() { return NCLS == 2 ? 4 : 2; }
template <int NCLS>
constexpr int oz_synth_smem() {
  return 1024 + NCLS * kOzClassA + oz_stages<NCLS>() * kOzStageB + kOzEpiWarps * kOzEpiWarpBytes + 512;
}
static_assert(oz_synth_smem<2>() <= kSmemLimit && oz_synth_smem<4>() <= kSmemLimit, "k_oz_synth shared memory");
static_assert(kOzEpiCols == 16 && kOzSlotB % 512 == 0 && kOzLevels * kOzBN <= 256, "k_oz_synth tiles");

struct OzSynthJob {
  double *out0, *out1;          // rows r < out_split -> out0 + r ldo, else out1 + (r - out_split) ldo
  const int *cell_exp;          // per row: power of two of a unit V
};

struct OzSynthArgs {
  int cells, cell_tiles;        // valid G rows; tiles of 256 rows (pairs of 128)
  int col_tiles;                // tiles of kOzBN columns
  // column c is longitude first + c - shift (c >= shift: the folded columns; a
  // column before them repeats column shift's cells, so that runs of 8 columns
  // start on even cells) and its mirror n_phi - 1 - that; half folded columns
  int n_phi, first, shift, half;
  int a_rows, b_rows;           // rows of one slice in the stacked G / trig operands
  int out_split;
  long long ldo;
  int n_jobs;
  OzSynthJob job[4];
  int *err;
};

struct OzSynthMaps {
  CUtensorMap a[4], b;          // G digits per field (box 32 x 128), trig digits (box 32 x 24)
};

__device__ __forceinline__ void tma_prefetch_2d(const CUtensorMap *map, int x, int y) {
  asm volatile("cp.async.bulk.prefetch.tensor.2d.L2.global.tile [%0, {%1, %2}];" ::"l"((uint64_t)map), "r"(x),
               "r"(y)
               : "memory");
}

__device__ __forceinline__ long long mad_wide(int x, int y, long long z) {
  long long d;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(d) : "r"(x), "r"(y), "l"(z));
  return d;
}

// i64_ldexp out of line: rows whose results may leave the normal range
static __device__ __noinline__ double i64_ldexp_any(long long v, int e) { return i64_ldexp(v, e); }

// 8 staged values per row of the warp's 32 rows to cells start .. start + 7 of
// the output rows, those in [lo, hi).  Rows of even length (even start, 16-byte
// aligned rows): lanes 4 c' + e take values 2 e and 2 e + 1 of rows 8 q + c', whose
// addresses row4[q] the lane keeps for the cell tile.
__device__ __forceinline__ void oz_store_runs2(const double *ebuf, double *const (&row4)[4], int lane, int start, int lo,
                                               int hi) {
  const int e = lane & 3, at = start + 2 * e;
  const double *src = ebuf + (lane >> 2) * kOzEpiPad + 2 * e;
  if (start >= lo && start + 8 <= hi) {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const double2 val = *reinterpret_cast<const double2 *>(src + 8 * q * kOzEpiPad);
      if (row4[q] != nullptr) *reinterpret_cast<double2 *>(row4[q] + at) = val;
    }
  } else {
    const bool v0 = at >= lo && at < hi, v1 = at + 1 >= lo && at + 1 < hi;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const double2 val = *reinterpret_cast<const double2 *>(src + 8 * q * kOzEpiPad);
      if (row4[q] != nullptr && v0) row4[q][at] = val.x;
      if (row4[q] != nullptr && v1) row4[q][at + 1] = val.y;
    }
  }
}
__device__ __forceinline__ void oz_store_runs1(const double *ebuf, double *const *rowp, int lane, int start, int lo, int hi) {
  const int e = lane & 7, at = start + e;
  const bool ok = at >= lo && at < hi;
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const int r = 4 * q + (lane >> 3);
    double *orow = rowp[r];
    if (orow != nullptr && ok) orow[at] = ebuf[r * kOzEpiPad + e];
  }
}

template <int NCLS>
__global__ void __launch_bounds__(kOzThreads, 1)
k_oz_synth(const __grid_constant__ OzSynthMaps maps, const __grid_constant__ OzSynthArgs a) {
  pdl_wait();
  typedef FormOzSynth F;
  constexpr int KSTEPS = kRowBytes / 32;        // MMAs of K = 16 per class
  constexpr int BH = kOzBN / 2;                 // trig rows per CTA and tile
  constexpr int S = oz_stages<NCLS>();
  constexpr int NB = 2;                         // TMEM buffers, 256 columns apart
  constexpr int NC = kOzEpiCols;

  extern __shared__ uint8_t smem_raw[];
  uint8_t *smem = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint8_t *tileA = smem;                                     // [class][slice][128 rows][64 B]
  uint8_t *ringB = smem + NCLS * kOzClassA;                  // [stage][slice][24 rows][64 B]
  uint8_t *epi = ringB + S * kOzStageB;                      // epilogue staging
  uint64_t *bars = (uint64_t *)(epi + kOzEpiWarps * kOzEpiWarpBytes);
  uint64_t *a_full = bars, *a_empty = bars + NCLS;           // per class
  uint64_t *b_full = a_empty + NCLS, *b_empty = b_full + S;
  uint64_t *tfull = b_empty + S, *tempty = tfull + NB;       // [NB] each, tempty counted in the even CTA
  uint32_t *tmem_slot = (uint32_t *)(tempty + NB);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rank = (int)cluster_rank();
  const int pair = (int)blockIdx.x >> 1, n_pairs = (int)gridDim.x >> 1;
  const int total = a.cell_tiles * a.n_jobs;     // job-major cell tiles

  if (threadIdx.x == 0) {
    for (int c = 0; c < NCLS; ++c) {
      mbar_init(&a_full[c], 1);
      mbar_init(&a_empty[c], 1);
    }
    for (int s = 0; s < S; ++s) {
      mbar_init(&b_full[s], 1);
      mbar_init(&b_empty[s], 1);
    }
    for (int b = 0; b < NB; ++b) {
      mbar_init(&tfull[b], 1);
      mbar_init(&tempty[b], 2 * kOzEpiWarps);
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
      int gs = 0, s = 0, n_tiles = 0;
      uint32_t ph = 0;
      bool ok = true;
      auto load_b = [&](int ctile, int cls) {   // the trig digits of one class and column tile into the ring
        if (gs >= S && !mbar_wait(&b_empty[s], ph ^ 1, a.err)) return false;
        if (rank == 0) mbar_expect_tx(&b_full[s], 2u * (uint32_t)kOzStageB);
        const uint32_t fbar = mapa_rank(smem_u32(&b_full[s]), 0);
        const uint32_t base = smem_u32(ringB + s * kOzStageB);
#pragma unroll
        for (int p = 0; p < F::kTrig; ++p)
          tma_load_2d_pair(&maps.b, base + p * kOzSlotB, fbar, cls * F::kClassSlots,
                           p * a.b_rows + ctile * kOzBN + rank * BH);
        ++gs;
        if (++s == S) {
          s = 0;
          ph ^= 1;
        }
        return true;
      };
      for (int t = pair; t < total && ok; t += n_pairs, ++n_tiles) {
        const int arow = (2 * (t % a.cell_tiles) + rank) * kPairRows;
        const CUtensorMap *tmA = &maps.a[t / a.cell_tiles];
        for (int c = 0; c < NCLS && ok; ++c) {
          // the previous cell tile's MMAs of the class have completed before its digits are replaced
          if (n_tiles > 0 && !mbar_wait(&a_empty[c], (n_tiles - 1) & 1, a.err)) {
            ok = false;
            break;
          }
          if (rank == 0) mbar_expect_tx(&a_full[c], 2u * (uint32_t)kOzClassA);
          const uint32_t a_bar = mapa_rank(smem_u32(&a_full[c]), 0);
#pragma unroll
          for (int p = 0; p < F::kSlices; ++p)
            tma_load_2d_pair(tmA, smem_u32(tileA + (c * F::kSlices + p) * kOzSlotA), a_bar, c * F::kClassSlots,
                             p * a.a_rows + arow);
          // the first column tile's trig digits of the class behind them
          ok = load_b(0, c);
        }
        if (!ok) break;
        if (t + n_pairs < total) {
          const int tn = t + n_pairs;
          const CUtensorMap *tmN = &maps.a[tn / a.cell_tiles];
          const int nrow = (2 * (tn % a.cell_tiles) + rank) * kPairRows;
#pragma unroll
          for (int c = 0; c < NCLS; ++c)
#pragma unroll
            for (int p = 0; p < F::kSlices; ++p) tma_prefetch_2d(tmN, c * F::kClassSlots, p * a.a_rows + nrow);
        }
        for (int ctile = 1; ctile < a.col_tiles && ok; ++ctile)
          for (int c = 0; c < NCLS && ok; ++c) ok = load_b(ctile, c);
      }
      // every load has been consumed before this CTA leaves: the last
      // stages of the ring and the last G tile
      if (ok) {
        for (int i = max(0, gs - S); i < gs; ++i)
          if (!mbar_wait(&b_empty[i % S], (i / S) & 1, a.err)) break;
        for (int c = 0; c < NCLS && n_tiles > 0; ++c)
          if (!mbar_wait(&a_empty[c], (n_tiles - 1) & 1, a.err)) break;
      }
    }
  } else if (warp == 1) {
    if (rank == 0 && lane == 0) {
      const uint32_t idesc = instr_desc_pair<F>(kOzBN);
      int it = 0, s = 0, n_tiles = 0;
      uint32_t ph = 0;
      bool ok = true;
      for (int t = pair; t < total && ok; t += n_pairs, ++n_tiles) {
        for (int ctile = 0; ctile < a.col_tiles && ok; ++ctile) {
#pragma unroll 1
          for (int c = 0; c < NCLS; ++c, ++it) {
            if ((ctile == 0 && !mbar_wait_cluster(&a_full[c], n_tiles & 1, a.err)) ||
                !mbar_wait_cluster(&b_full[s], ph, a.err)) {
              ok = false;
              break;
            }
            const int b = it % NB;
            if (it >= NB && !mbar_wait_cluster(&tempty[b], ((it / NB) & 1) ^ 1, a.err)) {
              ok = false;
              break;
            }
            tc_fence_after();
            const uint32_t sa = smem_u32(tileA + c * kOzClassA), sb = smem_u32(ringB + s * kOzStageB);
            auto product = [&](int L, int ga, int gb, bool first) {   // G slice ga with trig slice gb
#pragma unroll
              for (int kk = 0; kk < KSTEPS; ++kk)
                mma_pair<F>(tmem_base + (uint32_t)(b * 256 + L * kOzBN), smem_desc(sa + ga * kOzSlotA + kk * 32),
                            smem_desc(sb + gb * kOzSlotB + kk * 32), idesc, (!first || kk != 0) ? 1u : 0u);
            };
            // level 4 (scaled trig digits), then level 3 onto it; levels 2, 1, 0
#pragma unroll 1
            for (int g = 0; g < F::kSlices; ++g) product(3, g, F::kTrigScaled + 4 - g, g == 0);
#pragma unroll 1
            for (int g = 0; g < 4; ++g) product(3, g, 3 - g, false);
#pragma unroll 1
            for (int L = 2; L >= 0; --L)
#pragma unroll 1
              for (int g = 0; g <= L; ++g) product(L, g, L - g, g == 0);
            mma_commit_pair(&tfull[b]);
            mma_commit_pair(&b_empty[s]);   // the trig stage is free once these MMAs complete
            if (ctile == a.col_tiles - 1) mma_commit_pair(&a_empty[c]);   // and the class's G digits after the last
            if (++s == S) {
              s = 0;
              ph ^= 1;
            }
          }
        }
      }
    }
  } else {
    // epilogue: lane quarter `quarter` of the TMEM lanes (32 rows), column
    // group `sub` (NC columns) of each tile
    const int quarter = warp & 3;
    const int sub = (warp - 2) >> 2;
    const uint32_t tempty_even = mapa_rank(smem_u32(&tempty[0]), 0);
    uint8_t *wbuf = epi + (size_t)(warp - 2) * kOzEpiWarpBytes;
    double *ebuf = reinterpret_cast<double *>(wbuf);                            // [32][kOzEpiPad]
    double **rowp = reinterpret_cast<double **>(wbuf + 32 * kOzEpiPad * 8);     // [32] output rows
    const bool vec = (a.ldo & 1) == 0;
    // cells the columns reach, plus and mirrored (a cell that is its own mirror: plus only)
    const int p_lo = a.first - a.shift, p_hi = a.first + a.half;
    const int last = a.n_phi - 1 - a.first;
    const int m_lo = last - a.half + 1 + (last - a.half + 1 == p_hi - 1 ? 1 : 0);
    const int m_hi = last + 1 + a.shift - (last == a.first ? 1 : 0);
    int it = 0;
    bool ok = true;
    for (int t = pair; t < total && ok; t += n_pairs) {
      const OzSynthJob &J = a.job[t / a.cell_tiles];
      const int ct = t % a.cell_tiles;
      const int cell = (2 * ct + rank) * kPairRows + quarter * 32 + lane;
      const bool cell_ok = cell < a.cells;
      const int ce = cell_ok ? J.cell_exp[cell] : 0;
      // the whole warp's rows stay in the normal range, a sum of 1 as well as one of four classes, up to 2^54
      const bool rows_ok = __all_sync(0xffffffffu, i64_ldexp_row_ok(ce) && (NCLS == 2 || i64_ldexp_row_ok(ce + 1)));
      __syncwarp();   // the previous tile's row pointers are no longer read
      rowp[lane] = !cell_ok ? nullptr
                   : (cell < a.out_split) ? J.out0 + (size_t)cell * a.ldo
                                          : J.out1 + (size_t)(cell - a.out_split) * a.ldo;
      __syncwarp();
      double *row4[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) row4[q] = rowp[8 * q + (lane >> 2)];
      for (int ctile = 0; ctile < a.col_tiles && ok; ++ctile) {
        long long vc[NC], vs[NCLS == 4 ? NC : 1];
        const int col0 = ctile * kOzBN + sub * NC;
#pragma unroll
        for (int c = 0; c < NCLS; ++c, ++it) {
          const int b = it % NB;
          if (!mbar_wait_cluster(&tfull[b], (it / NB) & 1, a.err)) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint32_t tcol = tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(b * 256 + sub * NC);
#pragma unroll
          for (int g = 0; g < NC; g += 8) {
            uint32_t u[kOzLevels][8];
#pragma unroll
            for (int L = 0; L < kOzLevels; ++L) tmem_ld8_async(tcol + (uint32_t)(L * kOzBN + g), u[L]);
            tmem_wait_ld();
            if (g + 8 >= NC) {
              // the accumulators are no longer needed
              tc_fence_before();
              __syncwarp();
              if (lane == 0) mbar_arrive_cluster_relaxed(tempty_even + (uint32_t)(b * sizeof(uint64_t)));
            }
            long long v[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) {
              v[j] = mad_wide(oz_int(u[2][j]), 1024, (long long)oz_int(u[3][j]));
              v[j] = mad_wide(oz_int(u[1][j]), 1 << 20, v[j]);
              v[j] = mad_wide(oz_int(u[0][j]), 1 << 30, v[j]);
            }
            if (c == 0) {
#pragma unroll
              for (int j = 0; j < 8; ++j) vc[g + j] = v[j];
            } else if (c < NCLS / 2) {
#pragma unroll
              for (int j = 0; j < 8; ++j) vc[g + j] += v[j];
            } else if (c < NCLS - 1) {
#pragma unroll
              for (int j = 0; j < 8; ++j) vs[NCLS == 4 ? g + j : 0] = v[j];
            } else {
              if constexpr (NCLS == 4) {
#pragma unroll
                for (int j = 0; j < 8; ++j) v[j] += vs[g + j];
              }
              // the cells +phi, then their mirrors (in reversed order), staged
              // and stored as row runs
              const int c0 = col0 + g;
              const int plus = a.first - a.shift + c0, minus = last + a.shift - c0 - 7;
#pragma unroll
              for (int sg = 0; sg < 2; ++sg) {
                if (rows_ok) {
                  // half of the values through the float64 pipe's conversion,
                  // half by integer formatting: the epilogue's issue slots are its
                  // limit, and with more the float64 pipe (six of eight: 356
                  // against 352 us, all: 379).  Values of four classes
                  // may reach 2^54.
#pragma unroll
                  for (int j = 0; j < 8; ++j) {
                    const long long V = sg ? vc[g + j] - v[j] : vc[g + j] + v[j];
                    ebuf[lane * kOzEpiPad + (sg ? 7 - j : j)] = (j & 1) == 0 ? i64_ldexp_row_cvt(V, ce)
                                                                : NCLS == 4  ? i64_ldexp_row54(V, ce)
                                                                             : i64_ldexp_row(V, ce);
                  }
                } else {
#pragma unroll
                  for (int j = 0; j < 8; ++j)
                    ebuf[lane * kOzEpiPad + (sg ? 7 - j : j)] = i64_ldexp_any(sg ? vc[g + j] - v[j] : vc[g + j] + v[j], ce);
                }
                __syncwarp();
                const int start = sg ? minus : plus, lo = sg ? m_lo : p_lo, hi = sg ? m_hi : p_hi;
                if (vec)
                  oz_store_runs2(ebuf, row4, lane, start, lo, hi);
                else
                  oz_store_runs1(ebuf, rowp, lane, start, lo, hi);
                __syncwarp();   // the staged values are read before the next ones overwrite them
              }
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
