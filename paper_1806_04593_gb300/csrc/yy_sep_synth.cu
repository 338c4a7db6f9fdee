// Separable synthesis of the CUDA-core forms (YY_FP64, YY_FP32).  Per shell
// (patch p, radius i) and field (Phi, g_r, g_theta, g_phi):
//   theta stage  G[j][t] = sum_{l >= m} q[l^2 + t] P_f[j][l^2 + t]
//                (g_phi: the cos slot takes the sin coefficients and the sin
//                slot minus the cos ones, from d/dphi of cos / sin (m phi))
//   phi stage    out[j][k] = sum_t G[j][t] tr[t][k]
// with q the combined coefficients of the field (Q, Q_r, Q_t, Q_t).  Sums
// run from the top down (l from l_max, t from 2 l_max): the monopole (l = 0,
// t = 0) dominates Phi and g_r, and adding it last leaves one rounding of the
// large value instead of one per small term.
#include <math.h>

#include <algorithm>

#include "yy_internal.h"

namespace yy {
namespace {

struct SynthOut {
  double *o[4][2];     // field, patch
};

// ---------------------------------------------------------------------------
// float64
// ---------------------------------------------------------------------------
//
// The float64 pipe retires two operations per clock per SM, so the time is the
// number of float64 instructions and nothing else is near a limit: tables come
// through L1, and the symmetries of the cells cut the operations.
//  - theta: cell n_theta - 1 - j mirrors cell j.  K_lm P_l^m has the parity of
//    l + m, its theta derivative the opposite one: the sums over even and odd
//    l + m give both rows (E + O, E - O).
//  - g_phi: Q_t = -Q / r and the g_phi table is m / sin(theta) times Phi's, so
//    G_gphi[t] = (+-) m / (r sin theta) G_Phi[other slot of m].
//  - phi, every grid: the cells mirror about phi = 0 (pi on the polar grid), so
//    the cos slots' sum C and the sin slots' sum S give two cells (C + S, C - S).
//  - phi, where pi is a whole number of cells: cell phi also pairs with cell
//    pi - phi, where cos(m phi) takes the sign (-1)^m and sin(m phi) -(-1)^m;
//    the sums over even and odd m apart give up to four cells.
//  - phi, where pi / 2 is one too: pi / 2 -+ phi.  Even orders keep their functions
//    there up to signs that follow m mod 4, odd orders exchange cos and sin: sums
//    of even m apart by m mod 4 (one product per slot) and of odd m with both
//    functions (two per slot) give up to eight cells.
// The monopole (l = 0 of slot 0, then slot 0) is added last, to each row and to each
// cell apart: two roundings at the size of Phi and g_r.  (Inside the folded sums it
// took up to six: 4.7 units of 2^-53 at worst instead of 2, rms 1.05e-16 instead of 6.8e-17.)
// Columns and their images: AzFold.  On the 1-degree Yin-Yang grid 45 columns
// give the 270 cells: 16.4 float64 operations per output at l_max 25 instead of
// 51.  Measured there, 550 zones, with the gradient: 3.47 ms, against 12.9 ms for one
// thread per four cells without the folds; 2-degree grid, 200 zones, l_max 15: 254 us
// and 707.  (With the monopole inside the sums, 15.5 operations: 3.27 ms and 246 us, and
// with pi - phi alone, 18.7: 3.98 ms and 289 us.)
struct Synth64 {
  int n_r, n_theta, n_phi, lmax, n_lm, chunks;
  AzFold fold;
  const double *Q, *P, *dP, *tr, *isin, *r_edges;
  size_t qsz;
  SynthOut out;
};

// rows of G in shared memory: (field, row pair of the chunk, side), padded to
// the phi stage's groups of four (two with the quarter fold)
constexpr int kR64 = 4;
__host__ __device__ constexpr int rows64(int nf, int jp) { return (2 * nf * jp + kR64 - 1) / kR64 * kR64; }
// row stride of G: the theta stage's lanes write consecutive slots t, and two
// more values than the rows keep those writes off one another's banks
__host__ __device__ constexpr int stride_g(int rows) { return rows + 2; }

// The phi stage of two rows at one column, every fold in use.
__device__ __forceinline__ void phi_quarter(const Synth64 &a, const double *g, int ld, int c, double *const *dst) {
  constexpr int R = 2;
  // even m: cos and sin slots by m mod 4; odd m: cos slots with cos and with
  // sigma sin, sin slots with sin and with sigma cos (sigma = +1, -1 for m mod 4 = 1, 3)
  double c0[R] = {}, c2[R] = {}, s0[R] = {}, s2[R] = {}, cc[R] = {}, cs[R] = {}, ss[R] = {}, sc[R] = {};
  const int nb = a.fold.cols;
  const double *tr = a.tr + c;
  auto even = [&](int m, double (&x)[R], double (&y)[R]) {
    const double tc = tr[(size_t)(2 * m - 1) * nb], ts = tr[(size_t)(2 * m) * nb];
    const double2 u = *reinterpret_cast<const double2 *>(g + (size_t)(2 * m - 1) * ld);
    const double2 v = *reinterpret_cast<const double2 *>(g + (size_t)(2 * m) * ld);
    x[0] = fma(u.x, tc, x[0]);
    x[1] = fma(u.y, tc, x[1]);
    y[0] = fma(v.x, ts, y[0]);
    y[1] = fma(v.y, ts, y[1]);
  };
  auto odd = [&](int m, bool minus) {
    const double tc = tr[(size_t)(2 * m - 1) * nb], ts = tr[(size_t)(2 * m) * nb];
    const double xc = minus ? -tc : tc, xs = minus ? -ts : ts;
    const double2 u = *reinterpret_cast<const double2 *>(g + (size_t)(2 * m - 1) * ld);
    const double2 v = *reinterpret_cast<const double2 *>(g + (size_t)(2 * m) * ld);
    cc[0] = fma(u.x, tc, cc[0]);
    cc[1] = fma(u.y, tc, cc[1]);
    cs[0] = fma(u.x, xs, cs[0]);
    cs[1] = fma(u.y, xs, cs[1]);
    ss[0] = fma(v.x, ts, ss[0]);
    ss[1] = fma(v.y, ts, ss[1]);
    sc[0] = fma(v.x, xc, sc[0]);
    sc[1] = fma(v.y, xc, sc[1]);
  };
  int m = a.lmax;
  if ((m & 3) == 3) odd(m--, true);
  if ((m & 3) == 2) even(m--, c2, s2);
  if ((m & 3) == 1) odd(m--, false);
  for (; m > 0; m -= 4) {
    even(m, c0, s0);
    odd(m - 1, true);
    even(m - 2, c2, s2);
    odd(m - 3, false);
  }
  const int h = a.fold.half, first = a.fold.first, q = a.fold.quarter;
  const int kb = q - a.fold.odd - c, kc = q + c, kd = a.fold.partner - c;   // pi/2 - phi, pi/2 + phi, pi - phi
  const bool wb = kb != c && kb < h, wc = kc != kb && kc < h, wd = kd != kc && kd != c && kd < h;
#pragma unroll
  for (int r = 0; r < R; ++r) {
    double *o = dst[r];
    if (o == nullptr) continue;
    const double z = g[r];   // m = 0, added last
    const double e1 = c0[r] + c2[r], e2 = c0[r] - c2[r], f1 = s0[r] + s2[r], f2 = s0[r] - s2[r];
    auto put = [&](int col, double C, double S) {
      const int kp = first + col, km = a.n_phi - 1 - kp;
      o[kp] = z + (C + S);
      if (km != kp) o[km] = z + (C - S);
    };
    put(c, e1 + cc[r], f1 + ss[r]);
    if (wb) put(kb, e2 + cs[r], sc[r] - f2);
    if (wc) put(kc, e2 - cs[r], sc[r] + f2);
    if (wd) put(kd, e1 - cc[r], ss[r] - f1);
  }
}

template <int NF, bool QUARTER>
__global__ void __launch_bounds__(256, 3) k_synth_f64(const Synth64 a, int jp) {
  pdl_begin();
  extern __shared__ __align__(16) unsigned char smraw[];
  const int rp = rows64(NF, jp), ld = stride_g(rp), nt = 2 * a.lmax + 1;
  double *Gs = reinterpret_cast<double *>(smraw);                  // [nt][ld]
  double **dst = reinterpret_cast<double **>(Gs + (size_t)nt * ld);   // [rp] output row, NULL: none
  const int shell = blockIdx.x / a.chunks, chunk = blockIdx.x % a.chunks;
  const int p = shell / a.n_r, i = shell % a.n_r;
  const size_t n_ang = (size_t)a.n_theta * a.n_phi;
  for (int r = threadIdx.x; r < rp; r += blockDim.x) {
    const int f = r / (2 * jp), j = chunk * jp + (r % (2 * jp)) / 2, jm = a.n_theta - 1 - j;
    double *o = nullptr;
    if (f < NF && j <= jm && !((r & 1) && j == jm))
      o = a.out.o[f][p] + (size_t)i * n_ang + (size_t)((r & 1) ? jm : j) * a.n_phi;
    dst[r] = o;
  }
  // theta stage: one thread per (row pair, slot)
  const double inv_r = NF == 4 ? 1.0 / a.r_edges[i + 1] : 0.0;
  const double *q = a.Q + (size_t)shell * a.n_lm;
  for (int e = threadIdx.x; e < jp * nt; e += blockDim.x) {
    const int jj = e / nt, t = e % nt;
    const int j = chunk * jp + jj, m = (t + 1) / 2;
    const bool ok = 2 * j < a.n_theta;
    const size_t row = (size_t)(ok ? j : 0) * a.n_lm;
    // x: the terms of l_max's parity, y: of the other
    double x[3] = {0.0, 0.0, 0.0}, y[3] = {0.0, 0.0, 0.0};
    auto term = [&](int l, double (&s)[3]) {
      const int at = l * l + t;
      const double pv = a.P[row + at];
      s[0] = fma(q[at], pv, s[0]);
      if constexpr (NF == 4) {
        s[1] = fma(q[a.qsz + at], pv, s[1]);
        s[2] = fma(q[2 * a.qsz + at], a.dP[row + at], s[2]);
      }
    };
    const int least = t == 0 ? 1 : m;   // the monopole is added last
    int l = a.lmax;
    for (; l > least; l -= 2) {
      term(l, x);
      term(l - 1, y);
    }
    if (l == least) term(l, x);
    const bool odd = ((a.lmax + m) & 1) != 0;   // parity of x's terms
    double *g = Gs + (size_t)t * ld + 2 * jj;
    auto put = [&](double *at, double v0, double v1) { *reinterpret_cast<double2 *>(at) = make_double2(ok ? v0 : 0.0, ok ? v1 : 0.0); };
    auto sides = [&](const double *coef, double u, double v, double &plus, double &minus) {
      plus = u + v;
      minus = odd ? v - u : u - v;
      if (t == 0) {
        plus = fma(coef[0], a.P[row], plus);
        minus = fma(coef[0], a.P[row], minus);
      }
    };
    double up, um;
    sides(q, x[0], y[0], up, um);
    put(g, up, um);
    if constexpr (NF == 4) {
      double radial_p, radial_m;
      sides(q + a.qsz, x[1], y[1], radial_p, radial_m);
      put(g + 2 * jp, radial_p, radial_m);
      put(g + 4 * jp, x[2] + y[2], odd ? x[2] - y[2] : y[2] - x[2]);   // dP has the other parity
      const int to = t == 0 ? 0 : ((t & 1) ? t + 1 : t - 1);
      const double fac = (t & 1 ? 1.0 : -1.0) * m * a.isin[ok ? j : 0] * inv_r;
      put(Gs + (size_t)to * ld + 6 * jp + 2 * jj, fac * up, fac * um);
    }
  }
  if (rp > 2 * NF * jp)
    for (int e = threadIdx.x; e < nt * (rp - 2 * NF * jp); e += blockDim.x)
      Gs[(size_t)(e / (rp - 2 * NF * jp)) * ld + 2 * NF * jp + e % (rp - 2 * NF * jp)] = 0.0;
  __syncthreads();

  // phi stage: one thread per (group of four rows, or two, and column)
  const int nb = a.fold.cols;
  if constexpr (QUARTER) {
    for (int e = threadIdx.x; e < rp / 2 * nb; e += blockDim.x) phi_quarter(a, Gs + e / nb * 2, ld, e % nb, dst + e / nb * 2);
    return;
  }
  for (int e = threadIdx.x; e < rp / kR64 * nb; e += blockDim.x) {
    const int r0 = e / nb * kR64, c = e % nb;
    double ce[kR64], co[kR64], se[kR64], so[kR64];   // cos / sin slots of even / odd m
#pragma unroll
    for (int r = 0; r < kR64; ++r) ce[r] = co[r] = se[r] = so[r] = 0.0;
    const double *g = Gs + r0;
    const double *tr = a.tr + c;
    auto step = [&](int m, double (&cs)[kR64], double (&sn)[kR64]) {
      const double tc = tr[(size_t)(2 * m - 1) * nb], ts = tr[(size_t)(2 * m) * nb];
      const double *gc = g + (size_t)(2 * m - 1) * ld, *gs = gc + ld;
#pragma unroll
      for (int r = 0; r < kR64; r += 2) {
        const double2 u = *reinterpret_cast<const double2 *>(gc + r), v = *reinterpret_cast<const double2 *>(gs + r);
        cs[r] = fma(u.x, tc, cs[r]);
        cs[r + 1] = fma(u.y, tc, cs[r + 1]);
        sn[r] = fma(v.x, ts, sn[r]);
        sn[r + 1] = fma(v.y, ts, sn[r + 1]);
      }
    };
    int m = a.lmax;
    if (m & 1) step(m--, co, so);
    for (; m > 0; m -= 2) {
      step(m, ce, se);
      step(m - 1, co, so);
    }
    const int kp = a.fold.first + c, km = a.n_phi - 1 - kp;
    const int pc = a.fold.partner - c;
    const bool pair = a.fold.partner >= 0 && pc > c && pc < a.fold.half;
    const int kq = a.fold.first + pc;
#pragma unroll
    for (int r = 0; r < kR64; ++r) {
      double *o = dst[r0 + r];
      if (o == nullptr) continue;
      const double z = g[r];   // m = 0, added last
      const double C = ce[r] + co[r], S = se[r] + so[r];
      o[kp] = z + (C + S);
      if (km != kp) o[km] = z + (C - S);
      if (pair) {
        const double Cq = ce[r] - co[r], Sq = so[r] - se[r];
        o[kq] = z + (Cq + Sq);
        if (a.n_phi - 1 - kq != kq) o[a.n_phi - 1 - kq] = z + (Cq - Sq);
      }
    }
  }
}

// ---------------------------------------------------------------------------
// fp32
// ---------------------------------------------------------------------------
//
// Every output is one chain of fp32 multiply-adds over t (and every G one over
// l), in that order: no sum is split or folded.  Two kernels, G between them in
// tiles [field][tile][t][rows] of consecutive rows (shell, j): in one kernel the
// blocks' theta stages, bound by load latency, left the phi stage's registers
// idle (526 us on the 1-degree grid at l_max 25 with the gradient, against 55 +
// 342 us for the two; one thread per four cells with shared-memory G: 1909 us).
struct Synth32 {
  int n_shells, n_r, n_theta, n_phi, lmax, n_lm;
  int tile, tiles;                     // rows per tile, tiles per field
  int items;                           // (shell group, j) per block of the theta stage
  const float *Q, *P, *dP, *Qs, *tr;   // tables [mode][j]; tr [t][k]
  float *G;
  size_t qsz;
  SynthOut out;
};

// theta stage: a thread takes row j of S shells and the orders m and l_max - m
// (together l_max + 2 terms whatever m), both slots of an order and all fields,
// so a table value serves 2 S sums.  Lanes run over (shell group, j): the
// tables, [mode][j], load contiguously.  The coefficients of the block's groups
// are staged shell-minor, so that one 16-byte load serves the four shells.
constexpr int kS32 = 4, kThetaThreads = 128;

// groups of shells that a block of `items` (shell group, j) can meet
__host__ __device__ constexpr int theta_groups(int n_theta, int items) { return (items + n_theta - 2) / n_theta + 1; }

template <int NF>
__global__ void __launch_bounds__(kThetaThreads) k_theta32(const Synth32 a) {
  pdl_begin();
  constexpr int S = kS32, NQ = NF == 4 ? 3 : 1;   // g_phi uses the coefficients of g_theta
  extern __shared__ __align__(16) unsigned char smraw[];
  float *qs = reinterpret_cast<float *>(smraw);   // [group][l - m][NQ][cos, sin][S]
  const int groups = (a.n_shells + S - 1) / S, e0 = blockIdx.x * a.items;
  const int end = min(e0 + a.items, groups * a.n_theta);
  const int e = min(e0 + (int)threadIdx.x, end - 1);   // past the end: repeats the last
  const int g0 = e0 / a.n_theta, ng = min(theta_groups(a.n_theta, a.items), groups - g0);
  const int j = e % a.n_theta, group = e / a.n_theta, shell0 = group * S, nt = 2 * a.lmax + 1;
  size_t row[S];   // offset of the row's slot 0 in a field's tiles
#pragma unroll
  for (int s = 0; s < S; ++s) {
    const int r = (shell0 + s) * a.n_theta + j;
    row[s] = (size_t)(r / a.tile) * a.tile * nt + r % a.tile;
  }
  const size_t fsz = (size_t)a.tiles * a.tile * nt;
#pragma unroll 1
  for (int half = 0; half < 2; ++half) {
    const int m = half == 0 ? (int)blockIdx.y : a.lmax - (int)blockIdx.y;
    if (half == 1 && m <= (int)blockIdx.y) break;   // the middle order, or both done
    const int c = m == 0 ? 0 : 2 * m - 1, d = m == 0 ? 0 : 1;   // the cos slot; the sin slot is c + d
    const int nl = a.lmax - m + 1;
    if (half == 1) __syncthreads();   // the first order's coefficients are used up
    for (int x = threadIdx.x; x < ng * nl * NQ * S * 2; x += kThetaThreads) {
      // sin fastest, then l: neighbouring threads read both slots of a mode
      const int sn = x & 1, l = m + (x >> 1) % nl, y = (x >> 1) / nl, sh = y % S, f = y / S % NQ, gg = y / S / NQ;
      const int shell = min((g0 + gg) * S + sh, a.n_shells - 1);
      qs[(((gg * nl + l - m) * NQ + f) * 2 + sn) * S + sh] = a.Q[f * a.qsz + (size_t)shell * a.n_lm + l * l + c + sn * d];
    }
    __syncthreads();
    float gc[NF][S], gs[NF][S];
#pragma unroll
    for (int f = 0; f < NF; ++f)
#pragma unroll
      for (int s = 0; s < S; ++s) gc[f][s] = gs[f][s] = 0.0f;
    const float4 *q = reinterpret_cast<const float4 *>(qs) + (size_t)((group - g0 + 1) * nl - 1) * NQ * 2;
#pragma unroll 2
    for (int l = a.lmax; l >= m; --l, q -= NQ * 2) {
      const size_t at = (size_t)(l * l + c) * a.n_theta + j;
      const float pv = a.P[at];
      auto add = [&](float (&g)[S], const float4 &v, float w) {
        g[0] = fmaf(v.x, w, g[0]);
        g[1] = fmaf(v.y, w, g[1]);
        g[2] = fmaf(v.z, w, g[2]);
        g[3] = fmaf(v.w, w, g[3]);
      };
      add(gc[0], q[0], pv);
      add(gs[0], q[1], pv);
      if constexpr (NF == 4) {
        const float dv = a.dP[at], sv = a.Qs[at];
        add(gc[1], q[2], pv);
        add(gs[1], q[3], pv);
        const float4 tc = q[4], ts = q[5];
        add(gc[2], tc, dv);
        add(gs[2], ts, dv);
        add(gc[3], ts, sv);   // cos slot <- sin coefficient, sin slot <- cos
        add(gs[3], tc, sv);
      }
    }
    if (e0 + (int)threadIdx.x >= end) continue;
#pragma unroll
    for (int f = 0; f < NF; ++f)
#pragma unroll
      for (int s = 0; s < S; ++s) {
        if (shell0 + s >= a.n_shells) continue;
        float *g = a.G + f * fsz + row[s] + (size_t)c * a.tile;
        g[0] = (f == 3 && m == 0) ? 0.0f : gc[f][s];
        if (m > 0) g[a.tile] = f == 3 ? -gs[f][s] : gs[f][s];
      }
  }
}

// phi stage: 51 multiply-adds per output at l_max 25, bound by the fp32 pipe
// (its register ports: about 95 multiply-adds a clock per SM, scalar or packed).
// A thread holds 8 rows x 8 longitudes.  Rows of even length: four pairs of
// neighbouring longitudes, a quarter of a row apart, each pair one packed fp32
// instruction (its halves round as the scalar instruction does) and one 16-byte
// store: a warp's stores are 512 contiguous bytes (8 bytes a lane reach 4.7 TB/s,
// 16 bytes 6.4).  Odd rows, whose pairs would not be aligned: eight longitudes an
// eighth of a row apart.  The next tile of G is copied in while this one is used,
// and two blocks per SM run one's stores beside the other's sums.
constexpr int kR32 = 8, kC32 = 8;   // rows and longitudes of a thread
__host__ __device__ constexpr int cols32(int n_phi) { return (n_phi + kC32 - 1) / kC32; }   // threads across a row

__device__ __forceinline__ uint64_t twice(float x) {
  uint64_t d;
  asm("mov.b64 %0, {%1, %1};" : "=l"(d) : "f"(x));
  return d;
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ void copy16(float *dst, const float *src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}

constexpr int kPhiThreads = 256;

// TRS: the trig table in shared memory (else read through L1); PAIR: rows of even length
template <bool PAIR, bool TRS>
__global__ void __launch_bounds__(kPhiThreads, 2) k_phi32(const Synth32 a, int n_fields) {
  pdl_begin();
  extern __shared__ __align__(16) unsigned char smraw[];
  const int nt = 2 * a.lmax + 1, cols = cols32(a.n_phi), ldk = TRS ? cols * kC32 : a.n_phi;
  const int size = nt * a.tile;   // a multiple of 8 values
  float *Gs = reinterpret_cast<float *>(smraw);   // [2][nt][tile]
  float *trs = Gs + 2 * size;                     // [nt][ldk]
  const int total = n_fields * a.tiles;
  auto fetch = [&](int k, int buf) {
    const float *src = a.G + (size_t)k * size;
    float *to = Gs + buf * size;
    for (int e = threadIdx.x * 4; e < size; e += kPhiThreads * 4) copy16(to + e, src + e);
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  if ((int)blockIdx.x < total) fetch(blockIdx.x, 0);
  if constexpr (TRS)
    for (int e = threadIdx.x; e < nt * ldk; e += kPhiThreads) {
      const int t = e / ldk, k = e - t * ldk;
      trs[e] = k < a.n_phi ? a.tr[(size_t)t * a.n_phi + k] : 0.0f;
    }
  const int rows = a.n_shells * a.n_theta, patch_rows = a.n_r * a.n_theta;
  int buf = 0;
  for (int k = blockIdx.x; k < total; k += gridDim.x, buf ^= 1) {
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();   // tile k is in, and the tile before it is used up
    if (k + (int)gridDim.x < total) fetch(k + gridDim.x, buf ^ 1);
    const int f = k / a.tiles, first = (k - f * a.tiles) * a.tile;
    double *base0 = a.out.o[f][0], *base1 = a.out.o[f][1];
    for (int e = threadIdx.x; e < a.tile / kR32 * cols; e += kPhiThreads) {
      const int r0 = e / cols * kR32, c0 = e % cols;
      const float *g = Gs + buf * size + (size_t)(nt - 1) * a.tile + r0;
      const int k0 = PAIR ? 2 * c0 : c0, step = PAIR ? 2 * cols : cols;   // first longitude, distance of the next
      const float *tr = (TRS ? trs : a.tr) + (size_t)(nt - 1) * ldk + k0;
      auto out_row = [&](int r) -> double * {
        const int row = first + r0 + r;
        if (row >= rows) return nullptr;
        return (row >= patch_rows ? base1 + (size_t)(row - patch_rows) * a.n_phi : base0 + (size_t)row * a.n_phi) + k0;
      };
      if constexpr (PAIR) {
        constexpr int NP = kC32 / 2;
        uint64_t acc[kR32][NP];
#pragma unroll
        for (int r = 0; r < kR32; ++r)
#pragma unroll
          for (int u = 0; u < NP; ++u) acc[r][u] = 0;
#pragma unroll 1
        for (int t = nt - 1; t >= 0; --t, g -= a.tile, tr -= ldk) {
          uint64_t x[NP];
#pragma unroll
          for (int u = 0; u < NP; ++u) x[u] = *reinterpret_cast<const uint64_t *>(tr + (TRS ? u * step : min(u * step, a.n_phi - 2 - k0)));
#pragma unroll
          for (int r = 0; r < kR32; r += 4) {
            const float4 v = *reinterpret_cast<const float4 *>(g + r);
            const float y[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              const uint64_t yy = twice(y[i]);
#pragma unroll
              for (int u = 0; u < NP; ++u) acc[r + i][u] = fma2(yy, x[u], acc[r + i][u]);
            }
          }
        }
#pragma unroll
        for (int r = 0; r < kR32; ++r) {
          double *o = out_row(r);
          if (o == nullptr) break;
#pragma unroll
          for (int u = 0; u < NP; ++u)
            if (k0 + u * step < a.n_phi)
              *reinterpret_cast<double2 *>(o + u * step) = make_double2(widen_f32(__uint_as_float((uint32_t)acc[r][u])),
                                                                       widen_f32(__uint_as_float((uint32_t)(acc[r][u] >> 32))));
        }
      } else {
        float acc[kR32][kC32];
#pragma unroll
        for (int r = 0; r < kR32; ++r)
#pragma unroll
          for (int u = 0; u < kC32; ++u) acc[r][u] = 0.0f;
#pragma unroll 1
        for (int t = nt - 1; t >= 0; --t, g -= a.tile, tr -= ldk) {
          float x[kC32];
#pragma unroll
          for (int u = 0; u < kC32; ++u) x[u] = tr[TRS ? u * step : min(u * step, a.n_phi - 1 - k0)];
#pragma unroll
          for (int r = 0; r < kR32; r += 4) {
            const float4 v = *reinterpret_cast<const float4 *>(g + r);
            const float y[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
              for (int u = 0; u < kC32; ++u) acc[r + i][u] = fmaf(y[i], x[u], acc[r + i][u]);
          }
        }
#pragma unroll
        for (int r = 0; r < kR32; ++r) {
          double *o = out_row(r);
          if (o == nullptr) break;
#pragma unroll
          for (int u = 0; u < kC32; ++u)
            if (k0 + u * step < a.n_phi) o[u * step] = widen_f32(acc[r][u]);
        }
      }
    }
  }
}

// [j][mode] -> [mode][j]
__global__ void k_transpose_f32(int n_theta, int n_lm, const float *__restrict__ src, float *__restrict__ dst) {
  const size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e < (size_t)n_theta * n_lm) dst[e] = src[(e % n_theta) * n_lm + e / n_theta];
}

// 1, cos, sin at the folded columns
__global__ void k_fold_trig(int m1, AzFold f, double dph, double dph_low, double *__restrict__ out) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= m1 * f.cols) return;
  const int m = e / f.cols, c = e % f.cols;
  double sn, cs;
  fold_sincos(f, dph, dph_low, c, m, &sn, &cs);
  if (m == 0) {
    out[c] = 1.0;
  } else {
    out[(size_t)(2 * m - 1) * f.cols + c] = cs;
    out[(size_t)(2 * m) * f.cols + c] = sn;
  }
}

__global__ void k_inv_sin(int n_theta, double th0, double dth, double *__restrict__ isin) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j < n_theta) isin[j] = 1.0 / sin(th0 + dth * (j + 0.5));
}

// blocks per SM that should be in flight together, and how many rounds of
// them make the uneven end of the last one small
constexpr int kBlocksPerSm = 3, kRounds = 2;

SynthOut outputs(const yy_grid *g, double *phi_yin, double *phi_yang, double *grad_yin, double *grad_yang) {
  const size_t comp = (size_t)g->n_r * g->n_ang;
  SynthOut o = {};
  o.o[0][0] = phi_yin;
  o.o[0][1] = phi_yang;
  for (int c = 0; c < 3 && grad_yin; ++c) {
    o.o[1 + c][0] = grad_yin + c * comp;
    o.o[1 + c][1] = grad_yang ? grad_yang + c * comp : nullptr;
  }
  return o;
}

template <int NF>
size_t smem64(int lmax, int jp) {
  const size_t rows = rows64(NF, jp);
  return (size_t)stride_g((int)rows) * (2 * lmax + 1) * sizeof(double) + rows * sizeof(double *);
}
// Rows per block: as many as give the register tiles whole groups (nine row
// pairs of four fields: 72 rows), halved while the grid would leave the SMs
// short of blocks.
template <int NF>
cudaError_t run64(yy_grid *g, const Synth64 &a0, cudaStream_t s) {
  const int pairs = (g->n_theta + 1) / 2, want = g->sms * kBlocksPerSm * kRounds;
  int jp = NF == 4 ? 9 : 18;
  while (jp > 2 && (long long)grid_rows(g) * ((pairs + jp - 1) / jp) < want) jp = (jp + 1) / 2;
  Synth64 a = a0;
  a.chunks = (pairs + jp - 1) / jp;
  jp = (pairs + a.chunks - 1) / a.chunks;   // even chunks
  return launch_kernel(g, "k_synth_f64", a.fold.quarter > 0 ? k_synth_f64<NF, true> : k_synth_f64<NF, false>,
                       (unsigned)(grid_rows(g) * a.chunks), 256, smem64<NF>(g->lmax, jp), s, a, jp);
}

// Rows per tile of the fp32 form: multiples of eight whose items (eight rows x
// eight longitudes) best fill whole rounds of a block's threads and whose tiles
// best fill whole rounds of two blocks per SM.  The trig table stays out of
// shared memory where it leaves less than 64 rows room.
constexpr int kMaxTile32 = 256;
constexpr size_t kSmem32 = 113 * 1024;
struct Phi32 {
  int tile;
  size_t tiles_smem, trig_smem;
};

Phi32 phi32_shape(const yy_grid *g, int n_fields) {
  Phi32 f = {};
  const int cols = cols32(g->n_phi), slots = 2 * g->sms;
  const size_t per_row = 2 * (size_t)(2 * g->lmax + 1) * sizeof(float);   // two buffers
  f.trig_smem = (size_t)(2 * g->lmax + 1) * cols * kC32 * sizeof(float);
  if (f.trig_smem + 64 * per_row > kSmem32) f.trig_smem = 0;
  const long long rows = (long long)grid_rows(g) * g->n_theta;
  double least = 1e300;
  for (int tile = kR32; tile <= kMaxTile32 && (tile == kR32 || f.trig_smem + tile * per_row <= kSmem32); tile += kR32) {
    const long long tiles = (rows + tile - 1) / tile * n_fields;
    // rounds of the blocks, by a tile's rounds of the threads and its own cost
    const double cost = (double)((tiles + slots - 1) / slots) * ((tile / kR32 * cols + kPhiThreads - 1) / kPhiThreads + 0.15);
    if (cost < least) {
      least = cost;
      f.tile = tile;
    }
  }
  f.tiles_smem = f.tile * per_row;
  return f;
}

template <bool PAIR>
cudaError_t launch_phi32(yy_grid *g, const Synth32 &a, const Phi32 &f, int nf, cudaStream_t s) {
  return launch_kernel(g, "k_phi32", f.trig_smem ? k_phi32<PAIR, true> : k_phi32<PAIR, false>, std::min(nf * a.tiles, 2 * g->sms),
                       kPhiThreads, f.tiles_smem + f.trig_smem, s, a, nf);
}

cudaError_t run32(yy_grid *g, Synth32 a, bool grad, cudaStream_t s) {
  const int nf = grad ? 4 : 1;
  const Phi32 f = phi32_shape(g, nf);
  a.tile = f.tile;
  a.tiles = (grid_rows(g) * g->n_theta + f.tile - 1) / f.tile;
  auto qsm_of = [&](int items) { return (size_t)theta_groups(a.n_theta, items) * (a.lmax + 1) * (grad ? 3 : 1) * 2 * kS32 * sizeof(float); };
  a.items = kThetaThreads;   // less where short columns would bring too many groups into a block
  while (a.items > 1 && qsm_of(a.items) > 100 * 1024) a.items /= 2;
  const size_t qsm = qsm_of(a.items);
  const dim3 theta((unsigned)(((a.n_shells + kS32 - 1) / kS32 * a.n_theta + a.items - 1) / a.items), (unsigned)(a.lmax / 2 + 1));
  const cudaError_t e = launch_kernel(g, "k_theta32", grad ? k_theta32<4> : k_theta32<1>, theta, kThetaThreads, qsm, s, a);
  if (e != cudaSuccess) return e;
  return g->n_phi % 2 == 0 ? launch_phi32<true>(g, a, f, nf, s) : launch_phi32<false>(g, a, f, nf, s);
}

}  // namespace

AzFold az_fold(const yy_grid *g) {
  AzFold f;
  f.half = (g->n_phi + 1) / 2;
  const bool polar = g->n_patch == 1;
  f.first = polar ? 0 : g->n_phi / 2;
  // cells to phi = pi from the mirror axis: whole when the quotient is one to rounding
  int whole = 0;
  if (polar) {
    whole = g->n_phi % 2 == 0 ? g->n_phi / 2 : 0;
  } else {
    const double cells = 3.141592653589793238462643383279502884 / g->dph, near = rint(cells);
    if (fabs(cells - near) <= 4.0 * 2.220446049250313e-16 * near && near < 1e6) whole = (int)near;
  }
  f.odd = polar || g->n_phi % 2 == 0 ? 1 : 0;
  f.partner = whole > 0 ? whole - f.odd : -1;
  f.quarter = whole > 0 && whole % 2 == 0 ? whole / 2 : 0;
  f.cols = f.quarter > 0 ? (f.odd ? (f.quarter + 1) / 2 : f.quarter / 2 + 1) : f.partner >= 0 ? f.partner / 2 + 1 : f.half;
  f.cols = std::min(f.half, f.cols);
  return f;
}

// The cell width is (3 pi / 2 + 2 delta_phi) / n_phi (2 pi / n_phi on the polar grid), with pi
// beyond its double: pi / 4 is kQ + kQLow to 107 bits.
double fold_dph_low(const yy_grid *g) {
  const double kQ = 0.78539816339744830962, kQLow = 3.0616169978683829431e-17;
  const double n = g->n_phi, quarters = g->n_patch == 1 ? 8.0 : 6.0, d = 2.0 * g->delta_phi;
  const double range = quarters * kQ, low = fma(quarters, kQ, -range) + quarters * kQLow;
  const double sum = range + d, b = sum - range, err = (range - (sum - b)) + (d - b);   // exact: sum + err
  return (fma(-g->dph, n, sum) + (err + low)) / n;
}

cudaError_t synthesis_separable_prepare(yy_grid *g) {
  const int nt = 2 * g->lmax + 1;
  const AzFold f = az_fold(g);
  cudaError_t e = dmalloc((void **)&g->sep_trf, (size_t)nt * f.cols * sizeof(double));
  if (e == cudaSuccess) e = dmalloc((void **)&g->sep_isin, (size_t)g->n_theta * sizeof(double));
  if (e != cudaSuccess) return e;
  const int m1 = g->lmax + 1;
  k_fold_trig<<<(m1 * f.cols + 255) / 256, 256>>>(m1, f, g->dph, fold_dph_low(g), g->sep_trf);
  k_inv_sin<<<(g->n_theta + 255) / 256, 256>>>(g->n_theta, g->th0, g->dth, g->sep_isin);
  for (auto k : {(const void *)k_synth_f64<1, false>, (const void *)k_synth_f64<4, false>, (const void *)k_synth_f64<1, true>,
                 (const void *)k_synth_f64<4, true>, (const void *)k_theta32<1>, (const void *)k_theta32<4>,
                 (const void *)k_phi32<true, true>, (const void *)k_phi32<true, false>,
                 (const void *)k_phi32<false, true>, (const void *)k_phi32<false, false>})
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
  if (e != cudaSuccess) return e;
  // float64: any grid.  fp32: grids whose trig table (rows padded to a multiple
  // of four), coefficients and one row of G fit 227 KB; the others keep the
  // dense contraction, whose fp32 sums round differently.
  const int ntr = (g->n_phi + 3) & ~3;
  g->sep_syn_ok = 2;
  // (Rows (shell, j) are counted in 32 bits.)
  if (((size_t)nt * ntr + g->n_lm + (nt | 1)) * sizeof(float) <= 227 * 1024 && (long long)grid_rows(g) * g->n_theta <= 1 << 30)
    g->sep_syn_ok |= 1;
  return cudaGetLastError();
}

cudaError_t synthesis_separable_prepare_f32(yy_grid *g) {
  if (!(g->sep_syn_ok & 1)) return cudaSuccess;   // the dense contraction serves
  const size_t n_p = (size_t)g->n_theta * g->n_lm, rows = (size_t)grid_rows(g) * g->n_theta;
  const float *src[3] = {g->sep_P32, g->sep_dP32, g->sep_Qs32};
  cudaError_t e = cudaSuccess;
  for (int q = 0; q < 3 && e == cudaSuccess; ++q) {
    if (g->sep_T32[q]) continue;
    if ((e = dmalloc((void **)&g->sep_T32[q], n_p * sizeof(float))) == cudaSuccess)
      k_transpose_f32<<<(unsigned)((n_p + 255) / 256), 256>>>(g->n_theta, g->n_lm, src[q], g->sep_T32[q]);
  }
  // four fields of whole tiles
  if (e == cudaSuccess && !g->sep_G32)
    e = dmalloc((void **)&g->sep_G32, 4 * (rows + kMaxTile32 - 1) * (2 * g->lmax + 1) * sizeof(float));
  return e == cudaSuccess ? cudaGetLastError() : e;
}

cudaError_t synthesis_separable(yy_grid *g, double *phi_yin, double *phi_yang, double *grad_yin, double *grad_yang,
                                bool fp64, cudaStream_t s) {
  const SynthOut o = outputs(g, phi_yin, phi_yang, grad_yin, grad_yang);
  const size_t qsz = (size_t)grid_rows(g) * g->n_lm;
  if (fp64) {
    const Synth64 a = {g->n_r, g->n_theta, g->n_phi, g->lmax, g->n_lm, 0, az_fold(g), g->Q, g->sep_P, g->sep_dP,
                       g->sep_trf, g->sep_isin, g->r_edges, qsz, o};
    return grad_yin ? run64<4>(g, a, s) : run64<1>(g, a, s);
  }
  const Synth32 a = {grid_rows(g), g->n_r, g->n_theta, g->n_phi, g->lmax, g->n_lm, 0, 0, 0, g->Q32, g->sep_T32[0],
                     g->sep_T32[1], g->sep_T32[2], g->sep_tr32, g->sep_G32, qsz, o};
  return run32(g, a, grad_yin != nullptr, s);
}

}  // namespace yy
