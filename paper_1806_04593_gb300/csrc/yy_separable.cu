// Separable analysis (§3 Eqs. ac/as with the §4 weights):
//
//   A_p[i][lm] = sum_j K_lm T_j^(lm) sum_k rho_p[i][j][k] w_jk {C_k^(m) | S_k^(m)}
//
// The weight w_jk is not a product of a theta and a phi factor (it follows the
// overlap boundary), so it is folded into the density first; the remaining
// double sum factors into an azimuthal stage and a polar stage:
//
//   phi stage    F[p,i][j][t] = sum_k (rho w)_ijk az[t][k],
//                az[0] = d_phi (m = 0), az[2m-1] = C_k^(m), az[2m] = S_k^(m)
//   theta stage  A[p,i][l^2 + t] = sum_j (K_lm T_j^(lm)) F[p,i][j][t]
//
// which costs 2 N_ang (2 l_max + 1) + 2 n_theta n_lm flops per shell instead of
// 2 N_ang n_lm for the dense contraction (12.6 times fewer at the 1-degree grid
// with l_max = 25).  The float64 kernels (k_sep_phi64, k_sep_theta64) fold the cells by
// the symmetries of both angles.  The fp32 ones (k_sep_phi32, k_sep_theta32) sum
// in order, except that the m = 0 sums, which carry the monopole and so
// dominate Phi, are compensated fp32 pairs in the azimuthal stage and float64
// in the polar stage.
#include <math.h>

#include <algorithm>
#include <type_traits>

#include "yy_internal.h"

namespace yy {
namespace {

// exact float64 -> fp32 rounding by integer operations (round to nearest even):
// the rounding bias added at bit 29 of the 64-bit word, bits 29..60 kept and the
// exponent rebiased; values outside the normal fp32 range are converted
__device__ __forceinline__ float narrow(double x) {
  const unsigned long long u = (unsigned long long)__double_as_longlong(x);
  const unsigned int hi = (unsigned int)(u >> 32);
  if (((hi >> 20) & 0x7FFu) - 897u >= 254u) return (float)x;
  const unsigned int r = (unsigned int)((u + 0x0FFFFFFFull + ((u >> 29) & 1ull)) >> 29) - (896u << 23);
  return __uint_as_float((r & 0x7FFFFFFFu) | (hi & 0x80000000u));
}

// Knuth's two-sum into an unevaluated fp32 pair (h, l)
__device__ __forceinline__ void pair_add(float &h, float &l, float b) {
  const float s = h + b;
  const float bb = s - h;
  l += (h - (s - bb)) + (b - bb);
  h = s;
}

__device__ __forceinline__ int degree_of(int idx) {
  int l = (int)sqrtf((float)idx);   // corrected below; exact for idx < 2^24
  while (l * l > idx) --l;
  while ((l + 1) * (l + 1) <= idx) ++l;
  return l;
}

// az[k][t] (t fastest, padded to nt_pad): the azimuthal cell integrals
__global__ void k_az_table(int n_phi, int lmax, int nt_pad, double ph0, double dph, double *__restrict__ az) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= n_phi * nt_pad) return;
  const int k = e / nt_pad, t = e % nt_pad;
  double v = 0.0;
  if (t == 0) {
    v = dph;
  } else if (t <= 2 * lmax) {
    const int m = (t + 1) / 2;
    const double phc = ph0 + dph * (k + 0.5);
    const double half = 2.0 * sin(0.5 * m * dph) / m;   // closed forms of C_k^(m), S_k^(m) (§2)
    v = (t & 1) ? cos(m * phc) * half : sin(m * phc) * half;
  }
  az[e] = v;
}

// tb0[j][l] = K_l0 T_j^(l0) d_phi as an unevaluated fp32 pair (hi, lo)
__global__ void k_tb0(int n_theta, int lmax, int n_lm, double dph, const double *__restrict__ tbar,
                      float2 *__restrict__ tb0) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= n_theta * (lmax + 1)) return;
  const int j = e / (lmax + 1), l = e % (lmax + 1);
  const double v = tbar[(size_t)j * n_lm + l * l] * dph;
  const float hi = (float)v;
  tb0[e] = make_float2(hi, (float)(v - (double)hi));
}

__global__ void k_round(size_t n, const double *__restrict__ src, float *__restrict__ dst) {
  const size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e < n) dst[e] = (float)src[e];
}

constexpr int kTT = 4;     // azimuthal functions per thread of the fp32 azimuthal stage

// four consecutive values, 16-byte aligned
__device__ __forceinline__ void ld4(const float *p, float (&o)[4]) {
  const float4 v = *reinterpret_cast<const float4 *>(p);
  o[0] = v.x;
  o[1] = v.y;
  o[2] = v.z;
  o[3] = v.w;
}
__device__ __forceinline__ void st4(float *p, const float (&v)[4]) {
  *reinterpret_cast<float4 *>(p) = make_float4(v[0], v[1], v[2], v[3]);
}

// exact product a b = p + e (fma-based) and an unevaluated-pair dot step
__device__ __forceinline__ void pair_fma(float &h, float &l, float ah, float al, float bh, float bl) {
  const float p = ah * bh;
  const float e = fmaf(ah, bh, -p);
  pair_add(h, l, p);
  l += e + fmaf(ah, bl, al * bh);
}

// Azimuthal stage, float64.  The float64 pipe (two operations per clock per SM)
// sets the time, so the cells are folded by their symmetries first (AzFold):
// with E, O the sum and difference of a cell and its mirror, cos slots take E
// and sin slots O over half the columns; where cells phi and pi - phi both
// exist, E +- E' and O -+ O' serve the even and odd orders over a third of them;
// where pi / 2 is a whole number of cells, the columns at phi, pi / 2 -+ phi and
// pi - phi (A, B, C, D) become one: even orders take sums of the four by m mod 4 with
// one product per slot, odd orders A and D with their own function and B and C with
// the other one (on the 1-degree Yin-Yang grid 45 columns for 270 cells: 16.2
// float64 operations per cell instead of 52; 0.89 ms there at 550 zones and
// l_max 25 against 0.97 ms with pi - phi alone and 3.02 ms without the folds,
// 62 us, 72 and 214 on the 2-degree grid of 200 zones at l_max 15).  A
// block takes up to 16 consecutive rows (shell, j); each thread then sums both
// slots of an order m for two rows.
constexpr int kR64 = 2;

struct SepPhi64 {
  int rows, per, n_r, n_theta, n_phi, m1, nt_pad;   // per: rows of a block, even
  AzFold fold;
  const double *rho0, *rho1, *w;
  const double2 *az;   // [column][m]: the cell integrals of cos and sin (m phi)
  double *F;
};

// planes of the staged, folded rows: [plane][column][per]
//   pi - phi at most: E of even m, E of odd m, O of even m, O of odd m
//   quarter fold: E of m mod 4 = 0, 2, O of m mod 4 = 0, 2, then of odd m: E_A - E_D,
//   E_B - E_C, O_A + O_D, O_B + O_C
constexpr int kPlanes = 4, kPlanesQuarter = 8;

__global__ void k_sep_phi64(const SepPhi64 a) {
  pdl_begin();
  extern __shared__ __align__(16) unsigned char smraw[];
  double *xs = reinterpret_cast<double *>(smraw);
  const int row0 = blockIdx.x * a.per, cols = a.fold.cols, plane = cols * a.per;
  const int patch_rows = a.n_r * a.n_theta, h = a.fold.half;
  const bool quarter = a.fold.quarter > 0;
  for (int e = threadIdx.x; e < plane; e += blockDim.x) {
    const int r = e / cols, c = e % cols, row = row0 + r;
    double *o = xs + c * a.per + r;
    const bool ok = row < a.rows;
    const int rr = ok ? row : 0;
    const double *x = (rr >= patch_rows ? a.rho1 + (size_t)(rr - patch_rows) * a.n_phi : a.rho0 + (size_t)rr * a.n_phi);
    const double *w = a.w + (size_t)(rr % a.n_theta) * a.n_phi;
    auto fold = [&](bool on, int col, double &E, double &O) {
      E = O = 0.0;
      if (!ok || !on) return;
      const int kp = a.fold.first + col, km = a.n_phi - 1 - kp;
      const double u = x[kp] * w[kp];
      if (km == kp) {
        E = u;
      } else {
        const double v = x[km] * w[km];
        E = u + v;
        O = u - v;
      }
    };
    if (quarter) {
      const int kb = a.fold.quarter - a.fold.odd - c, kc = a.fold.quarter + c, kd = a.fold.partner - c;
      double ea, oa, eb, ob, ec, oc, ed, od;
      fold(true, c, ea, oa);
      fold(kb != c && kb < h, kb, eb, ob);
      fold(kc != kb && kc < h, kc, ec, oc);
      fold(kd != kc && kd != c && kd < h, kd, ed, od);
      const double e1 = ea + ed, e2 = eb + ec, o1 = oa - od, o2 = ob - oc;
      o[0] = e1 + e2;           // cos(m phi), m mod 4 = 0
      o[plane] = e1 - e2;       // 2
      o[2 * plane] = o1 - o2;   // sin(m phi), m mod 4 = 0
      o[3 * plane] = o1 + o2;   // 2
      o[4 * plane] = ea - ed;
      o[5 * plane] = eb - ec;
      o[6 * plane] = oa + od;
      o[7 * plane] = ob + oc;
    } else {
      double ee, oe, E, O;
      fold(true, c, ee, oe);
      const int pc = a.fold.partner - c;
      fold(a.fold.partner >= 0 && pc > c && pc < h, pc, E, O);
      o[0] = ee + E;            // cos(m (pi - phi)) = (-1)^m cos(m phi)
      o[plane] = ee - E;
      o[2 * plane] = oe - O;    // sin(m (pi - phi)) = -(-1)^m sin(m phi)
      o[3 * plane] = oe + O;
    }
  }
  __syncthreads();
  // items (pair of rows, order), the even orders first: with the quarter fold an
  // odd order costs twice an even one, and a warp should not hold both
  const int pairs = a.per / kR64, evens = (a.m1 + 1) / 2;
  for (int e = threadIdx.x; e < pairs * a.m1; e += blockDim.x) {
    const bool is_odd = e >= pairs * evens;
    const int e1 = is_odd ? e - pairs * evens : e, n = is_odd ? a.m1 - evens : evens;
    const int r = e1 / n * kR64, m = e1 % n * 2 + (is_odd ? 1 : 0);
    const double2 *az = a.az + m;
    double cs[kR64] = {0.0, 0.0}, sn[kR64] = {0.0, 0.0};
    auto sum = [&](const double *xe, const double *xo) {
#pragma unroll 4
      for (int c = 0; c < cols; ++c) {
        const double2 t = az[(size_t)c * a.m1];
        const double2 u = *reinterpret_cast<const double2 *>(xe + c * a.per), v = *reinterpret_cast<const double2 *>(xo + c * a.per);
        cs[0] = fma(u.x, t.x, cs[0]);
        cs[1] = fma(u.y, t.x, cs[1]);
        sn[0] = fma(v.x, t.y, sn[0]);
        sn[1] = fma(v.y, t.y, sn[1]);
      }
    };
    if (!quarter) {
      sum(xs + (is_odd ? plane : 0) + r, xs + (is_odd ? 3 : 2) * plane + r);
    } else if (!is_odd) {
      sum(xs + (m & 2 ? plane : 0) + r, xs + (m & 2 ? 3 : 2) * plane + r);
    } else {
      const double *ea = xs + 4 * plane + r, *eb = ea + plane, *oa = eb + plane, *ob = oa + plane;
      double cq[kR64] = {0.0, 0.0}, sq[kR64] = {0.0, 0.0};   // B and C, with the other function
#pragma unroll 2
      for (int c = 0; c < cols; ++c) {
        const double2 t = az[(size_t)c * a.m1];
        const double2 u = *reinterpret_cast<const double2 *>(ea + c * a.per), v = *reinterpret_cast<const double2 *>(oa + c * a.per);
        const double2 p = *reinterpret_cast<const double2 *>(eb + c * a.per), q = *reinterpret_cast<const double2 *>(ob + c * a.per);
        cs[0] = fma(u.x, t.x, cs[0]);
        cs[1] = fma(u.y, t.x, cs[1]);
        sn[0] = fma(v.x, t.y, sn[0]);
        sn[1] = fma(v.y, t.y, sn[1]);
        cq[0] = fma(p.x, t.y, cq[0]);
        cq[1] = fma(p.y, t.y, cq[1]);
        sq[0] = fma(q.x, t.x, sq[0]);
        sq[1] = fma(q.y, t.x, sq[1]);
      }
#pragma unroll
      for (int i = 0; i < kR64; ++i) {   // sin(m pi / 2) = 1, -1 for m mod 4 = 1, 3
        cs[i] += (m & 2) ? -cq[i] : cq[i];
        sn[i] += (m & 2) ? -sq[i] : sq[i];
      }
    }
#pragma unroll
    for (int i = 0; i < kR64; ++i) {
      if (row0 + r + i >= a.rows) break;
      double *F = a.F + (size_t)(row0 + r + i) * a.nt_pad;
      if (m == 0) {
        F[0] = cs[i];
      } else {
        F[2 * m - 1] = cs[i];
        F[2 * m] = sn[i];
      }
    }
  }
}

// az[column][m] = the cell integrals of cos and sin (m phi) at the folded columns
__global__ void k_fold_az(int m1, AzFold f, double dph, double dph_low, double2 *__restrict__ out) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= m1 * f.cols) return;
  const int c = e / m1, m = e % m1;
  double sn, cs;
  fold_sincos(f, dph, dph_low, c, m, &sn, &cs);
  const double width = m == 0 ? dph : 2.0 * sin(0.5 * m * dph) / m;
  out[e] = make_double2(cs * width, sn * width);
}

// Azimuthal stage, fp32: every F is one chain of fp32 multiply-adds over k in
// order.  A block takes 32 consecutive rows (shell, j) of a patch and walks k in
// pieces of 32.  Four warps copy the next piece while this one is summed (8 rows
// each, lane = k), round and weight it and write it transposed; all threads sum
// it, R rows x 4 functions each, the table's piece in shared memory beside it
// (through L1 it came from L2: the staged rows leave L1 little room).  On the
// 1-degree grid, 550 zones, l_max 25: 155 us (300 us with whole shells staged and
// the table read per 16 products), bound by instruction issue; 22 us
// against 48 on the 2-degree grid of 200 zones at l_max 15.  Every other row is narrowed
// by the conversion instruction, on the float64 pipe, idle here (same rounding: all by
// integer operations 168 us, all by the instruction 161); whole pieces of whole blocks
// take no checks per value (162 without).  The row's compensated sum (the m = 0
// azimuthal sum without the factor d_phi) is formed by the lanes as they convert:
// lane L adds k = L, L + 32, ... to an unevaluated fp32 pair, and shuffles add the
// lanes' pairs.
constexpr int kRows32 = 32, kPiece = 32, kLoadWarps = 4, kLoadRows = kRows32 / kLoadWarps;
constexpr int kLd32 = kRows32 + 4;   // row stride of a staged k: 16-byte writes of 8 lanes on 32 banks

struct SepPhi32 {
  int n_r, n_theta, n_phi, nt_pad;
  const double *rho[2];
  const float *w, *az;   // az [k][nt_pad]
  float *F;
  float2 *F0;
};

__device__ __forceinline__ void copy_async(double *dst, const double *src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void copy_async16(float *dst, const float *src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void copy_async(float *dst, const float *src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}

template <int kR32>
__global__ void k_sep_phi32(const SepPhi32 a) {
  pdl_begin();
  extern __shared__ __align__(16) float azs[];            // [2][kPiece][nt_pad]
  __shared__ __align__(16) double raw[kRows32][kPiece];
  __shared__ __align__(16) float wts[kRows32][kPiece];
  __shared__ __align__(16) float xs[2][kPiece * kLd32];   // [k][row]
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int patch_rows = a.n_r * a.n_theta, row0 = blockIdx.x * kRows32;
  const int rows = min(kRows32, patch_rows - row0), j0 = row0 % a.n_theta;
  const double *src = (blockIdx.y ? a.rho[1] : a.rho[0]) + (size_t)row0 * a.n_phi;
  const size_t out0 = (size_t)blockIdx.y * patch_rows + row0;
  const int tg = a.nt_pad / kTT, r = threadIdx.x / tg * kR32, tt = threadIdx.x % tg;
  const int pieces = (a.n_phi + kPiece - 1) / kPiece, q = warp * kLoadRows;
  const bool loads = warp < kLoadWarps;
  int wrow[kLoadRows];   // the rows' offsets in the weights
#pragma unroll
  for (int i = 0; i < kLoadRows; ++i) wrow[i] = (j0 + q + i) % a.n_theta * a.n_phi;
  // the rows: a thread reads only what it copied itself; the table: after a barrier
  auto fetch = [&](int p) {
    const int k = p * kPiece + lane;
    if (loads && k < a.n_phi) {
      const double *x = src + q * a.n_phi + k;
      if (rows == kRows32) {
#pragma unroll
        for (int i = 0; i < kLoadRows; ++i) {
          copy_async(&raw[q + i][lane], x + i * a.n_phi);
          copy_async(&wts[q + i][lane], a.w + wrow[i] + k);
        }
      } else {
        for (int i = 0; i < kLoadRows && q + i < rows; ++i) {
          copy_async(&raw[q + i][lane], x + i * a.n_phi);
          copy_async(&wts[q + i][lane], a.w + (j0 + q + i) % a.n_theta * a.n_phi + k);
        }
      }
    }
    const int n = min(kPiece, a.n_phi - p * kPiece) * a.nt_pad;
    for (int e = threadIdx.x * 4; e < n; e += blockDim.x * 4)
      copy_async16(azs + (p & 1) * kPiece * a.nt_pad + e, a.az + (size_t)p * kPiece * a.nt_pad + e);
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  fetch(0);
  float h[kLoadRows], l[kLoadRows];
#pragma unroll
  for (int i = 0; i < kLoadRows; ++i) h[i] = l[i] = 0.0f;
  float acc[kR32][kTT];
#pragma unroll
  for (int i = 0; i < kR32; ++i)
#pragma unroll
    for (int b = 0; b < kTT; ++b) acc[i][b] = 0.0f;
  for (int p = 0; p < pieces; ++p) {
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    if (loads) {
      float v[kLoadRows];
      auto convert = [&](auto whole) {
#pragma unroll
        for (int i = 0; i < kLoadRows; ++i) {
          v[i] = 0.0f;
          if (decltype(whole)::value || (p * kPiece + lane < a.n_phi && q + i < rows)) {
            const double x = raw[q + i][lane];
            // rounded before the pair's sum
            v[i] = __fmul_rn(i & 1 ? __double2float_rn(x) : narrow(x), wts[q + i][lane]);
            pair_add(h[i], l[i], v[i]);
          }
        }
      };
      if (rows == kRows32 && (p + 1) * kPiece <= a.n_phi)
        convert(std::true_type());
      else
        convert(std::false_type());
      float4 *to = reinterpret_cast<float4 *>(&xs[p & 1][lane * kLd32 + q]);
      to[0] = make_float4(v[0], v[1], v[2], v[3]);
      to[1] = make_float4(v[4], v[5], v[6], v[7]);
    }
    __syncthreads();   // piece p is in; the other buffers are used up
    if (p + 1 < pieces) fetch(p + 1);
    if (r < kRows32) {
      const float *x = &xs[p & 1][r], *az = azs + (p & 1) * kPiece * a.nt_pad + tt * kTT;
      const int n = min(kPiece, a.n_phi - p * kPiece);
#pragma unroll 8
      for (int k = 0; k < n; ++k) {
        float t4[4], u[kR32];
        ld4(az + k * a.nt_pad, t4);
        if constexpr (kR32 == 4) {
          ld4(x + k * kLd32, u);
        } else {
          const float2 u2 = *reinterpret_cast<const float2 *>(x + k * kLd32);
          u[0] = u2.x;
          u[1] = u2.y;
        }
#pragma unroll
        for (int i = 0; i < kR32; ++i)
#pragma unroll
          for (int b = 0; b < kTT; ++b) acc[i][b] = fmaf(u[i], t4[b], acc[i][b]);
      }
    }
  }
  if (r < kRows32)
#pragma unroll
    for (int i = 0; i < kR32; ++i)
      if (r + i < rows) st4(a.F + (out0 + r + i) * a.nt_pad + tt * kTT, acc[i]);
  if (!loads) return;
#pragma unroll
  for (int i = 0; i < kLoadRows; ++i) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
      const float oh = __shfl_xor_sync(0xffffffffu, h[i], off);
      const float ol = __shfl_xor_sync(0xffffffffu, l[i], off);
      pair_add(h[i], l[i], oh);
      l[i] += ol;
    }
    if (lane == 0 && q + i < rows) a.F0[out0 + q + i] = make_float2(h[i], l[i]);
  }
}

// The polar stages' dot products over j wait for table loads from L2, so a
// thread keeps eight of them in flight and a block has a thread per mode, up to
// 1024.
constexpr int kBatch = 8;
int theta_threads(int n_lm, int extra) { return std::min(1024, (n_lm + 31) / 32 * 32 + extra); }

// Polar stage, fp32: a block takes S shells, their F in shared memory, so that a
// table value serves all of them; per mode and shell an fp32 dot product over j
// in order.  The last warp takes the m = 0 modes: an unevaluated-pair dot product
// of the pair-split table (with d_phi folded in) and the pair row sums, then one
// float64 addition.  1-degree grid, 550 zones: 43 us with four shells a block,
// 70 with one; 200 zones of 2-degree cells: 14 with two, 12 with one.
template <int S>
__global__ void k_sep_theta32(int n_shells, int n_theta, int n_lm, int lmax1, int nt_pad, const float *__restrict__ tb,
                              const float2 *__restrict__ tb0, const float *__restrict__ F, const float2 *__restrict__ F0,
                              double *__restrict__ A) {
  pdl_begin();
  extern __shared__ __align__(16) unsigned char smraw[];
  const int shell0 = blockIdx.x * S, ns = min(S, n_shells - shell0), rows = S * n_theta;
  float2 *f0s = reinterpret_cast<float2 *>(smraw);                 // [S][n_theta]
  float *fs = reinterpret_cast<float *>(f0s + rows + (rows & 1));     // [S][n_theta][nt_pad]
  const size_t row0 = (size_t)shell0 * n_theta;
  for (int e = threadIdx.x; e < ns * n_theta * nt_pad / 4; e += blockDim.x)
    reinterpret_cast<float4 *>(fs)[e] = reinterpret_cast<const float4 *>(F + row0 * nt_pad)[e];
  for (int e = threadIdx.x; e < ns * n_theta; e += blockDim.x) f0s[e] = F0[row0 + e];
  __syncthreads();
  const int modes = blockDim.x - 32;   // threads of the m > 0 modes
  if ((int)threadIdx.x >= modes) {
    for (int e = threadIdx.x - modes; e < ns * lmax1; e += 32) {
      const int q = e / lmax1, l = e % lmax1;
      const float2 *y = f0s + q * n_theta;
      float h = 0.0f, lo = 0.0f;
      for (int j0 = 0; j0 < n_theta; j0 += kBatch) {
        float2 x[kBatch];
#pragma unroll
        for (int u = 0; u < kBatch; ++u) x[u] = tb0[(size_t)min(j0 + u, n_theta - 1) * lmax1 + l];
#pragma unroll
        for (int u = 0; u < kBatch; ++u)
          if (j0 + u < n_theta) pair_fma(h, lo, x[u].x, x[u].y, y[j0 + u].x, y[j0 + u].y);
      }
      A[(size_t)(shell0 + q) * n_lm + l * l] = widen_f32(h) + widen_f32(lo);
    }
    return;
  }
  for (int idx = threadIdx.x; idx < n_lm; idx += modes) {
    const int l = degree_of(idx);
    const int t = idx - l * l;
    if (t == 0) continue;
    const float *tab = tb + idx, *f = fs + t;
    float s[S];
#pragma unroll
    for (int q = 0; q < S; ++q) s[q] = 0.0f;
    for (int j0 = 0; j0 < n_theta; j0 += kBatch) {
      float v[kBatch];
#pragma unroll
      for (int u = 0; u < kBatch; ++u) v[u] = tab[(size_t)min(j0 + u, n_theta - 1) * n_lm];
#pragma unroll
      for (int u = 0; u < kBatch; ++u)
        if (j0 + u < n_theta) {
#pragma unroll
          for (int q = 0; q < S; ++q) s[q] = fmaf(v[u], f[(q * n_theta + j0 + u) * nt_pad], s[q]);
        }
    }
#pragma unroll
    for (int q = 0; q < S; ++q)
      if (q < ns) A[(size_t)(shell0 + q) * n_lm + idx] = widen_f32(s[q]);
  }
}

// Polar stage, float64: one block per shell, the shell's F staged in shared
// memory, one thread per mode.
__global__ void k_sep_theta64(int n_theta, int n_lm, int nt_pad, const double *__restrict__ tb,
                                                     const double *__restrict__ F, double *__restrict__ A) {
  pdl_begin();
  extern __shared__ __align__(16) unsigned char smraw[];
  const int shell = blockIdx.x;
  const double *Fs = F + (size_t)shell * n_theta * nt_pad;
  // The polar cells are symmetric about the equator (cell n_theta - 1 - j is
  // cell j reflected), so the cell integrals of P_l^m(cos theta) sin theta
  // have its parity: T_j' = (-1)^(l + m) T_j.  With S_j = F_j + F_j' and
  // D_j = F_j - F_j', a mode is the sum over j < ceil(n_theta / 2) of T_j S_j
  // (even l + m) or T_j D_j (odd): half the products.  A middle row (odd
  // n_theta) is its own mirror and enters once, as both S and D.
  const int half = (n_theta + 1) >> 1;
  double *cs = reinterpret_cast<double *>(smraw);                  // [2][half][nt_pad]: S, then D
  for (int e = threadIdx.x; e < half * nt_pad; e += blockDim.x) {
    const int j = e / nt_pad, jm = n_theta - 1 - j;
    const double a = Fs[e], b = Fs[(size_t)(jm - j) * nt_pad + e];
    cs[e] = jm == j ? a : a + b;
    cs[(size_t)half * nt_pad + e] = jm == j ? a : a - b;
  }
  __syncthreads();
  for (int idx = threadIdx.x; idx < n_lm; idx += blockDim.x) {
    const int l = degree_of(idx);
    const int t = idx - l * l;
    const double *c = cs + ((((l + ((t + 1) >> 1)) & 1) != 0) ? (size_t)half * nt_pad : 0) + t;
    const double *tab = tb + idx;
    double s = 0.0;
    for (int j0 = 0; j0 < half; j0 += kBatch) {
      double v[kBatch];
#pragma unroll
      for (int u = 0; u < kBatch; ++u) v[u] = tab[(size_t)min(j0 + u, half - 1) * n_lm];
#pragma unroll
      for (int u = 0; u < kBatch; ++u)
        if (j0 + u < half) s = fma(v[u], c[(j0 + u) * nt_pad], s);
    }
    A[(size_t)shell * n_lm + idx] = s;
  }
}

// Dynamic shared memory of the polar stages: the fp32 form stages a shell's F and
// m = 0 pair sums, the float64 form the mirrored sums S and D of ceil(n_theta / 2)
// rows each.
static size_t theta_smem(int n_theta, int nt_pad, size_t el) {
  if (el == sizeof(double)) return (size_t)(n_theta + 1) * nt_pad * sizeof(double);
  return (size_t)n_theta * nt_pad * el + (size_t)(n_theta + 1) * sizeof(float2);
}

// Polar stage after the tensor-core azimuthal stage: F of the rows (shell, j)
// comes from the raw fp32 sums part[t][row] of the centred and scaled rows,
// F = part * row_scale * t_scale + mean * colsum[t] (the centring undone with
// the column sums of the table), and the m = 0 row sums from their float64
// values.  A block takes kThetaShells shells (each table value read serves
// all of them); one measured fastest: with four, 275 blocks of 98 KB left
// most SMs with a single block.
constexpr int kThetaShells = 1;

__global__ void __launch_bounds__(256) k_sep_theta_partials(SepThetaPartials a, int n_shells) {
  constexpr int S = kThetaShells;
  extern __shared__ __align__(16) unsigned char smraw[];
  float2 *f0s = reinterpret_cast<float2 *>(smraw);                          // [S][n_theta]
  float *rsm = reinterpret_cast<float *>(f0s + S * a.n_theta);               // [S][n_theta][2]: scale, mean
  float *fs = rsm + 2 * S * a.n_theta;                                      // [S][n_theta][nt_pad + 1]
  const int fst = a.nt_pad + 1;                                             // odd stride: conflict-free fill
  const int shell0 = blockIdx.x * S;
  const int ns = min(S, n_shells - shell0);
  for (int e = threadIdx.x; e < S * a.n_theta; e += blockDim.x) {
    const int q = e / a.n_theta, j = e - q * a.n_theta;
    float2 f0 = make_float2(0.0f, 0.0f);
    float sc = 0.0f, mn = 0.0f;
    if (q < ns) {
      const size_t row = (size_t)(shell0 + q) * a.n_theta + j;
      const double d = a.F0[row];
      const float hi = narrow(d);
      f0 = make_float2(hi, narrow(d - widen_f32(hi)));
      sc = a.row_scale[row];
      mn = narrow(a.mean[row]);
    }
    f0s[e] = f0;
    rsm[2 * e] = sc;
    rsm[2 * e + 1] = mn;
  }
  __syncthreads();
  const int rows = S * a.n_theta;   // the block's rows are consecutive: (shell0 + q) n_theta + j
  const size_t row0 = (size_t)shell0 * a.n_theta;
  for (int e = threadIdx.x; e < a.nt_pad * rows; e += blockDim.x) {
    const int t = e / rows, qj = e - t * rows;
    float v = 0.0f;
    if (t >= 1 && t < a.nt && qj < ns * a.n_theta)
      v = fmaf(a.part[(size_t)t * a.part_ld + row0 + qj] * rsm[2 * qj], a.t_scale[t], rsm[2 * qj + 1] * a.colsum[t]);
    fs[(size_t)qj * fst + t] = v;
  }
  __syncthreads();
  // m = 0 modes: warp q < S takes shell q, lanes the degrees, compensated
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (warp < ns) {
    for (int l = lane; l < a.lmax1; l += 32) {
      float h = 0.0f, lo = 0.0f;
      for (int j = 0; j < a.n_theta; ++j) {
        const float2 x = a.tb0[(size_t)j * a.lmax1 + l], y = f0s[warp * a.n_theta + j];
        pair_fma(h, lo, x.x, x.y, y.x, y.y);
      }
      a.A[(size_t)(shell0 + warp) * a.n_lm + l * l] = widen_f32(h) + widen_f32(lo);
    }
  }
  // the other modes: fp32 dot products over j, one table read for all S shells
  for (int idx = threadIdx.x; idx < a.n_lm; idx += blockDim.x) {
    const int l = degree_of(idx);
    const int t = idx - l * l;
    if (t == 0) continue;
    float acc[S];
#pragma unroll
    for (int q = 0; q < S; ++q) acc[q] = 0.0f;
#pragma unroll 4
    for (int j = 0; j < a.n_theta; ++j) {
      const float tv = a.tb[(size_t)j * a.n_lm + idx];
#pragma unroll
      for (int q = 0; q < S; ++q) acc[q] = fmaf(tv, fs[((size_t)q * a.n_theta + j) * fst + t], acc[q]);
    }
#pragma unroll
    for (int q = 0; q < S; ++q)
      if (q < ns) a.A[(size_t)(shell0 + q) * a.n_lm + idx] = widen_f32(acc[q]);
  }
}

// Rows per block of the float64 azimuthal stage: 16 (two blocks or more per SM
// at the folded columns of one-degree cells), halved while the SMs are short of
// blocks or the staged rows do not fit; 0: not even two rows fit.
size_t phi64_smem(const AzFold &f, int rows) {
  return (size_t)(f.quarter > 0 ? kPlanesQuarter : kPlanes) * f.cols * rows * sizeof(double);
}
int phi64_rows(const yy_grid *g) {
  const AzFold f = az_fold(g);
  const long long rows = (long long)grid_rows(g) * g->n_theta;
  int per = 16;
  while (per > 2 && (phi64_smem(f, per) > 113 * 1024 || (rows + per - 1) / per < 2 * g->sms)) per /= 2;
  return phi64_smem(f, per) <= 227 * 1024 ? per : 0;
}

}  // namespace

cudaError_t separable_prepare(yy_grid *g) {
  const int nt_pad = (2 * g->lmax + 1 + kTT - 1) / kTT * kTT;
  g->sep_nt_pad = nt_pad;
  const size_t n_az = (size_t)g->n_phi * nt_pad;
  const size_t n_tb = (size_t)g->n_theta * g->n_lm;
  const size_t n_f = (size_t)grid_rows(g) * g->n_theta * nt_pad;
  cudaError_t e = cudaSuccess;
  auto A = [&](void **p, size_t bytes) {
    if (e == cudaSuccess) e = dmalloc(p, bytes);
  };
  A((void **)&g->sep_az, n_az * sizeof(double));
  A((void **)&g->sep_az32, n_az * sizeof(float));
  A((void **)&g->sep_w32, (size_t)g->n_ang * sizeof(float));
  A((void **)&g->sep_tb32, n_tb * sizeof(float));
  A((void **)&g->sep_F, n_f * sizeof(double));   // float64 or fp32 partial transforms
  A((void **)&g->sep_F0, (size_t)grid_rows(g) * g->n_theta * sizeof(float2));
  A((void **)&g->sep_tb0, (size_t)g->n_theta * (g->lmax + 1) * sizeof(float2));
  if (e != cudaSuccess) return e;
  k_tb0<<<(g->n_theta * (g->lmax + 1) + 255) / 256, 256>>>(g->n_theta, g->lmax, g->n_lm, g->dph, g->tbar,
                                                           g->sep_tb0);
  k_az_table<<<(unsigned)((n_az + 255) / 256), 256>>>(g->n_phi, g->lmax, nt_pad, g->ph0, g->dph, g->sep_az);
  k_round<<<(unsigned)((n_az + 255) / 256), 256>>>(n_az, g->sep_az, g->sep_az32);
  k_round<<<(unsigned)((g->n_ang + 255) / 256), 256>>>((size_t)g->n_ang, g->w, g->sep_w32);
  k_round<<<(unsigned)((n_tb + 255) / 256), 256>>>(n_tb, g->tbar, g->sep_tb32);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  {
    const size_t n_p = (size_t)g->n_theta * g->n_lm, n_tr = (size_t)(2 * g->lmax + 1) * g->n_phi;
    A((void **)&g->sep_P32, n_p * sizeof(float));
    A((void **)&g->sep_dP32, n_p * sizeof(float));
    A((void **)&g->sep_Qs32, n_p * sizeof(float));
    A((void **)&g->sep_tr32, n_tr * sizeof(float));
    if (e != cudaSuccess) return e;
    k_round<<<(unsigned)((n_p + 255) / 256), 256>>>(n_p, g->sep_P, g->sep_P32);
    k_round<<<(unsigned)((n_p + 255) / 256), 256>>>(n_p, g->sep_dP, g->sep_dP32);
    k_round<<<(unsigned)((n_p + 255) / 256), 256>>>(n_p, g->sep_Qs, g->sep_Qs32);
    k_round<<<(unsigned)((n_tr + 255) / 256), 256>>>(n_tr, g->sep_tr, g->sep_tr32);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    if ((e = synthesis_separable_prepare(g)) != cudaSuccess) return e;
  }
  const AzFold fold = az_fold(g);
  const int m1 = g->lmax + 1;
  A((void **)&g->sep_azf, (size_t)m1 * fold.cols * sizeof(double2));
  if (e != cudaSuccess) return e;
  k_fold_az<<<(m1 * fold.cols + 255) / 256, 256>>>(m1, fold, g->dph, fold_dph_low(g), (double2 *)g->sep_azf);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  // float64: the polar stage's sums and the folded rows in shared memory.
  // fp32: grids whose table and 16 padded rows of a shell fit 227 KB; the others
  // keep the dense contraction, whose fp32 sums round differently.  (Rows
  // (shell, j) are counted in 32 bits.)
  g->sep_ok = 0;
  const bool counted = (long long)grid_rows(g) * g->n_theta <= 1 << 30;
  const size_t tail_t = (size_t)(g->n_theta + 1) * sizeof(float2), limit = 227 * 1024;
  if (counted && theta_smem(g->n_theta, nt_pad, sizeof(double)) <= limit && phi64_rows(g) > 0) g->sep_ok |= 2;
  if (counted && (size_t)g->n_theta * nt_pad * sizeof(float) + tail_t <= limit &&
      theta_smem(g->n_theta, nt_pad, sizeof(float)) <= limit && (size_t)g->n_phi * (nt_pad + 20) * sizeof(float) <= limit)
    g->sep_ok |= 1;
  // the attribute belongs to the kernel, not to this grid: always the maximum
  for (auto f : {(const void *)k_sep_phi64, (const void *)k_sep_phi32<2>, (const void *)k_sep_phi32<4>, (const void *)k_sep_theta32<1>, (const void *)k_sep_theta32<2>,
                 (const void *)k_sep_theta32<4>, (const void *)k_sep_theta64, (const void *)k_sep_theta_partials})
    if ((e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  f == (const void *)k_sep_phi32<2> || f == (const void *)k_sep_phi32<4> ? 64 * 1024 : 227 * 1024)) != cudaSuccess)
      return e;
  return cudaSuccess;
}

size_t separable_theta_partials_smem(const yy_grid *g, int nt_pad) {
  return (size_t)kThetaShells * g->n_theta * (sizeof(float2) + 2 * sizeof(float) + (nt_pad + 1) * sizeof(float));
}

cudaError_t separable_theta_partials(yy_grid *g, SepThetaPartials a, cudaStream_t s) {
  a.n_theta = g->n_theta;
  a.n_lm = g->n_lm;
  a.lmax1 = g->lmax + 1;
  a.tb = g->sep_tb32;
  a.tb0 = (const float2 *)g->sep_tb0;
  a.A = g->A;
  const int S = kThetaShells;
  const size_t smem = separable_theta_partials_smem(g, a.nt_pad);
  if (smem > 227 * 1024) return cudaErrorInvalidConfiguration;
  k_sep_theta_partials<<<(grid_rows(g) + S - 1) / S, 256, smem, s>>>(a, grid_rows(g));
  note_launch(g, "k_sep_theta_partials", s);
  return cudaGetLastError();
}

cudaError_t separable_theta_f64(yy_grid *g, cudaStream_t s) {
  const int nt_pad = g->sep_nt_pad;
  return launch_kernel(g, "k_sep_theta64", k_sep_theta64, grid_rows(g), theta_threads(g->n_lm, 0),
                       theta_smem(g->n_theta, nt_pad, sizeof(double)), s, g->n_theta, g->n_lm, nt_pad, g->tbar, g->sep_F, g->A);
}

cudaError_t analysis_separable(yy_grid *g, const double *rho_yin, const double *rho_yang, bool fp64, cudaStream_t s) {
  const int nt_pad = g->sep_nt_pad, rows = grid_rows(g) * g->n_theta;
  if (fp64) {
    const int per = phi64_rows(g), m1 = g->lmax + 1;
    const SepPhi64 a = {rows, per, g->n_r, g->n_theta, g->n_phi, m1, nt_pad, az_fold(g), rho_yin, rho_yang, g->w,
                        (const double2 *)g->sep_azf, g->sep_F};
    const int threads = std::max(64, (per / kR64 * m1 + 31) / 32 * 32);   // one item per thread (672 at l_max 80)
    const cudaError_t e = launch_kernel(g, "k_sep_phi64", k_sep_phi64, (rows + per - 1) / per, threads, phi64_smem(a.fold, per), s, a);
    return e == cudaSuccess ? separable_theta_f64(g, s) : e;
  }
  const SepPhi32 a = {g->n_r, g->n_theta, g->n_phi, nt_pad, {rho_yin, rho_yang}, g->sep_w32, g->sep_az32, (float *)g->sep_F,
                      (float2 *)g->sep_F0};
  // rows per thread: four, or two where that leaves half of the loading warps without sums
  const int tg = nt_pad / kTT, R = kRows32 / 2 * tg <= 32 * kLoadWarps ? 2 : 4;
  const int threads = std::max(32 * kLoadWarps, (kRows32 / R * tg + 31) / 32 * 32);   // one item per thread (352 at l_max 80)
  const dim3 blocks((unsigned)((g->n_r * g->n_theta + kRows32 - 1) / kRows32), (unsigned)g->n_patch);
  const size_t table = 2 * (size_t)kPiece * nt_pad * sizeof(float);
  const cudaError_t e = launch_kernel(g, "k_sep_phi32", R == 2 ? k_sep_phi32<2> : k_sep_phi32<4>, blocks, threads, table, s, a);
  if (e != cudaSuccess) return e;
  // shells per block: as many as leave every SM a block (and fit two blocks per SM)
  const size_t shell = theta_smem(g->n_theta, nt_pad, sizeof(float));
  const int shells = grid_rows(g), mode_threads = theta_threads(g->n_lm, 32);
  auto polar = [&](auto k, int S) {
    return launch_kernel(g, "k_sep_theta32", k, (shells + S - 1) / S, mode_threads, S * shell, s, shells, g->n_theta, g->n_lm,
                         g->lmax + 1, nt_pad, g->sep_tb32, g->sep_tb0, (const float *)g->sep_F, (const float2 *)g->sep_F0, g->A);
  };
  if (shells >= 4 * g->sms && 4 * shell <= 113 * 1024) return polar(k_sep_theta32<4>, 4);
  if (shells >= 3 * g->sms && 2 * shell <= 113 * 1024) return polar(k_sep_theta32<2>, 2);
  return polar(k_sep_theta32<1>, 1);
}

}  // namespace yy
