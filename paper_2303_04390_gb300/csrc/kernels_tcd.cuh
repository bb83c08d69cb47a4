// FP64 kernels for 21..64 states (codon models) on the tensor cores.
//
// The FP64 pipe of this GPU issues half a lane per clock in each quarter of
// an SM, so a 61-state product on it costs 30 times what it costs in FP32.
// Here the contractions run on the tensor cores in exact integer arithmetic
// instead (the error-free slicing of Ozaki, Ogita, Oishi and Rump, Numer.
// Algorithms 59, 2012, in fixed point):
//
//   Each operand row is scaled by a power of two to magnitudes at most 1 and
//   written in fixed point with 62 fractional bits as eight signed base-256
//   digits, x = 2^e sum_i a_i 2^(-6 - 8 i), a_i in [-128, 127], the digits
//   stored as FP16 integers.  A digit product is an integer of at most 14
//   bits, and an MMA adds 64 of them, so the sums of all products a_i b_j with
//   one i + j = d <= 7 stay below 2^23 and accumulate exactly in FP32:
//   kind::f16 MMAs give the eight integers D_d = sum_{i + j = d} a_i . b_j
//   without any rounding.  The epilogue adds them in integer arithmetic,
//   sum_d D_d 256^(7 - d), and rounds once to FP64.
//
// What is dropped (digits past the 62nd bit, products with i + j > 7) is about
// 2^-59 of the product of the row's and the column's largest entries: an
// absolute error.  On a short branch P has entries of the order t, t^2 and t^3
// beside a diagonal near 1, and where the two sides of an internal branch
// disagree the site likelihood is one of those.  So the contractions take
// E = P - I = V diag(expm1) Vinv, whose rows and columns have scales of their
// own (of the order t), and the identity's part stays in FP64:
//   U = p + E p,   q_x = a_x + E' a_x.
// The error is then 2^-59 of E's entries times p, while the eigenvector route
// leaves one of about 2^-56 t in those entries themselves.  The matrix build
// and a_x Q, whose sums may be far below the largest product, are rounded at
// the 53rd bit of the sum instead of at a fixed place.  Measured: codons that
// differ by 1, 2 and 3 nucleotides across internal branches of 1e-8 to 2e-3 are
// as far from exact as FP64 products on the same eigenvectors are (with P in
// place of E: up to 1e8 times as far); simulated alignments, 20 to 61 taxa,
// mean branch lengths 0.002 to 0.1: gradient (2-norm) 1.2e-14 to 1.2e-13, 0.98
// to 1.01 times what FP64 products leave.  It costs 6% (61 taxa x 601 patterns
// x 4 categories 0.72 -> 0.76 ms): one FP64 addition per entry.
//
// The digits of slice i of the 128-row operand multiply the digits 0..7 - i
// of the 64-row operand, whose accumulators are adjacent TMEM columns: one
// MMA chain of N = 64 (8 - i) columns (at most 256 per instruction), 48 MMAs
// per contraction, 512 TMEM columns.
//
// Structure as in kernels_tc64.cuh (U form, per-category exponents, one CTA
// per 128-pattern tile, node and category), with FP64 vectors: the elementwise
// products, the dot products of Eq. 8 and the sums stay on the FP64 pipe.
//   post:  p_k = U_i o U_j, normalised per row,  U_k = p_k + p_k E_k'
//   pre:   a_x = q_k o U_y, den = a_x . U_x, num_x = gamma_r (a_x Q) . U_x,
//          q_x = a_x + a_x E_x  (a normalised per row)
//   a tip: U_x is column y of P_x and num_x = a_x . (column y of dP_x), from
//          FP64 tables; a tip with a partial vector multiplies them out.
#pragma once

#include <cuda_fp16.h>

namespace phylo {

constexpr int kTcdThreads = 512;
constexpr uint32_t kTcdA = 8 * 128 * 128;  // eight digit slices, 128 rows of 64
constexpr uint32_t kTcdB = kTcdDigits;     // eight digit slices, 64 rows
constexpr int kTcdLd = 66;                 // staging row (doubles), conflict-free
static_assert(128 * kTcdLd * 8 <= kTcdA, "staging fits in the operand buffer");
constexpr size_t kTcdSmem = 1024 + kTcdA + kTcdB;
constexpr uint32_t kTcdTab = 64 * 64 * 8;  // one FP64 table

// The digits' fixed point of x / 2^s, |x| <= 2^s, towards zero: x 2^(62 - s),
// plus the bias that makes every byte a digit + 128.
__device__ __forceinline__ unsigned long long tcd_fix(double x, int s) {
  const int hi = __double2hiint(x);
  const unsigned lo = (unsigned)__double2loint(x);
  // 2^62 <= m < 2^63; a zero or subnormal x is shifted out (k > 63)
  const unsigned long long m =
      ((unsigned long long)(((unsigned)hi & 0xfffffu) | 0x100000u) << 32 | lo) << 10;
  const int k = 1023 + s - ((hi >> 20) & 0x7ff);
  unsigned long long v;
  asm("shr.u64 %0, %1, %2;" : "=l"(v) : "l"(m), "r"(k));  // (shifts past 63 give 0)
  return (hi < 0 ? 0ull - v : v) + 0x8080808080808080ull;
}

// Digit slices of 8 consecutive elements (chunk j of row `row`), given in
// biased fixed point, of an operand at `op` with `slice` bytes per slice
// (128-byte rows, 128-byte swizzle).
__device__ __forceinline__ void tcd_put_fix(unsigned char* op, uint32_t slice, int row, int j,
                                            const unsigned long long (&t)[8]) {
  uint32_t h[8], l[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    h[i] = (uint32_t)(t[i] >> 32);
    l[i] = (uint32_t)t[i];
  }
  const uint32_t off = tc::b16_chunk(row, j);
  const __half2 bias = __floats2half2_rn(-1152.f, -1152.f);
#pragma unroll
  for (int s = 0; s < 8; ++s) {
    const int byte = 3 - (s & 3);
    uint32_t w[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const uint32_t a = s < 4 ? h[2 * i] : l[2 * i], b = s < 4 ? h[2 * i + 1] : l[2 * i + 1];
      // halves 1024 + digit + 128, exactly, less 1152
      const uint32_t u =
          (__byte_perm(a, b, byte | (4 + byte) << 8) & 0x00ff00ffu) | 0x64006400u;
      const __half2 v = __hadd2(*reinterpret_cast<const __half2*>(&u), bias);
      w[i] = *reinterpret_cast<const uint32_t*>(&v);
    }
    *reinterpret_cast<uint4*>(op + s * slice + off) = make_uint4(w[0], w[1], w[2], w[3]);
  }
}

__device__ __forceinline__ void tcd_put(unsigned char* op, uint32_t slice, int row, int j,
                                        const double (&x)[8], int s = 0) {
  unsigned long long t[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) t[i] = tcd_fix(x[i], s);
  tcd_put_fix(op, slice, row, j, t);
}

// The products V(s, m) e_m in fixed point without the FP64 pipe (a product
// there takes 64 clocks per warp; the 122-state matrix build 439 -> 406 us):
// x = m 2^(k - 63) with the sign apart, m in [2^63, 2^64) or zero.
struct __align__(16) TcdFactor {
  unsigned long long m;
  int k, neg;
};
constexpr int kTcdZero = -(1 << 20);  // exponent of a zero
__device__ __forceinline__ TcdFactor tcd_factor(double x) {
  const unsigned hi = (unsigned)__double2hiint(x);
  const unsigned lo = (unsigned)__double2loint(x);
  const int E = (hi >> 20) & 0x7ff;
  if (E == 0) return TcdFactor{0, kTcdZero, 0};  // (below 2^-1022: as zero)
  return TcdFactor{(unsigned long long)((hi & 0xfffffu) | 0x100000u) << 43 |
                       (unsigned long long)lo << 11,
                   E - 1023, (int)(hi >> 31)};
}
// Place of eigenvalue m's factor: the 8 lanes of a row read m = 8 j + i.
__device__ __forceinline__ int tcd_factor_at(int m) {
  return (m & ~63) | (m & 7) << 3 | (m >> 3 & 7);
}
// Exponent e with |v_i f_i| < 2^e over the row's 8 lanes; 0 for zeros.
__device__ __forceinline__ int tcd_products(const double (&v)[8], const TcdFactor* f, int j,
                                            TcdFactor (&p)[8]) {
  int k = kTcdZero;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const TcdFactor a = tcd_factor(v[i]), b = f[8 * i + j];
    p[i] = TcdFactor{__umul64hi(a.m, b.m), a.k + b.k, a.neg ^ b.neg};
    k = max(k, p[i].k);
  }
  k = max(k, __shfl_xor_sync(kFull, k, 1));
  k = max(k, __shfl_xor_sync(kFull, k, 2));
  k = max(k, __shfl_xor_sync(kFull, k, 4));
  return k < -4096 ? 0 : k + 2;
}
__device__ __forceinline__ void tcd_put(unsigned char* op, uint32_t slice, int row, int j,
                                        const TcdFactor (&p)[8], int e) {
  unsigned long long t[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) {  // |x| = m 2^(k - 62), times 2^(62 - e)
    unsigned long long v;
    asm("shr.u64 %0, %1, %2;" : "=l"(v) : "l"(p[i].m), "r"(e - p[i].k));  // >= 2
    t[i] = (p[i].neg ? 0ull - v : v) + 0x8080808080808080ull;
  }
  tcd_put_fix(op, slice, row, j, t);
}

// 64-bit shifts that give 0 past 63.
__device__ __forceinline__ unsigned long long tcd_shl(unsigned long long x, int k) {
  unsigned long long y;
  asm("shl.b64 %0, %1, %2;" : "=l"(y) : "l"(x), "r"(k));
  return y;
}
__device__ __forceinline__ unsigned long long tcd_shr(unsigned long long x, int k) {
  unsigned long long y;
  asm("shr.u64 %0, %1, %2;" : "=l"(y) : "l"(x), "r"(k));
  return y;
}

// D_d accumulators of one element -> sum_d D_d 2^(-12 - 8 d + scale).
// |D_d| <= 2^22 for d <= 4 (read from the float's bits), < 2^23 after.
// UNIT: the sum's magnitude is at most about 1 (tcd_sum_shift), and it is
// rounded once, at the 53rd bit or 2^-62, whichever is coarser; else it may
// reach 64 and is rounded at its 53rd bit.  A result below 2^-1022 is 0.
template <bool UNIT>
__device__ __forceinline__ double tcd_value(const float (&f)[8], int scale) {
  constexpr unsigned K = 0x4b400000u;  // bits of 1.5 2^23: D + K - K
  unsigned n[8];
#pragma unroll
  for (int d = 0; d < 5; ++d) n[d] = (unsigned)__float_as_int(f[d] + 12582912.f);
#pragma unroll
  for (int d = 5; d < 8; ++d) n[d] = (unsigned)__float2int_rn(f[d]);
  const int t01 = (int)(n[0] * 256u + n[1] - K * 257u), t23 = (int)(n[2] * 256u + n[3] - K * 257u);
  const int t45 = (int)(n[4] * 256u + n[5] - K * 256u), t67 = (int)(n[6] * 256u + n[7]);
  // the sum is top 2^32 + low in units of 2^-68
  const long long top = (long long)t01 * 65536 + t23, low = (long long)t45 * 65536 + t67;
  bool neg;
  unsigned long long X;  // the magnitude is X 2^-z, X in [2^63, 2^64) unless 0
  int z;
  if constexpr (UNIT) {
    const long long V = (top << 26) + (low >> 6);
    neg = V < 0;
    const unsigned long long m = neg ? 0ull - (unsigned long long)V : (unsigned long long)V;
    const int lz = __clzll((long long)m);
    X = m << (lz & 63);
    z = 62 + lz;
  } else {
    const long long t = top + (low >> 32);
    neg = t < 0;  // (the complement is one unit short of the magnitude)
    unsigned long long h = (unsigned long long)(neg ? ~t : t);
    unsigned long long l = (unsigned long long)(neg ? ~(unsigned)low : (unsigned)low) << 32;
    z = 36;
    if (h == 0) {  // less than 2^-36
      h = l;
      l = 0;
      z = 100;
    }
    const int lz = __clzll((long long)h);
    X = tcd_shl(h, lz) | tcd_shr(l, 64 - lz);  // (lz > 0 where l != 0)
    z += lz;
  }
  const int E = 1023 + 63 - z + scale;
  if (X == 0 || E <= 0) return 0.0;
  unsigned long long bits = (X >> 11) + ((X >> 10) & 1u);  // (carries into the exponent)
  bits += (unsigned long long)((unsigned)(E - 1) | (neg ? 0x800u : 0u)) << 52;
  return __longlong_as_double((long long)bits);
}

// Instruction descriptor: F16 x F16 -> FP32, both operands K-major, M = 128.
__host__ __device__ constexpr uint32_t tcd_idesc(int N) {
  return (1u << 4) | ((uint32_t)(N >> 3) << 17) | ((128u >> 4) << 24);
}

// Every digit product with i + j <= 7 into (or added to) the 512 columns at
// `tmem`.  One thread issues.
__device__ __forceinline__ void tcd_mma(uint32_t tmem, uint32_t A, uint32_t B,
                                        bool accumulate = false) {
#pragma unroll
  for (int i = 0; i < 8; ++i) {
#pragma unroll
    for (int n0 = 0; n0 < 64 * (8 - i); n0 += 256) {
      const int N = 64 * (8 - i) - n0 < 256 ? 64 * (8 - i) - n0 : 256;
#pragma unroll
      for (int kk = 0; kk < 4; ++kk)
        tc::mma_bf16(tmem + 64 * i + n0, tc::desc(A + i * 128 * 128 + kk * 32),
                     tc::desc(B + n0 * 128 + kk * 32), tcd_idesc(N),
                     (accumulate || (i | kk)) ? 1 : 0);
    }
  }
}

// 4 accumulator columns of this thread's row from each of the eight sums.
__device__ __forceinline__ void tcd_ld(uint32_t taddr, float (&v)[4][8]) {
  uint32_t r[8][4];
#pragma unroll
  for (int d = 0; d < 8; ++d)
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[d][0]), "=r"(r[d][1]), "=r"(r[d][2]), "=r"(r[d][3])
                 : "r"(taddr + 64 * d));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int d = 0; d < 8; ++d)
#pragma unroll
    for (int i = 0; i < 4; ++i) v[i][d] = __uint_as_float(r[d][i]);
}

// Cooperative layout: in iteration it (0, 1) lane l of warp w handles row
// 64 it + 4 w + l / 8 and elements 8 (l % 8) .. + 7.
__device__ __forceinline__ int tcd_row(int it) {
  return 64 * it + 4 * (int)(threadIdx.x >> 5) + (int)((threadIdx.x & 31) >> 3);
}

__device__ __forceinline__ void tcd_load8(const double* src, double (&v)[8]) {
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const double2 x = reinterpret_cast<const double2*>(src)[i];
    v[2 * i] = x.x;
    v[2 * i + 1] = x.y;
  }
}

// Divides a row (8 lanes) by the power of two that brings its largest
// magnitude into [1/2, 1); returns the exponent, 0 for a zero row.  Only
// entries below 2^-64 of the largest can be flushed.  A NaN or infinity raises
// ERR_ZERO_PARTIAL.  FP64 products are kept out of it: exponent fields.
__device__ __forceinline__ int tcd_row_max(const double (&x)[8]) {
  int m = 0;
#pragma unroll
  for (int i = 0; i < 8; ++i) m = max(m, tree_abs_bits(x[i]));
  m = max(m, __shfl_xor_sync(kFull, m, 1));
  m = max(m, __shfl_xor_sync(kFull, m, 2));
  return max(m, __shfl_xor_sync(kFull, m, 4)) >> 20;
}
__device__ __forceinline__ int tcd_normalise(double (&x)[8], bool valid, int* err) {
  int E = tcd_row_max(x), shift = 0;
  if (__any_sync(kFull, valid && E < 64)) {  // close to or among the subnormals
    if (valid && E < 64) {
      shift = -128;
#pragma unroll
      for (int i = 0; i < 8; ++i) x[i] *= 0x1p128;
    }
    E = tcd_row_max(x);
  }
  if (valid && E == 0x7ff) atomicOr(err, ERR_ZERO_PARTIAL);
  if (E == 0) return 0;
  const int e = E - 1022;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int hi = __double2hiint(x[i]), field = (hi >> 20) & 0x7ff;
    const bool keep = field > max(e, 0);
    x[i] = __hiloint2double(keep ? hi - (e << 20) : 0, keep ? __double2loint(x[i]) : 0);
  }
  return e + shift;
}

// s with sum |x| <= 2^s (about) over a normalised row.
__device__ __forceinline__ int tcd_sum_shift(const double (&x)[8]) {
  unsigned sum = 0;  // in units of 2^-20
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int hi = __double2hiint(x[i]), k = 1023 - ((hi >> 20) & 0x7ff);
    sum += k > 20 ? 0u : (((unsigned)hi & 0xfffffu) | 0x100000u) >> k;
  }
  sum += __shfl_xor_sync(kFull, sum, 1);
  sum += __shfl_xor_sync(kFull, sum, 2);
  sum += __shfl_xor_sync(kFull, sum, 4);
  return sum <= 1u << 20 ? 0 : 12 - __clz(sum - 1);
}

// Row sums over the 8 lanes of both iterations' rows: 3 additions for two.
// Lane j even returns iteration 0's sum, odd iteration 1's.
__device__ __forceinline__ double tcd_row_sums(double s0, double s1) {
  const bool odd = threadIdx.x & 1;
  double s = (odd ? s1 : s0) + __shfl_xor_sync(kFull, odd ? s0 : s1, 1);
  s += __shfl_xor_sync(kFull, s, 2);
  return s + __shfl_xor_sync(kFull, s, 4);
}

__device__ __forceinline__ double tcd_dot8(const double (&x)[8], const double (&y)[8]) {
  double s = x[0] * y[0];
#pragma unroll
  for (int i = 1; i < 8; ++i) s = fma(x[i], y[i], s);
  return s;
}

__device__ __forceinline__ const unsigned char* tcd_unit(const LevelArgs<double>& a, int b,
                                                         int r) {
  return reinterpret_cast<const unsigned char*>(a.P) + ((size_t)b * a.n_cat + r) * kTcdUnitBytes;
}

// Rows of a child's U in the cooperative layout (zero past the last pattern);
// y: a compact tip's states, -1 otherwise; e: an internal child's exponents.
// With `dp` the same for dP (tips only): column y of dP, or dP v.
__device__ __forceinline__ void tcd_child(const LevelArgs<double>& a, int b, bool compact, int r,
                                          int c0, bool dp, double (&u)[2][8], int (&y)[2],
                                          int (&e)[2]) {
  const int C = a.n_patterns, R = a.n_cat, S = a.n_states, j = threadIdx.x & 7;
#pragma unroll
  for (int it = 0; it < 2; ++it) {
    const int c = c0 + tcd_row(it);
    y[it] = -1;
    e[it] = 0;
#pragma unroll
    for (int i = 0; i < 8; ++i) u[it][i] = 0.0;
    if (c >= C) continue;
    if (b >= a.n_tips) {
      const size_t slot = (size_t)(b - a.n_tips);
      tcd_load8(a.post + ((slot * C + c) * R + r) * 64 + 8 * j, u[it]);
      e[it] = a.escale[(slot * R + r) * a.escale_stride + c];
      continue;
    }
    const double* tab = reinterpret_cast<const double*>(tcd_unit(a, b, r) + (dp ? kTcdTab : 0));
    if (compact) {
      y[it] = a.tip_states[(size_t)b * a.state_stride + c];
      if (y[it] < S) {
        tcd_load8(tab + y[it] * 64 + 8 * j, u[it]);
      } else {  // a gap: all ones, derivative 0
#pragma unroll
        for (int i = 0; i < 8; ++i) u[it][i] = !dp && 8 * j + i < S ? 1.0 : 0.0;
      }
      continue;
    }
    const double* v = a.tip_partials + ((size_t)b * C + c) * 64;
    for (int t = 0; t < S; ++t) {
      double row[8];
      tcd_load8(tab + t * 64 + 8 * j, row);
      const double vt = v[t];
#pragma unroll
      for (int i = 0; i < 8; ++i) u[it][i] = fma(row[i], vt, u[it][i]);
    }
  }
}

// Staging rows [128][kTcdLd], pairs of doubles: place of pair c of a row (of
// 32), so that the eight lanes of a row write their own pairs without conflict.
__device__ __forceinline__ int tcd_pair(int c) { return c ^ (c >> 3 & 3); }
__device__ __forceinline__ double2* tcd_at(double* st, int row, int c) {
  return reinterpret_cast<double2*>(st + row * kTcdLd) + tcd_pair(c);
}

struct TcdBars {
  uint64_t tma, mma;
  uint32_t tmem;
};

__device__ __forceinline__ void tcd_copy_b(unsigned char* B, const unsigned char* src,
                                           uint64_t* bar) {
  mbar_expect_tx(bar, kTcdB);
  for (uint32_t o = 0; o < kTcdB; o += 32768) bulk_g2s(B + o, src + o, 32768, bar);
}

// This thread's accumulator row and its 16 columns.
__device__ __forceinline__ int tcd_acc_row() {
  return 32 * ((int)(threadIdx.x >> 5) & 3) + (int)(threadIdx.x & 31);
}
__device__ __forceinline__ int tcd_acc_col() { return 16 * (int)(threadIdx.x >> 7); }
__device__ __forceinline__ uint32_t tcd_acc_addr(uint32_t tmem) {
  return tmem + ((uint32_t)(32 * ((threadIdx.x >> 5) & 3)) << 16) + tcd_acc_col();
}

// x + x E' -> global rows, from the rows x in the cooperative layout and the
// accumulators of x E' (column exponents ecol), by way of the staging rows.
// (Adding x on the way from there to the rows, straight from its registers,
// saves a pass over the staging but not the stores' coalescing: 0.79 ms
// against 0.76 for 61 taxa x 601 patterns.)
__device__ __forceinline__ void tcd_store_sum(double* st, const double (&x)[2][8], uint32_t tmem,
                                              const int* ecol, double* base, size_t stride, int c0,
                                              int C) {
  const int lane = threadIdx.x & 31, j = threadIdx.x & 7, col = tcd_acc_col();
#pragma unroll
  for (int it = 0; it < 2; ++it)
#pragma unroll
    for (int i = 0; i < 4; ++i)
      *tcd_at(st, tcd_row(it), 4 * j + i) = make_double2(x[it][2 * i], x[it][2 * i + 1]);
  __syncthreads();
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    float f[4][8];
    tcd_ld(tcd_acc_addr(tmem) + 4 * q, f);
#pragma unroll
    for (int i = 0; i < 4; i += 2) {
      const int c = col + 4 * q + i;
      double2* p = tcd_at(st, tcd_acc_row(), c >> 1);
      const double2 v = *p;
      *p = make_double2(v.x + tcd_value<true>(f[i], ecol[c]),
                        v.y + tcd_value<true>(f[i + 1], ecol[c + 1]));
    }
  }
  __syncthreads();
  for (int row = threadIdx.x >> 5; row < 128; row += kTcdThreads / 32) {
    if (c0 + row >= C) return;
    reinterpret_cast<double2*>(base + (size_t)(c0 + row) * stride)[lane] = *tcd_at(st, row, lane);
  }
}

// ---------------------------------------------------------------------------
// Matrices (Eq. 1): E = P - I = V diag(expm1) Vinv of two (branch, category)
// units per CTA (64 rows each), the rows V diag(e) sliced here, Vinv's digits
// from the host.  Internal branches get the digits of E and of E', every row
// with its own exponent, tips the FP64 tables P' and dP' (a second contraction
// with gamma lambda e^x).
// ---------------------------------------------------------------------------
template <typename T>  // double only
__global__ void __launch_bounds__(kTcdThreads) pmat_tcd_kernel(PmatArgs a) {
  extern __shared__ unsigned char smraw[];
  unsigned char* A = align1024(smraw);
  unsigned char* B = A + kTcdA;
  double* stage = reinterpret_cast<double*>(A);
  __shared__ TcdBars bars;
  __shared__ TcdFactor ex[2][64], dx[2][64];
  __shared__ int erow[128], ecol[64];
  const int tid = threadIdx.x, warp = tid >> 5, j = tid & 7;
  const int S = a.n_states, R = a.n_cat, units = a.n_branches * R;
  const int u0 = 2 * blockIdx.x;
  pdl_release();
  if (tid == 0) {
    mbar_init_fenced(&bars.tma, 1);
    mbar_init_fenced(&bars.mma, 1);
    tcd_copy_b(B, static_cast<const unsigned char*>(a.vdigits), &bars.tma);
  }
  if (tid < 64) ecol[tid] = reinterpret_cast<const int*>(
      static_cast<const unsigned char*>(a.vdigits) + kTcdB)[tid];
  if (tid < 128) {
    const int h = tid >> 6, m = tid & 63, unit = u0 + h;
    double e = 0.0, de = 0.0;
    if (unit < units && m < S) {
      double t = a.t[unit / R];
      if (!(t >= 0.0) || !isfinite(t)) {
        if (m == 0 && unit % R == 0) atomicOr(a.err, ERR_BAD_LENGTH);
        t = 0.0;
      }
      const double g = a.rates[unit % R], x = a.lambda[m] * g * t;
      e = expm1(x);
      if (unit / R < a.n_tips) de = g * a.lambda[m] * exp(x);
    }
    ex[h][tcd_factor_at(m)] = tcd_factor(e);
    dx[h][tcd_factor_at(m)] = tcd_factor(de);
  }
  if (warp == 0) tc::alloc(&bars.tmem, 512);
  __syncthreads();
  tc::fence_after();
  const uint32_t tmem = bars.tmem;
  uint32_t ptma = 0, pmma = 0;
  int pend_tma = -1, pend_mma = -1;
  const bool tips = u0 / R < a.n_tips;  // (a pair's first unit has the smaller branch)
  bool ok = true;
  for (int d = 0; d < (tips ? 2 : 1) && ok; ++d) {
#pragma unroll
    for (int it = 0; it < 2; ++it) {
      const int row = tcd_row(it), h = row >> 6, s = row & 63;
      double v[8];
      TcdFactor x[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const int m = 8 * j + i;
        v[i] = s < S && m < S ? a.V[s * S + m] : 0.0;
      }
      const int e = tcd_products(v, (d ? dx : ex)[h], j, x);
      if (j == 0) erow[row] = e;
      tcd_put(A, 128 * 128, row, j, x, e);
    }
    tc::fence_smem_for_async();
    if (d == 0) ok = tc_block_wait(&bars.tma, ptma, pend_tma, a.err);
    else __syncthreads();
    if (!ok) break;
    if (tid == 0) {
      tc::fence_after();
      tcd_mma(tmem, smem_addr(A), smem_addr(B));
      tc::commit(&bars.mma);
    }
    ok = tc_block_wait(&bars.mma, pmma, pend_mma, a.err);
    if (!ok) break;
    const int row = tcd_acc_row(), s = row & 63;
    const bool one = d == 0 && (u0 + (row >> 6)) / R < a.n_tips;  // a tip's P, not E
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      float f[4][8];
      const int t0 = tcd_acc_col() + 4 * q;
      tcd_ld(tcd_acc_addr(tmem) + 4 * q, f);
      double v[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        v[i] = tcd_value<false>(f[i], erow[row] + ecol[t0 + i]);
        if (one && s == t0 + i && s < S) v[i] += 1.0;
      }
#pragma unroll
      for (int i = 0; i < 2; ++i)
        *reinterpret_cast<double2*>(stage + row * kTcdLd + t0 + 2 * i) =
            make_double2(v[2 * i], v[2 * i + 1]);
    }
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    for (int hh = 0; hh < 2; ++hh) {
      const int unit = u0 + hh;
      if (unit >= units) continue;
      const bool tip = unit / R < a.n_tips;
      unsigned char* out = static_cast<unsigned char*>(a.P) + (size_t)unit * kTcdUnitBytes;
      const double* st = stage + hh * 64 * kTcdLd;
      if (tip) {  // row y of the table = column y
        double* tab = reinterpret_cast<double*>(out + (d ? kTcdTab : 0));
        for (int i = tid; i < 64 * 64; i += kTcdThreads)
          tab[i] = st[(i & 63) * kTcdLd + (i >> 6)];
      } else if (d == 0) {
        // one 8-element chunk of E and one of E' per thread
        const int r8 = tid >> 3;
        double x[8], y[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          x[i] = st[r8 * kTcdLd + 8 * j + i];
          y[i] = st[(8 * j + i) * kTcdLd + r8];
        }
        const int ep = tcd_normalise(x, r8 < S, a.err);
        const int sp = tcd_sum_shift(x);
        tcd_put(out, 64 * 128, r8, j, x, sp);
        const int e = tcd_normalise(y, r8 < S, a.err);
        const int sy = tcd_sum_shift(y);
        tcd_put(out + kTcdB, 64 * 128, r8, j, y, sy);
        if (j == 0) {
          reinterpret_cast<int*>(out + 2 * kTcdB)[r8] = e + sy;
          reinterpret_cast<int*>(out + 2 * kTcdB)[64 + r8] = ep + sp;
        }
      }
    }
    __syncthreads();  // the staging is the next contraction's operand
  }
  if (tid == 0) {  // bounded drain of whatever a timeout left in flight
    if (pend_tma >= 0) (void)mbar_wait(&bars.tma, (uint32_t)pend_tma);
    if (pend_mma >= 0) (void)mbar_wait(&bars.mma, (uint32_t)pend_mma);
  }
  tc::fence_before();
  __syncthreads();
  if (warp == 0) tc::dealloc(tmem, 512);
}

// ---------------------------------------------------------------------------
// Post-order level (Eq. 2), every level but the root's.
// ---------------------------------------------------------------------------
template <typename T>  // double only
__global__ void __launch_bounds__(kTcdThreads) post_tcd_kernel(LevelArgs<T> a) {
  extern __shared__ unsigned char smraw[];
  unsigned char* A = align1024(smraw);
  unsigned char* B = A + kTcdA;
  double* stage = reinterpret_cast<double*>(A);
  __shared__ TcdBars bars;
  __shared__ int erow[64];  // exponents of E_k's rows
  const int tid = threadIdx.x, warp = tid >> 5, j = tid & 7;
  const int R = a.n_cat, C = a.n_patterns;
  const int4 d = a.level_desc[blockIdx.y];
  const int k = d.x, r = blockIdx.z, c0 = blockIdx.x * 128;
  const size_t slot = (size_t)(k - a.n_tips);
  auto issue = [&] {
    if (tid != 0) return;
    mbar_init_fenced(&bars.tma, 1);
    mbar_init_fenced(&bars.mma, 1);
    tcd_copy_b(B, tcd_unit(a, k, r), &bars.tma);  // digits of E_k
  };
  if (a.mats_ready) issue();
  pdl_wait_and_release();
  if (!a.mats_ready) issue();
  if (tid < 64) erow[tid] = reinterpret_cast<const int*>(tcd_unit(a, k, r) + 2 * kTcdB)[64 + tid];
  if (warp == 0) tc::alloc(&bars.tmem, 512);
  double p[2][8], u[2][8];
  int y[2], e[2], e1[2];
  tcd_child(a, d.y, d.w & kDescFlagCompact0, r, c0, false, p, y, e);
  tcd_child(a, d.z, d.w & kDescFlagCompact1, r, c0, false, u, y, e1);
#pragma unroll
  for (int it = 0; it < 2; ++it) {
    const int row = tcd_row(it), c = c0 + row;
#pragma unroll
    for (int i = 0; i < 8; ++i) p[it][i] *= u[it][i];
    const int er = tcd_normalise(p[it], c < C, a.err);
    tcd_put(A, 128 * 128, row, j, p[it]);
    if (j == 0 && c < C) a.escale[(slot * R + r) * a.escale_stride + c] = e[it] + e1[it] + er;
  }
  tc::fence_smem_for_async();
  __syncthreads();  // barriers initialised, TMEM allocated, A written
  tc::fence_after();
  const uint32_t tmem = bars.tmem;
  uint32_t ptma = 0, pmma = 0;
  int pend_tma = -1, pend_mma = -1;
  bool ok = tc_block_wait(&bars.tma, ptma, pend_tma, a.err);
  if (ok) {
    if (tid == 0) {
      tc::fence_after();
      tcd_mma(tmem, smem_addr(A), smem_addr(B));
      tc::commit(&bars.mma);
    }
    ok = tc_block_wait(&bars.mma, pmma, pend_mma, a.err);
  }
  if (ok) {  // U_k = p_k + E_k p_k
    tcd_store_sum(stage, p, tmem, erow, a.post + (slot * C * R + r) * 64, (size_t)R * 64, c0, C);
  }
  if (tid == 0) {
    if (pend_tma >= 0) (void)mbar_wait(&bars.tma, (uint32_t)pend_tma);
    if (pend_mma >= 0) (void)mbar_wait(&bars.mma, (uint32_t)pend_mma);
  }
  tc::fence_before();
  __syncthreads();
  if (warp == 0) tc::dealloc(tmem, 512);
}

// Eq. 3 at the root from its children's U: 8 lanes per pattern, the
// categories summed relative to the largest exponent.
template <typename T>  // double only
__global__ void __launch_bounds__(kTcdThreads) root_tcd_kernel(LevelArgs<T> a) {
  pdl_wait_and_release();
  __shared__ double lred[kTcdThreads / 32];
  const int R = a.n_cat, C = a.n_patterns, S = a.n_states;
  const int tid = threadIdx.x, lane = tid & 31, j = tid & 7, c0 = blockIdx.x * 128;
  const int4 d = a.level_desc[0];
  double lsum[2] = {0.0, 0.0};
  int lexp[2] = {INT_MIN / 2, INT_MIN / 2};
  for (int r = 0; r < R; ++r) {
    double p[2][8], u[2][8];
    int y[2], e[2], e1[2];
    tcd_child(a, d.y, d.w & kDescFlagCompact0, r, c0, false, p, y, e);
    tcd_child(a, d.z, d.w & kDescFlagCompact1, r, c0, false, u, y, e1);
#pragma unroll
    for (int it = 0; it < 2; ++it) {
      double s = 0.0;
#pragma unroll
      for (int i = 0; i < 8; ++i)
        if (8 * j + i < S) s = fma(a.root_pi[8 * j + i], p[it][i] * u[it][i], s);
      s += __shfl_xor_sync(kFull, s, 1);
      s += __shfl_xor_sync(kFull, s, 2);
      s += __shfl_xor_sync(kFull, s, 4);
      if (s != 0.0) {  // running sum relative to the largest exponent
        const double t = a.cat_w[r] * s;
        const int E = e[it] + e1[it];
        if (E > lexp[it]) {
          lsum[it] = ldexp(lsum[it], max(lexp[it] - E, -2000)) + t;
          lexp[it] = E;
        } else {
          lsum[it] += ldexp(t, max(E - lexp[it], -2000));
        }
      }
    }
  }
  double term = 0.0;
#pragma unroll
  for (int it = 0; it < 2; ++it) {
    const int c = c0 + tcd_row(it);
    if (c >= C || j != 0) continue;
    if (!(lsum[it] > 0.0) || !isfinite(lsum[it])) atomicOr(a.err, ERR_ZERO_PARTIAL);
    term += a.pattern_w[c] * (log(lsum[it]) + (double)lexp[it] * 0.69314718055994530942);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) term += __shfl_down_sync(kFull, term, o);
  if (lane == 0) lred[tid >> 5] = term;
  __syncthreads();
  if (tid == 0) {
    double l = 0.0;
    for (int w = 0; w < kTcdThreads / 32; ++w) l += lred[w];
    a.lpart[blockIdx.x] = l;
  }
}

// x 2^e, e <= 0 or small.
__device__ __forceinline__ double tcd_scale(double x, int e) {
  return e >= -1022 && e <= 1023 ? x * __hiloint2double((1023 + e) << 20, 0) : ldexp(x, e);
}

// ---------------------------------------------------------------------------
// Pre-order level (Eq. 4) with the per-category Eq. 8 terms: one CTA per
// (tile, node k, category r, child x); blockIdx.z = 2 r + x.  (The FP32 path's
// units, which form a tip's numerator in its sibling's CTA, lost here: the
// elementwise FP64 products bound a CTA, and the tips' are better on SMs of
// their own: pre-order of 64 taxa x 570 patterns 0.46 -> 0.57 ms.)  rterm holds
// {w_r num_i, w_r num_j, w_r den, exponent} per (node, pattern, category).
// ---------------------------------------------------------------------------
template <typename T>  // double only
__global__ void __launch_bounds__(kTcdThreads) pre_tcd_kernel(LevelArgs<T> a) {
  extern __shared__ unsigned char smraw[];
  unsigned char* A = align1024(smraw);
  unsigned char* B = A + kTcdA;
  double* stage = reinterpret_cast<double*>(A);
  __shared__ TcdBars bars;
  __shared__ double nums[4][128];
  __shared__ int ecol[64], ecol_p[64];  // column exponents of Q and E_x
  const int tid = threadIdx.x, warp = tid >> 5, j = tid & 7;
  const int R = a.n_cat, C = a.n_patterns, S = a.n_states;
  const int4 d = a.level_desc[blockIdx.y];
  const int k = d.x, x = (int)(blockIdx.z & 1), r = (int)(blockIdx.z >> 1);
  const int bx = x ? d.z : d.y, by = x ? d.y : d.z;
  const bool cx = d.w & (x ? kDescFlagCompact1 : kDescFlagCompact0);
  const bool cy = d.w & (x ? kDescFlagCompact0 : kDescFlagCompact1);
  const bool internal = bx >= a.n_tips;  // only these need contractions
  const size_t kslot = (size_t)(k - a.n_tips), xslot = (size_t)(bx - a.n_tips);
  const int c0 = blockIdx.x * 128, estr = a.escale_stride;
  if (internal) {  // Q' and its digits are host-written
    if (tid == 0) {
      mbar_init_fenced(&bars.tma, 1);
      mbar_init_fenced(&bars.mma, 1);
      tcd_copy_b(B, a.qt, &bars.tma);
    }
    if (tid < 64) ecol[tid] = reinterpret_cast<const int*>(a.qt + kTcdB)[tid];
  }
  // The matrices and the children's U are read before the wait: the matrix
  // build and the post-order pass, which ended with its root level, are at
  // least one launch back; only q_k comes from the launch before.
  if (internal && tid < 64)
    ecol_p[tid] = reinterpret_cast<const int*>(tcd_unit(a, bx, r) + 2 * kTcdB)[tid];
  double av[2][8], u[2][8];
  int y[2], ey[2], ex[2], eq[2];
  tcd_child(a, by, cy, r, c0, false, u, y, ey);
  pdl_wait_and_release();
  if (internal && warp == 0) tc::alloc(&bars.tmem, 512);
#pragma unroll
  for (int it = 0; it < 2; ++it) {  // a_x = q_k o U_y
    const int c = c0 + tcd_row(it);
    eq[it] = 0;
    if (k == a.root) {
#pragma unroll
      for (int i = 0; i < 8; ++i) av[it][i] = 8 * j + i < S ? a.root_pi[8 * j + i] : 0.0;
    } else if (c < C) {
      tcd_load8(a.pre + ((kslot * C + c) * R + r) * 64 + 8 * j, av[it]);
      eq[it] = a.pre_escale[(kslot * R + r) * estr + c];
    } else {
#pragma unroll
      for (int i = 0; i < 8; ++i) av[it][i] = 0.0;
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) av[it][i] *= u[it][i];
  }
  double* rt = static_cast<double*>(a.rterm);
  const double wr = a.cat_w[r];
  const int mit = tid & 1;  // the iteration whose row sum this lane gets
  const int crow = c0 + tcd_row(0) + 64 * mit;
  const bool mine = (j >> 1) == 0 && crow < C;  // lanes j = 0, 1 write
  double* mine_t = rt + ((kslot * C + (mine ? crow : 0)) * R + r) * 4;
  if (x == 0 || !internal) {
    if (x == 0) {  // den = a_x . U_x
      tcd_child(a, bx, cx, r, c0, false, u, y, ex);
      const double s = tcd_row_sums(tcd_dot8(av[0], u[0]), tcd_dot8(av[1], u[1]));
      if (mine) {
        mine_t[2] = wr * s;
        mine_t[3] = (double)(mit ? eq[1] + ex[1] + ey[1] : eq[0] + ex[0] + ey[0]);
      }
    }
    if (!internal) {  // num_x = a_x . (column of dP_x, or dP_x v)
      tcd_child(a, bx, cx, r, c0, true, u, y, ex);
      const double s = tcd_row_sums(tcd_dot8(av[0], u[0]), tcd_dot8(av[1], u[1]));
      if (mine) mine_t[x] = wr * s;
      return;  // block-uniform: no barrier, copy or TMEM is in use
    }
  }
  // ---- internal child: W_x = a_x Q, q_x = a_x + a_x E_x, a_x normalised per row ----
  int ea[2];
#pragma unroll
  for (int it = 0; it < 2; ++it) {
    const int row = tcd_row(it), c = c0 + row;
    ea[it] = tcd_normalise(av[it], c < C, a.err);
    tcd_put(A, 128 * 128, row, j, av[it]);
    if (j == 0 && c < C)
      a.pre_escale[(xslot * R + r) * estr + c] = ea[it] + eq[it] + ey[it];
  }
  tc::fence_smem_for_async();
  __syncthreads();  // barriers initialised, TMEM allocated, A written
  tc::fence_after();
  const uint32_t tmem = bars.tmem;
  uint32_t ptma = 0, pmma = 0;
  int pend_tma = -1, pend_mma = -1;
  bool ok = tc_block_wait(&bars.tma, ptma, pend_tma, a.err);
  if (ok) {
    if (tid == 0) {
      tc::fence_after();
      tcd_mma(tmem, smem_addr(A), smem_addr(B));
      tc::commit(&bars.mma);
    }
    ok = tc_block_wait(&bars.mma, pmma, pend_mma, a.err);
  }
  const int arow = tcd_acc_row(), acol = tcd_acc_col();
  if (ok) {
    // Q's digits have been read: E_x' takes their place
    if (tid == 0) tcd_copy_b(B, tcd_unit(a, bx, r) + kTcdB, &bars.tma);
    const int c = c0 + arow;
    const double* ux = a.post + ((xslot * C + (c < C ? c : 0)) * R + r) * 64 + acol;
    double num = 0.0;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const double2 u0 = reinterpret_cast<const double2*>(ux)[2 * q],
                    u1 = reinterpret_cast<const double2*>(ux)[2 * q + 1];
      const double uu[4] = {u0.x, u0.y, u1.x, u1.y};
      float f[4][8];
      tcd_ld(tcd_acc_addr(tmem) + 4 * q, f);
#pragma unroll
      for (int i = 0; i < 4; ++i)
        num = fma(tcd_value<false>(f[i], ecol[acol + 4 * q + i]), uu[i], num);
    }
    nums[acol >> 4][arow] = num;
    tc::fence_before();
    ok = tc_block_wait(&bars.tma, ptma, pend_tma, a.err);  // (a block barrier)
  }
  if (ok) {
    if (tid == 0) {
      tc::fence_after();
      tcd_mma(tmem, smem_addr(A), smem_addr(B));
      tc::commit(&bars.mma);
    }
    if (mine) {
      const int row = crow - c0;
      const double s = (nums[0][row] + nums[1][row]) + (nums[2][row] + nums[3][row]);
      mine_t[x] = tcd_scale(wr * a.rates[r] * s, mit ? ea[1] : ea[0]);
    }
    ok = tc_block_wait(&bars.mma, pmma, pend_mma, a.err);
  }
  if (ok) {
    tcd_store_sum(stage, av, tmem, ecol_p, a.pre + (xslot * C * R + r) * 64, (size_t)R * 64, c0,
                  C);
  }
  if (tid == 0) {
    if (pend_tma >= 0) (void)mbar_wait(&bars.tma, (uint32_t)pend_tma);
    if (pend_mma >= 0) (void)mbar_wait(&bars.mma, (uint32_t)pend_mma);
  }
  tc::fence_before();
  __syncthreads();
  if (warp == 0) tc::dealloc(tmem, 512);
}

// Eq. 8 ratios and their per-tile sums (Eq. 7), from the per-category terms.
template <typename T>  // double only
__global__ void __launch_bounds__(128) ratio_tcd_kernel(LevelArgs<T> a) {
  pdl_wait_and_release();
  __shared__ double red[4][2];
  const int R = a.n_cat, C = a.n_patterns;
  const size_t slot = blockIdx.y;
  const int2 ch = a.children[a.n_tips + (int)slot];
  const int c = blockIdx.x * 128 + threadIdx.x;
  double gi = 0.0, gj = 0.0;
  if (c < C) {
    const double2* src = static_cast<const double2*>(a.rterm) + (slot * C + c) * R * 2;
    double Ni = 0.0, Nj = 0.0, D = 0.0;
    int g = INT_MIN / 2;
    for (int r = 0; r < R; ++r) {
      const double2 n = src[2 * r], de = src[2 * r + 1];
      // a category whose terms all vanish carries an arbitrary exponent
      if (n.x == 0.0 && n.y == 0.0 && de.x == 0.0) continue;
      const int E = (int)de.y;
      if (E > g) {
        const int s = max(g - E, -2000);
        Ni = tcd_scale(Ni, s) + n.x;
        Nj = tcd_scale(Nj, s) + n.y;
        D = tcd_scale(D, s) + de.x;
        g = E;
      } else {
        const int s = max(E - g, -2000);
        Ni += tcd_scale(n.x, s);
        Nj += tcd_scale(n.y, s);
        D += tcd_scale(de.x, s);
      }
    }
    if (!(D > 0.0) || !isfinite(D)) {
      atomicOr(a.err, ERR_BAD_RATIO);
    } else {
      gi = a.pattern_wt[c] * (Ni / D);
      gj = a.pattern_wt[c] * (Nj / D);
    }
  }
  block_sum2<128>(gi, gj, red);
  if (threadIdx.x == 0) {
    a.gpart[(size_t)ch.x * a.n_tiles + blockIdx.x] = gi;
    a.gpart[(size_t)ch.y * a.n_tiles + blockIdx.x] = gj;
  }
}

template <typename T = double>
inline cudaError_t launch_tcd(const LevelArgs<double>& a, bool post, cudaStream_t st) {
  if (post && a.root_level)
    return launch_pdl(root_tcd_kernel<double>, dim3(a.n_tiles), kTcdThreads, 0, st, a);
  if (post)
    return launch_pdl(post_tcd_kernel<double>, dim3(a.n_tiles, a.n_level, a.n_cat), kTcdThreads,
                      kTcdSmem, st, a);
  return launch_pdl(pre_tcd_kernel<double>, dim3(a.n_tiles, a.n_level, 2 * a.n_cat), kTcdThreads,
                    kTcdSmem, st, a);
}

template <typename T = double>
inline cudaError_t launch_ratio_tcd(const LevelArgs<double>& a, cudaStream_t st) {
  if (a.n_tiles <= 0 || a.n_tips < 2) return cudaSuccess;
  return launch_pdl(ratio_tcd_kernel<double>, dim3(a.n_tiles, a.n_tips - 1), 128, 0, st, a);
}

template <typename T = double>
inline cudaError_t launch_pmat_tcd(const PmatArgs& a, cudaStream_t st) {
  const int units = a.n_branches * a.n_cat;
  pmat_tcd_kernel<double><<<(units + 1) / 2, kTcdThreads, kTcdSmem, st>>>(a);
  return cudaGetLastError();
}

template <typename T = double>
inline cudaError_t prepare_tcd() {
  cudaError_t e = cudaFuncSetAttribute(
      pmat_tcd_kernel<double>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kTcdSmem);
  for (auto k : {post_tcd_kernel<double>, pre_tcd_kernel<double>})
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kTcdSmem);
  return e;
}

}  // namespace phylo
