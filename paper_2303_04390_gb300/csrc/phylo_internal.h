// Internal declarations shared by the host API (phylo_api.cu) and the kernel
// translation units (kernels_fp32.cu, kernels_fp64.cu).  Not installed.
#pragma once

#include <cmath>
#include <cstddef>
#include <cstdint>
#include <cstring>
#include <vector>

#include <cuda_runtime.h>

namespace phylo {

// Flags of a level-node descriptor: child 0 / child 1 is a tip with a
// compact state; child 0 / child 1 is a cherry fused into this node (FP32,
// 4 states: kernels_p4.cuh).
constexpr int kDescFlagCompact0 = 1, kDescFlagCompact1 = 2;
constexpr int kDescFlagCherry0 = 4, kDescFlagCherry1 = 8;

// Pre-order units of the FP32 tensor-core paths: {k, child x, sibling y, flags};
// a unit contracts the a of child x.  With tip tables (uses_tip_tables) only
// children that are internal or have partial vectors have one: a compact tip's
// numerator is a table lookup in its sibling's unit, and a node whose children
// are both compact tips has none (its terms are lookups only, which nothing
// waits for, and follow after the last level, for all such nodes in one
// launch).  Without, every child has one.
inline bool uses_units(int SP, bool fp64) { return (SP == 64 || SP == 128) && !fp64; }
constexpr int kUnitCompactY = 1;  // y is a compact tip
constexpr int kUnitSecond = 2;    // x is child 1 of k
constexpr int kUnitDen = 4;       // writes the denominator
constexpr int kUnitCompactX = 8;  // x is a compact tip
constexpr int kUnitNumY = 16;     // writes y's numerator, from y's table
// The tables (a launch after the matrix build) and the lookups of the nodes
// with two tips (a launch after the last level) halve the CTAs of a level,
// which pays once levels fill the GPU.  21..64 states, without -> with, by the
// product below: 64 taxa x 100 patterns x 4 categories (256) 205 -> 224 us,
// 64 x 1,100 x 1 (576) 185 -> 200, 128 x 200 x 4 (1,024) 275 -> 283,
// 64 x 600 x 4 (1,280) 268 -> 276, 40 x 1,500 x 4 (1,920) 280 -> 270,
// 30 x 3,000 x 4 (2,880) 310 -> 288.  65..128 states: with tables from the
// smallest (8 x 50).
inline bool uses_tip_tables(int SP, bool fp64, int n_tips, int n_tiles, int R) {
  return uses_units(SP, fp64) && (SP == 128 || (long long)n_tips * n_tiles * R >= 1536);
}
// The units of node k with children (i, j); returns their number (0 to 2).
inline int pre_units(int k, int i, int j, bool compact_i, bool compact_j, bool tables,
                     int4 (&out)[2]) {
  const int ci = compact_i ? 1 : 0, cj = compact_j ? 1 : 0;
  if (tables && ci && cj) return 0;
  if (tables && cj) {
    out[0] = make_int4(k, i, j, kUnitCompactY | kUnitNumY | kUnitDen);
    return 1;
  }
  if (tables && ci) {
    out[0] = make_int4(k, j, i, kUnitCompactY | kUnitNumY | kUnitSecond | kUnitDen);
    return 1;
  }
  out[0] = make_int4(k, i, j, kUnitDen | ci * kUnitCompactX | cj * kUnitCompactY);
  out[1] = make_int4(k, j, i, kUnitSecond | cj * kUnitCompactX | ci * kUnitCompactY);
  return 2;
}

// Device-side numeric flags (bit mask in the workspace's error word).
enum : int {
  ERR_ZERO_PARTIAL = 1,  // a partial vector was all zero / NaN for a pattern
  ERR_BAD_LENGTH = 2,    // a branch length was negative or not finite
  ERR_BAD_RATIO = 4,     // a gradient denominator was zero or not finite
  ERR_TIMEOUT = 8        // a bounded wait on an asynchronous copy expired
};

__host__ __device__ inline int round_up(int x, int m) { return (x + m - 1) / m * m; }

// Padded state count used by the kernels for a model with S states.
inline int padded_states(int S) {
  if (S <= 4) return 4;
  if (S <= 20) return 20;
  if (S <= 64) return 64;
  if (S <= 128) return 128;
  return 256;
}

// Lanes per pattern in the register kernels (next power of two >= R).
inline int lanes_per_pattern(int R) {
  int rp = 1;
  while (rp < R) rp <<= 1;
  return rp;
}

// Threads per block of the register kernels (one thread per (pattern, r)).
constexpr int kSmallThreads = 128;
// Patterns per block of the kernels for S_pad = 128 and 256 (kernels_big.cuh).
constexpr int kBigPatternsF32 = 16;
constexpr int kBigPatternsF64 = 8;
#ifndef PHYLO_BIG_SPT
#define PHYLO_BIG_SPT 2
#endif
constexpr int kBigStatesPerThread = PHYLO_BIG_SPT;  // FP32: states per thread
constexpr int kMaxStates = 256;

// FP32 4-state path (kernels_p4.cuh): one thread per pattern; patterns come
// in tiles of 32 (one warp), the unit of the partials' layout and of the
// per-tile sums.  Partials are tile-blocked, [slot][tile][r][32][4] floats,
// so a warp's access to one category is 512 contiguous bytes.
constexpr int kP4TilePatterns = 32;
__host__ __device__ inline size_t p4_index(size_t slot, int c, int r, int R, int n_tiles) {
  return ((slot * n_tiles + (size_t)(c >> 5)) * R + r) * 32 + (c & 31);
}
// Whether a path stores its partials tile-blocked (FP32, 4 padded states).
inline bool uses_p4_tiles(int SP, bool fp64) { return SP == 4 && !fp64; }
// Tip-state rows are padded to 16 bytes (row starts aligned for bulk copies).
inline int tip_state_stride(int C) { return round_up(C, 16); }
// The FP32 kernels for 4 and 20 padded states read their matrices in the
// orientations the products use, built that way by the matrix kernel: per
// branch, [P' of every category][dP' of every category][P of every
// category] (SP x SP floats each; P' rows are the columns of P).  The dP
// region is then empty.
inline bool uses_tr_layout(int SP, bool fp64) { return SP == 4 || (SP == 20 && !fp64); }
constexpr int kP4MatKinds = 3;
// How a pass of the level schedule runs.
enum PassMode {
  kByLevel,  // one launch per level
  kByTile,   // a pattern tile walks runs of levels (kernels_tree.cuh)
  kWalk      // one launch, every partial vector in shared memory
};
// These launches, 4 padded states: tiles of one warp of (pattern,
// category) lanes.
constexpr int kTreeWarps = 8;      // warps per block, kByTile
constexpr int kWalkMaxWarps = 16;  // warps per block, kWalk
constexpr int kSms = 152;          // SMs of the GPU: blocks of one wave
constexpr int kWalkMaxGroup = 2;   // at most 4 tiles per block, kWalk
constexpr size_t kWalkMaxSmem = 226 * 1024;
constexpr uint32_t kWalkCopy = 32768;  // bytes per bulk copy of the matrices
// Shared memory of a kWalk block with 2^g tiles: the matrices of every branch
// (at offset 0), the nodes' vectors, Q, both schedules (descriptors, level
// offsets), the tips' states.
struct WalkPlan {
  size_t vec, q, desc, off, states, total;
  __host__ __device__ WalkPlan(int n_tips, int R, int RP, int g, bool fp64) {
    const size_t elem = fp64 ? 8 : 4, N = n_tips;
    vec = (2 * N - 2) * kP4MatKinds * R * 16 * elem;
    q = vec + ((N - 2) << g) * 128 * elem;
    desc = q + RP * 16 * elem;
    off = desc + 2 * (N - 1) * 16;
    states = off + (2 * N * 4 + 15) / 16 * 16;
    total = states + ((N << g) * (32 / RP) + 15) / 16 * 16;
  }
};
// Tiles per block (log2) of a kWalk launch, -1 if the problem does not fit in
// one wave of blocks: the smallest group with a block per SM, else the
// largest that shared memory holds.  A second wave loses: 61 taxa x 5,000
// patterns took 100 us against 78 level by level, x 2,000 (one wave) 45
// against 77.
inline int walk_group(bool fp64, int n_tips, int C, int R, int RP) {
  const long long tiles = ((long long)C * RP + 31) / 32;
  auto smem = [&](int g) { return WalkPlan(n_tips, R, RP, g, fp64).total; };
  auto blocks = [&](int g) { return (tiles + (1 << g) - 1) >> g; };
  int g = 0;
  while (g < kWalkMaxGroup && blocks(g) > kSms) ++g;
  while (g >= 0 && smem(g) > kWalkMaxSmem) --g;
  if (g < 0) return -1;
  const int resident = !fp64 && 2 * (smem(g) + 2048) <= 228 * 1024 ? 2 : 1;
  return blocks(g) <= kSms * resident ? g : -1;
}
// FP32 with 5..20 states: whether enough of a tree's levels fill the GPU with
// four patterns per thread to lay the partials out for it (about a quarter of
// the nodes sit in the widest level).  4 categories, before -> after: 256 taxa x
// 5,000 patterns 0.99 -> 0.84 ms, 500 x 1,000 0.58 -> 0.55, 16 x 10,000 0.182 ->
// 0.176; below the line it loses (500 x 300: 0.37 -> 0.38, 96 x 1,201 0.25 ->
// 0.26).  With 3 categories or more a warp's matrix reads hit that many rows
// and are what it saves; with 1 or 2 it loses (256 x 5,000: 1 category 293 ->
// 306 us, 2 462 -> 490, 3 986 -> 909, 8 2,601 -> 1,984).
inline bool uses_quad(int SP, bool fp64, int n_tips, int n_tiles, int R) {
  return SP == 20 && !fp64 && R > 2 && n_tiles >= 32 &&
         (long long)((n_tiles + 3) / 4) * n_tips >= 8 * kSms;
}
inline PassMode pass_mode(int SP, bool fp64, int n_tips, int C, int R, int RP) {
  if (SP != 4) return kByLevel;
  if (walk_group(fp64, n_tips, C, R, RP) >= 0) return kWalk;
  return fp64 ? kByTile : kByLevel;
}

// FP32 with 21..64 states runs on the tensor cores (kernels_tc64.cuh):
// 128-pattern tiles and one rescale exponent per (node, category, pattern).
inline bool uses_tensor_cores(int SP, bool fp64) { return SP == 64 && !fp64; }
constexpr int kTcTilePatterns = 128;
// Matrix operand tiles of one (branch, category) on that path: P and P' as
// three-term BF16 splits, then P' in FP32 (kernels_tc64.cuh gives the
// layout); Q' as one more three-term 64 x 64 operand per model.
constexpr size_t kTcUnitBytes = 65536;
constexpr size_t kTcQtBytes = 3 * 64 * 128;

// FP64 with 21..64 states runs on the tensor cores as well, in exact integer
// arithmetic on base-256 digits (kernels_tcd.cuh): per (branch, category) an
// internal branch's E = P - I and E' as eight-digit operands, the exponents of
// their rows (E' first), a tip's P' and dP' in FP64.
inline bool uses_tcd(int SP, bool fp64) { return SP == 64 && fp64; }
constexpr uint32_t kTcdDigits = 8 * 64 * 128;           // one 64 x 64 operand
constexpr size_t kTcdUnitBytes = 2 * (size_t)kTcdDigits + 128 * sizeof(int);

// The digits of an operand with rows M(n, k), n, k < S (zero beyond) in blocks
// of 64 x 64 (block of rows n >> 6, columns k >> 6; columns fastest), row n
// scaled by 2^-e_n to magnitudes below 1: digit i of element (n, k) of
// round(M 2^(62 - e_n)) = sum_i a_i 256^(7 - i) as an FP16 integer in slice i
// (8 KB) of its block, K-major 128-byte swizzle; then e_n as ints.  SP: 64 or
// 128 padded states.  out: digit_bytes(SP).
inline size_t digit_bytes(int SP) {
  return (size_t)(SP / 64) * (SP / 64) * kTcdDigits + SP * sizeof(int);
}
// FP16 of the integers -128 .. 127 (index + 128).
struct DigitHalves {
  uint16_t h[256];
  DigitHalves() {
    for (int d = -128; d < 128; ++d) {
      int ex;
      const double f = std::frexp(std::fabs((double)d), &ex);
      h[d + 128] = d ? (uint16_t)((d < 0 ? 0x8000 : 0) + ((ex + 13) << 10) + (int)(f * 2048.0)) : 0;
    }
  }
};
template <typename F>
inline void build_digits(int S, int SP, F M, unsigned char* out) {
  static const DigitHalves halves;
  const int NB = SP / 64;
  std::memset(out, 0, digit_bytes(SP));
  for (int n = 0; n < S; ++n) {
    double mx = 0.0;
    for (int k = 0; k < S; ++k) mx = std::fmax(mx, std::fabs(M(n, k)));
    int e = 0;
    (void)std::frexp(mx, &e);
    std::memcpy(out + (size_t)NB * NB * kTcdDigits + n * sizeof(int), &e, sizeof(int));
    for (int k = 0; k < S; ++k) {
      unsigned char* blk = out + (size_t)((n >> 6) * NB + (k >> 6)) * kTcdDigits;
      const long long v = std::llrint(std::ldexp(M(n, k), 62 - e));
      const uint64_t t = (uint64_t)v + 0x8080808080808080ull;
      for (int i = 0; i < 8; ++i) {
        const size_t off = (size_t)(n & 63) * 128 +
                           ((size_t)(((k & 63) >> 3) ^ (n & 7)) << 4) + (k & 7) * 2;
        std::memcpy(blk + (size_t)i * 64 * 128 + off, &halves.h[t >> (56 - 8 * i) & 0xff], 2);
      }
    }
  }
}

// Eigenvectors for the digit contractions: fixed point keeps what each term
// V(s, m) Vinv(m, t) adds to an entry only while no term needs a row's or a
// column's scale to itself, so the free factor of every eigenvector pair is
// chosen to give column m of V and row m of Vinv the same size relative to
// the rows of V and the columns of Vinv.  Powers of two (exact); pairs within
// a factor of 16, as an orthonormal or a symmetrised basis has, stay as given.
inline void balance_eigen(int S, double* V, double* W) {
  std::vector<double> r(S), c(S);
  for (int pass = 0; pass < 32; ++pass) {
    bool changed = false;
    for (int s = 0; s < S; ++s) {
      r[s] = c[s] = 0.0;
      for (int m = 0; m < S; ++m) {
        r[s] = std::fmax(r[s], std::fabs(V[(size_t)s * S + m]));
        c[s] = std::fmax(c[s], std::fabs(W[(size_t)m * S + s]));
      }
    }
    for (int m = 0; m < S; ++m) {
      double a = 0.0, b = 0.0;
      for (int s = 0; s < S; ++s) {
        if (r[s] > 0.0) a = std::fmax(a, std::fabs(V[(size_t)s * S + m]) / r[s]);
        if (c[s] > 0.0) b = std::fmax(b, std::fabs(W[(size_t)m * S + s]) / c[s]);
      }
      if (!(a > 0.0 && b > 0.0)) continue;
      const int k = (std::ilogb(b) - std::ilogb(a)) / 2;
      if (k >= -2 && k <= 2) continue;
      changed = true;
      for (int s = 0; s < S; ++s) {
        V[(size_t)s * S + m] = std::ldexp(V[(size_t)s * S + m], k);
        W[(size_t)m * S + s] = std::ldexp(W[(size_t)m * S + s], -k);
      }
    }
    if (!changed) break;
  }
}

// Round-to-nearest-even BF16 of a finite float, and back (host side).
inline uint16_t host_bf16(float x) {
  uint32_t u;
  std::memcpy(&u, &x, 4);
  u += 0x7FFFu + ((u >> 16) & 1u);
  return (uint16_t)(u >> 16);
}
inline float host_bf16_value(uint16_t b) {
  const uint32_t u = (uint32_t)b << 16;
  float f;
  std::memcpy(&f, &u, 4);
  return f;
}

// Row t of Q = V diag(lambda) Vinv, every entry summed over m in order.
inline void q_row(int S, const double* V, const double* Vinv, const double* lambda, int t,
                  double (&row)[kMaxStates]) {
  for (int s = 0; s < S; ++s) row[s] = 0.0;
  for (int m = 0; m < S; ++m) {
    const double a = V[t * S + m] * lambda[m];
    for (int s = 0; s < S; ++s) row[s] += a * Vinv[m * S + s];
  }
}

// Bytes of the Q' operand for SP = 64 or 128 padded states: (SP / 64)^2
// blocks of 64 x 64 three-term BF16 values.
inline size_t qt_bytes(int SP) { return (size_t)(SP / 64) * (SP / 64) * kTcQtBytes; }

// Q' as the three-term BF16 operand of the tensor-core pre-order step (the
// Eq. 8 numerator through dP = gamma Q P): row s holds column s of
// Q = V diag(lambda) Vinv (FP64, rounded once to FP32), each FP32 value
// split as x = t0 + t1 + t2 with t_i the round-to-nearest BF16 of the
// remainder, cut into K-blocks of 64 columns, each an operand of SP rows stored
// in the K-major 128-byte-swizzle layout the MMAs read (element (row, k) of
// a term at row * 128 + (((k / 8) ^ (row % 8)) * 16) + (k % 8) * 2, terms
// SP * 128 bytes apart).  Rows and columns past S are zero.  out: qt_bytes(SP).
// With `rows` the operand holds Q itself (row s = row s of Q; the tips' tables
// Q P).
inline void build_qt_tile(int S, int SP, const double* V, const double* Vinv,
                          const double* lambda, unsigned char* out, bool rows = false) {
  std::memset(out, 0, qt_bytes(SP));
  const size_t term = 64 * 128;
  const int NB = SP / 64;
  double q[kMaxStates];
  for (int t = 0; t < S; ++t) {
    q_row(S, V, Vinv, lambda, t, q);
    for (int s = 0; s < S; ++s) {
      float rem = (float)q[s];
      const int on = rows ? t : s, ok = rows ? s : t;  // the entry's row and column
      const int n = on & 63, k = ok & 63;
      const size_t blk = (size_t)(ok >> 6) * NB * kTcQtBytes + (size_t)(on >> 6) * term;
      const size_t off = blk + (size_t)n * 128 + ((size_t)((k >> 3) ^ (n & 7)) << 4) + (k & 7) * 2;
      for (int i = 0; i < 3; ++i) {
        const uint16_t b = host_bf16(rem);
        std::memcpy(out + i * NB * term + off, &b, 2);
        rem = rem - host_bf16_value(b);
      }
    }
  }
}

// FP32 paths whose post-order pass stores U = P p per node instead of p
// (20 padded states, kernels.cuh; 21..64 and 65..128 states, kernels_tc64.cuh
// and kernels_tcb.cuh): tips
// with partial vectors keep their U in extra slots of the post region, and
// the pre-order step forms Eq. 8's numerator through Q.
inline bool uses_u_form(int SP, bool fp64) {
  return (SP == 20 || SP == 64 || SP == 128) && !fp64;
}

// Q = V diag(lambda) Vinv in FP64, rounded once to T, row-major SP x SP
// with zero padding (the pre-order step of the 4- and 20-state U form).
template <typename T>
inline void build_q_matrix(int S, int SP, const double* V, const double* Vinv,
                           const double* lambda, T* out) {
  for (int i = 0; i < SP * SP; ++i) out[i] = T(0);
  double q[kMaxStates];
  for (int t = 0; t < S; ++t) {
    q_row(S, V, Vinv, lambda, t, q);
    for (int s = 0; s < S; ++s) out[t * SP + s] = (T)q[s];
  }
}

// FP32 with 65..128 states runs on the tensor cores too (kernels_tcb.cuh):
// 128-pattern tiles, per-category exponents, and the matrices written by
// the matrix kernel directly as 64 x 64 BF16 operand blocks (kind P, P'
// x 2 x 2 blocks of 24 KB per (branch, category)).
inline bool uses_tc_big(int SP, bool fp64) { return SP == 128 && !fp64; }
constexpr size_t kTcbUnitBytes = 2 * 2 * 2 * (3 * 64 * 128);
// Offset of block (kind, jn, jk) in a (branch, category) unit: kind 0 = P,
// 1 = P' (its rows are the columns of P); block row n, column k
// holds M[64 jn + n][64 jk + k] as three BF16 terms in the K-major
// 128-byte-swizzle layout of tc.cuh.  The two row blocks of a K-block jk are
// one 128-row operand (terms 16 KB apart), which one bulk copy stages and one
// chain of N = 128 MMAs reads.
__host__ __device__ constexpr size_t tcb_block(int kind, int jn, int jk) {
  return ((size_t)kind * 2 + jk) * (3 * 128 * 128) + (size_t)jn * (64 * 128);
}
// Paths with per-category exponents and Eq. 8 terms combined by the ratio
// kernel (both tensor-core paths).
inline bool uses_tc_terms(int SP, bool fp64) {
  return uses_tensor_cores(SP, fp64) || uses_tc_big(SP, fp64) || uses_tcd(SP, fp64);
}

// The eigenvectors as double-float pairs for the tensor-core path's matrix
// kernel: out = [V' hi][V' lo][Vinv hi][Vinv lo] (each 64 x 64 floats, V'
// the transpose of V, zero outside S x S) then [pi hi][pi lo] (64 each).
// Returns whether the decomposition is the symmetric one of a reversible
// model, Vinv[m][t] = pi_t V[t][m] (then P(t) = I + V diag(e) V' diag(pi)
// and P_st pi_s = P_ts pi_t, which the kernel exploits).
// The same tables for the other padded sizes (S_pad = 256: the FP32 matrix
// build of kernels_big.cuh): each SP x SP, then pi, SP each.
inline size_t eigen_split_floats(int SP) { return 4 * (size_t)SP * SP + 2 * (size_t)SP; }
constexpr size_t kEigenSplitFloats = 4 * 64 * 64 + 2 * 64;
inline bool build_eigen_split(int S, int SP, const double* V, const double* Vinv,
                              const double* pi, float* out) {
  const size_t sq = (size_t)SP * SP;
  for (size_t i = 0; i < eigen_split_floats(SP); ++i) out[i] = 0.f;
  double vmax = 0.0;
  for (int i = 0; i < S * S; ++i) vmax = Vinv[i] > vmax ? Vinv[i] : (-Vinv[i] > vmax ? -Vinv[i] : vmax);
  bool reversible = true;
  for (int m = 0; m < S; ++m)
    for (int s = 0; s < S; ++s) {
      const double v = V[s * S + m], w = Vinv[m * S + s];
      const float vh = (float)v, wh = (float)w;
      out[0 * sq + (size_t)m * SP + s] = vh;
      out[1 * sq + (size_t)m * SP + s] = (float)(v - (double)vh);
      out[2 * sq + (size_t)m * SP + s] = wh;
      out[3 * sq + (size_t)m * SP + s] = (float)(w - (double)wh);
      const double dev = w - pi[s] * v;
      if (!(dev <= 1e-10 * vmax && -dev <= 1e-10 * vmax)) reversible = false;
    }
  for (int s = 0; s < S; ++s) {
    const float ph = (float)pi[s];
    out[4 * sq + s] = ph;
    out[4 * sq + SP + s] = (float)(pi[s] - (double)ph);
  }
  return reversible;
}
// FP32 paths build their matrices from the double-float tables, except those
// of 65..128 states (digits of the eigenvectors).
inline bool uses_eigen_split(int SP, bool fp64) { return !fp64 && SP != 128; }

// Exponent planes per node: R on the tensor-core path, else 1 (one
// exponent per (node, pattern) shared by all categories).
inline int escale_planes(int SP, int R, bool fp64) {
  return uses_tc_terms(SP, fp64) ? R : 1;
}

// Patterns of one tile (the unit of the per-tile gradient sums).
inline int patterns_per_tile(int SP, int R, bool fp64, PassMode mode = kByLevel) {
  if (mode != kByLevel) return 32 / lanes_per_pattern(R);
  if (SP == 4 && !fp64) return kP4TilePatterns;
  if (uses_tc_terms(SP, fp64)) return kTcTilePatterns;
  if (SP <= 20) return kSmallThreads / lanes_per_pattern(R);
  return fp64 ? kBigPatternsF64 : kBigPatternsF32;
}

// Partial-vector elements stored per node.  Tile-blocked paths pad the
// patterns to whole tiles: FP32 with 4 padded states ([tile][r][32][4]),
// FP32 with 20 padded states ([tile][chunk][kSmallThreads][4], every lane of
// the RP-wide category slots present); the others store [C][R][SP].
inline size_t partial_elems_per_node(int SP, bool fp64, int C, int R, int n_tiles,
                                     PassMode mode = kByLevel) {
  if (mode == kWalk) return (size_t)n_tiles * 32 * SP;
  if (uses_p4_tiles(SP, fp64) && mode == kByLevel) return (size_t)n_tiles * kP4TilePatterns * R * SP;
  if (SP == 20 && !fp64) return (size_t)n_tiles * kSmallThreads * SP;
  return (size_t)C * R * SP;
}

// Arguments of the post- and pre-order level kernels.  All arrays live in
// the caller's workspace.  Partials are pattern-major: [slot][c][r][SP],
// slot = node - n_tips for internal nodes.
template <typename T>
struct LevelArgs {
  const int2* children;        // [2N-1]; (-1,-1) for tips
  const int* level_nodes;      // internal nodes of this level
  const int4* level_desc;      // per level node: {k, child 0, child 1, flags}; the
                               // pre-order pass of the FP32 tensor-core paths: units
  int n_level;                 // number of nodes (units) in the level
  int root_level;              // 1 if the level is the root alone
  int level_cherry;            // 1 if a node of the level has a fused cherry child
  int n_tips, n_patterns, n_states, n_cat, root;
  const T* P;                  // [2N-2][R][SP][SP], row = parent state
                               // (tensor-core path: [2N-2][R] operand tiles;
                               // FP32 4 states: [2N-2][P' | dP' | P][R][16])
  const T* dP;                 // same layout: dP/dt = gamma_r Q P (null on
                               // the tensor-core and FP32 4-state paths,
                               // whose P region holds dP)
  T* post;                     // [N-1][C][R][SP] post-order partials (FP32,
                               // 20 and 64 padded states: U = P p of every
                               // internal node, then of every tip with partials)
  T* pre;                      // [N-1][C][R][SP] pre-order partials
  int* escale;                 // [N-1][planes][escale_stride] cumulative
                               // post-order exponents (planes: escale_planes)
  int* pre_escale;             // [N-1][R][escale_stride] cumulative pre-order
                               // exponents (tensor-core path only, else null)
  const uint8_t* tip_states;   // [N][state_stride]; value S = gap
  int state_stride;            // C rounded up to 16 (16-byte rows)
  int escale_stride;           // C rounded up to 4 (16-byte rows)
  const T* tip_partials;       // [N][C][SP] or nullptr
  const int* tip_has_partials; // [N] or nullptr
  const double* pattern_w;     // [C]
  const double* root_pi;       // [S]
  const double* cat_w;         // [R]
  const T* pattern_wt;         // [C] the same weights in T
  const T* cat_wt;             // [R] the same weights in T
  const T* root_pit;           // [S] the root distribution in T
  void* rterm;                 // tensor-core path: [N-1][C][R] float4 Eq. 8
                               // terms of each category (else null)
  double* gpart;               // [2N-2][n_tiles] per-tile gradient sums
  double* lpart;               // [n_tiles] per-tile log-likelihood sums
  int n_tiles;
  int* err;                    // numeric flags
  const unsigned char* tc_tiles;  // 65..128 states, FP32: the pre-split matrix
                                  // blocks [2N-2][R][kTcbUnitBytes] (else null)
  const unsigned char* qt;     // 21..128 states: Q' operand (FP64: its digits)
  const T* qmat;               // 4 and 20 padded states, U form: Q row-major [SP][SP]
  const double* rates;         // [R] category rates gamma_r
  int quad;                    // FP32, 20 padded states: the partials' layout for four
                               // patterns per thread (kernels.cuh, uses_quad)
  int tip_tables;              // uses_tip_tables
  int tip_level;               // U-form paths: the level's nodes are tips with
                               // partials (their U = P p, before level 1)
  int mats_ready;              // 1 if P was complete before the previous launch
                               // began (every launch but the first after the
                               // matrix kernel): the level may read P and its
                               // descriptors before griddepcontrol.wait
};

struct ReduceArgs {
  const double* gpart;   // [n_branches][n_tiles]; with gpart_pairs each entry
                         // holds a float pair {hi, lo} (value hi + lo)
  const double* lpart;   // [n_tiles]
  int n_tiles, n_branches;
  int gpart_pairs;       // FP32 with 4 or 20 padded states: tile sums as float
                         // pairs (no FP64 in those level kernels)
  double* out;           // [1 + n_branches]
};

// The level schedule of a pass on the device: descriptors in level order,
// level l in [off[l], off[l + 1]).
struct TreeSched {
  const int4* desc;
  const int* off;
  const int* host_off;  // the same offsets on the host
  int n_levels;
};
struct TreePass {
  TreeSched post, pre;
  bool do_post, do_pre;
  bool walk;
  int warps, group;  // kWalk: warps per block, log2 of its tiles
};

struct PmatArgs {
  const float* vsplit;   // tensor-core path: build_eigen_split's table
  const unsigned char* qn;  // uses_tip_tables: Q as an operand (its rows), for the tables
                            // Q P of compact tips (else null)
  const int* tip_has;    // [N] or nullptr: tips with partial vectors (no table)
  const void* vdigits;   // 21..64 states FP64, 65..128 FP32: the digits of Vinv'
                         // (build_digits)
  int n_tips;
  int reversible;        // tensor-core path: the table's decomposition is symmetric
  const double* V;       // [S][S]
  const double* Vinv;    // [S][S]
  const double* lambda;  // [S]
  const double* rates;   // [R]
  const double* t;       // [n_branches]
  int n_branches, n_states, n_cat;
  void* P;               // [n_branches][R][SP][SP] of T
  void* dP;
  void* tiles;           // 65..128 states, FP32: the matrices written as pre-split
                         // operand blocks instead of P and dP (else null)
  int* err;
};

// Launch with programmatic stream serialisation: the kernel may begin
// launching while its predecessor drains; every kernel launched this way
// starts with pdl_wait_and_release() (tma.cuh) before it touches memory
// that other kernels write.  PHYLO_PDL=0 at build time turns it off.
#ifndef PHYLO_PDL
#define PHYLO_PDL 1
#endif
template <typename... KArgs, typename... Args>
inline cudaError_t launch_pdl(void (*kern)(KArgs...), dim3 grid, dim3 block, size_t smem,
                              cudaStream_t st, Args... args) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = PHYLO_PDL;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, args...);
}

// Launchers (kernels_fp32.cu / kernels_fp64.cu).  SP = padded states.
template <typename T>
cudaError_t launch_pmat(const PmatArgs& a, int SP, cudaStream_t st);
template <typename T>
cudaError_t launch_post_level(const LevelArgs<T>& a, int SP, int RP,
                              cudaStream_t st);
template <typename T>
cudaError_t launch_pre_level(const LevelArgs<T>& a, int SP, int RP,
                             cudaStream_t st);
// The passes of a kByTile or kWalk problem.
template <typename T>
cudaError_t launch_tree_pass(const LevelArgs<T>& a, const TreePass& p, int RP, cudaStream_t st);
// Work after the last pre-order level (the tensor-core path's Eq. 8
// ratios); a no-op elsewhere.
template <typename T>
cudaError_t launch_pre_finish(const LevelArgs<T>& a, int SP, cudaStream_t st);
template <typename T>
cudaError_t prepare_kernels(int SP, int RP);
cudaError_t launch_reduce(const ReduceArgs& a, cudaStream_t st);

// Chain-rule epilogues on the gradient g [2N-2] (kernels_fp64.cu).
cudaError_t launch_grad_rate_time(const double* g, int n_br, const double* rates,
                                  const double* times, double* d_rates, double* d_times,
                                  cudaStream_t st);
cudaError_t launch_grad_heights(const double* g, const int2* children, int n_tips,
                                const double* rates, double* d_heights, cudaStream_t st);
cudaError_t launch_grad_branch_sum(const double* g, const int* branches, const double* weights,
                                   int n, double* out, cudaStream_t st);

}  // namespace phylo
