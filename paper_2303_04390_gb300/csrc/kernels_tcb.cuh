// FP32 kernels for 65..128 states (S_pad = 128: the paper's 122-state
// Markov-modulated codon model) on the tensor cores, K- and N-tiled.
//
// Arithmetic as on the 64-state tensor-core path (kernels_tc64.cuh, the U
// form: the post-order pass stores U_x = P_x p_x of every node), per
// (node k, tile of 128 patterns, category r):
//   post:  p_k = U_i o U_j (rescaled),  U_k = p_k P_k'            (Eq. 2)
//   root:  L_c = sum_r w_r pi' (U_i o U_j)                          (Eq. 3)
//   pre, per child x with sibling y (Eq. 4 with the Eq. 8 terms):
//          a_x = q_k o U_y,  den = a_x . U_x,
//          [q_x | W_x] = a_x [P_x | Q],  num_x = gamma_r W_x . U_x
// With 128 padded states every operand is cut into 64 x 64 blocks: a
// contraction D[128 x 128] = A[128 x 128] B[128 x 128]' is, for each of the
// two 64-column blocks of D, two MMA groups of K = 64 accumulated in TMEM.
// Each group is the BF16 x3 split of tc.cuh (six products per FP32
// product), so results carry FP32 accuracy.  One K-block of the A operand
// (p_k or a_x) at a time is formed in registers and split into its three BF16
// terms in shared memory; the matrix operands (P and P' written pre-split by
// the matrix kernel, tcb_block; Q' from the host) are bulk-copied
// (cp.async.bulk).  A compact tip child's U is its column of P, read from the
// split P' blocks.
//
// TMEM: post 128 columns [U_k]; pre 256 [q_x | W_x].  One buffer of A and one
// of B (97 KB) for two CTAs per SM: the kernels wait on loads, copies and MMAs
// in turn, and the second CTA fills those waits better than a second buffer
// did (one CTA, both K-blocks of A and a two-deep B ring, 193 KB: 122 states,
// 128 taxa x 2,000 patterns x 4 categories, post-order 0.68 -> 0.59 ms,
// pre-order 1.20 -> 0.99 ms).
//
// Rescaling, exponents and the Eq. 8 terms follow the 64-state path
// (per-category exponents; ratio_tc_kernel combines the categories).
// Every wait is bounded; on expiry the kernel raises ERR_TIMEOUT, drains
// (bounded) the copies and MMAs it issued, frees its TMEM and returns.
#pragma once

namespace phylo {

constexpr int kTcbSP = 128;                  // padded states of this path
constexpr int kTcbNB = kTcbSP / 64;          // 64-blocks per dimension
static_assert(kTcbUnitBytes == 2 * kTcbNB * kOp128, "matrix block size");
// Shared memory (+1024 for alignment).
constexpr size_t kTcbSmem = 1024 + 2 * (size_t)kOp128;   // level kernels: A, B
constexpr size_t kTipqBSmem = 1024 + 4 * (size_t)kOp128;  // tables: both K-blocks of A, B ring
constexpr int kTcbLd = kTcbSP + 4;           // output staging row stride (floats)
static_assert((size_t)kTcRows * kTcbLd * 4 <= 2 * (size_t)kOp128, "staging fits in A and B");

__device__ __forceinline__ const unsigned char* tcb_unit(const LevelArgs<float>& a, int b,
                                                         int r) {
  return a.tc_tiles + ((size_t)b * a.n_cat + r) * kTcbUnitBytes;
}

// Stored U rows of node x (pattern 0, category r); row stride R * 128 floats.
__device__ __forceinline__ const float* tcb_u_rows(const LevelArgs<float>& a, int x, int r) {
  return a.post + (u_slot(a, x) * a.n_patterns * a.n_cat + r) * kTcbSP;
}

// Entries 64 kb + 8 j .. 64 kb + 8 j + 7 of column y of P_x for branch b (row
// y of P', read from the split P' blocks: the three BF16 terms summed); a
// gap (y = S) gives ones up to S, y < 0 (past the last pattern) zeros.
__device__ __forceinline__ void tcb_col8(const LevelArgs<float>& a, int b, int r, int y, int kb,
                                         int j, float4& lo, float4& hi) {
  const int S = a.n_states;
  if (y < 0 || y >= S) {
    const float g = y < 0 ? 0.f : 1.f;
    const int s = 64 * kb + 8 * j;
    lo = make_float4(s < S ? g : 0.f, s + 1 < S ? g : 0.f, s + 2 < S ? g : 0.f,
                     s + 3 < S ? g : 0.f);
    hi = make_float4(s + 4 < S ? g : 0.f, s + 5 < S ? g : 0.f, s + 6 < S ? g : 0.f,
                     s + 7 < S ? g : 0.f);
    return;
  }
  const unsigned char* blk = tcb_unit(a, b, r) + tcb_block(1, y >> 6, kb);
  const uint32_t off = tc::b16_chunk(y & 63, j);
  const uint4 t0 = __ldg(reinterpret_cast<const uint4*>(blk + off));
  const uint4 t1 = __ldg(reinterpret_cast<const uint4*>(blk + kTerm128 + off));
  const uint4 t2 = __ldg(reinterpret_cast<const uint4*>(blk + 2 * kTerm128 + off));
  const uint32_t w0[4] = {t0.x, t0.y, t0.z, t0.w}, w1[4] = {t1.x, t1.y, t1.z, t1.w},
                 w2[4] = {t2.x, t2.y, t2.z, t2.w};
  float v[8];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    // element 2 i in the low half of word i, 2 i + 1 in the high half
    v[2 * i] = (__uint_as_float(w0[i] << 16) + __uint_as_float(w1[i] << 16)) +
               __uint_as_float(w2[i] << 16);
    v[2 * i + 1] = (__uint_as_float(w0[i] & 0xffff0000u) + __uint_as_float(w1[i] & 0xffff0000u)) +
                   __uint_as_float(w2[i] & 0xffff0000u);
  }
  lo = make_float4(v[0], v[1], v[2], v[3]);
  hi = make_float4(v[4], v[5], v[6], v[7]);
}

// A child's rows c0 + coop_row(it): each one's stored exponent (0 for a tip)
// and a compact tip's state (-1 otherwise, or past the last pattern).
__device__ __forceinline__ void tcb_child_meta(int (&E)[4], int (&y)[4],
                                               const LevelArgs<float>& a, const TcChild& x,
                                               int r, int c0) {
#pragma unroll
  for (int it = 0; it < 4; ++it) {
    const int c = c0 + coop_row(it);
    const bool on = c < a.n_patterns;
    y[it] = x.compact && on ? (int)a.tip_states[(size_t)x.b * a.state_stride + c] : -1;
    E[it] = x.internal && on
                ? a.escale[((size_t)(x.b - a.n_tips) * a.n_cat + r) * a.escale_stride + c]
                : 0;
  }
}

// K-block kb of a child's U rows in the cooperative layout.
__device__ __forceinline__ void tcb_child_kb(float4 (&v)[8], const int (&y)[4],
                                             const LevelArgs<float>& a, const TcChild& x, int r,
                                             int c0, int kb) {
  if (!x.compact) {
    coop_load(v, tcb_u_rows(a, x.b, r) + 64 * kb, (size_t)a.n_cat * kTcbSP, c0, a.n_patterns);
    return;
  }
#pragma unroll
  for (int it = 0; it < 4; ++it)
    tcb_col8(a, x.b, r, y[it], kb, threadIdx.x & 7, v[2 * it], v[2 * it + 1]);
}

// 32 floats of a child's stored U, from column col, for pattern c.
__device__ __forceinline__ void tcb_child_part(float (&u)[32], const LevelArgs<float>& a,
                                               const TcChild& x, int r, int c, int col) {
  const bool on = c < a.n_patterns;
  const float4* src = reinterpret_cast<const float4*>(
      tcb_u_rows(a, x.b, r) + (size_t)(on ? c : 0) * a.n_cat * kTcbSP + col);
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const float4 f = on ? __ldg(src + i) : make_float4(0.f, 0.f, 0.f, 0.f);
    u[4 * i] = f.x;
    u[4 * i + 1] = f.y;
    u[4 * i + 2] = f.z;
    u[4 * i + 3] = f.w;
  }
}

// D (+)= A B' for one K-block (the MMAs of one round).  N = 128 in one chain:
// two chains of N = 64 took 27 clocks per MMA for half the work.
__device__ __forceinline__ void tcb_mma_round(uint32_t d_tmem, const unsigned char* A,
                                              const unsigned char* B, bool accumulate) {
  uint32_t ta[3], tb[3];
  term_addrs(A, kTerm128, ta);
  term_addrs(B, kTerm128, tb);
  tc::mma_split_bf16x3_acc<128>(d_tmem, ta, tb, accumulate);
}

// Coalesced store of staged 128-float rows (a quarter warp writes one
// 128-byte quarter row per instruction).
__device__ __forceinline__ void tcb_store_rows(float* __restrict__ base, size_t stride, int c0,
                                               int C, const float* st) {
  const int jj = threadIdx.x & 7;
#pragma unroll
  for (int it = 0; it < 4; ++it) {
    const int row = coop_row(it), c = c0 + row;
    if (c < C) {
      float* dst = base + (size_t)c * stride;
#pragma unroll
      for (int q = 0; q < 4; ++q)
        *reinterpret_cast<float4*>(dst + 32 * q + 4 * jj) =
            *reinterpret_cast<const float4*>(st + row * kTcbLd + 32 * q + 4 * jj);
    }
  }
}

// Bookkeeping of the asynchronous phases a CTA has issued and waited on,
// so that a timeout can drain what is still in flight.  Barriers: 0, 1 =
// bulk copies into B buffer 0, 1; 2, 3 = MMA commits of rounds using B
// buffer 0, 1.  Scalars (not arrays), so that they stay in registers.
struct TcbPhases {
  uint32_t i0 = 0, i1 = 0, i2 = 0, i3 = 0;  // issued
  uint32_t w0 = 0, w1 = 0, w2 = 0, w3 = 0;  // waited
  __device__ uint32_t waited(int k) const { return k == 0 ? w0 : k == 1 ? w1 : k == 2 ? w2 : w3; }
  __device__ void wait_done(int k) {
    w0 += k == 0; w1 += k == 1; w2 += k == 2; w3 += k == 3;
  }
  __device__ void issue(int k) {
    i0 += k == 0; i1 += k == 1; i2 += k == 2; i3 += k == 3;
  }
};

__device__ __forceinline__ bool tcb_wait(uint64_t* bars, TcbPhases& ph, int k, int* err) {
  const bool mine = mbar_wait(&bars[k], ph.waited(k) & 1);
  const bool ok = __syncthreads_and(mine);
  if (ok) ph.wait_done(k);
  else if (threadIdx.x == 0) atomicOr(err, ERR_TIMEOUT);
  tc::fence_after();
  return ok;
}

__device__ __forceinline__ void tcb_drain(uint64_t* bars, const TcbPhases& ph) {
  if (threadIdx.x != 0) return;
  const uint32_t iss[4] = {ph.i0, ph.i1, ph.i2, ph.i3};
  const uint32_t wai[4] = {ph.w0, ph.w1, ph.w2, ph.w3};
#pragma unroll
  for (int k = 0; k < 4; ++k)
    for (uint32_t p = wai[k]; p < iss[k]; ++p) (void)mbar_wait(&bars[k], p & 1);
}

// Common prologue: barriers, TMEM, the block's row and half.
#define TCB_PROLOGUE(COLS)                                                   \
  extern __shared__ unsigned char smraw[];                                   \
  unsigned char* base = align1024(smraw);                                    \
  unsigned char* const A0 = base;                                           \
  unsigned char* const B0 = base + 2 * kOp128;                               \
  __shared__ uint64_t bars[4]; /* tma 0, tma 1, mma 0, mma 1 */              \
  __shared__ uint32_t tmem_slot;                                             \
  const int tid = threadIdx.x, warp = tid >> 5;                              \
  const int row = tid & (kTcRows - 1), h = tid / kTcRows;                    \
  if (warp == 0) tc::alloc(&tmem_slot, COLS);                                \
  if (tid == 0)                                                              \
    for (int i = 0; i < 4; ++i) mbar_init_fenced(&bars[i], 1);               \
  __syncthreads();                                                           \
  tc::fence_after();                                                         \
  const uint32_t tmem = tmem_slot;                                           \
  const uint32_t trow = tmem + ((uint32_t)((warp & 3) * 32) << 16);          \
  TcbPhases ph;

#define TCB_EPILOGUE(COLS)                                                   \
  tcb_drain(bars, ph);                                                       \
  tc::fence_before();                                                        \
  __syncthreads();                                                           \
  if (warp == 0) tc::dealloc(tmem, COLS);

// One round of a contraction: the matrix operand at bsrc (one K-block) times
// A buffer ab (that K-block of the A operand) into
// d_tmem.
struct TcbRound {
  const unsigned char* bsrc;
  int ab;
  uint32_t d_tmem;
  bool accumulate;
};

// A buffers at A0 + ab kOp128, B buffers at B0 + b kOp128.
__device__ __forceinline__ unsigned char* tcb_a(unsigned char* A0, int ab) {
  return A0 + (size_t)ab * kOp128;
}
__device__ __forceinline__ unsigned char* tcb_b(unsigned char* B0, int b) {
  return B0 + (size_t)b * kOp128;
}

__device__ __forceinline__ void tcb_issue_b(unsigned char* B0, uint64_t* bars, TcbPhases& ph,
                                            int i, const unsigned char* bsrc) {
  if (threadIdx.x == 0) {
    const int b = i & 1;
    mbar_expect_tx(&bars[b], kOp128);
    ph.issue(b);
    bulk_g2s(tcb_b(B0, b), bsrc, kOp128, &bars[b]);
  }
}

// Runs rounds 0 .. n-1 (round_of(i) generates round i) on A operands already
// staged; the caller has issued the block copies of rounds 0 and 1 (those
// that exist).  While round i's MMAs run, round i + 1's blocks are in flight
// and round i + 2's copy starts once round i's MMAs have freed its buffer.
// False on a timeout (ERR_TIMEOUT raised); on success every MMA is done.
template <class RoundOf>
__device__ __forceinline__ bool tcb_rounds(unsigned char* A0, unsigned char* B0, uint64_t* bars,
                                           TcbPhases& ph, int n, RoundOf round_of, int* err) {
#pragma unroll 1
  for (int i = 0; i < n; ++i) {
    const TcbRound cur = round_of(i);
    if (!tcb_wait(bars, ph, i & 1, err)) return false;  // round i's blocks (and the A operand)
    if (threadIdx.x == 0) {
      tcb_mma_round(cur.d_tmem, tcb_a(A0, cur.ab), tcb_b(B0, i & 1), cur.accumulate);
      tc::commit(&bars[2 + (i & 1)]);
      ph.issue(2 + (i & 1));
    }
    if (i + 2 < n) {  // round i's MMAs free its B buffer for round i + 2
      if (!tcb_wait(bars, ph, 2 + (i & 1), err)) return false;
      tcb_issue_b(B0, bars, ph, i + 2, round_of(i + 2).bsrc);
    }
  }
  for (int i = n >= 2 ? n - 2 : 0; i < n; ++i)
    if (!tcb_wait(bars, ph, 2 + (i & 1), err)) return false;
  return true;
}

// ---------------------------------------------------------------------------
// Tables of the compact tips, as on the 64-state path (tipq_tc_kernel): G = Q P
// of one (tip, category) per CTA, stored by columns in FP32 ([128][128]) in
// place of the tip's P blocks.
// ---------------------------------------------------------------------------
static_assert(kTcbSP * kTcbSP * 4 <= kTcbNB * kOp128, "a table fits in the P blocks");

template <typename T>  // float only
__global__ void __launch_bounds__(kTcThreads) tipq_tcb_kernel(PmatArgs a) {
  static_assert(std::is_same<T, float>::value, "tensor-core path is FP32");
  pdl_wait_and_release();
  const int unit = blockIdx.x;
  if (a.tip_has && a.tip_has[unit / a.n_cat]) return;  // block-uniform
  TCB_PROLOGUE(128)
  unsigned char* U = static_cast<unsigned char*>(a.tiles) + (size_t)unit * kTcbUnitBytes;
  auto round_of = [=, &a](int kb) {
    return TcbRound{a.qn + tcb_block(0, 0, kb), kb, tmem, kb > 0};
  };
  if (tid == 0) {  // A: P' (rows = columns of P), both K-blocks, on round 0's barrier
    mbar_expect_tx(&bars[0], (1 + kTcbNB) * kOp128);
    ph.issue(0);
    for (int kb = 0; kb < kTcbNB; ++kb)
      bulk_g2s(tcb_a(A0, kb), U + tcb_block(1, 0, kb), kOp128, &bars[0]);
    bulk_g2s(tcb_b(B0, 0), round_of(0).bsrc, kOp128, &bars[0]);
  }
  tcb_issue_b(B0, bars, ph, 1, round_of(1).bsrc);
  if (tcb_rounds(A0, B0, bars, ph, kTcbNB, round_of, a.err)) {
    float* st = reinterpret_cast<float*>(base);  // A is free: every MMA is done
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      float w[32];
      tc::ld32(trow + 64 * h + 32 * q, w);
#pragma unroll
      for (int i = 0; i < 32; i += 4)
        *reinterpret_cast<float4*>(st + row * kTcbLd + 64 * h + 32 * q + i) =
            make_float4(w[i], w[i + 1], w[i + 2], w[i + 3]);
    }
    __syncthreads();
    tcb_store_rows(reinterpret_cast<float*>(U + tcb_block(0, 0, 0)), kTcbSP, 0, kTcbSP, st);
  }
  TCB_EPILOGUE(128)
}

// Floats 64 kb + 8 j .. + 7 of row y of a tip's table (zeros for a gap or past
// the last pattern: the derivative of the all-ones vector is 0).
__device__ __forceinline__ void tcb_gtab8(const LevelArgs<float>& a, int b, int r, int y, int kb,
                                          int j, float4& lo, float4& hi) {
  lo = hi = make_float4(0.f, 0.f, 0.f, 0.f);
  if (y < 0 || y >= a.n_states) return;
  const float4* g = reinterpret_cast<const float4*>(
      reinterpret_cast<const float*>(tcb_unit(a, b, r) + tcb_block(0, 0, 0)) + y * kTcbSP +
      64 * kb + 8 * j);
  lo = __ldg(g);
  hi = __ldg(g + 1);
}

// ---------------------------------------------------------------------------
// Post-order level (Eq. 2), every level but the root's; with `tip_level`
// the level's nodes are tips with partial vectors, whose U = P p is formed
// from those vectors before the first level runs.
// ---------------------------------------------------------------------------
template <typename T>  // float only
__global__ void __launch_bounds__(kTcThreads, 2) post_tcb_kernel(LevelArgs<T> a) {
  static_assert(std::is_same<T, float>::value, "tensor-core path is FP32");
  extern __shared__ unsigned char smraw[];
  unsigned char* A = align1024(smraw);  // one K-block of p_k
  unsigned char* B = A + kOp128;        // one K-block of P_k
  __shared__ uint64_t bar_tma, bar_mma;
  __shared__ uint32_t tmem_slot;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int row = tid & (kTcRows - 1), h = tid / kTcRows;
  const int R = a.n_cat, C = a.n_patterns;
  const int4 d = a.level_desc[blockIdx.y];
  const int k = d.x, r = blockIdx.z;
  const int c0 = blockIdx.x * kTcRows;
  const bool tip = a.tip_level;
  // round kb: U_k (+)= p_k[:, kb] P_k[:, kb]'
  auto copy_b = [&](int kb) {
    if (tid != 0) return;
    mbar_expect_tx(&bar_tma, kOp128);
    bulk_g2s(B, tcb_unit(a, k, r) + tcb_block(0, 0, kb), kOp128, &bar_tma);
  };
  if (tid == 0) {
    mbar_init_fenced(&bar_tma, 1);
    mbar_init_fenced(&bar_mma, 1);
  }
  if (a.mats_ready) copy_b(0);
  pdl_wait_and_release();  // before TMEM or any other global access
  if (!a.mats_ready) copy_b(0);
  if (warp == 0) tc::alloc(&tmem_slot, 128);
  float4 v[2][8];
  if (tip) {
#pragma unroll
    for (int kb = 0; kb < kTcbNB; ++kb)
      coop_load(v[kb], a.tip_partials + (size_t)k * C * kTcbSP + 64 * kb, kTcbSP, c0, C);
  } else {
    // p_k = U_i o U_j, each row rescaled into [1/2, 1); a K-block at a time
    const TcChild x0 = tc_child(a.n_tips, d.y, d.w & kDescFlagCompact0);
    const TcChild x1 = tc_child(a.n_tips, d.z, d.w & kDescFlagCompact1);
    int E0[4], E1[4], y0[4], y1[4];
    tcb_child_meta(E0, y0, a, x0, r, c0);
    tcb_child_meta(E1, y1, a, x1, r, c0);
#pragma unroll
    for (int kb = 0; kb < kTcbNB; ++kb) {
      float4 u[8];
      tcb_child_kb(v[kb], y0, a, x0, r, c0, kb);
      tcb_child_kb(u, y1, a, x1, r, c0, kb);
#pragma unroll
      for (int i = 0; i < 8; ++i) v[kb][i] = mul4(v[kb][i], u[i]);
    }
#pragma unroll
    for (int it = 0; it < 4; ++it) {
      float m = 0.f;
#pragma unroll
      for (int kb = 0; kb < kTcbNB; ++kb) m = amax4(v[kb][2 * it + 1], amax4(v[kb][2 * it], m));
      m = row_max8(m);
      const int c = c0 + coop_row(it);
      const int e = rescale_exponent(m, c < C, a.err);
      const float sc = ldexpf(1.f, -e);
#pragma unroll
      for (int kb = 0; kb < kTcbNB; ++kb)
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          float4& w = v[kb][2 * it + q];
          w = make_float4(w.x * sc, w.y * sc, w.z * sc, w.w * sc);
        }
      if (c < C && (lane & 7) == 0)
        a.escale[((size_t)(k - a.n_tips) * R + r) * a.escale_stride + c] = E0[it] + E1[it] + e;
    }
  }
  coop_put(A, v[0]);
  tc::fence_smem_for_async();
  __syncthreads();  // barriers initialised, TMEM allocated, A written
  tc::fence_after();
  const uint32_t tmem = tmem_slot;
  const uint32_t trow = tmem + ((uint32_t)((warp & 3) * 32) << 16);
  uint32_t ptma = 0, pmma = 0;
  int pend_tma = -1, pend_mma = -1;
  bool ok = true;
#pragma unroll
  for (int kb = 0; kb < kTcbNB && ok; ++kb) {
    if (kb) {
      copy_b(kb);
      coop_put(A, v[kb]);
      tc::fence_smem_for_async();
    }
    ok = tc_block_wait(&bar_tma, ptma, pend_tma, a.err);
    if (!ok) break;
    if (tid == 0) {
      tc::fence_after();
      tcb_mma_round(tmem, A, B, kb > 0);
      tc::commit(&bar_mma);
    }
    ok = tc_block_wait(&bar_mma, pmma, pend_mma, a.err);
  }
  if (ok) {  // U_k, stored as computed (exponent: escale of k)
    float* st = reinterpret_cast<float*>(A);  // A and B are free: every MMA is done
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      float w[32];
      tc::ld32(trow + 64 * h + 32 * q, w);
#pragma unroll
      for (int i = 0; i < 32; i += 4)
        *reinterpret_cast<float4*>(st + row * kTcbLd + 64 * h + 32 * q + i) =
            make_float4(w[i], w[i + 1], w[i + 2], w[i + 3]);
    }
    __syncthreads();
    tcb_store_rows(a.post + (u_slot(a, k) * C * R + r) * kTcbSP, (size_t)R * kTcbSP, c0, C, st);
  }
  if (tid == 0) {  // bounded drain of whatever a timeout left in flight
    if (pend_tma >= 0) (void)mbar_wait(&bar_tma, (uint32_t)pend_tma);
    if (pend_mma >= 0) (void)mbar_wait(&bar_mma, (uint32_t)pend_mma);
  }
  tc::fence_before();
  __syncthreads();
  if (warp == 0) tc::dealloc(tmem, 128);
}

// ---------------------------------------------------------------------------
// Eq. 3 at the root: L_c = sum_r w_r 2^(E_i + E_j) pi' (U_i o U_j), the sum
// over r taken relative to the largest exponent; W_c log L_c summed per tile.
// ---------------------------------------------------------------------------
template <typename T>  // float only
__global__ void __launch_bounds__(kTcRows) root_tcb_kernel(LevelArgs<T> a) {
  static_assert(std::is_same<T, float>::value, "tensor-core path is FP32");
  pdl_wait_and_release();
  __shared__ double lred[kTcRows / 32];
  const int R = a.n_cat, C = a.n_patterns, S = a.n_states;
  const int4 d = a.level_desc[0];
  const TcChild xs[2] = {tc_child(a.n_tips, d.y, d.w & kDescFlagCompact0),
                         tc_child(a.n_tips, d.z, d.w & kDescFlagCompact1)};
  const int c = blockIdx.x * kTcRows + threadIdx.x;
  double term = 0.0;
  if (c < C) {
    int y[2] = {-1, -1};
    for (int x = 0; x < 2; ++x)
      if (xs[x].compact) y[x] = a.tip_states[(size_t)xs[x].b * a.state_stride + c];
    float lsum = 0.f;
    int lexp = INT_MIN / 2;
    for (int r = 0; r < R; ++r) {
      int E = 0;
      for (int x = 0; x < 2; ++x)
        if (xs[x].internal)
          E += a.escale[((size_t)(xs[x].b - a.n_tips) * R + r) * a.escale_stride + c];
      float dot = 0.f;
      for (int kb = 0; kb < kTcbNB; ++kb)
        for (int j = 0; j < 8; ++j) {
          float4 u[2][2];
          for (int x = 0; x < 2; ++x) {
            if (xs[x].compact) {
              tcb_col8(a, xs[x].b, r, y[x], kb, j, u[x][0], u[x][1]);
            } else {
              const float4* src = reinterpret_cast<const float4*>(
                  tcb_u_rows(a, xs[x].b, r) + (size_t)c * R * kTcbSP + 64 * kb + 8 * j);
              u[x][0] = __ldg(src);
              u[x][1] = __ldg(src + 1);
            }
          }
          const int s = 64 * kb + 8 * j;
          for (int q = 0; q < 2; ++q) {
            const float4 p4 = mul4(u[0][q], u[1][q]);
            const float pe[4] = {p4.x, p4.y, p4.z, p4.w};
            for (int i = 0; i < 4; ++i)
              if (s + 4 * q + i < S) dot = fmaf(a.root_pit[s + 4 * q + i], pe[i], dot);
          }
        }
      if (dot != 0.f) {
        const float t = a.cat_wt[r] * dot;
        if (E > lexp) {
          lsum = lsum * pow2i(lexp - E) + t;
          lexp = E;
        } else {
          lsum += t * pow2i(E - lexp);
        }
      }
    }
    if (!(lsum > 0.f) || !isfinite(lsum)) atomicOr(a.err, ERR_ZERO_PARTIAL);
    else term = (double)a.pattern_wt[c] * (log((double)lsum) + (double)lexp * 0.69314718055994530942);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) term += __shfl_down_sync(kFull, term, o);
  if ((threadIdx.x & 31) == 0) lred[threadIdx.x >> 5] = term;
  __syncthreads();
  if (threadIdx.x == 0) {
    double l = 0.0;
    for (int w = 0; w < kTcRows / 32; ++w) l += lred[w];
    a.lpart[blockIdx.x] = l;
  }
}

// ---------------------------------------------------------------------------
// Pre-order level (Eq. 4) with the per-category Eq. 8 terms: one CTA per
// (tile, unit (pre_units), category): as on the 64-state path, a compact tip's
// numerator is formed in its sibling's unit from the table G_y.
// ---------------------------------------------------------------------------
template <typename T>  // float only
__global__ void __launch_bounds__(kTcThreads, 2) pre_tcb_kernel(LevelArgs<T> a) {
  static_assert(std::is_same<T, float>::value, "tensor-core path is FP32");
  extern __shared__ unsigned char smraw[];
  unsigned char* A = align1024(smraw);  // one K-block of a_x
  unsigned char* B = A + kOp128;        // one K-block of Q or P_x
  __shared__ uint64_t bar_tma, bar_mma;
  __shared__ uint32_t tmem_slot;
  __shared__ float xn[2][kTcRows], xm[2][kTcRows];  // the halves' num and q maximum
  const int tid = threadIdx.x, warp = tid >> 5, j = tid & 7;
  const int row = tid & (kTcRows - 1), h = tid / kTcRows;
  const int R = a.n_cat, C = a.n_patterns, S = a.n_states;
  const int4 d = a.level_desc[blockIdx.z];
  const int k = d.x, r = (int)blockIdx.y;
  const int x = (d.w & kUnitSecond) ? 1 : 0;  // x's place among k's children
  const TcChild cx = tc_child(a.n_tips, d.y, false);
  const TcChild cy = tc_child(a.n_tips, d.z, d.w & kUnitCompactY);
  const bool root = k == a.root;
  const size_t kslot = (size_t)(k - a.n_tips);
  const int c0 = blockIdx.x * kTcRows, c = c0 + row;
  const int estr = a.escale_stride;
  if (tid == 0) {
    mbar_init_fenced(&bar_tma, 1);
    mbar_init_fenced(&bar_mma, 1);
  }
  auto copy_b = [&](bool p, int kb) {  // Q' (host-written) or P_x'
    if (tid != 0) return;
    mbar_expect_tx(&bar_tma, kOp128);
    bulk_g2s(B, p ? tcb_unit(a, cx.b, r) + tcb_block(1, 0, kb) : a.qt + tcb_block(0, 0, kb),
             kOp128, &bar_tma);
  };
  copy_b(false, 0);
  // The children's U and exponents are read before the wait: the post-order
  // pass that wrote them ended with its root level, at least one launch back;
  // only q_k comes from the launch before.
  int Ey[4], Ex[4], yy[4], yx[4];
  tcb_child_meta(Ey, yy, a, cy, r, c0);
  tcb_child_meta(Ex, yx, a, cx, r, c0);
  float4 q[8], ux[8], uy[8];
  float den[4], ny[4];  // this lane's parts of the rows' sums
  auto load_u = [&](int kb) {
    tcb_child_kb(ux, yx, a, cx, r, c0, kb);
    tcb_child_kb(uy, yy, a, cy, r, c0, kb);
  };
  load_u(0);
  pdl_wait_and_release();  // before TMEM or any other global access
  if (warp == 0) tc::alloc(&tmem_slot, 256);
  // row-layout values of this thread's row for the epilogue
  int eq_row = 0, ey_row = 0;
  if (c < C) {
    if (!root) eq_row = a.pre_escale[(kslot * R + r) * estr + c];
    if (cy.internal) ey_row = a.escale[((size_t)(cy.b - a.n_tips) * R + r) * estr + c];
  }
  auto load_q = [&](int kb) {
    if (root) {  // q_root = pi
      const int s = 64 * kb + 8 * j;
      float p[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) p[i] = s + i < S ? a.root_pit[s + i] : 0.f;
#pragma unroll
      for (int it = 0; it < 4; ++it) {
        q[2 * it] = make_float4(p[0], p[1], p[2], p[3]);
        q[2 * it + 1] = make_float4(p[4], p[5], p[6], p[7]);
      }
    } else {
      coop_load(q, a.pre + (kslot * C * R + r) * kTcbSP + 64 * kb, (size_t)R * kTcbSP, c0, C);
    }
  };
  // a_y = q_k o U_x: den = a_y . U_y and a tip sibling's numerator; then
  // a_x = q_k o U_y, split into A
  auto form = [&](int kb) {
#pragma unroll
    for (int it = 0; it < 4; ++it) {
      const float4 b0 = mul4(q[2 * it], ux[2 * it]), b1 = mul4(q[2 * it + 1], ux[2 * it + 1]);
      den[it] = dot4(b1, uy[2 * it + 1], dot4(b0, uy[2 * it], kb ? den[it] : 0.f));
      if (!kb) ny[it] = 0.f;
      if (cy.compact) {
        float4 lo, hi;
        tcb_gtab8(a, cy.b, r, yy[it], kb, j, lo, hi);
        ny[it] = dot4(b1, hi, dot4(b0, lo, ny[it]));
      }
      q[2 * it] = mul4(q[2 * it], uy[2 * it]);
      q[2 * it + 1] = mul4(q[2 * it + 1], uy[2 * it + 1]);
    }
    coop_put(A, q);
    tc::fence_smem_for_async();
  };
  load_q(0);
  form(0);
  __syncthreads();  // barriers initialised, TMEM allocated
  tc::fence_after();
  const uint32_t tmem = tmem_slot;  // columns [q_x | W_x]
  const uint32_t trow = tmem + ((uint32_t)((warp & 3) * 32) << 16);
  uint32_t ptma = 0, pmma = 0;
  int pend_tma = -1, pend_mma = -1;
  bool ok = tc_block_wait(&bar_tma, ptma, pend_tma, a.err);
  auto mma = [&](bool p, int kb) {
    if (tid != 0) return;
    tc::fence_after();
    tcb_mma_round(p ? tmem : tmem + 128u, A, B, kb > 0);
    tc::commit(&bar_mma);
  };
  // rounds W, q (internal x) of K-block 0, then of K-block 1
  if (ok) {
    mma(false, 0);
    load_q(1);
    load_u(1);
    ok = tc_block_wait(&bar_mma, pmma, pend_mma, a.err);
  }
  if (ok && cx.internal) {
    copy_b(true, 0);
    ok = tc_block_wait(&bar_tma, ptma, pend_tma, a.err);
    if (ok) {
      mma(true, 0);
      ok = tc_block_wait(&bar_mma, pmma, pend_mma, a.err);
    }
  }
  if (ok) {
    copy_b(false, 1);
    form(1);
    ok = tc_block_wait(&bar_tma, ptma, pend_tma, a.err);
  }
  const float wg = (float)(a.cat_w[r] * a.rates[r]);
  float* rt = reinterpret_cast<float*>(a.rterm);
  if (ok) {
    mma(false, 1);
    // the Eq. 8 terms that need no contraction, during the MMAs
    if (d.w & (kUnitDen | kUnitNumY)) {
#pragma unroll
      for (int it = 0; it < 4; ++it) {
        const float dn = row_sum8(den[it]), nn = row_sum8(ny[it]);
        const int cc = c0 + coop_row(it);
        if (cc < C && j == 0) {
          float* t4 = rt + ((kslot * C + cc) * R + r) * 4;
          if (cy.compact) t4[1 - x] = wg * nn;
          if (d.w & kUnitDen) {
            const int eq = root ? 0 : a.pre_escale[(kslot * R + r) * estr + cc];
            t4[2] = a.cat_wt[r] * dn;
            t4[3] = __int_as_float(eq + Ex[it] + Ey[it]);
          }
        }
      }
    }
    ok = tc_block_wait(&bar_mma, pmma, pend_mma, a.err);
  }
  if (ok && cx.internal) {
    copy_b(true, 1);
    ok = tc_block_wait(&bar_tma, ptma, pend_tma, a.err);
    if (ok) {
      mma(true, 1);
      ok = tc_block_wait(&bar_mma, pmma, pend_mma, a.err);
    }
  }
  if (ok) {
    // epilogue (row layout, thread (row, h) owns states 64 h .. 64 h + 63)
    float num = 0.f, m = 0.f;
#pragma unroll
    for (int qq = 0; qq < 2; ++qq) {
      float u[32], w[32];
      tcb_child_part(u, a, cx, r, c, 64 * h + 32 * qq);
      tc::ld32(trow + 128 + 64 * h + 32 * qq, w);
#pragma unroll
      for (int i = 0; i < 32; ++i) num = fmaf(w[i], u[i], num);
    }
    if (cx.internal) {
#pragma unroll
      for (int qq = 0; qq < 2; ++qq) {
        float w[32];
        tc::ld32(trow + 64 * h + 32 * qq, w);
#pragma unroll
        for (int i = 0; i < 32; ++i) m = fmaxf(m, fabsf(w[i]));
      }
    }
    xn[h][row] = num;
    xm[h][row] = m;
    __syncthreads();
    if (c < C && h == 0) rt[((kslot * C + c) * R + r) * 4 + x] = wg * (num + xn[1][row]);
    if (cx.internal) {  // q_x = a_x P_x, the row rescaled into [1/2, 1)
      m = fmaxf(m, xm[1 - h][row]);
      const int e = rescale_exponent(m, c < C, a.err);
      const float f = ldexpf(1.f, -e);
      float* st = reinterpret_cast<float*>(A);  // A and B are free: every MMA is done
#pragma unroll
      for (int qq = 0; qq < 2; ++qq) {
        float w[32];
        tc::ld32(trow + 64 * h + 32 * qq, w);
#pragma unroll
        for (int i = 0; i < 32; i += 4)
          *reinterpret_cast<float4*>(st + row * kTcbLd + 64 * h + 32 * qq + i) =
              make_float4(w[i] * f, w[i + 1] * f, w[i + 2] * f, w[i + 3] * f);
      }
      if (c < C && h == 0)  // q_x = P_x' (q_k o U_y): exponents of q_k and of U_y
        a.pre_escale[((size_t)(cx.b - a.n_tips) * R + r) * estr + c] = e + eq_row + ey_row;
      __syncthreads();
      tcb_store_rows(a.pre + ((size_t)(cx.b - a.n_tips) * C * R + r) * kTcbSP,
                     (size_t)R * kTcbSP, c0, C, st);
    }
  }
  if (tid == 0) {  // bounded drain of whatever a timeout left in flight
    if (pend_tma >= 0) (void)mbar_wait(&bar_tma, (uint32_t)pend_tma);
    if (pend_mma >= 0) (void)mbar_wait(&bar_mma, (uint32_t)pend_mma);
  }
  tc::fence_before();
  __syncthreads();
  if (warp == 0) tc::dealloc(tmem, 256);
}

#undef TCB_PROLOGUE
#undef TCB_EPILOGUE

struct Cols128 {
  template <bool G>
  __device__ __forceinline__ static void col(const LevelArgs<float>& a, int b, int r, int y,
                                             int kb, int j, float4& lo, float4& hi) {
    if (G) tcb_gtab8(a, b, r, y, kb, j, lo, hi);
    else tcb_col8(a, b, r, y, kb, j, lo, hi);
  }
};

// The nodes whose children are both compact tips (level_desc), then the ratios.
template <int SP>
inline cudaError_t launch_ratio_tc64(const LevelArgs<float>& a, cudaStream_t st) {
  if (a.n_tiles <= 0 || a.n_tips < 2) return cudaSuccess;
  if (a.n_level > 0) {
    const cudaError_t e =
        launch_pdl(SP == 64 ? cherry_kernel<64, Cols64> : cherry_kernel<128, Cols128>,
                   dim3(a.n_tiles, a.n_cat, a.n_level), kTcThreads, 0, st, a);
    if (e != cudaSuccess) return e;
  }
  dim3 grid(a.n_tiles, a.n_tips - 1);
  return launch_pdl(ratio_tc_kernel<float>, grid, kTcRows, 0, st, a);
}

inline cudaError_t launch_tcb(const LevelArgs<float>& a, bool post, cudaStream_t st) {
  if (post) {
    if (a.root_level) return launch_pdl(root_tcb_kernel<float>, dim3(a.n_tiles), kTcRows, 0, st, a);
    dim3 grid(a.n_tiles, a.n_level, a.n_cat);
    return launch_pdl(post_tcb_kernel<float>, grid, kTcThreads, kTcbSmem, st, a);
  }
  dim3 grid(a.n_tiles, a.n_cat, a.n_level);
  return launch_pdl(pre_tcb_kernel<float>, grid, kTcThreads, kTcbSmem, st, a);
}

// ---------------------------------------------------------------------------
// Matrices (Eq. 1): P = I + V diag(expm1) Vinv by the exact digit contractions
// of kernels_tcd.cuh (eight base-256 digits: the sum over eigenvalues, which
// cancels in the small entries of short branches, carries no rounding), each
// entry rounded to FP32 and written as the split operands.  One CTA per
// (branch, category) and half of the columns (64 nh ..), K in two blocks of
// 64 eigenvalues: the rows V diag(e) sliced here, Vinv's digits from the host.
// It replaces the double-float contraction on the CUDA cores (12 FP32
// operations a term; the step includes the tip tables): 254 branches x 4
// categories, 122 states, 0.76 -> 0.40 ms.  A CTA is a serial chain (slice,
// contract, slice, contract, split) that one CTA per SM (512 TMEM columns)
// does not hide.
// ---------------------------------------------------------------------------
// Sum of the accumulators of one element in FP32, infinite past its range (K = 128: |D_d| <= 2^22 only
// for d <= 2, < 2^24 after; the sum's magnitude below 2^8).
__device__ __forceinline__ float tcb_digit_value(const float (&f)[8], int scale, bool one) {
  constexpr unsigned K = 0x4b400000u;
  unsigned n[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) n[d] = (unsigned)__float_as_int(f[d] + 12582912.f);
  const int t01 = (int)(n[0] * 256u + n[1] - K * 257u);
  const int t23 = (int)(n[2] * 256u + (unsigned)__float2int_rn(f[3]) - K * 256u);
  const long long top = (long long)t01 * 65536 + t23;
  long long low = (long long)__float2int_rn(f[4]) * 256 + __float2int_rn(f[5]);
  low = low * 256 + __float2int_rn(f[6]);
  low = low * 256 + __float2int_rn(f[7]);
  long long V = (top << 19) + (low >> 13);  // in units of 2^(scale - 55)
  if (one) {  // 1 + the sum (a small one shifted to units of 2^-61)
    V >>= min(max(-6 - scale, 0), 63);
    scale = max(scale, -6);
    V += scale <= 55 ? 1ll << (55 - scale) : 0;
  }
  const unsigned long long m = V < 0 ? 0ull - (unsigned long long)V : (unsigned long long)V;
  const int lz = __clzll((long long)m);
  const unsigned long long X = m << lz;
  const int E = 127 + 63 + 7 - 62 - lz + scale;
  if (m == 0 || E <= 0) return 0.f;
  if (E > 254) return V < 0 ? -INFINITY : INFINITY;
  const unsigned bits = ((unsigned)(E - 1) << 23) + (unsigned)(X >> 40) +
                        ((unsigned)(X >> 39) & 1u);
  return __uint_as_float(bits | (V < 0 ? 0x80000000u : 0u));
}

template <typename T>  // float only
__global__ void __launch_bounds__(kTcdThreads) pmat_tcb_kernel(PmatArgs a) {
  static_assert(std::is_same<T, float>::value, "tensor-core path is FP32");
  extern __shared__ unsigned char smraw[];
  unsigned char* A = align1024(smraw);
  unsigned char* B = A + kTcdA;
  float* stage = reinterpret_cast<float*>(A);  // [128][kStageLd]
  __shared__ TcdBars bars;
  __shared__ TcdFactor ex[kTcbSP];
  __shared__ int erow[kTcRows], ecol[64];
  const int tid = threadIdx.x, warp = tid >> 5, j = tid & 7;
  const int S = a.n_states, R = a.n_cat;
  const int unit = blockIdx.x >> 1, nh = blockIdx.x & 1;
  const int b = unit / R, r = unit % R;
  const unsigned char* vd = static_cast<const unsigned char*>(a.vdigits);
  auto copy_b = [&](int kb) {
    if (tid == 0) tcd_copy_b(B, vd + (size_t)(2 * nh + kb) * kTcdB, &bars.tma);
  };
  if (tid == 0) {
    mbar_init_fenced(&bars.tma, 1);
    mbar_init_fenced(&bars.mma, 1);
  }
  copy_b(0);
  if (tid < 64) ecol[tid] = reinterpret_cast<const int*>(vd + 4 * (size_t)kTcdB)[64 * nh + tid];
  if (tid < kTcbSP) {
    double e = 0.0;
    if (tid < S) {
      double t = a.t[b];
      if (!(t >= 0.0) || !isfinite(t)) {
        if (tid == 0 && r == 0 && nh == 0) atomicOr(a.err, ERR_BAD_LENGTH);
        t = 0.0;
      }
      e = expm1(a.lambda[tid] * a.rates[r] * t);
    }
    ex[tcd_factor_at(tid)] = tcd_factor(e);
  }
  if (warp == 0) tc::alloc(&bars.tmem, 512);
  __syncthreads();
  tc::fence_after();
  const uint32_t tmem = bars.tmem;
  uint32_t ptma = 0, pmma = 0;
  int pend_tma = -1, pend_mma = -1;
  // V diag(e) of both K-blocks; a row's digits share one scale
  TcdFactor x[2][2][8];  // [kb][iteration]
  int er[2];
#pragma unroll
  for (int it = 0; it < 2; ++it) {
    const int s = tcd_row(it);
    int e[2];
#pragma unroll
    for (int kb = 0; kb < 2; ++kb) {
      double v[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const int m = 64 * kb + 8 * j + i;
        v[i] = s < S && m < S ? a.V[s * S + m] : 0.0;
      }
      e[kb] = tcd_products(v, ex + 64 * kb, j, x[kb][it]);
    }
    er[it] = max(e[0], e[1]);
    if (j == 0) erow[s] = er[it];
  }
  bool ok = true;
#pragma unroll
  for (int kb = 0; kb < 2; ++kb) {
    if (!ok) break;
    if (kb) copy_b(1);
#pragma unroll
    for (int it = 0; it < 2; ++it) tcd_put(A, 128 * 128, tcd_row(it), j, x[kb][it], er[it]);
    tc::fence_smem_for_async();
    ok = tc_block_wait(&bars.tma, ptma, pend_tma, a.err);
    if (!ok) break;
    if (tid == 0) {
      tc::fence_after();
      tcd_mma(tmem, smem_addr(A), smem_addr(B), kb > 0);
      tc::commit(&bars.mma);
    }
    ok = tc_block_wait(&bars.mma, pmma, pend_mma, a.err);
  }
  if (ok) {
    const int s = tcd_acc_row();
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      float f[4][8];
      const int t0 = tcd_acc_col() + 4 * q;
      tcd_ld(tcd_acc_addr(tmem) + 4 * q, f);
      float v[4];
#pragma unroll
      for (int i = 0; i < 4; ++i)
        v[i] = tcb_digit_value(f[i], erow[s] + ecol[t0 + i], s == 64 * nh + t0 + i && s < S);
      *reinterpret_cast<float4*>(stage + s * kStageLd + t0) = make_float4(v[0], v[1], v[2], v[3]);
    }
    __syncthreads();
    // P: K-block nh of the operand, every row; P': row block nh of both K-blocks
    unsigned char* U = static_cast<unsigned char*>(a.tiles) + (size_t)unit * kTcbUnitBytes;
    for (int i = tid; i < 128 * 16; i += kTcdThreads) {
      const int row = i >> 4, c4 = 4 * (i & 15);
      put_split3_4(U + tcb_block(0, 0, nh), kTerm128, row, c4,
                   *reinterpret_cast<const float4*>(stage + row * kStageLd + c4));
    }
    for (int i = tid; i < 64 * 32; i += kTcdThreads) {
      // row t of P', states s4 ..: four lanes fill 32 bytes
      const int s4 = 4 * (i & 3) + 16 * (i >> 8), t = i >> 2 & 63;
      put_split3_4(U + tcb_block(1, nh, s4 >> 6), kTerm128, t, s4 & 63,
                   make_float4(stage[s4 * kStageLd + t], stage[(s4 + 1) * kStageLd + t],
                               stage[(s4 + 2) * kStageLd + t], stage[(s4 + 3) * kStageLd + t]));
    }
  }
  if (tid == 0) {  // bounded drain of whatever a timeout left in flight
    if (pend_tma >= 0) (void)mbar_wait(&bars.tma, (uint32_t)pend_tma);
    if (pend_mma >= 0) (void)mbar_wait(&bars.mma, (uint32_t)pend_mma);
  }
  tc::fence_before();
  __syncthreads();
  if (warp == 0) tc::dealloc(tmem, 512);
}

inline cudaError_t launch_pmat_tcb(const PmatArgs& a, cudaStream_t st) {
  pmat_tcb_kernel<float><<<2 * a.n_branches * a.n_cat, kTcdThreads, kTcdSmem, st>>>(a);
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  return launch_pdl(tipq_tcb_kernel<float>, dim3(a.n_tips * a.n_cat), kTcThreads, kTipqBSmem, st, a);
}

inline cudaError_t prepare_tcb() {
  cudaError_t e = cudaFuncSetAttribute(post_tcb_kernel<float>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)kTcbSmem);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(pre_tcb_kernel<float>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)kTcbSmem);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(tipq_tcb_kernel<float>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)kTipqBSmem);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(pmat_tcb_kernel<float>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)kTcdSmem);
  return e;
}

}  // namespace phylo
