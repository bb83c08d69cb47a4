// Whole-pass kernels for 4 padded states (nucleotide models): one launch
// walks every level of a pass, or a run of levels, in FP64 at any size and in
// FP32 for problems too small to fill the GPU level by level.
//
// Site patterns never mix before the final sums, so a tile of patterns can
// climb (post-order) or descend (pre-order) the whole tree on its own: only
// the warps on that tile have to agree that a level is done before the next
// begins, which takes a block barrier instead of a kernel boundary.  A block
// owns one tile of 32 / RP patterns; the nodes of a level are dealt to its
// warps, one thread per (pattern, category), the RP lanes of a pattern
// adjacent.
//
// Arithmetic: the U form (kernels_p4.cuh) for every internal node, cherries
// included,
//   post:  p_k = U_i o U_j (rescaled), U_k = P_k p_k             (Eqs. 2, 3)
//   pre:   a_x = q_k o U_y, den = a_x . U_x, q_x = P_x' a_x,
//          num_x = (a_x' gamma_r Q) . U_x  (a tip: a_x' dP_x e_y) (Eqs. 4, 8)
// with q_root = w_r pi, so that the category weights ride along in q.
// A tip with a partial vector v gets U = P v where it is needed.
//
// What bounds it.  FP64: the FP64 pipe, which issues half a lane per clock in
// each quarter of an SM (64 clocks per warp instruction), so everything that
// is not a product or a sum is kept off it: the rescale maximum compares high
// words as integers, the scaling adds to the exponent fields, and the three
// sums over categories and the two ratios of a pattern are spread over its
// lanes, one instruction for all of them.  256 taxa x 3,001 patterns x 4
// categories: post-order 0.42 -> 0.19 ms, pre-order 0.98 -> 0.56 ms against
// per-level launches that formed P p, dP p and P' a (ncu: FP64 pipe 65% and
// 70% of the time, 24 and 80 FP64 instructions a step; the rest is the third
// block that some SMs hold and others do not).  Spreading a tile over a
// cluster of 2, 4 or 8 blocks lost at every size (the cluster barrier: 0.84,
// 1.12, 1.87 ms for both passes against 0.76).
// FP32 (small problems): the latency of a level, see the second half.
#pragma once

namespace phylo {

constexpr int kTreeThreads = 32 * kTreeWarps;

__device__ __forceinline__ void tree_load4(const float* p, float (&v)[4]) {
  const float4 x = *reinterpret_cast<const float4*>(p);
  v[0] = x.x; v[1] = x.y; v[2] = x.z; v[3] = x.w;
}
__device__ __forceinline__ void tree_load4(const double* p, double (&v)[4]) {
  const double2 x = reinterpret_cast<const double2*>(p)[0];
  const double2 y = reinterpret_cast<const double2*>(p)[1];
  v[0] = x.x; v[1] = x.y; v[2] = y.x; v[3] = y.y;
}
__device__ __forceinline__ void tree_store4(float* p, const float (&v)[4]) {
  *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
}
__device__ __forceinline__ void tree_store4(double* p, const double (&v)[4]) {
  reinterpret_cast<double2*>(p)[0] = make_double2(v[0], v[1]);
  reinterpret_cast<double2*>(p)[1] = make_double2(v[2], v[3]);
}

// out[j] = sum_i y[i] X[i][j]: X = M' gives M y, X = M gives M' y.
template <typename T>
__device__ __forceinline__ void tree_comb(const T* X, const T (&y)[4], T (&out)[4]) {
  T row[4];
  tree_load4(X, row);
#pragma unroll
  for (int j = 0; j < 4; ++j) out[j] = row[j] * y[0];
#pragma unroll
  for (int i = 1; i < 4; ++i) {
    tree_load4(X + 4 * i, row);
#pragma unroll
    for (int j = 0; j < 4; ++j) out[j] = fma(row[j], y[i], out[j]);
  }
}

template <typename T>
__device__ __forceinline__ T tree_dot(const T (&x)[4], const T (&y)[4]) {
  T s = x[0] * y[0];
#pragma unroll
  for (int j = 1; j < 4; ++j) s = fma(x[j], y[j], s);
  return s;
}

// |x| as an integer that orders like it: the bits of a float, the high word
// of a double.
__device__ __forceinline__ int tree_abs_bits(float x) { return __float_as_int(x) & 0x7fffffff; }
__device__ __forceinline__ int tree_abs_bits(double x) { return __double2hiint(x) & 0x7fffffff; }

// x > 0 and finite.
__device__ __forceinline__ bool tree_positive(float x) { return x > 0.f && isfinite(x); }
__device__ __forceinline__ bool tree_positive(double x) {
  const int hi = __double2hiint(x);
  return hi >= 0 && hi < 0x7ff00000 && (hi | __double2loint(x)) != 0;
}

// x 2^-e for finite x, exact unless it underflows: an addition to the
// exponent field of a double that stays normal, a product otherwise.
__device__ __forceinline__ float tree_scale(float x, int, float f) { return x * f; }
__device__ __forceinline__ double tree_scale(double x, int e, double f) {
  const int hi = __double2hiint(x), field = (hi >> 20) & 0x7ff;
  if (field > 0 && field - e > 0) return __hiloint2double(hi - (e << 20), __double2loint(x));
  return x * f;
}

// Divides the pattern's vector (RP lanes) by the power of two that brings
// its largest magnitude into [1/2, 1); returns the exponent.  A zero or
// non-finite vector raises ERR_ZERO_PARTIAL and keeps its values.
template <typename T, int RP>
__device__ __forceinline__ int tree_rescale(T (&v)[4], bool active, bool valid, int* err) {
  constexpr bool f64 = sizeof(T) == 8;
  constexpr int shift = f64 ? 20 : 23, bias = f64 ? 1022 : 126;
  int m = 0;
#pragma unroll
  for (int s = 0; s < 4; ++s) m = max(m, tree_abs_bits(v[s]));
  if (!active) m = 0;
#pragma unroll
  for (int o = 1; o < RP; o <<= 1) m = max(m, __shfl_xor_sync(kFull, m, o));
  const int field = m >> shift;
  int e = field - bias;
  T f;
  if (f64) f = (T)__hiloint2double((1023 - e) << 20, 0);
  else f = (T)__int_as_float((127 - e) << 23);
  // the exponents of a subnormal or huge maximum, and zero and non-finite
  // ones, take the general route (2^-e itself is not a normal number there)
  const bool usual = field >= 1 && field <= 2 * bias;
  if (!__all_sync(kFull, usual || !valid)) {
    const T mx = pattern_max<T, 4, RP>(v, active);
    if (!usual && valid) {
      e = 0;
      if (!(mx > T(0)) || !isfinite(mx) || field > 2 * bias + 2) atomicOr(err, ERR_ZERO_PARTIAL);
      else (void)frexp(mx, &e);
      const int h = e / 2;  // 2^-e may lie outside the type's range
      const T f1 = ldexp(T(1), -h), f2 = ldexp(T(1), h - e);
#pragma unroll
      for (int s = 0; s < 4; ++s) v[s] = v[s] * f1 * f2;
      return e;
    }
  }
  if (!valid) return 0;
#pragma unroll
  for (int s = 0; s < 4; ++s) v[s] = tree_scale(v[s], e, f);
  return e;
}

// This thread's place: pattern and category of the block's tile.
template <int RP>
struct TreeLane {
  int c, r, rr, warp, lane;
  bool valid, active;  // a pattern; a pattern and a category
  __device__ TreeLane(int C, int R) {
    lane = threadIdx.x & 31;
    warp = threadIdx.x >> 5;
    c = blockIdx.x * (32 / RP) + lane / RP;
    r = lane % RP;
    rr = r < R ? r : 0;
    valid = c < C;
    active = valid && r < R;
  }
};

// The matrices of branch b: P' of category rr, then (in steps of 16 R) dP'
// and P.
template <typename T>
__device__ __forceinline__ const T* tree_mats(const LevelArgs<T>& a, int b, int rr) {
  return a.P + ((size_t)b * kP4MatKinds * a.n_cat + rr) * 16;
}

// U of child b: column y of P_b for a compact tip in state y (a gap: all
// ones), the stored U of an internal node, P_b v of a tip with a partial
// vector; y = -1 unless the tip is compact.
template <typename T, int RP>
__device__ __forceinline__ void tree_child(const LevelArgs<T>& a, const TreeLane<RP>& t, int b,
                                           bool compact, int& y, T (&u)[4]) {
  const int C = a.n_patterns, R = a.n_cat, S = a.n_states;
  y = -1;
  if (!t.active) {
    if (compact) y = 0;  // (keeps idle lanes on their warp's branch)
#pragma unroll
    for (int s = 0; s < 4; ++s) u[s] = T(0);
  } else if (compact) {
    y = a.tip_states[(size_t)b * a.state_stride + t.c];
    if (y < S) {
      tree_load4(tree_mats(a, b, t.rr) + 4 * y, u);
    } else {
#pragma unroll
      for (int s = 0; s < 4; ++s) u[s] = s < S ? T(1) : T(0);
    }
  } else if (b >= a.n_tips) {
    tree_load4(a.post + (((size_t)(b - a.n_tips) * C + t.c) * R + t.r) * 4, u);
  } else {
    T v[4];
    tree_load4(a.tip_partials + ((size_t)b * C + t.c) * 4, v);
    tree_comb(tree_mats(a, b, t.rr), v, u);
  }
}

// gamma_r Q of every category.
template <typename T>
__device__ __forceinline__ void tree_put_q(T* Qs, const LevelArgs<T>& a) {
  for (int i = threadIdx.x; i < 16 * a.n_cat; i += blockDim.x)
    Qs[i] = (T)a.rates[i / 16] * a.qmat[i % 16];
}

template <typename T, int RP>
__global__ void __launch_bounds__(kTreeThreads)
tree4_post_kernel(LevelArgs<T> a, TreeSched s, int first, int last) {
  const TreeLane<RP> t(a.n_patterns, a.n_cat);
  const int C = a.n_patterns, R = a.n_cat, S = a.n_states;
  pdl_wait_and_release();
  int lo = s.off[first];
  for (int l = first; l < last; ++l) {
    const int hi = s.off[l + 1];
    for (int i = lo + blockIdx.y * kTreeWarps + t.warp; i < hi; i += gridDim.y * kTreeWarps) {
      const int4 d = s.desc[i];
      const int k = d.x;
      T p[4], uj[4];
      int yi, yj, e = 0;
      tree_child<T, RP>(a, t, d.y, d.w & kDescFlagCompact0, yi, p);
      tree_child<T, RP>(a, t, d.z, d.w & kDescFlagCompact1, yj, uj);
      if (t.valid) {
        if (d.y >= a.n_tips) e += a.escale[(size_t)(d.y - a.n_tips) * a.escale_stride + t.c];
        if (d.z >= a.n_tips) e += a.escale[(size_t)(d.z - a.n_tips) * a.escale_stride + t.c];
      }
#pragma unroll
      for (int x = 0; x < 4; ++x) p[x] *= uj[x];
      e += tree_rescale<T, RP>(p, t.active, t.valid, a.err);
      if (k != a.root) {
        T u[4];
        tree_comb(tree_mats(a, k, t.rr), p, u);  // U_k = P_k p_k
        if (t.active) {
          tree_store4(a.post + (((size_t)(k - a.n_tips) * C + t.c) * R + t.r) * 4, u);
          if (t.r == 0) a.escale[(size_t)(k - a.n_tips) * a.escale_stride + t.c] = e;
        }
        continue;
      }
      // Eq. 3: L_c = sum_r w_r pi' p_root, the exponents restored
      double lr = 0.0;
      if (t.active) {
#pragma unroll
        for (int x = 0; x < 4; ++x)
          if (x < S) lr += a.root_pi[x] * (double)p[x];
        lr *= a.cat_w[t.r];
      }
      lr = sum_over_lanes<RP>(lr);
      double term = 0.0;
      if (t.valid && t.r == 0) {
        if (!(lr > 0.0) || !isfinite(lr)) atomicOr(a.err, ERR_ZERO_PARTIAL);
        term = a.pattern_w[t.c] * (log(lr) + (double)e * 0.69314718055994530942);
      }
#pragma unroll
      for (int o = 16; o >= RP; o >>= 1) term += __shfl_down_sync(kFull, term, o);
      if (t.lane == 0) a.lpart[blockIdx.x] = term;
    }
    lo = hi;
    __syncthreads();  // end of the level
  }
}

// The ratios N_i / D and N_j / D of a pattern from its lanes' terms (Eq. 8):
// lane role 0 gets child i's, role 1 child j's (role -1: neither).  Summing
// a different quantity on each lane costs 3 additions instead of 6, and one
// division gives both ratios.
template <typename T, int RP>
__device__ __forceinline__ T tree_ratio(T D, T Ni, T Nj, int r, bool valid, int& role, int* err) {
  static_assert(RP >= 2, "two lanes for two ratios");
  T y, den;
  if constexpr (RP == 2) {
    const T x = r ? Nj : Ni, send = r ? Ni : Nj;
    y = x + __shfl_xor_sync(kFull, send, 1);
    den = D + __shfl_xor_sync(kFull, D, 1);
    role = r;
  } else {
    // after two exchanges lane r % 4 = 0, 1, 2 holds its four lanes' sum of
    // D, N_i, N_j
    const bool odd = r & 1, two = r & 2;
    T x0 = odd ? Ni : D, x1 = odd ? T(0) : Nj;
    x0 += __shfl_xor_sync(kFull, odd ? D : Ni, 1);
    x1 += __shfl_xor_sync(kFull, odd ? Nj : T(0), 1);
    y = (two ? x1 : x0) + __shfl_xor_sync(kFull, two ? x0 : x1, 2);
    if constexpr (RP == 8) y += __shfl_xor_sync(kFull, y, 4);
    den = __shfl_sync(kFull, y, (threadIdx.x & 31) & ~(RP - 1));
    role = r == 1 ? 0 : r == 2 ? 1 : -1;
  }
  if (!valid || role < 0) return T(0);
  if (!tree_positive(den)) {
    atomicOr(err, ERR_BAD_RATIO);
    return T(0);
  }
  return y / den;
}

// Sum of the tile's pattern terms for branch b (FP32: the pair as stored,
// which the final reduction converts).
template <typename T, int RP>
__device__ __forceinline__ void tree_tile_sum(const LevelArgs<T>& a, int tile, int b, T W, T g,
                                              bool on, bool writes) {
  using A = Acc<T>;
  typename A::type x = on ? A::prod(W, g) : A::zero();
#pragma unroll
  for (int o = 16; o >= RP; o >>= 1) x = A::add(x, A::shfl_down(x, o));
  if (!writes) return;
  if constexpr (sizeof(T) == 4)
    reinterpret_cast<float2*>(a.gpart)[(size_t)b * a.n_tiles + tile] = make_float2(x.hi, x.lo);
  else
    a.gpart[(size_t)b * a.n_tiles + tile] = x;
}

template <typename T, int RP>
__global__ void __launch_bounds__(kTreeThreads)
tree4_pre_kernel(LevelArgs<T> a, TreeSched s, int first, int last) {
  __shared__ __align__(16) T Qs[RP * 16];
  const TreeLane<RP> t(a.n_patterns, a.n_cat);
  const int C = a.n_patterns, R = a.n_cat, S = a.n_states;
  tree_put_q<T>(Qs, a);  // host-written, as the weights
  const T* Q = Qs + 16 * t.rr;
  const T wr = t.active ? a.cat_wt[t.r] : T(0);
  const T W = t.valid ? a.pattern_wt[t.c] : T(0);
  __syncthreads();
  pdl_wait_and_release();
  int lo = s.off[first];
  for (int l = first; l < last; ++l) {
    const int hi = s.off[l + 1];
    for (int i = lo + blockIdx.y * kTreeWarps + t.warp; i < hi; i += gridDim.y * kTreeWarps) {
      const int4 d = s.desc[i];
      const int k = d.x, b[2] = {d.y, d.z};
      T q[4], u[2][4];
      int yy[2];
      if (k == a.root) {  // Eq. 4 at the root: q = w_r pi
#pragma unroll
        for (int x = 0; x < 4; ++x) q[x] = x < S ? wr * a.root_pit[x] : T(0);
      } else if (t.active) {
        tree_load4(a.pre + (((size_t)(k - a.n_tips) * C + t.c) * R + t.r) * 4, q);
      } else {
#pragma unroll
        for (int x = 0; x < 4; ++x) q[x] = T(0);
      }
      tree_child<T, RP>(a, t, b[0], d.w & kDescFlagCompact0, yy[0], u[0]);
      tree_child<T, RP>(a, t, b[1], d.w & kDescFlagCompact1, yy[1], u[1]);
      T den = T(0), num[2];
#pragma unroll
      for (int x = 0; x < 2; ++x) {
        T av[4];  // a_x = q_k o U_y
#pragma unroll
        for (int j = 0; j < 4; ++j) av[j] = q[j] * u[1 - x][j];
        if (x == 0) den = tree_dot(av, u[0]);
        if (yy[x] >= 0) {  // compact tip: a_x' dP_x e_y (0 for a gap)
          num[x] = T(0);
          if (yy[x] < S) {
            T dp[4];
            tree_load4(tree_mats(a, b[x], t.rr) + 16 * R + 4 * yy[x], dp);
            num[x] = tree_dot(av, dp);
          }
        } else {  // (a_x' gamma_r Q) U_x
          T aq[4];
          tree_comb(Q, av, aq);
          num[x] = tree_dot(aq, u[x]);
        }
        if (b[x] >= a.n_tips) {  // q_x = P_x' a_x, rescaled (only ratios use it)
          T out[4];
          tree_comb(tree_mats(a, b[x], t.rr) + 32 * R, av, out);
          (void)tree_rescale<T, RP>(out, t.active, t.valid, a.err);
          if (t.active)
            tree_store4(a.pre + (((size_t)(b[x] - a.n_tips) * C + t.c) * R + t.r) * 4, out);
        }
      }
      if constexpr (RP == 1) {
        const bool ok = !t.valid || tree_positive(den);
        if (!ok) atomicOr(a.err, ERR_BAD_RATIO);
        const bool on = t.valid && ok;  // the only category's weight cancels
        tree_tile_sum<T, RP>(a, blockIdx.x, b[0], W, on ? num[0] / den : T(0), on, t.lane == 0);
        tree_tile_sum<T, RP>(a, blockIdx.x, b[1], W, on ? num[1] / den : T(0), on, t.lane == 0);
      } else {
        int role;
        const T g = tree_ratio<T, RP>(den, num[0], num[1], t.r, t.valid, role, a.err);
        tree_tile_sum<T, RP>(a, blockIdx.x, role == 1 ? b[1] : b[0], W, g, t.valid && role >= 0,
                             t.lane < RP && role >= 0);
      }
    }
    lo = hi;
    __syncthreads();  // end of the level
  }
}

// ---------------------------------------------------------------------------
// Problems that fit in shared memory: one block per tile group runs both
// passes of an evaluation with everything a step reads on the SM.
//
// A block takes 2^g tiles (32 / RP patterns each) and copies in the matrices
// of every branch (one contiguous region, bulk copies on one mbarrier), both
// schedules and its tips' states; every node's vector lives in shared memory
// from its step to its reader's: U_x from x's post-order step until its
// parent's pre-order step reads it, which then leaves q_x in its place.  The
// (node, tile) steps of a level are dealt to the block's warps and a block
// barrier ends the level, so a level costs shared-memory latencies, the
// step's arithmetic and the barrier, where a level's launch costs 2 to 4 us.
// The post-order exponents only enter log P as their sum over the nodes, so
// one integer per pattern is kept.
//
// Measured, whole evaluation: 61 taxa x 733 patterns x 4 categories FP32 68
// -> 37 us (20 levels: ~1 us each, which is one warp's arithmetic for a
// step), 8 taxa x 250 patterns FP64 80 -> 40 us.  Per-warp double buffers of
// the step's matrices instead of all of them were slower (55 us: a step is
// shorter than a bulk copy's latency), as were the blocks of the last tile
// summing the tiles themselves (45 us).
//
// The two passes alone (the forward and backward of reverse mode) are the
// same code; the forward pass leaves the vectors in the workspace, where the
// backward pass finds them.
// ---------------------------------------------------------------------------

// Vector of (slot, lane): 16-byte chunks of a warp adjacent.
template <typename T>
__device__ __forceinline__ void walk_load(const T* base, int slot, int lane, T (&v)[4]) {
  if constexpr (sizeof(T) == 4) {
    tree_load4(base + (slot * 32 + lane) * 4, v);
  } else {
    const double2* p = reinterpret_cast<const double2*>(base) + slot * 64 + lane;
    const double2 x = p[0], y = p[32];
    v[0] = x.x; v[1] = x.y; v[2] = y.x; v[3] = y.y;
  }
}
template <typename T>
__device__ __forceinline__ void walk_store(T* base, int slot, int lane, const T (&v)[4]) {
  if constexpr (sizeof(T) == 4) {
    tree_store4(base + (slot * 32 + lane) * 4, v);
  } else {
    double2* p = reinterpret_cast<double2*>(base) + slot * 64 + lane;
    p[0] = make_double2(v[0], v[1]);
    p[32] = make_double2(v[2], v[3]);
  }
}

template <typename T, int RP, bool POST, bool PRE>
__global__ void __launch_bounds__(32 * kWalkMaxWarps)
walk4_kernel(LevelArgs<T> a, TreeSched post, TreeSched pre, int g) {
  extern __shared__ __align__(16) unsigned char smraw[];
  constexpr int CT = 32 / RP;
  const int G = 1 << g, NT = blockDim.x, W = NT >> 5;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int N = a.n_tips, C = a.n_patterns, R = a.n_cat, S = a.n_states;
  const int n_int = N - 1, n_vec = (N - 2) * G;  // the root has no vector
  const int bstride = kP4MatKinds * R * 16;      // elements per branch
  const WalkPlan plan(N, R, RP, g, sizeof(T) == 8);
  T* P = reinterpret_cast<T*>(smraw);
  T* vec = reinterpret_cast<T*>(smraw + plan.vec);
  T* Qs = reinterpret_cast<T*>(smraw + plan.q);
  int4* desc = reinterpret_cast<int4*>(smraw + plan.desc);  // post, then pre
  int* off = reinterpret_cast<int*>(smraw + plan.off);      // post, then pre: N each
  uint8_t* states = smraw + plan.states;                    // [tip][G * CT]
  __shared__ uint64_t bar;
  __shared__ int esum[4 * CT];
  const int pat = lane / RP, r = lane % RP, rr = r < R ? r : 0;
  const int c0 = blockIdx.x * G * CT;  // the block's first pattern
  // what the host wrote: schedules, Q, tip states, weights
  for (int i = threadIdx.x; i < N; i += NT) {
    if (POST && i <= post.n_levels) off[i] = post.off[i];
    if (PRE && i <= pre.n_levels) off[N + i] = pre.off[i];
    if (POST && i < n_int) desc[i] = post.desc[i];
    if (PRE && i < n_int) desc[n_int + i] = pre.desc[i];
  }
  for (int i = threadIdx.x; i < N * G * CT; i += NT) {
    const int tip = i / (G * CT), c = c0 + i % (G * CT);
    states[i] = c < C ? a.tip_states[(size_t)tip * a.state_stride + c] : 0;
  }
  if constexpr (PRE) tree_put_q<T>(Qs, a);
  if (threadIdx.x < G * CT) esum[threadIdx.x] = 0;
  if (threadIdx.x == 0) mbar_init_fenced(&bar, 1);
  const T* Q = Qs + 16 * rr;
  const T wcat = PRE && r < R ? a.cat_wt[r] : T(0);
  pdl_wait_and_release();
  if (threadIdx.x == 0) {
    const uint32_t total = (uint32_t)((2 * N - 2) * bstride * sizeof(T));
    mbar_expect_tx(&bar, total);
    for (uint32_t o = 0; o < total; o += kWalkCopy)
      bulk_g2s(smraw + o, reinterpret_cast<const unsigned char*>(a.P) + o,
               min(kWalkCopy, total - o), &bar);
  }
  if constexpr (!POST) {  // the forward pass's vectors, [tile][slot][lane][4]
    for (int i = warp; i < n_vec; i += W) {
      const int slot = i >> g, tile = blockIdx.x * G + (i & (G - 1));
      if (tile >= a.n_tiles) continue;
      T v[4];
      tree_load4(a.post + (((size_t)tile * (N - 2) + slot) * 32 + lane) * 4, v);
      walk_store(vec, i, lane, v);
    }
  }
  // (the barrier also publishes the initialised mbarrier)
  __syncthreads();
  if (!__syncthreads_and(mbar_wait(&bar, 0))) {  // bounded drain, then give up
    if (threadIdx.x == 0) {
      atomicOr(a.err, ERR_TIMEOUT);
      (void)mbar_wait(&bar, 0);
    }
    return;
  }
#pragma unroll
  for (int pass = POST ? 0 : 1; pass < (PRE ? 2 : 1); ++pass) {
    const bool up = pass == 0;
    const int n_levels = up ? post.n_levels : pre.n_levels;
    int lo = 0;
    for (int l = 0; l < n_levels; ++l) {
      const int hi = off[(up ? 0 : N) + l + 1];
      for (int i = (lo << g) + warp; i < hi << g; i += W) {
        const int4 d = desc[(up ? 0 : n_int) + (i >> g)];
        const int sub = i & (G - 1), tile = blockIdx.x * G + sub;
        const int cl = sub * CT + pat, c = c0 + cl;
        const bool valid = c < C, active = valid && r < R;
        const int k = d.x, b[2] = {d.y, d.z};
        const bool compact[2] = {(d.w & kDescFlagCompact0) != 0, (d.w & kDescFlagCompact1) != 0};
        int y[2];
        T u[2][4];
#pragma unroll
        for (int x = 0; x < 2; ++x) {  // U of the children
          const T* Pt = P + b[x] * bstride + rr * 16;  // P'
          y[x] = compact[x] ? states[b[x] * (G * CT) + cl] : -1;
          if (y[x] >= S) {
#pragma unroll
            for (int j = 0; j < 4; ++j) u[x][j] = j < S ? T(1) : T(0);
          } else if (y[x] >= 0) {
            tree_load4(Pt + 4 * y[x], u[x]);
          } else if (b[x] >= N) {
            walk_load(vec, ((b[x] - N) << g) + sub, lane, u[x]);
          } else {
            T v[4];
            tree_load4(a.tip_partials + ((size_t)b[x] * C + (valid ? c : 0)) * 4, v);
            tree_comb(Pt, v, u[x]);
          }
        }
        if (up) {
          T p[4];
#pragma unroll
          for (int j = 0; j < 4; ++j) p[j] = active ? u[0][j] * u[1][j] : T(0);
          const int e = tree_rescale<T, RP>(p, active, valid, a.err);
          if (r == 0 && e != 0) atomicAdd(&esum[cl], e);
          if (k != a.root) {
            T uk[4];  // U_k = P_k p_k
            tree_comb(P + k * bstride + rr * 16, p, uk);
            walk_store(vec, ((k - N) << g) + sub, lane, uk);
          } else {  // Eq. 3; every other node's exponent is in (a barrier ago)
            double lr = 0.0;
            if (active) {
#pragma unroll
              for (int j = 0; j < 4; ++j)
                if (j < S) lr += a.root_pi[j] * (double)p[j];
              lr *= a.cat_w[r];
            }
            lr = sum_over_lanes<RP>(lr);
            __syncwarp();
            double term = 0.0;
            if (valid && r == 0) {
              if (!(lr > 0.0) || !isfinite(lr)) atomicOr(a.err, ERR_ZERO_PARTIAL);
              term = a.pattern_w[c] *
                     (log(lr) + (double)*(volatile int*)&esum[cl] * 0.69314718055994530942);
            }
#pragma unroll
            for (int o = 16; o >= RP; o >>= 1) term += __shfl_down_sync(kFull, term, o);
            if (lane == 0 && tile < a.n_tiles) a.lpart[tile] = term;
          }
        } else {
          T q[4], den = T(0), num[2];
          if (k == a.root) {  // Eq. 4 at the root: q = w_r pi
#pragma unroll
            for (int j = 0; j < 4; ++j) q[j] = j < S ? wcat * a.root_pit[j] : T(0);
          } else {
            walk_load(vec, ((k - N) << g) + sub, lane, q);
          }
#pragma unroll
          for (int x = 0; x < 2; ++x) {
            T av[4];  // a_x = q_k o U_y
#pragma unroll
            for (int j = 0; j < 4; ++j) av[j] = active ? q[j] * u[1 - x][j] : T(0);
            if (x == 0) den = tree_dot(av, u[0]);
            const T* mx = P + b[x] * bstride + rr * 16;
            if (y[x] >= 0) {  // compact tip: a_x' dP_x e_y (0 for a gap)
              num[x] = T(0);
              if (y[x] < S) {
                T dp[4];
                tree_load4(mx + 16 * R + 4 * y[x], dp);
                num[x] = tree_dot(av, dp);
              }
            } else {  // (a_x' gamma_r Q) U_x
              T aq[4];
              tree_comb(Q, av, aq);
              num[x] = tree_dot(aq, u[x]);
            }
            if (b[x] >= N) {  // q_x = P_x' a_x, rescaled, in U_x's place
              T out[4];
              tree_comb(mx + 32 * R, av, out);
              (void)tree_rescale<T, RP>(out, active, valid, a.err);
              walk_store(vec, ((b[x] - N) << g) + sub, lane, out);
            }
          }
          const T wt = valid ? a.pattern_wt[c] : T(0);
          const bool here = tile < a.n_tiles;
          if constexpr (RP == 1) {
            const bool good = !valid || tree_positive(den);
            if (!good) atomicOr(a.err, ERR_BAD_RATIO);
            const bool on = valid && good;  // the only category's weight cancels
            tree_tile_sum<T, RP>(a, tile, b[0], wt, on ? num[0] / den : T(0), on,
                                 here && lane == 0);
            tree_tile_sum<T, RP>(a, tile, b[1], wt, on ? num[1] / den : T(0), on,
                                 here && lane == 0);
          } else {
            int role;
            const T gr = tree_ratio<T, RP>(den, num[0], num[1], r, valid, role, a.err);
            tree_tile_sum<T, RP>(a, tile, role == 1 ? b[1] : b[0], wt, gr, valid && role >= 0,
                                 here && lane < RP && role >= 0);
          }
        }
      }
      lo = hi;
      __syncthreads();  // end of the level
    }
  }
  if constexpr (!PRE) {  // leave the vectors for the backward pass
    for (int i = warp; i < n_vec; i += W) {
      const int slot = i >> g, tile = blockIdx.x * G + (i & (G - 1));
      if (tile >= a.n_tiles) continue;
      T v[4];
      walk_load(vec, i, lane, v);
      tree_store4(a.post + (((size_t)tile * (N - 2) + slot) * 32 + lane) * 4, v);
    }
  }
}

template <typename T, int RP>
cudaError_t launch_walk4(const LevelArgs<T>& a, const TreePass& p, cudaStream_t st) {
  const int G = 1 << p.group;
  const dim3 grid((unsigned)((a.n_tiles + G - 1) / G)), block(32 * p.warps);
  const size_t smem = WalkPlan(a.n_tips, a.n_cat, RP, p.group, sizeof(T) == 8).total;
  auto k = p.do_post && p.do_pre ? walk4_kernel<T, RP, true, true>
           : p.do_post           ? walk4_kernel<T, RP, true, false>
                                 : walk4_kernel<T, RP, false, true>;
  return launch_pdl(k, grid, block, smem, st, a, p.post, p.pre, p.group);
}

template <typename T, int RP>
cudaError_t prepare_walk4() {
  cudaError_t e = cudaSuccess;
  for (auto k : {walk4_kernel<T, RP, true, true>, walk4_kernel<T, RP, true, false>,
                 walk4_kernel<T, RP, false, true>})
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               (int)kWalkMaxSmem);
  return e;
}

// The launches of a kByTile pass.  A block per tile leaves most of the GPU idle
// where there are few tiles, and a wide level then waits for the FP64 pipes of
// a few SMs.  So with room for two blocks per SM, a level of more than `wide`
// nodes is a launch of its own, its nodes split over them, eight nodes or more
// a block; the levels between two of those stay in one launch.  4 categories,
// one launch a pass -> with the split (one launch per level): 1,024 taxa x 100
// patterns 1103 -> 320 us (726), 4,096 x 1 4117 -> 333 (913), 1,024 x 640 1702
// -> 791 (1472), 100 x 100 184 -> 164 (386).  `wide`: a pre-order step has
// three times the FP64 instructions of a post-order one, and a launch costs
// about what 8 of its nodes take a block; 16 (and 48 for post-order) was slower
// with few tiles (64 x 100: 124 us against 112).
template <typename F>
cudaError_t tree_launches(const TreeSched& s, int n_tiles, int wide, F launch) {
  const int most = 2 * kSms / n_tiles;  // blocks per tile
  int first = 0;
  for (int l = 0; l <= s.n_levels; ++l) {
    const int w = l < s.n_levels ? s.host_off[l + 1] - s.host_off[l] : 0;
    const bool own = most > 1 && w > wide;
    if ((own || l == s.n_levels) && first < l) {
      const cudaError_t e = launch(first, l, 1);
      if (e != cudaSuccess) return e;
    }
    if (own) {
      const cudaError_t e =
          launch(l, l + 1, std::min(most, (w + kTreeWarps - 1) / kTreeWarps));
      if (e != cudaSuccess) return e;
      first = l + 1;
    }
  }
  return cudaSuccess;
}

// A block that starts early is placed while its predecessor's blocks hold
// their SMs, and stays where it is: with tiles on more than a quarter of the
// SMs some SMs then hold two long blocks and others none.  Those launches start
// in turn (128 taxa x 1,000 patterns 252 -> 195 us, 256 x 500 271 -> 248);
// below, the early start saves its microseconds (1,024 x 8: 256 -> 244).
template <typename K, typename... Args>
cudaError_t tree_launch(bool early, K kern, dim3 grid, cudaStream_t st, Args... args) {
  if (early) return launch_pdl(kern, grid, kTreeThreads, 0, st, args...);
  kern<<<grid, kTreeThreads, 0, st>>>(args...);
  return cudaGetLastError();
}

template <typename T, int RP>
cudaError_t launch_tree_rp(const LevelArgs<T>& a, const TreePass& p, cudaStream_t st) {
  if (p.walk) return launch_walk4<T, RP>(a, p, st);
  if constexpr (sizeof(T) == 8) {  // kByTile: FP64 only
    const bool early = 4 * a.n_tiles <= kSms;
    cudaError_t e = cudaSuccess;
    if (p.do_post)
      e = tree_launches(p.post, a.n_tiles, 24, [&](int first, int last, int split) {
        return tree_launch(early, tree4_post_kernel<T, RP>, dim3(a.n_tiles, split), st, a, p.post,
                           first, last);
      });
    if (p.do_pre && e == cudaSuccess)
      e = tree_launches(p.pre, a.n_tiles, 8, [&](int first, int last, int split) {
        return tree_launch(early, tree4_pre_kernel<T, RP>, dim3(a.n_tiles, split), st, a, p.pre,
                           first, last);
      });
    return e;
  }
  return cudaErrorInvalidValue;
}

template <typename T>
cudaError_t launch_tree(const LevelArgs<T>& a, const TreePass& p, int RP, cudaStream_t st) {
  if (a.n_tiles <= 0) return cudaSuccess;
  switch (RP) {
    case 1: return launch_tree_rp<T, 1>(a, p, st);
    case 2: return launch_tree_rp<T, 2>(a, p, st);
    case 4: return launch_tree_rp<T, 4>(a, p, st);
    case 8: return launch_tree_rp<T, 8>(a, p, st);
    default: return cudaErrorInvalidValue;
  }
}

template <typename T>
cudaError_t prepare_tree(int RP) {
  switch (RP) {
    case 1: return prepare_walk4<T, 1>();
    case 2: return prepare_walk4<T, 2>();
    case 4: return prepare_walk4<T, 4>();
    case 8: return prepare_walk4<T, 8>();
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace phylo
