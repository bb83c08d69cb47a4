// FP32 level kernels for 5..20 states (amino-acid models) on larger
// alignments: four patterns per thread.
//
// The products of the U form (kernels.cuh) are 20 x 20 matrices times one
// vector per (pattern, category).  With one vector per thread every 16-byte
// shared-memory read of a matrix row feeds two packed FMAs, and the reads, not
// the FMAs, set the time (a 16-byte read returns to the registers of a warp in
// four clocks of the SM; issue active was 31%).  Here a thread holds the
// vectors of four patterns, so a read feeds eight.
//
// Layout: a warp's tile is 128 / RP patterns, lane = (quad, category r), the
// RP lanes of four patterns adjacent; a node's vectors are [tile][state][lane]
// float4 over the quad's patterns, so every access is 512 contiguous bytes.
// A block is four warps: four tiles of one node, which share its matrices.
//
// Measured (256 taxa x 5,000 patterns x 4 categories): post-order 0.366 ->
// 0.299 ms, pre-order 0.590 -> 0.510 ms.  What bounds it now is latency at 8
// (pre-order) and 10 to 11 warps per SM and the last wave of a level (ncu:
// pre-order 5.3 clocks per warp and issue, 1.1 of them for global and 0.8 for
// shared loads, issue active 33 to 36%; post-order 9 to 10 clocks, 5 for global
// loads, issue active 22 to 37%).  Vectors in registers and the product
// unrolled over all 20 rows were slower (0.70 ms: instruction fetch).
//
// The pre-order step takes the numerator from the other side,
//   num_x = gamma_r (a_x Q) . U_x = gamma_r a_x . (Q U_x),
// so that registers hold one set of results (Q U_x, then P_x' a_x) and shared
// memory the vectors: U_x, over which a_x = q_k o U_y is formed state by state.
// A compact tip's U and dP are lookups.
#pragma once

namespace phylo {

constexpr int kQ20Threads = 128;

// Index (in float4) of state 0 of a tile's lane.
__device__ __forceinline__ size_t q20_index(size_t slot, int tile, int n_tiles, int lane) {
  return (slot * n_tiles + tile) * (kU20 * 32) + lane;
}

__device__ __forceinline__ float q20_p(float4 v, int p) {
  return p == 0 ? v.x : p == 1 ? v.y : p == 2 ? v.z : v.w;
}

// out[p][j] = sum_i f[p] y_i[p] X[i][j] for the four patterns p, i in order;
// y: the lane's vectors in shared memory, state i at y[32 i].
__device__ __forceinline__ void q20_comb(const float* __restrict__ X, const float4* y,
                                         const float (&f)[4], float2 (&out)[4][kU20 / 2]) {
#pragma unroll
  for (int p = 0; p < 4; ++p)
#pragma unroll
    for (int h = 0; h < kU20 / 2; ++h) out[p][h] = make_float2(0.f, 0.f);
#pragma unroll 4
  for (int i = 0; i < kU20; ++i) {
    const float4 v = y[32 * i];
    float4 row[kU20 / 4];
#pragma unroll
    for (int h = 0; h < kU20 / 4; ++h)
      row[h] = reinterpret_cast<const float4*>(X + i * kU20)[h];
#pragma unroll
    for (int p = 0; p < 4; ++p) {
      const float vp = q20_p(v, p) * f[p];
      const float2 yi = make_float2(vp, vp);
#pragma unroll
      for (int h = 0; h < kU20 / 4; ++h) {
        out[p][2 * h] = __ffma2_rn(lo2(row[h]), yi, out[p][2 * h]);
        out[p][2 * h + 1] = __ffma2_rn(hi2(row[h]), yi, out[p][2 * h + 1]);
      }
    }
  }
}

__device__ __forceinline__ float q20_el(const float2 (&v)[kU20 / 2], int s) {
  return s & 1 ? v[s >> 1].y : v[s >> 1].x;
}

// States 4 ch .. 4 ch + 3 of the quad's stored vectors: u[p][s].
__device__ __forceinline__ void q20_stored(const float4* v, int ch, bool active,
                                           float (&u)[4][4]) {
#pragma unroll
  for (int s = 0; s < 4; ++s) {
    const float4 x = active ? v[(4 * ch + s) * 32] : make_float4(0.f, 0.f, 0.f, 0.f);
    u[0][s] = x.x; u[1][s] = x.y; u[2][s] = x.z; u[3][s] = x.w;
  }
}

// The same of a table by the patterns' states y (rows of X; a gap: `gap` up to
// S states).
__device__ __forceinline__ void q20_lookup(const float* X, const int (&y)[4], int S, float gap,
                                           int ch, float (&u)[4][4]) {
#pragma unroll
  for (int p = 0; p < 4; ++p) {
    float4 x;
    if (y[p] < S) {
      x = reinterpret_cast<const float4*>(X + y[p] * kU20)[ch];
    } else {
      const int s = 4 * ch;
      x = make_float4(s < S ? gap : 0.f, s + 1 < S ? gap : 0.f, s + 2 < S ? gap : 0.f,
                      s + 3 < S ? gap : 0.f);
    }
    u[p][0] = x.x; u[p][1] = x.y; u[p][2] = x.z; u[p][3] = x.w;
  }
}

// A warp lane's place, and the exponents and states of a child.
template <int RP>
struct Q20Lane {
  int lane, r, rr, tile, c;  // c: the quad's first pattern
  bool active;               // a tile and a category
  __device__ Q20Lane(const LevelArgs<float>& a) {
    lane = threadIdx.x & 31;
    r = lane % RP;
    rr = r < a.n_cat ? r : 0;
    tile = blockIdx.x * (kQ20Threads / 32) + (threadIdx.x >> 5);
    c = tile * (128 / RP) + 4 * (lane / RP);
    active = tile < a.n_tiles && r < a.n_cat;
  }
};

// The quad's states of tip b (patterns past the last: state 0).
__device__ __forceinline__ void q20_states(const LevelArgs<float>& a, int b, int c,
                                           int (&y)[4]) {
  uint32_t w = 0;  // rows are padded to 16 bytes
  if (c < a.n_patterns)
    w = *reinterpret_cast<const uint32_t*>(a.tip_states + (size_t)b * a.state_stride + c);
#pragma unroll
  for (int p = 0; p < 4; ++p) y[p] = c + p < a.n_patterns ? (int)(w >> (8 * p) & 0xff) : 0;
}

// Rescales the four patterns' vectors (RP lanes each) as `rescale`; e: their
// exponents.
template <int RP>
__device__ __forceinline__ void q20_rescale(float2 (&v)[4][kU20 / 2], const Q20Lane<RP>& t,
                                            const LevelArgs<float>& a, int (&e)[4]) {
#pragma unroll
  for (int p = 0; p < 4; ++p) {
    float m = 0.f;
#pragma unroll
    for (int h = 0; h < kU20 / 2; ++h) m = fmaxf(m, fmaxf(fabsf(v[p][h].x), fabsf(v[p][h].y)));
    if (!t.active) m = 0.f;
#pragma unroll
    for (int o = 1; o < RP; o <<= 1) m = fmaxf(m, __shfl_xor_sync(kFull, m, o));
    e[p] = 0;
    float f = 1.f;
    if (!(m > 0.f) || !isfinite(m)) {
      if (t.tile < a.n_tiles && t.c + p < a.n_patterns) atomicOr(a.err, ERR_ZERO_PARTIAL);
    } else {
      e[p] = p4_rescale(m, f);
    }
    const float2 f2 = make_float2(f, f);
#pragma unroll
    for (int h = 0; h < kU20 / 2; ++h) v[p][h] = __fmul2_rn(v[p][h], f2);
  }
}

__device__ __forceinline__ void q20_store(float4* dst, const float2 (&v)[4][kU20 / 2]) {
#pragma unroll
  for (int h = 0; h < kU20 / 2; ++h) {
    dst[(2 * h) * 32] = make_float4(v[0][h].x, v[1][h].x, v[2][h].x, v[3][h].x);
    dst[(2 * h + 1) * 32] = make_float4(v[0][h].y, v[1][h].y, v[2][h].y, v[3][h].y);
  }
}

// Resident blocks the kernels' registers are bounded for.
#ifndef PHYLO_Q20_POST_BLOCKS
#define PHYLO_Q20_POST_BLOCKS 3
#endif
#ifndef PHYLO_Q20_PRE_BLOCKS
#define PHYLO_Q20_PRE_BLOCKS 2
#endif

template <int RP>
__global__ void __launch_bounds__(kQ20Threads, PHYLO_Q20_POST_BLOCKS)
post_q20_kernel(LevelArgs<float> a) {
  constexpr int MS = MatStride<float, kU20>::v;
  extern __shared__ __align__(16) unsigned char smraw[];
  float* mats = reinterpret_cast<float*>(smraw);  // P' of [child 0 | child 1 | node][RP][MS]
  __shared__ uint64_t bar;
  const int S = a.n_states;
  const Q20Lane<RP> t(a);
  const bool tip = a.tip_level;
  if (threadIdx.x == 0) mbar_init_fenced(&bar, 1);
  __syncthreads();
  const int4 d[1] = {a.level_desc[blockIdx.y]};  // host-written: readable before the wait
  if (a.mats_ready) post_u20_stage<RP, 1>(a, d, 1, tip, mats, &bar);
  const int k = d[0].x;
  const bool compact[2] = {!tip && (d[0].w & kDescCompactX), !tip && (d[0].w & kDescCompactY)};
  int y[2][4] = {};
  if (t.active) {
    if (compact[0]) q20_states(a, d[0].y, t.c, y[0]);
    if (compact[1]) q20_states(a, d[0].z, t.c, y[1]);
  }
  pdl_wait_and_release();
  if (!a.mats_ready) post_u20_stage<RP, 1>(a, d, 1, tip, mats, &bar);
  const bool in_c = t.active && t.c < a.n_patterns;
  int e[4] = {0, 0, 0, 0};
  if (!tip && in_c) {
    for (int x = 0; x < 2; ++x) {
      const int b = x ? d[0].z : d[0].y;
      if (b < a.n_tips) continue;
      const int4 v = *reinterpret_cast<const int4*>(
          a.escale + (size_t)(b - a.n_tips) * a.escale_stride + t.c);
      e[0] += v.x; e[1] += v.y; e[2] += v.z; e[3] += v.w;
    }
  }
  if (!__syncthreads_and(mbar_wait(&bar, 0))) {
    if (threadIdx.x == 0) atomicOr(a.err, ERR_TIMEOUT);
    return;
  }
  if (t.tile >= a.n_tiles) return;  // warp-uniform
  const float4* post = reinterpret_cast<const float4*>(a.post);
  const float* tab[2] = {mats + (size_t)t.rr * MS, mats + (size_t)(RP + t.rr) * MS};
  // p_k by state in shared memory (this lane's own slots), its maximum by pattern
  float4* v = reinterpret_cast<float4*>(mats + 3 * RP * MS) + (threadIdx.x >> 5) * (kU20 * 32) +
              t.lane;
  float m[4] = {0.f, 0.f, 0.f, 0.f}, f[4] = {1.f, 1.f, 1.f, 1.f};
  if (tip) {  // the tip's partial vectors, [c][20]
#pragma unroll 1
    for (int ch = 0; ch < kU20 / 4; ++ch) {
      float u[4][4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const bool on = t.active && t.c + i < a.n_patterns;
        const float4 x = on ? reinterpret_cast<const float4*>(
                                  a.tip_partials)[((size_t)k * a.n_patterns + t.c + i) * (kU20 / 4) + ch]
                            : make_float4(0.f, 0.f, 0.f, 0.f);
        u[i][0] = x.x; u[i][1] = x.y; u[i][2] = x.z; u[i][3] = x.w;
      }
#pragma unroll
      for (int s = 0; s < 4; ++s)
        v[32 * (4 * ch + s)] = make_float4(u[0][s], u[1][s], u[2][s], u[3][s]);
    }
  } else {  // p_k = U_i o U_j
    const float4* src[2] = {
        post + q20_index(compact[0] ? 0 : u20_slot(a, d[0].y), t.tile, a.n_tiles, t.lane),
        post + q20_index(compact[1] ? 0 : u20_slot(a, d[0].z), t.tile, a.n_tiles, t.lane)};
#pragma unroll
    for (int ch = 0; ch < kU20 / 4; ++ch) {
      float u[2][4][4];
#pragma unroll
      for (int x = 0; x < 2; ++x) {
        if (compact[x]) q20_lookup(tab[x], y[x], S, 1.f, ch, u[x]);
        else q20_stored(src[x], ch, t.active, u[x]);
      }
#pragma unroll
      for (int s = 0; s < 4; ++s) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          u[0][i][s] *= u[1][i][s];
          m[i] = fmaxf(m[i], fabsf(u[0][i][s]));
        }
        v[32 * (4 * ch + s)] = make_float4(u[0][0][s], u[0][1][s], u[0][2][s], u[0][3][s]);
      }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      if (!t.active) m[i] = 0.f;
#pragma unroll
      for (int o = 1; o < RP; o <<= 1) m[i] = fmaxf(m[i], __shfl_xor_sync(kFull, m[i], o));
      if (!(m[i] > 0.f) || !isfinite(m[i])) {
        if (t.c + i < a.n_patterns) atomicOr(a.err, ERR_ZERO_PARTIAL);
      } else {
        e[i] += p4_rescale(m[i], f[i]);
      }
    }
  }
  if (k != a.root) {  // U_k = P_k p_k
    float2 u[4][kU20 / 2];
    q20_comb(mats + (size_t)(2 * RP + t.rr) * MS, v, f, u);
    if (t.active)
      q20_store(reinterpret_cast<float4*>(a.post) +
                    q20_index(u20_slot(a, k), t.tile, a.n_tiles, t.lane), u);
    if (!tip && in_c && t.r == 0)
      *reinterpret_cast<int4*>(a.escale + (size_t)(k - a.n_tips) * a.escale_stride + t.c) =
          make_int4(e[0], e[1], e[2], e[3]);
    return;
  }
  // Root: L_c = sum_r w_r pi' p_root (Eq. 3), with the exponents restored.
  double lr[4] = {0.0, 0.0, 0.0, 0.0}, term = 0.0;
#pragma unroll 1
  for (int s = 0; s < S; ++s) {
    const float4 x = v[32 * s];
    const double pi = t.active ? a.root_pi[s] : 0.0;
    lr[0] += pi * (double)(x.x * f[0]);
    lr[1] += pi * (double)(x.y * f[1]);
    lr[2] += pi * (double)(x.z * f[2]);
    lr[3] += pi * (double)(x.w * f[3]);
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const double L = sum_over_lanes<RP>(t.active ? lr[i] * a.cat_w[t.r] : 0.0);
    if (t.r == 0 && t.c + i < a.n_patterns) {
      if (!(L > 0.0) || !isfinite(L)) atomicOr(a.err, ERR_ZERO_PARTIAL);
      term += a.pattern_w[t.c + i] * (log(L) + (double)e[i] * 0.69314718055994530942);
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) term += __shfl_down_sync(kFull, term, o);
  if (t.lane == 0) a.lpart[t.tile] = term;
}

// Sums over a quad's RP lanes: afterwards lane r < 4 holds the sum of its own
// pattern, r, in v[0].
template <int RP>
__device__ __forceinline__ void q20_sum(float (&v)[4], int r) {
  static_assert(RP >= 4, "a lane per pattern of the quad");
  const bool odd = r & 1, two = r & 2;
#pragma unroll
  for (int i = 0; i < 2; ++i)
    v[i] = (odd ? v[2 * i + 1] : v[2 * i]) +
           __shfl_xor_sync(kFull, odd ? v[2 * i] : v[2 * i + 1], 1);
  v[0] = (two ? v[1] : v[0]) + __shfl_xor_sync(kFull, two ? v[0] : v[1], 2);
  if constexpr (RP == 8) v[0] += __shfl_xor_sync(kFull, v[0], 4);
}

template <int RP>
__global__ void __launch_bounds__(kQ20Threads, PHYLO_Q20_PRE_BLOCKS)
pre_q20_kernel(LevelArgs<float> a) {
  constexpr int MS = MatStride<float, kU20>::v, SQ = kU20 * kU20;
  extern __shared__ __align__(16) unsigned char smraw[];
  // per child [P' | dP'] of a compact tip or [P] of an internal child, [RP][MS]
  // each; then Q' (rows = columns of Q)
  float* mats = reinterpret_cast<float*>(smraw);
  float* Qt = mats + 4 * RP * MS;
  // the stored children's U, then a, by state (this lane's own slots)
  float4* v[2];
  for (int x = 0; x < 2; ++x)
    v[x] = reinterpret_cast<float4*>(Qt + SQ) +
           (x * (kQ20Threads / 32) + (threadIdx.x >> 5)) * (kU20 * 32) + (threadIdx.x & 31);
  __shared__ uint64_t bar;
  const int S = a.n_states, R = a.n_cat;
  const Q20Lane<RP> t(a);
  if (threadIdx.x == 0) mbar_init_fenced(&bar, 1);
  const int4 d = a.level_desc[blockIdx.y];  // host-written, as Q and the tip states
  const int k = d.x, b[2] = {d.y, d.z};
  const bool compact[2] = {(d.w & kDescCompactX) != 0, (d.w & kDescCompactY) != 0};
  // The children's U, before the wait: the post-order pass that wrote them
  // ended with its root level, at least one launch back; only q_k comes from
  // the launch before.
  const float4* post = reinterpret_cast<const float4*>(a.post);
#pragma unroll
  for (int x = 0; x < 2; ++x) {
    if (compact[x]) continue;
    const float4* u =
        post + q20_index(u20_slot(a, b[x]), min(t.tile, a.n_tiles - 1), a.n_tiles, t.lane);
#pragma unroll
    for (int s = 0; s < kU20; ++s) {
      if (t.active) cp_async16(v[x] + 32 * s, u + 32 * s);
      else v[x][32 * s] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
  }
  cp_async_commit();
  for (int i = threadIdx.x; i < SQ; i += kQ20Threads) Qt[i] = a.qmat[(i % kU20) * kU20 + i / kU20];
  __syncthreads();
  auto stage = [&] {
    if (threadIdx.x != 0) return;
    uint32_t n = 0;
    for (int x = 0; x < 2; ++x) n += compact[x] ? 2 : b[x] >= a.n_tips;
    mbar_expect_tx(&bar, n * (uint32_t)(R * SQ * sizeof(float)));
    for (int x = 0; x < 2; ++x)
      for (int m = 0; m < 2; ++m) {
        const int kind = compact[x] ? m : 2;
        if (!compact[x] && (m || b[x] < a.n_tips)) continue;
        issue_mats<float, kU20, RP>(a.P, b + x, 1, R, mats + (size_t)(2 * x + m) * RP * MS, &bar,
                                    kP4MatKinds, kind);
      }
  };
  if (a.mats_ready) stage();
  int y[2][4] = {};
  if (t.active) {
    if (compact[0]) q20_states(a, b[0], t.c, y[0]);
    if (compact[1]) q20_states(a, b[1], t.c, y[1]);
  }
  const float w = t.active ? a.cat_wt[t.r] : 0.f;
  const float gam = t.active ? (float)a.rates[t.r] : 0.f;
  pdl_wait_and_release();
  if (!a.mats_ready) stage();
  cp_async_wait<0>();
  if (!__syncthreads_and(mbar_wait(&bar, 0))) {
    if (threadIdx.x == 0) atomicOr(a.err, ERR_TIMEOUT);
    return;
  }
  if (t.tile >= a.n_tiles) return;  // warp-uniform
  // q_k of every state, requested at once and used after the first product
  float4 q[kU20];
  {
    const float4* qk = reinterpret_cast<const float4*>(a.pre) +
                       q20_index(k == a.root ? 0 : k - a.n_tips, t.tile, a.n_tiles, t.lane);
#pragma unroll
    for (int s = 0; s < kU20; ++s) {
      if (k == a.root) {
        const float p = t.active && s < S ? a.root_pit[s] : 0.f;
        q[s] = make_float4(p, p, p, p);
      } else {
        q[s] = t.active ? __ldg(qk + 32 * s) : make_float4(0.f, 0.f, 0.f, 0.f);
      }
    }
  }
  const float one[4] = {1.f, 1.f, 1.f, 1.f};
  // child x's tables: P' (then dP') of a compact tip, P of an internal child
  const float* tab[2] = {mats + (size_t)t.rr * MS, mats + (size_t)(2 * RP + t.rr) * MS};
  float den[4] = {0.f, 0.f, 0.f, 0.f}, num[2][4] = {};
  if (compact[0] && compact[1]) {  // lookups only
#pragma unroll
    for (int ch = 0; ch < kU20 / 4; ++ch) {
      float u[4][4], uj[4][4], g[4][4];
      q20_lookup(tab[0], y[0], S, 1.f, ch, u);
      q20_lookup(tab[1], y[1], S, 1.f, ch, uj);
      q20_lookup(tab[1] + RP * MS, y[1], S, 0.f, ch, g);
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int s = 0; s < 4; ++s) {
          const float aj = q20_p(q[4 * ch + s], i) * u[i][s];
          den[i] = fmaf(aj, uj[i][s], den[i]);
          num[1][i] = fmaf(aj, g[i][s], num[1][i]);
        }
      q20_lookup(tab[0] + RP * MS, y[0], S, 0.f, ch, g);
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int s = 0; s < 4; ++s)
          num[0][i] = fmaf(q20_p(q[4 * ch + s], i) * uj[i][s], g[i][s], num[0][i]);
    }
  }
  // Stages 0, 1: Q U_x of a stored child x and its numerator; the last of them
  // leaves a in the place of U.  Stages 2, 3: q_x = P_x' a_x of an internal
  // child, rescaled (only ratios use it).  One loop, one copy of the product.
#pragma unroll 1
  for (int st = 0; st < 4; ++st) {
    const int x = st & 1, bx = x ? b[1] : b[0];
    if (st < 2 ? (x ? compact[1] : compact[0]) : bx < a.n_tips) continue;
    float4* vx = x ? v[1] : v[0];
    float2 z[4][kU20 / 2];
    q20_comb(st < 2 ? Qt : x ? tab[1] : tab[0], vx, one, z);
    if (st >= 2) {
      int e[4];
      q20_rescale<RP>(z, t, a, e);
      if (t.active)
        q20_store(reinterpret_cast<float4*>(a.pre) +
                      q20_index(bx - a.n_tips, t.tile, a.n_tiles, t.lane), z);
      continue;
    }
    float nx[4] = {0.f, 0.f, 0.f, 0.f}, ny[4] = {0.f, 0.f, 0.f, 0.f};
    const bool cy = x ? compact[0] : compact[1];
    if (cy) {
      const float* Ty = x ? tab[0] : tab[1];
      int ys[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) ys[i] = x ? y[0][i] : y[1][i];
#pragma unroll
      for (int ch = 0; ch < kU20 / 4; ++ch) {
        float u[4][4], g[4][4];
        q20_lookup(Ty, ys, S, 1.f, ch, u);
        q20_lookup(Ty + RP * MS, ys, S, 0.f, ch, g);
#pragma unroll
        for (int s = 0; s < 4; ++s) {
          const float4 w4 = vx[32 * (4 * ch + s)];
          float ax[4];
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const float qi = q20_p(q[4 * ch + s], i), wi = q20_p(w4, i);
            ny[i] = fmaf(qi * wi, g[i][s], ny[i]);  // a_y . (column of dP_y)
            ax[i] = qi * u[i][s];
            den[i] = fmaf(ax[i], wi, den[i]);
            nx[i] = fmaf(ax[i], q20_el(z[i], 4 * ch + s), nx[i]);
          }
          vx[32 * (4 * ch + s)] = make_float4(ax[0], ax[1], ax[2], ax[3]);
        }
      }
    } else {
      float4* vy = x ? v[0] : v[1];
#pragma unroll
      for (int s = 0; s < kU20; ++s) {
        const float4 x4 = vx[32 * s], y4 = vy[32 * s];
        float ax[4], ay[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const float qi = q20_p(q[s], i);
          ax[i] = qi * q20_p(y4, i);
          ay[i] = qi * q20_p(x4, i);
          if (!x) den[i] = fmaf(ax[i], q20_p(x4, i), den[i]);
          nx[i] = fmaf(ax[i], q20_el(z[i], s), nx[i]);
        }
        if (x) {
          vx[32 * s] = make_float4(ax[0], ax[1], ax[2], ax[3]);
          vy[32 * s] = make_float4(ay[0], ay[1], ay[2], ay[3]);
        }
      }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      if (x) num[1][i] = gam * nx[i];
      else num[0][i] = gam * nx[i];
      if (cy) {
        if (x) num[0][i] = ny[i];
        else num[1][i] = ny[i];
      }
    }
  }
  // sums over the categories (Eq. 8), the ratios, and the tile's sums
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    den[i] *= w;
    num[0][i] *= w;
    num[1][i] *= w;
  }
  q20_sum<RP>(den, t.r);
  q20_sum<RP>(num[0], t.r);
  q20_sum<RP>(num[1], t.r);
  using A = Acc<float>;
  F2 g[2] = {A::zero(), A::zero()};
  const int c = t.c + t.r;
  if (t.r < 4 && c < a.n_patterns) {  // (lane r: pattern r of the quad)
    if (!(den[0] > 0.f) || !isfinite(den[0])) {
      atomicOr(a.err, ERR_BAD_RATIO);
    } else {
      const float W = a.pattern_wt[c];
      g[0] = A::prod(W, num[0][0] / den[0]);
      g[1] = A::prod(W, num[1][0] / den[0]);
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    g[0] = A::add(g[0], A::shfl_down(g[0], o));
    g[1] = A::add(g[1], A::shfl_down(g[1], o));
  }
  if (t.lane == 0) {  // the pairs as stored (the reduction converts to FP64)
    float2* gp = reinterpret_cast<float2*>(a.gpart);
    gp[(size_t)b[0] * a.n_tiles + t.tile] = make_float2(g[0].hi, g[0].lo);
    gp[(size_t)b[1] * a.n_tiles + t.tile] = make_float2(g[1].hi, g[1].lo);
  }
}

template <int RP>
constexpr size_t q20_smem(bool post) {
  return ((size_t)(post ? 3 : 4) * RP * MatStride<float, kU20>::v + (post ? 0 : kU20 * kU20) +
          (post ? 1 : 2) * kQ20Threads * kU20 * 4) *
         sizeof(float);
}

template <int RP>
cudaError_t launch_q20(LevelArgs<float> a, bool post, cudaStream_t st) {
  // One node per grid row: 65,536 tips with partial vectors take two launches
  // (each waits for the one before it, so the level after them sees both).
  constexpr int kRows = 65535;
  cudaError_t e = cudaSuccess;
  for (int left = a.n_level; left > 0 && e == cudaSuccess; left -= kRows, a.level_desc += kRows) {
    a.n_level = std::min(left, kRows);
    const dim3 grid((a.n_tiles + kQ20Threads / 32 - 1) / (kQ20Threads / 32), a.n_level);
    e = post ? launch_pdl(post_q20_kernel<RP>, grid, kQ20Threads, q20_smem<RP>(true), st, a)
             : launch_pdl(pre_q20_kernel<RP>, grid, kQ20Threads, q20_smem<RP>(false), st, a);
    a.mats_ready = 0;
  }
  return e;
}

template <int RP>
cudaError_t prepare_q20() {
  cudaError_t e = cudaFuncSetAttribute(post_q20_kernel<RP>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)q20_smem<RP>(true));
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(pre_q20_kernel<RP>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)q20_smem<RP>(false));
}

}  // namespace phylo
