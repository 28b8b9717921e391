// window_split.cuh -- the split form of a minibatch step's window phase: the
// window kernel's arithmetic, bit for bit, in three kernels over strips of 16
// lines instead of one kernel of thread-block clusters.  Included by
// core.cuh inside namespace magpie_impl, after window_kernel.cuh.
//
//   split_exit     columns: exit wave Q . z_k, forward column FFTs
//   split_project  rows:    forward row FFTs, modulus projection, inverse row FFTs
//   split_grad     columns: inverse column FFTs, g^0, the MAGPS V-cycle
//
// A block takes 16 lines of one window, MS / 16 blocks per window, and the
// window travels between the kernels through its own slot of the increment
// buffer, which stays in L2 (64 windows of 256 x 256 are 32 MiB): the
// gradient kernel reads its 16 columns whole before it overwrites them with
// the increments.  A column strip is 128 bytes wide, so every global access
// of the column kernels is a whole 128-byte segment per half-warp and a line's
// exchange needs one pass through shared memory; the row kernel's lines stay
// inside a warp and need no block barrier at all.
//
// What bounds it: the chain of loads, line transforms and stores of a block,
// with 13 to 32 warps per SM in flight; the cluster kernel's clusters left
// 15 x 8 of the 152 SMs with one block each at m = 256, and waited twice per
// window for exchanges through distributed shared memory.  Sweeps (GB300, us,
// cluster kernel / split form): n = 1024, m = 256, 2500 windows, 4 levels,
// minibatch 64: 5240 / 2210; n = 512, m = 128, 900 windows, 3 levels,
// minibatch 64: 321 / 289.  Of the 56 us of an m = 256 step the kernels alone
// take 12.6, 16.5, 19.4 and the update 9 us.  Tried and left out: handing
// windows from kernel to kernel one by one with counters (2.86 ms against
// 2.54: the waiting blocks hold the slots of working ones), loading z and Q
// for g^0 before the gradient kernel's wait (no change), taking a large
// minibatch through the three kernels in L2-sized parts (no change at 64 MB,
// slower below).
#pragma once

template <int MS>
struct Split {
  static constexpr int E = Cfg<MS>::E, G = Cfg<MS>::G;
  static constexpr int NL = 16;           // lines per block
  static constexpr int T = NL * G;        // threads: G lanes of E points per line
  static constexpr int TILES = MS / NL;   // blocks (and partial-sum slots) per window
  static constexpr int M = MS * MS;
  // levels whose bins fit a thread's strip of E rows and the block's columns
  static constexpr int LMAX = E == 16 ? 5 : 4;
  // resident blocks per SM the three kernels' registers are bounded for.  The
  // line transforms want their 16 to 32 loads in flight (about 113 registers);
  // the 256-thread blocks of m = 256 gain more from a fourth resident block
  // in the first two kernels (64 registers): a 40-step sweep of 2500 windows
  // took 2.44 ms with (1, 1, 1), 2.22 with (4, 4, 1), 2.25 with (4, 4, 3),
  // 2.29 with (5, 4, 1).  At m = 128 any bound above 4 costs (0.296 ms per
  // 15-step sweep unbounded, 0.304 with (1, 5, 1), 0.309 with (1, 1, 5)).
  static constexpr int MB[3] = {MS == 256 ? 4 : 1, MS == 256 ? 4 : 1, 1};
};

// Sum of `v` over the block into part[...][0 or 1] (per-warp FP32 shuffle
// trees, the warps added in FP64 in warp order by thread 0).
template <int T>
__device__ __forceinline__ void split_sum(float v, double* out) {
  __shared__ float red[T / 32];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x == 0) {
    double s = 0.0;
#pragma unroll
    for (int i = 0; i < T / 32; ++i) s += (double)red[i];
    *out = s;
  }
}

// early: the window indices are final before the stream's previous kernel
// ends (a sweep's permutation), so the index and the corner are read before
// the wait for that kernel.
template <int MS>
__device__ __forceinline__ void split_exit_body(const StepArgs& A, int win, int tile, bool early) {
  using S = Split<MS>;
  constexpr int E = S::E, G = S::G, NL = S::NL;
  __shared__ float2 X[NL * MS];
  const int tid = threadIdx.x, l = tid % NL, g = tid / NL, c = tile * NL + l;
  if (!early) grid_dep_wait();
  const int k = A.idx[win];
  if ((unsigned)k >= (unsigned)A.n_pos) {
    if (early) grid_dep_wait();
    grid_dep_launch();
    if (tid == 0 && tile == 0) {
      atomicOr(A.err, 1);
      A.corner[win] = make_int2(-(1 << 30), -(1 << 30));
    }
    return;
  }
  const int pr = A.pos[2 * k], pc = A.pos[2 * k + 1];
  const float2* zp = A.z + (size_t)(pr + g) * A.n_cols + pc + c;
  const float2* qp = A.Q + g * MS + c;
  const size_t zs = (size_t)G * A.n_cols;
  float2 x[E];
  if (early) grid_dep_wait();
  grid_dep_launch();
  if (tid == 0 && tile == 0) A.corner[win] = make_int2(pr, pc);
#pragma unroll
  for (int e = 0; e < E; ++e) x[e] = cmul(__ldg(qp + e * (G * MS)), __ldcg(zp + e * zs));
  dft_reg<E, false>(x);
#pragma unroll
  for (int k1 = 1; k1 < E; ++k1) x[k1] = twmul<false>(x[k1], __ldg(&A.tw[(g * k1) & (MS - 1)]));
#pragma unroll
  for (int k1 = 0; k1 < E; ++k1) X[(k1 * G + g) * NL + l] = x[k1];
  __syncthreads();
  float2* out = A.contrib + (size_t)win * S::M + c;
#pragma unroll
  for (int j = 0; j < E / G; ++j) {
    const int k1 = g + G * j;
    float2 v[G];
#pragma unroll
    for (int gp = 0; gp < G; ++gp) v[gp] = X[(k1 * G + gp) * NL + l];
    dft_reg<G, false>(v);
#pragma unroll
    for (int k2 = 0; k2 < G; ++k2) out[(k1 + E * k2) * MS] = v[k2];
  }
}

template <int MS>
__device__ __forceinline__ void split_project_body(const StepArgs& A, int win, int tile) {
  using S = Split<MS>;
  constexpr int E = S::E, G = S::G, NL = S::NL;
  __shared__ float2 X[NL * MS];
  const int tid = threadIdx.x, rl = tid / G, g = tid % G, kr = tile * NL + rl;
  const int k = A.idx[win];
  const bool ok = (unsigned)k < (unsigned)A.n_pos;  // a skipped window waits as well: see split_exit_kernel
  const float* ampr = A.amp + (size_t)(ok ? k : 0) * S::M + kr * MS + g;
  float av[E];  // fetched while the exit kernel finishes
#pragma unroll
  for (int j = 0; j < E / G; ++j)
#pragma unroll
    for (int k2 = 0; k2 < G; ++k2) av[j * G + k2] = __ldg(ampr + G * j + E * k2);
  grid_dep_wait();
  if (!ok) return;
  grid_dep_launch();
  float2* row = A.contrib + (size_t)win * S::M + kr * MS + g;
  float2 x[E];
#pragma unroll
  for (int e = 0; e < E; ++e) x[e] = __ldcg(row + G * e);
  // rows of a half-warp (G = 8: two of them) kept in different banks
  float2* line = X + rl * MS;
  const int sw = G < 16 ? (rl & 1) << 3 : 0;
  auto slot = [&](int s) -> float2& { return line[s ^ sw]; };
  line_fwd<MS, false>(x, g, true, slot, A.tw);
  constexpr float inv_m = 1.0f / float(S::M);
  float res = 0.f;
#pragma unroll
  for (int i = 0; i < E; ++i) {
    const float a = A.amp_raw ? sqrtf(fmaxf(av[i], 0.f)) : av[i];
    const float2 P = x[i];
    const float p2 = cabs2(P);
    float mag;
    float2 Pp;
    if (p2 > 0.f) {
      const float rs = rsqrtf(p2);
      mag = __fmul_rn(p2, rs);
      const float sc = a * rs * inv_m;
      Pp = f2(__fmul_rn(P.x, sc), __fmul_rn(P.y, sc));
    } else {
      mag = 0.f;
      Pp = f2(__fmul_rn(a, inv_m), 0.f);  // theta(0) = 0
    }
    const float dlt = mag - a;
    res = __fmaf_rn(dlt, dlt, res);
    x[i] = Pp;
  }
  line_inv<MS>(x, g, true, slot, A.tw);
#pragma unroll
  for (int e = 0; e < E; ++e) row[G * e] = x[e];
  split_sum<S::T>(res, A.part + (size_t)(win * S::TILES + tile) * 2);
}

// The V-cycle of the window kernel for L levels on a strip: lane l of a
// half-warp owns column c, the thread the strip's E rows from R0 on.  Level-j
// values are held by all 2^j lanes of their bin, so a restriction is one or
// two shuffles and the whole cycle stays in registers.
// Y(r, l): g^0 at row r of the block's column l.  PREC: the precision form's
// roundings (its coarse kernel's: every bin summed row by row, and the other
// product of the up-pass fused), so that its results do not depend on whether
// the levels fit a strip.
template <int MS, int L, bool PREC, class Src, class Sink>
__device__ __forceinline__ void split_vcycle(const Src& Y, const float* pyr, int l, int c, int R0, const Sink& put) {
  constexpr int E = Split<MS>::E;
  float2 g[E];  // level j's E >> j values at offset E - (E >> (j - 1))
  constexpr auto off = [](int j) { return E - (E >> (j - 1)); };
  // ((x00 + x01) + x10) + x11 of a bin, this lane holding one column (p, q) of it
  const auto rows = [&](float2 p, float2 q, int x) {
    const float2 r0 = cadd(p, shfl_xor2(p, x)), o = shfl_xor2(q, x);
    const bool left = (l & x) == 0;
    return cadd(cadd(r0, left ? q : o), left ? o : q);
  };
#pragma unroll
  for (int a = 0; a < E / 2; ++a) {
    float2 v;
    if (PREC) {
      v = rows(Y(R0 + 2 * a, l), Y(R0 + 2 * a + 1, l), 1);
    } else {
      v = cadd(Y(R0 + 2 * a, l), Y(R0 + 2 * a + 1, l));
      v = cadd(v, shfl_xor2(v, 1));
    }
    g[a] = cscale_rn(v, 0.25f * __ldg(&pyr[lvl_off(MS, 1) + (R0 / 2 + a) * (MS / 2) + (c >> 1)]));
  }
#pragma unroll
  for (int j = 2; j < L; ++j) {
#pragma unroll
    for (int a = 0; a < (E >> j); ++a) {
      const float2 p = g[off(j - 1) + 2 * a], q = g[off(j - 1) + 2 * a + 1];
      float2 v;
      if (PREC) {
        v = rows(p, q, 1 << (j - 1));
      } else if (j == 2) {
        v = cadd(p, q);
        v = cadd(v, shfl_xor2(v, 2));
      } else {  // the window kernel sums these bins row by row
        v = cadd(cadd(p, shfl_xor2(p, 1 << (j - 1))), cadd(q, shfl_xor2(q, 1 << (j - 1))));
      }
      g[off(j) + a] =
          cscale_rn(v, 0.25f * __ldg(&pyr[lvl_off(MS, j) + ((R0 >> j) + a) * (MS >> j) + (c >> j)]));
    }
  }
#pragma unroll
  for (int j = L - 1; j >= 1; --j) {
    const int n = MS >> j;
    const float* iw = pyr + lvl_off(MS, j) + n * n + (R0 >> j) * n + (c >> j);
    const float* rr = iw + n * n;
#pragma unroll
    for (int a = 0; a < (E >> j); ++a) {
      if (j == L - 1)
        g[off(j) + a] = cscale_rn(g[off(j) + a], __ldg(iw + a * n));
      else if (PREC)  // prolong with u^l / w^l e^{l+1} as the fused product
        g[off(j) + a] = prolong(g[off(j + 1) + (a >> 1)], __ldg(rr + a * n), __ldg(iw + a * n), g[off(j) + a]);
      else
        g[off(j) + a] = prolong(g[off(j) + a], __ldg(iw + a * n), __ldg(rr + a * n), g[off(j + 1) + (a >> 1)]);
    }
  }
#pragma unroll
  for (int a = 0; a < E; ++a) {
    const float u = __ldg(&pyr[(R0 + a) * MS + c]);
    const float2 g0 = Y(R0 + a, l), e = g[a >> 1];
    put(R0 + a, c, f2(__fmaf_rn(u, e.x, g0.x), __fmaf_rn(u, e.y, g0.y)));
  }
}

template <int MS, bool PREC, class Src, class Sink>
__device__ __forceinline__ void split_vcycle_levels(int levels, const Src& Y, const float* pyr, int l, int c, int R0,
                                                    const Sink& put) {
  if (levels == 2)
    split_vcycle<MS, 2, PREC>(Y, pyr, l, c, R0, put);
  else if (levels == 3)
    split_vcycle<MS, 3, PREC>(Y, pyr, l, c, R0, put);
  else if (Split<MS>::LMAX == 4 || levels == 4)
    split_vcycle<MS, 4, PREC>(Y, pyr, l, c, R0, put);
  else
    split_vcycle<MS, Split<MS>::LMAX, PREC>(Y, pyr, l, c, R0, put);
}

template <int MS, bool ATOM>
__device__ __forceinline__ void split_grad_body(const StepArgs& A, int win, int tile) {
  using S = Split<MS>;
  constexpr int E = S::E, G = S::G, NL = S::NL;
  __shared__ float2 X[NL * MS];
  const int tid = threadIdx.x, l = tid % NL, g = tid / NL, c = tile * NL + l;
  const int k = A.idx[win];
  const bool ok = (unsigned)k < (unsigned)A.n_pos;  // a skipped window waits as well: see split_exit_kernel
  const int pr = A.pos[ok ? 2 * k : 0], pc = A.pos[ok ? 2 * k + 1 : 1];
  const float2* zp = A.z + (size_t)(pr + g) * A.n_cols + pc + c;
  const float2* qp = A.Q + g * MS + c;
  const size_t zs = (size_t)G * A.n_cols;
  grid_dep_wait();
  if (!ok) return;
  if (!ATOM) grid_dep_launch();  // the ordered update lists its windows meanwhile
  float2* col = A.contrib + (size_t)win * S::M + c;
  float2 x[E];
#pragma unroll
  for (int j = 0; j < E / G; ++j)
#pragma unroll
    for (int k2 = 0; k2 < G; ++k2) x[j * G + k2] = __ldcg(col + (g + G * j + E * k2) * MS);
#pragma unroll
  for (int j = 0; j < E / G; ++j) {
    const int k1 = g + G * j;
    float2 v[G];
#pragma unroll
    for (int k2 = 0; k2 < G; ++k2) v[k2] = x[j * G + k2];
    dft_reg<G, true>(v);
#pragma unroll
    for (int gp = 0; gp < G; ++gp)
      X[(k1 * G + gp) * NL + l] = gp ? twmul<true>(v[gp], __ldg(&A.tw[(gp * k1) & (MS - 1)])) : v[0];
  }
  __syncthreads();
#pragma unroll
  for (int k1 = 0; k1 < E; ++k1) x[k1] = X[(k1 * G + g) * NL + l];
  dft_reg<E, true>(x);
  // g^0 = conj(Q)(R_k - Q z_k) at rows g + G e of this column
  float gn2 = 0.f;
#pragma unroll
  for (int e = 0; e < E; ++e) {
    const float2 q = __ldg(qp + e * (G * MS));
    x[e] = cmul_cj(q, csub(x[e], cmul(q, __ldg(zp + e * zs))));
    gn2 += cabs2(x[e]);
  }
  IncrementSink<MS, ATOM> put;
  put.a = &A;
  put.out = A.contrib + (size_t)win * S::M;
  put.pr = pr;
  put.pc = pc;
  const bool direct = A.levels == 1 || A.grad_only;
  if (direct) {
#pragma unroll
    for (int e = 0; e < E; ++e) put(g + G * e, c, x[e]);
  } else {
    __syncthreads();  // the exchange has been read
#pragma unroll
    for (int e = 0; e < E; ++e) X[(g + G * e) * NL + l] = x[e];
  }
  split_sum<S::T>(gn2, A.part + (size_t)(win * S::TILES + tile) * 2 + 1);  // its barrier: g^0 in place
  if (direct) return;
  split_vcycle_levels<MS, false>(
      A.levels, [&](int r, int j) { return X[r * NL + j]; }, A.pyr, l, c, g * E, put);
}

// One problem.  Every block of a kernel waits for the kernel before, also
// where its window is skipped, then lets the next one's blocks be set up, so
// that a kernel's blocks start once every kernel but the one before theirs has
// ended: the update reads the corners that the exit kernel wrote before its
// own wait, which is for the gradient kernel, and would read an earlier step's
// if a grid of skipped windows ended without having waited.
template <int MS>
__global__ void __launch_bounds__(Split<MS>::T, Split<MS>::MB[0]) split_exit_kernel(const __grid_constant__ StepArgs A, bool early) {
  split_exit_body<MS>(A, blockIdx.x / Split<MS>::TILES, blockIdx.x % Split<MS>::TILES, early);
}
template <int MS>
__global__ void __launch_bounds__(Split<MS>::T, Split<MS>::MB[1]) split_project_kernel(const __grid_constant__ StepArgs A) {
  split_project_body<MS>(A, blockIdx.x / Split<MS>::TILES, blockIdx.x % Split<MS>::TILES);
}
template <int MS, bool ATOM>
__global__ void __launch_bounds__(Split<MS>::T, Split<MS>::MB[2]) split_grad_kernel(const __grid_constant__ StepArgs A) {
  split_grad_body<MS, ATOM>(A, blockIdx.x / Split<MS>::TILES, blockIdx.x % Split<MS>::TILES);
}

// Several problems: window i of the launch is window slot map[i].y of the
// problem table[map[i].x].
template <int MS, int STAGE>
__global__ void __launch_bounds__(Split<MS>::T, Split<MS>::MB[STAGE])
    split_kernel_batched(const StepArgs* __restrict__ table, const int2* __restrict__ map) {
  __shared__ StepArgs args;
  const int2 ent = map[blockIdx.x / Split<MS>::TILES];
  if (threadIdx.x == 0) args = table[ent.x];
  __syncthreads();
  const int tile = blockIdx.x % Split<MS>::TILES;
  if (STAGE == 0) split_exit_body<MS>(args, ent.y, tile, false);
  if (STAGE == 1) split_project_body<MS>(args, ent.y, tile);
  if (STAGE == 2) split_grad_body<MS, false>(args, ent.y, tile);
}
