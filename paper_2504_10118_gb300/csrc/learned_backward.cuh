// learned_backward.cuh -- the network's parameter gradient.  Included by
// magpie.cu inside namespace magpie_impl, after learned.cuh.
//
// Every contraction of the backward pass runs on the tensor cores without
// giving up FP32 operands: a gradient x is held as three BF16 planes,
// x = x1 + x2 + x3 exactly (8 + 8 + 8 significant bits; below about 2^-110 the
// last plane is a BF16 subnormal and drops bits), the other operand
// (weights, stored activations) is BF16 already, so a product is three exact
// BF16 products, and the FP32 accumulators of at most six instructions are
// added to FP32 totals with ordinary rounded additions.
//
// Layers whose input is upsampled (the last two) first sum the output
// gradients that read one input pixel through one tap,
//   S[q][tap][co] = sum of dz[p][co] over the outputs p whose tap reads q,
// in FP32: both gradients of such a layer are then plain products over the
// input pixels, dW = S^T a and dx = S W, with 4 or 16 times fewer terms.
//
// Launches for a batch: grad_last_kernel (layer 5 whole), grad_sum4_kernel
// (S of layer 4), one grad_gemm_kernel per layer 4 .. 1 whose blocks are part
// data gradient and part weight gradient (the two are independent),
// grad_first_kernel (layer 0) and grad_reduce_kernel (all partial sums).
// What bounds them: a few hundred MFLOP each, so a block's chain of loads and
// MMAs and the launch itself, not the tensor pipe.  The gradient alone (all
// launches above) of a 64-window batch at h = 32 (GB300): 2.36 ms with the
// former FP32 kernels (one thread per input gradient, 64 x 64 FP32 tiles for
// the weights), 0.16 ms now; the per-layer relative error against FP64 went
// from 1.4e-7 .. 2.4e-6 to 4e-8 .. 2.9e-7.
#pragma once

// ------------------------------------------------------------ three planes
// x = p[0] + p[1] + p[2] by truncation, so that nothing overflows; a
// non-finite x keeps its class in the first plane.
__device__ __forceinline__ void split3(float x, uint16_t (&p)[3]) {
  const uint32_t u = __float_as_uint(x);
  if ((u & 0x7f800000u) == 0x7f800000u) {
    p[0] = (uint16_t)((u >> 16) | ((u & 0x007fffffu) ? 0x40u : 0u));
    p[1] = p[2] = 0;
    return;
  }
  const float h = __uint_as_float(u & 0xffff0000u);
  const float r = x - h;  // exact
  const uint32_t v = __float_as_uint(r);
  const float m = __uint_as_float(v & 0xffff0000u);
  p[0] = (uint16_t)(u >> 16);
  p[1] = (uint16_t)(v >> 16);
  p[2] = (uint16_t)(__float_as_uint(r - m) >> 16);
}

__device__ __forceinline__ void ldsm4(uint32_t (&r)[4], uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(addr));
}
__device__ __forceinline__ void ldsm4t(uint32_t (&r)[4], uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(addr));
}
__device__ __forceinline__ void cp16(uint32_t dst, const void* src, bool ok) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(ok ? 16 : 0) : "memory");
}

// One layer's two gradients (layers 1 .. 4).
struct GradGemm {
  // weight gradient: C[m][n] = sum_p D[p][m] A[p][n] over chunks of pixels
  const uint16_t* d;   // [3][K][M] planes: dz of the layer (M = Cout), or S of an upsampled one (M = 9 Cout)
  size_t dplane;       // elements of a plane
  const bf16* act;     // [B][Hin][Hin][Cin] the layer's input
  float* part;         // [chunks][M N + M] partial sums (the last M: the bias gradient, not for S)
  int M, N, K, chunk;  // N = 9 Cin (S: Cin); K pixels; pixels per chunk (a multiple of 32)
  int Cin, Cout, lho, lhin;  // log2 of the output and input sides
  int gather;          // 1: row p of A is the tap's input pixel (stride 2); 0: row p of the input
  int wm, wn, wblocks; // 64-wide tiles of the weight gradient, its blocks
  // data gradient: X[q][ci] = sum_k D[q'][k] W[k][ci], masked by the input's ReLU
  const bf16* w;       // [Cout][9][Cin]
  void* out;           // planes [3][pixels][Cin], or FP32 [pixels][Cin]
  size_t oplane;
  int out_f32;
  int rows;            // input pixels per parity class (gather), or all of them
  int xm, xn, xblocks; // tiles of one class, blocks of all classes
};

constexpr int kGradStages = 3;
template <int BM, int BN, bool AT>
struct GradTile {
  static constexpr int APITCH = (AT ? BM : 32) * 2 + 16, AROWS = AT ? 32 : BM;
  static constexpr int BPITCH = BN * 2 + 16;
  static constexpr int APLANE = AROWS * APITCH, STAGE = 3 * APLANE + 32 * BPITCH;
  static constexpr int SMEM = kGradStages * STAGE;
};

// The product of a block's BM x BN tile over `steps` steps of 32 terms.
// Four warps, 2 x 2, each WM x WN.  load(stage address, step) issues the
// step's cp.async; A^T in shared memory (AT: [k][m], weight gradient) or
// [m][k].  bias: a column of ones beside the tile (its sums in bsum).
template <int BM, int BN, bool AT, class Load>
__device__ __forceinline__ void grad_tile(uint32_t sm, int steps, Load load, float (&tot)[BM / 32][BN / 16][4],
                                          bool bias, float (&bsum)[BM / 32][2]) {
  using T = GradTile<BM, BN, AT>;
  constexpr int MT = BM / 32, NT = BN / 16, WM = BM / 2, WN = BN / 2;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int wm = warp & 1, wn = warp >> 1;
#pragma unroll
  for (int i = 0; i < MT; ++i) {
    bsum[i][0] = bsum[i][1] = 0.f;
#pragma unroll
    for (int j = 0; j < NT; ++j)
#pragma unroll
      for (int e = 0; e < 4; ++e) tot[i][j][e] = 0.f;
  }
  const int l7 = lane & 7, mi = lane >> 3;
  const uint32_t ones[2] = {0x3f803f80u, 0x3f803f80u};
#pragma unroll
  for (int s = 0; s < kGradStages - 1; ++s) {
    if (s < steps) load(sm + (uint32_t)(s * T::STAGE), s);
    asm volatile("cp.async.commit_group;" ::: "memory");
  }
  for (int s = 0; s < steps; ++s) {
    asm volatile("cp.async.wait_group %0;" ::"n"(kGradStages - 2) : "memory");
    __syncthreads();
    const int nx = s + kGradStages - 1;
    if (nx < steps) load(sm + (uint32_t)((nx % kGradStages) * T::STAGE), nx);
    asm volatile("cp.async.commit_group;" ::: "memory");
    const uint32_t sa = sm + (uint32_t)((s % kGradStages) * T::STAGE), sb = sa + 3 * T::APLANE;
    float acc[MT][NT][4], bac[MT][4];
#pragma unroll
    for (int i = 0; i < MT; ++i) {
#pragma unroll
      for (int e = 0; e < 4; ++e) bac[i][e] = 0.f;
#pragma unroll
      for (int j = 0; j < NT; ++j)
#pragma unroll
        for (int e = 0; e < 4; ++e) acc[i][j][e] = 0.f;
    }
#pragma unroll
    for (int kk = 0; kk < 32; kk += 16) {
      uint32_t b[NT][2];
#pragma unroll
      for (int j = 0; j < NT; j += 2) {
        uint32_t r[4];
        ldsm4t(r, sb + (uint32_t)((kk + l7 + (mi & 1) * 8) * T::BPITCH + (wn * WN + j * 8 + (mi >> 1) * 8) * 2));
        b[j][0] = r[0];
        b[j][1] = r[1];
        b[j + 1][0] = r[2];
        b[j + 1][1] = r[3];
      }
#pragma unroll
      for (int p = 2; p >= 0; --p)  // the smallest plane first
#pragma unroll
        for (int i = 0; i < MT; ++i) {
          uint32_t a[4];
          const uint32_t pl = sa + (uint32_t)(p * T::APLANE);
          if (AT)
            ldsm4t(a, pl + (uint32_t)((kk + l7 + (mi >> 1) * 8) * T::APITCH + (wm * WM + i * 16 + (mi & 1) * 8) * 2));
          else
            ldsm4(a, pl + (uint32_t)((wm * WM + i * 16 + l7 + (mi & 1) * 8) * T::APITCH + (kk + (mi >> 1) * 8) * 2));
#pragma unroll
          for (int j = 0; j < NT; ++j) mma_bf16(acc[i][j], a, b[j]);
          if (bias) mma_bf16(bac[i], a, ones);
        }
    }
#pragma unroll
    for (int i = 0; i < MT; ++i) {
      bsum[i][0] += bac[i][0];
      bsum[i][1] += bac[i][2];
#pragma unroll
      for (int j = 0; j < NT; ++j)
#pragma unroll
        for (int e = 0; e < 4; ++e) tot[i][j][e] += acc[i][j][e];
    }
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
}

// A 64 x 64 tile of the weight gradient over one chunk of pixels.
__device__ __forceinline__ void grad_weights(const GradGemm& a, uint32_t sm, int blk) {
  using T = GradTile<64, 64, true>;
  const int tid = threadIdx.x, tiles = a.wm * a.wn;
  const int z = blk / tiles, tile = blk - z * tiles, m0 = (tile / a.wn) * 64, n0 = (tile % a.wn) * 64;
  const int p0 = z * a.chunk, p1 = min(a.K, p0 + a.chunk);
  // this thread's chunk of eight columns and its first row of a step
  const int c = tid & 7, r0 = tid >> 3;
  const int n = n0 + 8 * c;
  const int tap = a.gather ? n / a.Cin : 0, ci = a.gather ? n - tap * a.Cin : n;
  const int ky = tap / 3, kx = tap - 3 * ky, Ho = 1 << a.lho, Hin = 1 << a.lhin;
  auto load = [&](uint32_t st, int s) {
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const int r = r0 + 16 * i, p = p0 + 32 * s + r;
      const bool ok = p < p1;
#pragma unroll
      for (int pl = 0; pl < 3; ++pl)
        cp16(st + (uint32_t)(pl * T::APLANE + r * T::APITCH + c * 16),
             a.d + pl * a.dplane + (size_t)(ok ? p : 0) * a.M + m0 + 8 * c, ok);
      bool in = ok && n < a.N;
      size_t pix = p;
      if (a.gather) {
        const int ox = p & (Ho - 1), oy = (p >> a.lho) & (Ho - 1), b = p >> (2 * a.lho);
        const int iy = 2 * oy + ky - 1, ix = 2 * ox + kx - 1;
        in = in && (unsigned)iy < (unsigned)Hin && (unsigned)ix < (unsigned)Hin;
        pix = ((size_t)b * Hin + iy) * Hin + ix;
      }
      cp16(st + (uint32_t)(3 * T::APLANE + r * T::BPITCH + c * 16), a.act + (in ? pix * a.Cin + ci : 0), in);
    }
  };
  float tot[2][4][4], bs[2][2];
  const bool bias = n0 == 0 && a.gather;
  grad_tile<64, 64, true>(sm, (p1 - p0 + 31) / 32, load, tot, bias, bs);
  float* out = a.part + (size_t)z * ((size_t)a.M * a.N + a.M);
  const int lane = tid & 31, warp = tid >> 5, g = lane >> 2, t = lane & 3;
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const int m = m0 + (warp & 1) * 32 + i * 16 + g;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int nn = n0 + (warp >> 1) * 32 + j * 8 + 2 * t;
      if (nn >= a.N) continue;
      *reinterpret_cast<float2*>(out + (size_t)m * a.N + nn) = make_float2(tot[i][j][0], tot[i][j][1]);
      *reinterpret_cast<float2*>(out + (size_t)(m + 8) * a.N + nn) = make_float2(tot[i][j][2], tot[i][j][3]);
    }
    if (bias && (warp >> 1) == 0 && t == 0) {
      out[(size_t)a.M * a.N + m] = bs[i][0];
      out[(size_t)a.M * a.N + m + 8] = bs[i][1];
    }
  }
}

// A BM x BN tile of the data gradient.  Stride 2 (gather): the input pixels
// of one parity class (iy, ix parities), which share their 1, 2 or 4 taps;
// upsampled: one product over k = (co, tap).
template <int BM, int BN>
__device__ __forceinline__ void grad_data(const GradGemm& a, uint32_t sm, int blk) {
  using T = GradTile<BM, BN, false>;
  const int tid = threadIdx.x, tiles = a.xm * a.xn;
  // the class with the most taps first
  const int cls = a.gather ? 3 - blk / tiles : 0, tile = blk % tiles;
  const int py = cls >> 1, px = cls & 1, m0 = (tile / a.xn) * BM, n0 = (tile % a.xn) * BN;
  const int Ho = 1 << a.lho, Hin = 1 << a.lhin;
  const int ntap = a.gather ? (1 + py) * (1 + px) : 1, per = (a.gather ? a.Cout : a.M) / 32;
  const int ca = tid & 3, ra = tid >> 2;
  constexpr int CB = BN / 8, RB = 128 / CB;
  const int cb = tid % CB, rb = tid / CB;
  auto load = [&](uint32_t st, int s) {
    const int j = s / per, k0 = (s - j * per) * 32;
    // tap j of the class: along a row of parity 1, taps 0 (one output down) and 2
    const int jy = py ? j / (1 + px) : 0, jx = px ? j & 1 : 0;
    const int ky = py ? 2 * jy : 1, kx = px ? 2 * jx : 1;
    const int dy = py ? 1 - jy : 0, dx = px ? 1 - jx : 0;
#pragma unroll
    for (int i = 0; i < BM / 32; ++i) {
      const int r = ra + 32 * i, q = m0 + r;
      bool ok = q < a.rows;
      size_t row = q;
      if (a.gather) {
        const int ox = (q & (Ho - 1)) + dx, oy = ((q >> a.lho) & (Ho - 1)) + dy, b = q >> (2 * a.lho);
        ok = ok && ox < Ho && oy < Ho;
        row = ((size_t)b * Ho + oy) * Ho + ox;
      }
      const uint16_t* src = a.d + (ok ? row * a.M + k0 + 8 * ca : 0);
#pragma unroll
      for (int pl = 0; pl < 3; ++pl)
        cp16(st + (uint32_t)(pl * T::APLANE + r * T::APITCH + ca * 16), src + pl * a.dplane, ok);
    }
    const bf16* wp = a.gather ? a.w + ((size_t)k0 * 9 + ky * 3 + kx) * a.Cin : a.w + (size_t)k0 * a.Cin;
    const size_t ld = a.gather ? 9 * (size_t)a.Cin : (size_t)a.Cin;
#pragma unroll
    for (int i = 0; i < 32 / RB; ++i) {
      const int r = rb + RB * i;
      cp16(st + (uint32_t)(3 * T::APLANE + r * T::BPITCH + cb * 16), wp + r * ld + n0 + 8 * cb, true);
    }
  };
  constexpr int MT = BM / 32, NT = BN / 16;
  float tot[MT][NT][4], bs[MT][2];
  grad_tile<BM, BN, false>(sm, ntap * per, load, tot, false, bs);
  const int lane = tid & 31, warp = tid >> 5, g = lane >> 2, t = lane & 3;
#pragma unroll
  for (int i = 0; i < MT; ++i)
#pragma unroll
    for (int hh = 0; hh < 2; ++hh) {
      const int q = m0 + (warp & 1) * (BM / 2) + i * 16 + g + 8 * hh;
      if (q >= a.rows) continue;
      size_t pix = q;
      if (a.gather) {
        const int x = q & (Ho - 1), y = (q >> a.lho) & (Ho - 1), b = q >> (2 * a.lho);
        pix = ((size_t)b * Hin + 2 * y + py) * Hin + 2 * x + px;
      }
#pragma unroll
      for (int j = 0; j < NT; ++j) {
        const int ci = n0 + (warp >> 1) * (BN / 2) + j * 8 + 2 * t;
        const size_t o = pix * a.Cin + ci;
        const __nv_bfloat162 m2 = *reinterpret_cast<const __nv_bfloat162*>(a.act + o);
        const float v0 = __low2float(m2) > 0.f ? tot[i][j][2 * hh] : 0.f;
        const float v1 = __high2float(m2) > 0.f ? tot[i][j][2 * hh + 1] : 0.f;
        if (a.out_f32) {
          *reinterpret_cast<float2*>(static_cast<float*>(a.out) + o) = make_float2(v0, v1);
        } else {
          uint16_t s0[3], s1[3];
          split3(v0, s0);
          split3(v1, s1);
#pragma unroll
          for (int pl = 0; pl < 3; ++pl)
            *reinterpret_cast<uint32_t*>(static_cast<uint16_t*>(a.out) + pl * a.oplane + o) =
                (uint32_t)s0[pl] | ((uint32_t)s1[pl] << 16);
        }
      }
    }
}

// Both gradients of a layer: data-gradient blocks first (the next layer's
// launch waits for them), weight-gradient blocks behind them.
template <int BM, int BN>
__global__ void __launch_bounds__(128) grad_gemm_kernel(const __grid_constant__ GradGemm a) {
  extern __shared__ __align__(16) unsigned char grad_raw[];
  const uint32_t sm = smem_addr(grad_raw);
  if ((int)blockIdx.x < a.xblocks)
    grad_data<BM, BN>(a, sm, blockIdx.x);
  else
    grad_weights(a, sm, blockIdx.x - a.xblocks);
}
template <int BM, int BN>
constexpr size_t grad_smem() {
  return GradTile<BM, BN, false>::SMEM > GradTile<64, 64, true>::SMEM ? GradTile<BM, BN, false>::SMEM
                                                                      : GradTile<64, 64, true>::SMEM;
}

// Layer 5 (64 -> 2, input upsampled by 4), whole, in FP32: per input pixel q
// the 9 x 2 sums S of the output gradients, dz4[q] = S W (masked), and the
// block's share of dW = S^T a, of the bias gradient (the centre tap's S covers
// every output once) and of layer 4's bias gradient.  Blocks of 256 threads
// take 32 input pixels at a time.
constexpr int kLastQ = 32, kLastPart = 18 * 64 + 2 + 64;
__global__ void __launch_bounds__(256) grad_last_kernel(const float* __restrict__ dy, const bf16* __restrict__ w,
                                                        const bf16* __restrict__ act, float* __restrict__ dz,
                                                        float* __restrict__ part, int nq, int lhin) {
  __shared__ float S[kLastQ][18], A[kLastQ][64], W[18][64], Z[kLastQ][64];
  const int tid = threadIdx.x, Hin = 1 << lhin, Ho = 4 * Hin;
  for (int i = tid; i < 18 * 64; i += 256) W[i / 64][i % 64] = __bfloat162float(w[i]);  // row co * 9 + tap
  float acc[5] = {}, extra = 0.f;  // dW entries tid + 256 u; db5 (tid < 2) or db4 (64 <= tid < 128)
  for (int q0 = blockIdx.x * kLastQ; q0 < nq; q0 += gridDim.x * kLastQ) {
    __syncthreads();
    for (int i = tid; i < kLastQ * 18; i += 256) {
      const int qq = i / 18, k = i - qq * 18, co = k / 9, tap = k - 9 * co, ky = tap / 3, kx = tap - 3 * ky;
      const int q = q0 + qq;
      float s = 0.f;
      if (q < nq) {
        const int ix = q & (Hin - 1), iy = (q >> lhin) & (Hin - 1), b = q >> (2 * lhin);
        const int y0 = max(0, 4 * iy + 1 - ky), y1 = min(Ho, 4 * iy + 5 - ky);
        const int x0 = max(0, 4 * ix + 1 - kx), x1 = min(Ho, 4 * ix + 5 - kx);
        for (int y = y0; y < y1; ++y)
          for (int x = x0; x < x1; ++x) s += __ldg(&dy[(((size_t)b * Ho + y) * Ho + x) * 2 + co]);
      }
      S[qq][k] = s;
    }
    for (int i = tid; i < kLastQ * 64; i += 256) {
      const int q = q0 + i / 64;
      A[i / 64][i % 64] = q < nq ? __bfloat162float(act[(size_t)q * 64 + i % 64]) : 0.f;
    }
    __syncthreads();
    for (int i = tid; i < kLastQ * 64; i += 256) {
      const int qq = i / 64, ci = i % 64;
      float v = 0.f;
#pragma unroll
      for (int k = 0; k < 18; ++k) v = fmaf(S[qq][k], W[k][ci], v);
      v = A[qq][ci] > 0.f ? v : 0.f;
      Z[qq][ci] = v;
      if (q0 + qq < nq) dz[(size_t)(q0 + qq) * 64 + ci] = v;
    }
#pragma unroll
    for (int u = 0; u < 5; ++u) {
      const int e = tid + 256 * u;
      if (e < 18 * 64) {
        float s = 0.f;
#pragma unroll 8
        for (int qq = 0; qq < kLastQ; ++qq) s = fmaf(S[qq][e / 64], A[qq][e % 64], s);
        acc[u] += s;
      }
    }
    __syncthreads();
    if (tid < 2 || (tid >= 64 && tid < 128)) {
      float s = 0.f;
      for (int qq = 0; qq < kLastQ; ++qq) s += tid < 2 ? S[qq][tid * 9 + 4] : Z[qq][tid - 64];
      extra += s;
    }
  }
  float* o = part + (size_t)blockIdx.x * kLastPart;
#pragma unroll
  for (int u = 0; u < 5; ++u)
    if (tid + 256 * u < 18 * 64) o[tid + 256 * u] = acc[u];
  if (tid < 2) o[18 * 64 + tid] = extra;
  if (tid >= 64 && tid < 128) o[18 * 64 + 2 + tid - 64] = extra;
}

// S of layer 4 (512 -> 64, input upsampled by 2), as planes: S[q][co * 9 + tap]
// sums dz4 over the up to four outputs whose tap reads input pixel q.  One
// thread per (q, co): the 4 x 4 outputs around q, then their nine 2 x 2 sums.
__global__ void __launch_bounds__(256) grad_sum4_kernel(const float* __restrict__ dz, uint16_t* __restrict__ S,
                                                        size_t plane, int nq, int lhin) {
  const int Hin = 1 << lhin, Ho = 2 * Hin;
  const size_t i = (size_t)blockIdx.x * 256 + threadIdx.x;
  if (i >= (size_t)nq * 64) return;
  const int co = (int)(i & 63), q = (int)(i >> 6);
  const int ix = q & (Hin - 1), iy = (q >> lhin) & (Hin - 1), b = q >> (2 * lhin);
  float v[4][4];  // outputs 2 iy - 1 .. 2 iy + 2, likewise along x
#pragma unroll
  for (int y = 0; y < 4; ++y)
#pragma unroll
    for (int x = 0; x < 4; ++x) {
      const int oy = 2 * iy - 1 + y, ox = 2 * ix - 1 + x;
      v[y][x] = ((unsigned)oy < (unsigned)Ho && (unsigned)ox < (unsigned)Ho)
                    ? __ldg(&dz[(((size_t)b * Ho + oy) * Ho + ox) * 64 + co])
                    : 0.f;
    }
#pragma unroll
  for (int ky = 0; ky < 3; ++ky)
#pragma unroll
    for (int kx = 0; kx < 3; ++kx) {
      // outputs with (o + k - 1) / 2 = i: o = 2 i + 1 - k and the next
      const int y = 2 - ky, x = 2 - kx;
      const float s = (v[y][x] + v[y][x + 1]) + (v[y + 1][x] + v[y + 1][x + 1]);
      uint16_t p[3];
      split3(s, p);
#pragma unroll
      for (int pl = 0; pl < 3; ++pl) S[pl * plane + (size_t)q * 576 + co * 9 + ky * 3 + kx] = p[pl];
    }
}

// Layer 0 (4 -> 32): dW[co][tap][ci] and the bias gradient, 32 x 37 sums over
// the output pixels.  A warp takes 16 pixels per step: the gradients as A
// fragments split in registers, the 9 x 4 inputs (and a one, the bias column)
// as B fragments gathered from the image; the block's warps are added at the
// end.
constexpr int kFirstPart = 32 * 37;
__global__ void __launch_bounds__(128) grad_first_kernel(const float* __restrict__ dz, const bf16* __restrict__ act,
                                                         float* __restrict__ part, int npix, int lh) {
  __shared__ float red[4][32][40];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, t = lane & 3, H = 1 << lh;
  const uint16_t* in = reinterpret_cast<const uint16_t*>(act);
  float tot[2][5][4] = {};
  for (int p0 = (blockIdx.x * 4 + warp) * 16; p0 < npix; p0 += gridDim.x * 64) {
    uint32_t a[3][2][4];  // planes, m tiles
#pragma unroll
    for (int mt = 0; mt < 2; ++mt)
#pragma unroll
      for (int r = 0; r < 4; ++r) {  // rows g (+ 8), pixels 2 t, 2 t + 1 (+ 8)
        const int co = mt * 16 + g + (r & 1) * 8, p = p0 + 2 * t + (r >> 1) * 8;
        uint16_t s0[3], s1[3];
        split3(p < npix ? __ldg(&dz[(size_t)p * 32 + co]) : 0.f, s0);
        split3(p + 1 < npix ? __ldg(&dz[(size_t)(p + 1) * 32 + co]) : 0.f, s1);
#pragma unroll
        for (int pl = 0; pl < 3; ++pl) a[pl][mt][r] = (uint32_t)s0[pl] | ((uint32_t)s1[pl] << 16);
      }
    uint32_t b[5][2];
#pragma unroll
    for (int hh = 0; hh < 2; ++hh) {
      uint16_t v[2][5];
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const int p = p0 + 2 * t + 8 * hh + e;
        const int x = p & (H - 1), y = (p >> lh) & (H - 1), bb = p >> (2 * lh);
#pragma unroll
        for (int nt = 0; nt < 5; ++nt) {
          const int n = nt * 8 + g, tap = n >> 2, iy = y + tap / 3 - 1, ix = x + tap % 3 - 1;
          const bool ok = p < npix && n < 36 && (unsigned)iy < (unsigned)H && (unsigned)ix < (unsigned)H;
          v[e][nt] = ok ? __ldg(&in[(((size_t)bb * H + iy) * H + ix) * 4 + (n & 3)]) : n == 36 ? 0x3f80 : 0;
        }
      }
#pragma unroll
      for (int nt = 0; nt < 5; ++nt) b[nt][hh] = (uint32_t)v[0][nt] | ((uint32_t)v[1][nt] << 16);
    }
#pragma unroll
    for (int mt = 0; mt < 2; ++mt)
#pragma unroll
      for (int nt = 0; nt < 5; ++nt) {
        float acc[4] = {};
#pragma unroll
        for (int pl = 2; pl >= 0; --pl) mma_bf16(acc, a[pl][mt], b[nt]);
#pragma unroll
        for (int e = 0; e < 4; ++e) tot[mt][nt][e] += acc[e];
      }
  }
#pragma unroll
  for (int mt = 0; mt < 2; ++mt)
#pragma unroll
    for (int nt = 0; nt < 5; ++nt)
#pragma unroll
      for (int e = 0; e < 4; ++e) red[warp][mt * 16 + g + (e >> 1) * 8][nt * 8 + 2 * t + (e & 1)] = tot[mt][nt][e];
  __syncthreads();
  float* o = part + (size_t)blockIdx.x * kFirstPart;
  for (int i = threadIdx.x; i < kFirstPart; i += 128) {
    // weights [co][36], then the 32 biases
    const int co = i < 32 * 36 ? i / 36 : i - 32 * 36, n = i < 32 * 36 ? i % 36 : 36;
    o[i] = (red[0][co][n] + red[1][co][n]) + (red[2][co][n] + red[3][co][n]);
  }
}

// grad[dst + i] = sum over chunks of src[chunk stride + i], i < n, for every
// segment.  Segments of 16 chunks and more are summed by eight threads per
// entry (each every eighth chunk, then in order), the others by one.
struct GradSeg {
  const float* src;
  int dst, n, chunks, block0, wide;
  size_t stride;
};
constexpr int kGradSegs = 8;
struct GradSegs {
  GradSeg s[kGradSegs];
  int n;
};
__global__ void __launch_bounds__(256) grad_reduce_kernel(const __grid_constant__ GradSegs G, float* __restrict__ grad) {
  __shared__ float red[8][32];
  int k = 0;
  while (k + 1 < G.n && (int)blockIdx.x >= G.s[k + 1].block0) ++k;
  const GradSeg& s = G.s[k];
  const int blk = (int)blockIdx.x - s.block0;
  if (!s.wide) {
    const int i = blk * 256 + threadIdx.x;
    if (i >= s.n) return;
    float v = 0.f;
    for (int c = 0; c < s.chunks; ++c) v += s.src[c * s.stride + i];
    grad[s.dst + i] = v;
    return;
  }
  const int e = threadIdx.x & 31, w = threadIdx.x >> 5, i = blk * 32 + e;
  float v = 0.f;
  if (i < s.n)
#pragma unroll 8
    for (int c = w; c < s.chunks; c += 8) v += s.src[c * s.stride + i];
  red[w][e] = v;
  __syncthreads();
  if (w == 0 && i < s.n) {
    float t = 0.f;
#pragma unroll
    for (int j = 0; j < 8; ++j) t += red[j][e];
    grad[s.dst + i] = t;
  }
}
