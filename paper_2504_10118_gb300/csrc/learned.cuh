// learned.cuh -- the learned coarse-level correction: the network's forward
// pass (BF16 tensor-core implicit GEMM, FP32 accumulation), its Adam step
// (FP32; the backward pass is in learned_backward.cuh), and the per-window
// kernels that build the network's input on the coarsest grid of the V-cycle and apply its proposal with the
// surrogate acceptance test.  Included by magpie.cu inside its anonymous
// namespace.
//
// The paper has no network; its MAGPS (Algorithm MAGPS) ends the recursion on
// the coarsest grid with one proximal step, e_plain = g_H / w_H.  Here a
// six-layer convolutional network sees (z_H, e_plain / s) on that grid, s the
// RMS of e_plain over the window, and proposes e_nn = e_plain + s y.  Each
// window keeps the V-cycle output built on e_nn only when the window's
// quadratic surrogate 1/2 ||Q x - R_k||^2 (Eq. quadratic_surrogate) is no
// larger there than at the output built on e_plain.
#pragma once
#include <cuda_bf16.h>

constexpr int kCnnLayers = 6;
struct CnnLayer {
  int cin, cout, stride, up, relu;
};
// 3x3 convolutions, zero padding 1, nearest-neighbour upsampling of the input
// by `up`; sides h, h, h/2, h/4, h/8, h/4, h.
constexpr CnnLayer kCnn[kCnnLayers] = {
    {4, 32, 1, 1, 1}, {32, 64, 2, 1, 1}, {64, 128, 2, 1, 1}, {128, 512, 2, 1, 1}, {512, 64, 1, 2, 1}, {64, 2, 1, 4, 0},
};

typedef __nv_bfloat16 bf16;

// ------------------------------------------------------------ forward (MMA)
struct ConvFwd {
  const bf16* in;     // [B][Hin][Hin][Cin]
  const bf16* w;      // [Cout][3][3][Cin]
  const float* bias;  // [Cout]
  void* out;          // [B][Ho][Ho][Cout]: bf16 (hidden layers) or float (last)
  float* part;        // split-K: [splits][Mtot][Cout] partial sums, else null
  int B, Hin, Cin, Cout, stride, up, Ho, relu, out_f32;
  int K;       // 9 Cin
  int ksplit;  // K elements per split (multiple of 32)
  int lho, lup;  // log2 of Ho and up
  const float* x;  // first layer on the direct kernel: the FP32 input, rounded to BF16 into x16 as it is read
  uint2* x16;
};

__device__ __forceinline__ void mma_bf16(float* c, const uint32_t* a, const uint32_t* b) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};\n"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

// Implicit GEMM: rows = output pixels (b, oy, ox), columns = output channels,
// k = (ky, kx, ci).  Four warps; BM x BN tile, BK = 32 per stage.
template <int BM, int BN>
__global__ void __launch_bounds__(128) conv_fwd_kernel(const ConvFwd a) {
  constexpr int BK = 32, LDS = BK + 8;
  constexpr int WARPS_M = BM / 32, WARPS_N = 4 / WARPS_M, WTN = BN / WARPS_N, WN = WTN / 8;
  static_assert(WARPS_M * WARPS_N == 4 && WN >= 1, "tile");
  __shared__ __align__(16) bf16 As[BM * LDS];
  __shared__ __align__(16) bf16 Bs[BN * LDS];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int wm = warp % WARPS_M, wn = warp / WARPS_M;
  const int g = lane >> 2, t = lane & 3;
  const int HoHo = a.Ho * a.Ho;
  const int Mtot = a.B * HoHo;
  const int bm = blockIdx.x * BM, bn = blockIdx.y * BN;
  const int kbeg = blockIdx.z * a.ksplit;
  const int kend = min(a.K, kbeg + a.ksplit);
  const int Hv = a.Hin * a.up;
  const bool vec = (a.Cin % BK) == 0;
  float acc[2][WN][4];
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < WN; ++j)
#pragma unroll
      for (int e = 0; e < 4; ++e) acc[i][j][e] = 0.f;

  // global -> registers (the next stage, while the current one is multiplied)
  constexpr int AC = (BM * 4 + 127) / 128, BC = (BN * 4 + 127) / 128;
  uint4 ra[AC], rb[BC];
  auto load_a = [&](int c, int k0) -> uint4 {
    const int row = c >> 2, qd = c & 3;
    const int p = bm + row;
    uint4 v = make_uint4(0u, 0u, 0u, 0u);
    if (p < Mtot) {
      const int b = p / HoHo, rem = p - b * HoHo;
      const int oy = rem / a.Ho, ox = rem - oy * a.Ho;
      if (vec) {
        const int tap = k0 / a.Cin, ci0 = k0 - tap * a.Cin + 8 * qd;
        const int ky = tap / 3, kx = tap - 3 * ky;
        const int vy = oy * a.stride + ky - 1, vx = ox * a.stride + kx - 1;
        if (vy >= 0 && vy < Hv && vx >= 0 && vx < Hv) {
          const int iy = vy / a.up, ix = vx / a.up;
          v = *reinterpret_cast<const uint4*>(a.in + ((size_t)(b * a.Hin + iy) * a.Hin + ix) * a.Cin + ci0);
        }
      } else {
        bf16 e8[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const int k = k0 + 8 * qd + j;
          bf16 val = __float2bfloat16_rn(0.f);
          if (k < a.K) {
            const int tap = k / a.Cin, ci = k - tap * a.Cin;
            const int ky = tap / 3, kx = tap - 3 * ky;
            const int vy = oy * a.stride + ky - 1, vx = ox * a.stride + kx - 1;
            if (vy >= 0 && vy < Hv && vx >= 0 && vx < Hv)
              val = a.in[((size_t)(b * a.Hin + vy / a.up) * a.Hin + vx / a.up) * a.Cin + ci];
          }
          e8[j] = val;
        }
        v = *reinterpret_cast<const uint4*>(e8);
      }
    }
    return v;
  };
  auto load_b = [&](int c, int k0) -> uint4 {
    const int row = c >> 2, qd = c & 3;
    const int co = bn + row;
    uint4 v = make_uint4(0u, 0u, 0u, 0u);
    if (co < a.Cout) {
      const bf16* src = a.w + (size_t)co * a.K + k0 + 8 * qd;
      if (vec) {
        v = *reinterpret_cast<const uint4*>(src);
      } else {
        bf16 e8[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) e8[j] = (k0 + 8 * qd + j < a.K) ? src[j] : __float2bfloat16_rn(0.f);
        v = *reinterpret_cast<const uint4*>(e8);
      }
    }
    return v;
  };
  auto fetch = [&](int k0) {
#pragma unroll
    for (int u = 0; u < AC; ++u) {
      const int c = tid + 128 * u;
      if (c < BM * 4) ra[u] = load_a(c, k0);
    }
#pragma unroll
    for (int u = 0; u < BC; ++u) {
      const int c = tid + 128 * u;
      if (c < BN * 4) rb[u] = load_b(c, k0);
    }
  };
  if (kbeg < kend) fetch(kbeg);
  for (int k0 = kbeg; k0 < kend; k0 += BK) {
#pragma unroll
    for (int u = 0; u < AC; ++u) {
      const int c = tid + 128 * u;
      if (c < BM * 4) *reinterpret_cast<uint4*>(&As[(c >> 2) * LDS + 8 * (c & 3)]) = ra[u];
    }
#pragma unroll
    for (int u = 0; u < BC; ++u) {
      const int c = tid + 128 * u;
      if (c < BN * 4) *reinterpret_cast<uint4*>(&Bs[(c >> 2) * LDS + 8 * (c & 3)]) = rb[u];
    }
    __syncthreads();
    if (k0 + BK < kend) fetch(k0 + BK);
#pragma unroll
    for (int kk = 0; kk < BK; kk += 16) {
      uint32_t af[2][4], bfr[WN][2];
#pragma unroll
      for (int mi = 0; mi < 2; ++mi) {
        const int r = wm * 32 + mi * 16 + g;
        af[mi][0] = *reinterpret_cast<const uint32_t*>(&As[r * LDS + kk + 2 * t]);
        af[mi][1] = *reinterpret_cast<const uint32_t*>(&As[(r + 8) * LDS + kk + 2 * t]);
        af[mi][2] = *reinterpret_cast<const uint32_t*>(&As[r * LDS + kk + 8 + 2 * t]);
        af[mi][3] = *reinterpret_cast<const uint32_t*>(&As[(r + 8) * LDS + kk + 8 + 2 * t]);
      }
#pragma unroll
      for (int j = 0; j < WN; ++j) {
        const int n = wn * WTN + j * 8 + g;
        bfr[j][0] = *reinterpret_cast<const uint32_t*>(&Bs[n * LDS + kk + 2 * t]);
        bfr[j][1] = *reinterpret_cast<const uint32_t*>(&Bs[n * LDS + kk + 8 + 2 * t]);
      }
#pragma unroll
      for (int mi = 0; mi < 2; ++mi)
#pragma unroll
        for (int j = 0; j < WN; ++j) mma_bf16(acc[mi][j], af[mi], bfr[j]);
    }
    __syncthreads();
  }

  // ---- epilogue: C fragment (row g / g+8, columns 2t, 2t+1)
#pragma unroll
  for (int mi = 0; mi < 2; ++mi)
#pragma unroll
    for (int j = 0; j < WN; ++j) {
      const int co = bn + wn * WTN + j * 8 + 2 * t;
#pragma unroll
      for (int hh = 0; hh < 2; ++hh) {
        const int r = bm + wm * 32 + mi * 16 + g + 8 * hh;
        if (r >= Mtot || co >= a.Cout) continue;
        float v0 = acc[mi][j][2 * hh], v1 = acc[mi][j][2 * hh + 1];
        if (a.part) {
          *reinterpret_cast<float2*>(&a.part[((size_t)blockIdx.z * Mtot + r) * a.Cout + co]) = make_float2(v0, v1);
          continue;
        }
        v0 += a.bias[co];
        v1 += a.bias[co + 1];
        if (a.relu) {
          v0 = fmaxf(v0, 0.f);
          v1 = fmaxf(v1, 0.f);
        }
        if (a.out_f32)
          *reinterpret_cast<float2*>(&static_cast<float*>(a.out)[(size_t)r * a.Cout + co]) = make_float2(v0, v1);
        else
          *reinterpret_cast<__nv_bfloat162*>(&static_cast<bf16*>(a.out)[(size_t)r * a.Cout + co]) =
              __floats2bfloat162_rn(v0, v1);
      }
    }
}

// Direct convolutions for the thin layers, where an implicit-GEMM tile would
// be mostly padding.  Both read the BF16 inputs and weights (exact in FP32)
// and accumulate in FP32; consecutive lanes take consecutive 16-byte pieces of
// one pixel's channels, so a warp's loads and stores are contiguous.
//
// Few outputs (the last layer, 64 -> 2, input upsampled by 4): eight lanes per
// group of four output pixels of one row, which share their input pixels
// (three per tap row); lane `part` holds input channels 8 part .. 8 part + 7,
// and the eight partial sums of each output are added with butterfly shuffles.
// A tap's weights, FP32 in shared memory, are read once for the four pixels.
// Bound by its chain of loads and shuffles; 64 windows at h = 32: 9.3 us,
// against 20.3 with one output pixel per eight lanes, whose weights and
// inputs were read and converted for every pixel (same sums, same order).
// Needs `in` 16-byte aligned.
__global__ void __launch_bounds__(256) conv_thin_out_kernel(const ConvFwd a) {
  constexpr int CIN = 64, COUT = 2, S = CIN / 8;
  __shared__ __align__(16) float wsm[9 * COUT * CIN];
  for (int i = threadIdx.x; i < 9 * COUT * CIN; i += blockDim.x) {
    const int co = i / (9 * CIN), r = i - co * 9 * CIN, tap = r / CIN, ci = r - tap * CIN;
    wsm[(tap * COUT + co) * CIN + ci] = __bfloat162float(a.w[i]);
  }
  grid_dep_wait();
  grid_dep_launch();
  __syncthreads();
  const int Hq = a.Hin, HHq = a.Ho * Hq, groups = a.B * HHq;  // groups of four pixels: Ho rows x Hin columns
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const bool live = t < (long long)groups * S;  // whole groups: S divides 32
  const int grp = live ? (int)(t / S) : 0, part = (int)(t % S);
  const int b = grp / HHq, rem = grp - b * HHq, oy = rem / Hq, q = rem - oy * Hq;
  float acc[4][COUT];
#pragma unroll
  for (int j = 0; j < 4; ++j)
#pragma unroll
    for (int co = 0; co < COUT; ++co) acc[j][co] = 0.f;
#pragma unroll
  for (int ky = 0; ky < 3; ++ky) {
    const int vy = oy + ky - 1;
    if (!live || vy < 0 || vy >= a.Ho) continue;
    const bf16* rowp = a.in + ((size_t)(b * a.Hin + (vy >> 2)) * a.Hin + q) * CIN + part * 8;
    float x[3][8];  // input columns q - 1, q, q + 1
    bool ok[3];
#pragma unroll
    for (int e = 0; e < 3; ++e) {
      ok[e] = e == 0 ? q > 0 : e == 2 ? q + 1 < Hq : true;
      const uint4 raw = ok[e] ? __ldcg(reinterpret_cast<const uint4*>(rowp + (e - 1) * CIN)) : make_uint4(0, 0, 0, 0);
      const __nv_bfloat162* xh = reinterpret_cast<const __nv_bfloat162*>(&raw);
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        x[e][2 * j] = __low2float(xh[j]);
        x[e][2 * j + 1] = __high2float(xh[j]);
      }
    }
#pragma unroll
    for (int kx = 0; kx < 3; ++kx)
#pragma unroll
      for (int co = 0; co < COUT; ++co) {
        const float4* wr = reinterpret_cast<const float4*>(&wsm[((ky * 3 + kx) * COUT + co) * CIN + part * 8]);
        const float4 w0 = wr[0], w1 = wr[1];
        const float wv[8] = {w0.x, w0.y, w0.z, w0.w, w1.x, w1.y, w1.z, w1.w};
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const int e = (j + kx - 1 < 0) ? 0 : (j + kx - 1 > 3) ? 2 : 1;
          if (!ok[e]) continue;
#pragma unroll
          for (int c = 0; c < 8; ++c) acc[j][co] = fmaf(x[e][c], wv[c], acc[j][co]);
        }
      }
  }
#pragma unroll
  for (int j = 0; j < 4; ++j)
#pragma unroll
    for (int co = 0; co < COUT; ++co)
#pragma unroll
      for (int off = S / 2; off > 0; off >>= 1) acc[j][co] += __shfl_xor_sync(0xffffffffu, acc[j][co], off);
  if (!live || part != 0) return;
  float v[4][COUT];
#pragma unroll
  for (int j = 0; j < 4; ++j)
#pragma unroll
    for (int co = 0; co < COUT; ++co) v[j][co] = acc[j][co] + a.bias[co];
  float4* o = reinterpret_cast<float4*>(static_cast<float*>(a.out) + ((size_t)(b * a.Ho + oy) * a.Ho + 4 * q) * COUT);
  o[0] = make_float4(v[0][0], v[0][1], v[1][0], v[1][1]);
  o[1] = make_float4(v[2][0], v[2][1], v[3][0], v[3][1]);
}

// Few inputs (the first layer, 4 -> 32): four lanes per group of four output
// pixels of one row, lane `part` computing outputs 8 part .. 8 part + 7 of all
// four from the 3 x 6 inputs around them.  A tap's weights (FP32 [tap][ci][co]
// in shared memory) are read once for the four pixels, the FP32 input is
// rounded to BF16 as it is read and kept for the backward pass (no conversion
// pass).  64 windows at h = 32: 12 us, against 2.5 + 16.4 with a conversion
// pass and one pixel per four lanes, bound by its weight reads (same sums,
// same order).
__global__ void __launch_bounds__(128) conv_thin_in_kernel(const ConvFwd a) {
  constexpr int CIN = 4, COUT = 32;
  __shared__ __align__(16) float wsm[9 * CIN * COUT];
  grid_dep_wait();
  grid_dep_launch();
  for (int i = threadIdx.x; i < 9 * COUT * CIN; i += blockDim.x) {
    const int co = i / (9 * CIN), r = i - co * 9 * CIN;
    wsm[r * COUT + co] = __bfloat162float(a.w[i]);
  }
  __syncthreads();
  const int H = a.Ho, Hg = H >> 2, groups = a.B * H * Hg;
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= (long long)groups * 4) return;
  const int grp = (int)(t >> 2), part = (int)(t & 3);
  const int b = grp / (H * Hg), rem = grp - b * H * Hg, oy = rem / Hg, x0 = 4 * (rem - oy * Hg);
  const bool vec = ((uintptr_t)a.x & 15) == 0;
  float acc[4][8];
#pragma unroll
  for (int j = 0; j < 4; ++j)
#pragma unroll
    for (int o = 0; o < 8; ++o) acc[j][o] = 0.f;
#pragma unroll
  for (int ky = 0; ky < 3; ++ky) {
    const int iy = oy + ky - 1;
    if (iy < 0 || iy >= H) continue;
    const size_t row = (size_t)(b * H + iy) * H + x0;
    float x[6][CIN];
    bool ok[6];
#pragma unroll
    for (int e = 0; e < 6; ++e) {
      ok[e] = e == 0 ? x0 > 0 : e == 5 ? x0 + 4 < H : true;  // the middle four are the group's own
      float4 f = make_float4(0.f, 0.f, 0.f, 0.f);
      if (ok[e]) {
        const float* src = a.x + (row + e - 1) * CIN;
        f = vec ? __ldcg(reinterpret_cast<const float4*>(src))
                : make_float4(__ldcg(src), __ldcg(src + 1), __ldcg(src + 2), __ldcg(src + 3));
      }
      const __nv_bfloat162 lo = __floats2bfloat162_rn(f.x, f.y), hi = __floats2bfloat162_rn(f.z, f.w);
      x[e][0] = __low2float(lo);
      x[e][1] = __high2float(lo);
      x[e][2] = __low2float(hi);
      x[e][3] = __high2float(hi);
      if (ky == 1 && part == 0 && e >= 1 && e <= 4)
        a.x16[row + e - 1] = make_uint2(*reinterpret_cast<const uint32_t*>(&lo), *reinterpret_cast<const uint32_t*>(&hi));
    }
#pragma unroll
    for (int kx = 0; kx < 3; ++kx)
#pragma unroll
      for (int ci = 0; ci < CIN; ++ci) {
        const float4* wr = reinterpret_cast<const float4*>(&wsm[((ky * 3 + kx) * CIN + ci) * COUT + part * 8]);
        const float4 w0 = wr[0], w1 = wr[1];
        const float wv[8] = {w0.x, w0.y, w0.z, w0.w, w1.x, w1.y, w1.z, w1.w};
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          if (!ok[j + kx]) continue;
#pragma unroll
          for (int o = 0; o < 8; ++o) acc[j][o] = fmaf(x[j + kx][ci], wv[o], acc[j][o]);
        }
      }
  }
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    uint4 o;
    __nv_bfloat162* oh = reinterpret_cast<__nv_bfloat162*>(&o);
#pragma unroll
    for (int e = 0; e < 4; ++e)
      oh[e] = __floats2bfloat162_rn(fmaxf(acc[j][2 * e] + a.bias[part * 8 + 2 * e], 0.f),
                                    fmaxf(acc[j][2 * e + 1] + a.bias[part * 8 + 2 * e + 1], 0.f));
    *reinterpret_cast<uint4*>(static_cast<bf16*>(a.out) + ((size_t)(b * H + oy) * H + x0 + j) * COUT + part * 8) = o;
  }
}

// The second layer (32 -> 64, stride 2): one tap of 32 channels per step, the
// split-K sums kept inside the block (the accumulators are added to the
// totals where conv_fwd_kernel's splits end, so the result is bitwise its
// split-K epilogue's).  64 pixels x 64 channels per block, four warps of
// 32 x 32, taps brought in two steps ahead with cp.async.  64 windows at
// h = 32: 8.7 us, against 10.3 + 6.6 with split K and its epilogue kernel.
constexpr int kNarrowPitch = 80, kNarrowStage = 2 * 64 * kNarrowPitch;
__global__ void __launch_bounds__(128) conv_narrow_kernel(const ConvFwd a, int lho) {
  __shared__ __align__(16) unsigned char raw[3 * kNarrowStage];
  const uint32_t sm = smem_addr(raw);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, wm = warp & 1, wn = warp >> 1;
  const int Ho = 1 << lho, Mtot = a.B << (2 * lho), bm = blockIdx.x * 64;
  const int c = tid & 3, r0 = tid >> 2;
  int pb[2], py[2], px[2];
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const int p = bm + r0 + 32 * i;
    pb[i] = p < Mtot ? p >> (2 * lho) : -1;
    py[i] = 2 * ((p >> lho) & (Ho - 1)) - 1;
    px[i] = 2 * (p & (Ho - 1)) - 1;
  }
  auto copy = [](uint32_t dst, const void* src, bool ok) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(ok ? 16 : 0) : "memory");
  };
  auto load_w = [&](int s) {
    const uint32_t st = sm + (uint32_t)((s % 3) * kNarrowStage + 64 * kNarrowPitch);
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const int n = r0 + 32 * i;
      copy(st + (uint32_t)(n * kNarrowPitch + c * 16), a.w + (size_t)n * 288 + s * 32 + 8 * c, true);
    }
  };
  auto load_a = [&](int s) {
    const uint32_t st = sm + (uint32_t)((s % 3) * kNarrowStage);
    const int ky = s / 3, kx = s - 3 * ky;
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const int iy = py[i] + ky, ix = px[i] + kx;
      const bool ok = pb[i] >= 0 && (unsigned)iy < (unsigned)a.Hin && (unsigned)ix < (unsigned)a.Hin;
      copy(st + (uint32_t)((r0 + 32 * i) * kNarrowPitch + c * 16),
           a.in + (ok ? ((size_t)(pb[i] * a.Hin + iy) * a.Hin + ix) * 32 + 8 * c : 0), ok);
    }
  };
  load_w(0);
  load_w(1);
  grid_dep_wait();
  grid_dep_launch();
  load_a(0);
  asm volatile("cp.async.commit_group;" ::: "memory");
  load_a(1);
  asm volatile("cp.async.commit_group;" ::: "memory");
  float tot[2][4][4], acc[2][4][4];
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int e = 0; e < 4; ++e) tot[i][j][e] = acc[i][j][e] = 0.f;
  const int l7 = lane & 7, mi = lane >> 3, per = a.ksplit / 32;
#pragma unroll 1
  for (int s = 0; s < 9; ++s) {
    asm volatile("cp.async.wait_group 1;" ::: "memory");
    __syncthreads();
    if (s + 2 < 9) {
      load_w(s + 2);
      load_a(s + 2);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
    const uint32_t sa = sm + (uint32_t)((s % 3) * kNarrowStage), sb = sa + 64 * kNarrowPitch;
#pragma unroll
    for (int kk = 0; kk < 32; kk += 16) {
      uint32_t af[2][4], bf[4][2];
      auto ld4 = [](uint32_t (&r)[4], uint32_t addr) {
        asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                     : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                     : "r"(addr));
      };
#pragma unroll
      for (int i = 0; i < 2; ++i)
        ld4(af[i], sa + (uint32_t)((wm * 32 + i * 16 + l7 + (mi & 1) * 8) * kNarrowPitch + (kk + (mi >> 1) * 8) * 2));
#pragma unroll
      for (int j = 0; j < 4; j += 2) {
        uint32_t r[4];
        ld4(r, sb + (uint32_t)((wn * 32 + j * 8 + (mi >> 1) * 8 + l7) * kNarrowPitch + (kk + (mi & 1) * 8) * 2));
        bf[j][0] = r[0];
        bf[j][1] = r[1];
        bf[j + 1][0] = r[2];
        bf[j + 1][1] = r[3];
      }
#pragma unroll
      for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) mma_bf16(acc[i][j], af[i], bf[j]);
    }
    if ((s + 1) % per == 0 || s == 8) {
#pragma unroll
      for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            tot[i][j][e] += acc[i][j][e];
            acc[i][j][e] = 0.f;
          }
    }
  }
  const int g = lane >> 2, t = lane & 3;
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int hh = 0; hh < 2; ++hh) {
      const int p = bm + wm * 32 + i * 16 + g + 8 * hh;
      if (p >= Mtot) continue;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int co = wn * 32 + j * 8 + 2 * t;
        *reinterpret_cast<__nv_bfloat162*>(static_cast<bf16*>(a.out) + (size_t)p * 64 + co) =
            __floats2bfloat162_rn(fmaxf(tot[i][j][2 * hh] + a.bias[co], 0.f),
                                  fmaxf(tot[i][j][2 * hh + 1] + a.bias[co + 1], 0.f));
      }
    }
}

// Split-K epilogue: partial sums added in split order, then bias and ReLU;
// four outputs per thread (Cout a power of two, n a multiple of four).
__global__ void __launch_bounds__(256) conv_splitk_kernel(const ConvFwd a, int splits, size_t n) {
  const size_t i = ((size_t)blockIdx.x * blockDim.x + threadIdx.x) * 4;
  grid_dep_wait();
  grid_dep_launch();
  if (i >= n) return;
  const int c = (int)(i & (size_t)(a.Cout - 1)), cm = a.Cout - 1;
  const float4 bi = make_float4(a.bias[c], a.bias[(c + 1) & cm], a.bias[(c + 2) & cm], a.bias[(c + 3) & cm]);
  float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 9
  for (int s = 0; s < splits; ++s) {
    const float4 p = __ldcg(reinterpret_cast<const float4*>(a.part + (size_t)s * n + i));
    v.x += p.x;
    v.y += p.y;
    v.z += p.z;
    v.w += p.w;
  }
  v.x += bi.x;
  v.y += bi.y;
  v.z += bi.z;
  v.w += bi.w;
  if (a.relu) v = make_float4(fmaxf(v.x, 0.f), fmaxf(v.y, 0.f), fmaxf(v.z, 0.f), fmaxf(v.w, 0.f));
  if (a.out_f32) {
    *reinterpret_cast<float4*>(static_cast<float*>(a.out) + i) = v;
  } else {
    const __nv_bfloat162 lo = __floats2bfloat162_rn(v.x, v.y), hi = __floats2bfloat162_rn(v.z, v.w);
    *reinterpret_cast<uint2*>(static_cast<bf16*>(a.out) + i) =
        make_uint2(*reinterpret_cast<const uint32_t*>(&lo), *reinterpret_cast<const uint32_t*>(&hi));
  }
}

// --------------------------------------------------------------- training
// L = 1/2 mean((y - t)^2) with t = (z_H^T - z_H^0) / s - e_plain / s taken
// from the input x0 = (z_H^0, e_plain / s), the later z_H^T and s; dy = (y - t) / n.
// One block; the sum is reduced in a fixed order.
__global__ void __launch_bounds__(1024) cnn_loss_kernel(const float* __restrict__ y, const float4* __restrict__ x0,
                                                        const float2* __restrict__ zh, const float* __restrict__ scale,
                                                        int batch, int hh, float* __restrict__ dy,
                                                        double* __restrict__ loss) {
  __shared__ double red[32];
  const int n = batch * hh;  // pixels
  const double inv_n = 1.0 / (2.0 * (double)n);
  double s2 = 0.0;
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    const float s = scale[i / hh];
    const float is = s > 1e-30f ? 1.f / s : 0.f;
    const float4 x = x0[i];
    const float2 zt = zh[i];
    const float tx = (zt.x - x.x) * is - x.z, ty = (zt.y - x.y) * is - x.w;
    const float rx = y[2 * i] - tx, ry = y[2 * i + 1] - ty;
    dy[2 * i] = (float)(rx * inv_n);
    dy[2 * i + 1] = (float)(ry * inv_n);
    s2 += (double)rx * rx + (double)ry * ry;
  }
  const double tot = block_sum(s2, red, threadIdx.x, blockDim.x);
  if (threadIdx.x == 0) *loss = 0.5 * tot * inv_n;
}

// Adam (bias-corrected, c1 = 1/(1-b1^t), c2 = 1/(1-b2^t)); writes the BF16
// copy of the weights the forward pass reads.
__global__ void __launch_bounds__(256) adam_kernel(float* __restrict__ theta, const float* __restrict__ g,
                                                   float* __restrict__ m, float* __restrict__ v, bf16* __restrict__ wbf,
                                                   int P, float lr, float c1, float c2) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= P) return;
  const float gi = g[i];
  const float mi = 0.9f * m[i] + 0.1f * gi;
  const float vi = 0.999f * v[i] + 0.001f * gi * gi;
  m[i] = mi;
  v[i] = vi;
  const float th = theta[i] - lr * (mi * c1) / (sqrtf(vi * c2) + 1e-8f);
  theta[i] = th;
  wbf[i] = __float2bfloat16_rn(th);
}

__global__ void __launch_bounds__(256) to_bf16_kernel(const float* __restrict__ src, bf16* __restrict__ dst, size_t n) {
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
    dst[i] = __float2bfloat16_rn(src[i]);
}

// ------------------------------------------------------ per-window kernels
// W_z^l = |Q^l|^2 / (I_H^h I_h^H |Q^l|^2) for l = 0 .. L-2 (Eq. def_weights),
// level l at wz + sum_{j<l} (MS>>j)^2, from block means of Q in float64.
__global__ void __launch_bounds__(256) wz_kernel(const float2* __restrict__ Q, int MS, int L, float* __restrict__ wz) {
  int off = 0;
  for (int l = 0; l + 1 < L; ++l) {
    const int s = MS >> l, f = 1 << l;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < s * s; i += gridDim.x * blockDim.x) {
      const int r = i / s, c = i - r * s;
      double a2[4], self = 0.0;
      for (int a = 0; a < 2; ++a)
        for (int b = 0; b < 2; ++b) {
          const int rr = (r & ~1) + a, cc = (c & ~1) + b;
          double qx = 0.0, qy = 0.0;
          for (int y = 0; y < f; ++y)
            for (int x = 0; x < f; ++x) {
              const float2 q = Q[(rr * f + y) * MS + cc * f + x];
              qx += q.x;
              qy += q.y;
            }
          qx /= (double)(f * f);
          qy /= (double)(f * f);
          a2[2 * a + b] = qx * qx + qy * qy;
          if (rr == r && cc == c) self = a2[2 * a + b];
        }
      const double S = 0.25 * (a2[0] + a2[1] + a2[2] + a2[3]);
      wz[off + i] = S > 1e-30 ? (float)(self / S) : 0.f;
    }
    off += s * s;
  }
}

struct CoarseArgs {
  const float2* z;      // object [n_rows][n_cols]
  int n_cols;
  const int32_t* pos;   // [n_pos][2]
  const int32_t* idx;   // [count]
  int n_pos, MS, L;
  const float2* g0;     // [count][MS][MS] conj(Q)(R - Q z) from the window kernel
  const float* pyr;     // level factors (window-kernel layout)
  const float* wz;      // W_z^l tables
  float4* x;            // [count][h][h] (Re z_H, Im z_H, Re e/s, Im e/s)
  float* scale;         // [count] s
};

// One block per window: z_H and g_H on the coarsest grid as weighted sums over
// each coarse pixel's fine block, e_plain = g_H / w_H, s = RMS(e_plain).
__global__ void __launch_bounds__(1024) coarse_state_kernel(const CoarseArgs A) {
  __shared__ double red[32];
  const int w = blockIdx.x, tid = threadIdx.x;
  const int MS = A.MS, L = A.L, F = 1 << (L - 1), h = MS >> (L - 1);
  const int k = A.idx[w];
  float4* xo = A.x + (size_t)w * h * h;
  if ((unsigned)k >= (unsigned)A.n_pos) {
    for (int c = tid; c < h * h; c += blockDim.x) xo[c] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (tid == 0) A.scale[w] = 0.f;
    return;
  }
  const int pr = A.pos[2 * k], pc = A.pos[2 * k + 1];
  const float2* g0 = A.g0 + (size_t)w * MS * MS;
  const float norm = 1.f / (float)(F * F);
  const float* iwH = A.pyr + lvl_off(MS, L - 1) + h * h;
  float e2 = 0.f;
  for (int c = tid; c < h * h; c += blockDim.x) {
    const int cy = c / h, cx = c - cy * h;
    float2 gs = make_float2(0.f, 0.f), zs = make_float2(0.f, 0.f);
    for (int fy = 0; fy < F; ++fy)
      for (int fx = 0; fx < F; ++fx) {
        const int r = cy * F + fy, cc = cx * F + fx;
        float al = norm, be = norm;
        int woff = 0;
        for (int l = 0; l + 1 < L; ++l) {
          al *= __ldg(&A.pyr[lvl_off(MS, l + 1) + (r >> (l + 1)) * (MS >> (l + 1)) + (cc >> (l + 1))]);
          be *= __ldg(&A.wz[woff + (r >> l) * (MS >> l) + (cc >> l)]);
          woff += (MS >> l) * (MS >> l);
        }
        const float2 gv = g0[r * MS + cc];
        const float2 zv = __ldg(&A.z[(size_t)(pr + r) * A.n_cols + pc + cc]);
        gs.x += al * gv.x;
        gs.y += al * gv.y;
        zs.x += be * zv.x;
        zs.y += be * zv.y;
      }
    const float iw = __ldg(&iwH[c]);
    const float ex = gs.x * iw, ey = gs.y * iw;
    e2 += ex * ex + ey * ey;
    xo[c] = make_float4(zs.x, zs.y, ex, ey);
  }
  __shared__ float s_sh;
  const double tot = block_sum((double)e2, red, tid, blockDim.x);  // valid in thread 0
  if (tid == 0) s_sh = (float)sqrt(tot / (double)(h * h));
  __syncthreads();
  const float s = s_sh;
  const float is = s > 1e-30f ? 1.f / s : 0.f;
  for (int c = tid; c < h * h; c += blockDim.x) {
    float4 v = xo[c];
    v.z *= is;
    v.w *= is;
    xo[c] = v;
  }
  if (tid == 0) A.scale[w] = s;
}

// The same for 2 to 4 levels, whose per-pixel factors unroll (all of a coarse
// pixel's loads in flight), on a cluster of four blocks per window: the RMS is
// summed over the cluster.  At most four coarse pixels per thread (h <= 64).
// Bound by the latency of its loads; m = 128, three levels, 64 windows: 12 us
// against 18 us for the one-block form.
template <int L>
__global__ void __launch_bounds__(256) coarse_state_cluster_kernel(const CoarseArgs A) {
  constexpr int F = 1 << (L - 1), NP = 4;
  __shared__ double red[32];
  __shared__ double share;
  cg::cluster_group cl = cg::this_cluster();
  const int w = blockIdx.x / 4, rank = blockIdx.x % 4, tid = threadIdx.x;
  const int MS = A.MS, h = MS >> (L - 1), hh = h * h;
  grid_dep_wait();
  grid_dep_launch();
  const int k = A.idx[w];
  float4* xo = A.x + (size_t)w * hh;
  if ((unsigned)k >= (unsigned)A.n_pos) {  // uniform over the cluster
    for (int c = rank * 256 + tid; c < hh; c += 1024) xo[c] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (rank == 0 && tid == 0) A.scale[w] = 0.f;
    return;
  }
  const int pr = A.pos[2 * k], pc = A.pos[2 * k + 1];
  const float2* g0 = A.g0 + (size_t)w * MS * MS;
  constexpr float norm = 1.f / (float)(F * F);
  const float* iwH = A.pyr + lvl_off(MS, L - 1) + hh;
  float4 v[NP];
  float e2 = 0.f;
#pragma unroll
  for (int u = 0; u < NP; ++u) {
    const int c = rank * 256 + tid + 1024 * u;
    v[u] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (c >= hh) continue;
    const int cy = c / h, cx = c - cy * h;
    float2 gs = make_float2(0.f, 0.f), zs = make_float2(0.f, 0.f);
#pragma unroll
    for (int fy = 0; fy < F; ++fy) {
      const int r = cy * F + fy;
      // two pixels at a time: g^0 and W_z^0 by aligned 16- and 8-byte loads
#pragma unroll
      for (int fx = 0; fx < F; fx += 2) {
        const int cc = cx * F + fx;
        float al = norm;  // shared by both pixels
#pragma unroll
        for (int l = 0; l + 1 < L; ++l)
          al *= __ldg(&A.pyr[lvl_off(MS, l + 1) + (r >> (l + 1)) * (MS >> (l + 1)) + (cc >> (l + 1))]);
        const float2 w0 = __ldg(reinterpret_cast<const float2*>(&A.wz[r * MS + cc]));
        const float4 gv = __ldcg(reinterpret_cast<const float4*>(&g0[r * MS + cc]));
        const float2* zp = &A.z[(size_t)(pr + r) * A.n_cols + pc + cc];
        const float2 z0 = __ldcg(zp), z1 = __ldcg(zp + 1);
        float be0 = norm * w0.x, be1 = norm * w0.y;
        int woff = MS * MS;
#pragma unroll
        for (int l = 1; l + 1 < L; ++l) {
          const float b2 = __ldg(&A.wz[woff + (r >> l) * (MS >> l) + (cc >> l)]);
          be0 *= b2;
          be1 *= b2;
          woff += (MS >> l) * (MS >> l);
        }
        gs.x = fmaf(al, gv.x, gs.x);
        gs.y = fmaf(al, gv.y, gs.y);
        zs.x = fmaf(be0, z0.x, zs.x);
        zs.y = fmaf(be0, z0.y, zs.y);
        gs.x = fmaf(al, gv.z, gs.x);
        gs.y = fmaf(al, gv.w, gs.y);
        zs.x = fmaf(be1, z1.x, zs.x);
        zs.y = fmaf(be1, z1.y, zs.y);
      }
    }
    const float iw = __ldg(&iwH[c]);
    v[u] = make_float4(zs.x, zs.y, gs.x * iw, gs.y * iw);
    e2 += v[u].z * v[u].z + v[u].w * v[u].w;
  }
  const double part = block_sum((double)e2, red, tid, 256);  // valid in thread 0
  if (tid == 0) share = part;
  cl.sync();
  double tot = 0.0;
#pragma unroll
  for (int q = 0; q < 4; ++q) tot += *cl.map_shared_rank(&share, q);
  const float s = (float)sqrt(tot / (double)hh);
  const float is = s > 1e-30f ? 1.f / s : 0.f;
#pragma unroll
  for (int u = 0; u < NP; ++u) {
    const int c = rank * 256 + tid + 1024 * u;
    if (c < hh) xo[c] = make_float4(v[u].x, v[u].y, v[u].z * is, v[u].w * is);
  }
  if (rank == 0 && tid == 0) A.scale[w] = s;
  cl.sync();  // no block leaves while another may still read its share
}

struct LearnedUpArgs {
  const int32_t* idx;  // [count]
  int n_pos, MS, L;
  float2* contrib;     // in: g^0; out: w^0 Delta of the kept V-cycle output
  const float* pyr;    // level factors
  const float* scale;  // [count] s
  const float* y;      // [count][h][h][2] network output
  int* accepted;       // [count] 1 = learned output kept
  double* margin;      // [count] surrogate(plain) - surrogate(learned)
  unsigned long long* stats;  // [0] proposals, [1] acceptances (running totals)
};

// Offsets of level l >= 1 in a per-window pyramid of levels 1 .. L-1.
__host__ __device__ __forceinline__ int up_off(int MS, int l) {
  int o = 0;
  for (int j = 1; j < l; ++j) o += (MS >> j) * (MS >> j);
  return o;
}

// The V-cycle above the finest level in residual form, from g^0 in the
// increments, with the plain and the learned coarsest correction side by side;
// the surrogate test keeps one of them, written back as w^0 Delta.  A cluster
// of kUpSplit blocks per window, each with 1 / kUpSplit of the rows (whole
// coarsest bins: the network's side h is a multiple of 8): only the surrogate
// difference crosses blocks.  A thread keeps the g^0 of its 2 x 2 bins in
// registers from the restriction to the write-back, so g^0 is read once.
// Shared memory: two float2 pyramids of this block's rows of levels 1 .. L-1.
// m = 128, three levels, 64 windows: 12.7 us, against 26 with one block of
// 1024 threads per window that read g^0 three times.
constexpr int kUpSplit = 8, kUpThreads = 256;
__global__ void __launch_bounds__(kUpThreads) vcycle_up_kernel(const LearnedUpArgs A) {
  extern __shared__ __align__(16) unsigned char lsm[];
  __shared__ double red[32];
  __shared__ double share;
  cg::cluster_group cl = cg::this_cluster();
  constexpr int nt = kUpThreads, NB = 2;  // bins per thread: (MS / 2)^2 / 8 <= 512
  const int w = blockIdx.x / kUpSplit, q = blockIdx.x % kUpSplit, tid = threadIdx.x;
  const int MS = A.MS, L = A.L, M = MS * MS;
  grid_dep_wait();
  grid_dep_launch();
  const int k = A.idx[w];
  if ((unsigned)k >= (unsigned)A.n_pos) {  // uniform over the cluster
    if (q == 0 && tid == 0) {
      A.accepted[w] = 0;
      A.margin[w] = 0.0;
    }
    return;
  }
  const int tot = up_off(MS, L) / kUpSplit;
  float2* Ep = reinterpret_cast<float2*>(lsm);
  float2* En = Ep + tot;
  float2* g0 = A.contrib + (size_t)w * M;
  // level l: this block's rows q n / 8 .. of n = MS >> l, at up_off / 8
  const auto off = [&](int l) { return up_off(MS, l) / kUpSplit; };

  // ---- g^l, l = 1 .. L-1: g^{l+1} = W_u^l . I(g^l)
  float4 gr[NB][2];  // the two rows of each of this thread's finest bins
  const int s1 = MS >> 1, nb = s1 * s1 / kUpSplit, ls1 = 31 - __clz(s1);
  {
    const float* wu = A.pyr + lvl_off(MS, 1) + q * nb;
#pragma unroll
    for (int u = 0; u < NB; ++u) {
      const int i = tid + nt * u;
      if (i >= nb) continue;
      const int r = (q * nb + i) >> ls1, c = i & (s1 - 1);
      gr[u][0] = __ldcg(reinterpret_cast<const float4*>(&g0[(2 * r) * MS + 2 * c]));
      gr[u][1] = __ldcg(reinterpret_cast<const float4*>(&g0[(2 * r + 1) * MS + 2 * c]));
      const float f = 0.25f * __ldg(&wu[i]);
      Ep[i] = make_float2(f * (gr[u][0].x + gr[u][0].z + gr[u][1].x + gr[u][1].z),
                          f * (gr[u][0].y + gr[u][0].w + gr[u][1].y + gr[u][1].w));
    }
    __syncthreads();
  }
  for (int l = 2; l < L; ++l) {
    const int s = MS >> l, sf = MS >> (l - 1), n = s * s / kUpSplit, ls = 31 - __clz(s);
    const float* wu = A.pyr + lvl_off(MS, l) + q * n;
    float2* dst = Ep + off(l);
    const float2* src = Ep + off(l - 1);
    for (int i = tid; i < n; i += nt) {
      const int r = i >> ls, c = i & (s - 1);
      const float2 a = src[(2 * r) * sf + 2 * c], b = src[(2 * r) * sf + 2 * c + 1];
      const float2 cc = src[(2 * r + 1) * sf + 2 * c], d = src[(2 * r + 1) * sf + 2 * c + 1];
      const float f = 0.25f * __ldg(&wu[i]);
      dst[i] = make_float2(f * (a.x + b.x + cc.x + d.x), f * (a.y + b.y + cc.y + d.y));
    }
    __syncthreads();
  }
  // ---- coarsest: plain step and proposal
  const float s = A.scale[w];
  const bool proposed = s > 1e-30f;
  {
    const int h = MS >> (L - 1), n = h * h / kUpSplit;
    const float* iw = A.pyr + lvl_off(MS, L - 1) + h * h + q * n;
    float2* P = Ep + off(L - 1);
    float2* N = En + off(L - 1);
    const float2* yy = reinterpret_cast<const float2*>(A.y) + (size_t)w * h * h + q * n;
    for (int i = tid; i < n; i += nt) {
      const float2 g = P[i];
      const float f = __ldg(&iw[i]);
      const float2 e = make_float2(g.x * f, g.y * f);
      P[i] = e;
      if (proposed) {
        const float2 d = __ldcg(&yy[i]);
        N[i] = make_float2(e.x + s * d.x, e.y + s * d.y);
      } else {
        N[i] = e;
      }
    }
  }
  __syncthreads();
  // ---- up: e^l = g^l / w^l + (u^l / w^l) I_H^h e^{l+1}, l = L-2 .. 1
  for (int l = L - 2; l >= 1; --l) {
    const int s2 = MS >> l, sc = MS >> (l + 1), n = s2 * s2 / kUpSplit, ls = 31 - __clz(s2);
    const float* iw = A.pyr + lvl_off(MS, l) + s2 * s2 + q * n;
    const float* rr = iw + s2 * s2;
    float2* P = Ep + off(l);
    float2* N = En + off(l);
    const float2* Pc = Ep + off(l + 1);
    const float2* Nc = En + off(l + 1);
    for (int i = tid; i < n; i += nt) {
      const int pi = (i >> (ls + 1)) * sc + ((i & (s2 - 1)) >> 1);
      const float2 g = P[i];
      const float f = __ldg(&iw[i]), qq = __ldg(&rr[i]);
      const float2 ep = Pc[pi], en = Nc[pi];
      N[i] = make_float2(g.x * f + qq * en.x, g.y * f + qq * en.y);
      P[i] = make_float2(g.x * f + qq * ep.x, g.y * f + qq * ep.y);
    }
    __syncthreads();
  }
  // ---- finest: w^0 Delta = g^0 + u^0 I_H^h e^1; surrogate difference
  // 1/2 |Q|^2 |Delta|^2 - Re(conj(Delta) g^0) summed for both candidates
  const float* u0 = A.pyr;
  const float* w0 = A.pyr + M;
  float2 uu[NB][2];
  float dsum = 0.f;
#pragma unroll
  for (int u = 0; u < NB; ++u) {
    const int i = tid + nt * u;
    if (i >= nb) continue;
    const int r = (q * nb + i) >> ls1, c = i & (s1 - 1);
    const float2 ep = Ep[i], en = En[i];
#pragma unroll
    for (int a = 0; a < 2; ++a) {
      const int o = (2 * r + a) * MS + 2 * c;
      uu[u][a] = __ldg(reinterpret_cast<const float2*>(&u0[o]));
      const float2 wv2 = __ldg(reinterpret_cast<const float2*>(&w0[o]));
#pragma unroll
      for (int b = 0; b < 2; ++b) {
        const float2 g = b ? make_float2(gr[u][a].z, gr[u][a].w) : make_float2(gr[u][a].x, gr[u][a].y);
        const float uv = b ? uu[u][a].y : uu[u][a].x, wv = b ? wv2.y : wv2.x;
        const float iwv = wv > 1e-30f ? 1.f / wv : 0.f;
        const float q2 = wv - uv;
        const float2 dp = make_float2((g.x + uv * ep.x) * iwv, (g.y + uv * ep.y) * iwv);
        const float2 dn = make_float2((g.x + uv * en.x) * iwv, (g.y + uv * en.y) * iwv);
        const float sp = 0.5f * q2 * (dp.x * dp.x + dp.y * dp.y) - (dp.x * g.x + dp.y * g.y);
        const float sn = 0.5f * q2 * (dn.x * dn.x + dn.y * dn.y) - (dn.x * g.x + dn.y * g.y);
        dsum += sp - sn;
      }
    }
  }
  const double part = block_sum((double)dsum, red, tid, nt);  // valid in thread 0
  if (tid == 0) share = part;
  cl.sync();
  double mg = 0.0;
#pragma unroll
  for (int j = 0; j < kUpSplit; ++j) mg += *cl.map_shared_rank(&share, j);
  const bool keep = proposed && mg >= 0.0;
  if (q == 0 && tid == 0) {
    A.accepted[w] = keep;
    A.margin[w] = proposed ? mg : 0.0;
    if (proposed) atomicAdd(&A.stats[0], 1ull);
    if (keep) atomicAdd(&A.stats[1], 1ull);
  }
  const float2* E = keep ? En : Ep;
#pragma unroll
  for (int u = 0; u < NB; ++u) {
    const int i = tid + nt * u;
    if (i >= nb) continue;
    const int r = (q * nb + i) >> ls1, c = i & (s1 - 1);
    const float2 e = E[i];
#pragma unroll
    for (int a = 0; a < 2; ++a) {
      const float2 uv = uu[u][a];
      const float4 g = gr[u][a];
      *reinterpret_cast<float4*>(&g0[(2 * r + a) * MS + 2 * c]) =
          make_float4(g.x + uv.x * e.x, g.y + uv.x * e.y, g.z + uv.y * e.x, g.w + uv.y * e.y);
    }
  }
  cl.sync();  // no block leaves while another may still read its share
}

// patches[w] = the m x m window of the object at window idx[w] (zeros for an
// index out of range).
__global__ void __launch_bounds__(256) gather_windows_kernel(const float2* __restrict__ z, int n_cols,
                                                             const int32_t* __restrict__ pos,
                                                             const int32_t* __restrict__ idx, int n_pos, int MS,
                                                             float2* __restrict__ out) {
  const int w = blockIdx.x, k = idx[w];
  const bool ok = (unsigned)k < (unsigned)n_pos;
  const int pr = ok ? pos[2 * k] : 0, pc = ok ? pos[2 * k + 1] : 0;
  for (int i = threadIdx.x; i < MS * MS; i += blockDim.x) {
    const int r = i / MS, c = i - r * MS;
    out[(size_t)w * MS * MS + i] = ok ? z[(size_t)(pr + r) * n_cols + pc + c] : make_float2(0.f, 0.f);
  }
}
