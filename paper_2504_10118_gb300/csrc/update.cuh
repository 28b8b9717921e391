// update.cuh -- the ordered object update of a minibatch step (the tiled
// reduction of the windows' increments), shared by the update kernels and the
// persistent step kernel.  Included by core.cuh inside namespace magpie_impl.
#pragma once

// z += sum_b contrib_b / sum_b w0 over the windows covering each pixel, in
// minibatch order (bitwise reproducible).  One block of NT (256) threads per
// TW x TH object tile, TW TH / NT pixels of one column per thread: the block
// first lists, in minibatch order, the windows that overlap its tile (corners
// as recorded by the window kernel; a ballot compaction over all warps), each
// with its increments' offset; each thread then walks that list a few entries
// at a time with predicated loads, so several increments are in flight per
// thread.  Tile number tiles_x tiles_y turns the window phase's block partials
// into Phi_k and ||grad Phi_k||, in a block of its own beside the tiles.
// Dynamic smem: count entries.  Every tile shape sums each
// pixel's windows in minibatch order, so all give bitwise equal objects.
struct ApplyShape {
  int tw, th;
};
constexpr ApplyShape kApplyShapes[3] = {{16, 16}, {32, 8}, {32, 32}};
struct ApplyArgs {
  float2* z;               // object [n_rows][n_cols]
  int n_rows, n_cols;
  const int2* corners;     // [count] window corners from the window kernel
  const int32_t* idx;      // [count] window indices
  int count, n_pos;
  const float2* contrib;   // [count][MS][MS] increments w . Delta
  const float* w0;         // [MS][MS] u + |Q|^2
  int MS;
  const double* part;      // [count][slots][2] partial sums of the window phase
  int slots;               // partial-sum slots per window
  double* phi_pos;         // per-window Phi_k
  double* gn_pos;          // per-window ||grad Phi_k||
  int tiles_x, tiles_y;    // tiles per object row and column
  int block0;              // batched launches: first block of this problem
  // The precision form's V-cycle tail (apply_body<..., true>): contrib holds
  // g^0, and each window's w . Delta = g^0 + u^0 I_H^h e^1 is formed here as
  // it is summed (the finest prolongation of Algorithm MAGPS, residual form).
  const float2* e1;        // [count][MS/2][MS/2] e^1
  const float* u0;         // [MS][MS] u^0
  int* hand;               // precision form: the step's window hand-off counts, zeroed by
  int nhand;               // block 0 once the grid may run (null otherwise)
  int early;               // the object and the windows' positions are final before the stream's previous
                           // kernel ends: the windows are listed before the wait for it, their corners
                           // as an earlier kernel recorded them (1) or from idx and pos (2)
  const int32_t* pos;      // [n_pos][2] (early = 2)
};

// One window of a tile's list: its corner, the offset of its increments less
// that of its corner (so that pixel (r, c) is at off + r MS + c), its slot.
struct ApplyEntry {
  int qx, qy, off, b;
};

// Phi_k and ||grad Phi_k|| of the step's windows from the block partials, in block order.
__device__ __forceinline__ void apply_partials(const ApplyArgs& P) {
  const double scale = 0.5 / ((double)P.MS * (double)P.MS);  // a power of two
  for (int b = threadIdx.x; b < P.count; b += blockDim.x) {
    const int k = P.idx[b];
    if ((unsigned)k >= (unsigned)P.n_pos) continue;
    double a = 0.0, g = 0.0;
    for (int q = 0; q < P.slots; ++q) {
      a += P.part[(size_t)(b * P.slots + q) * 2];
      g += P.part[(size_t)(b * P.slots + q) * 2 + 1];
    }
    P.phi_pos[k] = a * scale;
    P.gn_pos[k] = sqrt(g);
  }
}

template <int TW, int TH, int NT = 256, bool TAIL = false, bool LEAVE = true>
__device__ __forceinline__ void apply_body(const ApplyArgs& P, const int tx, const int ty) {
  static_assert((TW * TH) % NT == 0 && NT % TW == 0 && NT % 32 == 0, "NT threads cover the tile in whole rows");
  constexpr int PPT = TW * TH / NT, RS = NT / TW, NW = NT / 32;  // pixels per thread, rows per pass, warps
  constexpr int U = PPT >= 4 ? 2 : kApplyUnroll;                  // list entries in flight
  extern __shared__ __align__(16) unsigned char apply_smem[];
  ApplyEntry* list = reinterpret_cast<ApplyEntry*>(apply_smem);
  __shared__ int warp_hits[NW];
  if (!P.early) grid_dep_wait();
  if (ty >= P.tiles_y) {  // the partial sums' block
    if (P.early) {
      grid_dep_wait();
      grid_dep_launch();
    }
    apply_partials(P);
    return;
  }
  const int count = P.count, MS = P.MS, M = MS * MS;
  const int R0 = ty * TH, C0 = tx * TW;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int r0 = R0 + (int)(threadIdx.x / TW), c = C0 + (int)(threadIdx.x % TW);
  // windows meeting this tile, listed in minibatch order: every warp takes
  // 32 consecutive windows per round, ballots, and the rounds are stitched
  // together by per-warp counts
  int nl = 0;
  for (int b0 = 0; b0 < count; b0 += NT) {
    const int b = b0 + threadIdx.x;
    bool hit = false;
    int2 q = make_int2(0, 0);
    if (b < count) {
      if (P.early == 2) {
        const int k = P.idx[b];
        q = (unsigned)k < (unsigned)P.n_pos ? make_int2(P.pos[2 * k], P.pos[2 * k + 1])
                                            : make_int2(-(1 << 30), -(1 << 30));
      } else {
        q = __ldcg(&P.corners[b]);
      }
      hit = q.x < R0 + TH && q.x + MS > R0 && q.y < C0 + TW && q.y + MS > C0;
    }
    const unsigned mask = __ballot_sync(0xffffffffu, hit);
    if (lane == 0) warp_hits[wid] = __popc(mask);
    __syncthreads();
    int off = nl;
#pragma unroll
    for (int i = 0; i < NW; ++i) {
      if (i < wid) off += warp_hits[i];
      nl += warp_hits[i];
    }
    if (hit) list[off + __popc(mask & ((1u << lane) - 1u))] = ApplyEntry{q.x, q.y, b * M - q.x * MS - q.y, b};
    __syncthreads();
  }
  // A tile that no window meets is left alone: nothing of the object outside
  // the windows is read.  Its block leaves at once (LEAVE; 2.215 ms per large
  // sweep, 2.275 if it first waits; a step of 8 windows at n = 700 9.2 / 10.4
  // us, at n = 4096 28.7 us against 45.7 with every tile read) or after the wait.
  // The block of the partial sums waits in any case, so the grid does not end
  // before the kernel it follows.
  float2 zz[PPT];
  const auto load_z = [&]() {  // on their way while the windows' increments are computed
#pragma unroll
    for (int p = 0; p < PPT; ++p)
      zz[p] = (r0 + p * RS < P.n_rows && c < P.n_cols) ? __ldcg(&P.z[(size_t)(r0 + p * RS) * P.n_cols + c])
                                                        : make_float2(0.f, 0.f);
  };
  if constexpr (LEAVE) {
    if (nl == 0) return;
    load_z();
  } else {
    if (nl > 0) load_z();
  }
  if (P.early) {
    grid_dep_wait();
    grid_dep_launch();
  }
  if constexpr (!LEAVE) {
    if (nl == 0) return;
  }
  float nx[PPT], ny[PPT], d[PPT];
#pragma unroll
  for (int p = 0; p < PPT; ++p) nx[p] = ny[p] = d[p] = 0.f;
  const int o0 = r0 * MS + c;
#pragma unroll 1
  for (int j0 = 0; j0 < nl; j0 += U) {
    float2 v[U][PPT];
    float wv[U][PPT];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const bool live = j0 + u < nl;
      const ApplyEntry q = list[live ? j0 + u : 0];
      const bool inc = live && (unsigned)(c - q.qy) < (unsigned)MS;
      const int qo = q.qx * MS + q.qy;
#pragma unroll
      for (int p = 0; p < PPT; ++p) {
        const int dr = r0 + p * RS - q.qx;
        const bool in = inc && (unsigned)dr < (unsigned)MS;
        const int o = o0 + p * RS * MS;
        v[u][p] = in ? __ldcg(&P.contrib[q.off + o]) : make_float2(0.f, 0.f);
        wv[u][p] = in ? __ldg(&P.w0[o - qo]) : 0.f;
        if constexpr (TAIL) {
          // w . Delta = g^0 + u^0 e^1 at this window pixel, e^1 of its 2 x 2 bin
          const int h = MS >> 1, dc = c - q.qy;
          const float2 e = in ? P.e1[q.b * h * h + (dr >> 1) * h + (dc >> 1)] : make_float2(0.f, 0.f);
          const float uo = in ? __ldg(&P.u0[o - qo]) : 0.f;
          v[u][p] = make_float2(__fmaf_rn(uo, e.x, v[u][p].x), __fmaf_rn(uo, e.y, v[u][p].y));
        }
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u)
#pragma unroll
      for (int p = 0; p < PPT; ++p) {
        nx[p] += v[u][p].x;
        ny[p] += v[u][p].y;
        d[p] += wv[u][p];
      }
  }
#pragma unroll
  for (int p = 0; p < PPT; ++p)
    if (d[p] > 0.f)  // only pixels of the object have windows
      P.z[(size_t)(r0 + p * RS) * P.n_cols + c] = make_float2(zz[p].x + nx[p] / d[p], zz[p].y + ny[p] / d[p]);
}
