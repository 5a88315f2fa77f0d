// olb_strip.cuh -- several D2Q9 pull steps per launch, the state between them in
// registers (FP32 arithmetic: FP32, FP16 and BF16 storage; every cell fluid, both axes
// periodic, nx even).
//
// A 2D step moves 72 bytes a cell (FP32) through L2 or, from about 1400^2, HBM, and a
// small one waits for its launch.  Here a block loads a tile of 64 x 32 cells once,
// advances it by up to `halo` steps and stores the cells that are still valid: one ring
// of cells is lost per step.  Every step collides the whole tile: 2048 cells for the 1344
// that are stored at halo 4 (1.5 times the arithmetic), for 768 at halo 8 (2.7 times).
// That pays against the traffic of a large lattice and the launches of a small one:
// 2048^2 FP32 45.9 -> 28.9 us a step, 64^2 2.07 -> 1.59.
// (The same with walls needs their links in every step: 1024^2 cavity 10.9 -> 13.8 us,
// 511 x 213 with an obstacle 3.1 -> 4.4; those lattices step one by one.)
//
// A warp holds 4 rows of 64 cells, two cells per lane: populations move along x by one
// shuffle per pair of values and along y by renaming registers; only the outer rows of
// each warp go through shared memory (3 populations each way), double-buffered, with
// one barrier per step.  Values are rounded to the storage type after every step and
// the arithmetic is that of the one-step kernel (collide_pair), so the result is the
// same bit for bit as that of single steps.
#pragma once

namespace olb {

struct StripGeom {
  int halo;   // cells around the stored part of a tile (even, >= steps)
  int steps;  // steps of this launch
};

constexpr int kStripX = 64, kStripRows = 4, kStripWarps = 8, kStripY = kStripRows * kStripWarps;

template <class S, bool TRT>
__global__ void __launch_bounds__(32 * kStripWarps, 2)
    k_strip(Params<float> p, const S* src, S* dst, StripGeom g) {
  using L = D2Q9;
  using H = Held<S>;
  constexpr int R = kStripRows;
  __shared__ float2 edge[2][2][3][kStripWarps][32];  // [step parity][0 up, 1 down][population][warp][lane]
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int halo = g.halo;
  const int xe = blockIdx.x * (kStripX - 2 * halo) - halo + 2 * lane;  // before wrapping
  const int ye = blockIdx.y * (kStripY - 2 * halo) - halo + warp * R;
  auto wrap = [](int v, int n) {
    v %= n;
    return v < 0 ? v + n : v;
  };
  const int x0 = wrap(xe, p.nx);
  int ys[R];
#pragma unroll
  for (int r = 0; r < R; ++r) ys[r] = wrap(ye + r, p.ny);
  pdl_wait_then_release();
  F2 f[R][L::Q];
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const PairNbr n = make_pair_nbr<L>(p, x0, ys[r], 0);
#pragma unroll
    for (int i = 0; i < L::Q; ++i)
      f[r][i] = ld_pair(src + (size_t)i * p.pitch, n, -L::c(i, 0), -L::c(i, 1), 0);
  }
  for (int k = 0; k < g.steps; ++k) {
#pragma unroll
    for (int r = 0; r < R; ++r) {
      F2 gamma(1.0f), rho, drho, j[3], u[3];
      if (p.gamma) gamma = F2(*reinterpret_cast<const float2*>(p.gamma + ys[r] * p.nx + x0));
      collide_pair<L, (int)PairStore<S>::SCALE, TRT>(p, gamma, f[r], drho, j, rho, u);
      if (sizeof(S) == 2) {
#pragma unroll
        for (int i = 0; i < L::Q; ++i) f[r][i] = H::get(H::put(f[r][i]));  // as it reads back from storage
      }
    }
    if (k + 1 == g.steps) break;
    int up = 0, down = 0;
#pragma unroll
    for (int i = 0; i < L::Q; ++i) {
      if (L::c(i, 1) == 1) edge[k & 1][0][up++][warp][lane] = f[R - 1][i].v;
      if (L::c(i, 1) == -1) edge[k & 1][1][down++][warp][lane] = f[0][i].v;
    }
    __syncthreads();
    // (the outermost rows take their own: those cells are no longer valid)
    const int below = warp == 0 ? 0 : warp - 1, above = warp == kStripWarps - 1 ? warp : warp + 1;
#pragma unroll
    for (int i = 1; i < L::Q; ++i) {
      const int cx = L::c(i, 0), cy = L::c(i, 1);
      int slot = 0;  // rank of i among the populations with its c_y
#pragma unroll
      for (int m = 0; m < i; ++m) slot += L::c(m, 1) == cy;
      if (cy == 1) {
#pragma unroll
        for (int r = R - 1; r > 0; --r) f[r][i] = f[r - 1][i];
        f[0][i] = F2(edge[k & 1][0][slot][below][lane]);
      } else if (cy == -1) {
#pragma unroll
        for (int r = 0; r < R - 1; ++r) f[r][i] = f[r + 1][i];
        f[R - 1][i] = F2(edge[k & 1][1][slot][above][lane]);
      }
      if (cx != 0) {
#pragma unroll
        for (int r = 0; r < R; ++r) {
          const F2 v = f[r][i];
          f[r][i] = cx == 1 ? F2(__shfl_up_sync(0xffffffffu, v.v.y, 1), v.v.x)
                            : F2(v.v.y, __shfl_down_sync(0xffffffffu, v.v.x, 1));
        }
      }
    }
  }
  // the valid part of the tile
  const int tx = 2 * lane;
  if (tx < halo || tx >= kStripX - halo || xe >= p.nx) return;
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int ty = warp * R + r;
    if (ty < halo || ty >= kStripY - halo || ye + r >= p.ny) continue;
#pragma unroll
    for (int i = 0; i < L::Q; ++i)
      PairStore<S>::st2(dst + (size_t)i * p.pitch + ys[r] * p.nx + x0, f[r][i]);
  }
}

}  // namespace olb
