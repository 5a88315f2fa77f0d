// olb_march.cuh -- two collide-and-stream steps of the D3Q19 pull pattern in one pass
// over memory (FP32 arithmetic: FP32, FP16 and BF16 storage).
//
// A step by itself reads and writes every population once and is bound by that
// traffic.  Here the state between the two steps never leaves the SM: a block owns a
// tile of 64 cells along x by ROWS - 2 rows along y and marches along z.  At plane t
//   stage A  collides plane t of the tile and of the ring of cells around it
//            (step 1, populations gathered from the source buffer) and keeps the
//            post-collision values on the SM;
//   stage B  gathers plane t - 1 of the tile from them, collides it (step 2) and
//            stores it to the destination buffer as the one-step kernel does.
// Both stages run the one-step kernel's own arithmetic (collide_pair, pair_update) on
// values rounded to the storage type in between, so the result is the same, bit for
// bit, as that of two single steps.
//
// Layout.  One warp per row of the extended tile (64 cells, two per lane); the two
// outer rows run stage A only, and collide the cells left (the first) and right (the
// last) of the tile for the next plane while the others run stage B (lane r holds the
// cell beside row r).  Of the 19 populations, the 10 that move along y go
// through a shared-memory ring of planes; the others stay in the registers of the
// thread that holds the column and move along x by shuffles.
// The ring keeps 4 planes of the populations with c_z = 1 (stage B reads planes t - 2
// and t - 1 of them while t + 1 may already be written by a warp that is ahead) and 3
// of the others (t - 1, t, t + 1), so one barrier per plane is enough.
//
// Walls.  Stage A reads bounce-back values where the one-step kernel left them (in the
// wall cells' slots).  Between the stages a cell's own slot i holds what returns to it
// when its link i ends at a wall (nobody else reads that slot then; on a moving wall
// the wall term is taken off before the value is rounded and stored), so stage B takes
// population i from the cell's own slot opp(i) when x - c_i is not a fluid cell.
#pragma once

namespace olb {

// c_z + 1 of the D3Q19 populations, for an index known at run time
__device__ constexpr unsigned char kMarchCz[19] = {1, 1, 1, 0, 1, 1, 0, 2, 0, 2, 1, 1, 2, 1, 1, 2, 0, 2, 0};

// p + n * i elements of 1 byte (n, i unsigned): one instruction
__device__ __forceinline__ uint64_t wide_add(uint64_t p, unsigned n, unsigned i) {
  uint64_t r;
  asm("mad.wide.u32 %0, %1, %2, %3;" : "=l"(r) : "r"(n), "r"(i), "l"(p));
  return r;
}
// The global-memory pointer at address q (stated, or the compiler would issue generic
// loads and stores).
template <class T>
__device__ __forceinline__ T* global_ptr(uint64_t q) {
  return static_cast<T*>(__cvta_global_to_generic(q));
}
__device__ __forceinline__ uint64_t wide_add_s(uint64_t p, int n, int i) {
  uint64_t r;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(n), "r"(i), "l"(p));
  return r;
}

// Source and destination buffers, and the bytes between two population planes (below
// 2^32): the address of a population is one wide multiply-add from a row's address.
template <class S>
struct MarchBuf {
  const S* src;
  S* dst;
  unsigned pitch;
};

struct MarchGeom {
  int cz;  // planes per block along z
};

template <class S>
struct March {
  using L = D3Q19;
  static constexpr int TX = 64;           // cells along x
  static constexpr int ROWS = 16;         // rows of stage A; ROWS - 2 rows are stored
  static constexpr int TY = ROWS - 2;
  static constexpr int THREADS = 32 * ROWS;
  static constexpr int RL = TX + 4;       // ring row: cells x - 2 .. x + 65 of the tile (pairs stay aligned)
  static constexpr int PT = ROWS * RL;    // values of one plane of one population
  __host__ __device__ static constexpr bool in_ring(int i) { return L::c(i, 1) != 0; }
  __host__ __device__ static constexpr bool on_side(int i) { return L::c(i, 1) == 0 && L::c(i, 0) != 0; }
  __host__ __device__ static constexpr int planes(int i) { return L::c(i, 2) == 1 ? 4 : 3; }
  // first plane of population i in the ring, and in the side columns
  __host__ __device__ static constexpr int first(int i) {
    int n = 0;
    for (int k = 0; k < i; ++k)
      if (in_ring(k)) n += planes(k);
    return n;
  }
  __host__ __device__ static constexpr int side(int i) {
    int n = 0;
    for (int k = 0; k < i; ++k)
      if (on_side(k)) n += planes(k);
    return n;
  }
  static constexpr size_t smem() { return ((size_t)first(L::Q) * PT + (size_t)side(L::Q) * ROWS) * sizeof(S); }
};

// A pair of stored values held in registers in the storage type.
template <class S>
struct Held {
  using T = F2;
  __device__ static T put(F2 v) { return v; }
  __device__ static F2 get(T v) { return v; }
};
template <>
struct Held<__half> {
  using T = __half2;
  __device__ static T put(F2 v) { return __float22half2_rn(v.v); }
  __device__ static F2 get(T v) { return F2(__half22float2(v)); }
};
template <>
struct Held<__nv_bfloat16> {
  using T = __nv_bfloat162;
  __device__ static T put(F2 v) { return __float22bfloat162_rn(v.v); }
  __device__ static F2 get(T v) { return F2(__bfloat1622float2(v)); }
};

// Link bits of the directions with c_a == s.
template <class L>
__host__ __device__ constexpr uint32_t face_mask(int a, int s) {
  uint32_t m = 0;
  for (int i = 1; i < L::Q; ++i)
    if (L::c(i, a) == s) m |= 1u << i;
  return m;
}

// An index that is a constant of its type, and fn(Idx<0>) ... fn(Idx<N - 1>): links are
// walked with constant indices, so that f[] stays in registers.
template <int I>
struct Idx {
  __host__ __device__ constexpr operator int() const { return I; }
};
template <class F, int... I>
__device__ __forceinline__ void static_for_impl(F&& fn, std::integer_sequence<int, I...>) {
  (fn(Idx<I>{}), ...);
}
template <int N, class F>
__device__ __forceinline__ void static_for(F&& fn) {
  static_for_impl(fn, std::make_integer_sequence<int, N>{});
}

// Calls fn(i) at least for every direction in `any` (the links of all lanes).  Every
// warp of a block waits for the slowest at each plane, so the directions that no lane
// needs are skipped by warp-wide tests: a wall across an axis brings the five links
// of that face, which one bit tells; links outside such faces (edges of obstacles)
// are tested one by one.
template <class L, class F>
__device__ __forceinline__ void for_links(uint32_t any, F&& fn) {
  uint32_t rest = any;
  static_for<6>([&](auto face) {
    constexpr int a = face / 2, s = (face & 1) ? 1 : -1;
    constexpr uint32_t five = face_mask<L>(a, s);
    // the link along the axis: the one that no other face holds
    constexpr uint32_t axis = five & ~(face_mask<L>((a + 1) % 3, 1) | face_mask<L>((a + 1) % 3, -1) |
                                       face_mask<L>((a + 2) % 3, 1) | face_mask<L>((a + 2) % 3, -1));
    if (any & axis) {
      static_for<L::Q>([&](auto i) {
        if constexpr ((five >> i) & 1u) fn(i);
      });
      rest &= ~five;
    }
  });
  if (rest) {
    static_for<L::Q>([&](auto i) {
      if constexpr (i > 0) {
        if (rest & (1u << i)) fn(i);
      }
    });
  }
}

// Takes the wall term off the post-collision populations whose links end at a moving
// wall (their own slots then hold what the bounce-back returns; no other cell reads
// them).  mv0, mv1: links of the pair's fluid cells that have moving ones.
__device__ __forceinline__ void moving_walls(const Params<float>& p, int x0, int y, int z, uint32_t mv0, uint32_t mv1,
                                             const uint32_t (&w)[2], F2 (&f)[19], F2 rho) {
  using L = D3Q19;
  const unsigned all = 0xffffffffu;
  const unsigned who = __ballot_sync(all, (mv0 | mv1) != 0);
  if (!who) return;
  const uint32_t form0 = (w[0] >> kWordPlaneShift) & 0x7ffu, form1 = (w[1] >> kWordPlaneShift) & 0x7ffu;
  const uint32_t form = __shfl_sync(all, mv0 ? form0 : form1, __ffs(who) - 1);
  if ((form & 7u) && __all_sync(all, (!mv0 || form0 == form) && (!mv1 || form1 == form))) {
    // one wall plane for the whole warp (a row along a flat lid): one table load per direction
    const float* tab = p.wall_f + 20 * (form >> (kWordMatShift - kWordPlaneShift));
    const int face = (int)(form & 7u) - 1;
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
      for (int s = 0; s < 2; ++s) {
        if (face == 2 * a + s) {
#pragma unroll
          for (int i = 1; i < L::Q; ++i)
            if (L::c(i, a) == 2 * s - 1) {
              const float t = tab[i];
              if (mv0 & (1u << i)) f[i].v.x -= rho.v.x * t;
              if (mv1 & (1u << i)) f[i].v.y -= rho.v.y * t;
            }
        }
      }
    return;
  }
#pragma unroll
  for (int i = 1; i < L::Q; ++i) {
    float t;
    if ((mv0 & (1u << i)) &&
        moving_term<L>(p, wrapped_cell<L>(p, x0, y, z, L::c(i, 0), L::c(i, 1), L::c(i, 2)), i, w[0], t))
      f[i].v.x -= rho.v.x * t;
    if ((mv1 & (1u << i)) &&
        moving_term<L>(p, wrapped_cell<L>(p, x0 + 1, y, z, L::c(i, 0), L::c(i, 1), L::c(i, 2)), i, w[1], t))
      f[i].v.y -= rho.v.y * t;
  }
}

// Stage B's stores: own slots, and bounce-back values into the wall cells' slots (the
// rules of pair_update).
template <class S, bool WALLS>
__device__ __forceinline__ void march_store(const Params<float>& p, const MarchBuf<S>& pl, bool act, int x0,
                                            int y, int z, int cell, const uint32_t (&w)[2], F2 (&f)[19], F2 rho) {
  using L = D3Q19;
  const uint64_t q0 = wide_add_s(__cvta_generic_to_global(pl.dst), cell, (int)sizeof(S));
  auto at = [&](int i) { return global_ptr<S>(wide_add(q0, pl.pitch, (unsigned)i)); };
  if (!WALLS) {
    if (act) {
#pragma unroll
      for (int i = 0; i < L::Q; ++i) PairStore<S>::st2(at(i), f[i]);
    }
    return;
  }
  const bool fl0 = act && (w[0] & kWordFluid), fl1 = act && (w[1] & kWordFluid);
  const uint32_t nb0 = w[0] & kWordLinks, nb1 = w[1] & kWordLinks;
  const uint32_t l0 = fl0 ? nb0 : 0u, l1 = fl1 ? nb1 : 0u;
  const uint32_t any = __reduce_or_sync(0xffffffffu, l0 | l1);
  if (any) {
    if (p.moving) moving_walls(p, x0, y, z, (w[0] & kWordMoving) ? l0 : 0u, (w[1] & kWordMoving) ? l1 : 0u, w, f, rho);
    // a link crosses a lattice face only along a periodic axis; elsewhere its target is
    // at a fixed offset
    const bool inner = (!(p.periodic & 1u) || (x0 > 0 && x0 + 2 < p.nx)) &&
                       (!(p.periodic & 2u) || (y > 0 && y + 1 < p.ny)) &&
                       (!(p.periodic & 4u) || (z > 0 && z + 1 < p.nz));
    if (__all_sync(0xffffffffu, inner || !(l0 | l1))) {
      for_links<L>(any, [&](auto i) {
        S* q = at(opp<L>(i)) + (L::c(i, 0) + p.nx * (L::c(i, 1) + p.ny * L::c(i, 2)));
        if (l0 & (1u << i)) PairStore<S>::st1(q, f[i].v.x);
        if (l1 & (1u << i)) PairStore<S>::st1(q + 1, f[i].v.y);
      });
    } else {
#pragma unroll
      for (int i = 1; i < L::Q; ++i) {
        if (l0 & (1u << i))
          PairStore<S>::st1(at(opp<L>(i)) + (wrapped_cell<L>(p, x0, y, z, L::c(i, 0), L::c(i, 1), L::c(i, 2)) - cell),
                            f[i].v.x);
        if (l1 & (1u << i))
          PairStore<S>::st1(at(opp<L>(i)) + (wrapped_cell<L>(p, x0 + 1, y, z, L::c(i, 0), L::c(i, 1), L::c(i, 2)) - cell),
                            f[i].v.y);
      }
    }
  }
  const bool lo = !fl0 && fl1 && !(nb0 & ~dir_mask<L>(1)), hi = fl0 && !fl1 && !(nb1 & ~dir_mask<L>(-1));
  if ((fl0 && fl1) || lo || hi) {
#pragma unroll
    for (int i = 0; i < L::Q; ++i) {
      S* q = at(i);
      if (L::c(i, 0) == 1 && lo)
        PairStore<S>::st1(q + 1, f[i].v.y);
      else if (L::c(i, 0) == -1 && hi)
        PairStore<S>::st1(q, f[i].v.x);
      else
        PairStore<S>::st2(q, f[i]);
    }
  } else if (fl0 || fl1) {
#pragma unroll
    for (int i = 0; i < L::Q; ++i) PairStore<S>::st1(at(i) + (fl0 ? 0 : 1), fl0 ? f[i].v.x : f[i].v.y);
  }
}

template <class S, bool WALLS, bool TRT>
__global__ void __launch_bounds__(March<S>::THREADS, 1)
    k_step2(Params<float> p, const __grid_constant__ MarchBuf<S> pl, MarchGeom g) {
  using L = D3Q19;
  using M = March<S>;
  using H = Held<S>;
  using HT = typename H::T;
  constexpr int SC_NUM = (int)PairStore<S>::SCALE;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  S* ring = reinterpret_cast<S*>(smem_raw);
  S* sides = ring + M::first(L::Q) * M::PT;
  const int row = threadIdx.x >> 5, lane = threadIdx.x & 31;  // row of the extended tile
  const int xt = blockIdx.x * M::TX;                  // the tile's first cell along x
  const int wx = min(M::TX, p.nx - xt);               // its width (even)
  const int yt = p.y0 + blockIdx.y * M::TY;           // its first row
  const int hy = min(M::TY, p.y1 + 1 - yt);           // its rows
  const int zs = p.z0 + blockIdx.z * g.cz;            // its planes
  const int ze = min(zs + g.cz, p.z1 + 1);
  const int sx = 2 * lane, x0 = xt + sx;              // the pair of this thread
  auto wrap_y = [&](int y) { return y < 0 ? y + p.ny : (y >= p.ny ? y - p.ny : y); };
  auto wrap_z = [&](int z) { return z < 0 ? z + p.nz : (z >= p.nz ? z - p.nz : z); };
  const int y = wrap_y(yt + row - 1);
  const bool act = sx < wx;
  const uint64_t src = __cvta_generic_to_global(pl.src);
  S* own = ring + row * M::RL + sx + 2;  // the ring row's index of x is x - xt + 2

  // The cells left or right of the tile at plane t (lane r: row r): the populations
  // that enter it.
  auto side_cells = [&](bool right, int t, int m4, int m3) {
    const int r = lane;
    if (r > hy + 1) return;
    int xe = right ? xt + wx : xt - 1;
    xe = xe < 0 ? p.nx - 1 : (xe >= p.nx ? xe - p.nx : xe);
    const Nbr n = make_nbr<L>(p, xe, wrap_y(yt + r - 1), wrap_z(t));
    F2 f[L::Q];
#pragma unroll
    for (int i = 0; i < L::Q; ++i)
      f[i] = F2(PairStore<S>::ld1(global_ptr<const S>(
          wide_add(wide_add_s(src, n.at(-L::c(i, 0), -L::c(i, 1), -L::c(i, 2)), (int)sizeof(S)), pl.pitch, i))));
    F2 gamma(1.0f);
    if (p.gamma) gamma = F2(p.gamma[n.cell]);
    F2 drho, j[3], rho, u[3];
    collide_pair<L, SC_NUM, TRT>(p, gamma, f, drho, j, rho, u);
    S* q = ring + r * M::RL + (right ? wx + 2 : 1);
#pragma unroll
    for (int i = 0; i < L::Q; ++i) {
      const int m = L::c(i, 2) == 1 ? m4 : m3;
      if (L::c(i, 0) != 0 && right == (L::c(i, 0) < 0)) {
        if (M::in_ring(i))
          PairStore<S>::st1(q + (M::first(i) + m) * M::PT, f[i].v.x);
        else
          PairStore<S>::st1(sides + (M::side(i) + m) * M::ROWS + r, f[i].v.x);
      }
    }
  };

  const int plane = p.nx * p.ny;
  const int xa = act ? x0 : xt;                            // lanes beyond the tile load its first pair
  const int xm = xa == 0 ? p.nx - 1 : -1;                  // from x0 to x0 - 1, and to x0 + 2
  const int xp = xa + 2 == p.nx ? 2 - p.nx : 2;
  const int yrow[3] = {wrap_y(y - 1) * p.nx + xa, y * p.nx + xa, wrap_y(y + 1) * p.nx + xa};
  // prefetch: 128-byte pieces of this row, one population each, spread over the lanes;
  // population i of plane t + 1 - c_z is first read at plane t + 1
  constexpr int LINES = M::TX * (int)sizeof(S) / 128, PFN = (L::Q * LINES + 31) / 32;
  uint64_t pf[PFN];
  int pf_cz[PFN];  // c_z + 1
  bool pf_ok[PFN];
#pragma unroll
  for (int b = 0; b < PFN; ++b) {
    const int e = b * 32 + lane, i = min(e / LINES, L::Q - 1), x = xt + (e % LINES) * (M::TX / LINES);
    pf_cz[b] = kMarchCz[i];
    pf_ok[b] = e < L::Q * LINES && x < p.nx;
    pf[b] = wide_add_s(wide_add(src, pl.pitch, i), y * p.nx + x - (pf_cz[b] - 1) * plane, (int)sizeof(S));
  }

  // Values of this thread's column that stay in registers, per population: plane t
  // (stage A), t - 1 (both stages) and, for c_z = 1, t - 2.
  HT h1[L::Q], h2[L::Q];
#pragma unroll
  for (int i = 0; i < L::Q; ++i) h1[i] = h2[i] = H::put(F2(0.0f));
  uint32_t wb[2] = {kWordFluid, kWordFluid};
  pdl_wait_then_release();
  const bool outer = row == 0 || row == hy + 1;
  if (outer) side_cells(row != 0, zs - 1, 0, 0);
  int m3 = 0;  // (t - zs + 1) mod 3
  for (int t = zs - 1; t <= ze; ++t) {
    const int m4 = (t - zs + 1) & 3;
    HT h0[L::Q];
    uint32_t wa[2] = {kWordFluid, kWordFluid};
    if (row <= hy + 1) {
      const int z = wrap_z(t);
      const int cell = (z * p.ny + y) * p.nx + xa;
      if (WALLS) {
        const uint2 ww = *reinterpret_cast<const uint2*>(p.word + cell);
        wa[0] = ww.x;
        wa[1] = ww.y;
      }
      const int zrow[3] = {wrap_z(z - 1) * plane, z * plane, wrap_z(z + 1) * plane};
      uint64_t rows[3][3];  // [dz + 1][dy + 1]: the pair's address in population 0
#pragma unroll
      for (int dz = 0; dz < 3; ++dz)
#pragma unroll
        for (int dy = 0; dy < 3; ++dy) rows[dz][dy] = wide_add_s(src, zrow[dz] + yrow[dy], (int)sizeof(S));
      F2 f[L::Q];
#pragma unroll
      for (int i = 0; i < L::Q; ++i) {
        const uint64_t q = wide_add(rows[1 - L::c(i, 2)][1 - L::c(i, 1)], pl.pitch, i);
        const S* a = global_ptr<const S>(q);
        if (L::c(i, 0) == 0)
          f[i] = PairStore<S>::ld2(a);
        else if (L::c(i, 0) == 1)
          f[i] = F2(PairStore<S>::ld1(global_ptr<const S>(wide_add_s(q, xm, (int)sizeof(S)))),
                    PairStore<S>::ld1(a));
        else
          f[i] = F2(PairStore<S>::ld1(a + 1),
                    PairStore<S>::ld1(global_ptr<const S>(wide_add_s(q, xp, (int)sizeof(S)))));
      }
      F2 gamma(1.0f);
      if (p.gamma) gamma = F2(*reinterpret_cast<const float2*>(p.gamma + cell));
      {
        // into L2 what stage A reads first at the next plane
#pragma unroll
        for (int b = 0; b < PFN; ++b)
          if (pf_ok[b] && (unsigned)(t + 2 - pf_cz[b]) < (unsigned)p.nz)
            asm volatile("prefetch.global.L2 [%0];" ::"l"(wide_add_s(pf[b], t + 1, plane * (int)sizeof(S))));
      }
      F2 drho, j[3], rho, u[3];
      collide_pair<L, SC_NUM, TRT>(p, gamma, f, drho, j, rho, u);
      if (WALLS && p.moving) {
        const uint32_t fm = kWordFluid | kWordMoving;
        moving_walls(p, x0, y, z, act && (wa[0] & fm) == fm ? wa[0] & kWordLinks : 0u,
                     act && (wa[1] & fm) == fm ? wa[1] & kWordLinks : 0u, wa, f, rho);
      }
#pragma unroll
      for (int i = 0; i < L::Q; ++i) {
        if (M::in_ring(i)) {
          if (act) PairStore<S>::st2(own + (M::first(i) + (L::c(i, 2) == 1 ? m4 : m3)) * M::PT, f[i]);
        } else {
          h0[i] = H::put(f[i]);
        }
      }
    }
    __syncthreads();
    const int m3b = m3 == 0 ? 2 : m3 - 1;  // ring plane of t - 1
    if (outer) {
      if (t < ze) side_cells(row != 0, t + 1, (m4 + 1) & 3, m3 == 2 ? 0 : m3 + 1);
    } else if (t > zs && row <= hy) {
      const int z = wrap_z(t - 1);
      // ring plane of population i in plane t - 1 - dz
      auto slot = [&](int i, int dz) { return L::c(i, 2) == 1 ? ((m4 - 1 - dz) & 3) : (dz < 0 ? m3 : m3b); };
      F2 f[L::Q];
#pragma unroll
      for (int i = 0; i < L::Q; ++i) {
        const int cx = L::c(i, 0), cz = L::c(i, 2);
        if (M::in_ring(i)) {
          const S* q = own + (M::first(i) + slot(i, cz)) * M::PT - L::c(i, 1) * M::RL;
          if (cx == 0)
            f[i] = PairStore<S>::ld2(q);
          else
            f[i] = F2(PairStore<S>::ld1(q - cx), PairStore<S>::ld1(q + 1 - cx));
        } else {
          const F2 v = H::get(cz == 0 ? h1[i] : (cz == 1 ? h2[i] : h0[i]));
          if (cx == 0) {
            f[i] = v;
          } else {
            const float side = PairStore<S>::ld1(sides + (M::side(i) + slot(i, cz)) * M::ROWS + row);
            if (cx == 1) {
              const float l = __shfl_up_sync(0xffffffffu, v.v.y, 1);
              f[i] = F2(lane == 0 ? side : l, v.v.x);
            } else {
              const float r = __shfl_down_sync(0xffffffffu, v.v.x, 1);
              f[i] = F2(v.v.y, sx + 2 == wx ? side : r);
            }
          }
        }
      }
      if (WALLS) {
        // links that end at a wall: population i returns from the cell's own slot opp(i)
        const uint32_t l0 = act && (wb[0] & kWordFluid) ? wb[0] & kWordLinks : 0u;
        const uint32_t l1 = act && (wb[1] & kWordFluid) ? wb[1] & kWordLinks : 0u;
        auto bounce = [&](auto link) {
          constexpr int o = link, i = opp<L>(link);
          const F2 v = M::in_ring(o) ? PairStore<S>::ld2(own + (M::first(o) + slot(o, 0)) * M::PT) : H::get(h1[o]);
          if ((l0 >> o) & 1u) f[i].v.x = v.v.x;
          if ((l1 >> o) & 1u) f[i].v.y = v.v.y;
        };
        const uint32_t any = __reduce_or_sync(0xffffffffu, l0 | l1);
        if (any) for_links<L>(any, bounce);
      }
      const int cell = (z * p.ny + y) * p.nx + xa;
      F2 gamma(1.0f);
      if (p.gamma) gamma = F2(*reinterpret_cast<const float2*>(p.gamma + cell));
      F2 drho, j[3], rho, u[3];
      collide_pair<L, SC_NUM, TRT>(p, gamma, f, drho, j, rho, u);
      march_store<S, WALLS>(p, pl, act, x0, y, z, cell, wb, f, rho);
    }
#pragma unroll
    for (int i = 0; i < L::Q; ++i) {
      if (!M::in_ring(i)) {
        if (L::c(i, 2) == 1) h2[i] = h1[i];
        h1[i] = h0[i];
      }
    }
    if (WALLS) {
      wb[0] = wa[0];
      wb[1] = wa[1];
    }
    m3 = m3 == 2 ? 0 : m3 + 1;
  }
}

}  // namespace olb
