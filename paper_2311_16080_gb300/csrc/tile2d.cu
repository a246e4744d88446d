// Several D2Q9 updates per launch on a lattice too large for one cluster.
//
// Small 2D lattices cost a launch (and with curved walls a boundary pass) per
// update while their populations sit in L2.  Here each block loads a tile with
// a ring of `halo` cells around it into shared memory, runs up to halo updates
// there and writes the tile: after each update one more cell of the ring is
// wrong (it lacks neighbours), after halo updates exactly the tile is right.
// Nothing is exchanged between blocks; the ring's cells are computed by every
// tile that holds them.
//
// Cells: FLUID and WALL anywhere, an INLET plane x = 0 and an OUTLET plane
// x = nx - 1, Bouzidi links.  In place as slots2d.cuh describes.  In these terms:
//   Bouzidi, wall distance q of the link i, j = opp(i): the pull of x + c_j in
//   direction i is what x itself pulls in direction i, so
//     q <  1/2: f_j = 2q h_i(x) + (1 - 2q) f_i(x) when x pulls;
//     q >= 1/2: h_i(x) / (2q) + (1 - 1/(2q)) h_j(x) is formed when x collides
//               and left in the slot that x will read;
//   OUTLET: the cell x - 1 (no WALL cell) leaves the populations it pulls with
//   c_x = -1 in a stash, and the outlet column is updated after a barrier of its
//   own.
#include <cuda_runtime.h>

#include <type_traits>

#include "../../include/xlb.h"
#include "overlap.cuh"
#include "slots2d.cuh"
#include "tile2d.h"

namespace xlb {
namespace {

constexpr int TILE_THREADS = 768;
constexpr long long TILE_SMEM = 220 * 1024;  // dynamic; the list is static

// meta word of a cell: bits 0-7: x + c_j is a WALL cell or outside the region
// (j = 1..8)
constexpr int M_SOLID = 1 << 8, M_INLET = 1 << 9, M_OUTLET = 1 << 10;
constexpr int M_BEFORE = 1 << 11;  // the cell beside an OUTLET cell
constexpr int M_BZ = 1 << 12;      // has Bouzidi links
constexpr int M_INNER = 1 << 13;   // of the tile, not of the ring
constexpr int M_WALLS = 0xff;
// cells with rules of their own: not in the main loop, where a few lanes would
// hold up every warp they sit in (the 1761 x 330 cylinder: 13 us an update),
// but packed in a list that a few warps work off beside it
constexpr int M_LISTED = M_INLET | M_BEFORE | M_BZ;

// The lattice's slot (direction j, cell) that the ghost value of the link from
// cell `self` in direction i = opp(j) is written to: BF16 rounds it by that
// number.  The wall may lie across a periodic seam.
template <typename S>
__device__ __forceinline__ uint32_t ghost_slot(const StepParams& p, int self, int i, int j) {
  if (!std::is_same<S, __nv_bfloat16>::value) return 0u;  // (no key)
  const int y = self / p.nx, x = self - y * p.nx;
  int xw = x + Lattice<9>::c(i, 0), yw = y + Lattice<9>::c(i, 1);
  xw = xw < 0 ? p.nx - 1 : (xw == p.nx ? 0 : xw);
  yw = yw < 0 ? p.ny - 1 : (yw == p.ny ? 0 : yw);
  return (uint32_t)((long long)j * p.plane + xw + p.nx * yw);
}

// A value as a ghost slot (k of the lattice) would store it.
template <typename S>
__device__ __forceinline__ float ghost_round(uint32_t slot, float v) {
  S s;
  st_ghost<S>(&s, slot, v);
  return Store<S>::ld_plain(&s);
}

struct TileCtx {
  uint32_t base;       // slots
  int rw;              // region's row length
};

template <typename S>
__device__ __forceinline__ void tile_slots(const TileCtx& t, int c, int m, uint32_t (&L)[9]) {
  constexpr int CB = Slots<S>::CELL, SB = (int)sizeof(S);
  const uint32_t a = t.base + (uint32_t)c * CB;
  L[0] = a;
#pragma unroll
  for (int j = 1; j < 9; ++j)
    L[j] = a + (Lattice<9>::c(j, 0) + Lattice<9>::c(j, 1) * t.rw) * CB + opposite<9>(j) * SB;
  if (m & M_WALLS) {
#pragma unroll
    for (int j = 1; j < 9; ++j)
      if (m >> (j - 1) & 1) L[j] = a + j * SB;
  }
}

// Rules of one cell that is INLET, OUTLET, beside an OUTLET or has Bouzidi
// links (rows of the table at q), on its pulled populations; `self` its cell in
// the lattice.
template <typename S>
__device__ __forceinline__ void special_pull(const StepParams& p, int m, int row, int self,
                                             const float2* __restrict__ q, float* stash, float (&f)[9]) {
  if (m & M_BZ) {
    const uint32_t low = __float_as_uint(__ldg(q).x);  // links with q < 1/2
    float g[9];
    g[0] = f[0];
#pragma unroll
    for (int i = 1; i < 9; ++i) {
      const int j = opposite<9>(i);
      const float2 w = __ldg(q + i);
      const float v = ghost_round<S>(ghost_slot<S>(p, self, i, j), __fmaf_rn(w.x, f[j], __fmul_rn(w.y, f[i])));
      g[j] = (low >> i & 1) ? v : f[j];
    }
#pragma unroll
    for (int i = 0; i < 9; ++i) f[i] = g[i];
  }
  if (m & (M_BEFORE | M_OUTLET)) {
    int k = 0;
#pragma unroll
    for (int i = 0; i < 9; ++i)
      if (Lattice<9>::c(i, 0) == -1) {
        if (m & M_BEFORE) stash[3 * row + k] = f[i];
        if (m & M_OUTLET) f[i] = stash[3 * row + k];
        ++k;
      }
  }
  if (m & M_INLET) inlet_rule<9>(p, self, f);
}

// What a cell with Bouzidi links leaves in its slots (at a): links with
// q >= 1/2 take the mixed value in place of h_i.
template <typename S>
__device__ __forceinline__ void special_push(const StepParams& p, int self, const float2* __restrict__ q, uint32_t a,
                                             float (&h)[9]) {
  constexpr int SB = (int)sizeof(S);
  const uint32_t high = __float_as_uint(__ldg(q).y);  // links with q >= 1/2
#pragma unroll
  for (int i = 1; i < 9; ++i) {
    const int j = opposite<9>(i);
    const float2 w = __ldg(q + i);
    S s;
    st_ghost<S>(&s, ghost_slot<S>(p, self, i, j), __fmaf_rn(w.x, h[i], __fmul_rn(w.y, h[j])));
    if (high >> i & 1) {
      if constexpr (sizeof(S) == 4) {
        asm volatile("st.shared.f32 [%0], %1;" ::"r"(a + i * SB), "f"(s) : "memory");
      } else {
        unsigned short u;
        memcpy(&u, &s, 2);
        asm volatile("st.shared.u16 [%0], %1;" ::"r"(a + i * SB), "h"(u) : "memory");
      }
    }
  }
}

// Bounds: FP32 instruction issue and the loads of a launch.  The 1761 x 330 cylinder,
// 4 updates a launch: 227 instructions per lattice cell and update (of which the
// ring and the meta words are some 100), 0.46 issued per cycle and scheduler; waits
// for the tile's loads lead the stalls.  A launch costs 7 us on regions of 2,100
// cells and 12 on 5,500, shared by its updates.
template <typename S, int COLL>
__global__ void __launch_bounds__(TILE_THREADS, 1) k_tile2d(const S* A, S* B,
                                                            const StepParams p, const int* __restrict__ bz,
                                                            const float2* __restrict__ bz_q, const Tile2dPlan plan,
                                                            int steps) {
  extern __shared__ __align__(16) unsigned char smem[];
  constexpr int CB = Slots<S>::CELL, SB = (int)sizeof(S);
  constexpr int MS = sizeof(S) == 4 ? 1 : Slots<S>::STRIDE;
  const int nx = p.nx, ny = p.ny, h = plan.halo;
  const int tx = blockIdx.x % plan.tx, ty = blockIdx.x / plan.tx;
  const int ix0 = tx * plan.bx, iy0 = ty * plan.by;
  const int ix1 = min(ix0 + plan.bx, nx), iy1 = min(iy0 + plan.by, ny);
  // the region; a lattice with inflow / outflow planes ends at them
  const bool clip = p.x_inlet || p.x_outlet;
  const int rx0 = clip ? max(ix0 - h, 0) : ix0 - h, rx1 = clip ? min(ix1 + h, nx) : ix1 + h;
  const int ry0 = iy0 - h, rw = rx1 - rx0, rh = iy1 + h - ry0;
  const int cells = rw * rh;
  const int cap = (plan.bx + 2 * h) * (plan.by + 2 * h);
  TileCtx t;
  t.base = (uint32_t)__cvta_generic_to_shared(smem);
  t.rw = rw;
  unsigned short* meta = reinterpret_cast<unsigned short*>(smem + (sizeof(S) == 4 ? (size_t)cap * CB : 9 * SB));
  float* stash = reinterpret_cast<float*>(
      smem + ((size_t)cap * (sizeof(S) == 4 ? CB + 2 : CB) + 15) / 16 * 16);
  __shared__ uint32_t list[TILE_LIST];  // cell | row of bz_q << 16
  __shared__ int n_list;
  if (threadIdx.x == 0) n_list = 0;
  __syncthreads();
  grid_wait();
  grid_release();
  auto lattice_cell = [&](int c) {
    const int ly = c / rw, lx = c - ly * rw;
    int gx = rx0 + lx, gy = ry0 + ly;
    gx = gx < 0 ? gx + nx : (gx >= nx ? gx - nx : gx);
    gy = gy < 0 ? gy + ny : (gy >= ny ? gy - ny : gy);
    return gx + nx * gy;
  };
  // the populations, with every round's loads in flight
  const int dly = TILE_THREADS / rw, dlx = TILE_THREADS - dly * rw;  // a round further
  auto wrapped = [&](int lx, int ly) {
    int gx = rx0 + lx, gy = ry0 + ly;
    gx = gx < 0 ? gx + nx : (gx >= nx ? gx - nx : gx);
    gy = gy < 0 ? gy + ny : (gy >= ny ? gy - ny : gy);
    return gx + nx * gy;
  };
  {
    int ly = (int)threadIdx.x / rw, lx = (int)threadIdx.x - ly * rw;
    auto next = [&]() {
      lx += dlx;
      ly += dly;
      if (lx >= rw) {
        lx -= rw;
        ++ly;
      }
    };
    if constexpr (sizeof(S) == 4) {
      for (int c = threadIdx.x; c < cells; c += TILE_THREADS, next()) {
        const S* g = A + wrapped(lx, ly);
        const uint32_t a = t.base + (uint32_t)c * CB;
#pragma unroll
        for (int i = 0; i < 9; ++i)
          asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(a + i * SB), "l"(g + (long long)i * p.plane)
                       : "memory");
      }
      asm volatile("cp.async.wait_all;" ::: "memory");
    } else {
      for (int c = threadIdx.x; c < cells; c += 3 * TILE_THREADS) {
        S v[3][9];
#pragma unroll
        for (int k = 0; k < 3; ++k, next()) {
          if (c + k * TILE_THREADS >= cells) continue;
          const S* g = A + wrapped(lx, ly);
#pragma unroll
          for (int i = 0; i < 9; ++i) v[k][i] = g[(long long)i * p.plane];
        }
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          if (c + k * TILE_THREADS >= cells) continue;
          S* cell = reinterpret_cast<S*>(smem + (size_t)(c + k * TILE_THREADS) * CB);
#pragma unroll
          for (int i = 0; i < 9; ++i) cell[i] = v[k][i];
        }
      }
    }
  }
  // the meta words; a thread handles the cells it loaded
  {
    int ly = (int)threadIdx.x / rw, lx = (int)threadIdx.x - ly * rw;
    for (int c = threadIdx.x; c < cells; c += TILE_THREADS) {
      int m = 0, row = 0;
      if (lx >= ix0 - rx0 && lx < ix1 - rx0 && ly >= h && ly < iy1 - ry0) m |= M_INNER;
#pragma unroll
      for (int j = 1; j < 9; ++j) {
        const int x = lx + Lattice<9>::c(j, 0), y = ly + Lattice<9>::c(j, 1);
        if (x < 0 || x >= rw || y < 0 || y >= rh) m |= 1 << (j - 1);
      }
      if (p.flags) {
        const int self = wrapped(lx, ly);
        const int f = p.flags[self], type = f & FLAG_TYPE;
        if (type == WALL) m |= M_SOLID;
        if (type == INLET) m |= M_INLET;
        if (type == OUTLET) m |= M_OUTLET;
        if (f & FLAG_SLOW) {
          const int gy = self / nx, gx = self - gy * nx;
          const int xs[3] = {gx == 0 ? nx - 1 : gx - 1, gx, gx == nx - 1 ? 0 : gx + 1};
          const int ys[3] = {gy == 0 ? ny - 1 : gy - 1, gy, gy == ny - 1 ? 0 : gy + 1};
#pragma unroll
          for (int j = 1; j < 9; ++j)
            if ((p.flags[xs[1 + Lattice<9>::c(j, 0)] + nx * ys[1 + Lattice<9>::c(j, 1)]] & FLAG_TYPE) == WALL)
              m |= 1 << (j - 1);
        }
        if (p.x_outlet && lx == rw - 2 && rx1 == nx && (p.flags[self + 1] & FLAG_TYPE) == OUTLET) m |= M_BEFORE;
        if (bz && (row = bz[self])) {
          m |= M_BZ;
          float v[9];
          const S* cell = reinterpret_cast<const S*>(smem + (size_t)c * CB);
#pragma unroll
          for (int i = 0; i < 9; ++i) v[i] = Store<S>::ld_plain(cell + i);
          special_push<S>(p, self, bz_q + 9 * (row - 1), t.base + (uint32_t)c * CB, v);
        }
      }
      meta[c * MS] = (unsigned short)m;
      if ((m & M_LISTED) && !(m & M_SOLID)) {
        const int k = atomicAdd(&n_list, 1);
        if (k < TILE_LIST) list[k] = (uint32_t)c | (uint32_t)row << 16;  // (the host takes no lattice with more)
      }
      lx += dlx;
      ly += dly;
      if (lx >= rw) {
        lx -= rw;
        ++ly;
      }
    }
  }
  __syncthreads();
  const bool outlet = p.x_outlet && rx1 == nx;
  const int listed = min(n_list, TILE_LIST);
  // the slots of cell c's update
  auto slots = [&](int c, int m, bool odd, uint32_t (&L)[9]) {
    if (odd) {
      tile_slots<S>(t, c, m, L);
    } else {
#pragma unroll
      for (int i = 0; i < 9; ++i) L[i] = t.base + (uint32_t)c * CB + i * SB;
    }
  };
  auto store = [&](const uint32_t (&L)[9], int m, int self, const CellRound<S>& r, const float (&v)[9], bool last) {
    if (m & M_SOLID) return;
    if (!last) {
#pragma unroll
      for (int i = 0; i < 9; ++i) slot_st<S, false>(L[i], r, i, v[i]);
    } else if (m & M_INNER) {
#pragma unroll
      for (int i = 0; i < 9; ++i) r.st(B + (long long)i * p.plane + self, i, v[i]);
    }
  };
  // one update of a cell with rules of its own
  auto special = [&](int c, int row, bool odd, bool last) {
    const int m = meta[c * MS], self = lattice_cell(c);
    uint32_t L[9];
    slots(c, m, odd, L);
    float f[9];
#pragma unroll
    for (int j = 0; j < 9; ++j) f[opposite<9>(j)] = slot_ld<S, false>(L[j]);
    const float2* q = bz_q + 9 * (row - 1);
    special_pull<S>(p, m, c / rw, self, q, stash, f);
    collide<9, COLL>(f, p);
    CellRound<S> r;
    r.begin((uint32_t)self, f);
    store(L, m, self, r, f, last);
    if ((m & M_BZ) && !last) {
#pragma unroll
      for (int i = 0; i < 9; ++i) f[i] = r.rounded(i, f[i]);
      special_push<S>(p, self, q, t.base + (uint32_t)c * CB, f);
    }
  };
  // The listed cells and the outlet column belong to the last warps, which take
  // no part in the main loop: one such cell costs a warp some 2 us of latency.
  int own = (listed + 31) / 32;
  if (outlet && own < 1) own = 1;
  if (own > 8) own = 8;
  const int n_main = TILE_THREADS - 32 * own;
  for (int k = 0; k < steps; ++k) {
    const bool odd = !(k & 1), last = k == steps - 1;
    // the rows whose neighbours are still right
    const int c_lo = (k + 1) * rw, c_hi = cells - (k + 1) * rw;
    if ((int)threadIdx.x >= n_main) {
      // the listed cells, then the outlet column, once the stash is whole
      for (int s = (int)threadIdx.x - n_main; s < listed; s += TILE_THREADS - n_main) {
        const int c = (int)(list[s] & 0xffffu);
        if (c >= c_lo && c < c_hi) special(c, (int)(list[s] >> 16), odd, last);
      }
      if (outlet) {
        asm volatile("bar.sync 1, %0;" ::"r"(TILE_THREADS - n_main) : "memory");
        for (int r = k + 1 + (int)threadIdx.x - n_main; r < rh - (k + 1); r += TILE_THREADS - n_main) {
          const int c = r * rw + rw - 1;
          if ((meta[c * MS] & (M_OUTLET | M_SOLID)) == M_OUTLET) special(c, 0, odd, last);
        }
      }
    } else
    for (int c0 = c_lo + threadIdx.x; c0 < c_hi; c0 += 2 * n_main) {
      const int c1 = c0 + n_main;
      int m0 = meta[c0 * MS], m1 = c1 < c_hi ? meta[c1 * MS] : M_SOLID;
      if (m0 & (M_LISTED | M_OUTLET)) m0 |= M_SOLID;  // not here
      if (m1 & (M_LISTED | M_OUTLET)) m1 |= M_SOLID;
      if (m0 & m1 & M_SOLID) continue;
      // a cell that takes no part reads the other's slots
      const int e0 = (m0 & M_SOLID) ? c1 : c0, e1 = (m1 & M_SOLID) ? c0 : c1;
      uint32_t L0[9], L1[9];
      slots(e0, (m0 & M_SOLID) ? m1 : m0, odd, L0);
      slots(e1, (m1 & M_SOLID) ? m0 : m1, odd, L1);
      F2 f[9];
#pragma unroll
      for (int j = 0; j < 9; ++j) f[opposite<9>(j)] = pack2(slot_ld<S, false>(L0[j]), slot_ld<S, false>(L1[j]));
      collide<9, COLL>(f, p);
      float a[9], b[9];
#pragma unroll
      for (int i = 0; i < 9; ++i) unpack2(f[i], a[i], b[i]);
      int s0 = 0, s1 = 0;
      if (std::is_same<S, __nv_bfloat16>::value || last) {  // (the rounding key, the cell to store)
        s0 = lattice_cell(e0);
        s1 = lattice_cell(e1);
      }
      CellRound<S> r0, r1;
      r0.begin((uint32_t)s0, a);
      r1.begin((uint32_t)s1, b);
      store(L0, m0, s0, r0, a, last);
      store(L1, m1, s1, r1, b, last);
    }
    __syncthreads();
  }
}

template <typename S>
long long tile_smem(int bx, int by, int h) {
  const long long cells = (long long)(bx + 2 * h) * (by + 2 * h);
  return (cells * (sizeof(S) == 4 ? Slots<S>::CELL + 2 : Slots<S>::CELL) + 15) / 16 * 16 + 12LL * (by + 2 * h);
}

template <typename S, int COLL>
int launch_tile_typed(const Tile2dArgs& a) {
  auto kern = k_tile2d<S, COLL>;
  const long long smem = tile_smem<S>(a.plan.bx, a.plan.by, a.plan.halo);
  if (smem > TILE_SMEM) return -1;
  if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TILE_SMEM) != cudaSuccess) return -3;
  return launch_overlapped(kern, dim3((unsigned)(a.plan.tx * a.plan.ty)), dim3(TILE_THREADS), (size_t)smem,
                           (cudaStream_t)a.stream, (const S*)a.src, (S*)a.dst, a.p, a.bz, (const float2*)a.bz_q, a.plan,
                           a.steps) == cudaSuccess ? 0 : -3;
}

template <typename S>
int tile_by_coll(const Tile2dArgs& a) {
  if (a.coll == COLL_BGK) return launch_tile_typed<S, COLL_BGK>(a);
  if (a.coll == COLL_KBC) return launch_tile_typed<S, COLL_KBC>(a);
  return -2;
}

}  // namespace

// Tiles that a model of the kernel expects to take the least time per update:
// waves of blocks over the SMs, 5 us a launch for load and store, and per update
// 0.8 us and a time for each round of two cells per thread.  (It ranks plans; what
// one takes is tile_us in api.cu.)
Tile2dPlan tile2d_plan(int storage, int coll, int nx, int ny) {
  Tile2dPlan best = {0, 0, 0, 0, 0, 0.f, 0};
  const float over = 5.0f, per = coll == COLL_KBC ? 2.9f : storage == XLB_STORE_BF16 ? 1.8f : 0.85f;
  for (int tx = 1; tx <= nx && tx <= 152; ++tx) {
    const int bx = (nx + tx - 1) / tx;
    if ((nx + bx - 1) / bx != tx) continue;
    for (int ty = 1; ty <= ny && tx * ty <= 2 * 152; ++ty) {
      const int by = (ny + ty - 1) / ty;
      if ((ny + by - 1) / by != ty) continue;
      for (int h = 2; h <= 12; ++h) {
        if (bx + 2 * h > nx || by + 2 * h > ny) break;  // a cell at most once in a region
        const long long smem = storage == XLB_STORE_F32 ? tile_smem<float>(bx, by, h) : tile_smem<__half>(bx, by, h);
        if (smem > TILE_SMEM) break;
        const int waves = (tx * ty + 151) / 152;
        // (a row of the ring less per update on either side)
        const long long busy = (long long)(bx + 2 * h) * (by + h - 1);
        const float rounds = (float)((busy + 2 * TILE_THREADS - 1) / (2 * TILE_THREADS));
        const float us = waves * (over + h * (0.8f + rounds * per)) / h;
        if (best.halo == 0 || us < best.us) best = {bx, by, tx, ty, h, us, waves};
      }
    }
  }
  return best;
}

int launch_tile2d(const Tile2dArgs& a) {
  if (a.plan.halo < 1 || a.steps < 1 || a.steps > a.plan.halo) return -1;
  switch (a.storage) {
    case XLB_STORE_F32: return tile_by_coll<float>(a);
    case XLB_STORE_F16: return tile_by_coll<__half>(a);
    case XLB_STORE_BF16: return tile_by_coll<__nv_bfloat16>(a);
  }
  return -5;
}

}  // namespace xlb
