// Resident D2Q9 updates: the populations of one domain stay in the shared
// memory of a thread-block cluster for all the updates of a call, so that
// between the first read and the last write nothing goes through L2 or HBM
// and a step costs a cluster barrier instead of a launch.
//
// The slots and the in-place scheme: slots2d.cuh.  The last update writes h
// straight to global memory.
#include <cuda_runtime.h>

#include "../../include/xlb.h"
#include "lbm_device.cuh"
#include "resident2d.h"
#include "slots2d.cuh"

namespace xlb {
namespace {

// Dynamic shared memory a block may take.  The kernels are allowed all of it,
// whatever a launch needs: that attribute belongs to the function, which other
// threads launch with other sizes.
constexpr int RESIDENT_SMEM = 220 * 1024;

// meta word of a cell: bits 0-7: x + c_j is a WALL cell (j = 1..8)
constexpr int M_SOLID = 1 << 8;                       // the cell itself is a WALL cell
constexpr int M_XL = 1 << 9, M_XR = 1 << 10;          // x = 0 / x = nx - 1
constexpr int M_YB = 1 << 11, M_YT = 1 << 12;         // first / last row of the block's part
constexpr int M_WALLS = 0xff;

__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ uint32_t cluster_size() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ uint32_t cluster_id() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%clusterid.x;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_barrier() {
  asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}
__device__ __forceinline__ uint32_t map_rank(uint32_t addr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}

// Addresses L_j(x), j = 1..8, of one cell's odd update, from the addresses of
// the cell itself (aM) and of its column in the rows above and below.
template <typename S>
__device__ __forceinline__ void odd_slots(uint32_t aM, uint32_t aU, uint32_t aD, int m, int nx, uint32_t (&L)[9]) {
  constexpr int CB = Slots<S>::CELL, SB = (int)sizeof(S);
  const int xp = (m & M_XR) ? (1 - nx) * CB : CB;
  const int xm = (m & M_XL) ? (nx - 1) * CB : -CB;
  L[0] = aM;
#pragma unroll
  for (int j = 1; j < 9; ++j) {
    const int cx = Lattice<9>::c(j, 0), cy = Lattice<9>::c(j, 1);
    const uint32_t row = cy == 0 ? aM : (cy == 1 ? aU : aD);
    L[j] = row + (cx == 0 ? 0 : (cx == 1 ? xp : xm)) + opposite<9>(j) * SB;
  }
  if (m & M_WALLS) {
#pragma unroll
    for (int j = 1; j < 9; ++j)
      if (m >> (j - 1) & 1) L[j] = aM + j * SB;
  }
}

// Cells per thread: one, whose slot addresses stay in registers for the whole
// call, or as many as it takes, two at a time.
enum ResidentMode { R_SINGLE, R_LOOP };

// Whether a slot in direction j of an odd update may lie in another block: a
// neighbouring row's, in the first and last rows (FAR).  (Upper and lower rows
// apart cost more in diverging warps than they spared: channel 203 x 67 573 ->
// 612 us.)
template <bool FAR>
__device__ constexpr bool is_far(int j) {
  return FAR && Lattice<9>::c(j, 1) != 0;
}

// The block's part of the domain and what an update needs of it.
struct Part {
  uint32_t base, topU, botD;  // slots; where the rows beyond the last / first one lie
  int nx, plane;
  bool split;                 // those rows belong to other blocks
  uint32_t key0;              // rounding key of the part's first cell
};

template <typename S>
__device__ __forceinline__ void cell_slots(const Part& d, int c, int m, uint32_t (&L)[9]) {
  constexpr int CB = Slots<S>::CELL;
  const uint32_t aM = d.base + (uint32_t)c * CB;
  const uint32_t aU = (m & M_YT) ? d.topU + (uint32_t)c * CB : aM + (uint32_t)d.nx * CB;
  const uint32_t aD = (m & M_YB) ? d.botD + (uint32_t)c * CB : aM - (uint32_t)d.nx * CB;
  odd_slots<S>(aM, aU, aD, m, d.nx, L);
}

// One update of one cell with slots L (L[0]: its own).
template <typename S, int COLL, bool ODD, bool FAR>
__device__ __forceinline__ void update_one(const uint32_t (&L)[9], int c, const Part& d, const StepParams& p, bool last,
                                           S* out) {
  constexpr int SB = (int)sizeof(S);
  float f[9];
#pragma unroll
  for (int j = 0; j < 9; ++j) {
    if (is_far<FAR>(j))
      f[opposite<9>(j)] = slot_ld<S, true>(ODD ? L[j] : L[0] + j * SB);
    else
      f[opposite<9>(j)] = slot_ld<S, false>(ODD ? L[j] : L[0] + j * SB);
  }
  collide<9, COLL>(f, p);
  CellRound<S> r;
  r.begin(d.key0 + c, f);
  if (last) {
#pragma unroll
    for (int i = 0; i < 9; ++i) r.st(out + (long long)i * d.plane + c, i, f[i]);
    return;
  }
#pragma unroll
  for (int i = 0; i < 9; ++i) {
    if (is_far<FAR>(i))
      slot_st<S, true>(ODD ? L[i] : L[0] + i * SB, r, i, f[i]);
    else
      slot_st<S, false>(ODD ? L[i] : L[0] + i * SB, r, i, f[i]);
  }
}

// One update of two cells (c0 and c1, the collision in packed arithmetic);
// m: their meta words, a cell that takes no part is marked M_SOLID and its
// addresses are then the other's.  In the call's last update the result goes
// to global memory (out: the part's first cell), else back to the slots.
template <typename S, int COLL, bool ODD, bool FAR>
__device__ __forceinline__ void update_pair(const uint32_t (&L0)[9], const uint32_t (&L1)[9], int c0, int c1, int m0,
                                            int m1, const Part& d, const StepParams& p, bool last, S* out) {
  constexpr int SB = (int)sizeof(S);
  float a[9], b[9];
  // odd: slot L_j holds f_opp(j); even: slot i of the cell holds f_opp(i)
#pragma unroll
  for (int j = 0; j < 9; ++j) {
    if (is_far<FAR>(j)) {
      a[opposite<9>(j)] = slot_ld<S, true>(ODD ? L0[j] : L0[0] + j * SB);
      b[opposite<9>(j)] = slot_ld<S, true>(ODD ? L1[j] : L1[0] + j * SB);
    } else {
      a[opposite<9>(j)] = slot_ld<S, false>(ODD ? L0[j] : L0[0] + j * SB);
      b[opposite<9>(j)] = slot_ld<S, false>(ODD ? L1[j] : L1[0] + j * SB);
    }
  }
  F2 f[9];
#pragma unroll
  for (int i = 0; i < 9; ++i) f[i] = pack2(a[i], b[i]);
  collide<9, COLL>(f, p);
#pragma unroll
  for (int i = 0; i < 9; ++i) unpack2(f[i], a[i], b[i]);
  CellRound<S> r0, r1;
  r0.begin(d.key0 + c0, a);
  r1.begin(d.key0 + c1, b);
  if (last) {
#pragma unroll
    for (int i = 0; i < 9; ++i) {
      if (!(m0 & M_SOLID)) r0.st(out + (long long)i * d.plane + c0, i, a[i]);
      if (!(m1 & M_SOLID)) r1.st(out + (long long)i * d.plane + c1, i, b[i]);
    }
    return;
  }
  if (!(m0 & M_SOLID)) {
#pragma unroll
    for (int i = 0; i < 9; ++i) {
      if (is_far<FAR>(i))
        slot_st<S, true>(ODD ? L0[i] : L0[0] + i * SB, r0, i, a[i]);
      else
        slot_st<S, false>(ODD ? L0[i] : L0[0] + i * SB, r0, i, a[i]);
    }
  }
  if (!(m1 & M_SOLID)) {
#pragma unroll
    for (int i = 0; i < 9; ++i) {
      if (is_far<FAR>(i))
        slot_st<S, true>(ODD ? L1[i] : L1[0] + i * SB, r1, i, b[i]);
      else
        slot_st<S, false>(ODD ? L1[i] : L1[0] + i * SB, r1, i, b[i]);
    }
  }
}

// Bounds: a batch by FP32 instruction issue (608 domains of 60 x 44, one block
// each: 128 instructions per cell and update, 0.58 issued per cycle and scheduler,
// then math pipe and barrier stalls); one small domain by the latency
// of a cluster barrier (287 ns) and of one cell's chain.  Each thread takes two
// cells a warp's width apart: the lanes of a warp stay on consecutive cells, the
// collision runs in packed arithmetic, and few warps hold cells of the rows
// whose neighbours are in another block (a pair a block apart instead: 1024
// channels 51.0 ms, this way 47.7).
template <typename S, int COLL, int MODE>
__global__ void __launch_bounds__(MODE == R_SINGLE ? 1024 : 768, 1) k_resident2d(const S* A, S* B, const uint8_t* __restrict__ flags,
                                                       const BatchDom* __restrict__ doms,
                                                       const int* __restrict__ order, const BatchDom one, float omega,
                                                       int steps) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int C = (int)cluster_size(), rank = (int)cluster_rank();
  const BatchDom d = doms ? doms[order[cluster_id()]] : one;
  const int nx = d.nx, ny = d.ny;
  // rows of block r: a whole number, the first ny % C blocks take one more
  const int rmin = ny / C, extra = ny % C;
  const int rows = rmin + (rank < extra), y0 = rank * rmin + min(rank, extra);
  const int cells = rows * nx, cap = (rmin + (extra > 0)) * nx;
  constexpr int CB = Slots<S>::CELL, SB = (int)sizeof(S);
  Part part;
  part.base = (uint32_t)__cvta_generic_to_shared(smem);
  unsigned short* meta = reinterpret_cast<unsigned short*>(smem + (sizeof(S) == 4 ? (size_t)cap * CB : 9 * SB));
  constexpr int MS = sizeof(S) == 4 ? 1 : Slots<S>::STRIDE;  // meta words between cells
  const int up = rank + 1 == C ? 0 : rank + 1, dn = rank == 0 ? C - 1 : rank - 1;
  part.topU = (C == 1 ? part.base : map_rank(part.base, up)) - (uint32_t)((rows - 1) * nx) * CB;
  part.botD = (C == 1 ? part.base : map_rank(part.base, dn)) + (uint32_t)((rmin + (dn < extra) - 1) * nx) * CB;
  part.nx = nx;
  part.plane = d.plane;
  part.split = C > 1;
  StepParams p;
  p.omega = omega;
  p.has_force = (d.Fx != 0.f || d.Fy != 0.f);
  p.F[0] = d.Fx;
  p.F[1] = d.Fy;
  p.F[2] = 0.f;
  const uint8_t* fl = flags ? flags + d.foff : nullptr;
  const int g0 = y0 * nx;  // the part's first cell in the domain
  const S* src = A + d.off + g0;
  S* dst = B + d.off + g0;
  part.key0 = (uint32_t)d.off + (uint32_t)g0;
  for (int c = threadIdx.x; c < cells; c += blockDim.x) {
    const int ry = c / nx, x = c - ry * nx, y = y0 + ry;
    int m = (x == 0 ? M_XL : 0) | (x == nx - 1 ? M_XR : 0) | (ry == 0 ? M_YB : 0) | (ry == rows - 1 ? M_YT : 0);
    if (fl) {
      if ((__ldg(fl + g0 + c) & FLAG_TYPE) != FLUID) m |= M_SOLID;
      if (__ldg(fl + g0 + c) & FLAG_SLOW) {
        const int xs[3] = {x == 0 ? nx - 1 : x - 1, x, x == nx - 1 ? 0 : x + 1};
        const int ys[3] = {y == 0 ? ny - 1 : y - 1, y, y == ny - 1 ? 0 : y + 1};
#pragma unroll
        for (int j = 1; j < 9; ++j)
          if ((__ldg(fl + xs[1 + Lattice<9>::c(j, 0)] + nx * ys[1 + Lattice<9>::c(j, 1)]) & FLAG_TYPE) != FLUID)
            m |= 1 << (j - 1);
      }
    }
    meta[c * MS] = (unsigned short)m;
    S* cell = reinterpret_cast<S*>(smem + (size_t)c * CB);
#pragma unroll
    for (int i = 0; i < 9; ++i) cell[i] = src[(long long)i * d.plane + c];
  }
  auto barrier = [&]() {
    if (C == 1)
      __syncthreads();
    else
      cluster_barrier();
  };
  barrier();
  if constexpr (MODE == R_SINGLE) {
    const int c = threadIdx.x, m = c < cells ? meta[c * MS] : M_SOLID;
    uint32_t L[9];
    if (!(m & M_SOLID)) cell_slots<S>(part, c, m, L);
    const bool far = part.split && (m & (M_YT | M_YB));
    for (int t = 0; t < steps; ++t) {
      const bool last = t == steps - 1;
      if (!(m & M_SOLID)) {
        if (t & 1)
          update_one<S, COLL, false, false>(L, c, part, p, last, dst);
        else if (far)
          update_one<S, COLL, true, true>(L, c, part, p, last, dst);
        else
          update_one<S, COLL, true, false>(L, c, part, p, last, dst);
      }
      barrier();
    }
  } else {
    for (int t = 0; t < steps; ++t) {
      const bool last = t == steps - 1;
      for (int c0 = 2 * (threadIdx.x & ~31) + (threadIdx.x & 31); c0 < cells; c0 += 2 * blockDim.x) {
        const int c1 = c0 + 32;
        const int m0 = meta[c0 * MS], m1 = c1 < cells ? meta[c1 * MS] : M_SOLID;
        if (m0 & m1 & M_SOLID) continue;
        uint32_t L0[9], L1[9];
        // a cell that takes no part reads the other's slots
        const int e0 = (m0 & M_SOLID) ? c1 : c0, e1 = (m1 & M_SOLID) ? c0 : c1;
        if (t & 1) {
          L0[0] = part.base + (uint32_t)e0 * CB;
          L1[0] = part.base + (uint32_t)e1 * CB;
          update_pair<S, COLL, false, false>(L0, L1, c0, c1, m0, m1, part, p, last, dst);
        } else {
          const int n0 = (m0 & M_SOLID) ? m1 : m0, n1 = (m1 & M_SOLID) ? m0 : m1;
          cell_slots<S>(part, e0, n0, L0);
          cell_slots<S>(part, e1, n1, L1);
          if (part.split && ((n0 | n1) & (M_YT | M_YB)))
            update_pair<S, COLL, true, true>(L0, L1, c0, c1, m0, m1, part, p, last, dst);
          else
            update_pair<S, COLL, true, false>(L0, L1, c0, c1, m0, m1, part, p, last, dst);
        }
      }
      barrier();  // also the last one: no block leaves while another reads its slots
    }
  }
}

// Where a launch goes instead of a.stream: a node of `graph`, or nowhere, only
// counting the clusters that fit the GPU.
struct Target {
  cudaGraph_t graph;
  int* clusters;
};

template <typename S, int COLL>
int launch_typed_resident(const ResidentArgs& a, const Target* t) {
  // (more than one cell per thread: the domains of a batch, which is BGK)
  if (COLL != COLL_BGK && !a.shape.one) return -2;
  auto kern = k_resident2d<S, COLL, R_SINGLE>;
  if constexpr (COLL == COLL_BGK)
    if (!a.shape.one) kern = k_resident2d<S, COLL, R_LOOP>;
  if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, RESIDENT_SMEM) != cudaSuccess ||
      (a.shape.ctas > 8 && cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess))
    return -3;
  const S* src = (const S*)a.src;
  S* dst = (S*)a.dst;
  const dim3 grid((unsigned)(a.n_dom * a.shape.ctas)), block((unsigned)a.shape.threads);
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = (unsigned)a.shape.ctas;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = (size_t)a.shape.smem;
  cfg.stream = (cudaStream_t)a.stream;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  if (t && t->clusters) return cudaOccupancyMaxActiveClusters(t->clusters, kern, &cfg) == cudaSuccess ? 0 : -3;
  if (t) {
    ResidentArgs c = a;  // the parameters' values are copied into the node
    void* args[] = {&src, &dst, &c.flags, &c.doms, &c.order, &c.dom, &c.omega, &c.steps};
    cudaKernelNodeParams kp = {};
    kp.func = (void*)kern;
    kp.gridDim = grid;
    kp.blockDim = block;
    kp.sharedMemBytes = (unsigned)a.shape.smem;
    kp.kernelParams = args;
    cudaGraphNode_t node;
    return cudaGraphAddKernelNode(&node, t->graph, nullptr, 0, &kp) == cudaSuccess &&
                   cudaGraphKernelNodeSetAttribute(node, cudaLaunchAttributeClusterDimension, &at[0].val) == cudaSuccess
               ? 0
               : -3;
  }
  return cudaLaunchKernelEx(&cfg, kern, src, dst, a.flags, a.doms, a.order, a.dom, a.omega, a.steps) == cudaSuccess
             ? 0
             : -3;
}

template <typename S>
int by_coll(const ResidentArgs& a, const Target* t) {
  if (a.coll == COLL_BGK) return launch_typed_resident<S, COLL_BGK>(a, t);
  if (a.coll == COLL_KBC) return launch_typed_resident<S, COLL_KBC>(a, t);
  return -2;
}

int launch_to(const ResidentArgs& a, const Target* t) {
  if (a.n_dom < 1 || a.steps < 1 || a.shape.ctas < 1) return -1;
  switch (a.storage) {
    case XLB_STORE_F32: return by_coll<float>(a, t);
    case XLB_STORE_F16: return by_coll<__half>(a, t);
    case XLB_STORE_BF16: return by_coll<__nv_bfloat16>(a, t);
  }
  return -5;
}

}  // namespace

ResidentShape resident2d_shape(int storage, int coll, int nx, int ny, bool alone) {
  const ResidentShape none = {0, 0, 0, false};
  if (coll != COLL_BGK && coll != COLL_KBC) return none;
  const long long cell = storage == XLB_STORE_F32 ? 9 * 4 + 2 : 10 * 2;  // Slots<S>, meta included
  auto fit = [&](int ctas, long long limit, bool one) {
    const int c = ctas > ny ? ny : ctas;
    const long long cells = (long long)((ny + c - 1) / c) * nx;
    const long long smem = (cells * cell + 15) / 16 * 16;
    if (smem > limit || (one && cells > 1024)) return none;
    if (cells <= 1024) return ResidentShape{c, (int)((cells + 31) / 32 * 32), smem, true};
    // 80 registers: 768 threads fill an SM
    return ResidentShape{c, limit == RESIDENT_SMEM ? 768 : 384, smem, false};
  };
  if (alone) return fit(16, RESIDENT_SMEM, true);
  // many domains: two blocks per SM where eight blocks' worth of that is
  // enough, else one
  for (long long limit : {112 * 1024, RESIDENT_SMEM})
    for (int ctas = 1; ctas <= 8; ++ctas) {
      const ResidentShape s = fit(ctas, limit, false);
      if (s.ctas > 0) return s;
    }
  return none;
}

int launch_resident2d(const ResidentArgs& a) { return launch_to(a, nullptr); }

int add_resident2d_node(const ResidentArgs& a, void* graph) {
  const Target t = {(cudaGraph_t)graph, nullptr};
  return launch_to(a, &t);
}

int resident2d_clusters(const ResidentShape& shape, int storage, int coll) {
  ResidentArgs a = {};
  a.n_dom = a.steps = 1;
  a.storage = storage;
  a.coll = coll;
  a.shape = shape;
  int n = 0;
  const Target t = {nullptr, &n};
  if (launch_to(a, &t) == 0) return n;
  cudaGetLastError();
  return 0;
}

}  // namespace xlb
