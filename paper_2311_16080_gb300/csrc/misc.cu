// Lattice-independent kernels: mask preparation and the final FP64
// reduction of block partial sums.
#include <cuda_runtime.h>

#include "launch.h"
#include "lattice.cuh"

namespace xlb {

long long row_blocks(const StepParams& p) {
  const long long nxb = (p.nx + 127) / 128;
  return nxb * (long long)p.ny * p.nz;
}

long long cell_blocks(const StepParams& p) {
  return p.mag_x ? ((long long)p.nx * p.ny * p.nz + 127) / 128 : row_blocks(p);
}

// Coordinates of a cell index; 32-bit divisions where the lattice allows.
__device__ __forceinline__ void cell_xyz(long long cell, int nx, int ny, bool small, int& x, int& y, int& z) {
  if (small) {
    const unsigned c = (unsigned)cell, r = c / (unsigned)nx;
    x = (int)(c - r * (unsigned)nx);
    y = (int)(r % (unsigned)ny);
    z = (int)(r / (unsigned)ny);
  } else {
    const long long r = cell / nx;
    x = (int)(cell - r * nx);
    y = (int)(r % ny);
    z = (int)(r / ny);
  }
}

// flags = type | FLAG_SLOW where a fluid-like cell has a WALL / LID / EQ cell
// in its Q-stencil, or is an INLET / OUTLET / FWALL cell.  Codes >= 7 set
// err[0]; an INLET, OUTLET or FWALL cell anywhere sets bit 0 of err[2], a LID
// or EQ cell bit 1, an OUTLET cell beside a WALL cell at x - 1 bit 2.
template <int Q>
__global__ void k_mask_prepare(const uint8_t* __restrict__ mask, uint8_t* __restrict__ flags, int nx, int ny,
                               int nz, int* err) {
  // blocks stride over the rows (y, z), threads over x: no division per cell
  const long long rows = (long long)ny * nz;
  int seen = 0;
  for (long long row = blockIdx.x; row < rows; row += gridDim.x) {
    const int y = (int)(row % ny), z = (int)(row / ny);
    const int ym = y == 0 ? ny - 1 : y - 1, yp = y == ny - 1 ? 0 : y + 1;
    const int zm = z == 0 ? nz - 1 : z - 1, zp = z == nz - 1 ? 0 : z + 1;
    const uint8_t* rb[3][3];
    {
      const int ys[3] = {ym, y, yp}, zs[3] = {zm, z, zp};
#pragma unroll
      for (int b = 0; b < 3; ++b)
#pragma unroll
        for (int c = 0; c < 3; ++c) rb[b][c] = mask + (long long)nx * (ys[b] + (long long)ny * zs[c]);
    }
    for (int x = threadIdx.x; x < nx; x += blockDim.x) {
      const long long cell = x + (long long)nx * row;
      const int t = mask[cell];
      if (t > FWALL) {
        atomicExch(err, 1);
        flags[cell] = WALL;
        continue;
      }
      int slow = (t == INLET || t == OUTLET || t == FWALL);
      seen |= slow | (t == LID || t == EQ ? 2 : 0);
      if (t == OUTLET && x > 0 && mask[cell - 1] == WALL) seen |= 4;
      if (fluid_like(t) && !slow) {
        const int xs[3] = {x == 0 ? nx - 1 : x - 1, x, x == nx - 1 ? 0 : x + 1};
#pragma unroll
        for (int i = 1; i < Q; ++i) {
          const int ts = rb[1 - Lattice<Q>::c(i, 1)][1 - Lattice<Q>::c(i, 2)][xs[1 - Lattice<Q>::c(i, 0)]];
          if (!holds_state(ts)) slow = 1;
        }
      }
      flags[cell] = (uint8_t)(t | (slow ? FLAG_SLOW : 0));
    }
  }
  if (seen) atomicOr(err + 2, seen);
}

int launch_mask_prepare(int Q, const uint8_t* mask, uint8_t* flags, int nx, int ny, int nz, int* err,
                        void* stream) {
  const long long rows = (long long)ny * nz;
  long long blocks = rows < 152LL * 64 ? rows : 152LL * 64;
  if (blocks < 1) blocks = 1;
  cudaStream_t s = (cudaStream_t)stream;
  if (Q == 9)
    k_mask_prepare<9><<<(unsigned)blocks, 256, 0, s>>>(mask, flags, nx, ny, nz, err);
  else if (Q == 19)
    k_mask_prepare<19><<<(unsigned)blocks, 256, 0, s>>>(mask, flags, nx, ny, nz, err);
  else if (Q == 27)
    k_mask_prepare<27><<<(unsigned)blocks, 256, 0, s>>>(mask, flags, nx, ny, nz, err);
  else
    return -1;
  return 0;
}

// Boundary tables, built once per mask by compaction in two launches over
// chunks of consecutive cells, each evaluating every table for its cells
// (per-chunk counts; an exclusive scan of the counts on the host; then
// ordered per-chunk writes):
//  - links, direction-major: for each direction i in turn, every FLUID cell,
//    every FWALL cell on an FWALL face plane and every inlet / outlet cell the
//    bulk pass serves, x (ascending), whose source x - c_i is WALL, LID or EQ
//    and not on a face plane, as {x, i | type << 8}.  Consecutive entries
//    then touch consecutive cells of one population plane wherever the wall
//    is not normal to x;
//  - fix-up cells: every other INLET and OUTLET cell and every FWALL cell off
//    the face planes, ascending.
constexpr int LIST_BLOCK = 256;

struct Pred {
  int face[6];     // described boundary faces: their sources need no ghost
  int x_in, x_out; // INLET cells of x = 0 / OUTLET cells of x = nx - 1 served by the bulk pass
};

// Does (x, y, z) lie on one of the described face planes?
__device__ __forceinline__ bool on_face_plane(int x, int y, int z, int nx, int ny, int nz, const Pred& pr) {
  return (x == 0 && pr.face[0]) || (x == nx - 1 && pr.face[1]) || (y == 0 && pr.face[2]) ||
         (y == ny - 1 && pr.face[3]) || (nz > 1 && z == 0 && pr.face[4]) || (nz > 1 && z == nz - 1 && pr.face[5]);
}

// Every table entry of one cell at once: bit i (1 <= i < Q) of the result
// says that the cell owns a link in direction i (types[i] = the source's
// type), bit Q that it is a fix-up cell.  The coordinates are found once and
// the Q - 1 neighbour flags are loaded together.
template <int Q>
__device__ __forceinline__ uint32_t cell_preds(const uint8_t* __restrict__ flags, long long cell, long long n, int nx,
                                               int ny, int nz, const Pred& pr, uint8_t (&types)[Q]) {
  // only FLUID cells with a WALL / LID / EQ neighbour and INLET / OUTLET /
  // FWALL cells carry FLAG_SLOW; every other cell has no entry
  if (cell >= n) return 0u;
  const int fl = flags[cell];
  if (!(fl & FLAG_SLOW)) return 0u;
  const int t = fl & FLAG_TYPE;
  if (!(t == FLUID || t == FWALL || t == INLET || t == OUTLET)) return 0u;
  int x, y, z;
  cell_xyz(cell, nx, ny, (long long)nx * ny * nz < 0x7fffffffLL, x, y, z);
  // inlet / outlet cells on the x-planes the bulk pass serves
  const bool io_bulk = (t == INLET && pr.x_in && x == 0) || (t == OUTLET && pr.x_out && x == nx - 1);
  // an FWALL cell on a face plane is updated by the bulk pass (it lies on an
  // FWALL face: the host keeps a face only where its plane's cells have the
  // type the faces derive); any other FWALL cell is a fix-up cell
  const bool fw_face = t == FWALL && on_face_plane(x, y, z, nx, ny, nz, pr);
  const bool fix = ((t == INLET || t == OUTLET) && !io_bulk) || (t == FWALL && !fw_face);
  uint32_t bits = fix ? 1u << Q : 0u;
  if (!(t == FLUID || fw_face || io_bulk)) return bits;
  const int xs[3] = {x == 0 ? nx - 1 : x - 1, x, x == nx - 1 ? 0 : x + 1};
  const int ys[3] = {y == 0 ? ny - 1 : y - 1, y, y == ny - 1 ? 0 : y + 1};
  const int zs[3] = {z == 0 ? nz - 1 : z - 1, z, z == nz - 1 ? 0 : z + 1};
  int ts[Q];
#pragma unroll
  for (int i = 1; i < Q; ++i)
    ts[i] = flags[xs[1 - Lattice<Q>::c(i, 0)] +
                  (long long)nx * (ys[1 - Lattice<Q>::c(i, 1)] + (long long)ny * zs[1 - Lattice<Q>::c(i, 2)])] &
            FLAG_TYPE;
#pragma unroll
  for (int i = 1; i < Q; ++i) {
    const int sx = xs[1 - Lattice<Q>::c(i, 0)], sy = ys[1 - Lattice<Q>::c(i, 1)], sz = zs[1 - Lattice<Q>::c(i, 2)];
    if (!holds_state(ts[i]) && !on_face_plane(sx, sy, sz, nx, ny, nz, pr)) {
      bits |= 1u << i;
      types[i] = (uint8_t)ts[i];
    }
  }
  return bits;
}

// Chunks of LIST_SUB x LIST_BLOCK consecutive cells, taken by a block in
// LIST_SUB rounds of LIST_BLOCK cells (ascending), so that the host scans one
// count per chunk and table.
constexpr int LIST_SUB = 16;

template <int Q>
__global__ void k_pred_count(const uint8_t* __restrict__ flags, long long n, int nx, int ny, int nz, Pred pr,
                             long long nchunks, int* counts) {
  for (long long chunk = blockIdx.x; chunk < nchunks; chunk += gridDim.x) {
    int acc[Q + 1];
#pragma unroll
    for (int pass = 0; pass <= Q; ++pass) acc[pass] = 0;
    for (int sub = 0; sub < LIST_SUB; ++sub) {
      uint8_t types[Q];
      const long long cell = (chunk * LIST_SUB + sub) * LIST_BLOCK + threadIdx.x;
      const uint32_t bits = cell_preds<Q>(flags, cell, n, nx, ny, nz, pr, types);
      if (!__syncthreads_or(bits != 0u)) continue;
#pragma unroll
      for (int pass = 1; pass <= Q; ++pass) acc[pass] += __syncthreads_count((bits >> pass) & 1u);
    }
    if (threadIdx.x == 0) {
#pragma unroll
      for (int pass = 1; pass <= Q; ++pass) counts[nchunks * pass + chunk] = acc[pass];
    }
  }
}

template <int Q>
__global__ void k_pred_write(const uint8_t* __restrict__ flags, long long n, int nx, int ny, int nz, Pred pr,
                             long long nchunks, const long long* __restrict__ offs, int2* links, int* cells) {
  __shared__ int warp_base[LIST_BLOCK / 32];
  __shared__ int round_total;
  __shared__ long long next[Q + 1];  // the next entry of each table in this chunk
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (long long chunk = blockIdx.x; chunk < nchunks; chunk += gridDim.x) {
    __syncthreads();  // next[] of the previous chunk has been read
    if (threadIdx.x <= Q && threadIdx.x > 0) next[threadIdx.x] = offs[nchunks * threadIdx.x + chunk];
    __syncthreads();
    for (int sub = 0; sub < LIST_SUB; ++sub) {
      const long long cell = (chunk * LIST_SUB + sub) * LIST_BLOCK + threadIdx.x;
      uint8_t types[Q];
      const uint32_t bits = cell_preds<Q>(flags, cell, n, nx, ny, nz, pr, types);
      if (!__syncthreads_or(bits != 0u)) continue;
#pragma unroll
      for (int pass = 1; pass <= Q; ++pass) {
        const int hit = (bits >> pass) & 1u;
        const unsigned ballot = __ballot_sync(0xffffffffu, hit);
        if (lane == 0) warp_base[warp] = __popc(ballot);
        __syncthreads();
        if (threadIdx.x == 0) {
          int run = 0;
          for (int w = 0; w < LIST_BLOCK / 32; ++w) {
            const int c = warp_base[w];
            warp_base[w] = run;
            run += c;
          }
          round_total = run;
        }
        __syncthreads();
        if (hit) {
          const long long o = next[pass] + warp_base[warp] + __popc(ballot & ((1u << lane) - 1u));
          if (pass == Q)
            cells[o] = (int)cell;
          else
            links[o] = make_int2((int)cell, pass | (types[pass] << 8));
        }
        __syncthreads();  // every thread has read warp_base and next[pass]
        if (threadIdx.x == 0) next[pass] += round_total;
      }
      __syncthreads();
    }
  }
}

long long bnd_list_blocks(long long n) { return (n + LIST_BLOCK * LIST_SUB - 1) / (LIST_BLOCK * LIST_SUB); }

static Pred make_pred(const int* face, bool x_in, bool x_out) {
  Pred pr;
  pr.x_in = x_in ? 1 : 0;
  pr.x_out = x_out ? 1 : 0;
  for (int f = 0; f < 6; ++f) pr.face[f] = face ? face[f] : 0;
  return pr;
}

static long long pred_grid(long long nchunks) { return nchunks < 152LL * 16 ? nchunks : 152LL * 16; }

int launch_pred_count(int Q, const int* face, bool x_in, bool x_out, const uint8_t* flags, int nx, int ny, int nz,
                      int* counts, void* stream) {
  const long long n = (long long)nx * ny * nz;
  const long long nc = bnd_list_blocks(n);
  if (nc < 1) return 0;
  const Pred pr = make_pred(face, x_in, x_out);
  const unsigned g = (unsigned)pred_grid(nc);
  cudaStream_t s = (cudaStream_t)stream;
  if (Q == 9)
    k_pred_count<9><<<g, LIST_BLOCK, 0, s>>>(flags, n, nx, ny, nz, pr, nc, counts);
  else if (Q == 19)
    k_pred_count<19><<<g, LIST_BLOCK, 0, s>>>(flags, n, nx, ny, nz, pr, nc, counts);
  else if (Q == 27)
    k_pred_count<27><<<g, LIST_BLOCK, 0, s>>>(flags, n, nx, ny, nz, pr, nc, counts);
  else
    return -1;
  return 0;
}

int launch_pred_write(int Q, const int* face, bool x_in, bool x_out, const uint8_t* flags, int nx, int ny, int nz,
                      const long long* offs, int2* links, int* cells, void* stream) {
  const long long n = (long long)nx * ny * nz;
  const long long nc = bnd_list_blocks(n);
  if (nc < 1) return 0;
  const Pred pr = make_pred(face, x_in, x_out);
  const unsigned g = (unsigned)pred_grid(nc);
  cudaStream_t s = (cudaStream_t)stream;
  if (Q == 9)
    k_pred_write<9><<<g, LIST_BLOCK, 0, s>>>(flags, n, nx, ny, nz, pr, nc, offs, links, cells);
  else if (Q == 19)
    k_pred_write<19><<<g, LIST_BLOCK, 0, s>>>(flags, n, nx, ny, nz, pr, nc, offs, links, cells);
  else if (Q == 27)
    k_pred_write<27><<<g, LIST_BLOCK, 0, s>>>(flags, n, nx, ny, nz, pr, nc, offs, links, cells);
  else
    return -1;
  return 0;
}

template <int Q>
__global__ void k_link_cells(const int2* __restrict__ links, long long n, const uint8_t* __restrict__ flags,
                             int nx, int ny, int nz, int2* __restrict__ cells) {
  const bool small = (long long)nx * ny * nz < 0x7fffffffLL;
  for (long long e = blockIdx.x * 256LL + threadIdx.x; e < n; e += (long long)gridDim.x * 256) {
    const int2 l = links[e];
    const int i = l.y & 0xff;
    int cx = 0, cy = 0, cz = 0;
#pragma unroll
    for (int j = 1; j < Q; ++j)
      if (j == i) {
        cx = Lattice<Q>::c(j, 0);
        cy = Lattice<Q>::c(j, 1);
        cz = Lattice<Q>::c(j, 2);
      }
    int x, y, z;
    cell_xyz(l.x, nx, ny, small, x, y, z);
    auto wrap = [](int v, int m) { return v < 0 ? m - 1 : (v >= m ? 0 : v); };
    const int w = wrap(x - cx, nx) + nx * (wrap(y - cy, ny) + ny * wrap(z - cz, nz));
    const int b = wrap(x + cx, nx) + nx * (wrap(y + cy, ny) + ny * wrap(z + cz, nz));
    cells[e] = make_int2(w, (flags[b] & FLAG_TYPE) == FLUID ? b : -1);
  }
}

__global__ void k_links_off_x(const int2* __restrict__ cells, long long n, int nx, bool face0, bool face1, int* flag) {
  bool off = false;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x) {
    const int x = cells[e].x % nx;
    off |= !((face0 && x == 0) || (face1 && x == nx - 1));
  }
  if (__syncthreads_or(off) && threadIdx.x == 0) atomicExch(flag, 1);
}

int launch_links_off_x(const int2* cells, long long n, int nx, bool face0, bool face1, int* flag, void* stream) {
  const long long b = (n + 255) / 256;
  k_links_off_x<<<(unsigned)(b < 152 * 8 ? b : 152 * 8), 256, 0, (cudaStream_t)stream>>>(cells, n, nx, face0, face1,
                                                                                       flag);
  return 0;
}

__global__ void k_number_cells(const int* __restrict__ cells, int n, int* __restrict__ number) {
  const int k = blockIdx.x * 256 + threadIdx.x;
  if (k < n) number[cells[k]] = k + 1;
}

void launch_number_cells(const int* cells, int n, int* number, void* stream) {
  if (n > 0) k_number_cells<<<(unsigned)((n + 255) / 256), 256, 0, (cudaStream_t)stream>>>(cells, n, number);
}

template <typename T>
__global__ void k_clear_walls(T* __restrict__ f, const uint8_t* __restrict__ flags, int Q, long long n,
                              long long plane) {
  for (long long cell = blockIdx.x * 256LL + threadIdx.x; cell < n; cell += (long long)gridDim.x * 256)
    if ((flags[cell] & FLAG_TYPE) == WALL)
      for (int i = 0; i < Q; ++i) f[i * plane + cell] = T(0);
}

int launch_clear_walls(void* f, int esize, const uint8_t* flags, int Q, long long n, long long plane, void* stream) {
  const long long b = (n + 255) / 256;
  const unsigned grid = (unsigned)(b < 152 * 32 ? b : 152 * 32);
  cudaStream_t s = (cudaStream_t)stream;
  if (esize == 4)
    k_clear_walls<<<grid, 256, 0, s>>>((uint32_t*)f, flags, Q, n, plane);
  else if (esize == 2)
    k_clear_walls<<<grid, 256, 0, s>>>((uint16_t*)f, flags, Q, n, plane);
  else
    return -1;
  return 0;
}

int launch_link_cells(int Q, const int2* links, long long n, const uint8_t* flags, int nx, int ny, int nz,
                      int2* cells, void* stream) {
  if (n <= 0) return 0;
  long long blocks = (n + 255) / 256;
  if (blocks > 152LL * 32) blocks = 152LL * 32;
  cudaStream_t s = (cudaStream_t)stream;
  if (Q == 9)
    k_link_cells<9><<<(unsigned)blocks, 256, 0, s>>>(links, n, flags, nx, ny, nz, cells);
  else if (Q == 19)
    k_link_cells<19><<<(unsigned)blocks, 256, 0, s>>>(links, n, flags, nx, ny, nz, cells);
  else if (Q == 27)
    k_link_cells<27><<<(unsigned)blocks, 256, 0, s>>>(links, n, flags, nx, ny, nz, cells);
  else
    return -1;
  return 0;
}

// The six boundary planes of a mask in one compact buffer: plane f (axis
// f / 2 at 0 or n - 1) holds its cells at a + n1 * b, (a, b) the coordinates
// on axes (f / 2 + 1) % 3 and (f / 2 + 2) % 3; axes of extent 1 have none.
__global__ void k_extract_planes(const uint8_t* __restrict__ mask, int nx, int ny, int nz, uint8_t* __restrict__ out) {
  const long long ext[3] = {nx, ny, nz};
  long long off = 0;
  for (int f = 0; f < 6; ++f) {
    const int ax = f / 2;
    if (ext[ax] < 2) continue;
    const long long n1 = ext[(ax + 1) % 3], n2 = ext[(ax + 2) % 3], pos = (f % 2) ? ext[ax] - 1 : 0;
    for (long long k = blockIdx.x * 256LL + threadIdx.x; k < n1 * n2; k += (long long)gridDim.x * 256) {
      long long q[3];
      q[ax] = pos;
      q[(ax + 1) % 3] = k % n1;
      q[(ax + 2) % 3] = k / n1;
      out[off + k] = mask[q[0] + nx * (q[1] + (long long)ny * q[2])];
    }
    off += n1 * n2;
  }
}

int launch_extract_planes(const uint8_t* mask, int nx, int ny, int nz, uint8_t* out, void* stream) {
  const long long big = (long long)(nx > ny ? nx : ny) * (ny > nz ? ny : nz) * 2;
  long long blocks = (big + 255) / 256;
  if (blocks > 152LL * 8) blocks = 152LL * 8;
  if (blocks < 1) blocks = 1;
  k_extract_planes<<<(unsigned)blocks, 256, 0, (cudaStream_t)stream>>>(mask, nx, ny, nz, out);
  return 0;
}

// n floats from src to dst (either may be mapped host memory), 16 bytes per
// access where both are 16-byte aligned.
__global__ void k_copy_f32(const float* __restrict__ src, float* __restrict__ dst, long long n) {
  const long long stride = (long long)gridDim.x * blockDim.x;
  const long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if ((((uintptr_t)src | (uintptr_t)dst) & 15) == 0) {
    const long long n4 = n / 4;
    for (long long k = t; k < n4; k += stride)
      reinterpret_cast<float4*>(dst)[k] = reinterpret_cast<const float4*>(src)[k];
    for (long long k = 4 * n4 + t; k < n; k += stride) dst[k] = src[k];
  } else {
    for (long long k = t; k < n; k += stride) dst[k] = src[k];
  }
}

int launch_copy_f32(const float* src, float* dst, long long n, void* stream) {
  if (n <= 0) return 0;
  long long blocks = (n / 4 + 255) / 256;
  if (blocks > 152LL * 8) blocks = 152LL * 8;
  if (blocks < 1) blocks = 1;
  k_copy_f32<<<(unsigned)blocks, 256, 0, (cudaStream_t)stream>>>(src, dst, n);
  return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

// Sums n rows of 4 doubles in a fixed order (deterministic): each thread
// strides over rows, then a fixed shared-memory tree.
__global__ void k_reduce_final(const double* __restrict__ partial, long long n, double* out) {
  __shared__ double s[4][256];
  double a[4] = {0.0, 0.0, 0.0, 0.0};
  for (long long r = threadIdx.x; r < n; r += blockDim.x)
#pragma unroll
    for (int k = 0; k < 4; ++k) a[k] += partial[4 * r + k];
#pragma unroll
  for (int k = 0; k < 4; ++k) s[k][threadIdx.x] = a[k];
  __syncthreads();
  for (int w = 128; w > 0; w >>= 1) {
    if ((int)threadIdx.x < w)
#pragma unroll
      for (int k = 0; k < 4; ++k) s[k][threadIdx.x] += s[k][threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x < 4) out[threadIdx.x] = s[threadIdx.x][0];
}

// FP64 sum of squares of n floats (the gradient norm of the differentiable
// workloads); grid-stride, one row (sum, 0, 0, 0) per block.
__global__ void k_sum_squares_partial(const float* __restrict__ x, long long n, double* partial) {
  double acc = 0.0;
  for (long long k = blockIdx.x * 256LL + threadIdx.x; k < n; k += (long long)gridDim.x * 256) {
    const double v = x[k];
    acc += v * v;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
  __shared__ double red[8];
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    double s = 0.0;
    for (int q = 0; q < 8; ++q) s += red[q];
    partial[4 * (long long)blockIdx.x] = s;
    partial[4 * (long long)blockIdx.x + 1] = 0.0;
    partial[4 * (long long)blockIdx.x + 2] = 0.0;
    partial[4 * (long long)blockIdx.x + 3] = 0.0;
  }
}

long long launch_sum_squares(const float* x, long long n, double* partial, long long capacity, void* stream) {
  long long b = (n + 2047) / 2048;
  if (b > capacity) b = capacity;
  if (b > 65535) b = 65535;
  if (b < 1) b = 1;
  k_sum_squares_partial<<<(unsigned)b, 256, 0, (cudaStream_t)stream>>>(x, n, partial);
  return b;
}

int launch_reduce_final(const double* partial, long long n, double* out, void* stream) {
  k_reduce_final<<<1, 256, 0, (cudaStream_t)stream>>>(partial, n, out);
  return 0;
}

}  // namespace xlb
