// Host interface of the resident D2Q9 kernel (resident2d.cu): a domain whose
// populations fit the shared memory of one thread-block cluster advances any
// number of updates in one launch.
#pragma once
#include <stdint.h>

namespace xlb {

// One D2Q9 domain of a batch (and the single domain of a small lattice).
struct BatchDom {
  long long off;   // element offset of the domain's populations in each buffer
  long long foff;  // offset of its flag bytes
  int nx, ny;
  int plane;       // elements between population planes (nx * ny rounded up to 64)
  float Fx, Fy;
};

// Launch shape of a resident domain: `ctas` thread blocks (one cluster) of
// `threads` threads share its rows.  ctas = 0: the domain does not fit.
struct ResidentShape {
  int ctas, threads;
  long long smem;  // dynamic shared memory per block
  bool one;        // one cell per thread
};

// Shape for an nx x ny domain: alone on the GPU (spread wide and with one cell
// per thread, so that the domain finishes early) or one of many (packed, so that
// all of them do).
ResidentShape resident2d_shape(int storage, int coll, int nx, int ny, bool alone);

// Clusters of that shape the GPU holds at once (0: it cannot launch one).
int resident2d_clusters(const ResidentShape& shape, int storage, int coll);

struct ResidentArgs {
  const void* src;        // post-collision populations (stored deviations)
  void* dst;              // the same after `steps` updates (may be src)
  const uint8_t* flags;   // flag byte per cell (FLUID and WALL only), or null: all FLUID
  const BatchDom* doms;   // device array, or null: `dom` below
  const int* order;       // device array: cluster k advances doms[order[k]] (with doms)
  BatchDom dom;
  int n_dom;
  int storage, coll;
  float omega;
  int steps;              // >= 1
  ResidentShape shape;
  void* stream;
};

// 0 on a successful launch request, else a negative code.
int launch_resident2d(const ResidentArgs& a);
// The same launch as a node of a graph (cudaGraph_t).
int add_resident2d_node(const ResidentArgs& a, void* graph);

}  // namespace xlb
