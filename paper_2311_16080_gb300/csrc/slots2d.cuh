// Shared-memory population slots of the D2Q9 kernels that keep cells on the SM
// for several updates (resident2d.cu, tile2d.cu): one buffer, in place (the swap
// of two directions per update that Bailey et al. 2009 call the AA pattern).
// Slot A[x][i] holds h_i(x) before an odd update.  With L_j(x) = A[x][j] where
// x + c_j is a WALL cell and A[x + c_j][opp(j)] elsewhere:
//   odd update:  f_opp(j)(x) is in L_j(x) (streamed, or bounced back from the
//                wall); after the collision h_j(x) goes to L_j(x);
//   even update: f_i(x) is then in A[x][opp(i)] and h_i(x) goes to A[x][i].
// Every slot is read and written by one thread per update, so one barrier
// per update is enough, and the even ones touch nothing but the own cell.
//
// A cell is 9 consecutive slots: with FP32 a stride of 9 words, which reaches
// every bank once per warp, and the direction is an immediate offset, so a
// neighbour costs one addition whatever the domain's size.  16-bit slots
// take a stride of 10 (5 words, again every bank once), the tenth being the
// cell's meta word.
#pragma once
#include <cuda_runtime.h>

#include "lbm_device.cuh"

namespace xlb {

template <typename S>
struct Slots {
  static constexpr int STRIDE = sizeof(S) == 4 ? 9 : 10;  // slots per cell
  static constexpr int CELL = STRIDE * (int)sizeof(S);    // bytes per cell
};

// slot access by 32-bit shared address; REMOTE: the address may lie in
// another block of the cluster
template <typename S, bool REMOTE>
__device__ __forceinline__ float slot_ld(uint32_t a) {
  if constexpr (sizeof(S) == 4) {
    float v;
    if (REMOTE)
      asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(a) : "memory");
    else
      asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(a) : "memory");
    return v;
  } else {
    unsigned short u;
    if (REMOTE)
      asm volatile("ld.shared::cluster.u16 %0, [%1];" : "=h"(u) : "r"(a) : "memory");
    else
      asm volatile("ld.shared.u16 %0, [%1];" : "=h"(u) : "r"(a) : "memory");
    S s;
    memcpy(&s, &u, 2);
    return Store<S>::ld_plain(&s);
  }
}

template <typename S, bool REMOTE>
__device__ __forceinline__ void slot_st(uint32_t a, const CellRound<S>& rnd, int i, float v) {
  if constexpr (sizeof(S) == 4) {
    if (REMOTE)
      asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory");
    else
      asm volatile("st.shared.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory");
  } else {
    const unsigned short u = rnd.bits(i, v);
    if (REMOTE)
      asm volatile("st.shared::cluster.u16 [%0], %1;" ::"r"(a), "h"(u) : "memory");
    else
      asm volatile("st.shared.u16 [%0], %1;" ::"r"(a), "h"(u) : "memory");
  }
}

}  // namespace xlb
