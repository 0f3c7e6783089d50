// Newton + preconditioned conjugate residual (PCR) substep solve on the GPU: the paper's
// own solver structure (Sec. IV-D) over the bilateral rows (stretch, yaw, pitch) of
// contact-free substeps, as an alternative to the Jacobi relaxation.
//
// Each Newton step linearises the rows at x = x_s + d and solves the Schur system of
// Eq. 8, (J M^-1 J^T + alpha~) dlambda = -(c + alpha~ lambda), with `pcr_iters`
// conjugate residual iterations preconditioned by its diagonal (the Jacobi denominators),
// then lambda += dlambda and d += M^-1 J^T dlambda.  Matrix-vector products are counted
// (one per PCR iteration, one per Newton step), like the update count of the Jacobi path.
//
// Layout: the lane group of a snake keeps its multipliers, the Newton increment, the CR search
// directions and the gradients of its nodes' segments (those before and after each node) in
// registers; what crosses a lane boundary (the multiplied vector's entries of the rows next
// door, M^-1 J^T of it at the nodes next door) moves by warp shuffles, eleven per product.
// What bounds it: the serial chain of products of a snake (its two reductions and shuffles
// in line) at few warps per scheduler.  Measured, 4096 uneven snakes in free fall to 1e-4:
// 2.68 ms per env-step with the gradients and vectors exchanged through shared memory (47
// loads per node and product), 1.48 ms now; same bits.
#pragma once

#include "internal.h"

namespace snakesim {

template <int G>
__device__ __forceinline__ float group_sum(float v) {
#pragma unroll
  for (int off = G / 2; off >= 1; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off, G);
  return v;
}

// Segment i -> i+1: n (3), heading gradient (2), elevation gradient (3); zero where there is
// no segment.
struct PcrSeg {
  float g[8];
  __device__ __forceinline__ float operator[](int c) const { return g[c]; }
};

// u_i = w_i (J^T v)_i for the NPL nodes of this lane; sg[j] is the segment before node j,
// sg[j + 1] the one after it; v[j][r] are this lane's entries (0 on rows that do not exist).
template <int NPL, int G>
__device__ __forceinline__ void pcr_jt(const SnakeK& S, const PcrSeg (&sg)[NPL + 1], int q, bool valid,
                                       const float (&v)[NPL][3], float (&u)[NPL][3]) {
  float vl[3], vr[3];
#pragma unroll
  for (int r = 0; r < 3; ++r) vl[r] = __shfl_up_sync(0xffffffffu, v[NPL - 1][r], 1, G);
#pragma unroll
  for (int r = 1; r < 3; ++r) vr[r] = __shfl_down_sync(0xffffffffu, v[0][r], 1, G);
#pragma unroll
  for (int j = 0; j < NPL; ++j) {
    const int i = q * NPL + j;
    const PcrSeg &A = sg[j], &B = sg[j + 1];
    float a0 = 0.f, a1 = 0.f, a2 = 0.f;
    if (valid && i < S.N && i >= S.nfix) {
      if (i >= 1) {  // stretch(i-1): +n_{i-1}; yaw/pitch(i-1): + segment i-1 gradients
        const float vs = j > 0 ? v[j > 0 ? j - 1 : 0][0] : vl[0], vy = j > 0 ? v[j > 0 ? j - 1 : 0][1] : vl[1],
                    vp = j > 0 ? v[j > 0 ? j - 1 : 0][2] : vl[2];
        a0 += A[0] * vs + A[3] * vy + A[5] * vp;
        a1 += A[1] * vs + A[4] * vy + A[6] * vp;
        a2 += A[2] * vs + A[7] * vp;
      }
      {  // rows of node i: stretch -n_i; yaw / pitch -(g_{i-1} + g_i)
        const float vs = v[j][0], vy = v[j][1], vp = v[j][2];
        float gy0 = 0.f, gy1 = 0.f, gp0 = 0.f, gp1 = 0.f, gp2 = 0.f;
        if (i >= 1) { gy0 = A[3]; gy1 = A[4]; gp0 = A[5]; gp1 = A[6]; gp2 = A[7]; }
        gy0 += B[3]; gy1 += B[4]; gp0 += B[5]; gp1 += B[6]; gp2 += B[7];
        a0 -= B[0] * vs + gy0 * vy + gp0 * vp;
        a1 -= B[1] * vs + gy1 * vy + gp1 * vp;
        a2 -= B[2] * vs + gp2 * vp;
      }
      if (i + 1 <= S.N - 1) {  // yaw/pitch(i+1): + segment i gradients
        const float vy = j + 1 < NPL ? v[j + 1 < NPL ? j + 1 : 0][1] : vr[1],
                    vp = j + 1 < NPL ? v[j + 1 < NPL ? j + 1 : 0][2] : vr[2];
        a0 += B[3] * vy + B[5] * vp;
        a1 += B[4] * vy + B[6] * vp;
        a2 += B[7] * vp;
      }
    }
    u[j][0] = S.inv_m * a0; u[j][1] = S.inv_m * a1; u[j][2] = S.inv_m * a2;
  }
}

// y = (J M^-1 J^T + alpha~) v on the rows of this lane's nodes; act[j][r] is non-zero on the
// rows that take part.
template <int NPL, int G>
__device__ __forceinline__ void pcr_matvec(const SnakeK& S, const PcrSeg (&sg)[NPL + 1], int q, bool valid,
                                           const float (&act)[NPL][3], const float (&v)[NPL][3], float (&y)[NPL][3]) {
  float u[NPL][3], ul[3], ur[3];
  pcr_jt<NPL, G>(S, sg, q, valid, v, u);
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    ul[d] = __shfl_up_sync(0xffffffffu, u[NPL - 1][d], 1, G);
    ur[d] = __shfl_down_sync(0xffffffffu, u[0][d], 1, G);
  }
#pragma unroll
  for (int j = 0; j < NPL; ++j) {
    const int i = q * NPL + j;
    const PcrSeg &A = sg[j], &B = sg[j + 1];
    const float* L = j > 0 ? u[j > 0 ? j - 1 : 0] : ul;
    const float* R = j + 1 < NPL ? u[j + 1 < NPL ? j + 1 : 0] : ur;
    y[j][0] = y[j][1] = y[j][2] = 0.f;
    if (!(valid && i < S.N)) continue;
    const float ux = u[j][0], uy = u[j][1], uz = u[j][2];
    if (act[j][0] != 0.f) {  // stretch(i): n_i . (u_{i+1} - u_i)
      y[j][0] = B[0] * (R[0] - ux) + B[1] * (R[1] - uy) + B[2] * (R[2] - uz) + S.at_s * v[j][0];
    }
    if (act[j][1] != 0.f || act[j][2] != 0.f) {  // yaw / pitch(i): g_{i-1} . (u_{i-1} - u_i) + g_i . (u_{i+1} - u_i)
      const float lx = L[0] - ux, ly = L[1] - uy, lz = L[2] - uz;
      const float rx = R[0] - ux, ry = R[1] - uy, rz = R[2] - uz;
      if (act[j][1] != 0.f) y[j][1] = A[3] * lx + A[4] * ly + B[3] * rx + B[4] * ry + S.at_b * v[j][1];
      if (act[j][2] != 0.f)
        y[j][2] = A[5] * lx + A[6] * ly + A[7] * lz + B[5] * rx + B[6] * ry + B[7] * rz + S.at_b * v[j][2];
    }
  }
}

}  // namespace snakesim
