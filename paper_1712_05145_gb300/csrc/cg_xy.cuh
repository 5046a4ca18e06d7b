// Row transforms of the FP32 CG iteration in Fourier space (cg_plane.cu, cg_rows.cu): packed
// complex-to-real and real-to-complex transforms of length H = n1 / 2, in place in shared memory.
//
// H = R1 R2.  A row's half spectrum X[0..H-1] (slot 0: X[0] + i X[H]) lies in natural order.
//  1. One task takes butterflies j and R2 - j of the first radix-R1 stage, k = j + r R2.  These hold k
//     and H - k together, so the merge of the half spectrum into the packed row's spectrum happens in
//     registers in front of the stage.
//  2. The radix-R2 stage over block b ends the inverse: z[n] = x[2n] + i x[2n+1], n = b + R1 s.  The
//     material law multiplies it and the forward radix-R2 stage over the same values follows at once.
//  3. The radix-R1 stage ends the forward transform, and the task pairs (j, R2 - j) hold k and H - k
//     again for the split.
// Every stage writes the positions it read, so one barrier separates two stages.
#pragma once
#include "ls_common.cuh"

namespace hom {

// R1 (pairs of radix-R1 butterflies per task) and R2 (1 or even) per row length
template <int H> struct RowPlan;
#define HOM_ROWPLAN(H_, A_, B_) \
  template <> struct RowPlan<H_> { static constexpr int R1 = A_, R2 = B_; };
HOM_ROWPLAN(2, 2, 1)
HOM_ROWPLAN(3, 3, 1)
HOM_ROWPLAN(4, 4, 1)
HOM_ROWPLAN(6, 6, 1)
HOM_ROWPLAN(8, 8, 1)
HOM_ROWPLAN(12, 6, 2)
HOM_ROWPLAN(16, 4, 4)
HOM_ROWPLAN(24, 6, 4)
HOM_ROWPLAN(32, 8, 4)
HOM_ROWPLAN(48, 6, 8)
HOM_ROWPLAN(64, 8, 8)
HOM_ROWPLAN(96, 8, 12)
HOM_ROWPLAN(128, 8, 16)
HOM_ROWPLAN(192, 8, 24)
HOM_ROWPLAN(256, 8, 32)
HOM_ROWPLAN(384, 12, 32)
HOM_ROWPLAN(512, 16, 32)
#undef HOM_ROWPLAN

template <int H> __host__ __device__ constexpr int row_pair_tasks() { return RowPlan<H>::R2 == 1 ? 1 : RowPlan<H>::R2 / 2; }

// X[k], X[H-k] -> Z[k], Z[H-k] of the packed row: s = X[k] + conj X[H-k], t = i W^-k (X[k] - conj X[H-k]),
// Z[k] = s + t, Z[H-k] = conj(s - t), W = exp(-2 pi i / n1) (the factor of H - k is minus the conjugate)
__device__ __forceinline__ void merge_pair(cx<float>& xk, cx<float>& xm, cx<float> wk) {
  const cx<float> s = xk + conj(xm), t = mul_i<float, 1>(cmul(conj(wk), xk - conj(xm)));
  xk = s + t;
  xm = conj(s - t);
}
// the reverse, times 2: X[k], X[H-k] from Z[k], Z[H-k]
__device__ __forceinline__ void split_pair(cx<float>& zk, cx<float>& zm, cx<float> wk) {
  const cx<float> s = zk + conj(zm), t = mul_i<float, -1>(cmul(wk, zk - conj(zm)));
  zk = s + t;
  zm = conj(s - t);
}

template <int R1, int R2, int DIR>
__device__ __forceinline__ void row_twiddle(cx<float> (&v)[R1], int j, const cx<float>* twh) {
  if constexpr (R2 > 1) {
#pragma unroll
    for (int r = 1; r < R1; ++r) {
      cx<float> w = twh[j * r];
      if (DIR > 0) w.im = -w.im;
      v[r] = cmul(v[r], w);
    }
  }
}

// pair task jp in [0, row_pair_tasks): merges and runs stage 1 of the inverse on A (butterfly j) and B
// (butterfly R2 - j; the self-paired R2 / 2 beside j = 0)
template <int H>
__device__ __forceinline__ void merge_and_stage(cx<float> (&A)[RowPlan<H>::R1], cx<float> (&B)[RowPlan<H>::R1], int jp,
                                                const cx<float>* tw1) {
  constexpr int R1 = RowPlan<H>::R1, R2 = RowPlan<H>::R2;
  if (jp == 0) {
    const float x0 = A[0].re, xn = A[0].im;
    A[0] = mk<float>(x0 + xn, x0 - xn);
#pragma unroll
    for (int r = 1; r <= R1 / 2; ++r) {
      if (2 * r == R1) A[r] = conj(A[r]) * 2.0f;
      else merge_pair(A[r], A[R1 - r], tw1[r * R2]);
    }
    if constexpr (R2 > 1) {
#pragma unroll
      for (int r = 0; r < (R1 + 1) / 2; ++r) {
        if (2 * r == R1 - 1) B[r] = conj(B[r]) * 2.0f;
        else merge_pair(B[r], B[R1 - 1 - r], tw1[R2 / 2 + r * R2]);
      }
    }
  } else {
#pragma unroll
    for (int r = 0; r < R1; ++r) merge_pair(A[r], B[R1 - 1 - r], tw1[jp + r * R2]);
  }
  SmallDFT<float, R1, +1>::run(A);
  if constexpr (R2 > 1) SmallDFT<float, R1, +1>::run(B);
}

// the forward counterpart: the last radix-R1 stage and the split (times 2)
template <int H>
__device__ __forceinline__ void stage_and_split(cx<float> (&A)[RowPlan<H>::R1], cx<float> (&B)[RowPlan<H>::R1], int jp,
                                                const cx<float>* tw1) {
  constexpr int R1 = RowPlan<H>::R1, R2 = RowPlan<H>::R2;
  SmallDFT<float, R1, -1>::run(A);
  if constexpr (R2 > 1) SmallDFT<float, R1, -1>::run(B);
  if (jp == 0) {
    const cx<float> z0 = A[0];
    A[0] = mk<float>(2.0f * (z0.re + z0.im), 2.0f * (z0.re - z0.im));
#pragma unroll
    for (int r = 1; r <= R1 / 2; ++r) {
      if (2 * r == R1) A[r] = conj(A[r]) * 2.0f;
      else split_pair(A[r], A[R1 - r], tw1[r * R2]);
    }
    if constexpr (R2 > 1) {
#pragma unroll
      for (int r = 0; r < (R1 + 1) / 2; ++r) {
        if (2 * r == R1 - 1) B[r] = conj(B[r]) * 2.0f;
        else split_pair(B[r], B[R1 - 1 - r], tw1[R2 / 2 + r * R2]);
      }
    }
  } else {
#pragma unroll
    for (int r = 0; r < R1; ++r) split_pair(A[r], B[R1 - 1 - r], tw1[jp + r * R2]);
  }
}

}  // namespace hom
