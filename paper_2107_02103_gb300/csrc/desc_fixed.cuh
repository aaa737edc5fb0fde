// The descriptor's contractions (Sec. II: D = S (S^<)^T and its backward) in fixed point (fixed.cuh), for
// f64 arrays: an atom's T, and its dE/dD, as two-limb integers against the atom's largest element, the
// products on the integer pipes, one conversion per element on the FP64 pipe.  Shared by descriptor.cu and
// the tensor-core forward's finish, so that both give D the same bits.
#pragma once

#include "fixed.cuh"

namespace dpc {
namespace {
namespace dfx {

// Binary places sh with |x| 2^sh < 2^places over the values whose largest high word (sign off) is hw, and
// `wild` where the sums are left to the FP64 pipe: an inf or NaN, or values so large or small that results
// could leave the normal range.  Zeros only: places 0.
__device__ __forceinline__ int places_of(int hw, int places, bool &wild) {
  const int eb = hw >> 20;
  wild |= hw != 0 && (eb < 650 || eb > 1400);
  return hw ? places + 1022 - eb : 0;
}

// The largest high word, sign off, of x[0 .. n) in shared memory: each warp by itself.
__device__ __forceinline__ int max_hiword(const double *x, int n, int lane) {
  int m = 0;
  for (int e = lane; e < n; e += 32) m = max(m, __double2hiint(x[e]) & 0x7fffffff);
  return __reduce_max_sync(0xffffffffu, m);
}

// D's products of 59 places each, in limbs of 30 bits: four of them stay below 2^61 (hi) and 2^63 (mid).
constexpr int kDescPlaces = 59, kDescLimb = 30;

// One atom's D [M1][M2] by the threads of a block, from its T in Ts [4][M1] (written and synchronised), with
// room for as many fixed points after it.  Consecutive threads take consecutive elements, M2 to a row.
// Why fixed point: four FP64 instructions an element, 272 sub-partition clocks of that pipe a warp, bound
// the kernels; one conversion takes it 64 and the 12 limb products the integer pipes 29.  Measured, the
// forward's finish: copper (4,096 atoms x 100 x 16) 0.053 -> 0.033 ms, water (12,288) 0.142 -> 0.076 ms.
__device__ __forceinline__ void desc_tile(const double *Ts, int M1, int M2, double *__restrict__ D) {
  bool wild = false;
  const int sh = places_of(max_hiword(Ts, 4 * M1, threadIdx.x & 31), kDescPlaces, wild);
  // a thread keeps its column n and takes every step-th row (a block's rows lie back to back; M2 above the
  // block: several columns a thread)
  const int cols = min(M2, (int)blockDim.x), step = (int)blockDim.x / cols;
  const int m0 = (int)threadIdx.x / cols, n0 = (int)threadIdx.x - m0 * cols;
  if (!wild) {  // uniform over the block
    fx::Fix *Tf = reinterpret_cast<fx::Fix *>(const_cast<double *>(Ts) + 4 * M1);
    for (int e = threadIdx.x; e < 4 * M1; e += blockDim.x) Tf[e] = fx::limbs<kDescLimb>(fx::from_double(Ts[e], sh));
    __syncthreads();
    const int ex = 2 * kDescLimb - 2 * sh;
    if (m0 < step)
      for (int n = n0; n < M2; n += cols) {
        const fx::Fix b0 = Tf[n], b1 = Tf[M1 + n], b2 = Tf[2 * M1 + n], b3 = Tf[3 * M1 + n];
#pragma unroll 2
        for (int m = m0; m < M1; m += step) {
          fx::Acc p;
          p.mad(Tf[m], b0);
          p.mad(Tf[M1 + m], b1);
          p.mad(Tf[2 * M1 + m], b2);
          p.mad(Tf[3 * M1 + m], b3);
          D[m * M2 + n] = fx::to_double(fx::over_unit<kDescLimb>(p), ex);
        }
      }
  } else if (m0 < step) {
    for (int n = n0; n < M2; n += cols)
      for (int m = m0; m < M1; m += step) {
        double v = Ts[m] * Ts[n];
#pragma unroll
        for (int k = 1; k < 4; ++k) v = fma(Ts[k * M1 + m], Ts[k * M1 + n], v);
        D[m * M2 + n] = v;
      }
  }
}

}  // namespace dfx
}  // namespace
}  // namespace dpc
