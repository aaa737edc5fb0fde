// The descriptor's contractions (Sec. II: D = S (S^<)^T and its backward) in fixed point (fixed.cuh), for
// f64 arrays: an atom's T, and its dE/dD, as two-limb integers against powers of two, the products on the
// integer pipes, one conversion per element on the FP64 pipe.  Shared by descriptor.cu and
// the tensor-core forward's finish, so that both give D the same bits.
#pragma once

#include "fixed.cuh"

namespace dpc {
namespace {
namespace dfx {

// A channel of an atom's T as fixed points against the largest of its four elements, in 60 places and limbs of
// 30 bits (four products: hi below 2^62, mid below 2^63), with their magnitudes as floats in units of 2^30.
struct alignas(16) Channel {
  fx::Fix f[4];
  float a[4];
  int sh, pad[7];  // 80 bytes: neither the threads' stores nor their loads of a column meet in a bank
};
constexpr int kDescPlaces = 60, kDescLimb = 30;
// The fixed-point sum of an element is off by at most 5.5 units: half a unit from either factor of each term, a
// quarter from each dropped product of low limbs, half from the rounding.  From this sum of magnitudes on, that is
// below 3 2^-53 of it, and with the rounding to f64 below the 4 2^-53 of four FP64 operations.
constexpr float kDescLeast = 0x1.d8p53f;
// Where D in fixed point pays: the channels' preparation (four conversions each, and 80 bytes of shared memory) has to
// be earned by their M2 elements.  Measured with 20,000 atoms, fixed over FP64 (a warp per atom): 16 x 8 1.01, 32 x 4
// 1.02, 24 x 6 0.92, 48 x 4 0.93, 100 x 3 1.03, 400 x 4 0.88; and above 512 channels, two or three blocks an SM, 600 x 6
// 1.09, 600 x 12 0.72, 800 x 12 1.12, 800 x 16 0.97.
__host__ __device__ constexpr bool desc_fixed_pays(int M1, int M2) {
  return M2 >= 4 && M1 * M2 >= 144 && (M1 <= 512 || 50 * M2 >= M1);
}
// Shared memory of desc_tile: T [4][M1] and the channels.
__host__ __device__ constexpr size_t desc_tile_bytes(int M1, int M2) {
  return (size_t)M1 * (4 * sizeof(double) + (desc_fixed_pays(M1, M2) ? sizeof(Channel) : 0));
}
// The element in FP64, in the order of descriptor_kernel.
__device__ __forceinline__ double desc_fp64(const double *Ts, int M1, int m, int n) {
  double v = Ts[m] * Ts[n];
#pragma unroll
  for (int k = 1; k < 4; ++k) v = fma(Ts[k * M1 + m], Ts[k * M1 + n], v);
  return v;
}

// One atom's D [M1][M2] by the threads of a block, from its T in Ts [4][M1] (written and synchronised), with
// room for the channels after it.  Consecutive threads take consecutive elements, M2 to a row.
// Why fixed point: four FP64 instructions an element, 272 sub-partition clocks of that pipe a warp, bound
// the kernels; one conversion takes it 64 and the 12 limb products the integer pipes 29.
// Why an exponent a channel: channels differ in size, and D[m][n] is to be as exact against its own terms as
// an FP64 sum (one exponent an atom lost 2^20 of an element whose channels were 2^-10 of the largest; an exponent
// a channel and the test below cost D by itself 59.7 -> 65.8 us, 12,288 atoms x 100 x 16).  Where its two channels
// have their large elements in different k the sum is far below the product of the two exponents; four FP32
// multiply-adds tell, and such an element (like those of a channel with an inf or NaN, or out of the exponents'
// range) is left to the FP64 pipe.
__device__ __forceinline__ void desc_tile(const double *Ts, int M1, int M2, double *__restrict__ D) {
  if (!desc_fixed_pays(M1, M2)) {  // uniform
    const int total = M1 * M2, dm = (int)blockDim.x / M2, dn = (int)blockDim.x - dm * M2;
    int m = (int)threadIdx.x / M2, n = (int)threadIdx.x - m * M2;
#pragma unroll 1
    for (int e = threadIdx.x; e < total; e += blockDim.x) {
      D[e] = desc_fp64(Ts, M1, m, n);
      m += dm, n += dn;
      if (n >= M2) n -= M2, ++m;
    }
    return;
  }
  Channel *C = reinterpret_cast<Channel *>(const_cast<double *>(Ts) + 4 * M1);
  for (int m = threadIdx.x; m < M1; m += blockDim.x) {
    double x[4];
    int hw = 0, any = 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      x[k] = Ts[k * M1 + m];
      hw = max(hw, __double2hiint(x[k]) & 0x7fffffff);
      any |= (__double2hiint(x[k]) & 0x7fffffff) | __double2loint(x[k]);
    }
    const int eb = hw >> 20;
    const bool fixed = eb >= 650 && eb <= 1022 + kDescPlaces;
    Channel c;
    c.sh = fixed ? kDescPlaces + 1022 - eb : 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      c.f[k] = fixed ? fx::limbs<kDescLimb>(fx::from_double(x[k], c.sh)) : fx::Fix{0, 0};
      // a channel of zeros passes the test with any other but one that is left to the FP64 pipe
      c.a[k] = fixed ? (float)abs(c.f[k].hi) : (any ? 0.0f : 0x1p30f);
    }
    C[m] = c;
  }
  __syncthreads();
  // a thread keeps its column n and takes every step-th row (a block's rows lie back to back; M2 above the
  // block: several columns a thread)
  const int cols = min(M2, (int)blockDim.x), step = (int)blockDim.x / cols;
  const int m0 = (int)threadIdx.x / cols, n0 = (int)threadIdx.x - m0 * cols;
  if (m0 >= step) return;
  for (int n = n0; n < M2; n += cols) {
    const Channel b = C[n];
#pragma unroll 2
    for (int m = m0; m < M1; m += step) {
      const Channel &c = C[m];
      fx::Acc p;
      float mag = 0.0f;
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        p.mad(c.f[k], b.f[k]);
        mag = fmaf(c.a[k], b.a[k], mag);
      }
      double v = fx::to_double(fx::over_unit<kDescLimb>(p), 2 * kDescLimb - c.sh - b.sh);
      if (mag < kDescLeast) v = desc_fp64(Ts, M1, m, n);
      D[m * M2 + n] = v;
    }
  }
}

}  // namespace dfx
}  // namespace
}  // namespace dpc
