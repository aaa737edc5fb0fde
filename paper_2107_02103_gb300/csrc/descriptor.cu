// Descriptor (Sec. II): S_i = T_i^T is M1 x 4, S_i^< its first M2 rows, and
// D_i = S_i (S_i^<)^T is M1 x M2:  D[i][m][n] = sum_k T[i][k][m] T[i][k][n].
//
// On f64 arrays (the f64 and the df64 calls) a block per atom, in fixed point on the integer pipes
// (desc_fixed.cuh).  In f32 one warp per atom: T_i (4 x M1) is staged in shared memory; the M1 x M2 output tile is
// contiguous, so lane l computes elements l, l + 32, ... of it in storage order, every lane busy (M1*M2 is a
// multiple of 32 for the paper's shapes) and every store coalesced.
// The warp-per-atom backward takes f32 and, in f64 or df64 arithmetic (io_t), the shapes too wide for the
// fixed-point one's shared memory.
#include <type_traits>

#include "desc_fixed.cuh"
#include "dp_common.cuh"

namespace dpc {

namespace {

constexpr int kDescWarps = 4;

template <typename real>
__global__ void __launch_bounds__(kDescWarps * 32)
    descriptor_kernel(const io_t<real> *__restrict__ T, int64_t nloc, int M1, int M2, io_t<real> *__restrict__ D) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int64_t i = (int64_t)blockIdx.x * kDescWarps + w;
  if (i >= nloc) return;  // warp-uniform; no block-wide barrier below
  real *Ts = reinterpret_cast<real *>(smem_raw) + (size_t)w * 4 * M1;
  const io_t<real> *__restrict__ Ti = T + i * 4 * M1;
#pragma unroll 4
  for (int e = lane; e < 4 * M1; e += 32) Ts[e] = from_io<real>(__ldg(Ti + e));
  __syncwarp();
  io_t<real> *__restrict__ Di = D + i * (int64_t)M1 * M2;
  const int total = M1 * M2;
  int m = lane / M2, n = lane - m * M2;
  const int dm = 32 / M2, dn = 32 - dm * M2;  // advance of (m, n) per 32 elements
  for (int e = lane; e < total; e += 32) {
    real v = Ts[m] * Ts[n];
    v = fma(Ts[M1 + m], Ts[M1 + n], v);
    v = fma(Ts[2 * M1 + m], Ts[2 * M1 + n], v);
    v = fma(Ts[3 * M1 + m], Ts[3 * M1 + n], v);
    Di[e] = to_io(v);
    m += dm;
    n += dn;
    if (n >= M2) {
      n -= M2;
      ++m;
    }
  }
}

// The same in f64: a block per atom, in fixed point (desc_fixed.cuh).
__global__ void __launch_bounds__(kDescWarps * 32)
    descriptor_f64_kernel(const double *__restrict__ T, int M1, int M2, double *__restrict__ D) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  double *Ts = reinterpret_cast<double *>(smem_raw);
  const int64_t i = blockIdx.x;
  for (int e = threadIdx.x; e < 4 * M1; e += blockDim.x) Ts[e] = __ldg(T + i * 4 * M1 + e);
  __syncthreads();
  dfx::desc_tile(Ts, M1, M2, D + i * (int64_t)M1 * M2);
}

// dD_i is staged in shared memory (read once, coalesced, converted once) in df64, where each
// element, read eight times, would otherwise cost eight conversions.  In f64 and f32 the
// second read of each element hits L1; staging there made the f32 kernel load-bound (both
// operands of every FMA from shared memory: 0.100 -> 0.146 ms on the water-like input).
template <typename real>
constexpr bool kStageDD = is_df64<real>;

// Shared memory per warp of the descriptor backward, in elements: T_i and the partial dT_i
// ([4][M1] each), and dD_i ([M1][M2 + 1], rows padded so that the eight rows one
// instruction reads fall in different banks) where it is staged.
template <typename real>
__host__ __device__ constexpr size_t desc_grad_smem_per_warp(int M1, int M2) {
  return (size_t)8 * M1 + (kStageDD<real> ? (size_t)M1 * (M2 + 1) : 0);
}

// Backward of the descriptor: D[m][n] = sum_k T[k][m] T[k][n] (n < M2) is
// quadratic in T, so for dD = dE/dD
//   dT[k][m] = sum_{n<M2} dD[m][n] T[k][n] + [m < M2] sum_{m'} dD[m'][m] T[k][m'].
// One warp per atom.  The 4*M1 (m, k) pairs of the first term are spread
// over the lanes (lane l: pairs l, l + 32, ...; 8 rows x 4 k per step, so the
// dD row reads of a step are 8 rows of M2 values); the 4*M2 (k, m) pairs of
// the second term walk the M1 rows of dD, each step reading one row.  Both
// terms meet in shared memory and dT is written coalesced.
template <typename real>
__global__ void __launch_bounds__(kDescWarps * 32)
    descriptor_grad_kernel(const io_t<real> *__restrict__ T, const io_t<real> *__restrict__ dD, int64_t nloc, int M1,
                           int M2, io_t<real> *__restrict__ dT) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int64_t i = (int64_t)blockIdx.x * kDescWarps + w;
  if (i >= nloc) return;  // warp-uniform; no block-wide barrier below
  real *Ts = reinterpret_cast<real *>(smem_raw) + (size_t)w * desc_grad_smem_per_warp<real>(M1, M2);  // [4][M1]
  real *Gs = Ts + 4 * M1;                                                                              // [4][M1]
  const io_t<real> *__restrict__ Ti = T + i * 4 * M1;
  const io_t<real> *__restrict__ Di = dD + i * (int64_t)M1 * M2;
#pragma unroll 4
  for (int e = lane; e < 4 * M1; e += 32) Ts[e] = from_io<real>(__ldg(Ti + e));
  // dD_i into shared memory ([M1][M2] after Gs) where staged; every element is read 8 times
  const real *Ds = Gs + 4 * M1;
  if constexpr (kStageDD<real>) {
    real *Dw = Gs + 4 * M1;
    // unrolled so that each lane has eight loads in flight, not one
#pragma unroll 8
    for (int e = lane; e < M1 * M2; e += 32) {
      const int r = e / M2;
      Dw[e + r] = from_io<real>(__ldg(Di + e));
    }
  }
  __syncwarp();
  auto dd = [&](int m, int n) -> real {  // dD_i[m][n]
    if constexpr (kStageDD<real>) return Ds[m * (M2 + 1) + n];
    else return __ldg(Di + (size_t)m * M2 + n);
  };
  // In df64 each sum runs in four interleaved partial sums: one chain of dependent df64 FMAs
  // (eight dependent instructions each) would leave the pipes idle between them.  In f64 and
  // f32 the extra adds cost more than they hide (f64: +13 % on the water-like input).
  constexpr int NP = is_df64<real> ? 4 : 1;
  // first term, pairs p = 4 m + k
  for (int p = lane; p < 4 * M1; p += 32) {
    const int m = p >> 2, k = p & 3;
    const real *tk = Ts + k * M1;
    real v[NP];
#pragma unroll
    for (int q = 0; q < NP; ++q) v[q] = real(0);
    int n = 0;
    for (; n + NP <= M2; n += NP)
#pragma unroll
      for (int q = 0; q < NP; ++q) v[q] = fma(dd(m, n + q), tk[n + q], v[q]);
    for (; n < M2; ++n) v[0] = fma(dd(m, n), tk[n], v[0]);
#pragma unroll
    for (int q = 1; q < NP; ++q) v[0] += v[q];
    Gs[k * M1 + m] = v[0];
  }
  __syncwarp();
  // second term, pairs p = M2 k + m (m < M2)
  for (int p = lane; p < 4 * M2; p += 32) {
    const int k = p / M2, m = p - k * M2;
    const real *tk = Ts + k * M1;
    real v[NP];
#pragma unroll
    for (int q = 0; q < NP; ++q) v[q] = real(0);
    int mp = 0;
    for (; mp + NP <= M1; mp += NP)
#pragma unroll
      for (int q = 0; q < NP; ++q) v[q] = fma(dd(mp + q, m), tk[mp + q], v[q]);
    for (; mp < M1; ++mp) v[0] = fma(dd(mp, m), tk[mp], v[0]);
#pragma unroll
    for (int q = 1; q < NP; ++q) v[0] += v[q];
    Gs[k * M1 + m] += v[0];
  }
  __syncwarp();
  io_t<real> *__restrict__ dTi = dT + i * 4 * M1;
  for (int e = lane; e < 4 * M1; e += 32) dTi[e] = to_io(Gs[e]);
}

// The same in f64, a block per atom, in fixed point (fixed.cuh): T_i [4][M1] and dD_i [M1][M2] staged in
// shared memory as two-limb integers (T against the largest of each k, dD against its own), every sum taken in
// pieces of 16 terms whose limb products stay exact in 64 bits (57 places, limbs of 28 bits: hi below 2^62),
// one conversion to f64 per piece.  First the 4 M1 sums over n (M2 terms), then the 4 M2 sums over m' (M1
// terms), spread over the block by piece and added in their order.  Rows of dD are padded to M2 + 1 entries.
// Why: 8 M1 M2 FP64 multiply-adds an atom bound the kernel above (79 % of that pipe, copper); as limb
// products they cost a ninth, and the FP64 pipe converts M1 M2 inputs and a sum per 16 terms.
// Measured: copper (4,096 x 100 x 16) 0.104 -> 0.058 ms; 1,536 atoms 0.047 -> 0.031 ms.
constexpr int kGradPiece = 16, kGradL = 28, kDescGradPlaces = 57;
constexpr int kDescGradThreads = 128;
__host__ __device__ constexpr int pieces_of(int n) { return (n + kGradPiece - 1) / kGradPiece; }
// 8-byte entries of shared memory: T, dD, the first term, the second term's pieces
__host__ __device__ constexpr size_t desc_grad_f64_entries(int M1, int M2) {
  return (size_t)8 * M1 + (size_t)M1 * (M2 + 1) + (size_t)4 * M2 * pieces_of(M1);
}
__global__ void __launch_bounds__(kDescGradThreads)
    descriptor_grad_f64_kernel(const double *__restrict__ T, const double *__restrict__ dD, int M1, int M2,
                               double *__restrict__ dT) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ int red[5];  // the largest high words: of T's rows, of dD
  using fx::Fix;
  Fix *Tf = reinterpret_cast<Fix *>(smem_raw);              // [4][M1]
  double *G = reinterpret_cast<double *>(Tf + 4 * M1);       // [4][M1]
  Fix *Df = reinterpret_cast<Fix *>(G + 4 * M1);             // [M1][M2 + 1]
  double *H = reinterpret_cast<double *>(Df + M1 * (M2 + 1));  // [pieces][4 M2]
  const int tid = threadIdx.x, lane = tid & 31;
  const int64_t i = blockIdx.x;
  const double *Ti = T + i * 4 * M1, *Di = dD + i * (int64_t)M1 * M2;
  double *Td = reinterpret_cast<double *>(Tf), *Dd = reinterpret_cast<double *>(Df);
  if (tid < 5) red[tid] = 0;
  __syncthreads();
  int hd = 0;
  {
    const int step_m = kDescGradThreads / M2, step_n = kDescGradThreads - step_m * M2;
    int m = tid / M2, n = tid - m * M2;
#pragma unroll 4
    for (int e = tid; e < M1 * M2; e += kDescGradThreads) {
      const double x = __ldg(Di + e);
      Dd[m * (M2 + 1) + n] = x;
      hd = max(hd, __double2hiint(x) & 0x7fffffff);
      m += step_m;
      n += step_n;
      if (n >= M2) n -= M2, ++m;
    }
  }
  hd = __reduce_max_sync(0xffffffffu, hd);
  if (lane == 0) atomicMax(red + 4, hd);
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    int ht = 0;
    for (int m = tid; m < M1; m += kDescGradThreads) {
      const double x = __ldg(Ti + k * M1 + m);
      Td[k * M1 + m] = x;
      ht = max(ht, __double2hiint(x) & 0x7fffffff);
    }
    ht = __reduce_max_sync(0xffffffffu, ht);
    if (lane == 0) atomicMax(red + k, ht);
  }
  __syncthreads();
  bool wild = false;
  const int sd = dfx::places_of(red[4], kDescGradPlaces, wild);
  int st[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) st[k] = dfx::places_of(red[k], kDescGradPlaces, wild);
  auto places_t = [&](int k) { return k < 2 ? (k ? st[1] : st[0]) : (k == 2 ? st[2] : st[3]); };
  const int np = pieces_of(M1);
  if (!wild) {  // uniform over the block
    // (the padding entries hold whatever the memory held and are not read again)
    for (int e = tid; e < M1 * (M2 + 1); e += kDescGradThreads) Df[e] = fx::limbs<kGradL>(fx::from_double(Dd[e], sd));
#pragma unroll
    for (int k = 0; k < 4; ++k)
      for (int m = tid; m < M1; m += kDescGradThreads)
        Tf[k * M1 + m] = fx::limbs<kGradL>(fx::from_double(Td[k * M1 + m], st[k]));
    __syncthreads();
    // sum over cnt <= 16 terms of a (stride sa) times b (consecutive), over 2^(2 L)
    auto piece = [&](const Fix *a, int sa, const Fix *b, int cnt) {
      fx::Acc p;
      if (cnt == kGradPiece) {
#pragma unroll
        for (int q = 0; q < kGradPiece; ++q, a += sa) p.mad(*a, b[q]);
      } else {
        for (int q = 0; q < cnt; ++q, a += sa) p.mad(*a, b[q]);
      }
      return fx::over_unit<kGradL>(p);
    };
    for (int p = tid; p < 4 * M1; p += kDescGradThreads) {  // pairs 4 m + k
      const int m = p >> 2, k = p & 3, ex = 2 * kGradL - sd - places_t(k);
      double v = 0.0;
      for (int n = 0; n < M2; n += kGradPiece)
        v += fx::to_double(piece(Df + m * (M2 + 1) + n, 1, Tf + k * M1 + n, min(kGradPiece, M2 - n)), ex);
      G[k * M1 + m] = v;
    }
    for (int p = tid; p < 4 * M2 * np; p += kDescGradThreads) {  // (piece, k, m), m fastest
      const int c = p / (4 * M2), r = p - c * 4 * M2, k = r / M2, m = r - k * M2, m0 = c * kGradPiece;
      H[p] = fx::to_double(piece(Df + m0 * (M2 + 1) + m, M2 + 1, Tf + k * M1 + m0, min(kGradPiece, M1 - m0)),
                           2 * kGradL - sd - places_t(k));
    }
  } else {
    for (int p = tid; p < 4 * M1; p += kDescGradThreads) {
      const int m = p >> 2, k = p & 3;
      double v = 0.0;
      for (int n = 0; n < M2; ++n) v = fma(Dd[m * (M2 + 1) + n], Td[k * M1 + n], v);
      G[k * M1 + m] = v;
    }
    for (int p = tid; p < 4 * M2 * np; p += kDescGradThreads) {
      const int c = p / (4 * M2), r = p - c * 4 * M2, k = r / M2, m = r - k * M2;
      double v = 0.0;
      for (int mp = c * kGradPiece; mp < min(M1, c * kGradPiece + kGradPiece); ++mp)
        v = fma(Dd[mp * (M2 + 1) + m], Td[k * M1 + mp], v);
      H[p] = v;
    }
  }
  __syncthreads();
  double *dTi = dT + i * 4 * M1;
  for (int e = tid; e < 4 * M1; e += kDescGradThreads) {
    const int k = e / M1, m = e - k * M1;
    double v = G[e];
    if (m < M2) {
      double s = H[k * M2 + m];
      for (int c = 1; c < np; ++c) s += H[c * 4 * M2 + k * M2 + m];
      v += s;
    }
    dTi[e] = v;
  }
}

template <typename real>
int descriptor_grad(const io_t<real> *T, const io_t<real> *dD, int64_t nloc, int M1, int M2, io_t<real> *dT,
                    void *stream) {
  clear_error();
  if (nloc < 0 || M1 < 1 || M2 < 1 || M2 > M1)
    return set_error(DP_ERR_SHAPE, "need nloc >= 0 and 1 <= M2 <= M1 (nloc %lld, M1 %d, M2 %d)", (long long)nloc, M1,
                     M2);
  if (M1 > 4096) return set_error(DP_ERR_UNSUPPORTED, "M1 = %d > 4096", M1);
  if (nloc == 0) return DP_OK;
  if (!T || !dD || !dT) return set_error(DP_ERR_NULL, "T, dD or dT is NULL");
  const int64_t blocks = (nloc + kDescWarps - 1) / kDescWarps;
  if (blocks > 2147483647LL) return set_error(DP_ERR_SHAPE, "nloc too large");
  if constexpr (std::is_same<io_t<real>, double>::value) {
    // in fixed point wherever the staged dD_i leaves at least four blocks to an SM; the kernel below for wider
    // ones.  Also for the df64 call, whose arrays are f64 (12,288 atoms x 100 x 16: 0.279 ms in df64 arithmetic,
    // 0.151 here; D 0.077 and 0.058)
    const size_t need = desc_grad_f64_entries(M1, M2) * sizeof(double);
    if (need <= 56 * 1024 && nloc <= 2147483647LL && M1 <= 1024) {
      if (need > 48 * 1024) {
        const cudaError_t e = cudaFuncSetAttribute(descriptor_grad_f64_kernel,
                                                   cudaFuncAttributeMaxDynamicSharedMemorySize, (int)need);
        if (e != cudaSuccess) return set_error(DP_ERR_CUDA, "dp_descriptor_contract_grad: %s", cudaGetErrorString(e));
      }
      descriptor_grad_f64_kernel<<<(unsigned)nloc, kDescGradThreads, need, (cudaStream_t)stream>>>(T, dD, M1, M2, dT);
      return launch_status("dp_descriptor_contract_grad");
    }
  }
  const size_t smem = (size_t)kDescWarps * desc_grad_smem_per_warp<real>(M1, M2) * sizeof(real);
  if (smem > 227 * 1024) return set_error(DP_ERR_UNSUPPORTED, "M1 = %d, M2 = %d need too much shared memory", M1, M2);
  if (smem > 48 * 1024) {
    const cudaError_t e = cudaFuncSetAttribute(descriptor_grad_kernel<real>,
                                               cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return set_error(DP_ERR_CUDA, "dp_descriptor_contract_grad: %s", cudaGetErrorString(e));
  }
  descriptor_grad_kernel<real>
      <<<(unsigned)blocks, kDescWarps * 32, smem, (cudaStream_t)stream>>>(T, dD, nloc, M1, M2, dT);
  return launch_status("dp_descriptor_contract_grad");
}

template <typename real>
int descriptor(const io_t<real> *T, int64_t nloc, int M1, int M2, io_t<real> *D, void *stream) {
  clear_error();
  if (nloc < 0 || M1 < 1 || M2 < 1 || M2 > M1)
    return set_error(DP_ERR_SHAPE, "need nloc >= 0 and 1 <= M2 <= M1 (nloc %lld, M1 %d, M2 %d)", (long long)nloc, M1,
                     M2);
  if (M1 > 4096) return set_error(DP_ERR_UNSUPPORTED, "M1 = %d > 4096", M1);
  if (nloc == 0) return DP_OK;
  if (!T || !D) return set_error(DP_ERR_NULL, "T or D is NULL");
  constexpr bool f64 = std::is_same<real, double>::value;
  const int64_t blocks = f64 ? nloc : (nloc + kDescWarps - 1) / kDescWarps;
  if (blocks > 2147483647LL) return set_error(DP_ERR_SHAPE, "nloc too large");
  if ((size_t)kDescWarps * 4 * M1 * sizeof(real) > 227 * 1024)
    return set_error(DP_ERR_UNSUPPORTED, "M1 = %d needs too much shared memory", M1);
  const size_t smem = f64 ? dfx::desc_tile_bytes(M1) : (size_t)kDescWarps * 4 * M1 * sizeof(real);
  const void *kernel = f64 ? (const void *)descriptor_f64_kernel : (const void *)descriptor_kernel<real>;
  if (smem > 48 * 1024) {
    const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return set_error(DP_ERR_CUDA, "dp_descriptor_contract: %s", cudaGetErrorString(e));
  }
  if constexpr (f64)
    descriptor_f64_kernel<<<(unsigned)blocks, kDescWarps * 32, smem, (cudaStream_t)stream>>>(T, M1, M2, D);
  else
    descriptor_kernel<real><<<(unsigned)blocks, kDescWarps * 32, smem, (cudaStream_t)stream>>>(T, nloc, M1, M2, D);
  return launch_status("dp_descriptor_contract");
}

}  // namespace

}  // namespace dpc

extern "C" {

int dp_descriptor_contract_f64(const double *T, int64_t nloc, int M1, int M2, double *D, void *stream) {
  return dpc::descriptor<double>(T, nloc, M1, M2, D, stream);
}

int dp_descriptor_contract_f32(const float *T, int64_t nloc, int M1, int M2, float *D, void *stream) {
  return dpc::descriptor<float>(T, nloc, M1, M2, D, stream);
}

int dp_descriptor_contract_df64(const double *T, int64_t nloc, int M1, int M2, double *D, void *stream) {
  return dpc::descriptor<double>(T, nloc, M1, M2, D, stream);
}

int dp_descriptor_contract_grad_df64(const double *T, const double *dD, int64_t nloc, int M1, int M2, double *dT,
                                     void *stream) {
  return dpc::descriptor_grad<dpc::df64>(T, dD, nloc, M1, M2, dT, stream);
}

int dp_descriptor_contract_grad_f64(const double *T, const double *dD, int64_t nloc, int M1, int M2, double *dT,
                                    void *stream) {
  return dpc::descriptor_grad<double>(T, dD, nloc, M1, M2, dT, stream);
}

int dp_descriptor_contract_grad_f32(const float *T, const float *dD, int64_t nloc, int M1, int M2, float *dT,
                                    void *stream) {
  return dpc::descriptor_grad<float>(T, dD, nloc, M1, M2, dT, stream);
}

}  // extern "C"
