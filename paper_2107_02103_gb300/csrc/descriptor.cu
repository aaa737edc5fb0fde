// Descriptor (Sec. II): S_i = T_i^T is M1 x 4, S_i^< its first M2 rows, and
// D_i = S_i (S_i^<)^T is M1 x M2:  D[i][m][n] = sum_k T[i][k][m] T[i][k][n].
//
// On f64 arrays (the f64 and the df64 calls) a block per atom, in fixed point on the integer pipes
// (desc_fixed.cuh), where the shape is large enough for that to pay.  In f32, and in f64 below, one warp per atom:
// T_i (4 x M1) is staged in shared memory; the M1 x M2 output tile is
// contiguous, so lane l computes elements l, l + 32, ... of it in storage order, every lane busy (M1*M2 is a
// multiple of 32 for the paper's shapes) and every store coalesced.
// The warp-per-atom backward takes f32, the small f64 shapes and, in f64 or df64 arithmetic (io_t), those too wide for
// the fixed-point one's shared memory.
#include <algorithm>
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
// shared memory as two-limb integers, every sum taken in pieces of 16 terms whose limb products stay exact in 64
// bits (57 places, limbs of 28 bits: hi below 2^62), one conversion to f64 per piece.  First the 4 M1 sums over n
// (M2 terms), then the 4 M2 sums over m' (M1 terms), spread over the block by piece and added in their order.
// Rows of dD are padded to M2 + 1 entries.
// Why: 8 M1 M2 FP64 multiply-adds an atom bound the kernel above (79 % of that pipe, copper); as limb
// products they cost a ninth, and the FP64 pipe converts M1 M2 inputs and a sum per 16 terms.
// Why the exponents: channels differ in size, so each row and column of dD has its own, 2^(C_n + r_m) above
// |dD[m][n]|, and what leaves a sum through them goes into its copy of T: T[k][n] 2^C_n against its largest over n
// for the first sums, T[k][m'] 2^r_m' against its largest over m' for the second.
// Measured, 4,096 x 100 x 16: FP64 0.104 ms, one exponent for all of dD 0.054, these 0.064; 12,288: the last two
// 0.152 and 0.181.
constexpr int kGradPiece = 16, kGradL = 28, kDescGradPlaces = 57;
constexpr int kDescGradThreads = 128;
__host__ __device__ constexpr int pieces_of(int n) { return (n + kGradPiece - 1) / kGradPiece; }
// What the choice of kernel goes by: the shared memory, in 8-byte entries, of T, dT, dD and the second sums' pieces.
__host__ __device__ constexpr size_t desc_grad_f64_entries(int M1, int M2) {
  return (size_t)8 * M1 + (size_t)M1 * (M2 + 1) + (size_t)4 * M2 * pieces_of(M1);
}
// What the kernel takes (dT stays in registers; nine blocks an SM, eight with it, for 100 x 16): the two copies of T,
// dD, the pieces, the exponents of dD's rows and columns.
__host__ __device__ constexpr size_t desc_grad_f64_bytes(int M1, int M2) {
  return ((size_t)4 * M1 + (size_t)M1 * (M2 + 1) + (size_t)4 * M2 * (pieces_of(M1) + 1)) * sizeof(double) +
         (size_t)(M1 + M2) * sizeof(int);
}
constexpr int kNoValue = -(1 << 20), kNoKey = -2147483647;  // the exponent of zeros
__global__ void __launch_bounds__(kDescGradThreads)
    descriptor_grad_f64_kernel(const double *__restrict__ T, const double *__restrict__ dD, int M1, int M2,
                               double *__restrict__ dT) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ int t1[4], t2[4], wild_s;  // exponents of the two copies of T; left to the FP64 pipe
  using fx::Fix;
  Fix *Tf = reinterpret_cast<Fix *>(smem_raw);               // [4][M1]
  Fix *Df = Tf + 4 * M1;                                      // [M1][M2 + 1]
  double *H = reinterpret_cast<double *>(Df + M1 * (M2 + 1));  // [pieces][4 M2]
  const int np = pieces_of(M1), tid = threadIdx.x, lane = tid & 31;
  Fix *Tn = reinterpret_cast<Fix *>(H + 4 * M2 * np);  // [4][M2]
  int *row_e = reinterpret_cast<int *>(Tn + 4 * M2);   // [M1]
  int *col_e = row_e + M1;                             // [M2]
  const int64_t i = blockIdx.x;
  const double *Ti = T + i * 4 * M1, *Di = dD + i * (int64_t)M1 * M2;
  double *Td = reinterpret_cast<double *>(Tf), *Dd = reinterpret_cast<double *>(Df);
  // exponents are compared as high words, sign off: the field in bits 20 up
  auto key = [](double x) { return __double2hiint(x) & 0x7fffffff; };
  auto tiny = [](double x, int h) { return h < (1 << 20) && (h | __double2loint(x)); };  // a subnormal
  for (int n = tid; n < M2; n += kDescGradThreads) col_e[n] = 0;
  if (tid < 4) t1[tid] = t2[tid] = kNoValue;
  if (tid == 4) wild_s = 0;
  __syncthreads();
  // a thread's element m, n of every kDescGradThreads, and how it moves on (its column stays where M2 divides the block)
  const int step_m = kDescGradThreads / M2, step_n = kDescGradThreads - step_m * M2;
  const int m_first = tid / M2, n_first = tid - m_first * M2;
  bool wild = false;
  {
    int m = m_first, n = n_first, c = 0;
#pragma unroll 4
    for (int e = tid; e < M1 * M2; e += kDescGradThreads) {
      const double x = __ldg(Di + e);
      Dd[m * (M2 + 1) + n] = x;
      const int h = key(x);
      wild |= tiny(x, h);
      c = max(c, h);
      m += step_m;
      n += step_n;
      if (n >= M2) n -= M2, ++m;
    }
    if (step_n == 0) atomicMax(col_e + n_first, c);
  }
  for (int e = tid; e < 4 * M1; e += kDescGradThreads) Td[e] = __ldg(Ti + e);
  __syncthreads();
  if (step_n != 0) {  // uniform
    const int cols = min(M2, kDescGradThreads), rows = kDescGradThreads / cols, m0 = tid / cols;
    for (int n = tid - m0 * cols; n < M2 && m0 < rows; n += cols) {
      int c = 0;
      for (int m = m0; m < M1; m += rows) c = max(c, key(Dd[m * (M2 + 1) + n]));
      atomicMax(col_e + n, c);
    }
    __syncthreads();
  }
  // columns: field C_n, kNoValue for zeros.  Rows: the largest of field - C_n
  for (int m = tid; m < M1; m += kDescGradThreads) {
    int r = kNoKey;
#pragma unroll 4
    for (int n = 0; n < M2; ++n) {
      const int h = key(Dd[m * (M2 + 1) + n]);
      r = max(r, h ? h - (col_e[n] & 0x7ff00000) : kNoKey);
    }
    row_e[m] = r == kNoKey ? kNoValue : r >> 20;
    wild |= r != kNoKey && r < -(200 << 20);
  }
  __syncthreads();
  for (int n = tid; n < M2; n += kDescGradThreads) {
    const int c = col_e[n] >> 20;
    wild |= c && (c < 800 || c > 1022 + kDescGradPlaces);
    col_e[n] = c ? c : kNoValue;
  }
  __syncthreads();
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    int a = kNoValue, b = kNoValue;
    for (int m = tid; m < M1; m += kDescGradThreads) {
      const double x = Td[k * M1 + m];
      const int h = key(x), e = h >> 20;
      wild |= e > 1500 || tiny(x, h);
      if (h) {  // (a sum with kNoValue stays far below any other)
        if (m < M2) a = max(a, e + col_e[m]);
        b = max(b, e + row_e[m]);
      }
    }
    a = __reduce_max_sync(0xffffffffu, a);
    b = __reduce_max_sync(0xffffffffu, b);
    if (lane == 0) atomicMax(t1 + k, a), atomicMax(t2 + k, b);
  }
  if (wild) wild_s = 1;
  __syncthreads();
  int e1[4], e2[4];  // the copies' exponents; zeros only: so high that all of T falls below the places
  wild = wild_s != 0;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    e1[k] = t1[k] < -(1 << 14) ? 1 << 14 : t1[k];
    e2[k] = t2[k] < -(1 << 14) ? 1 << 14 : t2[k];
    wild |= e1[k] < 1402 || e2[k] < 402;  // results stay normal: exponents sum to 1202 at least
  }
  auto pick = [](const int (&e)[4], int k) { return k < 2 ? (k ? e[1] : e[0]) : (k == 2 ? e[2] : e[3]); };
  double *dTi = dT + i * 4 * M1;
  auto finish = [&](int k, int m, double v) {  // the first sum and, m < M2, the second's pieces
    if (m < M2) {
      double s = H[k * M2 + m];
      for (int c = 1; c < np; ++c) s += H[c * 4 * M2 + k * M2 + m];
      v += s;
    }
    dTi[k * M1 + m] = v;
  };
  constexpr int kTop = kDescGradPlaces + 1022;  // x with field e <= E has |x| 2^(kTop - E) < 2^57
  if (!wild) {  // uniform over the block
    auto convert = [&](auto same_column) {
      int m = m_first, n = n_first;
      const int c = col_e[n];
#pragma unroll 4
      for (int e = tid; e < M1 * M2; e += kDescGradThreads) {
        Fix &d = Df[m * (M2 + 1) + n];
        // (zeros of a row or column of zeros: any shift up to 899)
        const int sh = min(kTop - (decltype(same_column)::value ? c : col_e[n]) - row_e[m], 899);
        d = fx::limbs<kGradL>(fx::from_double(Dd[m * (M2 + 1) + n], sh));
        m += step_m;
        if (!decltype(same_column)::value) {
          n += step_n;
          if (n >= M2) n -= M2, ++m;
        }
      }
    };
    if (step_n == 0)
      convert(std::true_type{});
    else
      convert(std::false_type{});
#pragma unroll
    for (int k = 0; k < 4; ++k)
      for (int m = tid; m < M1; m += kDescGradThreads) {
        const double x = Td[k * M1 + m];
        if (m < M2) Tn[k * M2 + m] = fx::limbs<kGradL>(fx::from_double_any(x, kTop - e1[k] + col_e[m]));
        Tf[k * M1 + m] = fx::limbs<kGradL>(fx::from_double_any(x, kTop - e2[k] + row_e[m]));
      }
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
    constexpr int kEx = 2 * kGradL - 2 * kTop;
    for (int p = tid; p < 4 * M2 * np; p += kDescGradThreads) {  // (piece, k, m), m fastest
      const int c = p / (4 * M2), r = p - c * 4 * M2, k = r / M2, m = r - k * M2, m0 = c * kGradPiece;
      H[p] = fx::to_double(piece(Df + m0 * (M2 + 1) + m, M2 + 1, Tf + k * M1 + m0, min(kGradPiece, M1 - m0)),
                           kEx + col_e[m] + pick(e2, k));
    }
    __syncthreads();
    for (int p = tid; p < 4 * M1; p += kDescGradThreads) {  // pairs 4 m + k
      const int m = p >> 2, k = p & 3, ex = kEx + row_e[m] + pick(e1, k);
      double v = 0.0;
      for (int n = 0; n < M2; n += kGradPiece)
        v += fx::to_double(piece(Df + m * (M2 + 1) + n, 1, Tn + k * M2 + n, min(kGradPiece, M2 - n)), ex);
      finish(k, m, v);
    }
  } else {
    for (int p = tid; p < 4 * M2 * np; p += kDescGradThreads) {
      const int c = p / (4 * M2), r = p - c * 4 * M2, k = r / M2, m = r - k * M2;
      double v = 0.0;
      for (int mp = c * kGradPiece; mp < min(M1, c * kGradPiece + kGradPiece); ++mp)
        v = fma(Dd[mp * (M2 + 1) + m], Td[k * M1 + mp], v);
      H[p] = v;
    }
    __syncthreads();
    for (int p = tid; p < 4 * M1; p += kDescGradThreads) {
      const int m = p >> 2, k = p & 3;
      double v = 0.0;
      for (int n = 0; n < M2; ++n) v = fma(Dd[m * (M2 + 1) + n], Td[k * M1 + n], v);
      finish(k, m, v);
    }
  }
}

// Launches of a block per atom over as many grids as nloc takes: f(first atom, blocks).
constexpr int64_t kMaxGrid = 2147483647;
template <class F>
int in_grids(int64_t nloc, F &&f) {
  for (int64_t i0 = 0; i0 < nloc; i0 += kMaxGrid)
    if (int rc = f(i0, (unsigned)std::min<int64_t>(kMaxGrid, nloc - i0))) return rc;
  return DP_OK;
}

// Where dT in fixed point pays.  Measured with 20,000 atoms, fixed over FP64 (a warp per atom): 16 x 16 1.25, 24 x 24
// 0.98, 32 x 12 1.04, 32 x 16 0.90, 48 x 8 1.17, 48 x 12 0.90, 64 x 6 1.02, 64 x 8 0.93, 80 x 3 1.06, 80 x 6 0.94,
// 100 x 1 0.74; with 1,500 atoms the same or less.
constexpr bool desc_grad_fixed_pays(int M1, int M2) { return M1 >= 80 || M1 * M2 >= 512; }

template <typename real>
int descriptor_grad_warps(const io_t<real> *T, const io_t<real> *dD, int64_t nloc, int M1, int M2, io_t<real> *dT,
                          void *stream) {
  const size_t smem = (size_t)kDescWarps * desc_grad_smem_per_warp<real>(M1, M2) * sizeof(real);
  if (smem > 227 * 1024) return set_error(DP_ERR_UNSUPPORTED, "M1 = %d, M2 = %d need too much shared memory", M1, M2);
  if (smem > 48 * 1024) {
    const cudaError_t e = cudaFuncSetAttribute(descriptor_grad_kernel<real>,
                                               cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return set_error(DP_ERR_CUDA, "dp_descriptor_contract_grad: %s", cudaGetErrorString(e));
  }
  descriptor_grad_kernel<real><<<(unsigned)((nloc + kDescWarps - 1) / kDescWarps), kDescWarps * 32, smem,
                                 (cudaStream_t)stream>>>(T, dD, nloc, M1, M2, dT);
  return launch_status("dp_descriptor_contract_grad");
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
  if (blocks > kMaxGrid) return set_error(DP_ERR_SHAPE, "nloc too large");
  if constexpr (std::is_same<io_t<real>, double>::value) {
    // in fixed point wherever that pays and the staged dD_i leaves at least four blocks to an SM; the warps in df64
    // arithmetic only for wider ones, so that the df64 call gives the f64 call's results (12,288 atoms x 100 x 16:
    // 0.279 ms in df64 arithmetic, 0.181 here; D 0.077 and 0.066)
    const size_t need = desc_grad_f64_bytes(M1, M2);
    if (desc_grad_f64_entries(M1, M2) * sizeof(double) <= 56 * 1024) {
      if (!desc_grad_fixed_pays(M1, M2)) return descriptor_grad_warps<double>(T, dD, nloc, M1, M2, dT, stream);
      if (need > 48 * 1024) {
        const cudaError_t e = cudaFuncSetAttribute(descriptor_grad_f64_kernel,
                                                   cudaFuncAttributeMaxDynamicSharedMemorySize, (int)need);
        if (e != cudaSuccess) return set_error(DP_ERR_CUDA, "dp_descriptor_contract_grad: %s", cudaGetErrorString(e));
      }
      return in_grids(nloc, [&](int64_t i0, unsigned n) {
        descriptor_grad_f64_kernel<<<n, kDescGradThreads, need, (cudaStream_t)stream>>>(
            T + i0 * 4 * M1, dD + i0 * M1 * M2, M1, M2, dT + i0 * 4 * M1);
        return launch_status("dp_descriptor_contract_grad");
      });
    }
  }
  return descriptor_grad_warps<real>(T, dD, nloc, M1, M2, dT, stream);
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
  const int64_t blocks = (nloc + kDescWarps - 1) / kDescWarps;
  if (blocks > kMaxGrid) return set_error(DP_ERR_SHAPE, "nloc too large");
  if ((size_t)kDescWarps * 4 * M1 * sizeof(real) > 227 * 1024)
    return set_error(DP_ERR_UNSUPPORTED, "M1 = %d needs too much shared memory", M1);
  auto allow = [&](const void *kernel, size_t smem) {
    const cudaError_t e = smem > 48 * 1024
                              ? cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)
                              : cudaSuccess;
    return e == cudaSuccess ? DP_OK : set_error(DP_ERR_CUDA, "dp_descriptor_contract: %s", cudaGetErrorString(e));
  };
  if constexpr (std::is_same<real, double>::value)
    if (dfx::desc_fixed_pays(M1, M2)) {
      const size_t smem = dfx::desc_tile_bytes(M1, M2);
      if (int rc = allow((const void *)descriptor_f64_kernel, smem)) return rc;
      return in_grids(nloc, [&](int64_t i0, unsigned n) {
        descriptor_f64_kernel<<<n, kDescWarps * 32, smem, (cudaStream_t)stream>>>(T + i0 * 4 * M1, M1, M2, D + i0 * M1 * M2);
        return launch_status("dp_descriptor_contract");
      });
    }
  const size_t smem = (size_t)kDescWarps * 4 * M1 * sizeof(real);
  if (int rc = allow((const void *)descriptor_kernel<real>, smem)) return rc;
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
