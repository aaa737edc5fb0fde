// Exact f64 GEMMs on the tcgen05 tensor cores, shared by the fitting net and the
// tensor-core form of the tabulated embedding.
#pragma once

#include <cuda_runtime.h>

#include <atomic>
#include <cstdint>

#include "dp_common.cuh"

namespace dpc {
namespace {

// ------------------------------------------------- f64 GEMMs on the tensor cores
// GB300 retires FP64 at 2 lanes per clock per SM but fp16 products on its
// tcgen05 tensor cores at ~1000 times that rate.  An f64 GEMM C = A B is
// recovered from fp16 products by splitting every operand element into base-64
// digits (the error-free splitting of Ozaki et al., here with balanced digits):
//   a_ik = 2^(E_i + 1) sum_{s=1..9} A_s[i][k] 64^-s + r_ik,  A_s integers in [-32, 32],  |r_ik| < 2^(E_i - 53),
// with max_k |a_ik| < 2^E_i: the row's 53-bit fixed point a 2^(53 - E) is truncated toward zero and
// biased by 32 (64^7 + ... + 1); its eight low 6-bit fields less 32 are digits 2 .. 9, and what lies
// above them (an arithmetic shift) is digit 1.  Likewise b_kj with a column exponent F_j, so that
//   C_ij = 2^(E_i + F_j + 2) sum_{d=2..10} 64^-d sum_{s+t=d} (A_s B_t)_ij + (terms with s + t > 10 and the r).
// Every (A_s B_t)_ij is a sum of integer products |A_s B_t| <= 1024; a diagonal
// d has at most 9 of them, so its fp32 sum on the tensor cores is exact while
// a block's share of K is at most kMaxShareK = 1792 (9 x 1792 x 1024 < 2^24).
// The diagonal sums of an output are recombined exactly as one 128-bit integer
// and rounded once (diag_s128, s128_to_f64).  What rounds is that conversion,
// the 53-bit truncation of the operands and the dropped terms: |error| <~
// K 2^-49 max_k|a_ik| max_k|b_kj|, against K 2^-53 sum_k |a_ik b_kj| for an f64
// dot product.  A row or column with an inf or NaN gives NaN outputs.
//
// Three schemes of digits (Digits below) serve the kernels: nine of 6 bits, the
// tabulation's forward (tab_gemm.cuh; K up to 1792 a share); eight of 7 bits,
// the fitting net (fit_gemm.cuh; 36 products, K up to 512 a share); seven of 8
// bits, the tabulation's backward, whose K is M1 <= 144 (tab_gemm_b8.cuh; 28
// products).  This file has what they share: the splitting of operands into
// digit planes (as the shared-memory image of each (tile, 16-deep K slice)
// block, the tcgen05 K-major layout without swizzle), the recombination, the
// descriptors and the bounded waits.  A wait on an mbarrier that gives up makes
// the kernel's outputs NaN and counts one timeout in g_wait_timeouts, which the
// host reads through dp_tc_wait_timeouts.
namespace tc {
constexpr int kS = 9;      // digits per operand element
constexpr int kBits = 6;   // bits per digit
constexpr int kFrac = kS * kBits - 1;  // 53 fractional bits; the ninth digit's spare bit keeps the balanced top digit in range
constexpr int kPad = kS * kBits - kFrac;  // a digit vector stands for 2^(E + kPad) sum_s d_s 64^-s
// 32 (64^7 + ... + 1): added to a fixed point f in (-2^53, 2^53), it makes each of the eight low 6-bit
// fields a digit plus 32 and leaves floor((f + bias) / 64^8) in [-32, 32] as the top digit
constexpr int64_t kDigitBias = 32ll * ((1ll << 48) - 1ll) / 63ll;
constexpr int kTM = 128, kTN = 48, kTK = 16;  // CTA tile; K per stage (one MMA)
constexpr int kStages = 4;
constexpr int kMaxShareK = 1792;
constexpr int kNonFinite = 1 << 20;  // exponent of a row or column holding inf or NaN
constexpr uint32_t kLBO = 128, kSBO = 256;  // core matrices: next along K at +128 B, next 8 rows at +256 B
constexpr int kPlaneA = kTM * kTK * 2, kPlaneB = kTN * kTK * 2;  // bytes of one digit plane in a stage
constexpr int kStageBytes = kS * (kPlaneA + kPlaneB);
constexpr uint32_t kTmemCols = 512;  // allocation (a power of two); kS * kTN = 432 used
constexpr int kMaxShareSlices = kMaxShareK / kTK;
constexpr int kScatKeys = kTM / 4 + 1, kScatAtoms = kTN / 4;  // scatter: keys (kq >= 4) and atoms of a tile
static_assert((size_t)kS * kMaxShareK * 32 * 32 < (1u << 24), "fp32 diagonal sums must stay exact");
static_assert(kDigitBias < (1ll << 48) && kFrac == 53 && kS == 9, "top digit floor((f + bias) / 2^48) within [-32, 32]");
static_assert(kMaxShareK % kTK == 0 && kS * kTN <= (int)kTmemCols, "shares and TMEM");

__host__ __device__ constexpr int64_t round_up(int64_t x, int64_t m) { return (x + m - 1) / m * m; }

__device__ __forceinline__ int exp_bits(double x) { return (int)(((uint64_t)__double_as_longlong(x) >> 52) & 0x7ff); }
__device__ __forceinline__ bool nonzero(double x) { return ((uint64_t)__double_as_longlong(x) << 1) != 0; }
// E with max |x| < 2^E from the largest biased exponent (normal x: |x| < 2^(eb - 1022))
__device__ __forceinline__ int exp_of_max(int ebmax) { return ebmax == 0x7ff ? kNonFinite : max(ebmax, 1) - 1022; }

// A digit scheme: NS balanced digits of NB bits (digit 1 in [-2^(NB-1), 2^(NB-1)], the others in
// [-2^(NB-1), 2^(NB-1) - 1]) for an element's NS NB - 1 fractional bits.  The tensor-core GEMMs use 9 x 6
// bits (kS, kBits: a share of K up to kMaxShareK = 1792) or, where K <= 144, 7 x 8 bits (products up to
// 2^14, seven of them on a diagonal: 7 x 2^14 x 144 < 2^24), which needs 28 digit products instead of 45.
template <int NS, int NB>
struct Digits {
  static constexpr int kNS = NS, kNB = NB;
  static constexpr int kFrac = NS * NB - 1;
  static constexpr int kPad = NS * NB - kFrac;  // a digit vector stands for 2^(E + kPad) sum_s d_s 2^(-NB s)
  static constexpr int64_t kBias = (1ll << (NB - 1)) * ((1ll << (NB * (NS - 1))) - 1ll) / ((1ll << NB) - 1ll);
  static constexpr uint32_t kHalf = 1u << (NB - 1);
  // the fp16 pair 1024 + kHalf: field u in [0, 2^NB] is encoded as 0x6400 | u (1024 + u) and this comes off
  static constexpr uint32_t kOffPair = (0x6400u + kHalf) * 0x10001u;
  static_assert(kBias < (1ll << (NB * (NS - 1))) && NB * (NS - 1) <= 56 && NB <= 9, "balanced top digit in range");
};
using Digits9x6 = Digits<9, 6>;
using Digits8x7 = Digits<8, 7>;
using Digits7x8 = Digits<7, 8>;
static_assert(Digits9x6::kBias == kDigitBias && Digits9x6::kFrac == kFrac && Digits9x6::kPad == kPad, "the 9 x 6 scheme");
static_assert(Digits8x7::kFrac == 55 && Digits8x7::kPad == 1 && Digits8x7::kBias < (1ll << 49), "the 8 x 7 scheme");
static_assert(Digits7x8::kFrac == 55 && Digits7x8::kPad == 1 && Digits7x8::kBias < (1ll << 48), "the 7 x 8 scheme");

// x 2^(kFrac - E) truncated toward zero (|x| < 2^E, so |.| < 2^kFrac), plus the scheme's bias (see digit_pairs)
template <class D = Digits9x6>
__device__ __forceinline__ int64_t biased_fixed(double x, int E) {
  const uint64_t b = (uint64_t)__double_as_longlong(x);
  const int eb = (int)((b >> 52) & 0x7ff);
  const uint64_t mant = b & 0xfffffffffffffull;
  const uint64_t m = eb ? (mant | (1ull << 52)) : mant;
  const int sh = (eb ? eb - 1075 : -1074) - E + D::kFrac;  // |x| 2^(kFrac - E) = m 2^sh, sh <= kFrac - 53 for finite x
  const int64_t mag = (int64_t)(sh >= 0 ? m << min(sh, 10) : (sh > -64 ? m >> -sh : 0ull));
  return (b >> 63 ? -mag : mag) + D::kBias;
}

// The NS balanced digits of two elements from their biased fixed points g, digit s of both packed as an
// fp16 pair (element 0 in the low half): field u in [0, 2^NB] (digit + 2^(NB-1)) is encoded as 0x6400 | u,
// the fp16 1024 + u, and 1024 + 2^(NB-1) comes off exactly.  Digits 2 .. NS are the low NB-bit fields;
// digit 1 is g shifted right by NB (NS - 1).
template <class D = Digits9x6>
__device__ __forceinline__ void digit_pairs(int64_t g0, int64_t g1, uint32_t (&h)[D::kNS]) {
  constexpr int NS = D::kNS, NB = D::kNB;
  constexpr uint32_t kMask = (1u << NB) - 1;
#pragma unroll
  for (int s = 1; s <= NS; ++s) {
    const int sh = NB * (NS - s);
    const uint32_t d0 = s == 1 ? (uint32_t)((g0 >> sh) + D::kHalf) : (uint32_t)(g0 >> sh) & kMask;
    const uint32_t d1 = s == 1 ? (uint32_t)((g1 >> sh) + D::kHalf) : (uint32_t)(g1 >> sh) & kMask;
    asm("sub.rn.f16x2 %0, %1, %2;" : "=r"(h[s - 1]) : "r"(0x64006400u | d0 | (d1 << 16)), "r"(D::kOffPair));
  }
}

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

// Rows of a matrix as digit planes, laid out as the shared-memory image of each (tile of RT rows,
// 16-deep K slice) block that the GEMM kernels copy in one piece: block (r / RT, k / 16) holds the kS
// planes of those rows and columns, plane s at s RT 32 bytes, and in a plane the tcgen05 K-major
// core matrices (8 rows x 8 k = 128 bytes; the second 8 k of the slice at +128 B, the next 8 rows
// at +256 B).  Also the rows' exponents [rows_p].  Element (r, k) of the source is X[r ld_r + k ld_k];
// rows >= nrows and columns >= K are zero (row_exps_kernel first finds the exponents).  Used for the A operand (rows of the
// layer input, RT = kTM) and for B (RT = kTN; forward: the columns of W, ld_r = 1, ld_k = N;
// backward: the rows of W).
__global__ void __launch_bounds__(128) row_exps_kernel(const double *__restrict__ X, int64_t ld_r, int64_t ld_k,
                                                       int64_t nrows, int K, int64_t rows_p, int zeros,
                                                       int *__restrict__ exps) {
  // one warp per row: E with max_k |x_rk| < 2^E, `zeros` for a row of zeros
  const int lane = threadIdx.x & 31;
  const int64_t r = (int64_t)blockIdx.x * 4 + (threadIdx.x >> 5);
  if (r >= rows_p) return;  // warp-uniform
  int eb = 0;
  if (r < nrows)
    for (int k = lane; k < K; k += 32) eb = max(eb, exp_bits(__ldg(X + r * ld_r + k * ld_k)));
  eb = __reduce_max_sync(0xffffffffu, eb);
  bool any = eb != 0;  // zeros, or subnormals?
  if (!any && r < nrows)
    for (int k = lane; k < K; k += 32) any |= nonzero(__ldg(X + r * ld_r + k * ld_k));
  any = __any_sync(0xffffffffu, any);
  if (lane == 0) exps[r] = any ? exp_of_max(eb) : zeros;
}

constexpr int kSplitK = 64;  // K per warp of split_rows_kernel
template <class D>
__global__ void __launch_bounds__(128) split_rows_kernel(const double *__restrict__ X, int64_t ld_r, int64_t ld_k,
                                                         int64_t nrows, int K, int64_t rows_p, int Kp, int RT,
                                                         unsigned char *__restrict__ planes,
                                                         const int *__restrict__ exps) {
  // one warp per (group of 8 rows, kSplitK of K): lane = (row ri8 = lane / 4, pair of k kp = lane % 4),
  // so that per plane and 8 k the warp writes one whole 128-byte core matrix
  const int lane = threadIdx.x & 31, ri8 = lane >> 2, kp = lane & 3;
  const int kchunks = (Kp + kSplitK - 1) / kSplitK;
  const int64_t w = (int64_t)blockIdx.x * 4 + (threadIdx.x >> 5);
  const int64_t g = w / kchunks;  // 8-row group
  if (g * 8 >= rows_p) return;    // warp-uniform
  const int kc = (int)(w - g * kchunks);
  const int64_t r = g * 8 + ri8;
  const double *__restrict__ xr = X + (r < nrows ? r : 0) * ld_r;
  auto x = [&](int k) { return (r < nrows && k < K) ? __ldg(xr + k * ld_k) : 0.0; };
  const int E = exps[r];
  constexpr int NS = D::kNS;
  const size_t plane = (size_t)RT * kTK * 2, block = NS * plane;
  const int ri = (int)(r % RT);
  unsigned char *rowbase = planes + (size_t)(r / RT) * (Kp / kTK) * block + (ri >> 3) * kSBO + (ri & 7) * 16 + kp * 4;
  for (int k0 = kc * kSplitK; k0 < min(Kp, kc * kSplitK + kSplitK); k0 += 8) {
    const int k = k0 + 2 * kp;
    const double x0 = x(k), x1 = x(k + 1);
    uint32_t h[NS];
    digit_pairs<D>(biased_fixed<D>(x0, E), biased_fixed<D>(x1, E), h);
    unsigned char *dst = rowbase + (size_t)(k0 / kTK) * block + ((k0 % kTK) >> 3) * kLBO;
#pragma unroll
    for (int s = 0; s < NS; ++s) *reinterpret_cast<uint32_t *>(dst + s * plane) = h[s];
  }
}

// shared-memory descriptor of a K-major operand without swizzle (tcgen05): start address, the byte
// offsets of the next core matrix along K (leading) and along the rows (stride), version 1
__device__ __forceinline__ uint64_t smem_desc(uint32_t saddr) {
  return (uint64_t)((saddr & 0x3FFFF) >> 4) | ((uint64_t)(kLBO >> 4) << 16) | ((uint64_t)(kSBO >> 4) << 32) |
         (1ull << 46);
}
// instruction descriptor, kind::f16: D f32 (bits 4-5 = 1), A and B f16 (0), both K-major, N >> 3 at
// bit 17 (set per MMA), M >> 4 at bit 24
constexpr uint32_t kIdescNoN = (1u << 4) | ((uint32_t)(kTM >> 4) << 24);  // N >> 3 goes in at bit 17
constexpr int kMaxPlanesPerMma = 256 / kTN;  // N <= 256 for M = 128
static_assert(kTN % 16 == 0 && kMaxPlanesPerMma >= 1, "MMA N: multiples of 16 up to 256");

// Bounded mbarrier waits that gave up, one count per CTA (this translation unit's kernels).
__device__ unsigned int g_wait_timeouts;

// The count, read after a device synchronisation, then cleared.
int take_wait_timeouts(unsigned int *count) {
  unsigned int v = 0, zero = 0;
  cudaError_t e = cudaDeviceSynchronize();
  if (e == cudaSuccess) e = cudaMemcpyFromSymbol(&v, g_wait_timeouts, sizeof v);
  if (e == cudaSuccess) e = cudaMemcpyToSymbol(g_wait_timeouts, &zero, sizeof zero);
  if (e != cudaSuccess) return set_error(DP_ERR_CUDA, "dp_tc_wait_timeouts: %s", cudaGetErrorString(e));
  *count += v;
  return DP_OK;
}

// A wait on an mbarrier phase, bounded in time (2 s on the global timer), that also gives up once another
// role has.  The waiting thread is suspended between polls (try_wait's time hint), so that a waiting
// thread takes no issue slots or shared-memory bandwidth from the copies and the MMAs.
__device__ __forceinline__ uint64_t global_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
__device__ __forceinline__ bool wait_or_abort(uint32_t bar, uint32_t parity, volatile int *abortf) {
  const uint64_t t0 = global_ns();
  for (;;) {
    uint32_t done;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n selp.u32 %0, 1, 0, p;\n}"
        : "=r"(done)
        : "r"(bar), "r"(parity), "r"(20000u)
        : "memory");
    if (done) return true;
    if (*abortf) return false;
    if (global_ns() - t0 > 2000000000ull) {
      *abortf = 1;
      return false;
    }
  }
}

// What a CTA still has in flight once a wait of it has given up: its copies into the stages that its producer issued
// last (the `full` barriers' phases) and the MMAs before its last commit.  The CTA waits for them before it gives up its
// shared memory and TMEM, each in at most kSettlePolls polls of about 20 us (a wait runs out by the clock, so also
// where the GPU was taken away from the kernel for seconds, and then all of this is still under way).  False if
// one did not end: a stage whose other arrivals are missing as well.
constexpr int kSettlePolls = 500;
__device__ __forceinline__ bool settle(uint32_t bar, uint32_t parity) {
  for (int i = 0; i < kSettlePolls; ++i) {
    uint32_t done;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n selp.u32 %0, 1, 0, p;\n}"
        : "=r"(done)
        : "r"(bar), "r"(parity), "r"(20000u)
        : "memory");
    if (done) return true;
  }
  return false;
}
// issued: slices whose copies the producer started, over a ring of `stages` (8-byte barriers from `full` on).
__device__ __forceinline__ bool settle_copies(uint32_t full, int stages, int issued) {
  bool all = true;
  for (int g = max(0, issued - stages); g < issued; ++g)
    all &= settle(full + 8 * (uint32_t)(g % stages), (uint32_t)((g / stages) & 1));
  return all;
}

// A float that holds an integer of at most 2^24 in magnitude (a diagonal sum) as an int: exact.
__device__ __forceinline__ int exact_int(float f) { return __float2int_rz(f); }

// The nine diagonal sums of one output (exact integers below 2^24; diagonal d weighs 64^-(d+2)) as one
// exact integer in units of 2^-60, S = sum_d v[d][c] 2^(6 (8 - d)), |S| < 2^74: integer adds, no rounding.
template <int W>
__device__ __forceinline__ __int128 diag_int(const float (&v)[kS][W], int c) {
  static_assert(kS == 9 && kBits == 6, "the integer recombination assumes nine 6-bit digits");
  long long lo = 0;  // diagonals 4 .. 10: below 2^24 2^36 64/63 < 2^61
#pragma unroll
  for (int d = 2; d < kS; ++d) lo += (long long)exact_int(v[d][c]) << (kBits * (kS - 1 - d));
  const long long hi = (long long)exact_int(v[0][c]) * 64 + exact_int(v[1][c]);  // diagonals 2, 3 over 2^42
  return ((__int128)hi << 42) + lo;
}

// S 2^e2 rounded once to the nearest f64 (ties to even), from its bits: integer operations only, except
// where the result falls outside the normal range (never for these sums in practice).
__device__ __forceinline__ double i128_to_double(__int128 S, int e2) {
  if (S == 0) return 0.0;
  const bool neg = S < 0;
  const unsigned __int128 U = neg ? (unsigned __int128)(-S) : (unsigned __int128)S;
  const unsigned long long uh = (unsigned long long)(U >> 64), ul = (unsigned long long)U;
  const int n = uh ? 128 - __clzll((long long)uh) : 64 - __clzll((long long)ul);  // bit length of |S|
  int ex = n - 1 + e2;  // exponent of the leading bit
  unsigned long long m;
  if (n <= 53) {
    m = ul << (53 - n);
  } else {
    const int sh = n - 53;
    m = (unsigned long long)(U >> sh);
    const unsigned long long rem = ul & ((1ull << sh) - 1ull), half = 1ull << (sh - 1);
    if (rem > half || (rem == half && (m & 1ull))) {
      ++m;
      if (m == (1ull << 53)) {
        m >>= 1;
        ++ex;
      }
    }
  }
  if (ex < -1022 || ex > 1023) return (neg ? -1.0 : 1.0) * scalbn((double)m, ex - 52);
  return __longlong_as_double((long long)(((unsigned long long)neg << 63) | ((unsigned long long)(ex + 1023) << 52) |
                                          (m & ((1ull << 52) - 1ull))));
}

// An output from its exact integer: NaN for a row or column with an inf or NaN.
__device__ __forceinline__ double output_value(__int128 S, int E, int F) {
  if (E >= kNonFinite || F >= kNonFinite) return __longlong_as_double(0x7ff8000000000000ll);
  return i128_to_double(S, E + F + 2 * kPad - 2 * kBits - kBits * (kS - 1));
}

// The exponent offset of output_value: an output is S 2^(E + F + kOutExp).
constexpr int kOutExp = 2 * kPad - 2 * kBits - kBits * (kS - 1);

// S 2^(E + F + X) rounded once to the nearest double (ties to even), S the two's complement pair (hi, lo)
// with |S| < 2^126, without branches: |S| is normalised by its leading-zero count, the top 53 bits are
// rounded from the round bit and the sticky bits, and the exponent is added into the bit pattern, so a
// rounding carry moves into it.  Sets `rare` where the result falls outside the normal range (never with
// these operands; the caller then takes output_value), NaN for a row or column with an inf or NaN.
template <int X>
__device__ __forceinline__ double s128_to_f64(long long hi, unsigned long long lo, int E, int F, bool &rare) {
  const unsigned long long sg = (unsigned long long)(hi >> 63);  // all ones when S < 0
  const unsigned long long ml = (lo ^ sg) - sg;                   // |S|, low word
  const unsigned long long mh = ((unsigned long long)hi ^ sg) + (sg & (ml == 0 ? 1ull : 0ull));
  const bool top = mh != 0;
  const int lz = top ? __clzll((long long)mh) : 64 + __clzll((long long)ml);
  const unsigned long long hN = top ? mh : ml, lN = top ? ml : 0ull;
  const int s1 = lz & 63;
  const unsigned long long N = (hN << s1) | ((lN >> 1) >> (63 - s1));  // the leading 64 bits
  const unsigned long long rest = lN << s1;
  const unsigned long long mant = N >> 11;
  const unsigned long long inc = ((N >> 10) & 1ull) & ((((N & 0x3ffull) | rest) != 0 ? 1ull : 0ull) | (mant & 1ull));
  const int ex = 127 - lz + E + F + X;  // exponent of the leading bit
  unsigned long long bits = (((unsigned long long)(ex + 1022) << 52) + mant + inc) | (sg << 63);
  const bool nonfinite = E >= kNonFinite || F >= kNonFinite, zero = lz == 128;
  rare |= !nonfinite && !zero && (unsigned)(ex + 1022) > 2045u;
  bits = zero ? 0ull : bits;
  bits = nonfinite ? 0x7ff8000000000000ull : bits;
  return __longlong_as_double((long long)bits);
}

// output_value without branches, for the wide epilogues: the nine diagonal sums become
// S = T 2^36 + M 2^18 + L (T, M, L each three diagonals, |.| < 2^36.03) as a 128-bit two's complement
// pair, rounded by s128_to_f64.  Equal to output_value(diag_int(v, c), E, F) except where `rare` is set:
// the caller then takes output_value for the group, after all of its outputs, so that no call or branch
// sits between their independent instruction chains (measured: a call site inside each conversion made
// it 3.5 times slower).
template <int W>
__device__ __forceinline__ void diag_s128(const float (&v)[kS][W], int c, long long &hi, unsigned long long &lo) {
  static_assert(kS == 9 && kBits == 6, "three groups of three 6-bit diagonals");
  int x[kS];
#pragma unroll
  for (int d = 0; d < kS; ++d) x[d] = exact_int(v[d][c]);
  const long long T = (long long)x[0] * 4096 + (long long)x[1] * 64 + x[2];
  const long long M = (long long)x[3] * 4096 + (long long)x[4] * 64 + x[5];
  const long long L = (long long)x[6] * 4096 + (long long)x[7] * 64 + x[8];
  const long long A = M * 262144 + L;  // |A| < 2^55
  const unsigned long long tl = (unsigned long long)T << 36;
  lo = tl + (unsigned long long)A;
  hi = (T >> 28) + (A >> 63) + (lo < tl ? 1 : 0);
}
template <int W>
__device__ __forceinline__ double diag_to_f64(const float (&v)[kS][W], int c, int E, int F, bool &rare) {
  long long hi;
  unsigned long long lo;
  diag_s128(v, c, hi, lo);
  return s128_to_f64<kOutExp>(hi, lo, E, F, rare);
}

// The 7 x 8-bit scheme (Digits7x8): seven diagonal sums, diagonal d weighing 256^-(d+2), as one exact
// integer S = sum_d v[d][c] 2^(8 (6 - d)), |S| < 2^72.01; an output is S 2^(E + F + kOutExp7x8).
constexpr int kOutExp7x8 = 2 * Digits7x8::kPad - 2 * 8 - 8 * 6;
// Its parts, S = T 2^32 + A, |T| < 2^40.01, |A| < 2^48.01.
template <int W>
__device__ __forceinline__ void diag7_parts(const float (&v)[7][W], int c, long long &T, long long &A) {
  int x[7];
#pragma unroll
  for (int d = 0; d < 7; ++d) x[d] = exact_int(v[d][c]);
  T = (long long)x[0] * 65536 + (long long)x[1] * 256 + x[2];
  A = (long long)x[3] * 16777216 + (long long)x[4] * 65536 + (long long)x[5] * 256 + x[6];
}

// The rare case of diag_to_f64 (a result outside the normal range), out of line so that the epilogue
// loops stay small: one output from its diagonal sums.
__device__ __noinline__ double output_value_rare(float v0, float v1, float v2, float v3, float v4, float v5, float v6,
                                                 float v7, float v8, int E, int F) {
  const float v[kS][1] = {{v0}, {v1}, {v2}, {v3}, {v4}, {v5}, {v6}, {v7}, {v8}};
  return output_value(diag_int(v, 0), E, F);
}

// split_rows_kernel with the row exponents found in the same kernel: one warp per group of 8 rows and
// all of K (lane = (row ri8 = lane / 4, pair of k kp = lane % 4)), a first pass over the rows for their
// largest exponents (reduced over the row's four lanes), a second for the digits.  For short rows
// (the tabulation's dT^T, K = M1 <= 256), where a launch per pass costs more than the passes.  Also G with
// sum_k |x_rk| < 2^G per row, G >= E (gexps; kNonFinite for a row with an inf or NaN).  A row of zeros (a plane of
// atoms, a masked gradient) gets the exponent of ordinary data: as the least one it sent every row of the atom out of
// the rows kernel's fast conversion (3,000 atoms of water, one component zero: the backward 131 us, 147 so).
constexpr int kZerosGrad = 0;  // the exponent of a column of zeros of dT^T
template <class D>
__global__ void __launch_bounds__(128) split_rows_1k_kernel(const double *__restrict__ X, int64_t ld_r, int64_t ld_k,
                                                            int64_t nrows, int K, int64_t rows_p, int Kp, int RT,
                                                            unsigned char *__restrict__ planes, int *__restrict__ exps,
                                                            int *__restrict__ gexps) {
  constexpr int NS = D::kNS;
  const int lane = threadIdx.x & 31, ri8 = lane >> 2, kp = lane & 3;
  const int64_t g = (int64_t)blockIdx.x * 4 + (threadIdx.x >> 5);  // 8-row group
  if (g * 8 >= rows_p) return;                                      // warp-uniform
  const int64_t r = g * 8 + ri8;
  const double *__restrict__ xr = X + (r < nrows ? r : 0) * ld_r;
  auto x = [&](int k) { return (r < nrows && k < K) ? __ldg(xr + k * ld_k) : 0.0; };
  int eb = 0;
  for (int k0 = 0; k0 < Kp; k0 += 8) eb = max(eb, max(exp_bits(x(k0 + 2 * kp)), exp_bits(x(k0 + 2 * kp + 1))));
  eb = max(eb, __shfl_xor_sync(0xffffffffu, eb, 1));
  eb = max(eb, __shfl_xor_sync(0xffffffffu, eb, 2));
  bool any = eb != 0;
  if (__any_sync(0xffffffffu, !any)) {  // zeros, or subnormals?
    for (int k0 = 0; k0 < Kp; k0 += 8) any |= nonzero(x(k0 + 2 * kp)) || nonzero(x(k0 + 2 * kp + 1));
    any = (__ballot_sync(0xffffffffu, any) >> (lane & ~3) & 0xfu) != 0;
  }
  const int E = any ? exp_of_max(eb) : kZerosGrad;
  // the row's sum of magnitudes in units of 2^(E - 20), each rounded up: below 2^28 + 2^8
  unsigned mag = 0;
  for (int k0 = 0; k0 < Kp; k0 += 8)
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const unsigned hw = (unsigned)__double2hiint(x(k0 + 2 * kp + h)) & 0x7fffffffu;  // |x| < (1 + m) 2^-20 2^(e - 1023)
      mag += hw ? (((hw & 0xfffffu) + 0x100001u) >> min(max(E + 1023 - (int)(hw >> 20), 0), 31)) + 1u : 0u;
    }
  mag += __shfl_xor_sync(0xffffffffu, mag, 1);
  mag += __shfl_xor_sync(0xffffffffu, mag, 2);
  if (kp == 0) {
    exps[r] = E;
    gexps[r] = E >= kNonFinite ? kNonFinite : max(E, E - 20 + 32 - __clz((int)mag));
  }
  const size_t plane = (size_t)RT * kTK * 2, block = NS * plane;
  const int ri = (int)(r % RT);
  unsigned char *rowbase = planes + (size_t)(r / RT) * (Kp / kTK) * block + (ri >> 3) * kSBO + (ri & 7) * 16 + kp * 4;
  for (int k0 = 0; k0 < Kp; k0 += 8) {
    const int k = k0 + 2 * kp;
    uint32_t h[NS];
    digit_pairs<D>(biased_fixed<D>(x(k), E), biased_fixed<D>(x(k + 1), E), h);
    unsigned char *dst = rowbase + (size_t)(k0 / kTK) * block + ((k0 % kTK) >> 3) * kLBO;
#pragma unroll
    for (int s = 0; s < NS; ++s) *reinterpret_cast<uint32_t *>(dst + s * plane) = h[s];
  }
}

template <class D>
int split_rows_1k(const double *X, int64_t ld_r, int64_t ld_k, int64_t nrows, int K, int64_t rows_p, int Kp, int RT,
                  unsigned char *planes, unsigned char *exps, int *gexps, cudaStream_t st, const char *who) {
  split_rows_1k_kernel<D><<<(unsigned)((rows_p / 8 + 3) / 4), 128, 0, st>>>(
      X, ld_r, ld_k, nrows, K, rows_p, Kp, RT, planes, reinterpret_cast<int *>(exps), gexps);
  return launch_status(who);
}

// zeros: the exponent of a row of zeros.  The plan's say that a coefficient is nowhere large (key_exps).
constexpr int kZerosPlan = -1021;
template <class D = Digits9x6>
int split_rows(const double *X, int64_t ld_r, int64_t ld_k, int64_t nrows, int K, int64_t rows_p, int Kp, int RT,
               unsigned char *planes, unsigned char *exps, cudaStream_t st, const char *who, int zeros = kZerosPlan) {
  row_exps_kernel<<<(unsigned)((rows_p + 3) / 4), 128, 0, st>>>(X, ld_r, ld_k, nrows, K, rows_p, zeros,
                                                                 reinterpret_cast<int *>(exps));
  int rc = launch_status(who);
  if (rc) return rc;
  const int64_t warps = rows_p / 8 * ((Kp + kSplitK - 1) / kSplitK);
  split_rows_kernel<D><<<(unsigned)((warps + 3) / 4), 128, 0, st>>>(X, ld_r, ld_k, nrows, K, rows_p, Kp, RT, planes,
                                                                 reinterpret_cast<const int *>(exps));
  return launch_status(who);
}
}  // namespace tc
}  // namespace
}  // namespace dpc
