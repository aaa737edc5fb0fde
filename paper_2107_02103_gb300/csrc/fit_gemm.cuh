// Persistent exact-f64 GEMM of the fitting net on the tcgen05 tensor cores, every centre type of a layer in
// one launch, with the layer's epilogue in it.
//
// A layer is C = A B per centre type: A the atoms' inputs (128-row tiles, a type's rows in tiles of their
// own), B the type's weights.  Both are split into eight balanced 7-bit digits (Digits8x7 of tc_gemm.cuh: 36
// digit products an output where nine 6-bit digits take 45; 55 binary places instead of 53), exact in fp32
// over a share of 512 of K.  One CTA per SM walks the units (128 rows, 64 columns, share of K) round-robin:
// warp 0 copies each slice's A and B blocks into a ring of four stages, lane 0 of warp 1 issues the slice's
// 12 MMAs, and 16 epilogue warps (four per TMEM lane quadrant, 16 columns each) read the unit's eight
// diagonals, recombine them exactly as a 128-bit integer, round once to f64 and apply the layer's epilogue
// (bias, tanh, skip; or the skip term and dE/dz) -- or, where K takes several shares, store the integers for
// fit_reduce_kernel to add.  The copies of the next unit run during the epilogue.
// Why: with a CTA per tile, four floats an output through memory and a kernel to finish them, the 240-wide
// GEMMs kept the tensor cores busy a third of the time and the epilogues took half as long as the GEMMs;
// launches per type and layer set the time of small systems.  64 columns a tile: a slice's copies are 12 % fewer
// bytes a column than with 48, and 4,096 atoms make 128 tiles of a 240-wide layer, one per SM, not 160.
// Measured, forward and backward of a 1600-240-240-240-1 net with every other kernel of theirs: 12,288 atoms
// of two types 2.19 -> 1.25 ms; a vector model's step on 192 atoms 0.92 -> 0.45 ms (102 -> 46 launches).
// What bounds it now (12,288 atoms, a backward's 1600-wide layer): of 18 us a tile 5 are copies alone, 12 with the
// MMAs, 6 the conversions that hold the accumulators; the rest runs beside the next tile.
// Every wait is bounded; a wait that gives up stops the CTA's copies and MMAs, its remaining outputs are NaN
// and one timeout is counted (dp_tc_wait_timeouts).
#pragma once

#include "tc_gemm.cuh"

namespace dpc {
namespace {
namespace tf {
using namespace tc;

using DF = Digits8x7;
constexpr int kSF = DF::kNS;
constexpr int kTNF = 64, kStagesF = 4;
constexpr int kPlaneAF = kTM * kTK * 2, kPlaneBF = kTNF * kTK * 2;
constexpr int kStageBytesF = kSF * (kPlaneAF + kPlaneBF);
constexpr int kMaxSharesK = 512 / kTK;  // slices of one exact share
constexpr int kPlanesPerMmaF = 256 / kTNF;
constexpr int kEpiWarpsF = 16, kThreadsF = 32 * (2 + kEpiWarpsF);
constexpr int kEpiColsF = 4 * kTNF / kEpiWarpsF;  // columns per epilogue warp, four warps to a lane quadrant
static_assert((long long)kSF * 64 * 64 * kMaxSharesK * kTK <= (1ll << 24), "exact fp32 diagonal sums");
static_assert(kSF * kTNF <= (int)kTmemCols, "accumulators");
constexpr size_t kBarOffF = (size_t)kStagesF * kStageBytesF;  // full, empty, acc_full, tmem_free
constexpr size_t kMiscOffF = kBarOffF + (2 * kStagesF + 2) * 8;
constexpr size_t kSmemF = kMiscOffF + 32;
static_assert(kSmemF <= 227 * 1024, "shared memory per block");

// The rows of a launch: 128-row tiles, those of type t being tiles t0[t] .. t0[t + 1] - 1 of the batch, of
// which the launch takes `tiles` from tile0 on.
struct Tiles {
  int ntypes, tile0, tiles;
  int t0[DP_MAX_TYPES + 1];
  int64_t start[DP_MAX_TYPES + 1];  // first atom of each type
};
struct TileRows {
  int type;      // within the batch
  int64_t row0;  // first atom
  int rows;
};
__device__ __forceinline__ TileRows tile_rows(const Tiles &G, int tile) {
  int t = 0;
  for (int q = 1; q < G.ntypes; ++q)
    if (tile >= G.t0[q]) t = q;
  TileRows R;
  R.type = t;
  R.row0 = G.start[t] + (int64_t)(tile - G.t0[t]) * kTM;
  R.rows = (int)min((int64_t)kTM, G.start[t + 1] - R.row0);
  return R;
}

// One entry of the table that tanh_tab below reads: T_j as f64 and as a float pair, S_j = 1 - T_j^2 as a pair.
constexpr int kTanhSteps = 32, kTanhEntries = 20 * kTanhSteps;
struct alignas(16) TanhEntry {
  double T;
  float Th, Tl, Sh, Sl, pad[2];
};

// A layer's epilogue.  Forward: z = acc + bias; lin: V = z; else t = tanh z, act = t, V = t (+ A: the skip).
// Backward: s = acc (+ S or g wo where the layer kept its width); out = s, or Snext = s and
// Z = s (1 - T^2).  Weights of type t lie pstride apart.
struct Epilogue {
  int N;
  int64_t pstride;
  const double *bias, *wo;
  const double *A, *S, *g, *T;
  int64_t lda, ldS, ldT;
  double *act, *V, *Snext, *Z, *out;
  int64_t ldact, ldv, ldz, ldo;
  bool skip, lin;
  const TanhEntry *tanh_table;
};

// tanh from a table of T_j = tanh(j / 32) and S_j = 1 - T_j^2:
//   |x| = j / 32 + d,  |d| <= 1/64,  tanh|x| = T_j + S_j t / (1 + T_j t),
//   t = tanh d = d + d z (-1/3 + z (2/15 - 17/315 z)),  z = d^2  (the next term is 2^-53 of t),
// d and the last sum in f64, the correction (at most 1/64) in float pairs on the FP32 pipes: a quarter of the
// instructions of dfl::tanh_d's degree-13 expm1, and more exact (its error is 2^-47 of the correction, not of
// the result).  j = 0 keeps small arguments' relative accuracy.
__device__ __forceinline__ double tanh_tab(double x, const TanhEntry *__restrict__ tab) {
  const double ax = fabs(x);
  const int h = __double2hiint(ax);
  if (h >= 0x40331999) return (h > 0x7ff00000 || (h == 0x7ff00000 && __double2loint(x))) ? x : copysign(1.0, x);  // 19.1
  if (h < 0x3bc79ca1) return x;  // below 1e-20
  const float af = __uint_as_float((unsigned)(h - 0x38000000) << 3 | (unsigned)__double2loint(ax) >> 29);  // truncated
  const int j = __float2int_rn(af * (float)kTanhSteps);
  const int4 e0 = __ldg(reinterpret_cast<const int4 *>(tab + j));
  const float2 S = __ldg(reinterpret_cast<const float2 *>(tab + j) + 2);
  const float Th = __int_as_float(e0.z), Tl = __int_as_float(e0.w);
  const dfl::df64 d = dfl::split(__dsub_rn(ax, dfl::widen((float)j * (1.0f / kTanhSteps))));  // exact
  const float dh = d.hi, dl = d.lo;
  // z = d^2, s = -1/3 + z (2/15 - 17/315 z), w = z s
  const float zh = __fmul_rn(dh, dh), zl = __fmaf_rn(__fadd_rn(dh, dh), dl, __fmaf_rn(dh, dh, -zh));
  const float q = __fmul_rn(zh, __fmaf_rn(zh, -0.053968254f, 0.13333334f));
  const float sh = __fadd_rn(-0.33333334f, q), sl = __fadd_rn(__fsub_rn(q, __fadd_rn(sh, 0.33333334f)), 9.9341075e-09f);
  const float wh = __fmul_rn(zh, sh), wl = __fmaf_rn(zl, sh, __fmaf_rn(zh, sl, __fmaf_rn(zh, sh, -wh)));
  // t = d + d w
  const float ph = __fmul_rn(dh, wh), pl = __fmaf_rn(dl, wh, __fmaf_rn(dh, wl, __fmaf_rn(dh, wh, -ph)));
  const float th = __fadd_rn(dh, ph), tl = __fadd_rn(__fadd_rn(__fsub_rn(ph, __fsub_rn(th, dh)), dl), pl);
  // S t over 1 + T t
  const float nh = __fmul_rn(S.x, th), nl = __fmaf_rn(S.y, th, __fmaf_rn(S.x, tl, __fmaf_rn(S.x, th, -nh)));
  const float mh = __fmul_rn(Th, th), ml = __fmaf_rn(Tl, th, __fmaf_rn(Th, tl, __fmaf_rn(Th, th, -mh)));
  const float eh = __fadd_rn(1.0f, mh), el = __fadd_rn(__fsub_rn(mh, __fsub_rn(eh, 1.0f)), ml);
  const float r = __frcp_rn(eh), q0 = __fmul_rn(nh, r);
  const float rem = __fadd_rn(__fmaf_rn(-q0, eh, nh), __fmaf_rn(-q0, el, nl));
  const double c = dfl::join(dfl::df64(q0, __fmul_rn(rem, r)));
  return copysign(__dadd_rn(__hiloint2double(e0.y, e0.x), c), x);
}

// Four tanhs side by side (measured, a 240-wide layer of 12,288 atoms: 0.106 ms; as a function of its own,
// called, 0.120).
__device__ __forceinline__ void tanh4(double &a, double &b, double &c, double &d, const TanhEntry *tab) {
  const double x = tanh_tab(a, tab), y = tanh_tab(b, tab), z = tanh_tab(c, tab), w = tanh_tab(d, tab);
  a = x, b = y, c = z, d = w;
}

__device__ __forceinline__ void store4(double *p, const double (&v)[4], int cnt) {
  if (cnt == 4 && (reinterpret_cast<uintptr_t>(p) & 15) == 0) {
    reinterpret_cast<double2 *>(p)[0] = make_double2(v[0], v[1]);
    reinterpret_cast<double2 *>(p)[1] = make_double2(v[2], v[3]);
  } else {
#pragma unroll
    for (int c = 0; c < 4; ++c)
      if (c < cnt) p[c] = v[c];
  }
}

// Columns n .. n + cnt - 1 (cnt <= 4) of one atom.  (Read-only loads: no input is an output of the same launch,
// and a group's loads may so pass the stores of the one before.)
template <bool kFwd>
__device__ __forceinline__ void finish4(const Epilogue &E, int type, int64_t row, int n, int cnt, double (&v)[4]) {
  if constexpr (kFwd) {
    const double *bias = E.bias + type * E.pstride + n;
#pragma unroll
    for (int c = 0; c < 4; ++c)
      if (c < cnt) v[c] += __ldg(bias + c);
    if (!E.lin) {
      tanh4(v[0], v[1], v[2], v[3], E.tanh_table);
      store4(E.act + row * E.ldact + n, v, cnt);
      if (E.skip)
#pragma unroll
        for (int c = 0; c < 4; ++c)
          if (c < cnt) v[c] += __ldg(E.A + row * E.lda + n + c);
    }
    store4(E.V + row * E.ldv + n, v, cnt);
  } else {
    if (E.skip) {
      const double g = E.S ? 0.0 : (E.g ? __ldg(E.g + row) : 1.0);
#pragma unroll
      for (int c = 0; c < 4; ++c)
        if (c < cnt) v[c] += E.S ? __ldg(E.S + row * E.ldS + n + c) : g * __ldg(E.wo + type * E.pstride + n + c);
    }
    if (E.T) {
      store4(E.Snext + row * E.ldz + n, v, cnt);
#pragma unroll
      for (int c = 0; c < 4; ++c)
        if (c < cnt) {
          const double t = __ldg(E.T + row * E.ldT + n + c);
          v[c] *= fma(-t, t, 1.0);
        }
      store4(E.Z + row * E.ldz + n, v, cnt);
    } else {
      store4(E.out + row * E.ldo + n, v, cnt);
    }
  }
}

struct Gemm {
  Tiles G;
  Epilogue E;
  int nt, ka, ks, per;           // column tiles, K slices, shares and slices per share
  const unsigned char *aplanes;  // [tiles][ka] blocks
  const int *Eexp;               // [128 tiles]
  const unsigned char *bplanes;  // of type t at t bstride: [nt][ka] blocks
  const int *Fexp;               // of type t at t fstride: [64 nt]
  size_t bstride, fstride;
  longlong2 *part;               // ks > 1: [ks][64 nt][128 tiles] exact integers (lo, hi); hi kPartBad: NaN
};
constexpr long long kPartBad = 1ll << 62;

// The eight diagonal sums of one output (exact integers up to 2^24; diagonal d weighs 128^-(d+2)) as one
// exact integer S = sum_d v[d] 2^(7 (7 - d)), two's complement; an output is S 2^(E + F + kOutExpF).
constexpr int kOutExpF = 2 * DF::kPad - 2 * DF::kNB - DF::kNB * (kSF - 1);
__device__ __forceinline__ void diag8_s128(const float (&v)[kSF][4], int c, long long &hi, unsigned long long &lo) {
  static_assert(kSF == 8 && DF::kNB == 7, "groups of three, three and two 7-bit diagonals");
  int x[kSF];
#pragma unroll
  for (int d = 0; d < kSF; ++d) x[d] = exact_int(v[d][c]);
  const long long T = (long long)x[0] * 16384 + (long long)x[1] * 128 + x[2];  // below 2^38.1
  const long long M = (long long)x[3] * 16384 + (long long)x[4] * 128 + x[5];
  const long long A = M * 16384 + ((long long)x[6] * 128 + x[7]);  // below 2^53
  const unsigned long long tl = (unsigned long long)T << 35;
  lo = tl + (unsigned long long)A;
  hi = (T >> 29) + (A >> 63) + (lo < tl ? 1 : 0);
}
// The same output rounded once to f64, times 2^e, on the FP64 pipe: the sum's two parts are exact doubles.
// `rare` where the exponents could leave the normal range, or belong to a row or column with an inf or NaN.  A zero
// is not: padding rows, and the rows of atoms without a gradient, have the least exponent (with one of them in each
// warp the GEMM's outputs went through output_any: 12,288 atoms' backward 0.38 ms, 0.46 so).
__device__ __forceinline__ double diag8_fp64(const float (&v)[kSF][4], int c, int e, bool &rare) {
  int x[kSF];
#pragma unroll
  for (int d = 0; d < kSF; ++d) x[d] = exact_int(v[d][c]);
  const long long T = (long long)x[0] * 16384 + (long long)x[1] * 128 + x[2];
  const long long M = (long long)x[3] * 16384 + (long long)x[4] * 128 + x[5];
  const double s = __fma_rn((double)T, 0x1p35, (double)(M * 16384 + ((long long)x[6] * 128 + x[7])));
  const bool zero = __double2hiint(s) == 0;  // (an integer)
  rare |= zero ? e > kNonFinite / 2 : abs(e) > 900;
  return zero ? 0.0 : __hiloint2double(__double2hiint(s) + (e << 20), __double2loint(s));
}
// A result outside the normal range (s128_to_f64's rare case), out of line.
__device__ __noinline__ double output_any(long long hi, unsigned long long lo, int E, int F) {
  if (E >= kNonFinite || F >= kNonFinite) return __longlong_as_double(0x7ff8000000000000ll);
  return i128_to_double((__int128)(((unsigned __int128)(unsigned long long)hi << 64) | lo), E + F + kOutExpF);
}
template <bool kFwd>
__global__ void __launch_bounds__(kThreadsF, 1) fit_gemm_kernel(const Gemm P) {
  extern __shared__ __align__(1024) unsigned char smem[];
  uint64_t *full = reinterpret_cast<uint64_t *>(smem + kBarOffF);
  uint64_t *empty = full + kStagesF;
  uint64_t *acc_full = empty + kStagesF;
  uint64_t *tmem_free = acc_full + 1;
  uint32_t *tmem_holder = reinterpret_cast<uint32_t *>(smem + kMiscOffF);
  volatile int *abortf = reinterpret_cast<volatile int *>(smem + kMiscOffF + 4);
  volatile int *uflag = reinterpret_cast<volatile int *>(smem + kMiscOffF + 8);  // the unit's accumulators are ready
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int nunits = P.G.tiles * P.nt * P.ks;

  if (tid == 0) {
    for (int s = 0; s < kStagesF; ++s) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(full + s)));
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(empty + s)));
    }
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(acc_full)));
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(tmem_free)), "r"(kEpiWarpsF));
    asm volatile("fence.mbarrier_init.release.cluster;");
    *abortf = 0;
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_holder)),
                 "r"(kTmemCols));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;");
  const uint32_t tmem = *tmem_holder;
  const uint32_t sbase = smem_u32(smem);
  // unit u: column tile u % nt (the CTAs at work together share A tiles), share, row tile
  auto slices_of = [&](int sh) { return min(P.per, P.ka - sh * P.per); };

  int issued = 0;  // thread 0: slices whose copies it started; thread 32: its commits on acc_full
  if (warp == 0) {
    // ---- producer
    if (lane == 0) {
      int &g = issued;
      bool ok = true;
      for (int u = blockIdx.x; u < nunits && ok; u += gridDim.x) {
        const int n = u % P.nt, r = u / P.nt, sh = r % P.ks, mt = r / P.ks;
        const int type = tile_rows(P.G, P.G.tile0 + mt).type;
        const unsigned char *a0 = P.aplanes + (size_t)mt * P.ka * (kSF * kPlaneAF);
        const unsigned char *b0 = P.bplanes + type * P.bstride + (size_t)n * P.ka * (kSF * kPlaneBF);
        const int ns = slices_of(sh);
        for (int j = 0; j < ns; ++j, ++g) {
          const int st = g % kStagesF;
          if (g >= kStagesF && !(ok = wait_or_abort(smem_u32(empty + st), (uint32_t)((g / kStagesF - 1) & 1), abortf)))
            break;
          const size_t sl = (size_t)sh * P.per + j;
          const uint32_t bar = smem_u32(full + st), dst = sbase + st * kStageBytesF;
          asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"((uint32_t)kStageBytesF)
                       : "memory");
          asm volatile(
              "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
              "l"(a0 + sl * (kSF * kPlaneAF)), "r"((uint32_t)(kSF * kPlaneAF)), "r"(bar)
              : "memory");
          asm volatile(
              "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                  dst + kSF * kPlaneAF),
              "l"(b0 + sl * (kSF * kPlaneBF)), "r"((uint32_t)(kSF * kPlaneBF)), "r"(bar)
              : "memory");
        }
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    // ---- MMA issuer: digit s of A against B's digits t <= 7 - s, up to four planes an MMA, the
    // accumulator moved by s + t diagonals (see tab_gemm.cuh)
    if (lane == 0) {
      int g = 0, &li = issued;
      bool ok = true;
      for (int u = blockIdx.x; u < nunits && ok; u += gridDim.x, ++li) {
        if (li > 0 && !(ok = wait_or_abort(smem_u32(tmem_free), (uint32_t)((li - 1) & 1), abortf))) break;
        asm volatile("tcgen05.fence::after_thread_sync;");
        const int ns = slices_of(u / P.nt % P.ks);
        for (int j = 0; j < ns; ++j, ++g) {
          const int st = g % kStagesF;
          if (!(ok = wait_or_abort(smem_u32(full + st), (uint32_t)((g / kStagesF) & 1), abortf))) break;
          asm volatile("tcgen05.fence::after_thread_sync;");
          const uint64_t a0 = smem_desc(sbase + st * kStageBytesF);
          const uint64_t b0 = smem_desc(sbase + st * kStageBytesF + kSF * kPlaneAF);
#pragma unroll
          for (int s = 0; s < kSF; ++s) {
#pragma unroll
            for (int t0 = 0; t0 < kSF - s; t0 += kPlanesPerMmaF) {
              const int np = min(kPlanesPerMmaF, kSF - s - t0);
              const uint32_t idesc = kIdescNoN | ((uint32_t)((np * kTNF) >> 3) << 17);
              const uint32_t acc = (j > 0 || s > 0) ? 1u : 0u;  // a unit's first digit product writes every diagonal
              asm volatile(
                  "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
                  " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(tmem + (uint32_t)((s + t0) * kTNF)),
                  "l"(a0 + (uint64_t)((s * kPlaneAF) >> 4)), "l"(b0 + (uint64_t)((t0 * kPlaneBF) >> 4)), "r"(idesc),
                  "r"(acc));
            }
          }
          asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
              smem_u32(empty + st)));
        }
        // completes when every MMA issued so far has (also after a wait that gave up)
        asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
            smem_u32(acc_full)));
      }
    }
    __syncwarp();
  } else {
    // ---- epilogue: warps 2 .. 17, TMEM lane quadrant warp % 4, columns 16 ((warp - 2) / 4) .. + 15
    const int q = warp & 3, c_lo = ((warp - 2) / 4) * kEpiColsF, rl = 32 * q + lane;
    const uint32_t trow = tmem + ((uint32_t)(32 * q) << 16);
    int li = 0;
    for (int u = blockIdx.x; u < nunits; u += gridDim.x, ++li) {
      const int n = u % P.nt, r = u / P.nt, sh = r % P.ks, mt = r / P.ks;
      if (tid == 64) *uflag = !*abortf && wait_or_abort(smem_u32(acc_full), (uint32_t)(li & 1), abortf);
      asm volatile("bar.sync 1, %0;" ::"r"(32 * kEpiWarpsF) : "memory");
      const bool ok = *uflag != 0;
      asm volatile("tcgen05.fence::after_thread_sync;");
      const TileRows R = tile_rows(P.G, P.G.tile0 + mt);
      const int Erow = P.Eexp[mt * kTM + rl];
      const int *F = P.Fexp + R.type * P.fstride + n * kTNF;
      auto load = [&](int c0, float (&v)[kSF][4]) {
        if (ok) {  // uniform over the CTA
#pragma unroll
          for (int d = 0; d < kSF; ++d)
            asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
                         : "=f"(v[d][0]), "=f"(v[d][1]), "=f"(v[d][2]), "=f"(v[d][3])
                         : "r"(trow + (uint32_t)(d * kTNF + c0)));
          asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
          for (int d = 0; d < kSF; ++d) asm volatile("" : "+f"(v[d][0]), "+f"(v[d][1]), "+f"(v[d][2]), "+f"(v[d][3]));
        } else {
#pragma unroll
          for (int d = 0; d < kSF; ++d) v[d][0] = v[d][1] = v[d][2] = v[d][3] = 0.f;
        }
      };
      auto release = [&]() {  // the next unit's MMAs may overwrite the accumulators
        asm volatile("tcgen05.fence::before_thread_sync;");
        __syncwarp();
        if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(tmem_free)) : "memory");
      };
      if (P.ks > 1) {
#pragma unroll 1
        for (int c0 = c_lo; c0 < c_lo + kEpiColsF; c0 += 4) {
          float v[kSF][4];
          load(c0, v);
          longlong2 *out = P.part + ((size_t)sh * P.nt * kTNF + n * kTNF + c0) * (P.G.tiles * kTM) + mt * kTM + rl;
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            long long hi;
            unsigned long long lo;
            diag8_s128(v, c, hi, lo);
            out[(size_t)c * (P.G.tiles * kTM)] = ok ? make_longlong2((long long)lo, hi) : make_longlong2(0, kPartBad);
          }
        }
        release();
      } else {
        // every column rounded to f64 first, so that the next unit's MMAs run beside the rest (memory, tanh)
        double val[kEpiColsF / 4][4];
        bool rare = false;
#pragma unroll
        for (int i = 0; i < kEpiColsF / 4; ++i) {
          const int c0 = c_lo + 4 * i;
          if (n * kTNF + c0 >= P.E.N) break;  // uniform
          float v[kSF][4];
          load(c0, v);
          // two outputs by integers, two on the FP64 pipe, side by side (a backward of 12,288 atoms: GEMMs
          // 0.468 ms; all by integers 0.495, one 0.475, three on the FP64 pipe 0.507)
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            const int Fc = __ldg(F + c0 + c);
            if (c >= 2) {
              val[i][c] = diag8_fp64(v, c, Erow + Fc + kOutExpF, rare);
            } else {
              long long hi;
              unsigned long long lo;
              diag8_s128(v, c, hi, lo);
              val[i][c] = s128_to_f64<kOutExpF>(hi, lo, Erow, Fc, rare);
            }
            if (!ok) val[i][c] = __longlong_as_double(0x7ff8000000000000ll);
          }
        }
        if (__any_sync(0xffffffffu, rare))  // apart, so that no call sits between the conversions above
#pragma unroll
          for (int i = 0; i < kEpiColsF / 4; ++i) {
            const int c0 = c_lo + 4 * i;
            if (n * kTNF + c0 >= P.E.N) break;
            float v[kSF][4];
            load(c0, v);
#pragma unroll
            for (int c = 0; c < 4; ++c) {
              long long hi;
              unsigned long long lo;
              diag8_s128(v, c, hi, lo);
              if (ok) val[i][c] = output_any(hi, lo, Erow, __ldg(F + c0 + c));
            }
          }
        release();
        if (rl < R.rows)
#pragma unroll
          for (int i = 0; i < kEpiColsF / 4; ++i) {
            const int col = n * kTNF + c_lo + 4 * i, cnt = min(4, P.E.N - col);
            if (cnt > 0) finish4<kFwd>(P.E, R.type, R.row0 + rl, col, cnt, val[i]);
          }
      }
      asm volatile("bar.sync 1, %0;" ::"r"(32 * kEpiWarpsF) : "memory");  // uflag is free
    }
  }

  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;");
  if (*abortf) {  // uniform
    if (tid == 0) settle_copies(smem_u32(full), kStagesF, issued);
    if (tid == 32 && issued > 0) settle(smem_u32(acc_full), (uint32_t)((issued - 1) & 1));
    __syncthreads();
  }
  if (tid == 0 && *abortf) atomicAdd(&g_wait_timeouts, 1u);
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols));
}

// ks > 1: the shares' integers of every output added and rounded once, then the epilogue.  A warp per 32 rows
// and four columns.
template <bool kFwd>
__global__ void __launch_bounds__(128) fit_reduce_kernel(const Gemm P) {
  const int lane = threadIdx.x & 31, nc = (P.E.N + 3) / 4;
  const int64_t w = (int64_t)blockIdx.x * 4 + (threadIdx.x >> 5);
  if (w >= (int64_t)P.G.tiles * 4 * nc) return;  // warp-uniform
  const int col = (int)(w % nc) * 4, m32 = (int)(w / nc), mt = m32 >> 2, mrow = m32 * 32 + lane;
  const TileRows R = tile_rows(P.G, P.G.tile0 + mt);
  const int rl = mrow - mt * kTM;
  if (rl >= R.rows) return;
  const int cnt = min(4, P.E.N - col);
  const size_t ld = (size_t)P.G.tiles * kTM, share = (size_t)P.nt * kTNF * ld;
  const int Erow = P.Eexp[mrow];
  const int *F = P.Fexp + R.type * P.fstride;
  double val[4];
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    val[c] = 0.0;
    if (c >= cnt) continue;
    const longlong2 *p = P.part + (size_t)(col + c) * ld + mrow;
    long long hi = 0;
    unsigned long long lo = 0;
    bool bad = false;
    for (int z = 0; z < P.ks; ++z) {
      const longlong2 x = p[z * share];
      const unsigned long long l = lo + (unsigned long long)x.x;
      hi += x.y + (l < lo ? 1 : 0);
      lo = l;
      bad = bad || x.y == kPartBad;
    }
    bool rare = false;
    val[c] = s128_to_f64<kOutExpF>(hi, lo, Erow, __ldg(F + col + c), rare);
    if (rare) val[c] = output_any(hi, lo, Erow, __ldg(F + col + c));
    if (bad) val[c] = __longlong_as_double(0x7ff8000000000000ll);
  }
  finish4<kFwd>(P.E, R.type, R.row0 + rl, col, cnt, val);
}

// ---- the operands' digit planes
// One group of eight rows by the block's NW warps, K shared out by 16s: first the rows' exponents (reduced
// over the row's four lanes and the warps), then the digits, a lane taking four consecutive k of its row.
// x4(k, v): the lane's row's elements k .. k + 3 (0 past its ends).
template <int NW, class X4>
__device__ __forceinline__ void split_group(X4 x4, int Kp, unsigned char *rowbase, size_t plane, int *exp_out) {
  __shared__ int red[NW][8];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, ri8 = lane >> 2, kq = lane & 3;
  int eb = 0;
#pragma unroll 2
  for (int k0 = kTK * warp; k0 < Kp; k0 += kTK * NW) {
    double v[4];
    x4(k0 + 4 * kq, v);
    eb = max(eb, max(max(exp_bits(v[0]), exp_bits(v[1])), max(exp_bits(v[2]), exp_bits(v[3]))));
  }
  eb = max(eb, __shfl_xor_sync(0xffffffffu, eb, 1));
  eb = max(eb, __shfl_xor_sync(0xffffffffu, eb, 2));
  if (kq == 0) red[warp][ri8] = eb;
  __syncthreads();
#pragma unroll
  for (int q = 0; q < NW; ++q) eb = max(eb, red[q][ri8]);
  const int E = exp_of_max(eb);
  if (warp == 0 && kq == 0) exp_out[ri8] = E;
  rowbase += ri8 * 16 + (kq >> 1) * kLBO + (kq & 1) * 8;
  const size_t block = kSF * plane;
#pragma unroll 2
  for (int k0 = kTK * warp; k0 < Kp; k0 += kTK * NW) {
    double v[4];
    x4(k0 + 4 * kq, v);
    uint32_t h[kSF], g[kSF];
    digit_pairs<DF>(biased_fixed<DF>(v[0], E), biased_fixed<DF>(v[1], E), h);
    digit_pairs<DF>(biased_fixed<DF>(v[2], E), biased_fixed<DF>(v[3], E), g);
    unsigned char *dst = rowbase + (size_t)(k0 / kTK) * block;
#pragma unroll
    for (int s = 0; s < kSF; ++s) *reinterpret_cast<uint2 *>(dst + s * plane) = make_uint2(h[s], g[s]);
  }
}
// Elements k .. k + 3 of a row of K, zeros past its end; 16-byte loads where the row allows them.
__device__ __forceinline__ void load4(const double *__restrict__ p, int64_t ld, int k, int K, bool wide, double (&v)[4]) {
  if (wide && k + 4 <= K) {
    const double2 a = __ldg(reinterpret_cast<const double2 *>(p + k)), b = __ldg(reinterpret_cast<const double2 *>(p + k) + 1);
    v[0] = a.x, v[1] = a.y, v[2] = b.x, v[3] = b.y;
  } else {
#pragma unroll
    for (int c = 0; c < 4; ++c) v[c] = k + c < K ? __ldg(p + (k + c) * ld) : 0.0;
  }
}

// The rows of A of a launch's tiles, a block per eight rows.  Source: X[row][k], or with wo or S given the
// last hidden layer's dz: s (1 - X^2), s = S[row][k] or g_row wo[k] (of the row's type).
struct SplitA {
  Tiles G;
  const double *X, *S, *g, *wo;
  int64_t ldx, ldS, pstride;
  int K, Kp;
  unsigned char *planes;
  int *exps;
};
template <int NW, bool kDz>
__global__ void __launch_bounds__(32 * NW) split_a_kernel(const SplitA P) {
  const int ri8 = (threadIdx.x & 31) >> 2;
  const int mt = blockIdx.x / (kTM / 8), g8 = blockIdx.x - mt * (kTM / 8);
  const TileRows R = tile_rows(P.G, P.G.tile0 + mt);
  const int rl = 8 * g8 + ri8;
  const bool valid = rl < R.rows;
  const int64_t row = R.row0 + (valid ? rl : 0);
  const double *xr = P.X + row * P.ldx;
  const double gr = kDz && !P.S && P.g ? P.g[row] : 1.0;
  const bool wide = (reinterpret_cast<uintptr_t>(xr) & 15) == 0;
  const int K = valid ? P.K : 0;
  auto x4 = [&](int k, double (&v)[4]) {
    load4(xr, 1, k, K, wide, v);
    if constexpr (kDz) {
#pragma unroll
      for (int c = 0; c < 4; ++c)
        if (k + c < K) {
          const double s = P.S ? __ldg(P.S + row * P.ldS + k + c) : gr * __ldg(P.wo + R.type * P.pstride + k + c);
          v[c] = s * fma(-v[c], v[c], 1.0);
        }
    }
  };
  split_group<NW>(x4, P.Kp, P.planes + (size_t)mt * (P.Kp / kTK) * (kSF * kPlaneAF) + (size_t)g8 * kSBO, kPlaneAF,
                  P.exps + mt * kTM + 8 * g8);
}

// The weights of every GEMM and type of a batch, a block per eight columns of B (blockIdx.y: the type).
constexpr int kMaxGemms = DP_MAX_LAYERS + 1;
struct SplitB {
  const double *params;  // the batch's first type's
  int64_t pstride;
  int count;
  int K[kMaxGemms], N[kMaxGemms], group0[kMaxGemms + 1];  // column groups of GEMM q: group0[q] ..
  int64_t woff[kMaxGemms];
  size_t planes[kMaxGemms], fexp[kMaxGemms];  // byte offsets in `work`
  size_t bstride;                             // bytes from type to type
  bool transposed;  // B[k][n] = W[n][k] (the backward: W's rows are the columns of B)
  unsigned char *work;
  TanhEntry *tanh_table;  // made by one block more (forward), or NULL
};
template <int NW>
__global__ void __launch_bounds__(32 * NW) split_b_kernel(const SplitB P) {
  if ((int)blockIdx.x == P.group0[P.count]) {
    if (blockIdx.y == 0)
      for (int j = threadIdx.x; j < kTanhEntries; j += blockDim.x) {
        TanhEntry e{};
        e.T = tanh((double)j / kTanhSteps);
        e.Th = (float)e.T;
        e.Tl = (float)(e.T - (double)e.Th);
        const double c = 1.0 / cosh((double)j / kTanhSteps), S = c * c;
        e.Sh = (float)S;
        e.Sl = (float)(S - (double)e.Sh);
        P.tanh_table[j] = e;
      }
    return;
  }
  int q = 0;
  for (int c = 1; c < P.count; ++c)
    if ((int)blockIdx.x >= P.group0[c]) q = c;
  const int g8 = blockIdx.x - P.group0[q], ri8 = (threadIdx.x & 31) >> 2;
  const int K = P.K[q], N = P.N[q], Kp = (int)round_up(K, kTK), n = 8 * g8 + ri8;
  const double *W = P.params + blockIdx.y * P.pstride + P.woff[q] + (n < N ? (P.transposed ? (int64_t)n * K : n) : 0);
  const int64_t ldk = P.transposed ? 1 : N;
  const bool wide = P.transposed && (reinterpret_cast<uintptr_t>(W) & 15) == 0;
  auto x4 = [&](int k, double (&v)[4]) { load4(W, ldk, k, n < N ? K : 0, wide, v); };
  unsigned char *base = P.work + blockIdx.y * P.bstride;
  const int tile = 8 * g8 / kTNF, r8 = g8 - tile * (kTNF / 8);
  split_group<NW>(x4, Kp, base + P.planes[q] + (size_t)tile * (Kp / kTK) * (kSF * kPlaneBF) + (size_t)r8 * kSBO, kPlaneBF,
                  reinterpret_cast<int *>(base + P.fexp[q]) + 8 * g8);
}

// E_i = v_i . wo + bo, the output layer of one output: a warp per atom, every type.
__global__ void __launch_bounds__(128) fit_energy_kernel(Tiles G, int64_t row0, int64_t n, const double *__restrict__ V,
                                                         int64_t ldv, int K, const double *__restrict__ wo,
                                                         int64_t pstride, double *__restrict__ E) {
  const int lane = threadIdx.x & 31;
  const int64_t i = (int64_t)blockIdx.x * 4 + (threadIdx.x >> 5);
  if (i >= n) return;  // warp-uniform
  const int64_t row = row0 + i;
  int t = 0;
  for (int q = 1; q < G.ntypes; ++q)
    if (row >= G.start[q]) t = q;
  const double *w = wo + t * pstride;
  double s = 0.0;
  for (int k = lane; k < K; k += 32) s = fma(V[row * ldv + k], __ldg(w + k), s);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (lane == 0) E[row] = s + w[K];
}

int set_smem(const char *who) {
  static std::atomic<unsigned long long> set_on{0};  // bit d: done on device d
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return set_error(DP_ERR_CUDA, "%s: %s", who, cudaGetErrorString(cudaGetLastError()));
  if (dev < 64 && (set_on.load(std::memory_order_acquire) >> dev & 1ull)) return DP_OK;
  for (const void *k : {(const void *)fit_gemm_kernel<true>, (const void *)fit_gemm_kernel<false>}) {
    const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemF);
    if (e != cudaSuccess) return set_error(DP_ERR_CUDA, "%s: %s", who, cudaGetErrorString(e));
  }
  if (dev < 64) set_on.fetch_or(1ull << dev, std::memory_order_acq_rel);
  return DP_OK;
}

}  // namespace tf
}  // namespace
}  // namespace dpc
