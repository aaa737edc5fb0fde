// Fitting net (Sec. II: the descriptor D_i is passed to a fully connected
// network that outputs the atomic energy E_i; E = sum_i E_i) and its
// backward dE/dD_i, for the atoms of each centre type with that type's net.
//
// A hidden layer is a GEMM over the atoms of one type, [n x a] x [a x b],
// with the bias and tanh fused into its epilogue; the output layer (width 1)
// is a dot product per atom.  The backward runs the layers in reverse, one
// GEMM each against the transposed weights, with d tanh / dz = 1 - tanh^2
// applied as the operand is loaded and the skip term added in the epilogue.
//
// Only the tanh outputs of the hidden layers are kept (act, an output of the
// forward): a layer's input is the sum of the tanh outputs of its run of
// equal-width layers (the skips telescope: v_l = t_l + v_{l-1}), formed as
// the operand is loaded.
//
// GEMM tiling: small output tiles (FitTile below), 256 threads, 16-deep
// slices of both operands staged in shared memory.  Every FMA
// instruction has its 32 lanes busy; the kernels are bound by the FP64 pipe
// (f64) or the FP32 pipe (f32, df64).
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <cstdint>

#include "dp_common.cuh"
#include "fit_gemm.cuh"

namespace dpc {
namespace {

// Output tile kBM x kBN per block, kTM x kTN per thread, 256 threads.
template <int BM, int BN, int TM, int TN>
struct Tile {
  static constexpr int kBM = BM, kBN = BN, kTM = TM, kTN = TN, kTX = BN / TN;  // kTX: threads across columns
  static_assert((BM / TM) * (BN / TN) == 256, "tile shape");
};
// By arithmetic and direction, measured on GB300 with the 240-wide nets of cu85 and water.  f64 is
// bound by the FP64 pipe alone, so its tiles are small: a type's few thousand atoms must still make
// many blocks per SM, or the SMs that get one block more than the others set the time (64 x 64
// tiles give 256 blocks for 4096 atoms on 152 SMs, 84 % at best; 16 x 16 tiles 3840, 97 %).  The
// backward's loader spends FP64 work on every element of A it stages (the factor 1 - t^2), once per
// column tile, so there wider tiles (16 x 48) pay for themselves.  df64 and f32 feed the FP32 pipes,
// where the shared-memory operand loads per product start to count: larger tiles.
template <typename real, bool kFwd>
struct FitTile {
  using T = Tile<16, 48, 1, 3>;
};
template <>
struct FitTile<double, true> {
  using T = Tile<16, 16, 1, 1>;
};
template <bool kFwd>
struct FitTile<float, kFwd> {
  using T = Tile<64, 64, 4, 4>;
};
template <>
struct FitTile<df64, true> {
  using T = Tile<32, 48, 2, 3>;
};
template <>
struct FitTile<df64, false> {
  using T = Tile<64, 64, 4, 4>;
};
constexpr int kBK = 16, kFitThreads = 256;
constexpr int kMaxChain = DP_MAX_LAYERS + 1;

// f64 and df64: tanh evaluated in double-float on the FP32 pipes (dfl::tanh_d), not on the FP64
// pipe, where a double tanh costs about a tenth of a 240-deep layer's products
__device__ __forceinline__ double tanh_r(const double z) { return dfl::tanh_d(z); }
__device__ __forceinline__ float tanh_r(const float z) { return tanhf(z); }
__device__ __forceinline__ df64 tanh_r(const df64 z) { return dfl::split(dfl::tanh_d(dfl::join(z))); }

template <typename real>
struct FitGemm {
  int64_t r0, n;  // the type's atoms: rows r0 .. r0 + n - 1
  int K, N;
  // forward operand: sum of nsrc row-major sources (D and/or tanh outputs), row strides lds
  const io_t<real> *src[kMaxChain];
  int64_t lds[kMaxChain];
  int nsrc;
  // backward operand: S (dE/dv, row stride ldS; NULL: S(i, o) = g_i wo[o]) times 1 - T^2
  const io_t<real> *S;
  int64_t ldS;
  const io_t<real> *g;   // [nloc] or NULL (= 1)
  const io_t<real> *wo;  // output-layer weights [K]
  const io_t<real> *T;
  int64_t ldT;
  const io_t<real> *W;     // forward: W [K][N] (wt: W [N][K] read as its transpose); backward: W [N][K] transposed
  const io_t<real> *bias;  // forward: [N], NULL (lin only) for none
  bool lin;                // forward: out = acc + bias, no tanh (an output layer of several outputs, or g W^T)
  bool wt;                 // forward: read W as [N][K]
  bool skip;               // backward: add S(i, n) (the layer had an identity skip)
  io_t<real> *out;
  int64_t ldo;
};

template <typename real, bool kFwd>
__device__ __forceinline__ real load_a(const FitGemm<real> &P, int64_t row, int k) {
  if constexpr (kFwd) {
    io_t<real> v = P.src[0][row * P.lds[0] + k];
    for (int s = 1; s < P.nsrc; ++s) v += P.src[s][row * P.lds[s] + k];
    return from_io<real>(v);
  } else {
    const real t = from_io<real>(P.T[row * P.ldT + k]);
    real s;
    if (P.S)
      s = from_io<real>(P.S[row * P.ldS + k]);
    else
      s = from_io<real>(P.g ? P.g[row] : io_t<real>(1)) * from_io<real>(P.wo[k]);
    return s * fma(-t, t, real(1));
  }
}

template <typename real, bool kFwd>
__device__ __forceinline__ real load_b(const FitGemm<real> &P, int k, int nn) {
  if constexpr (kFwd)
    return from_io<real>(P.wt ? P.W[(size_t)nn * P.K + k] : P.W[(size_t)k * P.N + nn]);
  else
    return from_io<real>(P.W[(size_t)nn * P.K + k]);
}

template <typename real, bool kFwd>
__global__ void __launch_bounds__(kFitThreads) fit_gemm_kernel(const FitGemm<real> P) {
  using TL = typename FitTile<real, kFwd>::T;
  constexpr int kBM = TL::kBM, kBN = TL::kBN, kTM = TL::kTM, kTN = TL::kTN, kTX = TL::kTX;
  __shared__ real As[kBK][kBM + 1];
  __shared__ real Bs[kBK][kBN];
  const int tx = threadIdx.x % kTX, ty = threadIdx.x / kTX;
  const int64_t m0 = (int64_t)blockIdx.y * kBM;
  const int n0 = blockIdx.x * kBN;
  real acc[kTM][kTN];
#pragma unroll
  for (int a = 0; a < kTM; ++a)
#pragma unroll
    for (int b = 0; b < kTN; ++b) acc[a][b] = real(0);
  for (int k0 = 0; k0 < P.K; k0 += kBK) {
    // A slice [kBM][kBK] and B slice [kBK][kBN], spread over the threads
    for (int e = threadIdx.x; e < kBM * kBK; e += kFitThreads) {
      const int am = e / kBK, ak = e - am * kBK;  // consecutive threads: consecutive k of one row
      const int64_t row = m0 + am;
      const int k = k0 + ak;
      As[ak][am] = (row < P.n && k < P.K) ? load_a<real, kFwd>(P, P.r0 + row, k) : real(0);
    }
    for (int e = threadIdx.x; e < kBK * kBN; e += kFitThreads) {
      const int bk = e / kBN, bn = e - bk * kBN;
      const int kb = k0 + bk, nb = n0 + bn;
      Bs[bk][bn] = (kb < P.K && nb < P.N) ? load_b<real, kFwd>(P, kb, nb) : real(0);
    }
    __syncthreads();
#pragma unroll
    for (int kk = 0; kk < kBK; ++kk) {
      real a[kTM], b[kTN];
#pragma unroll
      for (int q = 0; q < kTM; ++q) a[q] = As[kk][ty + (kBM / kTM) * q];
#pragma unroll
      for (int q = 0; q < kTN; ++q) b[q] = Bs[kk][tx + kTX * q];
#pragma unroll
      for (int p = 0; p < kTM; ++p)
#pragma unroll
        for (int q = 0; q < kTN; ++q) acc[p][q] = fma(a[p], b[q], acc[p][q]);
    }
    __syncthreads();
  }
  // epilogue: rows ty + (kBM / kTM) p, columns tx + kTX q (consecutive threads write consecutive columns)
#pragma unroll
  for (int p = 0; p < kTM; ++p) {
    const int64_t row = m0 + ty + (kBM / kTM) * p;
    if (row >= P.n) continue;
#pragma unroll
    for (int q = 0; q < kTN; ++q) {
      const int nn = n0 + tx + kTX * q;
      if (nn >= P.N) continue;
      real v = acc[p][q];
      if constexpr (kFwd) {
        if (P.lin)
          v = P.bias ? v + from_io<real>(P.bias[nn]) : v;
        else
          v = tanh_r(v + from_io<real>(P.bias[nn]));
      } else if (P.skip) {
        const int64_t r = P.r0 + row;
        v += P.S ? from_io<real>(P.S[r * P.ldS + nn])
                 : from_io<real>(P.g ? P.g[r] : io_t<real>(1)) * from_io<real>(P.wo[nn]);
      }
      P.out[(P.r0 + row) * P.ldo + nn] = to_io(v);
    }
  }
}

// Output layer: E_i = v_{L-1} . wo + bo, one warp per atom, lanes over the inputs.
template <typename real>
__global__ void __launch_bounds__(128) fit_out_kernel(const FitGemm<real> P, const io_t<real> *bo, io_t<real> *E) {
  const int lane = threadIdx.x & 31;
  const int64_t i = (int64_t)blockIdx.x * 4 + (threadIdx.x >> 5);
  if (i >= P.n) return;  // warp-uniform
  const int64_t row = P.r0 + i;
  real s = real(0);
  for (int k = lane; k < P.K; k += 32) s = fma(load_a<real, true>(P, row, k), from_io<real>(P.wo[k]), s);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += shfl_xor(s, o);
  if (lane == 0) E[row] = to_io(s + from_io<real>(bo[0]));
}

struct FitShape {
  int nlayer, ntypes, nout;  // nout = widths[nlayer], the outputs per atom
  int w[DP_MAX_LAYERS + 1];
  int64_t P;       // parameters per type
  int64_t H;       // sum of hidden widths (row length of act)
  int maxh;        // largest hidden width
  int64_t woff[DP_MAX_LAYERS + 1];  // offset of W_l in a type's parameters (l >= 1)
  int64_t aoff[DP_MAX_LAYERS + 1];  // column offset of hidden layer l in act
  int64_t start[DP_MAX_TYPES + 1];
};

// multi: whether the output layer may have several outputs (the FMA-pipe kernels); the tensor-core
// net has one (the energy).
int fit_shape(const int32_t *widths, int nlayer, int ntypes, const int64_t *type_start, FitShape *s,
              bool multi = false) {
  if (!widths || !type_start) return set_error(DP_ERR_NULL, "widths or type_start is NULL");
  if (nlayer < 1 || nlayer > DP_MAX_LAYERS)
    return set_error(DP_ERR_UNSUPPORTED, "nlayer = %d outside [1, %d]", nlayer, DP_MAX_LAYERS);
  if (ntypes < 1 || ntypes > DP_MAX_TYPES)
    return set_error(DP_ERR_UNSUPPORTED, "ntypes = %d outside [1, %d]", ntypes, DP_MAX_TYPES);
  if (!multi && widths[nlayer] != 1)
    return set_error(DP_ERR_SHAPE, "the output layer has width %d, not 1", widths[nlayer]);
  s->nout = widths[nlayer];
  s->nlayer = nlayer;
  s->ntypes = ntypes;
  s->P = 0;
  s->H = 0;
  s->maxh = 1;
  for (int l = 0; l <= nlayer; ++l) {
    if (widths[l] < 1 || widths[l] > (1 << 20)) return set_error(DP_ERR_SHAPE, "widths[%d] = %d", l, widths[l]);
    s->w[l] = widths[l];
  }
  for (int l = 1; l <= nlayer; ++l) {
    s->woff[l] = s->P;
    s->P += (int64_t)widths[l - 1] * widths[l] + widths[l];
    if (l < nlayer) {
      s->aoff[l] = s->H;
      s->H += widths[l];
      if (widths[l] > s->maxh) s->maxh = widths[l];
    }
  }
  for (int t = 0; t <= ntypes; ++t) {
    s->start[t] = type_start[t];
    if (t > 0 && type_start[t] < type_start[t - 1]) return set_error(DP_ERR_SHAPE, "type_start decreases");
  }
  if (type_start[0] != 0) return set_error(DP_ERR_SHAPE, "type_start[0] = %lld, not 0", (long long)type_start[0]);
  return DP_OK;
}

// Sources of the input of layer l (1 <= l <= nlayer): the tanh outputs of the run of
// equal-width layers that ends at l - 1, and D when that run reaches back to layer 0.
template <typename real>
void chain_sources(const FitShape &s, int l, const io_t<real> *D, const io_t<real> *act, FitGemm<real> &G) {
  G.nsrc = 0;
  int j = l - 1;
  while (true) {
    if (j == 0) {
      G.src[G.nsrc] = D;
      G.lds[G.nsrc++] = s.w[0];
      break;
    }
    G.src[G.nsrc] = act + s.aoff[j];
    G.lds[G.nsrc++] = s.H;
    if (s.w[j] != s.w[j - 1]) break;
    --j;
  }
}

template <typename real, bool kFwd>
int launch_gemm(const FitGemm<real> &G, cudaStream_t st, const char *who) {
  using TL = typename FitTile<real, kFwd>::T;
  const dim3 grid((unsigned)((G.N + TL::kBN - 1) / TL::kBN), (unsigned)((G.n + TL::kBM - 1) / TL::kBM));
  if (grid.y > 65535u) return set_error(DP_ERR_SHAPE, "%s: too many atoms of one type (%lld)", who, (long long)G.n);
  fit_gemm_kernel<real, kFwd><<<grid, kFitThreads, 0, st>>>(G);
  return launch_status(who);
}

template <typename real>
int fitting_fwd(const io_t<real> *params, const int32_t *widths, int nlayer, int ntypes, const int64_t *type_start,
                const io_t<real> *D, io_t<real> *E, io_t<real> *act, void *stream) {
  clear_error();
  FitShape s{};
  int rc = fit_shape(widths, nlayer, ntypes, type_start, &s, true);
  if (rc) return rc;
  const int64_t nloc = s.start[ntypes];
  if (nloc == 0) return DP_OK;
  if (!params || !D || !E || (s.H > 0 && !act)) return set_error(DP_ERR_NULL, "dp_fitting_fwd: NULL array");
  const cudaStream_t st = (cudaStream_t)stream;
  for (int t = 0; t < ntypes; ++t) {
    const int64_t n = s.start[t + 1] - s.start[t];
    if (n == 0) continue;
    const io_t<real> *pt = params + (size_t)t * s.P;
    FitGemm<real> G{};
    G.r0 = s.start[t];
    G.n = n;
    for (int l = 1; l < nlayer; ++l) {  // hidden layers
      G.K = s.w[l - 1];
      G.N = s.w[l];
      chain_sources<real>(s, l, D, act, G);
      G.W = pt + s.woff[l];
      G.bias = G.W + (size_t)G.K * G.N;
      G.out = act + s.aoff[l];
      G.ldo = s.H;
      rc = launch_gemm<real, true>(G, st, "dp_fitting_fwd");
      if (rc) return rc;
    }
    G.K = s.w[nlayer - 1];
    chain_sources<real>(s, nlayer, D, act, G);
    if (s.nout == 1) {  // E_i = v . wo + bo: a dot product per atom
      G.N = 1;
      G.wo = pt + s.woff[nlayer];
      fit_out_kernel<real><<<(unsigned)((n + 3) / 4), 128, 0, st>>>(G, G.wo + G.K, E);
      rc = launch_status("dp_fitting_fwd");
    } else {  // E_i = v W_out + b_out: a GEMM without tanh
      G.N = s.nout;
      G.W = pt + s.woff[nlayer];
      G.bias = G.W + (size_t)G.K * G.N;
      G.lin = true;
      G.out = E;
      G.ldo = s.nout;
      rc = launch_gemm<real, true>(G, st, "dp_fitting_fwd");
    }
    if (rc) return rc;
  }
  return DP_OK;
}

template <typename real>
int fitting_grad(const io_t<real> *params, const int32_t *widths, int nlayer, int ntypes, const int64_t *type_start,
                 const io_t<real> *act, const io_t<real> *g, io_t<real> *dD, io_t<real> *work, void *stream) {
  clear_error();
  FitShape s{};
  int rc = fit_shape(widths, nlayer, ntypes, type_start, &s, true);
  if (rc) return rc;
  const int64_t nloc = s.start[ntypes];
  if (nloc == 0) return DP_OK;
  if (!params || !dD || (s.H > 0 && !act) || ((nlayer > 2 || s.nout > 1) && !work))
    return set_error(DP_ERR_NULL, "dp_fitting_grad: NULL array");
  if (s.nout > 1 && !g) return set_error(DP_ERR_NULL, "dp_fitting_grad: g is NULL for a net of %d outputs", s.nout);
  const cudaStream_t st = (cudaStream_t)stream;
  io_t<real> *buf[2] = {work, work ? work + (size_t)nloc * s.maxh : nullptr};
  for (int t = 0; t < ntypes; ++t) {
    const int64_t n = s.start[t + 1] - s.start[t];
    if (n == 0) continue;
    const io_t<real> *pt = params + (size_t)t * s.P;
    FitGemm<real> G{};
    G.r0 = s.start[t];
    G.n = n;
    G.g = g;
    G.wo = pt + s.woff[nlayer];
    if (nlayer == 1) return set_error(DP_ERR_UNSUPPORTED, "a fitting net without hidden layers has dD = wo");
    const io_t<real> *S = nullptr;  // dE/dv of the layer being walked; NULL: g wo (the last hidden layer)
    int64_t ldS = 0;
    int cur = 0;
    if (s.nout > 1) {  // dE/dv_{nlayer-1} = g W_out^T, [n][nout] x [nout][widths[nlayer-1]], first
      FitGemm<real> Z{};
      Z.r0 = G.r0;
      Z.n = n;
      Z.K = s.nout;
      Z.N = s.w[nlayer - 1];
      Z.src[0] = g;
      Z.lds[0] = s.nout;
      Z.nsrc = 1;
      Z.W = pt + s.woff[nlayer];  // W_out [widths[nlayer-1]][nout], read transposed
      Z.wt = true;
      Z.lin = true;
      Z.out = buf[0];
      Z.ldo = s.maxh;
      if ((rc = launch_gemm<real, true>(Z, st, "dp_fitting_grad"))) return rc;
      S = buf[0];
      ldS = s.maxh;
      cur = 1;
    }
    for (int l = nlayer - 1; l >= 1; --l) {
      G.K = s.w[l];      // contraction over the layer's outputs
      G.N = s.w[l - 1];  // producing dE/dv_{l-1}
      G.S = S;
      G.ldS = ldS;
      G.T = act + s.aoff[l];
      G.ldT = s.H;
      G.W = pt + s.woff[l];
      G.skip = s.w[l] == s.w[l - 1];
      if (l == 1) {
        G.out = dD;
        G.ldo = s.w[0];
      } else {
        G.out = buf[cur];
        G.ldo = s.maxh;
      }
      rc = launch_gemm<real, false>(G, st, "dp_fitting_grad");
      if (rc) return rc;
      S = G.out;
      ldS = G.ldo;
      cur ^= 1;
    }
  }
  return DP_OK;
}

// ------------------------------------------------- f64 GEMMs on the tensor cores
// (tc_gemm.cuh: the digit splitting; fit_gemm.cuh: the GEMM with its epilogues and the split kernels)
namespace tf {

// The GEMMs on the tensor cores: the hidden layers, and with several outputs the output layer too
// (forward: v W_out + b_out; backward: g W_out^T, first).  GEMM q of a direction works on layer
// gemm_layer(s, fwd, q): forward 1 .. L-1 (then L), backward (L, then) L-1 .. 1.
int gemm_count(const FitShape &s) { return s.nlayer - 1 + (s.nout > 1 ? 1 : 0); }
int gemm_layer(const FitShape &s, bool fwd, int q) {
  return fwd ? q + 1 : s.nlayer - q - (s.nout > 1 ? 0 : 1);
}

// Where the B planes and column exponents of each GEMM sit in one type's share of the work buffer.
struct Layer {
  int K, N, Np, Kp;
  size_t planes, fexp;  // byte offsets
};
size_t layout(const FitShape &s, bool fwd, Layer *out) {
  size_t off = 0;
  for (int q = 0; q < gemm_count(s); ++q) {
    const int l = gemm_layer(s, fwd, q);
    Layer &L = out[q];
    L.K = fwd ? s.w[l - 1] : s.w[l];
    L.N = fwd ? s.w[l] : s.w[l - 1];
    L.Np = (int)round_up(L.N, kTNF);
    L.Kp = (int)round_up(L.K, kTK);
    L.planes = off;
    off += (size_t)round_up((int64_t)kSF * L.Np * L.Kp * 2, 256);
    L.fexp = off;
    off += (size_t)round_up((int64_t)L.Np * 4, 256);
  }
  return off;
}

// Shares of K of one GEMM: at most kMaxSharesK slices each (the exactness bound), and more where that still
// gives each SM at most one unit, but at least kMinShareSlices slices each (copper's hidden layers, 128 tiles:
// one share, the layer finished in the GEMM, 26 us; two shares and the reduction 53 us).
constexpr int kTargetUnits = 152;
constexpr int kMinShareSlices = 6;
int shares_for(int64_t tiles, int slices) {
  int want = (int)std::min<int64_t>(std::max<int64_t>(1, kTargetUnits / tiles), std::max(1, slices / kMinShareSlices));
  want = std::max(want, (slices + kMaxSharesK - 1) / kMaxSharesK);
  const int per = (slices + want - 1) / want;
  return (slices + per - 1) / per;  // no empty share
}

// The work buffer: the B planes of a batch of types, the A planes and row exponents of a chunk of row tiles,
// the shares' partial results, and the [nloc][max hidden width] buffers between layers (four).  Types go
// through in batches, and a batch's row tiles in chunks, of as many as the caller's buffer holds; the results
// do not depend on either (every output is summed exactly and rounded once).
constexpr int64_t kChunkRows = 16384;
struct WorkMap {
  int types, tiles;         // per batch, per chunk
  size_t bstride;           // bytes of one type's B planes (the larger of the two directions)
  size_t tanh_table, aplanes, aexp, part, buffers, total;
};
WorkMap work_map(const FitShape &s, int64_t nloc, int types, int tiles) {
  Layer L[kMaxGemms];
  WorkMap m{};
  m.types = types;
  m.tiles = tiles;
  m.bstride = std::max(layout(s, true, L), layout(s, false, L));
  int kmax = 1;
  for (int l = 0; l <= s.nlayer; ++l) kmax = std::max(kmax, s.w[l]);  // every GEMM's K is a layer width
  m.tanh_table = m.bstride * types;
  m.aplanes = m.tanh_table + (size_t)round_up((int64_t)kTanhEntries * (int64_t)sizeof(TanhEntry), 256);
  m.aexp = m.aplanes + (size_t)round_up((int64_t)tiles * kSF * kPlaneAF * (round_up(kmax, kTK) / kTK), 256);
  m.part = m.aexp + (size_t)round_up((int64_t)tiles * kTM * 4, 256);
  int64_t units = 0;  // of any chunk of at most `tiles` row tiles, where K takes several shares
  for (int dir = 0; dir < 2; ++dir) {
    layout(s, dir == 0, L);
    for (int q = 0; q < gemm_count(s); ++q) {
      const int64_t nt = L[q].Np / kTNF, slices = L[q].Kp / kTK, least = (slices + kMaxSharesK - 1) / kMaxSharesK;
      if (least > 1) units = std::max<int64_t>(units, least * tiles * nt);
      units = std::max<int64_t>(units, kTargetUnits + std::min<int64_t>(tiles * nt, kTargetUnits));
    }
  }
  m.buffers = m.part + (size_t)(units * kTM * kTNF) * sizeof(longlong2);
  m.total = m.buffers + (s.nlayer > 1 ? (size_t)4 * (size_t)nloc * (size_t)s.maxh * sizeof(double) : 0);
  return m;
}
int query_tiles(int64_t nloc) { return (int)(round_up(std::min<int64_t>(std::max<int64_t>(nloc, 1), kChunkRows), kTM) / kTM); }
size_t work_bytes(const FitShape &s, int64_t nloc) {
  const int types = (int)std::min<int64_t>(DP_MAX_TYPES, std::max<int64_t>(nloc, 1));
  return work_map(s, nloc, types, query_tiles(nloc) + types - 1).total;
}
// The smallest buffer taken: what the query gives, or, where that is less, what it gave when types went one by
// one with nine 6-bit digits and four floats an output through memory -- callers may hold buffers of that size.
size_t least_bytes(const FitShape &s, int64_t nloc) {
  Layer L[kMaxGemms];
  const int64_t Mp = (int64_t)query_tiles(nloc) * kTM;
  int64_t kmax = 1, nmax = 48, planes = 0, part = 0;
  for (int l = 0; l <= s.nlayer; ++l) {
    kmax = std::max<int64_t>(kmax, s.w[l]);
    nmax = std::max(nmax, round_up(s.w[l], 48));
  }
  for (int dir = 0; dir < 2; ++dir) {
    layout(s, dir == 0, L);
    int64_t sum = 0;
    for (int q = 0; q < gemm_count(s); ++q) {
      const int64_t Np = round_up(L[q].N, 48), slices = L[q].Kp / kTK, tiles = Mp / kTM * (Np / 48);
      sum += round_up(9 * Np * L[q].Kp * 2, 256) + round_up(Np * 4, 256);
      const int64_t want = std::max(std::min((608 + tiles - 1) / tiles, std::max<int64_t>(1, slices / 6)), (slices + 111) / 112);
      const int64_t per = (slices + want - 1) / want;
      part = std::max(part, (slices + per - 1) / per * Mp * Np);
    }
    planes = std::max(planes, sum);
  }
  part = std::max(part, 608 * 128 * 48 + Mp * nmax);
  const int64_t old = planes + round_up(9 * Mp * round_up(kmax, kTK) * 2, 256) + round_up(Mp * 4, 256) +
                      round_up(part * 16, 256) + (s.nlayer > 1 ? 4 * nloc * s.maxh * (int64_t)sizeof(double) : 0);
  return std::min(work_bytes(s, nloc), (size_t)old);
}
// The largest map that the buffer holds: fewer types a batch first, then fewer row tiles a chunk.
bool fit_map(const FitShape &s, int64_t nloc, size_t nbytes, WorkMap *out) {
  for (int types = s.ntypes; types >= 1; --types) {
    *out = work_map(s, nloc, types, query_tiles(nloc) + types - 1);
    if (out->total <= nbytes) return true;
  }
  for (int tiles = query_tiles(nloc); tiles >= 1; tiles /= 2) {
    *out = work_map(s, nloc, 1, tiles);
    if (out->total <= nbytes) return true;
  }
  return false;
}
int check_work(const FitShape &s, int64_t nloc, const void *work, size_t nbytes, const char *who, WorkMap *m) {
  if (gemm_count(s) == 0) return DP_OK;
  if (!work) return set_error(DP_ERR_NULL, "%s: work is NULL", who);
  if (nbytes < least_bytes(s, nloc) || !fit_map(s, nloc, nbytes, m))
    return set_error(DP_ERR_SHAPE, "%s: work holds %zu bytes, needs %zu", who, nbytes, work_bytes(s, nloc));
  if (reinterpret_cast<uintptr_t>(work) % 256) return set_error(DP_ERR_SHAPE, "%s: work is not 256-byte aligned", who);
  return DP_OK;
}

// One direction over one batch of types: its weights split, then `layers` called for each chunk of row tiles.
struct Run {
  const FitShape &s;
  const WorkMap &m;
  bool fwd;
  const double *params;  // the batch's first type's
  unsigned char *work;
  cudaStream_t st;
  const char *who;
  Tiles G;
  Layer L[kMaxGemms];
  int nsm;

  int split_weights(int types) {
    SplitB B{};
    B.params = params;
    B.pstride = s.P;
    B.count = gemm_count(s);
    layout(s, fwd, L);
    for (int q = 0; q < B.count; ++q) {
      B.K[q] = L[q].K;
      B.N[q] = L[q].N;
      B.woff[q] = s.woff[gemm_layer(s, fwd, q)];
      B.planes[q] = L[q].planes;
      B.fexp[q] = L[q].fexp;
      B.group0[q + 1] = B.group0[q] + L[q].Np / 8;
    }
    B.bstride = m.bstride;
    B.transposed = !fwd;
    B.work = work;
    B.tanh_table = fwd ? reinterpret_cast<TanhEntry *>(work + m.tanh_table) : nullptr;
    if (B.count == 0) return DP_OK;
    split_b_kernel<16><<<dim3((unsigned)(B.group0[B.count] + (fwd ? 1 : 0)), (unsigned)types), 512, 0, st>>>(B);
    return launch_status(who);
  }

  // GEMM q over the chunk's row tiles, from A's source to the epilogue's outputs
  int gemm(int q, const SplitA &src, const Epilogue &E, bool dz = false) {
    SplitA A = src;
    A.G = G;
    A.K = L[q].K;
    A.Kp = L[q].Kp;
    A.planes = work + m.aplanes;
    A.exps = reinterpret_cast<int *>(work + m.aexp);
    A.pstride = s.P;
    const unsigned blocks = (unsigned)(G.tiles * (kTM / 8));
    if (dz)
      split_a_kernel<4, true><<<blocks, 128, 0, st>>>(A);
    else
      split_a_kernel<4, false><<<blocks, 128, 0, st>>>(A);
    int rc = launch_status(who);
    if (rc) return rc;
    Gemm C{};
    C.G = G;
    C.E = E;
    C.E.N = L[q].N;
    C.E.pstride = s.P;
    C.E.tanh_table = reinterpret_cast<const TanhEntry *>(work + m.tanh_table);
    C.nt = L[q].Np / kTNF;
    C.ka = L[q].Kp / kTK;
    C.ks = shares_for((int64_t)G.tiles * C.nt, C.ka);
    C.per = (C.ka + C.ks - 1) / C.ks;
    C.aplanes = A.planes;
    C.Eexp = A.exps;
    C.bplanes = work + L[q].planes;
    C.Fexp = reinterpret_cast<const int *>(work + L[q].fexp);
    C.bstride = m.bstride;
    C.fstride = m.bstride / sizeof(int);
    C.part = reinterpret_cast<longlong2 *>(work + m.part);
    const unsigned grid = (unsigned)std::min<int64_t>(nsm, (int64_t)G.tiles * C.nt * C.ks);
    if (fwd)
      fit_gemm_kernel<true><<<grid, kThreadsF, kSmemF, st>>>(C);
    else
      fit_gemm_kernel<false><<<grid, kThreadsF, kSmemF, st>>>(C);
    if ((rc = launch_status(who))) return rc;
    if (C.ks > 1) {
      const int64_t warps = (int64_t)G.tiles * 4 * ((C.E.N + 3) / 4);
      const unsigned rb = (unsigned)((warps + 3) / 4);
      if (fwd)
        fit_reduce_kernel<true><<<rb, 128, 0, st>>>(C);
      else
        fit_reduce_kernel<false><<<rb, 128, 0, st>>>(C);
      rc = launch_status(who);
    }
    return rc;
  }
};

// Batches of types and chunks of row tiles; layers(run) runs a chunk, rows(run, row0, n) a batch's rows after.
template <class Layers, class Rows>
int over_batches(const FitShape &s, const WorkMap &m, bool fwd, const double *params, unsigned char *work,
                 cudaStream_t st, const char *who, Layers &&layers, Rows &&rows) {
  int dev = 0, nsm = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return set_error(DP_ERR_CUDA, "%s: %s", who, cudaGetErrorString(cudaGetLastError()));
  const int step = std::max(1, m.types);
  for (int t0 = 0; t0 < s.ntypes; t0 += step) {
    const int types = std::min(step, s.ntypes - t0);
    const int64_t r0 = s.start[t0], r1 = s.start[t0 + types];
    if (r0 == r1) continue;
    Run R{s, m, fwd, params + (size_t)t0 * s.P, work, st, who, Tiles{}, {}, std::max(1, nsm)};
    R.G.ntypes = types;
    for (int t = 0; t < types; ++t) {
      R.G.start[t] = s.start[t0 + t];
      R.G.t0[t + 1] = R.G.t0[t] + (int)((s.start[t0 + t + 1] - s.start[t0 + t] + kTM - 1) / kTM);
    }
    R.G.start[types] = r1;
    int rc = R.split_weights(types);
    const int all = R.G.t0[types];
    for (int c = 0; c < all && !rc && gemm_count(s) > 0; c += m.tiles) {
      R.G.tile0 = c;
      R.G.tiles = std::min(m.tiles, all - c);
      rc = layers(R);
    }
    if (!rc) rc = rows(R, r0, r1 - r0);
    if (rc) return rc;
  }
  return DP_OK;
}

int fwd(const double *params, const int32_t *widths, int nlayer, int ntypes, const int64_t *type_start, const double *D,
        double *E, double *act, void *work, size_t work_nbytes, void *stream) {
  clear_error();
  static const char *who = "dp_fitting_fwd_tc_f64";
  FitShape s{};
  int rc = fit_shape(widths, nlayer, ntypes, type_start, &s, true);
  if (rc) return rc;
  const int64_t nloc = s.start[ntypes];
  if (nloc == 0) return DP_OK;
  if (!params || !D || !E || (s.H > 0 && !act)) return set_error(DP_ERR_NULL, "%s: NULL array", who);
  WorkMap m{};
  if ((rc = check_work(s, nloc, work, work_nbytes, who, &m)) || (rc = set_smem(who))) return rc;
  const cudaStream_t st = (cudaStream_t)stream;
  unsigned char *wk = static_cast<unsigned char *>(work);
  double *V[2] = {reinterpret_cast<double *>(wk + m.buffers), nullptr};
  V[1] = V[0] + (size_t)nloc * s.maxh;
  auto layers = [&](Run &R) {
    for (int q = 0; q < gemm_count(s); ++q) {  // layer l = q + 1; input v_{l-1}: D, then the layers' outputs
      const int l = q + 1;
      SplitA A{};
      A.X = l == 1 ? D : V[l & 1];
      A.ldx = l == 1 ? s.w[0] : s.maxh;
      Epilogue P{};
      P.A = A.X;
      P.lda = A.ldx;
      P.bias = R.params + s.woff[l] + (size_t)s.w[l - 1] * s.w[l];
      if (l < nlayer) {
        P.skip = s.w[l] == s.w[l - 1];
        P.act = act + s.aoff[l];
        P.ldact = s.H;
        P.V = V[(l - 1) & 1];
        P.ldv = s.maxh;
      } else {  // several outputs: E_i = v W_out + b_out
        P.lin = true;
        P.V = E;
        P.ldv = s.nout;
      }
      if (int e = R.gemm(q, A, P)) return e;
    }
    return (int)DP_OK;
  };
  auto rows = [&](Run &R, int64_t r0, int64_t n) {
    if (s.nout > 1) return (int)DP_OK;
    fit_energy_kernel<<<(unsigned)((n + 3) / 4), 128, 0, st>>>(R.G, r0, n, nlayer == 1 ? D : V[nlayer & 1],
                                                               nlayer == 1 ? s.w[0] : s.maxh, s.w[nlayer - 1],
                                                               R.params + s.woff[nlayer], s.P, E);
    return launch_status(who);
  };
  return over_batches(s, m, true, params, wk, st, who, layers, rows);
}

int grad(const double *params, const int32_t *widths, int nlayer, int ntypes, const int64_t *type_start,
         const double *act, const double *g, double *dD, void *work, size_t work_nbytes, void *stream) {
  clear_error();
  static const char *who = "dp_fitting_grad_tc_f64";
  FitShape s{};
  int rc = fit_shape(widths, nlayer, ntypes, type_start, &s, true);
  if (rc) return rc;
  const int64_t nloc = s.start[ntypes];
  if (nloc == 0) return DP_OK;
  if (nlayer == 1) return set_error(DP_ERR_UNSUPPORTED, "a fitting net without hidden layers has dD = wo");
  if (!params || !dD || (s.H > 0 && !act)) return set_error(DP_ERR_NULL, "%s: NULL array", who);
  if (s.nout > 1 && !g) return set_error(DP_ERR_NULL, "%s: g is NULL for a net of %d outputs", who, s.nout);
  WorkMap m{};
  if ((rc = check_work(s, nloc, work, work_nbytes, who, &m)) || (rc = set_smem(who))) return rc;
  const cudaStream_t st = (cudaStream_t)stream;
  unsigned char *wk = static_cast<unsigned char *>(work);
  double *buf = reinterpret_cast<double *>(wk + m.buffers);
  const size_t bs = (size_t)nloc * s.maxh;
  double *Z[2] = {buf, buf + bs}, *Sb[2] = {buf + 2 * bs, buf + 3 * bs};
  auto layers = [&](Run &R) {
    const double *wo = R.params + s.woff[nlayer];
    const double *S = nullptr;  // dE/dv of the layer being walked; NULL: g wo (the last hidden layer)
    const int q0 = s.nout > 1 ? 1 : 0;  // the hidden layers' GEMMs come after g W_out^T
    if (s.nout > 1) {  // dE/dv_{nlayer-1} = g W_out^T into Sb[1], which the walk below first writes after
                       // its first GEMM has read it
      SplitA A{};
      A.X = g;
      A.ldx = s.nout;
      Epilogue P{};
      P.out = Sb[1];
      P.ldo = s.maxh;
      if (int e = R.gemm(0, A, P)) return e;
      S = Sb[1];
    }
    int cur = 0;
    for (int l = nlayer - 1; l >= 1; --l) {
      SplitA A{};
      const bool last = l == nlayer - 1;  // its dz is formed as it is split
      A.X = last ? act + s.aoff[l] : Z[cur];
      A.ldx = last ? s.H : s.maxh;
      A.S = last ? S : nullptr;
      A.ldS = s.maxh;
      A.g = g;
      A.wo = wo;
      Epilogue P{};
      P.skip = s.w[l] == s.w[l - 1];
      P.S = S;
      P.ldS = s.maxh;
      P.g = g;
      P.wo = wo;
      if (l > 1) {
        P.T = act + s.aoff[l - 1];
        P.ldT = s.H;
        P.Snext = Sb[cur];
        P.Z = Z[cur ^ 1];
        P.ldz = s.maxh;
      } else {
        P.out = dD;
        P.ldo = s.w[0];
      }
      if (int e = R.gemm(q0 + nlayer - 1 - l, A, P, last)) return e;
      S = P.Snext;
      cur ^= 1;
    }
    return (int)DP_OK;
  };
  return over_batches(s, m, false, params, wk, st, who, layers, [](Run &, int64_t, int64_t) { return (int)DP_OK; });
}

size_t work_bytes_api(const int32_t *widths, int nlayer, int64_t nloc) {
  clear_error();
  if (nloc < 0) return 0;
  const int64_t ts[2] = {0, nloc};
  FitShape s{};
  if (fit_shape(widths, nlayer, 1, ts, &s, true)) return 0;
  return work_bytes(s, nloc);
}
}  // namespace tf


// ------------------------------------------------- backward without allocation
// Some callers cannot hand this library a scratch buffer: an MD engine's force
// loop that owns all device memory, sized once at start-up, and gives a plugin
// only its input and output arrays -- allocating there would synchronise the
// device in the middle of a time step and fragment the engine's pool.  For
// them dp_fitting_grad_noalloc_f64 takes its scratch (the two buffers the
// backward passes between layers) from this fixed array, which every GPU that
// loads the library keeps until the process exits.
constexpr size_t kStaticScratchDoubles = (size_t)1 << 20;  // 8 MiB
static __device__ __align__(256) double g_fit_scratch[kStaticScratchDoubles];

// Device address of the array in the current context.  In host code the array's
// name only stands in for it; the runtime gives the address.  It is looked up
// on every call (the lookup allocates nothing), so that a context made anew --
// after cudaDeviceReset, or on another device -- is served at its own address.
int static_scratch(double **out) {
  void *q = nullptr;
  const cudaError_t e = cudaGetSymbolAddress(&q, g_fit_scratch);
  if (e != cudaSuccess)
    return set_error(DP_ERR_CUDA, "dp_fitting_grad_noalloc: cudaGetSymbolAddress: %s", cudaGetErrorString(e));
  *out = static_cast<double *>(q);
  return DP_OK;
}

int fitting_grad_noalloc(const double *params, const int32_t *widths, int nlayer, int ntypes,
                         const int64_t *type_start, const double *act, const double *g, double *dD, void *stream) {
  clear_error();
  FitShape s{};
  int rc = fit_shape(widths, nlayer, ntypes, type_start, &s, true);
  if (rc) return rc;
  const int64_t nloc = s.start[ntypes];
  const size_t need = (nlayer > 2 || s.nout > 1) ? (size_t)2 * (size_t)nloc * (size_t)s.maxh : 0;
  if (need > kStaticScratchDoubles)
    return set_error(DP_ERR_UNSUPPORTED,
                     "dp_fitting_grad_noalloc: needs 2 x %lld atoms x %d = %zu doubles of scratch, the static array "
                     "holds %zu; use dp_fitting_grad_f64 with a work buffer",
                     (long long)nloc, s.maxh, need, kStaticScratchDoubles);
  double *work = nullptr;
  if (need > 0 && nloc > 0) {
    rc = static_scratch(&work);
    if (rc) return rc;
  }
  return fitting_grad<double>(params, widths, nlayer, ntypes, type_start, act, g, dD, work, stream);
}

}  // namespace

// This unit's GEMM wait timeouts (see tc_gemm.cuh), for dp_tc_wait_timeouts.
int take_wait_timeouts_fitting(unsigned int *count) { return tc::take_wait_timeouts(count); }

}  // namespace dpc

extern "C" {

int dp_fitting_grad_noalloc_f64(const double *params, const int32_t *widths, int nlayer, int ntypes,
                                const int64_t *type_start, const double *act, const double *g, double *dD,
                                void *stream) {
  return dpc::fitting_grad_noalloc(params, widths, nlayer, ntypes, type_start, act, g, dD, stream);
}

int dp_fitting_fwd_f64(const double *params, const int32_t *widths, int nlayer, int ntypes, const int64_t *type_start,
                       const double *D, double *E, double *act, void *stream) {
  return dpc::fitting_fwd<double>(params, widths, nlayer, ntypes, type_start, D, E, act, stream);
}
int dp_fitting_fwd_f32(const float *params, const int32_t *widths, int nlayer, int ntypes, const int64_t *type_start,
                       const float *D, float *E, float *act, void *stream) {
  return dpc::fitting_fwd<float>(params, widths, nlayer, ntypes, type_start, D, E, act, stream);
}
int dp_fitting_fwd_df64(const double *params, const int32_t *widths, int nlayer, int ntypes,
                        const int64_t *type_start, const double *D, double *E, double *act, void *stream) {
  return dpc::fitting_fwd<dpc::df64>(params, widths, nlayer, ntypes, type_start, D, E, act, stream);
}
int dp_fitting_grad_f64(const double *params, const int32_t *widths, int nlayer, int ntypes,
                        const int64_t *type_start, const double *act, const double *g, double *dD, double *work,
                        void *stream) {
  return dpc::fitting_grad<double>(params, widths, nlayer, ntypes, type_start, act, g, dD, work, stream);
}
int dp_fitting_grad_f32(const float *params, const int32_t *widths, int nlayer, int ntypes, const int64_t *type_start,
                        const float *act, const float *g, float *dD, float *work, void *stream) {
  return dpc::fitting_grad<float>(params, widths, nlayer, ntypes, type_start, act, g, dD, work, stream);
}
int dp_fitting_grad_df64(const double *params, const int32_t *widths, int nlayer, int ntypes,
                         const int64_t *type_start, const double *act, const double *g, double *dD, double *work,
                         void *stream) {
  return dpc::fitting_grad<dpc::df64>(params, widths, nlayer, ntypes, type_start, act, g, dD, work, stream);
}

size_t dp_fitting_tc_work_bytes(const int32_t *widths, int nlayer, int64_t nloc) {
  return dpc::tf::work_bytes_api(widths, nlayer, nloc);
}
int dp_fitting_fwd_tc_f64(const double *params, const int32_t *widths, int nlayer, int ntypes,
                          const int64_t *type_start, const double *D, double *E, double *act, void *work,
                          size_t work_bytes, void *stream) {
  return dpc::tf::fwd(params, widths, nlayer, ntypes, type_start, D, E, act, work, work_bytes, stream);
}
int dp_fitting_grad_tc_f64(const double *params, const int32_t *widths, int nlayer, int ntypes,
                           const int64_t *type_start, const double *act, const double *g, double *dD, void *work,
                           size_t work_bytes, void *stream) {
  return dpc::tf::grad(params, widths, nlayer, ntypes, type_start, act, g, dD, work, work_bytes, stream);
}

}  // extern "C"
