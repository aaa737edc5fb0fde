// Tabulated embedding + contraction (Sec. II, kernel fusion) in f64 with the
// per-interval contraction on the tcgen05 tensor cores.
//
// The fused forward is a sum over the valid neighbour rows j of atom i,
//   T_i[k][m] = (1/N_c) sum_j R~_j[k] g_m^l(t_j),  g_m^l(t) = sum_q c_q^{l,m} t^q (q = 0..5),
// l the row's interval and t its offset from the interval's left node.  With
// u = t / Delta_l (Delta_l the interval's step, so 0 <= u <= 1) and the scaled
// coefficients c'_q^{l,m} = c_q^{l,m} Delta_l^q, it regroups per interval into
// moments of the rows that fall in it,
//   W_i[k][(l, q)] = sum_{j in l} R~_j[k] u_j^q,     T_i[k][m] = (1/N_c) sum_{(l, q)} W_i[k][(l, q)] c'_q^{l,m},
// a GEMM whose K index is (neighbour type, interval, power): the same sum as
// the per-row evaluation, associated per interval.  The backward is the
// transposed GEMM, on the unscaled coefficients (its A rows 6 key + q each
// carry their own exponent, so no scale is needed there), and the rows'
// polynomials in t itself:
//   dW_i[k][(l, q)] = (1/N_c) sum_m dT_i[k][m] c_q^{l,m},
//   dE/dR~_j[k] = sum_q dW_i[k][(l, q)] t_j^q,
//   dE/ds_j     = sum_k R~_j[k] sum_{q >= 1} q dW_i[k][(l, q)] t_j^(q-1)   (0 where s_j was clamped).
// The per-row work (24 multiply-adds per row for W, 40 for the derivatives) runs in fixed point on the
// integer pipes (fixed.cuh), the FP64 pipe converting; the per-interval work (24 M1 FMAs per interval and atom in
// each direction), which is most of it, runs as exact digit-split GEMMs on
// the tensor cores (tc_gemm.cuh), at f64 accuracy.
//
// K layout, per centre type: key = beta nint + l (neighbour type beta, interval
// l), and column 6 key + q of the GEMM holds power q, so an interval lies in
// one or two 16-deep K slices.  An atom touches only the intervals its
// rows fall in: the W values are stored per run of rows (one slot per
// interval an atom uses, found through a per-atom map), and the GEMMs skip the
// slices (forward) or output tiles (backward) that no atom of a tile uses.
//
// C'_alpha and its digit planes are made once per table by dp_tabulate_tc_plan_f64 (the plan).
// Per chunk of at most kChunkAtoms atoms:
//   forward:  runs_kernel<true> (slot keys, W, column exponents, slice flags), slice_list_kernel (each
//             tile's used slices), fwd_schedule_kernel (every centre type's items cut into pieces of
//             equal cost per CTA), tgemm_kernel<true> (tab_gemm.cuh, one launch; A = C'_alpha^T:
//             channels x K, B = W^T: K x (atom, k), its digit planes made in shared memory from W; an
//             uncut item writes its atoms' T, a piece its exact 128-bit partial sums),
//             fwd_finish_kernel (T of the cut items, and D_i = T_i^T T_i[:, :M2] when asked for);
//   backward: runs_kernel<false> (slot keys, slice flags; skipped when the forward's are reused),
//             the split of dT (B), the GEMM units, and the GEMM (A = C'_alpha: K x channels, B =
//             dT^T) scattering each used (atom, interval) block, as fixed points, to its run slot --
//             bgemm_kernel (tab_gemm_b8.cuh: every centre type in one launch, 8-atom tiles, seven 8-bit
//             digits) when M1 rounds up to at most 144, else tgemm_kernel<false> per centre type (12-atom
//             tiles, nine 6-bit digits) -- and rows_kernel (dE/ds, dE/dR~).
// The environment-fused calls (dp_tabulate_fusion_env_*_tc_f64) form each row from coordinates in
// runs_kernel<.., true> and add each row's force and virial in rows_force_kernel instead.
// The slot keys, their counts and the slice flags of every atom stay in the work buffer after
// the forward, so that a backward on the same inputs can skip its own key pass.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "desc_fixed.cuh"
#include "dp_common.cuh"
#include "env_row.cuh"
#include "fixed.cuh"
#include "tab_gemm.cuh"
#include "tab_gemm_b8.cuh"
#include "tc_gemm.cuh"

namespace dpc {
namespace {
namespace tt {
using namespace tc;

constexpr int kQ = 6;                 // K entries per interval: u^0 .. u^5
constexpr int kCols = 4;              // GEMM columns per atom: k = 0 .. 3
constexpr int kTileAtoms = kTN / kCols;  // 12 atoms per 48-column tile
constexpr int64_t kChunkAtoms = 16416;   // a multiple of 24 (12- and 8-atom tiles; 65,664 columns)
constexpr int kShareSlices = kMaxShareSlices;  // used K slices per forward share (112, the exactness bound)
constexpr size_t kPartBudget = (size_t)1 << 30;  // bytes of the forward's partial results per chunk at most
constexpr int kMaxCtasF = 160;  // CTAs of the forward GEMM at most (its part slots are sized for them)
constexpr int kEpiCost = 6;     // a forward unit's epilogue, in slices' time, for the forward schedule
constexpr int kBadFlag = DP_MAX_TYPES;  // after the backward's unit counts: set when a GEMM wait gave up
constexpr int kMaxKeys = 4096;  // ntypes x nint: each warp's key map (int16) lives in shared memory
static_assert(kChunkAtoms % kTileAtoms == 0 && kChunkAtoms % 8 == 0, "whole tiles per chunk");

// Shorts of one atom's key -> slot map: whole 16-byte words.
__host__ __device__ constexpr int map_stride(int nkeys) { return (nkeys + 7) / 8 * 8; }

// Sizes shared by the kernels, the plan and the work-buffer layout.
struct Shape {
  int ntypes, nint, nkeys, M1, cap;
  int Kp;    // round_up(6 nkeys, 16): K of the forward GEMM, rows of the backward A
  int nsl;   // Kp / 16
  int Mpf;   // round_up(M1, 128): rows of the forward A
  int Kpm;   // round_up(M1, 16): K of the backward GEMM
  int Mpb;   // round_up(Kp, 128): rows of the backward A
  int64_t nloc, tiles_all;    // atoms of the call and their 12-atom tiles
  int64_t chunk, Np, ntiles;  // atoms per chunk, its columns round_up(4 chunk, 48), Np / 48
  int zmax;                   // forward shares per tile at most
  int64_t maxunits;           // backward GEMM units (9 x 6 digits) per chunk and centre type at most
  int64_t nitems;             // forward items per chunk: (type, 12-atom tile, 128-row tile of A)
  int64_t maxpieces, maxslots;  // forward pieces and part slots per chunk at most
  bool b8;                    // the backward GEMM uses the 7 x 8-bit digits on 8-atom tiles (Kpm <= 144)
  int64_t Np8, ntiles8;       // its columns round_up(4 chunk, 32) and tiles Np8 / 32
  int64_t maxunits8;          // its units per chunk and centre type at most
};

// The plan: C' of every centre type and the digit planes of both GEMMs' A operands.
struct PlanLayout {
  size_t nodes, cp, afwd, efwd, abwd, ebwd, total;
};

// The work buffer: the slot keys, their counts and the slice flags of every atom of the call
// (kept from the forward for the backward), then one chunk's scratch.
struct Layout {
  size_t keys, nslots, occ, map, slist, scount, units, nunits, pieces, pcta, cta_start, npieces, pfirst, fexp, bplanes,
      w, part, total;
};

size_t take(size_t &off, size_t bytes) {
  const size_t at = off;
  off += (size_t)round_up((int64_t)bytes, 256);
  return at;
}

Shape table_shape(const TableGeom &g, int ntypes, int M1) {
  Shape s{};
  s.ntypes = ntypes;
  s.nint = g.nint;
  s.nkeys = ntypes * g.nint;
  s.M1 = M1;
  s.Kp = (int)round_up((int64_t)s.nkeys * kQ, kTK);
  s.nsl = s.Kp / kTK;
  s.Mpf = (int)round_up(M1, kTM);
  s.Kpm = (int)round_up(M1, kTK);
  s.Mpb = (int)round_up(s.Kp, kTM);
  s.zmax = (s.nsl + kShareSlices - 1) / kShareSlices;
  s.b8 = s.Kpm <= tb::kMaxKB;
  return s;
}

Shape make_shape(const TableGeom &g, int64_t nloc, int nnei, int ntypes, int M1) {
  Shape s = table_shape(g, ntypes, M1);
  s.cap = std::min(nnei, s.nkeys);
  s.nloc = nloc;
  s.tiles_all = (nloc + kTileAtoms - 1) / kTileAtoms;
  int64_t chunk = std::min<int64_t>(round_up(std::max<int64_t>(nloc, 1), kTileAtoms), kChunkAtoms);
  // part slots: two per CTA boundary, and every piece of an item whose used slices exceed one share
  auto slots_for = [&](int64_t c) {
    const int64_t items = (int64_t)s.ntypes * (round_up(kCols * c, kTN) / kTN) * (s.Mpf / kTM);
    return 2 * kMaxCtasF + (s.zmax > 1 ? items * s.zmax : 0);
  };
  while (chunk > kTileAtoms && (size_t)slots_for(chunk) * s.Mpf * kTN * sizeof(float4) > kPartBudget)
    chunk = round_up(chunk / 2, kTileAtoms);
  s.chunk = chunk;
  s.Np = round_up(kCols * chunk, kTN);
  s.ntiles = s.Np / kTN;
  s.maxunits = s.ntiles * (s.Mpb / kTM);
  s.nitems = (int64_t)s.ntypes * s.ntiles * (s.Mpf / kTM);
  s.maxpieces = s.nitems * s.zmax + kMaxCtasF;
  s.maxslots = slots_for(chunk);
  s.Np8 = round_up(kCols * chunk, tb::kTNB);
  s.ntiles8 = s.Np8 / tb::kTNB;
  s.maxunits8 = s.ntiles8 * (s.Mpb / kTM);
  return s;
}

PlanLayout plan_layout(const Shape &s) {
  PlanLayout L{};
  size_t off = 0;
  const size_t nt = (size_t)s.ntypes;
  L.nodes = take(off, (size_t)(s.nint + 1) * sizeof(double));
  L.cp = take(off, nt * s.Kp * s.M1 * sizeof(double));
  L.afwd = take(off, nt * kS * (size_t)s.Mpf * s.Kp * 2);
  L.efwd = take(off, nt * s.Mpf * sizeof(int));
  L.abwd = take(off, nt * (s.b8 ? tb::kSB : kS) * (size_t)s.Mpb * s.Kpm * 2);
  L.ebwd = take(off, nt * s.Mpb * sizeof(int));
  L.total = off;
  return L;
}

Layout make_layout(const Shape &s) {
  Layout L{};
  size_t off = 0;
  L.keys = take(off, (size_t)std::max<int64_t>(s.nloc, 1) * s.cap * sizeof(short));
  L.nslots = take(off, (size_t)std::max<int64_t>(s.nloc, 1) * sizeof(int));
  L.occ = take(off, (size_t)s.ntypes * std::max<int64_t>(s.tiles_all, 1) * s.nsl);
  L.map = take(off, std::max((size_t)s.chunk * s.nkeys * sizeof(int), (size_t)s.chunk * map_stride(s.nkeys) * sizeof(short)));
  L.slist = take(off, (size_t)s.ntypes * s.ntiles * s.nsl * sizeof(short));
  L.scount = take(off, (size_t)s.ntypes * s.ntiles * sizeof(int));
  L.units = take(off, (size_t)s.ntypes * std::max(s.maxunits, s.maxunits8) * sizeof(int));
  L.nunits = take(off, (size_t)(kBadFlag + 1) * sizeof(int));
  L.pieces = take(off, (size_t)s.maxpieces * sizeof(int4));
  L.pcta = take(off, (size_t)s.maxpieces * sizeof(int));
  L.cta_start = take(off, (size_t)(kMaxCtasF + 1) * sizeof(int));
  L.npieces = take(off, (size_t)s.nitems * sizeof(int));
  L.pfirst = take(off, (size_t)s.nitems * sizeof(int));
  L.fexp = take(off, (size_t)std::max(s.Np, s.Np8) * sizeof(int));
  L.bplanes = take(off, s.b8 ? (size_t)s.ntiles8 * (s.Kpm / kTK) * tb::kSB * tb::kPlaneBB  // the backward's dT planes
                             : (size_t)s.ntiles * (s.Kpm / kTK) * kS * kPlaneB);
  L.w = take(off, (size_t)s.chunk * s.cap * 24 * sizeof(double));  // moments (forward) or their gradients
  L.part = take(off, (size_t)s.maxslots * s.Mpf * kTN * sizeof(longlong2));
  L.total = off;
  return L;
}

// C'[alpha][6 key + q][m] = c_q Delta_l^q / N_c (key = beta nint + l; rows past the keys: 0).
// The interval's block of the table is pair-planar [3][M1][2] holding (a, b, c, d, e, f), the
// coefficients of t^5 .. t^0.
// kU: the coefficients of u^q, c_q Delta^q (the forward's); else of t^q, c_q (the backward's)
__global__ void __launch_bounds__(256) coef_kernel(const double *__restrict__ table, TableGeom g, int ntypes, int M1,
                                                   int Kp, double scale, bool kU, double *__restrict__ Cp) {
  const int64_t total = (int64_t)ntypes * Kp * M1;
  for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < total; x += (int64_t)gridDim.x * blockDim.x) {
    const int m = (int)(x % M1);
    const int64_t rest = x / M1;
    const int r = (int)(rest % Kp), alpha = (int)(rest / Kp);
    const int key = r / kQ, q = r - kQ * key;
    double v = 0.0;
    if (key < ntypes * g.nint) {
      const int beta = key / g.nint, l = key - beta * g.nint;
      const double *blk = table + ((size_t)(alpha * ntypes + beta) * g.nint + l) * M1 * 6;
      const int j = 5 - q;  // position of t^q's coefficient in (a .. f)
      const double c = blk[(size_t)(j >> 1) * 2 * M1 + 2 * m + (j & 1)];
      const double delta = l < g.n0 ? g.stride0 : g.stride1;
      double p = 1.0;
      if (kU)
        for (int e = 0; e < q; ++e) p *= delta;
      v = c * p * scale;
    }
    Cp[x] = v;
  }
}

// The grid's nodes x_0 .. x_nint as the interval search forms them (node_x), for the per-row kernels.
__global__ void nodes_kernel(TableGeom g, double *__restrict__ nodes) {
  for (int l = blockIdx.x * blockDim.x + threadIdx.x; l <= g.nint; l += gridDim.x * blockDim.x) nodes[l] = node_x(g, l);
}

// An f32 value within 2^-23 (relative) of s, formed from the fields of s by integer operations (no
// FP64 instruction); ok is false where that fails: |s| outside [2^-100, 2^100), zero, inf, NaN.
__device__ __forceinline__ float approx_f32(double s, bool &ok) {
  const unsigned hi = (unsigned)__double2hiint(s), lo = (unsigned)__double2loint(s);
  const int e = (int)((hi >> 20) & 0x7ff) - 1023;
  ok = e > -100 && e < 100;
  return __uint_as_float((hi & 0x80000000u) | ((unsigned)(e + 127) << 23) | ((hi & 0xfffffu) << 3) | (lo >> 29));
}

// floor(x) clamped into [0, n], for x below 2^22, on the FP32 pipe: 2^23 added with rounding down.
__device__ __forceinline__ int floor_clamped(float x, int n) {
  return __float_as_int(__fadd_rd(fminf(fmaxf(x, 0.0f), (float)n), 8388608.0f)) - 0x4B000000;
}

// The interval search of the tensor-core path's per-row kernels.  The segment and the index come from
// the f32 approximation of s; t = s - x_l is one f64 subtraction from the node table.  The f32 index can
// differ from floor((s - x_0) / Delta) by one where s lies within ~1e-4 steps of a node; either interval
// is correct there (the table is C2, so both polynomials agree to the rounding at the node, and t then
// lies a hair outside [0, Delta]).  Inputs within 2^-18 (relative) of lower, upper or upper_ext, where
// the f32 comparison could take the wrong side, and inputs outside the f32 range take the f64 search,
// whose clamping they follow exactly.  Deterministic: the forward and the backward find the same l.
__device__ __forceinline__ int locate_fast(const TableGeom &g, const TableGeomF &f, const double *__restrict__ nodes,
                                           double s, double &t, bool &clamped) {
  bool ok;
  const float sf = approx_f32(s, ok);
  const float tol = 0x1p-18f * fabsf(sf);
  if (!ok || fabsf(sf - f.lower) <= tol || fabsf(sf - f.upper) <= tol || fabsf(sf - f.upper_ext) <= tol)
    return locate(g, s, t, clamped);
  clamped = sf < f.lower || sf >= f.upper_ext;
  if (sf < f.lower) {
    t = 0.0;
    return 0;
  }
  if (sf >= f.upper_ext) {
    t = g.n1 > 0 ? g.stride1 : g.stride0;
    return g.nint - 1;
  }
  const int l = sf < f.upper ? floor_clamped((sf - f.lower) * f.inv0, g.n0 - 1)
                             : g.n0 + floor_clamped((sf - f.upper) * f.inv1, g.n1 - 1);
  t = s - __ldg(nodes + l);
  return l;
}

// The environment matrix's inputs, where the tensor-core path forms its rows from coordinates itself
// (dp_tabulate_fusion_env_*_tc_f64: s and R~ never reach HBM, nor ds and dR~ in the backward).
struct EnvRow {
  const double *coord;   // [nall][3]
  const int32_t *nlist;  // [nloc][nnei]: the neighbour's index into coord, or -1 (each segment's first)
  double rcs, rc, inv_width, mean, inv_std, inv_std_all;
  int kind;
  bool unit;  // mean 0, std 1, std_all 1: the normalisation's operations change no bit and are left out
};

// Row (i, j) as dp_env_mat forms it, by the same operations: d = x_j - x_i, r, 1/r, s(r) and ds/dr, the
// table input and R~[0] sh = (s - mean)/std, and R~[1 .. 3] = s d / (r std_all).
struct EnvVals {
  double d[3], inv_r, sv, dsv, a, r4[4];  // a = s / r
};
__device__ __forceinline__ EnvVals env_vals(const EnvRow &E, int64_t i, int j) {
  EnvVals v;
  const double xi = E.coord[3 * i], yi = E.coord[3 * i + 1], zi = E.coord[3 * i + 2];
  v.d[0] = E.coord[3 * (int64_t)j] - xi;
  v.d[1] = E.coord[3 * (int64_t)j + 1] - yi;
  v.d[2] = E.coord[3 * (int64_t)j + 2] - zi;
  const double r2 = fma(v.d[0], v.d[0], fma(v.d[1], v.d[1], v.d[2] * v.d[2]));
  double r;
  radius(r2, r, v.inv_r);
  weight(E, r, v.inv_r, v.sv, v.dsv);
  v.a = v.sv * v.inv_r;
  const double a = E.unit ? v.a : v.a * E.inv_std_all;
  v.r4[0] = E.unit ? v.sv : __dmul_rn(v.sv - E.mean, E.inv_std);  // (the offset s - x_l is formed from it)
  v.r4[1] = a * v.d[0];
  v.r4[2] = a * v.d[1];
  v.r4[3] = a * v.d[2];
  return v;
}

// Valid rows per type segment of atom i from its neighbour list (the rows with a neighbour, each
// segment's first, as dp_env_mat counts them) into nvb, and into nvalid_out when given; their total.
__device__ __forceinline__ int env_valid_rows(const EnvRow &E, int nnei, const int *sel, int ntypes, int64_t i,
                                              int lane, int *nvb, int32_t *nvalid_out) {
  int count = 0;  // lane b < ntypes: segment b's rows with a neighbour
  for (int q0 = 0; q0 < nnei; q0 += 32) {  // uniform
    const int q = q0 + lane;
    const int j = q < nnei ? __ldg(E.nlist + i * nnei + q) : -1;
    int b = 0, lim = sel[0];
#pragma unroll
    for (int c = 1; c < DP_MAX_TYPES; ++c)
      if (c < ntypes && q >= lim) {
        b = c;
        lim += sel[c];
      }
#pragma unroll
    for (int c = 0; c < DP_MAX_TYPES; ++c) {
      if (c >= ntypes) break;  // uniform
      const int n = __popc(__ballot_sync(0xffffffffu, j >= 0 && b == c));
      if (lane == c) count += n;
    }
  }
  if (lane < DP_MAX_TYPES) nvb[lane] = lane < ntypes ? count : 0;
  if (nvalid_out && lane < ntypes) nvalid_out[i * ntypes + lane] = count;
  __syncwarp();
  int nv = 0;
#pragma unroll
  for (int q = 0; q < DP_MAX_TYPES; ++q) nv += nvb[q];
  return nv;
}

struct RunsParams {
  const double *s, *Rt;
  EnvRow env;           // kEnv: rows from coordinates (s and Rt unused)
  int32_t *nvalid_out;  // kEnv forward: the counts of valid rows it finds
  const int32_t *nvalid, *atype;
  TableGeom g;
  TableGeomF gf;
  const double *nodes;  // [nint + 1] (the plan's)
  int64_t atom0, natoms, tiles_all;  // the chunk's first atom (a multiple of 12) and size; all tiles
  int nnei, ntypes, nkeys, cap, nsl;
  int sel[DP_MAX_TYPES];
  short *keys;         // [nloc][cap]: key of each slot (every atom of the call)
  int *nslots;         // [nloc]: slots in use
  unsigned char *occ;  // [ntypes][tiles_all][nsl]: the K slices some atom of the tile uses
  short *map;          // forward: [natoms][map_stride(nkeys)] run slot of the key, or -1 (this chunk)
  double *W;           // forward: [natoms][cap][24] moments W[k][q] at 6 k + q
  int *fexp;           // forward: [Np] exponents of the columns 4 a + k
};

// A batch of 32 rows: R~ and the powers of u as fixed points (fx::Fix), or as doubles in a wild batch.
// A row is a column of the stage (33 entries a row of it: neither the lanes' stores nor the reads of one row
// by the 24 (k, q) lanes meet in a bank).
struct alignas(16) RunsStage {
  long long r[4][33];
  long long tp[6][33];
  int nvb[DP_MAX_TYPES];
};
static_assert(sizeof(fx::Fix) == sizeof(double), "a stage entry holds either");

// The binary places of a batch's R~[k]: |R~[k]| 2^sh < 2^57 over its rows, from the largest high word
// (sign off) of its values.  `wild`: an inf, a NaN or values so large or small that the sums' exponents
// could leave the normal range; such a batch is summed on the FP64 pipe.
__device__ __forceinline__ int batch_places(int hiword, bool &wild) {
  const int eb = hiword >> 20;
  wild |= hiword != 0 && (eb < 200 || eb > 1800);
  return hiword ? 57 + 1022 - eb : 0;
}

// Valid rows per type segment of atom i (clamped into [0, sel]) into nvb; returns their total.
__device__ __forceinline__ int valid_rows(const int32_t *nvalid, const int *sel, int ntypes, int64_t i, int lane,
                                          int *nvb) {
  int sl = 0;
#pragma unroll
  for (int q = 0; q < DP_MAX_TYPES; ++q)
    if (lane == q) sl = sel[q];
  int x = 0;
  if (lane < ntypes) x = clampi(nvalid ? __ldg(nvalid + i * ntypes + lane) : sl, 0, sl);
  if (lane < DP_MAX_TYPES) nvb[lane] = x;
  __syncwarp();
  int nv = 0;
#pragma unroll
  for (int q = 0; q < DP_MAX_TYPES; ++q) nv += nvb[q];
  return nv;
}

// Row index of valid row v (type segments in order, the valid rows of each first) and its segment.
__device__ __forceinline__ int valid_row(int v, const int *nvb, const int *sel, int ntypes, int &b) {
  int row = v;
  b = 0;
  int lim = nvb[0];
  for (int q = 1; q < ntypes; ++q)  // uniform; none for one type
    if (v >= lim) {
      b = q;
      row += sel[q - 1] - nvb[q - 1];
      lim += nvb[q];
    }
  return row;
}

// Warps (one atom each) per block of the runs and rows kernels: a few per block, so that launching
// thousands of tiny blocks does not set the pace of a short kernel.
constexpr int kRunsWarps = 4, kRowsWarps = 4;
// One warp per atom: the runs of rows sharing an interval (consecutive rows with one key; rows
// sorted by distance give one run per interval, and a key met again adds to its slot), each
// interval's slot (a shared-memory map of the keys; each slot's key and the slot count are written
// out) and the flags of its K slices for the atom's tile; forward also the map, its moments W and
// the atom's four column exponents (over every value written, which bounds the final ones).
// Rows go in batches of 32, a lane per row.  The batch's new keys get their slots together (a lane per
// run; the lowest lane of a key met twice leads), then the runs are summed one by one, lane 6 k + q
// taking R~[k] u^q: limb products on the integer pipes (fixed.cuh) against the batch's largest R~[k] and
// unit u, one conversion to f64 per run and lane.  Why: with FP64 moments the kernel took 80 sub-partition
// clocks a row (24 of 32 lanes of a 68-clock FMA, the powers of u); 24 FMAs as limb products take 10.  And
// with one pass of bookkeeping per run short runs spent longer on that than on their sums.  Measured:
// copper 0.133 -> 0.078 ms, water (2.7 rows a run) 0.099 -> 0.084 ms.
template <bool kMom, bool kEnv = false>
__global__ void __launch_bounds__(32 * kRunsWarps, 7) runs_kernel(const RunsParams P) {
  constexpr int L = 28;  // limbs of the moments: 32 rows' products of 57 and 56 places stay below 2^63
  using fx::Fix;
  __shared__ RunsStage stw[kRunsWarps];
  extern __shared__ __align__(16) short smapw[];  // [kRunsWarps][map_stride(nkeys)]
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t a = (int64_t)blockIdx.x * kRunsWarps + warp;
  if (a >= P.natoms) return;  // warp-uniform
  RunsStage &st = stw[warp];
  short *smap = smapw + (size_t)warp * map_stride(P.nkeys);
  const int64_t i = P.atom0 + a;
  for (int k = lane; k < map_stride(P.nkeys) / 8; k += 32)
    reinterpret_cast<int4 *>(smap)[k] = make_int4(-1, -1, -1, -1);
  const int nv = kEnv ? env_valid_rows(P.env, P.nnei, P.sel, P.ntypes, i, lane, st.nvb, P.nvalid_out)
                      : valid_rows(P.nvalid, P.sel, P.ntypes, i, lane, st.nvb);  // (their __syncwarp orders the reset)
  const int alpha = P.atype ? clampi(__ldg(P.atype + i), 0, P.ntypes - 1) : 0;
  unsigned char *occ = P.occ + ((size_t)alpha * P.tiles_all + (size_t)(i / kTileAtoms)) * P.nsl;
  short *keys = P.keys + i * P.cap;
  double *Wl = kMom ? P.W + (size_t)a * P.cap * 24 + min(lane, 23) : nullptr;
  int nslot = 0;
  int eb = 0;  // largest exponent field written by this lane
  const int lk = min(lane / 6, 3), lq = lane - 6 * (lane / 6);
  const double *srow = P.s + i * P.nnei;
  const double *Rrow = P.Rt + i * P.nnei * 4;
  for (int base = 0; base < nv; base += 32) {
    const int v = base + lane;
    double r[4] = {0.0, 0.0, 0.0, 0.0}, u = 0.0;
    int key = -1;
    if (v < nv) {
      int b;
      double sv;
      double t;
      if constexpr (kEnv) {
        const int row = valid_row(v, st.nvb, P.sel, P.ntypes, b);
        const EnvVals ev = env_vals(P.env, i, __ldg(P.env.nlist + i * P.nnei + row));
        sv = ev.r4[0];
#pragma unroll
        for (int k = 0; k < 4; ++k) r[k] = ev.r4[k];
      } else {
        const int row = valid_row(v, st.nvb, P.sel, P.ntypes, b);
        sv = __ldg(srow + row);
        if constexpr (kMom) {
          const Vec4<double> rr = ld4(Rrow + (size_t)row * 4);
          r[0] = rr.x, r[1] = rr.y, r[2] = rr.z, r[3] = rr.w;
        }
      }
      bool clamped;
      const int l = locate_fast(P.g, P.gf, P.nodes, sv, t, clamped);
      key = b * P.g.nint + l;
      u = t * (l < P.g.n0 ? P.g.inv0 : P.g.inv1);
    }
    // the batch's runs and their slots
    const int prev = __shfl_up_sync(0xffffffffu, key, 1);
    const bool start = v < nv && (lane == 0 || key != prev);
    int slot = start ? (int)smap[key] : 0;
    const bool need = slot < 0;
    unsigned starts = __ballot_sync(0xffffffffu, start);
    bool fresh = false;
    if (__any_sync(0xffffffffu, need)) {
      const unsigned peers = __match_any_sync(0xffffffffu, need ? key : ~lane);
      fresh = need && lane == __ffs(peers) - 1;
      const unsigned lead = __ballot_sync(0xffffffffu, fresh);
      if (fresh) {
        slot = nslot + __popc(lead & ((1u << lane) - 1u));
        smap[key] = (short)slot;
        keys[slot] = (short)key;
        occ[kQ * key / kTK] = 1;  // the key's entries 6 key .. 6 key + 5, in one or two slices
        occ[(kQ * key + kQ - 1) / kTK] = 1;
      }
      const int led = __shfl_sync(0xffffffffu, slot, __ffs(peers) - 1);
      if (need) slot = led;
      nslot += __popc(lead);
    }
    if constexpr (kMom) {
      bool wild = false;  // uniform
      int sh[4];
#pragma unroll
      for (int k = 0; k < 4; ++k)
        sh[k] = batch_places(__reduce_max_sync(0xffffffffu, __double2hiint(r[k]) & 0x7fffffff), wild);
      // |u| < 1.125 unless s is NaN (t lies in its interval but for a hair)
      wild = wild || __any_sync(0xffffffffu, (__double2hiint(u) & 0x7fffffff) >= 0x3ff20000);
      if (!wild) {
        Fix *fr = reinterpret_cast<Fix *>(&st.r[0][lane]), *ft = reinterpret_cast<Fix *>(&st.tp[0][lane]);
#pragma unroll
        for (int k = 0; k < 4; ++k)  // (the shift is uniform, and negative from 2^57 up)
          fr[33 * k] = fx::limbs<L>(sh[k] < 0 ? fx::from_double_any(r[k], sh[k]) : fx::from_double(r[k], sh[k]));
        const Fix u1 = fx::limbs<L>(fx::from_double(u, 2 * L)), u2 = fx::limbs<L>(fx::mul<L>(u1, u1)),
                  u3 = fx::limbs<L>(fx::mul<L>(u2, u1));
        ft[33 * 0] = Fix{0, 1 << L};
        ft[33 * 1] = u1;
        ft[33 * 2] = u2;
        ft[33 * 3] = u3;
        ft[33 * 4] = fx::limbs<L>(fx::mul<L>(u2, u2));
        ft[33 * 5] = fx::limbs<L>(fx::mul<L>(u3, u2));
      } else {
#pragma unroll
        for (int k = 0; k < 4; ++k) st.r[k][lane] = __double_as_longlong(r[k]);
        double up = 1.0;
#pragma unroll
        for (int q = 0; q < 6; ++q, up *= u) st.tp[q][lane] = __double_as_longlong(up);
      }
      __syncwarp();
      const int scale = -(lk < 2 ? (lk ? sh[1] : sh[0]) : (lk == 2 ? sh[2] : sh[3]));
      const int tag = slot | (fresh ? 1 << 16 : 0);
      const int cnt = min(32, nv - base);
      while (starts) {  // uniform, run by run
        const int j0 = __ffs(starts) - 1;
        starts &= starts - 1;
        const int j1 = starts ? __ffs(starts) - 1 : cnt;
        const int run = __shfl_sync(0xffffffffu, tag, j0);
        if (lane < 24) {
          double *w = Wl + (run & 0xffff) * 24;
          const bool add = !(run >> 16);
          const double old = add ? *w : 0.0;
          double x = 0.0;
          if (!wild) {
            const Fix *pr = reinterpret_cast<const Fix *>(st.r[lk]), *pt = reinterpret_cast<const Fix *>(st.tp[lq]);
            fx::Acc acc;
            int j = j0;
            for (; j + 4 <= j1; j += 4)
#pragma unroll
              for (int h = 0; h < 4; ++h) acc.mad(pr[j + h], pt[j + h]);
#pragma unroll 1
            for (; j < j1; ++j) acc.mad(pr[j], pt[j]);
            x = fx::to_double(fx::over_unit<L>(acc), scale);
          } else {
            for (int j = j0; j < j1; ++j)
              x = fma(__longlong_as_double(st.r[lk][j]), __longlong_as_double(st.tp[lq][j]), x);
          }
          if (add) x += old;
          *w = x;
          eb = max(eb, exp_bits(x));
        }
      }
    }
    __syncwarp();
  }
  if (lane == 0) P.nslots[i] = nslot;
  if constexpr (kMom) {
    short *map = P.map + a * map_stride(P.nkeys);
    for (int k = lane; k < map_stride(P.nkeys) / 8; k += 32)
      reinterpret_cast<int4 *>(map)[k] = reinterpret_cast<const int4 *>(smap)[k];
    int m = eb;  // per k: the largest over its six lanes
#pragma unroll
    for (int q = 1; q < 6; ++q) m = max(m, __shfl_sync(0xffffffffu, eb, min(lane + q, 31)));
    if (lane < 24 && lane % 6 == 0) P.fexp[kCols * a + lane / 6] = exp_of_max(m);
  }
}

// The used K slices of each tile of the chunk, in order, and their count, per centre type (one warp per
// (type, tile)).
__global__ void __launch_bounds__(128) slice_list_kernel(const unsigned char *__restrict__ occ, int64_t tiles_all,
                                                         int64_t tile0, int64_t ntiles, int ntypes, int nsl,
                                                         short *__restrict__ list, int *__restrict__ count) {
  const int lane = threadIdx.x & 31;
  const int64_t w = (int64_t)blockIdx.x * 4 + (threadIdx.x >> 5);
  if (w >= (int64_t)ntypes * ntiles) return;  // warp-uniform
  const int t = (int)(w / ntiles);
  const int64_t tile = w - (int64_t)t * ntiles;
  const unsigned char *f = occ + ((size_t)t * tiles_all + tile0 + tile) * nsl;
  short *out = list + ((size_t)t * ntiles + tile) * nsl;
  int rank = 0;
  for (int b = 0; b < nsl; b += 32) {  // uniform
    const bool used = b + lane < nsl && f[b + lane] != 0;
    const unsigned m = __ballot_sync(0xffffffffu, used);
    if (used) out[rank + __popc(m & ((1u << lane) - 1u))] = (short)(b + lane);
    rank += __popc(m);
  }
  if (lane == 0) count[(size_t)t * ntiles + tile] = rank;
}

// The exponents of the backward's fixed points: from the row exponents Eexp [ntypes][Mp] of its A operand,
// kexp [ntypes][nkeys] and, of the chunk's dT columns, gexp.
struct GradExps {
  const int *Eexp;
  int64_t Mp;
  int nkeys, n0, nint, e0, e1;
  int2 *kexp;
  int *gexp;
};

// Exclusive prefix sum over a block of 1024 threads of one value per thread; the block's total in *total.
__device__ long long block_scan_1024(long long v, long long *red, long long *total) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  long long x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const long long y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) red[wid] = x;
  __syncthreads();
  if (wid == 0) {
    long long z = red[lane];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const long long y = __shfl_up_sync(0xffffffffu, z, o);
      if (lane >= o) z += y;
    }
    red[lane] = z;  // inclusive over the warps
  }
  __syncthreads();
  const long long before = (wid ? red[wid - 1] : 0ll) + x - v;
  *total = red[31];
  __syncthreads();  // red is reused by the next scan
  return before;
}

// The forward GEMM's schedule over one chunk: every item (type, tile, 128-row tile of A) with used slices
// costs its slice count plus kEpiCost; CTA b takes the cost range [b R, (b + 1) R) of the items' running
// sum, R = ceil(total / ncta), so that every CTA gets the same work.  An item is cut where a CTA's range
// begins and every 112 slices (the exactness bound of a share); the pieces of a cut item write their
// partial results to consecutive part slots, which fwd_finish_kernel sums.  R is at least kMinRange: on a few
// atoms, ranges of a slice or two took longer to sum than they saved in the GEMM.  One block of 1024 threads,
// each over a run of consecutive items; costs in 32 bits, a 64-bit division a piece having set its time.
// Measured, 64 atoms with 32 channels (schedule + GEMM + finish, us): 64 bits and no least range 38, 32 bits and
// none 33, least range 3: 30, 6: 29, 12: 31; 192 atoms of water 44 without, 42 with 6; above 1,000 atoms no
// difference but the schedule's own 6.6 -> 6.0.
constexpr int kMinRange = kEpiCost;
static_assert((int64_t)DP_MAX_TYPES * (kChunkAtoms / kTileAtoms) * ((DP_MAX_M1 + kTM - 1) / kTM) *
                      ((kMaxKeys * kQ + kTK - 1) / kTK + kEpiCost) < (1ll << 30), "a schedule's costs fit 32 bits");
__global__ void __launch_bounds__(1024) fwd_schedule_kernel(const int *__restrict__ scount, int64_t nitems,
                                                            int64_t ntiles, int nmt, int ncta, int4 *__restrict__ pieces,
                                                            int *__restrict__ pcta, int *__restrict__ cta_start,
                                                            int *__restrict__ npieces, int *__restrict__ pfirst) {
  __shared__ long long red[32];
  const int64_t per = (nitems + 1023) / 1024;
  const int64_t i0 = min(nitems, (int64_t)threadIdx.x * per), i1 = min(nitems, i0 + per);
  auto ns_of = [&](int64_t it) { return scount[it / nmt]; };  // item (t ntiles + tile) nmt + mt
  long long c = 0;
  for (int64_t it = i0; it < i1; ++it) {
    const int ns = ns_of(it);
    c += ns > 0 ? ns + kEpiCost : 0;
  }
  long long total;
  const int P0 = (int)block_scan_1024(c, red, &total);
  const int R = max(kMinRange, ((int)total + ncta - 1) / ncta);
  // the pieces of an item: cut where P + x reaches a multiple of R and where x reaches a multiple of 112
  auto for_pieces = [&](int P, int ns, auto &&f) {
    for (int x = 0; x < ns;) {
      const int b = (P + x) / R;
      const int e = min(ns, min((b + 1) * R - P, (x / kShareSlices + 1) * kShareSlices));
      f(x, e - x, min(b, ncta - 1));
      x = e;
    }
  };
  long long np = 0, nslot = 0;
  int P = P0;
  for (int64_t it = i0; it < i1; ++it) {
    const int ns = ns_of(it);
    int n = 0;
    for_pieces(P, ns, [&](int, int, int) { ++n; });
    np += n;
    nslot += n > 1 ? n : 0;
    P += ns > 0 ? ns + kEpiCost : 0;
  }
  long long np_total, nslot_total;
  long long pbase = block_scan_1024(np, red, &np_total);
  long long sbase = block_scan_1024(nslot, red, &nslot_total);
  P = P0;
  for (int64_t it = i0; it < i1; ++it) {
    const int ns = ns_of(it);
    int n = 0;
    for_pieces(P, ns, [&](int, int, int) { ++n; });
    npieces[it] = n;
    pfirst[it] = n > 1 ? (int)sbase : -1;
    const int64_t tt = it / nmt;
    const int mt = (int)(it - tt * nmt), t = (int)(tt / ntiles), tile = (int)(tt - (int64_t)t * ntiles);
    for_pieces(P, ns, [&](int x, int len, int cta) {
      // tile, (type | mt << 4 | slices << 8), first slice in the tile's list, part slot
      pieces[pbase] = make_int4(tile, t | mt << 4 | len << 8, x, n > 1 ? (int)sbase++ : -1);
      pcta[pbase++] = cta;
    });
    P += ns > 0 ? ns + kEpiCost : 0;
  }
  __syncthreads();
  // CTA b's pieces start at the first piece of a CTA >= b (pieces come in CTA order)
  for (long long i = threadIdx.x; i < np_total; i += blockDim.x) {
    const int cb = pcta[i], ca = i > 0 ? pcta[i - 1] : -1;
    for (int b = ca + 1; b <= cb; ++b) cta_start[b] = (int)i;
  }
  if (threadIdx.x == 0) {
    const int last = np_total > 0 ? pcta[np_total - 1] : -1;
    for (int b = last + 1; b <= ncta; ++b) cta_start[b] = (int)np_total;
  }
}

// The exponents of the backward's fixed points for every centre type and key (tg::key_exps), from the row
// exponents of its A operand; a share of them per block of the units kernels below.
__device__ __forceinline__ void fill_key_exps(const GradExps &X, int ntypes) {
  const int total = ntypes * X.nkeys;
  for (int x = blockIdx.x * blockDim.x + threadIdx.x; x < total; x += gridDim.x * blockDim.x) {
    const int t = x / X.nkeys, key = x - t * X.nkeys;
    X.kexp[x] = tg::key_exps(X.Eexp + (size_t)t * X.Mp + kQ * key, key % X.nint < X.n0 ? X.e0 : X.e1);
  }
}

// The backward GEMM's units: the (tile, 128-row output tile) pairs whose K slices some atom of the tile
// uses, per centre type (one thread per (type, tile)).
__global__ void __launch_bounds__(128) bwd_units_kernel(const unsigned char *__restrict__ occ, int64_t tiles_all,
                                                        int64_t tile0, int64_t ntiles, int ntypes, int nsl, int nmt,
                                                        int64_t maxunits, int *__restrict__ units,
                                                        int *__restrict__ nunits, const GradExps X,
                                                        const int *__restrict__ fexp, int log_M1) {
  fill_key_exps(X, ntypes);
  // sum_m |dT_km| < M1 2^F of every column
  for (int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; c < ntiles * kTN; c += (int64_t)gridDim.x * blockDim.x)
    X.gexp[c] = fexp[c] >= kNonFinite ? kNonFinite : fexp[c] + log_M1;
  const int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (x >= (int64_t)ntypes * ntiles) return;
  const int t = (int)(x / ntiles);
  const int64_t tile = x - (int64_t)t * ntiles;
  const unsigned char *f = occ + ((size_t)t * tiles_all + tile0 + tile) * nsl;
  constexpr int kPer = kTM / kTK;  // K slices per 128-row output tile
  for (int mt = 0; mt < nmt; ++mt) {
    bool any = false;
    for (int q = mt * kPer; q < min(nsl, mt * kPer + kPer); ++q) any |= f[q] != 0;
    if (any) units[(size_t)t * maxunits + atomicAdd(nunits + t, 1)] = tg::unit_code((int)tile, mt);
  }
}

// The 7 x 8-bit backward GEMM's units: the (8-atom tile, 128-row output tile) pairs that hold the slot
// of some atom of the tile of type t, from the atoms' slot keys (a key's rows are 6 key .. 6 key + 5), of every
// centre type in one list; one block per (type, tile), a warp per atom, the row tiles marked in a shared-memory
// bit set.
constexpr int kMaxRowTiles = 256;
static_assert((int64_t)kMaxKeys * kQ <= (int64_t)kMaxRowTiles * kTM, "row tiles of the backward A fit the bit set");
__global__ void __launch_bounds__(32 * tb::kAtomsB) bwd_units8_kernel(const short *__restrict__ keys,
                                                                    const int *__restrict__ nslots,
                                                                    const int32_t *__restrict__ atype, int ntypes,
                                                                    int cap, int64_t atom0, int64_t natoms,
                                                                    int64_t ntiles8,
                                                                    int *__restrict__ units, int *__restrict__ nunits,
                                                                    const GradExps X) {
  fill_key_exps(X, ntypes);
  __shared__ unsigned bits[kMaxRowTiles / 32];
  const int lane = threadIdx.x & 31, al = threadIdx.x >> 5;
  const int t = (int)(blockIdx.x / ntiles8);
  const int64_t tile = blockIdx.x - (int64_t)t * ntiles8;
  if (threadIdx.x < kMaxRowTiles / 32) bits[threadIdx.x] = 0u;
  __syncthreads();
  const int64_t a = tile * tb::kAtomsB + al, i = atom0 + a;
  if (a < natoms && (!atype || clampi(atype[i], 0, ntypes - 1) == t)) {  // warp-uniform
    const int ns = nslots[i];
    for (int slot = lane; slot < ns; slot += 32) {
      const int r0 = kQ * (int)keys[i * cap + slot], m_lo = r0 / kTM, m_hi = (r0 + kQ - 1) / kTM;
      atomicOr(&bits[m_lo >> 5], 1u << (m_lo & 31));
      atomicOr(&bits[m_hi >> 5], 1u << (m_hi & 31));
    }
  }
  __syncthreads();
  if (al != 0) return;
  const unsigned word = lane < kMaxRowTiles / 32 ? bits[lane] : 0u;
  const int cnt = __popc(word);
  int before = cnt;  // inclusive prefix over the lanes
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, before, o);
    if (lane >= o) before += y;
  }
  const int total = __shfl_sync(0xffffffffu, before, 31);
  int base = 0;
  if (lane == 0 && total) base = atomicAdd(nunits, total);
  base = __shfl_sync(0xffffffffu, base, 0) + before - cnt;
  for (unsigned m = word; m; m &= m - 1u) units[base++] = tb::unit_code((int)tile, 32 * lane + __ffs((int)m) - 1, t);
}

// The forward's finish, one block per atom of the chunk: T of an atom whose item (its centre type, its
// tile, a 128-row tile of A) was cut into several pieces -- the pieces' exact integers added as 128-bit
// integers and rounded once to f64 (s128_to_f64: no FP64 instruction) -- or has no used slices (T = 0);
// the other atoms' T the GEMM wrote.  Then, when D is wanted, the atom's descriptor D[m][n] =
// sum_k T[k][m] T[k][n] (n < M2) from its T staged in shared memory, by the descriptor call's own function,
// so that the two give the same bits.
__global__ void __launch_bounds__(128) fwd_finish_kernel(const longlong2 *__restrict__ part, int Mp,
                                                         const int *__restrict__ eexp, const int *__restrict__ fexp,
                                                         const int *__restrict__ npieces,
                                                         const int *__restrict__ pfirst, int64_t ntiles, int nmt,
                                                         int64_t atom0, const int32_t *__restrict__ atype,
                                                         int ntypes, int M1, double *__restrict__ T, int M2,
                                                         double *__restrict__ D) {
  extern __shared__ __align__(16) double Ts[];  // when D is wanted: [4][M1], T, and desc_tile's room after it
  const int64_t a = blockIdx.x;
  const int64_t tile = a / kTileAtoms;
  const int al = (int)(a - tile * kTileAtoms);
  const int t = atype ? clampi(atype[atom0 + a], 0, ntypes - 1) : 0;
  const int64_t item0 = ((int64_t)t * ntiles + tile) * nmt;
  bool direct = true;
  for (int mt = 0; mt < nmt; ++mt) direct = direct && npieces[item0 + mt] == 1;
  if (direct && !D) return;  // uniform
  double *Ta = T + (atom0 + a) * kCols * M1;
  for (int e = threadIdx.x; e < kCols * M1; e += blockDim.x) {
    const int k = e / M1, m = e - k * M1, col = al * kCols + k;
    const int np = npieces[item0 + m / kTM];
    double v;
    if (np == 1) {
      v = Ta[e];  // written by the GEMM (read only for D)
    } else {
      const int first = pfirst[item0 + m / kTM];
      long long hi = 0;
      unsigned long long lo = 0;
      bool nan = false;
      for (int z = 0; z < np; ++z) {  // np == 0: a tile without used slices, whose atoms have no valid rows
        const longlong2 x = part[((size_t)(first + z) * kTN + col) * Mp + m];
        const unsigned long long l = lo + (unsigned long long)x.x;
        hi += x.y + (l < lo ? 1 : 0);
        lo = l;
        nan = nan || x.y == tg::kPartNaN;
      }
      bool rare = false;
      const int E = eexp[(size_t)t * Mp + m], F = fexp[tile * kTN + col];
      v = s128_to_f64<kOutExp>(hi, lo, E, F, rare);
      if (rare) v = output_value((__int128)(((unsigned __int128)(unsigned long long)hi << 64) | lo), E, F);
      if (nan) v = __longlong_as_double(0x7ff8000000000000ll);
      Ta[e] = v;
    }
    if (D) Ts[e] = v;
  }
  if (!D) return;  // uniform
  __syncthreads();
  dfx::desc_tile(Ts, M1, M2, D + (atom0 + a) * (int64_t)M1 * M2);
}

struct RowsParams {
  const double *s, *Rt;
  const int32_t *nvalid, *atype;
  TableGeom g;
  TableGeomF gf;
  const double *nodes;  // [nint + 1] (the plan's)
  int64_t atom0;
  int nnei, ntypes, nkeys, cap;
  int sel[DP_MAX_TYPES];
  const short *keys;   // [nloc][cap]: key of each slot
  const int *nslots;   // [nloc]
  const fx::Fix *dW;   // [natoms][cap][24]: the backward GEMM's result per slot, dW[k][q] at 6 k + q
  const int2 *kexp;    // [ntypes][nkeys] exponents of those fixed points (key_exps), and
  const int *gexp;     // [4 natoms]: 2^gexp > sum_m |dT_km| of atom a at 4 a + k
  int e0, e1;          // binary places of u = t 2^e in the fine and the coarse segment
  const int *bad;      // nonzero: a GEMM wait gave up, the results are NaN
  double *ds, *dRt;
  int64_t natoms;
  EnvRow env;             // rows_force_kernel: rows from coordinates,
  double *F, *virial;     // and the forces [nall][3] and virial [9] they add to
};

// The atom's exponents gexp, every one nonfinite where a GEMM wait gave up; `plain`: results made with them
// and with plain key exponents (|.| <= 400) stay normal doubles, however small or large.
__device__ __forceinline__ int4 atom_exps(const RowsParams &P, int64_t a, bool &plain) {
  int4 g = __ldg(reinterpret_cast<const int4 *>(P.gexp) + a);
  if (__ldg(P.bad)) g = make_int4(kNonFinite, kNonFinite, kNonFinite, kNonFinite);
  plain = max(max(abs(g.x), abs(g.y)), max(abs(g.z), abs(g.w))) <= 400;
  return g;
}

__device__ __noinline__ double odd_double(long long v, int e, bool nan) {
  return nan ? __longlong_as_double(0x7ff8000000000000ll) : scalbn((double)v, e);
}

// One row's dE/dR~[k] = P_k(t) = sum_q dW[k][q] t^q and dE/ds = sum_k R~[k] P_k'(t), from its slot's 24
// fixed points (tg::key_exps), in integer arithmetic (fixed.cuh): with u = t 2^e,
//   P_k = d_0 + sum_q D_q u^q / q,   P_k' = 2^e sum_q D_q u^(q-1),
// two sums of products per k, each rounded once to f64.  Why: 42 FP64 instructions a row bound the kernel
// (91 % of that pipe); the limb products take the integer pipes 250 clocks of a sub-partition against 2,900,
// and the FP64 pipe keeps the conversions and the last dot product (14 instructions).  Measured with 1.7 M
// rows (copper, 4,096 atoms): 0.137 -> 0.073 ms; 1.1 M (water): 0.089 -> 0.061 ms.
struct RowPoly {
  fx::Fix u1, u2, u3, u4, w2, w3, w4, w5;  // u^q and u^q / q
  int2 ke;
  int e, drop, half;
  bool plain, nan;
};
// nan: the row's interval has no slot.
__device__ __forceinline__ RowPoly row_poly(const int2 ke, bool plain, double t, int e, bool nan) {
  constexpr int L = tg::kGradLimb;
  using fx::Fix;
  RowPoly R;
  R.u1 = fx::limbs<L>(fx::from_double_any(t, 2 * L + e));  // (any step of the table)
  const long long s2 = fx::mul<L>(R.u1, R.u1);
  R.u2 = fx::limbs<L>(s2);
  R.u3 = fx::limbs<L>(fx::mul<L>(R.u2, R.u1));
  const long long s4 = fx::mul<L>(R.u2, R.u2);
  R.u4 = fx::limbs<L>(s4);
  constexpr Fix third{0x15555555, 0x15555555}, fifth{-0x0ccccccd, 0x0ccccccd};  // 2^60 / 3, 2^60 / 5
  R.w2 = fx::limbs<L>(s2 >> 1);
  R.w3 = fx::limbs<L>(fx::mul<L>(R.u3, third));
  R.w4 = fx::limbs<L>(s4 >> 2);
  R.w5 = fx::limbs<L>(fx::mul<L>(fx::limbs<L>(fx::mul<L>(R.u4, R.u1)), fifth));
  R.ke = ke;
  R.e = e;
  R.drop = ke.x - ke.y;  // the constant's units over the slope's, as a shift: >= 1
  R.half = R.drop < 32 ? (int)((1u << R.drop) >> 1) : 0;  // so that it rounds (beyond, the constant decides alone)
  R.plain = plain && max(abs(ke.x), abs(ke.y)) <= 400 && R.drop < 32;
  R.nan = nan || (__double2hiint(t) & 0x7ff00000) == 0x7ff00000;  // (a NaN s)
  return R;
}
// P_k and P_k' of component k, whose column's exponent is g.
__device__ __forceinline__ void row_component(const RowPoly &R, const fx::Fix *__restrict__ slot, int k, int g,
                                              double &P, double &dP) {
  constexpr int L = tg::kGradLimb;
  using fx::Fix;
  const int4 *c = reinterpret_cast<const int4 *>(slot) + 3 * k;
  const int4 c01 = __ldg(c), c23 = __ldg(c + 1), c45 = __ldg(c + 2);
  const Fix c0{c01.x, c01.y}, c1{c01.z, c01.w}, c2{c23.x, c23.y}, c3{c23.z, c23.w}, c4{c45.x, c45.y},
      c5{c45.z, c45.w};
  fx::Acc p, q;
  p.hi = R.half;
  p.mad(c1, R.u1);
  p.mad(c2, R.w2);
  p.mad(c3, R.w3);
  p.mad(c4, R.w4);
  p.mad(c5, R.w5);
  q.mad(c2, R.u1);
  q.mad(c3, R.u2);
  q.mad(c4, R.u3);
  q.mad(c5, R.u4);
  const long long pv = fx::over_unit<L>(p), qv = fx::whole<L>(c1) + fx::over_unit<L>(q);
  const int ep = R.ke.x + g - tg::kGradPlaces, eq = R.ke.y + g - tg::kGradPlaces + R.e;
  if (R.plain) {
    const int ph = (int)(pv >> 32);
    const long long ps = (long long)(ph >> R.drop) << 32 | __funnelshift_r((unsigned)pv, (unsigned)ph, R.drop);
    P = fx::to_double(fx::whole<L>(c0) + ps, ep);
    dP = fx::to_double(qv, eq);
  } else {  // an inf or NaN in dT or the table, an abandoned GEMM wait, or an extreme scale
    P = odd_double(fx::whole<L>(c0) + (pv >> min(max(R.drop, 1), 63)), ep, R.ke.x >= kNonFinite || g >= kNonFinite);
    dP = odd_double(qv, eq, R.ke.y >= kNonFinite || g >= kNonFinite);
  }
  if (R.nan) P = dP = __longlong_as_double(0x7ff8000000000000ll);
}

// One warp per atom, a lane per valid row: the row's interval from s, its run slot from the atom's key map
// (shared memory), the slot's gradient coefficients dW[k][q] read through L1 (the rows of a run share
// them), and dE/dR~ and dE/ds from them (row_component); padded rows get zeros.  Seven blocks an SM keep 4,096
// atoms in one wave (copper: six 0.094 ms, eight, with spills, 0.079).
__global__ void __launch_bounds__(32 * kRowsWarps, 7) rows_kernel(const RowsParams P) {
  __shared__ int nvbw[kRowsWarps][DP_MAX_TYPES];
  extern __shared__ __align__(16) short smapw[];  // [kRowsWarps][map_stride(nkeys)]
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t a = (int64_t)blockIdx.x * kRowsWarps + warp;
  if (a >= P.natoms) return;  // warp-uniform
  int *nvb = nvbw[warp];
  short *smap = smapw + (size_t)warp * map_stride(P.nkeys);
  const int64_t i = P.atom0 + a;
  const short *keys = P.keys + i * P.cap;
  const int nslot = P.nslots[i];
  for (int k = lane; k < map_stride(P.nkeys) / 8; k += 32)
    reinterpret_cast<int4 *>(smap)[k] = make_int4(-1, -1, -1, -1);
  __syncwarp();
  for (int x = lane; x < nslot; x += 32) smap[keys[x]] = (short)x;  // the map of the atom's keys
  const int nv = valid_rows(P.nvalid, P.sel, P.ntypes, i, lane, nvb);  // (its __syncwarp orders the map)
  const fx::Fix *dWa = P.dW + (size_t)a * P.cap * 24;
  const int2 *kexp = P.kexp + (size_t)(P.atype ? clampi(__ldg(P.atype + i), 0, P.ntypes - 1) : 0) * P.nkeys;
  bool plain;
  const int4 ge = atom_exps(P, a, plain);
  const double *srow = P.s + i * P.nnei;
  const double *Rrow = P.Rt + i * P.nnei * 4;
  double *dsrow = P.ds + i * P.nnei;
  double *drow = P.dRt + i * P.nnei * 4;
  for (int v = lane; v < nv; v += 32) {
    int b;
    const int row = valid_row(v, nvb, P.sel, P.ntypes, b);
    const double sv = __ldg(srow + row);
    double t;
    bool clamped;
    const int l = locate_fast(P.g, P.gf, P.nodes, sv, t, clamped);
    const int key = b * P.g.nint + l;
    const int at = smap[key];  // -1: runs reused from a call on other rows
    const fx::Fix *slot = dWa + max(at, 0) * 24;
    const RowPoly R = row_poly(__ldg(kexp + key), plain, t, l < P.g.n0 ? P.e0 : P.e1, at < 0);
    const double2 *rr = reinterpret_cast<const double2 *>(Rrow + (size_t)row * 4);
    double2 *dr = reinterpret_cast<double2 *>(drow + (size_t)row * 4);
    double ds = 0.0;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const double2 r = __ldg(rr + h);
      double p0, p1, dp0, dp1;
      row_component(R, slot, 2 * h, h ? ge.z : ge.x, p0, dp0);
      row_component(R, slot, 2 * h + 1, h ? ge.w : ge.y, p1, dp1);
      dr[h] = make_double2(p0, p1);
      ds = fma(r.y, dp1, fma(r.x, dp0, ds));
    }
    dsrow[row] = clamped ? 0.0 : ds;
  }
  // padded rows of each segment
  int off = 0;
  for (int b = 0; b < P.ntypes; ++b) {  // uniform
    for (int j = nvb[b] + lane; j < P.sel[b]; j += 32) {
      dsrow[off + j] = 0.0;
      st4(drow + (size_t)(off + j) * 4, 0.0, 0.0, 0.0, 0.0);
    }
    off += P.sel[b];
  }
}

// rows_kernel fused with the environment and the force back end (dp_tabulate_fusion_env_grad_tc_f64): a
// lane per valid row forms the row from coordinates (env_vals, as dp_env_mat), its dE/ds and dE/dR~ as
// rows_kernel does, and from them, in registers, the row's force contribution g = dE/d(x_j - x_i) by
// dp_force_virial's arithmetic: F_i += g, F_j -= g (atomics), virial -= d (x) g; s, R~, ds and dR~ never
// reach memory.  The per-atom sums are reduced over the warp and added once.
__global__ void __launch_bounds__(32 * kRowsWarps, 4) rows_force_kernel(const RowsParams P) {
  __shared__ int nvbw[kRowsWarps][DP_MAX_TYPES];
  extern __shared__ __align__(16) short smapw[];  // [kRowsWarps][map_stride(nkeys)]
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t a = (int64_t)blockIdx.x * kRowsWarps + warp;
  if (a >= P.natoms) return;  // warp-uniform
  int *nvb = nvbw[warp];
  short *smap = smapw + (size_t)warp * map_stride(P.nkeys);
  const int64_t i = P.atom0 + a;
  const short *keys = P.keys + i * P.cap;
  const int nslot = P.nslots[i];
  for (int k = lane; k < map_stride(P.nkeys) / 8; k += 32)
    reinterpret_cast<int4 *>(smap)[k] = make_int4(-1, -1, -1, -1);
  __syncwarp();
  for (int x = lane; x < nslot; x += 32) smap[keys[x]] = (short)x;  // the map of the atom's keys
  const int nv = env_valid_rows(P.env, P.nnei, P.sel, P.ntypes, i, lane, nvb, nullptr);  // (orders the map)
  const fx::Fix *dWa = P.dW + (size_t)a * P.cap * 24;
  const int2 *kexp = P.kexp + (size_t)(P.atype ? clampi(__ldg(P.atype + i), 0, P.ntypes - 1) : 0) * P.nkeys;
  bool plain;
  const int4 ge = atom_exps(P, a, plain);
  double sum[16];  // the force on atom i, the virial (nine), padding
#pragma unroll
  for (int x = 0; x < 16; ++x) sum[x] = 0.0;
  for (int v = lane; v < nv; v += 32) {
    int b;
    const int row = valid_row(v, nvb, P.sel, P.ntypes, b);
    const int j = __ldg(P.env.nlist + i * P.nnei + row);
    const EnvVals ev = env_vals(P.env, i, j);
    double t;
    bool clamped;
    const int l = locate_fast(P.g, P.gf, P.nodes, ev.r4[0], t, clamped);
    const int key = b * P.g.nint + l;
    const int at = smap[key];  // -1: runs reused from a call on other rows
    const fx::Fix *slot = dWa + max(at, 0) * 24;
    const RowPoly R = row_poly(__ldg(kexp + key), plain, t, l < P.g.n0 ? P.e0 : P.e1, at < 0);
    // dE/ds = sum_k R~[k] P_k', R~[1 .. 3] = ce d
    double d4[4], dp[4];
#pragma unroll
    for (int k = 0; k < 4; ++k)
      row_component(R, slot, k, k == 0 ? ge.x : k == 1 ? ge.y : k == 2 ? ge.z : ge.w, d4[k], dp[k]);
    double ce = ev.a;
    if (!P.env.unit) ce *= P.env.inv_std_all;  // uniform
    double ds = fma(dp[1], ev.d[0], fma(dp[2], ev.d[1], dp[3] * ev.d[2]));
    ds = fma(ce, ds, ev.r4[0] * dp[0]);
    ds = clamped ? 0.0 : ds;
    // as dp_force_virial: the s column feeds both the table input and R~[0]
    const double g0 = ds + d4[0];
    const double p = fma(d4[1], ev.d[0], fma(d4[2], ev.d[1], d4[3] * ev.d[2]));
    double hs = g0 * ev.dsv, hp = (ev.dsv - ev.a) * ev.inv_r;
    if (!P.env.unit) hs *= P.env.inv_std, hp *= P.env.inv_std_all;
    const double cd = fma(hp, p, hs) * ev.inv_r;
    const double g[3] = {fma(cd, ev.d[0], ce * d4[1]), fma(cd, ev.d[1], ce * d4[2]), fma(cd, ev.d[2], ce * d4[3])};
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      sum[c] += g[c];
      atomicAdd(P.F + 3 * (int64_t)j + c, -g[c]);
    }
#pragma unroll
    for (int x = 0; x < 3; ++x)
#pragma unroll
      for (int y = 0; y < 3; ++y) sum[3 + 3 * x + y] = fma(-ev.d[x], g[y], sum[3 + 3 * x + y]);
  }
  // the twelve sums over the warp, halving the values a lane holds at each step (16 adds; 60 summed apart):
  // lane 16 a + 8 b + 4 c + 2 d holds value 8 a + 4 b + 2 c + d
#pragma unroll
  for (int h = 8; h >= 1; h >>= 1) {
    const bool up = lane & (2 * h);
#pragma unroll
    for (int x = 0; x < h; ++x) {
      const double send = up ? sum[x] : sum[x + h], keep = up ? sum[x + h] : sum[x];
      sum[x] = keep + __shfl_xor_sync(0xffffffffu, send, 2 * h);
    }
  }
  sum[0] += __shfl_xor_sync(0xffffffffu, sum[0], 1);
  const int at = lane >> 1;
  if ((lane & 1) == 0 && at < 12) atomicAdd(at < 3 ? P.F + 3 * i + at : P.virial + at - 3, sum[0]);
}

int check_work(const Layout &L, const void *work, size_t nbytes, const char *who) {
  if (!work) return set_error(DP_ERR_NULL, "%s: work is NULL", who);
  if (nbytes < L.total) return set_error(DP_ERR_SHAPE, "%s: work holds %zu bytes, needs %zu", who, nbytes, L.total);
  if (reinterpret_cast<uintptr_t>(work) % 256) return set_error(DP_ERR_SHAPE, "%s: work is not 256-byte aligned", who);
  return DP_OK;
}

// Sizes of a plan for this geometry; DP_OK or an error (message set).
int plan_shape(const dp_table_info *info, int nnei, int ntypes, int M1, TableGeom *g, Shape *S, const char *who) {
  int rc = make_geom(info, g);
  if (rc) return rc;
  if (nnei < 1 || ntypes < 1 || ntypes > DP_MAX_TYPES || M1 < 1 || M1 > DP_MAX_M1)
    return set_error(DP_ERR_SHAPE, "%s: nnei %d, ntypes %d, M1 %d out of range", who, nnei, ntypes, M1);
  if ((int64_t)ntypes * g->nint > kMaxKeys)
    return set_error(DP_ERR_UNSUPPORTED, "%s: ntypes x nint = %lld intervals per centre type, at most %d", who,
                     (long long)ntypes * g->nint, kMaxKeys);
  *S = table_shape(*g, ntypes, M1);
  return DP_OK;
}

// The plan of a call: present, large enough and made for the call's geometry (checked on the host).
int check_plan(const dp_tc_plan *plan, const dp_table_info *info, int nnei, int ntypes, int M1, const Shape &S,
               const char *who) {
  if (!plan || !plan->data) return set_error(DP_ERR_NULL, "%s: plan is NULL", who);
  const dp_table_info &a = plan->info;
  if (a.lower != info->lower || a.upper != info->upper || a.upper_ext != info->upper_ext ||
      a.stride0 != info->stride0 || a.stride1 != info->stride1 || plan->nnei != nnei || plan->ntypes != ntypes ||
      plan->M1 != M1)
    return set_error(DP_ERR_SHAPE, "%s: the plan was made for another table info, nnei, ntypes or M1", who);
  if (plan->bytes < plan_layout(S).total) return set_error(DP_ERR_SHAPE, "%s: plan buffer too short", who);
  return DP_OK;
}

// C' of every centre type from the table, then its digit planes: forward A = C'^T (rows: the
// channels, K: 6 key + q), backward A = C' (rows: 6 key + q, K: the channels).
int make_plan(const double *table, const dp_table_info *info, int nnei, int ntypes, int M1, void *buf,
              size_t bytes, dp_tc_plan *out, void *stream) {
  clear_error();
  static const char *who = "dp_tabulate_tc_plan_f64";
  TableGeom g;
  Shape s{};
  int rc = plan_shape(info, nnei, ntypes, M1, &g, &s, who);
  if (rc) return rc;
  if (!table || !buf || !out) return set_error(DP_ERR_NULL, "%s: table, plan buffer or plan is NULL", who);
  const PlanLayout P = plan_layout(s);
  if (bytes < P.total) return set_error(DP_ERR_SHAPE, "%s: plan buffer holds %zu bytes, needs %zu", who, bytes, P.total);
  if (reinterpret_cast<uintptr_t>(buf) % 256) return set_error(DP_ERR_SHAPE, "%s: plan buffer is not 256-byte aligned", who);
  const cudaStream_t st = (cudaStream_t)stream;
  unsigned char *wk = static_cast<unsigned char *>(buf);
  nodes_kernel<<<(unsigned)((g.nint + 256) / 256), 256, 0, st>>>(g, reinterpret_cast<double *>(wk + P.nodes));
  if ((rc = launch_status(who))) return rc;
  double *Cp = reinterpret_cast<double *>(wk + P.cp);
  const int64_t total = (int64_t)s.ntypes * s.Kp * s.M1;
  const unsigned cblocks = (unsigned)std::min<int64_t>((total + 255) / 256, 1 << 16);
  // forward: the u^q coefficients (the moments are in u, all K entries of a column of one scale)
  coef_kernel<<<cblocks, 256, 0, st>>>(table, g, s.ntypes, s.M1, s.Kp, 1.0 / (double)nnei, true, Cp);
  rc = launch_status(who);
  for (int t = 0; t < s.ntypes && !rc; ++t) {
    const double *Ct = Cp + (size_t)t * s.Kp * s.M1;
    rc = split_rows(Ct, 1, s.M1, s.M1, s.Kp, s.Mpf, s.Kp, kTM, wk + P.afwd + (size_t)t * kS * s.Mpf * s.Kp * 2,
                    wk + P.efwd + (size_t)t * s.Mpf * sizeof(int), st, who);
  }
  // backward: the t^q coefficients (each row 6 key + q of A has its own exponent), so that the rows
  // kernel evaluates its polynomials in t itself, with no 1/Delta on the way in or out
  if (!rc) {
    coef_kernel<<<cblocks, 256, 0, st>>>(table, g, s.ntypes, s.M1, s.Kp, 1.0 / (double)nnei, false, Cp);
    rc = launch_status(who);
  }
  for (int t = 0; t < s.ntypes && !rc; ++t) {
    const double *Ct = Cp + (size_t)t * s.Kp * s.M1;
    unsigned char *eb = wk + P.ebwd + (size_t)t * s.Mpb * sizeof(int);
    if (!rc && s.b8)
      rc = split_rows<Digits7x8>(Ct, s.M1, 1, s.Kp, s.M1, s.Mpb, s.Kpm, kTM,
                                 wk + P.abwd + (size_t)t * tb::kSB * s.Mpb * s.Kpm * 2, eb, st, who);
    else if (!rc)
      rc = split_rows(Ct, s.M1, 1, s.Kp, s.M1, s.Mpb, s.Kpm, kTM, wk + P.abwd + (size_t)t * kS * s.Mpb * s.Kpm * 2, eb,
                      st, who);
  }
  if (rc) return rc;
  out->data = buf;
  out->bytes = bytes;
  out->info = *info;
  out->nnei = nnei;
  out->ntypes = ntypes;
  out->M1 = M1;
  return DP_OK;
}

// Binary places e with |t| 2^e < 1 over an interval of this step, with 5 % to spare (t may lie a hair outside).
int unit_places(double stride) {
  int e = 0;
  std::frexp(1.05 * stride, &e);
  return -e;
}

RunsParams runs_params(const double *s, const double *Rt, const int32_t *nvalid, const int32_t *atype,
                       const TableGeom &g, const Segments &seg, const Shape &S, const Layout &L, unsigned char *wk,
                       int nnei, const double *nodes) {
  RunsParams R{};
  R.s = s;
  R.Rt = Rt;
  R.nvalid = nvalid;
  R.atype = atype;
  R.g = g;
  R.gf = to_f32(g);
  R.nnei = nnei;
  R.ntypes = S.ntypes;
  R.nkeys = S.nkeys;
  R.cap = S.cap;
  R.nsl = S.nsl;
  R.tiles_all = S.tiles_all;
  for (int b = 0; b < DP_MAX_TYPES; ++b) R.sel[b] = seg.sel[b];
  R.keys = reinterpret_cast<short *>(wk + L.keys);
  R.nslots = reinterpret_cast<int *>(wk + L.nslots);
  R.occ = wk + L.occ;
  R.map = reinterpret_cast<short *>(wk + L.map);
  R.fexp = reinterpret_cast<int *>(wk + L.fexp);
  R.nodes = nodes;
  return R;
}

// Validation shared by the forward and the backward; fills g, seg, S, L.
int tc_args(const dp_tc_plan *plan, const dp_table_info *info, const double *s, const double *Rt, int64_t nloc,
            int nnei, int ntypes, const int32_t *sel, int M1, const void *out0, const void *out1, void *work,
            size_t work_bytes, TableGeom *g, Segments *seg, Shape *S, Layout *L, const char *who) {
  int rc = check_fusion_args(plan ? plan->data : nullptr, info, s, Rt, nloc, nnei, ntypes, sel, M1, out0, out1, g, seg);
  if (rc || nloc == 0) return rc;
  Shape T{};
  if ((rc = plan_shape(info, nnei, ntypes, M1, g, &T, who))) return rc;
  if ((rc = check_plan(plan, info, nnei, ntypes, M1, T, who))) return rc;
  *S = make_shape(*g, nloc, nnei, ntypes, M1);
  *L = make_layout(*S);
  if ((rc = check_work(*L, work, work_bytes, who))) return rc;
  return tg::set_smem(who);
}

// env: the rows come from coordinates (dp_tabulate_fusion_env_fwd_tc_f64; s, Rt and nvalid unused, the
// counts of valid rows written to nvalid_out when given).
int fwd(const dp_tc_plan *plan, const dp_table_info *info, const double *s, const double *Rt, const int32_t *nvalid,
        const int32_t *atype, int64_t nloc, int nnei, int ntypes, const int32_t *sel, int M1, double *T, int M2,
        double *D, void *work, size_t work_bytes, void *stream, const EnvRow *env = nullptr,
        int32_t *nvalid_out = nullptr, const char *who = "dp_tabulate_fusion_fwd_tc_f64") {
  clear_error();
  TableGeom g;
  Segments seg;
  Shape S{};
  Layout L{};
  if (D && (M2 < 1 || M2 > M1)) return set_error(DP_ERR_SHAPE, "%s: M2 %d not in 1 .. M1 = %d", who, M2, M1);
  int rc = tc_args(plan, info, s, Rt, nloc, nnei, ntypes, sel, M1, T, T, work, work_bytes, &g, &seg, &S, &L, who);
  if (rc || nloc == 0) return rc;
  const PlanLayout PL = plan_layout(S);
  const unsigned char *pk = static_cast<const unsigned char *>(plan->data);
  const cudaStream_t st = (cudaStream_t)stream;
  unsigned char *wk = static_cast<unsigned char *>(work);
  prof_mark("tc_fwd", st);
  if (cudaMemsetAsync(wk + L.occ, 0, (size_t)ntypes * S.tiles_all * S.nsl, st) != cudaSuccess)
    return set_error(DP_ERR_CUDA, "%s: cudaMemsetAsync: %s", who, cudaGetErrorString(cudaGetLastError()));
  RunsParams R = runs_params(s, Rt, nvalid, atype, g, seg, S, L, wk, nnei,
                             reinterpret_cast<const double *>(pk + PL.nodes));
  R.W = reinterpret_cast<double *>(wk + L.w);
  if (env) {
    R.env = *env;
    R.nvalid_out = nvalid_out;
  }
  longlong2 *part = reinterpret_cast<longlong2 *>(wk + L.part);
  int dev = 0, nsm = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return set_error(DP_ERR_CUDA, "%s: %s", who, cudaGetErrorString(cudaGetLastError()));
  const int ncta = std::max(1, std::min(nsm, kMaxCtasF));
  for (int64_t c0 = 0; c0 < nloc; c0 += S.chunk) {
    const int64_t n = std::min<int64_t>(S.chunk, nloc - c0);
    const int64_t Np = round_up(kCols * n, kTN), ntiles = Np / kTN, tile0 = c0 / kTileAtoms;
    R.atom0 = c0;
    R.natoms = n;
    const dim3 rgrid((unsigned)((n + kRunsWarps - 1) / kRunsWarps));
    if (env)
      runs_kernel<true, true><<<rgrid, 32 * kRunsWarps, kRunsWarps * map_stride(S.nkeys) * sizeof(short), st>>>(R);
    else
      runs_kernel<true><<<rgrid, 32 * kRunsWarps, kRunsWarps * map_stride(S.nkeys) * sizeof(short), st>>>(R);
    if ((rc = launch_status(who))) return rc;
    prof_mark("tc_runs_moments", st);
    const int64_t nlist = (int64_t)ntypes * ntiles;
    slice_list_kernel<<<(unsigned)((nlist + 3) / 4), 128, 0, st>>>(wk + L.occ, S.tiles_all, tile0, ntiles, ntypes,
                                                                    S.nsl, reinterpret_cast<short *>(wk + L.slist),
                                                                    reinterpret_cast<int *>(wk + L.scount));
    if ((rc = launch_status(who))) return rc;
    const int nmt = S.Mpf / kTM;
    fwd_schedule_kernel<<<1, 1024, 0, st>>>(reinterpret_cast<const int *>(wk + L.scount), nlist * nmt, ntiles, nmt, ncta,
                                            reinterpret_cast<int4 *>(wk + L.pieces), reinterpret_cast<int *>(wk + L.pcta),
                                            reinterpret_cast<int *>(wk + L.cta_start),
                                            reinterpret_cast<int *>(wk + L.npieces),
                                            reinterpret_cast<int *>(wk + L.pfirst));
    if ((rc = launch_status(who))) return rc;
    prof_mark("tc_slice_lists", st);
    tg::Params G{};
    G.fwd = true;
    G.aplanes = pk + PL.afwd;
    G.astride = (size_t)kS * S.Mpf * S.Kp * 2;
    G.Eexp = reinterpret_cast<const int *>(pk + PL.efwd);
    G.estride = S.Mpf;
    G.ka = S.nsl;
    G.nmt = nmt;
    G.W = R.W;  // B made from the moments inside the GEMM
    G.map = R.map;
    G.nkeys = S.nkeys;
    G.mstride = map_stride(S.nkeys);
    G.cap = S.cap;
    G.Fexp = R.fexp;
    G.ntiles = ntiles;
    G.Np = Np;
    G.Mp = S.Mpf;
    G.slist = reinterpret_cast<const short *>(wk + L.slist);
    G.scount = reinterpret_cast<const int *>(wk + L.scount);
    G.zmax = S.zmax;
    G.part = part;
    G.tout = T;  // items in one piece write T themselves
    G.pieces = reinterpret_cast<const int4 *>(wk + L.pieces);
    G.cta_start = reinterpret_cast<const int *>(wk + L.cta_start);
    G.ldt = M1;
    G.atype = atype;
    G.natoms = n;
    G.atom0 = c0;
    G.ntypes = ntypes;
    if ((rc = tg::launch(G, st, who, ncta))) return rc;
    prof_mark("tc_gemm_fwd", st);
    fwd_finish_kernel<<<(unsigned)n, 128, D ? dfx::desc_tile_bytes(M1, M2) : 0, st>>>(
        part, S.Mpf, G.Eexp, R.fexp, reinterpret_cast<const int *>(wk + L.npieces),
        reinterpret_cast<const int *>(wk + L.pfirst), ntiles, nmt, c0, atype, ntypes, M1, T, M2, D);
    if ((rc = launch_status(who))) return rc;
    prof_mark("tc_finish_fwd", st);
  }
  return DP_OK;
}

// env: the rows come from coordinates and the rows kernel adds the forces and virial instead of writing
// ds and dRt (dp_tabulate_fusion_env_grad_tc_f64; s, Rt, nvalid, ds and dRt unused; F [nall][3] and
// virial [9] are zeroed first).
int grad(const dp_tc_plan *plan, const dp_table_info *info, const double *s, const double *Rt, const int32_t *nvalid,
         const int32_t *atype, int64_t nloc, int nnei, int ntypes, const int32_t *sel, int M1, const double *dT,
         double *ds, double *dRt, void *work, size_t work_bytes, int flags, void *stream, const EnvRow *env = nullptr,
         double *F = nullptr, double *virial = nullptr, int64_t nall = 0,
         const char *who = "dp_tabulate_fusion_grad_tc_f64") {
  clear_error();
  if (flags & ~DP_TC_REUSE_RUNS) return set_error(DP_ERR_SHAPE, "%s: unknown flags %#x", who, flags);
  TableGeom g;
  Segments seg;
  Shape S{};
  Layout L{};
  int rc = tc_args(plan, info, s, Rt, nloc, nnei, ntypes, sel, M1, env ? (void *)F : ds, env ? (void *)virial : dRt,
                   work, work_bytes, &g, &seg, &S, &L, who);
  if (rc) return rc;
  if (env) {  // the forces and virial are sums: zeroed first, also for nloc = 0
    cudaError_t e = cudaMemsetAsync(virial, 0, 9 * sizeof(double), (cudaStream_t)stream);
    if (e == cudaSuccess && nall > 0) e = cudaMemsetAsync(F, 0, (size_t)nall * 3 * sizeof(double), (cudaStream_t)stream);
    if (e != cudaSuccess) return set_error(DP_ERR_CUDA, "%s: %s", who, cudaGetErrorString(e));
  }
  if (nloc == 0) return DP_OK;
  if (!dT) return set_error(DP_ERR_NULL, "%s: dT is NULL", who);
  const PlanLayout PL = plan_layout(S);
  const unsigned char *pk = static_cast<const unsigned char *>(plan->data);
  const cudaStream_t st = (cudaStream_t)stream;
  unsigned char *wk = static_cast<unsigned char *>(work);
  const bool reuse = (flags & DP_TC_REUSE_RUNS) != 0;
  prof_mark("tc_grad", st);
  if (!reuse && cudaMemsetAsync(wk + L.occ, 0, (size_t)ntypes * S.tiles_all * S.nsl, st) != cudaSuccess)
    return set_error(DP_ERR_CUDA, "%s: cudaMemsetAsync: %s", who, cudaGetErrorString(cudaGetLastError()));
  RunsParams R = runs_params(s, Rt, nvalid, atype, g, seg, S, L, wk, nnei,
                             reinterpret_cast<const double *>(pk + PL.nodes));
  const int mtiles = S.Mpb / kTM;
  fx::Fix *dW = reinterpret_cast<fx::Fix *>(wk + L.w);
  GradExps X{};  // in the region of the forward's partial results, which the backward does not use
  X.Eexp = reinterpret_cast<const int *>(pk + PL.ebwd);
  X.Mp = S.Mpb;
  X.nkeys = S.nkeys;
  X.n0 = g.n0;
  X.nint = g.nint;
  X.e0 = unit_places(g.stride0);
  X.e1 = unit_places(g.stride1);
  X.gexp = reinterpret_cast<int *>(wk + L.part);
  X.kexp = reinterpret_cast<int2 *>(wk + L.part + (size_t)std::max(S.Np, S.Np8) * sizeof(int));
  RowsParams Q{};
  Q.s = s;
  Q.Rt = Rt;
  Q.nvalid = nvalid;
  Q.atype = atype;
  Q.g = g;
  Q.gf = R.gf;
  Q.nodes = R.nodes;
  Q.nnei = nnei;
  Q.ntypes = ntypes;
  Q.nkeys = S.nkeys;
  Q.cap = S.cap;
  for (int b = 0; b < DP_MAX_TYPES; ++b) Q.sel[b] = seg.sel[b];
  Q.keys = R.keys;
  Q.nslots = R.nslots;
  Q.dW = dW;
  Q.kexp = X.kexp;
  Q.gexp = X.gexp;
  Q.e0 = X.e0;
  Q.e1 = X.e1;
  Q.bad = reinterpret_cast<const int *>(wk + L.nunits) + kBadFlag;
  Q.ds = ds;
  Q.dRt = dRt;
  if (env) {
    R.env = *env;
    Q.env = *env;
    Q.F = F;
    Q.virial = virial;
  }
  for (int64_t c0 = 0; c0 < nloc; c0 += S.chunk) {
    const int64_t n = std::min<int64_t>(S.chunk, nloc - c0);
    const int64_t Np = round_up(kCols * n, kTN), ntiles = Np / kTN, tile0 = c0 / kTileAtoms;
    R.atom0 = c0;
    R.natoms = n;
    if (!reuse) {
      const dim3 rgrid((unsigned)((n + kRunsWarps - 1) / kRunsWarps));
      if (env)
        runs_kernel<false, true><<<rgrid, 32 * kRunsWarps, kRunsWarps * map_stride(S.nkeys) * sizeof(short), st>>>(R);
      else
        runs_kernel<false><<<rgrid, 32 * kRunsWarps, kRunsWarps * map_stride(S.nkeys) * sizeof(short), st>>>(R);
      if ((rc = launch_status(who))) return rc;
      prof_mark("tc_runs", st);
    }
    if (S.b8) {
      // B = dT^T on 8-atom tiles in the 7 x 8-bit digits: the columns 4 a + k are the rows of this chunk's dT
      if ((rc = split_rows_1k<Digits7x8>(dT + c0 * kCols * M1, M1, 1, kCols * n, M1, round_up(kCols * n, tb::kTNB),
                                         S.Kpm, tb::kTNB, wk + L.bplanes, wk + L.fexp, X.gexp, st, who)))
        return rc;
      prof_mark("tc_split_dT", st);
      if (cudaMemsetAsync(wk + L.nunits, 0, (kBadFlag + 1) * sizeof(int), st) != cudaSuccess)
        return set_error(DP_ERR_CUDA, "%s: cudaMemsetAsync: %s", who, cudaGetErrorString(cudaGetLastError()));
      const int64_t ntiles8 = (n + tb::kAtomsB - 1) / tb::kAtomsB, nlist = (int64_t)ntypes * ntiles8;
      bwd_units8_kernel<<<(unsigned)nlist, 32 * tb::kAtomsB, 0, st>>>(
          R.keys, R.nslots, atype, ntypes, S.cap, c0, n, ntiles8, reinterpret_cast<int *>(wk + L.units),
          reinterpret_cast<int *>(wk + L.nunits), X);
      if ((rc = launch_status(who))) return rc;
      prof_mark("tc_units", st);
      tb::Params G{};
      G.aplanes = pk + PL.abwd;
      G.astride = (size_t)tb::kSB * S.Mpb * S.Kpm * 2;
      G.Eexp = X.Eexp;
      G.ka = S.Kpm / kTK;
      G.bplanes = wk + L.bplanes;
      G.Fexp = R.fexp;
      G.Mp = S.Mpb;
      G.scat = dW;
      G.kexp = X.kexp;
      G.gexp = X.gexp;
      G.n0 = g.n0;
      G.nint = g.nint;
      G.e0 = X.e0;
      G.e1 = X.e1;
      G.bad = reinterpret_cast<int *>(wk + L.nunits) + kBadFlag;
      G.keys = R.keys;
      G.nslots = R.nslots;
      G.cap = S.cap;
      G.nkeys = S.nkeys;
      G.kq = kQ;
      G.atype = atype;
      G.natoms = n;
      G.atom0 = c0;
      G.ntypes = ntypes;
      G.units = reinterpret_cast<const int *>(wk + L.units);
      G.nunits = reinterpret_cast<const int *>(wk + L.nunits);
      if ((rc = tb::launch(G, st, who))) return rc;
      prof_mark("tc_gemm_grad", st);
    } else {
      // B = dT^T: the columns 4 a + k are the rows of this chunk's dT
      if ((rc = split_rows(dT + c0 * kCols * M1, M1, 1, kCols * n, M1, Np, S.Kpm, kTN, wk + L.bplanes, wk + L.fexp, st,
                           who, kZerosGrad)))
        return rc;
      prof_mark("tc_split_dT", st);
      if (cudaMemsetAsync(wk + L.nunits, 0, (kBadFlag + 1) * sizeof(int), st) != cudaSuccess)
        return set_error(DP_ERR_CUDA, "%s: cudaMemsetAsync: %s", who, cudaGetErrorString(cudaGetLastError()));
      const int64_t nlist = (int64_t)ntypes * ntiles;
      int log_M1 = 0;
      while ((1 << log_M1) < M1) ++log_M1;
      bwd_units_kernel<<<(unsigned)((nlist + 127) / 128), 128, 0, st>>>(wk + L.occ, S.tiles_all, tile0, ntiles, ntypes,
                                                                        S.nsl, mtiles, S.maxunits,
                                                                        reinterpret_cast<int *>(wk + L.units),
                                                                        reinterpret_cast<int *>(wk + L.nunits), X,
                                                                        R.fexp, log_M1);
      if ((rc = launch_status(who))) return rc;
      prof_mark("tc_units", st);
      for (int t = 0; t < ntypes; ++t) {
        tg::Params G{};
        G.fwd = false;
        G.aplanes = pk + PL.abwd + (size_t)t * kS * S.Mpb * S.Kpm * 2;
        G.Eexp = reinterpret_cast<const int *>(pk + PL.ebwd) + (size_t)t * S.Mpb;
        G.ka = S.Kpm / kTK;
        G.nmt = mtiles;
        G.bplanes = wk + L.bplanes;
        G.Fexp = R.fexp;
        G.ntiles = ntiles;
        G.Np = Np;
        G.Mp = S.Mpb;
        G.sflags = wk + L.occ + ((size_t)t * S.tiles_all + tile0) * S.nsl;
        G.nsf = S.nsl;
        G.scat = dW;
        G.kexp = X.kexp + (size_t)t * S.nkeys;
        G.gexp = X.gexp;
        G.n0 = g.n0;
        G.nint = g.nint;
        G.e0 = X.e0;
        G.e1 = X.e1;
        G.bad = reinterpret_cast<int *>(wk + L.nunits) + kBadFlag;
        G.keys = R.keys;
        G.nslots = R.nslots;
        G.cap = S.cap;
        G.nkeys = S.nkeys;
        G.kq = kQ;
        G.atype = atype;
        G.natoms = n;
        G.atom0 = c0;
        G.alpha = t;
        G.ntypes = ntypes;
        G.units = reinterpret_cast<const int *>(wk + L.units) + (size_t)t * S.maxunits;
        G.nunits = reinterpret_cast<const int *>(wk + L.nunits) + t;
        if ((rc = tg::launch(G, st, who))) return rc;
        prof_mark("tc_gemm_grad", st);
      }
    }
    Q.atom0 = c0;
    Q.natoms = n;
    const dim3 qgrid((unsigned)((n + kRowsWarps - 1) / kRowsWarps));
    if (env)
      rows_force_kernel<<<qgrid, 32 * kRowsWarps, kRowsWarps * map_stride(S.nkeys) * sizeof(short), st>>>(Q);
    else
      rows_kernel<<<qgrid, 32 * kRowsWarps, kRowsWarps * map_stride(S.nkeys) * sizeof(short), st>>>(Q);
    if ((rc = launch_status(who))) return rc;
    prof_mark("tc_rows", st);
  }
  return DP_OK;
}

EnvRow env_row(const dp_env_info *e, const double *coord, const int32_t *nlist) {
  EnvRow E{};
  E.coord = coord;
  E.nlist = nlist;
  E.rcs = e->rcs;
  E.rc = e->rc;
  E.inv_width = 1.0 / (e->rc - e->rcs);
  E.mean = e->mean;
  E.inv_std = 1.0 / e->std;
  E.inv_std_all = 1.0 / e->std_all;
  E.kind = e->kind;
  E.unit = e->mean == 0.0 && e->std == 1.0 && e->std_all == 1.0;
  return E;
}

int env_fwd(const dp_tc_plan *plan, const dp_table_info *info, const double *coord, const int32_t *nlist,
            const dp_env_info *env, const int32_t *atype, int64_t nloc, int nnei, int ntypes, const int32_t *sel,
            int M1, int32_t *nvalid, double *T, int M2, double *D, void *work, size_t work_bytes, void *stream) {
  clear_error();
  static const char *who = "dp_tabulate_fusion_env_fwd_tc_f64";
  if (int rc = check_env(env)) return rc;
  const EnvRow E = env_row(env, coord, nlist);
  // coord and nlist stand where the plain call's s and Rt are checked for NULL
  return fwd(plan, info, coord, reinterpret_cast<const double *>(nlist), nullptr, atype, nloc, nnei, ntypes, sel, M1,
             T, M2, D, work, work_bytes, stream, &E, nvalid, who);
}

int env_grad(const dp_tc_plan *plan, const dp_table_info *info, const double *coord, const int32_t *nlist,
             const dp_env_info *env, const int32_t *atype, int64_t nloc, int64_t nall, int nnei, int ntypes,
             const int32_t *sel, int M1, const double *dT, double *F, double *virial, void *work, size_t work_bytes,
             int flags, void *stream) {
  clear_error();
  static const char *who = "dp_tabulate_fusion_env_grad_tc_f64";
  if (int rc = check_env(env)) return rc;
  if (nall < nloc) return set_error(DP_ERR_SHAPE, "%s: nall = %lld < nloc = %lld", who, (long long)nall, (long long)nloc);
  if (!virial || (nall > 0 && !F)) return set_error(DP_ERR_NULL, "%s: NULL output", who);
  const EnvRow E = env_row(env, coord, nlist);
  return grad(plan, info, coord, reinterpret_cast<const double *>(nlist), nullptr, atype, nloc, nnei, ntypes, sel, M1,
              dT, nullptr, nullptr, work, work_bytes, flags, stream, &E, F, virial, nall, who);
}

size_t work_bytes_api(const dp_table_info *info, int64_t nloc, int nnei, int ntypes, int M1) {
  clear_error();
  TableGeom g;
  Shape S{};
  if (nloc < 0) {
    set_error(DP_ERR_SHAPE, "dp_tabulate_tc_work_bytes: nloc %lld < 0", (long long)nloc);
    return 0;
  }
  if (plan_shape(info, nnei, ntypes, M1, &g, &S, "dp_tabulate_tc_work_bytes")) return 0;
  return make_layout(make_shape(g, nloc, nnei, ntypes, M1)).total;
}

size_t plan_bytes_api(const dp_table_info *info, int nnei, int ntypes, int M1) {
  clear_error();
  TableGeom g;
  Shape S{};
  if (plan_shape(info, nnei, ntypes, M1, &g, &S, "dp_tabulate_tc_plan_bytes")) return 0;
  return plan_layout(S).total;
}

}  // namespace tt
}  // namespace

// This unit's GEMM wait timeouts (see tc_gemm.cuh), for dp_tc_wait_timeouts.
int take_wait_timeouts_tabulate(unsigned int *count) { return tc::take_wait_timeouts(count); }

}  // namespace dpc

extern "C" {

size_t dp_tabulate_tc_work_bytes(const dp_table_info *info, int64_t nloc, int nnei, int ntypes, int M1) {
  return dpc::tt::work_bytes_api(info, nloc, nnei, ntypes, M1);
}

size_t dp_tabulate_tc_plan_bytes(const dp_table_info *info, int nnei, int ntypes, int M1) {
  return dpc::tt::plan_bytes_api(info, nnei, ntypes, M1);
}

int dp_tabulate_tc_plan_f64(const double *table, const dp_table_info *info, int nnei, int ntypes, int M1, void *buf,
                            size_t bytes, dp_tc_plan *plan, void *stream) {
  return dpc::tt::make_plan(table, info, nnei, ntypes, M1, buf, bytes, plan, stream);
}

int dp_tabulate_fusion_fwd_tc_f64(const dp_tc_plan *plan, const dp_table_info *info, const double *s, const double *Rt,
                                  const int32_t *nvalid, const int32_t *atype, int64_t nloc, int nnei, int ntypes,
                                  const int32_t *sel, int M1, double *T, int M2, double *D, void *work,
                                  size_t work_bytes, void *stream) {
  return dpc::tt::fwd(plan, info, s, Rt, nvalid, atype, nloc, nnei, ntypes, sel, M1, T, M2, D, work, work_bytes,
                      stream);
}

int dp_tabulate_fusion_env_fwd_tc_f64(const dp_tc_plan *plan, const dp_table_info *info, const double *coord,
                                      const int32_t *nlist, const dp_env_info *env, const int32_t *atype, int64_t nloc,
                                      int nnei, int ntypes, const int32_t *sel, int M1, int32_t *nvalid, double *T,
                                      int M2, double *D, void *work, size_t work_bytes, void *stream) {
  return dpc::tt::env_fwd(plan, info, coord, nlist, env, atype, nloc, nnei, ntypes, sel, M1, nvalid, T, M2, D, work,
                          work_bytes, stream);
}

int dp_tabulate_fusion_env_grad_tc_f64(const dp_tc_plan *plan, const dp_table_info *info, const double *coord,
                                       const int32_t *nlist, const dp_env_info *env, const int32_t *atype,
                                       int64_t nloc, int64_t nall, int nnei, int ntypes, const int32_t *sel, int M1,
                                       const double *dT, double *F, double *virial, void *work, size_t work_bytes,
                                       int flags, void *stream) {
  return dpc::tt::env_grad(plan, info, coord, nlist, env, atype, nloc, nall, nnei, ntypes, sel, M1, dT, F, virial,
                           work, work_bytes, flags, stream);
}

int dp_tabulate_fusion_grad_tc_f64(const dp_tc_plan *plan, const dp_table_info *info, const double *s, const double *Rt,
                                   const int32_t *nvalid, const int32_t *atype, int64_t nloc, int nnei, int ntypes,
                                   const int32_t *sel, int M1, const double *dT, double *ds, double *dRt, void *work,
                                   size_t work_bytes, int flags, void *stream) {
  return dpc::tt::grad(plan, info, s, Rt, nvalid, atype, nloc, nnei, ntypes, sel, M1, dT, ds, dRt, work, work_bytes,
                       flags, stream);
}

}  // extern "C"
