// The AIM matrix-vector product on the grid (Sec. III-A, Eq. 8; filtered: Sec. III-B, Eq. 10).
//
// For each channel (one projection of one right-hand side) the product
//     y = P_t^T [ F^-1( F(c) .* F(b) ) ]_restr ,   b = zero-padded P_s x
// runs as an anterpolation, three grid passes and a gather:
//   k_anterpolate  u = P_s x at the active grid points (deterministic, no atomics).
//   k_row_fwd   the forward P-point row DFT of u. The row has nonzeros only in its first
//               m <= P/2 entries, so X[2k] = DFT_H(a)[k] and X[2k+1] = DFT_H(a w^n)[k],
//               H = P/2, w = exp(-2 pi i/P). Rows of few active points: only the later
//               passes are dense (row_fwd_sparse).
//   k_col_conv  per column q: the same pruned forward DFT along the rows, the product with
//               the stored spectrum column F(c)[., q] (even symmetric, so only
//               (P/2+1)^2 values are stored), and the inverse DFT keeping rows < P/2 only:
//               y[n] = IDFT_H(Y_even)[n] + w^-n IDFT_H(Y_odd)[n].
//   k_row_inv   the inverse row DFT with the same split, scaled by 1/P^2, evaluated at the
//               grid points the test projection reads (the restriction [.]_restr): the two
//               half-transforms are recombined only at those points.
//   k_gather    y_i = sum over projections of coef * (P_t^T v)_i plus the near-field row
//               (C x)_i, eight lanes per unknown, deterministic.
// Each length-H transform runs as register-resident radix-E passes (fft_reg.cuh, E = 16 or 8
// elements per thread, a schedule choice): the first pass reads its operands straight from
// global memory (column and inverse row passes) and the last pass writes straight to global memory (forward row and column passes; the inverse row
// pass keeps its last pass in shared memory for the restriction), so shared memory carries only
// the exchanges between passes. A thread owns TPT transforms: with TPT = 2 the even- and odd-half
// transforms of a line sit in the same thread; with TPT = 1 they sit in adjacent lanes and
// recombine through a lane shuffle (half the registers per thread, twice the threads). Which one
// is faster depends on the element type and on how much of the GPU a launch fills (pass_tpt); the
// autotuner measures both.
// The intermediate m x P grid of a channel is stored as column tiles of W entries
// (W * sizeof(complex) = 32 bytes) so that the column pass reads contiguous blocks and the
// row passes touch whole 32-byte sectors. Only grid rows that hold active points are stored.
#pragma once

#include <algorithm>
#include <climits>
#include <type_traits>
#include <vector>

#include "aim_internal.h"
#include "gridtypes.cuh"

namespace aim {

// ------------------------------------------------------------------------------------
// anterpolation
// ------------------------------------------------------------------------------------
struct AntArgs {
  const double2* x;    // n * nrhs
  int n, nrhs, n_act;
  const int* sc_ptr;
  const int* sc_col;
  const double* w[kMaxProj];
  void* u;             // element type of the grid, channel-major, n_act per channel
};

// u = P_s x at the active points, NP projections of one right-hand side per thread: the row pass
// then starts from values instead of from four dependent loads (row range, entry range, column,
// vector) that one warp of its CTA chases while the others wait at a barrier. Grid-point-major
// lists, so deterministic without atomics. A point has a handful of entries (about 7): the loads
// of up to kAntChunk entries are issued together before their FMAs, which run in entry order as a
// plain loop would.
constexpr int kAntChunk = 8, kAntThreads = 64;

template <typename CT, int NP>
__device__ __forceinline__ void ant_item(const AntArgs& a, long long t) {
  const bool valid = t < (long long)a.n_act * a.nrhs;
  const int r = valid ? (int)(t / a.n_act) : 0, ap = valid ? (int)(t - (long long)r * a.n_act) : 0;
  const double2* xv = a.x + (size_t)r * a.n;
  double re[NP], im[NP];
#pragma unroll
  for (int q = 0; q < NP; ++q) re[q] = im[q] = 0.0;
  const int e0 = a.sc_ptr[ap], e1 = valid ? a.sc_ptr[ap + 1] : e0;
  int col[kAntChunk];
  double ww[NP][kAntChunk];
  auto lists = [&](int e) {   // entries past the end repeat the last one with weight 0
#pragma unroll
    for (int u = 0; u < kAntChunk; ++u) {
      const int ee = min(e + u, e1 - 1);
      col[u] = a.sc_col[max(ee, 0)];
#pragma unroll
      for (int q = 0; q < NP; ++q) ww[q][u] = a.w[q][max(ee, 0)];
    }
  };
  lists(e0);
  grid_dependency_wait();   // the lists belong to the context: only x comes from an earlier kernel
  for (int e = e0; e < e1; e += kAntChunk) {
    if (e != e0) lists(e);
    double2 xx[kAntChunk];
#pragma unroll
    for (int u = 0; u < kAntChunk; ++u) xx[u] = xv[col[u]];
#pragma unroll
    for (int u = 0; u < kAntChunk; ++u) {
      if (e + u < e1) {
#pragma unroll
        for (int q = 0; q < NP; ++q) {
          re[q] = fma(ww[q][u], xx[u].x, re[q]);
          im[q] = fma(ww[q][u], xx[u].y, im[q]);
        }
      }
    }
  }
  if (!valid) return;
  CT* out = static_cast<CT*>(a.u) + (size_t)r * a.n_act + ap;
#pragma unroll
  for (int q = 0; q < NP; ++q) out[(size_t)q * a.nrhs * a.n_act] = cfrom<CT>(re[q], im[q]);
}

template <typename CT, int NP>
__global__ void __launch_bounds__(kAntThreads) k_anterpolate(AntArgs a) {
  ant_item<CT, NP>(a, (long long)blockIdx.x * kAntThreads + threadIdx.x);
}

// ------------------------------------------------------------------------------------
// row pass, forward
// ------------------------------------------------------------------------------------
struct RowFwdArgs {
  const double2* x;     // dense mode: m*m grid per channel
  const void* u;        // sparse mode: values at the active points, channel-major
  int dense;
  int m, n_act;
  const int* row_ptr;
  const int* act_ix;
  void* inter;
  const void* tw;
  int logH, logP, row_lo, nrows;
  int rows_per_cta;
  int qcut;            // columns q with min(q, P - q) > qcut carry a zero spectrum: not stored
  int sparse;          // few active points per row: the first radix runs at the active points only
  int dense_from;      // sparse: rows of more points than this take the dense passes all the same
};

// Output k of a row's transforms into the tiled intermediate: X[2k] and X[2k + 1] are neighbours in
// a tile. With both in the thread they go out as one vector store (32 bytes for the 16-byte types: a
// whole sector; as two stores each was half a sector written twice, 73 of 280 us of the double-float
// pass at 2048 points).
template <typename CT, int TPT>
__device__ __forceinline__ void store_row(CT* out, const RowFwdArgs& a, int rloc, bool live, int half, int k,
                                          const CT (&v)[TPT]) {
  constexpr int W = GridT<CT>::W;
  const int P = 1 << a.logP;
  if (!live) return;
  if constexpr (TPT == 2) {
    const int q = 2 * k;
    if (min(q, P - 1 - q) <= a.qcut) store_pair(&out[((size_t)(q / W) * a.nrows + rloc) * W + (q % W)], v[0], v[1]);
  } else {
    const int q = 2 * k + half;
    if (min(q, P - q) <= a.qcut) out[((size_t)(q / W) * a.nrows + rloc) * W + (q % W)] = v[0];
  }
}

// ------------------------------------------------------------------------------------
// sparse rows
// ------------------------------------------------------------------------------------
// A grid row of a contour holds few active points (about 18 of 2048 at the single-solve scale).
// The length-H transforms of a row split as H = R0 J, n = j + J r: the radix-R0 pass over r has at
// most one nonzero butterfly per active point, so it runs as a scatter of the active points into
// the R0 outputs of their j (forward), or as a sum over the R0 sub-transforms at the active points
// only (inverse), and only the J-point transforms are dense. J is a power of E, so the dense part
// has one or two radix-E passes instead of the three or four of the whole length.
template <int LOGE>
__host__ __device__ __forceinline__ int sparse_logj(int logH) {
  // two dense passes when the sparse radix then stays >= 2, else one
  return logH > 2 * LOGE ? 2 * LOGE : LOGE;
}

// The sparse radix of a transform length: R0 = 2^l0 <= 32, K2 = 2 R0 terms per point (both halves).
struct SparseGeom {
  int logj, l0, k2;
};
template <int LOGE>
__host__ __device__ __forceinline__ SparseGeom sparse_geom(int logH) {
  SparseGeom s;
  s.logj = sparse_logj<LOGE>(logH);
  s.l0 = logH - s.logj;
  s.k2 = 2 << s.l0;
  return s;
}

// Shared memory of the sparse stages behind the transforms' buffers: the forward pass's R0 roots of
// unity and, per row, the J masks of active r; the inverse pass's row ranges.
template <typename CT, int LOGE>
__host__ __device__ __forceinline__ size_t sparse_smem(int logH, int rows) {
  const SparseGeom s = sparse_geom<LOGE>(logH);
  return ((size_t)sizeof(CT) << s.l0) + ((size_t)rows << s.logj) * 4 + (size_t)(rows + 1) * 4;
}

// Whether a context's rows take the sparse stages. Counting operations, a point costs 2 R0 products
// and sums where the dense radix-R0 passes cost about 0.57 J log2(R0) of them per row; the line lies
// at half of that because the operations on single points are slower than those of the dense passes, and
// for binary64, where they run on the FP64 pipe of the few SMs that hold the longest rows, at a twelfth: at a
// twentieth (a contour of 1000 wavelengths, P = 4096) the row passes gain 29 %, at an eighth (100 wavelengths,
// P = 1024) 2 to 6 %, and at a half (P = 512) they take 79 -> 109 us.
template <typename CT, int LOGE>
static bool sparse_rows(const aim_ctx* ctx) {
  constexpr long long kCost = std::is_same<CT, double2>::value ? 24 : 4;
  const int logj = sparse_logj<LOGE>(ctx->logH), l0 = ctx->logH - logj;
  return kCost * ctx->n_act <= ((long long)ctx->nrows * l0) << logj;
}

// A row of a sparse context that holds more points than this takes the dense passes: where a contour runs
// along the grid a few rows hold hundreds of points each, their sums run in one CTA, and the launch waits
// for it. The line is at the points that cost kDenseRow times the dense radix of a row: a CTA that holds
// rows of both kinds runs one after the other, so with a lower line the few dozen points of a curved
// contour's extreme rows cost more than they save. (Row passes of a square of 2000 points a side, P = 4096,
// double-float S^alpha 378 -> 182 us; 900 a side, P = 2048, N 195 -> 132 us; complex64, 400 a side, P = 1024,
// N 41 -> 24 us. A line at 8 leaves the squares of P <= 512 at 22 to 28 us instead of 18 to 27, one at 2
// takes the star contour of P = 256 from 20 to 30.) It depends on the context alone, so that results depend
// neither on the number of right-hand sides nor on the launch.
template <int LOGE>
static int sparse_row_limit(const aim_ctx* ctx) {
  constexpr int kDenseRow = 4;
  const int logj = sparse_logj<LOGE>(ctx->logH), l0 = ctx->logH - logj, limit = (kDenseRow * l0 << logj) / 4;
  return ctx->row_most > limit ? limit : INT_MAX;
}

// Forward row pass of sparse rows. The points of a row go to their places n = j + J r of the row's two
// buffers (u in the even half's, u w^n in the odd half's) and into the masks that say which r of a j
// hold one; nothing else is written, so nothing is zeroed. The first dense pass forms its inputs
//     X0_half[j R0 + k1] = sum over the active r of j of u w^(half n) W_R0^(r k1)
// from them in registers (r ascending) and goes on at Ns = R0. Every factor comes from the table, so a value
// is rounded as often as in the dense passes, and not at all where W_R0 is 1, -1 or +-i (with w^j in place of
// w^n and roots of 2 R0 in the odd half, and Horner's rule in the inverse pass, S^alpha at P = 512 was off by
// 1.83e-14 in double-float instead of 1.66e-14, N at P = 1024 by 6.99e-14 instead of 6.48e-14). (Scattering
// every point into the R0
// outputs of its j by read-modify-write of shared memory took 38 of 280 us of the double-float pass
// at 2048 points, and 13 of 33 us at 512 points, where the rows along the contour's tangents set the
// time of the whole launch.)
template <typename CT, int TPT, int LOGE>
__device__ __forceinline__ void row_fwd_sparse(const RowFwdArgs& a, int row_block, int c, bool skip, unsigned char* smraw) {
  using T2 = CT;
  constexpr int NF = TPT, LPT = 3 - TPT;
  T2* sm = reinterpret_cast<T2*>(smraw);
  const int H = 1 << a.logH, P = 1 << a.logP, tpf = H >> LOGE, HS = padded_len<LOGE>(H);
  const int per_row = LPT * tpf;
  const int g = threadIdx.x / per_row, rem = threadIdx.x - g * per_row;
  const int half = TPT == 1 ? (rem & 1) : 0, j = TPT == 1 ? (rem >> 1) : rem;
  const int row0 = row_block * a.rows_per_cta, rloc = row0 + g;
  const bool live = rloc < a.nrows && !skip;
  const T2* tw = static_cast<const T2*>(a.tw);
  int fb[NF];
#pragma unroll
  for (int f = 0; f < NF; ++f) fb[f] = (2 * g + (TPT == 1 ? half : f)) * HS;
  const SparseGeom sg = sparse_geom<LOGE>(a.logH);
  const int J = 1 << sg.logj, R0 = 1 << sg.l0;
  T2* roots = sm + 2 * a.rows_per_cta * HS;
  unsigned* masks = reinterpret_cast<unsigned*>(roots + R0);
  {
    const int p0 = live ? a.row_ptr[a.row_lo + rloc] : 0, p1 = live ? a.row_ptr[a.row_lo + rloc + 1] : 0;
    for (int i = threadIdx.x; i < R0; i += blockDim.x) roots[i] = ldro(&tw[i << (sg.logj + 1)]);
    for (int i = rem; i < J; i += per_row) masks[(g << sg.logj) + i] = 0;
    int ix = p0 + rem < p1 ? a.act_ix[p0 + rem] : 0;
    T2 w = ldro(&tw[ix]);
    const T2* uv = static_cast<const T2*>(a.u) + (size_t)c * a.n_act;
    __syncthreads();
    grid_dependency_wait();
    for (int ap = p0 + rem; ap < p1; ap += per_row) {
      if (ap != p0 + rem) {
        ix = a.act_ix[ap];
        w = ldro(&tw[ix]);
      }
      const T2 u = uv[ap];
      sm[2 * g * HS + padi<LOGE>(ix)] = u;
      sm[(2 * g + 1) * HS + padi<LOGE>(ix)] = cmul(u, w);
      atomicOr(&masks[(g << sg.logj) + (ix & (J - 1))], 1u << (ix >> sg.logj));
    }
  }
  __syncthreads();
  const unsigned* rowmask = masks + (g << sg.logj);
  auto load = [&](int f, int i) {
    const int jj = i >> sg.l0, kk = i & (R0 - 1);
    const T2* src = sm + fb[f];
    unsigned m = rowmask[jj];
    T2 acc = czero<T2>();
    bool first = true;
    while (m) {
      const int r = __ffs(m) - 1;
      m &= m - 1;
      const T2 v = cmul(src[padi<LOGE>(jj + (r << sg.logj))], roots[(r * kk) & (R0 - 1)]);
      acc = first ? v : cadd(acc, v);
      first = false;
    }
    return acc;
  };
  T2* out = static_cast<T2*>(a.inter) + (size_t)c * P * a.nrows;
  auto emit = [&](int k, const T2 (&v)[NF]) { store_row<CT, TPT>(out, a, rloc, live, half, k, v); };
  // both dense passes have twiddles here, the first of a dense row has none: every factor from the table
  if (sg.logj == LOGE) {
    last_pass_from<LOGE, false, NF, LOGE, true>(j, tpf, a.logH, sg.l0, tw, a.logP, load, emit);
  } else {
    smem_pass_from<LOGE, false, NF, LOGE, true>(sm, fb, j, tpf, a.logH, sg.l0, tw, a.logP, load);
    last_pass_from<LOGE, false, NF, LOGE, true>(j, tpf, a.logH, sg.l0 + LOGE, tw, a.logP, PlainLoad<NF, LOGE, T2>{sm, fb}, emit);
  }
}

// CTA: rows_per_cta rows of one channel; (3 - TPT) * H/E threads per row (E = 2^LOGE elements each).

// One work item of the forward row pass: rows [row_block * rows_per_cta, +rows_per_cta) of channel c.
// Every thread of the CTA calls it (it holds barriers); `smraw` is the CTA's dynamic shared memory.
// LONG: rows of more points than a.dense_from may be among the sparse ones (a variant of its own: with the
// second path behind the first the double-float passes spill more, 469 -> 487 us at P = 4096).
template <typename CT, int TPT, int LOGE, bool LONG>
__device__ __forceinline__ void row_fwd_item(const RowFwdArgs& a, int row_block, int c, unsigned char* smraw) {
  if (!LONG && a.sparse) {
    row_fwd_sparse<CT, TPT, LOGE>(a, row_block, c, false, smraw);
    return;
  }
  using T2 = CT;
  constexpr int NF = TPT, LPT = 3 - TPT;
  T2* sm = reinterpret_cast<T2*>(smraw);
  const int H = 1 << a.logH, P = 1 << a.logP, tpf = H >> LOGE, HS = padded_len<LOGE>(H);
  const int per_row = LPT * tpf;
  const int g = threadIdx.x / per_row, rem = threadIdx.x - g * per_row;
  const int half = TPT == 1 ? (rem & 1) : 0, j = TPT == 1 ? (rem >> 1) : rem;
  const int rloc = row_block * a.rows_per_cta + g;
  bool live = rloc < a.nrows;
  if (LONG && a.sparse) {
    // each row by its own count: first the CTA's sparse rows, then its dense ones
    const bool full = live && a.row_ptr[a.row_lo + rloc + 1] - a.row_ptr[a.row_lo + rloc] > a.dense_from;
    const bool any_full = __syncthreads_or(full), any_sparse = __syncthreads_or(live && !full);
    if (any_sparse) row_fwd_sparse<CT, TPT, LOGE>(a, row_block, c, full, smraw);
    if (!any_full) return;
    __syncthreads();
    live = full;
  }
  const int iy = a.row_lo + rloc;
  const T2* tw = static_cast<const T2*>(a.tw);
  const int fbA = (2 * g) * HS;
  int fb[NF];
#pragma unroll
  for (int f = 0; f < NF; ++f) fb[f] = (2 * g + (TPT == 1 ? half : f)) * HS;
  // zero the row buffer, then put the row's values into it (the row's active-point range is
  // loaded first so that its latency overlaps the zeroing). Forming u w^n here, at the active
  // points only and into a second zeroed buffer, was measured: 0.6 % faster in double-float and
  // 3 % slower in complex64, so pass 0 keeps the products.
  int a0 = 0, a1 = 0;
  if (live && !a.dense) {
    a0 = a.row_ptr[iy];
    a1 = a.row_ptr[iy + 1];
  }
  for (int i = rem; i < HS; i += per_row) sm[fbA + i] = czero<T2>();
  __syncthreads();
  grid_dependency_wait();
  if (live) {
    if (a.dense) {
      const double2* u = a.x + (size_t)c * a.m * a.m + (size_t)iy * a.m;
      for (int ix = rem; ix < a.m; ix += per_row) {
        const double2 v = u[ix];
        sm[fbA + padi<LOGE>(ix)] = cfrom<T2>(v.x, v.y);
      }
    } else {
      const T2* uv = static_cast<const T2*>(a.u) + (size_t)c * a.n_act;
      for (int ap = a0 + rem; ap < a1; ap += per_row) sm[fbA + padi<LOGE>(a.act_ix[ap])] = uv[ap];
    }
  }
  __syncthreads();
  // pass 0 (radix E, Ns = 1): the transform of a and/or of a w^n
  {
    const int lognb = a.logH - LOGE;
    T2 v[NF][1 << LOGE];
#pragma unroll
    for (int r = 0; r < (1 << LOGE); ++r) {
      const int nn = j + (r << lognb);
      const T2 x = sm[fbA + padi<LOGE>(nn)];
#pragma unroll
      for (int f = 0; f < NF; ++f) v[f][r] = (TPT == 1 ? half : f) ? cmul(x, ldro(&tw[nn])) : x;
    }
#pragma unroll
    for (int f = 0; f < NF; ++f) dft_reg<(1 << LOGE), false>(v[f]);
    __syncthreads();
#pragma unroll
    for (int f = 0; f < NF; ++f)
#pragma unroll
      for (int r = 0; r < (1 << LOGE); ++r) sm[fb[f] + padi<LOGE>((j << LOGE) + r)] = v[f][r];
    __syncthreads();
  }
  const int np = fft_npass<LOGE>(a.logH);
  smem_passes<false, NF, LOGE>(sm, fb, j, tpf, a.logH, 1, np - 1, LOGE, tw, a.logP);
  int logNs = 0;
  for (int p = 0; p < np - 1; ++p) logNs += fft_logr<LOGE>(p, a.logH);
  // last pass: X[2k + half] straight to the tiled intermediate
  T2* out = static_cast<T2*>(a.inter) + (size_t)c * P * a.nrows;
  last_pass_dispatch<false, NF, LOGE>(sm, fb, j, tpf, a.logH, logNs, tw, a.logP, [&](int k, const T2 (&v)[NF]) {
    store_row<CT, TPT>(out, a, rloc, live, half, k, v);
  });
}

template <typename CT, int TPT, int LOGE, bool WIDE, bool LONG>
__global__ void __launch_bounds__(WIDE ? kWideMax : LaunchMax<CT, TPT, LOGE>::value) k_row_fwd(RowFwdArgs a) {
  extern __shared__ __align__(16) unsigned char smraw[];
  row_fwd_item<CT, TPT, LOGE, LONG>(a, blockIdx.x, blockIdx.y, smraw);
}

// ------------------------------------------------------------------------------------
// column pass: forward DFT x spectrum x inverse DFT
// ------------------------------------------------------------------------------------
struct ColArgs {
  void* inter;
  const void* spec;
  int qcut;            // columns q with min(q, P - q) > qcut carry a zero spectrum: neither read nor written
  const void* tw;
  int logH, logP, row_lo, nrows;
  int log_cols;        // log2 of the columns of one channel per CTA
  int chan_x;          // grid order: channels along x (1) or column tiles along x (0)
};

// Recombination of the even- and odd-half inverse transforms: with TPT = 2 both are in the
// thread; with TPT = 1 the partner lane holds the other one (all lanes must call this).
template <int TPT, typename T2>
__device__ __forceinline__ T2 recombine(const T2 (&v)[TPT], int half, const T2* __restrict__ tw, int nn) {
  if constexpr (TPT == 2) {
    return cadd(v[0], cmulc(v[1], ldro(&tw[nn])));
  } else {
    const T2 other = shfl_pair(v[0]);
    return half ? other : cadd(v[0], cmulc(other, ldro(&tw[nn])));
  }
}

// CTA: 2^log_cols consecutive columns of one channel; (3 - TPT) * H/E threads per column.
// Lane order puts the columns of a tile that the CTA holds (min(2^log_cols, W) of them) in
// adjacent lanes (lane pairs when TPT = 1), so with a whole tile per CTA the global loads and
// stores of a warp are whole 32-byte sectors; with fewer columns per CTA the CTAs of the
// neighbouring columns read the rest of each sector, through L2.
// One work item of the column pass: column tile `ctile` (2^log_cols columns) of channel c.
template <typename CT, int TPT, int LOGE>
__device__ __forceinline__ void col_conv_item(const ColArgs& a, int ctile, int c, unsigned char* smraw) {
  using T2 = CT;
  constexpr int W = GridT<CT>::W, NF = TPT, LPT = 3 - TPT;
  T2* sm = reinterpret_cast<T2*>(smraw);
  const int H = 1 << a.logH, P = 1 << a.logP, tpf = H >> LOGE, HS = padded_len<LOGE>(H);
  const int cw = min(1 << a.log_cols, W);               // columns side by side in the lanes
  const int per_grp = LPT * cw * tpf;
  const int g = threadIdx.x / per_grp, rem = threadIdx.x - g * per_grp;
  const int half = TPT == 1 ? (rem & 1) : 0;
  const int r2 = TPT == 1 ? (rem >> 1) : rem;
  const int wl = r2 & (cw - 1), j = r2 / cw;
  const int colc = g * cw + wl;                         // column within the CTA
  const int qcol = (ctile << a.log_cols) + colc;   // column of the grid
  const int w = qcol & (W - 1), tile = qcol / W;
  {
    // the filtered spectrum (Eq. 10) vanishes on columns beyond the mask radius. The row passes
    // neither store nor load those, so a CTA that holds nothing else has no work (a CTA's columns
    // are an aligned run, so its smallest distance from column 0 is at one of its ends; the same
    // decision in every thread: the early return is uniform)
    const int qa = ctile << a.log_cols, qb = qa + (1 << a.log_cols) - 1;
    if (min(min(qa, P - qa), min(qb, P - qb)) > a.qcut) {
      grid_dependency_wait();   // a launch of such CTAs alone must not complete before its predecessor
      return;
    }
  }
  int fb[NF];
#pragma unroll
  for (int f = 0; f < NF; ++f) fb[f] = (2 * colc + (TPT == 1 ? half : f)) * HS;
  const T2* tw = static_cast<const T2*>(a.tw);
  T2* blk = static_cast<T2*>(a.inter) + (size_t)c * P * a.nrows + (size_t)tile * a.nrows * W;
  const int row_hi = a.row_lo + a.nrows - 1;
  grid_dependency_wait();
  // pass 0 from global: a[n] and/or a[n] w^n, n = j + (H/E)-stride
  {
    const int lognb = a.logH - LOGE;
    T2 v[NF][1 << LOGE];
#pragma unroll
    for (int r = 0; r < (1 << LOGE); ++r) {
      const int nn = j + (r << lognb);
      const T2 x = (nn >= a.row_lo && nn <= row_hi) ? blk[(nn - a.row_lo) * W + w] : czero<T2>();
#pragma unroll
      for (int f = 0; f < NF; ++f) v[f][r] = (TPT == 1 ? half : f) ? cmul(x, ldro(&tw[nn])) : x;
    }
#pragma unroll
    for (int f = 0; f < NF; ++f) {
      dft_reg<(1 << LOGE), false>(v[f]);
#pragma unroll
      for (int r = 0; r < (1 << LOGE); ++r) sm[fb[f] + padi<LOGE>((j << LOGE) + r)] = v[f][r];
    }
    __syncthreads();
  }
  const int np = fft_npass<LOGE>(a.logH);
  // remaining forward passes but the last
  smem_passes<false, NF, LOGE>(sm, fb, j, tpf, a.logH, 1, np - 1, LOGE, tw, a.logP);
  // last forward pass, product with the spectrum column, first inverse pass (same radix), in
  // registers; the inverse then runs its radix-E passes
  const int lr0 = fft_logr<LOGE>(np - 1, a.logH);
  {
    const int qq = min(qcol, P - qcol);
    const T2* col = static_cast<const T2*>(a.spec) + (size_t)qq * (H + 1);
    const int half_h = H >> 1;
    auto spec_mul = [&](int f, int k, T2 v) {
      const int odd = TPT == 1 ? half : f;
      const T2 s = odd ? ldro(&col[half_h + 1 + min(k, H - 1 - k)]) : ldro(&col[min(k, H - k)]);
      return cmul(v, s);
    };
    conv_mid_dispatch<NF, LOGE>(lr0, sm, fb, j, tpf, a.logH, tw, a.logP, spec_mul);
  }
  for (int p = 1; p < np - 1; ++p)
    smem_pass<LOGE, true, NF, LOGE>(sm, fb, j, tpf, a.logH, lr0 + LOGE * (p - 1), tw, a.logP);
  // last inverse pass (radix E, Ns = H/E) recombines y[n] = A[n] + conj(w^n) B[n] for kept rows
  last_pass<LOGE, true, NF, LOGE>(sm, fb, j, tpf, a.logH, a.logH - LOGE, tw, a.logP, [&](int nn, const T2 (&v)[NF]) {
    const T2 y = recombine<TPT>(v, half, tw, nn);
    if (!half && nn >= a.row_lo && nn <= row_hi) blk[(nn - a.row_lo) * W + w] = y;
  });
}

// The middle of the column pass of one half: last forward pass, product with the spectrum, first
// inverse pass of the same radix (conv_mid_pass, in two parts around a barrier).
template <int LOGR, int LOGE, typename T2, typename Mul>
__device__ __forceinline__ void col_mid_half(T2* buf, int j, int tpf, int logH, const T2* tw, int logP, Mul mul) {
  constexpr int R = 1 << LOGR, NB = (1 << LOGE) >> LOGR;
  const int lognb = logH - LOGR;
  T2 v[1][NB][R];
  pass_compute<LOGR, false, LOGE>(v, j, tpf, logH, lognb, tw, logP, [&](int i) { return buf[padi<LOGE>(i)]; });
#pragma unroll
  for (int t = 0; t < NB; ++t) {
    const int b = j + t * tpf;
#pragma unroll
    for (int r = 0; r < R; ++r) v[0][t][r] = mul(b + (r << lognb), v[0][t][r]);
    dft_reg<R, true>(v[0][t]);
  }
  __syncthreads();
  pass_store<LOGR, LOGE>(v, buf, j, tpf, 0);
}

// The column pass with both halves of a column in one thread group, one half after the other through
// the same code: a thread holds one transform's E elements instead of two and the code of a pass is
// there once. The odd half's input waits in its own buffer, in the slots its thread reads next, and the
// even half's result in the slots its thread has just read, so neither needs a barrier; those two extra
// trips through shared memory are what it costs. The values and their order are those of col_conv_item.
template <typename CT, int LOGE>
__device__ __forceinline__ void col_conv_halves(const ColArgs& a, int ctile, int c, unsigned char* smraw) {
  using T2 = CT;
  constexpr int W = GridT<CT>::W, E = 1 << LOGE;
  T2* sm = reinterpret_cast<T2*>(smraw);
  const int H = 1 << a.logH, P = 1 << a.logP, tpf = H >> LOGE, HS = padded_len<LOGE>(H);
  const int cw = min(1 << a.log_cols, W);               // columns side by side in the lanes
  const int per_grp = cw * tpf;
  const int g = threadIdx.x / per_grp, rem = threadIdx.x - g * per_grp;
  const int wl = rem & (cw - 1), j = rem / cw;
  const int colc = g * cw + wl;                         // column within the CTA
  const int qcol = (ctile << a.log_cols) + colc;        // column of the grid
  const int w = qcol & (W - 1), tile = qcol / W;
  {
    const int qa = ctile << a.log_cols, qb = qa + (1 << a.log_cols) - 1;
    if (min(min(qa, P - qa), min(qb, P - qb)) > a.qcut) {   // as in col_conv_item
      grid_dependency_wait();
      return;
    }
  }
  const T2* tw = static_cast<const T2*>(a.tw);
  T2* buf0 = sm + 2 * colc * HS;
  T2* blk = static_cast<T2*>(a.inter) + (size_t)c * P * a.nrows + (size_t)tile * a.nrows * W;
  const int row_hi = a.row_lo + a.nrows - 1, lognb = a.logH - LOGE;
  grid_dependency_wait();
  // pass 0 (radix E, Ns = 1) of a and of a w^n
#pragma unroll 1
  for (int f = 0; f < 2; ++f) {
    T2* buf = buf0 + f * HS;
    T2 v[1][1][E];
    if (f == 0) {
#pragma unroll
      for (int r = 0; r < E; ++r) {
        const int nn = j + (r << lognb);
        v[0][0][r] = (nn >= a.row_lo && nn <= row_hi) ? blk[(nn - a.row_lo) * W + w] : czero<T2>();
      }
#pragma unroll
      for (int r = 0; r < E; ++r) {
        const int nn = j + (r << lognb);
        buf0[HS + padi<LOGE>(nn)] = cmul(v[0][0][r], ldro(&tw[nn]));
      }
    } else {
#pragma unroll
      for (int r = 0; r < E; ++r) v[0][0][r] = buf[padi<LOGE>(j + (r << lognb))];
    }
    dft_reg<E, false>(v[0][0]);
    if (f == 1) __syncthreads();
    pass_store<LOGE, LOGE>(v, buf, j, tpf, 0);
  }
  const int np = fft_npass<LOGE>(a.logH), lr0 = fft_logr<LOGE>(np - 1, a.logH);
  // a pass of half f reads, waits for the others' reads and writes; the next pass of the same half comes
  // after the other half's wait
  auto radix_e = [&](auto inv, int logNs) {
#pragma unroll 1
    for (int f = 0; f < 2; ++f) {
      T2* buf = buf0 + f * HS;
      T2 v[1][1][E];
      pass_compute<LOGE, decltype(inv)::value, LOGE>(v, j, tpf, a.logH, logNs, tw, a.logP, [&](int i) { return buf[padi<LOGE>(i)]; });
      __syncthreads();
      pass_store<LOGE, LOGE>(v, buf, j, tpf, logNs);
    }
  };
  for (int p = 1; p < np - 1; ++p) radix_e(std::false_type{}, LOGE * p);
  {
    const T2* col = static_cast<const T2*>(a.spec) + (size_t)min(qcol, P - qcol) * (H + 1);
#pragma unroll 1
    for (int f = 0; f < 2; ++f) {
      T2* buf = buf0 + f * HS;
      const T2* cf = f ? col + (H >> 1) + 1 : col;
      auto mul = [&](int k, T2 v) { return cmul(v, ldro(&cf[min(k, H - f - k)])); };
      if (lr0 == LOGE) {
        col_mid_half<LOGE, LOGE>(buf, j, tpf, a.logH, tw, a.logP, mul);
      } else {
        switch (lr0) {
          case 3: if constexpr (LOGE > 3) col_mid_half<3, LOGE>(buf, j, tpf, a.logH, tw, a.logP, mul); break;
          case 2: col_mid_half<2, LOGE>(buf, j, tpf, a.logH, tw, a.logP, mul); break;
          default: col_mid_half<1, LOGE>(buf, j, tpf, a.logH, tw, a.logP, mul); break;
        }
      }
    }
  }
  for (int p = 1; p < np - 1; ++p) radix_e(std::true_type{}, lr0 + LOGE * (p - 1));
  // last inverse pass (radix E, Ns = H/E: outputs where the inputs were), y[n] = A[n] + conj(w^n) B[n]
#pragma unroll 1
  for (int f = 0; f < 2; ++f) {
    T2* buf = buf0 + f * HS;
    T2 v[1][1][E];
    if (f == 1) __syncthreads();   // the odd half's last stores
    pass_compute<LOGE, true, LOGE>(v, j, tpf, a.logH, lognb, tw, a.logP, [&](int i) { return buf[padi<LOGE>(i)]; });
    if (f == 0) {
#pragma unroll
      for (int r = 0; r < E; ++r) buf[padi<LOGE>(j + (r << lognb))] = v[0][0][r];
    } else {
#pragma unroll
      for (int r = 0; r < E; ++r) {
        const int nn = j + (r << lognb);
        const T2 y = cadd(buf0[padi<LOGE>(nn)], cmulc(v[0][0][r], ldro(&tw[nn])));
        if (nn >= a.row_lo && nn <= row_hi) blk[(nn - a.row_lo) * W + w] = y;
      }
    }
  }
}

template <typename CT, int TPT, int LOGE, bool WIDE = false>
__global__ void __launch_bounds__(WIDE ? kWideMax : LaunchMax<CT, TPT, LOGE>::value) k_col_conv(ColArgs a) {
  extern __shared__ __align__(16) unsigned char smraw[];
  // with many channels they run along x: the channels of one column tile run back to back and
  // share its spectrum column through L2 (64 right-hand sides: 2.82 -> 2.67 ms per launch);
  // with few, column tiles run along x (no gain measured for 3 channels)
  const int tile = a.chan_x ? blockIdx.y : blockIdx.x, channel = a.chan_x ? blockIdx.x : blockIdx.y;
  if constexpr (std::is_same<CT, dfc>::value && TPT == 2 && LOGE == 3) {
    // one half after the other where columns are short (double-float, operator N: P = 256 with seven
    // right-hand sides 34.5 -> 31.1 us, P = 1024 70 -> 65 us); both at once from P = 2048 on (285 against
    // 291 us, P = 4096 1113 against 1155 us) and in complex64 (P = 4096 263 against 288 us)
    if (a.logP <= 10) {
      col_conv_halves<CT, LOGE>(a, tile, channel, smraw);
      return;
    }
  }
  col_conv_item<CT, TPT, LOGE>(a, tile, channel, smraw);
}

// ------------------------------------------------------------------------------------
// row pass, inverse + restriction
// ------------------------------------------------------------------------------------
struct RowInvArgs {
  const void* inter;
  const void* tw;
  void* vact;          // sparse mode output: channel-major, n_act per channel
  double2* dense_out;  // dense mode output: m*m per channel
  int dense;
  int m, n_act;
  const int* row_ptr;
  const int* act_ix;
  int logH, logP, row_lo, nrows;
  double scale;
  int rows_per_cta;
  int qcut;            // as in RowFwdArgs
  int sparse, dense_from;
};

// value of another lane (xor of the lane index); all 32 lanes call it together
__device__ __forceinline__ float2 shfl_xor_c(float2 v, int off) {
  return float2{__shfl_xor_sync(0xffffffffu, v.x, off), __shfl_xor_sync(0xffffffffu, v.y, off)};
}
__device__ __forceinline__ double2 shfl_xor_c(double2 v, int off) {
  return double2{__shfl_xor_sync(0xffffffffu, v.x, off), __shfl_xor_sync(0xffffffffu, v.y, off)};
}
__device__ __forceinline__ dfc shfl_xor_c(dfc v, int off) {
  dfc r;
  r.xh = __shfl_xor_sync(0xffffffffu, v.xh, off);
  r.yh = __shfl_xor_sync(0xffffffffu, v.yh, off);
  r.xl = __shfl_xor_sync(0xffffffffu, v.xl, off);
  r.yl = __shfl_xor_sync(0xffffffffu, v.yl, off);
  return r;
}

// Lanes that share one active point of a sparse row: four terms of its sum each (with one term each
// a point costs more in the shuffle tree than in products), at least two lanes.
__device__ __forceinline__ int sparse_point_lanes(int k2) { return max(2, k2 >> 2); }

// One work item of the inverse row pass: rows [row_block * rows_per_cta, +rows_per_cta) of channel c.
// LONG as in row_fwd_item.
template <typename CT, int TPT, int LOGE, bool LONG>
__device__ __forceinline__ void row_inv_item(const RowInvArgs& a, int row_block, int c, unsigned char* smraw) {
  using T2 = CT;
  using VT = typename GridT<CT>::VT;
  constexpr int W = GridT<CT>::W, NF = TPT, LPT = 3 - TPT;
  T2* sm = reinterpret_cast<T2*>(smraw);
  const int H = 1 << a.logH, P = 1 << a.logP, tpf = H >> LOGE, HS = padded_len<LOGE>(H);
  const int per_row = LPT * tpf;
  const int g = threadIdx.x / per_row, rem = threadIdx.x - g * per_row;
  const int half = TPT == 1 ? (rem & 1) : 0, j = TPT == 1 ? (rem >> 1) : rem;
  const int rloc = row_block * a.rows_per_cta + g;
  bool live = rloc < a.nrows;
  const int iy = a.row_lo + rloc;
  const T2* tw = static_cast<const T2*>(a.tw);
  const int fbA = (2 * g) * HS;
  int fb[NF];
#pragma unroll
  for (int f = 0; f < NF; ++f) fb[f] = (2 * g + (TPT == 1 ? half : f)) * HS;
  const T2* blk = static_cast<const T2*>(a.inter) + (size_t)c * P * a.nrows;
  // sparse rows: the CTA's active points, flat over its rows, lpp lanes each; the first
  // round's point is loaded here, so that its latency overlaps the transforms
  const int lpp = sparse_point_lanes(sparse_geom<LOGE>(a.logH).k2);
  int A0 = 0, A1 = 0, ix0 = 0;
  int* rps = reinterpret_cast<int*>(sm + 2 * a.rows_per_cta * HS);
  if (a.sparse) {
    const int row0 = row_block * a.rows_per_cta;
    A0 = a.row_ptr[a.row_lo + row0];
    A1 = a.row_ptr[a.row_lo + min(row0 + a.rows_per_cta, a.nrows)];
    for (int i = threadIdx.x; i <= a.rows_per_cta; i += blockDim.x) rps[i] = a.row_ptr[a.row_lo + min(row0 + i, a.nrows)];
  }
  grid_dependency_wait();
  // pass 0 (inverse, radix E, Ns = 1) from global: Y[2k] and/or Y[2k+1]
  {
    const int lognb = a.logH - LOGE;
    T2 v[NF][1 << LOGE];
#pragma unroll
    for (int r = 0; r < (1 << LOGE); ++r) {
      // every load is issued (from the channel's first tile where there is nothing to load) before
      // any value is looked at: a branch or a select per load would expose its latency 2^LOGE times
      if constexpr (TPT == 2) {
        // Y[2k] and Y[2k + 1] are neighbours in a tile: one vector load
        const int q = 2 * (j + (r << lognb));
        const bool ok = live && min(q, P - 1 - q) <= a.qcut;
        load_pair(&blk[ok ? ((size_t)(q / W) * a.nrows + rloc) * W + (q % W) : 0], v[0][r], v[1][r]);
      } else {
        const int q = 2 * (j + (r << lognb)) + half;
        const bool ok = live && min(q, P - q) <= a.qcut;
        v[0][r] = blk[ok ? ((size_t)(q / W) * a.nrows + rloc) * W + (q % W) : 0];
      }
    }
    if (a.sparse) {   // behind the loads above: their latencies overlap
      const int ap = A0 + threadIdx.x / lpp;
      if (ap < A1) ix0 = a.act_ix[ap];
    }
    if (!live || a.qcut < (P >> 1)) {   // zero the columns beyond the mask's disc
#pragma unroll
      for (int r = 0; r < (1 << LOGE); ++r)
#pragma unroll
        for (int f = 0; f < NF; ++f) {
          const int q = 2 * (j + (r << lognb)) + (TPT == 1 ? half : f);
          if (!live || min(q, P - q) > a.qcut) v[f][r] = czero<T2>();
        }
    }
#pragma unroll
    for (int f = 0; f < NF; ++f) {
      dft_reg<(1 << LOGE), true>(v[f]);
#pragma unroll
      for (int r = 0; r < (1 << LOGE); ++r) sm[fb[f] + padi<LOGE>((j << LOGE) + r)] = v[f][r];
    }
    __syncthreads();
  }
  int p0 = 1;   // the passes done
  if (a.sparse) {
    const int logj = sparse_logj<LOGE>(a.logH), J = 1 << logj, k2 = 2 << (a.logH - logj), tpl = k2 / lpp;
    if (logj > LOGE) smem_pass<LOGE, true, NF, LOGE>(sm, fb, j, tpf, a.logH, LOGE, tw, a.logP);
    // now sub-transform k1 of half h holds its J outputs at k1 J of the half's buffer, and
    //     y[n] = sum over k' = 2 k1 + h of Z_h[k1][n mod J] W_P^{-n k'}:
    // each lane of a point sums tpl <= 4 consecutive k', and the lanes add up over a fixed shuffle tree
    // (the order depends on the transform length alone). A lane's terms have W_P^{-n t}, t < 4, from the table
    // and its sum W_P^{-n k0}, so a term is rounded twice, as in a dense row's last pass and recombination
    // (Horner's rule in W_P^{-n} takes as many products in a chain and rounds all terms so far in each; a
    // table factor for every term, 64 scattered loads a point at P = 4096, cost 10 us of 190)
    const int l = threadIdx.x & (lpp - 1), grp = threadIdx.x / lpp, ngrp = blockDim.x / lpp;
    using VP = decltype(VT::x);
    VP* out = static_cast<VP*>(a.vact) + 2 * (size_t)c * a.n_act;
    const bool mixed = LONG && a.dense_from != INT_MAX;   // rows of too many points among them (sparse_row_limit)
    const bool full = mixed && live && rps[g + 1] - rps[g] > a.dense_from;
    const int a1 = mixed && !__syncthreads_or(live && !full) ? A0 : A1;
    for (int base = A0; base < a1; base += ngrp) {
      const int ap = base + grp;
      bool valid = ap < a1;
      int lo = 0;
      if (valid) {
        int hi = a.rows_per_cta;
        while (hi - lo > 1) {
          const int mid = (lo + hi) >> 1;
          if (rps[mid] <= ap) lo = mid; else hi = mid;
        }
        valid = !mixed || rps[lo + 1] - rps[lo] <= a.dense_from;
      }
      T2 acc = czero<T2>();
      if (valid) {
        const int ix = base == A0 ? ix0 : a.act_ix[ap];
        const T2* zb = sm + (size_t)(2 * lo) * HS;
        const int jj = ix & (J - 1), k0 = l * tpl;
        T2 zt[3];   // W_P^n, its square and its cube: the same in all lanes of the point
#pragma unroll
        for (int t = 1; t < 4; ++t) zt[t - 1] = ldro(&tw[(ix * min(t, tpl - 1)) & (P - 1)]);
        const T2 w0 = ldro(&tw[(ix * k0) & (P - 1)]);
#pragma unroll
        for (int t = 0; t < 4; ++t) {
          if (t < tpl) {
            const int kk = k0 + t;
            const T2 v = zb[(kk & 1) * HS + padi<LOGE>(((kk >> 1) << logj) + jj)];
            acc = t == 0 ? v : cadd(acc, cmulc(v, zt[t - 1]));
          }
        }
        acc = cmulc(acc, w0);
      }
      for (int off = lpp >> 1; off > 0; off >>= 1) acc = cadd(acc, shfl_xor_c(acc, off));
      // lane 0 stores the real part, lane 1 the imaginary part (every lane holds the sum): the
      // conversions of the double-float types run at the FP64 rate, once per component and warp
      if (valid && l < 2) out[2 * ap + l] = cto_vt_part(acc, l, a.scale);
    }
    if (!mixed || !__syncthreads_or(full)) return;
    // rows of too many points go on with the dense passes, of which they have those so far
    live = full;
    p0 = logj / LOGE;
  }
  const int np = fft_npass<LOGE>(a.logH);
  smem_passes<true, NF, LOGE>(sm, fb, j, tpf, a.logH, p0, np - 1, LOGE * p0, tw, a.logP);
  int logNs = 0;
  for (int p = 0; p < np - 1; ++p) logNs += fft_logr<LOGE>(p, a.logH);
  const double sc = a.scale;
  if (a.dense) {
    double2* out = a.dense_out + (size_t)c * a.m * a.m + (size_t)iy * a.m;
    last_pass_dispatch<true, NF, LOGE>(sm, fb, j, tpf, a.logH, logNs, tw, a.logP, [&](int nn, const T2 (&v)[NF]) {
      const T2 y = recombine<TPT>(v, half, tw, nn);
      if (!half && live && nn < a.m) out[nn] = cto_d2(y, sc);
    });
    return;
  }
  // sparse mode: the last pass as one more shared-memory pass leaves both half-transforms in
  // natural order in their own buffers, and the recombination y = Y_even + w^-n Y_odd runs only
  // at the row's active points (tens of the H outputs)
  smem_passes<true, NF, LOGE>(sm, fb, j, tpf, a.logH, np - 1, np, logNs, tw, a.logP);
  if (live) {
    VT* out = static_cast<VT*>(a.vact) + (size_t)c * a.n_act;
    const int a1 = a.row_ptr[iy + 1];
    for (int ap = a.row_ptr[iy] + rem; ap < a1; ap += per_row) {
      const int ix = a.act_ix[ap];
      const T2 y = cadd(sm[fbA + padi<LOGE>(ix)], cmulc(sm[fbA + HS + padi<LOGE>(ix)], ldro(&tw[ix])));
      out[ap] = cto_vt(y, sc);
    }
  }
}

template <typename CT, int TPT, int LOGE, bool WIDE, bool LONG>
__global__ void __launch_bounds__(WIDE ? kWideMax : LaunchMax<CT, TPT, LOGE>::value) k_row_inv(RowInvArgs a) {
  extern __shared__ __align__(16) unsigned char smraw[];
  row_inv_item<CT, TPT, LOGE, LONG>(a, blockIdx.x, blockIdx.y, smraw);
}

// ------------------------------------------------------------------------------------
// gather + near field, Gram inverse
// ------------------------------------------------------------------------------------
struct GatherArgs {
  const void* vact;
  int n_act, n, nrhs;
  const int* ga_ptr;
  const int* ga_act;
  const double* w[kMaxProj];
  double coef[kMaxProj];
  const int* nptr;
  const int* ncol;
  const void* nval;
  const double2* x;
  double2 out_scale;
  double2* y;
};

// A group of kGatherLanes adjacent lanes per unknown i and block of up to RB right-hand sides, four
// groups to a warp: the CSR entries of row i (weights, active-point indices, near-field values and
// columns) are loaded once and used for every right-hand side of the block. For each right-hand
// side, lane g of the group sums the entries e = e0 + g, e0 + g + 8, ... in order, projection by
// projection, and the group then adds its partial sums over a fixed tree, so the result does not
// depend on the block size. The FP64 pipe (1/64 of the FP32 rate, shared by the whole SM) sets the
// cost: the tree halves the values a lane still carries at each step (at xor distance 4, a lane
// keeps the right-hand sides of its half and passes the others on) instead of adding all of them
// in every lane, 14 additions for eight right-hand sides instead of 48, and small products spread
// over many short CTAs (gather_threads) so that they use many SMs' pipes. With a complex64 grid
// (mixed precision) the projection sums run in FP32 (Acc): converting every grid value to FP64 cost
// as much as the FP64 products. The coefficient products, the near-field rows and the sums over
// projections stay in FP64.
constexpr int kGatherLanes = 8;

// Gather for the threads of virtual block `vblock` (blockDim.x threads each); all 32 lanes of every
// warp call it (the group sums are shuffles).
template <typename T2, int NP, int RB>
__device__ __forceinline__ void gather_item(const GatherArgs& a, long long vblock) {
  static_assert(RB == 1 || RB == 2 || RB == 4 || RB == 8, "a power of two of at most kGatherLanes");
  using Acc = typename std::conditional<std::is_same<T2, float2>::value, float, double>::type;
  const long long grp = (vblock * blockDim.x + threadIdx.x) / kGatherLanes;
  const int g = threadIdx.x & (kGatherLanes - 1);
  const int nblk = (a.nrhs + RB - 1) / RB;
  const bool valid = grp < (long long)a.n * nblk;
  const int rb = valid ? (int)(grp / a.n) : 0, i = valid ? (int)(grp - (long long)rb * a.n) : 0;
  const int r0 = rb * RB, nr = min(RB, a.nrhs - r0);
  double re[RB], im[RB];
#pragma unroll
  for (int q = 0; q < RB; ++q) re[q] = im[q] = 0.0;
  // the lists belong to the context: those of the lane's first kPre entries (the usual row has about
  // 45 entries, six per lane) and of the near row are loaded before the wait for the grid values
  constexpr int kPre = 6;
  const int e0 = a.ga_ptr[i], e1 = valid ? a.ga_ptr[i + 1] : e0;
  int pre_act[kPre];
#pragma unroll
  for (int u = 0; u < kPre; ++u) pre_act[u] = a.ga_act[max(min(e0 + g + u * kGatherLanes, e1 - 1), 0)];
  // one or two right-hand sides: all projections of an entry together (their loads are
  // independent); more: projection by projection, which keeps the sums in registers. The sums
  // of a projection run over the same entries in the same order either way.
  constexpr int PG = RB <= 2 ? NP : 1;
  double pre_w[PG][kPre];
#pragma unroll
  for (int p = 0; p < PG; ++p)
#pragma unroll
    for (int u = 0; u < kPre; ++u) pre_w[p][u] = a.w[p][max(min(e0 + g + u * kGatherLanes, e1 - 1), 0)];
  int n0 = 0, n1 = 0;
  if (a.nptr != nullptr && valid) {
    n0 = a.nptr[i];
    n1 = a.nptr[i + 1];
  }
  grid_dependency_wait();
  if (valid) {
    const T2* v = static_cast<const T2*>(a.vact) + (size_t)r0 * a.n_act;
#pragma unroll
    for (int p0 = 0; p0 < NP; p0 += PG) {
      Acc cr[PG][RB], ci[PG][RB];
#pragma unroll
      for (int p = 0; p < PG; ++p)
#pragma unroll
        for (int q = 0; q < RB; ++q) cr[p][q] = ci[p][q] = Acc(0);
      auto entry = [&](int act, const double (&w)[PG]) {
#pragma unroll
        for (int p = 0; p < PG; ++p) {
          const Acc ww = static_cast<Acc>(w[p]);
#pragma unroll
          for (int q = 0; q < RB; ++q) {
            if (q < nr) {
              const T2 val = v[((size_t)(p0 + p) * a.nrhs + q) * a.n_act + act];
              cr[p][q] = fma(ww, static_cast<Acc>(val.x), cr[p][q]);
              ci[p][q] = fma(ww, static_cast<Acc>(val.y), ci[p][q]);
            }
          }
        }
      };
#pragma unroll
      for (int u = 0; u < kPre; ++u) {
        const int e = e0 + g + u * kGatherLanes;
        if (e < e1) {
          double w[PG];
#pragma unroll
          for (int p = 0; p < PG; ++p) w[p] = p0 == 0 ? pre_w[p][u] : a.w[p0 + p][e];
          entry(pre_act[u], w);
        }
      }
      for (int e = e0 + g + kPre * kGatherLanes; e < e1; e += kGatherLanes) {
        double w[PG];
#pragma unroll
        for (int p = 0; p < PG; ++p) w[p] = a.w[p0 + p][e];
        entry(a.ga_act[e], w);
      }
#pragma unroll
      for (int p = 0; p < PG; ++p) {
        const double cf = a.coef[p0 + p];
#pragma unroll
        for (int q = 0; q < RB; ++q) {
          re[q] = fma(cf, (double)cr[p][q], re[q]);
          im[q] = fma(cf, (double)ci[p][q], im[q]);
        }
      }
    }
    const T2* val = static_cast<const T2*>(a.nval);
#pragma unroll 3
    for (int e = n0 + g; e < n1; e += kGatherLanes) {
      const T2 cv = val[e];
      const double cx = cv.x, cy = cv.y;
      const int col = a.ncol[e];
#pragma unroll
      for (int q = 0; q < RB; ++q) {
        if (q < nr) {
          const double2 xx = a.x[(size_t)(r0 + q) * a.n + col];
          re[q] = fma(cx, xx.x, fma(-cy, xx.y, re[q]));
          im[q] = fma(cx, xx.y, fma(cy, xx.x, im[q]));
        }
      }
    }
  }
  // the tree: cnt right-hand sides left per lane; at each step a lane with bit `off` set keeps the
  // upper half of them (every lane of the warp takes part; groups past the end carry zeros)
  int q0 = 0;
#pragma unroll
  for (int off = kGatherLanes / 2, cnt = RB; off > 0; off >>= 1) {
    if (cnt > 1) {
      cnt >>= 1;
      const bool up = (g & off) != 0;
      if (up) q0 += cnt;
#pragma unroll
      for (int q = 0; q < cnt; ++q) {
        const double sr = up ? re[q] : re[q + cnt], si = up ? im[q] : im[q + cnt];
        const double kr = up ? re[q + cnt] : re[q], ki = up ? im[q + cnt] : im[q];
        re[q] = kr + __shfl_xor_sync(0xffffffffu, sr, off);
        im[q] = ki + __shfl_xor_sync(0xffffffffu, si, off);
      }
    } else {
      re[0] += __shfl_xor_sync(0xffffffffu, re[0], off);
      im[0] += __shfl_xor_sync(0xffffffffu, im[0], off);
    }
  }
  if (valid && (g & (kGatherLanes / RB - 1)) == 0 && q0 < nr) {
    const double2 s = a.out_scale;
    a.y[(size_t)(r0 + q0) * a.n + i] =
        double2{fma(s.x, re[0], -(s.y * im[0])), fma(s.x, im[0], s.y * re[0])};
  }
}

template <typename T2, int NP, int RB>
__global__ void __launch_bounds__(256) k_gather(GatherArgs a) {
  gather_item<T2, NP, RB>(a, blockIdx.x);
}

// Threads of a gather CTA: 256, fewer while that leaves fewer CTAs than twice the SMs.
inline int gather_threads(long long threads) {
  int tpb = 256;
  while (tpb > 32 && threads / tpb < 2 * kSMs) tpb >>= 1;
  return tpb;
}

// Right-hand sides of a gather group: the power of two at or above their number, at most 8 (their sums
// fill 128 registers and spill 24 bytes in double-float), and fewer while that leaves fewer warps than four per SM: a group's FP64 work
// grows with its right-hand sides, and short products are better off on more SMs (N = 400, seven
// right-hand sides: 19 us in groups of eight).
inline int gather_rhs_block(int n, int nrhs) {
  int rb = nrhs >= 5 ? 8 : nrhs >= 3 ? 4 : nrhs;
  while (rb > 1 && (long long)n * ((nrhs + rb - 1) / rb) * kGatherLanes < 4 * kSMs * 32) rb >>= 1;
  return rb;
}

// ------------------------------------------------------------------------------------
// launch configuration
// ------------------------------------------------------------------------------------
constexpr size_t kMaxDynSmem = 227 * 1024;   // opt-in dynamic shared memory per CTA

// Lets a kernel take as much dynamic shared memory as a CTA may have. The limit belongs to the device,
// not to a context: every context sets the same value, so none lowers another's, and each remembers the
// kernels for which it has done so (two host calls per launch otherwise).
template <typename K>
static aim_status ensure_smem(aim_ctx* ctx, K kernel, size_t bytes) {
  if (bytes <= 48 * 1024) return AIM_OK;
  const void* id = reinterpret_cast<const void*>(kernel);
  for (const void* raised : ctx->smem_raised)
    if (raised == id) return AIM_OK;
  cudaFuncAttributes fa;
  AIM_CUDA_TRY(cudaFuncGetAttributes(&fa, kernel));
  AIM_CUDA_TRY(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)(kMaxDynSmem - fa.sharedSizeBytes)));
  ctx->smem_raised.push_back(id);
  return AIM_OK;
}

// tables of the context in the element type of the grid product
static const void* twiddles(const aim_ctx* c, float2*) { return c->twf; }
static const void* twiddles(const aim_ctx* c, double2*) { return c->tw; }
static const void* twiddles(const aim_ctx* c, dfc*) { return c->twdf; }
static const void* spectrum(const aim_ctx* c, bool f, float2*) { return f ? (const void*)c->specAf : c->specUf; }
static const void* spectrum(const aim_ctx* c, bool f, double2*) { return f ? (const void*)c->specA : c->specU; }
static const void* spectrum(const aim_ctx* c, bool f, dfc*) { return f ? (const void*)c->specAdf : c->specUdf; }
static const void* near_values(const NearField* nf, int which, float2*) { return nf->valf[which]; }
static const void* near_values(const NearField* nf, int which, double2*) { return nf->val[which]; }
static const void* near_values(const NearField* nf, int which, dfc*) { return nf->val[which]; }
static int precision_of(float2*) { return AIM_MIXED; }
static int precision_of(double2*) { return AIM_FP64_NATIVE; }
static int precision_of(dfc*) { return AIM_FP64; }

// Which (transforms per thread, elements per thread) pairs are compiled for an element type:
// native binary64 keeps two transforms of 16 elements per thread
template <typename CT, int TPT, int LOGE>
struct Supports {
  static constexpr bool value = std::is_same<CT, double2>::value ? (TPT == 2 && LOGE == 4) : true;
};

inline int loge_of(const Schedule& sc) { return sc.elems == 8 ? 3 : 4; }

// columns per column-pass CTA: the schedule's choice. By default one column as soon as it has 256
// threads (64 with 16 complex64 elements per thread): CTAs of one column wait at barriers of their
// own, and several fit an SM, which gains more than the half or quarter sectors they load cost
// (operator N at P = 4096: double-float 1273 -> 1163 us, complex64 329 -> 277 us; complex64 at
// P = 2048, 32 right-hand sides: 2062 -> 1925 us; but double-float there 8.26 -> 9.35 ms). Shorter
// columns: the fewest whole tiles of W columns that give at least 128 threads.
template <typename CT, int TPT, int LOGE>
static int col_cols_of(const Schedule& sc, int logH, int logP) {
  constexpr int W = GridT<CT>::W, LPT = 3 - TPT;
  if (sc.col_cols > 0) return sc.col_cols;
  const int tpf = (1 << logH) >> LOGE, ntiles = (1 << logP) / W;
  if (LPT * tpf >= (std::is_same<CT, float2>::value && LOGE == 4 ? 64 : 256)) return 1;
  int tpc = 1;
  while (tpc * LPT * W * tpf < 128 && tpc < ntiles) tpc *= 2;
  return tpc * W;
}

template <typename CT, int TPT, int LOGE>
static bool feasible_tpt(const Schedule& sc, int logH, int logP) {
  if constexpr (!Supports<CT, TPT, LOGE>::value) {
    return false;
  } else {
    constexpr int LPT = 3 - TPT;
    if (logH < LOGE + 1) return false;   // at least two passes
    const int H = 1 << logH, tpf = H >> LOGE, cols = col_cols_of<CT, TPT, LOGE>(sc, logH, logP);
    if (cols < 1 || (cols & (cols - 1)) || cols > (1 << logP)) return false;
    if (LPT * cols * tpf > LaunchMax<CT, TPT, LOGE>::value || LPT * cols * tpf < 32) return false;
    if (2 * (size_t)cols * padded_len<LOGE>(H) * sizeof(CT) > kMaxDynSmem) return false;
    if (sc.min_row_threads < 32 || sc.min_row_threads > 1024) return false;
    // row passes: one row per CTA must fit too
    if (2 * (size_t)padded_len<LOGE>(H) * sizeof(CT) > kMaxDynSmem || LPT * tpf > LaunchMax<CT, TPT, LOGE>::value)
      return false;
    return true;
  }
}

template <typename CT>
static bool feasible_for(const Schedule& s, int logH, int logP) {
  if (s.tpt != 1 && s.tpt != 2) return false;
  if (s.elems != 0 && s.elems != 8 && s.elems != 16) return false;
  if (loge_of(s) == 3)
    return s.tpt == 1 ? feasible_tpt<CT, 1, 3>(s, logH, logP) : feasible_tpt<CT, 2, 3>(s, logH, logP);
  return s.tpt == 1 ? feasible_tpt<CT, 1, 4>(s, logH, logP) : feasible_tpt<CT, 2, 4>(s, logH, logP);
}

// rows per CTA: at least min_row_threads threads (fewer when the grid has fewer rows, but
// never less than a full warp: the recombination shuffles need all 32 lanes; rows past the
// last one load zeros and store nothing), within the launch bound
template <typename CT, int TPT, int LOGE>
static int rows_per_cta(const aim_ctx* ctx, const Schedule& sc) {
  constexpr int LPT = 3 - TPT;
  const int tpf = ctx->H >> LOGE;
  int rpc = 1;
  while (((rpc * LPT * tpf < sc.min_row_threads && rpc < ctx->nrows) || rpc * LPT * tpf < 32) &&
         2 * rpc * LPT * tpf <= LaunchMax<CT, TPT, LOGE>::value)
    rpc *= 2;
  return rpc;
}

template <typename CT, int TPT, int LOGE, bool WIDE>
aim_status launch_row_fwd(aim_ctx* ctx, int channels, RowFwdArgs fa, const Schedule& sc, cudaStream_t st) {
  constexpr int LPT = 3 - TPT;
  const int tpf = ctx->H >> LOGE, rpc = rows_per_cta<CT, TPT, LOGE>(ctx, sc);
  fa.sparse = !fa.dense && sparse_rows<CT, LOGE>(ctx);
  fa.dense_from = sparse_row_limit<LOGE>(ctx);
  fa.rows_per_cta = rpc;
  const size_t smem =
      2 * (size_t)rpc * padded_len<LOGE>(ctx->H) * sizeof(CT) + (fa.sparse ? sparse_smem<CT, LOGE>(ctx->logH, rpc) : 0);
  const auto kernel = fa.sparse && fa.dense_from != INT_MAX ? k_row_fwd<CT, TPT, LOGE, WIDE, true> : k_row_fwd<CT, TPT, LOGE, WIDE, false>;
  AIM_TRY(ensure_smem(ctx, kernel, smem));
  ProfScope ps(K_ROW_FWD, st);
  return launch_chained(kernel, dim3((ctx->nrows + rpc - 1) / rpc, channels), rpc * LPT * tpf, smem, st, fa);
}

template <typename CT, int TPT, int LOGE, bool WIDE>
aim_status launch_col_conv(aim_ctx* ctx, int channels, ColArgs ca, const Schedule& sc, cudaStream_t st) {
  constexpr int LPT = 3 - TPT;
  constexpr int kChanX = 8;   // channels from which the column-pass grid runs channels along x
  const int tpf = ctx->H >> LOGE, cols = col_cols_of<CT, TPT, LOGE>(sc, ctx->logH, ctx->logP);
  ca.log_cols = 0;
  while ((1 << ca.log_cols) < cols) ++ca.log_cols;
  if (ctx->P / cols > 65535) return fail(AIM_EINVAL, "too many column tiles for one column-pass grid");
  const size_t smem = 2 * (size_t)cols * padded_len<LOGE>(ctx->H) * sizeof(CT);
  AIM_TRY(ensure_smem(ctx, k_col_conv<CT, TPT, LOGE, WIDE>, smem));
  ca.chan_x = channels >= kChanX;
  const dim3 grid = ca.chan_x ? dim3(channels, ctx->P / cols) : dim3(ctx->P / cols, channels);
  ProfScope ps(K_COL_CONV, st);
  return launch_chained(k_col_conv<CT, TPT, LOGE, WIDE>, grid, cols * LPT * tpf, smem, st, ca);
}

template <typename CT, int TPT, int LOGE, bool WIDE>
aim_status launch_row_inv(aim_ctx* ctx, int channels, RowInvArgs ia, const Schedule& sc, cudaStream_t st) {
  constexpr int LPT = 3 - TPT;
  const int tpf = ctx->H >> LOGE, rpc = rows_per_cta<CT, TPT, LOGE>(ctx, sc);
  ia.sparse = !ia.dense && sparse_rows<CT, LOGE>(ctx);
  ia.dense_from = sparse_row_limit<LOGE>(ctx);
  ia.rows_per_cta = rpc;
  const size_t smem =
      2 * (size_t)rpc * padded_len<LOGE>(ctx->H) * sizeof(CT) + (ia.sparse ? sparse_smem<CT, LOGE>(ctx->logH, rpc) : 0);
  const auto kernel = ia.sparse && ia.dense_from != INT_MAX ? k_row_inv<CT, TPT, LOGE, WIDE, true> : k_row_inv<CT, TPT, LOGE, WIDE, false>;
  AIM_TRY(ensure_smem(ctx, kernel, smem));
  ProfScope ps(K_ROW_INV, st);
  return launch_chained(kernel, dim3((ctx->nrows + rpc - 1) / rpc, channels), rpc * LPT * tpf, smem, st, ia);
}

// Transforms per thread of a pass of `lines` lines whose two-transform form has tpf threads a line.
// The results do not depend on it. A schedule that the caller or the autotuner set is obeyed; with
// the context's default, one transform per thread where two leave the SMs short of warps: one has
// half the serial work per thread, two share their twiddles. The lines lie between the sizes where
// either was faster, one against two: forward row passes of full grids in double-float 14.4 against 16.5 us at
// 12 thousand threads, 33.7 against 41.7 at 93 thousand and 51 against 57 at 125 thousand, then 174 against 160
// at 500 thousand; in complex64 9.1 against 10.3 us at 7 thousand and 18.4 against 16.4 at 62 thousand; column
// passes 14.5 against 18.5 us at 16 thousand (S^alpha, P = 512) and 26.6 against 22.5 at 65 thousand
// (P = 1024). The inverse row pass of a full grid always takes two: with one, half of the lanes recombine and
// store every output (double-float 48 against 36 us at 125 thousand threads, 14.7 against 12.6 at 12 thousand;
// complex64 26 against 20 us at 62 thousand).
template <typename CT>
static int pass_tpt(const aim_ctx* ctx, const Schedule& sc, bool rows, long long lines) {
  if (std::is_same<CT, double2>::value || !sched_is_default(ctx, precision_of((CT*)nullptr))) return sc.tpt;
  const long long threads = lines * (ctx->H >> loge_of(sc));
  const long long most = !rows ? 32 << 10 : std::is_same<CT, float2>::value ? 64 << 10 : 128 << 10;
  return threads <= most ? 1 : 2;
}

// Whether a double-float pass with one transform of 8 elements per thread runs as its wide variant.
// The plain kernels are bounded to 1024 threads, 64 registers, and spill; bounded to 512 threads they
// take 102 to 128 registers and none, but half as many threads fit an SM. So the wide ones
// run launches that fit the GPU at once: 640 and 512 threads on each of 152 SMs. (N = 733 with three
// right-hand sides 151 -> 132 us, N = 64 62 -> 57 us; a grid product of 157 thousand row-pass threads
// 108 -> 116 us, so not there.)
inline bool wide_pass(const aim_ctx* ctx, const Schedule& sc, bool rows, long long lines) {
  const int per_line = ctx->H >> 2;   // two threads for every 8 elements
  const long long threads = lines * per_line;
  if (rows) return rows_per_cta<dfc, 1, 3>(ctx, sc) * per_line <= kWideMax && threads <= kSMs * 640;
  return col_cols_of<dfc, 1, 3>(sc, ctx->logH, ctx->logP) * per_line <= kWideMax && threads <= kSMs * 512;
}

template <typename CT>
static aim_status launch_three_passes(aim_ctx* ctx, int channels, bool filtered, RowFwdArgs fa, RowInvArgs ia,
                                      void* inter, cudaStream_t st) {
  if (channels > 65535) return fail(AIM_EINVAL, "too many channels in one grid pass");
  if (ctx->H < 32) return fail(AIM_EINVAL, "embedding side P must be >= 64");
  const Schedule sc = ctx->sched[precision_of((CT*)nullptr)];
  if (!feasible_for<CT>(sc, ctx->logH, ctx->logP)) return fail(AIM_EINVAL, "launch schedule not feasible");
  const void* tw = twiddles(ctx, (CT*)nullptr);
  const int qcut = filtered ? ctx->qcut : ctx->H;
  fa.tw = tw;
  fa.logH = ctx->logH;
  fa.logP = ctx->logP;
  fa.row_lo = ctx->row_lo;
  fa.nrows = ctx->nrows;
  fa.inter = inter;
  fa.qcut = qcut;
  ColArgs ca{};
  ca.inter = inter;
  ca.spec = spectrum(ctx, filtered, (CT*)nullptr);
  ca.qcut = qcut;
  ca.tw = tw;
  ca.logH = ctx->logH;
  ca.logP = ctx->logP;
  ca.row_lo = ctx->row_lo;
  ca.nrows = ctx->nrows;
  ia.inter = inter;
  ia.tw = tw;
  ia.logH = ctx->logH;
  ia.logP = ctx->logP;
  ia.row_lo = ctx->row_lo;
  ia.nrows = ctx->nrows;
  ia.scale = 1.0 / ((double)ctx->P * (double)ctx->P);
  ia.qcut = qcut;
  const long long rows = (long long)channels * ctx->nrows, cols = (long long)channels * std::min(ctx->P, 2 * qcut + 1);
  auto run = [&](auto tpt, auto loge, int pass) -> aim_status {
    constexpr int TPT = decltype(tpt)::value, LOGE = decltype(loge)::value;
    if constexpr (std::is_same<CT, dfc>::value && TPT == 1 && LOGE == 3) {
      if (wide_pass(ctx, sc, pass != 1, pass != 1 ? rows : cols)) {
        if (pass == 0) return launch_row_fwd<CT, TPT, LOGE, true>(ctx, channels, fa, sc, st);
        if (pass == 1) return launch_col_conv<CT, TPT, LOGE, true>(ctx, channels, ca, sc, st);
        return launch_row_inv<CT, TPT, LOGE, true>(ctx, channels, ia, sc, st);
      }
    }
    if (pass == 0) return launch_row_fwd<CT, TPT, LOGE, false>(ctx, channels, fa, sc, st);
    if (pass == 1) return launch_col_conv<CT, TPT, LOGE, false>(ctx, channels, ca, sc, st);
    return launch_row_inv<CT, TPT, LOGE, false>(ctx, channels, ia, sc, st);
  };
  using I1 = std::integral_constant<int, 1>;
  using I2 = std::integral_constant<int, 2>;
  using I3 = std::integral_constant<int, 3>;
  using I4 = std::integral_constant<int, 4>;
  for (int pass = 0; pass < 3; ++pass) {
    const bool full_inverse = pass == 2 && ia.dense && sched_is_default(ctx, precision_of((CT*)nullptr));
    const int tpt = full_inverse ? 2 : pass_tpt<CT>(ctx, sc, pass != 1, pass != 1 ? rows : cols);
    aim_status s;
    if constexpr (std::is_same<CT, double2>::value) {
      s = run(I2{}, I4{}, pass);
    } else if (loge_of(sc) == 3) {
      s = tpt == 1 ? run(I1{}, I3{}, pass) : run(I2{}, I3{}, pass);
    } else {
      s = tpt == 1 ? run(I1{}, I4{}, pass) : run(I2{}, I4{}, pass);
    }
    AIM_TRY(s);
  }
  return AIM_OK;
}

inline AntArgs ant_args(const aim_ctx* ctx, const PassSpec& spec, int nrhs, const double2* x) {
  AntArgs aa{};
  aa.x = x;
  aa.n = ctx->n;
  aa.nrhs = nrhs;
  aa.n_act = ctx->n_act;
  aa.sc_ptr = ctx->prj.sc_ptr;
  aa.sc_col = ctx->prj.sc_col;
  for (int pj = 0; pj < spec.nproj; ++pj) aa.w[pj] = ctx->prj.sc_w[spec.proj[pj]];
  // u and the restricted values are never alive together: the inverse row pass starts when the
  // forward row pass, the last reader of u, is long complete
  aa.u = ctx->vact;
  return aa;
}

template <typename CT>
GatherArgs gather_args(const aim_ctx* ctx, const PassSpec& spec, int nrhs, const double2* x, double2* y) {
  GatherArgs ga{};
  ga.vact = ctx->vact;
  ga.n_act = ctx->n_act;
  ga.n = ctx->n;
  ga.nrhs = nrhs;
  ga.ga_ptr = ctx->prj.ga_ptr;
  ga.ga_act = ctx->prj.ga_act;
  for (int pj = 0; pj < spec.nproj; ++pj) {
    ga.w[pj] = ctx->prj.ga_w[spec.proj[pj]];
    ga.coef[pj] = spec.coef[pj];
  }
  if (spec.near != nullptr && spec.near->nnz > 0) {
    ga.nptr = spec.near->ptr;
    ga.ncol = spec.near->col;
    ga.nval = near_values(spec.near, spec.near_which, (CT*)nullptr);
  }
  ga.x = x;
  ga.out_scale = spec.out_scale;
  ga.y = y;
  return ga;
}

template <typename CT>
aim_status grid_pass(aim_ctx* ctx, const PassSpec& spec, int nrhs, const double2* x, double2* y,
                     cudaStream_t st) {
  using VT = typename GridT<CT>::VT;
  const int precision = precision_of((CT*)nullptr);
  const int channels = spec.nproj * nrhs;
  if (inter_bytes_needed(ctx, channels, precision) > ctx->inter_bytes ||
      (size_t)channels * ctx->n_act * sizeof(VT) > ctx->vact_bytes)
    return fail(AIM_ESTATE, "grid workspace not reserved for this many right-hand sides");

  const AntArgs aa = ant_args(ctx, spec, nrhs, x);
  {
    ProfScope ps(K_ANTERP, st);
    const long long blocks = ((long long)ctx->n_act * nrhs + kAntThreads - 1) / kAntThreads;
    AIM_TRY(launch_chained(spec.nproj == 1 ? k_anterpolate<CT, 1> : k_anterpolate<CT, 3>, dim3((unsigned)blocks),
                           kAntThreads, 0, st, aa));
  }
  RowFwdArgs fa{};
  fa.u = ctx->vact;
  fa.dense = 0;
  fa.m = ctx->m;
  fa.n_act = ctx->n_act;
  fa.row_ptr = ctx->row_ptr;
  fa.act_ix = ctx->act_ix;
  RowInvArgs ia{};
  ia.vact = ctx->vact;
  ia.dense = 0;
  ia.m = ctx->m;
  ia.n_act = ctx->n_act;
  ia.row_ptr = ctx->row_ptr;
  ia.act_ix = ctx->act_ix;
  AIM_TRY(launch_three_passes<CT>(ctx, channels, spec.filtered, fa, ia, ctx->inter, st));

  const GatherArgs ga = gather_args<CT>(ctx, spec, nrhs, x, y);
  const int rb = gather_rhs_block(ctx->n, nrhs);
  const long long threads = (long long)ctx->n * ((nrhs + rb - 1) / rb) * kGatherLanes;
  const int tpb = gather_threads(threads);
  const dim3 blocks((unsigned)((threads + tpb - 1) / tpb));
  {
    ProfScope ps(K_GATHER, st);
    auto run = [&](auto np) {
      constexpr int NP = decltype(np)::value;
      switch (rb) {
        case 1: return launch_chained(k_gather<VT, NP, 1>, blocks, tpb, 0, st, ga);
        case 2: return launch_chained(k_gather<VT, NP, 2>, blocks, tpb, 0, st, ga);
        case 4: return launch_chained(k_gather<VT, NP, 4>, blocks, tpb, 0, st, ga);
        default: return launch_chained(k_gather<VT, NP, 8>, blocks, tpb, 0, st, ga);
      }
    };
    AIM_TRY(spec.nproj == 1 ? run(std::integral_constant<int, 1>{}) : run(std::integral_constant<int, 3>{}));
  }
  return AIM_OK;
}

// ------------------------------------------------------------------------------------
// several grid passes (contexts of any size) in one persistent launch
// ------------------------------------------------------------------------------------
// One job is a whole grid pass of one context (its channels, its spectrum, its gather). The
// persistent kernel runs five phases over all jobs' work items: anterpolation, forward row pass,
// column pass, inverse row pass, gather. Every CTA takes items c, c + G, c + 2G, ... of the flattened item list
// of a phase (G = CTAs of the launch); each item fills the CTA's threads with lines (rows or
// columns) of its job, so a job with a shorter transform puts more lines into one item. A grid
// barrier separates the phases. The launch is cooperative, so all CTAs are resident and the
// barrier completes; its waits are bounded all the same: after max_spins polls a CTA records the
// failure in *err and every CTA leaves at its next barrier, and the host reports AIM_ETIMEOUT.
struct MultiJob {
  AntArgs aa;
  RowFwdArgs fa;
  ColArgs ca;
  RowInvArgs ia;
  GatherArgs ga;
  int row_items;       // row blocks per channel
  int col_items;       // column tiles per channel
  int channels;
  int tile_major;      // column items ordered tile by tile (the channels of a tile adjacent)
  int nproj;           // 1 or 3
  int gather_rb;       // right-hand sides per gather group
};

// The whole job table travels as the kernel's parameter (read-only, in the constant bank: a
// uniform load per field, as for the single-context kernels' arguments).
struct MultiArgs {
  MultiJob jobs[kMaxMultiJobs];
  int njobs;
  long long off[5][kMaxMultiJobs + 1];   // prefix sums of the items of each phase over the jobs
  unsigned* bar;                         // [arrivals, generation]: arrivals are zero between launches
  int* err;                              // 1 when a barrier wait gave up (polled by the other waits)
  int* err_host;                         // the same for the host (pinned)
  long long max_spins;
};

static_assert(sizeof(MultiArgs) <= 32000, "the job table must fit the kernel parameter space (32 KB)");

__device__ __forceinline__ bool multi_grid_barrier(const MultiArgs& m) {
  __shared__ int ok;
  __syncthreads();
  if (threadIdx.x == 0) {
    volatile unsigned* gen = m.bar + 1;
    volatile int* err = m.err;
    const unsigned g0 = *gen;
    __threadfence();
    if (atomicAdd(m.bar, 1u) == gridDim.x - 1) {
      atomicExch(m.bar, 0u);
      __threadfence();
      atomicAdd(m.bar + 1, 1u);
    } else {
      long long spins = 0;
      while (*gen == g0) {
        if (*err != 0) break;
        if (++spins > m.max_spins) {
          atomicExch(m.err, 1);
          *static_cast<volatile int*>(m.err_host) = 1;
          break;
        }
        __nanosleep(128);
      }
    }
    __threadfence();
    ok = *err == 0;
  }
  __syncthreads();
  return ok != 0;
}

// Largest CTA of the persistent kernel: 512 threads, so that five phases' code keeps 128 registers.
// (With the 1024 threads of the single-context kernels' bound the complex64 kernel spilled 1.3 KB a
// thread: eight contexts of P = 64..512 took 136 us a launch instead of 102.)
template <typename CT, int TPT, int LOGE> struct MultiMax {
  static constexpr int value = LaunchMax<CT, TPT, LOGE>::value < 512 ? LaunchMax<CT, TPT, LOGE>::value : 512;
};

template <typename CT, int TPT, int LOGE>
__global__ void __launch_bounds__(MultiMax<CT, TPT, LOGE>::value) k_grid_multi(const __grid_constant__ MultiArgs m) {
  using VT = typename GridT<CT>::VT;
  extern __shared__ __align__(16) unsigned char smraw[];
  for (int phase = 0; phase < 5; ++phase) {
    const long long total = m.off[phase][m.njobs];
    for (long long it = blockIdx.x; it < total; it += gridDim.x) {
      int jb = 0;
      while (it >= m.off[phase][jb + 1]) ++jb;   // the same job in every thread of the CTA
      const MultiJob& J = m.jobs[jb];
      const long long local = it - m.off[phase][jb];
      if (phase == 0) {
        const long long t = local * blockDim.x + threadIdx.x;
        if (J.nproj == 1) ant_item<CT, 1>(J.aa, t); else ant_item<CT, 3>(J.aa, t);
      } else if (phase == 1) {
        row_fwd_item<CT, TPT, LOGE, true>(J.fa, (int)(local % J.row_items), (int)(local / J.row_items), smraw);
      } else if (phase == 2) {
        // many channels (right-hand sides): the channels of one column tile run back to back and
        // share its spectrum column through L2, as the single-context launch orders them
        const int tile = J.tile_major ? (int)(local / J.channels) : (int)(local % J.col_items);
        const int ch = J.tile_major ? (int)(local % J.channels) : (int)(local / J.col_items);
        col_conv_item<CT, TPT, LOGE>(J.ca, tile, ch, smraw);
      } else if (phase == 3) {
        row_inv_item<CT, TPT, LOGE, true>(J.ia, (int)(local % J.row_items), (int)(local / J.row_items), smraw);
      } else {
        auto gather = [&](auto np) {
          constexpr int NP = decltype(np)::value;
          if (J.gather_rb == 1) gather_item<VT, NP, 1>(J.ga, local);
          else if (J.gather_rb == 4) gather_item<VT, NP, 4>(J.ga, local);
          else gather_item<VT, NP, 8>(J.ga, local);
        };
        if (J.nproj == 1) gather(std::integral_constant<int, 1>{}); else gather(std::integral_constant<int, 3>{});
      }
      __syncthreads();   // the next item reuses the shared memory
    }
    if (phase < 4 && !multi_grid_barrier(m)) return;
  }
}

// Runs the passes (all of element type CT, all contexts on the schedule geometry of jobs[0]: the
// same transforms per thread and elements per thread) in one persistent cooperative launch.
// scratch: 16 device bytes for the barrier and the error flag, err_host: the host's flag, as
// MultiLauncher keeps them.
template <typename CT>
aim_status grid_pass_multi(const MultiPassSpec* passes, int count, unsigned* scratch, int* err_host, cudaStream_t st);

// Threads per CTA of a multi launch whose longest transform has half-length H: two lines of it and
// at least a whole 32-byte column tile of it (W columns), at least a warp, within the launch bound.
template <typename CT, int TPT, int LOGE>
static int multi_cta_threads(int H) {
  constexpr int LPT = 3 - TPT, W = GridT<CT>::W;
  constexpr int Lmax = MultiMax<CT, TPT, LOGE>::value;
  int B = 32;
  while (B < std::max(2, W) * LPT * (H >> LOGE) && B < Lmax) B *= 2;
  return B;
}

// Whether a context with half-length H can share a launch of B threads per CTA: a CTA takes
// B / (threads per line) of its lines, a power of two of at least one and at most its P columns.
template <typename CT, int TPT, int LOGE>
static bool multi_fits(int B, int H) {
  constexpr int LPT = 3 - TPT;
  const int per_line = LPT * (H >> LOGE);
  return per_line >= 1 && B >= per_line && B / per_line <= 2 * H;
}

// CTAs of a cooperative kernel that fit the device at once; the context remembers the shapes it has
// asked for.
template <typename K>
static aim_status resident_ctas(aim_ctx* ctx, K kernel, int threads, size_t smem, int* slots) {
  const void* id = reinterpret_cast<const void*>(kernel);
  for (const auto& s : ctx->coop_slots)
    if (s.kernel == id && s.threads == threads && s.smem == smem) {
      *slots = s.slots;
      return AIM_OK;
    }
  int sms = 0, per_sm = 0, coop = 0;
  AIM_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, ctx->device));
  AIM_CUDA_TRY(cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, ctx->device));
  if (!coop) return fail(AIM_ECUDA, "device does not support cooperative launches");
  AIM_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, smem));
  if (per_sm < 1) return fail(AIM_EINVAL, "multi-context kernel does not fit an SM");
  *slots = sms * per_sm;
  if (ctx->coop_slots.size() >= 64) ctx->coop_slots.clear();
  ctx->coop_slots.push_back({id, threads, smem, *slots});
  return AIM_OK;
}

template <typename CT, int TPT, int LOGE>
static aim_status launch_multi(const MultiPassSpec* passes, int count, unsigned* scratch, int* err_host, cudaStream_t st) {
  using T2 = CT;
  using VT = typename GridT<CT>::VT;
  constexpr int LPT = 3 - TPT;
  int maxH = 1;
  for (int i = 0; i < count; ++i) maxH = std::max(maxH, passes[i].ctx->H);
  const int B = multi_cta_threads<CT, TPT, LOGE>(maxH);
  if (B < LPT * (maxH >> LOGE)) return fail(AIM_EINVAL, "transform too long for the multi-context launch");
  static thread_local MultiArgs m;   // 19 KB: kept off the stack
  m = MultiArgs{};
  m.njobs = count;
  m.bar = scratch;
  m.err = reinterpret_cast<int*>(scratch + 2);
  m.err_host = err_host;
  m.max_spins = 20000000;   // ~2.5 s of 128 ns polls
  size_t smem = 0;
  for (int i = 0; i < count; ++i) {
    const MultiPassSpec& ps = passes[i];
    aim_ctx* ctx = ps.ctx;
    const PassSpec& spec = ps.spec;
    const int H = ctx->H, P = ctx->P, tpf = H >> LOGE, HS = padded_len<LOGE>(H);
    const int lines = B / (LPT * tpf);
    if (!multi_fits<CT, TPT, LOGE>(B, H) || lines > P || (lines & (lines - 1)))
      return fail(AIM_EINVAL, "contexts of too different sizes for one multi-context launch");
    const int channels = spec.nproj * ps.nrhs;
    const int precision = precision_of((CT*)nullptr);
    if (inter_bytes_needed(ctx, channels, precision) > ctx->inter_bytes ||
        (size_t)channels * ctx->n_act * sizeof(VT) > ctx->vact_bytes)
      return fail(AIM_ESTATE, "grid workspace not reserved for this many right-hand sides");
    const int sparse = sparse_rows<CT, LOGE>(ctx), qcut = spec.filtered ? ctx->qcut : ctx->H;
    smem = std::max(smem, 2 * (size_t)lines * HS * sizeof(T2) + (sparse ? sparse_smem<CT, LOGE>(ctx->logH, lines) : 0));
    MultiJob& J = m.jobs[i];
    const void* tw = twiddles(ctx, (CT*)nullptr);
    J.aa = ant_args(ctx, spec, ps.nrhs, ps.x);
    J.nproj = spec.nproj;
    RowFwdArgs& fa = J.fa;
    fa.u = ctx->vact;
    fa.dense = 0;
    fa.m = ctx->m;
    fa.n_act = ctx->n_act;
    fa.row_ptr = ctx->row_ptr;
    fa.act_ix = ctx->act_ix;
    fa.inter = ctx->inter;
    fa.tw = tw;
    fa.logH = ctx->logH;
    fa.logP = ctx->logP;
    fa.row_lo = ctx->row_lo;
    fa.nrows = ctx->nrows;
    fa.rows_per_cta = lines;
    fa.qcut = qcut;
    fa.sparse = sparse;
    fa.dense_from = sparse_row_limit<LOGE>(ctx);
    ColArgs& ca = J.ca;
    ca.inter = ctx->inter;
    ca.spec = spectrum(ctx, spec.filtered, (CT*)nullptr);
    ca.qcut = qcut;
    ca.tw = tw;
    ca.logH = ctx->logH;
    ca.logP = ctx->logP;
    ca.row_lo = ctx->row_lo;
    ca.nrows = ctx->nrows;
    int lc = 0;
    while ((1 << lc) < lines) ++lc;
    ca.log_cols = lc;
    ca.chan_x = 0;
    RowInvArgs& ia = J.ia;
    ia.inter = ctx->inter;
    ia.tw = tw;
    ia.vact = ctx->vact;
    ia.dense = 0;
    ia.m = ctx->m;
    ia.n_act = ctx->n_act;
    ia.row_ptr = ctx->row_ptr;
    ia.act_ix = ctx->act_ix;
    ia.logH = ctx->logH;
    ia.logP = ctx->logP;
    ia.row_lo = ctx->row_lo;
    ia.nrows = ctx->nrows;
    ia.scale = 1.0 / ((double)P * (double)P);
    ia.rows_per_cta = lines;
    ia.qcut = qcut;
    ia.sparse = sparse;
    ia.dense_from = fa.dense_from;
    J.ga = gather_args<CT>(ctx, spec, ps.nrhs, ps.x, ps.y);
    J.gather_rb = ps.nrhs == 1 ? 1 : ps.nrhs <= 4 ? 4 : 8;
    J.row_items = (ctx->nrows + lines - 1) / lines;
    J.col_items = P / lines;
    J.channels = channels;
    J.tile_major = channels >= 8;
    const long long groups = (long long)ctx->n * ((ps.nrhs + J.gather_rb - 1) / J.gather_rb);
    const long long gblocks = (groups * kGatherLanes + B - 1) / B;
    m.off[0][i + 1] = m.off[0][i] + ((long long)ctx->n_act * ps.nrhs + B - 1) / B;
    m.off[1][i + 1] = m.off[1][i] + (long long)J.row_items * channels;
    m.off[2][i + 1] = m.off[2][i] + (long long)J.col_items * channels;
    m.off[3][i + 1] = m.off[3][i] + (long long)J.row_items * channels;
    m.off[4][i + 1] = m.off[4][i] + gblocks;
  }
  if (smem > kMaxDynSmem) return fail(AIM_EINVAL, "multi-context launch needs too much shared memory");
  auto kernel = k_grid_multi<CT, TPT, LOGE>;
  AIM_TRY(ensure_smem(passes[0].ctx, kernel, smem));
  int slots = 0;
  AIM_TRY(resident_ctas(passes[0].ctx, kernel, B, smem, &slots));
  long long most = 0;
  for (int ph = 0; ph < 5; ++ph) most = std::max(most, m.off[ph][count]);
  const int grid = (int)std::max(1LL, std::min<long long>(slots, most));
  {
    // one launch: the three grid passes and the gathers of every job
    ProfScope ps(K_MULTI, st);
    void* params[] = {&m};
    AIM_CUDA_TRY(cudaLaunchCooperativeKernel((const void*)kernel, dim3(grid), dim3(B), params, smem, st));
  }
  return AIM_OK;
}

// Splits the passes into the fewest launches whose contexts can share one CTA size (longest
// transforms first; a context too short for the CTA size of a longer one goes to a later launch).
template <typename CT, int TPT, int LOGE>
aim_status launch_multi_groups(const MultiPassSpec* passes, int count, unsigned* scratch, int* err_host, cudaStream_t st) {
  std::vector<int> left(count);
  for (int i = 0; i < count; ++i) left[i] = i;
  std::stable_sort(left.begin(), left.end(), [&](int a, int b) { return passes[a].ctx->H > passes[b].ctx->H; });
  std::vector<MultiPassSpec> group;
  while (!left.empty()) {
    const int B = multi_cta_threads<CT, TPT, LOGE>(passes[left[0]].ctx->H);
    group.clear();
    std::vector<int> rest;
    for (int i : left) {
      if (multi_fits<CT, TPT, LOGE>(B, passes[i].ctx->H)) group.push_back(passes[i]);
      else rest.push_back(i);
    }
    AIM_TRY((launch_multi<CT, TPT, LOGE>(group.data(), (int)group.size(), scratch, err_host, st)));
    left.swap(rest);
  }
  return AIM_OK;
}

template <typename CT>
aim_status grid_pass_multi(const MultiPassSpec* passes, int count, unsigned* scratch, int* err_host, cudaStream_t st) {
  if (count < 1 || count > kMaxMultiJobs) return fail(AIM_EINVAL, "1 to 32 passes per multi-context launch");
  const int p = precision_of((CT*)nullptr);
  // Contexts may share a call when there is one pass geometry that all of them stand for; each runs with
  // its own elements per thread (so that its results are those of a launch of its own).
  const Schedule& sc = passes[0].ctx->sched[p];
  unsigned elems = 3;
  for (int i = 0; i < count; ++i) {
    elems &= multi_elems(passes[i].ctx, p);
    if (passes[i].ctx->sched[p].tpt != sc.tpt || elems == 0)
      return fail(AIM_EINVAL, "contexts of one multi-context launch must share the pass geometry of their schedule");
  }
  if constexpr (std::is_same<CT, double2>::value) {
    AIM_TRY((launch_multi_groups<CT, 2, 4>(passes, count, scratch, err_host, st)));
  } else {
    std::vector<MultiPassSpec> of[2];
    for (int i = 0; i < count; ++i) of[loge_of(passes[i].ctx->sched[p]) - 3].push_back(passes[i]);
    if (!of[0].empty())
      AIM_TRY((sc.tpt == 1 ? launch_multi_groups<CT, 1, 3>(of[0].data(), (int)of[0].size(), scratch, err_host, st)
                           : launch_multi_groups<CT, 2, 3>(of[0].data(), (int)of[0].size(), scratch, err_host, st)));
    if (!of[1].empty())
      AIM_TRY((sc.tpt == 1 ? launch_multi_groups<CT, 1, 4>(of[1].data(), (int)of[1].size(), scratch, err_host, st)
                           : launch_multi_groups<CT, 2, 4>(of[1].data(), (int)of[1].size(), scratch, err_host, st)));
  }
  return AIM_OK;
}


template <typename CT>
aim_status grid_product_dense(aim_ctx* ctx, bool filtered, int nrhs, const double2* u, double2* v, void* inter,
                              size_t inter_bytes, cudaStream_t st) {
  const int precision = precision_of((CT*)nullptr);
  if (inter == nullptr || inter_bytes_needed(ctx, nrhs, precision) > inter_bytes)
    return fail(AIM_ESTATE, "grid workspace not reserved for this many grids");
  AIM_CUDA_TRY(cudaMemsetAsync(v, 0, (size_t)nrhs * ctx->m * ctx->m * sizeof(double2), st));
  RowFwdArgs fa{};
  fa.x = u;
  fa.dense = 1;
  fa.m = ctx->m;
  RowInvArgs ia{};
  ia.dense = 1;
  ia.dense_out = v;
  ia.m = ctx->m;
  ia.n_act = ctx->n_act;
  return launch_three_passes<CT>(ctx, nrhs, filtered, fa, ia, inter, st);
}

}  // namespace aim
