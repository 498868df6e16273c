// Grid-product helpers shared by every element type: the banded Gram inverse (G^-1 of Eq. 3),
// workspace sizing, and the feasibility of a launch schedule.
#include <cmath>

#include "matvec_kernels.cuh"

namespace aim {

// y = G^-1 x from the stored band (or the dense inverse for small n). Each output (i, r) belongs
// to a group of kGramLanes adjacent lanes: lane g of the group sums the entries d = g, g + 8, ...
// in order, and the group then adds its partial sums by xor shuffles, so the order of every sum
// is fixed whatever the number of right-hand sides. FP64 throughput sets the cost of this kernel
// on this GPU: a whole warp per output spent twice as many FP64 operations on its shuffle tree
// as on the band itself, and a thread per output left the GPU idle for one vector (n threads,
// each a chain of cnt dependent loads and FMAs).
constexpr int kGramLanes = 8;

struct GramArgs {
  const double* gi;    // stored rows, `stride` entries each: entry d of row i belongs to column i - blo + d
  int stride, blo, d0, cnt;   // the entries applied: d0 <= d < d0 + cnt
  int n, nrhs;
  const double2* x;
  double2* y;
};

// all 32 lanes of every warp call it (the group sums are shuffles)
__device__ __forceinline__ void gram_item(const GramArgs& a, long long t) {
  const long long o = t / kGramLanes;
  const int g = threadIdx.x & (kGramLanes - 1);
  const bool valid = o < (long long)a.n * a.nrhs;
  const int r = valid ? (int)(o / a.n) : 0, i = valid ? (int)(o - (long long)r * a.n) : 0;
  const double* row = a.gi + (size_t)i * a.stride;
  // the row belongs to the context: the lane's first kPre entries (a band of 81 has at most 11 per
  // lane) are loaded before the wait for x
  constexpr int kPre = 11;
  double pre[kPre];
#pragma unroll
  for (int u = 0; u < kPre; ++u) pre[u] = row[min(a.d0 + g + u * kGramLanes, a.d0 + a.cnt - 1)];
  grid_dependency_wait();
  double re = 0.0, im = 0.0;
  if (valid) {
    const double2* xv = a.x + (size_t)r * a.n;
    auto entry = [&](int d, double gv) {
      int j = i - a.blo + d;
      if (j < 0) j += a.n;
      if (j >= a.n) j -= a.n;
      const double2 xx = xv[j];
      re = fma(gv, xx.x, re);
      im = fma(gv, xx.y, im);
    };
#pragma unroll
    for (int u = 0; u < kPre; ++u) {
      const int d = a.d0 + g + u * kGramLanes;
      if (d < a.d0 + a.cnt) entry(d, pre[u]);
    }
#pragma unroll 4
    for (int d = a.d0 + g + kPre * kGramLanes; d < a.d0 + a.cnt; d += kGramLanes) entry(d, row[d]);
  }
  // every lane of the warp takes part in the shuffles (groups past the end carry zeros)
#pragma unroll
  for (int off = kGramLanes / 2; off > 0; off >>= 1) {
    re += __shfl_xor_sync(0xffffffffu, re, off);
    im += __shfl_xor_sync(0xffffffffu, im, off);
  }
  if (valid && g == 0) a.y[o] = double2{re, im};
}

__global__ void __launch_bounds__(256) k_gram_inv(GramArgs a) {
  gram_item(a, (long long)blockIdx.x * blockDim.x + threadIdx.x);
}

// Several contexts in one launch: the CTAs are dealt out to the jobs in order.
struct GramMultiArgs {
  GramArgs jobs[kMaxMultiJobs];
  int first[kMaxMultiJobs + 1];   // first CTA of each job
  int njobs;
};

__global__ void __launch_bounds__(256) k_gram_inv_multi(const __grid_constant__ GramMultiArgs m) {
  int jb = 0;
  while (jb + 1 < m.njobs && (int)blockIdx.x >= m.first[jb + 1]) ++jb;   // the same job in every thread of the CTA
  gram_item(m.jobs[jb], (long long)((int)blockIdx.x - m.first[jb]) * blockDim.x + threadIdx.x);
}

static GramArgs gram_args(const aim_ctx* ctx, int nrhs, const double2* x, double2* y) {
  const int blo = ctx->gram_band;
  return {ctx->gram_inv, (blo * 2 + 1 <= ctx->n) ? 2 * blo + 1 : ctx->n, blo, ctx->gram_d0, ctx->gram_cnt, ctx->n, nrhs, x, y};
}

// G^-1 decays geometrically off its diagonal (by 0.27 per entry on a uniform mesh), so most of a
// densely stored row (n <= kGramDenseMax) is far below the rounding of its sum: entries under 2^-70
// of the row's diagonal at every offset beyond the window are not applied. (n = 400: 75 of 400
// entries left; seven right-hand sides 21 -> 8 us.) A row stored as a band is applied whole.
void gram_window(aim_ctx* ctx, const double* gi) {
  const int n = ctx->n, blo = ctx->gram_band, stride = (blo * 2 + 1 <= n) ? 2 * blo + 1 : n;
  ctx->gram_d0 = 0;
  ctx->gram_cnt = stride;
  if (n > kGramDenseMax) return;
  int reach = 0;   // largest |d - blo| of an entry that counts
  for (int i = 0; i < n; ++i) {
    const double* row = gi + (size_t)i * stride;
    const double least = std::ldexp(std::fabs(row[blo]), -70);
    int e = std::max(blo, stride - 1 - blo);
    while (e > reach && !(blo - e >= 0 && !(std::fabs(row[blo - e]) < least)) &&
           !(blo + e < stride && !(std::fabs(row[blo + e]) < least)))
      --e;
    reach = std::max(reach, e);
  }
  ctx->gram_d0 = std::max(0, blo - reach);
  ctx->gram_cnt = std::min(stride, blo + reach + 1) - ctx->gram_d0;
}

size_t inter_bytes_needed(const aim_ctx* ctx, int channels, int precision) {
  const size_t el = precision == AIM_MIXED ? sizeof(float2) : sizeof(double2);   // dfc is 16 bytes too
  return (size_t)channels * ctx->P * ctx->nrows * el;
}

bool schedule_feasible(int precision, int logH, int logP, const Schedule& s) {
  switch (precision) {
    case AIM_MIXED: return feasible_for<float2>(s, logH, logP);
    case AIM_FP64: return feasible_for<dfc>(s, logH, logP);
    case AIM_FP64_NATIVE: return feasible_for<double2>(s, logH, logP);
    default: return false;
  }
}

aim_status gram_inv_apply(aim_ctx* ctx, int nrhs, const double2* x, double2* y, cudaStream_t st) {
  if (ctx->gram_inv == nullptr) return fail(AIM_ESTATE, "no Gram matrix on a TM context");
  const long long threads = (long long)ctx->n * nrhs * kGramLanes;
  const int tpb = gather_threads(threads);
  ProfScope ps(K_GRAM, st);
  return launch_chained(k_gram_inv, dim3((unsigned)((threads + tpb - 1) / tpb)), tpb, 0, st, gram_args(ctx, nrhs, x, y));
}

aim_status gram_inv_apply_multi(const GramCall* calls, int count, cudaStream_t st) {
  if (count == 0) return AIM_OK;
  if (count > kMaxMultiJobs) return fail(AIM_EINVAL, "1 to 32 contexts per multi-context launch");
  long long threads = 0;
  for (int i = 0; i < count; ++i) {
    if (calls[i].ctx->gram_inv == nullptr) return fail(AIM_ESTATE, "no Gram matrix on a TM context");
    threads += (long long)calls[i].ctx->n * calls[i].nrhs * kGramLanes;
  }
  const int tpb = gather_threads(threads);
  GramMultiArgs m{};
  m.njobs = count;
  for (int i = 0; i < count; ++i) {
    m.jobs[i] = gram_args(calls[i].ctx, calls[i].nrhs, calls[i].x, calls[i].y);
    const long long blocks = ((long long)calls[i].ctx->n * calls[i].nrhs * kGramLanes + tpb - 1) / tpb;
    if (m.first[i] + blocks > 0x7fffffffLL) return fail(AIM_EINVAL, "too many right-hand sides in one multi-context call");
    m.first[i + 1] = m.first[i] + (int)blocks;
  }
  ProfScope ps(K_GRAM, st);
  return launch_chained(k_gram_inv_multi, dim3((unsigned)m.first[count]), tpb, 0, st, m);
}

}  // namespace aim
