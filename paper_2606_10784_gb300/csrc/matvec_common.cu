// Grid-product helpers shared by every element type: the banded Gram inverse (G^-1 of Eq. 3),
// workspace sizing, and the feasibility of a launch schedule.
#include "matvec_kernels.cuh"

namespace aim {

// y = G^-1 x from the stored band (or the whole inverse for small n). Each output (i, r) belongs
// to a group of adjacent lanes, eight for a band and sixteen for long whole rows: lane g of the group sums
// the entries d = g, g + lanes, ... in order, and the group then adds its partial sums by xor shuffles, so the
// order of every sum is fixed whatever the number of right-hand sides. FP64 throughput sets the cost of this
// kernel on this GPU: a whole warp per output spends more FP64 operations on its shuffle tree than it gains
// (a band: twice as many as on the band itself; rows of 512 entries, 64 right-hand sides 77 us with a warp,
// 67 with sixteen lanes, 66 with eight, where one vector takes 18 us instead of 5), and a thread per
// output left the GPU idle for one vector (n threads, each a chain of cnt dependent loads and FMAs).
// Whole rows are applied whole: G^-1 decays by 0.27 per entry on a uniform mesh, but the far entries are the
// result for a vector of one nonzero, and carry what is not finite to every unknown.
struct GramArgs {
  const double* gi;    // stored rows, cnt entries each: entry d of row i belongs to column i - blo + d
  int blo, cnt, log_lanes;
  int n, nrhs;
  const double2* x;
  double2* y;
};
constexpr int kGramWideRows = 89;   // entries from which a row gets 16 lanes: eight load 88 before the wait for x

// all 32 lanes of every warp call it (the group sums are shuffles)
__device__ __forceinline__ void gram_item(const GramArgs& a, long long t) {
  const int lanes = 1 << a.log_lanes;
  const long long o = t >> a.log_lanes;
  const int g = threadIdx.x & (lanes - 1);
  const bool valid = o < (long long)a.n * a.nrhs;
  const int r = valid ? (int)(o / a.n) : 0, i = valid ? (int)(o - (long long)r * a.n) : 0;
  const double* row = a.gi + (size_t)i * a.cnt;
  // the row belongs to the context: the lane's first kPre entries (a band of 81 has at most 11 per
  // lane) are loaded before the wait for x
  constexpr int kPre = 11;
  double pre[kPre];
#pragma unroll
  for (int u = 0; u < kPre; ++u) pre[u] = row[min(g + (u << a.log_lanes), a.cnt - 1)];
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
      const int d = g + (u << a.log_lanes);
      if (d < a.cnt) entry(d, pre[u]);
    }
#pragma unroll 4
    for (int d = g + (kPre << a.log_lanes); d < a.cnt; d += lanes) entry(d, row[d]);
  }
  // every lane of the warp takes part in the shuffles (groups past the end carry zeros)
  for (int off = lanes >> 1; off > 0; off >>= 1) {
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
  const int blo = ctx->gram_band, cnt = blo * 2 + 1 <= ctx->n ? 2 * blo + 1 : ctx->n;
  return {ctx->gram_inv, blo, cnt, cnt >= kGramWideRows ? 4 : 3, ctx->n, nrhs, x, y};
}
static long long gram_threads(const GramArgs& a) { return ((long long)a.n * a.nrhs) << a.log_lanes; }

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
  const GramArgs a = gram_args(ctx, nrhs, x, y);
  const long long threads = gram_threads(a);
  const int tpb = gather_threads(threads);
  ProfScope ps(K_GRAM, st);
  return launch_chained(k_gram_inv, dim3((unsigned)((threads + tpb - 1) / tpb)), tpb, 0, st, a);
}

aim_status gram_inv_apply_multi(const GramCall* calls, int count, cudaStream_t st) {
  if (count == 0) return AIM_OK;
  if (count > kMaxMultiJobs) return fail(AIM_EINVAL, "1 to 32 contexts per multi-context launch");
  long long threads = 0;
  GramMultiArgs m{};
  m.njobs = count;
  for (int i = 0; i < count; ++i) {
    if (calls[i].ctx->gram_inv == nullptr) return fail(AIM_ESTATE, "no Gram matrix on a TM context");
    m.jobs[i] = gram_args(calls[i].ctx, calls[i].nrhs, calls[i].x, calls[i].y);
    threads += gram_threads(m.jobs[i]);
  }
  const int tpb = gather_threads(threads);
  for (int i = 0; i < count; ++i) {
    const long long blocks = (gram_threads(m.jobs[i]) + tpb - 1) / tpb;
    if (m.first[i] + blocks > 0x7fffffffLL) return fail(AIM_EINVAL, "too many right-hand sides in one multi-context call");
    m.first[i + 1] = m.first[i] + (int)blocks;
  }
  ProfScope ps(K_GRAM, st);
  return launch_chained(k_gram_inv_multi, dim3((unsigned)m.first[count]), tpb, 0, st, m);
}

}  // namespace aim
