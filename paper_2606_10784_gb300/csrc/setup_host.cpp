// Host-side setup of the AIM operators (FP64): the parts of Secs. II-III that are sparse
// bookkeeping rather than arithmetic over the grid.
//
//   * flat segments, tangents and outward normals of the closed polygon (Sec. II);
//   * Gauss-Legendre nodes per segment and the hat values at them (Eq. 7);
//   * the grid (Sec. III-A): half side L, spacing eps = 2L/(m-1), and for every node the
//     tensor-product Lagrange stencil of s points per axis (the interpolation Lambda);
//   * the composed projections P = Lambda W Phi, stored twice: grid-point-major (for the
//     anterpolation fused into the row DFT) and unknown-major (for the interpolation gather);
//   * near pairs for the near-field correction, found by spatial hashing;
//   * G^-1 (Gram matrix of Eq. 3): dense for small N, otherwise its band (the inverse of this
//     diagonally dominant cyclic tridiagonal matrix decays geometrically off the diagonal);
//   * the FFT twiddle table exp(-2 pi i t / P).
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>

#include "aim_internal.h"

namespace aim {

void gauss_legendre01(int n, std::vector<double>* x, std::vector<double>* w) {
  // Newton iteration on P_n from the three-term recurrence (Golub & Welsch's classical
  // alternative; initial guesses cos(pi (i - 1/4) / (n + 1/2))).
  x->assign(n, 0.0);
  w->assign(n, 0.0);
  for (int i = 0; i < (n + 1) / 2; ++i) {
    double z = std::cos(M_PI * (i + 0.75) / (n + 0.5));
    double dp = 0.0;
    for (int it = 0; it < 100; ++it) {
      double p0 = 1.0, p1 = 0.0;
      for (int j = 1; j <= n; ++j) {
        const double p2 = p1;
        p1 = p0;
        p0 = ((2.0 * j - 1.0) * z * p1 - (j - 1.0) * p2) / j;
      }
      dp = n * (z * p0 - p1) / (z * z - 1.0);
      const double dz = p0 / dp;
      z -= dz;
      if (std::fabs(dz) < 1e-16) {
        // one more evaluation of the derivative at the converged root
        p0 = 1.0; p1 = 0.0;
        for (int j = 1; j <= n; ++j) {
          const double p2 = p1;
          p1 = p0;
          p0 = ((2.0 * j - 1.0) * z * p1 - (j - 1.0) * p2) / j;
        }
        dp = n * (z * p0 - p1) / (z * z - 1.0);
        break;
      }
    }
    const double wt = 2.0 / ((1.0 - z * z) * dp * dp);
    // map [-1,1] -> [0,1]; roots come in +- pairs, z > 0 here
    (*x)[i] = 0.5 * (1.0 - z);
    (*x)[n - 1 - i] = 0.5 * (1.0 + z);
    (*w)[i] = 0.5 * wt;
    (*w)[n - 1 - i] = 0.5 * wt;
  }
}

double host_grid_half_side(const double* xy, int n, int m, int s) {
  double R = 0.0;
  for (int i = 0; i < 2 * n; ++i) R = std::max(R, std::fabs(xy[i]));
  return R / (1.0 - (s + 2.0) / (m - 1.0));
}

// Lagrange weights of s points per axis at fractional grid coordinate xi.
static inline int lagrange(double xi, int s, double* w) {
  const int base = (s % 2 == 0) ? (int)std::floor(xi) - s / 2 + 1 : (int)std::floor(xi + 0.5) - (s - 1) / 2;
  const double t = xi - base;
  for (int a = 0; a < s; ++a) {
    double num = 1.0, den = 1.0;
    for (int b = 0; b < s; ++b) {
      if (b == a) continue;
      num *= (t - b);
      den *= (double)(a - b);
    }
    w[a] = num / den;
  }
  return base;
}

static double pt_seg_dist(double px, double py, double ax, double ay, double bx, double by) {
  const double ex = bx - ax, ey = by - ay;
  double t = ((px - ax) * ex + (py - ay) * ey) / (ex * ex + ey * ey);
  t = std::min(1.0, std::max(0.0, t));
  return std::hypot(px - (ax + t * ex), py - (ay + t * ey));
}

static double pt_seg_dist2(double px, double py, double ax, double ay, double bx, double by) {
  const double ex = bx - ax, ey = by - ay;
  double t = ((px - ax) * ex + (py - ay) * ey) / (ex * ex + ey * ey);
  t = std::min(1.0, std::max(0.0, t));
  const double dx = px - (ax + t * ex), dy = py - (ay + t * ey);
  return dx * dx + dy * dy;
}

static double seg_seg_dist(const double* p0, const double* p1, const double* q0, const double* q1) {
  return std::min(std::min(pt_seg_dist(p0[0], p0[1], q0[0], q0[1], q1[0], q1[1]),
                           pt_seg_dist(p1[0], p1[1], q0[0], q0[1], q1[0], q1[1])),
                  std::min(pt_seg_dist(q0[0], q0[1], p0[0], p0[1], p1[0], p1[1]),
                           pt_seg_dist(q1[0], q1[1], p0[0], p0[1], p1[0], p1[1])));
}

// Whether two segments come within rad: decided by squares (no square root) unless the distance is
// within rounding of rad.
static bool seg_seg_within(const double* p0, const double* p1, const double* q0, const double* q1, double rad) {
  const double d2 = std::min(std::min(pt_seg_dist2(p0[0], p0[1], q0[0], q0[1], q1[0], q1[1]),
                                      pt_seg_dist2(p1[0], p1[1], q0[0], q0[1], q1[0], q1[1])),
                             std::min(pt_seg_dist2(q0[0], q0[1], p0[0], p0[1], p1[0], p1[1]),
                                      pt_seg_dist2(q1[0], q1[1], p0[0], p0[1], p1[0], p1[1])));
  const double r2 = rad * rad;
  if (d2 < r2 * (1.0 - 1e-12)) return true;
  if (d2 > r2 * (1.0 + 1e-12)) return false;
  return seg_seg_dist(p0, p1, q0, q1) <= rad;
}

namespace {
// Stencil entries of the unknowns of one side, unknown-major: grid indices iy*m + ix (iy major) and
// nval weights each.
struct SideList {
  std::vector<int> ptr{0}, g;
  std::vector<double> w;
  int nval = 1;
};

// The stencils of a set of quadrature points, computed once: start indices and weights per axis.
struct Stencils {
  int s;
  std::vector<int> bx, by;
  std::vector<double> wx, wy;
  Stencils(int s_, size_t count) : s(s_), bx(count), by(count), wx(count * s_), wy(count * s_) {}
};

// Accumulates the stencils of a set of points into a dense local box, then emits the
// nonzero box entries in grid order (iy major, ix minor).
template <int nval>
struct BoxAccumulator {
  int s, m;
  int x0 = 0, y0 = 0, nx = 0, ny = 0;
  std::vector<double> box;   // ny * nx * nval
  std::vector<char> hit;
  void begin(int bx0, int by0, int bx1, int by1) {
    x0 = bx0; y0 = by0; nx = bx1 - bx0 + 1; ny = by1 - by0 + 1;
    box.assign((size_t)nx * ny * nval, 0.0);
    hit.assign((size_t)nx * ny, 0);
  }
  void add(int bx, int by, const double* wx, const double* wy, const double* val) {
    for (int b = 0; b < s; ++b) {
      const size_t cell = (size_t)(by + b - y0) * nx + (bx - x0);
      double* o = &box[cell * nval];
      for (int a = 0; a < s; ++a) {
        hit[cell + a] = 1;
        const double ww = wy[b] * wx[a];
        for (int q = 0; q < nval; ++q) o[a * nval + q] += ww * val[q];
      }
    }
  }
  void emit(SideList* out) {
    for (int yy = 0; yy < ny; ++yy)
      for (int xx = 0; xx < nx; ++xx) {
        const size_t cell = (size_t)yy * nx + xx;
        if (!hit[cell]) continue;
        out->g.push_back((y0 + yy) * m + (x0 + xx));
        for (int q = 0; q < nval; ++q) out->w.push_back(box[cell * nval + q]);
      }
    out->ptr.push_back((int)out->g.size());
  }
};

// Ranks of the active grid points: one bit per point and a running count per 64 of them.
struct ActiveSet {
  std::vector<uint64_t> bits;
  std::vector<int> before;
  explicit ActiveSet(size_t points) : bits((points + 63) / 64, 0), before((points + 63) / 64) {}
  void add(int g) { bits[(size_t)g >> 6] |= (uint64_t)1 << (g & 63); }
  int rank(int g) const {
    return before[(size_t)g >> 6] + __builtin_popcountll(bits[(size_t)g >> 6] & (((uint64_t)1 << (g & 63)) - 1));
  }
};
}  // namespace

aim_status host_setup(aim_ctx* ctx, HostSetup* hs) {
  const int n = ctx->n, m = ctx->m, s = ctx->s, p = ctx->p;
  const double* xy = ctx->xy.data();
  const double L = ctx->L, eps = ctx->eps;
  const bool te = ctx->form == AIM_TE_P1_GALERKIN;

  // ---- segments
  hs->dx.resize(n); hs->dy.resize(n); hs->h.resize(n);
  hs->tx.resize(n); hs->ty.resize(n); hs->nx.resize(n); hs->ny.resize(n);
  double hmax = 0.0;
  for (int e = 0; e < n; ++e) {
    const int f = (e + 1) % n;
    hs->dx[e] = xy[2 * f] - xy[2 * e];
    hs->dy[e] = xy[2 * f + 1] - xy[2 * e + 1];
    hs->h[e] = std::hypot(hs->dx[e], hs->dy[e]);
    if (!(hs->h[e] > 0.0)) return fail(AIM_EINVAL, "degenerate (zero-length) segment");
    hs->tx[e] = hs->dx[e] / hs->h[e];
    hs->ty[e] = hs->dy[e] / hs->h[e];
    hs->nx[e] = hs->ty[e];
    hs->ny[e] = -hs->tx[e];
    hmax = std::max(hmax, hs->h[e]);
  }
  gauss_legendre01(p, &hs->gx, &hs->gw);

  // ---- twiddles
  const int P = ctx->P;
  hs->tw.resize(2 * (size_t)P);
  for (int t = 0; t < P; ++t) {
    const double ang = 2.0 * M_PI * (double)t / (double)P;
    hs->tw[2 * t] = std::cos(ang);
    hs->tw[2 * t + 1] = -std::sin(ang);
  }

  // ---- projections: per unknown, the accumulated stencils of its quadrature nodes. The stencils of
  // all segments' nodes are computed once (a TE node serves two hats); TM adds the midpoints.
  auto stencil_of = [&](double x, double y, Stencils* st, size_t k) {
    st->bx[k] = lagrange((x + L) / eps, s, &st->wx[k * s]);
    st->by[k] = lagrange((y + L) / eps, s, &st->wy[k * s]);
    return st->bx[k] >= 0 && st->by[k] >= 0 && st->bx[k] + s - 1 <= m - 1 && st->by[k] + s - 1 <= m - 1;
  };
  Stencils node_st(s, (size_t)n * p);
  for (int e = 0; e < n; ++e)
    for (int u = 0; u < p; ++u)
      if (!stencil_of(xy[2 * e] + hs->gx[u] * hs->dx[e], xy[2 * e + 1] + hs->gx[u] * hs->dy[e], &node_st, (size_t)e * p + u))
        return fail(AIM_EINVAL, "contour too close to the grid edge for this stencil (increase L)");

  // unknown-major lists: source side (scatter) and test side (gather)
  SideList src, tst;
  hs->nproj = te ? 4 : 1;
  src.nval = hs->nproj;
  auto sources = [&](auto& box) {
    for (int i = 0; i < n; ++i) {
      // TE hat i: segment i (falling piece, phi = 1 - xi) and segment i-1 (rising piece, phi = xi);
      // TM pulse i: segment i
      const int segs[2] = {i, (i + n - 1) % n}, npc = te ? 2 : 1;
      int x0 = 1 << 30, y0 = 1 << 30, x1 = -1, y1 = -1;
      for (int pc = 0; pc < npc; ++pc)
        for (int u = 0; u < p; ++u) {
          const size_t k = (size_t)segs[pc] * p + u;
          x0 = std::min(x0, node_st.bx[k]); y0 = std::min(y0, node_st.by[k]);
          x1 = std::max(x1, node_st.bx[k] + s - 1); y1 = std::max(y1, node_st.by[k] + s - 1);
        }
      box.begin(x0, y0, x1, y1);
      for (int pc = 0; pc < npc; ++pc) {
        const int e = segs[pc];
        for (int u = 0; u < p; ++u) {
          const size_t k = (size_t)e * p + u;
          const double wq = hs->gw[u] * hs->h[e];
          const double phi = pc == 0 ? 1.0 - hs->gx[u] : hs->gx[u];
          const double dphi = (pc == 0 ? -1.0 : 1.0) / hs->h[e];
          const double te_val[4] = {wq * phi, wq * dphi, wq * phi * hs->nx[e], wq * phi * hs->ny[e]};
          box.add(node_st.bx[k], node_st.by[k], &node_st.wx[k * s], &node_st.wy[k * s], te ? te_val : &wq);
        }
      }
      box.emit(&src);
    }
  };
  BoxAccumulator<4> box4{s, m};
  BoxAccumulator<1> box{s, m};
  if (te) sources(box4);
  else sources(box);
  if (!te) {
    Stencils mid_st(s, n);
    const double one[1] = {1.0};
    for (int j = 0; j < n; ++j) {
      // collocation at the midpoint
      if (!stencil_of(xy[2 * j] + 0.5 * hs->dx[j], xy[2 * j + 1] + 0.5 * hs->dy[j], &mid_st, j))
        return fail(AIM_EINVAL, "contour too close to the grid edge");
      box.begin(mid_st.bx[j], mid_st.by[j], mid_st.bx[j] + s - 1, mid_st.by[j] + s - 1);
      box.add(mid_st.bx[j], mid_st.by[j], &mid_st.wx[(size_t)j * s], &mid_st.wy[(size_t)j * s], one);
      box.emit(&tst);
    }
  }
  const SideList& gat = te ? src : tst;

  // ---- active grid points: union of both sides, ordered by grid index
  ActiveSet act((size_t)m * m);
  for (int g : src.g) act.add(g);
  if (!te)
    for (int g : tst.g) act.add(g);
  int n_act = 0;
  hs->row_ptr.assign(m + 1, 0);
  hs->act_ix.clear();
  hs->act_iy.clear();
  for (size_t wd = 0; wd < act.bits.size(); ++wd) {
    act.before[wd] = n_act;
    for (uint64_t b = act.bits[wd]; b != 0; b &= b - 1) {
      const int g = (int)(wd * 64) + __builtin_ctzll(b);
      ++n_act;
      hs->act_ix.push_back(g % m);
      hs->act_iy.push_back(g / m);
      hs->row_ptr[g / m + 1]++;
    }
  }
  for (int iy = 0; iy < m; ++iy) hs->row_ptr[iy + 1] += hs->row_ptr[iy];
  hs->n_act = n_act;
  hs->row_lo = hs->act_iy.front();
  hs->row_hi = hs->act_iy.back();

  // ---- gather CSR (unknown-major)
  hs->ga_ptr = gat.ptr;
  const int nga = hs->ga_ptr[n];
  hs->ga_act.resize(nga);
  for (int e = 0; e < nga; ++e) hs->ga_act[e] = act.rank(gat.g[e]);
  for (int q = 0; q < hs->nproj; ++q) {
    hs->ga_w[q].resize(nga);
    for (int e = 0; e < nga; ++e) hs->ga_w[q][e] = gat.w[(size_t)e * gat.nval + q];
  }
  // ---- scatter CSR (active-point-major), by counting sort of the source entries
  const int nsc = src.ptr[n];
  std::vector<int> src_act(nsc);
  if (te) src_act = hs->ga_act;
  else
    for (int e = 0; e < nsc; ++e) src_act[e] = act.rank(src.g[e]);
  hs->sc_ptr.assign(n_act + 1, 0);
  for (int a : src_act) hs->sc_ptr[a + 1]++;
  for (int a = 0; a < n_act; ++a) hs->sc_ptr[a + 1] += hs->sc_ptr[a];
  hs->sc_col.resize(nsc);
  for (int q = 0; q < hs->nproj; ++q) hs->sc_w[q].resize(nsc);
  {
    std::vector<int> fill(hs->sc_ptr.begin(), hs->sc_ptr.end() - 1);
    for (int j = 0; j < n; ++j)
      for (int e = src.ptr[j]; e < src.ptr[j + 1]; ++e) {
        const int o = fill[src_act[e]]++;
        hs->sc_col[o] = j;
        for (int q = 0; q < hs->nproj; ++q) hs->sc_w[q][o] = src.w[(size_t)e * src.nval + q];
      }
  }
  // source-major list for the TM near field (the TE source list equals the gather list)
  if (!te) {
    hs->sr_ptr = src.ptr;
    hs->sr_act = src_act;
    hs->sr_w = src.w;
  }

  // ---- near pairs by spatial hashing of segment midpoints
  const double rad = ctx->near_radius;
  const double cell = rad + hmax;
  double bxmin = 1e300, bymin = 1e300, bxmax = -1e300, bymax = -1e300;
  std::vector<double> mx(n), my(n);
  for (int e = 0; e < n; ++e) {
    mx[e] = xy[2 * e] + 0.5 * hs->dx[e];
    my[e] = xy[2 * e + 1] + 0.5 * hs->dy[e];
    bxmin = std::min(bxmin, mx[e]); bxmax = std::max(bxmax, mx[e]);
    bymin = std::min(bymin, my[e]); bymax = std::max(bymax, my[e]);
  }
  const int ncx = std::max(1, (int)std::floor((bxmax - bxmin) / cell) + 1);
  const int ncy = std::max(1, (int)std::floor((bymax - bymin) / cell) + 1);
  if ((double)ncx * ncy > 4.0e7) return fail(AIM_EINVAL, "near radius too small relative to the contour size");
  std::vector<int> cstart((size_t)ncx * ncy + 1, 0), cseg(n), ccell(n);
  for (int e = 0; e < n; ++e) {
    const int cx = std::min(ncx - 1, (int)std::floor((mx[e] - bxmin) / cell));
    const int cy = std::min(ncy - 1, (int)std::floor((my[e] - bymin) / cell));
    ccell[e] = cy * ncx + cx;
    cstart[ccell[e] + 1]++;
  }
  for (size_t c = 0; c < (size_t)ncx * ncy; ++c) cstart[c + 1] += cstart[c];
  {
    std::vector<int> fill(cstart.begin(), cstart.end() - 1);
    for (int e = 0; e < n; ++e) cseg[fill[ccell[e]]++] = e;
  }
  auto for_candidates = [&](double px, double py, auto&& fn) {
    const int cx = std::min(ncx - 1, std::max(0, (int)std::floor((px - bxmin) / cell)));
    const int cy = std::min(ncy - 1, std::max(0, (int)std::floor((py - bymin) / cell)));
    for (int yy = std::max(0, cy - 1); yy <= std::min(ncy - 1, cy + 1); ++yy)
      for (int xx = std::max(0, cx - 1); xx <= std::min(ncx - 1, cx + 1); ++xx) {
        const int c = yy * ncx + xx;
        for (int q = cstart[c]; q < cstart[c + 1]; ++q) fn(cseg[q]);
      }
  };

  // A pair within `rad` has midpoints within rad and the half lengths (with a margin for rounding),
  // which rules most candidates out without their distances. Segment distances are symmetric, so each
  // pair of segments is looked at once.
  auto far_apart = [&](int e, int f, double reach) {
    const double dx = mx[e] - mx[f], dy = my[e] - my[f];
    return dx * dx + dy * dy > reach * reach * (1.0 + 1e-9);
  };
  std::vector<std::vector<int>> rows(n);
  if (te) {
    std::vector<std::vector<int>> seg_near(n);
    for (int e = 0; e < n; ++e) {
      seg_near[e].push_back(e);
      const double* p0 = &xy[2 * e];
      const double* p1 = &xy[2 * ((e + 1) % n)];
      for_candidates(mx[e], my[e], [&](int f) {
        if (f <= e || far_apart(e, f, rad + 0.5 * (hs->h[e] + hs->h[f]))) return;
        const double* q0 = &xy[2 * f];
        const double* q1 = &xy[2 * ((f + 1) % n)];
        if (seg_seg_within(p0, p1, q0, q1, rad)) {
          seg_near[e].push_back(f);
          seg_near[f].push_back(e);
        }
      });
    }
    // hats i and j are near when a segment of i (i-1 or i) is near a segment of j
    for (int i = 0; i < n; ++i) {
      auto& r = rows[i];
      for (int e : {(i + n - 1) % n, i})
        for (int f : seg_near[e]) {
          r.push_back(f);
          r.push_back((f + 1) % n);
        }
    }
  } else {
    for (int i = 0; i < n; ++i) {
      for_candidates(mx[i], my[i], [&](int j) {
        if (far_apart(i, j, rad + 0.5 * hs->h[j])) return;
        const double* q0 = &xy[2 * j];
        const double* q1 = &xy[2 * ((j + 1) % n)];
        if (pt_seg_dist(mx[i], my[i], q0[0], q0[1], q1[0], q1[1]) <= rad) rows[i].push_back(j);
      });
    }
  }
  hs->near_ptr.assign(n + 1, 0);
  for (int i = 0; i < n; ++i) {
    auto& r = rows[i];
    std::sort(r.begin(), r.end());
    r.erase(std::unique(r.begin(), r.end()), r.end());
    hs->near_ptr[i + 1] = hs->near_ptr[i] + (int)r.size();
  }
  hs->near_col.resize(hs->near_ptr[n]);
  for (int i = 0; i < n; ++i) std::copy(rows[i].begin(), rows[i].end(), hs->near_col.begin() + hs->near_ptr[i]);

  // segment pairs needed by the exact near entries: (e, f) with e <= f only, since the integrals of
  // (f, e) are those of (e, f) with the two hats exchanged. Segment e needs the segments j and j - 1 of
  // every hat j near hat e or e + 1.
  hs->seg_e.clear(); hs->seg_f.clear(); hs->pair_seg_idx.clear();
  if (te) {
    std::vector<int> base(n + 1, 0), lst;
    for (int e = 0; e < n; ++e) {
      lst.clear();
      for (int i : {e, (e + 1) % n})
        for (int j : rows[i]) {
          if (j >= e) lst.push_back(j);
          const int f = (j + n - 1) % n;
          if (f >= e) lst.push_back(f);
        }
      std::sort(lst.begin(), lst.end());
      lst.erase(std::unique(lst.begin(), lst.end()), lst.end());
      hs->seg_f.insert(hs->seg_f.end(), lst.begin(), lst.end());
      hs->seg_e.insert(hs->seg_e.end(), lst.size(), e);
      base[e + 1] = (int)hs->seg_f.size();
    }
    auto pair_id = [&](int e, int f) {   // ~id: the pair (f, e), hats exchanged
      const int lo = std::min(e, f), hi = std::max(e, f);
      const int id = (int)(std::lower_bound(hs->seg_f.begin() + base[lo], hs->seg_f.begin() + base[lo + 1], hi) - hs->seg_f.begin());
      return e <= f ? id : ~id;
    };
    hs->pair_seg_idx.resize((size_t)hs->near_ptr[n] * 4);
    for (int i = 0; i < n; ++i)
      for (int q = hs->near_ptr[i]; q < hs->near_ptr[i + 1]; ++q) {
        const int j = hs->near_col[q], im = (i + n - 1) % n, jm = (j + n - 1) % n;
        int* id = &hs->pair_seg_idx[(size_t)q * 4];
        id[0] = pair_id(i, j);
        id[1] = pair_id(i, jm);
        id[2] = pair_id(im, j);
        id[3] = pair_id(im, jm);
      }
  }

  // ---- G^-1 (TE)
  if (te) {
    // cyclic tridiagonal: diag_i = (h_{i-1}+h_i)/3, G[i][i+1] = G[i+1][i] = h_i/6
    auto diag = [&](int i) { return (hs->h[(i + n - 1) % n] + hs->h[i]) / 3.0; };
    auto off = [&](int i) { return hs->h[i] / 6.0; };   // couples i and i+1
    if (n < kGramRingMin) {
      // dense inverse: Sherman-Morrison on the cyclic system, one Thomas solve per column
      const int blo = n / 2;
      hs->gram_band = blo;
      hs->gram_inv.assign((size_t)n * n, 0.0);
      std::vector<double> a(n), b(n), c(n);
      for (int i = 0; i < n; ++i) {
        b[i] = diag(i);
        a[i] = off((i + n - 1) % n);   // G[i][i-1]
        c[i] = off(i);                 // G[i][i+1]
      }
      const double alpha = c[n - 1], beta = a[0];   // G[n-1][0], G[0][n-1]
      const double gamma = -b[0];
      std::vector<double> bb(b);
      bb[0] = b[0] - gamma;
      bb[n - 1] = b[n - 1] - alpha * beta / gamma;
      // the elimination's factors, shared by all columns; a column's right-hand side is zero before `from`
      std::vector<double> cp(n), inv(n), dp(n);
      for (int i = 0; i < n; ++i) {
        inv[i] = 1.0 / (i == 0 ? bb[0] : bb[i] - a[i] * cp[i - 1]);
        cp[i] = c[i] * inv[i];
      }
      auto thomas = [&](const std::vector<double>& rhs, int from, std::vector<double>* x) {
        std::fill(dp.begin(), dp.begin() + from, 0.0);
        dp[from] = rhs[from] * inv[from];
        for (int i = from + 1; i < n; ++i) dp[i] = (rhs[i] - a[i] * dp[i - 1]) * inv[i];
        (*x)[n - 1] = dp[n - 1];
        for (int i = n - 2; i >= 0; --i) (*x)[i] = dp[i] - cp[i] * (*x)[i + 1];
      };
      std::vector<double> u(n, 0.0), z(n), y(n), rhs(n);
      u[0] = gamma;
      u[n - 1] = alpha;
      thomas(u, 0, &z);
      const double vz = z[0] + beta / gamma * z[n - 1];
      for (int col = 0; col < n; ++col) {
        std::fill(rhs.begin(), rhs.end(), 0.0);
        rhs[col] = 1.0;
        thomas(rhs, col, &y);
        const double vy = y[0] + beta / gamma * y[n - 1];
        const double f = vy / (1.0 + vz);
        // column col of G^-1 = row col (symmetric); store row col at offsets d = 0..n-1 from col-blo
        double* row = &hs->gram_inv[(size_t)col * n];
        int j = ((col - blo) % n + n) % n;
        for (int d = 0; d < n; ++d) {
          row[d] = y[j] - f * z[j];
          if (++j == n) j = 0;
        }
      }
    } else {
      // Elimination along the unrolled ring from either side: x_t = -pl[t] x_{t+1} left of a unit right-hand
      // side, x_t = -pr[t] x_{t-1} right of it. The ratios are below 1/2 on any mesh (the row sums of
      // the off-diagonals are half the diagonal; 0.27 on a uniform one) and forget their start by their
      // square per step, so kLead steps ahead of the first one that is used stand for the whole line. On the
      // ring an unknown is reached from both sides, over d and over n - d segments: its entry is the sum of the
      // two products of ratios (a third, once around the ring more, is below 2^-n of them). A row is a band of
      // half-width kGramBand for large n, where what comes the other way round is below 2^-(n - kGramBand) of
      // the diagonal, and whole for smaller n. (n divisions in place of a window
      // system per row: 2.6 -> 0.7 ms at n = 1500.)
      const bool band = n > kGramDenseMax;
      const int stride = band ? 2 * kGramBand + 1 : n, mid = band ? kGramBand : n / 2;
      constexpr int kLead = 64;
      hs->gram_band = mid;
      hs->gram_inv.assign((size_t)n * stride, 0.0);
      std::vector<double> pl(n, 0.0), pr(n, 0.0);
      double r = 0.0;
      for (int t = -kLead; t < n; ++t) {
        const int g = (t + n) % n;
        r = off(g) / (diag(g) - off((g + n - 1) % n) * r);
        if (t >= 0) pl[g] = r;
      }
      r = 0.0;
      for (int t = n - 1 + kLead; t >= 0; --t) {
        const int g = t % n;
        r = off((g + n - 1) % n) / (diag(g) - off(g) * r);
        if (t < n) pr[g] = r;
      }
      // kRows rows at a time: the products along a row are a chain
      constexpr int kRows = 8;
      const int len = band ? kGramBand : n - 1;
      std::vector<double> left((size_t)(len + 1) * kRows), right(left.size());   // d segments away, row by row
      for (int i0 = 0; i0 < n; i0 += kRows) {
        int gl[kRows], gr[kRows];
        for (int q = 0; q < kRows; ++q) {
          const int i = (i0 + q) % n, il = (i + n - 1) % n, ir = (i + 1) % n;
          left[q] = right[q] = 1.0 / (diag(i) - off(il) * pl[il] - off(i) * pr[ir]);
          gl[q] = il;
          gr[q] = ir;
        }
        for (int d = 1; d <= len; ++d)
          for (int q = 0; q < kRows; ++q) {
            left[(size_t)d * kRows + q] = -pl[gl[q]] * left[(size_t)(d - 1) * kRows + q];
            right[(size_t)d * kRows + q] = -pr[gr[q]] * right[(size_t)(d - 1) * kRows + q];
            gl[q] = gl[q] == 0 ? n - 1 : gl[q] - 1;
            gr[q] = gr[q] + 1 == n ? 0 : gr[q] + 1;
          }
        for (int q = 0; q < kRows && i0 + q < n; ++q) {
          double* row = &hs->gram_inv[(size_t)(i0 + q) * stride + mid];
          row[0] = left[q];
          for (int d = 1; d <= mid; ++d)
            row[-d] = left[(size_t)d * kRows + q] + (band ? 0.0 : right[(size_t)(n - d) * kRows + q]);
          for (int d = 1; d < stride - mid; ++d)
            row[d] = right[(size_t)d * kRows + q] + (band ? 0.0 : left[(size_t)(n - d) * kRows + q]);
        }
      }
    }
  }
  return AIM_OK;
}

}  // namespace aim
