// fc_geom.cu -- finite cell element data on the GPU (paper Sec. 2).
//
// Per background cell:
//   a(v,u) = (eta grad v, alpha grad u) - (v, n.eta grad u)_G - (n.eta grad v, u)_G + (v, lambda u)_G
//   b(v,p) = -(div v, alpha p) + (v, n p)_G
//   f(v)   = (v, alpha f)
// for the nodal functions of the cell (eq. stokes_disc_weak_fcm_2): the 2^d
// Q1 functions for velocity and pressure (the paper's pair), or the 3^d Q2
// velocity functions with the Q1 pressure functions (Taylor-Hood variant),
// with Gamma_D the obstacle boundary (no-slip, w = 0).  The volume rule is
// the recursive box split: a box is split into 2^d children when the level
// set changes sign among its 3^d sample points, down to the quadrature depth;
// leaves take the tensor 2-point (Q1) or 3-point (Q2) Gauss rule with alpha
// evaluated at each point.  The boundary rule is composite 2-point Gauss in the curve
// parameter (circle / ellipse) or in cos(theta) times a uniform rule in the
// azimuth (sphere); every rule point is owned by the cell that contains it.
//
// Q1: moments of the rule (cell_moments_kernel).  Q2: one warp per cell walks
// the split tree in depth-first order (children in lexicographic order) and
// adds point contributions in rule order, every entry a sum over the points;
// the points themselves (level set, basis, force) are evaluated one per lane
// and broadcast.  This translation unit is compiled with --fmad=false, so
// that a point's cell and side of the level set do not depend on contraction.
#include <math.h>

#include "fc_internal.cuh"

namespace fc {

namespace {

constexpr double kPi = 3.14159265358979323846;
constexpr int kStack = 48;

__device__ __forceinline__ double phi_shape(const Shape& s, int dim, const double* x) {
  double dx = x[0] - s.c[0], dy = x[1] - s.c[1];
  if (s.type == 0) {
    double q = dx * dx + dy * dy;
    if (dim == 3) {
      double dz = x[2] - s.c[2];
      q = q + dz * dz;
    }
    return s.r[0] - sqrt(q);
  }
  double xp = s.rot[0] * dx + s.rot[1] * dy;
  double yp = -s.rot[1] * dx + s.rot[0] * dy;
  double u = xp / s.r[0], v = yp / s.r[1];
  return 1.0 - (u * u + v * v);
}

// Sign of the level set: only shapes whose bounding box meets the cell can
// be positive at a point of the cell, so the candidate list decides it.
__device__ __forceinline__ bool inside_obstacle(const Shape* sh, const int* cand, int nc, int dim,
                                                const double* x) {
  double p = -1.0;
  for (int t = 0; t < nc; ++t) {
    double q = phi_shape(sh[cand[t]], dim, x);
    if (t == 0 || q > p) p = q;
  }
  return p > 0.0;
}

__device__ __forceinline__ void force_at(const LevelGeom& g, const double* x, double* f) {
  f[0] = f[1] = f[2] = 0.0;
  switch (g.force_kind) {
    case 0:
      f[0] = g.force[0]; f[1] = g.force[1]; f[2] = g.force[2];
      break;
    case 1:
      f[0] = g.force[0] * sin(kPi * x[0]);
      f[1] = g.force[1] * cos(kPi * x[1]);
      break;
    case 2:
      f[0] = g.force[0] * sin(kPi * x[1]);
      if (g.dim == 3) f[0] = f[0] * sin(kPi * x[2]);
      break;
    case 3:
      f[0] = -g.force[0] * (kPi / 2.0) * sin(kPi * x[0] / 2.0);
      break;
    default:
      break;
  }
}

// Q2-Q1 entries handled by one lane: e = lane + 32 t.  Entry index space:
// [A upper triangle (a <= b, a-major)] [B (c, a, b)] [F (c, a)], with NV = 3^d
// velocity and NP = 2^d pressure functions per cell.
template <int DIM>
struct Entries {
  static constexpr int NV = DIM == 3 ? 27 : 9;
  static constexpr int NP = 1 << DIM;
  static constexpr int NA = NV * (NV + 1) / 2;
  static constexpr int NB = DIM * NV * NP;
  static constexpr int NF = DIM * NV;
  static constexpr int NE = NA + NB + NF;
  static constexpr int PER = (NE + 31) / 32;
  static constexpr int NG = DIM == 3 ? 27 : 9;  // Gauss points on a leaf, 3 per direction
  // warps per CTA: the per-warp point queue grows with the basis and static
  // shared memory is limited to 48 KB per CTA
  static constexpr int WARPS = DIM == 3 ? 1 : 3;
};

struct EntryId {
  int kind, c, a, b;  // kind 0 A, 1 B, 2 F, -1 none
};

template <int DIM>
__device__ EntryId entry_of(int e) {
  using E = Entries<DIM>;
  EntryId id{-1, 0, 0, 0};
  if (e < E::NA) {
    int a = 0, rem = e;
    while (rem >= E::NV - a) { rem -= E::NV - a; ++a; }
    id.kind = 0; id.a = a; id.b = a + rem;
  } else if (e < E::NA + E::NB) {
    int t = e - E::NA;
    id.kind = 1; id.c = t / (E::NV * E::NP); id.a = (t / E::NP) % E::NV; id.b = t % E::NP;
  } else if (e < E::NE) {
    int t = e - E::NA - E::NB;
    id.kind = 2; id.c = t / E::NV; id.a = t % E::NV;
  }
  return id;
}

// Q2 functions on [0, 1]: q0 = (1-t)(1-2t), q1 = 4t(1-t), q2 = t(2t-1)
__device__ __forceinline__ void q2_1d(double t, double* v, double* d) {
  v[0] = (1.0 - t) * (1.0 - 2.0 * t);
  v[1] = 4.0 * t * (1.0 - t);
  v[2] = t * (2.0 * t - 1.0);
  d[0] = 4.0 * t - 3.0;
  d[1] = 4.0 - 8.0 * t;
  d[2] = 4.0 * t - 1.0;
}

// velocity values / gradients (NV) and pressure values (NP) at x
template <int DIM>
__device__ __forceinline__ void elem_basis(const double* x0, const double* h, const double* x, double* val,
                                           double (*grad)[3], double* pval) {
  double v[3][3], d[3][3], t[3] = {0.0, 0.0, 0.0};
  for (int k = 0; k < 3; ++k) {
    t[k] = k < DIM ? (x[k] - x0[k]) / h[k] : 0.0;
    q2_1d(t[k], v[k], d[k]);
  }
  constexpr int NV = DIM == 3 ? 27 : 9;
  for (int a = 0; a < NV; ++a) {
    const int ia[3] = {a % 3, (a / 3) % 3, a / 9};
    double f = 1.0;
    for (int k = 0; k < DIM; ++k) f = f * v[k][ia[k]];
    val[a] = f;
    grad[a][0] = grad[a][1] = grad[a][2] = 0.0;
    for (int k = 0; k < DIM; ++k) {
      double gk = d[k][ia[k]] / h[k];
      for (int m = 0; m < DIM; ++m)
        if (m != k) gk = gk * v[m][ia[m]];
      grad[a][k] = gk;
    }
  }
  for (int b = 0; b < (1 << DIM); ++b) {
    double f = 1.0;
    for (int k = 0; k < DIM; ++k) f = f * (((b >> k) & 1) ? t[k] : 1.0 - t[k]);
    pval[b] = f;
  }
}

template <int DIM>
struct WarpShared {
  static constexpr int NV = Entries<DIM>::NV, NP = Entries<DIM>::NP;
  int cand[kMaxShapesPerCell];
  double stk_lo[kStack][3];
  int stk_lev[kStack];
  // Gauss points of the volume rule waiting for evaluation, in rule order:
  // position and weight, then per point alpha, force, basis values and
  // gradients (filled one point per lane)
  double px[32][3];
  double pw[32];
  double pal[32];
  double pf[32][3];
  double pval[32][NV];
  double pgrad[32][NV][3];
  double ppv[32][NP];
};

// Angular index range [lo, hi] (before wrapping) of rule points t = step *
// (m + off) that can fall in the box [bx0, bx1] x [by0, by1], seen from the
// centre (cx, cy) after the map (dx, dy) -> ((R^T d)_x / a, (R^T d)_y / b).
// Returns false when the box contains the centre (all indices).
__device__ bool angular_range(double bx0, double bx1, double by0, double by1, double cx, double cy,
                              double ca, double sa, double a, double b, double step, double off,
                              long long* mlo, long long* mhi) {
  if (cx >= bx0 && cx <= bx1 && cy >= by0 && cy <= by1) return false;
  double mx = 0.5 * (bx0 + bx1) - cx, my = 0.5 * (by0 + by1) - cy;
  double ur = (ca * mx + sa * my) / a, vr = (-sa * mx + ca * my) / b;
  double tref = atan2(vr, ur);
  double dmin = 0.0, dmax = 0.0;
  for (int k = 0; k < 4; ++k) {
    double X = (k & 1) ? bx1 : bx0, Y = (k & 2) ? by1 : by0;
    double dx = X - cx, dy = Y - cy;
    double u = (ca * dx + sa * dy) / a, v = (-sa * dx + ca * dy) / b;
    // angle of (u, v) relative to the reference direction
    double cr = ur * v - vr * u, dt = ur * u + vr * v;
    double d = atan2(cr, dt);
    if (k == 0 || d < dmin) dmin = d;
    if (k == 0 || d > dmax) dmax = d;
  }
  double tlo = tref + dmin, thi = tref + dmax;
  *mlo = (long long)floor(tlo / step - off) - 1;
  *mhi = (long long)floor(thi / step - off) + 1;
  return true;
}

template <int DIM>
__global__ void __launch_bounds__(Entries<DIM>::WARPS * 32)
    cell_elements_q2_kernel(LevelGeom g, double* __restrict__ eA, double* __restrict__ eB,
                            double* __restrict__ eF, double* __restrict__ estat, unsigned* __restrict__ d_err) {
  using E = Entries<DIM>;
  constexpr int NL = E::NV, NP = E::NP, WARPS = E::WARPS;
  __shared__ WarpShared<DIM> wsh[WARPS];
  const int lane = threadIdx.x & 31;
  const int wib = threadIdx.x >> 5;
  WarpShared<DIM>& S = wsh[wib];
  const long long cell = (long long)blockIdx.x * WARPS + wib;
  if (cell >= g.ncell) return;
  const unsigned FULL = 0xffffffffu;

  long long ci = cell % g.n[0];
  long long cj = (cell / g.n[0]) % g.n[1];
  long long ck = DIM == 3 ? cell / ((long long)g.n[0] * g.n[1]) : 0;
  double x0[3];
  x0[0] = g.lo[0] + (double)ci * g.h[0];
  x0[1] = g.lo[1] + (double)cj * g.h[1];
  x0[2] = DIM == 3 ? g.lo[2] + (double)ck * g.h[2] : 0.0;
  double x1[3] = {x0[0] + g.h[0], x0[1] + g.h[1], DIM == 3 ? x0[2] + g.h[2] : 0.0};

  // ---- candidate shapes (bounding boxes meeting the slightly enlarged cell)
  int nc = 0;
  for (int base = 0; base < g.nshape; base += 32) {
    int s = base + lane;
    bool hit = false;
    if (s < g.nshape) {
      const Shape& sh = g.shapes[s];
      hit = true;
      for (int k = 0; k < DIM; ++k) {
        double m = 1e-9 * g.h[k];
        if (sh.c[k] + sh.bbr < x0[k] - m || sh.c[k] - sh.bbr > x1[k] + m) hit = false;
      }
    }
    unsigned bal = __ballot_sync(FULL, hit);
    int pos = nc + __popc(bal & ((1u << lane) - 1u));
    if (hit && pos < kMaxShapesPerCell) S.cand[pos] = s;
    nc += __popc(bal);
  }
  if (nc > kMaxShapesPerCell) {
    if (lane == 0) atomicOr(d_err, kErrTooManyShapes);
    nc = kMaxShapesPerCell;
  }
  __syncwarp();

  double acc[E::PER];
#pragma unroll
  for (int t = 0; t < E::PER; ++t) acc[t] = 0.0;
  double fluid_volume = 0.0, bmeasure = 0.0;
  int nvol = 0, nbnd = 0;

  // ---- volume rule: depth-first over the split tree.  The Gauss points of
  // the leaves are queued in rule order and evaluated 32 at a time, one
  // point per lane (level set, alpha, basis, force); the lanes then add the
  // queued points to their entries in queue order, so every entry is still
  // the sum over the points in rule order.
  const double gq[2] = {0.5 - 0.5 / sqrt(3.0), 0.5 + 0.5 / sqrt(3.0)};  // boundary rule
  // 3-point Gauss on the leaves: nodes 1/2 -+ sqrt(3/5)/2, 1/2, weights 5/18, 8/18, 5/18
  const double gq3[3] = {0.5 - 0.5 * sqrt(0.6), 0.5, 0.5 + 0.5 * sqrt(0.6)};
  const double gw3[3] = {5.0 / 18.0, 8.0 / 18.0, 5.0 / 18.0};
  constexpr int NG = E::NG;
  int npt = 0;
  auto flush = [&]() {
    if (lane < npt) {
      const double x[3] = {S.px[lane][0], S.px[lane][1], S.px[lane][2]};
      S.pal[lane] = inside_obstacle(g.shapes, S.cand, nc, DIM, x) ? g.alpha : 1.0;
      double val[NL], grad[NL][3], pv[NP];
      elem_basis<DIM>(x0, g.h, x, val, grad, pv);
      for (int a = 0; a < NL; ++a) {
        S.pval[lane][a] = val[a];
        for (int k = 0; k < 3; ++k) S.pgrad[lane][a][k] = grad[a][k];
      }
      for (int b = 0; b < NP; ++b) S.ppv[lane][b] = pv[b];
      double f[3] = {0.0, 0.0, 0.0};
      force_at(g, x, f);
      for (int k = 0; k < 3; ++k) S.pf[lane][k] = f[k];
    }
    __syncwarp();
    for (int q = 0; q < npt; ++q) {
      const double w = S.pw[q], al = S.pal[q];
#pragma unroll
      for (int t = 0; t < E::PER; ++t) {
        EntryId id = entry_of<DIM>(lane + 32 * t);
        if (id.kind == 0) {
          double gg = 0.0;
          for (int kk = 0; kk < DIM; ++kk) gg = gg + S.pgrad[q][id.a][kk] * S.pgrad[q][id.b][kk];
          acc[t] = acc[t] + w * al * g.eta * gg;
        } else if (id.kind == 1) {
          acc[t] = acc[t] - w * al * S.pgrad[q][id.a][id.c] * S.ppv[q][id.b];
        } else if (id.kind == 2) {
          acc[t] = acc[t] + w * al * S.pf[q][id.c] * S.pval[q][id.a];
        }
      }
      if (al == 1.0) fluid_volume = fluid_volume + w;
      nvol++;
    }
    __syncwarp();
    npt = 0;
  };
  int sp = 0;
  if (lane == 0) {
    S.stk_lo[0][0] = x0[0]; S.stk_lo[0][1] = x0[1]; S.stk_lo[0][2] = x0[2];
    S.stk_lev[0] = 0;
  }
  sp = 1;
  __syncwarp();
  while (sp > 0) {
    --sp;
    double lo[3] = {S.stk_lo[sp][0], S.stk_lo[sp][1], S.stk_lo[sp][2]};
    int level = S.stk_lev[sp];
    __syncwarp();
    double hb[3];
    for (int k = 0; k < 3; ++k) {
      double v = g.h[k];
      for (int l = 0; l < level; ++l) v = v * 0.5;
      hb[k] = v;
    }
    // sign at the 3^d sample points
    constexpr int NS = DIM == 3 ? 27 : 9;
    bool pos = false;
    if (lane < NS) {
      int i = lane % 3, j = (lane / 3) % 3, k = lane / 9;
      double x[3] = {lo[0] + hb[0] * (0.5 * i), lo[1] + hb[1] * (0.5 * j),
                     DIM == 3 ? lo[2] + hb[2] * (0.5 * k) : 0.0};
      pos = inside_obstacle(g.shapes, S.cand, nc, DIM, x);
    }
    unsigned bal = __ballot_sync(FULL, pos);
    int npos = __popc(bal);
    bool cut = (npos != 0 && npos != NS);
    if (cut && level < g.qdepth) {
      // push the 2^d children in reverse so that child 0 is processed first
      constexpr int NCH = 1 << DIM;
      if (lane == 0) {
        for (int ch = NCH - 1; ch >= 0; --ch) {
          double lc[3] = {lo[0], lo[1], lo[2]};
          for (int k = 0; k < DIM; ++k)
            if ((ch >> k) & 1) lc[k] = lo[k] + hb[k] * 0.5;
          if (sp + (NCH - 1 - ch) < kStack) {
            S.stk_lo[sp + (NCH - 1 - ch)][0] = lc[0];
            S.stk_lo[sp + (NCH - 1 - ch)][1] = lc[1];
            S.stk_lo[sp + (NCH - 1 - ch)][2] = lc[2];
            S.stk_lev[sp + (NCH - 1 - ch)] = level + 1;
          }
        }
      }
      sp += NCH;
      if (sp > kStack) {
        if (lane == 0) atomicOr(d_err, kErrBadIndex);
        sp = 0;
      }
      __syncwarp();
      continue;
    }
    // a leaf: queue its Gauss points
    if (npt + NG > 32) flush();
    if (lane < NG) {
      const int i = lane % 3, j = (lane / 3) % 3, k = lane / 9;
      S.px[npt + lane][0] = lo[0] + hb[0] * gq3[i];
      S.px[npt + lane][1] = lo[1] + hb[1] * gq3[j];
      S.px[npt + lane][2] = DIM == 3 ? lo[2] + hb[2] * gq3[k] : 0.0;
      double w = (hb[0] * gw3[i]) * (hb[1] * gw3[j]);
      if (DIM == 3) w = w * (hb[2] * gw3[k]);
      S.pw[npt + lane] = w;
    }
    npt += NG;
    __syncwarp();
  }
  if (npt > 0) flush();

  // ---- boundary rule of every candidate shape, points owned by this cell
  const int k2 = 1 << g.qdepth;
  for (int t = 0; t < nc; ++t) {
    const int s = S.cand[t];
    const Shape sh = g.shapes[s];
    if (DIM == 2) {
      double rmax = sh.type == 0 ? sh.r[0] : (sh.r[0] > sh.r[1] ? sh.r[0] : sh.r[1]);
      long long N = 8LL * (long long)ceil(2.0 * kPi * rmax / g.hmin) * k2;
      if (N < 64) N = 64;
      double dt = 2.0 * kPi / (double)N;
      double a = sh.type == 0 ? sh.r[0] : sh.r[0], b = sh.type == 0 ? sh.r[0] : sh.r[1];
      double ca = sh.type == 0 ? 1.0 : sh.rot[0], sa = sh.type == 0 ? 0.0 : sh.rot[1];
      double mg = 1e-9 * g.h[0];
      long long mlo = 0, mhi = N - 1;
      if (angular_range(x0[0] - mg, x1[0] + mg, x0[1] - mg, x1[1] + mg, sh.c[0], sh.c[1], ca, sa,
                        a, b, dt, 0.5, &mlo, &mhi)) {
        if (mhi - mlo + 1 >= N) { mlo = 0; mhi = N - 1; }
      }
      long long cnt = mhi - mlo + 1;
      long long start = ((mlo % N) + N) % N;
      // ascending order of m: the wrapped head [0, e] precedes [start, N-1]
      long long e_wrap = start + cnt - 1 - N;  // last index of the wrapped part, < 0 if none
      long long seg_b[2], seg_e[2];
      int nseg = 0;
      if (e_wrap >= 0) { seg_b[nseg] = 0; seg_e[nseg] = e_wrap; nseg++; seg_b[nseg] = start; seg_e[nseg] = N - 1; nseg++; }
      else { seg_b[0] = start; seg_e[0] = start + cnt - 1; nseg = 1; }
      for (int sg = 0; sg < nseg; ++sg) {
        long long npts = 2 * (seg_e[sg] - seg_b[sg] + 1);
        for (long long base = 0; base < npts; base += 32) {
          long long pidx = base + lane;
          bool ok = false;
          double px = 0, py = 0, nx = 0, ny = 0, wgt = 0;
          if (pidx < npts) {
            long long m = seg_b[sg] + pidx / 2;
            int j = (int)(pidx & 1);
            double tt = dt * ((double)m + gq[j]);
            double ct = cos(tt), st = sin(tt);
            if (sh.type == 0) {
              px = sh.c[0] + sh.r[0] * ct;
              py = sh.c[1] + sh.r[0] * st;
              nx = -ct; ny = -st;
              wgt = 0.5 * dt * sh.r[0];
            } else {
              double cr = sh.rot[0], sr = sh.rot[1];
              px = sh.c[0] + (cr * (a * ct) - sr * (b * st));
              py = sh.c[1] + (sr * (a * ct) + cr * (b * st));
              double tx = b * ct, ty = a * st;
              double nl = sqrt(tx * tx + ty * ty);
              nx = -(cr * tx - sr * ty) / nl;
              ny = -(sr * tx + cr * ty) / nl;
              double spd = sqrt((a * st) * (a * st) + (b * ct) * (b * ct));
              wgt = 0.5 * dt * spd;
            }
            double xx[3] = {px, py, 0.0};
            ok = true;
            long long idx[2];
            for (int k = 0; k < 2; ++k) {
              if (xx[k] < g.lo[k] || xx[k] > g.hi[k]) { ok = false; break; }
              long long ii = (long long)floor((xx[k] - g.lo[k]) / g.h[k]);
              if (ii >= g.n[k]) ii = g.n[k] - 1;
              if (ii < 0) ii = 0;
              idx[k] = ii;
            }
            if (ok && (idx[0] != ci || idx[1] != cj)) ok = false;
            if (ok) {
              for (int u = 0; u < nc; ++u)
                if (S.cand[u] != s && phi_shape(g.shapes[S.cand[u]], 2, xx) > 0.0) { ok = false; break; }
            }
          }
          // each lane evaluates the basis at its own point; the points are
          // then added in rule order with their values broadcast by shuffle
          double lval[NL], ldn[NL], lpv[NP];
          {
            double bx[3] = {px, py, 0.0};
            double val[NL], grad[NL][3];
            elem_basis<DIM>(x0, g.h, bx, val, grad, lpv);
            for (int q = 0; q < NL; ++q) {
              double sdn = 0.0;
              const double bnl[3] = {nx, ny, 0.0};
              for (int k = 0; k < DIM; ++k) sdn = sdn + bnl[k] * grad[q][k];
              lval[q] = val[q];
              ldn[q] = sdn;
            }
          }
          unsigned vb = __ballot_sync(FULL, ok);
          while (vb) {
            int src = __ffs(vb) - 1;
            vb &= vb - 1;
            double bn[3] = {__shfl_sync(FULL, nx, src), __shfl_sync(FULL, ny, src), 0.0};
            double bw = __shfl_sync(FULL, wgt, src);
            double val[NL], dn[NL], pv[NP];
#pragma unroll
            for (int q = 0; q < NL; ++q) {
              val[q] = __shfl_sync(FULL, lval[q], src);
              dn[q] = __shfl_sync(FULL, ldn[q], src);
            }
#pragma unroll
            for (int q = 0; q < NP; ++q) pv[q] = __shfl_sync(FULL, lpv[q], src);
#pragma unroll
            for (int u = 0; u < E::PER; ++u) {
              EntryId id = entry_of<DIM>(lane + 32 * u);
              if (id.kind == 0) {
                double tv = -g.eta * val[id.a] * dn[id.b] - g.eta * dn[id.a] * val[id.b] +
                            g.lambda * val[id.a] * val[id.b];
                acc[u] = acc[u] + bw * tv;
              } else if (id.kind == 1) {
                acc[u] = acc[u] + bw * val[id.a] * bn[id.c] * pv[id.b];
              }
            }
            bmeasure = bmeasure + bw;
            nbnd++;
          }
        }
      }
    } else {
      const double r = sh.r[0];
      long long Nm = (long long)ceil(2.0 * r / g.hmin) * k2;
      if (Nm < 8) Nm = 8;
      long long Nf = 2LL * (long long)ceil(2.0 * kPi * r / g.hmin) * k2;
      if (Nf < 16) Nf = 16;
      double dm = 2.0 / (double)Nm, df = 2.0 * kPi / (double)Nf;
      double wgt = r * r * (0.5 * dm) * df;
      double mz = 1e-9 * g.h[2];
      long long m0 = (long long)floor((((x0[2] - mz) - sh.c[2]) / r + 1.0) / dm) - 1;
      long long m1 = (long long)floor((((x1[2] + mz) - sh.c[2]) / r + 1.0) / dm) + 1;
      if (m0 < 0) m0 = 0;
      if (m1 > Nm - 1) m1 = Nm - 1;
      double mgx = 1e-9 * g.h[0], mgy = 1e-9 * g.h[1];
      for (long long m = m0; m <= m1; ++m) {
        for (int j = 0; j < 2; ++j) {
          double mu = -1.0 + dm * ((double)m + gq[j]);
          double st = sqrt(1.0 - mu * mu);
          double rho = r * st;
          // ring bounding box against the cell's xy box
          if (sh.c[0] + rho < x0[0] - mgx || sh.c[0] - rho > x1[0] + mgx ||
              sh.c[1] + rho < x0[1] - mgy || sh.c[1] - rho > x1[1] + mgy)
            continue;
          long long qlo = 0, qhi = Nf - 1;
          if (angular_range(x0[0] - mgx, x1[0] + mgx, x0[1] - mgy, x1[1] + mgy, sh.c[0], sh.c[1],
                            1.0, 0.0, 1.0, 1.0, df, 0.5, &qlo, &qhi)) {
            if (qhi - qlo + 1 >= Nf) { qlo = 0; qhi = Nf - 1; }
          }
          long long cnt = qhi - qlo + 1;
          long long start = ((qlo % Nf) + Nf) % Nf;
          long long e_wrap = start + cnt - 1 - Nf;
          long long seg_b[2], seg_e[2];
          int nseg = 0;
          if (e_wrap >= 0) { seg_b[nseg] = 0; seg_e[nseg] = e_wrap; nseg++; seg_b[nseg] = start; seg_e[nseg] = Nf - 1; nseg++; }
          else { seg_b[0] = start; seg_e[0] = start + cnt - 1; nseg = 1; }
          for (int sg = 0; sg < nseg; ++sg) {
            long long npts = seg_e[sg] - seg_b[sg] + 1;
            for (long long base = 0; base < npts; base += 32) {
              long long pidx = base + lane;
              bool ok = false;
              double ex = 0, ey = 0;
              double xx[3] = {0, 0, 0};
              if (pidx < npts) {
                long long q = seg_b[sg] + pidx;
                double ph = df * ((double)q + 0.5);
                double cp = cos(ph), spv = sin(ph);
                ex = st * cp;
                ey = st * spv;
                xx[0] = sh.c[0] + r * ex;
                xx[1] = sh.c[1] + r * ey;
                xx[2] = sh.c[2] + r * mu;
                ok = true;
                long long idx[3];
                for (int k = 0; k < 3; ++k) {
                  if (xx[k] < g.lo[k] || xx[k] > g.hi[k]) { ok = false; break; }
                  long long ii = (long long)floor((xx[k] - g.lo[k]) / g.h[k]);
                  if (ii >= g.n[k]) ii = g.n[k] - 1;
                  if (ii < 0) ii = 0;
                  idx[k] = ii;
                }
                if (ok && (idx[0] != ci || idx[1] != cj || idx[2] != ck)) ok = false;
                if (ok) {
                  for (int u = 0; u < nc; ++u)
                    if (S.cand[u] != s && phi_shape(g.shapes[S.cand[u]], 3, xx) > 0.0) { ok = false; break; }
                }
              }
              double lval[NL], ldn[NL], lpv[NP];
              {
                double val[NL], grad[NL][3];
                elem_basis<DIM>(x0, g.h, xx, val, grad, lpv);
                const double bnl[3] = {-ex, -ey, -mu};
                for (int qq = 0; qq < NL; ++qq) {
                  double sdn = 0.0;
                  for (int k = 0; k < DIM; ++k) sdn = sdn + bnl[k] * grad[qq][k];
                  lval[qq] = val[qq];
                  ldn[qq] = sdn;
                }
              }
              unsigned vb = __ballot_sync(FULL, ok);
              while (vb) {
                int src = __ffs(vb) - 1;
                vb &= vb - 1;
                double bn[3] = {-__shfl_sync(FULL, ex, src), -__shfl_sync(FULL, ey, src), -mu};
                double val[NL], dn[NL], pv[NP];
#pragma unroll
                for (int qq = 0; qq < NL; ++qq) {
                  val[qq] = __shfl_sync(FULL, lval[qq], src);
                  dn[qq] = __shfl_sync(FULL, ldn[qq], src);
                }
#pragma unroll
                for (int qq = 0; qq < NP; ++qq) pv[qq] = __shfl_sync(FULL, lpv[qq], src);
#pragma unroll
                for (int u = 0; u < E::PER; ++u) {
                  EntryId id = entry_of<DIM>(lane + 32 * u);
                  if (id.kind == 0) {
                    double tv = -g.eta * val[id.a] * dn[id.b] - g.eta * dn[id.a] * val[id.b] +
                                g.lambda * val[id.a] * val[id.b];
                    acc[u] = acc[u] + wgt * tv;
                  } else if (id.kind == 1) {
                    acc[u] = acc[u] + wgt * val[id.a] * bn[id.c] * pv[id.b];
                  }
                }
                bmeasure = bmeasure + wgt;
                nbnd++;
              }
            }
          }
        }
      }
    }
  }

  // ---- write back (A mirrored)
  double* A = eA + cell * NL * NL;
  double* B = eB + cell * DIM * NL * NP;
  double* F = eF + cell * DIM * NL;
#pragma unroll
  for (int t = 0; t < E::PER; ++t) {
    EntryId id = entry_of<DIM>(lane + 32 * t);
    if (id.kind == 0) {
      A[id.a * NL + id.b] = acc[t];
      A[id.b * NL + id.a] = acc[t];
    } else if (id.kind == 1) {
      B[(id.c * NL + id.a) * NP + id.b] = acc[t];
    } else if (id.kind == 2) {
      F[id.c * NL + id.a] = acc[t];
    }
  }
  if (lane == 0 && estat) {
    estat[cell * 4 + 0] = fluid_volume;
    estat[cell * 4 + 1] = bmeasure;
    estat[cell * 4 + 2] = (double)nvol;
    estat[cell * 4 + 3] = (double)nbnd;
  }
}

// ---------------------------------------------------------------------------
// Q1 element data by moments.
//
// Every entry of the Q1 matrices is an integral of a product of 1D functions
// that are quadratic at most in each direction, so a cell needs 3^d moments of
// its rule, not one sum per entry: with l0 = 1 - t, l1 = t on [0, 1] and the
// quadratic basis (l0^2, l0 l1, l1^2),
//   T[i,j,k] = sum_q w alpha beta_i beta_j beta_k   over the volume points,
//   U_0[..] = sum_q w beta beta beta, U_{1+c}[..] = sum_q w n_c beta beta beta
// over the obstacle points of the cell.  l_a l_b is beta_{a+b}, l_b alone is
// l_b (l0 + l1) and 1 is (l0 + l1)^2, so each entry is a sum of moments with
// positive weights (no cancellation beyond the entry's own).  FP64 is the
// bound (one warp instruction per 64 clocks and SM partition): a volume point
// costs a warp 2 FP64 instructions instead of about 55, an obstacle point 6
// instead of about 70.
//
// Split over the GPU: a first pass, one warp per cell, finishes the cells that
// no obstacle surface can reach (alpha times the reference element matrices)
// and lists the others; the second takes a CTA per listed cell, a warp per
// child box of the cell and all warps over the obstacle points, so that the
// few large cells of the coarse levels do not leave one warp with thousands of
// points.  Setup and solve of 40 spheres on 32^3 to 4^3 cells: 153.3 ms with a
// warp per cell and a sum per entry (71.6 ms of it this rule), 87.6 ms so.
constexpr int kRing = 128;  // azimuths of a sphere rule tabulated at a time

// phi > 0 for the circle / sphere without the square root where the distance
// decides by more than rounding; the same answer as phi_shape() > 0
__device__ __forceinline__ bool in_shape(const Shape& s, int dim, const double* x) {
  if (s.type != 0) return phi_shape(s, dim, x) > 0.0;
  const double dx = x[0] - s.c[0], dy = x[1] - s.c[1];
  double q = dx * dx + dy * dy;
  if (dim == 3) {
    const double dz = x[2] - s.c[2];
    q = q + dz * dz;
  }
  const double rr = s.r[0] * s.r[0];
  if (q < rr * (1.0 - 1e-12)) return true;
  if (q > rr * (1.0 + 1e-12)) return false;
  return s.r[0] - sqrt(q) > 0.0;
}

__device__ __forceinline__ bool in_any(const Shape* sh, const int* cand, int nc, int dim, const double* x) {
  for (int t = 0; t < nc; ++t)
    if (in_shape(sh[cand[t]], dim, x)) return true;
  return false;
}

// the shapes whose bounding boxes meet the slightly enlarged cell, in
// ascending order (one warp); the count may exceed the list's length
template <int DIM>
__device__ int find_candidates(const LevelGeom& g, const double* x0, const double* x1, int lane, int* cand) {
  int nc = 0;
  for (int base = 0; base < g.nshape; base += 32) {
    const int s = base + lane;
    bool hit = s < g.nshape;
    if (hit) {
      const Shape& sh = g.shapes[s];
      // float32 first: a box that is clear of the cell by more than rounding
      for (int k = 0; k < DIM; ++k) {
        const float c = (float)sh.c[k], r = (float)sh.bbr, a = (float)x0[k], b = (float)x1[k];
        const float m = 1e-5f * (fabsf(c) + r + fabsf(a) + fabsf(b));
        if (c + r < a - m || c - r > b + m) hit = false;
      }
      if (hit)
        for (int k = 0; k < DIM; ++k) {
          const double m = 1e-9 * g.h[k];
          if (sh.c[k] + sh.bbr < x0[k] - m || sh.c[k] - sh.bbr > x1[k] + m) hit = false;
        }
    }
    const unsigned bal = __ballot_sync(0xffffffffu, hit);
    const int pos = nc + __popc(bal & ((1u << lane) - 1u));
    if (hit && pos < kMaxShapesPerCell) cand[pos] = s;
    nc += __popc(bal);
  }
  __syncwarp();
  return nc;
}

template <int DIM>
__device__ __forceinline__ void cell_box(const LevelGeom& g, long long cell, int* ic, double* x0, double* x1) {
  const unsigned u = (unsigned)cell, n0 = (unsigned)g.n[0], n1 = (unsigned)g.n[1], t = u / n0;
  ic[0] = (int)(u - t * n0);
  ic[1] = DIM == 3 ? (int)(t % n1) : (int)t;
  ic[2] = DIM == 3 ? (int)(t / n1) : 0;
  for (int k = 0; k < 3; ++k) {
    x0[k] = k < DIM ? g.lo[k] + (double)ic[k] * g.h[k] : 0.0;
    x1[k] = k < DIM ? x0[k] + g.h[k] : 0.0;
  }
}

// alpha times the reference element matrices (a warp), see the write-back of
// the second pass for what a plain cell is
template <int DIM>
__device__ __forceinline__ void write_plain(double al, const double* __restrict__ refA, const double* __restrict__ refB,
                                            double* __restrict__ A, double* __restrict__ B, int t0, int nt) {
  constexpr int NL = 1 << DIM;
  for (int t = t0; t < NL * NL; t += nt) A[t] = al * refA[t];
  for (int t = t0; t < DIM * NL * NL; t += nt) B[t] = al * refB[t];
}

// Pass 1: a warp per cell.
template <int DIM>
__global__ void __launch_bounds__(256)
    cell_plain_kernel(LevelGeom g, double* __restrict__ eA, double* __restrict__ eB, double* __restrict__ eF,
                      double* __restrict__ estat, unsigned* __restrict__ d_err, const double* __restrict__ refA,
                      const double* __restrict__ refB, unsigned char* __restrict__ cclass, int* __restrict__ list,
                      int* __restrict__ count) {
  constexpr int NL = 1 << DIM;
  __shared__ int scand[8][kMaxShapesPerCell];
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  const long long cell = (long long)blockIdx.x * 8 + wib;
  if (cell >= g.ncell) return;
  int ic[3];
  double x0[3], x1[3];
  cell_box<DIM>(g, cell, ic, x0, x1);
  int* cand = scand[wib];
  int nc = find_candidates<DIM>(g, x0, x1, lane, cand);
  if (nc > kMaxShapesPerCell) {
    if (lane == 0) atomicOr(d_err, kErrTooManyShapes);
    nc = kMaxShapesPerCell;
  }
  // near: the surface of some candidate may meet the cell (nearest and
  // farthest point of the box against the radius, with room for rounding)
  bool near = false, inside = false;
  for (int t = lane; t < nc; t += 32) {
    const Shape& sh = g.shapes[cand[t]];
    double dn = 0.0, df = 0.0;
    for (int k = 0; k < DIM; ++k) {
      const double a = x0[k] - sh.c[k], b = x1[k] - sh.c[k];
      const double lo = a > 0.0 ? a : (b < 0.0 ? -b : 0.0), hi = fmax(fabs(a), fabs(b));
      dn = dn + lo * lo;
      df = df + hi * hi;
    }
    const double rr = sh.r[0] * sh.r[0], m = 1e-7 * (rr + df);
    if (sh.type != 0 || !(dn > rr + m || df < rr - m)) near = true;
    else if (df < rr) inside = true;
  }
  if (__any_sync(0xffffffffu, near)) {
    if (lane == 0) list[atomicAdd(count, 1)] = (int)cell;
    return;
  }
  const double al = __any_sync(0xffffffffu, inside) ? g.alpha : 1.0;
  write_plain<DIM>(al, refA, refB, eA + cell * NL * NL, eB + cell * DIM * NL * NL, lane, 32);
  double w = 1.0;
  for (int k = 0; k < DIM; ++k) w = w * (g.h[k] * 0.5);
  if (lane < DIM * NL) {
    const int c = lane / NL, a = lane % NL;
    double f;
    if (g.force_kind == 0) {
      f = w * al * g.force[c];  // the functions of a cell have the same mean: 2^d points, 2^-d each
    } else {
      const double gq[2] = {0.5 - 0.5 / sqrt(3.0), 0.5 + 0.5 / sqrt(3.0)};
      f = 0.0;
      for (int q = 0; q < NL; ++q) {
        double x[3] = {0.0, 0.0, 0.0}, v = 1.0, fo[3];
        for (int k = 0; k < DIM; ++k) {
          const double t = gq[(q >> k) & 1];
          x[k] = x0[k] + g.h[k] * t;
          v = v * (((a >> k) & 1) ? t : 1.0 - t);
        }
        force_at(g, x, fo);
        f = f + w * al * fo[c] * v;
      }
    }
    eF[cell * DIM * NL + lane] = f;
  }
  if (lane == 0) {
    if (cclass) cclass[cell] = al == 1.0 ? 1 : 2;
    if (estat) {
      estat[cell * 4 + 0] = al == 1.0 ? w * NL : 0.0;
      estat[cell * 4 + 1] = 0.0;
      estat[cell * 4 + 2] = (double)NL;
      estat[cell * 4 + 3] = 0.0;
    }
  }
}

template <int DIM>
struct MomQueue {
  double x[32][3], w[32];    // volume points as they come, in rule order
  double b[3][32][3];        // beta per direction; direction 0 times the weight on volume points
  double wn[32][4];          // obstacle points: w, w n
  double l[3][32][2], f[32][3];  // force other than constant: 1D functions, w alpha f
};

template <int DIM>
struct MomShared {
  static constexpr int W = 1 << DIM, NM = DIM == 3 ? 27 : 9, NL = 1 << DIM;
  int cand[kMaxShapesPerCell];
  int nc, item, rootcut;
  double stk_lo[W][kStack][3];
  int stk_lev[W][kStack];
  MomQueue<DIM> q[W];
  double T[W][NM], U[W][4][NM], F[W][DIM * NL];
  double fluid[W], bmeas[W];
  int nvol[W], nbnd[W], first[W], mixed[W];  // alpha of the first point: 0 none, 1 fluid, 2 fictitious
  double ct[kRing], sn[kRing];
};

// Pass 2: a CTA of 2^d warps per listed cell (all cells of `cells` or of the
// grid when list is null).
template <int DIM>
__global__ void __launch_bounds__(32 << DIM)
    cell_moments_kernel(LevelGeom g, double* __restrict__ eA, double* __restrict__ eB, double* __restrict__ eF,
                        double* __restrict__ estat, unsigned* __restrict__ d_err, const double* __restrict__ refA,
                        const double* __restrict__ refB, unsigned char* __restrict__ cclass,
                        const long long* __restrict__ cells, const int* __restrict__ list,
                        const int* __restrict__ count, int* __restrict__ next, long long nitems) {
  using MS = MomShared<DIM>;
  constexpr int NL = MS::NL, W = MS::W, NM = MS::NM, NCH = 1 << DIM, NS = DIM == 3 ? 27 : 9;
  constexpr int PAR = DIM == 3 ? 1 : 3;  // points whose moments a warp adds at a time
  extern __shared__ double mom_raw[];
  MS& S = *reinterpret_cast<MS*>(mom_raw);
  const int tid = threadIdx.x, lane = tid & 31, wib = tid >> 5;
  const unsigned FULL = 0xffffffffu;
  const int total = list ? *count : (int)nitems;
  MomQueue<DIM>& Q = S.q[wib];
  const double gq[2] = {0.5 - 0.5 / sqrt(3.0), 0.5 + 0.5 / sqrt(3.0)};
  // the moment of this lane and, in 2D, its point of a group of three
  const int mom = lane % NM, grp = lane / NM;
  const bool owner = grp < PAR;
  const int mi = mom % 3, mj = (mom / 3) % 3, mk = DIM == 3 ? mom / 9 : 0;
  for (;;) {
    if (tid == 0) S.item = atomicAdd(next, 1);
    __syncthreads();
    const int item = S.item;
    if (item >= total) break;
    const long long slot = list ? list[item] : item;
    const long long cell = cells ? cells[slot] : slot;
    int ic[3];
    double x0[3], x1[3];
    cell_box<DIM>(g, cell, ic, x0, x1);
    if (wib == 0) {
      const int found = find_candidates<DIM>(g, x0, x1, lane, S.cand);
      if (lane == 0) {
        if (found > kMaxShapesPerCell) atomicOr(d_err, kErrTooManyShapes);
        S.nc = found < kMaxShapesPerCell ? found : kMaxShapesPerCell;
      }
      __syncwarp();
    }
    __syncthreads();
    const int nc = S.nc;

    // sign at the 3^d sample points of a box of the split tree
    auto box_cut = [&](const double* lo, const double* hb) {
      bool pos = false;
      if (lane < NS) {
        const int i = lane % 3, j = (lane / 3) % 3, k = lane / 9;
        const double x[3] = {lo[0] + hb[0] * (0.5 * i), lo[1] + hb[1] * (0.5 * j),
                             DIM == 3 ? lo[2] + hb[2] * (0.5 * k) : 0.0};
        pos = in_any(g.shapes, S.cand, nc, DIM, x);
      }
      const int npos = __popc(__ballot_sync(FULL, pos));
      return npos != 0 && npos != NS;
    };
    if (wib == 0) {
      const bool cut = g.qdepth > 0 && box_cut(x0, g.h);
      if (lane == 0) S.rootcut = cut;
    }
    __syncthreads();
    const bool split = S.rootcut;

    // ---- volume rule: warp w walks child w of a split cell depth first; an
    // uncut cell is one leaf (warp 0)
    double acc = 0.0, accf = 0.0, fluid = 0.0;
    int nvol = 0, npt = 0, first = 0;
    bool mixed = false;
    auto flush = [&]() {
      double al = 1.0;
      if (lane < npt) {
        const double x[3] = {Q.x[lane][0], Q.x[lane][1], Q.x[lane][2]};
        const bool in = in_any(g.shapes, S.cand, nc, DIM, x);
        al = in ? g.alpha : 1.0;
        const double wal = Q.w[lane] * al;
#pragma unroll
        for (int k = 0; k < DIM; ++k) {
          const double t = (x[k] - x0[k]) / g.h[k], u = 1.0 - t, m = k == 0 ? wal : 1.0;
          Q.b[k][lane][0] = m * (u * u);
          Q.b[k][lane][1] = m * (u * t);
          Q.b[k][lane][2] = m * (t * t);
          Q.l[k][lane][0] = u;
          Q.l[k][lane][1] = t;
        }
        if (g.force_kind != 0) {
          double f[3];
          force_at(g, x, f);
          for (int k = 0; k < DIM; ++k) Q.f[lane][k] = wal * f[k];
        }
        if (al == 1.0) fluid = fluid + Q.w[lane];
      }
      const unsigned live = __ballot_sync(FULL, lane < npt);
      const unsigned one = __ballot_sync(FULL, lane < npt && al == 1.0);
      if (first == 0) first = (one & 1u) ? 1 : 2;
      if (first == 1 ? one != live : one != 0u) mixed = true;
      __syncwarp();
      for (int q = 0; q < npt; q += PAR) {
        const int p = q + grp;
        if (owner && p < npt) {
          double v = Q.b[0][p][mi] * Q.b[1][p][mj];
          if (DIM == 3) acc = fma(v, Q.b[2][p][mk], acc);
          else acc = acc + v;
        }
      }
      if (g.force_kind != 0 && lane < DIM * NL) {
        const int c = lane / NL, a = lane % NL;
        for (int q = 0; q < npt; ++q) {
          double v = Q.f[q][c];
          for (int k = 0; k < DIM; ++k) v = v * Q.l[k][q][(a >> k) & 1];
          accf = accf + v;
        }
      }
      nvol += npt;
      npt = 0;
      __syncwarp();
    };
    int sp = 0;
    if (split || wib == 0) {
      if (lane == 0) {
        for (int k = 0; k < 3; ++k)
          S.stk_lo[wib][0][k] = x0[k] + (split && k < DIM && ((wib >> k) & 1) ? g.h[k] * 0.5 : 0.0);
        S.stk_lev[wib][0] = split ? 1 : 0;
      }
      sp = 1;
    }
    __syncwarp();
    while (sp > 0) {
      --sp;
      const double lo[3] = {S.stk_lo[wib][sp][0], S.stk_lo[wib][sp][1], S.stk_lo[wib][sp][2]};
      const int level = S.stk_lev[wib][sp];
      __syncwarp();
      double hb[3];
      for (int k = 0; k < 3; ++k) hb[k] = ldexp(g.h[k], -level);
      // (the root was tested above; boxes at the last depth are leaves)
      if (level > 0 && level < g.qdepth && box_cut(lo, hb)) {
        if (sp + NCH > kStack) {
          if (lane == 0) atomicOr(d_err, kErrBadIndex);
          break;
        }
        if (lane < NCH) {
          // reverse order, so that child 0 is taken first
          const int ch = NCH - 1 - lane;
          for (int k = 0; k < 3; ++k)
            S.stk_lo[wib][sp + lane][k] = k < DIM && ((ch >> k) & 1) ? lo[k] + hb[k] * 0.5 : lo[k];
          S.stk_lev[wib][sp + lane] = level + 1;
        }
        sp += NCH;
        __syncwarp();
        continue;
      }
      if (npt + NL > 32) flush();
      if (lane < NL) {
        const int i = lane & 1, j = (lane >> 1) & 1, k = lane >> 2;
        double w = 1.0;
        for (int m = 0; m < DIM; ++m) w = w * (hb[m] * 0.5);
        Q.x[npt + lane][0] = lo[0] + hb[0] * gq[i];
        Q.x[npt + lane][1] = lo[1] + hb[1] * gq[j];
        Q.x[npt + lane][2] = DIM == 3 ? lo[2] + hb[2] * gq[k] : 0.0;
        Q.w[npt + lane] = w;
      }
      npt += NL;
      __syncwarp();
    }
    if (npt > 0) flush();

    // ---- obstacle points of the cell: the index ranges of each candidate's
    // rule that can meet it, spread over the CTA's threads
    double au[4] = {0.0, 0.0, 0.0, 0.0}, bmeas = 0.0;
    int nbnd = 0;
    // a warp's points (one per lane, ok: in this cell) into its moments
    auto add_points = [&](bool ok, const double* x, const double* n, double w) {
      const unsigned vb = __ballot_sync(FULL, ok);
      if (vb == 0u) return;
      const int cnt = __popc(vb);
      if (ok) {
        const int p = __popc(vb & ((1u << lane) - 1u));
#pragma unroll
        for (int k = 0; k < DIM; ++k) {
          const double t = (x[k] - x0[k]) / g.h[k], u = 1.0 - t;
          Q.b[k][p][0] = u * u;
          Q.b[k][p][1] = u * t;
          Q.b[k][p][2] = t * t;
          Q.wn[p][1 + k] = w * n[k];
        }
        Q.wn[p][0] = w;
        bmeas = bmeas + w;
      }
      __syncwarp();
      for (int q = 0; q < cnt; q += PAR) {
        const int p = q + grp;
        if (owner && p < cnt) {
          double v = Q.b[0][p][mi] * Q.b[1][p][mj];
          if (DIM == 3) v = v * Q.b[2][p][mk];
#pragma unroll
          for (int c = 0; c <= DIM; ++c) au[c] = fma(v, Q.wn[p][c], au[c]);
        }
      }
      nbnd += cnt;
      __syncwarp();
    };
    auto owned_by_cell = [&](const double* x, int s) {
      for (int k = 0; k < DIM; ++k) {
        if (x[k] < g.lo[k] || x[k] > g.hi[k]) return false;
        int ii = (int)floor((x[k] - g.lo[k]) / g.h[k]);
        if (ii >= g.n[k]) ii = g.n[k] - 1;
        if (ii < 0) ii = 0;
        if (ii != ic[k]) return false;
      }
      for (int u = 0; u < nc; ++u)
        if (S.cand[u] != s && in_shape(g.shapes[S.cand[u]], DIM, x)) return false;
      return true;
    };
    const int k2 = 1 << g.qdepth;
    for (int t = 0; t < nc; ++t) {
      const int s = S.cand[t];
      const Shape sh = g.shapes[s];
      const double mgx = 1e-9 * g.h[0], mgy = 1e-9 * g.h[1];
      const double r = sh.r[0], a = sh.r[0], b = sh.type == 0 ? sh.r[0] : sh.r[1];
      const double cr = sh.type == 0 ? 1.0 : sh.rot[0], sr = sh.type == 0 ? 0.0 : sh.rot[1];
      long long N, m0 = 0, m1 = 0;
      double dm = 0.0;
      if (DIM == 2) {
        N = 8LL * (long long)ceil(2.0 * kPi * (a > b ? a : b) / g.hmin) * k2;
        if (N < 64) N = 64;
      } else {
        long long Nm = (long long)ceil(2.0 * r / g.hmin) * k2;
        if (Nm < 8) Nm = 8;
        N = 2LL * (long long)ceil(2.0 * kPi * r / g.hmin) * k2;
        if (N < 16) N = 16;
        dm = 2.0 / (double)Nm;
        const double mz = 1e-9 * g.h[2];
        m0 = (long long)floor((((x0[2] - mz) - sh.c[2]) / r + 1.0) / dm) - 1;
        m1 = (long long)floor((((x1[2] + mz) - sh.c[2]) / r + 1.0) / dm) + 1;
        if (m0 < 0) m0 = 0;
        if (m1 > Nm - 1) m1 = Nm - 1;
      }
      const double dt = 2.0 * kPi / (double)N;
      long long mlo = 0, mhi = N - 1;
      if (angular_range(x0[0] - mgx, x1[0] + mgx, x0[1] - mgy, x1[1] + mgy, sh.c[0], sh.c[1], cr, sr, a, b, dt, 0.5,
                        &mlo, &mhi)) {
        if (mhi - mlo + 1 >= N) { mlo = 0; mhi = N - 1; }
      }
      // (64 bits: N passes 2^31 for radii of a million cells)
      const long long cnt = mhi - mlo + 1, start = ((mlo % N) + N) % N;
      if (DIM == 2) {
        for (long long base = wib * 32; base < 2 * cnt; base += 32 * W) {
          const long long p = base + lane;
          bool ok = false;
          double x[3] = {0.0, 0.0, 0.0}, nv[3] = {0.0, 0.0, 0.0}, w = 0.0;
          if (p < 2 * cnt) {
            long long m = start + p / 2;
            if (m >= N) m -= N;
            const double tt = dt * ((double)m + gq[p & 1]);
            const double ct = cos(tt), st = sin(tt);
            if (sh.type == 0) {
              x[0] = sh.c[0] + r * ct;
              x[1] = sh.c[1] + r * st;
              nv[0] = -ct; nv[1] = -st;
              w = 0.5 * dt * r;
            } else {
              x[0] = sh.c[0] + (cr * (a * ct) - sr * (b * st));
              x[1] = sh.c[1] + (sr * (a * ct) + cr * (b * st));
              const double tx = b * ct, ty = a * st;
              const double nl = sqrt(tx * tx + ty * ty);
              nv[0] = -(cr * tx - sr * ty) / nl;
              nv[1] = -(sr * tx + cr * ty) / nl;
              w = 0.5 * dt * sqrt((a * st) * (a * st) + (b * ct) * (b * ct));
            }
            ok = owned_by_cell(x, s);
          }
          add_points(ok, x, nv, w);
        }
      } else {
        // rings m0 .. m1 (two Gauss rings each) x the azimuth range, the
        // azimuths' cosines and sines tabulated kRing at a time
        const double w = r * r * (0.5 * dm) * dt;
        const long long nr = m1 >= m0 ? 2 * (m1 - m0 + 1) : 0;
        for (long long q0 = 0; q0 < cnt; q0 += kRing) {
          const int nq = cnt - q0 < kRing ? (int)(cnt - q0) : kRing;
          __syncthreads();
          for (int q = tid; q < nq; q += 32 * W) {
            long long m = start + q0 + q;
            if (m >= N) m -= N;
            const double ph = dt * ((double)m + 0.5);
            S.ct[q] = cos(ph);
            S.sn[q] = sin(ph);
          }
          __syncthreads();
          for (long long base = wib * 32; base < nr * nq; base += 32 * W) {
            const long long p = base + lane;
            bool ok = false;
            double x[3] = {0.0, 0.0, 0.0}, nv[3] = {0.0, 0.0, 0.0};
            if (p < nr * nq) {
              const long long ring = p / nq;
              const int q = (int)(p - ring * nq);
              const double mu = -1.0 + dm * ((double)(m0 + ring / 2) + gq[ring & 1]);
              const double st = sqrt(1.0 - mu * mu);
              const double ex = st * S.ct[q], ey = st * S.sn[q];
              x[0] = sh.c[0] + r * ex;
              x[1] = sh.c[1] + r * ey;
              x[2] = sh.c[2] + r * mu;
              nv[0] = -ex; nv[1] = -ey; nv[2] = -mu;
              ok = owned_by_cell(x, s);
            }
            add_points(ok, x, nv, w);
          }
        }
      }
    }

    // ---- sums over the warps (fixed order)
    if (DIM == 2) {
      // the three groups of nine lanes
      const double a1 = __shfl_down_sync(FULL, acc, 9), a2 = __shfl_down_sync(FULL, acc, 18);
      acc = acc + a1 + a2;
#pragma unroll
      for (int c = 0; c <= DIM; ++c) {
        const double u1 = __shfl_down_sync(FULL, au[c], 9), u2 = __shfl_down_sync(FULL, au[c], 18);
        au[c] = au[c] + u1 + u2;
      }
    }
    for (int o = 16; o > 0; o >>= 1) {
      fluid = fluid + __shfl_xor_sync(FULL, fluid, o);
      bmeas = bmeas + __shfl_xor_sync(FULL, bmeas, o);
    }
    if (lane < NM) {
      S.T[wib][lane] = acc;
#pragma unroll
      for (int c = 0; c <= DIM; ++c) S.U[wib][c][lane] = au[c];
    }
    if (lane < DIM * NL) S.F[wib][lane] = accf;
    if (lane == 0) {
      S.fluid[wib] = fluid; S.bmeas[wib] = bmeas;
      S.nvol[wib] = nvol; S.nbnd[wib] = nbnd; S.first[wib] = first; S.mixed[wib] = mixed;
    }
    __syncthreads();
    for (int e = tid; e < NM * (2 + DIM) + DIM * NL; e += 32 * W) {
      double* p;
      int step;
      if (e < NM) { p = &S.T[0][e]; step = NM; }
      else if (e < NM * (2 + DIM)) { p = &S.U[0][(e - NM) / NM][(e - NM) % NM]; step = 4 * NM; }
      else { p = &S.F[0][e - NM * (2 + DIM)]; step = DIM * NL; }
      double v = p[0];
      for (int w = 1; w < W; ++w) v = v + p[w * step];
      p[0] = v;
    }
    __syncthreads();

    // ---- write back (A mirrored).  A plain cell (not split, one alpha at all
    // its Gauss points, no boundary points) takes alpha times the reference
    // element matrices of the same rule on an uncut cell: the same values up
    // to rounding, but bit-identical across plain cells, which makes the
    // patch blocks of uncut regions bit-identical (patch classes).
    int nb = 0, nvl = 0;
    double fl = 0.0, bm = 0.0;
    for (int w = 0; w < W; ++w) { nb += S.nbnd[w]; nvl += S.nvol[w]; fl = fl + S.fluid[w]; bm = bm + S.bmeas[w]; }
    const bool plain = refA != nullptr && !split && nb == 0 && !S.mixed[0];
    const double al1 = S.first[0] == 1 ? 1.0 : g.alpha;
    double* A = eA + slot * NL * NL;
    double* B = eB + slot * DIM * NL * NL;
    const double* T = S.T[0];
    constexpr int st[3] = {1, 3, 9};
    double hi[3];
    for (int k = 0; k < DIM; ++k) hi[k] = 1.0 / g.h[k];
    if (plain) {
      write_plain<DIM>(al1, refA, refB, A, B, tid, 32 * W);
    } else {
      for (int e = tid; e < NL * NL * (1 + DIM); e += 32 * W) {
        const int a = (e / NL) % NL, b = e % NL, kind = e / (NL * NL);
        int at = 0;  // beta_{a+b} in every direction
        for (int k = 0; k < DIM; ++k) at += (((a >> k) & 1) + ((b >> k) & 1)) * st[k];
        if (kind == 0) {
          if (a > b) continue;
          double v = 0.0, dn = 0.0;
          for (int k = 0; k < DIM; ++k) {
            const int ak = (a >> k) & 1, bk = (b >> k) & 1, z = at - (ak + bk) * st[k];
            const double sa = ak ? hi[k] : -hi[k], sb = bk ? hi[k] : -hi[k];
            v = v + sa * sb * (T[z] + 2.0 * T[z + st[k]] + T[z + 2 * st[k]]);
            const double* n = S.U[0][1 + k];
            dn = dn + sb * (n[z + ak * st[k]] + n[z + (ak + 1) * st[k]]) +
                 sa * (n[z + bk * st[k]] + n[z + (bk + 1) * st[k]]);
          }
          v = g.eta * (v - dn) + g.lambda * S.U[0][0][at];
          A[a * NL + b] = v;
          A[b * NL + a] = v;
        } else {
          const int c = kind - 1, ak = (a >> c) & 1, bk = (b >> c) & 1, z = at - (ak + bk) * st[c];
          const double sa = ak ? hi[c] : -hi[c];
          B[(c * NL + a) * NL + b] = S.U[0][1 + c][at] - sa * (T[z + bk * st[c]] + T[z + (bk + 1) * st[c]]);
        }
      }
    }
    if (tid < DIM * NL) {
      const int c = tid / NL, a = tid % NL;
      double f = S.F[0][tid];
      if (g.force_kind == 0) {
        f = 0.0;
        for (int t = 0; t < NL; ++t) {
          int z = 0;
          for (int k = 0; k < DIM; ++k) z += (((a >> k) & 1) + ((t >> k) & 1)) * st[k];
          f = f + T[z];
        }
        f = f * g.force[c];
      }
      eF[slot * DIM * NL + tid] = f;
    }
    if (tid == 0) {
      if (cclass) cclass[slot] = plain ? (al1 == 1.0 ? 1 : 2) : 0;
      if (estat) {
        estat[slot * 4 + 0] = fl;
        estat[slot * 4 + 1] = bm;
        estat[slot * 4 + 2] = (double)nvl;
        estat[slot * 4 + 3] = (double)nb;
      }
    }
    __syncthreads();
  }
}

template <int DIM>
cudaError_t run_moments(const LevelGeom& g, double* eA, double* eB, double* eF, double* estat, unsigned* d_err,
                        const double* refA, const double* refB, unsigned char* cclass, const long long* cells,
                        long long ncells, cudaStream_t s) {
  const long long n = cells ? ncells : g.ncell;
  if (n <= 0) return cudaSuccess;
  int* buf = nullptr;  // [0] listed cells, [1] next item, then the list
  cudaError_t e = cudaMallocAsync((void**)&buf, sizeof(int) * (size_t)(2 + (refA ? n : 0)), s);
  if (e != cudaSuccess) return e;
  e = cudaMemsetAsync(buf, 0, 2 * sizeof(int), s);
  if (e == cudaSuccess && refA) {
    cell_plain_kernel<DIM><<<(unsigned)((n + 7) / 8), 256, 0, s>>>(g, eA, eB, eF, estat, d_err, refA, refB, cclass,
                                                                 buf + 2, buf);
    note_launches(1);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) {
    auto kern = cell_moments_kernel<DIM>;
    const size_t sm = sizeof(MomShared<DIM>);
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    // CTAs take listed cells from a counter: enough of them to fill the GPU
    const long long grid = n < 152LL * 8 ? n : 152LL * 8;
    if (e == cudaSuccess) {
      kern<<<(unsigned)grid, 32 << DIM, sm, s>>>(g, eA, eB, eF, estat, d_err, refA, refB, cclass, cells,
                                               refA ? buf + 2 : nullptr, buf, buf + 1, n);
      note_launches(1);
      e = cudaGetLastError();
    }
  }
  const cudaError_t f = cudaFreeAsync(buf, s);
  return e != cudaSuccess ? e : f;
}

template <int DIM>
void run_elements_q2(const LevelGeom& g, double* eA, double* eB, double* eF, double* estat, unsigned* d_err,
                     cudaStream_t s) {
  constexpr int W = Entries<DIM>::WARPS;
  cell_elements_q2_kernel<DIM><<<(unsigned)((g.ncell + W - 1) / W), W * 32, 0, s>>>(g, eA, eB, eF, estat, d_err);
}

}  // namespace

cudaError_t launch_cell_elements(const LevelGeom& g, double* eA, double* eB, double* eF,
                                 double* estat, unsigned* d_err, const double* refA, const double* refB,
                                 unsigned char* cclass, cudaStream_t s) {
  return g.dim == 2 ? run_moments<2>(g, eA, eB, eF, estat, d_err, refA, refB, cclass, nullptr, 0, s)
                    : run_moments<3>(g, eA, eB, eF, estat, d_err, refA, refB, cclass, nullptr, 0, s);
}

cudaError_t launch_cell_elements_list(const LevelGeom& g, const long long* cells, long long ncells, double* eA,
                                      double* eB, double* eF, unsigned* d_err, cudaStream_t s) {
  return g.dim == 2 ? run_moments<2>(g, eA, eB, eF, nullptr, d_err, nullptr, nullptr, nullptr, cells, ncells, s)
                    : run_moments<3>(g, eA, eB, eF, nullptr, d_err, nullptr, nullptr, nullptr, cells, ncells, s);
}

cudaError_t launch_cell_elements_q2(const LevelGeom& g, double* eA, double* eB, double* eF, double* estat,
                                    unsigned* d_err, cudaStream_t s) {
  if (g.dim == 2) run_elements_q2<2>(g, eA, eB, eF, estat, d_err, s);
  else run_elements_q2<3>(g, eA, eB, eF, estat, d_err, s);
  note_launches(1);
  return cudaGetLastError();
}

}  // namespace fc
