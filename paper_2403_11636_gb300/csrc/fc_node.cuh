// fc_node.cuh -- the FP64 products of one node or patch, shared by the kernels
// that run them over whole levels (fc_mg.cu, fc_patch.cu) and over the nodes
// that the digit products leave (fc_digits.cu).
#pragma once

#include "fc_internal.cuh"

namespace fc {

// slot geometry of the cached rows: velocity nodes of the 5^d box (x fastest,
// component inner), then the pressures of the 3^d box
template <int DIM>
struct SlotDims {
  static constexpr int NU = DIM == 3 ? 125 : 25, NP = DIM == 3 ? 27 : 9, ND = DIM + 1, NSLOT = NU * DIM + NP;
};

// residual offset of every slot from the patch's node in the padded vector
template <int DIM>
__device__ __forceinline__ void slot_table(const LevelGeom& g, int* soff) {
  using P = SlotDims<DIM>;
  const int px = g.nn[0] + 4, py = g.nn[1] + 4;
  for (int j = threadIdx.x; j < P::NSLOT; j += blockDim.x) {
    // constant divisors: a CTA of few patches pays for its table (8 patches
    // of float32 rows: 0.213 ms per 65^3 launch with `% w`, 0.197 so)
    int o0, o1, o2, c;
    if (j < P::NU * DIM) {
      const int v = j / DIM;
      c = j % DIM;
      o0 = v % 5 - 2;
      o1 = DIM == 3 ? v / 5 % 5 - 2 : v / 5 - 2;
      o2 = DIM == 3 ? v / 25 - 2 : 0;
    } else {
      const int v = j - P::NU * DIM;
      c = DIM;
      o0 = v % 3 - 1;
      o1 = DIM == 3 ? v / 3 % 3 - 1 : v / 3 - 1;
      o2 = DIM == 3 ? v / 9 - 1 : 0;
    }
    soff[j] = (o0 + px * (o1 + py * o2)) * P::ND + c;
  }
  __syncthreads();
}

template <int DIM>
__device__ __forceinline__ void decode_node(const LevelGeom& g, unsigned i, int* ia) {
  // 32-bit: 64-bit division would run on the slow FP64 pipe
  const unsigned nx = (unsigned)g.nn[0], ny = (unsigned)g.nn[1];
  const unsigned t = i / nx;
  ia[0] = (int)(i - t * nx);
  if (DIM == 3) {
    const unsigned u = t / ny;
    ia[1] = (int)(t - u * ny);
    ia[2] = (int)u;
  } else {
    ia[1] = (int)t;
    ia[2] = 0;
  }
}

// Row loads: rows shared by a class of patches stay in the caches; a
// patch's own rows are read once per sweep and streamed past L2.
template <typename V>
__device__ __forceinline__ V ldrow(const V* p, bool cached) {
  return cached ? __ldg(p) : __ldcs(p);
}

// Restricted prolongation R~_i^T for the apply kernels: lane c < d+1
// updates component c of node i from the warp-reduced y (all lanes hold the
// sums); constrained velocity components take the residual (identity row).
// x2, when given, receives the (hi, lo) float pair of the new value.
template <int ND>
__device__ __forceinline__ void owned_update(unsigned i, int lane, const unsigned char* mask, double rcv,
                                             double yv, double omega, double* x, float2* x2) {
  if (lane >= ND) return;
  const int c = lane;
  const size_t k = (size_t)i * ND + c;
  const bool fixed = c < ND - 1 && ((mask[i] >> c) & 1);
  const double nv = x[k] + (fixed ? rcv : omega * yv);
  x[k] = nv;
  if (x2) {
    float hi = (float)nv;
    x2[k] = make_float2(hi, (float)(nv - (double)hi));
  }
}

template <int N, typename T>
__device__ __forceinline__ T pick(const T* v, int c) {
  T r = v[0];
#pragma unroll
  for (int k = 1; k < N; ++k)
    if (c == k) r = v[k];
  return r;
}

// FP64 patch apply of patch i by a group of TPP lanes: y = Inv_i r_i, then
// x[node i] += omega y.  Groups past the last patch (valid false) take part in
// the shuffles of their warp; i is any patch for them.
template <int DIM, int TPP>
__device__ __forceinline__ void apply_fp64_patch(const LevelGeom& g, const double* __restrict__ coef,
                                                 const unsigned char* __restrict__ mask,
                                                 const double* __restrict__ rpad, double omega,
                                                 double* __restrict__ x, const int* __restrict__ prow,
                                                 const int* soff, unsigned i, bool valid) {
  using P = SlotDims<DIM>;
  constexpr int ND = P::ND, NSLOT = P::NSLOT;
  const int lane = threadIdx.x % TPP;
  int ia[3];
  decode_node<DIM>(g, i, ia);
  const long long pbase = pad_node(g, ia[0], ia[1], ia[2]);
  const double* rp = rpad + pbase * ND;
  const int pr = prow ? prow[i] : (int)i;
  const bool shared_rows = pr < 0;  // class rows: read through the cache
  const double* cf = coef + (size_t)(shared_rows ? -pr - 1 : pr) * NSLOT * ND;
  double y[4] = {0.0, 0.0, 0.0, 0.0};  // 2D: y[3] stays zero
  // Live velocity slots.  Slots of out-of-grid nodes and of wall layers
  // (every velocity component constrained) have zero coefficients; in 3D the
  // 5 x 5 x 5 velocity box is clipped per direction to its live layers
  // [x0, x1] x [y0, y1] x [z0, z1]: a patch walks rows of rx = 3 (x1 - x0 + 1)
  // contiguous slots (a y row of a z-plane holds 15), ny rows per z-plane,
  // nz planes, then its 3^d pressure slots.  Patches of a warp are
  // consecutive nodes of an x row and mostly share the clipping.
  int nv = P::NU * DIM, rx = nv, ny = 1, vbase = 0;  // unclipped: one run of all velocity slots
  if (DIM == 3 && g.dead_layer) {
    const unsigned char* dx = g.dead_layer;
    const unsigned char* dy = dx + g.nn[0];
    const unsigned char* dz = dy + g.nn[1];
    int x0 = -2, x1 = 2, y0 = -2, y1 = 2, z0 = -2, z1 = 2;
    while (x0 <= 2 && (ia[0] + x0 < 0 || ia[0] + x0 > g.n[0] || dx[ia[0] + x0])) ++x0;
    while (x1 >= x0 && (ia[0] + x1 < 0 || ia[0] + x1 > g.n[0] || dx[ia[0] + x1])) --x1;
    while (y0 <= 2 && (ia[1] + y0 < 0 || ia[1] + y0 > g.n[1] || dy[ia[1] + y0])) ++y0;
    while (y1 >= y0 && (ia[1] + y1 < 0 || ia[1] + y1 > g.n[1] || dy[ia[1] + y1])) --y1;
    while (z0 <= 2 && (ia[2] + z0 < 0 || ia[2] + z0 > g.n[2] || dz[ia[2] + z0])) ++z0;
    while (z1 >= z0 && (ia[2] + z1 < 0 || ia[2] + z1 > g.n[2] || dz[ia[2] + z1])) --z1;
    rx = 3 * (x1 - x0 + 1);
    ny = y1 - y0 + 1;
    nv = x1 >= x0 && y1 >= y0 && z1 >= z0 ? rx * ny * (z1 - z0 + 1) : 0;
    vbase = (z0 + 2) * 75 + (y0 + 2) * 15 + (x0 + 2) * 3;
  }
  // a patch whose node has every velocity component constrained owns only
  // its pressure: its velocity rows are zero and only row d is summed
  const bool wall = DIM == 3 && (mask[i] & 7) == 7;
  const int tot = nv + P::NP;
  int zi = 0, yi = 0, o = lane;  // loop index t = (zi ny + yi) rx + o while t < nv
  if (nv > 0)
    while (o >= rx) {
      o -= rx;
      if (++yi == ny) { yi = 0; ++zi; }
    }
  if (DIM == 3 && wall) {
    for (int t = lane; t < tot; t += TPP) {
      const int j = t < nv ? vbase + zi * 75 + yi * 15 + o : P::NU * DIM + (t - nv);
      if (nv > 0) {
        o += TPP;
        while (o >= rx) {
          o -= rx;
          if (++yi == ny) { yi = 0; ++zi; }
        }
      }
      y[ND - 1] += ldrow(cf + (size_t)j * ND + (ND - 1), shared_rows) * rp[soff[j]];
    }
  } else {
#pragma unroll 4
    for (int t = lane; t < tot; t += TPP) {
      const int j = t < nv ? vbase + zi * 75 + yi * 15 + o : P::NU * DIM + (t - nv);
      if (nv > 0) {
        o += TPP;
        while (o >= rx) {
          o -= rx;
          if (++yi == ny) { yi = 0; ++zi; }
        }
      }
      double rv = rp[soff[j]];
      if (ND == 4) {
        const double2* c2 = reinterpret_cast<const double2*>(cf + (size_t)j * 4);
        double2 a = ldrow(c2, shared_rows), b = ldrow(c2 + 1, shared_rows);
        y[0] += a.x * rv; y[1] += a.y * rv; y[2] += b.x * rv; y[3] += b.y * rv;
      } else {
#pragma unroll
        for (int k = 0; k < ND; ++k) y[k] += ldrow(cf + (size_t)j * ND + k, shared_rows) * rv;
      }
    }
  }
  if constexpr (TPP >= 4) {
    // the lane whose group-lane bits below TPP/4 are zero writes component c
    int c = 0;
    const double yc = reduce_scatter4<TPP>(y, lane, &c);
    if (valid && c < ND && (lane & (TPP / 4 - 1)) == 0) owned_update<ND>(i, c, mask, rp[c], yc, omega, x, nullptr);
  } else {
#pragma unroll
    for (int k = 0; k < ND; ++k)
#pragma unroll
      for (int o = TPP / 2; o > 0; o >>= 1) y[k] += __shfl_xor_sync(0xffffffffu, y[k], o);
    if (valid && lane < ND) owned_update<ND>(i, lane, mask, rp[lane], pick<ND>(y, lane), omega, x, nullptr);
  }
}

// ---------------------------------------------------------------------------
// residual / apply of one node by TPP lanes (1, or a group of 4 or 8 of a warp):
// lane l takes the neighbours l, l + TPP, ... of the 3^d blocks of the
// compressed stencil, the d+1 sums are reduce-scattered over the group.  Groups
// past the last node (valid false) take part in the shuffles; node is any node
// for them.  Constrained rows are identity rows and constrained columns are
// skipped (their values live in b).
// OUT: 0 -> r (unpadded, optional) and rpad (padded, optional) in float64,
//      1 -> rpad as float32 pairs (hi, lo), 2 -> rpad as float32.
template <int DIM, int OUT, int TPP>
__device__ __forceinline__ void residual_node(const LevelGeom& g, const double* __restrict__ st,
                                              const unsigned char* __restrict__ mask, const double* __restrict__ x,
                                              const double* __restrict__ b, double* __restrict__ r,
                                              double* __restrict__ rpad, float* __restrict__ rpadf, long long node,
                                              bool valid) {
  constexpr int NB = DIM == 3 ? 27 : 9, SP = 2 * DIM + 2, ND = DIM + 1;
  const int lane = TPP == 1 ? 0 : threadIdx.x % TPP;
  int ia[3];
  decode_node<DIM>(g, (unsigned)node, ia);
  double acc[4] = {0.0, 0.0, 0.0, 0.0};  // 2D: acc[3] stays zero
#pragma unroll
  for (int k = 0; k < (NB + TPP - 1) / TPP; ++k) {
    const int nb = k * TPP + lane;
    if (TPP > 1 && nb >= NB) continue;
    const int ib0 = ia[0] + nb % 3 - 1, ib1 = ia[1] + (nb / 3) % 3 - 1, ib2 = DIM == 3 ? ia[2] + nb / 9 - 1 : 0;
    if (ib0 < 0 || ib0 > g.n[0] || ib1 < 0 || ib1 > g.n[1]) continue;
    if (DIM == 3 && (ib2 < 0 || ib2 > g.n[2])) continue;
    const long long bn = ib0 + (long long)g.nn[0] * (ib1 + (long long)g.nn[1] * ib2);
    const unsigned char mb = mask[bn];
    double xb[ND];
#pragma unroll
    for (int c = 0; c < ND; ++c) xb[c] = x[bn * ND + c];
#pragma unroll
    for (int c = 0; c < DIM; ++c)
      if ((mb >> c) & 1) xb[c] = 0.0;
    const double* s = st + (long long)nb * SP * g.nnodes + node;
    const double vA = s[0];
#pragma unroll
    for (int c = 0; c < DIM; ++c) {
      acc[c] = acc[c] + vA * xb[c];
      acc[c] = acc[c] + s[(1 + c) * g.nnodes] * xb[DIM];
    }
#pragma unroll
    for (int c = 0; c < DIM; ++c) acc[DIM] = acc[DIM] + s[(1 + DIM + c) * g.nnodes] * xb[c];
    acc[DIM] = acc[DIM] + s[(1 + 2 * DIM) * g.nnodes] * xb[DIM];
  }
  const unsigned char ma = mask[node];
  const long long pn = pad_node(g, ia[0], ia[1], ia[2]);
  auto store = [&](int c, double sum) {
    const double y = (c < DIM && ((ma >> c) & 1)) ? x[node * ND + c] : sum;
    const double v = b ? b[node * ND + c] - y : y;
    if (OUT == 0) {
      if (r) r[node * ND + c] = v;
      if (rpad) rpad[pn * ND + c] = v;
    } else if (OUT == 1) {
      const float hi = (float)v;
      rpadf[(pn * ND + c) * 2 + 0] = hi;
      rpadf[(pn * ND + c) * 2 + 1] = (float)(v - (double)hi);
    } else {
      rpadf[pn * ND + c] = (float)v;
    }
  };
  if constexpr (TPP == 1) {
    if (!valid) return;
#pragma unroll
    for (int c = 0; c < ND; ++c) store(c, acc[c]);
  } else {
    int c = 0;
    const double sum = reduce_scatter4<TPP>(acc, lane, &c);
    if (valid && c < ND && (lane & (TPP / 4 - 1)) == 0) store(c, sum);
  }
}

}  // namespace fc
