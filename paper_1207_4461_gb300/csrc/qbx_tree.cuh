// qbx_tree.cuh -- cluster moments of the sources and their evaluation through
// the truncated expansions of distant centres.
//
// The truncated Graf sum about a centre c is linear in the source field, so
// the sources of a cluster (a run of leaves inside a disc of radius R about
// z) may be replaced, for every centre c whose disc keeps away from theirs,
// by the cluster's outgoing expansion u(y) = sum_m M_m H_m(k|y-z|) e^{im arg(y-z)}
// (the addition theorem, Sec. 2 eq. graf-addition with the roles of source and
// centre exchanged): with V = c - z = D e^{iTheta},
//   H_m(k|y-z|) e^{im arg(y-z)} = sum_l H_{m-l}(kD) e^{i(m-l)Theta} J_l(k|y-c|) e^{il arg(y-c)},
// of which the centre keeps |l| <= p.  The result is the same truncated sum
// G_p (Sec. 2, eq. qbx-kernel) as pair by pair; only the cluster's series in m
// is cut, where its terms fall below kTreeTol of the kernel (series_order).
// Per (centre, cluster) that is (P+1) p products instead of p products for
// each of the cluster's 64, 128, 256, ... sources.
//
// Clusters: node (lev, j) holds leaves [j 2^lev, (j+1) 2^lev), a leaf half a
// panel.  Targets come in blocks of 32 consecutive nodes; for every block
// k_tree_lists names the highest nodes that are far enough from all its
// centres' discs, and the leaves that no such node covers (near leaves: pair
// by pair).
//
// Per target of the 256-panel starfish (p = 12, k = 20, S, D and grad S, both
// sides) this leaves about 4.4 panels of pairs of 256 (146k FP64 instructions
// of 8.5M), 9 nodes taken centre by centre and 33 gathered into the block's
// local expansion (150k), most of these for several blocks at once
// (k_tree_super).  The apply: 63.2 ms -> 3.2 ms; k = 20 + 1i at 128 panels
// 26.9 -> 3.4 ms; S and D at 32 panels, p = 8: 751 -> 336 us.
// The pair route stays for fewer than kTreeMinPanels panels (nothing is far),
// for workspaces without room for the arrays below, and where the clusters'
// chain of launches is not repaid: by pairs, columns, sources per leaf and
// operators, with both sides measured, at the calls (qbx_capi.cu: applies of
// many columns, stored coefficients, points off the curve; qbx_batch.cu,
// qbx_adjoint.cu, qbx_shape.cu; matrix_tree_setup for the assembled matrix).
#pragma once
#include <cuda_runtime.h>
#include "qbx_apply_impl.cuh"
#include "qbx_internal.h"

namespace qbx {

// Terms below this fraction of the kernel are left out: half a unit in the
// last place of the result, below the rounding of a single kernel value.
constexpr float kTreeTol = 5e-17f;

// Order at which a Graf series of inner radius R (k R = kr) and outer
// distance rho (k rho = z; q = R / rho) may be cut: the terms beyond it, with
// nd derivatives on the inner side, add up to less than kTreeTol of
// |H_nd(z)|.  |J_l(kr)| <= (kr/2)^l/l! e^{Im} (DLMF 10.14.4); |H_l| by its
// recurrence with absolute values.  damp = e^{2 Im k R}.  FP32: an estimate,
// on the safe side by an order or so.  Returns limit + 1 when limit orders do
// not do.
__device__ __forceinline__ int series_order(float kr, float z, float q, float damp, int nd, int limit) {
  if (!(q < 0.75f)) return limit + 1;   // (NaN too)
  const float a = 0.5f * kr, iz = 1.0f / z;
  // <= |H_nd/H0| (|H_1/H_0| > 1/(2 z (1 + log(1 + 1/z))), |H_2/H_0| > 1/(z^2 (1 + log(1 + 1/z))))
  const float qlo = fmaxf(1.0f, (nd == 2 ? iz * iz : 0.5f * iz) / (1.0f + log1pf(iz)));
  const float fac = 2.0f * damp / (1.0f - q), dw = nd == 2 ? 1.0f / (kr * kr * qlo) : nd ? 1.0f / (kr * qlo) : 1.0f;
  float g0 = 1.0f, g1 = a * (1.0f + iz);
  int last = 0;
  for (int l = 1; l <= limit + 1; ++l) {
    const float w = g1 * fac * (nd == 2 ? (float)(l * l) * dw : nd ? (float)l * dw : 1.0f);
    if (!(w <= kTreeTol)) last = l;
    const float g2 = __fdividef(a, (float)(l + 1)) * (2.0f * l * iz * g1 + __fdividef(a, (float)l) * g0);
    g0 = g1;
    g1 = g2;
  }
  return last;
}

__device__ __forceinline__ double neg_if(bool neg, double v) {
  return __hiloint2double(__double2hiint(v) ^ (neg ? 0x80000000 : 0), __double2loint(v));
}
__device__ __forceinline__ cplx neg_if(bool neg, cplx v) {   // on the integer pipe
  const int m = neg ? 0x80000000 : 0;
  return cplx{__hiloint2double(__double2hiint(v.re) ^ m, __double2loint(v.re)),
              __hiloint2double(__double2hiint(v.im) ^ m, __double2loint(v.im))};
}

}  // namespace qbx
