// qbx_tree.cu -- cluster moments (qbx_tree.cuh): nodes, block lists, moments,
// and the far sums of the fused apply.
#include <cuda_runtime.h>
#include <algorithm>
#include "qbx_tree.cuh"

namespace qbx {
namespace {

__device__ __forceinline__ float warp_min(float v) {
  for (int o = 16; o > 0; o >>= 1) v = fminf(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}
__device__ __forceinline__ float warp_max(float v) {
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}
__device__ __forceinline__ float block_reduce_max(float v, float* s, int n_warps) {
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  __syncthreads();
  if ((threadIdx.x & 31) == 0) s[threadIdx.x >> 5] = v;
  __syncthreads();
  v = s[0];
  for (int w = 1; w < n_warps; ++w) v = fmaxf(v, s[w]);
  return v;
}

// Nodes: about the centre of the bounding box of the node's points, and (a bit
// more than) the largest distance from it.  One CTA per node; the points
// relative to the node's first one in FP32 (the centre may be any point, its
// radius has to hold for it), so the FP64 pipe sees four subtractions a point.
__global__ void __launch_bounds__(256) k_tree_nodes(TreeArgs a) {
  __shared__ float s_red[8];
  const int id = blockIdx.x;
  int l = 0;
  while (id >= a.off[l + 1]) ++l;
  const int j = id - a.off[l];
  const int s0 = (j << l) * a.q_src, s1 = min(a.M, (j + 1) << l) * a.q_src;
  const double x0 = a.sx[s0], y0 = a.sy[s0];
  float xa = 0.0f, xb = 0.0f, ya = 0.0f, yb = 0.0f, bad = 0.0f;   // max of -x, x, -y, y
  for (int s = s0 + threadIdx.x; s < s1; s += 256) {
    const float x = (float)(a.sx[s] - x0), y = (float)(a.sy[s] - y0);
    if (!(fabsf(x) < 1e30f && fabsf(y) < 1e30f)) bad = 1.0f;   // a node with such a point is never far
    xa = fmaxf(xa, -x);
    xb = fmaxf(xb, x);
    ya = fmaxf(ya, -y);
    yb = fmaxf(yb, y);
  }
  xa = block_reduce_max(xa, s_red, 8);
  xb = block_reduce_max(xb, s_red, 8);
  ya = block_reduce_max(ya, s_red, 8);
  yb = block_reduce_max(yb, s_red, 8);
  bad = block_reduce_max(bad, s_red, 8);
  const double zx = x0 + (double)(0.5f * (xb - xa)), zy = y0 + (double)(0.5f * (yb - ya));
  float r = 0.0f;
  for (int s = s0 + threadIdx.x; s < s1; s += 256) {
    const float dx = (float)(a.sx[s] - zx), dy = (float)(a.sy[s] - zy);
    r = fmaxf(r, fmaf(dx, dx, dy * dy));
  }
  r = block_reduce_max(r, s_red, 8);
  if (threadIdx.x == 0) {
    double* n = a.node + 4 * (size_t)id;
    n[0] = zx;
    n[1] = zy;
    n[2] = bad > 0.0f ? INFINITY : (double)(sqrtf(r) * 1.00001f);
    n[3] = 0.0;
  }
}

// Lists: one CTA per block of 32 targets, one thread per leaf.  A leaf's
// thread looks from the largest node down for the first that is far from the
// block; the first leaf of that node names it.  In leaf order, so the sums
// do not depend on timing.
constexpr int kListWarps = 8;
__global__ void __launch_bounds__(32 * kListWarps) k_tree_lists(TreeArgs a) {
  __shared__ float s_c[64][3];                   // the centres (both sides) from the block's centre, their radii
  __shared__ double s_z[2];
  __shared__ float s_blk[3];                     // radius of all discs about it; largest, smallest radius
  __shared__ int s_n[kListWarps][3], s_at[3], s_ord[2];   // per warp / so far: near, far, local; largest local orders
  const int b = blockIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int nc = 32 * (a.n_ctr / a.n_tgt);
  if (warp == 0) {
    const int t = min(b * 32 + lane, a.n_tgt - 1);
    const double x0 = a.tx[b * 32], y0 = a.ty[b * 32];
    const float x = (float)(a.tx[t] - x0), y = (float)(a.ty[t] - y0);
    const float xa = warp_max(-x), xb = warp_max(x), ya = warp_max(-y), yb = warp_max(y);
    const double bx = x0 + (double)(0.5f * (xb - xa)), by = y0 + (double)(0.5f * (yb - ya));
    float rd = 0.0f, rm = 0.0f, rn = INFINITY;
    bool bad = false;
    for (int c = t, i = lane; c < a.n_ctr; c += a.n_tgt, i += 32) {
      const float ex = (float)(a.tx[t] - a.cx[c]), ey = (float)(a.ty[t] - a.cy[c]);
      const float r = sqrtf(fmaf(ex, ex, ey * ey)) * 1.00001f;
      const float ox = (float)(a.cx[c] - bx), oy = (float)(a.cy[c] - by);
      s_c[i][0] = ox;
      s_c[i][1] = oy;
      s_c[i][2] = r;
      const float rr = sqrtf(fmaf(ox, ox, oy * oy)) + r;
      bad |= !(rr < 1e30f);
      rd = fmaxf(rd, rr);
      rm = fmaxf(rm, r);
      rn = fminf(rn, r * 0.99998f);
    }
    rd = warp_max(rd) * 1.00001f;
    rm = warp_max(rm);
    rn = warp_min(rn);
    bad = __any_sync(0xffffffffu, bad);
    if (lane == 0) {
      s_z[0] = bx;
      s_z[1] = by;
      s_blk[0] = bad ? INFINITY : rd;   // (no node is far from such a block)
      s_blk[1] = bad ? INFINITY : rm;
      s_blk[2] = rn;
      s_at[0] = s_at[1] = s_at[2] = s_ord[0] = s_ord[1] = 0;
      double* n = a.node + 4 * (size_t)(a.off[a.lev] + b);   // the block's own entry: centre of its local expansion
      n[0] = bx;
      n[1] = by;
      n[2] = rd;
      n[3] = 0.0;
    }
  }
  __syncthreads();
  const double bx = s_z[0], by = s_z[1];
  const float rd = s_blk[0], rm = s_blk[1], rn = s_blk[2];
  const float ka = (float)sqrt(a.kre * a.kre + a.kim * a.kim), ki = (float)a.kim;
  int* near = a.near + (size_t)b * a.M;
  int2* far = reinterpret_cast<int2*>(a.far) + (size_t)b * (a.M + 1);
  int2* loc = reinterpret_cast<int2*>(a.loc) + (size_t)b * a.M;

  // orders (cluster | centre << 8 | block << 16; block 0: not through the
  // block's local expansion) and bit 24 if the node is far from the block, else 0
  auto test = [&](int id) -> int {
    const double* n = a.node + 4 * (size_t)id;
    const float dx = (float)(n[0] - bx), dy = (float)(n[1] - by), R = (float)n[2] * 1.00001f;
    const float d = sqrtf(fmaf(dx, dx, dy * dy));
    if (!(d > R)) return 0;
    // the two ends of the block on both sides first: most nodes fail there
    float du = INFINITY;
    for (int i = 0; i < nc; i += 31 - (i & 1) * 30) {
      const float vx = dx - s_c[i][0], vy = dy - s_c[i][1];
      du = fminf(du, sqrtf(fmaf(vx, vx, vy * vy)) - s_c[i][2]);
    }
    if (!(du > 1.34f * R)) return 0;
    const float damp = expf(2.0f * ki * R);
    if (series_order(ka * R, ka * du, R / du, damp, a.nd, kTreeP) > kTreeP) return 0;
    float dm = INFINITY, rho = INFINITY, dx1 = 0.0f;   // nearest disc point, nearest and farthest centre
    for (int i = 0; i < nc; ++i) {
      const float vx = dx - s_c[i][0], vy = dy - s_c[i][1];
      const float v = sqrtf(fmaf(vx, vx, vy * vy));
      dm = fminf(dm, v - s_c[i][2]);
      rho = fminf(rho, v);
      dx1 = fmaxf(dx1, v);
    }
    dm = 0.99999f * dm;             // nearest point of a centre's disc to the node's centre
    rho = 0.99999f * (rho - R);     // nearest source to a centre
    if (!(dm > 1.34f * R) || !(rho > 1.34f * rm)) return 0;
    const int om = series_order(ka * R, ka * dm, R / dm, damp, a.nd, kTreeP);
    if (om > kTreeP) return 0;
    int ol = series_order(ka * rm, ka * rho, rm / rho, expf(2.0f * ki * rm), a.nd, a.pl);
    // local expansion about the block's centre, good in all its discs
    const float dl = 0.99999f * (d - R);
    int oq = dl > 1.34f * rd ? series_order(ka * rd, ka * dl, rd / dl, expf(2.0f * ki * rd), a.nd, kTreeP) : kTreeP + 1;
    if (oq > kTreeP) oq = 0;
    if (a.eta > 0.0) {
      // every pair by the smooth rule (an expansion of enough orders at the
      // centre gives its value), or every pair through the expansion
      const float eta = (float)a.eta;
      if (rho >= 1.00001f * eta * rm) {
        if (ol > a.pl) return 0;
      } else if (dx1 + R < 0.99999f * eta * rn) {
        ol = min(ol, a.p);
        oq = 0;   // (the block's local expansion holds smooth-rule sources only)
      } else {
        return 0;
      }
    } else {
      ol = min(ol, a.p);
    }
    // H of order om + ol and the moments of order om stay in FP64's range
    const float no = (float)(om + max(ol, oq));
    if (!(no * log10f(fmaxf(2.0f * no / (2.7f * ka * dm), 1.0f)) < 280.0f) ||
        !((float)om * log10f(fmaxf(2.0f * om / (2.7f * ka * R), 1.0f)) < 280.0f))
      return 0;
    return om | ol << 8 | oq << 16 | 1 << 24;
  };

  for (int base = 0; base < a.M; base += 32 * kListWarps) {
    const int j = base + threadIdx.x;
    int code = 0, l = a.lev - 1;
    if (j < a.M) {
      for (; l >= 0; --l) {
        code = test(a.off[l] + (j >> l));
        if (code) break;
      }
    }
    const bool is_near = j < a.M && !code;
    const bool is_node = code && (j & ((1 << l) - 1)) == 0, has_loc = (code >> 16 & 0xff) > 0;
    const bool is_far = is_node && !has_loc, is_loc = is_node && has_loc;
    const unsigned below = (1u << lane) - 1;
    const unsigned mn = __ballot_sync(0xffffffffu, is_near), mf = __ballot_sync(0xffffffffu, is_far),
                   ml = __ballot_sync(0xffffffffu, is_loc);
    if (lane == 0) {
      s_n[warp][0] = __popc(mn);
      s_n[warp][1] = __popc(mf);
      s_n[warp][2] = __popc(ml);
    }
    if (is_loc) {
      atomicMax(&s_ord[0], code >> 16 & 0xff);
      atomicMax(&s_ord[1], code >> 8 & 0xff);
    }
    __syncthreads();
    int an = s_at[0], af = s_at[1], al = s_at[2];
    for (int w = 0; w < warp; ++w) {
      an += s_n[w][0];
      af += s_n[w][1];
      al += s_n[w][2];
    }
    const int id = a.off[max(l, 0)] + (j >> max(l, 0));
    if (is_near) near[an + __popc(mn & below)] = j;
    if (is_far) far[af + __popc(mf & below)] = make_int2(id, code & 0xffff);
    if (is_loc) loc[al + __popc(ml & below)] = make_int2(id, (code & 0xff) | (code >> 16 & 0xff) << 8);
    __syncthreads();
    if (threadIdx.x < 3)
      for (int w = 0; w < kListWarps; ++w) s_at[threadIdx.x] += s_n[w][threadIdx.x];
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    int nf = s_at[1];
    if (s_at[2] > 0)   // the block's local expansion, after the far nodes
      far[nf++] = make_int2(a.off[a.lev] + b, s_ord[0] | s_ord[1] << 8 | 1 << 16);
    a.cnt[3 * b] = s_at[0];
    a.cnt[3 * b + 1] = nf;
    a.cnt[3 * b + 2] = s_at[2];
  }
}

// Moments of one leaf about the centre of one of its nodes (blockIdx = leaf,
// level): with C_m = J_m(k rho) cos(m theta), S_m = J_m(k rho) sin(m theta) of
// the source's position about it,
//   A_m = sum_s w_s C_m, B_m = sum_s w_s S_m  (dipoles: their derivatives along
//   the source's direction, (k/2)(C_{m-1} - C_{m+1}) along x and so on),
// the coefficients of H_m cos(m Theta) and H_m sin(m Theta) (the factor 2 of
// m > 0 in k_tree_fold).  Phase 1: one thread per source forms its columns in
// shared memory; phase 2: one thread per (set, rhs, m) sums over the sources.
template <typename T>
__global__ void __launch_bounds__(128) k_tree_moments(TreeArgs a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int q = a.q_src, Q = q | 1, P = kTreeP;
  T* sC = reinterpret_cast<T*>(smem_raw);    // [P + 3][Q]
  T* sS = sC + (P + 3) * Q;
  const int panel = blockIdx.x, l = blockIdx.y;
  const double* n = a.node + 4 * (size_t)(a.off[l] + (panel >> l));
  const double zx = n[0], zy = n[1];
  KW<T> kw;
  kw.init(a.kre, a.kim, a.hk_tab);
  const T kk = kw.kval();
  const float kr = (float)sc_abs(kk) * (float)n[2];   // orders at any distance beyond kTreeP: in no list
  if (!(kr < 64.0f) || series_order(kr, 1e4f * kr + 1e4f, 1e-4f, 1.0f, 0, kTreeP) > kTreeP) return;
  for (int i = threadIdx.x; i < q; i += 128) {
    const double dx = a.sx[panel * q + i] - zx, dy = a.sy[panel * q + i] - zy;
    const double rho = sqrt(dx * dx + dy * dy);
    besselj_column<T>(rmul(kk, rho), P + 2, sC + i, Q);
    const double cs = rho > 0.0 ? dx / rho : 1.0, sn = rho > 0.0 ? dy / rho : 0.0;
    double c = 1.0, s = 0.0;
    for (int m = 0; m <= P + 2; ++m) {
      const T j = sC[m * Q + i];
      sC[m * Q + i] = rmul(j, c);
      sS[m * Q + i] = rmul(j, s);
      const double cn = fma(c, cs, -s * sn);
      s = fma(s, cs, c * sn);
      c = cn;
    }
  }
  __syncthreads();
  const int ncol = a.nset * a.nrhs;
  cplx* out = reinterpret_cast<cplx*>(a.mom) + (size_t)(l * a.M + panel) * ncol * (P + 2) * 2;
  const T hk = rmul(kk, 0.5);
  for (int e = threadIdx.x; e < ncol * (P + 2); e += 128) {
    const int col = e / (P + 2), m = e - col * (P + 2);
    const int set = col / a.nrhs, r = col - set * a.nrhs, kind = a.kind[set];
    const cplx* w = reinterpret_cast<const cplx*>(a.wd[set]) + (size_t)panel * q * a.nrhs + r;
    cplx A{0.0, 0.0}, B{0.0, 0.0};
    if (kind == kSetMono) {
      for (int i = 0; i < q; ++i) {
        madd(A, sC[m * Q + i], w[(size_t)i * a.nrhs]);
        madd(B, sS[m * Q + i], w[(size_t)i * a.nrhs]);
      }
    } else {
      const double* px = a.snx + (size_t)panel * q;
      const double* py = a.sny + (size_t)panel * q;
      const int mm = m > 0 ? m - 1 : 1;
      const double sg = m > 0 ? 1.0 : -1.0;   // C_{-1} = -C_1, S_{-1} = S_1
      for (int i = 0; i < q; ++i) {
        const double nx = kind == kSetNormal ? px[i] : kind == kSetX ? 1.0 : 0.0;
        const double ny = kind == kSetNormal ? py[i] : kind == kSetY ? 1.0 : 0.0;
        const T cm = rmul(sC[mm * Q + i], sg), cp = sC[(m + 1) * Q + i];
        const T sm = sS[mm * Q + i], sp = sS[(m + 1) * Q + i];
        const cplx v = w[(size_t)i * a.nrhs];
        madd(A, sc_sub(rmul(sc_sub(cm, cp), nx), rmul(sadd(sm, sp), ny)), v);
        madd(B, sadd(rmul(sc_sub(sm, sp), nx), rmul(sadd(cm, cp), ny)), v);
      }
      A = smul(hk, A);
      B = smul(hk, B);
    }
    out[(size_t)e * 2] = A;
    out[(size_t)e * 2 + 1] = B;
  }
}

// The coefficient columns of one node or local expansion from its moments
// [col][m][2] (m <= n): column set i is moment set `base`, itself or its
// derivative along x or y (the series of d/dx u has the coefficients
//   A^x_m = (k/2)(A_{m+1} - A_{m-1}), B^x_m = (k/2)(B_{m+1} - B_{m-1}),
//   A^y_m = (k/2)(B_{m+1} + B_{m-1}), B^y_m = -(k/2)(A_{m+1} + A_{m-1}),
// A_0 counted twice).
__device__ __forceinline__ void shifted_coef(const TreeArgs& a, int set, const cplx* mom, int stride, int n, int m,
                                             cplx* out) {
  auto at = [&](int i, int ab) {
    if (i < 0 || i > n) return cplx{0.0, 0.0};
    return mom[i * stride + ab];
  };
  const int sh = a.shift[set];
  if (sh == 0) {
    out[0] = at(m, 0);
    out[1] = at(m, 1);
    return;
  }
  const cplx hk{0.5 * a.kre, 0.5 * a.kim};
  const double f = m == 1 ? 2.0 : 1.0;
  const cplx Ap = at(m + 1, 0), Bp = at(m + 1, 1), Am = f * at(m - 1, 0), Bm = at(m - 1, 1);
  if (sh == 1) {
    out[0] = hk * (Ap - Am);
    out[1] = m ? hk * (Bp - Bm) : cplx{0.0, 0.0};
  } else {
    out[0] = hk * (Bp + Bm);
    out[1] = m ? -(hk * (Ap + Am)) : cplx{0.0, 0.0};
  }
}

// Node coefficients: the leaves' contributions added in leaf order, then the
// columns.  One CTA per (node, moment column).
__global__ void __launch_bounds__(64) k_tree_fold(TreeArgs a) {
  constexpr int N = kTreeP + 2;
  __shared__ cplx s_m[N][2];
  const int id = blockIdx.x, set = blockIdx.y / a.nrhs, r = blockIdx.y - set * a.nrhs;
  int l = 0;
  while (id >= a.off[l + 1]) ++l;
  const int j = id - a.off[l];
  const int p0 = j << l, p1 = min(a.M, (j + 1) << l);
  const int ncol = a.nset * a.nrhs;
  const cplx* mom = reinterpret_cast<const cplx*>(a.mom) + ((size_t)l * a.M * ncol + blockIdx.y) * N * 2;
  for (int i = threadIdx.x; i < N * 2; i += 64) {
    cplx v{0.0, 0.0};
    for (int p = p0; p < p1; ++p) v = v + mom[(size_t)p * ncol * N * 2 + i];
    s_m[i >> 1][i & 1] = (i > 1 ? 2.0 : 1.0) * v;
  }
  __syncthreads();
  for (int i = threadIdx.x; i < a.ncset * (kTreeP + 1); i += 64) {
    const int cs = i / (kTreeP + 1), m = i - cs * (kTreeP + 1);
    if (a.base[cs] != set) continue;
    shifted_coef(a, cs, &s_m[0][0], 2, kTreeP + 1, m,
                 reinterpret_cast<cplx*>(a.coef) + (((size_t)id * (kTreeP + 1) + m) * a.ncset * a.nrhs + cs * a.nrhs + r) * 2);
  }
}

// Local expansions: the nodes that are far from a whole block of targets (its
// radius included) are first gathered into one expansion about the block's
// centre z_b, u = sum_q J_q(k d) [A'_q cos(q phi) + B'_q sin(q phi)], which then
// counts as one more node for the block's centres.  With V = z_b - z of length
// D and direction Theta, s_m = A_m cos(m Theta) + B_m sin(m Theta),
// d_m = i (A_m sin(m Theta) - B_m cos(m Theta)):
//   S_q = sum_m s_m (H_{m-q} + (-1)^q H_{m+q}),  T_q = sum_m d_m (H_{m-q} - (-1)^q H_{m+q}),
//   A'_q = cos(q Theta) S_q - i sin(q Theta) T_q,  B'_q = sin(q Theta) S_q + i cos(q Theta) T_q
// (A'_0 halved).  One warp per node, lane = q: a tenth of the FP64 work of
// taking the node through each of the block's 32 or 64 centres.
constexpr int kLocWarps = 8, kLocCols = 2;   // moment columns per CTA
template <typename T>
__global__ void __launch_bounds__(32 * kLocWarps) k_tree_local(TreeArgs a) {
  constexpr int NC = kLocCols;
  __shared__ cplx s_h[kLocWarps][2 * kTreeP + 2];
  __shared__ cplx s_sd[kLocWarps][2 * NC][32];
  static_assert(kTreeP < 32, "one lane per order");
  const int b = blockIdx.x, col0 = blockIdx.y * NC, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int nc = min(NC, a.nset * a.nrhs - col0);
  int ccol[NC];   // coefficient column of each moment column
#pragma unroll
  for (int c = 0; c < NC; ++c) {
    const int set = min(col0 + c, a.nset * a.nrhs - 1) / a.nrhs;
    ccol[c] = a.plain[set] * a.nrhs + min(col0 + c, a.nset * a.nrhs - 1) - set * a.nrhs;
  }
  const int ncol = a.ncset * a.nrhs;
  const int cnt = a.cnt[3 * b + 2];
  if (cnt == 0) return;
  const double* blk = a.node + 4 * (size_t)(a.off[a.lev] + b);
  const int2* loc = reinterpret_cast<const int2*>(a.loc) + (size_t)b * a.M;
  KW<T> kw;
  kw.init(a.kre, a.kim, a.hk_tab);
  cplx accA[NC], accB[NC];
#pragma unroll
  for (int c = 0; c < NC; ++c) accA[c] = accB[c] = cplx{0.0, 0.0};
  for (int e = warp; e < cnt; e += kLocWarps) {
    const int2 ent = loc[e];
    const int om = ent.y & 0xff, oq = ent.y >> 8;
    const double* nd = a.node + 4 * (size_t)ent.x;
    const double vx = blk[0] - nd[0], vy = blk[1] - nd[1];
    double inv, rho, yq;
    kw.geom(fma(vx, vx, vy * vy), inv, rho, yq);
    cplx h0, h1;
    T twoz;
    kw.hankel(rho, inv, yq, h0, h1, twoz);
    const double ct = vx * inv, st = vy * inv;
    double cl = 1.0, sl = 0.0;   // cos, sin of lane * Theta, by squaring
    {
      double c = ct, s = st;
#pragma unroll
      for (int i = 0; i < 5; ++i) {
        if (lane >> i & 1) {
          const double cn = fma(cl, c, -sl * s);
          sl = fma(sl, c, cl * s);
          cl = cn;
        }
        const double c2 = fma(c, c, -s * s);
        s = 2.0 * c * s;
        c = c2;
      }
    }
    __syncwarp();   // the previous node's tables are no longer read
    if (lane == 0) s_h[warp][0] = h0;
    T s = twoz;
    for (int i = 1; i <= om + oq; ++i) {
      if (lane == 0) s_h[warp][i] = h1;
      const cplx h2 = hrec(s, h1, h0);
      h0 = h1;
      h1 = h2;
      s = sadd(s, twoz);
    }
    if (lane <= om) {
      const double2* co = reinterpret_cast<const double2*>(a.coef) + ((size_t)ent.x * (kTreeP + 1) + lane) * ncol * 2;
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        if (c >= nc) break;
        const double2 A = co[2 * ccol[c]], B = co[2 * ccol[c] + 1];
        s_sd[warp][2 * c][lane] = cplx{fma(A.x, cl, B.x * sl), fma(A.y, cl, B.y * sl)};
        s_sd[warp][2 * c + 1][lane] = cplx{fma(B.y, cl, -A.y * sl), fma(A.x, sl, -B.x * cl)};
      }
    }
    __syncwarp();
    if (lane <= oq) {
      cplx S[NC], D[NC];
#pragma unroll
      for (int c = 0; c < NC; ++c) S[c] = D[c] = cplx{0.0, 0.0};
      for (int m = 0; m <= om; ++m) {
        const int d = m - lane;
        const cplx ha = neg_if(d < 0 && (d & 1), s_h[warp][d < 0 ? -d : d]);
        const cplx hb = neg_if(lane & 1, s_h[warp][m + lane]);
        const cplx hp = ha + hb, hm = ha - hb;
#pragma unroll
        for (int c = 0; c < NC; ++c) {
          if (c >= nc) break;
          cfma(S[c], s_sd[warp][2 * c][m], hp);
          cfma(D[c], s_sd[warp][2 * c + 1][m], hm);
        }
      }
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        // A' += cos S - i sin D, B' += sin S + i cos D
        accA[c] = accA[c] + cplx{fma(cl, S[c].re, sl * D[c].im), fma(cl, S[c].im, -sl * D[c].re)};
        accB[c] = accB[c] + cplx{fma(sl, S[c].re, -cl * D[c].im), fma(sl, S[c].im, cl * D[c].re)};
      }
    }
  }
  // the warps' sums, in warp order
  __shared__ cplx s_sum[2 * NC][32], s_mom[NC][kTreeP + 1][2];
  for (int w = 0; w < kLocWarps; ++w) {
    if (warp == w) {
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        if (w > 0) {
          accA[c] = s_sum[2 * c][lane] + accA[c];
          accB[c] = s_sum[2 * c + 1][lane] + accB[c];
        }
        s_sum[2 * c][lane] = accA[c];
        s_sum[2 * c + 1][lane] = accB[c];
      }
    }
    __syncthreads();
  }
  if (warp == 0 && lane <= kTreeP) {
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      s_mom[c][lane][0] = (lane == 0 ? 0.5 : 1.0) * s_sum[2 * c][lane];
      s_mom[c][lane][1] = lane == 0 ? cplx{0.0, 0.0} : s_sum[2 * c + 1][lane];
    }
  }
  __syncthreads();
  cplx* out = reinterpret_cast<cplx*>(a.coef) + (size_t)(a.off[a.lev] + b) * (kTreeP + 1) * ncol * 2;
  for (int i = threadIdx.x; i < nc * a.ncset * (kTreeP + 1); i += 32 * kLocWarps) {
    const int c = i / (a.ncset * (kTreeP + 1)), rem = i - c * a.ncset * (kTreeP + 1);
    const int cs = rem / (kTreeP + 1), m = rem - cs * (kTreeP + 1);
    const int set = (col0 + c) / a.nrhs, r = col0 + c - set * a.nrhs;
    if (a.base[cs] == set)
      shifted_coef(a, cs, &s_mom[c][0][0], 2, kTreeP, m, out + ((size_t)m * ncol + cs * a.nrhs + r) * 2);
  }
}

// J_0..J_n at z as complex values of stride 32
template <typename T>
__device__ __forceinline__ void besselj_wave(T z, int n, cplx* out) {
  if constexpr (IsCplx<T>::value) {
    besselj_column<cplx>(z, n, out, 32);
  } else {
    besselj_column<double>(z, n, reinterpret_cast<double*>(out), 64);
    for (int i = 0; i <= n; ++i) out[i * 32].im = 0.0;
  }
}

// Shared memory of the far kernel: the centres' J column; per warp H_0.. per
// lane, and per order l the products J_l cos(l psi), J_l sin(l psi).
template <typename T>
__host__ __device__ size_t far_warp_bytes(int pl) {
  return (size_t)(kTreeP + pl + 2) * 32 * 16 + (size_t)pl * 2 * 32 * sizeof(T);
}
template <typename T>
__host__ __device__ size_t far_col_bytes(int pl) {
  return (size_t)(pl + 2) * 32 * sizeof(T);
}

// Far sums: a warp holds 32 centres of one side (one per lane) and takes the
// far nodes of their block in turn.  Per node: H_0..H_{om+ol} at the distance
// from the node's centre z to c, then for every m <= om
//   X_m = J_0 H_m + sum_l J_l cos(l psi) (H_{m-l} + (-1)^l H_{m+l}),
//   Y_m = sum_l J_l sin(l psi) (H_{m-l} - (-1)^l H_{m+l}),   psi = theta_t - Theta,
// the truncated expansion about c of H_m cos(m Theta), H_m sin(m Theta):
//   X cos(m Theta) - Y sin(m Theta),  X sin(m Theta) + Y cos(m Theta),
// times the node's coefficient columns.
// grad S: the derivative of the expansion cut at |l| <= p is the cut expansion
// of the derived columns up to the orders p, p + 1 at the cut,
//   (d_x - i d_y): -(k/2) e^{-i theta_t} [J_p e^{i(p+1) psi} (U_{p+1} + V_{p+1}) + J_{p+1} e^{-i p psi} (U_p - V_p)],
//   (d_x + i d_y): -(k/2) e^{i theta_t} [J_p e^{-i(p+1) psi} (U_{p+1} - V_{p+1}) + J_{p+1} e^{i p psi} (U_p + V_p)],
//   U_l = sum_m s_m (H_{m-l} + (-1)^l H_{m+l}), V_l = sum_m d_m (H_{m-l} - (-1)^l H_{m+l})
// with s_m, d_m of the density's own column as in k_tree_local (32 FP64
// instructions per m instead of 16 per (m, l) for the two derivatives).
// FP64-bound: 8 instructions per (m, l), l up to what order m needs, and 8
// per (m, column).
template <int OPS, typename T, int NR>
__global__ void __launch_bounds__(128) k_far_clusters(TreeArgs a) {
  constexpr bool kS = OPS & OPB_S, kD = OPS & OPB_D, kG = OPS & OPB_G, kX = OPS & OPB_X;
  constexpr int kC = kS + kD + 2 * kG + 2 * kX;   // columns per rhs: S, D, grad S x, y, X x, y
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int p = a.p, pl = a.pl, W = blockDim.x >> 5, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  T* colJ = reinterpret_cast<T*>(smem_raw) + lane;   // [pl + 2][32]
  unsigned char* mine = smem_raw + far_col_bytes<T>(pl) + (size_t)warp * far_warp_bytes<T>(pl);
  cplx* sH = reinterpret_cast<cplx*>(mine) + lane;                                   // [kTreeP + pl + 2][32]
  T* sF = reinterpret_cast<T*>(mine + (size_t)(kTreeP + pl + 2) * 32 * 16) + lane;   // [pl][2][32]

  const int nblk = a.n_blk * (a.n_ctr / a.n_tgt);
  const int unit = (int)(blockIdx.x % (unsigned)nblk), split = (int)(blockIdx.x / (unsigned)nblk);
  const int side = unit / a.n_blk, blk = unit - side * a.n_blk;
  const bool active = blk * 32 + lane < a.n_tgt;
  const int t = active ? blk * 32 + lane : a.n_tgt - 1;
  const int c = side * a.n_tgt + t;
  const double cx = a.cx[c], cy = a.cy[c];
  double ux = a.tx[t] - cx, uy = a.ty[t] - cy;
  const double r = hypot(ux, uy), ir = 1.0 / r;
  ux *= ir;
  uy *= ir;
  KW<T> kw;
  kw.init(a.kre, a.kim, a.hk_tab);
  const T kk = kw.kval();
  if (warp == 0) besselj_column<T>(rmul(kk, r), pl + 1, colJ, 32);
  __syncthreads();
  const T J0 = colJ[0];
  int set[kC];   // coefficient column set of each column
  {
    int i = 0;
    if (kS) set[i++] = a.set_s;
    if (kD) set[i++] = a.set_d;
    if (kG) {
      set[i++] = a.set_gx;
      set[i++] = a.set_gx + 1;
    }
    if (kX) {
      set[i++] = a.set_x;
      set[i++] = a.set_x + 1;
    }
  }
  cplx acc[kC][NR];
#pragma unroll
  for (int q = 0; q < kC; ++q)
#pragma unroll
    for (int i = 0; i < NR; ++i) acc[q][i] = cplx{0.0, 0.0};
  constexpr int iG = kS + kD;   // first column of grad S
  const int ncol = a.ncset * a.nrhs;
  const int cnt = a.cnt[3 * blk + 1];
  const int2* far = reinterpret_cast<const int2*>(a.far) + (size_t)blk * (a.M + 1);
  const float ka = (float)sc_abs(kk);
  // an entry may be shared by nparts warps, each with every nparts-th pair of orders m
  const int np = a.nparts;
  for (int e = split * W + warp; e < cnt * np; e += a.nsplit * W) {
    const int mpart = e % np;
    const int2 ent = far[cnt - 1 - e / np];   // the local expansion, the longest entry, first
    const int om = ent.y & 0xff, ol = ent.y >> 8 & 0xff;
    const bool local = ent.y >> 16;
    int lmax = ol;   // of order m = lane
    const double* nd = a.node + 4 * (size_t)ent.x;
    const double vx = cx - nd[0], vy = cy - nd[1];
    double inv, rho, yq;
    const double d2 = fma(vx, vx, vy * vy);
    double ct, st;   // Theta
    const int nH = om + ol + 1;   // (pairs of orders and the cut reach one further)
    if (local) {
      // regular waves: J_n(k d) in the place of H_n
      rho = sqrt(d2);
      const bool off = rho > 0.0;   // (the centre may be the block's)
      ct = off ? vx / rho : 1.0;
      st = off ? vy / rho : 0.0;
      besselj_wave<T>(rmul(kk, rho), nH, sH);
    } else {
      kw.geom(d2, inv, rho, yq);
      cplx h0, h1;
      T twoz;
      kw.hankel(rho, inv, yq, h0, h1, twoz);
      ct = vx * inv;
      st = vy * inv;
      T s = twoz;
      sH[0] = h0;
      for (int i = 1; i <= nH; ++i) {
        sH[i * 32] = h1;
        const cplx h2 = hrec(s, h1, h0);
        h0 = h1;
        h1 = h2;
        s = sadd(s, twoz);
      }
      // Orders l that order m needs (lane = m): the terms (kR/2)^m/m!
      // (kr/2)^l/l! |H_{m+l}| of the nearest centre against |H_nd|, dropped
      // below 2^-61 (their count is below 2^6); in exponents, FP32.
      const float rf = (float)rho, rmin = warp_min(rf), rc = warp_max((float)r);
      const int nl = __ffs(__ballot_sync(0xffffffffu, rf == rmin)) - 1;
      __syncwarp();
      const cplx* col = sH - lane + nl;
      auto ex = [&](int n) {
        const cplx h = col[n * 32];
        return (float)(max(__double2hiint(h.re) >> 20 & 0x7ff, __double2hiint(h.im) >> 20 & 0x7ff) - 1022);
      };
      if (lane <= om) {
        const float R = (float)nd[2], fm = (float)lane;
        const float lr = __log2f(0.5f * ka * rc);
        float base = fm * __log2f(0.5f * ka * R) - lgammaf(fm + 1.0f) * 1.442695f - ex(a.nd) + 3.0f +
                     1.442695f * (float)a.kim * (R + rc);
        const float wm = a.nd ? fm / (ka * R) : 1.0f, wl = a.nd ? 1.0f / (ka * rc) : 0.0f;
        lmax = 0;
        for (int l = 1; l <= ol; ++l) {
          base += lr - __log2f((float)l);
          if (base + ex(lane + l) + __log2f(fmaxf(wm, wl * (float)l)) > -61.0f) lmax = l;
        }
      }
      __syncwarp();
    }
    // orders m whose expansions reach the cut at l = p (grad S)
    const unsigned cut = ol == p ? __ballot_sync(0xffffffffu, lane <= om && lmax >= p) : 0u;
    const int mcut = cut ? 32 - __clz(cut) : -1;   // one order further: the derivative shifts m by one
    const double cp = fma(ux, ct, uy * st), sp = fma(uy, ct, -ux * st);   // psi
    double cP = 1.0, sP = 0.0;   // p psi, after the loop for ol == p
    for (int l = 1; l <= ol; ++l) {
      const double cn = fma(cP, cp, -sP * sp);
      sP = fma(sP, cp, cP * sp);
      cP = cn;
      const T j = colJ[l * 32];
      T* f = sF + (l - 1) * 64;
      f[0] = rmul(j, cP);
      f[32] = rmul(j, sP);
    }
    const cplx* co = reinterpret_cast<const cplx*>(a.coef) + ((size_t)ent.x * (kTreeP + 1) * ncol + a.rhs0) * 2;
    cplx U0[NR], V0[NR], U1[NR], V1[NR];
    if (kG) {
#pragma unroll
      for (int i = 0; i < NR; ++i) U0[i] = V0[i] = U1[i] = V1[i] = cplx{0.0, 0.0};
    }
    // e^{i m Theta} of this warp's first m and the step between its pairs
    double cm = 1.0, sm = 0.0, cstep = fma(ct, ct, -st * st), sstep = 2.0 * ct * st;
    if (np > 1) {
      const double c2 = cstep, s2 = sstep;
      for (int i = 1; i < np; ++i) {
        if (i == mpart) {
          cm = cstep;
          sm = sstep;
        }
        const double cn = fma(cstep, c2, -sstep * s2);
        sstep = fma(sstep, c2, cstep * s2);
        cstep = cn;
      }
      if (mpart == 0) {
        cm = 1.0;
        sm = 0.0;
      }
    }
    auto wave = [&](int n) {   // H_n, any sign of n
      return neg_if(n < 0 && (n & 1), sH[(n < 0 ? -n : n) * 32]);
    };
    auto finish = [&](int m, double c, double s, cplx X, cplx Y) {
      const cplx fc = lin2(c, X, -s, Y), fs = lin2(s, X, c, Y);
#pragma unroll
      for (int q = 0; q < kC; ++q) {
        const double2* v = reinterpret_cast<const double2*>(co + ((size_t)m * ncol + (size_t)set[q] * a.nrhs) * 2);
#pragma unroll
        for (int i = 0; i < NR; ++i) {
          if (i > 0 && i >= a.nr) break;
          const double2 A = __ldg(v + 2 * i), B = __ldg(v + 2 * i + 1);
          cfma(acc[q][i], cplx{A.x, A.y}, fc);
          cfma(acc[q][i], cplx{B.x, B.y}, fs);
        }
      }
      if (kG && m <= mcut) {
        const cplx a0 = wave(m - p), b0 = neg_if(p & 1, wave(m + p));
        const cplx a1 = wave(m - p - 1), b1 = neg_if(!(p & 1), wave(m + p + 1));
        const double2* v = reinterpret_cast<const double2*>(co + ((size_t)m * ncol + (size_t)a.set_g * a.nrhs) * 2);
#pragma unroll
        for (int i = 0; i < NR; ++i) {
          if (i > 0 && i >= a.nr) break;
          const double2 A = __ldg(v + 2 * i), B = __ldg(v + 2 * i + 1);
          const cplx s_{fma(A.x, c, B.x * s), fma(A.y, c, B.y * s)};
          const cplx d_{fma(B.y, c, -A.y * s), fma(A.x, s, -B.x * c)};
          cfma(U0[i], s_, a0 + b0);
          cfma(V0[i], d_, a0 - b0);
          cfma(U1[i], s_, a1 + b1);
          cfma(V1[i], d_, a1 - b1);
        }
      }
    };
    // two orders m, m + 1 at a time: their waves overlap (H_{m+l+1} serves both
    // at consecutive l), and the sums are eight independent chains
    for (int m = 2 * mpart; m <= om; m += 2 * np) {
      const bool two = m < om;
      cplx lo1 = sH[m * 32], hi0 = lo1, hi1 = sH[(m + 1) * 32];   // H_{m+1-l}, H_{m+l}, H_{m+1+l}
      cplx X0 = smul(J0, hi0), X1 = smul(J0, hi1), Y0{0.0, 0.0}, Y1{0.0, 0.0};
      const int lm = max(__shfl_sync(0xffffffffu, lmax, m), __shfl_sync(0xffffffffu, lmax, min(m + 1, om)));
      auto order = [&](int l, bool odd) {
        // lo0 = H_{m-l}, lo1 = H_{m+1-l}, hi0 = H_{m+l}, hi1 = H_{m+1+l}
        const cplx lo0 = wave(m - l);
        hi0 = hi1;
        hi1 = sH[(m + 1 + l) * 32];
        const T jc = sF[(l - 1) * 64], js = sF[(l - 1) * 64 + 32];
        const cplx s0 = lo0 + hi0, d0 = lo0 - hi0, s1 = lo1 + hi1, d1 = lo1 - hi1;
        madd(X0, jc, odd ? d0 : s0);
        madd(Y0, js, odd ? s0 : d0);
        madd(X1, jc, odd ? d1 : s1);
        madd(Y1, js, odd ? s1 : d1);
        lo1 = lo0;
      };
      int l = 1;
      for (; l < lm; l += 2) {
        order(l, true);
        order(l + 1, false);
      }
      if (l <= lm) order(l, true);
      finish(m, cm, sm, X0, Y0);
      if (two) finish(m + 1, fma(cm, ct, -sm * st), fma(sm, ct, cm * st), X1, Y1);
      const double cn = fma(cm, cstep, -sm * sstep);
      sm = fma(sm, cstep, cm * sstep);
      cm = cn;
    }
    if (kG && mcut >= 0) {
      const T hk = rmul(kk, -0.5);
      const T jp = sc_mul(hk, colJ[p * 32]), jq = sc_mul(hk, colJ[(p + 1) * 32]);   // -(k/2) J_p, J_{p+1}
      const cplx e0{cP, sP}, e1{fma(cP, cp, -sP * sp), fma(sP, cp, cP * sp)};         // e^{i p psi}, e^{i(p+1) psi}
      const cplx et{ux, uy};
#pragma unroll
      for (int i = 0; i < NR; ++i) {
        cplx d = smul(jp, e1 * (U1[i] + V1[i])), b = smul(jp, conj(e1) * (U1[i] - V1[i]));
        madd(d, jq, conj(e0) * (U0[i] - V0[i]));
        madd(b, jq, e0 * (U0[i] + V0[i]));
        d = conj(et) * d;
        b = et * b;
        acc[iG][i] = acc[iG][i] + 0.5 * (d + b);
        acc[iG + 1][i] = acc[iG + 1][i] + mul_i(0.5 * (d - b));
      }
    }
  }
  // ---- the warps' sums, in warp order (through the warps' areas) ----
  cplx* s_sum = reinterpret_cast<cplx*>(smem_raw + far_col_bytes<T>(pl)) + lane;
  for (int w = 0; w < W; ++w) {
    __syncthreads();
    if (warp == w) {
#pragma unroll
      for (int q = 0; q < kC; ++q)
#pragma unroll
        for (int i = 0; i < NR; ++i) {
          cplx* m = s_sum + (q * NR + i) * 32;
          if (w > 0) acc[q][i] = *m + acc[q][i];
          *m = acc[q][i];
        }
    }
  }
  if (warp != W - 1 || !active) return;
  cplx* part = reinterpret_cast<cplx*>(a.part);
  const size_t row = ((size_t)(a.split0 + split) * a.n_ctr + c) * kC;
#pragma unroll
  for (int i = 0; i < NR; ++i) {
    if (i >= a.nr) break;
#pragma unroll
    for (int q = 0; q < kC; ++q) part[(row + q) * a.nrhs + a.rhs0 + i] = acc[q][i];
  }
}

// warps per CTA with the most warps on an SM (at least two CTAs on it, where
// that many fit), and the CTA's shared memory; 0: none fits
template <typename T>
size_t far_smem(int pl, int n_acc, int* warps) {
  size_t best = 0;
  int most = 0;
  *warps = 0;
  for (int w = 4; w >= 1; --w) {
    const size_t b = far_col_bytes<T>(pl) + std::max(w * far_warp_bytes<T>(pl), (size_t)n_acc * 32 * 16);
    if (b > 220 * 1024) continue;
    const int ctas = (int)std::min<size_t>((size_t)227 * 1024 / (b + 1024), 16);
    const int on = w * ctas * 2 - (ctas < 2 ? 1 : 0);
    if (on > most) {
      most = on;
      best = b;
      *warps = w;
    }
  }
  return best;
}

// rhs per launch: grad S keeps four more sums per rhs and node
constexpr int far_nr(int ops) { return (ops & OPB_G) ? 2 : 4; }
int acc_count(int ops, int nr) {
  return ((ops & 1) + (ops >> 1 & 1) + 2 * (ops >> 2 & 1) + 2 * (ops >> 3 & 1)) * nr;
}

template <int OPS, typename T, int NR>
cudaError_t launch_far_t(const TreeArgs& a, cudaStream_t st) {
  int w = 0;
  const size_t smem = far_smem<T>(a.pl, acc_count(OPS, NR), &w);
  if (!smem) return cudaErrorInvalidValue;
  auto kern = k_far_clusters<OPS, T, NR>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  kern<<<(unsigned)(a.n_blk * (a.n_ctr / a.n_tgt)) * (unsigned)a.nsplit, 32 * w, smem, st>>>(a);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_far_ops(const TreeArgs& a, cudaStream_t st) {
#define QBX_FAR(O) case O: return a.nr <= 1 ? launch_far_t<O, T, 1>(a, st) : launch_far_t<O, T, far_nr(O)>(a, st);
  switch (a.ops) {
    QBX_FAR(1) QBX_FAR(2) QBX_FAR(3) QBX_FAR(4) QBX_FAR(5) QBX_FAR(6) QBX_FAR(7) QBX_FAR(12)
    default: return cudaErrorInvalidValue;
  }
#undef QBX_FAR
}

template <typename T>
size_t moments_smem(int q_src) {
  return (size_t)2 * (kTreeP + 3) * (q_src | 1) * sizeof(T);
}

template <typename T>
cudaError_t launch_moments_t(const TreeArgs& a, cudaStream_t st) {
  const size_t smem = moments_smem<T>(a.q_src);
  cudaError_t e = cudaFuncSetAttribute(k_tree_moments<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  k_tree_moments<T><<<dim3(a.M, a.lev), 128, smem, st>>>(a);
  k_tree_fold<<<dim3(a.off[a.lev], a.nset * a.nrhs), 64, 0, st>>>(a);
  k_tree_local<T><<<dim3(a.n_blk, (a.nset * a.nrhs + kLocCols - 1) / kLocCols), 32 * kLocWarps, 0, st>>>(a);
  return cudaGetLastError();
}

}  // namespace

int tree_levels(int panels, int q_src, TreeArgs* a) {
  // half panels as leaves where that leaves them 16 sources or more: near
  // pairs 2.05 -> 1.65 ms, far nodes 0.77 -> 0.99 ms (starfish, 256 panels)
  const int half = q_src % 2 == 0 && q_src >= 32;
  const int M = panels << half;
  a->M = M;
  a->q_src = q_src >> half;
  a->n_src = panels * q_src;
  int l = 0, n = 0;
  do {
    a->off[l] = n;
    n += (M + (1 << l) - 1) >> l;
    ++l;
  } while (l < kTreeLevels && (M >> l) >= 8);   // nodes of up to about an eighth of the curve
  a->lev = l;
  a->off[l] = n;
  return n;
}

size_t tree_layout(TreeArgs* a, char* base) {
  size_t at = 0;
  auto take = [&](size_t bytes) {
    char* v = base ? base + at : nullptr;
    at += host_align256(bytes);
    return v;
  };
  const size_t nodes = (size_t)a->off[a->lev] + a->n_blk, ncol = (size_t)a->ncset * a->nrhs;
  a->node = (double*)take(nodes * 4 * 8);
  a->near = (int*)take((size_t)a->n_blk * a->M * 4);
  a->far = (int*)take((size_t)a->n_blk * (a->M + 1) * 8);
  a->loc = (int*)take((size_t)a->n_blk * a->M * 8);
  a->cnt = (int*)take((size_t)a->n_blk * 12);
  a->mom = take((size_t)a->lev * a->M * a->nset * a->nrhs * (kTreeP + 2) * 2 * 16);
  a->coef = take(nodes * ncol * (kTreeP + 1) * 2 * 16);
  return at;
}

cudaError_t launch_tree_lists(const TreeArgs& a, cudaStream_t st) {
  k_tree_nodes<<<a.off[a.lev], 256, 0, st>>>(a);
  k_tree_lists<<<a.n_blk, 32 * kListWarps, 0, st>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_tree_moments(const TreeArgs& a, cudaStream_t st) {
  return a.kim != 0.0 ? launch_moments_t<cplx>(a, st) : launch_moments_t<double>(a, st);
}

cudaError_t launch_far_clusters(TreeArgs a, cudaStream_t st) {
  const int n = far_nr(a.ops);
  for (int r0 = 0; r0 < a.nrhs; r0 += n) {
    a.rhs0 = r0;
    a.nr = std::min(n, a.nrhs - r0);
    const cudaError_t e = a.kim != 0.0 ? launch_far_ops<cplx>(a, st) : launch_far_ops<double>(a, st);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

bool far_clusters_fit(const TreeArgs& a) {
  int w;
  const int n = acc_count(a.ops, a.nrhs <= 1 ? 1 : far_nr(a.ops));
  return (a.kim != 0.0 ? far_smem<cplx>(a.pl, n, &w) : far_smem<double>(a.pl, n, &w)) > 0;
}

// moment set of `kind` of density `slot` (one per pair); its own coefficient
// columns always exist
static int moment_set(TreeArgs* a, int kind, int slot) {
  for (int i = 0; i < a->nset; ++i)
    if (a->kind[i] == kind && a->slot[i] == slot) return i;
  const int i = a->nset++;
  a->kind[i] = kind;
  a->slot[i] = slot;
  a->plain[i] = a->ncset;
  a->base[a->ncset] = i;
  a->shift[a->ncset++] = 0;
  return i;
}

void tree_columns(TreeArgs* a, const int slot[3]) {
  a->nset = a->ncset = 0;
  if (a->ops & OPB_S) a->set_s = a->plain[moment_set(a, kSetMono, slot[0])];
  if (a->ops & OPB_D) a->set_d = a->plain[moment_set(a, kSetNormal, slot[1])];
  if (a->ops & OPB_G) {
    const int m = moment_set(a, kSetMono, slot[2]);
    a->set_g = a->plain[m];
    a->set_gx = a->ncset;
    for (int sh = 1; sh <= 2; ++sh) {
      a->base[a->ncset] = m;
      a->shift[a->ncset++] = sh;
    }
  }
  if (a->ops & OPB_X) {
    a->set_x = a->plain[moment_set(a, kSetX, slot[2])];
    moment_set(a, kSetY, slot[2]);
  }
}

}  // namespace qbx
