// qbx_misc.cu -- geometry (a0), density oversampling (a1), the unfused
// coefficient formation (a4) and evaluation (a5 + a6), the split reductions
// with the jump epilogue (a7), centre assignment and diagnostics.
#include <cuda_runtime.h>
#include <stdint.h>
#include "qbx_apply_impl.cuh"
#include "qbx_internal.h"

namespace qbx {

__device__ __forceinline__ bool finite_c(cplx v) { return isfinite(v.re) && isfinite(v.im); }

// ---------------------------------------------------------------------------
// a0 Geometry (Sec. 3.3 step 4a; Sec. 3.2 n = (t_2, -t_1); Sec. 4.1 panels).
// ---------------------------------------------------------------------------
__global__ void k_geom_nodes(int n, int q, const double* t_edges, const double* gam,
                             const double* dgam, const double* wgl, double* x, double* y,
                             double* nx, double* ny, double* w) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int m = i / q, j = i - m * q;
  const double half = 0.5 * (t_edges[m + 1] - t_edges[m]);
  const double gx = dgam[2 * i], gy = dgam[2 * i + 1];
  const double sp = hypot(gx, gy);
  x[i] = gam[2 * i];
  y[i] = gam[2 * i + 1];
  nx[i] = gy / sp;
  ny[i] = -gx / sp;
  w[i] = wgl[j] * half * sp;
}

// h_m: sum of the panel's source weights in node order (deterministic).
__global__ void k_panel_h(int M, int q_src, const double* w, double* h) {
  const int m = blockIdx.x * blockDim.x + threadIdx.x;
  if (m >= M) return;
  double s = 0.0;
  for (int j = 0; j < q_src; ++j) s += w[m * q_src + j];
  h[m] = s;
}

__global__ void k_centres(int n_tgt, int q_tgt, double r_factor, int rule, const double* h, const double* tx,
                          const double* ty, const double* tnx, const double* tny, double* cx,
                          double* cy, double* cr) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n_tgt) return;
  const double hm = h[t / q_tgt];
  const double r = rule == QBX_RADIUS_SQRT_H ? r_factor * sqrt(hm) : r_factor * hm;
  cx[t] = tx[t] - r * tnx[t];
  cy[t] = ty[t] - r * tny[t];
  cr[t] = r;
  cx[n_tgt + t] = tx[t] + r * tnx[t];
  cy[n_tgt + t] = ty[t] + r * tny[t];
  cr[n_tgt + t] = r;
}

// Radius rule QBX_RADIUS_ADMISSIBLE (a departure from Sec. 3.3 step 4a for
// corners of 90 degrees or less): each centre's radius lowered to the largest
// r whose disk holds no source node.  With d = x_s - x and c = x + sg r n,
// |d - sg r n|^2 >= r^2 reads |d|^2 - 2 sg r (d.n) >= 0: a bound
// r <= |d|^2 / (2 sg d.n) for every source with sg d.n > 0.
__global__ void k_cap_radius(int n_tgt, const double* tx, const double* ty, const double* tnx, const double* tny,
                             int n_src, const double* sx, const double* sy, double* cx, double* cy, double* cr) {
  __shared__ double bx[256], by[256];
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  const int cc = c < 2 * n_tgt ? c : 2 * n_tgt - 1;
  const int t = cc % n_tgt;
  const double sg = cc < n_tgt ? -1.0 : 1.0;
  const double x = tx[t], y = ty[t], nx = sg * tnx[t], ny = sg * tny[t];
  double r = cr[cc];
  for (int base = 0; base < n_src; base += 256) {
    const int nt = min(256, n_src - base);
    __syncthreads();
    for (int i = threadIdx.x; i < nt; i += blockDim.x) {
      bx[i] = sx[base + i];
      by[i] = sy[base + i];
    }
    __syncthreads();
    for (int j = 0; j < nt; ++j) {
      const double dx = bx[j] - x, dy = by[j] - y;
      const double a = fma(dx, nx, dy * ny);
      if (a > 0.0) r = fmin(r, fma(dx, dx, dy * dy) / (2.0 * a));
    }
  }
  if (c < 2 * n_tgt) {
    cr[c] = r;
    cx[c] = fma(r, nx, x);
    cy[c] = fma(r, ny, y);
  }
}

// ratio = min_s |x_s - c| / r  (eq. x-c-closest).  A CTA of eight warps holds
// 32 centres, one per lane, and the warps share the sources.  The distances are
// first taken in FP32 relative to the CTA's first centre, with a bound of their
// error; only sources that can be the closest are then measured in FP64 (the
// FP32 pipe has 64 times the FP64 rate here).  The all-FP64 loop of one thread
// per centre: 2.94 ms at 128 panels (4096 centres, 8192 sources).
constexpr int kRatioWarps = 8, kRatioTile = 128;
__global__ void __launch_bounds__(32 * kRatioWarps)
k_ratio(int n_ctr, const double* cx, const double* cy, const double* cr, int n_src, const double* sx, const double* sy,
        double* ratio) {
  __shared__ float2 s_p[kRatioWarps][kRatioTile];
  __shared__ float s_ub[kRatioWarps][32];
  __shared__ double s_best[kRatioWarps][32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int c = blockIdx.x * 32 + lane, cc = min(c, n_ctr - 1), c0 = blockIdx.x * 32;
  const double x0 = cx[c0], y0 = cy[c0], x = cx[cc], y = cy[cc];
  const float fx = (float)(x - x0), fy = (float)(y - y0);
  float ec = 4e-7f * (fabsf(fx) + fabsf(fy));
  for (int o = 16; o > 0; o >>= 1) ec = fmaxf(ec, __shfl_xor_sync(0xffffffffu, ec, o));
  // one tile of sources relative to the first centre; returns the error bound
  // of its distances (to any of the centres)
  auto stage = [&](int base) {
    __syncwarp();
    float e = 0.0f;
    for (int i = lane; i < kRatioTile && base + i < n_src; i += 32) {
      const float bx = (float)(sx[base + i] - x0), by = (float)(sy[base + i] - y0);
      s_p[warp][i] = make_float2(bx, by);
      e = fmaxf(e, 4e-7f * (fabsf(bx) + fabsf(by)));
    }
    for (int o = 16; o > 0; o >>= 1) e = fmaxf(e, __shfl_xor_sync(0xffffffffu, e, o));
    __syncwarp();
    return e + ec;
  };
  auto dist2 = [&](int j) {
    const float2 v = s_p[warp][j];
    const float dx = v.x - fx, dy = v.y - fy;
    return fmaf(dx, dx, dy * dy);
  };
  // upper bound of the smallest distance
  float ub = INFINITY;
  for (int base = warp * kRatioTile; base < n_src; base += kRatioWarps * kRatioTile) {
    const float e = stage(base);
    const int nt = min(kRatioTile, n_src - base);
    float m = INFINITY;
#pragma unroll 8
    for (int j = 0; j < nt; ++j) m = fminf(m, dist2(j));
    ub = fminf(ub, sqrtf(m) + e);
  }
  s_ub[warp][lane] = ub;
  __syncthreads();
  for (int w = 0; w < kRatioWarps; ++w) ub = fminf(ub, s_ub[w][lane]);
  // the sources that may be closer, in FP64 (also those whose FP32 distance is no number)
  double best = INFINITY;
  for (int base = warp * kRatioTile; base < n_src; base += kRatioWarps * kRatioTile) {
    const float e = stage(base), t = (ub + e) * 1.000001f, t2 = t * t;
    const int nt = min(kRatioTile, n_src - base);
    float m = INFINITY;   // a tile with none, at the price of the minimum
    bool odd = false;
#pragma unroll 8
    for (int j = 0; j < nt; ++j) {
      const float v = dist2(j);
      odd |= !(v <= 3e38f);
      m = fminf(m, v);
    }
    if (!odd && m > t2) continue;
    for (int j = 0; j < nt; ++j) {
      if (dist2(j) > t2) continue;
      const double ex = sx[base + j] - x, ey = sy[base + j] - y;
      best = fmin(best, fma(ex, ex, ey * ey));
    }
  }
  s_best[warp][lane] = best;
  __syncthreads();
  if (warp == 0 && c < n_ctr) {
    for (int w = 1; w < kRatioWarps; ++w) best = fmin(best, s_best[w][lane]);
    ratio[c] = sqrt(best) / cr[c];
  }
}

cudaError_t launch_geometry(int M, int q_tgt, int q_src, const double* t_edges,
                            const double* gam_tgt, const double* dgam_tgt,
                            const double* gam_src, const double* dgam_src,
                            const double* wgl_tgt, const double* wgl_src, double r_factor, int rule,
                            const qbx_geom& g, cudaStream_t st) {
  const int n_t = M * q_tgt, n_s = M * q_src;
  k_geom_nodes<<<(n_s + 255) / 256, 256, 0, st>>>(n_s, q_src, t_edges, gam_src, dgam_src, wgl_src,
                                                 g.src_x, g.src_y, g.src_nx, g.src_ny, g.src_w);
  k_geom_nodes<<<(n_t + 255) / 256, 256, 0, st>>>(n_t, q_tgt, t_edges, gam_tgt, dgam_tgt, wgl_tgt,
                                                 g.tgt_x, g.tgt_y, g.tgt_nx, g.tgt_ny, g.tgt_w);
  k_panel_h<<<(M + 127) / 128, 128, 0, st>>>(M, q_src, g.src_w, g.panel_h);
  k_centres<<<(n_t + 255) / 256, 256, 0, st>>>(n_t, q_tgt, r_factor, rule, g.panel_h, g.tgt_x, g.tgt_y,
                                              g.tgt_nx, g.tgt_ny, g.ctr_x, g.ctr_y, g.ctr_r);
  if (rule == QBX_RADIUS_ADMISSIBLE)
    k_cap_radius<<<(2 * n_t + 255) / 256, 256, 0, st>>>(n_t, g.tgt_x, g.tgt_y, g.tgt_nx, g.tgt_ny, n_s, g.src_x,
                                                       g.src_y, g.ctr_x, g.ctr_y, g.ctr_r);
  k_ratio<<<(2 * n_t + 31) / 32, 32 * kRatioWarps, 0, st>>>(2 * n_t, g.ctr_x, g.ctr_y, g.ctr_r, n_s, g.src_x,
                                                g.src_y, g.ctr_ratio);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// a1 Oversampling (Sec. 3.4.2): wdens[s][r] = w_s sum_i P[j][i] dens[m q_tgt + i][r].
// ---------------------------------------------------------------------------
__global__ void k_upsample(int n_src, int q_tgt, int q_src, int nrhs, const double* P,
                           const double* w, const cplx* dens, cplx* out) {
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= n_src * nrhs) return;
  const int s = idx / nrhs, r = idx - s * nrhs;
  const int m = s / q_src, j = s - m * q_src;
  const double* row = P + (size_t)j * q_tgt;
  const cplx* d = dens + (size_t)m * q_tgt * nrhs + r;
  double re = 0.0, im = 0.0;
  for (int i = 0; i < q_tgt; ++i) {
    const double c = row[i];
    const cplx v = d[(size_t)i * nrhs];
    re = fma(c, v.re, re);
    im = fma(c, v.im, im);
  }
  out[idx] = cplx{w[s] * re, w[s] * im};
}

// Unit tangents t = (-n_y, n_x) of the source nodes (the R operator of
// Sec. 3.2, eq. riesz-def, takes the D kernel with t in place of n).
__global__ void k_tangents(int n, const double* nx, const double* ny, double* tx, double* ty) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  tx[i] = -ny[i];
  ty[i] = nx[i];
}

cudaError_t launch_tangents(int n, const double* nx, const double* ny, double* tx, double* ty, cudaStream_t st) {
  if (n < 1) return cudaSuccess;
  k_tangents<<<(n + 255) / 256, 256, 0, st>>>(n, nx, ny, tx, ty);
  return cudaGetLastError();
}

// grad D finish (Sec. 3.2, eq. dlpderiv): ev [n_ctr][2][nrhs] are the
// gradients of the D expansions at the targets (interior centres first for
// two sides).  Two-sided: the average; PV from one side: lim -/+ t dmu/ds / 2
// (+ exterior), t = (-n_y, n_x), dmu/ds = (sum_j Dx[i][j] mu_j) w^GL_i / w_t.
__global__ void k_grad_d_finish(int n_tgt, int q_tgt, int nsides, int side0, int limit, int nrhs,
                                const cplx* ev, const cplx* dens, const double* tnx, const double* tny,
                                const double* tw, const double* wgl, const double* Dx, cplx* out, int* status) {
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= n_tgt * nrhs) return;
  const int t = idx / nrhs, r = idx - t * nrhs;
  cplx gx{0.0, 0.0}, gy{0.0, 0.0};
  for (int sd = 0; sd < nsides; ++sd) {
    const size_t row = ((size_t)(sd * n_tgt + t) * 2) * nrhs + r;
    gx = gx + ev[row];
    gy = gy + ev[row + nrhs];
  }
  if (nsides == 2) {
    gx = 0.5 * gx;
    gy = 0.5 * gy;
  } else if (limit == QBX_LIMIT_PV) {
    const int m = t / q_tgt, i = t - m * q_tgt;
    const cplx* d = dens + (size_t)m * q_tgt * nrhs + r;
    double re = 0.0, im = 0.0;
    for (int j = 0; j < q_tgt; ++j) {
      const double c = Dx[i * q_tgt + j];
      re = fma(c, d[(size_t)j * nrhs].re, re);
      im = fma(c, d[(size_t)j * nrhs].im, im);
    }
    const double f = wgl[i] / tw[t];
    const cplx ds{re * f, im * f};
    const double sg = side0 == QBX_SIDE_EXT ? 1.0 : -1.0;
    gx = gx - (0.5 * sg * -tny[t]) * ds;
    gy = gy - (0.5 * sg * tnx[t]) * ds;
  }
  out[((size_t)t * 2) * nrhs + r] = gx;
  out[((size_t)t * 2 + 1) * nrhs + r] = gy;
  if (!(isfinite(gx.re) && isfinite(gx.im) && isfinite(gy.re) && isfinite(gy.im))) atomicOr(status, 1);
}

cudaError_t launch_grad_d_finish(int n_tgt, int q_tgt, int nsides, int side0, int limit, int nrhs, const void* ev,
                                 const void* dens, const double* tnx, const double* tny, const double* tw,
                                 const double* wgl, const double* Dx, void* out, int* status, cudaStream_t st) {
  const int n = n_tgt * nrhs;
  k_grad_d_finish<<<(n + 255) / 256, 256, 0, st>>>(n_tgt, q_tgt, nsides, side0, limit, nrhs, (const cplx*)ev,
                                                   (const cplx*)dens, tnx, tny, tw, wgl, Dx, (cplx*)out, status);
  return cudaGetLastError();
}

cudaError_t launch_upsample(int M, int q_tgt, int q_src, int nrhs, const double* interp,
                            const double* src_w, const void* dens_tgt, void* wdens,
                            cudaStream_t st) {
  const int n = M * q_src * nrhs;
  k_upsample<<<(n + 255) / 256, 256, 0, st>>>(M * q_src, q_tgt, q_src, nrhs, interp, src_w,
                                              (const cplx*)dens_tgt, (cplx*)wdens);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// a7 Reduction over splits (fixed order), factor i/4, jump / average (Sec. 3.2).
// part: [nsplit][n_ctr][ncomp][nrhs]; for side TWO, centre t (interior) and
// n_tgt + t (exterior) are averaged.
// ---------------------------------------------------------------------------
__global__ void k_apply_finish(int op, int side, int limit, int n_tgt, int nsplit, int n_ctr,
                               int nrhs, int comp0, int ncomp_total, const cplx* part, const cplx* dens,
                               const double* tnx, const double* tny, cplx* out, int* status) {
  const int ncomp = op == QBX_OP_GRAD_S ? 2 : 1;
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= n_tgt * ncomp * nrhs) return;
  const int t = idx / (ncomp * nrhs);
  const int rem = idx - t * ncomp * nrhs;
  const int comp = rem / nrhs, r = rem - comp * nrhs;
  const int nsides = side == QBX_SIDE_TWO ? 2 : 1;
  cplx res{0.0, 0.0};
  for (int sd = 0; sd < nsides; ++sd) {
    const int c = t + sd * n_tgt;
    cplx u{0.0, 0.0};
    for (int k = 0; k < nsplit; ++k)
      u = u + part[(((size_t)k * n_ctr + c) * ncomp_total + comp0 + comp) * nrhs + r];
    u = mul_i(0.25 * u);
    if (side != QBX_SIDE_TWO && limit == QBX_LIMIT_PV) {
      const double sg = side == QBX_SIDE_EXT ? 1.0 : -1.0;
      const cplx dv = dens[(size_t)t * nrhs + r];
      if (op == QBX_OP_D) u = u - (0.5 * sg) * dv;
      else if (op == QBX_OP_GRAD_S) u = u + (0.5 * sg * (comp == 0 ? tnx[t] : tny[t])) * dv;
    }
    res = res + u;
  }
  if (nsides == 2) res = 0.5 * res;
  out[idx] = res;
  if (!finite_c(res)) atomicOr(status, 1);
}

cudaError_t launch_apply_finish(int op, int side, int limit, int n_tgt, int nsplit, int n_ctr,
                                int nrhs, int comp0, int ncomp_total, const void* part,
                                const void* dens_tgt, const double* tgt_nx, const double* tgt_ny,
                                void* out, int* status, cudaStream_t st) {
  const int ncomp = op == QBX_OP_GRAD_S ? 2 : 1;
  const int n = n_tgt * ncomp * nrhs;
  k_apply_finish<<<(n + 255) / 256, 256, 0, st>>>(op, side, limit, n_tgt, nsplit, n_ctr, nrhs, comp0,
                                                  ncomp_total, (const cplx*)part, (const cplx*)dens_tgt,
                                                  tgt_nx, tgt_ny, (cplx*)out, status);
  return cudaGetLastError();
}

// Fused apply dispatch: real k (fitted real-argument Hankel path) or complex k.
cudaError_t launch_apply_fused(const ApplyArgs& a, cudaStream_t st) {
  if (a.eta2 > 0.0) return a.kim == 0.0 ? launch_apply_fused_local_real(a, st) : launch_apply_fused_local_cplx(a, st);
  return a.kim == 0.0 ? launch_apply_fused_real(a, st) : launch_apply_fused_cplx(a, st);
}

size_t apply_smem_bytes(int ops, bool ck, int p, int nr) {
  return ck ? apply_smem_bytes_cplx(ops, p, nr) : apply_smem_bytes_real(ops, p, nr);
}

// rhs per launch: accumulators for one operator take 8 rhs in registers,
// several operators together 4.
int apply_chunk(int ops) { return (ops == 1 || ops == 2 || ops == 4) ? 8 : 4; }

__global__ void k_far_finish(int op, double kre, double kim, int n_far, int nsplit, int nrhs,
                             const cplx* part, cplx* out, int* status) {
  const int ncomp = op == QBX_OP_GRAD_S ? 2 : 1;
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= n_far * ncomp * nrhs) return;
  cplx u{0.0, 0.0};
  for (int k = 0; k < nsplit; ++k) u = u + part[(size_t)k * n_far * ncomp * nrhs + idx];
  cplx f = op == QBX_OP_S ? cplx{0.0, 0.25} : cplx{-0.25 * kim, 0.25 * kre};  // i/4 or ik/4
  if (op == QBX_OP_GRAD_S) f = -f;
  u = f * u;
  out[idx] = u;
  if (!finite_c(u)) atomicOr(status, 1);
}

cudaError_t launch_far_finish(int op, double kre, double kim, int n_far, int nsplit, int nrhs,
                              const void* part, void* out, int* status, cudaStream_t st) {
  const int ncomp = op == QBX_OP_GRAD_S ? 2 : 1;
  const int n = n_far * ncomp * nrhs;
  k_far_finish<<<(n + 255) / 256, 256, 0, st>>>(op, kre, kim, n_far, nsplit, nrhs,
                                                (const cplx*)part, (cplx*)out, status);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// a4 Unfused coefficients (Sec. 3.3 step 4b).  A CTA holds 32 centres of one
// side, one per lane; its two warps take the sources (all, or the block's near
// leaves) in turn, with accumulators for the 2p+1 orders of `nr` rhs in shared
// memory, added up at the end.
// (factor i/4 in the finishing kernel).
// ---------------------------------------------------------------------------
// With E_n = H_n e^{-i n theta}, E_{-n} = (-1)^n H_n e^{i n theta}:
//   S: alpha_l += w E_l;  D: alpha_l += w (k/2)[conj(nu) E_{l-1} - nu E_{l+1}]
// (the factor k/2 on the sums).  ONE: a single rhs, w folded into the seeds
// H_0, H_1; otherwise one product per rhs.
template <typename T, bool ONE>
__global__ void __launch_bounds__(kFormThreads) k_form(FormArgs a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  cplx* s_acc = reinterpret_cast<cplx*>(smem_raw);              // [(2p+1)*nr][threads]
  const int nr = ONE ? 1 : a.nr;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int blks = (a.n_tgt + 31) / 32, side = blockIdx.x / blks, blk = blockIdx.x - side * blks;
  const bool active = blk * 32 + lane < a.n_tgt;
  const int c = side * a.n_tgt + (active ? blk * 32 + lane : a.n_tgt - 1);
  const int p = a.p, nl = 2 * p + 1;
  for (int i = 0; i < nl * nr; ++i) s_acc[i * kFormThreads + tid] = cplx{0.0, 0.0};
  const double cx = a.cx[c], cy = a.cy[c];
  KW<T> kw;
  kw.init(a.kre, a.kim, a.hk_tab);
  const int* near = a.near ? a.near + (size_t)blk * a.near_stride : nullptr;
  int v0 = blockIdx.y * a.src_per_split, v1 = min(a.src.n, v0 + a.src_per_split);
  if (near) {
    const long n = (long)a.near_cnt[3 * blk] * a.near_q;
    v0 = (int)(n * blockIdx.y / a.nsplit);
    v1 = (int)(n * (blockIdx.y + 1) / a.nsplit);
  }
  const cplx* wd = reinterpret_cast<const cplx*>(a.wd) + a.rhs0;   // the caller's: 8-byte aligned
  auto weight = [&](int s, int rr) {
    const cplx* w = wd + (size_t)s * a.nrhs + rr;
    return cplx{__ldg(&w->re), __ldg(&w->im)};
  };
  for (int v = v0 + warp; v < v1; v += kFormThreads / 32) {
    int s = v;
    if (near) {
      const int i = v / a.near_q;
      s = near[i] * a.near_q + (v - i * a.near_q);
    }
    const double dx = __ldg(a.src.x + s) - cx, dy = __ldg(a.src.y + s) - cy;
    double inv, rho, yq;
    kw.geom(fma(dx, dx, dy * dy), inv, rho, yq);
    const double ct = dx * inv, st = dy * inv;
    cplx Hm, H;   // H_{n-1}, H_n
    T twoz;
    if constexpr (ONE) {
      kw.hankel_w(rho, inv, yq, weight(s, 0), Hm, H, twoz);
    } else {
      kw.hankel(rho, inv, yq, Hm, H, twoz);
    }
    auto add = [&](int l, cplx v_) {   // alpha_l, l = -p..p
#pragma unroll 1
      for (int rr = 0; rr < nr; ++rr) {
        cplx* A = s_acc + ((size_t)(l + p) * nr + rr) * kFormThreads + tid;
        if constexpr (ONE) {
          *A = *A + v_;
        } else {
          cplx u = *A;
          cfma(u, weight(s, rr), v_);
          *A = u;
        }
      }
    };
    double cn = ct, sn = st;   // n theta
    T sz = twoz;
    auto waves = [&](cplx& Ep, cplx& En, int n) {   // E_n, E_{-n} of H
      const cplx hc = cn * H, hs = sn * H;
      Ep = cplx{hc.re + hs.im, hc.im - hs.re};      // H (cos - i sin)
      En = cplx{hc.re - hs.im, hc.im + hs.re};
      if (n & 1) En = -En;
    };
    auto step = [&] {
      const cplx h = hrec(sz, H, Hm);
      Hm = H;
      H = h;
      sz = sadd(sz, twoz);
      const double c2 = fma(cn, ct, -sn * st);
      sn = fma(sn, ct, cn * st);
      cn = c2;
    };
    if (a.kind == QBX_OP_S) {
      add(0, Hm);
      for (int n = 1; n <= p; ++n) {
        cplx Ep, En;
        waves(Ep, En, n);
        add(n, Ep);
        add(-n, En);
        if (n < p) step();
      }
    } else {
      const double nx = __ldg(a.src.nx + s), ny = __ldg(a.src.ny + s);
      const cplx nu{nx, ny}, nub{nx, -ny};
      // at n: E_{+-n}, E_{+-(n-1)}, E_{+-(n-2)}; alpha_{n-1} and alpha_{-(n-1)} complete
      cplx E1p = Hm, E1n = Hm, E2p{0.0, 0.0}, E2n{0.0, 0.0};
      for (int n = 1; n <= p + 1; ++n) {
        cplx Ep, En;
        waves(Ep, En, n);
        if (n == 1) {
          add(0, nub * En - nu * Ep);
        } else {
          add(n - 1, nub * E2p - nu * Ep);
          add(1 - n, nub * En - nu * E2n);
        }
        E2p = E1p;
        E2n = E1n;
        E1p = Ep;
        E1n = En;
        if (n <= p) step();
      }
    }
  }
  __syncthreads();
  if (!active) return;
  const cplx f = a.kind == QBX_OP_S ? cplx{1.0, 0.0} : cplx{0.5 * a.kre, 0.5 * a.kim};
  cplx* part = reinterpret_cast<cplx*>(a.part);
  for (int i = warp; i < nl * nr; i += kFormThreads / 32) {   // the warps' sums in warp order
    cplx u = s_acc[(size_t)i * kFormThreads + lane];
    for (int w = 1; w < kFormThreads / 32; ++w) u = u + s_acc[(size_t)i * kFormThreads + 32 * w + lane];
    const int l = i / nr, rr = i - l * nr;
    part[(((size_t)blockIdx.y * a.n_ctr + c) * nl + l) * a.nrhs + a.rhs0 + rr] = f * u;
  }
}

size_t form_smem_bytes(int p, int nr) { return (size_t)(2 * p + 1) * nr * kFormThreads * 16; }

template <typename T>
static cudaError_t launch_form_t(const FormArgs& a, cudaStream_t st) {
  const size_t smem = form_smem_bytes(a.p, a.nr);
  auto kern = a.nr == 1 ? k_form<T, true> : k_form<T, false>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  kern<<<dim3(apply_units(a.n_ctr, a.n_tgt), a.nsplit), kFormThreads, smem, st>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_form(const FormArgs& a, cudaStream_t st) {
  return a.kim != 0.0 ? launch_form_t<cplx>(a, st) : launch_form_t<double>(a, st);
}

__global__ void k_form_finish(int n_ctr, int ncoef, int nsplit, int nrhs, const cplx* part,
                              cplx* alpha, int* status) {
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;
  const size_t n = (size_t)n_ctr * ncoef * nrhs;
  if (idx >= n) return;
  cplx u{0.0, 0.0};
  for (int k = 0; k < nsplit; ++k) u = u + part[(size_t)k * n + idx];
  u = mul_i(0.25 * u);
  alpha[idx] = u;
  if (!finite_c(u)) atomicOr(status, 1);
}

cudaError_t launch_form_finish(int n_ctr, int ncoef, int nsplit, int nrhs, const void* part,
                               void* alpha, int* status, cudaStream_t st) {
  const size_t n = (size_t)n_ctr * ncoef * nrhs;
  k_form_finish<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(n_ctr, ncoef, nsplit, nrhs,
                                                            (const cplx*)part, (cplx*)alpha, status);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// a5 + a6: evaluate stored coefficients (Sec. 3.3 step 4c), value or gradient
//   u = sum_l alpha_l J_l(k rho) e^{i l theta}
//   (d_x + i d_y) u = -k sum alpha_l J_{l+1} e^{i(l+1)theta},
//   (d_x - i d_y) u =  k sum alpha_l J_{l-1} e^{i(l-1)theta}.
// ---------------------------------------------------------------------------
template <typename T>
__device__ __forceinline__ cplx jc(const T* J, int l) {
  const int al = l < 0 ? -l : l;
  cplx v = to_c(J[al]);
  if (l < 0 && (al & 1)) v = -v;
  return v;
}

template <typename T> __device__ __forceinline__ T make_kr(double kre, double kim, double rho);
template <> __device__ __forceinline__ double make_kr<double>(double kre, double, double rho) { return kre * rho; }
template <> __device__ __forceinline__ cplx make_kr<cplx>(double kre, double kim, double rho) {
  return cplx{kre * rho, kim * rho};
}

template <typename T>
__global__ void k_eval(EvalArgs a) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= a.n_eval) return;
  const int c = a.ectr ? a.ectr[e] : e;
  if (c < 0 || c >= a.n_ctr) {   // invalid centre index: NaN output, status flag
    const int nout = (a.what == QBX_GRAD ? 2 : 1) * a.nrhs;
    cplx* o = reinterpret_cast<cplx*>(a.out) + (size_t)e * nout;
    for (int i = 0; i < nout; ++i) o[i] = cplx{NAN, NAN};
    atomicOr(a.status, 2);
    return;
  }
  double x, y;
  if (a.ex) {
    x = a.ex[e];
    y = a.ey[e];
  } else {
    x = a.tx[c % a.n_tgt];
    y = a.ty[c % a.n_tgt];
  }
  const double dx = x - a.cx[c], dy = y - a.cy[c];
  const double rho = hypot(dx, dy);
  const cplx eith = rho > 0.0 ? cplx{dx / rho, dy / rho} : cplx{1.0, 0.0};
  T J[QBX_MAX_P + 2];
  const T kr = make_kr<T>(a.kre, a.kim, rho);
  if (rho > 0.0) besselj_column<T>(kr, a.p + 1, J, 1);
  else {
    for (int l = 0; l <= a.p + 1; ++l) sc_zero(J[l]);
    sc_set(J[0], 1.0);
  }
  cplx E[QBX_MAX_P + 2];   // e^{i m theta}, m = 0..p+1
  E[0] = cplx{1.0, 0.0};
  for (int m = 1; m <= a.p + 1; ++m) E[m] = E[m - 1] * eith;
  const int p = a.p, nl = 2 * p + 1;
  const cplx k = cplx{a.kre, a.kim};
  const cplx* alpha = reinterpret_cast<const cplx*>(a.alpha) + (size_t)c * nl * a.nrhs;
  cplx* out = reinterpret_cast<cplx*>(a.out);
  for (int r = 0; r < a.nrhs; ++r) {
    if (a.what == QBX_GRAD) {
      cplx up{0, 0}, um{0, 0};
      for (int l = -p; l <= p; ++l) {
        const cplx al = alpha[(size_t)(l + p) * a.nrhs + r];
        const int mp1 = l + 1, mm1 = l - 1;
        const cplx ep = mp1 >= 0 ? E[mp1] : conj(E[-mp1]);
        const cplx em = mm1 >= 0 ? E[mm1] : conj(E[-mm1]);
        up = up + al * (jc(J, mp1) * ep);
        um = um + al * (jc(J, mm1) * em);
      }
      up = -(k * up);
      um = k * um;
      const cplx gx = 0.5 * (up + um);
      const cplx d = up - um;
      const cplx gy = cplx{0.5 * d.im, -0.5 * d.re};   // d / (2i)
      out[((size_t)e * 2 + 0) * a.nrhs + r] = gx;
      out[((size_t)e * 2 + 1) * a.nrhs + r] = gy;
    } else {
      cplx u{0, 0};
      for (int l = -p; l <= p; ++l) {
        const cplx el = l >= 0 ? E[l] : conj(E[-l]);
        u = u + alpha[(size_t)(l + p) * a.nrhs + r] * (jc(J, l) * el);
      }
      out[(size_t)e * a.nrhs + r] = u;
    }
  }
}

cudaError_t launch_eval(const EvalArgs& a, cudaStream_t st) {
  const int threads = 128;
  const int blocks = (a.n_eval + threads - 1) / threads;
  if (a.kim == 0.0) k_eval<double><<<blocks, threads, 0, st>>>(a);
  else k_eval<cplx><<<blocks, threads, 0, st>>>(a);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Centre assignment for off-surface points (smallest |x-c|/r <= 1, lowest index).
// ---------------------------------------------------------------------------
// A CTA of eight warps holds 32 points, one per lane, and the warps share the
// centres; a centre is measured in FP64 only where FP32 (relative to the CTA's
// first point) leaves open whether its disc holds the point.  The all-FP64
// loop of one thread per point: 2.28 ms for 2048 points and centres.
constexpr int kAssignWarps = 8;
__global__ void __launch_bounds__(32 * kAssignWarps)
k_assign(int n, const double* xy, int n_ctr, const double* cx, const double* cy, const double* cr, int* out) {
  __shared__ float s_p[kAssignWarps][32][3];
  __shared__ double s_q[kAssignWarps][32];
  __shared__ int s_i[kAssignWarps][32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int e = blockIdx.x * 32 + lane, ee = min(e, n - 1), e0 = blockIdx.x * 32;
  const double x0 = xy[2 * e0], y0 = xy[2 * e0 + 1], x = xy[2 * ee], y = xy[2 * ee + 1];
  const float fx = (float)(x - x0), fy = (float)(y - y0);
  int best = -1;
  double bq = INFINITY;
  for (int base = warp * 32; base < n_ctr; base += kAssignWarps * 32) {
    __syncwarp();
    if (base + lane < n_ctr) {
      const float bx = (float)(cx[base + lane] - x0), by = (float)(cy[base + lane] - y0);
      s_p[warp][lane][0] = bx;
      s_p[warp][lane][1] = by;
      // a distance beyond this cannot lie inside the disc
      const float r = (float)cr[base + lane];
      s_p[warp][lane][2] = r > 0.0f ? r * 1.00001f + 4e-7f * (fabsf(bx) + fabsf(by)) : INFINITY;
    }
    __syncwarp();
    const float ex = 8e-7f * (fabsf(fx) + fabsf(fy));
    for (int j = 0; j < min(32, n_ctr - base); ++j) {
      const float dx = s_p[warp][j][0] - fx, dy = s_p[warp][j][1] - fy;
      if (sqrtf(fmaf(dx, dx, dy * dy)) > s_p[warp][j][2] + ex) continue;
      const int c = base + j;
      const double q = hypot(x - cx[c], y - cy[c]) / cr[c];
      if (q <= 1.0 && q < bq) {
        bq = q;
        best = c;
      }
    }
  }
  s_q[warp][lane] = bq;
  s_i[warp][lane] = best;
  __syncthreads();
  if (warp == 0 && e < n) {
    for (int w = 1; w < kAssignWarps; ++w) {   // ties to the lowest index
      const double q = s_q[w][lane];
      const int i = s_i[w][lane];
      if (i >= 0 && (best < 0 || q < bq || (q == bq && i < best))) {
        bq = q;
        best = i;
      }
    }
    out[e] = best;
  }
}

cudaError_t launch_assign(int n, const double* xy, int n_ctr, const double* cx, const double* cy,
                          const double* cr, int* out, cudaStream_t st) {
  k_assign<<<(n + 31) / 32, 32 * kAssignWarps, 0, st>>>(n, xy, n_ctr, cx, cy, cr, out);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Diagnostics: the device special functions at given points.
// ---------------------------------------------------------------------------
__global__ void k_debug_hankel(const cplx* z, int n, cplx* h0, cplx* h1) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const cplx zz = z[i];
  cplx a, b;
  if (zz.im == 0.0 && zz.re > 0.0) hankel01_real(zz.re, 1.0 / zz.re, sqrt(1.0 / zz.re), a, b);
  else hankel01_cplx(zz, a, b);
  h0[i] = a;
  h1[i] = b;
}

__global__ void k_debug_besselj(const cplx* z, int n, int nmax, cplx* j) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const cplx zz = z[i];
  if (zz.im == 0.0) {
    double J[QBX_MAX_P + 2];
    besselj_column<double>(zz.re, nmax, J, 1);
    for (int l = 0; l <= nmax; ++l) j[(size_t)i * (nmax + 1) + l] = cplx{J[l], 0.0};
  } else {
    cplx J[QBX_MAX_P + 2];
    besselj_column<cplx>(zz, nmax, J, 1);
    for (int l = 0; l <= nmax; ++l) j[(size_t)i * (nmax + 1) + l] = J[l];
  }
}

cudaError_t launch_debug_hankel(const void* z, int n, void* h0, void* h1, cudaStream_t st) {
  k_debug_hankel<<<(n + 127) / 128, 128, 0, st>>>((const cplx*)z, n, (cplx*)h0, (cplx*)h1);
  return cudaGetLastError();
}

cudaError_t launch_debug_besselj(const void* z, int n, int nmax, void* j, cudaStream_t st) {
  k_debug_besselj<<<(n + 127) / 128, 128, 0, st>>>((const cplx*)z, n, nmax, (cplx*)j);
  return cudaGetLastError();
}

}  // namespace qbx
