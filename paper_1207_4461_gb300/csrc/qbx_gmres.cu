// qbx_gmres.cu -- device kernels of the batched GMRES solve for the
// second-kind exterior Dirichlet (sound-soft) problem of Sec. 4.2:
//   (1/2) mu + D mu - i eta S mu = f   (eq. dirichlet-inteq with the exterior
//   sign, D and S as two-sided averages, Sec. 3.5 and Sec. 4.2),
// with unknowns scaled by the square roots of the target weights (Sec. 4.2:
// sqrt-weight unknowns).  Every system (right-hand side) has its own Krylov
// basis; the systems advance in lockstep so that one matvec call serves all.
// Vectors are [n][nrhs] complex; bases [m+1][n][nrhs].  Reductions add in a
// fixed order, so results are deterministic.
#include <cuda_runtime.h>
#include <math.h>
#include <stdio.h>
#include <cooperative_groups.h>
#include <algorithm>
#include "../../include/qbx.h"
#include "qbx_device.cuh"
#include "qbx_internal.h"

using namespace qbx;

namespace {

constexpr int kRedThreads = 256;
constexpr int kRedBlocks = 152;   // first-pass blocks (one per SM)

// x = y / sqrt(w)  (scaled unknowns -> density) or x = y * sqrt(w)
__global__ void k_scale_sqrtw(int n, int nrhs, const double* w, const cplx* in, cplx* out, int inverse) {
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= n * nrhs) return;
  const double s = sqrt(w[idx / nrhs]);
  out[idx] = (inverse ? 1.0 / s : s) * in[idx];
}

// y = sqrt(w) * (x_density / 2 + D - i eta S), x_density = x / sqrt(w);
// s == NULL: d holds (D - i eta S) x_density
__global__ void k_cfie_combine(int n, int nrhs, const double* w, const cplx* xden, const cplx* d, const cplx* s,
                               double eta_re, double eta_im, cplx* y) {
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= n * nrhs) return;
  const double sw = sqrt(w[idx / nrhs]);
  const cplx ie = cplx{-eta_im, eta_re};   // i eta
  cplx v = 0.5 * xden[idx] + d[idx];
  if (s) v = v - ie * s[idx];
  y[idx] = sw * v;
}

// partial dots: part[b][j][r] = sum_{i in block b's range} conj(V_j[i][r]) w[i][r],
// grid (kRedBlocks, nv): block (b, j) takes row range b of vector j.  Lanes
// own right-hand sides (rows of [n][nrhs] are read whole and coalesced):
// thread t takes rhs r0 + t % R and every S-th row of the range,
// S = blockDim / R; the S partial sums of each r are then added in a fixed
// order, so the result does not depend on timing.
__global__ void k_dots_pass1(int n, int nrhs, int nv, const cplx* V, const cplx* w, cplx* part) {
  extern __shared__ cplx sred[];
  const int j = blockIdx.y;
  const int per = (n + gridDim.x - 1) / gridDim.x;
  const int i0 = blockIdx.x * per, i1 = min(n, i0 + per);
  const int R = min(nrhs, (int)blockDim.x), S = blockDim.x / R;
  const int rr = threadIdx.x % R, sub = threadIdx.x / R;
  const cplx* Vj = V + (size_t)j * n * nrhs;
  for (int r0 = 0; r0 < nrhs; r0 += R) {
    const int r = r0 + rr;
    cplx acc{0.0, 0.0};
    if (sub < S && r < nrhs) {
#pragma unroll 4
      for (int i = i0 + sub; i < i1; i += S) acc = acc + conj(Vj[(size_t)i * nrhs + r]) * w[(size_t)i * nrhs + r];
    }
    sred[threadIdx.x] = acc;
    __syncthreads();
    if (sub == 0 && r < nrhs) {
      cplx tot = sred[rr];
      for (int q = 1; q < S; ++q) tot = tot + sred[q * R + rr];
      part[((size_t)blockIdx.x * nv + j) * nrhs + r] = tot;
    }
    __syncthreads();
  }
}

// one warp per product: its lanes take every 32nd partial sum, then a tree
__global__ void k_dots_pass2(int nblocks, int nrhs, int nv, const cplx* part, cplx* out) {
  const int jr = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  if (jr >= nv * nrhs) return;
  cplx acc{0.0, 0.0};
  for (int b = lane; b < nblocks; b += 32) acc = acc + part[(size_t)b * nv * nrhs + jr];
  for (int o = 16; o > 0; o >>= 1) {
    acc.re += __shfl_xor_sync(0xffffffffu, acc.re, o);
    acc.im += __shfl_xor_sync(0xffffffffu, acc.im, o);
  }
  if (lane == 0) out[jr] = acc;
}

// w -= sum_j V_j h[j][r]
__global__ void k_orth_update(int n, int nrhs, int nv, const cplx* V, const cplx* h, cplx* w) {
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= n * nrhs) return;
  const int r = idx % nrhs;
  cplx acc = w[idx];
  for (int j = 0; j < nv; ++j) acc = acc - V[(size_t)j * n * nrhs + idx] * h[(size_t)j * nrhs + r];
  w[idx] = acc;
}

// out[i][r] = a[r] * in[i][r] (a real per rhs; 0 where a is not finite)
__global__ void k_scale_cols(int n, int nrhs, const double* a, const cplx* in, cplx* out) {
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= n * nrhs) return;
  const double s = a[idx % nrhs];
  out[idx] = isfinite(s) ? s * in[idx] : cplx{0.0, 0.0};
}

// x += sum_j V_j y[j][r]
__global__ void k_combine(int n, int nrhs, int nv, const cplx* V, const cplx* y, cplx* x) {
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= n * nrhs) return;
  const int r = idx % nrhs;
  cplx acc = x[idx];
  for (int j = 0; j < nv; ++j) acc = acc + V[(size_t)j * n * nrhs + idx] * y[(size_t)j * nrhs + r];
  x[idx] = acc;
}

int gfail(int code, const char* what) {
  char buf[320];
  snprintf(buf, sizeof(buf), "qbx_gmres: %s", what);
  return host_fail(code, buf);
}

int gcuda(cudaError_t e, const char* what) {
  char buf[320];
  snprintf(buf, sizeof(buf), "qbx_gmres: %s: %s", what, cudaGetErrorString(e));
  return host_fail(QBX_ECUDA, buf);
}

inline unsigned blocks(long n) { return (unsigned)((n + 255) / 256); }

}  // namespace

extern "C" {

int qbx_vec_scale_sqrtw(int n, int nrhs, const double* w, const qbx_c64* in, qbx_c64* out, int inverse,
                        void* stream) {
  if (n < 0 || nrhs < 1 || !w || !in || !out) return gfail(QBX_EINVAL, "bad arguments to qbx_vec_scale_sqrtw");
  if (n == 0) return QBX_OK;
  k_scale_sqrtw<<<blocks((long)n * nrhs), 256, 0, (cudaStream_t)stream>>>(n, nrhs, w, (const cplx*)in, (cplx*)out,
                                                                          inverse);
  cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? QBX_OK : gcuda(e, "scale kernel");
}

int qbx_cfie_combine(int n, int nrhs, const double* w, const qbx_c64* xden, const qbx_c64* dmu,
                     const qbx_c64* smu, qbx_c64 eta, qbx_c64* y, void* stream) {
  if (n < 0 || nrhs < 1 || !w || !xden || !dmu || !y) return gfail(QBX_EINVAL, "bad arguments to qbx_cfie_combine");
  if (n == 0) return QBX_OK;
  k_cfie_combine<<<blocks((long)n * nrhs), 256, 0, (cudaStream_t)stream>>>(
      n, nrhs, w, (const cplx*)xden, (const cplx*)dmu, (const cplx*)smu, eta.re, eta.im, (cplx*)y);
  cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? QBX_OK : gcuda(e, "combine kernel");
}

int qbx_vec_dots(int n, int nrhs, int nv, const qbx_c64* V, const qbx_c64* w, qbx_c64* work, qbx_c64* out,
                 void* stream) {
  if (n < 1 || nrhs < 1 || nv < 1 || nv > 65535 || !V || !w || !work || !out)
    return gfail(QBX_EINVAL, "bad arguments to qbx_vec_dots");
  cudaStream_t st = (cudaStream_t)stream;
  k_dots_pass1<<<dim3(kRedBlocks, nv), kRedThreads, kRedThreads * sizeof(cplx), st>>>(n, nrhs, nv, (const cplx*)V,
                                                                            (const cplx*)w, (cplx*)work);
  k_dots_pass2<<<blocks(32 * (long)nv * nrhs), 256, 0, st>>>(kRedBlocks, nrhs, nv, (const cplx*)work, (cplx*)out);
  cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? QBX_OK : gcuda(e, "dot kernels");
}

size_t qbx_vec_dots_work_bytes(int nrhs, int nv) { return (size_t)kRedBlocks * nv * nrhs * 16; }

int qbx_vec_orth_update(int n, int nrhs, int nv, const qbx_c64* V, const qbx_c64* h, qbx_c64* w, void* stream) {
  if (n < 1 || nrhs < 1 || nv < 0 || !V || !h || !w) return gfail(QBX_EINVAL, "bad arguments to qbx_vec_orth_update");
  if (nv == 0) return QBX_OK;
  k_orth_update<<<blocks((long)n * nrhs), 256, 0, (cudaStream_t)stream>>>(n, nrhs, nv, (const cplx*)V,
                                                                          (const cplx*)h, (cplx*)w);
  cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? QBX_OK : gcuda(e, "orthogonalisation kernel");
}

int qbx_vec_scale_cols(int n, int nrhs, const double* a, const qbx_c64* in, qbx_c64* out, void* stream) {
  if (n < 1 || nrhs < 1 || !a || !in || !out) return gfail(QBX_EINVAL, "bad arguments to qbx_vec_scale_cols");
  k_scale_cols<<<blocks((long)n * nrhs), 256, 0, (cudaStream_t)stream>>>(n, nrhs, a, (const cplx*)in, (cplx*)out);
  cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? QBX_OK : gcuda(e, "scale kernel");
}

int qbx_vec_combine(int n, int nrhs, int nv, const qbx_c64* V, const qbx_c64* y, qbx_c64* x, void* stream) {
  if (n < 1 || nrhs < 1 || nv < 0 || !V || !y || !x) return gfail(QBX_EINVAL, "bad arguments to qbx_vec_combine");
  if (nv == 0) return QBX_OK;
  k_combine<<<blocks((long)n * nrhs), 256, 0, (cudaStream_t)stream>>>(n, nrhs, nv, (const cplx*)V, (const cplx*)y,
                                                                      (cplx*)x);
  cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? QBX_OK : gcuda(e, "combine kernel");
}

}  // extern "C"

// ---------------------------------------------------------------------------
// The solve: restarted GMRES(m) per right-hand side, all systems in lockstep,
// driven from the device.  Arnoldi by classical Gram-Schmidt with one
// re-orthogonalisation (CGS2); the Hessenberg columns, the Givens rotations,
// the residual estimates |g_{j+1}| / ||f||, the convergence test and the
// back-substitution of each restart cycle run on the device, so the host waits
// for it once per restart cycle.  The kernels of an Arnoldi step read the step index and
// the state (done, matvec count) from a control block in device memory and
// do nothing once the step is inactive (all systems converged, maxiter
// reached or the cycle full); with the assembled matrix one step is
// captured as a CUDA graph and launched `restart` times per cycle.
// ---------------------------------------------------------------------------
#include <vector>

namespace {

// control block
enum { C_J = 0, C_DONE, C_TOTAL, C_MAXITER, C_M, C_ACTIVE, C_NOTCONV, C_JDONE, C_TICKET, C_N };

struct Dev {
  void* p = nullptr;
  ~Dev() { cudaFree(p); }
};

struct GraphGuard {
  cudaGraph_t g = nullptr;
  cudaGraphExec_t x = nullptr;
  cudaStream_t cap = nullptr;
  ~GraphGuard() {
    if (x) cudaGraphExecDestroy(x);
    if (g) cudaGraphDestroy(g);
    if (cap) cudaStreamDestroy(cap);
  }
};

// after ctl[C_J], C_DONE or C_TOTAL changed: does the next step run?
__device__ void set_active(int* ctl) {
  ctl[C_ACTIVE] = (!ctl[C_DONE] && ctl[C_TOTAL] < ctl[C_MAXITER] && ctl[C_J] < ctl[C_M]) ? 1 : 0;
}

// s[0 .. R) = the sums over q < S of s[q R + .] in a fixed order (a tree over
// q); sub = this thread's q (threads with sub >= S only take part in the barriers)
template <typename V>
__device__ __forceinline__ void tree_sum(V* s, int R, int S, int sub) {
  for (int h = S; h > 1;) {
    const int half = (h + 1) >> 1;
    __syncthreads();
    if (sub < h - half) s[threadIdx.x] = s[threadIdx.x] + s[threadIdx.x + half * R];
    h = half;
  }
  __syncthreads();
}

constexpr int kDotCluster = 8, kDotThreads = 256, kDotRows = 76;   // CTAs per vector; threads; clusters

// h[jv][r] = <V_jv, V_{j+1}>, jv <= j.  A cluster of 8 CTAs per vector, its
// CTAs' sums added in rank order through distributed shared memory, so that
// one launch gives the finished products; 76 clusters (all resident at once)
// take the vectors in turn.  FP64-bound from some 20 vectors on (4 multiply-
// adds per element).  With 152 row ranges x (m + 1) vectors of CTAs, most of
// which had nothing to do, and a second kernel for the 152 sums, the products
// of one step at n = 1152, 16 right-hand sides took 28 us, now 8.
__global__ void __cluster_dims__(kDotCluster, 1, 1) __launch_bounds__(kDotThreads)
k_dots_step(int n, int nrhs, const cplx* __restrict__ V, const int* ctl, cplx* h) {
  if (!ctl[C_ACTIVE]) return;
  __shared__ cplx sred[kDotThreads];
  __shared__ cplx stot[2][kDotThreads];
  auto cluster = cooperative_groups::this_cluster();
  const int nv = ctl[C_J] + 1, rank = blockIdx.x;
  const size_t vec = (size_t)n * nrhs;
  const cplx* w = V + (size_t)nv * vec;
  const int per = (n + kDotCluster - 1) / kDotCluster;
  const int i0 = min(n, rank * per), i1 = min(n, i0 + per);
  const int R = min(nrhs, kDotThreads), S = kDotThreads / R;
  const int rr = threadIdx.x % R, sub = threadIdx.x / R;
  int buf = 0;
  for (int jv = blockIdx.y; jv < nv; jv += gridDim.y) {
    const cplx* Vj = V + (size_t)jv * vec;
    for (int r0 = 0; r0 < nrhs; r0 += R) {
      const int r = r0 + rr;
      cplx acc{0.0, 0.0};
      if (sub < S && r < nrhs) {
#pragma unroll 4
        for (int i = i0 + sub; i < i1; i += S) acc = acc + conj(Vj[(size_t)i * nrhs + r]) * w[(size_t)i * nrhs + r];
      }
      sred[threadIdx.x] = acc;
      tree_sum(sred, R, S, sub);
      if (sub == 0) stot[buf][rr] = sred[rr];
      cluster.sync();   // (a buffer is written again only after the next one's barrier)
      if (rank == 0 && sub == 0 && r < nrhs) {
        cplx tot = stot[buf][rr];
#pragma unroll
        for (int q = 1; q < kDotCluster; ++q) tot = tot + cluster.map_shared_rank(stot[buf], q)[rr];
        h[(size_t)jv * nrhs + r] = tot;
      }
      buf ^= 1;
    }
  }
  cluster.sync();   // rank 0 has read the others' shared memory
}

constexpr int kOrthThreads = 512;

// V_{j+1} -= sum_{i <= j} V_i h[i][r]; NORM: also the partial ||V_{j+1}||^2 of
// the CTA's rows, part[block][r].  152 row ranges; where a range has fewer
// rows than the CTA has room for, up to 8 threads share an element's vectors
// (one warp alone reaches an eighth of the FP64 rate).
template <bool NORM>
__global__ void __launch_bounds__(kOrthThreads) k_orth_step(int n, int nrhs, cplx* __restrict__ V,
                                                            const cplx* __restrict__ h, const int* ctl, double* part) {
  if (!ctl[C_ACTIVE]) return;
  __shared__ cplx sred[kOrthThreads];
  __shared__ double snrm[kOrthThreads];
  const int nv = ctl[C_J] + 1;
  const size_t vec = (size_t)n * nrhs;
  cplx* w = V + (size_t)nv * vec;
  const int per = (n + gridDim.x - 1) / gridDim.x;
  const int i0 = min(n, (int)blockIdx.x * per), i1 = min(n, i0 + per);
  const int R = min(nrhs, kOrthThreads), S = kOrthThreads / R;
  const int rows = min(per, S), Q = min(8, S / rows);   // rows per pass, threads per element
  const int rr = threadIdx.x % R, sub = threadIdx.x / R, row = sub % rows, qp = sub / rows;
  for (int r0 = 0; r0 < nrhs; r0 += R) {
    const int r = r0 + rr;
    double nrm = 0.0;
    for (int ib = i0; ib < i1; ib += rows) {
      const int i = ib + row;
      const bool act = qp < Q && r < nrhs && i < i1;
      const size_t idx = (size_t)i * nrhs + r;
      cplx acc{0.0, 0.0};
      if (act) {
        if (qp == 0) acc = w[idx];
#pragma unroll 4
        for (int q = qp; q < nv; q += Q) acc = acc - V[(size_t)q * vec + idx] * h[(size_t)q * nrhs + r];
      }
      if (Q > 1) {
        sred[threadIdx.x] = acc;
        __syncthreads();
        if (act && qp == 0)
          for (int q = 1; q < Q; ++q) acc = acc + sred[threadIdx.x + q * rows * R];
        __syncthreads();
      }
      if (act && qp == 0) {
        w[idx] = acc;
        if (NORM) nrm += abs2(acc);
      }
    }
    if (NORM) {
      snrm[threadIdx.x] = nrm;
      tree_sum(snrm, R, S, sub);
      if (sub == 0 && r < nrhs) part[(size_t)blockIdx.x * nrhs + r] = snrm[rr];
      __syncthreads();
    }
  }
}

// End of a step.  Every CTA adds the partial norms (in a fixed order) and
// scales its rows, V_{j+1} *= 1 / ||V_{j+1}|| (0 where not finite); the CTA
// that finishes last then takes the Hessenberg column of every system: h(i) =
// h1 + h2 (i <= j), h(j+1) = ||V_{j+1}||; the earlier rotations, a new one
// zeroing h(j+1), the updated g, the residual estimate |g_{j+1}| / ||f|| and
// the convergence test.  A rotation is (a, b) -> (conj(c) a + s b, c b - s a)
// with s real (h(j+1) is); only a <- c b - s a is a chain, two multiply-adds
// per rotation in one warp, the products around it are formed by all threads.
// One thread per system for the whole column in its own launch took 21 us at
// 60 steps of 16 systems, inside this kernel from registers 18 with norm and
// scaling; now 10.
constexpr int kRotItems = 1024, kRotRhs = 128;
__global__ void __launch_bounds__(256) k_finish_step(int n, int nrhs, int m, cplx* __restrict__ V,
                                                     const double* __restrict__ part, int npart, const cplx* __restrict__ h1,
                                                     const cplx* __restrict__ h2, double* hn, cplx* __restrict__ Hm,
                                                     cplx* __restrict__ cs, cplx* __restrict__ sn, cplx* gv, const double* fnorm, double* rel, double tol,
                                                     int* ctl) {
  if (!ctl[C_ACTIVE]) return;
  __shared__ double s[256];
  __shared__ int s_last;
  const int j = ctl[C_J];
  cplx* w = V + (size_t)(j + 1) * n * nrhs;
  const int per = (n + gridDim.x - 1) / gridDim.x;
  const int i0 = min(n, (int)blockIdx.x * per), i1 = min(n, i0 + per);
  const int R = min(nrhs, 256), S = 256 / R;
  const int rr = threadIdx.x % R, sub = threadIdx.x / R;
  for (int r0 = 0; r0 < nrhs; r0 += R) {
    const int r = r0 + rr;
    double acc = 0.0;
    if (sub < S && r < nrhs) {
#pragma unroll 4
      for (int b = sub; b < npart; b += S) acc += part[(size_t)b * nrhs + r];
    }
    s[threadIdx.x] = acc;
    tree_sum(s, R, S, sub);
    const double hnn = sqrt(fmax(s[rr], 0.0));
    const double a = hnn > 0.0 ? 1.0 / hnn : 0.0;
    if (sub < S && r < nrhs) {
      if (blockIdx.x == 0 && sub == 0) hn[r] = hnn;
      for (int i = i0 + sub; i < i1; i += S) {
        const size_t idx = (size_t)i * nrhs + r;
        w[idx] = isfinite(a) ? a * w[idx] : cplx{0.0, 0.0};
      }
    }
    __syncthreads();
  }
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) s_last = atomicAdd(&ctl[C_TICKET], 1) == (int)gridDim.x - 1;
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  __shared__ cplx s_u[kRotItems], s_a[kRotItems + kRotRhs];   // c b, a before and after each rotation: [i][r]
  __shared__ double s_d[kRotItems];
  int open = 0;
  for (int r0 = 0; r0 < nrhs; r0 += kRotRhs) {
    const int nt = min(kRotRhs, nrhs - r0), I = kRotItems / nt;   // systems, rotations at a time
    auto hcol = [&](int i, int r) { return h1[(size_t)i * nrhs + r] + h2[(size_t)i * nrhs + r]; };
    __syncthreads();
    if (threadIdx.x < nt) s_a[threadIdx.x] = hcol(0, r0 + threadIdx.x);
    for (int ib = 0; ib < j; ib += I) {
      const int ni = min(I, j - ib);
      for (int e = threadIdx.x; e < ni * nt; e += 256) {
        const int i = ib + e / nt, r = r0 + e % nt;
        s_u[e] = cs[(size_t)i * nrhs + r] * hcol(i + 1, r);
        s_d[e] = sn[(size_t)i * nrhs + r].re;
      }
      __syncthreads();
      if (threadIdx.x < nt) {
        cplx a = s_a[threadIdx.x];
        for (int e = threadIdx.x; e < ni * nt; e += nt) {
          a = cplx{fma(-s_d[e], a.re, s_u[e].re), fma(-s_d[e], a.im, s_u[e].im)};
          s_a[e + nt] = a;
        }
      }
      __syncthreads();
      for (int e = threadIdx.x; e < ni * nt; e += 256) {
        const int i = ib + e / nt, r = r0 + e % nt;
        Hm[((size_t)i * m + j) * nrhs + r] = conj(cs[(size_t)i * nrhs + r]) * s_a[e] + s_d[e] * hcol(i + 1, r);
      }
      __syncthreads();
      if (threadIdx.x < nt) s_a[threadIdx.x] = s_a[ni * nt + threadIdx.x];
    }
    if (threadIdx.x < nt) {
      const int r = r0 + threadIdx.x;
      const cplx a = s_a[threadIdx.x];
      const double hnn = __ldcg(hn + r);
      const double den = sqrt(abs2(a) + hnn * hnn);
      const cplx c = den > 0.0 ? (1.0 / den) * a : cplx{1.0, 0.0};
      const double d = den > 0.0 ? hnn / den : 0.0;
      cs[(size_t)j * nrhs + r] = c;
      sn[(size_t)j * nrhs + r] = cplx{d, 0.0};
      Hm[((size_t)j * m + j) * nrhs + r] = conj(c) * a + cplx{d * hnn, 0.0};
      Hm[((size_t)(j + 1) * m + j) * nrhs + r] = cplx{0.0, 0.0};
      const cplx gj = gv[(size_t)j * nrhs + r];
      gv[(size_t)j * nrhs + r] = conj(c) * gj;
      const cplx gn = -(d * gj);
      gv[(size_t)(j + 1) * nrhs + r] = gn;
      const double e = fnorm[r] > 0.0 ? sqrt(abs2(gn)) / fnorm[r] : 0.0;
      rel[r] = e;
      if (!(e <= tol)) open = 1;
    }
  }
  open = __syncthreads_or(open);
  if (threadIdx.x == 0) {
    ctl[C_J] = j + 1;
    ctl[C_TOTAL] += 1;
    ctl[C_JDONE] = j + 1;
    ctl[C_DONE] = !open;
    ctl[C_TICKET] = 0;
    set_active(ctl);
  }
}

// start of a restart cycle, from hn = ||f~ - A x~||^2 per rhs: beta, the
// residual estimates, scl = 1/beta for V_0, g = (beta, 0, ...)
__global__ void k_cycle_init(int nrhs, int m, const cplx* hn, const double* fnorm, double* rel, double* scl, cplx* gv,
                             double tol, int* ctl) {
  const int r = blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= nrhs) return;
  const double beta = sqrt(fmax(hn[r].re, 0.0));
  scl[r] = beta > 0.0 ? 1.0 / beta : 0.0;
  const double e = fnorm[r] > 0.0 ? beta / fnorm[r] : 0.0;
  rel[r] = e;
  gv[r] = cplx{beta, 0.0};
  for (int i = 1; i <= m; ++i) gv[(size_t)i * nrhs + r] = cplx{0.0, 0.0};
  if (!(e <= tol)) atomicAdd(&ctl[C_NOTCONV], 1);
}

__global__ void k_cycle_init2(int* ctl) {
  ctl[C_J] = 0;
  ctl[C_JDONE] = 0;
  ctl[C_DONE] = ctl[C_NOTCONV] == 0;
  ctl[C_NOTCONV] = 0;
  set_active(ctl);
}

__global__ void k_fnorm(int nrhs, const cplx* hn, double* fnorm) {
  const int r = blockIdx.x * blockDim.x + threadIdx.x;
  if (r < nrhs) fnorm[r] = sqrt(fmax(hn[r].re, 0.0));
}

// y = H^{-1} g per system (upper triangular, jdone columns).  A CTA per system:
// with y_i known every thread takes its rows' product from g, so that the chain
// is one complex product and two barriers per column (one thread per system for
// the whole triangle: 266 us at 60 columns, now 38).  y holds g, then y.
__global__ void __launch_bounds__(128) k_backsolve(int nrhs, int m, const cplx* __restrict__ Hm,
                                                   const cplx* __restrict__ gv, cplx* y, const int* ctl) {
  const int r = blockIdx.x, jd = ctl[C_JDONE];
  __shared__ cplx s_y;
  // row l of thread l (mod 128): the running g_l, and 1 / H_ll of its first row
  for (int l = threadIdx.x; l < jd; l += 128) y[(size_t)l * nrhs + r] = gv[(size_t)l * nrhs + r];
  auto inv = [&](int i) {
    const cplx d = Hm[((size_t)i * m + i) * nrhs + r];
    return abs2(d) > 0.0 ? cdiv(cplx{1.0, 0.0}, d) : cplx{0.0, 0.0};
  };
  cplx own{0.0, 0.0}, id{0.0, 0.0};
  if (threadIdx.x < jd) {
    own = y[(size_t)threadIdx.x * nrhs + r];
    id = inv(threadIdx.x);
  }
  for (int i = jd - 1; i >= 0; --i) {
    cplx h{0.0, 0.0};
    if (threadIdx.x < i) h = Hm[((size_t)threadIdx.x * m + i) * nrhs + r];
    if (threadIdx.x == (i & 127)) {
      s_y = i < 128 ? own * id : y[(size_t)i * nrhs + r] * inv(i);
      y[(size_t)i * nrhs + r] = s_y;
    }
    __syncthreads();
    const cplx v = s_y;
    if (threadIdx.x < i) own = own - h * v;
    for (int l = threadIdx.x + 128; l < i; l += 128)
      y[(size_t)l * nrhs + r] = y[(size_t)l * nrhs + r] - Hm[((size_t)l * m + i) * nrhs + r] * v;
    __syncthreads();
  }
}

// x += sum_{i < jdone} V_i y[i][r]
__global__ void k_combine_cycle(int n, int nrhs, const cplx* V, const cplx* y, cplx* x, const int* ctl) {
  const long idx = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= (long)n * nrhs) return;
  const int r = (int)(idx % nrhs), nv = ctl[C_JDONE];
  cplx acc = x[idx];
  for (int q = 0; q < nv; ++q) acc = acc + V[(size_t)q * n * nrhs + idx] * y[(size_t)q * nrhs + r];
  x[idx] = acc;
}

// V_0 = f~ - w
__global__ void k_sub(long nel, const cplx* f, const cplx* w, cplx* out) {
  const long idx = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx < nel) out[idx] = f[idx] - w[idx];
}

}  // namespace

// Adense: the sqrt-weighted matrix from qbx_assemble_cfie (column-major), or
// NULL for matrix-free matvecs through qbx_apply_cfie.
static int solve_impl(qbx_plan* plan, const qbx_geom* g, qbx_c64 k, qbx_c64 eta, int p, const qbx_c64* Adense,
                      const qbx_c64* f, int nrhs, double tol, int restart, int maxiter, qbx_c64* mu, int* iters,
                      double* resid, void* stream) {
  if (!plan || !g || !f || !mu || nrhs < 1 || restart < 1 || maxiter < 1 || !(tol > 0.0))
    return gfail(QBX_EINVAL, "bad arguments to qbx_solve_exterior_dirichlet");
  const int n = g->n_tgt;
  const size_t vec = (size_t)n * nrhs;
  cudaStream_t st = (cudaStream_t)stream;
  const int m = restart;
  const size_t zw = Adense ? qbx_matmul_cm_work_bytes(n, nrhs) : 0;
  if (Adense && zw == 0) return gfail(QBX_ECUDA, "matrix product set-up failed");
  // one allocation: the basis, W, X~, F~, matrix-free: the density and
  // (D - i eta S) of it; the reductions' partial sums; small state: h1, h2
  // [(m+1)][nrhs], Hm [(m+1)][m][nrhs], cs, sn [m][nrhs], gv [(m+1)][nrhs],
  // y [m][nrhs], hn [nrhs] (complex); fnorm, rel, scl, hnorm [nrhs] (real);
  // the matrix product's splits; the control block
  const size_t nst = (size_t)nrhs * (2 * (m + 1) + (size_t)(m + 1) * m + 2 * m + (m + 1) + m + 1);
  Dev mem;
  size_t total_bytes = 0;
  auto room = [&](size_t b) {
    const size_t o = total_bytes;
    total_bytes += (b + 255) / 256 * 256;
    return o;
  };
  const size_t oV = room((size_t)(m + 1) * vec * 16), oW = room(vec * 16), oX = room(vec * 16), oF = room(vec * 16);
  const size_t oDEN = room(Adense ? 0 : vec * 16), oDM = room(Adense ? 0 : vec * 16);
  const size_t oWORK = room(qbx_vec_dots_work_bytes(nrhs, 1)), oST = room(nst * 16 + 4 * (size_t)nrhs * 8);
  const size_t oZW = room(zw), oCTL = room(C_N * sizeof(int));
  cudaError_t e = cudaMalloc(&mem.p, total_bytes);
  if (e != cudaSuccess) return gcuda(e, "allocation");
  char* base = (char*)mem.p;
  cplx *Vb = (cplx*)(base + oV), *W = (cplx*)(base + oW), *X = (cplx*)(base + oX), *F = (cplx*)(base + oF);
  cplx *DEN = (cplx*)(base + oDEN), *DM = (cplx*)(base + oDM), *WORK = (cplx*)(base + oWORK);
  void* ZW = base + oZW;
  cplx* h1 = (cplx*)(base + oST);
  cplx* h2 = h1 + (size_t)(m + 1) * nrhs;
  cplx* Hm = h2 + (size_t)(m + 1) * nrhs;
  cplx* cs = Hm + (size_t)(m + 1) * m * nrhs;
  cplx* sn = cs + (size_t)m * nrhs;
  cplx* gv = sn + (size_t)m * nrhs;
  cplx* yv = gv + (size_t)(m + 1) * nrhs;
  cplx* hn = yv + (size_t)m * nrhs;
  double* fnorm = (double*)(hn + nrhs);
  double* rel = fnorm + nrhs;
  double* scl = rel + nrhs;
  double* hnorm = scl + nrhs;
  int* ctl = (int*)(base + oCTL);
  {
    const int init[C_N] = {0, 0, 0, maxiter, m, 0, 0, 0, 0};
    e = cudaMemcpyAsync(ctl, init, sizeof(init), cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);   // (init lives on the host stack)
    if (e != cudaSuccess) return gcuda(e, "control block");
  }
  const unsigned ebl = blocks((long)vec), rbl = (unsigned)((nrhs + 127) / 128);
  int rc;
  // scaled right-hand side and initial guess: f~ = sqrt(w) f, x~ = sqrt(w) mu
  if ((rc = qbx_vec_scale_sqrtw(n, nrhs, g->tgt_w, f, (qbx_c64*)F, 0, stream))) return rc;
  if ((rc = qbx_vec_scale_sqrtw(n, nrhs, g->tgt_w, mu, (qbx_c64*)X, 0, stream))) return rc;
  // y = A~ x~ : density x~/sqrt(w), (D - i eta S) two-sided with the two
  // kernel values of each pair combined (qbx_apply_cfie), plus x/2; or one
  // complex matrix product with the assembled A~ (qbx_matmul_cm)
  auto matvec = [&](const qbx_c64* xs, qbx_c64* y, cudaStream_t s) -> int {
    int r;
    if (Adense) return qbx_matmul_cm(n, nrhs, Adense, xs, y, ZW, zw, s);
    if ((r = qbx_vec_scale_sqrtw(n, nrhs, g->tgt_w, xs, (qbx_c64*)DEN, 1, s))) return r;
    if ((r = qbx_apply_cfie(plan, g, k, eta, p, (qbx_c64*)DEN, nrhs, (qbx_c64*)DM, s))) return r;
    return qbx_cfie_combine(n, nrhs, g->tgt_w, (qbx_c64*)DEN, (qbx_c64*)DM, nullptr, eta, y, s);
  };
  // one Arnoldi step on stream s, every kernel gated by the control block:
  // V_{j+1} = A~ V_j, CGS2 against V_0..V_j, the norm, V_{j+1} normalised, the
  // Givens update and the convergence test.  jh: the step's j where the host
  // has to know it (matrix-free).
  auto step = [&](cudaStream_t s, int jh) -> int {
    if (Adense) {
      if (int r = matmul_cm_step(n, nrhs, Adense, (qbx_c64*)Vb, ZW, zw, ctl + C_ACTIVE, ctl + C_J, s)) return r;
    } else {
      cplx* vj = Vb + (size_t)jh * vec;
      if (int r = matvec((qbx_c64*)vj, (qbx_c64*)(vj + vec), s)) return r;   // (host-checked: runs only when active)
    }
    const dim3 dots(kDotCluster, (unsigned)std::min(m, kDotRows));
    k_dots_step<<<dots, kDotThreads, 0, s>>>(n, nrhs, Vb, ctl, h1);   // CGS2
    k_orth_step<false><<<kRedBlocks, kOrthThreads, 0, s>>>(n, nrhs, Vb, h1, ctl, nullptr);
    k_dots_step<<<dots, kDotThreads, 0, s>>>(n, nrhs, Vb, ctl, h2);
    k_orth_step<true><<<kRedBlocks, kOrthThreads, 0, s>>>(n, nrhs, Vb, h2, ctl, (double*)WORK);
    k_finish_step<<<kRedBlocks, 256, 0, s>>>(n, nrhs, m, Vb, (const double*)WORK, kRedBlocks, h1, h2, hnorm, Hm, cs, sn,
                                             gv, fnorm, rel, tol, ctl);
    cudaError_t ee = cudaGetLastError();
    return ee == cudaSuccess ? QBX_OK : gcuda(ee, "Arnoldi step kernels");
  };
  // ||f~|| per rhs
  if ((rc = qbx_vec_dots(n, nrhs, 1, (qbx_c64*)F, (qbx_c64*)F, (qbx_c64*)WORK, (qbx_c64*)hn, stream)))
    return rc;
  k_fnorm<<<rbl, 128, 0, st>>>(nrhs, hn, fnorm);
  // the assembled operator: one Arnoldi step as a CUDA graph
  GraphGuard gg;
  if (Adense) {
    e = cudaStreamCreateWithFlags(&gg.cap, cudaStreamNonBlocking);
    if (e == cudaSuccess) e = cudaStreamBeginCapture(gg.cap, cudaStreamCaptureModeRelaxed);
    if (e != cudaSuccess) return gcuda(e, "graph capture");
    rc = step(gg.cap, 0);
    e = cudaStreamEndCapture(gg.cap, &gg.g);
    if (rc) return rc;
    if (e == cudaSuccess) e = cudaGraphInstantiate(&gg.x, gg.g, 0);
    if (e != cudaSuccess) return gcuda(e, "Arnoldi step graph");
  }
  int hctl[C_N] = {0};
  bool done = false;
  int total = 0;
  while (!done && total < maxiter) {
    // r = f~ - A~ x~, beta, V_0 = r / beta, g = beta e_1
    if ((rc = matvec((qbx_c64*)X, (qbx_c64*)W, st))) return rc;
    k_sub<<<ebl, 256, 0, st>>>((long)vec, (const cplx*)F, (const cplx*)W, Vb);
    if ((rc = qbx_vec_dots(n, nrhs, 1, (qbx_c64*)Vb, (qbx_c64*)Vb, (qbx_c64*)WORK, (qbx_c64*)hn, stream)))
      return rc;
    k_cycle_init<<<rbl, 128, 0, st>>>(nrhs, m, hn, fnorm, rel, scl, gv, tol, ctl);
    k_cycle_init2<<<1, 1, 0, st>>>(ctl);
    if ((rc = qbx_vec_scale_cols(n, nrhs, scl, (qbx_c64*)Vb, (qbx_c64*)Vb, stream))) return rc;
    if (Adense) {
      for (int j = 0; j < m; ++j) {   // gated steps: those after convergence do nothing
        e = cudaGraphLaunch(gg.x, st);
        if (e != cudaSuccess) return gcuda(e, "Arnoldi step graph launch");
      }
    } else {
      for (int j = 0; j < m; ++j) {   // one host check per step (each step is a full QBX apply)
        e = cudaMemcpyAsync(hctl, ctl, sizeof(hctl), cudaMemcpyDeviceToHost, st);
        if (e == cudaSuccess) e = cudaStreamSynchronize(st);
        if (e != cudaSuccess) return gcuda(e, "control block copy");
        if (hctl[C_DONE] || hctl[C_TOTAL] >= maxiter || hctl[C_J] >= m) break;
        if ((rc = step(st, hctl[C_J]))) return rc;
      }
    }
    // y = H^{-1} g per system; x~ += V y
    k_backsolve<<<nrhs, 128, 0, st>>>(nrhs, m, Hm, gv, yv, ctl);
    k_combine_cycle<<<ebl, 256, 0, st>>>(n, nrhs, Vb, yv, (cplx*)X, ctl);
    e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaMemcpyAsync(hctl, ctl, sizeof(hctl), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);   // the one wait of the cycle
    if (e != cudaSuccess) return gcuda(e, "end of restart cycle");
    done = hctl[C_DONE] != 0;
    total = hctl[C_TOTAL];
  }
  // mu = x~ / sqrt(w); residual estimates of the last cycle
  if ((rc = qbx_vec_scale_sqrtw(n, nrhs, g->tgt_w, (qbx_c64*)X, mu, 1, stream))) return rc;
  if (resid) e = cudaMemcpyAsync(resid, rel, (size_t)nrhs * 8, cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) return gcuda(e, "final sync");
  if (iters) *iters = total;
  if (!done) return gfail(QBX_ENOCONV, "GMRES did not reach the tolerance within maxiter iterations");
  return QBX_OK;
}

extern "C" int qbx_solve_exterior_dirichlet(qbx_plan* plan, const qbx_geom* g, qbx_c64 k, qbx_c64 eta, int p,
                                            const qbx_c64* f, int nrhs, double tol, int restart, int maxiter,
                                            qbx_c64* mu, int* iters, double* resid, void* stream) {
  return solve_impl(plan, g, k, eta, p, nullptr, f, nrhs, tol, restart, maxiter, mu, iters, resid, stream);
}

extern "C" int qbx_solve_exterior_dirichlet_assembled(qbx_plan* plan, const qbx_geom* g, const qbx_c64* A,
                                                      const qbx_c64* f, int nrhs, double tol, int restart,
                                                      int maxiter, qbx_c64* mu, int* iters, double* resid,
                                                      void* stream) {
  if (!A) return gfail(QBX_EINVAL, "NULL matrix");
  return solve_impl(plan, g, qbx_c64{1.0, 0.0}, qbx_c64{0.0, 0.0}, 0, A, f, nrhs, tol, restart, maxiter, mu, iters,
                    resid, stream);
}
