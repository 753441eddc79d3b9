// qbx_grad_d.cu -- storage-free grad D (Sec. 3.2, eq. dlpderiv): the
// gradient at the target of the D expansion about each centre, summed pair
// by pair without forming the coefficients (Sec. 3.3's remark that every
// source may add to the target sum directly).
//
// With x - c = r e^{i theta_t}, x_s - c = rho e^{i theta_s}, psi = theta_t -
// theta_s, the truncated Graf kernel is G_p = sum_{|l|<=p} H_l(k rho)
// e^{-i l theta_s} J_l(k r) e^{i l theta_t}.  Writing d = d_x - i d_y and
// dbar = d_x + i d_y, the Bessel identities dbar[Z_m e^{i m theta}] =
// -k Z_{m+1} e^{i(m+1) theta}, d[Z_m e^{i m theta}] = k Z_{m-1} e^{i(m-1) theta}
// (Z = J or H) give, for n_s . grad_{x_s} G_p differentiated at the target,
//   d D    =  (k^2/2) e^{-i theta_t} [-nu~ R(psi)  + conj(nu~) Q(-psi)],
//   dbar D = -(k^2/2) e^{ i theta_t} [-nu~ Q(psi)  + conj(nu~) R(-psi)],
// nu~ = (a + i b) e^{-i psi}, a = n_s . e_rho, b = n_s . e_theta, and
//   Q(psi) = sum_{m=-p+1}^{p+1} H_m J_m     e^{i m psi},
//   R(psi) = sum_{m=-p+1}^{p+1} H_m J_{m-2} e^{i m psi}.
// Folding +-m over |m| <= p-1 (H_{-m} = (-1)^m H_m, J likewise):
//   Q(+-psi) = H_0 J_0 + 2 sum_{m=1}^{p-1} J_m cos(m psi) H_m + edges,
//   R(+-psi) = H_0 J_2 + sum_{m=1}^{p-1} [(J_{m-2}+J_{m+2}) cos(m psi)
//              +- i (J_{m-2}-J_{m+2}) sin(m psi)] H_m + edges,
// the edges being the orders m = p, p+1 with e^{+-i m psi}.  Then
// grad = ((d D + dbar D)/2, i (d D - dbar D)/2).  Per order: three sums and
// the H and Chebyshev recurrences; one rhs per pass with the weighted
// density multiplied into the seeds H0, H1 (every sum is linear in H_m).
#include <cuda_runtime.h>
#include "qbx_apply_impl.cuh"
#include "qbx_internal.h"

namespace qbx {
namespace {

constexpr int kGdWarps = 4;                  // warps per CTA, which take its sources in turn

// shared memory: columns J (J_0..J_{p+1}), C (J_{m-2}+J_{m+2})/2 and
// S (J_{m-2}-J_{m+2})/2 for m = 1..p-1 (row m), 32 centres wide; the warps' sums
template <typename T>
__host__ __device__ size_t gd_smem(int p) {
  return (size_t)((p + 2) + 2 * p) * 32 * sizeof(T) + 2 * 32 * 16;
}

template <typename T>
__device__ __forceinline__ T jl_signed(const T* cJ, int l) {   // J_l for l >= -1 from the column
  return l >= 0 ? cJ[l * 32] : rmul(cJ[32], -1.0);
}

// A CTA owns 32 centres of one side (one per lane); its warps take its share
// of the sources (all, or the block's near leaves: ApplyArgs::near) in turn.
template <typename T>
__global__ void __launch_bounds__(32 * kGdWarps) k_grad_d_fused(ApplyArgs a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int p = a.p;
  T* sJ = reinterpret_cast<T*>(smem_raw);
  T* sC = sJ + (p + 2) * 32;
  T* sS = sC + p * 32;
  cplx* s_sum = reinterpret_cast<cplx*>(sS + p * 32);   // [2][32]

  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  // work item (centre block of one side, source split), near-field splits first
  const int blks = (a.n_tgt + 31) / 32, nblk = blks * (a.n_ctr / a.n_tgt);
  const int unit = (int)(blockIdx.x % (unsigned)nblk), rank = (int)(blockIdx.x / (unsigned)nblk);
  const int side = unit / blks, blk = unit - side * blks;
  const bool active = blk * 32 + lane < a.n_tgt;
  const int t = active ? blk * 32 + lane : a.n_tgt - 1;
  const int c = side * a.n_tgt + t;
  const int* near = a.near ? a.near + (size_t)blk * a.near_stride : nullptr;
  int split = rank, v0, v1;
  if (near) {
    const long n = (long)a.near_cnt[3 * blk] * a.near_q_src;
    v0 = (int)(n * rank / a.nsplit);
    v1 = (int)(n * (rank + 1) / a.nsplit);
  } else {
    if (a.near_q_tgt > 0)
      split = near_first_split(rank, min(blk * 32 + 16, a.n_tgt - 1), a.near_q_tgt, a.near_q_src, a.src_per_split,
                               a.nsplit);
    v0 = split * a.src_per_split;
    v1 = min(a.src.n, v0 + a.src_per_split);
  }

  // ---- per-centre set-up ----
  const double cx = a.cx[c], cy = a.cy[c];
  double ux = a.tx[t] - cx, uy = a.ty[t] - cy;
  const double r = hypot(ux, uy);
  ux /= r;
  uy /= r;
  KW<T> kw;
  kw.init(a.kre, a.kim, a.hk_tab);
  const T kk = kw.kval();
  T* colJ = sJ + lane;
  T* colC = sC + lane;
  T* colS = sS + lane;
  if (warp == 0) {
    besselj_column<T>(rmul(kk, r), p + 1, colJ, 32);
    for (int m = 1; m <= p - 1; ++m) {
      const T jm2 = jl_signed(colJ, m - 2), jp2 = colJ[(m + 2) * 32];
      colC[m * 32] = rmul(sadd(jm2, jp2), 0.5);
      colS[m * 32] = rmul(sc_sub(jm2, jp2), 0.5);
    }
  }
  __syncthreads();
  const T J0 = colJ[0], J2 = colJ[2 * 32];
  // edge coefficients (halved: the Chebyshev values below are doubled)
  const T eQ0 = rmul(colJ[p * 32], 0.5), eQ1 = rmul(colJ[(p + 1) * 32], 0.5);
  const T eR0 = rmul(jl_signed(colJ, p - 2), 0.5), eR1 = rmul(colJ[(p - 1) * 32], 0.5);

  cplx accP{0.0, 0.0}, accM{0.0, 0.0};   // sums of the d and dbar brackets
  const double2* wd = reinterpret_cast<const double2*>(a.wd[0]) + a.rhs0;
  {
    for (int v = v0 + warp; v < v1; v += kGdWarps) {
      int s_ = v;
      if (near) {
        const int i = v / a.near_q_src;
        s_ = near[i] * a.near_q_src + (v - i * a.near_q_src);
      }
      const double dx = __ldg(a.src.x + s_) - cx, dy = __ldg(a.src.y + s_) - cy;
      const double nx = __ldg(a.src.nx + s_), ny = __ldg(a.src.ny + s_);
      const double2 w2 = __ldg(wd + (size_t)s_ * a.nrhs);
      const double rho2 = fma(dx, dx, dy * dy);
      double inv, rho, yq;
      kw.geom(rho2, inv, rho, yq);
      const double cs = fma(ux, dx, uy * dy) * inv;   // cos psi
      const double sn = fma(uy, dx, -ux * dy) * inv;  // sin psi
      const double av = fma(nx, dx, ny * dy) * inv;   // n_s . e_rho
      const double bv = fma(ny, dx, -nx * dy) * inv;  // n_s . e_theta
      cplx H0, H1;
      T twoz;
      kw.hankel_w(rho, inv, yq, cplx{w2.x, w2.y}, H0, H1, twoz);   // w H0, w H1
      // core sums over m = 1..p-1 with 2 cos(m psi), 2 sin(m psi)
      cplx SQ{0.0, 0.0}, CR{0.0, 0.0}, SR{0.0, 0.0};
      const double tw = 2.0 * cs;
      cplx Hm = H0, H = H1;
      T s = twoz;
      double cp = 2.0, cl = tw, sp = 0.0, sl = sn + sn;
      for (int m = 1; m < p; ++m) {
        const int o = m * 32;
        madd(SQ, rmul(colJ[o], cl), H);
        madd(CR, rmul(colC[o], cl), H);
        madd(SR, rmul(colS[o], sl), H);
        const cplx Hn = hrec(s, H, Hm);
        Hm = H;
        H = Hn;
        s = sadd(s, twoz);
        const double cn = fma(tw, cl, -cp), sq = fma(tw, sl, -sp);
        cp = cl;
        cl = cn;
        sp = sl;
        sl = sq;
      }
      // edges: orders p (H, cl, sl) and p + 1
      const cplx Hp1 = hrec(s, H, Hm);
      const double cl1 = fma(tw, cl, -cp), sl1 = fma(tw, sl, -sp);
      cplx A1Q{0.0, 0.0}, A2Q{0.0, 0.0}, A1R{0.0, 0.0}, A2R{0.0, 0.0};
      madd(A1Q, rmul(eQ0, cl), H);
      madd(A1Q, rmul(eQ1, cl1), Hp1);
      madd(A2Q, rmul(eQ0, sl), H);
      madd(A2Q, rmul(eQ1, sl1), Hp1);
      madd(A1R, rmul(eR0, cl), H);
      madd(A1R, rmul(eR1, cl1), Hp1);
      madd(A2R, rmul(eR0, sl), H);
      madd(A2R, rmul(eR1, sl1), Hp1);
      // Q(+-psi) = Qa +- i Qb, R(+-psi) = Ra +- i Rb
      cplx Qa = SQ + A1Q, Ra = CR + A1R;
      madd(Qa, J0, H0);
      madd(Ra, J2, H0);
      const cplx Qb = A2Q, Rb = SR + A2R;
      const cplx iQb{-Qb.im, Qb.re}, iRb{-Rb.im, Rb.re};
      // nu~ = (a + i b) e^{-i psi}
      const cplx nu{fma(av, cs, bv * sn), fma(bv, cs, -av * sn)};
      const cplx nuc = conj(nu);
      // d bracket: -nu~ R(psi) + conj(nu~) Q(-psi); dbar bracket: -nu~ Q(psi) + conj(nu~) R(-psi)
      cfma(accP, nuc, Qa - iQb);
      cfma(accP, -nu, Ra + iRb);
      cfma(accM, nuc, Ra - iRb);
      cfma(accM, -nu, Qa + iQb);
    }
  }
  // the warps' sums in warp order
  for (int w = 0; w < kGdWarps; ++w) {
    if (warp == w) {
      if (w > 0) {
        accP = s_sum[lane] + accP;
        accM = s_sum[32 + lane] + accM;
      }
      s_sum[lane] = accP;
      s_sum[32 + lane] = accM;
    }
    __syncthreads();
  }
  if (warp != kGdWarps - 1 || !active) return;
  // d D = (k^2/2) e^{-i theta_t} P, dbar D = -(k^2/2) e^{i theta_t} M (without the factor i/4)
  const cplx h = 0.5 * sc_mul(to_c(kk), to_c(kk));
  const cplx et{ux, uy};
  const cplx dD = h * (conj(et) * accP);
  const cplx dbD = -(h * (et * accM));
  const cplx gx = 0.5 * (dD + dbD);
  const cplx dm = dD - dbD;
  const cplx gy = cplx{-0.5 * dm.im, 0.5 * dm.re};
  cplx* part = reinterpret_cast<cplx*>(a.part);
  const size_t row = ((size_t)split * a.n_ctr + c) * 2;
  part[row * a.nrhs + a.rhs0] = gx;
  part[(row + 1) * a.nrhs + a.rhs0] = gy;
}

template <typename T>
cudaError_t launch_gd(const ApplyArgs& a, cudaStream_t st) {
  const size_t smem = gd_smem<T>(a.p);
  cudaError_t e = cudaFuncSetAttribute(k_grad_d_fused<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  const unsigned grid = (unsigned)apply_units(a.n_ctr, a.n_tgt) * (unsigned)a.nsplit;
  k_grad_d_fused<T><<<grid, 32 * kGdWarps, smem, st>>>(a);
  return cudaGetLastError();
}

template <typename T>
int occ_gd(int p) {
  const size_t smem = gd_smem<T>(p);
  int n = 0;
  if (cudaFuncSetAttribute(k_grad_d_fused<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess)
    return 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_grad_d_fused<T>, 32 * kGdWarps, smem) != cudaSuccess) return 0;
  return n;
}

}  // namespace

cudaError_t launch_grad_d_fused(const ApplyArgs& a, cudaStream_t st) {
  return a.kim == 0.0 ? launch_gd<double>(a, st) : launch_gd<cplx>(a, st);
}
size_t grad_d_fused_smem(bool ck, int p) { return ck ? gd_smem<cplx>(p) : gd_smem<double>(p); }
int grad_d_fused_occupancy(bool ck, int p) { return ck ? occ_gd<cplx>(p) : occ_gd<double>(p); }

}  // namespace qbx
