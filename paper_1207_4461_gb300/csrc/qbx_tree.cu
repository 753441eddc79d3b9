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
__global__ void __launch_bounds__(256) k_tree_nodes(TreeArgs q) {
  const TreeArgs& a = q.inst ? q.inst[blockIdx.z] : q;
  __shared__ float s_red[8];
  const int id = blockIdx.x;
  if (id >= a.off[a.lev]) return;
  int l = 0;
  while (id >= a.off[l + 1]) ++l;
  const int j = id - a.off[l];
  const int s0 = (j << l) * a.q_src, s1 = min(a.M, (j + 1) << l) * a.q_src;
  // discs: the node's points are the targets, each with its centres' discs
  const int nd = a.discs ? a.n_ctr_n / a.n_src : 1;
  const double* px = a.discs ? a.dcx : a.sx;
  const double* py = a.discs ? a.dcy : a.sy;
  const double x0 = px[s0], y0 = py[s0];
  float xa = -INFINITY, xb = -INFINITY, ya = -INFINITY, yb = -INFINITY, bad = 0.0f;   // max of -x, x, -y, y
  for (int sd = 0; sd < nd; ++sd)
    for (int s = s0 + threadIdx.x; s < s1; s += 256) {
      const float x = (float)(px[sd * a.n_src + s] - x0), y = (float)(py[sd * a.n_src + s] - y0);
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
  const double zx = x0 + (double)(0.5f * (xb - xa)), zy = y0 + (double)(0.5f * (yb - ya));
  float r = 0.0f;
  for (int s = s0 + threadIdx.x; s < s1; s += 256) {
    if (!a.discs) {
      const float dx = (float)(a.sx[s] - zx), dy = (float)(a.sy[s] - zy);
      r = fmaxf(r, sqrtf(fmaf(dx, dx, dy * dy)));
      continue;
    }
    for (int sd = 0; sd < nd; ++sd) {
      const double cx = a.dcx[sd * a.n_src + s], cy = a.dcy[sd * a.n_src + s];
      const float dx = (float)(cx - zx), dy = (float)(cy - zy);
      const float ex = (float)(a.sx[s] - cx), ey = (float)(a.sy[s] - cy);
      const float v = sqrtf(fmaf(dx, dx, dy * dy)) + sqrtf(fmaf(ex, ex, ey * ey));
      if (!(v < 1e30f)) bad = 1.0f;
      r = fmaxf(r, v);
    }
  }
  r = block_reduce_max(r, s_red, 8);
  bad = block_reduce_max(bad, s_red, 8);
  if (threadIdx.x == 0) {
    double* n = a.node + 4 * (size_t)id;
    n[0] = zx;
    n[1] = zy;
    n[2] = bad > 0.0f ? INFINITY : (double)(r * 1.00001f);
    n[3] = 0.0;
  }
}

// Super-blocks: a node that is far from 2^B consecutive blocks
// of targets goes into one expansion about them all, which the blocks take up
// as one more entry (k_tree_local), instead of into every block's own.  At 256
// panels, k = 40: 49 entries per block become 8, and 20 per block in the super-
// blocks (12 curves, 64 columns: 17.9 -> 11.4 ms of local expansions; teardrop,
// k = 30: 4.4 -> 2.4).  First their discs: one CTA per super-block.
__global__ void __launch_bounds__(256) k_tree_super(TreeArgs q) {
  const TreeArgs& a = q.inst ? q.inst[blockIdx.z] : q;
  __shared__ float s_red[8];
  const int id = blockIdx.x;
  if (id >= a.n_sup) return;
  int B = 1;
  while (id >= a.sup_off[B + 1]) ++B;
  const int t0 = (id - a.sup_off[B]) * (32 << B), t1 = min(a.n_tgt, t0 + (32 << B));
  const double x0 = a.tx[t0], y0 = a.ty[t0];
  float xa = -INFINITY, xb = -INFINITY, ya = -INFINITY, yb = -INFINITY;
  for (int t = t0 + threadIdx.x; t < t1; t += 256) {
    const float x = (float)(a.tx[t] - x0), y = (float)(a.ty[t] - y0);
    xa = fmaxf(xa, -x);
    xb = fmaxf(xb, x);
    ya = fmaxf(ya, -y);
    yb = fmaxf(yb, y);
  }
  xa = block_reduce_max(xa, s_red, 8);
  xb = block_reduce_max(xb, s_red, 8);
  ya = block_reduce_max(ya, s_red, 8);
  yb = block_reduce_max(yb, s_red, 8);
  const double zx = x0 + (double)(0.5f * (xb - xa)), zy = y0 + (double)(0.5f * (yb - ya));
  float rd = 0.0f, rm = 0.0f, bad = 0.0f;
  for (int t = t0 + threadIdx.x; t < t1; t += 256)
    for (int c = t; c < a.n_ctr; c += a.n_tgt) {
      const float ex = (float)(a.tx[t] - a.cx[c]), ey = (float)(a.ty[t] - a.cy[c]);
      const float ox = (float)(a.cx[c] - zx), oy = (float)(a.cy[c] - zy);
      const float r = sqrtf(fmaf(ex, ex, ey * ey)) * 1.00001f, v = sqrtf(fmaf(ox, ox, oy * oy)) + r;
      if (!(v < 1e30f)) bad = 1.0f;
      rd = fmaxf(rd, v);
      rm = fmaxf(rm, r);
    }
  rd = block_reduce_max(rd, s_red, 8);
  rm = block_reduce_max(rm, s_red, 8);
  bad = block_reduce_max(bad, s_red, 8);
  if (threadIdx.x == 0) {
    double* n = a.node + 4 * (size_t)(a.off[a.lev] + a.n_blk + id);
    n[0] = zx;
    n[1] = zy;
    n[2] = bad > 0.0f ? INFINITY : (double)(rd * 1.00001f);   // (no node is far from such a one)
    n[3] = rm;
  }
}

// Their lists: for the super-blocks above this one and then itself, from the
// largest down, the nodes of its own size and twice it that are far from all
// its discs and not covered yet; its own go into its list in node order.
// Every super-block goes through its ancestors' tests itself (same
// instructions, same numbers), so all agree on what is covered.
__global__ void __launch_bounds__(256) k_super_lists(TreeArgs q) {
  const TreeArgs& a = q.inst ? q.inst[blockIdx.z] : q;
  const int id = blockIdx.x;
  if (id >= a.n_sup) return;
  __shared__ int s_n[8], s_at, s_ol;
  int B = 1;
  while (id >= a.sup_off[B + 1]) ++B;
  const int j = id - a.sup_off[B], lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  unsigned char* cov = a.scov + (size_t)id * a.M;
  int2* out = reinterpret_cast<int2*>(a.sloc) + (size_t)id * a.sup_stride;
  const float ka = (float)sqrt(a.kre * a.kre + a.kim * a.kim), ki = (float)a.kim;
  for (int i = threadIdx.x; i < a.M; i += 256) cov[i] = 0;
  if (threadIdx.x == 0) s_at = s_ol = 0;
  __syncthreads();
  for (int Bb = a.sup_lev; Bb >= B; --Bb) {
    const double* sb = a.node + 4 * (size_t)(a.off[a.lev] + a.n_blk + a.sup_off[Bb] + (j >> (Bb - B)));
    const double bx = sb[0], by = sb[1];
    const float rd = (float)sb[2] * 1.00001f, rm = (float)sb[3];
    for (int l = min(Bb + a.sup_c + 1, a.lev - 1); l >= Bb + a.sup_c; --l) {
      const int nl = a.off[l + 1] - a.off[l];
      for (int i0 = 0; i0 < nl; i0 += 256) {
        const int i = i0 + threadIdx.x;
        int code = 0;
        if (i < nl && !cov[i << l]) {
          const double* n = a.node + 4 * (size_t)(a.off[l] + i);
          const float dx = (float)(n[0] - bx), dy = (float)(n[1] - by), R = (float)n[2] * 1.00001f;
          const float d = 0.99999f * sqrtf(fmaf(dx, dx, dy * dy)), dl = d - R, dm = d - rd, rho = dl - rd;
          if (dl > 1.34f * rd && dm > 1.34f * R && rho > 1.34f * rm) {
            const int oq = series_order(ka * rd, ka * dl, rd / dl, expf(2.0f * ki * rd), a.nd, kTreeP);
            const int om = series_order(ka * R, ka * dm, R / dm, expf(2.0f * ki * R), a.nd, kTreeP);
            int ol = rm > 0.0f ? series_order(ka * rm, ka * rho, rm / rho, expf(2.0f * ki * rm), a.nd, a.pl) : 0;
            bool ok = oq <= kTreeP && om <= kTreeP;
            if (a.eta > 0.0) ok = ok && rho >= 1.00001f * (float)a.eta * rm && ol <= a.pl;   // (all by the smooth rule)
            else ol = min(ol, a.p);
            // H of order om + ol and the moments of order om stay in FP64's range
            const float no = (float)(om + max(ol, oq));
            ok = ok && no * log10f(fmaxf(2.0f * no / (2.7f * ka * dm), 1.0f)) < 280.0f &&
                 (float)om * log10f(fmaxf(2.0f * om / (2.7f * ka * R), 1.0f)) < 280.0f;
            if (ok) code = om | oq << 8 | ol << 16 | 1 << 24;
          }
        }
        if (Bb == B) {
          const unsigned mine = __ballot_sync(0xffffffffu, code != 0);
          if (lane == 0) s_n[warp] = __popc(mine);
          __syncthreads();
          int at = s_at;
          for (int w = 0; w < warp; ++w) at += s_n[w];
          if (code) {
            out[at + __popc(mine & ((1u << lane) - 1))] = make_int2(a.off[l] + i, code & 0xffff);
            atomicMax(&s_ol, code >> 16 & 0xff);
          }
          __syncthreads();
          if (threadIdx.x == 0)
            for (int w = 0; w < 8; ++w) s_at += s_n[w];
          __syncthreads();
        }
        if (code)
          for (int v = i << l; v < min(a.M, (i + 1) << l); ++v) cov[v] = 1;
      }
      __syncthreads();
    }
  }
  if (threadIdx.x == 0) {
    a.scnt[2 * id] = s_at;
    a.scnt[2 * id + 1] = s_ol;
  }
}

// Lists: one CTA per block of 32 targets, one thread per leaf.  A leaf's
// thread looks from the largest node down for the first that is far from the
// block; the first leaf of that node names it.  In leaf order, so the sums
// do not depend on timing.
constexpr int kListWarps = 8;
constexpr int kSupMinLeaves = 128;   // fewer: no node of that size is far from a super-block
__global__ void __launch_bounds__(32 * kListWarps) k_tree_lists(TreeArgs q) {
  const TreeArgs& a = q.inst ? q.inst[blockIdx.z] : q;
  if (blockIdx.x >= a.n_blk) return;
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

  const unsigned char* cov = a.n_sup ? a.scov + (size_t)(a.sup_off[1] + (b >> 1)) * a.M : nullptr;   // by super-blocks

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
    // (evaluation points, rm = 0: the field itself)
    int ol = rm > 0.0f ? series_order(ka * rm, ka * rho, rm / rho, expf(2.0f * ki * rm), a.nd, a.pl) : 0;
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
    // (stored coefficients: a node taken directly goes into every order l <= p)
    const float no = (float)(om + (a.all_l && !oq ? a.p : max(ol, oq)));
    if (!(no * log10f(fmaxf(2.0f * no / (2.7f * ka * dm), 1.0f)) < 280.0f) ||
        !((float)om * log10f(fmaxf(2.0f * om / (2.7f * ka * R), 1.0f)) < 280.0f))
      return 0;
    return om | ol << 8 | oq << 16 | 1 << 24;
  };

  for (int base = 0; base < a.M; base += 32 * kListWarps) {
    const int j = base + threadIdx.x;
    int code = 0, l = a.lev - 1;
    const bool covered = cov && j < a.M && cov[j];
    if (j < a.M && !covered) {
      for (; l >= 0; --l) {
        if (cov) {   // no leaf of the node may be covered (covered are whole nodes of level sup_c + 1 and up)
          bool hit = false;
          for (int i = j >> l << l; i < min(a.M, ((j >> l) + 1) << l) && !hit; i += 2 << a.sup_c) hit = cov[i];
          if (hit) continue;
        }
        code = test(a.off[l] + (j >> l));
        if (code) break;
      }
    }
    if (a.only_loc && !(code >> 16 & 0xff)) code = 0;
    const bool is_near = j < a.M && !code && !covered;
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
    bool sup = false;
    for (int B = 1; a.n_sup && B <= a.sup_lev; ++B) {
      const int* sc = a.scnt + 2 * (a.sup_off[B] + (b >> B));
      if (sc[0] == 0) continue;
      sup = true;
      s_ord[0] = kTreeP;
      s_ord[1] = max(s_ord[1], sc[1]);
    }
    if (s_at[2] > 0 || sup)   // the block's local expansion, after the far nodes
      far[nf++] = make_int2(a.off[a.lev] + b, s_ord[0] | s_ord[1] << 8 | 1 << 16);
    a.cnt[3 * b] = s_at[0];
    a.cnt[3 * b + 1] = nf;
    a.cnt[3 * b + 2] = s_at[2];
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

// H0, H1 at k |v|, v = (ax - bx, ay - by), with v's, its length's and the
// product's rounding carried to first order (H_0' = -H_1, H_1' = H_0 - H_1/z).
// All sources of a cluster share one argument, so its rounding (z eps in the
// phase) does not average out over them as it does pair by pair; 30
// instructions per node (D at 12000 points, k = 16: off by 6.8e-15 without,
// 3.2e-15 with it; pair by pair 4.0e-15).
template <typename T>
__device__ __forceinline__ void far_hankel(const KW<T>& kw, const T kk, double ax, double bx, double ay, double by,
                                           double& ct, double& st, cplx& h0, cplx& h1, T& twoz) {
  const double vx = ax - bx, vy = ay - by;
  const double tx = vx - ax, ty = vy - ay;
  const double ex = (ax - (vx - tx)) - (bx + tx), ey = (ay - (vy - ty)) - (by + ty);   // rounding of v
  const double xx = vx * vx, d2 = fma(vy, vy, xx);
  double inv, rho, yq;
  kw.geom(d2, inv, rho, yq);
  kw.hankel(rho, inv, yq, h0, h1, twoz);
  ct = vx * inv;
  st = vy * inv;
  // |v|^2 - rho^2, the larger square's product exact
  const double yy = vy * vy, s = xx + yy, ts = s - xx;
  const double es = (xx - (s - ts)) + (yy - ts) + (fma(vx, vx, -xx) + fma(vy, vy, -yy)) + 2.0 * fma(vx, ex, vy * ey);
  const double rl = 0.5 * inv * (fma(-rho, rho, s) + es);   // rho's rounding
  // z = k rho: the product's rounding and k rl
  T d;
  if constexpr (IsCplx<T>::value) {
    const double zr = kk.re * rho, zi = kk.im * rho;
    d = cplx{fma(kk.re, rho, -zr) + kk.re * rl, fma(kk.im, rho, -zi) + kk.im * rl};
  } else {
    const double z = kk * rho;
    d = fma(kk, rho, -z) + kk * rl;
  }
  const cplx g0 = h0, g1 = h1;
  msub(h0, d, g1);
  madd(h1, d, g0);
  msub(h1, sc_mul(d, rmul(twoz, 0.5)), g1);
}

// Waves of one far entry (index, orders om | ol << 8 | local << 16) at this
// lane's centre, v = c - z: H_n(k d), or J_n(k d) for a local expansion,
// n <= om + ol + 1, stride 32; the direction Theta of v; and for m = lane the
// orders l that order m needs.
template <typename T>
__device__ __forceinline__ void far_waves(const KW<T>& kw, const T kk, float ka, int2 ent, int nder, double kim,
                                          const double* nd, double cx, double cy, double r, cplx* sH, double& ct,
                                          double& st, int& lmax) {
  const int om = ent.y & 0xff, ol = ent.y >> 8 & 0xff, lane = threadIdx.x & 31;
  const bool local = ent.y >> 16;
  const int nH = om + ol + 1;   // (pairs of orders and the cut reach one further)
  lmax = ol;
  const double vx = cx - nd[0], vy = cy - nd[1];
  if (local) {
    const double rho = sqrt(fma(vx, vx, vy * vy));
    const bool off = rho > 0.0;   // (the centre may be the block's)
    ct = off ? vx / rho : 1.0;
    st = off ? vy / rho : 0.0;
    besselj_wave<T>(rmul(kk, rho), nH, sH);
    return;
  }
  cplx h0, h1;
  T twoz;
  far_hankel<T>(kw, kk, cx, nd[0], cy, nd[1], ct, st, h0, h1, twoz);
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
  const float fx = (float)vx, fy = (float)vy, rf = fmaf(fx, fx, fy * fy), rmin = warp_min(rf), rc = warp_max((float)r);
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
    float base = fm * __log2f(0.5f * ka * R) - lgammaf(fm + 1.0f) * 1.442695f - ex(nder) + 3.0f +
                 1.442695f * (float)kim * (R + rc);
    const float wm = nder ? fm / (ka * R) : 1.0f, wl = nder && rc > 0.0f ? 1.0f / (ka * rc) : 0.0f;
    lmax = 0;
    for (int l = 1; l <= ol; ++l) {
      base += lr - __log2f((float)l);
      if (base + ex(lane + l) + (nder == 2 ? 2.0f : 1.0f) * __log2f(fmaxf(wm, wl * (float)l)) > -61.0f) lmax = l;
    }
  }
  __syncwarp();
}

// J_l cos(l psi), J_l sin(l psi) for l = 1..ol; optionally cos, sin of ol psi
template <typename T>
__device__ __forceinline__ void far_orders(double cp, double sp, int ol, const T* colJ, T* sF, double* cl = nullptr,
                                           double* sl = nullptr) {
  double c = 1.0, s = 0.0;
  for (int l = 1; l <= ol; ++l) {
    const double cn = fma(c, cp, -s * sp);
    s = fma(s, cp, c * sp);
    c = cn;
    const T j = colJ[l * 32];
    sF[(l - 1) * 64] = rmul(j, c);
    sF[(l - 1) * 64 + 32] = rmul(j, s);
  }
  if (cl) {
    *cl = c;
    *sl = s;
  }
}

// X, Y of the orders m and m + 1, l <= lm: their waves overlap (H_{m+l+1}
// serves both at consecutive l), and the sums are eight independent chains.
template <typename T>
__device__ __forceinline__ void far_pair(const cplx* sH, const T* sF, const T J0, int m, int lm, cplx& X0, cplx& Y0,
                                         cplx& X1, cplx& Y1) {
  cplx lo1 = sH[m * 32], hi0 = lo1, hi1 = sH[(m + 1) * 32];   // H_{m+1-l}, H_{m+l}, H_{m+1+l}
  X0 = smul(J0, hi0);
  X1 = smul(J0, hi1);
  Y0 = Y1 = cplx{0.0, 0.0};
  auto order = [&](int l, bool odd) {
    const int n = m - l;
    const cplx lo0 = neg_if(n < 0 && (n & 1), sH[(n < 0 ? -n : n) * 32]);   // H_{m-l}
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
}

// cos, sin of lane times the angle of (ct, st), by squaring
__device__ __forceinline__ void lane_power(int lane, double ct, double st, double& cl, double& sl) {
  double c = ct, s = st;
  cl = 1.0;
  sl = 0.0;
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

// Output orders q of a translation (k_tree_local has the formulas), lane = q:
// W_n the waves (H or J), sd the rows s_m, d_m of NC columns, m <= om, ss their
// Re + Im.  Complex waves: three real products per complex one (Re + Im of the
// waves formed once for all columns): 6 + 6 NC instructions per order m instead
// of 4 + 8 NC.  Real waves (J at real k): 2 + 4 NC.  Up to q = 15 the
// two halves of the warp share the orders m.
template <int NC, typename TW>
__device__ __forceinline__ void translate(const TW* W, const cplx (*sd)[32], const double (*ss)[32], int om, int oq,
                                          int nc, int lane, double cl, double sl, cplx* accA, cplx* accB) {
  constexpr bool kC = IsCplx<TW>::value;
  constexpr int K = kC ? 3 : 2;
  const bool half = oq < 16;
  const int q = half ? lane & 15 : lane, dm = half ? 2 : 1;
  double S[NC][K], D[NC][K];
#pragma unroll
  for (int c = 0; c < NC; ++c)
#pragma unroll
    for (int i = 0; i < K; ++i) S[c][i] = D[c][i] = 0.0;
  for (int m = half ? lane >> 4 : 0; m <= om; m += dm) {
    const int d = m - q;
    const TW ha = neg_if(d < 0 && (d & 1), W[d < 0 ? -d : d]);
    const TW hb = neg_if(q & 1, W[m + q]);
    const TW hp = sadd(ha, hb), hm = sc_sub(ha, hb);
    if constexpr (kC) {
      const double tp = hp.re + hp.im, tm = hm.re + hm.im;
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        if (c >= nc) break;
        const cplx u = sd[2 * c][m], v = sd[2 * c + 1][m];
        S[c][0] = fma(u.re, hp.re, S[c][0]);
        S[c][1] = fma(u.im, hp.im, S[c][1]);
        S[c][2] = fma(ss[2 * c][m], tp, S[c][2]);
        D[c][0] = fma(v.re, hm.re, D[c][0]);
        D[c][1] = fma(v.im, hm.im, D[c][1]);
        D[c][2] = fma(ss[2 * c + 1][m], tm, D[c][2]);
      }
    } else {
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        if (c >= nc) break;
        const cplx u = sd[2 * c][m], v = sd[2 * c + 1][m];
        S[c][0] = fma(u.re, hp, S[c][0]);
        S[c][1] = fma(u.im, hp, S[c][1]);
        D[c][0] = fma(v.re, hm, D[c][0]);
        D[c][1] = fma(v.im, hm, D[c][1]);
      }
    }
  }
  __syncwarp();
  if (half) {
    cl = __shfl_sync(0xffffffffu, cl, q);
    sl = __shfl_sync(0xffffffffu, sl, q);
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      if (c >= nc) break;
#pragma unroll
      for (int i = 0; i < K; ++i) {
        S[c][i] += __shfl_xor_sync(0xffffffffu, S[c][i], 16);
        D[c][i] += __shfl_xor_sync(0xffffffffu, D[c][i], 16);
      }
    }
  }
  if (lane > oq) return;
#pragma unroll
  for (int c = 0; c < NC; ++c) {
    if constexpr (kC) {
      S[c][2] -= S[c][0] + S[c][1];
      S[c][0] -= S[c][1];
      S[c][1] = S[c][2];
      D[c][2] -= D[c][0] + D[c][1];
      D[c][0] -= D[c][1];
      D[c][1] = D[c][2];
    }
    // A' += cos S - i sin D, B' += sin S + i cos D
    accA[c] = accA[c] + cplx{fma(cl, S[c][0], sl * D[c][1]), fma(cl, S[c][1], -sl * D[c][0])};
    accB[c] = accB[c] + cplx{fma(sl, S[c][0], -cl * D[c][1]), fma(sl, S[c][1], cl * D[c][0])};
  }
}

// s_m, d_m of the order m = lane of one column from its coefficients A, B
__device__ __forceinline__ void rotate_in(const cplx A, const cplx B, double cl, double sl, cplx* s, cplx* d, double* ss,
                                          double* ds) {
  const cplx u{fma(A.re, cl, B.re * sl), fma(A.im, cl, B.im * sl)};
  const cplx v{fma(B.im, cl, -A.im * sl), fma(A.re, sl, -B.re * cl)};
  *s = u;
  *d = v;
  if (ss) {
    *ss = u.re + u.im;
    *ds = v.re + v.im;
  }
}

// Whether node j of level l gets moments: it may be in a list (at no distance do
// kTreeP orders do beyond |k| R = 7.23), or, moments carried upward, those of a
// node above it that may be come from it.  A node's points lie in the disc of
// every node above it, but its own radius is about the centre of its bounding box and
// up to (1 + sqrt 2)/2 = 1.207 times that disc's (half a circle: 1.118 circles).
// (All nodes up to 1.25 times the limit, whether needed or not: one level of
// k_tree_up more on the teardrop of 256 panels at k = 30, 8.25 ms instead of 8.14.)
__device__ __forceinline__ bool has_moments(const TreeArgs& a, float ka, int l, int j) {
  auto listed = [&](float kr) {
    return kr < 64.0f && series_order(kr, 1e4f * kr + 1e4f, 1e-4f, 1.0f, 0, kTreeP) <= kTreeP;
  };
  const float kr = ka * (float)a.node[4 * (size_t)(a.off[l] + j) + 2];
  if (listed(kr)) return true;
  if (!a.up || !listed(0.8f * kr)) return false;
  for (++l, j >>= 1; l < a.lev; ++l, j >>= 1)
    if (listed(ka * (float)a.node[4 * (size_t)(a.off[l] + j) + 2])) return true;
  return false;
}

// whether k_tree_moments has room for the dipoles' columns (complex k: up to 99 sources a leaf)
template <typename T>
__host__ __device__ constexpr bool dipole_rows(int q) {
  return (size_t)(4 * kTreeP + 12) * (q | 1) * sizeof(T) <= 210 * 1024;
}

// Moments of one leaf about the centre of one of its nodes (blockIdx = leaf,
// level): with C_m = J_m(k rho) cos(m theta), S_m = J_m(k rho) sin(m theta) of
// the source's position about it,
//   A_m = sum_s w_s C_m, B_m = sum_s w_s S_m  (dipoles: their derivatives along
//   the source's direction, (k/2)(C_{m-1} - C_{m+1}) along x and so on),
// the coefficients of H_m cos(m Theta) and H_m sin(m Theta) (the factor 2 of
// m > 0 in k_tree_fold).  Phase 1: one thread per source forms its columns in
// shared memory, then the normal dipoles' columns from them (formed anew for
// every right-hand side they were two thirds of the kernel: 12 curves, 24
// columns 3.4 ms, now 1.6); phase 2: one thread per (set, rhs, m) sums over the sources.
template <typename T>
__global__ void __launch_bounds__(128) k_tree_moments(TreeArgs b) {
  const TreeArgs& a = b.inst ? b.inst[blockIdx.z] : b;
  if (blockIdx.x >= a.M) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int q = a.q_src, Q = q | 1, P = kTreeP;
  T* sC = reinterpret_cast<T*>(smem_raw);    // [P + 4][Q]
  T* sS = sC + (P + 4) * Q;
  T* dC = sS + (P + 4) * Q;                  // dipoles along the sources' normals: [P + 2][Q]
  T* dS = dC + (P + 2) * Q;
  const int panel = blockIdx.x, l = blockIdx.y;
  const double* n = a.node + 4 * (size_t)(a.off[l] + (panel >> l));
  const double zx = n[0], zy = n[1];
  KW<T> kw;
  kw.init(a.kre, a.kim, a.hk_tab);
  const T kk = kw.kval();
  if (!has_moments(a, (float)sc_abs(kk), l, panel >> l)) return;
  for (int i = threadIdx.x; i < q; i += 128) {
    const double dx = a.sx[panel * q + i] - zx, dy = a.sy[panel * q + i] - zy;
    const double rho = sqrt(dx * dx + dy * dy);
    besselj_column<T>(rmul(kk, rho), P + 3, sC + i, Q);
    const double cs = rho > 0.0 ? dx / rho : 1.0, sn = rho > 0.0 ? dy / rho : 0.0;
    double c = 1.0, s = 0.0;
    for (int m = 0; m <= P + 3; ++m) {
      const T j = sC[m * Q + i];
      sC[m * Q + i] = rmul(j, c);
      sS[m * Q + i] = rmul(j, s);
      const double cn = fma(c, cs, -s * sn);
      s = fma(s, cs, c * sn);
      c = cn;
    }
  }
  __syncthreads();
  bool dip = false;
  for (int i = 0; i < a.nset; ++i) dip |= a.kind[i] == kSetNormal || a.kind[i] == kSetCombined;
  dip = dip && dipole_rows<T>(q);
  if (dip) {
    for (int e = threadIdx.x; e < q * (P + 2); e += 128) {
      const int m = e / q, i = e - m * q, mm = m > 0 ? m - 1 : 1;
      const double nx = a.snx[(size_t)panel * q + i], ny = a.sny[(size_t)panel * q + i];
      const T cm = rmul(sC[mm * Q + i], m > 0 ? 1.0 : -1.0), cp = sC[(m + 1) * Q + i];   // C_{-1} = -C_1, S_{-1} = S_1
      const T sm = sS[mm * Q + i], sp = sS[(m + 1) * Q + i];
      dC[m * Q + i] = sc_sub(rmul(sc_sub(cm, cp), nx), rmul(sadd(sm, sp), ny));
      dS[m * Q + i] = sadd(rmul(sc_sub(sm, sp), nx), rmul(sadd(cm, cp), ny));
    }
    __syncthreads();
  }
  const int ncol = a.nset * a.nrhs;
  // few columns: [leaf, level][col][m][2]; many: the leaf's own rows of the coefficients
  cplx* out = a.up ? reinterpret_cast<cplx*>(a.coef) + (size_t)panel * (P + 2) * ncol * 2
                   : reinterpret_cast<cplx*>(a.mom) + (size_t)(l * a.M + panel) * ncol * (P + 2) * 2;
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
    } else if (kind == kSetQuadX || kind == kSetQuadY) {
      // n . grad of d/dx or d/dy: with F = C, S and F_{m-2}, F_m, F_{m+2}
      //   d_xx F = (k^2/4)(F_{m-2} - 2 F_m + F_{m+2}), d_yy F = -(k^2/4)(F_{m-2} + 2 F_m + F_{m+2}),
      //   d_xy C = -(k^2/4)(S_{m-2} - S_{m+2}), d_xy S = (k^2/4)(C_{m-2} - C_{m+2})
      const double* px = a.snx + (size_t)panel * q;
      const double* py = a.sny + (size_t)panel * q;
      const int mm = m >= 2 ? m - 2 : 2 - m;
      const double sc = m == 1 ? -1.0 : 1.0, ss = m == 0 ? -1.0 : 1.0;   // C_{-n} = (-1)^n C_n, S_{-n} = -(-1)^n S_n
      for (int i = 0; i < q; ++i) {
        const T cm = rmul(sC[mm * Q + i], sc), c0 = sC[m * Q + i], cp = sC[(m + 2) * Q + i];
        const T sm = rmul(sS[mm * Q + i], ss), s0 = sS[m * Q + i], sp = sS[(m + 2) * Q + i];
        const T cxy = sc_sub(sp, sm), sxy = sc_sub(cm, cp);
        const double nx = px[i], ny = py[i];
        const cplx v = w[(size_t)i * a.nrhs];
        if (kind == kSetQuadX) {
          const T cxx = sc_sub(sadd(cm, cp), rmul(c0, 2.0)), sxx = sc_sub(sadd(sm, sp), rmul(s0, 2.0));
          madd(A, sadd(rmul(cxx, nx), rmul(cxy, ny)), v);
          madd(B, sadd(rmul(sxx, nx), rmul(sxy, ny)), v);
        } else {
          const T cyy = sadd(sadd(cm, cp), rmul(c0, 2.0)), syy = sadd(sadd(sm, sp), rmul(s0, 2.0));
          madd(A, sc_sub(rmul(cxy, nx), rmul(cyy, ny)), v);
          madd(B, sc_sub(rmul(sxy, nx), rmul(syy, ny)), v);
        }
      }
      const T k2 = sc_mul(hk, hk);
      A = smul(k2, A);
      B = smul(k2, B);
    } else {
      if (dip && (kind == kSetNormal || kind == kSetCombined)) {
        for (int i = 0; i < q; ++i) {
          const cplx v = w[(size_t)i * a.nrhs];
          madd(A, dC[m * Q + i], v);
          madd(B, dS[m * Q + i], v);
        }
      } else {
        const double* px = a.snx + (size_t)panel * q;
        const double* py = a.sny + (size_t)panel * q;
        const int mm = m > 0 ? m - 1 : 1;
        const double sg = m > 0 ? 1.0 : -1.0;   // C_{-1} = -C_1, S_{-1} = S_1
        for (int i = 0; i < q; ++i) {
          const double nx = kind == kSetX ? 1.0 : kind == kSetY ? 0.0 : px[i];
          const double ny = kind == kSetY ? 1.0 : kind == kSetX ? 0.0 : py[i];
          const T cm = rmul(sC[mm * Q + i], sg), cp = sC[(m + 1) * Q + i];
          const T sm = sS[mm * Q + i], sp = sS[(m + 1) * Q + i];
          const cplx v = w[(size_t)i * a.nrhs];
          madd(A, sc_sub(rmul(sc_sub(cm, cp), nx), rmul(sadd(sm, sp), ny)), v);
          madd(B, sadd(rmul(sc_sub(sm, sp), nx), rmul(sadd(cm, cp), ny)), v);
        }
      }
      A = smul(hk, A);
      B = smul(hk, B);
      if (kind == kSetCombined) {   // - i eta times the density's own
        cplx A1{0.0, 0.0}, B1{0.0, 0.0};
        for (int i = 0; i < q; ++i) {
          madd(A1, sC[m * Q + i], w[(size_t)i * a.nrhs]);
          madd(B1, sS[m * Q + i], w[(size_t)i * a.nrhs]);
        }
        const cplx f{a.eta_im, -a.eta_re};
        cfma(A, f, A1);
        cfma(B, f, B1);
      }
    }
    const double f = a.up && m > 0 ? 2.0 : 1.0;
    cplx* o = out + (a.up ? (size_t)m * ncol + col : (size_t)e) * 2;
    o[0] = f * A;
    o[1] = f * B;
  }
}

// Moments of the centres of one leaf (adjoint sweeps: a centre with gradient g
// sends conj(g) times its truncated expansion to the sources).  As a function
// of the source position the truncated Graf sum of a centre c is the outgoing
// field sum_{|n|<=p} J_n(kr) e^{-i n theta_t} H_n e^{i n theta} about c; carried
// to the node's centre its coefficients of H_m cos, H_m sin are the values
// that k_far_clusters forms, with J_n(k |c - z|) in the place of H_n.  One
// centre per lane, a warp per 32 centres of the leaf (blockIdx = leaf, level);
// the lanes' products are added up over the leaf.
template <typename T>
__global__ void __launch_bounds__(32) k_tree_disc_moments(TreeArgs a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int P = kTreeP, p = a.p, lane = threadIdx.x;
  cplx* sH = reinterpret_cast<cplx*>(smem_raw) + lane;                     // [P + p + 4][32]
  T* colJ = reinterpret_cast<T*>(sH - lane + (P + p + 4) * 32) + lane;     // [p + 2][32]
  T* sF = colJ + (p + 2) * 32;                                             // [p][2][32]
  const int leaf = blockIdx.x, l = blockIdx.y;
  const double* n = a.node + 4 * (size_t)(a.off[l] + (leaf >> l));
  KW<T> kw;
  kw.init(a.kre, a.kim, a.hk_tab);
  const T kk = kw.kval();
  if (!has_moments(a, (float)sc_abs(kk), l, leaf >> l)) return;
  const int nside = a.n_ctr_n / a.n_src, nc = a.q_src * nside, ncol = a.nset * a.nrhs;
  cplx* out = reinterpret_cast<cplx*>(a.mom) + (size_t)(l * a.M + leaf) * ncol * (P + 2) * 2;
  for (int c0 = 0; c0 < nc; c0 += 32) {
    const bool active = c0 + lane < nc;
    const int i = active ? c0 + lane : 0, sd = i / a.q_src, t = leaf * a.q_src + i - sd * a.q_src;
    const int c = sd * a.n_src + t;
    const double cx = a.dcx[c], cy = a.dcy[c];
    double ux = a.sx[t] - cx, uy = a.sy[t] - cy;
    const double r = hypot(ux, uy);
    ux /= r;
    uy /= r;
    besselj_column<T>(rmul(kk, r), p + 1, colJ, 32);
    const double vx = cx - n[0], vy = cy - n[1], d = sqrt(fma(vx, vx, vy * vy));
    const double ct = d > 0.0 ? vx / d : 1.0, st = d > 0.0 ? vy / d : 0.0;
    besselj_wave<T>(rmul(kk, d), P + p + 3, sH);
    far_orders<T>(fma(ux, ct, uy * st), fma(uy, ct, -ux * st), p, colJ, sF);
    const T J0 = colJ[0];
    double cm = 1.0, sm = 0.0;
    for (int m = 0; m <= P + 1; m += 2) {
      cplx X0, Y0, X1, Y1;
      far_pair<T>(sH, sF, J0, m, p, X0, Y0, X1, Y1);
      for (int h = 0; h < 2; ++h) {
        const cplx X = h ? X1 : X0, Y = h ? Y1 : Y0;
        const cplx fc = lin2(cm, X, -sm, Y), fs = lin2(sm, X, cm, Y);
        for (int col = 0; col < ncol; ++col) {
          cplx A{0.0, 0.0}, B{0.0, 0.0};
          if (active) {
            const cplx g = conj(reinterpret_cast<const cplx*>(a.wd[0])[(size_t)c * a.nrhs + col]);
            A = g * fc;
            B = g * fs;
          }
          for (int o = 16; o > 0; o >>= 1) {
            A.re += __shfl_xor_sync(0xffffffffu, A.re, o);
            A.im += __shfl_xor_sync(0xffffffffu, A.im, o);
            B.re += __shfl_xor_sync(0xffffffffu, B.re, o);
            B.im += __shfl_xor_sync(0xffffffffu, B.im, o);
          }
          if (lane == 0) {
            cplx* v = out + ((size_t)col * (P + 2) + m + h) * 2;
            v[0] = c0 ? v[0] + A : A;
            v[1] = c0 ? v[1] + B : B;
          }
        }
        const double cn = fma(cm, ct, -sm * st);
        sm = fma(sm, ct, cm * st);
        cm = cn;
      }
    }
    __syncwarp();
  }
}

// Node moments upward (many columns): a node's moments from its two children's
// (the addition theorem for outgoing waves about a new centre z', V = z' - z:
// M'_q = sum_m M_m J_{m-q}(k|V|) e^{i(m-q) arg V}), in the form of k_tree_local
// with J in the place of H.  One launch per level; a CTA per (node, 32
// columns), warp = 4 columns, lane = q.  Per column 1/16 of the FP64 work of
// summing the sources again at every level.
constexpr int kUpWarps = 8, kUpCols = 4;
template <typename T>
__global__ void __launch_bounds__(32 * kUpWarps) k_tree_up(TreeArgs q, int l) {
  const TreeArgs& a = q.inst ? q.inst[blockIdx.z] : q;
  if (l >= a.lev || blockIdx.x >= a.off[l + 1] - a.off[l]) return;
  constexpr int NC = kUpCols, N = kTreeP + 2;
  static_assert(N == 32, "one lane per order");
  __shared__ T s_w[2][2 * N];
  __shared__ cplx s_sd[kUpWarps][2 * NC][32];
  __shared__ double s_ss[kUpWarps][IsCplx<T>::value ? 2 * NC : 1][32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int id = a.off[l] + blockIdx.x, c0 = a.off[l - 1] + 2 * blockIdx.x;
  const int nch = min(2, a.off[l] - c0);
  const int ncol = a.nset * a.nrhs;
  KW<T> kw;
  kw.init(a.kre, a.kim, a.hk_tab);
  const T kk = kw.kval();
  const double* z = a.node + 4 * (size_t)id;
  if (!has_moments(a, (float)sc_abs(kk), l, (int)blockIdx.x)) return;
  if (warp < nch && lane == 0) {
    const double* y = a.node + 4 * (size_t)(c0 + warp);
    const double vx = z[0] - y[0], vy = z[1] - y[1];
    besselj_column<T>(rmul(kk, sqrt(vx * vx + vy * vy)), 2 * N - 2, s_w[warp], 1);
  }
  __syncthreads();
  for (int col0 = (blockIdx.y * kUpWarps + warp) * NC; col0 < ncol; col0 += gridDim.y * kUpWarps * NC) {
    const int nc = min(NC, ncol - col0);
    cplx accA[NC], accB[NC];
#pragma unroll
    for (int c = 0; c < NC; ++c) accA[c] = accB[c] = cplx{0.0, 0.0};
    for (int ch = 0; ch < nch; ++ch) {
      const double* y = a.node + 4 * (size_t)(c0 + ch);
      const double vx = z[0] - y[0], vy = z[1] - y[1], d = sqrt(vx * vx + vy * vy);
      const double ct = d > 0.0 ? vx / d : 1.0, st = d > 0.0 ? vy / d : 0.0;
      double cl, sl;
      lane_power(lane, ct, st, cl, sl);
      __syncwarp();
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        if (c >= nc) break;
        const cplx* m = reinterpret_cast<const cplx*>(a.coef) + (((size_t)(c0 + ch) * N + lane) * ncol + col0 + c) * 2;
        const cplx A = m[0], B = m[1];
        constexpr bool kC = IsCplx<T>::value;
        rotate_in(A, B, cl, sl, &s_sd[warp][2 * c][lane], &s_sd[warp][2 * c + 1][lane],
                  kC ? &s_ss[warp][kC ? 2 * c : 0][lane] : nullptr, kC ? &s_ss[warp][kC ? 2 * c + 1 : 0][lane] : nullptr);
      }
      __syncwarp();
      translate<NC, T>(s_w[ch], s_sd[warp], s_ss[warp], N - 1, N - 1, nc, lane, cl, sl, accA, accB);
    }
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      if (c >= nc) break;
      cplx* m = reinterpret_cast<cplx*>(a.coef) + (((size_t)id * N + lane) * ncol + col0 + c) * 2;
      m[0] = (lane > 0 ? 1.0 : 0.5) * accA[c];
      m[1] = lane > 0 ? accB[c] : cplx{0.0, 0.0};
    }
  }
}

// The coefficient columns of one node or local expansion from its moments
// (m <= n; strides si of m, sab of A, B): column set i is moment set `base`, itself or its
// derivative along x or y (the series of d/dx u has the coefficients
//   A^x_m = (k/2)(A_{m+1} - A_{m-1}), B^x_m = (k/2)(B_{m+1} - B_{m-1}),
//   A^y_m = (k/2)(B_{m+1} + B_{m-1}), B^y_m = -(k/2)(A_{m+1} + A_{m-1}),
// A_0 counted twice).
__device__ __forceinline__ void shifted_coef(const TreeArgs& a, int set, const cplx* mom, int si, int sab, int n,
                                             int m, cplx* out) {
  auto at = [&](int i, int ab) {
    if (i < 0 || i > n) return cplx{0.0, 0.0};
    return mom[i * si + ab * sab];
  };
  const int sh = a.shift[set];
  if (sh == 0) {
    out[0] = at(m, 0);
    out[1] = at(m, 1);
    return;
  }
  const cplx hk{0.5 * a.kre, 0.5 * a.kim};
  if (sh >= 3) {
    // second derivatives along x, x (3) and x, y (4): the x derivative's
    // coefficients at m - 1 and m + 1, shifted again
    auto dx = [&](int i, cplx* v) {
      const double f = i == 1 ? 2.0 : 1.0;
      v[0] = i < 0 ? cplx{0.0, 0.0} : hk * (at(i + 1, 0) - f * at(i - 1, 0));
      v[1] = i < 1 ? cplx{0.0, 0.0} : hk * (at(i + 1, 1) - at(i - 1, 1));
    };
    cplx p[2], q[2];
    dx(m + 1, p);
    dx(m - 1, q);
    const double f = m == 1 ? 2.0 : 1.0;
    if (sh == 3) {
      out[0] = hk * (p[0] - f * q[0]);
      out[1] = m ? hk * (p[1] - q[1]) : cplx{0.0, 0.0};
    } else {
      out[0] = hk * (p[1] + q[1]);
      out[1] = m ? -(hk * (p[0] + f * q[0])) : cplx{0.0, 0.0};
    }
    return;
  }
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
    shifted_coef(a, cs, &s_m[0][0], 2, 1, kTreeP + 1, m,
                 reinterpret_cast<cplx*>(a.coef) + (((size_t)id * (kTreeP + 2) + m) * a.ncset * a.nrhs + cs * a.nrhs + r) * 2);
  }
}

// Waves H_0..H_{om+oq} and direction of one entry (node, orders om | oq << 8) of a local expansion about blk
template <typename T>
__device__ __forceinline__ void loc_waves(const KW<T>& kw, const double* blk, const double* node, int2 ent, cplx* h,
                                          double2* dir) {
  const int n = (ent.y & 0xff) + (ent.y >> 8);
  const double* nd = node + 4 * (size_t)ent.x;
  double ct, st;
  cplx h0, h1;
  T twoz;
  far_hankel<T>(kw, kw.kval(), blk[0], nd[0], blk[1], nd[1], ct, st, h0, h1, twoz);
  *dir = make_double2(ct, st);
  h[0] = h0;
  T s = twoz;
  for (int i = 1; i <= n; ++i) {
    h[i] = h1;
    const cplx h2 = hrec(s, h1, h0);
    h0 = h1;
    h1 = h2;
    s = sadd(s, twoz);
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
// (A'_0 halved).  Lane = q: a tenth of the FP64 work of taking the node through
// each of the block's 32 or 64 centres.  A CTA takes a block and four columns,
// its warps the block's nodes in turn.  The waves of 32 nodes at a time are
// formed with one node per lane (by every warp for its own node they were a
// quarter of the FP64 work: 12 curves, 64 columns 22.4 -> 17.9 ms with the
// three-product form).  Eight groups of columns to a CTA share the waves, but
// leave few and long CTAs: 64 columns at 256 panels with super-blocks 4.8 ms
// against 2.4, although the waves are then formed once per group (2 % of the work).
constexpr int kLocWarps = 8, kLocCols = 4, kLocNodes = 32, kLocRow = 2 * kTreeP + 3;
struct LocSmem {
  cplx h[kLocNodes][kLocRow];
  cplx sd[kLocWarps][2 * kLocCols][32];
  double ss[kLocWarps][2 * kLocCols][32];
  double2 dir[kLocNodes];
};
template <typename T>
__global__ void __launch_bounds__(32 * kLocWarps, 2) k_tree_local(TreeArgs q, bool super) {
  const TreeArgs& a = q.inst ? q.inst[blockIdx.z] : q;
  if (blockIdx.x >= (super ? a.n_sup : a.n_blk)) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  LocSmem& sm = *reinterpret_cast<LocSmem*>(smem_raw);
  constexpr int NC = kLocCols;
  static_assert(kTreeP < 32, "one lane per order");
  const int b = blockIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int cnt = super ? a.scnt[2 * b] : a.cnt[3 * b + 2];
  __shared__ int s_anc[kSupLevels];   // the super-blocks above the block with a list, as node entries
  int nanc = 0;
  if (!super && a.n_sup) {
    for (int B = 1; B <= a.sup_lev; ++B) {
      const int id = a.sup_off[B] + (b >> B);
      if (a.scnt[2 * id] == 0) continue;
      if (threadIdx.x == 0) s_anc[nanc] = a.off[a.lev] + a.n_blk + id;
      ++nanc;
    }
  }
  const int nmom = a.nset * a.nrhs, col0 = blockIdx.y * NC;
  if (cnt + nanc == 0 || col0 >= nmom) return;
  const int nc = min(NC, nmom - col0);
  int ccol[NC];   // coefficient column of each moment column
#pragma unroll
  for (int c = 0; c < NC; ++c) {
    const int col = min(col0 + c, nmom - 1), set = col / a.nrhs;
    ccol[c] = a.plain[set] * a.nrhs + col - set * a.nrhs;
  }
  const int ncol = a.ncset * a.nrhs;
  const int own = a.off[a.lev] + (super ? a.n_blk : 0) + b;   // this expansion's entry
  const double* blk = a.node + 4 * (size_t)own;
  const int2* loc = super ? reinterpret_cast<const int2*>(a.sloc) + (size_t)b * a.sup_stride
                          : reinterpret_cast<const int2*>(a.loc) + (size_t)b * a.M;
  KW<T> kw;
  kw.init(a.kre, a.kim, a.hk_tab);
  cplx accA[NC], accB[NC];
#pragma unroll
  for (int c = 0; c < NC; ++c) accA[c] = accB[c] = cplx{0.0, 0.0};
  // rows s_m, d_m of this warp's columns of node or super-block id; cos, sin of lane * Theta
  auto rows = [&](int id, int om, const double2 dir, double& cl, double& sl) {
    lane_power(lane, dir.x, dir.y, cl, sl);
    __syncwarp();   // the previous rows are no longer read
    if (lane <= om) {
      const double2* co = reinterpret_cast<const double2*>(a.coef) + ((size_t)id * (kTreeP + 2) + lane) * ncol * 2;
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        if (c >= nc) break;
        const double2 A = co[2 * ccol[c]], B = co[2 * ccol[c] + 1];
        rotate_in(cplx{A.x, A.y}, cplx{B.x, B.y}, cl, sl, &sm.sd[warp][2 * c][lane], &sm.sd[warp][2 * c + 1][lane],
                  &sm.ss[warp][2 * c][lane], &sm.ss[warp][2 * c + 1][lane]);
      }
    }
    __syncwarp();
  };
  for (int e0 = 0; e0 < cnt; e0 += kLocNodes) {
    __syncthreads();   // the previous nodes' waves are no longer read
    if (warp == 0 && e0 + lane < cnt) loc_waves<T>(kw, blk, a.node, loc[e0 + lane], sm.h[lane], &sm.dir[lane]);
    __syncthreads();
    for (int e = warp; e < min(kLocNodes, cnt - e0); e += kLocWarps) {
      const int2 ent = loc[e0 + e];
      const int om = ent.y & 0xff, oq = ent.y >> 8;
      double cl, sl;
      rows(ent.x, om, sm.dir[e], cl, sl);
      translate<NC, cplx>(sm.h[e], sm.sd[warp], sm.ss[warp], om, oq, nc, lane, cl, sl, accA, accB);
    }
  }
  if (nanc > 0) {   // the expansions of the super-blocks: the same translation with J about the block's centre
    __syncthreads();
    if (warp == 0 && lane < nanc) {
      const double* nd = a.node + 4 * (size_t)s_anc[lane];
      const double vx = blk[0] - nd[0], vy = blk[1] - nd[1], d = sqrt(fma(vx, vx, vy * vy));
      sm.dir[lane] = d > 0.0 ? make_double2(vx / d, vy / d) : make_double2(1.0, 0.0);
      besselj_column<T>(rmul(kw.kval(), d), 2 * kTreeP + 1, reinterpret_cast<T*>(sm.h[lane]), 1);
    }
    __syncthreads();
    for (int e = warp; e < nanc; e += kLocWarps) {
      double cl, sl;
      rows(s_anc[e], kTreeP, sm.dir[e], cl, sl);
      translate<NC, T>(reinterpret_cast<const T*>(sm.h[e]), sm.sd[warp], sm.ss[warp], kTreeP, kTreeP, nc, lane, cl, sl,
                       accA, accB);
    }
  }
  // the warps' sums, in warp order
  __syncwarp();
#pragma unroll
  for (int c = 0; c < NC; ++c) {
    sm.sd[warp][2 * c][lane] = accA[c];
    sm.sd[warp][2 * c + 1][lane] = accB[c];
  }
  __syncthreads();
  for (int i = threadIdx.x; i < 2 * NC * 32; i += 32 * kLocWarps) {
    const int row = i >> 5, m = i & 31;
    cplx v = sm.sd[0][row][m];
    for (int w = 1; w < kLocWarps; ++w) v = v + sm.sd[w][row][m];
    sm.sd[0][row][m] = m > 0 ? v : row & 1 ? cplx{0.0, 0.0} : 0.5 * v;
  }
  __syncthreads();
  cplx* out = reinterpret_cast<cplx*>(a.coef) + (size_t)own * (kTreeP + 2) * ncol * 2;
  const int per = a.ncset * (kTreeP + 1);
  for (int i = threadIdx.x; i < nc * per; i += 32 * kLocWarps) {
    const int c = i / per, rem = i - c * per, cs = rem / (kTreeP + 1), m = rem - cs * (kTreeP + 1);
    const int col = col0 + c, set = col / a.nrhs, r = col - set * a.nrhs;
    if (a.base[cs] == set)
      shifted_coef(a, cs, &sm.sd[0][2 * c][0], 1, 32, kTreeP, m, out + ((size_t)m * ncol + cs * a.nrhs + r) * 2);
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

// Matrix entries of the assembled combined field from the panels that are far
// from a block of 32 targets: the panel's q_tgt columns of moments (one per
// column of the interpolation) go into local expansions about the block's
// centre, whose waves' truncated expansions about the two centres of a target
// are the same for every panel: their sums C_q, S_q over both sides are formed
// once per CTA, and an entry is sum_q (A'_q C_q + B'_q S_q).  A warp takes one
// panel, four columns at a time (lane = q in the translation, then lane =
// target).  FP64-bound: 4000 instructions per panel and block, pair by pair
// 20700 (assembly at 72 panels, p = 10, 18 of them near a block: 5.7 -> 2.8 ms).
struct MatrixSmem {
  union {
    LocSmem loc;
    unsigned char setup[sizeof(LocSmem)];   // per side: J column, waves, orders (while C, S are formed)
  };
  cplx basis[kTreeP + 1][2][32];
};
template <typename T>
__global__ void __launch_bounds__(32 * kLocWarps) k_tree_matrix(MatrixFarArgs q) {
  const TreeArgs& a = q.t;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  MatrixSmem& ms = *reinterpret_cast<MatrixSmem*>(smem_raw);
  LocSmem& sm = ms.loc;
  constexpr int NC = kLocCols;
  const int b = blockIdx.x, split = blockIdx.y, nsplit = gridDim.y, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int cnt = a.cnt[3 * b + 2], mine = cnt > split ? (cnt - split + nsplit - 1) / nsplit : 0;
  if (mine == 0) return;
  const double* blk = a.node + 4 * (size_t)(a.off[a.lev] + b);
  const int2* loc = reinterpret_cast<const int2*>(a.loc) + (size_t)b * a.M;
  const bool active = b * 32 + lane < a.n_tgt;
  const int t = active ? b * 32 + lane : a.n_tgt - 1;
  KW<T> kw;
  kw.init(a.kre, a.kim, a.hk_tab);
  const T kk = kw.kval();
  int oqmax = 0;
  for (int e = lane; e < mine; e += 32) oqmax = max(oqmax, loc[split + nsplit * e].y >> 8);
  oqmax = __reduce_max_sync(0xffffffffu, oqmax);
  // the basis: the columns of a side by two warps of four, then all warps' pairs of orders on both sides
  for (int phase = 0; phase < 3; ++phase) {
    const int p = a.p;
    for (int sd = phase < 2 ? warp >> 2 : 0; sd < (phase < 2 ? (warp >> 2) + 1 : 2); ++sd) {
      const int c = sd * a.n_tgt + t;
      unsigned char* set = ms.setup + sd * (far_col_bytes<T>(p) + far_warp_bytes<T>(p));
      T* colJ = reinterpret_cast<T*>(set) + lane;
      cplx* sH = reinterpret_cast<cplx*>(set + far_col_bytes<T>(p)) + lane;
      T* sF = reinterpret_cast<T*>(sH - lane + (kTreeP + p + 2) * 32) + lane;
      const double cx = a.cx[c], cy = a.cy[c];
      double ux = a.tx[t] - cx, uy = a.ty[t] - cy;
      const double r = hypot(ux, uy), vx = cx - blk[0], vy = cy - blk[1], rho = sqrt(fma(vx, vx, vy * vy));
      ux /= r;
      uy /= r;
      const double ct = rho > 0.0 ? vx / rho : 1.0, st = rho > 0.0 ? vy / rho : 0.0;
      if (phase == 0) {
        if ((warp & 3) == 0) besselj_column<T>(rmul(kk, r), p + 1, colJ, 32);
        if ((warp & 3) == 1) besselj_wave<T>(rmul(kk, rho), oqmax + p + 1, sH);
        continue;
      }
      if (phase == 1) {
        if ((warp & 3) == 0) far_orders<T>(fma(ux, ct, uy * st), fma(uy, ct, -ux * st), p, colJ, sF);
        continue;
      }
      double cm = 1.0, sn = 0.0;
      for (int m = 0; m <= oqmax; ++m) {
        const double c1 = fma(cm, ct, -sn * st), s1 = fma(sn, ct, cm * st);
        if (!(m & 1) && (m >> 1) % kLocWarps == warp) {
          cplx X0, Y0, X1, Y1;
          far_pair<T>(sH, sF, colJ[0], m, p, X0, Y0, X1, Y1);
          auto add = [&](int n, const cplx fc, const cplx fs) {
            ms.basis[n][0][lane] = sd ? ms.basis[n][0][lane] + fc : fc;
            ms.basis[n][1][lane] = sd ? ms.basis[n][1][lane] + fs : fs;
          };
          add(m, lin2(cm, X0, -sn, Y0), lin2(sn, X0, cm, Y0));
          if (m < oqmax) add(m + 1, lin2(c1, X1, -s1, Y1), lin2(s1, X1, c1, Y1));
        }
        cm = c1;
        sn = s1;
      }
    }
    __syncthreads();
  }
  const double swt = sqrt(q.tw[t]);
  cplx* out = reinterpret_cast<cplx*>(q.out);
  const int ncol = a.nrhs;
  for (int e0 = 0; e0 < mine; e0 += kLocNodes) {
    if (e0) __syncthreads();
    if (warp == 0 && e0 + lane < mine) loc_waves<T>(kw, blk, a.node, loc[split + nsplit * (e0 + lane)], sm.h[lane], &sm.dir[lane]);
    __syncthreads();
    for (int e = warp; e < min(kLocNodes, mine - e0); e += kLocWarps) {
      const int2 ent = loc[split + nsplit * (e0 + e)];
      const int om = ent.y & 0xff, oq = ent.y >> 8;
      const double2 dir = sm.dir[e];
      double cl, sl;
      lane_power(lane, dir.x, dir.y, cl, sl);
      for (int c0 = 0; c0 < ncol; c0 += NC) {
        const int nc = min(NC, ncol - c0);
        __syncwarp();
        if (lane <= om) {
          const cplx* co = reinterpret_cast<const cplx*>(a.coef) + (((size_t)ent.x * (kTreeP + 2) + lane) * ncol + c0) * 2;
#pragma unroll
          for (int c = 0; c < NC; ++c) {
            if (c >= nc) break;
            rotate_in(co[2 * c], co[2 * c + 1], cl, sl, &sm.sd[warp][2 * c][lane], &sm.sd[warp][2 * c + 1][lane],
                      &sm.ss[warp][2 * c][lane], &sm.ss[warp][2 * c + 1][lane]);
          }
        }
        __syncwarp();
        cplx accA[NC], accB[NC];
#pragma unroll
        for (int c = 0; c < NC; ++c) accA[c] = accB[c] = cplx{0.0, 0.0};
        translate<NC, cplx>(sm.h[e], sm.sd[warp], sm.ss[warp], om, oq, nc, lane, cl, sl, accA, accB);
        __syncwarp();
#pragma unroll
        for (int c = 0; c < NC; ++c) {
          sm.sd[warp][2 * c][lane] = (lane == 0 ? 0.5 : 1.0) * accA[c];
          sm.sd[warp][2 * c + 1][lane] = lane == 0 ? cplx{0.0, 0.0} : accB[c];
        }
        __syncwarp();
        cplx v[NC];
#pragma unroll
        for (int c = 0; c < NC; ++c) v[c] = cplx{0.0, 0.0};
        for (int m = 0; m <= oq; ++m) {
          const cplx fc = ms.basis[m][0][lane], fs = ms.basis[m][1][lane];
#pragma unroll
          for (int c = 0; c < NC; ++c) {
            cfma(v[c], sm.sd[warp][2 * c][m], fc);
            cfma(v[c], sm.sd[warp][2 * c + 1][m], fs);
          }
        }
        if (active) {
#pragma unroll
          for (int c = 0; c < NC; ++c) {
            if (c >= nc) break;
            const int col = ent.x * ncol + c0 + c;
            const double sc = swt / sqrt(q.tw[col]);
            out[(size_t)col * a.n_tgt + t] = cplx{sc * (-0.125 * v[c].im), sc * (0.125 * v[c].re)};
          }
        }
      }
    }
  }
}

// the columns of the interpolation as weighted densities: wd[s][i] = w_s P[s mod q_src][i]
__global__ void k_matrix_density(int n, int q_src, int q_tgt, const double* w, const double* P, cplx* wd) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n * q_tgt) return;
  const int s = i / q_tgt;
  wd[i] = cplx{w[s] * P[(s % q_src) * q_tgt + i - s * q_tgt], 0.0};
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
    int lmax;   // of order m = lane
    const double* nd = a.node + 4 * (size_t)ent.x;
    double ct, st;   // Theta
    far_waves<T>(kw, kk, ka, ent, a.nd, a.kim, nd, cx, cy, r, sH, ct, st, lmax);
    // orders m whose expansions reach the cut at l = p (grad S)
    const unsigned cut = !a.discs && ol == p ? __ballot_sync(0xffffffffu, lane <= om && lmax >= p) : 0u;
    const int mcut = cut ? 32 - __clz(cut) : -1;   // one order further: the derivative shifts m by one
    const double cp = fma(ux, ct, uy * st), sp = fma(uy, ct, -ux * st);   // psi
    double cP, sP;   // cos, sin of ol psi (= p psi where the cut is reached)
    far_orders<T>(cp, sp, ol, colJ, sF, &cP, &sP);
    const cplx* co = reinterpret_cast<const cplx*>(a.coef) + ((size_t)ent.x * (kTreeP + 2) * ncol + a.rhs0) * 2;
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
    for (int m = 2 * mpart; m <= om; m += 2 * np) {
      const bool two = m < om;
      cplx X0, Y0, X1, Y1;
      far_pair<T>(sH, sF, J0, m, max(__shfl_sync(0xffffffffu, lmax, m), __shfl_sync(0xffffffffu, lmax, min(m + 1, om))),
                  X0, Y0, X1, Y1);
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

// Far sums for many columns (S, D, S + D or the combined field, 16 or more
// rhs): a CTA of eight warps holds 32 targets; for every far node of the block
// the warps form the values of H_m cos(m Theta), H_m sin(m Theta) through the
// target's centre (or the average over its two centres) in shared memory, as
// k_far_clusters does, and then multiply them into RG columns each, three real
// products per complex one (the coefficients' Re + Im formed once per warp for
// its 32 targets, five orders at a time in the place of the waves): a column costs 6 FP64 instructions per
// order where the pairs of a leaf cost 96 (with four products, 8: 12 curves, 64
// columns 9.5 ms, now 8.5).
constexpr int kFgWarps = 8, kFgOrders = 5, kFgCols = 8;
template <typename T>
struct FarGroupSmem {
  static __host__ __device__ size_t rows(int pl) { return (size_t)kTreeP + pl + 2; }
  static __host__ __device__ size_t bytes(int pl, int nsd) {
    return (size_t)nsd * ((pl + 2) * sizeof(T) + rows(pl) * 16 + (size_t)pl * 2 * sizeof(T) + 2 * 8 + 4) * 32 +
           (size_t)2 * (kTreeP + 1) * 32 * 16;
  }
};

template <typename T, int RG>
__global__ void __launch_bounds__(32 * kFgWarps) k_far_group(TreeArgs q) {
  const TreeArgs& a = q.inst ? q.inst[blockIdx.z] : q;
  const int pl = a.pl, nsd = a.n_ctr / a.n_tgt;
  const int blk = (int)blockIdx.x % q.n_blk, split = (int)blockIdx.x / q.n_blk;   // q: the largest n_blk
  if (blk >= a.n_blk || split >= a.nsplit) return;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const size_t rows = FarGroupSmem<T>::rows(pl);
  cplx* sB = reinterpret_cast<cplx*>(smem_raw);                        // [2 (kTreeP + 1)][32] values
  cplx* sH = sB + 2 * (kTreeP + 1) * 32;                               // [side][rows][32]
  T* sJ = reinterpret_cast<T*>(sH + nsd * rows * 32);                  // [side][pl + 2][32]
  T* sF = sJ + (size_t)nsd * (pl + 2) * 32;                            // [side][pl][2][32]
  double* sT = reinterpret_cast<double*>(sF + (size_t)nsd * pl * 64);  // [side][2][32] Theta
  int* sL = reinterpret_cast<int*>(sT + nsd * 64);                     // [side][32] orders l by m
  // per warp: coefficients of its columns, [order][column][A, B], and their Re + Im
  // (where the waves of the first side were: at least kTreeP + 2 rows)
  static_assert(RG <= kFgCols && kFgWarps * kFgOrders * kFgCols * 2 * 24 <= (kTreeP + 2) * 32 * 16, "columns of the warps");
  double* mine = reinterpret_cast<double*>(sH) + (size_t)warp * kFgOrders * kFgCols * 6;
  cplx* sC = reinterpret_cast<cplx*>(mine);
  double* sS = mine + kFgOrders * kFgCols * 4;
  const bool active = blk * 32 + lane < a.n_tgt;
  const int t = active ? blk * 32 + lane : a.n_tgt - 1;
  KW<T> kw;
  kw.init(a.kre, a.kim, a.hk_tab);
  const T kk = kw.kval();
  const float ka = (float)sc_abs(kk);
  double cx = 0.0, cy = 0.0, ux = 0.0, uy = 0.0, r = 0.0;   // of side `warp`
  if (warp < nsd) {
    cx = a.cx[warp * a.n_tgt + t];
    cy = a.cy[warp * a.n_tgt + t];
    ux = a.tx[t] - cx;
    uy = a.ty[t] - cy;
    r = hypot(ux, uy);
    ux /= r;
    uy /= r;
    besselj_column<T>(rmul(kk, r), pl + 1, sJ + (size_t)warp * (pl + 2) * 32 + lane, 32);
  }
  const int ncomp = (a.ops & OPB_C) ? 1 : popc3(a.ops), ncols = ncomp * a.nrhs;
  const int ccol = a.ncset * a.nrhs;
  const int cnt = a.cnt[3 * blk + 1];
  const int2* far = reinterpret_cast<const int2*>(a.far) + (size_t)blk * (a.M + 1);
  // columns in the coefficient rows: S's set, then D's (or the combined one)
  const int set0 = (a.ops & OPB_S) ? a.set_s : a.set_d, set1 = a.set_d;
  for (int g0 = 0; g0 < ncols; g0 += kFgWarps * RG) {
    double acc[RG][3];
#pragma unroll
    for (int i = 0; i < RG; ++i) acc[i][0] = acc[i][1] = acc[i][2] = 0.0;
    const int mycol = g0 + warp * RG;
    for (int e = split; e < cnt; e += a.nsplit) {
      const int2 ent = far[cnt - 1 - e];
      const int om = ent.y & 0xff, ol = ent.y >> 8 & 0xff;
      __syncthreads();   // the previous node's waves and values are no longer read
      if (warp < nsd) {
        cplx* H = sH + (size_t)warp * rows * 32 + lane;
        const double* nd = a.node + 4 * (size_t)ent.x;
        double ct, st;
        int lmax;
        far_waves<T>(kw, kk, ka, ent, a.nd, a.kim, nd, cx, cy, r, H, ct, st, lmax);
        sT[warp * 64 + lane] = ct;
        sT[warp * 64 + 32 + lane] = st;
        sL[warp * 32 + lane] = lmax;
        far_orders<T>(fma(ux, ct, uy * st), fma(uy, ct, -ux * st), ol, sJ + (size_t)warp * (pl + 2) * 32 + lane,
                      sF + (size_t)warp * pl * 64 + lane);
      }
      __syncthreads();
      for (int m = 2 * warp; m <= om; m += 2 * kFgWarps) {
        cplx c0{0.0, 0.0}, s0 = c0, c1 = c0, s1 = c0;
        const double wgt = nsd == 2 ? 0.5 : 1.0;
        for (int sd = 0; sd < nsd; ++sd) {
          const cplx* H = sH + (size_t)sd * rows * 32 + lane;
          cplx X0, Y0, X1, Y1;
          far_pair<T>(H, sF + (size_t)sd * pl * 64 + lane, sJ[(size_t)sd * (pl + 2) * 32 + lane], m,
                      max(sL[sd * 32 + m], sL[sd * 32 + min(m + 1, om)]), X0, Y0, X1, Y1);
          const double ct = sT[sd * 64 + lane], st = sT[sd * 64 + 32 + lane];
          double cm, sm;
          lane_power(m, ct, st, cm, sm);
          cm *= wgt;
          sm *= wgt;
          const double cn = fma(cm, ct, -sm * st), sn = fma(sm, ct, cm * st);
          c0 = c0 + lin2(cm, X0, -sm, Y0);
          s0 = s0 + lin2(sm, X0, cm, Y0);
          c1 = c1 + lin2(cn, X1, -sn, Y1);
          s1 = s1 + lin2(sn, X1, cn, Y1);
        }
        sB[(2 * m) * 32 + lane] = c0;
        sB[(2 * m + 1) * 32 + lane] = s0;
        if (m < om) {
          sB[(2 * m + 2) * 32 + lane] = c1;
          sB[(2 * m + 3) * 32 + lane] = s1;
        }
      }
      __syncthreads();
      if (mycol < ncols) {
        const double2* co = reinterpret_cast<const double2*>(a.coef) + (size_t)ent.x * (kTreeP + 2) * ccol * 2;
        for (int m0 = 0; m0 <= om; m0 += kFgOrders) {
          const int nm = min(kFgOrders, om + 1 - m0);
          __syncwarp();
          for (int v = lane; v < nm * RG * 2; v += 32) {
            const int m = v / (RG * 2), i = v / 2 % RG, c = min(mycol + i, ncols - 1), comp = c / a.nrhs;
            const double2 w = __ldg(co + (size_t)(m0 + m) * ccol * 2 +
                                    2 * ((comp ? set1 : set0) * a.nrhs + c - comp * a.nrhs) + (v & 1));
            sC[v] = cplx{w.x, w.y};
            sS[v] = w.x + w.y;
          }
          __syncwarp();
          for (int m = 0; m < nm; ++m) {
            const cplx fc = sB[2 * (m0 + m) * 32 + lane], fs = sB[(2 * (m0 + m) + 1) * 32 + lane];
            const double tc = fc.re + fc.im, ts = fs.re + fs.im;
#pragma unroll
            for (int i = 0; i < RG; ++i) {
              const int v = (m * RG + i) * 2;
              const cplx A = sC[v], B = sC[v + 1];
              acc[i][0] = fma(A.re, fc.re, acc[i][0]);
              acc[i][1] = fma(A.im, fc.im, acc[i][1]);
              acc[i][2] = fma(sS[v], tc, acc[i][2]);
              acc[i][0] = fma(B.re, fs.re, acc[i][0]);
              acc[i][1] = fma(B.im, fs.im, acc[i][1]);
              acc[i][2] = fma(sS[v + 1], ts, acc[i][2]);
            }
          }
        }
      }
    }
    if (active) {
      cplx* part = reinterpret_cast<cplx*>(a.part) + ((size_t)(a.split0 + split) * a.n_tgt + t) * ncols;
#pragma unroll
      for (int i = 0; i < RG; ++i)
        if (mycol + i < ncols)
          part[mycol + i] = cplx{acc[i][0] - acc[i][1], acc[i][2] - acc[i][0] - acc[i][1]};
    }
  }
}

// Coefficients alpha_l, |l| <= p, of every centre from the far nodes of its
// block: the translation of k_tree_local to each centre (lane), with the
// directions Theta of the lanes apart,
//   alpha_l = e^{-il Theta} (S_l + T_l)/2, alpha_{-l} = (-1)^l e^{il Theta} (S_l - T_l)/2.
template <typename T>
__host__ __device__ size_t form_far_bytes(int p) {   // per warp: waves, s_m and d_m, the sums
  return ((size_t)(kTreeP + p + 2) + 2 * (kTreeP + 1) + (2 * p + 1)) * 32 * 16;
}
template <typename T>
__global__ void __launch_bounds__(64) k_form_far(TreeArgs a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int p = a.p, nl = 2 * p + 1, W = blockDim.x >> 5, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  cplx* sH = reinterpret_cast<cplx*>(smem_raw + (size_t)warp * form_far_bytes<T>(p)) + lane;
  cplx* sD = sH + (kTreeP + p + 2) * 32;          // [kTreeP + 1][2][32]
  cplx* sA = sD + 2 * (kTreeP + 1) * 32;          // [2p + 1][32]
  const int units = a.n_blk * (a.n_ctr / a.n_tgt);
  const int unit = blockIdx.x % units, split = blockIdx.x / units, r = blockIdx.y;
  const int side = unit / a.n_blk, blk = unit - side * a.n_blk;
  const bool active = blk * 32 + lane < a.n_tgt;
  const int t = active ? blk * 32 + lane : a.n_tgt - 1, c = side * a.n_tgt + t;
  const double cx = a.cx[c], cy = a.cy[c], rad = hypot(a.tx[t] - cx, a.ty[t] - cy);
  KW<T> kw;
  kw.init(a.kre, a.kim, a.hk_tab);
  const T kk = kw.kval();
  const float ka = (float)sc_abs(kk);
  for (int l = 0; l < nl; ++l) sA[l * 32] = cplx{0.0, 0.0};
  const int cnt = a.cnt[3 * blk + 1], ncol = a.ncset * a.nrhs;
  const int2* far = reinterpret_cast<const int2*>(a.far) + (size_t)blk * (a.M + 1);
  for (int e = split * W + warp; e < cnt; e += a.nsplit * W) {
    int2 ent = far[cnt - 1 - e];
    const int om = ent.y & 0xff;
    ent.y = (ent.y & ~0xff00) | p << 8;   // every order l <= p
    const double* nd = a.node + 4 * (size_t)ent.x;
    double ct, st;
    int lmax;
    __syncwarp();
    far_waves<T>(kw, kk, ka, ent, a.nd, a.kim, nd, cx, cy, rad, sH, ct, st, lmax);
    const double2* co = reinterpret_cast<const double2*>(a.coef) +
                        ((size_t)ent.x * (kTreeP + 2) * ncol + (size_t)a.set_s * a.nrhs + r) * 2;
    double cm = 1.0, sm = 0.0;
    for (int m = 0; m <= om; ++m) {
      const double2 A = __ldg(co + (size_t)m * ncol * 2), B = __ldg(co + (size_t)m * ncol * 2 + 1);
      sD[(2 * m) * 32] = cplx{fma(A.x, cm, B.x * sm), fma(A.y, cm, B.y * sm)};
      sD[(2 * m + 1) * 32] = cplx{fma(B.y, cm, -A.y * sm), fma(A.x, sm, -B.x * cm)};
      const double cn = fma(cm, ct, -sm * st);
      sm = fma(sm, ct, cm * st);
      cm = cn;
    }
    double cl = 0.5, sl = 0.0;   // e^{i l Theta} / 2
    for (int l = 0; l <= p; ++l) {
      cplx S{0.0, 0.0}, D{0.0, 0.0};
      for (int m = 0; m <= om; ++m) {
        const int d = m - l;
        const cplx ha = neg_if(d < 0 && (d & 1), sH[(d < 0 ? -d : d) * 32]);
        const cplx hb = neg_if(l & 1, sH[(m + l) * 32]);
        cfma(S, sD[(2 * m) * 32], ha + hb);
        cfma(D, sD[(2 * m + 1) * 32], ha - hb);
      }
      const cplx e{cl, sl};
      sA[(p + l) * 32] = sA[(p + l) * 32] + conj(e) * (S + D);
      if (l > 0) sA[(p - l) * 32] = sA[(p - l) * 32] + neg_if(l & 1, e * (S - D));
      const double cn = fma(cl, ct, -sl * st);
      sl = fma(sl, ct, cl * st);
      cl = cn;
    }
  }
  __syncthreads();
  if (!active) return;
  cplx* part = reinterpret_cast<cplx*>(a.part) + ((size_t)(a.split0 + split) * a.n_ctr + c) * nl * a.nrhs + r;
  for (int l = warp; l < nl; l += W) {   // the warps' sums in warp order
    const cplx* v = reinterpret_cast<const cplx*>(smem_raw) + ((kTreeP + p + 2) + 2 * (kTreeP + 1) + l) * 32 + lane;
    cplx u = *v;
    for (int w = 1; w < W; ++w) u = u + v[w * (form_far_bytes<T>(p) / 16)];
    part[(size_t)l * a.nrhs] = u;
  }
}

// Plain quadrature at points anywhere: a lane owns a point and walks the nodes
// from the top of its share of the curve, taking a node whose disc is far
// enough through its moments, descending otherwise, and a leaf that never is
// source by source.  The lanes of a warp step together: each finds its next
// node, then all evaluate theirs (points in random order share no node, so
// lists per block would hold every leaf).  About 15 FP64 instructions per order
// of a node, 100 per source of a leaf.
template <typename T, int NR, bool GRAD>
__global__ void __launch_bounds__(128) k_far_points(FarPointArgs q) {
  const TreeArgs& a = q.t;
  constexpr int kC = GRAD ? 2 : 1;
  const int chunks = (q.n_far + 127) / 128;
  const int e = (int)(blockIdx.x % chunks) * 128 + threadIdx.x, split = blockIdx.x / chunks;
  const bool active = e < q.n_far;
  const int ee = active ? e : q.n_far - 1;
  const double x = q.xy[2 * ee], y = q.xy[2 * ee + 1];
  KW<T> kw;
  kw.init(a.kre, a.kim, a.hk_tab);
  const T kk = kw.kval();
  const float ka = (float)sc_abs(kk), ki = (float)a.kim;
  cplx acc[kC][NR];
#pragma unroll
  for (int g = 0; g < kC; ++g)
#pragma unroll
    for (int i = 0; i < NR; ++i) acc[g][i] = cplx{0.0, 0.0};
  const int top = a.lev - 1, ntop = a.off[top + 1] - a.off[top], ncol = a.ncset * a.nrhs;
  int l = top, j = (int)((long)ntop * split / q.nsplit);
  const int jend = (int)((long)ntop * (split + 1) / q.nsplit);   // of the top level
  const int set = GRAD ? a.set_gx : a.set_s;
  const cplx* wd = reinterpret_cast<const cplx*>(q.wd);
  for (;;) {
    // ---- the next node to take: om >= 0 through its moments, -1 a near leaf ----
    int om = 0, id = -1;
    while ((j << l) < a.M && (j >> (top - l)) < jend) {
      const double* n = a.node + 4 * (size_t)(a.off[l] + j);
      const float dx = (float)(x - n[0]), dy = (float)(y - n[1]), R = (float)n[2] * 1.00001f;
      const float d = 0.99999f * sqrtf(fmaf(dx, dx, dy * dy));
      om = kTreeP + 1;
      if (d > 1.34f * R) {
        om = series_order(ka * R, ka * d, R / d, expf(2.0f * ki * R), a.nd, kTreeP);
        if (om <= kTreeP) {
          const float o = (float)om;   // H and the moments of order om stay in range
          if (!(o * log10f(fmaxf(2.0f * o / (2.7f * ka * d), 1.0f)) < 280.0f) ||
              !(o * log10f(fmaxf(2.0f * o / (2.7f * ka * R), 1.0f)) < 280.0f))
            om = kTreeP + 1;
        }
      }
      if (om > kTreeP && l > 0) {   // descend
        --l;
        j <<= 1;
        continue;
      }
      id = a.off[l] + j;
      if (om > kTreeP) om = -1;
      ++j;
      while (l < top && !(j & 1)) {
        j >>= 1;
        ++l;
      }
      break;
    }
    if (!__any_sync(0xffffffffu, id >= 0)) break;
    if (id < 0) continue;
    if (om >= 0) {
      const double* n = a.node + 4 * (size_t)id;
      double ct, st;
      cplx h, h1;
      T twoz;
      far_hankel<T>(kw, kk, x, n[0], y, n[1], ct, st, h, h1, twoz);
      T s = twoz;
      double cm = 1.0, sm = 0.0;
      const double2* co =
          reinterpret_cast<const double2*>(a.coef) + ((size_t)id * (kTreeP + 2) * ncol + (size_t)set * a.nrhs + q.rhs0) * 2;
      for (int m = 0; m <= om; ++m) {
        const cplx fc = cm * h, fs = sm * h;
#pragma unroll
        for (int g = 0; g < kC; ++g)
#pragma unroll
          for (int i = 0; i < NR; ++i) {
            if (i > 0 && i >= q.nr) break;
            const double2* v = co + ((size_t)m * ncol + (size_t)g * a.nrhs + i) * 2;
            const double2 A = __ldg(v), B = __ldg(v + 1);
            cfma(acc[g][i], cplx{A.x, A.y}, fc);
            cfma(acc[g][i], cplx{B.x, B.y}, fs);
          }
        const cplx h2 = hrec(s, h1, h);
        h = h1;
        h1 = h2;
        s = sadd(s, twoz);
        const double cn = fma(cm, ct, -sm * st);
        sm = fma(sm, ct, cm * st);
        cm = cn;
      }
    } else {
      const int s0 = (id - a.off[0]) * a.q_src;
      for (int i0 = 0; i0 < a.q_src; ++i0) {
        const int sr = s0 + i0;
        const double rx = x - __ldg(a.sx + sr), ry = y - __ldg(a.sy + sr);
        double inv, d, yq;
        kw.geom(fma(rx, rx, ry * ry), inv, d, yq);
        cplx h0, h1;
        T twoz;
        kw.hankel(d, inv, yq, h0, h1, twoz);
        cplx v[2];
        if (GRAD) {
          const cplx g = -smul(kk, h1);
          v[0] = (rx * inv) * g;
          v[1] = (ry * inv) * g;
        } else {
          v[0] = q.dip ? smul(rmul(kk, fma(rx, __ldg(a.snx + sr), ry * __ldg(a.sny + sr)) * inv), h1) : h0;
        }
#pragma unroll
        for (int i = 0; i < NR; ++i) {
          if (i > 0 && i >= q.nr) break;
          const cplx w = wd[(size_t)sr * a.nrhs + q.rhs0 + i];
#pragma unroll
          for (int g = 0; g < kC; ++g) cfma(acc[g][i], w, v[g]);
        }
      }
    }
  }
  if (!active) return;
  cplx* part = reinterpret_cast<cplx*>(q.part);
#pragma unroll
  for (int g = 0; g < kC; ++g)
#pragma unroll
    for (int i = 0; i < NR; ++i) {
      if (i >= q.nr) break;
      part[(((size_t)split * q.n_far + e) * kC + g) * a.nrhs + q.rhs0 + i] = acc[g][i];
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
    QBX_FAR(1) QBX_FAR(2) QBX_FAR(3) QBX_FAR(4) QBX_FAR(5) QBX_FAR(6) QBX_FAR(7) QBX_FAR(12) QBX_FAR(13)
    default: return cudaErrorInvalidValue;
  }
#undef QBX_FAR
}

template <typename T>
size_t moments_smem(int q_src) {
  return (size_t)((dipole_rows<T>(q_src) ? 4 * kTreeP + 12 : 2 * kTreeP + 8)) * (q_src | 1) * sizeof(T);
}

template <typename T>
size_t disc_moments_smem(int p) {
  return (size_t)(kTreeP + p + 4) * 32 * 16 + (size_t)(3 * p + 2) * 32 * sizeof(T);
}

template <typename T>
cudaError_t launch_moments_t(const TreeArgs& a, cudaStream_t st, int n_inst) {
  const int ncol = a.nset * a.nrhs;
  if (a.discs) {
    const size_t smem = disc_moments_smem<T>(a.p);
    cudaError_t e = cudaFuncSetAttribute(k_tree_disc_moments<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    k_tree_disc_moments<T><<<dim3(a.M, a.lev), 32, smem, st>>>(a);
  } else {
    const size_t smem = moments_smem<T>(a.q_src);
    cudaError_t e = cudaFuncSetAttribute(k_tree_moments<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    k_tree_moments<T><<<dim3(a.M, a.up ? 1 : a.lev, n_inst), 128, smem, st>>>(a);
  }
  if (a.up)
    for (int l = 1; l < a.lev; ++l)
      k_tree_up<T><<<dim3((a.M + (1 << l) - 1) >> l, (ncol + kUpWarps * kUpCols - 1) / (kUpWarps * kUpCols), n_inst),
                     32 * kUpWarps, 0, st>>>(a, l);
  if (!a.up) k_tree_fold<<<dim3(a.off[a.lev], ncol), 64, 0, st>>>(a);
  if (a.n_blk == 0) return cudaGetLastError();
  cudaError_t e = cudaFuncSetAttribute(k_tree_local<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(LocSmem));
  if (e != cudaSuccess) return e;
  const int ng = (ncol + kLocCols - 1) / kLocCols;
  if (a.n_sup) k_tree_local<T><<<dim3(a.n_sup, ng, n_inst), 32 * kLocWarps, sizeof(LocSmem), st>>>(a, true);
  k_tree_local<T><<<dim3(a.n_blk, ng, n_inst), 32 * kLocWarps, sizeof(LocSmem), st>>>(a, false);
  return cudaGetLastError();
}

}  // namespace

int tree_levels(int panels, int q_src, TreeArgs* a) {
  // (the discs of an adjoint's leaves reach past half a panel: whole panels there)
  // half panels as leaves where that leaves them 16 sources or more: near
  // pairs 2.05 -> 1.65 ms, far nodes 0.77 -> 0.99 ms (starfish, 256 panels)
  const int half = q_src % 2 == 0 && q_src >= 32 && !a->discs;
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
  // Super-blocks: nodes of a super-block's size are sup_c levels above it, by
  // the number of leaves next to 32 targets.  Many columns: from kSupMinLeaves
  // leaves on; few: from 64 blocks on (complex k: 128), where they are worth
  // their three launches (S + D + grad S, 128 blocks 3.25 -> 3.18 ms; shape step
  // of S, 64 and 256 blocks 4.68 -> 4.43; 64 blocks, complex k 3.41 -> 3.44)
  a->n_sup = a->sup_lev = a->sup_c = 0;
  if (!a->only_loc && (a->up ? a->M >= kSupMinLeaves : a->n_blk >= (a->kim != 0.0 ? 128 : 64))) {
    for (double r = 32.0 * a->M / a->n_tgt; r > 1.5; r *= 0.5) ++a->sup_c;
    a->sup_off[1] = 0;
    for (int B = 1; B <= kSupLevels && B + a->sup_c < a->lev; ++B) {
      a->sup_lev = B;
      a->n_sup += (a->n_blk + (1 << B) - 1) >> B;
      a->sup_off[B + 1] = a->n_sup;
    }
    a->sup_stride = (a->M >> (a->sup_c + 1)) + 2;
  }
  const size_t nodes = (size_t)a->off[a->lev] + a->n_blk + a->n_sup, ncol = (size_t)a->ncset * a->nrhs;
  a->node = (double*)take(nodes * 4 * 8);
  a->near = (int*)take((size_t)a->n_blk * a->M * 4);
  a->far = (int*)take((size_t)a->n_blk * (a->M + 1) * 8);
  a->loc = (int*)take((size_t)a->n_blk * a->M * 8);
  a->cnt = (int*)take((size_t)a->n_blk * 12);
  a->sloc = (int*)take((size_t)a->n_sup * a->sup_stride * 8);
  a->scnt = (int*)take((size_t)a->n_sup * 8);
  a->scov = (unsigned char*)take((size_t)a->n_sup * a->M);
  a->mom = take(a->up ? 0 : (size_t)a->lev * a->M * a->nset * a->nrhs * (kTreeP + 2) * 2 * 16);
  a->coef = take(nodes * ncol * (kTreeP + 2) * 2 * 16);
  return at;
}

cudaError_t launch_tree_lists(const TreeArgs& a, cudaStream_t st, int n_inst) {
  k_tree_nodes<<<dim3(a.off[a.lev], 1, n_inst), 256, 0, st>>>(a);
  if (a.n_sup) {
    k_tree_super<<<dim3(a.n_sup, 1, n_inst), 256, 0, st>>>(a);
    k_super_lists<<<dim3(a.n_sup, 1, n_inst), 256, 0, st>>>(a);
  }
  k_tree_lists<<<dim3(a.n_blk, 1, n_inst), 32 * kListWarps, 0, st>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_tree_moments(const TreeArgs& a, bool ck, cudaStream_t st, int n_inst) {
  return ck ? launch_moments_t<cplx>(a, st, n_inst) : launch_moments_t<double>(a, st, n_inst);
}

// Assembled matrix: the set-up of the tree over whole panels and its bytes
// (base null: only those); 0 where the entries are formed pair by pair.
size_t matrix_tree_setup(MatrixFarArgs* q, const qbx_geom* g, qbx_c64 k, qbx_c64 eta, int p, const double* hk_tab,
                         char* base) {
  *q = MatrixFarArgs{};
  TreeArgs& t = q->t;
  // (a panel's q_tgt columns of moments against its q_src sources: at 16/16 nodes
  // 1.25 to 1.42 times the pairs' time, 80 panels; at 16/64 0.36 to 0.99, at 8/32
  // 0.31 to 1.04)
  if (g->M < kTreeMinPanels || g->q_src > 128 || g->q_src < 2 * g->q_tgt) return 0;
  const bool ck = k.im != 0.0;
  const size_t setup = 2 * (ck ? far_col_bytes<cplx>(p) + far_warp_bytes<cplx>(p) : far_col_bytes<double>(p) + far_warp_bytes<double>(p));
  if (setup > sizeof(LocSmem) || (ck ? moments_smem<cplx>(g->q_src) : moments_smem<double>(g->q_src)) > 220 * 1024) return 0;
  t.kre = k.re;
  t.kim = k.im;
  t.eta_re = eta.re;
  t.eta_im = eta.im;
  t.p = t.pl = p;
  t.nd = 1;
  t.only_loc = 1;
  t.M = g->M;
  t.q_src = g->q_src;
  t.n_src = g->n_src;
  t.lev = 1;
  t.off[0] = 0;
  t.off[1] = g->M;
  t.sx = g->src_x;
  t.sy = g->src_y;
  t.snx = g->src_nx;
  t.sny = g->src_ny;
  t.n_tgt = g->n_tgt;
  t.n_ctr = 2 * g->n_tgt;
  t.cx = g->ctr_x;
  t.cy = g->ctr_y;
  t.tx = g->tgt_x;
  t.ty = g->tgt_y;
  t.hk_tab = hk_tab;
  t.n_blk = (g->n_tgt + 31) / 32;
  t.nrhs = g->q_tgt;
  t.up = 1;
  t.ops = OPB_C;
  const int none[3] = {0, 0, 0};
  tree_columns(&t, none);
  size_t at = tree_layout(&t, base);
  t.wd[0] = base ? base + at : nullptr;
  at += host_align256((size_t)g->n_src * g->q_tgt * 16);
  q->tw = g->tgt_w;
  return at;
}

template <typename T>
static cudaError_t launch_matrix_far_t(const MatrixFarArgs& q, const double* sw, const double* P, int num_sms,
                                       cudaStream_t st) {
  const TreeArgs& a = q.t;
  const int n = a.n_src * a.nrhs;
  k_matrix_density<<<(n + 255) / 256, 256, 0, st>>>(a.n_src, a.q_src, a.nrhs, sw, P, (cplx*)a.wd[0]);
  const size_t sm = moments_smem<T>(a.q_src);
  cudaError_t e = cudaFuncSetAttribute(k_tree_moments<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_tree_matrix<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(MatrixSmem));
  if (e != cudaSuccess) return e;
  k_tree_moments<T><<<dim3(a.M, 1, 1), 128, sm, st>>>(a);
  // one CTA (8 warps) per SM
  const unsigned ns = (unsigned)std::max(1, std::min((num_sms + a.n_blk - 1) / a.n_blk, (a.M + kLocWarps - 1) / kLocWarps));
  k_tree_matrix<T><<<dim3(a.n_blk, ns), 32 * kLocWarps, sizeof(MatrixSmem), st>>>(q);
  return cudaGetLastError();
}
cudaError_t launch_matrix_far(const MatrixFarArgs& q, const double* sw, const double* P, int num_sms, cudaStream_t st) {
  return q.t.kim != 0.0 ? launch_matrix_far_t<cplx>(q, sw, P, num_sms, st) : launch_matrix_far_t<double>(q, sw, P, num_sms, st);
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

cudaError_t launch_tree_nodes(const TreeArgs& a, cudaStream_t st) {
  k_tree_nodes<<<a.off[a.lev], 256, 0, st>>>(a);
  return cudaGetLastError();
}

template <typename T>
static int form_far_warps(int p) { return 2 * form_far_bytes<T>(p) <= 200 * 1024 ? 2 : form_far_bytes<T>(p) <= 200 * 1024 ? 1 : 0; }
bool form_far_fit(const TreeArgs& a) { return form_far_warps<double>(a.p) > 0; }

template <typename T>
static cudaError_t launch_form_far_t(const TreeArgs& a, cudaStream_t st) {
  const int w = form_far_warps<T>(a.p);
  const size_t smem = w * form_far_bytes<T>(a.p);
  cudaError_t e = cudaFuncSetAttribute(k_form_far<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  k_form_far<T><<<dim3((unsigned)(a.n_blk * (a.n_ctr / a.n_tgt)) * a.nsplit, a.nrhs), 32 * w, smem, st>>>(a);
  return cudaGetLastError();
}
cudaError_t launch_form_far(const TreeArgs& a, cudaStream_t st) {
  return a.kim != 0.0 ? launch_form_far_t<cplx>(a, st) : launch_form_far_t<double>(a, st);
}

template <typename T, int NR>
static cudaError_t launch_far_points_t(const FarPointArgs& a, cudaStream_t st) {
  const unsigned grid = (unsigned)((a.n_far + 127) / 128) * (unsigned)a.nsplit;
  if (a.grad) k_far_points<T, NR, true><<<grid, 128, 0, st>>>(a);
  else k_far_points<T, NR, false><<<grid, 128, 0, st>>>(a);
  return cudaGetLastError();
}
cudaError_t launch_far_points(FarPointArgs a, cudaStream_t st) {
  for (int r0 = 0; r0 < a.t.nrhs; r0 += 4) {
    a.rhs0 = r0;
    a.nr = std::min(4, a.t.nrhs - r0);
    cudaError_t e;
    if (a.t.kim != 0.0) e = a.nr == 1 ? launch_far_points_t<cplx, 1>(a, st) : launch_far_points_t<cplx, 4>(a, st);
    else e = a.nr == 1 ? launch_far_points_t<double, 1>(a, st) : launch_far_points_t<double, 4>(a, st);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

// Far sums of the adjoint sweeps (columns [split][source][ncol][nrhs]: value,
// gradient, d_xx, d_xy of the field of conj(g), as ops asks) to one row of
// their partial sums: conj of the value (S); of n . gradient (D); of value and
// gradient (S with the source-position gradient); of K_D = n . grad, grad K_D
// and grad (D's shape sweep, d_yy = -k^2 value - d_xx).
__global__ void k_adj_far(int mode, int n_src, int nsplit, int ncol, int nrhs, cplx k2, const cplx* in,
                          const double* snx, const double* sny, cplx* out) {
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= n_src * nrhs) return;
  const int s = idx / nrhs, r = idx - s * nrhs;
  cplx v[5];
  for (int q = 0; q < ncol; ++q) {
    v[q] = cplx{0.0, 0.0};
    for (int i = 0; i < nsplit; ++i) v[q] = v[q] + in[(((size_t)i * n_src + s) * ncol + q) * nrhs + r];
  }
  const double nx = snx[s], ny = sny[s];
  cplx o[5];
  int n = 0;
  if (mode == 0) {
    o[n++] = v[0];
  } else if (mode == 1) {
    o[n++] = nx * v[0] + ny * v[1];
  } else if (mode == 2) {
    for (int q = 0; q < 3; ++q) o[n++] = v[q];
  } else {
    const cplx yy = -(k2 * v[0]) - v[3];
    o[n++] = nx * v[1] + ny * v[2];
    o[n++] = nx * v[3] + ny * v[4];
    o[n++] = nx * v[4] + ny * yy;
    o[n++] = v[1];
    o[n++] = v[2];
  }
  for (int q = 0; q < n; ++q) out[((size_t)s * n + q) * nrhs + r] = conj(o[q]);
}

cudaError_t launch_adj_far(const TreeArgs& a, int mode, const double* snx, const double* sny, void* row,
                           cudaStream_t st) {
  const int ncol = (a.ops & 1) + 2 * (a.ops >> 2 & 1) + 2 * (a.ops >> 3 & 1);
  const cplx k{a.kre, a.kim};
  k_adj_far<<<(a.n_tgt * a.nrhs + 127) / 128, 128, 0, st>>>(mode, a.n_tgt, a.nsplit, ncol, a.nrhs, k * k,
                                                           (const cplx*)a.part, snx, sny, (cplx*)row);
  return cudaGetLastError();
}

size_t adj_tree_setup(TreeArgs* t, const qbx_geom* g, int c0, int nc, qbx_c64 k, int p, int ops, int nd, int nrhs,
                      const double* hk_tab, const void* gc, int num_sms, char* base) {
  *t = TreeArgs{};
  if (g->M < kTreeMinPanels) return 0;
  t->kre = k.re;
  t->kim = k.im;
  t->p = p;
  t->pl = 0;
  t->nd = nd;
  t->ops = ops;
  t->nrhs = nrhs;
  t->discs = 1;
  t->sx = g->tgt_x;
  t->sy = g->tgt_y;
  t->dcx = g->ctr_x + c0;
  t->dcy = g->ctr_y + c0;
  t->n_ctr_n = nc;
  t->tx = t->cx = g->src_x;
  t->ty = t->cy = g->src_y;
  t->n_tgt = t->n_ctr = g->n_src;
  t->n_blk = (g->n_src + 31) / 32;
  t->hk_tab = hk_tab;
  t->wd[0] = gc;
  tree_columns_discs(t);
  tree_levels(g->M, g->q_tgt, t);
  const size_t smem = k.im != 0.0 ? disc_moments_smem<cplx>(p) : disc_moments_smem<double>(p);
  if (smem > 220 * 1024 || !far_clusters_fit(*t)) return 0;
  t->nparts = std::max(1, std::min(4, num_sms * 8 / (t->n_blk * 16)));
  t->nsplit = std::max(1, std::min(4, (num_sms * 2 + t->n_blk - 1) / t->n_blk));
  size_t at = tree_layout(t, base);
  const int ncol = (ops & 1) + 2 * (ops >> 2 & 1) + 2 * (ops >> 3 & 1);
  t->part = base ? base + at : nullptr;
  return at + host_align256((size_t)t->nsplit * g->n_src * ncol * nrhs * 16);
}

bool far_group_fit(const TreeArgs& a, bool ck, int nsd) {
  return (ck ? FarGroupSmem<cplx>::bytes(a.pl, nsd) : FarGroupSmem<double>::bytes(a.pl, nsd)) <= 220 * 1024;
}

template <typename T, int RG>
static cudaError_t launch_far_group_t(const TreeArgs& a, cudaStream_t st, int n_inst) {
  const size_t smem = FarGroupSmem<T>::bytes(a.pl, a.n_ctr / a.n_tgt);
  auto kern = k_far_group<T, RG>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  kern<<<dim3((unsigned)a.n_blk * a.nsplit, 1, n_inst), 32 * kFgWarps, smem, st>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_far_group(const TreeArgs& a, bool ck, cudaStream_t st, int n_inst) {
  const int cols = ((a.ops & OPB_C) ? 1 : popc3(a.ops)) * a.nrhs;
  if (cols > 32) return ck ? launch_far_group_t<cplx, 8>(a, st, n_inst) : launch_far_group_t<double, 8>(a, st, n_inst);
  return ck ? launch_far_group_t<cplx, 4>(a, st, n_inst) : launch_far_group_t<double, 4>(a, st, n_inst);
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

static int shift_set(TreeArgs* a, int moment, int sh) {
  a->base[a->ncset] = moment;
  a->shift[a->ncset] = sh;
  return a->ncset++;
}

void tree_columns_grad_d(TreeArgs* a, bool sources) {
  a->nset = a->ncset = 0;
  const int m = moment_set(a, kSetNormal, 0);
  a->set_g = a->plain[m];
  a->set_gx = shift_set(a, m, 1);
  shift_set(a, m, 2);
  if (sources) {
    a->set_x = a->plain[moment_set(a, kSetQuadX, 0)];
    moment_set(a, kSetQuadY, 0);
  }
}

void tree_columns_discs(TreeArgs* a) {
  a->nset = a->ncset = 0;
  const int m = moment_set(a, kSetMono, 0);
  a->set_s = a->set_g = a->plain[m];
  if (a->ops & OPB_G) {
    a->set_gx = shift_set(a, m, 1);
    shift_set(a, m, 2);
  }
  if (a->ops & OPB_X) {
    a->set_x = shift_set(a, m, 3);
    shift_set(a, m, 4);
  }
}

void tree_columns(TreeArgs* a, const int slot[3]) {
  a->nset = a->ncset = 0;
  if (a->ops & OPB_C) {
    a->set_d = a->plain[moment_set(a, kSetCombined, slot[1])];
    return;
  }
  if (a->ops & OPB_S) a->set_s = a->plain[moment_set(a, kSetMono, slot[0])];
  if (a->ops & OPB_D) a->set_d = a->plain[moment_set(a, kSetNormal, slot[1])];
  if (a->ops & OPB_G) {
    const int m = moment_set(a, kSetMono, slot[2]);
    a->set_g = a->plain[m];
    a->set_gx = shift_set(a, m, 1);
    shift_set(a, m, 2);
  }
  if (a->ops & OPB_X) {
    a->set_x = a->plain[moment_set(a, kSetX, slot[2])];
    moment_set(a, kSetY, slot[2]);
  }
}

}  // namespace qbx
