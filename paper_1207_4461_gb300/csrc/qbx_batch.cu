// qbx_batch.cu -- many curves (each with its own panels, wavenumber and
// densities) applied in one persistent launch of the group kernel, run as a
// CUDA graph: [zero the item counter] -> [oversample every curve's
// densities] -> [cluster lists] -> [group kernel over the longest-first item
// list of near sources, beside cluster moments and far sums] -> [scale, jump
// terms / two-sided average into every curve's outputs].
#include <cuda_runtime.h>
#include <math.h>
#include <stdio.h>
#include <algorithm>
#include <map>
#include <mutex>
#include <numeric>
#include <tuple>
#include <vector>
#include "../../include/qbx.h"
#include "qbx_device.cuh"
#include "qbx_internal.h"

using namespace qbx;

struct qbx_batch {
  int device = 0, n_inst = 0, p = 0, ops = 0, side = 0, limit = 0, nrhs = 0, ncomp = 0, rg = 8;
  bool ck = false;
  int n_items = 0, grid = 0, max_src = 0, max_tgt = 0, num_sms = 0;
  int chunk = 0;                    // sources per work item (multiple of 32)
  double eta2 = 0.0;                // near-only QBX when > 0 (qbx_batch_set_eta)
  double* d_hk = nullptr;           // amplitude tables of the complex-k curves' rays
  size_t part_cap = 0;              // bytes allocated for the partial sums
  std::vector<qbx::GroupInst> h_inst;
  GroupInst* d_inst = nullptr;
  GroupItem* d_items = nullptr;
  int* d_counter = nullptr;
  int* d_status = nullptr;
  void* d_wd = nullptr;
  void* d_part = nullptr;
  const double* d_interp = nullptr;  // the plan's
  int q_tgt = 0, q_src = 0;
  cudaGraph_t graph = nullptr;
  cudaGraphExec_t exec = nullptr;
  int nsd = 1;                      // 2: both sides of a target averaged per pair (two-sided S, D, S + D)
  // distant sources through cluster moments (qbx_tree.cu): per-curve arguments
  bool tree = false;
  std::vector<qbx::TreeArgs> h_tree;
  TreeArgs* d_tree = nullptr;
  void* d_tree_mem = nullptr;
  int ns_far = 0;                   // far splits of every clustered curve
  int tree_q = 0;                   // sources per leaf
  cudaStream_t cap[2] = {nullptr, nullptr};   // the graph's two branches are captured from these
  cudaEvent_t ev[2] = {nullptr, nullptr};
};

namespace {

int bfail(int code, const char* what) {
  char buf[320];
  snprintf(buf, sizeof(buf), "qbx_batch: %s", what);
  return host_fail(code, buf);
}

int bcuda(cudaError_t e, const char* what) {
  char buf[320];
  snprintf(buf, sizeof(buf), "qbx_batch: %s: %s", what, cudaGetErrorString(e));
  return host_fail(QBX_ECUDA, buf);
}

// a1 for every curve: blockIdx.y = curve, wd[s][r] = w_s sum_i P[j][i] dens[m q_tgt + i][r]
__global__ void k_batch_upsample(const GroupInst* inst, int q_tgt, int q_src, int nrhs, const double* P) {
  const GroupInst& in = inst[blockIdx.y];
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= in.n_src * nrhs) return;
  const int s = idx / nrhs, r = idx - s * nrhs;
  const int m = s / q_src, j = s - m * q_src;
  const double* row = P + (size_t)j * q_tgt;
  const cplx* d = reinterpret_cast<const cplx*>(in.dens) + (size_t)m * q_tgt * nrhs + r;
  double re = 0.0, im = 0.0;
  for (int i = 0; i < q_tgt; ++i) {
    const double c = row[i];
    const cplx v = d[(size_t)i * nrhs];
    re = fma(c, v.re, re);
    im = fma(c, v.im, im);
  }
  const double w = in.sw[s];
  reinterpret_cast<cplx*>(const_cast<void*>(in.wd))[idx] = cplx{w * re, w * im};
}

// a7 for every curve: blockIdx.y = curve; component q of the partial rows
// belongs to operator op_of[q] (S, D, grad S x, grad S y in that order).
__global__ void k_batch_finish(const GroupInst* inst, int ops, int ncomp, int limit, int nrhs, int* status) {
  const GroupInst& in = inst[blockIdx.y];
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= in.n_tgt * ncomp * nrhs) return;
  const int t = idx / (ncomp * nrhs);
  const int rem = idx - t * ncomp * nrhs;
  const int q = rem / nrhs, r = rem - q * nrhs;
  // operator and component within it
  int op = 0, comp = 0, qq = q;
  for (int o = 0; o < 3; ++o) {
    if (!(ops >> o & 1)) continue;
    const int n = (o == QBX_OP_GRAD_S) ? 2 : 1;
    if (qq < n) {
      op = o;
      comp = qq;
      break;
    }
    qq -= n;
  }
  const cplx* part = reinterpret_cast<const cplx*>(in.part);
  const int nsides = in.n_row / in.n_tgt;   // (merged: the sums are the two-sided average already)
  cplx res{0.0, 0.0};
  for (int sd = 0; sd < nsides; ++sd) {
    const int c = t + sd * in.n_tgt;
    cplx u{0.0, 0.0};
    for (int k = 0; k < in.nsplit; ++k) u = u + part[(((size_t)k * in.n_row + c) * ncomp + q) * nrhs + r];
    u = mul_i(0.25 * u);
    if (in.side != QBX_SIDE_TWO && limit == QBX_LIMIT_PV) {
      const double sg = in.side == QBX_SIDE_EXT ? 1.0 : -1.0;
      const cplx dv = reinterpret_cast<const cplx*>(in.dens)[(size_t)t * nrhs + r];
      if (op == QBX_OP_D) u = u - (0.5 * sg) * dv;
      else if (op == QBX_OP_GRAD_S) u = u + (0.5 * sg * (comp == 0 ? in.tnx[t] : in.tny[t])) * dv;
    }
    res = res + u;
  }
  if (nsides == 2) res = 0.5 * res;
  const int nc_op = op == QBX_OP_GRAD_S ? 2 : 1;
  cplx* out = reinterpret_cast<cplx*>(in.out[op]);
  out[((size_t)t * nc_op + comp) * nrhs + r] = res;
  if (!(isfinite(res.re) && isfinite(res.im))) atomicOr(status, 1);
}

void destroy(qbx_batch* b) {
  if (!b) return;
  cudaSetDevice(b->device);
  if (b->exec) cudaGraphExecDestroy(b->exec);
  if (b->graph) cudaGraphDestroy(b->graph);
  cudaFree(b->d_inst);
  cudaFree(b->d_items);
  cudaFree(b->d_counter);
  cudaFree(b->d_status);
  cudaFree(b->d_wd);
  cudaFree(b->d_part);
  cudaFree(b->d_hk);
  cudaFree(b->d_tree);
  cudaFree(b->d_tree_mem);
  for (int i = 0; i < 2; ++i) {
    if (b->cap[i]) cudaStreamDestroy(b->cap[i]);
    if (b->ev[i]) cudaEventDestroy(b->ev[i]);
  }
  delete b;
}


// Sources of a work item's block: all of the curve's, or with clusters about
// the six panels that stay near (the kernel takes the list's actual share).
int block_sources(const GroupInst& in) {
  return in.near ? std::min(in.n_src, 6 * (in.n_src / in.M)) : in.n_src;
}

// Work items of a configuration: 32 rows of one curve (with a near list: of one
// side, otherwise across the sides: both sides of 400 centres are 25 blocks, not
// 26) x a range of at most `chunk` of its sources (equal ranges per curve),
// longest first.  Both sides of a target in one item take twice as long per
// source: a curve without a near list has twice the ranges then (one curve of
// 16 panels, S, both sides, 32 rhs: 1460 us; with the ranges of one side 2289;
// with one side per item 1442).
std::vector<GroupItem> make_items(const std::vector<GroupInst>& inst, int nsd, int chunk, std::vector<int>& nsplit) {
  std::vector<GroupItem> items;
  nsplit.assign(inst.size(), 1);
  for (size_t i = 0; i < inst.size(); ++i) {
    const int n = block_sources(inst[i]);
    int ns = std::max(1, (n + chunk - 1) / chunk);
    if (nsd == 2 && !inst[i].near) ns = std::min(2 * ns, std::max(1, n / 16));
    const int len = (n + ns - 1) / ns;
    ns = (n + len - 1) / len;   // every range non-empty
    nsplit[i] = ns;
    const int run = inst[i].near ? inst[i].n_tgt : inst[i].n_row;
    for (int r = 0; r < inst[i].n_row; r += run)
      for (int c = r; c < r + run; c += kGrpCentres)
        for (int k = 0; k < ns; ++k)
          items.push_back(GroupItem{(int)i, c, std::min(r + run, c + kGrpCentres), k, k * len, std::min(n, (k + 1) * len)});
  }
  std::stable_sort(items.begin(), items.end(), [&](const GroupItem& x, const GroupItem& y) {
    const long cx = (long)(x.row1 - x.row0) * (x.src1 - x.src0);
    const long cy = (long)(y.row1 - y.row0) * (y.src1 - y.src0);
    return cx > cy;
  });
  return items;
}

// (the pair kernel's nsplit rows, and a clustered curve's ns_far more)
size_t part_bytes(const std::vector<GroupInst>& inst, const std::vector<int>& nsplit, int ns_far, int ncomp, int nrhs) {
  size_t t = 0;
  for (size_t i = 0; i < inst.size(); ++i)
    t += host_align256((size_t)(nsplit[i] + (inst[i].near ? ns_far : 0)) * inst[i].n_row * ncomp * nrhs * 16);
  return t;
}

// Predicted makespan (in pair units) of the persistent grid taking the items
// in list order: each of `slots` CTAs takes the next item when it finishes
// (the atomic counter), an item costs its pairs plus a fixed set-up share.
double lpt_makespan(const std::vector<GroupItem>& items, int slots) {
  std::vector<double> heap(std::max(1, slots), 0.0);   // min-heap of finish times
  auto cmp = [](double x, double y) { return x > y; };
  for (const GroupItem& it : items) {
    std::pop_heap(heap.begin(), heap.end(), cmp);
    const double pairs = (double)(it.row1 - it.row0) * (it.src1 - it.src0);
    heap.back() += pairs + 32.0 * kGrpTile;   // + one tile's worth of set-up per item
    std::push_heap(heap.begin(), heap.end(), cmp);
  }
  return *std::max_element(heap.begin(), heap.end());
}

// smallest source range of an item (with clusters a block has few hundred sources in all)
int min_chunk(const qbx_batch* b) { return b->tree ? 64 : 512; }

// sources of an item that has the range `chunk` (make_items)
int item_sources(const qbx_batch* b, int chunk) { return b->nsd == 2 && !b->tree ? (chunk + 1) / 2 : chunk; }

// The source chunk the model prefers: the smallest predicted makespan over
// chunks 2^j * 32 (and all sources), ties to the larger chunk (fewer
// partial sums), within the partial-sum memory budget.
int model_chunk(const qbx_batch* b, int slots, size_t budget) {
  std::vector<int> cand{(b->max_src + kGrpTile - 1) / kGrpTile * kGrpTile};
  for (int c = 1 << 20; c >= min_chunk(b); c /= 2)
    if (c < b->max_src) cand.push_back(c);
  int best = cand[0];
  double bt = 1e300;
  std::vector<int> ns;
  for (int c : cand) {
    std::vector<GroupItem> items = make_items(b->h_inst, b->nsd, c, ns);
    if (part_bytes(b->h_inst, ns, b->ns_far, b->ncomp, b->nrhs) > budget) break;
    const double t = lpt_makespan(items, slots);
    if (t < bt * 0.995) {
      bt = t;
      best = c;
    }
  }
  return best;
}

// (Re)build the batch for (rg, chunk): items, partial-sum layout, device
// tables, and the graph [counter := 0] -> [oversample] -> [group] -> [finish].
int configure(qbx_batch* b, int rg, int chunk) {
  cudaError_t e = cudaSetDevice(b->device);
  if (e != cudaSuccess) return bcuda(e, "device");
  std::vector<int> ns;
  std::vector<GroupItem> items = make_items(b->h_inst, b->nsd, chunk, ns);
  const size_t pb = part_bytes(b->h_inst, ns, b->ns_far, b->ncomp, b->nrhs);
  if (pb > b->part_cap) {
    cudaFree(b->d_part);
    b->d_part = nullptr;
    b->part_cap = 0;
    e = cudaMalloc(&b->d_part, pb);
    if (e != cudaSuccess) return bcuda(e, "partial-sum allocation");
    b->part_cap = pb;
  }
  if (items.size() > (size_t)b->n_items) {
    cudaFree(b->d_items);
    b->d_items = nullptr;
    e = cudaMalloc(&b->d_items, sizeof(GroupItem) * items.size());
    if (e != cudaSuccess) return bcuda(e, "item-list allocation");
  }
  size_t off = 0;
  for (int i = 0; i < b->n_inst; ++i) {
    GroupInst& in = b->h_inst[i];
    in.nsplit_near = ns[i];
    in.nsplit = ns[i] + (in.near ? b->ns_far : 0);
    in.part = static_cast<char*>(b->d_part) + off;
    off += host_align256((size_t)in.nsplit * in.n_row * b->ncomp * b->nrhs * 16);
    if (b->tree) {
      b->h_tree[i].part = in.part;
      b->h_tree[i].split0 = ns[i];
      b->h_tree[i].nsplit = in.near ? b->ns_far : 0;
    }
  }
  e = cudaMemcpy(b->d_inst, b->h_inst.data(), sizeof(GroupInst) * b->n_inst, cudaMemcpyHostToDevice);
  if (e == cudaSuccess && b->tree)
    e = cudaMemcpy(b->d_tree, b->h_tree.data(), sizeof(TreeArgs) * b->n_inst, cudaMemcpyHostToDevice);
  if (e == cudaSuccess)
    e = cudaMemcpy(b->d_items, items.data(), sizeof(GroupItem) * items.size(), cudaMemcpyHostToDevice);
  if (e != cudaSuccess) return bcuda(e, "upload");
  b->n_items = (int)items.size();
  b->rg = rg;
  b->chunk = chunk;
  const bool local = b->eta2 > 0.0;
  const int occ = local ? group_occupancy_local(b->ops, b->ck, b->p, rg, b->nsd)
                        : (b->ck ? group_occupancy_cplx(b->ops, b->p, rg, b->nsd)
                                 : group_occupancy_real(b->ops, b->p, rg, b->nsd));
  const size_t gsmem = b->ck ? group_smem_cplx(b->ops, b->p, rg, b->nsd) : group_smem_real(b->ops, b->p, rg, b->nsd);
  if (occ < 1 || gsmem > 220 * 1024) return bfail(QBX_EINVAL, "p too large for the group kernel");
  b->grid = std::min(b->n_items, b->num_sms * occ);
  if (b->exec) cudaGraphExecDestroy(b->exec);
  if (b->graph) cudaGraphDestroy(b->graph);
  b->exec = nullptr;
  b->graph = nullptr;
  GroupArgs ga{};
  ga.ops = b->ops;
  ga.p = b->p;
  ga.nrhs = b->nrhs;
  ga.nsd = b->nsd;
  ga.inst = b->d_inst;
  ga.n_items = b->n_items;
  ga.items = b->d_items;
  ga.counter = b->d_counter;
  ga.eta2 = b->eta2;
  // the graph, captured from two streams of the batch's own: the pair sums
  // beside the cluster moments and far sums
  for (int i = 0; i < 2 && e == cudaSuccess; ++i) {
    if (!b->cap[i]) e = cudaStreamCreateWithFlags(&b->cap[i], cudaStreamNonBlocking);
    if (e == cudaSuccess && !b->ev[i]) e = cudaEventCreateWithFlags(&b->ev[i], cudaEventDisableTiming);
  }
  if (e == cudaSuccess) e = cudaStreamBeginCapture(b->cap[0], cudaStreamCaptureModeThreadLocal);
  if (e != cudaSuccess) return bcuda(e, "graph capture");
  cudaStream_t s0 = b->cap[0], s1 = b->tree ? b->cap[1] : b->cap[0];
  auto ok = [&](cudaError_t x) {
    if (e == cudaSuccess) e = x;
  };
  ok(cudaMemsetAsync(b->d_counter, 0, sizeof(int), s0));
  k_batch_upsample<<<dim3((b->max_src * b->nrhs + 255) / 256, b->n_inst), 256, 0, s0>>>(b->d_inst, b->q_tgt, b->q_src,
                                                                                       b->nrhs, b->d_interp);
  ok(cudaGetLastError());
  TreeArgs tr{};
  if (b->tree) {   // launch sizes: the largest over the curves
    tr = b->h_tree[0];
    tr.inst = b->d_tree;
    for (const TreeArgs& t : b->h_tree) {
      tr.M = std::max(tr.M, t.M);
      tr.n_blk = std::max(tr.n_blk, t.n_blk);
      tr.n_sup = std::max(tr.n_sup, t.n_sup);
      if (t.off[t.lev] > tr.off[tr.lev]) {
        tr.lev = t.lev;
        for (int l = 0; l <= t.lev; ++l) tr.off[l] = t.off[l];
      }
    }
    tr.q_src = b->tree_q;
    tr.nsplit = b->ns_far;
    ok(launch_tree_lists(tr, s0, b->n_inst));
    ok(cudaEventRecord(b->ev[0], s0));
    ok(cudaStreamWaitEvent(s1, b->ev[0], 0));
  }
  if (local) ok(launch_group_local(ga, b->ck, rg, b->grid, s1));
  else ok(b->ck ? launch_group_cplx(ga, rg, b->grid, s1) : launch_group_real(ga, rg, b->grid, s1));
  if (b->tree) {
    ok(launch_tree_moments(tr, b->ck, s0, b->n_inst));
    ok(launch_far_group(tr, b->ck, s0, b->n_inst));
    ok(cudaEventRecord(b->ev[1], s1));
    ok(cudaStreamWaitEvent(s0, b->ev[1], 0));
  }
  k_batch_finish<<<dim3((b->max_tgt * b->ncomp * b->nrhs + 255) / 256, b->n_inst), 256, 0, s0>>>(
      b->d_inst, b->ops, b->ncomp, b->limit, b->nrhs, b->d_status);
  ok(cudaGetLastError());
  const cudaError_t ec = cudaStreamEndCapture(s0, &b->graph);   // (also after an error)
  ok(ec);
  if (e == cudaSuccess) e = cudaGraphInstantiate(&b->exec, b->graph, 0);
  if (e != cudaSuccess) return bcuda(e, "graph construction");
  return QBX_OK;
}

// Cluster arrays of every curve with enough panels (many columns: S, D or
// S + D), for the batch's eta: sizes them, allocates on first use, and points
// the curves' pair sums at their near lists.  Without memory for them, or for
// orders the far kernel cannot hold, every pair goes pair by pair.
int prepare_tree(qbx_batch* b, size_t budget) {
  b->tree = false;
  for (GroupInst& in : b->h_inst) in.near = nullptr;
  if (b->ops == (QBX_OPS_S | QBX_OPS_D | QBX_OPS_GRAD_S)) return QBX_OK;
  // (the clusters' chain of launches is repaid from about 2.3e6 pairs on: one
  // curve of 48 panels, 32 rhs, S + D; up to 16 rhs from 1e6; near-only and with
  // leaves of few sources later, as one curve's apply: 12 curves of 100 panels of
  // 4/8 nodes, S + D of 32 rhs, 3.8e6 pairs in all, 5164 us against 4205)
  double pairs = 0.0;
  for (const GroupInst& in : b->h_inst) pairs += (double)in.n_ctr * in.n_src;
  const bool many = b->nrhs > 16, half_leaves = b->q_src % 2 == 0 && b->q_src >= 32;
  const double leaf = std::max(1.0, 20.0 / (half_leaves ? b->q_src / 2 : b->q_src));
  if (pairs < leaf * (b->eta2 > 0.0 ? (b->side == QBX_SIDE_TWO ? 3.2e6 : many ? 3.6e6 : 2.0e6) : many ? 2.3e6 : 1.0e6))
    return QBX_OK;
  const int none[3] = {0, 0, 0};
  std::vector<TreeArgs> v(b->n_inst);
  size_t total = 0;
  long blocks = 0;
  for (int i = 0; i < b->n_inst; ++i) {
    const GroupInst& in = b->h_inst[i];
    TreeArgs& t = v[i];
    t = TreeArgs{};
    t.kre = in.kre;
    t.kim = in.kim;
    t.p = b->p;
    t.pl = b->eta2 > 0.0 ? std::max(b->p, kTreeLocal) : b->p;
    t.nd = (b->ops & QBX_OPS_D) ? 1 : 0;
    t.eta = sqrt(b->eta2);
    t.n_tgt = in.n_tgt;
    t.n_ctr = in.n_ctr;
    t.ops = b->ops;
    t.nrhs = b->nrhs;
    t.up = 1;
    tree_columns(&t, none);
    if (in.M < kTreeMinPanels) continue;   // (no levels, leaves or blocks)
    tree_levels(in.M, b->q_src, &t);
    b->tree_q = t.q_src;
    t.n_blk = (in.n_tgt + kGrpCentres - 1) / kGrpCentres;
    blocks += t.n_blk;
    t.sx = in.sx;
    t.sy = in.sy;
    t.snx = in.snx;
    t.sny = in.sny;
    t.cx = in.cx;
    t.cy = in.cy;
    t.tx = in.tx;
    t.ty = in.ty;
    t.hk_tab = in.hk_tab;
    for (int s = 0; s < t.nset; ++s) t.wd[s] = in.wd;
    total += tree_layout(&t, nullptr);
  }
  if (total == 0 || !far_group_fit(v[0], b->ck, b->h_inst[0].n_ctr / b->h_inst[0].n_tgt)) return QBX_OK;
  if (!b->d_tree_mem) {
    if (total > budget) return QBX_OK;
    cudaError_t e = cudaMalloc(&b->d_tree_mem, total);
    if (e == cudaSuccess) e = cudaMalloc(&b->d_tree, sizeof(TreeArgs) * b->n_inst);
    if (e != cudaSuccess) {
      cudaGetLastError();
      cudaFree(b->d_tree_mem);
      b->d_tree_mem = nullptr;
      return QBX_OK;
    }
  }
  b->tree = true;
  b->ns_far = (int)std::max<long>(1, std::min<long>(4, (b->num_sms * 3 + blocks - 1) / blocks));
  size_t off = 0;
  for (int i = 0; i < b->n_inst; ++i) {
    if (v[i].n_blk == 0) continue;
    off += tree_layout(&v[i], static_cast<char*>(b->d_tree_mem) + off);
    b->h_inst[i].near = v[i].near;
    b->h_inst[i].near_cnt = v[i].cnt;
    b->h_inst[i].near_stride = v[i].M;
    b->h_inst[i].near_q = v[i].q_src;
  }
  b->h_tree = v;
  return QBX_OK;
}

// Tuned configurations, cached per (device, p, operators, side, nrhs, real or
// complex k, global or near-only, with clusters or without (whose thresholds
// lie inside the buckets), and the power-of-two buckets of the largest curve,
// the total pairs and the curve count): a batch created later with the same key
// starts from the measured choice instead of the model's.
typedef std::tuple<int, int, int, int, int, int, int, int, int, int, int> TuneKey;
std::mutex g_tune_mu;
std::map<TuneKey, std::pair<int, int>> g_tune_cache;

int log2i(double v) { return v < 1.0 ? 0 : (int)std::floor(std::log2(v)); }

TuneKey tune_key(const qbx_batch* b) {
  double pairs = 0.0;
  for (const GroupInst& in : b->h_inst) pairs += (double)in.n_ctr * in.n_src;
  return TuneKey{b->device, b->p, b->ops, b->side, b->nrhs, b->ck ? 1 : 0, b->eta2 > 0.0 ? 1 : 0,
                 b->tree ? 1 : 0, log2i(b->max_src), log2i(pairs), log2i(b->n_inst)};
}

// partial-sum budget: a quarter of the free device memory
size_t part_budget(int device) {
  size_t fr = 0, tot = 0;
  cudaSetDevice(device);
  if (cudaMemGetInfo(&fr, &tot) != cudaSuccess) return (size_t)1 << 30;
  return fr / 4;
}

}  // namespace

extern "C" {

int qbx_batch_create(qbx_batch** batch, qbx_plan* plan, int n_inst, const qbx_geom* geoms, const qbx_c64* k,
                     int p, int ops, int side, int limit, int nrhs, const qbx_c64* const* dens,
                     qbx_c64* const* out) {
  if (!batch) return bfail(QBX_EINVAL, "batch out-pointer is NULL");
  *batch = nullptr;
  if (!plan) return bfail(QBX_EINVAL, "plan is NULL");
  if (n_inst < 1 || !geoms || !k || !dens || !out) return bfail(QBX_EINVAL, "empty batch or NULL table");
  if (ops != QBX_OPS_S && ops != QBX_OPS_D && ops != (QBX_OPS_S | QBX_OPS_D) &&
      ops != (QBX_OPS_S | QBX_OPS_D | QBX_OPS_GRAD_S))
    return bfail(QBX_EINVAL, "operator set must be S, D, S+D or S+D+grad S");
  if (side != QBX_SIDE_INT && side != QBX_SIDE_EXT && side != QBX_SIDE_TWO) return bfail(QBX_EINVAL, "bad side");
  if (limit != QBX_LIMIT_ONE_SIDED && limit != QBX_LIMIT_PV) return bfail(QBX_EINVAL, "bad limit");
  if (p < 0 || p > QBX_MAX_P) return bfail(QBX_EINVAL, "p outside [0, QBX_MAX_P]");
  if (nrhs < 1) return bfail(QBX_EINVAL, "nrhs < 1");
  qbx_batch* b = new qbx_batch();
  b->n_inst = n_inst;
  b->p = p;
  b->ops = ops;
  b->side = side;
  b->limit = limit;
  b->nrhs = nrhs;
  b->ncomp = (ops & 1) + ((ops >> 1) & 1) + 2 * ((ops >> 2) & 1);
  b->rg = nrhs > 8 ? 8 : 2;
  b->nsd = side == QBX_SIDE_TWO && b->ncomp <= 2 ? 2 : 1;
  // the plan's device, grid pair and interpolation matrix
  int num_sms = 0;
  host_plan_info(plan, &b->device, &b->q_tgt, &b->q_src, &b->d_interp);
  cudaError_t e = cudaSetDevice(b->device);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&num_sms, cudaDevAttrMultiProcessorCount, b->device);
  if (e != cudaSuccess) {
    destroy(b);
    return bcuda(e, "device");
  }
  // ---- instances ----
  std::vector<GroupInst> inst(n_inst);
  size_t wd_total = 0;
  std::vector<size_t> wd_off(n_inst);
  for (int i = 0; i < n_inst; ++i) {
    const qbx_geom& g = geoms[i];
    if (g.q_tgt != b->q_tgt || g.q_src != b->q_src || g.M < 1 || g.n_tgt != g.M * g.q_tgt ||
        g.n_src != g.M * g.q_src || !g.src_x || !g.ctr_x || !g.tgt_x || !g.src_w) {
      destroy(b);
      return bfail(QBX_EINVAL, "geometry of an instance inconsistent with the plan");
    }
    if (!isfinite(k[i].re) || !isfinite(k[i].im) || k[i].im < 0.0 || (k[i].im == 0.0 && !(k[i].re > 0.0))) {
      destroy(b);
      return bfail(QBX_EINVAL, "k of an instance must be finite with Im k >= 0 (real k > 0)");
    }
    if (!dens[i]) {
      destroy(b);
      return bfail(QBX_EINVAL, "NULL density");
    }
    for (int o = 0; o < 3; ++o)
      if ((ops >> o & 1) && !out[3 * i + o]) {
        destroy(b);
        return bfail(QBX_EINVAL, "NULL output of a requested operator");
      }
    if (k[i].im != 0.0) b->ck = true;
    GroupInst& in = inst[i];
    in.kre = k[i].re;
    in.kim = k[i].im;
    in.n_src = g.n_src;
    in.n_tgt = g.n_tgt;
    in.M = g.M;
    in.side = side;
    in.n_ctr = side == QBX_SIDE_TWO ? 2 * g.n_tgt : g.n_tgt;
    in.n_row = b->nsd == 2 ? g.n_tgt : in.n_ctr;
    const int c0 = side == QBX_SIDE_EXT ? g.n_tgt : 0;
    in.nsplit = 1;
    in.sx = g.src_x;
    in.sy = g.src_y;
    in.snx = g.src_nx;
    in.sny = g.src_ny;
    in.sw = g.src_w;
    in.cx = g.ctr_x + c0;
    in.cy = g.ctr_y + c0;
    in.tx = g.tgt_x;
    in.ty = g.tgt_y;
    in.tnx = g.tgt_nx;
    in.tny = g.tgt_ny;
    in.dens = dens[i];
    for (int o = 0; o < 3; ++o) in.out[o] = out[3 * i + o];
    wd_off[i] = wd_total;
    wd_total += host_align256((size_t)g.n_src * nrhs * 16);
    b->max_src = std::max(b->max_src, g.n_src);
    b->max_tgt = std::max(b->max_tgt, g.n_tgt);
  }
  b->num_sms = num_sms;
  b->h_inst = inst;
  // ---- device memory: instance table, densities, counter, status ----
  int n_ck = 0;
  for (int i = 0; i < n_inst; ++i) n_ck += inst[i].kim != 0.0 ? 1 : 0;
  e = cudaMalloc(&b->d_wd, wd_total);
  if (e == cudaSuccess && n_ck > 0) e = cudaMalloc(&b->d_hk, (size_t)n_ck * hk_table_doubles() * sizeof(double));
  if (e == cudaSuccess) e = cudaMalloc(&b->d_inst, sizeof(GroupInst) * n_inst);
  if (e == cudaSuccess) e = cudaMalloc(&b->d_counter, sizeof(int));
  if (e == cudaSuccess) e = cudaMalloc(&b->d_status, sizeof(int));
  if (e == cudaSuccess) e = cudaMemset(b->d_status, 0, sizeof(int));
  if (e != cudaSuccess) {
    destroy(b);
    return bcuda(e, "allocation");
  }
  for (int i = 0; i < n_inst; ++i) b->h_inst[i].wd = static_cast<char*>(b->d_wd) + wd_off[i];
  // complex k: each curve's amplitude table (the k of a curve is fixed for the batch's life)
  for (int i = 0, j = 0; i < n_inst; ++i) {
    GroupInst& in = b->h_inst[i];
    in.hk_tab = nullptr;
    if (in.kim == 0.0) continue;
    double* t = b->d_hk + (size_t)(j++) * hk_table_doubles();
    e = launch_hk_table(in.kre, in.kim, t, 0);
    if (e != cudaSuccess) {
      destroy(b);
      return bcuda(e, "complex-k amplitude tables");
    }
    in.hk_tab = t;
  }
  e = cudaStreamSynchronize(0);   // made before any apply, on whatever stream it runs
  if (e != cudaSuccess) {
    destroy(b);
    return bcuda(e, "complex-k amplitude tables");
  }
  // ---- items: the source chunk the makespan model prefers ----
  const int occ = b->ck ? group_occupancy_cplx(ops, p, b->rg, b->nsd) : group_occupancy_real(ops, p, b->rg, b->nsd);
  if (occ < 1) {
    destroy(b);
    return bfail(QBX_EINVAL, "p too large for the group kernel");
  }
  prepare_tree(b, part_budget(b->device));
  int rg = b->rg, chunk = 0;
  {
    std::lock_guard<std::mutex> lk(g_tune_mu);
    auto it = g_tune_cache.find(tune_key(b));
    if (it != g_tune_cache.end()) {
      rg = it->second.first;
      chunk = it->second.second;
    }
  }
  if (chunk > 0) {   // a cached choice, if its partial sums fit
    std::vector<int> ns;
    make_items(b->h_inst, b->nsd, chunk, ns);
    if (part_bytes(b->h_inst, ns, b->ns_far, b->ncomp, b->nrhs) > part_budget(b->device)) chunk = 0;
  }
  if (chunk == 0) {
    rg = b->rg;
    chunk = model_chunk(b, num_sms * occ, part_budget(b->device));
  }
  if (int rc = configure(b, rg, chunk)) {
    destroy(b);
    return rc;
  }
  *batch = b;
  return QBX_OK;
}

int qbx_batch_tune(qbx_batch* b, void* stream, int* rg_out, int* chunk_out) {
  if (!b) return bfail(QBX_EINVAL, "batch is NULL");
  cudaError_t e = cudaSetDevice(b->device);
  if (e != cudaSuccess) return bcuda(e, "device");
  cudaStream_t st = (cudaStream_t)stream;
  // candidates: the model's chunk and its neighbours, for the rhs groupings
  // that apply (8 rhs per warp needs more than 8 rhs to pay off)
  const size_t budget = part_budget(b->device) + b->part_cap;
  const int c0 = b->chunk;
  std::vector<int> chunks{c0};
  if (c0 / 2 >= min_chunk(b)) chunks.push_back(c0 / 2);
  if (c0 < b->max_src) chunks.push_back(std::min(2 * c0, (b->max_src + kGrpTile - 1) / kGrpTile * kGrpTile));
  std::vector<int> rgs{b->nrhs > 8 ? 8 : 2};
  if (b->nrhs > 2 && b->nrhs % 32 != 0) rgs.push_back(rgs[0] == 8 ? 2 : 8);
  cudaEvent_t e0, e1;
  if ((e = cudaEventCreate(&e0)) != cudaSuccess) return bcuda(e, "event");
  if ((e = cudaEventCreate(&e1)) != cudaSuccess) {
    cudaEventDestroy(e0);
    return bcuda(e, "event");
  }
  float best_ms = 1e30f;
  int best_rg = b->rg, best_chunk = c0;
  int rc = QBX_OK;
  for (int rg : rgs) {
    for (int c : chunks) {
      std::vector<int> ns;
      make_items(b->h_inst, b->nsd, c, ns);
      if (part_bytes(b->h_inst, ns, b->ns_far, b->ncomp, b->nrhs) > budget) continue;
      if ((rc = configure(b, rg, c))) break;
      // one untimed launch, then one timed
      e = cudaGraphLaunch(b->exec, st);
      if (e == cudaSuccess) e = cudaEventRecord(e0, st);
      if (e == cudaSuccess) e = cudaGraphLaunch(b->exec, st);
      if (e == cudaSuccess) e = cudaEventRecord(e1, st);
      if (e == cudaSuccess) e = cudaEventSynchronize(e1);
      float ms = 0.0f;
      if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, e0, e1);
      if (e != cudaSuccess) {
        rc = bcuda(e, "tuning launch");
        break;
      }
      if (ms < best_ms) {
        best_ms = ms;
        best_rg = rg;
        best_chunk = c;
      }
    }
    if (rc) break;
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  if (rc) return rc;
  if ((rc = configure(b, best_rg, best_chunk))) return rc;
  {
    std::lock_guard<std::mutex> lk(g_tune_mu);
    g_tune_cache[tune_key(b)] = std::make_pair(best_rg, best_chunk);
  }
  if (rg_out) *rg_out = best_rg;
  if (chunk_out) *chunk_out = item_sources(b, best_chunk);
  return QBX_OK;
}

int qbx_batch_set_eta(qbx_batch* b, double eta) {
  if (!b) return bfail(QBX_EINVAL, "NULL batch");
  if (!(eta >= 0.0) || !isfinite(eta)) return bfail(QBX_EINVAL, "eta must be finite and >= 0");
  b->eta2 = eta * eta;
  const bool was = b->tree;
  prepare_tree(b, part_budget(b->device));
  if (was != b->tree)   // other items, other ranges
    b->chunk = model_chunk(b, b->grid, part_budget(b->device) + b->part_cap);
  return configure(b, b->rg, b->chunk);
}

int qbx_batch_info(const qbx_batch* b, int* rg, int* chunk, int* n_items, int* grid) {
  if (!b) return bfail(QBX_EINVAL, "batch is NULL");
  if (rg) *rg = b->rg;
  if (chunk) *chunk = item_sources(b, b->chunk);
  if (n_items) *n_items = b->n_items;
  if (grid) *grid = b->grid;
  return QBX_OK;
}

int qbx_batch_apply(qbx_batch* b, void* stream) {
  if (!b) return bfail(QBX_EINVAL, "batch is NULL");
  cudaError_t e = cudaSetDevice(b->device);
  if (e == cudaSuccess) e = cudaGraphLaunch(b->exec, (cudaStream_t)stream);
  if (e != cudaSuccess) return bcuda(e, "graph launch");
  return QBX_OK;
}

int qbx_batch_status(qbx_batch* b, void* stream) {
  if (!b) return bfail(QBX_EINVAL, "batch is NULL");
  int h = 0;
  cudaStream_t st = (cudaStream_t)stream;
  cudaError_t e = cudaMemcpyAsync(&h, b->d_status, sizeof(int), cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e == cudaSuccess) e = cudaMemsetAsync(b->d_status, 0, sizeof(int), st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) return bcuda(e, "status");
  if (h) return bfail(QBX_ENONFINITE, "a kernel produced a non-finite value");
  return QBX_OK;
}

int qbx_debug_batch_route(const qbx_batch* b, int* clusters) {
  if (!b || !clusters) return bfail(QBX_EINVAL, "NULL argument");
  *clusters = b->tree ? 1 : 0;
  return QBX_OK;
}

int qbx_batch_destroy(qbx_batch* b) {
  destroy(b);
  return QBX_OK;
}

}  // extern "C"
