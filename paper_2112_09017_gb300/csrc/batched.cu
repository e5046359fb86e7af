// Batched Newton-Schulz polar factorisations: many independent problems of uneven sizes, each with its own
// stop rule. A run is seven launches, captured once in a CUDA graph: norms, the planes of every problem, the
// small problems' loops on one SM each (onchip.cu), the other problems' loops in one cooperative launch that
// also forms U^T A of all of them (coop_batch.cu), U, H, and the results.
#include <math.h>
#include <stdint.h>
#include <string.h>

#include <algorithm>
#include <new>
#include <numeric>
#include <vector>

#include "batched.cuh"
#include "device_util.cuh"

namespace polar {

namespace {

constexpr int kThreads = 256;
constexpr int kStored = 3;       // BF16 planes kept for X and G
constexpr int kTile = 128;       // rows and columns of the loop's tiles
constexpr int kMaxSplit = 64;    // most blocks per problem of the passes over A, U and H

int64_t up(int64_t x, int64_t a) { return (x + a - 1) / a * a; }

__device__ __forceinline__ double block_sum_b(double v) {
  __shared__ double red[kThreads / 32];
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  __syncthreads();
  if (l == 0) red[w] = v;
  __syncthreads();
  double t = 0.0;
  if (threadIdx.x == 0)
    for (int i = 0; i < (int)(blockDim.x >> 5); ++i) t += red[i];
  return t;
}

// Sums of squares of every problem's A, one per block at the head of its residual history (which the loop
// fills later). Grid (count, Y), Y <= kMaxSplit. One block per problem, in FP64, took 1845 us for the
// 256-problem batch (n 64..1024).
__global__ void b_norm_kernel(const float* const* __restrict__ A, const BMeta* __restrict__ meta,
                              DevState* __restrict__ st, BShared* sh) {
  const int p = blockIdx.x;
  const float* a = A[p];
  const int64_t total = meta[p].m * meta[p].n, units = (total + 7) / 8;
  const bool vec = (reinterpret_cast<uintptr_t>(a) & 15u) == 0;
  SquareSum acc;
  for (int64_t u = (int64_t)blockIdx.y * kThreads + threadIdx.x; u < units; u += (int64_t)gridDim.y * kThreads) {
    float v[8];
    load_row8(a + 8 * u, total - 8 * u, vec, v);   // the problem is packed: rows do not matter here
    acc.add8(v);
  }
  const double t = block_sum_b(acc.value());
  if (threadIdx.x == 0) {
    st[p].res_hist[blockIdx.y] = t;
    if (p == 0 && blockIdx.y == 0) {
      sh->err = 0;
      for (int i = 0; i < 4; ++i) sh->running[i] = 0;
    }
  }
}

// The initial state of every problem, X_0 = A_p / ||A_p||_F as three planes, and P planes of A_p (for H).
// Grid (count, Y), units of 8 columns strided over the problem's blocks.
__global__ void b_scale_split_kernel(const float* const* __restrict__ A, const BMeta* __restrict__ meta,
                                     DevState* __restrict__ st, int P, int norm_blocks) {
  const int p = blockIdx.x;
  __shared__ double nrm_s;
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int i = 0; i < norm_blocks; ++i) t += st[p].res_hist[i];
    nrm_s = sqrt(t);
  }
  __syncthreads();
  const double nrm = nrm_s;
  const bool good = isfinite(nrm) && nrm > 0.0;
  const BMeta& mt = meta[p];
  if (blockIdx.y == 0 && threadIdx.x == 0) {
    DevState& s = st[p];
    s.normA = nrm;
    s.inv_sqrt_n = 1.0 / sqrt((double)mt.n);
    s.iters = 0;
    s.hist_len = 0;
    s.err_flags = 0;
    s.planes_next = P;
    s.sym_err = 0.0;
    s.upd_c1 = 1.5f;
    s.upd_c3 = -0.5f;
    for (int i = 0; i < 4; ++i) s.ring[i] = 0.0;
    s.status = good ? ST_RUNNING : ST_NONFINITE;
  }
  if (!good) return;
  const float* a = A[p];
  const float s = (float)nrm;
  const bool vec = (reinterpret_cast<uintptr_t>(a) & 15u) == 0 && mt.n % 4 == 0;
  const int n = (int)mt.n, c8 = (n + 7) / 8;
  const int64_t units = mt.m * c8;
  for (int64_t u = (int64_t)blockIdx.y * kThreads + threadIdx.x; u < units; u += (int64_t)gridDim.y * kThreads) {
    const int64_t r = u / c8;
    const int c = (int)(u - r * c8) * 8;
    float v[8], x[8];
    load_row8(a + r * n + c, n - c, vec, v);
#pragma unroll
    for (int j = 0; j < 8; ++j) x[j] = __fdiv_rn(v[j], s);
    split_store8(mt.xp[0] + r * mt.ldp + c, mt.xps, kStored, x);
    split_store8(mt.ap + r * mt.ldp + c, mt.xps, P, v);
  }
}

// U_p = the planes of its final iterate summed (exact). Grid (count, Y), units of 8 columns strided.
__global__ void b_u_kernel(const BMeta* __restrict__ meta, const DevState* __restrict__ st, float* const* __restrict__ U,
                           const BShared* sh) {
  const int p = blockIdx.x;
  if (sh->err || !finished_ok(st[p].status)) return;
  const BMeta& mt = meta[p];
  const uint16_t* X = mt.xp[st[p].iters & 1];
  float* u = U[p];
  const bool vec = (reinterpret_cast<uintptr_t>(u) & 15u) == 0 && mt.n % 4 == 0;
  const int n = (int)mt.n, c8 = (n + 7) / 8;
  const int64_t units = mt.m * c8;
  for (int64_t i = (int64_t)blockIdx.y * kThreads + threadIdx.x; i < units; i += (int64_t)gridDim.y * kThreads) {
    const int64_t r = i / c8;
    const int c = (int)(i - r * c8) * 8;
    float v[8];
    sum_row8(X + r * mt.ldp + c, mt.xps, v);
    store_row8(u + r * n + c, n - c, vec, v);
  }
}

// H_p = (C_p + C_p^T) / 2 by pairs of 32 x 32 tiles (bi <= bj) through shared memory. Grid (count, Y).
__global__ void b_h_kernel(const BMeta* __restrict__ meta, const DevState* __restrict__ st, float* const* __restrict__ H,
                           const BShared* sh) {
  const int p = blockIdx.x;
  if (sh->err || !finished_ok(st[p].status)) return;
  const BMeta& mt = meta[p];
  __shared__ float ta[32][33];
  __shared__ float tb[32][33];
  const int n = (int)mt.n, nt = (n + 31) / 32, npair = nt * (nt + 1) / 2;
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  float* h = H[p];
  for (int t = blockIdx.y; t < npair; t += gridDim.y) {
    int bj = (int)((sqrtf(8.0f * (float)t + 1.0f) - 1.0f) * 0.5f);
    while (bj > 0 && bj * (bj + 1) / 2 > t) --bj;
    while ((bj + 1) * (bj + 2) / 2 <= t) ++bj;
    const int bi = t - bj * (bj + 1) / 2, i0 = bi * 32, j0 = bj * 32;
    __syncthreads();
    for (int yy = ty; yy < 32; yy += kThreads / 32) {
      ta[yy][tx] = (i0 + yy < n && j0 + tx < n) ? mt.C[(int64_t)(i0 + yy) * n + j0 + tx] : 0.0f;
      tb[yy][tx] = (j0 + yy < n && i0 + tx < n) ? mt.C[(int64_t)(j0 + yy) * n + i0 + tx] : 0.0f;
    }
    __syncthreads();
    for (int yy = ty; yy < 32; yy += kThreads / 32) {
      if (i0 + yy < n && j0 + tx < n) h[(int64_t)(i0 + yy) * n + j0 + tx] = 0.5f * (ta[yy][tx] + tb[tx][yy]);
      if (bi < bj && j0 + yy < n && i0 + tx < n) h[(int64_t)(j0 + yy) * n + i0 + tx] = 0.5f * (tb[yy][tx] + ta[tx][yy]);
    }
  }
}

// Per-problem results: updates applied (negative, -1 - updates, when not converged;
// INT32_MIN after a device timeout) and the final residual.
__global__ void b_results_kernel(const DevState* __restrict__ st, const BShared* sh, int count, int32_t* iters_dev,
                                 double* resid_dev) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= count) return;
  const DevState& s = st[p];
  const int it = s.iters;
  int32_t code = s.status == ST_CONVERGED ? it : -1 - it;
  double r = (it < POLAR_HIST && it < s.hist_len) ? s.res_hist[it] : s.ring[it & 3];
  if (!finished_ok(s.status)) r = NAN;
  if (sh->err) {
    code = INT32_MIN;
    r = NAN;
  }
  iters_dev[p] = code;
  resid_dev[p] = r;
}

}  // namespace

struct BatchedPlan {
  int count = 0;
  int P = 3;
  int prec = POLAR_BF16X6;
  polar_options_t opt{};
  std::vector<int64_t> m, n;
  std::vector<void*> allocs;
  size_t ws_bytes = 0;
  BMeta* meta_d = nullptr;
  DevState* st_d = nullptr;
  BShared* sh_d = nullptr;
  const float** A_tab = nullptr;   // device tables of the caller's pointers (per run)
  float** U_tab = nullptr;
  float** H_tab = nullptr;
  void** host_tab = nullptr;       // pinned staging: A, U, H pointers, then tol
  // operand maps of the loop's products per parity of k, and of U^T A per problem and parity
  TcMapPair* gram_m[2] = {nullptr, nullptr};
  TcMapPair* upd_m[2] = {nullptr, nullptr};
  TcMapPair* h_m = nullptr;
  TcTile *gram_t = nullptr, *upd_t = nullptr, *h_t = nullptr;
  int n_gram = 0, n_upd = 0, n_h = 0;
  int64_t deepest = 0;             // most K of all tiles that one block takes in a product
  int sms = 0;
  OcTask* oc_tasks = nullptr;      // problems solved on one SM each (largest first)
  int n_oc = 0;
  cudaStream_t cap = nullptr;
  cudaGraph_t graph = nullptr;
  cudaGraphExec_t exec = nullptr;
  int32_t* iters_cap = nullptr;    // the graph writes results here; copied out per run
  double* resid_cap = nullptr;
  cudaEvent_t tab_ev = nullptr;    // the last upload of host_tab has been consumed
  int grid() const { return std::max(1, std::min(sms, std::max(std::max(n_gram, n_upd), n_h))); }
};

namespace {

polar_status_t b_alloc(BatchedPlan* b, size_t bytes, void** out) {
  if (b->opt.ws_limit && b->ws_bytes + bytes > b->opt.ws_limit) return POLAR_ENOMEM;
  void* p = nullptr;
  if (device_alloc(&p, bytes) != cudaSuccess) return POLAR_ENOMEM;
  b->allocs.push_back(p);
  b->ws_bytes += bytes;
  *out = p;
  return POLAR_OK;
}


// Tiles of a rows x cols product; tri: those that hold an entry on or above the diagonal.
int64_t tile_count(int64_t rows, int64_t cols, bool tri) {
  const int64_t tm = (rows + kTile - 1) / kTile, tn = (cols + kTile - 1) / kTile;
  return tri ? tn * (tn + 1) / 2 : tm * tn;
}

// Tile table: problems by decreasing work, each problem's tiles contiguous and column by column (neighbouring
// blocks of a wave share that problem's operand panels in L2).
void build_tiles(const std::vector<int>& order, const std::vector<int64_t>& rows, const std::vector<int64_t>& cols,
                 const std::vector<int64_t>& depth, bool tri, std::vector<TcTile>& out) {
  out.clear();
  for (int p : order) {
    const int64_t tm = (rows[p] + kTile - 1) / kTile, tn = (cols[p] + kTile - 1) / kTile;
    for (int64_t j = 0; j < tn; ++j)
      for (int64_t i = 0; i < (tri ? j + 1 : tm); ++i) out.push_back({p, (int32_t)i, (int32_t)j, (int32_t)depth[p]});
  }
}

// Most K of all tiles that one of `grid` blocks takes from a table.
int64_t deepest_block(const std::vector<TcTile>& t, int grid) {
  std::vector<int64_t> sum(grid, 0);
  for (size_t i = 0; i < t.size(); ++i) sum[i % grid] += t[i].K;
  return *std::max_element(sum.begin(), sum.end());
}

TcOperand opnd(const uint16_t* planes, int64_t rows, int64_t cols, int64_t ld, int64_t stride, int kmajor) {
  TcOperand o;
  o.planes = planes; o.rows = rows; o.cols = cols; o.ld = ld; o.plane_stride = stride; o.kmajor = kmajor;
  return o;
}

polar_status_t enqueue_all(BatchedPlan* b, cudaStream_t s) {
  const int count = b->count;
  StopRule rule;
  rule.tol = b->opt.tol;
  rule.stagnation = b->opt.stagnation;
  rule.stag_floor = b->opt.stag_floor;
  rule.switch_residual = b->opt.switch_residual;
  rule.max_iter = b->opt.max_iter;
  rule.sched = 0;   // batched plans have a fixed plane count
  rule.planes_fixed = b->P;
  rule.n_pre = b->opt.precondition ? precond_steps(b->opt.s_minus, b->opt.s0) : 0;
  rule.pre_a = 1.5 * sqrt(3.0) - b->opt.s_minus;
#define BK_(x) do { if ((x) != cudaSuccess) return POLAR_ECUDA; } while (0)
  // blocks per problem of the passes over A, U and H: about 8192 in all, so that a few large problems spread too, but
  // no more than the largest problem has work for (123 problems of 30 x 30: 174 us with 64 blocks each, 120 with one)
  int64_t units = 1;
  for (int p = 0; p < count; ++p) units = std::max(units, b->m[p] * ((b->n[p] + 7) / 8));
  const int most = std::max(8, std::min(kMaxSplit, 8192 / count));
  const int ys = (int)std::min<int64_t>(most, (units + kThreads - 1) / kThreads);
  b_norm_kernel<<<dim3(count, ys), kThreads, 0, s>>>(b->A_tab, b->meta_d, b->st_d, b->sh_d);
  BK_(cudaGetLastError());
  b_scale_split_kernel<<<dim3(count, ys), kThreads, 0, s>>>(b->A_tab, b->meta_d, b->st_d, b->P, ys);
  BK_(cudaGetLastError());
  // the small problems' whole loops, one SM each; the loop below skips them
  BK_(launch_onchip_ns(b->oc_tasks, b->n_oc, rule, &b->sh_d->tol, &b->sh_d->err, b->P, s));
  CoBatch c{};
  c.gram_t = b->gram_t; c.upd_t = b->upd_t; c.h_t = b->h_t;
  c.n_gram = b->n_gram; c.n_upd = b->n_upd; c.n_h = b->n_h;
  for (int i = 0; i < 2; ++i) {
    c.gram_m[i] = b->gram_m[i];
    c.upd_m[i] = b->upd_m[i];
  }
  c.h_m = b->h_m;
  c.meta = b->meta_d; c.st = b->st_d; c.sh = b->sh_d;
  c.count = count;
  c.P = b->P;
  c.rule = rule;
  update_coeffs(rule, 0, c.pre_c1, c.pre_c3);   // of the preconditioning steps, where there are any
  c.withhold = tc_withhold();
  // a block may wait for one that has all its tiles to do: about 14 ns per unit of K and tile, four times that
  c.wait_ns = 2000000000ull + 56ull * (uint64_t)b->deepest;
  BK_(launch_co_batch(c, b->grid(), s));
  b_u_kernel<<<dim3(count, ys), kThreads, 0, s>>>(b->meta_d, b->st_d, b->U_tab, b->sh_d);
  BK_(cudaGetLastError());
  b_h_kernel<<<dim3(count, ys), kThreads, 0, s>>>(b->meta_d, b->st_d, b->H_tab, b->sh_d);
  BK_(cudaGetLastError());
  b_results_kernel<<<(count + 127) / 128, 128, 0, s>>>(b->st_d, b->sh_d, count, b->iters_cap, b->resid_cap);
  BK_(cudaGetLastError());
#undef BK_
  return POLAR_OK;
}

}  // namespace

polar_status_t batched_create(BatchedPlan** out, int count, const int64_t* m, const int64_t* n,
                              const polar_options_t& opt, int prec) {
  BatchedPlan* b = new (std::nothrow) BatchedPlan();
  if (!b) return POLAR_ENOMEM;
  b->count = count;
  b->opt = opt;
  b->prec = prec;
  b->P = product_planes(prec);
  if (!device_is_sm103(&b->sms)) { delete b; return POLAR_ECUDA; }
  b->m.assign(m, m + count);
  b->n.assign(n, n + count);
  // k-blocks of 32 per promoted slice: the first matching tuning entry's, else the library's (entries' tile widths
  // are accepted and have no effect: every tile is 128 wide)
  std::vector<int> slice_of(count, tc_default_slice(b->P));
  for (int p = 0; p < count && opt.tune; ++p) {
    const double aspect = (double)m[p] / (double)n[p];
    for (int e = 0; e < opt.n_tune; ++e) {
      const polar_tune_entry_t& te = opt.tune[e];
      if (n[p] < te.n_lo || n[p] > te.n_hi || aspect < te.aspect_lo || aspect > te.aspect_hi) continue;
      if (te.slice_stages >= 1 && te.slice_stages <= 8) slice_of[p] = te.slice_stages;
      break;
    }
  }
  polar_status_t r = POLAR_OK;
  void* v = nullptr;
  auto fail = [&](polar_status_t e) {
    batched_destroy(b);
    return e;
  };
  // per-problem layout, packed into one allocation per buffer kind
  std::vector<BMeta> meta(count);
  size_t x_bytes = 0, g_bytes = 0, a_bytes = 0, c_bytes = 0;
  std::vector<int> ntg(count, 0);
  for (int p = 0; p < count; ++p) {
    BMeta& mt = meta[p];
    mt.m = m[p];
    mt.n = n[p];
    mt.ldp = up(n[p], 64);
    mt.xps = up(m[p] * mt.ldp, 64);
    mt.gps = up(n[p] * mt.ldp, 64);
    x_bytes += (size_t)kStored * mt.xps * 2;
    g_bytes += (size_t)kStored * mt.gps * 2;
    a_bytes += (size_t)b->P * mt.xps * 2;
    c_bytes += (size_t)up(n[p] * n[p], 64) * 4;
  }
  std::vector<int> order(count);
  std::iota(order.begin(), order.end(), 0);
  std::stable_sort(order.begin(), order.end(),
                   [&](int x, int y) { return (double)m[x] * n[x] * n[x] > (double)m[y] * n[y] * n[y]; });
  // problems that fit one SM run their loop there; the rest go through the tiles, which all problems share for H
  std::vector<int> order_tc, order_oc;
  for (int p : order) (opt.small_onchip != 0 && onchip_fits(m[p], n[p]) ? order_oc : order_tc).push_back(p);
  size_t part_count = 0;
  for (int p : order_tc) {
    ntg[p] = (int)tile_count(n[p], n[p], true);
    part_count += (size_t)ntg[p] * kBatchEpiWarps;
  }

  uint8_t *xb[2], *gb, *ab, *cb;
  for (int i = 0; i < 2; ++i) {
    if ((r = b_alloc(b, x_bytes, &v)) != POLAR_OK) return fail(r);
    xb[i] = (uint8_t*)v;
    if (cudaMemset(v, 0, x_bytes) != cudaSuccess) return fail(POLAR_ECUDA);
  }
  if ((r = b_alloc(b, g_bytes, &v)) != POLAR_OK) return fail(r);
  gb = (uint8_t*)v;
  if (cudaMemset(v, 0, g_bytes) != cudaSuccess) return fail(POLAR_ECUDA);
  if ((r = b_alloc(b, a_bytes, &v)) != POLAR_OK) return fail(r);
  ab = (uint8_t*)v;
  if (cudaMemset(v, 0, a_bytes) != cudaSuccess) return fail(POLAR_ECUDA);
  if ((r = b_alloc(b, c_bytes, &v)) != POLAR_OK) return fail(r);
  cb = (uint8_t*)v;
  if ((r = b_alloc(b, std::max<size_t>(part_count, 1) * 8, &v)) != POLAR_OK) return fail(r);
  double* partials = (double*)v;
  size_t xo = 0, go = 0, ao = 0, co = 0, po = 0;
  for (int p = 0; p < count; ++p) {
    BMeta& mt = meta[p];
    mt.xp[0] = (uint16_t*)(xb[0] + xo);
    mt.xp[1] = (uint16_t*)(xb[1] + xo);
    mt.gp = (uint16_t*)(gb + go);
    mt.ap = (uint16_t*)(ab + ao);
    mt.C = (float*)(cb + co);
    mt.partials = partials + po;
    mt.ntiles_gram = ntg[p];
    mt.slice = slice_of[p];
    xo += (size_t)kStored * mt.xps * 2;
    go += (size_t)kStored * mt.gps * 2;
    ao += (size_t)b->P * mt.xps * 2;
    co += (size_t)up(mt.n * mt.n, 64) * 4;
    po += (size_t)ntg[p] * kBatchEpiWarps;
  }
  if ((r = b_alloc(b, sizeof(BMeta) * count, &v)) != POLAR_OK) return fail(r);
  b->meta_d = (BMeta*)v;
  if (cudaMemcpy(b->meta_d, meta.data(), sizeof(BMeta) * count, cudaMemcpyHostToDevice) != cudaSuccess)
    return fail(POLAR_ECUDA);
  if ((r = b_alloc(b, sizeof(DevState) * count, &v)) != POLAR_OK) return fail(r);
  b->st_d = (DevState*)v;
  if (cudaMemset(v, 0, sizeof(DevState) * count) != cudaSuccess) return fail(POLAR_ECUDA);
  if (!order_oc.empty()) {
    std::vector<OcTask> tasks;
    for (int p : order_oc) {
      OcTask t;
      t.m = meta[p].m; t.n = meta[p].n; t.ldp = meta[p].ldp; t.xps = meta[p].xps;
      t.x0 = meta[p].xp[0];
      t.xp[0] = meta[p].xp[0];
      t.xp[1] = meta[p].xp[1];
      t.st = b->st_d + p;
      tasks.push_back(t);
    }
    if ((r = b_alloc(b, sizeof(OcTask) * tasks.size(), &v)) != POLAR_OK) return fail(r);
    b->oc_tasks = (OcTask*)v;
    b->n_oc = (int)tasks.size();
    if (cudaMemcpy(v, tasks.data(), sizeof(OcTask) * tasks.size(), cudaMemcpyHostToDevice) != cudaSuccess)
      return fail(POLAR_ECUDA);
  }
  if ((r = b_alloc(b, sizeof(BShared), &v)) != POLAR_OK) return fail(r);
  b->sh_d = (BShared*)v;
  if (cudaMemset(v, 0, sizeof(BShared)) != cudaSuccess) return fail(POLAR_ECUDA);
  if ((r = b_alloc(b, sizeof(void*) * 3 * count, &v)) != POLAR_OK) return fail(r);
  b->A_tab = (const float**)v;
  b->U_tab = (float**)v + count;
  b->H_tab = (float**)v + 2 * count;
  if (cudaMallocHost((void**)&b->host_tab, sizeof(void*) * 3 * count + 16) != cudaSuccess) return fail(POLAR_ENOMEM);
  if ((r = b_alloc(b, sizeof(int32_t) * count, &v)) != POLAR_OK) return fail(r);
  b->iters_cap = (int32_t*)v;
  if ((r = b_alloc(b, sizeof(double) * count, &v)) != POLAR_OK) return fail(r);
  b->resid_cap = (double*)v;

  // operand maps
  auto put = [&](const void* src, size_t bytes, void** dst) -> polar_status_t {
    polar_status_t rr = b_alloc(b, std::max<size_t>(bytes, 16), dst);
    if (rr != POLAR_OK) return rr;
    if (bytes && cudaMemcpy(*dst, src, bytes, cudaMemcpyHostToDevice) != cudaSuccess) return POLAR_ECUDA;
    return POLAR_OK;
  };
  std::vector<TcMapPair> hm(2 * (size_t)count);
  for (int par = 0; par < 2; ++par) {
    std::vector<TcMapPair> gm(count), um(count);
    for (int p = 0; p < count; ++p) {
      const BMeta& mt = meta[p];
      const TcOperand x = opnd(mt.xp[par], mt.m, mt.n, mt.ldp, mt.xps, 0);
      const TcOperand g = opnd(mt.gp, mt.n, mt.n, mt.ldp, mt.gps, 0);
      const TcOperand a = opnd(mt.ap, mt.m, mt.n, mt.ldp, mt.xps, 0);
      TcMapPair& h = hm[2 * (size_t)p + par];
      if (!tc_make_map(gm[p].a, x, b->P, true, 0) || !tc_make_map(gm[p].b, g, b->P, false, kTile) ||
          !tc_make_map(um[p].a, x, b->P, false, kTile) || !tc_make_map(um[p].b, g, b->P, true, 0) ||
          !tc_make_map(h.a, x, b->P, true, 0) || !tc_make_map(h.b, a, b->P, true, 0))
        return fail(POLAR_ECUDA);
    }
    if ((r = put(gm.data(), sizeof(TcMapPair) * count, &v)) != POLAR_OK) return fail(r);
    b->gram_m[par] = (TcMapPair*)v;
    if ((r = put(um.data(), sizeof(TcMapPair) * count, &v)) != POLAR_OK) return fail(r);
    b->upd_m[par] = (TcMapPair*)v;
  }
  if ((r = put(hm.data(), sizeof(TcMapPair) * hm.size(), &v)) != POLAR_OK) return fail(r);
  b->h_m = (TcMapPair*)v;
  std::vector<TcTile> gram_t, upd_t, h_t;
  build_tiles(order_tc, b->n, b->n, b->m, true, gram_t);
  build_tiles(order_tc, b->m, b->n, b->n, false, upd_t);
  build_tiles(order, b->n, b->n, b->m, false, h_t);
  if ((r = put(gram_t.data(), sizeof(TcTile) * gram_t.size(), &v)) != POLAR_OK) return fail(r);
  b->gram_t = (TcTile*)v;
  b->n_gram = (int)gram_t.size();
  if ((r = put(upd_t.data(), sizeof(TcTile) * upd_t.size(), &v)) != POLAR_OK) return fail(r);
  b->upd_t = (TcTile*)v;
  b->n_upd = (int)upd_t.size();
  if ((r = put(h_t.data(), sizeof(TcTile) * h_t.size(), &v)) != POLAR_OK) return fail(r);
  b->h_t = (TcTile*)v;
  b->n_h = (int)h_t.size();
  for (const auto* t : {&gram_t, &upd_t}) b->deepest = std::max(b->deepest, deepest_block(*t, b->grid()));

  // the buffers are cleared and filled on the default stream, which a run's stream need not wait for
  if (cudaStreamSynchronize(cudaStreamLegacy) != cudaSuccess) return fail(POLAR_ECUDA);

  // capture the whole sequence once; each run uploads its pointer tables and replays it
  if (cudaStreamCreateWithFlags(&b->cap, cudaStreamNonBlocking) != cudaSuccess) return fail(POLAR_ECUDA);
  if (cudaEventCreateWithFlags(&b->tab_ev, cudaEventDisableTiming) != cudaSuccess) return fail(POLAR_ECUDA);
  if (cudaStreamBeginCapture(b->cap, cudaStreamCaptureModeRelaxed) != cudaSuccess) return fail(POLAR_ECUDA);
  polar_status_t er = enqueue_all(b, b->cap);
  cudaGraph_t gph = nullptr;
  cudaError_t ce = cudaStreamEndCapture(b->cap, &gph);
  if (er != POLAR_OK || ce != cudaSuccess || !gph) {
    if (gph) cudaGraphDestroy(gph);
    cudaGetLastError();
    b->graph = nullptr;  // the run enqueues the sequence directly instead
  } else {
    b->graph = gph;
    if (cudaGraphInstantiate(&b->exec, gph, 0) != cudaSuccess) {
      cudaGetLastError();
      b->exec = nullptr;
    }
  }
  *out = b;
  return POLAR_OK;
}

polar_status_t batched_run(BatchedPlan* b, const float* const* A, float* const* U, float* const* H, double tol,
                           int32_t* iters_dev, double* resid_dev, cudaStream_t s) {
  const int count = b->count;
  // the previous run's upload from the pinned table must have been consumed
  if (cudaEventSynchronize(b->tab_ev) != cudaSuccess) return POLAR_ECUDA;
  for (int p = 0; p < count; ++p) {
    b->host_tab[p] = (void*)A[p];
    b->host_tab[count + p] = (void*)U[p];
    b->host_tab[2 * count + p] = (void*)H[p];
  }
  if (cudaMemcpyAsync(b->A_tab, b->host_tab, sizeof(void*) * 3 * count, cudaMemcpyHostToDevice, s) != cudaSuccess)
    return POLAR_ECUDA;
  // tol is read by the finalize kernel from the shared block (0: the plan's tolerance)
  double* tol_pinned = reinterpret_cast<double*>(b->host_tab + 3 * count);
  *tol_pinned = tol > 0 ? tol : 0.0;
  if (cudaMemcpyAsync(&b->sh_d->tol, tol_pinned, sizeof(double), cudaMemcpyHostToDevice, s) != cudaSuccess)
    return POLAR_ECUDA;
  if (cudaEventRecord(b->tab_ev, s) != cudaSuccess) return POLAR_ECUDA;
  if (b->exec) {
    if (cudaGraphLaunch(b->exec, s) != cudaSuccess) return POLAR_ECUDA;
  } else {
    polar_status_t r = enqueue_all(b, s);
    if (r != POLAR_OK) return r;
  }
  if (iters_dev &&
      cudaMemcpyAsync(iters_dev, b->iters_cap, sizeof(int32_t) * count, cudaMemcpyDeviceToDevice, s) != cudaSuccess)
    return POLAR_ECUDA;
  if (resid_dev &&
      cudaMemcpyAsync(resid_dev, b->resid_cap, sizeof(double) * count, cudaMemcpyDeviceToDevice, s) != cudaSuccess)
    return POLAR_ECUDA;
  return POLAR_OK;
}

void batched_destroy(BatchedPlan* b) {
  if (!b) return;
  cudaDeviceSynchronize();
  if (b->exec) cudaGraphExecDestroy(b->exec);
  if (b->graph) cudaGraphDestroy(b->graph);
  if (b->cap) cudaStreamDestroy(b->cap);
  if (b->tab_ev) cudaEventDestroy(b->tab_ev);
  for (void* p : b->allocs) cudaFree(p);
  if (b->host_tab) cudaFreeHost(b->host_tab);
  delete b;
}

size_t batched_workspace_bytes(const BatchedPlan* b) { return b ? b->ws_bytes : 0; }

}  // namespace polar
