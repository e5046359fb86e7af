// One polar solve in one cooperative launch (Sec. III.D, Eq. NewtonSchulz, Algorithm 1), for matrices whose
// products are a few waves of 128 x 64 or 128 x 128 tiles; the pieces are in coop_kernel.cuh.
//
// Where the products have so few 128 x 64 tiles that most SMs would idle, clusters of four blocks share tiles
// along K (co_epilogue_split).
//
//   ||A||_F | X_0 = A / ||A||_F and the planes of A | per step: Gram | update | ... | U^T A | U, H
//
// with a grid barrier at every bar. The update of step k runs before its stop test is known (each block
// evaluates the test in a warp of its own, from the same partials in the same order, while the products run): when the test
// stops the iteration at X_k, the update has written the other buffer and is ignored.
#include <math.h>

#include <algorithm>
#include <mutex>
#include <new>

#include "coop_kernel.cuh"

namespace polar {
namespace {

struct CoSolve {
  CUtensorMap xmn[2], xk[2], gmn, gk, amn;   // X_k as MN-major and K-major operand, G, mirrored G, A
  const float* A;
  int64_t lda;
  float* U;
  int64_t ldu;
  float* H;
  int64_t ldh;
  uint16_t* xp[2];
  uint16_t* gp;
  uint16_t* ap;
  float* C;
  int64_t ldc, ldp, xps, gps;
  double* partials;                          // one per block, two per block at the end
  double* part2;                             // residual sums, EPI_WARPS per block
  DevState* st;
  int m, n;
  double v_tol, stag2, v_floor;              // the stop rule on squares: n tol^2, stagnation^2, n stag_floor^2
  int n_pre, max_iter;
  float pre_c1, pre_c3;                      // update coefficients of the first n_pre steps
  double inv_sqrt_n;
  int withhold;
  int sg, su, sh;                            // split chains: blocks per tile of the Gram, the update and U^T A
};

// The stop rule of step k on v = ||G - I||_F^2 = n r^2 against squared thresholds: r <= tol is
// v <= n tol^2 and r > s r_{k-2} is v > s^2 v_{k-2}.
__device__ __forceinline__ int co_stop_status(const CoSolve& p, int k, double v, double v_km2) {
  const bool testing = k >= p.n_pre;
  if (!isfinite(v)) return ST_NONFINITE;
  if (testing && v <= p.v_tol) return ST_CONVERGED;
  if (testing && k >= p.n_pre + 2 && v > p.stag2 * v_km2 && v < p.v_floor) return ST_NOT_CONVERGED;
  if (k >= p.max_iter) return ST_NOT_CONVERGED;
  return ST_RUNNING;
}

template <int TN, bool SPLIT>
__device__ __forceinline__ void co_solve(const CoSolve& p, uint8_t* co_raw) {
  CoCtx x = co_setup<TN, CO_P, SPLIT>(co_raw, &p.st->bar);
  const int m = p.m, n = p.n, tid = threadIdx.x, nthr = CO_THREADS;
  const int gtid = blockIdx.x * nthr + tid, gthr = gridDim.x * nthr;
  const bool vec_a = (reinterpret_cast<uintptr_t>(p.A) & 15u) == 0 && p.lda % 4 == 0;
  const bool vec_u = (reinterpret_cast<uintptr_t>(p.U) & 15u) == 0 && p.ldu % 4 == 0;
  const int c8n = (n + 7) / 8;
  DevState* st = p.st;
  CoPipe pipe;
  bool run = true;
  // ---- ||A||_F, float64 sums in a fixed order
  {
    SquareSum acc;
    for (int u = gtid; u < m * c8n; u += gthr) {
      const int r = u / c8n, c = (u - r * c8n) * 8;
      float v[8];
      load_row8(p.A + (int64_t)r * p.lda + c, n - c, vec_a, v);
      acc.add8(v);
    }
    const double t = co_block_sum(x, acc.value());
    if (tid == 0) p.partials[blockIdx.x] = t;
    run = co_grid_sync(x);
  }
  if (run) {
    const double nrm = sqrt(co_warp_sum(p.partials, gridDim.x, 1, x.lane));
    const bool good = isfinite(nrm) && nrm > 0.0;
    if (gtid == 0) {
      st->normA = nrm;
      st->inv_sqrt_n = p.inv_sqrt_n;
      st->iters = 0;
      st->hist_len = 0;
      st->err_flags = 0;
      st->planes_next = CO_P;
      st->fp8_on = 0;
      st->sym_err = 0.0;
      st->status = good ? ST_RUNNING : ST_NONFINITE;
    }
    run = good;            // the same in every block
    if (run) {
      // ---- X_0 = A / ||A||_F and A as planes; columns from n to the next multiple of 8 are zeros
      const float s = (float)nrm;
      for (int u = gtid; u < m * c8n; u += gthr) {
        const int r = u / c8n, c = (u - r * c8n) * 8;
        float v[8], y[8];
        load_row8(p.A + (int64_t)r * p.lda + c, n - c, vec_a, v);
#pragma unroll
        for (int j = 0; j < 8; ++j) y[j] = __fdiv_rn(v[j], s);
        const int64_t o = (int64_t)r * p.ldp + c;
        store_planes8(p.xp[0] + o, p.xps, 3, y);
        store_planes8(p.ap + o, p.xps, 3, v);
      }
      run = co_grid_sync(x);
    }
  }
  // ---- the iteration
  const CoTiles tg = co_tiles<TN>(n, n, true), tu = co_tiles<TN>(m, n, false);
  double v_km1 = 0.0, v_km2 = 0.0;   // the control warp's last two residual sums
  int it = 0, status = ST_TIMEOUT;
  for (int k = 0; run; ++k) {
    const int b = k & 1;
    // Gram of X_k: the upper triangle's tiles, and this block's part of ||G - I||_F^2
    {
      CoEpi e{};
      e.M = n; e.N = n;
      e.out = p.gp; e.ldo = p.ldp; e.os = p.gps;
      e.part = p.part2;
      co_product<TN, SPLIT, true, false, TC_EPI_GRAM>(x, pipe, &p.xmn[b], &p.xmn[b], nullptr, tg, m, e, p.sg,
                                                      p.withhold);
    }
    run = co_grid_sync(x);
    if (!run) break;
    // the update, and beside it the stop test of X_k and its record
    if (k < p.max_iter) {
      CoEpi e{};
      e.M = m; e.N = n;
      e.x = p.xp[b]; e.ldx = p.ldp; e.xs = p.xps;
      e.out = p.xp[b ^ 1]; e.ldo = p.ldp; e.os = p.xps;
      e.c1 = k < p.n_pre ? p.pre_c1 : 1.5f;
      e.c3 = k < p.n_pre ? p.pre_c3 : -0.5f;
      co_product<TN, SPLIT, false, true, TC_EPI_NS>(x, pipe, &p.xk[b], &p.gmn, &p.gk, tu, n, e, p.su, p.withhold);
    }
    if (x.warp == CO_CTL_WARP) {
      const double v = co_warp_sum(p.part2, gridDim.x * EPI_WARPS, 1, x.lane);
      const int s = co_stop_status(p, k, v, v_km2);
      v_km2 = v_km1;
      v_km1 = v;
      if (x.lane == 0) {
        x.ctl->status = s;
        if (blockIdx.x == 0) {
          st->res_hist[k] = sqrt(v) * p.inv_sqrt_n;   // k <= max_iter < POLAR_HIST
          st->planes_hist[k] = (unsigned char)CO_P;
          st->hist_len = k + 1;
          st->iters = k;
          st->status = s;
        }
      }
    }
    run = co_grid_sync(x);
    if (!run) break;
    status = *reinterpret_cast<volatile int*>(&x.ctl->status);
    it = k;
    if (status != ST_RUNNING) break;
  }
  // ---- C = U^T A, then U and H = (C + C^T) / 2
  if (run && (status == ST_CONVERGED || status == ST_NOT_CONVERGED)) {
    const CoTiles th = co_tiles<TN>(n, n, false);
    {
      CoEpi e{};
      e.M = n; e.N = n;
      e.C = p.C; e.ldc = p.ldc;
      co_product<TN, SPLIT, true, false, TC_EPI_STORE>(x, pipe, &p.xmn[it & 1], &p.amn, nullptr, th, m, e, p.sh,
                                                       p.withhold);
    }
    run = co_grid_sync(x);
    if (run) {
      const uint16_t* X = p.xp[it & 1];
      for (int u = gtid; u < m * c8n; u += gthr) {
        const int r = u / c8n, c = (u - r * c8n) * 8;
        float v[8];
        sum_planes8(load_planes8(X + (int64_t)r * p.ldp + c, p.xps, true), v);
        store_row8(p.U + (int64_t)r * p.ldu + c, n - c, vec_u, v);
      }
      // H by pairs of 32 x 32 tiles (bi <= bj) through shared memory (the stages are idle)
      float* ta = reinterpret_cast<float*>(x.smem);
      float* tb = ta + 32 * 33;
      const int nt = (n + 31) / 32, npair = nt * (nt + 1) / 2;
      double skew = 0.0, full = 0.0;
      for (int t = blockIdx.x; t < npair; t += gridDim.x) {
        int bj = (int)((sqrtf(8.0f * (float)t + 1.0f) - 1.0f) * 0.5f);
        while (bj > 0 && bj * (bj + 1) / 2 > t) --bj;
        while ((bj + 1) * (bj + 2) / 2 <= t) ++bj;
        const int bi = t - bj * (bj + 1) / 2, i0 = bi * 32, j0 = bj * 32;
        __syncthreads();
        for (int u = tid; u < 1024; u += nthr) {
          const int yy = u >> 5, xx = u & 31;
          ta[yy * 33 + xx] = (i0 + yy < n && j0 + xx < n) ? __ldcg(p.C + (int64_t)(i0 + yy) * p.ldc + j0 + xx) : 0.0f;
          tb[yy * 33 + xx] = (j0 + yy < n && i0 + xx < n) ? __ldcg(p.C + (int64_t)(j0 + yy) * p.ldc + i0 + xx) : 0.0f;
        }
        __syncthreads();
        for (int u = tid; u < 1024; u += nthr) {
          const int yy = u >> 5, xx = u & 31;
          if (i0 + yy < n && j0 + xx < n) {   // C(i, j) and C(j, i) of the upper tile's entry
            const float c = ta[yy * 33 + xx], ct = tb[xx * 33 + yy];
            p.H[(int64_t)(i0 + yy) * p.ldh + j0 + xx] = 0.5f * (c + ct);
            const double d = 0.5 * ((double)c - (double)ct), w = bi < bj ? 2.0 : 1.0;
            skew = fma(w * d, d, skew);
            full = fma((double)c, (double)c, full);
            if (bi < bj) full = fma((double)ct, (double)ct, full);
          }
          if (bi < bj && j0 + yy < n && i0 + xx < n)
            p.H[(int64_t)(j0 + yy) * p.ldh + i0 + xx] = 0.5f * (tb[yy * 33 + xx] + ta[xx * 33 + yy]);
        }
      }
      const double s1 = co_block_sum(x, skew);
      const double s2 = co_block_sum(x, full);
      if (tid == 0) {
        p.partials[2 * blockIdx.x] = s1;
        p.partials[2 * blockIdx.x + 1] = s2;
      }
      run = co_grid_sync(x);
      if (run && blockIdx.x == 0 && x.warp == 0) {
        const double a = co_warp_sum(p.partials, gridDim.x, 2, x.lane);
        const double c = co_warp_sum(p.partials + 1, gridDim.x, 2, x.lane);
        if (x.lane == 0) st->sym_err = c > 0.0 ? sqrt(a / c) : 0.0;
      }
    }
  }
  co_teardown<TN, SPLIT>(x, st);
}

template <int TN>
__global__ void __launch_bounds__(CO_THREADS, 1) co_solve_kernel(const __grid_constant__ CoSolve p) {
  extern __shared__ uint8_t co_raw[];
  co_solve<TN, false>(p, co_raw);
}

// Clusters whose blocks share tiles along K: products with few 128 x 64 tiles.
__global__ void __cluster_dims__(CO_CLUSTER, 1, 1) __launch_bounds__(CO_THREADS, 1)
    co_solve_split_kernel(const __grid_constant__ CoSolve p) {
  extern __shared__ uint8_t co_raw[];
  co_solve<64, true>(p, co_raw);
}

template <int TN>
cudaError_t co_prepare() {
  return cudaFuncSetAttribute(co_solve_kernel<TN>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)co_smem<TN>());
}

cudaError_t co_launch_split(const CoSolve& p, int grid, cudaStream_t s) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid, 1, 1);
  cfg.blockDim = dim3(CO_THREADS, 1, 1);
  cfg.dynamicSmemBytes = co_smem<64, CO_P, true>();
  cfg.stream = s;
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeCooperative;
  attr.val.cooperative = 1;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  void* args[] = {const_cast<CoSolve*>(&p)};
  return cudaLaunchKernelExC(&cfg, reinterpret_cast<const void*>(co_solve_split_kernel), args);
}

// Clusters of the split form that can be resident at once; 0 when it cannot run. Asked once per device.
int co_split_clusters_now(int sms) {
  const int smem = (int)co_smem<64, CO_P, true>();
  int n = 0;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(sms / CO_CLUSTER * CO_CLUSTER), 1, 1);
  cfg.blockDim = dim3(CO_THREADS, 1, 1);
  cfg.dynamicSmemBytes = (size_t)smem;
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeClusterDimension;
  attr.val.clusterDim.x = CO_CLUSTER;
  attr.val.clusterDim.y = 1;
  attr.val.clusterDim.z = 1;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  if (cudaFuncSetAttribute(co_solve_split_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) != cudaSuccess ||
      cudaOccupancyMaxActiveClusters(&n, reinterpret_cast<const void*>(co_solve_split_kernel), &cfg) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return n;
}

int co_split_clusters(int sms) {
  static std::mutex mu;
  static int known[64];   // clusters + 1
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
  std::lock_guard<std::mutex> lk(mu);
  if (!known[dev]) known[dev] = co_split_clusters_now(sms) + 1;
  return known[dev] - 1;
}

template <int TN>
cudaError_t co_launch(const CoSolve& p, int grid, cudaStream_t s) {
  void* args[] = {const_cast<CoSolve*>(&p)};
  return cudaLaunchCooperativeKernel(reinterpret_cast<const void*>(co_solve_kernel<TN>), dim3((unsigned)grid),
                                     dim3(CO_THREADS), args, co_smem<TN>(), s);
}

}  // namespace

struct CoopSolve {
  CoSolve p;
  int tn, grid;
  bool split;
};

// Cycles of a chain's products with tiles of one width: whole waves, a k-block of 32 costing about 750 cycles
// with 64-wide tiles and 870 with 128-wide ones (measured inside the solve; the MMAs alone take 494 and 786),
// a tile's output step about 4000 and 7000. Waves: the most of any product.
template <int TN>
static double co_cost(const CoopProduct* p, int count, int sms, int64_t* waves) {
  double c = 0.0;
  *waves = 0;
  for (int i = 0; i < count; ++i) {
    const int64_t w = ((int64_t)co_tiles<TN>(p[i].M, p[i].N, p[i].tri).ntiles + sms - 1) / sms;
    c += (double)w * ((double)((p[i].K + BK - 1) / BK) * (TN == 64 ? 750.0 : 870.0) + (TN == 64 ? 4000.0 : 7000.0));
    *waves = std::max(*waves, w);
  }
  return c;
}

// One launch against separate ones, per step at kappa 100: 512^2 23 against 84 us, 1024^2 36 against 111, 2048^2
// 113 against 174, 3072^2 326 against 445, 8192 x 2048 (7 waves of 128-wide tiles) 415 against 563, 4096^2 (7)
// 798 against 796; 8192^2 (27 waves) 6782 against 5600, where wider tiles read less from L2. So the line lies at
// eight waves.
CoopForm coop_form(const CoopProduct* p, int count, int sms) {
  int64_t w64, w128;
  const double c64 = co_cost<64>(p, count, sms, &w64), c128 = co_cost<128>(p, count, sms, &w128);
  CoopForm f;
  if (w128 > 8) return f;
  // few tiles: share each between blocks along K, where that shortens a step by a tenth
  f.split = coop_split_plan(p, count, sms, f.S, &f.blocks);
  if (!f.split) {
    f.S[0] = f.S[1] = 1;
    f.blocks = 0;
  }
  f.tn = f.split || c64 <= c128 ? 64 : 128;
  return f;
}

// Blocks per 128 x 64 tile of one product on `blocks` blocks (1, 2 or 4), and its cycles (co_cost's measure). A
// split tile's exchange costs a little more than its smaller output step saves; k-blocks cost a little more than
// in the other form, whose stages hold two.
static int co_split_of(const CoopProduct& q, int blocks, double* cycles) {
  const int64_t tiles = co_tiles<64>(q.M, q.N, q.tri).ntiles;
  int best = 1;
  *cycles = (double)((tiles + blocks - 1) / blocks) * ((double)((q.K + 31) / 32) * 850.0 + 4000.0);
  for (int S = 2; S <= CO_CLUSTER; S *= 2) {
    if (tiles * S > blocks) break;
    const int64_t kc = ((q.K + S - 1) / S + 63) / 64 * 64;
    const double c = (double)((std::min(kc, q.K) + 31) / 32) * 800.0 + 5000.0;
    if (c < *cycles) {
      *cycles = c;
      best = S;
    }
  }
  return best;
}

bool coop_split_plan(const CoopProduct* p, int count, int sms, int* S, int* blocks, double* cycles) {
  int64_t waves;
  const double whole = co_cost<64>(p, count, sms, &waves), wide = co_cost<128>(p, count, sms, &waves);
  if (cycles) *cycles = whole;
  *blocks = CO_CLUSTER * co_split_clusters(sms);
  if (*blocks <= 0) return false;
  double split = 0.0, c;
  int64_t want = CO_CLUSTER;
  for (int i = 0; i < count; ++i) {
    S[i] = co_split_of(p[i], *blocks, &c);
    split += c;
    want = std::max<int64_t>(want, (int64_t)co_tiles<64>(p[i].M, p[i].N, p[i].tri).ntiles * S[i]);
    want = std::max<int64_t>(want, (p[i].M * p[i].N + 8191) / 8192);
  }
  *blocks = (int)std::min<int64_t>(*blocks, (want + CO_CLUSTER - 1) / CO_CLUSTER * CO_CLUSTER);
  if (split >= 0.9 * std::min(whole, wide)) return false;
  if (cycles) *cycles = split;
  return true;
}

CoopSolve* coop_solve_create(const CoopBuffers& b, int64_t m, int64_t n, int sms) {
  const CoopProduct prod[2] = {{n, n, m, true}, {m, n, n, false}};
  const CoopForm f = coop_form(prod, 2, sms);
  if (!f.tn) return nullptr;
  CoopSolve* c = new (std::nothrow) CoopSolve();
  if (!c) return nullptr;
  c->tn = f.tn;
  c->split = f.split && f.blocks <= b.nparts / 2;
  c->p.sg = c->p.su = c->p.sh = 1;
  if (c->split) {
    double ch;
    c->p.sg = f.S[0];
    c->p.su = f.S[1];
    c->p.sh = co_split_of({n, n, m, false}, f.blocks, &ch);
  }
  // enough blocks for the larger product's tiles, and for the passes over A
  const int64_t tiles = c->tn == 64 ? co_tiles<64>(m, n, false).ntiles : co_tiles<128>(m, n, false).ntiles;
  int64_t grid = std::max<int64_t>(tiles, (m * n + 8191) / 8192);
  grid = std::min<int64_t>(grid, std::min<int64_t>(sms, b.nparts / 2));
  if (c->split) grid = f.blocks;
  if (!c->split && tiles <= 2) grid = 1;   // a second tile takes less time than two grid barriers
  c->grid = (int)std::max<int64_t>(grid, 1);
  if (8 * c->grid > b.nparts && (size_t)8 * c->grid * 8 > (size_t)n * b.ldc * 4) {
    c->split = false;   // no room for a sum per block and warp
    c->p.sg = c->p.su = c->p.sh = 1;
    c->grid = std::max(1, b.nparts / 8);
  }
  CoSolve& p = c->p;
  TcOperand x[2], g, a;
  for (int i = 0; i < 2; ++i) {
    x[i].planes = b.xp[i]; x[i].rows = m; x[i].cols = n; x[i].ld = b.ldp; x[i].plane_stride = b.xps;
    p.xp[i] = b.xp[i];
  }
  g = x[0];
  g.planes = b.gp; g.rows = n; g.plane_stride = b.gps;
  a = x[0];
  a.planes = b.ap;
  bool ok = tc_make_map(&p.gmn, g, CO_P, true, 0) && tc_make_map(&p.gk, g, CO_P, false, c->tn) &&
            tc_make_map(&p.amn, a, CO_P, true, 0);
  for (int i = 0; i < 2; ++i)
    ok = ok && tc_make_map(&p.xmn[i], x[i], CO_P, true, 0) && tc_make_map(&p.xk[i], x[i], CO_P, false, BM);
  ok = ok && (c->tn == 64 ? co_prepare<64>() : co_prepare<128>()) == cudaSuccess;
  if (!ok) {
    cudaGetLastError();
    delete c;
    return nullptr;
  }
  p.gp = b.gp; p.ap = b.ap; p.C = b.C; p.ldc = b.ldc; p.ldp = b.ldp; p.xps = b.xps; p.gps = b.gps;
  p.partials = b.partials; p.st = b.st;
  // the residual sums take C's place (written only after the iteration) where the partials are too few
  p.part2 = 8 * c->grid <= b.nparts ? b.partials : reinterpret_cast<double*>(b.C);
  p.m = (int)m; p.n = (int)n;
  p.inv_sqrt_n = 1.0 / sqrt((double)n);
  return c;
}

void coop_solve_destroy(CoopSolve* c) { delete c; }

CoopForm coop_solve_form(const CoopSolve* c) {
  CoopForm f;
  f.tn = c->tn;
  f.blocks = c->grid;
  f.S[0] = c->p.sg;
  f.S[1] = c->p.su;
  f.split = c->split;
  return f;
}

cudaError_t coop_solve_launch(CoopSolve* c, const float* A, int64_t lda, float* U, int64_t ldu, float* H, int64_t ldh,
                              const StopRule& rule, cudaStream_t s) {
  CoSolve& p = c->p;
  p.A = A; p.lda = lda; p.U = U; p.ldu = ldu; p.H = H; p.ldh = ldh;
  p.v_tol = rule.tol * rule.tol * (double)p.n;
  p.stag2 = rule.stagnation * rule.stagnation;
  p.v_floor = rule.stag_floor * rule.stag_floor * (double)p.n;
  p.n_pre = rule.n_pre;
  p.max_iter = rule.max_iter;
  update_coeffs(rule, 0, p.pre_c1, p.pre_c3);   // of the preconditioning steps, where there are any
  p.withhold = tc_withhold();
  if (c->split) return co_launch_split(p, c->grid, s);
  return c->tn == 64 ? co_launch<64>(p, c->grid, s) : co_launch<128>(p, c->grid, s);
}

}  // namespace polar
