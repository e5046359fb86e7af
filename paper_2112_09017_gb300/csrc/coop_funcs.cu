// The Newton-Schulz inverse (Algorithm 2) and the Chebyshev matrix function (Clenshaw summation), each as one
// cooperative launch, for matrices whose products are a few waves of 128 x 64 or 128 x 128 tiles; the
// pieces are in coop_kernel.cuh. What bounds them there is what bounds the solve: with separate launches a
// 1001 x 1001 product ran as 32 tiles of 128 x 256 (56 us, and 145 us for a Clenshaw step at 1536 with its
// mirrored two-byte stores); here it is 128 tiles, and a Clenshaw step stores only the upper triangle.
#include <math.h>

#include <algorithm>

#include "coop_kernel.cuh"

namespace polar {
namespace {

// ------------------------------------------------------------------ inverse

struct CoInverse {
  CUtensorMap amn, ak, xmn[2], xk[2], pmn;   // A (rows x cols), X_k (cols x rows), P = A X_k
  const float* A;
  int64_t lda;
  float* X;
  int64_t ldx;
  uint16_t* ap;
  uint16_t* xp[2];
  uint16_t* pp;
  int64_t lpa, sa, lpx, sx, sp;
  double* norm;                              // EPI_WARPS per block
  double* step;                              // 2 EPI_WARPS per block
  DevState* st;
  int rows, cols, max_iter, withhold;
  int sa2, su;                               // split chains: blocks per tile of A X and of the update
};

template <int TN, bool SPLIT>
__device__ __forceinline__ void co_inverse(const CoInverse& p, uint8_t* co_raw) {
  CoCtx x = co_setup<TN, CO_P, SPLIT>(co_raw, &p.st->bar);
  const int N = p.rows, M = p.cols, tid = threadIdx.x;
  const int gtid = blockIdx.x * CO_THREADS + tid, gthr = gridDim.x * CO_THREADS;
  DevState* st = p.st;
  CoPipe pipe;
  bool run;
  // ---- planes of A
  {
    const bool vec = (reinterpret_cast<uintptr_t>(p.A) & 15u) == 0 && p.lda % 4 == 0;
    const int c8 = (M + 7) / 8;
    for (int u = gtid; u < N * c8; u += gthr) {
      const int r = u / c8, c = (u - r * c8) * 8;
      float v[8];
      load_row8(p.A + (int64_t)r * p.lda + c, M - c, vec, v);
      store_planes8(p.ap + (int64_t)r * p.lpa + c, p.sa, 3, v);
    }
    if (gtid == 0) {
      st->iters = 0;
      st->hist_len = 0;
      st->err_flags = 0;
      st->sym_err = 0.0;
      st->status = ST_RUNNING;
    }
    run = co_grid_sync(x);
  }
  // ---- a = ||A A^T||_F = ||A^T A||_F, from the upper triangle of A^T A
  if (run) {
    const CoTiles t = co_tiles<TN>(M, M, true);
    CoEpi e{};
    e.M = M; e.N = M;
    e.part = p.norm;
    co_product<TN, SPLIT, true, false, CO_EPI_NORM>(x, pipe, &p.amn, &p.amn, nullptr, t, N, e, 1, p.withhold);
    run = co_grid_sync(x);
  }
  int status = ST_TIMEOUT;
  if (run) {
    const double a = sqrt(co_warp_sum(p.norm, gridDim.x * EPI_WARPS, 1, x.lane));
    const bool good = isfinite(a) && a > 0.0;
    if (gtid == 0) {
      st->normA = a;
      if (!good) st->status = ST_NONFINITE;
    }
    run = good;   // the same in every block
    if (run) {
      // ---- X_0 = A^T / a, 32 x 32 tiles through shared memory (the stages are idle); the columns from
      // rows to the next multiple of 32 are zeros, as the step sums need them
      float* t = reinterpret_cast<float*>(x.smem);
      const float sc = (float)a;
      const int tr = (N + 31) / 32, tc = (M + 31) / 32;
      for (int b = blockIdx.x; b < tr * tc; b += gridDim.x) {
        const int r0 = (b / tc) * 32, c0 = (b % tc) * 32;
        __syncthreads();
        for (int u = tid; u < 1024; u += CO_THREADS) {
          const int yy = u >> 5, xx = u & 31;
          t[yy * 33 + xx] = (r0 + yy < N && c0 + xx < M) ? p.A[(int64_t)(r0 + yy) * p.lda + c0 + xx] : 0.0f;
        }
        __syncthreads();
        for (int u = tid; u < 1024; u += CO_THREADS) {
          const int yy = u >> 5, xx = u & 31;   // row c0 + yy of X_0, column r0 + xx
          if (c0 + yy >= M) continue;
          uint16_t q[3];
          split_planes_dev<3>(__fdiv_rn(t[xx * 33 + yy], sc), q);
          uint16_t* d = p.xp[0] + (int64_t)(c0 + yy) * p.lpx + r0 + xx;
#pragma unroll
          for (int i = 0; i < 3; ++i) d[i * p.sx] = q[i];
        }
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // before the next copies into the stages
      run = co_grid_sync(x);
    }
  }
  // ---- X <- 2 X - X (A X); the test of step k runs beside the product A X of step k + 1
  const CoTiles ta = co_tiles<TN>(N, N, false), tu = co_tiles<TN>(M, N, false);
  int k = 0;
  for (; run; ++k) {
    const int b = k & 1;
    {
      CoEpi e{};
      e.M = N; e.N = N;
      e.out = p.pp; e.ldo = p.lpx; e.os = p.sp;
      co_product<TN, SPLIT, false, false, TC_EPI_PLANES>(x, pipe, &p.ak, &p.xmn[b], nullptr, ta, M, e, p.sa2,
                                                         p.withhold);
    }
    if (x.warp == CO_CTL_WARP && k > 0) {
      // Algorithm 2's test after update k - 1: ||X' - X||_F / ||X'||_F against u 2^(k-1), u = 2^-24
      const double sd = co_warp_sum(p.step, gridDim.x * EPI_WARPS, 2, x.lane);
      const double sx = co_warp_sum(p.step + 1, gridDim.x * EPI_WARPS, 2, x.lane);
      if (x.lane == 0) {
        const double delta = sx > 0.0 ? sqrt(sd / sx) : INFINITY;
        const int s = !isfinite(delta) ? ST_NONFINITE
                      : delta <= ldexp(1.0, k - 1 - 24) ? ST_CONVERGED
                      : k >= p.max_iter ? ST_NOT_CONVERGED : ST_RUNNING;
        x.ctl->status = s;
        if (blockIdx.x == 0) {
          if (k <= POLAR_HIST) {
            st->res_hist[k - 1] = delta;
            st->hist_len = k;
          }
          st->sym_err = delta;
          st->iters = k;
          st->status = s;
        }
      }
    }
    run = co_grid_sync(x);
    if (!run) break;
    if (k > 0) status = *reinterpret_cast<volatile int*>(&x.ctl->status);
    else status = ST_RUNNING;
    if (status != ST_RUNNING) break;
    CoEpi e{};
    e.M = M; e.N = N;
    e.x = p.xp[b]; e.ldx = p.lpx; e.xs = p.sx;
    e.out = p.xp[b ^ 1]; e.ldo = p.lpx; e.os = p.sx;
    e.c1 = 2.0f; e.c3 = -1.0f;
    e.part = p.step;
    co_product<TN, SPLIT, false, false, TC_EPI_NS_STEP>(x, pipe, &p.xk[b], &p.pmn, nullptr, tu, N, e, p.su,
                                                        p.withhold);
    run = co_grid_sync(x);
  }
  if (run && (status == ST_CONVERGED || status == ST_NOT_CONVERGED)) {
    const uint16_t* X = p.xp[k & 1];
    const bool vec = (reinterpret_cast<uintptr_t>(p.X) & 15u) == 0 && p.ldx % 4 == 0;
    const int c8 = (N + 7) / 8;
    for (int u = gtid; u < M * c8; u += gthr) {
      const int r = u / c8, c = (u - r * c8) * 8;
      float v[8];
      sum_planes8(load_planes8(X + (int64_t)r * p.lpx + c, p.sx, true), v);
      store_row8(p.X + (int64_t)r * p.ldx + c, N - c, vec, v);
    }
  }
  co_teardown<TN, SPLIT>(x, st);
}

template <int TN>
__global__ void __launch_bounds__(CO_THREADS, 1) co_inverse_kernel(const __grid_constant__ CoInverse p) {
  extern __shared__ uint8_t co_raw[];
  co_inverse<TN, false>(p, co_raw);
}
__global__ void __cluster_dims__(CO_CLUSTER, 1, 1) __launch_bounds__(CO_THREADS, 1)
    co_inverse_split_kernel(const __grid_constant__ CoInverse p) {
  extern __shared__ uint8_t co_raw[];
  co_inverse<64, true>(p, co_raw);
}

// ------------------------------------------------------------------ Chebyshev

struct CoCheb {
  CUtensorMap tmn, bmn[3], bk[3];            // T; the rotating B_k, and mirrored
  const float* A;
  int64_t lda;
  float* F;
  int64_t ldf;
  uint16_t* tp;
  uint16_t* bp[3];
  int64_t ldp, sp;
  double am, bm, cd, cd1;                    // T = am A + bm I; c_d and c_{d-1}
  DevState* st;
  int n, degree, withhold;
  int S;                                     // split chains: blocks per tile
  float coef[COOP_MAX_DEGREE + 1];
};

// The planes of float32 value v at entry (i, j).
__device__ __forceinline__ void co_put(uint16_t* P, int64_t ld, int64_t ps, int i, int j, float v) {
  uint16_t q[3];
  split_planes_dev<3>(v, q);
  uint16_t* d = P + (int64_t)i * ld + j;
#pragma unroll
  for (int s = 0; s < 3; ++s) d[s * ps] = q[s];
}

template <int TN, bool SPLIT>
__device__ __forceinline__ void co_cheb(const CoCheb& p, uint8_t* co_raw) {
  CoCtx x = co_setup<TN, CO_P, SPLIT>(co_raw, &p.st->bar);
  const int n = p.n, d = p.degree, tid = threadIdx.x;
  const int nt = (n + 31) / 32, npair = nt * (nt + 1) / 2;
  CoPipe pipe;
  float* ta = reinterpret_cast<float*>(x.smem);
  float* tb = ta + 32 * 33;
  if (blockIdx.x == 0 && tid == 0) {
    p.st->err_flags = 0;
    p.st->status = ST_RUNNING;
  }
  // ---- T, B_d = c_d I and B_{d-1} = c_{d-1} I + 2 c_d T from the upper triangle of A: pairs of 32 x 32
  // tiles, the columns from n to the next multiple of 32 zeros. Each value is rounded once from float64.
  for (int t = blockIdx.x; t < npair; t += gridDim.x) {
    int bj = (int)((sqrtf(8.0f * (float)t + 1.0f) - 1.0f) * 0.5f);
    while (bj > 0 && bj * (bj + 1) / 2 > t) --bj;
    while ((bj + 1) * (bj + 2) / 2 <= t) ++bj;
    const int bi = t - bj * (bj + 1) / 2, i0 = bi * 32, j0 = bj * 32;
    __syncthreads();
    for (int u = tid; u < 1024; u += CO_THREADS) {
      const int yy = u >> 5, xx = u & 31, i = i0 + yy, j = j0 + xx;
      const bool in = i < n && j < n && i <= j;
      const double s = in ? p.am * (double)p.A[(int64_t)i * p.lda + j] + (i == j ? p.bm : 0.0) : 0.0;
      ta[yy * 33 + xx] = (float)s;
      tb[yy * 33 + xx] = in ? (float)(2.0 * p.cd * s + (i == j ? p.cd1 : 0.0)) : 0.0f;
    }
    __syncthreads();
    for (int u = tid; u < 1024; u += CO_THREADS) {
      const int yy = u >> 5, xx = u & 31;
      for (int side = 0; side < (bi < bj ? 2 : 1); ++side) {
        const int i = (side ? j0 : i0) + yy, j = (side ? i0 : j0) + xx;
        if (i >= n) continue;
        // above the diagonal as stored, below it (the other tile of the pair, or within a diagonal one) transposed
        const int s = (side || (bi == bj && yy > xx)) ? xx * 33 + yy : yy * 33 + xx;
        co_put(p.tp, p.ldp, p.sp, i, j, ta[s]);
        co_put(p.bp[(d - 1) % 3], p.ldp, p.sp, i, j, tb[s]);
        co_put(p.bp[d % 3], p.ldp, p.sp, i, j, i == j ? (float)p.cd : 0.0f);
      }
    }
  }
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // before the first copies into the stages
  bool run = co_grid_sync(x);
  // ---- B_k = 2 T B_{k+1} - B_{k+2} + c_k I for k = d-2 .. 1, F = T B_1 - B_2 + c_0 I
  const CoTiles tt = co_tiles<TN>(n, n, true);
  for (int k = d - 2; k >= 0 && run; --k) {
    CoEpi e{};
    e.M = n; e.N = n;
    e.x = p.bp[(k + 2) % 3]; e.ldx = p.ldp; e.xs = p.sp;
    e.out = p.bp[k % 3]; e.ldo = p.ldp; e.os = p.sp;
    e.c1 = -1.0f;
    e.c3 = k > 0 ? 2.0f : 1.0f;
    e.diag = p.coef[k];
    co_product<TN, SPLIT, true, true, TC_EPI_CLENSHAW>(x, pipe, &p.tmn, &p.bmn[(k + 1) % 3], &p.bk[(k + 1) % 3], tt, n,
                                                       e, p.S, p.withhold);
    run = co_grid_sync(x);
  }
  // ---- F from the upper triangle
  if (run) {
    const uint16_t* B = p.bp[0];
    for (int t = blockIdx.x; t < npair; t += gridDim.x) {
      int bj = (int)((sqrtf(8.0f * (float)t + 1.0f) - 1.0f) * 0.5f);
      while (bj > 0 && bj * (bj + 1) / 2 > t) --bj;
      while ((bj + 1) * (bj + 2) / 2 <= t) ++bj;
      const int bi = t - bj * (bj + 1) / 2, i0 = bi * 32, j0 = bj * 32;
      __syncthreads();
      for (int u = tid; u < 128; u += CO_THREADS) {   // 32 rows of four 16-byte groups per plane
        const int yy = u >> 2, g = (u & 3) * 8;
        float v[8];
        sum_planes8(load_planes8(B + (int64_t)(i0 + yy) * p.ldp + j0 + g, p.sp, i0 + yy < n), v);
#pragma unroll
        for (int e = 0; e < 8; ++e) ta[yy * 33 + g + e] = v[e];
      }
      __syncthreads();
      for (int u = tid; u < 1024; u += CO_THREADS) {
        const int yy = u >> 5, xx = u & 31;
        if (i0 + yy < n && j0 + xx < n)
          p.F[(int64_t)(i0 + yy) * p.ldf + j0 + xx] = (bi == bj && yy > xx) ? ta[xx * 33 + yy] : ta[yy * 33 + xx];
        if (bi < bj && j0 + yy < n && i0 + xx < n) p.F[(int64_t)(j0 + yy) * p.ldf + i0 + xx] = ta[xx * 33 + yy];
      }
    }
  }
  co_teardown<TN, SPLIT>(x, p.st);
}

template <int TN>
__global__ void __launch_bounds__(CO_THREADS, 1) co_cheb_kernel(const __grid_constant__ CoCheb p) {
  extern __shared__ uint8_t co_raw[];
  co_cheb<TN, false>(p, co_raw);
}
__global__ void __cluster_dims__(CO_CLUSTER, 1, 1) __launch_bounds__(CO_THREADS, 1)
    co_cheb_split_kernel(const __grid_constant__ CoCheb p) {
  extern __shared__ uint8_t co_raw[];
  co_cheb<64, true>(p, co_raw);
}

// ------------------------------------------------------------------ host

template <class Params>
cudaError_t co_run(void (*kernel)(Params), const Params& p, size_t smem, int grid, cudaStream_t s) {
  cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid, 1, 1);
  cfg.blockDim = dim3(CO_THREADS, 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeCooperative;
  attr.val.cooperative = 1;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  void* args[] = {const_cast<Params*>(&p)};
  return cudaLaunchKernelExC(&cfg, reinterpret_cast<const void*>(kernel), args);
}

TcOperand co_operand(const uint16_t* planes, int64_t rows, int64_t cols, int64_t ld, int64_t stride) {
  TcOperand o{};
  o.planes = planes; o.rows = rows; o.cols = cols; o.ld = ld; o.plane_stride = stride;
  return o;
}

// Blocks for products of at most m x n and passes over that many entries.
int co_grid(int64_t m, int64_t n, int tn, int sms) {
  const int64_t tiles = tn == 64 ? co_tiles<64>(m, n, false).ntiles : co_tiles<128>(m, n, false).ntiles;
  return (int)std::min<int64_t>(sms, std::max<int64_t>(tiles, (m * n + 8191) / 8192));
}

}  // namespace

size_t coop_inverse_sums(int sms) { return (size_t)sms * EPI_WARPS * 3 * sizeof(double); }

cudaError_t coop_inverse_launch(const CoopInverseArgs& a, const CoopForm& f, int sms, cudaStream_t s) {
  CoInverse p{};
  const TcOperand A = co_operand(a.ap, a.rows, a.cols, a.lpa, a.sa), P = co_operand(a.pp, a.rows, a.rows, a.lpx, a.sp);
  bool ok = tc_make_map(&p.amn, A, CO_P, true, 0) && tc_make_map(&p.ak, A, CO_P, false, BM) &&
            tc_make_map(&p.pmn, P, CO_P, true, 0);
  for (int i = 0; i < 2; ++i) {
    const TcOperand X = co_operand(a.xp[i], a.cols, a.rows, a.lpx, a.sx);
    ok = ok && tc_make_map(&p.xmn[i], X, CO_P, true, 0) && tc_make_map(&p.xk[i], X, CO_P, false, BM);
    p.xp[i] = a.xp[i];
  }
  if (!ok) return cudaErrorInvalidValue;
  p.A = a.A; p.lda = a.lda; p.X = a.X; p.ldx = a.ldx;
  p.ap = a.ap; p.pp = a.pp;
  p.lpa = a.lpa; p.sa = a.sa; p.lpx = a.lpx; p.sx = a.sx; p.sp = a.sp;
  const int grid = co_grid(a.rows, a.rows, f.tn, sms);
  p.sa2 = f.S[0];
  p.su = f.S[1];
  p.norm = a.sums;
  p.step = a.sums + (size_t)sms * EPI_WARPS;
  p.st = a.st;
  p.rows = (int)a.rows; p.cols = (int)a.cols; p.max_iter = a.max_iter;
  p.withhold = tc_withhold();
  if (f.split) return co_run(co_inverse_split_kernel, p, co_smem<64, CO_P, true>(), f.blocks, s);
  return f.tn == 64 ? co_run(co_inverse_kernel<64>, p, co_smem<64>(), grid, s)
                    : co_run(co_inverse_kernel<128>, p, co_smem<128>(), grid, s);
}

cudaError_t coop_cheb_launch(const CoopChebArgs& a, const CoopForm& f, int sms, cudaStream_t s) {
  CoCheb p{};
  if (a.degree < 2 || a.degree > COOP_MAX_DEGREE) return cudaErrorInvalidValue;
  bool ok = tc_make_map(&p.tmn, co_operand(a.tp, a.n, a.n, a.ldp, a.sp), CO_P, true, 0);
  for (int i = 0; i < 3; ++i) {
    const TcOperand B = co_operand(a.bp[i], a.n, a.n, a.ldp, a.sp);
    ok = ok && tc_make_map(&p.bmn[i], B, CO_P, true, 0) && tc_make_map(&p.bk[i], B, CO_P, false, f.tn);
    p.bp[i] = a.bp[i];
  }
  if (!ok) return cudaErrorInvalidValue;
  p.A = a.A; p.lda = a.lda; p.F = a.F; p.ldf = a.ldf;
  p.tp = a.tp; p.ldp = a.ldp; p.sp = a.sp;
  p.am = a.am; p.bm = a.bm; p.cd = a.coef[a.degree]; p.cd1 = a.coef[a.degree - 1];
  for (int k = 0; k <= a.degree; ++k) p.coef[k] = (float)a.coef[k];
  p.st = a.st;
  p.n = (int)a.n; p.degree = a.degree;
  p.S = f.S[0];
  p.withhold = tc_withhold();
  const int grid = co_grid(a.n, a.n, f.tn, sms);
  if (f.split) return co_run(co_cheb_split_kernel, p, co_smem<64, CO_P, true>(), f.blocks, s);
  return f.tn == 64 ? co_run(co_cheb_kernel<64>, p, co_smem<64>(), grid, s)
                    : co_run(co_cheb_kernel<128>, p, co_smem<128>(), grid, s);
}

}  // namespace polar
