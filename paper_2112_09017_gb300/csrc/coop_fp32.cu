// One plain-form (float32, SIMT) polar solve in one cooperative launch, for matrices whose products have few
// 128 x 128 tiles: the 32 x 32 tiles of simt_small.cuh, a grid barrier between products, the structure of
// coop_solve.cu. 300 x 200 took 2520 us as separate launches (per step a Gram of 45 us on three SMs, an
// update of 25 us on six, and the small kernels between them).
#include <math.h>

#include <algorithm>
#include <new>

#include "coop_barrier.cuh"
#include "simt_small.cuh"

namespace polar {
namespace {

struct Co32 {
  const float* A;
  int64_t lda;
  float* U;
  int64_t ldu;
  float* H;
  int64_t ldh;
  float* x[2];
  int64_t ldx;
  float* G;                 // G, and C = U^T A at the end
  int64_t ldg;
  double* partials;         // one per block, two per block at the end
  DevState* st;
  int m, n;
  double v_tol, stag2, v_floor;
  int n_pre, max_iter;
  float pre_c1, pre_c3;
  double inv_sqrt_n;
  int withhold;             // test hook: the first block leaves at once, the others' waits expire
};

struct Co32Ctl {
  double red[SS_THREADS / 32];
  double v;
  int abort;
  int status;
};

// Block sum of one double per thread, in a fixed order; every thread gets it.
__device__ __forceinline__ double c32_block_sum(Co32Ctl& c, double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) c.red[threadIdx.x >> 5] = v;
  __syncthreads();
  double t = 0.0;
#pragma unroll
  for (int w = 0; w < SS_THREADS / 32; ++w) t += c.red[w];
  return t;
}

// Sum of the blocks' partials, in a fixed order, by one warp.
__device__ __forceinline__ double c32_grid_sum(const double* p, int n, int stride, int lane) {
  double v = 0.0;
  for (int i = lane; i < n; i += 32) v += __ldcg(p + (size_t)i * stride);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

__device__ __forceinline__ void c32_tri(int t, int& bi, int& bj) {
  int j = (int)((sqrtf(8.0f * (float)t + 1.0f) - 1.0f) * 0.5f);
  while (j > 0 && j * (j + 1) / 2 > t) --j;
  while ((j + 1) * (j + 2) / 2 <= t) ++j;
  bj = j;
  bi = t - j * (j + 1) / 2;
}

__global__ void __launch_bounds__(SS_THREADS, 1) co_fp32_kernel(const __grid_constant__ Co32 p) {
  extern __shared__ __align__(16) unsigned char c32_raw[];
  SsSmem& sm = *reinterpret_cast<SsSmem*>(c32_raw);
  Co32Ctl& ctl = *reinterpret_cast<Co32Ctl*>(c32_raw + sizeof(SsSmem));
  const int m = p.m, n = p.n, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int r0t = tid >> 5, ct = tid & 31;        // a tile's entries (r0t, ct) and (r0t + 16, ct) are this thread's
  const int tm = (m + SS_T - 1) / SS_T, tn = (n + SS_T - 1) / SS_T, ntri = tn * (tn + 1) / 2;
  DevState* st = p.st;
  GridBarrier bar(reinterpret_cast<GridBarWords*>(&st->bar), &ctl.abort);
  if (tid == 0) ctl.abort = p.withhold && blockIdx.x == 0 ? 1 : 0;
  __syncthreads();
  // ---- ||A||_F
  double acc = 0.0;
  for (int r = blockIdx.x * (SS_THREADS / 32) + warp; r < m; r += gridDim.x * (SS_THREADS / 32))
    for (int c = lane; c < n; c += 32) {
      const double v = (double)p.A[(int64_t)r * p.lda + c];
      acc = fma(v, v, acc);
    }
  acc = c32_block_sum(ctl, acc);
  if (tid == 0) p.partials[blockIdx.x] = acc;
  bool run = bar.sync();
  if (run) {
    const double nrm = sqrt(c32_grid_sum(p.partials, gridDim.x, 1, lane));
    const bool good = isfinite(nrm) && nrm > 0.0;
    if (blockIdx.x == 0 && tid == 0) {
      st->normA = nrm;
      st->inv_sqrt_n = p.inv_sqrt_n;
      st->iters = 0;
      st->hist_len = 0;
      st->err_flags = 0;
      st->planes_next = 0;
      st->fp8_on = 0;
      st->sym_err = 0.0;
      st->status = good ? ST_RUNNING : ST_NONFINITE;
    }
    run = good;            // the same in every block
    if (run) {
      const float s = (float)nrm;
      for (int r = blockIdx.x * (SS_THREADS / 32) + warp; r < m; r += gridDim.x * (SS_THREADS / 32))
        for (int c = lane; c < n; c += 32)
          p.x[0][(int64_t)r * p.ldx + c] = __fdiv_rn(p.A[(int64_t)r * p.lda + c], s);
      run = bar.sync();
    }
  }
  // ---- the iteration
  double v_km1 = 0.0, v_km2 = 0.0;
  int it = 0, status = ST_TIMEOUT;
  for (int k = 0; run; ++k) {
    const int b = k & 1;
    const SsOperand xmn{p.x[b], p.ldx, n, true}, xk{p.x[b], p.ldx, m, true}, gmn{p.G, p.ldg, n, true};
    double part = 0.0;
    for (int t = blockIdx.x; t < ntri; t += gridDim.x) {
      int bi, bj;
      c32_tri(t, bi, bj);
      ss_tile<false, false>(sm, xmn, xmn, bi * SS_T, bj * SS_T, m);
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int rr = r0t + 16 * h, r = bi * SS_T + rr, c = bj * SS_T + ct;
        if (r < n && c < n && r <= c) {
          const float v = ss_sum(sm, rr, ct);
          p.G[(int64_t)r * p.ldg + c] = v;
          const double d = (double)v - (r == c ? 1.0 : 0.0);
          part += (r == c ? 1.0 : 2.0) * d * d;
        }
        // the mirrored entry: row bj * 32 + rr, column bi * 32 + ct
        const int r2 = bj * SS_T + rr, c2 = bi * SS_T + ct;
        if (r2 < n && c2 < n && c2 < r2) p.G[(int64_t)r2 * p.ldg + c2] = ss_sum(sm, ct, rr);
      }
      __syncthreads();
    }
    part = c32_block_sum(ctl, part);
    if (tid == 0) p.partials[blockIdx.x] = part;
    run = bar.sync();
    if (!run) break;
    if (k < p.max_iter) {
      const float c1 = k < p.n_pre ? p.pre_c1 : 1.5f, c3 = k < p.n_pre ? p.pre_c3 : -0.5f;
      const float* xo = p.x[b];
      float* xn = p.x[b ^ 1];
      for (int t = blockIdx.x; t < tm * tn; t += gridDim.x) {
        const int bj = t / tm, bi = t - bj * tm;
        ss_tile<true, false>(sm, xk, gmn, bi * SS_T, bj * SS_T, n);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int rr = r0t + 16 * h, r = bi * SS_T + rr, c = bj * SS_T + ct;
          if (r < m && c < n) {
            const int64_t o = (int64_t)r * p.ldx + c;
            xn[o] = fmaf(c1, __ldcg(xo + o), c3 * ss_sum(sm, rr, ct));   // c3 = -0.5: one rounding
          }
        }
        __syncthreads();
      }
    }
    // the stop test of X_k on squares (co_stop_status's rule), by the last warp of every block
    if (warp == SS_THREADS / 32 - 1) {
      const double v = c32_grid_sum(p.partials, gridDim.x, 1, lane);
      const bool testing = k >= p.n_pre;
      const int s = !isfinite(v) ? ST_NONFINITE
                    : testing && v <= p.v_tol ? ST_CONVERGED
                    : testing && k >= p.n_pre + 2 && v > p.stag2 * v_km2 && v < p.v_floor ? ST_NOT_CONVERGED
                    : k >= p.max_iter ? ST_NOT_CONVERGED : ST_RUNNING;
      v_km2 = v_km1;
      v_km1 = v;
      if (lane == 0) {
        ctl.status = s;
        if (blockIdx.x == 0) {
          st->res_hist[k] = sqrt(v) * p.inv_sqrt_n;   // k <= max_iter < POLAR_HIST
          st->planes_hist[k] = 0;
          st->hist_len = k + 1;
          st->iters = k;
          st->status = s;
        }
      }
    }
    run = bar.sync();
    if (!run) break;
    status = *reinterpret_cast<volatile int*>(&ctl.status);
    it = k;
    if (status != ST_RUNNING) break;
  }
  // ---- C = U^T A, then U and H = (C + C^T) / 2
  if (run && (status == ST_CONVERGED || status == ST_NOT_CONVERGED)) {
    const SsOperand u{p.x[it & 1], p.ldx, n, true};
    const SsOperand a{p.A, p.lda, n, (reinterpret_cast<uintptr_t>(p.A) & 15u) == 0 && p.lda % 4 == 0};
    for (int t = blockIdx.x; t < tn * tn; t += gridDim.x) {
      const int bj = t / tn, bi = t - bj * tn;
      ss_tile<false, false>(sm, u, a, bi * SS_T, bj * SS_T, m);
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int rr = r0t + 16 * h, r = bi * SS_T + rr, c = bj * SS_T + ct;
        if (r < n && c < n) p.G[(int64_t)r * p.ldg + c] = ss_sum(sm, rr, ct);
      }
      __syncthreads();
    }
    run = bar.sync();
    if (run) {
      const float* X = p.x[it & 1];
      for (int r = blockIdx.x * (SS_THREADS / 32) + warp; r < m; r += gridDim.x * (SS_THREADS / 32))
        for (int c = lane; c < n; c += 32) p.U[(int64_t)r * p.ldu + c] = __ldcg(X + (int64_t)r * p.ldx + c);
      double skew = 0.0, full = 0.0;
      float* ta = &sm.red[0][0][0];   // two 32 x 33 tiles
      float* tb = &sm.red[1][0][0];
      for (int t = blockIdx.x; t < ntri; t += gridDim.x) {
        int bi, bj;
        c32_tri(t, bi, bj);
        const int i0 = bi * SS_T, j0 = bj * SS_T;
        __syncthreads();
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int yy = r0t + 16 * h;
          ta[yy * 33 + ct] = (i0 + yy < n && j0 + ct < n) ? __ldcg(p.G + (int64_t)(i0 + yy) * p.ldg + j0 + ct) : 0.0f;
          tb[yy * 33 + ct] = (j0 + yy < n && i0 + ct < n) ? __ldcg(p.G + (int64_t)(j0 + yy) * p.ldg + i0 + ct) : 0.0f;
        }
        __syncthreads();
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int yy = r0t + 16 * h;
          if (i0 + yy < n && j0 + ct < n) {
            const float c = ta[yy * 33 + ct], cc = tb[ct * 33 + yy];
            p.H[(int64_t)(i0 + yy) * p.ldh + j0 + ct] = 0.5f * (c + cc);
            const double d = 0.5 * ((double)c - (double)cc);
            skew = fma(bi < bj ? 2.0 * d : d, d, skew);
            full = fma((double)c, (double)c, full);
            if (bi < bj) full = fma((double)cc, (double)cc, full);
          }
          if (bi < bj && j0 + yy < n && i0 + ct < n)
            p.H[(int64_t)(j0 + yy) * p.ldh + i0 + ct] = 0.5f * (tb[yy * 33 + ct] + ta[ct * 33 + yy]);
        }
      }
      const double s1 = c32_block_sum(ctl, skew);
      const double s2 = c32_block_sum(ctl, full);
      if (tid == 0) {
        p.partials[2 * blockIdx.x] = s1;
        p.partials[2 * blockIdx.x + 1] = s2;
      }
      run = bar.sync();
      if (run && blockIdx.x == 0 && warp == 0) {
        const double a2 = c32_grid_sum(p.partials, gridDim.x, 2, lane);
        const double c2 = c32_grid_sum(p.partials + 1, gridDim.x, 2, lane);
        if (lane == 0) st->sym_err = c2 > 0.0 ? sqrt(a2 / c2) : 0.0;
      }
    }
  }
  __syncthreads();
  if (tid == 0 && ctl.abort) {
    atomicOr(&st->err_flags, 1u);
    st->status = ST_TIMEOUT;
  }
  bar.leave();
}

constexpr size_t c32_smem() { return sizeof(SsSmem) + sizeof(Co32Ctl); }

}  // namespace

struct CoopFp32 {
  Co32 p;
  int grid;
};

// Taken where a step finishes first. In SM cycles, fitted to the steps of 45 solves of up to 2^24 entries (5 % off): a
// wave of 32 x 32 tiles takes 26 per K, a step's barriers and stop test 21000; in separate launches a wave of 128 x
// 128 tiles 236 per K, a step's launches 64000. One launch against separate ones, us per step: 300 x 200 18 and 98,
// 1024^2 167 and 245, 1256^2 291 and 323, 1580^2 524 and 562; 1755^2 708 and 630, 2108^2 1143 and 972, 3159 x 1757
// 1222 and 981.
bool coop_fp32_fits(int64_t m, int64_t n, int sms) {
  auto tri = [](int64_t t) { return t * (t + 1) / 2; };
  auto waves = [](int64_t t, int64_t on) { return (double)((t + on - 1) / on); };
  const int64_t um = (m + 127) / 128, un = (n + 127) / 128;
  const double big = 236.0 * (waves(tri(un), sms) * (double)m + waves(um * un, sms) * (double)n) + 64000.0;
  const int64_t tm = (m + SS_T - 1) / SS_T, tn = (n + SS_T - 1) / SS_T, grid = std::min<int64_t>(tm * tn, sms);
  const double small = 26.0 * (waves(tri(tn), grid) * (double)m + waves(tm * tn, grid) * (double)n) + 21000.0;
  return m * n <= (int64_t)1 << 24 && small < big;
}

CoopFp32* coop_fp32_create(const CoopFp32Buffers& b, int64_t m, int64_t n, int sms) {
  if (!coop_fp32_fits(m, n, sms)) return nullptr;
  CoopFp32* c = new (std::nothrow) CoopFp32();
  if (!c) return nullptr;
  if (cudaFuncSetAttribute(co_fp32_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)c32_smem()) !=
      cudaSuccess) {
    cudaGetLastError();
    delete c;
    return nullptr;
  }
  const int64_t tiles = ((m + SS_T - 1) / SS_T) * ((n + SS_T - 1) / SS_T);
  c->grid = (int)std::max<int64_t>(1, std::min<int64_t>(std::min<int64_t>(tiles, sms), b.nparts / 2));
  Co32& p = c->p;
  p.x[0] = b.x[0]; p.x[1] = b.x[1]; p.ldx = b.ldx;
  p.G = b.G; p.ldg = b.ldg;
  p.partials = b.partials; p.st = b.st;
  p.m = (int)m; p.n = (int)n;
  p.inv_sqrt_n = 1.0 / sqrt((double)n);
  return c;
}

void coop_fp32_destroy(CoopFp32* c) { delete c; }

int coop_fp32_blocks(const CoopFp32* c) { return c->grid; }

cudaError_t coop_fp32_launch(CoopFp32* c, const float* A, int64_t lda, float* U, int64_t ldu, float* H, int64_t ldh,
                             const StopRule& rule, cudaStream_t s) {
  Co32& p = c->p;
  p.A = A; p.lda = lda; p.U = U; p.ldu = ldu; p.H = H; p.ldh = ldh;
  p.v_tol = rule.tol * rule.tol * (double)p.n;
  p.stag2 = rule.stagnation * rule.stagnation;
  p.v_floor = rule.stag_floor * rule.stag_floor * (double)p.n;
  p.n_pre = rule.n_pre;
  p.max_iter = rule.max_iter;
  update_coeffs(rule, 0, p.pre_c1, p.pre_c3);   // of the preconditioning steps, where there are any
  p.withhold = tc_withhold();
  void* args[] = {&p};
  return cudaLaunchCooperativeKernel(reinterpret_cast<const void*>(co_fp32_kernel), dim3((unsigned)c->grid),
                                     dim3(SS_THREADS), args, c32_smem(), s);
}

}  // namespace polar
