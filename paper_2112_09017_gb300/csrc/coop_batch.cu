// The loops of a batch of uneven problems in one cooperative launch: per step the Gram tiles of every running
// problem, the stop rules, the update tiles, with a grid barrier after each; then U^T A of every problem.
//
// Tiles are 128 x 128, taken from tables (problems by decreasing work) by the roles of coop_kernel.cuh. With
// separate grouped launches of 128 x 256 tiles the 256-problem batch (n 64..1024) spent 682 us on the Grams,
// 1371 us on the updates and 200 us on mirroring G per step: K is a few hundred, so a tile's output step is
// as long as its products unless it overlaps the next tile's. Here four slice buffers let the products run
// 256 of K ahead of the output step, narrower tiles pad less, G needs no mirror, and the steps after the last
// problem's stop cost nothing (they were three hundred launches that returned at once).
#include <math.h>

#include "batched.cuh"
#include "coop_kernel.cuh"
#include "stop_rule.cuh"

namespace polar {
namespace {

enum : int { CB_GRAM = 0, CB_UPDATE = 1, CB_H = 2 };

// Tiles of a table: this block's are blockIdx.x, blockIdx.x + gridDim.x, ..., without those of problems that
// have stopped (for H: that failed). Each role walks the table for itself, the next record and its problem's
// status on their way while a tile is worked on; no status changes during a product.
template <int KIND>
struct CoTableSrc {
  static constexpr bool TABLE = true, SPLIT = false, BKM = false;
  const CoBatch& p;
  const TcTile* tiles;
  int n, par, t;
  float c1, c3;
  int4 rec;          // of tile t
  int2 stat;         // its problem's (status, iters), once `have`
  bool have;
  int prob;          // of the tile given out last
  int cur_par;
  CoEpi e;

  __device__ __forceinline__ CoTableSrc(const CoBatch& b, int parity, float k1 = 0.f, float k3 = 0.f)
      : p(b), tiles(KIND == CB_GRAM ? b.gram_t : KIND == CB_UPDATE ? b.upd_t : b.h_t),
        n(KIND == CB_GRAM ? b.n_gram : KIND == CB_UPDATE ? b.n_upd : b.n_h), par(parity), t((int)blockIdx.x), c1(k1),
        c3(k3), have(false) {
    if (t < n) rec = __ldg(reinterpret_cast<const int4*>(tiles + t));
  }
  __device__ __forceinline__ int2 load_status(int prob_) const {
    return __ldcg(reinterpret_cast<const int2*>(&p.st[prob_].status));   // status and iters, adjacent
  }
  __device__ __forceinline__ const TcMapPair* maps(int prob_, int par_) const {
    return KIND == CB_GRAM ? p.gram_m[par_] + prob_ : KIND == CB_UPDATE ? p.upd_m[par_] + prob_
                                                                       : p.h_m + 2 * prob_ + par_;
  }
  __device__ __forceinline__ bool next(CoTile& c) {
    while (t < n) {
      if (!have) stat = load_status(rec.x);
      const int4 r = rec;
      const int2 s = stat;
      t += (int)gridDim.x;
      have = false;
      if (t < n) rec = __ldg(reinterpret_cast<const int4*>(tiles + t));
      if (KIND == CB_H ? !finished_ok(s.x) : s.x != ST_RUNNING) continue;
      prob = r.x;
      cur_par = KIND == CB_H ? (s.y & 1) : par;
      const TcMapPair* mp = maps(prob, cur_par);
      c.ma = reinterpret_cast<const CUtensorMap*>(mp->a);
      c.mb = KIND == CB_GRAM ? c.ma : reinterpret_cast<const CUtensorMap*>(mp->b);
      c.mbt = KIND == CB_UPDATE ? reinterpret_cast<const CUtensorMap*>(p.gram_m[0][prob].b) : nullptr;
      c.bi = r.y;
      c.bj = r.z;
      c.kbeg = 0;
      c.K = r.w;
      c.slice = __ldg(&p.meta[prob].slice);
      return true;
    }
    return false;
  }
  __device__ __forceinline__ void poke(bool producer) {
    if (have || t >= n) return;
    stat = load_status(rec.x);
    have = true;
    if (producer && KIND != CB_H) {
      const TcMapPair* mp = maps(rec.x, par);
      asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(mp->a)) : "memory");
      if (KIND == CB_UPDATE)
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(mp->b)) : "memory");
    }
  }
  __device__ __forceinline__ const CoEpi& epi(const CoTile& c) {
    const BMeta& m = p.meta[prob];
    e.N = (int)m.n;
    e.M = KIND == CB_UPDATE ? (int)m.m : (int)m.n;
    if (KIND == CB_H) {
      e.C = m.C;
      e.ldc = m.n;
    } else {
      e.ldo = m.ldp;
      e.out = KIND == CB_GRAM ? m.gp : m.xp[par ^ 1];
      e.os = KIND == CB_GRAM ? m.gps : m.xps;
      // the triangle's tiles are counted column by column
      if (KIND == CB_GRAM) e.tile_part = m.partials + ((int64_t)c.bj * (c.bj + 1) / 2 + c.bi) * EPI_WARPS;
      if (KIND == CB_UPDATE) {
        e.x = m.xp[par];
        e.ldx = m.ldp;
        e.xs = m.xps;
        e.c1 = c1;
        e.c3 = c3;
      }
    }
    return e;
  }
};

template <int P>
__global__ void __launch_bounds__(CO_THREADS, 1) co_batch_kernel(const __grid_constant__ CoBatch p) {
  extern __shared__ uint8_t co_raw[];
  constexpr int TN = 128;
  CoCtx x = co_setup<TN, P>(co_raw, p.sh->bar, p.wait_ns);
  CoPipe pipe;
  bool run = true;
  const double tol = p.sh->tol > 0 ? p.sh->tol : p.rule.tol;
  for (int k = 0; run && p.n_gram > 0; ++k) {
    const int b = k & 1;
    if (x.warp == 0) {
      if (x.lane == 0) co_producer<TN, P, true, false>(x, pipe, CoTableSrc<CB_GRAM>(p, b), p.withhold);
    } else if (x.warp == 1) {
      co_mma<TN, P, true, false>(x, pipe, CoTableSrc<CB_GRAM>(p, b));
    } else if (x.warp < CO_CTL_WARP) {
      co_epilogue<TN, TC_EPI_GRAM>(x, pipe, CoTableSrc<CB_GRAM>(p, b));
    }
    run = co_grid_sync(x);
    if (!run) break;
    // the stop rule of step k, one warp per running problem, its partials summed in a fixed order
    for (int q = blockIdx.x * CO_WARPS + x.warp; q < p.count; q += gridDim.x * CO_WARPS) {
      DevState& s = p.st[q];
      if (__ldcg(&s.status) != ST_RUNNING) continue;
      const BMeta& mt = p.meta[q];
      const double v = co_warp_sum<1>(mt.partials, mt.ntiles_gram * EPI_WARPS, 1, x.lane);
      if (x.lane == 0) {
        const double r = sqrt(v) * s.inv_sqrt_n;
        float c1, c3;
        if (batched_step_rule(s, p.rule, tol, r, k >= 2 ? s.ring[(k - 2) & 3] : 0.0, k, P, c1, c3))
          atomicAdd(&p.sh->running[k & 3], 1);
      }
    }
    run = co_grid_sync(x);
    if (!run || __ldcg(&p.sh->running[k & 3]) == 0) break;   // the same in every block
    if (blockIdx.x == 0 && threadIdx.x == 0) p.sh->running[(k + 2) & 3] = 0;   // read last at step k - 2
    const float c1 = k < p.rule.n_pre ? p.pre_c1 : 1.5f, c3 = k < p.rule.n_pre ? p.pre_c3 : -0.5f;
    if (x.warp == 0) {
      if (x.lane == 0) co_producer<TN, P, false, true>(x, pipe, CoTableSrc<CB_UPDATE>(p, b), p.withhold);
    } else if (x.warp == 1) {
      co_mma<TN, P, false, true>(x, pipe, CoTableSrc<CB_UPDATE>(p, b));
    } else if (x.warp < CO_CTL_WARP) {
      co_epilogue<TN, TC_EPI_NS>(x, pipe, CoTableSrc<CB_UPDATE>(p, b, c1, c3));
    }
    run = co_grid_sync(x);
  }
  // C = U^T A of every finished problem, from the planes of its own final iterate
  if (run) {
    if (x.warp == 0) {
      if (x.lane == 0) co_producer<TN, P, true, false>(x, pipe, CoTableSrc<CB_H>(p, 0), p.withhold);
    } else if (x.warp == 1) {
      co_mma<TN, P, true, false>(x, pipe, CoTableSrc<CB_H>(p, 0));
    } else if (x.warp < CO_CTL_WARP) {
      co_epilogue<TN, TC_EPI_STORE>(x, pipe, CoTableSrc<CB_H>(p, 0));
    }
  }
  __syncthreads();
  co_teardown<TN>(x, nullptr, &p.sh->err);
}

template <int P>
cudaError_t launch_p(const CoBatch& b, int grid, cudaStream_t s) {
  constexpr size_t smem = co_smem<128, P>();
  auto k = co_batch_kernel<P>;
  cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  void* args[] = {const_cast<CoBatch*>(&b)};
  return cudaLaunchCooperativeKernel(reinterpret_cast<const void*>(k), dim3((unsigned)grid), dim3(CO_THREADS), args,
                                     smem, s);
}

}  // namespace

cudaError_t launch_co_batch(const CoBatch& b, int max_grid, cudaStream_t s) {
  // Any number of blocks solves the batch: where fewer SMs are available than the device has, half as many, each
  // with twice the tiles.
  cudaError_t e = cudaSuccess;
  CoBatch c = b;
  for (int grid = max_grid; grid >= 1; grid /= 2, c.wait_ns *= 2) {
    e = c.P == 1 ? launch_p<1>(c, grid, s) : c.P == 2 ? launch_p<2>(c, grid, s) : launch_p<3>(c, grid, s);
    if (e != cudaErrorCooperativeLaunchTooLarge) return e;
    cudaGetLastError();
  }
  return e;
}

}  // namespace polar
