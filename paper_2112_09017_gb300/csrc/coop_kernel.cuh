// Persistent cooperative kernels: a whole chain of split-BF16 tensor-core products (three planes, six
// passes) in one launch, for sizes at which a product is a few waves of small tiles. The chain's
// products depend on each other through global memory, so a grid barrier separates them; what it replaces
// per product is a kernel launch, the set-up of barriers, TMEM and descriptors, and the small kernels
// between the products (residual and stop rule, mirror).
//
// The product itself is that of gemm_tc_kernel.cuh: TMA producer, one MMA-issuing thread, eight epilogue
// warps that promote every 64-deep k-slice into FP32 registers with round-to-nearest, the same passes in
// the same order. What differs is the tile: 128 x TN with TN = 64 or 128, all eight epilogue warps on one
// tile (TN / 2 columns each), so that a matrix of a few hundred rows spreads over the chip and the output
// step of a tile is short. G is kept as its upper triangle only: a k-block of the update's B operand below
// the triangle is read from the mirrored place as a K-major operand, above it as an MN-major one.
//
// The blocks wait on one another, so the launch is cooperative (every block resident, or an error), and
// every wait is bounded: a grid barrier that expires raises the block's abort flag like an mbarrier that
// expires, the block leaves, and the others leave when their own waits expire.
#pragma once

#include "coop_barrier.cuh"
#include "gemm_tc_kernel.cuh"

namespace polar {
namespace {

constexpr int CO_P = 3;                     // planes of the chains (the batched ones take 1, 2 or 3)
constexpr int CO_THREADS = NTHREADS + 32;   // one warp more, for what must not hold up the products: the stop test
constexpr int CO_WARPS = CO_THREADS / 32;
constexpr int CO_CTL_WARP = CO_WARPS - 1;
// beside the TcEpi kinds: no output, ||C||_F^2 of a symmetric product; C = c3 acc + c1 C, any pitch and alignment
constexpr int CO_EPI_NORM = 16, CO_EPI_GEMM = 17;

template <int TN, int P = CO_P, bool SPLIT = false>
struct CoCfg {
  // A stage holds SUB k-blocks of 32: with 64-wide tiles two, because the twelve short MMAs of one do not
  // cover the waits and commits of a stage (1024 x 1024: 766 us per solve against 824 with six stages of one).
  // A split chain has 34 KiB less (the exchange of partial tiles) and takes five stages of one: two of two
  // are too few in flight (1000 x 700: 684 against 537 us).
  static constexpr int SUB = TN == 64 && !SPLIT ? 2 : 1;
  // 72, 48 or (split) 36 KiB each
  static constexpr int STAGES = TN == 64 ? (SPLIT ? 5 : 3) : 4;
  static constexpr uint32_t A_BYTES = P * A_PLANE;         // of one k-block
  static constexpr uint32_t B_BYTES = P * TN * BK * 2;
  static constexpr uint32_t KB_BYTES = A_BYTES + B_BYTES;
  static constexpr uint32_t STAGE_BYTES = SUB * KB_BYTES;
  static constexpr int BKS = SUB * BK;                     // K of one stage
  static constexpr int NBUF = 4;                           // TMEM slice buffers of TN columns
  static constexpr uint32_t TCOLS = NBUF * TN;
  static constexpr int CW = TN / 2;                        // columns of one epilogue warp
  static constexpr int SLICE = 64 / BKS;                   // stages per promoted slice
};

// Clusters of a split chain, and floats per row of the exchange buffer: [source][row][columns].
constexpr int CO_CLUSTER = 4;
constexpr int CO_XLD = 64 + 4;
constexpr size_t CO_XBUF = (size_t)128 * CO_XLD * 4;

// Shared control block, behind the stages (and the exchange buffer).
struct CoCtl {
  uint64_t bars[2 * 5 + 2 * 4 + 2];
  double red[CO_WARPS];
  uint32_t tmem;
  int abort;
  int status;              // of the last stop test
};

template <int TN, int P = CO_P, bool SPLIT = false>
constexpr size_t co_smem() {
  return (size_t)CoCfg<TN, P, SPLIT>::STAGES * CoCfg<TN, P, SPLIT>::STAGE_BYTES + (SPLIT ? CO_XBUF : 0) + sizeof(CoCtl) + 1024;
}

// What a role carries from one product to the next.
struct CoPipe {
  int stage = 0;
  uint32_t phase = 0;
  int buf = 0;
  uint32_t buf_phase = 0;
};

struct CoCtx {
  CoCtl* ctl;
  uint8_t* smem;             // 1024-byte aligned, the stages
  uint32_t smem_base, tmem;
  uint32_t xbuf, xfull;      // split chains: the exchange buffer and its barrier (shared addresses)
  uint32_t xphase;
  Bars br;
  GridBarrier bar;
  int warp, lane;
  volatile int* abort_flag;
};

// One product of a chain: tiles of 128 x TN, rectangular (column by column) or the upper triangle's.
struct CoTiles {
  int tm, tn, ntiles, tri;
};

template <int TN>
__host__ __device__ inline CoTiles co_tiles(int64_t M, int64_t N, bool tri) {
  CoTiles t;
  t.tm = (int)((M + BM - 1) / BM);
  t.tn = (int)((N + TN - 1) / TN);
  t.tri = tri ? 1 : 0;
  if (!tri) t.ntiles = t.tm * t.tn;
  else if (TN == 128) t.ntiles = t.tn * (t.tn + 1) / 2;
  else t.ntiles = (t.tn / 2) * (t.tn / 2 + 1) + (t.tn & 1) * (t.tn / 2 + 1);
  return t;
}

template <int TN>
__device__ __forceinline__ void co_coords(const CoTiles& c, int t, int& bi, int& bj) {
  if (!c.tri) {
    bj = t / c.tm;
    bi = t - bj * c.tm;
  } else if (TN == 128) {   // column bj holds bj + 1 tiles
    int j = (int)((sqrtf(8.0f * (float)t + 1.0f) - 1.0f) * 0.5f);
    while (j > 0 && j * (j + 1) / 2 > t) --j;
    while ((j + 1) * (j + 2) / 2 <= t) ++j;
    bj = j;
    bi = t - j * (j + 1) / 2;
  } else {                  // columns 2j and 2j + 1 hold j + 1 tiles each
    int j = (int)((sqrtf(4.0f * (float)t + 1.0f) - 1.0f) * 0.5f);
    while (j > 0 && j * (j + 1) > t) --j;
    while ((j + 1) * (j + 2) <= t) ++j;
    const int r = t - j * (j + 1);
    bj = 2 * j + (r > j ? 1 : 0);
    bi = r > j ? r - j - 1 : r;
  }
}

// What the roles need of one tile: its operand maps, place, K, and stages per promoted slice.
struct CoTile {
  const CUtensorMap* ma;
  const CUtensorMap* mb;
  const CUtensorMap* mbt;    // the mirrored (K-major) map of a B whose upper triangle alone is stored
  int bi, bj;
  int kbeg, K;               // from kbeg to below K
  int slice;                 // k-blocks of 32 per promoted slice
};

struct CoEpi;

// Tiles of one product of a chain: this block's are blockIdx.x, blockIdx.x + gridDim.x, ... With S > 1 (split
// chains) S neighbouring blocks of a cluster share a tile, each taking a part of K, and there are at least as
// many such groups as tiles.
template <int TN, bool SPLIT_ = false, bool BKM_ = false>
struct CoChainSrc {
  static constexpr bool TABLE = false, SPLIT = SPLIT_;
  static constexpr bool BKM = BKM_;          // B is a K-major operand (its map is mbt)
  const CUtensorMap *ma, *mb, *mbt;
  CoTiles ct;
  int K, kbeg;
  const CoEpi* e;
  int t, dt;
  __device__ __forceinline__ CoChainSrc(const CUtensorMap* a, const CUtensorMap* b, const CUtensorMap* bt, CoTiles c,
                                        int k, const CoEpi* ep = nullptr, int S = 1)
      : ma(a), mb(b), mbt(bt), ct(c), K(k), kbeg(0), e(ep), t((int)blockIdx.x), dt((int)gridDim.x) {
    if (SPLIT && S > 1) {
      const int sub = t % S, kc = ((k + S - 1) / S + 63) / 64 * 64;
      t /= S;
      dt /= S;
      kbeg = sub * kc;
      K = min(k, kbeg + kc);
    }
  }
  __device__ __forceinline__ bool next(CoTile& c) {
    if (t >= ct.ntiles) return false;
    co_coords<TN>(ct, t, c.bi, c.bj);
    t += dt;
    c.ma = ma; c.mb = mb; c.mbt = mbt;
    c.kbeg = kbeg;
    c.K = K;
    c.slice = 64 / BK;
    return true;
  }
  __device__ __forceinline__ void poke(bool) {}
  __device__ __forceinline__ const CoEpi& epi(const CoTile&) { return *e; }
};

// First k of the B operand that a column tile at n0 reads from the mirrored place: the rows above it were
// stored by the upper triangle's tiles (whole 128-row tiles that hold an entry on or above the diagonal).
template <int TN>
__device__ __forceinline__ int co_mirror_from(int n0) { return 128 * ((n0 + TN - 1) / 128 + 1); }

// ------------------------------------------------------------------ set-up, grid barrier, teardown

template <int TN, int P = CO_P, bool SPLIT = false>
__device__ __forceinline__ CoCtx co_setup(uint8_t* smem_raw, void* bar, uint64_t wait_ns = 2 * WAIT_LIMIT_NS) {
  using C = CoCfg<TN, P, SPLIT>;
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  CoCtl* ctl = reinterpret_cast<CoCtl*>(smem + C::STAGES * C::STAGE_BYTES + (SPLIT ? CO_XBUF : 0));
  CoCtx x{ctl, smem, 0, 0, 0, 0, 0, Bars(), GridBarrier(static_cast<GridBarWords*>(bar), &ctl->abort, wait_ns)};
  x.smem_base = smem_u32(x.smem);
  x.br.full0 = smem_u32(&x.ctl->bars[0]);
  x.br.empty0 = smem_u32(&x.ctl->bars[C::STAGES]);
  x.br.tfull0 = smem_u32(&x.ctl->bars[2 * C::STAGES]);
  x.br.tempty0 = smem_u32(&x.ctl->bars[2 * C::STAGES + C::NBUF]);
  x.br.drain = smem_u32(&x.ctl->bars[2 * C::STAGES + 2 * C::NBUF]);
  x.xfull = smem_u32(&x.ctl->bars[2 * C::STAGES + 2 * C::NBUF + 1]);
  x.xbuf = x.smem_base + C::STAGES * C::STAGE_BYTES;
  x.warp = threadIdx.x >> 5;
  x.lane = threadIdx.x & 31;
  x.abort_flag = reinterpret_cast<volatile int*>(&x.ctl->abort);
  if (threadIdx.x == 0) {
    for (int s = 0; s < C::STAGES; ++s) {
      mbar_init(x.br.full0 + 8 * s, 1);
      mbar_init(x.br.empty0 + 8 * s, 1);
    }
    for (int b = 0; b < C::NBUF; ++b) {
      mbar_init(x.br.tfull0 + 8 * b, 1);
      mbar_init(x.br.tempty0 + 8 * b, EPI_WARPS);
    }
    mbar_init(x.br.drain, 1);
    mbar_init(x.xfull, EPI_WARPS);
    x.ctl->abort = 0;
    x.ctl->status = ST_RUNNING;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (x.warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&x.ctl->tmem)),
                 "r"(C::TCOLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  if (SPLIT) cluster_sync_all();   // the cluster's barriers are initialised before anyone arrives on them
  tc_fence_after();
  x.tmem = *reinterpret_cast<volatile uint32_t*>(&x.ctl->tmem);
  return x;
}

// Orders what the last grid barrier made visible to this thread before the copies (the async proxy) that it
// issues from here on.
__device__ __forceinline__ void co_fence_proxy() { asm volatile("fence.proxy.async.global;" ::: "memory"); }

__device__ __forceinline__ bool co_grid_sync(CoCtx& x) { return x.bar.sync(); }

// Leaves the kernel: every thread of the block, after its last product. Reports an expired wait.
template <int TN, bool SPLIT = false>
__device__ __forceinline__ void co_teardown(CoCtx& x, DevState* st, int* err_word = nullptr) {
  if (x.warp == 1) {   // every MMA issued has completed before TMEM is released; a commit covers its own thread's
    if (elect_one()) tc_commit(x.br.drain);   // the lane that issued them (co_mma)
    __syncwarp();
    mbar_drain(x.br.drain, 0);
  }
  tc_fence_before();
  __syncthreads();
  if (SPLIT) cluster_sync_all();   // no block leaves while another may still write into its exchange buffer
  if (threadIdx.x == 0 && *x.abort_flag) {
    if (err_word) atomicOr(err_word, 1);
    if (st) {
      atomicOr(&st->err_flags, 1u);
      st->status = ST_TIMEOUT;
    }
  }
  x.bar.leave();
  if (x.warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(x.tmem), "r"(CoCfg<TN>::TCOLS)
                 : "memory");
  }
}

// ------------------------------------------------------------------ the roles of one product
//
// All in line, so that what they carry stays in registers: the grid barrier's acquire empties L1, and a
// context kept in local memory for calls was read back from L2 at the start of every product.

// SYM: B is symmetric and only its upper triangle is stored.
template <int TN, int P, bool A_MN, bool SYM, class Src>
__device__ __forceinline__ void co_producer(const CoCtx& x, CoPipe& pp, Src src, int withhold) {
  using C = CoCfg<TN, P, Src::SPLIT>;
  if (withhold) return;   // test hook: no copies are issued, the consumers' bounded waits expire
  co_fence_proxy();
  int stage = pp.stage;
  uint32_t phase = pp.phase;
  bool ok = true;
  uint32_t armed = 0, armed_phase = 0;
  CoTile c;
  while (ok && src.next(c)) {
    const int m0 = c.bi * BM, n0 = c.bj * TN, K = c.K;
    const int km = Src::BKM ? 0 : SYM ? co_mirror_from<TN>(n0) : 0x7fffffff;
    const CUtensorMap *ma = c.ma, *mb = c.mb, *mbt = c.mbt;
    for (int k0 = c.kbeg; k0 < K; k0 += C::BKS) {
      if (!mbar_wait(x.br.empty0 + 8 * stage, phase ^ 1u, x.abort_flag)) { ok = false; break; }
      const uint32_t fb = x.br.full0 + 8 * stage;
      mbar_expect_tx(fb, C::SUB == 2 && k0 + BK < K ? 2 * C::KB_BYTES : C::KB_BYTES);
      armed |= 1u << stage;
      armed_phase = (armed_phase & ~(1u << stage)) | (phase << stage);
#pragma unroll
      for (int s = 0; s < C::SUB; ++s) {
        const int k = k0 + s * BK;
        if (s > 0 && k >= K) break;
        const uint32_t a_dst = x.smem_base + stage * C::STAGE_BYTES + s * C::KB_BYTES, b_dst = a_dst + C::A_BYTES;
        if (A_MN) {
#pragma unroll
          for (int cc = 0; cc < BM / 64; ++cc) tma_load_3d(a_dst + cc * P * MN_CHUNK, ma, fb, m0 + 64 * cc, k, 0);
        } else {
          tma_load_3d(a_dst, ma, fb, k, m0, 0);
        }
        if (k < km) {
#pragma unroll
          for (int cc = 0; cc < TN / 64; ++cc) tma_load_3d(b_dst + cc * P * MN_CHUNK, mb, fb, n0 + 64 * cc, k, 0);
        } else {
          tma_load_3d(b_dst, mbt, fb, k, n0, 0);
        }
      }
      if (++stage == C::STAGES) { stage = 0; phase ^= 1u; }
      if (k0 == c.kbeg) src.poke(true);
    }
  }
  pp.stage = stage;
  pp.phase = phase;
  // every copy this thread started lands before the block can leave (another role may have aborted)
  for (int s = 0; s < C::STAGES; ++s)
    if (armed & (1u << s)) mbar_drain(x.br.full0 + 8 * s, (armed_phase >> s) & 1u);
}

// The whole warp runs the loop and one elected lane issues, a stage's waits between the halves of the stage
// before it (see role_mma; with four slice buffers the wait for one is rarely a real one).
template <int TN, int P, bool A_MN, bool SYM, class Src>
__device__ __forceinline__ void co_mma(const CoCtx& x, CoPipe& pp, Src src) {
  using C = CoCfg<TN, P, Src::SPLIT>;
  const bool issuer = elect_one();
  const uint64_t a0 = A_MN ? smem_desc(x.smem_base, P * MN_CHUNK, 1024, 2)
                           : smem_desc(x.smem_base, 16, KM_SBO, KM_SWZ);
  const uint64_t bm0 = smem_desc(x.smem_base + C::A_BYTES, P * MN_CHUNK, 1024, 2);
  const uint64_t bk0 = smem_desc(x.smem_base + C::A_BYTES, 16, KM_SBO, KM_SWZ);
  const Bars br = x.br;
  volatile int* abort_flag = x.abort_flag;
  const uint32_t tmem = x.tmem;
  int stage = pp.stage, buf = pp.buf;
  uint32_t phase = pp.phase, buf_phase = pp.buf_phase;
  bool ok = true;
  CoTile c;
  while (ok && src.next(c)) {
    const int K = c.K, kin_last = Src::TABLE ? c.slice / C::SUB - 1 : C::SLICE - 1;
    const int km = Src::BKM ? 0 : SYM ? co_mirror_from<TN>(c.bj * TN) : 0x7fffffff;
    int kin = 0;
    if (Src::SPLIT && c.kbeg >= K) continue;   // no part of K for this block
    ok = mbar_wait_warp(br.tempty0 + 8 * buf, buf_phase ^ 1u, abort_flag) &&
         mbar_wait_warp(br.full0 + 8 * stage, phase, abort_flag);
    for (int k0 = c.kbeg; k0 < K && ok; k0 += C::BKS) {
      const bool last = kin == kin_last || k0 + C::BKS >= K;
      const uint32_t d = tmem + (uint32_t)(buf * TN), acc = kin == 0 ? 0u : 1u;
      const uint64_t so = (uint64_t)((stage * C::STAGE_BYTES) >> 4);
      const int this_stage = stage, this_buf = buf;
      const bool two = C::SUB == 2 && k0 + BK < K;   // the stage's second k-block exists
      tc_fence_after();
      if (issuer) {
        // km and the stages are multiples of 64: a stage lies on one side of it
        if (k0 < km) {
          issue_half<P, A_MN, true, P, TN, 1, 0>(d, a0 + so, bm0 + so, acc);
          if (two) issue_half<P, A_MN, true, P, TN, 1, 1>(d, a0 + so, bm0 + so, 1u);
        } else {
          issue_half<P, A_MN, false, P, TN, 1, 0>(d, a0 + so, bk0 + so, acc);
          if (two) issue_half<P, A_MN, false, P, TN, 1, 1>(d, a0 + so, bk0 + so, 1u);
        }
      }
      if (k0 == c.kbeg) src.poke(false);
      if (++stage == C::STAGES) { stage = 0; phase ^= 1u; }
      if (last) {
        if (++buf == C::NBUF) { buf = 0; buf_phase ^= 1u; }
        kin = 0;
      } else {
        ++kin;
      }
      if (k0 + C::BKS < K)
        ok = mbar_wait_warp(br.full0 + 8 * stage, phase, abort_flag) &&
             (!last || mbar_wait_warp(br.tempty0 + 8 * buf, buf_phase ^ 1u, abort_flag));
      if (issuer) {
        const uint64_t so2 = so + (two ? (uint64_t)(C::KB_BYTES >> 4) : 0u);
        if (k0 < km) {
          if (two) issue_half<P, A_MN, true, P, TN, 1, 0>(d, a0 + so2, bm0 + so2, 1u);
          issue_half<P, A_MN, true, P, TN, 1, 1>(d, a0 + so2, bm0 + so2, 1u);
        } else {
          if (two) issue_half<P, A_MN, false, P, TN, 1, 0>(d, a0 + so2, bk0 + so2, 1u);
          issue_half<P, A_MN, false, P, TN, 1, 1>(d, a0 + so2, bk0 + so2, 1u);
        }
        tc_commit(br.empty0 + 8 * this_stage);
        if (last) tc_commit(br.tfull0 + 8 * this_buf);
      }
      __syncwarp();
    }
  }
  pp.stage = stage;
  pp.phase = phase;
  pp.buf = buf;
  pp.buf_phase = buf_phase;
}

// What the output step of a product needs.
struct CoEpi {
  int M, N;
  const uint16_t* x;         // NS, NS_STEP: three planes of X_k; CLENSHAW: of Z
  int64_t ldx, xs;
  uint16_t* out;             // planes (every kind but STORE)
  int64_t ldo, os;
  float* C;                  // STORE
  int64_t ldc;
  float c1, c3;              // NS: c1 X + c3 acc; CLENSHAW: c3 acc + c1 Z + diag I
  float diag;
  double* part;              // GRAM, NORM: per epilogue warp of every block; NS_STEP: two each
  double* tile_part;         // GRAM from a table: this tile's EPI_WARPS sums
};

// 8 consecutive entries of a row of C = c3 v + c1 C (C is not read for c1 = 0), `n` of them existing.
__device__ __forceinline__ void co_gemm_store8(float* c, int n, bool vec, float c1, float c3, const float* v) {
  if (vec && n >= 8) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      float4 o = make_float4(c3 * v[4 * h], c3 * v[4 * h + 1], c3 * v[4 * h + 2], c3 * v[4 * h + 3]);
      if (c1 != 0.0f) {
        const float4 x = reinterpret_cast<const float4*>(c)[h];
        o = make_float4(fmaf(c1, x.x, o.x), fmaf(c1, x.y, o.y), fmaf(c1, x.z, o.z), fmaf(c1, x.w, o.w));
      }
      reinterpret_cast<float4*>(c)[h] = o;
    }
  } else {
#pragma unroll
    for (int j = 0; j < 8; ++j)
      if (j < n) c[j] = c1 != 0.0f ? fmaf(c1, c[j], c3 * v[j]) : c3 * v[j];
  }
}

// Sums over each warp's tiles, in float64 from a warp's 32 row chunks on, go to e.part: GRAM ||G - I||_F^2,
// NS_STEP ||X' - X||^2 and ||X'||^2, NORM ||C||_F^2.
template <int TN, int EPI, class Src>
__device__ __forceinline__ void co_epilogue(const CoCtx& x, CoPipe& pp, Src src) {
  using C = CoCfg<TN>;
  constexpr int CW = C::CW, NCH = CW / 32;
  constexpr bool NS = EPI == TC_EPI_NS || EPI == TC_EPI_NS_STEP, STEP = EPI == TC_EPI_NS_STEP;
  constexpr bool READS_X = NS || EPI == TC_EPI_CLENSHAW;
  const int q = x.warp & 3, half = (x.warp - 2) >> 2, lane = x.lane, lq = lane & 3;
  const uint32_t t_lane = x.tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(half * CW);
  int buf = pp.buf;
  uint32_t buf_phase = pp.buf_phase;
  double sum0 = 0.0, sum1 = 0.0, norm = 0.0;   // norm: this lane's
  bool ok = true;
  CoTile ti;
  while (ok && src.next(ti)) {
    const CoEpi& e = src.epi(ti);
    const int bi = ti.bi, bj = ti.bj, nslices = (ti.K - ti.kbeg + ti.slice * BK - 1) / (ti.slice * BK);
    const int r = bi * BM + q * 32 + lane, r4 = r - lq;
    const int cb = bj * TN + half * CW;
    unsigned rows4 = 0;
#pragma unroll
    for (int i = 0; i < 4; ++i) rows4 |= (r4 + i < e.M) ? (1u << i) : 0u;
    // one chunk per warp: X_k's planes are read while the products run
    Planes8 pre[4];
    if (READS_X && NCH == 1 && cb < e.N) {
      const uint16_t* xr = e.x + r4 * e.ldx + cb + 8 * lq;
#pragma unroll
      for (int i = 0; i < 4; ++i) pre[i] = load_planes8(xr + i * e.ldx, e.xs, (rows4 & (1u << i)) != 0);
    }
    float acc[CW];
#pragma unroll
    for (int i = 0; i < CW; ++i) acc[i] = 0.0f;
    for (int sl = 0; sl < nslices; ++sl) {
      if (!mbar_wait(x.br.tfull0 + 8 * buf, buf_phase, x.abort_flag)) { ok = false; break; }
      tc_fence_after();
#pragma unroll
      for (int c = 0; c < CW / 16; ++c) {
        float v[16];
        tmem_ld16(t_lane + (uint32_t)(buf * TN + c * 16), v);
        add16_packed(&acc[c * 16], v);   // round-to-nearest promotion
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(x.br.tempty0 + 8 * buf);
      if (++buf == C::NBUF) { buf = 0; buf_phase ^= 1u; }
      if (sl == 0) src.poke(false);
    }
    if (!__all_sync(0xffffffffu, ok)) { ok = false; break; }
    float d2 = 0.f, x2 = 0.f;
    float t[NCH] = {};   // GRAM: the chunks' residual terms
#pragma unroll
    for (int c = 0; c < NCH; ++c) {
      const int c0 = cb + 32 * c;
      float* v = &acc[32 * c];
      if (c0 >= e.N) continue;                       // the same for every lane of the warp
      if (EPI == TC_EPI_GRAM) {
        // residual terms: twice the squares above the diagonal, (g - 1)^2 on it (columns past N hold zeros)
        if (r < e.M && c0 + 31 >= r) {
          float s4[4] = {0.f, 0.f, 0.f, 0.f};
          if (c0 > r) {
#pragma unroll
            for (int j = 0; j < 32; ++j) s4[j & 3] = fmaf(v[j], v[j], s4[j & 3]);
#pragma unroll
            for (int j = 0; j < 4; ++j) s4[j] *= 2.0f;
          } else {
            const int d = r - c0;
#pragma unroll
            for (int j = 0; j < 32; ++j) {
              const float g = j == d ? v[j] - 1.0f : v[j], w = j < d ? 0.0f : j == d ? 1.0f : 2.0f;
              s4[j & 3] = fmaf(w * g, g, s4[j & 3]);
            }
          }
          t[c] = (s4[0] + s4[1]) + (s4[2] + s4[3]);
        }
      }
      if (EPI == CO_EPI_NORM) {   // twice the squares above the diagonal, the squares on it
        if (r < e.M && c0 + 31 >= r) {
          double on = 0.0, off = 0.0;
#pragma unroll
          for (int j = 0; j < 32; ++j) {
            const double g = (double)v[j];
            if (c0 + j > r) off = fma(g, g, off);
            else if (c0 + j == r) on = g * g;
          }
          norm += 2.0 * off + on;
        }
        continue;
      }
      if (EPI == CO_EPI_GEMM) {
        store_c32(e.C + (r - lane) * e.ldc + c0, e.ldc, e.M - (r - lane), lane < e.N - c0 ? 31 : -1, lane, e.c3, e.c1, v);
        continue;
      }
      quad_rows(v, lq);
      if (EPI == TC_EPI_GRAM || EPI == TC_EPI_PLANES) {
        // columns past N hold zeros (the operand maps stop at N) and land in the pitch's padding
        store_chunk(e.out + r4 * e.ldo + c0 + 8 * lq, e.ldo, e.os, 3, v, rows4);
      } else if (READS_X) {
        const uint16_t* xr = e.x + r4 * e.ldx + c0 + 8 * lq;
        uint16_t* pr = e.out + r4 * e.ldo + c0 + 8 * lq;
        Planes8 xv;
        if (NCH > 1) xv = load_planes8(xr, e.xs, (rows4 & 1u) != 0);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          float xo[8];
          if (NCH == 1) {
            sum_planes8(pre[i], xo);
          } else {
            sum_planes8(xv, xo);
            if (i < 3) xv = load_planes8(xr + (i + 1) * e.ldx, e.xs, (rows4 & (2u << i)) != 0);
          }
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            if (NS) {
              const float xn = fmaf(e.c1, xo[j], e.c3 * v[8 * i + j]);   // c3 = -0.5, -1: one rounding
              if (STEP) {
                d2 = fmaf(xn - xo[j], xn - xo[j], d2);
                x2 = fmaf(xn, xn, x2);
              }
              v[8 * i + j] = xn;
            } else {
              float o = fmaf(e.c3, v[8 * i + j], e.c1 * xo[j]);
              if (r4 + i == c0 + 8 * lq + j) o += e.diag;
              v[8 * i + j] = o;
            }
          }
          if (rows4 & (1u << i)) store_planes8(pr + i * e.ldo, e.os, 3, v + 8 * i);
        }
      } else {   // STORE: whole 16-byte groups up to a pitch that is a multiple of 4, else single entries
        float* cr = e.C + r4 * e.ldc + c0 + 8 * lq;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          if (!(rows4 & (1u << i))) continue;
          if (Src::TABLE && (e.ldc & 3)) {
#pragma unroll
            for (int j = 0; j < 8; ++j)
              if (c0 + 8 * lq + j < e.N) cr[i * e.ldc + j] = v[8 * i + j];
            continue;
          }
          if (c0 + 8 * lq < e.ldc)
            *reinterpret_cast<float4*>(cr + i * e.ldc) = make_float4(v[8 * i], v[8 * i + 1], v[8 * i + 2], v[8 * i + 3]);
          if (c0 + 8 * lq + 4 < e.ldc)
            *reinterpret_cast<float4*>(cr + i * e.ldc + 4) =
                make_float4(v[8 * i + 4], v[8 * i + 5], v[8 * i + 6], v[8 * i + 7]);
        }
      }
    }
    if (EPI == TC_EPI_GRAM) sum0 += warp_sum64<NCH>(t);
    if (Src::TABLE && EPI == TC_EPI_GRAM) {
      if (lane == 0) e.tile_part[x.warp - 2] = sum0;
      sum0 = 0.0;
    }
    if (STEP) {
      sum0 += warp_sum64(d2);
      sum1 += warp_sum64(x2);
    }
  }
  pp.buf = buf;
  pp.buf_phase = buf_phase;
  if (EPI == CO_EPI_NORM) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) norm += __shfl_xor_sync(0xffffffffu, norm, o);
    if (lane == 0) __stcg(src.epi(ti).part + blockIdx.x * EPI_WARPS + x.warp - 2, norm);
  }
  if (!Src::TABLE && (EPI == TC_EPI_GRAM || STEP) && lane == 0) {
    double* dst = src.epi(ti).part + (STEP ? 2 : 1) * (blockIdx.x * EPI_WARPS + x.warp - 2);
    __stcg(dst, sum0);
    if (STEP) __stcg(dst + 1, sum1);
  }
}

// mbar_wait on a barrier that other blocks of the cluster arrive on after writing into this block's shared
// memory.
__device__ __noinline__ bool mbar_wait_cluster(uint32_t bar, uint32_t parity, volatile int* abort_flag) {
  const uint64_t t0 = gtime();
  for (uint32_t i = 1;; ++i) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    if (ok) return true;
    if ((i & 63u) == 0) {
      if (*abort_flag) return false;
      if (gtime() - t0 > WAIT_LIMIT_NS) {
        *abort_flag = 1;
        return false;
      }
    }
  }
}

// The epilogue of a product whose tiles are shared by S blocks (2 or 4), each with its part of K: every warp
// sends its 32 x 32 partial to the block that finishes those rows (rows 128 / S * sub of the tile belong to the
// group's block `sub`), which adds the S partials in a fixed order and runs the output step on 128 / S rows,
// 8 columns per lane. At most one tile per group.
template <int EPI, class Src>
__device__ __forceinline__ void co_epilogue_split(CoCtx& x, CoPipe& pp, Src src, int S) {
  using C = CoCfg<64, CO_P, true>;
  const int q = x.warp & 3, half = (x.warp - 2) >> 2, lane = x.lane, w = x.warp - 2;
  const int sub = (int)blockIdx.x % S, rows = 128 / S, units = 4 / S;
  constexpr bool NS = EPI == TC_EPI_NS || EPI == TC_EPI_NS_STEP, STEP = EPI == TC_EPI_NS_STEP;
  constexpr bool READS_X = NS || EPI == TC_EPI_CLENSHAW;
  CoTile ti;
  double sum0 = 0.0, sum1 = 0.0, norm = 0.0;   // norm: this lane's
  const bool have = src.next(ti);        // the same in every block of the group
  const CoEpi& e = src.epi(ti);
  if (have) {
    const int nslices = (ti.K - ti.kbeg + 63) / 64;
    const int col = ti.bj * 64 + 8 * (lane & 7);
    Planes8 pre[2];
    if (READS_X) {
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const int r = ti.bi * BM + sub * rows + (u * EPI_WARPS + w) * 4 + (lane >> 3);
        if (u < units) pre[u] = load_planes8(e.x + r * e.ldx + col, e.xs, r < e.M && col < e.N);
      }
    }
    float acc[32];
#pragma unroll
    for (int i = 0; i < 32; ++i) acc[i] = 0.0f;
    bool ok = true;
    for (int sl = 0; sl < nslices; ++sl) {
      if (!mbar_wait(x.br.tfull0 + 8 * pp.buf, pp.buf_phase, x.abort_flag)) { ok = false; break; }
      tc_fence_after();
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        float v[16];
        tmem_ld16(x.tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(pp.buf * 64 + half * 32 + c * 16), v);
        add16_packed(&acc[c * 16], v);   // round-to-nearest promotion
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(x.br.tempty0 + 8 * pp.buf);
      if (++pp.buf == C::NBUF) { pp.buf = 0; pp.buf_phase ^= 1u; }
    }
    if (__all_sync(0xffffffffu, ok)) {
      // to the block that finishes these rows: [sub][row][column] of its exchange buffer
      const uint32_t dst_rank = cluster_rank() - sub + q * S / 4;
      const uint32_t row = (uint32_t)((q % units) * 32 + lane);
      const uint32_t dst = mapa_shared(x.xbuf, dst_rank) + (((uint32_t)sub * rows + row) * CO_XLD + half * 32) * 4;
#pragma unroll
      for (int i = 0; i < 8; ++i)
        asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(dst + 16 * i), "f"(acc[4 * i]),
                     "f"(acc[4 * i + 1]), "f"(acc[4 * i + 2]), "f"(acc[4 * i + 3])
                     : "memory");
      __syncwarp();
      if (lane == 0) mbar_arrive_cluster(mapa_shared(x.xfull, dst_rank));
      ok = mbar_wait_cluster(x.xfull, x.xphase, x.abort_flag);
      x.xphase ^= 1u;
    }
    if (__all_sync(0xffffffffu, ok)) {
      const float* xb = reinterpret_cast<const float*>(x.smem + C::STAGES * C::STAGE_BYTES);
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        if (u >= units) break;
        const int lr = (u * EPI_WARPS + w) * 4 + (lane >> 3), r = ti.bi * BM + sub * rows + lr;
        float v[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) v[i] = 0.0f;
        for (int s = 0; s < S; ++s) {
          const float4* src4 = reinterpret_cast<const float4*>(xb + (s * rows + lr) * CO_XLD + 8 * (lane & 7));
          const float4 a = src4[0], b = src4[1];
          v[0] += a.x; v[1] += a.y; v[2] += a.z; v[3] += a.w;
          v[4] += b.x; v[5] += b.y; v[6] += b.z; v[7] += b.w;
        }
        float d2 = 0.0f, x2 = 0.0f;   // GRAM: the residual terms; STEP: the step's
        if (r >= e.M || col >= e.N) {   // past the matrix: nothing but zeros to the sums
        } else if (EPI == TC_EPI_GRAM) {
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            const int d = col + j - r;   // above the diagonal twice, on it (g - 1)^2 (columns past N hold zeros)
            const float g = d == 0 ? v[j] - 1.0f : v[j], wt = d < 0 ? 0.0f : d == 0 ? 1.0f : 2.0f;
            d2 = fmaf(wt * g, g, d2);
          }
          store_planes8(e.out + r * e.ldo + col, e.os, 3, v);
        } else if (READS_X) {
          float xo[8];
          sum_planes8(pre[u], xo);
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            if (NS) {
              v[j] = fmaf(e.c1, xo[j], e.c3 * v[j]);   // c3 = -0.5, -1: one rounding
              if (STEP) {
                d2 = fmaf(v[j] - xo[j], v[j] - xo[j], d2);
                x2 = fmaf(v[j], v[j], x2);
              }
            } else {
              v[j] = fmaf(e.c3, v[j], e.c1 * xo[j]);
              if (r == col + j) v[j] += e.diag;
            }
          }
          store_planes8(e.out + r * e.ldo + col, e.os, 3, v);
        } else if (EPI == TC_EPI_PLANES) {
          store_planes8(e.out + r * e.ldo + col, e.os, 3, v);
        } else if (EPI == CO_EPI_GEMM) {
          co_gemm_store8(e.C + r * e.ldc + col, e.N - col,
                         (reinterpret_cast<uintptr_t>(e.C) & 15u) == 0 && (e.ldc & 3) == 0, e.c1, e.c3, v);
        } else if (EPI == CO_EPI_NORM) {
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            const double g = (double)v[j], wt = col + j < r ? 0.0 : col + j == r ? 1.0 : 2.0;
            norm = fma(wt * g, g, norm);
          }
        } else {   // STORE (a pitch that is a multiple of 4)
          float* cr = e.C + r * e.ldc + col;
          if (col < e.ldc) *reinterpret_cast<float4*>(cr) = make_float4(v[0], v[1], v[2], v[3]);
          if (col + 4 < e.ldc) *reinterpret_cast<float4*>(cr + 4) = make_float4(v[4], v[5], v[6], v[7]);
        }
        if (EPI == TC_EPI_GRAM || STEP) sum0 += warp_sum64(d2);
        if (STEP) sum1 += warp_sum64(x2);
      }
    }
  }
  if (EPI == CO_EPI_NORM) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) norm += __shfl_xor_sync(0xffffffffu, norm, o);
    if (lane == 0) __stcg(e.part + blockIdx.x * EPI_WARPS + w, norm);
  }
  if ((EPI == TC_EPI_GRAM || STEP) && lane == 0) {
    double* dst = e.part + (STEP ? 2 : 1) * (blockIdx.x * EPI_WARPS + w);
    __stcg(dst, sum0);
    if (STEP) __stcg(dst + 1, sum1);
  }
}


// One product of a chain by all its roles, its tiles shared by S blocks.
template <int TN, bool SPLIT, bool A_MN, bool SYM, int EPI, bool BKM = false>
__device__ __forceinline__ void co_product(CoCtx& x, CoPipe& pipe, const CUtensorMap* ma, const CUtensorMap* mb,
                                           const CUtensorMap* mbt, CoTiles t, int K, const CoEpi& e, int S,
                                           int withhold) {
  using Src = CoChainSrc<TN, SPLIT, BKM>;
  if (x.warp == 0) {
    if (x.lane == 0) co_producer<TN, CO_P, A_MN, SYM>(x, pipe, Src(ma, mb, mbt, t, K, nullptr, S), withhold);
  } else if (x.warp == 1) {
    co_mma<TN, CO_P, A_MN, SYM>(x, pipe, Src(nullptr, nullptr, nullptr, t, K, nullptr, S));
  } else if (x.warp < CO_CTL_WARP) {
    if constexpr (SPLIT) {
      if (S > 1) {
        co_epilogue_split<EPI>(x, pipe, Src(nullptr, nullptr, nullptr, t, K, &e, S), S);
        return;
      }
    }
    co_epilogue<TN, EPI>(x, pipe, Src(nullptr, nullptr, nullptr, t, K, &e));
  }
}

// Sum of n doubles in device memory in a fixed order, by one warp (every lane gets it). AHEAD loads in flight and
// their sums as a tree: at 512^2 the stop test adds 36 per lane, and one at a time they took longer than the
// products beside which it runs.
template <int AHEAD = 8>
__device__ __forceinline__ double co_warp_sum(const double* p, int n, int stride, int lane) {
  double v = 0.0;
  for (int i = lane; i < n; i += 32 * AHEAD) {
    double a[AHEAD];
#pragma unroll
    for (int j = 0; j < AHEAD; ++j) a[j] = i + 32 * j < n ? __ldcg(p + (size_t)(i + 32 * j) * stride) : 0.0;
#pragma unroll
    for (int o = AHEAD / 2; o > 0; o >>= 1)
#pragma unroll
      for (int j = 0; j < o; ++j) a[j] += a[j + o];
    v += a[0];
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Block sum of one double per thread (valid in thread 0).
__device__ __forceinline__ double co_block_sum(CoCtx& x, double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  __syncthreads();
  if (x.lane == 0) x.ctl->red[x.warp] = v;
  __syncthreads();
  double t = 0.0;
  if (threadIdx.x == 0)
    for (int w = 0; w < CO_WARPS; ++w) t += x.ctl->red[w];
  return t;
}

}  // namespace
}  // namespace polar
