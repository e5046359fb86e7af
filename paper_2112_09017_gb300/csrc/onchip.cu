// Batched small problems (n <= 128, m <= 256) solved entirely on one SM each: the
// whole Newton-Schulz loop of Sec. III.D (Eq. NewtonSchulz with the residual stop
// rule; Algorithm 1's preconditioning steps when asked) in one CTA per problem, with
// no global-memory traffic between iterations.
//
//   shared memory  the three BF16 planes of X_k, rows padded to 16 and columns to 128,
//                  in 64-column chunks of 128-byte rows with the 128-byte swizzle: the
//                  same bytes are the MN-major operands of the Gram (K = rows of X)
//                  and the K-major operand of the update (N = rows of X)
//   TMEM           two Gram accumulators (columns 0 and 128), the planes of G as the
//                  A operand of the update (two BF16 per 32-bit column, from column
//                  256), and the update accumulator (columns 0 .. m, once the Gram's
//                  have been read)
//   Gram           G = X^T X in 64-row slices into alternating accumulators, each
//                  promoted by the workers with round-to-nearest adds (the tensor-core
//                  accumulator itself truncates)
//   update         P^T = G X^T (G is symmetric): A = G from TMEM (M = 128 lanes = the
//                  columns of X), B = X, N = the rows of X; then
//                  X_{k+1}(r, i) = c1 X_k(r, i) + c3 P^T(i, r), split back into the
//                  planes in place
// Sixteen worker warps, four per TMEM lane quarter taking 16-wide chunks of columns or rows in turn, load X_0,
// promote accumulators, sum the residual, write G into TMEM and X back into shared memory; a warp of its own
// issues the MMAs once the workers have handed over their operands and decides (warp 0 allocates TMEM). Every
// mbarrier wait is bounded (about one second); on expiry the problem reports a timeout, the MMAs in flight
// drain and TMEM is freed.
#include <cuda.h>
#include <math.h>
#include <stdint.h>
#include <stdlib.h>

#include "device_util.cuh"
#include "internal.cuh"
#include "tc_ptx.cuh"

namespace polar {
namespace {

constexpr int OC_WARPS = 16;          // workers (12 and 8, with more registers each, measured 6 and 15 % slower)
constexpr int OC_SUB = OC_WARPS / 4;  // per TMEM lane quarter
static_assert(OC_WARPS == 16, "the stop test adds 16 sums");
constexpr int OC_GT = (128 / 16 + OC_SUB - 1) / OC_SUB;   // 16-wide chunks of G per worker, at most
constexpr int OC_WORKERS = OC_WARPS * 32;
constexpr int OC_THREADS = OC_WORKERS + 32;   // and one warp that issues the MMAs and decides
constexpr uint32_t OC_TMEM_COLS = 512;
constexpr uint32_t OC_G_COL = 256;          // first TMEM column of G's planes
constexpr int64_t OC_MAX_M = 256, OC_MAX_N = 128;

// Plane pairs (A plane, B plane) of the split product, smallest terms first:
// (1,1) (0,2) (2,0) (0,1) (1,0) (0,0); P planes use the last 6, 3 or 1 of them.
__host__ __device__ constexpr uint32_t oc_pass_a(int i) { return i == 0 ? 1u : i == 2 ? 2u : i == 4 ? 1u : 0u; }
__host__ __device__ constexpr uint32_t oc_pass_b(int i) { return i == 0 ? 1u : i == 1 ? 2u : i == 3 ? 1u : 0u; }

// The stop rule of the batched finalize on squares: with v = ||G - I||_F^2 = n r^2,
// r <= tol is v <= n tol^2 and r > s r_{k-2} is v > s^2 v_{k-2} (one FP64 compare each
// instead of a square root on the critical path).
struct OcRule {
  double v_tol, stag2, v_floor;
  int n_pre, max_iter;
  float pre_c1, pre_c3;
};

struct OcCtl {
  uint64_t full[2];    // tcgen05.commit -> all warps: accumulator ready
  uint64_t empty[2];   // the workers' warps have read a Gram accumulator that another slice takes
  uint64_t drain;
  int abort;           // a bounded wait expired
  int decision;        // 0: keep iterating, 1: stop, 2: abort
  OcRule dr;
  uint32_t tmem_base;
  int pad;
  float c1, c3;
  uint64_t red_s[OC_WARPS];   // the warps' sums
  int red_e[OC_WARPS];
};

__host__ __device__ __forceinline__ uint32_t oc_rows(int64_t m) { return (uint32_t)((m + 15) / 16 * 16); }

size_t oc_smem_bytes(int64_t max_m) { return (size_t)6 * oc_rows(max_m) * 128 + sizeof(OcCtl) + 1024; }
static_assert(6 * 256 * 128 + sizeof(OcCtl) + 1024 > 232448 / 2 && 6 * 256 * 128 + sizeof(OcCtl) + 1024 <= 232448,
              "one CTA per SM and within the opt-in shared memory of a CTA");

// Byte offset of element (r, c) in a plane: chunk c / 64, row r, 16-byte unit swizzled by r % 8.
__device__ __forceinline__ uint32_t oc_off(uint32_t r, uint32_t c, uint32_t ch) {
  return (c >> 6) * ch + r * 128u + ((((c & 63u) >> 3) ^ (r & 7u)) << 4) + ((c & 7u) << 1);
}

// Workers hand over to the issuing warp (X_k complete: 2, G's planes stored: 3) without waiting; the whole
// block meets once per step (4), so that no hand-over can overtake another, whatever a wait that expired skips.
template <int ID>
__device__ __forceinline__ void oc_arrive() { asm volatile("bar.arrive %0, %1;" ::"n"(ID), "n"(OC_THREADS) : "memory"); }
template <int ID>
__device__ __forceinline__ void oc_sync() { asm volatile("bar.sync %0, %1;" ::"n"(ID), "n"(OC_THREADS) : "memory"); }

// 8 consecutive 32-bit columns of this thread's TMEM lane (completed by tmem_st_wait).
__device__ __forceinline__ void oc_st8(uint32_t taddr, const uint32_t (&r)[8]) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"r"(taddr), "r"(r[0]),
               "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7])
               : "memory");
}

__device__ __forceinline__ void oc_fence_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// Instruction descriptor: D = F32, A = B = BF16, M = 128, N = n, majors as given.
__device__ __forceinline__ uint32_t oc_idesc(bool a_mn, bool b_mn, uint32_t n) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((a_mn ? 1u : 0u) << 15) | ((b_mn ? 1u : 0u) << 16) | ((n >> 3) << 17) |
         ((128u >> 4) << 24);
}

struct OcBars {
  uint32_t full, empty, drain;
};

// TMEM loads without the wait, and the wait tied to the loaded registers so that no use
// is scheduled before it (tcgen05.wait::ld covers every earlier load of the thread).
__device__ __forceinline__ void oc_ld16(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
}
__device__ __forceinline__ void oc_wait16(uint32_t (&r)[16]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
                 "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15])
               :
               : "memory");
}

// Two floats to BF16 with round-to-nearest-even: lo in the low half, hi in the high half.
__device__ __forceinline__ uint32_t oc_bf16x2(float lo, float hi) {
  uint32_t d;
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(d) : "f"(hi), "f"(lo));
  return d;
}
// The issuing warp: the Gram's 64-row slices of X_k into accumulators s % 2, the update P^T = G X^T into columns
// 0 .. mp, each completed on its full barrier, and the stop test between. Plane q of X is read through
// MN-major descriptors (chunk stride ch, 8-row groups of 1024 bytes) and K-major ones (rows of 128 bytes).
//
// A warp of its own, every lane of it in the loops and one elected lane issuing, keeps the descriptors in uniform
// registers; as thread 0 of a worker warp the MMAs took 85 to 115 cycles each to issue instead of about 55, and
// the stop test stood between the Gram and the update.
template <int P>
__device__ __noinline__ void oc_issue(const OcTask& tk, uint32_t xbase, uint32_t ch, uint32_t mp, uint32_t np,
                                      uint32_t tmem, OcBars br, volatile OcCtl* ctl, int lane, int withhold) {
  // descriptor high word: stride between 8-row groups 1024 bytes, version 1, 128-byte swizzle
  constexpr uint64_t HI = (uint64_t)((1024u >> 4) | (1u << 14) | (2u << 29)) << 32;
  volatile int* abort_flag = &ctl->abort;
  xbase = __shfl_sync(0xffffffffu, xbase, 0);
  ch = __shfl_sync(0xffffffffu, ch, 0);
  mp = __shfl_sync(0xffffffffu, mp, 0);
  np = __shfl_sync(0xffffffffu, np, 0);
  tmem = __shfl_sync(0xffffffffu, tmem, 0);
  const bool issuer = elect_one();
  const uint32_t idesc_g = oc_idesc(true, true, np), idesc_u = oc_idesc(false, false, mp);
  const uint32_t ks_g = mp / 16, ks_u = np / 16, nslices = (ks_g + 3) / 4;
  const uint64_t mn0 = HI | ((uint64_t)((ch >> 4) & 0x3FFFu) << 16) | ((xbase >> 4) & 0x3FFFu);   // plane 0, MN-major
  const uint64_t km0 = HI | (1u << 16) | ((xbase >> 4) & 0x3FFFu);                                // plane 0, K-major
  const uint64_t pl = (2 * ch) >> 4;   // from one plane to the next
  DevState* st = tk.st;
  const double inv_sqrt_n = st->inv_sqrt_n;
  double v_km1 = 0.0, v_stag = 0.0;    // the last sum of squares, and the one before it times stagnation^2
  uint32_t ephase = 0;                 // completions awaited on empty[0], empty[1] (one bit each)
  bool issued = false;
  for (int k = 0;; ++k) {
    oc_sync<2>();
    bool go = !withhold && __all_sync(0xffffffffu, !*abort_flag);
    for (uint32_t s = 0; s < nslices && go; ++s) {
      const uint32_t bsl = s & 1u, d = tmem + 128 * bsl, nkk = min(4u, ks_g - 4 * s);
      if (s >= 2) {
        go = mbar_wait_warp(br.empty + 8 * bsl, (ephase >> bsl) & 1u, abort_flag);
        ephase ^= 1u << bsl;
        if (!go) break;
      }
      tc_fence_after();
      issued = true;
      // small terms first, hi*hi last; neighbours share A (see mma_step of the tiled products)
      for (uint32_t kk = 0; kk < nkk; ++kk) {
        const uint64_t x = mn0 + (4 * s + kk) * 128;   // 16 rows of X: 2048 bytes
        const uint32_t first = kk == 0 ? 0u : 1u;
        if (issuer) {
          if (P == 3) {
            tc_mma_step<1>(d, x + pl, x + pl, idesc_g, first, 1);
            tc_mma_step<1>(d, x + pl, x, idesc_g, 1u, 3);
            tc_mma_step<1>(d, x + 2 * pl, x, idesc_g, 1u, 0);
            tc_mma_step<1>(d, x, x + 2 * pl, idesc_g, 1u, 1);
            tc_mma_step<1>(d, x, x + pl, idesc_g, 1u, 3);
          } else if (P == 2) {
            tc_mma(d, x + pl, x, idesc_g, first);
            tc_mma(d, x, x + pl, idesc_g, 1u);
          }
        }
        __syncwarp();
      }
      for (uint32_t kk = 0; kk < nkk; ++kk) {
        const uint64_t x = mn0 + (4 * s + kk) * 128;
        if (issuer) tc_mma(d, x, x, idesc_g, P == 1 && kk == 0 ? 0u : 1u);
        __syncwarp();
      }
      if (issuer) tc_commit(br.full + 8 * bsl);
      __syncwarp();
    }
    oc_sync<3>();
    // the update starts at once, whatever the stop rule will say (its result is not used after a stop)
    go = go && __all_sync(0xffffffffu, !*abort_flag);
    if (go) {
      tc_fence_after();
#pragma unroll
      for (int ps = P == 3 ? 0 : P == 2 ? 3 : 5; ps < 6; ++ps) {
        const uint64_t b0 = km0 + oc_pass_b(ps) * pl;
        const uint32_t a0 = tmem + OC_G_COL + 64 * oc_pass_a(ps);
        for (uint32_t kk = 0; kk < ks_u; ++kk) {   // 16 columns of X: 32 bytes within its 64-column chunk
          const uint64_t b = b0 + (kk >> 2) * (ch >> 4) + (kk & 3u) * 2;
          const uint32_t first = ps == (P == 3 ? 0 : P == 2 ? 3 : 5) && kk == 0 ? 0u : 1u;
          if (issuer) tc_mma_ts(tmem, a0 + 8 * kk, b, idesc_u, first);
          __syncwarp();
        }
      }
      if (issuer) {
        tc_commit(br.full);
        tc_commit(br.full + 8);
      }
      __syncwarp();
    }
    // the stop test: the warps' sums added up (every lane has the sum), v = n r^2 against squared thresholds
    const double v = warp_sum16({ctl->red_s[lane & 15], ctl->red_e[lane & 15]}, lane);
    int dec = 2, status = ST_TIMEOUT;
    if (go) {
      const bool testing = k >= ctl->dr.n_pre;
      if (!isfinite(v)) status = ST_NONFINITE;
      else if (testing && v <= ctl->dr.v_tol) status = ST_CONVERGED;
      else if (testing && k >= ctl->dr.n_pre + 2 && v > v_stag && v < ctl->dr.v_floor) status = ST_NOT_CONVERGED;
      else if (k >= ctl->dr.max_iter) status = ST_NOT_CONVERGED;
      else status = ST_RUNNING;
      dec = status == ST_RUNNING ? 0 : 1;
    }
    const float c1 = k < ctl->dr.n_pre ? ctl->dr.pre_c1 : 1.5f, c3 = k < ctl->dr.n_pre ? ctl->dr.pre_c3 : -0.5f;
    if (lane == 0) {
      ctl->c1 = c1;
      ctl->c3 = c3;
      ctl->decision = dec;
    }
    v_stag = ctl->dr.stag2 * v_km1;
    v_km1 = v;
    oc_sync<4>();
    if (lane == 0 && dec != 2) {
      // the record of step k, as the batched finalize keeps it
      const double r = sqrt(v) * inv_sqrt_n;
      if (k < POLAR_HIST) {
        st->res_hist[k] = r;
        st->planes_hist[k] = (unsigned char)P;
        st->hist_len = k + 1;
      }
      st->ring[k & 3] = r;
      st->iters = k;
      if (status != ST_RUNNING) st->status = status;
      else {
        st->upd_c1 = c1;
        st->upd_c3 = c3;
      }
    }
    if (dec != 0) break;
  }
  // everything issued has completed before the CTA frees TMEM
  if (issued) {
    if (issuer) tc_commit(br.drain);
    __syncwarp();
    mbar_drain(br.drain, 0);
  }
}

// The whole loop for one problem by the workers. The four warps of a TMEM lane quarter take 16-wide chunks in
// turn: chunk c of the Gram's columns and of the update's rows belongs to warp sub = c % 4 of the quarter.
template <int P>
__device__ __noinline__ void oc_solve(const OcTask& tk, uint8_t* xs, uint32_t ch, uint32_t mp, uint32_t np,
                                      uint32_t tmem, OcBars br, volatile OcCtl* ctl, int warp, int lane) {
  const int tid = warp * 32 + lane;
  const uint32_t sub = (uint32_t)warp >> 2;
  const uint32_t i = (uint32_t)((warp & 3) * 32 + lane);           // TMEM lane: a row of G, a column of X
  const uint32_t lane_addr = (uint32_t)((warp & 3) * 32) << 16;
  const int64_t m = tk.m, n = tk.n;
  volatile int* abort_flag = &ctl->abort;
  uint32_t use0 = 0, use1 = 0;                                     // completions awaited on full[0], full[1]
  const uint32_t nslices = (mp / 16 + 3) / 4;
  const uint32_t gch = np / 16, uch = mp / 16;                     // 16-wide chunks of G's columns, X's rows
  int k = 0;
  for (;; ++k) {
    // X_k complete in shared memory (and the last accumulator read)
    oc_fence_async();
    tc_fence_before();
    oc_arrive<2>();
    // ---- Gram: promote this warp's chunks (at most two) of every slice
    float g[OC_GT][16];
#pragma unroll
    for (int t = 0; t < OC_GT; ++t)
#pragma unroll
      for (int e = 0; e < 16; ++e) g[t][e] = 0.0f;
    for (uint32_t s = 0; s < nslices; ++s) {
      const uint32_t b = s & 1u;
      bool ok = !*abort_flag && mbar_wait(br.full + 8 * b, (b ? use1 : use0) & 1u, abort_flag);
      ok = __all_sync(0xffffffffu, ok);
      if (ok) {
        tc_fence_after();
#pragma unroll
        for (int t = 0; t < OC_GT; ++t) {
          if (sub + OC_SUB * t < gch) {
            float f[16];
            tmem_ld16(tmem + lane_addr + 128u * b + 16u * (sub + OC_SUB * t), f);
            add16_packed(g[t], f);
          }
        }
      }
      if (b) ++use1; else ++use0;
      if (s + 2 < nslices) {   // this accumulator takes slice s + 2
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(br.empty + 8 * b);
      }
    }
    // ---- residual ||G - I||_F^2 over the n x n block (float per thread, at most 32 terms;
    // FP64 is slow on this part), and G's planes into TMEM as the update's A operand (two
    // BF16 per column, low half first) whatever the decision
    float part32 = 0.0f;
    bool stored = false;
#pragma unroll
    for (int t = 0; t < OC_GT; ++t) {
      const uint32_t c = sub + OC_SUB * t;
      if (c < gch) {
#pragma unroll
        for (int e = 0; e < 16; ++e) {
          const int64_t jj = 16 * c + e;
          if (jj >= n) g[t][e] = 0.0f;   // columns beyond n
          if ((int64_t)i < n && jj < n) {
            const float d = g[t][e] - ((int64_t)i == jj ? 1.0f : 0.0f);
            part32 = fmaf(d, d, part32);
          }
        }
#pragma unroll
        for (int qp = 0; qp < P; ++qp) {
          uint32_t w[8];
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            w[j] = oc_bf16x2(g[t][2 * j], g[t][2 * j + 1]);
            const float2 rest = sub_x2(make_float2(g[t][2 * j], g[t][2 * j + 1]), bf16_pair(w[j]));
            g[t][2 * j] = rest.x;
            g[t][2 * j + 1] = rest.y;
          }
          oc_st8(tmem + lane_addr + OC_G_COL + 64u * qp + 8u * c, w);
        }
        stored = true;
      }
    }
    if (stored) tmem_st_wait();
    const Fixed part = warp_fixed<1>({part32});
    if (lane == 0) {
      ctl->red_s[warp] = part.s;
      ctl->red_e[warp] = part.e;
    }
    tc_fence_before();
    oc_arrive<3>();
    oc_sync<4>();   // the decision
    if (ctl->decision != 0) break;
    // ---- update: P^T = G X^T, then X_{k+1} = c1 X_k + c3 P in place, this warp's 16-row
    // chunks one at a time from TMEM with the next in flight
    bool ok = !*abort_flag && mbar_wait(br.full, use0 & 1u, abort_flag) && mbar_wait(br.full + 8, use1 & 1u, abort_flag);
    ok = __all_sync(0xffffffffu, ok);
    ++use0;
    ++use1;
    if (ok && sub < uch) {
      tc_fence_after();
      const float c1 = ctl->c1, c3 = ctl->c3;
      // Lanes 2j and 2j + 1 share columns 2j and 2j + 1: the even lane takes rows 0..3 and 8..11 of a chunk of
      // 16, the odd lane rows 4..7 and 12..15, both columns of each, so that X moves as 32-bit words and the
      // arithmetic as FP32 pairs (rows four apart lie in different halves of the swizzled 128 bytes: no bank
      // conflicts). Columns past n are zeros in X and in the product and stay so.
      const uint32_t odd = i & 1u, i2 = i & ~1u;
      const bool active = (int64_t)i2 < n;
      const uint32_t cb = (i2 >> 6) * ch + ((i2 & 7u) << 1), unit = (i2 & 63u) >> 3;
      uint32_t cur[16], nxt[16];
      oc_ld16(tmem + lane_addr + 16u * sub, cur);
      oc_wait16(cur);
      for (uint32_t c = sub; c < uch; c += OC_SUB) {
        const bool more = c + OC_SUB < uch;
        if (more) oc_ld16(tmem + lane_addr + 16u * (c + OC_SUB), nxt);
        const uint32_t rb = 16u * c;
#pragma unroll
        for (int t = 0; t < 8; ++t) {
          const int re = (t & 3) + 8 * (t >> 2), ro = re + 4;   // the even and the odd lane's row
          const uint32_t got = __shfl_xor_sync(0xffffffffu, odd ? cur[re] : cur[ro], 1);
          const float2 pr = make_float2(__uint_as_float(odd ? got : cur[re]), __uint_as_float(odd ? cur[ro] : got));
          const uint32_t row = rb + (uint32_t)(odd ? ro : re);
          if (active && row < (uint32_t)m) {
            uint8_t* a = xs + row * 128u + ((unit ^ (row & 7u)) << 4) + cb;
            const uint32_t h = *reinterpret_cast<uint32_t*>(a), md = *reinterpret_cast<uint32_t*>(a + 2 * ch),
                           l = *reinterpret_cast<uint32_t*>(a + 4 * ch);
            const float2 x = add_x2(add_x2(bf16_pair(h), bf16_pair(md)), bf16_pair(l));
            // c1 X + (c3 P), the product with c3 = -0.5 exact
            float2 r = fma_x2(make_float2(c1, c1), x, make_float2(c3 * pr.x, c3 * pr.y));
#pragma unroll
            for (int q = 0; q < 3; ++q) {
              const uint32_t w = oc_bf16x2(r.x, r.y);
              r = sub_x2(r, bf16_pair(w));
              *reinterpret_cast<uint32_t*>(a + 2 * q * ch) = w;
            }
          }
        }
        if (more) {
          oc_wait16(nxt);
#pragma unroll
          for (int e = 0; e < 16; ++e) cur[e] = nxt[e];
        }
      }
    }
  }
  if (ctl->decision != 1) return;
  // ---- the final iterate's planes to global memory, where the H product and U read them
  uint16_t* dst = tk.xp[k & 1];
  for (uint32_t u = (uint32_t)tid; u < 3u * (uint32_t)m * 16u; u += OC_WORKERS) {
    const uint32_t q = u / ((uint32_t)m * 16u), rem = u % ((uint32_t)m * 16u), r = rem >> 4, c8 = (rem & 15u) * 8u;
    if (c8 >= n) continue;
    const uint4 v = *reinterpret_cast<const uint4*>(xs + 2 * q * ch + oc_off(r, c8, ch));
    uint16_t* d = dst + q * tk.xps + r * tk.ldp + c8;
    if (c8 + 8 <= n) {
      *reinterpret_cast<uint4*>(d) = v;
    } else {
      const uint16_t* e = reinterpret_cast<const uint16_t*>(&v);
      for (uint32_t t = 0; c8 + t < n; ++t) d[t] = e[t];
    }
  }
}

template <int P>
__global__ void __launch_bounds__(OC_THREADS, 1)
    onchip_ns_kernel(const OcTask* __restrict__ tasks, StopRule rule, const double* tol_dev, int* err_word,
                     int withhold) {
  extern __shared__ uint8_t oc_smem[];
  const OcTask tk = tasks[blockIdx.x];
  // nothing in this kernel has written the status yet, so every thread sees the same value
  if (tk.st->status != ST_RUNNING) return;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t raw = smem_u32(oc_smem);
  const uint32_t xbase = (raw + 1023u) & ~1023u;     // swizzle atoms need 1024-byte alignment
  uint8_t* xs = oc_smem + (xbase - raw);
  const uint32_t mp = oc_rows(tk.m), np = oc_rows(tk.n), ch = mp * 128u;
  volatile OcCtl* ctl = reinterpret_cast<volatile OcCtl*>(xs + 6 * ch);
  OcBars br;
  br.full = smem_u32((const void*)&ctl->full[0]);
  br.empty = smem_u32((const void*)&ctl->empty[0]);
  br.drain = smem_u32((const void*)&ctl->drain);
  if (threadIdx.x == 0) {
    mbar_init(br.full, 1);
    mbar_init(br.full + 8, 1);
    mbar_init(br.empty, OC_WARPS);
    mbar_init(br.empty + 8, OC_WARPS);
    mbar_init(br.drain, 1);
    ctl->abort = 0;
    ctl->decision = 0;
    const double tol = (tol_dev && *tol_dev > 0) ? *tol_dev : rule.tol;
    const double nn = (double)tk.n;
    ctl->dr.v_tol = tol * tol * nn;
    ctl->dr.stag2 = rule.stagnation * rule.stagnation;
    ctl->dr.v_floor = rule.stag_floor * rule.stag_floor * nn;
    ctl->dr.n_pre = rule.n_pre;
    ctl->dr.max_iter = rule.max_iter;
    ctl->dr.pre_c1 = (float)rule.pre_a;
    ctl->dr.pre_c3 = (float)(-(4.0 / 27.0) * rule.pre_a * rule.pre_a * rule.pre_a);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    oc_fence_async();
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32((const void*)&ctl->tmem_base)),
                 "n"(OC_TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  // X_0's three planes into shared memory, zero beyond m x n
  {
    const int64_t m = tk.m, n = tk.n;
    for (uint32_t u = threadIdx.x; u < 3u * mp * 16u; u += OC_THREADS) {
      const uint32_t q = u / (mp * 16u), rem = u % (mp * 16u), r = rem >> 4, c8 = (rem & 15u) * 8u;
      uint4 v = make_uint4(0u, 0u, 0u, 0u);
      if (r < m && c8 < n) {
        const uint16_t* src = tk.x0 + q * tk.xps + r * tk.ldp + c8;
        if (c8 + 8 <= n) {
          v = *reinterpret_cast<const uint4*>(src);
        } else {
          uint16_t* e = reinterpret_cast<uint16_t*>(&v);
          for (uint32_t t = 0; c8 + t < n; ++t) e[t] = src[t];
        }
      }
      *reinterpret_cast<uint4*>(xs + 2 * q * ch + oc_off(r, c8, ch)) = v;
    }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = ctl->tmem_base;
  if (warp < OC_WARPS) oc_solve<P>(tk, xs, ch, mp, np, tmem, br, ctl, warp, lane);
  else oc_issue<P>(tk, xbase, ch, mp, np, tmem, br, ctl, lane, withhold);
  tc_fence_before();
  __syncthreads();
  if (threadIdx.x == 0 && ctl->decision == 2) {
    atomicOr(&tk.st->err_flags, 1u);
    tk.st->status = ST_TIMEOUT;
    if (err_word) atomicOr(err_word, 1);
  }
  if (warp == 0) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "n"(OC_TMEM_COLS) : "memory");
  }
}

template <int P>
cudaError_t launch_p(const OcTask* tasks, int ntasks, const StopRule& rule, const double* tol_dev, int* err_word,
                     int withhold, cudaStream_t s) {
  // sized for the largest problem whatever the batch holds: more than half an SM's shared
  // memory keeps one CTA per SM, so no CTA waits for another's 512 TMEM columns
  const size_t smem = oc_smem_bytes(OC_MAX_M);
  auto k = onchip_ns_kernel<P>;
  cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  k<<<ntasks, OC_THREADS, smem, s>>>(tasks, rule, tol_dev, err_word, withhold);
  return cudaGetLastError();
}

}  // namespace

bool onchip_fits(int64_t m, int64_t n) { return n >= 1 && m >= n && m <= OC_MAX_M && n <= OC_MAX_N; }

// Test hook for the bounded waits of this kernel: with POLAR_TEST_WITHHOLD_MMA=1 in the
// environment the MMA thread issues nothing, so the workers' waits expire after about
// one second and the problems report a timeout.
int onchip_withhold() {
  const char* e = getenv("POLAR_TEST_WITHHOLD_MMA");
  return (e && e[0] == '1') ? 1 : 0;
}

cudaError_t launch_onchip_ns(const OcTask* tasks, int ntasks, const StopRule& rule, const double* tol_dev,
                             int* err_word, int P, cudaStream_t s) {
  if (ntasks <= 0) return cudaSuccess;
  const int withhold = onchip_withhold();
  switch (P) {
    case 1: return launch_p<1>(tasks, ntasks, rule, tol_dev, err_word, withhold, s);
    case 2: return launch_p<2>(tasks, ntasks, rule, tol_dev, err_word, withhold, s);
    case 3: return launch_p<3>(tasks, ntasks, rule, tol_dev, err_word, withhold, s);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace polar
