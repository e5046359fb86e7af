// Plain-form float32 products in 32 x 32 tiles: one tile of C = op(A) op(B) per pass of a 512-thread block.
//
// For products with fewer 128 x 128 tiles than SMs the large SIMT kernel leaves most of the chip idle and
// walks K alone: a 300 x 200 Gram was three blocks of 45 us. Here a tile is 1/16 of that, and the block's
// eight groups of 64 threads share its K: each chunk of 64 is copied asynchronously (three in flight) and
// group g sums its k = 8 g .. 8 g + 7 into a fresh 4 x 4 register tile per thread before adding it to the
// running one (blocked summation); the groups' tiles are added at the end, in a fixed order.
#pragma once

#include "internal.cuh"

namespace polar {
namespace {

constexpr int SS_T = 32;                 // tile rows and columns
constexpr int SS_KC = 64;                // K of a chunk
constexpr int SS_THREADS = 512;
constexpr int SS_GROUPS = SS_THREADS / 64;
constexpr int SS_STAGES = 3;
constexpr int SS_LDM = SS_T + 4;         // floats per k-row of an MN-major chunk [64][36]
constexpr int SS_LDK = SS_KC + 4;        // floats per row of a K-major chunk [32][68]
constexpr int SS_OP = SS_KC * SS_LDM;    // floats kept for either (the K-major form takes 32 * 68)
static_assert(SS_T * SS_LDK <= SS_OP, "one buffer holds either form of a chunk");

struct SsSmem {
  float op[SS_STAGES][2][SS_OP];
  float red[SS_GROUPS][SS_T][SS_T + 1];
};

struct SsOperand {
  const float* p;
  int64_t ld;
  int mn;       // extent along M or N
  bool vec;     // 16-byte aligned rows
};

__device__ __forceinline__ void ss_cp16(float* dst, const float* src, int bytes) {
  const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void ss_cp4(float* dst, const float* src, int bytes) {
  const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(d), "l"(src), "r"(bytes) : "memory");
}

// This thread's 16 bytes of a chunk: 4 entries along the operand's contiguous direction, zeros outside.
template <bool KMAJOR>
__device__ __forceinline__ void ss_copy(float* dst, const SsOperand& o, int mn0, int k0, int K) {
  const int t = threadIdx.x;
  int row, col, lim;                     // position in the stored chunk; entries that exist from there
  int64_t off;
  bool row_ok;
  if (KMAJOR) {
    row = t >> 4;
    col = (t & 15) * 4;
    row_ok = mn0 + row < o.mn;
    off = (int64_t)(mn0 + row) * o.ld + k0 + col;
    lim = K - (k0 + col);
    dst += row * SS_LDK + col;
  } else {
    row = t >> 3;
    col = (t & 7) * 4;
    row_ok = k0 + row < K;
    off = (int64_t)(k0 + row) * o.ld + mn0 + col;
    lim = o.mn - (mn0 + col);
    dst += row * SS_LDM + col;
  }
  if (!row_ok || lim < 0) lim = 0;
  if (lim > 4) lim = 4;
  const float* src = lim > 0 ? o.p + off : o.p;   // a zero-byte copy reads nothing, from a valid address
  if (o.vec) {
    ss_cp16(dst, src, 4 * lim);
  } else {
#pragma unroll
    for (int j = 0; j < 4; ++j) ss_cp4(dst + j, j < lim ? src + j : o.p, j < lim ? 4 : 0);
  }
}

// One tile: on return the eight groups' sums are in sm.red and every thread of the block has passed a
// barrier; ss_sum gives an entry. The caller reads sm.red before the next tile's first barrier.
template <bool AK, bool BK_>
__device__ __forceinline__ void ss_tile(SsSmem& sm, const SsOperand& a, const SsOperand& b, int m0, int n0, int K) {
  const int g = threadIdx.x >> 6, t = threadIdx.x & 63;
  const int tx = t & 7, ty = t >> 3;
  const int nk = (K + SS_KC - 1) / SS_KC;
  float acc[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = 0.0f;
#pragma unroll
  for (int s = 0; s < SS_STAGES - 1; ++s) {
    if (s < nk) {
      ss_copy<AK>(sm.op[s][0], a, m0, s * SS_KC, K);
      ss_copy<BK_>(sm.op[s][1], b, n0, s * SS_KC, K);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  }
  for (int kt = 0; kt < nk; ++kt) {
    asm volatile("cp.async.wait_group %0;" ::"n"(SS_STAGES - 2) : "memory");
    __syncthreads();   // chunk kt is here for everyone, and everyone has left the buffer refilled next
    if (kt + SS_STAGES - 1 < nk) {
      const int s = (kt + SS_STAGES - 1) % SS_STAGES;
      ss_copy<AK>(sm.op[s][0], a, m0, (kt + SS_STAGES - 1) * SS_KC, K);
      ss_copy<BK_>(sm.op[s][1], b, n0, (kt + SS_STAGES - 1) * SS_KC, K);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
    const float* pa = sm.op[kt % SS_STAGES][0];
    const float* pb = sm.op[kt % SS_STAGES][1];
    float part[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) part[i][j] = 0.0f;
#pragma unroll
    for (int kq = 0; kq < 2; ++kq) {
      const int k = 8 * g + 4 * kq;
      float av[4][4], bv[4][4];          // [k][row], [k][column]
      // MN-major: rows 4 ty .. 4 ty + 3 of one k per load; K-major: four k of rows ty, ty + 8, ... (rows of
      // neighbouring ty lie 68 floats apart: different banks)
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        if (AK) {
          const float4 v = *reinterpret_cast<const float4*>(pa + (ty + 8 * i) * SS_LDK + k);
          av[0][i] = v.x; av[1][i] = v.y; av[2][i] = v.z; av[3][i] = v.w;
        } else {
          const float4 v = *reinterpret_cast<const float4*>(pa + (k + i) * SS_LDM + 4 * ty);
          av[i][0] = v.x; av[i][1] = v.y; av[i][2] = v.z; av[i][3] = v.w;
        }
        if (BK_) {
          const float4 v = *reinterpret_cast<const float4*>(pb + (tx + 8 * i) * SS_LDK + k);
          bv[0][i] = v.x; bv[1][i] = v.y; bv[2][i] = v.z; bv[3][i] = v.w;
        } else {
          const float4 v = *reinterpret_cast<const float4*>(pb + (k + i) * SS_LDM + 4 * tx);
          bv[i][0] = v.x; bv[i][1] = v.y; bv[i][2] = v.z; bv[i][3] = v.w;
        }
      }
#pragma unroll
      for (int kk = 0; kk < 4; ++kk)
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int j = 0; j < 4; ++j) part[i][j] = fmaf(av[kk][i], bv[kk][j], part[i][j]);
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) acc[i][j] += part[i][j];
  }
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j)
      sm.red[g][AK ? ty + 8 * i : 4 * ty + i][BK_ ? tx + 8 * j : 4 * tx + j] = acc[i][j];
  __syncthreads();
}

__device__ __forceinline__ float ss_sum(const SsSmem& sm, int r, int c) {
  float s[SS_GROUPS];
#pragma unroll
  for (int g = 0; g < SS_GROUPS; ++g) s[g] = sm.red[g][r][c];
  return ((s[0] + s[1]) + (s[2] + s[3])) + ((s[4] + s[5]) + (s[6] + s[7]));
}

}  // namespace
}  // namespace polar
