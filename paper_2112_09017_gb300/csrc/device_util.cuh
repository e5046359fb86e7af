// Device helpers shared by the kernels of libpolar.so.
#pragma once

#include <stdint.h>

namespace polar {

// Round-to-nearest-even BF16 bit pattern of a float32 (NaN stays NaN).
__device__ __forceinline__ uint16_t bf16_rne_bits_dev(float x) {
  uint32_t u = __float_as_uint(x);
  if ((u & 0x7fffffffu) > 0x7f800000u) return (uint16_t)((u >> 16) | 0x40u);
  uint32_t lsb = (u >> 16) & 1u;
  return (uint16_t)((u + 0x7fffu + lsb) >> 16);
}

__device__ __forceinline__ float bf16_to_f32_dev(uint16_t b) { return __uint_as_float(((uint32_t)b) << 16); }

// Plane q of the split x = x_0 + x_1 + x_2 (each the BF16 rounding of what the
// previous planes left), for q < NP; planes[q] receives the bit pattern.
template <int NP>
__device__ __forceinline__ void split_planes_dev(float x, uint16_t (&planes)[3]) {
  float rem = x;
#pragma unroll
  for (int q = 0; q < NP; ++q) {
    uint16_t b = bf16_rne_bits_dev(rem);
    planes[q] = b;
    rem = rem - bf16_to_f32_dev(b);
  }
}

// Two FP32 operations per instruction (round-to-nearest each): a + b, a b + c, a - b.
__device__ __forceinline__ float2 add_x2(float2 a, float2 b) {
  float2 d;
  asm("{\n\t.reg .b64 a, b, c;\n\tmov.b64 a, {%2, %3};\n\tmov.b64 b, {%4, %5};\n\tadd.rn.f32x2 c, a, b;\n\t"
      "mov.b64 {%0, %1}, c;\n\t}"
      : "=f"(d.x), "=f"(d.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return d;
}
__device__ __forceinline__ float2 fma_x2(float2 a, float2 b, float2 c) {
  float2 d;
  asm("{\n\t.reg .b64 a, b, c;\n\tmov.b64 a, {%2, %3};\n\tmov.b64 b, {%4, %5};\n\tmov.b64 c, {%6, %7};\n\t"
      "fma.rn.f32x2 a, a, b, c;\n\tmov.b64 {%0, %1}, a;\n\t}"
      : "=f"(d.x), "=f"(d.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
  return d;
}
__device__ __forceinline__ float2 sub_x2(float2 a, float2 b) { return fma_x2(b, make_float2(-1.0f, -1.0f), a); }

// The two BF16 values of a word as floats.
__device__ __forceinline__ float2 bf16_pair(uint32_t w) {
  return make_float2(__uint_as_float(w << 16), __uint_as_float(w & 0xffff0000u));
}

// A non-negative number s 2^e; e = FIXED_BAD for one that is not finite.
struct Fixed {
  uint64_t s;
  int e;
};
constexpr int FIXED_BAD = 1024;

__device__ __forceinline__ double fixed_double(Fixed f) {   // rounded to nearest; for -900 < e
  if (f.e == FIXED_BAD) return __longlong_as_double(0x7ff8000000000000ll);
  if (f.s == 0) return 0.0;
  const int lz = __clzll((long long)f.s);
  const uint64_t n = f.s << lz, r = (n >> 11) + ((n >> 10) & 1u);   // 53 bits; the top one adds one to the exponent
  return __longlong_as_double((long long)(((uint64_t)(1023 + 63 - 1 - lz + f.e) << 52) + r));
}

// The sum of the lanes' q, each below 2^59 (2^60 in half of the lanes, the others zero).
__device__ __forceinline__ uint64_t warp_add59(uint64_t q) {
  const uint32_t s0 = __reduce_add_sync(0xffffffffu, (uint32_t)q & 0x1fffffu),
                 s1 = __reduce_add_sync(0xffffffffu, (uint32_t)(q >> 21) & 0x1fffffu),
                 s2 = __reduce_add_sync(0xffffffffu, (uint32_t)(q >> 42));
  return ((uint64_t)s2 << 42) + ((uint64_t)s1 << 21) + s0;
}

// The sum of N non-negative floats of every lane, the same in every lane of a converged warp, whatever their
// magnitudes: fixed point with 36 - N bits below the largest value's last one, so that what is cut off is no more
// than a float64 sum's rounding, in integers because a chain of FP64 shuffles costs a step of a small solve more
// than the warp-wide integer sums (FP64 runs at two operations a cycle and SM).
template <int N>
__device__ __forceinline__ Fixed warp_fixed(const float (&v)[N]) {
  static_assert(N == 1 || N == 2, "a lane's values add up to less than 2^59");
  uint32_t top = 0;
#pragma unroll
  for (int i = 0; i < N; ++i) top = max(top, __float_as_uint(v[i]));
  top = __reduce_max_sync(0xffffffffu, top);
  if (top >= 0x7f800000u) return {0, FIXED_BAD};
  const int ex = max((int)(top >> 23), 1);
  uint64_t q = 0;
#pragma unroll
  for (int i = 0; i < N; ++i) {
    const uint32_t b = __float_as_uint(v[i]);
    const int down = ex - max((int)(b >> 23), 1);
    const uint64_t man = (b & 0x7fffffu) | (b >> 23 ? 0x800000u : 0u);
    q += down < 60 - N ? (man << (36 - N)) >> down : 0u;
  }
  return {warp_add59(q), ex - 186 + N};
}
template <int N>
__device__ __forceinline__ double warp_sum64(const float (&v)[N]) {
  return fixed_double(warp_fixed<N>(v));
}
__device__ __forceinline__ double warp_sum64(float v) { return warp_sum64<1>({v}); }

// The sum of 16 of them, in lanes 0 to 15.
__device__ __forceinline__ double warp_sum16(Fixed f, int lane) {
  const int top = (int)__reduce_max_sync(0xffffffffu, (uint32_t)(f.e + FIXED_BAD)) - FIXED_BAD;
  if (top == FIXED_BAD) return fixed_double({0, FIXED_BAD});
  const int down = top - f.e;
  return fixed_double({warp_add59(lane < 16 && down < 60 ? (f.s >> 4) >> down : 0u), top + 4});
}

// s <- s + b rounded, and its rounding error, exactly (Knuth's two-sum).
__device__ __forceinline__ float two_sum(float& s, float b) {
  const float t = s + b, bb = t - s, e = (s - (t - bb)) + (b - bb);
  s = t;
  return e;
}

// A float64 sum of squares of float32 values. FP64 runs at 1/64 of the FP32 rate here (two FMAs a cycle and SM),
// which made the norm of a batch take longer than reading it; so squares are split exactly into FP32 pairs
// (p = x x, e = fma(x, x, -p)) and added by two-sums into three floats, the last of which alone rounds, at about
// 2^-68 of the sum, and only every eighth group of eight goes through FP64. Groups whose largest magnitude is
// outside [2^-50, 2^60], where squares or their errors could leave float32's range, are summed in FP64 as they are.
struct SquareSum {
  double total = 0.0;
  float hi = 0.f, mid = 0.f, lo = 0.f;
  int held = 0;
  __device__ __forceinline__ void add8(const float (&v)[8]) {
    float top = 0.f;
#pragma unroll
    for (int j = 0; j < 8; ++j) top = fmaxf(top, fabsf(v[j]));
    if (top <= 0x1p60f && (top >= 0x1p-50f || top == 0.f)) {   // a NaN among smaller values passes through the sums
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const float p = v[j] * v[j];
        lo += two_sum(mid, two_sum(hi, p));
        lo += two_sum(mid, fmaf(v[j], v[j], -p));
      }
      if (++held == 8) flush();
    } else {
#pragma unroll
      for (int j = 0; j < 8; ++j) total = fma((double)v[j], (double)v[j], total);
    }
  }
  __device__ __forceinline__ void flush() {
    total += (double)hi + ((double)mid + (double)lo);
    hi = mid = lo = 0.f;
    held = 0;
  }
  __device__ __forceinline__ double value() {
    flush();
    return total;
  }
};

// 8 consecutive values of a float32 row, `n` of them existing (zeros beyond), 16-byte loads when vec.
__device__ __forceinline__ void load_row8(const float* p, int64_t n, bool vec, float (&v)[8]) {
  if (vec && n >= 8) {
    const float4 a = __ldg(reinterpret_cast<const float4*>(p)), b = __ldg(reinterpret_cast<const float4*>(p) + 1);
    v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
    v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
  } else {
#pragma unroll
    for (int j = 0; j < 8; ++j) v[j] = j < n ? __ldg(p + j) : 0.0f;
  }
}

// The reverse for stores.
__device__ __forceinline__ void store_row8(float* p, int64_t n, bool vec, const float (&v)[8]) {
  if (vec && n >= 8) {
    reinterpret_cast<float4*>(p)[0] = make_float4(v[0], v[1], v[2], v[3]);
    reinterpret_cast<float4*>(p)[1] = make_float4(v[4], v[5], v[6], v[7]);
  } else {
#pragma unroll
    for (int j = 0; j < 8; ++j)
      if (j < n) p[j] = v[j];
  }
}

// np planes of 8 consecutive values, one 16-byte store per plane (base 16-byte aligned, pstride a multiple of 8).
// Each plane is the round-to-nearest-even BF16 of what the previous planes left.
__device__ __forceinline__ void split_store8(uint16_t* base, int64_t pstride, int np, const float (&v)[8]) {
  float r[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) r[j] = v[j];
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    if (q >= np) break;
    uint32_t w[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(w[k]) : "f"(r[2 * k + 1]), "f"(r[2 * k]));
      r[2 * k] -= __uint_as_float(w[k] << 16);
      r[2 * k + 1] -= __uint_as_float(w[k] & 0xffff0000u);
    }
    *reinterpret_cast<uint4*>(base + q * pstride) = make_uint4(w[0], w[1], w[2], w[3]);
  }
}

// The exact sum of three planes' 8 consecutive values.
__device__ __forceinline__ void sum_row8(const uint16_t* p, int64_t pstride, float (&v)[8]) {
  uint4 q[3];
#pragma unroll
  for (int i = 0; i < 3; ++i) q[i] = *reinterpret_cast<const uint4*>(p + i * pstride);
  const uint32_t h[4] = {q[0].x, q[0].y, q[0].z, q[0].w}, m[4] = {q[1].x, q[1].y, q[1].z, q[1].w},
                 l[4] = {q[2].x, q[2].y, q[2].z, q[2].w};
#pragma unroll
  for (int w = 0; w < 4; ++w) {
    v[2 * w] = (__uint_as_float(h[w] << 16) + __uint_as_float(m[w] << 16)) + __uint_as_float(l[w] << 16);
    v[2 * w + 1] = (__uint_as_float(h[w] & 0xffff0000u) + __uint_as_float(m[w] & 0xffff0000u)) +
                   __uint_as_float(l[w] & 0xffff0000u);
  }
}

// The strictly lower triangle of a symmetric n x n matrix kept as three BF16 planes (pitch ldp,
// plane stride ps) from its upper triangle: 64 x 64 blocks (bi <= bj) of the upper triangle, taken
// t0, t0 + dt, ... in column order, read with 16-byte accesses into shared memory (`tile`, at least
// 3 x 64 x 66 halves) and written transposed with 16-byte accesses (diagonal blocks element by
// element below their diagonal). Columns from n up to the next multiple of 8 are padding: they may
// be written with zeros. All threads of the block take part (blockDim.x a multiple of 32).
__device__ __forceinline__ void mirror3_tiles(uint16_t* P, int64_t ldp, int64_t ps, int64_t n, int64_t t0, int64_t dt,
                                              uint16_t* tile) {
  constexpr int LD = 66;   // halves per shared row: 33 words, so column reads of eight rows miss each other's banks
  const int64_t nt = (n + 63) / 64, ntri = nt * (nt + 1) / 2;
  const int tid = threadIdx.x, nthr = blockDim.x;
  for (int64_t t = t0; t < ntri; t += dt) {
    int64_t bj = (int64_t)((sqrt(8.0 * (double)t + 1.0) - 1.0) * 0.5);
    while (bj * (bj + 1) / 2 > t) --bj;
    while ((bj + 1) * (bj + 2) / 2 <= t) ++bj;
    const int64_t bi = t - bj * (bj + 1) / 2;
    const int64_t i0 = bi * 64, j0 = bj * 64;
    __syncthreads();
    for (int u = tid; u < 3 * 512; u += nthr) {   // rows i0.., columns j0.. of the upper block
      const int q = u >> 9, rr = (u >> 3) & 63, cv = u & 7;
      const int64_t i = i0 + rr, j = j0 + 8 * cv;
      uint4 v = make_uint4(0u, 0u, 0u, 0u);
      if (i < n && j < n) v = *reinterpret_cast<const uint4*>(P + q * ps + i * ldp + j);
      uint32_t* d = reinterpret_cast<uint32_t*>(tile + (q * 64 + rr) * LD + 8 * cv);
      d[0] = v.x; d[1] = v.y; d[2] = v.z; d[3] = v.w;
    }
    __syncthreads();
    for (int u = tid; u < 3 * 512; u += nthr) {   // rows j0.. of the lower block, columns i0..
      const int q = u >> 9, jj = (u >> 3) & 63, iv = u & 7;
      const int64_t j = j0 + jj, i = i0 + 8 * iv;
      if (j >= n || i >= n) continue;
      const uint16_t* col = tile + (q * 64 + 8 * iv) * LD + jj;
      uint16_t* dst = P + q * ps + j * ldp + i;
      if (bi < bj) {
        uint32_t w[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) w[e] = (uint32_t)col[(2 * e) * LD] | ((uint32_t)col[(2 * e + 1) * LD] << 16);
        *reinterpret_cast<uint4*>(dst) = make_uint4(w[0], w[1], w[2], w[3]);
      } else {
#pragma unroll
        for (int e = 0; e < 8; ++e)
          if (i + e < j && i + e < n) dst[e] = col[e * LD];
      }
    }
  }
}

}  // namespace polar
