// One split-BF16 product C = alpha op(A) op(B) + beta C (three planes) in 128 x 64 tiles, for shapes with few
// 128 x 256 tiles; the pieces are in coop_kernel.cuh (no grid barrier here: an ordinary launch). A 48 x 48 x 6000
// product was one tile of 165 us. Where even the narrow tiles are few, clusters of four blocks share them
// along K.
#include <algorithm>

#include "coop_kernel.cuh"

namespace polar {
namespace {

struct CoGemm {
  CUtensorMap a, b;
  float* C;
  int64_t ldc;
  int M, N, K, tri, S;
  float alpha, beta;
  unsigned int* err;
  int withhold;
};

template <bool SPLIT, bool A_MN, bool BKM>
__device__ __forceinline__ void co_gemm(const CoGemm& p, uint8_t* co_raw) {
  CoCtx x = co_setup<64, CO_P, SPLIT>(co_raw, nullptr);
  CoPipe pipe;
  CoEpi e{};
  e.M = p.M; e.N = p.N;
  e.C = p.C; e.ldc = p.ldc;
  e.c1 = p.beta; e.c3 = p.alpha;
  const CoTiles t = co_tiles<64>(p.M, p.N, p.tri != 0);
  co_product<64, SPLIT, A_MN, false, CO_EPI_GEMM, BKM>(x, pipe, &p.a, BKM ? nullptr : &p.b, BKM ? &p.b : nullptr, t, p.K,
                                                       e, p.S, p.withhold);
  __syncthreads();
  co_teardown<64, SPLIT>(x, nullptr, reinterpret_cast<int*>(p.err));
}

template <bool A_MN, bool BKM>
__global__ void __launch_bounds__(CO_THREADS, 1) co_gemm_kernel(const __grid_constant__ CoGemm p) {
  extern __shared__ uint8_t co_raw[];
  co_gemm<false, A_MN, BKM>(p, co_raw);
}

template <bool A_MN, bool BKM>
__global__ void __cluster_dims__(CO_CLUSTER, 1, 1) __launch_bounds__(CO_THREADS, 1)
    co_gemm_split_kernel(const __grid_constant__ CoGemm p) {
  extern __shared__ uint8_t co_raw[];
  co_gemm<true, A_MN, BKM>(p, co_raw);
}

template <bool A_MN, bool BKM>
cudaError_t launch_t(const CoGemm& p, bool split, int blocks, cudaStream_t s) {
  auto k = split ? co_gemm_split_kernel<A_MN, BKM> : co_gemm_kernel<A_MN, BKM>;
  const size_t smem = split ? co_smem<64, CO_P, true>() : co_smem<64>();
  cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  k<<<(unsigned)blocks, CO_THREADS, smem, s>>>(p);
  return cudaGetLastError();
}

int gemm_sms() {
  int n = 0;
  return device_is_sm103(&n) && n > 0 ? n : 1;
}

}  // namespace

// 128 x 256 tiles take about 1600 cycles per k-block of 32 and 17000 for set-up and output step, in whole waves
// (co_cost's measure; narrow ones about 750). Whole calls (splits and product) on 128 x 256 tiles and on narrow
// ones: 48 x 48 x 6000 165 and 36 us, 128 x 128 x 512 31 and 17, 512^3 35 and 17, 1024^3 52 and 27, 100 x 5000 x
// 500 38 and 25, 5000 x 100 x 5000 183 and 120, 1500^3 68 and 56, 971 x 1725 x 2232 109 and 76. From about one wave
// of wide tiles on the costs decide for those (2048^3, 128 of them, 88 us; 3000 x 2500 x 500, 240, 60 us): twice the
// operand traffic per product is what bounds narrow tiles there; past two waves they are not asked.
CoopForm co_gemm_form(int64_t M, int64_t N, int64_t K, bool tri) {
  CoopForm f;
  const int64_t lim = (int64_t)1 << 30;
  if (M > lim || N > lim || K > lim) return f;
  const int sms = gemm_sms();
  const int64_t tm = (M + 127) / 128, tn = (N + 255) / 256;
  const int64_t wide = tri ? tri_tiles(tm, tn) : tm * tn;
  if (wide > 2 * sms) return f;
  const CoopProduct p = {M, N, K, tri};
  double narrow;
  f.split = coop_split_plan(&p, 1, sms, f.S, &f.blocks, &narrow);
  const double big = (double)((wide + sms - 1) / sms) * ((double)((K + 31) / 32) * 1600.0 + 17000.0);
  if (narrow + 4000.0 >= big) return CoopForm();
  f.tn = 64;
  const int tiles = co_tiles<64>(M, N, tri).ntiles;
  if (!f.split) f.S[0] = 1;
  f.blocks = f.split ? (tiles * f.S[0] + CO_CLUSTER - 1) / CO_CLUSTER * CO_CLUSTER : std::min(sms, tiles);
  return f;
}

cudaError_t launch_co_gemm(const TcArgs& a, const CoopForm& f, cudaStream_t s) {
  CoGemm p{};
  p.S = f.S[0];
  if (!tc_make_map(&p.a, a.a, CO_P, !a.a.kmajor, BM) || !tc_make_map(&p.b, a.b, CO_P, !a.b.kmajor, 64))
    return cudaErrorInvalidValue;
  p.C = a.C; p.ldc = a.ldc;
  p.M = (int)a.M; p.N = (int)a.N; p.K = (int)a.K; p.tri = a.triangular ? 1 : 0;
  p.alpha = a.alpha; p.beta = a.beta;
  p.err = a.err_out;
  p.withhold = a.withhold_tma;
  auto launch = a.a.kmajor ? (a.b.kmajor ? launch_t<false, true> : launch_t<false, false>)
                           : (a.b.kmajor ? launch_t<true, true> : launch_t<true, false>);
  return launch(p, f.split, f.blocks, s);
}

}  // namespace polar
