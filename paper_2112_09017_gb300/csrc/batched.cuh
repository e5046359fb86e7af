// What the kernels of the batched solves share (batched.cu, coop_batch.cu).
#pragma once

#include "internal.cuh"

namespace polar {

constexpr int kBatchEpiWarps = 8;   // residual sums per Gram tile

// Per-problem layout of the workspace (device memory).
struct BMeta {
  int64_t m, n;
  uint16_t* xp[2];   // three planes each, pitch ldp, plane stride xps
  uint16_t* gp;      // three planes of G's upper triangle (whole 128-wide tiles), pitch ldp, plane stride gps
  uint16_t* ap;      // P planes of A
  float* C;          // n x n, U^T A
  double* partials;  // Gram partials: ntiles_gram * kBatchEpiWarps
  int64_t ldp, xps, gps;
  int ntiles_gram;
  int slice;         // k-blocks of 32 per promoted slice
};

struct BShared {     // device: shared state of the batch
  unsigned int bar[2];   // the grid barrier of the loop's launch, zero between launches
  int err;           // a bounded wait expired
  int pad;
  double tol;
  int running[4];    // problems still running after the finalize of step k, at slot k % 4
};

// Operand maps of one problem's product (CUtensorMap).
struct alignas(128) TcMapPair {
  unsigned char a[128], b[128];
};

// One 128 x 128 tile of one problem: its row and column, and the product's K.
struct TcTile {
  int32_t prob, bi, bj;
  int32_t K;
};

struct CoBatch {
  const TcTile *gram_t, *upd_t, *h_t;
  int n_gram, n_upd, n_h;
  const TcMapPair* gram_m[2];   // a: X_k as MN-major operand; b: G mirrored (K-major)
  const TcMapPair* upd_m[2];    // a: X_k as K-major operand; b: G
  const TcMapPair* h_m;         // [problem][parity] a: X_k, b: A, both MN-major
  const BMeta* meta;
  DevState* st;
  BShared* sh;
  int count, P;
  StopRule rule;
  float pre_c1, pre_c3;
  int withhold;
  uint64_t wait_ns;             // bound of a grid barrier's wait
};

// The loop of every problem in the tables, then U^T A of every finished problem, in one cooperative launch
// of at most max_grid blocks.
cudaError_t launch_co_batch(const CoBatch& b, int max_grid, cudaStream_t s);

__device__ __forceinline__ bool finished_ok(int status) {
  return status == ST_CONVERGED || status == ST_NOT_CONVERGED;
}

}  // namespace polar
