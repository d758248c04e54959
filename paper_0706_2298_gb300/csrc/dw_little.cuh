// FP32 little GCR of one system in one persistent cooperative kernel (dw_little.cu), as used by
// dw_dfl.cu: even-odd preconditioned (A.2), deflated by the global modes (A.3), GCR (A.4).
#pragma once

#include "dw_common.cuh"

constexpr int LITTLE_NKV = 24;        // Krylov vectors per cycle, at most
constexpr int LITTLE_COPIES = 4;      // accumulators of a value: CTA b adds to copy b mod 4
constexpr int LITTLE_NV = 128;        // values per grid reduction, at most (2 Ns + 2 nkv + 3)

constexpr size_t LITTLE_ACC_BYTES = (size_t)3 * LITTLE_COPIES * LITTLE_NV * sizeof(double);

struct LittleArgs {
  int Ne, No, nkv, maxit, a3;
  const int *list_e, *list_o, *lnb_e, *lnb_o;   // block rows of a parity; their neighbours' positions [row][8]
  const float *M;                               // [Nb][8][Ns][Ns] complex, column-major blocks
  const float *g, *Bg, *Ainv;                   // [Ns][Ne Ns], [Ns][Ne Ns], [Ns][Ns]
  const float* b;
  float* v;
  float* work;                                  // 2 nkv + 5 vectors of Ne Ns complex
  double* acc;                                  // [3][LITTLE_COPIES][LITTLE_NV] reduction accumulators, zero at launch
  double* out;                                  // [0] iterations, [1] relative residual
  double tol;
};

// whether a kernel for this Ns and number of block rows per CTA exists and `grid` CTAs of it are resident at
// once (sets its attributes)
bool little_warp_ready(int Ns, int rows, int grid, int sms);
cudaError_t little_warp_launch(const LittleArgs& a, int Ns, int grid, cudaStream_t s);
