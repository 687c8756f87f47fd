// The whole degree loop of the dense filter (Algorithms 2 and 3) as one launch (tc_loop.cu).
#pragma once
#include "common.cuh"

namespace rchfsi {

// Launch shape of the loop for an M x M operator and N columns (es: element size of the storage).
struct TcLoopPlan {
  bool ok = false;  // false: the per-step products of tc_gemm.cu are used
  int64_t M = 0, N = 0;  // the shape it was made for (with bf16)
  bool bf16 = false;
  int BN = 0, m_tiles = 0, nsplit = 0, kb_per_split = 0, stages = 0, elems = 0;
  uint32_t acc_cols = 0;
  size_t smem = 0;
  size_t ws_floats = 0;  // partial tiles of two steps
  size_t counters = 0;   // ints, zero before the launch
};
TcLoopPlan tc_loop_plan(int num_sms, int64_t M, int64_t N, bool bf16);

// steps k = 0 .. steps - 1:  out = a_k A R + b_k R + c_k R_prev + a_k W diag(lam_k), R_prev = R, R = out.
// R starts in R0 (R_prev is 0); step k writes R1 for even k and R0 for odd k.  A: M x M row-major (pitch ld,
// K-contiguous); R0, R1, W: M x N column-major (pitch ld); W may be null.  coef: a_k, b_k, c_k per step;
// lam: N floats per step (unused without W).  bf16: bfloat16 storage, else FP32 storage with TF32 products.
void tc_loop(cudaStream_t s, const TcLoopPlan& p, int64_t M, int64_t N, bool bf16, const void* A, int64_t ld, void* R0,
             void* R1, const void* W, const float* coef, const float* lam, int steps, float* ws, int* counters,
             int* err);

}  // namespace rchfsi
