// A projection of the CUDA-core family's step, as its kernels take it (simt.cu, gemm_f32.cu).
#pragma once

#include "dare_internal.h"

namespace dare {

enum { SG_Q = 0, SG_KV = 1, SG_OUT = 2 };
struct SgemmParams {
  const void* a;
  const int* idx;        // gathered rows of A (tokens), or nullptr
  const int* count;      // device count of them
  int a_cache_rows;      // A is addressed by cache row
  StepGeom g;
  int rows;              // rows of the launch (capacity of the list if gathered)
  const void* w0;
  const void* w1;        // SG_KV: W_V
  void* out0;
  void* out1;
  const float2* rope;
  float* q_prev;
  float* scores;
  float* q_raw;          // heads wider than 64: un-rotated scoring head of every token, for score_kernel
  int has_prev;
  int* status;
};

// fp32 projection on the tensor cores, operands split into three bf16 parts (gemm_f32.cu): width a multiple of 64.
cudaError_t launch_gemm_f32(int epi, const SgemmParams& p, cudaStream_t st);

}  // namespace dare
