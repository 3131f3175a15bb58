// Registry of the instantiated FFT engines (one translation unit per group so the
// build compiles them in parallel).
#pragma once

#include <cuda_runtime.h>

#include "top_internal.h"

namespace top {

struct EngineInfo {
  int M;      // line length handled (half of an even padded size)
  int G;      // threads per line
  int NS;     // number of radix stages
  int R[4];   // radices
  int tw_size;
  int rows;         // rows per block of the row passes
  int ci;           // workspace lines interleaved by the row passes
};

// PASS_ROWS_CHAIN: the inverse row pass of one propagation fused with the forward row pass of
// the next (the second parameter block).
enum PassKind : int { PASS_ROWS_FWD = 0, PASS_COLS = 1, PASS_ROWS_INV = 2, PASS_ROWS_CHAIN = 3 };

#define TOP_DECLARE_UNIT(name)                                                                        \
  bool engine_info_##name(int M, EngineInfo* info);                                                   \
  cudaError_t launch_pass_##name(int kind, int M, const PassParams& p, const PassParams* next, cudaStream_t s, \
                                 bool* found);

TOP_DECLARE_UNIT(small)
TOP_DECLARE_UNIT(m128)
TOP_DECLARE_UNIT(m256)
TOP_DECLARE_UNIT(m512)
TOP_DECLARE_UNIT(m1024)
TOP_DECLARE_UNIT(m2048)
TOP_DECLARE_UNIT(m4096)
TOP_DECLARE_UNIT(m250)
TOP_DECLARE_UNIT(m500)
TOP_DECLARE_UNIT(m768)
TOP_DECLARE_UNIT(m1000)

#undef TOP_DECLARE_UNIT

// Bluestein line transforms (CztParams) on the power-of-two engines of a unit.
cudaError_t launch_czt_small(int M, const CztParams& p, cudaStream_t s, bool* found);
cudaError_t launch_czt_m128(int M, const CztParams& p, cudaStream_t s, bool* found);
cudaError_t launch_czt_m256(int M, const CztParams& p, cudaStream_t s, bool* found);
cudaError_t launch_czt_m512(int M, const CztParams& p, cudaStream_t s, bool* found);
cudaError_t launch_czt_m1024(int M, const CztParams& p, cudaStream_t s, bool* found);
cudaError_t launch_czt_m2048(int M, const CztParams& p, cudaStream_t s, bool* found);
cudaError_t launch_czt_m4096(int M, const CztParams& p, cudaStream_t s, bool* found);
// The same as two halves on the 4096-point engine (convolution length 8192).
cudaError_t launch_czt_split_m4096(int M, const CztParams& p, cudaStream_t s, bool* found);

}  // namespace top
