// Tensor-core Gram-Schmidt projections (arnoldi_tc.cu) as the block FGMRES
// cycle uses them.
#pragma once

#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <cstdint>

#include "tc_plan.h"

namespace mtf {

constexpr int kPrepParts = 32;          // partial maxima and norms per column (block32.cu, k_bprep)
constexpr float kBasisScale = 16384.f;  // 2^14: unit-norm basis entries stay below the FP16 range limit

struct TcArnoldi;
TcArnoldi* tca_create();
void tca_destroy(TcArnoldi* t);
void tca_set_dots_hi(TcArnoldi& t, bool on);
void tca_prepare(TcArnoldi& t, int s, int m, int64_t ldn, cudaStream_t st);
void tca_store(TcArnoldi& t, const float* Vn, int q0, cudaStream_t st);
unsigned* tca_hmax(TcArnoldi& t);
void tca_project(TcArnoldi& t, int nq, float* W, int nc, double* H, int ldh, const float* maxparts, int ncm,
                 unsigned* err, cudaStream_t st);

// the basis's tiled FP16 hi / lo copies (dots, update; tc_plan.h)
struct TcaTiles {
  __half* Vd = nullptr;
  __half* Vu = nullptr;
  int nkc = 0, nbc = 0;
};
TcaTiles tca_tiles(const TcArnoldi& t);

#ifdef __CUDACC__
__device__ __forceinline__ void tca_split(float v, __half& hi, __half& lo) {
  hi = __float2half_rn(v);
  lo = __float2half_rn(v - __half2float(hi));
}
#endif

}  // namespace mtf
