// FP16-storage forward row transforms (the inverses: rows_f16_inv.cu), and the
// tensor-core compression lines.
#include "launch.h"
#include "tc_fft.cuh"

namespace bfp {

cudaError_t launch_rows_f16(int log2n, int mode, bool naive, const RowArgs& a, cudaStream_t s) {
  if (mode == kForward) return launch_rows<__half2, __half2, kForward, false, false>(log2n, a, s);
  if (mode == kInverse) return launch_rows_f16_inverse(log2n, naive, a, s);
  return cudaErrorInvalidValue;
}

cudaError_t launch_tc_compress(bool in32, const RowArgs& a, cudaStream_t s) {
  if (a.tc_b == nullptr || a.h == nullptr) return cudaErrorInvalidValue;
  return in32 ? launch_tc_kernel<kCompress, float2>(a, s) : launch_tc_kernel<kCompress, __half2>(a, s);
}

}  // namespace bfp
