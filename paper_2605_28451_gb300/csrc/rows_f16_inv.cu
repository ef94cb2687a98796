// FP16-storage inverse row transforms: the block-floating-point path (Eq. 1)
// and the naive unshifted path of Section III-B.
#include "launch.h"
#include "tc_fft.cuh"

namespace bfp {

cudaError_t launch_rows_f16_inverse(int log2n, bool naive, const RowArgs& a, cudaStream_t s) {
  return naive ? launch_rows<__half2, __half2, kInverse, true, false>(log2n, a, s)
               : launch_rows<__half2, __half2, kInverse, false, false>(log2n, a, s);
}

}  // namespace bfp
