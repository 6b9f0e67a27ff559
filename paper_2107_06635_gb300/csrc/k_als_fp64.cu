// Instantiations of the ALS kernel k_als for the FP64 contexts (one CTA per
// item at two or three CTAs per SM).
#include "als_kernel.cuh"

namespace ntu {

cudaError_t als_launch_fp64(const AlsArgs& a, int n, int split, bool three, size_t smem,
                             cudaStream_t stream) {
  return als_launch_impl<-1>(a, n, split, three, smem, stream);
}

}  // namespace ntu
