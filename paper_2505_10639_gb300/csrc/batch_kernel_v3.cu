// The batch kernel of batch_kernels.cuh compiled for 3 CTAs per SM
// (up to 80 registers a thread).
#include "batch_kernels.cuh"

namespace mfbd_dev {

template int batch_max_ctas_variant<3>(size_t smem, bool half_box);
template cudaError_t launch_batch_variant<3>(const BatchParams& prm, int ctas, size_t smem, cudaStream_t s);

}  // namespace mfbd_dev
