// Pass kernels of 48 px patches (the CTA-per-unit kernels of generic_kernels.cuh).
#include "generic_kernels.cuh"

namespace mfbd_dev {

template int generic_adjoint_ctas_n<48>(bool half_box, int sms);
template cudaError_t launch_generic_forward_n<48>(const GenericParams& prm, int sms, cudaStream_t s);
template cudaError_t launch_generic_adjoint_n<48>(const GenericParams& prm, int sms, cudaStream_t s);

}  // namespace mfbd_dev
