// Host side of the batched persistent kernel (batch_kernels.cuh): shared-memory
// size and the dispatch over its two register variants.
#include "batch_internal.h"

#include <algorithm>

namespace mfbd_dev {

size_t batch_smem(const bool (&sizes)[4], bool half_box) {
    // the twiddles, then the exchange buffers of an item, a P part's coefficient
    // tile (up to 256 modes) or a G part's sums
    size_t unit = (size_t)kJC * std::max(256, kBT / 32 * kGM) * sizeof(float) / sizeof(float2);
    const int n[4] = {48, 64, 96, 128};
    for (int i = 0; i < 4; ++i)
        if (sizes[i])
            unit = std::max(unit, (size_t)(n[i] <= 64 ? kSmallUnits : 1) * n[i] * (half_box ? n[i] / 2 + 4 : n[i] + 4));
    return (kBatchTwiddles + unit) * sizeof(float2);
}

int batch_max_ctas_per_sm(size_t smem, bool half_box, int variant) {
    return variant == 1 ? batch_max_ctas_variant<3>(smem, half_box) : batch_max_ctas_variant<2>(smem, half_box);
}

cudaError_t launch_batch(const BatchParams& prm, int ctas, size_t smem, int variant, cudaStream_t s) {
    if (prm.n_items == 0) return cudaSuccess;
    return variant == 1 ? launch_batch_variant<3>(prm, ctas, smem, s) : launch_batch_variant<2>(prm, ctas, smem, s);
}

}  // namespace mfbd_dev
