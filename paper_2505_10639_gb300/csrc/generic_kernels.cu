// Frame reduction of the CTA-per-unit kernels (any patch size) and the
// size dispatch of their pass kernels, which are instantiated per patch
// size in generic_n48.cu ... generic_n128.cu (generic_kernels.cuh).
#include <algorithm>

#include "mfbd_internal.h"
#include "chained.cuh"
#include "frame_reduction.cuh"

namespace mfbd_dev {

namespace {

using namespace reduction;

// A CTA takes 1/S of the frequencies of one (patch, object) at a time (S =
// rsplit); with one object and one split its sum is the patch's loss,
// otherwise the sums of a patch's objects and splits are added in order by
// loss_combine_kernel. HOLD frames of a frequency are held by each of FS lanes. Against
// one warp per (patch, object, split) and four frames' loads in flight: 2,904
// units of 96 px 0.126 -> 0.081 ms, 735 of 128 px 0.085 -> 0.056, 12,800 of 128
// px 0.852 -> 0.442 (60 % of the copy peak on what it cannot do without).
constexpr int kRedWarps = 8;

template <int HOLD, int FS, bool EXPL = false>
__global__ void __launch_bounds__(32 * kRedWarps, HOLD == 32 ? 1 : 2) generic_reduce_kernel(const GenericParams prm) {
    constexpr int kF = 32 / FS;  // frequencies of a warp
    __shared__ double part[kRedWarps];
    const int N = prm.N, half = N * (N / 2 + 1), J = prm.J, S = prm.rsplit;
    const size_t dstride = (size_t)N * prm.spec_ld;
    const long long work = (long long)prm.P * prm.K * S;
    chain_wait();
    chain_release();
    for (long long u = blockIdx.x; u < work; u += gridDim.x) {
        const long long pk = u / S;
        const int s = (int)(u - pk * S), k = (int)(pk % prm.K);
        RedPtr r;
        r.N = N;
        r.J = J;
        r.spec_ld = prm.spec_ld;
        r.gamma = prm.gamma;
        r.d = prm.spectra + (size_t)pk * J * dstride;
        r.h = prm.gscr + (size_t)pk * J * half;
        r.w = prm.weights + (size_t)k * J;
        r.supp = prm.obj[k].supp;
        r.sw = prm.sw;
        r.obj = prm.object ? prm.object + (size_t)pk * dstride : nullptr;
        r.oin = prm.oin ? prm.oin + (size_t)pk * dstride : nullptr;
        r.gobj = prm.gobj ? prm.gobj + (size_t)pk * dstride : nullptr;
        const double v = cta_sum<kRedWarps>(
            reduce_lane<HOLD, FS, EXPL>(r, kF * (kRedWarps * s + (threadIdx.x >> 5)), kF * kRedWarps * S), part);
        if (threadIdx.x == 0) (prm.K * S == 1 ? prm.loss : prm.lpart)[u] = v;
        __syncthreads();
    }
}

__global__ void loss_combine_kernel(const double* __restrict__ lpart, int S, double* __restrict__ loss, int P) {
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    chain_wait();
    chain_release();
    if (p >= P) return;
    double tot = 0.0;
    for (int i = 0; i < S; ++i) tot += lpart[(size_t)p * S + i];
    loss[p] = tot;
}

}  // namespace

size_t generic_smem(int N, bool half_box) {
    const int stride = half_box ? N / 2 + 4 : N + 4;  // Geo<N>::S_HALF, S_FULL
    return ((size_t)2 * N + (size_t)N * stride) * sizeof(float2);  // at most 2 N twiddles
}

int generic_adjoint_ctas(int N, bool half_box, int sms) {
    switch (N) {
        case 48: return generic_adjoint_ctas_n<48>(half_box, sms);
        case 64: return generic_adjoint_ctas_n<64>(half_box, sms);
        case 96: return generic_adjoint_ctas_n<96>(half_box, sms);
        case 128: return generic_adjoint_ctas_n<128>(half_box, sms);
        default: return 0;
    }
}

cudaError_t launch_generic_forward(const GenericParams& prm, int sms, cudaStream_t s) {
    const long long units = (long long)prm.P * prm.K * prm.J;
    if (units == 0) return cudaSuccess;
    switch (prm.N) {
        case 48: return launch_generic_forward_n<48>(prm, sms, s);
        case 64: return launch_generic_forward_n<64>(prm, sms, s);
        case 96: return launch_generic_forward_n<96>(prm, sms, s);
        case 128: return launch_generic_forward_n<128>(prm, sms, s);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_generic_adjoint(const GenericParams& prm, int sms, cudaStream_t s) {
    const long long units = (long long)prm.P * prm.K * prm.J;
    if (units == 0) return cudaSuccess;
    const bool rec = prm.pscr == nullptr;
    if (rec && (!prm.e2scr || prm.e2_ctas < 1)) return cudaErrorInvalidValue;
    switch (prm.N) {
        case 48: return launch_generic_adjoint_n<48>(prm, sms, s);
        case 64: return launch_generic_adjoint_n<64>(prm, sms, s);
        case 96: return launch_generic_adjoint_n<96>(prm, sms, s);
        case 128: return launch_generic_adjoint_n<128>(prm, sms, s);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_generic_reduction(const GenericParams& prm, int sms, cudaStream_t s) {
    if (prm.P == 0) return cudaSuccess;
    const int per_patch = prm.K * prm.rsplit;
    if (per_patch > 1 && !prm.lpart) return cudaErrorInvalidValue;
    // up to 16 frames of a frequency in a lane's registers, then two and four
    // lanes a frequency, then chunks: 2,904 units of 12 frames (96 px) 0.081 ms
    // (0.110 in chunks, 0.097 over two lanes of 8); 12,800 of 32 frames (128 px)
    // 0.442 (0.460 as 32 in one lane, 0.477 in chunks); 22,500 of 100 frames (64
    // px) 0.283 (0.329 in chunks). The object-inferring form is not split; held
    // against read twice, whole evaluations: 900 patches of 15 frames (64 px) 824
    // -> 707 us, 100 of 16 167 -> 154, 225 of 12 (96 px) 387 -> 345.
    auto kern = prm.oin        ? (prm.J <= 8    ? generic_reduce_kernel<8, 1, true>
                                  : prm.J <= 16 ? generic_reduce_kernel<16, 1, true>
                                                : generic_reduce_kernel<0, 1, true>)
                : prm.J <= 8   ? generic_reduce_kernel<8, 1>
                : prm.J <= 16  ? generic_reduce_kernel<16, 1>
                : prm.J <= 32  ? generic_reduce_kernel<16, 2>
                : prm.J <= 64  ? generic_reduce_kernel<16, 4>
                : prm.J <= 128 ? generic_reduce_kernel<32, 4>
                               : generic_reduce_kernel<0, 1>;
    int per_sm = 0;
    cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, 32 * kRedWarps, 0);
    if (e != cudaSuccess) return e;
    long long ctas = (long long)sms * (per_sm > 0 ? per_sm : 1);
    if (ctas > (long long)prm.P * per_patch) ctas = (long long)prm.P * per_patch;
    e = launch_chained(prm.chain, kern, (int)ctas, 32 * kRedWarps, 0, s, prm);
    if (e != cudaSuccess || per_patch == 1) return e;
    return launch_loss_combine(prm.lpart, per_patch, prm.loss, prm.P, s, prm.chain);
}

int generic_reduction_split(int P, int K, int N, int sms) {
    const long long ctas = (long long)P * K, want = 8LL * sms;
    if (ctas <= 0 || ctas >= want) return 1;
    const long long smax = std::max(1, N * (N / 2 + 1) / (32 * kRedWarps));
    return (int)std::min((want + ctas - 1) / ctas, smax);
}

int reduction_split(int P, int K, int N, int sms) {
    const long long warps = (long long)P * K, want = 8LL * sms;
    if (warps <= 0 || warps >= want) return 1;
    const long long smax = std::max(1, N * (N / 2 + 1) / 128);
    return (int)std::min((want + warps - 1) / warps, smax);
}

cudaError_t launch_loss_combine(const double* lpart, int S, double* loss, int P, cudaStream_t s, bool chain) {
    if (P == 0) return cudaSuccess;
    return launch_chained(chain, loss_combine_kernel, (P + 127) / 128, 128, 0, s, lpart, S, loss, P);
}

}  // namespace mfbd_dev
