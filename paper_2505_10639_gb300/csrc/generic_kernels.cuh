// Pass kernels of one problem for patch sizes other than 64 (48, 96, 128),
// and for 64 px plans outside the fused kernel's range (more than 12 frames,
// pupil boxes over 37 px, recompute, on request): one CTA per unit (patch, object, frame),
// persistent over the units. The passes themselves (Sec. 3.1, Eqs. 20-22 and
// their adjoint) are in lane_passes.cuh. Each patch size is instantiated in a
// translation unit of its own (generic_n48.cu ... generic_n128.cu) so that
// they compile in parallel.
#pragma once

#include <algorithm>

#include "chained.cuh"
#include "mfbd_internal.h"
#include "lane_passes.cuh"

namespace mfbd_dev {

namespace generic_detail {

namespace {

using namespace lanepass;

// CTAs per SM that the register budget is set for: two to three times 8 warps
// at 80-128 registers a thread. Timed with one more or one less at each size
// (forward / adjoint / recomputing adjoint, ms): 12,800 units of 128 px 0.668 /
// 0.868 / 1.002 with 2 (0.948 / 1.148 / 1.533 with 3); 2,904 units of 96 px
// 0.107 / 0.129 / 0.161 with 3, 4, 3 (0.111 / 0.146 / 0.164 with 4, 3, 4); 6,750
// units of 64 px 0.101 / 0.128 with 6 (0.102 / 0.132 with 5), 23,064 units 0.333
// / 0.414 (0.326 / 0.411); 23,064 units of 48 px 0.193 / 0.214 with 12 (0.195 /
// 0.226 with 9).
template <int N, bool ADJ, bool RECOMPUTE>
constexpr int kMinCtas = N == 128 ? 2 : N == 96 ? (ADJ && !RECOMPUTE ? 4 : 3) : N == 64 ? 6 : 12;

template <int N>
__device__ __forceinline__ UnitPtr unit_ptr(const GenericParams& prm, long long u) {
    const int J = prm.J, K = prm.K;
    const int j = (int)(u % J);
    const long long pk = u / J;
    const int k = (int)(pk % K);
    const long long p = pk / K;
    const GenericObj& ob = prm.obj[k];
    const long long img = (p * J + j) * (long long)ob.W * ob.W;
    UnitPtr q;
    q.phi = prm.phi + ob.phi_off + img;
    q.gphi = prm.gphi + ob.phi_off + img;
    q.h = prm.gscr + (size_t)u * N * Geo<N>::NH;
    q.pf = prm.pscr ? prm.pscr + (size_t)u * N * N : nullptr;
    q.W = ob.W;
    q.inv_z = ob.inv_z;
    q.cmask = ob.cmask;
    q.csupp = ob.csupp;
    return q;
}

// Warps of a CTA: half of a pass's N / 8 groups of four lines, so that every
// warp runs two of them.
template <int N>
constexpr int kWarps = N / 16;

template <int N, int S, bool OTF_ONLY>
__global__ void __launch_bounds__(32 * kWarps<N>, kMinCtas<N, false, false>) generic_forward_kernel(const GenericParams prm) {
    extern __shared__ __align__(16) unsigned char gsm[];
    float2* tw = reinterpret_cast<float2*>(gsm);
    float2* E = tw + Twiddles<N>::kElems;
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    load_twiddles<N>(tw, threadIdx.x, 32 * kWarps<N>);
    chain_wait();  // no chain_release: the reduction, resident early, would run with these CTAs' L1 split
    __syncthreads();
    const long long units = (long long)prm.P * prm.K * prm.J;
    for (long long u = blockIdx.x; u < units; u += gridDim.x)
        unit_forward<N, S, kWarps<N>, OTF_ONLY>(unit_ptr<N>(prm, u), E, tw, w, lane, CtaBar{});
}

template <int N, int S, bool RECOMPUTE>
__global__ void __launch_bounds__(32 * kWarps<N>, kMinCtas<N, true, RECOMPUTE>) generic_adjoint_kernel(const GenericParams prm) {
    extern __shared__ __align__(16) unsigned char gsm[];
    float2* tw = reinterpret_cast<float2*>(gsm);
    float2* E = tw + Twiddles<N>::kElems;
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // RECOMPUTE: the column transforms of P, in this CTA's global buffer (kept
    // in L2) so that shared memory holds one exchange buffer
    float2* E2 = RECOMPUTE ? prm.e2scr + (size_t)blockIdx.x * N * prm.es2 : nullptr;
    load_twiddles<N>(tw, threadIdx.x, 32 * kWarps<N>);
    chain_wait();
    chain_release();
    __syncthreads();
    const long long units = (long long)prm.P * prm.K * prm.J;
    for (long long u = blockIdx.x; u < units; u += gridDim.x) {
        // the next unit's seed (and phase) from HBM into L2 under this unit: 12,800
        // units of 128 px 1.038 -> 1.000 ms, 6,750 of 64 px 0.138 -> 0.129; not where
        // it was slower (96 px 0.130 -> 0.133, 48 px 0.216 -> 0.221, 128 px with the
        // field kept 0.866 -> 0.892)
        if (N == 64 || (N == 128 && RECOMPUTE))
            if (threadIdx.x == 32 * kWarps<N> - 1 && u + gridDim.x < units) {
                const UnitPtr n = unit_ptr<N>(prm, u + gridDim.x);
                prefetch_l2(n.h, 8u * N * Geo<N>::NH);
                if (RECOMPUTE && n.W % 2 == 0) prefetch_l2(n.phi, 4u * n.W * n.W);  // rows of whole 16-byte groups
            }
        unit_adjoint<N, S, kWarps<N>, RECOMPUTE>(unit_ptr<N>(prm, u), E, E2, prm.es2, tw, w, lane, CtaBar{});
    }
}

template <class Kern>
cudaError_t persistent_ctas(Kern kern, int threads, size_t smem, int sms, long long* ctas) {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, threads, smem);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) return cudaErrorInvalidConfiguration;
    *ctas = (long long)sms * per_sm;
    return cudaSuccess;
}

template <class Kern>
cudaError_t launch_persistent(Kern kern, int threads, size_t smem, long long units, int sms, const GenericParams& prm,
                              cudaStream_t s, int max_ctas = 0) {
    long long ctas = 0;
    cudaError_t e = persistent_ctas(kern, threads, smem, sms, &ctas);
    if (e != cudaSuccess) return e;
    if (max_ctas > 0 && ctas > max_ctas) ctas = max_ctas;
    if (ctas > units) ctas = units;
    return launch_chained(prm.chain, kern, (int)ctas, threads, smem, s, prm);
}

}  // namespace

}  // namespace generic_detail

// f(integral constant of the buffer's row stride)
template <int N, class F>
auto with_stride(bool half_box, F&& f) {
    using lanepass::Geo;
    return half_box ? f(fftreg::IC<Geo<N>::S_HALF>{}) : f(fftreg::IC<Geo<N>::S_FULL>{});
}

template <int N>
int generic_adjoint_ctas_n(bool half_box, int sms) {
    using namespace generic_detail;
    return with_stride<N>(half_box, [&](auto s) {
        constexpr int S = decltype(s)::value;
        long long c = 0;
        const cudaError_t e = persistent_ctas(generic_adjoint_kernel<N, S, true>, 32 * kWarps<N>,
                                              generic_smem(N, half_box), sms, &c);
        return e == cudaSuccess ? (int)c : 0;
    });
}

template <int N>
cudaError_t launch_generic_forward_n(const GenericParams& prm, int sms, cudaStream_t s) {
    using namespace generic_detail;
    const long long units = (long long)prm.P * prm.K * prm.J;
    const size_t smem = generic_smem(N, prm.half_box);
    return with_stride<N>(prm.half_box, [&](auto st) {
        constexpr int S = decltype(st)::value;
        return prm.otf_only
                   ? launch_persistent(generic_forward_kernel<N, S, true>, 32 * kWarps<N>, smem, units, sms, prm, s)
                   : launch_persistent(generic_forward_kernel<N, S, false>, 32 * kWarps<N>, smem, units, sms, prm, s);
    });
}

template <int N>
cudaError_t launch_generic_adjoint_n(const GenericParams& prm, int sms, cudaStream_t s) {
    using namespace generic_detail;
    const long long units = (long long)prm.P * prm.K * prm.J;
    const size_t smem = generic_smem(N, prm.half_box);
    return with_stride<N>(prm.half_box, [&](auto st) {
        constexpr int S = decltype(st)::value;
        return prm.pscr == nullptr ? launch_persistent(generic_adjoint_kernel<N, S, true>, 32 * kWarps<N>, smem, units,
                                                       sms, prm, s, prm.e2_ctas)
                                   : launch_persistent(generic_adjoint_kernel<N, S, false>, 32 * kWarps<N>, smem,
                                                       units, sms, prm, s);
    });
}

}  // namespace mfbd_dev
