// Batched persistent kernel: the whole loss + gradient of an uneven batch of
// problems (patch sizes 48, 64, 96, 128; objects, frames and modes per
// problem) in one launch, or (staged) in one launch per kind of item.
//
// The work is a list of items, each of one kind (BatchKind), those of a whole
// patch cut into parts: P, the phases
// phi = c_k B_k a of every object and frame of a patch (Sec. 3.1, Eq. 22);
// F, the forward passes of a unit (Eqs. 20-21 and the OTF); R, the frame
// reduction of a patch (Sec. 2.2.1, Eqs. 11-12, and the adjoint seeds); A,
// the adjoint passes of a unit (-> dL/dphi); G, the modal adjoint of a patch
// (dL/da = sum_k c_k B_k^T dL/dphi_k). CTAs (256 threads) take items in list
// order from a ticket counter. In one-launch mode an item first waits for
// the items it depends on (P -> F -> R -> A -> G of the same patch), which
// all come earlier in the list: the holder of the smallest unfinished ticket
// never waits, so the launch always progresses. Every wait is bounded: on
// giving up it sets the error flag and the item is skipped. In staged mode
// the host launches each kind's range of the list separately and nothing
// waits.
//
// F and A items of patches of N <= 64 px cover up to two consecutive units
// (k J + j) of one patch: four warps run one unit each on their own exchange
// buffer and named barrier. Larger patches use all eight warps on one unit.
// The passes are those of lane_passes.cuh. Measured on 500 drawn problems
// (15,788 units): 6.76 ms with a unit per warp (N <= 64) or per 128 threads
// and one or two lanes a line, 3.59 ms with these, 1.98 ms with P, R and G in
// parts; staged P 0.87 -> 0.16, F 1.17 -> 0.51, R 2.04 -> 0.36, A 1.52 -> 0.68, G
// 1.53 -> 0.25 ms.
//
// Data written by one CTA and read by another inside the launch (phases,
// OTFs and seeds, fields, dL/dphi) is published by the writer's barrier,
// fence and counter increment and acquired by the reader's thread 0
// (ld.acquire.gpu, fence) before its CTA barrier: the PTX memory model then
// orders the readers' plain loads after the writes. Every per-unit and
// per-patch scratch block also starts on a 256-byte boundary, so no cache
// line is shared by blocks of different writers.
//
// The kernel is instantiated for its two register budgets in
// batch_kernel_v2.cu and batch_kernel_v3.cu, which compile in parallel.
#pragma once

#include "batch_internal.h"
#include "frame_reduction.cuh"
#include "lane_passes.cuh"

#include <algorithm>


namespace mfbd_dev {

namespace {

using namespace lanepass;
using namespace reduction;

constexpr long long kSpinLimit = 1ll << 22; // polls of a dependency counter (~1 s)

__device__ __forceinline__ int ld_acquire(const int* p) {
    int v;
    asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// Thread 0: wait until *c >= target. false (and the error flag set) when the
// wait gives up or another CTA has given up already.
__device__ bool wait_ctr(const int* c, int target, int* err) {
    for (long long it = 0; it < kSpinLimit; ++it) {
        if (ld_acquire(c) >= target) {
            __threadfence();
            return true;
        }
        if (*(volatile int*)err) return false;
        __nanosleep(200);
    }
    atomicExch(err, 1);
    return false;
}

__device__ __forceinline__ long long unit_stride_phi(int W) { return ((long long)W * W + 63) & ~63ll; }

// Pointers of unit (patch p, object k, frame j) of problem pr.
template <int N>
__device__ __forceinline__ UnitPtr batch_unit(const BatchParams& prm, const BatchProblem& pr, int p, int k, int j) {
    const BatchObj& ob = pr.obj[k];
    const long long u = ((long long)p * pr.K + k) * pr.J + j;
    const long long phi = pr.phi_off + (long long)p * pr.phi_patch + ob.phi_koff + (long long)j * unit_stride_phi(ob.W);
    UnitPtr q;
    q.phi = prm.phi + phi;
    q.gphi = prm.gphi + phi;
    q.h = prm.gscr + pr.gscr_off + u * N * Geo<N>::NH;
    q.pf = prm.pscr + pr.pscr_off + u * N * N;
    q.W = ob.W;
    q.inv_z = ob.inv_z;
    q.cmask = ob.cmask;
    q.csupp = ob.csupp;
    return q;
}

// Barrier of a group of `n` threads (a multiple of 32) on named barrier `id`.
struct GroupBar {
    int id, n;
    __device__ __forceinline__ void operator()() const {
        asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(n) : "memory");
    }
};

// Twiddles of every patch size, one after the other at the start of the
// CTA's shared memory (complex elements).
template <int N>
constexpr int kTwOff = N == 48 ? 0 : N == 64 ? 96 : N == 96 ? 160 : 352;
static_assert(kTwOff<64> == Twiddles<48>::kElems && kTwOff<96> == kTwOff<64> + Twiddles<64>::kElems &&
                  kTwOff<128> == kTwOff<96> + Twiddles<96>::kElems && kTwOff<128> + Twiddles<128>::kElems == kBatchTwiddles, "room for the four tables");

// F or A item: two units of one patch, four warps each (N <= 64), or one unit
// on the whole CTA (N = 96, 128).
template <int N, bool HALF, bool ADJ>
__device__ void item_unit(const BatchParams& prm, const BatchProblem& pr, const BatchItem& it, float2* smem) {
    constexpr int S = HALF ? Geo<N>::S_HALF : Geo<N>::S_FULL;
    constexpr int kUnits = N <= 64 ? kSmallUnits : 1, kW = kBT / 32 / kUnits;
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, g = w / kW;
    if (g > it.extra) return;
    const int kj = it.kj + g, k = kj / pr.J, j = kj - k * pr.J;
    const UnitPtr q = batch_unit<N>(prm, pr, it.patch, k, j);
    const float2* tw = smem + kTwOff<N>;
    float2* E = smem + kBatchTwiddles + (size_t)g * N * S;
    auto run = [&](auto bar) {
        if constexpr (ADJ) unit_adjoint<N, S, kW, false>(q, E, nullptr, 0, tw, w - g * kW, lane, bar);
        else if ((prm.kinds >> BK_RED) & 1) unit_forward<N, S, kW, false>(q, E, tw, w - g * kW, lane, bar);
        else unit_forward<N, S, kW, true>(q, E, tw, w - g * kW, lane, bar);  // the OTFs alone
    };
    if constexpr (kUnits > 1) run(GroupBar{1 + g, 32 * kW});
    else run(CtaBar{});
}

// P part: phi_kj[i] = c_k sum_m a_j[m] B_k[m][i] on every box pixel i for one
// object and kJC frames of the patch, their coefficients staged in shared
// memory mode-major ([m][kJC]: two 16-byte loads per mode).
__device__ void item_proj(const BatchParams& prm, const BatchProblem& pr, int p, int part, float* sa) {
    const int t = threadIdx.x, J = pr.J, M = pr.M;
    const int k = part % pr.K, jc = part / pr.K * kJC, nj = min(kJC, J - jc);
    const float* a = prm.coeffs + pr.coeff_off + (size_t)p * J * M;
    for (int e = t; e < kJC * M; e += kBT) {
        const int m = e / kJC, jj = e - m * kJC;
        sa[e] = jj < nj ? a[(size_t)(jc + jj) * M + m] : 0.f;
    }
    __syncthreads();
    const float4* sa4 = reinterpret_cast<const float4*>(sa);
    const BatchObj& ob = pr.obj[k];
    const int npix = ob.W * ob.W;
    const long long us = unit_stride_phi(ob.W);
    float* phi = prm.phi + pr.phi_off + (long long)p * pr.phi_patch + ob.phi_koff + jc * us;
    for (int i = t; i < npix; i += kBT) {
        float acc[kJC];
#pragma unroll
        for (int jj = 0; jj < kJC; ++jj) acc[jj] = 0.f;
#pragma unroll 8
        for (int m = 0; m < M; ++m) {
            const float b = ob.bm[(size_t)m * npix + i];
            const float4 c0 = sa4[2 * m], c1 = sa4[2 * m + 1];
            acc[0] = fmaf(c0.x, b, acc[0]);
            acc[1] = fmaf(c0.y, b, acc[1]);
            acc[2] = fmaf(c0.z, b, acc[2]);
            acc[3] = fmaf(c0.w, b, acc[3]);
            acc[4] = fmaf(c1.x, b, acc[4]);
            acc[5] = fmaf(c1.y, b, acc[5]);
            acc[6] = fmaf(c1.z, b, acc[6]);
            acc[7] = fmaf(c1.w, b, acc[7]);
        }
#pragma unroll
        for (int jj = 0; jj < kJC; ++jj)
            if (jj < nj) phi[jj * us + i] = ob.scale * acc[jj];
    }
}

// G part: grad[j][m] = sum_k c_k sum_i dL/dphi_kj[i] B_k[m][i] for kJC frames
// and kGM modes (one per lane), the objects added in order. The warps take an
// eighth of an object's pixels each and add their sums in warp order through
// shared memory (kBT / 32 x kJC x kGM floats).
__device__ void item_grad(const BatchParams& prm, const BatchProblem& pr, int p, int part, float* sums) {
    constexpr int kW = kBT / 32;
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, J = pr.J, M = pr.M;
    const int mt = (M + kGM - 1) / kGM, jc = part / mt * kJC, nj = min(kJC, J - jc);
    const int m0 = part % mt * kGM, m = min(m0 + lane, M - 1);
    float acc[kJC];
#pragma unroll
    for (int jj = 0; jj < kJC; ++jj) acc[jj] = 0.f;
    for (int k = 0; k < pr.K; ++k) {
        const BatchObj& ob = pr.obj[k];
        const int npix = ob.W * ob.W;
        const long long us = unit_stride_phi(ob.W);
        const float* g = prm.gphi + pr.phi_off + (long long)p * pr.phi_patch + ob.phi_koff + jc * us;
        const float* row[kJC];
#pragma unroll
        for (int jj = 0; jj < kJC; ++jj) row[jj] = g + min(jj, nj - 1) * us;
        const float* bt = ob.bt + m;
        float sum[kJC];
#pragma unroll
        for (int jj = 0; jj < kJC; ++jj) sum[jj] = 0.f;
        // four pixels per step: one 16-byte load of each frame's dL/dphi (rows
        // are 256-byte aligned), the same for all lanes; then the tail
        const int n4 = npix & ~3, per = (n4 / 4 + kW - 1) / kW * 4;
        const int i1 = min(n4, (w + 1) * per);
#pragma unroll 2
        for (int i = w * per; i < i1; i += 4) {
            const float b0 = bt[(size_t)i * ob.ldt], b1 = bt[(size_t)(i + 1) * ob.ldt];
            const float b2 = bt[(size_t)(i + 2) * ob.ldt], b3 = bt[(size_t)(i + 3) * ob.ldt];
#pragma unroll
            for (int jj = 0; jj < kJC; ++jj) {
                const float4 gv = *reinterpret_cast<const float4*>(row[jj] + i);
                float x = fmaf(gv.x, b0, sum[jj]);
                x = fmaf(gv.y, b1, x);
                x = fmaf(gv.z, b2, x);
                sum[jj] = fmaf(gv.w, b3, x);
            }
        }
        if (w == kW - 1)
            for (int i = n4; i < npix; ++i) {
                const float b = bt[(size_t)i * ob.ldt];
#pragma unroll
                for (int jj = 0; jj < kJC; ++jj) sum[jj] = fmaf(row[jj][i], b, sum[jj]);
            }
#pragma unroll
        for (int jj = 0; jj < kJC; ++jj) acc[jj] = fmaf(ob.scale, sum[jj], acc[jj]);
    }
#pragma unroll
    for (int jj = 0; jj < kJC; ++jj) sums[(w * kJC + jj) * kGM + lane] = acc[jj];
    __syncthreads();
    float* grad = prm.grad + pr.coeff_off + (size_t)p * J * M;
    for (int e = threadIdx.x; e < kJC * kGM; e += kBT) {
        const int jj = e / kGM, mm = m0 + e % kGM;
        float v = 0.f;
#pragma unroll
        for (int q = 0; q < kW; ++q) v += sums[q * kJC * kGM + e];
        if (jj < nj && mm < M) grad[(size_t)(jc + jj) * M + mm] = v;
    }
}

// R part: the CTA's threads share the part's frequencies of each object; the
// patch loss adds an object's warps in order, then the objects, then (the last
// part to arrive) the parts. The lanes that a frequency's frames are split over
// follow from J alone, so that every kernel variant sums in the same order (and
// the autotuner's choice cannot change the bits); HOLD, what the variant's
// register budget holds, only decides whether a lane keeps its frames (16) or
// reads them twice in chunks. (Splitting 9 to 16 frames over two lanes in the
// 80-register variant alone read them once, with other bits: 400 problems of 48
// and 64 px, for which that variant was the fastest, 812 us; now the other one
// is, 859 us.)
constexpr int kRedFrames = 16;  // frames of a frequency in a lane

template <int HOLD>
__device__ void item_reduce(const BatchParams& prm, const BatchProblem& pr, int p, int part, double* warps) {
    const int N = pr.N, NH = N / 2 + 1, J = pr.J, parts = red_parts(N);
    const size_t dstride = (size_t)N * NH;
    double tot = 0.0;
    for (int k = 0; k < pr.K; ++k) {
        const size_t unit0 = ((size_t)p * pr.K + k) * J;
        RedPtr r;
        r.N = N;
        r.J = J;
        r.spec_ld = NH;
        r.gamma = pr.gamma;
        r.d = prm.spectra + pr.spec_off + unit0 * dstride;
        r.h = prm.gscr + pr.gscr_off + unit0 * dstride;
        r.w = pr.weights + (size_t)k * J;
        r.supp = pr.obj[k].supp;
        r.sw = pr.sw;
        r.obj = prm.object ? prm.object + pr.obj_off + ((size_t)p * pr.K + k) * dstride : nullptr;
        auto share = [&](auto fs, auto hold) {
            constexpr int FS = decltype(fs)::value, kF = 32 / FS;
            return reduce_lane<decltype(hold)::value, FS>(r, kF * (kBT / 32 * part + (threadIdx.x >> 5)),
                                                          kF * (kBT / 32) * parts);
        };
        using fftreg::IC;
        constexpr int kFull = HOLD >= kRedFrames ? HOLD : 0;
        const double v = J <= HOLD             ? share(IC<1>{}, IC<HOLD>{})
                         : J <= kRedFrames     ? share(IC<1>{}, IC<kFull>{})
                         : J <= 2 * kRedFrames ? share(IC<2>{}, IC<kFull>{})
                                               : share(IC<1>{}, IC<0>{});
        tot += cta_sum<kBT / 32>(v, warps);
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        if (parts > 1) {
            const long long patch = pr.ctr_off + p;
            volatile double* lp = prm.lpart + patch * kMaxRedParts;
            lp[part] = tot;
            __threadfence();
            if (atomicAdd(prm.ctr + patch * BC_COUNT + BC_LOSS, 1) != parts - 1) return;
            __threadfence();
            tot = 0.0;
            for (int i = 0; i < parts; ++i) tot += lp[i];
        }
        prm.loss[pr.loss_off + p] = tot;
    }
}

template <bool HALF, bool ADJ>
__device__ void dispatch_unit(const BatchParams& prm, const BatchProblem& pr, const BatchItem& it, float2* smem) {
    switch (pr.N) {
        case 48: item_unit<48, HALF, ADJ>(prm, pr, it, smem); break;
        case 64: item_unit<64, HALF, ADJ>(prm, pr, it, smem); break;
        case 96: item_unit<96, HALF, ADJ>(prm, pr, it, smem); break;
        default: item_unit<128, HALF, ADJ>(prm, pr, it, smem); break;
    }
}

// MINB: CTAs per SM the register budget is set for (2: up to 128 registers a
// thread; 3: up to 80). The autotuner picks one. HALF: every pupil box of the
// batch is at most half its patch, and the exchange buffers are the half-box
// ones.
template <int MINB, bool HALF>
__global__ void __launch_bounds__(kBT, MINB) batch_kernel(const BatchParams prm) {
    extern __shared__ __align__(16) unsigned char bsm[];
    float2* smem = reinterpret_cast<float2*>(bsm);
    load_twiddles<48>(smem + kTwOff<48>, threadIdx.x, kBT);
    load_twiddles<64>(smem + kTwOff<64>, threadIdx.x, kBT);
    load_twiddles<96>(smem + kTwOff<96>, threadIdx.x, kBT);
    load_twiddles<128>(smem + kTwOff<128>, threadIdx.x, kBT);
    __shared__ int s_item, s_ok;
    __shared__ double warps[kBT / 32];
    float* scratch = reinterpret_cast<float*>(smem + kBatchTwiddles);  // of the P and G parts
    for (;;) {
        if (threadIdx.x == 0) s_item = atomicAdd(prm.ticket, 1);
        __syncthreads();
        const int i = s_item;
        if (i >= prm.n_items) break;
        const BatchItem it = prm.items[prm.item0 + i];
        const BatchProblem& pr = prm.probs[it.prob];
        int* ctr = prm.ctr + (pr.ctr_off + it.patch) * BC_COUNT;
        if (threadIdx.x == 0) {
            bool ok = true;
            if (prm.wait) {
                const int units = pr.K * pr.J;
                switch (it.kind) {
                    case BK_FWD: ok = wait_ctr(ctr + BC_PROJ, proj_parts(pr.K, pr.J), prm.err); break;
                    case BK_RED: ok = wait_ctr(ctr + BC_FWD, units, prm.err); break;
                    case BK_ADJ: ok = wait_ctr(ctr + BC_RED, red_parts(pr.N), prm.err); break;
                    case BK_GRAD: ok = wait_ctr(ctr + BC_ADJ, units, prm.err); break;
                    default: break;
                }
            }
            s_ok = ok;
        }
        __syncthreads();
        if (s_ok && ((prm.kinds >> it.kind) & 1)) {
            switch (it.kind) {
                case BK_PROJ: item_proj(prm, pr, it.patch, it.part, scratch); break;
                case BK_FWD: dispatch_unit<HALF, false>(prm, pr, it, smem); break;
                case BK_RED: item_reduce<MINB == 2 ? 16 : 8>(prm, pr, it.patch, it.part, warps); break;
                case BK_ADJ: dispatch_unit<HALF, true>(prm, pr, it, smem); break;
                default: item_grad(prm, pr, it.patch, it.part, scratch); break;
            }
        }
        __syncthreads();  // the item's writes precede the signal; s_item is free again
        if (prm.wait && threadIdx.x == 0 && it.kind != BK_GRAD) {
            __threadfence();
            const int n = (it.kind == BK_FWD || it.kind == BK_ADJ) ? 1 + it.extra : 1;
            const int slot = it.kind == BK_PROJ ? BC_PROJ : it.kind == BK_FWD ? BC_FWD : it.kind == BK_RED ? BC_RED
                                                                                                      : BC_ADJ;
            atomicAdd(ctr + slot, n);
        }
    }
}

}  // namespace

template <int MINB>
int batch_max_ctas_variant(size_t smem, bool half_box) {
    auto kern = half_box ? batch_kernel<MINB, true> : batch_kernel<MINB, false>;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) return 0;
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kBT, smem) != cudaSuccess) return 0;
    return per_sm;
}

template <int MINB>
cudaError_t launch_batch_variant(const BatchParams& prm, int ctas, size_t smem, cudaStream_t s) {
    if (prm.half_box) batch_kernel<MINB, true><<<ctas, kBT, smem, s>>>(prm);
    else batch_kernel<MINB, false><<<ctas, kBT, smem, s>>>(prm);
    return cudaGetLastError();
}

}  // namespace mfbd_dev
