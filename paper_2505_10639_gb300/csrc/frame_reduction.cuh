// Frame reduction of one (patch, object) at any patch size (Sec. 2.2.1, Eqs.
// 11-12, and the adjoint seeds), shared by the single-problem kernels
// (generic_kernels.cu) and the batched persistent kernel (batch_kernels.cuh).
#pragma once

#include <cstdint>

#include "fft_reg.cuh"
#include "mfbd_device.cuh"

namespace mfbd_dev {
namespace reduction {

using fftreg::cadd;
using fftreg::cconj;
using fftreg::cmul;
using fftreg::cscale;
using fftreg::csub;

__device__ __forceinline__ bool wbit(const uint32_t* rows, int words, int r, int c) {
    return (rows[r * words + (c >> 5)] >> (c & 31)) & 1u;
}

// Frame reduction of one (patch, object) by one warp, any patch size: the
// residual form of Eq. 12 in FP32 with FP64 where it would cancel, Kahan sums
// per lane and an FP64 warp combine; writes the object (Eq. 11) when `obj`
// is not null and the adjoint seeds G_j = -w_j conj(O) (D_j - O H_j) over H_j.
// Returns the (patch, object) loss on every lane.
struct RedPtr {
    int N, J, spec_ld;      // spectra / object row stride: N/2 + 1 or N
    double gamma;
    const float2* d;        // frame 0 of D; frames N spec_ld apart
    float2* h;              // frame 0 of H; frames N (N/2 + 1) apart
    const float* w;         // [J] frame weights
    const uint32_t* supp;   // [N][sw] OTF support rows
    int sw;
    float2* obj = nullptr;           // [N][spec_ld] or null
    const float2* oin = nullptr;     // object-inferring loss: the given object [N][spec_ld], else null
    float2* gobj = nullptr;          // with oin: dL/dconj(O) [N][spec_ld], or null
};

// Lanes take the frequencies f0 + lane, f0 + lane + fstep, ... (fstep a
// multiple of 32: several warps can share one (patch, object)); the returned
// sum covers this warp's frequencies.
__device__ __forceinline__ double reduce_warp(const RedPtr& r, int lane, int f0 = 0, int fstep = 32) {
    const int N = r.N, NH = N / 2 + 1, half = N * NH, J = r.J;
    const size_t dstride = (size_t)N * r.spec_ld;
    const float gam = (float)r.gamma;
    KahanSum acc;
    for (int f = f0 + lane; f < half; f += fstep) {
        const int ky = f / NH, kx = f - ky * NH;
        const size_t doff = (size_t)ky * r.spec_ld + kx;
        const float2* dp = r.d + doff;
        float2* hp = r.h + f;
        const bool seed = (f != 0) && wbit(r.supp, r.sw, ky, kx);
        if (r.oin) {  // object-inferring loss: the object is given
            float2 g;
            const float t = explicit_frequency(J, dp, dstride, hp, half, r.w, r.gamma, seed, r.oin[doff], g);
            acc.add((kx == 0 || kx == N / 2) ? t : 2.0f * t);
            if (r.gobj) {
                r.gobj[doff] = g;
                if (r.spec_ld == N && kx > 0 && kx < N / 2) r.gobj[(size_t)((N - ky) % N) * N + (N - kx)] = cconj(g);
            }
            continue;
        }
        float2 num = make_float2(0.f, 0.f), o;
        float e = 0.f, qs = 0.f, tval;
#pragma unroll 4
        for (int j = 0; j < J; ++j) {
            const float2 d = dp[(size_t)j * dstride];
            const float2 h = hp[(size_t)j * half];
            const float wj = r.w[j];
            num.x += wj * (d.x * h.x + d.y * h.y);
            num.y += wj * (d.y * h.x - d.x * h.y);
            e += wj * (d.x * d.x + d.y * d.y);
            qs += wj * (h.x * h.x + h.y * h.y);
        }
        qs += gam;
        const float invq = 1.0f / qs;
        o = cscale(num, invq);
        const float t_est = e - (num.x * num.x + num.y * num.y) * invq;
        if (f != 0 && t_est < kCancel * e) {
            fp64_frequency(J, dp, dstride, hp, half, r.w, r.gamma, seed, tval, o);
        } else {
            float tsum = 0.f;
#pragma unroll 4
            for (int j = 0; j < J; ++j) {
                const float2 d = dp[(size_t)j * dstride];
                const float2 h = hp[(size_t)j * half];
                const float wj = r.w[j];
                const float2 res = csub(d, cmul(o, h));
                tsum += wj * (res.x * res.x + res.y * res.y);
                hp[(size_t)j * half] = seed ? cscale(cmul(cconj(o), res), -wj) : make_float2(0.f, 0.f);
            }
            tval = tsum + gam * (o.x * o.x + o.y * o.y);
        }
        acc.add((kx == 0 || kx == N / 2) ? tval : 2.0f * tval);
        if (r.obj) {
            r.obj[doff] = o;
            if (r.spec_ld == N && kx > 0 && kx < N / 2) r.obj[(size_t)((N - ky) % N) * N + (N - kx)] = cconj(o);
        }
    }
    double v = (double)acc.s - (double)acc.c;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    return v;
}

}  // namespace reduction
}  // namespace mfbd_dev
