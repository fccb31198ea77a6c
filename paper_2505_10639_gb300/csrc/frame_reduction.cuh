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

// Frame reduction of one (patch, object), any patch size: the residual form of
// Eq. 12 in FP32 with FP64 where it would cancel, Kahan sums per lane; writes
// the object (Eq. 11) when `obj` is not null and the adjoint seeds
// G_j = -w_j conj(O) (D_j - O H_j) over H_j.
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

// One warp takes the 32 / FS frequencies f0, f0 + 1, ... and then every fstep
// further on; lane q (32 / FS) + i holds frames q ceil(J / FS), ... of
// frequency i, and the FS lanes of a frequency add their sums by shuffles. The
// returned sum covers the lane's share. Outside the OTF support H vanishes and
// G with it: neither is read or written there (the passes of the larger sizes
// do not store or load them either), which at pupils of 0.35 to 0.5 N px leaves
// 40 to 80 % of the half spectrum.
//
// HBM is the floor (D once, H and G once on the support); what it needs is
// loads in flight and no second read: a frequency's frames are loaded once, all
// at once, into the registers of its lanes (J <= HOLD FS), or (HOLD = 0, any J)
// in chunks of kChunk frames, twice; both add a lane's frames in order, so FS
// alone decides the bits. Lanes outside the support take the same
// way with their loads of H predicated off: a path of their own, which most
// warps would run as well as the other, was slower (96 px 0.081 -> 0.100 ms).
// EXPL: the object-inferring loss (r.oin), FS = 1.
template <int HOLD, int FS, bool EXPL = false>
__device__ __forceinline__ double reduce_lane(const RedPtr& r, int f0, int fstep) {
    static_assert(FS == 1 || !EXPL, "the object-inferring loss is not split over lanes");
    constexpr int kChunk = 8, kF = 32 / FS;
    const int N = r.N, NH = N / 2 + 1, half = N * NH, J = r.J;
    const unsigned dstride = (unsigned)N * r.spec_ld;  // J * dstride < 2^32
    const float gam = (float)r.gamma;
    const int lane = threadIdx.x & 31, q = FS > 1 ? lane / kF : 0;
    const int jq = (J + FS - 1) / FS, jb = q * jq, nj = FS > 1 ? max(0, min(jq, J - jb)) : J;  // this lane's frames
    KahanSum acc;
    for (int fb = f0; fb < half; fb += fstep) {
        const bool live = fb + lane % kF < half;
        if (FS == 1 && !live) break;
        const int f = live ? fb + lane % kF : half - 1;
        const int ky = f / NH, kx = f - ky * NH;
        const size_t doff = (size_t)ky * r.spec_ld + kx;
        const float2 *dp0 = r.d + doff, *dp = dp0 + (unsigned)jb * dstride;
        float2 *hp0 = r.h + f, *hp = hp0 + (unsigned)jb * (unsigned)half;
        const float* wp = r.w + jb;
        const bool sup = wbit(r.supp, r.sw, ky, kx), seed = sup && f != 0;
        const float twice = (kx == 0 || kx == N / 2) ? 1.f : 2.f;
        float2 o = EXPL ? r.oin[doff] : make_float2(0.f, 0.f), g = make_float2(gam * o.x, gam * o.y);
        float t = 0.f;
        constexpr int kHeld = HOLD > 0 ? HOLD : 1;
        float2 d[kHeld], h[kHeld];
        float wv[kHeld];
        if constexpr (HOLD > 0) {
#pragma unroll
            for (int j = 0; j < HOLD; ++j) {
                const bool in = j < nj;
                d[j] = in ? dp[(unsigned)j * dstride] : make_float2(0.f, 0.f);
                h[j] = in && sup ? hp[(unsigned)j * (unsigned)half] : make_float2(0.f, 0.f);
                wv[j] = in ? wp[j] : 0.f;
            }
        }
        if (EXPL && sup) {  // the object is given
            if constexpr (HOLD > 0)
                t = explicit_held<HOLD>(J, d, h, wv, dp, dstride, hp, half, r.w, r.gamma, seed, o, g);
            else t = explicit_frequency(J, dp, dstride, hp, half, r.w, r.gamma, seed, o, g);
        } else {
            float2 num = make_float2(0.f, 0.f);
            float e = 0.f, qs = 0.f;
            auto gather = [&](float2 d, float2 h, float wj) {
                num.x += wj * (d.x * h.x + d.y * h.y);
                num.y += wj * (d.y * h.x - d.x * h.y);
                e += wj * (d.x * d.x + d.y * d.y);
                qs += wj * (h.x * h.x + h.y * h.y);
            };
            auto scatter = [&](float2 d, float2 h, float wj, int j) {
                const float2 res = csub(d, cmul(o, h));
                t += wj * (res.x * res.x + res.y * res.y);
                if (sup && live)
                    hp[(unsigned)j * (unsigned)half] = seed ? cscale(cmul(cconj(o), res), -wj) : make_float2(0.f, 0.f);
            };
            // false where the residual cancels (seed frequencies only)
            auto solve = [&]() {
                if constexpr (EXPL) {
                    return true;  // outside the support: the data's energy, O as given
                } else {
#pragma unroll
                    for (int off = kF; off < 32; off <<= 1) {
                        num.x += __shfl_xor_sync(0xffffffffu, num.x, off);
                        num.y += __shfl_xor_sync(0xffffffffu, num.y, off);
                        e += __shfl_xor_sync(0xffffffffu, e, off);
                        qs += __shfl_xor_sync(0xffffffffu, qs, off);
                    }
                    qs += gam;
                    const float invq = 1.0f / qs;
                    o = cscale(num, invq);
                    const float t_est = e - (num.x * num.x + num.y * num.y) * invq;
                    return !(seed && t_est < kCancel * e);
                }
            };
            bool fine;
            if constexpr (HOLD > 0) {
#pragma unroll
                for (int j = 0; j < HOLD; ++j)
                    if (j < nj) gather(d[j], h[j], wv[j]);
                fine = solve();
                if (fine) {
#pragma unroll
                    for (int j = 0; j < HOLD; ++j)
                        if (j < nj) scatter(d[j], h[j], wv[j], j);
                }
            } else {
                auto chunks = [&](bool on, auto&& use) {
#pragma unroll 1
                    for (int j0 = 0; j0 < nj; j0 += kChunk) {
                        float2 d[kChunk], h[kChunk];
                        float wv[kChunk];
#pragma unroll
                        for (int c = 0; c < kChunk; ++c) {
                            const bool in = on && j0 + c < nj;
                            d[c] = in ? dp[(unsigned)(j0 + c) * dstride] : make_float2(0.f, 0.f);
                            h[c] = in && sup ? hp[(unsigned)(j0 + c) * (unsigned)half] : make_float2(0.f, 0.f);
                            wv[c] = in ? wp[j0 + c] : 0.f;
                        }
#pragma unroll
                        for (int c = 0; c < kChunk; ++c)
                            if (j0 + c < nj) use(d[c], h[c], wv[c], j0 + c);
                    }
                };
                chunks(true, [&](float2 d, float2 h, float wj, int) { gather(d, h, wj); });
                const float own = e;  // this lane's share
                fine = solve();
                if (fine) {  // outside the support the residual is the data
                    chunks(sup, scatter);
                    if (!sup) t = own;
                }
            }
            if (!fine) {
                t = 0.f;
                if (q == 0 && live) fp64_frequency(J, dp0, dstride, hp0, half, r.w, r.gamma, true, t, o);
            } else if (q == 0) {
                t += gam * (o.x * o.x + o.y * o.y);
            }
        }
        if (!live) continue;
        acc.add(twice * t);
        if (q != 0) continue;
        if (r.obj) {
            r.obj[doff] = o;
            if (r.spec_ld == N && kx > 0 && kx < N / 2) r.obj[(size_t)((N - ky) % N) * N + (N - kx)] = cconj(o);
        }
        if (EXPL && r.gobj) {
            r.gobj[doff] = g;
            if (r.spec_ld == N && kx > 0 && kx < N / 2) r.gobj[(size_t)((N - ky) % N) * N + (N - kx)] = cconj(g);
        }
    }
    return (double)acc.s - (double)acc.c;
}

// Sum over a CTA of WARPS warps in a fixed order (lanes by a butterfly, then
// the warps in order), returned by thread 0. `part`: WARPS doubles of shared
// memory, free again after the caller's next barrier.
template <int WARPS>
__device__ __forceinline__ double cta_sum(double v, double* part) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = v;
    __syncthreads();
    double tot = 0.0;
    if (threadIdx.x == 0)
        for (int w = 0; w < WARPS; ++w) tot += part[w];
    return tot;
}

}  // namespace reduction
}  // namespace mfbd_dev
