// Line transforms held by one lane (N <= 64) or a lane pair (N = 96, 128), for
// the patch images of the mosaic and the aligned 64 px spectra: a line of N
// points is held by S = 1 or 2 lanes, L = N / S points each; a register FFT of L
// points on the decimated samples x[S n + s] of each lane s and, for S = 2, one
// radix-2 stage across the lane pair by shuffles, leaving X[s L + k] in lane s.
#pragma once

#include <cstdint>

#include "fft_reg.cuh"
#include "mfbd_device.cuh"

namespace mfbd_dev {
namespace linefft {

using fftreg::cadd;
using fftreg::cconj;
using fftreg::cscale;
using fftreg::csub;

template <int N>
struct Geo {
    static constexpr int S = N > 64 ? 2 : 1;  // lanes per line
    static constexpr int L = N / S;           // points per lane
    static constexpr int NH = N / 2 + 1;
    static constexpr int LINES = 64;          // lines per round of a 64 S-thread group
    static constexpr int THREADS = LINES * S;
};

__device__ __forceinline__ float2 shfl_xor2(float2 v, int m) {
    return make_float2(__shfl_xor_sync(0xffffffffu, v.x, m), __shfl_xor_sync(0xffffffffu, v.y, m));
}

// Forward (DIR = -1) line transform, decimation in time: lane s holds
// x[S n + s] on entry and X[s L + k] on exit.
template <int N, int DIR>
__device__ __forceinline__ void line_fft(float2 (&v)[Geo<N>::L], int sub) {
    constexpr int S = Geo<N>::S, L = Geo<N>::L;
    fftreg::fft_line<L, DIR>(v);
    if constexpr (S == 2) {
        fftreg::static_for<0, L>([&](auto kk) {
            constexpr int k = decltype(kk)::value;
            const float2 t = sub ? fftreg::twmul<N, k, DIR>(v[k]) : v[k];  // lane 1: W^k O[k]
            const float2 o = shfl_xor2(t, 1);
            v[k] = sub ? csub(o, t) : cadd(t, o);
        });
    }
}

// Conjugate partner conj Z[(N - kx) mod N] of element K of this lane (which
// holds kx = sub L + K after line_fft). With S = 2 it comes from the pair
// lane by a shuffle that every lane of the warp executes; the callers take
// one partner at a time so that no second register array is live.
template <int N, int K>
__device__ __forceinline__ float2 conj_partner(const float2 (&v)[Geo<N>::L]) {
    constexpr int S = Geo<N>::S, L = Geo<N>::L;
    if constexpr (S == 1) return cconj(v[(L - K) % L]);
    else if constexpr (K == 0) return cconj(v[0]);  // kx = 0 or N/2: its own partner
    else return cconj(shfl_xor2(v[L - K], 1));
}

}  // namespace linefft
}  // namespace mfbd_dev
