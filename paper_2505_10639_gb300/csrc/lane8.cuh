// N-point complex transforms of a line held by eight lanes of a warp
// (N = 48, 64, 96, 128), exchanged through the line's own shared-memory
// storage.
//
// With R = N / 8, lane t of a line holds either
//   strided  a[q] = x[t + 8 q],                q < R, or
//   blocked  u[8 m + k2] = X[t + 8 m + R k2],  k2 < 8, m < ceil(R / 8)
// (blocked elements with t + 8 m >= R do not exist). strided_to_blocked
// transforms one into the other (decimation in time: an R-point transform
// per lane, the exchange with the twiddles W_N^(t k1) on one of its sides,
// 8-point transforms);
// blocked_to_strided is its mirror (8-point transforms, twiddles, exchange,
// an R-point transform). A line that was transformed one way can be
// multiplied pointwise and transformed again the other way without a change
// of layout.
//
// Why eight lanes: a lane that holds a whole 64-point line (or half a
// 128-point one) needs 170-255 registers, so an SM runs 8-12 warps, and the
// unrolled 64-point network is about 1,060 instructions per copy; eight lanes
// hold 6 to 16 points each (32 registers of data at 128), an SM runs two to
// three times as many warps, and each network is a few hundred instructions.
// The price is one shared-memory exchange per transform: N complex written
// and read, 2 N / 16 wavefronts of 128 bytes.
//
// The exchange uses N slots in blocks of eight; element (k1, t) sits in block
// k1 at position t ^ (k1 mod 8). Writes go through the lanes' t at a fixed k1,
// reads at a fixed t through the lanes' k1; with the storage strides of
// RowLine and ColLine (S = 4 mod 8 complex) a half warp's 16 accesses fall on
// 16 different 8-byte banks both times.
#pragma once

#include "fft_reg.cuh"

namespace mfbd_dev {
namespace lane8 {

using fftreg::cadd;
using fftreg::cconj;
using fftreg::cmul;
using fftreg::cscale;
using fftreg::csub;
using fftreg::static_for;
using fftreg::twmul;

// Forward 3-point transform.
MFBD_HD void dft3(float2& x0, float2& x1, float2& x2) {
    constexpr float s3 = -0.86602540378443864676f;  // -sin(2 pi / 3)
    const float2 sum = cadd(x1, x2), dif = csub(x1, x2);
    const float2 m = make_float2(x0.x - 0.5f * sum.x, x0.y - 0.5f * sum.y);
    const float2 r = make_float2(-s3 * dif.y, s3 * dif.x);
    x0 = cadd(x0, sum);
    x1 = cadd(m, r);
    x2 = csub(m, r);
}

// Forward R-point transform in registers, natural order in and out: a power
// of two, or 3 P points (P prime to 3) by the prime-factor map: with
// n = P n1 + 3 n2 the factor W_R^(n k) is W_3^(n1 k) W_P^(n2 k), so three
// P-point transforms over n2 and P 3-point ones over n1 are the whole of it,
// the output k in (k mod 3, k mod P). Without the rounded twiddles that
// x[3 n + r] needs between the two, the error of a whole line falls from
// 8.4e-8 to 7.9e-8 (48 points) and from 8.9e-8 to 8.5e-8 (96).
template <int R>
MFBD_HD void dft(float2 (&a)[R]) {
    if constexpr (R == 3) {
        dft3(a[0], a[1], a[2]);
    } else if constexpr (R % 3 == 0) {
        constexpr int P = R / 3;
        static_assert(P % 3 != 0, "the map needs coprime factors");
        float2 b[3][P];
        static_for<0, R>([&](auto i) {
            constexpr int n1 = decltype(i)::value / P, n2 = decltype(i)::value % P;
            b[n1][n2] = a[(P * n1 + 3 * n2) % R];
        });
        dft<P>(b[0]);
        dft<P>(b[1]);
        dft<P>(b[2]);
        static_for<0, P>([&](auto kk) {
            constexpr int k = decltype(kk)::value;
            dft3(b[0][k], b[1][k], b[2][k]);
        });
        static_for<0, R>([&](auto kk) { a[decltype(kk)::value] = b[decltype(kk)::value % 3][decltype(kk)::value % P]; });
    } else if constexpr (R == 4 || R == 16) {
        fftreg::fft4<R, -1>(a);
    } else if constexpr (R == 8) {  // two 4-point transforms of the even and the odd points
        float2 e[4], o[4];
        static_for<0, 4>([&](auto i) {
            e[decltype(i)::value] = a[2 * decltype(i)::value];
            o[decltype(i)::value] = a[2 * decltype(i)::value + 1];
        });
        fftreg::fft4<4, -1>(e);
        fftreg::fft4<4, -1>(o);
        static_for<0, 4>([&](auto kk) {
            constexpr int k = decltype(kk)::value;
            const float2 t = twmul<8, k, -1>(o[k]);
            a[k] = cadd(e[k], t);
            a[k + 4] = csub(e[k], t);
        });
    } else {
        fftreg::fft<R, -1>(a);
    }
}

// dft<R> of a line whose points R/2.. are zero: the even outputs are the
// R/2-point transform of a, the odd ones that of a[q] W_R^q.
template <int R>
MFBD_HD void dft_half_in(const float2 (&x)[R / 2], float2 (&a)[R]) {
    float2 e[R / 2], o[R / 2];
    static_for<0, R / 2>([&](auto qq) {
        constexpr int q = decltype(qq)::value;
        e[q] = x[q];
        o[q] = twmul<R, q, -1>(x[q]);
    });
    dft<R / 2>(e);
    dft<R / 2>(o);
    static_for<0, R / 2>([&](auto kk) {
        a[2 * decltype(kk)::value] = e[decltype(kk)::value];
        a[2 * decltype(kk)::value + 1] = o[decltype(kk)::value];
    });
}

// The first R/2 outputs of dft<R>.
template <int R>
MFBD_HD void dft_half_out(const float2 (&a)[R], float2 (&x)[R / 2]) {
    float2 e[R / 2], o[R / 2];
    static_for<0, R / 2>([&](auto qq) {
        e[decltype(qq)::value] = a[2 * decltype(qq)::value];
        o[decltype(qq)::value] = a[2 * decltype(qq)::value + 1];
    });
    dft<R / 2>(e);
    dft<R / 2>(o);
    static_for<0, R / 2>([&](auto kk) {
        constexpr int k = decltype(kk)::value;
        x[k] = cadd(e[k], twmul<R, k, -1>(o[k]));
    });
}

// Where a transform takes its twiddles W_N^(j k1) (j < 8, k1 < R). N = 64 and
// 128 multiply on the blocked side of the exchange in both directions: one set
// per lane, taken from shared memory once per pass into registers, serves
// every transform of the pass (against reading them at each transform, which
// is a third of the shared-memory wavefronts: 128 px forward passes 0.603 ->
// 0.590 ms, 64 px 0.350 -> 0.337). At 48 and 96 the register budget has no
// room for that (96 px 0.109 -> 0.111, adjoint 0.129 -> 0.142 ms): they read
// them at each transform, 16 bytes at a time, on the side that has fewer.
template <int N>
constexpr bool kTwiddlesInRegisters = N % 3 != 0;

// Twiddle tables: in registers, [j][k1]; else for strided_to_blocked, per pair
// of k1, the lanes' j ([k1 / 2][j][k1 % 2]) and for blocked_to_strided, per
// pair of j, the lanes' k1 ([j / 2][k1][j % 2]).
template <int N>
struct Twiddles {
    static constexpr int R = N / 8;
    static constexpr int kElems = kTwiddlesInRegisters<N> ? N : 2 * N;
    float v[2 * kElems];
    constexpr Twiddles() : v{} {
        for (int j = 0; j < 8; ++j)
            for (int k1 = 0; k1 < R; ++k1) {
                const fftreg::SinCos sc = fftreg::sincos_2pi(j * k1, N);
                if (kTwiddlesInRegisters<N>) {
                    put(j * R + k1, sc);
                } else {
                    put(((k1 / 2) * 8 + j) * 2 + k1 % 2, sc);
                    put(N + ((j / 2) * R + k1) * 2 + j % 2, sc);
                }
            }
    }
    constexpr void put(int i, const fftreg::SinCos& sc) {
        v[2 * i] = (float)sc.c;
        v[2 * i + 1] = (float)-sc.s;
    }
};

template <int N>
__device__ const Twiddles<N> kTwiddles = Twiddles<N>();

template <int N>
struct Geo {
    static constexpr int R = N / 8;
    static constexpr int M2 = (R + 7) / 8;      // groups of 8 blocked elements per lane
    static constexpr int NH = N / 2 + 1;
    // Row strides (complex) of the N x S exchange buffer: pupil boxes up to
    // N / 2 px, and any box.
    static constexpr int S_HALF = N / 2 + 4, S_FULL = N + 4;
};

// Copies the twiddles (Twiddles<N>::kElems complex) to shared memory; the
// caller synchronises.
template <int N>
__device__ __forceinline__ void load_twiddles(float2* tw, int t, int threads) {
    for (int i = t; i < Twiddles<N>::kElems / 2; i += threads)
        reinterpret_cast<float4*>(tw)[i] = reinterpret_cast<const float4*>(kTwiddles<N>.v)[i];
}

// A lane's twiddles for one pass.
template <int N>
struct LaneTwiddles {
    static constexpr int R = Geo<N>::R;
    float2 w[kTwiddlesInRegisters<N> ? 7 * Geo<N>::M2 : 1];  // W_N^(j (t + 8 m)) at [7 m + j - 1]
    const float4* table;
    __device__ __forceinline__ LaneTwiddles(const float2* shared, int t)
        : table(reinterpret_cast<const float4*>(shared)) {
        if constexpr (kTwiddlesInRegisters<N>) {
#pragma unroll
            for (int m = 0; m < Geo<N>::M2; ++m)
#pragma unroll
                for (int j = 1; j < 8; ++j) w[7 * m + j - 1] = shared[j * R + t + 8 * m];
        }
    }
    // strided side of strided_to_blocked
    __device__ __forceinline__ void strided(float2 (&a)[R], int t) const {
        if constexpr (!kTwiddlesInRegisters<N>) {
#pragma unroll
            for (int p = 0; p < R / 2; ++p) {
                const float4 v = table[p * 8 + t];
                if (p > 0) a[2 * p] = cmul(a[2 * p], make_float2(v.x, v.y));
                a[2 * p + 1] = cmul(a[2 * p + 1], make_float2(v.z, v.w));
            }
        }
    }
    // blocked side, group m: of strided_to_blocked, and (BACK) of blocked_to_strided
    template <bool BACK>
    __device__ __forceinline__ void blocked(float2 (&b)[8], int m, int k1) const {
        if constexpr (kTwiddlesInRegisters<N>) {
#pragma unroll
            for (int j = 1; j < 8; ++j) b[j] = cmul(b[j], w[7 * m + j - 1]);
        } else if constexpr (BACK) {
#pragma unroll
            for (int p = 0; p < 4; ++p) {
                const float4 v = table[N / 2 + p * R + k1];
                if (p > 0) b[2 * p] = cmul(b[2 * p], make_float2(v.x, v.y));
                b[2 * p + 1] = cmul(b[2 * p + 1], make_float2(v.z, v.w));
            }
        }
    }
};

// Storage of a line in the N x S buffer, in R blocks of 8 elements: element x
// of block b sits at block(b) + x * kStep.
//
// RowLine: the N complex of the row pair (i, i + N/2): elements 0 .. N/2 - 1
// in row i, the rest in row i + N/2.
template <int N, int S>
struct RowLine {
    static constexpr int kStep = 1;
    float2* lo;  // row i
    __device__ __forceinline__ float2* block(int b) const { return lo + b * 8 + (b >= N / 16 ? (N / 2) * S - N / 2 : 0); }
};
// ColLine: element y in row y; rows N/2.. `shift` columns further.
template <int N, int S>
struct ColLine {
    static constexpr int kStep = S;
    float2* top;  // row 0 of the column
    int shift;
    __device__ __forceinline__ float2* block(int b) const { return top + b * 8 * S + (b >= N / 16 ? shift : 0); }
};

// strided a (already transformed over q by dft<R>) -> blocked u.
template <int N, class Line>
__device__ __forceinline__ void finish_blocked(const Line& ln, float2 (&a)[N / 8], float2 (&u)[8 * Geo<N>::M2],
                                               const LaneTwiddles<N>& tw, int t) {
    constexpr int R = Geo<N>::R, M2 = Geo<N>::M2;
    tw.strided(a, t);
    __syncwarp();  // every lane of the line has read what the storage held
#pragma unroll
    for (int k1 = 0; k1 < R; ++k1) ln.block(k1)[(t ^ (k1 & 7)) * Line::kStep] = a[k1];
    __syncwarp();
#pragma unroll
    for (int m = 0; m < M2; ++m) {
        float2 b[8];
        const int k1 = t + 8 * m;
        if (R % 8 == 0 || k1 < R) {
            const float2* src = ln.block(k1);
#pragma unroll
            for (int j = 0; j < 8; ++j) b[j] = src[(j ^ t) * Line::kStep];
            tw.template blocked<false>(b, m, k1);
        } else {
#pragma unroll
            for (int j = 0; j < 8; ++j) b[j] = make_float2(0.f, 0.f);
        }
        dft<8>(b);
#pragma unroll
        for (int j = 0; j < 8; ++j) u[8 * m + j] = b[j];
    }
}

template <int N, class Line>
__device__ __forceinline__ void strided_to_blocked(const Line& ln, float2 (&a)[N / 8], float2 (&u)[8 * Geo<N>::M2],
                                                   const LaneTwiddles<N>& tw, int t) {
    dft<N / 8>(a);
    finish_blocked<N>(ln, a, u, tw, t);
}

// The same for a line whose elements N/2.. are zero (x: the first R / 2).
template <int N, class Line>
__device__ __forceinline__ void strided_to_blocked(const Line& ln, const float2 (&x)[N / 16],
                                                   float2 (&u)[8 * Geo<N>::M2], const LaneTwiddles<N>& tw, int t) {
    float2 a[N / 8];
    dft_half_in<N / 8>(x, a);
    finish_blocked<N>(ln, a, u, tw, t);
}

// blocked u -> strided a before its R-point transform.
template <int N, class Line>
__device__ __forceinline__ void start_strided(const Line& ln, const float2 (&u)[8 * Geo<N>::M2], float2 (&a)[N / 8],
                                              const LaneTwiddles<N>& tw, int t) {
    constexpr int R = Geo<N>::R, M2 = Geo<N>::M2;
    __syncwarp();
#pragma unroll
    for (int m = 0; m < M2; ++m) {
        const int k1 = t + 8 * m;
        if (R % 8 == 0 || k1 < R) {
            float2 b[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) b[j] = u[8 * m + j];
            dft<8>(b);
            tw.template blocked<true>(b, m, k1);
            float2* dst = ln.block(k1);
#pragma unroll
            for (int j = 0; j < 8; ++j) dst[(j ^ t) * Line::kStep] = b[j];
        }
    }
    __syncwarp();
#pragma unroll
    for (int k1 = 0; k1 < R; ++k1) a[k1] = ln.block(k1)[(t ^ (k1 & 7)) * Line::kStep];
}

template <int N, class Line>
__device__ __forceinline__ void blocked_to_strided(const Line& ln, const float2 (&u)[8 * Geo<N>::M2],
                                                   float2 (&a)[N / 8], const LaneTwiddles<N>& tw, int t) {
    start_strided<N>(ln, u, a, tw, t);
    dft<N / 8>(a);
}

// The same, the first half of the outputs only.
template <int N, class Line>
__device__ __forceinline__ void blocked_to_strided(const Line& ln, const float2 (&u)[8 * Geo<N>::M2],
                                                   float2 (&x)[N / 16], const LaneTwiddles<N>& tw, int t) {
    float2 a[N / 8];
    start_strided<N>(ln, u, a, tw, t);
    dft_half_out<N / 8>(a, x);
}

}  // namespace lane8
}  // namespace mfbd_dev
