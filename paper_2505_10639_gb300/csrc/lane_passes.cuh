// Per-unit passes of the CTA-per-unit kernels (patch sizes 48, 64, 96, 128;
// generic_kernels.cuh).
//
// The passes are those of Sec. 3.1, Eqs. 20-22 and their adjoint, on lines of
// eight lanes (lane8.cuh), four lines per warp, WARPS warps on one unit
// (patch, object, frame). The 2-D transforms go through one N x S exchange
// buffer in shared memory in three passes each way; within a pass every line
// reads and writes only its own storage, so a warp runs its lines without a
// barrier and the group's barrier stands between passes:
//   PUPIL  box columns of P = exp(i phi), zero-padded, along y;
//   ROWS   row pairs (i, i + N/2): the two field rows p = F P, the PSF rows
//          |p|^2 / (N^2 n_pup), their transform as one complex row;
//   OTF    half-spectrum columns: the two rows' half spectra split on load,
//          transformed along y, masked by the OTF support, H(0) = 1;
// and back:
//   SEED   conj of the columns of the seed G along y, the row pairs packed on
//          store;
//   ROWS   row pairs: the g_q rows (2 Re / (N^2 n_pup)) from the packed row,
//          then conj of the rows of F^H(g_q p) on the box columns;
//   ADJ    box columns along y -> 2 Im(conj(P) G_P) on the pupil.
// Half-spectrum line 0 packs the real columns 0 and N/2.
//
// The field p is kept in global memory by the forward passes, or (RECOMPUTE)
// its column transforms are redone by the adjoint into a global buffer of the
// CTA (L2) and each row just before it is needed.
//
// What bounds it: instruction issue and shared-memory wavefronts, about level
// (a 128-point line is some 3,400 lane instructions and 4 KB of shared-memory
// traffic). Measured against one or two lanes a line (64 registers of data a
// lane, 8-12 warps an SM, stalled on instruction fetch), forward + adjoint:
// 2,904 units of 96 px 0.402 + 0.508 -> 0.107 + 0.129 ms; 12,800 units of
// 128 px with the field recomputed 1.95 + 2.74 -> 0.60 + 1.00 ms, kept
// 2.68 + 2.64 -> 0.67 + 0.87 ms; 23,064 units of 64 px 1.35 + 1.07 -> 0.33 +
// 0.41 ms.
#pragma once

#include <cstdint>

#include "lane8.cuh"
#include "mfbd_device.cuh"

namespace mfbd_dev {
namespace lanepass {

using namespace lane8;

// Barrier of the threads that work on one unit.
struct CtaBar {
    __device__ __forceinline__ void operator()() const { __syncthreads(); }
};

// A column of up to 128 mask bits, shifted so that bit<B>() is row t + B.
struct ColumnBits {
    uint32_t w[4];
    __device__ __forceinline__ ColumnBits(const uint64_t* col, bool act, int t) {
        const uint64_t a = act ? col[0] : 0ull, b = act ? col[1] : 0ull;
        const uint32_t r[5] = {(uint32_t)a, (uint32_t)(a >> 32), (uint32_t)b, (uint32_t)(b >> 32), 0u};
#pragma unroll
        for (int i = 0; i < 4; ++i) w[i] = __funnelshift_r(r[i], r[i + 1], t);
    }
    __device__ __forceinline__ bool bit(int b) const { return (w[b >> 5] >> (b & 31)) & 1u; }
};

// L2 prefetch of `bytes` (a multiple of 16) from a 16-byte aligned address.
__device__ __forceinline__ void prefetch_l2(const void* p, uint32_t bytes) {
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(__cvta_generic_to_global(p)), "r"(bytes) : "memory");
}

// Everything one unit's passes touch.
struct UnitPtr {
    const float* phi;       // [W][W] box phase
    float* gphi;            // [W][W] dL/dphi (0 outside the pupil)
    float2* h;              // [N][N/2+1]: OTF, then the adjoint seed; read on the OTF support only
    float2* pf;             // [N][N] field rows, or null (recomputed)
    int W;
    float inv_z;            // 1 / (N^2 n_pup)
    const uint64_t* cmask;  // [W][2] box column c: bit y = pupil pixel at box (y, c)
    const uint64_t* csupp;  // [N/2+1][2] column kx: bit ky = OTF support
};

// Lines of a warp: columns c0 .. c0 + 3 with a line's lanes four apart, or row
// pairs p0 .. p0 + 3 (in the order p0, p0 + 2, p0 + 1, p0 + 3) with a line's
// lanes adjacent; both orders keep the accesses of a half warp on 16 banks.
struct ColLanes {
    int t, c;
    __device__ __forceinline__ explicit ColLanes(int lane) : t(lane >> 2), c(lane & 3) {}
};
struct RowLanes {
    int t, p;
    __device__ __forceinline__ explicit RowLanes(int lane)
        : t(lane & 7), p((((lane >> 3) & 1) << 1) | (lane >> 4)) {}
};

// Inputs of a line that are not zero by construction: the pupil box takes at
// most the first half of a line when the buffer is the half-box one.
template <int N, int S>
struct BoxPoints {
    static constexpr bool kHalf = S == Geo<N>::S_HALF;
    static constexpr int kQ = kHalf ? N / 16 : N / 8;
};

// PUPIL. Columns of the transform go to the buffer E, or (dst != null) to
// dst [N][ld], the buffer then only carrying the exchange.
template <int N, int S, int WARPS>
__device__ __forceinline__ void pass_pupil(const UnitPtr& q, float2* E, const float2* table, int w, int lane, float2* dst,
                                           int ld) {
    constexpr int R = Geo<N>::R, M2 = Geo<N>::M2, Q = BoxPoints<N, S>::kQ;
    const ColLanes cl(lane);
    const int t = cl.t;
    const LaneTwiddles<N> tw(table, t);
    for (int c0 = 4 * w; c0 < q.W; c0 += 4 * WARPS) {
        const int c = c0 + cl.c;
        const bool act = c < q.W;
        const ColumnBits in(q.cmask + 2 * c, act, t);
        float2 a[Q], u[8 * M2];
#pragma unroll
        for (int i = 0; i < Q; ++i)
            a[i] = in.bit(8 * i) ? expi(q.phi[(t + 8 * i) * q.W + c]) : make_float2(0.f, 0.f);
        const ColLine<N, S> ln{E + c, 0};
        strided_to_blocked<N>(ln, a, u, tw, t);
        if (dst == nullptr) {
            __syncwarp();
#pragma unroll
            for (int m = 0; m < M2; ++m)
                if (R % 8 == 0 || t + 8 * m < R)
#pragma unroll
                    for (int k = 0; k < 8; ++k) E[(t + 8 * m + R * k) * S + c] = u[8 * m + k];
        } else if (act) {
#pragma unroll
            for (int m = 0; m < M2; ++m)
                if (R % 8 == 0 || t + 8 * m < R)
#pragma unroll
                    for (int k = 0; k < 8; ++k) dst[(t + 8 * m + R * k) * ld + c] = u[8 * m + k];
        }
    }
}

// Forward passes of one unit -> q.h (and the field q.pf when kept); OTF_ONLY:
// q.h is also written (0) outside the OTF support. E: the group's N x S
// exchange buffer; w, lane: warp of the group and lane. Ends with the group's
// barrier.
template <int N, int S, int WARPS, bool OTF_ONLY, class Bar>
__device__ __forceinline__ void unit_forward(const UnitPtr& q, float2* E, const float2* table, int w, int lane, Bar bar) {
    constexpr int R = Geo<N>::R, M2 = Geo<N>::M2, NH = Geo<N>::NH, Q = BoxPoints<N, S>::kQ;
    // skipping the stores outside the support costs a branch each, which pays at
    // the larger sizes only (128 px forward 0.655 -> 0.603 ms, 48 px 0.193 -> 0.214)
    constexpr bool kAll = OTF_ONLY || N <= 64;
    pass_pupil<N, S, WARPS>(q, E, table, w, lane, nullptr, 0);
    bar();
    {  // ROWS
        const RowLanes rl(lane);
        const int t = rl.t;
        const LaneTwiddles<N> tw(table, t);
#pragma unroll 1
        for (int p0 = 4 * w; p0 < N / 2; p0 += 4 * WARPS) {
            const int i = p0 + rl.p;
            const RowLine<N, S> ln{E + i * S};
            float2 x0[Q], x1[Q], z[8 * M2];
#pragma unroll
            for (int e = 0; e < Q; ++e) {
                const bool in = t + 8 * e < q.W;
                x0[e] = in ? E[i * S + t + 8 * e] : make_float2(0.f, 0.f);
                x1[e] = in ? E[(i + N / 2) * S + t + 8 * e] : make_float2(0.f, 0.f);
            }
            {
                float2 u[8 * M2];
                strided_to_blocked<N>(ln, x0, u, tw, t);
#pragma unroll
                for (int m = 0; m < M2; ++m) {
                    if (q.pf && (R % 8 == 0 || t + 8 * m < R))
#pragma unroll
                        for (int k = 0; k < 8; ++k) q.pf[i * N + t + 8 * m + R * k] = u[8 * m + k];
#pragma unroll
                    for (int k = 0; k < 8; ++k)
                        z[8 * m + k].x = (u[8 * m + k].x * u[8 * m + k].x + u[8 * m + k].y * u[8 * m + k].y) * q.inv_z;
                }
            }
            {
                float2 u[8 * M2];
                strided_to_blocked<N>(ln, x1, u, tw, t);
#pragma unroll
                for (int m = 0; m < M2; ++m) {
                    if (q.pf && (R % 8 == 0 || t + 8 * m < R))
#pragma unroll
                        for (int k = 0; k < 8; ++k) q.pf[(i + N / 2) * N + t + 8 * m + R * k] = u[8 * m + k];
#pragma unroll
                    for (int k = 0; k < 8; ++k)
                        z[8 * m + k].y = (u[8 * m + k].x * u[8 * m + k].x + u[8 * m + k].y * u[8 * m + k].y) * q.inv_z;
                }
            }
            float2 a[R];
            blocked_to_strided<N>(ln, z, a, tw, t);
            __syncwarp();
#pragma unroll
            for (int e = 0; e < R; ++e) ln.block(e)[t] = a[e];
        }
    }
    bar();
    {  // OTF
        const ColLanes cl(lane);
        const int t = cl.t;
        const LaneTwiddles<N> tw(table, t);
#pragma unroll 1
        for (int l0 = 4 * w; l0 < N / 2; l0 += 4 * WARPS) {
            const int kx = l0 + cl.c;
            const ColLine<N, S> ln{E + kx, kx ? N / 2 - 2 * kx : 0};
            float2 v[R], u[8 * M2];
#pragma unroll
            for (int e = 0; e < R / 2; ++e) {
                // X[kx] and X[N - kx] (line 0: X[0] and X[N/2]) of the rows i + i (i + N/2)
                const float2 a = ln.block(e)[t * S], b = ln.block(e + R / 2)[t * S];
                if (kx == 0) {
                    v[e] = make_float2(a.x, b.x);
                    v[e + R / 2] = make_float2(a.y, b.y);
                } else {
                    v[e] = make_float2(0.5f * (a.x + b.x), 0.5f * (a.y - b.y));
                    v[e + R / 2] = make_float2(0.5f * (a.y + b.y), 0.5f * (b.x - a.x));
                }
            }
            strided_to_blocked<N>(ln, v, u, tw, t);
            const ColumnBits in(q.csupp + 2 * kx, true, t);
            if (l0 == 0) {  // the warp of line 0 splits its packed columns through the line's storage
                const ColumnBits in2(q.csupp + 2 * (N / 2), kx == 0, t);
                __syncwarp();
                if (kx == 0) {
#pragma unroll
                    for (int m = 0; m < M2; ++m)
                        if (R % 8 == 0 || t + 8 * m < R)
#pragma unroll
                            for (int k = 0; k < 8; ++k) E[(t + 8 * m + R * k) * S] = u[8 * m + k];
                }
                __syncwarp();
                if (kx == 0) {
#pragma unroll
                    for (int m = 0; m < M2; ++m)
                        if (R % 8 == 0 || t + 8 * m < R)
#pragma unroll
                            for (int k = 0; k < 8; ++k) {
                                const int ky = t + 8 * m + R * k;
                                const float2 z = u[8 * m + k], c = E[(ky ? N - ky : 0) * S];
                                const float2 hn = make_float2(0.5f * (z.y + c.y), 0.5f * (c.x - z.x));
                                const bool sup = in2.bit(8 * m + R * k);
                                if constexpr (kAll) q.h[ky * NH + N / 2] = sup ? hn : make_float2(0.f, 0.f);
                                else if (sup) q.h[ky * NH + N / 2] = hn;
                                u[8 * m + k] = ky ? make_float2(0.5f * (z.x + c.x), 0.5f * (z.y - c.y))
                                                  : make_float2(1.f, 0.f);
                            }
                }
            }
#pragma unroll
            for (int m = 0; m < M2; ++m)
                if (R % 8 == 0 || t + 8 * m < R)
#pragma unroll
                    for (int k = 0; k < 8; ++k) {
                        const int ky = t + 8 * m + R * k;
                        const bool sup = in.bit(8 * m + R * k);
                        if constexpr (kAll) q.h[ky * NH + kx] = sup ? u[8 * m + k] : make_float2(0.f, 0.f);
                        else if (sup) q.h[ky * NH + kx] = u[8 * m + k];
                    }
        }
    }
    bar();
}

// One row of F^H(g p) on the box columns: u the field row (blocked), g the
// g_q row; conj(g p) transformed back to strided.
template <int N, int S, int Q>
__device__ __forceinline__ void adjoint_row(const RowLine<N, S>& ln, float2 (&u)[8 * Geo<N>::M2],
                                            const float (&g)[8 * Geo<N>::M2], float2 (&out)[Q],
                                            const LaneTwiddles<N>& tw, int t) {
#pragma unroll
    for (int e = 0; e < 8 * Geo<N>::M2; ++e) u[e] = make_float2(g[e] * u[e].x, -g[e] * u[e].y);
    blocked_to_strided<N>(ln, u, out, tw, t);
}

// Adjoint passes of one unit: q.h (the seed G) -> q.gphi (0 in the box
// outside the pupil). E2 (row stride es2): RECOMPUTE's global buffer for the
// column transforms of P. Ends with the group's barrier.
template <int N, int S, int WARPS, bool RECOMPUTE, class Bar>
__device__ __forceinline__ void unit_adjoint(const UnitPtr& q, float2* E, float2* E2, int es2, const float2* table, int w,
                                             int lane, Bar bar) {
    constexpr int R = Geo<N>::R, M2 = Geo<N>::M2, NH = Geo<N>::NH, Q = BoxPoints<N, S>::kQ;
    if constexpr (RECOMPUTE) {
        pass_pupil<N, S, WARPS>(q, E, table, w, lane, E2, es2);
        bar();
    }
    {  // SEED
        const ColLanes cl(lane);
        const int t = cl.t;
        const LaneTwiddles<N> tw(table, t);
#pragma unroll 1
        for (int l0 = 4 * w; l0 < N / 2; l0 += 4 * WARPS) {
            const int kx = l0 + cl.c;
            const ColLine<N, S> ln{E + kx, kx ? N / 2 - 2 * kx : 0};
            float2 a[R], u[8 * M2];
            const ColumnBits in(q.csupp + 2 * kx, true, t);
#pragma unroll
            for (int e = 0; e < R; ++e)
                a[e] = N <= 64 || in.bit(8 * e) ? cconj(q.h[(t + 8 * e) * NH + kx]) : make_float2(0.f, 0.f);
            if (kx == 0) {  // conj(G_0 + i G_N/2)
                const ColumnBits in2(q.csupp + 2 * (N / 2), true, t);
#pragma unroll
                for (int e = 0; e < R; ++e) {
                    const float2 b = N <= 64 || in2.bit(8 * e) ? q.h[(t + 8 * e) * NH + N / 2] : make_float2(0.f, 0.f);
                    a[e] = make_float2(a[e].x - b.y, a[e].y - b.x);
                }
            }
            strided_to_blocked<N>(ln, a, u, tw, t);
            __syncwarp();
            // rows y and y + N/2 of T = conj(u): conj of T_y + i T_(y+N/2) at kx, and its mirror at N - kx
#pragma unroll
            for (int m = 0; m < M2; ++m)
                if (R % 8 == 0 || t + 8 * m < R)
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const float2 u0 = u[8 * m + k], u1 = u[8 * m + k + 4];
                        float2 lo = make_float2(u0.x + u1.y, u0.y - u1.x), hi = make_float2(u0.x - u1.y, -u0.y - u1.x);
                        if (kx == 0) {  // T_0 and T_N/2 are the real and imaginary parts
                            lo = make_float2(u0.x, -u1.x);
                            hi = make_float2(-u0.y, u1.y);
                        }
                        float2* row = E + (t + 8 * m + R * k) * S;
                        row[kx] = lo;
                        row[(N / 2) * S + (kx ? N / 2 - kx : 0)] = hi;
                    }
        }
    }
    bar();
    {  // ROWS
        const RowLanes rl(lane);
        const int t = rl.t;
        const LaneTwiddles<N> tw(table, t);
        const float sc = 2.0f * q.inv_z;
#pragma unroll 1
        for (int p0 = 4 * w; p0 < N / 2; p0 += 4 * WARPS) {
            const int i = p0 + rl.p;
            const RowLine<N, S> ln{E + i * S};
            float g0[8 * M2], g1[8 * M2];
            {
                float2 a[R], u[8 * M2];
#pragma unroll
                for (int e = 0; e < R; ++e) a[e] = ln.block(e)[t];
                strided_to_blocked<N>(ln, a, u, tw, t);
#pragma unroll
                for (int e = 0; e < 8 * M2; ++e) {
                    g0[e] = u[e].x * sc;
                    g1[e] = -u[e].y * sc;
                }
            }
            float2 x0[Q], x1[Q], u[8 * M2];
            auto field_row = [&](int y) {
                if constexpr (RECOMPUTE) {
                    float2 a[Q];
#pragma unroll
                    for (int e = 0; e < Q; ++e)
                        a[e] = t + 8 * e < q.W ? E2[y * es2 + t + 8 * e] : make_float2(0.f, 0.f);
                    strided_to_blocked<N>(ln, a, u, tw, t);
                } else {
#pragma unroll
                    for (int m = 0; m < M2; ++m)
#pragma unroll
                        for (int k = 0; k < 8; ++k)
                            u[8 * m + k] = (R % 8 == 0 || t + 8 * m < R) ? q.pf[y * N + t + 8 * m + R * k]
                                                                         : make_float2(0.f, 0.f);
                }
            };
            field_row(i);
            adjoint_row<N, S>(ln, u, g0, x0, tw, t);
            field_row(i + N / 2);
            adjoint_row<N, S>(ln, u, g1, x1, tw, t);
            __syncwarp();
#pragma unroll
            for (int e = 0; e < Q; ++e)
                if (t + 8 * e < q.W) {
                    E[i * S + t + 8 * e] = x0[e];
                    E[(i + N / 2) * S + t + 8 * e] = x1[e];
                }
        }
    }
    bar();
    {  // ADJ: dL/dphi = 2 Im(conj(P) G_P) on the pupil
        const ColLanes cl(lane);
        const int t = cl.t;
        const LaneTwiddles<N> tw(table, t);
#pragma unroll 1
        for (int c0 = 4 * w; c0 < q.W; c0 += 4 * WARPS) {
            const int c = c0 + cl.c;
            const bool act = c < q.W;
            const ColumnBits in(q.cmask + 2 * c, act, t);
            float2 a[R], u[8 * M2];
#pragma unroll
            for (int e = 0; e < R; ++e) a[e] = E[(t + 8 * e) * S + c];
            const ColLine<N, S> ln{E + c, 0};
            strided_to_blocked<N>(ln, a, u, tw, t);
#pragma unroll
            for (int m = 0; m < M2; ++m)
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    const int y = t + 8 * m + R * k;
                    if (BoxPoints<N, S>::kHalf && k >= 4) continue;  // y >= N/2 >= W
                    if (act && y < q.W && (R % 8 == 0 || t + 8 * m < R)) {
                        float gv = 0.f;
                        if (in.bit(8 * m + R * k)) {
                            const float2 p = expi(q.phi[y * q.W + c]), g = u[8 * m + k];
                            gv = 2.0f * (-p.x * g.y - p.y * g.x);  // G_P = conj(g)
                        }
                        q.gphi[y * q.W + c] = gv;
                    }
                }
        }
    }
    bar();
}

}  // namespace lanepass
}  // namespace mfbd_dev
