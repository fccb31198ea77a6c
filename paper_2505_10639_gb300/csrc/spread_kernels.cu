// The fused evaluation for few (patch, object) pairs: a cluster of CTAs per
// pair instead of one CTA.
//
// fused_kernels.cu carries a pair on one SM, one warp and one lane per line
// for each frame: with fewer pairs than SMs the rest of the chip is idle and
// the pair takes some 50 us whatever its number of frames, most of it the
// latency of 64-point lines transformed in one lane. Here the frames of a pair
// are dealt to the CTAs of a cluster (two at most per CTA) and a line is held
// by four lanes, 16 points each, so that 256 threads run all 64 lines of a
// pass at once. The OTFs and seeds go through the plan's per-unit buffers
// (L2), the CTAs of a cluster meeting at the cluster barrier before and after
// the frame reduction, whose frequencies they share.
//
// The transforms and every elementwise step are those of the fused kernel and
// of the three-kernel path in the same order: object and dL/da agree with both
// bit for bit. So does the loss with the fused kernel's: every CTA puts the
// terms of its frequencies into the shared memory of the cluster's last one,
// which adds them in the order of the fused kernel's threads. For that the
// twiddle products across lanes round as the compiler contracts twmul's
// constant ones (fused_over_s; the pupil columns beyond 32, which the other
// kernels transform by fft64_quarters, go through it here).
// Stating those roundings in twmul itself would tie the kernels together by
// construction, but made the fused kernel 1 % slower.
#include "chained.cuh"
#include "fft_reg.cuh"
#include "mfbd_device.cuh"
#include "mfbd_internal.h"
#include "pass64.cuh"

#include <algorithm>

namespace mfbd_dev {

using fftreg::cadd;
using fftreg::cconj;
using fftreg::cscale;
using fftreg::csub;

namespace {

using namespace pass64;

constexpr int kSW = 8, kST = 32 * kSW;  // warps and threads of a CTA
constexpr int kQ = kN / 4;              // points of a line in a lane
constexpr int kMaxBox = 36;             // pupil boxes: at most five warps of columns
// Exchange buffer: element (y, x) at 68 y + 4 (y / 16) + x + x / 16. A half
// warp (four lines of four lanes) then falls on 16 different 8-byte banks for
// lines along x and along y, both where a lane's points are four apart (loads)
// and where they are sixteen apart between lanes (stores).
constexpr int kLd = 68, kBufElems = kN * kLd + 16;

__device__ __forceinline__ int row_base(int y) { return y * kLd + 4 * (y >> 4); }

// How twmul's v (c + i s) rounds, c and s being constants there: the real part
// fused over c v.x; the imaginary part over s v.x where |c| = |s| or c < 0 < s,
// else over c v.y.
constexpr bool fused_over_s(float c, float s) { return c == s || c == -s || (c < 0.f && s > 0.f); }

// fft4<64> of a line over four lanes: lane l holds x[4 n + l] on entry and
// X[k + 16 q] with q = split_q(l) on exit.
__device__ __forceinline__ void fft64_lanes(float2 (&a)[kQ], int l) {
    fftreg::fft4<kQ, -1>(a);
    fftreg::static_for<1, kQ>([&](auto kk) {
        constexpr int k = decltype(kk)::value;
        constexpr fftreg::SinCos w1 = fftreg::sincos_2pi(k, kN), w2 = fftreg::sincos_2pi(2 * k, kN),
                                 w3 = fftreg::sincos_2pi(3 * k, kN);
        constexpr float c1 = (float)w1.c, c2 = (float)w2.c, c3 = (float)w3.c;
        constexpr float n1 = (float)-w1.s, n2 = (float)-w2.s, n3 = (float)-w3.s;
        constexpr bool f1 = fused_over_s(c1, n1), f2 = fused_over_s(c2, n2), f3 = fused_over_s(c3, n3);
        const float c = l == 0 ? 1.f : l == 1 ? c1 : l == 2 ? c2 : c3;
        const float s = l == 0 ? 0.f : l == 1 ? n1 : l == 2 ? n2 : n3;
        const float2 v = a[k];
        float2 r = make_float2(__fmaf_rn(c, v.x, -__fmul_rn(s, v.y)), __fmaf_rn(c, v.y, __fmul_rn(s, v.x)));
        if constexpr (f1 || f2 || f3)
            if ((f1 && l == 1) || (f2 && l == 2) || (f3 && l == 3)) r.y = __fmaf_rn(s, v.x, __fmul_rn(c, v.y));
        a[k] = r;
    });
    const float s2 = (l & 2) ? -1.f : 1.f, s1 = (l & 1) ? -1.f : 1.f;
    const bool rot = l == 3;
#pragma unroll
    for (int k = 0; k < kQ; ++k) {
        const float ox = __shfl_xor_sync(0xffffffffu, a[k].x, 2), oy = __shfl_xor_sync(0xffffffffu, a[k].y, 2);
        const float tx = fmaf(s2, a[k].x, ox), ty = fmaf(s2, a[k].y, oy);
        const float ux = rot ? ty : tx, uy = rot ? -tx : ty;
        const float px = __shfl_xor_sync(0xffffffffu, ux, 1), py = __shfl_xor_sync(0xffffffffu, uy, 1);
        a[k] = make_float2(fmaf(s1, ux, px), fmaf(s1, uy, py));
    }
}

// A thread's line and lane: thread = 4 line + l.
struct Lane {
    int line, l, q;
    __device__ __forceinline__ Lane() : line(threadIdx.x >> 2), l(threadIdx.x & 3), q(split_q(threadIdx.x & 3)) {}
};

// Forward passes of one frame: phases -> h (OTF, masked, H(0) = 1), the field
// kept in `field` (this thread's 16 points, kST apart).
__device__ __forceinline__ void frame_forward(const ObjParams& ob, const float* __restrict__ ph, float2* E,
                                              float2* field, float2* __restrict__ h) {
    const Lane t;
    float* Ef = reinterpret_cast<float*>(E);
    const int W = ob.W;
    float2 a[kQ];
    if (t.line < 8 * ((W + 7) / 8)) {  // PUPIL: column c of P along y (whole warps)
        const int c = t.line;
        const uint64_t cm = c < W ? ob.cmask[c] : 0ull;
        float phv[kQ];
#pragma unroll
        for (int n = 0; n < kQ; ++n) phv[n] = bit(cm, 4 * n + t.l) ? ph[(4 * n + t.l) * ob.phi_ld + c] : 0.f;
#pragma unroll
        for (int n = 0; n < kQ; ++n) a[n] = bit(cm, 4 * n + t.l) ? expi(phv[n]) : make_float2(0.f, 0.f);
        if (c < 32) fft64_lanes(a, t.l);  // uniform in a warp
        else fft64_quarters(a, t.l);
        if (c < W)
#pragma unroll
            for (int k = 0; k < kQ; ++k) E[row_base(16 * t.q) + k * kLd + c + (c >> 4)] = a[k];
    }
    __syncthreads();
    {  // FIELD: row y of p; the PSF row |p|^2 / (N^2 n_pup) as floats
        float2* row = E + row_base(t.line);
#pragma unroll
        for (int n = 0; n < kQ; ++n)
            a[n] = 4 * n + t.l < W ? row[4 * n + t.l + (n >> 2)] : make_float2(0.f, 0.f);
        fft64_lanes(a, t.l);
        __syncwarp();
        float* srow = Ef + 2 * row_base(t.line) + 18 * t.q;
        const float iz = ob.inv_z;
#pragma unroll
        for (int k = 0; k < kQ; ++k) {
            field[k * kST + threadIdx.x] = a[k];
            srow[k] = (a[k].x * a[k].x + a[k].y * a[k].y) * iz;
        }
    }
    __syncthreads();
    if (t.line < kN / 2) {  // PSF rows i and i + 32 as one complex line, split into their half spectra
        const int i = t.line;
        const float *s0 = Ef + 2 * row_base(i), *s1 = Ef + 2 * row_base(i + kN / 2);
#pragma unroll
        for (int n = 0; n < kQ; ++n) {
            const int x = 4 * n + t.l + 2 * (n >> 2);
            a[n] = make_float2(s0[x], s1[x]);
        }
        fft64_lanes(a, t.l);
        __syncwarp();
        float2 *r0 = E + row_base(i), *r1 = E + row_base(i + kN / 2);
#pragma unroll
        for (int k = 0; k < kQ; ++k) r0[k + 17 * t.q] = a[k];
        __syncwarp();
        float2 u[9], v[9];  // kx = 4 m + l; lane 0 also kx = 32
#pragma unroll
        for (int m = 0; m < 9; ++m) {
            const int kx = 4 * m + t.l, mx = (kN - kx) & (kN - 1);
            if (m == 8 && t.l > 0) continue;
            const float2 z = r0[kx + (kx >> 4)], zc = cconj(r0[mx + (mx >> 4)]);
            u[m] = cscale(cadd(z, zc), 0.5f);
            const float2 d = cscale(csub(z, zc), 0.5f);
            v[m] = make_float2(d.y, -d.x);
        }
        __syncwarp();
#pragma unroll
        for (int m = 0; m < 8; ++m) {
            const int kx = 4 * m + t.l, at = kx + (kx >> 4);
            if (m == 0 && t.l == 0) {  // the real columns 0 and 32 share slot 0
                r0[0] = make_float2(u[0].x, u[8].x);
                r1[0] = make_float2(v[0].x, v[8].x);
            } else {
                r0[at] = u[m];
                r1[at] = v[m];
            }
        }
    }
    __syncthreads();
    if (t.line < kN / 2) {  // OTF: half-spectrum columns along y, column 0 packed with column 32
        const int kx = t.line, at = kx + (kx >> 4);
#pragma unroll
        for (int n = 0; n < kQ; ++n) a[n] = E[row_base(4 * n + t.l) + at];
        fft64_lanes(a, t.l);
        if (kx > 0) {
            const uint64_t cs = ob.csupp[kx];
#pragma unroll
            for (int k = 0; k < kQ; ++k) {
                const int ky = k + 16 * t.q;
                h[ky * kNH + kx] = bit(cs, ky) ? a[k] : make_float2(0.f, 0.f);
            }
        }
        if (threadIdx.x < 32) {  // the warp of column 0 splits it through its storage
            __syncwarp();
            if (kx == 0)
#pragma unroll
                for (int k = 0; k < kQ; ++k) E[row_base(16 * t.q) + k * kLd] = a[k];
            __syncwarp();
            const uint64_t cs0 = ob.csupp[0], cs32 = ob.csupp[kN / 2];
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                const int ky = threadIdx.x + 32 * i;
                const float2 z = E[row_base(ky)];
                const float2 zc = cconj(E[row_base((kN - ky) & (kN - 1))]);
                float2 h0 = cscale(cadd(z, zc), 0.5f);
                const float2 d = cscale(csub(z, zc), 0.5f);
                float2 h32 = make_float2(d.y, -d.x);
                if (!bit(cs0, ky)) h0 = make_float2(0.f, 0.f);
                if (!bit(cs32, ky)) h32 = make_float2(0.f, 0.f);
                if (ky == 0) h0 = make_float2(1.f, 0.f);
                h[ky * kNH] = h0;
                h[ky * kNH + 32] = h32;
            }
        }
    }
    __syncthreads();
}

// Adjoint passes of one frame: h (the seed G) -> gphi. The first two occupy the
// lower warps; the upper four (128 threads) run beside(0) and, a CTA barrier
// later, beside(1).
template <class Beside>
__device__ __forceinline__ void frame_adjoint(const ObjParams& ob, const float* __restrict__ ph,
                                              float* __restrict__ gphi, float2* E, const float2* field,
                                              const float2* h, Beside&& beside) {
    const Lane t;
    float* Ef = reinterpret_cast<float*>(E);
    const int W = ob.W;
    float2 a[kQ];
    if (t.line < kN / 2) {  // SEED: conj of the columns of G, column 0 as G_0 + i G_32
        const int kx = t.line;
#pragma unroll
        for (int n = 0; n < kQ; ++n) {
            const int ky = 4 * n + t.l;
            const float2 g = h[ky * kNH + kx];
            const float2 b = kx == 0 ? h[ky * kNH + 32] : make_float2(0.f, 0.f);
            a[n] = make_float2(g.x - b.y, -(g.y + b.x));
        }
        fft64_lanes(a, t.l);
#pragma unroll
        for (int k = 0; k < kQ; ++k) E[row_base(16 * t.q) + k * kLd + kx + (kx >> 4)] = a[k];
    } else {
        beside(0);
    }
    __syncthreads();
    if (t.line < kN / 2) {  // C2R: conj of T_i + i T_(i+32), Hermitian-extended; g_q rows as floats
        const int i = t.line;
        const float2 *r0 = E + row_base(i), *r1 = E + row_base(i + kN / 2);
#pragma unroll
        for (int n = 0; n < kQ; ++n) {
            const int x = 4 * n + t.l, m = x <= kN / 2 ? x : kN - x;
            if (x == 0) {
                a[n] = make_float2(r0[0].x, -r1[0].x);
            } else if (x == kN / 2) {
                a[n] = make_float2(-r0[0].y, r1[0].y);
            } else {
                const float2 p = r0[m + (m >> 4)], q = r1[m + (m >> 4)];
                a[n] = x < kN / 2 ? make_float2(p.x + q.y, p.y - q.x) : make_float2(p.x - q.y, -(p.y + q.x));
            }
        }
        fft64_lanes(a, t.l);
        __syncwarp();
        const float sc = 2.0f * ob.inv_z;
        float *g0 = Ef + 2 * row_base(i) + 18 * t.q, *g1 = Ef + 2 * row_base(i + kN / 2) + 18 * t.q;
#pragma unroll
        for (int k = 0; k < kQ; ++k) {
            g0[k] = a[k].x * sc;
            g1[k] = a[k].y * -sc;
        }
    } else {
        beside(1);
    }
    __syncthreads();
    {  // rows of conj(g_q p), transformed; the box columns kept
        float2* row = E + row_base(t.line);
        const float* grow = Ef + 2 * row_base(t.line) + 18 * t.q;
#pragma unroll
        for (int k = 0; k < kQ; ++k) {
            const float2 p = field[k * kST + threadIdx.x];
            const float g = grow[k];
            a[k] = make_float2(g * p.x, -g * p.y);
        }
        __syncwarp();
#pragma unroll
        for (int k = 0; k < kQ; ++k) row[k + 17 * t.q] = a[k];
        __syncwarp();
#pragma unroll
        for (int n = 0; n < kQ; ++n) a[n] = row[4 * n + t.l + (n >> 2)];
        fft64_lanes(a, t.l);
        __syncwarp();
#pragma unroll
        for (int k = 0; k < kQ; ++k)
            if (k + 16 * t.q < W) row[k + 17 * t.q] = a[k];
    }
    __syncthreads();
    if (t.line < 8 * ((W + 7) / 8)) {  // ADJ: dL/dphi = 2 Im(conj(P) G_P) on the pupil, G_P = conj(a)
        const int c = t.line, at = c + (c >> 4);
#pragma unroll
        for (int n = 0; n < kQ; ++n) a[n] = E[row_base(4 * n + t.l) + at];
        fft64_lanes(a, t.l);
        if (c < W) {
            const uint64_t cm = ob.cmask[c];
#pragma unroll
            for (int k = 0; k < kQ; ++k) {
                const int y = k + 16 * t.q;
                if (y < W) {
                    const float2 pv = expi(ph[y * ob.phi_ld + c]);
                    gphi[y * ob.phi_ld + c] = bit(cm, y) ? 2.0f * fmaf(pv.x, -a[k].y, -(pv.y * a[k].x)) : 0.f;
                }
            }
        }
    }
    __syncthreads();
}

__device__ __forceinline__ void cluster_sync() {
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

constexpr int kSpreadFrames = 2;  // frames of a CTA
constexpr size_t kSpreadSmem = (kBufElems + (size_t)kSpreadFrames * kQ * kST) * sizeof(float2);

// Address of this CTA's shared-memory object in CTA `rank` of the cluster.
__device__ __forceinline__ uint32_t in_rank(const void* p, int rank) {
    uint32_t a;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(rank));
    return a;
}

// EXPL: the object-inferring loss. Cluster c of prm.csize CTAs carries pair c.
template <bool EXPL>
__global__ void __launch_bounds__(kST, 2) spread_pair_kernel(const FusedParams prm) {
    extern __shared__ __align__(16) unsigned char spsm[];
    // The last CTA sums the pair's loss: chain c adds the terms c, c + kChains,
    // ... as thread c of the fused kernel does, so a patch's loss does not depend
    // on which of the two kernels its plan takes. Half its warps do so beside the
    // first adjoint passes (1 pair of 8 frames: 43.6 us an evaluation; the sum before
    // them 45.7, each CTA summing its own frequencies, with other bits, 44.5).
    constexpr int kChains = 32 * kFusedFrames;
    __shared__ float terms[kHalf];
    __shared__ double swarp[kFusedFrames];
    float2* E = reinterpret_cast<float2*>(spsm);
    float2* field = E + kBufElems;
    const int csize = prm.csize;
    const int rank = (int)(blockIdx.x % csize), lane = threadIdx.x & 31;
    const long long pair = blockIdx.x / csize;
    const int J = prm.J, K = prm.K;
    const long long p = pair / K;
    const int k = (int)(pair - p * K);
    const ObjParams& ob = prm.obj[k];
    float2* const hpair = prm.gscr + (size_t)pair * J * kHalf;
    chain_wait();
    chain_release();
    for (int f = 0; f < kSpreadFrames; ++f) {
        const int j = rank + f * csize;
        if (j < J)
            frame_forward(ob, prm.phi + ob.phi_off + (p * J + j) * ob.phi_unit + ob.phi_org, E,
                          field + (size_t)f * kQ * kST, hpair + (size_t)j * kHalf);
    }
    cluster_sync();  // every frame's OTF
    const uint32_t sums = in_rank(terms, csize - 1);
    each_frequency<kFusedFrames, EXPL ? 2 : 1, false>(
        prm, (int)p, k, hpair, rank * kST + threadIdx.x, csize * kST,
        [&](int f, float x) { asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(sums + 4 * f), "f"(x) : "memory"); });
    cluster_sync();  // every seed and term of the loss
    auto sum_loss = [&](int step) {  // the upper four warps of the last CTA
        if (step == 0) {
            for (int c = threadIdx.x - kST / 2; c < kChains; c += kST / 2) {  // whole warps
                KahanSum acc;
                for (int f = c; f < kHalf; f += kChains) acc.add(terms[f]);
                double v = (double)acc.s - (double)acc.c;
#pragma unroll
                for (int off = 16; off > 0; off >>= 1) v += __shfl_down_sync(0xffffffffu, v, off);
                if (lane == 0) swarp[c >> 5] = v;
            }
        } else if (threadIdx.x == kST / 2) {
            double tot = 0.0;
            for (int w = 0; w < kFusedFrames; ++w) tot += swarp[w];
            __stcg(&prm.lpair[pair], tot);
            // the pair that finishes the patch sums its objects in order and resets the count
            __threadfence();
            if (atomicAdd(&prm.lcnt[p], 1) == K - 1) {
                __threadfence();
                double sum = 0.0;
                for (int kk = 0; kk < K; ++kk) sum += __ldcg(&prm.lpair[p * K + kk]);
                prm.loss[p] = sum;
                prm.lcnt[p] = 0;
            }
        }
    };
    for (int f = 0; f < kSpreadFrames; ++f) {
        const int j = rank + f * csize;
        const long long img = ob.phi_off + (p * J + j) * ob.phi_unit + ob.phi_org;
        if (j < J)
            frame_adjoint(ob, prm.phi + img, prm.gphi + img, E, field + (size_t)f * kQ * kST,
                          hpair + (size_t)j * kHalf, [&](int step) {
                              if (f == 0 && rank == csize - 1) sum_loss(step);
                          });
    }
}

// Launches the kernel, or (clusters) asks how many of its clusters fit the GPU
// at once.
template <bool EXPL>
cudaError_t launch_spread(const FusedParams& prm, cudaStream_t s, int* clusters) {
    auto kern = spread_pair_kernel<EXPL>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSpreadSmem);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
    cudaLaunchAttribute attr[2]{};
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = prm.csize;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = prm.chain ? 1 : 0;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)((long long)prm.P * prm.K * prm.csize));
    cfg.blockDim = dim3(kST);
    cfg.dynamicSmemBytes = kSpreadSmem;
    cfg.stream = s;
    cfg.attrs = attr;
    cfg.numAttrs = clusters ? 1 : 2;
    if (clusters) return cudaOccupancyMaxActiveClusters(clusters, kern, &cfg);
    e = cudaLaunchKernelEx(&cfg, kern, prm);
    if (e != cudaSuccess) cudaGetLastError();
    return e;
}

}  // namespace

// One frame per CTA if all pairs are then resident at once, else (more than 8
// frames, where the fused kernel runs three warps a scheduler) two; beyond that
// the fused kernel. us per evaluation, this kernel and the fused one, both with
// chained launches: 1 pair of 8 frames 44 and 69, 41 of 6 frames 57 and 83, 20 of
// 12 frames 50 and 91; two frames to a CTA: 40 pairs of 12 frames 73 and 87, but
// 64 of 6 frames 72 and 64. A second wave is slower (48 pairs of 12 frames 115
// and 88).
//
// chain: whether the kernel may be launched over the projection's tail. Its
// clusters then go to the SMs that are already free. While they are few, that
// saves 2 to 3 us (15 pairs of 12 frames 50 against 52); near the most that fit,
// what the projection's CTAs leave is cut up and a second wave forms: 28 pairs of
// 10 frames 74 us chained, 52 not, 83 on the fused kernel; 45 pairs of 12 frames
// (28 px) 108, 71, 75. A second wave was seen from 80 % of the clusters that fit
// up, so the line is at three quarters; clusters of two take the two places of
// an SM and always fit (152 pairs 65 and 68 us). Single CTAs (one frame) double
// up on the free SMs as soon as they are nearly as many as all SMs: 130 pairs 85
// and 87 us, 142 pairs 112 and 87, the fused kernel 101; there the line is at 0.8
// of the SMs.
int spread_cluster(int P, int K, int J, int max_box, bool* chain) {
    if (J > kFusedFrames || max_box > kMaxBox || P < 1 || (long long)P * K > 4096) return 0;
    for (int frames = 1; frames <= (J > 8 ? kSpreadFrames : 1); ++frames) {
        FusedParams prm{};
        prm.P = P;
        prm.K = K;
        prm.csize = (J + frames - 1) / frames;
        int n0 = 0, n1 = 0;
        const bool ok = launch_spread<false>(prm, nullptr, &n0) == cudaSuccess &&
                        launch_spread<true>(prm, nullptr, &n1) == cudaSuccess;
        if (!ok) cudaGetLastError();
        const long long pairs = (long long)P * K, fit = std::min(n0, n1);
        if (ok && pairs <= fit) {
            *chain = prm.csize == 2 || (4 * pairs <= 3 * fit && (prm.csize > 1 || 5 * pairs <= 2 * fit));
            return prm.csize;
        }
    }
    return 0;
}

cudaError_t launch_spread_pairs(const FusedParams& prm, cudaStream_t s) {
    if (prm.P == 0) return cudaSuccess;
    return prm.oin ? launch_spread<true>(prm, s, nullptr) : launch_spread<false>(prm, s, nullptr);
}

}  // namespace mfbd_dev
