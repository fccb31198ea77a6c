// The spatially variant PSF model on a dictionary (Sec. 2.2.2, "Spatially
// variant convolution"): the PSF at object point r' is sum_i a_i(r') phi_i,
// the image of object k in frame j is sum_i (o_k a_ikj) * phi_i, and the data
// term of the log-posterior in the Fourier domain is
//   L = sum_kj gamma_kj sum_u |I_kj(u) - sum_i F(o_k a_ikj)(u) Phi_i(u)|^2
// (full frequency plane). With R_kj = I_kj - sum_i F(o_k a_ikj) Phi_i and
// g_ikj = Re F^H[conj(Phi_i) (-2 gamma_kj R_kj)] (F^H unnormalised):
//   dL/da_ikj = o_k g_ikj,  dL/do_k = sum_j sum_i a_ikj g_ikj.
//
// dict_unit_kernel: one CTA of eight warps per unit (patch, object, frame),
// N = 64, persistent; lines of eight lanes (lane8.cuh), every warp holding the
// same four row pairs and four half-spectrum columns of every atom.
//   Forward, per atom i: rows y and y + N/2 of o a_i as one complex line,
//   transformed; then the half-spectrum columns (the two rows' spectra split
//   on load, columns 0 and N/2 packed in line 0), transformed, times Phi_i,
//   accumulated in registers: a lane owns eight frequencies of one column.
//   Then the residual, the unit's loss (FP64 sums of FP32 terms; columns 0 and
//   N/2 once, the others twice) and conj(G) = -2 gamma conj(R) in place.
//   Backward, per atom i: the inverse of the half spectrum conj(Phi_i) G
//   (columns along ky, then the packed row pairs) gives g_i; dL/da_i = o g_i
//   is stored and a_i g_i accumulated in registers into the unit's share of
//   dL/do, written out at the end.
// The atoms alternate between two exchange buffers, so that one CTA barrier
// per atom (rows to columns, or back) is enough.
//   HBM is the floor (coefficient maps in and their gradient out); the L1 data
//   path bounds it (shared-memory exchanges, atom transforms: 65 % of its
//   wavefronts, issue 32 %). 5,400 units of 8 atoms: 2.63 ms with one warp per
//   unit (a 64-point line per lane, 4 warps an SM), 0.936 ms with this.
// dict_combine_kernel: dL/do_k = the units' shares summed over frames in
// frame order; the patch loss = the units' losses summed over (k, j) in order.
#include "../../include/mfbd.h"
#include "mfbd_internal.h"
#include "lane_passes.cuh"

#include <cuda_runtime.h>

#include <cstdint>

using namespace mfbd_dev;

namespace {

using namespace mfbd_dev::lanepass;

constexpr int kDN = 64, kDNH = kDN / 2 + 1;
constexpr int kDS = Geo<kDN>::S_HALF;  // row stride of an exchange buffer
constexpr int kDWarps = 8;             // one group of four lines each, in every pass
// shared memory of a CTA: the twiddles and two exchange buffers
constexpr size_t kDictSmem = ((size_t)kDN + 2 * (size_t)kDN * kDS) * sizeof(float2);

struct DictParams {
    int P, K, J, M;
    const float2* atom_otf;  // [M][N][NH]
    const float* gamma;      // [K][J]
    const float* object;     // [P][K][N][N]
    const float* coeff;      // [P][K][J][M][N][N]
    const float2* spectra;   // [P][K][J][N][NH]
    float* grad_coeff;       // [P][K][J][M][N][N] or null
    float* unit_gobj;        // [P][K][J][N][N] or null (workspace)
    double* unit_loss;       // [P][K][J] (workspace)
};

}  // namespace

namespace {

__global__ void __launch_bounds__(32 * kDWarps, 2) dict_unit_kernel(const DictParams prm) {
    extern __shared__ __align__(16) unsigned char dsm[];
    float2* table = reinterpret_cast<float2*>(dsm);
    float2* const buf0 = table + kDN;
    __shared__ double part[kDWarps];
    __shared__ float2 snyq[kDN];  // column N/2, each element private to a lane of line 0
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    load_twiddles<kDN>(table, threadIdx.x, 32 * kDWarps);
    __syncthreads();
    const long long units = (long long)prm.P * prm.K * prm.J;
    const bool backward = prm.grad_coeff != nullptr || prm.unit_gobj != nullptr;
    // this lane's four-line group: the row pair (i, i + 32) and the column kx;
    // at 64 points a blocked line holds the same elements t + 8 e as a strided one
    const RowLanes rl(lane);
    const ColLanes cl(lane);
    const int i = 4 * w + rl.p, tr = rl.t, kx = 4 * w + cl.c, tc = cl.t;
    const int shift = kx ? kDN / 2 - 2 * kx : 0;
    const int r0 = i * kDN + tr, r1 = (i + kDN / 2) * kDN + tr;  // first element of the rows' lines
    int b = 0;  // exchange buffer of the next atom: one barrier per atom and pass pair
    for (long long u = blockIdx.x; u < units; u += gridDim.x) {
        const int j = (int)(u % prm.J);
        const long long pk = u / prm.J;
        const int k = (int)(pk % prm.K);
        const float* o = prm.object + (size_t)pk * kDN * kDN;
        const float* a = prm.coeff + (size_t)u * prm.M * kDN * kDN;
        const float2* I = prm.spectra + (size_t)u * kDN * kDNH;
        const float gam = prm.gamma[k * prm.J + j];
        // ------------------------------------------- model: sum_i F(o a_i) Phi_i
        float2 mod[8];  // column kx
        float2* const nyq = snyq + tc;  // and, in the lanes of line 0, column N/2
#pragma unroll
        for (int e = 0; e < 8; ++e) mod[e] = make_float2(0.f, 0.f);
        if (kx == 0) {
#pragma unroll
            for (int e = 0; e < 8; ++e) nyq[8 * e] = make_float2(0.f, 0.f);
        }
        float o0[8], o1[8], a0[8], a1[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            o0[e] = o[r0 + 8 * e];
            o1[e] = o[r1 + 8 * e];
            a0[e] = a[r0 + 8 * e];
            a1[e] = a[r1 + 8 * e];
        }
        for (int m = 0; m < prm.M; ++m) {
            float2* E = buf0 + b * (kDN * kDS);
            b ^= 1;
            {
                const RowLine<kDN, kDS> ln{E + i * kDS};
                float2 v[8], z[8];
#pragma unroll
                for (int e = 0; e < 8; ++e) v[e] = make_float2(o0[e] * a0[e], o1[e] * a1[e]);
                if (m + 1 < prm.M) {  // the next atom's maps arrive under this atom's transforms
                    const float* an = a + (size_t)(m + 1) * kDN * kDN;
#pragma unroll
                    for (int e = 0; e < 8; ++e) {
                        a0[e] = an[r0 + 8 * e];
                        a1[e] = an[r1 + 8 * e];
                    }
                }
                strided_to_blocked<kDN>(ln, v, z, LaneTwiddles<kDN>(table, tr), tr);
                __syncwarp();
#pragma unroll
                for (int e = 0; e < 8; ++e) ln.block(e)[tr] = z[e];
            }
            __syncthreads();
            const float2* Phi = prm.atom_otf + (size_t)m * kDN * kDNH;
            const ColLine<kDN, kDS> ln{E + kx, shift};
            float2 v[8], x[8];
#pragma unroll
            for (int e = 0; e < 4; ++e) {  // the two rows' half spectra at kx; line 0: columns 0 and N/2 packed
                const float2 p = ln.block(e)[tc * kDS], q = ln.block(e + 4)[tc * kDS];
                v[e] = kx ? make_float2(0.5f * (p.x + q.x), 0.5f * (p.y - q.y)) : make_float2(p.x, q.x);
                v[e + 4] = kx ? make_float2(0.5f * (p.y + q.y), 0.5f * (q.x - p.x)) : make_float2(p.y, q.y);
            }
            strided_to_blocked<kDN>(ln, v, x, LaneTwiddles<kDN>(table, tc), tc);
            if (w == 0) {  // the warp of line 0 splits its packed columns through the line's storage
                __syncwarp();
                if (kx == 0) {
#pragma unroll
                    for (int e = 0; e < 8; ++e) E[(tc + 8 * e) * kDS] = x[e];
                }
                __syncwarp();
                if (kx == 0) {
#pragma unroll
                    for (int e = 0; e < 8; ++e) {
                        const int ky = tc + 8 * e;
                        const float2 z = x[e], c = E[((kDN - ky) & (kDN - 1)) * kDS];
                        const float2 h = make_float2(0.5f * (z.y + c.y), 0.5f * (c.x - z.x));
                        nyq[8 * e] = cadd(nyq[8 * e], cmul(h, Phi[ky * kDNH + kDN / 2]));
                        x[e] = make_float2(0.5f * (z.x + c.x), 0.5f * (z.y - c.y));
                    }
                }
            }
#pragma unroll
            for (int e = 0; e < 8; ++e) mod[e] = cadd(mod[e], cmul(x[e], Phi[(tc + 8 * e) * kDNH + kx]));
        }
        // --------------------- residual, loss, conj(G) = -2 gamma conj(R) in place
        double lacc = 0.0;
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            const float2 d = I[(tc + 8 * e) * kDNH + kx];
            const float2 r = make_float2(d.x - mod[e].x, d.y - mod[e].y);
            lacc += (kx ? 2.0 : 1.0) * (double)(r.x * r.x + r.y * r.y);
            mod[e] = make_float2(-2.f * gam * r.x, 2.f * gam * r.y);
            if (kx == 0) {
                const float2 dn = I[(tc + 8 * e) * kDNH + kDN / 2];
                const float2 rn = make_float2(dn.x - nyq[8 * e].x, dn.y - nyq[8 * e].y);
                lacc += (double)(rn.x * rn.x + rn.y * rn.y);
                nyq[8 * e] = make_float2(-2.f * gam * rn.x, 2.f * gam * rn.y);
            }
        }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) lacc += __shfl_xor_sync(0xffffffffu, lacc, off);
        if (lane == 0) part[w] = lacc;
        __syncthreads();
        if (threadIdx.x == 0) {
            double s = 0.0;
            for (int q = 0; q < kDWarps; ++q) s += part[q];
            prm.unit_loss[u] = (double)gam * s;
        }
        if (!backward) {
            __syncthreads();  // part is free again
            continue;
        }
        // ------------------------------ g_i = F^H[conj(Phi_i) G] (real), per atom
        float s0[8], s1[8];  // the unit's share of dL/do
#pragma unroll
        for (int e = 0; e < 8; ++e) s0[e] = s1[e] = 0.f;
        for (int m = 0; m < prm.M; ++m) {
            float2* E = buf0 + b * (kDN * kDS);
            b ^= 1;
            const float2* Phi = prm.atom_otf + (size_t)m * kDN * kDNH;
            {
                // columns along ky: F^H x = conj(F conj x); line 0 the packed real columns
                const ColLine<kDN, kDS> ln{E + kx, shift};
                float2 v[8], x[8];
#pragma unroll
                for (int e = 0; e < 8; ++e) v[e] = cmul(Phi[(tc + 8 * e) * kDNH + kx], mod[e]);
                if (kx == 0) {
#pragma unroll
                    for (int e = 0; e < 8; ++e) {
                        const float2 c = cmul(Phi[(tc + 8 * e) * kDNH + kDN / 2], nyq[8 * e]);
                        v[e] = make_float2(v[e].x + c.y, v[e].y - c.x);
                    }
                }
                strided_to_blocked<kDN>(ln, v, x, LaneTwiddles<kDN>(table, tc), tc);
                __syncwarp();
                // rows y and y + N/2 of T = conj(x): conj of T_y + i T_(y+N/2) at kx, and its mirror
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const float2 u0 = x[e], u1 = x[e + 4];
                    float2 lo = make_float2(u0.x + u1.y, u0.y - u1.x), hi = make_float2(u0.x - u1.y, -u0.y - u1.x);
                    if (kx == 0) {
                        lo = make_float2(u0.x, -u1.x);
                        hi = make_float2(-u0.y, u1.y);
                    }
                    ln.block(e)[tc * kDS] = lo;
                    ln.block(e + 4)[tc * kDS] = hi;
                }
            }
            __syncthreads();
            const RowLine<kDN, kDS> ln{E + i * kDS};
            float2 v[8], g[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) v[e] = ln.block(e)[tr];
            if (prm.unit_gobj) {
                const float* am = a + (size_t)m * kDN * kDN;
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    a0[e] = am[r0 + 8 * e];
                    a1[e] = am[r1 + 8 * e];
                }
            }
            strided_to_blocked<kDN>(ln, v, g, LaneTwiddles<kDN>(table, tr), tr);
            // g.x = g_i(y, x), -g.y = g_i(y + N/2, x)
            if (prm.grad_coeff) {
                float* gc = prm.grad_coeff + ((size_t)u * prm.M + m) * kDN * kDN;
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    gc[r0 + 8 * e] = o0[e] * g[e].x;
                    gc[r1 + 8 * e] = -o1[e] * g[e].y;
                }
            }
            if (prm.unit_gobj) {
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    s0[e] = fmaf(a0[e], g[e].x, s0[e]);
                    s1[e] = fmaf(a1[e], -g[e].y, s1[e]);
                }
            }
        }
        if (prm.unit_gobj) {
            float* out = prm.unit_gobj + (size_t)u * kDN * kDN;
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                out[r0 + 8 * e] = s0[e];
                out[r1 + 8 * e] = s1[e];
            }
        }
    }
}

// dL/do_k = sum_j of the units' shares (frame order); loss_p = sum_kj of the
// units' losses (in order). One CTA per patch.
__global__ void __launch_bounds__(256) dict_combine_kernel(int K, int J, const double* __restrict__ unit_loss,
                                                           const float* __restrict__ unit_gobj,
                                                           float* __restrict__ grad_object, double* __restrict__ loss) {
    const int p = blockIdx.x;
    if (grad_object) {
        const int per = K * kDN * kDN;
        for (int e = threadIdx.x; e < per; e += blockDim.x) {
            const int k = e / (kDN * kDN), r = e - k * kDN * kDN;
            const float* src = unit_gobj + (((size_t)p * K + k) * J) * kDN * kDN + r;
            float s = 0.f;
            for (int j = 0; j < J; ++j) s += src[(size_t)j * kDN * kDN];
            grad_object[(size_t)p * per + e] = s;
        }
    }
    if (threadIdx.x == 0) {
        double s = 0.0;
        for (int e = 0; e < K * J; ++e) s += unit_loss[(size_t)p * K * J + e];
        loss[p] = s;
    }
}

}  // namespace

namespace {

// workspace: the units' losses, then (256-byte aligned) their dL/do shares
size_t dict_gobj_offset(long long units) { return ((size_t)units * sizeof(double) + 255) & ~(size_t)255; }

int dict_check_desc(const mfbd_dict_desc* d) {
    if (!d) return set_error(MFBD_ERR_INVALID_ARG, "dictionary descriptor is NULL");
    if (d->n_patches < 0 || d->n_objects < 1 || d->n_frames < 1 || d->n_atoms < 1)
        return set_error(MFBD_ERR_INVALID_ARG, "dictionary sizes: n_patches >= 0, n_objects, n_frames, n_atoms >= 1");
    if (d->n != kDN) return set_error(MFBD_ERR_UNSUPPORTED, "the dictionary model supports n = 64");
    if ((long long)d->n_patches * d->n_objects * d->n_frames * d->n_atoms > (1ll << 40))
        return set_error(MFBD_ERR_INVALID_ARG, "dictionary problem too large");
    return MFBD_OK;
}

bool aligned(const void* p, size_t a) { return (reinterpret_cast<uintptr_t>(p) & (a - 1)) == 0; }

}  // namespace

extern "C" size_t mfbd_dict_workspace_bytes(const mfbd_dict_desc* desc) {
    if (dict_check_desc(desc) != MFBD_OK) return 0;
    const long long units = (long long)desc->n_patches * desc->n_objects * desc->n_frames;
    return dict_gobj_offset(units) + (size_t)units * kDN * kDN * sizeof(float);
}

extern "C" int mfbd_dict_loss_grad(const mfbd_dict_desc* desc, const void* atom_otf, const float* gamma,
                                   const float* object, const float* coeff, const void* spectra, void* workspace,
                                   double* loss, float* grad_object, float* grad_coeff, void* stream) {
    int st = dict_check_desc(desc);
    if (st != MFBD_OK) return st;
    const long long units = (long long)desc->n_patches * desc->n_objects * desc->n_frames;
    if (units == 0) return MFBD_OK;
    if (!atom_otf || !gamma || !object || !coeff || !spectra || !workspace || !loss)
        return set_error(MFBD_ERR_INVALID_ARG, "a required dictionary-model pointer is NULL");
    if (!aligned(object, 16) || !aligned(coeff, 16) || (grad_coeff && !aligned(grad_coeff, 16)) ||
        !aligned(workspace, 16) || !aligned(atom_otf, 8) || !aligned(spectra, 8) || !aligned(loss, 8) ||
        (grad_object && !aligned(grad_object, 4)))
        return set_error(MFBD_ERR_INVALID_ARG,
                         "object, coeff, grad_coeff and workspace need 16-byte alignment; atom_otf, spectra, loss 8");
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    int dev = 0, sms = 0, per_sm = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(dict_unit_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kDictSmem);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, dict_unit_kernel, 32 * kDWarps, kDictSmem);
    if (e != cudaSuccess) return set_cuda_error(e, "mfbd_dict_loss_grad setup");
    if (per_sm < 1) return set_error(MFBD_ERR_UNSUPPORTED, "the dictionary kernel does not fit an SM");
    unsigned char* ws = static_cast<unsigned char*>(workspace);
    DictParams prm;
    prm.P = desc->n_patches;
    prm.K = desc->n_objects;
    prm.J = desc->n_frames;
    prm.M = desc->n_atoms;
    prm.atom_otf = static_cast<const float2*>(atom_otf);
    prm.gamma = gamma;
    prm.object = object;
    prm.coeff = coeff;
    prm.spectra = static_cast<const float2*>(spectra);
    prm.grad_coeff = grad_coeff;
    prm.unit_loss = reinterpret_cast<double*>(ws);
    prm.unit_gobj = grad_object ? reinterpret_cast<float*>(ws + dict_gobj_offset(units)) : nullptr;
    long long ctas = (long long)sms * per_sm;
    if (ctas > units) ctas = units;
    dict_unit_kernel<<<(int)ctas, 32 * kDWarps, kDictSmem, s>>>(prm);
    if ((e = cudaGetLastError()) != cudaSuccess) return set_cuda_error(e, "dict_unit_kernel launch");
    dict_combine_kernel<<<desc->n_patches, 256, 0, s>>>(prm.K, prm.J, prm.unit_loss, prm.unit_gobj, grad_object,
                                                        loss);
    if ((e = cudaGetLastError()) != cudaSuccess) return set_cuda_error(e, "dict_combine_kernel launch");
    return MFBD_OK;
}
