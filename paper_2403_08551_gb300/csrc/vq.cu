// vq.cu -- codec decode (Sec. 3.3): FP16 positions, and Cholesky / colour
// attributes as the sum over M residual-VQ stages of codebook rows,
//   hat c^M = sum_{k=1..M} C^k[i^k].
// The result equals the sum evaluated exactly and rounded once to FP32: for
// M <= 2 a single FP32 addition already is that (rounding a double-precision
// sum of two floats to float is innocuous since 53 >= 2*24 + 2); for M > 2
// it is what an FP64 sum in stage order, rounded once, gives (RowSum).
#include <algorithm>

#include <cuda_fp16.h>

#include "kernels.cuh"

namespace gi {
namespace {

// The FP64 sum of up to eight floats rounded to FP32, on the FP32 units (with
// FP64 a three-stage decode took five times a two-stage one): s + e is the
// running sum and the errors of its additions (Knuth, TAOCP 2, 4.2.2), p the sum
// of the magnitudes, q the smallest but for zeros. With u the last unit of q, every
// term is a multiple of u and q < 2^24 u. If q >= 2^-22 p, then p < 2^46 u at every
// addition, |s| <= p (rounding is monotone), and an addition's error is a multiple
// of u of at most 2^21 u. The first addition is exact, so the seven others of eight
// terms leave |e| <= 7 * 2^21 u < 2^24 u: e is exact in FP32 (for more terms it
// need not be), the FP64 sum is exact below 2^53 u, and s + e rounds as it does.
// Otherwise (terms of very different size, infinities, NaN) get() is false and the
// caller sums in FP64. Three stages, 64 entries: 1 M Gaussians 88 -> 16.5 us, 3.2 M
// x 256 entries 256 -> 43.6 us (what bounds it there is the codebook rows' bank
// conflicts).
constexpr int kRowSumTerms = 8;
struct RowSum {
    float s = 0.f, e = 0.f, p = 0.f, q = 3.402823466e38f;
    __device__ __forceinline__ void add(float x) {
        const float t = __fadd_rn(s, x), v = __fsub_rn(t, s);
        e = __fadd_rn(e, __fadd_rn(__fsub_rn(s, __fsub_rn(t, v)), __fsub_rn(x, v)));
        s = t;
        p = __fadd_rn(p, fabsf(x));
        if (x != 0.f) q = fminf(q, fabsf(x));
    }
    __device__ __forceinline__ bool get(float& r) const {
        r = __fadd_rn(s, e);
        return q >= __fmul_rn(p, 0x1p-22f);
    }
};

__global__ void __launch_bounds__(256) k_vq_decode(const uint16_t* __restrict__ means16,
                                                   const uint8_t* __restrict__ idx, const float* __restrict__ cb,
                                                   int n, int stages, int cbs, float* __restrict__ means,
                                                   float* __restrict__ chol, float* __restrict__ color,
                                                   int aos_stride, uint32_t* status) {
    extern __shared__ float scb[];  // [2][stages][cbs][3]
    const int ncb = 2 * stages * cbs * 3;
    for (int i = threadIdx.x; i < ncb; i += blockDim.x) scb[i] = cb[i];
    __syncthreads();
    for (int g = blockIdx.x * blockDim.x + threadIdx.x; g < n; g += gridDim.x * blockDim.x) {
        const float mx = __half2float(__ushort_as_half(means16[2 * (size_t)g]));
        const float my = __half2float(__ushort_as_half(means16[2 * (size_t)g + 1]));
        float o[2][3];
        for (int a = 0; a < 2; ++a) {
            if (stages <= 2) {
                float acc[3] = {0.f, 0.f, 0.f};
                for (int s = 0; s < stages; ++s) {
                    int i = idx[((size_t)a * stages + s) * n + g];
                    if (i >= cbs) {  // index outside the codebook: skip the read
                        flag_error(status, kErrBounds);
                        i = 0;
                    }
                    const float* row = scb + (((size_t)a * stages + s) * cbs + i) * 3;
                    acc[0] = __fadd_rn(acc[0], row[0]);
                    acc[1] = __fadd_rn(acc[1], row[1]);
                    acc[2] = __fadd_rn(acc[2], row[2]);
                }
                o[a][0] = acc[0]; o[a][1] = acc[1]; o[a][2] = acc[2];
            } else {
                RowSum sum[3];
                for (int s = 0; s < stages; ++s) {
                    int i = idx[((size_t)a * stages + s) * n + g];
                    if (i >= cbs) {
                        flag_error(status, kErrBounds);
                        i = 0;
                    }
                    const float* row = scb + (((size_t)a * stages + s) * cbs + i) * 3;
                    for (int c = 0; c < 3; ++c) sum[c].add(row[c]);
                }
                bool ok = true;
                for (int c = 0; c < 3; ++c) ok &= sum[c].get(o[a][c]);
                if (!ok) {
                    double acc[3] = {0.0, 0.0, 0.0};
                    for (int s = 0; s < stages; ++s) {
                        int i = idx[((size_t)a * stages + s) * n + g];
                        if (i >= cbs) i = 0;
                        const float* row = scb + (((size_t)a * stages + s) * cbs + i) * 3;
                        for (int c = 0; c < 3; ++c) acc[c] += (double)row[c];
                    }
                    for (int c = 0; c < 3; ++c) o[a][c] = (float)acc[c];
                }
            }
        }
        if (aos_stride == 8) {
            float4* p = reinterpret_cast<float4*>(means) + 2 * (size_t)g;
            p[0] = make_float4(mx, my, o[0][0], o[0][1]);
            p[1] = make_float4(o[0][2], o[1][0], o[1][1], o[1][2]);
        } else {
            means[2 * (size_t)g] = mx;
            means[2 * (size_t)g + 1] = my;
            chol[3 * (size_t)g] = o[0][0];
            chol[3 * (size_t)g + 1] = o[0][1];
            chol[3 * (size_t)g + 2] = o[0][2];
            color[3 * (size_t)g] = o[1][0];
            color[3 * (size_t)g + 1] = o[1][1];
            color[3 * (size_t)g + 2] = o[1][2];
        }
    }
}

constexpr int kVqQuads = 2;  // quads per thread and round of the fast path
// From this count on, two-stage decodes keep eight copies of the codebook rows
// in shared memory (lane l reads copy l mod 8, so the eight rows of a 16-byte
// load phase fall on different banks; 128 KB for 2 x 256 entries, one block of
// 1024 threads per SM). Random rows otherwise collide about 2.7-fold, which
// alone takes 18 us of shared-memory time at 3.2 M. Graph-replayed, 2 x 256
// entries, eight copies / one: 600,000 Gaussians 7.4 / 7.0 us, 800,000 12.5 /
// 10.6, 1.2 M 14.0 / 15.7, 3.2 M 28.5 / 33.7 (before the staged stores 34.6). One
// stage gains nothing (25 us either way).
constexpr int kVqReplicated = 1200000;

// RowSum's FP64 case for Gaussian j of a quad. Not inlined: the compiler would
// otherwise run it for every value and choose.
template <int MAXS>
struct VqWords {
    uint32_t w[MAXS];
};
template <int MAXS>
__device__ __noinline__ float3 row_sum_fp64(VqWords<MAXS> ws, int j, const float4* rows, int copies, int stages,
                                            int cbs) {
    double d[3] = {0.0, 0.0, 0.0};
#pragma unroll
    for (int st = 0; st < MAXS; ++st) {
        if (st < stages) {
            int i = (ws.w[st] >> (8 * j)) & 0xff;
            if (i >= cbs) i = 0;
            const float4 r = rows[(st * cbs + i) * copies];
            d[0] += (double)r.x;
            d[1] += (double)r.y;
            d[2] += (double)r.z;
        }
    }
    return make_float3((float)d[0], (float)d[1], (float)d[2]);
}

// The decoded attribute a (0: Cholesky vector, 1: colour) of a quad from its
// index words w[stage] and the padded codebook rows: up to two stages as FP32
// sums (exact), more as RowSum.
template <int MAXS>
__device__ __forceinline__ void vq_quad(const uint32_t (&w)[MAXS], const float4* rows, int copies, int stages,
                                        int cbs, float (&o)[4][3], uint32_t* status) {
    auto row = [&](int st, int j) {
        int i = (w[st] >> (8 * j)) & 0xff;
        if (i >= cbs) {  // index outside the codebook: skip the read
            flag_error(status, kErrBounds);
            i = 0;
        }
        return rows[(st * cbs + i) * copies];
    };
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        if constexpr (MAXS <= 2) {
            float f[3] = {0.f, 0.f, 0.f};
#pragma unroll
            for (int st = 0; st < MAXS; ++st) {
                if (st < stages) {
                    const float4 r = row(st, j);
                    f[0] = __fadd_rn(f[0], r.x);
                    f[1] = __fadd_rn(f[1], r.y);
                    f[2] = __fadd_rn(f[2], r.z);
                }
            }
#pragma unroll
            for (int c = 0; c < 3; ++c) o[j][c] = f[c];
        } else {
            static_assert(MAXS <= kRowSumTerms, "RowSum is exact for eight terms");
            RowSum sum[3];
#pragma unroll
            for (int st = 0; st < MAXS; ++st) {
                if (MAXS == 3 || st < stages) {
                    const float4 r = row(st, j);
                    sum[0].add(r.x);
                    sum[1].add(r.y);
                    sum[2].add(r.z);
                }
            }
            bool ok = true;
#pragma unroll
            for (int c = 0; c < 3; ++c) ok &= sum[c].get(o[j][c]);
            if (!ok) {
                VqWords<MAXS> ws;
#pragma unroll
                for (int st = 0; st < MAXS; ++st) ws.w[st] = w[st];
                const float3 d = row_sum_fp64<MAXS>(ws, j, rows, copies, MAXS == 3 ? 3 : stages, cbs);
                o[j][0] = d.x;
                o[j][1] = d.y;
                o[j][2] = d.z;
            }
        }
    }
}

// Four consecutive Gaussians (a quad) per lane when every array is 16-byte
// aligned (the usual case): the FP16 positions of the four as one 16-byte
// load, each index plane as one 4-byte load, codebook rows from shared memory
// as one 16-byte load each (rows padded to four floats). Same arithmetic as
// k_vq_decode. 80 % of the bytes are written: the positions leave as one
// 32-byte store per lane, and the 48 bytes of each attribute go through the
// warp's corner of shared memory so that every store instruction writes 512
// contiguous bytes (three 16-byte stores 48 bytes apart fill half a sector
// each; one stage, 3.2 M: 32.5 -> 24.5 us).
template <int MAXS, int THREADS>
__global__ void __launch_bounds__(THREADS) k_vq_decode4(const uint4* __restrict__ means16,
                                                           const uint8_t* __restrict__ idx,
                                                           const float* __restrict__ cb, int n, int stages, int cbs,
                                                           float4* __restrict__ means, float4* __restrict__ chol,
                                                           float4* __restrict__ color, int copies, bool v8,
                                                           uint32_t* status) {
    extern __shared__ float4 srow[];  // [2][stages][cbs][copies] rows (x, y, z, 0), then [warps][96]
    const int nrow = 2 * stages * cbs * copies;
    for (int i = threadIdx.x; i < nrow; i += blockDim.x) {
        const int r = i / copies;
        srow[i] = make_float4(cb[3 * r], cb[3 * r + 1], cb[3 * r + 2], 0.f);
    }
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const float4* rows = srow + (lane & (copies - 1));  // this lane's copy
    float4* stage = srow + nrow + 96 * (threadIdx.x >> 5);
    const int nq = n >> 2;
    const int stride = gridDim.x * blockDim.x;
    for (int q0 = blockIdx.x * blockDim.x + (threadIdx.x & ~31); q0 < nq; q0 += kVqQuads * stride) {
        // every load of the round is issued before any quad is decoded
        uint4 h[kVqQuads];
        uint32_t w[kVqQuads][2][MAXS];
#pragma unroll
        for (int u = 0; u < kVqQuads; ++u) {
            const int q = q0 + u * stride + lane;
            const bool in = q < nq;
            h[u] = in ? means16[q] : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
            for (int a = 0; a < 2; ++a)
#pragma unroll
                for (int st = 0; st < MAXS; ++st) {
                    const uint32_t* I = reinterpret_cast<const uint32_t*>(idx + ((size_t)a * stages + st) * n);
                    w[u][a][st] = st < stages && in ? I[q] : 0u;
                }
        }
#pragma unroll
        for (int u = 0; u < kVqQuads; ++u) {
            const int qb = q0 + u * stride;  // the warp's first quad
            if (qb >= nq) break;
            const int valid = min(32, nq - qb);
            if (lane < valid) {
                const uint32_t hw[4] = {h[u].x, h[u].y, h[u].z, h[u].w};
                float mf[8];
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    mf[2 * j] = __half2float(__ushort_as_half((unsigned short)(hw[j] & 0xffffu)));
                    mf[2 * j + 1] = __half2float(__ushort_as_half((unsigned short)(hw[j] >> 16)));
                }
                const float4 m0 = make_float4(mf[0], mf[1], mf[2], mf[3]), m1 = make_float4(mf[4], mf[5], mf[6], mf[7]);
                float4* m = means + 2 * (size_t)(qb + lane);
                if (v8) {
                    st_global_v8(m, m0, m1);
                } else {
                    m[0] = m0;
                    m[1] = m1;
                }
            }
#pragma unroll
            for (int a = 0; a < 2; ++a) {
                float o[4][3];
                if (lane < valid) {
                    vq_quad<MAXS>(w[u][a], rows + a * stages * cbs * copies, copies, stages, cbs, o, status);
                    stage[3 * lane] = make_float4(o[0][0], o[0][1], o[0][2], o[1][0]);
                    stage[3 * lane + 1] = make_float4(o[1][1], o[1][2], o[2][0], o[2][1]);
                    stage[3 * lane + 2] = make_float4(o[2][2], o[3][0], o[3][1], o[3][2]);
                }
                __syncwarp();
                float4* dst = (a == 0 ? chol : color) + 3 * (size_t)qb;
#pragma unroll
                for (int i = 0; i < 3; ++i)
                    if (lane + 32 * i < 3 * valid) dst[lane + 32 * i] = stage[lane + 32 * i];
                __syncwarp();
            }
        }
    }
}

// The paper's codec (Sec. 3.3): FP16 positions, the b-bit Cholesky codes
// reconstructed as l_bar_i = code_i gamma_i + beta_i (Eq. 9, the same two
// roundings as the fit's quantiser), and the RVQ colour as the FP64 sum of
// the chosen entries in stage order, rounded once (as the fit's formation).
__global__ void __launch_bounds__(256) k_codec_decode(const uint16_t* __restrict__ means16,
                                                      const uchar4* __restrict__ codes, GammaBeta gb,
                                                      const uint8_t* __restrict__ idx, const float* __restrict__ cb,
                                                      int n, int stages, int size, float* __restrict__ means,
                                                      float* __restrict__ chol, float* __restrict__ color,
                                                      uint32_t* status) {
    extern __shared__ float scb[];  // [stages][size][3]
    pdl_wait();
    for (int i = threadIdx.x; i < stages * size * 3; i += blockDim.x) scb[i] = cb[i];
    __syncthreads();
    const bool two = stages <= 2;  // then one FP32 addition is the exact sum rounded once
    for (int g = blockIdx.x * blockDim.x + threadIdx.x; g < n; g += gridDim.x * blockDim.x) {
        means[2 * (size_t)g] = __half2float(__ushort_as_half(means16[2 * (size_t)g]));
        means[2 * (size_t)g + 1] = __half2float(__ushort_as_half(means16[2 * (size_t)g + 1]));
        const uchar4 q = codes[g];
        chol[3 * (size_t)g] = __fadd_rn(__fmul_rn((float)q.x, gb.v[0]), gb.v[3]);
        chol[3 * (size_t)g + 1] = __fadd_rn(__fmul_rn((float)q.y, gb.v[1]), gb.v[4]);
        chol[3 * (size_t)g + 2] = __fadd_rn(__fmul_rn((float)q.z, gb.v[2]), gb.v[5]);
        double s0 = 0.0, s1 = 0.0, s2 = 0.0;
        float f0 = 0.f, f1 = 0.f, f2 = 0.f;
        for (int m = 0; m < stages; ++m) {
            int j = idx[(size_t)m * n + g];
            if (j >= size) {  // index outside the codebook: skip the read
                flag_error(status, kErrBounds);
                j = 0;
            }
            const float* e = scb + ((size_t)m * size + j) * 3;
            if (two) {
                f0 = __fadd_rn(f0, e[0]);
                f1 = __fadd_rn(f1, e[1]);
                f2 = __fadd_rn(f2, e[2]);
            } else {
                s0 = __dadd_rn(s0, (double)e[0]);
                s1 = __dadd_rn(s1, (double)e[1]);
                s2 = __dadd_rn(s2, (double)e[2]);
            }
        }
        color[3 * (size_t)g] = two ? f0 : (float)s0;
        color[3 * (size_t)g + 1] = two ? f1 : (float)s1;
        color[3 * (size_t)g + 2] = two ? f2 : (float)s2;
    }
}

}  // namespace

cudaError_t launch_codec_decode(const uint16_t* means16, const uint8_t* codes, const float* gamma_beta,
                                const uint8_t* idx, const float* cb, int32_t n, int32_t stages, int32_t size,
                                float* means, float* chol, float* color, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    GammaBeta gb;
    for (int i = 0; i < 6; ++i) gb.v[i] = gamma_beta[i];
    const int blocks = std::max(1, std::min((n + 255) / 256, sm_count() * 4));
    return launch_pdl(k_codec_decode, dim3(blocks), dim3(256), (size_t)stages * size * 3 * sizeof(float), s, means16,
                      reinterpret_cast<const uchar4*>(codes), gb, idx, cb, n, stages, size, means, chol, color,
                      device_status());
}

cudaError_t launch_vq_decode(const uint16_t* means16, const uint8_t* idx, const float* cb, int32_t n, int32_t stages,
                             int32_t cb_size, float* means, float* chol, float* color, int32_t out_stride_aos,
                             cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    auto a16 = [](const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; };
    if (out_stride_aos == 0 && n % 4 == 0 && a16(means16) && (reinterpret_cast<uintptr_t>(idx) & 3) == 0 &&
        a16(means) && a16(chol) && a16(color)) {
        auto go = [&](auto kern, int threads, int copies, int per_sm) {
            const size_t smem = ((size_t)2 * stages * cb_size * copies + 96 * (threads / 32)) * sizeof(float4);
            cudaError_t e = smem_optin(reinterpret_cast<const void*>(kern), (int)smem);
            if (e != cudaSuccess) return e;
            const int blocks = std::max(1, std::min((n / 4 + threads - 1) / threads, sm_count() * per_sm));
            kern<<<blocks, threads, smem, s>>>(reinterpret_cast<const uint4*>(means16), idx, cb, n, stages, cb_size,
                                               reinterpret_cast<float4*>(means), reinterpret_cast<float4*>(chol),
                                               reinterpret_cast<float4*>(color), copies,
                                               (reinterpret_cast<uintptr_t>(means) & 31) == 0, device_status());
            return cudaGetLastError();
        };
        if (stages == 2 && n >= kVqReplicated) return go(k_vq_decode4<2, 1024>, 1024, 8, 1);
        if (stages <= 2) return go(k_vq_decode4<2, 256>, 256, 1, 8);
        return stages == 3 ? go(k_vq_decode4<3, 256>, 256, 1, 8) : go(k_vq_decode4<8, 256>, 256, 1, 8);
    }
    const size_t smem = (size_t)2 * stages * cb_size * 3 * sizeof(float);
    {
        cudaError_t e = smem_optin(reinterpret_cast<const void*>(k_vq_decode), (int)smem);
        if (e != cudaSuccess) return e;
    }
    int dev = 0, nsm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    if (nsm <= 0) nsm = 148;
    const int blocks = std::max(1, std::min((n + 255) / 256, nsm * 4));
    k_vq_decode<<<blocks, 256, smem, s>>>(means16, idx, cb, n, stages, cb_size, means, chol, color, out_stride_aos,
                                          device_status());
    return cudaGetLastError();
}

}  // namespace gi
