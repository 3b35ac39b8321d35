// blend.cu -- sorted alpha-blending render and its gradients (Sec. 3.2,
// Eq. 3-4): the rasterisation that accumulated summation replaces, built to
// measure that replacement on the same hardware (Table 3's "w/o AR").
//
//   alpha_n = min(0.99, o_n exp(-sigma_n)), skipped when alpha_n < 1/255,
//   C_i = sum_n c_n alpha_n T_n, T_n = prod_{m < n} (1 - alpha_m),
//   the walk stopping before the Gaussian that would take T below 1e-4
//
// over each tile's list in ascending Gaussian index (a 2D image has no depth
// to sort by). One CTA per 16 x 16 tile, a few pixels per thread: the list is
// staged through shared memory in chunks and every pixel walks it front to
// back, the CTA stopping once all its pixels have saturated.
//
// Gradients, per pixel and front to back again with the same operations
// (so the same decisions), using the final colour C from the forward pass:
// with the prefix P_n = sum_{m <= n} c_m alpha_m T_m and the suffix
// S = C - P_n,
//   dL/dc_n     = sum_i dL/dC_i alpha_n T_n
//   dL/dalpha_n = sum_ch dL/dC (c_n T_n - S / (1 - alpha_n))
// and, unless alpha_n was clamped, dL/dsigma_n = -dL/dalpha_n alpha_n and
// dL/do_n = dL/dalpha_n exp(-sigma_n). The per-pixel terms of each list entry
// are summed over the tile's 256 pixels (a thread's pixels in registers, warp
// butterflies, then the warps in order) into the same eight per-pair sums the accumulated backward writes
// (colour, and e~ (dx, dy, dx^2, dx dy, dy^2) with e~ = -dL/dsigma) plus a
// ninth for the opacity, at the pair's emission index; the per-Gaussian
// reduction is then shared with the accumulated path. Deterministic.
#include <type_traits>

#include "kernels.cuh"

namespace gi {
namespace {

constexpr int kBT = 16;
constexpr int kBPix = kBT * kBT;
constexpr int kBWarps = kBPix / 32;
constexpr int kBChunk = 32;  // list entries per backward chunk
#ifndef GI_BLEND_RENDER_PX
#define GI_BLEND_RENDER_PX 2
#endif
#ifndef GI_BLEND_BACKWARD_PX
#define GI_BLEND_BACKWARD_PX 4
#endif
constexpr int kBlendRenderPx = GI_BLEND_RENDER_PX;      // pixels per thread, forward
constexpr int kBlendBackwardPx = GI_BLEND_BACKWARD_PX;  // pixels per thread, backward

// Packed products and sums that stay separate operations: the walk's decisions
// (alpha >= 1/255, T >= 1e-4) depend on every rounding. The assembler contracts
// a mul.rn.f32x2 whose result feeds an add.rn.f32x2 into one fused operation
// (unlike the scalar forms; seen as different last bits in 45 % of the
// pixels), so such a sum is written as product * one + c with one = 1.0f from
// a kernel argument, which rounds exactly as the addition.
__device__ __forceinline__ float2 add_product(float2 product, float2 c, float one) {
    return __ffma2_rn(product, make_float2(one, one), c);
}

// Pixels of a thread: PX rows of one column (so dx and its products are shared),
// a warp covers a block of 8 x 8 pixels (PX = 2) or 16 x 8 (PX = 4).
template <int PX>
struct PixMap {
    static constexpr int BW = PX == 2 ? 8 : 16, BH = 8;  // a warp's block
    static constexpr int NW = kBPix / (32 * PX);         // warps (blocks) per tile
    static __device__ __forceinline__ int bx(int warp) { return (warp * BW) % kBT; }
    static __device__ __forceinline__ int by(int warp) { return (warp * BW) / kBT * BH; }
    static __device__ __forceinline__ int x(int tid) { return bx(tid >> 5) + (tid & 31) % BW; }
    static __device__ __forceinline__ int y(int tid) { return by(tid >> 5) + (tid & 31) / BW * PX; }
};

// exp(-sigma) of a record at two pixels of a column, with explicit roundings
// (packed operations round as the scalar ones) so that the forward and the
// backward kernel compute the same values. z1s = (m11 dx)^2, t = m21 dx.
__device__ __forceinline__ float2 blend_w2(float m22, float z1s, float t, float2 dy, float one) {
    const float2 z2 = add_product(__fmul2_rn(make_float2(m22, m22), dy), make_float2(t, t), one);
    const float2 q = add_product(__fmul2_rn(z2, z2), make_float2(z1s, z1s), one);
    return make_float2(ex2(-q.x), ex2(-q.y));
}

// Blocks of the tile at (x0, y0) in which some pixel may reach alpha >= 1/255
// (bit = block of Map): the smallest q = |M d|^2 over each block's pixel centres, on
// its edges unless the Gaussian's centre lies inside, against log2(255 o).
// An entry left out of a block would be skipped at each of its pixels, so
// the results do not change. The margin of 0.02 covers the rounding of both
// sides while the terms of z1 and z2 stay below 1000 (their errors then stay
// below 4e-4, and q's, near the threshold of at most 8, below 3e-3); larger
// ones (needles) keep every block, as does anything that is not a number.
// About 47 % of the (entry, 8 x 8 block) pairs of a fit's lists drop out.
template <class Map>
__device__ __forceinline__ uint32_t reach_mask(const float4 r0, const float4 r1, float o, float x0, float y0) {
    const float thr = log2f(255.f * o) + 0.02f;
    const float m11 = r0.z, m21 = r0.w, m22 = r1.x;
    const float inv22 = 1.f / m22, k = m21 * m22 / (m11 * m11 + m21 * m21);
    const float ax = x0 + 0.5f - r0.x, ay = y0 + 0.5f - r0.y;  // the tile's first pixel centre - mu
    const float far = (fabsf(m11) + fabsf(m21)) * fmaxf(fabsf(ax), fabsf(ax + 15.f)) +
                      fabsf(m22) * fmaxf(fabsf(ay), fabsf(ay + 15.f));
    if (!(far < 1000.f)) return (1u << Map::NW) - 1u;
    uint32_t mask = 0;
#pragma unroll
    for (int w = 0; w < Map::NW; ++w) {
        const float xl = ax + (float)Map::bx(w), xh = xl + (float)(Map::BW - 1);
        const float yl = ay + (float)Map::by(w), yh = yl + (float)(Map::BH - 1);
        float q = 0.f;
        if (xl > 0.f || xh < 0.f || yl > 0.f || yh < 0.f) {
            q = __int_as_float(0x7f800000);
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                const float dx = i ? xh : xl;  // edge of fixed x
                const float t = m21 * dx, z1 = m11 * dx;
                const float z2 = fmaf(m22, fminf(fmaxf(-t * inv22, yl), yh), t);
                q = fminf(q, fmaf(z2, z2, z1 * z1));
                const float dy = i ? yh : yl;  // edge of fixed y
                const float d = fminf(fmaxf(-k * dy, xl), xh);
                const float u1 = m11 * d, u2 = fmaf(m21, d, m22 * dy);
                q = fminf(q, fmaf(u2, u2, u1 * u1));
            }
        }
        if (!(q > thr)) mask |= 1u << w;
    }
    return mask;
}

// Reduce-scatter of the first 8 per-lane values over the warp (9 shuffles
// instead of 8 x 5): lanes 4s .. 4s + 3 return the warp sum of slot s. Fixed
// order, so deterministic.
__device__ __forceinline__ float warp_reduce_scatter8(float (&v)[9], int lane) {
#pragma unroll
    for (int w = 4; w >= 1; w >>= 1) {  // offsets 16, 8, 4: keep w slots
        const int off = 4 * w;
        const bool up = (lane & off) != 0;
#pragma unroll
        for (int i = 0; i < w; ++i) {
            const float send = up ? v[i] : v[i + w];
            const float keep = up ? v[i + w] : v[i];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, send, off);
        }
    }
    v[0] += __shfl_xor_sync(0xffffffffu, v[0], 2);
    v[0] += __shfl_xor_sync(0xffffffffu, v[0], 1);
    return v[0];
}

struct TileGeo {
    ImgDesc d;
    int img, tx, ty, b, e;
};

__device__ __forceinline__ TileGeo tile_geo(const Batch& B, const int2* ranges, int t, uint32_t* status) {
    TileGeo g;
    g.img = image_of_tile(B, t);
    g.d = img_desc(B, g.img);
    const int lt = t - g.d.tile_base;
    g.tx = lt % g.d.tw;
    g.ty = lt / g.d.tw;
    const int2 rg = ranges[t];
    const bool ok = gi_in_bounds(rg.x >= 0 && rg.x <= rg.y, status);
    g.b = ok ? rg.x : 0;
    g.e = ok ? rg.y : 0;
    return g;
}

// PX pixels per thread: each staged record is read from shared memory once
// per thread and applied to all its pixels; a warp only walks the entries
// that reach its block (reach_mask), and stops when its pixels have saturated.
// Bound by instruction issue. Skipping by block, packed arithmetic on two rows
// and selects instead of branches: 39.7 -> 20 M warp instructions, 49.5 -> 31
// us at 768x512 / 30,000 (four pixels a thread: 36 us).
template <int PX>
__global__ void __launch_bounds__(kBPix / PX) k_render_blend(const float4* __restrict__ rec_binned,
                                                             const uint32_t* __restrict__ ids,
                                                             const float* __restrict__ o_eff,
                                                             const int2* __restrict__ ranges, Batch B,
                                                             const float* __restrict__ target,
                                                             float* __restrict__ out, int32_t* __restrict__ n_last,
                                                             float* __restrict__ dl_tiled,
                                                             double* __restrict__ loss_sum, float one, uint32_t* status) {
    constexpr int NT = kBPix / PX;
    constexpr int kStage = 128;  // list entries staged per chunk
    static_assert(PX % 2 == 0, "pixels in packed pairs");
    __shared__ float4 s_rec[kStage][2];
    __shared__ float s_o[kStage];
    __shared__ uint32_t s_mask[kStage];
    __shared__ float s_red[32];
    pdl_wait();
    const int t = blockIdx.x;
    const TileGeo tg = tile_geo(B, ranges, t, status);
    const ImgDesc& d = tg.d;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int px = PixMap<PX>::x(tid), py = PixMap<PX>::y(tid);
    const int x = tg.tx * kBT + px, y0 = tg.ty * kBT + py;
    const float cx = (float)x + 0.5f;
    float2 cy[PX / 2], C0[PX / 2], C1[PX / 2], C2[PX / 2], Tr[PX / 2];  // pairs of rows
    int last[PX];
    unsigned done = 0u;  // bit i: pixel i has stopped (or lies outside the image)
#pragma unroll
    for (int i = 0; i < PX; ++i) {
        if (i % 2 == 0) {
            cy[i / 2] = make_float2((float)(y0 + i) + 0.5f, (float)(y0 + i + 1) + 0.5f);
            C0[i / 2] = C1[i / 2] = C2[i / 2] = make_float2(0.f, 0.f);
            Tr[i / 2] = make_float2(1.f, 1.f);
        }
        last[i] = 0;
        if (!(x < d.W && y0 + i < d.H)) done |= 1u << i;
    }
    constexpr unsigned kAll = (1u << PX) - 1u;
    for (int base = tg.b; base < tg.e; base += kStage) {
        if (__syncthreads_and(done == kAll)) break;  // also orders the restaging after the last chunk's reads
        for (int s = tid; s < kStage; s += NT) {
            const int k = base + s;
            uint32_t m = 0;
            if (k < tg.e) {
                uint32_t g = ids[k];
                if (!gi_in_bounds(g < (uint32_t)B.total_gauss, status)) g = 0;
                const float4 r0 = rec_binned[2 * (size_t)k], r1 = rec_binned[2 * (size_t)k + 1];
                const float o = o_eff[g];
                s_rec[s][0] = r0;
                s_rec[s][1] = r1;
                s_o[s] = o;
                m = reach_mask<PixMap<PX>>(r0, r1, o, (float)(tg.tx * kBT), (float)(tg.ty * kBT));
            }
            s_mask[s] = m;
        }
        __syncthreads();
        for (int g0 = 0; g0 < kStage && base + g0 < tg.e; g0 += 32) {
            uint32_t todo = __ballot_sync(0xffffffffu, (s_mask[g0 + lane] >> warp) & 1u);
            if (__all_sync(0xffffffffu, done == kAll)) break;
            while (todo) {
                const int j = g0 + __ffs(todo) - 1;
                todo &= todo - 1u;
                const float4 r0 = s_rec[j][0], r1 = s_rec[j][1];
                const float o = s_o[j];
                const float dx = __fsub_rn(cx, r0.x);
                const float z1 = __fmul_rn(r0.z, dx);
                const float z1s = __fmul_rn(z1, z1), tt = __fmul_rn(r0.w, dx);
                // Branch-free: a pixel that skips the entry (or has stopped)
                // adds zero and keeps its state.
#pragma unroll
                for (int h = 0; h < PX / 2; ++h) {
                    const float2 dy = __fadd2_rn(cy[h], make_float2(-r0.y, -r0.y));
                    float2 a = __fmul2_rn(make_float2(o, o), blend_w2(r1.x, z1s, tt, dy, one));
                    bool u0 = !(a.x < kBlendAlphaMin) && !(done & (1u << (2 * h)));
                    bool u1 = !(a.y < kBlendAlphaMin) && !(done & (2u << (2 * h)));
                    a = make_float2(fminf(a.x, kBlendAlphaMax), fminf(a.y, kBlendAlphaMax));
                    const float2 test =
                        __fmul2_rn(Tr[h], __fadd2_rn(make_float2(1.f, 1.f), make_float2(-a.x, -a.y)));
                    if (u0 && test.x < kBlendTMin) done |= 1u << (2 * h);
                    if (u1 && test.y < kBlendTMin) done |= 2u << (2 * h);
                    u0 = u0 && !(test.x < kBlendTMin);
                    u1 = u1 && !(test.y < kBlendTMin);
                    float2 at = __fmul2_rn(a, Tr[h]);
                    at = make_float2(u0 ? at.x : 0.f, u1 ? at.y : 0.f);
                    C0[h] = add_product(__fmul2_rn(make_float2(r1.y, r1.y), at), C0[h], one);
                    C1[h] = add_product(__fmul2_rn(make_float2(r1.z, r1.z), at), C1[h], one);
                    C2[h] = add_product(__fmul2_rn(make_float2(r1.w, r1.w), at), C2[h], one);
                    Tr[h] = make_float2(u0 ? test.x : Tr[h].x, u1 ? test.y : Tr[h].y);
                    const int pos = base - tg.b + j + 1;
                    last[2 * h] = u0 ? pos : last[2 * h];
                    last[2 * h + 1] = u1 ? pos : last[2 * h + 1];
                }
            }
        }
    }
    const float scale = 2.0f / (3.0f * (float)d.W * (float)d.H);
    float lsum = 0.f;
#pragma unroll
    for (int i = 0; i < PX; ++i) {
        const int y = y0 + i;
        float dl0 = 0.f, dl1 = 0.f, dl2 = 0.f;
        if (x < d.W && y < d.H) {
            const int64_t pix = d.pix_base + (int64_t)y * d.W + x;
            const float c0 = i % 2 ? C0[i / 2].y : C0[i / 2].x, c1 = i % 2 ? C1[i / 2].y : C1[i / 2].x,
                        c2 = i % 2 ? C2[i / 2].y : C2[i / 2].x;
            out[3 * pix] = c0;
            out[3 * pix + 1] = c1;
            out[3 * pix + 2] = c2;
            if (n_last) n_last[pix] = last[i];
            if (target) {
                const float r0 = c0 - target[3 * pix], r1 = c1 - target[3 * pix + 1], r2 = c2 - target[3 * pix + 2];
                lsum = fmaf(r2, r2, fmaf(r1, r1, fmaf(r0, r0, lsum)));
                dl0 = r0 * scale;
                dl1 = r1 * scale;
                dl2 = r2 * scale;
            }
        }
        if (dl_tiled) {  // planar per tile, as the accumulated render writes it
            float* dt = dl_tiled + (size_t)t * 3 * kBPix + (py + i) * kBT + px;
            dt[0] = dl0;
            dt[kBPix] = dl1;
            dt[2 * kBPix] = dl2;
        }
    }
    if (target && loss_sum) {
        lsum = warp_sum(lsum);
        if (lane == 0) s_red[warp] = lsum;
        __syncthreads();
        if (tid == 0) {
            float s = 0.f;
            for (int w = 0; w < NT / 32; ++w) s += s_red[w];
            atomicAdd(&loss_sum[tg.img], (double)s);
        }
    }
}

// Emission index of pair (tile tx, ty; Gaussian g): pair_off[g] plus the
// tile's row-major rank inside g's rect; -1 when out of range.
__device__ __forceinline__ int64_t emission_index(const int4* rect, const int64_t* pair_off, uint32_t g, int tx,
                                                  int ty, int64_t capacity) {
    const int4 r = rect[g];
    const int64_t e = pair_off[g] + (int64_t)(ty - r.y) * (r.z - r.x) + (tx - r.x);
    return (e >= 0 && e < capacity) ? e : -1;
}

// The same walk for the gradients. Also bound by issue; two pixels per packed
// operation, selects instead of branches, rows no pixel of which sees the
// entry passed over and a reduce-scatter of 8 values plus one butterfly instead
// of 16: 105 -> 85 us at 768x512 / 30,000 with the same sums bit for bit (a
// pixel's column, the threads' row order and the reduction tree are kept).
// Warps on 8 x 8 or 16 x 8 blocks with the forward's reach mask take 74 us but
// round the sums in another order, which moves the discontinuous walk of the
// next step; a mask over two-row strips saves less than it costs.
template <int PX>
__global__ void __launch_bounds__(kBPix / PX) k_backward_blend(
    const float4* __restrict__ rec_binned, const uint32_t* __restrict__ ids, const float* __restrict__ o_eff,
    const int2* __restrict__ ranges, const int4* __restrict__ rect, const int64_t* __restrict__ pair_off, Batch B,
    const float* __restrict__ out, const int32_t* __restrict__ n_last, const float* __restrict__ dl_tiled,
    int64_t capacity, float* __restrict__ partial, float* __restrict__ partial_o, float one, AdamCfg adam,
    uint32_t* status) {
    constexpr int NT = kBPix / PX, NW = NT / 32;
    __shared__ float4 s_rec[kBChunk][2];
    __shared__ float s_o[kBChunk];
    __shared__ int64_t s_e[kBChunk];
    __shared__ float s_red[kBChunk][NW][9];
    __shared__ uint32_t s_has[NW];  // entries of the chunk with a sum from warp w
    __shared__ int s_max[NW];
    pdl_wait();
    if (adam.step && blockIdx.x == 0 && threadIdx.x == 0) begin_update(adam);
    const int t = blockIdx.x;
    const TileGeo tg = tile_geo(B, ranges, t, status);
    const ImgDesc& d = tg.d;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const float* dt = dl_tiled + (size_t)t * 3 * kBPix;
    // The thread's pixels lie in one column, rows tid / 16 + i NT / 16, held in
    // pairs: row centres, dL/dC, final colour, colour so far, T.
    const int x = tg.tx * kBT + tid % kBT;
    const float cx = (float)x + 0.5f;
    float2 cy[PX / 2], g0[PX / 2], g1[PX / 2], g2[PX / 2], Cf0[PX / 2], Cf1[PX / 2], Cf2[PX / 2], P0[PX / 2],
        P1[PX / 2], P2[PX / 2], Tr[PX / 2];
    int nl[PX];
    auto put = [](float2& v, int i, float f) { (i % 2 ? v.y : v.x) = f; };
    auto get = [](const float2& v, int i) { return i % 2 ? v.y : v.x; };
    int mine = 0;
    bool finite = true;
#pragma unroll
    for (int i = 0; i < PX; ++i) {
        const int q = tid + NT * i, h = i / 2;
        const int y = tg.ty * kBT + q / kBT;
        put(cy[h], i, (float)y + 0.5f);
        put(g0[h], i, dt[q]);
        put(g1[h], i, dt[kBPix + q]);
        put(g2[h], i, dt[2 * kBPix + q]);
        float c0 = 0.f, c1 = 0.f, c2 = 0.f;
        nl[i] = 0;
        if (x < d.W && y < d.H) {
            const int64_t pix = d.pix_base + (int64_t)y * d.W + x;
            c0 = out[3 * pix];
            c1 = out[3 * pix + 1];
            c2 = out[3 * pix + 2];
            nl[i] = min(n_last[pix], tg.e - tg.b);
        }
        put(Cf0[h], i, c0);
        put(Cf1[h], i, c1);
        put(Cf2[h], i, c2);
        P0[h] = P1[h] = P2[h] = make_float2(0.f, 0.f);
        Tr[h] = make_float2(1.f, 1.f);
        mine = max(mine, nl[i]);
        finite = finite && isfinite(dt[q]) && isfinite(dt[kBPix + q]) && isfinite(dt[2 * kBPix + q]);
    }
    const bool all_finite = __all_sync(0xffffffffu, finite);
    const int wmax = __reduce_max_sync(0xffffffffu, mine);  // entries this warp walks
    if (lane == 0) s_max[warp] = wmax;
    __syncthreads();
    int nmax = 0;
#pragma unroll
    for (int w = 0; w < NW; ++w) nmax = max(nmax, s_max[w]);
    for (int base = tg.b; base < tg.b + nmax; base += kBChunk) {
        const int n = min(kBChunk, tg.b + nmax - base);
        if (tid < n) {
            const int k = base + tid;
            uint32_t g = ids[k];
            const bool ok = gi_in_bounds(g < (uint32_t)B.total_gauss, status);
            if (!ok) g = 0;
            s_rec[tid][0] = rec_binned[2 * (size_t)k];
            s_rec[tid][1] = rec_binned[2 * (size_t)k + 1];
            s_o[tid] = o_eff[g];
            s_e[tid] = ok ? emission_index(rect, pair_off, g, tg.tx, tg.ty, capacity) : -1;
        }
        __syncthreads();
        const int walk = min(n, wmax - (base - tg.b));
        uint32_t has = 0;
        // A pixel that skips an entry adds dL/dC * 0, which is zero only while
        // dL/dC is finite: with a non-finite target pixel in the warp's rows the
        // skipped products are left out (as a branch in every walk it would cost
        // issue slots; here the usual walk is unchanged).
        auto walk_entries = [&](auto skip_zeros) {
            for (int j = 0; j < walk; ++j) {
                const float4 r0 = s_rec[j][0], r1 = s_rec[j][1];
                const float o = s_o[j];
                const int pos = base - tg.b + j;
                const float dx = __fsub_rn(cx, r0.x);
                const float z1 = __fmul_rn(r0.z, dx);
                const float z1s = __fmul_rn(z1, z1), tt = __fmul_rn(r0.w, dx);
                const float2 c0 = make_float2(r1.y, r1.y), c1 = make_float2(r1.z, r1.z), c2 = make_float2(r1.w, r1.w);
                const float2 m1 = make_float2(-1.f, -1.f);
                float v[9] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
                // Branch-free, two pixels at a time: a pixel that skips the entry
                // (or stopped before it) adds zeros and keeps its state; a pair of
                // rows none of whose pixels sees the entry is passed over.
#pragma unroll
                for (int h = 0; h < PX / 2; ++h) {
                    const float2 dy = __fadd2_rn(cy[h], make_float2(-r0.y, -r0.y));
                    const float2 w = blend_w2(r1.x, z1s, tt, dy, one);
                    float2 a = __fmul2_rn(make_float2(o, o), w);
                    const bool u0 = !(a.x < kBlendAlphaMin) && pos < nl[2 * h];
                    const bool u1 = !(a.y < kBlendAlphaMin) && pos < nl[2 * h + 1];
                    if (!__any_sync(0xffffffffu, u0 || u1)) continue;
                    has |= 1u << j;
                    const bool f0 = u0 && !(a.x > kBlendAlphaMax), f1 = u1 && !(a.y > kBlendAlphaMax);  // not clamped
                    a = make_float2(fminf(a.x, kBlendAlphaMax), fminf(a.y, kBlendAlphaMax));
                    float2 at = __fmul2_rn(a, Tr[h]);
                    at = make_float2(u0 ? at.x : 0.f, u1 ? at.y : 0.f);
                    P0[h] = add_product(__fmul2_rn(c0, at), P0[h], one);  // as the forward pass rounds them
                    P1[h] = add_product(__fmul2_rn(c1, at), P1[h], one);
                    P2[h] = add_product(__fmul2_rn(c2, at), P2[h], one);
                    const float2 keep = __fadd2_rn(make_float2(1.f, 1.f), make_float2(-a.x, -a.y));
                    const float2 ninv = make_float2(-__fdividef(1.f, keep.x), -__fdividef(1.f, keep.y));
                    // dL/dalpha = sum_ch dL/dC (c T - (C - P) / (1 - alpha))
                    const float2 A = __ffma2_rn(c0, Tr[h], __fmul2_rn(__ffma2_rn(P0[h], m1, Cf0[h]), ninv));
                    const float2 Bb = __ffma2_rn(c1, Tr[h], __fmul2_rn(__ffma2_rn(P1[h], m1, Cf1[h]), ninv));
                    const float2 C = __ffma2_rn(c2, Tr[h], __fmul2_rn(__ffma2_rn(P2[h], m1, Cf2[h]), ninv));
                    float2 dla = __ffma2_rn(g2[h], C, __ffma2_rn(g0[h], A, __fmul2_rn(g1[h], Bb)));
                    dla = make_float2(f0 ? dla.x : 0.f, f1 ? dla.y : 0.f);
                    const float2 ee = __fmul2_rn(dla, a);  // -dL/dsigma
                    const float2 ex = __fmul2_rn(ee, make_float2(dx, dx)), ey = __fmul2_rn(ee, dy);
#pragma unroll
                    for (int i = 0; i < 2; ++i) {  // one pixel after the other: the order of the sums
                        if (decltype(skip_zeros)::value ? (i ? u1 : u0) : true) {
                            v[0] = fmaf(get(g0[h], i), get(at, i), v[0]);
                            v[1] = fmaf(get(g1[h], i), get(at, i), v[1]);
                            v[2] = fmaf(get(g2[h], i), get(at, i), v[2]);
                        }
                        v[3] = __fadd_rn(v[3], get(ex, i));
                        v[4] = __fadd_rn(v[4], get(ey, i));
                        v[5] = fmaf(get(ex, i), dx, v[5]);
                        v[6] = fmaf(get(ex, i), get(dy, i), v[6]);
                        v[7] = fmaf(get(ey, i), get(dy, i), v[7]);
                        v[8] = fmaf(get(dla, i), get(w, i), v[8]);
                    }
                    const float2 Tn = __fmul2_rn(Tr[h], keep);
                    Tr[h] = make_float2(u0 ? Tn.x : Tr[h].x, u1 ? Tn.y : Tr[h].y);
                }
                if (!((has >> j) & 1u)) continue;
                const float s8 = warp_sum(v[8]), sum = warp_reduce_scatter8(v, lane);
                if ((lane & 3) == 0) s_red[j][warp][lane >> 2] = sum;
                if (lane == 1) s_red[j][warp][8] = s8;
            }
        };
        if (all_finite)
            walk_entries(std::false_type{});
        else
            walk_entries(std::true_type{});
        if (lane == 0) s_has[warp] = has;
        __syncthreads();
        for (int i = tid; i < n * 9; i += NT) {
            const int j = i / 9, q = i % 9;
            float s = 0.f;
#pragma unroll
            for (int w = 0; w < NW; ++w)
                if ((s_has[w] >> j) & 1u) s += s_red[j][w][q];
            const int64_t ei = s_e[j];
            if (ei >= 0) {
                if (q < 8)
                    partial[8 * ei + q] = s;
                else
                    partial_o[ei] = s;
            }
        }
        __syncthreads();
    }
    // Entries past every pixel's stop contribute nothing: zero their sums.
    for (int k = tg.b + nmax + tid; k < tg.e; k += NT) {
        const uint32_t g = ids[k];
        if (!gi_in_bounds(g < (uint32_t)B.total_gauss, status)) continue;
        const int64_t ei = emission_index(rect, pair_off, g, tg.tx, tg.ty, capacity);
        if (ei >= 0) {
            reinterpret_cast<float4*>(partial)[2 * ei] = make_float4(0.f, 0.f, 0.f, 0.f);
            reinterpret_cast<float4*>(partial)[2 * ei + 1] = make_float4(0.f, 0.f, 0.f, 0.f);
            partial_o[ei] = 0.f;
        }
    }
}

}  // namespace

cudaError_t launch_render_blend(const float4* rec_binned, const uint32_t* ids, const int2* ranges, const Batch& B,
                                const float* target, float* out, float* dl_tiled, double* loss_sum, uint32_t* status,
                                cudaStream_t s) {
    if (B.total_tiles <= 0) return cudaSuccess;
    if (B.tile != kBT) return cudaErrorInvalidValue;
    return launch_pdl(k_render_blend<kBlendRenderPx>, dim3(B.total_tiles), dim3(kBPix / kBlendRenderPx), 0, s,
                      rec_binned, ids, B.opac.o, ranges, B, target, out, B.opac.n_last, dl_tiled, loss_sum, 1.0f, status);
}

cudaError_t launch_backward_blend(const float4* rec_binned, const uint32_t* ids, const int2* ranges, const int4* rect,
                                  const int64_t* pair_off, const Batch& B, const float* out, const float* dl_tiled,
                                  int64_t capacity, float4* partial, uint32_t* status, cudaStream_t s, const AdamCfg* adam) {
    if (B.total_tiles <= 0) return cudaSuccess;
    if (B.tile != kBT) return cudaErrorInvalidValue;
    return launch_pdl(k_backward_blend<kBlendBackwardPx>, dim3(B.total_tiles), dim3(kBPix / kBlendBackwardPx), 0, s,
                      rec_binned, ids, B.opac.o, ranges, rect, pair_off, B, out, B.opac.n_last, dl_tiled, capacity,
                      reinterpret_cast<float*>(partial), B.opac.partial, 1.0f, adam ? *adam : AdamCfg{}, status);
}

}  // namespace gi
