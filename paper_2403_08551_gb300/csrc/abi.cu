// abi.cu -- extern "C" entry points of libgi for the per-stage operations:
// validation, workspace carve-up and launches. See include/gi.h.
#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <map>
#include <mutex>
#include <utility>

#include "kernels.cuh"
#include "pairs_wait.cuh"

namespace gi {

namespace {
thread_local char t_err[512] = "";
__device__ uint32_t g_dev_status;

bool aligned(const void* p, size_t a) { return (reinterpret_cast<uintptr_t>(p) % a) == 0; }

bool valid_tile(int t) { return t == 8 || t == 16 || t == 32; }

gi_status check_image(const gi_image& img, const char* fn) {
    if (img.width <= 0 || img.height <= 0 || !valid_tile(img.tile))
        return set_error(GI_ERR_INVALID_ARG, "%s: bad image %dx%d tile %d (tile must be 8, 16 or 32)", fn,
                         img.width, img.height, img.tile);
    const int64_t tw = (img.width + img.tile - 1) / img.tile, th = (img.height + img.tile - 1) / img.tile;
    if (tw * th >= (int64_t(1) << 30))
        return set_error(GI_ERR_INVALID_ARG, "%s: too many tiles (%lld)", fn, (long long)(tw * th));
    return GI_OK;
}

Batch single(const gi_image& img, int32_t n) {
    Batch b{};
    const int tw = (img.width + img.tile - 1) / img.tile, th = (img.height + img.tile - 1) / img.tile;
    b.one = ImgDesc{img.width, img.height, tw, th, 0, 0, 0};
    b.many = nullptr;
    b.nimg = 1;
    b.tile = img.tile;
    b.total_tiles = tw * th;
    b.total_gauss = n;
    return b;
}

// Buffers of a fused formation + binning + render.
struct RasterBufs {
    float4* rec;
    int4* rect;
    int32_t* cnt;
    uint32_t *keys, *ids;
    int2* ranges;
    float4* rec_binned;
    uint32_t* emit;  // nullable
    int64_t *pair_off, *k_dev;
    BinWs ws;
};

size_t up256(size_t x) { return (x + 255) / 256 * 256; }
size_t raster_partial_bytes(int64_t capacity) { return up256((size_t)capacity * 32); }
size_t raster_dl_bytes(const gi_image& img) {
    return up256((size_t)single(img, 0).total_tiles * img.tile * img.tile * 12);
}

struct RasterBytes {
    size_t state, scratch, backward;
};

// Carve-up of a differentiable pass: in `state` what its backward reads, in
// `scratch` what the forward needs besides.
RasterBufs raster_layout(void* state, void* scratch, int32_t n, const gi_image& img, int64_t capacity,
                         RasterBytes& bytes) {
    RasterBufs b{};
    const int tiles = single(img, n).total_tiles;
    const size_t N = (size_t)(n > 0 ? n : 1), cap = (size_t)capacity;
    char* p = static_cast<char*>(state);
    size_t off = 0;
    auto take = [&](size_t x) -> void* {
        const size_t o = off;
        off += up256(x);
        return p ? p + o : nullptr;
    };
    b.rec_binned = static_cast<float4*>(take(cap * 32));
    b.keys = static_cast<uint32_t*>(take(cap * 4));
    b.emit = static_cast<uint32_t*>(take(cap * 4));
    b.cnt = static_cast<int32_t*>(take(N * 4));
    b.pair_off = static_cast<int64_t*>(take((N + 1) * 8));
    b.k_dev = static_cast<int64_t*>(take(8));
    bytes.state = off;
    b.ws = bin_ws_layout(scratch, n, capacity, tiles);
    p = static_cast<char*>(scratch);
    off = up256(b.ws.bytes);
    b.rec = static_cast<float4*>(take(N * 32));
    b.rect = static_cast<int4*>(take(N * 16));
    b.ids = static_cast<uint32_t*>(take(cap * 4));
    b.ranges = static_cast<int2*>(take((size_t)tiles * 8));
    bytes.scratch = off;
    bytes.backward = raster_partial_bytes(capacity) + raster_dl_bytes(img);
    return b;
}

// Formation (which also writes the counts the binning starts from) and binning.
cudaError_t enqueue_form_bin(const float* means, const float* chol, const float* color, const Batch& B,
                             int64_t capacity, const RasterBufs& b, cudaStream_t s) {
    ZeroJob zj{};
    zj.p[0] = b.ws.zero;
    zj.n32[0] = b.ws.zero_words;
    zj.p[1] = reinterpret_cast<uint32_t*>(b.ranges);
    zj.n32[1] = (int64_t)B.total_tiles * 2;
    const cudaError_t e = launch_project(params_soa(means, chol, color), B, b.rec, b.rect, b.cnt, b.ws.blk_sum, zj, s,
                                         &b.ws);
    if (e != cudaSuccess) return e;
    return launch_bin(b.rect, b.cnt, b.rec, B, capacity, b.ws, true, b.keys, b.ids, b.ranges, b.rec_binned, b.emit,
                      b.pair_off, b.k_dev, nullptr, device_status(), s);
}

cudaError_t enqueue_plain_render(const Batch& B, const RasterBufs& b, float* out, cudaStream_t s) {
    return launch_render(b.rec_binned, b.ranges, B, nullptr, out, nullptr, nullptr, nullptr, nullptr, device_status(),
                         s);
}

#define GI_REQUIRE(cond, ...)                                   \
    do {                                                        \
        if (!(cond)) return set_error(GI_ERR_INVALID_ARG, __VA_ARGS__); \
    } while (0)

}  // namespace

gi_status set_error(gi_status st, const char* fmt, ...) {
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(t_err, sizeof(t_err), fmt, ap);
    va_end(ap);
    return st;
}

gi_status set_cuda_error(cudaError_t e, const char* what) {
    snprintf(t_err, sizeof(t_err), "%s: CUDA error %d (%s)", what, (int)e, cudaGetErrorString(e));
    return GI_ERR_CUDA;
}

cudaError_t smem_optin(const void* kernel, int bytes) {
    static std::mutex mu;
    static std::map<std::pair<const void*, int>, int> done;  // (kernel, device) -> limit set
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    std::lock_guard<std::mutex> lk(mu);
    int& have = done[{kernel, dev}];
    if (have >= bytes) return cudaSuccess;
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e == cudaSuccess) have = bytes;
    return e;
}

int sm_count() {
    static std::mutex mu;
    static std::map<int, int> cached;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 152;
    std::lock_guard<std::mutex> lk(mu);
    int& v = cached[dev];
    if (v <= 0 && (cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || v <= 0)) {
        v = 0;
        return 152;
    }
    return v;
}

uint32_t* device_status() {
    static uint32_t* cache[64] = {nullptr};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return nullptr;
    if (!cache[dev]) {
        void* p = nullptr;
        if (cudaGetSymbolAddress(&p, g_dev_status) != cudaSuccess) return nullptr;
        cache[dev] = static_cast<uint32_t*>(p);
    }
    return cache[dev];
}

}  // namespace gi

using namespace gi;

extern "C" {

int32_t gi_abi_version(void) { return 8; }

const char* gi_last_error(void) { return t_err; }

const char* gi_status_string(int32_t st) {
    switch (st) {
        case GI_OK: return "GI_OK";
        case GI_ERR_INVALID_ARG: return "GI_ERR_INVALID_ARG";
        case GI_ERR_CUDA: return "GI_ERR_CUDA";
        case GI_ERR_CAPACITY: return "GI_ERR_CAPACITY";
        case GI_ERR_TIMEOUT: return "GI_ERR_TIMEOUT";
        case GI_ERR_UNSUPPORTED: return "GI_ERR_UNSUPPORTED";
        case GI_ERR_NO_MEMORY: return "GI_ERR_NO_MEMORY";
        default: return "GI_ERR_UNKNOWN";
    }
}

gi_status gi_device_errors(uint32_t* bits, int32_t clear, gi_stream stream) {
    GI_REQUIRE(bits, "gi_device_errors: bits is NULL");
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    uint32_t* st = device_status();
    if (!st) return set_error(GI_ERR_CUDA, "gi_device_errors: no device status word");
    uint32_t v = 0;
    GI_CUDA_TRY(cudaStreamSynchronize(s));
    GI_CUDA_TRY(cudaMemcpy(&v, st, sizeof(v), cudaMemcpyDeviceToHost));
    if (clear) GI_CUDA_TRY(cudaMemset(st, 0, sizeof(uint32_t)));
    *bits = v;
    return GI_OK;
}

gi_status gi_project(const float* means, const float* chol, const float* color, int32_t n, gi_image img,
                     float* rec, int32_t* rect, int32_t* cnt, gi_stream stream) {
    NvtxRange nvtx_("gi_project");
    gi_status st = check_image(img, "gi_project");
    if (st != GI_OK) return st;
    GI_REQUIRE(n >= 0, "gi_project: n < 0");
    if (n == 0) return GI_OK;
    GI_REQUIRE(means && chol && color && rec && rect && cnt, "gi_project: NULL pointer");
    GI_REQUIRE(aligned(rec, 16) && aligned(rect, 16) && aligned(means, 4) && aligned(chol, 4) &&
                   aligned(color, 4) && aligned(cnt, 4),
               "gi_project: misaligned pointer");
    const Batch B = single(img, n);
    ZeroJob zj{};
    cudaError_t e = launch_project(params_soa(means, chol, color), B, reinterpret_cast<float4*>(rec),
                                   reinterpret_cast<int4*>(rect), cnt, nullptr, zj,
                                   reinterpret_cast<cudaStream_t>(stream));
    if (e != cudaSuccess) return set_cuda_error(e, "gi_project");
    return GI_OK;
}

gi_status gi_bin_workspace_size(int32_t n, gi_image img, int64_t capacity, size_t* bytes) {
    gi_status st = check_image(img, "gi_bin_workspace_size");
    if (st != GI_OK) return st;
    GI_REQUIRE(bytes, "gi_bin_workspace_size: bytes is NULL");
    GI_REQUIRE(n >= 0 && capacity >= 1 && capacity <= kMaxCapacity,
               "gi_bin_workspace_size: bad n (%d) or capacity (%lld)", n, (long long)capacity);
    const Batch B = single(img, n);
    *bytes = bin_ws_layout(nullptr, n, capacity, B.total_tiles).bytes;
    return GI_OK;
}

gi_status gi_bin_tiles(const int32_t* rect, const int32_t* cnt, const float* rec, int32_t n, gi_image img,
                       int64_t capacity, void* ws, size_t ws_bytes, uint32_t* keys, uint32_t* ids,
                       int32_t* ranges, float* rec_binned, int64_t* pair_off, int64_t* k_dev,
                       gi_stream stream) {
    NvtxRange nvtx_("gi_bin_tiles");
    gi_status st = check_image(img, "gi_bin_tiles");
    if (st != GI_OK) return st;
    GI_REQUIRE(n >= 0, "gi_bin_tiles: n < 0");
    GI_REQUIRE(capacity >= 1 && capacity <= kMaxCapacity, "gi_bin_tiles: capacity %lld outside [1, 2^30)",
               (long long)capacity);
    GI_REQUIRE(ws && keys && ids && ranges && pair_off && k_dev && (n == 0 || (rect && cnt)),
               "gi_bin_tiles: NULL pointer");
    GI_REQUIRE(!rec_binned || rec || n == 0, "gi_bin_tiles: rec_binned needs rec");
    GI_REQUIRE(aligned(ws, 256), "gi_bin_tiles: workspace must be 256-byte aligned");
    GI_REQUIRE(aligned(ranges, 16) && aligned(keys, 4) && aligned(ids, 4) && aligned(pair_off, 8) &&
                   aligned(k_dev, 8) && (!rec || aligned(rec, 16)) && (!rec_binned || aligned(rec_binned, 16)) &&
                   (!rect || aligned(rect, 16)),
               "gi_bin_tiles: misaligned pointer");
    const Batch B = single(img, n);
    const BinWs w = bin_ws_layout(ws, n, capacity, B.total_tiles);
    GI_REQUIRE(ws_bytes >= w.bytes, "gi_bin_tiles: workspace %zu bytes < %zu needed", ws_bytes, w.bytes);
    cudaError_t e = launch_bin(reinterpret_cast<const int4*>(rect), cnt, reinterpret_cast<const float4*>(rec), B,
                               capacity, w, false, keys, ids, reinterpret_cast<int2*>(ranges),
                               reinterpret_cast<float4*>(rec_binned), nullptr, pair_off, k_dev, nullptr, device_status(),
                               reinterpret_cast<cudaStream_t>(stream));
    if (e != cudaSuccess) return set_cuda_error(e, "gi_bin_tiles");
    return GI_OK;
}

gi_status gi_render(const float* rec_binned, const int32_t* ranges, gi_image img, const float* target, float* out,
                    float* dl_dout, double* loss_sum, gi_stream stream) {
    NvtxRange nvtx_("gi_render");
    gi_status st = check_image(img, "gi_render");
    if (st != GI_OK) return st;
    GI_REQUIRE(rec_binned && ranges && out, "gi_render: NULL pointer");
    GI_REQUIRE(!dl_dout || target, "gi_render: dl_dout needs target");
    GI_REQUIRE(!loss_sum || target, "gi_render: loss_sum needs target");
    GI_REQUIRE(aligned(rec_binned, 16) && aligned(ranges, 8) && aligned(out, 4) && (!target || aligned(target, 4)) &&
                   (!dl_dout || aligned(dl_dout, 4)) && (!loss_sum || aligned(loss_sum, 8)),
               "gi_render: misaligned pointer");
    const Batch B = single(img, 0);
    cudaError_t e = launch_render(reinterpret_cast<const float4*>(rec_binned), reinterpret_cast<const int2*>(ranges),
                                  B, target, out, dl_dout, nullptr, loss_sum, nullptr, device_status(),
                                  reinterpret_cast<cudaStream_t>(stream));
    if (e != cudaSuccess) return set_cuda_error(e, "gi_render");
    return GI_OK;
}

gi_status gi_backward_workspace_size(int32_t n, gi_image img, int64_t capacity, size_t* bytes) {
    gi_status st = check_image(img, "gi_backward_workspace_size");
    if (st != GI_OK) return st;
    GI_REQUIRE(bytes, "gi_backward_workspace_size: bytes is NULL");
    GI_REQUIRE(n >= 0 && capacity >= 1 && capacity <= kMaxCapacity, "gi_backward_workspace_size: bad n or capacity");
    const Batch B = single(img, n);
    const size_t part = ((size_t)capacity * 32 + 255) / 256 * 256;
    const size_t dl = ((size_t)B.total_tiles * img.tile * img.tile * 12 + 255) / 256 * 256;
    const size_t emit = ((size_t)capacity * 4 + 255) / 256 * 256;
    *bytes = part + dl + emit;
    return GI_OK;
}

gi_status gi_render_backward(const float* rec_binned, const uint32_t* keys, const uint32_t* ids,
                             const int32_t* ranges, const int32_t* rect, const int32_t* cnt,
                             const int64_t* pair_off, const int64_t* k_dev, const float* chol, int32_t n,
                             gi_image img, int64_t capacity, const float* dl_dout, void* ws, size_t ws_bytes,
                             float* g_means, float* g_chol, float* g_color, float* g_conic, gi_stream stream) {
    NvtxRange nvtx_("gi_render_backward");
    gi_status st = check_image(img, "gi_render_backward");
    if (st != GI_OK) return st;
    GI_REQUIRE(n >= 0, "gi_render_backward: n < 0");
    GI_REQUIRE(capacity >= 1 && capacity <= kMaxCapacity, "gi_render_backward: bad capacity");
    (void)ranges;
    if (n == 0) return GI_OK;
    GI_REQUIRE(rec_binned && keys && ids && rect && cnt && pair_off && k_dev && chol && dl_dout && ws && g_means &&
                   g_chol && g_color,
               "gi_render_backward: NULL pointer");
    GI_REQUIRE(aligned(rec_binned, 16) && aligned(keys, 16) && aligned(rect, 16) && aligned(ws, 256) &&
                   aligned(pair_off, 8) && aligned(k_dev, 8),
               "gi_render_backward: misaligned pointer");
    size_t need = 0;
    gi_backward_workspace_size(n, img, capacity, &need);
    GI_REQUIRE(ws_bytes >= need, "gi_render_backward: workspace %zu bytes < %zu needed", ws_bytes, need);
    const Batch B = single(img, n);
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    const size_t part_bytes = ((size_t)capacity * 32 + 255) / 256 * 256;
    const size_t dl_bytes = ((size_t)B.total_tiles * img.tile * img.tile * 12 + 255) / 256 * 256;
    float4* partial = static_cast<float4*>(ws);
    float* dl_tiled = reinterpret_cast<float*>(static_cast<char*>(ws) + part_bytes);
    uint32_t* emit = reinterpret_cast<uint32_t*>(static_cast<char*>(ws) + part_bytes + dl_bytes);
    cudaError_t e = launch_pack_dl(dl_dout, B, dl_tiled, s);
    if (e == cudaSuccess)
        e = launch_emit_index(keys, ids, reinterpret_cast<const int4*>(rect), pair_off, B, k_dev, capacity, emit,
                              device_status(), s);
    if (e == cudaSuccess)
        e = launch_backward(reinterpret_cast<const float4*>(rec_binned), keys, emit, dl_tiled, B, k_dev, capacity,
                            partial, device_status(), s);
    if (e == cudaSuccess)
        e = launch_reduce(partial, pair_off, cnt, capacity, n, params_soa(nullptr, chol, nullptr), g_means, g_chol,
                          g_color, g_conic, nullptr, nullptr, nullptr, nullptr, nullptr, B, s);
    if (e != cudaSuccess) return set_cuda_error(e, "gi_render_backward");
    return GI_OK;
}

gi_status gi_render_pass(const float* means, const float* chol, const float* color, int32_t n, gi_image img,
                         int64_t capacity, void* ws, size_t ws_bytes, float* rec, int32_t* rect, int32_t* cnt,
                         uint32_t* keys, uint32_t* ids, int32_t* ranges, float* rec_binned, int64_t* pair_off,
                         int64_t* k_dev, float* out, gi_stream stream) {
    NvtxRange nvtx_("gi_render_pass");
    if (n <= 0) {  // nothing to form: the separate calls (and their checks of n)
        gi_status st = gi_project(means, chol, color, n, img, rec, rect, cnt, stream);
        if (st == GI_OK)
            st = gi_bin_tiles(rect, cnt, rec, n, img, capacity, ws, ws_bytes, keys, ids, ranges, rec_binned, pair_off,
                              k_dev, stream);
        return st == GI_OK ? gi_render(rec_binned, ranges, img, nullptr, out, nullptr, nullptr, stream) : st;
    }
    gi_status st = check_image(img, "gi_render_pass");
    if (st != GI_OK) return st;
    GI_REQUIRE(capacity >= 1 && capacity <= kMaxCapacity, "gi_render_pass: capacity %lld outside [1, 2^30)",
               (long long)capacity);
    GI_REQUIRE(means && chol && color && ws && rec && rect && cnt && keys && ids && ranges && rec_binned && pair_off &&
                   k_dev && out,
               "gi_render_pass: NULL pointer");
    GI_REQUIRE(aligned(ws, 256) && aligned(rec, 16) && aligned(rect, 16) && aligned(ranges, 16) &&
                   aligned(rec_binned, 16) && aligned(pair_off, 8) && aligned(k_dev, 8) && aligned(means, 4) &&
                   aligned(chol, 4) && aligned(color, 4) && aligned(cnt, 4) && aligned(keys, 4) && aligned(ids, 4) &&
                   aligned(out, 4),
               "gi_render_pass: misaligned pointer");
    const BinWs w = bin_ws_layout(ws, n, capacity, single(img, n).total_tiles);
    GI_REQUIRE(ws_bytes >= w.bytes, "gi_render_pass: workspace %zu bytes < %zu needed", ws_bytes, w.bytes);
    const RasterBufs b{reinterpret_cast<float4*>(rec), reinterpret_cast<int4*>(rect), cnt, keys, ids,
                       reinterpret_cast<int2*>(ranges), reinterpret_cast<float4*>(rec_binned), nullptr, pair_off, k_dev,
                       w};
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    cudaError_t e = enqueue_form_bin(means, chol, color, single(img, n), capacity, b, s);
    if (e == cudaSuccess) e = enqueue_plain_render(single(img, 0), b, out, s);
    if (e != cudaSuccess) return set_cuda_error(e, "gi_render_pass");
    return GI_OK;
}

gi_status gi_rasterize_split_size(int32_t n, gi_image img, int64_t capacity, size_t* state_bytes,
                                  size_t* scratch_bytes, size_t* backward_bytes) {
    gi_status st = check_image(img, "gi_rasterize_split_size");
    if (st != GI_OK) return st;
    GI_REQUIRE(state_bytes && scratch_bytes && backward_bytes, "gi_rasterize_split_size: NULL pointer");
    GI_REQUIRE(n >= 0 && capacity >= 1 && capacity <= kMaxCapacity,
               "gi_rasterize_split_size: bad n (%d) or capacity (%lld)", n, (long long)capacity);
    RasterBytes bytes{};
    raster_layout(nullptr, nullptr, n, img, capacity, bytes);
    *state_bytes = bytes.state;
    *scratch_bytes = bytes.scratch;
    *backward_bytes = bytes.backward;
    return GI_OK;
}

gi_status gi_rasterize_size(int32_t n, gi_image img, int64_t capacity, size_t* forward_bytes, size_t* backward_bytes) {
    GI_REQUIRE(forward_bytes && backward_bytes, "gi_rasterize_size: NULL pointer");
    size_t state = 0, scratch = 0, backward = 0;
    gi_status st = gi_rasterize_split_size(n, img, capacity, &state, &scratch, &backward);
    if (st != GI_OK) return st;
    *forward_bytes = state + scratch;
    *backward_bytes = backward;
    return GI_OK;
}

gi_status gi_rasterize_forward_split(const float* means, const float* chol, const float* color, int32_t n,
                                     gi_image img, int64_t capacity, void* state, size_t state_bytes, void* scratch,
                                     size_t scratch_bytes, float* out, int64_t* pairs, gi_stream stream) {
    NvtxRange nvtx_("gi_rasterize_forward");
    size_t need_state = 0, need_scratch = 0, unused = 0;
    gi_status st = gi_rasterize_split_size(n, img, capacity, &need_state, &need_scratch, &unused);
    if (st != GI_OK) return st;
    GI_REQUIRE(state && scratch && out && pairs && (n == 0 || (means && chol && color)),
               "gi_rasterize_forward: NULL pointer");
    GI_REQUIRE(aligned(state, 256) && aligned(scratch, 256) && aligned(means, 4) && aligned(chol, 4) &&
                   aligned(color, 4) && aligned(out, 4),
               "gi_rasterize_forward: misaligned pointer");
    GI_REQUIRE(state_bytes >= need_state && scratch_bytes >= need_scratch,
               "gi_rasterize_forward: state %zu or scratch %zu bytes < %zu, %zu needed", state_bytes, scratch_bytes,
               need_state, need_scratch);
    RasterBytes bytes{};
    const RasterBufs b = raster_layout(state, scratch, n, img, capacity, bytes);
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    *pairs = 0;
    if (n == 0) {
        st = gi_bin_tiles(nullptr, nullptr, nullptr, 0, img, capacity, scratch, b.ws.bytes, b.keys, b.ids,
                          reinterpret_cast<int32_t*>(b.ranges), reinterpret_cast<float*>(b.rec_binned), b.pair_off,
                          b.k_dev, stream);
        return st == GI_OK ? gi_render(reinterpret_cast<float*>(b.rec_binned), reinterpret_cast<int32_t*>(b.ranges),
                                       img, nullptr, out, nullptr, nullptr, stream)
                           : st;
    }
    PairsWait* w = pairs_wait();
    if (!w) return set_error(GI_ERR_NO_MEMORY, "gi_rasterize_forward: no pinned word or event");
    cudaError_t e = enqueue_form_bin(means, chol, color, single(img, n), capacity, b, s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(w->k, b.k_dev, sizeof(int64_t), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaEventRecord(w->ev, s);
    if (e == cudaSuccess) e = cudaEventSynchronize(w->ev);
    if (e != cudaSuccess) return set_cuda_error(e, "gi_rasterize_forward");
    *pairs = *w->k;
    // Behind the count: a list cut off at a short capacity is not worth
    // rendering (the caller repeats the pass).
    if (*pairs <= capacity) e = enqueue_plain_render(single(img, 0), b, out, s);
    return e == cudaSuccess ? GI_OK : set_cuda_error(e, "gi_rasterize_forward");
}

gi_status gi_rasterize_forward(const float* means, const float* chol, const float* color, int32_t n, gi_image img,
                               int64_t capacity, void* state, size_t state_bytes, float* out, int64_t* pairs,
                               gi_stream stream) {
    size_t need = 0, scratch = 0, unused = 0;
    gi_status st = gi_rasterize_split_size(n, img, capacity, &need, &scratch, &unused);
    if (st != GI_OK) return st;
    GI_REQUIRE(state_bytes >= need + scratch, "gi_rasterize_forward: state %zu bytes < %zu needed", state_bytes,
               need + scratch);
    return gi_rasterize_forward_split(means, chol, color, n, img, capacity, state, need,
                                      state ? static_cast<char*>(state) + need : nullptr, scratch, out, pairs, stream);
}

gi_status gi_rasterize_backward(const void* state, size_t state_bytes, const float* chol, int32_t n, gi_image img,
                                int64_t capacity, const float* dl_dout, void* ws, size_t ws_bytes, float* g_means,
                                float* g_chol, float* g_color, gi_stream stream) {
    NvtxRange nvtx_("gi_rasterize_backward");
    size_t need = 0, unused = 0, bwd = 0;
    gi_status st = gi_rasterize_split_size(n, img, capacity, &need, &unused, &bwd);
    if (st != GI_OK) return st;
    if (n == 0) return GI_OK;
    GI_REQUIRE(state && chol && dl_dout && ws && g_means && g_chol && g_color, "gi_rasterize_backward: NULL pointer");
    GI_REQUIRE(aligned(state, 256) && aligned(ws, 256), "gi_rasterize_backward: misaligned pointer");
    GI_REQUIRE(state_bytes >= need && ws_bytes >= bwd, "gi_rasterize_backward: state %zu or workspace %zu bytes < %zu, %zu",
               state_bytes, ws_bytes, need, bwd);
    RasterBytes bytes{};
    const RasterBufs b = raster_layout(const_cast<void*>(state), nullptr, n, img, capacity, bytes);
    const Batch B = single(img, n);
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    float4* partial = static_cast<float4*>(ws);
    float* dl_tiled = reinterpret_cast<float*>(static_cast<char*>(ws) + raster_partial_bytes(capacity));
    cudaError_t e = launch_pack_dl(dl_dout, B, dl_tiled, s);
    if (e == cudaSuccess)
        e = launch_backward(b.rec_binned, b.keys, b.emit, dl_tiled, B, b.k_dev, capacity, partial, device_status(), s);
    if (e == cudaSuccess)
        e = launch_reduce(partial, b.pair_off, b.cnt, capacity, n, params_soa(nullptr, chol, nullptr), g_means, g_chol,
                          g_color, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, B, s);
    if (e != cudaSuccess) return set_cuda_error(e, "gi_rasterize_backward");
    return GI_OK;
}

gi_status gi_vq_decode(const uint16_t* means16, const uint8_t* idx, const float* codebooks, int32_t n,
                       int32_t stages, int32_t cb_size, float* means, float* chol, float* color, gi_stream stream) {
    NvtxRange nvtx_("gi_vq_decode");
    GI_REQUIRE(n >= 0, "gi_vq_decode: n < 0");
    GI_REQUIRE(stages >= 1 && stages <= 8 && cb_size >= 1 && cb_size <= 256,
               "gi_vq_decode: stages must be 1..8 and cb_size 1..256");
    if (n == 0) return GI_OK;
    GI_REQUIRE(means16 && idx && codebooks && means && chol && color, "gi_vq_decode: NULL pointer");
    GI_REQUIRE(aligned(means16, 2) && aligned(codebooks, 4) && aligned(means, 4) && aligned(chol, 4) &&
                   aligned(color, 4),
               "gi_vq_decode: misaligned pointer");
    cudaError_t e = launch_vq_decode(means16, idx, codebooks, n, stages, cb_size, means, chol, color, 0,
                                     reinterpret_cast<cudaStream_t>(stream));
    if (e != cudaSuccess) return set_cuda_error(e, "gi_vq_decode");
    return GI_OK;
}

gi_status gi_codec_decode(const uint16_t* means16, const uint8_t* codes, const float* gamma_beta,
                          const uint8_t* idx, const float* codebooks, int32_t n, int32_t stages, int32_t size,
                          float* means, float* chol, float* color, gi_stream stream) {
    NvtxRange nvtx_("gi_codec_decode");
    GI_REQUIRE(n >= 0, "gi_codec_decode: n < 0");
    GI_REQUIRE(stages >= 1 && stages <= 8 && size >= 1 && size <= 256,
               "gi_codec_decode: stages must be 1..8 and size 1..256");
    GI_REQUIRE(gamma_beta, "gi_codec_decode: NULL gamma_beta");
    if (n == 0) return GI_OK;
    GI_REQUIRE(means16 && codes && idx && codebooks && means && chol && color, "gi_codec_decode: NULL pointer");
    GI_REQUIRE(aligned(means16, 2) && aligned(codes, 4) && aligned(codebooks, 4) && aligned(means, 4) &&
                   aligned(chol, 4) && aligned(color, 4),
               "gi_codec_decode: misaligned pointer");
    cudaError_t e = launch_codec_decode(means16, codes, gamma_beta, idx, codebooks, n, stages, size, means, chol,
                                        color, reinterpret_cast<cudaStream_t>(stream));
    if (e != cudaSuccess) return set_cuda_error(e, "gi_codec_decode");
    return GI_OK;
}

}  // extern "C"
