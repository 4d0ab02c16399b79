// a4: renderer stand-in, and a5: normalised splat (Eq. stoch_rnoisy) with the
// average-pool pyramid (Eq. app-pyramid) of arXiv 2602.08642.
#include "render_common.cuh"
#include "spp_internal.cuh"

namespace spp {
namespace {

constexpr int kRenderThreads = 256;

// Sample t of the list: pixel i = sample_pixel[t], slot k = t - offsets[i];
// value clean_i * render_factor(key, i, k).
__global__ void __launch_bounds__(kRenderThreads)
render_kernel(const __grid_constant__ BatchImages images, const int32_t *__restrict__ offsets,
              const int32_t *__restrict__ sample_pixel, const long long *__restrict__ total,
              long long capacity, long long N, const __grid_constant__ StreamKeys keys,
              float4 *__restrict__ rgb) {
    pdl_wait();
    pdl_trigger();
    // image blockIdx.y of a batch
    const float *__restrict__ clean = images.p[blockIdx.y];
    const uint64_t key = keys.k[blockIdx.y];
    offsets += blockIdx.y * (N + SPP_BATCH_OFFSETS_PAD);
    sample_pixel += blockIdx.y * capacity;
    total += blockIdx.y * 2;
    rgb += blockIdx.y * capacity;
    long long T = *total;
    if (T > capacity) T = capacity;
    const long long stride = static_cast<long long>(gridDim.x) * blockDim.x;
    for (long long t = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x; t < T;
         t += stride) {
        const int i = sample_pixel[t];
        if (i < 0 || i >= N) continue;
        const uint64_t k = static_cast<uint64_t>(t - offsets[i]);
        const float g = render_factor(key, static_cast<uint64_t>(i), k);
        rgb[t] = make_float4(clean[i] * g, clean[N + i] * g, clean[2 * N + i] * g, 0.0f);
    }
}

constexpr int kSplatTX = 32;
constexpr int kSplatTY = 8;
constexpr int kSplatRows = 2;                    // rows per thread
constexpr int kSplatH = kSplatTY * kSplatRows;   // 16: covers one level-4 block
constexpr int kMaxLevels = 5;

struct LayerPtrs {
    float *p[kMaxLevels];
};

// One block = 32 x 16 full-resolution pixels.  Each pixel gathers its slots
// (the list is ordered by pixel), normalises by s_i, and the block reduces
// 2x2 means level by level in shared memory.
__global__ void __launch_bounds__(kSplatTX *kSplatTY)
splat_kernel(const int32_t *__restrict__ offsets, const float4 *__restrict__ rgb,
             const float *__restrict__ s, const float *__restrict__ hw, long long capacity, int W,
             int H, int L, LayerPtrs layers) {
    __shared__ float buf[2][3][kSplatH][kSplatTX + 1];
    pdl_wait();
    pdl_trigger();
    const int tx = threadIdx.x, ty = threadIdx.y;
    const int x0 = blockIdx.x * kSplatTX, y0 = blockIdx.y * kSplatH;
    const long long N = static_cast<long long>(W) * H;
    // image blockIdx.z of a batch
    offsets += blockIdx.z * (N + SPP_BATCH_OFFSETS_PAD);
    rgb += blockIdx.z * capacity;
    s += blockIdx.z * N;
    hw += blockIdx.z * N;
#pragma unroll
    for (int l = 0; l < kMaxLevels; ++l)
        layers.p[l] += blockIdx.z * 3 * (static_cast<long long>(W >> l) * (H >> l));
    // all independent per-pixel loads of both rows first, then the samples
    long long beg[kSplatRows], end[kSplatRows];
    float wl[kSplatRows], si[kSplatRows];
    bool in[kSplatRows];
#pragma unroll
    for (int r = 0; r < kSplatRows; ++r) {
        const int x = x0 + tx, y = y0 + ty + kSplatTY * r;
        in[r] = x < W && y < H;
        beg[r] = 0;
        end[r] = 0;
        wl[r] = 1.0f;
        si[r] = 1.0f;
        if (in[r]) {
            const long long i = static_cast<long long>(y) * W + x;
            beg[r] = __ldg(offsets + i);
            end[r] = __ldg(offsets + i + 1);
            wl[r] = __ldg(hw + i);
            si[r] = __ldg(s + i);
        }
    }
    float4 first[kSplatRows], last[kSplatRows];
#pragma unroll
    for (int r = 0; r < kSplatRows; ++r) {
        if (beg[r] < 0) beg[r] = 0;
        if (end[r] > capacity) end[r] = capacity;
        first[r] = make_float4(0.f, 0.f, 0.f, 0.f);
        last[r] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (end[r] > beg[r]) {
            last[r] = __ldcs(rgb + end[r] - 1);                       // the holdout slot
            if (end[r] - beg[r] >= 2) first[r] = __ldcs(rgb + beg[r]);  // the first regular slot
        }
    }
#pragma unroll
    for (int r = 0; r < kSplatRows; ++r) {
        const int ly = ty + kSplatTY * r;
        float a0 = 0.0f, a1 = 0.0f, a2 = 0.0f;
        if (in[r]) {
            const long long i = static_cast<long long>(y0 + ly) * W + x0 + tx;
            if (end[r] > beg[r]) {
                a0 = first[r].x;
                a1 = first[r].y;
                a2 = first[r].z;
                for (long long t = beg[r] + 1; t < end[r] - 1; ++t) {  // slots beyond two
                    const float4 v = __ldcs(rgb + t);
                    a0 += v.x;
                    a1 += v.y;
                    a2 += v.z;
                }
                a0 = __fmaf_rn(wl[r], last[r].x, a0);
                a1 = __fmaf_rn(wl[r], last[r].y, a1);
                a2 = __fmaf_rn(wl[r], last[r].z, a2);
                a0 = __fdiv_rn(a0, si[r]);
                a1 = __fdiv_rn(a1, si[r]);
                a2 = __fdiv_rn(a2, si[r]);
            }
            float *L0 = layers.p[0];
            __stcs(L0 + i, a0);
            __stcs(L0 + N + i, a1);
            __stcs(L0 + 2 * N + i, a2);
        }
        buf[0][0][ly][tx] = a0;
        buf[0][1][ly][tx] = a1;
        buf[0][2][ly][tx] = a2;
    }
    __syncthreads();
    const int tid = ty * kSplatTX + tx;
#pragma unroll
    for (int l = 1; l < kMaxLevels; ++l) {
        if (l >= L) break;
        const int src = (l - 1) & 1, dst = l & 1;
        const int bw = kSplatTX >> l, bh = kSplatH >> l;
        const int Wl = W >> l, Hl = H >> l;
        const long long Nl = static_cast<long long>(Wl) * Hl;
        if (tid < bw * bh) {
            const int cx = tid % bw, cy = tid / bw;
            const int gx = (x0 >> l) + cx, gy = (y0 >> l) + cy;
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const float v = 0.25f * ((buf[src][c][2 * cy][2 * cx] + buf[src][c][2 * cy][2 * cx + 1]) +
                                         (buf[src][c][2 * cy + 1][2 * cx] +
                                          buf[src][c][2 * cy + 1][2 * cx + 1]));
                buf[dst][c][cy][cx] = v;
                if (gx < Wl && gy < Hl) layers.p[l][c * Nl + static_cast<long long>(gy) * Wl + gx] = v;
            }
        }
        __syncthreads();
    }
}

constexpr int kQuadTX = 128;  // 32 lanes x 4 pixels
constexpr int kQuadTY = 16;   // 8 warps x 2 rows: covers one level-4 block

// The same for widths that are a multiple of 4: a thread owns 4 x 2 pixels, reads
// offsets, weights and s in 16-byte pieces and forms its two level-1 pixels in
// registers, so that only the levels below pass through shared memory.  Same sums
// in the same order.
//
// Bound by latency (offsets, then samples, then divisions), with 32 bytes per pixel
// to move: eight pixels per thread keep four times the loads in flight that two
// did, in a quarter of the instructions.  1920 x 1080: 23.0 -> 17.9 us, the 4K frame
// 739 -> 715 us.  (The same over arrays of a templated length took 90 registers for
// 78, and the frame 738 us.)
__global__ void __launch_bounds__(256)
splat_quad_kernel(const int32_t *__restrict__ offsets, const float4 *__restrict__ rgb,
                  const float *__restrict__ s, const float *__restrict__ hw, long long capacity,
                  int W, int H, int L, LayerPtrs layers) {
    __shared__ float lvl1[3][kQuadTY / 2][kQuadTX / 2 + 1];
    __shared__ float lvl2[3][kQuadTY / 4][kQuadTX / 4 + 1];
    pdl_wait();
    pdl_trigger();
    const int tid = threadIdx.x, lane = tid & 31, pair = tid >> 5;
    const int x0 = blockIdx.x * kQuadTX, y0 = blockIdx.y * kQuadTY;
    const int x = x0 + 4 * lane;
    const long long N = static_cast<long long>(W) * H;
    // image blockIdx.z of a batch
    offsets += blockIdx.z * (N + SPP_BATCH_OFFSETS_PAD);
    rgb += blockIdx.z * capacity;
    s += blockIdx.z * N;
    hw += blockIdx.z * N;
    float *L0 = layers.p[0] + blockIdx.z * 3 * N;

    // the loads of both rows first; W is a multiple of 4, so four pixels are inside
    // or none
    int o[2][5];
    float4 w[2], sv[2];
    bool in[2];
#pragma unroll
    for (int r = 0; r < 2; ++r) {
        const int y = y0 + 2 * pair + r;
        in[r] = x < W && y < H;
        int4 q = make_int4(0, 0, 0, 0);
        o[r][4] = 0;
        w[r] = sv[r] = make_float4(1.0f, 1.0f, 1.0f, 1.0f);
        if (in[r]) {
            const long long i = static_cast<long long>(y) * W + x;
            q = __ldg(reinterpret_cast<const int4 *>(offsets + i));
            o[r][4] = __ldg(offsets + i + 4);
            w[r] = __ldg(reinterpret_cast<const float4 *>(hw + i));
            sv[r] = __ldg(reinterpret_cast<const float4 *>(s + i));
        }
        o[r][0] = q.x;
        o[r][1] = q.y;
        o[r][2] = q.z;
        o[r][3] = q.w;
    }
    float a[2][3][4];
#pragma unroll
    for (int r = 0; r < 2; ++r) {
        const float wq[4] = {w[r].x, w[r].y, w[r].z, w[r].w};
        const float sq[4] = {sv[r].x, sv[r].y, sv[r].z, sv[r].w};
        float4 first[4], last[4];
        int beg[4], end[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            beg[q] = max(o[r][q], 0);
            end[q] = o[r][q + 1] > capacity ? static_cast<int>(capacity) : o[r][q + 1];
            first[q] = last[q] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (end[q] > beg[q]) {
                last[q] = __ldcs(rgb + end[q] - 1);                         // the holdout slot
                if (end[q] - beg[q] >= 2) first[q] = __ldcs(rgb + beg[q]);  // the first regular one
            }
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            float a0 = 0.0f, a1 = 0.0f, a2 = 0.0f;
            if (end[q] > beg[q]) {
                a0 = first[q].x;
                a1 = first[q].y;
                a2 = first[q].z;
                for (int t = beg[q] + 1; t < end[q] - 1; ++t) {  // slots beyond two
                    const float4 v = __ldcs(rgb + t);
                    a0 += v.x;
                    a1 += v.y;
                    a2 += v.z;
                }
                a0 = __fdiv_rn(__fmaf_rn(wq[q], last[q].x, a0), sq[q]);
                a1 = __fdiv_rn(__fmaf_rn(wq[q], last[q].y, a1), sq[q]);
                a2 = __fdiv_rn(__fmaf_rn(wq[q], last[q].z, a2), sq[q]);
            }
            a[r][0][q] = a0;
            a[r][1][q] = a1;
            a[r][2][q] = a2;
        }
        if (in[r]) {
            const long long i = static_cast<long long>(y0 + 2 * pair + r) * W + x;
#pragma unroll
            for (int c = 0; c < 3; ++c)
                __stcs(reinterpret_cast<float4 *>(L0 + c * N + i),
                       make_float4(a[r][c][0], a[r][c][1], a[r][c][2], a[r][c][3]));
        }
    }
    if (L < 2) return;
    {
        const int W1 = W >> 1, H1 = H >> 1;
        const long long N1 = static_cast<long long>(W1) * H1;
        const int gx = x >> 1, gy = (y0 >> 1) + pair;
        float *L1 = layers.p[1] + blockIdx.z * 3 * N1 + static_cast<long long>(gy) * W1 + gx;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            float2 v;
            v.x = 0.25f * ((a[0][c][0] + a[0][c][1]) + (a[1][c][0] + a[1][c][1]));
            v.y = 0.25f * ((a[0][c][2] + a[0][c][3]) + (a[1][c][2] + a[1][c][3]));
            lvl1[c][pair][2 * lane] = v.x;
            lvl1[c][pair][2 * lane + 1] = v.y;
            if (gx < W1 && gy < H1) *reinterpret_cast<float2 *>(L1 + c * N1) = v;
        }
    }
    // levels 2 to 4: from lvl1 into lvl2, back, and once more
    auto reduce = [&](int l, auto &src, auto &dst) {
        const int bw = kQuadTX >> l, bh = kQuadTY >> l;
        const int Wl = W >> l, Hl = H >> l;
        const long long Nl = static_cast<long long>(Wl) * Hl;
        __syncthreads();
        if (tid < bw * bh) {
            const int cx = tid % bw, cy = tid / bw;
            const int gx = (x0 >> l) + cx, gy = (y0 >> l) + cy;
            float *out = layers.p[l] + blockIdx.z * 3 * Nl;
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const float v = 0.25f * ((src[c][2 * cy][2 * cx] + src[c][2 * cy][2 * cx + 1]) +
                                         (src[c][2 * cy + 1][2 * cx] + src[c][2 * cy + 1][2 * cx + 1]));
                dst[c][cy][cx] = v;
                if (gx < Wl && gy < Hl) out[c * Nl + static_cast<long long>(gy) * Wl + gx] = v;
            }
        }
    };
    if (L > 2) reduce(2, lvl1, lvl2);
    if (L > 3) reduce(3, lvl2, lvl1);
    if (L > 4) reduce(4, lvl1, lvl2);
}

}  // namespace
}  // namespace spp

namespace spp {
namespace {

int render(int B, const float *const *clean, const int32_t *offsets, const int32_t *sample_pixel,
           const int64_t *total, int64_t capacity, int W, int H, const uint64_t *seeds,
           uint32_t frame, float *rgb, cudaStream_t stream) {
    if (B < 0 || B > kMaxBatch || W < 0 || H < 0 || capacity < 0) return SPP_ERR_ARG;
    if (!clean || !offsets || !total || !seeds) return SPP_ERR_ARG;
    if (capacity > 0 && (!sample_pixel || !rgb)) return SPP_ERR_ARG;
    BatchImages images{};
    StreamKeys keys{};
    for (int b = 0; b < B; ++b) {
        if (!clean[b]) return SPP_ERR_ARG;
        if (!aligned16(clean[b])) return SPP_ERR_ALIGN;
        images.p[b] = clean[b];
        keys.k[b] = stream_key(seeds[b], frame);
    }
    if (!aligned16(offsets) || !aligned16(total) || (rgb && !aligned16(rgb)) ||
        (sample_pixel && !aligned16(sample_pixel)))
        return SPP_ERR_ALIGN;
    const long long N = static_cast<long long>(W) * H;
    if (B == 0 || N == 0 || capacity == 0) return SPP_OK;
    long long grid = (capacity + kRenderThreads - 1) / kRenderThreads;
    const long long max_grid = static_cast<long long>(sm_count()) * 8;
    if (grid > max_grid) grid = max_grid;
    launch_dependent(render_kernel, dim3(static_cast<unsigned>(grid), B), dim3(kRenderThreads), 0,
                     stream, images, offsets, sample_pixel,
                     reinterpret_cast<const long long *>(total), capacity, N, keys,
                     reinterpret_cast<float4 *>(rgb));
    count_launch();
    return launch_status();
}

int splat(int B, const int32_t *offsets, const float *rgb, const float *s, const float *holdout_w,
          int64_t capacity, int W, int H, int L, float *const *layers, cudaStream_t stream) {
    if (B < 0 || W < 0 || H < 0 || capacity < 0 || !layers) return SPP_ERR_ARG;
    if (L < 1 || L > kMaxLevels) return SPP_ERR_SHAPE;
    if ((W % (1 << (L - 1))) != 0 || (H % (1 << (L - 1))) != 0) return SPP_ERR_SHAPE;
    if (!offsets || !s || !holdout_w || (capacity > 0 && !rgb)) return SPP_ERR_ARG;
    LayerPtrs lp{};
    for (int l = 0; l < L; ++l) {
        if (!layers[l]) return SPP_ERR_ARG;
        if (!aligned16(layers[l])) return SPP_ERR_ALIGN;
        lp.p[l] = layers[l];
    }
    if (!aligned16(offsets) || !aligned16(s) || !aligned16(holdout_w) || (rgb && !aligned16(rgb)))
        return SPP_ERR_ALIGN;
    if (B == 0 || static_cast<long long>(W) * H == 0) return SPP_OK;
    if (W % 4 == 0) {  // 16-byte pieces of a row
        dim3 grid((W + kQuadTX - 1) / kQuadTX, (H + kQuadTY - 1) / kQuadTY, B);
        launch_dependent(splat_quad_kernel, grid, dim3(256), 0, stream, offsets,
                         reinterpret_cast<const float4 *>(rgb), s, holdout_w, capacity, W, H, L, lp);
        count_launch();
        return launch_status();
    }
    dim3 block(kSplatTX, kSplatTY);
    dim3 grid((W + kSplatTX - 1) / kSplatTX, (H + kSplatH - 1) / kSplatH, B);
    launch_dependent(splat_kernel, grid, block, 0, stream, offsets,
                     reinterpret_cast<const float4 *>(rgb), s, holdout_w, capacity, W, H, L, lp);
    count_launch();
    return launch_status();
}

}  // namespace
}  // namespace spp

extern "C" {

int spp_render_synthetic(const float *clean, const int32_t *offsets, const int32_t *sample_pixel,
                         const int64_t *total, int64_t capacity, int W, int H, uint64_t seed,
                         uint32_t frame, float *rgb, cudaStream_t stream) {
    return spp::render(1, &clean, offsets, sample_pixel, total, capacity, W, H, &seed, frame, rgb,
                       stream);
}

int spp_render_synthetic_batch(int B, const float *const *clean, const int32_t *offsets,
                               const int32_t *sample_pixel, const int64_t *total, int64_t capacity,
                               int W, int H, const uint64_t *seeds, uint32_t frame, float *rgb,
                               cudaStream_t stream) {
    using namespace spp;
    if (B < 0 || W < 0 || H < 0 || capacity < 0 || !clean || !offsets || !sample_pixel || !total ||
        !seeds || !rgb)
        return SPP_ERR_ARG;
    const int64_t n = static_cast<int64_t>(W) * H;
    if (B > 1 && n % 4) return SPP_ERR_ALIGN;
    for (int b = 0; b < B; b += kMaxBatch) {
        const int k = B - b < kMaxBatch ? B - b : kMaxBatch;
        const int rc = render(k, clean + b, offsets + b * (n + SPP_BATCH_OFFSETS_PAD),
                              sample_pixel + b * capacity, total + 2 * b, capacity, W, H, seeds + b,
                              frame, rgb + 4 * b * capacity, stream);
        if (rc != SPP_OK) return rc;
    }
    return SPP_OK;
}

int spp_splat_samples(const int32_t *offsets, const float *rgb, const float *s,
                      const float *holdout_w, int64_t capacity, int W, int H, int L,
                      float *const *layers, cudaStream_t stream) {
    return spp::splat(1, offsets, rgb, s, holdout_w, capacity, W, H, L, layers, stream);
}

int spp_splat_samples_batch(int B, const int32_t *offsets, const float *rgb, const float *s,
                            const float *holdout_w, int64_t capacity, int W, int H, int L,
                            float *const *layers, cudaStream_t stream) {
    return spp::splat(B, offsets, rgb, s, holdout_w, capacity, W, H, L, layers, stream);
}

}  // extern "C"
