// a11: backward pass of the sampling + reconstruction path (arXiv 2602.08642):
// the joint-softmax gather pyramid (App. A), the reprojection W_t, the tone
// map (Sec. 5), the L1 loss in sRGB (Eq. loss_spatial with m = 1), the
// average-pool pyramid, the density-normalised splat with the relaxed ramp
// (Eq. stoch_rnoisy, Eq. relaxed_holdout) and the spatial softmax of the
// sampler output (Sec. 3).
//
// The reconstruction backward recomputes each pixel's softmax weights from
// its logits instead of storing the K x K tap products, and takes the
// transpose of the gathers in gather form (each source pixel sums the
// contributions of the pixels that read it, in a fixed order): its result
// is the same from run to run.  The bilinear warp's backward scatters with
// atomics (a source pixel's readers are not bounded for arbitrary motion),
// and so may differ in its last bits from run to run.
#include "recon_common.cuh"
#include "render_common.cuh"

namespace spp {
namespace {

constexpr int kBX = 32, kBY = 8, kBH = 2;
constexpr int kRX = kBX + 2 * kBH, kRY = kBY + 2 * kBH;  // consumer region 36 x 12
constexpr int kRN = kRX * kRY;                           // 432 consumers
// a thread per consumer (with 256 threads the halo's 176 consumers, 54 dependent
// loads each, were a second round)
constexpr int kBwdThreads = (kRN + 31) / 32 * 32;
constexpr int kFX = kBX / 2 + 1, kFY = kBY / 2 + 1;      // coarse cells the tile's taps read

// Shared memory of the backward of one 32 x 8 tile: per consumer pixel of
// the tile and its 2-pixel halo the normalised weights of its kernels and
// dLoss/d out; the tap values the tile's own pixels read.
template <bool UP, bool TEMP>
struct BwdSmem {
    float wd[25][kRN];
    float wu[UP ? 4 : 1][UP ? kRN : 1];
    float wt[TEMP ? 25 : 1][TEMP ? kRN : 1];
    float g[3][kRN];
    float nz[3][kRN];
    float wp[TEMP ? 3 : 1][TEMP ? kRN : 1];
    float cv[UP ? 3 : 1][UP ? kFY * kFX : 1];
};

// Taps i in [lo, hi] of a consumer at q whose clamped source, clamp(q + i -
// 2) to [0, n - 1], is p (the transpose of clamp-to-edge along one axis);
// lo > hi when there is none.
__device__ __forceinline__ void tap_range(int q, int p, int n, int &lo, int &hi) {
    if (n == 1) {
        lo = 0;
        hi = 4;
    } else if (p == 0) {
        lo = 0;
        hi = min(2 - q, 4);
    } else if (p == n - 1) {
        lo = max(n + 1 - q, 0);
        hi = 4;
    } else {
        lo = hi = p - q + 2;
        if (lo < 0 || lo > 4) hi = lo - 1;
    }
}

// Backward of one reconstruction level in gather form: every output
// gradient element has exactly one writer, which adds its consumers'
// contributions in a fixed order, so the result does not depend on
// scheduling.  A block owns a 32 x 8 tile; a thread owns one of the 36 x 12
// consumers of the tile's sources: it computes that pixel's softmax weights
// and, inside the tile, dLoss/d logits; then the tile's threads sum for their
// source pixel (and for each coarse cell under the tile) w_k g over the
// consumers and taps that read it.
//
// Bound by its shared-memory and L1 accesses (about 560 and 110 per consumer of
// the tile), not by its bytes, so a warp takes whole rows of the tile.
// Two CTAs of 448 threads per SM (the weights of one tile take 109 KB) leave 72
// registers, so the products q_k are formed twice (once for their mean, once for
// the gradients) instead of being kept.  960 x 540, cold caches: level 0 with the
// temporal term 144 -> 137 us, level 1 27 -> 20.6 us, level 2 14 -> 10.1 us
// against 256 threads per tile and two rounds of loads.
template <bool UP, bool TEMP>
__global__ void __launch_bounds__(kBwdThreads, 2)
recon_backward_kernel(const float *__restrict__ noisy, const float *__restrict__ logits, int C,
                      const float *__restrict__ coarse, const float *__restrict__ warped,
                      const uint8_t *__restrict__ mask, int Wl, int Hl,
                      const float *__restrict__ g, float *__restrict__ grad_logits,
                      float *__restrict__ grad_noisy, float *__restrict__ grad_coarse,
                      float *__restrict__ grad_warped, int Cg, long long gl_stride,
                      bool accumulate) {
    constexpr int kSpatial = 25 + (UP ? 4 : 0);
    extern __shared__ __align__(16) unsigned char bwd_smem_raw[];
    BwdSmem<UP, TEMP> &sm = *reinterpret_cast<BwdSmem<UP, TEMP> *>(bwd_smem_raw);

    const int tid = threadIdx.x;
    const int bx0 = blockIdx.x * kBX, by0 = blockIdx.y * kBY;
    const long long Nl = static_cast<long long>(Wl) * Hl;
    const int Wc = Wl >> 1, Hc = Hl >> 1;
    const long long Nc = static_cast<long long>(Wc) * Hc;
    const int cbx = bx0 >> 1, cby = by0 >> 1;  // first coarse cell under the tile
    // image blockIdx.z of a batch (which shares the mask); gl_stride: floats
    // between the images' logit gradients
    noisy += blockIdx.z * 3 * Nl;
    logits += blockIdx.z * C * Nl;
    g += blockIdx.z * 3 * Nl;
    grad_logits += blockIdx.z * gl_stride;
    if (grad_noisy) grad_noisy += blockIdx.z * 3 * Nl;
    if (UP) coarse += blockIdx.z * 3 * Nc;
    if (UP && grad_coarse) grad_coarse += blockIdx.z * 3 * Nc;
    if (TEMP) warped += blockIdx.z * 3 * Nl;
    if (TEMP && grad_warped) grad_warped += blockIdx.z * 3 * Nl;

    // this thread's consumer: cell (rx, ry) of the region, pixel (px, py).  Warps
    // 0-7 have the tile's rows (whole 128-byte lines of every plane), the others the
    // halo: rows 0-1 and 10-11, then columns 0-1 and 34-35.
    const bool tile = tid < kBX * kBY;
    int rx, ry;
    if (tile) {
        rx = kBH + tid % kBX;
        ry = kBH + tid / kBX;
    } else if (tid < kBX * kBY + 4 * kRX) {
        const int h = tid - kBX * kBY;
        rx = h % kRX;
        ry = h / kRX < 2 ? h / kRX : kRY - 4 + h / kRX;
    } else {
        const int h = min(tid, kRN - 1) - kBX * kBY - 4 * kRX;
        ry = kBH + h / 4;
        rx = (h % 4) < 2 ? (h % 4) : kBX + (h % 4);
    }
    const int cell = ry * kRX + rx;
    const int px = bx0 + rx - kBH, py = by0 + ry - kBH;
    const bool in = tid < kRN && px >= 0 && px < Wl && py >= 0 && py < Hl;
    const long long pix = in ? static_cast<long long>(py) * Wl + px : 0;

    // spatial logits into registers, temporal ones straight into this thread's
    // cells of shared memory (all of them in registers would spill)
    float w[kSpatial];
    bool use_t = false;
    if (in) {
        use_t = TEMP && !(mask && mask[pix]);
        if (TEMP && use_t) {
#pragma unroll
            for (int k = 0; k < 25; ++k) copy_async4(&sm.wt[k][cell], logits + (29 + k) * Nl + pix);
        }
#pragma unroll
        for (int k = 0; k < kSpatial; ++k) w[k] = __ldg(logits + k * Nl + pix);
    }
    // tap values of the region (clamp-to-edge)
    if (tid < kRN) {
        const long long q = static_cast<long long>(clampi(py, 0, Hl - 1)) * Wl +
                            clampi(px, 0, Wl - 1);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            sm.nz[c][cell] = __ldg(noisy + c * Nl + q);
            if (TEMP) sm.wp[c][cell] = __ldg(warped + c * Nl + q);
            sm.g[c][cell] = in ? __ldg(g + c * Nl + pix) : 0.0f;
        }
    }
    if (UP && tid < kFX * kFY) {
        const int cx = min(cbx + tid % kFX, Wc - 1), cy = min(cby + tid / kFX, Hc - 1);
        const long long q = static_cast<long long>(cy) * Wc + cx;
#pragma unroll
        for (int c = 0; c < 3; ++c) sm.cv[c][tid] = __ldg(coarse + c * Nc + q);
    }
    // the normalised weights of the consumer; a cell that is no pixel reads
    // nothing and contributes nothing
    if (TEMP) copy_async_wait();
    if (in) {
        float m = w[0];
#pragma unroll
        for (int k = 1; k < kSpatial; ++k) m = fmaxf(m, w[k]);
        if (use_t) {
#pragma unroll
            for (int k = 0; k < 25; ++k) m = fmaxf(m, sm.wt[k][cell]);
        }
        float wsum = 0.0f;
#pragma unroll
        for (int k = 0; k < kSpatial; ++k) {
            w[k] = __expf(w[k] - m);
            wsum += w[k];
        }
        if (use_t) {
#pragma unroll
            for (int k = 0; k < 25; ++k) {
                const float e = __expf(sm.wt[k][cell] - m);
                sm.wt[k][cell] = e;
                wsum += e;
            }
        }
        const float inv = 1.0f / wsum;
#pragma unroll
        for (int k = 0; k < kSpatial; ++k) w[k] *= inv;
        if (use_t) {
#pragma unroll
            for (int k = 0; k < 25; ++k) sm.wt[k][cell] *= inv;
        }
    } else {
#pragma unroll
        for (int k = 0; k < kSpatial; ++k) w[k] = 0.0f;
    }
    if (tid < kRN) {
#pragma unroll
        for (int k = 0; k < 25; ++k) sm.wd[k][cell] = w[k];
        if (UP) {
#pragma unroll
            for (int k = 0; k < 4; ++k) sm.wu[k][cell] = w[25 + k];
        }
        if (TEMP && !use_t) {
#pragma unroll
            for (int k = 0; k < 25; ++k) sm.wt[k][cell] = 0.0f;
        }
    }
    __syncthreads();

    // dLoss/d logits of the tile: dLoss/dz_k = w_k (q_k - qbar), q_k = g . v_k
    const bool inside = in && tile;
    const float g0 = sm.g[0][cell], g1 = sm.g[1][cell], g2 = sm.g[2][cell];
    const int o0 = cell - kBH * kRX - kBH;
    auto up_cell = [&](int j, int i) {
        return (min((py + j) >> 1, Hc - 1) - cby) * kFX + min((px + i) >> 1, Wc - 1) - cbx;
    };
    auto dot = [&](const auto &v, int o) { return g0 * v[0][o] + g1 * v[1][o] + g2 * v[2][o]; };
    float qbar = 0.0f;
    if (inside) {
#pragma unroll
        for (int k = 0; k < 25; ++k) qbar = fmaf(w[k], dot(sm.nz, o0 + k / 5 * kRX + k % 5), qbar);
        if (UP) {
#pragma unroll
            for (int k = 0; k < 4; ++k)
                qbar = fmaf(w[25 + k], dot(sm.cv, up_cell(k / 2, k % 2)), qbar);
        }
        if (TEMP) {
#pragma unroll
            for (int k = 0; k < 25; ++k)
                qbar = fmaf(sm.wt[k][cell], dot(sm.wp, o0 + k / 5 * kRX + k % 5), qbar);
        }
    }
    __syncthreads();  // or the compiler would keep the products, in local memory
    if (inside) {
        float *gl = grad_logits + pix;
#pragma unroll
        for (int k = 0; k < 25; ++k)
            gl[k * Nl] = w[k] * (dot(sm.nz, o0 + k / 5 * kRX + k % 5) - qbar);
        if (UP) {
#pragma unroll
            for (int k = 0; k < 4; ++k)
                gl[(25 + k) * Nl] = w[25 + k] * (dot(sm.cv, up_cell(k / 2, k % 2)) - qbar);
        }
        if (TEMP) {
#pragma unroll
            for (int k = 0; k < 25; ++k)
                gl[(29 + k) * Nl] =
                    use_t ? sm.wt[k][cell] * (dot(sm.wp, o0 + k / 5 * kRX + k % 5) - qbar) : 0.0f;
        }
        // channels without a kernel get 0
        for (int k = TEMP ? 54 : kSpatial; k < Cg; ++k) gl[k * Nl] = 0.0f;
    }

    // sources of the tile: the sum of w_k g over the taps that read them
    if (inside && (grad_noisy || (TEMP && grad_warped))) {
        float an[3] = {0.0f, 0.0f, 0.0f}, aw[3] = {0.0f, 0.0f, 0.0f};
        // CTA-uniform: every source of the tile is 2 or more pixels from the
        // border, so each consumer reads it through exactly one tap
        const bool inner = bx0 >= 2 && bx0 + kBX + 2 <= Wl && by0 >= 2 && by0 + kBY + 2 <= Hl;
        if (inner) {
#pragma unroll
            for (int dy = -2; dy <= 2; ++dy)
#pragma unroll
                for (int dx = -2; dx <= 2; ++dx) {
                    const int from = cell + dy * kRX + dx;
                    const int k = (2 - dy) * 5 + (2 - dx);
                    const float wk = sm.wd[k][from];
#pragma unroll
                    for (int c = 0; c < 3; ++c) an[c] = fmaf(wk, sm.g[c][from], an[c]);
                    if (TEMP) {
                        const float wt = sm.wt[k][from];
#pragma unroll
                        for (int c = 0; c < 3; ++c) aw[c] = fmaf(wt, sm.g[c][from], aw[c]);
                    }
                }
        } else {
            for (int dy = -2; dy <= 2; ++dy) {
                const int qy = py + dy;
                if (qy < 0 || qy >= Hl) continue;
                int jlo, jhi;
                tap_range(qy, py, Hl, jlo, jhi);
                for (int dx = -2; dx <= 2; ++dx) {
                    const int qx = px + dx;
                    if (qx < 0 || qx >= Wl) continue;
                    int ilo, ihi;
                    tap_range(qx, px, Wl, ilo, ihi);
                    const int from = cell + dy * kRX + dx;
                    for (int j = jlo; j <= jhi; ++j)
                        for (int i = ilo; i <= ihi; ++i) {
                            const float wk = sm.wd[j * 5 + i][from];
#pragma unroll
                            for (int c = 0; c < 3; ++c) an[c] = fmaf(wk, sm.g[c][from], an[c]);
                            if (TEMP) {
                                const float wt = sm.wt[j * 5 + i][from];
#pragma unroll
                                for (int c = 0; c < 3; ++c)
                                    aw[c] = fmaf(wt, sm.g[c][from], aw[c]);
                            }
                        }
                }
            }
        }
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            if (grad_noisy) {
                float *o = grad_noisy + c * Nl + pix;
                *o = accumulate ? *o + an[c] : an[c];
            }
            if (TEMP && grad_warped) {
                float *o = grad_warped + c * Nl + pix;
                *o = accumulate ? *o + aw[c] : aw[c];
            }
        }
    }
    // coarse cells under the tile: the upsampling taps of the full-resolution
    // pixels 2c - 1 .. 2c + 1 that read them
    if (UP && grad_coarse && tid < (kBX / 2) * (kBY / 2)) {
        const int cx = cbx + tid % (kBX / 2), cy = cby + tid / (kBX / 2);
        if (cx < Wc && cy < Hc) {
            float ac[3] = {0.0f, 0.0f, 0.0f};
            for (int qy = 2 * cy - 1; qy <= 2 * cy + 1; ++qy) {
                if (qy < 0 || qy >= Hl) continue;
                for (int qx = 2 * cx - 1; qx <= 2 * cx + 1; ++qx) {
                    if (qx < 0 || qx >= Wl) continue;
                    const int from = (qy - by0 + kBH) * kRX + qx - bx0 + kBH;
#pragma unroll
                    for (int j = 0; j < 2; ++j)
#pragma unroll
                        for (int i = 0; i < 2; ++i) {
                            if (min((qx + i) >> 1, Wc - 1) != cx || min((qy + j) >> 1, Hc - 1) != cy)
                                continue;
                            const float wk = sm.wu[2 * j + i][from];
#pragma unroll
                            for (int c = 0; c < 3; ++c) ac[c] = fmaf(wk, sm.g[c][from], ac[c]);
                        }
                }
            }
            const long long q = static_cast<long long>(cy) * Wc + cx;
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                float *o = grad_coarse + c * Nc + q;
                *o = accumulate ? *o + ac[c] : ac[c];
            }
        }
    }
}

// W_t backward: each pixel's bilinear weights scatter its gradient to the
// four previous-frame pixels it read.
__global__ void __launch_bounds__(256)
warp_backward_kernel(const float *__restrict__ mv, int W, int H, const float *__restrict__ g,
                     float *__restrict__ grad_prev) {
    const int gx = blockIdx.x * 64 + (threadIdx.x & 63);
    const int gy = blockIdx.y * 4 + (threadIdx.x >> 6);
    if (gx >= W || gy >= H) return;
    const long long N = static_cast<long long>(W) * H;
    const long long i = static_cast<long long>(gy) * W + gx;
    const float mx = __ldg(mv + i), my = __ldg(mv + N + i);
    const float ix = fminf(fmaxf(floorf(mx), -1048576.0f), 1048576.0f);
    const float iy = fminf(fmaxf(floorf(my), -1048576.0f), 1048576.0f);
    float fx = mx - floorf(mx), fy = my - floorf(my);
    int X0 = gx + static_cast<int>(ix), Y0 = gy + static_cast<int>(iy);
    if (X0 < 0) { X0 = 0; fx = 0.0f; } else if (X0 >= W - 1) { X0 = W - 1; fx = 0.0f; }
    if (Y0 < 0) { Y0 = 0; fy = 0.0f; } else if (Y0 >= H - 1) { Y0 = H - 1; fy = 0.0f; }
    const int X1 = X0 + 1 < W ? X0 + 1 : W - 1;
    const int Y1 = Y0 + 1 < H ? Y0 + 1 : H - 1;
    const long long r0 = static_cast<long long>(Y0) * W, r1 = static_cast<long long>(Y1) * W;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const float v = __ldg(g + c * N + i);
        if (v == 0.0f) continue;
        float *P = grad_prev + c * N;
        atomicAdd(P + r0 + X0, (1.0f - fy) * (1.0f - fx) * v);
        atomicAdd(P + r0 + X1, (1.0f - fy) * fx * v);
        atomicAdd(P + r1 + X0, fy * (1.0f - fx) * v);
        atomicAdd(P + r1 + X1, fy * fx * v);
    }
}

__device__ __forceinline__ float tau_prime(float x, float s, float h) {
    if (x < s - 1.0f) return 0.5f * expf((x + 1.0f - s) / s);
    if (x < 1.0f - h) return 0.5f;
    return 0.5f * expf(-(x + h - 1.0f) / h);
}

__device__ __forceinline__ float tau_exact(float x, float s, float h) {
    if (x < s - 1.0f) return 0.5f * s * expf((x + 1.0f - s) / s);
    if (x < 1.0f - h) return 0.5f * (1.0f + x);
    return 1.0f - 0.5f * h * expf(-(x + h - 1.0f) / h);
}

__device__ __forceinline__ float srgb_prime(float v) {
    return v <= 0.0031308f ? 12.92f : (1.055f / 2.4f) * powf(v, 1.0f / 2.4f - 1.0f);
}

// Sec. 5 backward: gh = base + d sRGB(tau(x)) / d hdr applied to grad_ldr; base
// NULL is 0, and may be gh itself (accumulation).
__global__ void __launch_bounds__(256)
tonemap_backward_kernel(const float *__restrict__ hdr, long long N, ToneArgs tm,
                        const float *__restrict__ gl, const float *base, float *gh) {
    const long long i = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (i >= N) return;
    // image blockIdx.y of a batch
    hdr += blockIdx.y * 3 * N;
    gl += blockIdx.y * 3 * N;
    if (base) base += blockIdx.y * 3 * N;
    gh += blockIdx.y * 3 * N;
    float v[3], l[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        v[c] = hdr[c * N + i];
        l[c] = logf(fmaxf(v[c], 0x1p-24f));
    }
    const float mean = (l[0] + l[1] + l[2]) * (1.0f / 3.0f);
    float gx[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const float x = tm.alpha * (mean + tm.beta * (l[c] - mean) + tm.k);
        gx[c] = gl[c * N + i] * srgb_prime(tau_exact(x, tm.s, tm.h)) * tau_prime(x, tm.s, tm.h);
    }
    const float gs = gx[0] + gx[1] + gx[2];
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        const float glog = tm.alpha * (tm.beta * gx[j] + (1.0f - tm.beta) * (1.0f / 3.0f) * gs);
        const float b = base ? base[j * N + i] : 0.0f;
        gh[j * N + i] = v[j] >= 0x1p-24f ? b + glog / v[j] : b;
    }
}

// floats between the losses of a batch's images
constexpr int kScalarStride = 4;
// elements of a loss per thread: a block sum and one atomic per 2048 elements
// (per 256, the atomics on the one sum and the block reductions made the loss of
// 8 x 256 x 256 pixels take 15 us)
constexpr int kLossItems = 8;

inline unsigned loss_blocks(int64_t n) {
    return static_cast<unsigned>((n + 256 * kLossItems - 1) / (256 * kLossItems));
}

// Mean absolute error and its gradient sign(ldr - ref) / n.
__global__ void __launch_bounds__(256)
l1_loss_kernel(const float *__restrict__ a, const float *__restrict__ b, long long n,
               float *__restrict__ loss, float *__restrict__ grad) {
    const long long i0 = static_cast<long long>(blockIdx.x) * (256 * kLossItems) + threadIdx.x;
    // image blockIdx.y of a batch
    a += blockIdx.y * n;
    b += blockIdx.y * n;
    if (grad) grad += blockIdx.y * n;
    loss += blockIdx.y * kScalarStride;
    float v = 0.0f;
    const float unit = 1.0f / static_cast<float>(n);
#pragma unroll
    for (int k = 0; k < kLossItems; ++k) {
        const long long i = i0 + 256 * k;
        if (i >= n) continue;
        const float d = a[i] - b[i];
        v += fabsf(d);
        if (grad) grad[i] = d > 0.0f ? unit : (d < 0.0f ? -unit : 0.0f);
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) v += __shfl_down_sync(0xffffffffu, v, off);
    __shared__ float part[8];
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
        float t = 0.0f;
        for (int w = 0; w < 8; ++w) t += part[w];
        atomicAdd(loss, t / static_cast<float>(n));
    }
}

// Eq. loss_combined: mean over elements of max(wt |dI - dI_ref|, ws |I - I_ref|)
// with dI = I - Wprev, dI_ref = I_ref - Wref (warped previous frames), and
// its gradient with respect to I (ties go to the spatial term).
__global__ void combined_loss_kernel(const float *__restrict__ I, const float *__restrict__ R,
                                     const float *__restrict__ P, const float *__restrict__ Q,
                                     long long n, float w, float ws,
                                     float *__restrict__ loss, float *__restrict__ grad) {
    const long long i0 = static_cast<long long>(blockIdx.x) * (256 * kLossItems) + threadIdx.x;
    // image blockIdx.y of a batch
    I += blockIdx.y * n;
    R += blockIdx.y * n;
    P += blockIdx.y * n;
    Q += blockIdx.y * n;
    if (grad) grad += blockIdx.y * n;
    loss += blockIdx.y * kScalarStride;
    float v = 0.0f;
#pragma unroll
    for (int q = 0; q < kLossItems; ++q) {
        const long long i = i0 + 256 * q;
        if (i >= n) continue;
        const float ds = I[i] - R[i];
        const float dt = (I[i] - P[i]) - (R[i] - Q[i]);
        const float s = ws * fabsf(ds), t = w * fabsf(dt);
        const bool temporal = t > s;
        v += temporal ? t : s;
        if (grad) {
            const float sg = temporal ? (dt > 0.0f ? w : (dt < 0.0f ? -w : 0.0f))
                                      : (ds > 0.0f ? ws : (ds < 0.0f ? -ws : 0.0f));
            grad[i] = sg / static_cast<float>(n);
        }
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) v += __shfl_down_sync(0xffffffffu, v, off);
    __shared__ float part[8];
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
        float t = 0.0f;
        for (int k = 0; k < 8; ++k) t += part[k];
        atomicAdd(loss, t / static_cast<float>(n));
    }
}

// Mean squared difference (for PSNR); partial sums in FP64, one atomic per block.
__global__ void sq_err_kernel(const float *__restrict__ a, const float *__restrict__ b, long long n,
                              double *__restrict__ out) {
    double v = 0.0;
    for (long long i = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x; i < n;
         i += static_cast<long long>(gridDim.x) * blockDim.x) {
        const double d = static_cast<double>(a[i]) - static_cast<double>(b[i]);
        v += d * d;
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) v += __shfl_down_sync(0xffffffffu, v, off);
    __shared__ double part[8];
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < 8; ++w) t += part[w];
        atomicAdd(out, t / static_cast<double>(n));
    }
}

// Eq. app-pyramid backward: grad_L0 += 4^-l grad_L^l at the parent cell.
struct GradLayers {
    const float *p[5];
};

__global__ void __launch_bounds__(256)
pyramid_backward_kernel(GradLayers gl, int W, int H, int L, float *__restrict__ g0) {
    const int x = blockIdx.x * 64 + (threadIdx.x & 63);
    const int y = blockIdx.y * 4 + (threadIdx.x >> 6);
    if (x >= W || y >= H) return;
    const long long N = static_cast<long long>(W) * H;
    const long long i = static_cast<long long>(y) * W + x;
    g0 += blockIdx.z * 3 * N;  // image blockIdx.z of a batch
    float a[3] = {0.0f, 0.0f, 0.0f};
#pragma unroll
    for (int l = 1; l < 5; ++l) {
        if (l >= L) break;
        const int Wl = W >> l, Hl = H >> l;
        const long long Nl = static_cast<long long>(Wl) * Hl;
        const long long q = blockIdx.z * 3 * Nl + static_cast<long long>(y >> l) * Wl + (x >> l);
        const float sc = 1.0f / static_cast<float>(1 << (2 * l));
#pragma unroll
        for (int c = 0; c < 3; ++c) a[c] = fmaf(sc, __ldg(gl.p[l] + c * Nl + q), a[c]);
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) g0[c * N + i] += a[c];
}

// Splat backward with respect to s (Eq. stoch_rnoisy, Eq. relaxed_holdout):
//   grad_s_i = sum_c g_ic (-L0_ic / s_i)
//            + [extra, linear ramp] sum_c g_ic S_i,last,c / s_i * h lam (1 - u_i) / p_i^2
__global__ void __launch_bounds__(256)
splat_backward_kernel(const int32_t *__restrict__ offsets, const int32_t *__restrict__ counts,
                      const float4 *__restrict__ rgb, const float *__restrict__ s,
                      const float *__restrict__ L0, const float *__restrict__ gL0, long long N,
                      long long capacity, const __grid_constant__ StreamKeys keys, float lam,
                      float h, int hard,
                      float *__restrict__ grad_s) {
    const long long i = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (i >= N) return;
    // image blockIdx.y of a batch
    const uint64_t key = keys.k[blockIdx.y];
    offsets += blockIdx.y * (N + SPP_BATCH_OFFSETS_PAD);
    counts += blockIdx.y * N;
    rgb += blockIdx.y * capacity;
    s += blockIdx.y * N;
    L0 += blockIdx.y * 3 * N;
    gL0 += blockIdx.y * 3 * N;
    grad_s += blockIdx.y * N;
    const float si = s[i];
    float acc = 0.0f;
#pragma unroll
    for (int c = 0; c < 3; ++c) acc -= gL0[c * N + i] * L0[c * N + i] / si;
    if (!hard) {
        const float f = floorf(si);
        const float p = si - f;
        const int n = counts[i];
        const bool extra = n > static_cast<int>(f) && p > 0.0f;
        const long long last = static_cast<long long>(offsets[i]) + n - 1;
        if (extra && last >= 0 && last < capacity) {
            const uint64_t bits = stream_bits(key, static_cast<uint64_t>(i));
            const float u = static_cast<float>(static_cast<double>(bits >> 16) * 0x1p-48);
            const float r = lam / p * (u + p - 1.0f);
            if (r > 0.0f && r < 1.0f) {
                const float dw = h * lam * (1.0f - u) / (p * p);
                const float4 S = rgb[last];
                acc += (gL0[i] * S.x + gL0[N + i] * S.y + gL0[2 * N + i] * S.z) * dw / si;
            }
        }
    }
    grad_s[i] = acc;
}

// Straight-through (estimator 1) and Gumbel-softmax (estimator 2) gradients
// of the splat with respect to s; see spp_splat_backward_estimator.
__global__ void __launch_bounds__(256)
splat_backward_est_kernel(const int32_t *__restrict__ offsets, const int32_t *__restrict__ counts,
                          const float4 *__restrict__ rgb, const float *__restrict__ s,
                          const float *__restrict__ L0, const float *__restrict__ gL0,
                          const float *__restrict__ hw, long long N, long long capacity,
                          int estimator, float lam,
                          const __grid_constant__ BatchImages images,
                          const __grid_constant__ StreamKeys render_keys,
                          float *__restrict__ grad_s) {
    const long long i = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (i >= N) return;
    // image blockIdx.y of a batch
    const float *__restrict__ clean = images.p[blockIdx.y];
    const uint64_t render_key = render_keys.k[blockIdx.y];
    offsets += blockIdx.y * (N + SPP_BATCH_OFFSETS_PAD);
    counts += blockIdx.y * N;
    rgb += blockIdx.y * capacity;
    s += blockIdx.y * N;
    L0 += blockIdx.y * 3 * N;
    gL0 += blockIdx.y * 3 * N;
    hw += blockIdx.y * N;
    grad_s += blockIdx.y * N;
    const float si = s[i];
    float acc = 0.0f;
#pragma unroll
    for (int c = 0; c < 3; ++c) acc -= gL0[c * N + i] * L0[c * N + i] / si;
    const float f = floorf(si);
    const float p = si - f;
    const int n = counts[i];
    const bool extra = n > static_cast<int>(f) && p > 0.0f;
    const long long last = static_cast<long long>(offsets[i]) + n - 1;
    float3 S = make_float3(0.f, 0.f, 0.f);
    float scale = 0.0f;
    if (estimator == 2) {
        if (extra && last >= 0 && last < capacity) {
            const float w = hw[i];
            scale = lam * w * (1.0f - w) / (p * (1.0f - p));
            const float4 v = rgb[last];
            S = make_float3(v.x, v.y, v.z);
        }
    } else if (p > 0.0f) {
        scale = 1.0f;
        if (extra && last >= 0 && last < capacity) {
            const float4 v = rgb[last];
            S = make_float3(v.x, v.y, v.z);
        } else {  // the sample of slot f, which the forward did not trace
            const float g = render_factor(render_key, static_cast<uint64_t>(i),
                                          static_cast<uint64_t>(f));
            S = make_float3(clean[i] * g, clean[N + i] * g, clean[2 * N + i] * g);
        }
    }
    if (scale != 0.0f)
        acc += (gL0[i] * S.x + gL0[N + i] * S.y + gL0[2 * N + i] * S.z) * scale / si;
    grad_s[i] = acc;
}

// The DASR surrogate (Sec. 4.1, Eq. kuz_grad): (ref - L0) / n dotted with
// the loss gradient where the pixel has n >= 1 samples, ref dotted with it
// where it has none.
__global__ void __launch_bounds__(256)
splat_backward_dasr_kernel(const int32_t *__restrict__ counts, const float *__restrict__ L0,
                           const float *__restrict__ gL0,
                           const __grid_constant__ BatchImages refs, long long N,
                           float *__restrict__ grad_s) {
    const long long i = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (i >= N) return;
    // image blockIdx.y of a batch
    const float *__restrict__ ref = refs.p[blockIdx.y];
    counts += blockIdx.y * N;
    L0 += blockIdx.y * 3 * N;
    gL0 += blockIdx.y * 3 * N;
    grad_s += blockIdx.y * N;
    const int n = counts[i];
    float acc = 0.0f;
    if (n >= 1) {
#pragma unroll
        for (int c = 0; c < 3; ++c) acc = fmaf(gL0[c * N + i], ref[c * N + i] - L0[c * N + i], acc);
        acc /= static_cast<float>(n);
    } else {
#pragma unroll
        for (int c = 0; c < 3; ++c) acc = fmaf(gL0[c * N + i], ref[c * N + i], acc);
    }
    grad_s[i] = acc;
}

// Density backward, pass 1: per block, sum d and sum d g (FP64), written to
// the block's own slot; pass 1b adds the slots in index order.  No atomics:
// the sums, and the gradient, are the same from run to run.
constexpr int kDensityMaxBlocks = 2048;
// workspace of an image: the two sums, then the blocks' slots
constexpr int kDensityWsDoubles = 32 + 2 * kDensityMaxBlocks;

__global__ void __launch_bounds__(256)
density_reduce_kernel(const float *__restrict__ d, const float *__restrict__ g, long long N,
                      double *__restrict__ partial) {
    // image blockIdx.y of a batch
    d += blockIdx.y * N;
    g += blockIdx.y * N;
    partial += blockIdx.y * kDensityWsDoubles;
    double a = 0.0, b = 0.0;
    for (long long i = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x; i < N;
         i += static_cast<long long>(gridDim.x) * blockDim.x) {
        const float di = d[i];
        a += di;
        b += static_cast<double>(di) * g[i];
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        a += __shfl_down_sync(0xffffffffu, a, off);
        b += __shfl_down_sync(0xffffffffu, b, off);
    }
    __shared__ double pa[8], pb[8];
    if ((threadIdx.x & 31) == 0) {
        pa[threadIdx.x >> 5] = a;
        pb[threadIdx.x >> 5] = b;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double ta = 0.0, tb = 0.0;
        for (int w = 0; w < 8; ++w) {
            ta += pa[w];
            tb += pb[w];
        }
        partial[2 * blockIdx.x] = ta;
        partial[2 * blockIdx.x + 1] = tb;
    }
}

__global__ void __launch_bounds__(256)
density_sum_kernel(const double *__restrict__ partial, int blocks, double K,
                   double *__restrict__ sums) {
    partial += blockIdx.y * kDensityWsDoubles;
    sums += blockIdx.y * kDensityWsDoubles;
    double a = 0.0, b = 0.0;
    for (int k = threadIdx.x; k < blocks; k += blockDim.x) {
        a += partial[2 * k];
        b += partial[2 * k + 1];
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        a += __shfl_down_sync(0xffffffffu, a, off);
        b += __shfl_down_sync(0xffffffffu, b, off);
    }
    __shared__ double pa[8], pb[8];
    if ((threadIdx.x & 31) == 0) {
        pa[threadIdx.x >> 5] = a;
        pb[threadIdx.x >> 5] = b;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double ta = 0.0, tb = 0.0;
        for (int w = 0; w < 8; ++w) {
            ta += pa[w];
            tb += pb[w];
        }
        sums[0] = K / ta;
        sums[1] = tb / ta;
    }
}

// Pass 2 (Sec. 3): dLoss/dz_j = (1 - phi) B N pi_j (g_j - sum_i pi_i g_i), the
// divisions by the sum done once (per pixel they kept the FP64 pipe busy).
__global__ void __launch_bounds__(256)
density_grad_kernel(const float *__restrict__ d, const float *__restrict__ g, long long N,
                    const double *__restrict__ sums, float *__restrict__ gz,
                    long long gz_stride) {
    const long long i = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (i >= N) return;
    // image blockIdx.y of a batch
    d += blockIdx.y * N;
    g += blockIdx.y * N;
    sums += blockIdx.y * kDensityWsDoubles;
    gz += blockIdx.y * gz_stride;
    const double scale = sums[0], dot = sums[1];
    gz[i] = static_cast<float>(scale * static_cast<double>(d[i]) *
                               (static_cast<double>(g[i]) - dot));
}

ToneArgs tone_args_bwd(const spp_tonemap *tm) {
    ToneArgs t{1.0f, 1.0f, 0.0f, 0.5f, 0.5f, 2.0f, 2.0f};
    if (tm) {
        t.alpha = tm->alpha;
        t.beta = tm->beta;
        t.k = tm->exposure;
        t.s = tm->shadow;
        t.h = tm->highlight;
    }
    t.inv_s = 1.0f / t.s;
    t.inv_h = 1.0f / t.h;
    return t;
}

template <bool UP, bool TEMP>
int launch_recon_backward(dim3 grid, cudaStream_t stream, const float *noisy,
                          const float *logits, int C, const float *coarse, const float *warped,
                          const uint8_t *mask, int Wl, int Hl, const float *g, float *grad_logits,
                          float *grad_noisy, float *grad_coarse, float *grad_warped, int Cg,
                          long long gl_stride, bool accumulate) {
    constexpr int kSmem = static_cast<int>(sizeof(BwdSmem<UP, TEMP>));
    static int configured_dev = -1;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return SPP_ERR_CUDA;
    if (configured_dev != dev) {
        if (cudaFuncSetAttribute(recon_backward_kernel<UP, TEMP>,
                                 cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem) != cudaSuccess)
            return SPP_ERR_CUDA;
        configured_dev = dev;
    }
    recon_backward_kernel<UP, TEMP><<<grid, kBwdThreads, kSmem, stream>>>(
        noisy, logits, C, coarse, warped, mask, Wl, Hl, g, grad_logits, grad_noisy, grad_coarse,
        grad_warped, Cg, gl_stride, accumulate);
    return SPP_OK;
}

// accumulate: whether the gradients of the tap sources are added to what their
// buffers hold or stored
int level_backward(int B, const float *noisy, const float *logits, int C, const float *coarse,
                   const float *warped_prev, const uint8_t *mask, int Wl, int Hl,
                   const float *grad_out, float *grad_logits, int Cg, float *grad_noisy,
                   float *grad_coarse, float *grad_warped, bool accumulate, cudaStream_t stream) {
    if (B < 0 || B > 65535 || Wl < 0 || Hl < 0 || !noisy || !logits || !grad_out || !grad_logits)
        return SPP_ERR_ARG;
    if (warped_prev && !coarse) return SPP_ERR_ARG;
    const int need = warped_prev ? 54 : 25 + (coarse ? 4 : 0);
    if (C < need || Cg < need || Cg > C) return SPP_ERR_ARG;
    if (coarse && ((Wl & 1) || (Hl & 1))) return SPP_ERR_SHAPE;
    if (!aligned16(noisy) || !aligned16(logits) || !aligned16(grad_out) ||
        !aligned16(grad_logits) || (coarse && !aligned16(coarse)) ||
        (warped_prev && !aligned16(warped_prev)) || (mask && !aligned16(mask)) ||
        (grad_noisy && !aligned16(grad_noisy)) || (grad_coarse && !aligned16(grad_coarse)) ||
        (grad_warped && !aligned16(grad_warped)))
        return SPP_ERR_ALIGN;
    const long long n = static_cast<long long>(Wl) * Hl;
    if (B == 0 || n == 0) return SPP_OK;
    if (B > 1 && (C * n) % 4) return SPP_ERR_ALIGN;
    dim3 grid((Wl + kBX - 1) / kBX, (Hl + kBY - 1) / kBY, B);
    int rc;
    if (!coarse)
        rc = launch_recon_backward<false, false>(grid, stream, noisy, logits, C, coarse,
                                                 warped_prev, mask, Wl, Hl, grad_out, grad_logits,
                                                 grad_noisy, grad_coarse, grad_warped, Cg, C * n, accumulate);
    else if (!warped_prev)
        rc = launch_recon_backward<true, false>(grid, stream, noisy, logits, C, coarse,
                                                warped_prev, mask, Wl, Hl, grad_out, grad_logits,
                                                grad_noisy, grad_coarse, grad_warped, Cg, C * n, accumulate);
    else
        rc = launch_recon_backward<true, true>(grid, stream, noisy, logits, C, coarse,
                                               warped_prev, mask, Wl, Hl, grad_out, grad_logits,
                                               grad_noisy, grad_coarse, grad_warped, Cg, C * n, accumulate);
    count_launch();
    return rc != SPP_OK ? rc : launch_status();
}

}  // namespace
}  // namespace spp

extern "C" {

int spp_reconstruct_level_backward(const float *noisy, const float *logits, int C,
                                   const float *coarse, const float *warped_prev,
                                   const uint8_t *mask, int Wl, int Hl, const float *grad_out,
                                   float *grad_logits, float *grad_noisy, float *grad_coarse,
                                   float *grad_warped, cudaStream_t stream) {
    return spp_reconstruct_level_backward_batch(1, noisy, logits, C, coarse, warped_prev, mask, Wl,
                                                Hl, grad_out, grad_logits, C, grad_noisy,
                                                grad_coarse, grad_warped, stream);
}

int spp_reconstruct_level_backward_batch(int B, const float *noisy, const float *logits, int C,
                                         const float *coarse, const float *warped_prev,
                                         const uint8_t *mask, int Wl, int Hl,
                                         const float *grad_out, float *grad_logits, int Cg,
                                         float *grad_noisy, float *grad_coarse,
                                         float *grad_warped, cudaStream_t stream) {
    return spp::level_backward(B, noisy, logits, C, coarse, warped_prev, mask, Wl, Hl, grad_out,
                               grad_logits, Cg, grad_noisy, grad_coarse, grad_warped, true, stream);
}

int spp_reconstruct_pyramid_backward(const float *const *layers, const float *const *logits,
                                     const int *channels, const float *const *hats,
                                     const float *warped_prev, const uint8_t *mask,
                                     const float *hdr, int W, int H, int L, const spp_tonemap *tm,
                                     const float *grad_hdr, const float *grad_ldr, float *grad_out,
                                     float *const *grad_layers, float *const *grad_logits,
                                     float *const *grad_hats, float *grad_warped,
                                     cudaStream_t stream) {
    using namespace spp;
    if (!layers || !logits || !channels || !hats || !grad_layers || !grad_logits || !grad_hats ||
        !hdr || !grad_out || W < 0 || H < 0)
        return SPP_ERR_ARG;
    if (L < 2 || L > 16) return SPP_ERR_SHAPE;
    if (!aligned16(hdr) || !aligned16(grad_out) || (grad_hdr && !aligned16(grad_hdr)) ||
        (grad_ldr && !aligned16(grad_ldr)))
        return SPP_ERR_ALIGN;
    const ToneArgs ta = tone_args_bwd(tm);
    if (grad_ldr && !(ta.s > 0.0f && ta.s < 1.0f && ta.h > 0.0f && ta.h < 1.0f)) return SPP_ERR_ARG;
    const long long N = static_cast<long long>(W) * H;
    const float *g = grad_out;
    if (N && grad_ldr) {
        tonemap_backward_kernel<<<static_cast<unsigned>((N + 255) / 256), 256, 0, stream>>>(
            hdr, N, ta, grad_ldr, grad_hdr, grad_out);
        count_launch();
    } else if (N && grad_hdr) {
        g = grad_hdr;
    } else if (N && cudaMemsetAsync(grad_out, 0, 3 * N * sizeof(float), stream) != cudaSuccess) {
        return SPP_ERR_CUDA;
    }
    for (int l = 0; l < L; ++l) {
        const bool up = l + 1 < L;
        const int rc = level_backward(1, layers[l], logits[l], channels[l], up ? hats[l + 1] : nullptr,
                                      l == 0 ? warped_prev : nullptr, l == 0 ? mask : nullptr, W >> l,
                                      H >> l, g, grad_logits[l], channels[l], grad_layers[l],
                                      up ? grad_hats[l + 1] : nullptr,
                                      l == 0 ? grad_warped : nullptr, false, stream);
        if (rc != SPP_OK) return rc;
        if (up) g = grad_hats[l + 1];
    }
    return launch_status();
}

int spp_warp_previous_backward(const float *mv, int W, int H, const float *grad_warped,
                               float *grad_prev, cudaStream_t stream) {
    using namespace spp;
    if (W < 0 || H < 0 || !mv || !grad_warped || !grad_prev) return SPP_ERR_ARG;
    if (!aligned16(mv) || !aligned16(grad_warped) || !aligned16(grad_prev)) return SPP_ERR_ALIGN;
    if (static_cast<long long>(W) * H == 0) return SPP_OK;
    dim3 grid((W + 63) / 64, (H + 3) / 4);
    warp_backward_kernel<<<grid, 256, 0, stream>>>(mv, W, H, grad_warped, grad_prev);
    count_launch();
    return launch_status();
}

int spp_tonemap_backward(const float *hdr, int W, int H, const spp_tonemap *tm,
                         const float *grad_ldr, float *grad_hdr, cudaStream_t stream) {
    return spp_tonemap_backward_batch(1, hdr, W, H, tm, grad_ldr, grad_hdr, stream);
}

int spp_tonemap_backward_batch(int B, const float *hdr, int W, int H, const spp_tonemap *tm,
                               const float *grad_ldr, float *grad_hdr, cudaStream_t stream) {
    using namespace spp;
    if (B < 0 || B > 65535 || W < 0 || H < 0 || !hdr || !grad_ldr || !grad_hdr) return SPP_ERR_ARG;
    if (!aligned16(hdr) || !aligned16(grad_ldr) || !aligned16(grad_hdr)) return SPP_ERR_ALIGN;
    const ToneArgs ta = tone_args_bwd(tm);
    if (!(ta.s > 0.0f && ta.s < 1.0f && ta.h > 0.0f && ta.h < 1.0f)) return SPP_ERR_ARG;
    const long long N = static_cast<long long>(W) * H;
    if (B == 0 || N == 0) return SPP_OK;
    tonemap_backward_kernel<<<dim3(static_cast<unsigned>((N + 255) / 256), B), 256, 0, stream>>>(
        hdr, N, ta, grad_ldr, grad_hdr, grad_hdr);
    count_launch();
    return launch_status();
}

int spp_l1_loss(const float *ldr, const float *ref, int64_t n, float *loss, float *grad_ldr,
                cudaStream_t stream) {
    using namespace spp;
    if (n < 0 || !ldr || !ref || !loss) return SPP_ERR_ARG;
    if (!aligned16(ldr) || !aligned16(ref) || (grad_ldr && !aligned16(grad_ldr)) || !aligned16(loss))
        return SPP_ERR_ALIGN;
    if (cudaMemsetAsync(loss, 0, sizeof(float), stream) != cudaSuccess) return SPP_ERR_CUDA;
    if (n == 0) return SPP_OK;
    l1_loss_kernel<<<loss_blocks(n), 256, 0, stream>>>(
        ldr, ref, static_cast<long long>(n), loss, grad_ldr);
    count_launch();
    return launch_status();
}

int spp_l1_loss_batch(int B, const float *ldr, const float *ref, int64_t n, float *loss,
                      float *grad_ldr, cudaStream_t stream) {
    using namespace spp;
    if (B < 0 || B > 65535 || n < 0 || !ldr || !ref || !loss) return SPP_ERR_ARG;
    if (!aligned16(ldr) || !aligned16(ref) || (grad_ldr && !aligned16(grad_ldr)) || !aligned16(loss))
        return SPP_ERR_ALIGN;
    if (B == 0) return SPP_OK;
    if (cudaMemsetAsync(loss, 0, sizeof(float) * kScalarStride * B, stream) != cudaSuccess)
        return SPP_ERR_CUDA;
    if (n == 0) return SPP_OK;
    l1_loss_kernel<<<dim3(loss_blocks(n), B), 256, 0, stream>>>(
        ldr, ref, static_cast<long long>(n), loss, grad_ldr);
    count_launch();
    return launch_status();
}

int spp_combined_loss(const float *ldr, const float *ref, const float *prev_warped,
                      const float *ref_prev_warped, int64_t n, float temporal_weight,
                      float spatial_weight, float *loss, float *grad_ldr, cudaStream_t stream) {
    using namespace spp;
    if (n < 0 || !ldr || !ref || !prev_warped || !ref_prev_warped || !loss) return SPP_ERR_ARG;
    if (!aligned16(ldr) || !aligned16(ref) || !aligned16(prev_warped) ||
        !aligned16(ref_prev_warped) || !aligned16(loss) || (grad_ldr && !aligned16(grad_ldr)))
        return SPP_ERR_ALIGN;
    if (cudaMemsetAsync(loss, 0, sizeof(float), stream) != cudaSuccess) return SPP_ERR_CUDA;
    if (n == 0) return SPP_OK;
    combined_loss_kernel<<<loss_blocks(n), 256, 0, stream>>>(
        ldr, ref, prev_warped, ref_prev_warped, static_cast<long long>(n), temporal_weight,
        spatial_weight, loss, grad_ldr);
    count_launch();
    return launch_status();
}

int spp_combined_loss_batch(int B, const float *ldr, const float *ref, const float *prev_warped,
                            const float *ref_prev_warped, int64_t n, float temporal_weight,
                            float spatial_weight, float *loss, float *grad_ldr,
                            cudaStream_t stream) {
    using namespace spp;
    if (B < 0 || B > 65535 || n < 0 || !ldr || !ref || !prev_warped || !ref_prev_warped || !loss)
        return SPP_ERR_ARG;
    if (!aligned16(ldr) || !aligned16(ref) || !aligned16(prev_warped) ||
        !aligned16(ref_prev_warped) || !aligned16(loss) || (grad_ldr && !aligned16(grad_ldr)))
        return SPP_ERR_ALIGN;
    if (B == 0) return SPP_OK;
    if (cudaMemsetAsync(loss, 0, sizeof(float) * kScalarStride * B, stream) != cudaSuccess)
        return SPP_ERR_CUDA;
    if (n == 0) return SPP_OK;
    combined_loss_kernel<<<dim3(loss_blocks(n), B), 256, 0, stream>>>(
        ldr, ref, prev_warped, ref_prev_warped, static_cast<long long>(n), temporal_weight,
        spatial_weight, loss, grad_ldr);
    count_launch();
    return launch_status();
}

int spp_mse(const float *a, const float *b, int64_t n, double *mse, cudaStream_t stream) {
    using namespace spp;
    if (n < 0 || !a || !b || !mse) return SPP_ERR_ARG;
    if (!aligned16(a) || !aligned16(b) || !aligned16(mse)) return SPP_ERR_ALIGN;
    if (cudaMemsetAsync(mse, 0, sizeof(double), stream) != cudaSuccess) return SPP_ERR_CUDA;
    if (n == 0) return SPP_OK;
    const long long blocks = std::min<long long>((n + 255) / 256, 4LL * sm_count());
    sq_err_kernel<<<static_cast<unsigned>(blocks), 256, 0, stream>>>(a, b, n, mse);
    count_launch();
    return launch_status();
}

int spp_pyramid_backward(const float *const *grad_layers, int W, int H, int L, float *grad_L0,
                         cudaStream_t stream) {
    return spp_pyramid_backward_batch(1, grad_layers, W, H, L, grad_L0, stream);
}

int spp_pyramid_backward_batch(int B, const float *const *grad_layers, int W, int H, int L,
                               float *grad_L0, cudaStream_t stream) {
    using namespace spp;
    if (B < 0 || B > 65535 || W < 0 || H < 0 || !grad_layers || !grad_L0) return SPP_ERR_ARG;
    if (L < 1 || L > 5) return SPP_ERR_SHAPE;
    if ((W % (1 << (L - 1))) != 0 || (H % (1 << (L - 1))) != 0) return SPP_ERR_SHAPE;
    GradLayers gl{};
    for (int l = 1; l < L; ++l) {
        if (!grad_layers[l]) return SPP_ERR_ARG;
        if (!aligned16(grad_layers[l])) return SPP_ERR_ALIGN;
        gl.p[l] = grad_layers[l];
    }
    if (!aligned16(grad_L0)) return SPP_ERR_ALIGN;
    if (B == 0 || static_cast<long long>(W) * H == 0 || L == 1) return SPP_OK;
    dim3 grid((W + 63) / 64, (H + 3) / 4, B);
    pyramid_backward_kernel<<<grid, 256, 0, stream>>>(gl, W, H, L, grad_L0);
    count_launch();
    return launch_status();
}

}  // extern "C"

namespace spp {
namespace {

// The splat's gradient for at most kMaxBatch images; offsets, counts, rgb, s,
// layer0 and the gradients hold the images one after the other.
int splat_backward(int B, const int32_t *offsets, const int32_t *counts, const float *rgb,
                   const float *s, const float *layer0, const float *grad_layer0, int64_t capacity,
                   int W, int H, const spp_params *p, const uint64_t *seeds, float *grad_s,
                   cudaStream_t stream) {
    if (W < 0 || H < 0 || capacity < 0 || !p || !seeds || !offsets || !counts || !s || !layer0 ||
        !grad_layer0 || !grad_s || (capacity > 0 && !rgb))
        return SPP_ERR_ARG;
    if (!aligned16(offsets) || !aligned16(counts) || (rgb && !aligned16(rgb)) || !aligned16(s) ||
        !aligned16(layer0) || !aligned16(grad_layer0) || !aligned16(grad_s))
        return SPP_ERR_ALIGN;
    const long long N = static_cast<long long>(W) * H;
    if (B == 0 || N == 0) return SPP_OK;
    const bool hard = p->holdout_mode == SPP_HOLDOUT_HARD;
    const double lam = hard ? 1.0 : p->lambda;
    const double h = 2.0 * lam / (2.0 * lam - 1.0);
    StreamKeys keys{};
    for (int b = 0; b < B; ++b) keys.k[b] = stream_key(seeds[b], p->frame);
    splat_backward_kernel<<<dim3(static_cast<unsigned>((N + 255) / 256), B), 256, 0, stream>>>(
        offsets, counts, reinterpret_cast<const float4 *>(rgb), s, layer0, grad_layer0, N, capacity,
        keys, static_cast<float>(lam), static_cast<float>(h), hard ? 1 : 0, grad_s);
    count_launch();
    return launch_status();
}

int splat_backward_estimator(int B, const int32_t *offsets, const int32_t *counts, const float *rgb,
                             const float *s, const float *layer0, const float *grad_layer0,
                             const float *holdout_w, int64_t capacity, int W, int H,
                             const spp_params *p, const uint64_t *seeds, int estimator,
                             const float *const *clean, const uint64_t *render_seeds, float *grad_s,
                             cudaStream_t stream) {
    if (estimator == SPP_ESTIMATOR_RELAXED)
        return splat_backward(B, offsets, counts, rgb, s, layer0, grad_layer0, capacity, W, H, p,
                              seeds, grad_s, stream);
    BatchImages images{};
    bool all_clean = clean != nullptr, clean_aligned = true;
    for (int b = 0; all_clean && b < B; ++b) {
        images.p[b] = clean[b];
        clean_aligned = clean_aligned && aligned16(clean[b]);
        all_clean = clean[b] != nullptr;
    }
    const long long N = static_cast<long long>(W) * H;
    const dim3 grid(static_cast<unsigned>((N + 255) / 256), B);
    if (estimator == SPP_ESTIMATOR_DASR) {
        if (W < 0 || H < 0 || !counts || !layer0 || !grad_layer0 || !all_clean || !grad_s)
            return SPP_ERR_ARG;
        if (!aligned16(counts) || !aligned16(layer0) || !aligned16(grad_layer0) ||
            !clean_aligned || !aligned16(grad_s))
            return SPP_ERR_ALIGN;
        if (B == 0 || N == 0) return SPP_OK;
        splat_backward_dasr_kernel<<<grid, 256, 0, stream>>>(counts, layer0, grad_layer0, images, N,
                                                             grad_s);
        count_launch();
        return launch_status();
    }
    if (estimator != SPP_ESTIMATOR_STRAIGHT_THROUGH && estimator != SPP_ESTIMATOR_GUMBEL)
        return SPP_ERR_ARG;
    if (!p || W < 0 || H < 0 || capacity < 0 || !offsets || !counts || !s || !layer0 ||
        !grad_layer0 || !grad_s || (capacity > 0 && !rgb))
        return SPP_ERR_ARG;
    if (estimator == SPP_ESTIMATOR_GUMBEL && (!holdout_w || !(p->lambda > 0.0)))
        return SPP_ERR_ARG;
    if (estimator == SPP_ESTIMATOR_STRAIGHT_THROUGH && !all_clean) return SPP_ERR_ARG;
    if (!aligned16(offsets) || !aligned16(counts) || !aligned16(s) || !aligned16(layer0) ||
        !aligned16(grad_layer0) || !aligned16(grad_s) || (rgb && !aligned16(rgb)) ||
        (holdout_w && !aligned16(holdout_w)) || !clean_aligned)
        return SPP_ERR_ALIGN;
    if (B == 0 || N == 0) return SPP_OK;
    StreamKeys keys{};
    for (int b = 0; b < B; ++b) keys.k[b] = stream_key(render_seeds[b], p->frame);
    splat_backward_est_kernel<<<grid, 256, 0, stream>>>(
        offsets, counts, reinterpret_cast<const float4 *>(rgb), s, layer0, grad_layer0, holdout_w,
        N, capacity, estimator, static_cast<float>(p->lambda), images, keys, grad_s);
    count_launch();
    return launch_status();
}

}  // namespace
}  // namespace spp

extern "C" {

int spp_splat_backward(const int32_t *offsets, const int32_t *counts, const float *rgb,
                       const float *s, const float *layer0, const float *grad_layer0,
                       int64_t capacity, int W, int H, const spp_params *p, float *grad_s,
                       cudaStream_t stream) {
    return spp::splat_backward(1, offsets, counts, rgb, s, layer0, grad_layer0, capacity, W, H, p,
                               p ? &p->seed : nullptr, grad_s, stream);
}

int spp_splat_backward_estimator(const int32_t *offsets, const int32_t *counts, const float *rgb,
                                 const float *s, const float *layer0, const float *grad_layer0,
                                 const float *holdout_w, int64_t capacity, int W, int H,
                                 const spp_params *p, int estimator, const float *clean,
                                 uint64_t render_seed, float *grad_s, cudaStream_t stream) {
    return spp::splat_backward_estimator(1, offsets, counts, rgb, s, layer0, grad_layer0, holdout_w,
                                         capacity, W, H, p, p ? &p->seed : nullptr, estimator,
                                         &clean, &render_seed, grad_s, stream);
}

int spp_splat_backward_batch(int B, const int32_t *offsets, const int32_t *counts, const float *rgb,
                             const float *s, const float *layer0, const float *grad_layer0,
                             const float *holdout_w, int64_t capacity, int W, int H,
                             const spp_params *p, const uint64_t *seeds, int estimator,
                             const float *const *clean, const uint64_t *render_seeds,
                             float *grad_s, cudaStream_t stream) {
    using namespace spp;
    if (B < 0 || W < 0 || H < 0 || capacity < 0 || !p || !seeds || !render_seeds || !offsets ||
        !counts || !rgb || !s || !layer0 || !grad_layer0 || !holdout_w || !clean || !grad_s)
        return SPP_ERR_ARG;
    const int64_t n = static_cast<int64_t>(W) * H;
    if (B > 1 && n % 4) return SPP_ERR_ALIGN;
    for (int b = 0; b < B; b += kMaxBatch) {
        const int k = B - b < kMaxBatch ? B - b : kMaxBatch;
        const int rc = splat_backward_estimator(
            k, offsets + b * (n + SPP_BATCH_OFFSETS_PAD), counts + b * n, rgb + 4 * b * capacity,
            s + b * n, layer0 + b * 3 * n, grad_layer0 + b * 3 * n, holdout_w + b * n, capacity, W,
            H, p, seeds + b, estimator, clean + b, render_seeds + b, grad_s + b * n, stream);
        if (rc != SPP_OK) return rc;
    }
    return SPP_OK;
}

size_t spp_density_backward_workspace_bytes(void) {
    return spp::kDensityWsDoubles * sizeof(double);
}

int spp_density_backward(const float *d, int64_t N, double budget, double uniform_fraction,
                         const float *grad_s, float *grad_z, void *ws, size_t ws_bytes,
                         cudaStream_t stream) {
    return spp_density_backward_batch(1, d, N, budget, uniform_fraction, grad_s, grad_z, N, ws,
                                      ws_bytes, stream);
}

int spp_density_backward_batch(int B, const float *d, int64_t N, double budget,
                               double uniform_fraction, const float *grad_s, float *grad_z,
                               int64_t grad_z_stride, void *ws, size_t ws_bytes,
                               cudaStream_t stream) {
    using namespace spp;
    if (B < 0 || B > 65535 || N < 0 || !d || !grad_s || !grad_z || !ws) return SPP_ERR_ARG;
    if (ws_bytes < B * spp_density_backward_workspace_bytes()) return SPP_ERR_WORKSPACE;
    if (!aligned16(d) || !aligned16(grad_s) || !aligned16(grad_z) || !aligned16(ws))
        return SPP_ERR_ALIGN;
    if (B == 0 || N == 0) return SPP_OK;
    double *sums = static_cast<double *>(ws);
    double *partial = sums + 32;
    long long blocks = (N + 255) / 256;
    // 16 pixels per thread: with fewer, the block reductions (FP64 adds) are
    // most of the work
    long long rblocks = (blocks + 15) / 16;
    if (rblocks > kDensityMaxBlocks) rblocks = kDensityMaxBlocks;
    density_reduce_kernel<<<dim3(static_cast<unsigned>(rblocks), B), 256, 0, stream>>>(d, grad_s, N,
                                                                                    partial);
    const double K = (1.0 - uniform_fraction) * budget * static_cast<double>(N);
    density_sum_kernel<<<dim3(1, B), 256, 0, stream>>>(partial, static_cast<int>(rblocks), K, sums);
    density_grad_kernel<<<dim3(static_cast<unsigned>(blocks), B), 256, 0, stream>>>(
        d, grad_s, N, sums, grad_z, grad_z_stride);
    count_launch(3);
    return launch_status();
}

}  // extern "C"
