// Weight gradient of the 3x3 convolution on the tcgen05 tensor cores:
//   gw[co][ci][dy][dx] = sum over pixels p of g[p][co] * x[p + (dy-1, dx-1)][ci]
//   gb[co]             = sum over pixels p of g[p][co]
// BF16 operands, FP32 accumulation.
//
// GEMM view: K = the pixels, so that both operands are stored with K as the
// slow axis (NHWC: a pixel's channels are contiguous).  tcgen05 reads such
// "MN-major" operands directly, so TMA boxes of the tensors are the operands
// and nothing is transposed: a box row is one pixel of 32 channels (64 bytes,
// 64-byte swizzle), a core matrix is 8 consecutive pixels.
//   A (M = 128): 4 atoms of 32 input channels, each atom one pixel (64 bytes)
//     after the one before it: the taps dx = 0, 1, 2 of an input row are the
//     same bytes at row shifts 0, 1, 2 (the fourth atom is a spare shift whose
//     32 accumulator rows are not read).
//   B (N = cout padded to 32): the row of g, one atom per 32 output channels.
// A CTA owns one block of 32 input channels, one dy and one share ("split") of
// the pixel chunks of 64 pixels of a row; its 128 x N accumulator stays in TMEM
// for the whole kernel and is written once as a partial sum.  A second kernel
// adds the partials in a fixed order (the result is deterministic) and writes
// gw and gb in the natural layout.
//
// The accumulation in TMEM truncates, so a sum's error grows with the length
// of its chain of MMAs, and where the chains are cut shows in the 5th digit of
// a gradient.  The cut is part of the result: split s of S takes the chunks s,
// s + S, ... in order, S = (SM count) / ceil(9 cin / 128), and the partials are
// added in the order of s.
//
// Bound: the TMA feed (8.3 KB per chunk for 32 output channels, 4 MMAs of
// about 40 cycles), with up to 150 to 190 CTAs resident.  Pixels as the fast
// axis, the form before this one, made four warps transpose every operand
// through registers for each of the 9 taps (1.21 ms instead of 0.16 ms for
// the three gradients of a 64 -> 64 layer on 2 x 500 x 281 pixels) and left the
// tensor cores idle.
//
// Warp roles (192 threads): warps 0-3 sum g over the pixels of each stage
// (the bias gradient, on CTAs of the first input block and dy) and read TMEM at
// the end; warp 4 issues the TMA boxes; warp 5 issues the MMAs.  Every wait is
// bounded as in conv_tc.cu: on expiry the CTA records SPP_ERR_TIMEOUT, the
// other roles leave at their next wait, the issuing threads wait for their
// copies and MMAs in flight, and TMEM is freed before the kernel returns.
#include <cuda_bf16.h>

#include <algorithm>
#include <cstring>

#include "conv_src.cuh"
#include "conv_tc.cuh"
#include "spp_internal.cuh"
#include "tc_common.cuh"
#include "tma_host.cuh"

namespace spp {
namespace conv {
namespace {

constexpr int kThreads = 192;
constexpr int kPX = 64;                 // pixels per K chunk (of one row)
constexpr int kHX = kPX + 2;            // input pixels under a chunk's three dx taps
constexpr int kBlk = 32;                // channels of a block (64 bytes)
constexpr int kLanes = 3 * kBlk;        // accumulator rows that are read: dx 0, 1, 2
constexpr int kXBytes = kHX * 64;                    // one x box
constexpr int kXSlot = (kXBytes + 511) / 512 * 512;  // its slot (swizzle period)
constexpr int kGBytes = kPX * 64;                    // one g box
constexpr int kHeader = 512;
constexpr int kMaxStages = 3;
constexpr int kBiasGroups = 8;          // pixel groups of a chunk in the bias sums
// shared memory per CTA: two CTAs fit an SM where the grid exceeds the SMs
constexpr int kSmemLimit = 110 * 1024;
// the spare fourth shift of the last pixel stays inside the x slot
static_assert(kXSlot - kXBytes >= 64, "no room for the spare tap");

struct WBars {
    uint64_t full[kMaxStages];
    uint64_t empty[kMaxStages];
    uint64_t accf;
    uint64_t drain;
    uint32_t tmem_base;
    int abort;
};
static_assert(sizeof(WBars) <= kHeader, "header");

struct WKernelArgs {
    int H, W;
    int64_t nchunks;
    int nci, nco;    // 32-channel blocks of x and of g
    int n0;          // blocks of x that come from the first source
    int ns, nch;     // stages, chunks per stage
    float *partial;  // [split][nci][dy][nco * 32][96 rows]
    float *pbias;    // [split][8][nco * 32]
    int32_t *status;
};

// MN-major operand in the 64-byte swizzle (layout type 4): atoms of 32
// channels x 8 pixels; atoms along M / N are lbo bytes apart, groups of 8
// pixels 512 bytes.  The swizzle follows the absolute address (boxes start on
// its 512-byte period), so any pixel may be the first.
__device__ __forceinline__ uint64_t desc_mn64(uint32_t saddr, uint32_t lbo) {
    return static_cast<uint64_t>((saddr & 0x3FFFFu) >> 4) |
           (static_cast<uint64_t>(lbo >> 4) << 16) | (static_cast<uint64_t>(512 >> 4) << 32) |
           (1ull << 46) | (4ull << 61);
}
// both operands MN-major (bits 15 and 16)
__host__ __device__ constexpr uint32_t idesc_mn(int N) {
    return tc::idesc_bf16_f32(128, N) | (1u << 15) | (1u << 16);
}

__device__ __forceinline__ void tma_box(const CUtensorMap *map, uint32_t dst, uint64_t *bar, int c,
                                        int x, int y, int b) {
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes "
        "[%0], [%1, {%3, %4, %5, %6}], [%2];" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(tc::smem_u32(bar)), "r"(c), "r"(x), "r"(y),
        "r"(b)
        : "memory");
}

__global__ void __launch_bounds__(kThreads)
wgrad_kernel(const WKernelArgs a, const __grid_constant__ CUtensorMap xmap0,
             const __grid_constant__ CUtensorMap xmap1, const __grid_constant__ CUtensorMap gmap) {
    extern __shared__ __align__(128) unsigned char smem_raw[];
    unsigned char *base = smem_raw + ((512u - (tc::smem_u32(smem_raw) & 511u)) & 511u);
    WBars &bars = *reinterpret_cast<WBars *>(base);
    unsigned char *stages = base + kHeader;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int split = blockIdx.x, splits = gridDim.x;
    const int ci = blockIdx.y / 3, dy = blockIdx.y % 3;
    const int N = a.nco * kBlk;
    const int cw = (a.W + kPX - 1) / kPX;
    // chunks of this split, and the stages they fill
    const int mine = static_cast<int>((a.nchunks - split + splits - 1) / splits);
    const int nstages = (mine + a.nch - 1) / a.nch;
    const int chunk_bytes = kXSlot + a.nco * kGBytes, stage_bytes = a.nch * chunk_bytes;
    const bool has_bias = blockIdx.y == 0;
    const uint32_t cols = N <= 32 ? 32 : N <= 64 ? 64 : 128;

    if (tid == 0) {
        for (int s = 0; s < a.ns; ++s) {
            tc::mbar_init(&bars.full[s], 1);
            tc::mbar_init(&bars.empty[s], has_bias ? 5 : 1);
        }
        tc::mbar_init(&bars.accf, 1);
        tc::mbar_init(&bars.drain, 1);
        bars.abort = 0;
        tc::fence_mbar_init();
    }
    if (warp == 5) tc::tmem_alloc(&bars.tmem_base, cols);
    pdl_wait();
    pdl_trigger();
    tc::tc_fence_before();
    __syncthreads();
    tc::tc_fence_after();
    const uint32_t tmem = bars.tmem_base;
    volatile int *abort_flag = &bars.abort;
    auto fail = [&]() {
        *abort_flag = 1;
        set_status(a.status, SPP_ERR_TIMEOUT);
    };

    if (warp == 4) {
        // --------------------------------------------------------- TMA boxes
        if (lane == 0) {
            const CUtensorMap *xmap = ci < a.n0 ? &xmap0 : &xmap1;
            const int cx = (ci < a.n0 ? ci : ci - a.n0) * kBlk;
            int s = 0, issued = 0;
            uint32_t ph = 0;
            for (; issued < nstages; ++issued) {
                if (!tc::mbar_wait(&bars.empty[s], ph ^ 1u, abort_flag)) {
                    fail();
                    break;
                }
                const int k0 = issued * a.nch, kn = min(a.nch, mine - k0);
                uint32_t at = tc::smem_u32(stages + s * stage_bytes);
                tc::mbar_arrive_expect_tx(&bars.full[s],
                                          static_cast<uint32_t>(kn * (kXBytes + a.nco * kGBytes)));
                for (int k = 0; k < kn; ++k, at += chunk_bytes) {
                    const int64_t q = split + static_cast<int64_t>(k0 + k) * splits;
                    const int64_t by = q / cw;  // b H + y
                    const int x0 = static_cast<int>(q - by * cw) * kPX;
                    const int b = static_cast<int>(by / a.H);
                    const int y = static_cast<int>(by - static_cast<int64_t>(b) * a.H);
                    tma_box(xmap, at, &bars.full[s], cx, x0 - 1, y + dy - 1, b);
                    for (int j = 0; j < a.nco; ++j)
                        tma_box(&gmap, at + kXSlot + j * kGBytes, &bars.full[s], j * kBlk, x0, y, b);
                }
                if (++s == a.ns) {
                    s = 0;
                    ph ^= 1u;
                }
            }
            // after a wait gave up: the copies of the last stages issued have to
            // land before the CTA exits
            if (issued < nstages)
                for (int k = max(issued - a.ns, 0); k < issued; ++k)
                    (void)tc::mbar_wait(&bars.full[k % a.ns], (k / a.ns) & 1u, nullptr);
        }
        __syncwarp();
    } else if (warp == 5) {
        // -------------------------------------------------------- MMA issuer
        if (lane == 0) {
            const uint32_t idesc = idesc_mn(N);
            bool ok = true;
            int s = 0;
            uint32_t ph = 0, acc = 0;
            for (int g = 0; g < nstages; ++g) {
                if (!tc::mbar_wait(&bars.full[s], ph, abort_flag)) {
                    fail();
                    ok = false;
                    break;
                }
                tc::tc_fence_after();
                const int kn = min(a.nch, mine - g * a.nch);
                uint32_t at = tc::smem_u32(stages + s * stage_bytes);
                for (int k = 0; k < kn; ++k, at += chunk_bytes) {
                    const uint64_t ad = desc_mn64(at, 64), bd = desc_mn64(at + kXSlot, kGBytes);
#pragma unroll
                    for (int ks = 0; ks < kPX / 16; ++ks) {
                        tc::mma_bf16(tmem, ad + ((ks * 16 * 64) >> 4), bd + ((ks * 16 * 64) >> 4),
                                     idesc, acc);
                        acc = 1;
                    }
                }
                tc::mma_commit(&bars.empty[s]);
                if (++s == a.ns) {
                    s = 0;
                    ph ^= 1u;
                }
            }
            if (ok) {
                tc::mma_commit(&bars.accf);
            } else if (acc) {
                tc::mma_commit(&bars.drain);
                (void)tc::mbar_wait(&bars.drain, 0, nullptr);
            }
        }
        __syncwarp();
    } else {
        // ----------------------------- bias gradient, then the accumulator
        bool ok = true;
        if (has_bias) {
            // thread: 8 channels (16-byte piece c4 of block j) of the pixels 8 pg
            // .. 8 pg + 7 of every chunk, added one after the other
            const int c4 = lane & 3, pg = lane >> 2, j = warp;
            float bs[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) bs[e] = 0.f;
            int s = 0;
            uint32_t ph = 0;
            for (int g = 0; g < nstages; ++g) {
                if (!tc::mbar_wait(&bars.full[s], ph, abort_flag)) {
                    fail();
                    ok = false;
                    break;
                }
                if (j < a.nco) {
                    const int kn = min(a.nch, mine - g * a.nch);
                    const unsigned char *gs =
                        stages + s * stage_bytes + kXSlot + j * kGBytes + 8 * pg * 64;
                    for (int k = 0; k < kn; ++k, gs += chunk_bytes) {
                        uint4 v[8];
#pragma unroll
                        for (int p = 0; p < 8; ++p)
                            v[p] = *reinterpret_cast<const uint4 *>(gs + p * 64 +
                                                                    16 * (c4 ^ ((p >> 1) & 3)));
#pragma unroll
                        for (int p = 0; p < 8; ++p) {
                            const uint32_t *u = &v[p].x;
#pragma unroll
                            for (int h = 0; h < 4; ++h) {
                                const float2 f = unpack_bf16x2(u[h]);
                                bs[2 * h] += f.x;
                                bs[2 * h + 1] += f.y;
                            }
                        }
                    }
                }
                __syncwarp();
                if (lane == 0) tc::mbar_arrive(&bars.empty[s]);
                if (++s == a.ns) {
                    s = 0;
                    ph ^= 1u;
                }
            }
            if (j < a.nco) {
                float *pb = a.pbias + (static_cast<int64_t>(split) * kBiasGroups + pg) * N +
                            j * kBlk + 8 * c4;
#pragma unroll
                for (int e = 0; e < 8; ++e) pb[e] = bs[e];
            }
        }
        if (ok && !tc::mbar_wait(&bars.accf, 0, abort_flag)) {
            fail();
            ok = false;
        }
        if (ok && warp < 3) {  // TMEM lanes 32 dx + channel
            tc::tc_fence_after();
            const uint32_t lbase = tmem + (static_cast<uint32_t>(warp * 32) << 16);
            float *o = a.partial +
                       ((static_cast<int64_t>(split) * a.nci + ci) * 3 + dy) * N * kLanes + tid;
#pragma unroll 1
            for (int c = 0; c < N; c += 32) {
                uint32_t v[32];
                tc::tmem_ld16(lbase + c, *reinterpret_cast<uint32_t(*)[16]>(v));
                tc::tmem_ld16(lbase + c + 16, *reinterpret_cast<uint32_t(*)[16]>(v + 16));
                tc::tmem_wait_ld();
#pragma unroll
                for (int e = 0; e < 32; ++e) o[(c + e) * kLanes] = __uint_as_float(v[e]);
            }
        }
    }

    tc::tc_fence_before();
    __syncthreads();
    if (warp == 5) {
        tc::tc_fence_after();
        tc::tmem_dealloc(tmem, cols);
    }
}

// gw[co][ci][dy][dx] = sum over the splits of their partial sums, gb[co] =
// sum over the splits and their eight pixel groups, one thread per value, in
// order (the loads of 16 splits are in flight together).  Blocks of 64 threads
// spread a small layer's 9216 values over the SMs.
constexpr int kRedThreads = 64;

__global__ void __launch_bounds__(kRedThreads)
wgrad_reduce_kernel(const float *__restrict__ partial, const float *__restrict__ pbias, int splits,
                    int nci, int nco, int cin, int cout, float *__restrict__ gw,
                    float *__restrict__ gb) {
    pdl_wait();
    pdl_trigger();
    const int N = nco * kBlk;
    const int64_t nw = static_cast<int64_t>(nci) * 3 * N * kLanes;
    const int64_t at = static_cast<int64_t>(blockIdx.x) * kRedThreads + threadIdx.x;
    const bool weight = at < nw;
    const int co_b = static_cast<int>(at - nw);
    if (!weight && co_b >= N) return;
    const float *p = weight ? partial + at : pbias + co_b;
    const int64_t stride = weight ? nw : N;
    const int terms = weight ? splits : kBiasGroups * splits;
    float acc = 0.f;
    constexpr int kU = 16;
    int s = 0;
    for (; s + kU <= terms; s += kU) {
        float v[kU];
#pragma unroll
        for (int u = 0; u < kU; ++u) v[u] = p[(s + u) * stride];
#pragma unroll
        for (int u = 0; u < kU; ++u) acc += v[u];
    }
    for (; s < terms; ++s) acc += p[s * stride];
    if (weight) {
        const int row = static_cast<int>(at % kLanes);
        const int64_t r = at / kLanes;
        const int co = static_cast<int>(r % N), cd = static_cast<int>(r / N);  // ci 3 + dy
        const int ci = (cd / 3) * kBlk + row % kBlk;
        if (ci < cin && co < cout)
            gw[(static_cast<int64_t>(co) * cin + ci) * 9 + (cd % 3) * 3 + row / kBlk] = acc;
    } else if (co_b < cout && gb) {
        gb[co_b] = acc;
    }
}

// NHWC BF16 [B][H][W][C] as a 4-D tensor (channel, x, y, image), box 32
// channels x bx pixels of one row; channels beyond C and pixels outside the image
// arrive as zeros.
bool nhwc_map(CUtensorMap *map, const __nv_bfloat16 *p, int B, int H, int W, int C, int bx) {
    auto enc = tensor_map_encoder();
    if (!enc) return false;
    cuuint64_t dims[4] = {static_cast<cuuint64_t>(C), static_cast<cuuint64_t>(W),
                          static_cast<cuuint64_t>(H), static_cast<cuuint64_t>(B)};
    cuuint64_t strides[3] = {static_cast<cuuint64_t>(C) * 2, static_cast<cuuint64_t>(W) * C * 2,
                             static_cast<cuuint64_t>(H) * W * C * 2};
    cuuint32_t box[4] = {kBlk, static_cast<cuuint32_t>(bx), 1, 1};
    cuuint32_t estr[4] = {1, 1, 1, 1};
    return enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<__nv_bfloat16 *>(p), dims,
               strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B,
               CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

struct Plan {
    int nci, nco, splits, nch, ns;
    int64_t nchunks;
};

Plan plan(int B, int W, int H, int cin, int cout) {
    Plan p;
    p.nci = (cin + kBlk - 1) / kBlk;
    p.nco = (cout + kBlk - 1) / kBlk;
    p.nchunks = static_cast<int64_t>(B) * H * ((W + kPX - 1) / kPX);
    // the cut of the sums (see the top of this file)
    const int want = std::max(1, sm_count() / ((9 * ((cin + 15) / 16 * 16) + 127) / 128));
    p.splits = static_cast<int>(std::max<int64_t>(1, std::min<int64_t>(p.nchunks, want)));
    // four chunks per stage (one barrier round trip for 16 MMAs), two where g
    // is wide
    p.nch = p.nco <= 2 ? 4 : 2;
    const int stage = p.nch * (kXSlot + p.nco * kGBytes);
    p.ns = std::min(kMaxStages, (kSmemLimit - kHeader - 512) / stage);  // 512: alignment slack
    return p;
}

}  // namespace

size_t wgrad_workspace_bytes(int B, int W, int H, int cin, int cout) {
    const Plan p = plan(B, W, H, cin, cout);
    return sizeof(float) * static_cast<size_t>(p.splits) * p.nco * kBlk *
               (static_cast<size_t>(p.nci) * 3 * kLanes + kBiasGroups) +
           256;
}

int wgrad(const WgradArgs &a, float *gw, float *gb, void *ws, cudaStream_t stream) {
    if (a.cin <= 0 || a.cout <= 0 || a.c0 % 8 || a.c1 % 8 || a.cg % 8 ||
        (a.c1 && a.c0 % kBlk) || (a.cout + kBlk - 1) / kBlk > 4)
        return SPP_ERR_ARG;
    if (static_cast<int64_t>(a.B) * a.W * a.H == 0) {
        if (cudaMemsetAsync(gw, 0, sizeof(float) * 9 * static_cast<size_t>(a.cin) * a.cout,
                            stream) != cudaSuccess)
            return SPP_ERR_CUDA;
        if (gb && cudaMemsetAsync(gb, 0, sizeof(float) * a.cout, stream) != cudaSuccess)
            return SPP_ERR_CUDA;
        return SPP_OK;
    }
    const Plan p = plan(a.B, a.W, a.H, a.cin, a.cout);
    CUtensorMap xm0, xm1, gm;
    if (!nhwc_map(&xm0, a.x0, a.B, a.H, a.W, a.c0, kHX) ||
        !nhwc_map(&gm, a.g, a.B, a.H, a.W, a.cg, kPX))
        return SPP_ERR_CUDA;
    xm1 = xm0;
    if (a.c1 && !nhwc_map(&xm1, a.x1, a.B, a.H, a.W, a.c1, kHX)) return SPP_ERR_CUDA;
    WKernelArgs k;
    k.H = a.H;
    k.W = a.W;
    k.nchunks = p.nchunks;
    k.nci = p.nci;
    k.nco = p.nco;
    k.n0 = a.c1 ? a.c0 / kBlk : p.nci;
    k.ns = p.ns;
    k.nch = p.nch;
    k.partial = static_cast<float *>(ws);
    k.pbias = k.partial + static_cast<size_t>(p.splits) * p.nci * 3 * p.nco * kBlk * kLanes;
    k.status = a.status;
    const int smem = kHeader + 512 + p.ns * p.nch * (kXSlot + p.nco * kGBytes);
    static int configured_dev = -1;
    int dev = 0;
    cudaGetDevice(&dev);
    if (configured_dev != dev) {
        if (cudaFuncSetAttribute(wgrad_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 kSmemLimit) != cudaSuccess)
            return SPP_ERR_CUDA;
        configured_dev = dev;
    }
    launch_dependent(wgrad_kernel, dim3(p.splits, 3 * p.nci), dim3(kThreads), smem, stream, k, xm0,
                     xm1, gm);
    const int64_t vals = static_cast<int64_t>(p.nci) * 3 * p.nco * kBlk * kLanes + p.nco * kBlk;
    launch_dependent(wgrad_reduce_kernel,
                     dim3(static_cast<unsigned>((vals + kRedThreads - 1) / kRedThreads)),
                     dim3(kRedThreads), 0, stream, k.partial, k.pbias, p.splits, p.nci, p.nco,
                     a.cin, a.cout, gw, gb);
    count_launch(2);
    return launch_status();
}

}  // namespace conv
}  // namespace spp
