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
// Past the end of a row g is 0, but the dx = 0 rows still hold the row's last pixel
// there, and an infinity times 0 is NaN.  So a row's last chunk stops at its last
// pixel, and where that is inside a K step of 16 (W % 16 != 0) the step is two MMAs:
// one that leaves out the dx = 0 lanes, one for them alone with the 8 pixels around
// the edge from a box of the tensor without its last column (kEdgeBytes).
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
// through registers for each of the 9 taps (1.21 ms instead of 0.14 ms for
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
constexpr int kEdgeBytes = 8 * 64;                   // 8 pixels at the edge of a row
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
    int nchunks;     // B H ceil(W / 64)
    int nci, nco;    // 32-channel blocks of x and of g
    int n0;          // blocks of x that come from the first source
    int ns, nch;     // stages, chunks per stage
    int steps, rem;  // whole K steps of a row's last chunk, and the pixels after them
    // places in a chunk of its x box, its edge box (when rem > 0; it starts at pixel
    // edge_x of the row) and its g boxes
    int x_off, edge_off, edge_x, g_off;
    float *partial;  // [split][nci][dy][nco * 32][96 rows]
    float *pbias;    // [split][8][nco * 32]
    int32_t *status;
};

// MN-major operand in the 64-byte swizzle (layout type 4): atoms of 32
// channels x 8 pixels; atoms along M / N are lbo bytes apart, groups of 8
// pixels sbo bytes.  The swizzle follows the absolute address (boxes start on
// its 512-byte period), so any pixel may be the first.
__device__ __forceinline__ uint64_t desc_mn64(uint32_t saddr, uint32_t lbo, uint32_t sbo = 512) {
    return static_cast<uint64_t>((saddr & 0x3FFFFu) >> 4) |
           (static_cast<uint64_t>(lbo >> 4) << 16) | (static_cast<uint64_t>(sbo >> 4) << 32) |
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

// EDGE: rows that do not end with a chunk (W % 64 != 0).  Its tests in the other
// instance made the gradients of 8 x 256 x 256 take 1229 us instead of 1204.
template <bool EDGE>
__global__ void __launch_bounds__(kThreads)
wgrad_kernel(const WKernelArgs a, const __grid_constant__ CUtensorMap xmap0,
             const __grid_constant__ CUtensorMap xmap1, const __grid_constant__ CUtensorMap gmap,
             const __grid_constant__ CUtensorMap emap0, const __grid_constant__ CUtensorMap emap1) {
    // emap0, emap1: the sources without the last pixel of every row
    extern __shared__ __align__(128) unsigned char smem_raw[];
    unsigned char *base = smem_raw + ((512u - (tc::smem_u32(smem_raw) & 511u)) & 511u);
    WBars &bars = *reinterpret_cast<WBars *>(base);
    unsigned char *stages = base + kHeader;
    const int tid = threadIdx.x, lane = tid & 31;
    const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);  // known to be the warp's
    const int split = blockIdx.x, splits = gridDim.x;
    const int ci = blockIdx.y / 3, dy = blockIdx.y % 3;
    const int N = a.nco * kBlk;
    const int cw = (a.W + kPX - 1) / kPX;
    // chunks of this split, and the stages they fill
    const int mine = (a.nchunks - split + splits - 1) / splits;
    const int nstages = (mine + a.nch - 1) / a.nch;
    const int x_off = EDGE ? a.x_off : 0, g_off = EDGE ? a.g_off : kXSlot;
    const int chunk_bytes = g_off + a.nco * kGBytes, stage_bytes = a.nch * chunk_bytes;
    // a chunk's place in its row, advanced by `splits` chunks with carries (a division
    // per chunk made the copy thread the kernel's bound)
    const int dxc = splits % cw;
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
            const CUtensorMap *emap = ci < a.n0 ? &emap0 : &emap1;
            const int cx = (ci < a.n0 ? ci : ci - a.n0) * kBlk;
            const int dby = splits / cw, dyy = dby % a.H, db = dby / a.H;
            int xc = split % cw, y = (split / cw) % a.H, b = split / cw / a.H;
            int s = 0, issued = 0;
            uint32_t ph = 0;
            for (; issued < nstages; ++issued) {
                if (!tc::mbar_wait(&bars.empty[s], ph ^ 1u, abort_flag)) {
                    fail();
                    break;
                }
                const int k0 = issued * a.nch, kn = min(a.nch, mine - k0);
                uint32_t at = tc::smem_u32(stages + s * stage_bytes);
                int edges = 0;  // edge boxes of the stage
                if (EDGE && a.rem)
                    for (int k = 0, q = xc; k < kn; ++k) {
                        edges += q == cw - 1;
                        q += dxc;
                        if (q >= cw) q -= cw;
                    }
                tc::mbar_arrive_expect_tx(&bars.full[s],
                                          static_cast<uint32_t>(kn * (kXBytes + a.nco * kGBytes) +
                                                                edges * kEdgeBytes));
                for (int k = 0; k < kn; ++k, at += chunk_bytes) {
                    const int x0 = xc * kPX;
                    tma_box(xmap, at + x_off, &bars.full[s], cx, x0 - 1, y + dy - 1, b);
                    if (EDGE && a.rem && xc == cw - 1)
                        tma_box(emap, at + a.edge_off, &bars.full[s], cx, a.edge_x, y + dy - 1, b);
                    for (int j = 0; j < a.nco; ++j)
                        tma_box(&gmap, at + g_off + j * kGBytes, &bars.full[s], j * kBlk, x0, y, b);
                    xc += dxc;
                    y += dyy;
                    b += db;
                    if (xc >= cw) {
                        xc -= cw;
                        ++y;
                    }
                    if (y >= a.H) {
                        y -= a.H;
                        ++b;
                    }
                }
                if (++s == a.ns) {
                    s = 0;
                    ph ^= 1u;
                }
            }
            // the copies of the last stages issued have to land before the CTA exits,
            // also where another role gave up on them
            for (int k = max(issued - a.ns, 0); k < issued; ++k)
                (void)tc::mbar_wait(&bars.full[k % a.ns], (k / a.ns) & 1u, nullptr);
        }
        __syncwarp();
    } else if (warp == 5) {
        // -------------------------------------------------------- MMA issuer
        {
            // warp-uniform code, one lane issues: descriptors in uniform registers
            const uint32_t lead = tc::elect_one();
            const uint32_t idesc = idesc_mn(N);
            bool ok = true;
            int s = 0, xc = split % cw;
            uint32_t ph = 0, acc = 0;
            for (int g = 0; g < nstages; ++g) {
                if (!tc::mbar_wait_warp(&bars.full[s], ph, abort_flag)) {
                    fail();
                    ok = false;
                    break;
                }
                tc::tc_fence_after();
                const int kn = min(a.nch, mine - g * a.nch);
                uint32_t at = tc::smem_u32(stages + s * stage_bytes);
                for (int k = 0; k < kn; ++k, at += chunk_bytes) {
                    const uint64_t ad = desc_mn64(at + x_off, 64),
                                   bd = desc_mn64(at + g_off, kGBytes);
                    const bool last = EDGE && xc == cw - 1;
                    const int steps = last ? a.steps : kPX / 16;
#pragma unroll
                    for (int ks = 0; ks < kPX / 16; ++ks) {
                        if (EDGE && ks >= steps) break;
                        tc::mma_bf16(tmem, ad + tc::desc_offset(ks * 16 * 64),
                                     bd + tc::desc_offset(ks * 16 * 64), idesc, acc, lead);
                        acc = 1;
                    }
                    if (last && a.rem) {
                        // the step over the edge: dx = 1, 2; then dx = 0, whose group of
                        // 8 pixels with the edge is the edge box.  The other group is in
                        // its place: before the edge when rem >= 8 (then the edge box lies
                        // behind the x box), all zeros after it (then it lies before)
                        const uint32_t off = steps * 16 * 64;
                        const uint64_t bs = bd + tc::desc_offset(off);
                        tc::mma_bf16_lanes<1>(tmem, ad + tc::desc_offset(off), bs, idesc, acc, lead);
                        const uint64_t es =
                            a.rem < 8 ? desc_mn64(at + a.edge_off, 64, x_off + off + 512 - a.edge_off)
                                      : desc_mn64(at + x_off + off, 64, a.edge_off - x_off - off);
                        tc::mma_bf16_lanes<14>(tmem, es, bs, idesc, acc, lead);
                        acc = 1;
                    }
                    if (EDGE) {
                        xc += dxc;
                        if (xc >= cw) xc -= cw;
                    }
                }
                tc::mma_commit(&bars.empty[s], lead);
                if (++s == a.ns) {
                    s = 0;
                    ph ^= 1u;
                }
            }
            if (ok) tc::mma_commit(&bars.accf, lead);
            if (acc) {
                tc::mma_commit(&bars.drain, lead);
                (void)tc::mbar_wait(&bars.drain, 0, nullptr);
            }
        }
        __syncwarp();
    } else {
        // ----------------------------- bias gradient, then the accumulator
        bool ok = true;
        if (has_bias) {
            // thread: channel pair `pair` of every block, of the pixels 8 pg .. 8
            // pg + 7 of every chunk, added one after the other (all four warps
            // share the sums: with 8 channels per thread one warp had them all
            // for 32 output channels and held the stages back)
            const int pair = lane & 15, pg = 2 * warp + (lane >> 4);
            float bs[4][2];
#pragma unroll
            for (int j = 0; j < 4; ++j) bs[j][0] = bs[j][1] = 0.f;
            int s = 0;
            uint32_t ph = 0;
            for (int g = 0; g < nstages; ++g) {
                if (!tc::mbar_wait_warp(&bars.full[s], ph, abort_flag)) {
                    fail();
                    ok = false;
                    break;
                }
                const int kn = min(a.nch, mine - g * a.nch);
                const unsigned char *gs = stages + s * stage_bytes + g_off + 8 * pg * 64;
                for (int k = 0; k < kn; ++k, gs += chunk_bytes) {
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        if (j >= a.nco) break;
                        uint32_t v[8];
#pragma unroll
                        for (int p = 0; p < 8; ++p)
                            v[p] = *reinterpret_cast<const uint32_t *>(
                                gs + j * kGBytes + p * 64 +
                                16 * ((pair >> 2) ^ ((p >> 1) & 3)) + 4 * (pair & 3));
#pragma unroll
                        for (int p = 0; p < 8; ++p) {
                            const float2 f = unpack_bf16x2(v[p]);
                            bs[j][0] += f.x;
                            bs[j][1] += f.y;
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
            float *pb = a.pbias + (static_cast<int64_t>(split) * kBiasGroups + pg) * N + 2 * pair;
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (j < a.nco)
                    *reinterpret_cast<float2 *>(pb + j * kBlk) = make_float2(bs[j][0], bs[j][1]);
        }
        if (ok && !tc::mbar_wait_warp(&bars.accf, 0, abort_flag)) {
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
// sum over the splits and their eight pixel groups, each added one after the
// other in order.  A weight has one thread (the loads of 32 splits are in flight
// together; blocks of 64 threads spread a small layer's 9216 values over the
// SMs).  A bias is a chain of 8 x splits terms, up to 608: a block of its own
// brings 8 channels' terms into shared memory, then 8 threads add (as a
// thread's loop over global memory this chain took 26 to 39 us of a layer).
constexpr int kRedThreads = 64;
constexpr int kBiasChannels = 8, kBiasTerms = 320;

__global__ void __launch_bounds__(kRedThreads)
wgrad_reduce_kernel(const float *__restrict__ partial, const float *__restrict__ pbias, int splits,
                    int nci, int nco, int cin, int cout, float *__restrict__ gw,
                    float *__restrict__ gb) {
    __shared__ float s_terms[kBiasTerms][kBiasChannels];
    pdl_wait();
    pdl_trigger();
    const int N = nco * kBlk, tid = threadIdx.x;
    const int bias_blocks = N / kBiasChannels;
    if (static_cast<int>(blockIdx.x) < bias_blocks) {
        const int co0 = blockIdx.x * kBiasChannels, terms = kBiasGroups * splits;
        float acc = 0.f;
        for (int t0 = 0; t0 < terms; t0 += kBiasTerms) {
            constexpr int kPer = kBiasTerms * kBiasChannels / kRedThreads;
            float v[kPer];
#pragma unroll
            for (int k = 0; k < kPer; ++k) {
                const int e = k * kRedThreads + tid, t = t0 + e / kBiasChannels;
                v[k] = t < terms ? pbias[static_cast<int64_t>(t) * N + co0 + e % kBiasChannels] : 0.f;
            }
            __syncthreads();
#pragma unroll
            for (int k = 0; k < kPer; ++k) {
                const int e = k * kRedThreads + tid;
                s_terms[e / kBiasChannels][e % kBiasChannels] = v[k];
            }
            __syncthreads();
            if (tid < kBiasChannels) {
#pragma unroll 16
                for (int t = 0; t < kBiasTerms; ++t) acc += s_terms[t][tid];  // zeros past the end
            }
        }
        if (tid < kBiasChannels && co0 + tid < cout && gb) gb[co0 + tid] = acc;
        return;
    }
    const int64_t nw = static_cast<int64_t>(nci) * 3 * N * kLanes;
    const int64_t at = static_cast<int64_t>(blockIdx.x - bias_blocks) * kRedThreads + tid;
    if (at >= nw) return;
    const float *p = partial + at;
    float acc = 0.f;
    constexpr int kU = 32;
    for (int s = 0; s < splits; s += kU) {
        float v[kU];
#pragma unroll
        for (int u = 0; u < kU; ++u) v[u] = s + u < splits ? p[(s + u) * nw] : 0.f;
#pragma unroll
        for (int u = 0; u < kU; ++u) acc += v[u];
    }
    const int row = static_cast<int>(at % kLanes);
    const int r = static_cast<int>(at / kLanes);
    const int co = r % N, cd = r / N;  // cd = ci 3 + dy
    const int ci = (cd / 3) * kBlk + row % kBlk;
    if (ci < cin && co < cout)
        gw[(static_cast<int64_t>(co) * cin + ci) * 9 + (cd % 3) * 3 + row / kBlk] = acc;
}

// NHWC BF16 [B][H][W][C] as a 4-D tensor (channel, x, y, image) of its first
// `columns` columns, box 32 channels x bx pixels of one row; channels beyond C and
// pixels outside those columns or the image arrive as zeros.
bool nhwc_map(CUtensorMap *map, const __nv_bfloat16 *p, int B, int H, int W, int C, int columns,
              int bx) {
    auto enc = tensor_map_encoder();
    if (!enc) return false;
    cuuint64_t dims[4] = {static_cast<cuuint64_t>(C), static_cast<cuuint64_t>(columns),
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
    int rem, chunk;  // W % 16, bytes of a chunk
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
    p.rem = W % 16;
    p.chunk = kXSlot + (p.rem ? kEdgeBytes : 0) + p.nco * kGBytes;
    const int stage = p.nch * p.chunk;
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
    if (p.nchunks > 0x7fffffff) return SPP_ERR_ARG;
    CUtensorMap xm0, xm1, gm, em0, em1;
    if (!nhwc_map(&xm0, a.x0, a.B, a.H, a.W, a.c0, a.W, kHX) ||
        !nhwc_map(&gm, a.g, a.B, a.H, a.W, a.cg, a.W, kPX))
        return SPP_ERR_CUDA;
    xm1 = xm0;
    if (a.c1 && !nhwc_map(&xm1, a.x1, a.B, a.H, a.W, a.c1, a.W, kHX)) return SPP_ERR_CUDA;
    em0 = xm0;
    em1 = xm1;
    const int without_last = std::max(1, a.W - 1);
    if (p.rem && (!nhwc_map(&em0, a.x0, a.B, a.H, a.W, a.c0, without_last, 8) ||
                  (a.c1 && !nhwc_map(&em1, a.x1, a.B, a.H, a.W, a.c1, without_last, 8))))
        return SPP_ERR_CUDA;
    WKernelArgs k;
    k.H = a.H;
    k.W = a.W;
    k.nchunks = static_cast<int>(p.nchunks);
    k.nci = p.nci;
    k.nco = p.nco;
    k.n0 = a.c1 ? a.c0 / kBlk : p.nci;
    k.ns = p.ns;
    k.nch = p.nch;
    k.steps = ((a.W - 1) % kPX + 1) / 16;
    k.rem = p.rem;
    const bool edge_first = p.rem > 0 && p.rem < 8;
    k.x_off = edge_first ? kEdgeBytes : 0;
    k.edge_off = edge_first ? 0 : kXSlot;
    // a row of one pixel has no other column: a box past the end, all zeros
    k.edge_x = a.W == 1 ? 8 : a.W - p.rem - 1 + (edge_first ? 0 : 8);
    k.g_off = kXSlot + (p.rem ? kEdgeBytes : 0);
    k.partial = static_cast<float *>(ws);
    k.pbias = k.partial + static_cast<size_t>(p.splits) * p.nci * 3 * p.nco * kBlk * kLanes;
    k.status = a.status;
    const int smem = kHeader + 512 + p.ns * p.nch * p.chunk;
    static int configured_dev = -1;
    int dev = 0;
    cudaGetDevice(&dev);
    if (configured_dev != dev) {
        for (auto *kernel : {wgrad_kernel<false>, wgrad_kernel<true>})
            if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     kSmemLimit) != cudaSuccess)
                return SPP_ERR_CUDA;
        configured_dev = dev;
    }
    launch_dependent(a.W % kPX ? wgrad_kernel<true> : wgrad_kernel<false>,
                     dim3(p.splits, 3 * p.nci), dim3(kThreads), smem, stream, k, xm0, xm1, gm, em0,
                     em1);
    const int blocks = p.nci * 3 * p.nco * kBlk * kLanes / kRedThreads + p.nco * kBlk / kBiasChannels;
    launch_dependent(wgrad_reduce_kernel, dim3(blocks), dim3(kRedThreads), 0, stream, k.partial, k.pbias, p.splits, p.nci, p.nco,
                     a.cin, a.cout, gw, gb);
    count_launch(2);
    return launch_status();
}

}  // namespace conv
}  // namespace spp
