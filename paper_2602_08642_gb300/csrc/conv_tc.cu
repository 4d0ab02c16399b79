// 3x3 convolution (zero padding, stride 1) as an implicit GEMM on the
// tcgen05 tensor cores: BF16 operands, FP32 accumulation in TMEM.
//
// GEMM view: M = 128 output pixels of one image row, N = output channels,
// K = 9 taps x input channels.  One CTA per SM runs persistently over
// tiles of TR rows x 128 pixels; the accumulator of each row is an
// M=128 x N block of TMEM columns, double-buffered across tiles so the
// epilogue of one tile overlaps the main loop of the next.
//
// Warp roles (320 threads):
//   warps 0-3  epilogue: tcgen05.ld of the accumulator (warp w reads TMEM
//              lanes 32w..32w+31 = pixels), bias / ReLU / mask, stores;
//   warps 4-7  a second set of epilogue warps (the second half of each
//              tile's rows, TMEM lanes 32 (w - 4)..) when the input arrives by
//              TMA and N <= 64 or N = 128, with warp 9 issuing the copies; otherwise
//              producers: per K chunk of 16 input channels they stage the
//              (TR+2) x 130 pixel halo of the tile in shared memory as K-major
//              rows of 32 bytes per pixel in the 32-byte swizzle ([row][pixel]
//              [16 ch], a_off), with zero padding and the fused upsample +
//              concat on the way (a TMA box writes the plain NHWC case
//              directly); one elected thread
//              bulk-copies the pre-packed weights of the chunk;
//   warp 8     issues the MMAs (one lane): for each row r and tap (dy, dx) the A
//              operand is the halo window starting at row r+dy, pixel dx
//              (a start address moved by whole 32-byte pixel rows, which the
//              swizzled descriptor allows because the swizzle follows the
//              absolute address), the B operand the tap's weight block.  No
//              im2col copy is made.
//
// Stages are recycled through full/empty mbarriers (producers -> MMA via
// arrival counts and transaction bytes, MMA -> producers via
// tcgen05.commit).  Every wait is bounded: on expiry the CTA records
// SPP_ERR_TIMEOUT in the status word, the other roles leave at their next
// wait, and TMEM is freed before the kernel returns.  On every path the MMA warp
// waits for its issued MMAs and the copy thread for its last copies before they
// leave: another role may have given up on them.  (0.15 us a launch: 1080p forward
// 714.0 -> 716.2 us.  The same waits behind the block's last barrier, only where a role
// gave up, changed the roles' code: 735 us.)
#include <cuda_bf16.h>

#include <algorithm>
#include <cstdlib>
#include <cstring>
#include <type_traits>

#include "conv_src.cuh"
#include "conv_tc.cuh"
#include "spp_internal.cuh"
#include "tc_common.cuh"
#include "tma_host.cuh"

namespace spp {
namespace conv {
namespace {

constexpr int kTileX = 128;  // output pixels per row tile (MMA M)
constexpr int kPitch = 130;  // staged halo pixels per row
constexpr int kThreads = 320;
constexpr int kHeader = 384;  // barriers, TMEM slot, abort flag
constexpr int kUpW = kTileX / 2 + 2;  // coarse pixels under a tile's halo (upsampling layers)
constexpr int kSmemLimit = 227 * 1024;             // dynamic shared memory per CTA
constexpr int kSmemBudget = kSmemLimit - 512;      // minus alignment slack

constexpr int kResidentMax = 80 * 1024;  // weights kept in shared memory up to this size

// RES: all weights of the layer stay resident in shared memory (loaded once
// per CTA); otherwise each stage carries its chunk's weights.
template <int N, bool RES>
struct Cfg {
    static constexpr int TR = N <= 64 ? 4 : N <= 128 ? 2 : 1;  // rows per tile
    // halo bytes per stage: (TR+2) x 130 pixel rows of 32 bytes (16 channels),
    // 32-byte swizzled (a_off), a multiple of the 256-byte swizzle period
    static constexpr int kA = ((TR + 2) * kPitch * 32 + 255) / 256 * 256;
    static constexpr int kB = 9 * 2 * N * 16;                   // weight bytes per K chunk
    static constexpr int kStage = RES ? kA : kA + kB;
    static constexpr int kWRegion = RES ? kResidentMax : 0;
    static constexpr int kEpiBytes = RES ? 4 * 2 * (N >= 32 ? 32 : 16) * 32 * 4 : 0;
    static constexpr int kBiasOff = kHeader;                     // FP32 bias [N]
    static constexpr int kZeroOff = kBiasOff + 1024;             // zero operand (stacked)
    // N = 32 and 64: the three dy taps of a halo row are one MMA of 3 N columns
    // whose output spans three neighbouring output rows (below)
    static constexpr bool kStack = (N == 32 || N == 64);
    // rows of the zero operand that resets the TR accumulator rows (at least
    // the 128 rows of the A side), in both 8-channel groups
    static constexpr int kZeroRows = TR * N > 128 ? TR * N : 128;
    static constexpr int kZeroBytes = kStack ? 2 * kZeroRows * 16 : 0;
    static constexpr int kWOff = kZeroOff + kZeroBytes;          // resident weights
    static constexpr int kStagesOff = (kWOff + kWRegion + 255) / 256 * 256;
    // BF16 NHWC outputs leave through TMA tensor stores: a warp stages 32 pixels
    // x kCBs channels in one of its two slots, in the swizzle of that row length
    // (64 or 32 bytes; 16-byte shared stores without bank conflicts)
    static constexpr int kCBs = N < 32 ? N : 32;
    static constexpr int kSlot = 32 * 2 * kCBs;
    // eight epilogue warps (two per TMEM sub-partition, each taking half of
    // a tile's rows) when the layer's input comes by TMA and N <= 64 or N = 128, else four
    // (N = 96 and the resident N = 128 would spill).
    // A block of 32 pixels x 32 channels takes a warp about 1300 cycles, mostly
    // latency: with eight warps 64 -> 128 channels at 960 x 540 takes 64 us, with four
    // 92 us, 128 -> 128 103 and 113 us.
    static constexpr int kEpiWarps = N <= 64 || (N == 128 && !RES) ? 8 : 4;
    static constexpr int kStoreBytes = kEpiWarps * 2 * kSlot;
    // the FP32 planar staging buffers and the BF16 slots share one
    // region (a launch uses one of the two epilogues)
    static constexpr int kOutBytes = kEpiBytes > kStoreBytes ? kEpiBytes : kStoreBytes;
    static constexpr int kNS0 = (kSmemBudget - kStagesOff - kOutBytes) / kStage;
    static constexpr int kNS = kNS0 > 8 ? 8 : kNS0;
    // a stage is published kLag stages after its copies were issued; kLag <=
    // kNS - 2 lets the MMAs of one stage run while the next is published
    static constexpr int kLag = kNS - 2;
    // Stacked MMAs: halo row h feeds output rows h - 2, h - 1, h (dy = 2, 1,
    // 0); the first two and the last two halo rows of a tile feed only the
    // output rows inside the tile, through the matching part of the stacked
    // weights, so each accumulator holds exactly the TR rows; one 0 x 0 MMA
    // with accumulate off resets them at the start of a tile, after which
    // every MMA accumulates
    static constexpr int kRowOff = 0;
    static constexpr int kAccCols = TR * N;
    static constexpr int kCols = tc::pow2_cols(2 * kAccCols);
    static_assert(2 * kAccCols <= 512, "accumulators exceed TMEM");
    // FP32 planar outputs leave through two 8 KB staging buffers ([16 ch][128 px])
    // and TMA tensor stores (resident-weight variants; the heads are)
    static constexpr int kEpiOff = (kStagesOff + kNS * kStage + 511) / 512 * 512;
    static constexpr int kStoreOff = kEpiOff;
    static constexpr int kSmem = kEpiOff + kOutBytes + 512;  // + alignment slack
    // Upsampling layers (tma_in == 3): the coarse rows under a tile's halo,
    // one TMA box of 16 channels, in two buffers after the other areas (when
    // they fit): [buffer 2][kUpRows][kUpW][16 ch], not swizzled
    static constexpr int kUpRows = TR / 2 + 2;
    static constexpr int kUpBox = kUpRows * kUpW * 32;         // bytes of one box
    static constexpr int kUpG = (kUpBox + 127) / 128 * 128;     // its 128-byte aligned slot
    // (upsampling layers have BF16 outputs from four epilogue warps: the buffers
    // may overlap the rest of the staging area)
    static constexpr int kUpOff = (kStoreOff + 4 * 2 * kSlot + 127) / 128 * 128;
    static constexpr int kSmemUp0 = kUpOff + 2 * kUpG + 512;
    static constexpr int kSmemUp = kSmemUp0 > kSmem ? kSmemUp0 : kSmem;
    static constexpr bool kUpFits = kSmemUp <= kSmemLimit;
    static_assert(kSmem <= kSmemLimit, "shared memory over the per-CTA limit");
    static_assert(kNS >= 2, "stage does not fit twice");
};

struct Bars {
    uint64_t full[8];   // producers' halo stores (128 arrivals)
    uint64_t wfull[8];  // weight bulk copies (1 arrival + bytes); [0] only when resident
    uint64_t empty[8];  // MMA done with the stage (tcgen05.commit)
    uint64_t accf[2];   // accumulator ready (tcgen05.commit)
    uint64_t acce[2];   // accumulator drained by the epilogue (128 arrivals)
    uint64_t drain;     // abort path: all issued MMAs complete
    uint64_t upfull[2]; // coarse boxes of an upsampling layer landed (1 arrival + bytes)
    uint64_t updone[2]; // coarse buffer expanded by every producer (160 arrivals)
    uint32_t tmem_base;
    int abort;
};
static_assert(sizeof(Bars) <= kHeader, "header");

// Byte offset in a stage of the 8 channels kg (0, 1) of halo pixel (row, px):
// rows of 32 bytes (one 16-channel K chunk) in the K-major 32-byte swizzle
// (the 16-byte half kg of row q sits at half kg ^ bit 2 of q), the layout a
// TMA box with CU_TENSOR_MAP_SWIZZLE_32B writes to a 256-byte aligned stage
// and the one the MMA reads through a SWIZZLE_32B descriptor at any row start
__device__ __forceinline__ int a_off(int row, int px, int kg) {
    const int q = row * kPitch + px;
    return q * 32 + 16 * (kg ^ ((q >> 2) & 1));
}


// TMA load of an NHWC halo box [1 group][TR+2 rows][130 px][8 ch] (5-D map:
// channel-in-group, x, y, group, image) into shared memory, completing on bar.
__device__ __forceinline__ void tma_load_halo(const CUtensorMap *map, void *dst, uint64_t *bar,
                                              int x, int y, int g, int b) {
    asm volatile(
        "cp.async.bulk.tensor.5d.shared::cluster.global.mbarrier::complete_tx::bytes "
        "[%0], [%1, {%3, %4, %5, %6, %7}], [%2];" ::"r"(tc::smem_u32(dst)),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(tc::smem_u32(bar)), "r"(0), "r"(x), "r"(y),
        "r"(g), "r"(b)
        : "memory");
}

// TMA tensor store of an FP32 box of 32 pixels x 32 (16) planes at (x, y, c, b).
__device__ __forceinline__ void tma_store_planes(const CUtensorMap *map, const void *src, int x,
                                                 int y, int c, int b) {
    asm volatile(
        "cp.async.bulk.tensor.4d.global.shared::cta.bulk_group [%0, {%2, %3, %4, %5}], [%1];" ::"l"(
            reinterpret_cast<uint64_t>(map)),
        "r"(tc::smem_u32(src)), "r"(x), "r"(y), "r"(c), "r"(b)
        : "memory");
}
// TMA tensor store of 32 pixels x kCBs channels of BF16 NHWC from a warp's
// staging slot at (c, x, y, b), clipped at the image's edges.
__device__ __forceinline__ void tma_store_nhwc(const CUtensorMap *map, const void *src, int c, int x,
                                               int y, int b) {
    asm volatile(
        "cp.async.bulk.tensor.4d.global.shared::cta.bulk_group [%0, {%2, %3, %4, %5}], [%1];" ::"l"(
            reinterpret_cast<uint64_t>(map)),
        "r"(tc::smem_u32(src)), "r"(c), "r"(x), "r"(y), "r"(b)
        : "memory");
}
__device__ __forceinline__ void tma_store_commit() {
    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
}
// Two FP32 additions in one instruction (each rounded to nearest even).
__device__ __forceinline__ float2 add2(float2 a, float2 b) {
    float2 d;
    asm("{\n\t.reg .b64 x, y, z;\n\t"
        "mov.b64 x, {%2, %3};\n\tmov.b64 y, {%4, %5};\n\t"
        "add.rn.f32x2 z, x, y;\n\tmov.b64 {%0, %1}, z;\n\t}"
        : "=f"(d.x), "=f"(d.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return d;
}
// bf16x2 maximum with 0 of each half (NaN gives 0, as fmaxf(x, 0) does)
__device__ __forceinline__ uint32_t relu_bf16x2(uint32_t u) {
    uint32_t d;
    asm("max.bf16x2 %0, %1, %2;" : "=r"(d) : "r"(u), "r"(0u));
    return d;
}
// the BF16 pair u where the halves of m are positive, else 0
__device__ __forceinline__ uint32_t mask_bf16x2(uint32_t u, uint32_t m) {
    uint32_t on;
    asm("set.gt.u32.bf16x2 %0, %1, %2;" : "=r"(on) : "r"(m), "r"(0u));
    return u & on;
}
// the stores committed before the last `pending` have finished reading shared memory
template <int P>
__device__ __forceinline__ void tma_store_wait_read() {
    asm volatile("cp.async.bulk.wait_group.read %0;" ::"n"(P) : "memory");
}
__device__ __forceinline__ void tma_store_wait_all() {
    asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
}

template <int N, bool RES>
__global__ void __launch_bounds__(kThreads, 1) conv3x3_kernel(const ConvArgs a,
                                                             const __grid_constant__ CUtensorMap omap,
                                                             const __grid_constant__ CUtensorMap imap,
                                                             const __grid_constant__ CUtensorMap umap) {
    // omap: the output (FP32 planes or BF16 NHWC), imap: the NHWC input, umap: the
    // coarse source of an upsampling layer
    using C = Cfg<N, RES>;
    constexpr int TR = C::TR, NS = C::kNS;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    unsigned char *base = smem_raw + ((512u - (tc::smem_u32(smem_raw) & 511u)) & 511u);
    Bars &bars = *reinterpret_cast<Bars *>(base);
    unsigned char *wres = base + C::kWOff;              // resident weights (RES)
    unsigned char *stages = base + C::kStagesOff;
    float *sbias = reinterpret_cast<float *>(base + C::kBiasOff);
    const int tid = threadIdx.x, lane = tid & 31;
    const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);  // known to be the warp's

    const int tiles_x = (a.W + kTileX - 1) / kTileX;
    const int tiles_y = (a.H + TR - 1) / TR;
    const int per_img = tiles_x * tiles_y;
    const int ntiles = a.B * per_img;
    const int kchunks = a.cin_pad / 16;

    // the second set of epilogue warps: for a plain NHWC input (TMA halo, one
    // issuing thread) the producer warps 4-7 take half of each tile's output
    // rows and warp 9 issues the copies
    const bool ep8 = C::kEpiWarps == 8 && a.tma_in == 1 && !(TR < 4 && a.pool_out);
    if (tid == 0) {
        for (int s = 0; s < NS; ++s) {
            tc::mbar_init(&bars.full[s], a.tma_in == 1 ? 1 : a.tma_in == 3 ? 160 : 128);
            tc::mbar_init(&bars.wfull[s], 1);
            tc::mbar_init(&bars.empty[s], 1);
        }
        for (int i = 0; i < 2; ++i) {
            tc::mbar_init(&bars.accf[i], 1);
            tc::mbar_init(&bars.acce[i], ep8 ? 256 : 128);
        }
        tc::mbar_init(&bars.drain, 1);
        for (int i = 0; i < 2; ++i) {
            tc::mbar_init(&bars.upfull[i], 1);
            tc::mbar_init(&bars.updone[i], 160);
        }
        bars.abort = 0;
        tc::fence_mbar_init();
    }
    if (C::kStack) {
        // the zero operand that resets an accumulator (0 x 0 with accumulate off)
        for (int i = tid; i < C::kZeroBytes / 16; i += kThreads)
            reinterpret_cast<uint4 *>(base + C::kZeroOff)[i] = make_uint4(0, 0, 0, 0);
        tc::fence_proxy_async();
    }
    if (warp == 8) tc::tmem_alloc(&bars.tmem_base, C::kCols);
    // launched as a programmatic dependent: the set-up above touches no global
    // memory; every global access below comes after the previous kernel of the
    // stream has completed
    pdl_wait();
    pdl_trigger();
    for (int i = tid; i < N; i += kThreads) sbias[i] = (a.bias && i < a.cout) ? a.bias[i] : 0.f;
    tc::tc_fence_before();
    __syncthreads();
    tc::tc_fence_after();
    const uint32_t tmem = bars.tmem_base;
    volatile int *abort_flag = &bars.abort;
    auto fail = [&]() {
        *abort_flag = 1;
        set_status(a.status, SPP_ERR_TIMEOUT);
    };

    // producers: warps 4-7, joined by warp 9 for an upsampling layer (whose
    // expansion of the coarse boxes bounds it), or warp 9 alone (TMA-fed
    // layers with eight epilogue warps)
    const bool up5 = a.tma_in == 3;
    if (ep8 ? warp == 9 : (warp >= 4 && warp < 8) || (up5 && warp == 9)) {
        // ---------------------------------------------------------- producers
        const int ptid = ep8 ? tid - 288 : warp == 9 ? tid - 160 : tid - 128;
        const int nprod = up5 ? 160 : 128;  // threads sharing the expansion tasks
        constexpr int kTasks = 2 * (TR + 2) * kPitch;  // 16-byte chunks per stage
        // upsampling layers: this thread's coarse pieces (the same in every
        // chunk): coarse row << 10 | coarse column << 1 | 8-channel half
        constexpr int kUpTasks = C::kUpRows * kUpW * 2;
        constexpr int kUpPer = (kUpTasks + 127) / 128;
        int uinfo[kUpPer];
#pragma unroll
        for (int k = 0; k < kUpPer; ++k) {
            const int j = k * nprod + ptid;
            uinfo[k] = j < kUpTasks ? (((j >> 1) / kUpW) << 10) | (((j >> 1) % kUpW) << 1) | (j & 1)
                                    : -1;
        }
        uint32_t it = 0;
        uint32_t issued = 0;  // weight copies issued (by ptid 0)
        bool ok = true;
        // Without TMA the halo goes through cp.async (zero-fill for the
        // padding); a stage is published kLag stages later, so that up to kLag
        // stages of copies are in flight per thread.
        constexpr uint32_t kLag = C::kLag;
        uint32_t published = 0;
        // arrival for a cp.async stage whose copies have landed (TMA stages of
        // an upsampling layer arrived when they were issued)
        auto publish_lagged = [&](uint32_t k) {
            const int ck = static_cast<int>(k % static_cast<uint32_t>(kchunks));
            if (a.tma_in == 2 && ck * 16 < a.c0) return;
            tc::fence_proxy_async();
            tc::mbar_arrive(&bars.full[k % NS]);
        };
        // tma_in == 3: the u-th upsampled chunk of this CTA (tile blockIdx.x +
        // (u / nup) * gridDim.x, chunk c0 / 16 + u % nup) has its coarse box in
        // buffer u & 1; the box of chunk u + 1 is requested while chunk u is
        // expanded
        const int nup = a.tma_in == 3 ? kchunks - a.c0 / 16 : 0;
        uint32_t u_next = 0, u_issued = 0;
        auto issue_up = [&](uint32_t u) {  // thread ptid 0
            const int t = blockIdx.x + static_cast<int>(u / nup) * gridDim.x;
            if (t >= ntiles) return;
            const int b = t / per_img, r = t - b * per_img;
            const int y0 = (r / tiles_x) * TR, x0 = (r % tiles_x) * kTileX;
            uint64_t *bar = &bars.upfull[u & 1];
            tc::mbar_arrive_expect_tx(bar, C::kUpBox);
            tma_load_halo(&umap, base + C::kUpOff + (u & 1) * C::kUpG, bar, (x0 >> 1) - 1,
                          (y0 - 1) >> 1, static_cast<int>(u % nup), b);
            u_issued = u + 1;
        };
        if (nup > 0 && ptid == 0) issue_up(0);
        if (RES && ptid == 0) {
            // the whole packed weight operand, once
            tc::mbar_arrive_expect_tx(&bars.wfull[0], static_cast<uint32_t>(kchunks * C::kB));
            for (int c = 0; c < kchunks; ++c)
                tc::bulk_g2s(wres + c * C::kB,
                             reinterpret_cast<const unsigned char *>(a.wpack) +
                                 static_cast<size_t>(c) * C::kB,
                             C::kB, &bars.wfull[0]);
            issued = 1;
        }
        for (int t = blockIdx.x; t < ntiles && ok; t += gridDim.x) {
            const int b = t / per_img, r = t - b * per_img;
            const int y0 = (r / tiles_x) * TR, x0 = (r % tiles_x) * kTileX;
            for (int c = 0; c < kchunks; ++c) {
                const int s = static_cast<int>(it % NS);
                const uint32_t ph = (it / NS) & 1u;
                if (!tc::mbar_wait(&bars.empty[s], ph ^ 1u, abort_flag)) {
                    fail();
                    ok = false;
                    break;
                }
                unsigned char *As = stages + s * C::kStage;
                if (!RES && ptid == 0) {
                    tc::mbar_arrive_expect_tx(&bars.wfull[s], C::kB);
                    tc::bulk_g2s(As + C::kA,
                                 reinterpret_cast<const unsigned char *>(a.wpack) +
                                     static_cast<size_t>(c) * C::kB,
                                 C::kB, &bars.wfull[s]);
                    ++issued;
                }
                // task j -> 8-channel group j & 1 (fastest), then pixel, then row;
                // shared-memory offset a_off(row, px, kg)
                if (a.tma_in == 1) {
                    // the halo of both 8-channel groups as two TMA boxes (zero fill
                    // outside the image and beyond the channels)
                    if (ptid == 0) {
                        tc::mbar_arrive_expect_tx(&bars.full[s], kPitch * (TR + 2) * 32);
                        tma_load_halo(&imap, As, &bars.full[s], x0 - 1, y0 - 1, c, b);
                    }
                    ++it;
                    ++published;
                } else if (a.tma_in == 3) {
                    if (c * 16 < a.c0) {
                        // skip-connection chunk: TMA as above, every producer arrives
                        if (ptid == 0) {
                            tc::mbar_arrive_expect_tx(&bars.full[s], kPitch * (TR + 2) * 32);
                            tma_load_halo(&imap, As, &bars.full[s], x0 - 1, y0 - 1, c, b);
                        } else {
                            tc::mbar_arrive(&bars.full[s]);
                        }
                    } else {
                        // upsampled chunk: request the next chunk's coarse box once
                        // its buffer (used by chunk u_next - 1) is expanded, then
                        // expand this one: halo pixel (x, y) <- coarse (x/2, y/2),
                        // zero outside the output grid
                        const uint32_t u = u_next++;
                        if (ptid == 0) {
                            if (u >= 1 && !tc::mbar_wait(&bars.updone[(u - 1) & 1], ((u - 1) >> 1) & 1u,
                                                         abort_flag)) {
                                fail();
                                ok = false;
                                break;
                            }
                            issue_up(u + 1);
                        }
                        if (!tc::mbar_wait(&bars.upfull[u & 1], (u >> 1) & 1u, abort_flag)) {
                            fail();
                            ok = false;
                            break;
                        }
                        const unsigned char *ub = base + C::kUpOff + (u & 1) * C::kUpG;
                        // each coarse piece (cr, cx) goes to the halo rows and
                        // pixels that read it: rows 2 cr - p, 2 cr + 1 - p (p = 1
                        // when y0 is even) and pixels 2 cx - 1, 2 cx (x0 is even),
                        // those inside the halo.  W and H are even, so a halo
                        // pixel outside the image reads a coarse cell outside the
                        // coarse image, which the TMA box filled with zeros.
                        const int par = (y0 - 1) & 1;
#pragma unroll
                        for (int k = 0; k < kUpPer; ++k) {
                            if (uinfo[k] < 0) continue;
                            const int cr = uinfo[k] >> 10, cx = (uinfo[k] >> 1) & 511,
                                      kg = uinfo[k] & 1;
                            const uint4 v = *reinterpret_cast<const uint4 *>(
                                ub + (cr * kUpW + cx) * 32 + kg * 16);
#pragma unroll
                            for (int dr = 0; dr < 2; ++dr) {
                                const int row = 2 * cr + dr - par;
                                if (row < 0 || row > TR + 1) continue;
#pragma unroll
                                for (int dc = 0; dc < 2; ++dc) {
                                    const int px = 2 * cx + dc - 1;
                                    if (px < 0 || px >= kPitch) continue;
                                    *reinterpret_cast<uint4 *>(As + a_off(row, px, kg)) = v;
                                }
                            }
                        }
                        tc::fence_proxy_async();
                        tc::mbar_arrive(&bars.full[s]);
                        tc::mbar_arrive(&bars.updone[u & 1]);
                    }
                    ++it;
                    ++published;
                } else if (a.tma_in == 2 && c * 16 < a.c0) {
                    // upsampling layer, skip-connection chunk: TMA as above, every
                    // producer arrives now; an empty copy group keeps the count of
                    // groups equal to the count of stages for the lagged ones
                    if (ptid == 0) {
                        tc::mbar_arrive_expect_tx(&bars.full[s], kPitch * (TR + 2) * 32);
                        tma_load_halo(&imap, As, &bars.full[s], x0 - 1, y0 - 1, c, b);
                    } else {
                        tc::mbar_arrive(&bars.full[s]);
                    }
                    cp_async_commit();
                    ++it;
                    if (it > kLag) {
                        cp_async_wait<kLag>();
                        publish_lagged(published);
                        ++published;
                    }
                } else {
                    const uint32_t sbase = tc::smem_u32(As);
#pragma unroll 4
                    for (int j = ptid; j < kTasks; j += nprod) {
                        const int row = (j >> 1) / kPitch, px = (j >> 1) % kPitch, kg = j & 1;
                        const __nv_bfloat16 *src = chunk_address(a, b, y0 - 1 + row, x0 - 1 + px,
                                                                 c * 16 + kg * 8);
                        cp_async16(sbase + a_off(row, px, kg),
                                   src ? src : a.src0, src ? 16u : 0u);
                    }
                    cp_async_commit();
                    ++it;
                    if (it > kLag) {
                        cp_async_wait<kLag>();
                        publish_lagged(published);
                        ++published;
                    }
                }
            }
        }
        // publish the stages still in flight (also on the abort path, where the
        // copies must land before the CTA exits)
        cp_async_wait<0>();
        for (; published < it; ++published) publish_lagged(published);
        if (ptid == 0) {
            // wait (bounded, ignoring the abort flag) for the copies still in flight:
            // those of the last stages, of which the MMA warp may have given up
            if (a.tma_in == 1) {
                const uint32_t first = it > NS ? it - NS : 0;
                for (uint32_t k = first; k < it; ++k)
                    (void)tc::mbar_wait(&bars.full[k % NS], (k / NS) & 1u, nullptr);
            }
            if (a.tma_in >= 2) {
                // the skip-connection boxes (TMA) among the last stages
                const uint32_t first = it > NS ? it - NS : 0;
                for (uint32_t k = first; k < it; ++k)
                    if (static_cast<int>(k % static_cast<uint32_t>(kchunks)) * 16 < a.c0)
                        (void)tc::mbar_wait(&bars.full[k % NS], (k / NS) & 1u, nullptr);
            }
            // coarse boxes requested (the last two, one per buffer)
            for (uint32_t k = u_issued > 2 ? u_issued - 2 : 0; k < u_issued; ++k)
                (void)tc::mbar_wait(&bars.upfull[k & 1], (k >> 1) & 1u, nullptr);
            if (RES) {
                if (issued) (void)tc::mbar_wait(&bars.wfull[0], 0, nullptr);
            } else {
                const uint32_t first = issued > NS ? issued - NS : 0;
                for (uint32_t k = first; k < issued; ++k)
                    (void)tc::mbar_wait(&bars.wfull[k % NS], (k / NS) & 1u, nullptr);
            }
        }
    } else if (warp == 8) {
        // -------------------------------------------------------- MMA issuer
        {
            // One lane issues, but the code is the whole warp's, so that descriptors,
            // each one addition from a stage's first, can stay in uniform registers.
            // The issue rate bounds the layers of N <= 64: 4K forward 2.48 ms with a
            // descriptor built for every MMA in one lane's branch, 2.42 with
            // additions, 2.38 with warp-uniform code.  All lanes take part in every
            // wait: the warp stays converged, which uniform registers rely on.
            const uint32_t lead = tc::elect_one();
            auto wait = [&](uint64_t *bar, uint32_t parity) {
                return tc::mbar_wait_warp(bar, parity, abort_flag);
            };
            constexpr uint32_t idesc = tc::idesc_bf16_f32(128, N);
            constexpr uint32_t kLboB = N * 16;
            uint32_t it = 0, tl = 0;
            bool ok = true, pending = false;
            if (RES && ntiles > static_cast<int>(blockIdx.x) && !wait(&bars.wfull[0], 0)) {
                fail();
                ok = false;
            }
            for (int t = blockIdx.x; t < ntiles && ok; t += gridDim.x, ++tl) {
                const int acc = tl & 1;
                if (!wait(&bars.acce[acc], ((tl >> 1) & 1u) ^ 1u)) {
                    fail();
                    ok = false;
                    break;
                }
                tc::tc_fence_after();
                const uint32_t d0 = tmem + acc * C::kAccCols;
                pending = true;
                if (C::kStack) {
                    // reset the TR accumulator rows
                    const uint64_t zd = tc::smem_desc(tc::smem_u32(base + C::kZeroOff),
                                                      C::kZeroRows * 16, 128);
                    tc::mma_bf16(d0, zd, zd, tc::idesc_bf16_f32(128, TR * N), 0u, lead);
                }
                for (int c = 0; c < kchunks; ++c, ++it) {
                    const int s = static_cast<int>(it % NS);
                    const uint32_t ph = (it / NS) & 1u;
                    if (!wait(&bars.full[s], ph) || (!RES && !wait(&bars.wfull[s], ph))) {
                        fail();
                        ok = false;
                        break;
                    }
                    tc::tc_fence_after();
                    const uint32_t a_base = tc::smem_u32(stages + s * C::kStage);
                    const uint64_t a_desc = tc::smem_desc_sw32(a_base);
                    const uint64_t b_desc =
                        tc::smem_desc(RES ? tc::smem_u32(wres + c * C::kB) : a_base + C::kA,
                                      C::kStack ? 3 * N * 16 : kLboB, 128);
                    if (C::kStack) {
                        // halo row h feeds output rows h-2, h-1, h through the
                        // stacked weights [dy = 2; dy = 1; dy = 0] of its dx tap;
                        // rows outside the tile are left out (the matching part of
                        // the stacked weights, fewer MMA columns)
#pragma unroll
                        for (int dx = 0; dx < 3; ++dx) {
#pragma unroll
                            for (int h = 0; h < TR + 2; ++h) {
                                const int rlo = h - 2 < 0 ? 0 : h - 2;   // first row fed
                                const int rhi = h < TR - 1 ? h : TR - 1;  // last row fed
                                const int k0 = rlo - (h - 2);             // its dy block
                                const uint64_t bd =
                                    b_desc + tc::desc_offset((dx * 6 + k0) * N * 16);
                                const uint64_t ad =
                                    a_desc + tc::desc_offset((h * kPitch + dx) * 32);
                                tc::mma_bf16(d0 + rlo * N, ad, bd,
                                             tc::idesc_bf16_f32(128, (rhi - rlo + 1) * N), 1u,
                                             lead);
                            }
                        }
                    } else {
#pragma unroll
                        for (int tap = 0; tap < 9; ++tap) {
                            const int dy = tap / 3, dx = tap % 3;
                            const uint64_t bd = b_desc + tc::desc_offset(tap * 2 * N * 16);
#pragma unroll
                            for (int r = 0; r < TR; ++r) {
                                const uint64_t ad =
                                    a_desc + tc::desc_offset(((r + dy) * kPitch + dx) * 32);
                                tc::mma_bf16(d0 + r * N, ad, bd, idesc, (c | tap) != 0, lead);
                            }
                        }
                    }
                    tc::mma_commit(&bars.empty[s], lead);
                }
                if (!ok) break;
                tc::mma_commit(&bars.accf[acc], lead);
            }
            if (pending) {
                tc::mma_commit(&bars.drain, lead);
                (void)tc::mbar_wait(&bars.drain, 0, nullptr);
            }
        }
        __syncwarp();
    } else if (warp < 4 || (ep8 && warp < 8)) {
        // ----------------------------------------------------------- epilogue
        // warp w reads TMEM lanes 32 (w % 4) ..; with eight epilogue warps,
        // warps 0-3 take the first half of a tile's rows and 4-7 the second
        const int sub = warp & 3;
        const int row_lo = ep8 ? (warp >> 2) * (TR / 2) : 0;
        const int row_hi = ep8 ? row_lo + TR / 2 : TR;
        uint32_t tl = 0;
        uint32_t eblk = 0;  // TMA-stored blocks
        const uint32_t lane_base = static_cast<uint32_t>(sub * 32) << 16;
        // BF16 NHWC blocks: 32 pixels x kCB channels, kW packed pairs per pixel
        constexpr int kCB = C::kCBs, kW = kCB / 2;
        unsigned char *slots = base + C::kStoreOff + warp * 2 * C::kSlot;
        // this lane's pixel row in a slot, and its swizzle (bits 7.. of the address)
        const uint32_t swz = kCB == 32 ? (lane >> 1) & 3 : (lane >> 2) & 1;
        auto store_block = [&](const uint32_t (&w)[kW], int c, int x0, int y, int b) {
            unsigned char *slot = slots + (eblk & 1) * C::kSlot;
            if (lane == 0) tma_store_wait_read<1>();  // the slot's previous store
            __syncwarp();
            uint4 *row = reinterpret_cast<uint4 *>(slot + lane * 2 * kCB);
#pragma unroll
            for (int q = 0; q < kW / 4; ++q)
                row[q ^ swz] = make_uint4(w[4 * q], w[4 * q + 1], w[4 * q + 2], w[4 * q + 3]);
            tc::fence_proxy_async();
            __syncwarp();
            if (lane == 0) {
                if (y < a.H && x0 < a.W) tma_store_nhwc(&omap, slot, c, x0, y, b);
                tma_store_commit();
            }
            ++eblk;
        };
        // accumulators + bias as BF16 pairs
        auto pack_bias = [&](const uint32_t *v, int j0, bool relu, uint32_t (&w)[kW]) {
#pragma unroll
            for (int e = 0; e < kCB; e += 4) {
                const float4 bb = *reinterpret_cast<const float4 *>(sbias + j0 + e);
                const float2 f0 = add2(make_float2(__uint_as_float(v[e]), __uint_as_float(v[e + 1])),
                                       make_float2(bb.x, bb.y));
                const float2 f1 =
                    add2(make_float2(__uint_as_float(v[e + 2]), __uint_as_float(v[e + 3])),
                         make_float2(bb.z, bb.w));
                w[e / 2] = pack_bf16x2(f0.x, f0.y);
                w[e / 2 + 1] = pack_bf16x2(f1.x, f1.y);
                if (relu) {
                    w[e / 2] = relu_bf16x2(w[e / 2]);
                    w[e / 2 + 1] = relu_bf16x2(w[e / 2 + 1]);
                }
            }
        };
        for (int t = blockIdx.x; t < ntiles; t += gridDim.x, ++tl) {
            const int acc = tl & 1;
            const int b = t / per_img, rr = t - b * per_img;
            const int y0 = (rr / tiles_x) * TR, x = (rr % tiles_x) * kTileX + sub * 32 + lane;
            // the layer below's activations (mask) of block k of the tile; each
            // block's are requested one block ahead, the first before the wait
            constexpr int kRowBlocks = N / kCB;
            constexpr int kBlocks = TR * kRowBlocks;
            uint4 mask[2][kW / 4];
            auto load_mask = [&](int k, uint4 (&m)[kW / 4]) {
                const int y = y0 + k / kRowBlocks, j0 = (k % kRowBlocks) * kCB;
                const bool inside = x < a.W && y < a.H;
                const size_t pix = (static_cast<size_t>(b) * a.H + y) * a.W + x;
                const uint4 *src = reinterpret_cast<const uint4 *>(a.act + pix * N + j0);
#pragma unroll
                for (int q = 0; q < kW / 4; ++q)
                    m[q] = inside ? __ldg(src + q) : make_uint4(0, 0, 0, 0);
            };
            if (a.epi_mode == kEpiMaskBF16) load_mask(row_lo * kRowBlocks, mask[0]);
            if (!tc::mbar_wait_warp(&bars.accf[acc], (tl >> 1) & 1u, abort_flag)) {
                fail();
                break;
            }
            tc::tc_fence_after();
            const uint32_t abase = tmem + lane_base + acc * C::kAccCols + C::kRowOff * N;
            // hands the accumulator back to the MMA warp
            auto release_acc = [&]() {
                tc::tc_fence_before();
                tc::mbar_arrive(&bars.acce[acc]);
            };
            const int xw = x - lane;  // the warp's first pixel
            if (TR % 2 == 0 && a.pool_out) {
                // ReLU rows in pairs, plus the 2x2 average of their BF16 values
                // (lanes x and x^1 hold horizontal neighbours), up to 32 columns
                // of both rows per TMEM round trip.  Each lane of a pair averages
                // half of the channels and stores them as one 32-byte sector.
#pragma unroll 1
                for (int r = row_lo; r < row_hi; r += 2) {
                    const int y = y0 + r;
#pragma unroll 1
                    for (int j0 = 0; j0 < N; j0 += kCB) {
                        uint32_t v0[kCB], v1[kCB];
#pragma unroll
                        for (int q = 0; q < kCB / 16; ++q) {
                            tc::tmem_ld16(abase + r * N + j0 + 16 * q,
                                          *reinterpret_cast<uint32_t(*)[16]>(v0 + 16 * q));
                            tc::tmem_ld16(abase + (r + 1) * N + j0 + 16 * q,
                                          *reinterpret_cast<uint32_t(*)[16]>(v1 + 16 * q));
                        }
                        tc::tmem_wait_ld();
                        uint32_t w0[kW], w1[kW];
                        pack_bias(v0, j0, true, w0);
                        pack_bias(v1, j0, true, w1);
                        store_block(w0, j0, xw, y, b);
                        store_block(w1, j0, xw, y + 1, b);
                        const bool odd = lane & 1;
                        uint32_t wp[kW / 2];
                        auto sum2 = [](uint32_t p, uint32_t q) {  // p + q, as FP32 pairs
                            return add2(make_float2(__uint_as_float(p << 16),
                                                    __uint_as_float(p & 0xffff0000u)),
                                        make_float2(__uint_as_float(q << 16),
                                                    __uint_as_float(q & 0xffff0000u)));
                        };
#pragma unroll
                        for (int k = 0; k < kW / 2; ++k) {
                            const uint32_t mine0 = odd ? w0[k + kW / 2] : w0[k];
                            const uint32_t mine1 = odd ? w1[k + kW / 2] : w1[k];
                            const uint32_t other0 = __shfl_xor_sync(
                                0xffffffffu, odd ? w0[k] : w0[k + kW / 2], 1);
                            const uint32_t other1 = __shfl_xor_sync(
                                0xffffffffu, odd ? w1[k] : w1[k + kW / 2], 1);
                            const float2 s = add2(sum2(mine0, mine1), sum2(other0, other1));
                            wp[k] = pack_bf16x2(0.25f * s.x, 0.25f * s.y);
                        }
                        if (x - (lane & 1) < a.W && y + 1 < a.H) {
                            uint4 *o = reinterpret_cast<uint4 *>(
                                a.pool_out +
                                ((static_cast<size_t>(b) * (a.H >> 1) + (y >> 1)) * (a.W >> 1) +
                                 (x >> 1)) * N + j0 + (odd ? kCB / 2 : 0));
#pragma unroll
                            for (int q = 0; q < kW / 8; ++q)
                                o[q] = make_uint4(wp[4 * q], wp[4 * q + 1], wp[4 * q + 2],
                                                  wp[4 * q + 3]);
                        }
                    }
                }
                release_acc();
                continue;
            }
            if (RES && a.epi_mode == kEpiF32Planar && a.tma_out) {
                // each epilogue warp stages kPB output planes of its 32 pixels of
                // the row in its own buffer and stores them with one TMA tensor
                // store (clipped at W and at cout); two buffers per warp, one
                // when eight warps share the staging area
                constexpr int kPB = N >= 32 ? 32 : 16;  // planes per block
                // (from the thread index: with addresses from the uniform warp index
                // h0 took 464 us at 3840 x 2160, so 424; the BF16 blocks are faster
                // with the uniform one, e0a 137 against 147 us)
                const int wv = tid >> 5, sv = wv & 3;
                const uint32_t vbase = tmem + (static_cast<uint32_t>(sv * 32) << 16) +
                                       acc * C::kAccCols + C::kRowOff * N;
                float *ebuf = reinterpret_cast<float *>(base + C::kEpiOff);
                const int x0 = (rr % tiles_x) * kTileX;
                constexpr int kRowBlocks = N / kPB;
                constexpr int kBlocks = TR * kRowBlocks;
                auto tmem_read = [&](int k, uint32_t (&vv)[kPB]) {
#pragma unroll
                    for (int q = 0; q < kPB / 16; ++q)
                        tc::tmem_ld16(vbase + (k / kRowBlocks) * N + (k % kRowBlocks) * kPB + 16 * q,
                                      *reinterpret_cast<uint32_t(*)[16]>(vv + 16 * q));
                };
                auto pblocks = [&](auto count_c, int kb_lo) {
                    constexpr int kCount = decltype(count_c)::value;
                    uint32_t fbuf[2][kPB];
                    tmem_read(kb_lo, fbuf[0]);
                    tc::tmem_wait_ld();
#pragma unroll
                    for (int kk = 0; kk < kCount; ++kk) {
                        const int kb = kb_lo + kk;
                        if (kk + 1 < kCount) tmem_read(kb + 1, fbuf[(kk + 1) & 1]);
                        const uint32_t (&v)[kPB] = fbuf[kk & 1];
                        const int y = y0 + kb / kRowBlocks, j0 = (kb % kRowBlocks) * kPB;
                        if (j0 < a.cout) {  // padding columns are not stored
                            float *buf = ebuf + (ep8 ? wv : wv * 2 + static_cast<int>(eblk & 1)) *
                                                    kPB * 32;
                            if (lane == 0) {
                                if (ep8)
                                    tma_store_wait_read<0>();
                                else
                                    tma_store_wait_read<1>();
                            }
                            __syncwarp();
#pragma unroll
                            for (int e = 0; e < kPB; e += 4) {
                                const float4 bb = *reinterpret_cast<const float4 *>(sbias + j0 + e);
                                buf[e * 32 + lane] = __uint_as_float(v[e]) + bb.x;
                                buf[(e + 1) * 32 + lane] = __uint_as_float(v[e + 1]) + bb.y;
                                buf[(e + 2) * 32 + lane] = __uint_as_float(v[e + 2]) + bb.z;
                                buf[(e + 3) * 32 + lane] = __uint_as_float(v[e + 3]) + bb.w;
                            }
                            tc::fence_proxy_async();
                            __syncwarp();
                            if (lane == 0) {
                                if (y < a.H && x0 + sv * 32 < a.W)
                                    tma_store_planes(&omap, buf, x0 + sv * 32, y, j0, b);
                                // a group per block, or a block outside the image would
                                // shift the count of stores still to wait for
                                tma_store_commit();
                            }
                            ++eblk;
                        }
                        tc::tmem_wait_ld();
                    }
                };
                if (ep8)
                    pblocks(std::integral_constant<int, kBlocks / 2>{}, row_lo * kRowBlocks);
                else
                    pblocks(std::integral_constant<int, kBlocks>{}, 0);
                release_acc();
                continue;
            }
            // one row at a time, up to 32 columns per TMEM round trip; the
            // next block's TMEM read is in flight while this one is stored
            // (tcgen05.wait::ld waits for every outstanding read, so each
            // wait covers exactly the one issued before the stores)
            auto tmem_read = [&](int k, uint32_t (&vv)[kCB]) {
                const int r = k / kRowBlocks, j0 = (k % kRowBlocks) * kCB;
#pragma unroll
                for (int q = 0; q < kCB / 16; ++q)
                    tc::tmem_ld16(abase + r * N + j0 + 16 * q,
                                  *reinterpret_cast<uint32_t(*)[16]>(vv + 16 * q));
            };
            // blocks [kb_lo, kb_lo + kCount) of the tile (kCount a constant, so
            // that the double buffer stays in registers)
            auto blocks = [&](auto count_c, int kb_lo) {
                constexpr int kCount = decltype(count_c)::value;
                uint32_t vbuf[2][kCB];
                tmem_read(kb_lo, vbuf[0]);
                tc::tmem_wait_ld();
#pragma unroll
                for (int kk = 0; kk < kCount; ++kk) {
                    const int kb = kb_lo + kk;
                    if (kk + 1 < kCount) {
                        tmem_read(kb + 1, vbuf[(kk + 1) & 1]);
                        if (a.epi_mode == kEpiMaskBF16) load_mask(kb + 1, mask[(kk + 1) & 1]);
                    }
                    const uint32_t (&v)[kCB] = vbuf[kk & 1];
                    const int r = kb / kRowBlocks, j0 = (kb % kRowBlocks) * kCB;
                    const int y = y0 + r;
                    if (a.epi_mode == kEpiF32Planar) {
                        if (x < a.W && y < a.H) {
                            const size_t plane = static_cast<size_t>(a.H) * a.W;
                            float *o = a.outf + static_cast<size_t>(b) * a.cout * plane +
                                       static_cast<size_t>(y) * a.W + x;
#pragma unroll
                            for (int e = 0; e < kCB; ++e) {
                                const int n = j0 + e;
                                if (n < a.cout) __stcs(o + n * plane, __uint_as_float(v[e]) + sbias[n]);
                            }
                        }
                    } else {
                        uint32_t w[kW];
                        if (a.epi_mode == kEpiMaskBF16) {
#pragma unroll
                            for (int q = 0; q < kW / 4; ++q) {
                                const uint32_t *mu = &mask[kk & 1][q].x;
#pragma unroll
                                for (int k = 0; k < 4; ++k)
                                    w[4 * q + k] = mask_bf16x2(
                                        pack_bf16x2(__uint_as_float(v[8 * q + 2 * k]),
                                                    __uint_as_float(v[8 * q + 2 * k + 1])),
                                        mu[k]);
                            }
                        } else {
                            pack_bias(v, j0, a.epi_mode == kEpiReluBF16, w);
                        }
                        store_block(w, j0, xw, y, b);
                    }
                    tc::tmem_wait_ld();
                }
            };
            if (ep8)
                blocks(std::integral_constant<int, kBlocks / 2>{}, row_lo * kRowBlocks);
            else
                blocks(std::integral_constant<int, kBlocks>{}, 0);
            release_acc();
        }
        if (lane == 0 && eblk) tma_store_wait_all();
    }

    tc::tc_fence_before();
    __syncthreads();
    if (warp == 8) {
        tc::tc_fence_after();
        tc::tmem_dealloc(tmem, C::kCols);
    }
}

// Eight consecutive input channels of one operand row per thread (a 16-byte
// store); a block works on one item of the table.
constexpr int kPackThreads = 256;

__global__ void __launch_bounds__(kPackThreads)
pack_weights_kernel(const __grid_constant__ PackTable table) {
    int i = 0;
    while (i + 1 < table.count && static_cast<int>(blockIdx.x) >= table.it[i + 1].first_block) ++i;
    const PackItem &it = table.it[i];
    const int cin = it.cin, cout = it.cout, n = it.n;
    const int block = blockIdx.x - it.first_block;
    if (block == 0 && it.bias_dst)
        for (int j = threadIdx.x; j < n; j += kPackThreads)
            it.bias_dst[j] = j < cout ? it.bias[j] : 0.f;
    const int idx = block * kPackThreads + threadIdx.x;
    if (idx >= it.cin_pad / 16 * 18 * n) return;
    int o, kg, c, dy, dx;
    if (n == 32 || n == 64) {
        // stacked: [chunk][dx][kg][3 n = (dy = 2, 1, 0) x n][8]
        const int S = 3 * n, n3 = idx % S;
        kg = (idx / S) % 2;
        dx = (idx / (2 * S)) % 3;
        c = idx / (6 * S);
        o = n3 % n;
        dy = 2 - n3 / n;
    } else {
        // [chunk][tap][kg][n][8]
        o = idx % n;
        kg = (idx / n) % 2;
        const int tap = (idx / (2 * n)) % 9;
        c = idx / (18 * n);
        dy = tap / 3;
        dx = tap % 3;
    }
    uint32_t w[4];
#pragma unroll
    for (int h = 0; h < 4; ++h) {
        float v[2];
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const int k = c * 16 + kg * 8 + 2 * h + e;  // input channel of this convolution
            v[e] = 0.f;
            if (!it.transpose) {
                if (o < cout && k < cin)
                    v[e] = it.w[((static_cast<int64_t>(o) * cin + k) * 3 + dy) * 3 + dx];
            } else {  // data gradient: input channel k is an output channel of w
                if (o < cin && k < cout)
                    v[e] = it.w[((static_cast<int64_t>(k) * cin + o) * 3 + (2 - dy)) * 3 + (2 - dx)];
            }
        }
        w[h] = pack_bf16x2(v[0], v[1]);
    }
    reinterpret_cast<uint4 *>(it.dst)[idx] = make_uint4(w[0], w[1], w[2], w[3]);
}

// SPP_CONV_NO_TMA_IN=1 selects the cp.async halo producers instead of TMA
// (comparison and fallback).
bool getenv_disable_tma_in() {
    static const bool off = [] {
        const char *v = getenv("SPP_CONV_NO_TMA_IN");
        return v && v[0] == '1';
    }();
    return off;
}

// Upsampling layers (kSrcConcatUp: a skip tensor concatenated with the 2x
// nearest upsampling of a coarse one) without expanding anything in shared
// memory: the columns of the output are split into their even and odd ones.
// Row m of an MMA is the pixel pair at coarse column xc = xc0 + m; output phase
// a (pixel 2 xc + a) has its own accumulators, and tap dx of it reads
//   the upsampled tensor at coarse column (2 xc + a + dx - 1) >> 1, one of
//     xc - 1, xc, xc + 1;
//   the skip tensor at pixel 2 xc + a + dx - 1, a column of its even or its odd
//     plane, which TMA boxes with a doubled x stride bring.
// Every operand is then a window of a staged row, as in conv3x3_kernel: the same
// MMAs and weights, and every sum in the same order (dx by dx within a K chunk, so
// both planes of a skip chunk are staged together): the same bits.
// The rows of an upsampled chunk are shared too: halo row h reads coarse row
// (h + 1) >> 1 of the box.
//
// The expansion (a thread per coarse piece, up to four 16-byte stores) bounds these
// layers, the largest of the network, in conv3x3_kernel: 96 -> 32 channels at
// 3840 x 2160 take 554 us there and 360 us here, 192 -> 64 at 1920 x 1080 329 and
// 289 us (of which handing the phases over one by one is 3 %).
//
// A tile is TR x 256 pixels.  Accumulators take 2 TR N columns: double-buffered
// for N = 32, one set for N = 64 (half-height tiles with two sets would fetch the
// streamed weights twice as often, and L2 is what they are close to), whose phases
// are handed over one by one: phase 0 is read while phase 1 of the last chunk runs.
// Warps 0-3 and 4-7 are the epilogues of phase 0 and 1, warp 8 issues the MMAs,
// warp 9 the copies.
template <int N, bool RES>
__global__ void __launch_bounds__(kThreads, 1)
conv3x3_up_kernel(const ConvArgs a, const __grid_constant__ CUtensorMap omap0,
                  const __grid_constant__ CUtensorMap omap1,
                  const __grid_constant__ CUtensorMap emap,
                  const __grid_constant__ CUtensorMap dmap,
                  const __grid_constant__ CUtensorMap umap) {
    // omap0, omap1: the output's even and odd columns; emap, dmap: the skip
    // tensor's; umap: the coarse tensor
    using C = Cfg<N, RES>;
    constexpr int TR = C::TR, NS = C::kNS;
    static_assert(C::kStack && TR % 2 == 0 && C::kEpiWarps == 8, "stacked layers of even tiles");
    constexpr int kPhase = C::kAccCols;  // accumulator columns of a phase
    constexpr int kSets = 2 * 2 * kPhase <= 512 ? 2 : 1;
    constexpr int kCols = 512;
    constexpr int kUpBytes = (TR / 2 + 2) * kPitch * 32;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    unsigned char *base = smem_raw + ((512u - (tc::smem_u32(smem_raw) & 511u)) & 511u);
    Bars &bars = *reinterpret_cast<Bars *>(base);
    unsigned char *wres = base + C::kWOff;
    unsigned char *stages = base + C::kStagesOff;
    float *sbias = reinterpret_cast<float *>(base + C::kBiasOff);
    const int tid = threadIdx.x, lane = tid & 31;
    const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);  // known to be the warp's

    const int tiles_x = (a.W + 2 * kTileX - 1) / (2 * kTileX);
    const int tiles_y = (a.H + TR - 1) / TR;
    const int per_img = tiles_x * tiles_y;
    const int ntiles = a.B * per_img;
    const int kc0 = a.c0 / 16, kchunks = a.cin_pad / 16;
    const int nst = kchunks + kc0;  // stages per tile: two planes of a skip chunk, an upsampled one

    if (tid == 0) {
        for (int s = 0; s < NS; ++s) {
            tc::mbar_init(&bars.full[s], 1);
            tc::mbar_init(&bars.wfull[s], 1);
            tc::mbar_init(&bars.empty[s], 1);
        }
        for (int i = 0; i < 2; ++i) {
            tc::mbar_init(&bars.accf[i], 1);
            tc::mbar_init(&bars.acce[i], kSets == 2 ? 256 : 128);
        }
        tc::mbar_init(&bars.drain, 1);
        bars.abort = 0;
        tc::fence_mbar_init();
    }
    for (int i = tid; i < C::kZeroBytes / 16; i += kThreads)
        reinterpret_cast<uint4 *>(base + C::kZeroOff)[i] = make_uint4(0, 0, 0, 0);
    tc::fence_proxy_async();
    if (warp == 8) tc::tmem_alloc(&bars.tmem_base, kCols);
    pdl_wait();
    pdl_trigger();
    for (int i = tid; i < N; i += kThreads) sbias[i] = (a.bias && i < a.cout) ? a.bias[i] : 0.f;
    tc::tc_fence_before();
    __syncthreads();
    tc::tc_fence_after();
    const uint32_t tmem = bars.tmem_base;
    volatile int *abort_flag = &bars.abort;
    auto fail = [&]() {
        *abort_flag = 1;
        set_status(a.status, SPP_ERR_TIMEOUT);
    };

    if (warp == 9) {
        // ------------------------------------------------------------- copies
        if (lane == 0) {
            uint32_t it = 0;
            bool ok = true;
            if (RES && static_cast<int>(blockIdx.x) < ntiles) {
                tc::mbar_arrive_expect_tx(&bars.wfull[0], static_cast<uint32_t>(kchunks * C::kB));
                for (int c = 0; c < kchunks; ++c)
                    tc::bulk_g2s(wres + c * C::kB,
                                 reinterpret_cast<const unsigned char *>(a.wpack) +
                                     static_cast<size_t>(c) * C::kB,
                                 C::kB, &bars.wfull[0]);
            }
            for (int t = blockIdx.x; t < ntiles && ok; t += gridDim.x) {
                const int b = t / per_img, r = t - b * per_img;
                const int y0 = (r / tiles_x) * TR, xc0 = (r % tiles_x) * kTileX;
                for (int st = 0; st < nst; ++st, ++it) {
                    const int s = static_cast<int>(it % NS);
                    if (!tc::mbar_wait(&bars.empty[s], ((it / NS) & 1u) ^ 1u, abort_flag)) {
                        fail();
                        ok = false;
                        break;
                    }
                    unsigned char *As = stages + s * C::kStage;
                    const bool skip = st < 2 * kc0;
                    const int c = skip ? st >> 1 : st - kc0;
                    if (!RES && skip && (st & 1)) {
                        tc::mbar_arrive(&bars.wfull[s]);  // its chunk's weights are there
                    } else if (!RES) {
                        tc::mbar_arrive_expect_tx(&bars.wfull[s], C::kB);
                        tc::bulk_g2s(As + C::kA,
                                     reinterpret_cast<const unsigned char *>(a.wpack) +
                                         static_cast<size_t>(c) * C::kB,
                                     C::kB, &bars.wfull[s]);
                    }
                    if (skip) {
                        tc::mbar_arrive_expect_tx(&bars.full[s], kPitch * (TR + 2) * 32);
                        tma_load_halo(st & 1 ? &dmap : &emap, As, &bars.full[s], xc0 - 1, y0 - 1, c, b);
                    } else {
                        tc::mbar_arrive_expect_tx(&bars.full[s], kUpBytes);
                        tma_load_halo(&umap, As, &bars.full[s], xc0 - 1, y0 / 2 - 1, c - kc0, b);
                    }
                }
            }
            // wait (bounded, ignoring the abort flag) for the copies in flight, as in
            // conv3x3_kernel
            for (uint32_t k = it > NS ? it - NS : 0; k < it; ++k) {
                (void)tc::mbar_wait(&bars.full[k % NS], (k / NS) & 1u, nullptr);
                if (!RES) (void)tc::mbar_wait(&bars.wfull[k % NS], (k / NS) & 1u, nullptr);
            }
            if (RES && static_cast<int>(blockIdx.x) < ntiles)
                (void)tc::mbar_wait(&bars.wfull[0], 0, nullptr);
        }
        __syncwarp();
    } else if (warp == 8) {
        // -------------------------------------------------------- MMA issuer
        {
            // warp-uniform, as in conv3x3_kernel
            const uint32_t lead = tc::elect_one();
            auto wait = [&](uint64_t *bar, uint32_t parity) {
                return tc::mbar_wait_warp(bar, parity, abort_flag);
            };
            uint32_t it = 0, tl = 0;
            bool ok = true, pending = false;
            if (RES && static_cast<int>(blockIdx.x) < ntiles && !wait(&bars.wfull[0], 0)) {
                fail();
                ok = false;
            }
            for (int t = blockIdx.x; t < ntiles && ok; t += gridDim.x, ++tl) {
                const int acc = kSets == 2 ? tl & 1 : 0;
                const uint32_t free_parity = ((tl / kSets) & 1u) ^ 1u;
                const uint32_t d0 = tmem + acc * 2 * kPhase;
                // resets the accumulators of a phase, once the epilogue that reads them
                // (of both phases with two sets) is through with them
                auto begin = [&](int phase) {
                    if (!wait(&bars.acce[kSets == 2 ? acc : phase], free_parity))
                        return false;
                    tc::tc_fence_after();
                    pending = true;
                    const uint64_t zd =
                        tc::smem_desc(tc::smem_u32(base + C::kZeroOff), C::kZeroRows * 16, 128);
                    tc::mma_bf16(d0 + phase * kPhase, zd, zd, tc::idesc_bf16_f32(128, kPhase), 0u,
                                 lead);
                    return true;
                };
                if (!begin(0) || (kSets == 2 && !begin(1))) {
                    fail();
                    ok = false;
                    break;
                }
                for (int c = 0; c < kchunks; ++c) {
                    // the two stages of a skip chunk (its even and odd columns; the
                    // first brings the weights) or the one of an upsampled chunk
                    const bool skip = c < kc0;
                    const int s = static_cast<int>(it % NS);
                    const uint32_t ph = (it / NS) & 1u;
                    const int s1 = static_cast<int>((it + 1) % NS);
                    if (!wait(&bars.full[s], ph) || (!RES && !wait(&bars.wfull[s], ph)) ||
                        (skip && !wait(&bars.full[s1], ((it + 1) / NS) & 1u))) {
                        fail();
                        ok = false;
                        break;
                    }
                    tc::tc_fence_after();
                    const uint32_t a_base = tc::smem_u32(stages + s * C::kStage);
                    const uint64_t even = tc::smem_desc_sw32(a_base);
                    const uint64_t odd = tc::smem_desc_sw32(tc::smem_u32(stages + s1 * C::kStage));
                    const uint64_t b_desc =
                        tc::smem_desc(RES ? tc::smem_u32(wres + c * C::kB) : a_base + C::kA,
                                      3 * N * 16, 128);
                    // tap dx of a phase from the staged columns starting at `col`
                    // (0: xc0 - 1); rows as in conv3x3_kernel
                    auto taps = [&](int phase, int dx, uint64_t rows, int col, bool up) {
#pragma unroll
                        for (int h = 0; h < TR + 2; ++h) {
                            const int rlo = h - 2 < 0 ? 0 : h - 2;
                            const int rhi = h < TR - 1 ? h : TR - 1;
                            const int k0 = rlo - (h - 2);
                            const int row = up ? (h + 1) >> 1 : h;
                            tc::mma_bf16(d0 + phase * kPhase + rlo * N,
                                         rows + tc::desc_offset((row * kPitch + col) * 32),
                                         b_desc + tc::desc_offset((dx * 6 + k0) * N * 16),
                                         tc::idesc_bf16_f32(128, (rhi - rlo + 1) * N), 1u, lead);
                        }
                    };
                    // dx = 0, 1, 2 for each phase, as in conv3x3_kernel: the same sums
                    if (skip) {
                        taps(0, 0, odd, 0, false);
                        taps(0, 1, even, 1, false);
                        taps(0, 2, odd, 1, false);
                    } else {
                        taps(0, 0, even, 0, true);
                        taps(0, 1, even, 1, true);
                        taps(0, 2, even, 1, true);
                    }
                    if (kSets == 1 && c == kchunks - 1) tc::mma_commit(&bars.accf[0], lead);
                    if (kSets == 1 && c == 0 && !begin(1)) {
                        fail();
                        ok = false;
                        break;
                    }
                    if (skip) {
                        taps(1, 0, even, 1, false);
                        taps(1, 1, odd, 1, false);
                        taps(1, 2, even, 2, false);
                    } else {
                        taps(1, 0, even, 1, true);
                        taps(1, 1, even, 1, true);
                        taps(1, 2, even, 2, true);
                    }
                    tc::mma_commit(&bars.empty[s], lead);
                    if (skip) tc::mma_commit(&bars.empty[s1], lead);
                    it += skip ? 2 : 1;
                }
                if (!ok) break;
                tc::mma_commit(&bars.accf[kSets == 2 ? acc : 1], lead);
            }
            if (pending) {
                tc::mma_commit(&bars.drain, lead);
                (void)tc::mbar_wait(&bars.drain, 0, nullptr);
            }
        }
        __syncwarp();
    } else {
        // ----------------------------------------------------------- epilogue
        const int sub = warp & 3, phase = warp >> 2;
        const CUtensorMap *omap = phase ? &omap1 : &omap0;
        constexpr int kCB = C::kCBs, kW = kCB / 2;
        static_assert(kCB == 32, "64-byte slots");
        constexpr int kRowBlocks = N / kCB, kBlocks = TR * kRowBlocks;
        unsigned char *slots = base + C::kStoreOff + warp * 2 * C::kSlot;
        const uint32_t swz = (lane >> 1) & 3;
        const uint32_t lane_base = static_cast<uint32_t>(sub * 32) << 16;
        const int Wc = a.W >> 1;
        uint32_t tl = 0, eblk = 0;
        for (int t = blockIdx.x; t < ntiles; t += gridDim.x, ++tl) {
            const int acc = kSets == 2 ? tl & 1 : 0;
            const int b = t / per_img, r = t - b * per_img;
            const int y0 = (r / tiles_x) * TR, xw = (r % tiles_x) * kTileX + sub * 32;
            const int bar = kSets == 2 ? acc : phase;
            if (!tc::mbar_wait_warp(&bars.accf[bar], (tl / kSets) & 1u, abort_flag)) {
                fail();
                break;
            }
            tc::tc_fence_after();
            const uint32_t abase = tmem + lane_base + (acc * 2 + phase) * kPhase;
            auto tmem_read = [&](int k, uint32_t (&v)[kCB]) {
#pragma unroll
                for (int q = 0; q < kCB / 16; ++q)
                    tc::tmem_ld16(abase + (k / kRowBlocks) * N + (k % kRowBlocks) * kCB + 16 * q,
                                  *reinterpret_cast<uint32_t(*)[16]>(v + 16 * q));
            };
            uint32_t vbuf[2][kCB];
            tmem_read(0, vbuf[0]);
            tc::tmem_wait_ld();
#pragma unroll
            for (int k = 0; k < kBlocks; ++k) {
                if (k + 1 < kBlocks) tmem_read(k + 1, vbuf[(k + 1) & 1]);
                const uint32_t (&v)[kCB] = vbuf[k & 1];
                const int y = y0 + k / kRowBlocks, j0 = (k % kRowBlocks) * kCB;
                uint32_t w[kW];
#pragma unroll
                for (int e = 0; e < kCB; e += 2) {
                    const float2 bb = *reinterpret_cast<const float2 *>(sbias + j0 + e);
                    const float2 f =
                        add2(make_float2(__uint_as_float(v[e]), __uint_as_float(v[e + 1])), bb);
                    w[e / 2] = pack_bf16x2(f.x, f.y);
                    if (a.epi_mode == kEpiReluBF16) w[e / 2] = relu_bf16x2(w[e / 2]);
                }
                unsigned char *slot = slots + (eblk & 1) * C::kSlot;
                if (lane == 0) tma_store_wait_read<1>();  // the slot's previous store
                __syncwarp();
                uint4 *row = reinterpret_cast<uint4 *>(slot + lane * 2 * kCB);
#pragma unroll
                for (int q = 0; q < kW / 4; ++q)
                    row[q ^ swz] = make_uint4(w[4 * q], w[4 * q + 1], w[4 * q + 2], w[4 * q + 3]);
                tc::fence_proxy_async();
                __syncwarp();
                if (lane == 0) {
                    if (y < a.H && xw < Wc) tma_store_nhwc(omap, slot, j0, xw, y, b);
                    tma_store_commit();
                }
                ++eblk;
                tc::tmem_wait_ld();
            }
            tc::tc_fence_before();
            tc::mbar_arrive(&bars.acce[bar]);
        }
        if (lane == 0 && eblk) tma_store_wait_all();
    }

    tc::tc_fence_before();
    __syncthreads();
    if (warp == 8) {
        tc::tc_fence_after();
        tc::tmem_dealloc(tmem, kCols);
    }
}

// Launches conv3x3_up_kernel where it applies and pays; false: not launched.
template <int N, bool RES>
bool launch_up(const ConvArgs &a, cudaStream_t stream, int *rc) {
    using C = Cfg<N, RES>;
    // The rounds of tiles per SM decide: padding columns and a last round that is
    // nearly empty can cost more than the expansion.  A round of tiles of 256 columns
    // takes 1.23 to 1.30 (N = 32) or 1.49 to 1.58 (N = 64) times a round of 128 columns
    // of the expanding kernel (both kernels on the network's layers at 3840 x 2160,
    // 1920 x 1080, 1368 x 768, 1280 x 720 and 640 x 360: 360 us in 54 rounds against
    // 554 us in 107 at N = 32, 289 us in 15 against 329 us in 27 at N = 64).  The line
    // asks for 1.5 and 1.78 times the rounds, a margin of about an eighth.
    const int64_t rows = static_cast<int64_t>(a.B) * ((a.H + C::TR - 1) / C::TR), sms = sm_count();
    const int64_t ntiles = rows * ((a.W + 2 * kTileX - 1) / (2 * kTileX));
    const int64_t rounds = (ntiles + sms - 1) / sms;
    const int64_t rounds128 = (rows * ((a.W + kTileX - 1) / kTileX) + sms - 1) / sms;
    if (a.src_mode != kSrcConcatUp || a.pool_out ||
        (a.epi_mode != kEpiReluBF16 && a.epi_mode != kEpiBF16) || a.W % 2 || a.H % 2 ||
        a.c0 % 16 || a.c1 % 16 || a.c0 <= 0 || a.c1 <= 0 || a.cin_pad != a.c0 + a.c1 ||
        ntiles <= 0 || ntiles > 0x7fffffff || getenv_disable_tma_in() ||
        (N == 32 ? 3 * rounds > 2 * rounds128 : 16 * rounds > 9 * rounds128))
        return false;
    auto enc = tensor_map_encoder();
    if (!enc) return false;
    const cuuint64_t Wc = a.W / 2, H = a.H, B = a.B, c0 = a.c0, c1 = a.c1;
    cuuint32_t estr[5] = {1, 1, 1, 1, 1};
    CUtensorMap omap[2], smap[2], umap;
    for (int p = 0; p < 2; ++p) {
        // output columns 2 x + p, a block of 32 of them and 32 channels
        cuuint64_t dims[4] = {static_cast<cuuint64_t>(N), Wc, H, B};
        cuuint64_t strides[3] = {4ull * N, 4ull * N * Wc, 4ull * N * Wc * H};
        cuuint32_t box[4] = {32, 32, 1, 1};
        if (enc(&omap[p], CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, a.out + p * N, dims, strides, box, estr,
                CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B,
                CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return false;
        // skip columns 2 x + p: (channel in chunk, x, y, 16-channel chunk, image)
        cuuint64_t sdims[5] = {16, Wc, H, c0 / 16, B};
        cuuint64_t sstr[4] = {4 * c0, 4 * c0 * Wc, 32, 4 * c0 * Wc * H};
        cuuint32_t sbox[5] = {16, kPitch, C::TR + 2, 1, 1};
        if (enc(&smap[p], CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5,
                const_cast<__nv_bfloat16 *>(a.src0 + p * c0), sdims, sstr, sbox, estr,
                CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_32B,
                CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return false;
    }
    cuuint64_t udims[5] = {16, Wc, H / 2, c1 / 16, B};
    cuuint64_t ustr[4] = {2 * c1, 2 * c1 * Wc, 32, 2 * c1 * Wc * (H / 2)};
    cuuint32_t ubox[5] = {16, kPitch, C::TR / 2 + 2, 1, 1};
    if (enc(&umap, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, const_cast<__nv_bfloat16 *>(a.src1), udims,
            ustr, ubox, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_32B,
            CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
        return false;
    static int configured_dev = -1;
    int dev = 0;
    cudaGetDevice(&dev);
    if (configured_dev != dev) {
        if (cudaFuncSetAttribute(conv3x3_up_kernel<N, RES>,
                                 cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 C::kSmem) != cudaSuccess) {
            *rc = SPP_ERR_CUDA;
            return true;
        }
        configured_dev = dev;
    }
    const int grid = static_cast<int>(std::min(ntiles, sms));
    launch_dependent(conv3x3_up_kernel<N, RES>, dim3(grid), dim3(kThreads), C::kSmem, stream, a,
                     omap[0], omap[1], smap[0], smap[1], umap);
    count_launch();
    *rc = launch_status();
    return true;
}

template <int N, bool RES>
int launch_variant(const ConvArgs &a, cudaStream_t stream) {
    using C = Cfg<N, RES>;
    if constexpr (C::kStack) {
        int rc;
        if (launch_up<N, RES>(a, stream, &rc)) return rc;
    }
    static int configured_dev = -1;
    int dev = 0;
    cudaGetDevice(&dev);
    if (configured_dev != dev) {
        if (cudaFuncSetAttribute(conv3x3_kernel<N, RES>,
                                 cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 C::kUpFits ? C::kSmemUp : C::kSmem) != cudaSuccess)
            return SPP_ERR_CUDA;
        configured_dev = dev;
    }
    const int64_t ntiles = static_cast<int64_t>(a.B) * ((a.H + C::TR - 1) / C::TR) *
                           ((a.W + kTileX - 1) / kTileX);
    if (ntiles == 0) return SPP_OK;
    const int grid = static_cast<int>(std::min<int64_t>(ntiles, sm_count()));
    CUtensorMap omap;
    memset(&omap, 0, sizeof(omap));
    ConvArgs b = a;
    b.tma_out = 0;
    if (RES && a.epi_mode == kEpiF32Planar && a.W % 4 == 0) {
        // [B][cout][H][W] FP32 as a 4-D tensor (x, y, plane, image), box 128 x 1 x 16 x 1
        auto enc = tensor_map_encoder();
        cuuint64_t dims[4] = {static_cast<cuuint64_t>(a.W), static_cast<cuuint64_t>(a.H),
                              static_cast<cuuint64_t>(a.cout), static_cast<cuuint64_t>(a.B)};
        cuuint64_t strides[3] = {static_cast<cuuint64_t>(a.W) * 4ull,
                                 static_cast<cuuint64_t>(a.W) * a.H * 4ull,
                                 static_cast<cuuint64_t>(a.W) * a.H * a.cout * 4ull};
        cuuint32_t box[4] = {32, 1, static_cast<cuuint32_t>(N >= 32 ? 32 : 16), 1};
        cuuint32_t estr[4] = {1, 1, 1, 1};
        if (enc && enc(&omap, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, a.outf, dims, strides, box, estr,
                       CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                       CU_TENSOR_MAP_L2_PROMOTION_NONE,
                       CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS)
            b.tma_out = 1;
    }
    if (a.epi_mode != kEpiF32Planar) {
        // BF16 NHWC [B][H][W][N] as (channel, x, y, image), box kCBs x 32 x 1 x 1
        auto enc = tensor_map_encoder();
        cuuint64_t dims[4] = {static_cast<cuuint64_t>(N), static_cast<cuuint64_t>(a.W),
                              static_cast<cuuint64_t>(a.H), static_cast<cuuint64_t>(a.B)};
        cuuint64_t strides[3] = {static_cast<cuuint64_t>(N) * 2,
                                 static_cast<cuuint64_t>(a.W) * N * 2,
                                 static_cast<cuuint64_t>(a.W) * a.H * N * 2};
        cuuint32_t box[4] = {static_cast<cuuint32_t>(C::kCBs), 32, 1, 1};
        cuuint32_t estr[4] = {1, 1, 1, 1};
        if (!enc || enc(&omap, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, a.out, dims, strides, box, estr,
                        CU_TENSOR_MAP_INTERLEAVE_NONE,
                        C::kCBs == 32 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_32B,
                        CU_TENSOR_MAP_L2_PROMOTION_NONE,
                        CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return SPP_ERR_CUDA;
    }
    CUtensorMap imap;
    memset(&imap, 0, sizeof(imap));
    b.tma_in = 0;
    if ((a.src_mode == kSrcNHWC || a.src_mode == kSrcConcatUp) && a.c0 % 16 == 0 &&
        !getenv_disable_tma_in()) {
        // NHWC BF16 [B][H][W][c0] as 5-D (channel in chunk, x, y, 16-channel chunk,
        // image); box 16 x 130 x (TR+2) x 1 x 1 = one K chunk of the halo, written
        // with the 32-byte swizzle of the A operand (32-byte pieces: about twice
        // the TMA throughput of 16-byte ones)
        auto enc = tensor_map_encoder();
        cuuint64_t dims[5] = {16, static_cast<cuuint64_t>(a.W), static_cast<cuuint64_t>(a.H),
                              static_cast<cuuint64_t>(a.c0 / 16), static_cast<cuuint64_t>(a.B)};
        cuuint64_t strides[4] = {static_cast<cuuint64_t>(a.c0) * 2,
                                 static_cast<cuuint64_t>(a.W) * a.c0 * 2, 32,
                                 static_cast<cuuint64_t>(a.H) * a.W * a.c0 * 2};
        cuuint32_t box[5] = {16, static_cast<cuuint32_t>(kPitch), static_cast<cuuint32_t>(C::TR + 2),
                             1, 1};
        cuuint32_t estr[5] = {1, 1, 1, 1, 1};
        if (enc && enc(&imap, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, const_cast<__nv_bfloat16 *>(a.src0),
                       dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                       CU_TENSOR_MAP_SWIZZLE_32B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                       CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS)
            b.tma_in = a.src_mode == kSrcNHWC ? 1 : 2;
    }
    CUtensorMap umap;
    memset(&umap, 0, sizeof(umap));
    if (b.tma_in == 2 && C::kUpFits && a.epi_mode != kEpiF32Planar && a.c1 % 16 == 0 && a.c1 > 0 && a.W % 2 == 0 &&
        a.H % 2 == 0) {
        // the coarse source [B][H/2][W/2][c1] as 5-D (channel in chunk, x, y,
        // 16-channel chunk, image); box 16 x kUpW x kUpRows x 1 x 1 = one K chunk of
        // the coarse rows under a tile's halo
        auto enc = tensor_map_encoder();
        const int Wc = a.W / 2, Hc = a.H / 2;
        cuuint64_t dims[5] = {16, static_cast<cuuint64_t>(Wc), static_cast<cuuint64_t>(Hc),
                              static_cast<cuuint64_t>(a.c1 / 16), static_cast<cuuint64_t>(a.B)};
        cuuint64_t strides[4] = {static_cast<cuuint64_t>(a.c1) * 2,
                                 static_cast<cuuint64_t>(Wc) * a.c1 * 2, 32,
                                 static_cast<cuuint64_t>(Hc) * Wc * a.c1 * 2};
        cuuint32_t box[5] = {16, static_cast<cuuint32_t>(kUpW), static_cast<cuuint32_t>(C::kUpRows),
                             1, 1};
        cuuint32_t estr[5] = {1, 1, 1, 1, 1};
        if (enc && enc(&umap, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, const_cast<__nv_bfloat16 *>(a.src1),
                       dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                       CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                       CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS)
            b.tma_in = 3;
    }
    launch_dependent(conv3x3_kernel<N, RES>, dim3(grid), dim3(kThreads),
                     b.tma_in == 3 ? C::kSmemUp : C::kSmem, stream, b, omap, imap, umap);
    count_launch();
    return launch_status();
}

template <int N>
int launch(const ConvArgs &a, cudaStream_t stream) {
    const int64_t wbytes = static_cast<int64_t>(a.cin_pad / 16) * Cfg<N, false>::kB;
    // N = 192 (data gradients of the 192-channel decoder input) always streams:
    // its weights exceed the resident region at every cin_pad above 16
    if constexpr (N != 192) {
        if (wbytes <= kResidentMax) return launch_variant<N, true>(a, stream);
    }
    return launch_variant<N, false>(a, stream);
}

}  // namespace

int pack_weights(PackTable &table, cudaStream_t stream) {
    int blocks = 0;
    for (int i = 0; i < table.count; ++i) {
        PackItem &it = table.it[i];
        it.first_block = blocks;
        blocks += std::max(1, (it.cin_pad / 16 * 18 * it.n + kPackThreads - 1) / kPackThreads);
    }
    if (blocks == 0) return SPP_OK;
    pack_weights_kernel<<<blocks, kPackThreads, 0, stream>>>(table);
    count_launch();
    return launch_status();
}

int pack_weights(const float *w, int cin, int cout, int transpose, int cin_pad, int n,
                 __nv_bfloat16 *dst, cudaStream_t stream) {
    PackTable table;
    table.count = 1;
    table.it[0] = PackItem{w, dst, nullptr, nullptr, cin, cout, transpose, cin_pad, n, 0};
    return pack_weights(table, stream);
}

int conv3x3(const ConvArgs &a, cudaStream_t stream) {
    if (a.B < 0 || a.H < 0 || a.W < 0 || a.cin_pad <= 0 || a.cin_pad % 16 || !supported_n(a.n))
        return SPP_ERR_ARG;
    if (!a.wpack || !aligned16(a.wpack)) return SPP_ERR_ALIGN;
    switch (a.n) {
        case 16: return launch<16>(a, stream);
        case 32: return launch<32>(a, stream);
        case 64: return launch<64>(a, stream);
        case 96: return launch<96>(a, stream);
        case 128: return launch<128>(a, stream);
        default: return launch<192>(a, stream);
    }
}

}  // namespace conv
}  // namespace spp
