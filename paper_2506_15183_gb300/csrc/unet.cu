// The learned hole inpainter on the tensor cores (sm_103a): a 4-level U-Net over
// 64 x 64 tiles, BF16 weights and activations, FP32 accumulation.
//
// Each 3x3 convolution is an implicit GEMM: M = output pixels (128 per accumulator), N =
// output channels (32..256, or a part of them on small grids), K = taps x input channels,
// taken 32 or 64 channels (64 or 128 bytes: the swizzle span) at a time.  Operands are TMA
// tiled loads into shared memory, swizzled by the copy engine (the zero padding of the
// convolution is the part of a box outside the tensor, which TMA fills with zeros); one thread
// each issues the activation and the weight copies, one warp the tcgen05.mma (kind::f16, BF16
// operands, FP32 accumulator in tensor memory, K = 16), with mbarriers between them.  The
// epilogue reads the accumulators with tcgen05.ld, adds the bias, applies ReLU, rounds to BF16
// and stores NHWC at a channel offset of a wider buffer (so a concatenation is written in
// place), or, for the layer below a decoder level, to the 2 x 2 pixels of the nearest
// upsampling.  Three forms:
//   - conv3x3_rows (conv_rows.cu), for 32 or 64 output channels on tiles 32 to 128 pixels
//     wide: one image row per accumulator, the three taps of a kernel column in one MMA.
//   - conv3x3_halo, for the other tiles of whole rows of one image: a band of 128 or 256 pixels
//     goes into one or two accumulators (each CTA walks bands blockIdx.x, + gridDim.x, ..., as
//     many CTAs as fit on the SMs at once); a K step is one (32-channel block, dx) pair, a single
//     box of the band's R rows plus one above and below, shared by the three dy taps through the
//     start address of the MMA operand (whole 512-byte swizzle atoms apart), and one box of the
//     three taps' weights.  Each input pixel is copied 3 (R + 2) / R times instead of 9.
//   - conv3x3_tc, one CTA per one or two 128-pixel tiles (the 8 x 8 level, where 128 pixels are
//     two images, and 256 output channels): a K step is one (block of 32 or 64 channels, tap),
//     the activation boxes {channels, W, rows, images} at the tap's offset and the weight box
//     {channels, the CTA's output channels} of the K-major weights (k = tap * Cin + ci).
// The last two use CTAs of 128 threads and rings of up to 12 stages: two, and several CTAs per SM,
// where there are enough of them that the copies of one overlap the set-up, MMAs and
// epilogue of the others; deeper where a CTA has its SM to itself.
//
// Every wait on an mbarrier has a deadline (1 s of %globaltimer): a wait that runs out
// records kUnetTimeout in a status word, the kernel waits (again bounded) for the copies
// it issued, frees its tensor memory and returns.  Nothing traps.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <new>
#include <vector>

#include "ring.h"
#include "tc.cuh"
#include "unet_device.cuh"
#include "unet_internal.h"
#include "yoro.h"
#include "yoro_internal.h"
#include "yoro_unet.h"

namespace yoro {

namespace {

__device__ unsigned g_unet_status;  // kernel-side failures of this file's kernels

constexpr int kMaxStages = 12;

struct ConvArgs {
    int T, H, W;          // tiles and their size (the output has the input's size)
    int Cin, Cout;        // Cin: channels of the input tensor, a multiple of 32
    int bn;               // output channels of a CTA: Cout, or a part of it (blockIdx.y) on small grids
    const float* bias;    // Cout
    int y_coff;           // first output channel in y (the output's tensor map)
    int upsample;         // 1: pixel (yy, xx) goes to (2yy + a, 2xx + b), a, b in {0, 1}
    int relu;
    int ncols;            // tensor-memory columns allocated (a power of two >= mt bn, >= 32)
    const int* count;     // optional: tiles at or after *count are skipped (the tile list's length)
    uint16_t* pool;       // optional (16-pixel rows only): T x H/2 x W/2 x Cout, the 2x2 maximum of the output
    int mt, stages;       // 128-pixel accumulators per CTA (halo form) and copy stages
};

// The epilogue of both forms: the CTA's mt accumulators of 128 pixels (pixel i of
// accumulator j is the CTA tile's pixel 128 j + i, row-major over its rows) are read
// back 32 channels at a time, the bias added, ReLU applied, rounded to BF16 and staged in
// shared memory (`stg`, 1024-aligned: the copy stages, free once every MMA has
// completed), one slice of 64 bytes per pixel for each 32 channels, in the 64-byte
// swizzle (bias: the CTA's bn values; 16-byte chunk k of pixel p at p 64 + (k ^ (p / 2 mod 4)) 16, so a warp's
// writes meet no bank twice).  One thread then writes every slice with TMA tensor
// stores: a box {32 channels, W, rows, images} at channel y_coff + 32 s, or, for the
// nearest upsampling, the same box four times through a 5-D view of the output that
// splits each coordinate into (pixel, replica).  The CTA ends once the stores have read
// shared memory.
__device__ __forceinline__ void epilogue_store(const ConvArgs& a, const CUtensorMap* tmY, uint32_t tmem,
                                               unsigned char* stg, const float* bias, int mt, int n0, int y0)
{
    const int nb = blockIdx.y * a.bn;  // the CTA's first output channel
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int m = warp * 32 + lane;  // this thread's pixel of each accumulator = its TMEM lane
    const int slice = mt * kTileM * 64;
    for (int c0 = 0; c0 < a.bn; c0 += 32) {
        unsigned char* sl = stg + (c0 >> 5) * slice;
        for (int j = 0; j < mt; ++j) {
            uint32_t r[32];
            tmem_ld32(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)(j * a.bn + c0), r);
            uint4 q[4];
            uint32_t* qw = reinterpret_cast<uint32_t*>(q);
#pragma unroll
            for (int i = 0; i < 16; ++i) {
                float v0 = __fadd_rn(__uint_as_float(r[2 * i]), bias[c0 + 2 * i]);
                float v1 = __fadd_rn(__uint_as_float(r[2 * i + 1]), bias[c0 + 2 * i + 1]);
                if (a.relu) {
                    v0 = fmaxf(v0, 0.0f);
                    v1 = fmaxf(v1, 0.0f);
                }
                qw[i] = pack_bf16x2(v0, v1);
            }
            const int px = j * kTileM + m;
            unsigned char* row = sl + px * 64;
            const int sw = (px >> 1) & 3;
#pragma unroll
            for (int k = 0; k < 4; ++k) *reinterpret_cast<uint4*>(row + ((k ^ sw) << 4)) = q[k];
            // 16-pixel rows: a warp holds two of them; the 2x2 maximum of its pixels
            if (a.pool) {
#pragma unroll
                for (int i = 0; i < 16; ++i) {
                    qw[i] = max_bf16x2(qw[i], __shfl_xor_sync(0xffffffffu, qw[i], 16));
                    qw[i] = max_bf16x2(qw[i], __shfl_xor_sync(0xffffffffu, qw[i], 1));
                }
                const int yy = y0 + ((j * kTileM + warp * 32) >> 4);  // the first of its rows
                const size_t pp = ((size_t)n0 * (a.H >> 1) + (yy >> 1)) * 8 + ((lane & 15) >> 1);
                // the four lanes of a pooled pixel write 16 bytes each
                const int k = (lane & 1) + 2 * (lane >> 4);
                reinterpret_cast<uint4*>(a.pool + pp * a.Cout + nb + c0)[k] =
                    k == 0 ? q[0] : k == 1 ? q[1] : k == 2 ? q[2] : q[3];
            }
        }
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // the writes, seen by the copy engine
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int c0 = 0; c0 < a.bn; c0 += 32) {
            const unsigned char* sl = stg + (c0 >> 5) * slice;
            if (!a.upsample) {
                tma_store_4d(tmY, sl, a.y_coff + nb + c0, 0, y0, n0);
            } else {
#pragma unroll
                for (int ab = 0; ab < 4; ++ab) tma_store_5d(tmY, sl, a.y_coff + nb + c0, ab & 1, 0, ab >> 1, n0 * a.H + y0);
            }
        }
        asm volatile("cp.async.bulk.commit_group;" ::: "memory");
        asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
    }
}

// The one-tile form: MT tiles of 128 consecutive pixels (whole images where an image is
// smaller), a K step being KC channels of one tap.  The activation boxes and the weight box of
// a step are issued by two threads (warps 0 and 2): an issue costs a thread about 300 cycles
// plus 100 per copy whatever its size, so one thread with two copies of 32 channels per step
// was the pace of small grids (690 cycles a step).  With 64 channels a step (128-byte
// swizzle) half as many are needed.  The sums keep their order (tap, channel).
//
// MT = 2 for grids of two tiles per SM and more: both tiles use the weights of one copy (256
// channels: 64 instead of 96 bytes per cycle from L2, which 128-pixel CTAs were bound by).
//
// Measured (KC = 32, MT = 1, one issuing thread -> this): enc3b on 8 tiles 26.5 -> 15.6 us, on
// 870 89 -> 76; enc3a 15.0 -> 9.2 us on 8 tiles, 43 on 870 before and after.
template <int KC, int MT>
__global__ void __launch_bounds__(128, 1)
    conv3x3_tc(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
               const __grid_constant__ CUtensorMap tmY, const ConvArgs a)
{
    extern __shared__ unsigned char smem_raw[];
    const int hw = a.H * a.W;
    const int p0 = blockIdx.x * MT * kTileM;
    if (a.count && p0 / hw >= *a.count) return;  // no such tile (uniform)
    unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                                           ~static_cast<uintptr_t>(1023));
    constexpr int kA = kTileM * KC * 2;  // one tile's activation box
    const int S = a.stages, nb = blockIdx.y * a.bn;
    const int b_bytes = a.bn * KC * 2;
    const int stage_bytes = MT * kA + b_bytes;
    uint64_t* full = reinterpret_cast<uint64_t*>(smem + S * stage_bytes);
    uint64_t* empty = full + S;
    uint64_t* done = empty + S;
    uint32_t* tslot = reinterpret_cast<uint32_t*>(done + 1);
    // steps issued by warp 0 (activations), consumed, issued by warp 2 (weights)
    volatile int* counts = reinterpret_cast<volatile int*>(tslot + 1);
    const int warp = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0), lane = threadIdx.x & 31;

    if (threadIdx.x == 0) {
        for (int s = 0; s < S; ++s) {
            mbar_init(&full[s], 2);
            mbar_init(&empty[s], 1);
        }
        mbar_init(done, 1);
        counts[0] = 0;
        counts[1] = 0;
        counts[2] = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tslot)),
                     "r"(a.ncols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    pdl_wait();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tslot;

    const int cb_n = a.Cin / KC;
    const int nk = 9 * cb_n;
    const uint64_t deadline = globaltimer() + kWaitNs;

    if ((warp == 0 || warp == 2) && lane == 0) {  // copies: activations, weights
        int s = 0, ph = 1, tap = 0, cb = 0;
        for (int k = 0; k < nk; ++k) {
            if (!mbar_wait(&empty[s], ph, deadline)) {
                atomicOr(&g_unet_status, kUnetTimeout);
                break;
            }
            unsigned char* sa = smem + s * stage_bytes;
            if (warp == 0) {
                const int dy = tap / 3, dx = tap - 3 * dy;
                mbar_expect_tx(&full[s], (uint32_t)(MT * kA));
#pragma unroll
                for (int j = 0; j < MT; ++j) {  // a tile past the last image arrives as zeros
                    const int p = p0 + j * kTileM, n = p / hw, y = (p - n * hw) / a.W;
                    tma_load_4d(sa + j * kA, &tmA, &full[s], cb * KC, dx - 1, y + dy - 1, n);
                }
                counts[0] = k + 1;
            } else {
                mbar_expect_tx(&full[s], (uint32_t)b_bytes);
                tma_load_2d(sa + MT * kA, &tmB, &full[s], tap * a.Cin + cb * KC, nb);
                counts[2] = k + 1;
            }
            if (++cb == cb_n) {
                cb = 0;
                ++tap;
            }
            if (++s == S) {
                s = 0;
                ph ^= 1;
            }
        }
    } else if (warp == 1) {  // MMAs: the whole warp runs the loop, one lane issues
        const uint32_t idesc = idesc_bf16(a.bn), el = elect_one();
        const uint64_t dbase = KC == 64 ? desc_sw128(smem_u32(smem)) : desc_sw64(smem_u32(smem));
        int s = 0, ph = 0;
        for (int k = 0; k < nk; ++k) {
            if (!mbar_wait_warp(&full[s], ph, deadline)) {
                if (el) atomicOr(&g_unet_status, kUnetTimeout);
                break;
            }
            tc_fence_after();
            const uint64_t da = dbase + (uint64_t)((uint32_t)(s * stage_bytes) >> 4), db = da + (MT * kA >> 4);
#pragma unroll
            for (int q = 0; q < KC / 16; ++q)
#pragma unroll
                for (int j = 0; j < MT; ++j)
                    mma_bf16_elected(el, tmem + (uint32_t)(j * a.bn), da + (uint64_t)(j * (kA >> 4) + 2 * q),
                                     db + (uint64_t)(2 * q), idesc, k + q > 0 ? 1u : 0u);
            mma_commit_elected(el, &empty[s]);
            if (el) counts[1] = k + 1;
            if (++s == S) {
                s = 0;
                ph ^= 1;
            }
        }
        mma_commit_elected(el, done);  // arrives once every MMA issued above has completed
    }
    __syncwarp();

    const bool ok = mbar_wait(done, 0, deadline + kWaitNs);
    if (!ok) atomicOr(&g_unet_status, kUnetTimeout);
    if (ok) {
        tc_fence_after();
#pragma unroll
        for (int j = 0; j < MT; ++j) {
            const int p = p0 + j * kTileM, n = p / hw, y = (p - n * hw) / a.W;
            if (n < a.T)  // uniform
                epilogue_store(a, &tmY, tmem + (uint32_t)(j * a.bn), smem + j * (a.bn >> 5) * kTileM * 64, a.bias + nb, 1,
                               n, y);
        }
    }
    tc_fence_before();
    __syncthreads();
    if (threadIdx.x == 0 && counts[1] < nk) {  // copies still in flight after a timeout: wait for them (bounded)
        const uint64_t d2 = globaltimer() + kWaitNs;
        ring_drain(counts[1], counts[0], counts[2], [&](int k) { mbar_arrive(&full[k % S]); },
                   [&](int k) { mbar_wait(&full[k % S], (k / S) & 1, d2); });
    }
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(a.ncols) : "memory");
    }
}

// Halo form of the same convolution, for layers whose 128-pixel tile is whole rows of
// one image: a CTA computes R = mt 128 / W whole rows of one image into mt accumulators
// of 128 pixels (mt Cout tensor-memory columns).  A K step is one (channel block, dx)
// pair rather than one (channel block, tap): a single activation box of R + 2 rows x W
// pixels x 32 channels at column offset dx - 1 (rows y0 - 1 and y0 + R and columns -1 and
// W lie outside the image and arrive as zeros) and the three weight boxes of the taps
// (0, dx), (1, dx), (2, dx).  In NHWC the box is R + 2 rows of W pixels of 64 bytes, so
// the operand of tap dy for accumulator j is the same box read from pixel row j 128 +
// dy W: a start (j 128 + dy W) 64 bytes in, a whole number of 512-byte swizzle atoms
// for W a multiple of 8, and the three dy taps share one copy.  Activation bytes copied
// per output pixel: 3 (R + 2) / R boxes instead of 9; weight bytes: 1 / mt of the
// one-tile form.
__global__ void __launch_bounds__(128, 1)
    conv3x3_halo(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                 const __grid_constant__ CUtensorMap tmY, const ConvArgs a, int nbands)
{
    extern __shared__ unsigned char smem_raw[];
    const int mt = a.mt, S = a.stages;
    const int tile_px = mt * kTileM;
    const int R = tile_px / a.W;
    const int bands_per_tile = a.H / R;
    // bands of tiles at or after *count are skipped (the tile list's length)
    const int live = a.count ? min(nbands, *a.count * bands_per_tile) : nbands;
    if ((int)blockIdx.x >= live) return;  // uniform
    unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                                           ~static_cast<uintptr_t>(1023));
    const int a_bytes = (R + 2) * a.W * kKc * 2;
    const int a_span = (a_bytes + 1023) & ~1023;
    const int b_tap = a.bn * kKc * 2, nb = blockIdx.y * a.bn;
    const int stage_bytes = a_span + ((3 * b_tap + 1023) & ~1023);
    uint64_t* full = reinterpret_cast<uint64_t*>(smem + S * stage_bytes);
    uint64_t* empty = full + kMaxStages;
    uint64_t* done = empty + kMaxStages;
    uint32_t* tslot = reinterpret_cast<uint32_t*>(done + 1);
    // activation boxes issued, steps consumed, abort, weight boxes issued
    volatile int* counts = reinterpret_cast<volatile int*>(tslot + 1);
    float* sbias = reinterpret_cast<float*>(smem + S * stage_bytes + 1024);
    const int warp = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0), lane = threadIdx.x & 31;

    const int cb_n = a.Cin / kKc;
    const int nk = 3 * cb_n;  // K steps of a band: (channel block, dx)
    // K step kk of the CTA (band kk / nk of its walk, step kk % nk) into stage kk % S: the
    // activation box (issued by warp 0) and the three taps' weights (one box, warp 2)
    auto issue_a = [&](int kk, int n0, int y0) {
        const int s = kk % S, k = kk % nk, cb = k / 3, dx = k - 3 * cb;
        mbar_expect_tx(&full[s], (uint32_t)a_bytes);
        tma_load_4d(smem + s * stage_bytes, &tmA, &full[s], cb * kKc, dx - 1, y0 - 1, n0);
        counts[0] = kk + 1;
    };
    auto issue_b = [&](int kk) {
        const int s = kk % S, k = kk % nk, cb = k / 3, dx = k - 3 * cb;
        mbar_expect_tx(&full[s], (uint32_t)(3 * b_tap));
        tma_load_4d(smem + s * stage_bytes + a_span, &tmB, &full[s], cb * kKc, nb, 0, dx);
        counts[3] = kk + 1;
    };
    const int first = nk < S ? nk : S;  // copies issued before the CTA-wide barrier

    // The first copies start as soon as the barriers exist (their stages are free), while
    // warp 1 allocates the tensor memory and the bias is staged in shared memory.
    if (threadIdx.x == 0) {
        for (int s = 0; s < S; ++s) {
            mbar_init(&full[s], 2);
            mbar_init(&empty[s], 1);
        }
        mbar_init(done, 1);
        counts[0] = 0;
        counts[1] = 0;
        counts[2] = 0;
        counts[3] = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        pdl_wait();
        const int b0 = blockIdx.x, n0 = b0 / bands_per_tile, y0 = (b0 - n0 * bands_per_tile) * R;
        for (int k = 0; k < first; ++k) {
            issue_a(k, n0, y0);
            issue_b(k);
        }
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tslot)),
                     "r"(a.ncols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    for (int c = threadIdx.x; c < a.bn; c += blockDim.x) sbias[c] = __ldg(a.bias + nb + c);
    pdl_wait();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tslot;

    // The CTA walks bands blockIdx.x, + gridDim.x, ...: per band its K steps, then the
    // epilogue; the barriers' phases run on across bands (step kk of the walk), and the
    // accumulators are reused once every thread's reads of them are done.
    // Where a band's output fits one stage, the epilogue stages it in the stage of the
    // band's last K step, and the next band's first copy (into the other stage) is issued
    // by the MMA thread once that stage is free, so it lands during the last MMAs and the
    // epilogue.
    const bool early = mt * kTileM * a.bn * 2 <= stage_bytes && S >= 2;
    int it = 0;
    for (int band = blockIdx.x; band < live; band += gridDim.x, ++it) {
        const int n0 = band / bands_per_tile, y0 = (band - n0 * bands_per_tile) * R;
        const uint64_t deadline = globaltimer() + kWaitNs;
        if ((warp == 0 || warp == 2) && lane == 0) {  // copies: activations, weights
            for (int k = it == 0 ? first : (early ? 1 : 0); k < nk; ++k) {
                const int kk = it * nk + k, s = kk % S;
                if (!mbar_wait(&empty[s], ((kk / S) & 1) ^ 1, deadline)) {
                    atomicOr(&g_unet_status, kUnetTimeout);
                    counts[2] = 1;
                    break;
                }
                if (warp == 0) issue_a(kk, n0, y0);
                else issue_b(kk);
            }
        } else if (warp == 1) {  // MMAs: the whole warp runs the loop, one lane issues
            // Descriptors: a stage's bases plus constants in the 16-byte start-address
            // field (the smem window is below 256 KB, so the field never carries over).
            const uint32_t idesc = idesc_bf16(a.bn), el = elect_one();
            const uint64_t dbase = desc_sw64(smem_u32(smem));
            const uint32_t aW = (uint32_t)a.W * 4u, aT = (uint32_t)kTileM * 4u, bT = (uint32_t)b_tap >> 4;
            const uint32_t d1 = tmem + (uint32_t)a.bn;
            bool run = true;
            for (int k = 0; k < nk; ++k) {
                const int kk = it * nk + k, s = kk % S;
                if (!(run = mbar_wait_warp(&full[s], (kk / S) & 1, deadline))) {
                    if (el) {
                        atomicOr(&g_unet_status, kUnetTimeout);
                        counts[2] = 1;
                    }
                    break;
                }
                tc_fence_after();
                const uint64_t da = dbase + (uint64_t)((uint32_t)(s * stage_bytes) >> 4);
                const uint64_t db = da + (uint64_t)((uint32_t)a_span >> 4);
#pragma unroll
                for (int dy = 0; dy < 3; ++dy) {
                    const uint64_t bt = db + dy * bT;
                    const uint64_t a0 = da + dy * aW, a1 = a0 + aT;
                    const uint32_t acc = (k > 0 || dy > 0) ? 1u : 0u;
                    mma_bf16_elected(el, tmem, a0, bt, idesc, acc);
                    mma_bf16_elected(el, tmem, a0 + 2, bt + 2, idesc, 1u);
                    if (mt > 1) {  // uniform
                        mma_bf16_elected(el, d1, a1, bt, idesc, acc);
                        mma_bf16_elected(el, d1, a1 + 2, bt + 2, idesc, 1u);
                    }
                }
                mma_commit_elected(el, &empty[s]);
                if (el) counts[1] = kk + 1;
            }
            mma_commit_elected(el, done);  // arrives once every MMA issued above has completed
            // early: the next band's first copy, into the stage the second-to-last K step
            // frees, while this band's last MMAs run
            const int next = band + (int)gridDim.x;
            if (early && next < live && run && el) {
                const int kk = (it + 1) * nk, s = kk % S;
                const int n1 = next / bands_per_tile, y1 = (next - n1 * bands_per_tile) * R;
                if (mbar_wait(&empty[s], ((kk / S) & 1) ^ 1, deadline)) {
                    issue_a(kk, n1, y1);
                    issue_b(kk);
                } else {
                    atomicOr(&g_unet_status, kUnetTimeout);
                    counts[2] = 1;
                }
            }
        }
        __syncwarp();
        const bool ok = mbar_wait(done, it & 1, deadline + kWaitNs);
        if (!ok) {
            atomicOr(&g_unet_status, kUnetTimeout);
            counts[2] = 1;
        }
        __syncthreads();
        const bool go = ok && !counts[2];  // the same for every thread (read after the barrier)
        if (go) {
            tc_fence_after();
            // early: the stage of this band's last K step (its copies were consumed)
            unsigned char* stg = early ? smem + ((it * nk + nk - 1) % S) * stage_bytes : smem;
            epilogue_store(a, &tmY, tmem, stg, sbias, mt, n0, y0);
        }
        // every thread's reads of the accumulators are done before the next band's MMAs
        tc_fence_before();
        __syncthreads();
        tc_fence_after();
        if (!go) break;
    }
    __syncthreads();
    if (threadIdx.x == 0 && counts[2]) {  // copies still in flight after a timeout: wait for them (bounded)
        const uint64_t d2 = globaltimer() + kWaitNs;
        ring_drain(counts[1], counts[0], counts[3], [&](int k) { mbar_arrive(&full[k % S]); },
                   [&](int k) { mbar_wait(&full[k % S], (k / S) & 1, d2); });
    }
    __syncthreads();
    if (warp == 1) {  // the allocating warp frees
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(a.ncols) : "memory");
    }
}

}  // namespace

EncodeTiled tensor_map_encoder()
{
    static EncodeTiled fn = nullptr;
    if (!fn) {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) !=
                cudaSuccess ||
            q != cudaDriverEntryPointSuccess)
            return nullptr;
        fn = reinterpret_cast<EncodeTiled>(p);
    }
    return fn;
}

namespace {

// One-tile form: bytes of one copy stage, and of a CTA.
int conv_stage_bytes(int bn, int kc, int mt) { return (mt * kTileM + bn) * kc * 2; }

size_t conv_smem_bytes(int stage, int stages) { return 1024 + (size_t)stages * stage + (2 * stages + 1) * 8 + 16; }

// Output channels per CTA where `ctas` CTAs with all Cout would leave SMs idle: halved, down to
// 64 (an MMA takes 55 cycles at N = 64 and at N = 32), while twice as many CTAs still get an
// SM of their own.  Each part runs the same K steps (its sums
// are the same), but its copies are smaller, and a lone CTA's ring can be as deep as its SM's
// shared memory: on few tiles these layers wait for their copies.
int split_channels(int Cout, long long ctas, int sms)
{
    int bn = Cout;
    while (bn > 64 && 2 * ctas * (Cout / bn) <= sms) bn /= 2;
    return bn;
}

// Halo form: bytes of one copy stage (activation box of R + 2 rows, three weight boxes).
int halo_stage_bytes(int W, int rows, int cout)
{
    return ((((rows + 2) * W * kKc * 2) + 1023) & ~1023) + ((3 * cout * kKc * 2 + 1023) & ~1023);
}

// Halo form: the stages, then 1 KB of barriers and counters, then the bias (256 floats).
size_t halo_smem_bytes(int stage_bytes, int stages)
{
    return 1024 + (size_t)stages * stage_bytes + 1024 + 256 * 4;
}

// Shared memory a halo-form CTA of two stages may take: two CTAs share an SM (228 KB, 1 KB
// reserved per CTA).
constexpr int kHaloSmemBudget = 112 * 1024;

// The halo form's shape for a layer, or mt = 0 where the one-tile form runs: whole-row
// tiles of one image (W in 16..128), two accumulators of 128 pixels (R = 256 / W rows,
// a divisor of H), Cout <= 128 (2 Cout tensor-memory columns), two copy stages within
// the budget.  It also says which layers the row form may take.  At 128 output channels, which
// the halo form still runs, two accumulators with two stages (two CTAs per SM) measured
// fastest against one or four accumulators and two to four stages at one to four CTAs per SM:
// more CTAs per SM overlap one CTA's set-up, last MMAs and epilogue with the others' copies.
// unet_conv3x3 takes one accumulator and a deeper ring on grids that leave SMs idle.
void halo_shape(int H, int W, int Cout, int* mt, int* stages)
{
    *mt = 0;
    *stages = 0;
    if (W < 16 || W > kTileM || kTileM % W || Cout > 128) return;
    const int rows = 2 * kTileM / W;
    if (rows > H || H % rows) return;
    if (halo_smem_bytes(halo_stage_bytes(W, rows, Cout), 2) > (size_t)kHaloSmemBudget) return;
    if ((Cout / kKc) * 2 * kTileM * 64 > 2 * halo_stage_bytes(W, rows, Cout)) return;  // the epilogue's staging
    *mt = 2;
    *stages = 2;
}

}  // namespace

unsigned unet_status_take()
{
    unsigned v = 0, z = 0;
    if (cudaMemcpyFromSymbol(&v, g_unet_status, sizeof v) != cudaSuccess ||
        cudaMemcpyToSymbol(g_unet_status, &z, sizeof z) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return v | conv_rows_status_take() | conv_dw_status_take();
}

// One 3x3 convolution (zero padding 1) of x (T tiles of H x W, NHWC bf16 with Cin
// channels, Cin a multiple of 32) with K-major weights wk (Cout rows of 9 Cin, k = (3 dy +
// dx) Cin + ci) and bias, ReLU if relu, into y at channel offset y_coff of a tensor with
// y_cstride channels (upsample: into the 2H x 2W grid of the nearest upsampling).
// Shared memory of one SM (228 KB) and the SM count of the current device.
constexpr size_t kSmemPerSm = 228 * 1024;
constexpr int kSmemPerBlock = 227 * 1024;  // the most one CTA can take

int sm_count()
{
    static int n = 0;
    if (!n) {
        int dev = 0, v = 0;
        if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) !=
                                                      cudaSuccess || v < 1) {
            cudaGetLastError();
            return 148;
        }
        n = v;
    }
    return n;
}

// Needs T H W a multiple of 128, W in {8, 16, 32, 64, 128} with 128 / W rows per tile or
// whole tiles per 128 pixels, Cout in {32, 64, 128, 256}.  Returns cudaErrorInvalidValue
// for shapes it does not take.
cudaError_t unet_conv3x3(const ConvCall& call, cudaStream_t stream)
{
    const int T = call.T, H = call.H, W = call.W, Cin = call.Cin, Cout = call.Cout;
    const int y_cstride = call.y_cstride, y_coff = call.y_coff, upsample = call.upsample;
    const void *x = call.x, *wk = call.wk;
    void* y = call.y;
    if (call.pool && (W < 16 || W > 64 || H % 2 || upsample)) return cudaErrorInvalidValue;
    if (T < 1 || H < 1 || W < 1 || Cin < kKc || Cin % kKc || (Cout != 32 && Cout != 64 && Cout != 128 && Cout != 256))
        return cudaErrorInvalidValue;
    if (W > kTileM || kTileM % W) return cudaErrorInvalidValue;
    int hb = kTileM / W, nb = 1;
    if (hb > H) {
        if (hb % H) return cudaErrorInvalidValue;
        nb = hb / H;
        hb = H;
    } else if (H % hb) {
        return cudaErrorInvalidValue;
    }
    const long long pixels = (long long)T * H * W;
    if (pixels % kTileM || (nb > 1 && T % nb)) return cudaErrorInvalidValue;
    if (y_cstride % 8 || y_coff % 8 || y_coff + Cout > y_cstride) return cudaErrorInvalidValue;
    if (reinterpret_cast<uintptr_t>(y) % 16) return cudaErrorInvalidValue;  // a TMA store's base
    EncodeTiled enc = tensor_map_encoder();
    if (!enc) return cudaErrorNotSupported;

    // the form, and the output channels of a CTA
    const int sms = sm_count();
    int mt = 0, stages = 0;
    if (nb == 1) halo_shape(H, W, Cout, &mt, &stages);
    if (mt && conv_rows_takes(H, W, Cout)) return conv_rows_launch(call, sms, kSmemPerBlock, stream);
    // the output layer and half-resolution inputs are the row form's; the others pool 16-pixel rows
    if (call.rgb || call.frames || call.low || (call.pool && W != 16)) return cudaErrorInvalidValue;
    // on small grids one accumulator per CTA: twice the CTAs, half the MMAs of each (the halo
    // rows' overhead does not matter there)
    if (mt && pixels / (mt * kTileM) * 2 <= sms) mt = 1;
    const int kc = !mt && Cin % 64 == 0 ? 64 : kKc;  // one-tile form: channels of a K step
    const int tt = !mt && pixels >= 2ll * kTileM * sms ? 2 : 1;  // one-tile form: tiles of a CTA
    const int cta_px = (mt ? mt : tt) * kTileM;
    const long long ctas = (pixels + cta_px - 1) / cta_px;
    const int bn = split_channels(Cout, ctas, sms);
    const bool alone = ctas * (Cout / bn) <= sms;  // every CTA has an SM of its own

    CUtensorMap ta, tb;
    const cuuint64_t adim[4] = {(cuuint64_t)Cin, (cuuint64_t)W, (cuuint64_t)H, (cuuint64_t)T};
    const cuuint64_t astr[3] = {(cuuint64_t)Cin * 2, (cuuint64_t)W * Cin * 2, (cuuint64_t)H * W * Cin * 2};
    const cuuint32_t one4[4] = {1, 1, 1, 1};
    auto load_map = [&](CUtensorMap* m, const void* ptr, int rank, const cuuint64_t* dim, const cuuint64_t* str,
                        const cuuint32_t* box) {
        return enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, (cuuint32_t)rank, const_cast<void*>(ptr), dim, str, box, one4,
                   CU_TENSOR_MAP_INTERLEAVE_NONE,
                   box[0] == 64 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B,
                   CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
    };
    if (mt) {  // weights as {channel, co, dy, dx}: the three taps of a kernel column in one box
        const cuuint64_t ci = (cuuint64_t)Cin;
        const cuuint64_t bdim[4] = {ci, (cuuint64_t)Cout, 3, 3};
        const cuuint64_t bstr[3] = {9 * ci * 2, 3 * ci * 2, ci * 2};
        const cuuint32_t bbox[4] = {(cuuint32_t)kKc, (cuuint32_t)bn, 3, 1};
        const cuuint32_t abox[4] = {(cuuint32_t)kKc, (cuuint32_t)W, (cuuint32_t)(mt * kTileM / W + 2), 1u};
        if (!load_map(&ta, x, 4, adim, astr, abox) || !load_map(&tb, wk, 4, bdim, bstr, bbox)) return cudaErrorInvalidValue;
    } else {
        const cuuint64_t bdim[2] = {(cuuint64_t)9 * Cin, (cuuint64_t)Cout};
        const cuuint64_t bstr[1] = {(cuuint64_t)9 * Cin * 2};
        const cuuint32_t bbox[2] = {(cuuint32_t)kc, (cuuint32_t)bn};
        const cuuint32_t abox[4] = {(cuuint32_t)kc, (cuuint32_t)W, (cuuint32_t)hb, (cuuint32_t)nb};
        if (!load_map(&ta, x, 4, adim, astr, abox) || !load_map(&tb, wk, 2, bdim, bstr, bbox)) return cudaErrorInvalidValue;
    }

    // The output map: the epilogue's box of 32 channels x the CTA's pixels (rows x W x
    // images), or for the upsampling a 5-D view {channel, b, x, a, n H + y} of the 2H x 2W
    // output with pixel (2y + a, 2x + b), whose box {32, 1, W, 1, rows} takes one replica.
    const cuuint64_t cs = (cuuint64_t)y_cstride;
    auto y_map = [&](CUtensorMap* m, int rows, int imgs) -> bool {
        if (!upsample) {
            const cuuint64_t d[4] = {cs, (cuuint64_t)W, (cuuint64_t)H, (cuuint64_t)T};
            const cuuint64_t st[3] = {cs * 2, (cuuint64_t)W * cs * 2, (cuuint64_t)H * W * cs * 2};
            const cuuint32_t box[4] = {(cuuint32_t)kKc, (cuuint32_t)W, (cuuint32_t)rows, (cuuint32_t)imgs};
            return enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, y, d, st, box, one4, CU_TENSOR_MAP_INTERLEAVE_NONE,
                       CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_NONE,
                       CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
        }
        const cuuint64_t d[5] = {cs, 2, (cuuint64_t)W, 2, (cuuint64_t)T * H};
        const cuuint64_t st[4] = {cs * 2, 2 * cs * 2, (cuuint64_t)2 * W * cs * 2, (cuuint64_t)4 * W * cs * 2};
        const cuuint32_t box[5] = {(cuuint32_t)kKc, 1, (cuuint32_t)W, 1, (cuuint32_t)(rows * imgs)};
        const cuuint32_t one5[5] = {1, 1, 1, 1, 1};
        return enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, y, d, st, box, one5, CU_TENSOR_MAP_INTERLEAVE_NONE,
                   CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_NONE,
                   CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
    };

    ConvArgs a;
    a.T = T;
    a.H = H;
    a.W = W;
    a.Cin = Cin;
    a.Cout = Cout;
    a.bias = call.bias;
    a.y_coff = y_coff;
    a.upsample = upsample;
    a.relu = call.relu;
    a.bn = bn;
    a.ncols = bn;
    a.count = call.count;
    a.pool = static_cast<uint16_t*>(call.pool);
    a.mt = mt;
    const unsigned parts = (unsigned)(Cout / bn);
    if (mt) {
        const int rows = mt * kTileM / W;
        CUtensorMap ty;
        if (!y_map(&ty, rows, 1)) return cudaErrorInvalidValue;
        const int stage = halo_stage_bytes(W, rows, bn);
        a.ncols = mt * bn;
        a.stages = stages;  // two
        if (alone)
            while (a.stages < kMaxStages && halo_smem_bytes(stage, a.stages + 1) <= (size_t)kSmemPerBlock) ++a.stages;
        const cudaError_t e =
            cudaFuncSetAttribute(conv3x3_halo, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemPerBlock);
        if (e != cudaSuccess) return e;
        const size_t hsmem = halo_smem_bytes(stage, a.stages);
        // as many CTAs as fit at once (shared memory; registers allow 5), each walking bands
        const int per_sm = std::min(5, (int)(kSmemPerSm / (hsmem + 1024)));
        const long long grid = std::min<long long>(ctas, (long long)std::max(per_sm, 1) * sms);
        return launch_kernel(conv3x3_halo, dim3((unsigned)grid, parts), 128, hsmem, stream, call.pdl, ta, tb, ty, a,
                           (int)ctas);
    }
    // one-tile form: a lone CTA (and one with two tiles, whose accumulators take the tensor
    // memory) rings as deep as its SM's shared memory, else two CTAs share an SM
    const int stage = conv_stage_bytes(bn, kc, tt);
    const size_t budget = alone || tt > 1 ? (size_t)kSmemPerBlock : kSmemPerSm / 2 - 1024;
    a.ncols = tt * bn;
    a.stages = 1;
    while (a.stages < kMaxStages && conv_smem_bytes(stage, a.stages + 1) <= budget) ++a.stages;
    CUtensorMap ty;
    if (!y_map(&ty, hb, nb)) return cudaErrorInvalidValue;
    auto go = [&](auto kernel) -> cudaError_t {
        const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemPerBlock);
        if (e != cudaSuccess) return e;
        return launch_kernel(kernel, dim3((unsigned)ctas, parts), 128, conv_smem_bytes(stage, a.stages), stream, call.pdl,
                           ta, tb, ty, a);
    };
    if (kc == 64) return tt == 2 ? go(conv3x3_tc<64, 2>) : go(conv3x3_tc<64, 1>);
    return tt == 2 ? go(conv3x3_tc<32, 2>) : go(conv3x3_tc<32, 1>);
}

namespace {

constexpr int kInCh = 6;   // network input channels (padded to 32 in memory)
constexpr int kLevels = 4;
constexpr int kWidths[kLevels] = {32, 64, 128, 256};

// ---- small CUDA-core kernels around the convolutions

// Per 64 x 64 cell of each frame (blockIdx.x: cell, blockIdx.y: frame): 1 if it holds a
// hole pixel (mask == 1), at the cell's entry of the concatenated grids.
__global__ void tile_flags_kernel(const __grid_constant__ FrameTable ft, int* __restrict__ flags)
{
    const int f = blockIdx.y, cell = blockIdx.x;
    const int w = ft.w[f], h = ft.h[f], ntx = ft.ntx[f];
    if (cell >= ntx * ((h + kTile - 1) / kTile)) return;  // uniform
    const int tx = cell % ntx, ty = cell / ntx;
    const uint8_t* mask = ft.mask[f];
    int any = 0;
    for (int i = threadIdx.x; i < kTile * kTile; i += blockDim.x) {
        const int x = tx * kTile + (i & (kTile - 1)), y = ty * kTile + (i >> 6);
        if (x < w && y < h && mask[(size_t)y * w + x]) any = 1;
    }
    any = __syncthreads_or(any);
    if (threadIdx.x == 0) flags[ft.off[f] + cell] = any;
}

// Ordered list of the flagged tiles (index ty * ntx + tx) and its length, one CTA.
__global__ void tile_list_kernel(const int* __restrict__ flags, int ntiles, int* __restrict__ list,
                                 int* __restrict__ count)
{
    __shared__ int warp_sums[32];
    __shared__ int base;
    if (threadIdx.x == 0) base = 0;
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int c0 = 0; c0 < ntiles; c0 += blockDim.x) {
        const int i = c0 + threadIdx.x;
        const int f = i < ntiles ? flags[i] : 0;
        int incl = f;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += v;
        }
        if (lane == 31) warp_sums[warp] = incl;
        __syncthreads();
        if (warp == 0) {
            const int nw = blockDim.x >> 5;
            int ws = lane < nw ? warp_sums[lane] : 0;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int v = __shfl_up_sync(0xffffffffu, ws, o);
                if (lane >= o) ws += v;
            }
            if (lane < nw) warp_sums[lane] = ws;  // inclusive prefix of warp totals
        }
        __syncthreads();
        const int before = base + (warp ? warp_sums[warp - 1] : 0) + incl - f;
        if (f) list[before] = i;
        __syncthreads();
        if (threadIdx.x == blockDim.x - 1) base = before + f;
        __syncthreads();
    }
    if (threadIdx.x == 0) *count = base;
}

__device__ __forceinline__ uint16_t bf16_bits(float v)
{
    const __nv_bfloat16 b = __float2bfloat16_rn(v);
    return *reinterpret_cast<const uint16_t*>(&b);
}

// The network input of listed tile ti, pixel (py, px) of its window: the six channels of
// the definition (the plain path's right eye / 255: warped colors and the Patcher's fill
// at holes; the hole mask; near / warped depth, 0 at holes; near / source depth), rounded
// to bfloat16, then 26 zero channels.
// Pixels outside the frame (frames smaller than a tile) are all zero.
__global__ void tile_input_kernel(const __grid_constant__ FrameTable ft, const int* __restrict__ list,
                                  const int* __restrict__ count, uint16_t* __restrict__ x)
{
    const int ti = blockIdx.y;
    if (ti >= *count) return;
    const int p = blockIdx.x * blockDim.x + threadIdx.x;  // pixel of the tile
    if (p >= kTile * kTile) return;
    const int g = list[ti];
    const int f = table_frame(ft, g);
    const int tile = g - ft.off[f];
    const int w = ft.w[f], h = ft.h[f], ntx = ft.ntx[f];
    const float near_ = ft.near_[f];
    const int gx = window_origin(tile % ntx, w) + (p & (kTile - 1)), gy = window_origin(tile / ntx, h) + (p >> 6);
    float c[kInCh] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
    if (gx < w && gy < h) {
        const size_t o = (size_t)gy * w + gx;
        const bool hole = ft.mask[f][o] != 0;
        const uint32_t v = ft.rgba[f][o];
        c[0] = __fdiv_rn((float)(v & 255u), 255.0f);
        c[1] = __fdiv_rn((float)((v >> 8) & 255u), 255.0f);
        c[2] = __fdiv_rn((float)((v >> 16) & 255u), 255.0f);
        if (!hole) c[4] = __fdiv_rn(near_, fmaxf(ft.zt[f][o], near_));
        c[3] = hole ? 1.0f : 0.0f;
        c[5] = __fdiv_rn(near_, fmaxf(ft.zsrc[f][o], near_));
    }
    uint4 q[4] = {};
    uint32_t* qw = reinterpret_cast<uint32_t*>(q);
    qw[0] = (uint32_t)bf16_bits(c[0]) | ((uint32_t)bf16_bits(c[1]) << 16);
    qw[1] = (uint32_t)bf16_bits(c[2]) | ((uint32_t)bf16_bits(c[3]) << 16);
    qw[2] = (uint32_t)bf16_bits(c[4]) | ((uint32_t)bf16_bits(c[5]) << 16);
    uint4* dst = reinterpret_cast<uint4*>(x + ((size_t)ti * kTile * kTile + p) * 32);
#pragma unroll
    for (int i = 0; i < 4; ++i) dst[i] = q[i];
}

// The three colors of every pixel of the first T tiles to rgb (T x 64 x 64 x 3 floats), from
// stored activations (the training forward, which keeps them for its backward pass).
__global__ void output_kernel(const uint16_t* a, const float* wo, int T, float* rgb)
{
    pdl_wait();
    const int ti = blockIdx.y;
    if (ti >= T) return;
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= kTile * kTile) return;
    const uint4* src = reinterpret_cast<const uint4*>(a + ((size_t)ti * kTile * kTile + p) * 32);
    float v[32];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const uint4 q = src[i];
        const uint32_t qw[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            v[8 * i + 2 * k] = __uint_as_float(qw[k] << 16);
            v[8 * i + 2 * k + 1] = __uint_as_float(qw[k] & 0xffff0000u);
        }
    }
    float col[3];
    net_colors(v, wo, col);
    float* o = rgb + ((size_t)ti * kTile * kTile + p) * 3;
    o[0] = col[0];
    o[1] = col[1];
    o[2] = col[2];
}

void host_bf16_impl(const float* src, size_t n, uint16_t* dst)
{
    for (size_t i = 0; i < n; ++i) {
        uint32_t u;
        std::memcpy(&u, &src[i], 4);
        if ((u & 0x7fffffffu) > 0x7f800000u) {  // NaN stays NaN
            dst[i] = (uint16_t)((u >> 16) | 0x40u);
            continue;
        }
        u += 0x7fffu + ((u >> 16) & 1u);
        dst[i] = (uint16_t)(u >> 16);
    }
}

}  // namespace

void host_bf16(const float* src, size_t n, uint16_t* dst) { host_bf16_impl(src, n, dst); }

cudaError_t unet_output_rgb(const UnetNet* n, int T, float* rgb, cudaStream_t s)
{
    return launch_kernel(output_kernel, dim3(16, (unsigned)T), 256, 0, s, true, n->d0b, n->wout, T, rgb);
}

size_t unet_param_count()
{
    size_t n = 0;
    int cin = kInCh;
    for (int l = 0; l < kLevels; ++l) {
        n += (size_t)kWidths[l] * cin * 9 + kWidths[l] + (size_t)kWidths[l] * kWidths[l] * 9 + kWidths[l];
        cin = kWidths[l];
    }
    for (int l = kLevels - 2; l >= 0; --l) {
        const int c = kWidths[l];
        n += (size_t)c * (c + kWidths[l + 1]) * 9 + c + (size_t)c * c * 9 + c;
    }
    return n + 3 * 32 + 3;
}

void unet_layer_dims(int i, int* cin, int* cout)
{
    // i = 0..7 encoder (level i / 2), 8..13 decoder (levels 2, 1, 0)
    if (i < 8) {
        const int l = i / 2;
        *cout = kWidths[l];
        *cin = (i % 2) ? kWidths[l] : (l ? kWidths[l - 1] : kInCh);
    } else {
        const int l = 2 - (i - 8) / 2;
        *cout = kWidths[l];
        *cin = ((i - 8) % 2) ? kWidths[l] : kWidths[l] + kWidths[l + 1];
    }
}

void unet_free(UnetNet* n)
{
    if (!n) return;
    for (auto& L : n->conv) {
        cudaFree(L.wk);
        cudaFree(L.bias);
    }
    cudaFree(n->wout);
    uint16_t* bufs[] = {n->in0, n->e0a, n->cat0, n->skip0, n->d1b, n->p0,  n->e1a, n->cat1, n->skip1, n->d2b,
                        n->p1,  n->e2a, n->cat2, n->p2,    n->e3a, n->d2a, n->d1a, n->d0a,  n->d0b};
    for (uint16_t* b : bufs) cudaFree(b);
    cudaFree(n->flags);
    cudaFree(n->list);
    cudaFree(n->count);
    delete n;
}

UnetNet* unet_create(const float* params, size_t n_params, int max_tiles, int max_grid_tiles, bool train)
{
    if (!params || n_params != unet_param_count() || max_tiles < 1 || max_grid_tiles < 1) return nullptr;
    UnetNet* n = new UnetNet();
    std::memset(n, 0, sizeof *n);
    n->max_tiles = (max_tiles + 1) & ~1;  // even: the 8 x 8 level takes two tiles per 128-pixel MMA tile
    n->max_grid_tiles = max_grid_tiles;
    bool ok = true;
    const float* p = params;
    std::vector<uint16_t> hk;
    for (int i = 0; i < 14 && ok; ++i) {
        int cin, cout;
        unet_layer_dims(i, &cin, &cout);
        UnetLayer& L = n->conv[i];
        L.cin = cin;
        L.cout = cout;
        L.cin_pad = (cin + 31) / 32 * 32;
        // (cout, cin, 3, 3) -> (cout, 3, 3, cin_pad), bfloat16
        std::vector<float> km((size_t)cout * 9 * L.cin_pad, 0.0f);
        for (int co = 0; co < cout; ++co)
            for (int ci = 0; ci < cin; ++ci)
                for (int t = 0; t < 9; ++t) km[((size_t)co * 9 + t) * L.cin_pad + ci] = p[((size_t)co * cin + ci) * 9 + t];
        p += (size_t)cout * cin * 9;
        hk.resize(km.size());
        host_bf16(km.data(), km.size(), hk.data());
        ok = cudaMalloc(&L.wk, hk.size() * 2) == cudaSuccess && cudaMalloc(&L.bias, cout * 4) == cudaSuccess &&
             cudaMemcpy(L.wk, hk.data(), hk.size() * 2, cudaMemcpyHostToDevice) == cudaSuccess &&
             cudaMemcpy(L.bias, p, cout * 4, cudaMemcpyHostToDevice) == cudaSuccess;
        p += cout;
    }
    if (ok) {  // output layer: bfloat16-rounded weights kept as floats, FP32 biases
        std::vector<uint16_t> b16(96);
        host_bf16(p, 96, b16.data());
        float wo[99];
        for (int i = 0; i < 96; ++i) {
            const uint32_t u = (uint32_t)b16[i] << 16;
            std::memcpy(&wo[i], &u, 4);
        }
        for (int i = 0; i < 3; ++i) wo[96 + i] = p[96 + i];
        ok = cudaMalloc(&n->wout, sizeof wo) == cudaSuccess &&
             cudaMemcpy(n->wout, wo, sizeof wo, cudaMemcpyHostToDevice) == cudaSuccess;
    }
    const size_t T = n->max_tiles, P0 = T * 64 * 64, P1 = T * 32 * 32, P2 = T * 16 * 16, P3 = T * 8 * 8;
    struct {
        uint16_t** b;
        size_t elems;
    } al[] = {{&n->e0a, P0 * 32}, {&n->p0, P1 * 32}, {&n->e1a, P1 * 64}, {&n->p1, P2 * 64}, {&n->e2a, P2 * 128},
              {&n->cat2, P2 * 384}, {&n->p2, P3 * 128}, {&n->e3a, P3 * 256}, {&n->d2a, P2 * 128}, {&n->d1a, P1 * 64},
              {&n->d0a, P0 * 32},
              // training
              {&n->cat0, train ? P0 * 96 : 0}, {&n->cat1, train ? P1 * 192 : 0}, {&n->d0b, train ? P0 * 32 : 0},
              // inference
              {&n->in0, train ? 0 : P0 * 32}, {&n->skip0, train ? 0 : P0 * 32}, {&n->d1b, train ? 0 : P1 * 64},
              {&n->skip1, train ? 0 : P1 * 64}, {&n->d2b, train ? 0 : P2 * 128}};
    for (auto& x : al)
        if (ok && x.elems) ok = cudaMalloc(x.b, x.elems * 2) == cudaSuccess;
    if (ok) {
        // the in0 buffer of tiles never written stays zero (T rounded up to even)
        ok = (train || cudaMemset(n->in0, 0, P0 * 32 * 2) == cudaSuccess) &&
             cudaMalloc(&n->flags, (size_t)max_grid_tiles * 4) == cudaSuccess &&
             cudaMalloc(&n->list, (size_t)max_grid_tiles * 4) == cudaSuccess &&
             cudaMalloc(&n->count, 4) == cudaSuccess;
    }
    if (!ok) {
        cudaGetLastError();
        unet_free(n);
        return nullptr;
    }
    return n;
}

// The 14 convolutions over the first T tiles of x (tiles at or after *count skipped when
// count is given), the 2x2 pools in the epilogues of the layers they follow.  In an inference
// net the decoder's first layers of levels 1 and 0 read the skip and the lower level's output
// at its own resolution; in a training net they read the concatenation, written by the
// layers before.  The output layer rides on the last one: colors to out.rgb, or composed into
// out.frames; with neither (training), the last layer's activations end in d0b.
cudaError_t unet_run(UnetNet* n, const uint16_t* x, int T, const int* count, const NetOut& out, cudaStream_t s)
{
    const int Te = (T + 1) & ~1;  // the 8 x 8 level takes two tiles per 128-pixel accumulator
    const bool cat = n->cat0 != nullptr;
    cudaError_t e = cudaSuccess;
    // layer i on H x H tiles: input (and half-resolution input), output at channel offset coff of
    // cstride, upsampled store, pooled copy
    auto conv = [&](int i, const uint16_t* in, const uint16_t* low, int cskip, int H, void* y, int cstride, int coff,
                    int up, void* pool) {
        if (e != cudaSuccess) return;
        const UnetLayer& L = n->conv[i];
        ConvCall c{in, L.wk, y, L.bias, count, pool, i == 0 ? T : Te, H, H, L.cin_pad, L.cout, cstride, coff, up, 1};
        c.low = low;
        c.cskip = cskip;
        // the kernel before is the layer before.  The frame path (count) is launched plainly: it
        // shares the GPU with other streams' batches in the serving loop, whose learned frames met
        // stalls with it (p99 4 to 27 ms in two runs, 1.3 to 2.8 in four without; one frame alone
        // 604 against 639 us).
        c.pdl = i > 0 && !count;
        if (i == 13) {
            c.T = T;
            c.wout = n->wout;
            c.rgb = out.rgb;
            c.frames = out.frames;
            c.list = out.frames ? n->list : nullptr;
        }
        e = unet_conv3x3(c, s);
    };
    uint16_t* const none = nullptr;
    conv(0, x, none, 0, 64, n->e0a, 32, 0, 0, nullptr);                                       // enc0a
    conv(1, n->e0a, none, 0, 64, cat ? n->cat0 : n->skip0, cat ? 96 : 32, 0, 0, n->p0);       // enc0b
    conv(2, n->p0, none, 0, 32, n->e1a, 64, 0, 0, nullptr);                                   // enc1a
    conv(3, n->e1a, none, 0, 32, cat ? n->cat1 : n->skip1, cat ? 192 : 64, 0, 0, n->p1);      // enc1b
    conv(4, n->p1, none, 0, 16, n->e2a, 128, 0, 0, nullptr);                                  // enc2a
    conv(5, n->e2a, none, 0, 16, n->cat2, 384, 0, 0, n->p2);                                  // enc2b
    conv(6, n->p2, none, 0, 8, n->e3a, 256, 0, 0, nullptr);                                   // enc3a
    conv(7, n->e3a, none, 0, 8, n->cat2, 384, 128, 1, nullptr);                               // enc3b, upsampled
    conv(8, n->cat2, none, 0, 16, n->d2a, 128, 0, 0, nullptr);                                // dec2a
    if (cat) {
        conv(9, n->d2a, none, 0, 16, n->cat1, 192, 64, 1, nullptr);                           // dec2b, upsampled
        conv(10, n->cat1, none, 0, 32, n->d1a, 64, 0, 0, nullptr);                            // dec1a
        conv(11, n->d1a, none, 0, 32, n->cat0, 96, 32, 1, nullptr);                           // dec1b, upsampled
        conv(12, n->cat0, none, 0, 64, n->d0a, 32, 0, 0, nullptr);                            // dec0a
    } else {
        conv(9, n->d2a, none, 0, 16, n->d2b, 128, 0, 0, nullptr);
        conv(10, n->skip1, n->d2b, 64, 32, n->d1a, 64, 0, 0, nullptr);
        conv(11, n->d1a, none, 0, 32, n->d1b, 64, 0, 0, nullptr);
        conv(12, n->skip0, n->d1b, 32, 64, n->d0a, 32, 0, 0, nullptr);
    }
    conv(13, n->d0a, none, 0, 64, n->d0b, 32, 0, 0, nullptr);                                 // dec0b
    return e;
}

}  // namespace yoro

struct yoro_unet_ctx {
    yoro::UnetNet* net;
    int device;
    int max_w, max_h;
};

extern "C" {

yoro_status yoro_unet_conv3x3(const void* x, int T, int H, int W, int Cin, const void* wk, const float* bias,
                              void* y, int Cout, int y_cstride, int y_coff, int upsample, int relu,
                              void* cuda_stream)
{
    if (!x || !wk || !bias || !y) return YORO_EINVAL;
    if (((uintptr_t)x | (uintptr_t)wk | (uintptr_t)y) & 15u) return YORO_EALIGN;
    const cudaError_t e = yoro::unet_conv3x3(yoro::ConvCall{x, wk, y, bias, nullptr, nullptr, T, H, W, Cin, Cout, y_cstride,
                                                            y_coff, upsample, relu},
                                             (cudaStream_t)cuda_stream);
    if (e == cudaErrorInvalidValue) return YORO_EINVAL;
    return e == cudaSuccess ? YORO_OK : YORO_ECUDA;
}

long long yoro_unet_param_count(void) { return (long long)yoro::unet_param_count(); }

yoro_unet yoro_unet_create(const float* params, long long n_params, int max_tiles, int max_w, int max_h)
{
    if (!params || n_params <= 0 || max_tiles < 0 || max_w < 0 || max_h < 0 || max_w > 65536 || max_h > 65536)
        return nullptr;
    const int grid_tiles = ((max_w + 63) / 64) * ((max_h + 63) / 64);
    const int tiles = std::max(std::max(max_tiles, grid_tiles), 2);
    yoro_unet_ctx* c = new (std::nothrow) yoro_unet_ctx();
    if (!c) return nullptr;
    if (cudaGetDevice(&c->device) != cudaSuccess) {
        cudaGetLastError();
        delete c;
        return nullptr;
    }
    c->max_w = max_w;
    c->max_h = max_h;
    c->net = yoro::unet_create(params, (size_t)n_params, tiles, tiles, false);  // flags and list hold `tiles` cells
    if (!c->net) {
        delete c;
        return nullptr;
    }
    return c;
}

void yoro_unet_destroy(yoro_unet u)
{
    if (!u) return;
    yoro::unet_free(u->net);
    delete u;
}

yoro_status yoro_unet_forward(yoro_unet u, const void* x, int T, float* rgb, void* cuda_stream)
{
    if (!u || !x || !rgb || T < 0 || T > u->net->max_tiles) return YORO_EINVAL;
    if (T == 0) return YORO_OK;
    if (((uintptr_t)x & 15u) || ((uintptr_t)rgb & 3u)) return YORO_EALIGN;
    const yoro::NetOut out{rgb, nullptr};
    return yoro::unet_run(u->net, static_cast<const uint16_t*>(x), T, nullptr, out, (cudaStream_t)cuda_stream) ==
                   cudaSuccess
               ? YORO_OK
               : YORO_ECUDA;
}

}  // extern "C"

namespace {

// Checks of one frame of the inpainting entry points; YORO_OK, or the status to return.
yoro_status check_frame(const yoro_unet_ctx* u, int w, int h, float near_, const void* rgba,
                        const unsigned char* mask, const float* zt, const float* src_depth)
{
    if (w < 0 || h < 0 || !(near_ > 0.0f) || !std::isfinite(near_)) return YORO_EINVAL;
    if ((size_t)w * h == 0) return YORO_OK;
    if (w > u->max_w || h > u->max_h) return YORO_ETOOBIG;
    if (!rgba || !mask || !zt || !src_depth) return YORO_EINVAL;
    if (((uintptr_t)rgba | (uintptr_t)zt | (uintptr_t)src_depth) & 3u) return YORO_EALIGN;
    return YORO_OK;
}

// Appends frame i to the table (its cells after those already there).
void table_add(yoro::FrameTable& ft, const yoro_unet_frame& fr)
{
    const int k = ft.n;
    ft.w[k] = fr.w;
    ft.h[k] = fr.h;
    ft.ntx[k] = (fr.w + 63) / 64;
    ft.near_[k] = fr.near_;
    ft.rgba[k] = static_cast<uint32_t*>(fr.rgba);
    ft.mask[k] = fr.mask;
    ft.zt[k] = fr.zt;
    ft.zsrc[k] = fr.src_depth;
    ft.off[k + 1] = ft.off[k] + ft.ntx[k] * ((fr.h + 63) / 64);
    ft.n = k + 1;
}

// One pass of the network over the hole cells of the table's frames: the cells' flags, the
// list of the flagged ones and its length on the device (launches cover every cell; those
// past the list's length return at once), the inputs, and the 14 layers, the last of which
// composes.
yoro_status inpaint_table(yoro_unet_ctx* u, const yoro::FrameTable& ft, cudaStream_t s)
{
    yoro::UnetNet* n = u->net;
    const int total = ft.off[ft.n];
    int maxcells = 0;
    for (int f = 0; f < ft.n; ++f) maxcells = std::max(maxcells, ft.off[f + 1] - ft.off[f]);
    if (total == 0) return YORO_OK;
    yoro::tile_flags_kernel<<<dim3((unsigned)maxcells, (unsigned)ft.n), 256, 0, s>>>(ft, n->flags);
    yoro::tile_list_kernel<<<1, 1024, 0, s>>>(n->flags, total, n->list, n->count);
    yoro::tile_input_kernel<<<dim3(16, (unsigned)total), 256, 0, s>>>(ft, n->list, n->count, n->in0);
    if (cudaGetLastError() != cudaSuccess) return YORO_ECUDA;
    const yoro::NetOut out{nullptr, &ft};
    return yoro::unet_run(n, n->in0, total, n->count, out, s) == cudaSuccess ? YORO_OK : YORO_ECUDA;
}

}  // namespace

extern "C" {

yoro_status yoro_unet_inpaint(yoro_unet u, int w, int h, float near_, void* rgba, const unsigned char* mask,
                              const float* zt, const float* src_depth, void* cuda_stream)
{
    if (!u) return YORO_EINVAL;
    const yoro_status st = check_frame(u, w, h, near_, rgba, mask, zt, src_depth);
    if (st != YORO_OK || (size_t)w * h == 0) return st;
    yoro::FrameTable ft;
    ft.n = 0;
    ft.off[0] = 0;
    table_add(ft, yoro_unet_frame{w, h, near_, rgba, mask, zt, src_depth});
    return inpaint_table(u, ft, (cudaStream_t)cuda_stream);
}

yoro_status yoro_unet_inpaint_batch(yoro_unet u, int n, const yoro_unet_frame* frames, void* cuda_stream)
{
    if (!u || n < 0 || (n > 0 && !frames)) return YORO_EINVAL;
    for (int i = 0; i < n; ++i) {
        const yoro_unet_frame& fr = frames[i];
        const yoro_status st = check_frame(u, fr.w, fr.h, fr.near_, fr.rgba, fr.mask, fr.zt, fr.src_depth);
        if (st != YORO_OK) return st;
    }
    // groups of frames whose cells fit the network's buffers, up to kMaxInpaintFrames each
    const int capacity = std::min(u->net->max_tiles, u->net->max_grid_tiles);
    yoro::FrameTable ft;
    ft.n = 0;
    ft.off[0] = 0;
    for (int i = 0; i < n; ++i) {
        const yoro_unet_frame& fr = frames[i];
        if ((size_t)fr.w * fr.h == 0) continue;
        const int cells = ((fr.w + 63) / 64) * ((fr.h + 63) / 64);
        if (ft.n == yoro::kMaxInpaintFrames || (ft.n > 0 && ft.off[ft.n] + cells > capacity)) {
            const yoro_status st = inpaint_table(u, ft, (cudaStream_t)cuda_stream);
            if (st != YORO_OK) return st;
            ft.n = 0;
        }
        table_add(ft, fr);
    }
    return ft.n ? inpaint_table(u, ft, (cudaStream_t)cuda_stream) : YORO_OK;
}

yoro_status yoro_unet_prepare(yoro_unet u, int w, int h, float near_, const void* rgba, const unsigned char* mask,
                              const float* zt, const float* src_depth, void* x_out, int max_out, int* list_host,
                              int* count_host, void* cuda_stream)
{
    if (!u || !list_host || !count_host) return YORO_EINVAL;
    *count_host = 0;
    yoro_status st = check_frame(u, w, h, near_, rgba, mask, zt, src_depth);
    if (st != YORO_OK || (size_t)w * h == 0) return st;
    const int ntx = (w + 63) / 64, nty = (h + 63) / 64;
    if (!x_out || max_out < ntx * nty) return YORO_EINVAL;
    if ((uintptr_t)x_out & 15u) return YORO_EALIGN;
    yoro::UnetNet* n = u->net;
    const cudaStream_t s = (cudaStream_t)cuda_stream;
    yoro::FrameTable ft;
    ft.n = 0;
    ft.off[0] = 0;
    table_add(ft, yoro_unet_frame{w, h, near_, const_cast<void*>(rgba), mask, zt, src_depth});
    yoro::tile_flags_kernel<<<dim3((unsigned)(ntx * nty), 1), 256, 0, s>>>(ft, n->flags);
    yoro::tile_list_kernel<<<1, 1024, 0, s>>>(n->flags, ntx * nty, n->list, n->count);
    yoro::tile_input_kernel<<<dim3(16, (unsigned)(ntx * nty)), 256, 0, s>>>(ft, n->list, n->count,
                                                                          static_cast<uint16_t*>(x_out));
    if (cudaGetLastError() != cudaSuccess) return YORO_ECUDA;
    if (cudaMemcpyAsync(count_host, n->count, 4, cudaMemcpyDeviceToHost, s) != cudaSuccess ||
        cudaMemcpyAsync(list_host, n->list, (size_t)ntx * nty * 4, cudaMemcpyDeviceToHost, s) != cudaSuccess ||
        cudaStreamSynchronize(s) != cudaSuccess) {
        cudaGetLastError();
        return YORO_ECUDA;
    }
    return YORO_OK;
}

yoro_status yoro_unet_status(void* cuda_stream)
{
    if (cudaStreamSynchronize((cudaStream_t)cuda_stream) != cudaSuccess) {
        cudaGetLastError();
        return YORO_ECUDA;
    }
    return yoro::unet_status_take() ? YORO_EDEVICE : YORO_OK;
}

}  // extern "C"
