// Weight gradient of the inpainter's 3x3 layers on the tensor cores:
//   dW[co][ci][dy][dx] = sum over pixels p of dZ[p][co] X[p + (dy - 1, dx - 1)][ci]
// with bfloat16 dZ and X and FP32 accumulation: per layer a product of K = pixels (4,096 per
// tile at the top level), M = co, N = 9 ci.
//
// Both operands lie in memory as NHWC rows, channels contiguous, so in shared memory the K
// index (the pixel) strides by 64 bytes per 32 channels: MN-major operands of tcgen05.mma
// with the 64-byte swizzle the copy engine writes, no transposition pass.  A box is 8 rows
// of one image: of dZ its W columns alone, of X the ten rows around them with a column of
// padding on each side (what lies outside the image arrives as zeros).  A K step is 16 pixels
// of dZ (of one row; of two where W = 8, whose X rows are 16 pixels apart for that) and the
// 16 pixels of X at a constant distance: the three dy are the three 32-column blocks of N =
// 96 (block stride one row), the dx are three MMAs from starts one pixel apart.  So every
// product is one of the sum's, a gradient pixel with an input pixel or with the padding's
// zero: an infinite input reaches the taps it lies under and no others.  (With padding columns
// in dZ too, one box walked as one run of pixels, their zeros met the columns 0 and W - 1 of
// X, and 0 x infinity put NaN into taps that never meet such a pixel.)
//
// Precision.  The tensor core cuts an accumulator off after every step of 16 pixels, toward
// zero, so a long chain loses half a unit in the last place per step, always in the same
// direction.  An accumulator therefore takes a few steps only (8 at 64 pixels a side, 4, 2, 1
// below), is read back and added in FP32, rounded to nearest, in the registers of twelve
// accumulating warps, while the MMAs go on in the next of five accumulators of 96 columns (one
// dx each); the shares' sums are added with their rounding errors beside them.  The chains'
// lengths are the longest that stay within the error of chains of FP32 fused multiply-adds at
// every batch from 4 tiles on (relative error of a layer's gradient against 64 bits, random
// dense inputs / sparse gradients on non-negative inputs):
//                                    multiply-adds      one chain per CTA  these chains
//   64 tiles, 64 px, 96 channels     3.8e-7 / 3.1e-7    5.6e-6 / 1.5e-6    1.7e-7 / 1.3e-7
//   64 tiles, 32 px, 192 channels    2.9e-7 / 1.7e-7    2.7e-6 / 6.4e-7    1.4e-7 / 1.1e-7
//   64 tiles, 16 px, 384 channels    2.5e-7 / 1.1e-7    1.3e-6 / 3.3e-7    1.3e-7 / 8.4e-8
//   64 tiles, 8 px, 256 channels     1.6e-7 / 7.8e-8    3.8e-7 / 1.2e-7    9.8e-8 / 5.5e-8
//   4 tiles, 8 px, 256 channels      9.7e-8 / 4.1e-8    (6 tiles: 3.1e-7)  4.9e-8 / 3.4e-8
// They cost 44, 32, 37 and 31 us for the first four layers, where one chain took 40, 27, 26 and
// 22: reading 96 columns back takes a warp about 700 cycles, three warps take turns, and an MMA
// 56.  (Chains of 4 and 2 steps at 64 and 32 px: 45 and 43 us; 32 columns per read and
// packed additions, which spill: 47, 49, 48, 40.)
//
// A CTA sums one (32 or 64 or 128 co) x (32 ci) x 9 tile over its share of the boxes; the
// shares' sums go to a workspace and dw_reduce_kernel adds them in order (so the gradient is
// the same bits on every run).  M is always 128: with 32 or 64 output channels the other rows
// multiply whatever follows in shared memory and are not read back.  One MMA takes 56 cycles
// at N = 96 whatever M holds.
#include <algorithm>

#include "tc.cuh"
#include "unet_internal.h"

namespace yoro {

namespace {

__device__ unsigned g_dw_status;  // waits that ran out in this file's kernel

// Warps: one copies, one issues MMAs, twelve accumulate (four lane quarters for each dx).
constexpr int kDwThreads = 64 + 12 * 32;
constexpr int kDwAcc = 5;                  // accumulators of kDwN columns
constexpr int kDwRows = 8;                 // rows of a box
constexpr int kDwN = 96;                   // N of an MMA: three dy times 32 ci
constexpr int kDwTile = 9 * 32;            // columns of a tile: 9 taps times 32 ci

// A level's shapes: W pixels wide, COB blocks of 32 output channels.
template <int W, int COB, int STAGES, int FLUSH>
struct DwShape {
    static constexpr int kPitch = W == 8 ? 16 : W + 2;  // pixels of an X row
    static constexpr int kSteps = kDwRows * W / 16;     // K steps of a box
    static constexpr int kPlane = kDwRows * W * 64;     // one 32-channel block of dZ
    static constexpr int kZ = COB * kPlane;
    static constexpr int kX = (kDwRows + 2) * kPitch * 64;
    static constexpr int kStage = (kZ + kX + 1023) / 1024 * 1024;
    // 16-byte units from the box's first X pixel to that of K step k
    __device__ static constexpr uint32_t x_start(int k) { return 4u * (uint32_t)(W == 8 ? 2 * k * kPitch : 16 * k / W * kPitch + 16 * k % W); }
    static constexpr int kStages = STAGES;
    static constexpr int kFlush = FLUSH;                // K steps of an accumulator
    static constexpr int kFlushes = kSteps / FLUSH;     // per box and dx
    // block stride of A: the next plane; with one plane the next pixel (those rows are not read back)
    static constexpr int kLboA = COB == 1 ? 64 : kPlane;
    // rows 64..127 of two planes read two more planes' worth past the last stage
    static constexpr int kSlack = COB == 2 ? std::max(0, 4 * kPlane - kStage) : 0;
    static constexpr int kSmem = 1024 + 1024 + STAGES * kStage + kSlack;
    static_assert(kSteps % FLUSH == 0, "whole chains");
    static_assert((W % 16 == 0 || W == 8) && kPlane % 1024 == 0, "K steps of 16 pixels, whole swizzle atoms");
    static_assert(kSmem <= 227 * 1024, "shared memory of one CTA");
};

__device__ __forceinline__ uint64_t desc_mn_sw64(uint32_t saddr, uint32_t block_stride, uint32_t group_stride)
{
    uint64_t d = (uint64_t)((saddr >> 4) & 0x3fffu);
    d |= (uint64_t)(block_stride >> 4) << 16;  // next 32 channels
    d |= (uint64_t)(group_stride >> 4) << 32;  // next 8 pixels
    d |= (uint64_t)1u << 46;
    d |= (uint64_t)4u << 61;
    return d;
}

// Wait for the phase of parity `parity` to complete; false after kWaitNs.
__device__ __forceinline__ bool mbar_wait_limit(uint64_t* bar, uint32_t parity)
{
    return mbar_try_wait(bar, parity) || mbar_wait(bar, parity, globaltimer() + kWaitNs);
}

template <class S, int COB>
__global__ void __launch_bounds__(kDwThreads, 1)
    conv3x3_dw(const __grid_constant__ CUtensorMap tmZ, const __grid_constant__ CUtensorMap tmX, int H, int boxes,
               int cbs, float* ws)
{
    extern __shared__ unsigned char smem_raw[];
    unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                                           ~static_cast<uintptr_t>(1023));
    uint64_t* full = reinterpret_cast<uint64_t*>(smem);
    uint64_t* empty = full + S::kStages;
    uint64_t* afull = empty + S::kStages;
    uint64_t* aempty = afull + kDwAcc;
    uint64_t* drain = aempty + kDwAcc;
    uint32_t* tslot = reinterpret_cast<uint32_t*>(drain + 1);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tslot + 1);
    unsigned char* stages = smem + 1024;
    const int warp = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
    const int cb = blockIdx.y % cbs, ct = blockIdx.y / cbs;
    const int b0 = (int)((long long)boxes * blockIdx.x / gridDim.x);
    const int b1 = (int)((long long)boxes * (blockIdx.x + 1) / gridDim.x);

    if (threadIdx.x == 0) {
        for (int s = 0; s < S::kStages; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        for (int s = 0; s < kDwAcc; ++s) {
            mbar_init(&afull[s], 1);
            mbar_init(&aempty[s], COB);  // the warps of the lane quarters that are read back
        }
        mbar_init(drain, 1);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tslot)),
                     "r"(512)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    pdl_wait();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tslot;
    auto timed_out = [&]() {
        atomicOr(&g_dw_status, kUnetTimeout);
        *abort_flag = 1;
    };
    int issued = 0;

    if (warp == 0) {
        if (lane == 0) {  // copies
            const int bands = H / kDwRows;
            for (int b = b0; b < b1; ++b) {
                const int i = b - b0, s = i % S::kStages;
                if (!mbar_wait_limit(&empty[s], ((i / S::kStages) & 1) ^ 1)) {
                    timed_out();
                    break;
                }
                const int n = b / bands, y0 = (b - n * bands) * kDwRows;
                unsigned char* st = stages + s * S::kStage;
                mbar_expect_tx(&full[s], (uint32_t)(S::kZ + S::kX));
#pragma unroll
                for (int j = 0; j < COB; ++j)
                    tma_load_4d(st + j * S::kPlane, &tmZ, &full[s], (ct * COB + j) * 32, 0, y0, n);
                tma_load_4d(st + S::kZ, &tmX, &full[s], cb * 32, -1, y0 - 1, n);
                ++issued;
            }
        }
    } else if (warp == 1) {  // MMAs: the whole warp runs the loop, one lane issues
        constexpr uint32_t idesc = idesc_bf16(kDwN) | (1u << 15) | (1u << 16);  // both operands MN-major
        const uint32_t el = elect_one();
        const uint64_t da = desc_mn_sw64(smem_u32(stages), S::kLboA, 512);
        const uint64_t db = desc_mn_sw64(smem_u32(stages) + S::kZ, S::kPitch * 64, S::kPitch == 16 ? 1024 : 512);
        auto issue_all = [&]() -> bool {
            int slot = 0, ph = 1;
            for (int b = b0; b < b1; ++b) {
                const int i = b - b0, s = i % S::kStages;
                if (!__all_sync(0xffffffffu, mbar_wait_limit(&full[s], (i / S::kStages) & 1))) return false;
                tc_fence_after();
                const uint64_t as = da + (uint64_t)((uint32_t)(s * S::kStage) >> 4);
                const uint64_t bs = db + (uint64_t)((uint32_t)(s * S::kStage) >> 4);
                for (int f = 0; f < S::kFlushes; ++f) {
#pragma unroll
                    for (int dx = 0; dx < 3; ++dx) {
                        if (!__all_sync(0xffffffffu, mbar_wait_limit(&aempty[slot], ph))) return false;
                        tc_fence_after();
#pragma unroll
                        for (int q = 0; q < S::kFlush; ++q) {
                            const int k = f * S::kFlush + q;
                            mma_bf16_elected(el, tmem + slot * kDwN, as + 64 * k, bs + S::x_start(k) + 4 * dx, idesc,
                                             q > 0 ? 1u : 0u);
                        }
                        mma_commit_elected(el, &afull[slot]);
                        if (++slot == kDwAcc) {
                            slot = 0;
                            ph ^= 1;
                        }
                    }
                }
                mma_commit_elected(el, &empty[s]);
            }
            return true;
        };
        bool ok = issue_all();
        mma_commit_elected(el, drain);  // arrives once every MMA issued above has completed
        ok = mbar_wait_warp(drain, 0, globaltimer() + kWaitNs) && ok;
        if (!ok && el) timed_out();
    } else if ((warp & 3) < COB) {  // accumulate: rows co = 32 (warp & 3) + lane, column blocks of one dx
        const int q = warp & 3, dx = (warp - 2) >> 2;
        const uint32_t tq = tmem + ((uint32_t)(q * 32) << 16);
        float sum[kDwN];
#pragma unroll
        for (int c = 0; c < kDwN; ++c) sum[c] = 0.0f;
        int slot = dx, ph = 0;
        bool ok = true;
        for (int e = (b1 - b0) * S::kFlushes; e > 0; --e) {
            if (!(ok = __all_sync(0xffffffffu, mbar_wait_limit(&afull[slot], ph)))) break;
            tc_fence_after();
#pragma unroll
            for (int c0 = 0; c0 < kDwN; c0 += 16) {  // 96 sums and 16 values: within 128 registers
                uint32_t v[16];
                tmem_ld16(tq + slot * kDwN + c0, v);
#pragma unroll
                for (int c = 0; c < 16; ++c) sum[c0 + c] = __fadd_rn(sum[c0 + c], __uint_as_float(v[c]));
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&aempty[slot]);
            slot += 3;
            if (slot >= kDwAcc) {
                slot -= kDwAcc;
                ph ^= 1;
            }
        }
        if (!ok && lane == 0) timed_out();
        if (ok) {  // row co of the tile, 3 x 32 of its sums: column dy 32 + ci is tap (dy, dx)
            float* row = ws + ((((size_t)blockIdx.y * gridDim.x + blockIdx.x) * COB + q) * 32 + lane) * kDwTile;
#pragma unroll
            for (int dy = 0; dy < 3; ++dy)
#pragma unroll
                for (int i = 0; i < 8; ++i)
                    reinterpret_cast<float4*>(row + (3 * dy + dx) * 32)[i] = make_float4(
                        sum[dy * 32 + 4 * i], sum[dy * 32 + 4 * i + 1], sum[dy * 32 + 4 * i + 2], sum[dy * 32 + 4 * i + 3]);
        }
    }
    __syncwarp();
    tc_fence_before();
    __syncthreads();
    if (threadIdx.x == 0 && *abort_flag) {  // copies still in flight after a timeout: wait for them (bounded)
        const uint64_t d = globaltimer() + kWaitNs;
        for (int i = max(0, issued - S::kStages); i < issued; ++i) mbar_wait(&full[i % S::kStages], (i / S::kStages) & 1, d);
    }
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
    }
}

// A sum with the roundings of its additions beside it (Knuth, "The Art of Computer Programming",
// vol. 2, 4.2.2: a + b = RN(a + b) + e, e by five more operations).
struct Sum2 {
    float s, e;
};

__device__ __forceinline__ void add(Sum2& a, float v)
{
    const float t = __fadd_rn(a.s, v), z = __fsub_rn(t, a.s);
    a.e = __fadd_rn(a.e, __fadd_rn(__fsub_rn(a.s, __fsub_rn(t, z)), __fsub_rn(v, z)));
    a.s = t;
}

// Where the sum is infinite or NaN, its error term means nothing.
__device__ __forceinline__ float value(const Sum2& a) { return isfinite(a.s) ? __fadd_rn(a.s, a.e) : a.s; }

// dW[co][ci][tap] = the sum over the shares of ws[ct cbs + cb][share][co][tap][ci], rounded once.
// A block takes 128 consecutive floats of a tile (32 loads of 16 bytes), its eight warps every
// eighth share, and adds the warps' sums in order.  Bound by reading the workspace from L2 (up to 22
// MB a layer); one thread per element over all shares was 13 us a layer, latency.
__global__ void __launch_bounds__(256) dw_reduce_kernel(const float* ws, int shares, int co_tile, int cbs, int cin,
                                                        float* dW)
{
    pdl_wait();
    __shared__ float4 part[8][32], rest[8][32];
    const int l = threadIdx.x & 31, g = threadIdx.x >> 5;
    const int quads = co_tile * (kDwTile / 4);  // of a tile
    const int tile = blockIdx.x / (quads / 32), q = (blockIdx.x - tile * (quads / 32)) * 32 + l;
    const float4* p = reinterpret_cast<const float4*>(ws) + (size_t)tile * shares * quads + q;
    Sum2 s[4] = {};
#pragma unroll 4
    for (int i = g; i < shares; i += 8) {
        const float4 v = p[(size_t)i * quads];
        add(s[0], v.x);
        add(s[1], v.y);
        add(s[2], v.z);
        add(s[3], v.w);
    }
    part[g][l] = make_float4(s[0].s, s[1].s, s[2].s, s[3].s);
    rest[g][l] = make_float4(s[0].e, s[1].e, s[2].e, s[3].e);
    __syncthreads();
    if (threadIdx.x < 128) {  // thread k: float k of the 128
        const int k = threadIdx.x, e = (q - l) * 4 + k;  // place in the tile: [co][tap][ci]
        Sum2 t = {0.0f, 0.0f};
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            add(t, reinterpret_cast<const float*>(&part[i][0])[k]);
            t.e = __fadd_rn(t.e, reinterpret_cast<const float*>(&rest[i][0])[k]);
        }
        const int c = e & 31, r = e >> 5, tap = r % 9, col = r / 9;
        const int ci = (tile % cbs) * 32 + c, co = tile / cbs * co_tile + col;  // tile = ct cbs + cb
        if (ci < cin) dW[((size_t)co * cin + ci) * 9 + tap] = value(t);  // the first layer's padding channels are dropped
    }
}

template <int W, int COB, int STAGES, int FLUSH>
cudaError_t launch(const CUtensorMap& tz, const CUtensorMap& tx, int H, int boxes, int tiles, int cbs, int shares,
                   float* ws, cudaStream_t s)
{
    using S = DwShape<W, COB, STAGES, FLUSH>;
    const cudaError_t e =
        cudaFuncSetAttribute(conv3x3_dw<S, COB>, cudaFuncAttributeMaxDynamicSharedMemorySize, S::kSmem);
    if (e != cudaSuccess) return e;
    return launch_kernel(conv3x3_dw<S, COB>, dim3((unsigned)shares, (unsigned)tiles), kDwThreads, S::kSmem, s, true, tz, tx,
                         H, boxes, cbs, ws);
}

}  // namespace

size_t conv_dw_workspace(int sms) { return (size_t)sms * 128 * kDwTile * sizeof(float); }

cudaError_t conv_dw_launch(const void* dZ, const void* X, int xcs, int T, int side, int cin, int cout, int sms, float* ws,
                           float* dW, cudaStream_t s)
{
    EncodeTiled enc = tensor_map_encoder();
    if (!enc) return cudaErrorNotSupported;
    const int cob = cout == 32 ? 1 : cout == 64 ? 2 : 4;
    if ((side != 64 || cob != 1) && (side != 32 || cob != 2) && ((side != 16 && side != 8) || cob != 4 || cout % 128))
        return cudaErrorInvalidValue;
    const int cbs = (cin + 31) / 32, tiles = cbs * (cout / (32 * cob));
    const int boxes = T * (side / kDwRows);
    const int shares = std::max(1, std::min(boxes, sms / tiles));  // of the pixels: a CTA for every SM
    if ((size_t)shares * tiles > (size_t)sms) return cudaErrorInvalidValue;  // the workspace holds `sms` tiles
    const cuuint32_t one[4] = {1, 1, 1, 1};
    auto map = [&](CUtensorMap* m, const void* p, int cs, int cols, int rows) {
        const cuuint64_t c = (cuuint64_t)cs, w = (cuuint64_t)side;
        const cuuint64_t d[4] = {c, w, w, (cuuint64_t)T};
        const cuuint64_t st[3] = {c * 2, w * c * 2, w * w * c * 2};
        const cuuint32_t box[4] = {32, (cuuint32_t)cols, (cuuint32_t)rows, 1};
        return enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(p), d, st, box, one,
                   CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                   CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
    };
    CUtensorMap tz, tx;
    if (!map(&tz, dZ, cout, side, kDwRows) || !map(&tx, X, xcs, side == 8 ? 16 : side + 2, kDwRows + 2)) return cudaErrorInvalidValue;
    cudaError_t e;
    if (side == 64) e = launch<64, 1, 3, 8>(tz, tx, side, boxes, tiles, cbs, shares, ws, s);
    else if (side == 32) e = launch<32, 2, 3, 4>(tz, tx, side, boxes, tiles, cbs, shares, ws, s);
    else if (side == 16) e = launch<16, 4, 4, 2>(tz, tx, side, boxes, tiles, cbs, shares, ws, s);
    else e = launch<8, 4, 4, 1>(tz, tx, side, boxes, tiles, cbs, shares, ws, s);
    if (e != cudaSuccess) return e;
    return launch_kernel(dw_reduce_kernel, dim3((unsigned)(tiles * (32 * cob * kDwTile / 128))), 256, 0, s, true, (const float*)ws, shares, 32 * cob, cbs, cin,
                         dW);
}

unsigned conv_dw_status_take()
{
    unsigned v = 0, z = 0;
    if (cudaMemcpyFromSymbol(&v, g_dw_status, sizeof v) != cudaSuccess ||
        cudaMemcpyToSymbol(g_dw_status, &z, sizeof z) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return v;
}

}  // namespace yoro
