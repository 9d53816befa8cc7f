// 3x3 convolution of the inpainter's wide, shallow layers (32 or 64 output channels on tiles
// 32, 64 or 128 pixels wide) on the tensor cores: the row form.
//
// What bounds these layers: one tcgen05.mma of M = 128 pixels x N = Cout x K = 16 reads its
// A tile (4 KB) and its weights (Cout x 32 bytes) from shared memory at 128 bytes per
// cycle, and one thread issues at most one MMA per ~55 cycles (measured), so at N = 32 the
// tensor core does 16 cycles of work per 55.  The three taps of a kernel column share
// their input, so here they share the MMA: M is one image row (128 / W images side by
// side, so the lanes of an accumulator are the same pixels of every row), the accumulators
// of R rows lie next to each other in tensor memory, and input row r is multiplied once
// with the weights of taps dy = 0, 1, 2 (N = 3 Cout) into the accumulators of rows r + 1, r,
// r - 1 (later rows lie in lower columns): 56 cycles where three MMAs took 164 (N = 96), 96
// where they took 164 (N = 192).
//
// The kernel columns share the copy of a row as well: tap dx reads the same shared-memory
// row from a start one pixel (64 bytes) to the left or right (the swizzle is a function
// of the shared-memory address, so any pixel start reads what the copy engine wrote), and
// the lanes whose neighbour lies outside the image (x = 0 for dx = 0, x = W - 1 for dx = 2)
// are left out by the MMA's lane mask, which is the convolution's zero padding.  A row is
// copied once per 32 channels, (R + 2) / R times in all, instead of three times that.
//
// Per output element the products are accumulated in the order (channel block, dx, dy,
// K half) of conv3x3_halo, so both forms give the same bits.
//
// One CTA per SM walks units of (image group, R rows).  Warp 0 streams rows (two per
// copy, 16 KB: a wait, an expect and a copy cost the issuing thread 300-450 cycles whatever
// the size) and weights (nine taps per copy), warp 1 issues the MMAs, warps 2-5 read back one of two accumulator sets (256
// columns each) while the other is being filled, zero it for its next use, and store: each
// warp stages its 32 pixels of two rows and writes them with its own TMA store.  Where the
// next level follows, the 2x2 maximum of the rows a warp holds goes to the pooled tensor
// in the same pass.
//
// The issuing warp runs its loop as a whole (one lane elected per instruction): in uniform
// control flow the descriptors are built in uniform registers, where a single-lane branch
// cost about 100 more cycles per MMA (155 against 56 at N = 96).
//
// Measured, 870 tiles, halo form -> row form as the network runs it, us: enc0a 143 -> 71, enc0b
// 144 -> 83 (with the pooling), enc1a 51 -> 33, enc1b 78 -> 49 (with the pooling), dec1a 166 ->
// 137 and dec0a 305 -> 186 (half-resolution input), dec1b 141 -> 46 (stored at its own
// resolution), dec0b 152 -> 95 (with the output layer).  enc0a moves its 405 MB at 5.7 TB/s;
// dec0a keeps the tensor pipe 43 % and shared memory 57 % busy, dec1a 59 and 59 % (304 tiles):
// neither unit is full, the one CTA's roles wait on one another.
#include <algorithm>
#include <cmath>

#include "tc.cuh"
#include "unet_device.cuh"
#include "unet_internal.h"

namespace yoro {

namespace {

__device__ unsigned g_rows_status;  // waits that ran out in this file's kernel

constexpr int kRowBytes = kTileM * kKc * 2;     // one row of 128 pixels x 32 channels
constexpr int kPairBytes = 2 * kRowBytes;       // rows are copied two at a time
constexpr int kAccCols = 256;                   // tensor-memory columns of an accumulator set
constexpr int kMaxPairs = 11;                   // row-pair slots (bounds the barrier array)
constexpr int kStageBytes = 2 * 32 * kKc * 2;   // a warp's 32 pixels of two rows, 32 channels
constexpr int kStores = 4 * 2 * kStageBytes;    // two staging buffers for each of four warps
// Warps: one copies, one issues MMAs, four read back and store; the output layer's epilogues
// take eight (its 96 products and sums per pixel kept four busy longer than the MMAs: dec0b on
// 870 tiles 127 us), an upsampled input one more that doubles its rows.
__host__ __device__ constexpr int epilogue_warps(int mode) { return mode >= 2 ? 8 : 4; }
__host__ __device__ constexpr int rows_threads(int mode, bool up) { return 64 + 32 * epilogue_warps(mode) + (up ? 32 : 0); }
constexpr int kLowBytes = kRowBytes / 2;        // a row of the half-resolution input: 64 pixels
constexpr int kLow = 6;                         // its landing slots

struct RowsArgs {
    int T, H, W, Cin;
    int pairs;         // row-pair slots
    int cskip;         // channels of the first input; the other Cin - cskip come from the half-resolution one
    int wslots;        // weight slots (9 taps of one channel block each); resident when wslots == Cin / 32
    int y_coff, upsample, relu;
    const float* bias;
    const int* count;  // optional: tiles at or after *count are skipped
    uint16_t* pool;    // kPool: T x H/2 x W/2 x Cout, the 2x2 maximum of the output
    const float* wout; // kColors, kCompose: the output layer
    float* rgb;        // kColors: T x H x W x 3
    const int* list;   // kCompose: the cells of the tiles
};

// What the epilogue does with a pixel's channels.
enum { kStore, kPool, kColors, kCompose };
static_assert(kColors == 2, "epilogue_warps()");

// One 32-channel slice of one pixel: bias, ReLU, rounding to bfloat16.
__device__ __forceinline__ void finish(const uint32_t (&r)[32], const float* bias, int relu, uint32_t (&q)[16])
{
#pragma unroll
    for (int i = 0; i < 16; ++i) {
        float v0 = __fadd_rn(__uint_as_float(r[2 * i]), bias[2 * i]);
        float v1 = __fadd_rn(__uint_as_float(r[2 * i + 1]), bias[2 * i + 1]);
        if (relu) {
            v0 = fmaxf(v0, 0.0f);
            v1 = fmaxf(v1, 0.0f);
        }
        q[i] = pack_bf16x2(v0, v1);
    }
}

struct NoFrames {};

// UP: the input is a concatenation of cskip channels at the layer's resolution (tmA) and the
// nearest upsampling of the rest (tmU, H/2 x W/2), which is never stored: a fifth kind of warp
// writes each of its rows, pixels doubled, into the row slots (8 KB of shared-memory writes),
// where it serves as both input rows it is upsampled to.  Written out and read back, the
// upsampled tensors were half of the memory traffic of the decoder's first layers and most of
// what the layers below them wrote.
template <int COUT, int R, int MODE, bool UP, class Frames>
__global__ void __launch_bounds__(rows_threads(MODE, UP), 1)
    conv3x3_rows(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                 const __grid_constant__ CUtensorMap tmY, const __grid_constant__ CUtensorMap tmU, const RowsArgs a,
                 const __grid_constant__ Frames ft)
{
    constexpr int kThreads = rows_threads(MODE, UP), kEpi = epilogue_warps(MODE);
    constexpr int kSkipSlots = (R + 2) / 2;             // slots of a channel block: rows -1 .. R
    constexpr int kLowRows = R / 2 + 2;                 // half-resolution rows under them
    constexpr int kUpSlots = (kLowRows + 1) / 2;
    extern __shared__ unsigned char smem_raw[];
    const int W = a.W, H = a.H, NP = a.pairs, WS = a.wslots;
    const int nimg = kTileM / W, bands = H / R;
    const int cb_n = a.Cin / kKc, cb_skip = UP ? a.cskip / kKc : cb_n;
    const int tiles = a.count ? min(a.T, *a.count) : a.T;
    const int units = (tiles + nimg - 1) / nimg * bands;
    if ((int)blockIdx.x >= units) return;  // uniform

    unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                                           ~static_cast<uintptr_t>(1023));
    // 1 KB of barriers first: the row before slot 0 that a dx = 0 operand starts 64 bytes into
    uint64_t* full = reinterpret_cast<uint64_t*>(smem);
    uint64_t* empty = full + kMaxPairs;
    uint64_t* wfull = empty + kMaxPairs;
    uint64_t* wempty = wfull + 4;
    uint64_t* afull = wempty + 4;
    uint64_t* aempty = afull + 2;
    uint64_t* lfull = aempty + 2;
    uint64_t* lempty = lfull + kLow;
    uint64_t* drain = lempty + kLow;
    uint32_t* tslot = reinterpret_cast<uint32_t*>(drain + 1);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tslot + 1);
    float* sbias = reinterpret_cast<float*>(smem + 480);  // COUT floats
    float* swout = reinterpret_cast<float*>(smem + 608);  // kColors, kCompose: 99 floats after 32 biases
    unsigned char* rows = smem + 1024;
    constexpr int kWBytes = 9 * COUT * kKc * 2;
    unsigned char* wts = rows + NP * kPairBytes;
    unsigned char* stage = wts + WS * kWBytes;
    unsigned char* land = stage + kStores;
    const bool resident = WS == cb_n;
    const int warp = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0), lane = threadIdx.x & 31;

    if (threadIdx.x == 0) {
        for (int s = 0; s < NP; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        for (int s = 0; s < WS && s < 4; ++s) {
            mbar_init(&wfull[s], 1);
            mbar_init(&wempty[s], 1);
        }
        for (int s = 0; s < 2; ++s) {
            mbar_init(&afull[s], 1);
            mbar_init(&aempty[s], kEpi);
        }
        for (int s = 0; s < kLow; ++s) {
            mbar_init(&lfull[s], 1);
            mbar_init(&lempty[s], 1);
        }
        mbar_init(drain, 1);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tslot)),
                     "r"(2 * kAccCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    for (int c = threadIdx.x; c < COUT; c += kThreads) sbias[c] = __ldg(a.bias + c);
    if (MODE == kColors || MODE == kCompose)
        for (int c = threadIdx.x; c < 99; c += kThreads) swout[c] = __ldg(a.wout + c);
    pdl_wait();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tslot;

    auto timed_out = [&]() {
        atomicOr(&g_rows_status, kUnetTimeout);
        *abort_flag = 1;
    };
    // what thread 0 has copied: row slots (bits) and the parity of their last copy's phase; counts
    uint32_t copied = 0u, parity = 0u;
    int wissued = 0, lissued = 0;

    if (warp == 0) {
        if (lane == 0) {  // copies
            int slot = 0, ph = 1, ws = 0, wph = 1, ls = 0, lph = 1;
            bool ok = true;
            for (int u = blockIdx.x; u < units && ok; u += gridDim.x) {
                const int g = u / bands, y0 = (u - g * bands) * R;
                const uint64_t deadline = globaltimer() + kWaitNs;
                for (int cb = 0; cb < cb_n && ok; ++cb) {
                    if (!resident || u == (int)blockIdx.x) {
                        if (!(ok = mbar_wait(&wempty[ws], wph, deadline))) break;
                        mbar_expect_tx(&wfull[ws], kWBytes);
                        tma_load_4d(wts + ws * kWBytes, &tmB, &wfull[ws], cb * kKc, 0, 0, 0);  // all nine taps
                        ++wissued;
                        if (++ws == WS) {
                            ws = 0;
                            wph ^= 1;
                        }
                    }
                    // rows -1 and H arrive as zeros
                    if (UP && cb >= cb_skip) {
                        for (int i = 0; i < kLowRows; ++i) {
                            if (!(ok = mbar_wait(&lempty[ls], lph, deadline))) break;
                            mbar_expect_tx(&lfull[ls], kLowBytes);
                            tma_load_4d(land + ls * kLowBytes, &tmU, &lfull[ls], (cb - cb_skip) * kKc, 0, g * nimg,
                                        y0 / 2 - 1 + i);
                            ++lissued;
                            if (++ls == kLow) {
                                ls = 0;
                                lph ^= 1;
                            }
                        }
                        for (int i = 0; i < kUpSlots; ++i)  // filled by the doubling warp
                            if (++slot == NP) {
                                slot = 0;
                                ph ^= 1;
                            }
                        continue;
                    }
                    for (int r = -1; r <= R; r += 2) {
                        if (!(ok = mbar_wait(&empty[slot], ph, deadline))) break;
                        mbar_expect_tx(&full[slot], kPairBytes);
                        tma_load_4d(rows + slot * kPairBytes, &tmA, &full[slot], cb * kKc, 0, g * nimg, y0 + r);
                        copied |= 1u << slot;
                        parity = (parity & ~(1u << slot)) | ((uint32_t)(ph ^ 1) << slot);
                        if (++slot == NP) {
                            slot = 0;
                            ph ^= 1;
                        }
                    }
                }
            }
            if (!ok) timed_out();
        }
    } else if (warp == 1) {  // MMAs: the whole warp runs the loop, one lane issues
        constexpr uint32_t id1 = idesc_bf16(COUT), id2 = idesc_bf16(2 * COUT), id3 = idesc_bf16(3 * COUT);
        const uint32_t el = elect_one();
        const uint64_t drow = desc_sw64(smem_u32(rows));
        const uint64_t dw = desc_sw64(smem_u32(wts));
        // lanes x = 0 and x = W - 1 of each image
        const uint32_t lo2 = W == 128 ? 0u : 1u, lo13 = W == 32 ? 1u : 0u;
        const uint32_t hi3 = 0x80000000u, hi1 = W == 128 ? 0u : hi3, hi02 = W == 32 ? hi3 : 0u;
        // false once a wait ran out.  Every value below is the same in all lanes and no issue
        // hangs on a condition that only a vote makes uniform, so the loop stays in the uniform
        // datapath.
        auto issue_all = [&]() -> bool {
            int slot0 = 0, ph0 = 0, ws = 0, wph = 0, it = 0;
            for (int u = blockIdx.x; u < units; u += gridDim.x, ++it) {
                const int g = u / bands, y0 = (u - g * bands) * R;
                const bool top = y0 == 0, bottom = y0 + R == H;  // row -1 or R lies outside the image
                const uint32_t acc = tmem + (uint32_t)((it & 1) * kAccCols);
                const uint64_t deadline = globaltimer() + kWaitNs;
                if (!mbar_wait_warp(&aempty[it & 1], (it >> 1) & 1, deadline)) return false;
                tc_fence_after();
                for (int cb = 0; cb < cb_n; ++cb) {
                    if (resident) ws = cb;
                    if (!resident || it == 0)
                        if (!mbar_wait_warp(&wfull[ws], wph, deadline)) return false;
                    const bool up = UP && cb >= cb_skip;
                    int slot = slot0, ph = ph0;
#pragma unroll
                    for (int dx = 0; dx < 3; ++dx) {
                        const uint32_t m0 = dx == 0 ? 1u : dx == 2 ? hi02 : 0u;
                        const uint32_t m1 = dx == 0 ? lo13 : dx == 2 ? hi1 : 0u;
                        const uint32_t m2 = dx == 0 ? lo2 : dx == 2 ? hi02 : 0u;
                        const uint32_t m3 = dx == 0 ? lo13 : dx == 2 ? hi3 : 0u;
                        const uint64_t wb = dw + (uint64_t)((uint32_t)(ws * kWBytes + dx * 3 * COUT * kKc * 2) >> 4);
                        slot = slot0;
                        ph = ph0;
                        // input row r, in row `half` of the current slot, into output rows r + 1 .. r - 1
                        // inside the unit (ascending columns)
                        auto row = [&](int r, int half) {
                            const int lo = r < 1 ? 0 : r - 1, hi = r + 1 > R - 1 ? R - 1 : r + 1, n = hi - lo + 1;
                            const uint32_t id = n == 3 ? id3 : n == 2 ? id2 : id1;
                            const uint64_t da = drow + (uint64_t)((uint32_t)slot * (uint32_t)(kPairBytes >> 4) +
                                                                  (uint32_t)(half * (kRowBytes >> 4) + 4 * dx)) - 4;
                            const uint64_t db = wb + (uint64_t)((r + 1 - hi) * (COUT * kKc * 2 >> 4));
                            const uint32_t d = acc + (uint32_t)((R - 1 - hi) * COUT);
                            mma_bf16_masked(el, d, da, db, id, m0, m1, m2, m3);
                            mma_bf16_masked(el, d, da + 2, db + 2, id, m0, m1, m2, m3);
                        };
                        auto next = [&]() {
                            if (dx == 2) mma_commit_elected(el, &empty[slot]);
                            if (++slot == NP) {
                                slot = 0;
                                ph ^= 1;
                            }
                        };
                        if (!up) {
#pragma unroll
                            for (int r = -1; r <= R; ++r) {
                                const bool second = (r & 1) == 0;  // of the pair in this slot
                                if (dx == 0 && !second) {
                                    if (!mbar_wait_warp(&full[slot], ph, deadline)) return false;
                                    tc_fence_after();
                                }
                                if (!(r == -1 && top) && !(r == R && bottom)) row(r, second ? 1 : 0);
                                if (second) next();
                            }
                        } else {
                            // half-resolution row i = 0 .. kLowRows - 1 of the unit, in row i & 1 of its slot,
                            // is input rows 2i - 2 and 2i - 1
#pragma unroll
                            for (int i = 0; i < kLowRows; ++i) {
                                if (dx == 0 && !(i & 1)) {
                                    if (!mbar_wait_warp(&full[slot], ph, deadline)) return false;
                                    tc_fence_after();
                                }
#pragma unroll
                                for (int r = 2 * i - 2; r <= 2 * i - 1; ++r)
                                    if (r >= -1 && r <= R && !(r == -1 && top) && !(r == R && bottom)) row(r, i & 1);
                                if ((i & 1) || i == kLowRows - 1) next();
                            }
                        }
                    }
                    slot0 = slot;
                    ph0 = ph;
                    if (!resident) {
                        mma_commit_elected(el, &wempty[ws]);
                        if (++ws == WS) {
                            ws = 0;
                            wph ^= 1;
                        }
                    }
                }
                mma_commit_elected(el, &afull[it & 1]);
            }
            return true;
        };
        const bool ok = issue_all();
        if (!ok) {  // the MMAs issued so far: wait for them (bounded)
            if (el) timed_out();
            mma_commit_elected(el, drain);
            mbar_wait_warp(drain, 0, globaltimer() + kWaitNs);
        }
    } else if (UP && warp == 6) {  // doubles the half-resolution rows
        int slot = 0, ph = 1, ls = 0, lph = 0;
        bool ok = true;
        for (int u = blockIdx.x; u < units && ok; u += gridDim.x) {
            const uint64_t deadline = globaltimer() + kWaitNs;
            for (int cb = 0; cb < cb_n && ok; ++cb) {
                const bool up = cb >= cb_skip;
                for (int t = 0; t < (up ? kUpSlots : kSkipSlots); ++t) {
                    if (up) {
                        if (!(ok = mbar_wait_warp(&empty[slot], ph, deadline))) break;
                        for (int half = 0; half < 2 && 2 * t + half < kLowRows; ++half) {
                            if (!(ok = mbar_wait_warp(&lfull[ls], lph, deadline))) break;
                            const unsigned char* src = land + ls * kLowBytes;
                            unsigned char* dst = rows + slot * kPairBytes + half * kRowBytes;
#pragma unroll
                            for (int i = 0; i < 8; ++i) {  // 16-byte chunk e & 3 of pixel e >> 2, twice
                                const int e = i * 32 + lane, q = e >> 2, k = e & 3;
                                const uint4 v = *reinterpret_cast<const uint4*>(src + q * 64 + ((k ^ ((q >> 1) & 3)) << 4));
                                unsigned char* o = dst + q * 128 + ((k ^ (q & 3)) << 4);
                                *reinterpret_cast<uint4*>(o + (q & 1) * 64) = v;  // odd q the other way round:
                                *reinterpret_cast<uint4*>(o + 64 - (q & 1) * 64) = v;  // no bank met twice
                            }
                            __syncwarp();
                            if (lane == 0) mbar_arrive(&lempty[ls]);
                            if (++ls == kLow) {
                                ls = 0;
                                lph ^= 1;
                            }
                        }
                        if (!ok) break;
                        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                        __syncwarp();
                        if (lane == 0) mbar_arrive(&full[slot]);
                    }
                    if (++slot == NP) {
                        slot = 0;
                        ph ^= 1;
                    }
                }
            }
        }
        if (!ok && lane == 0) timed_out();
    } else {  // read back, store
        const int q = warp & 3;  // this warp's quarter of the tensor-memory lanes
        const uint32_t tq = tmem + ((uint32_t)(q * 32) << 16);
        for (int c = 0; c < 2 * kAccCols; c += 32) tmem_zero32_async(tq + c);
        tmem_wait_st();
        tc_fence_before();
        if (lane == 0) {
            mbar_arrive(&aempty[0]);
            mbar_arrive(&aempty[1]);
        }
        unsigned char* st = stage + (warp - 2) * 2 * kStageBytes;
        const int img = W == 32 ? q : W == 64 ? q >> 1 : 0;           // image of the group
        const int x0 = W == 32 ? 0 : W == 64 ? (q & 1) * 32 : q * 32;  // first pixel of the row
        int it = 0, nst = 0;
        for (int u = blockIdx.x; u < units; u += gridDim.x, ++it) {
            const int g = u / bands, y0 = (u - g * bands) * R;
            const int n = g * nimg + img;
            const uint32_t acc = tq + (uint32_t)((it & 1) * kAccCols);
            bool ok = mbar_wait(&afull[it & 1], (it >> 1) & 1, globaltimer() + 2 * kWaitNs);
            ok = __all_sync(0xffffffffu, ok);
            if (!ok || *abort_flag) {
                if (!ok && lane == 0) timed_out();
                break;
            }
            __syncwarp();
            tc_fence_after();
            if constexpr (MODE == kColors || MODE == kCompose) {  // the output layer, a row of pixels at a time
                bool live = n < tiles;
                float* rgb = nullptr;
                const uint8_t* mask = nullptr;
                uint32_t* rgba = nullptr;
                int pitch = 0, r0 = 0, r1 = R;  // rows of the unit that are written
                if constexpr (MODE == kColors) {
                    rgb = a.rgb + (((size_t)n * H + y0) * W + x0 + lane) * 3;
                } else if (live) {
                    const int cell = a.list[n];
                    const int f = table_frame(ft, cell), tile = cell - ft.off[f];
                    const int tx = tile % ft.ntx[f], ty = tile / ft.ntx[f];
                    const int gx = window_origin(tx, ft.w[f]) + x0 + lane, gy = window_origin(ty, ft.h[f]) + y0;
                    // the pixels of the window outside the cell belong to the neighbouring tile
                    live = gx >= kTile * tx && gx < ft.w[f];
                    r0 = max(0, kTile * ty - gy);
                    r1 = min(R, ft.h[f] - gy);
                    pitch = ft.w[f];
                    mask = ft.mask[f] + (ptrdiff_t)gy * pitch + gx;
                    rgba = ft.rgba[f] + (ptrdiff_t)gy * pitch + gx;
                }
                // the two groups of four warps take every other row
#pragma unroll 1
                for (int r = (warp - 2) >> 2; r < R; r += kEpi / 4) {
                    uint32_t v[32], p[16];
                    const uint32_t t = acc + (uint32_t)((R - 1 - r) * COUT);
                    tmem_ld32_async(t, v);
                    bool put = live && r >= r0 && r < r1;
                    if constexpr (MODE == kCompose) {  // hole pixels only
                        put = put && mask[(ptrdiff_t)r * pitch];
                    }
                    tmem_wait_ld();
                    tmem_zero32_async(t);
                    if (!__any_sync(0xffffffffu, put)) continue;
                    finish(v, sbias, a.relu, p);
                    float x[32], col[3];
#pragma unroll
                    for (int i = 0; i < 16; ++i) {
                        x[2 * i] = __uint_as_float(p[i] << 16);
                        x[2 * i + 1] = __uint_as_float(p[i] & 0xffff0000u);
                    }
                    net_colors(x, swout, col);
                    if (put) {
                        if constexpr (MODE == kColors) {
                            float* o = rgb + (size_t)r * W * 3;
                            o[0] = col[0];
                            o[1] = col[1];
                            o[2] = col[2];
                        } else {
                            rgba[(ptrdiff_t)r * pitch] = net_rgba(col);
                        }
                    }
                }
            }
            for (int rr = 0; rr < R && MODE < kColors; rr += 2) {
#pragma unroll
                for (int c0 = 0; c0 < COUT; c0 += 32) {
                    uint32_t v0[32], v1[32];
                    const uint32_t t0 = acc + (uint32_t)((R - 1 - rr) * COUT + c0), t1 = t0 - COUT;
                    tmem_ld32_async(t0, v0);
                    tmem_ld32_async(t1, v1);
                    tmem_wait_ld();
                    tmem_zero32_async(t0);
                    tmem_zero32_async(t1);
                    uint32_t p0[16], p1[16];
                    finish(v0, sbias + c0, a.relu, p0);
                    finish(v1, sbias + c0, a.relu, p1);
                    // a staging buffer is free once the store issued from it two slices ago has read it
                    unsigned char* sb = st + (nst & 1) * kStageBytes;
                    if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");
                    __syncwarp();
                    const int sw = (lane >> 1) & 3;
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        *reinterpret_cast<uint4*>(sb + lane * 64 + ((k ^ sw) << 4)) =
                            make_uint4(p0[4 * k], p0[4 * k + 1], p0[4 * k + 2], p0[4 * k + 3]);
                        *reinterpret_cast<uint4*>(sb + 2048 + lane * 64 + ((k ^ sw) << 4)) =
                            make_uint4(p1[4 * k], p1[4 * k + 1], p1[4 * k + 2], p1[4 * k + 3]);
                    }
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                    __syncwarp();
                    if (lane == 0) {
                        if (n < a.T) {
                            if (!a.upsample) {
                                tma_store_4d(&tmY, sb, a.y_coff + c0, x0, n, y0 + rr);
                            } else {
#pragma unroll
                                for (int ab = 0; ab < 4; ++ab)
                                    tma_store_5d(&tmY, sb, a.y_coff + c0, ab & 1, x0, ab >> 1, n * H + y0 + rr);
                            }
                        }
                        asm volatile("cp.async.bulk.commit_group;" ::: "memory");
                    }
                    ++nst;
                    if constexpr (MODE == kPool) {  // 2x2 maximum: the two rows, then the neighbouring pixel
#pragma unroll
                        for (int i = 0; i < 16; ++i) {
                            const uint32_t m = max_bf16x2(p0[i], p1[i]);
                            p0[i] = max_bf16x2(m, __shfl_xor_sync(0xffffffffu, m, 1));
                        }
                        if (n < a.T) {  // lanes 2i and 2i + 1 write 16 bytes of each 32 of pooled pixel i
                            const size_t px = ((size_t)n * (H / 2) + ((y0 + rr) >> 1)) * (W / 2) + ((x0 + lane) >> 1);
                            uint4* dst = reinterpret_cast<uint4*>(a.pool + px * COUT + c0) + (lane & 1);
#pragma unroll
                            for (int k = 0; k < 2; ++k)
                                dst[2 * k] = (lane & 1) ? make_uint4(p0[8 * k + 4], p0[8 * k + 5], p0[8 * k + 6], p0[8 * k + 7])
                                                        : make_uint4(p0[8 * k], p0[8 * k + 1], p0[8 * k + 2], p0[8 * k + 3]);
                        }
                    }
                }
            }
            tmem_wait_st();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&aempty[it & 1]);
        }
        if (lane == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
    }
    __syncwarp();
    tc_fence_before();
    __syncthreads();
    if (threadIdx.x == 0 && *abort_flag) {  // copies still in flight after a timeout: wait for them (bounded)
        const uint64_t d = globaltimer() + kWaitNs;
        for (int i = 0; i < NP; ++i)
            if ((copied >> i) & 1u) mbar_wait(&full[i], (parity >> i) & 1u, d);
        for (int i = max(0, lissued - kLow); i < lissued; ++i) mbar_wait(&lfull[i % kLow], (i / kLow) & 1, d);
        for (int i = max(0, wissued - WS); i < wissued; ++i) mbar_wait(&wfull[i % WS], (i / WS) & 1, d);
    }
    __syncthreads();
    if (warp == 1) {  // the allocating warp frees
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(2 * kAccCols) : "memory");
    }
}

size_t rows_smem(int pairs, int wslots, int cout, bool up)
{
    return 2048 + (up ? kLow * kLowBytes : 0) + (size_t)pairs * kPairBytes + (size_t)wslots * 9 * cout * kKc * 2 + kStores;
}

}  // namespace

// 16-pixel rows and 128 channels stay with the halo form: at N = 128 an MMA already does 64
// cycles of work for 64 of operand reads, so sharing it between taps gains nothing.  The
// form wins at every tile count measured (T = 64: dec0a 33.9 -> 25.0 us, enc0b 18.8 -> 14.9;
// at T = 2 and 8 both are bound by the call, 11-12 us).
bool conv_rows_takes(int H, int W, int Cout)
{
    return (W == 32 || W == 64 || W == 128) && (Cout == 32 || Cout == 64) && H % 2 == 0;
}

cudaError_t conv_rows_launch(const ConvCall& c, int sms, int smem_max, cudaStream_t stream)
{
    EncodeTiled enc = tensor_map_encoder();
    if (!enc) return cudaErrorNotSupported;
    const int nimg = kTileM / c.W, groups = (c.T + nimg - 1) / nimg;
    RowsArgs a;
    a.T = c.T;
    a.H = c.H;
    a.W = c.W;
    a.Cin = c.Cin;
    // rows of a unit: an accumulator set's 256 columns, fewer while that leaves SMs without a unit
    int R = kAccCols / c.Cout;
    while (c.H % R) R /= 2;
    while (R > 2 && groups * (c.H / R) < sms) R /= 2;
    const bool up = c.low != nullptr;
    if (up && (c.rgb || c.frames || c.pool || c.W > 64 || c.cskip < kKc || c.cskip % kKc || c.cskip >= c.Cin))
        return cudaErrorInvalidValue;
    a.cskip = c.cskip;
    const int cb_n = c.Cin / kKc;
    a.wslots = cb_n <= 3 && 9 * c.Cin * c.Cout * 2 <= 80 * 1024 ? cb_n : 2;
    a.pairs = std::min(kMaxPairs, (int)((smem_max - (int)rows_smem(0, a.wslots, c.Cout, up)) / kPairBytes));
    if (2 * a.pairs < R + 2) return cudaErrorInvalidValue;
    a.y_coff = c.y_coff;
    a.upsample = c.upsample;
    a.relu = c.relu;
    a.bias = c.bias;
    a.count = c.count;
    a.pool = static_cast<uint16_t*>(c.pool);
    a.wout = c.wout;
    a.rgb = c.rgb;
    a.list = c.list;
    if ((c.rgb || c.frames) && (c.Cout != 32 || c.upsample || c.pool)) return cudaErrorInvalidValue;

    CUtensorMap ta, tb, ty, tu;
    const cuuint32_t one[5] = {1, 1, 1, 1, 1};
    // {channel, x, image, y}: a box of two rows of nimg images is 2 x 128 consecutive pixels
    const cuuint64_t ci = (cuuint64_t)c.Cin, W = (cuuint64_t)c.W, H = (cuuint64_t)c.H, T = (cuuint64_t)c.T;
    const cuuint64_t ca = up ? (cuuint64_t)c.cskip : ci;
    const cuuint64_t ad[4] = {ca, W, T, H};
    const cuuint64_t as[3] = {ca * 2, H * W * ca * 2, W * ca * 2};
    const cuuint32_t abox[4] = {(cuuint32_t)kKc, (cuuint32_t)c.W, (cuuint32_t)nimg, 2};
    if (enc(&ta, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(c.x), ad, as, abox, one,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
        return cudaErrorInvalidValue;
    tu = ta;  // unused without a half-resolution input
    if (up) {  // the same of one half-resolution row: 64 pixels
        const cuuint64_t cu = ci - ca, Wl = W / 2, Hl = H / 2;
        const cuuint64_t ud[4] = {cu, Wl, T, Hl};
        const cuuint64_t us[3] = {cu * 2, Hl * Wl * cu * 2, Wl * cu * 2};
        const cuuint32_t ubox[4] = {(cuuint32_t)kKc, (cuuint32_t)Wl, (cuuint32_t)nimg, 1};
        if (enc(&tu, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(c.low), ud, us, ubox, one,
                CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return cudaErrorInvalidValue;
    }
    // {channel, co, dy, dx}: a box of all taps lands as the three dy blocks of each dx
    const cuuint64_t bd[4] = {ci, (cuuint64_t)c.Cout, 3, 3};
    const cuuint64_t bs[3] = {9 * ci * 2, 3 * ci * 2, ci * 2};
    const cuuint32_t bbox[4] = {(cuuint32_t)kKc, (cuuint32_t)c.Cout, 3, 3};
    if (enc(&tb, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(c.wk), bd, bs, bbox, one,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
        return cudaErrorInvalidValue;
    // a store's box: 32 channels x 32 pixels x two rows of one image
    const cuuint64_t cs = (cuuint64_t)c.y_cstride;
    CUresult r = CUDA_SUCCESS;
    if (c.rgb || c.frames) {
        ty = ta;  // nothing is stored
    } else if (!c.upsample) {
        const cuuint64_t d[4] = {cs, W, T, H};
        const cuuint64_t s[3] = {cs * 2, H * W * cs * 2, W * cs * 2};
        const cuuint32_t box[4] = {(cuuint32_t)kKc, 32, 1, 2};
        r = enc(&ty, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, c.y, d, s, box, one, CU_TENSOR_MAP_INTERLEAVE_NONE,
                CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    } else {  // {channel, b, x, a, n H + y}: pixel (2y + a, 2x + b)
        const cuuint64_t d[5] = {cs, 2, W, 2, T * H};
        const cuuint64_t s[4] = {cs * 2, 2 * cs * 2, 2 * W * cs * 2, 4 * W * cs * 2};
        const cuuint32_t box[5] = {(cuuint32_t)kKc, 1, 32, 1, 2};
        r = enc(&ty, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, c.y, d, s, box, one, CU_TENSOR_MAP_INTERLEAVE_NONE,
                CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    }
    if (r != CUDA_SUCCESS) return cudaErrorInvalidValue;

    const size_t smem = rows_smem(a.pairs, a.wslots, c.Cout, up);
    const int grid = std::min(groups * (c.H / R), sms);
    auto go = [&](auto kernel, const auto& frames) -> cudaError_t {
        const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_max);
        if (e != cudaSuccess) return e;
        return launch_kernel(kernel, dim3((unsigned)grid), rows_threads(c.frames || c.rgb ? kColors : kStore, up), smem,
                           stream, c.pdl, ta, tb, ty, tu, a, frames);
    };
    const NoFrames none;
#define YORO_ROWS32(MODE, FRAMES, TABLE)                                \
    (R == 8   ? go(conv3x3_rows<32, 8, MODE, false, FRAMES>, TABLE)            \
     : R == 4 ? go(conv3x3_rows<32, 4, MODE, false, FRAMES>, TABLE)            \
              : go(conv3x3_rows<32, 2, MODE, false, FRAMES>, TABLE))
    if (up) {
        if (c.Cout == 64)
            return R == 4 ? go(conv3x3_rows<64, 4, kStore, true, NoFrames>, none)
                          : go(conv3x3_rows<64, 2, kStore, true, NoFrames>, none);
        return R == 8   ? go(conv3x3_rows<32, 8, kStore, true, NoFrames>, none)
               : R == 4 ? go(conv3x3_rows<32, 4, kStore, true, NoFrames>, none)
                        : go(conv3x3_rows<32, 2, kStore, true, NoFrames>, none);
    }
    if (c.Cout == 64) {
        if (c.pool) return R == 4 ? go(conv3x3_rows<64, 4, kPool, false, NoFrames>, none) : go(conv3x3_rows<64, 2, kPool, false, NoFrames>, none);
        return R == 4 ? go(conv3x3_rows<64, 4, kStore, false, NoFrames>, none) : go(conv3x3_rows<64, 2, kStore, false, NoFrames>, none);
    }
    if (c.frames) return YORO_ROWS32(kCompose, FrameTable, *c.frames);
    if (c.rgb) return YORO_ROWS32(kColors, NoFrames, none);
    if (c.pool) return YORO_ROWS32(kPool, NoFrames, none);
    return YORO_ROWS32(kStore, NoFrames, none);
#undef YORO_ROWS32
}

unsigned conv_rows_status_take()
{
    unsigned v = 0, z = 0;
    if (cudaMemcpyFromSymbol(&v, g_rows_status, sizeof v) != cudaSuccess ||
        cudaMemcpyToSymbol(g_rows_status, &z, sizeof z) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return v;
}

}  // namespace yoro
