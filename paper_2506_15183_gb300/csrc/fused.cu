// Fused second-eye synthesis kernel for GB300 (sm_103a).
//
// One CTA synthesizes a band of B output rows at once; shared memory holds the
// band's warped rows plus the kernel's halo rows above and below (the window; one halo
// row per side for the paper's 3-row kernel): per target pixel a 32-bit word that is
// first the source column and then the depth, a 32-bit RGBA8 word, a reached bit, and
// per 32-pixel word a hole prefix sum.  The steps, separated by CTA barriers:
//
//   0.  one warp starts 1-D bulk prefetches of the window's depth and color rows
//       into L2 (cp.async.bulk.prefetch.L2), while all threads clear the window;
//   P1  disparity + forward warp (Alg. 1 closed form, Alg. 2 nearest kept): every
//       source pixel of every window row takes the atomic maximum of its source
//       column into its target's word (O1: a row never writes another row).  In a
//       row, of two sources that reach the same target the one further right is
//       the nearer (see scatter_window), so the maximum column is the z-test's
//       winner.  A thread takes whole columns (two, five rows of each per load
//       group) where they split evenly over the threads, else pixels round-robin;
//   P2  resolve + gather: each reached target loads its source's depth and color;
//       warp ballots write the rows' reached-pixel bitmasks, and the band rows'
//       reached pixels and hole mask leave for global memory at once;
//   P3a per band row: its last reached pixel, the border holes right of it (the
//       fallback), and per word the counts of cracks and wider holes with prefix sums;
//   P3b the other holes are filled (Alg. 3, Eq. 6) in chunks dealt to whichever warp
//       is free (32 pixels of wider holes, one per lane, or 64 one-pixel cracks, two
//       per lane), so a wide disocclusion is spread over many warps; a chunk inside
//       one hole is filled by the whole warp together.  Hole
//       edges and kernel candidates come from the bitmasks (leading/trailing-zero
//       counts over 32-pixel words).
//
// No thread ever waits on another CTA or on an asynchronous copy: the prefetches
// only warm L2, and every read is an ordinary load.
#include <cuda_runtime.h>

#include <cstdint>
#include <type_traits>

#include "yoro_device.cuh"
#include "yoro_internal.h"

namespace yoro {

namespace {

#ifdef YORO_DEBUG_BOUNDS
__device__ unsigned g_status;  // debug-bounds status word of this file's kernels
__device__ __forceinline__ void yoro_status_record(unsigned code) { atomicOr(&g_status, code); }
#endif

// Records kSelfTest in the debug-bounds build (no memory is touched); nothing otherwise.
__global__ void selftest_kernel()
{
    if (threadIdx.x == 0) (void)YORO_BOUND(false, kSelfTest);
}

// Remaining weight below which the exact early exit is tested after each contribution
// (2^-9: measured fastest among 2^-8 .. 2^-15 on the 1832x1920 workload).
constexpr float kSettleFrom = 0.001953125f;

__device__ __forceinline__ void prefetch_l2(const void* p, uint32_t bytes)
{
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(bytes) : "memory");
}

// The band window in shared memory.  Window row j (frame row ra + j) has its words at
// zt + j*wpad (source column during P1, -1 for none; clamped depth bits of the source
// after P2), rgba + j*wpad (color of the source after P2) and its reached bitmask at
// bits + j*nwords.
struct Window {
    uint32_t* zt;
    uint32_t* rgba;
    uint32_t* bits;
    uint32_t* pre;  // band row vj's hole prefix sums per word at pre + vj*nwords
    uint32_t* zmax; // fills with ZMAX: per word of window row j, its largest reached depth (bits; 0: none)
    int wpad, nwords, ra, slots;
    __device__ __forceinline__ const uint32_t* zrow(int v) const { return zt + (v - ra) * wpad; }
    __device__ __forceinline__ const uint32_t* crow(int v) const { return rgba + (v - ra) * wpad; }
    __device__ __forceinline__ const uint32_t* brow(int v) const { return bits + (v - ra) * nwords; }
};

// The Patcher's kernel shape (Sec. Patcher): rows v - halo .. v + halo (the kernel
// height h = 2 halo + 1, the paper's default 3) and the column order in each row:
// farthest first, min(R + w, W - 1) down to R (the paper's order, mirrored), or nearest
// first, R up.  VAR = false compiles the paper's defaults as constants; VAR = true
// takes them from the frame (the variant launch).
template <bool VAR>
struct KernelShape {
    int halo;
    bool nearest;
    __device__ __forceinline__ explicit KernelShape(const FrameArgs& f)
        : halo(VAR ? f.halo : 1), nearest(VAR ? f.nearest != 0 : false)
    {
    }
};

// Hole edges of pixel (v, x): L = highest reached column < x (or -1), R = lowest
// reached column > x (or w), from the row's reached bitmask.
__device__ __forceinline__ void find_edges(int x, int v, const Window& s, int w, int& L, int& R)
{
    const uint32_t* bv = s.brow(v);
    L = -1;
    {
        int wi = x >> 5;
        uint32_t m = bv[wi] & ((1u << (x & 31)) - 1u);
        for (;;) {
            if (m) {
                L = (wi << 5) + 31 - __clz(m);
                break;
            }
            if (--wi < 0) break;
            m = bv[wi];
        }
    }
    R = w;  // bits past the row end are zero
    {
        int wi = x >> 5;
        uint32_t m = ((x & 31) == 31) ? 0u : (bv[wi] & (~0u << ((x & 31) + 1)));
        for (;;) {
            if (m) {
                R = (wi << 5) + __ffs(m) - 1;
                break;
            }
            if (++wi >= s.nwords) break;
            m = bv[wi];
        }
    }
}

// Hole fill of pixel (v, x) with edges L, R (R < w).  Rows outside [0, h) are skipped.
// ZMAX: words whose reached pixels are all foreground are passed over by their largest depth.
// The stereo pair's holes are narrow (24 candidates walked at the 99th percentile), but where
// the second eye is rotated or shifted out of its row, holes up to 900 columns wide lie
// beside wide occluders and their kernels hold more than a thousand foreground candidates;
// walked one by one they kept single bands' CTAs busy for 100 us (figures at fill_keys).
template <bool VAR, bool ZMAX>
__device__ __forceinline__ uint32_t fill_from_edges(int x, int v, int L, int R, int h, int w, const Window& s,
                                                    const KernelShape<VAR>& ks)
{
    const int wd = R - L;
    const float d_occ = (L >= 0) ? __uint_as_float(s.zrow(v)[L]) : 0.0f;
    FillAcc f;
    f.init(__fdiv_rn((float)(R - x), (float)wd));
    const int jhi = min(R + wd, w - 1);
    const int whi = jhi >> 5, wlo = R >> 5;
    const uint32_t mhi = ((jhi & 31) == 31) ? ~0u : ((2u << (jhi & 31)) - 1u);
    const uint32_t mlo = ~0u << (R & 31);
#pragma unroll 1
    for (int vv = v - ks.halo; vv <= v + ks.halo; ++vv) {
        if (vv < 0 || vv >= h || !YORO_BOUND(vv - s.ra >= 0 && vv - s.ra < s.slots, kBadHoles)) continue;
        const uint32_t* b = s.brow(vv);
        const uint32_t* zr = s.zrow(vv);
        const uint32_t* cr = s.crow(vv);
#pragma unroll 1
        for (int step = 0; step <= whi - wlo; ++step) {
            const int wi = ks.nearest ? wlo + step : whi - step;
            if (ZMAX && YORO_BOUND(wi >= 0 && wi < s.nwords, kBadHoles) &&
                __uint_as_float(s.zmax[(vv - s.ra) * s.nwords + wi]) < d_occ)
                continue;
            uint32_t m = b[wi];
            if (wi == whi) m &= mhi;
            if (wi == wlo) m &= mlo;
            while (m) {
                const int bit = ks.nearest ? __ffs(m) - 1 : 31 - __clz(m);
                m &= ~(1u << bit);
                const int c = (wi << 5) + bit;
                if (__uint_as_float(zr[c]) < d_occ) continue;  // foreground (O2)
                if (!f.add(cr[c])) return f.result();          // weight reached exactly 0
                uint32_t out;
                if (f.wrem <= kSettleFrom && f.settled(out)) return out;
            }
        }
    }
    return f.any() ? f.result() : s.crow(v)[R];
}

// Hole fill of the pixels x of one hole (row v, edges L, R with R < w), one per active
// lane, by the whole warp.  The depth gate and the candidates are the same for every
// pixel of the hole, so the warp tests 32 kernel columns at a time (ballot of the
// contributing ones) and hands each contributor's color, in Alg. 3's order, to all
// lanes; each lane accumulates it with its own t and stops at its own exact exit.  A
// kernel full of foreground candidates is thus crossed 32 columns per step instead of
// one candidate per step.
//
// ZMAX: 32 words per step by their largest depth first, then the columns of those that are not
// all foreground.  The two forms are written out apart: with the contributor test and the
// accumulation shared between them as lambdas the form without ZMAX took up to 17 % longer on
// whole frames with wide holes (1439x1601, 24 seeds: up to 5.8 us more on three, the others
// the same).
template <bool VAR, bool ZMAX>
__device__ __forceinline__ uint32_t fill_hole_warp(int x, bool act, int v, int L, int R, int h, int w,
                                                   const Window& s, const KernelShape<VAR>& ks)
{
    const int lane = threadIdx.x & 31;
    const int wd = R - L;
    const float d_occ = (L >= 0) ? __uint_as_float(s.zrow(v)[L]) : 0.0f;
    FillAcc f;
    f.init(__fdiv_rn((float)(R - (act ? x : L + 1)), (float)wd));
    bool done = !act;
    uint32_t res = 0u;
    const int jhi = min(R + wd, w - 1);
    const int jlast = min(v + ks.halo, h - 1) - s.ra;
    for (int j = max(v - ks.halo, 0) - s.ra; j <= jlast; ++j) {
        if constexpr (!ZMAX) {
            for (int g0 = 0; g0 <= jhi - R; g0 += 32) {
                // lane 0 takes the group's first column in kernel order
                const int c = ks.nearest ? R + g0 + lane : jhi - g0 - lane;
                bool contrib = false;
                uint32_t col = 0u;
                if ((ks.nearest ? c <= jhi : c >= R) &&
                    YORO_BOUND(j >= 0 && j < s.slots && c >= 0 && c < s.wpad, kBadHoles)) {
                    const int i = j * s.wpad + c;
                    const bool reached = (s.bits[j * s.nwords + (c >> 5)] >> (c & 31)) & 1u;
                    contrib = reached && !(__uint_as_float(s.zt[i]) < d_occ);  // not foreground (O2)
                    if (contrib) col = s.rgba[i];
                }
                uint32_t cm = __ballot_sync(0xffffffffu, contrib);
                while (cm) {  // contributors in kernel order
                    const int k = __ffs(cm) - 1;
                    cm &= cm - 1u;
                    const uint32_t cc = __shfl_sync(0xffffffffu, col, k);
                    if (!done) {
                        if (!f.add(cc)) {  // weight reached exactly 0
                            res = f.result();
                            done = true;
                        } else {
                            uint32_t out;
                            if (f.wrem <= kSettleFrom && f.settled(out)) {
                                res = out;
                                done = true;
                            }
                        }
                    }
                    if (__all_sync(0xffffffffu, done)) return res;
                }
            }
        } else {
            const int wlo = R >> 5, whi = jhi >> 5;
            for (int g0 = 0; g0 <= whi - wlo; g0 += 32) {
                const int wi = ks.nearest ? wlo + g0 + lane : whi - g0 - lane;
                const bool some = wi >= wlo && wi <= whi && YORO_BOUND(j >= 0 && j < s.slots, kBadHoles) &&
                                  !(__uint_as_float(s.zmax[j * s.nwords + wi]) < d_occ);
                for (uint32_t wm = __ballot_sync(0xffffffffu, some); wm; wm &= wm - 1u) {
                    const int q = __ffs(wm) - 1, word = ks.nearest ? wlo + g0 + q : whi - g0 - q;
                    const int c = (word << 5) + (ks.nearest ? lane : 31 - lane);
                    bool contrib = false;
                    uint32_t col = 0u;
                    if (c >= R && c <= jhi && YORO_BOUND(j >= 0 && j < s.slots && c >= 0 && c < s.wpad, kBadHoles)) {
                        const int i = j * s.wpad + c;
                        const bool reached = (s.bits[j * s.nwords + word] >> (c & 31)) & 1u;
                        contrib = reached && !(__uint_as_float(s.zt[i]) < d_occ);
                        if (contrib) col = s.rgba[i];
                    }
                    uint32_t cm = __ballot_sync(0xffffffffu, contrib);
                    while (cm) {
                        const int k = __ffs(cm) - 1;
                        cm &= cm - 1u;
                        const uint32_t cc = __shfl_sync(0xffffffffu, col, k);
                        if (!done) {
                            if (!f.add(cc)) {
                                res = f.result();
                                done = true;
                            } else {
                                uint32_t out;
                                if (f.wrem <= kSettleFrom && f.settled(out)) {
                                    res = out;
                                    done = true;
                                }
                            }
                        }
                        if (__all_sync(0xffffffffu, done)) return res;
                    }
                }
            }
        }
    }
    if (!done) res = f.any() ? f.result() : (YORO_BOUND(R < s.wpad, kBadHoles) ? s.crow(v)[R] : 0u);
    return res;
}

// Hole fill of a one-pixel crack (v, x): reached pixels at x-1 and x+1, so L = x-1,
// R = x+1, w = 2 and t = 1/2.  The kernel is rows v-1, v, v+1 (v - halo .. v + halo)
// times columns min(x+3, W-1) .. x+1 (or x+1 .. x+3 nearest first); all slots are
// visited in the same order as fill_from_edges,
// without early exits.  A slot that does not contribute (outside the image, a hole, or
// nearer than the occluder) is given weight 0, which leaves acc and wrem unchanged
// exactly, so the result equals the general loop's.
template <bool VAR>
__device__ __forceinline__ uint32_t fill_crack(int x, int v, int h, int w, const Window& s,
                                               const KernelShape<VAR>& ks)
{
    const float d_occ = __uint_as_float(s.zrow(v)[x - 1]);
    FillAcc f;
    f.init(0.5f);
#pragma unroll
    for (int k = 0; k <= 2 * ks.halo; ++k) {
        const int vv = v - ks.halo + k;
        const bool row_in = vv >= 0 && vv < h;
        // a valid row to read when vv is outside
        const int vr = (row_in && YORO_BOUND(vv - s.ra >= 0 && vv - s.ra < s.slots, kBadHoles)) ? vv : v;
        const uint32_t* b = s.brow(vr);
        const uint32_t* zr = s.zrow(vr);
        const uint32_t* cr = s.crow(vr);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const int col = ks.nearest ? x + 1 + c : x + 3 - c;
            const bool col_in = col < w;
            const int cc = col_in ? col : x + 1;
            const bool reached = (b[cc >> 5] >> (cc & 31)) & 1u;
            const bool contributes = row_in && col_in && reached && !(__uint_as_float(zr[cc]) < d_occ);
            f.add_if(contributes, cr[cc]);
        }
    }
    return f.any() ? f.result() : s.crow(v)[x + 1];
}

// Interior holes of 32-pixel word g of a band row with reached bitmask bv and last
// reached column `last`: one-pixel cracks (both neighbours reached) in cm, wider holes
// in gm.  Holes right of `last` are border holes and in neither.
__device__ __forceinline__ void hole_masks(const uint32_t* bv, int g, int nwords, int last, uint32_t& cm,
                                           uint32_t& gm)
{
    const uint32_t reach = bv[g];
    const uint32_t prev = g > 0 ? bv[g - 1] : 0u;
    const uint32_t next = g + 1 < nwords ? bv[g + 1] : 0u;
    const int rem = last - (g << 5);
    const uint32_t inb = rem >= 31 ? ~0u : (rem >= 0 ? ((2u << rem) - 1u) : 0u);
    const uint32_t hw = ~reach & inb;
    const uint32_t left = (reach << 1) | (prev >> 31);   // bit i: column 32g + i - 1 reached
    const uint32_t right = (reach >> 1) | (next << 31);  // bit i: column 32g + i + 1 reached
    cm = hw & left & right;
    gm = hw & ~cm;
}

// Position of the k-th (0-based) set bit of m; m must have more than k set bits.
__device__ __forceinline__ int nth_set_bit(uint32_t m, int k)
{
    int pos = 0, c;
    c = __popc(m & 0xffffu);
    if (k >= c) { k -= c; pos += 16; m >>= 16; }
    c = __popc(m & 0xffu);
    if (k >= c) { k -= c; pos += 8; m >>= 8; }
    c = __popc(m & 0xfu);
    if (k >= c) { k -= c; pos += 4; m >>= 4; }
    c = __popc(m & 0x3u);
    if (k >= c) { k -= c; pos += 2; m >>= 2; }
    c = (int)(m & 1u);
    if (k >= c) pos += 1;
    return pos;
}

// P1 (Alg. 1 closed form, Alg. 2 nearest kept) over the window's nr rows.
//
// Alg. 2 keeps, per target, the nearest source, on equal depth the one met first.  In
// one row that is the source with the largest column: with k = fx * ipd >= 0,
// Q = RN(k / zc) does not grow with the clamped depth zc, and the target
// floor(RN(x + 0.5 - Q)) rises by at least one per column at fixed Q (for targets in
// [0, 2^22) the rounding unit is at most 1/2, and a round-half-even tie resolves the
// same way one column apart).  So if sources x1 < x2 reach
// one target, Q1 < Q2, i.e. zc1 > zc2: the right one is strictly nearer, and equal
// depths never meet.  Each source therefore takes an atomic maximum of its column into
// its target's word (one native 32-bit shared atomic), and the depth is fetched for
// the winner alone in P2.
//
// Two forms deal the window's pixels to the threads.  In the two-column form each
// thread takes the columns x = tid and x + NT of every window row: consecutive lanes take
// consecutive columns, so a warp's loads of one row are one 128-byte line; a column's
// centre x + 0.5 and its depth pointer are set once, so a pixel costs only its row step;
// and the thread issues the loads of U = 5 rows of both columns before it processes any
// (a 15-row window is three groups; the rows left over form one group of their own
// height).  At 1832 columns it executes 12 % fewer
// instructions than the flat form below and keeps more loads in flight (measured
// against one column at a time with 3 to 15 rows per group, two columns with 3, 4 or 7
// rows, and (row group, column) units dealt round-robin).  But a thread's share is whole
// columns, so where the columns do not split evenly over the threads the flat form,
// pixels dealt round-robin in memory order, balances better.
template <int NT, int U>
__device__ __forceinline__ void scatter_rows(const FrameArgs& f, const float* dcol, int j, int nr, int x, float xc,
                                             bool two, int* srow, int wpad, uint32_t near_m1, uint32_t far_m1)
{
    const int w = f.w;
    float z[2][U];
#pragma unroll
    for (int c = 0; c < 2; ++c)
#pragma unroll
        for (int u = 0; u < U; ++u)
            z[c][u] = ((c == 0 || two) && YORO_BOUND(j + u < nr, kBadScatter))
                          ? dcol[c * NT + (size_t)u * w]
                          : 0.0f;
#pragma unroll
    for (int c = 0; c < 2; ++c)
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (c == 0 || two) {
                uint32_t zb;
                const int xt = disparity_target(z[c][u], __fadd_rn(xc, (float)(c * NT)), f.k, near_m1, far_m1,
                                                f.half_m, zb);
                if ((unsigned)xt < (unsigned)w && YORO_BOUND(j + u < nr, kBadScatter))
                    atomicMax(srow + u * wpad + xt, x + c * NT);
            }
        }
}

// Next pixel of a flat (row, column) enumeration of a region `rw` columns wide dealt
// round-robin: advance by `dq` columns and `dr` rows (the stride split as rows and a
// remainder), carrying a row.
__device__ __forceinline__ void advance(int& r, int& q, int dr, int dq, int rw)
{
    q += dq;
    r += dr;
    if (q >= rw) {
        q -= rw;
        ++r;
    }
}

// The flat form over columns x0 .. w-1 of the window rows: pixel i = r * rw + q
// (rw = w - x0) goes to thread i mod NT, which issues the loads of U = 4 pixels before
// it processes any.
template <int NT, int U, bool FULL>
__device__ __forceinline__ void scatter_flat(const FrameArgs& f, const float* depth, int n, int i, int& r, int& q,
                                             int dr, int dq, int x0, int rw, int* src, int wpad, uint32_t near_m1,
                                             uint32_t far_m1)
{
    const int w = f.w;
    float z[U];
    int ru[U], xu[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
        ru[u] = r;
        xu[u] = x0 + q;
        z[u] = ((FULL || i + u * NT < n) && YORO_BOUND(i + u * NT < n, kBadScatter))
                   ? depth[(size_t)r * w + x0 + q]
                   : 0.0f;
        advance(r, q, dr, dq, rw);
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
        if (FULL || i + u * NT < n) {
            uint32_t zb;
            const int xt = disparity_target(z[u], __fadd_rn((float)xu[u], 0.5f), f.k, near_m1, far_m1, f.half_m, zb);
            if ((unsigned)xt < (unsigned)w) atomicMax(src + ru[u] * wpad + xt, xu[u]);
        }
    }
}

template <int NT>
__device__ __forceinline__ void scatter_window(const FrameArgs& f, const float* depth, int nr, int* src, int wpad)
{
    constexpr int U = 5;
    const int w = f.w;
    const uint32_t near_m1 = __float_as_uint(f.near_) - 1u, far_m1 = __float_as_uint(f.far_) - 1u;
    // Columns of the two-column form: the first 2 NT of a frame at least that wide, else
    // all of them if no thread's share exceeds the mean share by more than a quarter
    // (2 NT / w or NT / w <= 5/4; at 1440 columns, 2 NT / w = 1.42 and the flat form
    // measured 3 % faster), else none.
    const int pc = w >= 2 * NT ? 2 * NT : (w > NT ? (5 * w >= 8 * NT ? w : 0) : (5 * w >= 4 * NT ? w : 0));
    const int x = threadIdx.x;
    if (x < pc) {
        const bool two = x + NT < pc;
        const float xc = __fadd_rn((float)x, 0.5f);  // exact: x < 2^23
        const float* dcol = depth + x;
        int* srow = src;
        int j = 0;
        for (; j + U <= nr; j += U) {  // every row of the group in the window
            scatter_rows<NT, U>(f, dcol, j, nr, x, xc, two, srow, wpad, near_m1, far_m1);
            dcol += (size_t)U * w;
            srow += U * wpad;
        }
        switch (nr - j) {  // the last rows as one group of their own height
        case 1: scatter_rows<NT, 1>(f, dcol, j, nr, x, xc, two, srow, wpad, near_m1, far_m1); break;
        case 2: scatter_rows<NT, 2>(f, dcol, j, nr, x, xc, two, srow, wpad, near_m1, far_m1); break;
        case 3: scatter_rows<NT, 3>(f, dcol, j, nr, x, xc, two, srow, wpad, near_m1, far_m1); break;
        case 4: scatter_rows<NT, 4>(f, dcol, j, nr, x, xc, two, srow, wpad, near_m1, far_m1); break;
        default: break;
        }
    }
    // the other columns (none at 1832 columns; 16 at 2064) in the flat form
    const int rw = w - pc;
    if (rw > 0) {
        constexpr int UF = 4;
        const int n = nr * rw;
        const int dr = NT / rw, dq = NT - dr * rw;
        int r = (int)threadIdx.x / rw, q = (int)threadIdx.x - r * rw;
        int i = threadIdx.x;
        for (; i + (UF - 1) * NT < n; i += UF * NT)  // every load of the group in range
            scatter_flat<NT, UF, true>(f, depth, n, i, r, q, dr, dq, pc, rw, src, wpad, near_m1, far_m1);
        if (i < n) scatter_flat<NT, UF, false>(f, depth, n, i, r, q, dr, dq, pc, rw, src, wpad, near_m1, far_m1);
    }
}

// P2 (resolve + gather) over the window: warp `warp` owns the 32-pixel words
// g = warp, warp + NW, ... of every row and takes RB rows per batch.  A reached target
// loads its source's depth (clamped as in P1) and color; ballots give the reached
// bitmasks.  Band rows send their reached pixels and hole mask to global memory right
// here; their holes are written in P3.  The loads of a batch are unconditional (a hole
// or a lane past the row end reads column 0, a batch row past the window reads the
// last window row), so the batch has no branches around its loads.
template <int RB, bool FULL, int NWI, int DX, bool ZT>
__device__ __forceinline__ void resolve_batch(const FrameArgs& f, const float* depth, const uint32_t* color,
                                              const Window& s, int g, int j0, int nb, int nr, int jb0, int jb1,
                                              uint32_t near_m1, uint32_t far_m1)
{
    // NWI words of the row batch at once: word g and, if NWI == 2, word g + DX / 32
    // (the next word the same warp owns), DX columns to the right.
    const int lane = threadIdx.x & 31;
    const int w = f.w, wpad = s.wpad;
    const int x = (g << 5) + lane;
    bool xin[NWI];
#pragma unroll
    for (int q = 0; q < NWI; ++q) xin[q] = x + q * DX < w;
    int sc[NWI][RB];
    float zs[NWI][RB];
    uint32_t cs[NWI][RB];
    // offsets advance by one row stride per row: no multiplies in the batch
    int so = j0 * wpad + x;  // shared-memory word of (row, x)
    int go = j0 * w;         // global pixel offset of the row in the window
#pragma unroll
    for (int u = 0; u < RB; ++u) {
#pragma unroll
        for (int q = 0; q < NWI; ++q)
            sc[q][u] = ((FULL || u < nb) && xin[q] && YORO_BOUND(so + q * DX < nr * wpad, kBadResolve))
                           ? (int)s.zt[so + q * DX]
                           : -1;
        so += wpad;
    }
#pragma unroll
    for (int u = 0; u < RB; ++u) {
#pragma unroll
        for (int q = 0; q < NWI; ++q) {
            const int o = go + max(sc[q][u], 0);
            zs[q][u] = 0.0f;
            cs[q][u] = 0u;
            if ((FULL || u < nb) && YORO_BOUND(o < nr * w, kBadResolve)) {
                zs[q][u] = depth[o];
                cs[q][u] = color[o];
            }
        }
        go += w;
    }
    so = j0 * wpad + x;
    int vo = (s.ra + j0) * w + x;  // frame pixel offset of (row, x)
#pragma unroll
    for (int u = 0; u < RB; ++u) {
        if (FULL || u < nb) {
            const int j = j0 + u;
            const bool band = j >= jb0 && j < jb1;
#pragma unroll
            for (int q = 0; q < NWI; ++q) {
                const bool reached = sc[q][u] >= 0;
                const uint32_t m = __ballot_sync(0xffffffffu, reached);
                const uint32_t zbits = clamped_depth_bits(zs[q][u], near_m1, far_m1);
                if (reached && YORO_BOUND(so + q * DX < nr * wpad, kBadResolve)) {
                    s.zt[so + q * DX] = zbits;
                    s.rgba[so + q * DX] = cs[q][u];
                }
                if (lane == 0 && YORO_BOUND(g + q * (DX >> 5) < s.nwords && j < nr, kBadResolve))
                    s.bits[j * s.nwords + g + q * (DX >> 5)] = m;
                // a band row: the pixel and its mask byte leave
                if (band && xin[q] && YORO_BOUND(vo + q * DX < f.h * w, kBadResolve)) {
                    if (reached) f.out[vo + q * DX] = cs[q][u];
                    f.mask[vo + q * DX] = reached ? 0 : 1;
                    if (ZT && f.zt_out) f.zt_out[vo + q * DX] = reached ? __uint_as_float(zbits) : 0.0f;
                }
            }
        }
        so += wpad;
        vo += w;
    }
}

// WIDE (windows wider than 2 NT words): the words from 2 NT on are dealt as (word, row
// batch) items over all warps instead of as a third word of the first warps (2064-wide
// frames: 29.0 -> 27.5 us per frame).  A separate instantiation, so that the code of the
// common width is untouched (compiled into one kernel the extra loop cost 1832-wide
// frames 2.5 %).
template <int NT, bool ZT, bool WIDE = false>
__device__ __forceinline__ void resolve_window(const FrameArgs& f, const float* depth, const uint32_t* color,
                                               int nr, int y0, int y1, const Window& s)
{
    constexpr int NW = NT / 32, RB = 3;  // 15-row windows: five full batches (2..8 measured)
    constexpr int DX = 32 * NW;          // columns between the two words a warp takes at once
    const int warp = threadIdx.x >> 5;
    const uint32_t near_m1 = __float_as_uint(f.near_) - 1u, far_m1 = __float_as_uint(f.far_) - 1u;
    const int jb0 = y0 - s.ra, jb1 = y1 - s.ra;  // band rows of the window: [jb0, jb1)
    for (int g = warp; g < (WIDE ? min(s.nwords, 2 * NW) : s.nwords); g += 2 * NW) {
        const bool two = g + NW < s.nwords;  // warp-uniform
        int j0 = 0;
        for (; j0 + RB <= nr; j0 += RB) {
            if (two) resolve_batch<RB, true, 2, DX, ZT>(f, depth, color, s, g, j0, RB, nr, jb0, jb1, near_m1, far_m1);
            else resolve_batch<RB, true, 1, DX, ZT>(f, depth, color, s, g, j0, RB, nr, jb0, jb1, near_m1, far_m1);
        }
        if (j0 < nr) {
            if (two) resolve_batch<RB, false, 2, DX, ZT>(f, depth, color, s, g, j0, nr - j0, nr, jb0, jb1, near_m1,
                                                     far_m1);
            else resolve_batch<RB, false, 1, DX, ZT>(f, depth, color, s, g, j0, nr - j0, nr, jb0, jb1, near_m1,
                                                     far_m1);
        }
    }
    if (WIDE) {
        const int nbat = (nr + RB - 1) / RB;
        for (int it = warp; it < (s.nwords - 2 * NW) * nbat; it += NW) {
            const int gw = 2 * NW + it / nbat, j0 = (it - (it / nbat) * nbat) * RB;
            if (j0 + RB <= nr)
                resolve_batch<RB, true, 1, DX, ZT>(f, depth, color, s, gw, j0, RB, nr, jb0, jb1, near_m1, far_m1);
            else
                resolve_batch<RB, false, 1, DX, ZT>(f, depth, color, s, gw, j0, nr - j0, nr, jb0, jb1, near_m1,
                                                    far_m1);
        }
    }
}

// One band [y0, y1) of one frame; shared memory holds the window rows ra..rb
// (ra = y0-1 or 0, rb = y1 or h-1).  Ends with a barrier, so the next band may reuse
// shared memory.
template <int NT, bool VAR, bool ZMAX = false>
__device__ __forceinline__ void fill_band(const FrameArgs& f, int y0, int y1, const Window& s, int* ctr,
                                          int* rowinfo);

template <int NT, bool VAR, bool ZT, bool WIDE = false>
__device__ __forceinline__ void run_band(const FrameArgs& f, int y0, int y1, Window s, int* ctr, int* rowinfo)
{
    constexpr int NW = NT / 32;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int w = f.w, h = f.h;
    const KernelShape<VAR> ks(f);
    const int ra = max(y0 - ks.halo, 0), rb = min(y1 - 1 + ks.halo, h - 1);
    const int nr = rb - ra + 1;
    s.ra = ra;
    const float* depth = f.depth + (size_t)ra * w;
    const uint32_t* color = f.color + (size_t)ra * w;

    if (f.bulk && lane == 0) {  // one depth row, then its color row, per warp
        for (int j = warp; j < nr; j += NW) {
            prefetch_l2(depth + (size_t)j * w, (uint32_t)w * 4u);
            prefetch_l2(color + (size_t)j * w, (uint32_t)w * 4u);
        }
    }
    {
        uint4* z4 = reinterpret_cast<uint4*>(s.zt);  // four words per 16 bytes; wpad % 8 == 0
        const int n4 = nr * (s.wpad >> 2);
        const uint4 e = make_uint4(~0u, ~0u, ~0u, ~0u);
        for (int i = tid; i < n4; i += NT) z4[i] = e;
        if (tid == 0) *ctr = 0;
    }
    __syncthreads();

    // ---- P1: disparity and nearest-wins scatter of rows ra..rb
    scatter_window<NT>(f, depth, nr, reinterpret_cast<int*>(s.zt), s.wpad);
    __syncthreads();

    // ---- P2: resolve, gather depths and colors, reached bitmasks; band rows' reached
    // pixels and hole mask leave
    resolve_window<NT, ZT, WIDE>(f, depth, color, nr, y0, y1, s);
    __syncthreads();

    fill_band<NT, VAR>(f, y0, y1, s, ctr, rowinfo);
}

// P3 of one band [y0, y1) whose window (s.ra set) holds the reached pixels' depths and
// colors and every window row's reached bitmask.  Writes the band rows' holes to
// f.out (reached pixels and masks are not touched).  Ends with a barrier.
template <int NT, bool VAR, bool ZMAX>
__device__ __forceinline__ void fill_band(const FrameArgs& f, int y0, int y1, const Window& s, int* ctr,
                                          int* rowinfo)
{
    constexpr int NW = NT / 32;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int w = f.w, h = f.h;
    const int nwords = s.nwords;
    const KernelShape<VAR> ks(f);

    // ---- P3a: per band row (one warp per row; rows with every pixel reached are done):
    // its last reached column, the border holes right of it, and per 32-pixel word the
    // number of interior cracks and wider holes with their prefix sums within the row.  Border holes have no
    // background edge (R = W) and take the fallback, the color of the last reached pixel
    // (zero if the row has none).  Counts are packed as cracks | wider << 16: a band
    // holds fewer than 2^16 pixels.
    const int nb = y1 - y0;
    int* lastr = rowinfo;           // last reached column of band row vj
    int* rowoff = lastr + s.slots;  // holes of the band rows before row vj
    for (int vj = warp; vj < nb; vj += NW) {
        uint32_t tot = 0u;
        const int v = y0 + vj;
        const uint32_t* bv = s.brow(v);
        int last = -1;
        bool full = true;  // every pixel of the row reached
        for (int gg = lane; gg < nwords; gg += 32) {
            const uint32_t b = bv[gg];
            if (b) last = (gg << 5) + 31 - __clz(b);
            const uint32_t inrow = (gg == nwords - 1 && (w & 31)) ? (1u << (w & 31)) - 1u : ~0u;
            full = full && b == inrow;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) last = max(last, __shfl_xor_sync(0xffffffffu, last, o));
        if (!__all_sync(0xffffffffu, full)) {  // warp-uniform
            const uint32_t border = last >= 0 ? s.crow(v)[last] : 0u;
            uint32_t* orow = f.out + (size_t)v * w;
            for (int x = last + 1 + lane; x < w; x += 32) orow[x] = border;
            if (lane == 0) lastr[vj] = last;
            uint32_t* pre = s.pre + vj * nwords;
            for (int g0 = 0; g0 < nwords; g0 += 32) {
                const int g = g0 + lane;
                uint32_t c = 0u;
                if (g < nwords) {
                    uint32_t cm, gm;
                    hole_masks(bv, g, nwords, last, cm, gm);
                    c = (uint32_t)__popc(cm) | ((uint32_t)__popc(gm) << 16);
                }
                uint32_t sc = c;  // inclusive scan over the lanes
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const uint32_t y = __shfl_up_sync(0xffffffffu, sc, o);
                    if (lane >= o) sc += y;
                }
                if (g < nwords) pre[g] = tot + sc - c;
                tot += __shfl_sync(0xffffffffu, sc, 31);
            }
        }
        if (lane == 0) rowoff[vj] = (int)tot;
    }
    __syncthreads();
    if (warp == 0) {  // exclusive scan of the row totals; the band total goes to ctr[1]
        uint32_t run = 0u;
        for (int c0 = 0; c0 < nb; c0 += 32) {
            const uint32_t c = c0 + lane < nb ? (uint32_t)rowoff[c0 + lane] : 0u;
            uint32_t sc = c;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t y = __shfl_up_sync(0xffffffffu, sc, o);
                if (lane >= o) sc += y;
            }
            if (c0 + lane < nb) rowoff[c0 + lane] = (int)(run + sc - c);
            run += __shfl_sync(0xffffffffu, sc, 31);
        }
        if (lane == 0) ctr[1] = (int)run;
    }
    __syncthreads();

    // ---- P3b: fill of the interior holes (Alg. 3, Eq. 6).  The band's wider holes, then
    // its cracks, in row-major order, are dealt in chunks to whichever warp takes the next
    // chunk from a shared counter, so a wide disocclusion is spread over many warps and
    // every chunk but the last of each kind is full: 32 wider-hole pixels (one per lane),
    // or 64 cracks (two consecutive ones per lane: a crack's nine-slot fill is short, so
    // the search that locates it is a large part of its cost, and the second crack is
    // found from the first by the next crack bit of its row; 1832x1920, four streams:
    // 19.67 -> 19.52 us per frame, four per lane 20.52).  A lane finds its first hole by
    // binary search over the row and word prefix sums.
    {
        const uint32_t tot = (uint32_t)ctr[1];
        const int tc = (int)(tot & 0xffffu), tg = (int)(tot >> 16);
        const int ng = (tg + 31) >> 5, nchunks = ng + ((tc + 63) >> 6);
        // hole idx of the kind selected by sh (16: wider holes, 0: cracks) -> band row vj,
        // its rank r in the row, word g, rank k in the word, the word's hole masks
        auto locate = [&](int idx, int sh, int& vj, int& r, int& g, int& k, uint32_t& cm, uint32_t& gm) {
            // band row: the last row whose offset is <= idx
            int lo = 0, hi = nb - 1;
            while (lo < hi) {
                const int mid = (lo + hi + 1) >> 1;
                if ((int)(((uint32_t)rowoff[mid] >> sh) & 0xffffu) <= idx) lo = mid;
                else hi = mid - 1;
            }
            vj = lo;
            r = idx - (int)(((uint32_t)rowoff[vj] >> sh) & 0xffffu);
            // word of the row: the last word whose prefix is <= r
            const uint32_t* pre = s.pre + vj * nwords;
            lo = 0;
            hi = nwords - 1;
            while (lo < hi) {
                const int mid = (lo + hi + 1) >> 1;
                if ((int)((pre[mid] >> sh) & 0xffffu) <= r) lo = mid;
                else hi = mid - 1;
            }
            g = lo;
            k = r - (int)((pre[g] >> sh) & 0xffffu);
            hole_masks(s.brow(y0 + vj), g, nwords, lastr[vj], cm, gm);
        };
        for (;;) {
            int chunk = 0;
            if (lane == 0) chunk = atomicAdd(ctr, 1);
            chunk = __shfl_sync(0xffffffffu, chunk, 0);
            if (chunk >= nchunks) break;
            if (chunk < ng) {  // 32 pixels of wider holes, one per lane (warp-uniform branch)
                const int idx = (chunk << 5) + lane;
                bool act = idx < tg;  // lane 0 is always active
                int v = 0, x = 0;
                if (act) {
                    int vj, r, g, k;
                    uint32_t cm, gm;
                    locate(idx, 16, vj, r, g, k, cm, gm);
                    v = y0 + vj;
                    x = (g << 5) + nth_set_bit(gm, k);
                    // the located pixel is a hole of the band row (checked in the debug-bounds build)
                    act = YORO_BOUND((unsigned)x < (unsigned)w && !((s.brow(v)[x >> 5] >> (x & 31)) & 1u),
                                     kBadHoles);
                }
                uint32_t o = 0u;
                int L = -1, R = 0;
                if (act) find_edges(x, v, s, w, L, R);
                // one hole for the whole chunk: its kernel is scanned once by the warp
                const int v0 = __shfl_sync(0xffffffffu, v, 0), L0 = __shfl_sync(0xffffffffu, L, 0),
                          R0 = __shfl_sync(0xffffffffu, R, 0);
                if (__all_sync(0xffffffffu, !act || (v == v0 && L == L0 && R == R0)))
                    o = fill_hole_warp<VAR, ZMAX>(x, act, v0, L0, R0, h, w, s, ks);
                else if (act)
                    o = fill_from_edges<VAR, ZMAX>(x, v, L, R, h, w, s, ks);
                if (act && YORO_BOUND(v >= y0 && v < y1, kBadHoles)) f.out[(size_t)v * w + x] = o;
            } else {  // 64 cracks, two consecutive ones per lane
                const int idx = ((chunk - ng) << 6) + 2 * lane;
                bool act0 = idx < tc, act1 = idx + 1 < tc;
                int v0 = 0, x0 = 0, v1 = 0, x1 = 0;
                if (act0) {
                    int vj, r, g, k;
                    uint32_t cm, gm;
                    locate(idx, 0, vj, r, g, k, cm, gm);
                    const int b0 = nth_set_bit(cm, k);
                    v0 = y0 + vj;
                    x0 = (g << 5) + b0;
                    act0 = YORO_BOUND((unsigned)x0 < (unsigned)w && !((s.brow(v0)[x0 >> 5] >> (x0 & 31)) & 1u),
                                      kBadHoles);
                    if (act1) {
                        const int rowc = (vj + 1 < nb ? (int)((uint32_t)rowoff[vj + 1] & 0xffffu) : tc) -
                                         (int)((uint32_t)rowoff[vj] & 0xffffu);  // cracks of row vj
                        if (r + 1 < rowc) {  // the next crack of the same row: the next crack bit
                            const uint32_t* bv = s.brow(v0);
                            uint32_t rest = b0 == 31 ? 0u : (cm & (~0u << (b0 + 1)));
                            int g1 = g;
                            while (!rest && YORO_BOUND(g1 + 1 < nwords, kBadHoles)) {
                                ++g1;
                                hole_masks(bv, g1, nwords, lastr[vj], rest, gm);
                            }
                            v1 = v0;
                            x1 = (g1 << 5) + __ffs(rest) - 1;
                        } else {  // the first crack of a later row
                            locate(idx + 1, 0, vj, r, g, k, cm, gm);
                            v1 = y0 + vj;
                            x1 = (g << 5) + nth_set_bit(cm, k);
                        }
                        act1 = YORO_BOUND(
                            (unsigned)x1 < (unsigned)w && !((s.brow(v1)[x1 >> 5] >> (x1 & 31)) & 1u), kBadHoles);
                    }
                }
                if (act0 && YORO_BOUND(v0 >= y0 && v0 < y1, kBadHoles))
                    f.out[(size_t)v0 * w + x0] = fill_crack<VAR>(x0, v0, h, w, s, ks);
                if (act1 && YORO_BOUND(v1 >= y0 && v1 < y1, kBadHoles))
                    f.out[(size_t)v1 * w + x1] = fill_crack<VAR>(x1, v1, h, w, s, ks);
            }
        }
    }
    __syncthreads();
}

// Shared-memory layout of a window of `slots` rows (see fused_smem_bytes).
__device__ __forceinline__ Window window_layout(unsigned char* smem, int slots, int wpad, int w, int*& ctr,
                                                int*& rowinfo)
{
    Window s;
    s.zt = reinterpret_cast<uint32_t*>(smem);
    s.rgba = s.zt + slots * wpad;
    s.bits = s.rgba + slots * wpad;
    s.wpad = wpad;
    s.nwords = (w + 31) >> 5;
    s.ra = 0;
    s.slots = slots;
    s.pre = s.bits + slots * ((wpad + 31) / 32);
    s.zmax = nullptr;
    ctr = reinterpret_cast<int*>(s.pre + slots * ((wpad + 31) / 32));
    rowinfo = ctr + 4;
    return s;
}

template <int NT, int MINB, bool VAR, bool ZT = false, bool WIDE = false>
__global__ void __launch_bounds__(NT, MINB) fused_single(FrameArgs f, int wpad)
{
    after_wait();
    extern __shared__ __align__(128) unsigned char smem_raw[];
    int *ctr, *rowinfo;
    const Window s = window_layout(smem_raw, f.band + 2 * KernelShape<VAR>(f).halo, wpad, f.w, ctr, rowinfo);
    const int nbands = (f.h + f.band - 1) / f.band;
    for (int b = blockIdx.x; b < nbands; b += gridDim.x) {
        const int y0 = b * f.band;
        run_band<NT, VAR, ZT, WIDE>(f, y0, min(y0 + f.band, f.h), s, ctr, rowinfo);
    }
}

template <int NT, int MINB, bool ZT = false, bool WIDE = false>
__global__ void __launch_bounds__(NT, MINB) fused_batch(const __grid_constant__ BatchArgs a, int wpad)
{
    after_wait();
    extern __shared__ __align__(128) unsigned char smem_raw[];
    for (int item = blockIdx.x; item < a.total_items; item += gridDim.x) {
        int lo = 0, hi = a.n - 1;  // frame whose item range holds `item`
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (a.item_start[mid] <= item) lo = mid;
            else hi = mid - 1;
        }
        const FrameArgs& f = a.f[lo];
        int *ctr, *rowinfo;
        // the frame's own row stride: a narrower frame fits more rows (f.band) in the
        // shared memory sized for max_band rows of the widest
        const Window s = window_layout(smem_raw, f.band + 2, (f.w + 7) / 8 * 8, f.w, ctr, rowinfo);
        const int y0 = (item - a.item_start[lo]) * f.band;
        run_band<NT, false, ZT, WIDE>(f, y0, min(y0 + f.band, f.h), s, ctr, rowinfo);
    }
}

// P3 alone over an image that is already resolved in global memory: the reached pixels'
// colors in f.out, their depths in zt, the hole mask in f.mask (the row-downsampled
// intermediate buffer's and the general pose's full-resolution image).  Each band's window
// is loaded (the reached bitmasks by ballot over the mask bytes, depths and colors of the
// reached pixels; each warp takes four 32-pixel words at a time, their loads issued
// before any is used), then filled exactly as the fused kernel fills its bands.  VAR as
// in the fused kernel: false compiles the paper's kernel shape as constants.
template <int NT, bool VAR>
__global__ void __launch_bounds__(NT, 1) fill_only(FrameArgs f, const float* zt, int wpad)
{
    after_wait();
    extern __shared__ __align__(128) unsigned char smem_raw[];
    constexpr int NW = NT / 32;
    int *ctr, *rowinfo;
    const KernelShape<VAR> ks(f);
    Window s = window_layout(smem_raw, f.band + 2 * ks.halo, wpad, f.w, ctr, rowinfo);
    const int w = f.w, h = f.h, nwords = s.nwords;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int nbands = (h + f.band - 1) / f.band;
    for (int b = blockIdx.x; b < nbands; b += gridDim.x) {
        const int y0 = b * f.band, y1 = min(y0 + f.band, h);
        const int ra = max(y0 - ks.halo, 0), rb = min(y1 - 1 + ks.halo, h - 1);
        const int nr = rb - ra + 1;
        s.ra = ra;
        const int items = nr * nwords;
        for (int it0 = warp; it0 < items; it0 += 4 * NW) {
            uint32_t mk[4], zv[4], cv[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int it = it0 + q * NW;
                const int j = it / nwords, g = it - j * nwords;
                const int x = (g << 5) + lane;
                const size_t o = (size_t)(ra + j) * w + x;
                const bool ld = it < items && x < w;
                mk[q] = ld ? f.mask[o] : 1u;
                zv[q] = ld ? __float_as_uint(zt[o]) : 0u;
                cv[q] = ld ? f.out[o] : 0u;
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int it = it0 + q * NW;
                if (it >= items) break;  // warp-uniform
                const int j = it / nwords, g = it - j * nwords;
                const int x = (g << 5) + lane;
                const bool reached = mk[q] == 0u;
                const uint32_t m = __ballot_sync(0xffffffffu, reached);
                if (lane == 0 && YORO_BOUND(j < s.slots, kBadHoles)) s.bits[j * nwords + g] = m;
                if (reached && YORO_BOUND(j * wpad + x < s.slots * wpad, kBadHoles)) {
                    s.zt[j * wpad + x] = zv[q];
                    s.rgba[j * wpad + x] = cv[q];
                }
            }
        }
        if (threadIdx.x == 0) *ctr = 0;
        __syncthreads();
        fill_band<NT, VAR>(f, y0, y1, s, ctr, rowinfo);
    }
}

// The band fill straight from a frame-wide z-buffer of 64-bit keys (clamped depth bits
// above the source pixel's index, the empty key at holes: the general pose's Alg. 2 over
// the frame): each band's window is loaded from the keys (reached bitmask, the depth from
// the key, the winner's color gathered from f.color), the band rows' colors of reached
// pixels and their hole mask leave for global memory, and the holes are filled as in
// fill_only.  It stands in for a gather pass that writes the image out and fill_only's
// reading it back.  The loading takes about 19 us of the pass at 1832x1920; the rest is the
// holes' fill, bound by the bands that hold the most of it.  With each word's largest reached
// depth at hand (one warp reduction and 4 bytes per word) the fill passes over words that
// are all foreground: eight seeds of 1832x1920 took 103, 52, 66, 56, 72, 95, 52 and 60 us with
// one lane or one warp crossing them column by column, 64, 53, 61, 54, 68, 61, 50 and 48 so.
// ZMAX = false, without them, is for the widths whose window just fits shared memory.
template <int NT, bool VAR, bool ZMAX>
__global__ void __launch_bounds__(NT, 1) fill_keys(FrameArgs f, const unsigned long long* keys, int wpad)
{
    after_wait();
    extern __shared__ __align__(128) unsigned char smem_raw[];
    constexpr int NW = NT / 32, RB = 5;  // bands of 13 rows: windows of three full batches
    int *ctr, *rowinfo;
    const KernelShape<VAR> ks(f);
    Window s = window_layout(smem_raw, f.band + 2 * ks.halo, wpad, f.w, ctr, rowinfo);
    if (ZMAX) s.zmax = reinterpret_cast<uint32_t*>(rowinfo + 2 * s.slots);  // after the window (keys_smem_bytes)
    const int w = f.w, h = f.h, nwords = s.nwords;
    const size_t n = (size_t)w * (size_t)h;  // source indices are below n (checked in the debug-bounds build)
    (void)n;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int nbands = (h + f.band - 1) / f.band;
    for (int b = blockIdx.x; b < nbands; b += gridDim.x) {
        const int y0 = b * f.band, y1 = min(y0 + f.band, h);
        const int ra = max(y0 - ks.halo, 0), rb = min(y1 - 1 + ks.halo, h - 1);
        const int nr = rb - ra + 1;
        s.ra = ra;
        if (f.bulk && lane == 0)  // most winners come from rows near their target's
            for (int j = warp; j < nr; j += NW) prefetch_l2(f.color + (size_t)(ra + j) * w, (uint32_t)w * 4u);
        // as in the resolve, a warp owns the words g = warp, warp + NW, ... of every row and takes
        // RB rows at a time, with offsets that advance by a row
        for (int g = warp; g < nwords; g += NW) {
            const int x = (g << 5) + lane;
            const bool xin = x < w;
            auto batch = [&](auto full, int j0, int nb) {
                constexpr bool FULL = decltype(full)::value;
                unsigned long long kv[RB];
                uint32_t cv[RB];
                const unsigned long long* kp = keys + ((ra + j0) * w + x);
#pragma unroll
                for (int u = 0; u < RB; ++u) {
                    kv[u] = ((FULL || u < nb) && xin) ? *kp : kEmptyKey;
                    kp += w;
                }
#pragma unroll
                for (int u = 0; u < RB; ++u) {
                    const uint32_t src = (uint32_t)kv[u];
                    cv[u] = (kv[u] != kEmptyKey && YORO_BOUND(src < n, kBadPose)) ? f.color[src] : 0u;
                }
                int so = j0 * wpad + x, vo = (ra + j0) * w + x;
#pragma unroll
                for (int u = 0; u < RB; ++u) {
                    if (FULL || u < nb) {  // uniform
                        const bool reached = kv[u] != kEmptyKey;
                        const uint32_t m = __ballot_sync(0xffffffffu, reached);
                        uint32_t zm = 0u;
                        if (ZMAX) zm = __reduce_max_sync(0xffffffffu, reached ? (uint32_t)(kv[u] >> 32) : 0u);
                        if (lane == 0 && YORO_BOUND(j0 + u < s.slots, kBadHoles)) {
                            s.bits[(j0 + u) * nwords + g] = m;
                            if (ZMAX) s.zmax[(j0 + u) * nwords + g] = zm;
                        }
                        if (reached && YORO_BOUND(so < s.slots * wpad, kBadHoles)) {
                            s.zt[so] = (uint32_t)(kv[u] >> 32);
                            s.rgba[so] = cv[u];
                        }
                        // a band row: the pixel and its mask byte leave
                        if (ra + j0 + u >= y0 && ra + j0 + u < y1 && xin) {
                            if (reached) f.out[vo] = cv[u];
                            f.mask[vo] = reached ? 0 : 1;
                        }
                    }
                    so += wpad;
                    vo += w;
                }
            };
            int j0 = 0;
            for (; j0 + RB <= nr; j0 += RB) batch(std::true_type{}, j0, RB);
            if (j0 < nr) batch(std::false_type{}, j0, nr - j0);
        }
        if (threadIdx.x == 0) *ctr = 0;
        __syncthreads();
        fill_band<NT, VAR, ZMAX>(f, y0, y1, s, ctr, rowinfo);
    }
}

// The row-downsampled intermediate buffer in one kernel: per band, the window rows'
// cells are reprojected into 64-bit cell keys in shared memory (after the window),
// every window pixel is sampled from its cell's winner into the window (depth, color,
// reached bitmask; the band rows' reached pixels and masks leave for global memory),
// and the band's holes are filled as the fused kernel fills them.  The steps and their
// rounding are those of imbuffer.cu's separate kernels (the reading is stated there).  Bound
// by its instructions: per 32-pixel word the sampling takes 105 and the cells 35 (four seeds
// of 1832x1920, 4 px per cell: 70, 69, 71, 81 us before the balanced bands and the row
// batches, 51, 48, 54, 59 us with them; without holes about 30).
template <int NT, bool VAR>
__global__ void __launch_bounds__(NT, 1) imb_band(FrameArgs f, int div, int interp, int wpad, int cells_off)
{
    after_wait();
    extern __shared__ __align__(128) unsigned char smem_raw[];
    constexpr int NW = NT / 32, RB = 3;  // bands of 7 rows: windows of three full batches
    int *ctr, *rowinfo;
    const KernelShape<VAR> ks(f);
    const int slots = f.band + 2 * ks.halo;
    Window s = window_layout(smem_raw, slots, wpad, f.w, ctr, rowinfo);
    const int w = f.w, h = f.h, nwords = s.nwords, ws = (w + div - 1) / div;
    unsigned long long* cells = reinterpret_cast<unsigned long long*>(smem_raw + cells_off);  // after the window
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t near_m1 = __float_as_uint(f.near_) - 1u, far_m1 = __float_as_uint(f.far_) - 1u;
    const float inv_s = 1.0f / (float)div;
    const int lg = __ffs(div) - 1;  // div is a power of two
    const int nbands = (h + f.band - 1) / f.band;
    for (int b = blockIdx.x; b < nbands; b += gridDim.x) {
        const int y0 = b * f.band, y1 = min(y0 + f.band, h);
        const int ra = max(y0 - ks.halo, 0), rb = min(y1 - 1 + ks.halo, h - 1);
        const int nr = rb - ra + 1;
        s.ra = ra;
        if (f.bulk && lane == 0) {  // one depth row, then its color row, per warp
            for (int j = warp; j < nr; j += NW) {
                prefetch_l2(f.depth + (size_t)(ra + j) * w, (uint32_t)w * 4u);
                prefetch_l2(f.color + (size_t)(ra + j) * w, (uint32_t)w * 4u);
            }
        }
        for (int i = threadIdx.x; i < nr * ws; i += NT) cells[i] = kEmptyKey;
        if (threadIdx.x == 0) *ctr = 0;
        __syncthreads();
        // cells: Alg. 1 on each cell's pixel, Alg. 2 by a 64-bit minimum of the key.  Only the
        // target cell floor(t / s) is needed, so the exact t = (p + 0.5) - RN(k / zc) is
        // computed only when the estimate cannot decide it (disparity_target's margin, which
        // holds for t and so for t / s, s >= 1).  Four cells' loads are in flight at a time;
        // (row j, cell i) of flat index c advance without a division per cell.
        const int dj = NT / ws, di = NT - dj * ws;
        int cj = (int)threadIdx.x / ws, ci = (int)threadIdx.x - cj * ws;
        for (int c = threadIdx.x; c < nr * ws; c += 4 * NT) {
            float z[4];
            int jq = cj, iq = ci;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                z[q] = c + q * NT < nr * ws
                           ? f.depth[(size_t)(ra + jq) * w + min((iq << lg) + (div >> 1), w - 1)]
                           : 0.0f;
                advance(jq, iq, dj, di, ws);
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                if (c + q * NT < nr * ws) {
                    const float pc = __fadd_rn((float)min((ci << lg) + (div >> 1), w - 1), 0.5f);
                    const uint32_t zb = clamped_depth_bits(z[q], near_m1, far_m1);
                    const float zc = __uint_as_float(zb);
                    const float te = __fmul_rn(__fmaf_rn(-f.k, rcp_approx(zc), pc), inv_s);
                    float tc = floorf(te);
                    if (!(fabsf(__fsub_rn(__fsub_rn(te, tc), 0.5f)) < f.half_m))
                        tc = floorf(__fmul_rn(__fsub_rn(pc, __fdiv_rn(f.k, zc)), inv_s));
                    if (tc >= 0.0f && tc < (float)ws && YORO_BOUND(cj < slots && ci < ws, kBadScatter))
                        atomicMin(&cells[cj * ws + (int)tc], zkey(zb, ci));
                }
                advance(cj, ci, dj, di, ws);
            }
        }
        __syncthreads();
        if (interp) {  // the winner's shift once per cell: its key's low word becomes disp
            for (int c = threadIdx.x; c < nr * ws; c += NT) {
                const unsigned long long key = cells[c];
                if (key != kEmptyKey) {
                    const uint32_t zb = (uint32_t)(key >> 32);
                    cells[c] = ((unsigned long long)zb << 32) | __float_as_uint(__fdiv_rn(f.k, __uint_as_float(zb)));
                }
            }
            __syncthreads();
        }
        // sampling: each window pixel from its cell's winner.  As in the resolve, a warp owns the
        // words g = warp, warp + NW, ... of every row and takes RB rows at a time, their color
        // loads issued before any is used, with offsets that advance by a row (an enumeration of
        // (row, word) items took 153 instructions per word, this one 105).  div divides 32, so
        // a lane's place in its cell is the same in every word: the neighbour's side and its
        // weight |x + 0.5 - (div cj + div / 2)| / div are constants of the lane (all exact).
        const float off = __fsub_rn(__fadd_rn((float)(lane & (div - 1)), 0.5f), 0.5f * (float)div);
        const int nside = off == 0.0f ? 0 : off < 0.0f ? -1 : 1;
        const float nwt = __fmul_rn(fabsf(off), inv_s);
        const float wlast = (float)(w - 1);
        for (int g = warp; g < nwords; g += NW) {
            const int x = (g << 5) + lane;
            const bool xin = x < w;
            const int cj = xin ? x >> lg : 0;
            const bool side = nside != 0 && (unsigned)(cj + nside) < (unsigned)ws;
            const float xf = (float)x;
            auto batch = [&](auto full, int j0, int nb) {
                constexpr bool FULL = decltype(full)::value;
                uint32_t zb[RB], c0[RB], c1[RB];
                float fr[RB];
                uint32_t reach = 0u;  // bit u: this lane's pixel of row j0 + u is reached
                const unsigned long long* kc = cells + j0 * ws + cj;
                const uint32_t* crow = f.color + (ra + j0) * w;
#pragma unroll
                for (int u = 0; u < RB; ++u) {
                    unsigned long long key = kEmptyKey;
                    if ((FULL || u < nb) && xin) key = kc[0];
                    zb[u] = (uint32_t)(key >> 32);
                    fr[u] = 0.0f;
                    c0[u] = c1[u] = 0u;
                    if (key != kEmptyKey) {
                        reach |= 1u << u;
                        if (!interp) {
                            c0[u] = crow[min(((int)(uint32_t)key << lg) + (lane & (div - 1)), w - 1)];
                        } else {
                            float d = __uint_as_float((uint32_t)key);  // disp of the winner
                            if (side) {
                                const unsigned long long kn = kc[nside];
                                if (kn != kEmptyKey)
                                    d = __fadd_rn(d, __fmul_rn(__fsub_rn(__uint_as_float((uint32_t)kn), d), nwt));
                            }
                            // the row's end texels: a coordinate clamped to [0, w - 1] (where the
                            // fraction is 0, the second texel does not count)
                            const float uc = fminf(fmaxf(__fadd_rn(xf, d), 0.0f), wlast);
                            const float fl = floorf(uc);
                            const int i0 = (int)fl;
                            fr[u] = __fsub_rn(uc, fl);
                            c0[u] = crow[i0];
                            c1[u] = crow[min(i0 + 1, w - 1)];
                        }
                    }
                    kc += ws;
                    crow += w;
                }
                int so = j0 * wpad + x, vo = (ra + j0) * w + x;
#pragma unroll
                for (int u = 0; u < RB; ++u) {
                    if (FULL || u < nb) {  // uniform
                        const bool reached = (reach >> u) & 1u;
                        const uint32_t m = __ballot_sync(0xffffffffu, reached);
                        if (lane == 0 && YORO_BOUND(j0 + u < slots, kBadResolve)) s.bits[(j0 + u) * nwords + g] = m;
                        const bool band = ra + j0 + u >= y0 && ra + j0 + u < y1;
                        if (band && xin) f.mask[vo] = reached ? 0 : 1;
                        if (reached) {
                            uint32_t col = c0[u];
                            if (interp) {
                                // per channel RN(v0 + RN((v1 - v0) fr)), rounded half to even: bytes under
                                // the exponent of 2^23 give v1 - v0 exactly, and adding 2^23 to the result
                                // (in [0, 255]) rounds it to an integer in the low byte
                                uint32_t b[4];
#pragma unroll
                                for (int ch = 0; ch < 4; ++ch) {
                                    const float e0 = __uint_as_float(__byte_perm(c0[u], 0x4B00u, 0x5440u + ch));
                                    const float e1 = __uint_as_float(__byte_perm(c1[u], 0x4B00u, 0x5440u + ch));
                                    const float r =
                                        __fadd_rn(__fsub_rn(e0, 8388608.0f), __fmul_rn(__fsub_rn(e1, e0), fr[u]));
                                    b[ch] = __float_as_uint(__fadd_rn(r, 8388608.0f));
                                }
                                col = __byte_perm(__byte_perm(b[0], b[1], 0x0040u), __byte_perm(b[2], b[3], 0x0040u),
                                                  0x5410u);
                            }
                            if (YORO_BOUND(so < slots * wpad, kBadResolve)) {
                                s.zt[so] = zb[u];
                                s.rgba[so] = col;
                            }
                            if (band) f.out[vo] = col;
                        }
                    }
                    so += wpad;
                    vo += w;
                }
            };
            int j0 = 0;
            for (; j0 + RB <= nr; j0 += RB) batch(std::true_type{}, j0, RB);
            if (j0 < nr) batch(std::false_type{}, j0, nr - j0);
        }
        __syncthreads();
        fill_band<NT, VAR>(f, y0, y1, s, ctr, rowinfo);
    }
}

// Two shapes: 1024 threads with one CTA per SM (large bands), or 512 threads with
// two CTAs per SM (bands small enough that two fit in shared memory).
constexpr int kBig = 1024;
constexpr int kSmall = 512;

}  // namespace

int fused_wpad(int w) { return ((w + 7) / 8) * 8; }

unsigned fused_status_take()
{
#ifdef YORO_DEBUG_BOUNDS
    unsigned v = 0, z = 0;
    if (cudaMemcpyFromSymbol(&v, g_status, sizeof v) != cudaSuccess ||
        cudaMemcpyToSymbol(g_status, &z, sizeof z) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return v;
#else
    return 0;
#endif
}

cudaError_t debug_selftest_launch(cudaStream_t stream)
{
    selftest_kernel<<<1, 32, 0, stream>>>();
    return cudaGetLastError();
}

bool debug_bounds_built()
{
#ifdef YORO_DEBUG_BOUNDS
    return true;
#else
    return false;
#endif
}

size_t fused_smem_bytes(int wpad, int band, int halo)
{
    const size_t slots = (size_t)band + 2 * (size_t)halo;
    // per pixel a source/depth word and a color word; per 32-pixel word a reached
    // bitmask and a hole prefix sum; two counters (16 bytes); per window row a last
    // reached column and a hole offset
    return slots * (size_t)wpad * 8 + slots * (size_t)((wpad + 31) / 32) * 8 + 16 + slots * 8;
}

cudaError_t fused_configure(int device, FusedLimits* lim)
{
    int smem_optin = 0, sms = 0, smem_sm = 0;
    cudaError_t e = cudaDeviceGetAttribute(&smem_optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, device);
    if (e != cudaSuccess) return e;
    e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device);
    if (e != cudaSuccess) return e;
    e = cudaDeviceGetAttribute(&smem_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, device);
    if (e != cudaSuccess) return e;
    lim->sms = sms;
    lim->smem_per_block = smem_optin;
    lim->smem_per_sm = smem_sm;
    int wmax = 0;  // widest frame with a band of one row
    while (fused_smem_bytes(fused_wpad(wmax + 32), 1, 1) <= (size_t)smem_optin && wmax + 32 <= 65535) wmax += 32;
    lim->max_width = wmax;
    const void* fns[] = {(const void*)fused_single<kBig, 1, false>, (const void*)fused_single<kSmall, 2, false>,
                         (const void*)fused_single<kBig, 1, true>,  (const void*)fused_single<kSmall, 2, true>,
                         (const void*)fused_single<kBig, 1, false, true>, (const void*)fused_single<kSmall, 2, false, true>,
                         (const void*)fused_batch<kBig, 1>,         (const void*)fused_batch<kSmall, 2>,
                         (const void*)fused_batch<kBig, 1, true>,   (const void*)fused_batch<kSmall, 2, true>,
                         (const void*)fused_single<kBig, 1, false, false, true>,
                         (const void*)fused_batch<kBig, 1, false, true>,
                         (const void*)fill_only<kBig, false>,       (const void*)fill_only<kBig, true>,
                         (const void*)fill_keys<kBig, false, true>, (const void*)fill_keys<kBig, true, true>,
                         (const void*)fill_keys<kBig, false, false>, (const void*)fill_keys<kBig, true, false>,
                         (const void*)imb_band<kBig, false>,        (const void*)imb_band<kBig, true>};
    for (const void* fn : fns) {
        e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_optin);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

// Largest band whose rows fit the per-CTA shared memory.
static int max_band(const FusedLimits& lim, int wpad, int halo)
{
    if (wpad <= 0) return 1;
    int b = 1;
    while (b < 4096 && fused_smem_bytes(wpad, b + 1, halo) <= (size_t)lim.smem_per_block) ++b;
    return b;
}

// Band height for h rows in bands of at most bmax rows on `sms` CTAs at a time: the height with
// the least (waves of bands) x (rows a band works on, plus about three rows' worth of fixed
// cost).  Bands of all bmax rows can leave the last wave nearly empty: 1920 rows in bands of
// 10 are 192 bands, two waves for 152 SMs, and bands of 7 (275) are two waves of 9 rows
// each instead of 12 (1832x1920 through the intermediate buffer, 4 px per cell: 69 -> 58 us with
// the bands alone).  A frame whose slowest band falls into the last wave can lose what the others
// gain: of 24 seeds each, against bands of bmax rows dealt by stride, plain frames of 2064x2208
// take 0.68 to 0.95 of the time (mean 0.82), 1832x1920 with 5 kernel rows 0.67 to 1.23 (0.84; three
// seeds above 1), through the buffer 1832x1920 0.58 to 0.98 (2 and 4 px per cell: 0.81 and
// 0.72), 2064x2208 0.63 to 1.10 (0.81 and 0.88; one seed each above 1).
static int balanced_band(int h, int halo, int bmax, int sms)
{
    int best = 1;
    long long cost = -1;
    for (int b = 1; b <= bmax; ++b) {
        const long long waves = ((h + b - 1) / b + sms - 1) / sms;
        const long long c = waves * (b + 2 * halo + 3);
        if (cost < 0 || c <= cost) {
            cost = c;
            best = b;
        }
        if (waves <= 1) break;  // taller bands only leave SMs idle
    }
    return best;
}

// Band height for a w x h frame: enough bands for every SM, each as tall as shared
// memory allows up to that.  Two CTAs per SM when two such bands fit on an SM.
FusedShape fused_shape(const FusedLimits& lim, int w, int h, int halo)
{
    const int wpad = fused_wpad(w);
    const int bmax = max_band(lim, wpad, halo);
    FusedShape s;
    int band = (h + lim.sms - 1) / lim.sms;
    if (band > bmax) {  // more than one wave: one CTA per SM fills it
        s.band = balanced_band(h, halo, bmax, lim.sms);
        s.two_per_sm = 0;
        return s;
    }
    if (band < 1) band = 1;
    // two CTAs of half the band height, if they fit beside each other
    const int half = (band + 1) / 2;
    if (band >= 2 && 2 * (fused_smem_bytes(wpad, half, halo) + 1024) <= (size_t)lim.smem_per_sm) {
        s.band = half;
        s.two_per_sm = 1;
    } else {
        s.band = band;
        s.two_per_sm = 0;
    }
    return s;
}

cudaError_t fused_launch(const FrameArgs& f, const FusedLimits& lim, int two_per_sm, cudaStream_t stream)
{
    const int wpad = fused_wpad(f.w);
    const size_t smem = fused_smem_bytes(wpad, f.band, f.halo);
    const bool var = f.halo != 1 || f.nearest != 0;  // a Patcher variant: its own instantiation
    const int nbands = (f.h + f.band - 1) / f.band;
    // One CTA per band, as in the other band kernels: the hardware deals the later waves' bands to
    // whichever SM is free.  Striding over the bands left a slow band's CTA with its next one
    // (2064x2208, 24 seeds: mean 45.3 -> 42.6 us, one seed 48.1 -> 38.3).
    const int grid = nbands;
    if (f.zt_out && var) return cudaErrorInvalidValue;  // the depth output exists for the default kernel
    const bool wide = (f.w + 31) / 32 > 2 * (kBig / 32);  // wider than 2 words per warp
    auto go = [&](auto kernel, int threads) {
        return launch_after(kernel, (unsigned)grid, threads, smem, stream, f, wpad);
    };
    if (two_per_sm) {
        if (f.zt_out) return go(fused_single<kSmall, 2, false, true>, kSmall);
        return var ? go(fused_single<kSmall, 2, true>, kSmall) : go(fused_single<kSmall, 2, false>, kSmall);
    }
    if (f.zt_out) return go(fused_single<kBig, 1, false, true>, kBig);
    if (var) return go(fused_single<kBig, 1, true>, kBig);
    return wide ? go(fused_single<kBig, 1, false, false, true>, kBig) : go(fused_single<kBig, 1, false>, kBig);
}

cudaError_t fused_launch_batch(const BatchArgs& a, int wmax, const FusedLimits& lim, cudaStream_t stream, bool zt)
{
    const int wpad = fused_wpad(wmax);
    const size_t smem = fused_smem_bytes(wpad, a.max_band, 1);  // batch frames use the default kernel
    const bool two = 2 * (smem + 1024) <= (size_t)lim.smem_per_sm;
    // One CTA per (frame, band) item: the hardware block scheduler hands the next item to
    // whichever SM frees up first, so bands with heavy disocclusions do not hold back the
    // rest of the batch.
    const int grid = a.total_items;
    if (grid < 1) return cudaSuccess;
    const bool wide = (wmax + 31) / 32 > 2 * (kBig / 32);  // a frame wider than 2 words per warp
    auto go = [&](auto kernel, int threads) {
        return launch_after(kernel, (unsigned)grid, threads, smem, stream, a, wpad);
    };
    if (two) return zt ? go(fused_batch<kSmall, 2, true>, kSmall) : go(fused_batch<kSmall, 2>, kSmall);
    if (zt) return go(fused_batch<kBig, 1, true>, kBig);
    return wide ? go(fused_batch<kBig, 1, false, true>, kBig) : go(fused_batch<kBig, 1>, kBig);
}

int fused_max_band(const FusedLimits& lim, int w, int halo) { return max_band(lim, fused_wpad(w), halo); }

static size_t imb_cells_offset(int w, int band, int halo)
{
    return (fused_smem_bytes(fused_wpad(w), band, halo) + 15) & ~(size_t)15;
}

size_t imb_band_smem_bytes(int w, int band, int halo, int div)
{
    const int ws = (w + div - 1) / div;
    return imb_cells_offset(w, band, halo) + (size_t)(band + 2 * halo) * (size_t)ws * sizeof(unsigned long long);
}

int imb_band_max(const FusedLimits& lim, int w, int halo, int div)
{
    int b = 0;
    while (b < 4096 && imb_band_smem_bytes(w, b + 1, halo, div) <= (size_t)lim.smem_per_block) ++b;
    return b;
}

cudaError_t imb_band_launch(FrameArgs f, int div, int interp, const FusedLimits& lim, cudaStream_t stream)
{
    f.band = balanced_band(f.h, f.halo, max(1, imb_band_max(lim, f.w, f.halo, div)), lim.sms);
    const size_t smem = imb_band_smem_bytes(f.w, f.band, f.halo, div);
    const int nbands = (f.h + f.band - 1) / f.band;
    if (nbands < 1) return cudaSuccess;
    const int wpad = fused_wpad(f.w), cells = (int)imb_cells_offset(f.w, f.band, f.halo);
    const auto kernel = f.halo == 1 && !f.nearest ? imb_band<kBig, false> : imb_band<kBig, true>;
    return launch_after(kernel, (unsigned)nbands, kBig, smem, stream, f, div, interp, wpad, cells);
}

cudaError_t fill_only_launch(FrameArgs f, const float* zt, const FusedLimits& lim, cudaStream_t stream)
{
    const int wpad = fused_wpad(f.w);
    f.band = balanced_band(f.h, f.halo, max(1, max_band(lim, wpad, f.halo)), lim.sms);
    const size_t smem = fused_smem_bytes(wpad, f.band, f.halo);
    const int grid = (f.h + f.band - 1) / f.band;
    if (grid < 1) return cudaSuccess;
    const auto kernel = f.halo == 1 && !f.nearest ? fill_only<kBig, false> : fill_only<kBig, true>;
    return launch_after(kernel, (unsigned)grid, kBig, smem, stream, f, zt, wpad);
}

// fill_keys: the window and, if any, its words' largest depths.
static size_t keys_smem_bytes(int wpad, int band, int halo, bool zmax)
{
    return fused_smem_bytes(wpad, band, halo) + (zmax ? (size_t)(band + 2 * halo) * (size_t)((wpad + 31) / 32) * 4 : 0);
}

static bool keys_zmax(const FusedLimits& lim, int w, int halo)
{
    return keys_smem_bytes(fused_wpad(w), 1, halo, true) <= (size_t)lim.smem_per_block;
}

// The largest depths take 1.5 % more shared memory, so some frames' one-row window fits without
// them only (9,249 to 9,384 columns for 3 kernel rows, 1,849 to 1,872 for 15).  Those with up to 7
// rows go without, still filled by bands; with more rows, where a band is mostly halo, a gather
// and one thread per hole pixel is faster.  h = 1024, wide occluders / 40-pixel runs of depths,
// bands against gather, us: 3 rows at 9317 columns 344 / 420 against 786 / 862, 5 rows at 5589
// 248 / 348 against 390 / 516, 7 rows at 3989 447 / 331 against 410 / 374, 9 rows at 3105
// 307 / 340 against 276 / 281, 15 rows at 1861 205 / 356 against 212 / 281.
bool fill_keys_takes(const FusedLimits& lim, int w, int halo) { return keys_zmax(lim, w, halo) || halo <= 3; }

cudaError_t fill_keys_launch(FrameArgs f, const unsigned long long* keys, const FusedLimits& lim, cudaStream_t stream)
{
    const int wpad = fused_wpad(f.w);
    const bool zmax = keys_zmax(lim, f.w, f.halo);
    int bmax = 1;
    while (bmax < 4096 && keys_smem_bytes(wpad, bmax + 1, f.halo, zmax) <= (size_t)lim.smem_per_block) ++bmax;
    f.band = balanced_band(f.h, f.halo, bmax, lim.sms);
    const size_t smem = keys_smem_bytes(wpad, f.band, f.halo, zmax);
    const int grid = (f.h + f.band - 1) / f.band;
    if (grid < 1) return cudaSuccess;
    const bool var = f.halo != 1 || f.nearest;
    const auto kernel = zmax ? (var ? fill_keys<kBig, true, true> : fill_keys<kBig, false, true>)
                             : (var ? fill_keys<kBig, true, false> : fill_keys<kBig, false, false>);
    return launch_after(kernel, (unsigned)grid, kBig, smem, stream, f, keys, wpad);
}

}  // namespace yoro
