// Second-eye synthesis for a general pose of the second eye: Eq. 5 with a general
// M = (VP_left)^-1 VP_right, the eye rotated and offset in any direction, so a pixel
// may leave its row (observation O1 no longer holds).
//
// Reading (the oracle's, step for step): both eyes share the pinhole intrinsics; the
// second eye sits at c (left-eye camera coordinates) with rotation rot, p' = rot (p - c).
//   1. Per source pixel (y, x): zc = clamp(depth) (Alg. 1);
//      p = (((x + 0.5) - cx) zc / fx, ((y + 0.5) - cy) zc / fy, zc); q = p - c;
//      p' = rot q, each component ((r0 q0 + r1 q1) + r2 q2); dropped unless p'.z > 0;
//      target (floor(fx p'.x / p'.z + cx), floor(fy p'.y / p'.z + cy)), dropped outside.
//   2. Alg. 2 over the frame: the nearest p'.z per target, the lower source index
//      y w + x on equal depth: a 64-bit atomicMin of (p'.z bits << 32 | index).
//   3. Gather: the winner's color; p'.z is the target's depth.
//   4. Holes along each row and the Patcher (Alg. 3, Eq. 6) over the gathered image:
//      when a band fits shared memory, the fused kernel's band fill reading the keys
//      itself (fill_keys in fused.cu: steps 3 and 4 in one kernel), else a gather pass
//      and one thread per hole pixel.
// Every float operation is an explicit round-to-nearest intrinsic (IEEE division
// included), never contracted, so the result equals the oracle's byte for byte.
#include <cuda_runtime.h>

#include <cstdint>

#include "pose_grid.h"
#include "yoro_device.cuh"
#include "yoro_internal.h"

namespace yoro {

namespace {

#ifdef YORO_DEBUG_BOUNDS
__device__ unsigned g_status;  // debug-bounds status word of this file's kernels
__device__ __forceinline__ void yoro_status_record(unsigned code) { atomicOr(&g_status, code); }
#endif

__device__ __forceinline__ float dot3(const float* r, float q0, float q1, float q2)
{
    return __fadd_rn(__fadd_rn(__fmul_rn(r[0], q0), __fmul_rn(r[1], q1)), __fmul_rn(r[2], q2));
}

// a / b, correctly rounded, for a constant b whose correctly rounded reciprocal y is at hand:
// the quotient estimate a y is corrected twice by its exact remainder (Markstein, "Computation
// of elementary functions on the IBM RISC System/6000 processor", 1990: with y = RN(1/b) and a
// faithful q, RN(q + RN(a - b q) y) is RN(a / b); the first correction makes q faithful).
// Needs normal numbers throughout (pose_fast()).
__device__ __forceinline__ float div_const(float a, float b, float y)
{
    float q = __fmul_rn(a, y);
    q = __fmaf_rn(__fmaf_rn(-q, b, a), y, q);
    return __fmaf_rn(__fmaf_rn(-q, b, a), y, q);
}

// floor(RN(RN(a / Z) + c)) as a float.  The estimate t = RN(a r + c), r = rcp.approx(Z) (within
// 1 ulp), differs from RN(RN(a / Z) + c) by less than (2^-23 + 2^-24) |a / Z| + 2^-23 |t| (1 +
// 2^-20), and |a / Z| <= (|t| + |c|) (1 + 2^-20): by less than 3.1e-7 (|t| + |c|).  Unless an
// integer lies within m = 3.4e-7 (|t| + |c|) + 1e-6 of t, both have the same floor; else, and
// where the estimate is not finite, the division decides.
__device__ __forceinline__ float project(float a, float Z, float c)
{
    const float t = __fmaf_rn(a, rcp_approx(Z), c);
    const float fl = floorf(t);
    const float m = __fmaf_rn(__fadd_rn(fabsf(t), fabsf(c)), 3.4e-7f, 1.0e-6f);
    const float fr = __fsub_rn(t, fl);
    if (fr > m && fr < __fsub_rn(1.0f, m)) return fl;
    return floorf(__fadd_rn(__fdiv_rn(a, Z), c));
}

// Steps 1 and 2.  A block takes 256 columns of kScatterRows rows, a thread one column of
// them: its column's centre is set once and its loads are all in flight before the first is
// used.  The pass is bound by its arithmetic: with four IEEE divisions and a 64-bit division
// for the row per pixel it took 21.9 us at 1832x1920 (18.6 M warp instructions); now 16.6 us
// (12.9 M).  FAST: the divisions by fx and fy
// through their reciprocals, the two by p'.z only where an estimate leaves the target open.
template <bool FAST>
__global__ void __launch_bounds__(kScatterCols) pose_scatter_kernel(FrameArgs f, PoseArgs p, unsigned cols)
{
    const int w = f.w, h = f.h;
    const uint32_t near_m1 = __float_as_uint(f.near_) - 1u, far_m1 = __float_as_uint(f.far_) - 1u;
    const unsigned rg = blockIdx.x / cols, xu = (blockIdx.x - rg * cols) * kScatterCols + threadIdx.x;
    if (xu >= (unsigned)w) return;
    const int x = (int)xu, y0 = (int)rg * kScatterRows;
    const int nr = min(kScatterRows, h - y0);
    const int i0 = y0 * w + x;  // w h < 2^31
    float z[kScatterRows];
#pragma unroll
    for (int r = 0; r < kScatterRows; ++r) z[r] = r < nr ? __ldg(f.depth + i0 + r * w) : 0.0f;
    const float xc = __fsub_rn(__fadd_rn((float)x, 0.5f), p.cx);
#pragma unroll
    for (int r = 0; r < kScatterRows; ++r) {
        if (r >= nr) break;
        const float zc = __uint_as_float(clamped_depth_bits(z[r], near_m1, far_m1));
        const float ax = __fmul_rn(xc, zc);
        const float ay = __fmul_rn(__fsub_rn(__fadd_rn((float)(y0 + r), 0.5f), p.cy), zc);
        const float px = FAST ? div_const(ax, p.fx, p.inv_fx) : __fdiv_rn(ax, p.fx);
        const float py = FAST ? div_const(ay, p.fy, p.inv_fy) : __fdiv_rn(ay, p.fy);
        const float q0 = __fsub_rn(px, p.c[0]), q1 = __fsub_rn(py, p.c[1]), q2 = __fsub_rn(zc, p.c[2]);
        const float X = dot3(p.rot, q0, q1, q2), Y = dot3(p.rot + 3, q0, q1, q2), Z = dot3(p.rot + 6, q0, q1, q2);
        if (!(Z > 0.0f)) continue;
        float u, v;
        if (FAST) {
            u = project(__fmul_rn(p.fx, X), Z, p.cx);
            v = project(__fmul_rn(p.fy, Y), Z, p.cy);
        } else {
            u = floorf(__fadd_rn(__fdiv_rn(__fmul_rn(p.fx, X), Z), p.cx));
            v = floorf(__fadd_rn(__fdiv_rn(__fmul_rn(p.fy, Y), Z), p.cy));
        }
        if (!(u >= 0.0f && u < (float)w && v >= 0.0f && v < (float)h)) continue;
        const size_t o = (size_t)(int)v * w + (int)u;
        if (YORO_BOUND(o < (size_t)w * (size_t)h, kBadPose))
            atomicMin(&p.zbuf[o], zkey(__float_as_uint(Z), i0 + r * w));
    }
}

// Whether every division by fx and fy stays among normal numbers (the numerators are zero or
// between 2^-25 near and (2^31 + |c|) far in magnitude), and p'.z below 2^126, where
// rcp.approx.ftz would flush its reciprocal to zero: |p| < 2^93, so |p'.z| < 3 2^30 (2^93 +
// 2^30) < 2^125.  Rotations and positions are only checked to be finite when a handle is made.
bool pose_fast(const FrameArgs& f, const PoseArgs& p)
{
    const float lo = 9.3e-10f, hi = 1.0e9f;  // 2^-30, 2^30
    for (float r : p.rot)
        if (!(r >= -hi && r <= hi)) return false;
    for (float c : p.c)
        if (!(c >= -hi && c <= hi)) return false;
    return p.fx >= lo && p.fx <= hi && p.fy >= lo && p.fy <= hi && f.near_ >= lo && f.far_ <= hi && p.cx >= -hi &&
           p.cx <= hi && p.cy >= -hi && p.cy <= hi;
}

// Step 3: one thread per target pixel.
__global__ void pose_gather_kernel(FrameArgs f, PoseArgs p)
{
    const size_t n = (size_t)f.w * (size_t)f.h;
    for (size_t o = (size_t)blockIdx.x * blockDim.x + threadIdx.x; o < n; o += (size_t)gridDim.x * blockDim.x) {
        const unsigned long long key = p.zbuf[o];
        if (key == kEmptyKey) {
            f.mask[o] = 1;
            continue;
        }
        const uint32_t src = (uint32_t)key;
        f.mask[o] = 0;
        p.zt[o] = __uint_as_float((uint32_t)(key >> 32));
        f.out[o] = YORO_BOUND(src < n, kBadPose) ? f.color[src] : 0u;
    }
}

unsigned blocks_for(size_t n, int threads)
{
    size_t b = (n + threads - 1) / threads;
    return (unsigned)(b > 65535u * 8u ? 65535u * 8u : b);
}

}  // namespace

size_t pose_scratch_bytes(int w, int h)
{
    const size_t n = (size_t)w * (size_t)h;
    return ((n * sizeof(unsigned long long) + 255) & ~(size_t)255) + n * sizeof(float);
}

void pose_bind_scratch(PoseArgs* p, void* scratch, int w, int h)
{
    const size_t n = (size_t)w * (size_t)h;
    p->zbuf = static_cast<unsigned long long*>(scratch);
    p->zt = reinterpret_cast<float*>(static_cast<unsigned char*>(scratch) +
                                     ((n * sizeof(unsigned long long) + 255) & ~(size_t)255));
}

cudaError_t pose_launch(const FrameArgs& f, const PoseArgs& p, const FusedLimits& lim, bool band_fill,
                        cudaStream_t stream)
{
    const size_t n = (size_t)f.w * f.h;
    if (n == 0) return cudaSuccess;
    cudaError_t e = cudaMemsetAsync(p.zbuf, 0xFF, n * sizeof(unsigned long long), stream);
    if (e != cudaSuccess) return e;
    const int threads = 256;
    const ScatterGrid g = scatter_grid(f.w, f.h);
    if (pose_fast(f, p)) pose_scatter_kernel<true><<<g.blocks, kScatterCols, 0, stream>>>(f, p, g.cols);
    else pose_scatter_kernel<false><<<g.blocks, kScatterCols, 0, stream>>>(f, p, g.cols);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    // a band fits shared memory: the band fill reads the keys itself (gather included)
    if (band_fill && fill_keys_takes(lim, f.w, f.halo)) return fill_keys_launch(f, p.zbuf, lim, stream);
    pose_gather_kernel<<<blocks_for(n, threads), threads, 0, stream>>>(f, p);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    return fill_pixels_launch(f, p.zt, stream);
}

unsigned pose_status_take()
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

}  // namespace yoro
