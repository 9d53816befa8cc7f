// Device helpers shared by the inpainter's kernels: the frames of a launch and their 64 x 64
// cells, and the output layer of one pixel.
#pragma once

#include <cuda_runtime.h>

#include <cstddef>
#include <cstdint>

namespace yoro {

constexpr int kTile = 64;  // inference tile: 64 x 64 pixels

// The frames of one inpainting launch.  Their cell grids are concatenated: cell c of frame
// f (c = ty * ntx + tx) is entry off[f] + c, so their hole cells form one list and one pass
// of the network takes them all.
constexpr int kMaxInpaintFrames = 32;

struct FrameTable {
    int n;
    int off[kMaxInpaintFrames + 1];  // off[n]: cells of all frames
    int w[kMaxInpaintFrames], h[kMaxInpaintFrames], ntx[kMaxInpaintFrames];
    float near_[kMaxInpaintFrames];
    uint32_t* rgba[kMaxInpaintFrames];
    const uint8_t* mask[kMaxInpaintFrames];
    const float* zt[kMaxInpaintFrames];
    const float* zsrc[kMaxInpaintFrames];
};

// Frame of concatenated cell g.
__device__ __forceinline__ int table_frame(const FrameTable& ft, int g)
{
    int lo = 0, hi = ft.n - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (ft.off[mid] <= g) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

// Origin of the 64 x 64 window of grid cell (tx, ty): the cell itself, except that the
// last column and row are shifted inward so the window ends at the frame's edge (a frame
// narrower or lower than 64 keeps origin 0 and is padded).  A tile writes its cell only.
__device__ __forceinline__ int window_origin(int t, int size) { return max(0, min(kTile * t, size - kTile)); }

// The output layer at one pixel: a 1x1 convolution of its 32 activations (FP32 sums in
// channel order, then the bias) and the logistic sigmoid 1 / (1 + exp(-z)).  wo (16-byte
// aligned): 3 x 32 weights, then 3 biases.
__device__ __forceinline__ void net_colors(const float (&v)[32], const float* wo, float (&col)[3])
{
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        float acc = 0.0f;
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const float4 w = reinterpret_cast<const float4*>(wo)[c * 8 + q];
            acc = __fadd_rn(acc, __fmul_rn(w.x, v[4 * q]));
            acc = __fadd_rn(acc, __fmul_rn(w.y, v[4 * q + 1]));
            acc = __fadd_rn(acc, __fmul_rn(w.z, v[4 * q + 2]));
            acc = __fadd_rn(acc, __fmul_rn(w.w, v[4 * q + 3]));
        }
        const float z = __fadd_rn(acc, wo[96 + c]);
        col[c] = __fdiv_rn(1.0f, __fadd_rn(1.0f, expf(-z)));
    }
}

// RGBA8 of a repainted pixel: rint(clamp(c, 0, 1) * 255) per color, alpha 255.
__device__ __forceinline__ uint32_t net_rgba(const float (&col)[3])
{
    uint32_t out = 0xff000000u;
#pragma unroll
    for (int c = 0; c < 3; ++c)
        out |= (uint32_t)rintf(__fmul_rn(fminf(fmaxf(col[c], 0.0f), 1.0f), 255.0f)) << (8 * c);
    return out;
}

}  // namespace yoro
