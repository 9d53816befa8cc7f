// Internal interface of the learned inpainter (unet.cu, unet_train.cu).
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>

#include <cstddef>
#include <cstdint>

namespace yoro {

// Parameters of the network: 14 3x3 layers (enc0a, enc0b, ..., enc3b, dec2a, dec2b, dec1a,
// dec1b, dec0a, dec0b) and the 1x1 output layer, in the order of the definition.
struct UnetLayer {
    int cin, cout, cin_pad;
    uint16_t* wk;  // device, K-major bfloat16
    float* bias;   // device
};

struct UnetNet {
    UnetLayer conv[14];
    float* wout;  // device: 3 x 32 (bfloat16 values as floats), then 3 biases
    int max_tiles;
    // activations, NHWC bfloat16, for max_tiles tiles.  A training net keeps the concatenations
    // of levels 0 and 1 (the weight gradients read them); an inference net keeps their parts:
    // the skips, and the lower levels' outputs at their own resolution.
    uint16_t *in0, *e0a, *cat0, *skip0, *d1b, *p0, *e1a, *cat1, *skip1, *d2b, *p1, *e2a, *cat2, *p2, *e3a, *d2a, *d1a,
        *d0a, *d0b;
    int *flags, *list, *count;
    int max_grid_tiles;  // capacity of flags / list
};

// Driver entry point for tensor-map encoding, looked up once through the runtime (no link
// against the driver library); nullptr if it is missing.
using EncodeTiled = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                 const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                 CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
EncodeTiled tensor_map_encoder();

struct FrameTable;

// One 3x3 convolution: x (T tiles of H x W, NHWC bf16 with Cin channels), K-major weights wk,
// bias, output y at channel y_coff of y_cstride channels (upsample: into the 2H x 2W grid).
// count: optional device count of live tiles.  pool: optional T x H/2 x W/2 x Cout copy of
// the output's 2x2 maximum.  rgb or frames: instead of y, the network's output layer (wout:
// 3 x 32 weights and 3 biases) of every pixel, as colors (T x H x W x 3 floats) or composed
// into the frames of the listed tiles.
struct ConvCall {
    const void* x;
    const void* wk;
    void* y;
    const float* bias;
    const int* count;
    void* pool;
    int T, H, W, Cin, Cout, y_cstride, y_coff, upsample, relu;
    const float* wout = nullptr;
    float* rgb = nullptr;
    const FrameTable* frames = nullptr;
    const int* list = nullptr;
    // optional (row form only): x holds the first cskip channels, low (T x H/2 x W/2, dense) the
    // others, read through their nearest upsampling
    const void* low = nullptr;
    int cskip = 0;
    // the kernel before in the stream writes nothing that this one reads in its prologue (biases,
    // output weights, count): start the prologue while it ends
    bool pdl = false;
};

// Where a pass of the network ends: colors, frames, or (neither) the activations in d0b.
struct NetOut {
    float* rgb;
    const FrameTable* frames;
};

// conv_rows.cu: the row form of the convolution.  conv_rows_takes(): whether a shape that
// the halo form accepts can run as rows.
bool conv_rows_takes(int H, int W, int Cout);
cudaError_t conv_rows_launch(const ConvCall& c, int sms, int smem_max, cudaStream_t stream);
unsigned conv_rows_status_take();

// conv_dw.cu: the weight gradient of one layer from its dZ (T x side x side x cout, dense) and
// input X (channel stride xcs), into dW (cout, cin, 3, 3), overwritten.  ws: workspace of
// conv_dw_workspace() bytes for the same sms.  The network's levels only (side 64, 32, 16, 8
// with 32, 64, 128, 256 output channels).
size_t conv_dw_workspace(int sms);
cudaError_t conv_dw_launch(const void* dZ, const void* X, int xcs, int T, int side, int cin, int cout, int sms, float* ws,
                           float* dW, cudaStream_t s);
unsigned conv_dw_status_take();
int sm_count();

size_t unet_param_count();
void unet_layer_dims(int i, int* cin, int* cout);
UnetNet* unet_create(const float* params, size_t n_params, int max_tiles, int max_grid_tiles, bool train);
void unet_free(UnetNet* n);
cudaError_t unet_run(UnetNet* n, const uint16_t* x, int T, const int* count, const NetOut& out, cudaStream_t s);
cudaError_t unet_conv3x3(const ConvCall& call, cudaStream_t stream);
// The output layer (1x1 convolution, sigmoid) of T tiles' d0b activations into rgb (T x 64 x 64 x 3).
cudaError_t unet_output_rgb(const UnetNet* n, int T, float* rgb, cudaStream_t s);
// The host's round-to-nearest-even float -> bfloat16 rule (NaN kept NaN).
void host_bf16(const float* src, size_t n, uint16_t* dst);

}  // namespace yoro
