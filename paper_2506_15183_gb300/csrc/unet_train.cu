// Training of the learned hole inpainter on the GPU: forward, loss, backward and Adam, all
// in this library's kernels.
//
// Loss of a batch: the mean over hole pixels and color channels of (s - g)^2, s the
// network's color and g the ground truth in [0, 1].  The backward pass is the chain rule
// layer by layer:
//   output layer  dz = dL/ds s (1 - s); its weight gradient and the gradient of the last
//                 activations (the 1x1 layer's transpose);
//   3x3 layer     dZ = dY where the layer's output is positive (ReLU'), rounded to
//                 bfloat16; the bias gradient sums dZ; the weight gradient correlates the
//                 layer's input with dZ over every pixel (a K = pixels product on the
//                 tensor cores, conv_dw.cu); the input gradient is a 3x3 convolution of dZ with the
//                 kernel flipped in both directions and its channels transposed, run by the
//                 same tcgen05 kernel as the forward (no ReLU, zero bias; outputs wider than
//                 256 channels in slices);
//   routing       a concatenation splits the input gradient by channels, nearest
//                 upsampling sums each 2x2 block, 2x2 max pooling sends each window's
//                 gradient to its first maximum (row-major), and an encoder level's output
//                 gathers its skip path and its pooling path.
// Gradients of activations are bfloat16 where a tensor-core convolution writes or reads
// them and FP32 sums in between.  Adam keeps FP32 master weights and rebuilds the forward's
// K-major bfloat16 weights and the backward's flipped, transposed ones in the same pass.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <new>
#include <vector>

#include "tc.cuh"
#include "unet_internal.h"
#include "yoro.h"
#include "yoro_unet.h"

namespace yoro {

namespace {

__device__ __forceinline__ float bf2f(uint16_t b) { return __uint_as_float((uint32_t)b << 16); }

__device__ __forceinline__ uint16_t f2bf(float v)
{
    const __nv_bfloat16 b = __float2bfloat16_rn(v);
    return *reinterpret_cast<const uint16_t*>(&b);
}

__device__ __forceinline__ float warp_sum(float v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

__global__ void count_holes_kernel(const uint8_t* hole, long long n, int* cnt)
{
    pdl_wait();
    int c = 0;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        c += hole[i] != 0;
    c = (int)warp_sum((float)c);
    if ((threadIdx.x & 31) == 0 && c) atomicAdd(cnt, c);
}

// Eight bfloat16 channels of a 16-byte load.
__device__ __forceinline__ void unpack8(const uint16_t* p, float (&v)[8])
{
    const uint4 q = *reinterpret_cast<const uint4*>(p);
    const uint32_t w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        v[2 * k] = __uint_as_float(w[k] << 16);
        v[2 * k + 1] = __uint_as_float(w[k] & 0xffff0000u);
    }
}

// dZ of eight channels of a pixel: v where the layer's output y is positive (ReLU'), rounded
// to bfloat16 and stored; the bias gradient adds v.
__device__ __forceinline__ void mask8(const float (&v)[8], const float (&y)[8], uint16_t* dz, float (&db)[8])
{
    uint32_t w[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const float a = y[2 * k] > 0.0f ? v[2 * k] : 0.0f, b = y[2 * k + 1] > 0.0f ? v[2 * k + 1] : 0.0f;
        db[2 * k] += a;
        db[2 * k + 1] += b;
        w[k] = (uint32_t)f2bf(a) | ((uint32_t)f2bf(b) << 16);
    }
    *reinterpret_cast<uint4*>(dz) = make_uint4(w[0], w[1], w[2], w[3]);
}

// Adds every thread's sums of N channels (channel group threadIdx.x % groups, the groups a
// power of two up to 32) into s[group * N ..] of shared memory, then adds s to dst.
template <int N>
__device__ __forceinline__ void block_sums(float (&v)[N], int groups, float* s, float* dst)
{
    for (int i = threadIdx.x; i < groups * N; i += blockDim.x) s[i] = 0.0f;
    __syncthreads();
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int k = 0; k < N; ++k) {
        for (int o = groups; o < 32; o <<= 1) v[k] += __shfl_xor_sync(0xffffffffu, v[k], o);
        if (lane < groups) atomicAdd(&s[(threadIdx.x & (groups - 1)) * N + k], v[k]);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < groups * N; i += blockDim.x) atomicAdd(&dst[i], s[i]);
    __syncthreads();
}

// The gradient dZ of a layer's sums (before ReLU), with its bias gradient, from the input
// gradients of the layers that read its output.  A thread takes eight channels of a pixel
// (kDirect, kUp) or of a 2x2 window (kPooled); the blocks stride by whole pixels, so its
// channels stay the same.  These passes are bound by memory (bfloat16 in, bfloat16 out),
// so the routing, ReLU' and the bias sums are one pass with 16-byte accesses and nothing
// is accumulated in global memory in between.
//   kDirect   one consumer at the same pixels: D at channel doff of dcs
//   kUp       the consumer read this layer's output upsampled: the sum of D's 2x2 block; the
//             output itself is the upsampled copy (read at (2y, 2x))
//   kPooled   an encoder level's last layer: its skip consumer's D plus, at the first maximum
//             of each window of its output (row-major), the pooled consumer's P (dense)
enum { kDirect, kUp, kPooled };

template <int KIND>
__global__ void __launch_bounds__(256) dz_kernel(const uint16_t* D, int dcs, int doff, const uint16_t* P,
                                                 const uint16_t* Y, int ycs, int yoff, int side, int C, long long items,
                                                 uint16_t* dZ, float* gb)
{
    pdl_wait();
    __shared__ float s[256];
    const int cg = C >> 3;  // channel groups, a power of two
    const int c = (threadIdx.x & (cg - 1)) << 3;
    float db[8] = {};
    // log2 of the groups and of the side (powers of two)
    const int lc = __ffs(cg) - 1, ls = __ffs(KIND == kPooled ? side >> 1 : side) - 1;
    for (long long i = blockIdx.x * 256ll + threadIdx.x; i < items; i += gridDim.x * 256ll) {
        const long long p = i >> lc;  // pixel, or window
        float v[8], y[8];
        if (KIND == kDirect) {
            unpack8(D + p * dcs + doff + c, v);
            unpack8(Y + p * ycs + yoff + c, y);
            mask8(v, y, dZ + p * C + c, db);
        } else if (KIND == kUp) {
            const long long x = p & (side - 1), r = p >> ls, t = r >> ls, yy = r & (side - 1);
            const long long q = (t * 2 * side + 2 * yy) * 2 * side + 2 * x;
            float e[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) v[k] = 0.0f;
#pragma unroll
            for (int ab = 0; ab < 4; ++ab) {
                unpack8(D + (q + (ab >> 1) * 2 * side + (ab & 1)) * dcs + doff + c, e);
#pragma unroll
                for (int k = 0; k < 8; ++k) v[k] += e[k];
            }
            unpack8(Y + q * ycs + yoff + c, y);
            mask8(v, y, dZ + p * C + c, db);
        } else {
            const int h = side >> 1;
            const long long x = p & (h - 1), r = p >> ls, t = r >> ls, yy = r & (h - 1);
            const long long q0 = (t * side + 2 * yy) * side + 2 * x;
            float g[8], w[4][8];
            int best[8];
            unpack8(P + p * C + c, g);
#pragma unroll
            for (int ab = 0; ab < 4; ++ab) unpack8(Y + (q0 + (ab >> 1) * side + (ab & 1)) * ycs + yoff + c, w[ab]);
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                best[k] = 0;
                float m = w[0][k];
#pragma unroll
                for (int ab = 1; ab < 4; ++ab)
                    if (w[ab][k] > m) {
                        m = w[ab][k];
                        best[k] = ab;
                    }
            }
#pragma unroll
            for (int ab = 0; ab < 4; ++ab) {
                const long long q = q0 + (ab >> 1) * side + (ab & 1);
                unpack8(D + q * dcs + doff + c, v);
#pragma unroll
                for (int k = 0; k < 8; ++k) v[k] += best[k] == ab ? g[k] : 0.0f;
                mask8(v, w[ab], dZ + q * C + c, db);
            }
        }
    }
    block_sums(db, cg, s, gb);
}

// The loss, and the backward pass through the output layer and the last layer's ReLU: dz of
// the sigmoid input at every pixel (0 outside holes), the gradient of the 1x1 weights and
// biases, and dZ of the last 3x3 layer with its bias gradient.  A thread takes eight
// channels of a pixel (four threads a pixel; the first of them adds the loss).
__global__ void __launch_bounds__(256) out_bwd_kernel(const float* rgb, const uint8_t* gt, const uint8_t* hole, long long npx,
                                                      const int* cnt, const uint16_t* a, const float* wout, uint16_t* dZ,
                                                      float* gw, float* gwb, float* gb, float* loss)
{
    pdl_wait();
    __shared__ float s[128];
    const float inv_n = 1.0f / (3.0f * (float)max(*cnt, 1));
    const int c = (threadIdx.x & 3) << 3;
    float w[3][8], dw[3][8] = {}, db[8] = {}, dwb[4] = {};  // dwb: three biases and the loss
#pragma unroll
    for (int j = 0; j < 3; ++j)
#pragma unroll
        for (int k = 0; k < 8; ++k) w[j][k] = wout[32 * j + c + k];
    for (long long i = blockIdx.x * 256ll + threadIdx.x; i < 4 * npx; i += gridDim.x * 256ll) {
        const long long p = i >> 2;
        if (!hole[p]) {  // dz = 0
            *reinterpret_cast<uint4*>(dZ + p * 32 + c) = make_uint4(0u, 0u, 0u, 0u);
            continue;
        }
        float dz[3], v[8], y[8];
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            const float sg = rgb[3 * p + j];
            const float e = sg - (float)gt[3 * p + j] / 255.0f;
            dz[j] = 2.0f * e * inv_n * sg * (1.0f - sg);
            if (c == 0) {
                dwb[j] += dz[j];
                dwb[3] += e * e;
            }
        }
        unpack8(a + p * 32 + c, y);
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            v[k] = w[0][k] * dz[0] + w[1][k] * dz[1] + w[2][k] * dz[2];
#pragma unroll
            for (int j = 0; j < 3; ++j) dw[j][k] += dz[j] * y[k];
        }
        mask8(v, y, dZ + p * 32 + c, db);
    }
    block_sums(db, 4, s, gb);
#pragma unroll
    for (int j = 0; j < 3; ++j) block_sums(dw[j], 4, s, gw + 32 * j);
    dwb[3] *= inv_n;
    // the sums sit in the threads of channel group 0; the others add zeros
    for (int o = 1; o < 32; o <<= 1)
#pragma unroll
        for (int j = 0; j < 4; ++j) dwb[j] += __shfl_xor_sync(0xffffffffu, dwb[j], o);
    if (threadIdx.x < 4) s[threadIdx.x] = 0.0f;
    __syncthreads();
    if ((threadIdx.x & 31) == 0)
#pragma unroll
        for (int j = 0; j < 4; ++j) atomicAdd(&s[j], dwb[j]);
    __syncthreads();
    if (threadIdx.x < 3) atomicAdd(&gwb[threadIdx.x], s[threadIdx.x]);
    if (threadIdx.x == 3) atomicAdd(loss, s[3]);
}

// Adam and the layers' weights, one pass.  A block takes 32 x 32 (co, ci) of one layer (a run
// of 288 consecutive parameters per co; the first layer has 6 ci), updates them (lr = 0: leaves
// them) with coalesced accesses to the parameters, gradient and moments, and writes from
// shared memory, 64 bytes at a time, the forms the kernels read:
//   wk[co][tap][ci]       the forward's K-major weights (bfloat16; the first layer's padding
//                         channels keep the zeros they were created with)
//   wt[ci][8 - tap][co]   the kernel flipped in both directions: the input gradient is a 3x3
//                         convolution of dZ with these
// The last block takes the biases and the output layer (FP32 biases; bfloat16-rounded weights
// as floats).  31 us for 1.9 M parameters; one thread per (co, ci), which wrote wt two bytes at
// a time, took 49, and eight elements' loads in flight per thread 40.
struct WeightTable {
    int block0[15];  // first block of each layer; [14]: the last block
    int woff[14], boff[14], cin[14], cout[14], cin_pad[14];
    uint16_t* wk[14];
    uint16_t* wt[14];
    float* bias[14];
    int out_off;  // 96 weights, then 3 biases
    float* wout;
};

struct AdamArgs {
    float *p, *m, *v;
    const float* g;
    float lr, b1, b2, eps, c1, c2;
    int update;
};

__device__ __forceinline__ float adam_step(const AdamArgs& a, int i)
{
    float p = a.p[i];
    if (a.update) {
        const float gi = a.g[i];
        const float mi = a.b1 * a.m[i] + (1.0f - a.b1) * gi;
        const float vi = a.b2 * a.v[i] + (1.0f - a.b2) * gi * gi;
        a.m[i] = mi;
        a.v[i] = vi;
        p -= a.lr * (mi / a.c1) / (sqrtf(vi / a.c2) + a.eps);
        a.p[i] = p;
    }
    return p;
}

constexpr int kWeightThreads = 576;  // two of a tile's rows of 288

__global__ void __launch_bounds__(kWeightThreads) weights_kernel(const __grid_constant__ WeightTable w, const AdamArgs a)
{
    pdl_wait();
    __shared__ uint16_t s[32][290];  // [co][ci 9 + tap]; 145 words per row: no bank conflict along co
    if ((int)blockIdx.x == w.block0[14]) {
        for (int l = 0; l < 14; ++l)
            for (int i = threadIdx.x; i < w.cout[l]; i += kWeightThreads) w.bias[l][i] = adam_step(a, w.boff[l] + i);
        if (threadIdx.x < 99) {
            const int i = threadIdx.x;
            const float p = adam_step(a, w.out_off + i);
            w.wout[i] = i < 96 ? bf2f(f2bf(p)) : p;
        }
        return;
    }
    int l = 0;
    while ((int)blockIdx.x >= w.block0[l + 1]) ++l;
    const int cin = w.cin[l], cout = w.cout[l], cp = w.cin_pad[l];
    const int cbs = (cin + 31) >> 5, b = blockIdx.x - w.block0[l];
    const int co0 = b / cbs * 32, ci0 = b % cbs * 32;
    const int nci = min(32, cin - ci0), run = nci * 9;
    const int base = w.woff[l] + (co0 * cin + ci0) * 9;
#pragma unroll 4
    for (int i = threadIdx.x; i < 32 * run; i += kWeightThreads) {
        const int co = i / run, k = i - co * run;
        s[co][k] = f2bf(adam_step(a, base + co * cin * 9 + k));
    }
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int r = warp; r < 32 * 9; r += kWeightThreads / 32) {
        const int row = r / 9, tap = r - row * 9;
        if (lane < nci) w.wk[l][((size_t)(co0 + row) * 9 + tap) * cp + ci0 + lane] = s[row][lane * 9 + tap];
        if (row < nci) w.wt[l][((size_t)(ci0 + row) * 9 + 8 - tap) * cout + co0 + lane] = s[lane][row * 9 + tap];
    }
}

// Blocks of a grid-stride pass: at most about four waves, so that the blocks' closing atomics
// on the same few sums stay few.
unsigned blocks_for(long long n) { return (unsigned)std::min<long long>((n + 255) / 256, 608); }

}  // namespace

struct Trainer {
    UnetNet* net;
    int B;
    size_t np;
    float *params, *grads, *m, *v;
    size_t woff[14], boff[14], wout_off, bout_off;
    WeightTable table;
    uint16_t* wt[14];
    // bfloat16 gradients: dZ of the current layer; DX[0]: its input gradient; DX[1..3]: those
    // of the decoder levels' first layers (8, 10, 12), which two layers read
    uint16_t *dZ, *DX[4];
    float *zero_bias, *rgb, *loss;  // loss and nhole follow the gradients in memory
    float* ws;  // partial sums of the weight gradients
    int sms;
    int* nhole;
    int step;
    float lr, b1, b2, eps;
};

namespace {

int layer_side(int i) { return i < 8 ? (64 >> (i / 2)) : (64 >> (2 - (i - 8) / 2)); }

// Where layer i's input gradient lives (Trainer::DX).
int dx_buffer(int i) { return i == 8 ? 1 : i == 10 ? 2 : i == 12 ? 3 : 0; }

void trainer_free(Trainer* t)
{
    if (!t) return;
    unet_free(t->net);
    for (uint16_t* w : t->wt) cudaFree(w);
    for (uint16_t* d : t->DX) cudaFree(d);
    void* bufs[] = {t->params, t->grads, t->m, t->v, t->dZ, t->zero_bias, t->rgb, t->ws};
    for (void* b : bufs) cudaFree(b);
    delete t;
}

// The layers' weights from the parameters, after an Adam step if update.
cudaError_t update_weights(Trainer* t, bool update, cudaStream_t s)
{
    AdamArgs a{t->params, t->m, t->v, t->grads, t->lr, t->b1, t->b2, t->eps, 1.0f, 1.0f, update ? 1 : 0};
    if (update) {
        a.c1 = 1.0f - std::pow(t->b1, (float)t->step);
        a.c2 = 1.0f - std::pow(t->b2, (float)t->step);
    }
    return launch_kernel(weights_kernel, dim3((unsigned)t->table.block0[14] + 1), kWeightThreads, 0, s, true, t->table, a);
}

}  // namespace

Trainer* trainer_create(const float* params, size_t np, int batch, float lr, float b1, float b2, float eps)
{
    if (!params || np != unet_param_count() || batch < 2 || (batch & 1)) return nullptr;
    Trainer* t = new (std::nothrow) Trainer();
    if (!t) return nullptr;
    std::memset(t, 0, sizeof *t);
    t->B = batch;
    t->np = np;
    t->lr = lr;
    t->b1 = b1;
    t->b2 = b2;
    t->eps = eps;
    t->sms = sm_count();
    t->net = unet_create(params, np, batch, 1, true);
    bool ok = t->net != nullptr;
    size_t off = 0;
    for (int i = 0; i < 14; ++i) {
        int cin, cout;
        unet_layer_dims(i, &cin, &cout);
        t->woff[i] = off;
        off += (size_t)cout * cin * 9;
        t->boff[i] = off;
        off += cout;
    }
    t->wout_off = off;
    t->bout_off = off + 96;
    const size_t B = batch;
    size_t dz_max = 0, dx_max[4] = {};
    WeightTable& w = t->table;
    for (int i = 0; i < 14 && ok; ++i) {
        int cin, cout;
        unet_layer_dims(i, &cin, &cout);
        const size_t P = B * layer_side(i) * layer_side(i);
        dz_max = std::max(dz_max, P * cout);
        size_t& dx = dx_max[dx_buffer(i)];
        dx = std::max(dx, P * (size_t)cin);
        ok = cudaMalloc(&t->wt[i], (size_t)cin * 9 * cout * 2) == cudaSuccess;
        const UnetLayer& L = t->net->conv[i];
        w.block0[i + 1] = w.block0[i] + cout / 32 * ((cin + 31) / 32);
        w.woff[i] = (int)t->woff[i];
        w.boff[i] = (int)t->boff[i];
        w.cin[i] = cin;
        w.cout[i] = cout;
        w.cin_pad[i] = L.cin_pad;
        w.wk[i] = L.wk;
        w.wt[i] = t->wt[i];
        w.bias[i] = L.bias;
    }
    if (ok) {
        w.out_off = (int)t->wout_off;
        w.wout = t->net->wout;
        for (int k = 0; k < 4 && ok; ++k) ok = cudaMalloc(&t->DX[k], dx_max[k] * 2) == cudaSuccess;
    }
    if (ok)
        ok = cudaMalloc(&t->params, np * 4) == cudaSuccess && cudaMalloc(&t->grads, (np + 2) * 4) == cudaSuccess &&
             cudaMalloc(&t->m, np * 4) == cudaSuccess && cudaMalloc(&t->v, np * 4) == cudaSuccess &&
             cudaMalloc(&t->dZ, dz_max * 2) == cudaSuccess && cudaMalloc(&t->zero_bias, 384 * 4) == cudaSuccess &&
             cudaMalloc(&t->rgb, B * 4096 * 3 * 4) == cudaSuccess &&
             cudaMalloc(&t->ws, conv_dw_workspace(t->sms)) == cudaSuccess;
    if (ok) {
        t->loss = t->grads + np;
        t->nhole = reinterpret_cast<int*>(t->grads + np + 1);
        ok = cudaMemcpy(t->params, params, np * 4, cudaMemcpyHostToDevice) == cudaSuccess &&
             cudaMemset(t->m, 0, np * 4) == cudaSuccess && cudaMemset(t->v, 0, np * 4) == cudaSuccess &&
             cudaMemset(t->zero_bias, 0, 384 * 4) == cudaSuccess &&
             cudaMemset(t->grads, 0, (np + 2) * 4) == cudaSuccess && update_weights(t, false, nullptr) == cudaSuccess &&
             cudaDeviceSynchronize() == cudaSuccess;
    }
    if (!ok) {
        cudaGetLastError();
        trainer_free(t);
        return nullptr;
    }
    return t;
}

// One step on B tiles (B even, <= the trainer's batch): x (B x 64 x 64 x 32 bfloat16), gt
// (B x 64 x 64 x 3 bytes), hole (B x 64 x 64 bytes).  lr = 0 leaves the weights as they
// are (the gradients stay readable).
cudaError_t trainer_step(Trainer* t, const void* x, const uint8_t* gt, const uint8_t* hole, int B, cudaStream_t s)
{
    UnetNet* n = t->net;
    const long long npx = (long long)B * 4096;
    const uint16_t* xin = static_cast<const uint16_t*>(x);
    // gradients, loss and hole count
    cudaError_t e = cudaMemsetAsync(t->grads, 0, (t->np + 2) * 4, s);
    if (e == cudaSuccess) e = unet_run(n, xin, B, nullptr, NetOut{nullptr, nullptr}, s);
    if (e == cudaSuccess) e = unet_output_rgb(n, B, t->rgb, s);
    if (e != cudaSuccess) return e;
    e = launch_kernel(count_holes_kernel, dim3(blocks_for(npx)), 256, 0, s, true, hole, npx, t->nhole);
    if (e == cudaSuccess)
        e = launch_kernel(out_bwd_kernel, dim3(blocks_for(4 * npx)), 256, 0, s, true, (const float*)t->rgb, gt, hole, npx,
                          (const int*)t->nhole, (const uint16_t*)n->d0b, (const float*)n->wout, t->dZ,
                          t->grads + t->wout_off, t->grads + t->bout_off, t->grads + t->boff[13], t->loss);
    if (e != cudaSuccess) return e;

    // per layer: forward input X (channel stride), output Y (stride, offset)
    struct IO {
        const uint16_t* x;
        int xcs;
        const uint16_t* y;
        int ycs, ycoff;
    };
    const IO io[14] = {{xin, 32, n->e0a, 32, 0},       {n->e0a, 32, n->cat0, 96, 0},
                       {n->p0, 32, n->e1a, 64, 0},     {n->e1a, 64, n->cat1, 192, 0},
                       {n->p1, 64, n->e2a, 128, 0},    {n->e2a, 128, n->cat2, 384, 0},
                       {n->p2, 128, n->e3a, 256, 0},   {n->e3a, 256, n->cat2, 384, 128},
                       {n->cat2, 384, n->d2a, 128, 0}, {n->d2a, 128, n->cat1, 192, 64},
                       {n->cat1, 192, n->d1a, 64, 0},  {n->d1a, 64, n->cat0, 96, 32},
                       {n->cat0, 96, n->d0a, 32, 0},   {n->d0a, 32, n->d0b, 32, 0}};
    // who reads layer i's output: the form of dZ, and the consumer's input gradient
    struct Route {
        int kind, from, off, pooled;  // consumer's layer, channel offset in its input, pooled consumer
    };
    const Route route[13] = {{kDirect, 1, 0, 0},  {kPooled, 12, 0, 2},  {kDirect, 3, 0, 0},  {kPooled, 10, 0, 4},
                             {kDirect, 5, 0, 0},  {kPooled, 8, 0, 6},   {kDirect, 7, 0, 0},  {kUp, 8, 128, 0},
                             {kDirect, 9, 0, 0},  {kUp, 10, 64, 0},     {kDirect, 11, 0, 0}, {kUp, 12, 32, 0},
                             {kDirect, 13, 0, 0}};
    for (int i = 13; i >= 0; --i) {
        const UnetLayer& L = n->conv[i];
        const int side = layer_side(i);
        const long long P = (long long)B * side * side;
        if (i < 13) {
            const Route& r = route[i];
            const uint16_t* D = t->DX[dx_buffer(r.from)];
            const int dcs = n->conv[r.from].cin;
            const long long items = P * (L.cout / 8) / (r.kind == kPooled ? 4 : 1);
            const unsigned blocks = blocks_for(items);
            float* gb = t->grads + t->boff[i];
            const uint16_t* pooled = r.kind == kPooled ? t->DX[dx_buffer(r.pooled)] : nullptr;
            const auto kernel = r.kind == kDirect ? dz_kernel<kDirect> : r.kind == kUp ? dz_kernel<kUp> : dz_kernel<kPooled>;
            e = launch_kernel(kernel, dim3(blocks), 256, 0, s, true, D, dcs, r.off, pooled, io[i].y, io[i].ycs, io[i].ycoff,
                              side, L.cout, items, t->dZ, gb);
            if (e != cudaSuccess) return e;
        }
        e = conv_dw_launch(t->dZ, io[i].x, io[i].xcs, B, side, L.cin, L.cout, t->sms, t->ws, t->grads + t->woff[i], s);
        if (e != cudaSuccess) return e;
        if (i == 0) break;
        // input gradient: slices of 256 / 128 / 64 / 32 output channels
        for (int c0 = 0; c0 < L.cin && e == cudaSuccess;) {
            const int rem = L.cin - c0;
            const int w = rem >= 256 ? 256 : rem >= 128 ? 128 : rem >= 64 ? 64 : 32;
            ConvCall c{t->dZ, t->wt[i] + (size_t)c0 * 9 * L.cout, t->DX[dx_buffer(i)], t->zero_bias, nullptr, nullptr, B,
                       side, side, L.cout, w, L.cin, c0, 0, 0};
            c.pdl = true;
            e = unet_conv3x3(c, s);
            c0 += w;
        }
        if (e != cudaSuccess) return e;
    }
    if (t->lr != 0.0f) {
        ++t->step;
        e = update_weights(t, true, s);
    }
    return e;
}

}  // namespace yoro

struct yoro_unet_trainer_ctx {
    yoro::Trainer* t;
};

extern "C" {

yoro_unet_trainer yoro_unet_trainer_create(const float* params, long long n_params, int batch_tiles, float lr,
                                           float beta1, float beta2, float eps)
{
    if (!params || n_params <= 0 || !(lr >= 0.0f) || !(beta1 >= 0.0f && beta1 < 1.0f) ||
        !(beta2 >= 0.0f && beta2 < 1.0f) || !(eps > 0.0f))
        return nullptr;
    yoro::Trainer* t = yoro::trainer_create(params, (size_t)n_params, batch_tiles, lr, beta1, beta2, eps);
    if (!t) return nullptr;
    yoro_unet_trainer_ctx* c = new (std::nothrow) yoro_unet_trainer_ctx();
    if (!c) {
        yoro::trainer_free(t);
        return nullptr;
    }
    c->t = t;
    return c;
}

void yoro_unet_trainer_destroy(yoro_unet_trainer tr)
{
    if (!tr) return;
    yoro::trainer_free(tr->t);
    delete tr;
}

yoro_status yoro_unet_train_step(yoro_unet_trainer tr, const void* x, const unsigned char* gt,
                                 const unsigned char* hole, int tiles, void* cuda_stream)
{
    if (!tr || !x || !gt || !hole || tiles < 2 || (tiles & 1) || tiles > tr->t->B) return YORO_EINVAL;
    if ((uintptr_t)x & 15u) return YORO_EALIGN;
    return yoro::trainer_step(tr->t, x, gt, hole, tiles, (cudaStream_t)cuda_stream) == cudaSuccess ? YORO_OK
                                                                                                 : YORO_ECUDA;
}

yoro_status yoro_unet_trainer_set_lr(yoro_unet_trainer tr, float lr)
{
    if (!tr || !(lr >= 0.0f) || !std::isfinite(lr)) return YORO_EINVAL;
    tr->t->lr = lr;
    return YORO_OK;
}

yoro_status yoro_unet_trainer_read(yoro_unet_trainer tr, int what, float* host_out, void* cuda_stream)
{
    if (!tr || !host_out || what < 0 || what > 2) return YORO_EINVAL;
    const cudaStream_t s = (cudaStream_t)cuda_stream;
    const float* src = what == 0 ? tr->t->params : what == 1 ? tr->t->grads : tr->t->loss;
    const size_t bytes = what == 2 ? 4 : tr->t->np * 4;
    if (cudaMemcpyAsync(host_out, src, bytes, cudaMemcpyDeviceToHost, s) != cudaSuccess ||
        cudaStreamSynchronize(s) != cudaSuccess) {
        cudaGetLastError();
        return YORO_ECUDA;
    }
    return YORO_OK;
}

}  // extern "C"
