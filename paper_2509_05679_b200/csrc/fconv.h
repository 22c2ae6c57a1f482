// Geometry and small device helpers shared by the convolutions off the TMA/tcgen05 path: the packed-FMA kernels (fconv.cu) and the
// warp-level tensor-core kernels (mconv.cu), which cut an image into the same tiles.
#pragma once
#include "kernels.h"

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace fdg {

typedef __nv_bfloat16 bf16;

constexpr int FC_PIX = 128;              // destination pixels per tile
constexpr int FC_CO = 16;
constexpr int FC_KC = 16;                // channels per chunk
constexpr int PITCH = 20;                // floats per pixel (or weight row) in shared memory: 16 + 4, so that the eight 16-byte reads
                                         // of neighbouring pixels fall into different banks
constexpr int FW_CO = 16, FW_CI = 16;
constexpr int FW_CTAS = 3 * 148, MW_CTAS = 4 * 148;      // of a weight gradient, fconv.cu's and mconv.cu's: as many as registers allow at a time
constexpr size_t FC_SMEM_MAX = 224 * 1024;

struct FcParams {
    int H, W, C;                         // input tensor (the error gradient in the backward direction)
    int Ho, Wo, Co;                      // output tensor
    int Hd, Wd, os, xs;                  // destination grid of a class, its stride in the output, stride of the input per destination pixel
    int ngroup;                          // images per group (a group has its own weights)
    int ncls, cls_tap0[5], cls_oph[4], cls_opw[4];       // output parity classes (one, unless this is a stride-2 input gradient)
    int cls_h0[4], cls_w0[4], cls_rh[4], cls_rw[4];      // per class: offset and size of the input region of a tile
    int toff[9], wtap[9];                // per tap: offset inside the region (floats), index of its weights
    int Wt, Ht, Nt, lw, lh, tiles_w, tiles_h;            // tile = Wt x Ht x Nt = 128 destination pixels (powers of two)
    int taps;                            // taps of the weight tensor
    int back;                            // 0: B[n][k] = W[n][tap][k]; 1: B[n][k] = W[k][tap][n]
    size_t w_group, b_group;             // elements between the groups' weights / biases
    int epi;
    int x_floats, w_floats, buffers;     // shared memory of one buffer
};

struct FwParams {
    int H, W, C, Ho, Wo, Co;
    int step;                            // pixels of x between neighbours of the region (the stride for 1x1 layers, else 1)
    int pad, hstep;                      // region origin = tile origin * hstep - pad
    int RH, RW, ntaps, toff[9];          // region of a tile; per tap: offset inside it (floats)
    int Wt, Ht, Nt, lw, lh, tiles_w, tiles_h, tiles;     // tile = Wt x Ht x Nt output pixels (powers of two)
    int ngroup, splits, ci_blocks;
    int nslices, pps;                    // pixel slices of a tile, pixels per slice
    int x_floats;
};

// Geometry of a forward (back == false) or input-gradient launch over `groups` groups of g.N / groups images; false: not covered.
bool plan_fc(const ConvGeom& g, int groups, bool back, FcParams& p);
// Of a weight gradient by `ctas` CTAs; smem: of fw_kernel.
bool plan_fw(const ConvGeom& g, int groups, int ctas, FwParams& p, int& G, int& run, size_t& smem);

// Work of one pass of a layer for the profiler: multiply-adds, and its two activations and its weights (fp32 gradients) once each.
inline double conv_flops(const ConvGeom& g) { return 2.0 * g.N * g.Ho * g.Wo * g.Co * g.R * g.R * g.C; }
inline double conv_bytes(int dt, const ConvGeom& g, bool wgrad) {
    const double w = (double)g.R * g.R * g.C * g.Co, e = dt ? 2.0 : 4.0;
    return e * ((double)g.N * g.H * g.W * g.C + (double)g.N * g.Ho * g.Wo * g.Co) + (wgrad ? 4.0 : e) * w;
}

// The tensor-core forms (mconv.cu), tried first by the fconv_* functions; false / 0: not covered or refused, nothing launched.
// mconv_wgrad leaves partial matrices as fw_kernel does and returns their number per block.
bool mconv_forward(int dt, const void* x, const void* w, const Packed& pk, const float* bias, void* y, float* stat, const ConvGeom& g, int epi, int groups, size_t w_group, size_t b_group,
                   cudaStream_t s);
bool mconv_dgrad(int dt, const void* dy, const void* w, const Packed& pk, void* dx, const ConvGeom& g, int epi, int groups, size_t w_group, cudaStream_t s);
int  mconv_wgrad(int dt, const void* x, const void* dy, float* ws, const ConvGeom& g, int groups, cudaStream_t s);

__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, bool valid) {
    const int n = valid ? 16 : 0;        // 0: the 16 bytes are zero-filled
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(n) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

template <typename T> __device__ __forceinline__ float stored(float v);
template <> __device__ __forceinline__ float stored<float>(float v) { return v; }
template <> __device__ __forceinline__ float stored<bf16>(float v) { return __bfloat162float(__float2bfloat16_rn(v)); }

// sum += part, compensated: part, which started at what the sum lost last time, becomes what it loses this time
__device__ __forceinline__ void kahan(float2& sum, float2& part) {
    const float2 t = __fadd2_rn(sum, part);
    const float2 d = __fadd2_rn(t, make_float2(-sum.x, -sum.y));
    part = __fadd2_rn(part, make_float2(-d.x, -d.y));
    sum = t;
}

}  // namespace fdg
