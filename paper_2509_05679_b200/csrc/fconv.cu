// FMA convolutions (CUDA cores, fp32 arithmetic, fp32 or bf16 storage) for the layers the tensor-core kernels do not take: channel counts that
// are no multiple of 16 (the first layer's 3 among them), launches of such channels in which mconv.cu would be slower (worth_it there: small images, few 1x1
// tiles), all of them with kernel_path 1.  3x3 and 1x1, stride 1 and 2, any channel counts, any image size.  The tiles, the partial matrices of a weight gradient and their reduction are shared with mconv.cu.
//
//   fc_kernel : forward and input gradient.  A CTA computes 128 pixels x 16 output channels: the input region of its
//               pixels (halo included) is fetched ONCE per 16-channel chunk and every filter tap reads it from shared memory.
//   fw_kernel : weight gradient.  A CTA keeps a 16 c_out x (taps x 16 c_in) tile of dW in registers over all the pixels of
//               its split; partial sums per CTA, added in a fixed order by fw_reduce_kernel.
//
// Arithmetic: packed fp32 (fma.rn.f32x2: 65.6 TFLOP/s on a B200 where scalar fma gives 46.7).  The pairs lie along the
// contraction (channels 2i and 2i + 1) in fc_kernel and along c_in in fw_kernel, so that operands come out of NHWC data as
// 16-byte vectors without shuffling.  Chains of at most 16 products (fw_kernel: 32 in long sums) are added to a compensated (Kahan) running sum, so the
// rounding error of a long contraction stays at a few ulps.
//
// What bounds them: the FMA pipe (fc_kernel issues 32 packed FMAs for eight 16-byte shared loads, or 16 for six, fw_kernel 16 for four).
// The implicit-GEMM kernel they replace fetched every operand element by itself with two integer divisions and reached
// 2.5-9 TFLOP/s on the ResNet-20 layers.
#include "fconv.h"
#include "kernels.h"
#include "launch.h"

#include <cuda_bf16.h>

namespace fdg {

typedef __nv_bfloat16 bf16;

namespace {

// fc_kernel: 4 rows of 32 pixels x 16 output channels; a thread has PP = 4 or 2 pixels x 4 channels: 4 or 8 warps
constexpr int FW_THREADS = 160;          // 9 taps x 2 groups of 8 c_in x 4 groups of 4 c_out x 2 pixel slices = 144, in five warps: three CTAs put
                                         // four warps on each scheduler and leave 128 registers a thread (nine warps, two CTAs: 96, and spills)

__device__ __forceinline__ float to_f(float v) { return v; }
__device__ __forceinline__ float to_f(bf16 v) { return __bfloat162float(v); }
__device__ __forceinline__ void put(float* p, float v) { *p = v; }
__device__ __forceinline__ void put(bf16* p, float v) { *p = __float2bfloat16_rn(v); }
__device__ __forceinline__ float4 ld4(const float* p) { return *(const float4*)p; }
__device__ __forceinline__ float4 ld4(const bf16* p) {
    const uint2 v = *(const uint2*)p;
    return make_float4(__uint_as_float(v.x << 16), __uint_as_float(v.x & 0xffff0000u), __uint_as_float(v.y << 16), __uint_as_float(v.y & 0xffff0000u));
}
__device__ __forceinline__ void st4(float* p, float4 v) { *(float4*)p = v; }
__device__ __forceinline__ void st4(bf16* p, float4 v) {
    const __nv_bfloat162 a = __floats2bfloat162_rn(v.x, v.y), b = __floats2bfloat162_rn(v.z, v.w);
    *(uint2*)p = make_uint2(*(const uint32_t*)&a, *(const uint32_t*)&b);
}

// The input region of a tile, channels c0 .. c0 + 15, into dst[pixel][PITCH]: nimg images x RH rows x RW pixels whose first
// pixel is (h0, w0) and whose neighbours are `step` pixels apart in the tensor; zeros outside the image, past image n_end
// and past channel C.  A warp takes whole rows, so that the loop has no division.
// VEC: C is a multiple of 4 (16-byte fp32 / 8-byte bf16 pieces); fp32 pieces travel by cp.async.
template <typename T>
__device__ __forceinline__ void load_region(const bool VEC, const T* __restrict__ x, float* dst, int n0, int n_end, int nimg, int h0, int w0, int RH, int RW, int step,
                                            int H, int W, int C, int c0, int nq, int warp, int nwarps, int lane) {
    int ni = 0, rh = warp;
    while (rh >= RH) { rh -= RH; ++ni; }
    while (ni < nimg) {
        const int n = n0 + ni, h = h0 + rh * step;
        const bool row_ok = n < n_end && h >= 0 && h < H;
        const T* src = x + (((size_t)(row_ok ? n : n0) * H + (row_ok ? h : 0)) * W) * C + c0;
        float* d = dst + (size_t)((ni * RH + rh) * RW) * PITCH;
        for (int j = lane; j < RW * 4; j += 32) {
            const int rw = j >> 2, q = j & 3;
            if (q >= nq) continue;
            const int w = w0 + rw * step, c = 4 * q;
            const bool ok = row_ok && w >= 0 && w < W;
            if (VEC) {
                const bool in = ok && c0 + c < C;
                const T* s = src + (in ? (size_t)w * C + c : 0);
                if (sizeof(T) == 4) cp_async16(smem_addr(d + rw * PITCH + c), s, in);
                else *(float4*)(d + rw * PITCH + c) = in ? ld4(s) : make_float4(0.f, 0.f, 0.f, 0.f);
            } else {
                float v[4];
#pragma unroll
                for (int e = 0; e < 4; ++e) v[e] = ok && c0 + c + e < C ? to_f(src[(size_t)w * C + c + e]) : 0.f;
                *(float4*)(d + rw * PITCH + c) = make_float4(v[0], v[1], v[2], v[3]);
            }
        }
        rh += nwarps;
        while (rh >= RH) { rh -= RH; ++ni; }
    }
}

// the two lanes of a sum, with what either has lost
__device__ __forceinline__ float lanes_sum(float2 sum, float2 lost) {
    const float s = __fadd_rn(sum.x, sum.y), b = __fsub_rn(s, sum.x);
    const float e = __fadd_rn(__fsub_rn(sum.x, __fsub_rn(s, b)), __fsub_rn(sum.y, b));          // two-sum: sum.x + sum.y = s + e
    return __fadd_rn(s, __fadd_rn(e, __fadd_rn(lost.x, lost.y)));
}

struct Yes { static constexpr bool value = true; };
struct No { static constexpr bool value = false; };

// 16 output channels x up to 16 input channels of every tap of the class into dst[tap][row][PITCH]; channel n sits in row
// (n % 4) * 4 + n / 4, so that the four channel groups of a warp read neighbouring rows.
template <typename T, bool VEC>
__device__ __forceinline__ void load_weights(const T* __restrict__ w, float* dst, const FcParams& p, int t0, int t1, int co0, int c0, int nq, int tid, int nthreads) {
    for (int i = tid; i < (t1 - t0) * 64; i += nthreads) {
        const int t = i >> 6, e = i & 63;
        const int tap = p.wtap[t0 + t];
        if (!p.back) {
            const int n = e >> 2, q = e & 3;
            if (q >= nq) continue;
            const int co = co0 + n, c = c0 + 4 * q;
            const T* s = w + ((size_t)(co < p.Co ? co : 0) * p.taps + tap) * p.C;
            float4 v;
            if (VEC) v = co < p.Co && c < p.C ? ld4(s + c) : make_float4(0.f, 0.f, 0.f, 0.f);
            else {
                float f[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) f[j] = co < p.Co && c + j < p.C ? to_f(s[c + j]) : 0.f;
                v = make_float4(f[0], f[1], f[2], f[3]);
            }
            *(float4*)(dst + (t * 16 + (n & 3) * 4 + (n >> 2)) * PITCH + 4 * q) = v;
        } else {
            // k runs over the layer's output channels, n over its input channels (contiguous in memory)
            const int k = e >> 2, g = e & 3;
            if (k >= 4 * nq) continue;
            const bool kin = c0 + k < p.C;
            const T* s = w + ((size_t)(kin ? c0 + k : 0) * p.taps + tap) * p.Co;
            float f[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) { const int n = co0 + 4 * g + j; f[j] = kin && n < p.Co ? to_f(s[n]) : 0.f; }
#pragma unroll
            for (int j = 0; j < 4; ++j) dst[(t * 16 + j * 4 + g) * PITCH + k] = f[j];          // channel 4 g + j: row j * 4 + g
        }
    }
}

// CTAs per SM that the register allocation allows: fp32 at four pixels a thread without spills (168 registers: ResNet-20 with one module
// 2.77 -> 2.70 ms per step; bf16, whose operands are unpacked to the same registers, is 3 % faster with four CTAs and ten words spilled).
template <typename T> constexpr int fc_ctas(int pp) { return pp == 2 ? 2 : sizeof(T) == 4 ? 3 : 4; }

// grid = (pixel tiles, blocks of 16 output channels, groups x classes).  NQ: 4-channel quads per chunk (1: at most 4 channels).
template <typename T, int NQ, bool VEC, int PP>
__global__ void __launch_bounds__(512 / PP, fc_ctas<T>(PP)) fc_kernel(const T* __restrict__ x, const T* __restrict__ w, const float* __restrict__ bias, T* __restrict__ y,
                                                           float* __restrict__ stat, const __grid_constant__ FcParams p) {
    extern __shared__ __align__(16) float fsm[];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int cls = blockIdx.z % p.ncls, grp = blockIdx.z / p.ncls;
    int tile = blockIdx.x;
    const int tw = tile % p.tiles_w; tile /= p.tiles_w;
    const int th = tile % p.tiles_h, tn = tile / p.tiles_h;
    const int n_end = (grp + 1) * p.ngroup, n0 = grp * p.ngroup + tn * p.Nt;
    const int hd0 = th * p.Ht, wd0 = tw * p.Wt, co0 = blockIdx.y * FC_CO;
    const int t0 = p.cls_tap0[cls], t1 = p.cls_tap0[cls + 1];
    const int RH = p.cls_rh[cls], RW = p.cls_rw[cls], h0 = hd0 * p.xs + p.cls_h0[cls], w0 = wd0 * p.xs + p.cls_w0[cls];
    w += (size_t)grp * p.w_group;

    // this thread: pixels px0 + 8 i (i = 0..PP - 1), channels co0 + 4 cg + j; warps of the same `row` share 32 pixels
    constexpr int NT = 512 / PP, PARTS = 4 / PP;
    const int g = lane & 7, cg = lane >> 3, row = warp / PARTS, part_of = warp % PARTS, px0 = row * 32 + g + 8 * PP * part_of;
    uint32_t xb[PP];
#pragma unroll
    for (int i = 0; i < PP; ++i) {
        const int px = px0 + 8 * i;
        const int pw = px & (p.Wt - 1), ph = (px >> p.lw) & (p.Ht - 1), pn = px >> (p.lw + p.lh);
        xb[i] = (uint32_t)(((pn * RH + ph * p.xs) * RW + pw * p.xs) * PITCH);
    }
    // fp32 storage: per channel the sums of its even and of its odd products.  bf16 storage: per pair of channels their sums (0, 1) and what the last
    // additions lost (2, 3); rounding the two lanes' sum at every flush adds 2.6 % to an error that the rounded result hides, and the other form
    // spills there (+5 % per step).
    constexpr bool LANES = sizeof(T) == 4;
    float2 acc[PP][4], part[PP][4];
#pragma unroll
    for (int i = 0; i < PP; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) { acc[i][j] = make_float2(0.f, 0.f); part[i][j] = make_float2(0.f, 0.f); }

    const int chunks = t1 > t0 ? (p.C + FC_KC - 1) / FC_KC : 0;
    auto fetch = [&](int c, int buf) {
        float* xs_ = fsm + (size_t)buf * (p.x_floats + p.w_floats);
        load_region<T>(VEC, x, xs_, n0, n_end, p.Nt, h0, w0, RH, RW, 1, p.H, p.W, p.C, c * FC_KC, NQ, warp, NT / 32, lane);
        load_weights<T, VEC>(w, xs_ + p.x_floats, p, t0, t1, co0, c * FC_KC, NQ, tid, NT);
        cp_commit();
    };
    if (chunks) fetch(0, 0);
    for (int c = 0; c < chunks; ++c) {
        const int buf = p.buffers > 1 ? c & 1 : 0;
        if (p.buffers > 1 && c + 1 < chunks) { fetch(c + 1, buf ^ 1); cp_wait<1>(); } else cp_wait<0>();
        __syncthreads();
        const float* xs_ = fsm + (size_t)buf * (p.x_floats + p.w_floats);
        const float* ws_ = xs_ + p.x_floats + cg * PITCH;
        auto tap = [&](int t, auto first) {
            const float* xt = xs_ + p.toff[t0 + t];
            const float* wt = ws_ + t * (16 * PITCH);
#pragma unroll
            for (int q = 0; q < NQ; ++q) {
                float4 wv[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) wv[j] = *(const float4*)(wt + j * (4 * PITCH) + 4 * q);
#pragma unroll
                for (int i = 0; i < PP; ++i) {
                    const float4 xv = *(const float4*)(xt + xb[i] + 4 * q);
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const float2 lo = make_float2(xv.x, xv.y), hi = make_float2(xv.z, xv.w);
                        if (!LANES && decltype(first)::value && q == 0) part[i][j] = __fmul2_rn(lo, make_float2(wv[j].x, wv[j].y));
                        else part[i][j] = __ffma2_rn(lo, make_float2(wv[j].x, wv[j].y), part[i][j]);
                        part[i][j] = __ffma2_rn(hi, make_float2(wv[j].z, wv[j].w), part[i][j]);
                    }
                }
            }
        };
        auto flush = [&]() {             // Kahan
#pragma unroll
            for (int i = 0; i < PP; ++i) {
                if (LANES) {
#pragma unroll
                    for (int j = 0; j < 4; ++j) kahan(acc[i][j], part[i][j]);
                } else {
#pragma unroll
                    for (int j = 0; j < 2; ++j) {
                        const float2 s = make_float2(part[i][2 * j].x + part[i][2 * j].y, part[i][2 * j + 1].x + part[i][2 * j + 1].y);
                        const float2 yv = __fadd2_rn(s, make_float2(-acc[i][2 + j].x, -acc[i][2 + j].y));
                        const float2 t = __fadd2_rn(acc[i][j], yv);
                        const float2 d = __fadd2_rn(t, make_float2(-acc[i][j].x, -acc[i][j].y));
                        acc[i][2 + j] = __fadd2_rn(d, make_float2(-yv.x, -yv.y));
                        acc[i][j] = t;
                    }
                }
            }
        };
        int t = 0;
#pragma unroll 1
        for (; t + 1 < t1 - t0; t += 2) { tap(t, Yes()); tap(t + 1, No()); flush(); }      // two taps x 16 channels: pair chains of 16 products
        if (t < t1 - t0) { tap(t, Yes()); flush(); }
        __syncthreads();
        if (p.buffers == 1 && c + 1 < chunks) fetch(c + 1, 0);
    }

    float val[PP][4];
    bool valid[PP];
    const int co = co0 + 4 * cg;
#pragma unroll
    for (int i = 0; i < PP; ++i) {
        const int px = px0 + 8 * i;
        const int wd = wd0 + (px & (p.Wt - 1)), hd = hd0 + ((px >> p.lw) & (p.Ht - 1)), n = n0 + (px >> (p.lw + p.lh));
        valid[i] = n < n_end && hd < p.Hd && wd < p.Wd;
        float (&v)[4] = val[i];
#pragma unroll
        for (int j = 0; j < 4; ++j) v[j] = LANES ? lanes_sum(acc[i][j], part[i][j]) : (j & 1 ? acc[i][j >> 1].y : acc[i][j >> 1].x);
        if (!valid[i] || co >= p.Co) continue;
        const size_t o = (((size_t)n * p.Ho + (hd * p.os + p.cls_oph[cls])) * p.Wo + (wd * p.os + p.cls_opw[cls])) * p.Co + co;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            if (bias && co + j < p.Co) v[j] += bias[(size_t)grp * p.b_group + co + j];
            if (p.epi & EPI_RELU) v[j] = fmaxf(v[j], 0.f);
        }
        if (p.epi & EPI_OUT_F32) {
#pragma unroll
            for (int j = 0; j < 4; ++j) if (co + j < p.Co) ((float*)y)[o + j] = v[j];
        } else if ((p.Co & 3) == 0) {
            if (p.epi & EPI_ACCUM) { const float4 old = ld4(y + o); v[0] += old.x; v[1] += old.y; v[2] += old.z; v[3] += old.w; }
            st4(y + o, make_float4(v[0], v[1], v[2], v[3]));
        } else {
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (co + j < p.Co) { if (p.epi & EPI_ACCUM) v[j] += to_f(y[o + j]); put(y + o + j, v[j]); }
        }
    }
    if (!stat) return;
    // batch-norm statistics of the tile, from the values as stored: per channel the mean over its pixels and the sum of squared
    // deviations from that mean (no cancellation, whatever the mean)
    const int cnt = min(p.Wt, p.Wd - wd0) * min(p.Ht, p.Hd - hd0) * min(p.Nt, n_end - n0);
    float s[4], m[4];
    float* const red = fsm + row * 16 + 4 * cg;
    float4* const carry = (float4*)(fsm + 64) + row * 32 + lane;
    // sums over the tile's pixels in a fixed order, the same for every PP: 4 pixels of a lane one after the other (over the warps that share
    // them), 8 lanes, 4 rows of 32 pixels.  add(s) adds this thread's pixels.
    auto over_pixels = [&](auto add) {
#pragma unroll
        for (int j = 0; j < 4; ++j) s[j] = 0.f;
#pragma unroll
        for (int k = 0; k < PARTS; ++k) {
            if (part_of == k) {
                if (k > 0) { const float4 c4 = *carry; s[0] = c4.x; s[1] = c4.y; s[2] = c4.z; s[3] = c4.w; }
                add();
                if (k + 1 < PARTS) *carry = make_float4(s[0], s[1], s[2], s[3]);
            }
            if (k + 1 < PARTS) __syncthreads();
        }
        if (part_of == PARTS - 1) {
#pragma unroll
            for (int j = 0; j < 4; ++j) {
#pragma unroll
                for (int d = 1; d < 8; d <<= 1) s[j] += __shfl_xor_sync(0xffffffffu, s[j], d);
                if (g == 0) red[j] = s[j];
            }
        }
        __syncthreads();
#pragma unroll
        for (int j = 0; j < 4; ++j) s[j] = (fsm[4 * cg + j] + fsm[16 + 4 * cg + j]) + (fsm[32 + 4 * cg + j] + fsm[48 + 4 * cg + j]);
        __syncthreads();
    };
    over_pixels([&] {
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int i = 0; i < PP; ++i) { val[i][j] = stored<T>(val[i][j]); if (valid[i]) s[j] += val[i][j]; }
    });
#pragma unroll
    for (int j = 0; j < 4; ++j) m[j] = s[j] / (float)cnt;
    over_pixels([&] {
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int i = 0; i < PP; ++i) if (valid[i]) { const float d = val[i][j] - m[j]; s[j] = fmaf(d, d, s[j]); }
    });
    if (warp == 0 && g == 0) {
        const int tiles = gridDim.x, groups = gridDim.z;
        const size_t rec = (size_t)grp * tiles + blockIdx.x;
#pragma unroll
        for (int j = 0; j < 4; ++j) if (co + j < p.Co) *(float2*)(stat + (rec * p.Co + co + j) * 2) = make_float2(m[j], s[j]);
        if (blockIdx.y == 0 && cg == 0) stat[(size_t)groups * tiles * p.Co * 2 + rec] = (float)cnt;
    }
}

// grid = (splits, c_out blocks x c_in blocks, groups).  Thread = 4 c_out x 8 c_in of one tap, for one slice of every tile's
// pixels.  dy is kept twice in shared memory ((d, d) pairs: the multiplier of a packed FMA), x as in fc_kernel.  While a tile is used, the
// next one's x is on its way into the other buffer (fp32: cp.async) and its dy into registers.
// Compensated sum: a chain of CHAIN products starts at what the running sum lost at its last addition, so that the compensation
// costs neither registers nor an instruction of its own.  Chains of 32 (16 take 3 to 4 % of a ResNet-20 step) where a group has FW_LONG or more pixels: the
// sums over slices and splits in double leave the error below that of the implicit GEMM this replaced, which added its splits in fp32 (rms
// error against double sums, normal data, of the result's rms: 12288 pixels of 8x8, 64 -> 64 channels 1.06e-7 against 1.50e-7, of 32x32, 16 -> 16
// 1.08e-7 against 1.47e-7).  Shorter sums were better there (4096 pixels: 1.12e-7 against 1.13e-7 with chains of 32; 768: 8.5e-8, 1.06e-7) and get chains of 16
// (768: 8.5e-8).  bf16 storage: chains of 32, sums over slices and splits in fp32 (its inputs are rounded to 4e-3).
// part: [group][block][split][16 c_out][taps][8 * G c_in]
template <typename T> struct FwSum { typedef float type; };
template <> struct FwSum<float> { typedef double type; };
constexpr long FW_LONG = 6144;
constexpr int FW_DYV = 4;                                    // float4s of dy per thread and tile: 128 pixels x 4 / 160 threads
template <typename T, int XS, int G, int RUN, int CHAIN>
__global__ void __launch_bounds__(FW_THREADS, 3) fw_kernel(const T* __restrict__ x, const T* __restrict__ dy, float* __restrict__ part_out,
                                                           const __grid_constant__ FwParams p) {
    extern __shared__ __align__(16) float fsm[];
    float* const ds_ = fsm + 2 * p.x_floats;                 // [pixel][16][2]
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int grp = blockIdx.z, cob = blockIdx.y / p.ci_blocks, cib = blockIdx.y % p.ci_blocks;
    const int co0 = cob * FW_CO, ci0 = cib * FW_CI;
    const int per_slice = p.ntaps * G * 4;
    const int slice = tid / per_slice, rest = tid - slice * per_slice;
    const int cog = rest & 3, ng = rest >> 2, tap = ng / G, half = ng - tap * G;
    const bool active = slice < p.nslices;
    const int npix = p.Wt * p.Ht * p.Nt;
    float2 acc[4][4], part[4][4];                            // [c_out][c_in pair]
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) { acc[i][j] = make_float2(0.f, 0.f); part[i][j] = make_float2(0.f, 0.f); }
    const int xoff = (active ? p.toff[tap] : 0) + half * 8;
    const float* const dt = ds_ + cog * 8;
    const int per = (p.tiles + p.splits - 1) / p.splits;
    const int tile0 = blockIdx.x * per, tile_end = min(p.tiles, tile0 + per), n_end = (grp + 1) * p.ngroup;
    float4 dv[FW_DYV];
    auto fetch = [&](int tl, int buf) {
        const int tw = tl % p.tiles_w; tl /= p.tiles_w;
        const int th = tl % p.tiles_h, tn = tl / p.tiles_h;
        const int n0 = grp * p.ngroup + tn * p.Nt, ho0 = th * p.Ht, wo0 = tw * p.Wt;
        load_region<T>((p.C & 3) == 0, x, fsm + buf * p.x_floats, n0, n_end, p.Nt, ho0 * p.hstep - p.pad, wo0 * p.hstep - p.pad, p.RH, p.RW, p.step, p.H, p.W, p.C,
                       ci0, G == 2 ? 4 : 2, warp, FW_THREADS / 32, lane);
        cp_commit();
#pragma unroll
        for (int u = 0; u < FW_DYV; ++u) {
            const int i = tid + u * FW_THREADS;
            dv[u] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (i >= npix * 4) continue;
            const int px = i >> 2, q = i & 3;
            const int w = wo0 + (px & (p.Wt - 1)), h = ho0 + ((px >> p.lw) & (p.Ht - 1)), n = n0 + (px >> (p.lw + p.lh));
            const int c = co0 + 4 * q;
            if (n >= n_end || h >= p.Ho || w >= p.Wo || c >= p.Co) continue;
            const T* s = dy + (((size_t)n * p.Ho + h) * p.Wo + w) * p.Co + c;
            if ((p.Co & 3) == 0) dv[u] = ld4(s);
            else { dv[u].x = to_f(s[0]); dv[u].y = c + 1 < p.Co ? to_f(s[1]) : 0.f; dv[u].z = c + 2 < p.Co ? to_f(s[2]) : 0.f; dv[u].w = c + 3 < p.Co ? to_f(s[3]) : 0.f; }
        }
    };
    if (tile0 < tile_end) fetch(tile0, 0);
    for (int tile = tile0; tile < tile_end; ++tile) {
        const int buf = (tile - tile0) & 1;
#pragma unroll
        for (int u = 0; u < FW_DYV; ++u) {
            const int i = tid + u * FW_THREADS;
            if (i >= npix * 4) continue;
            float* d = ds_ + (i >> 2) * 32 + (i & 3) * 8;
            *(float4*)d = make_float4(dv[u].x, dv[u].x, dv[u].y, dv[u].y);
            *(float4*)(d + 4) = make_float4(dv[u].z, dv[u].z, dv[u].w, dv[u].w);
        }
        cp_wait<0>();
        __syncthreads();
        if (tile + 1 < tile_end) fetch(tile + 1, buf ^ 1);
        if (active) {
            const float* const xt = fsm + buf * p.x_floats + xoff;
#pragma unroll 1
            for (int r = 0; r < p.pps; r += CHAIN) {
#pragma unroll
                for (int rr = 0; rr < CHAIN; rr += RUN) {
                    const int px = slice * p.pps + r + rr;
                    if (rr > 0 && r + rr >= p.pps) break;
                    const int pw = px & (p.Wt - 1), ph = (px >> p.lw) & (p.Ht - 1), pn = px >> (p.lw + p.lh);
                    const float* xp = xt + ((pn * p.RH + ph * XS) * p.RW + pw * XS) * PITCH;
                    const float* dp = dt + px * 32;
#pragma unroll
                    for (int k = 0; k < RUN; ++k) {
                        const float4 xa = *(const float4*)(xp + k * XS * PITCH), xc = *(const float4*)(xp + k * XS * PITCH + 4);
                        const float4 d0 = *(const float4*)(dp + k * 32), d1 = *(const float4*)(dp + k * 32 + 4);
                        const float2 xv[4] = {make_float2(xa.x, xa.y), make_float2(xa.z, xa.w), make_float2(xc.x, xc.y), make_float2(xc.z, xc.w)};
                        const float2 d2[4] = {make_float2(d0.x, d0.y), make_float2(d0.z, d0.w), make_float2(d1.x, d1.y), make_float2(d1.z, d1.w)};
#pragma unroll
                        for (int i = 0; i < 4; ++i)
#pragma unroll
                            for (int j = 0; j < 4; ++j) part[i][j] = __ffma2_rn(d2[i], xv[j], part[i][j]);
                    }
                }
#pragma unroll
                for (int i = 0; i < 4; ++i)
#pragma unroll
                    for (int j = 0; j < 4; ++j) kahan(acc[i][j], part[i][j]);
            }
        }
        __syncthreads();                                     // dy and this x buffer are consumed
    }
    // the slices' sums in slice order, then the CTA's partial matrix
    const int nout = FW_CO * p.ntaps * 8 * G;
    float* const red = fsm;                                  // [slice][16][taps][8 G]
    if (active) {
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j)
                *(float2*)(red + (size_t)slice * nout + ((cog * 4 + i) * p.ntaps + tap) * (8 * G) + half * 8 + 2 * j) = acc[i][j];
    }
    __syncthreads();
    float* out = part_out + (((size_t)grp * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x) * nout;
    for (int i = tid; i < nout; i += FW_THREADS) {
        typename FwSum<T>::type s = 0;
        for (int k = 0; k < p.nslices; ++k) s += red[(size_t)k * nout + i];
        out[i] = (float)s;
    }
}

// dW[c_out][tap][c_in] = sum over the splits (at most 592): 8 lanes per element take every 8th split, eight loads in flight each, then a
// fixed tree.  S: what they are added in.
template <typename S>
__global__ void __launch_bounds__(256) fw_reduce_kernel(const float* __restrict__ part, float* __restrict__ dw, int splits, int nout, int ntaps, int cw, int ci_blocks,
                                                        int C, int Co, size_t w_group, bool accum) {
    __shared__ S sh[8][33];
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    const int e = blockIdx.x * 32 + tx, blk = blockIdx.y, grp = blockIdx.z;
    const float* src = part + ((size_t)grp * gridDim.y + blk) * splits * nout + e;
    S s = 0;
    if (e < nout) {
        int k = ty;
        for (; k + 56 < splits; k += 64) {
            float v[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) v[u] = src[(size_t)(k + 8 * u) * nout];
#pragma unroll
            for (int u = 0; u < 8; ++u) s += v[u];
        }
        for (; k < splits; k += 8) s += src[(size_t)k * nout];
    }
    sh[ty][tx] = s;
    __syncthreads();
    if (ty != 0 || e >= nout) return;
    s = ((sh[0][tx] + sh[1][tx]) + (sh[2][tx] + sh[3][tx])) + ((sh[4][tx] + sh[5][tx]) + (sh[6][tx] + sh[7][tx]));
    const int co = (blk / ci_blocks) * FW_CO + e / (ntaps * cw), tap = e / cw % ntaps, ci = (blk % ci_blocks) * FW_CI + e % cw;
    if (co >= Co || ci >= C) return;
    float* d = dw + (size_t)grp * w_group + ((size_t)co * ntaps + tap) * C + ci;
    *d = accum ? *d + (float)s : (float)s;
}

}  // namespace

static int ilog2(int v) { int l = 0; while ((1 << l) < v) ++l; return l; }

// The largest power of two <= cap that wastes least when it tiles `n`.
static int best_tile(int n, int cap) {
    int best = 1; long best_cover = n;
    for (int t = 2; t <= cap; t *= 2) {
        const long cover = (long)((n + t - 1) / t) * t;
        if (t / 2 >= n) break;
        if (cover <= best_cover + best_cover / 8) { best = t; if (cover < best_cover) best_cover = cover; }   // a wider tile may waste an eighth
    }
    return best;
}

namespace { struct Tile { int Wt, Ht, Nt; }; }
// Tile of `pixels` pixels for n images of H x W per group; a tile needs R x R windows, `step` apart, of what it reads.
// First choice: the exact cover of an image, as best_tile has it.  Images that no power of two covers (7x7, 5x7) leave it tiles of single pixels from
// 128 images: half empty for the images of one worker, nine pixels read for one.  Where another tile costs less than three quarters
// (pixels computed, used or not, plus a quarter per pixel read), that one (step times of 24-channel networks on 4 workers x 48: 7x7 fp32 590 us
// with the exact cover, 290 so; 489 with the implicit GEMM that these kernels replaced; 5x7 511, 291, 483).
static Tile pick_tile(int H, int W, int n, int pixels, int R, int step) {
    auto cost = [&](int wt, int ht) {
        const int nt = pixels / (wt * ht);
        const double tiles = (double)((W + wt - 1) / wt) * ((H + ht - 1) / ht) * ((n + nt - 1) / nt);
        return tiles * (pixels + 0.25 * nt * ((wt - 1) * step + R) * ((ht - 1) * step + R));
    };
    Tile t;
    t.Wt = best_tile(W, pixels < 32 ? pixels : 32);
    t.Ht = best_tile(H, pixels / t.Wt);
    const auto pow2 = [](int v) { return (v & (v - 1)) == 0; };
    double best = pow2(H) && pow2(W) ? 0.0 : 0.75 * cost(t.Wt, t.Ht);
    for (int wt = pixels < 32 ? pixels : 32; wt >= 1; wt /= 2)
        for (int ht = pixels / wt; ht >= 1; ht /= 2)
            if (cost(wt, ht) < best) { best = cost(wt, ht); t.Wt = wt; t.Ht = ht; }
    t.Nt = pixels / (t.Wt * t.Ht);
    return t;
}

// Geometry of a forward (back == 0) or input-gradient launch over `groups` groups of g.N / groups images; false: not covered.
bool plan_fc(const ConvGeom& g, int groups, bool back, FcParams& p) {
    if ((g.H * g.W == 1 && g.R == 1) || (g.R != 3 && g.R != 1) || (g.stride != 1 && g.stride != 2) || g.N % groups) return false;
    p = FcParams{};
    p.taps = g.R * g.R; p.back = back; p.ngroup = g.N / groups;
    p.w_group = 0; p.b_group = 0;
    int dh[9], dw[9];
    if (!back) {
        p.H = g.H; p.W = g.W; p.C = g.C; p.Ho = g.Ho; p.Wo = g.Wo; p.Co = g.Co; p.Hd = g.Ho; p.Wd = g.Wo; p.os = 1; p.xs = g.stride;
        p.ncls = 1; p.cls_tap0[0] = 0; p.cls_tap0[1] = p.taps;
        for (int t = 0; t < p.taps; ++t) { dh[t] = t / g.R - g.pad; dw[t] = t % g.R - g.pad; p.wtap[t] = t; }
    } else {
        // dx[h][w] = sum over taps of dy[(h + pad - r) / stride][(w + pad - s) / stride] . W[:][r][s][:]; a stride-2 layer by output parity
        p.H = g.Ho; p.W = g.Wo; p.C = g.Co; p.Ho = g.H; p.Wo = g.W; p.Co = g.C; p.os = g.stride; p.xs = 1;
        p.Hd = (g.H + g.stride - 1) / g.stride; p.Wd = (g.W + g.stride - 1) / g.stride;
        if (g.stride == 2 && ((g.H | g.W) & 1)) return false;
        int n = 0;
        for (int ph = 0; ph < g.stride; ++ph) for (int pw = 0; pw < g.stride; ++pw) {
            p.cls_oph[p.ncls] = ph; p.cls_opw[p.ncls] = pw; p.cls_tap0[p.ncls] = n;
            for (int r = 0; r < g.R; ++r) for (int s = 0; s < g.R; ++s) {
                const int a = ph + g.pad - r, b = pw + g.pad - s;
                if (a % g.stride || b % g.stride) continue;
                dh[n] = a / g.stride; dw[n] = b / g.stride; p.wtap[n] = r * g.R + s; ++n;
            }
            p.cls_tap0[++p.ncls] = n;
        }
    }
    const Tile t = pick_tile(p.Hd, p.Wd, p.ngroup, FC_PIX, g.R, p.xs);
    p.Wt = t.Wt; p.Ht = t.Ht; p.Nt = t.Nt; p.lw = ilog2(t.Wt); p.lh = ilog2(t.Ht);
    p.tiles_w = (p.Wd + t.Wt - 1) / t.Wt; p.tiles_h = (p.Hd + t.Ht - 1) / t.Ht;
    int maxt = 0;
    for (int c = 0; c < p.ncls; ++c) {
        const int a = p.cls_tap0[c], b = p.cls_tap0[c + 1];
        int h0 = 0, h1 = 0, w0 = 0, w1 = 0;
        for (int i = a; i < b; ++i) {
            if (i == a || dh[i] < h0) h0 = dh[i];
            if (i == a || dh[i] > h1) h1 = dh[i];
            if (i == a || dw[i] < w0) w0 = dw[i];
            if (i == a || dw[i] > w1) w1 = dw[i];
        }
        p.cls_h0[c] = h0; p.cls_w0[c] = w0;
        p.cls_rh[c] = (t.Ht - 1) * p.xs + (h1 - h0) + 1; p.cls_rw[c] = (t.Wt - 1) * p.xs + (w1 - w0) + 1;
        for (int i = a; i < b; ++i) p.toff[i] = ((dh[i] - h0) * p.cls_rw[c] + (dw[i] - w0)) * PITCH;
        const int f = t.Nt * p.cls_rh[c] * p.cls_rw[c] * PITCH;
        if (f > p.x_floats) p.x_floats = f;
        if (b - a > maxt) maxt = b - a;
    }
    p.w_floats = maxt * 16 * PITCH;
    const size_t one = (size_t)(p.x_floats + p.w_floats) * sizeof(float);
    // two buffers as long as four CTAs (the register limit) or at least two fit on an SM
    p.buffers = p.C > FC_KC && 2 * one <= 110 * 1024 ? 2 : 1;
    return one <= FC_SMEM_MAX;
}

namespace {

template <typename T, int NQ, bool VEC, int PP>
void launch_fc_pp(const void* x, const void* w, const float* bias, void* y, float* stat, const FcParams& p, int groups, cudaStream_t s) {
    const size_t smem = (size_t)p.buffers * (p.x_floats + p.w_floats) * sizeof(float);
    static OncePerDevice once;
    allow_smem(once, (const void*)fc_kernel<T, NQ, VEC, PP>, (int)FC_SMEM_MAX);
    const int tiles = p.tiles_w * p.tiles_h * ((p.ngroup + p.Nt - 1) / p.Nt);
    klaunch(fc_kernel<T, NQ, VEC, PP>, dim3(tiles, (p.Co + FC_CO - 1) / FC_CO, groups * p.ncls), 512 / PP, smem, s, (const T*)x, (const T*)w, bias, (T*)y, stat, p);
}
// Two pixels a thread while all CTAs fit at two per SM: such launches leave each scheduler one to three warps of four pixels a thread, which wait for
// shared memory (short scoreboard, ncu: 41 % of the issue slots used at 2.6 warps), and twice the warps pay for half as many FMAs per shared load.
// ResNet-20 fp32, 2 x 7 samples, K = 2: 701 -> 584 us per step, 4 x 9, K = 1: 1364 -> 1080; with every launch that way, 4 x 48 goes from 2.70
// to 2.88 ms.  One pixel a thread below 60 to 148 CTAs gave nothing (584 -> 626, 1075 -> 1125).  Both give the same bits.
template <typename T, int NQ, bool VEC>
void launch_fc(const void* x, const void* w, const float* bias, void* y, float* stat, const FcParams& p, int groups, cudaStream_t s) {
    const long ctas = (long)p.tiles_w * p.tiles_h * ((p.ngroup + p.Nt - 1) / p.Nt) * ((p.Co + FC_CO - 1) / FC_CO) * groups * p.ncls;
    if (ctas <= 2 * 148) launch_fc_pp<T, NQ, VEC, 2>(x, w, bias, y, stat, p, groups, s);
    else launch_fc_pp<T, NQ, VEC, 4>(x, w, bias, y, stat, p, groups, s);
}
template <typename T>
void dispatch_fc(const void* x, const void* w, const float* bias, void* y, float* stat, const FcParams& p, int groups, cudaStream_t s) {
    // 16-byte (fp32) / 8-byte (bf16) pieces of a pixel's channels need a channel count that is a multiple of 4; the weight
    // rows of the backward direction are read element by element
    const bool vec = p.C % 4 == 0;
    if (p.C <= 4) { if (vec) launch_fc<T, 1, true>(x, w, bias, y, stat, p, groups, s); else launch_fc<T, 1, false>(x, w, bias, y, stat, p, groups, s); }
    else { if (vec) launch_fc<T, 4, true>(x, w, bias, y, stat, p, groups, s); else launch_fc<T, 4, false>(x, w, bias, y, stat, p, groups, s); }
}

}  // namespace

// Weight gradient: 128 pixels per tile (64 for 3x3 stride 2, whose input region is four times its output).
bool plan_fw(const ConvGeom& g, int groups, int ctas, FwParams& p, int& G, int& run, size_t& smem) {
    if ((g.H * g.W == 1 && g.R == 1) || (g.R != 3 && g.R != 1) || (g.stride != 1 && g.stride != 2) || g.N % groups) return false;
  for (int pixels = g.R == 3 && g.stride == 2 ? 64 : 128; pixels >= 32; pixels /= 2) {        // smaller tiles where the halo of tiny images outgrows shared memory
    p = FwParams{};
    const Tile t = pick_tile(g.Ho, g.Wo, g.N / groups, pixels, g.R, g.R == 1 ? 1 : g.stride);
    run = t.Wt >= 8 ? 8 : (t.Wt >= 4 ? 4 : 1);
    p.H = g.H; p.W = g.W; p.C = g.C; p.Ho = g.Ho; p.Wo = g.Wo; p.Co = g.Co;
    p.Wt = t.Wt; p.Ht = t.Ht; p.Nt = t.Nt; p.lw = ilog2(t.Wt); p.lh = ilog2(t.Ht);
    p.tiles_w = (g.Wo + t.Wt - 1) / t.Wt; p.tiles_h = (g.Ho + t.Ht - 1) / t.Ht;
    p.ngroup = g.N / groups;
    p.tiles = p.tiles_w * p.tiles_h * ((p.ngroup + t.Nt - 1) / t.Nt);
    p.pad = g.pad; p.hstep = g.stride; p.ntaps = g.R * g.R;
    p.step = g.R == 1 ? g.stride : 1;
    const int xs = g.R == 1 ? 1 : g.stride;
    p.RH = (t.Ht - 1) * xs + g.R; p.RW = (t.Wt - 1) * xs + g.R;
    for (int i = 0; i < p.ntaps; ++i) p.toff[i] = ((i / g.R) * p.RW + i % g.R) * PITCH;
    G = g.C <= 8 ? 1 : 2;
    const int npix = t.Wt * t.Ht * t.Nt, per_slice = p.ntaps * G * 4;
    p.nslices = 1;
    while (p.nslices * 2 * per_slice <= FW_THREADS && npix / (p.nslices * 2) >= run) p.nslices *= 2;
    p.pps = npix / p.nslices;
    p.ci_blocks = (g.C + FW_CI - 1) / FW_CI;
    const int blocks = p.ci_blocks * ((g.Co + FW_CO - 1) / FW_CO) * groups;
    // once around the device, each CTA with at least one tile
    int want = ctas / blocks;
    if (want > p.tiles) want = p.tiles;
    if (want < 1) want = 1;
    const int per = (p.tiles + want - 1) / want;
    p.splits = (p.tiles + per - 1) / per;
    p.x_floats = t.Nt * p.RH * p.RW * PITCH;
    smem = ((size_t)2 * p.x_floats + (size_t)npix * 32) * sizeof(float);
    const size_t red = (size_t)p.nslices * FW_CO * p.ntaps * 8 * G * sizeof(float);
    if (red > smem) smem = red;
    if (smem <= FC_SMEM_MAX) return true;
  }
    return false;
}
namespace {

template <typename T, int XS, int G, int RUN, int CHAIN>
void launch_fw_chain(const void* x, const void* dy, float* ws, const FwParams& p, int groups, size_t smem, cudaStream_t s) {
    static OncePerDevice once;
    allow_smem(once, (const void*)fw_kernel<T, XS, G, RUN, CHAIN>, (int)FC_SMEM_MAX);
    klaunch(fw_kernel<T, XS, G, RUN, CHAIN>, dim3(p.splits, p.ci_blocks * ((p.Co + FW_CO - 1) / FW_CO), groups), FW_THREADS, smem, s, (const T*)x, (const T*)dy, ws, p);
}
template <typename T, int XS, int G, int RUN>
void launch_fw(const void* x, const void* dy, float* ws, const FwParams& p, int groups, size_t smem, cudaStream_t s) {
    if (sizeof(T) == 4 && (long)p.ngroup * p.Ho * p.Wo < FW_LONG) launch_fw_chain<T, XS, G, RUN, 16>(x, dy, ws, p, groups, smem, s);
    else launch_fw_chain<T, XS, G, RUN, 32>(x, dy, ws, p, groups, smem, s);
}
template <typename T, int XS, int G>
void dispatch_fw_run(const void* x, const void* dy, float* ws, const FwParams& p, int run, int groups, size_t smem, cudaStream_t s) {
    if (run == 8) launch_fw<T, XS, G, 8>(x, dy, ws, p, groups, smem, s);
    else if (run == 4) launch_fw<T, XS, G, 4>(x, dy, ws, p, groups, smem, s);
    else launch_fw<T, XS, G, 1>(x, dy, ws, p, groups, smem, s);
}
template <typename T>
void dispatch_fw(const void* x, const void* dy, float* ws, const FwParams& p, int xs, int G, int run, int groups, size_t smem, cudaStream_t s) {
    if (xs == 1) { if (G == 1) dispatch_fw_run<T, 1, 1>(x, dy, ws, p, run, groups, smem, s); else dispatch_fw_run<T, 1, 2>(x, dy, ws, p, run, groups, smem, s); }
    else { if (G == 1) dispatch_fw_run<T, 2, 1>(x, dy, ws, p, run, groups, smem, s); else dispatch_fw_run<T, 2, 2>(x, dy, ws, p, run, groups, smem, s); }
}

}  // namespace

bool fconv_supported(const ConvGeom& g) {
    FcParams p; FwParams q; int G, run; size_t smem;
    return plan_fc(g, 1, false, p) && plan_fc(g, 1, true, p) && plan_fw(g, 1, FW_CTAS, q, G, run, smem);
}
bool fconv_forward(int dt, const void* x, const void* w, const float* bias, void* y, const ConvGeom& g, int epi, int groups, size_t w_group, size_t b_group,
                   float* stat, const Packed& pk, cudaStream_t s) {
    FcParams p;
    if (!plan_fc(g, groups, false, p)) return false;
    p.epi = epi; p.w_group = w_group; p.b_group = b_group;
    if (pk.data && mconv_forward(dt, x, w, pk, bias, y, stat, g, epi, groups, w_group, b_group, s)) return true;
    Scope sc(KC_FMA_FWD, conv_flops(g), conv_bytes(dt, g, false), s);
    if (dt) dispatch_fc<bf16>(x, w, bias, y, stat, p, groups, s); else dispatch_fc<float>(x, w, bias, y, stat, p, groups, s);
    return true;
}
bool fconv_dgrad(int dt, const void* dy, const void* w, void* dx, const ConvGeom& g, int epi, int groups, size_t w_group, const Packed& pk, cudaStream_t s) {
    FcParams p;
    if (!plan_fc(g, groups, true, p)) return false;
    p.epi = epi; p.w_group = w_group;
    if (pk.data && mconv_dgrad(dt, dy, w, pk, dx, g, epi, groups, w_group, s)) return true;
    Scope sc(KC_FMA_DGRAD, conv_flops(g), conv_bytes(dt, g, false), s);
    if (dt) dispatch_fc<bf16>(dy, w, nullptr, dx, nullptr, p, groups, s); else dispatch_fc<float>(dy, w, nullptr, dx, nullptr, p, groups, s);
    return true;
}
int fconv_stat_tiles(const ConvGeom& g, int groups) {
    FcParams p;
    return plan_fc(g, groups, false, p) ? p.tiles_w * p.tiles_h * ((p.ngroup + p.Nt - 1) / p.Nt) : 0;
}
size_t fconv_wgrad_workspace_elems(const ConvGeom& g, int groups) {
    FwParams p; int G, run; size_t smem;
    if (!plan_fw(g, groups, FW_CTAS, p, G, run, smem)) return 0;
    // a window of the batch may be cut into other tiles, but never uses more splits than fill the device
    const int blocks = p.ci_blocks * ((g.Co + FW_CO - 1) / FW_CO) * groups;
    return (size_t)blocks * (MW_CTAS > blocks ? MW_CTAS / blocks : 1) * FW_CO * p.ntaps * 8 * G;
}
bool fconv_wgrad(int dt, const void* x, const void* dy, float* dw, float* ws, const ConvGeom& g, int groups, size_t w_group, bool accum, bool tensor, cudaStream_t s) {
    FwParams p; int G, run; size_t smem;
    if (!plan_fw(g, groups, FW_CTAS, p, G, run, smem)) return false;
    const int xs = g.R == 1 ? 1 : g.stride, blocks = p.ci_blocks * ((g.Co + FW_CO - 1) / FW_CO), nout = FW_CO * p.ntaps * 8 * G;
    const int splits = tensor ? mconv_wgrad(dt, x, dy, ws, g, groups, s) : 0;
    if (splits) p.splits = splits;
    else {
        Scope sc(KC_FMA_WGRAD, conv_flops(g), conv_bytes(dt, g, true), s);
        if (dt) dispatch_fw<bf16>(x, dy, ws, p, xs, G, run, groups, smem, s); else dispatch_fw<float>(x, dy, ws, p, xs, G, run, groups, smem, s);
    }
    Scope sc(KC_SPLITK, 0.0, 4.0 * groups * (p.splits + 1) * blocks * nout, s);
    const dim3 rgrid((nout + 31) / 32, blocks, groups);
    // bf16: the packed-FMA kernel's partial matrices in fp32, mconv.cu's in double (in fp32 the error was up to 1.1 times that of the former); one is only copied
    if (dt && splits <= 1) klaunch(fw_reduce_kernel<FwSum<bf16>::type>, rgrid, 256, 0, s, ws, dw, p.splits, nout, p.ntaps, 8 * G, p.ci_blocks, g.C, g.Co, w_group, accum);
    else klaunch(fw_reduce_kernel<FwSum<float>::type>, rgrid, 256, 0, s, ws, dw, p.splits, nout, p.ntaps, 8 * G, p.ci_blocks, g.C, g.Co, w_group, accum);
    return true;
}

}  // namespace fdg
