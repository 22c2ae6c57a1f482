// Convolutions (3x3 and 1x1, stride 1 and 2) of channel counts that are multiples of 16 on the warp-level tensor-core instruction: the fp32
// path, and with bf16 storage the layers whose channels are no multiple of 64 (the paper's ResNet-20 has 16, 32 and 64).
//
//   mc_kernel : forward and input gradient.  A CTA computes 128 pixels x 16 or 32 output channels; the input region of its pixels (halo
//               included) is fetched once per 16-channel chunk and every filter tap reads it from shared memory, shifted.
//   mw_kernel : weight gradient.  A CTA keeps a 16 c_out x (taps x 16 c_in) tile of dW in registers over the pixels of its split.
//   mc_pack_kernel : a layer's weights in the order in which the lanes of a warp hold them (one launch per pass for all layers of a module).
//
// Arithmetic with fp32 storage: a value is the sum of three bf16 values, x = hi + mid + lo (8 bits each or, see below, 6 in hi; rounded to nearest, so that nothing is left), and
// a product the sum of the six that matter: lo hi + mid mid + hi lo + mid hi + hi mid + hi hi (the rest is 2e-8 of it, of either sign; 6e-8, and one-sided, with parts by
// truncation).  Every product is exact; an mma adds 16 of them to its running sum and truncates to 24 bits of the largest term: 2.5e-8 of the
// result's rms for 16 fresh products of 16 bits, 1.3e-7 for nine such steps in a chain, 5.3e-7 for 36, 1e-7 as soon as a 24-bit running sum of
// like size is among the terms.  So hi hi starts from zero in every step and goes into an fp32 sum on the CUDA cores, two taps of it into a
// compensated (Kahan) sum, in a weight gradient of fp32 storage every step (four CTAs per SM have no registers for both); the other five, 2^-6 of
// it at the most, run on in one accumulator per chunk.  What truncation takes away has the sign of the sum: 1.7e-8 of a sum of products of one sign with 16-bit
// products.  One operand's hi (the weights', where the pack does it once; dy's in a weight gradient) therefore has 6 bits, as few as three parts allow: 14-bit
// products, 6e-9.
// Error against double sums, of the result's rms (packed-FMA kernels of fconv.cu beside it), 3x3: normal data, forward and input gradient 4.1e-8 to 4.8e-8
// (7.6e-8), weight gradient 4.5e-8 (8e-8 to 1.1e-7); ReLU'd x, weights and dy with a mean of half their deviation 2.4e-8 to 3.7e-8 (2.5e-8 to
// 4.7e-8), weight gradient 2.6e-8 to 3.0e-8 (2.8e-8 to 3.8e-8); every product of one sign 2.5e-8 to 3.5e-8 (2.5e-8 to 3.9e-8; 2 % more than there from 256
// channels on), weight gradient 2.0e-8 (1.9e-8; 1x1 6 % more).  With 8 bits and nine taps a run the last two of forward and input gradient were up to
// 1.6 and 1.75 times those of the packed-FMA kernels (22.7 us for what takes 25 now).  Two fp16 parts and three products were off by 9.4e-8:
// 22-bit products lose more where the terms are aligned.  bf16 storage: one exact product a step, weight gradients flushed every MW_RUN steps and the splits
// added in double: 1.00 times the packed-FMA kernels' errors at the most, 0.8 on average (1.19 with a flush per tile).  Forward and input gradient keep to
// one flush per chunk there: 6.5e-8 before the result is rounded to bf16, by 1.7e-3 (4.4e-8; one every two taps gives 4.6e-8 for 4.5 % of a step).
//
// Time, 192 images, launch included (packed FMA beside it): fp32 32x32 16 -> 16 forward 25 us (38), weight gradient with its reduction 38 (54); 16x16 32 -> 32 25
// (40), 36 (53); 8x8 64 -> 64 29 (41), 39 (57).  What bounds them: a third to 40 % of the mma.sync rate (980 multiply-adds per clock and SM, six per
// product), the rest is latency of one warp's chain (fixed-latency waits, ncu) and the splitting, which every block of 16 or 32 output channels repeats.
#include "fconv.h"
#include "launch.h"

#include <algorithm>

namespace fdg {

namespace {

constexpr int MC_THREADS = 128;
constexpr int W_HI = 6, DY_HI = 6;       // bits of hi in the weights and, in a weight gradient, in dy
constexpr int MW_RUN = 4;                // steps of a weight gradient that are added before they go into the compensated sum (bf16 storage)

template <typename T> constexpr bool SPLIT = sizeof(T) == 4;
template <typename T> constexpr int PARTS = SPLIT<T> ? 3 : 1;             // bf16 values per value
template <typename T> constexpr int PACK16 = 32 * PARTS<T>;               // 16-byte words of the packed weights per (16 x 16 block, tap)

__device__ __forceinline__ void ldsm4(uint32_t (&r)[4], uint32_t a) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];" : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(a) : "memory");
}
__device__ __forceinline__ void ldsm4t(uint32_t (&r)[4], uint32_t a) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];" : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(a) : "memory");
}
__device__ __forceinline__ void ldsm2t(uint32_t (&r)[2], uint32_t a) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x2.trans.shared.b16 {%0,%1}, [%2];" : "=r"(r[0]), "=r"(r[1]) : "r"(a) : "memory");
}
// d = a b (+ d): 16 x 16 times 16 x 8
__device__ __forceinline__ void mma(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1, bool add) {
    const float c0 = add ? d[0] : 0.f, c1 = add ? d[1] : 0.f, c2 = add ? d[2] : 0.f, c3 = add ? d[3] : 0.f;
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%11,%12,%13};"
        : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3]) : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1), "f"(c0), "f"(c1), "f"(c2), "f"(c3));
}
// product `k` of a step, smallest first: parts of a and of b (0 hi, 1 mid, 2 lo)
template <typename T> constexpr int PRODUCTS = SPLIT<T> ? 6 : 1;
template <typename T> __host__ __device__ constexpr int part_a(int k) { return !SPLIT<T> ? 0 : k == 0 ? 2 : k == 1 || k == 3 ? 1 : 0; }
template <typename T> __host__ __device__ constexpr int part_b(int k) { return !SPLIT<T> ? 0 : k == 2 ? 2 : k == 1 || k == 4 ? 1 : 0; }

// Range: before the split a value is multiplied by RANGE = 2^16, so that lo of the smallest normal number, 2^-126, still is a multiple of bf16's smallest, 2^-133
// (the exponents reach as far down as fp32's, the digits 16 places less far); sums carry RANGE^2 until they are stored.  The price is at the other
// end: from 2^111 on (sums: 2^95) parts are infinite, and since a part that overflows leaves NaN in the next one, so is no sum that they enter.  Such outputs are computed
// once more, product by product (direct_*).
constexpr float RANGE = 65536.f, UNRANGE2 = 1.f / (65536.f * 65536.f);
// two values' parts.  HI: significant bits of hi, 8 or fewer (at least 6: mid and lo hold 8 each and a sign)
__device__ __forceinline__ uint32_t pair_rn(float a, float b) { const __nv_bfloat162 v = __floats2bfloat162_rn(a, b); return *(const uint32_t*)&v; }
__device__ __forceinline__ float2 pair_value(uint32_t v) { return make_float2(__uint_as_float(v << 16), __uint_as_float(v & 0xffff0000u)); }
template <int HI> __device__ __forceinline__ void split2(float a, float b, uint32_t& hi, uint32_t& mid, uint32_t& lo) {
    const float2 minus = make_float2(-1.f, -1.f);
    if (HI == 8) hi = pair_rn(a, b);
    else {
        constexpr uint32_t half = 1u << (23 - HI), keep = (0xffffu << (8 - HI)) & 0xffffu;
        hi = __byte_perm(__float_as_uint(a) + half, __float_as_uint(b) + half, 0x7632) & (keep << 16 | keep);
    }
    const float2 r = __ffma2_rn(pair_value(hi), minus, make_float2(a, b));
    mid = pair_rn(r.x, r.y);
    const float2 l = __ffma2_rn(pair_value(mid), minus, r);
    lo = pair_rn(l.x, l.y);
}

// fp32 values of a pixel's 16 channels as they arrive: quad q sits at position q ^ (pixel / 2 % 4), so that eight pixels' quads q lie in different banks
__device__ __forceinline__ int raw_at(int pix, int q) { return pix * 16 + ((q ^ ((pix >> 1) & 3)) << 2); }

// A region (see load_region in fconv.cu) of 16 channels from c0 on.  fp32: into raw.  bf16: into planes[half][pixel][8], halves `xp` pixels apart.
template <typename T>
__device__ __forceinline__ void fetch_region(const T* __restrict__ x, char* dst, int xp, int n0, int n_end, int nimg, int h0, int w0, int RH, int RW, int step,
                                             int H, int W, int C, int c0, int warp, int nwarps, int lane) {
    constexpr int Q = SPLIT<T> ? 4 : 2;              // 16-byte pieces of a pixel
    int ni = 0, rh = warp;
    while (rh >= RH) { rh -= RH; ++ni; }
    while (ni < nimg) {
        const int n = n0 + ni, h = h0 + rh * step;
        const bool row_ok = n < n_end && h >= 0 && h < H;
        // a lane keeps its piece q and steps over pixels, 8 (fp32) or 16 at a time: the position in dst moves by a constant (raw_at: pixel / 2 % 4 stays)
        constexpr int STEP = 32 / Q;
        const int q = lane % Q, pix = (ni * RH + rh) * RW + lane / Q;
        int w = w0 + lane / Q * step;
        const T* s = x + (((ptrdiff_t)n * H + h) * W + w) * C + c0 + q * (16 / Q);
        uint32_t d = smem_addr(dst) + (uint32_t)(SPLIT<T> ? raw_at(pix, q) * 4 : (q * xp + pix) * 16);
        for (int rw = lane / Q; rw < RW; rw += STEP) {
            const bool in = row_ok && w >= 0 && w < W;
            cp_async16(d, in ? s : x, in);
            w += STEP * step; s += (size_t)STEP * step * C; d += STEP * (SPLIT<T> ? 64 : 16);
        }
        rh += nwarps;
        while (rh >= RH) { rh -= RH; ++ni; }
    }
}
// raw -> planes [hi, mid, lo][half][pixel][8], parts `part_bytes` apart
template <int HI> __device__ __forceinline__ void split_pixels(const float* raw, char* dst, int xp, int part_bytes, int npix, int tid, int nthreads) {
    for (int pix = tid; pix < npix; pix += nthreads)
#pragma unroll
        for (int half = 0; half < 2; ++half) {
            const float4 a = *(const float4*)(raw + raw_at(pix, 2 * half)), b = *(const float4*)(raw + raw_at(pix, 2 * half + 1));
            const float2 range = make_float2(RANGE, RANGE);
            const float2 v[4] = {__fmul2_rn(make_float2(a.x, a.y), range), __fmul2_rn(make_float2(a.z, a.w), range), __fmul2_rn(make_float2(b.x, b.y), range),
                                 __fmul2_rn(make_float2(b.z, b.w), range)};
            uint4 h, m, l;
            split2<HI>(v[0].x, v[0].y, h.x, m.x, l.x); split2<HI>(v[1].x, v[1].y, h.y, m.y, l.y); split2<HI>(v[2].x, v[2].y, h.z, m.z, l.z); split2<HI>(v[3].x, v[3].y, h.w, m.w, l.w);
            char* const d = dst + (half * xp + pix) * 16;
            *(uint4*)d = h; *(uint4*)(d + part_bytes) = m; *(uint4*)(d + 2 * part_bytes) = l;
        }
}

// sum += y + lost, compensated; lost: what the sum has lost so far
__device__ __forceinline__ void add_kahan(float2& sum, float2& lost, float2 y) {
    const float2 minus = make_float2(-1.f, -1.f);
    y = __fadd2_rn(y, lost);
    const float2 t = __fadd2_rn(sum, y);
    lost = __ffma2_rn(__ffma2_rn(sum, minus, t), minus, y);          // y - (t - sum)
    sum = t;
}

struct McParams {
    FcParams p;                          // geometry; toff in pixels
    int xp;                              // pixels of the largest class's region
    int wtaps;                           // taps of the largest class
    size_t pack_group;                   // 16-byte words between the groups' packed weights
};
// a compensated sum that overflowed has lost NaN
__device__ __forceinline__ float total(float sum, float lost) { return isinf(sum) ? sum : __fadd_rn(sum, lost); }
// the compensated sums of the packed-FMA kernels end as NaN where they overflow
__device__ __forceinline__ float finite_or_nan(double s) { const float v = (float)s; return isfinite(v) ? v : __int_as_float(0x7fffffff); }

// One output of mc_kernel, product by product; w: this group's weights.
__device__ __noinline__ float direct_output(const float* __restrict__ x, const float* __restrict__ w, const FcParams& p, int cls, int n, int hd, int wd, int co) {
    double s = 0.0;
    for (int t = p.cls_tap0[cls]; t < p.cls_tap0[cls + 1] && isfinite(s); ++t) {
        const int h = hd * p.xs + p.cls_h0[cls] + p.toff[t] / p.cls_rw[cls], wi = wd * p.xs + p.cls_w0[cls] + p.toff[t] % p.cls_rw[cls];
        const bool in = h >= 0 && h < p.H && wi >= 0 && wi < p.W;
        const float* const xs = x + (((size_t)n * p.H + (in ? h : 0)) * p.W + (in ? wi : 0)) * p.C;
        const float* const ws = p.back ? w + (size_t)p.wtap[t] * p.Co + co : w + ((size_t)co * p.taps + p.wtap[t]) * p.C;
        const size_t step = p.back ? (size_t)p.taps * p.Co : 1;
        for (int c = 0; c < p.C; ++c) s += (in ? (double)xs[c] : 0.0) * (double)ws[c * step];
    }
    return finite_or_nan(s);
}
// Of a lane's outputs, in the order of mc_kernel's loops, those that one look says are NaN: the first channel of the middle tap (in the image with stride 1) is no
// finite number in the weights or in x.  With NaN in all weights direct_output for each made a step of ResNet-20 take 18.7 ms (2.6 now, 2.0 without NaN).
template <int NB>
__device__ __noinline__ uint32_t surely_nan(const float* __restrict__ x, const float* __restrict__ w, const FcParams& p, int cls, int n0, int hd0, int wd0, int px0, int n_end, int co0) {
    const int t = (p.cls_tap0[cls] + p.cls_tap0[cls + 1]) / 2, dh = p.cls_h0[cls] + p.toff[t] / p.cls_rw[cls], dw = p.cls_w0[cls] + p.toff[t] % p.cls_rw[cls];
    const float* const ws = p.back ? w + (size_t)p.wtap[t] * p.Co : w + (size_t)p.wtap[t] * p.C;
    const size_t step = p.back ? 1 : (size_t)p.taps * p.C;
    uint32_t nan = 0;
#pragma unroll
    for (int j = 0; j < NB; ++j)
#pragma unroll
        for (int e = 0; e < 2; ++e)
            if (!isfinite(ws[(co0 + 8 * j + e) * step])) nan |= (1u << 2 | 1u | (1u << 2 | 1u) << 4 * NB) << (4 * j + e);
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const int px = px0 + i * 16 + r * 8, n = n0 + (px >> (p.lw + p.lh));
            const int h = (hd0 + ((px >> p.lw) & (p.Ht - 1))) * p.xs + dh, wi = (wd0 + (px & (p.Wt - 1))) * p.xs + dw;
            if (n < n_end && h >= 0 && h < p.H && wi >= 0 && wi < p.W && !isfinite(x[(((size_t)n * p.H + h) * p.W + wi) * p.C])) {
#pragma unroll
                for (int j = 0; j < NB; ++j) nan |= 3u << ((i * NB + j) * 4 + r * 2);
            }
        }
    return nan;
}
// One element of mw_kernel's partial matrix.
__device__ __noinline__ float direct_wgrad(const float* __restrict__ x, const float* __restrict__ dy, const FwParams& p, int grp, int tile0, int tile_end, int co, int tap, int ci) {
    const int R = p.ntaps == 9 ? 3 : 1, n_end = (grp + 1) * p.ngroup;
    double s = 0.0;
    for (int t = tile0; t < tile_end && isfinite(s); ++t) {
        const int tw = t % p.tiles_w, th = t / p.tiles_w % p.tiles_h, tn = t / p.tiles_w / p.tiles_h;
        for (int px = 0; px < p.Wt * p.Ht * p.Nt; ++px) {
            const int wo = tw * p.Wt + (px & (p.Wt - 1)), ho = th * p.Ht + ((px >> p.lw) & (p.Ht - 1)), n = grp * p.ngroup + tn * p.Nt + (px >> (p.lw + p.lh));
            const int h = ho * p.hstep - p.pad + tap / R, w = wo * p.hstep - p.pad + tap % R;
            if (n >= n_end || ho >= p.Ho || wo >= p.Wo) continue;
            const bool in = h >= 0 && h < p.H && w >= 0 && w < p.W;
            if (!isfinite(s)) break;
            s += (in ? (double)x[(((size_t)n * p.H + h) * p.W + w) * p.C + ci] : 0.0) * (double)dy[(((size_t)n * p.Ho + ho) * p.Wo + wo) * p.Co + co];
        }
    }
    return finite_or_nan(s);
}

template <typename T> constexpr int mc_x_bytes(int xp) { return xp * (SPLIT<T> ? 64 + 96 : 2 * 32); }            // fp32: raw + parts; bf16: two buffers
template <typename T, int NB> constexpr int mc_w_bytes(int taps, int chunks) { return (chunks > 1 ? 2 : 1) * taps * (NB / 2) * PACK16<T> * 16; }

// grid = (pixel tiles, blocks of 8 NB output channels, groups x classes); a warp computes 32 pixels x 8 NB channels.
template <typename T, int NB>
__global__ void __launch_bounds__(MC_THREADS, NB == 4 ? SPLIT<T> ? 2 : 3 : 4) mc_kernel(const T* __restrict__ x, const T* __restrict__ w, const uint4* __restrict__ pk,
                                                                        const float* __restrict__ bias, T* __restrict__ y, float* __restrict__ stat, const __grid_constant__ McParams q) {
    constexpr bool S = SPLIT<T>;
    constexpr int NW = MC_THREADS / 32, BLKS = NB / 2, U = PACK16<T>;
    extern __shared__ __align__(16) char msm[];
    const FcParams& p = q.p;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, tq = lane & 3;
    const int cls = blockIdx.z % p.ncls, grp = blockIdx.z / p.ncls;
    int tile = blockIdx.x;
    const int tw = tile % p.tiles_w; tile /= p.tiles_w;
    const int th = tile % p.tiles_h, tn = tile / p.tiles_h;
    const int n_end = (grp + 1) * p.ngroup, n0 = grp * p.ngroup + tn * p.Nt;
    const int hd0 = th * p.Ht, wd0 = tw * p.Wt, co0 = blockIdx.y * (8 * NB);
    const int t0 = p.cls_tap0[cls], nt = p.cls_tap0[cls + 1] - t0;
    const int RH = p.cls_rh[cls], RW = p.cls_rw[cls], h0 = hd0 * p.xs + p.cls_h0[cls], w0 = wd0 * p.xs + p.cls_w0[cls];
    const int kc = p.C >> 4, chunks = nt > 0 ? kc : 0, npix = p.Nt * RH * RW;
    pk += (size_t)grp * q.pack_group;
    w += (size_t)grp * p.w_group;                    // read by direct_output only

    float* const raw = (float*)msm;                                              // fp32 only
    char* const planes = msm + (S ? q.xp * 64 : 0);                              // fp32: [part][half][pixel] 16 bytes; bf16: [buffer][half][pixel]
    const int plane_bytes = q.xp * 32;
    char* const wst = planes + (S ? 3 : 2) * plane_bytes;
    const int wbuf = q.wtaps * BLKS * U * 16;

    // the pixel whose 16 bytes this lane hands to ldmatrix (row lane % 16 of the 16-pixel group i; channels 8 (lane / 16) ...)
    uint32_t abase[2];
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const int px = warp * 32 + i * 16 + (lane & 15);
        const int pw = px & (p.Wt - 1), ph = (px >> p.lw) & (p.Ht - 1), pn = px >> (p.lw + p.lh);
        abase[i] = smem_addr(planes) + (uint32_t)(((lane >> 4) * q.xp + (pn * RH + ph * p.xs) * RW + pw * p.xs) * 16);
    }
    float2 sum[2][NB][2], lost[2][NB][2];
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < NB; ++j)
#pragma unroll
            for (int r = 0; r < 2; ++r) sum[i][j][r] = lost[i][j][r] = make_float2(0.f, 0.f);

    auto fetch_w = [&](int c, int buf) {
        for (int tb = warp; tb < nt * BLKS; tb += NW) {
            const int b = tb % BLKS, t = tb / BLKS;
            const uint4* const s = pk + ((size_t)((blockIdx.y * BLKS + b) * kc + c) * p.taps + p.wtap[t0 + t]) * U + lane;
            const uint32_t d = smem_addr(wst + buf * wbuf + (tb * U + lane) * 16);
#pragma unroll
            for (int i = 0; i < U / 32; ++i) cp_async16(d + i * 512, s + i * 32, true);
        }
    };
    auto fetch_x = [&](int c, int buf) {
        fetch_region<T>(x, S ? (char*)raw : planes + buf * plane_bytes, q.xp, n0, n_end, p.Nt, h0, w0, RH, RW, 1, p.H, p.W, p.C, c * FC_KC, warp, NW, lane);
    };
    if (chunks) { fetch_x(0, 0); fetch_w(0, 0); cp_commit(); }
    for (int c = 0; c < chunks; ++c) {
        const int buf = c & 1;
        if (S) {
            cp_wait<0>();
            __syncthreads();
            split_pixels<8>(raw, planes, q.xp, plane_bytes, npix, tid, MC_THREADS);
            __syncthreads();
            if (c + 1 < chunks) { fetch_x(c + 1, 0); fetch_w(c + 1, buf ^ 1); cp_commit(); }
        } else {
            if (c + 1 < chunks) { fetch_x(c + 1, buf ^ 1); fetch_w(c + 1, buf ^ 1); cp_commit(); cp_wait<1>(); } else cp_wait<0>();
            __syncthreads();
        }
        float rest[2][NB][4];                        // fp32 storage: of all products but hi hi, over the chunk
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int j = 0; j < NB; ++j) rest[i][j][0] = rest[i][j][1] = rest[i][j][2] = rest[i][j][3] = 0.f;
        const char* const ws_ = wst + buf * wbuf + lane * (S ? 16 : 8);
        const uint32_t xo = S ? 0u : (uint32_t)(buf * plane_bytes);
        auto tap = [&](int t, float (&part)[2][NB][4]) {
            const uint32_t off = xo + (uint32_t)p.toff[t0 + t] * 16u;
            uint32_t a[2][PARTS<T>][4], b[NB][PARTS<T>][2];
#pragma unroll
            for (int i = 0; i < 2; ++i)
#pragma unroll
                for (int k = 0; k < PARTS<T>; ++k) ldsm4(a[i][k], abase[i] + off + k * plane_bytes);
#pragma unroll
            for (int j = 0; j < NB; ++j) {
                const char* const s = ws_ + (t * BLKS + (j >> 1)) * (U * 16);
                if (S) {
                    const uint4 v = *(const uint4*)(s + (j & 1) * 512);
                    const uint2 l = *(const uint2*)(s - lane * 8 + 1024 + (j & 1) * 256);
                    b[j][0][0] = v.x; b[j][0][1] = v.y; b[j][PARTS<T> / 2][0] = v.z; b[j][PARTS<T> / 2][1] = v.w; b[j][PARTS<T> - 1][0] = l.x; b[j][PARTS<T> - 1][1] = l.y;
                } else { const uint2 v = *(const uint2*)(s + (j & 1) * 256); b[j][0][0] = v.x; b[j][0][1] = v.y; }
            }
#pragma unroll
            for (int k = 0; k < PRODUCTS<T>; ++k)
#pragma unroll
                for (int j = 0; j < NB; ++j)
#pragma unroll
                    for (int i = 0; i < 2; ++i) {
                        if (k + 1 < PRODUCTS<T>) mma(rest[i][j], a[i][part_a<T>(k)], b[j][part_b<T>(k)][0], b[j][part_b<T>(k)][1], true);
                        else mma(part[i][j], a[i][0], b[j][0][0], b[j][0][1], false);
                    }
        };
        auto each = [&](auto f) {                    // over the lane's pairs of outputs
#pragma unroll
            for (int i = 0; i < 2; ++i)
#pragma unroll
                for (int j = 0; j < NB; ++j)
#pragma unroll
                    for (int r = 0; r < 2; ++r) f(i, j, r);
        };
        auto pair = [](const float (&v)[4], int r) { return make_float2(v[2 * r], v[2 * r + 1]); };
        float one[2][NB][4];
        if constexpr (S) {                           // two taps into the compensated sum at a time
            int t = 0;
#pragma unroll 1
            for (; t + 1 < nt; t += 2) {
                float two[2][NB][4];
                tap(t, one); tap(t + 1, two);
                each([&](int i, int j, int r) { add_kahan(sum[i][j][r], lost[i][j][r], __fadd2_rn(pair(one[i][j], r), pair(two[i][j], r))); });
            }
            if (t < nt) { tap(t, one); each([&](int i, int j, int r) { add_kahan(sum[i][j][r], lost[i][j][r], pair(one[i][j], r)); }); }
            each([&](int i, int j, int r) { lost[i][j][r] = __fadd2_rn(lost[i][j][r], pair(rest[i][j], r)); });
        } else {                                     // the whole chunk
            float2 acc[2][NB][2];
            each([&](int i, int j, int r) { acc[i][j][r] = make_float2(0.f, 0.f); });
#pragma unroll 1
            for (int t = 0; t < nt; ++t) { tap(t, one); each([&](int i, int j, int r) { acc[i][j][r] = __fadd2_rn(acc[i][j][r], pair(one[i][j], r)); }); }
            each([&](int i, int j, int r) { add_kahan(sum[i][j][r], lost[i][j][r], acc[i][j][r]); });
        }
        if (!S) __syncthreads();                     // this buffer is consumed
    }

    float val[2][NB][2][2];
    bool valid[2][2];
    if constexpr (S) {
        uint32_t direct = 0;                         // outputs that are not finite, in the order of the loops
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int j = 0; j < NB; ++j)
#pragma unroll
                for (int r = 0; r < 2; ++r)
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        const float v = e ? total(sum[i][j][r].y, lost[i][j][r].y) : total(sum[i][j][r].x, lost[i][j][r].x);
                        val[i][j][r][e] = v * UNRANGE2;
                        direct |= (uint32_t)!isfinite(v) << (((i * NB + j) * 2 + r) * 2 + e);
                    }
        if (direct) {                                // apart from the loop above, whose code it would triple (2 us a launch)
            float redo[2 * NB * 4];
            const uint32_t nan = surely_nan<NB>(x, w, p, cls, n0, hd0, wd0, warp * 32 + g, n_end, co0 + 2 * tq);
#pragma unroll 1
            for (int k = 0; k < 2 * NB * 4; ++k) {
                const int px = warp * 32 + k / (NB * 4) * 16 + (k >> 1 & 1) * 8 + g;
                const int wd = wd0 + (px & (p.Wt - 1)), hd = hd0 + ((px >> p.lw) & (p.Ht - 1)), n = n0 + (px >> (p.lw + p.lh));
                if (nan >> k & 1) redo[k] = __int_as_float(0x7fffffff);
                else if (direct >> k & 1 && n < n_end && hd < p.Hd && wd < p.Wd) redo[k] = direct_output(x, w, p, cls, n, hd, wd, co0 + 8 * (k / 4 % NB) + 2 * tq + (k & 1));
            }
#pragma unroll
            for (int k = 0; k < 2 * NB * 4; ++k) if (direct >> k & 1) val[k / (NB * 4)][k / 4 % NB][k >> 1 & 1][k & 1] = redo[k];
        }
    }
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const int px = warp * 32 + i * 16 + r * 8 + g;
            const int wd = wd0 + (px & (p.Wt - 1)), hd = hd0 + ((px >> p.lw) & (p.Ht - 1)), n = n0 + (px >> (p.lw + p.lh));
            valid[i][r] = n < n_end && hd < p.Hd && wd < p.Wd;
            const size_t o = (((size_t)n * p.Ho + (hd * p.os + p.cls_oph[cls])) * p.Wo + (wd * p.os + p.cls_opw[cls])) * p.Co + co0 + 2 * tq;
#pragma unroll
            for (int j = 0; j < NB; ++j) {
                float a = S ? val[i][j][r][0] : total(sum[i][j][r].x, lost[i][j][r].x), b = S ? val[i][j][r][1] : total(sum[i][j][r].y, lost[i][j][r].y);
                if (valid[i][r]) {
                    const int co = co0 + 8 * j + 2 * tq;
                    if (bias) { a += bias[(size_t)grp * p.b_group + co]; b += bias[(size_t)grp * p.b_group + co + 1]; }
                    if (p.epi & EPI_RELU) { a = fmaxf(a, 0.f); b = fmaxf(b, 0.f); }
                    if (S || (p.epi & EPI_OUT_F32)) {
                        float2* const d = (float2*)((float*)y + o + 8 * j);
                        if (p.epi & EPI_ACCUM) { const float2 old = *d; a += old.x; b += old.y; }
                        *d = make_float2(a, b);
                    } else {
                        __nv_bfloat162* const d = (__nv_bfloat162*)((bf16*)y + o + 8 * j);
                        if (p.epi & EPI_ACCUM) { const __nv_bfloat162 old = *d; a += __low2float(old); b += __high2float(old); }
                        *d = __floats2bfloat162_rn(a, b);
                    }
                }
                val[i][j][r][0] = stored<T>(a); val[i][j][r][1] = stored<T>(b);
            }
        }
    if (!stat) return;
    // batch-norm statistics of the tile, from the values as stored: per channel the mean over its pixels and the sum of squared
    // deviations from that mean (no cancellation, whatever the mean); in a fixed order
    const int cnt = min(p.Wt, p.Wd - wd0) * min(p.Ht, p.Hd - hd0) * min(p.Nt, n_end - n0);
    float* const red = (float*)msm;                  // [warp][8 NB]
    float s[NB][2], mean[NB][2];
    auto over_pixels = [&](auto term) {
#pragma unroll
        for (int j = 0; j < NB; ++j)
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                s[j][e] = 0.f;
#pragma unroll
                for (int i = 0; i < 2; ++i)
#pragma unroll
                    for (int r = 0; r < 2; ++r) if (valid[i][r]) s[j][e] += term(val[i][j][r][e], mean[j][e]);
#pragma unroll
                for (int d = 4; d < 32; d <<= 1) s[j][e] += __shfl_xor_sync(0xffffffffu, s[j][e], d);
            }
        __syncthreads();
        if (g == 0)
#pragma unroll
            for (int j = 0; j < NB; ++j) *(float2*)(red + warp * (8 * NB) + 8 * j + 2 * tq) = make_float2(s[j][0], s[j][1]);
        __syncthreads();
#pragma unroll
        for (int j = 0; j < NB; ++j)
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const float* const c = red + 8 * j + 2 * tq + e;
                s[j][e] = (c[0] + c[8 * NB]) + (c[16 * NB] + c[24 * NB]);
            }
    };
    over_pixels([](float v, float) { return v; });
#pragma unroll
    for (int j = 0; j < NB; ++j)
#pragma unroll
        for (int e = 0; e < 2; ++e) mean[j][e] = s[j][e] / (float)cnt;
    over_pixels([](float v, float m) { const float d = v - m; return d * d; });
    if (warp == 0 && g == 0) {
        const int tiles = gridDim.x, groups = gridDim.z;
        const size_t rec = (size_t)grp * tiles + blockIdx.x;
#pragma unroll
        for (int j = 0; j < NB; ++j)
            *(float4*)(stat + (rec * p.Co + co0 + 8 * j + 2 * tq) * 2) = make_float4(mean[j][0], s[j][0], mean[j][1], s[j][1]);
        if (blockIdx.y == 0 && tq == 0) stat[(size_t)groups * tiles * p.Co * 2 + rec] = (float)cnt;
    }
}

constexpr int MW_WARPS = 6;              // two halves of c_in x (3x3: three rows of taps; 1x1: three pixel slices)
struct MwParams {
    FwParams p;                          // geometry; toff in pixels
    int npix, xp;                        // pixels of a tile, of its region
};
__host__ __device__ constexpr int mw_slices(int taps_a_warp) { return taps_a_warp == 3 ? 1 : 3; }
template <typename T> constexpr int mw_smem(int npix, int xp) { return (npix + xp) * (SPLIT<T> ? 64 + 96 : 2 * 32); }      // fp32: raw + parts; bf16: two buffers

// grid = (splits, c_out blocks x c_in blocks, groups).  part_out: [group][block][split][16 c_out][taps][16 c_in], as fw_kernel's.
template <typename T, int XS, int TW>
__global__ void __launch_bounds__(MW_WARPS * 32, SPLIT<T> ? 4 : 3) mw_kernel(const T* __restrict__ x, const T* __restrict__ dy, float* __restrict__ part_out,
                                                              const __grid_constant__ MwParams q) {
    constexpr bool S = SPLIT<T>;
    constexpr int SL = mw_slices(TW);
    extern __shared__ __align__(16) char msm[];
    const FwParams& p = q.p;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, tq = lane & 3;
    const int grp = blockIdx.z, cob = blockIdx.y / p.ci_blocks, cib = blockIdx.y % p.ci_blocks;
    const int co0 = cob * FW_CO, ci0 = cib * FW_CI;
    const int half = warp & 1, slice = SL > 1 ? warp >> 1 : 0, tap0 = SL > 1 ? 0 : (warp >> 1) * TW;
    const int xp = q.xp, npix = q.npix;
    float* const raw_x = (float*)msm;                                            // fp32 only
    float* const raw_d = raw_x + xp * 16;
    char* const px_ = msm + (S ? (xp + npix) * 64 : 0);                          // planes of x: fp32 [part][half][pixel] 16 bytes; bf16 [buffer][half][pixel]
    char* const pd_ = px_ + xp * 32 * (S ? 3 : 2);                               // planes of dy
    float2 sum[TW][2], lost[TW][2];
#pragma unroll
    for (int s = 0; s < TW; ++s)
#pragma unroll
        for (int r = 0; r < 2; ++r) sum[s][r] = lost[s][r] = make_float2(0.f, 0.f);
    const int per = (p.tiles + p.splits - 1) / p.splits;
    const int tile0 = blockIdx.x * per, tile_end = min(p.tiles, tile0 + per), n_end = (grp + 1) * p.ngroup;
    auto fetch = [&](int tl, int buf) {
        const int tw = tl % p.tiles_w; tl /= p.tiles_w;
        const int th = tl % p.tiles_h, tn = tl / p.tiles_h;
        const int n0 = grp * p.ngroup + tn * p.Nt, ho0 = th * p.Ht, wo0 = tw * p.Wt;
        fetch_region<T>(x, S ? (char*)raw_x : px_ + buf * xp * 32, xp, n0, n_end, p.Nt, ho0 * p.hstep - p.pad, wo0 * p.hstep - p.pad, p.RH, p.RW, p.step, p.H, p.W, p.C,
                        ci0, warp, MW_WARPS, lane);
        constexpr int Q = S ? 4 : 2;
        const int c = tid % Q;
        const T* const d0 = dy + co0 + c * (16 / Q);
        for (int px = tid / Q; px < npix; px += MW_WARPS * 32 / Q) {
            const int w = wo0 + (px & (p.Wt - 1)), h = ho0 + ((px >> p.lw) & (p.Ht - 1)), n = n0 + (px >> (p.lw + p.lh));
            const bool in = n < n_end && h < p.Ho && w < p.Wo;
            cp_async16(smem_addr(S ? (char*)(raw_d + raw_at(px, c)) : pd_ + buf * npix * 32 + (c * npix + px) * 16), in ? d0 + (((size_t)n * p.Ho + h) * p.Wo + w) * p.Co : dy, in);
        }
        cp_commit();
    };
    auto region_pixel = [&](int px) { return ((px >> (p.lw + p.lh)) * p.RH + ((px >> p.lw) & (p.Ht - 1)) * XS) * p.RW + (px & (p.Wt - 1)) * XS; };
    if (tile0 < tile_end) fetch(tile0, 0);
    for (int tile = tile0; tile < tile_end; ++tile) {
        const int buf = (tile - tile0) & 1;
        if (S) {
            cp_wait<0>();
            __syncthreads();
            split_pixels<8>(raw_x, px_, xp, xp * 32, xp, tid, MW_WARPS * 32);
            split_pixels<DY_HI>(raw_d, pd_, npix, npix * 32, npix, tid, MW_WARPS * 32);
            __syncthreads();
            if (tile + 1 < tile_end) fetch(tile + 1, 0);
        } else {
            if (tile + 1 < tile_end) { fetch(tile + 1, buf ^ 1); cp_wait<1>(); } else cp_wait<0>();
            __syncthreads();
        }
        const uint32_t dbase = smem_addr(pd_) + (S ? 0 : buf * npix * 32) + (((lane >> 3) & 1) * npix + (lane & 7) + 8 * (lane >> 4)) * 16;
        // rows of x that this lane hands to ldmatrix: pixel lane % 16; lanes 16..31 those of the second part (fp32), nobody's (bf16)
        const uint32_t xbase = smem_addr(px_) + (S ? 0 : buf * xp * 32) + (half * xp + p.toff[tap0]) * 16;
        float rest[TW][4];                           // fp32 storage: this tile's sum of all products but hi hi
        float2 acc[TW][2];                           // bf16 storage: of MW_RUN steps
#pragma unroll
        for (int s = 0; s < TW; ++s) {
            rest[s][0] = rest[s][1] = rest[s][2] = rest[s][3] = 0.f;
            acc[s][0] = acc[s][1] = make_float2(0.f, 0.f);
        }
        int run = 0;
#pragma unroll 1
        for (int ks = slice; ks * 16 < npix; ks += SL) {
            uint32_t a[PARTS<T>][4], b[TW][PARTS<T>][2];
            float part[TW][4];
            const uint32_t xa = xbase + region_pixel(ks * 16 + (lane & 15)) * 16;
#pragma unroll
            for (int k = 0; k < PARTS<T>; ++k) ldsm4t(a[k], dbase + ks * 256 + k * npix * 32);
#pragma unroll
            for (int s = 0; s < TW; ++s) {
                if (S) {
                    uint32_t v[4];
                    ldsm4t(v, xa + s * 16 + (lane >> 4) * xp * 32);
                    b[s][0][0] = v[0]; b[s][0][1] = v[1]; b[s][PARTS<T> / 2][0] = v[2]; b[s][PARTS<T> / 2][1] = v[3];
                }
                ldsm2t(b[s][PARTS<T> - 1], xa + s * 16 + (PARTS<T> - 1) * xp * 32);
            }
#pragma unroll
            for (int k = 0; k < PRODUCTS<T>; ++k)
#pragma unroll
                for (int s = 0; s < TW; ++s) {
                    if (k + 1 < PRODUCTS<T>) mma(rest[s], a[part_a<T>(k)], b[s][part_b<T>(k)][0], b[s][part_b<T>(k)][1], true);
                    else mma(part[s], a[0], b[s][0][0], b[s][0][1], false);
                }
#pragma unroll
            for (int s = 0; s < TW; ++s)
#pragma unroll
                for (int r = 0; r < 2; ++r) {
                    const float2 v = make_float2(part[s][2 * r], part[s][2 * r + 1]);
                    if (S) add_kahan(sum[s][r], lost[s][r], v); else acc[s][r] = __fadd2_rn(acc[s][r], v);
                }
            if (!S && (++run == MW_RUN || (ks + SL) * 16 >= npix)) {
                run = 0;
#pragma unroll
                for (int s = 0; s < TW; ++s)
#pragma unroll
                    for (int r = 0; r < 2; ++r) { add_kahan(sum[s][r], lost[s][r], acc[s][r]); acc[s][r] = make_float2(0.f, 0.f); }
            }
        }
        if (S)
#pragma unroll
            for (int s = 0; s < TW; ++s)
#pragma unroll
                for (int r = 0; r < 2; ++r) lost[s][r] = __fadd2_rn(lost[s][r], make_float2(rest[s][2 * r], rest[s][2 * r + 1]));
        if (!S) __syncthreads();                     // this buffer is consumed
    }
    // the slices' sums in slice order, then the CTA's partial matrix
    const int nout = FW_CO * p.ntaps * FW_CI;
    float* const red = (float*)msm;                  // [slice][16][taps][16]
    __syncthreads();
#pragma unroll
    for (int s = 0; s < TW; ++s)
#pragma unroll
        for (int r = 0; r < 2; ++r)
            *(float2*)(red + (size_t)slice * nout + ((g + 8 * r) * p.ntaps + tap0 + s) * 16 + 8 * half + 2 * tq) =
                make_float2(total(sum[s][r].x, lost[s][r].x), total(sum[s][r].y, lost[s][r].y));
    __syncthreads();
    float* const out = part_out + (((size_t)grp * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x) * nout;
    bool direct = false;
    for (int i = tid; i < nout; i += MW_WARPS * 32) {
        double s = 0;
        for (int k = 0; k < SL; ++k) s += (double)red[(size_t)k * nout + i];
        if (S) { direct |= !isfinite(s); s *= UNRANGE2; }
        out[i] = (float)s;
    }
    if constexpr (S)
        if (direct)
#pragma unroll 1
            for (int i = tid; i < nout; i += MW_WARPS * 32)
                if (!isfinite(out[i])) out[i] = direct_wgrad(x, dy, p, grp, tile0, tile_end, co0 + i / (p.ntaps * 16), i / 16 % p.ntaps, ci0 + i % 16);
}

// One CTA per 16 x 16 block of a layer's matrices (all taps): [n block][k chunk][tap][n8][lane], per lane the B operand of one mma: the values (k = 2 t, 2 t + 1
// and 2 t + 8, 2 t + 9; n = lane / 4), t = lane % 4; fp32: 16 bytes of hi and mid each, then 8 of lo each.  Forward: n = output, k = input channel; back: the reverse.
template <typename T>
__global__ void __launch_bounds__(256) mc_pack_kernel(const T* __restrict__ wbig, size_t w_group, uint4* __restrict__ out, size_t out_group, const __grid_constant__ PackArgs a) {
    __shared__ float ws[9 * 256 + 16];
    int l = 0;
    while (l + 1 < a.n && (int)blockIdx.x >= a.layer[l + 1].block0) ++l;
    const PackLayer& L = a.layer[l];
    const int blk = blockIdx.x - L.block0, cib = blk % (L.C / 16), cob = blk / (L.C / 16), tid = threadIdx.x;
    wbig += (size_t)blockIdx.y * w_group + L.w_off;
    out += (size_t)blockIdx.y * out_group + L.out_off;
    for (int i = tid; i < L.taps * 256; i += 256) {
        const int ci = i & 15, tap = (i >> 4) % L.taps, co = (i >> 4) / L.taps;
        ws[(co * L.taps + tap) * 16 + ci] = (float)wbig[((size_t)(cob * 16 + co) * L.taps + tap) * L.C + cib * 16 + ci];
    }
    __syncthreads();
    const int nb = a.back ? cib : cob, kb = a.back ? cob : cib, kc = (a.back ? L.Co : L.C) / 16;
    for (int i = tid; i < L.taps * 64; i += 256) {
        const int lane = i & 31, n8 = (i >> 5) & 1, tap = i >> 6, n = n8 * 8 + (lane >> 2), k0 = 2 * (lane & 3);
        uint32_t h[2], mid[2], lo[2];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            float v[2];
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                const int k = k0 + 8 * u + j;
                v[j] = ws[((a.back ? k : n) * L.taps + tap) * 16 + (a.back ? n : k)];
            }
            if (SPLIT<T>) {
                split2<W_HI>(v[0] * RANGE, v[1] * RANGE, h[u], mid[u], lo[u]);
            } else {
                const __nv_bfloat162 b = __floats2bfloat162_rn(v[0], v[1]);
                h[u] = *(const uint32_t*)&b;
            }
        }
        uint4* const d = out + ((size_t)(nb * kc + kb) * L.taps + tap) * PACK16<T>;
        if (SPLIT<T>) { d[n8 * 32 + lane] = make_uint4(h[0], h[1], mid[0], mid[1]); ((uint2*)(d + 64))[n8 * 32 + lane] = make_uint2(lo[0], lo[1]); }
        else ((uint2*)d)[n8 * 32 + lane] = make_uint2(h[0], h[1]);
    }
}

constexpr int SM_SMEM = 228 * 1024, CTA_SMEM = 1024;      // of an SM; what every CTA takes beside its own

bool channels_ok(const ConvGeom& g) { return g.C % 16 == 0 && g.Co % 16 == 0; }
template <typename T, int NB> size_t mc_smem(const McParams& q) { return (size_t)mc_x_bytes<T>(q.xp) + mc_w_bytes<T, NB>(q.wtaps, q.p.C / 16); }

// CTAs of 16 output channels; the four parity classes of a 1x1 stride-2 input gradient, three of which have no tap and only write, count as two
long mc_ctas(const McParams& q, int groups) {
    const int classes = q.p.ncls > 1 && q.p.taps == 1 ? 2 : q.p.ncls;
    return (long)classes * q.p.tiles_w * q.p.tiles_h * ((q.p.ngroup + q.p.Nt - 1) / q.p.Nt) * groups * (q.p.Co / 16);
}
// Whether mc_kernel takes a launch; the packed-FMA kernel has the others.  Both cut images into the same tiles.  A tile's region is fetched row by row, a warp a
// row, and with fp32 storage split pixel by pixel before it is used; the packed-FMA kernel reads it as it is.  So the line lies where a
// tile has many rows or, per tap, many pixels for its 128 outputs: small images, sides that exact covers of 2x2x32 or 1x1x128 pixels leave
// (5, 6, 9, 10, 13, 14 ...), 1x1 layers; and further out where the CTAs of one wave have nobody to cover for them.  From 3 to 25 sides of 1 to
// 56, 16 to 256 channels, 4 to 768 images (tensor core : packed FMA of the launches just inside / just outside):
//   fp32 3x3            region of 300 pixels in up to one wave, 512 beyond      0.92 / 1.2 (5x5 and 6x6 images, 16 of them), 1.05 / 2.0 (1x1)
//   fp32 3x3 stride 2   forward: 36 rows; backward: 180 pixels, 288 beyond      1.08 / 1.6 (20x20, 28x28 in 16 channels); 1.07 / 1.27 (4x4)
//   fp32 1x1            4 rows in up to one wave, 16 in up to two, any beyond   1.0 / 1.25, 1.05 / 1.18, 1.05 / -
//   bf16                128 rows in up to one wave, any beyond; 1x1 with fewer images than a tile holds: 32     0.96 / 1.26, 1.0 / 1.17
// Some launches outside would gain: 0.7 at the best (bf16, 1x1 images, one wave).
template <typename T> bool worth_it(const McParams& q, int groups) {
    int rows = 0;
    for (int c = 0; c < q.p.ncls; ++c) rows = std::max(rows, q.p.Nt * q.p.cls_rh[c]);
    const long ctas = mc_ctas(q, groups);
    const bool few = ctas <= 148;
    if (!SPLIT<T>) return (rows <= 128 || !few) && !(q.p.taps == 1 && rows > 32 && q.p.ngroup < q.p.Nt);
    if (q.p.taps == 1) return ctas > 2 * 148 || rows <= (few ? 4 : 16);
    if (q.p.xs == 2) return rows <= 36;
    if (q.p.ncls > 1) return q.xp <= (few ? 180 : 288);
    return q.xp <= (few ? 300 : 512);
}
template <typename T>
bool plan_mc(const ConvGeom& g, int groups, bool back, McParams& q) {
    if (!channels_ok(g) || !plan_fc(g, groups, back, q.p)) return false;
    q.xp = q.p.x_floats / PITCH;
    q.wtaps = q.p.w_floats / (16 * PITCH);
    for (int& t : q.p.toff) t /= PITCH;
    return mc_smem<T, 4>(q) <= FC_SMEM_MAX && worth_it<T>(q, groups);
}
template <typename T>
bool plan_mw(const ConvGeom& g, int groups, MwParams& q, size_t& smem) {
    int G, run; size_t fw;
    if (!channels_ok(g) || !plan_fw(g, groups, FW_CTAS, q.p, G, run, fw)) return false;
    q.npix = q.p.Wt * q.p.Ht * q.p.Nt;
    q.xp = q.p.x_floats / PITCH;
    // splits for one wave: registers allow four CTAs per SM (bf16 storage three), shared memory as few as one where regions are large (stride 2, small
    // images); with four for all of them a second wave ran: 32 -> 64 stride 2, 64 images of 28x28 52 us (packed FMA 49), now 45; 768 of 20x20 263 (233), now 203
    const int fit = (int)(SM_SMEM / (mw_smem<T>(q.npix, q.xp) + CTA_SMEM)), most = (SPLIT<T> ? MW_CTAS : FW_CTAS) / 148;
    if (!plan_fw(g, groups, 148 * std::max(1, std::min(fit, most)), q.p, G, run, fw)) return false;
    for (int i = 0; i < q.p.ntaps; ++i) q.p.toff[i] /= PITCH;
    const size_t red = (size_t)mw_slices(g.R) * FW_CO * q.p.ntaps * FW_CI * sizeof(float);
    smem = mw_smem<T>(q.npix, q.xp);
    if (red > smem) smem = red;
    return q.npix % 16 == 0 && smem <= FC_SMEM_MAX;
}

template <typename T, int NB>
cudaError_t launch_mc(const void* x, const void* w, const void* pk, const float* bias, void* y, float* stat, const McParams& q, int groups, cudaStream_t s) {
    static OncePerDevice once;
    if (cudaError_t e = allow_smem(once, (const void*)mc_kernel<T, NB>, (int)FC_SMEM_MAX)) return e;
    const int tiles = q.p.tiles_w * q.p.tiles_h * ((q.p.ngroup + q.p.Nt - 1) / q.p.Nt);
    return klaunch(mc_kernel<T, NB>, dim3(tiles, q.p.Co / (8 * NB), groups * q.p.ncls), MC_THREADS, mc_smem<T, NB>(q), s, (const T*)x, (const T*)w, (const uint4*)pk, bias, (T*)y, stat, q);
}
template <typename T>
bool run_mc(const void* x, const void* w, const void* pk, const float* bias, void* y, float* stat, const ConvGeom& g, int epi, int groups, size_t w_group, size_t b_group, size_t pack_group, bool back,
            cudaStream_t s) {
    McParams q;
    if (!plan_mc<T>(g, groups, back, q)) return false;
    Scope sc(back ? KC_MMA_DGRAD : KC_MMA_FWD, conv_flops(g), conv_bytes(SPLIT<T> ? 0 : 1, g, false), s);
    q.p.epi = epi; q.p.w_group = w_group; q.p.b_group = b_group;
    q.pack_group = pack_group / 16;
    const long tiles = (long)q.p.tiles_w * q.p.tiles_h * ((q.p.ngroup + q.p.Nt - 1) / q.p.Nt) * groups * q.p.ncls;
    // 32 output channels a CTA (a third less shared-memory traffic per product, the region split for twice the work), unless 16 fill the device more evenly;
    // large regions (stride 2) leave an SM two CTAs at the most either way.  fp32 3x3 stride 1: 16 also where they make one wave of four per SM and up to three
    // quarters of another, 0.82 to 0.98 of the time of 32 (192 images of 16x16, 32 -> 32: 25 us against 30; from 1.95 waves on 1.16 and more)
    const auto waves = [](long ctas) { return (ctas + 147) / 148; };
    const long narrow = tiles * (q.p.Co / 16);
    const bool tail = SPLIT<T> && q.p.taps == 9 && q.p.ncls == 1 && q.p.xs == 1 && narrow > 4 * 148 && narrow <= 7 * 148;
    const bool wide = q.p.Co % 32 == 0 && (mc_smem<T, 2>(q) > 75 * 1024 || (!tail && 2 * waves(tiles * (q.p.Co / 32)) <= 1.15 * waves(narrow)));
    return launched(wide ? launch_mc<T, 4>(x, w, pk, bias, y, stat, q, groups, s) : launch_mc<T, 2>(x, w, pk, bias, y, stat, q, groups, s));
}
template <typename T, int XS, int TW>
cudaError_t launch_mw(const void* x, const void* dy, float* ws, const MwParams& q, int groups, int blocks, size_t smem, cudaStream_t s) {
    static OncePerDevice once;
    if (cudaError_t e = allow_smem(once, (const void*)mw_kernel<T, XS, TW>, (int)FC_SMEM_MAX)) return e;
    return klaunch(mw_kernel<T, XS, TW>, dim3(q.p.splits, blocks, groups), MW_WARPS * 32, smem, s, (const T*)x, (const T*)dy, ws, q);
}
template <typename T>
int run_mw(const void* x, const void* dy, float* ws, const ConvGeom& g, int groups, cudaStream_t s) {
    MwParams q; size_t smem;
    if (!plan_mw<T>(g, groups, q, smem)) return 0;
    Scope sc(KC_MMA_WGRAD, conv_flops(g), conv_bytes(SPLIT<T> ? 0 : 1, g, true), s);
    const int blocks = q.p.ci_blocks * (g.Co / FW_CO);
    cudaError_t e;
    if (g.R == 1) e = launch_mw<T, 1, 1>(x, dy, ws, q, groups, blocks, smem, s);
    else if (g.stride == 1) e = launch_mw<T, 1, 3>(x, dy, ws, q, groups, blocks, smem, s);
    else e = launch_mw<T, 2, 3>(x, dy, ws, q, groups, blocks, smem, s);
    return launched(e) ? q.p.splits : 0;
}

}  // namespace

bool mconv_takes(int dt, const ConvGeom& g, int groups, bool back) {
    McParams q;
    return dt ? plan_mc<bf16>(g, groups, back, q) : plan_mc<float>(g, groups, back, q);
}
size_t mconv_pack_bytes(int dt, const ConvGeom& g) { return (size_t)(g.C / 16) * (g.Co / 16) * g.R * g.R * (dt ? PACK16<bf16> : PACK16<float>) * 16; }
bool mconv_pack(int dt, const void* wbig, size_t w_group, void* out, size_t out_group, const PackArgs& a, int blocks, int groups, cudaStream_t s) {
    Scope sc(KC_TC_AUX, 0.0, (double)blocks * groups * 9 * 256 * (dt ? 4.0 : 8.0), s);
    return launched(dt ? klaunch(mc_pack_kernel<bf16>, dim3(blocks, groups), 256, 0, s, (const bf16*)wbig, w_group, (uint4*)out, out_group / 16, a)
                       : klaunch(mc_pack_kernel<float>, dim3(blocks, groups), 256, 0, s, (const float*)wbig, w_group, (uint4*)out, out_group / 16, a));
}
bool mconv_forward(int dt, const void* x, const void* w, const Packed& pk, const float* bias, void* y, float* stat, const ConvGeom& g, int epi, int groups, size_t w_group, size_t b_group,
                   cudaStream_t s) {
    return (dt ? run_mc<bf16> : run_mc<float>)(x, w, pk.data, bias, y, stat, g, epi, groups, w_group, b_group, pk.group, false, s);
}
bool mconv_dgrad(int dt, const void* dy, const void* w, const Packed& pk, void* dx, const ConvGeom& g, int epi, int groups, size_t w_group, cudaStream_t s) {
    return (dt ? run_mc<bf16> : run_mc<float>)(dy, w, pk.data, nullptr, dx, nullptr, g, epi, groups, w_group, 0, pk.group, true, s);
}
int mconv_wgrad(int dt, const void* x, const void* dy, float* ws, const ConvGeom& g, int groups, cudaStream_t s) {
    return dt ? run_mw<bf16>(x, dy, ws, g, groups, s) : run_mw<float>(x, dy, ws, g, groups, s);
}

}  // namespace fdg
