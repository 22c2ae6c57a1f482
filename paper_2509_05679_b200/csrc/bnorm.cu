// Batch-norm with fp32 storage (statistics per worker), two launches per layer and direction at most:
//   forward : the producing convolution has left per-tile (mean, sum of squared deviations) (fconv.cu); ONE kernel merges them
//             and normalises.  Backward: one kernel of partial sums, one that finishes the sums and applies them.
// The generic kernels (kernels.cu) take three launches each, read 4 bytes per thread and load instruction and use half of
// their lanes at 16 channels; the paper's ResNet-20 has 21 batch-norms per step, all of them resident in L2 (12.6 MB at the most),
// so that launches and bytes in flight count, not DRAM.  A thread keeps 4 consecutive channels (16-byte accesses) for every row
// it visits; a CTA owns a contiguous row range of one worker.  Used when C / 4 is a power of two <= 256.
// Every sum has a fixed order.
#include "kernels.h"
#include "launch.h"

#include <cuda_bf16.h>

namespace fdg {

typedef __nv_bfloat16 bf16;

namespace {

constexpr int BT = 256;
constexpr int BNF_MAX_CHUNKS = 64;

struct BnfArgs {
    const float* x; const float* out; const float* dout; const float* res;
    const float* gamma; const float* beta; size_t p_group;      // floats between the workers' gamma / beta (0: shared)
    float* stats;                                               // [worker][C][4]: mean, invstd, and what those fp32 values are off by
    const float* tile_part; int tiles;                          // forward: the convolution's records (see fconv_stat_tiles)
    float* part;                                                // backward: [chunk][worker][C][2]
    float* y; float* dres; int accum_dx, accum_dres;
    float* dgamma; float* dbeta; size_t g_group; int accum_params;
    long rpw; int C, relu, mask_from_x;
};

// (mean, invstd) of worker w from its tiles' (mean m_t, sum of squared deviations q_t, count n_t), in double, in one pass: with the first
// tile's mean as the pivot p and d_t = m_t - p,  mean = p + S1 / N,  N var = S2 - S1^2 / N,  S1 = sum n_t d_t,  S2 = sum (q_t + n_t d_t^2);
// for the channels c0 .. c0 + nc - 1 (nc <= BT, a power of two).  Every CTA of a normalising launch does this by itself, so it is the
// launch's latency that counts: four records in flight per thread.  tmp: BT double2.
__device__ __forceinline__ void merge_tiles(const float* __restrict__ part, int tiles, int w, int nw, int C, int c0, int nc, long rows, float4* dst, double2* tmp) {
    const int tid = threadIdx.x, lanes = BT / nc, c = tid % nc, pt = tid / nc;
    const float2* p = (const float2*)part + (size_t)w * tiles * C + c0 + c;
    const float* cnt = part + (size_t)nw * tiles * C * 2 + (size_t)w * tiles;
    const double pivot = (double)p[0].x;
    double s1 = 0.0, s2 = 0.0;
    auto add = [&](float2 v, float n) { const double d = (double)v.x - pivot, nd = (double)n * d; s1 += nd; s2 += (double)v.y + nd * d; };
    int t = pt;
    for (; t + 3 * lanes < tiles; t += 4 * lanes) {
        float2 v[4]; float n[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) { v[u] = p[(size_t)(t + u * lanes) * C]; n[u] = cnt[t + u * lanes]; }
#pragma unroll
        for (int u = 0; u < 4; ++u) add(v[u], n[u]);
    }
    for (; t < tiles; t += lanes) add(p[(size_t)t * C], cnt[t]);
    tmp[tid] = make_double2(s1, s2);
    __syncthreads();
    for (int d = lanes / 2; d > 0; d >>= 1) {
        if (pt < d) { const double2 o = tmp[tid + d * nc]; tmp[tid].x += o.x; tmp[tid].y += o.y; }
        __syncthreads();
    }
    if (pt == 0) {
        const double2 a = tmp[c];
        const double mean = pivot + a.x / (double)rows, m2 = fmax(a.y - a.x * a.x / (double)rows, 0.0);
        const double istd = 1.0 / sqrt(m2 / (double)rows + 1e-5);
        const float mh = (float)mean, ih = (float)istd;
        dst[c] = make_float4(mh, ih, (float)(mean - (double)mh), (float)(istd - (double)ih));
    }
    __syncthreads();
}

// stats only (bf16 storage: the streamed apply kernel of kernels.cu follows).  grid = (channel blocks of min(C, 64), workers)
__global__ void __launch_bounds__(BT) bn_merge_tiles_k(const float* __restrict__ part, float* __restrict__ stats, int tiles, int C, int nc, long rows) {
    __shared__ double2 tmp[BT];
    __shared__ float4 res[BT];
    const int c0 = blockIdx.x * nc, w = blockIdx.y;
    merge_tiles(part, tiles, w, gridDim.y, C, c0, nc, rows, res, tmp);
    if ((int)threadIdx.x < nc) *(float2*)(stats + ((size_t)w * C + c0 + threadIdx.x) * 2) = make_float2(res[threadIdx.x].x, res[threadIdx.x].y);
}

// gamma * (x - mean) * invstd + beta with the roundings that matter near zero carried along: a ReLU decides on the sign of this
// value, and the plain fp32 expression (four roundings, two of them of constants that a whole channel shares) is off by more
// than the stored x and the stored result are.  scale + scale_lo = gamma * invstd, mean + mean_lo, invstd + invstd_lo from the double-
// precision merge.  One expression for both directions, so that the backward pass finds the same sign.
struct BnCoef { float mean, scale, scale_lo, beta, mean_lo; };
__device__ __forceinline__ BnCoef bn_coef(float4 st, float gamma, float beta) {
    BnCoef k;
    k.mean = st.x; k.mean_lo = st.z; k.beta = beta;
    k.scale = __fmul_rn(gamma, st.y);
    k.scale_lo = __fmaf_rn(gamma, st.w, __fmaf_rn(gamma, st.y, -k.scale));
    return k;
}
__device__ __forceinline__ float bn_value(float x, const BnCoef& k) {
    const float d = __fsub_rn(x, k.mean), t = __fadd_rn(d, k.mean);          // two-sum: x - mean = d + e exactly (as far as fp32 holds e)
    const float e = __fadd_rn(__fsub_rn(x, t), __fsub_rn(__fsub_rn(t, d), k.mean));
    return __fadd_rn(__fmaf_rn(d, k.scale, k.beta), __fmaf_rn(d, k.scale_lo, __fmul_rn(__fsub_rn(e, k.mean_lo), k.scale)));
}

__device__ __forceinline__ float2 warp_sum(float2 v) {
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) { v.x += __shfl_xor_sync(0xffffffffu, v.x, d); v.y += __shfl_xor_sync(0xffffffffu, v.y, d); }
    return v;
}

// MODE 0: y = bn(x) (+ res) (relu).  MODE 1: partial sums of (dy, dy * xhat), dy = dout * [out > 0] if relu.
// MODE 2: dx (+)= gamma * invstd * (dy - mean(dy) - xhat * mean(dy xhat)), dres (+)= dy, dgamma, dbeta.
template <int MODE>
__global__ void __launch_bounds__(BT) bnf_kernel(const BnfArgs a) {
    __shared__ double2 tmp[BT];
    __shared__ float4 st4[1024];                 // MODE 0: statistics; MODE 2: (sum dy, sum dy xhat); MODE 1: reduction
    float2* const st = (float2*)st4;
    const int C = a.C, cgs = C / 4, rows_it = BT / cgs, tid = threadIdx.x, cg = tid % cgs, rl = tid / cgs;
    const int w = blockIdx.y, nw = gridDim.y, chunks = gridDim.x;
    long per = (a.rpw + chunks - 1) / chunks;
    per = (per + rows_it - 1) / rows_it * rows_it;
    const long r0 = (long)blockIdx.x * per, r1 = min(a.rpw, r0 + per);
    if (MODE == 0) {
        const int nc = C < BT ? C : BT;
        for (int c0 = 0; c0 < C; c0 += nc) merge_tiles(a.tile_part, a.tiles, w, nw, C, c0, nc, a.rpw, st4 + c0, tmp);
        if (blockIdx.x == 0) for (int c = tid; c < C; c += BT) *(float4*)(a.stats + ((size_t)w * C + c) * 4) = st4[c];
    }
    if (MODE == 2) {
        const float2* const part = (const float2*)a.part;
        float2* const t2 = (float2*)tmp;
        const int nc = C < BT ? C : BT, lanes = BT / nc, c = tid % nc, pt = tid / nc;
        for (int c0 = 0; c0 < C; c0 += nc) {
            float2 s = make_float2(0.f, 0.f);
            for (int k = pt; k < chunks; k += lanes) { const float2 v = part[((size_t)k * nw + w) * C + c0 + c]; s.x += v.x; s.y += v.y; }
            t2[tid] = s;
            __syncthreads();
            if (pt == 0) {
                float2 t = make_float2(0.f, 0.f);
                for (int q = 0; q < lanes; ++q) { t.x += t2[q * nc + c].x; t.y += t2[q * nc + c].y; }
                st[c0 + c] = t;
            }
            __syncthreads();
        }
        if (a.g_group) {                         // every worker has parameters of its own
            if (blockIdx.x == 0) for (int e = tid; e < C; e += BT) { a.dbeta[w * a.g_group + e] = st[e].x; a.dgamma[w * a.g_group + e] = st[e].y; }
        } else {                                 // sums over all workers: one warp per channel, spread over the launch's CTAs
            const int warp = tid >> 5, lane = tid & 31, rows = nw * chunks, me = w * chunks + blockIdx.x;
            for (int e = me + warp * rows; e < C; e += (BT / 32) * rows) {
                float2 s = make_float2(0.f, 0.f);
                for (int r = lane; r < rows; r += 32) { const float2 v = part[((size_t)(r % chunks) * nw + r / chunks) * C + e]; s.x += v.x; s.y += v.y; }
                s = warp_sum(s);
                if (lane == 0) { a.dbeta[e] = a.accum_params ? a.dbeta[e] + s.x : s.x; a.dgamma[e] = a.accum_params ? a.dgamma[e] + s.y : s.y; }
            }
        }
    }
    float mean[4], istd[4], ga[4], c1[4], c2[4], s1[4], s2[4];
    BnCoef k[4];
    const float inv_n = 1.f / (float)a.rpw;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const int c = cg * 4 + j;
        const float4 ms = MODE == 0 ? st4[c] : *(const float4*)(a.stats + ((size_t)w * C + c) * 4);
        mean[j] = ms.x; istd[j] = ms.y;
        ga[j] = a.gamma[w * a.p_group + c];
        k[j] = bn_coef(ms, ga[j], a.beta[w * a.p_group + c]);
        if (MODE == 2) { c1[j] = st[c].x * inv_n; c2[j] = st[c].y * inv_n; }
        s1[j] = s2[j] = 0.f;
    }
    const size_t base = ((size_t)w * a.rpw) * C + (size_t)cg * 4;
    const bool need_out = MODE != 0 && a.relu && !a.mask_from_x;
    constexpr int U = 4;                         // rows in flight per thread
    for (long r = r0 + rl; r < r1; r += (long)rows_it * U) {
        float4 xv[U], dv[U], ov[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const long rr = r + (long)u * rows_it;
            if (rr >= r1) continue;
            const size_t o = base + (size_t)rr * C;
            xv[u] = *(const float4*)(a.x + o);
            if (MODE == 0) { if (a.res) ov[u] = *(const float4*)(a.res + o); }
            else { dv[u] = *(const float4*)(a.dout + o); if (need_out) ov[u] = *(const float4*)(a.out + o); }
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const long rr = r + (long)u * rows_it;
            if (rr >= r1) continue;
            const size_t o = base + (size_t)rr * C;
            const float x[4] = {xv[u].x, xv[u].y, xv[u].z, xv[u].w};
            if (MODE == 0) {
                float v[4];
                const float re[4] = {ov[u].x, ov[u].y, ov[u].z, ov[u].w};
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    v[j] = bn_value(x[j], k[j]);
                    if (a.res) v[j] += re[j];
                    if (a.relu) v[j] = fmaxf(v[j], 0.f);
                }
                *(float4*)(a.y + o) = make_float4(v[0], v[1], v[2], v[3]);
            } else {
                float d[4] = {dv[u].x, dv[u].y, dv[u].z, dv[u].w};
                const float ou[4] = {ov[u].x, ov[u].y, ov[u].z, ov[u].w};
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    if (a.relu && !((need_out ? ou[j] : bn_value(x[j], k[j])) > 0.f)) d[j] = 0.f;
                    if (MODE == 1) { s1[j] += d[j]; s2[j] += d[j] * (x[j] - mean[j]) * istd[j]; }
                }
                if (MODE == 2) {
                    float v[4];
#pragma unroll
                    for (int j = 0; j < 4; ++j) { const float xh = (x[j] - mean[j]) * istd[j]; v[j] = ga[j] * istd[j] * (d[j] - c1[j] - xh * c2[j]); }
                    if (a.y) {
                        if (a.accum_dx) { const float4 old = *(const float4*)(a.y + o); v[0] += old.x; v[1] += old.y; v[2] += old.z; v[3] += old.w; }
                        *(float4*)(a.y + o) = make_float4(v[0], v[1], v[2], v[3]);
                    }
                    if (a.dres) {
                        if (a.accum_dres) { const float4 old = *(const float4*)(a.dres + o); d[0] += old.x; d[1] += old.y; d[2] += old.z; d[3] += old.w; }
                        *(float4*)(a.dres + o) = make_float4(d[0], d[1], d[2], d[3]);
                    }
                }
            }
        }
    }
    if (MODE == 1) {
        static_assert(sizeof(float) * BT * 8 <= sizeof(st4), "reduction space");
        float* const r8 = (float*)st;            // [8][256]: value i of thread t at i * 256 + t (no bank conflicts)
#pragma unroll
        for (int j = 0; j < 4; ++j) { r8[j * BT + tid] = s1[j]; r8[(4 + j) * BT + tid] = s2[j]; }
        __syncthreads();
        for (int t = tid; t < 2 * C; t += BT) {
            const int c = t >> 1, v = (t & 1) * 4 + (c & 3), q = c >> 2;
            float acc = 0.f;
            for (int i = 0; i < rows_it; ++i) acc += r8[v * BT + i * cgs + q];
            a.part[(((size_t)blockIdx.x * nw + w) * C + c) * 2 + (t & 1)] = acc;
        }
    }
}

// ------------------------------------------------------------------------------------------ bf16 storage, small tensors
// Batch-norm of a tensor that fits in L2, ONE launch per direction: a cluster of eight CTAs owns one worker's rows of SL channels (each CTA an
// eighth of the rows), sums over its rows, adds the eight sums through distributed shared memory (in double, in rank order), and goes
// over the same rows again, now out of L2.  The streamed kernels of kernels.cu are built for tensors that do not fit: 96 KB rings, two or
// three launches, a handful of CTAs here; on 18 samples of 4x4x512 they took 8 + 5 + 4 us forward and 6 + 11 us backward for 300 KB.
// A thread keeps 8 consecutive channels (16-byte accesses) for every row it visits, four rows in flight.
struct BncArgs {
    const bf16* x; const bf16* out; const bf16* dout; const bf16* res;
    const float* gamma; const float* beta;
    float* stats;                                // [worker][C][2] (mean, invstd)
    float* red;                                  // backward: [worker][C][2] (sum dy, sum dy xhat)
    bf16* y; bf16* dres; int accum_dx, accum_dres;   // backward: y = dx, or nullptr (not needed)
    int rpw, C, relu, mask_from_x;
};
constexpr int BNC_RANKS = 8;

__device__ __forceinline__ void unpack(const uint4& v, float (&f)[8]) {
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int j = 0; j < 4; ++j) { f[2 * j] = __uint_as_float(w[j] << 16); f[2 * j + 1] = __uint_as_float(w[j] & 0xffff0000u); }
}
__device__ __forceinline__ uint4 pack(const float (&f)[8]) {
    uint32_t w[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) { const __nv_bfloat162 t = __floats2bfloat162_rn(f[2 * j], f[2 * j + 1]); w[j] = *(const uint32_t*)&t; }
    return make_uint4(w[0], w[1], w[2], w[3]);
}
// the streamed kernels' expression (bn_pair), so that a ReLU mask recomputed from x is the forward pass's whichever kernels ran
__device__ __forceinline__ float bn_plain(float x, float mean, float istd, float gamma, float beta) {
    return __fmaf_rn(gamma, __fmul_rn(__fsub_rn(x, mean), istd), beta);
}

template <int SL, bool BWD>
__global__ void __launch_bounds__(BT) bnc_kernel(const BncArgs a) {
    constexpr int L = SL / 8, R = BT / L;        // threads per row, rows per pass
    __shared__ float wsum[BT / 32][SL][2];
    __shared__ double2 cta[SL];
    __shared__ float2 tot[SL];                   // forward: (mean, invstd); backward: (sum dy, sum dy (x - mean)) / rows
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, cl = tid % L, rl = tid / L;
    uint32_t rank; asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
    const int c0 = (blockIdx.x / BNC_RANKS) * SL, w = blockIdx.y, C = a.C;
    const int per = (a.rpw + BNC_RANKS - 1) / BNC_RANKS, r0 = (int)rank * per, r1 = min(a.rpw, r0 + per);
    const size_t base = (size_t)w * a.rpw * C + c0 + cl * 8;
    float mean[8], istd[8], ga[8], be[8], s1[8], s2[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        const int c = c0 + cl * 8 + j;
        ga[j] = a.gamma[c]; be[j] = a.beta[c]; s1[j] = s2[j] = 0.f;
        if (BWD) { const float2 st = *(const float2*)(a.stats + ((size_t)w * C + c) * 2); mean[j] = st.x; istd[j] = st.y; }
    }
    constexpr int U = 4;
    const bool need_out = BWD && a.relu && !a.mask_from_x;
    // dy with the ReLU's mask applied; d = x - mean
    auto masked = [&](const uint4& xv, const uint4& dv, const uint4& ov, float (&d)[8], float (&dy)[8]) {
        float o[8];
        unpack(xv, d); unpack(dv, dy);
        if (need_out) unpack(ov, o);
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            if (a.relu && !((need_out ? o[j] : bn_plain(d[j], mean[j], istd[j], ga[j], be[j])) > 0.f)) dy[j] = 0.f;
            d[j] = __fsub_rn(d[j], mean[j]);
        }
    };
    for (int r = r0 + rl; r < r1; r += R * U) {
        uint4 xv[U], dv[U], ov[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int rr = r + u * R;
            if (rr >= r1) continue;
            const size_t o = base + (size_t)rr * C;
            xv[u] = *(const uint4*)(a.x + o);
            if (BWD) { dv[u] = *(const uint4*)(a.dout + o); if (need_out) ov[u] = *(const uint4*)(a.out + o); }
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (r + u * R >= r1) continue;
            float f[8];
            if (!BWD) {
                unpack(xv[u], f);
#pragma unroll
                for (int j = 0; j < 8; ++j) { s1[j] += f[j]; s2[j] = fmaf(f[j], f[j], s2[j]); }
            } else {
                float dy[8];
                masked(xv[u], dv[u], ov[u], f, dy);
#pragma unroll
                for (int j = 0; j < 8; ++j) { s1[j] += dy[j]; s2[j] = fmaf(dy[j], f[j], s2[j]); }
            }
        }
    }
    // over the rows: lanes of equal channels, warps, CTAs of the cluster, each in a fixed order
#pragma unroll
    for (int d = L; d < 32; d <<= 1)
#pragma unroll
        for (int j = 0; j < 8; ++j) { s1[j] += __shfl_xor_sync(0xffffffffu, s1[j], d); s2[j] += __shfl_xor_sync(0xffffffffu, s2[j], d); }
    if (lane < L)
#pragma unroll
        for (int j = 0; j < 8; ++j) { wsum[warp][lane * 8 + j][0] = s1[j]; wsum[warp][lane * 8 + j][1] = s2[j]; }
    __syncthreads();
    if (tid < SL) {
        double2 t = make_double2(0.0, 0.0);
#pragma unroll
        for (int q = 0; q < BT / 32; ++q) { t.x += (double)wsum[q][tid][0]; t.y += (double)wsum[q][tid][1]; }
        cta[tid] = t;
    }
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
    if (tid < SL) {
        const uint32_t mine = (uint32_t)__cvta_generic_to_shared(&cta[tid]);
        double x[BNC_RANKS], y[BNC_RANKS];
#pragma unroll
        for (int q = 0; q < BNC_RANKS; ++q) {
            uint32_t src;
            asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(src) : "r"(mine), "r"(q));
            asm volatile("ld.shared::cluster.v2.f64 {%0, %1}, [%2];" : "=d"(x[q]), "=d"(y[q]) : "r"(src) : "memory");
        }
        double tx = 0.0, ty = 0.0;
#pragma unroll
        for (int q = 0; q < BNC_RANKS; ++q) { tx += x[q]; ty += y[q]; }
        const size_t so = ((size_t)w * C + c0 + tid) * 2;
        if (!BWD) {
            const double m = tx / a.rpw;
            double var = ty / a.rpw - m * m;
            if (var < 0.0) var = 0.0;
            tot[tid] = make_float2((float)m, (float)(1.0 / sqrt(var + 1e-5)));
            if (rank == 0) *(float2*)(a.stats + so) = tot[tid];
        } else {
            const double is = (double)a.stats[so + 1];
            if (rank == 0) *(float2*)(a.red + so) = make_float2((float)tx, (float)(ty * is));
            tot[tid] = make_float2((float)(tx / a.rpw), (float)(ty * is / a.rpw));
        }
    }
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");      // this CTA has read its neighbours' sums
    __syncthreads();
    float sc[8], ka[8], kb[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        const float2 t = tot[cl * 8 + j];
        if (!BWD) { mean[j] = t.x; istd[j] = t.y; }
        else { sc[j] = ga[j] * istd[j]; ka[j] = -sc[j] * istd[j] * t.y; kb[j] = -sc[j] * t.x; }      // dx = sc dy + (d ka + kb)
    }
    for (int r = r0 + rl; r < r1; r += R * U) {
        uint4 xv[U], dv[U], ov[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int rr = r + u * R;
            if (rr >= r1) continue;
            const size_t o = base + (size_t)rr * C;
            xv[u] = *(const uint4*)(a.x + o);
            if (BWD) { dv[u] = *(const uint4*)(a.dout + o); if (need_out) ov[u] = *(const uint4*)(a.out + o); }
            else if (a.res) ov[u] = *(const uint4*)(a.res + o);
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int rr = r + u * R;
            if (rr >= r1) continue;
            const size_t o = base + (size_t)rr * C;
            float f[8], g[8];
            if (!BWD) {
                unpack(xv[u], f);
                if (a.res) unpack(ov[u], g);
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    f[j] = bn_plain(f[j], mean[j], istd[j], ga[j], be[j]);
                    if (a.res) f[j] += g[j];
                    if (a.relu) f[j] = fmaxf(f[j], 0.f);
                }
                *(uint4*)(a.y + o) = pack(f);
            } else {
                masked(xv[u], dv[u], ov[u], f, g);
                if (a.y) {                           // none for the network's input
#pragma unroll
                    for (int j = 0; j < 8; ++j) f[j] = fmaf(sc[j], g[j], fmaf(f[j], ka[j], kb[j]));
                    if (a.accum_dx) {
                        float old[8];
                        unpack(*(const uint4*)(a.y + o), old);
#pragma unroll
                        for (int j = 0; j < 8; ++j) f[j] += old[j];
                    }
                    *(uint4*)(a.y + o) = pack(f);
                }
                if (a.dres) {
                    if (a.accum_dres) {
                        float old[8];
                        unpack(*(const uint4*)(a.dres + o), old);
#pragma unroll
                        for (int j = 0; j < 8; ++j) g[j] += old[j];
                    }
                    *(uint4*)(a.dres + o) = pack(g);
                }
            }
        }
    }
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");         // none of the neighbours reads this CTA's sums any more
}
// dbeta, dgamma = sums over the workers (ascending)
__global__ void __launch_bounds__(128) bnc_params_k(const float* __restrict__ red, float* __restrict__ dgamma, float* __restrict__ dbeta, int nw, int C) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= C) return;
    float g = 0.f, b = 0.f;
    for (int w = 0; w < nw; ++w) { const float2 v = *(const float2*)(red + ((size_t)w * C + c) * 2); b += v.x; g += v.y; }
    dgamma[c] = g; dbeta[c] = b;
}

// Three CTAs per SM over all workers, at least four rows per thread.
int bnf_chunks(int nw, long rpw, int C) {
    const long rows_it = BT / (C / 4), want = (3 * 148 + nw - 1) / nw, maxc = (rpw + rows_it * 4 - 1) / (rows_it * 4);
    long c = want < maxc ? want : maxc;
    if (c > BNF_MAX_CHUNKS) c = BNF_MAX_CHUNKS;
    return (int)(c < 1 ? 1 : c);
}

}  // namespace

template <bool BWD>
static void bnc_launch(const BncArgs& a, int nw, int nw_all, int modules, cudaStream_t s) {
    // channels per cluster: 64 (whole 128-byte lines), fewer where that makes less than 25 CTAs: many small CTAs end one launch sooner, but the SMs are
    // wanted by the other modules (18 samples, 4 modules: 386 us per step with this line, 432 with 100 CTAs; by the number of ALL workers: a launch for
    // a group of them adds in the same order).
    // Long columns, more than 20 rows a thread: fewer until no SM is without a CTA, if the SMs are free for it.  With one module they are (us per step, left without):
    // ResNet-18 2 x 12 931 (958), 4 x 6 904 (965), ResNet-20 4 x 48 1164 (1234).  With two, the other one's convolutions leave room on their SMs
    // if they are those of mconv.cu, which is where channels are no multiple of 64 (ResNet-20 4 x 48 828 (849), 4 x 42 779 (792)), not if a
    // CTA of theirs fills an SM (ResNet-18 2 x 12 553 (540)); with more modules somebody wants them (ResNet-20 4 x 48 K=3 765 (756), K=4 774 (755), ResNet-18 K=4 2 x 12
    // 425 (406), 1 x 48 528 (514), 4 x 6 464 (444)).  Up to 20 rows a launch is short enough as it is (2 x 9, 18 rows: 378 (377)).
    int sl = 64;
    const bool room = modules == 1 || (modules == 2 && a.C % 64 != 0);
    const auto ctas = [&] { return (a.C / sl) * nw_all * BNC_RANKS; };
    const auto long_columns = [&] { return (long)(a.rpw + BNC_RANKS - 1) / BNC_RANKS * (sl / 8) > 20L * BT; };
    while (sl > 16 && (a.C % sl || ctas() < 25 || (room && long_columns() && ctas() < 148))) sl /= 2;
    const dim3 grid((a.C / sl) * BNC_RANKS, nw);
    if (sl == 64) klaunch_cluster(bnc_kernel<64, BWD>, grid, BT, 0, s, BNC_RANKS, a);
    else if (sl == 32) klaunch_cluster(bnc_kernel<32, BWD>, grid, BT, 0, s, BNC_RANKS, a);
    else klaunch_cluster(bnc_kernel<16, BWD>, grid, BT, 0, s, BNC_RANKS, a);
}
// Tensors up to 4 MB: read twice out of L2 (beyond that the streamed kernels' rate counts, not the launches: 4 workers x 16, 693 us per step with the
// line at 4 MB, 729 at 8 MB, 820 at 17 MB), and few enough rows per thread for plain fp32 sums (at most 16 384 / 8 / 32 = 64).
bool bnc_supported(int dt, int nw, long rpw, int C) { return dt == 1 && C % 16 == 0 && rpw <= 16384 && (double)nw * rpw * C * 2.0 <= 4e6; }
void bnc_forward(const void* x, const float* gamma, const float* beta, const void* res, void* y, float* stats, int nw, int nw_all, int modules, long rpw, int C, bool relu,
                 cudaStream_t s) {
    BncArgs a{};
    a.x = (const bf16*)x; a.gamma = gamma; a.beta = beta; a.res = (const bf16*)res; a.y = (bf16*)y; a.stats = stats; a.rpw = (int)rpw; a.C = C; a.relu = relu;
    Scope sc(KC_BN_FWD_APPLY, 0.0, 2.0 * nw * rpw * C * (res ? 3 : 2), s);
    bnc_launch<false>(a, nw, nw_all, modules, s);
}
void bnc_backward(const void* x, const void* out, const void* dout, const float* gamma, const float* beta, const float* stats, void* dx, bool accum_dx, void* dres,
                  bool accum_dres, float* red, int nw, int nw_all, int modules, long rpw, int C, bool relu, bool has_res, cudaStream_t s) {
    BncArgs a{};
    a.x = (const bf16*)x; a.out = (const bf16*)out; a.dout = (const bf16*)dout; a.gamma = gamma; a.beta = beta; a.stats = (float*)stats; a.y = (bf16*)dx;
    a.accum_dx = accum_dx; a.dres = (bf16*)dres; a.accum_dres = accum_dres; a.red = red; a.rpw = (int)rpw; a.C = C; a.relu = relu; a.mask_from_x = relu && !has_res;
    Scope sc(KC_BN_BWD_APPLY, 0.0, 2.0 * nw * rpw * C * (3 + (relu && has_res ? 1 : 0) + (accum_dx ? 1 : 0) + (dres ? (accum_dres ? 2 : 1) : 0)), s);
    bnc_launch<true>(a, nw, nw_all, modules, s);
}
void bnc_params(const float* red, float* dgamma, float* dbeta, int nw, int C, cudaStream_t s) {
    Scope sc(KC_BN_BWD_REDUCE, 0.0, 8.0 * nw * C, s);
    klaunch(bnc_params_k, (C + 127) / 128, 128, 0, s, red, dgamma, dbeta, nw, C);
}

bool bnf_supported(int dt, int C) { return dt == 0 && C % 4 == 0 && C / 4 <= BT && ((C / 4) & (C / 4 - 1)) == 0; }

void bn_merge_tiles(const float* tile_part, float* stats, int tiles, int nw, long rpw, int C, cudaStream_t s) {
    int nc = 1;                                  // channels per block: a power of two that divides C
    while (nc < 64 && C % (2 * nc) == 0) nc *= 2;
    Scope sc(KC_BN_FWD_STATS, 0.0, 8.0 * tiles * nw * C, s);
    klaunch(bn_merge_tiles_k, dim3(C / nc, nw), BT, 0, s, tile_part, stats, tiles, C, nc, rpw);
}

void bnf_forward(const float* x, const float* gamma, const float* beta, size_t p_group, const float* res, float* y, float* stats, const float* tile_part,
                 int tiles, int nw, long rpw, int C, bool relu, cudaStream_t s) {
    BnfArgs a{};
    a.x = x; a.gamma = gamma; a.beta = beta; a.p_group = p_group; a.res = res; a.y = y; a.stats = stats; a.tile_part = tile_part; a.tiles = tiles;
    a.rpw = rpw; a.C = C; a.relu = relu;
    Scope sc(KC_BN_FWD_APPLY, 0.0, 4.0 * nw * rpw * C * (res ? 3 : 2), s);
    klaunch(bnf_kernel<0>, dim3(bnf_chunks(nw, rpw, C), nw), BT, 0, s, a);
}

void bnf_backward(const float* x, const float* out, const float* dout, const float* gamma, const float* beta, size_t p_group, const float* stats, float* dx,
                  bool accum_dx, float* dres, bool accum_dres, float* dgamma, float* dbeta, size_t g_group, float* scratch, int nw, long rpw, int C, bool relu,
                  bool mask_from_x, bool accum_params, cudaStream_t s) {
    BnfArgs a{};
    a.x = x; a.out = out; a.dout = dout; a.gamma = gamma; a.beta = beta; a.p_group = p_group; a.stats = (float*)stats; a.y = dx; a.accum_dx = accum_dx;
    a.dres = dres; a.accum_dres = accum_dres; a.dgamma = dgamma; a.dbeta = dbeta; a.g_group = g_group; a.accum_params = accum_params; a.part = scratch;
    a.rpw = rpw; a.C = C; a.relu = relu; a.mask_from_x = mask_from_x;
    const dim3 grid(bnf_chunks(nw, rpw, C), nw);
    const double total = (double)nw * rpw * C;
    const int reads = 2 + (relu && !mask_from_x ? 1 : 0);
    { Scope sc(KC_BN_BWD_REDUCE, 0.0, 4.0 * total * reads, s);
      klaunch(bnf_kernel<1>, grid, BT, 0, s, a); }
    Scope sc(KC_BN_BWD_APPLY, 0.0, 4.0 * total * (reads + 1 + (accum_dx ? 1 : 0) + (dres ? (accum_dres ? 2 : 1) : 0)), s);
    klaunch(bnf_kernel<2>, grid, BT, 0, s, a);
}

}  // namespace fdg
