// Linear layers on the CUDA cores (fp32 arithmetic, fp32 or bf16 storage): the whole fp32 path and, with bf16 storage, widths that are
// no multiple of 64.  Any sizes.
//   forward  : one launch, y = x W^T (+ b) (relu).
//   backward : one launch: dx (+)= dy W and dW (+)= dy^T x, db (+)= column sums of dy; the ReLU mask dy * [y > 0] is applied while dy is
//              read, so that there is no pass of its own for it, for the bias gradient or for either gradient matrix.
//
// What bounds these layers is latency, not arithmetic: 64 samples through 3072 -> 512 are 0.2 GFLOP, and the kernels they replace took
// two launches each with serial chains of up to 3072 / 16 slices or a few CTAs (62 us for the input gradient of 512 -> 256 on 64
// samples).  So: 32 x 64 tiles of 128 threads, and a forward or input-gradient tile is split over the contraction among the CTAs of a
// cluster, which add their partial tiles through distributed shared memory in rank order: no workspace, no second launch.  A
// weight-gradient tile contracts over the samples; the CTAs of a cluster take tiles of their own.  From 1024 samples on that chain
// is split over CTAs that leave partial matrices in a workspace, and a second launch (off the chain of the backward pass) adds them.
// Arithmetic as in fconv.cu: packed FMAs with the pairs along the contraction, chains of at most 16 products into a compensated sum.
#include "kernels.h"
#include "launch.h"

#include <cuda_bf16.h>

namespace fdg {

typedef __nv_bfloat16 bf16;

namespace {

constexpr int LT = 128, LM = 32, LN = 64, LK = 32;
constexpr int LP = 36;                   // floats per row of a 32-wide chunk: rows fall into different banks for 16-byte reads

__device__ __forceinline__ float to_f(float v) { return v; }
__device__ __forceinline__ float to_f(bf16 v) { return __bfloat162float(v); }
__device__ __forceinline__ void put(float* p, float v) { *p = v; }
__device__ __forceinline__ void put(bf16* p, float v) { *p = __float2bfloat16_rn(v); }
__device__ __forceinline__ float4 ld4(const float* p) { return *(const float4*)p; }
__device__ __forceinline__ float4 ld4(const bf16* p) {
    const uint2 v = *(const uint2*)p;
    return make_float4(__uint_as_float(v.x << 16), __uint_as_float(v.x & 0xffff0000u), __uint_as_float(v.y << 16), __uint_as_float(v.y & 0xffff0000u));
}

// Four consecutive elements of row r (columns c .. c + 3) of a row-major matrix, zero outside rows x cols.
template <typename T>
__device__ __forceinline__ float4 fetch4(const T* __restrict__ p, int r, int c, int rows, int cols, bool vec) {
    if (r >= rows || c >= cols) return make_float4(0.f, 0.f, 0.f, 0.f);
    const T* s = p + (size_t)r * cols + c;
    if (vec) return ld4(s);              // cols is a multiple of 4 and the matrix starts on a 4-element boundary
    return make_float4(to_f(s[0]), c + 1 < cols ? to_f(s[1]) : 0.f, c + 2 < cols ? to_f(s[2]) : 0.f, c + 3 < cols ? to_f(s[3]) : 0.f);
}
__device__ __forceinline__ float4 masked(float4 d, float4 y) { return make_float4(y.x > 0.f ? d.x : 0.f, y.y > 0.f ? d.y : 0.f, y.z > 0.f ? d.z : 0.f, y.w > 0.f ? d.w : 0.f); }

struct LinArgs {
    const void* x; const void* w; const void* dy; const void* y;     // [M][K], [N][K], [M][N], [M][N] (y: mask of the backward pass, or nullptr)
    const float* bias;
    void* out;                           // forward: y [M][N]; backward: dx [M][K] or nullptr
    float* dw; float* db;
    int M, N, K, epi, accum_p;
    int vec_k, vec_n;                    // rows of length K / N can be read 4 elements at a time
    int split;                           // CTAs per cluster
    int dx_clusters, dx_tiles_n, dw_tiles_n, dw_tiles;
    int dw_splits; float* part;          // > 1: every dW tile in this many parts of the samples, to part: [group][split][N * K, then N sums of db]
    size_t w_group, b_group, g_group;    // grid.y groups of M samples each: elements between their weights, biases, parameter gradients
};

// the arguments of group blockIdx.y
template <typename T>
__device__ __forceinline__ LinArgs of_group(const LinArgs& in, bool fwd) {
    LinArgs a = in;
    const size_t g = blockIdx.y, mk = g * a.M * a.K, mn = g * a.M * a.N;
    a.x = (const T*)a.x + mk; a.w = (const T*)a.w + g * a.w_group;
    if (a.dy) a.dy = (const T*)a.dy + mn;
    if (a.y) a.y = (const T*)a.y + mn;
    if (a.bias) a.bias += g * a.b_group;
    if (a.out) a.out = (a.epi & EPI_OUT_F32) ? (void*)((float*)a.out + mn) : (void*)((T*)a.out + (fwd ? mn : mk));
    if (a.dw) a.dw += g * a.g_group;
    if (a.db) a.db += g * a.g_group;
    if (a.part) a.part += g * a.dw_splits * ((size_t)a.N * a.K + a.N);
    return a;
}

enum { L_FWD, L_DX, L_DW };

// What a CTA hands on of its part of a contraction.  fp32 storage: both lanes' compensated sums together, in double, so that neither the lanes nor the
// split cost precision (with parts rounded to fp32 the error of 512 samples through 500 -> 300 was 9 % above that of an unsplit sum).  bf16 storage: fp32, the
// lanes added at every flush; the rounded result hides the difference, and the sums in double take 3 % of a small network's step.
template <typename T> struct Part { typedef float type; };
template <> struct Part<float> { typedef double type; };

// One 32 x 64 tile over the contraction range [k0, k1).  Operands in shared memory as [row][contraction], double buffered; the next
// chunk travels in registers while this one is used.
template <typename T, int MODE>
__device__ __forceinline__ void tile_product(const LinArgs& a, int row0, int col0, int k0, int k1, float* sm, typename Part<T>::type (&out)[4][4], float* bias_sum) {
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane & 7, cg = lane >> 3;
    constexpr bool LANES = sizeof(T) == 4;
    float2 acc[4][4], part[4][4];            // LANES: per output even and odd products; else per pair of outputs their sums (0, 1), what these have lost (2, 3)
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = part[i][j] = make_float2(0.f, 0.f);
    float4 ra[2], rb[4];
    const T* const X = (const T*)a.x; const T* const W = (const T*)a.w; const T* const DY = (const T*)a.dy; const T* const Y = (const T*)a.y;
    // column n of the tile sits in row (n / 16) * 16 + (n % 4) * 4 + (n % 16) / 4 of the B tile: a warp's four channel groups read neighbours
    auto brow = [](int n) { return (n & ~15) + (n & 3) * 4 + ((n & 15) >> 2); };
    auto fetch = [&](int kc) {
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int i = tid + u * LT;
            if (MODE == L_FWD) ra[u] = fetch4(X, row0 + (i >> 3), kc + 4 * (i & 7), a.M, a.K, a.vec_k);
            else if (MODE == L_DX) {
                ra[u] = fetch4(DY, row0 + (i >> 3), kc + 4 * (i & 7), a.M, a.N, a.vec_n);
                if (Y) ra[u] = masked(ra[u], fetch4(Y, row0 + (i >> 3), kc + 4 * (i & 7), a.M, a.N, a.vec_n));
            } else {                     // sample i >> 3, four output features
                ra[u] = fetch4(DY, kc + (i >> 3), row0 + 4 * (i & 7), a.M, a.N, a.vec_n);
                if (Y) ra[u] = masked(ra[u], fetch4(Y, kc + (i >> 3), row0 + 4 * (i & 7), a.M, a.N, a.vec_n));
            }
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int i = tid + u * LT;
            if (MODE == L_FWD) rb[u] = fetch4(W, col0 + (i >> 3), kc + 4 * (i & 7), a.N, a.K, a.vec_k);
            else if (MODE == L_DX) rb[u] = fetch4(W, kc + (i >> 4), col0 + 4 * (i & 15), a.N, a.K, a.vec_k);
            else rb[u] = fetch4(X, kc + (i >> 4), col0 + 4 * (i & 15), a.M, a.K, a.vec_k);
        }
    };
    // what lies past k1 belongs to another CTA of the cluster (ranges are multiples of LK except the last, which ends with the matrix)
    auto stash = [&](float* A, float* B) {
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int i = tid + u * LT;
            if (MODE != L_DW) *(float4*)(A + (i >> 3) * LP + 4 * (i & 7)) = ra[u];
            else {
                const float v[4] = {ra[u].x, ra[u].y, ra[u].z, ra[u].w};
#pragma unroll
                for (int e = 0; e < 4; ++e) A[(4 * (i & 7) + e) * LP + (i >> 3)] = v[e];
            }
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int i = tid + u * LT;
            if (MODE == L_FWD) *(float4*)(B + brow(i >> 3) * LP + 4 * (i & 7)) = rb[u];
            else {
                const float v[4] = {rb[u].x, rb[u].y, rb[u].z, rb[u].w};
#pragma unroll
                for (int e = 0; e < 4; ++e) B[brow(4 * (i & 15) + e) * LP + (i >> 4)] = v[e];
            }
        }
    };
    constexpr int BUF = (LM + LN) * LP;
    const int chunks = k1 > k0 ? (k1 - k0 + LK - 1) / LK : 0;
    if (chunks) fetch(k0);
    float bsum = 0.f;
    for (int c = 0; c < chunks; ++c) {
        float* const A = sm + (c & 1) * BUF;
        float* const B = A + LM * LP;
        stash(A, B);
        __syncthreads();                 // the other buffer's readers of chunk c - 1 have all passed here before chunk c + 1 overwrites it
        if (c + 1 < chunks) fetch(k0 + (c + 1) * LK);
        const float* const pa = A + g * LP;
        const float* const pb = B + (warp * 16 + cg) * LP;
#pragma unroll
        for (int q = 0; q < LK / 4; ++q) {
            float4 wv[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) wv[j] = *(const float4*)(pb + j * (4 * LP) + 4 * q);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float4 xv = *(const float4*)(pa + i * (8 * LP) + 4 * q);
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const float2 lo = make_float2(xv.x, xv.y), hi = make_float2(xv.z, xv.w);
                    if (!LANES && q == 0) part[i][j] = __fmul2_rn(lo, make_float2(wv[j].x, wv[j].y));
                    else part[i][j] = __ffma2_rn(lo, make_float2(wv[j].x, wv[j].y), part[i][j]);
                    part[i][j] = __ffma2_rn(hi, make_float2(wv[j].z, wv[j].w), part[i][j]);
                }
            }
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {                // Kahan
            if (LANES) {
#pragma unroll
                for (int j = 0; j < 4; ++j) {        // the next chain starts at what the sum lost
                    const float2 t = __fadd2_rn(acc[i][j], part[i][j]);
                    const float2 d = __fadd2_rn(t, make_float2(-acc[i][j].x, -acc[i][j].y));
                    part[i][j] = __fadd2_rn(part[i][j], make_float2(-d.x, -d.y));
                    acc[i][j] = t;
                }
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
        if (MODE == L_DW && bias_sum && tid < LM) {
            float s = 0.f;
#pragma unroll
            for (int k = 0; k < LK; ++k) s += A[tid * LP + k];
            bsum += s;
        }
    }
    if (MODE == L_DW && bias_sum) *bias_sum = bsum;
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            if (LANES) out[i][j] = (typename Part<T>::type)(((double)acc[i][j].x + (double)acc[i][j].y) + ((double)part[i][j].x + (double)part[i][j].y));    // part: what the lanes have lost
            else out[i][j] = j & 1 ? acc[i][j >> 1].y : acc[i][j >> 1].x;
        }
}

__device__ __forceinline__ uint32_t ctarank() { uint32_t r; asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r)); return r; }
__device__ __forceinline__ void cluster_sync() { asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ void st_part(float* d, const float (&v)[4]) { *(float4*)d = make_float4(v[0], v[1], v[2], v[3]); }
__device__ __forceinline__ void st_part(double* d, const double (&v)[4]) { *(double2*)d = make_double2(v[0], v[1]); *(double2*)(d + 2) = make_double2(v[2], v[3]); }
// four consecutive parts of another CTA of the cluster
__device__ __forceinline__ void ld_cluster(uint32_t local, uint32_t rank, float (&v)[4]) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(local), "r"(rank));
    asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]) : "r"(r) : "memory");
}
__device__ __forceinline__ void ld_cluster(uint32_t local, uint32_t rank, double (&v)[4]) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(local), "r"(rank));
    asm volatile("ld.shared::cluster.v2.f64 {%0, %1}, [%2];" : "=d"(v[0]), "=d"(v[1]) : "r"(r) : "memory");
    asm volatile("ld.shared::cluster.v2.f64 {%0, %1}, [%2];" : "=d"(v[2]), "=d"(v[3]) : "r"(r + 16) : "memory");
}

// Four consecutive outputs of one row: bias, ReLU, accumulation, store (T, or fp32 with EPI_OUT_F32).
template <typename T>
__device__ __forceinline__ void emit(const LinArgs& a, int r, int c, int rows, int cols, float (&v)[4], const float* bias) {
    if (r >= rows) return;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        if (c + j >= cols) continue;
        const size_t o = (size_t)r * cols + c + j;
        float t = v[j];
        if (bias) t += bias[c + j];
        if (a.epi & EPI_RELU) t = fmaxf(t, 0.f);
        if (a.epi & EPI_OUT_F32) ((float*)a.out)[o] = t;
        else {
            T* const d = (T*)a.out + o;
            if (a.epi & EPI_ACCUM) t += to_f(*d);
            put(d, t);
        }
    }
}

// A tile that the cluster's CTAs have each done a part of: CTA `rank` adds rows rank, rank + split, ... over the CTAs in rank order.
template <typename T>
__device__ __forceinline__ void join_tile(const LinArgs& a, int row0, int col0, int rows, int cols, typename Part<T>::type (&v)[4][4], const float* bias, float* sm) {
    typedef typename Part<T>::type P;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane & 7, cg = lane >> 3;
    if (a.split == 1) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            float f[4] = {(float)v[i][0], (float)v[i][1], (float)v[i][2], (float)v[i][3]};
            emit<T>(a, row0 + g + 8 * i, col0 + warp * 16 + 4 * cg, rows, cols, f, bias);
        }
        return;
    }
    __syncthreads();                     // the operand buffers are no longer read
    constexpr int TP = LN + 16 / (int)sizeof(P);
    static_assert(LM * TP * sizeof(P) <= 2 * (LM + LN) * LP * sizeof(float), "the parts reuse the operand buffers");
    P* const part = (P*)sm;
#pragma unroll
    for (int i = 0; i < 4; ++i) st_part(part + (g + 8 * i) * TP + warp * 16 + 4 * cg, v[i]);
    cluster_sync();
    const uint32_t base = (uint32_t)__cvta_generic_to_shared(sm);
    const int rank = (int)ctarank();
    for (int e = tid; e < LM * LN / 4 / a.split; e += LT) {
        const int r = (e / (LN / 4)) * a.split + rank, c = 4 * (e % (LN / 4));
        const uint32_t at = base + (uint32_t)((r * TP + c) * sizeof(P));
        P s[4] = {0, 0, 0, 0};
        for (int q = 0; q < a.split; q += 2) {       // split is a power of two; two CTAs' parts in flight
            P t[2][4];
            ld_cluster(at, q, t[0]);
            ld_cluster(at, q + 1, t[1]);
#pragma unroll
            for (int u = 0; u < 2; ++u)
#pragma unroll
                for (int j = 0; j < 4; ++j) s[j] += t[u][j];
        }
        float f[4] = {(float)s[0], (float)s[1], (float)s[2], (float)s[3]};
        emit<T>(a, row0 + r, col0 + c, rows, cols, f, bias);
    }
    cluster_sync();                      // no CTA leaves while another reads its tile
}

__device__ __forceinline__ void my_range(int K, int split, int rank, int& k0, int& k1) {
    const int per = ((K + split - 1) / split + LK - 1) / LK * LK;
    k0 = min(K, rank * per); k1 = min(K, k0 + per);
}

// grid = column tiles x row tiles x split (the cluster) along x
template <typename T>
__global__ void __launch_bounds__(LT) lin_fwd_kernel(const LinArgs args) {
    const LinArgs a = of_group<T>(args, true);
    __shared__ __align__(16) float sm[2 * (LM + LN) * LP];
    const int tile = blockIdx.x / a.split, rank = blockIdx.x % a.split;
    const int tiles_n = (a.N + LN - 1) / LN, row0 = tile / tiles_n * LM, col0 = tile % tiles_n * LN;
    int k0, k1; my_range(a.K, a.split, rank, k0, k1);
    typename Part<T>::type v[4][4];
    tile_product<T, L_FWD>(a, row0, col0, k0, k1, sm, v, nullptr);
    join_tile<T>(a, row0, col0, a.M, a.N, v, a.bias, sm);
}

// The first dx_clusters clusters: input gradient; the others: `split` weight-gradient tiles (or parts of tiles) each.
template <typename T>
__global__ void __launch_bounds__(LT) lin_bwd_kernel(const LinArgs args) {
    const LinArgs a = of_group<T>(args, false);
    __shared__ __align__(16) float sm[2 * (LM + LN) * LP];
    const int cl = blockIdx.x / a.split, rank = blockIdx.x % a.split;
    typename Part<T>::type v[4][4];
    if (cl < a.dx_clusters) {
        const int row0 = cl / a.dx_tiles_n * LM, col0 = cl % a.dx_tiles_n * LN;
        int k0, k1; my_range(a.N, a.split, rank, k0, k1);
        tile_product<T, L_DX>(a, row0, col0, k0, k1, sm, v, nullptr);
        join_tile<T>(a, row0, col0, a.M, a.K, v, nullptr, sm);
        return;
    }
    const int item = (cl - a.dx_clusters) * a.split + rank;
    if (item >= a.dw_tiles * a.dw_splits) return;
    const int tile = item % a.dw_tiles, sp = item / a.dw_tiles;
    const int row0 = tile / a.dw_tiles_n * LM, col0 = tile % a.dw_tiles_n * LN;
    float* dw = a.dw; float* db = a.db;
    int s0 = 0, s1 = a.M, accum = a.accum_p;
    if (a.dw_splits > 1) {
        my_range(a.M, a.dw_splits, sp, s0, s1);
        dw = a.part + sp * ((size_t)a.N * a.K + a.N); accum = 0;
        if (db) db = dw + (size_t)a.N * a.K;
    }
    float bs = 0.f;
    tile_product<T, L_DW>(a, row0, col0, s0, s1, sm, v, db && col0 == 0 ? &bs : nullptr);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane & 7, cg = lane >> 3;
    const int c = col0 + warp * 16 + 4 * cg;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int r = row0 + g + 8 * i;
        if (r >= a.N || c >= a.K) continue;
        float* const d = dw + (size_t)r * a.K + c;
        if ((a.K & 3) == 0 && (((uintptr_t)dw) & 15) == 0) {
            float4 o = make_float4((float)v[i][0], (float)v[i][1], (float)v[i][2], (float)v[i][3]);
            if (accum) { const float4 old = *(const float4*)d; o.x += old.x; o.y += old.y; o.z += old.z; o.w += old.w; }
            *(float4*)d = o;
        } else {
#pragma unroll
            for (int j = 0; j < 4; ++j) if (c + j < a.K) d[j] = accum ? d[j] + (float)v[i][j] : (float)v[i][j];
        }
    }
    if (db && col0 == 0 && tid < LM && row0 + tid < a.N) db[row0 + tid] = accum ? db[row0 + tid] + bs : bs;
}

// dW and db from the partial matrices: 32 elements per CTA, eight threads of different splits per element, four loads in flight each, then their
// sums in order, in double.
__global__ void __launch_bounds__(256) lin_reduce_kernel(const float* __restrict__ part, float* __restrict__ dw, float* __restrict__ db, int splits, size_t nk, int N,
                                                         size_t g_group, bool accum) {
    __shared__ double sh[8][32];
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    const size_t e = (size_t)blockIdx.x * 32 + tx, n = nk + N;
    const float* const src = part + blockIdx.y * (splits * n) + e;
    double s = 0.0;
    if (e < n) {
        int k = ty;
        for (; k + 24 < splits; k += 32) {
            float v[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) v[u] = src[(size_t)(k + 8 * u) * n];
#pragma unroll
            for (int u = 0; u < 4; ++u) s += (double)v[u];
        }
        for (; k < splits; k += 8) s += (double)src[(size_t)k * n];
    }
    sh[ty][tx] = s;
    __syncthreads();
    if (ty != 0 || e >= n || (e >= nk && !db)) return;
#pragma unroll
    for (int k = 1; k < 8; ++k) s += sh[k][tx];
    float* const d = (e < nk ? dw + e : db + (e - nk)) + blockIdx.y * g_group;
    *d = accum ? *d + (float)s : (float)s;
}

// CTAs per cluster: as many as fill the device once (148 SMs, four CTAs each take the latency), a power of two up to 8 (the portable
// cluster size), with at least two chunks of the contraction each.
int pick_split(int tiles, int contraction) {
    int s = 1;
    while (s < 8 && tiles * s * 2 <= 148 * 2 && contraction >= s * 2 * 2 * LK) s *= 2;
    return s;
}
// Parts of a weight-gradient tile's samples: at least DW_CHUNKS chunks each, and no more CTAs than four per SM.  Without them 16 x 1024 samples of
// a 70-33-65-17-5 network took 2565 us per step (the implicit GEMM that these kernels replaced 385), 784-64-32-10 1100 (380), bf16 4352 (397) and 1670
// (394); 8 x 256 samples 344 (210) and 144 (128).  With them 296, 262, 366, 290, 125 and 80.
constexpr int DW_CHUNKS = 16;
int max_dw_splits(int tiles, int samples) {
    const int by_samples = (samples + LK - 1) / LK / DW_CHUNKS, by_ctas = 4 * 148 / tiles, s = by_samples < by_ctas ? by_samples : by_ctas;
    return s < 2 ? 1 : s;
}
int pick_dw_splits(int tiles, int samples) {                          // parts that are not empty
    const int s = max_dw_splits(tiles, samples), per = ((samples + s - 1) / s + LK - 1) / LK * LK;       // as my_range
    return (samples + per - 1) / per;
}
int dw_tile_count(const ConvGeom& g) { return ((g.Co + LM - 1) / LM) * ((g.C + LN - 1) / LN); }
bool aligned4(const void* p, int dt) { return ((uintptr_t)p & (dt ? 7 : 15)) == 0; }

}  // namespace

bool linear_supported(const ConvGeom& g) { return g.H * g.W == 1 && g.R == 1; }
size_t linear_workspace_elems(const ConvGeom& g, int groups) {
    const int s = max_dw_splits(dw_tile_count(g) * groups, g.N / groups);     // a window of the batch has no more
    return s > 1 ? (size_t)groups * s * ((size_t)g.Co * g.C + g.Co) : 0;
}

void linear_forward(int dt, const void* x, const void* w, const float* bias, void* y, const ConvGeom& g, int epi, int groups, size_t w_group, size_t b_group,
                    cudaStream_t s) {
    LinArgs a{};
    a.x = x; a.w = w; a.bias = bias; a.out = y; a.M = g.N / groups; a.N = g.Co; a.K = g.C; a.epi = epi; a.w_group = w_group; a.b_group = b_group;
    a.vec_k = g.C % 4 == 0 && w_group % 4 == 0 && aligned4(x, dt) && aligned4(w, dt);
    const int tiles = ((a.M + LM - 1) / LM) * ((a.N + LN - 1) / LN);
    a.split = pick_split(tiles * groups, a.K);
    const double esz = dt ? 2.0 : 4.0;
    Scope sc(KC_FMA_FWD, 2.0 * g.N * a.N * a.K, esz * ((double)a.M * a.K + (double)a.N * a.K + (double)a.M * a.N), s);
    if (dt) klaunch_cluster(lin_fwd_kernel<bf16>, dim3(tiles * a.split, groups), LT, 0, s, a.split, a);
    else klaunch_cluster(lin_fwd_kernel<float>, dim3(tiles * a.split, groups), LT, 0, s, a.split, a);
}

void linear_backward(int dt, const void* x, const void* w, const void* y_or_null, const void* dy, void* dx_or_null, bool accum_dx, float* dw_or_null, float* db_or_null,
                     const ConvGeom& g, int groups, size_t w_group, size_t g_group, bool accum_p, float* workspace, cudaStream_t s, cudaStream_t s_reduce,
                     cudaEvent_t ready) {
    LinArgs a{};
    a.x = x; a.w = w; a.y = y_or_null; a.dy = dy; a.out = dx_or_null; a.dw = dw_or_null; a.db = db_or_null; a.M = g.N / groups; a.N = g.Co; a.K = g.C;
    a.w_group = w_group; a.g_group = g_group;
    a.epi = accum_dx ? EPI_ACCUM : 0; a.accum_p = accum_p;
    a.vec_k = g.C % 4 == 0 && w_group % 4 == 0 && aligned4(x, dt) && aligned4(w, dt);
    a.vec_n = g.Co % 4 == 0 && aligned4(dy, dt) && (!y_or_null || aligned4(y_or_null, dt));
    a.dx_tiles_n = (a.K + LN - 1) / LN;
    const int dx_tiles = dx_or_null ? ((a.M + LM - 1) / LM) * a.dx_tiles_n : 0;
    a.split = dx_tiles ? pick_split(dx_tiles * groups, a.N) : 1;
    a.dx_clusters = dx_tiles;
    a.dw_tiles_n = (a.K + LN - 1) / LN;
    a.dw_tiles = dw_or_null ? dw_tile_count(g) : 0;
    a.dw_splits = dw_or_null && workspace ? pick_dw_splits(a.dw_tiles * groups, a.M) : 1;
    if (a.dw_splits > 1) a.part = workspace;
    const int clusters = dx_tiles + (a.dw_tiles * a.dw_splits + a.split - 1) / a.split;
    const double esz = dt ? 2.0 : 4.0;
    {
        Scope sc(KC_FMA_WGRAD, (dx_or_null ? 4.0 : 2.0) * g.N * a.N * a.K, esz * ((double)a.M * a.K * (dx_or_null ? 2 : 1) + (double)a.N * a.K + (double)a.M * a.N * (y_or_null ? 2 : 1)) + 4.0 * a.N * a.K, s);
        if (dt) klaunch_cluster(lin_bwd_kernel<bf16>, dim3(clusters * a.split, groups), LT, 0, s, a.split, a);
        else klaunch_cluster(lin_bwd_kernel<float>, dim3(clusters * a.split, groups), LT, 0, s, a.split, a);
    }
    if (a.dw_splits == 1) return;
    const size_t nk = (size_t)a.N * a.K;
    if (s_reduce != s) { step_record(ready, s); step_wait(s_reduce, ready); }
    Scope sc(KC_SPLITK, 0.0, 4.0 * groups * (a.dw_splits + 1) * (nk + a.N), s_reduce);
    klaunch(lin_reduce_kernel, dim3((unsigned)((nk + a.N + 31) / 32), groups), 256, 0, s_reduce, workspace, dw_or_null, db_or_null, a.dw_splits, nk, a.N, g_group, accum_p);
}

}  // namespace fdg
