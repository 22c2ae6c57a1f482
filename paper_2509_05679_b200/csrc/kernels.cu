// Memory-bound and small kernels in fp32 or bf16 storage with fp32 arithmetic: elementwise layers, pooling, streamed batch-norm,
// the classifier head with the loss, column sums, mixing and SGD, input copies; and the profiler all launchers report to.
#include "kernels.h"
#include "launch.h"

#include <cuda_bf16.h>
#include <atomic>
#include <cstdio>
#include <map>
#include <mutex>
#include <string>
#include <vector>

namespace fdg {

static std::atomic<uint64_t> g_launches{0};
uint64_t launches() { return g_launches.load(); }

// ---- per-kernel-class device timing (off by default): every launcher opens a Scope, which counts the
// launch and, while profiling is on, brackets it with two events on the launching stream.
static const char* kClassNames[KC_COUNT] = {
    "fma_fwd", "fma_dgrad", "fma_wgrad", "splitk_reduce", "bias_grad", "relu_fwd", "relu_bwd", "add_fwd",
    "copy_accumulate", "maxpool_fwd", "maxpool_bwd", "gap_fwd", "gap_bwd", "bn_fwd_stats", "bn_fwd_apply", "bn_bwd_reduce",
    "bn_bwd_apply", "softmax_ce", "sgd_update", "tags", "fill", "tc_gemm_fwd", "tc_gemm_dgrad", "tc_gemm_wgrad", "tc_aux", "ingest",
    "mma_fwd", "mma_dgrad", "mma_wgrad",
};
namespace prof {
struct Rec { int cls; cudaEvent_t a, b; };
static bool g_on = false;
static std::mutex g_mu;
static std::vector<Rec> g_recs;
static std::vector<cudaEvent_t> g_pool;
static KernelStat g_stat[KC_COUNT];
static std::map<std::string, KernelStat> g_detail;          // "class[detail]" -> statistics
static thread_local const char* t_detail = nullptr;
struct DRec { std::string key; cudaEvent_t a, b; };
static std::vector<DRec> g_drecs;
static cudaEvent_t get_event() {
    if (!g_pool.empty()) { cudaEvent_t e = g_pool.back(); g_pool.pop_back(); return e; }
    cudaEvent_t e = nullptr; cudaEventCreate(&e); return e;
}
}  // namespace prof
void profile_detail(const char* d) { prof::t_detail = d; }
Scope::Scope(int cls_, double flops, double bytes, cudaStream_t s) : cls(cls_), st(s), a(nullptr), detail(prof::t_detail) {
    g_launches.fetch_add(1, std::memory_order_relaxed);
    if (!prof::g_on) return;
    std::lock_guard<std::mutex> lk(prof::g_mu);
    prof::g_stat[cls].launches += 1; prof::g_stat[cls].flops += flops; prof::g_stat[cls].bytes += bytes;
    if (detail) {
        KernelStat& d = prof::g_detail[std::string(kClassNames[cls]) + "[" + detail + "]"];
        d.launches += 1; d.flops += flops; d.bytes += bytes;
    }
    a = prof::get_event();
    cudaEventRecord(a, st);
}
Scope::~Scope() {
    if (!a) return;
    std::lock_guard<std::mutex> lk(prof::g_mu);
    cudaEvent_t b = prof::get_event();
    cudaEventRecord(b, st);
    prof::g_recs.push_back({cls, a, b});
    if (detail) prof::g_drecs.push_back({std::string(kClassNames[cls]) + "[" + detail + "]", a, b});
}
void profile_enable(bool on) {
    std::lock_guard<std::mutex> lk(prof::g_mu);
    if (on) { for (auto& k : prof::g_stat) k = KernelStat{}; prof::g_detail.clear(); }
    prof::g_on = on;
}
int profile_read(KernelStat* out, const char** names) {
    cudaDeviceSynchronize();
    std::lock_guard<std::mutex> lk(prof::g_mu);
    for (auto& r : prof::g_drecs) {
        float ms = 0.f;
        if (cudaEventElapsedTime(&ms, r.a, r.b) == cudaSuccess) prof::g_detail[r.key].ms += ms;
    }
    prof::g_drecs.clear();
    for (auto& r : prof::g_recs) {
        float ms = 0.f;
        if (cudaEventElapsedTime(&ms, r.a, r.b) == cudaSuccess) prof::g_stat[r.cls].ms += ms;
        prof::g_pool.push_back(r.a); prof::g_pool.push_back(r.b);
    }
    prof::g_recs.clear();
    for (int i = 0; i < KC_COUNT; ++i) { out[i] = prof::g_stat[i]; names[i] = kClassNames[i]; }
    return KC_COUNT;
}
int profile_read_detail(KernelStat* out, char (*names)[48], int capacity) {
    std::lock_guard<std::mutex> lk(prof::g_mu);
    int n = 0;
    for (auto& kv : prof::g_detail) {
        if (n >= capacity) break;
        out[n] = kv.second;
        std::snprintf(names[n], 48, "%s", kv.first.c_str());
        ++n;
    }
    return n;
}

typedef __nv_bfloat16 bf16;

__device__ __forceinline__ long long device_time_ns() { long long t; asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t)); return t; }
__device__ __forceinline__ float ld(const float* p) { return *p; }
__device__ __forceinline__ float ld(const bf16* p) { return __bfloat162float(*p); }
__device__ __forceinline__ void st(float* p, float v) { *p = v; }
__device__ __forceinline__ void st(bf16* p, float v) { *p = __float2bfloat16_rn(v); }

template <typename T> __device__ __forceinline__ float rounded(float v);        // v as T stores it
template <> __device__ __forceinline__ float rounded<float>(float v) { return v; }
template <> __device__ __forceinline__ float rounded<bf16>(float v) { return __bfloat162float(__float2bfloat16_rn(v)); }

static inline unsigned cdiv(size_t a, size_t b) { return (unsigned)((a + b - 1) / b); }

// Convolutions and linear layers on the CUDA cores: fconv.cu and linear.cu.
size_t wgrad_workspace_elems(const ConvGeom& g) { return linear_supported(g) ? 0 : fconv_wgrad_workspace_elems(g, 1); }
bool conv_supported(const ConvGeom& g) { return linear_supported(g) || fconv_supported(g); }
void conv_forward(int dt, const void* x, const void* w, const float* bias, void* y, const ConvGeom& g, int epi, const Packed& pk, cudaStream_t s) {
    if (linear_supported(g)) linear_forward(dt, x, w, bias, y, g, epi, 1, 0, 0, s);
    else fconv_forward(dt, x, w, bias, y, g, epi, 1, 0, 0, nullptr, pk, s);
}

// ------------------------------------------------------------------------------------------
// column sums (bias gradient): two stages, fixed order
// ------------------------------------------------------------------------------------------
constexpr int RED_CHUNKS = 64;

template <typename T>
__global__ void colsum_partial(const T* __restrict__ dy, float* __restrict__ part, long rows, int C) {
    int c = blockIdx.x * 32 + threadIdx.x;
    long per = (rows + gridDim.y - 1) / gridDim.y;
    long r0 = (long)blockIdx.y * per, r1 = min(rows, r0 + per);
    float s = 0.f;
    if (c < C) for (long r = r0 + threadIdx.y; r < r1; r += blockDim.y) s += ld(dy + r * C + c);
    __shared__ float sh[8][33];
    sh[threadIdx.y][threadIdx.x] = s;
    __syncthreads();
    if (threadIdx.y == 0 && c < C) {
        float t = 0.f;
        for (int i = 0; i < 8; ++i) t += sh[i][threadIdx.x];
        part[(size_t)blockIdx.y * C + c] = t;
    }
}
__global__ void colsum_final(const float* __restrict__ part, float* __restrict__ out, int chunks, int C, bool accum) {
    int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= C) return;
    float s = 0.f;
    for (int i = 0; i < chunks; ++i) s += part[(size_t)i * C + c];
    out[c] = accum ? out[c] + s : s;
}
void bias_grad(int dt, const void* dy, float* db, float* scratch, long rows, int C, bool accum, cudaStream_t s) {
    int chunks = (int)(rows < RED_CHUNKS ? rows : RED_CHUNKS);
    dim3 grid(cdiv(C, 32), chunks), blk(32, 8);
    { Scope sc(KC_BIAS_GRAD, 0.0, (dt ? 2.0 : 4.0) * rows * C, s);
      if (dt) klaunch(colsum_partial<bf16>, grid, blk, 0, s, (const bf16*)dy, scratch, rows, C);
      else klaunch(colsum_partial<float>, grid, blk, 0, s, (const float*)dy, scratch, rows, C); }
    Scope sc(KC_BIAS_GRAD, 0.0, 4.0 * chunks * C, s);
    klaunch(colsum_final, cdiv(C, 128), 128, 0, s, scratch, db, chunks, C, accum);
}

// ------------------------------------------------------------------------------------------
// elementwise layers: 128-bit accesses (8 bf16 or 4 fp32 values per thread and pass), grid-stride loops over a grid of
// a few CTAs per SM; the last n % V elements are handled one by one by the first threads
// ------------------------------------------------------------------------------------------
template <typename T> struct Vec;
template <> struct Vec<float> {
    static constexpr int V = 4;
    static __device__ __forceinline__ void load(const float* p, float (&f)[8]) { const float4 v = *(const float4*)p; f[0] = v.x; f[1] = v.y; f[2] = v.z; f[3] = v.w; }
    static __device__ __forceinline__ void store(float* p, const float (&f)[8]) { *(float4*)p = make_float4(f[0], f[1], f[2], f[3]); }
};
template <> struct Vec<bf16> {
    static constexpr int V = 8;
    static __device__ __forceinline__ void load(const bf16* p, float (&f)[8]) {
        const uint4 v = *(const uint4*)p; const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int j = 0; j < 4; ++j) { f[2 * j] = __uint_as_float(w[j] << 16); f[2 * j + 1] = __uint_as_float(w[j] & 0xffff0000u); }
    }
    static __device__ __forceinline__ void store(bf16* p, const float (&f)[8]) {
        uint32_t w[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) { const __nv_bfloat162 t = __floats2bfloat162_rn(f[2 * j], f[2 * j + 1]); w[j] = *(const uint32_t*)&t; }
        *(uint4*)p = make_uint4(w[0], w[1], w[2], w[3]);
    }
};
static unsigned ew_grid(size_t nvec) { size_t b = (nvec + 255) / 256; return (unsigned)(b < 1 ? 1 : (b > 148 * 8 ? 148 * 8 : b)); }

// OP 0: y = max(x, 0).  OP 1: dx (+)= dy * (y > 0)   (a = y, b = dy, o = dx).  OP 2: y = a + b.  OP 3: dst (+)= src   (a = src, o = dst).
template <typename T, int OP>
__global__ void __launch_bounds__(256) ew_k(const T* __restrict__ a, const T* __restrict__ b, T* o, size_t n, bool accum, bool aligned) {
    constexpr int V = Vec<T>::V;
    const size_t nvec = aligned ? n / V : 0, stride = (size_t)gridDim.x * blockDim.x, t0 = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    for (size_t i = t0; i < nvec; i += stride) {
        float fa[8], fb[8], fo[8];
        Vec<T>::load(a + i * V, fa);
        if (OP == 1 || OP == 2) Vec<T>::load(b + i * V, fb);
        if ((OP == 1 || OP == 3) && accum) Vec<T>::load(o + i * V, fo);
#pragma unroll
        for (int j = 0; j < V; ++j) {
            float v;
            if (OP == 0) v = fmaxf(fa[j], 0.f);
            else if (OP == 1) v = fa[j] > 0.f ? fb[j] : 0.f;
            else if (OP == 2) v = fa[j] + fb[j];
            else v = fa[j];
            if ((OP == 1 || OP == 3) && accum) v += fo[j];
            fo[j] = v;
        }
        Vec<T>::store(o + i * V, fo);
    }
    for (size_t i = nvec * V + t0; i < n; i += stride) {
        float v;
        if (OP == 0) v = fmaxf(ld(a + i), 0.f);
        else if (OP == 1) v = ld(a + i) > 0.f ? ld(b + i) : 0.f;
        else if (OP == 2) v = ld(a + i) + ld(b + i);
        else v = ld(a + i);
        if ((OP == 1 || OP == 3) && accum) v += ld(o + i);
        st(o + i, v);
    }
}
template <int OP>
static void ew_launch(int dt, const void* a, const void* b, void* o, size_t n, bool accum, cudaStream_t s) {
    // a window of a tensor whose rows are no multiple of 16 bytes can start anywhere: such calls go element by element
    const bool aligned = (((uintptr_t)a | (uintptr_t)b | (uintptr_t)o) & 15) == 0;
    const size_t work = aligned ? n / (dt ? 8 : 4) : n;
    if (dt) klaunch(ew_k<bf16, OP>, ew_grid(work), 256, 0, s, (const bf16*)a, (const bf16*)b, (bf16*)o, n, accum, aligned);
    else klaunch(ew_k<float, OP>, ew_grid(work), 256, 0, s, (const float*)a, (const float*)b, (float*)o, n, accum, aligned);
}

void relu_forward(int dt, const void* x, void* y, size_t n, cudaStream_t s) {
    Scope sc(KC_RELU_FWD, 0.0, 2 * (dt ? 2.0 : 4.0) * n, s);
    ew_launch<0>(dt, x, nullptr, y, n, false, s);
}
void relu_backward(int dt, const void* y, const void* dy, void* dx, size_t n, bool accum, cudaStream_t s) {
    Scope sc(KC_RELU_BWD, 0.0, (accum ? 4 : 3) * (dt ? 2.0 : 4.0) * n, s);
    ew_launch<1>(dt, y, dy, dx, n, accum, s);
}
void add_forward(int dt, const void* a, const void* b, void* y, size_t n, cudaStream_t s) {
    Scope sc(KC_ADD_FWD, 0.0, 3 * (dt ? 2.0 : 4.0) * n, s);
    ew_launch<2>(dt, a, b, y, n, false, s);
}
void copy_or_accumulate(int dt, const void* src, void* dst, size_t n, bool accum, cudaStream_t s) {
    Scope sc(KC_COPY_ACC, 0.0, (accum ? 3 : 2) * (dt ? 2.0 : 4.0) * n, s);
    ew_launch<3>(dt, src, nullptr, dst, n, accum, s);
}

// ------------------------------------------------------------------------------------------
// Backward pass through "+ bias, ReLU" of a linear / conv layer in ONE pass over dy:  dy *= (y > 0) in place (if the layer
// has a ReLU) and db[c] = sum over rows of the masked dy (if it has a bias).  A thread keeps one 128-bit channel group for
// every row it visits; a CTA owns a contiguous row range; partial sums per CTA, then a fixed-order final sum.
// Used when C / V is a power of two <= 256 (V = 8 bf16 / 4 fp32 values per access); other widths take the generic kernels.
// ------------------------------------------------------------------------------------------
constexpr int RB_MAX_CHUNKS = 592;
template <typename T>
__global__ void __launch_bounds__(256) relu_bias_bwd_k(const T* __restrict__ y, T* dy, float* __restrict__ part, long rows, int C, long rows_per_cta) {
    constexpr int V = Vec<T>::V;
    const int cgs = C / V, rows_it = 256 / cgs, cg = threadIdx.x % cgs, rl = threadIdx.x / cgs;
    const long r0 = (long)blockIdx.x * rows_per_cta, r1 = min(rows, r0 + rows_per_cta);
    float s[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) s[j] = 0.f;
    for (long r = r0 + rl; r < r1; r += rows_it) {
        const size_t o = (size_t)r * C + (size_t)cg * V;
        float g[8];
        Vec<T>::load(dy + o, g);
        if (y) {
            float a[8];
            Vec<T>::load(y + o, a);
#pragma unroll
            for (int j = 0; j < V; ++j) if (!(a[j] > 0.f)) g[j] = 0.f;
            Vec<T>::store(dy + o, g);
        }
#pragma unroll
        for (int j = 0; j < V; ++j) s[j] += g[j];
    }
    if (!part) return;
    __shared__ float sh[256][9];
#pragma unroll
    for (int j = 0; j < V; ++j) sh[threadIdx.x][j] = s[j];
    __syncthreads();
    for (int t = threadIdx.x; t < C; t += 256) {
        const int q = t / V, k = t % V;
        float acc = 0.f;
        for (int rr = 0; rr < rows_it; ++rr) acc += sh[rr * cgs + q][k];
        part[(size_t)blockIdx.x * C + t] = acc;
    }
}
// one warp per channel: lanes take the partials round-robin, then a fixed shuffle tree
__global__ void colsum_final_warp(const float* __restrict__ part, float* __restrict__ out, int chunks, int C, bool accum) {
    const int c = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (c >= C) return;
    float a = 0.f;
    for (int k = lane; k < chunks; k += 32) a += part[(size_t)k * C + c];
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) a += __shfl_xor_sync(0xffffffffu, a, d);
    if (lane == 0) out[c] = accum ? out[c] + a : a;
}
// out[c] = sum over the records of part[rec][c][0] (records that a kernel's epilogue left, see KmParams::stat_part): one block per 4
// channels, a thread owns one channel and every 64th record, eight loads in flight, then a fixed tree.
__global__ void __launch_bounds__(256) colsum_records_k(const float* __restrict__ part, float* __restrict__ out, int recs, int C, bool accum) {
    __shared__ float sh[64][5];
    const int cl = threadIdx.x & 3, kl = threadIdx.x >> 2, c = blockIdx.x * 4 + cl;
    const float* p = part + (size_t)c * 2;
    float a = 0.f;
    int k = kl;
    for (; k + 448 < recs; k += 512) {
        float v[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) v[j] = p[(size_t)(k + 64 * j) * C * 2];
        a += ((v[0] + v[1]) + (v[2] + v[3])) + ((v[4] + v[5]) + (v[6] + v[7]));
    }
    for (; k < recs; k += 64) a += p[(size_t)k * C * 2];
    sh[kl][cl] = a;
    __syncthreads();
    for (int d = 32; d > 0; d >>= 1) { if (kl < d) sh[kl][cl] += sh[kl + d][cl]; __syncthreads(); }
    if (kl == 0) out[c] = accum ? out[c] + sh[0][cl] : sh[0][cl];
}
void colsum_records(const float* part, float* out, int recs, int C, bool accum, cudaStream_t s) {
    Scope sc(KC_BIAS_GRAD, 0.0, 8.0 * recs * C, s);
    klaunch(colsum_records_k, C / 4, 256, 0, s, part, out, recs, C, accum);
}
// The sums a block's threads hold for their channel group (thread t: group t % cgs, V values) -> rec[c][0], in a fixed order.
template <int V>
__device__ __forceinline__ void block_colsum(const float (&s)[8], float* rec, int cgs) {
    __shared__ float sh[256][9];
#pragma unroll
    for (int j = 0; j < V; ++j) sh[threadIdx.x][j] = s[j];
    __syncthreads();
    for (int t = threadIdx.x; t < cgs * V; t += 256) {
        const int q = t / V, k = t % V;
        float a = 0.f;
        for (int r = q; r < 256; r += cgs) a += sh[r][k];
        rec[(size_t)t * 2] = a;
    }
}
bool relu_bias_backward_supported(int dt, int C) {
    const int V = dt ? 8 : 4;
    if (C % V) return false;
    const int cgs = C / V;
    return cgs <= 256 && (cgs & (cgs - 1)) == 0;
}
size_t relu_bias_backward_scratch_elems(int C) { return (size_t)RB_MAX_CHUNKS * C; }
void relu_bias_backward(int dt, const void* y_or_null, void* dy, float* db_or_null, float* scratch, long rows, int C, bool accum, cudaStream_t s) {
    const int V = dt ? 8 : 4, rows_it = 256 / (C / V);
    long chunks = (rows + (long)rows_it * 8 - 1) / ((long)rows_it * 8);              // at least eight passes per CTA
    if (chunks > RB_MAX_CHUNKS) chunks = RB_MAX_CHUNKS;
    if (chunks < 1) chunks = 1;
    long per = (rows + chunks - 1) / chunks;
    per = (per + rows_it - 1) / rows_it * rows_it;
    chunks = (rows + per - 1) / per;
    const double esz = dt ? 2.0 : 4.0;
    { Scope sc(db_or_null ? KC_BIAS_GRAD : KC_RELU_BWD, 0.0, esz * rows * C * (y_or_null ? 3 : 1), s);
      if (dt) klaunch(relu_bias_bwd_k<bf16>, (unsigned)chunks, 256, 0, s, (const bf16*)y_or_null, (bf16*)dy, db_or_null ? scratch : nullptr, rows, C, per);
      else klaunch(relu_bias_bwd_k<float>, (unsigned)chunks, 256, 0, s, (const float*)y_or_null, (float*)dy, db_or_null ? scratch : nullptr, rows, C, per); }
    if (db_or_null) {
        Scope sc(KC_BIAS_GRAD, 0.0, 4.0 * chunks * C, s);
        klaunch(colsum_final_warp, cdiv((size_t)C * 32, 256), 256, 0, s, scratch, db_or_null, (int)chunks, C, accum);
    }
}

template <typename T>
__global__ void maxpool_fwd_k(const T* x, T* y, int N, int H, int W, int C) {
    size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    int Ho = H / 2, Wo = W / 2;
    size_t total = (size_t)N * Ho * Wo * C;
    if (i >= total) return;
    int c = i % C; size_t p = i / C; int ox = p % Wo; p /= Wo; int oy = p % Ho; int n = p / Ho;
    const T* b = x + (((size_t)n * H + 2 * oy) * W + 2 * ox) * C + c;
    float m = ld(b);
    m = fmaxf(m, ld(b + C)); m = fmaxf(m, ld(b + (size_t)W * C)); m = fmaxf(m, ld(b + (size_t)W * C + C));
    st(y + i, m);
}
template <typename T>
__global__ void maxpool_bwd_k(const T* x, const T* dy, T* dx, int N, int H, int W, int C, bool accum) {
    size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    int Ho = H / 2, Wo = W / 2;
    size_t total = (size_t)N * Ho * Wo * C;
    if (i >= total) return;
    int c = i % C; size_t p = i / C; int ox = p % Wo; p /= Wo; int oy = p % Ho; int n = p / Ho;
    size_t base = (((size_t)n * H + 2 * oy) * W + 2 * ox) * C + c;
    size_t o[4] = {base, base + (size_t)C, base + (size_t)W * C, base + (size_t)W * C + C};
    int best = 0; float m = ld(x + o[0]);
#pragma unroll
    for (int j = 1; j < 4; ++j) { float v = ld(x + o[j]); if (v > m) { m = v; best = j; } }   // first maximum wins
    float g = ld(dy + i);
#pragma unroll
    for (int j = 0; j < 4; ++j) { float v = (j == best) ? g : 0.f; if (accum) v += ld(dx + o[j]); st(dx + o[j], v); }
}
// the same with one 128-bit channel group per thread (C a multiple of the vector width)
template <typename T>
__global__ void __launch_bounds__(256) maxpool_fwd_vk(const T* __restrict__ x, T* __restrict__ y, int N, int H, int W, int C) {
    constexpr int V = Vec<T>::V;
    const int Ho = H / 2, Wo = W / 2, cgs = C / V;
    const size_t total = (size_t)N * Ho * Wo * cgs;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x) {
        const int cg = (int)(i % cgs); size_t p = i / cgs; const int ox = (int)(p % Wo); p /= Wo; const int oy = (int)(p % Ho); const size_t n = p / Ho;
        const T* b = x + ((n * H + 2 * oy) * W + 2 * ox) * C + (size_t)cg * V;
        float a0[8], a1[8], a2[8], a3[8];
        Vec<T>::load(b, a0); Vec<T>::load(b + C, a1); Vec<T>::load(b + (size_t)W * C, a2); Vec<T>::load(b + (size_t)W * C + C, a3);
#pragma unroll
        for (int j = 0; j < V; ++j) a0[j] = fmaxf(fmaxf(a0[j], a1[j]), fmaxf(a2[j], a3[j]));
        Vec<T>::store(y + i * V, a0);
    }
}
template <typename T>
__global__ void __launch_bounds__(256) maxpool_bwd_vk(const T* __restrict__ x, const T* __restrict__ dy, T* dx, int N, int H, int W, int C, bool accum, float* col) {
    constexpr int V = Vec<T>::V;
    const int Ho = H / 2, Wo = W / 2, cgs = C / V;
    const size_t total = (size_t)N * Ho * Wo * cgs;
    float sum[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) sum[j] = 0.f;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x) {
        const int cg = (int)(i % cgs); size_t p = i / cgs; const int ox = (int)(p % Wo); p /= Wo; const int oy = (int)(p % Ho); const size_t n = p / Ho;
        const size_t base = ((n * H + 2 * oy) * W + 2 * ox) * C + (size_t)cg * V;
        const size_t o[4] = {base, base + (size_t)C, base + (size_t)W * C, base + (size_t)W * C + C};
        float a[4][8], g[8];
#pragma unroll
        for (int q = 0; q < 4; ++q) Vec<T>::load(x + o[q], a[q]);
        Vec<T>::load(dy + i * V, g);
        int best[8];
#pragma unroll
        for (int j = 0; j < V; ++j) {
            int b = 0; float m = a[0][j];
#pragma unroll
            for (int q = 1; q < 4; ++q) if (a[q][j] > m) { m = a[q][j]; b = q; }            // first maximum wins
            best[j] = b;
            if (col) { if (!(m > 0.f)) g[j] = 0.f; sum[j] += g[j]; }        // x is a ReLU's output: its gradient, masked, and that layer's bias gradient
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            float v[8];
            if (accum) Vec<T>::load(dx + o[q], v);
#pragma unroll
            for (int j = 0; j < V; ++j) { const float t = best[j] == q ? g[j] : 0.f; v[j] = accum ? v[j] + t : t; }
            Vec<T>::store(dx + o[q], v);
        }
    }
    if (col) block_colsum<V>(sum, col + (size_t)blockIdx.x * C * 2, cgs);
}
void maxpool_forward(int dt, const void* x, void* y, int N, int H, int W, int C, cudaStream_t s) {
    const double esz_ = dt ? 2.0 : 4.0;
    Scope sc(KC_POOL_FWD, 0.0, 1.25 * esz_ * (double)N * H * W * C, s);
    size_t n = (size_t)N * (H / 2) * (W / 2) * C;
    if (C % (dt ? 8 : 4) == 0) {
        if (dt) klaunch(maxpool_fwd_vk<bf16>, ew_grid(n / 8), 256, 0, s, (const bf16*)x, (bf16*)y, N, H, W, C);
        else klaunch(maxpool_fwd_vk<float>, ew_grid(n / 4), 256, 0, s, (const float*)x, (float*)y, N, H, W, C);
        return;
    }
    if (dt) klaunch(maxpool_fwd_k<bf16>, cdiv(n, 256), 256, 0, s, (const bf16*)x, (bf16*)y, N, H, W, C);
    else klaunch(maxpool_fwd_k<float>, cdiv(n, 256), 256, 0, s, (const float*)x, (float*)y, N, H, W, C);
}
int pool_col_records(int dt, int N, int H, int W, int C) { return (int)ew_grid((size_t)N * (H / 2) * (W / 2) * C / (dt ? 8 : 4)); }
void maxpool_backward(int dt, const void* x, const void* dy, void* dx, int N, int H, int W, int C, bool accum, float* col_or_null, cudaStream_t s) {
    const double esz_ = dt ? 2.0 : 4.0;
    Scope sc(KC_POOL_BWD, 0.0, 2.25 * esz_ * (double)N * H * W * C, s);
    size_t n = (size_t)N * (H / 2) * (W / 2) * C;
    if (C % (dt ? 8 : 4) == 0) {
        if (dt) klaunch(maxpool_bwd_vk<bf16>, ew_grid(n / 8), 256, 0, s, (const bf16*)x, (const bf16*)dy, (bf16*)dx, N, H, W, C, accum, col_or_null);
        else klaunch(maxpool_bwd_vk<float>, ew_grid(n / 4), 256, 0, s, (const float*)x, (const float*)dy, (float*)dx, N, H, W, C, accum, col_or_null);
        return;
    }
    if (dt) klaunch(maxpool_bwd_k<bf16>, cdiv(n, 256), 256, 0, s, (const bf16*)x, (const bf16*)dy, (bf16*)dx, N, H, W, C, accum);
    else klaunch(maxpool_bwd_k<float>, cdiv(n, 256), 256, 0, s, (const float*)x, (const float*)dy, (float*)dx, N, H, W, C, accum);
}

template <typename T>
__global__ void gap_fwd_k(const T* x, T* y, int N, int HW, int C) {
    size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= (size_t)N * C) return;
    int c = i % C; size_t n = i / C;
    float s = 0.f;
    for (int p = 0; p < HW; ++p) s += ld(x + (n * HW + p) * C + c);
    st(y + i, s / (float)HW);
}
template <typename T>
__global__ void gap_bwd_k(const T* dy, T* dx, int N, int HW, int C, bool accum) {
    size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= (size_t)N * HW * C) return;
    int c = i % C; size_t n = i / ((size_t)HW * C);
    float v = ld(dy + n * C + c) / (float)HW;
    if (accum) v += ld(dx + i);
    st(dx + i, v);
}
// the same with one 16-byte vector (4 fp32 / 8 bf16 channels) per thread; C a multiple of the vector length
template <typename T>
__global__ void __launch_bounds__(256) gap_bwd_vk(const T* __restrict__ dy, T* __restrict__ dx, size_t nvec, int HW, int Cv, bool accum, const T* __restrict__ x, float* col) {
    constexpr int V = Vec<T>::V;
    float sum[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) sum[j] = 0.f;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < nvec; i += (size_t)gridDim.x * blockDim.x) {
        const int cv = (int)(i % Cv); const size_t n = i / ((size_t)HW * Cv);
        float g[8], o[8];
        Vec<T>::load(dy + (n * Cv + cv) * V, g);
        if (accum) Vec<T>::load(dx + i * V, o);
#pragma unroll
        for (int j = 0; j < V; ++j) g[j] = accum ? g[j] / (float)HW + o[j] : g[j] / (float)HW;
        if (x) {                             // x is a ReLU's output: its gradient, masked, and (col) that layer's bias gradient
            float xv[8];
            Vec<T>::load(x + i * V, xv);
#pragma unroll
            for (int j = 0; j < V; ++j) { if (!(xv[j] > 0.f)) g[j] = 0.f; sum[j] += rounded<T>(g[j]); }
        }
        Vec<T>::store(dx + i * V, g);
    }
    if (col) block_colsum<V>(sum, col + (size_t)blockIdx.x * Cv * V * 2, Cv);
}
void gap_forward(int dt, const void* x, void* y, int N, int HW, int C, cudaStream_t s) {
    const double esz_ = dt ? 2.0 : 4.0; (void)esz_;
    Scope sc(KC_GAP_FWD, 0.0, esz_ * (double)N * (HW + 1) * C, s);
    size_t n = (size_t)N * C;
    if (dt) klaunch(gap_fwd_k<bf16>, cdiv(n, 128), 128, 0, s, (const bf16*)x, (bf16*)y, N, HW, C);
    else klaunch(gap_fwd_k<float>, cdiv(n, 128), 128, 0, s, (const float*)x, (float*)y, N, HW, C);
    
}
int gap_col_records(int dt, int N, int HW, int C) { return (int)ew_grid((size_t)N * HW * C / (dt ? 8 : 4)); }
void gap_backward(int dt, const void* dy, void* dx, int N, int HW, int C, bool accum, const void* mask_x_or_null, float* col_or_null, cudaStream_t s) {
    const double esz_ = dt ? 2.0 : 4.0; (void)esz_;
    Scope sc(KC_GAP_BWD, 0.0, esz_ * (double)N * (HW + 1) * C, s);
    size_t n = (size_t)N * HW * C;
    const int V = dt ? 8 : 4;
    if (C % V == 0 && ((uintptr_t)dy | (uintptr_t)dx) % 16 == 0) {
        const size_t nvec = n / V;
        if (dt) klaunch(gap_bwd_vk<bf16>, ew_grid(nvec), 256, 0, s, (const bf16*)dy, (bf16*)dx, nvec, HW, C / V, accum, (const bf16*)mask_x_or_null, col_or_null);
        else klaunch(gap_bwd_vk<float>, ew_grid(nvec), 256, 0, s, (const float*)dy, (float*)dx, nvec, HW, C / V, accum, (const float*)mask_x_or_null, col_or_null);
        return;
    }
    if (dt) klaunch(gap_bwd_k<bf16>, cdiv(n, 256), 256, 0, s, (const bf16*)dy, (bf16*)dx, N, HW, C, accum);
    else klaunch(gap_bwd_k<float>, cdiv(n, 256), 256, 0, s, (const float*)dy, (float*)dx, N, HW, C, accum);
    
}

// ------------------------------------------------------------------------------------------
// batch-norm, statistics per worker
// ------------------------------------------------------------------------------------------
// grid (C/32, chunks, workers), block (32, 8).  part: [chunk][worker][C][2]
template <typename T, bool BWD>
__global__ void bn_reduce_partial(const T* __restrict__ x, const T* __restrict__ out, const T* __restrict__ dout,
                                  const float* __restrict__ stats, float* __restrict__ part, long rpw, int C, bool relu) {
    int c = blockIdx.x * 32 + threadIdx.x;
    int w = blockIdx.z, nw = gridDim.z;
    long per = (rpw + gridDim.y - 1) / gridDim.y;
    long r0 = (long)blockIdx.y * per, r1 = min(rpw, r0 + per);
    float s1 = 0.f, s2 = 0.f;
    if (c < C) {
        float mean = 0.f, istd = 0.f;
        if (BWD) { mean = stats[((size_t)w * C + c) * 2]; istd = stats[((size_t)w * C + c) * 2 + 1]; }
        const float pivot = BWD ? 0.f : ld(x + (size_t)w * rpw * C + c);
        for (long r = r0 + threadIdx.y; r < r1; r += blockDim.y) {
            size_t o = ((size_t)w * rpw + r) * C + c;
            if (BWD) {
                float dy = ld(dout + o);
                if (relu && !(ld(out + o) > 0.f)) dy = 0.f;
                s1 += dy; s2 += dy * (ld(x + o) - mean) * istd;
            } else {
                // sums of (x - pivot): the pivot (the worker's first value of the channel) keeps the variance
                // formula E[d^2] - E[d]^2 from cancelling when |mean| >> std
                float v = ld(x + o) - pivot; s1 += v; s2 += v * v;
            }
        }
    }
    __shared__ float sh1[8][33], sh2[8][33];
    sh1[threadIdx.y][threadIdx.x] = s1; sh2[threadIdx.y][threadIdx.x] = s2;
    __syncthreads();
    if (threadIdx.y == 0 && c < C) {
        float a = 0.f, b = 0.f;
        for (int i = 0; i < 8; ++i) { a += sh1[i][threadIdx.x]; b += sh2[i][threadIdx.x]; }
        size_t o = (((size_t)blockIdx.y * nw + w) * C + c) * 2;
        part[o] = a; part[o + 1] = b;
    }
}
// forward: stats[w][c] = (mean, invstd).  One thread per (w, c).
template <typename T>
__global__ void bn_stats_final(const float* __restrict__ part, const T* __restrict__ x, float* __restrict__ stats, int chunks, int nwC,
                               int C, long rpw) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= nwC) return;
    double s1 = 0.0, s2 = 0.0;
    for (int k = 0; k < chunks; ++k) { s1 += part[((size_t)k * nwC + i) * 2]; s2 += part[((size_t)k * nwC + i) * 2 + 1]; }
    const int w = i / C, c = i - w * C;
    const double pivot = (double)ld(x + (size_t)w * rpw * C + c);       // the partial sums are sums of (x - pivot)
    double dm = s1 / (double)rpw, var = s2 / (double)rpw - dm * dm;
    if (var < 0.0) var = 0.0;
    stats[(size_t)i * 2] = (float)(pivot + dm);
    stats[(size_t)i * 2 + 1] = (float)(1.0 / sqrt(var + 1e-5));
}
// backward: red[w][c] = (sum dy, sum dy xhat); dgamma[c] = sum_w red[w][c].y; dbeta[c] = sum_w red[w][c].x
__global__ void bn_bwd_final(const float* __restrict__ part, float* __restrict__ red, float* __restrict__ dgamma,
                             float* __restrict__ dbeta, int chunks, int nw, int C, bool accum) {
    int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= C) return;
    float g = 0.f, b = 0.f;
    for (int w = 0; w < nw; ++w) {
        float s1 = 0.f, s2 = 0.f;
        for (int k = 0; k < chunks; ++k) { size_t o = (((size_t)k * nw + w) * C + c) * 2; s1 += part[o]; s2 += part[o + 1]; }
        red[((size_t)w * C + c) * 2] = s1; red[((size_t)w * C + c) * 2 + 1] = s2;
        b += s1; g += s2;
    }
    dgamma[c] = accum ? dgamma[c] + g : g; dbeta[c] = accum ? dbeta[c] + b : b;
}
template <typename T>
__global__ void bn_apply_k(const T* __restrict__ x, const float* __restrict__ gamma, const float* __restrict__ beta,
                           const T* __restrict__ res, T* __restrict__ y, const float* __restrict__ stats,
                           long rpw, int C, size_t total, bool relu) {
    size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= total) return;
    int c = i % C; size_t row = i / C; int w = (int)(row / rpw);
    float mean = stats[((size_t)w * C + c) * 2], istd = stats[((size_t)w * C + c) * 2 + 1];
    float v = gamma[c] * (ld(x + i) - mean) * istd + beta[c];
    if (res) v += ld(res + i);
    if (relu) v = fmaxf(v, 0.f);
    st(y + i, v);
}
template <typename T>
__global__ void bn_bwd_apply_k(const T* __restrict__ x, const T* __restrict__ out, const T* __restrict__ dout,
                               const float* __restrict__ gamma, const float* __restrict__ stats, const float* __restrict__ red,
                               T* __restrict__ dx, bool accum_dx, T* __restrict__ dres, bool accum_dres,
                               long rpw, int C, size_t total, bool relu) {
    size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= total) return;
    int c = i % C; size_t row = i / C; int w = (int)(row / rpw);
    size_t so = ((size_t)w * C + c) * 2;
    float mean = stats[so], istd = stats[so + 1];
    float dy = ld(dout + i);
    if (relu && !(ld(out + i) > 0.f)) dy = 0.f;
    float xh = (ld(x + i) - mean) * istd;
    float inv_n = 1.f / (float)rpw;
    if (dx) {
        float v = gamma[c] * istd * (dy - red[so] * inv_n - xh * red[so + 1] * inv_n);
        if (accum_dx) v += ld(dx + i);
        st(dx + i, v);
    }
    if (dres) { float r = dy; if (accum_dres) r += ld(dres + i); st(dres + i, r); }
}

// ------------------------------------------------------------------------------------------
// Batch-norm, bf16 storage, streamed: a CTA owns a contiguous range of one worker's rows, which is one
// contiguous range of memory (NHWC).  One thread feeds a ring of shared-memory stages with bulk asynchronous
// copies (cp.async.bulk, completion on an mbarrier), 16 KB per input tensor and stage, so that about 90 KB per
// CTA are in flight whatever the registers hold; all 256 threads read 16-byte vectors (8 channels) from the
// stage, and results go straight to global memory.  A thread keeps the same 8 channels for every row.
// grid = (row chunks, workers).  Used when C/8 is a power of two <= 256.
// ------------------------------------------------------------------------------------------
constexpr int BNV_THREADS = 256;
constexpr int BNV_MAX_CHUNKS = 128;
constexpr int BV = 8;                               // channels per thread (one 128-bit access)
// ring geometry: the best of the measured family (rings of 48..192 KB, 1..4 CTAs per SM, tiles of 8..32 KB)
constexpr int BNS_TILE = 16384;                     // bytes per input tensor and stage
constexpr int BNS_CTAS = 2;                         // CTAs per SM the ring size allows
constexpr int BNS_RING = 96 * 1024;                 // shared memory of the ring (stages = tiles in the ring / input tensors, at most 8)
constexpr int BNS_VPT = BNS_TILE / 16 / 256;        // 16-byte vectors per thread and tile
constexpr long long BNS_WAIT_CYCLES = 4000000000LL; // ~2 s

constexpr int BP = BV / 2;                          // channel pairs per thread
__device__ __forceinline__ void unpack8(const uint4& v, float2 (&f)[BP]) {
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int j = 0; j < BP; ++j) f[j] = make_float2(__uint_as_float(w[j] << 16), __uint_as_float(w[j] & 0xffff0000u));
}
// round to nearest even; RELU: negative values become zero in the same conversion
template <bool RELU>
__device__ __forceinline__ uint4 pack8(const float2 (&f)[BP]) {
    uint32_t w[BP];
#pragma unroll
    for (int j = 0; j < BP; ++j) {
        if (RELU) asm("cvt.rn.relu.bf16x2.f32 %0, %1, %2;" : "=r"(w[j]) : "f"(f[j].y), "f"(f[j].x));
        else asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(w[j]) : "f"(f[j].y), "f"(f[j].x));
    }
    return make_uint4(w[0], w[1], w[2], w[3]);
}
// the one expression both passes use for the normalised value, so that the backward pass can recompute the sign of
// the forward output from x alone: gamma * ((x - mean) * invstd) + beta, the product rounded before the fused last
// step, two channels per instruction
__device__ __forceinline__ float2 bn_pair(float2 x, float2 neg_mean, float2 invstd, float2 gamma, float2 beta) {
    return __ffma2_rn(gamma, __fmul2_rn(__fadd2_rn(x, neg_mean), invstd), beta);
}

__device__ __forceinline__ uint32_t bns_smem(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ bool bns_wait(uint32_t bar, uint32_t parity, int* err) {
    uint32_t ok;
    long long t0 = 0;
    for (;;) {
        asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                     : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
        if (ok) return true;
        if (t0 == 0) t0 = clock64();
        else if (clock64() - t0 > BNS_WAIT_CYCLES) { atomicCAS(err, 0, 20); return false; }
    }
}

// p[0] + p[stride] + ... (n terms, in that order), eight loads in flight
__device__ __forceinline__ float2 sum_strided(const float2* p, size_t stride, int n) {
    float2 acc = make_float2(0.f, 0.f);
    int i = 0;
    for (; i + 8 <= n; i += 8) {
        float2 v[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) v[j] = p[(size_t)(i + j) * stride];
#pragma unroll
        for (int j = 0; j < 8; ++j) { acc.x += v[j].x; acc.y += v[j].y; }
    }
    for (; i < n; ++i) { const float2 v = p[(size_t)i * stride]; acc.x += v.x; acc.y += v.y; }
    return acc;
}
// a fixed shuffle tree: the summation order never changes
__device__ __forceinline__ float2 warp_sum2(float2 v) {
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) { v.x += __shfl_xor_sync(0xffffffffu, v.x, d); v.y += __shfl_xor_sync(0xffffffffu, v.y, d); }
    return v;
}

struct BnsArgs {
    const bf16* in[3];          // input tensors streamed through the ring: x, then dout, then the forward output (as the mode needs)
    int n_in;
    const float* gamma; const float* beta; const float* stats; const bf16* res;
    float* part;                // modes 0, 1: partial sums [chunk][worker][C][2], written; mode 3: the same, read (gridDim.x chunks)
    float* dgamma; float* dbeta; int accum_params;   // mode 3: parameter gradients, written by one CTA
    bf16* y;                    // mode 2: output; mode 3: dx, or nullptr (the network's input: not needed)
    bf16* dres;                 // mode 3: gradient of the residual input, or nullptr
    long rpw; int C; int relu; int mask_from_x; int accum_dx; int accum_dres;
    int reverse;                // walk the CTA's tiles from the last to the first: a kernel that re-reads what the kernel before it
                                // has just streamed in ascending order (backward apply after backward sums) starts with the part
                                // that is still in L2
    int* err;
};

// MODE 0: (sum x, sum x^2).  MODE 1: (sum dy, sum dy * xhat) with dy = dout * [forward output > 0] if relu.
// MODE 2: y = bn(x) (+ res) (relu).  MODE 3: dx (+)= BN backward of dy, dres (+)= dy.
// mask_from_x: the forward output had no residual, so its sign is the sign of bn_pair(x).
template <int MODE>
__global__ void __launch_bounds__(BNV_THREADS, BNS_CTAS) bns_kernel(const BnsArgs a) {
    extern __shared__ __align__(128) uint8_t bns_sm[];
    const int C = a.C, cgs = C / BV, rows_it = BNV_THREADS / cgs;
    const int tid = threadIdx.x, cg = tid % cgs, rl = tid / cgs;
    const int w = blockIdx.y, nw = gridDim.y;
    const int n_in = a.n_in, stages = (BNS_RING / BNS_TILE) / n_in < 8 ? (BNS_RING / BNS_TILE) / n_in : 8;
    const int tile_rows = BNS_TILE / (C * 2);
    long per = (a.rpw + gridDim.x - 1) / gridDim.x;
    per = (per + tile_rows - 1) / tile_rows * tile_rows;
    const long r0 = (long)blockIdx.x * per, r1 = min(a.rpw, r0 + per);
    const int ntiles = r1 > r0 ? (int)((r1 - r0 + tile_rows - 1) / tile_rows) : 0;
    uint64_t* full = (uint64_t*)(bns_sm + BNS_RING);
    const uint32_t full0 = bns_smem(full), ring0 = bns_smem(bns_sm);
    if (tid == 0) {
        for (int s = 0; s < stages; ++s) asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(full0 + 8 * s), "r"(1) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    const size_t wbase = (size_t)w * a.rpw * C;           // first element of this worker
    auto issue = [&](int i) {                             // thread 0: fill stage i % stages with tile i
        const int st = i % stages;
        const long row = r0 + (long)(a.reverse ? ntiles - 1 - i : i) * tile_rows;
        const long rows = r1 - row < tile_rows ? r1 - row : tile_rows;
        const uint32_t bytes = (uint32_t)(rows * C * 2), bar = full0 + 8 * st;
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes * n_in) : "memory");
        for (int k = 0; k < n_in; ++k)
            asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                         ::"r"(ring0 + (st * n_in + k) * BNS_TILE), "l"(a.in[k] + wbase + (size_t)row * C), "r"(bytes), "r"(bar) : "memory");
    };
    if (tid == 0) for (int i = 0; i < stages - 1 && i < ntiles; ++i) issue(i);

    // MODE 3: (sum dy, sum dy xhat) of this worker from the chunk partials of the sums kernel (same grid), while the first
    // tiles are on their way: all threads take part (up to 256 / C interleaved chunk subsets per channel, then a
    // fixed-order sum of the subsets), so every CTA of a worker gets the same sums in the same order.  dgamma / dbeta:
    // CTA i of the launch takes the channels c = i (mod number of CTAs), one warp per channel, lanes over the
    // (worker, chunk) partials and a fixed shuffle tree.
    float2* const red_s = (float2*)(bns_sm + BNS_RING + 64);
    if (MODE == 3) {
        const int chunks = gridDim.x;
        const float2* const part = (const float2*)a.part;
        if (C <= BNV_THREADS) {
            float2* const tmp = red_s + C;                  // [256 / C][C]
            const int nparts = BNV_THREADS / C, c = tid % C, pt = tid / C;
            tmp[pt * C + c] = sum_strided(part + ((size_t)pt * nw + w) * C + c, (size_t)nparts * nw * C, (chunks - pt + nparts - 1) / nparts);
            __syncthreads();
            if (tid < C) {
                float2 t = make_float2(0.f, 0.f);
                for (int q = 0; q < nparts; ++q) { t.x += tmp[q * C + tid].x; t.y += tmp[q * C + tid].y; }
                red_s[tid] = t;
            }
        } else {
            for (int c = tid; c < C; c += BNV_THREADS) red_s[c] = sum_strided(part + (size_t)w * C + c, (size_t)nw * C, chunks);
        }
        {
            const int warp = tid >> 5, lane = tid & 31, rows = nw * chunks, me = w * chunks + blockIdx.x;      // rows = CTAs of the launch
            for (int c = me + warp * rows; c < C; c += (BNV_THREADS / 32) * rows) {
                float2 acc = make_float2(0.f, 0.f);
                for (int r0w = lane; r0w < rows; r0w += 32 * 4) {              // four loads in flight
                    float2 v[4];
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const int r = r0w + 32 * j;
                        v[j] = r < rows ? part[((size_t)(r % chunks) * nw + r / chunks) * C + c] : make_float2(0.f, 0.f);
                    }
#pragma unroll
                    for (int j = 0; j < 4; ++j) { acc.x += v[j].x; acc.y += v[j].y; }
                }
                acc = warp_sum2(acc);
                if (lane == 0) { a.dbeta[c] = a.accum_params ? a.dbeta[c] + acc.x : acc.x; a.dgamma[c] = a.accum_params ? a.dgamma[c] + acc.y : acc.y; }
            }
        }
        __syncthreads();
    }
    // Per-channel coefficients, two channels per register pair (the arithmetic below is packed fp32: one instruction per
    // channel pair).  With d = x - mean and scale = gamma * invstd the input gradient gamma * invstd * (dy - c1 - xhat * c2)
    // is scale * dy + (d * ka + kb), ka = -scale * invstd * c2, kb = -scale * c1; sum dy * xhat = invstd * sum dy * d.
    float2 s1[BP], s2[BP], nmean[BP], is[BP], ga[BP], be[BP], sc[BP], ka[BP], kb[BP];
    const float inv_n = 1.f / (float)a.rpw;
#pragma unroll
    for (int j = 0; j < BP; ++j) {
        float* const f1 = &s1[j].x; float* const f2 = &s2[j].x; float* const fnm = &nmean[j].x; float* const fis = &is[j].x;
        float* const fga = &ga[j].x; float* const fbe = &be[j].x; float* const fsc = &sc[j].x; float* const fka = &ka[j].x; float* const fkb = &kb[j].x;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int c = cg * BV + 2 * j + h;
            const size_t so = ((size_t)w * C + c) * 2;
            f1[h] = 0.f; f2[h] = 0.f;
            if (MODE != 0) { fnm[h] = -a.stats[so]; fis[h] = a.stats[so + 1]; fga[h] = a.gamma[c]; fbe[h] = a.beta[c]; }
            if (MODE == 3) {
                const float c1 = red_s[c].x * inv_n, c2 = red_s[c].y * inv_n;
                fsc[h] = fga[h] * fis[h]; fka[h] = -fsc[h] * fis[h] * c2; fkb[h] = -fsc[h] * c1;
            }
        }
    }
    const bool need_out = (MODE == 1 || MODE == 3) && a.relu && !a.mask_from_x;
    const bool res_in_ring = MODE == 2 && a.res && n_in > 1;
    bool ok = true;
    for (int i = 0; i < ntiles; ++i) {
        // every thread left tile i - 1 at the barrier below, so its stage can take tile i + stages - 1
        if (tid == 0 && i + stages - 1 < ntiles) issue(i + stages - 1);
        const int st = i % stages;
        if (ok && !bns_wait(full0 + 8 * st, (uint32_t)(i / stages) & 1u, a.err)) ok = false;
        const uint8_t* sx = bns_sm + (size_t)(st * n_in) * BNS_TILE + tid * 16;      // row lr, channel group cg: vector lr * cgs + cg = tid + k * 256
        const long trow = r0 + (long)(a.reverse ? ntiles - 1 - i : i) * tile_rows;
        const size_t o0 = wbase + (size_t)trow * C + (size_t)tid * BV;
        const int vec_rows = ok ? (int)min((long)tile_rows, r1 - trow) : 0;            // rows of this tile that exist
        // one 16-byte vector (row rl + k * rows_it of the tile, channel group cg) per call
        auto vec = [&](const int k) {
            const uint4 xw = *(const uint4*)(sx + k * (BNV_THREADS * 16));
            const size_t o = o0 + (size_t)k * (BNV_THREADS * BV);
            float2 xv[BP];
            unpack8(xw, xv);
            if (MODE == 0) {
#pragma unroll
                for (int j = 0; j < BP; ++j) { s1[j] = __fadd2_rn(s1[j], xv[j]); s2[j] = __ffma2_rn(xv[j], xv[j], s2[j]); }
            } else if (MODE == 2) {
#pragma unroll
                for (int j = 0; j < BP; ++j) xv[j] = bn_pair(xv[j], nmean[j], is[j], ga[j], be[j]);
                if (a.res) {
                    float2 rv[BP];
                    unpack8(res_in_ring ? *(const uint4*)(sx + BNS_TILE + k * (BNV_THREADS * 16)) : __ldg((const uint4*)(a.res + o)), rv);
#pragma unroll
                    for (int j = 0; j < BP; ++j) xv[j] = __fadd2_rn(xv[j], rv[j]);
                }
                *(uint4*)(a.y + o) = a.relu ? pack8<true>(xv) : pack8<false>(xv);
            } else {
                float2 dv[BP];
                unpack8(*(const uint4*)(sx + BNS_TILE + k * (BNV_THREADS * 16)), dv);
#pragma unroll
                for (int j = 0; j < BP; ++j) xv[j] = __fadd2_rn(xv[j], nmean[j]);          // d = x - mean from here on
                if (a.relu) {
                    float2 f[BP];
                    if (need_out) unpack8(*(const uint4*)(sx + 2 * BNS_TILE + k * (BNV_THREADS * 16)), f);
                    else {
#pragma unroll
                        for (int j = 0; j < BP; ++j) f[j] = __ffma2_rn(ga[j], __fmul2_rn(xv[j], is[j]), be[j]);   // bn_pair after its first step
                    }
#pragma unroll
                    for (int j = 0; j < BP; ++j) { if (!(f[j].x > 0.f)) dv[j].x = 0.f; if (!(f[j].y > 0.f)) dv[j].y = 0.f; }
                }
                if (MODE == 1) {
#pragma unroll
                    for (int j = 0; j < BP; ++j) { s1[j] = __fadd2_rn(s1[j], dv[j]); s2[j] = __ffma2_rn(dv[j], xv[j], s2[j]); }
                } else {
                    if (a.y) {
                        float2 t[BP];
#pragma unroll
                        for (int j = 0; j < BP; ++j) t[j] = __ffma2_rn(sc[j], dv[j], __ffma2_rn(xv[j], ka[j], kb[j]));
                        if (a.accum_dx) {
                            float2 old[BP]; unpack8(*(const uint4*)(a.y + o), old);
#pragma unroll
                            for (int j = 0; j < BP; ++j) t[j] = __fadd2_rn(t[j], old[j]);
                        }
                        *(uint4*)(a.y + o) = pack8<false>(t);
                    }
                    if (a.dres) {
                        if (a.accum_dres) {
                            float2 old[BP]; unpack8(*(const uint4*)(a.dres + o), old);
#pragma unroll
                            for (int j = 0; j < BP; ++j) dv[j] = __fadd2_rn(dv[j], old[j]);
                        }
                        *(uint4*)(a.dres + o) = pack8<false>(dv);
                    }
                }
            }
        };
        if (vec_rows == tile_rows) {
            // a whole tile: no per-vector test, so that the four vectors of a thread are independent instruction streams
#pragma unroll
            for (int k = 0; k < BNS_VPT; ++k) vec(k);
        } else {
#pragma unroll
            for (int k = 0; k < BNS_VPT; ++k) if (rl + k * rows_it < vec_rows) vec(k);
        }
        __syncthreads();
    }
    if (MODE == 0 || MODE == 1) {
        // the ring is idle now (every issued tile was waited for): reuse it for the reduction over the row lanes
        float (*red_sh)[2 * BV + 1] = (float (*)[2 * BV + 1])bns_sm;
#pragma unroll
        for (int j = 0; j < BP; ++j) {
            if (MODE == 1) s2[j] = __fmul2_rn(s2[j], is[j]);            // sum dy * d -> sum dy * xhat
            red_sh[tid][2 * j] = s1[j].x; red_sh[tid][2 * j + 1] = s1[j].y; red_sh[tid][BV + 2 * j] = s2[j].x; red_sh[tid][BV + 2 * j + 1] = s2[j].y;
        }
        __syncthreads();
        // thread t < 2*BV*cgs sums one (channel group, value) column over the rows_it row lanes, in a fixed order
        for (int t = tid; t < cgs * 2 * BV; t += BNV_THREADS) {
            const int q = t / (2 * BV), k = t % (2 * BV);
            float acc = 0.f;
            for (int rr = 0; rr < rows_it; ++rr) acc += red_sh[rr * cgs + q][k];
            const int c = q * BV + (k % BV);
            a.part[(((size_t)blockIdx.x * nw + w) * C + c) * 2 + (k / BV)] = acc;
        }
    }
}

// One warp per (worker, channel): lanes take the chunk partials round-robin, then a fixed shuffle tree adds the
// lanes, so the summation order never changes.  stats[w][c] = (mean, invstd).
__global__ void bnv_stats_final(const float* __restrict__ part, float* __restrict__ stats, int chunks, int nwC, long rpw) {
    const int i = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (i >= nwC) return;
    float2 a = make_float2(0.f, 0.f);
    for (int k = lane; k < chunks; k += 32) { const float2 v = *(const float2*)(part + ((size_t)k * nwC + i) * 2); a.x += v.x; a.y += v.y; }
    a = warp_sum2(a);
    if (lane == 0) {
        const double mean = (double)a.x / (double)rpw;
        double var = (double)a.y / (double)rpw - mean * mean;
        if (var < 0.0) var = 0.0;
        *(float2*)(stats + (size_t)i * 2) = make_float2((float)mean, (float)(1.0 / sqrt(var + 1e-5)));
    }
}
// same, from the partials a convolution epilogue left: [w * cpw + k][C][2], k < cpw.  One block of 256 threads per
// (worker, 4 channels): a thread owns one channel and every 64th partial, so that a warp's loads cover whole
// 32-byte sectors; then a fixed-order tree over the 64 partial lanes in shared memory.
__global__ void __launch_bounds__(256) bnv_stats_final_tiles(const float* __restrict__ part, float* __restrict__ stats, int cpw, int nw, int C, long rpw) {
    __shared__ float2 sh[64][5];
    const int w = blockIdx.y, tid = threadIdx.x, cl = tid & 3, kl = tid >> 2;
    const int c = blockIdx.x * 4 + cl;
    const float* p = part + ((size_t)w * cpw * C + c) * 2;
    float2 a = make_float2(0.f, 0.f);
    int k = kl;
    for (; k + 448 < cpw; k += 512) {                      // eight independent loads in flight
        float2 v[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) v[j] = *(const float2*)(p + (size_t)(k + 64 * j) * C * 2);
        a.x += ((v[0].x + v[1].x) + (v[2].x + v[3].x)) + ((v[4].x + v[5].x) + (v[6].x + v[7].x));
        a.y += ((v[0].y + v[1].y) + (v[2].y + v[3].y)) + ((v[4].y + v[5].y) + (v[6].y + v[7].y));
    }
    for (; k + 192 < cpw; k += 256) {                      // four
        const float2 v0 = *(const float2*)(p + (size_t)k * C * 2), v1 = *(const float2*)(p + (size_t)(k + 64) * C * 2);
        const float2 v2 = *(const float2*)(p + (size_t)(k + 128) * C * 2), v3 = *(const float2*)(p + (size_t)(k + 192) * C * 2);
        a.x += (v0.x + v1.x) + (v2.x + v3.x); a.y += (v0.y + v1.y) + (v2.y + v3.y);
    }
    for (; k < cpw; k += 64) { const float2 v = *(const float2*)(p + (size_t)k * C * 2); a.x += v.x; a.y += v.y; }
    sh[kl][cl] = a;
    __syncthreads();
    for (int d = 32; d > 0; d >>= 1) {
        if (kl < d) { sh[kl][cl].x += sh[kl + d][cl].x; sh[kl][cl].y += sh[kl + d][cl].y; }
        __syncthreads();
    }
    if (kl == 0) {
        const double mean = (double)sh[0][cl].x / (double)rpw;
        double var = (double)sh[0][cl].y / (double)rpw - mean * mean;
        if (var < 0.0) var = 0.0;
        *(float2*)(stats + ((size_t)w * C + c) * 2) = make_float2((float)mean, (float)(1.0 / sqrt(var + 1e-5)));
    }
}
static bool bnv_ok(int dt, int C) { int cgs = C / BV; return dt == 1 && C % BV == 0 && cgs <= BNV_THREADS && (cgs & (cgs - 1)) == 0; }
constexpr int BNS_SMEM = BNS_RING + 8 * 8;
constexpr int BNS_RED_BYTES = BNV_THREADS * BV * 8;   // backward apply: (sum dy, sum dy xhat) per channel, up to 256 * 8 channels (C <= 256: + 256 subset sums)
// Row chunks per worker such that chunks * nw CTAs fill the SMs the caller sizes for once (two CTAs per SM; 0: all SMs),
// each with at least four tiles.
static int bn_device_sms() {
    static int sms = 0;
    if (!sms) { int dev = 0; cudaGetDevice(&dev); cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev); if (sms <= 0) sms = 148; }
    return sms;
}
static int bns_chunks(int nw, long rpw, int C, int sms_wanted) {
    const int sms = sms_wanted > 0 && sms_wanted < bn_device_sms() ? sms_wanted : bn_device_sms();
    const long tile_rows = BNS_TILE / (C * 2);
    long want = ((long)sms * BNS_CTAS) / nw, maxc = (rpw + tile_rows * 4 - 1) / (tile_rows * 4);
    long c = want < maxc ? want : maxc;
    if (c > BNV_MAX_CHUNKS) c = BNV_MAX_CHUNKS;
    return (int)(c < 1 ? 1 : c);
}
template <int MODE>
static void bns_launch(const BnsArgs& a, int chunks, int nw, cudaStream_t s) {
    constexpr int smem = BNS_SMEM + (MODE == 3 ? BNS_RED_BYTES : 0);
    static OncePerDevice once;
    allow_smem(once, (const void*)bns_kernel<MODE>, smem);
    klaunch(bns_kernel<MODE>, dim3(chunks, nw), BNV_THREADS, smem, s, a);
}

bool bn_accepts_conv_partials(int dt, int C) { return bnv_ok(dt, C); }

void bn_forward(int dt, const void* x, const float* gamma, const float* beta, const void* res, void* y, float* stats,
                float* scratch, int nw, long rpw, int C, bool relu, const float* conv_part, int conv_chunks, int sms, int* err, cudaStream_t s) {
    if (bnv_ok(dt, C) && err) {
        const int chunks = bns_chunks(nw, rpw, C, sms);
        const double total = (double)nw * rpw * C;
        BnsArgs a{};
        a.in[0] = (const bf16*)x; a.n_in = 1; a.gamma = gamma; a.beta = beta; a.stats = stats; a.rpw = rpw; a.C = C; a.relu = relu; a.err = err;
        if (conv_part) {
            Scope sc(KC_BN_FWD_STATS, 0.0, 8.0 * conv_chunks * nw * C, s);
            klaunch(bnv_stats_final_tiles, dim3(C / 4, nw), 256, 0, s, conv_part, stats, conv_chunks, nw, C, rpw);
        } else if (conv_chunks >= 0) {
            { Scope sc(KC_BN_FWD_STATS, 0.0, 2.0 * total, s);
              BnsArgs r = a; r.part = scratch;
              bns_launch<0>(r, chunks, nw, s); }
            { Scope sc(KC_BN_FWD_STATS, 0.0, 8.0 * chunks * nw * C, s);
              klaunch(bnv_stats_final, cdiv((size_t)nw * C * 32, 256), 256, 0, s, scratch, stats, chunks, nw * C, rpw); }
        }
        Scope sc(KC_BN_FWD_APPLY, 0.0, 2.0 * total * (res ? 3 : 2), s);
        a.y = (bf16*)y; a.res = (const bf16*)res;
        if (res) { a.in[1] = (const bf16*)res; a.n_in = 2; }
        a.reverse = conv_part || conv_chunks < 0 ? 0 : 1;       // after a statistics pass of its own: x was just read front to back
        bns_launch<2>(a, chunks, nw, s);
        return;
    }
    int chunks = (int)(rpw < RED_CHUNKS ? rpw : RED_CHUNKS);
    dim3 grid(cdiv(C, 32), chunks, nw), blk(32, 8);
    const double esz_ = dt ? 2.0 : 4.0;
    size_t total = (size_t)nw * rpw * C;
    { Scope sc(KC_BN_FWD_STATS, 0.0, esz_ * total, s);
      if (dt) klaunch(bn_reduce_partial<bf16, false>, grid, blk, 0, s, (const bf16*)x, nullptr, nullptr, nullptr, scratch, rpw, C, false);
      else klaunch(bn_reduce_partial<float, false>, grid, blk, 0, s, (const float*)x, nullptr, nullptr, nullptr, scratch, rpw, C, false); }
    { Scope sc(KC_BN_FWD_STATS, 0.0, 8.0 * chunks * nw * C, s);
      if (dt) klaunch(bn_stats_final<bf16>, cdiv((size_t)nw * C, 128), 128, 0, s, scratch, (const bf16*)x, stats, chunks, nw * C, C, rpw);
      else klaunch(bn_stats_final<float>, cdiv((size_t)nw * C, 128), 128, 0, s, scratch, (const float*)x, stats, chunks, nw * C, C, rpw); }
    Scope sc(KC_BN_FWD_APPLY, 0.0, esz_ * total * (res ? 3 : 2), s);
    if (dt) klaunch(bn_apply_k<bf16>, cdiv(total, 256), 256, 0, s, (const bf16*)x, gamma, beta, (const bf16*)res, (bf16*)y, stats, rpw, C, total, relu);
    else klaunch(bn_apply_k<float>, cdiv(total, 256), 256, 0, s, (const float*)x, gamma, beta, (const float*)res, (float*)y, stats, rpw, C, total, relu);
}

void bn_backward(int dt, const void* x, const void* out, const void* dout, const float* gamma, const float* beta,
                 const float* stats, void* dx, bool accum_dx, void* dres, bool accum_dres, float* dgamma, float* dbeta, float* red,
                 float* scratch, int nw, long rpw, int C, bool relu, bool has_res, bool accum_params, int sms, int* err, cudaStream_t s) {
    if (bnv_ok(dt, C) && err) {
        const int chunks = bns_chunks(nw, rpw, C, sms);
        const double total = (double)nw * rpw * C;
        const int mask_from_x = relu && !has_res;
        const bool need_out = relu && !mask_from_x;
        const int reads = 2 + (need_out ? 1 : 0);
        BnsArgs a{};
        a.in[0] = (const bf16*)x; a.in[1] = (const bf16*)dout; a.in[2] = (const bf16*)out; a.n_in = reads;
        a.gamma = gamma; a.beta = beta; a.stats = stats; a.rpw = rpw; a.C = C; a.relu = relu; a.mask_from_x = mask_from_x; a.err = err;
        { Scope sc(KC_BN_BWD_REDUCE, 0.0, 2.0 * total * reads, s);
          BnsArgs r = a; r.part = scratch;
          bns_launch<1>(r, chunks, nw, s); }
        Scope sc(KC_BN_BWD_APPLY, 0.0, 2.0 * total * (reads + 1 + (accum_dx ? 1 : 0) + (dres ? (accum_dres ? 2 : 1) : 0)), s);
        a.y = (bf16*)dx; a.accum_dx = accum_dx; a.dres = (bf16*)dres; a.accum_dres = accum_dres;
        a.part = scratch; a.dgamma = dgamma; a.dbeta = dbeta; a.accum_params = accum_params;   // the apply kernel finishes the sums itself
        a.reverse = 1;                       // the sums kernel above has just read the same tensors front to back
        bns_launch<3>(a, chunks, nw, s);
        return;
    }
    int chunks = (int)(rpw < RED_CHUNKS ? rpw : RED_CHUNKS);
    dim3 grid(cdiv(C, 32), chunks, nw), blk(32, 8);
    const double esz_ = dt ? 2.0 : 4.0;
    size_t total = (size_t)nw * rpw * C;
    { Scope sc(KC_BN_BWD_REDUCE, 0.0, esz_ * total * (relu ? 3 : 2), s);
      if (dt) klaunch(bn_reduce_partial<bf16, true>, grid, blk, 0, s, (const bf16*)x, (const bf16*)out, (const bf16*)dout, stats, scratch, rpw, C, relu);
      else klaunch(bn_reduce_partial<float, true>, grid, blk, 0, s, (const float*)x, (const float*)out, (const float*)dout, stats, scratch, rpw, C, relu); }
    { Scope sc(KC_BN_BWD_REDUCE, 0.0, 8.0 * chunks * nw * C, s);
      klaunch(bn_bwd_final, cdiv(C, 128), 128, 0, s, scratch, red, dgamma, dbeta, chunks, nw, C, accum_params); }
    Scope sc(KC_BN_BWD_APPLY, 0.0, esz_ * total * ((relu ? 3 : 2) + 1 + (dres ? (accum_dres ? 2 : 1) : 0) + (accum_dx ? 1 : 0)), s);
    if (dt) klaunch(bn_bwd_apply_k<bf16>, cdiv(total, 256), 256, 0, s, (const bf16*)x, (const bf16*)out, (const bf16*)dout, gamma, stats, red,
                                                                  (bf16*)dx, accum_dx, (bf16*)dres, accum_dres, rpw, C, total, relu);
    else klaunch(bn_bwd_apply_k<float>, cdiv(total, 256), 256, 0, s, (const float*)x, (const float*)out, (const float*)dout, gamma, stats, red,
                                                                (float*)dx, accum_dx, (float*)dres, accum_dres, rpw, C, total, relu);
}

// ------------------------------------------------------------------------------------------
// softmax cross-entropy: one block; thread i handles rows i, i+256, ...; fixed-order tree sum
// ------------------------------------------------------------------------------------------
// The loss goes straight to the host (a record in pinned memory): loss and error word first, then the number the host waits for.
__device__ __forceinline__ void publish_loss(LossRecord* rec, float loss, const int* err, long long seq) {
    volatile LossRecord* const r = rec;
    r->loss = loss;
    r->err = err ? *(const volatile int*)err : 0;
    __threadfence_system();
    r->seq = seq;
}
__global__ void stamp_k(long long* stamp) { *stamp = device_time_ns(); }
void stamp_time(long long* stamp, cudaStream_t s) {
    Scope sc(KC_FILL, 0.0, 8.0, s);
    klaunch(stamp_k, 1, 1, 0, s, stamp);
}
__global__ void publish_k(LossRecord* rec, float loss, const int* err, long long seq) { publish_loss(rec, loss, err, seq); }
void publish_loss_value(LossRecord* rec, float loss, const int* err, long long seq, cudaStream_t s) {
    Scope sc(KC_FILL, 0.0, sizeof(LossRecord), s);
    klaunch(publish_k, 1, 1, 0, s, rec, loss, err, seq);
}

template <typename T>
__global__ void softmax_ce_k(const float* __restrict__ z, const int32_t* __restrict__ labels, T* __restrict__ dz,
                             LossRecord* rec, const int* err, long long seq, int M, int C, float scale) {
    __shared__ float sh[256];
    float local = 0.f;
    const float inv_m = 1.f / (float)M;
    // exp / log in double: a few thousand values per step, and it keeps the error of (softmax - onehot) at the rounding
    // of the stored result instead of |z| * ulp(expf)
    for (int r = threadIdx.x; r < M; r += blockDim.x) {
        const float* zr = z + (size_t)r * C;
        float m = zr[0];
        for (int c = 1; c < C; ++c) m = fmaxf(m, zr[c]);
        double se = 0.0;
        for (int c = 0; c < C; ++c) se += exp((double)zr[c] - (double)m);
        const double lse = (double)m + log(se);
        int y = labels[r];
        local += (float)(lse - (double)zr[y]);
        for (int c = 0; c < C; ++c) st(dz + (size_t)r * C + c, (float)((exp((double)zr[c] - lse) - (c == y ? 1.0 : 0.0)) * (double)scale));
    }
    sh[threadIdx.x] = local;
    __syncthreads();
    for (int s = 128; s > 0; s >>= 1) { if ((int)threadIdx.x < s) sh[threadIdx.x] += sh[threadIdx.x + s]; __syncthreads(); }
    if (threadIdx.x == 0) publish_loss(rec, sh[0] * inv_m, err, seq);
}
void softmax_ce(int dt, const float* logits, const int32_t* labels, void* dlogits, LossRecord* rec, const int* err, long long seq, int M, int classes, float scale,
                cudaStream_t s) {
    Scope sc(KC_SOFTMAX_CE, 0.0, (double)M * classes * (dt ? 6.0 : 8.0) + 4.0 * M, s);
    if (dt) klaunch(softmax_ce_k<bf16>, 1, 256, 0, s, logits, labels, (bf16*)dlogits, rec, err, seq, M, classes, scale);
    else klaunch(softmax_ce_k<float>, 1, 256, 0, s, logits, labels, (float*)dlogits, rec, err, seq, M, classes, scale);
}

// ------------------------------------------------------------------------------------------
// Classifier head: the network's last linear layer (c_in -> a few classes) fused with the loss.
//   head_fwd_loss_k : one warp per sample: logits = x W^T + b (fp32, kept for the caller), softmax cross-entropy,
//                     dlogits = (softmax - onehot) * scale in the storage dtype, per-CTA loss partials.
//   head_bwd_k      : a CTA owns a range of samples: dx = dlogits W (one warp per sample) and the partial sums of
//                     dW[c][k] = sum_rows dlogits[row][c] x[row][k] and db[c] = sum_rows dlogits[row][c] (column k = K).
//   head_reduce_k   : dW / db = partials added in CTA order; one CTA more adds the loss partials and hands the mean loss to the host.
// The first two stand in the last module's chain, so latency is all that counts: operands come in one round trip to L2 (weights and tiles through shared
// memory, HEAD_W_SMEM, HEAD_STAGE_VECS; a loop over the classes waited for four to eight), and what waits for other CTAs or for the host's memory is in
// the third, off the chain.  512 samples, 1024 columns, 10 classes in bf16, cold: forward 20.3 -> 9.9 us, backward 10.5 -> 8.0; steps of the 512-wide fp32 MLP 62 -> 58 us.
// Replaces an implicit-GEMM launch on 64 x 64 tiles (8-16 CTAs), a one-CTA loss kernel, two bias-gradient launches, a
// split weight gradient with its reduction and an input-gradient launch.  classes <= 16, c_in a multiple of the vector width.
// ------------------------------------------------------------------------------------------
constexpr int HEAD_MAX_C = 16;
constexpr int HEAD_ROWS_PER_CTA = 32;       // samples per CTA of head_bwd_k
constexpr size_t HEAD_W_SMEM = 40 * 1024;   // a larger W is read from L2 by every warp (static and dynamic shared memory stay below the 48 KB of any launch)
constexpr int HEAD_STAGE_VECS = 32;         // wider slices are there for many samples, where other CTAs cover the latency
// W_SMEM: W fits into HEAD_W_SMEM (a kernel of its own: through a pointer to either, loads from L2 are no longer known to be of constant global memory:
// one bf16 layer of 4096 columns and 16 classes, one sample, 68 us a step instead of 47)
template <typename T, bool W_SMEM>
__global__ void __launch_bounds__(256) head_fwd_loss_k(const T* __restrict__ x, const T* __restrict__ W, const float* __restrict__ bias,
                                                       const int32_t* __restrict__ labels, float* __restrict__ logits, T* __restrict__ dz,
                                                       float* __restrict__ loss_part, int M, int K, int C, float scale) {
    constexpr int V = Vec<T>::V;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int row = blockIdx.x * 8 + warp;
    __shared__ float wl[8];
    extern __shared__ __align__(16) char hsm[];
    if constexpr (W_SMEM) {                  // all of W, 16 bytes a thread at a time
        for (int i = threadIdx.x; i < C * K / V; i += 256) ((uint4*)hsm)[i] = ((const uint4*)W)[i];
        __syncthreads();
    }
    float rloss = 0.f;
    if (row < M) {
        float acc[HEAD_MAX_C];
#pragma unroll
        for (int c = 0; c < HEAD_MAX_C; ++c) acc[c] = 0.f;
        const T* xr = x + (size_t)row * K;
        for (int kv = lane; kv < K / V; kv += 32) {
            float xv[8];
            Vec<T>::load(xr + (size_t)kv * V, xv);
#pragma unroll
            for (int c = 0; c < HEAD_MAX_C; c += 8) {            // eight classes' loads in flight; a class that does not exist repeats the last one
                if (c >= C) break;
                float wv[8][8];
#pragma unroll
                for (int q = 0; q < 8; ++q) Vec<T>::load((W_SMEM ? (const T*)hsm : W) + (size_t)min(c + q, C - 1) * K + (size_t)kv * V, wv[q]);
#pragma unroll
                for (int q = 0; q < 8; ++q)
#pragma unroll
                    for (int j = 0; j < V; ++j) acc[c + q] = fmaf(xv[j], wv[q][j], acc[c + q]);
            }
        }
        float z = 0.f;                       // lane c keeps logit c
#pragma unroll
        for (int c = 0; c < HEAD_MAX_C; ++c) {
            if (c >= C) break;
            float v = acc[c];
#pragma unroll
            for (int d = 16; d > 0; d >>= 1) v += __shfl_xor_sync(0xffffffffu, v, d);
            if (lane == c) z = v + (bias ? bias[c] : 0.f);
        }
        const bool mine = lane < C;
        if (mine) logits[(size_t)row * C + lane] = z;
        float m = mine ? z : -INFINITY;
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, d));
        // exp / log in double: it keeps the error of (softmax - onehot) at the rounding of the stored result
        double e = mine ? exp((double)z - (double)m) : 0.0;
        double se = e;
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) se += __shfl_xor_sync(0xffffffffu, se, d);
        const double lse = (double)m + log(se);
        const int y = labels[row];
        const float zy = __shfl_sync(0xffffffffu, z, y);
        rloss = (float)(lse - (double)zy);
        if (mine) st(dz + (size_t)row * C + lane, (float)((e / se - (lane == y ? 1.0 : 0.0)) * (double)scale));
    }
    if (lane == 0) wl[warp] = rloss;
    __syncthreads();
    if (threadIdx.x == 0) {
        float s = 0.f;
        for (int i = 0; i < 8; ++i) s += wl[i];
        loss_part[blockIdx.x] = s;
    }
}
// grid = (ceil(M / HEAD_ROWS_PER_CTA), slices of `kvs` vectors of the K columns): the sums over a CTA's 32 samples are serial chains, so the
// columns are what is spread over the device.  part: [CTA row][C][K + 1].
// mask: the head's input is the output of a ReLU layer: dx *= (x > 0), and col receives the column sums of the masked dx (that layer's bias
// gradient), [CTA row][K][2].
template <typename T>
__global__ void __launch_bounds__(256) head_bwd_k(const T* __restrict__ x, const T* __restrict__ W, const T* __restrict__ dz, T* dx, float* __restrict__ part,
                                                  float* __restrict__ col, int M, int K, int C, int kvs, bool accum_dx, bool mask, bool staged) {
    constexpr int V = Vec<T>::V;
    const int r0 = blockIdx.x * HEAD_ROWS_PER_CTA, r1 = min(M, r0 + HEAD_ROWS_PER_CTA);
    const int nkv = K / V, kv0 = blockIdx.y * kvs, nk = min(nkv - kv0, kvs);
    __shared__ float dzs[HEAD_ROWS_PER_CTA][HEAD_MAX_C];
    __shared__ float cs[256][V + 1];
    extern __shared__ __align__(16) char hsm[];
    // this CTA's part of x and of W; staged (kvs <= HEAD_STAGE_VECS): copies [rows][kvs], [C][kvs] in shared memory
    const T* xp = x + (size_t)r0 * K + (size_t)kv0 * V;
    const T* wp = W + (size_t)kv0 * V;
    size_t pitch = K;
    if (staged) {
        uint4* const xs = (uint4*)hsm;
        for (int i = threadIdx.x; i < (r1 - r0 + C) * kvs; i += 256) {
            const int r = i / kvs, kv = i - r * kvs;
            if (kv < nk) xs[i] = *(const uint4*)(r < r1 - r0 ? xp + (size_t)r * K + kv * V : wp + (size_t)(r - (r1 - r0)) * K + kv * V);
        }
        xp = (const T*)xs; wp = (const T*)(xs + (size_t)(r1 - r0) * kvs); pitch = (size_t)kvs * V;
    }
    for (int i = threadIdx.x; i < (r1 - r0) * C; i += 256) dzs[i / C][i % C] = ld(dz + (size_t)r0 * C + i);
    __syncthreads();
    if (dx) {
        // thread = one vector of columns for every (256 / kvs)-th sample
        const int kv = threadIdx.x % kvs, rl = threadIdx.x / kvs, rstep = 256 / kvs;
        float sum[8];
#pragma unroll
        for (int j = 0; j < V; ++j) sum[j] = 0.f;
        if (kv < nk && rl < rstep)
            for (int r = r0 + rl; r < r1; r += rstep) {
                float a[8];
#pragma unroll
                for (int j = 0; j < V; ++j) a[j] = 0.f;
                for (int c = 0; c < C; ++c) {
                    float wv[8];
                    Vec<T>::load(wp + c * pitch + kv * V, wv);
                    const float g = dzs[r - r0][c];
#pragma unroll
                    for (int j = 0; j < V; ++j) a[j] = fmaf(g, wv[j], a[j]);
                }
                T* d = dx + (size_t)r * K + (size_t)(kv0 + kv) * V;
                if (accum_dx) {
                    float old[8];
                    Vec<T>::load(d, old);
#pragma unroll
                    for (int j = 0; j < V; ++j) a[j] += old[j];
                }
                if (mask) {
                    float xv[8];
                    Vec<T>::load(xp + (r - r0) * pitch + kv * V, xv);
#pragma unroll
                    for (int j = 0; j < V; ++j) { if (!(xv[j] > 0.f)) a[j] = 0.f; sum[j] += rounded<T>(a[j]); }
                }
                Vec<T>::store(d, a);
            }
        if (mask && col) {
#pragma unroll
            for (int j = 0; j < V; ++j) cs[threadIdx.x][j] = sum[j];
            __syncthreads();
            for (int t = threadIdx.x; t < nk * V; t += 256) {
                float a = 0.f;
                for (int q = 0; q < rstep; ++q) a += cs[q * kvs + t / V][t % V];
                col[((size_t)blockIdx.x * K + kv0 * V + t) * 2] = a;
            }
        }
    }
    // partial sums: (class, vector of V columns) pairs round-robin over the threads, rows in ascending order
    float* out = part + (size_t)blockIdx.x * C * (K + 1);
    for (int p = threadIdx.x; p < C * nk; p += 256) {
        const int c = p / nk, kv = p - c * nk;
        float a[8];
#pragma unroll
        for (int j = 0; j < V; ++j) a[j] = 0.f;
#pragma unroll 8
        for (int r = r0; r < r1; ++r) {
            float xv[8];
            Vec<T>::load(xp + (r - r0) * pitch + kv * V, xv);
            const float g = dzs[r - r0][c];
#pragma unroll
            for (int j = 0; j < V; ++j) a[j] = fmaf(g, xv[j], a[j]);
        }
#pragma unroll
        for (int j = 0; j < V; ++j) out[(size_t)c * (K + 1) + (kv0 + kv) * V + j] = a[j];
    }
    if (blockIdx.y == 0 && threadIdx.x < C) {
        float a = 0.f;
        for (int r = r0; r < r1; ++r) a += dzs[r - r0][threadIdx.x];
        out[(size_t)threadIdx.x * (K + 1) + K] = a;
    }
}
// blockDim = (elements, lanes): lane y adds the CTAs y, y + lanes, ...  The last CTA: the mean of the M losses from `blocks` partials, for the host.
__global__ void head_reduce_k(const float* __restrict__ part, float* __restrict__ dW, float* __restrict__ db, int ctas, int K, int C, const float* __restrict__ loss_part,
                              int blocks, int M, LossRecord* rec, const int* err, long long seq) {
    if (blockIdx.x == gridDim.x - 1) {
        __shared__ double ls[256];
        const int tid = threadIdx.y * blockDim.x + threadIdx.x, nt = blockDim.x * blockDim.y;      // nt: a power of two
        double s = 0.0;
        for (int i = tid; i < blocks; i += nt) s += (double)loss_part[i];
        ls[tid] = s;
        __syncthreads();
        for (int d = nt / 2; d > 0; d >>= 1) { if (tid < d) ls[tid] += ls[tid + d]; __syncthreads(); }
        if (tid == 0) publish_loss(rec, (float)(ls[0] / (double)M), err, seq);
        return;
    }
    __shared__ float sh[8][32];
    const int i = blockIdx.x * blockDim.x + threadIdx.x, lanes = blockDim.y, n = C * (K + 1);
    float s = 0.f;
    if (i < n) {
#pragma unroll 8
        for (int b = threadIdx.y; b < ctas; b += lanes) s += part[(size_t)b * n + i];
    }
    if (lanes > 1) {
        sh[threadIdx.y][threadIdx.x] = s;
        __syncthreads();
        if (threadIdx.y > 0) return;
        for (int y = 1; y < lanes; ++y) s += sh[y][threadIdx.x];
    }
    if (i >= n) return;
    const int c = i / (K + 1), k = i - c * (K + 1);
    if (k < K) dW[(size_t)c * K + k] = s;
    else if (db) db[c] = s;
}
bool head_supported(int dt, int K, int C) { return C >= 2 && C <= HEAD_MAX_C && K % (dt ? 8 : 4) == 0; }
size_t head_scratch_elems(int M, int K, int C) {
    const size_t ctas = (M + HEAD_ROWS_PER_CTA - 1) / HEAD_ROWS_PER_CTA;
    return ctas * C * (K + 1) + (M + 7) / 8;
}
void head_forward_loss(int dt, const void* x, const void* W, const float* bias, const int32_t* labels, float* logits, void* dlogits, float* loss_part, int M, int K, int C,
                       float scale, cudaStream_t s) {
    Scope sc(KC_SOFTMAX_CE, 2.0 * M * K * C, (dt ? 2.0 : 4.0) * ((double)M * K + (double)C * K + (double)M * C) + 4.0 * M * C, s);
    const unsigned grid = (M + 7) / 8;
    const size_t w_bytes = (size_t)C * K * (dt ? 2 : 4), smem = w_bytes <= HEAD_W_SMEM ? w_bytes : 0;
    if (dt) klaunch(smem ? head_fwd_loss_k<bf16, true> : head_fwd_loss_k<bf16, false>, grid, 256, smem, s, (const bf16*)x, (const bf16*)W, bias, labels, logits, (bf16*)dlogits, loss_part, M, K, C,
                    scale);
    else klaunch(smem ? head_fwd_loss_k<float, true> : head_fwd_loss_k<float, false>, grid, 256, smem, s, (const float*)x, (const float*)W, bias, labels, logits, (float*)dlogits, loss_part, M, K, C,
                 scale);
}
int head_col_records(int M) { return (M + HEAD_ROWS_PER_CTA - 1) / HEAD_ROWS_PER_CTA; }
void head_backward(int dt, const void* x, const void* W, const void* dlogits, void* dx_or_null, bool accum_dx, bool mask_dx, float* col_or_null, float* scratch, int M,
                   int K, int C, cudaStream_t s) {
    const unsigned ctas = (M + HEAD_ROWS_PER_CTA - 1) / HEAD_ROWS_PER_CTA;
    const int nkv = K / (dt ? 8 : 4);
    // vectors of columns per CTA: a power of two that puts about one CTA on every SM, at least eight (a warp then reads whole sectors), and no
    // more than there are: the other threads take other samples (16384 samples, 256 columns in bf16: 50 us with 256 whatever there are, 31 so)
    int kvs = 8;
    while (kvs < 256 && kvs < nkv) kvs *= 2;
    while (kvs > 8 && ctas * ((nkv + kvs - 1) / kvs) < 148) kvs /= 2;
    const dim3 grid(ctas, (nkv + kvs - 1) / kvs);
    const bool staged = kvs <= HEAD_STAGE_VECS;
    const size_t smem = staged ? (size_t)(HEAD_ROWS_PER_CTA + C) * kvs * 16 : 0;
    Scope sc(KC_FMA_WGRAD, (dx_or_null ? 4.0 : 2.0) * M * K * C, (dt ? 2.0 : 4.0) * ((double)M * K * (dx_or_null ? 2 : 1) + (double)C * K + (double)M * C), s);
    if (dt) klaunch(head_bwd_k<bf16>, grid, 256, smem, s, (const bf16*)x, (const bf16*)W, (const bf16*)dlogits, (bf16*)dx_or_null, scratch, col_or_null, M, K, C, kvs, accum_dx, mask_dx, staged);
    else klaunch(head_bwd_k<float>, grid, 256, smem, s, (const float*)x, (const float*)W, (const float*)dlogits, (float*)dx_or_null, scratch, col_or_null, M, K, C, kvs, accum_dx, mask_dx, staged);
}
void head_reduce(float* dW, float* db_or_null, const float* scratch, const float* loss_part, LossRecord* rec, const int* err, long long seq, int M, int K, int C, cudaStream_t s) {
    const unsigned ctas = (M + HEAD_ROWS_PER_CTA - 1) / HEAD_ROWS_PER_CTA;
    Scope sc(KC_SPLITK, 0.0, 4.0 * (ctas + 1) * C * (K + 1), s);
    // from 65 partial matrices on eight threads per element (512 of them, 2570 elements: 62 us with one, 10 so; 68: 15 and 7)
    const bool many = ctas > 64;
    klaunch(head_reduce_k, cdiv((size_t)C * (K + 1), many ? 32 : 64) + 1, many ? dim3(32, 8) : dim3(64), 0, s, scratch, dW, db_or_null, (int)ctas, K, C, loss_part, (M + 7) / 8, M, rec,
            err, seq);
}

// ------------------------------------------------------------------------------------------
// SGD update fused with the emission of the next weight version (Eq. dl_update with P = 11^T/N)
// 128-bit loads and stores; grid sized to a multiple of the SM count by the grid-stride loop.
// ------------------------------------------------------------------------------------------
template <typename T>
__global__ void sgd_k(float4* __restrict__ master, const float4* __restrict__ grad, T* __restrict__ copy, size_t n4, float lr, long long* stamp) {
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n4; i += (size_t)gridDim.x * blockDim.x) {
        float4 w = master[i];
        if (grad) {
            float4 g = grad[i];
            w.x = fmaf(-lr, g.x, w.x); w.y = fmaf(-lr, g.y, w.y); w.z = fmaf(-lr, g.z, w.z); w.w = fmaf(-lr, g.w, w.w);
            master[i] = w;
        }
        if (sizeof(T) == 4) {
            ((float4*)copy)[i] = w;
        } else {
            __nv_bfloat162 lo = __floats2bfloat162_rn(w.x, w.y), hi = __floats2bfloat162_rn(w.z, w.w);
            uint2 pk; pk.x = *(unsigned*)&lo; pk.y = *(unsigned*)&hi;
            ((uint2*)copy)[i] = pk;
        }
    }
    if (stamp && blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) *stamp = device_time_ns();
}
void sgd_update(int dt, float* master, const float* grad, void* copy_next, size_t n, float lr, long long* stamp, cudaStream_t s) {
    size_t n4 = n / 4;
    if (n4 == 0) return;
    unsigned blocks = cdiv(n4, 256);
    if (blocks > 148 * 8) blocks = 148 * 8;
    // per parameter: read master (4) [+ read grad (4) + write master (4)] + write the copy (2 or 4)
    Scope sc(KC_SGD, 0.0, (double)n * ((grad ? 12.0 : 4.0) + (dt ? 2.0 : 4.0)), s);
    if (dt) klaunch(sgd_k<bf16>, blocks, 256, 0, s, (float4*)master, (const float4*)grad, (bf16*)copy_next, n4, lr, stamp);
    else klaunch(sgd_k<float>, blocks, 256, 0, s, (float4*)master, (const float4*)grad, (float*)copy_next, n4, lr, stamp);
}

// ------------------------------------------------------------------------------------------
// General mixing matrix (Eq. dl_update (a), (b)): R replicas of a module's parameters, each with its own gradient.
//   u_r = w_r - lr * g_r ;  w_s(t+1) = sum_r P[s][r] * u_r  (r ascending) ;  copies of w_s(t+1) in the storage dtype.
// A thread owns 4 consecutive parameters of ALL replicas: it reads the R masters (and gradients) first and writes the R
// results afterwards, so the update is in place.  master / grad: [R][n_big + n_small]; the copies of replica r start
// slot_bytes * r after copy0: n_big values in the storage dtype, then n_small floats.
// ------------------------------------------------------------------------------------------
constexpr int MIX_MAX_R = 32;
template <typename T>
__global__ void __launch_bounds__(256) mix_k(float* master, const float* __restrict__ grad, char* copy0, size_t n_big, size_t n_small, size_t slot_bytes,
                                              int R, const float* __restrict__ P, float lr, long long* stamp) {
    __shared__ float Ps[MIX_MAX_R * MIX_MAX_R];
    for (int i = threadIdx.x; i < R * R; i += blockDim.x) Ps[i] = P[i];
    __syncthreads();
    const size_t n = n_big + n_small, n4 = n / 4;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n4; i += (size_t)gridDim.x * blockDim.x) {
        float4 u[MIX_MAX_R];
        for (int r = 0; r < R; ++r) {
            float4 w = ((const float4*)(master + (size_t)r * n))[i];
            if (grad) {
                const float4 g = ((const float4*)(grad + (size_t)r * n))[i];
                w.x = fmaf(-lr, g.x, w.x); w.y = fmaf(-lr, g.y, w.y); w.z = fmaf(-lr, g.z, w.z); w.w = fmaf(-lr, g.w, w.w);
            }
            u[r] = w;
        }
        for (int s = 0; s < R; ++s) {
            float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
            for (int r = 0; r < R; ++r) {
                const float p = Ps[s * R + r];
                a.x = fmaf(p, u[r].x, a.x); a.y = fmaf(p, u[r].y, a.y); a.z = fmaf(p, u[r].z, a.z); a.w = fmaf(p, u[r].w, a.w);
            }
            ((float4*)(master + (size_t)s * n))[i] = a;
            char* slot = copy0 + (size_t)s * slot_bytes;
            const size_t e = i * 4;
            if (e < n_big) {
                if (sizeof(T) == 4) ((float4*)slot)[i] = a;
                else {
                    __nv_bfloat162 lo = __floats2bfloat162_rn(a.x, a.y), hi = __floats2bfloat162_rn(a.z, a.w);
                    uint2 pk; pk.x = *(unsigned*)&lo; pk.y = *(unsigned*)&hi;
                    ((uint2*)slot)[i] = pk;
                }
            } else {
                *(float4*)((float*)(slot + n_big * sizeof(T)) + (e - n_big)) = a;
            }
        }
    }
    if (stamp && blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) *stamp = device_time_ns();
}
int mix_max_replicas() { return MIX_MAX_R; }
void mix_update(int dt, float* master, const float* grad, void* copy0, size_t n_big, size_t n_small, size_t slot_bytes, int R, const float* P, float lr,
                long long* stamp, cudaStream_t s) {
    const size_t n4 = (n_big + n_small) / 4;
    if (n4 == 0) return;
    unsigned blocks = cdiv(n4, 256);
    if (blocks > 148 * 4) blocks = 148 * 4;
    Scope sc(KC_SGD, 0.0, (double)R * (n_big + n_small) * ((grad ? 12.0 : 8.0) + (dt ? 2.0 : 4.0)), s);
    if (dt) klaunch(mix_k<bf16>, blocks, 256, 0, s, master, grad, (char*)copy0, n_big, n_small, slot_bytes, R, P, lr, stamp);
    else klaunch(mix_k<float>, blocks, 256, 0, s, master, grad, (char*)copy0, n_big, n_small, slot_bytes, R, P, lr, stamp);
}

// ------------------------------------------------------------------------------------------
// schedule tags
// ------------------------------------------------------------------------------------------
__global__ void tags_k(TagOps o) {
    if (threadIdx.x != 0) return;
    if (o.time_start) *o.time_start = device_time_ns();
    // tags of what this step produces first: the last module reads the stash slot it fills itself
    if (o.wr_in) { o.wr_in[0] = o.version_now; o.wr_in[1] = -1; }      // module 1: the batch sampled now
    if (o.wr_out) { o.wr_out[0] = o.fwd_batch; o.wr_out[1] = -1; }
    if (o.wr_stash) { o.wr_stash[0] = o.fwd_batch; o.wr_stash[1] = o.version_now; }
    if (o.wr_grad) { o.wr_grad[0] = o.bwd_batch; o.wr_grad[1] = -1; }
    int64_t fb = o.rd_act ? o.rd_act[0] : -1;
    int64_t bb = -1, bv = -1;
    if (o.rd_stash) {
        bb = o.rd_stash[0];
        if (o.rd_grad && o.rd_grad[0] != bb) bb = -2;
        bv = o.rd_wbwd ? o.rd_wbwd[1] : -1;
        if (o.rd_stash[1] != bv) bv = -2;                 // the stash records the version the forward used
    }
    o.trace[0] = fb; o.trace[1] = bb; o.trace[2] = bv; o.trace[3] = o.rd_wfwd ? o.rd_wfwd[1] : -1;
    // the next weight version replaces a slot only at the end of the step, after the reads above
    if (o.wr_wnext) { o.wr_wnext[0] = -1; o.wr_wnext[1] = o.version_now + 1; }
}
void tags_step(const TagOps& ops, cudaStream_t s) { Scope sc(KC_TAGS, 0.0, 128.0, s); klaunch(tags_k, 1, 32, 0, s, ops); }

// Zeros, 16 bytes per thread and access (n16 vectors).
__global__ void __launch_bounds__(256) zero_k(uint4* p, size_t n16) {
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n16; i += (size_t)gridDim.x * blockDim.x) p[i] = make_uint4(0u, 0u, 0u, 0u);
}
void zero_fill(void* p, size_t bytes, cudaStream_t s) { klaunch(zero_k, ew_grid(bytes / 16), 256, 0, s, (uint4*)p, bytes / 16); }

// The step's batch and labels into their FIFO slots, one launch.  vec: both input addresses are 16-byte aligned (labels go word by word).
__global__ void __launch_bounds__(256) ingest_k(const char* __restrict__ x, char* __restrict__ xd, size_t x_bytes, const int32_t* __restrict__ y, int32_t* __restrict__ yd, int m, bool vec) {
    const size_t t0 = (size_t)blockIdx.x * blockDim.x + threadIdx.x, stride = (size_t)gridDim.x * blockDim.x;
    const size_t n16 = vec ? x_bytes / 16 : 0;
    size_t i = t0;
    for (; i + 3 * stride < n16; i += 4 * stride) {              // four loads in flight
        uint4 v[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) v[u] = ((const uint4*)x)[i + u * stride];
#pragma unroll
        for (int u = 0; u < 4; ++u) ((uint4*)xd)[i + u * stride] = v[u];
    }
    for (; i < n16; i += stride) ((uint4*)xd)[i] = ((const uint4*)x)[i];
    for (size_t b = n16 * 16 + 2 * t0; b < x_bytes; b += 2 * stride) *(uint16_t*)(xd + b) = *(const uint16_t*)(x + b);     // both storage types are whole 2-byte words
    for (size_t l = t0; l < (size_t)m; l += stride) yd[l] = y[l];
}
void ingest(const void* x, void* xd, size_t x_bytes, const int32_t* y, int32_t* yd, int m, cudaStream_t s) {
    const bool vec = (((uintptr_t)x | (uintptr_t)xd) & 15) == 0;
    Scope sc(KC_INGEST, 0.0, 2.0 * (double)x_bytes + 8.0 * m, s);
    klaunch(ingest_k, ew_grid(vec ? x_bytes / 64 : x_bytes / 2), 256, 0, s, (const char*)x, (char*)xd, x_bytes, y, yd, m, vec);
}

bool profile_active() { return prof::g_on; }

}  // namespace fdg
