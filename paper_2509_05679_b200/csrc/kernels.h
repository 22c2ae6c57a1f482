// Internal launch interface between the step executor (fdg_api.cu) and the kernels.
// All pointers are device pointers; `dt` is 0 for fp32 storage, 1 for bf16 storage.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace fdg {

struct ConvGeom {            // x: [N,H,W,C]  ->  y: [N,Ho,Wo,Co], R x R window
    int N, H, W, C, Ho, Wo, Co, R, stride, pad;
};

enum { EPI_RELU = 1, EPI_ACCUM = 2, EPI_OUT_F32 = 4 };

// y = conv(x, W) (+ bias) (relu)            (Eq. forward_step for linear / conv layers, CUDA cores)

bool   conv_supported(const ConvGeom& g);
size_t wgrad_workspace_elems(const ConvGeom& g);      // fp32 elements fconv_wgrad needs
struct Packed;
void   conv_forward(int dt, const void* x, const void* w, const float* bias, void* y, const ConvGeom& g, int epi, const Packed& pk, cudaStream_t st);
// Linear layers (linear.cu).  linear_backward: dx (+)= dy' W (dx_or_null == nullptr: not needed), dW (+)= dy'^T x, db (+)= column sums of
// dy' in one launch; dy' = dy * [y > 0] if y_or_null is given (the layer ends in a ReLU), else dy.  The sums run over the worker x
// batch axis, which is the worker average of Eq. dl_update (b) for P = 11^T/N.  accum_p: dW and db are added to (a second group of workers).  dw_or_null ==
// nullptr: dx alone; dx_or_null == nullptr: w is not read.  Many samples: dW and db go through partial matrices in workspace
// (linear_workspace_elems floats, the layer's own; nullptr: one part) that a second launch on st_reduce, behind `ready`, adds up.
bool   linear_supported(const ConvGeom& g);
size_t linear_workspace_elems(const ConvGeom& g, int groups);
// groups, w_group, b_group, g_group: as for the convolutions below (g.N counts the samples of all groups).
void   linear_forward(int dt, const void* x, const void* w, const float* bias, void* y, const ConvGeom& g, int epi, int groups, size_t w_group, size_t b_group,
                      cudaStream_t st);
void   linear_backward(int dt, const void* x, const void* w, const void* y_or_null, const void* dy, void* dx_or_null, bool accum_dx, float* dw_or_null, float* db_or_null,
                       const ConvGeom& g, int groups, size_t w_group, size_t g_group, bool accum_p, float* workspace, cudaStream_t st, cudaStream_t st_reduce,
                       cudaEvent_t ready);
// Convolutions (3x3 and 1x1, stride 1 and 2) in the packed-FMA kernels of fconv.cu: forward, dx (+)= conv_transpose(dy, W), dW (+)= the sum
// over all N*Ho*Wo rows of dy^T (x) patches(x) (fp32).  `groups`: consecutive equal groups of images, each with its own weights
// (w_group elements apart; biases b_group apart; weight gradients w_group apart).  false: shape not covered, nothing launched.
bool   fconv_supported(const ConvGeom& g);
// Layers of channel counts that are multiples of 16 run on warp-level tensor-core instructions (mconv.cu) if their weights are there in the order
// that these read: mconv_pack lays out a module's layers (PackArgs, `blocks` 16 x 16 blocks in all) for one direction, per group `group` bytes apart.
// mconv_takes: whether a forward (back == false) or input-gradient launch of this many images and groups goes that way, given them.
// mconv_pack_bytes: of one such layer and direction, a multiple of 16.
struct Packed { const void* data; size_t group; };       // data == nullptr: the packed-FMA kernels
struct PackLayer { size_t w_off, out_off; int C, Co, taps, block0; };        // elements into the matrices, 16-byte words into the result; first block
struct PackArgs { enum { MAX = 48 }; PackLayer layer[MAX]; int n, back; };
bool   mconv_takes(int dt, const ConvGeom& g, int groups, bool back);
size_t mconv_pack_bytes(int dt, const ConvGeom& g);
bool   mconv_pack(int dt, const void* wbig, size_t w_group, void* out, size_t out_group, const PackArgs& a, int blocks, int groups, cudaStream_t st);      // false: refused
bool   fconv_forward(int dt, const void* x, const void* w, const float* bias, void* y, const ConvGeom& g, int epi, int groups, size_t w_group, size_t b_group,
                     float* stat_or_null, const Packed& pk, cudaStream_t st);
// Batch-norm statistics taken along by fconv_forward (groups = workers): per worker and pixel tile the channels' (mean, sum of
// squared deviations), then the tiles' pixel counts: [groups][tiles][Co][2], [groups][tiles] floats.  0: shape not covered.
int    fconv_stat_tiles(const ConvGeom& g, int groups);
bool   fconv_dgrad(int dt, const void* dy, const void* w, void* dx, const ConvGeom& g, int epi, int groups, size_t w_group, const Packed& pk, cudaStream_t st);
size_t fconv_wgrad_workspace_elems(const ConvGeom& g, int groups);
// tensor: by mconv.cu where it covers the shape.
bool   fconv_wgrad(int dt, const void* x, const void* dy, float* dw, float* workspace, const ConvGeom& g, int groups, size_t w_group, bool accum, bool tensor, cudaStream_t st);
// db[c] = sum over rows of dy[row][c]; scratch: fp32 [64 * C]
void bias_grad(int dt, const void* dy, float* db, float* scratch, long rows, int C, bool accum, cudaStream_t st);

// Backward pass through "+ bias, ReLU" of a layer in one pass over dy: dy *= (y > 0) in place (y_or_null == nullptr: no
// ReLU) and db = column sums of the masked dy (db_or_null == nullptr: no bias).  scratch: relu_bias_backward_scratch_elems(C)
// floats.  Only for widths relu_bias_backward_supported() accepts.
bool   relu_bias_backward_supported(int dt, int C);
size_t relu_bias_backward_scratch_elems(int C);
void   relu_bias_backward(int dt, const void* y_or_null, void* dy, float* db_or_null, float* scratch, long rows, int C, bool accum, cudaStream_t st);

// First-layer convolution (3x3, stride 1, <= 4 input channels, bf16): dedicated kernels (stem.cu).
bool   stem_supported(int dt, const ConvGeom& g);
size_t stem_wgrad_workspace_elems(const ConvGeom& g);
void   stem_forward(const void* x, const void* w, const float* bias, void* y, const ConvGeom& g, bool relu, cudaStream_t st);
void   stem_wgrad(const void* x, const void* dy, float* dw, float* workspace, const ConvGeom& g, bool accum, cudaStream_t st);

void relu_forward(int dt, const void* x, void* y, size_t n, cudaStream_t st);
// dx (+)= dy * (y > 0)
void relu_backward(int dt, const void* y, const void* dy, void* dx, size_t n, bool accum, cudaStream_t st);
// y = a + b ; backward is two copies / accumulations
void add_forward(int dt, const void* a, const void* b, void* y, size_t n, cudaStream_t st);
void copy_or_accumulate(int dt, const void* src, void* dst, size_t n, bool accum, cudaStream_t st);
void maxpool_forward(int dt, const void* x, void* y, int N, int H, int W, int C, cudaStream_t st);
// Where the input of a backward pass's layer is a ReLU layer's output, the pass can apply that ReLU's mask to the gradient it produces and leave
// the masked gradient's column sums (the layer's bias gradient) as records [rec][C][2], the sums in element 0: col_or_null (C / V a power
// of two <= 256, V = 8 bf16 / 4 fp32 values), *_col_records records, added by colsum_records.
void colsum_records(const float* part, float* out, int recs, int C, bool accum, cudaStream_t st);
int  pool_col_records(int dt, int N, int H, int W, int C);
int  gap_col_records(int dt, int N, int HW, int C);
void maxpool_backward(int dt, const void* x, const void* dy, void* dx, int N, int H, int W, int C, bool accum, float* col_or_null, cudaStream_t st);
void gap_forward(int dt, const void* x, void* y, int N, int HW, int C, cudaStream_t st);
void gap_backward(int dt, const void* dy, void* dx, int N, int HW, int C, bool accum, const void* mask_x_or_null, float* col_or_null, cudaStream_t st);

// Batch-norm with per-worker statistics.  x: [n_workers * rows_per_worker, C].
// err: device word that a kernel sets non-zero if a bounded wait on an asynchronous copy gave up (nullptr: the
// kernels that stream through shared memory are not used).
// stats: fp32 [n_workers][C][2] = (mean, invstd).  scratch: fp32 [128 * n_workers * C * 2].
// conv_part / conv_chunks: if non-null, the producing convolution already left per-tile (sum, sum of squares)
// partials [n_workers * conv_chunks][C][2] (worker-major); the statistics pass over x is skipped.
// sms: the SMs the streamed kernels size their grids for (0 or >= the device's count: all); the partial sums depend on it
// through the number of row chunks (fp32 summation order).
void bn_forward(int dt, const void* x, const float* gamma, const float* beta, const void* residual_or_null,
                void* y, float* stats, float* scratch, int n_workers, long rows_per_worker, int C, bool relu,
                const float* conv_part, int conv_chunks, int sms, int* err, cudaStream_t st);
bool bn_accepts_conv_partials(int dt, int C);
// conv_part == nullptr and conv_chunks < 0: `stats` already holds (mean, invstd) of every worker (bn_merge_tiles).

// fp32 storage (bnorm.cu), C / 4 a power of two: forward from the records fconv_forward left (tile_part, see fconv_stat_tiles), backward in
// two launches.  p_group / g_group: floats between the workers' parameters / parameter gradients (0: shared by all workers, gradients
// summed over them).  mask_from_x: the forward output was bnf_forward's without a residual, so its sign can be recomputed from x.
// scratch: as in bn_backward.  bn_merge_tiles: (mean, invstd) per worker and channel from such records, any storage type.
// bf16 storage, tensors of a few MB (bnorm.cu): one launch per direction, statistics included.  red: [n_workers][C][2] floats, from which
// bnc_params adds up dgamma, dbeta.  nw: the workers of this launch (pointers to the first one's), nw_all: all of them; modules: of the network,
// which share the device.
bool bnc_supported(int dt, int nw, long rpw, int C);
void bnc_forward(const void* x, const float* gamma, const float* beta, const void* res, void* y, float* stats, int nw, int nw_all, int modules, long rpw, int C, bool relu,
                 cudaStream_t st);
void bnc_backward(const void* x, const void* out, const void* dout, const float* gamma, const float* beta, const float* stats, void* dx, bool accum_dx, void* dres,
                  bool accum_dres, float* red, int nw, int nw_all, int modules, long rpw, int C, bool relu, bool has_res, cudaStream_t st);
void bnc_params(const float* red, float* dgamma, float* dbeta, int nw, int C, cudaStream_t st);
bool bnf_supported(int dt, int C);
void bn_merge_tiles(const float* tile_part, float* stats, int tiles, int nw, long rpw, int C, cudaStream_t st);
void bnf_forward(const float* x, const float* gamma, const float* beta, size_t p_group, const float* res, float* y, float* stats, const float* tile_part,
                 int tiles, int nw, long rpw, int C, bool relu, cudaStream_t st);
void bnf_backward(const float* x, const float* out, const float* dout, const float* gamma, const float* beta, size_t p_group, const float* stats, float* dx,
                  bool accum_dx, float* dres, bool accum_dres, float* dgamma, float* dbeta, size_t g_group, float* scratch, int nw, long rpw, int C, bool relu,
                  bool mask_from_x, bool accum_params, cudaStream_t st);
// dy_eff = dout * (out > 0 if relu).  dx (+)= BN backward of dy_eff (dx == nullptr: not needed, in every backward of this file); dres (+)= dy_eff;
// dgamma, dbeta (fp32) = sums over all workers.  red: fp32 [n_workers][C][2] scratch for (sum dy, sum dy xhat).
void bn_backward(int dt, const void* x, const void* out, const void* dout, const float* gamma, const float* beta,
                 const float* stats, void* dx, bool accum_dx, void* dres_or_null, bool accum_dres, float* dgamma, float* dbeta,
                 float* red, float* scratch, int n_workers, long rows_per_worker, int C, bool relu, bool has_res, bool accum_params,
                 int sms, int* err, cudaStream_t st);

// Where a step's loss reaches the host: pinned memory the kernel that computes it writes to (seq last).
struct LossRecord { float loss; int err; long long seq; };
void publish_loss_value(LossRecord* rec, float loss, const int* err, long long seq, cudaStream_t st);

// Softmax cross-entropy over fp32 logits [M, classes]: dlogits (storage dtype) = (softmax - onehot) * scale,
// rec: the mean loss, the error word `err` and the number `seq`.  Deterministic single-block reduction.
void softmax_ce(int dt, const float* logits, const int32_t* labels, void* dlogits, LossRecord* rec, const int* err, long long seq, int M, int classes,
                float scale, cudaStream_t st);

// Classifier head (the last linear layer, c_in = K -> C classes, C <= 16) fused with the loss.  head_forward_loss: logits
// (fp32), dlogits = (softmax - onehot) * scale (storage dtype) and partial sums of the loss in one launch.  head_backward: dx (+)= dlogits W
// (dx_or_null == nullptr: not needed) and the partial sums of dW, db, which head_reduce adds, with those of the loss; mask_dx, col: see above.
// scratch: head_scratch_elems floats: the weight-gradient partials, then the loss partials.
bool   head_supported(int dt, int K, int C);
size_t head_scratch_elems(int M, int K, int C);
void   head_forward_loss(int dt, const void* x, const void* W, const float* bias, const int32_t* labels, float* logits, void* dlogits, float* loss_part, int M, int K, int C,
                         float scale, cudaStream_t st);
int    head_col_records(int M);
void   head_backward(int dt, const void* x, const void* W, const void* dlogits, void* dx_or_null, bool accum_dx, bool mask_dx, float* col_or_null, float* scratch, int M,
                     int K, int C, cudaStream_t st);
// what head_backward left in scratch, and the mean loss
void   head_reduce(float* dW, float* db_or_null, const float* scratch, const float* loss_part, LossRecord* rec, const int* err, long long seq, int M, int K, int C,
                   cudaStream_t st);

// master -= lr * grad (skipped when grad == nullptr: w(t+1) = w(t)); copy_next = storage-dtype copy of
// the new master (the next weight version).  n must be a multiple of 4; pointers 16-byte aligned.
// stamp: device word that receives the device's time in ns at the end, or nullptr.
void sgd_update(int dt, float* master, const float* grad, void* copy_next, size_t n, float lr, long long* stamp, cudaStream_t st);

// General mixing matrix: R replicas [R][n_big + n_small] of master and grad; u_r = w_r - lr g_r (grad == nullptr: u_r = w_r),
// w_s = sum_r P[s][r] u_r in place, and the storage-dtype copies of the next version (replica r at copy0 + r * slot_bytes:
// n_big values of the storage dtype, then n_small floats).  R <= mix_max_replicas().
int  mix_max_replicas();
void mix_update(int dt, float* master, const float* grad, void* copy0, size_t n_big, size_t n_small, size_t slot_bytes, int R, const float* P, float lr,
                long long* stamp, cudaStream_t st);

// Schedule tags (see fdg_trace).  tags are int64 pairs {batch id, weight version}.
struct TagOps {
    const int64_t* rd_act;  const int64_t* rd_stash; const int64_t* rd_grad; const int64_t* rd_wbwd; const int64_t* rd_wfwd;
    int64_t* wr_in; int64_t* wr_out; int64_t* wr_stash; int64_t* wr_grad; int64_t* wr_wnext;
    int64_t fwd_batch, bwd_batch, version_now;   // what this step produces (-1: nothing)
    long long* time_start;                       // device time in ns, or nullptr
    int64_t* trace;                              // [4]: fwd batch, bwd batch, bwd weight version, fwd weight version
};
void tags_step(const TagOps& ops, cudaStream_t st);

void stamp_time(long long* stamp, cudaStream_t st);              // the device's time in ns
void zero_fill(void* p, size_t bytes, cudaStream_t st);          // p and bytes multiples of 16
// x_bytes of a batch and its m labels into their FIFO slots
void ingest(const void* x, void* x_slot, size_t x_bytes, const int32_t* y, int32_t* y_slot, int m, cudaStream_t st);
uint64_t launches();     // kernels launched so far through this interface

// Kernel classes for launch counting and optional device timing.
enum KernelClass {
    KC_FMA_FWD, KC_FMA_DGRAD, KC_FMA_WGRAD, KC_SPLITK, KC_BIAS_GRAD, KC_RELU_FWD, KC_RELU_BWD, KC_ADD_FWD, KC_COPY_ACC,
    KC_POOL_FWD, KC_POOL_BWD, KC_GAP_FWD, KC_GAP_BWD, KC_BN_FWD_STATS, KC_BN_FWD_APPLY, KC_BN_BWD_REDUCE, KC_BN_BWD_APPLY,
    KC_SOFTMAX_CE, KC_SGD, KC_TAGS, KC_FILL, KC_TC_FWD, KC_TC_DGRAD, KC_TC_WGRAD, KC_TC_AUX, KC_INGEST,
    KC_MMA_FWD, KC_MMA_DGRAD, KC_MMA_WGRAD,        // mconv.cu
    KC_COUNT
};
struct KernelStat { uint64_t launches; double ms, flops, bytes; };
// Opened around every launch: counts it and, while profiling is enabled, records an event before and
// after it on the launching stream.  flops / bytes are the launch's ALGORITHMIC work.
struct Scope {
    int cls; cudaStream_t st; cudaEvent_t a; const char* detail;
    Scope(int cls, double flops, double bytes, cudaStream_t s);
    ~Scope();
};
void profile_detail(const char* detail);                    // tag (e.g. a layer shape) for the Scopes this thread opens next; nullptr clears
int  profile_read_detail(KernelStat* out, char (*names)[48], int capacity);   // call after profile_read
bool profile_active();
void profile_enable(bool on);                               // on: clears the statistics
int  profile_read(KernelStat* out, const char** names);     // synchronises the device; returns KC_COUNT

}  // namespace fdg
