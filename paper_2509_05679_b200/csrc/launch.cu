// See launch.h.
#include "launch.h"

namespace fdg {

static thread_local StepGraph* t_graph = nullptr;
StepGraph* StepGraph::current() { return t_graph; }

cudaError_t allow_smem(OncePerDevice& once, const void* kernel, int bytes) {
    int dev = -1;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess || once.done(dev)) return e;
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e == cudaSuccess) once.set(dev);
    return e;
}

static cudaError_t launch_now(const void* func, dim3 grid, dim3 block, size_t smem, cudaStream_t s, void** args, int cluster) {
    if (!cluster) return cudaLaunchKernel(func, grid, block, args, smem, s);
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = cluster; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
    cfg.gridDim = grid; cfg.blockDim = block; cfg.dynamicSmemBytes = smem; cfg.stream = s; cfg.attrs = at; cfg.numAttrs = 1;
    return cudaLaunchKernelExC(&cfg, func, args);
}

cudaError_t launch_raw(const void* func, dim3 grid, dim3 block, size_t smem, cudaStream_t s, void** args, const size_t* sizes, int nargs, int cluster) {
    if (t_graph) return t_graph->on_launch(func, grid, block, smem, s, args, sizes, nargs, cluster);
    return launch_now(func, grid, block, smem, s, args, cluster);
}
cudaError_t step_record(cudaEvent_t e, cudaStream_t s) {
    return t_graph && t_graph->mode() == StepGraph::UPDATE ? cudaSuccess : cudaEventRecord(e, s);
}
cudaError_t step_wait(cudaStream_t s, cudaEvent_t e) {
    return t_graph && t_graph->mode() == StepGraph::UPDATE ? cudaSuccess : cudaStreamWaitEvent(s, e, 0);
}

bool StepGraph::begin_capture(cudaStream_t origin) {
    clear();
    if (cudaStreamBeginCapture(origin, cudaStreamCaptureModeThreadLocal) != cudaSuccess) { cudaGetLastError(); return false; }
    mode_ = CAPTURE; bad_ = false; t_graph = this;
    return true;
}
bool StepGraph::end_capture(cudaStream_t origin) {
    t_graph = nullptr; mode_ = OFF;
    const bool ok = cudaStreamEndCapture(origin, &graph_) == cudaSuccess && graph_ && !bad_ && cudaGraphInstantiate(&exec_, graph_, 0) == cudaSuccess;
    if (!ok) { cudaGetLastError(); clear(); }
    return ok;
}
void StepGraph::begin_update() { mode_ = UPDATE; next_ = 0; bad_ = false; t_graph = this; }
bool StepGraph::end_update() {
    t_graph = nullptr; mode_ = OFF;
    if (!bad_ && next_ == nodes_.size()) return true;
    clear();
    return false;
}
void StepGraph::clear() {
    if (exec_) cudaGraphExecDestroy(exec_);
    if (graph_) cudaGraphDestroy(graph_);
    exec_ = nullptr; graph_ = nullptr; nodes_.clear(); next_ = 0;
}

cudaError_t StepGraph::on_launch(const void* func, dim3 grid, dim3 block, size_t smem, cudaStream_t s, void** args, const size_t* sizes, int nargs, int cluster) {
    size_t total = 0;
    for (int i = 0; i < nargs; ++i) total += sizes[i];
    if (mode_ == CAPTURE) {
        cudaError_t e = launch_now(func, grid, block, smem, s, args, cluster);
        if (e != cudaSuccess) { bad_ = true; return e; }
        // the node just added is what the stream's next work depends on
        cudaStreamCaptureStatus st;
        const cudaGraphNode_t* deps = nullptr;
        size_t ndeps = 0;
        e = cudaStreamGetCaptureInfo_v2(s, &st, nullptr, nullptr, &deps, &ndeps);
        if (e != cudaSuccess || st != cudaStreamCaptureStatusActive || ndeps != 1) { bad_ = true; return e; }
        Node n{deps[0], func, grid, block, smem, std::vector<char>(total)};
        size_t at = 0;
        for (int i = 0; i < nargs; ++i) { std::memcpy(n.params.data() + at, args[i], sizes[i]); at += sizes[i]; }
        nodes_.push_back(std::move(n));
        return cudaSuccess;
    }
    if (bad_ || next_ >= nodes_.size()) { bad_ = true; return cudaSuccess; }
    Node& n = nodes_[next_++];
    if (n.func != func || n.grid.x != grid.x || n.grid.y != grid.y || n.grid.z != grid.z || n.block.x != block.x || n.block.y != block.y || n.smem != smem ||
        n.params.size() != total) { bad_ = true; return cudaSuccess; }
    bool same = true;
    size_t at = 0;
    for (int i = 0; i < nargs; ++i) {
        if (same && std::memcmp(n.params.data() + at, args[i], sizes[i]) != 0) same = false;
        if (!same) std::memcpy(n.params.data() + at, args[i], sizes[i]);
        at += sizes[i];
    }
    if (same) return cudaSuccess;
    cudaKernelNodeParams kp = {};
    kp.func = const_cast<void*>(func); kp.gridDim = grid; kp.blockDim = block; kp.sharedMemBytes = (unsigned)smem; kp.kernelParams = args;
    const cudaError_t e = cudaGraphExecKernelNodeSetParams(exec_, n.node, &kp);
    if (e != cudaSuccess) { cudaGetLastError(); bad_ = true; }
    return cudaSuccess;
}

}  // namespace fdg
