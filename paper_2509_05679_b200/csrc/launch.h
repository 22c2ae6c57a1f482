// How the step executor puts kernels on streams: every launch goes through klaunch(), every event between the streams of one
// module's step through step_record() / step_wait(), so that the same code that enqueues a step can also record it into a CUDA graph
// once and afterwards only refresh the kernels' parameters (the FIFO slots rotate, everything else stays).
//
// Why: a launch costs the host 3.6 us on a B200 host, refreshing a graph node 0.2 us and launching a graph about 3 us, and inside a graph
// dependent kernels follow each other in 0.3-0.6 us.  A step of a small network is 35 to 170 launches.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>
#include <cstring>
#include <tuple>
#include <utility>
#include <vector>

namespace fdg {

// The graph of one module's step.
class StepGraph {
public:
    enum Mode { OFF, CAPTURE, UPDATE };
    ~StepGraph() { clear(); }
    bool ready() const { return exec_ != nullptr; }
    // capture: everything this thread enqueues until end_capture() becomes the graph (origin: a stream of the library's own)
    bool begin_capture(cudaStream_t origin);
    bool end_capture(cudaStream_t origin);
    // update: the same calls again, with new parameters; false if they were not the same calls (the graph is dropped then)
    void begin_update();
    bool end_update();
    cudaError_t launch(cudaStream_t s) { return cudaGraphLaunch(exec_, s); }
    void clear();
    cudaError_t on_launch(const void* func, dim3 grid, dim3 block, size_t smem, cudaStream_t s, void** args, const size_t* sizes, int nargs, int cluster);
    Mode mode() const { return mode_; }
    static StepGraph* current();                 // of this thread, or nullptr
private:
    struct Node { cudaGraphNode_t node; const void* func; dim3 grid, block; size_t smem; std::vector<char> params; };
    Mode mode_ = OFF;
    cudaGraph_t graph_ = nullptr;
    cudaGraphExec_t exec_ = nullptr;
    std::vector<Node> nodes_;
    size_t next_ = 0;
    bool bad_ = false;
};

// Something done once per device and process (devices 0 to 63; done again every time on others).  Two threads may both do it.
class OncePerDevice {
public:
    bool done(int device) const { return device >= 0 && device < 64 && (mask_.load(std::memory_order_acquire) >> device & 1); }
    void set(int device) { if (device >= 0 && device < 64) mask_.fetch_or(1ull << device, std::memory_order_release); }
private:
    std::atomic<uint64_t> mask_{0};
};
// Lets `kernel` have `bytes` of dynamic shared memory on the current device (a kernel's attributes are those of one device); `once` is the kernel's.
cudaError_t allow_smem(OncePerDevice& once, const void* kernel, int bytes);

// cluster: CTAs per cluster along x (0: none)
cudaError_t launch_raw(const void* func, dim3 grid, dim3 block, size_t smem, cudaStream_t s, void** args, const size_t* sizes, int nargs, int cluster);
// Whether a launch went through.  A refused one leaves no error behind: its caller has another way, and the next launch is not to be blamed for it.
inline bool launched(cudaError_t e) { if (e != cudaSuccess) cudaGetLastError(); return e == cudaSuccess; }
// the order between streams inside one module's step: nothing to do while a graph is only refreshed
cudaError_t step_record(cudaEvent_t e, cudaStream_t s);
cudaError_t step_wait(cudaStream_t s, cudaEvent_t e);

namespace detail {
template <typename Tuple, size_t... I>
cudaError_t launch_tuple(const void* f, dim3 grid, dim3 block, size_t smem, cudaStream_t s, int cluster, Tuple& t, std::index_sequence<I...>) {
    void* args[sizeof...(I) + 1] = {(void*)&std::get<I>(t)..., nullptr};
    const size_t sizes[sizeof...(I) + 1] = {sizeof(std::tuple_element_t<I, Tuple>)..., 0};
    return launch_raw(f, grid, block, smem, s, args, sizes, (int)sizeof...(I), cluster);
}
}  // namespace detail

template <typename... P, typename... A>
cudaError_t klaunch_cluster(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, int cluster, A&&... a) {
    static_assert(sizeof...(P) == sizeof...(A), "kernel arguments");
    std::tuple<std::remove_cv_t<std::remove_reference_t<P>>...> t(std::forward<A>(a)...);
    return detail::launch_tuple((const void*)kernel, grid, block, smem, s, cluster, t, std::index_sequence_for<P...>());
}
template <typename... P, typename... A>
cudaError_t klaunch(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, A&&... a) {
    return klaunch_cluster(kernel, grid, block, smem, s, 0, std::forward<A>(a)...);
}

}  // namespace fdg
