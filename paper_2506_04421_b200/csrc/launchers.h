// Internal launcher prototypes shared between the C-ABI layer and the kernel files.
#pragma once
#include <cuda_runtime.h>
#include <atomic>
#include "hmar_common.h"

namespace hmar {

void count_launch(int n);

// Per-kernel timing (diagnostics): when profiling is on, a kernel launch wrapped in KernelTimer is
// bracketed by two events on its stream; hmar_profile_end() sums them per kernel name.
bool profile_enabled();
struct KernelTimer {
    KernelTimer(const char* name, cudaStream_t stream);
    ~KernelTimer();
    const char* name_;
    cudaStream_t stream_;
    cudaEvent_t begin_;
    bool on_;
};

// Opts a kernel in to `bytes` of dynamic shared memory on the current device: once per kernel and device, not on every
// call (0.4 us of host time each, three of them in a backward call).
struct SmemOptIn {
    std::atomic<unsigned long long> done{0};                // a bit per device
    cudaError_t operator()(const void* kernel, size_t bytes) {
        int dev = 0;
        cudaError_t e = cudaGetDevice(&dev);
        if (e != cudaSuccess) return e;
        const unsigned long long bit = dev < 64 ? 1ull << dev : 0;
        if (done.load(std::memory_order_acquire) & bit) return cudaSuccess;
        e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
        if (e == cudaSuccess) done.fetch_or(bit, std::memory_order_release);
        return e;
    }
};

// What an entry point returns for the outcome of its launches.  A refused launch or copy leaves its error in the runtime,
// where the check behind the next launch, which nothing refused, would find it: it is taken out here.
inline int launch_status(cudaError_t e) {
    if (e == cudaSuccess) return HMAR_OK;
    cudaGetLastError();
    return HMAR_ERR_CUDA;
}

// Launches a kernel whose blocks may start as soon as the last block of the previous kernel of its stream has ended: its
// parameters and its own set-up no longer wait for that kernel's stores to be flushed.  It calls grid_wait() before it
// touches anything that another kernel writes or reads, and before it takes tensor memory.  1.5 to 3 us per launch: forward
// + backward of L = 1300, 39 heads 107 -> 99.5 us, L = 680 128 heads 87 -> 80, L = 2240 96 heads 312 -> 305; forward of
// L = 680, 32 heads 14.3 -> 12.3.  (Letting the next kernel start earlier, while blocks of this one still run, is slower:
// backward of L = 2240, 384 heads 829 -> 853 us, without the overlap 835.)
template <typename... P, typename... A>
cudaError_t launch_overlapped(void (*kernel)(P...), unsigned grid, unsigned threads, size_t smem, cudaStream_t stream, A&&... args) {
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t config{};
    config.gridDim = dim3(grid);
    config.blockDim = dim3(threads);
    config.dynamicSmemBytes = smem;
    config.stream = stream;
    config.attrs = &attr;
    config.numAttrs = 1;
    return cudaLaunchKernelEx(&config, kernel, static_cast<A&&>(args)...);
}

template <typename T>
cudaError_t simt_fwd(const T* q, const T* k, const T* v, T* out, float* lse, int BH, int D,
                     const ScaleTable& st, float scale, cudaStream_t stream);
template <typename T>
cudaError_t simt_scale_step(const T* q, const T* k_prev, const T* v_prev, const T* k_cur, const T* v_cur,
                            T* out, float* lse, int BH, int D, int n_prev, int n_cur, float scale,
                            cudaStream_t stream);
template <typename T>
cudaError_t simt_bwd(const T* q, const T* k, const T* v, const T* out, const float* lse, const T* dout,
                     T* dq, T* dk, T* dv, float* delta, int BH, int D, const ScaleTable& st, float scale,
                     cudaStream_t stream);

cudaError_t launch_recon_accumulate(float* xhat, const float* codebook, const int* tokens_old, const int* tokens_new,
                                    const unsigned char* mask, int* tokens_out, int B, int C, int V, int side, int out_side,
                                    cudaStream_t stream);
cudaError_t launch_recon_downsample(const float* xhat, float* out, int B, int C, int in_side, int out_side,
                                    cudaStream_t stream);

}  // namespace hmar
