// Shared host-side plumbing of the library: status codes, per-device scratch,
// CUDA error capture, launch counting.  No kernel arithmetic lives here.
#pragma once

#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include "../../include/dualdiff.h"

namespace dd {

// Per-device scratch owned by the library.
struct DeviceCtx {
    void *verify_ws = nullptr;      // dd_verify chunk partials and row results
    size_t verify_ws_bytes = 0;
    void *verify_cnt = nullptr;     // dd_verify completion counters: all zero between launches
    size_t verify_cnt_bytes = 0;
    void *head_ws = nullptr;        // dd_lm_head_verify: the flagged rows' hidden states, where there is room for them
    size_t head_ws_bytes = 0;
    void *staging = nullptr;        // device copies of host buffers (the *_host calls)
    size_t staging_bytes = 0;
    unsigned int *attn_status = nullptr;  // one word: first expired wait of the attention kernel
    // Host copy of the two health words (pinned, mapped): [0] attention, [1] verify.  A kernel that
    // records an expired wait writes the code here as well, so the next call sees it without a
    // device synchronisation.
    volatile unsigned int *mirror = nullptr;
    unsigned int *mirror_dev = nullptr;   // the same two words as the kernels address them
};

// Returns the context of the current device (creating it on first use), or
// nullptr after recording a CUDA error.
DeviceCtx *current_ctx(int *device_out = nullptr);

// Allocates the host copy of the health words on first use (pinned host memory, no device memory).
int ensure_mirror(DeviceCtx *ctx);

// DD_ERR_TIMEOUT (with error text) if the host copy shows that kernel `which` (0 attention,
// 1 verify) has recorded an expired wait on this device; DD_OK otherwise.
int check_mirror(const DeviceCtx *ctx, int which);

// Grows (never shrinks) a scratch buffer; new memory is zero-filled.
int ensure_bytes(void **ptr, size_t *have, size_t need);
// The same for scratch that a call can do without, a quarter of the free memory at most and never while `stream` is
// being captured: DD_OK if it is there; if not, nothing has changed.
int try_bytes(void **ptr, size_t *have, size_t need, cudaStream_t stream);

// Records a CUDA error text for dd_last_cuda_error() and returns DD_ERR_CUDA.
int cuda_fail(cudaError_t e, const char *where);

// Sets the text dd_last_cuda_error() returns.
void set_error_text(const char *text);

void count_launch(unsigned n = 1);

// Launches a kernel that may be brought onto the SMs while the one before it on the stream is still running, once every CTA of that one
// has executed ddptx::grid_trigger() or ended.  Every CTA of the launched kernel executes ddptx::grid_wait() before its threads read or
// write global memory (or depends, through a barrier of its own, on a thread that has): the wait returns when the kernels before it have
// ended and what they wrote can be seen, so that calls on one stream keep their order.  `cluster`: CTAs per cluster.
// Calls that follow one another directly lose the gap between two kernels and the set-up before the wait (barriers, TMEM, tensor map
// prefetch): attention 1 x 4 x 128 x 64 4.6 -> 3.6 us a call, 1 x 32 x 1024 x 128 19.7 -> 19.0, verification of 128 rows of 1024 7.5 ->
// 6.8, the head's three kernels over 64 rows of 1000
// 14.8 -> 12.2.  A captured graph keeps these edges.  `early` false: an ordinary launch, behind the end of the kernel before.
template <typename... Params, typename... Args>
cudaError_t launch_as(bool early, void (*kernel)(Params...), unsigned grid, unsigned threads, int smem, cudaStream_t stream, int cluster,
                      const Args &...args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = (size_t)smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = early ? 1 : 0;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = (unsigned)cluster;
    attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = cluster > 1 ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, kernel, args...);
}

template <typename... Params, typename... Args>
cudaError_t launch(void (*kernel)(Params...), unsigned grid, unsigned threads, int smem, cudaStream_t stream, int cluster, const Args &...args)
{
    return launch_as(true, kernel, grid, threads, smem, stream, cluster, args...);
}

#define DD_CUDA_TRY(expr)                                         \
    do {                                                          \
        cudaError_t _e = (expr);                                  \
        if (_e != cudaSuccess) return ::dd::cuda_fail(_e, #expr); \
    } while (0)

}  // namespace dd
