// Internal launch interfaces between the C-ABI layer and the kernels.
#pragma once
#include <cuda_runtime.h>
#include <cstdint>

#include "layout.h"

namespace bigbird {

struct FwdArgs {
    const void* q;
    const void* k;
    const void* v;
    const uint8_t* kpm;      // [B, N] or nullptr
    void* out;
    float* lse;              // may be nullptr
    int B, H, D, b, nb;
    int64_t N;
    float scale;
    int dtype;               // BIGBIRD_FP32 / BIGBIRD_BF16
    cudaStream_t stream;
};

struct BwdArgs {
    const void* q;
    const void* k;
    const void* v;
    const void* out;         // the forward result
    const float* lse;        // [B, H, N] from the forward pass
    const void* dout;        // gradient of the loss with respect to out
    const uint8_t* kpm;      // [B, N] or nullptr
    void* dq;
    void* dk;
    void* dv;
    int B, H, D, b, nb;
    int64_t N;
    float scale;
    int dtype;
    cudaStream_t stream;
};

// Per-device scratch owned by the library.
constexpr int kCounterSlots = 64;
struct DeviceScratch {
    int* status = nullptr;          // [2]: code, detail
    int* counters = nullptr;        // [kCounterSlots * 2] work counters of the dynamic scheduler, a pair per stream, zero between calls
    unsigned long long stream_ids[kCounterSlots] = {};     // the streams that own them
    int streams = 0;
};

// CUDA-core kernel (fp32 arithmetic).  Returns a cudaError_t.  *launches is incremented per kernel enqueued.
cudaError_t launch_attn_fwd_simt(const FwdArgs& a, const bigbird_layout& L, const DeviceLayout& dl, int sms, int* launches);

// CUDA-core gradient kernels (fp32 arithmetic): dq by query block, dk and dv by key block over the transposed lists.
// The workspace of a call comes from `pool`, in stream order.
cudaError_t launch_attn_bwd_simt(const BwdArgs& a, const bigbird_layout& L, const DeviceLayout& dl, cudaMemPool_t pool, int sms, int* launches);

// tcgen05 gradient kernels (bf16 tensors, b = D = 64).  The workspace of a call comes from `pool`, in stream order.  Returns a
// BIGBIRD_* code; *cuda_err receives the cudaError_t on BIGBIRD_ECUDA.
bool attn_bwd_sm100_takes(const BwdArgs& a);
int launch_attn_bwd_sm100(const BwdArgs& a, const bigbird_layout& L, const DeviceLayout& dl, cudaMemPool_t pool, int* status,
                          int* launches, cudaError_t* cuda_err);

// tcgen05 kernel (bf16 operands).  Returns a BIGBIRD_* code; *cuda_err receives the cudaError_t on BIGBIRD_ECUDA.
// Scratch of a call comes from `pool`, in stream order.
int launch_attn_fwd_sm100(const FwdArgs& a, const bigbird_layout& L, const DeviceLayout& dl, DeviceScratch& sc, cudaMemPool_t pool,
                          int* launches, cudaError_t* cuda_err);

// One-thread kernel whose bounded wait is left to expire (about two seconds); sets the device status word.
cudaError_t launch_wait_expiry_selftest(DeviceScratch& sc, cudaStream_t stream);

#ifdef __CUDACC__
// Every kernel of the library is launched so that it may begin before the kernel in front of it in the stream has drained: it lets
// the next one begin as soon as there is room, and waits for those in front before it touches memory that they may use.
__device__ __forceinline__ void grid_dependency_release() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void grid_dependency_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
#endif

}  // namespace bigbird
