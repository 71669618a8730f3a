// Shared host-side helpers of libmpipe_enc (argument checks, status reporting).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>
#include "../../include/mpipe_enc.h"

namespace mpipe {

inline bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }
inline int cdiv(int a, int b) { return (a + b - 1) / b; }

// Number of SMs of the current device (cached per device id).
int sm_count();

// A kernel that uses more than 48 KB of dynamic shared memory must opt in once per device; doing it on every
// launch costs host time that shows on small microbatches.  The kernel is a template VALUE argument, so every
// kernel (every instantiation of a kernel template) has its own function-local table of the devices set up.
template <auto kernel>
inline bool ensure_dynamic_smem(int bytes) {
    static bool done[64] = {};
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0) return false;
    if (dev < 64 && done[dev]) return true;
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes) != cudaSuccess) return false;
    if (dev < 64) done[dev] = true;
    return true;
}

// Programmatic dependent launch.  Every kernel of the library is launched with the attribute that lets it start while the
// kernel before it in the stream is still running, runs its set-up (barriers, TMEM, descriptors) there, and calls pdl_wait()
// before it touches global memory: that returns when everything earlier in the stream has completed and is visible.  Only
// then does it call pdl_launch(), which lets the NEXT kernel start early in turn -- so a kernel that is running implies that
// everything before its predecessor has completed.  A predecessor from outside the library (a torch kernel, a copy) never
// triggers early; the wait then ends when it has finished, as in plain stream order.
// Takes the ~1.5 us of launch latency and the ~0.7 us of set-up between two kernels of a layer out of the critical path
// (24 layers on one 777-token image, seven kernels each: 2194 -> 1752 us).  A grid of more than one wave of small blocks is
// launched plainly: its blocks sit in the slots of the kernel that still runs and the start of the copy it is made of comes
// no earlier (gradient of 200 small images at head_dim 80: 383 us plain, 400 us with an early prepass and convert).
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
template <typename... KArgs, typename... Args>
inline cudaError_t launch_kernel_as(bool early, void (*kernel)(KArgs...), unsigned grid, unsigned block, size_t smem, cudaStream_t st,
                                    unsigned cluster, Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = early ? 1 : 0;
    at[1].id = cudaLaunchAttributeClusterDimension;
    at[1].val.clusterDim.x = cluster;
    at[1].val.clusterDim.y = at[1].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = cluster > 1 ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}
template <typename... KArgs, typename... Args>
inline cudaError_t launch_kernel(void (*kernel)(KArgs...), unsigned grid, unsigned block, size_t smem, cudaStream_t st,
                                 unsigned cluster, Args... args) {
    return launch_kernel_as(grid <= unsigned(8 * sm_count()), kernel, grid, block, smem, st, cluster, args...);
}

// Defined in gemm.cu, used by the layer forward: one projection that stores both GELU(u) and u.
int32_t linear_fwd_gelu_keep_preact(const void* a, const void* w, const void* bias, void* act, void* pre, int32_t M, int32_t N,
                                    int32_t K, int64_t lda, int64_t ldw, int64_t ldact, int64_t ldpre, int32_t* status_buf,
                                    void* stream);

// Up to two matrices that a projection brings into L2 for the kernels behind it.
struct LayerAhead {
    const void* ptr[2] = {nullptr, nullptr};
    uint32_t bytes[2] = {0, 0};
};

// Defined in gemm.cu, used by the layer: mpipe_linear_fwd / mpipe_linear_dgrad whose weights were complete before the previous kernel
// of the stream started (true behind any other kernel of the layer): they are loaded while that kernel still runs.
int32_t linear_fwd_in_layer(const void* a, const void* w, const void* bias, const void* residual, void* c, int32_t M, int32_t N, int32_t K,
                            int64_t lda, int64_t ldw, int64_t ldr, int64_t ldc, int32_t flags, int32_t* status_buf, void* stream,
                            const LayerAhead& ahead);
int32_t linear_dgrad_in_layer(const void* dy, const void* w, const void* gelu_input, void* dx, int32_t M, int32_t N, int32_t K, int64_t lddy,
                              int64_t ldw, int64_t ldu, int64_t lddx, int32_t* status_buf, void* stream);

// Defined in gemm.cu, used by the layer backward: mpipe_linear_wgrad that also adds the column sums of dy to db (fp32 [N]).
int32_t linear_wgrad_bias(const void* dy, const void* x, float* dw, float* db, int32_t n_tokens, int32_t N, int32_t K, int64_t lddy,
                          int64_t ldx, int64_t lddw, int32_t* status_buf, void* stream, const LayerAhead& ahead);

// Defined in attn_bwd.cu, used by the layer backward: mpipe_varlen_attn_bwd whose dQ and dK leave turned back by the rotary tables
// (both NULL: as they are).
int32_t varlen_attn_bwd_rope(const void* dout, const void* q, const void* k, const void* v, const void* o, const float* lse, void* dq,
                             void* dk, void* dv, int64_t tok_stride_qkv, int64_t head_stride_qkv, int64_t tok_stride_o,
                             int64_t head_stride_o, int64_t tok_stride_grad, int64_t head_stride_grad, const int32_t* cu_seqlens_dev,
                             int32_t n_seg, int32_t total_tokens, int32_t max_seqlen, const mpipe_work_item_t* bwd_items_dev,
                             int32_t n_bwd_items, int32_t n_heads, int32_t head_dim, float softmax_scale, const float* rope_cos,
                             const float* rope_sin, void* workspace, size_t workspace_bytes, int32_t* status_buf, void* stream);

// Defined in attn_fwd.cu, used by the layer forward: mpipe_varlen_attn_fwd; `settled` says that the device copy of the plan was
// complete before the previous kernel of the stream started (true behind any other kernel of the layer).
int32_t varlen_attn_fwd(const void* q, const void* k, const void* v, void* o, float* lse, int64_t tok_stride_qkv,
                        int64_t head_stride_qkv, int64_t tok_stride_o, int64_t head_stride_o, const int32_t* cu_seqlens_dev,
                        int32_t n_seg, int32_t total_tokens, int32_t max_seqlen, const mpipe_work_item_t* fwd_items_dev,
                        int32_t n_fwd_items, int32_t n_heads, int32_t head_dim, float softmax_scale, int32_t mode,
                        int32_t* status_buf, void* stream, bool settled);

// Optional measurement aid (mpipe_set_profile_events): events recorded around one kernel launch.  The slots
// are thread-local: they affect only launches made by the thread that set them, so concurrent callers of the
// library share no mutable state.
struct ProfileEvents {
    cudaEvent_t start = nullptr, stop = nullptr;
};
enum { kProfileFwd = 0, kProfileBwdMain = 1, kProfileMerge = 2, kProfileLinear = 3, kProfileLayerNorm = 4, kProfileSlots = 5 };
extern thread_local ProfileEvents g_profile[kProfileSlots];
inline void profile_start(int which, cudaStream_t st) {
    if (g_profile[which].start != nullptr) cudaEventRecord(g_profile[which].start, st);
}
inline void profile_stop(int which, cudaStream_t st) {
    if (g_profile[which].stop != nullptr) cudaEventRecord(g_profile[which].stop, st);
}

// Device-side: record the first finding in the caller's status buffer.
__device__ __forceinline__ void report_status(int32_t* status_buf, int32_t code, int32_t detail) {
    if (status_buf != nullptr && atomicCAS(status_buf, 0, code) == 0) status_buf[1] = detail;
}

// Work items are read from device memory that the host cannot inspect when it launches, so every CTA checks
// the whole list before it does anything else: an item is acceptable if its row range and its key range are
// non-empty, lie inside [0, T) and the row range is at most one tile.  One bad item rejects the plan as a whole --
// the kernel reports MPIPE_ERR_INDEX with the item's index and returns without reading or writing a tensor --
// which keeps every check out of the pipeline's loops.  A plan made by mpipe_seg_plan for the same total_tokens
// always passes.
__device__ __forceinline__ bool plan_item_ok(const mpipe_work_item_t& it, int32_t tile_rows, int32_t T) {
    return it.row_start >= 0 && it.row_len >= 1 && it.row_len <= tile_rows && it.row_start <= T - it.row_len &&
           it.kv_start >= 0 && it.kv_len >= 1 && it.kv_start <= T - it.kv_len;
}
// Returns true if every item passes.  All threads of the CTA must call it; `flag` is a shared-memory word.
static __device__ __noinline__ bool plan_ok_cta(const mpipe_work_item_t* items, int32_t n_items, int32_t tile_rows, int32_t T,
                                            int32_t* status_buf, int* flag) {
    if (threadIdx.x == 0) *flag = -1;
    __syncthreads();
    for (int i = threadIdx.x; i < n_items; i += blockDim.x)
        if (!plan_item_ok(items[i], tile_rows, T)) atomicMax(flag, i);
    __syncthreads();
    const int bad = *flag;
    if (bad >= 0 && blockIdx.x == 0 && threadIdx.x == 0) report_status(status_buf, MPIPE_ERR_INDEX, bad);
    return bad < 0;
}

}  // namespace mpipe
