// Host-side pieces of libmpipe_enc: the segment planner, the position validator, status strings.
#include <algorithm>
#include <cstring>
#include <numeric>
#include <vector>
#include "common.h"
#include "plan_words.h"
#include "sm100_ptx.cuh"

namespace mpipe {

// A segment plan's words on their way to the device as the arguments of a kernel: they are taken over when the kernel is launched, so
// there is no staging buffer to allocate, guard by an event and keep, and the kernels around it keep their early launches, which a
// copy engine between them forbids.  Bound by the launch (a few KB).  us, pinned copy -> arguments: the host's part of an upload of
// 0.3 KB 10.6 -> 6.8, of 19 KB 11.5 -> 9.4; steps of four images (229 tokens) 33 -> 28, of eight (6553 tokens) 182 -> 173, of 200
// thumbnails 500 -> 491.
template <int kWords>
struct alignas(16) PlanWords {
    uint32_t w[kWords];
};
template <int kWords>
__global__ void __launch_bounds__(256) plan_words_kernel(const __grid_constant__ PlanWords<kWords> src, uint32_t* __restrict__ dst, int32_t n) {
    pdl_wait();
    pdl_launch();
    for (int i = blockIdx.x * 256 + threadIdx.x; i < n; i += gridDim.x * 256) dst[i] = src.w[i];
}
template <int kWords>
static int32_t launch_plan_words(const void* words, int32_t n, void* dst, cudaStream_t st) {
    PlanWords<kWords> src;
    std::memcpy(src.w, words, size_t(n) * 4);
    uint32_t* out = static_cast<uint32_t*>(dst);
    void* args[3] = {&src, &out, &n};
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(unsigned((n + 255) / 256));
    cfg.blockDim = dim3(256);
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    const cudaError_t e = cudaLaunchKernelExC(&cfg, reinterpret_cast<const void*>(plan_words_kernel<kWords>), args);
    return e == cudaSuccess && cudaGetLastError() == cudaSuccess ? MPIPE_OK : MPIPE_ERR_CUDA;
}

thread_local ProfileEvents g_profile[kProfileSlots];

int sm_count() {
    static int cached[64] = {0};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 148;
    if (cached[dev] == 0) {
        int n = 0;
        if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0) n = 148;
        cached[dev] = n;
    }
    return cached[dev];
}

// Tiles of every non-empty segment, longest segment first (ties: lower index first).
static int32_t emit_items(const int32_t* counts, const int32_t* cu, const std::vector<int32_t>& order,
                          int32_t tile_rows, mpipe_work_item_t* out) {
    int64_t n_items = 0;
    for (int32_t s : order) {
        const int32_t n = counts[s];
        if (n == 0) continue;
        const int32_t tiles = (n + tile_rows - 1) / tile_rows;
        if (out != nullptr) {
            for (int32_t t = 0; t < tiles; ++t) {
                mpipe_work_item_t& it = out[n_items + t];
                it.seg = s;
                it.tile = t;
                it.row_start = cu[s] + t * tile_rows;
                it.row_len = std::min(tile_rows, n - t * tile_rows);
                it.kv_start = cu[s];
                it.kv_len = n;
            }
        }
        n_items += tiles;
    }
    return static_cast<int32_t>(n_items);
}

}  // namespace mpipe

extern "C" {

int32_t mpipe_plan_words_to_device(const void* words, int32_t n, void* dst, void* stream) {
    using namespace mpipe;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (n < 0 || n > kPlanWordsMax || (n > 0 && (words == nullptr || dst == nullptr))) return MPIPE_ERR_INVALID_ARG;
    if (n == 0) return MPIPE_OK;
    if (n <= 256) return launch_plan_words<256>(words, n, dst, st);      // (what a launch costs grows with the arguments' size)
    if (n <= 1024) return launch_plan_words<1024>(words, n, dst, st);
    if (n <= 3072) return launch_plan_words<3072>(words, n, dst, st);
    return launch_plan_words<kPlanWordsMax>(words, n, dst, st);
}

int32_t mpipe_seg_plan(const int32_t* patch_counts, int32_t n_seg, int32_t fwd_tile_rows, int32_t bwd_tile_rows,
                       int32_t mode, int32_t* cu_seqlens, int32_t* total_tokens, int32_t* max_seqlen,
                       mpipe_work_item_t* fwd_items, int32_t* n_fwd_items, mpipe_work_item_t* bwd_items,
                       int32_t* n_bwd_items) {
    if (n_seg < 0 || (n_seg > 0 && patch_counts == nullptr) || cu_seqlens == nullptr || total_tokens == nullptr ||
        max_seqlen == nullptr || n_fwd_items == nullptr || n_bwd_items == nullptr)
        return MPIPE_ERR_INVALID_ARG;
    if (fwd_tile_rows <= 0 || bwd_tile_rows <= 0) return MPIPE_ERR_INVALID_ARG;
    if (mode != MPIPE_ENC_FROZEN && mode != MPIPE_ENC_TRAINED) return MPIPE_ERR_INVALID_ARG;
    int64_t acc = 0;
    int32_t mx = 0;
    for (int32_t i = 0; i < n_seg; ++i) {
        if (patch_counts[i] < 0) return MPIPE_ERR_INVALID_ARG;
        acc += patch_counts[i];
        if (acc >= (int64_t(1) << 31)) return MPIPE_ERR_INVALID_ARG;
        mx = std::max(mx, patch_counts[i]);
    }
    cu_seqlens[0] = 0;
    for (int32_t i = 0; i < n_seg; ++i) cu_seqlens[i + 1] = cu_seqlens[i] + patch_counts[i];
    *total_tokens = cu_seqlens[n_seg];
    *max_seqlen = mx;

    std::vector<int32_t> order(static_cast<size_t>(n_seg));
    std::iota(order.begin(), order.end(), 0);
    std::stable_sort(order.begin(), order.end(),
                     [&](int32_t a, int32_t b) { return patch_counts[a] > patch_counts[b]; });
    *n_fwd_items = mpipe::emit_items(patch_counts, cu_seqlens, order, fwd_tile_rows, fwd_items);
    *n_bwd_items = (mode == MPIPE_ENC_TRAINED)
                       ? mpipe::emit_items(patch_counts, cu_seqlens, order, bwd_tile_rows, bwd_items)
                       : 0;
    return MPIPE_OK;
}

int32_t mpipe_validate_positions(const int32_t* positions, int32_t n, int32_t n_llm_tokens) {
    if (n < 0 || n_llm_tokens < 0 || (n > 0 && positions == nullptr)) return MPIPE_ERR_INVALID_ARG;
    std::vector<uint8_t> seen(static_cast<size_t>(n_llm_tokens), 0);
    for (int32_t i = 0; i < n; ++i) {
        const int32_t p = positions[i];
        if (p < 0 || p >= n_llm_tokens) return MPIPE_ERR_INDEX;
        if (seen[p]) return MPIPE_ERR_INVALID_ARG;
        seen[p] = 1;
    }
    return MPIPE_OK;
}

const char* mpipe_status_str(int32_t status) {
    switch (status) {
        case MPIPE_OK: return "ok";
        case MPIPE_ERR_INVALID_ARG: return "invalid argument";
        case MPIPE_ERR_UNSUPPORTED: return "unsupported configuration";
        case MPIPE_ERR_WORKSPACE: return "workspace missing or too small";
        case MPIPE_ERR_CUDA: return "CUDA call failed";
        case MPIPE_ERR_TIMEOUT: return "device wait timed out";
        case MPIPE_ERR_INDEX: return "index out of range";
        default: return "unknown status";
    }
}

int32_t mpipe_version(void) { return 100; }

int32_t mpipe_set_profile_events(int32_t which, void* start_event, void* stop_event) {
    if (which < 0 || which >= mpipe::kProfileSlots) return MPIPE_ERR_INVALID_ARG;
    mpipe::g_profile[which].start = static_cast<cudaEvent_t>(start_event);
    mpipe::g_profile[which].stop = static_cast<cudaEvent_t>(stop_event);
    return MPIPE_OK;
}

}  // extern "C"
