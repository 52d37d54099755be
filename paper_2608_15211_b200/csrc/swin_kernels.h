// Host-side launch interface between the C ABI (api.cu) and the kernel files.
#pragma once
#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include "swin_common.cuh"

namespace terra {

void count_launch(cudaStream_t stream);   // after every launch: bumps the launch counter, closes an open timing scope
// Optional per-kernel timing (terra_profile_*): opens a scope (CUDA event on `stream`) that the next
// count_launch closes.  Does nothing unless profiling is enabled.
void prof_begin(const char* name, cudaStream_t stream);

// Launches `kernel` so that it may be brought up (barriers, tensor memory, shared memory) while the launch before it in the stream is
// still running; the kernel calls wait_for_prerequisites() before it touches what that launch reads or writes.  A chain of
// small kernels loses 2 to 3 us less at each joint.
template <typename... P, typename... A>
cudaError_t launch_dependent(void (*kernel)(P...), unsigned grid, unsigned block, size_t smem, cudaStream_t stream, A&&... args) {
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

// Launches `kernel`, where its CTAs wait for one another (`together`) only if all can be on the device at the same time.
template <typename... P, typename... A>
cudaError_t launch_together(void (*kernel)(P...), unsigned grid, unsigned block, size_t smem, cudaStream_t stream, bool together, A&&... args) {
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeCooperative;
    attr.val.cooperative = together;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

// Before a kernel's launch: allows it `smem` bytes of dynamic shared memory on the current device and, where `occupancy` is
// given, says how many CTAs of `threads` threads fit an SM.  Each thread remembers its last few kernels: the two runtime
// calls cost more host time than the launch of a small kernel.
cudaError_t prepare_kernel(const void* kernel, size_t smem, int threads = 0, int* occupancy = nullptr);

cudaError_t launch_route(const Geo& g, int32_t* perm, int32_t* inv_perm, int32_t* win_offsets,
                         int32_t* pos, int32_t* label, cudaStream_t stream);

cudaError_t launch_fwd_mma(const Geo& g, const void* q, const void* k, const void* v, const float* bias,
                           void* o, float* lse, int sm_count, cudaStream_t stream);
// the register-tile kernels for fp16 activations and gradients (same arguments)
cudaError_t launch_fwd_mma_f16(const Geo& g, const void* q, const void* k, const void* v, const float* bias,
                               void* o, float* lse, int sm_count, cudaStream_t stream);
bool bwd_small_supported_f16(const Geo& g);
cudaError_t launch_bwd_small_f16(const Geo& g, const void* q, const void* k, const void* v, const void* o, const void* d_o,
                                 const float* bias, const float* lse, void* dq, void* dk, void* dv, float* dbias,
                                 int sm_count, cudaStream_t stream);
// the tcgen05 kernels compiled for fp16 activations (same shapes, workspaces and helpers as the bf16 ones)
cudaError_t launch_fwd_tc_f16(const Geo& g, const void* q, const void* k, const void* v, const float* bias,
                              void* o, float* lse, void* workspace, int sm_count, cudaStream_t stream);
cudaError_t read_tc_status_f16(int* timed_out, cudaStream_t stream);
cudaError_t launch_bwd_tc_f16(const Geo& g, const void* q, const void* k, const void* v, const float* bias,
                              const void* o, const float* lse, const void* d_o, void* dq, void* dk, void* dv, float* dbias,
                              void* workspace, int sm_count, cudaStream_t stream);
cudaError_t read_bwd_tc_status_f16(int* timed_out);
cudaError_t launch_bwd_delta_f16(const Geo& g, const void* o, const void* d_o, float* delta, cudaStream_t stream);
cudaError_t launch_bwd_mma_f16(const Geo& g, const void* q, const void* k, const void* v, const float* bias,
                               const float* lse, const float* delta, const void* d_o,
                               void* dq, void* dk, void* dv, float* dbias, int sm_count, cudaStream_t stream);

// tcgen05 forward path (head dim 32, window side <= 16)
constexpr int kFwdBiasFloats = 2304;   // prepared bias table per head (padded rows, -inf zone, maximum in the last float)
bool fwd_tc_supported(const Geo& g);
bool pad16_layout(const Geo& g);       // window sides 9 .. 15: slots laid out 16 to a window row, bias codes with stride 48
size_t fwd_tc_workspace_bytes(const Geo& g);
cudaError_t launch_fwd_tc(const Geo& g, const void* q, const void* k, const void* v, const float* bias,
                          void* o, float* lse, void* workspace, int sm_count, cudaStream_t stream);
// synchronises the stream, reads and clears the device-side "a bounded wait expired" word
cudaError_t read_tc_status(int* timed_out, cudaStream_t stream);

// TMA variants of the two kernels above (grids of 16-wide windows whose window rows are runs of consecutive tokens):
// the shape test, and the encoder of a [tokens][channels] tensor map with a box of 32 channels x box_tokens tokens
bool tma_row_shape(const Geo& g);
bool make_row_map(void* cu_tensor_map, const Geo& g, const void* base, int token_stride, int box_tokens, int box_ch = 32);

// tcgen05 forward path for window sides 9 .. 128 (head dim 32: 17 .. 128) on any grid (attn_fwd_win.cu)
bool fwd_win_supported(const Geo& g);
size_t fwd_win_workspace_bytes(const Geo& g);
cudaError_t launch_fwd_win(const Geo& g, const void* q, const void* k, const void* v, const float* bias, void* o, float* lse, void* workspace,
                           int sm_count, cudaStream_t stream);
cudaError_t launch_fwd_win_f16(const Geo& g, const void* q, const void* k, const void* v, const float* bias, void* o, float* lse, void* workspace,
                               int sm_count, cudaStream_t stream);
cudaError_t read_fwd_win_status(int* timed_out);
cudaError_t read_fwd_win_status_f16(int* timed_out);
// tcgen05 forward path for head dims 64 and 128 and many complete windows of side 64 and 128 without mask labels (attn_fwd_tc64.cu)
bool fwd_tc64_pays(const Geo& g);
size_t fwd_tc64_workspace_bytes(const Geo& g);
cudaError_t launch_fwd_tc64(const Geo& g, const void* q, const void* k, const void* v, const float* bias, void* o, float* lse, void* workspace,
                            int sm_count, cudaStream_t stream);
cudaError_t launch_fwd_tc64_f16(const Geo& g, const void* q, const void* k, const void* v, const float* bias, void* o, float* lse, void* workspace,
                                int sm_count, cudaStream_t stream);
cudaError_t read_fwd_tc64_status(int* timed_out);     // after the stream has been synchronised
cudaError_t read_fwd_tc64_status_f16(int* timed_out);
// One-pass tcgen05 backward for window sides 9 .. 128 at head dim 128, 11 .. 128 at 64 and 17 .. 128 at 32, any grid.
struct OnePassPlan {
    int rw;                  // slots per window row
    int npad, rmax;          // slots of a window rounded up to 128; window rows rounded up to whole key tiles
    int strips, rl;          // strips of a full window row (0: sides up to 32); floats of a bias-table row
    int split_log2;          // a window's key tiles are shared by 1 << split_log2 units
    int gangs, gang, ring, rotate;   // or by `gang` CTAs, that add to one slab in turn: `gangs` of them, `ring` slabs each (gang 1: none)
    long long units;
    size_t off_bias0, off_bias1, off_acc, off_slabs, off_flags, bytes;      // workspace
    int flags;               // ints at off_flags
};
constexpr int kPlanSms = 148;          // SM count the plan is made for
constexpr int kMaxCtas = 160;          // CTAs whose dQ slabs fit the workspace
constexpr int kGangMin = 4;            // CTAs of a gang at least
constexpr double kGangLag = 5.5;       // half chunks from a CTA's turn to the next one's
bool bwd_onepass_supported(const Geo& g);
OnePassPlan bwd_onepass_plan(const Geo& g);
struct GangShape { int gangs, gang, rotate; };
GangShape fit_gangs(const OnePassPlan& p, long long units, int ctas);
int sms_of_stream(cudaStream_t stream, int device_sms);
cudaError_t launch_bwd_onepass(const Geo& g, const void* q, const void* k, const void* v, const float* bias, const void* o, const float* lse,
                               const void* d_o, void* dq, void* dk, void* dv, float* dbias, void* workspace, int sm_count, cudaStream_t stream);
cudaError_t launch_bwd_onepass_f16(const Geo& g, const void* q, const void* k, const void* v, const float* bias, const void* o, const float* lse,
                                   const void* d_o, void* dq, void* dk, void* dv, float* dbias, void* workspace, int sm_count, cudaStream_t stream);
cudaError_t read_bwd_onepass_status(int* timed_out);
cudaError_t read_bwd_onepass_status_f16(int* timed_out);

cudaError_t launch_bounded_wait_selftest(long long limit_cycles, cudaStream_t stream);
cudaError_t launch_bias_prep(const Geo& g, const float* bias, float* prep, cudaStream_t stream);

// tcgen05 backward path (head dim 32, window side <= 16)
bool bwd_tc_supported(const Geo& g);
size_t bwd_tc_workspace_bytes(const Geo& g);
cudaError_t launch_bwd_tc(const Geo& g, const void* q, const void* k, const void* v, const float* bias,
                          const void* o, const float* lse, const void* d_o, void* dq, void* dk, void* dv, float* dbias,
                          void* workspace, int sm_count, cudaStream_t stream);
cudaError_t read_bwd_tc_status(int* timed_out);

// delta[b, token, head] = sum_c dO * O   (fp32, same indexing as lse)
// the whole backward in one kernel for windows of at most 64 tokens (no delta kernel, no workspace)
bool bwd_small_supported(const Geo& g);
cudaError_t launch_bwd_small(const Geo& g, const void* q, const void* k, const void* v, const void* o, const void* d_o,
                             const float* bias, const float* lse, void* dq, void* dk, void* dv, float* dbias,
                             int sm_count, cudaStream_t stream);
cudaError_t launch_bwd_delta(const Geo& g, const void* o, const void* d_o, float* delta, cudaStream_t stream);

// dK, dV (key-tile CTAs) and dQ, dBias (query-tile CTAs)
cudaError_t launch_bwd_mma(const Geo& g, const void* q, const void* k, const void* v, const float* bias,
                           const float* lse, const float* delta, const void* d_o,
                           void* dq, void* dk, void* dv, float* dbias, int sm_count, cudaStream_t stream);

}  // namespace terra
