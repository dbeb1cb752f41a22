// Internal declarations shared by the translation units of libfp8attn.so.
#pragma once
#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include "fp8attn.h"

namespace fp8attn {

// Workspace layout (device memory, caller-owned, zero-filled once):
//   [0,4)    device status word (fp8attn_status_t, 0 = ok); first error wins
//   [4,8)    detail code of that error (which wait expired, which CTA)
//   [16,20)  blocks of a one-pass kernel that are done; zero between calls
//   [256, 4352) the one-pass kernels' own words (values that their blocks publish to one another);
//                       zero between calls.  Their place must not depend on B*H: one workspace
//                       serves calls of all sizes up to its own, and nothing but these kernels
//                       may ever write there.
//   [4352, 4352 + 12*B*H) three sets of per-(b,h) absmax accumulators (fp32 bit
//                       patterns): one is used by fp8attn_quantize, all three (Q, K, V)
//                       by fp8attn_quantize_qkv; cleared at the start of every call that uses
//                       them, left as they are at its end.  fp8attn_perturb keeps its per-head
//                       sums of squares (fp64) here too.
constexpr size_t kWsStatusOffset = 0;
constexpr size_t kWsDetailOffset = 4;
constexpr size_t kWsCounterOffset = 16;
constexpr size_t kWsWordsOffset = 256;
constexpr int kOnePassWords = 1024;
constexpr size_t kWsAmaxOffset = kWsWordsOffset + sizeof(uint32_t) * kOnePassWords;
// detail code (bits 24..31 of the detail word) of an expired grid-wide wait of a one-pass kernel
constexpr uint32_t kDetailGridWait = 32;

// (16 bytes per head beyond the accumulators are unused: the size that callers were told before)
inline size_t workspace_bytes(int B, int H) {
    const size_t heads = (size_t)B * (size_t)H;
    auto up = [](size_t x) { return (x + 255) / 256 * 256; };
    return kWsWordsOffset + up(12 * heads) + up(sizeof(uint32_t) * kOnePassWords + 16 * heads);
}

// Scratch of the tail split (FP8ATTN_SPLIT_TAIL), appended to the workspace: partial results
// of fewer than one CTA per SM of the current device, `rows` rows of d + 4 floats each (api.cu).
// A caller may bring scratch for CTAs of 256 rows; with 384 at d = 64 the split has all the room it
// can use.
size_t split_scratch_bytes(int d, int rows);
inline int split_scratch_rows(int d) { return d == 64 ? 384 : 256; }

void count_launch();

// quantize.cu
int launch_quantize(const void* x_bf16, int64_t n_heads, int64_t elems_per_head,
                    const float* scale_in, void* x_fp8, float* scale_out,
                    uint32_t* amax_bits, uint32_t flags, uint32_t* status, uint32_t* counters, uint32_t* words,
                    cudaStream_t stream);

// `status`, `counters`, `words`: the workspace's status words, its counters and the one-pass kernels'
// own words (NULL: no workspace, two passes).
int launch_quantize_qkv(const void* q_train, const void* k, const void* v, const void* q_test,
                        int64_t n_heads, int64_t elems_train, int64_t elems_test, void* q_train_fp8,
                        void* k_fp8, void* v_fp8, void* q_test_fp8, float* scale_q, float* scale_k,
                        float* scale_v, uint32_t* amax_bits, uint32_t flags, uint32_t* status,
                        uint32_t* counters, uint32_t* words, cudaStream_t stream,
                        int32_t* key_dest = nullptr, int d = 64);

// The form that a quantization of these sizes takes (tensors: 1 or 3): stages of the staged kernel, -1: a
// block per head, 0: two passes.
int quantize_stages(int tensors, int64_t n_heads, int64_t elems_train, int64_t elems_test, uint32_t flags, int sms);

// launch_quantize of a bf16 tensor by the staged kernel, every wait of which ends after that many clocks
int launch_quantize_timeout_selftest(const void* x_bf16, int64_t n_heads, int64_t elems_per_head, void* x_fp8,
                                     float* scale_out, uint32_t* amax_bits, uint32_t* status, uint32_t* counters,
                                     uint32_t* words, int64_t wait_clocks, cudaStream_t stream);

// key_order.cu
// dest[b,h,r] = the row that key r of head (b,h) moves to: the keys of largest norm first.
// norm_scratch: device memory for one fp32 per key (its squared norm), the heads
// norm_stride_bytes apart; compute_norms: fill it from k16 first (else it is filled already).
int launch_key_order(const void* k16, int64_t n_heads, int64_t n_train, int d, bool half, int32_t* dest,
                     void* norm_scratch, int64_t norm_stride_bytes, bool compute_norms, cudaStream_t stream);
// out[b,h,dest[b,h,r],:] = x[b,h,r,:] for a 16-bit tensor
int launch_reorder_rows(const void* x16, int64_t n_heads, int64_t rows, int d, const int32_t* dest, void* out16,
                        cudaStream_t stream);

// perturb.cu
int launch_perturb(const void* x_bf16, int64_t n_heads, int64_t elems_per_head, float epsilon,
                   uint64_t seed, uint32_t stream_id, void* out_bf16, float* rho_out, double* sumsq,
                   cudaStream_t stream);

// attention.cu
struct AttnParams {
    const void* q_train; const void* q_test; const void* k; const void* v;
    const float* scale_q; const float* scale_k; const float* scale_v;  // NULL for bf16
    int B, H; int64_t n_train, n_test; int d;
    float softmax_scale;
    uint32_t flags;    // FP8ATTN_* forward flags
    void* out_train; void* out_test;
    uint32_t* status;  // workspace status words
    float* partial;    // scratch of the tail split (NULL: none)
    size_t partial_bytes;
};
int launch_icl_attention(const AttnParams& p, bool fp8, cudaStream_t stream);
// Query rows per CTA that a forward call of these sizes and flags uses on a device with `sms` SMs and
// with that much scratch for the tail split: 256, 128 in small launches, or at d = 64 also 384 (attention.cu says when).
int attention_rows_per_cta(int B, int H, int64_t n_train, int64_t n_test, int d, uint32_t flags, int sms,
                           size_t partial_bytes = (size_t)1 << 40);
int launch_wait_timeout_selftest(uint32_t* status, uint64_t limit_ns, cudaStream_t stream);

}  // namespace fp8attn
