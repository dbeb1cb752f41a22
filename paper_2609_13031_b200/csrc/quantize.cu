// Per-head absmax quantization of bf16 (or IEEE fp16) tensors to e4m3 (paper Eq. 2).
//
// Calls whose heads fit on chip take one pass: short heads a block each (quantize_heads_kernel), longer
// ones all SMs together (staged.cuh): 2 B read + 1 B written per element.  The others
// (heads of more than 16 MB, an order of the keys, scales given, or on request) take two HBM-bound kernels:
//   absmax_kernel    max |x| per head, packed bf16x2 max, one atomicMax per block
//   quantize_kernel  s = amax/448, y = x/s (IEEE fp32), cvt.rn.satfinite.e4m3x2
// Algorithmic traffic: 2 B read per element for the maximum, 2 B read + 1 B
// written for the conversion (5 B per element; 3 B when the scale is given).
// The conversion walks each head backwards so that it starts on the part of the
// head the maximum pass touched last, which is still in L2.
// The IEEE division x/s is not evaluated per element but by three multiply-adds that give the same
// quotient (quantize_math.cuh).
#include <mutex>

#include "common.h"
#include "quantize_math.cuh"
#include "staged.cuh"

namespace fp8attn {
namespace {

constexpr int kThreads = 256;

// SMs of the current device (0 on error)
int sm_count() {
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return 0;
    return sms;
}

// One block's share of max |x| over head blockIdx.y (vecs_per_head 16-byte vectors),
// merged into amax_bits[blockIdx.y].
// With kNorm it also leaves the squared norm of every row (vecs_per_row 16-byte vectors, 8 or
// 16; fp32 bit pattern) in row_norm[row] of the head: the vectors of a row sit in neighbouring
// lanes, whose loop conditions agree (all bounds are multiples of the row length), so the lanes
// of a row add up under a mask of their own.
template <bool kHalf, bool kNorm = false>
__device__ __forceinline__ void absmax_body(const uint4* __restrict__ x, int64_t vecs_per_head,
                                            uint32_t* __restrict__ amax_bits,
                                            uint32_t* __restrict__ row_norm = nullptr, int vecs_per_row = 8) {
    using T = In16<kHalf>;
    using V2 = typename T::V2;
    auto am = [](uint32_t a, uint32_t b) { return __hmax2(__habs2(T::as2(a)), __habs2(T::as2(b))); };
    const uint32_t row_mask = (vecs_per_row == 16 ? 0xffffu : 0xffu) << (threadIdx.x & 31 & ~(vecs_per_row - 1));
    auto norm_of = [&](const uint4& v, int64_t vec) {
        const uint32_t w[4] = {v.x, v.y, v.z, v.w};
        float q = 0.f;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const float lo = T::lo(w[k]), hi = T::hi(w[k]);
            q = fmaf(lo, lo, q);
            q = fmaf(hi, hi, q);
        }
        for (int o = vecs_per_row >> 1; o > 0; o >>= 1) q += __shfl_xor_sync(row_mask, q, o);
        if ((vec & (vecs_per_row - 1)) == 0) row_norm[vec / vecs_per_row] = __float_as_uint(q);
    };
    const uint4* xh = x + (int64_t)blockIdx.y * vecs_per_head;
    V2 m = T::as2(0u);
    int64_t stride = (int64_t)gridDim.x * kThreads;
    int64_t i = (int64_t)blockIdx.x * kThreads + threadIdx.x;
    for (; i + 3 * stride < vecs_per_head; i += 4 * stride) {
        uint4 a = ld_nc_v4(xh + i), b = ld_nc_v4(xh + i + stride);
        uint4 c = ld_nc_v4(xh + i + 2 * stride), e = ld_nc_v4(xh + i + 3 * stride);
        if (kNorm) {
            norm_of(a, i);
            norm_of(b, i + stride);
            norm_of(c, i + 2 * stride);
            norm_of(e, i + 3 * stride);
        }
        V2 m0 = am(a.x, a.y), m1 = am(a.z, a.w), m2 = am(b.x, b.y), m3 = am(b.z, b.w);
        V2 m4 = am(c.x, c.y), m5 = am(c.z, c.w), m6 = am(e.x, e.y), m7 = am(e.z, e.w);
        m = __hmax2(m, __hmax2(__hmax2(__hmax2(m0, m1), __hmax2(m2, m3)),
                               __hmax2(__hmax2(m4, m5), __hmax2(m6, m7))));
    }
    for (; i < vecs_per_head; i += stride) {
        uint4 a = ld_nc_v4(xh + i);
        if (kNorm) norm_of(a, i);
        m = __hmax2(m, __hmax2(am(a.x, a.y), am(a.z, a.w)));
    }
    // |x| as a non-negative fp32 bit pattern orders like an unsigned integer
    float f = fmaxf(__low2float(m), __high2float(m));
    uint32_t bits = __float_as_uint(f);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) bits = max(bits, __shfl_xor_sync(0xffffffffu, bits, o));
    __shared__ uint32_t warp_max[kThreads / 32];
    if ((threadIdx.x & 31) == 0) warp_max[threadIdx.x >> 5] = bits;
    __syncthreads();
    if (threadIdx.x < 32) {
        bits = threadIdx.x < kThreads / 32 ? warp_max[threadIdx.x] : 0u;
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) bits = max(bits, __shfl_xor_sync(0xffffffffu, bits, o));
        if (threadIdx.x == 0) atomicMax(amax_bits + blockIdx.y, bits);
    }
}

// grid: (blocks_per_head, n_heads).
template <bool kHalf>
__global__ void __launch_bounds__(kThreads)
absmax_kernel(const uint4* __restrict__ x, int64_t vecs_per_head, uint32_t* __restrict__ amax_bits) {
    absmax_body<kHalf>(x, vecs_per_head, amax_bits);
}

// One block's share of head blockIdx.y.  Each thread turns 32 B of 16-bit input into
// 16 B of e4m3 per step.  pairs_per_head = elems_per_head / 16.
// `row_dest` (NULL: none) sends the codes of row r of a head to row row_dest[r] of the output;
// a row is 2^pairs_per_row_shift pairs.
template <bool kHalf>
__device__ __forceinline__ void quantize_body(const uint4* __restrict__ x, int64_t pairs_per_head,
                                              const float* __restrict__ scale_in,
                                              const uint32_t* __restrict__ amax_bits,
                                              uint4* __restrict__ out, float* __restrict__ scale_out,
                                              const int32_t* __restrict__ row_dest = nullptr,
                                              int pairs_per_row_shift = 0) {
    const float s = scale_in != nullptr ? scale_in[blockIdx.y] : head_scale(__uint_as_float(amax_bits[blockIdx.y]));
    if (blockIdx.x == 0 && threadIdx.x == 0 && scale_out != nullptr) scale_out[blockIdx.y] = s;
    const Divisor dv = divisor(s);
    const uint4* xh = x + (int64_t)blockIdx.y * pairs_per_head * 2;
    uint4* oh = out + (int64_t)blockIdx.y * pairs_per_head;
    int64_t stride = (int64_t)gridDim.x * kThreads;
    // walk the head from its end towards its start
    for (int64_t r = (int64_t)blockIdx.x * kThreads + threadIdx.x; r < pairs_per_head; r += stride) {
        int64_t i = pairs_per_head - 1 - r;
        uint4 a = ld_nc_v4(xh + 2 * i), b = ld_nc_v4(xh + 2 * i + 1);
        const uint2 o0 = dv.direct ? quant8_direct<kHalf>(a, dv) : quant8<kHalf, true>(a, dv);
        const uint2 o1 = dv.direct ? quant8_direct<kHalf>(b, dv) : quant8<kHalf, true>(b, dv);
        const uint4 o = make_uint4(o0.x, o0.y, o1.x, o1.y);
        int64_t dst = i;
        if (row_dest != nullptr) {
            const int64_t row = i >> pairs_per_row_shift;
            dst = ((int64_t)row_dest[(int64_t)blockIdx.y * (pairs_per_head >> pairs_per_row_shift) + row]
                   << pairs_per_row_shift) + (i - (row << pairs_per_row_shift));
        }
        oh[dst] = o;
    }
}

// grid: (blocks_per_head, n_heads).
template <bool kHalf>
__global__ void __launch_bounds__(kThreads)
quantize_kernel(const uint4* __restrict__ x, int64_t pairs_per_head,
                const float* __restrict__ scale_in, const uint32_t* __restrict__ amax_bits,
                uint4* __restrict__ out, float* __restrict__ scale_out) {
    quantize_body<kHalf>(x, pairs_per_head, scale_in, amax_bits, out, scale_out);
}

// All tensors of one attention call in two launches: blockIdx.z picks the tensor.
struct QuantBatch {
    const uint4* x[4];
    uint4* out[4];
    int64_t pairs_per_head[4];
    const float* scale_in[4];     // given scales (NULL: derive the scale from amax_in)
    const uint32_t* amax_in[4];   // accumulators the scale is derived from
    uint32_t* amax_acc[4];        // accumulators this tensor's maximum goes to (NULL: none)
    float* scale_out[4];
    const int32_t* row_dest[4];   // output row of every input row, per head (NULL: the same row)
    int pairs_per_row_shift;      // log2(d / 16)
};

// kNorm: the pass over K (z = 1) also leaves the keys' squared norms in key_norm (one word per
// key, the heads key_norm_stride words apart).
template <bool kHalf, bool kNorm = false>
__global__ void __launch_bounds__(kThreads)
absmax_batch_kernel(const QuantBatch b, uint32_t* key_norm = nullptr, int64_t key_norm_stride = 0) {
    const int z = blockIdx.z;
    if (b.amax_acc[z] == nullptr || b.pairs_per_head[z] <= 0) return;
    if (kNorm && z == 1)
        absmax_body<kHalf, true>(b.x[z], b.pairs_per_head[z] * 2, b.amax_acc[z],
                                 key_norm + (int64_t)blockIdx.y * key_norm_stride, 2 << b.pairs_per_row_shift);
    else
        absmax_body<kHalf>(b.x[z], b.pairs_per_head[z] * 2, b.amax_acc[z]);
}

template <bool kHalf>
__global__ void __launch_bounds__(kThreads) quantize_batch_kernel(const QuantBatch b) {
    const int z = blockIdx.z;
    quantize_body<kHalf>(b.x[z], b.pairs_per_head[z], b.scale_in[z], b.amax_in[z], b.out[z], b.scale_out[z],
                         b.row_dest[z], b.pairs_per_row_shift);
}


// Calls of more than this many 16-bit input bytes clear their words in a launch of their own first
// (which also starts on the data); smaller ones rely on what the last call left.
constexpr int64_t kOneLaunchMaxBytes = 48ll << 20;

// Short heads: one block per head holds it in registers between the maximum and the conversion.
// Nothing is exchanged between blocks.  Test rows are cut into pieces with blocks of their own, each of
// which takes the maximum of the train queries' head once more (from L2) instead of waiting for it; where
// there are heads enough to fill the SMs, the block of the train queries converts them.
// What bounds it: latency in small calls (one way in, one block-wide maximum, one way out); the
// exchange of the staged kernel took half of such a call.  With many heads HBM.
// Graph-replayed, staged kernel -> this one: 2 heads of 512 + 128 rows x 64 9.4 -> 3.5 us, 8 heads
// 11.0 -> 3.7 us, 8 heads of 1,024 + 256 11.1 -> 4.7 us; two passes -> this one (where the staged kernel
// took longer or did not take the call): 1,024 heads of 64 + 16 rows x 64 18.6 -> 9.3 us, 4,096 heads of
// 128 + 32 rows x 64 88 -> 64 us.
constexpr int kHeadPer = 8;                         // vectors per thread, at most
constexpr int kHeadVecs = 1024 * kHeadPer;          // 131,072 bytes: 1,024 rows x 64, 512 x 128

struct HeadArgs {
    const uint4* x[4];
    uint2* out[4];
    float* scale_out[4];
    const uint32_t* status;     // write nothing while an error is recorded there (NULL: do not look)
    int tensors, n_heads;
    int vecs;                   // per head of the tensors that are reduced
    int counts;                 // the test rows enter the maximum of tensor 0
    int64_t test_vecs;          // per head
    int pieces;                 // of the test rows of a head; 0: the block of tensor 0 converts them
    int64_t piece_vecs;
};

__device__ __forceinline__ uint32_t recorded_error(const HeadArgs& a) {
    return threadIdx.x == 0 && a.status != nullptr ? *reinterpret_cast<const volatile uint32_t*>(a.status) : 0u;
}
template <bool kHalf>
__device__ __forceinline__ bool block_divisor(typename In16<kHalf>::V2 m, uint32_t* warp_max, uint32_t error, Divisor& dv) {
    const uint32_t w = *reinterpret_cast<const uint32_t*>(&m);
    uint32_t top = __reduce_max_sync(0xffffffffu, max(w & 0xffffu, w >> 16));
    if ((threadIdx.x & 31) == 0) warp_max[threadIdx.x >> 5] = top;
    if (__syncthreads_or((int)error)) return false;
    top = __reduce_max_sync(0xffffffffu, (threadIdx.x & 31) < blockDim.x / 32 ? warp_max[threadIdx.x & 31] : 0u);
    dv = divisor(head_scale(In16<kHalf>::lo(top)));
    return true;
}
// (the per-element division stays out of the unrolled loops: small calls pay for the code they fetch)
template <bool kHalf>
__device__ __noinline__ void convert_direct(const uint4* x, uint2* out, int64_t n, Divisor dv) {
#pragma unroll 1
    for (int64_t i = threadIdx.x; i < n; i += blockDim.x) out[i] = quant8_direct<kHalf>(ld_nc_v4(x + i), dv);
}
// `n` vectors, four loads of a thread under way at a time
template <bool kHalf>
__device__ __forceinline__ void convert_rows(const uint4* x, uint2* out, int64_t n, const Divisor& dv) {
    if (dv.direct) return convert_direct<kHalf>(x, out, n, dv);
    for (int64_t i = threadIdx.x; i < n; i += 4 * blockDim.x) {
        uint4 v[4];
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (i + k * blockDim.x < n) v[k] = ld_nc_v4(x + i + k * blockDim.x);
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (i + k * blockDim.x < n) out[i + k * blockDim.x] = quant8<kHalf, true>(v[k], dv);
    }
}

template <bool kHalf>
__global__ void __launch_bounds__(1024) quantize_heads_kernel(const __grid_constant__ HeadArgs a) {
    using T = In16<kHalf>;
    __shared__ uint32_t warp_max[32];
    const int tid = threadIdx.x, mains = a.tensors * a.n_heads;
    typename T::V2 m = T::as2(0u);
    if ((int)blockIdx.x < mains) {
        const int head = (int)blockIdx.x / a.tensors, z = (int)blockIdx.x - head * a.tensors;
        const uint4* x = a.x[z] + (int64_t)head * a.vecs;
        uint4 v[kHeadPer];
#pragma unroll
        for (int k = 0; k < kHeadPer; ++k) {
            const int i = tid + k * (int)blockDim.x;
            v[k] = i < a.vecs ? ld_nc_v4(x + i) : make_uint4(0u, 0u, 0u, 0u);
        }
        const uint32_t error = recorded_error(a);
#pragma unroll
        for (int k = 0; k < kHeadPer; ++k) m = absmax8<kHalf>(m, v[k]);
        const uint4* test_x = a.x[3] + head * a.test_vecs;
        if (a.counts && z == 0)
            for (int64_t i = tid; i < a.test_vecs; i += blockDim.x) m = absmax8<kHalf>(m, ld_nc_v4(test_x + i));
        Divisor dv;
        if (!block_divisor<kHalf>(m, warp_max, error, dv)) return;
        if (tid == 0) a.scale_out[z][head] = dv.s;
        uint2* out = a.out[z] + (int64_t)head * a.vecs;
        if (dv.direct) {
            convert_direct<kHalf>(x, out, a.vecs, dv);
        } else {
#pragma unroll
            for (int k = 0; k < kHeadPer; ++k) {
                const int i = tid + k * (int)blockDim.x;
                if (i < a.vecs) out[i] = quant8<kHalf, false>(v[k], dv);
            }
        }
        if (z == 0 && a.pieces == 0) convert_rows<kHalf>(test_x, a.out[3] + head * a.test_vecs, a.test_vecs, dv);
    } else {
        const int item = (int)blockIdx.x - mains, head = item / a.pieces;
        const int64_t first = (int64_t)(item - head * a.pieces) * a.piece_vecs;
        const uint4* head_x = a.x[0] + (int64_t)head * a.vecs;
        const uint4* test_x = a.x[3] + head * a.test_vecs;
        const uint32_t error = recorded_error(a);
#pragma unroll 4
        for (int i = tid; i < a.vecs; i += blockDim.x) m = absmax8<kHalf>(m, ld_nc_v4(head_x + i));
        if (a.counts)
            for (int64_t i = tid; i < a.test_vecs; i += blockDim.x) m = absmax8<kHalf>(m, ld_nc_v4(test_x + i));
        Divisor dv;
        if (!block_divisor<kHalf>(m, warp_max, error, dv)) return;
        convert_rows<kHalf>(test_x + first, a.out[3] + head * a.test_vecs + first, min(a.piece_vecs, a.test_vecs - first), dv);
    }
}

// Whether a call of more than kOneLaunchMaxBytes, two launches in either form, is faster in one pass.  Every
// byte crosses the HBM interface once instead of twice, but a stage has a cost of its own, so small calls,
// and heads that leave much of a stage empty (8.5 MB of the 16.8 MB that the SMs hold: one head per stage),
// do better in two passes.  Both times in us, fitted to 80 measured sizes (50 .. 900 MB, 1 .. 64 heads, graph-
// replayed, mean of inputs in L2 and not), within 15 % of each.  One pass / two: 8 heads of 12,289 + 3,000 x 128
// 42 / 39 us, 4 heads of 33,000 + 5,000 56 / 49 us, 2 heads of 33,200 + 8,300 33 / 28 us, 8 heads of 35,000 +
// 5,000 100 / 101 us, of 44,000 + 1,000 102 / 120 us, of 65,536 + 16,384 129 / 183 us.  Test rows that enter the
// maximum of the train queries are read by the blocks that hold those: 8 heads of 20,011 + 3,001 x 128 76 /
// 58 us, of 65,536 + 16,384 157 / 185 us.  Calls of two stages have had a kernel of their own since, 1-2 us faster
// than the estimate knows: 8 heads of 5,000 + 12,000 x 128 26.2 / 28.8 us (two passes here), of 5,000 + 32,768 43.1 / 41.5
// and 16 heads of 2,600 + 32,768 65.8 / 61.0 (one pass here).
bool one_pass_pays(const staged::Shape& a) {
    const double heads = a.units / a.tensors, mb = 16e-6;
    const double train = mb * (double)a.vecs * a.units, test = mb * (double)a.follow_vecs * heads;
    double one = 12.4 + 1.74 * a.stages + 0.175 * train;
    if (a.follow_vecs > 0) one += 5.5 + 0.21 * test;
    if (a.follow_counts) one += 3.3 * (a.stages < heads ? a.stages : heads);
    return one < 6.3 + 0.407 * (train + test);
}

// How a quantization runs.
struct Form {
    enum { kTwoPasses, kHeads, kStaged } kind;
    unsigned grid;
    staged::Shape shape;        // kStaged
    HeadArgs heads;             // kHeads: without its pointers
    unsigned threads;           // kHeads
    bool heed_status;           // a fused call that is one launch writes nothing while an error is recorded
};
Form quantize_form(int tensors, int64_t n_heads, int64_t elems_train, int64_t elems_test, uint32_t flags, int sms) {
    Form f = {};
    if ((flags & (FP8ATTN_SCALES_GIVEN | FP8ATTN_QKV_TWO_LAUNCHES)) || elems_train <= 0) return f;
    const int64_t vecs = elems_train / 8, follow = elems_test / 8;
    const bool counts = follow > 0 && (flags & FP8ATTN_QUERY_SCALE_FROM_ALL_ROWS);
    const bool large = (vecs * tensors + follow) * n_heads * 16 > kOneLaunchMaxBytes;
    f.heed_status = tensors == 3 && !large;
    if (vecs <= kHeadVecs) {
        if (counts && follow > kHeadVecs) return f;
        // Pieces of the test rows: two per SM, but none so small that reading the train queries again is
        // most of its work.  None where the train heads fill the SMs by themselves.
        // (16 heads of 300 + 20,000 x 128: 30 us, two passes 37 us; 4,096 heads of 128 + 32 x 64 with a block
        // for the test rows of every head took 90 us)
        int64_t piece = (follow * n_heads + 2 * sms - 1) / (2 * sms);
        if (piece < vecs / 4) piece = vecs / 4;
        if (piece < 1024) piece = 1024;
        if (piece > follow) piece = follow;
        const bool own = follow > 0 && !(tensors * n_heads >= 4 * sms && follow <= vecs);
        const int64_t pieces = own ? (follow + piece - 1) / piece : 0;
        if (n_heads * (tensors + pieces) > 0x7fffffffll) return f;
        f.kind = Form::kHeads;
        f.grid = (unsigned)(n_heads * (tensors + pieces));
        HeadArgs& a = f.heads;
        a.tensors = tensors;
        a.n_heads = (int)n_heads;
        a.vecs = (int)vecs;
        a.counts = counts;
        a.test_vecs = follow;
        a.pieces = (int)pieces;
        a.piece_vecs = piece;
        // four vectors per thread, more where a block is full
        const int64_t threads = (vecs + 4 * 32 - 1) / (4 * 32) * 32, least = pieces > 0 ? 256 : 64;
        f.threads = (unsigned)(threads < least ? least : threads > 1024 ? 1024 : threads);
        return f;
    }
    if (follow > 0x7fffffffll) return f;
    staged::Shape& a = f.shape;
    a.tensors = tensors;
    a.units = (int)(tensors * n_heads);
    a.vecs = vecs;
    a.follow_vecs = (uint32_t)follow;
    a.follow_counts = counts;
    a.cleared = large;
    f.grid = staged::plan(a, sms);
    if (f.grid > 0 && (!a.cleared || one_pass_pays(a))) f.kind = Form::kStaged;
    return f;
}

template <bool kHalf>
int launch_heads(const Form& f, const QuantBatch& b, const uint32_t* status, cudaStream_t stream) {
    HeadArgs a = f.heads;
    a.status = f.heed_status ? status : nullptr;
    for (int z = 0; z < 4; ++z) {
        a.x[z] = b.x[z];
        a.out[z] = reinterpret_cast<uint2*>(b.out[z]);
        a.scale_out[z] = b.scale_out[z];
    }
    quantize_heads_kernel<kHalf><<<f.grid, f.threads, 0, stream>>>(a);
    count_launch();
    return cudaGetLastError() == cudaSuccess ? FP8ATTN_OK : FP8ATTN_ERR_CUDA;
}

// The one-pass kernel for the tensors of `b`: tensors [0, tensors) and, if there are test rows, tensor 3
// with the scale of tensor 0.  amax_bits: the accumulators of the two-pass form, free here.
template <bool kHalf, bool kSelfTest = false>
int launch_staged(const Form& f, const QuantBatch& b, uint32_t* status, uint32_t* counters, uint32_t* words,
                  uint32_t* amax_bits, cudaStream_t stream, int64_t wait_clocks = 0) {
    staged::Args a = {};
    static_cast<staged::Shape&>(a) = f.shape;
    for (int z = 0; z < a.tensors; ++z) {
        a.x[z] = b.x[z];
        a.out[z] = b.out[z];
        a.result_out[z] = b.scale_out[z];
    }
    a.follow_x = b.x[3];
    a.follow_out = b.out[3];
    a.wait_clocks = wait_clocks;
    a.heed_status = f.heed_status;
    a.status = status;
    a.counter = counters;
    a.slots = words;
    a.heads = a.cleared ? amax_bits : words + a.sets * a.slots_per_set;
    return staged::launch<kHalf, kSelfTest>(a, f.grid, stream);
}

}  // namespace

int launch_quantize_qkv(const void* q_train, const void* k, const void* v, const void* q_test,
                        int64_t n_heads, int64_t elems_train, int64_t elems_test, void* q_train_fp8,
                        void* k_fp8, void* v_fp8, void* q_test_fp8, float* scale_q, float* scale_k,
                        float* scale_v, uint32_t* amax_bits, uint32_t flags, uint32_t* status,
                        uint32_t* counters, uint32_t* words, cudaStream_t stream, int32_t* key_dest, int d) {
    if (n_heads <= 0) return FP8ATTN_OK;
    if (n_heads > 65535) return FP8ATTN_ERR_UNSUPPORTED;
    QuantBatch b;
    const void* xs[4] = {q_train, k, v, q_test};
    void* outs[4] = {q_train_fp8, k_fp8, v_fp8, q_test_fp8};
    float* scales[4] = {scale_q, scale_k, scale_v, nullptr};
    for (int z = 0; z < 4; ++z) {
        b.x[z] = static_cast<const uint4*>(xs[z]);
        b.out[z] = static_cast<uint4*>(outs[z]);
        b.pairs_per_head[z] = (z == 3 ? elems_test : elems_train) / 16;
        // the test queries reuse the train-query maximum (slot 0): shared query scale
        b.amax_in[z] = amax_bits + (z == 3 ? 0 : z) * n_heads;
        b.amax_acc[z] = z == 3 ? nullptr : amax_bits + z * n_heads;
        // single-call form: the query scale covers train and test queries alike
        if (z == 3 && (flags & FP8ATTN_QUERY_SCALE_FROM_ALL_ROWS) && elems_test > 0) b.amax_acc[z] = amax_bits;
        b.scale_out[z] = scales[z];
        b.scale_in[z] = nullptr;
        // a key order applies to K and V alike: the attention sums over keys
        b.row_dest[z] = (z == 1 || z == 2) ? key_dest : nullptr;
        if (flags & FP8ATTN_SCALES_GIVEN) {
            // scales computed upstream: nothing to reduce, nothing to write back
            b.scale_in[z] = scales[z == 3 ? 0 : z];
            b.scale_out[z] = nullptr;
            b.amax_acc[z] = nullptr;
        }
    }
    b.pairs_per_row_shift = d == 128 ? 3 : 2;
    const int tensors = elems_test > 0 ? 4 : 3;
    const int sms = sm_count();
    if (sms <= 0) return FP8ATTN_ERR_CUDA;
    const bool half = (flags & FP8ATTN_INPUT_FP16) != 0;
    if (key_dest == nullptr) {
        const Form f = quantize_form(3, n_heads, elems_train, elems_test, flags, sms);
        if (f.kind == Form::kHeads) return half ? launch_heads<true>(f, b, status, stream) : launch_heads<false>(f, b, status, stream);
        if (f.kind == Form::kStaged) {
            const int rc = half ? launch_staged<true>(f, b, status, counters, words, amax_bits, stream)
                                : launch_staged<false>(f, b, status, counters, words, amax_bits, stream);
            if (rc != staged::kRefused) return rc;
        }
    }
    const int64_t want = ((int64_t)sms * 16 + n_heads * 3 - 1) / (n_heads * 3);
    // (blocks for the train rows; more only where the test rows are many times as many: blocks with
    // nothing to do cost 2 us in calls of 12 us, too few took 4 heads of 64 + 32,768 x 128 350 us, not 20)
    const int64_t most = elems_test / 4 > elems_train ? elems_test / 4 : elems_train;
    const int64_t have = (most / 16 + kThreads - 1) / kThreads;
    const unsigned bx = (unsigned)(want < have ? (want < 1 ? 1 : want) : (have < 1 ? 1 : have));
    if (!(flags & FP8ATTN_SCALES_GIVEN) &&
        cudaMemsetAsync(amax_bits, 0, sizeof(uint32_t) * 3 * n_heads, stream) != cudaSuccess)
        return FP8ATTN_ERR_CUDA;
    // A key order is built between the two passes: the keys' norms come out of the maximum pass
    // (or, where the scales are given and there is none, out of a pass of their own) and sit in
    // the K8 buffer until the conversion overwrites them.
    uint32_t* key_norm = reinterpret_cast<uint32_t*>(k_fp8);
    const int64_t key_norm_stride = elems_train / 4;        // K8 bytes per head, in words
    const int64_t keys = elems_train / d;
    if (elems_train > 0 && !(flags & FP8ATTN_SCALES_GIVEN)) {
        const dim3 grid(bx, (unsigned)n_heads, 4);
        if (key_dest != nullptr) {
            if (half) absmax_batch_kernel<true, true><<<grid, kThreads, 0, stream>>>(b, key_norm, key_norm_stride);
            else absmax_batch_kernel<false, true><<<grid, kThreads, 0, stream>>>(b, key_norm, key_norm_stride);
        } else {
            if (half) absmax_batch_kernel<true><<<grid, kThreads, 0, stream>>>(b);
            else absmax_batch_kernel<false><<<grid, kThreads, 0, stream>>>(b);
        }
        count_launch();
    }
    if (key_dest != nullptr && elems_train > 0) {
        const int rc = launch_key_order(k, n_heads, keys, d, half, key_dest, key_norm,
                                        key_norm_stride * 4, (flags & FP8ATTN_SCALES_GIVEN) != 0, stream);
        if (rc != FP8ATTN_OK) return rc;
    }
    if (half) quantize_batch_kernel<true><<<dim3(bx, (unsigned)n_heads, tensors), kThreads, 0, stream>>>(b);
    else quantize_batch_kernel<false><<<dim3(bx, (unsigned)n_heads, tensors), kThreads, 0, stream>>>(b);
    count_launch();
    return cudaGetLastError() == cudaSuccess ? FP8ATTN_OK : FP8ATTN_ERR_CUDA;
}

int launch_quantize(const void* x_bf16, int64_t n_heads, int64_t elems_per_head,
                    const float* scale_in, void* x_fp8, float* scale_out,
                    uint32_t* amax_bits, uint32_t flags, uint32_t* status, uint32_t* counters, uint32_t* words,
                    cudaStream_t stream) {
    const bool half = (flags & FP8ATTN_INPUT_FP16) != 0;
    if (n_heads <= 0) return FP8ATTN_OK;
    if (n_heads > 65535) return FP8ATTN_ERR_UNSUPPORTED;
    const int64_t vecs = elems_per_head / 8, pairs = elems_per_head / 16;
    // enough blocks to fill the SMs several times over, never more than the work
    const int sms = sm_count();
    if (sms <= 0) return FP8ATTN_ERR_CUDA;
    auto blocks_for = [&](int64_t units) {
        int64_t want = ((int64_t)sms * 16 + n_heads - 1) / n_heads;
        int64_t have = (units + kThreads - 1) / kThreads;
        int64_t b = want < have ? want : have;
        return (unsigned)(b < 1 ? 1 : b);
    };
    if (scale_in == nullptr && status != nullptr) {
        const Form f = quantize_form(1, n_heads, elems_per_head, 0, flags, sms);
        if (f.kind != Form::kTwoPasses) {
            QuantBatch b = {};
            b.x[0] = static_cast<const uint4*>(x_bf16);
            b.out[0] = static_cast<uint4*>(x_fp8);
            b.scale_out[0] = scale_out;
            if (f.kind == Form::kHeads) return half ? launch_heads<true>(f, b, status, stream) : launch_heads<false>(f, b, status, stream);
            const int rc = half ? launch_staged<true>(f, b, status, counters, words, amax_bits, stream)
                                : launch_staged<false>(f, b, status, counters, words, amax_bits, stream);
            if (rc != staged::kRefused) return rc;
        }
    }
    if (scale_in == nullptr) {
        if (cudaMemsetAsync(amax_bits, 0, sizeof(uint32_t) * n_heads, stream) != cudaSuccess)
            return FP8ATTN_ERR_CUDA;
        if (elems_per_head > 0) {
            const dim3 grid(blocks_for((vecs + 3) / 4), (unsigned)n_heads);
            if (half) absmax_kernel<true><<<grid, kThreads, 0, stream>>>((const uint4*)x_bf16, vecs, amax_bits);
            else absmax_kernel<false><<<grid, kThreads, 0, stream>>>((const uint4*)x_bf16, vecs, amax_bits);
            count_launch();
        }
    }
    // also launched for empty heads when the scale must be written out
    if (elems_per_head > 0 || scale_out != nullptr) {
        const dim3 grid(blocks_for(pairs), (unsigned)n_heads);
        if (half)
            quantize_kernel<true><<<grid, kThreads, 0, stream>>>((const uint4*)x_bf16, pairs, scale_in,
                                                                 amax_bits, (uint4*)x_fp8, scale_out);
        else
            quantize_kernel<false><<<grid, kThreads, 0, stream>>>((const uint4*)x_bf16, pairs, scale_in,
                                                                  amax_bits, (uint4*)x_fp8, scale_out);
        count_launch();
    }
    return cudaGetLastError() == cudaSuccess ? FP8ATTN_OK : FP8ATTN_ERR_CUDA;
}

int launch_quantize_timeout_selftest(const void* x_bf16, int64_t n_heads, int64_t elems_per_head, void* x_fp8,
                                     float* scale_out, uint32_t* amax_bits, uint32_t* status, uint32_t* counters,
                                     uint32_t* words, int64_t wait_clocks, cudaStream_t stream) {
    const int sms = sm_count();
    if (sms <= 0) return FP8ATTN_ERR_CUDA;
    const Form f = quantize_form(1, n_heads, elems_per_head, 0, 0u, sms);
    if (f.kind != Form::kStaged) return FP8ATTN_ERR_UNSUPPORTED;
    QuantBatch b = {};
    b.x[0] = static_cast<const uint4*>(x_bf16);
    b.out[0] = static_cast<uint4*>(x_fp8);
    b.scale_out[0] = scale_out;
    const int rc = launch_staged<false, true>(f, b, status, counters, words, amax_bits, stream, wait_clocks);
    return rc == staged::kRefused ? FP8ATTN_ERR_UNSUPPORTED : rc;
}

int quantize_stages(int tensors, int64_t n_heads, int64_t elems_train, int64_t elems_test, uint32_t flags, int sms) {
    const Form f = quantize_form(tensors, n_heads, elems_train, elems_test, flags, sms);
    return f.kind == Form::kHeads ? -1 : f.kind == Form::kStaged ? f.shape.stages : 0;
}

}  // namespace fp8attn

// ---------------------------------------------------------------------------
// Allocation-free variant of the quantizer.
//
// The per-head absmax accumulators normally live in the caller's workspace.
// Here they live in a fixed array inside the library image, so a caller needs
// nothing but its input and output buffers.
// ---------------------------------------------------------------------------
namespace fp8attn {
namespace {

constexpr int kStaticMaxHeads = FP8ATTN_NOALLOC_MAX_HEADS;

// Resident on every GPU that loads the library, until the process exits.
static __device__ __align__(256) uint32_t g_static_amax[kStaticMaxHeads];

constexpr int kMaxDevices = 64;
std::mutex g_static_mutex;
uint32_t* g_static_amax_addr[kMaxDevices] = {};

// Device address of g_static_amax on the current device.  In host code the
// symbol's name is only a handle, so the address is looked up once per device.
int static_amax_address(uint32_t** out) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return FP8ATTN_ERR_CUDA;
    if (dev < 0 || dev >= kMaxDevices) return FP8ATTN_ERR_UNSUPPORTED;
    std::lock_guard<std::mutex> lock(g_static_mutex);
    if (g_static_amax_addr[dev] == nullptr) {
        void* p = nullptr;
        if (cudaGetSymbolAddress(&p, g_static_amax) != cudaSuccess || p == nullptr)
            return FP8ATTN_ERR_CUDA;
        g_static_amax_addr[dev] = static_cast<uint32_t*>(p);
    }
    *out = g_static_amax_addr[dev];
    return FP8ATTN_OK;
}

}  // namespace
}  // namespace fp8attn

extern "C" int fp8attn_quantize_noalloc(const void* x_bf16, int B, int H, int64_t rows, int d,
                                        const float* scale_in, void* x_fp8, float* scale_out,
                                        void* cuda_stream) {
    using namespace fp8attn;
    if (B <= 0 || H <= 0 || rows < 0) return FP8ATTN_ERR_INVALID_ARG;
    if (d != 64 && d != 128) return FP8ATTN_ERR_UNSUPPORTED;
    if ((int64_t)B * H > kStaticMaxHeads) return FP8ATTN_ERR_TOO_LARGE;
    if (rows > 0 && (!x_bf16 || !x_fp8)) return FP8ATTN_ERR_INVALID_ARG;
    if (!scale_in && !scale_out) return FP8ATTN_ERR_INVALID_ARG;
    if (reinterpret_cast<uintptr_t>(x_bf16) % 16 || reinterpret_cast<uintptr_t>(x_fp8) % 16 ||
        reinterpret_cast<uintptr_t>(scale_in) % 4 || reinterpret_cast<uintptr_t>(scale_out) % 4)
        return FP8ATTN_ERR_INVALID_ARG;
    int dev = 0, major = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev) != cudaSuccess)
        return FP8ATTN_ERR_CUDA;
    if (major != 10) return FP8ATTN_ERR_UNSUPPORTED;
    uint32_t* amax = nullptr;
    int rc = static_amax_address(&amax);
    if (rc != FP8ATTN_OK) return rc;
    // launch_quantize clears the accumulators it uses at the start of every call
    return launch_quantize(x_bf16, (int64_t)B * H, rows * (int64_t)d, scale_in, x_fp8, scale_out, amax, 0u,
                           nullptr, nullptr, nullptr, static_cast<cudaStream_t>(cuda_stream));
}
