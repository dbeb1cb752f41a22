// The quantizer in one pass for heads that a block cannot hold by itself: an element crosses the HBM
// interface once on its way in and once on its way out, although its head's maximum comes first.
//
// What bounds it: HBM.  Two kernels, one per pass, read every element twice (5 bytes per element
// of the quantizer instead of 3), because a large call is more than L2 can hold between them.
// Here the first read stays on chip, in shared memory: 148 SMs hold 33 MB in two buffers per SM.
//
// A "unit" is one head of one tensor that is reduced.  The units of a call form a flat range, cut
// into stages of whole units that fit one buffer of every SM; of each stage every block (one per
// SM) holds an equal contiguous share, loaded by cp.async.bulk.  Per stage: the share has landed ->
// the worker warps reduce it, segment by segment (segment = the part of one unit inside the
// share) -> the exchange warp publishes the segments' values and collects those of the other
// blocks that share its units, while the workers convert the second half of the stage before ->
// they convert the first half of this one.  The load warp refills each half of a buffer as soon as
// it is converted, and has what there is no room for yet fetched to L2, so that HBM is read without
// a pause.  A value is published in words of its own together with a tag (the stage), so that a
// store and a poll carry it: no atomics, no fence, no counter (those took 3 us a stage, as much as
// the work).
//
// The blocks are launched cooperatively, i.e. resident together or not at all; the waits are
// bounded all the same (kWaitClocks: FP8ATTN_ERR_TIMEOUT in the status word).  The last block whose
// exchange warp has read all that it will read leaves the published words and the counter at zero for
// the next call, while the workers convert.  (At the end of the kernel the fence that orders this waits
// for the block's output stores: 1 us a call.)
//
// Measured, graph-replayed, one pass / two passes: 8 heads of 65,536 + 16,384 rows x 128 (654 MB in and
// out, 100 us at the copy rate) 126-130 / 183 us; x 64 72 / 94 us; 16 heads of 20,011 + 3,001 x 128 92-97 / 115 us;
// 8 heads 52-57 / 56 us; 8,192 + 2,048 x 64 14.5 / 20.5 us.  About 10 us go before the second stage: launch,
// the first stage's way in, and its exchange under the second's loads.
// (Tried before: 24 KB chunks handed out by tickets to a control thread and worker warps: 2.5 us per
// chunk for the hand-overs.  Accumulators and a grid-wide counter instead of tagged words: 154 us.
// Without the fetch to L2: 159 us.)
#pragma once
#include "common.h"
#include "quantize_math.cuh"
#include "sm100_ptx.cuh"

namespace fp8attn {
namespace staged {

using namespace ptx;

constexpr int kThreads = 1024;
constexpr int kWorkers = kThreads - 64;        // and one warp that issues the loads, one that exchanges values
constexpr int kBufVecs = 7088;                 // 16-byte vectors per buffer: a head of 65,536 x 128 over 148 SMs
constexpr int kParts = 2;                      // a buffer is given up in halves
constexpr size_t kSmemBytes = (size_t)2 * kBufVecs * 16;
constexpr int kMinVecs = kBufVecs;             // heads are longer than that, so that ...
constexpr int kMaxSegments = 2;                // ... a share is part of two at most
constexpr int kMaxFollowHeads = 32;            // whose rows follow in one block, in calls that clear nothing first
constexpr int64_t kWaitClocks = 4000000000ll;  // 2 s

// The sizes of a call and how it is cut (host arithmetic only, see plan()).
struct Shape {
    int tensors, units;         // tensors that are reduced; their heads
    int64_t vecs;               // 16-byte vectors per unit
    uint32_t follow_vecs;       // per head, of a tensor that takes the results of tensor 0 as they are ...
    int follow_counts;          // ... after entering its reduction
    bool cleared;               // a launch before clears the published words
    int stage_units;            // per stage (the last one may have fewer)
    int stages;
    // Published values: `sets` sets of slots_per_set.  Alternate stages use alternate sets: a block is in
    // stage s + 2 only after every block that it shares a unit with has collected stage s.  A shorter
    // last stage pairs other blocks with one another and has a set of its own.
    uint32_t slots_per_set;
    int sets, last_set;
};

struct Args : Shape {
    const uint4* x[3];          // the tensors that are reduced: unit u is head u / tensors of tensor u % tensors
    void* out[3];
    float* result_out[3];       // per head (NULL: none)
    const uint4* follow_x;      // values may lie outside the range of tensor 0
    void* follow_out;
    int64_t wait_clocks;        // limit of every wait of the self-test
    bool heed_status;           // write nothing while an error is recorded
    uint32_t* status;
    uint32_t* counter;          // blocks done
    uint32_t* slots;            // published values
    uint32_t* heads;            // published results of tensor 0, for the rows that follow it
};

// the workers and the exchange warp (barrier 0 is __syncthreads)
__device__ __forceinline__ void sync_exchange() { asm volatile("bar.sync 1, %0;" ::"n"(kWorkers + 32) : "memory"); }
__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
                 "l"(src), "r"(bytes), "r"(bar)
                 : "memory");
}
__device__ __forceinline__ void bulk_prefetch(const void* src, uint32_t bytes) {
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(src), "r"(bytes) : "memory");
}

// first position of block b's share of `total` vectors (128-byte lines stay whole).  A stage is at
// most kBufVecs vectors per SM: everything fits 32 bits.
__device__ __forceinline__ uint32_t cut(uint32_t total, uint32_t b) {
    return b == gridDim.x ? total : total * b / gridDim.x & ~7u;
}
// One block's share of one stage: n positions from cut(total, block) on, which are `segs` segments of
// the units from `unit` (of the stage) on; the first begins at vector `skip` of its unit.
struct Share {
    uint32_t total, unit, segs, skip, n;
    __device__ __forceinline__ Share(uint32_t stage_units, uint32_t vecs) {
        total = stage_units * vecs;
        const uint32_t lo = cut(total, blockIdx.x);
        n = cut(total, blockIdx.x + 1) - lo;
        unit = lo / vecs;
        skip = lo - unit * vecs;
        segs = n == 0 ? 0 : (skip + n + vecs - 1) / vecs;
    }
    // first and last + 1 position of segment g, and the vector of its unit that the first is
    __device__ __forceinline__ uint32_t begin(uint32_t g, uint32_t vecs) const { return g == 0 ? 0 : g * vecs - skip; }
    __device__ __forceinline__ uint32_t end(uint32_t g, uint32_t vecs) const { return min((g + 1) * vecs - skip, n); }
    __device__ __forceinline__ uint32_t at(uint32_t g) const { return g == 0 ? skip : 0; }
    __device__ __forceinline__ uint32_t half() const { return n / 2 & ~7u; }
    // the block that holds position x
    __device__ __forceinline__ uint32_t holder(uint32_t x) const {
        uint32_t b = min(x * gridDim.x / total, gridDim.x - 1);
        while (cut(total, b) > x) --b;
        while (cut(total, b + 1) <= x) ++b;
        return b;
    }
};

// A published value is one word: tag << 16 | maximum, the bit pattern of max |x| in the 16-bit type, which
// orders like an integer.
constexpr uint32_t kLost = 0xffffffffu;     // published: no tag (tags are below 0xffff)
__device__ __forceinline__ void publish(uint32_t* word, uint32_t tag, uint32_t v) {
    *reinterpret_cast<volatile uint32_t*>(word) = tag << 16 | v;
}
__device__ __forceinline__ uint32_t peek(const uint32_t* word) { return *reinterpret_cast<const volatile uint32_t*>(word); }
__device__ __forceinline__ bool tagged(uint32_t word, uint32_t tag) { return word >> 16 == tag; }
__device__ __forceinline__ uint32_t value(uint32_t word) { return word & 0xffffu; }

// What the conversion needs to know about a segment.
struct Segment {
    Divisor divisor;
    uint8_t* out;               // where position 0 of the share would go
    uint32_t begin, end;        // positions
    uint32_t head;
    int32_t at;                 // vector of the unit = position + at
};

// thread `tid`'s part of max |x| over `vecs` vectors
template <bool kHalf>
__device__ __forceinline__ uint32_t reduce(const uint4* x, int vecs, int tid) {
    typename In16<kHalf>::V2 m = In16<kHalf>::as2(0u);
#pragma unroll 4
    for (int i = tid; i < vecs; i += kWorkers) m = absmax8<kHalf>(m, x[i]);
    const uint32_t w = *reinterpret_cast<const uint32_t*>(&m);
    return max(w & 0xffffu, w >> 16);
}
// positions [i0, i1) of a segment; kFollows: the scale is another tensor's
template <bool kHalf, bool kFollows>
__device__ __forceinline__ void convert(const Segment& seg, const uint4* x, uint32_t i0, uint32_t i1, int tid) {
    constexpr uint32_t kStep = kWorkers;
    const Divisor dv = seg.divisor;
    uint2* o = reinterpret_cast<uint2*>(seg.out);
    if (dv.direct) {
        for (uint32_t i = i0 + tid; i < i1; i += kStep) o[i] = quant8_direct<kHalf>(x[i], dv);
        return;
    }
    uint32_t i = i0 + tid;
    for (; i + kStep < i1; i += 2 * kStep) {    // two vectors under way at a time
        const uint4 v0 = x[i], v1 = x[i + kStep];
        o[i] = quant8<kHalf, kFollows>(v0, dv);
        o[i + kStep] = quant8<kHalf, kFollows>(v1, dv);
    }
    if (i < i1) o[i] = quant8<kHalf, kFollows>(x[i], dv);
}

// every contiguous piece of half `part` of a share: to(first position, source, vectors)
template <class To>
__device__ __forceinline__ void half_share(const Args& a, const Share& s, int stage, uint32_t part, To to) {
    const uint32_t vecs = (uint32_t)a.vecs, tensors = (uint32_t)a.tensors;
    const uint32_t u0 = (uint32_t)(stage * a.stage_units) + s.unit;
    const uint32_t p0 = part == 0 ? 0 : s.half(), p1 = part == 0 ? s.half() : s.n;
    for (uint32_t g = 0; g < s.segs; ++g) {
        const uint32_t b = s.begin(g, vecs), i0 = max(p0, b), i1 = min(p1, s.end(g, vecs));
        if (i0 >= i1) continue;
        const uint32_t unit = u0 + g, head = unit / tensors;
        to(i0, a.x[unit - head * tensors] + (int64_t)head * vecs + s.at(g) + (i0 - b), i1 - i0);
    }
}

// A launch of its own before large calls: clears the words and has the first stage fetched to L2
// meanwhile (the launch then costs nothing).  One warp per block, the grid of staged_kernel.
__global__ void clear_and_fetch_kernel(const __grid_constant__ Args a) {
    const Share s((uint32_t)min(a.stage_units, a.units), (uint32_t)a.vecs);
    if (threadIdx.x == 0)
        for (uint32_t part = 0; part < kParts; ++part)
            half_share(a, s, 0, part, [](uint32_t, const uint4* src, uint32_t n) { bulk_prefetch(src, n * 16); });
    const uint32_t t = blockIdx.x * 32 + threadIdx.x, threads = gridDim.x * 32;
    for (uint32_t i = t; i < a.sets * a.slots_per_set; i += threads) a.slots[i] = 0u;
    if (a.follow_vecs > 0)
        for (uint32_t i = t; i < (uint32_t)(a.units / a.tensors); i += threads) a.heads[i] = 0u;
}

// kSelfTest: waits end after a.wait_clocks.  (A limit and checks that only an expired wait needs stay out of
// the exchange's path in all other calls: a variable limit and a look at `lost` before a share is published
// cost 0.4 us a stage, 89 -> 96 us for 16 heads of 20,011 + 3,001 x 128.)
template <bool kHalf, bool kSelfTest>
__global__ void __launch_bounds__(kThreads, 1) staged_kernel(const __grid_constant__ Args a) {
    const int64_t limit = kSelfTest ? a.wait_clocks : kWaitClocks;
    extern __shared__ __align__(128) uint8_t smem[];
    __shared__ uint64_t full[2], known[2], part_free[2][kParts];
    __shared__ uint32_t seg_acc[kMaxSegments];
    __shared__ Segment segment[2][kMaxSegments];
    __shared__ uint16_t holders[kMaxSegments][2];       // first and last block of every segment's unit
    __shared__ uint32_t follow_acc[kMaxFollowHeads];
    __shared__ volatile int lost, give_up;
    static_assert(kSmemBytes + sizeof(segment) + sizeof(seg_acc) + sizeof(follow_acc) + 768 <= 232448, "shared memory of a block");
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int stages = a.stages;
    const uint32_t vecs = (uint32_t)a.vecs, tensors = (uint32_t)a.tensors;
    if (tid == 0) {
        for (int i = 0; i < 2; ++i) {
            mbar_init(smem_u32(&full[i]), kParts);
            mbar_init(smem_u32(&known[i]), 1);
            for (int part = 0; part < kParts; ++part) mbar_init(smem_u32(&part_free[i][part]), kWorkers / 32);
        }
        fence_mbar_init();
        lost = give_up = 0;
    }
    if (tid < kMaxSegments) seg_acc[tid] = 0u;
    // rows that follow tensor 0 without counting are converted last, an equal share of them per block;
    // those of a small call are on their way to L2 from the start
    uint32_t f_lo = 0, f_hi = 0;
    if (a.follow_vecs > 0 && !a.follow_counts) {
        const uint32_t total = (uint32_t)(a.units / a.tensors) * a.follow_vecs;
        const uint32_t each = total / gridDim.x, more = total - each * gridDim.x;
        f_lo = each * blockIdx.x + min(blockIdx.x, more);
        f_hi = f_lo + each + (blockIdx.x < more ? 1u : 0u);
        if (f_lo + tid * 8 < f_hi) asm volatile("prefetch.global.L2 [%0];" ::"l"(a.follow_x + f_lo + tid * 8));
    }
    __syncthreads();
    int parts = 0;      // halves of stages that the load thread has requested
    const Share share_full((uint32_t)min(a.stage_units, a.units), vecs);
    const Share share_last((uint32_t)(a.units - (stages - 1) * a.stage_units), vecs);

    auto timed_out = [&] {
        if (atomicCAS(a.status, 0u, (uint32_t)FP8ATTN_ERR_TIMEOUT) == 0u)
            a.status[1] = (kDetailGridWait << 24) | (blockIdx.x & 0xFFFFFFu);
    };

    if (warp == kWorkers / 32) {
        // ============================== loads ==============================
        if (lane == 0) {
            bool on = true;
            auto pieces = [&](int stage, uint32_t part, auto to) {
                half_share(a, stage + 1 < stages ? share_full : share_last, stage, part, to);
            };
            auto wait = [&](uint32_t bar, uint32_t parity) {
                const int64_t t0 = clock64();
                bool done = mbar_test_wait(bar, parity);
                while (!done && !give_up && clock64() - t0 < limit) done = mbar_try_wait(bar, parity);
                return done;
            };
            auto load = [&](int stage, uint32_t part) {
                const uint32_t buf = stage & 1, bar = smem_u32(&full[buf]);
                const Share& s = stage + 1 < stages ? share_full : share_last;
                mbar_arrive_expect_tx(bar, (part == 0 ? s.half() : s.n - s.half()) * 16);
                ++parts;
                pieces(stage, part, [&](uint32_t i0, const uint4* src, uint32_t n) {
                    bulk_load(smem_u32(smem) + (buf * kBufVecs + i0) * 16, src, n * 16, bar);
                });
            };
            // What is requested waits in line before the exchange's words: a stage is requested when
            // the exchange of the stage two before it is over, and is in L2 by the next exchange.
            load(0, 0);
            load(0, 1);
            if (stages > 1) {
                on = wait(smem_u32(&full[0]), 0);
                if (on) load(1, 0);
                if (on) load(1, 1);
            }
            for (int stage = 2; stage < stages && on; ++stage) {
                const uint32_t buf = stage & 1, parity = ((stage >> 1) - 1) & 1;
                on = wait(smem_u32(&known[buf]), parity);
                for (uint32_t part = 0; part < kParts && on; ++part)
                    pieces(stage, part, [&](uint32_t, const uint4* src, uint32_t n) { bulk_prefetch(src, n * 16); });
                for (uint32_t part = 0; part < kParts && on; ++part) {
                    on = wait(smem_u32(&part_free[buf][part]), parity);
                    if (on) load(stage, part);
                }
            }
            if (!on) lost = 1;
        }
        __syncwarp();
    } else if (warp > kWorkers / 32) {
        // ============================== exchange ==============================
        // (recorded before this launch, so all blocks decide alike; asked for under the first loads)
        const bool pending = a.heed_status && *reinterpret_cast<volatile uint32_t*>(a.status) != 0u;
        for (int stage = 0; stage < stages; ++stage) {
            const Share& s = stage + 1 < stages ? share_full : share_last;
            const uint32_t u0 = (uint32_t)(stage * a.stage_units) + s.unit;
            uint32_t* const slots =
                a.slots + (stage + 1 == stages ? a.last_set : stage & 1) * a.slots_per_set;
            const uint32_t tag = (uint32_t)stage + 1;
            if (stage == 0 || (stage + 1 == stages && share_last.total != share_full.total)) {
                for (uint32_t g = lane; g < s.segs; g += 32) {
                    holders[g][0] = (uint16_t)s.holder((s.unit + g) * vecs);
                    holders[g][1] = (uint16_t)s.holder((s.unit + g + 1) * vecs - 1);
                }
            }
            sync_exchange();        // A: the share is reduced
            // (block b and unit u of the stage meet at most once, and b + u names the meeting)
            for (uint32_t g = lane; g < s.segs; g += 32) {
                publish(slots + blockIdx.x + s.unit + g, tag, seg_acc[g]);
                seg_acc[g] = 0u;
            }
            __syncwarp();
            // Collect the values of this share's units: `width` lanes per segment.
            const uint32_t width = s.segs <= 1 ? 32 : 16;
            const bool none_empty = s.total >= 8 * gridDim.x;
            bool there = !lost && !pending;
            const int64_t t0 = clock64();
            for (uint32_t g0 = 0; g0 < s.segs; g0 += 32 / width) {
                const uint32_t g = g0 + lane / width;
                uint32_t v = 0u;
                if (g < s.segs) {
                    constexpr int kBatch = 5;       // polls under way at a time: 148 blocks at 32 a row
                    const uint32_t u = s.unit + g, b1 = holders[g][1];
                    for (uint32_t b0 = holders[g][0] + lane % width; b0 <= b1; b0 += kBatch * width) {
                        uint32_t raw[kBatch];
                        for (bool all = false; there && !all;) {
#pragma unroll
                            for (int k = 0; k < kBatch; ++k) raw[k] = peek(slots + min(b0 + k * width, b1) + u);
                            all = true;
#pragma unroll
                            for (int k = 0; k < kBatch; ++k) {
                                const uint32_t b = min(b0 + k * width, b1);
                                all &= tagged(raw[k], tag) || (!none_empty && cut(s.total, b) == cut(s.total, b + 1));
                            }
                            if (!all) there = !lost && clock64() - t0 < limit;
                        }
#pragma unroll
                        for (int k = 0; k < kBatch; ++k)
                            if (b0 + k * width <= b1 && there && tagged(raw[k], tag)) v = max(v, value(raw[k]));
                    }
                }
                __syncwarp();
                for (uint32_t o = width >> 1; o > 0; o >>= 1) v = max(v, __shfl_xor_sync(0xffffffffu, v, o));
                if (g < s.segs && lane % width == 0) {
                    const uint32_t unit = u0 + g, head = unit / tensors, z = unit - head * tensors;
                    Segment& seg = segment[stage & 1][g];
                    seg.divisor = divisor(head_scale(In16<kHalf>::lo(v)));
                    seg.begin = s.begin(g, vecs);
                    seg.end = s.end(g, vecs);
                    seg.head = head;
                    seg.at = (int32_t)(s.at(g) - seg.begin);
                    seg.out = static_cast<uint8_t*>(a.out[z]) + ((int64_t)head * vecs + seg.at) * 8;
                    if (there && (g > 0 || s.skip == 0)) {      // the unit begins here
                        if (a.result_out[z] != nullptr) a.result_out[z][head] = seg.divisor.s;
                        if (z == 0 && a.follow_vecs > 0 && !a.follow_counts) publish(a.heads + head, 1, v);
                    }
                }
            }
            if (!__all_sync(0xffffffffu, there) && lane == 0) {
                if (!pending) timed_out();
                give_up = 1;
            }
            if (lane == 0) mbar_arrive(smem_u32(&known[stage & 1]));
            sync_exchange();        // B: results are known
            if (give_up) break;
        }
        // The heads that this block's following rows belong to (calls that cleared the words read them
        // when they convert).
        if (f_lo < f_hi && !a.cleared && !give_up) {
            const uint32_t h = f_lo / a.follow_vecs + lane;
            bool there = true;
            if (h <= (f_hi - 1) / a.follow_vecs) {
                const int64_t t0 = clock64();
                uint32_t raw = peek(a.heads + h);
                while (there && !tagged(raw, 1)) {
                    there = clock64() - t0 < limit;
                    raw = peek(a.heads + h);
                }
                follow_acc[lane] = value(raw);
            }
            if (!__all_sync(0xffffffffu, there) && lane == 0) {
                timed_out();
                give_up = 1;
            }
        }
        // The last warp to get here leaves everything at zero for the next call: its fence and those of the
        // others put all stores and polls of the words before that.
        __syncwarp();
        uint32_t done = 0;
        if (lane == 0) {
            __threadfence();
            done = atomicAdd(a.counter, 1u);
            __threadfence();
        }
        if (__shfl_sync(0xffffffffu, done, 0) == gridDim.x - 1) {
            for (uint32_t i = lane; i < a.sets * a.slots_per_set; i += 32) a.slots[i] = 0u;
            if (a.follow_vecs > 0 && !a.cleared)
                for (int i = lane; i < a.units / a.tensors; i += 32) a.heads[i] = 0u;
            if (lane == 0) *a.counter = 0u;
        }
    } else {
        // ============================== workers ==============================
        // Rows that follow tensor 0 and count: a block takes them in proportion to its segment of the
        // head (so that their values join the segment's).
        auto follow_range = [&](const Share& s, uint32_t g, uint32_t u0, uint32_t& head, uint32_t& f0, uint32_t& f1) {
            const uint32_t unit = u0 + s.unit + g, at = s.at(g);
            head = unit / tensors;
            if (unit - head * tensors != 0) return false;
            f0 = (uint32_t)((uint64_t)at * a.follow_vecs / vecs);
            f1 = (uint32_t)((uint64_t)(at + s.end(g, vecs) - s.begin(g, vecs)) * a.follow_vecs / vecs);
            return true;
        };
        auto convert_half = [&](int stage, uint32_t part) {
            const Share& s = stage + 1 < stages ? share_full : share_last;
            const uint4* buf = reinterpret_cast<const uint4*>(smem) + (stage & 1) * kBufVecs;
            const uint32_t p0 = part == 0 ? 0 : s.half(), p1 = part == 0 ? s.half() : s.n;
            for (uint32_t g = 0; g < s.segs; ++g) {
                const Segment& seg = segment[stage & 1][g];
                const uint32_t i0 = max(p0, seg.begin), i1 = min(p1, seg.end);
                if (i0 < i1) convert<kHalf, false>(seg, buf, i0, i1, tid);
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&part_free[stage & 1][part]));
        };
        for (int stage = 0; stage <= stages; ++stage) {
            if (stage < stages) {
                const Share& s = stage + 1 < stages ? share_full : share_last;
                const uint4* buf = reinterpret_cast<const uint4*>(smem) + (stage & 1) * kBufVecs;
                const uint32_t bar = smem_u32(&full[stage & 1]), parity = (stage >> 1) & 1;
                bool landed = mbar_test_wait(bar, parity);
                if (!landed) {
                    const int64_t t0 = clock64();
                    while (!landed && !lost && clock64() - t0 < limit) landed = mbar_try_wait(bar, parity);
                }
                if (!__all_sync(0xffffffffu, landed)) {     // what is published then bears no tag
                    lost = 1;
                    for (uint32_t g = lane; g < s.segs; g += 32) atomicMax(&seg_acc[g], kLost);
                }
                for (uint32_t g = 0; g < s.segs; ++g) {
                    const uint32_t b = s.begin(g, vecs), e = s.end(g, vecs);
                    if (b + (tid & ~31) >= e && !a.follow_counts) continue;      // (whole warps)
                    uint32_t v = 0u;
                    if (b + tid < e) v = reduce<kHalf>(buf + b, e - b, tid);
                    uint32_t head, f0, f1;
                    if (a.follow_counts && follow_range(s, g, (uint32_t)(stage * a.stage_units), head, f0, f1) && f0 + tid < f1)
                        v = max(v, reduce<kHalf>(a.follow_x + (int64_t)head * a.follow_vecs + f0, f1 - f0, tid));
                    v = __reduce_max_sync(0xffffffffu, v);
                    if (lane == 0) atomicMax(&seg_acc[g], v);
                }
                sync_exchange();    // A
            }
            if (stage > 0) {
                convert_half(stage - 1, 1);
                const Share& s = stage < stages ? share_full : share_last;
                for (uint32_t g = 0; a.follow_counts && g < s.segs; ++g) {
                    Segment seg = segment[(stage - 1) & 1][g];
                    uint32_t head, f0, f1;
                    if (!follow_range(s, g, (uint32_t)((stage - 1) * a.stage_units), head, f0, f1)) continue;
                    const int64_t first = (int64_t)head * a.follow_vecs;
                    seg.out = static_cast<uint8_t*>(a.follow_out) + first * 8;
                    convert<kHalf, true>(seg, a.follow_x + first, f0, f1, tid);
                }
            }
            if (stage < stages) {
                sync_exchange();    // B
                if (give_up) break;
                convert_half(stage, 0);
            }
        }
    }
    __syncthreads();
    // ---- a block that gives up leaves when its copies have landed ----
    if (give_up && tid == kWorkers) {
        if (parts & 1) mbar_arrive(smem_u32(&full[parts >> 1 & 1]));      // for the half that was never requested
        const int64_t t0 = clock64();
        for (int n = (parts + 1) / 2, stage = max(0, n - 2); stage < n; ++stage)
            while (!mbar_try_wait(smem_u32(&full[stage & 1]), (stage >> 1) & 1) && clock64() - t0 < kWaitClocks) {}
    }
    // ---- rows that follow tensor 0 ----
    if (!give_up) {
        bool there = true;
        const int64_t t0 = clock64();
        Segment seg;
        seg.at = 0;
        seg.out = static_cast<uint8_t*>(a.follow_out);
        for (uint32_t x = f_lo; x < f_hi && there;) {
            seg.head = x / a.follow_vecs;
            const uint32_t end = f_hi - seg.head * a.follow_vecs < a.follow_vecs ? f_hi : (seg.head + 1) * a.follow_vecs;
            uint32_t v = follow_acc[a.cleared ? 0 : seg.head - f_lo / a.follow_vecs];
            if (a.cleared) {
                uint32_t raw = peek(a.heads + seg.head);
                while (there && !tagged(raw, 1)) {
                    there = clock64() - t0 < limit;
                    raw = peek(a.heads + seg.head);
                }
                v = value(raw);
            }
            seg.divisor = divisor(head_scale(In16<kHalf>::lo(v)));
            if (there && tid < kWorkers) convert<kHalf, true>(seg, a.follow_x, x, end, tid);
            x = end;
        }
        if (!there) timed_out();
    }
}

// Two stages fill both buffers and wait for no room: they are loaded at once and exchanged together, so that the
// workers stand still once, under the second load, instead of twice (2 us each, 3 us where the words wait behind loads
// from HBM).  Graph-replayed, inputs not in L2 / in L2: 16 heads of 12,289 x 64 19.0 -> 18.0 / 12.9 -> 12.9 us, 8 heads of
// 16,384 x 128 22.7 -> 19.8 / 13.6 -> 13.7, 2 heads of 40,000 x 128 17.3 -> 16.2 / 12.5 -> 11.4, three tensors of 8 heads of
// 8,192 + 2,048 x 64 20.8 -> 19.4 / 15.2 -> 14.7, of 5,000 + 32,768 x 128 46.2 -> 44.7 / 42.6 -> 41.4.  Rows
// that count in the maximum stay with the general form.  (A kernel of its own: as a template parameter of the general
// one it moved that by up to 3 % through its schedule.)
template <bool kHalf, bool kSelfTest>
__global__ void __launch_bounds__(kThreads, 1) staged_pair_kernel(const __grid_constant__ Args a) {
    const int64_t limit = kSelfTest ? a.wait_clocks : kWaitClocks;
    extern __shared__ __align__(128) uint8_t smem[];
    __shared__ uint64_t full[2];
    __shared__ uint32_t seg_acc[2][kMaxSegments];
    __shared__ Segment segment[2][kMaxSegments];
    __shared__ uint16_t holders[2][kMaxSegments][2];    // first and last block of every segment's unit
    __shared__ uint32_t follow_acc[kMaxFollowHeads];
    __shared__ volatile int lost, give_up;
    static_assert(kSmemBytes + sizeof(segment) + sizeof(seg_acc) + sizeof(follow_acc) + 768 <= 232448, "shared memory of a block");
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    constexpr int stages = 2;
    const uint32_t vecs = (uint32_t)a.vecs, tensors = (uint32_t)a.tensors;
    if (tid == 0) {
        for (int i = 0; i < 2; ++i) mbar_init(smem_u32(&full[i]), kParts);
        fence_mbar_init();
        lost = give_up = 0;
    }
    if (tid < (int)(sizeof(seg_acc) / sizeof(uint32_t))) (&seg_acc[0][0])[tid] = 0u;
    // rows that follow tensor 0 without counting are converted last, an equal share of them per block;
    // those of a small call are on their way to L2 from the start
    uint32_t f_lo = 0, f_hi = 0;
    if (a.follow_vecs > 0) {
        const uint32_t total = (uint32_t)(a.units / a.tensors) * a.follow_vecs;
        const uint32_t each = total / gridDim.x, more = total - each * gridDim.x;
        f_lo = each * blockIdx.x + min(blockIdx.x, more);
        f_hi = f_lo + each + (blockIdx.x < more ? 1u : 0u);
        if (f_lo + tid * 8 < f_hi) asm volatile("prefetch.global.L2 [%0];" ::"l"(a.follow_x + f_lo + tid * 8));
    }
    __syncthreads();
    const Share share_full((uint32_t)min(a.stage_units, a.units), vecs);
    const Share share_last((uint32_t)(a.units - (stages - 1) * a.stage_units), vecs);

    auto timed_out = [&] {
        if (atomicCAS(a.status, 0u, (uint32_t)FP8ATTN_ERR_TIMEOUT) == 0u)
            a.status[1] = (kDetailGridWait << 24) | (blockIdx.x & 0xFFFFFFu);
    };

    if (warp == kWorkers / 32) {
        // ============================== loads ==============================
        if (lane == 0) {
            for (int stage = 0; stage < stages; ++stage) {
                const Share& s = stage == 0 ? share_full : share_last;
                const uint32_t bar = smem_u32(&full[stage]);
                for (uint32_t part = 0; part < kParts; ++part) {
                    mbar_arrive_expect_tx(bar, (part == 0 ? s.half() : s.n - s.half()) * 16);
                    half_share(a, s, stage, part, [&](uint32_t i0, const uint4* src, uint32_t n) {
                        bulk_load(smem_u32(smem) + (stage * kBufVecs + i0) * 16, src, n * 16, bar);
                    });
                }
            }
        }
        __syncwarp();
    } else if (warp > kWorkers / 32) {
        // ============================== exchange ==============================
        // (recorded before this launch, so all blocks decide alike; asked for under the first loads)
        const bool pending = a.heed_status && *reinterpret_cast<volatile uint32_t*>(a.status) != 0u;
        // One stage's exchange: what of it can be known before the share is reduced (the barrier comes between).
        struct Round {
            const Share& s;
            uint32_t u0, *slots, tag;
            uint16_t (*holders)[2];
            int stage;
        };
        auto round = [&](int stage) {
            const Share& s = stage + 1 < stages ? share_full : share_last;
            uint16_t (*const h)[2] = holders[stage];
            for (uint32_t g = lane; g < s.segs; g += 32) {
                h[g][0] = (uint16_t)s.holder((s.unit + g) * vecs);
                h[g][1] = (uint16_t)s.holder((s.unit + g + 1) * vecs - 1);
            }
            return Round{s, (uint32_t)(stage * a.stage_units) + s.unit,
                         a.slots + stage * a.slots_per_set, (uint32_t)stage + 1, h, stage};
        };
        auto put = [&](const Round& r) {
            const Share& s = r.s;
            // (block b and unit u of the stage meet at most once, and b + u names the meeting)
            for (uint32_t g = lane; g < s.segs; g += 32) {
                publish(r.slots + blockIdx.x + s.unit + g, r.tag, seg_acc[r.stage][g]);
                seg_acc[r.stage][g] = 0u;
            }
            __syncwarp();
        };
        // true: this lane's values are there
        auto collect = [&](const Round& r) {
            const Share& s = r.s;
            uint32_t* const slots = r.slots;
            const uint32_t tag = r.tag, u0 = r.u0;
            const int stage = r.stage;
            // Collect the values of this share's units: `width` lanes per segment.
            const uint32_t width = s.segs <= 1 ? 32 : 16;
            const bool none_empty = s.total >= 8 * gridDim.x;
            bool there = !lost && !pending;
            const int64_t t0 = clock64();
            for (uint32_t g0 = 0; g0 < s.segs; g0 += 32 / width) {
                const uint32_t g = g0 + lane / width;
                uint32_t v = 0u;
                if (g < s.segs) {
                    constexpr int kBatch = 5;       // polls under way at a time: 148 blocks at 32 a row
                    const uint32_t u = s.unit + g, b1 = r.holders[g][1];
                    for (uint32_t b0 = r.holders[g][0] + lane % width; b0 <= b1; b0 += kBatch * width) {
                        uint32_t raw[kBatch];
                        for (bool all = false; there && !all;) {
#pragma unroll
                            for (int k = 0; k < kBatch; ++k) raw[k] = peek(slots + min(b0 + k * width, b1) + u);
                            all = true;
#pragma unroll
                            for (int k = 0; k < kBatch; ++k) {
                                const uint32_t b = min(b0 + k * width, b1);
                                all &= tagged(raw[k], tag) || (!none_empty && cut(s.total, b) == cut(s.total, b + 1));
                            }
                            if (!all) there = !lost && clock64() - t0 < limit;
                        }
#pragma unroll
                        for (int k = 0; k < kBatch; ++k)
                            if (b0 + k * width <= b1 && there && tagged(raw[k], tag)) v = max(v, value(raw[k]));
                    }
                }
                __syncwarp();
                for (uint32_t o = width >> 1; o > 0; o >>= 1) v = max(v, __shfl_xor_sync(0xffffffffu, v, o));
                if (g < s.segs && lane % width == 0) {
                    const uint32_t unit = u0 + g, head = unit / tensors, z = unit - head * tensors;
                    Segment& seg = segment[stage & 1][g];
                    seg.divisor = divisor(head_scale(In16<kHalf>::lo(v)));
                    seg.begin = s.begin(g, vecs);
                    seg.end = s.end(g, vecs);
                    seg.head = head;
                    seg.at = (int32_t)(s.at(g) - seg.begin);
                    seg.out = static_cast<uint8_t*>(a.out[z]) + ((int64_t)head * vecs + seg.at) * 8;
                    if (there && (g > 0 || s.skip == 0)) {      // the unit begins here
                        if (a.result_out[z] != nullptr) a.result_out[z][head] = seg.divisor.s;
                        if (z == 0 && a.follow_vecs > 0) publish(a.heads + head, 1, v);
                    }
                }
            }
            return there;
        };
        const Round r0 = round(0), r1 = round(1);
        sync_exchange();        // A: both shares are reduced
        put(r0);
        put(r1);
        bool there = collect(r0);
        there = collect(r1) && there;
        if (!__all_sync(0xffffffffu, there) && lane == 0) {
            if (!pending) timed_out();
            give_up = 1;
        }
        sync_exchange();        // B: results are known
        // The heads that this block's following rows belong to (calls that cleared the words read them
        // when they convert).
        if (f_lo < f_hi && !a.cleared && !give_up) {
            const uint32_t h = f_lo / a.follow_vecs + lane;
            bool there = true;
            if (h <= (f_hi - 1) / a.follow_vecs) {
                const int64_t t0 = clock64();
                uint32_t raw = peek(a.heads + h);
                while (there && !tagged(raw, 1)) {
                    there = clock64() - t0 < limit;
                    raw = peek(a.heads + h);
                }
                follow_acc[lane] = value(raw);
            }
            if (!__all_sync(0xffffffffu, there) && lane == 0) {
                timed_out();
                give_up = 1;
            }
        }
        // The last warp to get here leaves everything at zero for the next call: its fence and those of the
        // others put all stores and polls of the words before that.
        __syncwarp();
        uint32_t done = 0;
        if (lane == 0) {
            __threadfence();
            done = atomicAdd(a.counter, 1u);
            __threadfence();
        }
        if (__shfl_sync(0xffffffffu, done, 0) == gridDim.x - 1) {
            for (uint32_t i = lane; i < a.sets * a.slots_per_set; i += 32) a.slots[i] = 0u;
            if (a.follow_vecs > 0 && !a.cleared)
                for (int i = lane; i < a.units / a.tensors; i += 32) a.heads[i] = 0u;
            if (lane == 0) *a.counter = 0u;
        }
    } else {
        // ============================== workers ==============================
        auto convert_half = [&](int stage, uint32_t part) {
            const Share& s = stage + 1 < stages ? share_full : share_last;
            const uint4* buf = reinterpret_cast<const uint4*>(smem) + (stage & 1) * kBufVecs;
            const uint32_t p0 = part == 0 ? 0 : s.half(), p1 = part == 0 ? s.half() : s.n;
            for (uint32_t g = 0; g < s.segs; ++g) {
                const Segment& seg = segment[stage & 1][g];
                const uint32_t i0 = max(p0, seg.begin), i1 = min(p1, seg.end);
                if (i0 < i1) convert<kHalf, false>(seg, buf, i0, i1, tid);
            }
        };
        // the share's values, once it has landed
        auto reduce_share = [&](int stage) {
            const Share& s = stage + 1 < stages ? share_full : share_last;
            const uint4* buf = reinterpret_cast<const uint4*>(smem) + (stage & 1) * kBufVecs;
            const uint32_t bar = smem_u32(&full[stage]), parity = 0;
            bool landed = mbar_test_wait(bar, parity);
            if (!landed) {
                const int64_t t0 = clock64();
                while (!landed && !lost && clock64() - t0 < limit) landed = mbar_try_wait(bar, parity);
            }
            if (!__all_sync(0xffffffffu, landed)) {     // what is published then bears no tag
                lost = 1;
                for (uint32_t g = lane; g < s.segs; g += 32) atomicMax(&seg_acc[stage][g], kLost);
            }
            for (uint32_t g = 0; g < s.segs; ++g) {
                const uint32_t b = s.begin(g, vecs), e = s.end(g, vecs);
                if (b + (tid & ~31) >= e) continue;      // (whole warps)
                uint32_t v = 0u;
                if (b + tid < e) v = reduce<kHalf>(buf + b, e - b, tid);
                v = __reduce_max_sync(0xffffffffu, v);
                if (lane == 0) atomicMax(&seg_acc[stage][g], v);
            }
        };
#pragma unroll 1
        for (int stage = 0; stage < stages; ++stage) reduce_share(stage);
        sync_exchange();    // A
        sync_exchange();    // B
#pragma unroll 1
        for (uint32_t half = 0; half < 2 * kParts && !give_up; ++half) convert_half(half / kParts, half % kParts);
    }
    __syncthreads();
    // ---- a block that gives up leaves when its copies have landed ----
    if (give_up && tid == kWorkers) {
        const int64_t t0 = clock64();
        for (int stage = 0; stage < stages; ++stage)
            while (!mbar_try_wait(smem_u32(&full[stage]), 0) && clock64() - t0 < kWaitClocks) {}
    }
    // ---- rows that follow tensor 0 ----
    if (!give_up) {
        bool there = true;
        const int64_t t0 = clock64();
        Segment seg;
        seg.at = 0;
        seg.out = static_cast<uint8_t*>(a.follow_out);
        for (uint32_t x = f_lo; x < f_hi && there;) {
            seg.head = x / a.follow_vecs;
            const uint32_t end = f_hi - seg.head * a.follow_vecs < a.follow_vecs ? f_hi : (seg.head + 1) * a.follow_vecs;
            uint32_t v = follow_acc[a.cleared ? 0 : seg.head - f_lo / a.follow_vecs];
            if (a.cleared) {
                uint32_t raw = peek(a.heads + seg.head);
                while (there && !tagged(raw, 1)) {
                    there = clock64() - t0 < limit;
                    raw = peek(a.heads + seg.head);
                }
                v = value(raw);
            }
            seg.divisor = divisor(head_scale(In16<kHalf>::lo(v)));
            if (there && tid < kWorkers) convert<kHalf, true>(seg, a.follow_x, x, end, tid);
            x = end;
        }
        if (!there) timed_out();
    }
}

// Fills what plan() does not get (stage_units and everything behind it) and returns the grid, or 0 where
// this path does not take the call: a unit that does not fit one buffer of every SM or is no longer than a
// share, or more words than the workspace has for them.
inline unsigned plan(Shape& a, int sms) {
    if (a.units <= 0 || a.vecs <= kMinVecs || a.vecs % 8 != 0) return 0;     // (shares end on multiples of eight vectors)
    if ((uint64_t)a.follow_vecs * (uint64_t)(a.units / a.tensors) > 0x7fffffffull) return 0;
    // at least 8 KB per block, test rows included: with fewer blocks there is less to exchange, but all of
    // them share the test rows (1 head of 1,100 + 200,000 x 64 with the blocks that its train rows are worth:
    // 19.4 us, with all of them 14.7)
    const int64_t all = a.vecs * a.units + (int64_t)a.follow_vecs * (a.units / a.tensors);
    const int64_t grid = all / 512 < 1 ? 1 : all / 512 > sms ? sms : all / 512;
    const int64_t room = grid * kBufVecs;
    if (a.vecs > room) return 0;
    // (stages as large as fit: half as large, calls of many short heads take a third longer, because
    // a stage costs 3.5 us however short)
    const int64_t fit = room / a.vecs;
    int64_t stages = (a.units + fit - 1) / fit;
    a.stage_units = (int)((a.units + stages - 1) / stages);
    stages = (a.units + a.stage_units - 1) / a.stage_units;
    if (stages > 0xfff0) return 0;
    a.stages = (int)stages;
    const bool shorter = stages > 2 && stages * a.stage_units != a.units;
    a.sets = shorter ? 3 : stages > 1 ? 2 : 1;
    a.last_set = shorter ? 2 : (int)(stages - 1) & 1;
    const int64_t per_set = grid + a.stage_units;
    // the words of the heads sit behind the slots, or where the call clears them first
    const int64_t head_words = !a.cleared && a.follow_vecs > 0 ? a.units / a.tensors : 0;
    if (a.sets * per_set + head_words > kOnePassWords || (head_words > 0 && head_words / grid + 2 > kMaxFollowHeads)) return 0;
    a.slots_per_set = (uint32_t)per_set;
    return (unsigned)grid;
}

// The device does not hold all blocks of a cooperative launch at once, as in a context that was given only
// some of the SMs: nothing was launched that waits, the caller takes two passes.
constexpr int kRefused = -1;

template <bool kHalf, bool kSelfTest>
int launch(const Args& a, unsigned grid, cudaStream_t stream) {
    // Two stages whose test rows do not count: the pair kernel, 2 .. 13 % faster where the inputs are not in L2, between
    // the same and 10 % where they are (see there).
    // (the opt-in to large dynamic shared memory is per device and context: set on every call)
    auto kernel = a.stages == 2 && !a.follow_counts ? staged_pair_kernel<kHalf, kSelfTest> : staged_kernel<kHalf, kSelfTest>;
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemBytes) !=
        cudaSuccess)
        return FP8ATTN_ERR_CUDA;
    cudaLaunchAttribute attr = {};
    attr.id = cudaLaunchAttributeCooperative;
    attr.val.cooperative = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = kSmemBytes;
    cfg.stream = stream;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    if (a.cleared) {
        clear_and_fetch_kernel<<<grid, 32, 0, stream>>>(a);
        if (cudaGetLastError() != cudaSuccess) return FP8ATTN_ERR_CUDA;
        count_launch();
    }
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, a);
    if (e == cudaErrorCooperativeLaunchTooLarge || e == cudaErrorNotSupported) {
        cudaGetLastError();     // (reported here and nowhere else)
        return kRefused;
    }
    if (e != cudaSuccess) return FP8ATTN_ERR_CUDA;
    count_launch();
    return FP8ATTN_OK;
}

}  // namespace staged
}  // namespace fp8attn
