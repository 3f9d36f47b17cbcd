// The walk over a stash, shared by the restore (bt_decompress.cu) and the ReLU6 backward (bt_relu6_bwd.cu).
//
// A warp takes a part of a chunk (4096 bytes of dense elements: half a chunk of 2-byte, a quarter of 4-byte elements) and
// first brings its packed run into shared memory with one bulk copy -- the run starts wherever its rank puts it: the
// 16-byte vectors that cover it are copied whole, the last one element by element so that nothing behind the caller's
// values is read -- and the gather reads shared memory: a test of the element's bit, a shared load, a select, a
// predicated 32-bit add.  Words and their places in the run come from a small table in shared memory.
//
// What this is for.  2-byte elements: the kernels are bound by instruction issue; a gather straight from global memory
// costs a load and a 64-bit address per element, and with a quarter chunk per warp half of the 500 instructions per 1024
// elements came before the first element (restore of [64,128,112,112] bf16: 59 us with a quarter chunk per warp, 51 this
// way).  4-byte elements: the gathered values of a quarter occupy 32 registers a lane until they arrive, which keeps 35
// warps on an SM with two dependent round trips each (fp32 2^28 at half zeros: 266 us gathered from global memory, 243
// this way; 2^27 at 90 % zeros 108 and 94; 200704 elements 4.2 and 2.3).  4096 bytes a warp keep 48 warps on an SM (44 with
// 2-byte elements, whose table is larger).
#pragma once

#include "bt_internal.cuh"

namespace bt {
namespace walk {

constexpr uint32_t kFull = 0xFFFFFFFFu;

// A lane's consecutive elements under the low bits of `bits` (four; two of 8 bytes): for every set bit the next value at
// shared address `a`, kFill for a clear bit (8-byte elements: in the upper half, 0 in the lower), as they are stored
// (8 bytes of 2-byte elements, else 16).
template <typename U, uint32_t kFill = 0>
__device__ __forceinline__ auto expand(uint32_t a, const uint32_t bits)
{
    if constexpr (sizeof(U) == 2) {
        uint2 r;
#define BT_PAIR(OUT, B0, B1, LAST)                                                                                   \
    "and.b32 t, %3, " #B0 ";\n\tsetp.ne.u32 p, t, 0;\n\tld.shared.u16 lo, [%2];\n\tselp.b32 lo, lo, %4, p;\n\t@p add.u32 %2, %2, 2;\n\t" \
    "and.b32 t, %3, " #B1 ";\n\tsetp.ne.u32 p, t, 0;\n\tld.shared.u16 hi, [%2];\n\tselp.b32 hi, hi, %4, p;\n\t" LAST      \
    "prmt.b32 " OUT ", lo, hi, 0x5410;\n\t"
        asm volatile("{\n\t.reg .pred p;\n\t.reg .b32 t, lo, hi;\n\t" BT_PAIR("%0", 1, 2, "@p add.u32 %2, %2, 2;\n\t") BT_PAIR("%1", 4, 8, "") "}"
                     : "=&r"(r.x), "=&r"(r.y), "+r"(a) : "r"(bits), "n"(kFill));
#undef BT_PAIR
        return r;
    } else if constexpr (sizeof(U) == 4) {
        uint4 r;
#define BT_ONE(OUT, BIT, LAST) "and.b32 t, %5, " #BIT ";\n\tsetp.ne.u32 p, t, 0;\n\tld.shared.u32 " OUT ", [%4];\n\tselp.b32 " OUT ", " OUT ", %6, p;\n\t" LAST
#define BT_STEP "@p add.u32 %4, %4, 4;\n\t"
        asm volatile("{\n\t.reg .pred p;\n\t.reg .b32 t;\n\t" BT_ONE("%0", 1, BT_STEP) BT_ONE("%1", 2, BT_STEP) BT_ONE("%2", 4, BT_STEP) BT_ONE("%3", 8, "") "}"
                     : "=&r"(r.x), "=&r"(r.y), "=&r"(r.z), "=&r"(r.w), "+r"(a) : "r"(bits), "n"(kFill));
#undef BT_STEP
#undef BT_ONE
        return r;
    } else {
        uint4 r;
        asm volatile("{\n\t.reg .pred p;\n\t.reg .b32 t;\n\t"
                     "and.b32 t, %5, 1;\n\tsetp.ne.u32 p, t, 0;\n\tld.shared.v2.u32 {%0, %1}, [%4];\n\tselp.b32 %0, %0, 0, p;\n\tselp.b32 %1, %1, %6, p;\n\t@p add.u32 %4, %4, 8;\n\t"
                     "and.b32 t, %5, 2;\n\tsetp.ne.u32 p, t, 0;\n\tld.shared.v2.u32 {%2, %3}, [%4];\n\tselp.b32 %2, %2, 0, p;\n\tselp.b32 %3, %3, %6, p;\n\t}"
                     : "=&r"(r.x), "=&r"(r.y), "=&r"(r.z), "=&r"(r.w), "+r"(a) : "r"(bits), "n"(kFill));
        return r;
    }
}

// Bounded wait for a warp's own bulk copy (phase 0 of its mbarrier): false if it has not landed within the limit.
constexpr uint64_t kLandLimitNs = 2000000000ull, kLandLastNs = 20000000ull;
__device__ __forceinline__ bool landed(uint64_t *bar, const uint64_t limit_ns)
{
    uint64_t t0 = 0;
    for (uint32_t probes = 1; !mbar_try_wait(bar, 0); ++probes) {
        if ((probes & 63u) == 0) {
            uint64_t now;
            asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(now));
            if (t0 == 0) t0 = now;
            if (now - t0 > limit_ns) return false;
        }
    }
    return true;
}

// What a warp knows about its part once the run is staged.
struct Part {
    uint32_t words;     // shared address of its (bitmap word, shared address of the word's first value) pairs
    uint64_t e0;        // index of its first element
    bool     whole;     // all its elements exist
};
template <typename U>
struct Of {
    static constexpr int      kElems   = 4096 / sizeof(U);             // elements of a part
    static constexpr int      kWords   = kElems / 32;
    static constexpr int      kPerLane = sizeof(U) == 8 ? 2 : 4;       // consecutive elements of a lane in a step
    static constexpr int      kSteps   = kElems / (32 * kPerLane);
    static constexpr int      kParts   = BT_CHUNK_ELEMS / kElems;      // of a chunk
    static constexpr uint32_t kLanes   = kWords / 4;                   // lanes that hold a part's words, four each
    // CTAs of `warps` warps for a tensor
    static uint64_t blocks_of(const uint64_t n, const int warps)
    {
        const uint64_t per = static_cast<uint64_t>(warps) * kElems;
        return (n + per - 1) / per;
    }
};

// Reads the chunk's bitmap words and prefix entry, ranks the part's words and stages its packed run.  False if
// this warp has no part.  `block`: index of the CTA among those that work on the tensor.
template <typename U, int kWarps>
__device__ __forceinline__ bool stage_part(const uint32_t *__restrict__ bitmap, const U *values,
                                           const uint64_t *__restrict__ values_offset, const uint64_t *__restrict__ prefix,
                                           const uint64_t n, const uint64_t block, Part &pt)
{
    using P = Of<U>;
    constexpr uint32_t kES = sizeof(U);
    // a part's run (at most 4096 bytes) behind less than 16 bytes of its first vector, whole vectors
    __shared__ __align__(16) unsigned char s_run[kWarps][4096 + 32];
    __shared__ __align__(16) uint2         s_words[kWarps][P::kWords];
    __shared__ __align__(8) uint64_t       s_landed[kWarps];   // the warp's bulk copy has landed

    const uint32_t lane        = threadIdx.x & 31u;
    const uint32_t wic         = threadIdx.x >> 5;
    const uint64_t warp_global = block * kWarps + wic;
    if (warp_global >= (n + P::kElems - 1) / P::kElems) return false;
    if (lane == 0) {
        mbar_init(&s_landed[wic], 1);
        fence_proxy_async();
    }
    __syncwarp();

    const uint64_t chunk = warp_global / P::kParts;
    const uint32_t part  = static_cast<uint32_t>(warp_global % P::kParts);

    // the chunk's 128 words, four per lane (zero past the end of the bitmap), and its prefix entry: independent loads
    const uint4    w4         = load_words4(bitmap, chunk * 128 + 4 * lane, (n + 31) >> 5);
    const uint64_t chunk_base = prefix[chunk];
    if (values_offset) values = reinterpret_cast<const U *>(reinterpret_cast<const unsigned char *>(values) + *values_offset);

    const uint32_t c1 = __popc(w4.x), c2 = c1 + __popc(w4.y), c3 = c2 + __popc(w4.z), c4 = c3 + __popc(w4.w);
    uint32_t       incl = c4;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t u = __shfl_up_sync(kFull, incl, o);
        if (lane >= static_cast<uint32_t>(o)) incl += u;
    }
    const uint32_t last   = __shfl_sync(kFull, incl, (part + 1) * P::kLanes - 1);
    const uint32_t front  = __shfl_sync(kFull, incl, part * P::kLanes - 1);        // part 0: some lane's, not used
    const uint32_t before = part ? front : 0u;             // non-zeros of the chunk in front of this part
    const uint32_t cnt    = last - before;                 // values of this part

    // ---- the run into shared memory: one bulk copy per warp.  The copy engine writes shared memory by itself;
    // brought in through registers (16-byte loads, then 16-byte shared stores) the same bytes pass the L1 data pipe
    // twice.  The copy covers the whole 16-byte vectors of the run; the elements of the last, partial
    // vector are fetched one by one so that nothing behind the caller's values is read.
    const U *const src   = values + (chunk_base + before);
    const uint32_t shift = static_cast<uint32_t>(reinterpret_cast<uintptr_t>(src) & 15u);                // bytes
    const uint32_t bytes = shift + kES * cnt;                                                            // of the staging area in use
    const uint32_t full  = cnt ? bytes >> 4 : 0u;                                                        // whole vectors
    const unsigned char *const gv = reinterpret_cast<const unsigned char *>(src) - shift;
    if (full && lane == 0) {
        mbar_arrive_expect_tx(&s_landed[wic], 16u * full);
        bulk_load(&s_run[wic][0], gv, 16u * full, &s_landed[wic]);
    }
    // the part's words and where their values start, for the steps
    if (lane / P::kLanes == part) {
        const uint32_t a  = smem_addr(&s_run[wic][0]) + shift + kES * (incl - c4 - before);
        const uint32_t to = smem_addr(&s_words[wic][4 * (lane % P::kLanes)]);
        asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(to), "r"(w4.x), "r"(a), "r"(w4.y), "r"(a + kES * c1) : "memory");
        asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(to + 16u), "r"(w4.z), "r"(a + kES * c2), "r"(w4.w), "r"(a + kES * c3) : "memory");
    }
    const uint32_t tail0 = full * 16u > shift ? full * 16u : shift;
    for (uint32_t b = tail0 + kES * lane; b < bytes; b += 32u * kES) *reinterpret_cast<U *>(&s_run[wic][b]) = *reinterpret_cast<const U *>(gv + b);
    // Not seen so far: the copy engine has not delivered within two seconds.  The calls built on this have no
    // status word; the warp gives the copy a last, short time (so that the CTA does not retire with a copy into
    // its shared memory in flight) and leaves its part of the output unwritten.
    if (full && !landed(&s_landed[wic], kLandLimitNs)) {
        landed(&s_landed[wic], kLandLastNs);
        return false;
    }
    __syncwarp();
    pt.words = smem_addr(&s_words[wic][0]);
    pt.e0    = warp_global * P::kElems;
    pt.whole = pt.e0 + P::kElems <= n;
    return true;
}

// Step k (0 .. kSteps - 1) of the expansion: the lane's kPerLane consecutive elements from e0 + 32 kPerLane k + kPerLane
// lane on.  (2-byte elements: with 8 elements per lane the 32 lanes of one shared load reach over 256 bytes of the run and
// every load takes two passes: 0.131 ms instead of 0.126 on 205 M elements; with 2 per lane the table reads and stores
// double: 0.153 ms.)
template <typename U, uint32_t kFill = 0>
__device__ __forceinline__ auto expand_step(const Part &pt, const int k, const uint32_t lane)
{
    constexpr uint32_t kPer = Of<U>::kPerLane, kShare = 32 / kPer;     // lanes that share a word
    uint32_t           w, at;
    asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(w), "=r"(at) : "r"(pt.words + 8u * kPer * static_cast<uint32_t>(k) + 8u * (lane / kShare)));
    const uint32_t sh = (lane % kShare) * kPer;
    return expand<U, kFill>(at + static_cast<uint32_t>(sizeof(U)) * __popc(w & ((1u << sh) - 1u)), w >> sh);
}

}  // namespace walk
}  // namespace bt
