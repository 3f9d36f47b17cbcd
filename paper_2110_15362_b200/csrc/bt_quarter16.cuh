// The walk over a stash of 2-byte values, shared by the restore (bt_decompress.cu) and the ReLU6 backward
// (bt_relu6_bwd.cu).
//
// The generic kernels gather every stashed value with one global load and a 64-bit address computation per
// element, which makes a 2-byte element cost as many instructions as a 4-byte one.  Here a warp takes half a chunk
// (2048 elements) and first brings its packed run into shared memory with one bulk copy -- the run starts wherever its
// rank puts it: the 16-byte vectors that cover it are copied whole, the last one element by element so that
// nothing behind the caller's values is read -- and the gather reads shared memory: a test of the element's bit,
// a 2-byte shared load, a select, a predicated 32-bit add.
//
// These kernels are bound by instruction issue.  A quarter chunk per warp spent half of its 500 instructions before the
// first element (bitmap words, ranks, staging); with half a chunk, and the words and their places in the run read from a
// small table in shared memory instead of two shuffles per step, the restore of [64,128,112,112] bf16 takes 51 us
// instead of 57.  A whole chunk per warp would want 9 KB of shared memory a warp: 24 of them per SM, not 48.
#pragma once

#include "bt_internal.cuh"

namespace bt {
namespace q16 {

constexpr uint32_t kFull = 0xFFFFFFFFu;

__device__ __forceinline__ uint4 ldg_vec_stream(const uint4 *p)
{
    uint4 v;
    asm volatile("ld.global.L1::no_allocate.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
    return v;
}

// Four consecutive elements under the four low bits of `bits`: for every set bit the next 2-byte value at shared
// address `a` (which moves on), kFill for a clear bit; packed two to a word.
template <uint32_t kFill = 0>
__device__ __forceinline__ uint2 expand4_u16(uint32_t a, const uint32_t bits)
{
    uint2 r;
#define BT_PAIR(OUT, B0, B1, LAST) \
    "and.b32 t, %3, " #B0 ";\n\tsetp.ne.u32 p, t, 0;\n\tld.shared.u16 lo, [%2];\n\tselp.b32 lo, lo, %4, p;\n\t@p add.u32 %2, %2, 2;\n\t" \
    "and.b32 t, %3, " #B1 ";\n\tsetp.ne.u32 p, t, 0;\n\tld.shared.u16 hi, [%2];\n\tselp.b32 hi, hi, %4, p;\n\t" LAST \
    "prmt.b32 " OUT ", lo, hi, 0x5410;\n\t"
    asm volatile("{\n\t.reg .pred p;\n\t.reg .b32 t, lo, hi;\n\t" BT_PAIR("%0", 1, 2, "@p add.u32 %2, %2, 2;\n\t") BT_PAIR("%1", 4, 8, "") "}" : "=r"(r.x), "=r"(r.y), "+r"(a) : "r"(bits), "n"(kFill));
#undef BT_PAIR
    return r;
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

// What a warp knows about its half chunk once the run is staged.
struct Part {
    uint32_t words;     // shared address of its 64 (bitmap word, shared address of the word's first value) pairs
    uint64_t e0;        // index of its first element
    bool     whole;     // all 2048 elements exist
};
constexpr int kPartElems = 2048;
constexpr int kPartSteps = kPartElems / 128;
// CTAs of `warps` warps for a tensor
inline uint64_t blocks_of(const uint64_t n, const int warps)
{
    const uint64_t per = static_cast<uint64_t>(warps) * kPartElems;
    return (n + per - 1) / per;
}

// Reads the chunk's bitmap words and prefix entry, ranks the half chunk's words and stages its packed run.  False if
// this warp has no part.  `block`: index of the CTA among those that work on the tensor.
template <int kWarps>
__device__ __forceinline__ bool stage_part(const uint32_t *__restrict__ bitmap, const uint16_t *values,
                                           const uint64_t *__restrict__ values_offset, const uint64_t *__restrict__ prefix,
                                           const uint64_t n, const uint64_t block, Part &pt)
{
    // a part's run (at most 2048 values) behind up to 14 bytes of its first vector, whole vectors
    __shared__ __align__(16) unsigned char s_run[kWarps][2 * kPartElems + 32];
    __shared__ __align__(16) uint2         s_words[kWarps][kPartElems / 32];
    __shared__ __align__(8) uint64_t       s_landed[kWarps];   // the warp's bulk copy has landed

    const uint32_t lane        = threadIdx.x & 31u;
    const uint32_t wic         = threadIdx.x >> 5;
    const uint64_t warp_global = block * kWarps + wic;
    if (warp_global >= (n + kPartElems - 1) / kPartElems) return false;
    if (lane == 0) {
        mbar_init(&s_landed[wic], 1);
        fence_proxy_async();
    }
    __syncwarp();

    const uint64_t chunk = warp_global >> 1;
    const bool     late  = warp_global & 1u;               // the second half of the chunk

    // the chunk's 128 words, four per lane (zero past the end of the bitmap), and its prefix entry: independent loads
    const uint4    w4         = load_words4(bitmap, chunk * 128 + 4 * lane, (n + 31) >> 5);
    const uint64_t chunk_base = prefix[chunk];
    if (values_offset) values = reinterpret_cast<const uint16_t *>(reinterpret_cast<const unsigned char *>(values) + *values_offset);

    const uint32_t c1 = __popc(w4.x), c2 = c1 + __popc(w4.y), c3 = c2 + __popc(w4.z), c4 = c3 + __popc(w4.w);
    uint32_t       incl = c4;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t u = __shfl_up_sync(kFull, incl, o);
        if (lane >= static_cast<uint32_t>(o)) incl += u;
    }
    const uint32_t half = __shfl_sync(kFull, incl, 15), all = __shfl_sync(kFull, incl, 31);
    const uint32_t before = late ? half : 0u;              // non-zeros of the chunk in front of this part
    const uint32_t cnt    = late ? all - half : half;      // values of this part

    // ---- the run into shared memory: one bulk copy per warp.  The copy engine writes shared memory by itself;
    // brought in through registers (16-byte loads, then 16-byte shared stores) the same bytes pass the L1 data pipe
    // twice.  The copy covers the whole 16-byte vectors of the run; the elements of the last, partial
    // vector are fetched one by one so that nothing behind the caller's values is read.
    const uint16_t *const src   = values + (chunk_base + before);
    const uint32_t        shift = static_cast<uint32_t>(reinterpret_cast<uintptr_t>(src) & 15u);         // bytes
    const uint32_t        bytes = shift + 2u * cnt;                                                      // of the staging area in use
    const uint32_t        full  = cnt ? bytes >> 4 : 0u;                                                 // whole vectors
    const unsigned char  *const gv = reinterpret_cast<const unsigned char *>(src) - shift;
    if (full && lane == 0) {
        mbar_arrive_expect_tx(&s_landed[wic], 16u * full);
        bulk_load(&s_run[wic][0], gv, 16u * full, &s_landed[wic]);
    }
    // the part's words and where their values start, for the steps
    if ((lane >> 4) == (late ? 1u : 0u)) {
        const uint32_t a  = smem_addr(&s_run[wic][0]) + shift + 2u * (incl - c4 - before);
        const uint32_t to = smem_addr(&s_words[wic][4 * (lane & 15u)]);
        asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(to), "r"(w4.x), "r"(a), "r"(w4.y), "r"(a + 2u * c1) : "memory");
        asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(to + 16u), "r"(w4.z), "r"(a + 2u * c2), "r"(w4.w), "r"(a + 2u * c3) : "memory");
    }
    const uint32_t tail0 = full * 16u > shift ? full * 16u : shift;
    for (uint32_t b = tail0 + 2u * lane; b < bytes; b += 64u) s_run[wic][b] = gv[b], s_run[wic][b + 1] = gv[b + 1];
    // Not seen so far: the copy engine has not delivered within two seconds.  The calls built on this have no
    // status word; the warp gives the copy a last, short time (so that the CTA does not retire with a copy into
    // its shared memory in flight) and leaves its part of the output unwritten.
    if (full && !landed(&s_landed[wic], kLandLimitNs)) {
        landed(&s_landed[wic], kLandLastNs);
        return false;
    }
    __syncwarp();
    pt.words = smem_addr(&s_words[wic][0]);
    pt.e0    = warp_global * kPartElems;
    pt.whole = pt.e0 + kPartElems <= n;
    return true;
}

// Step k (0 .. kPartSteps - 1) of the expansion: the lane's four consecutive elements e0 + 128k + 4 lane .. + 3, packed
// two to a word, kFill (+0 unless the caller asks otherwise) where the bit is clear.  (With 8 elements per lane the 32
// lanes of one shared load reach over 256 bytes of the run and every load takes two passes: 0.131 ms instead of
// 0.126 on 205 M elements; with 2 per lane the table reads and stores double: 0.153 ms.)
template <uint32_t kFill = 0>
__device__ __forceinline__ uint2 expand_step(const Part &pt, const int k, const uint32_t lane)
{
    uint32_t w, at;
    asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(w), "=r"(at) : "r"(pt.words + 32u * static_cast<uint32_t>(k) + 8u * (lane >> 3)));
    const uint32_t sh = (lane & 7u) * 4u;
    return expand4_u16<kFill>(at + 2u * __popc(w & ((1u << sh) - 1u)), w >> sh);
}

}  // namespace q16
}  // namespace bt
