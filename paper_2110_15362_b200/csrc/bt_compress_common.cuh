// What the single-tensor and the batched compress kernels share: constants of the workspace protocol, small PTX
// wrappers, the bounded mbarrier wait, the steps of a worker warp on a segment (into registers, flags, ranks, bitmap
// words, survivors packed into the worker's own ring in shared memory, copy-out from there), the worker and the store
// warp built of them, and the host-side launch shape.
#pragma once

#include <mutex>
#include <type_traits>

#include "bt_internal.cuh"

namespace bt {

// A value no other call of this process gets (bt_compress.cu).
uint64_t next_call_tag();
// The calling thread's limit on the CTAs of one compress launch, 0: none (bt_compress.cu).
uint32_t compress_max_ctas();
// The bound of the kernels' waits in nanoseconds; only a test build can change it (bt_compress.cu).
uint64_t compress_wait_ns();

namespace cmp {

constexpr uint32_t kFull       = 0xFFFFFFFFu;
constexpr int      kMaxWindows = 5;                   // 32 * kMaxWindows descriptors are read at a time (six: bf16 2^27 82.4 us, five: 80.1)
constexpr uint32_t kMaxGrid    = 32 * kMaxWindows;    // CTAs that tiles are dealt to
constexpr int      kHdrSeq     = 0;                   // header words (64-bit): launch sequence number,
constexpr int      kHdrAbort   = 1;                   //   abort word (== the launch's tag once a wait ran out),
constexpr int      kHdrCursor  = 2;                   //   batched arena form: the cursor as the launch found it, and
constexpr int      kHdrPushed  = 3;                   //   its tag once its last tile is finished

__device__ __forceinline__ uint64_t now_ns()
{
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ uint64_t warp_sum_u64(uint64_t v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
    return v;
}

__device__ __forceinline__ void mbar_arrive(uint64_t *bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr(bar)) : "memory");
}

__device__ __forceinline__ void red_add_u64(uint64_t *p, uint64_t v)
{
    asm volatile("red.relaxed.gpu.global.add.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

// A bijective mixer of 64-bit words (the finaliser of splitmix64).
__host__ __device__ __forceinline__ uint64_t mix64(uint64_t x)
{
    x ^= x >> 30;
    x *= 0xBF58476D1CE4E5B9ull;
    x ^= x >> 27;
    x *= 0x94D049BB133111EBull;
    x ^= x >> 31;
    return x;
}

// The tag of a launch that found the sequence number `seq` in its workspace (never 0).
__device__ __forceinline__ uint64_t tag_of(const uint64_t call_tag, const uint64_t seq)
{
    return mix64(call_tag + seq * 0x9E3779B97F4A7C15ull) | 1ull;
}

// Raise the abort flag (shared, and global under this launch's tag if a scan warp got as far as reading it),
// move the workspace's sequence number so that the next launch cannot take this one's words for its own, and
// report the timeout.
static __device__ __noinline__ void raise_timeout(uint64_t *ws_header, int32_t *dev_status, volatile uint32_t *s_abort,
                                           const uint64_t tag)
{
    *s_abort = 1u;
    if (tag) st_relaxed_u64(ws_header + kHdrAbort, tag);
    red_add_u64(ws_header + kHdrSeq, 1ull << 32);
    __threadfence();
    if (dev_status) *reinterpret_cast<volatile int32_t *>(dev_status) = BT_ERR_TIMEOUT;
}

// A limit below this is kept to the nanosecond (see mbar_wait_strict).  Only the test build of the library
// (-DBT_TEST_HOOKS) can set such a limit, and only that build carries the code for it: the product's waits
// are the same instructions with or without it.
constexpr uint64_t kStrictLimitNs = 1000;
constexpr uint64_t kLastNs        = 20000000;         // the last wait for a copy that is in flight
#ifdef BT_TEST_HOOKS
constexpr bool kTestHooks = true;
#else
constexpr bool kTestHooks = false;
#endif

// The wait under a limit of less than a microsecond, which only a test build of the library can set: probes that
// return at once (a try_wait may itself suspend the thread for longer than such a limit), the clock read after
// every probe.  A phase that is not complete at the first probe and does not complete within the limit fails.
static __device__ __noinline__ bool mbar_wait_strict(uint64_t *bar, const uint32_t parity, const uint64_t limit_ns)
{
    const uint64_t t0 = now_ns();
    for (;;) {
        uint32_t ok;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(ok)
            : "r"(smem_addr(bar)), "r"(parity)
            : "memory");
        if (ok) return true;
        if (now_ns() - t0 > limit_ns) return false;
    }
}

// Bounded wait on an mbarrier phase.  False once the limit passed or the CTA is aborting.  The limit is checked
// every 32 probes, each of which may suspend the thread for a while: exact enough for the product's two seconds.
template <bool kStopOnAbort = true>
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, uint32_t parity, volatile uint32_t *s_abort, const uint64_t limit_ns)
{
    if (kTestHooks && limit_ns < kStrictLimitNs) return mbar_wait_strict(bar, parity, limit_ns);
    if (mbar_try_wait(bar, parity)) return true;
    const uint64_t t0 = now_ns();
    for (;;) {
#pragma unroll 1
        for (int i = 0; i < 32; ++i)
            if (mbar_try_wait(bar, parity)) return true;
        if ((kStopOnAbort && *s_abort) || now_ns() - t0 > limit_ns) return false;
    }
}

// ---------------------------------------------------------------------------------------------
// A segment of a tile as one warp compacts it: one block, for 2-byte elements two, of kRows rows of 32 * kE elements,
// lane l owning the kE consecutive elements l * kE .. of every row.  A lane keeps its elements in registers and four
// flag bits per row (bit j of nibble r: element j of row r survives) in ONE 32-bit word per block; the ranks come from
// counts packed four rows to a register (bytes: at most 128 survivors of a row), so that a warp scan of two registers
// ranks all eight rows of a block at once.
//
// Four elements per lane and row keep the survivors of a row within 256 (2-byte) or 512 bytes, so that the predicated
// stores of a row meet in few banks (eight 2-byte elements per lane were measured to lose there what they save).
template <typename U>
struct Rows {
    static constexpr int kE      = sizeof(U) == 8 ? 2 : 4;                 // consecutive elements of a lane in a row
    static constexpr int kRows   = 8;
    static constexpr int kBlock  = kRows * 32 * kE;                        // 1024 elements (512 of 8 bytes)
    static constexpr int kBlocks = sizeof(U) == 2 ? 2 : 1;
    static constexpr int kSeg    = kBlocks * kBlock;                       // 4096 bytes whatever the type
    static constexpr int kRegs   = kE * static_cast<int>(sizeof(U)) / 4;   // registers of a lane per row: 2 or 4
    uint32_t x[kBlocks][kRows][kRegs];
};

template <typename U>
__device__ __forceinline__ void load_rows(Rows<U> &s, const uint32_t seg_addr, const uint32_t lane)
{
    using R = Rows<U>;
#pragma unroll
    for (int r = 0; r < R::kBlocks * R::kRows; ++r) {
        const uint32_t at = seg_addr + static_cast<uint32_t>(r) * (128u * R::kRegs) + lane * (4u * R::kRegs);
        uint32_t(&x)[R::kRegs] = s.x[r / R::kRows][r % R::kRows];
        if constexpr (R::kRegs == 4)
            asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(x[0]), "=r"(x[1]), "=r"(x[2]), "=r"(x[3]) : "r"(at));
        else
            asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(x[0]), "=r"(x[1]) : "r"(at));
    }
}

// acc += bit where the element is not the zero pattern / is kept by the ReLU (greater than zero, or a NaN); the latter
// also gives the ReLU's dense value.
__device__ __forceinline__ void flag_nonzero(uint32_t &acc, const uint32_t x, const uint32_t bit)
{
    asm("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %1, 0;\n\t@p add.u32 %0, %0, %2;\n\t}" : "+r"(acc) : "r"(x), "r"(bit));
}
__device__ __forceinline__ uint32_t flag_relu(uint32_t &acc, const uint32_t x, const uint32_t bit)
{
    uint32_t y;
    asm("{\n\t.reg .pred p;\n\tsetp.gtu.f32 p, %2, 0f00000000;\n\t@p add.u32 %0, %0, %3;\n\tselp.b32 %1, %2, 0, p;\n\t}"
        : "+r"(acc), "=r"(y) : "f"(__uint_as_float(x)), "r"(bit));
    return y;
}

// Two packed 2-byte elements compared in their own type: 0xFFFF in the half of an element that is kept by the ReLU
// (greater than zero or a NaN) resp. saturated by the ReLU6 (at least 6), else 0.
template <int DT>
__device__ __forceinline__ uint32_t relu_keeps_pair(const uint32_t x)
{
    uint32_t m;
    if constexpr (DT == BT_F16) asm("set.gtu.u32.f16x2 %0, %1, %2;" : "=r"(m) : "r"(x), "r"(0u));
    else asm("set.gtu.u32.bf16x2 %0, %1, %2;" : "=r"(m) : "r"(x), "r"(0u));
    return m;
}
template <int DT>
__device__ __forceinline__ uint32_t relu6_saturates_pair(const uint32_t x)
{
    uint32_t m;
    if constexpr (DT == BT_F16) asm("set.ge.u32.f16x2 %0, %1, %2;" : "=r"(m) : "r"(x), "r"(0x46004600u));
    else asm("set.ge.u32.bf16x2 %0, %1, %2;" : "=r"(m) : "r"(x), "r"(0x40C040C0u));
    return m;
}

// The flag word of the lane's elements of a block (its rows); the fused forms replace the elements by their forward value
// on the way (the forms decided by one compare leave elements that are not kept as they are: their flag is clear) and,
// with WRITE_Y, put it in the elements' place in the input slot (`slot`: shared address of the block).
template <typename U, int FUSED, bool WRITE_Y>
__device__ __forceinline__ uint32_t flag_rows(uint32_t (&rows)[8][Rows<U>::kRegs], const uint32_t lane, const uint32_t slot, const float tau)
{
    using R                = Rows<U>;
    constexpr bool kDirect = FUSED >= kFusedReluDirect;
    uint32_t acc[4] = {0, 0, 0, 0};                       // byte b of the flag word: rows 2b and 2b + 1
#pragma unroll
    for (int r = 0; r < R::kRows; ++r) {
        uint32_t yv[R::kRegs];
        if constexpr (sizeof(U) == 2) {
#pragma unroll
            for (int h = 0; h < R::kRegs; ++h) {
                uint32_t &x = rows[r][h];
                const int i = 4 * (r & 1) + 2 * h;        // bit of the pair's first element within the byte
                if constexpr (FUSED < 0) {
                    // 1 per non-zero half, then both flags into place by one multiply-add of bytes
                    acc[r >> 1] = __dp4a(__vminu2(x, 0x00010001u), (1u << i) | ((2u << i) << 16), acc[r >> 1]);
                } else if constexpr (kDirect) {
                    const uint32_t m = relu_keeps_pair<FUSED & 3>(x);
                    if constexpr (FUSED >= kFusedRelu6Direct) {
                        const uint32_t q = relu6_saturates_pair<FUSED & 3>(x);
                        x                = (x & ~q) | (Elem<FUSED & 3>::kSix * 0x00010001u & q);
                    }
                    // bytes 0 and 2 of the mask are 0 or -1
                    const uint32_t c = (static_cast<uint32_t>(-(1 << i)) & 0xFFu) | ((static_cast<uint32_t>(-(2 << i)) & 0xFFu) << 16);
                    acc[r >> 1]      = static_cast<uint32_t>(__dp4a(static_cast<int>(m), static_cast<int>(c), static_cast<int>(acc[r >> 1])));
                    yv[h]            = x & m;
                } else {
                    const uint32_t lo = fused_forward<FUSED>(x & 0xFFFFu, tau), hi = fused_forward<FUSED>(x >> 16, tau);
                    flag_nonzero(acc[r >> 1], lo, 1u << i);
                    flag_nonzero(acc[r >> 1], hi, 2u << i);
                    x     = lo | (hi << 16);
                    yv[h] = x;
                }
            }
        } else {
#pragma unroll
            for (int j = 0; j < R::kE; ++j) {
                const uint32_t bit = 1u << (4 * (r & 1) + j);
                if constexpr (sizeof(U) == 4) {
                    uint32_t &x = rows[r][j];
                    if constexpr (kDirect) {
                        yv[j] = flag_relu(acc[r >> 1], x, bit);
                    } else {
                        if constexpr (FUSED >= 0) x = fused_forward<FUSED>(x, tau);
                        flag_nonzero(acc[r >> 1], x, bit);
                        yv[j] = x;
                    }
                } else {
                    uint64_t x = rows[r][2 * j] | (static_cast<uint64_t>(rows[r][2 * j + 1]) << 32);
                    if constexpr (FUSED >= 0) {
                        x                 = fused_forward<FUSED>(x, tau);
                        rows[r][2 * j]     = static_cast<uint32_t>(x);
                        rows[r][2 * j + 1] = static_cast<uint32_t>(x >> 32);
                    }
                    flag_nonzero(acc[r >> 1], static_cast<uint32_t>(x) | static_cast<uint32_t>(x >> 32), bit);
                    yv[2 * j] = static_cast<uint32_t>(x), yv[2 * j + 1] = static_cast<uint32_t>(x >> 32);
                }
            }
        }
        if constexpr (WRITE_Y) {
            const uint32_t at = slot + static_cast<uint32_t>(r) * (128u * R::kRegs) + lane * (4u * R::kRegs);
            if constexpr (R::kRegs == 4)
                asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(at), "r"(yv[0]), "r"(yv[1]), "r"(yv[2]), "r"(yv[3]) : "memory");
            else
                asm volatile("st.shared.v2.u32 [%0], {%1, %2};" ::"r"(at), "r"(yv[0]), "r"(yv[1]) : "memory");
        }
    }
    return acc[0] | (acc[1] << 8) | (acc[2] << 16) | (acc[3] << 24);
}

// Ranks: byte k of excl[i] is the number of survivors in the lanes below within row 2k + i, of total[i] the survivors
// of that row.
struct RowRanks {
    uint32_t excl[2], total[2];
    __device__ __forceinline__ uint32_t count() const { return __dp4a(total[0], 0x01010101u, __dp4a(total[1], 0x01010101u, 0u)); }
};

template <int kBy>
__device__ __forceinline__ void scan_step(uint32_t &v)
{
    asm volatile("{\n\t.reg .pred p;\n\t.reg .b32 t;\n\tshfl.sync.up.b32 t|p, %0, %1, 0, 0xFFFFFFFF;\n\t@p add.u32 %0, %0, t;\n\t}" : "+r"(v) : "n"(kBy));
}

__device__ __forceinline__ void rank_rows(RowRanks &k, const uint32_t flags)
{
    // survivors per row: population counts of the nibbles, all eight at once
    uint32_t c = flags - ((flags >> 1) & 0x55555555u);
    c          = (c & 0x33333333u) + ((c >> 2) & 0x33333333u);
    const uint32_t own0 = c & 0x0F0F0F0Fu, own1 = (c >> 4) & 0x0F0F0F0Fu;
    uint32_t       v0 = own0, v1 = own1;
    scan_step<1>(v0), scan_step<1>(v1);
    scan_step<2>(v0), scan_step<2>(v1);
    scan_step<4>(v0), scan_step<4>(v1);
    scan_step<8>(v0), scan_step<8>(v1);
    scan_step<16>(v0), scan_step<16>(v1);
    k.total[0] = __shfl_sync(kFull, v0, 31), k.total[1] = __shfl_sync(kFull, v1, 31);
    k.excl[0] = v0 - own0, k.excl[1] = v1 - own1;
}

// A block's bitmap words.  A lane's nibbles are exchanged with three neighbours (four for 8-byte elements, whose
// rows give a lane two bits) until it holds one whole word; `index` receives the word's place within the block.
// True if this lane has a word (all lanes; every other one for 8-byte elements).
template <int kE>
__device__ __forceinline__ bool block_word(const uint32_t flags, const uint32_t lane, uint32_t &word, uint32_t &index)
{
    uint32_t a = flags, v = lane;                          // v: lane number among those that hold distinct bits
    if constexpr (kE == 2) {
        const uint32_t b = __shfl_xor_sync(kFull, a, 1);   // two lanes' pairs of bits make a nibble, on both lanes
        a                = (lane & 1u) ? (b | (a << 2)) : (a | (b << 2));
        v                = lane >> 1;
    }
    constexpr int kX = kE == 2 ? 2 : 1;
    // rows 0..3 to the even, rows 4..7 to the odd holder: the nibbles of the two, interleaved into four bytes
    uint32_t b = __shfl_xor_sync(kFull, a, kX);
    a          = __byte_perm(a, b, (v & 1u) ? 0x3726u : 0x5140u);
    const uint32_t m = (a ^ (a >> 4)) & 0x00F000F0u;
    a                = a ^ m ^ (m << 4);
    b = __shfl_xor_sync(kFull, a, 2 * kX);                 // two rows each: 16 bits per row
    a = __byte_perm(a, b, (v & 2u) ? 0x3726u : 0x5140u);
    b = __shfl_xor_sync(kFull, a, 4 * kX);                 // one row each: 32 bits
    a = __byte_perm(a, b, (v & 4u) ? 0x3276u : 0x5410u);
    word               = a;
    const uint32_t row = 4u * (v & 1u) + (v & 2u) + ((v >> 2) & 1u);
    index              = row * static_cast<uint32_t>(kE) + (v >> 3);
    return kE == 4 || (lane & 1u) == 0;
}

// The survivors of a block to shared memory, packed from address `out` on.  kES: bytes of a stored value, kE: a lane's elements
// per row; x[r] holds row r.  Returns the address behind the last survivor.
template <int kES, int kE>
__device__ __forceinline__ uint32_t place_rows(const uint32_t (&x)[8][kES * kE / 4], const uint32_t flags, const RowRanks &k, uint32_t out)
{
#pragma unroll
    for (int r = 0; r < 8; ++r) {
        const uint32_t f  = static_cast<uint32_t>(kES) << (8 * (r >> 1));   // picks the row's byte and scales it
        uint32_t       at = __dp4a(k.excl[r & 1], f, out);
        out               = __dp4a(k.total[r & 1], f, out);
#pragma unroll
        for (int j = 0; j < kE; ++j) {
            const uint32_t bit = 1u << (4 * r + j);
            if constexpr (kES == 2)
                asm volatile("{\n\t.reg .pred p;\n\t.reg .b32 t;\n\tand.b32 t, %1, %2;\n\tsetp.ne.u32 p, t, 0;\n\t@p st.shared.u16 [%0], %3;\n\t}"
                             :: "r"(at), "r"(flags), "r"(bit), "h"(static_cast<uint16_t>(x[r][j >> 1] >> (16 * (j & 1)))) : "memory");
            else if constexpr (kES == 4)
                asm volatile("{\n\t.reg .pred p;\n\t.reg .b32 t;\n\tand.b32 t, %1, %2;\n\tsetp.ne.u32 p, t, 0;\n\t@p st.shared.u32 [%0], %3;\n\t}"
                             :: "r"(at), "r"(flags), "r"(bit), "r"(x[r][j]) : "memory");
            else
                asm volatile("{\n\t.reg .pred p;\n\t.reg .b32 t;\n\tand.b32 t, %1, %2;\n\tsetp.ne.u32 p, t, 0;\n\t@p st.shared.v2.u32 [%0], {%3, %4};\n\t}"
                             :: "r"(at), "r"(flags), "r"(bit), "r"(x[r][2 * j]), "r"(x[r][2 * j + 1]) : "memory");
            if (j + 1 < kE) asm("{\n\t.reg .pred p;\n\t.reg .b32 t;\n\tand.b32 t, %1, %2;\n\tsetp.ne.u32 p, t, 0;\n\t@p add.u32 %0, %0, %3;\n\t}" : "+r"(at) : "r"(flags), "r"(bit), "n"(kES));
        }
    }
    return out;
}

// Down-cast on stash: two binary32 patterns narrowed to a packed pair of binary16 (CAST 1) or bfloat16 (CAST 2), round
// to nearest even by the hardware conversion, every NaN to the one quiet NaN 0x7FFF (a NaN always narrows to a NaN and
// nothing else does, so the packed result is what is asked).
template <int CAST>
__device__ __forceinline__ uint32_t narrowed_pair(const uint32_t lo, const uint32_t hi)
{
    uint32_t h, m;
    if constexpr (CAST == 1) {
        asm("cvt.rn.f16x2.f32 %0, %1, %2;" : "=r"(h) : "f"(__uint_as_float(hi)), "f"(__uint_as_float(lo)));
        asm("set.nan.u32.f16x2 %0, %1, %1;" : "=r"(m) : "r"(h));
    } else {
        asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(h) : "f"(__uint_as_float(hi)), "f"(__uint_as_float(lo)));
        asm("set.nan.u32.bf16x2 %0, %1, %1;" : "=r"(m) : "r"(h));
    }
    return (h & ~m) | (0x7FFF7FFFu & m);
}
template <int CAST, typename U>
using Stored = std::conditional_t<CAST == 0, U, uint16_t>;

__device__ __forceinline__ uint4 lds_vec(const uint32_t addr)
{
    uint4 v;
    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr));
    return v;
}
template <typename V>
__device__ __forceinline__ V lds_value(const uint32_t addr)
{
    V v;
    if constexpr (sizeof(V) == 8) asm volatile("ld.shared.u64 %0, [%1];" : "=l"(v) : "r"(addr));
    else if constexpr (sizeof(V) == 4) asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(addr));
    else asm volatile("ld.shared.u16 %0, [%1];" : "=h"(v) : "r"(addr));
    return v;
}

// 16 bytes of a packed run kBytes (0 .. 14) behind a 16-byte boundary of shared memory.
template <int kWords, bool kHalf>
__device__ __forceinline__ uint4 lds_vec_shifted(const uint32_t addr)
{
    const uint4 a = lds_vec(addr);
    if constexpr (kWords == 0 && !kHalf) {
        return a;
    } else {
        const uint4    b    = lds_vec(addr + 16);
        const uint32_t w[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
        if constexpr (kHalf)
            return make_uint4(__byte_perm(w[kWords], w[kWords + 1], 0x5432), __byte_perm(w[kWords + 1], w[kWords + 2], 0x5432),
                              __byte_perm(w[kWords + 2], w[kWords + 3], 0x5432), __byte_perm(w[kWords + 3], w[kWords + 4], 0x5432));
        else return make_uint4(w[kWords], w[kWords + 1], w[kWords + 2], w[kWords + 3]);
    }
}

template <typename V, int kWords, bool kHalf>
__device__ __forceinline__ void copy_vectors(const uint32_t from, const uint32_t lane, const uint32_t vecs, V *to, const Extent vx)
{
    constexpr uint32_t kPer = 16 / sizeof(V);
#pragma unroll 2
    for (uint32_t v = lane; v < vecs; v += 32) {
        const uint4 d = lds_vec_shifted<kWords, kHalf>(from + 16u * v);
        if (vx.holds(to + kPer * v, 16)) *reinterpret_cast<uint4 *>(to + kPer * v) = d;
    }
}

// One warp copies the `cnt` packed values at the 16-byte aligned shared address `from` to out[0 .. cnt).  The
// destination is wherever the run's rank puts it: the values in front of its first 16-byte boundary and behind its last
// one leave as single elements, the rest as 16-byte vectors put together from two shared vectors (the shift is the same
// for the whole warp).  Never reads past the last whole 16 bytes that the run touches.
template <typename V>
__device__ __forceinline__ void copy_out_run(const uint32_t from, const uint32_t lane, const uint32_t cnt, V *out, const Extent vx)
{
    constexpr uint32_t kPer = 16 / sizeof(V);
    uint32_t           h    = (static_cast<uint32_t>(16u - (reinterpret_cast<uintptr_t>(out) & 15u)) & 15u) / static_cast<uint32_t>(sizeof(V));
    h                       = h < cnt ? h : cnt;                 // values in front of the first boundary
    const uint32_t vecs = (cnt - h) / kPer;                      // whole 16-byte units behind them
    const uint32_t tail = h + kPer * vecs;                       // first of the values behind the last unit
    const bool     is_head = lane < h, is_tail = lane >= 16u && tail + (lane - 16u) < cnt;
    if (is_head || is_tail) {
        const uint32_t e = is_head ? lane : tail + (lane - 16u);
        const V        v = lds_value<V>(from + e * static_cast<uint32_t>(sizeof(V)));
        if (vx.holds(out + e, sizeof(V))) out[e] = v;
    }
    V *const to = out + h;
    if constexpr (sizeof(V) == 8) {
        if (h == 0) copy_vectors<V, 0, false>(from, lane, vecs, to, vx);
        else copy_vectors<V, 2, false>(from, lane, vecs, to, vx);
    } else if constexpr (sizeof(V) == 4) {
        switch (h) {
        case 0: copy_vectors<V, 0, false>(from, lane, vecs, to, vx); break;
        case 1: copy_vectors<V, 1, false>(from, lane, vecs, to, vx); break;
        case 2: copy_vectors<V, 2, false>(from, lane, vecs, to, vx); break;
        default: copy_vectors<V, 3, false>(from, lane, vecs, to, vx); break;
        }
    } else {
        switch (h) {
        case 0: copy_vectors<V, 0, false>(from, lane, vecs, to, vx); break;
        case 1: copy_vectors<V, 0, true>(from, lane, vecs, to, vx); break;
        case 2: copy_vectors<V, 1, false>(from, lane, vecs, to, vx); break;
        case 3: copy_vectors<V, 1, true>(from, lane, vecs, to, vx); break;
        case 4: copy_vectors<V, 2, false>(from, lane, vecs, to, vx); break;
        case 5: copy_vectors<V, 2, true>(from, lane, vecs, to, vx); break;
        case 6: copy_vectors<V, 3, false>(from, lane, vecs, to, vx); break;
        default: copy_vectors<V, 3, true>(from, lane, vecs, to, vx); break;
        }
    }
}

// The same where the values buffer ends inside the run: only the first `room` values leave.
template <typename V>
__device__ __forceinline__ void copy_out_clipped(const uint32_t from, const uint32_t lane, const uint32_t cnt, V *out, const uint64_t room,
                                                 const Extent vx)
{
    for (uint32_t j = lane; j < cnt && j < room; j += 32) {
        const V v = lds_value<V>(from + j * static_cast<uint32_t>(sizeof(V)));
        if (vx.holds(out + j, sizeof(V))) out[j] = v;
    }
}

// ---------------------------------------------------------------------------------------------
// Shared memory of a CTA besides the ring of tiles and the worker warps' rings of packed values.  A tile goes round
// through five mbarriers: its ring slot through `full` and `empty` (forms with the dense output: `written` in between),
// its place in the queue of the last kQueue tiles through `counted`, `ready` and `done`.
constexpr int kQueue = 8;   // tiles of a CTA between their count and the end of their copy-out
// The numbers of a CTA's last kTiles tiles.  The load warp writes the number of tile `it` once tile it - kStages is in
// registers.  Every worker has then posted the counts up to tile it - 2 kStages, and so all is done with the tiles kQueue
// before that one.
constexpr int      kTiles  = 16;
constexpr uint32_t kNoTile = 0xFFFFFFFFu;             // behind a CTA's last tile, kStages times
template <int kSegs, int kStages>
struct CtaState {
    uint64_t full[kStages];           // the bulk copy of the tile has landed               (copy engine -> workers)
    uint64_t empty[kStages];          // every segment of the tile is in registers          (workers -> load warp),
                                      // or the dense output has left the slot              (store warp -> load warp)
    uint64_t written[kStages];        // the dense output is in the slot                    (workers -> store warp)
    uint64_t counted[kQueue];         // every segment's count is posted                    (workers -> scan warps)
    uint64_t ready[kQueue];           // base and offsets are in shared, the count is out   (scan, publishing warps -> workers)
    uint64_t done[kQueue];            // every segment has been copied out                  (workers -> workers)
    uint64_t base[kQueue];            // exclusive base of the tile
    uint64_t dst[kQueue];             // batched arena form: byte offset of the tile's tensor in the arena
    uint32_t job[kQueue];             // batched form: the tile's tensor
    uint32_t cnt[kQueue][kSegs];      // packed count of each segment
    uint32_t off[kQueue][kSegs];      // exclusive offset of each segment in the tile
    uint32_t at[kQueue][kSegs];       // where in its worker's ring a segment's values start
    uint32_t tile[kTiles];            // the tiles' numbers (kNoTile: the stream has ended)
    __align__(16) uint64_t offer[2];  // the answer to the load warp's request for the tile of a CTA that has not started,
    uint64_t offered;                 // and the barrier that it arrives on
    volatile uint64_t tag;            // this launch's tag once the first scan warp has it, else 0
    uint64_t          arena_c0;       // arena forms: the cursor as the launch found it
    volatile uint32_t abort;
    // by the first threads of the CTA, one barrier each; a CTA-wide barrier follows
    __device__ __forceinline__ void init(const bool dense_output, const bool publisher, const uint32_t tid)
    {
        if (tid == 0) abort = 0, tag = 0;
        if (tid < kStages) {
            mbar_init(&full[tid], 1), mbar_init(&empty[tid], dense_output ? 1 : kSegs), mbar_init(&written[tid], kSegs);
        } else if (tid - kStages < kQueue) {
            const uint32_t q = tid - kStages;
            mbar_init(&counted[q], kSegs), mbar_init(&ready[q], publisher ? 2 : 1), mbar_init(&done[q], kSegs);
        }
        static_assert(2 * kStages + kQueue <= kTiles, "a tile's number outlives the tile");
        if (tid < kStages + kQueue) fence_proxy_async();
    }
};

// One CTA per SM; the input ring and the workers' rings take nearly all of its shared memory.  Three slots of 32 KB keep
// the loads going (measured with loads alone: 6.2 to 6.4 TB/s with 3 to 7 slots), since a slot is free again as soon as
// its tile is in registers.
struct Shape {
    static constexpr int kSegs = 8, kWorkers = 24, kStages = 3, kRing = 5376;
};
// Do the CTAs have a warp for publishing the counts (see scan_tiles)?
template <typename U>
constexpr bool kPublisher = sizeof(U) >= 4;
// load warp, two scan warps, and as the form has them a publishing and a store warp
template <typename U>
constexpr int warps_of(const bool dense_output)
{
    return Shape::kWorkers + 3 + (kPublisher<U> ? 1 : 0) + (dense_output ? 1 : 0);
}

// A tile's descriptor: its count under the launch's tag, twice.
__device__ __forceinline__ void post(uint64_t *desc, const uint32_t count, const uint64_t tag)
{
    st_relaxed_2xu64(desc, (tag & 0xFFFFFFFF00000000ull) | count, (tag << 32) | count);
}

// The launch's tag as the first scan warp left it in shared memory (bounded wait; 0 if the CTA is aborting).
__device__ __forceinline__ uint64_t wait_tag(volatile uint64_t *s_tag, volatile uint32_t *s_abort, const uint64_t limit_ns)
{
    uint64_t t = *s_tag;
    if (t) return t;
    const uint64_t t0 = now_ns();
    for (;;) {
#pragma unroll 1
        for (int i = 0; i < 32; ++i) {
            t = *s_tag;
            if (t) return t;
        }
        if (*s_abort || now_ns() - t0 > limit_ns) return 0;
    }
}

// The counts in front of a tile, as a scan warp reads them: d0[k], d1[k], lane l <-> descriptor from + l + 32k.
struct Window {
    uint64_t d0[kMaxWindows], d1[kMaxWindows];
    uint32_t from, size;
    __device__ static __forceinline__ bool valid(const uint64_t w0, const uint64_t w1, const uint64_t tag)
    {
        return ((w0 ^ tag) >> 32) == 0 && ((w1 >> 32) ^ (tag & 0xFFFFFFFFull)) == 0 && static_cast<uint32_t>(w0) == static_cast<uint32_t>(w1);
    }
    // One batch of independent loads, from `from` on towards tile `to`.
    __device__ __forceinline__ void read(const uint64_t *desc, const uint32_t to, const uint64_t tag, const uint32_t lane)
    {
        size = to - from < 32u * kMaxWindows ? to - from : 32u * kMaxWindows;
#pragma unroll
        for (int k = 0; k < kMaxWindows; ++k) {
            if (lane + 32u * k < size) ld_relaxed_2xu64(desc + 2 * (static_cast<uint64_t>(from) + lane + 32u * k), d0[k], d1[k]);
            else d0[k] = tag & 0xFFFFFFFF00000000ull, d1[k] = tag << 32;             // no such tile: a valid count of 0
        }
    }
    // Polls until all are published.  False if the wait ran out or the launch is giving up.
    __device__ __forceinline__ bool settle(const uint64_t *desc, const uint64_t *header, const uint64_t tag, const uint32_t lane, const uint32_t pause_ns,
                                           const uint64_t wait_ns)
    {
        uint32_t polls = 0;
        uint64_t t0    = 0;
        for (;;) {
            bool missing = false;
#pragma unroll
            for (int k = 0; k < kMaxWindows; ++k) missing |= !valid(d0[k], d1[k], tag);
            if (!__any_sync(kFull, missing)) return true;
            __nanosleep(pause_ns);
            if ((++polls & 255u) == 0 || (kTestHooks && wait_ns < kStrictLimitNs)) {
                if (t0 == 0) t0 = now_ns();
                if (__any_sync(kFull, (now_ns() - t0 > wait_ns) || ld_relaxed_u64(header + kHdrAbort) == tag)) return false;
            }
#pragma unroll
            for (int k = 0; k < kMaxWindows; ++k)
                if (!valid(d0[k], d1[k], tag)) ld_relaxed_2xu64(desc + 2 * (static_cast<uint64_t>(from) + lane + 32u * k), d0[k], d1[k]);
        }
    }
    // The sum of the counts (of those from tile lo to before hi): at most 160 tiles of 16384 elements.
    __device__ __forceinline__ uint32_t sum() const
    {
        uint32_t part = 0;
#pragma unroll
        for (int k = 0; k < kMaxWindows; ++k) part += static_cast<uint32_t>(d0[k]);
        return __reduce_add_sync(kFull, part);
    }
    __device__ __forceinline__ uint32_t sum(const uint32_t lo, const uint32_t hi, const uint32_t lane) const
    {
        uint32_t part = 0;
#pragma unroll
        for (int k = 0; k < kMaxWindows; ++k) {
            const uint64_t at = static_cast<uint64_t>(from) + lane + 32u * k;
            part += at >= lo && at < hi ? static_cast<uint32_t>(d0[k]) : 0u;
        }
        return __reduce_add_sync(kFull, part);
    }
};

// A tile's counts as a scan warp has them.
template <int kSegs>
struct TileCounts {
    uint32_t own, upto;       // lane s: the count of the tile's segment s, and of its segments up to s
    uint32_t count;           // of the tile
    // from the counts of the CTA's tile j; leaves the segments' offsets in the tile for the workers
    template <typename State>
    __device__ __forceinline__ void take(State &sh, const uint32_t j, const uint32_t lane)
    {
        own  = lane < kSegs ? sh.cnt[j % kQueue][lane] : 0u;
        upto = own;
#pragma unroll
        for (int o = 1; o < kSegs; o <<= 1) {
            const uint32_t u = __shfl_up_sync(kFull, upto, o);
            if (lane >= static_cast<uint32_t>(o)) upto += u;
        }
        if (lane < kSegs) sh.off[j % kQueue][lane] = upto - own;
        count = __shfl_sync(kFull, upto, kSegs - 1);
    }
};

// A scan warp's tag: the first one makes it from the sequence number, which changes only once all counts of the launch are
// published, or two seconds into a failure; a CTA publishes none before it has the tag.  0 if the CTA is aborting.
template <int kSegs, int kStages>
__device__ __forceinline__ uint64_t scan_tag(CtaState<kSegs, kStages> &sh, const uint32_t p, const uint32_t lane, const uint64_t call_tag,
                                             const uint64_t *header, const uint64_t wait_ns)
{
    uint64_t tag = 0;
    if (lane == 0) {
        if (p == 0) sh.tag = tag = tag_of(call_tag, ld_relaxed_u64(header + kHdrSeq));
        else tag = wait_tag(&sh.tag, &sh.abort, wait_ns);
    }
    return __shfl_sync(kFull, tag, 0);
}

// What the two scan warps of a CTA do.  Warp p takes the CTA's tiles p, p + 2, p + 4, ... (in the order the CTA takes them).
// Its turn for the CTA's tile j:
//   wait until tile j + 1 is counted -- about one tile later, when the tiles in front of tile j, taken at about the same
//     time by other CTAs, are counted and published too -- and read, in ONE batch of independent loads, the descriptors
//     from the CTA's tile j - 1 up to tile j.  2-byte types and dense tiles (11/16 and more survive), whose CTAs are further
//     apart, read 0.1 us later, so that the first read usually finds everything: fp32 2^26 without zeros 94.1 -> 88.7 us,
//     2^27 at 30 % zeros with the restore 290.9 -> 281.9, bf16 2^27 78.4 -> 76.8 (fp32 at 90 % zeros 51.6 and 51.8);
//   wait until tile j + 2 is counted: the loads have arrived by then (the round trip to L2 takes 1.3 us under load).
//     Handed to the workers as soon as the loads are there, bases come before the workers are through with the counting,
//     and dense tensors, whose values then leave in smaller pieces, lose what sparse ones gain: fp32 2^26 without zeros
//     103 us against 94, with 90 % zeros 53 against 54;
//   finish tile j: its base is that of tile j - 1, which is the other scan warp's, plus the counts.
// Each warp has two tiles' time for a turn.  What the workers wait for most is this exchange, not data (fp32 2^26 at half
// zeros: a third of their time for bases, a tenth for tiles), so nothing else is done between the last wait and the base.
//
// Who publishes the counts.  All CTAs wait for every count, so nothing may hold it up.  4- and 8-byte types: a warp of its own
// (publish_tiles).  2-byte types: the scan warps, in the wait for tile j + 2; their SMs are short of issue slots, and another
// warp costs more than it gives (bf16 2^27 82.7 us against 81; fp32 2^26 with 90 % zeros 54 against 58 the other way).
//
// Stream: tile numbers and tensors.  Scan: what a kernel does with a tile,
//   begin(tile, j)   what does not depend on the counts in front of it,
//   resume(j)        the base of the CTA's tile before,
//   add(window)      the counts from there on,
//   finish(tile, j)  base and offsets for the workers, prefix entries; at a tensor's end nnz and status.
// False if a wait ran out.
template <typename U, bool LISTED, int kSegs, int kStages, typename Stream, typename Scan>
__device__ __forceinline__ bool scan_tiles(CtaState<kSegs, kStages> &sh, const uint32_t p, const uint32_t lane, Stream &stream, Scan &scan,
                                           const uint64_t *desc, const uint64_t *header, const uint64_t tag, const bool one_wave, const uint64_t wait_ns)
{
    auto counted = [&](const uint32_t j) { return mbar_wait(&sh.counted[j % kQueue], (j / kQueue) & 1u, &sh.abort, wait_ns); };
    // waits until tile j is counted and publishes it; its number, or kNoTile behind the last one
    auto next = [&](const uint32_t j, uint32_t &tile) {
        tile = LISTED ? 0u : stream.dealt(j);
        if (tile == kNoTile) return true;
        if (!counted(j)) return false;
        if constexpr (LISTED) tile = sh.tile[j % kTiles];
        if constexpr (!kPublisher<U>) {
            const uint32_t count = __reduce_add_sync(kFull, lane < kSegs ? sh.cnt[j % kQueue][lane] : 0u);
            if (lane == 0 && tile != kNoTile) stream.publish(tile, count, tag);
        }
        return true;
    };
    uint32_t tile, after;
    if (!next(p, tile)) return false;
    for (uint32_t j = p; tile != kNoTile; j += 2, tile = after) {
        uint32_t behind = LISTED ? 0u : stream.dealt(j + 1);
        if (behind != kNoTile && !counted(j + 1)) return false;
        if constexpr (LISTED) behind = sh.tile[(j + 1) % kTiles];
        // The CTA's last tile: there is no next tile to wait for.  A short pause gives the counts in front of it
        // time to land, so that the reads below usually succeed at once instead of costing a second
        // round trip; a launch of one wave, whose counts come all at once, does not pause (fp32 200704
        // elements 7.2 -> 6.7 us; 2.4 M elements, two waves: 9.9 -> 10.4 without the pause).
        if (behind == kNoTile) __nanosleep(one_wave ? 20 : 300);
        Window w;
        w.from = j == 0 ? 0u : LISTED ? sh.tile[(j - 1) % kTiles] : tile - gridDim.x;
        scan.begin(tile, j);
        if (behind != kNoTile && (sizeof(U) == 2 || scan.count * 16u >= 11u * kSegs * Rows<U>::kSeg)) __nanosleep(100);
        w.read(desc, tile, tag, lane);
        after = kNoTile;
        if (behind != kNoTile && !next(j + 2, after)) return false;
        if (!w.settle(desc, header, tag, lane, one_wave ? 20 : 100, wait_ns)) return false;
        if (j > 0 && !mbar_wait(&sh.ready[(j - 1) % kQueue], ((j - 1) / kQueue) & 1u, &sh.abort, wait_ns)) return false;
        scan.resume(j);
        // (a window is cut only where a CTA was slow or started late, behind a kernel that took its SM for a while)
        for (;;) {
            scan.add(w);
            if (w.from + w.size == tile) break;
            w.from += w.size;
            w.read(desc, tile, tag, lane);
            if (!w.settle(desc, header, tag, lane, 100, wait_ns)) return false;
        }
        scan.finish(tile, j);
    }
    return true;
}

// The tile a worker looks at, and where a tile's values go.
struct TileIn {
    uint64_t    n, first;       // elements of the tensor, first element of the tile
    const void *src;
    void       *y;
    uint32_t   *bitmap;
};
struct TileOut {
    void    *values;
    uint64_t capacity;          // in values
};

// ---------------------------------------------------------------------------------------------
// Which tiles a CTA takes (deal_of says when).  Stealing: the launch has one CTA per tile; a CTA that runs takes its own tile
// first and then, while it works, those of CTAs that have not started (clusterlaunchcontrol.try_cancel), until none is
// left.  Tiles are handed out in ascending order, so whoever waits for the counts of lower tiles waits for tiles that are
// done or in the hands of CTAs that run: no CTA needs another one to be resident.  Else CTA b takes the tiles b, b + G, ...
__device__ __forceinline__ void ask_for_tile(uint64_t (&offer)[2], uint64_t *bar)
{
    fence_proxy_async();                               // the answer before was read by an ordinary load
    mbar_arrive_expect_tx(bar, 16);
    asm volatile("clusterlaunchcontrol.try_cancel.async.shared::cta.mbarrier::complete_tx::bytes.b128 [%0], [%1];" ::"r"(smem_addr(offer)),
                 "r"(smem_addr(bar))
                 : "memory");
}
// kNoTile: refused.  No request may follow a refusal.
__device__ __forceinline__ uint32_t offered_tile(const uint64_t (&offer)[2])
{
    uint32_t tile;
    asm volatile(
        "{\n\t.reg .b128 r;\n\t.reg .pred p;\n\t"
        "ld.shared.b128 r, [%1];\n\t"
        "mov.u32 %0, 0xFFFFFFFF;\n\t"
        "clusterlaunchcontrol.query_cancel.is_canceled.pred.b128 p, r;\n\t"
        "@p clusterlaunchcontrol.query_cancel.get_first_ctaid::x.b32.b128 %0, r;\n\t}"
        : "=r"(tile)
        : "r"(smem_addr(offer))
        : "memory");
    return tile;
}

// The first request goes out before the CTA waits for the kernel in front (by the load warp's lane).
template <int kSegs, int kStages>
__device__ __forceinline__ void ask_first(CtaState<kSegs, kStages> &sh)
{
    mbar_init(&sh.offered, 1);
    ask_for_tile(sh.offer, &sh.offered);
}

// The load warp's lane: one bulk copy per tile into the ring, kStages tiles ahead of the workers at most.  One request for a
// tile is under way at a time, so that a CTA's tiles ascend; its answer has a tile's time to arrive (two or four under way
// are no faster: bf16 64 MiB with dense output 31.2 us, 31.5, 31.9).
template <typename U, bool LISTED, int kSegs, int kStages, typename Stream>
__device__ __forceinline__ void load_tiles(CtaState<kSegs, kStages> &sh, U *tiles, Stream &stream, const uint32_t num_tiles, const bool stealing,
                                           const uint64_t wait_ns)
{
    constexpr uint32_t kTile = kSegs * Rows<U>::kSeg;
    uint64_t tile = blockIdx.x;                        // 64-bit: running past the end cannot wrap
    uint32_t it = 0, ends = 0, answers = 0;
    bool     asked = stealing;
    for (; ends < kStages; ++it) {
        const uint32_t s = it % kStages;
        if (it >= static_cast<uint32_t>(kStages) && !mbar_wait(&sh.empty[s], ((it / kStages) - 1) & 1u, &sh.abort, wait_ns)) break;
        if (tile >= num_tiles) {
            if (!LISTED) break;
            sh.tile[it % kTiles] = kNoTile;
            mbar_arrive(&sh.full[s]);
            ++ends;
            continue;
        }
        if (LISTED) sh.tile[it % kTiles] = static_cast<uint32_t>(tile);
        TileIn t;
        stream.locate(static_cast<uint32_t>(tile), t);
        const uint64_t left  = t.n - t.first;
        const uint32_t valid = left < static_cast<uint64_t>(kTile) ? static_cast<uint32_t>(left) : kTile;
        const uint32_t bytes = (valid * static_cast<uint32_t>(sizeof(U))) & ~15u;   // whole 16-byte units
        fence_proxy_async();                       // the workers' accesses to the slot come first
        mbar_arrive_expect_tx(&sh.full[s], bytes);  // bytes == 0 simply completes the phase
        if (bytes) bulk_load(tiles + static_cast<size_t>(s) * kTile, static_cast<const U *>(t.src) + t.first, bytes, &sh.full[s]);
        if (!LISTED || !stealing) {
            tile += gridDim.x;
            continue;
        }
        const uint64_t before = tile;
        tile                  = kNoTile;
        if (asked) {
            if (!mbar_wait(&sh.offered, answers & 1u, &sh.abort, wait_ns)) {
                ++it;
                break;
            }
            ++answers;
            tile  = offered_tile(sh.offer);
            asked = tile != kNoTile;
            if (asked) ask_for_tile(sh.offer, &sh.offered);
            if (tile <= before) {                  // not in ascending order: the launch gives up
                sh.abort = 1u;
                ++it;
                break;
            }
        }
    }
    // This lane stays until everything it asked for has landed, whatever the other warps do (they may leave early once a
    // bounded wait has run out somewhere): the CTA never retires with a copy into its shared memory in flight.  The last
    // kStages copies can be pending, behind the first markers of the end too; a marker's phase is complete.  A launch that
    // gives up takes the CTAs that have not started with it, else each of them would wait anew.  Every wait is bounded.
    for (uint32_t i = it > static_cast<uint32_t>(kStages) ? it - kStages : 0; i < it; ++i)
        mbar_wait<false>(&sh.full[i % kStages], (i / kStages) & 1u, &sh.abort, kLastNs);
    while (asked && mbar_wait<false>(&sh.offered, answers & 1u, &sh.abort, kLastNs)) {
        ++answers;
        asked = offered_tile(sh.offer) != kNoTile;
        if (asked) ask_for_tile(sh.offer, &sh.offered);
    }
}

// One worker warp of a CTA (worker w of kWorkers): takes the segments w, w + kWorkers, w + 2 kWorkers, ... of the CTA's
// stream of tiles -- into registers, flags, ranks, count posted, packed into its own ring in shared memory -- and copies
// each out once its base is known, a few tiles later.  `pack`: false where no values are wanted (a capacity of 0: the call
// is made for bitmap, prefix and count), then neither packing nor copying takes place.  False if a wait ran out.
//
// Every worker does everything, so that what one waits for (a shuffle, a shared load, a base) is filled by the others;
// a warp's chain of dependent steps per segment is about 1500 cycles, as long as a tile takes at full bandwidth, and
// eight warps in step with each tile (which the first version of this kernel had) left the SM waiting half the time.
//
// No worker waits for a base before it has posted the counts that the base needs: the scan makes tile t ready once the
// tiles up to t + 2 are counted, and a worker that waits for tile t has posted its segments of the tiles up to t + 2.
// (After placing a segment of tile `it` it copies out the one of tile it - 3; a lack of room in its ring can only make it do so
// before.)
template <typename U, int FUSED, bool WRITE_Y, int CAST, bool LISTED, int kSegs, int kWorkers, int kStages, int kRing, typename Stream>
__device__ __forceinline__ bool work(CtaState<kSegs, kStages> &sh, U *tiles, const uint32_t ring, const uint32_t w, const uint32_t lane,
                                     Stream &stream, const float tau, const uint64_t wait_ns, const bool pack)
{
    using V                  = Stored<CAST, U>;
    constexpr int      kE    = Rows<U>::kE;
    constexpr int      kSeg  = Rows<U>::kSeg;
    constexpr int      kTile = kSegs * kSeg;
    constexpr uint32_t kES   = sizeof(V);
    constexpr int      kMax  = kSeg * static_cast<int>(kES);        // a segment without zeros
    static_assert(kWorkers == 3 * kSegs, "a worker that packs a segment has its last one, three tiles back, and no other to copy out");
    static_assert(kRing % 16 == 0 && kRing >= kMax, "a segment alone always fits");
    static_assert(3 * kSegs <= kQueue * kSegs - kWorkers - kSegs, "the queue holds every tile not copied out");
    // A wait on a barrier's parity tells two phases apart, not three: a worker that comes to a ring slot must have seen
    // the slot's tile before.  (The copies of different slots may land in any order.)
    static_assert((kStages * kSegs) % kWorkers == 0, "a worker visits a ring slot once per round, in its turn");

    uint32_t it = w / kSegs, seg = w % kSegs;                       // the segment in hand
    uint32_t o_it = it, o_seg = seg, pending = 0;                   // the oldest not yet copied out; their number
    uint32_t held = 0, end = 0;                                     // bytes of the last one packed; the ring's end for the next, 0 or ~0
    auto     next = [](uint32_t &i, uint32_t &s) {
        i += kWorkers / kSegs, s += kWorkers % kSegs;
        if (kWorkers % kSegs != 0 && s >= static_cast<uint32_t>(kSegs)) s -= kSegs, ++i;
    };
    auto copy_oldest = [&]() -> bool {
        const uint32_t q = o_it % kQueue;
        if (!mbar_wait(&sh.ready[q], (o_it / kQueue) & 1u, &sh.abort, wait_ns)) return false;
        const TileOut  o   = stream.out(q);
        const uint32_t cnt = sh.cnt[q][o_seg], from = ring + sh.at[q][o_seg];
        const uint64_t dst = sh.base[q] + sh.off[q][o_seg];
        V *const       to  = static_cast<V *>(o.values) + dst;
        const Extent   vx  = extent_of(o.values, o.capacity * sizeof(V));
        if (dst + cnt <= o.capacity) copy_out_run<V>(from, lane, cnt, to, vx);
        else copy_out_clipped<V>(from, lane, cnt, to, dst < o.capacity ? o.capacity - dst : 0, vx);
        __syncwarp();
        if (lane == 0) mbar_arrive(&sh.done[q]);
        next(o_it, o_seg);
        --pending;
        return true;
    };

    for (TileIn t;; next(it, seg)) {
        const uint32_t s    = it % kStages, q = it % kQueue;
        U *const       tile = tiles + static_cast<size_t>(s) * kTile;
        if (!LISTED && !stream.seek(it, t)) break;
        if (!mbar_wait(&sh.full[s], (it / kStages) & 1u, &sh.abort, wait_ns)) return false;
        if constexpr (LISTED) {
            const uint32_t number = sh.tile[it % kTiles];
            if (number == kNoTile) break;
            stream.locate(number, t);
        }
        if (t.n - t.first < static_cast<uint64_t>(kTile)) {
            // Ragged last tile: each warp completes its own segment -- the elements of the last 16 bytes that the bulk copy
            // left out, zeros behind the end of the tensor -- and meets no other warp over it.  (A barrier among the workers
            // here would never open if one of them had left the kernel because its wait ran out.)  One element per lane for
            // those 16 bytes, then whole vectors: the ragged tile is the last one and everything waits for its count.
            // (Filled element by element, 64 steps for 2-byte types: bf16 200704 elements 7.7 us, this way 6.2.)
            constexpr uint32_t kPer = 16 / sizeof(U);
            const U *const src     = static_cast<const U *>(t.src);
            const uint32_t have    = static_cast<uint32_t>(t.n - t.first);
            const uint32_t by_bulk = have / kPer * kPer;
            const uint32_t seg0    = seg * kSeg;
            if (by_bulk >= seg0 && by_bulk < seg0 + kSeg && lane < kPer)
                tile[by_bulk + lane] = by_bulk + lane < have ? src[t.first + by_bulk + lane] : U(0);
            for (uint32_t e = (by_bulk >= seg0 ? by_bulk + kPer : seg0) + kPer * lane; e < seg0 + kSeg; e += 32 * kPer)
                *reinterpret_cast<uint4 *>(tile + e) = make_uint4(0, 0, 0, 0);
            __syncwarp();
        }
        // the segment into registers; the slot is free for the next tile once every segment is
        Rows<U> rows;
        load_rows<U>(rows, smem_addr(tile + seg * kSeg), lane);
        if constexpr (!WRITE_Y) {
            __syncwarp();
            if (lane == 0) mbar_arrive(&sh.empty[s]);
        }

        const uint64_t e0 = t.first + seg * kSeg;                   // first element of the segment
        constexpr int  kBlocks = Rows<U>::kBlocks, kBlock = Rows<U>::kBlock;
        uint32_t       flags[kBlocks], run = 0;
        RowRanks       ranks[kBlocks];
#pragma unroll
        for (int h = 0; h < kBlocks; ++h) {
            flags[h] = flag_rows<U, FUSED, WRITE_Y>(rows.x[h], lane, smem_addr(tile + seg * kSeg + h * kBlock), tau);
            rank_rows(ranks[h], flags[h]);
            run += ranks[h].count();
        }
        if constexpr (WRITE_Y) {
            fence_proxy_async();                                    // the copy engine reads the dense output next
            __syncwarp();
            if (lane == 0) mbar_arrive(&sh.written[s]);
        }
        // the count first: the exchange of counts waits for nothing else (without values to copy out, a place in the queue
        // is free again once the scan is done with it)
        if (it >= static_cast<uint32_t>(kQueue) && !mbar_wait(pack ? &sh.done[q] : &sh.ready[q], ((it / kQueue) - 1) & 1u, &sh.abort, wait_ns)) return false;
        if (lane == 0) {
            sh.cnt[q][seg] = run;
            mbar_arrive(&sh.counted[q]);
        }
#pragma unroll
        for (int h = 0; h < kBlocks; ++h) {
            uint32_t word, index;
            if (block_word<kE>(flags[h], lane, word, index)) {
                const uint64_t wd = (e0 + h * kBlock) / 32 + index;
                if (wd < ((t.n + 31) >> 5) && extent_of(t.bitmap, 4 * ((t.n + 31) >> 5)).holds(t.bitmap + wd, 4)) t.bitmap[wd] = word;
            }
        }
        if (!pack) continue;
        // Room in the ring: one segment at most is not copied out yet, the worker's last one, three tiles back, and it lies at one of
        // the ring's ends.  This one goes to the other end, if the two fit together; else the last one has to leave first.  (Laid
        // one behind the other instead, two segments with about half of their elements kept end where the next one fits only by
        // chance, and the worker waits for a base early: bf16 2^29 elements at half zeros 313 us, this way 297; fp32 2^24 21.3
        // and 20.4; at a third of zeros, where two never fit, the same.)
        const uint32_t need = run ? (run * kES + 15u) & ~15u : 16u;
        if (pending && held + need > static_cast<uint32_t>(kRing) && !copy_oldest()) return false;
        const uint32_t at = (static_cast<uint32_t>(kRing) - need) & end;
        end = ~end, held = need;
        ++pending;
        if constexpr (CAST != 0) {
            uint32_t h[8][2];
#pragma unroll
            for (int r = 0; r < 8; ++r)
                h[r][0] = narrowed_pair<CAST>(rows.x[0][r][0], rows.x[0][r][1]), h[r][1] = narrowed_pair<CAST>(rows.x[0][r][2], rows.x[0][r][3]);
            place_rows<2, 4>(h, flags[0], ranks[0], ring + at);
        } else {
            uint32_t to = ring + at;
#pragma unroll
            for (int h = 0; h < kBlocks; ++h) to = place_rows<sizeof(U), kE>(rows.x[h], flags[h], ranks[h], to);
        }
        if (lane == 0) sh.at[q][seg] = at;
        __syncwarp();
        // (Copying out whatever is ready already, three tiles later or at once, is slower where the memory is the bound:
        // fp32 2^28 at half zeros 267 us against 256.5.)
        while (pending && o_it + 3 <= it)
            if (!copy_oldest()) return false;
    }
    if constexpr (LISTED) {
        // the end goes on to the scan and store warps like a tile (each worker has a segment in one of its markers)
        const uint32_t s = it % kStages, q = it % kQueue;
        if (it >= static_cast<uint32_t>(kQueue) && !mbar_wait(pack ? &sh.done[q] : &sh.ready[q], ((it / kQueue) - 1) & 1u, &sh.abort, wait_ns)) return false;
        if (lane == 0) {
            if constexpr (WRITE_Y) mbar_arrive(&sh.written[s]);
            mbar_arrive(&sh.counted[q]);
        }
    }
    while (pending)
        if (!copy_oldest()) return false;
    return true;
}

// The publishing warp of the 4- and 8-byte types: sends a tile's count out to the other CTAs as soon as every segment is
// counted.  Published by the worker that counts last, whose chain of steps that lengthens, bf16 2^27 takes 88 us instead of 78;
// by the store warp, behind its wait for the copy engine, fp32 8 MiB with the dense output 7.2 instead of 5.7.  False if a
// wait ran out.
template <typename U, bool LISTED, int kSegs, int kStages, typename Stream>
__device__ __forceinline__ bool publish_tiles(CtaState<kSegs, kStages> &sh, const uint32_t lane, Stream &stream, const uint64_t wait_ns)
{
    const uint64_t tag = wait_tag(&sh.tag, &sh.abort, wait_ns);
    if (tag == 0) return false;
    for (uint32_t it = 0;; ++it) {
        const uint32_t q      = it % kQueue;
        uint32_t       number = LISTED ? 0u : stream.dealt(it);
        if (number == kNoTile) return true;
        if (!mbar_wait(&sh.counted[q], (it / kQueue) & 1u, &sh.abort, wait_ns)) return false;
        if constexpr (LISTED) number = sh.tile[it % kTiles];
        if (number == kNoTile) return true;
        const uint32_t count = __reduce_add_sync(kFull, lane < kSegs ? sh.cnt[q][lane] : 0u);
        if (lane == 0) {
            stream.publish(number, count, tag);
            mbar_arrive(&sh.ready[q]);             // (until then the counts of the tile's segments stay)
        }
    }
}

// The store warp of the forms with the dense output: sends every tile off from its slot, whole 16-byte units by ONE bulk
// copy, and hands the slot back.  Stored by the workers themselves, 4 KB here and 4 KB there, the same bytes are slower
// than in one piece (fp32 2^28 at half zeros 422 us against 418, fp32 2^25 without values 52.9 against 50.4, bf16
// [61,144,57,55] 31.6 against 30.5).  False if a wait ran out.
template <typename U, int kSegs, int kStages, typename Stream>
__device__ __forceinline__ bool store_dense(CtaState<kSegs, kStages> &sh, const U *tiles, const uint32_t lane, Stream &stream, const uint64_t wait_ns)
{
    constexpr uint32_t kTile = kSegs * Rows<U>::kSeg;
    TileIn t;
    for (uint32_t it = 0;; ++it) {
        const uint32_t s    = it % kStages;
        const U *const tile = tiles + static_cast<size_t>(s) * kTile;
        if (!mbar_wait(&sh.written[s], (it / kStages) & 1u, &sh.abort, wait_ns)) return false;
        const uint32_t number = sh.tile[it % kTiles];
        if (number == kNoTile) return true;
        stream.locate(number, t);
        const uint64_t left  = t.n - t.first;
        const uint32_t have  = left < kTile ? static_cast<uint32_t>(left) : kTile;
        const uint32_t whole = (have * static_cast<uint32_t>(sizeof(U))) & ~15u;
        U *const       y     = static_cast<U *>(t.y) + t.first;
        const Extent   yx    = extent_of(t.y, t.n * sizeof(U));
        if (lane == 0 && whole && yx.holds(y, whole)) {
            bulk_store(y, tile, whole);
            bulk_commit();
        }
        const uint32_t e = whole / static_cast<uint32_t>(sizeof(U)) + lane;       // behind the last whole unit
        if (e < have && yx.holds(y + e, sizeof(U))) y[e] = tile[e];
        __syncwarp();
        if (lane == 0) {
            bulk_wait_read<0>();
            mbar_arrive(&sh.empty[s]);
        }
    }
}

// Launch shape of one kernel instantiation on one device: the opt-in shared
// memory size is set and the number of co-resident CTAs is looked up once.
struct LaunchShape {
    std::mutex lock;
    int        grid_of_device[64] = {};
    template <typename Kernel>
    cudaError_t max_grid(Kernel kernel, int threads, size_t smem, int &grid)
    {
        int         dev = 0;
        cudaError_t e   = reported(cudaGetDevice(&dev));
        if (e != cudaSuccess) return e;
        if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
        std::lock_guard<std::mutex> g(lock);
        if (grid_of_device[dev] == 0) {
            e = reported(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem)));
            if (e != cudaSuccess) return e;
            int sms = 0, per_sm = 0;
            e = reported(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
            if (e != cudaSuccess) return e;
            e = reported(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, smem));
            if (e != cudaSuccess) return e;
            if (per_sm < 1 || sms < 1) return cudaErrorLaunchOutOfResources;
            grid_of_device[dev] = sms * per_sm;
        }
        grid = grid_of_device[dev];
        return cudaSuccess;
    }
};

// How a compressor of `tiles` tiles is launched.
//   No more tiles than CTAs that fit: a CTA per tile.  A CTA waits for the counts of lower CTAs alone; those are dispatched
//     first and retire without waiting for it (single-pass scans with look-back rest on that order as well; and the waits
//     are bounded), so a plain launch will do.
//   Stealing: a CTA per tile too, of which those that run take over the others' (load_tiles).  A plain launch, which takes the
//     device 2.2 us less than a cooperative one, and a slow SM takes fewer tiles.  With the dense output at every size
//     (f32 64 MiB 33.5 -> 30.2 us, 1 GiB 421 -> 416); without it up to `steal_waves` tiles per CTA: beyond, the CTAs no longer read
//     and write in step, which costs the DRAM more than the launch is worth.  Dealt out and stolen, half zeros, us:
//       f32 8 MiB 6.5 5.2, 64 21.3 20.2, 128 (28 waves) 37.1 36.1, 196 52.5 52.6 (2 % zeros 69.2 72.8), 256 65.8 66.3, 1 GiB 246 256;
//       f64 128 MiB 35.9 34.8, 256 64.5 64.6, 1 GiB 235 244;
//       bf16, whose kernel is bound by the SM before the DRAM, 128 MiB 42.1 38.5, 256 78.2 74.6, 384 (83 waves) 118.2 113.8 (2 % zeros
//       149.1 148.9), 768 226.7 223.1 (30 % zeros 263.9 268.7), 1 GiB 294 292;
//       batches, where a CTA looks for each tile's tensor: ResNet-18 f32 batch 16 (30 waves) 42.0 41.8, 32 73.9 77.5, bf16 batch 32
//       (30 waves) 44.8 45.5, 64 81.5 85.2.
//   Else, or under a limit on the CTAs that is in force: the tiles are dealt to CTAs that wait for one another and must be
//     resident together: a cooperative launch, or an error.
struct Deal {
    uint32_t grid, resident, stealing;
    bool     cooperative;
};
template <typename U>
constexpr uint32_t kStealWaves      = sizeof(U) == 2 ? 80 : 28;       // one tensor
constexpr uint32_t kBatchStealWaves = 20;
template <typename Kernel>
inline cudaError_t deal_of(const uint32_t tiles, const bool dense_output, const uint32_t steal_waves, Kernel dealt, Kernel listed, LaunchShape (&shapes)[2], const int threads,
                           const size_t smem, Deal &d)
{
    int         resident = 0;
    cudaError_t e        = shapes[0].max_grid(dealt, threads, smem, resident);
    if (e != cudaSuccess) return e;
    const uint32_t limit = compress_max_ctas(), all = static_cast<uint32_t>(resident) < kMaxGrid ? static_cast<uint32_t>(resident) : kMaxGrid;
    const bool     limited = limit != 0 && limit < all;
    d.resident = limited ? limit : all;
    d.stealing = !limited && tiles > all && tiles <= 0x7FFFFFFFu && (dense_output || tiles <= steal_waves * all);   // (a grid has fewer than 2^31 CTAs)
    d.grid     = d.stealing || tiles < d.resident ? tiles : d.resident;
    d.cooperative = tiles > d.grid;
    return d.stealing ? shapes[1].max_grid(listed, threads, smem, resident) : cudaSuccess;
}

}  // namespace cmp
}  // namespace bt
