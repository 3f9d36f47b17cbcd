// 2x2 / stride 2 max pooling with winner codes, and its backward pass from the codes.
//
// The tensor is planes x height x width elements, row-major, height and width even, so the two input rows of
// an output row are adjacent in memory and output row R (counted across all planes) reads input rows 2R and
// 2R + 1.  The framework's comparison rule on the exactly widened values: a later window element replaces the
// maximum when it is greater or when it is a NaN; a 2-bit code keeps the winner's position (2*dy + dx), and
// neighbouring lanes merge their codes into words with a few shuffles.  The backward pass reads a gradient and a
// code per output and writes the four window positions: the gradient where the code points, +0 elsewhere.
//
// Three forms of each pass, by what the rows allow: rows that hold whole 16-byte vectors of window pairs (width a
// multiple of 8 for 2-byte, of 4 for 4-byte elements) take 8 bytes of outputs per group and two groups per thread;
// other rows of 2-byte elements two outputs per thread, which need not be in one row; the rest one.
//
// With the codes kept, neither the pooling layer's input nor an index tensor is needed for its backward pass:
// 2 bits per output instead of 8 bytes per output plus the saved input.
#include "bt_internal.cuh"

namespace bt {
namespace {

constexpr uint32_t kFull    = 0xFFFFFFFFu;
constexpr int      kThreads = 256;

// a pair of adjacent elements as one register-sized load / store
template <typename U>
struct Pair;
template <>
struct Pair<uint32_t> {
    using T = uint2;
    __device__ static uint32_t lo(T p) { return p.x; }
    __device__ static uint32_t hi(T p) { return p.y; }
    __device__ static T make(uint32_t a, uint32_t b) { return make_uint2(a, b); }
};
template <>
struct Pair<uint64_t> {
    using T = ulonglong2;
    __device__ static uint64_t lo(T p) { return p.x; }
    __device__ static uint64_t hi(T p) { return p.y; }
    __device__ static T make(uint64_t a, uint64_t b) { return make_ulonglong2(a, b); }
};

// Two windows of 2-byte elements at once: A, B, C, D hold the two windows' elements (0,0), (0,1), (1,0), (1,1), one
// window per half.  The comparison rule on packed pairs in the element's own type (an exact widening changes no
// comparison); `code` receives the winner's position per half.
template <int DT>
__device__ __forceinline__ uint32_t later_wins(const uint32_t v, const uint32_t best)
{
    uint32_t gt, nan;
    if constexpr (DT == BT_F16) {
        asm("set.gt.u32.f16x2 %0, %1, %2;" : "=r"(gt) : "r"(v), "r"(best));
        asm("set.nan.u32.f16x2 %0, %1, %1;" : "=r"(nan) : "r"(v));
    } else {
        asm("set.gt.u32.bf16x2 %0, %1, %2;" : "=r"(gt) : "r"(v), "r"(best));
        asm("set.nan.u32.bf16x2 %0, %1, %1;" : "=r"(nan) : "r"(v));
    }
    return gt | nan;                                        // 0xFFFF in the half of a window where v replaces the maximum
}
template <int DT>
__device__ __forceinline__ uint32_t pool_pair(const uint32_t a, const uint32_t b, const uint32_t c, const uint32_t d, uint32_t &code)
{
    uint32_t m = later_wins<DT>(b, a), best = (b & m) | (a & ~m);
    code       = 0x00010001u & m;
    m          = later_wins<DT>(c, best), best = (c & m) | (best & ~m);
    code       = (0x00020002u & m) | (code & ~m);
    m          = later_wins<DT>(d, best), best = (d & m) | (best & ~m);
    code       = (0x00030003u & m) | (code & ~m);
    return best;
}

// g / d for g < 2^31 by one multiplication (d >= 1): floor(g (2^32 + m) / 2^(32 + s)) with s = ceil(log2 d) and
// m = floor(2^32 (2^s - d) / d) + 1 is exact (Granlund and Montgomery, Division by invariant integers).
struct DivBy {
    uint32_t m, s;
    static DivBy of(const uint32_t d)
    {
        uint32_t s = 0;
        while ((1ull << s) < d) ++s;
        return DivBy{static_cast<uint32_t>((((1ull << s) - d) << 32) / d + 1), s};
    }
    __device__ __forceinline__ uint32_t operator()(const uint32_t g) const { return (__umulhi(g, m) + g) >> s; }
};
// rows of more than 2^31 groups in all: the plain division
struct DivWide {
    uint64_t d;
    __device__ __forceinline__ uint64_t operator()(const uint64_t g) const { return g / d; }
};

// One output per thread.  I: uint32_t while every element index fits 32 bits, else uint64_t (Div likewise)
template <typename U, int DT, typename I, typename Div>
__global__ void __launch_bounds__(kThreads)
maxpool2x2_fwd_kernel(const U *__restrict__ x, const uint64_t outputs, const Div row_of, const I wo, const I width, U *__restrict__ y,
                      uint32_t *__restrict__ codes)
{
    in_stream_order();
    using P             = Pair<U>;
    const uint32_t lane = threadIdx.x & 31u;
    const uint64_t o64  = static_cast<uint64_t>(blockIdx.x) * kThreads + threadIdx.x;
    const bool     live = o64 < outputs;
    uint32_t       code = 0;
    if (live) {
        const I        o   = static_cast<I>(o64);
        const I        row = row_of(o);                    // output row, counted across the planes
        const I        col = o - row * wo;
        const uint64_t at  = 2ull * row * width + 2ull * col;
        const typename P::T top = *reinterpret_cast<const typename P::T *>(x + at);
        const typename P::T bot = *reinterpret_cast<const typename P::T *>(x + at + width);
        const U e[4] = {P::lo(top), P::hi(top), P::lo(bot), P::hi(bot)};
        U    best  = e[0];
        auto bestv = Elem<DT>::widen(e[0]);
#pragma unroll
        for (uint32_t k = 1; k < 4; ++k) {
            const auto v    = Elem<DT>::widen(e[k]);
            const bool take = greater_or_nan(v, bestv) != 0;
            best            = take ? e[k] : best;
            bestv           = take ? v : bestv;
            code            = take ? k : code;
        }
        if (extent_of(y, outputs * sizeof(U)).holds(y + o64, sizeof(U))) y[o64] = best;
    }
    if (codes) {
        uint32_t word = code << (2u * (lane & 15u));
#pragma unroll
        for (int d = 8; d > 0; d >>= 1) word |= __shfl_xor_sync(kFull, word, d);
        if (live && (lane & 15u) == 0 && extent_of(codes, 4 * ((outputs + 15) >> 4)).holds(codes + (o64 >> 4), 4)) codes[o64 >> 4] = word;
    }
}

template <typename U, typename I, typename Div>
__global__ void __launch_bounds__(kThreads)
maxpool2x2_bwd_kernel(const uint32_t *__restrict__ codes, const uint32_t *__restrict__ mask, const U *__restrict__ gout,
                      const uint64_t outputs, const Div row_of, const I wo, const I width, U *__restrict__ gin)
{
    in_stream_order();
    // mask (may be NULL): bitmap over the outputs; the gradient of an output whose bit is clear counts as +0
    using P            = Pair<U>;
    const uint64_t o64 = static_cast<uint64_t>(blockIdx.x) * kThreads + threadIdx.x;
    if (o64 >= outputs) return;
    const I        o    = static_cast<I>(o64);
    const I        row  = row_of(o);
    const I        col  = o - row * wo;
    const uint64_t at   = 2ull * row * width + 2ull * col;
    const uint32_t k    = (codes[o64 >> 4] >> (2u * (static_cast<uint32_t>(o64) & 15u))) & 3u;
    U              g    = gout[o64];
    if (mask != nullptr && ((mask[o64 >> 5] >> (static_cast<uint32_t>(o64) & 31u)) & 1u) == 0) g = U(0);
    const Extent gx = extent_of(gin, 4 * outputs * sizeof(U));
    if (gx.holds(gin + at, 2 * sizeof(U))) *reinterpret_cast<typename P::T *>(gin + at) = P::make(k == 0 ? g : U(0), k == 1 ? g : U(0));
    if (gx.holds(gin + at + width, 2 * sizeof(U)))
        *reinterpret_cast<typename P::T *>(gin + at + width) = P::make(k == 2 ? g : U(0), k == 3 ? g : U(0));
}

// 0xFFFF or 0xFFFF0000 where the 2-bit code in bits 4 and 5 of s (all others clear) names that element of a pair of
// codes 0 and 1, else 0: shifts past the register give 0.
__device__ __forceinline__ uint32_t pair_mask(const uint32_t s)
{
    uint32_t m;
    asm("shl.b32 %0, %1, %2;" : "=r"(m) : "r"(0x0000FFFFu), "r"(s));
    return m;
}

// ---------------------------------------------------------------------------------------------
// Two outputs o, o + 1 (o even) of a tensor of 2-byte elements per thread.  kEven: rows of an even number of outputs, so
// the two are neighbours in one row and their windows one 8-byte access per input row; else they may lie in different rows.
struct TwoOutputs {
    uint64_t first, second;    // element indices of their windows
};
template <typename I, typename Div>
__device__ __forceinline__ TwoOutputs windows_of(const I o, const Div row_of, const I wo, const I width)
{
    const I        row = row_of(o), col = o - row * wo;
    const uint64_t at  = 2ull * row * width + 2ull * col;
    return TwoOutputs{at, col + 1 == wo ? 2ull * (row + 1) * width : at + 2};
}

template <int DT, bool kEven, typename I, typename Div>
__global__ void __launch_bounds__(kThreads)
maxpool2x2_fwd_pair_kernel(const uint16_t *__restrict__ x, const uint64_t outputs, const Div row_of, const I wo, const I width,
                           uint16_t *__restrict__ y, uint32_t *__restrict__ codes)
{
    in_stream_order();
    const uint32_t lane = threadIdx.x & 31u;
    const uint64_t o    = 2 * (static_cast<uint64_t>(blockIdx.x) * kThreads + threadIdx.x);
    uint32_t       bits = 0;
    if (o < outputs) {
        const TwoOutputs w    = windows_of<I>(static_cast<I>(o), row_of, wo, width);
        const bool       both = kEven || o + 1 < outputs;
        uint32_t         t0, t1, b0, b1;
        if constexpr (kEven) {
            const uint2 top = *reinterpret_cast<const uint2 *>(x + w.first), bot = *reinterpret_cast<const uint2 *>(x + w.first + width);
            t0 = top.x, t1 = top.y, b0 = bot.x, b1 = bot.y;
        } else {
            auto pair = [&](const uint64_t at) { return *reinterpret_cast<const uint32_t *>(x + at); };
            t0 = pair(w.first), b0 = pair(w.first + width);
            t1 = both ? pair(w.second) : 0u, b1 = both ? pair(w.second + width) : 0u;
        }
        uint32_t       code;
        const uint32_t best = pool_pair<DT>(__byte_perm(t0, t1, 0x5410), __byte_perm(t0, t1, 0x7632), __byte_perm(b0, b1, 0x5410),
                                            __byte_perm(b0, b1, 0x7632), code);
        bits = __dp4a(code, both ? 0x00040001u : 1u, 0u);
        const Extent yx = extent_of(y, outputs * 2);
        if (both) {
            if (yx.holds(y + o, 4)) *reinterpret_cast<uint32_t *>(y + o) = best;
        } else if (yx.holds(y + o, 2)) {
            y[o] = static_cast<uint16_t>(best);
        }
    }
    if (codes) {
        uint32_t word = bits << (4u * (lane & 7u));
#pragma unroll
        for (int d = 4; d > 0; d >>= 1) word |= __shfl_xor_sync(kFull, word, d);
        if (o < outputs && (lane & 7u) == 0 && extent_of(codes, 4 * ((outputs + 15) >> 4)).holds(codes + (o >> 4), 4)) codes[o >> 4] = word;
    }
}

template <bool kEven, typename I, typename Div>
__global__ void __launch_bounds__(kThreads)
maxpool2x2_bwd_pair_kernel(const uint32_t *__restrict__ codes, const uint32_t *__restrict__ mask, const uint16_t *__restrict__ gout,
                           const uint64_t outputs, const Div row_of, const I wo, const I width, uint16_t *__restrict__ gin)
{
    in_stream_order();
    const uint64_t o = 2 * (static_cast<uint64_t>(blockIdx.x) * kThreads + threadIdx.x);
    if (o >= outputs) return;
    const TwoOutputs w    = windows_of<I>(static_cast<I>(o), row_of, wo, width);
    const bool       both = kEven || o + 1 < outputs;
    const uint32_t   bits = codes[o >> 4] >> (2u * (static_cast<uint32_t>(o) & 15u));
    const uint32_t   live = mask != nullptr ? mask[o >> 5] >> (static_cast<uint32_t>(o) & 31u) : 0xFFFFFFFFu;
    const uint32_t   g    = both ? *reinterpret_cast<const uint32_t *>(gout + o) : gout[o];
    const uint32_t   s0 = (bits << 4) & 0x30u, s1 = (bits << 2) & 0x30u;
    const uint32_t   g0 = live & 1u ? __byte_perm(g, 0, 0x1010) : 0u, g1 = live & 2u ? __byte_perm(g, 0, 0x3232) : 0u;
    const Extent     gx = extent_of(gin, 4 * outputs * 2);
    if constexpr (kEven) {
        auto put = [&](const uint64_t at, const uint32_t v0, const uint32_t v1) {
            if (gx.holds(gin + at, 8)) *reinterpret_cast<uint2 *>(gin + at) = make_uint2(v0, v1);
        };
        put(w.first, g0 & pair_mask(s0), g1 & pair_mask(s1));
        put(w.first + width, g0 & pair_mask(s0 ^ 0x20u), g1 & pair_mask(s1 ^ 0x20u));
    } else {
        auto put = [&](const uint64_t at, const uint32_t v) {
            if (gx.holds(gin + at, 4)) *reinterpret_cast<uint32_t *>(gin + at) = v;
        };
        put(w.first, g0 & pair_mask(s0));
        put(w.first + width, g0 & pair_mask(s0 ^ 0x20u));
        if (both) {
            put(w.second, g1 & pair_mask(s1));
            put(w.second + width, g1 & pair_mask(s1 ^ 0x20u));
        }
    }
}

// ---------------------------------------------------------------------------------------------
// Rows of whole vectors: a group is kOut adjacent outputs, i.e. one 16-byte load per input row, one 8-byte store of the
// winners and 2 * kOut code bits; 16 / kOut consecutive lanes share a code word.  Group g starts at element
// 2 * kOut * g + row * width of the input: the rows of outputs in front of it cover two input rows each, and a row of
// groups covers one.  A thread takes kGroups groups, kThreads apart, all of their loads first.
constexpr int kGroups = 2;

template <typename U, int DT, typename I, typename Div>
__global__ void __launch_bounds__(kThreads)
maxpool2x2_fwd_vec_kernel(const U *__restrict__ x, const uint64_t groups, const Div row_of, const I width,
                          U *__restrict__ y, uint32_t *__restrict__ codes)
{
    in_stream_order();
    constexpr int      kOut          = 8 / sizeof(U);          // outputs per group
    constexpr uint32_t kLanesPerWord = 16 / kOut;
    const uint32_t     lane          = threadIdx.x & 31u;
    const uint64_t     g0            = static_cast<uint64_t>(blockIdx.x) * (kThreads * kGroups) + threadIdx.x;
    uint4              top[kGroups], bot[kGroups];
#pragma unroll
    for (int u = 0; u < kGroups; ++u) {
        const uint64_t g64 = g0 + u * kThreads;
        if (g64 < groups) {
            const I        row = row_of(static_cast<I>(g64));
            const uint64_t at  = 2ull * kOut * g64 + static_cast<uint64_t>(row) * width;
            top[u] = *reinterpret_cast<const uint4 *>(x + at), bot[u] = *reinterpret_cast<const uint4 *>(x + at + width);
        }
    }
#pragma unroll
    for (int u = 0; u < kGroups; ++u) {
        const uint64_t g64  = g0 + u * kThreads;
        const bool     live = g64 < groups;
        uint32_t       bits = 0;
        if (live) {
            uint2 pack;
            if constexpr (sizeof(U) == 2) {
                const uint4 &p = top[u], &q = bot[u];
                uint32_t     c0, c1;
                pack.x = pool_pair<DT>(__byte_perm(p.x, p.y, 0x5410), __byte_perm(p.x, p.y, 0x7632), __byte_perm(q.x, q.y, 0x5410),
                                       __byte_perm(q.x, q.y, 0x7632), c0);
                pack.y = pool_pair<DT>(__byte_perm(p.z, p.w, 0x5410), __byte_perm(p.z, p.w, 0x7632), __byte_perm(q.z, q.w, 0x5410),
                                       __byte_perm(q.z, q.w, 0x7632), c1);
                bits = __dp4a(c0, 0x00040001u, __dp4a(c1, 0x00400010u, 0u));
            } else {
                const U t[4] = {top[u].x, top[u].y, top[u].z, top[u].w}, b[4] = {bot[u].x, bot[u].y, bot[u].z, bot[u].w};
                U       win[kOut];
#pragma unroll
                for (int j = 0; j < kOut; ++j) {
                    const U  e[4]  = {t[2 * j], t[2 * j + 1], b[2 * j], b[2 * j + 1]};
                    U        best  = e[0];
                    auto     bestv = Elem<DT>::widen(e[0]);
                    uint32_t code  = 0;
#pragma unroll
                    for (uint32_t k = 1; k < 4; ++k) {
                        const auto v    = Elem<DT>::widen(e[k]);
                        const bool take = greater_or_nan(v, bestv) != 0;
                        best            = take ? e[k] : best;
                        bestv           = take ? v : bestv;
                        code            = take ? k : code;
                    }
                    win[j] = best;
                    bits |= code << (2 * j);
                }
                pack = make_uint2(win[0], win[1]);
            }
            if (extent_of(y, groups * kOut * sizeof(U)).holds(y + g64 * kOut, 8)) *reinterpret_cast<uint2 *>(y + g64 * kOut) = pack;
        }
        if (codes) {
            uint32_t word = bits << (2u * kOut * (lane % kLanesPerWord));
#pragma unroll
            for (int d = kLanesPerWord / 2; d > 0; d >>= 1) word |= __shfl_xor_sync(kFull, word, d);
            if (live && (lane % kLanesPerWord) == 0 && extent_of(codes, 4 * ((groups * kOut + 15) >> 4)).holds(codes + ((g64 * kOut) >> 4), 4))
                codes[(g64 * kOut) >> 4] = word;
        }
    }
}

template <typename U, typename I, typename Div>
__global__ void __launch_bounds__(kThreads)
maxpool2x2_bwd_vec_kernel(const uint32_t *__restrict__ codes, const uint32_t *__restrict__ mask, const U *__restrict__ gout,
                          const uint64_t groups, const Div row_of, const I width, U *__restrict__ gin)
{
    in_stream_order();
    constexpr int  kOut = 8 / sizeof(U);
    const uint64_t g0   = static_cast<uint64_t>(blockIdx.x) * (kThreads * kGroups) + threadIdx.x;
    const Extent   gx   = extent_of(gin, 4 * groups * kOut * sizeof(U));
    uint32_t       bits[kGroups], live[kGroups];
    uint2          gv[kGroups];
#pragma unroll
    for (int u = 0; u < kGroups; ++u) {
        const uint64_t g64 = g0 + u * kThreads, o0 = g64 * kOut;
        if (g64 < groups) {
            bits[u] = codes[o0 >> 4];
            // the kOut mask bits of this group's outputs sit in one word (kOut divides 32)
            live[u] = mask != nullptr ? mask[o0 >> 5] : 0xFFFFFFFFu;
            gv[u]   = *reinterpret_cast<const uint2 *>(gout + o0);
        }
    }
#pragma unroll
    for (int u = 0; u < kGroups; ++u) {
        const uint64_t g64 = g0 + u * kThreads, o0 = g64 * kOut;
        if (g64 >= groups) return;
        const I        row = row_of(static_cast<I>(g64));
        const uint64_t at  = 2ull * kOut * g64 + static_cast<uint64_t>(row) * width;
        const uint32_t b = bits[u] >> (2u * (static_cast<uint32_t>(o0) & 15u)), l = live[u] >> (static_cast<uint32_t>(o0) & 31u);
        uint4          top, bot;
        if constexpr (sizeof(U) == 2) {
            // an output's gradient in both halves of a word, +0 where its bit is clear; the code's mask picks one half of
            // the top or of the bottom pair (code ^ 2 puts the bottom codes where the top ones are)
            const uint32_t g[4] = {__byte_perm(gv[u].x, 0, 0x1010), __byte_perm(gv[u].x, 0, 0x3232), __byte_perm(gv[u].y, 0, 0x1010),
                                   __byte_perm(gv[u].y, 0, 0x3232)};
            uint32_t       tp[4], bp[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const uint32_t s = j < 2 ? (b << (4 - 2 * j)) & 0x30u : (b >> (2 * j - 4)) & 0x30u;
                const uint32_t v = (l >> j) & 1u ? g[j] : 0u;
                tp[j] = v & pair_mask(s), bp[j] = v & pair_mask(s ^ 0x20u);
            }
            top = make_uint4(tp[0], tp[1], tp[2], tp[3]), bot = make_uint4(bp[0], bp[1], bp[2], bp[3]);
        } else {
            U gr[2] = {gv[u].x, gv[u].y}, t[4], c[4];
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                const uint32_t k = (b >> (2 * j)) & 3u;
                gr[j]            = (l >> j) & 1u ? gr[j] : U(0);
                t[2 * j]         = k == 0 ? gr[j] : U(0);
                t[2 * j + 1]     = k == 1 ? gr[j] : U(0);
                c[2 * j]         = k == 2 ? gr[j] : U(0);
                c[2 * j + 1]     = k == 3 ? gr[j] : U(0);
            }
            top = make_uint4(t[0], t[1], t[2], t[3]), bot = make_uint4(c[0], c[1], c[2], c[3]);
        }
        if (gx.holds(gin + at, 16)) *reinterpret_cast<uint4 *>(gin + at) = top;
        if (gx.holds(gin + at + width, 16)) *reinterpret_cast<uint4 *>(gin + at + width) = bot;
    }
}

// CTAs for `items` threads' worth of work
inline bool grid_of(const uint64_t items, const uint64_t per_block, unsigned &grid)
{
    const uint64_t g = (items + per_block - 1) / per_block;
    grid             = static_cast<unsigned>(g);
    return g <= 0x7FFFFFFFull;
}

template <typename U, int DT>
cudaError_t fwd_typed(const void *vx, uint64_t outputs, uint64_t wo, uint64_t width, uint64_t elements, void *vy, uint32_t *codes,
                      cudaStream_t s)
{
    const U *const x      = static_cast<const U *>(vx);
    U *const       y      = static_cast<U *>(vy);
    const bool     narrow = elements <= 0xFFFFFFFFull;         // every index in 32 bits
    const uint32_t w32 = static_cast<uint32_t>(width), wo32 = static_cast<uint32_t>(wo);
    unsigned       grid;
    if constexpr (sizeof(U) <= 4) {
        constexpr uint64_t kOut = 8 / sizeof(U);
        if (width % (2 * kOut) == 0) {
            const uint64_t groups = outputs / kOut, per_row = wo / kOut;
            if (!grid_of(groups, kThreads * kGroups, grid)) return cudaErrorInvalidValue;
            return narrow ? launch(maxpool2x2_fwd_vec_kernel<U, DT, uint32_t, DivBy>, grid, kThreads, 0, s, x, groups,
                                   DivBy::of(static_cast<uint32_t>(per_row)), w32, y, codes)
                          : launch(maxpool2x2_fwd_vec_kernel<U, DT, uint64_t, DivWide>, grid, kThreads, 0, s, x, groups, DivWide{per_row},
                                   width, y, codes);
        }
    }
    if constexpr (sizeof(U) == 2) {
        if (!grid_of((outputs + 1) / 2, kThreads, grid)) return cudaErrorInvalidValue;
        if (!narrow) return launch(maxpool2x2_fwd_pair_kernel<DT, false, uint64_t, DivWide>, grid, kThreads, 0, s, x, outputs, DivWide{wo}, wo, width, y, codes);
        return wo % 2 == 0 ? launch(maxpool2x2_fwd_pair_kernel<DT, true, uint32_t, DivBy>, grid, kThreads, 0, s, x, outputs, DivBy::of(wo32), wo32, w32, y, codes)
                           : launch(maxpool2x2_fwd_pair_kernel<DT, false, uint32_t, DivBy>, grid, kThreads, 0, s, x, outputs, DivBy::of(wo32), wo32, w32, y, codes);
    } else {
        if (!grid_of(outputs, kThreads, grid)) return cudaErrorInvalidValue;
        return narrow ? launch(maxpool2x2_fwd_kernel<U, DT, uint32_t, DivBy>, grid, kThreads, 0, s, x, outputs, DivBy::of(wo32), wo32, w32, y, codes)
                      : launch(maxpool2x2_fwd_kernel<U, DT, uint64_t, DivWide>, grid, kThreads, 0, s, x, outputs, DivWide{wo}, wo, width, y, codes);
    }
}

template <typename U>
cudaError_t bwd_typed(const uint32_t *codes, const uint32_t *mask, const void *vg, uint64_t outputs, uint64_t wo,
                      uint64_t width, uint64_t elements, void *vi, cudaStream_t s)
{
    const U *const gout   = static_cast<const U *>(vg);
    U *const       gin    = static_cast<U *>(vi);
    const bool     narrow = elements <= 0xFFFFFFFFull;
    const uint32_t w32 = static_cast<uint32_t>(width), wo32 = static_cast<uint32_t>(wo);
    unsigned       grid;
    if constexpr (sizeof(U) <= 4) {
        constexpr uint64_t kOut = 8 / sizeof(U);
        if (width % (2 * kOut) == 0) {
            const uint64_t groups = outputs / kOut, per_row = wo / kOut;
            if (!grid_of(groups, kThreads * kGroups, grid)) return cudaErrorInvalidValue;
            return narrow ? launch(maxpool2x2_bwd_vec_kernel<U, uint32_t, DivBy>, grid, kThreads, 0, s, codes, mask, gout, groups,
                                   DivBy::of(static_cast<uint32_t>(per_row)), w32, gin)
                          : launch(maxpool2x2_bwd_vec_kernel<U, uint64_t, DivWide>, grid, kThreads, 0, s, codes, mask, gout, groups,
                                   DivWide{per_row}, width, gin);
        }
    }
    if constexpr (sizeof(U) == 2) {
        if (!grid_of((outputs + 1) / 2, kThreads, grid)) return cudaErrorInvalidValue;
        if (!narrow) return launch(maxpool2x2_bwd_pair_kernel<false, uint64_t, DivWide>, grid, kThreads, 0, s, codes, mask, gout, outputs, DivWide{wo}, wo, width, gin);
        return wo % 2 == 0 ? launch(maxpool2x2_bwd_pair_kernel<true, uint32_t, DivBy>, grid, kThreads, 0, s, codes, mask, gout, outputs, DivBy::of(wo32), wo32, w32, gin)
                           : launch(maxpool2x2_bwd_pair_kernel<false, uint32_t, DivBy>, grid, kThreads, 0, s, codes, mask, gout, outputs, DivBy::of(wo32), wo32, w32, gin);
    } else {
        if (!grid_of(outputs, kThreads, grid)) return cudaErrorInvalidValue;
        return narrow ? launch(maxpool2x2_bwd_kernel<U, uint32_t, DivBy>, grid, kThreads, 0, s, codes, mask, gout, outputs, DivBy::of(wo32), wo32, w32, gin)
                      : launch(maxpool2x2_bwd_kernel<U, uint64_t, DivWide>, grid, kThreads, 0, s, codes, mask, gout, outputs, DivWide{wo}, wo, width, gin);
    }
}

}  // namespace

cudaError_t launch_maxpool2x2_fwd(const void *x, uint64_t planes, uint64_t height, uint64_t width, int dtype, void *y,
                                  uint32_t *codes, cudaStream_t s)
{
    const uint64_t wo = width / 2, outputs = planes * (height / 2) * wo, elements = planes * height * width;
    switch (dtype) {
    case BT_F64: return fwd_typed<uint64_t, BT_F64>(x, outputs, wo, width, elements, y, codes, s);
    case BT_F32: return fwd_typed<uint32_t, BT_F32>(x, outputs, wo, width, elements, y, codes, s);
    case BT_F16: return fwd_typed<uint16_t, BT_F16>(x, outputs, wo, width, elements, y, codes, s);
    default: return fwd_typed<uint16_t, BT_BF16>(x, outputs, wo, width, elements, y, codes, s);
    }
}

cudaError_t launch_maxpool2x2_bwd(const uint32_t *codes, const uint32_t *mask, const void *gout, uint64_t planes,
                                  uint64_t height, uint64_t width, int elem_size, void *gin, cudaStream_t s)
{
    const uint64_t wo = width / 2, outputs = planes * (height / 2) * wo, elements = planes * height * width;
    if (elem_size == 8) return bwd_typed<uint64_t>(codes, mask, gout, outputs, wo, width, elements, gin, s);
    return elem_size == 4 ? bwd_typed<uint32_t>(codes, mask, gout, outputs, wo, width, elements, gin, s)
                          : bwd_typed<uint16_t>(codes, mask, gout, outputs, wo, width, elements, gin, s);
}

}  // namespace bt
