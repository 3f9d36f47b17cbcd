// ReLU6 backward from the stash: grad_in[i] = (bit i set and the stashed
// activation is below 6) ? grad_out[i] : +0.  Unlike plain ReLU, the bitmap alone
// does not say whether a unit is saturated (its stashed value is 6), so the
// values are consulted: the staged walk of the restore (bt_staged_walk.cuh), one
// comparison per value, and a select on the gradient.
//
// Elements under a clear bit come out of the expansion as a NaN, so the one
// comparison "below 6" -- false for a stored 6 and for a NaN -- decides both
// conditions; 2-byte elements take it in their own type, two at a time.
#include <type_traits>

#include "bt_staged_walk.cuh"

namespace bt {
namespace {

// Two packed 2-byte values compared with 6 in their own type: 0xFFFF in the half of a value below 6, else 0 (a NaN
// is not below 6).
template <int DT>
__device__ __forceinline__ uint32_t below_six_mask(const uint32_t pair)
{
    uint32_t m;
    if constexpr (DT == BT_F16) asm("set.lt.u32.f16x2 %0, %1, %2;" : "=r"(m) : "r"(pair), "r"(0x46004600u));
    else asm("set.lt.u32.bf16x2 %0, %1, %2;" : "=r"(m) : "r"(pair), "r"(0x40C040C0u));
    return m;
}

template <int DT>
constexpr uint32_t kNanFill = DT == BT_F32 || DT == BT_F64 ? 0x7FFFFFFFu : 0x7FFFu;

// The lane's gradient g under its stashed values v.
template <int DT>
__device__ __forceinline__ uint2 passed(const uint2 g, const uint2 v)
{
    return make_uint2(g.x & below_six_mask<DT>(v.x), g.y & below_six_mask<DT>(v.y));
}
template <int DT>
__device__ __forceinline__ uint4 passed(const uint4 g, const uint4 v)
{
    if constexpr (DT == BT_F32) {
        return make_uint4(__uint_as_float(v.x) < 6.0f ? g.x : 0u, __uint_as_float(v.y) < 6.0f ? g.y : 0u, __uint_as_float(v.z) < 6.0f ? g.z : 0u,
                          __uint_as_float(v.w) < 6.0f ? g.w : 0u);
    } else {
        const bool a = __hiloint2double(static_cast<int>(v.y), static_cast<int>(v.x)) < 6.0;
        const bool b = __hiloint2double(static_cast<int>(v.w), static_cast<int>(v.z)) < 6.0;
        return make_uint4(a ? g.x : 0u, a ? g.y : 0u, b ? g.z : 0u, b ? g.w : 0u);
    }
}

constexpr int kWarps = 4;   // warps per CTA

// The gradient does not depend on the stash: that of the first kAhead steps (an 8- or 16-byte load per lane and step) is
// requested before the run is staged, that of a later step when the step kAhead before it has used its registers.
template <typename U, int DT, int kAhead, int kCtas>
__global__ void __launch_bounds__(kWarps * 32, kCtas)
relu6_bwd_kernel(const uint32_t *__restrict__ bitmap, const U *__restrict__ values, const uint64_t *__restrict__ values_offset,
                 const uint64_t *__restrict__ prefix, const U *gout, const uint64_t n, U *gin)   // gin may alias gout
{
    using P            = walk::Of<U>;
    using V            = std::conditional_t<sizeof(U) == 2, uint2, uint4>;       // a lane's elements of a step
    constexpr int kPer = P::kPerLane;
    in_stream_order();
    const uint32_t lane = threadIdx.x & 31u;
    const uint64_t e0   = (static_cast<uint64_t>(blockIdx.x) * kWarps + (threadIdx.x >> 5)) * P::kElems;
    if (e0 >= n) return;
    const bool     whole = e0 + P::kElems <= n;
    const U *const from  = gout + e0 + lane * kPer;
    auto gradient = [&](const int k) {
        if (whole) return *reinterpret_cast<const V *>(from + k * 32 * kPer);
        const uint64_t at = e0 + static_cast<uint64_t>(k) * (32 * kPer) + lane * kPer;
        if (at + kPer <= n) return *reinterpret_cast<const V *>(gout + at);
        V g{};
        U h[kPer];
#pragma unroll
        for (int j = 0; j < kPer; ++j) h[j] = at + j < n ? gout[at + j] : U(0);
        if constexpr (sizeof(U) == 2) g = make_uint2(h[0] | (uint32_t(h[1]) << 16), h[2] | (uint32_t(h[3]) << 16));
        else if constexpr (sizeof(U) == 4) g = make_uint4(h[0], h[1], h[2], h[3]);
        else g = make_uint4(static_cast<uint32_t>(h[0]), static_cast<uint32_t>(h[0] >> 32), static_cast<uint32_t>(h[1]), static_cast<uint32_t>(h[1] >> 32));
        return g;
    };
    V g[kAhead];
#pragma unroll
    for (int k = 0; k < kAhead; ++k) g[k] = gradient(k);
    walk::Part pt;
    if (!walk::stage_part<U, kWarps>(bitmap, values, values_offset, prefix, n, blockIdx.x, pt)) return;
    const Extent ox = extent_of(gin, n * sizeof(U));
    U *const     to = gin + e0 + lane * kPer;
#pragma unroll
    for (int k = 0; k < P::kSteps; ++k) {
        const V r = passed<DT>(g[k % kAhead], walk::expand_step<U, kNanFill<DT>>(pt, k, lane));
        if (k + kAhead < P::kSteps) g[k % kAhead] = gradient(k + kAhead);
        if (whole) {
            if (ox.holds(to + k * 32 * kPer, sizeof(V))) *reinterpret_cast<V *>(to + k * 32 * kPer) = r;
        } else {
            const uint64_t at = e0 + static_cast<uint64_t>(k) * (32 * kPer) + lane * kPer;
            const U *const e  = reinterpret_cast<const U *>(&r);
#pragma unroll
            for (int j = 0; j < kPer; ++j)
                if (at + j < n && ox.holds(gin + at + j, sizeof(U))) gin[at + j] = e[j];
        }
    }
}

template <typename U, int DT, int kAhead, int kCtas>
cudaError_t launch_typed(const uint32_t *bitmap, const void *values, const uint64_t *values_offset, const uint64_t *prefix,
                         const void *gout, uint64_t n, void *gin, cudaStream_t stream)
{
    const uint64_t grid = walk::Of<U>::blocks_of(n, kWarps);
    if (grid > 0x7FFFFFFFull) return cudaErrorInvalidValue;
    return launch(relu6_bwd_kernel<U, DT, kAhead, kCtas>, static_cast<unsigned>(grid), kWarps * 32, 0, stream, bitmap,
                  static_cast<const U *>(values), values_offset, prefix, static_cast<const U *>(gout), n, static_cast<U *>(gin));
}

}  // namespace

cudaError_t launch_relu6_bwd(const uint32_t *bitmap, const void *values, const uint64_t *values_offset,
                             const uint64_t *prefix, const void *gout, uint64_t n, int dtype, void *gin,
                             cudaStream_t stream)
{
    // 64 bytes of gradient ahead per lane: 8 steps of 2-byte elements on 10 CTAs per SM ([61,144,57,55] bf16: 23.5 us; 4
    // steps on 11 CTAs 27.1, 12 on 8 23.2, 16 on 8 23.8), 4 steps of wider ones on 8 (fp32 2^27: 197.8 us; 8 steps on 10
    // CTAs 205.6, 2 on 12 204.4).  Gathered from global memory the two took 28.8 and 217.7 us.
    switch (dtype) {
    case BT_F64: return launch_typed<uint64_t, BT_F64, 4, 8>(bitmap, values, values_offset, prefix, gout, n, gin, stream);
    case BT_F32: return launch_typed<uint32_t, BT_F32, 4, 8>(bitmap, values, values_offset, prefix, gout, n, gin, stream);
    case BT_F16: return launch_typed<uint16_t, BT_F16, 8, 10>(bitmap, values, values_offset, prefix, gout, n, gin, stream);
    default: return launch_typed<uint16_t, BT_BF16, 8, 10>(bitmap, values, values_offset, prefix, gout, n, gin, stream);
    }
}

}  // namespace bt
