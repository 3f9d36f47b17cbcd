// Algorithm 2 (bitmap -> dense), chunk-parallel.  The single running counter j
// of the algorithm is replaced by chunk_prefix[c] plus popcounts inside the
// chunk, so every warp decodes its part of a chunk without talking to any other
// (bt_staged_walk.cuh): it stages the part's packed run in shared memory, ranks
// the part's words and expands it with 8- or 16-byte stores, a lane owning a few
// consecutive elements per step.
#include <type_traits>

#include "bt_internal.cuh"
#include "bt_staged_walk.cuh"

namespace bt {
namespace {

// WIDEN: 0, or the 16-bit type of the stashed values of a binary32 tensor (1 binary16, 2 bfloat16): the value
// is widened exactly on its way out (the restore side of the down-cast on stash).
template <int WIDEN>
__device__ __forceinline__ uint32_t widened(const uint16_t h)
{
    if constexpr (WIDEN == 1) {
        // exponent and mantissa moved into place, then rebiased by an exact multiplication (subnormals included);
        // infinities and NaNs get the all-ones exponent by hand, which keeps a NaN payload and sign
        const uint32_t t = static_cast<uint32_t>(h & 0x7FFFu) << 13;
        uint32_t       r = __float_as_uint(__uint_as_float(t) * 5.192296858534828e33f);      // 2^112
        r                = (h & 0x7C00u) == 0x7C00u ? (t | 0x7F800000u) : r;
        return r | (static_cast<uint32_t>(h & 0x8000u) << 16);
    } else {
        return static_cast<uint32_t>(h) << 16;
    }
}

// One tensor restored by a batched launch (see decompress_batch_kernel).
struct RestoreJob {
    const uint32_t *bitmap;
    const void     *values;
    const uint64_t *values_offset;  // NULL, or the device word holding the byte offset of the values inside `values`
    const uint64_t *prefix;
    void           *out;
    uint64_t        n;
    uint32_t        first_block;    // the launch's blocks [first_block, next job's first_block) restore this tensor
};
template <int kJobs>
struct RestoreParams {
    RestoreJob job[kJobs];
    uint32_t   jobs;
};

// `block`: index of this CTA among those that restore the tensor.  WIDEN: 0 restores the elements as they are; 1
// (binary16) / 2 (bfloat16) widens every restored 2-byte value to binary32 on its way out.
template <typename U, int kWarps, int WIDEN = 0>
__device__ __forceinline__ void
decompress_body(const uint32_t *__restrict__ bitmap, const U *values, const uint64_t *__restrict__ values_offset,
                const uint64_t *__restrict__ prefix, const uint64_t n, std::conditional_t<WIDEN != 0, uint32_t, U> *__restrict__ out,
                const uint64_t block)
{
    using P = walk::Of<U>;
    walk::Part pt;
    if (!walk::stage_part<U, kWarps>(bitmap, values, values_offset, prefix, n, block, pt)) return;
    const uint32_t lane = threadIdx.x & 31u;
    const Extent   ox   = extent_of(out, n * sizeof(*out));
#pragma unroll
    for (int k = 0; k < P::kSteps; ++k) {
        const auto     v  = walk::expand_step<U>(pt, k, lane);
        const uint64_t at = pt.e0 + static_cast<uint64_t>(k) * (32 * P::kPerLane) + lane * P::kPerLane;
        if constexpr (WIDEN == 0) {
            if (pt.whole || at + P::kPerLane <= n) {
                if (ox.holds(out + at, sizeof(v))) *reinterpret_cast<std::remove_const_t<decltype(v)> *>(out + at) = v;
            } else {
                const U *const e = reinterpret_cast<const U *>(&v);
#pragma unroll
                for (int j = 0; j < P::kPerLane; ++j)
                    if (at + j < n && ox.holds(out + at + j, sizeof(U))) out[at + j] = e[j];
            }
        } else {
            // a clear bit gave the pattern 0, which widens to +0
            uint32_t f[4];
            if constexpr (WIDEN == 2) {
                f[0] = v.x << 16, f[1] = v.x & 0xFFFF0000u, f[2] = v.y << 16, f[3] = v.y & 0xFFFF0000u;
            } else {
                f[0] = widened<WIDEN>(static_cast<uint16_t>(v.x)), f[1] = widened<WIDEN>(static_cast<uint16_t>(v.x >> 16));
                f[2] = widened<WIDEN>(static_cast<uint16_t>(v.y)), f[3] = widened<WIDEN>(static_cast<uint16_t>(v.y >> 16));
            }
            if (pt.whole || at + 4 <= n) {
                if (ox.holds(out + at, 16)) *reinterpret_cast<uint4 *>(out + at) = make_uint4(f[0], f[1], f[2], f[3]);
            } else {
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    if (at + j < n && ox.holds(out + at + j, 4)) out[at + j] = f[j];
            }
        }
    }
}

// Warps per CTA.  The bound of twelve CTAs per SM keeps the registers at 42 at most.  Twelve fit with 4- and 8-byte elements
// (17.6 and 17.1 KB of shared memory each); with 2-byte elements the table of words takes 18.6 KB, and eleven do.
constexpr int kWarps = 4;

template <typename U, int WIDEN = 0>
__global__ void __launch_bounds__(kWarps * 32, 12)
decompress_kernel(const uint32_t *__restrict__ bitmap, const U *values, const uint64_t *__restrict__ values_offset,
                  const uint64_t *__restrict__ prefix, const uint64_t n, std::conditional_t<WIDEN != 0, uint32_t, U> *__restrict__ out)
{
    in_stream_order();
    decompress_body<U, kWarps, WIDEN>(bitmap, values, values_offset, prefix, n, out, blockIdx.x);
}

// The tensor a CTA of a batched launch works on: the last job whose first block is not behind this one.
template <int kJobs>
__device__ __forceinline__ uint32_t job_of_block(const RestoreParams<kJobs> &p)
{
    uint32_t k = 0;
    for (uint32_t j = 1; j < p.jobs; ++j) k = p.job[j].first_block <= blockIdx.x ? j : k;
    return k;
}

// Several tensors of one element type restored by ONE launch: every CTA looks up its tensor in the job table (in
// the kernel's parameters) and restores its parts of it exactly as the single-tensor kernel does.
template <typename U, int kJobs>
__global__ void __launch_bounds__(kWarps * 32, 12)
decompress_batch_kernel(const __grid_constant__ RestoreParams<kJobs> p)
{
    in_stream_order();
    const RestoreJob &j = p.job[job_of_block(p)];
    decompress_body<U, kWarps>(j.bitmap, static_cast<const U *>(j.values), j.values_offset, j.prefix, j.n, static_cast<U *>(j.out),
                               blockIdx.x - j.first_block);
}

template <typename U, int WIDEN = 0>
cudaError_t launch_typed(const uint32_t *bitmap, const void *values, const uint64_t *values_offset,
                         const uint64_t *prefix, uint64_t n, void *out, cudaStream_t stream)
{
    using O             = std::conditional_t<WIDEN != 0, uint32_t, U>;
    const uint64_t grid = walk::Of<U>::blocks_of(n, kWarps);
    if (grid > 0x7FFFFFFFull) return cudaErrorInvalidValue;
    return launch(decompress_kernel<U, WIDEN>, static_cast<unsigned>(grid), kWarps * 32, 0, stream, bitmap,
                  static_cast<const U *>(values), values_offset, prefix, n, static_cast<O *>(out));
}

template <typename U>
cudaError_t launch_batch_typed(const DecompressJob *jobs, uint32_t count, cudaStream_t stream)
{
    RestoreParams<kMaxBatch> p{};
    uint64_t                 blocks = 0;
    for (uint32_t k = 0; k < count; ++k) {
        p.job[k] = RestoreJob{jobs[k].bitmap, jobs[k].values, jobs[k].values_offset, jobs[k].prefix, jobs[k].out, jobs[k].n, static_cast<uint32_t>(blocks)};
        blocks += walk::Of<U>::blocks_of(jobs[k].n, kWarps);
        if (blocks > 0x7FFFFFFFull) return cudaErrorInvalidValue;
    }
    p.jobs = count;
    return launch(decompress_batch_kernel<U, kMaxBatch>, static_cast<unsigned>(blocks), kWarps * 32, 0, stream, p);
}

}  // namespace

cudaError_t launch_decompress_widen(const uint32_t *bitmap, const void *values16, const uint64_t *values_offset,
                                    const uint64_t *prefix, uint64_t n, int from_dtype, void *out_f32, cudaStream_t stream)
{
    return from_dtype == BT_F16 ? launch_typed<uint16_t, 1>(bitmap, values16, values_offset, prefix, n, out_f32, stream)
                                : launch_typed<uint16_t, 2>(bitmap, values16, values_offset, prefix, n, out_f32, stream);
}

cudaError_t launch_decompress(const uint32_t *bitmap, const void *values, const uint64_t *values_offset,
                              const uint64_t *prefix, uint64_t n, int elem_size, void *out, cudaStream_t stream)
{
    if (elem_size == 8) return launch_typed<uint64_t>(bitmap, values, values_offset, prefix, n, out, stream);
    if (elem_size == 4) return launch_typed<uint32_t>(bitmap, values, values_offset, prefix, n, out, stream);
    return launch_typed<uint16_t>(bitmap, values, values_offset, prefix, n, out, stream);
}

cudaError_t launch_decompress_batch(const DecompressJob *jobs, uint32_t count, int elem_size, cudaStream_t stream)
{
    if (count == 0 || count > kMaxBatch) return cudaErrorInvalidValue;
    if (elem_size == 8) return launch_batch_typed<uint64_t>(jobs, count, stream);
    return elem_size == 4 ? launch_batch_typed<uint32_t>(jobs, count, stream) : launch_batch_typed<uint16_t>(jobs, count, stream);
}

}  // namespace bt
