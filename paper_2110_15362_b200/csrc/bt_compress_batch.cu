// The batched forms of Algorithm 1 and of its fused ReLU form: the tensors of a batch in ONE launch of the
// persistent compaction kernel (bt_compress.cu describes the pipeline of a CTA, the compaction and the scan).
//
// What a batch adds.  The tiles of all tensors are numbered through, tensor after tensor, and handed out in that order as
// those of one tensor are, so the CTAs share the batch evenly whatever the tensors' sizes.  The prefix restarts at every
// tensor: the base of a tile is that of the CTA's tile before, where that is in the same tensor, plus the counts of the
// tensor's tiles in between.  Every tensor gets exactly the bitmap, values, chunk prefix, count and status the
// single-tensor call would give it.  A step that
// stashes many activations of a few megabytes pays the fixed cost of a launch (load, compact, exchange counts, copy
// out: each a memory round trip) once per batch instead of once per tensor.
#include "bt_compress_common.cuh"

namespace bt {
namespace {

using namespace cmp;

template <int kJobs>
struct CompressParams {
    CompressCommon c;
    CompressJob    job[kJobs];
};

// Raise the abort flag (shared, and global under this launch's tag if the CTA got as far as reading it), move
// the workspace's sequence number so that the next launch cannot take this one's words for its own, and report
// the timeout in every tensor's status word.
template <int kJobs>
__device__ __noinline__ void raise_timeout(const CompressParams<kJobs> &p, volatile uint32_t *s_abort, const uint64_t tag)
{
    *s_abort = 1u;
    if (tag) st_relaxed_u64(p.c.ws_header + kHdrAbort, tag);
    red_add_u64(p.c.ws_header + kHdrSeq, 1ull << 32);
    __threadfence();
    for (uint32_t k = 0; k < p.c.jobs; ++k)
        if (p.job[k].dev_status) *reinterpret_cast<volatile int32_t *>(p.job[k].dev_status) = BT_ERR_TIMEOUT;
}

// The tensor of a tile, looked for from tensor k on.
template <int kJobs>
__device__ __forceinline__ uint32_t tensor_of(const CompressParams<kJobs> &p, uint32_t k, const uint32_t tile)
{
    while (tile - p.job[k].desc0 >= p.job[k].tiles) ++k;
    return k;
}

// values of `size` bytes that fit behind a cursor of an arena
__device__ __forceinline__ uint64_t arena_room(const uint64_t cursor, const uint64_t bytes, const uint32_t size)
{
    return cursor <= bytes ? (bytes - cursor) / size : 0;
}

// The tiles of a CTA of a batched launch, as `work` takes them.
template <typename U, int kTile, int kJobs, typename State>
struct ManyTensors {
    const CompressParams<kJobs> &p;
    const State                 &sh;
    uint32_t                     k;         // the tensor looked at last: a CTA's tiles ascend
    // tile `it` of the CTA where they are dealt out beforehand
    __device__ __forceinline__ uint32_t dealt(const uint32_t it) const
    {
        const uint64_t tile = blockIdx.x + static_cast<uint64_t>(it) * gridDim.x;        // 64-bit: running past the end cannot wrap
        return tile < p.c.tiles ? static_cast<uint32_t>(tile) : kNoTile;
    }
    __device__ __forceinline__ bool seek(const uint32_t it, TileIn &t)
    {
        const uint32_t tile = dealt(it);
        if (tile == kNoTile) return false;
        locate(tile, t);
        return true;
    }
    __device__ __forceinline__ void locate(const uint32_t tile, TileIn &t)
    {
        k                    = tensor_of(p, k, tile);
        const CompressJob &j = p.job[k];
        t.n = j.n, t.first = static_cast<uint64_t>(tile - j.desc0) * kTile, t.src = j.src, t.y = j.y, t.bitmap = j.bitmap;
    }
    __device__ __forceinline__ void publish(const uint32_t tile, const uint32_t count, const uint64_t tag) const
    {
        uint64_t *const d = p.c.ws_desc + 2 * static_cast<uint64_t>(tile);
        if (extent_of(p.c.ws_desc, 8 * p.c.ws_words).holds(d, 16)) post(d, count, tag);
    }
    __device__ __forceinline__ TileOut out(const uint32_t q) const
    {
        if (p.c.arena == nullptr) {
            const CompressJob &j = p.job[sh.job[q]];
            return TileOut{j.values, j.capacity};
        }
        const uint64_t at0 = sh.dst[q];
        return TileOut{static_cast<unsigned char *>(p.c.arena) + at0, arena_room(at0, p.c.arena_bytes, sizeof(U))};
    }
};

// What a scan warp of a batched launch does with a tile (see scan_tiles).  A window covers the tiles from the CTA's tile
// before on, whatever tensors they belong to.
template <typename U, int kSegs, int kChunksPerTile, int kJobs, typename State>
struct ManyScan : TileCounts<kSegs> {
    const CompressParams<kJobs> &p;
    State                       &sh;
    const uint32_t               lane;
    const uint64_t               tag;
    uint32_t                     k = 0;         // the tile's tensor
    uint32_t                     m;             // as far as add() has come: tensor m, `base` values of it, which start at
    uint64_t                     base, at;      // byte `at` of the arena
    __device__ __forceinline__ ManyScan(const CompressParams<kJobs> &params, State &state, uint32_t l, uint64_t t) : p(params), sh(state), lane(l), tag(t) {}
    __device__ __forceinline__ bool in_arena() const { return p.c.arena != nullptr; }
    __device__ __forceinline__ void begin(const uint32_t tile, const uint32_t j)
    {
        k = tensor_of(p, k, tile);
        this->take(sh, j, lane);
    }
    __device__ __forceinline__ void resume(const uint32_t j)
    {
        m = 0, base = 0, at = sh.arena_c0;
        if (j) m = sh.job[(j - 1) % kQueue], base = sh.base[(j - 1) % kQueue], at = sh.dst[(j - 1) % kQueue];
    }
    // Tensor by tensor, as far as the window goes or to the tile's tensor.  A tensor of the arena form starts where the tensor
    // before it ended: the window goes back to the CTA's tile before, whatever tensor that is in, so every CTA adds
    // up the tensors that end in between by itself and nobody waits for a cursor from another CTA (MobileNetV2 layers at
    // batch 2: 70 us with the cursors handed on, 38 this way; at batch 64 361 and 351).
    __device__ __forceinline__ void add(const Window &w)
    {
        const uint32_t to = w.from + w.size;
        for (uint32_t lo = w.from;; ++m) {
            const uint32_t end = p.job[m].desc0 + p.job[m].tiles, hi = end < to ? end : to;
            if (in_arena() || m == k) base += w.sum(lo, hi, lane);
            lo = hi;
            if (m == k || hi < end) break;
            // tensor m is complete: the cursor moves past it if it fits
            if (in_arena() && base <= arena_room(at, p.c.arena_bytes, sizeof(U))) at += (base * sizeof(U) + 15) & ~15ull;
            base = 0;
        }
    }
    __device__ __forceinline__ void finish(const uint32_t tile, const uint32_t j)
    {
        constexpr int      kSegsPerChunk = kSegs / kChunksPerTile;
        const CompressJob &jb            = p.job[k];
        const uint64_t     chunks_total  = (jb.n + BT_CHUNK_ELEMS - 1) / BT_CHUNK_ELEMS;
        const uint32_t     pt            = tile - jb.desc0, ps = j % kQueue;        // pt: the tile within its tensor
        // exclusive count in front of each chunk of the tile
        if (lane < kSegs && (lane % kSegsPerChunk) == 0) {
            const uint64_t ch = static_cast<uint64_t>(pt) * kChunksPerTile + lane / kSegsPerChunk;
            if (ch < chunks_total && extent_of(jb.prefix, 8 * chunks_total).holds(jb.prefix + ch, 8)) jb.prefix[ch] = base + (this->upto - this->own);
        }
        __syncwarp();
        if (lane != 0) return;
        sh.base[ps] = base;
        sh.dst[ps]  = at;
        sh.job[ps]  = k;
        mbar_arrive(&sh.ready[ps]);                      // the tile's values may leave; what follows takes two trips to L2 and fences
        if (pt != jb.tiles - 1) return;
        const uint64_t nnz = base + this->count;
        *jb.nnz_out        = nnz;
        // (the status word needs no look at the abort word here: it is looked at after the store, below)
        const bool aborted  = in_arena() && ld_relaxed_u64(p.c.ws_header + kHdrAbort) == tag;
        uint64_t   capacity = jb.capacity;
        if (in_arena()) {
            // the cursor moves past the tensor only when everything fitted
            capacity        = arena_room(at, p.c.arena_bytes, sizeof(U));
            const bool fits = !aborted && nnz <= capacity;
            if (fits) *jb.offset_out = at;
            if (k + 1 == p.c.jobs) {
                *p.c.arena_cursor = fits ? at + ((nnz * sizeof(U) + 15) & ~15ull) : at;
                __threadfence();
                st_relaxed_u64(p.c.ws_header + kHdrCursor, sh.arena_c0);
                if (!aborted) st_relaxed_u64(p.c.ws_header + kHdrPushed, tag);
            }
        }
        if (jb.dev_status) {
            *reinterpret_cast<volatile int32_t *>(jb.dev_status) = aborted ? BT_ERR_TIMEOUT : (nnz > capacity ? BT_ERR_CAPACITY : BT_OK);
            // a CTA that gives up from now on stores its BT_ERR_TIMEOUT after this word; one that gave
            // up just before is seen here
            __threadfence();
            if (!aborted && ld_relaxed_u64(p.c.ws_header + kHdrAbort) == tag)
                *reinterpret_cast<volatile int32_t *>(jb.dev_status) = BT_ERR_TIMEOUT;
        }
        // the launch's last tile: all counts are published by now, so every CTA has read the sequence number:
        // the next launch on this workspace gets another tag
        if (k + 1 == p.c.jobs) red_add_u64(p.c.ws_header + kHdrSeq, 1ull);
    }
};

// U: uint64_t, uint32_t or uint16_t (the element's width).
// FUSED: -1 for the plain compressor, else the number of the fused forward form.
// kJobs: room for tensors in the kernel's parameters.
// kSegs segments per tile, kWorkers worker warps, kStages slots of the input ring, kRing bytes of packed values per worker.
template <typename U, int FUSED, bool WRITE_Y, bool LISTED, int kJobs, int kSegs, int kWorkers, int kStages, int kRing>
__global__ void __launch_bounds__(warps_of<U>(WRITE_Y) * 32)
compress_kernel(const __grid_constant__ CompressParams<kJobs> p)
{
    constexpr int kSeg           = Rows<U>::kSeg;
    constexpr int kTile          = kSegs * kSeg;
    constexpr int kChunksPerTile = kTile / BT_CHUNK_ELEMS;
    // warp roles
    constexpr int kScanWarp = kWorkers;                   // and kScanWarp + 1
    constexpr int kLoadWarp = kWorkers + 2;               // and behind it a publishing and a store warp, as the form has them
    static_assert(BT_CHUNK_ELEMS % kSeg == 0 && kTile % BT_CHUNK_ELEMS == 0, "segments tile a chunk, chunks a tile");
    static_assert(kSegs <= 32, "one lane per segment count");

    extern __shared__ __align__(128) unsigned char smem_raw[];
    U *const       tiles  = reinterpret_cast<U *>(smem_raw);                                        // input ring
    const uint32_t packed = smem_addr(smem_raw) + kStages * kTile * static_cast<int>(sizeof(U));    // packed rings
    __shared__ CtaState<kSegs, kStages> sh;

    const uint32_t tid  = threadIdx.x;
    const uint32_t lane = tid & 31u;
    // broadcast from lane 0 so that the compiler knows the role branches below are warp-uniform
    const uint32_t warp    = __shfl_sync(kFull, tid >> 5, 0);
    const uint64_t wait_ns = p.c.wait_ns;

    // The arena's cursor is read before the barrier below: the launch's first update of it follows a tensor's last base,
    // which needs a publication from every CTA in front of it, and the sequence number moves only behind all of them.
    const bool in_arena = p.c.arena != nullptr;
    if (LISTED && p.c.stealing && tid == kLoadWarp * 32) ask_first(sh);
    sh.init(WRITE_Y, kPublisher<U>, tid);
    in_stream_order();
    if (tid == 0) sh.arena_c0 = in_arena ? *reinterpret_cast<const volatile uint64_t *>(p.c.arena_cursor) : 0;
    __syncthreads();

    ManyTensors<U, kTile, kJobs, CtaState<kSegs, kStages>> stream{p, sh, 0};

    if (warp == kLoadWarp) {
        if (lane == 0) load_tiles<U, LISTED>(sh, tiles, stream, p.c.tiles, p.c.stealing != 0, wait_ns);
        return;
    }

    if (warp == kScanWarp || warp == kScanWarp + 1) {
        // ------------------------------------------------------------ scan warps
        const uint32_t q   = warp - kScanWarp;
        const uint64_t tag = scan_tag(sh, q, lane, p.c.call_tag, p.c.ws_header, wait_ns);
        ManyScan<U, kSegs, kChunksPerTile, kJobs, CtaState<kSegs, kStages>> scan(p, sh, lane, tag);
        if ((tag == 0 || !scan_tiles<U, LISTED>(sh, q, lane, stream, scan, p.c.ws_desc, p.c.ws_header, tag, false, wait_ns)) && lane == 0)
            raise_timeout(p, &sh.abort, tag);
        return;
    }

    if constexpr (kPublisher<U>) {
        if (warp == kLoadWarp + 1) {
            if (!publish_tiles<U, LISTED>(sh, lane, stream, wait_ns) && lane == 0) raise_timeout(p, &sh.abort, sh.tag);
            return;
        }
    }
    if constexpr (WRITE_Y) {
        if (warp == kLoadWarp + 1 + (kPublisher<U> ? 1 : 0)) {
            if (!store_dense<U>(sh, tiles, lane, stream, wait_ns) && lane == 0) raise_timeout(p, &sh.abort, sh.tag);
            return;
        }
    }

    // ---------------------------------------------------------------- workers
    if (!work<U, FUSED, WRITE_Y, 0, LISTED, kSegs, kWorkers, kStages, kRing>(sh, tiles, packed + warp * kRing, warp, lane, stream, 0.0f, wait_ns, true) && lane == 0)
        raise_timeout(p, &sh.abort, sh.tag);
}

// Behind an arena launch of more than one tensor: the values of the tensors that fit behind one that did not.  Such a
// tensor starts where the one that did not fit started, and that one's first values went there as well (its tiles leave
// before its count is known), in no order.  Once the launch is complete they are gathered again, from the dense input under
// the bitmap: a kept element is the input's own pattern, in the fused ReLU too, whose dense output may lie over the input.
//
// Where everything fitted, as the counts and the cursor tell, there is nothing to do, and what it costs is a launch: 2 us
// with few CTAs, 2.9 with one per SM (35 layers of MobileNetV2 at batch 1, two such launches: 39.0 us without, 43.1, 44.8).
// So the CTAs go by the tiles of the launch, one per 64 and at least 8 (8 take 10 ms for 400 MB, one per SM 0.6).  Leave
// to start early, given by the launch in front, costs 0.2 us more.  Ordering the launch's own stores instead would take a
// published end of every CTA's copy-out, fences included, in every launch.
constexpr uint32_t kAgainThreads = 256;
inline uint32_t again_ctas(const uint64_t tiles, const uint32_t most)
{
    const uint64_t n = tiles / 64 < 8 ? 8 : tiles / 64;
    return n < most ? static_cast<uint32_t>(n) : most;
}
template <typename U, int kJobs>
__global__ void __launch_bounds__(kAgainThreads) values_again_kernel(const __grid_constant__ CompressParams<kJobs> p)
{
    in_stream_order();
    const uint32_t lane = threadIdx.x & 31u;
    const uint64_t nnz  = lane < p.c.jobs ? *p.job[lane].nnz_out : 0;
    const uint64_t at0  = p.c.ws_header[kHdrCursor];
    // A launch that finished moved the sequence number by one, one that gave up by more (and may not have come to this word,
    // which then holds an earlier launch's tag, beside that launch's cursor): every output of it is undefined.
    if (p.c.ws_header[kHdrPushed] != tag_of(p.c.call_tag, p.c.ws_header[kHdrSeq] - 1)) return;
    const uint64_t all = warp_sum_u64((nnz * sizeof(U) + 15) & ~15ull);
    if (at0 <= p.c.arena_bytes && all <= p.c.arena_bytes - at0) return;
    uint64_t at      = at0;
    bool     refused = false;
    for (uint32_t k = 0; k < p.c.jobs; ++k) {
        const uint64_t count = __shfl_sync(kFull, nnz, k);
        if (count > arena_room(at, p.c.arena_bytes, sizeof(U))) {
            refused = true;
            continue;
        }
        if (refused) {
            const CompressJob &j    = p.job[k];
            const U *const     src  = static_cast<const U *>(j.src);
            U *const           to   = reinterpret_cast<U *>(static_cast<unsigned char *>(p.c.arena) + at);
            const Extent       vx   = extent_of(to, count * sizeof(U));
            const uint64_t     step = static_cast<uint64_t>(gridDim.x) * (kAgainThreads / 32);
            // a chunk per warp and turn, its bitmap words four per lane
            for (uint64_t ch = static_cast<uint64_t>(blockIdx.x) * (kAgainThreads / 32) + (threadIdx.x >> 5); ch * BT_CHUNK_ELEMS < j.n; ch += step) {
                const uint64_t e0   = ch * BT_CHUNK_ELEMS + lane;
                const uint4    w4   = load_words4(j.bitmap, ch * (BT_CHUNK_ELEMS / 32) + 4 * lane, (j.n + 31) >> 5);
                uint64_t       rank = j.prefix[ch];
#pragma unroll 2
                for (uint32_t q = 0; q < 32; ++q) {
                    const uint32_t w[4] = {__shfl_sync(kFull, w4.x, q), __shfl_sync(kFull, w4.y, q), __shfl_sync(kFull, w4.z, q), __shfl_sync(kFull, w4.w, q)};
                    U              v[4];
#pragma unroll
                    for (uint32_t i = 0; i < 4; ++i) {
                        const uint64_t e = e0 + 32 * (4 * q + i);
                        v[i]             = ((w[i] >> lane) & 1u) && e < j.n ? src[e] : U(0);
                    }
#pragma unroll
                    for (uint32_t i = 0; i < 4; ++i) {
                        const uint64_t e = e0 + 32 * (4 * q + i), at_rank = rank + __popc(w[i] & lanemask_lt());
                        if (((w[i] >> lane) & 1u) && e < j.n && at_rank < count && vx.holds(to + at_rank, sizeof(U))) to[at_rank] = v[i];
                        rank += __popc(w[i]);
                    }
                }
            }
        }
        at += (count * sizeof(U) + 15) & ~15ull;
    }
}

template <typename U, int FUSED, bool WRITE_Y, int kJobs, int kSegs, int kWorkers, int kStages, int kRing>
cudaError_t launch_shaped(const CompressCommon &c, const CompressJob *jobs, uint32_t count, void *workspace, cudaStream_t stream)
{
    constexpr int    kTile    = kSegs * Rows<U>::kSeg;
    constexpr int    kThreads = warps_of<U>(WRITE_Y) * 32;
    constexpr size_t kSmem    = static_cast<size_t>(kStages) * kTile * sizeof(U) + static_cast<size_t>(kWorkers) * kRing;
    static LaunchShape shapes[2];   // one per instantiation
    // 2-byte types: the listed form when the tiles are dealt out, too.  In the other one, where every worker looks for the tensor
    // of its next tile before it waits for it, their registers no longer go round, and the loop over the segments spills
    // (bf16 VGG-16 at batch 32, 60 % zeros: 258 us that way, 225 listed; fp32 at batch 16: 197 and 200).
    constexpr bool kListed = WRITE_Y || sizeof(U) == 2;
    auto dealt  = compress_kernel<U, FUSED, WRITE_Y, kListed, kJobs, kSegs, kWorkers, kStages, kRing>;
    auto listed = compress_kernel<U, FUSED, WRITE_Y, true, kJobs, kSegs, kWorkers, kStages, kRing>;
    if (count == 0 || count > static_cast<uint32_t>(kJobs)) return cudaErrorInvalidValue;

    CompressParams<kJobs> p;
    p.c             = c;
    uint64_t tiles  = 0, chunks = 0;
    for (uint32_t k = 0; k < count; ++k) {
        p.job[k]            = jobs[k];
        const uint64_t t    = (jobs[k].n + kTile - 1) / kTile;
        if (t == 0 || t > 0xFFFFFFFFull) return cudaErrorInvalidValue;
        p.job[k].tiles      = static_cast<uint32_t>(t);
        tiles += t;
        chunks += (jobs[k].n + BT_CHUNK_ELEMS - 1) / BT_CHUNK_ELEMS;
    }
    if (tiles > 0xFFFFFFFFull) return cudaErrorInvalidValue;
    for (uint32_t k = count; k < static_cast<uint32_t>(kJobs); ++k) p.job[k] = CompressJob{};

    Deal        deal;
    cudaError_t e = deal_of(static_cast<uint32_t>(tiles), WRITE_Y, kBatchStealWaves, dealt, listed, shapes, kThreads, kSmem, deal);
    if (e != cudaSuccess) return e;
    p.c.stealing = deal.stealing;

    uint64_t first = 0;                         // tiles are numbered tensor after tensor
    for (uint32_t k = 0; k < count; ++k) {
        p.job[k].desc0 = static_cast<uint32_t>(first);
        first += p.job[k].tiles;
    }
    p.c.tiles     = static_cast<uint32_t>(tiles);
    p.c.jobs      = count;
    p.c.ws_header = static_cast<uint64_t *>(workspace);
    p.c.ws_desc   = reinterpret_cast<uint64_t *>(static_cast<unsigned char *>(workspace) + kWsHeaderBytes);
    p.c.ws_words  = (batch_workspace_bytes(chunks, count) - kWsHeaderBytes) / 8;
    p.c.call_tag  = next_call_tag();
    p.c.wait_ns   = compress_wait_ns();
    e = launch_as(deal.cooperative, deal.stealing ? listed : dealt, deal.grid, kThreads, kSmem, stream, p);
    if (e != cudaSuccess || p.c.arena == nullptr || count < 2) return e;
    return launch(values_again_kernel<U, kJobs>, again_ctas(tiles, deal.resident), kAgainThreads, 0, stream, p);
}

template <typename U, int FUSED, bool WRITE_Y>
cudaError_t launch_typed(const CompressCommon &c, const CompressJob *jobs, uint32_t count, void *workspace, cudaStream_t stream)
{
    using S = Shape;   // as the single-tensor kernel
    return launch_shaped<U, FUSED, WRITE_Y, kMaxBatch, S::kSegs, S::kWorkers, S::kStages, S::kRing>(c, jobs, count, workspace, stream);
}

}  // namespace

cudaError_t launch_compress_batch(const CompressJob *jobs, uint32_t count, void *workspace, int dtype, int fused,
                                  const BatchArena *arena, cudaStream_t stream)
{
    // fused: 0 plain compressor, 1 ReLU
    // the dense output is written for all tensors of a launch or for none
    if (count == 0 || count > kMaxBatch || fused > 1) return cudaErrorInvalidValue;
    const bool y = jobs[0].y != nullptr;
    for (uint32_t k = 1; k < count; ++k)
        if ((jobs[k].y != nullptr) != y) return cudaErrorInvalidValue;
    CompressCommon c{};
    if (arena) {
        c.arena        = arena->arena;
        c.arena_bytes  = arena->arena_bytes;
        c.arena_cursor = arena->arena_cursor;
    }
    if (fused == 0) {
        return dtype == BT_F64   ? launch_typed<uint64_t, -1, false>(c, jobs, count, workspace, stream)
               : dtype == BT_F32 ? launch_typed<uint32_t, -1, false>(c, jobs, count, workspace, stream)
                                 : launch_typed<uint16_t, -1, false>(c, jobs, count, workspace, stream);
    }
    // the ReLU: for 2- and 4-byte types decided by one compare in the element's own type (as in the single-tensor kernel)
    constexpr int kd = kFusedReluDirect;
    switch (dtype) {
    case BT_F64:
        return y ? launch_typed<uint64_t, BT_F64, true>(c, jobs, count, workspace, stream)
                 : launch_typed<uint64_t, BT_F64, false>(c, jobs, count, workspace, stream);
    case BT_F32:
        return y ? launch_typed<uint32_t, kd + BT_F32, true>(c, jobs, count, workspace, stream)
                 : launch_typed<uint32_t, kd + BT_F32, false>(c, jobs, count, workspace, stream);
    case BT_F16:
        return y ? launch_typed<uint16_t, kd + BT_F16, true>(c, jobs, count, workspace, stream)
                 : launch_typed<uint16_t, kd + BT_F16, false>(c, jobs, count, workspace, stream);
    default:
        return y ? launch_typed<uint16_t, kd + BT_BF16, true>(c, jobs, count, workspace, stream)
                 : launch_typed<uint16_t, kd + BT_BF16, false>(c, jobs, count, workspace, stream);
    }
}

}  // namespace bt
