// Algorithm 1 (dense -> bitmap) and its fused forms (ReLU, activation pruning) as ONE
// compaction pass: a stream compaction by one CTA per SM whose prefix sum rides on
// the tiles being taken in ascending order.
//
// A CTA takes tile after tile, each time a higher one; how the tiles are shared out
// is decided per launch (bt_compress_common.cuh: `load_tiles`, `deal_of`).  The warps
// of a CTA are specialised: a load warp, two scan warps, by the form a publishing and a
// store warp, and workers for everything else (bt_compress_common.cuh: `work`).
//
// Workers.  A tile is cut into segments of 4096 bytes, dealt to the workers in turn.  A worker takes its segment from the input ring into
// registers (the slot is free for the next bulk copy at once), finds the
// survivors, ranks them with one packed warp scan, posts the count, writes the
// segment's bitmap words, packs the survivors into its own ring in shared memory
// and, some tiles later, copies them from there to values[base + offset ...].
//
// Prefix.  Tile t's exclusive base is that of tile s, the one that the same CTA
// took before, plus the counts of the tiles from s on:
//     base(t) = base(s) + count(s) + ... + count(t - 1).
// As soon as a tile is counted its count is published in a descriptor.  About one
// tile later -- when the other CTAs have published what they took at the same
// time -- a scan warp reads the descriptors in front of its tile in ONE batch of
// independent loads, and uses them a tile after that (bt_compress_common.cuh:
// `scan_tiles`).  No tile waits on another CTA's base: only on counts of lower
// tiles, which never wait on anything but data.
//
// Nothing has to be zero before it starts: a tile's descriptor carries the
// launch's 64-bit tag in both of its halves, and a reader takes only descriptors
// with its own launch's tag, so the CTAs never meet.  (Sums of whole waves made
// by reductions, as an earlier version kept beside the descriptors, halve the
// descriptors read but want zeroed words and with them a grid-wide barrier in
// every launch of more than one wave.)
#include <atomic>
#include <chrono>

#include "bt_compress_common.cuh"

namespace bt {
namespace {

using namespace cmp;

// The tiles of a CTA of a single-tensor launch, as `work` takes them.
template <typename U, typename V, int kTile, typename State>
struct OneTensor {
    const CompressArgs &a;
    const State        &sh;
    const uint32_t      num_tiles, cta, G;
    // tile `it` of the CTA where they are dealt out beforehand
    __device__ __forceinline__ uint32_t dealt(const uint32_t it) const
    {
        const uint64_t tile = cta + static_cast<uint64_t>(it) * G;       // 64-bit: running past the end cannot wrap
        return tile < num_tiles ? static_cast<uint32_t>(tile) : kNoTile;
    }
    __device__ __forceinline__ bool seek(const uint32_t it, TileIn &t) const
    {
        // (as dealt() and locate(), spelt out, with the CTA's number at hand: bf16 2^29 304 us, 311 the other way)
        const uint64_t tile = cta + static_cast<uint64_t>(it) * G;
        if (tile >= num_tiles) return false;
        t.n = a.n, t.first = tile * kTile, t.src = a.src, t.y = a.y, t.bitmap = a.bitmap;
        return true;
    }
    __device__ __forceinline__ void locate(const uint32_t tile, TileIn &t) const
    {
        t.n = a.n, t.first = static_cast<uint64_t>(tile) * kTile, t.src = a.src, t.y = a.y, t.bitmap = a.bitmap;
    }
    __device__ __forceinline__ void publish(const uint32_t tile, const uint32_t count, const uint64_t tag) const
    {
        uint64_t *const d = a.ws_desc + 2 * static_cast<uint64_t>(tile);
        // the part of the workspace behind its header, as large as the size query promises the caller
        if (extent_of(a.ws_desc, compress_workspace_bytes((a.n + BT_CHUNK_ELEMS - 1) / BT_CHUNK_ELEMS) - kWsHeaderBytes).holds(d, 16)) post(d, count, tag);
    }
    __device__ __forceinline__ TileOut out(const uint32_t) const
    {
        if (!a.arena_cursor) return TileOut{a.values, a.capacity};
        const uint64_t c0 = sh.arena_c0;
        return TileOut{static_cast<unsigned char *>(a.values) + c0, c0 <= a.arena_bytes ? (a.arena_bytes - c0) / sizeof(V) : 0};
    }
};

// What a scan warp of a single-tensor launch does with a tile (see scan_tiles).
template <typename V, int kSegs, int kChunksPerTile, typename State>
struct OneScan : TileCounts<kSegs> {
    const CompressArgs &a;
    State              &sh;
    const uint32_t      num_tiles, lane;
    const uint64_t      tag;
    uint64_t            base;
    __device__ __forceinline__ OneScan(const CompressArgs &args, State &state, uint32_t tiles, uint32_t l, uint64_t t)
        : a(args), sh(state), num_tiles(tiles), lane(l), tag(t)
    {
    }
    __device__ __forceinline__ void begin(const uint32_t, const uint32_t j) { this->take(sh, j, lane); }
    __device__ __forceinline__ void resume(const uint32_t j) { base = j ? sh.base[(j - 1) % kQueue] : 0ull; }
    __device__ __forceinline__ void add(const Window &w) { base += w.sum(); }
    __device__ __forceinline__ void finish(const uint32_t tile, const uint32_t j)
    {
        constexpr int  kSegsPerChunk = kSegs / kChunksPerTile;
        const uint64_t chunks_total  = (a.n + BT_CHUNK_ELEMS - 1) / BT_CHUNK_ELEMS;
        const uint32_t ps            = j % kQueue;
        // exclusive count in front of each chunk of the tile
        if (lane < kSegs && (lane % kSegsPerChunk) == 0) {
            const uint64_t ch = static_cast<uint64_t>(tile) * kChunksPerTile + lane / kSegsPerChunk;
            if (ch < chunks_total && extent_of(a.prefix, 8 * chunks_total).holds(a.prefix + ch, 8)) a.prefix[ch] = base + (this->upto - this->own);
        }
        __syncwarp();
        if (lane != 0) return;
        sh.base[ps] = base;
        mbar_arrive(&sh.ready[ps]);                      // the tile's values may leave; what follows takes two trips to L2 and fences
        if (tile != num_tiles - 1) return;
        const uint64_t nnz = base + this->count;
        *a.nnz_out = nnz;
        // (the status word needs no look at the abort word here: it is looked at after the store, below)
        const bool aborted = a.arena_cursor && ld_relaxed_u64(a.ws_header + kHdrAbort) == tag;
        uint64_t capacity = a.capacity;
        if (a.arena_cursor) {
            // arena form: the room left behind the cursor; the cursor moves only when everything fitted
            const uint64_t c0 = sh.arena_c0;
            capacity          = c0 <= a.arena_bytes ? (a.arena_bytes - c0) / sizeof(V) : 0;
            if (!aborted && nnz <= capacity) {
                *a.values_offset_out = c0;
                *a.arena_cursor      = c0 + ((nnz * sizeof(V) + 15) & ~15ull);
            }
        }
        if (a.dev_status) {
            *reinterpret_cast<volatile int32_t *>(a.dev_status) = aborted ? BT_ERR_TIMEOUT : (nnz > capacity ? BT_ERR_CAPACITY : BT_OK);
            // a CTA that gives up from now on stores its BT_ERR_TIMEOUT after this word; one that gave up
            // just before is seen here
            __threadfence();
            if (!aborted && ld_relaxed_u64(a.ws_header + kHdrAbort) == tag)
                *reinterpret_cast<volatile int32_t *>(a.dev_status) = BT_ERR_TIMEOUT;
        }
        // all counts are published by now, so every CTA has read the sequence number:
        // the next launch on this workspace gets another tag
        red_add_u64(a.ws_header + kHdrSeq, 1ull);
    }
};

// U: uint64_t, uint32_t or uint16_t (the element's width).
// FUSED: -1 for the plain compressor, else the number of the fused forward form.
// CAST: 0, or the 16-bit type the kept binary32 values are narrowed to (1 binary16, 2 bfloat16).
// kSegs segments per tile, kWorkers worker warps, kStages slots of the input ring, kRing bytes of packed values per worker.
template <typename U, int FUSED, bool WRITE_Y, int CAST, bool LISTED, int kSegs, int kWorkers, int kStages, int kRing>
__global__ void __launch_bounds__(warps_of<U>(WRITE_Y) * 32) compress_kernel(const CompressArgs a, const uint32_t num_tiles)
{
    constexpr int kSeg          = Rows<U>::kSeg;
    constexpr int kTile         = kSegs * kSeg;
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
    const uint32_t warp = __shfl_sync(kFull, tid >> 5, 0);
    const uint64_t wait_ns = a.wait_ns;          // bound of every wait below

    // The arena's cursor is read before the barrier below: the kernel's one update of it follows the last tile's base,
    // which needs a publication from every CTA, and a CTA publishes only after this barrier.
    if (LISTED && a.stealing && tid == kLoadWarp * 32) ask_first(sh);
    sh.init(WRITE_Y, kPublisher<U>, tid);
    in_stream_order();
    if (tid == 0) sh.arena_c0 = a.arena_cursor ? *reinterpret_cast<const volatile uint64_t *>(a.arena_cursor) : 0;
    __syncthreads();

    OneTensor<U, Stored<CAST, U>, kTile, CtaState<kSegs, kStages>> stream{a, sh, num_tiles, blockIdx.x, gridDim.x};

    if (warp == kLoadWarp) {
        if (lane == 0) load_tiles<U, LISTED>(sh, tiles, stream, num_tiles, a.stealing != 0, wait_ns);
        return;
    }

    if (warp == kScanWarp || warp == kScanWarp + 1) {
        // ------------------------------------------------------------ scan warps
        const uint32_t p   = warp - kScanWarp;
        const uint64_t tag = scan_tag(sh, p, lane, a.call_tag, a.ws_header, wait_ns);
        OneScan<Stored<CAST, U>, kSegs, kChunksPerTile, CtaState<kSegs, kStages>> scan(a, sh, num_tiles, lane, tag);
        if ((tag == 0 || !scan_tiles<U, LISTED>(sh, p, lane, stream, scan, a.ws_desc, a.ws_header, tag, num_tiles <= gridDim.x && !a.stealing, wait_ns)) && lane == 0)
            raise_timeout(a.ws_header, a.dev_status, &sh.abort, sh.tag);
        return;
    }

    if constexpr (kPublisher<U>) {
        if (warp == kLoadWarp + 1) {
            if (!publish_tiles<U, LISTED>(sh, lane, stream, wait_ns) && lane == 0) raise_timeout(a.ws_header, a.dev_status, &sh.abort, sh.tag);
            return;
        }
    }
    if constexpr (WRITE_Y) {
        if (warp == kLoadWarp + 1 + (kPublisher<U> ? 1 : 0)) {
            if (!store_dense<U>(sh, tiles, lane, stream, wait_ns) && lane == 0) raise_timeout(a.ws_header, a.dev_status, &sh.abort, sh.tag);
            return;
        }
    }

    // ---------------------------------------------------------------- workers
    if (!work<U, FUSED, WRITE_Y, CAST, LISTED, kSegs, kWorkers, kStages, kRing>(sh, tiles, packed + warp * kRing, warp, lane, stream, a.tau, wait_ns,
                                                                               a.capacity != 0 || a.arena_cursor) && lane == 0)
        raise_timeout(a.ws_header, a.dev_status, &sh.abort, sh.tag);
}

}  // namespace

// A value no other call of this process gets: a counter that starts at a salt drawn from the clock and the
// address space, so that words left in recycled memory by another run of the library do not line up either.
uint64_t next_call_tag()
{
    static std::atomic<uint64_t> counter{
        cmp::mix64(static_cast<uint64_t>(std::chrono::steady_clock::now().time_since_epoch().count()) ^
                   cmp::mix64(reinterpret_cast<uintptr_t>(&counter)))};
    return counter.fetch_add(1, std::memory_order_relaxed);
}

// The calling thread's limit on the CTAs of one compress launch (0: none).  A launch of this kernel fills the SMs with one CTA
// each, and a cooperative one (deal_of) starts only when all its CTAs can be resident, so two launches of more than half the
// SMs each run one after the other even on different streams; a caller that keeps several in flight gives each a share of the SMs.
thread_local uint32_t t_max_ctas = 0;
uint32_t compress_max_ctas() { return t_max_ctas; }
uint32_t set_compress_max_ctas(uint32_t max_ctas)
{
    const uint32_t before = t_max_ctas;
    t_max_ctas            = max_ctas;
    return before;
}

// The bound of the kernels' waits; only a test build can change it.
std::atomic<uint64_t> g_wait_ns{kDefaultWaitNs};
uint64_t compress_wait_ns() { return g_wait_ns.load(std::memory_order_relaxed); }
uint64_t set_compress_wait_ns(uint64_t wait_ns) { return g_wait_ns.exchange(wait_ns, std::memory_order_relaxed); }

namespace {

template <typename U, int FUSED, bool WRITE_Y, int CAST, int kSegs, int kWorkers, int kStages, int kRing>
cudaError_t launch_shaped(const CompressArgs &a, cudaStream_t stream)
{
    constexpr int kTile    = kSegs * Rows<U>::kSeg;
    constexpr int kThreads = warps_of<U>(WRITE_Y) * 32;
    constexpr size_t kSmem = static_cast<size_t>(kStages) * kTile * sizeof(U) + static_cast<size_t>(kWorkers) * kRing;
    static LaunchShape shapes[2];   // one per instantiation
    auto dealt  = compress_kernel<U, FUSED, WRITE_Y, CAST, WRITE_Y, kSegs, kWorkers, kStages, kRing>;
    auto listed = compress_kernel<U, FUSED, WRITE_Y, CAST, true, kSegs, kWorkers, kStages, kRing>;

    const uint32_t num_tiles = static_cast<uint32_t>((a.n + kTile - 1) / kTile);
    Deal           deal;
    cudaError_t    e = deal_of(num_tiles, WRITE_Y, kStealWaves<U>, dealt, listed, shapes, kThreads, kSmem, deal);
    if (e != cudaSuccess) return e;
    CompressArgs args = a;
    args.call_tag     = next_call_tag();
    args.wait_ns      = compress_wait_ns();
    args.stealing     = deal.stealing;
    return launch_as(deal.cooperative, deal.stealing ? listed : dealt, deal.grid, kThreads, kSmem, stream, args, num_tiles);
}

template <typename U, int FUSED, bool WRITE_Y, int CAST = 0>
cudaError_t launch_typed(const CompressArgs &a, cudaStream_t stream)
{
    using S = Shape;
    return launch_shaped<U, FUSED, WRITE_Y, CAST, S::kSegs, S::kWorkers, S::kStages, S::kRing>(a, stream);
}

}  // namespace

cudaError_t launch_compress(const CompressArgs &a, int dtype, int fused, cudaStream_t stream)
{
    // fused: 0 plain compressor, 1 threshold form (ReLU at tau = 0), 2 ReLU6
    const bool y = a.y != nullptr;
    if (a.cast != 0) {
        // down-cast on stash: binary32 tensors, plain and threshold forms
        if (dtype != BT_F32 || fused == 2) return cudaErrorInvalidValue;
        const bool h = a.cast == BT_F16;
        if (fused == 0) return h ? launch_typed<uint32_t, -1, false, 1>(a, stream) : launch_typed<uint32_t, -1, false, 2>(a, stream);
        if (a.tau == 0.0f) {
            constexpr int kd = kFusedReluDirect + BT_F32;
            if (y) return h ? launch_typed<uint32_t, kd, true, 1>(a, stream) : launch_typed<uint32_t, kd, true, 2>(a, stream);
            return h ? launch_typed<uint32_t, kd, false, 1>(a, stream) : launch_typed<uint32_t, kd, false, 2>(a, stream);
        }
        if (y) return h ? launch_typed<uint32_t, BT_F32, true, 1>(a, stream) : launch_typed<uint32_t, BT_F32, true, 2>(a, stream);
        return h ? launch_typed<uint32_t, BT_F32, false, 1>(a, stream) : launch_typed<uint32_t, BT_F32, false, 2>(a, stream);
    }
    if (fused == 0) {
        return dtype == BT_F64   ? launch_typed<uint64_t, -1, false>(a, stream)
               : dtype == BT_F32 ? launch_typed<uint32_t, -1, false>(a, stream)
                                 : launch_typed<uint16_t, -1, false>(a, stream);
    }
    constexpr int k6 = kFusedRelu6;
    if (fused == 2) {
        switch (dtype) {
        case BT_F64:
            return y ? launch_typed<uint64_t, k6 + BT_F64, true>(a, stream) : launch_typed<uint64_t, k6 + BT_F64, false>(a, stream);
        case BT_F32:
            return y ? launch_typed<uint32_t, k6 + BT_F32, true>(a, stream) : launch_typed<uint32_t, k6 + BT_F32, false>(a, stream);
        // 2-byte types: the decisions by compares in the element's own type
        case BT_F16:
            return y ? launch_typed<uint16_t, kFusedRelu6Direct + BT_F16, true>(a, stream) : launch_typed<uint16_t, kFusedRelu6Direct + BT_F16, false>(a, stream);
        default:
            return y ? launch_typed<uint16_t, kFusedRelu6Direct + BT_BF16, true>(a, stream)
                     : launch_typed<uint16_t, kFusedRelu6Direct + BT_BF16, false>(a, stream);
        }
    }
    if (a.tau == 0.0f && dtype != BT_F64) {
        // the ReLU itself: decided by one compare in the element's own type instead of a compare with the threshold, a
        // select and the zero test
        constexpr int kd = kFusedReluDirect;
        if (dtype == BT_F32) return y ? launch_typed<uint32_t, kd + BT_F32, true>(a, stream) : launch_typed<uint32_t, kd + BT_F32, false>(a, stream);
        if (dtype == BT_F16) return y ? launch_typed<uint16_t, kd + BT_F16, true>(a, stream) : launch_typed<uint16_t, kd + BT_F16, false>(a, stream);
        return y ? launch_typed<uint16_t, kd + BT_BF16, true>(a, stream) : launch_typed<uint16_t, kd + BT_BF16, false>(a, stream);
    }
    switch (dtype) {
    case BT_F64:
        return y ? launch_typed<uint64_t, BT_F64, true>(a, stream) : launch_typed<uint64_t, BT_F64, false>(a, stream);
    case BT_F32:
        return y ? launch_typed<uint32_t, BT_F32, true>(a, stream) : launch_typed<uint32_t, BT_F32, false>(a, stream);
    case BT_F16:
        return y ? launch_typed<uint16_t, BT_F16, true>(a, stream) : launch_typed<uint16_t, BT_F16, false>(a, stream);
    default:
        return y ? launch_typed<uint16_t, BT_BF16, true>(a, stream)
                 : launch_typed<uint16_t, BT_BF16, false>(a, stream);
    }
}

}  // namespace bt
