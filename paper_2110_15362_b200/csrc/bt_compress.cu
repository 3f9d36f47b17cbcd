// Algorithm 1 (dense -> bitmap) and its fused forms (ReLU, activation pruning) as ONE
// compaction pass: a persistent-CTA stream compaction whose prefix sum rides on the
// wave structure of the grid.
//
// The grid has exactly as many CTAs (G) as fit on the device at once and is
// launched cooperatively, so that all of them are co-resident (a tensor of at
// most G tiles: one CTA per tile, a plain launch), and CTA b takes tiles
// b, b+G, b+2G, ...: iteration j of every CTA together forms "wave j", G
// consecutive tiles.  The warps of a CTA are specialised: one load warp, two
// scan warps, and workers for everything else (bt_compress_common.cuh: `work`).
//
// Workers.  A tile is cut into segments of 4096 bytes, dealt to the workers in turn.  A worker takes its segment from the input ring into
// registers (the slot is free for the next bulk copy at once), finds the
// survivors, ranks them with one packed warp scan, posts the count, writes the
// segment's bitmap words, packs the survivors into its own ring in shared memory
// and, some tiles later, copies them from there to values[base + offset ...].
//
// Prefix.  Tile t's exclusive base is that of tile t - G, which the same CTA
// took in the wave before, plus the counts of the G tiles in between:
//     base(t) = base(t - G) + count(t - G) + ... + count(t - 1).
// As soon as a tile is counted a scan warp publishes the count in a descriptor.
// About one tile later -- when every CTA has published wave j -- it reads the G
// descriptors in front of its tile in ONE batch of independent loads, and uses
// them a tile after that.  The two scan warps alternate tiles, so that each has
// two tiles' time for that round trip to L2.  No tile waits on another CTA's
// base: only on counts, which never wait on anything but data.
//
// Nothing has to be zero before it starts: a tile's descriptor carries the
// launch's 64-bit tag in both of its halves, and a reader takes only descriptors
// with its own launch's tag, so the CTAs never meet.  (Sums of whole waves made
// by reductions, as an earlier version kept beside the descriptors, halve the
// descriptors read but want zeroed words and with them a grid-wide barrier in
// every launch of more than one wave.)
//
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
    __device__ __forceinline__ bool seek(const uint32_t it, TileIn &t) const
    {
        const uint64_t tile = cta + static_cast<uint64_t>(it) * G;       // 64-bit: running past the end cannot wrap
        if (tile >= num_tiles) return false;
        t.n = a.n, t.first = tile * kTile, t.src = a.src, t.y = a.y, t.bitmap = a.bitmap;
        return true;
    }
    __device__ __forceinline__ TileOut out(const uint32_t) const
    {
        if (!a.arena_cursor) return TileOut{a.values, a.capacity};
        const uint64_t c0 = sh.arena_c0;
        return TileOut{static_cast<unsigned char *>(a.values) + c0, c0 <= a.arena_bytes ? (a.arena_bytes - c0) / sizeof(V) : 0};
    }
};

// U: uint64_t, uint32_t or uint16_t (the element's width).
// FUSED: -1 for the plain compressor, else the number of the fused forward form.
// CAST: 0, or the 16-bit type the kept binary32 values are narrowed to (1 binary16, 2 bfloat16).
// kSegs segments per tile, kWorkers worker warps, kStages slots of the input ring, kRing bytes of packed values per worker.
template <typename U, int FUSED, bool WRITE_Y, int CAST, int kSegs, int kWorkers, int kStages, int kRing>
__global__ void __launch_bounds__((kWorkers + 3 + WRITE_Y) * 32) compress_kernel(const CompressArgs a, const uint32_t num_tiles)
{
    constexpr int kSeg          = Rows<U>::kSeg;
    constexpr int kTile         = kSegs * kSeg;
    constexpr int kChunksPerTile = kTile / BT_CHUNK_ELEMS;
    constexpr int kSegsPerChunk = BT_CHUNK_ELEMS / kSeg;
    // warp roles
    constexpr int kScanWarp = kWorkers;                   // and kScanWarp + 1
    constexpr int kLoadWarp = kWorkers + 2;               // and, with the dense output, a store warp behind it
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
    const uint32_t G    = gridDim.x;
    const uint32_t cta  = blockIdx.x;
    const U *const src  = static_cast<const U *>(a.src);
    const uint64_t n    = a.n;
    const uint64_t wait_ns = a.wait_ns;          // bound of every wait below

    // tile of iteration `it` of this CTA (64-bit so that running past the end cannot wrap)
    auto tile_of = [&](uint32_t it) { return cta + static_cast<uint64_t>(it) * G; };

    // The arena's cursor is read before the barrier below: the kernel's one update of it follows the last tile's base,
    // which needs a publication from every CTA, and a CTA publishes only after this barrier.
    sh.init(WRITE_Y, tid);
    in_stream_order();
    if (tid == 0) sh.arena_c0 = a.arena_cursor ? *reinterpret_cast<const volatile uint64_t *>(a.arena_cursor) : 0;
    __syncthreads();

    // bulk copy of tile `it` of this CTA into its ring slot (issued by lane 0 of the load warp)
    auto issue_load = [&](const uint32_t it) {
        const uint32_t s     = it % kStages;
        const uint64_t first = tile_of(it) * kTile;
        const uint64_t left  = n - first;
        const uint32_t valid = left < static_cast<uint64_t>(kTile) ? static_cast<uint32_t>(left) : kTile;
        const uint32_t bytes = (valid * static_cast<uint32_t>(sizeof(U))) & ~15u;   // whole 16-byte units
        fence_proxy_async();                       // the workers' accesses to the slot come first
        mbar_arrive_expect_tx(&sh.full[s], bytes);  // bytes == 0 simply completes the phase
        if (bytes) bulk_load(tiles + static_cast<size_t>(s) * kTile, src + first, bytes, &sh.full[s]);
    };

    // the part of the workspace behind its header, as large as the size query promises the caller
    const Extent wsx = extent_of(a.ws_desc, compress_workspace_bytes((n + BT_CHUNK_ELEMS - 1) / BT_CHUNK_ELEMS) - kWsHeaderBytes);

    if (warp == kLoadWarp) {
        // ------------------------------------------------------------ load warp (one lane)
        if (lane == 0) {
            uint32_t issued = 0;
            for (; tile_of(issued) < num_tiles; ++issued) {
                if (issued >= static_cast<uint32_t>(kStages) && !mbar_wait(&sh.empty[issued % kStages], ((issued / kStages) - 1) & 1u, &sh.abort, wait_ns)) break;
                issue_load(issued);
            }
            // This lane stays until every bulk copy it issued has landed, whatever the other warps do (they may
            // leave early once a bounded wait has run out somewhere): the CTA never retires with a copy into its
            // shared memory in flight.  Only the last kStages copies can still be pending; each wait is bounded.
            for (uint32_t it = issued > static_cast<uint32_t>(kStages) ? issued - kStages : 0; it < issued; ++it)
                mbar_wait<false>(&sh.full[it % kStages], (it / kStages) & 1u, &sh.abort, 20000000ull);
        }
        return;
    }

    if (warp == kScanWarp || warp == kScanWarp + 1) {
        // ------------------------------------------------------------ scan warps
        // Two warps share the scan: warp p takes this CTA's tiles p, p + 2, p + 4, ...  A warp's turn for
        // tile j is
        //   (a) wait until the workers have counted tile j, publish the count,
        //   (c) finish tile j - 2 (its own previous tile) from the loads of its previous turn and hand it
        //       to the workers; the base of tile j - 3 is the other scan warp's,
        //   (b) wait until tile j + 1 is counted -- about one tile later, when every CTA has published
        //       wave j -- and issue, in ONE batch of independent loads, the reads of the descriptors of
        //       the G tiles in front of tile j.
        // The loads of (b) are used a whole tile later, in (c) of the next turn, so the round trip to L2
        // (1.3 us under load, longer than one tile) never stalls a turn for long: a turn has two tiles' time.
        // (One warp doing every tile cannot hide that round trip however deep its software pipeline is:
        // its loads of consecutive tiles retire through the same scoreboard.)
        const uint32_t  p            = warp - kScanWarp;
        uint64_t *const desc         = a.ws_desc;                  // two words per tile
        const uint64_t  chunks_total = (n + BT_CHUNK_ELEMS - 1) / BT_CHUNK_ELEMS;
        const uint32_t  last_it      = static_cast<uint32_t>((num_tiles - 1 - cta) / G);   // this CTA's last iteration
        bool            failed       = false;

        // The tag of this launch.  Both scan warps read the same sequence number: it changes only once every CTA
        // has published all its counts, or two seconds into a failure.
        uint64_t seq = 0;
        if (lane == 0) seq = ld_relaxed_u64(a.ws_header + kHdrSeq);
        seq                   = __shfl_sync(kFull, seq, 0);
        const uint64_t tag    = mix64(a.call_tag + seq * 0x9E3779B97F4A7C15ull) | 1ull;
        const uint64_t tag_w0 = tag & 0xFFFFFFFF00000000ull, tag_w1 = tag << 32;
        if (p == 0 && lane == 0) sh.tag = tag;
        auto valid = [&](const uint64_t w0, const uint64_t w1) {
            return ((w0 ^ tag_w0) >> 32) == 0 && ((w1 ^ tag_w1) >> 32) == 0 && static_cast<uint32_t>(w0) == static_cast<uint32_t>(w1);
        };

        // d0[k], d1[k], lane l <-> descriptor l + 32k of the window in front of this warp's previous tile: `window` tiles
        // from tile `from` on
        uint64_t d0[kMaxWindows], d1[kMaxWindows], from = 0;
        uint32_t window = 0;
#pragma unroll
        for (int k = 0; k < kMaxWindows; ++k) d0[k] = tag_w0, d1[k] = tag_w1;

        for (uint32_t j = p; !failed && j <= last_it + 2; j += 2) {
            if (j <= last_it) {
                // ---- (a)
                const uint32_t q = j % kQueue;
                if (!mbar_wait(&sh.counted[q], (j / kQueue) & 1u, &sh.abort, wait_ns)) {
                    failed = true;
                    break;
                }
                const uint32_t c   = lane < kSegs ? sh.cnt[q][lane] : 0u;
                uint32_t       inc = c;
#pragma unroll
                for (int o = 1; o < kSegs; o <<= 1) {
                    const uint32_t u = __shfl_up_sync(kFull, inc, o);
                    if (lane >= static_cast<uint32_t>(o)) inc += u;
                }
                const uint32_t agg = __shfl_sync(kFull, inc, kSegs - 1);
                if (lane == 0) {
                    if (wsx.holds(desc + 2 * tile_of(j), 16)) st_relaxed_2xu64(desc + 2 * tile_of(j), tag_w0 | agg, tag_w1 | agg);
                    sh.agg[q] = agg;
                }
                if (lane < kSegs) sh.off[q][lane] = inc - c;
            }
            if (j >= 2) {
                // ---- (c): tile j - 2 <= last_it
                const uint32_t f     = j - 2;
                uint32_t       polls = 0;
                uint64_t       t0    = 0;
                for (;;) {
                    bool missing = false;
#pragma unroll
                    for (int k = 0; k < kMaxWindows; ++k) missing |= !valid(d0[k], d1[k]);
                    if (!__any_sync(kFull, missing)) break;
                    __nanosleep(num_tiles > G ? 100 : 20);
                    if ((++polls & 255u) == 0 || (kTestHooks && wait_ns < kStrictLimitNs)) {
                        if (t0 == 0) t0 = now_ns();
                        if (__any_sync(kFull, (now_ns() - t0 > wait_ns) || ld_relaxed_u64(a.ws_header + kHdrAbort) == tag)) {
                            failed = true;
                            break;
                        }
                    }
#pragma unroll
                    for (int k = 0; k < kMaxWindows; ++k)
                        if (!valid(d0[k], d1[k]))
                            ld_relaxed_2xu64(desc + 2 * (from + lane + 32u * k), d0[k], d1[k]);
                }
                if (failed) break;
                uint32_t part = 0;                                   // at most 160 tiles of 16384 elements
#pragma unroll
                for (int k = 0; k < kMaxWindows; ++k) part += static_cast<uint32_t>(d0[k]);
                uint64_t base = __reduce_add_sync(kFull, part);
                if (f > 0) {
                    if (!mbar_wait(&sh.ready[(f - 1) % kQueue], ((f - 1) / kQueue) & 1u, &sh.abort, wait_ns)) {
                        failed = true;
                        break;
                    }
                    base += sh.base[(f - 1) % kQueue];
                }
                const uint32_t ps = f % kQueue;
                const uint64_t pt = tile_of(f);
                // exclusive count in front of each chunk of that tile
                if (lane < kSegs && (lane % kSegsPerChunk) == 0) {
                    const uint64_t ch = pt * kChunksPerTile + lane / kSegsPerChunk;
                    if (ch < chunks_total && extent_of(a.prefix, 8 * chunks_total).holds(a.prefix + ch, 8)) a.prefix[ch] = base + sh.off[ps][lane];
                }
                const uint32_t agg_last = sh.agg[ps];
                __syncwarp();
                if (lane == 0) {
                    sh.base[ps] = base;
                    mbar_arrive(&sh.ready[ps]);                      // the tile's values may leave; what follows takes two trips to L2 and fences
                }
                if (pt == num_tiles - 1 && lane == 0) {
                    const uint64_t nnz = base + agg_last;
                    *a.nnz_out = nnz;
                    // (the status word needs no look at the abort word here: it is looked at after the store, below)
                    const bool aborted = a.arena_cursor && ld_relaxed_u64(a.ws_header + kHdrAbort) == tag;
                    uint64_t capacity = a.capacity;
                    if (a.arena_cursor) {
                        // arena form: the room left behind the cursor; the cursor moves only when everything fitted
                        const uint64_t c0 = sh.arena_c0;
                        capacity          = c0 <= a.arena_bytes ? (a.arena_bytes - c0) / sizeof(Stored<CAST, U>) : 0;
                        if (!aborted && nnz <= capacity) {
                            *a.values_offset_out = c0;
                            *a.arena_cursor      = c0 + ((nnz * sizeof(Stored<CAST, U>) + 15) & ~15ull);
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
                    // every CTA has published all its counts by now, so every CTA has read the sequence number:
                    // the next launch on this workspace gets another tag
                    red_add_u64(a.ws_header + kHdrSeq, 1ull);
                }
            }
            if (j <= last_it) {
                // ---- (b): a tile later (when the other scan warp's next tile is counted, if there is one)
                if (j + 1 > last_it) {
                    // This CTA's last tile: no next tile to wait for.  A short pause gives the other counts of the
                    // wave time to land, so that the reads below usually succeed at once instead of costing a second
                    // round trip; a launch of one wave, whose counts come all at once, does not pause (fp32 200704
                    // elements 7.2 -> 6.7 us; 2.4 M elements, two waves: 9.9 -> 10.4 without the pause).
                    __nanosleep(num_tiles > G ? 300 : 20);
                } else if (!mbar_wait(&sh.counted[(j + 1) % kQueue], ((j + 1) / kQueue) & 1u, &sh.abort, wait_ns)) {
                    failed = true;
                    break;
                }
                window = tile_of(j) < G ? static_cast<uint32_t>(tile_of(j)) : G;
                from   = tile_of(j) - window;
#pragma unroll
                for (int k = 0; k < kMaxWindows; ++k) {
                    if (lane + 32u * k < window) ld_relaxed_2xu64(desc + 2 * (from + lane + 32u * k), d0[k], d1[k]);
                    else d0[k] = tag_w0, d1[k] = tag_w1;             // no such tile: a valid count of 0
                }
            }
        }
        if (failed && lane == 0) raise_timeout(a.ws_header, a.dev_status, &sh.abort, sh.tag);
        return;
    }

    OneTensor<U, Stored<CAST, U>, kTile, CtaState<kSegs, kStages>> stream{a, sh, num_tiles, cta, G};
    if constexpr (WRITE_Y) {
        if (warp == kLoadWarp + 1) {
            if (!store_dense<U>(sh, tiles, lane, stream, wait_ns) && lane == 0) raise_timeout(a.ws_header, a.dev_status, &sh.abort, sh.tag);
            return;
        }
    }

    // ---------------------------------------------------------------- workers
    if (!work<U, FUSED, WRITE_Y, CAST, kSegs, kWorkers, kStages, kRing>(sh, tiles, packed + warp * kRing, warp, lane, stream, a.tau, wait_ns,
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

// The calling thread's limit on the CTAs of one compress launch (0: none).  A cooperative launch needs all its
// CTAs resident at once and a CTA of this kernel fills an SM, so two launches of more than half the SMs each run
// one after the other even on different streams; a caller that keeps several launches in flight gives each a
// share of the SMs.
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
    constexpr int kThreads = (kWorkers + 3 + WRITE_Y) * 32;
    constexpr size_t kSmem = static_cast<size_t>(kStages) * kTile * sizeof(U) + static_cast<size_t>(kWorkers) * kRing;
    static LaunchShape shape;   // one per instantiation
    auto kernel = compress_kernel<U, FUSED, WRITE_Y, CAST, kSegs, kWorkers, kStages, kRing>;

    const uint32_t num_tiles = static_cast<uint32_t>((a.n + kTile - 1) / kTile);
    int            max_grid  = 0;
    cudaError_t    e         = shape.max_grid(kernel, kThreads, kSmem, max_grid);
    if (e != cudaSuccess) return e;
    if (max_grid > 32 * kMaxWindows) max_grid = 32 * kMaxWindows;
    if (t_max_ctas != 0 && static_cast<uint32_t>(max_grid) > t_max_ctas) max_grid = static_cast<int>(t_max_ctas);
    const uint32_t grid  = num_tiles < static_cast<uint32_t>(max_grid) ? num_tiles : static_cast<uint32_t>(max_grid);
    CompressArgs args = a;
    args.call_tag     = next_call_tag();
    args.wait_ns      = compress_wait_ns();
    return launch_waiting(num_tiles, kernel, grid, kThreads, kSmem, stream, args, num_tiles);
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
