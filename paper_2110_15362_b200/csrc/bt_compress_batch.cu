// The batched forms of Algorithm 1 and of its fused ReLU form: the tensors of a batch in ONE launch of the
// persistent compaction kernel (bt_compress.cu describes the pipeline of a CTA, the compaction and the scan).
//
// What a batch adds.  The tiles of all tensors are dealt round robin to the same resident grid: tile t of
// tensor k goes to CTA (rot_k + t) mod G, where rot_k continues the deal of the tensor before it, so every CTA
// gets the same share of the batch whatever the tensors' sizes.  The prefix restarts at every tensor: the base of
// tile t of a tensor is that of its tile t - G, which the same CTA took before, plus the counts of the G tiles in
// between (of all tiles in front of it where t < G).  Every tensor has its own descriptors in the workspace and gets
// exactly the bitmap, values, chunk prefix, count and status the single-tensor call would give it.  A step that
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

// ---------------------------------------------------------------------------------------------
// The tiles of a launch in the order one CTA takes them: tensor after tensor; inside tensor k the tiles
// v, v + G, v + 2G, ... with v = (cta - rot_k) mod G, the CTA's place in the deal of that tensor.
struct Walk {
    uint32_t k;       // tensor
    uint32_t j;       // wave of the tensor; the tile is v + j * G
    uint32_t v;       // this CTA's virtual index in the tensor
    uint32_t tiles;   // tiles of the tensor
    bool     valid;
    __device__ __forceinline__ uint32_t tile(const uint32_t G) const { return v + j * G; }
};

template <int kJobs>
__device__ __forceinline__ void walk_seek(Walk &w, const CompressParams<kJobs> &p, const uint32_t cta, const uint32_t G)
{
    while (w.k < p.c.jobs) {
        const uint32_t rot = p.job[w.k].rot;
        w.tiles            = p.job[w.k].tiles;
        w.v                = cta >= rot ? cta - rot : cta + G - rot;
        if (w.v < w.tiles) {
            w.j     = 0;
            w.valid = true;
            return;
        }
        ++w.k;
    }
    w.valid = false;
}
template <int kJobs>
__device__ __forceinline__ void walk_begin(Walk &w, const CompressParams<kJobs> &p, const uint32_t cta, const uint32_t G)
{
    w.k = 0, w.j = 0, w.v = 0, w.tiles = 0;
    walk_seek(w, p, cta, G);
}
template <int kJobs>
__device__ __forceinline__ void walk_next(Walk &w, const CompressParams<kJobs> &p, const uint32_t cta, const uint32_t G)
{
    ++w.j;
    if (static_cast<uint64_t>(w.v) + static_cast<uint64_t>(w.j) * G >= w.tiles) {
        ++w.k;
        walk_seek(w, p, cta, G);
    }
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
    const uint32_t               cta, G;
    Walk                         w;
    uint32_t                     at;        // the walk stands at this tile of the CTA
    __device__ __forceinline__ bool seek(const uint32_t it, TileIn &t)
    {
        for (; at < it && w.valid; ++at) walk_next(w, p, cta, G);
        if (!w.valid) return false;
        const CompressJob &j = p.job[w.k];
        t.n = j.n, t.first = static_cast<uint64_t>(w.tile(G)) * kTile, t.src = j.src, t.y = j.y, t.bitmap = j.bitmap;
        return true;
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

// U: uint64_t, uint32_t or uint16_t (the element's width).
// FUSED: -1 for the plain compressor, else the number of the fused forward form.
// kJobs: room for tensors in the kernel's parameters.
// kSegs segments per tile, kWorkers worker warps, kStages slots of the input ring, kRing bytes of packed values per worker.
template <typename U, int FUSED, bool WRITE_Y, int kJobs, int kSegs, int kWorkers, int kStages, int kRing>
__global__ void __launch_bounds__((kWorkers + 3 + WRITE_Y) * 32)
compress_kernel(const __grid_constant__ CompressParams<kJobs> p)
{
    constexpr int kSeg           = Rows<U>::kSeg;
    constexpr int kTile          = kSegs * kSeg;
    constexpr int kChunksPerTile = kTile / BT_CHUNK_ELEMS;
    constexpr int kSegsPerChunk  = BT_CHUNK_ELEMS / kSeg;
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
    const uint32_t warp    = __shfl_sync(kFull, tid >> 5, 0);
    const uint32_t G       = gridDim.x;
    const uint32_t cta     = blockIdx.x;
    const uint64_t wait_ns = p.c.wait_ns;

    // The arena's cursor is read before the barrier below: the launch's first update of it follows a tensor's last base,
    // which needs a publication from every CTA in front of it, and the sequence number moves only behind all of them.
    const bool in_arena = p.c.arena != nullptr;
    sh.init(WRITE_Y, tid);
    in_stream_order();
    if (tid == 0) sh.arena_c0 = in_arena ? *reinterpret_cast<const volatile uint64_t *>(p.c.arena_cursor) : 0;
    __syncthreads();

    const Extent wsx = extent_of(p.c.ws_desc, 8 * p.c.ws_words);

    if (warp == kLoadWarp) {
        // ------------------------------------------------------------ load warp (one lane)
        if (lane == 0) {
            uint32_t issued = 0;
            Walk     w;
            walk_begin(w, p, cta, G);
            for (uint32_t it = 0; w.valid; ++it, walk_next(w, p, cta, G)) {
                if (it >= static_cast<uint32_t>(kStages) && !mbar_wait(&sh.empty[it % kStages], ((it / kStages) - 1) & 1u, &sh.abort, wait_ns)) break;
                // bulk copy of the tile into its ring slot
                const uint32_t s     = it % kStages;
                const U *const src   = static_cast<const U *>(p.job[w.k].src);
                const uint64_t first = static_cast<uint64_t>(w.tile(G)) * kTile;
                const uint64_t left  = p.job[w.k].n - first;
                const uint32_t valid = left < static_cast<uint64_t>(kTile) ? static_cast<uint32_t>(left) : kTile;
                const uint32_t bytes = (valid * static_cast<uint32_t>(sizeof(U))) & ~15u;   // whole 16-byte units
                fence_proxy_async();                       // the workers' accesses to the slot come first
                mbar_arrive_expect_tx(&sh.full[s], bytes);  // bytes == 0 simply completes the phase
                if (bytes) bulk_load(tiles + static_cast<size_t>(s) * kTile, src + first, bytes, &sh.full[s]);
                issued = it + 1;
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
        // Two warps share the scan: warp q takes this CTA's tiles q, q + 2, q + 4, ... (counted in the order the
        // CTA takes them); a turn is that of the single-tensor kernel (bt_compress.cu).
        const uint32_t  q          = warp - kScanWarp;
        uint64_t *const desc       = p.c.ws_desc;
        bool            failed     = false;

        // number of tiles this CTA takes
        uint32_t my_tiles = 0;
        for (uint32_t k = 0; k < p.c.jobs; ++k) {
            const uint32_t rot = p.job[k].rot, t = p.job[k].tiles;
            const uint32_t v   = cta >= rot ? cta - rot : cta + G - rot;
            if (v < t) my_tiles += (t - v + G - 1) / G;
        }
        const uint32_t last_i = my_tiles - 1;       // every CTA has a tile: the grid is no larger than the tile count

        // The tag of this launch.  One warp reads the sequence number; it moves only once every CTA has published a
        // count, which a CTA does after this read.
        uint64_t tag = 0;
        if (q == 0) {
            if (lane == 0) {
                const uint64_t seq = ld_relaxed_u64(p.c.ws_header + kHdrSeq);
                tag                = mix64(p.c.call_tag + seq * 0x9E3779B97F4A7C15ull) | 1ull;
                sh.tag             = tag;
            }
        } else if (lane == 0) {
            tag = wait_tag(&sh.tag, &sh.abort, wait_ns);
        }
        tag = __shfl_sync(kFull, tag, 0);
        if (tag == 0) {
            if (lane == 0) raise_timeout(p, &sh.abort, 0);
            return;
        }
        // (before this CTA's first count: whoever finishes the launch's last tile has seen it)
        if (in_arena && cta == 0 && q == 0 && lane == 0) {
            st_relaxed_u64(p.c.ws_header + kHdrPushed, 0);
            __threadfence();
        }
        const uint64_t tag_w0 = tag & 0xFFFFFFFF00000000ull, tag_w1 = tag << 32;
        auto valid = [&](const uint64_t w0, const uint64_t w1) {
            return ((w0 ^ tag_w0) >> 32) == 0 && ((w1 ^ tag_w1) >> 32) == 0 && static_cast<uint32_t>(w0) == static_cast<uint32_t>(w1);
        };

        // d0[k], d1[k], lane l <-> descriptor l + 32k of the window in front of this warp's previous tile: `window` tiles
        // from descriptor `from` on
        uint64_t d0[kMaxWindows], d1[kMaxWindows], from = 0;
        uint32_t window = 0;
#pragma unroll
        for (int k = 0; k < kMaxWindows; ++k) d0[k] = tag_w0, d1[k] = tag_w1;

        Walk cur;                                   // this warp's tile of the turn
        walk_begin(cur, p, cta, G);
        if (q == 1 && cur.valid) walk_next(cur, p, cta, G);
        uint32_t pk = 0, pj = 0, pv = 0;            // this warp's previous tile: tensor, wave, virtual CTA

        for (uint32_t i = q; !failed && i <= last_i + 2; i += 2) {
            const bool has = i <= last_i;
            if (has) {
                // ---- (a)
                const uint32_t s = i % kQueue;
                if (!mbar_wait(&sh.counted[s], (i / kQueue) & 1u, &sh.abort, wait_ns)) {
                    failed = true;
                    break;
                }
                const uint32_t c   = lane < kSegs ? sh.cnt[s][lane] : 0u;
                uint32_t       inc = c;
#pragma unroll
                for (int o = 1; o < kSegs; o <<= 1) {
                    const uint32_t u = __shfl_up_sync(kFull, inc, o);
                    if (lane >= static_cast<uint32_t>(o)) inc += u;
                }
                const uint32_t agg = __shfl_sync(kFull, inc, kSegs - 1);
                if (lane == 0) {
                    uint64_t *const d = desc + 2 * (static_cast<uint64_t>(p.job[cur.k].desc0) + cur.tile(G));
                    if (wsx.holds(d, 16)) st_relaxed_2xu64(d, tag_w0 | agg, tag_w1 | agg);
                    sh.agg[s] = agg;
                }
                if (lane < kSegs) sh.off[s][lane] = inc - c;
            }
            if (i >= 2) {
                // ---- (c): this warp's previous tile, (pk, pj, pv)
                const CompressJob &jb    = p.job[pk];
                uint32_t           polls = 0;
                uint64_t           t0    = 0;
                for (;;) {
                    bool missing = false;
#pragma unroll
                    for (int k = 0; k < kMaxWindows; ++k) missing |= !valid(d0[k], d1[k]);
                    if (!__any_sync(kFull, missing)) break;
                    __nanosleep(100);
                    if ((++polls & 255u) == 0 || (kTestHooks && wait_ns < kStrictLimitNs)) {
                        if (t0 == 0) t0 = now_ns();
                        if (__any_sync(kFull, (now_ns() - t0 > wait_ns) || ld_relaxed_u64(p.c.ws_header + kHdrAbort) == tag)) {
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
                const uint64_t pt = pv + static_cast<uint64_t>(pj) * G;
                if ((in_arena ? i > 2 : pj > 0) && !mbar_wait(&sh.ready[(i - 3) % kQueue], ((i - 3) / kQueue) & 1u, &sh.abort, wait_ns)) {
                    failed = true;
                    break;
                }
                // the sum of the window's counts from descriptor lo to before hi: at most 160 tiles of 16384 elements
                auto counts = [&](const uint64_t lo, const uint64_t hi) {
                    uint32_t part = 0;
#pragma unroll
                    for (int k = 0; k < kMaxWindows; ++k) {
                        const uint64_t at = from + lane + 32u * k;
                        part += at >= lo && at < hi ? static_cast<uint32_t>(d0[k]) : 0u;
                    }
                    return __reduce_add_sync(kFull, part);
                };
                uint64_t base = 0, arena_at = 0;
                if (!in_arena) {
                    // the CTA's tile before is tile pt - G of the same tensor, if it is not the first here
                    base = (pj > 0 ? sh.base[(i - 3) % kQueue] : 0ull) + counts(0, ~0ull);
                } else {
                    // Arena form: the tensor's values start where the tensor before it ended.  The window goes back to the
                    // CTA's tile before, whatever tensor that is in, so every CTA adds up the tensors that end in between by
                    // itself and nobody waits for a cursor from another CTA (MobileNetV2 layers at batch 2: 70 us with the
                    // cursors handed on, 38 this way; at batch 64 361 and 351).
                    uint32_t m = 0;
                    uint64_t lo = from;
                    arena_at    = sh.arena_c0;
                    if (i > 2) m = sh.job[(i - 3) % kQueue], base = sh.base[(i - 3) % kQueue], arena_at = sh.dst[(i - 3) % kQueue];
                    for (;; ++m) {
                        const uint64_t end = static_cast<uint64_t>(p.job[m].desc0) + p.job[m].tiles, lin = jb.desc0 + pt;
                        const uint64_t hi  = end < lin ? end : lin;
                        base += counts(lo, hi);
                        lo = hi;
                        if (m == pk) break;
                        // tensor m is complete: the cursor moves past it if it fits
                        if (base <= arena_room(arena_at, p.c.arena_bytes, sizeof(U))) arena_at += (base * sizeof(U) + 15) & ~15ull;
                        base = 0;
                    }
                }
                const uint32_t ps = (i - 2) % kQueue;
                // exclusive count in front of each chunk of that tile
                if (lane < kSegs && (lane % kSegsPerChunk) == 0) {
                    const uint64_t ch = pt * kChunksPerTile + lane / kSegsPerChunk;
                    const uint64_t chunks_total = (jb.n + BT_CHUNK_ELEMS - 1) / BT_CHUNK_ELEMS;
                    if (ch < chunks_total && extent_of(jb.prefix, 8 * chunks_total).holds(jb.prefix + ch, 8)) jb.prefix[ch] = base + sh.off[ps][lane];
                }
                const uint32_t agg_last = sh.agg[ps];
                __syncwarp();
                if (lane == 0) {
                    sh.base[ps] = base;
                    sh.dst[ps]  = arena_at;
                    sh.job[ps]  = pk;
                    mbar_arrive(&sh.ready[ps]);                      // the tile's values may leave; what follows takes two trips to L2 and fences
                }
                bool bump = false;              // lane 0: this is the launch's last tile
                if (pt == jb.tiles - 1 && lane == 0) {
                    const uint64_t nnz = base + agg_last;
                    *jb.nnz_out        = nnz;
                    // (the status word needs no look at the abort word here: it is looked at after the store, below)
                    const bool aborted = in_arena && ld_relaxed_u64(p.c.ws_header + kHdrAbort) == tag;
                    uint64_t   capacity = jb.capacity;
                    if (in_arena) {
                        // the cursor moves past the tensor only when everything fitted
                        capacity        = arena_room(arena_at, p.c.arena_bytes, sizeof(U));
                        const bool fits = !aborted && nnz <= capacity;
                        if (fits) *jb.offset_out = arena_at;
                        if (pk + 1 == p.c.jobs) {
                            *p.c.arena_cursor = fits ? arena_at + ((nnz * sizeof(U) + 15) & ~15ull) : arena_at;
                            __threadfence();
                            st_relaxed_u64(p.c.ws_header + kHdrCursor, sh.arena_c0);
                            if (!aborted) st_relaxed_u64(p.c.ws_header + kHdrPushed, 1);
                        }
                    }
                    bump = pk + 1 == p.c.jobs;
                    if (jb.dev_status) {
                        *reinterpret_cast<volatile int32_t *>(jb.dev_status) = aborted ? BT_ERR_TIMEOUT : (nnz > capacity ? BT_ERR_CAPACITY : BT_OK);
                        // a CTA that gives up from now on stores its BT_ERR_TIMEOUT after this word; one that gave
                        // up just before is seen here
                        __threadfence();
                        if (!aborted && ld_relaxed_u64(p.c.ws_header + kHdrAbort) == tag)
                            *reinterpret_cast<volatile int32_t *>(jb.dev_status) = BT_ERR_TIMEOUT;
                    }
                }
                __syncwarp();
                if (__shfl_sync(kFull, bump ? 1 : 0, 0)) {
                    // The launch's last tile.  The next launch on this workspace must get another tag, and the sequence
                    // number may move only once every CTA has read it, i.e. has published a count.  The first G tiles
                    // of the launch are one per CTA: wait for their counts (they have been out for a long time).
                    bool seen[kMaxWindows];
#pragma unroll
                    for (int k = 0; k < kMaxWindows; ++k) seen[k] = lane + 32u * k >= G;
                    bool           all = true;
                    const uint64_t ts  = now_ns();
                    for (;;) {
                        bool miss = false;
#pragma unroll
                        for (int k = 0; k < kMaxWindows; ++k) {
                            if (!seen[k]) {
                                uint64_t x0, x1;
                                ld_relaxed_2xu64(desc + 2 * static_cast<uint64_t>(lane + 32u * k), x0, x1);
                                seen[k] = valid(x0, x1);
                                miss |= !seen[k];
                            }
                        }
                        if (!__any_sync(kFull, miss)) break;
                        if (__any_sync(kFull, now_ns() - ts > wait_ns)) {
                            all = false;
                            break;
                        }
                        __nanosleep(200);
                    }
                    if (lane == 0) red_add_u64(p.c.ws_header + kHdrSeq, all ? 1ull : 1ull << 32);
                }
            }
            if (has) {
                // ---- (b): a tile later (when the other scan warp's next tile is counted, if there is one)
                if (i + 1 > last_i) {
                    // This CTA's last tile: no next tile to wait for.  A short pause gives the other counts of the
                    // wave time to land, so that the reads below usually succeed at once instead of costing a second
                    // round trip.
                    __nanosleep(300);
                } else if (!mbar_wait(&sh.counted[(i + 1) % kQueue], ((i + 1) / kQueue) & 1u, &sh.abort, wait_ns)) {
                    failed = true;
                    break;
                }
                // the descriptors in front of the tile back to the CTA's tile before: in the arena form whatever tensor they
                // belong to, else those of the tile's own tensor
                const uint64_t lin  = static_cast<uint64_t>(p.job[cur.k].desc0) + cur.tile(G);
                const uint64_t back = in_arena ? lin : cur.tile(G);
                window = back < G ? static_cast<uint32_t>(back) : G;
                from   = lin - window;
#pragma unroll
                for (int k = 0; k < kMaxWindows; ++k) {
                    if (lane + 32u * k < window) ld_relaxed_2xu64(desc + 2 * (from + lane + 32u * k), d0[k], d1[k]);
                    else d0[k] = tag_w0, d1[k] = tag_w1;             // no such tile: a valid count of 0
                }
                pk = cur.k, pj = cur.j, pv = cur.v;
                walk_next(cur, p, cta, G);
                if (cur.valid) walk_next(cur, p, cta, G);
            }
        }
        if (failed && lane == 0) raise_timeout(p, &sh.abort, tag);
        return;
    }

    ManyTensors<U, kTile, kJobs, CtaState<kSegs, kStages>> stream{p, sh, cta, G, {}, 0};
    walk_begin(stream.w, p, cta, G);
    if constexpr (WRITE_Y) {
        if (warp == kLoadWarp + 1) {
            if (!store_dense<U>(sh, tiles, lane, stream, wait_ns) && lane == 0) raise_timeout(p, &sh.abort, sh.tag);
            return;
        }
    }

    // ---------------------------------------------------------------- workers
    if (!work<U, FUSED, WRITE_Y, 0, kSegs, kWorkers, kStages, kRing>(sh, tiles, packed + warp * kRing, warp, lane, stream, p.c.tau, wait_ns, true) && lane == 0)
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
inline uint32_t again_ctas(const uint64_t tiles, const uint32_t grid)
{
    const uint64_t n = tiles / 64 < 8 ? 8 : tiles / 64;
    return n < grid ? static_cast<uint32_t>(n) : grid;
}
template <typename U, int kJobs>
__global__ void __launch_bounds__(kAgainThreads) values_again_kernel(const __grid_constant__ CompressParams<kJobs> p)
{
    in_stream_order();
    const uint32_t lane = threadIdx.x & 31u;
    const uint64_t nnz  = lane < p.c.jobs ? *p.job[lane].nnz_out : 0;
    const uint64_t at0  = p.c.ws_header[kHdrCursor];
    if (p.c.ws_header[kHdrPushed] != 1) return;                     // a wait ran out: every output is undefined
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
    constexpr int    kThreads = (kWorkers + 3 + WRITE_Y) * 32;
    constexpr size_t kSmem    = static_cast<size_t>(kStages) * kTile * sizeof(U) + static_cast<size_t>(kWorkers) * kRing;
    static LaunchShape shape;   // one per instantiation
    auto kernel = compress_kernel<U, FUSED, WRITE_Y, kJobs, kSegs, kWorkers, kStages, kRing>;
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

    int         max_grid = 0;
    cudaError_t e        = shape.max_grid(kernel, kThreads, kSmem, max_grid);
    if (e != cudaSuccess) return e;
    if (max_grid > 32 * kMaxWindows) max_grid = 32 * kMaxWindows;
    if (compress_max_ctas() != 0 && static_cast<uint32_t>(max_grid) > compress_max_ctas()) max_grid = static_cast<int>(compress_max_ctas());
    const uint32_t grid = tiles < static_cast<uint64_t>(max_grid) ? static_cast<uint32_t>(tiles) : static_cast<uint32_t>(max_grid);

    // the deal: tile t of tensor k goes to CTA (rot_k + t) mod grid; descriptors tensor after tensor
    uint64_t dealt = 0;
    for (uint32_t k = 0; k < count; ++k) {
        p.job[k].rot    = static_cast<uint32_t>(dealt % grid);
        p.job[k].desc0  = static_cast<uint32_t>(dealt);
        dealt += p.job[k].tiles;
    }
    p.c.jobs      = count;
    p.c.ws_header = static_cast<uint64_t *>(workspace);
    p.c.ws_desc   = reinterpret_cast<uint64_t *>(static_cast<unsigned char *>(workspace) + kWsHeaderBytes);
    p.c.ws_words  = (batch_workspace_bytes(chunks, count) - kWsHeaderBytes) / 8;
    p.c.call_tag  = next_call_tag();
    p.c.wait_ns   = compress_wait_ns();
    // (with no more tiles than CTAs, CTA b takes descriptor b: what launch_waiting asks for)
    e = launch_waiting(tiles, kernel, grid, kThreads, kSmem, stream, p);
    if (e != cudaSuccess || p.c.arena == nullptr || count < 2) return e;
    return launch(values_again_kernel<U, kJobs>, again_ctas(tiles, grid), kAgainThreads, 0, stream, p);
}

template <typename U, int FUSED, bool WRITE_Y>
cudaError_t launch_typed(const CompressCommon &c, const CompressJob *jobs, uint32_t count, void *workspace, cudaStream_t stream)
{
    using S = Shape;   // as the single-tensor kernel
    return launch_shaped<U, FUSED, WRITE_Y, kMaxBatch, S::kSegs, S::kWorkers, S::kStages, S::kRing>(c, jobs, count, workspace, stream);
}

}  // namespace

cudaError_t launch_compress_batch(const CompressJob *jobs, uint32_t count, float tau, void *workspace, int dtype, int fused,
                                  const BatchArena *arena, cudaStream_t stream)
{
    // fused: 0 plain compressor, 1 threshold form (ReLU at tau = 0)
    // the dense output is written for all tensors of a launch or for none
    if (count == 0 || count > kMaxBatch || fused > 1) return cudaErrorInvalidValue;
    const bool y = jobs[0].y != nullptr;
    for (uint32_t k = 1; k < count; ++k)
        if ((jobs[k].y != nullptr) != y) return cudaErrorInvalidValue;
    CompressCommon c{};
    c.tau = tau;
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
    if (tau == 0.0f && dtype != BT_F64) {
        // the ReLU itself: decided by one compare in the element's own type (as in the single-tensor kernel)
        constexpr int kd = kFusedReluDirect;
        if (dtype == BT_F32)
            return y ? launch_typed<uint32_t, kd + BT_F32, true>(c, jobs, count, workspace, stream)
                     : launch_typed<uint32_t, kd + BT_F32, false>(c, jobs, count, workspace, stream);
        if (dtype == BT_F16)
            return y ? launch_typed<uint16_t, kd + BT_F16, true>(c, jobs, count, workspace, stream)
                     : launch_typed<uint16_t, kd + BT_F16, false>(c, jobs, count, workspace, stream);
        return y ? launch_typed<uint16_t, kd + BT_BF16, true>(c, jobs, count, workspace, stream)
                 : launch_typed<uint16_t, kd + BT_BF16, false>(c, jobs, count, workspace, stream);
    }
    switch (dtype) {
    case BT_F64:
        return y ? launch_typed<uint64_t, BT_F64, true>(c, jobs, count, workspace, stream)
                 : launch_typed<uint64_t, BT_F64, false>(c, jobs, count, workspace, stream);
    case BT_F32:
        return y ? launch_typed<uint32_t, BT_F32, true>(c, jobs, count, workspace, stream)
                 : launch_typed<uint32_t, BT_F32, false>(c, jobs, count, workspace, stream);
    case BT_F16:
        return y ? launch_typed<uint16_t, BT_F16, true>(c, jobs, count, workspace, stream)
                 : launch_typed<uint16_t, BT_F16, false>(c, jobs, count, workspace, stream);
    default:
        return y ? launch_typed<uint16_t, BT_BF16, true>(c, jobs, count, workspace, stream)
                 : launch_typed<uint16_t, BT_BF16, false>(c, jobs, count, workspace, stream);
    }
}

}  // namespace bt
