"""Sizes at the edges of the kernels' own units, against the oracle: segments and blocks of the compressors (a worker's
2048 two-byte, 1024 four-byte, 512 eight-byte elements; blocks of 1024), parts of the staged walk (4096 bytes), calls
without room for values over more tiles than a CTA's queue holds, and pooling rows of every kind."""
import numpy as np
import pytest
import torch

from paper_2110_15362_b200 import binding as B
from paper_2110_15362_b200 import workloads as W
from tests.gpu_util import Guarded, from_raw

pytestmark = pytest.mark.gpu

UNIT = {"f32": 1024, "bf16": 2048, "f16": 2048, "f64": 512}


@pytest.fixture(scope="module")
def G():
    from tests import gpu_util
    return gpu_util


@pytest.mark.parametrize("kind", ["f32", "bf16", "f64"])
@pytest.mark.parametrize("units,off", [(1, -1), (1, 0), (1, 1), (2, 31), (7, -33), (8, 0), (8, 1), (9, 130), (24, -1), (25, 2), (65, 127)])
def test_sizes_around_segments_and_parts(G, oracle, kind, units, off):
    n = units * UNIT[kind] + off
    for zf in (0.0, 0.5, 0.98):
        x = W.random_patterns(n, kind, zf, seed=n + int(100 * zf))
        c = oracle.compress(x)
        g = G.gpu_compress(from_raw(x, kind))
        assert g.guards_ok and g.status == B.BT_OK and g.nnz == c.nnz
        assert np.array_equal(g.bitmap, c.bitmap) and np.array_equal(g.prefix, c.prefix) and np.array_equal(g.values, c.values)
        back, ok = G.gpu_decompress(c.bitmap, c.values, c.prefix, n, kind)
        assert ok and np.array_equal(back, x)


@pytest.mark.parametrize("kind", ["f32", "bf16", "f64"])
@pytest.mark.parametrize("seg", [0, 3, 7])
def test_ragged_tile_in_a_used_slot(G, oracle, kind, seg):
    """The fifth tile of the only CTA ends within segment `seg`, around 16-byte units, over the dense data of the second."""
    unit = 16 // np.dtype(W.random_patterns(1, kind, 0.0, seed=0).dtype).itemsize
    before = B.bt_set_max_ctas(1)
    try:
        for off in (1, unit - 1, unit, unit + 1, UNIT[kind] // 2, UNIT[kind] - unit - 1, UNIT[kind] - 1, UNIT[kind]):
            n = (4 * 8 + seg) * UNIT[kind] + off
            x = W.random_patterns(n, kind, 0.01, seed=n)
            y_ref, c = oracle.prune_fwd_compress(x, kind, 0.0)
            g = G.gpu_compress(from_raw(x, kind), relu=True, want_y=True)
            assert g.guards_ok and g.status == B.BT_OK and g.nnz == c.nnz and np.array_equal(g.y, y_ref)
            assert np.array_equal(g.bitmap, c.bitmap) and np.array_equal(g.prefix, c.prefix) and np.array_equal(g.values, c.values)
    finally:
        B.bt_set_max_ctas(before)


@pytest.mark.parametrize("kind", ["f32", "bf16"])
def test_one_tile_per_cta_on_two_streams(oracle, kind):
    """Launches of one tile per CTA need not be resident as a whole: two streams, each launch with more than half the SMs,
    alone and as batches, against the oracle; the largest such launch and the next tile."""
    B.lib()
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    tile = 8 * UNIT[kind]
    sizes = [tile * sms, tile * (sms - 1) + 1, tile * sms + 1, tile * (sms - 20) - 5]
    raws = [W.random_patterns(n, kind, 0.5, seed=n % 1000) for n in sizes]
    refs = [oracle.compress(r) for r in raws]
    xs = [from_raw(r, kind) for r in raws]
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    half = [from_raw(r[: r.size // 2], kind) for r in raws[:2]]      # batches: two tensors that fill the SMs together
    for _ in range(5):
        stashes, wss = [B.Stash(n, x.dtype) for n, x in zip(sizes, xs)], [B.new_workspace(n) for n in sizes]
        bst = [[B.Stash(h.numel(), h.dtype) for h in half] for _ in streams]
        bws = [torch.empty(B.bt_batch_workspace_bytes([h.numel() for h in half]), dtype=torch.uint8, device="cuda") for _ in streams]
        torch.cuda.synchronize()
        for k in range(len(sizes)):
            st, s = stashes[k], streams[k % 2]
            B.bt_compress(xs[k], st.bitmap, st.values, st.chunk_prefix, st.nnz_out, wss[k], st.dev_status, stream=s)
            if k < 2:
                B.bt_compress_batch(B.batch_items(half, bst[k]), half[0].dtype, bws[k], stream=s)
        torch.cuda.synchronize()
        for st, c in zip(stashes, refs):
            assert st.status == B.BT_OK and st.nnz == c.nnz
            assert np.array_equal(W.raw_numpy(st.bitmap).view(np.uint32), c.bitmap)
            assert np.array_equal(W.raw_numpy(st.values[: c.nnz]), c.values)
        for pair in bst:
            for st, r in zip(pair, raws):
                c = oracle.compress(r[: r.size // 2])
                assert st.status == B.BT_OK and st.nnz == c.nnz and np.array_equal(W.raw_numpy(st.values[: c.nnz]), c.values)


@pytest.mark.parametrize("kind", ["f32", "bf16", "f64"])
@pytest.mark.parametrize("fused", [False, True])
@pytest.mark.parametrize("tiles", [1, 2 * 8, 2 * 8 + 1, 2 * 19 + 1])
def test_no_room_for_values(oracle, kind, fused, tiles):
    """Bitmap, prefix array and count with a capacity of 0: two CTAs, up to twenty tiles each (a CTA's queue holds eight)."""
    n = tiles * 8 * UNIT[kind] - 77
    x = W.random_patterns(n, kind, 0.5, seed=tiles)
    t = from_raw(x, kind)
    y_ref, c = oracle.prune_fwd_compress(x, kind, 0.0) if fused else (None, oracle.compress(x))
    bitmap, prefix = Guarded((n + 31) // 32, torch.int32), Guarded((n + 4095) // 4096, torch.int64)
    nnz, status, y = Guarded(1, torch.int64), Guarded(1, torch.int32), Guarded(n, t.dtype)
    before = B.bt_set_max_ctas(2)
    try:
        tail = (bitmap.inner, None, prefix.inner, nnz.inner, B.new_workspace(n), status.inner)
        if fused:
            B.bt_relu_fwd_compress(t, y.inner, *tail, n=n, values_capacity=0)
        else:
            B.bt_compress(t, *tail, n=n, values_capacity=0)
        torch.cuda.synchronize()
    finally:
        B.bt_set_max_ctas(before)
    assert int(nnz.inner.item()) == c.nnz
    assert int(status.inner.item()) == (B.BT_ERR_CAPACITY if c.nnz else B.BT_OK)
    assert np.array_equal(bitmap.raw().view(np.uint32), c.bitmap) and np.array_equal(prefix.raw().view(np.uint64), c.prefix)
    if fused:
        assert np.array_equal(y.raw(), y_ref)
    assert all(g.guards_intact() for g in (bitmap, prefix, nnz, status, y))


# (planes, height, width): whole vectors of a row or not, odd numbers of outputs, rows of one output, blocks of threads
POOL = [(1, 2, 2), (3, 2, 2), (1, 2, 6), (5, 6, 2), (7, 2, 14), (1, 14, 14), (9, 14, 14), (3, 30, 30), (2, 28, 28), (1, 2, 1030), (1, 34, 62),
        (1, 2, 8), (3, 2, 8), (1, 2, 4096), (1, 2, 4104), (3, 18, 24), (5, 64, 40)]


@pytest.mark.parametrize("kind", ["f32", "bf16", "f16", "f64"])
@pytest.mark.parametrize("shape", POOL)
def test_pooling_rows(oracle, kind, shape):
    planes, h, w = shape
    n, m = planes * h * w, planes * h * w // 4
    x = W.random_patterns(n, kind, 0.4, seed=n)
    y_ref, codes_ref = oracle.maxpool2x2_fwd(x, planes, h, w, kind)
    t = from_raw(x, kind)
    y, codes, gin = Guarded(m, t.dtype), Guarded((m + 15) // 16, torch.int32), Guarded(n, t.dtype)
    B.bt_maxpool2x2_fwd(t, y.inner, codes.inner, planes=planes, height=h, width=w)
    torch.cuda.synchronize()
    assert np.array_equal(y.raw(), y_ref) and np.array_equal(codes.raw().view(np.uint32), codes_ref)
    g = W.random_patterns(m, kind, 0.1, seed=m + 1)
    B.bt_maxpool2x2_bwd(codes.inner, from_raw(g, kind), gin.inner, planes=planes, height=h, width=w)
    torch.cuda.synchronize()
    assert np.array_equal(gin.raw(), oracle.maxpool2x2_bwd(codes_ref, g, planes, h, w))
    # under the bitmap of the pooled output: the gradient of an output whose bit is clear counts as zero
    c = oracle.compress(y_ref)
    bitmap = torch.from_numpy(c.bitmap.view(np.int32).copy()).cuda()
    B.bt_maxpool2x2_bwd_masked(codes.inner, bitmap, from_raw(g, kind), gin.inner, planes=planes, height=h, width=w)
    torch.cuda.synchronize()
    assert np.array_equal(gin.raw(), oracle.maxpool2x2_bwd(codes_ref, oracle.relu_bwd_from_bitmap(c.bitmap, g), planes, h, w))
    assert all(q.guards_intact() for q in (y, codes, gin))
