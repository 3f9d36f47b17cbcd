"""How the compress launches share out their tiles: a CTA per tile up to one wave, tiles of CTAs that have not started taken
over by those that run above it (always with the dense output; without it up to 28 waves, 80 of 2-byte types, 20 of a batch), dealt
out beforehand to resident CTAs beyond that.  Sizes on both sides of every line, ragged last tiles, against the oracle; and launches that get
the SMs late, because others on streams of their own hold them."""
import numpy as np
import pytest
import torch

from paper_2110_15362_b200 import binding as B
from paper_2110_15362_b200 import workloads as W
from tests import test_gpu_batch
from tests.gpu_util import TDT, from_raw

pytestmark = pytest.mark.gpu

TILE_BYTES = 32768
SIZE = {"f32": 4, "bf16": 2, "f64": 8}
LINE = {"f32": 28, "bf16": 80, "f64": 28}                        # waves of tiles of one tensor without the dense output


@pytest.fixture(scope="module")
def G():
    assert torch.cuda.is_available(), "these tests need a CUDA device"
    from tests import gpu_util
    B.lib()
    return gpu_util


def _sms():
    return torch.cuda.get_device_properties(0).multi_processor_count


@pytest.mark.parametrize("kind", ["f32", "bf16", "f64"])
@pytest.mark.parametrize("want_y", [False, True])
@pytest.mark.parametrize("waves,more", [(1, -1), (1, 0), (1, 1), (2, 1), (None, 0), (None, 1)])
def test_lines_of_the_rule(G, oracle, kind, want_y, waves, more):
    waves = waves or (20 if want_y else LINE[kind])
    tiles = waves * _sms() + more
    n = tiles * TILE_BYTES // SIZE[kind] - 1027                  # the last tile is ragged
    assert -(-n * SIZE[kind] // TILE_BYTES) == tiles
    x = W.near_threshold_patterns(n, kind, seed=waves + more + 2)
    y_ref, c = oracle.prune_fwd_compress(x, kind, 0.05)
    g = G.gpu_compress(G.from_raw(x, kind), tau=0.05, want_y=want_y)
    assert g.guards_ok and g.status == B.BT_OK and g.nnz == c.nnz
    assert np.array_equal(g.bitmap, c.bitmap) and np.array_equal(g.prefix, c.prefix)
    assert np.array_equal(g.values.view(c.values.dtype), c.values)
    if want_y:
        assert np.array_equal(g.y, y_ref)


@pytest.mark.parametrize("kind", ["f32", "bf16", "f64"])
@pytest.mark.parametrize("fused,want_y", [(False, False), (True, False), (True, True)])
def test_batch_beyond_twenty_waves(oracle, kind, fused, want_y):
    """Tensors of a tile, of a wave and of many, ragged, in one launch of more than twenty waves of tiles."""
    per_tile, sms = TILE_BYTES // SIZE[kind], _sms()
    sizes = [per_tile * t - r for t, r in ((1, 5), (sms, 0), (12 * sms + 3, 1027), (2, 1), (7 * sms + 40, 7), (1, per_tile - 1), (sms // 2, 33))]
    assert sum(-(-n // per_tile) for n in sizes) > 20 * sms
    raws, sts, ys, _ = test_gpu_batch.run_batch(kind, sizes, 5000, fused, want_y)
    test_gpu_batch.check_batch(oracle, kind, raws, sts, ys, fused)


@pytest.mark.parametrize("kind", ["f32", "bf16", "f64"])
def test_arena_batch_beyond_twenty_waves(oracle, kind):
    es, sms = SIZE[kind], _sms()
    sizes = [TILE_BYTES // es * t - r for t, r in ((1, 5), (13 * sms + 3, 1027), (2, 1), (7 * sms + 40, 7), (sms // 2, 33))]
    raws, sts, _, arena, cursor, offsets = test_gpu_batch._arena_batch(kind, sizes, 6000, False, sum(sizes) * es)
    at = 0
    for k, raw in enumerate(raws):
        c = oracle.compress(raw)
        assert sts[k].status == B.BT_OK and sts[k].nnz == c.nnz and int(offsets[k].item()) == at
        assert np.array_equal(W.raw_numpy(sts[k].chunk_prefix).view(np.uint64), c.prefix)
        assert np.array_equal(arena[at:at + c.nnz * es].cpu().numpy().view(raw.dtype), c.values)
        at += (c.nnz * es + 15) // 16 * 16
    assert int(cursor.item()) == at and bool((arena[at:] == 0x5A).all().item())


def test_launches_that_get_the_sms_late(oracle):
    """Streams, one of them of higher priority, keep one another's CTAs from starting, so that a CTA's first tile can lie far behind
    tile 0 and more descriptors in front of it than are read at a time: with and without the dense output, and a batch.
    Every stash of every repetition is the oracle's."""
    dev, reps = torch.device("cuda"), 12
    tiles = 6 * _sms() + 5
    bits = {2: torch.int16, 4: torch.int32}
    work = []
    for k, (kind, form) in enumerate((("f32", "plain"), ("bf16", "plain"), ("f32", "y"), ("bf16", "batch"))):
        per_tile = TILE_BYTES // SIZE[kind]
        n = tiles * per_tile - 77 * (k + 1)
        sizes = [n // 3, 5, n - n // 3 - 5] if form == "batch" else [n]
        raws = [W.random_patterns(m, kind, 0.5, seed=300 + 10 * k + i) for i, m in enumerate(sizes)]
        refs = [oracle.relu_fwd_compress(r, kind) if form == "y" else (None, oracle.compress(r)) for r in raws]
        xs = [from_raw(r, kind) for r in raws]
        sts = [[B.Stash(m, TDT[kind], dev) for m in sizes] for _ in range(reps)]
        for st in sum(sts, []):
            st.nnz_out.fill_(-1), st.dev_status.fill_(-1)
        ys = [torch.empty_like(xs[0]) for _ in range(reps)] if form == "y" else None
        ws = torch.empty(max(B.bt_batch_workspace_bytes(sizes), B.bt_workspace_bytes(n)), dtype=torch.uint8, device=dev)
        work.append((form, refs, xs, sts, ys, ws, torch.cuda.Stream(priority=-1 if k == 1 else 0), [B.batch_items(xs, s) for s in sts]))
    torch.cuda.synchronize()
    for rep in range(reps):
        for form, _, xs, sts, ys, ws, stream, items in work:
            st = sts[rep][0]
            with torch.cuda.stream(stream):
                if form == "batch":
                    B.bt_compress_batch(items[rep], xs[0].dtype, ws)
                elif form == "y":
                    B.bt_relu_fwd_compress(xs[0], ys[rep], st.bitmap, st.values, st.chunk_prefix, st.nnz_out, ws, st.dev_status)
                else:
                    B.bt_compress(xs[0], st.bitmap, st.values, st.chunk_prefix, st.nnz_out, ws, st.dev_status)
    torch.cuda.synchronize()
    for form, refs, xs, sts, ys, _, _, _ in work:
        for i, (y_ref, c) in enumerate(refs):
            es = c.values.dtype.itemsize
            want = [torch.from_numpy(a.view({2: np.int16, 4: np.int32, 8: np.int64}[a.dtype.itemsize])).to(dev) for a in (c.bitmap, c.prefix, c.values)]
            for rep in range(reps):
                st = sts[rep][i]
                assert st.status == B.BT_OK and st.nnz == c.nnz, (form, rep)
                got = (st.bitmap, st.chunk_prefix, st.values[:c.nnz].view(bits[es]))
                assert all(torch.equal(a, b) for a, b in zip(got, want)), (form, rep)
                if form == "y":
                    assert np.array_equal(W.raw_numpy(ys[rep]), y_ref), rep
