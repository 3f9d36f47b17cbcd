"""How the compress launches share out their tiles: a CTA per tile up to one wave, tiles of CTAs that have not started taken
over by those that run above it (always with the dense output, up to twenty waves without), dealt out beforehand to resident
CTAs beyond that.  Sizes on both sides of every line, ragged last tiles, against the oracle; and launches that get
the SMs late, because others on streams of their own hold them."""
import numpy as np
import pytest
import torch

from paper_2110_15362_b200 import binding as B
from paper_2110_15362_b200 import workloads as W

pytestmark = pytest.mark.gpu

TILE_BYTES = 32768
SIZE = {"f32": 4, "bf16": 2, "f64": 8}


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
@pytest.mark.parametrize("waves,more", [(1, -1), (1, 0), (1, 1), (2, 1), (20, 0), (20, 1)])
def test_lines_of_the_rule(G, oracle, kind, want_y, waves, more):
    tiles = waves * _sms() + more
    n = tiles * TILE_BYTES // SIZE[kind] - 4099                  # the last tile is ragged
    x = W.near_threshold_patterns(n, kind, seed=waves + more + 2)
    y_ref, c = oracle.prune_fwd_compress(x, kind, 0.05)
    g = G.gpu_compress(G.from_raw(x, kind), tau=0.05, want_y=want_y)
    assert g.guards_ok and g.status == B.BT_OK and g.nnz == c.nnz
    assert np.array_equal(g.bitmap, c.bitmap) and np.array_equal(g.prefix, c.prefix)
    assert np.array_equal(g.values.view(c.values.dtype), c.values)
    if want_y:
        assert np.array_equal(g.y, y_ref)


def test_launches_that_get_the_sms_late(oracle):
    """Three streams, one of them of higher priority, keep one another's CTAs from starting; every stash is the oracle's."""
    dev = torch.device("cuda")
    tiles = 6 * _sms() + 5
    cases = []
    for k, kind in enumerate(("f32", "bf16", "f32")):
        n = tiles * TILE_BYTES // SIZE[kind] - 77 * (k + 1)
        raw = W.random_patterns(n, kind, 0.5, seed=300 + k)
        x = torch.from_numpy(raw.view(np.int32 if kind == "f32" else np.int16)).to(dev).view(torch.float32 if kind == "f32" else torch.bfloat16)
        cases.append((oracle.compress(raw), x, B.Stash(n, x.dtype, dev), B.new_workspace(n, dev), torch.cuda.Stream(priority=-1 if k == 1 else 0)))
    torch.cuda.synchronize()
    for _ in range(20):
        for _, x, st, ws, stream in cases:
            with torch.cuda.stream(stream):
                B.bt_compress(x, st.bitmap, st.values, st.chunk_prefix, st.nnz_out, ws, st.dev_status)
    torch.cuda.synchronize()
    for c, _, st, _, _ in cases:
        assert st.status == B.BT_OK and st.nnz == c.nnz
        assert np.array_equal(W.raw_numpy(st.bitmap).view(np.uint32), c.bitmap)
        assert np.array_equal(W.raw_numpy(st.chunk_prefix).view(np.uint64), c.prefix)
        assert np.array_equal(W.raw_numpy(st.values[:c.nnz]), c.values)
