"""A bounded wait that runs out: the kernel must return by itself, report BT_ERR_TIMEOUT in the status
word, write nothing outside its buffers, and leave the workspace and the context usable.

The failure is made without faulting or hanging anything: a build of the library with test hooks
(tests/checking_libs.py, -DBT_TEST_HOOKS; the product library has no such entry point) sets the bound of
every wait inside the compress kernels to a few nanoseconds, far less than the first bulk copy of a tile
takes, so the first wait of every CTA runs out although nothing is wrong.  The copies already in flight
are still awaited (with their own, fixed bound) before a CTA retires.
"""
import time

import numpy as np
import pytest
import torch

from paper_2110_15362_b200 import binding as B
from paper_2110_15362_b200 import workloads as W
from tests import checking_libs as C
from tests.gpu_util import Guarded, from_raw

pytestmark = pytest.mark.gpu


@pytest.fixture()
def hooks(monkeypatch):
    L = C.hooks_lib()
    monkeypatch.setattr(B, "_lib", L)
    yield L
    L.bt_test_set_wait_ns(2_000_000_000)
    B.bt_set_max_ctas(0)


# How a launch's tiles are shared out: `ctas` 0: as its size has it; 74: dealt out to that many CTAs, a cooperative launch
def _buffers(n, dtype, cap=None):
    return (Guarded((n + 31) // 32, torch.int32), Guarded(n if cap is None else cap, dtype),
            Guarded((n + 4095) // 4096, torch.int64), Guarded(1, torch.int64), Guarded(1, torch.int32))


@pytest.mark.parametrize("kind,limit_ns,waves,ctas", [(k, ns, w, c) for k, ns in (("f32", 0), ("f32", 50), ("bf16", 100), ("f64", 50))
                                                      for w, c in ((5, 0), (5, 74), (81 if k == "bf16" else 29, 0))])
def test_wait_runs_out_then_workspace_is_reusable(hooks, oracle, kind, limit_ns, waves, ctas):
    n = 148 * 8192 * 5 + 4097 * 3 + 5          # several waves of tiles on every SM and a ragged tail
    if waves > 5:                              # so many that they are dealt out to a CTA per SM, a cooperative launch
        n = 148 * (32768 // {"f32": 4, "bf16": 2, "f64": 8}[kind]) * waves + 4097 * 3 + 5
    B.bt_set_max_ctas(ctas)
    raw_a = W.random_patterns(n, kind, 0.5, seed=41)
    raw_b = W.random_patterns(n, kind, 0.7, seed=42)
    x_a, x_b = from_raw(raw_a, kind), from_raw(raw_b, kind)
    ws = B.new_workspace(n)
    bitmap, values, prefix, nnz, status = _buffers(n, x_a.dtype)
    status.inner.fill_(-1)

    before = hooks.bt_test_set_wait_ns(limit_ns)
    assert before == 2_000_000_000              # the product's bound
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    rc = B.bt_compress(x_a, bitmap.inner, values.inner, prefix.inner, nnz.inner, ws, status.inner, check=False)
    torch.cuda.synchronize()
    took = time.perf_counter() - t0
    assert rc == B.BT_OK                        # the host saw nothing wrong: the launch itself succeeded
    assert int(status.inner.item()) == B.BT_ERR_TIMEOUT
    assert took < 1.0, f"the kernel took {took:.3f} s to give up"
    assert all(g.guards_intact() for g in (bitmap, values, prefix, nnz, status))

    # the next ordinary launch on the same workspace, other data: exactly the oracle's result
    assert hooks.bt_test_set_wait_ns(2_000_000_000) == limit_ns
    B.bt_compress(x_b, bitmap.inner, values.inner, prefix.inner, nnz.inner, ws, status.inner)
    torch.cuda.synchronize()
    c = oracle.compress(raw_b)
    assert int(status.inner.item()) == B.BT_OK and int(nnz.inner.item()) == c.nnz
    assert np.array_equal(bitmap.raw().view(np.uint32), c.bitmap)
    assert np.array_equal(prefix.raw().view(np.uint64), c.prefix)
    assert np.array_equal(values.raw()[:c.nnz], c.values)
    assert all(g.guards_intact() for g in (bitmap, values, prefix, nnz, status))


@pytest.mark.parametrize("kind,limit_ns", [("f32", 0), ("f32", 50), ("f16", 20), ("f64", 100)])
@pytest.mark.parametrize("tiles", [1, 3, 25, 148])
def test_one_tile_per_cta_with_the_dense_output(hooks, oracle, kind, limit_ns, tiles):
    """A CTA with one tile comes to the end of its stream with its only copy still under way; the first wait that runs out
    there finds the end markers already in place.  It stays until the copy has landed all the same."""
    n = tiles * 32768 // {"f32": 4, "f16": 2, "f64": 8}[kind] - 3
    raws = [W.random_patterns(n, kind, 0.5, seed=60 + i) for i in range(2)]
    x_a, x_b = (from_raw(r, kind) for r in raws)
    ws, y = B.new_workspace(n), Guarded(n, x_a.dtype)
    bitmap, values, prefix, nnz, status = _buffers(n, x_a.dtype)
    status.inner.fill_(-1)
    hooks.bt_test_set_wait_ns(limit_ns)
    t0 = time.perf_counter()
    for _ in range(20):                          # the CTAs of one launch take the place of those of the one before
        rc = B.bt_relu_fwd_compress(x_a, y.inner, bitmap.inner, values.inner, prefix.inner, nnz.inner, ws, status.inner, check=False)
        assert rc == B.BT_OK
    torch.cuda.synchronize()
    assert time.perf_counter() - t0 < 1.0 and int(status.inner.item()) == B.BT_ERR_TIMEOUT
    hooks.bt_test_set_wait_ns(2_000_000_000)
    B.bt_relu_fwd_compress(x_b, y.inner, bitmap.inner, values.inner, prefix.inner, nnz.inner, ws, status.inner)
    torch.cuda.synchronize()
    y_ref, c = oracle.relu_fwd_compress(raws[1], kind)
    assert int(status.inner.item()) == B.BT_OK and int(nnz.inner.item()) == c.nnz
    assert np.array_equal(bitmap.raw().view(np.uint32), c.bitmap) and np.array_equal(prefix.raw().view(np.uint64), c.prefix)
    assert np.array_equal(values.raw()[:c.nnz], c.values) and np.array_equal(y.raw(), y_ref)
    assert all(g.guards_intact() for g in (bitmap, values, prefix, nnz, status, y))


@pytest.mark.parametrize("ctas", [0, 74])
def test_fused_and_batched_forms_time_out_cleanly(hooks, oracle, ctas):
    B.bt_set_max_ctas(ctas)
    sizes = [8192 * 300 + 77, 5, 8192 * 40, 4096 * 3 + 1]
    raws = [W.random_patterns(n, "f16", 0.5, seed=50 + i) for i, n in enumerate(sizes)]
    xs = [from_raw(r, "f16") for r in raws]
    stashes = [B.Stash(n, torch.float16, "cuda") for n in sizes]
    ys = [Guarded(n, torch.float16) for n in sizes]
    ws = torch.empty(B.bt_batch_workspace_bytes(sizes), dtype=torch.uint8, device="cuda")
    items = B.batch_items(xs, stashes, [y.inner for y in ys])

    hooks.bt_test_set_wait_ns(20)
    t0 = time.perf_counter()
    rc = B.bt_relu_fwd_compress_batch(items, torch.float16, ws, check=False)
    torch.cuda.synchronize()
    assert rc == B.BT_OK and time.perf_counter() - t0 < 1.0
    assert stashes[0].status == B.BT_ERR_TIMEOUT          # the tensor with tiles on every SM
    assert all(y.guards_intact() for y in ys)

    hooks.bt_test_set_wait_ns(2_000_000_000)
    B.bt_relu_fwd_compress_batch(items, torch.float16, ws)
    torch.cuda.synchronize()
    for raw, st, y in zip(raws, stashes, ys):
        y_ref, c = oracle.relu_fwd_compress(raw, "f16")
        assert st.status == B.BT_OK and st.nnz == c.nnz
        assert np.array_equal(W.raw_numpy(st.bitmap).view(np.uint32), c.bitmap)
        assert np.array_equal(W.raw_numpy(st.chunk_prefix).view(np.uint64), c.prefix)
        assert np.array_equal(W.raw_numpy(st.values[:c.nnz]), c.values)
        assert np.array_equal(y.raw(), y_ref) and y.guards_intact()


@pytest.mark.parametrize("ctas", [0, 74])
@pytest.mark.parametrize("kind", ["f32", "bf16"])
def test_batched_arena_form_times_out_cleanly(hooks, oracle, kind, ctas):
    """The batched arena form under a limit of a few nanoseconds: the launch gives up by itself, and the next ordinary launch
    on the same workspace and arena is the oracle's."""
    B.bt_set_max_ctas(ctas)
    es, dt = {"f32": (4, torch.float32), "bf16": (2, torch.bfloat16)}[kind]
    sizes = [8192 * 200 + 5, 8192 * 150, 4097, 8192 * 170 + 1]
    raws = [W.random_patterns(n, kind, 0.5, seed=90 + i) for i, n in enumerate(sizes)]
    xs = [from_raw(r, kind) for r in raws]
    stashes = [B.Stash(n, dt, "cuda", values_capacity=1) for n in sizes]
    items = B.batch_items(xs, stashes)
    arena = Guarded(sum(sizes) + 3, dt)
    cursor = torch.zeros(1, dtype=torch.int64, device="cuda")
    offsets = torch.zeros(len(sizes), dtype=torch.int64, device="cuda")
    ws = torch.empty(B.bt_batch_workspace_bytes(sizes), dtype=torch.uint8, device="cuda")

    hooks.bt_test_set_wait_ns(30)
    t0 = time.perf_counter()
    rc = B.bt_compress_arena_batch(items, dt, arena.inner.view(torch.uint8), cursor, offsets, ws, check=False)
    torch.cuda.synchronize()
    assert rc == B.BT_OK and time.perf_counter() - t0 < 1.0
    assert stashes[0].status == B.BT_ERR_TIMEOUT and arena.guards_intact()

    hooks.bt_test_set_wait_ns(2_000_000_000)
    cursor.zero_()
    B.bt_compress_arena_batch(items, dt, arena.inner.view(torch.uint8), cursor, offsets, ws)
    torch.cuda.synchronize()
    at = 0
    raw_arena = arena.inner.view(torch.uint8)
    for k, raw in enumerate(raws):
        c = oracle.compress(raw)
        assert stashes[k].status == B.BT_OK and stashes[k].nnz == c.nnz and int(offsets[k].item()) == at
        assert np.array_equal(raw_arena[at:at + es * c.nnz].cpu().numpy().view(raw.dtype), c.values)
        at += (es * c.nnz + 15) // 16 * 16
    assert int(cursor.item()) == at and arena.guards_intact()


def test_batch_that_times_out_leaves_earlier_stashes_alone(hooks, oracle):
    """An arena batch that gives up may leave anything behind the cursor, but nothing in front of it: there lie the values
    of calls that reported BT_OK.  Its counts are whatever the caller's memory held; here they are such that the second tensor
    would fit behind a first one that does not, which is what the launch behind a batch looks for."""
    sizes = [8192 * 160 + 5, 8192 * 140 + 1]
    raws = [W.random_patterns(n, "f32", 0.5, seed=70 + i) for i, n in enumerate(sizes)]
    xs = [from_raw(r, "f32") for r in raws]
    new_stashes = lambda: [B.Stash(n, torch.float32, "cuda", values_capacity=1) for n in sizes]
    first, second = new_stashes(), new_stashes()
    refs = [oracle.compress(r) for r in raws]
    step = [(4 * c.nnz + 15) // 16 * 16 for c in refs]
    # room for the first batch and, behind it, for the second tensor of another one but not for the first
    arena = Guarded((sum(step) + step[1] + 64) // 4, torch.float32)
    assert step[0] > step[1] + 64
    raw_arena = arena.inner.view(torch.uint8)
    cursor = torch.zeros(1, dtype=torch.int64, device="cuda")
    offsets = torch.zeros(len(sizes), dtype=torch.int64, device="cuda")
    ws = torch.empty(B.bt_batch_workspace_bytes(sizes), dtype=torch.uint8, device="cuda")
    B.bt_compress_arena_batch(B.batch_items(xs, first), torch.float32, raw_arena, cursor, offsets, ws)
    torch.cuda.synchronize()
    assert [st.status for st in first] == [B.BT_OK] * 2 and int(cursor.item()) == sum(step)
    before = raw_arena[:sum(step)].clone()

    for st, left in zip(second, (sum(sizes), 5000)):
        st.nnz_out.fill_(left)
        st.bitmap.fill_(-1)
        st.chunk_prefix.zero_()
    hooks.bt_test_set_wait_ns(30)
    assert B.bt_compress_arena_batch(B.batch_items(xs, second), torch.float32, raw_arena, cursor, offsets, ws, check=False) == B.BT_OK
    torch.cuda.synchronize()
    assert second[0].status == B.BT_ERR_TIMEOUT and int(cursor.item()) == sum(step)
    assert torch.equal(raw_arena[:sum(step)], before) and arena.guards_intact()

    # and the launch behind a batch is back at work in the next one: the second tensor whole behind a first that does not fit
    hooks.bt_test_set_wait_ns(2_000_000_000)
    B.bt_compress_arena_batch(B.batch_items(xs, second), torch.float32, raw_arena, cursor, offsets, ws)
    torch.cuda.synchronize()
    assert [st.status for st in second] == [B.BT_ERR_CAPACITY, B.BT_OK] and int(offsets[1].item()) == sum(step)
    assert np.array_equal(raw_arena[sum(step):sum(step) + 4 * refs[1].nnz].cpu().numpy().view(np.uint32), refs[1].values)
    assert int(cursor.item()) == sum(step) + step[1] and torch.equal(raw_arena[:sum(step)], before) and arena.guards_intact()
