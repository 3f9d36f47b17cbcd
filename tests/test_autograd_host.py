"""Host side of the autograd integration, without a GPU: the words that calls report in, and what a context keeps alive."""
import gc
import threading
import weakref

import pytest
import torch

from paper_2110_15362_b200 import autograd as A
from paper_2110_15362_b200 import binding as B


def _hooks(**kw):
    return A.stash_saved_activations(min_numel=16, device="cpu", **kw)


@pytest.mark.parametrize("keep_values", [True, False])
def test_a_call_that_raises_leaves_no_status_word(keep_values):
    """The native node refuses a CPU tensor after its status word is handed out; nothing will ever write that word."""
    hooks = _hooks(arena_bytes=1 << 16)
    with pytest.raises(RuntimeError, match="CUDA"):
        A.relu_stash(torch.zeros(64), hooks, keep_values=keep_values)
    assert not hooks.statuses and not hooks.loose_statuses
    with hooks:                                  # reads the words of the pass before
        pass


@pytest.mark.parametrize("call", [A.relu6_stash, A.relu_maxpool2x2_stash])
def test_a_call_that_fails_leaves_no_status_word(call, monkeypatch):
    class Calls:
        def __getattr__(self, name):
            return lambda *args: B.BT_ERR_WORKSPACE if "arena" in name else B.BT_OK
    hooks = _hooks(arena_bytes=1 << 16)
    monkeypatch.setattr(B, "_calls", Calls)
    monkeypatch.setattr(B, "_tensor_calls", Calls)
    monkeypatch.setattr(B, "_stream", lambda stream: 0)
    with pytest.raises(B.BitTrainError):
        call(torch.zeros(4, 16), hooks)
    assert not hooks.statuses
    with hooks:
        pass


def test_status_words_are_distinct_and_read_once_made():
    words = A._StatusWords()
    taken = [words.next(torch.device("cpu")) for _ in range(3 * A._StatusBlock.SIZE + 5)]
    assert len({w[0] for w in taken}) == len(taken) and not words
    for k, w in enumerate(taken):
        w[1].words[w[2]] = k
        if k % 3 == 0:
            words.made(w)
    assert words and sorted(words.drain()) == list(range(0, len(taken), 3)) and not words
    # a word handed out before a check and made after it still has its memory
    w = words.next(torch.device("cpu"))
    assert words.drain() == []
    w[1].words[w[2]] = 7
    words.made(w)
    assert words.drain() == [7] and words.drain() == []


def test_status_words_of_several_threads():
    words, got, seen = A._StatusWords(), [], []

    def take(base):
        for k in range(500):
            w = words.next(torch.device("cpu"))
            w[1].words[w[2]] = base + k
            words.made(w)
            if k % 50 == 49:
                seen.extend(words.drain())
    threads = [threading.Thread(target=take, args=(1000 * t,)) for t in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    got = sorted(seen + words.drain())
    assert got == sorted(1000 * t + k for t in range(4) for k in range(500))


@pytest.mark.parametrize("entered", [False, True])
def test_a_dropped_context_frees_its_arena_at_once(entered):
    gc.collect()
    gc.disable()
    try:
        hooks = _hooks(arena_bytes=1 << 16)
        arena = weakref.ref(hooks.arena)
        if entered:
            x = torch.randn(64, requires_grad=True)
            with hooks:
                y = (x * x).sum()
            y.backward()
            assert torch.equal(x.grad, 2 * x)
        del hooks
        assert arena() is None
    finally:
        gc.enable()


def test_an_entered_context_needs_no_other_reference():
    """Entered by hand and dropped: its hooks stay in force until it is left."""
    class Counted(A.stash_saved_activations):
        packed = 0

        def _pack(self, t):
            Counted.packed += 1
            return super()._pack(t)

    gone = weakref.ref(Counted(device="cpu"))
    assert gone() is None
    h = Counted(device="cpu")
    h.__enter__()
    leave = torch._C._autograd._pop_saved_tensors_default_hooks
    del h
    try:
        x = torch.randn(8, requires_grad=True)
        (x * x).sum().backward()
        assert Counted.packed == 2
    finally:
        leave()
