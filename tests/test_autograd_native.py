"""The native node of the stashing ReLU and the native restore: what they refuse (no GPU), and on the GPU every form of the
node against torch.relu -- inputs and gradients that are views, in place, retained and released graphs, empty tensors."""
import pytest
import torch

from paper_2110_15362_b200 import autograd as A
from paper_2110_15362_b200 import binding as B


def test_arguments_are_checked():
    x = torch.zeros(64)
    none = (0, 0, 0, 0, False, None, 0, None, None, None, 0, None)
    with pytest.raises(TypeError):
        A._native.relu_stash(x)
    with pytest.raises(TypeError):
        A._native.relu_stash(None, *none)
    with pytest.raises(RuntimeError, match="CUDA"):
        A._native.relu_stash(x, *none)
    with pytest.raises(OverflowError):
        A._native.relu_stash(x, -1 << 70, *none[1:])
    with pytest.raises(TypeError):
        A._native.restore(0, x, None, False, 0, [64], torch.float32)
    with pytest.raises(RuntimeError, match="record"):
        A._native.restore(0, torch.zeros(8, dtype=torch.uint8), None, False, 0, (64,), torch.float32)


def _views(kind, dtype):
    """(a leaf, a function of it whose result the ReLU takes)"""
    g = torch.Generator().manual_seed(7)
    if kind == "empty":
        return torch.zeros(0, device="cuda", dtype=dtype), lambda t: t * 1
    t = torch.randn(96, 203, generator=g).to(dtype).cuda()
    if kind == "transposed":
        return t, lambda t: (t * 1).t()
    if kind == "misaligned":
        return t, lambda t: (t * 1).flatten()[1:]
    return t, lambda t: t * 1


@pytest.mark.gpu
@pytest.mark.parametrize("form", ["exact", "full", "arena", "bits", "bits_alone", "alone", "narrow", "narrow_arena"])
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16, torch.float64])
@pytest.mark.parametrize("kind", ["whole", "transposed", "misaligned", "empty"])
@pytest.mark.parametrize("inplace", [False, True])
def test_every_form_of_the_node(form, dtype, kind, inplace):
    opts = {"exact": {}, "full": {"two_pass": False}, "arena": {"arena_bytes": 1 << 20}, "bits": {}, "narrow": {"narrow": torch.bfloat16},
            "narrow_arena": {"narrow": torch.bfloat16, "arena_bytes": 1 << 20}}
    hooks = A.stash_saved_activations(min_numel=16, **opts[form]) if form in opts else None
    t, view = _views(kind, dtype)
    leaf, ref = t.clone().requires_grad_(), t.clone().requires_grad_()

    def step():
        h = view(leaf)
        # an activation may be written over its input only where that is not a view of something saved
        return A.relu_stash(h, hooks, inplace=inplace, keep_values=not form.startswith("bits"))

    if hooks is not None:
        with hooks:
            y = step()
    else:
        y = step()
    y_ref = torch.relu(view(ref))
    assert torch.equal(y, y_ref) and y.requires_grad
    for grad in (torch.randn_like(y_ref), torch.ones((), device="cuda", dtype=dtype).expand_as(y_ref)):
        leaf.grad = ref.grad = None
        y.backward(grad, retain_graph=True)
        y_ref.backward(grad, retain_graph=True)
        assert torch.equal(leaf.grad, ref.grad)
    y.sum().backward()
    with pytest.raises(RuntimeError, match="second time"):
        y.sum().backward()
    if hooks is not None:
        packed = getattr(y, "_bt_packed", None)
        assert (packed is None) == form.startswith("bits")
        if packed is not None and t.numel():
            back, want = packed.unpack(), y.detach()
            assert torch.equal(back, want.bfloat16().to(dtype) if form.startswith("narrow") and dtype == torch.float32 else want)
        hooks.check_statuses()
    with torch.no_grad():
        assert not A.relu_stash(view(ref), keep_values=not form.startswith("bits")).requires_grad


@pytest.mark.gpu
@pytest.mark.parametrize("two_pass", [True, False])
def test_a_hook_that_raises_leaves_no_kernel_writing_the_threads_words(two_pass):
    """The count of an exact-size stash goes to page-locked words of the thread; a hook that raises behind the launch must not
    leave that store to a later moment, when the thread may be waiting for another stash's count on another stream."""
    class Raised(Exception):
        pass

    def pack(t):
        raise Raised

    x = torch.randn(1 << 16, device="cuda").requires_grad_()
    hooks = A.stash_saved_activations(min_numel=16, two_pass=two_pass)
    with hooks:
        A.relu_stash(x * 1, hooks).sum().backward()
    torch.cuda.synchronize()
    h, host = x.detach().clone().requires_grad_() * 1, A._read_back()
    host.view[:] = -1
    torch.cuda._sleep(100_000_000)
    with torch.autograd.graph.saved_tensors_hooks(pack, lambda t: t):
        with pytest.raises(Raised):
            A.relu_stash(h, hooks)
    seen = int(host.view[0])
    torch.cuda.synchronize()
    assert seen == int((h > 0).sum())
    with hooks:
        y = A.relu_stash(x * 1, hooks)
    assert torch.equal(y, torch.relu(x)) and y._bt_packed.nnz == seen


@pytest.mark.gpu
@pytest.mark.parametrize("mode", ["arena", "full"])
def test_a_dropped_context_on_a_side_stream(mode):
    """A context's buffers go back to the allocator as soon as it is dropped, but to no other stream before the one that the
    pass ran on is done with them."""
    n, opts = 3 << 20, {"arena": {"arena_bytes": 37 << 20}, "full": {"two_pass": False}}[mode]
    x = torch.randn(n, device="cuda").requires_grad_()
    hooks = A.stash_saved_activations(min_numel=16, **opts)
    with hooks:
        A.relu_stash(x.detach(), hooks)                                  # the scratch buffers: the default stream's
    side = torch.cuda.Stream()
    used = {t.data_ptr(): t.numel() * t.element_size() for t in (*hooks.scratch.kept, *hooks.scratch.ws.values(), *hooks.scratch.values.values())}
    assert len(used) == (3 if mode == "arena" else 2)

    def spare():
        return [torch.empty(size, dtype=torch.uint8, device="cuda") for size in used.values() for _ in range(4)]
    spare()                                                              # (device allocations would wait for the pause below)
    for pause in (0, 400_000_000):
        torch.cuda.synchronize()
        x.grad = None
        with torch.cuda.stream(side):
            with hooks:
                y = A.relu_stash(x * 1, hooks) * 2
                z = (y * y).sum()
            hooks.check_statuses()                                       # its host read here, not behind the pause
            torch.cuda._sleep(pause)
            z.backward()
        del y, z
    del hooks
    taken = spare()
    assert not side.query()                                              # the backward pass is still to run
    assert not set(used) & {t.data_ptr() for t in taken}
    torch.cuda.synchronize()
    r = x.detach().clone().requires_grad_()
    ((torch.relu(r * 1) * 2) ** 2).sum().backward()
    assert torch.equal(x.grad, r.grad)
