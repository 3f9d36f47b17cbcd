"""A launch that the runtime refuses is reported by the call it belongs to, and by no later one."""
import ctypes

import pytest
import torch

from paper_2110_15362_b200 import binding as B

pytestmark = pytest.mark.gpu

UNSUPPORTED, INVALIDATED, THREAD_LOCAL = 900, 901, 1


@pytest.mark.parametrize("refused", ["compress", "compress_many_tiles", "decompress", "relu_bwd", "relu6_bwd", "pool", "mask"])
def test_a_refused_launch_is_not_reported_again(refused):
    """The stream's capture is made invalid by a wait inside it, so the runtime refuses what is launched there."""
    n = 40000 if refused != "compress_many_tiles" else 1 << 23
    x = torch.randn(n, device="cuda")
    st, ws, out = B.Stash(n, x.dtype), B.new_workspace(n), torch.empty_like(x)
    good = lambda: B.bt_compress(x, st.bitmap, st.values, st.chunk_prefix, st.nnz_out, ws, st.dev_status)   # noqa: E731
    good()
    calls = {
        "compress": lambda s: B.bt_compress(x, st.bitmap, st.values, st.chunk_prefix, st.nnz_out, ws, st.dev_status, stream=s, check=False),
        "decompress": lambda s: B.bt_decompress(st.bitmap, st.values, st.chunk_prefix, out, stream=s, check=False),
        "relu_bwd": lambda s: B.bt_relu_bwd_from_bitmap(st.bitmap, x, out, stream=s, check=False),
        "relu6_bwd": lambda s: B.bt_relu6_bwd_from_stash(st.bitmap, st.values, st.chunk_prefix, x, out, stream=s, check=False),
        "pool": lambda s: B.bt_maxpool2x2_fwd(x, out, None, planes=1, height=n // 4, width=4, stream=s, check=False),
        "mask": lambda s: B.bt_mask_compress(x, st.bitmap, st.chunk_prefix, None, st.values, stream=s, check=False),
    }
    torch.cuda.synchronize()
    rt, stream = ctypes.CDLL("libcudart.so.12"), torch.cuda.Stream()
    handle, graph = ctypes.c_void_p(stream.cuda_stream), ctypes.c_void_p()
    assert rt.cudaStreamBeginCapture(handle, THREAD_LOCAL) == 0
    try:
        assert rt.cudaStreamSynchronize(handle) == UNSUPPORTED
        assert calls[refused if refused != "compress_many_tiles" else "compress"](stream) == B.BT_ERR_CUDA
    finally:
        assert rt.cudaStreamEndCapture(handle, ctypes.byref(graph)) == INVALIDATED
        rt.cudaGetLastError()                                        # torch's runtime forgets the two as well
    for name, call in calls.items():
        assert call(None) == B.BT_OK, name
    staging = torch.empty(B.bt_host_staging_bytes(n, x.dtype), dtype=torch.uint8, device="cuda")
    host = [t.pin_memory() for t in (x.cpu(), st.bitmap.cpu(), st.values.cpu(), st.chunk_prefix.cpu(), torch.zeros(1, dtype=torch.int64))]
    B.bt_compress_host(*host, staging)
    torch.cuda.synchronize()
    assert int(host[4]) == st.nnz
