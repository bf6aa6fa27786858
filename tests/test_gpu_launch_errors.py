"""A launch that the runtime refuses is reported by the call that made it, and by no later one."""
import ctypes

import pytest
import torch

import paper_2602_00523_b200 as sage
from helpers import dev_f32, dev_i32

pytestmark = pytest.mark.gpu


def test_a_refused_launch_is_not_reported_by_the_next_call():
    cudart = ctypes.CDLL("libcudart.so.12")              # the one that torch has loaded
    path_len, window, count, d_max = dev_i32([3]), dev_i32([[0] * 10]), dev_i32([0]), dev_f32([8.0])
    pool = torch.zeros(1, 2, 1, 64, 128, dtype=torch.bfloat16, device="cuda")
    table, seq, path, one = dev_i32([[0, 1]]), dev_i32([10]), dev_i32([[0, -1]]), dev_i32([1])
    logits = torch.randn(2, 4096, device="cuda")
    policy, stream = sage.make_history_policy(), torch.cuda.Stream()
    sage.sage_compact_kv(pool, pool.clone(), table, seq, path, one)
    sage.sage_update_history(path_len, policy, window, count, d_max)
    out = sage.sage_expand_topk(logits, 2, 2)
    ws = torch.empty(sage.sage_expand_topk_workspace_size(2, 4096), dtype=torch.uint8, device="cuda")
    root, offsets = dev_i32([-1]), dev_i32([0, 1])
    accepted = sage.sage_accept(root, one, one, offsets, 2)
    torch.cuda.synchronize()
    handle = ctypes.c_void_p(stream.cuda_stream)
    assert cudart.cudaStreamBeginCapture(handle, 1) == 0
    try:
        assert cudart.cudaStreamSynchronize(handle) != 0           # not allowed: spoils the capture, every launch into it is refused
        for call in (lambda: sage.sage_compact_kv(pool, pool, table, seq, path, one, stream=stream),
                     lambda: sage.sage_expand_topk(logits, 2, 2, out=out, ws=ws, stream=stream),
                     lambda: sage.sage_accept(root, one, one, offsets, 2, out=accepted, stream=stream)):
            with pytest.raises(sage.SageError) as e:
                call()
            assert e.value.code == sage.SAGE_ERR_CUDA
            sage.sage_update_history(path_len, policy, window, count, d_max)       # on the stream that is not captured
    finally:
        graph = ctypes.c_void_p()
        cudart.cudaStreamEndCapture(handle, ctypes.byref(graph))
        cudart.cudaGetLastError()
    torch.cuda.synchronize()
    assert count.item() == 4 and seq.item() == 11
