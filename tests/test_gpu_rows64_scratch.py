"""The FP64 path's scratch follows the events: a context without events has none,
small ones have little, and no call allocates any, so that its first call may be
one that the caller captures."""
import numpy as np
import pytest

from paper_2407_11349_gb300 import synth
from paper_2407_11349_gb300.hawkes import HAWKES_F64, Hawkes

pytestmark = pytest.mark.gpu

P0 = synth.DEFAULT_PARAMS


def test_small_contexts_are_small():
    torch = pytest.importorskip("torch")
    ds = synth.grid_dataset(40, 100.0, 20, 20, seed=3)
    stream = torch.cuda.Stream().cuda_stream  # the caller's: only the contexts' own buffers count
    hks = [Hawkes(0, stream).load(ds)]
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    try:
        # about 100 KB a context, 0.6 MB more with 40 events (their arrays are
        # padded to 2,048); memory comes in pieces of 2 MB
        hks += [Hawkes(0, stream) for _ in range(64)]
        empty = free - torch.cuda.mem_get_info()[0]
        assert empty <= 64 * (1 << 19)
        for h in hks[1:]:
            h.load(ds)
        assert free - torch.cuda.mem_get_info()[0] <= 64 * (1 << 20)
    finally:
        for h in hks:
            h.close()


def test_first_call_under_capture():
    torch = pytest.importorskip("torch")
    ds = synth.grid_dataset(700, 100.0, 20, 20, seed=3)
    stream = torch.cuda.Stream()
    dp = torch.tensor(P0, dtype=torch.float64, device="cuda")
    out = torch.zeros(7, dtype=torch.float64, device="cuda")
    hk = Hawkes(0, stream.cuda_stream).load(ds)
    ref = Hawkes(0).load(ds)
    try:
        graph = torch.cuda.CUDAGraph()
        torch.cuda.synchronize()
        with torch.cuda.graph(graph, stream=stream):
            hk.loglik_grad_async(dp.data_ptr(), out.data_ptr(), HAWKES_F64)
        graph.replay()
        torch.cuda.synchronize()
        assert np.array_equal(out.cpu().numpy(), np.concatenate(ref.loglik_grad(P0, HAWKES_F64), axis=None))
        assert np.array_equal(out.cpu().numpy(), np.concatenate(hk.loglik_grad(P0, HAWKES_F64), axis=None))
    finally:
        hk.close()
        ref.close()
