"""A context of the default stream is asked about its bricks while another stream captures (needs a
GPU)."""
import ctypes

import pytest

from paper_1507_07294_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def test_the_question_leaves_no_error_behind():
    """The default stream's state cannot be asked for while a stream that synchronises with it
    captures; the next caller that looks for an error must not find that one."""
    import torch

    from paper_1507_07294_gb300 import lbm as L
    cudart = torch.cuda.cudart()
    with L.Solver(I.droplet(n=16, R=4.0), stream=0) as s:
        s.step(2)
        torch.cuda.synchronize()
        handle = ctypes.c_uint64(0)  # a blocking stream: PyTorch's own do not synchronise with 0
        assert int(cudart.cudaStreamCreate(ctypes.addressof(handle))) == 0
        stream = torch.cuda.ExternalStream(handle.value)
        x = torch.ones(4, device="cuda")
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            y = x + 1
            assert L.lbm_get_tuning(s.ctx, L.LBM_TUNE_BRICKS) == 0
            z = y + 1
        graph.replay()
        torch.cuda.synchronize()
        assert z.tolist() == [3.0] * 4
        assert L.lbm_get_tuning(s.ctx, L.LBM_TUNE_BRICKS) == 1
        del graph
        torch.cuda.synchronize()
        cudart.cudaStreamDestroy(handle.value)
