"""The end of a batch whose status has been read, while a graph of other work is captured by this thread or
another: the capture goes on."""
import threading

import pytest

from gpu_common import lib

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", ["global", "thread_local"])
@pytest.mark.parametrize("where", ["same thread", "other thread"])
def test_close_beside_a_capture(where, mode):
    import torch
    F = lib()
    s = F.Solver([F.Params(nx=40, qx_half=4, qy=4, qz=0, kn=0.3, eta0=0.1, U_left=-0.2, U_right=0.2)], stream=torch.cuda.Stream())
    s.step(3)
    assert s.status()[2][0] == 3
    x = torch.zeros(8, device="cuda")
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.stream(torch.cuda.Stream()):
        graph.capture_begin(capture_error_mode=mode)
        try:
            x.add_(1.0)
            if where == "same thread":
                s.close()
            else:
                t = threading.Thread(target=s.close)
                t.start()
                t.join()
            x.add_(1.0)
        finally:
            graph.capture_end()
    graph.replay()
    torch.cuda.synchronize()
    assert x.eq(2.0).all()
