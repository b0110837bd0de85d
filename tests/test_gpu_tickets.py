"""The arrival tickets of a tile's update chunks after an update that gave up: its blocks leave without
taking theirs, and the next state of the instance must not find the count short."""
import numpy as np
import pytest

from gpu_common import lib

pytestmark = pytest.mark.gpu


def tickets(F, s):
    """The ticket counters of a batch of one instance of up to 64 tiles: the last 256 bytes of its workspace."""
    import torch
    pad = -s.ws.data_ptr() % 256
    end = pad + F.workspace_bytes(s.params)
    return s.ws[end - 256:end].view(torch.int32)


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("how", ["profiles", "state"])
def test_new_state_clears_the_tickets(how, precision):
    F = lib()
    p = F.Params(nx=45, qx_half=6, qy=6, qz=0, kn=0.1, eta0=0.2, U_left=-0.42, U_right=0.42, grid="tanh", precision=precision)
    x = np.linspace(-1.0, 1.0, p.nx)
    got = []
    for left in (0, 1):                                   # tickets left in place: none, one per tile
        s = F.Solver([p])
        assert s.layout()[1] > 2                          # several chunks per tile
        s.step(3)
        state = s.get_state()
        t = tickets(F, s)
        assert not t.any()
        t[:2] = left
        if how == "profiles":
            s.set_profiles(0, 1.0 + 0.1 * x, 0.2 * x, 1.0 - 0.1 * x * x)
        else:
            s.set_state(0, state)
        assert not t.any()
        s.step(4)
        got.append((s.moments(), s.get_state()))
    assert got[0][1] == got[1][1]
    for k, v in got[0][0].items():
        assert np.array_equal(v, got[1][0][k]), k
