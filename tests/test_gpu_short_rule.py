"""Orders just above the 8-point auxiliary rule's, in a start-up wave that is slow enough for it (|u_x|/sqrt T
just below 0.02), against the oracle."""
import numpy as np
import pytest

from gpu_common import compare, lib, oracle_for

pytestmark = pytest.mark.gpu


def test_slow_waves_match_oracle():
    F = lib()
    ps = [F.Params(nx=33, qx_half=q, qy=0, qz=0, kn=0.3, eta0=0.1, T_left=0.86, T_right=1.14) for q in (9, 10, 11, 12)]
    s = F.Solver(ps)
    s.step(20)
    for i, p in enumerate(ps):
        o = oracle_for(p)
        v = []
        for _ in range(20):
            o.step(1)
            M = o.moments()
            v.append(np.max(np.abs(M["ux"]) / np.sqrt(M["T"])))
        assert 0.018 < max(v) < 0.02
        compare(s.moments(i), M, 1e-12, f"order {p.qx_half}")
