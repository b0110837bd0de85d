"""Full-range x projections in FP32 storage on both sides of the double-float range's line (T = 1.8): tiles that
are below it, above it and mixed, against the oracle."""
import pytest

from gpu_common import compare, lib, oracle_for

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("qx_half,tol", [(8, 1e-5), (20, 1e-5)])
def test_hot_full_range_matches_oracle(qx_half, tol):
    F = lib()
    ps = [F.Params(nx=40, kn=0.3, eta0=0.05, qx_half=qx_half, qy=0, qz=0, T_left=1.5, T_right=1.7, x_quadrature="full",
                   precision="fp32"),
          F.Params(nx=70, kn=0.3, eta0=0.05, qx_half=qx_half, qy=3, qz=0, T_left=1.2, T_right=2.2, T_init=1.7, x_quadrature="full",
                   precision="fp32")]
    s = F.Solver(ps)
    s.step(10)
    for i, p in enumerate(ps):
        o = oracle_for(p)
        o.step(10)
        M = o.moments()
        compare(s.moments(i), M, tol, f"instance {i}")
        assert (M["T"].max() > 1.8) == (i == 1)
