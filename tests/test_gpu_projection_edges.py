"""Velocity-space projections at the edges of their code paths against the oracle: orders around
the register blocks (8 and 16 polynomials) and the double-float range (up to 32), the smallest
and odd transverse orders, each velocity-space form and x rule, and a start-up wave strong
enough for the long auxiliary rule (|u_x|/sqrt T > 0.02).  The bars are the repository's: 1e-12
(FP64) and 1e-5 (FP32 storage).  (Orders 9 to 12 in a wave of |u_x|/sqrt T just below 0.02 do not
reach 1e-12 with the 8-point auxiliary rule, see the comment at its use.)"""
import numpy as np
import pytest

from gpu_common import compare, lib, oracle_for

pytestmark = pytest.mark.gpu

WAVE = dict(nx=33, kn=0.3, eta0=0.1, T_left=0.7, T_right=1.3)
SHEAR = dict(nx=35, kn=0.2, eta0=0.1, U_left=-0.4, U_right=0.3, T_left=0.9, T_right=1.0, grid="tanh")
LOW = [dict(WAVE, qx_half=2, qy=0, qz=0), dict(WAVE, qx_half=3, qy=3, qz=0), dict(SHEAR, qx_half=7, qy=5, qz=3),
       dict(SHEAR, qx_half=8, qy=8, qz=8, j1_shear=True), dict(SHEAR, qx_half=4, qy=2, qz=0, accel_y=0.1),
       dict(WAVE, qx_half=3, qy=0, qz=0, x_quadrature="full"), dict(SHEAR, qx_half=4, qy=4, qz=3, x_quadrature="full")]
HIGH = [dict(SHEAR, qx_half=13, qy=7, qz=0),
        dict(WAVE, qx_half=16, qy=0, qz=0), dict(SHEAR, qx_half=17, qy=3, qz=0), dict(WAVE, qx_half=32, qy=0, qz=0),
        dict(WAVE, qx_half=33, qy=0, qz=0), dict(SHEAR, qx_half=17, qy=4, qz=0, x_quadrature="full")]


@pytest.mark.parametrize("precision,tol", [("fp64", 1e-12), ("fp32", 1e-5)])
@pytest.mark.parametrize("batch", [LOW, HIGH], ids=["low", "high"])
def test_projection_edges_match_oracle(batch, precision, tol):
    F = lib()
    s = F.Solver([F.Params(**d, precision=precision) for d in batch])
    s.set_schedule("tiled")
    s.step(20)
    for i, d in enumerate(batch):
        o = oracle_for(F.Params(**d))
        o.step(20)
        Mo = o.moments()
        compare(s.moments(i), Mo, tol, f"instance {i} ({precision})")
        if d["nx"] == WAVE["nx"]:
            assert np.max(np.abs(Mo["ux"]) / np.sqrt(Mo["T"])) > 0.02     # the long rule was in use


# FP32 storage above 32 polynomials: double-float with scaled points up to T = 1.8, FP64 in hotter
# tiles; an instance below and one whose tiles differ (x projections split over blocks)
HOT = [dict(nx=40, kn=0.3, eta0=0.05, qx_half=40, qy=0, qz=0, T_left=1.5, T_right=1.7),
       dict(nx=70, kn=0.3, eta0=0.05, qx_half=36, qy=3, qz=0, T_left=1.0, T_right=2.4, T_init=1.7)]


def test_hot_high_orders_match_oracle():
    F = lib()
    s = F.Solver([F.Params(**d, precision="fp32") for d in HOT])
    s.set_schedule("tiled")
    s.step(10)
    for i, d in enumerate(HOT):
        o = oracle_for(F.Params(**d))
        o.step(10)
        compare(s.moments(i), o.moments(), 1e-5, f"instance {i}")
