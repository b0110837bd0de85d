"""The arithmetic of the update kernel by itself, compiled from its headers, against wider arithmetic
on the host."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def dev(tmp_path_factory):
    from paper_2308_15407_gb300 import build
    so = str(tmp_path_factory.mktemp("arith") / "arith.so")
    subprocess.run([build.nvcc(), *build.ARCH, *build.FLAGS, "-I", build.CSRC, "-shared", "-o", so,
                    os.path.join(HERE, "device_arithmetic.cu")], check=True)
    return C.CDLL(so)


def faces(dev, v):
    """Device faces of the stencils v[n, 5], in v's type."""
    import torch
    x = torch.tensor(v, device="cuda")
    y = torch.empty(len(v), dtype=x.dtype, device="cuda")
    torch.cuda.synchronize()
    fn = dev.faces32 if v.dtype == np.float32 else dev.faces64
    assert fn(C.c_void_p(x.data_ptr()), len(v), C.c_void_p(y.data_ptr())) == 0
    return y.cpu().numpy()


def faces_wide(v):
    """The three candidates and their weights 1/10, 6/10, 3/10 over the squared indicators, in long double."""
    a, b, c, d, e = v.astype(np.longdouble).T
    F = np.stack([2 * a - 7 * b + 11 * c, -b + 5 * c + 2 * d, 2 * c + 5 * d - e]) / 6
    s = np.stack([13 * (a - 2 * b + c) ** 2 + 3 * (a - 4 * b + 3 * c) ** 2,
                  13 * (b - 2 * c + d) ** 2 + 3 * (b - d) ** 2,
                  13 * (c - 2 * d + e) ** 2 + 3 * (3 * c - 4 * d + e) ** 2])
    w = np.array([1, 6, 3], dtype=np.longdouble)[:, None] * (s.min(axis=0) / s) ** 2
    return (w * F).sum(axis=0) / w.sum(axis=0)


def fronts(jump, falling, dtype, seed=0):
    """Two levels 1 : jump with the front at any of the four gaps, each sloping by 2 % a node, with 0.5 %
    of noise (as far as the weights of FP32 resolve it: jumps up to 1e3)."""
    rng = np.random.default_rng(seed)
    n = 4000
    at = rng.integers(1, 5, n)[:, None]
    j = np.arange(5)[None]
    high = (j < at) if falling else (j >= at)
    noise = 0.005 if dtype == np.float64 or jump <= 1e3 else 0.0
    v = (1 + 0.02 * j + noise * rng.uniform(-1, 1, (n, 5))) * np.where(high, 1.0, 1.0 / jump)
    return v.astype(dtype)


JUMPS = [1.0, 3.0, 1e2, 1e3, 1e4, 1e6, 1e8, 1e12]


# A candidate is a sum of three products whose coefficients add up to 10/3 at most: up to seven roundings of
# the face with those of the coefficients themselves; the weighted mean adds the weights' products, their
# sum and a quotient (in FP32 an approximate reciprocal of two units, but of the offset from c only).
BARS = [(np.float32, 10 * 2.0 ** -24), (np.float64, 12 * 2.0 ** -53)]


@pytest.mark.parametrize("falling", [False, True], ids=["rising", "falling"])
@pytest.mark.parametrize("jump", JUMPS)
@pytest.mark.parametrize("dtype,tol", BARS, ids=["fp32", "fp64"])
def test_faces_at_fronts(dev, dtype, tol, jump, falling):
    v = fronts(jump, falling, dtype)
    ref = faces_wide(v)
    assert np.max(np.abs(faces(dev, v) / ref - 1)) <= tol


# FP64 takes its weights in double-float up to third differences of 2^-7 of the value
@pytest.mark.parametrize("noise", [1e-4, 1e-3, 2e-3, 4e-3, 0.03, 0.3])
@pytest.mark.parametrize("dtype,tol", BARS, ids=["fp32", "fp64"])
def test_faces_across_the_smoothness_line(dev, dtype, tol, noise):
    v = (1 + noise * np.random.default_rng(3).uniform(-1, 1, (20000, 5))).astype(dtype)
    ref = faces_wide(v)
    assert np.max(np.abs(faces(dev, v) / ref - 1)) <= tol
