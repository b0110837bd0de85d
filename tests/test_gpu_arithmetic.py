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


# The velocity tails: the same stencils, smaller by powers of two.
@pytest.mark.parametrize("falling", [False, True], ids=["rising", "falling"])
@pytest.mark.parametrize("jump", [*JUMPS, 3e4, 1e5, 2e5])
@pytest.mark.parametrize("dtype,tol,e", [(np.float32, BARS[0][1], e) for e in (0, -20, -30, -36, -45)] +
                         [(np.float64, BARS[1][1], e) for e in (-60, -80, -99, -130, -400)])
def test_small_faces_at_fronts(dev, dtype, tol, e, jump, falling):
    v = np.ldexp(fronts(jump, falling, dtype), e)
    ref = faces_wide(np.ldexp(v, -e))
    assert np.max(np.abs(np.ldexp(faces(dev, v), -e) / ref - 1)) <= tol


# FP64 takes its weights in double-float up to third differences of 2^-7 of the value
@pytest.mark.parametrize("noise", [1e-4, 1e-3, 2e-3, 4e-3, 0.03, 0.3])
@pytest.mark.parametrize("dtype,tol", BARS, ids=["fp32", "fp64"])
def test_faces_across_the_smoothness_line(dev, dtype, tol, noise):
    v = (1 + noise * np.random.default_rng(3).uniform(-1, 1, (20000, 5))).astype(dtype)
    ref = faces_wide(v)
    assert np.max(np.abs(faces(dev, v) / ref - 1)) <= tol


def rounding(dev, base, inc, lo, hi):
    """Of all 2^24 random numbers, how many round base + inc to lo, to hi, and to neither."""
    import torch
    n = torch.zeros(3, dtype=torch.int64, device="cuda")
    torch.cuda.synchronize()
    assert dev.rounding(C.c_float(base), C.c_float(inc), C.c_float(lo), C.c_float(hi), C.c_void_p(n.data_ptr())) == 0
    return n.cpu().tolist()


# base, exponent of the last place there, increment in units of it
ROUNDINGS = [(1.5, -23, 0.25), (1.5, -23, 0.75), (1.25, -23, 1e-3), (1.0, -23, 0.125),      # inside a binade
             (1.0, -24, -1e-3), (1.0, -24, -0.5), (1.0, -24, -0.875),                     # down from a power of two
             (1.0 - 2.0 ** -24, -24, 0.999), (1.0 - 2.0 ** -24, -24, 1e-3),                # up to one
             (2.0 ** -110, -133, 0.25), (2.0 ** -110, -134, -0.25), (2.0 ** -126, -149, 0.0),   # 2^-103 and below
             (3.0 * 2.0 ** -120, -142, 0.375), (1.5, -23, 0.0), (0.0, -23, 1.0), (1.75, -23, 2.0 ** -20)]


@pytest.mark.parametrize("sign", [1.0, -1.0], ids=["plus", "minus"])
@pytest.mark.parametrize("case", ROUNDINGS, ids=str)
def test_rounding_is_exact_in_expectation(dev, case, sign):
    """A sum goes to one of its two neighbouring floats, to each as often as the other is near: of the 2^24
    random numbers to within one (half a step of the comparison, half a unit of the remainder)."""
    base, e, units = case
    inc = np.float32(units * 2.0 ** e)
    s = np.float64(base) + np.float64(inc)                   # exact: at most 47 bits apart
    lo = np.float32(s)
    if lo > s:
        lo = np.nextafter(lo, np.float32(-np.inf))
    hi = lo if lo == s else np.nextafter(lo, np.float32(np.inf))
    up = 0.0 if lo == s else float((s - np.float64(lo)) / (np.float64(hi) - np.float64(lo)))
    n = rounding(dev, sign * base, sign * float(inc), sign * float(lo), sign * float(hi))
    assert n[2] == 0
    assert abs(n[1] - up * 2 ** 24) <= 1
    if sign < 0:
        assert n == rounding(dev, base, float(inc), float(lo), float(hi))


def test_rounding_keeps_what_is_not_finite(dev):
    inf, big = float("inf"), float(np.finfo(np.float32).max)
    assert rounding(dev, inf, 1.0, inf, 0.0)[0] == 2 ** 24
    assert rounding(dev, 1.0, -inf, -inf, 0.0)[0] == 2 ** 24
    assert rounding(dev, float("nan"), 1.0, 1.0, inf)[2] == 2 ** 24
    assert rounding(dev, big, 0.0, big, inf)[0] == 2 ** 24
