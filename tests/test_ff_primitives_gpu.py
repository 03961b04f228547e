"""The float-float primitives of the mixed path (csrc/ff.cuh), compiled on their own
(ff_primitives.cu) and compared with mpmath at 40 digits over the ranges that they
serve. Bounds: FP64 is truncated to 2^-46, a product or sum errs by a unit of 2^-46,
the root by 2^-44, so k r by 2.6 times that (below 2^-42); the Hankel tables by two
FP32 roundings (2^-23) of the first FP32 degree, 17^-3 or 17^-6 of |H| (0.25^3 / 6 or
0.25^6 / 720 where H oscillates, beyond x = 1), and 1/17 of it for the next, plus a
unit per Horner step; Miller's recurrence by a few units per order and what its
argument's 2^-42 makes of J_j (j or x times that)."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from tests.conftest import ROOT

pytestmark = pytest.mark.gpu
U = 2.0 ** -46


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    torch = pytest.importorskip("torch")
    pytest.importorskip("mpmath")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1602_05301_gb300 import build as b
    so = str(tmp_path_factory.mktemp("ff") / "ff_primitives.so")
    r = subprocess.run([b.nvcc()] + b.ARCH + b.FLAGS + ["-I" + b.CSRC, "-shared", "-o", so,
                       os.path.join(ROOT, "tests", "ff_primitives.cu")],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    lib = ctypes.CDLL(so)
    vp, i, d = ctypes.c_void_p, ctypes.c_int, ctypes.c_double
    lib.ff_probe.argtypes = [i, i, vp, vp, i, d, i, vp]

    def run(op, a, width, b=None, iarg=0, k=1.0):
        a = np.ascontiguousarray(a, float)
        b = None if b is None else np.ascontiguousarray(b, float)
        out = np.empty((a.size, width))
        assert lib.ff_probe(op, a.size, a.ctypes.data, None if b is None else b.ctypes.data,
                            iarg, k, width, out.ctypes.data) == 0
        return out

    return run


def _pair(x):
    """x rounded to a pair of FP32 numbers, exactly representable in FP64."""
    h = np.asarray(x, float).astype(np.float32).astype(float)
    return h + (x - h).astype(np.float32)


@pytest.mark.parametrize("op,near,far", [(0, 2.6e-11, 3.3e-10), (1, 5.3e-15, 4.3e-14)])
def test_hankel(probe, op, near, far):
    import mpmath as mp
    mp.mp.dps = 40
    rng = np.random.default_rng(op)
    # interval ends and random points of both tables, and arguments outside them
    ends = np.concatenate([2.0 ** np.arange(-16, 4), 8.0 + 0.5 * np.arange(48)])
    x = _pair(np.concatenate([ends, ends * (1 - 2.0 ** -24), np.geomspace(2.0 ** -16, 8, 300),
                              rng.uniform(8, 31.98, 300), [2.0 ** -20, 1e-12, 32.0, 40.5, 300.0]]))
    h = probe(op, x, 4)
    h = h[:, 0::2] + 1j * h[:, 1::2]
    ref = np.array([[complex(mp.hankel1(n, mp.mpf(v))) for n in (0, 1)] for v in x])
    err = np.max(np.abs(h - ref) / np.abs(ref), axis=1)
    # (outside the tables the value is FP64's rounded to a pair)
    assert np.all(err < np.where(x < 1, near, far) + 10 * U)


def test_rounding_of_fp64(probe):
    rng = np.random.default_rng(1)
    v = np.concatenate([rng.uniform(-2, 2, 500), np.ldexp(rng.uniform(-1, 1, 500),
                        rng.integers(-70, 100, 500)), [0.0, -0.0, 1.0, 2.0 ** -100, 1 - 2.0 ** -53]])
    for sh in (-20, 0, 7):
        w = np.ldexp(v, -sh)
        got = probe(2, v, 1, iarg=sh)[:, 0]
        assert np.all(np.abs(got - w) <= 2.0 ** -46 * np.abs(w))
    # below FP32's normal range zero, the second part zero where it would be subnormal
    got = probe(2, [2.0 ** -127, -2.0 ** -149, 2.0 ** -126 * (1 + 2.0 ** -30), 2.0 ** 128], 1)[:, 0]
    assert got[0] == 0 and got[1] == 0 and got[2] == 2.0 ** -126 and np.isinf(got[3])


def test_fp32_to_fp64(probe):
    rng = np.random.default_rng(4)
    v = np.concatenate([rng.standard_normal(500), np.ldexp(rng.uniform(-1, 1, 500),
                        rng.integers(-125, 128, 500)), [0.0, -0.0, 1.0, np.inf, -np.inf, np.nan,
                        2.0 ** -126, -2.0 ** -126, np.finfo(np.float32).max]])
    v = v.astype(np.float32)
    v[np.abs(v) < 2.0 ** -126] = 0  # subnormals become zero
    assert np.array_equal(probe(5, v, 1)[:, 0], v.astype(float), equal_nan=True)


def test_reciprocal_root(probe):
    x = _pair(np.random.default_rng(2).uniform(1, 4, 2000) * 4.0 ** np.repeat(np.arange(-35, 45), 25))
    got = probe(3, x, 1)[:, 0]
    ref = 1 / np.sqrt(x)  # FP64: 2^-53
    assert np.max(np.abs(got - ref) / ref) < 2.0 ** -44


@pytest.mark.parametrize("k", [1.0, 20.0, 3e-7, 1.9e9])
def test_polar(probe, k):
    """From the largest distances to those whose square is below FP32's range."""
    rng = np.random.default_rng(3)
    r = np.concatenate([10.0 ** rng.uniform(-30, 3, 2000), 10.0 ** rng.uniform(-24, -18, 500)]) / k
    th = rng.uniform(0, 2 * np.pi, r.size)
    dx, dy = r * np.cos(th), r * np.sin(th)
    o = probe(4, dx, 5, b=dy, k=k)
    rr, unit = np.hypot(dx, dy), 2.0 ** np.floor(np.log2(k))
    assert np.all(o[:, 0] == 1)
    # the second parts of components below 2^-102 may be lost
    tol = np.where(k * r > 2.0 ** -90, 2.0 ** -42, 2.0 ** -22)
    assert np.all(np.abs(o[:, 1] - k * rr) <= tol * k * rr)
    assert np.all(np.abs(o[:, 2] * rr * unit - 1) <= tol)
    assert np.all(np.hypot(o[:, 3] - dx / rr, o[:, 4] - dy / rr) < 2.0 ** -21)
    o = probe(4, [0.0, 1e-39, 1e-45], 5, b=[0.0, -1e-39, 0.0], k=1.0)
    assert not o[:, 0].any()


@pytest.mark.parametrize("M,x,s", [(5, 1e-4, -12), (20, 0.4, -5), (20, 3.0, -2), (60, 0.05, -9),
                                   (60, 20.0, 0), (126, 0.5, -7), (126, 60.0, 0)])
def test_miller(probe, M, x, s):
    import mpmath as mp
    mp.mp.dps = 40
    xs = np.array([x, 0.7 * x])
    got = probe(100 + M, xs, M + 1, iarg=s)
    for v, row in zip(xs, got):
        J = [mp.besselj(j, mp.mpf(v)) for j in range(M + 1)]
        ref = np.array([float(t * mp.mpf(2) ** (-s * j)) for j, t in enumerate(J)])
        # relative to the row's envelope where J has zeros (orders below x), to the
        # values above; orders whose scaled value nears FP32's least are lost
        env = np.where(np.arange(M + 1) < v, np.abs(ref[:int(v) + 1]).max(), np.abs(ref))
        ok = env > 2.0 ** -40
        assert ok.sum() >= 3
        assert np.all(np.abs(row - ref)[ok] <= (16 + 20 * M + 16 * v) * U * env[ok])
