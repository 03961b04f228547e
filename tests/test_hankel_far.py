"""H_0 and H_1 beyond the geometric tables (x >= 8): the committed table of
[8, 32) is its generator's output, and the device values there and in Hankel's
expansion above match mpmath, both orders in each branch, at interval ends, on
warps that straddle the branches and at large arguments. Bound: the four
roundings of a Horner step on values up to |H| (2e-15) below 32; above it the
reduced argument is exact, the amplitude, the rotation and P + iQ add a few
roundings (4e-15)."""
import os
import subprocess
import sys

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1602_05301_gb300", "csrc")


@pytest.mark.parametrize("name", ["far"])
def test_header_is_the_generator_output(name):
    pytest.importorskip("mpmath")
    r = subprocess.run([sys.executable, os.path.join(CSRC, "gen_hankel_table_%s.py" % name)],
                       capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stderr
    assert r.stdout == open(os.path.join(CSRC, "hankel_table_%s.h" % name)).read()


@pytest.mark.gpu
@pytest.mark.parametrize("variant", [0, 1])
def test_values_against_mpmath(variant):
    torch = pytest.importorskip("torch")
    mp = pytest.importorskip("mpmath")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1602_05301_gb300 import build as b
    b.build()
    from paper_1602_05301_gb300 import qbx
    mp.mp.dps = 30
    rng = np.random.default_rng(3)
    ends = 8.0 + 0.5 * np.arange(49)
    x = np.concatenate([ends, np.nextafter(ends, 0)[1:], rng.uniform(8, 40, 400),
                        np.geomspace(32, 1e6, 200)])
    x = x[rng.permutation(x.size)]
    h = qbx.qbx_hankel01(x, variant)
    ref = np.array([[complex(mp.hankel1(0, v)), complex(mp.hankel1(1, v))] for v in x])
    err = np.max(np.abs(h - ref) / np.abs(ref), axis=1)
    assert err[x < 32].max() < 2e-15
    assert err[x >= 32].max() < 4e-15
