"""A batch that captures its graph anew at every evaluation in one thread while
others build, evaluate and destroy plans: distinct handles are independent, so each
gives what it gives alone."""
import threading

import numpy as np
import pytest

from qbx_workloads import discretise_curve, starfish

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def qbxmod():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1602_05301_gb300 import build as b
    b.build()
    from paper_1602_05301_gb300 import qbx
    return qbx


def _plan(qbxmod, panels):
    g = discretise_curve(*starfish(0.25, 5), panels, 12, k=4.0)
    lp = qbxmod.LayerPotential(g.as_dict(), 6, sides=2)
    lp.build(g.node_xy, np.arange(g.n), np.ones(g.n, np.int8), mode=qbxmod.QBX_FMM, p_fmm=20,
             n_max=20)
    return lp, np.cos(np.arange(g.n)) + 1j * np.sin(3.0 * np.arange(g.n))


def test_captures_beside_other_threads(qbxmod):
    probs = [_plan(qbxmod, m) for m in (30, 44, 61)]
    batch = qbxmod.Batch([lp for lp, _ in probs])
    sig = np.concatenate([s for _, s in probs])
    coefs = [1.0, 2j, -0.5]
    ref = [batch.eval(sigma_S=sig, cS=c) for c in coefs]

    def alone():
        lp, s = _plan(qbxmod, 37)
        u = lp.eval(sigma_S=s, cS=1.0)
        lp.close()
        return u

    x = np.linspace(0.1, 40.0, 1000)
    ref_u, ref_h = alone(), qbxmod.qbx_hankel01(x)
    done, errors = threading.Event(), []

    def work(fn, ref):
        try:
            while not done.is_set():
                assert np.array_equal(fn(), ref)
        except BaseException as e:
            errors.append(e)
            done.set()

    threads = [threading.Thread(target=work, args=a) for a in
               ((lambda: qbxmod.qbx_hankel01(x), ref_h), (alone, ref_u))]
    for t in threads:
        t.start()
    try:
        for i in range(120):
            if done.is_set():
                break
            assert np.array_equal(batch.eval(sigma_S=sig, cS=coefs[i % 3]), ref[i % 3]), i
    finally:
        done.set()
        for t in threads:
            t.join()
    batch.close()
    for lp, _ in probs:
        lp.close()
    assert not errors, errors
