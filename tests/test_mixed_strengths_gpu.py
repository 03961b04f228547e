"""The mixed path at densities of any size: it is linear, and a power of two times
a density changes no rounding, so the potentials and the coefficients are the same
power of two times those of the density, bit for bit (no value of either comes
near FP64's limits). On targets that every list and both one-sided limits feed,
with a caller's grid and a library-made one, alone and as a batch."""
import numpy as np
import pytest

from qbx_workloads import discretise_curve, fourier_radial
from qbx_workloads.configs import grid_targets

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


def _plan(qbxmod, k, p_fmm, panels=120, q_src=0, n_max=30):
    curve = fourier_radial(np.array([0.0, 0.1, 0.15]), np.array([0.0, 0.4, 1.0]), 1.0)
    g = discretise_curve(*curve, panels, 10, k=k)
    on = np.arange(0, g.n, 3)
    off = grid_targets(40, -2.5, 2.5)
    tgt = np.concatenate([g.node_xy[on], off])
    node = np.concatenate([on, np.full(len(off), -1)]).astype(np.int64)
    side = np.where(node >= 0, 1 - 2 * (np.arange(len(tgt)) % 2), 0).astype(np.int8)
    lp = qbxmod.LayerPotential(g.as_dict(), 7, sides=2, q_src=q_src)
    lp.build(tgt, node, side, mode=qbxmod.QBX_FMM, p_fmm=p_fmm, p_add=0, n_max=n_max)
    return lp, g


# p_fmm = 130 has levels without a power-of-two scale: the kernels for those too
@pytest.mark.parametrize("k,p_fmm,q_src,layers", [
    (6.0, 20, 0, "DS"), (0.02, 14, 24, "D"), (40.0, 30, 0, "S"), (3.0, 130, 0, "DS")])
@pytest.mark.parametrize("e", [-900, -110, -70, 50, 110, 700])
def test_power_of_two(qbxmod, k, p_fmm, q_src, layers, e):
    lp, g = _plan(qbxmod, k, p_fmm, q_src=q_src)
    rng = np.random.default_rng(7)
    sig = rng.standard_normal(g.n) + 1j * rng.standard_normal(g.n)
    sig *= 10.0 ** rng.uniform(-3, 0, g.n)
    n_ctr = int(lp.stats()["n_centres"])
    res = []
    for f in (1.0, 2.0 ** e):
        alpha = np.empty((n_ctr, 15), complex)
        kw = {}
        if "S" in layers:
            kw.update(sigma_S=f * sig, cS=0.3 - k * 1j)
        if "D" in layers:
            kw.update(sigma_D=f * sig, cD=1.1)
        u = lp.eval(precision=qbxmod.QBX_MIXED, alpha_out=alpha, **kw)
        res.append((u / f, alpha / f))
    lp.close()
    assert np.isfinite(res[0][0]).all() and np.linalg.norm(res[0][0]) > 0
    for a, b in zip(*res):
        assert np.array_equal(a, b)


def test_batch(qbxmod):
    probs = [_plan(qbxmod, 2.0 + 3 * i, 18, panels=40 + 23 * i) for i in range(3)]
    rng = np.random.default_rng(3)
    sig = [rng.standard_normal(g.n) + 1j * rng.standard_normal(g.n) for _, g in probs]
    b = qbxmod.Batch([lp for lp, _ in probs])
    scale = np.concatenate([np.full(lp.n_targets, 2.0 ** e) for (lp, _), e in
                            zip(probs, (-100, 0, 90))])
    cat = np.concatenate
    u = b.eval(sigma_S=cat(sig), cS=1j, precision=qbxmod.QBX_MIXED)
    v = b.eval(sigma_S=cat([2.0 ** e * s for e, s in zip((-100, 0, 90), sig)]), cS=1j,
               precision=qbxmod.QBX_MIXED)
    b.close()
    for lp, _ in probs:
        lp.close()
    assert np.array_equal(np.asarray(v), scale * np.asarray(u))


def test_no_strengths(qbxmod):
    lp, g = _plan(qbxmod, 5.0, 20)
    u = lp.eval(sigma_S=np.zeros(g.n, complex), cS=1.0, precision=qbxmod.QBX_MIXED)
    lp.close()
    assert np.array_equal(u, np.zeros_like(u))
