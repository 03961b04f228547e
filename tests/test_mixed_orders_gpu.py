"""Mixed precision at box orders and box sizes where a scaled quantity leaves its
format (x = k times the box side, sig_j = (x/2)^j / j!): finite, and FP32 against
FP64 of the same truncated expansions within the mixed tolerance 1e-6, on targets
far, near and on the curve and on a tree deep enough for every list."""
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


def _plan(qbxmod, k, p_fmm):
    curve = fourier_radial(np.array([0.0, 0.1, 0.15]), np.array([0.0, 0.4, 1.0]), 1.0)
    g = discretise_curve(*curve, 160, 8, k=k)
    on = np.arange(0, g.n, 5)
    off = grid_targets(40, -3.0, 3.0)  # its corners set the root box
    tgt = np.concatenate([g.node_xy[on], off])
    node = np.concatenate([on, np.full(len(off), -1)]).astype(np.int64)
    side = np.where(node >= 0, 1 - 2 * (np.arange(len(tgt)) % 2), 0).astype(np.int8)
    lp = qbxmod.LayerPotential(g.as_dict(), 6, sides=2)
    assoc = lp.build(tgt, node, side, mode=qbxmod.QBX_FMM, p_fmm=p_fmm, p_add=0, n_max=12)
    return lp, g, assoc


def _check(qbxmod, order, x):
    # the finest level's boxes have k side = x: its depth does not depend on k
    lp, _, _ = _plan(qbxmod, 1.0, 8)
    depth = int(lp.stats()["depth"])
    lp.close()
    k = x * 2.0 ** depth / 6.0
    p_fmm = next(p for p in range(order, 0, -1)
                 if qbxmod.qbx_fmm_level_orders(k, 6.0, depth + 1, p, 0)[depth] <= order)
    lp, g, assoc = _plan(qbxmod, k, p_fmm)
    assert int(lp.stats()["depth"]) == depth and lp.box_orders()[depth] == order
    st = lp.stats()
    assert min(st["v_pairs"], st["w_pairs"], st["x_pairs"]) > 0
    rng = np.random.default_rng(order)
    sig = rng.standard_normal(g.n) + 1j * rng.standard_normal(g.n)
    kw = dict(sigma_S=sig, cS=1.0, sigma_D=sig, cD=0.3j)
    u = lp.eval(**kw)
    v = lp.eval(precision=qbxmod.QBX_MIXED, **kw)
    lp.close()
    assert np.isfinite(u).all() and np.isfinite(v).all()
    for sel in (assoc >= 0, assoc < 0):
        assert np.linalg.norm((u - v)[sel]) < 1e-6 * np.linalg.norm(u[sel])


# 2^{s j} / sig_j beyond FP32 where 2^{s m} H_m is within its bound, and next to it
@pytest.mark.parametrize("order,x", [
    (126, 5.856), (125, 5.7848), (124, 5.7144), (123, 5.6456), (122, 5.6)])
def test_scaled_powers_beyond_fp32(qbxmod, order, x):
    _check(qbxmod, order, x)


# 1 / sig_j beyond FP64
@pytest.mark.parametrize("order,x", [
    (54, 2.0 ** -13.7), (54, 2.0 ** -14), (64, 2.0 ** -10.5)])
def test_inverse_sigma_beyond_fp64(qbxmod, order, x):
    _check(qbxmod, order, x)


# H_m of the M2L, m <= 2 order, beyond FP64, with and without the above
@pytest.mark.parametrize("order,x", [
    (126, 0.732), (123, 0.7057), (120, 0.24), (130, 0.5)])
def test_m2l_hankel_beyond_fp64(qbxmod, order, x):
    _check(qbxmod, order, x)


# the same in FP64 on the CUDA cores (m2l_engine 2)
def test_m2l_hankel_beyond_fp64_cuda_cores(qbxmod):
    g = discretise_curve(*fourier_radial(np.array([0.2]), np.array([0.3]), 1.0), 160, 8, k=4.0)
    sig = np.exp(1j * np.arange(g.n))
    u = []
    for engine in (0, 2):
        lp = qbxmod.LayerPotential(g.as_dict(), 6, sides=2)
        lp.build(grid_targets(40, -3.0, 3.0), mode=qbxmod.QBX_FMM, p_fmm=126, p_add=0, n_max=12,
                 m2l_engine=engine)
        u.append(lp.eval(sigma_S=sig, cS=1.0))
        lp.close()
    assert np.isfinite(u[1]).all()
    assert np.linalg.norm(u[1] - u[0]) < 1e-10 * np.linalg.norm(u[0])
