"""The all-pairs and U-list FP64 coefficient kernels at the sizes where their
work split changes: fewer sources than a block has lanes, few and many centres
(four warps or one per centre), orders at the ends of the reduction's layout
(0, 1, 15, 16), each layer alone and both, and the direct plan that forms only
the centres its targets use. Against the FP64 oracle, within the FP64 tolerance."""
import numpy as np
import pytest

from qbx_workloads import discretise_curve, starfish

pytestmark = pytest.mark.gpu

TOL64 = 1e-10


@pytest.fixture(scope="module")
def qbxmod():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1602_05301_gb300 import build as b
    b.build()
    from paper_1602_05301_gb300 import qbx
    return qbx


@pytest.mark.parametrize("mode", ["direct", "fmm"])
@pytest.mark.parametrize("panels,q,p", [(7, 5, 0), (12, 11, 1), (40, 13, 15), (64, 16, 16)])
@pytest.mark.parametrize("layers", ["S", "D", "DS"])
def test_coefficients_and_potential(qbxmod, oracle, mode, panels, q, p, layers):
    k = 1.3
    g = discretise_curve(*starfish(0.2, 3), panels, q, k=k)
    rng = np.random.default_rng(100 * panels + p)
    sig = rng.standard_normal(g.n) + 1j * rng.standard_normal(g.n)
    # every third node from outside, every fifth from inside, and targets off the curve
    on = np.concatenate([np.arange(0, g.n, 3), np.arange(0, g.n, 5)])
    side = np.concatenate([np.ones(len(range(0, g.n, 3))), -np.ones(len(range(0, g.n, 5)))])
    off = 3.0 * np.exp(2j * np.pi * np.arange(33) / 33)
    tgt = np.concatenate([g.node_xy[on], np.stack([off.real, off.imag], -1)])
    node = np.concatenate([on, np.full(33, -1)]).astype(np.int64)
    side = np.concatenate([side, np.zeros(33)]).astype(np.int8)
    lp = qbxmod.LayerPotential(g.as_dict(), p, sides=2)
    assoc = lp.build(tgt, node, side, p_fmm=40, n_max=24,
                     mode=qbxmod.QBX_FMM if mode == "fmm" else qbxmod.QBX_DIRECT)
    kw = {}
    if "S" in layers:
        kw.update(sigma_S=sig, cS=0.7 - 0.2j)
    if "D" in layers:
        kw.update(sigma_D=sig, cD=1.1j)
    alpha = np.zeros((2 * g.n, 2 * p + 1), np.complex128)
    u = lp.eval(**kw)                    # the used centres only
    ua = lp.eval(alpha_out=alpha, **kw)  # every centre
    lp.close()
    u_ref, _ = oracle.layer_potential(
        g.as_dict(), tgt, p, sigma_S=kw.get("sigma_S"), sigma_D=kw.get("sigma_D"),
        cS=kw.get("cS", 0.0), cD=kw.get("cD", 0.0), sides=2, centre_of_target=assoc)
    for v in (u, ua):
        assert np.linalg.norm(v - u_ref) <= TOL64 * np.linalg.norm(u_ref)
    cxy, rad = oracle.centres(g.node_xy, g.normal_xy, g.panel_of_node, g.panel_h, 2)
    a_ref = oracle.qbx_coefficients(g.node_xy, g.normal_xy, g.weight, k, cxy, p,
                                    kw.get("sigma_S"), kw.get("sigma_D"), kw.get("cS", 0.0),
                                    kw.get("cD", 0.0))
    from scipy.special import jv
    w = np.abs(jv(np.arange(-p, p + 1)[None, :], k * np.asarray(rad)[:, None]))
    assert np.linalg.norm((alpha - a_ref) * w) <= TOL64 * np.linalg.norm(a_ref * w)
