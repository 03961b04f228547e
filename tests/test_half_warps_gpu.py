"""P2QBXL with a warp and with half a warp per centre: handles of 6112 centres (a warp
each) and of 6144 (half a warp), an odd number of them used, so that the last half
warp stays without one, in one-warp blocks (fewer than 8192 formed). Against the
FP64 oracle at some of the targets; and every centre formed (coefficients asked
for) gives the bits of the used ones formed."""
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


@pytest.mark.parametrize("precision,tol", [("fp64", 1e-10), ("mixed", 1e-6)])
@pytest.mark.parametrize("p,layers", [(3, "S"), (12, "DS"), (16, "D")])
@pytest.mark.parametrize("panels", [191, 192])
def test_odd_number_of_centres(qbxmod, oracle, panels, p, layers, precision, tol):
    g = discretise_curve(*starfish(0.25, 5), panels, 16, k=6.0)
    rng = np.random.default_rng(panels)
    sig = rng.standard_normal(g.n) + 1j * rng.standard_normal(g.n)
    n = 1001
    node = np.arange(n, dtype=np.int64)
    tgt = g.node_xy[node]
    lp = qbxmod.LayerPotential(g.as_dict(), p, sides=2)
    assoc = lp.build(tgt, node, np.ones(n, np.int8), p_fmm=45, n_max=24, mode=qbxmod.QBX_FMM)
    assert lp.n_centres == 32 * panels and (assoc >= 0).all() and np.unique(assoc).size == n
    kw = dict(precision=qbxmod.QBX_MIXED if precision == "mixed" else qbxmod.QBX_FP64)
    if "S" in layers:
        kw.update(sigma_S=sig, cS=0.7 - 2.2j)
    if "D" in layers:
        kw.update(sigma_D=sig, cD=1.1j)
    u = lp.eval(**kw)
    v = lp.eval(alpha_out=np.empty((lp.n_centres, 2 * p + 1), complex), **kw)
    lp.close()
    assert np.array_equal(u, v)
    pick = np.r_[0:n:40, n - 3:n]
    u_ref, _ = oracle.layer_potential(
        g.as_dict(), tgt[pick], p, sigma_S=kw.get("sigma_S"), sigma_D=kw.get("sigma_D"),
        cS=kw.get("cS", 0.0), cD=kw.get("cD", 0.0), sides=2, centre_of_target=assoc[pick])
    assert np.linalg.norm(u[pick] - u_ref) < tol * np.linalg.norm(u_ref)
