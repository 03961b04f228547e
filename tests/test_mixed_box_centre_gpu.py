"""Mixed precision with sources so close to a box centre that the square of their
distance is below FP32's normal range (k r from 1e-23 to 1e-19): finite, and the
FP64 potential within the mixed tolerance 1e-6 (such a source's expansion is its
charge alone)."""
from fractions import Fraction

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


def _centre(tree, b):
    """Centre of box b as one rounding of x0 + (i + 1/2) s, and as two."""
    x0, y0, side = tree["root"]
    s = side / 2.0 ** int(tree["level"][b])
    i, j = tree["ij"][b] + 0.5
    one = [float(Fraction(o) + Fraction(a) * Fraction(s)) for o, a in ((x0, i), (y0, j))]
    return np.array(one), np.array([x0 + i * s, y0 + j * s])


@pytest.mark.parametrize("k,r", [(1.0, 3e-23), (1.3, 1e-21), (5.0, 1e-20), (1.0, 9e-20)])
def test_source_at_a_box_centre(qbxmod, k, r):
    curve = fourier_radial(np.array([0.0, 0.1, 0.15]), np.array([0.0, 0.4, 1.0]), 1.0)
    g = discretise_curve(*curve, 80, 10, k=k)
    off = grid_targets(30, -3.0, 3.0)  # its corners set the root box
    rng = np.random.default_rng(5)
    sig = rng.standard_normal(g.n) + 1j * rng.standard_normal(g.n)
    geom = g.as_dict()
    src = dict(q=g.q, node_xy=np.array(geom["node_xy"]), normal_xy=np.array(geom["normal_xy"]),
               weight=np.array(geom["weight"]))
    shift = np.zeros(2)

    def plan():
        lp = qbxmod.LayerPotential(dict(geom, node_xy=geom["node_xy"] + shift), 5, sides=2,
                                   src=src, defer_conditions=True)
        lp.build(off + shift, mode=qbxmod.QBX_FMM, p_fmm=20, n_max=24)
        return lp, lp.export_tree()

    lp, tree = plan()
    lp.close()
    leaf = np.flatnonzero((tree["child"] < 0).all(1) & (tree["range"][:, 0, 1] -
                          tree["range"][:, 0, 0] >= 4) & (tree["level"] >= 3))[0]
    moved = tree["perm_src"][tree["range"][leaf, 0, 0]:][:2]
    shift = -_centre(tree, leaf)[0]  # the leaf's centre goes to the origin, up to rounding
    src["node_xy"] = src["node_xy"] + shift
    lp, tree = plan()
    lp.close()
    for node, c in zip(moved, _centre(tree, leaf)):
        assert np.abs(c).max() < 1e-14
        src["node_xy"][node] = c + r * np.array([0.8, -0.6])
    lp, tree2 = plan()
    assert np.array_equal(tree["root"], tree2["root"])
    kw = dict(sigma_S=sig, cS=1.0, sigma_D=sig, cD=0.5j)
    u = lp.eval(**kw)
    v = lp.eval(precision=qbxmod.QBX_MIXED, **kw)
    lp.close()
    assert np.isfinite(v).all()
    assert np.linalg.norm(u - v) < 1e-6 * np.linalg.norm(u)
