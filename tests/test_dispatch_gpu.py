"""The rules that choose a kernel by size, on both sides of each line: the block
widths of the FP32 M2L (64, 96, 128 output orders, and more than one block), the
narrow and wide M2M / L2L kernels, and two centres per warp where there are at
least 8192 of them (an odd number, so that a half warp stays without one)."""
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


def _problem(k, panels, q, n_on):
    g = discretise_curve(*starfish(0.25, 5), panels, q, k=k)
    rng = np.random.default_rng(panels)
    sig = rng.standard_normal(g.n) + 1j * rng.standard_normal(g.n)
    node = np.arange(n_on, dtype=np.int64)
    off = 2.5 * np.exp(2j * np.pi * np.arange(21) / 21)
    tgt = np.concatenate([g.node_xy[node], np.stack([off.real, off.imag], -1)])
    node = np.concatenate([node, np.full(21, -1)])
    side = np.where(node >= 0, 1, 0).astype(np.int8)
    return g, sig, tgt, node, side


# box orders on either side of each width, at leaf sizes that give a few and many
# boxes; FP32 against FP64 of the same truncated expansions, within the mixed
# tolerance
@pytest.mark.parametrize("p_fmm,panels,n_max", [
    (8, 24, 16), (31, 160, 8), (32, 64, 24), (47, 100, 16), (48, 500, 16), (63, 64, 24), (64, 200, 64)])
def test_mixed_translations(qbxmod, p_fmm, panels, n_max):
    g, sig, tgt, node, side = _problem(0.8, panels, 16, panels * 16)
    lp = qbxmod.LayerPotential(g.as_dict(), 6, sides=2)
    assoc = lp.build(tgt, node, side, mode=qbxmod.QBX_FMM, p_fmm=p_fmm, n_max=n_max)
    kw = dict(sigma_S=sig, cS=1j, sigma_D=sig, cD=1.0)
    u = lp.eval(**kw)
    v = lp.eval(precision=qbxmod.QBX_MIXED, **kw)
    lp.close()
    for sel in (assoc >= 0, assoc < 0):
        assert np.linalg.norm((u - v)[sel]) < 1e-6 * np.linalg.norm(u[sel])


@pytest.mark.parametrize("mode,precision,p,layers,tol", [
    ("direct", "fp64", 0, "DS", 1e-10), ("direct", "fp64", 15, "S", 1e-10),
    ("direct", "fp64", 16, "DS", 1e-10), ("fmm", "fp64", 7, "D", 1e-10),
    ("fmm", "fp64", 16, "DS", 1e-10), ("fmm", "mixed", 1, "DS", 1e-6),
    ("fmm", "mixed", 12, "D", 1e-6), ("fmm", "mixed", 16, "S", 1e-6)])
def test_many_centres(qbxmod, oracle, mode, precision, p, layers, tol):
    g, sig, tgt, node, side = _problem(6.0, 513, 16, 8193)
    lp = qbxmod.LayerPotential(g.as_dict(), p, sides=2)
    assoc = lp.build(tgt, node, side, p_fmm=45, n_max=24,
                     mode=qbxmod.QBX_FMM if mode == "fmm" else qbxmod.QBX_DIRECT)
    kw = {}
    if "S" in layers:
        kw.update(sigma_S=sig, cS=0.7 - 2.2j)
    if "D" in layers:
        kw.update(sigma_D=sig, cD=1.1j)
    u = lp.eval(precision=qbxmod.QBX_MIXED if precision == "mixed" else qbxmod.QBX_FP64, **kw)
    lp.close()
    pick = np.concatenate([np.arange(0, 8193, 256), np.arange(8193 - 5, len(tgt))])
    u_ref, _ = oracle.layer_potential(
        g.as_dict(), tgt[pick], p, sigma_S=kw.get("sigma_S"), sigma_D=kw.get("sigma_D"),
        cS=kw.get("cS", 0.0), cD=kw.get("cD", 0.0), sides=2, centre_of_target=assoc[pick])
    assert (assoc[:8193] >= 0).all()
    assert np.linalg.norm(u[pick] - u_ref) < tol * np.linalg.norm(u_ref)
