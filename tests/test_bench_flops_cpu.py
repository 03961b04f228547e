"""bench.py's flop model in direct mode, which runs FP64 kernels in either precision."""
import importlib.util
import os

from tests.conftest import ROOT


def test_direct_mode_is_charged_in_fp64():
    spec = importlib.util.spec_from_file_location("bench", os.path.join(ROOT, "bench.py"))
    bench = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(bench)
    stats = dict(p2qbxl_pairs=1000, p2p_pairs=500, n_qbx_targets=20)
    f = [bench.flop_model(None, stats, 8, True, True, None, False, mixed=m)
         for m in (False, True)]
    assert f[0] == f[1] and all(v[1] == 0.0 for v in f[1].values())
