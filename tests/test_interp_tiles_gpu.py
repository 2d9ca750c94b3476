"""Interpolation lists across many tiles and launches: sparse matches on an
image of several hundred tiles (long paths, tiles open and stable in turn,
neighbours found late), a single match whose list reaches every tile, ragged
tiles at the right and lower edge, and every specialised and run-time k."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

from test_interp_gpu import api, compare, gpu_interp, oracle_interp  # noqa: F401


@pytest.mark.parametrize("k,n,size", [(16, 60, (401, 259)), (8, 25, (401, 259)), (3, 9, (130, 65)),
                                      (16, 1, (273, 150)), (16, 3000, (257, 255))])
def test_lists_across_tiles(api, k, n, size):  # noqa: F811
    from paper_1704_03217_gb300 import synth
    w, h = size
    img, _, _ = synth.sintel_like_pair(5, w, h, t_max=10.0)
    rng = np.random.default_rng(k * 1000 + n)
    rows = np.stack([rng.integers(0, w, n), rng.integers(0, h, n), rng.integers(0, w, n),
                     rng.integers(0, h, n)], 1).astype(np.int32)
    prm_d = dict(levels=2, color=1)
    ip = api.InterpParams(k=k, cost_shift=6)
    flow, keys = gpu_interp(api, api.Params(**prm_d), img, rows, ip)
    okeys, oflow, _ = oracle_interp(prm_d, img, rows, ip)
    compare(flow, keys, okeys, oflow, "k %d n %d" % (k, n))
