"""Search phases of few seeds (a warp per seed, patches read from global
memory): every field equals the oracle's for both descriptors and channel
counts, even, odd and largest patches, more than two search candidates, the
refresh alone (a level without iterations), lattices of one seed and ragged
rows, and a batch of unequal sizes against each pair alone."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from paper_1704_03217_gb300 import synth
from pgm_compare import assert_parity


@pytest.fixture(scope="module")
def api():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1704_03217_gb300 import build
    build.build()
    from paper_1704_03217_gb300 import api as A
    return A


@pytest.mark.parametrize("name,prm,size", [
    ("colour", dict(levels=3, color=1), (121, 83)),
    ("colour-16-1", dict(levels=2, color=1, patch_fwd=16, patch_bwd=1), (97, 61)),
    ("gray-wide", dict(levels=3, color=0, rs_W=9, patch_fwd=8, patch_bwd=13), (121, 83)),
    ("bits", dict(levels=3, color=1, descriptor=1), (121, 83)),
    ("bits-gray-l1", dict(levels=3, color=0, descriptor=1, norm=1, rs_W=5, patch_fwd=16), (140, 90)),
    ("sector", dict(levels=2, color=1, descriptor=2, rs_grid=2), (97, 61)),
    ("refresh-only", dict(levels=3, color=1, iters_level=(2, 0, 3)), (121, 83)),
    ("one-seed", dict(levels=1, color=0, seed_stride=7), (7, 7)),
    ("dense", dict(levels=2, color=1, seed_stride=1, patch_fwd=5, patch_bwd=3), (33, 21)),
])
def test_direct_search_parity(api, name, prm, size):
    mk = synth.sintel_like_pair if prm["color"] else synth.noise_affine_pair
    f1, f2, _ = mk(31, *size)
    assert_parity(api, prm, f1, f2, stream_id=9, what=name)


def test_direct_search_batch(api):
    """Pairs of unequal sizes in shared launches, each as alone."""
    p = api.Params(levels=3, color=1)
    sizes = [(64, 48), (121, 83), (97, 150)]
    one, P1, P2 = [], [], []
    for k, (w, h) in enumerate(sizes):
        f1, f2, _ = synth.sintel_like_pair(40 + k, w, h)
        a, b = torch.from_numpy(f1).cuda(), torch.from_numpy(f2).cuda()
        P1.append(api.build_pyramid(p, a))
        P2.append(api.build_pyramid(p, b))
        one.append(api.match(p, P1[-1], P2[-1], stream_id=k))
    ws = [api.Workspace(p, w, h, w, h) for w, h in sizes]
    api.match_batch(p, P1, P2, [0, 1, 2], ws)
    torch.cuda.synchronize()
    for a, b in zip(one, ws):
        b.sync_status()
        for l in range(3):
            for d in (0, 1):
                x, y = a.field(l, d), b.field(l, d)
                for k in x:
                    assert np.array_equal(x[k].cpu().numpy(), y[k].cpu().numpy()), (l, d, k)
