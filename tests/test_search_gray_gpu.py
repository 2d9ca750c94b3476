"""The gray search with two seeds per warp: every field equals the oracle's on
images of more than one tile per SM (one launch per direction) and of fewer
(both directions in one), for each specialised patch side and the run-time one,
for more than two search candidates (drawn by the lanes), for a search on a
grid only and for odd tile tails."""
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
    ("15-11", dict(levels=3), (413, 307)),
    ("8-8", dict(levels=2, patch_fwd=8, patch_bwd=8, seed_stride=2), (251, 173)),
    ("16-1", dict(levels=2, patch_fwd=16, patch_bwd=1), (331, 290)),
    ("wide-search", dict(levels=3, rs_W=9), (413, 307)),
    ("floor-search", dict(levels=3, rs_W=4, rs_mode=1, patch_fwd=11, patch_bwd=15), (201, 133)),
    ("one-candidate", dict(levels=2, rs_W=1), (201, 133)),
    ("grid-search", dict(levels=2, rs_grid=4, patch_fwd=7, patch_bwd=5), (331, 290)),
    ("tiny", dict(levels=1, patch_fwd=3, patch_bwd=2), (9, 7)),
])
def test_gray_search_parity(api, name, prm, size):
    f1, f2, _ = synth.noise_affine_pair(21, *size)
    assert_parity(api, dict(prm, color=0), f1, f2, stream_id=3, what=name)
