"""The tensor-core initialisation where patches are staged in chunks of rows
(wide or dense lattices) and on the two-channel descriptor: the coarsest
level's fields right after it equal the oracle's brute force at every seed."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from paper_1704_03217_gb300 import synth
from pgm_compare import compare_fields, run_both


@pytest.fixture(scope="module")
def api():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1704_03217_gb300 import build
    build.build()
    from paper_1704_03217_gb300 import api as A
    return A


@pytest.mark.parametrize("name,prm,size", [
    ("dense", dict(levels=2, color=1, seed_stride=1), (499, 17)),          # 15 and 11 in chunks
    ("stride2", dict(levels=2, color=1, seed_stride=2, patch_fwd=14, patch_bwd=5), (901, 37)),
    ("one-row-chunks", dict(levels=1, color=1, seed_stride=5, patch_fwd=15, patch_bwd=12), (731, 21)),
    ("gray", dict(levels=4, color=0), (501, 157)),
    ("gray-dense", dict(levels=2, color=0, seed_stride=1), (401, 19)),
    ("gray-even", dict(levels=3, color=0, patch_fwd=8, patch_bwd=12, seed_stride=2), (300, 90)),
    ("gray-small", dict(levels=2, color=0, patch_fwd=1, patch_bwd=2), (61, 33)),
])
def test_init_equals_brute_force(api, name, prm, size):
    mk = synth.sintel_like_pair if prm["color"] else synth.noise_affine_pair
    f1, f2, _ = mk(9, *size)
    L = prm["levels"]
    p = dict(prm, max_visits=1, iters_level=tuple([-1] * (L - 1) + [0]))
    (_, _, ws, _, _), (_, _, M, _, _) = run_both(api, p, f1, f2, stream_id=2)
    compare_fields(ws, M, L, name)
    assert ws.field(L - 1, 0)["valid"].all().item(), name
