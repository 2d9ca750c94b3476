"""The staged searches at sizes that reach them (phases of fewer seeds go a
warp per seed, straight from global memory): the gray one for each specialised
patch side and the run-time one, one, two and more search candidates, both
search modes, a search on a grid only, every tile shape and the refresh alone;
and the bit-planes' two forms under the L1 cost.  Every field equals the
oracle's.  That the staged kernel ran is read from the evaluation counters:
it scores almost all candidates in its shared-memory window, the other
kernel none."""
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


def tiles(size):
    """Tiles of 8 x 8 seeds of one direction's level-0 lattice of stride 1."""
    return -(-size[0] // 8) * -(-size[1] // 8)


def check(api, prm, size, what):
    """A dense lattice whose level 0 has most of the work."""
    prm = dict(dict(levels=3, seed_stride=1, iters_coarse=1, iters_fine=3), **prm)
    # the level-0 seeds of a colour in both directions, against 128 per SM
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    assert 2 * ((size[0] + 1) // 2) * size[1] > 128 * sms, "phase too small for the staged kernels"
    mk = synth.sintel_like_pair if prm["color"] else synth.noise_affine_pair
    f1, f2, _ = mk(17, *size)
    (_, _, ws, rows, keep), (_, _, M, orows, okeep) = run_both(api, prm, f1, f2, stream_id=4)
    ev = ws.evals()
    total = sum(ev["pm"]) + sum(ev["cost"])
    assert 0 < sum(ev["pm_global"]) < 0.75 * total, ev
    compare_fields(ws, M, prm["levels"], what)
    assert (keep == okeep).all() and (rows == orows).all(), what


@pytest.mark.parametrize("name,prm,size", [
    ("15-11", dict(), (201, 133)),
    ("11-15", dict(patch_fwd=11, patch_bwd=15), (203, 131)),
    ("8-8", dict(patch_fwd=8, patch_bwd=8), (201, 133)),
    ("16-1", dict(patch_fwd=16, patch_bwd=1), (201, 133)),
    ("7-4", dict(patch_fwd=7, patch_bwd=4), (197, 140)),
    ("wide", dict(rs_W=9), (201, 133)),
    ("wide-8", dict(rs_W=5, patch_fwd=8, patch_bwd=6), (201, 133)),
    ("floor", dict(rs_W=4, rs_mode=1, patch_fwd=11, patch_bwd=8), (201, 133)),
    ("one-candidate", dict(rs_W=1), (201, 133)),
    ("grid", dict(rs_grid=4, patch_fwd=7, patch_bwd=5), (201, 133)),
    ("refresh-only", dict(iters_level=(0, 0, 0), refine_rounds=1), (201, 133)),
])
def test_gray(api, name, prm, size):
    check(api, dict(prm, color=0), size, name)


@pytest.mark.parametrize("tile_w", [4, 16])
def test_gray_tile_shapes(api, tile_w):
    from paper_1704_03217_gb300 import tune
    tune.set(tile_w=tile_w)
    try:
        check(api, dict(color=0, patch_fwd=15, patch_bwd=8), (205, 131), "tile_w %d" % tile_w)
    finally:
        tune.set()


@pytest.mark.parametrize("name,color,prm,size,per_lane", [
    ("gray-warp", 0, dict(patch_fwd=9, patch_bwd=16), (201, 133), False),
    ("gray-lane", 0, dict(patch_fwd=7, patch_bwd=5, rs_W=4), (259, 243), True),
    ("gray-lane-split", 0, dict(levels=4, patch_fwd=4, patch_bwd=3), (353, 341), True),
    ("colour-warp", 1, dict(patch_fwd=11, patch_bwd=16, rs_W=5), (201, 133), False),
    ("colour-lane", 1, dict(levels=4, patch_fwd=12, patch_bwd=11), (259, 243), True),
])
def test_bit_planes_under_l1(api, name, color, prm, size, per_lane):
    # a lane per seed from 12 tiles per SM, each direction alone above 24 of both
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    n = tiles(size) if 2 * tiles(size) > 24 * sms else 2 * tiles(size)
    assert (n >= 12 * sms) == per_lane
    check(api, dict(prm, color=color, descriptor=1, norm=1), size, name)
