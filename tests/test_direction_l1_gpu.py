"""The direction descriptor under the L1 cost, through every visit: the search
kernels that take the bit-planes also refresh the costs of a visit's current
matches, whichever the norm."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from paper_1704_03217_gb300 import synth
from pgm_compare import assert_parity


@pytest.mark.parametrize("name,prm,size", [
    ("gray", dict(levels=3, color=0), (140, 90)),
    ("colour", dict(levels=3, color=1), (301, 157)),
])
def test_direction_l1_parity(name, prm, size):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1704_03217_gb300 import build
    build.build()
    from paper_1704_03217_gb300 import api
    mk = synth.sintel_like_pair if prm["color"] else synth.noise_affine_pair
    f1, f2, _ = mk(31, *size)
    assert_parity(api, dict(prm, descriptor=1, norm=1), f1, f2, stream_id=9, what=name)
