"""Interpolation where entries travel far: one match on long images lower than
a tile, and corridors that wind through the image, whose paths are many times
the image's sides.  The call settles, and its lists equal the oracle's."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

from test_interp_gpu import api, compare, gpu_interp, oracle_interp  # noqa: F401


def serpentine(w, h, pitch, gap):
    """Dark corridors `pitch` rows high between bright lines that leave a gap
    at alternate ends."""
    img = np.zeros((h, w), np.uint8)
    for n, y in enumerate(range(pitch, h - 2, pitch)):
        img[y:y + 2, :] = 255
        img[y:y + 2, (slice(0, gap) if n & 1 else slice(w - gap, w))] = 0
    return img


def check(api, img, rows, ip, what):  # noqa: F811
    prm_d = dict(levels=1, color=0)
    rows = np.asarray(rows, np.int32)
    flow, keys = gpu_interp(api, api.Params(**prm_d), img, rows, ip)
    okeys, oflow, _ = oracle_interp(prm_d, img, rows, ip)
    compare(flow, keys, okeys, oflow, what)


@pytest.mark.parametrize("w,h", [(1024, 8), (2048, 12), (2048, 8), (3000, 1), (1, 1500), (8, 1024)])
def test_one_match_on_a_long_image(api, w, h):  # noqa: F811
    rng = np.random.default_rng(w + h)
    img = rng.integers(0, 256, size=(h, w)).astype(np.uint8)
    check(api, img, [[0, 0, 5, 3]], api.InterpParams(), "%dx%d" % (w, h))


@pytest.mark.parametrize("w,h,pitch,shift,k", [(256, 192, 12, 0, 16), (256, 256, 9, 0, 3),
                                               (128, 512, 12, 6, 8)])
def test_winding_corridors(api, w, h, pitch, shift, k):  # noqa: F811
    check(api, serpentine(w, h, pitch, 24), [[1, 1, 2, 3], [4, 2, 9, 9]],
          api.InterpParams(k=k, cost_shift=shift), "serpentine %dx%d" % (w, h))
