"""Level images, converted images and descriptors of narrow images of every
width from 1 to 44: the last words of rows and the borders of the kernels that
make four pixels a thread, and blocks of several levels and directions in one
launch, equal the oracle's."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

import oracle as O
from pgm_compare import compare_pyramid


@pytest.mark.parametrize("color,descriptor,h", [(1, 0, 7), (0, 1, 20), (1, 1, 33)])
def test_every_width(color, descriptor, h):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1704_03217_gb300 import api, build
    build.build()
    prm = dict(levels=3, color=color, descriptor=descriptor)
    p = api.Params(**prm)
    rng = np.random.default_rng(h)
    imgs = [rng.integers(0, 256, size=(h, w, 3) if color else (h, w), dtype=np.uint8)
            for w in range(1, 45)]
    dev = [torch.from_numpy(i).cuda() for i in imgs]
    pyrs = [api.Pyramid(p, i.shape[1], i.shape[0]) for i in imgs]
    api.build_pyramids(p, dev, pyrs)                 # 44 images: several launches' items
    torch.cuda.synchronize()
    for i, q in zip(imgs, pyrs):
        compare_pyramid(q, O.Pyramid(O.make_params(prm), i), "w %d" % i.shape[1])
