"""Waits of the tensor-core initialisation that run out at different moments,
where patches are staged in chunks and where they are staged whole: the call
ends, a limit of a few cycles is reported as PGM_ERR_TIMEOUT, and with the
default limit the same pair is initialised exactly as before."""
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def api():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1704_03217_gb300 import build
    build.build()
    from paper_1704_03217_gb300 import api as A
    return A


@pytest.mark.parametrize("name,prm,size", [
    ("chunks", dict(levels=2, color=1, seed_stride=1), (499, 37)),
    ("chunks-stride2", dict(levels=2, color=1, seed_stride=2, patch_fwd=14, patch_bwd=5), (901, 37)),
    ("gray-chunks", dict(levels=1, color=0, seed_stride=2), (451, 37)),
    ("whole", dict(levels=2, color=1), (160, 96)),
])
def test_waits_that_run_out(api, name, prm, size):
    from paper_1704_03217_gb300 import _lib, synth
    L = _lib.load()
    mk = synth.sintel_like_pair if prm["color"] else synth.noise_affine_pair
    f1, f2, _ = mk(12, *size)
    n = prm["levels"]
    p = api.Params(**dict(prm, max_visits=1, iters_level=tuple([-1] * (n - 1) + [0])))
    P1 = api.build_pyramid(p, torch.from_numpy(f1).cuda())
    P2 = api.build_pyramid(p, torch.from_numpy(f2).cuda())
    ref = api.match(p, P1, P2, stream_id=5)
    ref.sync_status()
    want = {d: {k: v.clone() for k, v in ref.field(n - 1, d).items()} for d in (0, 1)}
    try:
        for limit in (2, 1000, 4000, 16000, 64000):       # cycles; nothing is staged within 2
            assert L.pgm_set_wait_limit(limit) == 0
            ws = api.match(p, P1, P2, stream_id=5)
            torch.cuda.synchronize()
            try:
                ws.sync_status()
                code = 0
            except _lib.PGMError as e:
                code = e.code
            assert code == 5 if limit == 2 else code in (0, 5), (name, limit, code)
            if code == 0:
                for d in (0, 1):
                    got = ws.field(n - 1, d)
                    for k in want[d]:
                        assert torch.equal(got[k], want[d][k]), (name, limit, d, k)
    finally:
        assert L.pgm_set_wait_limit(0) == 0
    again = api.match(p, P1, P2, stream_id=5)
    again.sync_status()
    for d in (0, 1):
        got = again.field(n - 1, d)
        for k in want[d]:
            assert torch.equal(got[k], want[d][k]), (name, d, k)
