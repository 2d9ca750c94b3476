"""Region removal on fields whose regions cross warps and rows in every way:
the exported matches equal the oracle's on random fields (thin, wide, narrower
and wider than a warp), on combs and spirals of one seed's width, on one region
that spans the field and on fields without a region."""
import ctypes as C

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

import oracle as O


def _spiral(n):
    a = np.zeros((n, n), bool)
    i, j, di, dj = 0, 0, 0, 1
    a[0, 0] = True
    for _ in range(n * n):
        i2, j2 = i + 2 * di, j + 2 * dj
        inside = 0 <= i2 < n and 0 <= j2 < n
        if not inside or a[i2, j2]:
            if 0 <= i + di < n and 0 <= j + dj < n and not inside and not a[i + di, j + dj]:
                pass
            di, dj = dj, -di
            if not (0 <= i + 2 * di < n and 0 <= j + 2 * dj < n) or a[i + 2 * di, j + 2 * dj]:
                break
            continue
        i, j = i + di, j + dj
        a[i, j] = True
    return a


def _case(name, ny, nx, rng):
    u = np.zeros((ny, nx), np.int64)
    if name == "random":
        keep = rng.random((ny, nx)) < 0.6
        u = rng.choice([0, 3, 14, 40], size=(ny, nx), p=[0.7, 0.1, 0.1, 0.1])
    elif name == "comb":                       # teeth joined by the last row alone
        keep = np.zeros((ny, nx), bool)
        keep[:, ::2] = True
        keep[-1] = True
    elif name == "spiral":
        keep = _spiral(max(ny, nx))[:ny, :nx]
    elif name == "steps":                      # every row another motion: runs only
        keep = np.ones((ny, nx), bool)
        u = np.repeat(np.arange(ny)[:, None] * 12, nx, 1)
    else:
        keep = np.full((ny, nx), name == "all")
    return u, keep


@pytest.mark.parametrize("name,ny,nx", [
    ("random", 37, 61), ("random", 1, 300), ("random", 300, 1), ("random", 64, 32), ("random", 150, 333),
    ("comb", 40, 97), ("spiral", 75, 75), ("steps", 20, 129), ("all", 131, 257), ("none", 9, 40)])
def test_regions_equal_oracle(name, ny, nx):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1704_03217_gb300 import _lib, api, build
    build.build()
    L = _lib.load()
    rng = np.random.default_rng(ny * 1000 + nx)
    ux, valid = _case(name, ny, nx, rng)
    uy = np.zeros_like(ux)
    outl = (rng.random((ny, nx)) < 0.1) if name == "random" else np.zeros((ny, nx), bool)
    prm = api.Params(min_region=5)
    u = torch.from_numpy(((ux & 0xffff) | (uy << 16)).astype(np.int32)).cuda()
    f = torch.from_numpy((valid.astype(np.uint8) | (outl.astype(np.uint8) << 1))).cuda()
    rows = torch.zeros((ny * nx, 4), dtype=torch.int32, device="cuda")
    cnt = torch.zeros(1, dtype=torch.int32, device="cuda")
    code = L.pgm_filter_noalloc(C.byref(prm.cstruct()), nx, ny, C.c_void_p(u.data_ptr()),
                                C.c_void_p(f.data_ptr()), C.c_void_p(rows.data_ptr()), ny * nx,
                                C.c_void_p(cnt.data_ptr()),
                                C.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert code == 0
    torch.cuda.synchronize()
    want, _ = O.filter_arrays(dict(min_region=5), ux, uy, valid, outl)
    got = rows[:int(cnt.item())].cpu().numpy()
    assert got.shape == want.shape and (got == want).all()
