"""The tensor-core initialisation's staging in chunks of patch rows and its
gray runs, on a CPU model (no GPU): for images wider than a seed tile, for
patches cut into chunks, and for the two-channel descriptor, every read of a
step stays inside its staged buffer, second offsets are positive, and the
accumulated cross terms equal a direct correlation of border-replicated
patches."""
import numpy as np
import pytest

BORD, M, N, NT, NTC = 8, 128, 160, 2, 4


def lattice_n(W, s):
    return (W - 1 - s // 2) // s + 1


def geom(P, s, nx, ny, tw, th, Q, nchunk, gray):
    e = (P - 1) // s
    g = dict(e=e, Wu=nx + e, ph=s * s, copies=2 if gray and P % 4 else 1)
    g["mtiles"] = -(-ny * g["Wu"] // M)
    ra = M + e + 1
    g["pa"] = min(g["Wu"], ra)
    g["LA"] = g["pa"] * (Q - 1) + ra
    g["NT"] = 1 if nchunk > 1 else NT
    g["Wt"] = tw + P - 1
    g["ntiles"] = -(-th * g["Wt"] // N)
    rb, rows = g["NT"] * N + P - 1, min(Q * s, P)
    g["pb"] = min(g["Wt"], rb)
    g["LB"] = g["pb"] * (rows - 1) + rb
    return g


def chunk_steps(P, s, g, gray, Q, c):
    """(a1, a2, b1, b2) offsets of every step of chunk c (b2 None: zeros)."""
    ra, rb = c * Q * s, min(P, (c + 1) * Q * s)
    tail = 4 * ((P - 1) // 4)
    us = [(p, r) for r in range(ra, rb) for p in range(0, P, 4 if gray else 1)]

    def aoff(p, r):
        cp = 1 if gray and g["copies"] == 2 and p == tail else 0
        return ((cp * s + r % s) * s + p % s) * g["LA"] + ((r - ra) // s) * g["pa"] + p // s

    key = lambda u: (gray and P % 4 and u[0] == tail, u[1] % s, u[0] % s, u[1] // s, u[0] // s)
    used, out = set(), []
    for i, u in enumerate(us):
        if u in used:
            continue
        used.add(u)
        v = next((v for v in us[i + 1:] if v not in used and key(v) > key(u)), None)
        b1 = (u[1] - ra) * g["pb"] + u[0]
        if v is None:
            out.append((aoff(*u), aoff(*u) + 1, b1, None))
        else:
            used.add(v)
            out.append((aoff(*u), aoff(*v), b1, (v[1] - ra) * g["pb"] + v[0]))
    return out


def unit(img, X, Y, gray, keep=4):
    """Staged unit(s) at arrays X, Y of a (h, w, c) image with replicated border."""
    h, w, c = img.shape
    y = np.clip(np.clip(Y, -BORD, h + BORD - 1), 0, h - 1)
    if not gray:
        x = np.clip(np.clip(X, -BORD, w + BORD - 1), 0, w - 1)
        return np.concatenate([img[y, x], np.zeros(x.shape + (2,), img.dtype)], -1)
    out = []
    for k in range(4):
        x = np.clip(np.clip(X + k, -BORD, w + BORD - 1), 0, w - 1)
        out.append(img[y, x] * (k < keep))
    return np.concatenate(out, -1)


@pytest.mark.parametrize("P,s,w,h,tw,th,Q,gray", [
    (15, 1, 150, 20, 190, 23, 5, False),        # three chunks, runs shorter than a row
    (11, 1, 200, 17, 97, 30, 4, False),         # a last chunk of fewer rows
    (15, 3, 420, 40, 210, 31, 2, False),        # three chunks of 6 patch rows, ragged
    (8, 2, 300, 25, 40, 33, 1, False),          # a chunk per two rows
    (5, 3, 40, 30, 44, 28, 2, False),           # whole patch in one chunk
    (15, 3, 60, 40, 71, 37, 5, True),           # gray, one chunk, masked last run
    (15, 1, 160, 20, 150, 22, 5, True),
    (8, 3, 90, 30, 100, 31, 3, True),           # P a multiple of four: no second copy
    (11, 2, 130, 21, 70, 25, 2, True),
    (1, 3, 20, 11, 30, 12, 1, True),
])
def test_chunked_staging_gives_exact_cross_terms(P, s, w, h, tw, th, Q, gray):
    rng = np.random.default_rng(P * 100 + s * 10 + Q)
    C = 2 if gray else 6
    ref = rng.integers(-12240, 12241, size=(h, w, C)).astype(np.int64)
    tgt = rng.integers(-12240, 12241, size=(th, tw, C)).astype(np.int64)
    nx, ny, c0, hp = lattice_n(w, s), lattice_n(h, s), s // 2, P // 2
    nchunk = -(-((P - 1) // s + 1) // Q)
    g = geom(P, s, nx, ny, tw, th, Q, nchunk, gray)
    tail, o = 4 * ((P - 1) // 4), c0 - hp
    rows = min(Q * s, P)
    assert 2 ** 14 > g["ph"] * g["copies"] * g["LA"] and 2 ** 14 > g["LB"]
    for mt in sorted({0, g["mtiles"] // 2, g["mtiles"] - 1}):
        for tile in sorted({0, g["ntiles"] // 3, g["ntiles"] - 1}):
            acc = np.zeros((M, N), np.int64)
            if nchunk == 1:                          # staged for two tiles from an even one
                t0, kb = tile - tile % NT, (tile % NT) * N
            else:
                t0, kb = tile, 0
            nsteps = 0
            for c in range(nchunk):
                e = np.arange(g["ph"] * g["LA"])
                ph, k = e // g["LA"], e % g["LA"]
                q = np.minimum(k // g["pa"], Q - 1)
                f = mt * M + (c * Q + q) * g["Wu"] + k - q * g["pa"]
                X, Y = s * (f % g["Wu"]) + ph % s + o, s * (f // g["Wu"]) + ph // s + o
                A = unit(ref, X, Y, gray)
                if g["copies"] == 2:
                    A = np.concatenate([A, unit(ref, X, Y, gray, P - tail)])
                k = np.arange(g["LB"])
                r = np.minimum(k // g["pb"], rows - 1)
                f = t0 * N + (c * Q * s + r) * g["Wt"] + k - r * g["pb"]
                B = unit(tgt, f % g["Wt"] - hp, f // g["Wt"] - hp, gray)
                for a1, a2, b1, b2 in chunk_steps(P, s, g, gray, Q, c):
                    nsteps += 1
                    assert a2 > a1 and (b2 is None or b2 > b1)
                    assert max(a1, a2) + M <= len(A) and max(b1, b2 or 0) + kb + N <= len(B)
                    acc += A[a1:a1 + M] @ B[b1 + kb:b1 + kb + N].T
                    if b2 is not None:
                        acc += A[a2:a2 + M] @ B[b2 + kb:b2 + kb + N].T
            assert nsteps <= 128
            pad = lambda im: np.pad(im, ((hp, P), (hp, P), (0, 0)), mode="edge")
            rp, tp = pad(ref), pad(tgt)
            for m in range(0, M, 7):
                i, j = (mt * M + m) % g["Wu"], (mt * M + m) // g["Wu"]
                if i >= nx or j >= ny:
                    continue
                a = rp[c0 + s * j:c0 + s * j + P, c0 + s * i:c0 + s * i + P]
                for n in range(0, N, 11):
                    x, y = (tile * N + n) % g["Wt"], (tile * N + n) // g["Wt"]
                    if x >= tw or y >= th:
                        continue
                    assert acc[m, n] == (a * tp[y:y + P, x:x + P]).sum(), (mt, tile, m, n)
