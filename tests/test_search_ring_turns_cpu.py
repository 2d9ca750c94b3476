"""The search kernels' ring with one full and one empty barrier per buffer,
every interleaving on a model of parity-waited mbarriers (CPU only).  A
producer reads the seeds of tile n, waits for its turn (handed on by the
producer of tile n - 1 once that is staged), waits until the buffer's last tile
is released, and stages; consumers take every tile.  No buffer is refilled
before its tile has been read, and no consumer reads another tile than its own.

Without turns a ring of fewer buffers than producers is not safe: a producer
can come to a buffer whose last tile but one is still held, and the parity of
that phase is the one that it waits for."""
import pytest


def walk(tiles, nbuf, nprod, ncons, turns):
    """A violation message or None."""
    # producers: (tile, past its turn); consumers: (tile, reading); barriers of
    # the buffers: (phase, arrivals); turns: phases; contents: (tile, copied)
    start = (tuple((p, False) for p in range(nprod)), ((0, False),) * ncons, ((0, 0),) * nbuf,
             ((0, 0),) * nbuf, (0,) * nprod, (None,) * nbuf, ())
    todo, seen = [start], {start}

    def put(t, i, v):
        return t[:i] + (v,) + t[i + 1:]

    def arrive(bars, b, count):
        ph, k = bars[b]
        return put(bars, b, (ph + 1, 0) if k + 1 == count else (ph, k + 1))

    while todo:
        prod, cons, full, empty, turn, content, flight = todo.pop()
        out = []
        for x, (b, n) in enumerate(flight):                # a copy lands
            out.append((prod, cons, arrive(full, b, 1), empty, turn, put(content, b, (n, True)),
                        flight[:x] + flight[x + 1:]))
        for p, (n, ready) in enumerate(prod):
            if n >= tiles:
                continue
            if not ready:
                if turns and n > 0 and turn[p] % 2 == (n // nprod - (p == 0)) & 1:
                    continue
                out.append((put(prod, p, (n, True)), cons, full, empty, turn, content, flight))
                continue
            b = n % nbuf
            if n >= nbuf and empty[b][0] % 2 == (n // nbuf - 1) & 1:
                continue
            if content[b] is not None and min(c[0] for c in cons) <= content[b][0]:
                return "tile %d in buffer %d refilled with %d" % (content[b][0], b, n)
            q = (p + 1) % nprod
            out.append((put(prod, p, (n + nprod, False)), cons, full, empty,
                        put(turn, q, turn[q] + 1) if turns else turn, put(content, b, (n, False)),
                        tuple(sorted(flight + ((b, n),)))))
        for c, (n, reading) in enumerate(cons):
            if n >= tiles:
                continue
            b = n % nbuf
            if reading:
                out.append((prod, put(cons, c, (n + 1, False)), full, arrive(empty, b, ncons), turn,
                            content, flight))
            elif full[b][0] % 2 != (n // nbuf) & 1:
                if content[b] != (n, True):
                    return "consumer of tile %d read %s" % (n, content[b])
                out.append((prod, put(cons, c, (n, True)), full, empty, turn, content, flight))
        if not out and any(c[0] < tiles for c in cons):
            return "stuck"
        for s in out:
            if s not in seen:
                seen.add(s)
                todo.append(s)
    return None


@pytest.mark.parametrize("nprod,nbuf", [(2, 2), (2, 3), (4, 2), (4, 3), (4, 4), (4, 5), (4, 8)])
def test_rings_with_turns_are_safe(nprod, nbuf):
    """Two producers on 2 or 3 buffers (int16 descriptors), four on 2 to 8 (bit-planes)."""
    assert walk(14, nbuf, nprod, 2 if nbuf < 5 else 1, True) is None


@pytest.mark.parametrize("nprod,nbuf", [(2, 1), (4, 2), (4, 3)])
def test_fewer_buffers_than_producers_need_turns(nprod, nbuf):
    assert walk(14, nbuf, nprod, 2, False) is not None
