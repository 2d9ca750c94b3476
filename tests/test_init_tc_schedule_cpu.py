"""The schedule of the tensor-core initialisation's CTA on a model of its
parity-waited mbarriers (CPU only): worker warps that stage chunks and read
accumulators, one issuing thread, and the tensor pipe that completes its
commits at some later time.  Every bounded wait may run out at any moment, as
it may on the GPU, where the lanes of a warp look at the barrier, the abort
flag and the clock one after another.  All interleavings of two workers are
walked: each ends with every warp at the block's last barrier, behind which no
product is in flight when the tensor memory is freed; no wait passes
on a phase that it does not mean; a centre table is read complete and not
written meanwhile; a buffer is not staged again under the products that read
it; and accumulators are neither read before their products
are complete nor overwritten before every worker has read them."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1704_03217_gb300", "csrc")


def worker(nchunk, ntile, meet):
    """The operations of a worker warp.  meet: how the workers meet before
    the tables are read, "mbarrier" (bounded) or "named" (no limit)."""
    ops, nstage = [], nchunk * ntile
    if nchunk == 1:
        ops += [("write", k) for k in range(ntile)] + [("arrive", "full0", 0)]
        ops += [("arrive", "tab", 0), ("wait", "tab", 0)] if meet == "mbarrier" else [("sync",)]
        for k in range(ntile):
            ops += [("wait", "done0", k), ("read", k), ("arrive", "acc", k)]
        return ops + [("join",)]
    for i in range(nstage + 1):
        b, k, c = i & 1, i // nchunk, i % nchunk
        if i > 0 and c == 0 and meet == "mbarrier":
            ops.append(("wait", "tab", k - 1))
        if i < nstage:
            if i >= 2:
                ops.append(("wait", "done%d" % b, i // 2 - 1))
            if c == 0:
                ops.append(("write", k))
            ops.append(("arrive", "full%d" % b, i // 2))
        if i > 0 and c == 0:
            if meet == "named":
                ops.append(("sync",))
            ops += [("wait", "done%d" % (b ^ 1), (i - 1) // 2), ("read", k - 1), ("arrive", "acc", k - 1)]
        if c == 0 and i < nstage and meet == "mbarrier":
            ops.append(("arrive", "tab", k))
    return ops + [("join",)]


def issuer(nchunk, ntile, drain):
    """drain: who waits for the products in flight after an abort: "joined",
    the issuer behind the block's barrier, or "own", the issuer when its own
    wait ran out."""
    ops = []
    for k in range(ntile):
        if k:
            ops.append(("wait", "acc", k - 1))
        for c in range(nchunk):
            i = k * nchunk + c if nchunk > 1 else 0
            b = i & 1 if nchunk > 1 else 0
            if nchunk > 1 or k == 0:
                ops.append(("wait", "full%d" % b, i // 2))
            ops.append(("issue", k, b))
    return ops + ([("drain",)] if drain == "own" else []) + [("join",)]


BARS = ("full0", "full1", "done0", "done1", "acc", "tab")


def walk(nchunk, ntile, meet, failing, drain="joined", workers=2):
    """Every interleaving; a violation message or None.  failing: waits may
    run out."""
    progs = [worker(nchunk, ntile, meet)] * workers + [issuer(nchunk, ntile, drain)]
    count = {b: 1 if b.startswith("done") else workers for b in BARS}
    # program counters; barriers (phase, arrived); abort; commits in flight
    # (tile, buffer); tiles of both tables' parts per worker; workers that
    # have read each tile; products completed
    start = ((0,) * (workers + 1), tuple((0, 0) for _ in BARS), False, (),
             ((None,) * workers,) * 2, (0,) * ntile, 0)
    todo, seen = [start], {start}
    while todo:
        pcs, bars, abort, flight, tabs, reads, done = state = todo.pop()
        out = []

        def arrive(bs, name):
            j = BARS.index(name)
            ph, n = bs[j]
            n += 1
            new = (ph + 1, 0) if n == count[name] else (ph, n)
            return bs[:j] + (new,) + bs[j + 1:]

        def step(a, pc, **kw):
            s = dict(bars=bars, abort=abort, flight=flight, tabs=tabs, reads=reads, done=done)
            s.update(kw)
            out.append((pcs[:a] + (pc,) + pcs[a + 1:], s["bars"], s["abort"], s["flight"], s["tabs"],
                        s["reads"], s["done"]))

        if flight:                                         # the oldest commit's products complete
            out.append((pcs, arrive(bars, "done%d" % flight[0][1]), abort, flight[1:], tabs, reads,
                        done + 1))
        for a, prog in enumerate(progs):
            op, pc = prog[pcs[a]], pcs[a]
            if op[0] == "join":
                continue
            if op[0] == "wait":
                ph = bars[BARS.index(op[1])][0]
                if ph % 2 != op[2] % 2:
                    if ph != op[2] + 1:
                        return "wait for phase %d of %s passed in phase %d" % (op[2], op[1], ph)
                    step(a, pc + 1)
                if failing:                                # (abort seen, or out of time)
                    step(a, len(prog) - (2 if prog[-2] == ("drain",) else 1), abort=True)
            elif op[0] == "drain":
                if not flight:
                    step(a, pc + 1)
            elif op[0] == "arrive":
                if op[1].startswith("full") and nchunk > 1 and done < 2 * op[2] + int(op[1][4]) - 1:
                    return "buffer %s restaged under its products" % op[1][4]
                step(a, pc + 1, bars=arrive(bars, op[1]))
            elif op[0] == "sync":                          # no limit: passes when every worker is there
                if all(progs[w][pcs[w]] == op for w in range(workers)):
                    out.append((tuple(p + 1 for p in pcs[:workers]) + pcs[workers:], bars, abort, flight,
                                tabs, reads, done))
            elif op[0] == "write":                         # this worker's part of the table
                if op[1] >= 2 and reads[op[1] - 2] < workers:
                    return "table of tile %d overwritten under a reader" % (op[1] - 2)
                t = tabs[op[1] & 1]
                t = t[:a] + (op[1],) + t[a + 1:]
                step(a, pc + 1, tabs=(t, tabs[1]) if op[1] & 1 == 0 else (tabs[0], t))
            elif op[0] == "read":
                k = op[1]
                if tabs[k & 1] != (k,) * workers:
                    return "table of tile %d read as %s" % (k, tabs[k & 1])
                if done < (k + 1) * nchunk:
                    return "accumulators of tile %d read after %d commits" % (k, done)
                step(a, pc + 1, reads=reads[:k] + (reads[k] + 1,) + reads[k + 1:])
            elif op[0] == "issue":
                k = op[1]
                if k and reads[k - 1] < workers:
                    return "accumulators of tile %d overwritten before they were read" % (k - 1)
                step(a, pc + (2 if prog[pc + 1] == ("drain",) else 1), flight=flight + ((k, op[2]),))
        if flight and all(progs[a][pcs[a]] == ("join",) for a in range(workers + 1)):
            if drain == "own" or not abort:
                return "tensor memory freed under %d commits" % len(flight)
            if len({b for _, b in flight}) < len(flight):
                return "two commits outstanding on one buffer"
        if not out:
            if any(progs[a][pcs[a]] != ("join",) for a in range(workers + 1)):
                return "stuck at %s" % [progs[a][pcs[a]] for a in range(workers + 1)]
            if not failing and reads != (workers,) * ntile:
                return "ended early"
        for s in out:
            if s not in seen:
                seen.add(s)
                todo.append(s)
    return None


SHAPES = [(1, 1), (1, 2), (2, 1), (2, 2), (2, 4), (3, 1), (3, 2), (3, 4), (4, 3), (5, 2), (15, 2)]


@pytest.mark.parametrize("nchunk,ntile", SHAPES)
def test_every_interleaving_is_ordered(nchunk, ntile):
    assert walk(nchunk, ntile, "mbarrier", False) is None


@pytest.mark.parametrize("nchunk,ntile", SHAPES)
def test_every_interleaving_ends_when_waits_run_out(nchunk, ntile):
    assert walk(nchunk, ntile, "mbarrier", True) is None


@pytest.mark.parametrize("nchunk,ntile", [(3, 1), (2, 2), (3, 2)])
def test_a_barrier_without_a_limit_strands_a_worker(nchunk, ntile):
    """Workers that met on a named barrier after bounded waits: one leaves on
    a wait that ran out, another passes it and waits for the first for ever."""
    assert walk(nchunk, ntile, "named", False) is None
    assert "stuck" in walk(nchunk, ntile, "named", True)


@pytest.mark.parametrize("nchunk,ntile", [(1, 1), (1, 2), (2, 2), (3, 1)])
def test_a_drain_on_the_issuers_own_failure_alone_is_not_enough(nchunk, ntile):
    """A worker's wait runs out after the issuer has issued everything."""
    assert walk(nchunk, ntile, "mbarrier", False, drain="own") is None
    assert "freed" in walk(nchunk, ntile, "mbarrier", True, drain="own")


def test_the_kernel_has_no_other_unbounded_barrier():
    src = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, "init_tc.cu")).read())
    assert not re.search(r"\b(bar|barrier)\.(cta\.)?(sync|red|arrive)\b", src)
