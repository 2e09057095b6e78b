"""The host sampler's shared threads: the same bits from one thread and from
many, from calls that overlap, at sizes around its pieces, after the helpers
have gone idle and ended, and in a forked child (which has none of them)."""
import multiprocessing
import threading
import time

import numpy as np
import pytest

import aeb_inputs as ai


@pytest.fixture(scope="module")
def aeb():
    import paper_2604_27193_gb300 as m
    m.build()
    return m


def _draw(aeb, seed, n, threads, first=0):
    out = aeb.aeb_sample_params(ai.single_model(), ai.single_scenario(seed), first, n,
                                n_threads=threads)
    return b"".join(out[f].tobytes() for f in aeb.FIELDS)


@pytest.mark.parametrize("n", [1, 255, 256, 257, 511, 4097, 20_001])
@pytest.mark.parametrize("threads", [0, 2, 3, 64])
def test_same_bits_whatever_the_threads(aeb, n, threads):
    assert _draw(aeb, 5, n, threads, first=11) == _draw(aeb, 5, n, 1, first=11)


def test_overlapping_calls(aeb):
    want = [_draw(aeb, s, 3000 + 700 * s, 1) for s in range(8)]
    bad = []

    def work(s):
        for _ in range(20):
            if _draw(aeb, s, 3000 + 700 * s, 0) != want[s]:
                bad.append(s)

    ts = [threading.Thread(target=work, args=(s,)) for s in range(8)]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    assert not bad


def test_after_the_helpers_have_ended(aeb):
    want = _draw(aeb, 9, 10_000, 0)
    time.sleep(1.5)  # idle helpers end after a second
    assert _draw(aeb, 9, 10_000, 0) == want


def _child(q):
    import paper_2604_27193_gb300 as m
    q.put(_draw(m, 3, 10_000, 0))


def test_forked_child(aeb):
    want = _draw(aeb, 3, 10_000, 0)  # the parent has helpers now
    ctx = multiprocessing.get_context("fork")
    q = ctx.Queue()
    p = ctx.Process(target=_child, args=(q,))
    p.start()
    got = q.get(timeout=60)
    p.join(60)
    assert got == want and p.exitcode == 0
