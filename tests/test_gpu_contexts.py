"""Contexts of different meshes side by side, each driven by a thread of its own.

A context's calls are serialized by its caller; different contexts run at the same time, on streams of their
own.  Every sum is added in a fixed order, so each thread gets the bits that its context gives alone.
"""
import threading

import numpy as np
import pytest

from paper_2007_14228_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ofks():
    from paper_2007_14228_gb300 import build
    build.build()
    from paper_2007_14228_gb300 import ofks as mod
    return mod


def evaluations(ofks, cells, p, count, start=None):
    s = I.lih().with_cells(cells).with_p(p, occ=1.0)
    m = I.make_mesh(s)
    X = I.initial_block(m.n_free, p, 5)
    ctx = ofks.context_for(s, m, beta=10.0)
    if start is not None:
        start.wait()
    out = []
    for i in range(count):
        ctx.set_orbitals(X * (1.0 - 0.01 * (i % 3)))
        r = ctx.evaluate()
        out.append((r["e_total"], r["kkt"], r["hartree_iters"], ctx.get_field("U"), ctx.get_field("G")))
    ctx.close()
    return out


# one persistent Hartree solve per SM in every pair; axes of 15 to 127 points, 1 to 152 CTAs, few and many columns
@pytest.mark.parametrize("cells", [[(8, 8, 8), (9, 8, 10)], [(8, 8, 8), (24, 24, 24)], [(64, 6, 5), (24, 24, 24)],
                                   [(8, 8, 8), (8, 8, 9), (12, 10, 9)]], ids=str)
def test_threads_get_the_same_bits_as_alone(ofks, cells):
    jobs = [(c, 2 if i % 2 == 0 else 17, 12) for i, c in enumerate(cells)]
    alone = [evaluations(ofks, *j) for j in jobs]
    got, start = [None] * len(jobs), threading.Barrier(len(jobs))

    def work(i):
        try:
            got[i] = evaluations(ofks, *jobs[i], start)
        except Exception as e:                    # noqa: BLE001 (reported by the main thread)
            got[i] = e
            start.abort()

    threads = [threading.Thread(target=work, args=(i,)) for i in range(len(jobs))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for a, g in zip(alone, got):
        assert not isinstance(g, Exception), g
        for x, y in zip(a, g):
            assert x[:3] == y[:3]
            assert np.array_equal(x[3], y[3]) and np.array_equal(x[4], y[4])
