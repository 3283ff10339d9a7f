"""Products and PCG of blocks whose last chunk of four columns is partly padding.

A column's product does not depend on the others, so the first p columns of an eight-column block give the
same bits at every p.  The PCG's sums may be added in another order (1e-16 of a sum of positive terms, a few
iterations): 1e-12.  In float32 a row's 65 products round to 4e-6 normwise per iteration; 5e-5 for three.
"""
import numpy as np
import pytest

from paper_2007_14228_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def run(p, precision="fp64", iters=3):
    from paper_2007_14228_gb300 import build
    build.build()
    from paper_2007_14228_gb300 import ofks
    s = I.lih().with_cells((8, 7, 9)).with_p(p, occ=1.0)
    m = I.make_mesh(s)
    X = np.ascontiguousarray(np.random.default_rng(4).standard_normal((m.n_free, 8))[:, :p])
    ctx = ofks.context_for(s, m, beta=10.0, precision=precision, pcg_iters=iters)
    out = ctx.apply("L", X), ctx.apply("B", X), ctx.precondition("pcg", X, -np.linspace(0.5, 2.0, 8)[:p])
    ctx.close()
    return out


@pytest.mark.parametrize("p", [1, 2, 3, 4, 5, 6, 7])
def test_float64_columns_do_not_depend_on_the_padding(p):
    full, part = run(8), run(p)
    for a, b in zip(full[:2], part[:2]):
        assert np.array_equal(a[:, :p], b)
    assert np.linalg.norm(full[2][:, :p] - part[2]) <= 1e-12 * np.linalg.norm(part[2])


@pytest.mark.parametrize("iters", [1, 2, 3])
@pytest.mark.parametrize("p", [5, 8])
def test_float32_direction_after_each_count_of_iterations(p, iters):
    ref, got = run(p, "fp64", iters)[2], run(p, "mixed", iters)[2]
    assert np.linalg.norm(got - ref) <= 5e-5 * np.linalg.norm(ref)
