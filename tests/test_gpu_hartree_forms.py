"""The forms of the separable Hartree CG against its CUDA-core form, at the edges of their tiles.

The CG runs as one persistent kernel, as three kernels per application or as six, by the interior
extents (2 cells - 1 per axis): rows of 16 (15, 17), 128-row tiles (127, 129), axes too long for one
form or the other.  Every form solves the same system, so the potentials agree within the tolerance.

Tolerances: two solves to a 1e-12 relative residual agree within 1e-9 of the potential's norm (the
bound of the parity tests); in the float32 phase the density is float32 (1e-6) and the operator's
values carry 48 bits (3.6e-15 times a condition number near 1e7), so 5e-6.
"""
import numpy as np
import pytest

from paper_2007_14228_gb300 import inputs as I

pytestmark = pytest.mark.gpu

CELLS = [(6, 4, 4), (8, 8, 8), (9, 8, 10), (24, 24, 24), (64, 6, 5), (65, 9, 7), (7, 64, 6), (6, 5, 65), (6, 64, 65),
         (100, 5, 6), (6, 70, 72), (6, 96, 97), (80, 40, 41)]


@pytest.fixture(scope="module")
def ofks():
    from paper_2007_14228_gb300 import build
    build.build()
    from paper_2007_14228_gb300 import ofks as mod
    return mod


def potential(ofks, s, m, X, **kw):
    ctx = ofks.context_for(s, m, beta=10.0, **kw)
    out = []
    for scale in (1.0, 0.9):                      # a cold start and a warm one
        ctx.set_orbitals(X * scale)
        r = ctx.evaluate()
        out.append(ctx.get_field("U"))
    ctx.close()
    return out, r["hartree_iters"]


@pytest.mark.parametrize("cells", CELLS, ids=lambda c: "x".join(map(str, c)))
def test_forms_agree(ofks, cells):
    s = I.lih().with_cells(cells)
    m = I.make_mesh(s)
    x = m.xyz[m.free_ids()]
    d = np.linalg.norm(x, axis=1)
    X = np.stack([np.exp(-2.0 * d), x[:, 0] * np.exp(-0.7 * d)], axis=1)
    X /= np.sqrt(np.mean(X * X, axis=0))
    ref, _ = potential(ofks, s, m, X, poisson_sep_tc=0)
    got, its = potential(ofks, s, m, X)
    assert 0 < its < 60
    for g, r in zip(got, ref):
        assert np.linalg.norm(g - r) <= 1e-9 * np.linalg.norm(r)
    got, _ = potential(ofks, s, m, X, precision="mixed", poisson_tol_mixed=1e-12)
    for g, r in zip(got, ref):
        assert np.linalg.norm(g - r) <= 5e-6 * np.linalg.norm(r)


def test_iteration_limit_and_recovery(ofks):
    s = I.lih().with_cells((8, 8, 8))
    m = I.make_mesh(s)
    X = I.initial_block(m.n_free, s.p, 0)
    ctx = ofks.context_for(s, m, beta=10.0, poisson_max_iter=1)
    ctx.set_orbitals(X)
    with pytest.raises(ofks.OfksError) as e:
        ctx.evaluate()
    assert e.value.code == ofks.ETIMEOUT
    X2 = X.copy()
    X2[0, 0] = np.inf
    ctx.set_params(poisson_max_iter=100)
    ctx.set_orbitals(X2)
    with pytest.raises(ofks.OfksError) as e:
        ctx.evaluate()
    assert e.value.code == ofks.ENONFINITE
    ctx.close()
