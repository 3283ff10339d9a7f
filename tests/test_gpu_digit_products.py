"""The float64 products formed from exact digits on the tensor cores, against extended precision.

Gradient G = H X + B X C, C = beta (S - I) - Lambda: the product is rounded once (2^-53 of its value),
the sum once (2^-53 of G), dropped digits are below 48 2^-58 of the largest entry of B X's row times the
largest of C's column, and C itself is formed in float64 on the device (2^-52 of |B X| |C|).
"""
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


def block(m, p, kind):
    rng = np.random.default_rng(p)
    X = rng.standard_normal((m.n_free, p))
    if kind == "localized":           # columns of very different size and place, exact zeros, tiny values
        d = np.linalg.norm(m.xyz[m.free_ids()], axis=1)
        X *= np.exp(-np.linspace(0.2, 30.0, p)[None, :] * d[:, None])
        X[::7] = 0.0
        X[3] *= 1e-300
    return X


@pytest.mark.parametrize("kind", ["plain", "localized"])
@pytest.mark.parametrize("p", [13, 16, 17, 31, 32, 33, 41, 45, 48, 49])
def test_gradient(ofks, p, kind):
    s = I.lih().with_cells((8, 7, 6)).with_p(p, occ=1.0)
    m = I.make_mesh(s)
    X = block(m, p, kind)
    ctx = ofks.context_for(s, m, beta=10.0)
    ctx.set_orbitals(X)
    r = ctx.evaluate()
    HX, BX, G = (ctx.get_field(k) for k in ("HX", "BX", "G"))
    L0, S, Lam = (ctx.get_field(k) for k in ("Lambda0", "S", "Lambda"))
    ctx.close()
    q = np.longdouble
    C = (10.0 * (S - np.eye(p)).astype(q) - Lam.astype(q)).astype(np.float64)   # one rounding, as a fused multiply-add
    val = BX.astype(q) @ C.astype(q)
    ref = HX.astype(q) + val
    big = np.abs(BX).max(axis=1, keepdims=True) * np.abs(C).max(axis=0, keepdims=True)
    bound = 1.01 * 2.0 ** -53 * (np.abs(val) + np.abs(ref)) + 48 * 2.0 ** -58 * big + 2.0 ** -51 * (np.abs(BX) @ np.abs(C))
    if p <= 48:                       # beyond, the gradient is a sum of p rounded products
        assert np.all(np.abs(G - ref) <= bound + 1e-290)
    kkt = np.sqrt(np.sum((HX.astype(q) - BX.astype(q) @ L0.astype(q)) ** 2))
    assert abs(r["kkt"] - kkt) <= 1e-13 * kkt + 1e-13 * np.linalg.norm(np.abs(BX) @ np.abs(L0))


def test_non_finite_rows_are_reported(ofks):
    s = I.lih().with_cells((8, 7, 6)).with_p(20, occ=1.0)
    m = I.make_mesh(s)
    for bad in (np.inf, np.nan):
        X = block(m, 20, "plain")
        X[5, 3] = bad
        ctx = ofks.context_for(s, m, beta=10.0, hartree=0)
        ctx.set_orbitals(X)
        with pytest.raises(ofks.OfksError) as e:
            ctx.evaluate()
        assert e.value.code == ofks.ENONFINITE
        ctx.close()
