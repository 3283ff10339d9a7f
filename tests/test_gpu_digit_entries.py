"""Every entry of the float64 gradient and Grams, however small beside its row's or column's largest.

The direct sum of p products is off by at most p 2^-53 of the sum of their magnitudes, entry by entry; the digit
forms keep that bound, and add directly where the digits alone would not (and for infinities, as before).
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


Q = np.longdouble


# The gradient of a block X grows like X^3 through beta (S - I): scaled so that its largest entry is just below
# float64's largest, entries of 2^1023 and more are finite.  Bound: float64 rounding of a sum of 16 products of
# one dominant size, 2^-45.
def test_the_largest_results_stay_finite(ofks):
    p = 16
    s = I.lih().with_cells((6, 4, 5)).with_p(p, occ=1.0)
    m = I.make_mesh(s)
    X = np.abs(np.random.default_rng(2).standard_normal((m.n_free, p)))
    ctx = ofks.context_for(s, m, beta=10.0, hartree=0, xc=0, method="plam")
    BX = ctx.apply("B", X)
    top = np.max(np.abs(BX @ (10.0 * (X.T @ BX))))
    X *= (1.7e308 / top) ** (1.0 / 3.0)
    ctx.set_orbitals(X)
    with pytest.raises(ofks.OfksError) as e:      # its norm is beyond float64
        ctx.evaluate()
    assert e.value.code == ofks.ENONFINITE
    HX, BX, G, L0, S = (ctx.get_field(k) for k in ("HX", "BX", "G", "Lambda0", "S"))
    ctx.close()
    C = 10.0 * (S - np.eye(p)) - L0
    with np.errstate(over="ignore"):
        ref = (HX.astype(Q) + BX.astype(Q) @ C.astype(Q)).astype(np.float64)
    big = np.isfinite(ref) & (np.abs(ref) >= 2.0 ** 1023)
    assert big.any()
    assert np.all(np.abs(G[big] / ref[big] - 1.0) <= 2.0 ** -45)
