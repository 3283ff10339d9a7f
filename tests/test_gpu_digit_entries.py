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


def block(m, p, kind):
    rng = np.random.default_rng(p)
    n = m.n_free
    X = rng.standard_normal((n, p))
    if kind == "spikes":              # each column one node's, nodes side by side, over a floor of 1e-14
        X *= 1e-14
        X[(7 + 5 * np.arange(p)) % n, np.arange(p)] += 1.0
    elif kind == "localized":         # decaying from centres of their own, with zeros and a tiny row
        x = m.xyz[m.free_ids()]
        for k in range(p):
            X[:, k] *= np.exp(-np.linspace(0.5, 6.0, p)[k] * np.linalg.norm(x - x[(37 * k) % n], axis=1))
        X[::7] = 0.0
        X[3] *= 1e-300
    elif kind == "graded":            # rows and columns over forty orders of magnitude, some below float64's normal range
        X *= 10.0 ** rng.uniform(-20, 20, p) * 10.0 ** rng.uniform(-3, 3, n)[:, None]
        X[11] *= 1e-306
    return X


def fields(ofks, s, m, X, names, **kw):
    ctx = ofks.context_for(s, m, beta=10.0, hartree=0, **kw)
    ctx.set_orbitals(X)
    try:
        ctx.evaluate()
    except ofks.OfksError as e:       # the record of an infinite block; its fields stand
        assert e.code == ofks.ENONFINITE
    out = {k: ctx.get_field(k) for k in names}
    ctx.close()
    return out


# G = H X + B X C: the sum, two roundings more, and C = 10 (S - I) - Lambda formed in float64
@pytest.mark.parametrize("kind", ["plain", "spikes", "localized", "graded"])
@pytest.mark.parametrize("p", [13, 16, 17, 23, 32, 33, 41, 43, 45, 48])
def test_every_entry_of_the_gradient(ofks, p, kind):
    s = I.lih().with_cells((8, 7, 6)).with_p(p, occ=1.0)
    m = I.make_mesh(s)
    X = block(m, p, kind)
    f = fields(ofks, s, m, X, ("HX", "BX", "G", "S", "Lambda"), xc=0)
    HX, BX, G = f["HX"], f["BX"], f["G"]
    C = (10.0 * (f["S"] - np.eye(p)).astype(Q) - f["Lambda"].astype(Q)).astype(np.float64)
    ref = HX.astype(Q) + BX.astype(Q) @ C.astype(Q)
    eps = 2.0 ** -53
    bound = (p + 3) * eps * (np.abs(HX) + np.abs(BX) @ np.abs(C)) \
        + 4 * eps * np.abs(BX) @ (10.0 * np.abs(f["S"] - np.eye(p)) + np.abs(f["Lambda"]))
    assert np.all(np.abs(G - ref) <= 1.001 * bound + 1e-307 * 2.0 ** -40)


# an infinity gives the infinities and NaNs of the direct sum
def test_infinities_of_the_gradient(ofks):
    p = 17
    s = I.lih().with_cells((6, 4, 5)).with_p(p, occ=1.0)
    m = I.make_mesh(s)
    X = block(m, p, "plain")
    X[5, 3] = np.inf
    f = fields(ofks, s, m, X, ("HX", "BX", "G", "S", "Lambda"), xc=0, method="moptqr")
    C = -f["Lambda"]
    with np.errstate(invalid="ignore", over="ignore"):
        # no NaN where every product is an infinity of one sign or finite
        parts = np.concatenate([f["HX"][:, None, :], f["BX"][:, :, None] * C[None, :, :]], axis=1)
        ref = parts.sum(axis=1)
    assert np.isinf(ref).any() or np.isnan(ref).any()
    assert np.array_equal(np.isnan(f["G"]), np.isnan(ref))
    inf = np.isinf(ref)
    assert np.array_equal(f["G"][inf], ref[inf])
