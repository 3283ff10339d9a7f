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


# Lambda0 = X^T H X and S = X^T B X: sums of 64 rows by digits, or direct sums over at most 256 rows, added over
# the ranges of rows
@pytest.mark.parametrize("kind", ["plain", "spikes", "localized", "graded"])
@pytest.mark.parametrize("p", [13, 16, 17, 23, 32, 33, 41, 48, 49, 64, 65, 97, 129])
def test_every_entry_of_the_grams(ofks, p, kind):
    s = I.lih().with_cells((8, 7, 6)).with_p(p, occ=1.0)
    m = I.make_mesh(s)
    X = block(m, p, kind)
    f = fields(ofks, s, m, X, ("HX", "BX", "Lambda0", "S"), xc=0)
    for A, got in ((f["HX"], f["Lambda0"]), (f["BX"], f["S"])):
        ref = np.triu(X.astype(Q).T @ A.astype(Q))
        ref = ref + np.triu(ref, 1).T
        bound = (256 + len(X) / 64 + 3) * 2.0 ** -53 * np.triu(np.abs(X).T @ np.abs(A))
        bound = np.maximum(bound, bound.T)
        assert np.all(np.abs(got - ref) <= 1.001 * bound + 1e-307 * 2.0 ** -40)


# an infinity gives the infinities and NaNs of the direct sum
def test_infinities_of_the_grams(ofks):
    p, j = 17, 3
    s = I.lih().with_cells((6, 4, 5)).with_p(p, occ=1.0)
    m = I.make_mesh(s)
    X = block(m, p, "plain")
    ctx = ofks.context_for(s, m, beta=10.0)
    e = np.zeros_like(X)
    # a node with the most neighbours: its row has no padding entries, whose zeros would give NaN
    x = m.xyz[m.free_ids()]
    best, count = 0, 0
    for r in np.argsort(np.linalg.norm(x - x.mean(axis=0), axis=1))[:16]:
        e[:, 0] = 0.0
        e[r, 0] = 1.0
        c = np.count_nonzero(ctx.apply("B", e)[:, 0])
        if c > count:
            best, count = r, c
    e[:, 0] = 0.0
    e[best, 0] = 1.0
    col = ctx.apply("B", e)[:, 0]
    ctx.close()
    X[:, j] = np.where(col < 0, -1.0, 1.0)        # every product with the column's infinities has one sign
    X[best, j] = np.inf
    f = fields(ofks, s, m, X, ("BX", "S"), xc=0)
    with np.errstate(invalid="ignore", over="ignore"):
        ref = np.array([[np.sum(X[:, min(a, b)] * f["BX"][:, max(a, b)]) for b in range(p)] for a in range(p)])
    assert np.isinf(ref).sum() > p // 2
    assert np.array_equal(np.isnan(f["S"]), np.isnan(ref))
    inf = np.isinf(ref)
    assert np.array_equal(f["S"][inf], ref[inf])
