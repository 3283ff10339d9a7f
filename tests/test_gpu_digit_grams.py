"""The float64 Grams formed from exact digits on the tensor cores, against extended precision.

Lambda0 = X^T H X, S = X^T B X.  Entries of a column smaller than 2^-9 of its largest among 64 rows lose
up to 2^-62 of that largest, and what the dropped digit products add is below 7.1 2^-60 of the product of
the two largest magnitudes, in each of 64 rows; each sum of 64 rows is rounded once, and these sums are
added in float64, 2^-53 of the sum of magnitudes each time.
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


def largest(M):                       # largest magnitude of each column among 64 rows, summed over the steps
    return np.array([np.abs(M[r:r + 64]).max(axis=0) for r in range(0, len(M), 64)])


@pytest.mark.parametrize("kind", ["plain", "localized"])
@pytest.mark.parametrize("p", [13, 16, 17, 31, 32, 33, 41, 48, 49, 64, 65, 97, 129])
def test_grams(ofks, p, kind):
    s = I.lih().with_cells((6, 6, 7) if p % 2 else (6, 4, 5)).with_p(p, occ=1.0)
    m = I.make_mesh(s)
    X = block(m, p, kind)
    ctx = ofks.context_for(s, m, beta=10.0)
    ctx.set_orbitals(X)
    ctx.evaluate()
    fields = {k: ctx.get_field(k) for k in ("HX", "BX", "Lambda0", "S")}
    ctx.close()
    q = np.longdouble
    for prod, gram in (("HX", "Lambda0"), ("BX", "S")):
        A, got = fields[prod], fields[gram]
        ref = np.triu(X.astype(q).T @ A.astype(q))
        ref = ref + np.triu(ref, 1).T
        mag = np.abs(X).T @ np.abs(A)
        big = 64 * largest(X).T @ largest(A)
        bound = (len(X) / 64 + 2) * 2.0 ** -53 * mag + 2.0 ** -57 * big
        bound = np.maximum(np.triu(bound), np.triu(bound).T)
        assert np.all(np.abs(got - ref) <= bound + 1e-290)
