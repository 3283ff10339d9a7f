"""The persistent Hartree CG: what a solve depends on, where it stops, and what follows a failure."""
import re

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


def lih(cells):
    s = I.lih().with_cells(cells)
    m = I.make_mesh(s)
    return s, m, I.initial_block(m.n_free, s.p, 0)


# few iterations to many: the residual is tested after every one of them, whatever came before
@pytest.mark.parametrize("tol", [1e-3, 1e-5, 1e-8, 1e-12])
@pytest.mark.parametrize("cells", [(8, 8, 8), (16, 15, 17)], ids=str)
def test_a_solve_depends_on_its_start_and_tolerance_alone(ofks, cells, tol, tmp_path):
    s, m, V = lih(cells)
    path = str(tmp_path / "state")

    def potential(ctx):
        r = ctx.evaluate()
        return r["hartree_iters"], ctx.get_field("U")

    ctx = ofks.context_for(s, m, beta=10.0, poisson_tol=tol)
    ctx.init_orbitals(V)
    ctx.step(3)
    ctx.save_state(path)
    its, U = potential(ctx)                       # the run goes on
    for earlier in ((), (1e-12,), (1e-2, 1e-6)):  # a new context, after no solve and after others
        other = ofks.context_for(s, m, beta=10.0, poisson_tol=tol)
        other.init_orbitals(V)
        for k, t in enumerate(earlier):
            other.set_params(poisson_tol=t)
            other.set_orbitals(V * (1.0 + k))
            other.evaluate()
        other.set_params(poisson_tol=tol)
        other.load_state(path)
        its2, U2 = potential(other)
        assert its2 == its and np.array_equal(U, U2)
        other.close()
    ctx.close()


@pytest.mark.parametrize("limit", [1, 2, 3, 5])
def test_the_iteration_limit_is_kept(ofks, limit):
    s, m, V = lih((8, 8, 8))
    ctx = ofks.context_for(s, m, beta=10.0, poisson_max_iter=limit)
    ctx.init_orbitals(V)
    with pytest.raises(ofks.OfksError) as e:
        ctx.evaluate()
    assert e.value.code == ofks.ETIMEOUT
    assert int(re.search(r"Hartree CG: (\d+) iterations", str(e.value)).group(1)) == limit
    ctx.close()
