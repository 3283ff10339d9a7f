"""Blocks of more than 64 float32 columns against the float64 form: the warp-per-row products.

Widths at the edges of the kernel's 128- and 256-column pieces and of the padding to four columns.
Tolerance: H's values and the blocks are rounded to float32 (6e-8 each) and a row sums about 65
products, so a normwise error of a few 1e-7; 5e-6 leaves room for cancellation in H X.
"""
import numpy as np
import pytest

from paper_2007_14228_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("p", [65, 68, 127, 129, 133, 210, 255, 256])
def test_products_and_normalization(p):
    from paper_2007_14228_gb300 import build
    build.build()
    from paper_2007_14228_gb300 import ofks
    s = I.lih().with_cells((8, 7, 9)).with_p(p, occ=1.0)
    m = I.make_mesh(s)
    X = I.initial_block(m.n_free, p, 3)
    fields = {}
    for precision in ("fp64", "mixed"):
        ctx = ofks.context_for(s, m, beta=10.0, precision=precision)
        ctx.init_orbitals(X)
        ctx.evaluate()
        fields[precision] = {k: ctx.get_field(k) for k in ("HX", "Lambda0", "S")}
        ctx.step(1)
        X1 = ctx.get_orbitals()
        norms = np.einsum("ij,ij->j", X1, ctx.apply("B", X1))
        assert np.max(np.abs(norms - 1.0)) < 2e-5     # Eq. (PCAL-main), float32 sums
        ctx.close()
    for k, ref in fields["fp64"].items():
        assert np.linalg.norm(fields["mixed"][k] - ref) <= 5e-6 * np.linalg.norm(ref), k
