"""Coupling regenerated in the product (k_coupling_regen) at every order and every width of
its passes (4, 8, 12 and 16 columns, and several passes), against the FP64 oracle:
FP32 arithmetic, as the stored coupling's 1e-6 of the other tests; order 5 sums 125 terms
with an absolute sum of the Lagrange polynomials of 2 per direction: 4e-6."""
import numpy as np
import pytest

import oracle
from paper_2203_05665_gb300 import H2Matrix, inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("order", [1, 2, 3, 4, 5])
def test_widths(require_gpu, order):
    v, f = I.ellipsoid(3, (1.5, 1.0, 0.7))
    n = f.shape[0]
    o = oracle.Oracle(v, f, leaf_size=16, eta=2.0, order=order)
    h = H2Matrix(v, f, leaf_size=16, eta=2.0, order=order, prec="f32", coupling="regen")
    assert h.stats["coupling"] == 2 and h.stats["adm_blocks"] > 0
    for nrhs in (1, 4, 5, 8, 12, 16, 17, 32):
        x = I.uniform_rhs(n, nrhs, 8300 + nrhs)
        y, ref = h.matvec_host(x), o.matvec(x)
        for c in range(nrhs):
            e = np.linalg.norm(y[:, c] - ref[:, c]) / np.linalg.norm(ref[:, c])
            assert e <= (4e-6 if order == 5 else 1e-6), (nrhs, c, e)
    h.close()
