"""Products of more columns than one block-row tile takes run in groups of columns (order 5
from 17, order 4 and leaves of 64 triangles from 33 columns in FP64): on every route, each
group's results are those of a product of these columns alone, bit for bit, and agree with
the FP64 oracle.  Tolerance: double-float, 2^-44 = 5.7e-14 per operation; order 5 sums 125
terms of both signs (the Lagrange polynomials' absolute sum per direction is 2, so 8 for a
coefficient), 1e-12."""
import numpy as np
import pytest

import oracle
from paper_2203_05665_gb300 import H2Matrix, HelmholtzMatrix, colmajor, inputs as I
from paper_2203_05665_gb300._lib import H2Error

pytestmark = pytest.mark.gpu


def _rel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


@pytest.mark.parametrize("prec, order, leaf, nrhs, most", [
    ("f64", 5, 32, 16, 16), ("f64", 5, 32, 17, 16), ("f64", 5, 32, 32, 16), ("f64", 5, 64, 23, 16),
    ("f64n", 5, 32, 31, 16), ("f64", 4, 32, 33, 32), ("f64", 4, 32, 64, 32), ("f64", 3, 40, 64, 50),
    ("f64", 2, 64, 64, 32), ("f64n", 3, 64, 50, 32), ("f32", 5, 32, 32, 64)])
def test_groups_of_columns(require_gpu, prec, order, leaf, nrhs, most):
    import torch
    v, f = I.icosphere(3)
    f = np.ascontiguousarray(f[:16 * leaf]) if leaf > 32 else f
    n = f.shape[0]
    o = oracle.Oracle(v, f, leaf_size=leaf, eta=2.0, order=order)
    h = H2Matrix(v, f, leaf_size=leaf, eta=2.0, order=order, prec=prec)
    dt = torch.float32 if prec == "f32" else torch.float64
    x = I.uniform_rhs(n, nrhs, 5600 + nrhs)
    xd = colmajor(torch.from_numpy(x).to(dt).cuda())
    ref = o.matvec(x)
    # products, graphs kept for repeated ones, the accumulating form, a captured graph, no allocation
    ys = [colmajor(torch.zeros_like(xd)) for _ in range(5)]
    for y in ys[:3]:
        h.matvec(xd, y)
    h.matvec_acc(xd, ys[3])
    h.matvec_noalloc(xd, ys[4])
    y, tol = ys[0].double().cpu().numpy(), 1e-12 if prec != "f32" else 1e-5
    for c in range(nrhs):
        assert _rel(y[:, c], ref[:, c]) <= tol, c
    assert all(torch.equal(ys[0], z) for z in ys[1:])
    assert _rel(h.matvec_host(x), ref) <= tol
    g = h.graph(xd, ys[1])
    ys[1].zero_()
    g.launch()
    torch.cuda.synchronize()
    assert torch.equal(ys[0], ys[1])
    g.close()
    passes = -(-nrhs // most)
    if passes > 1:
        width = -(-(-(-nrhs // passes)) // 2) * 2
        for c0 in range(0, nrhs, width):
            part = colmajor(xd[:, c0:c0 + width].clone())
            one = colmajor(torch.empty_like(part))
            h.matvec(part, one)
            assert torch.equal(ys[0][:, c0:c0 + width], one), c0
        h.matvec(xd, ys[2])
        with pytest.raises(H2Error):
            h.coefficients(0, nrhs)
        h.profile(True)
        h.matvec(xd, ys[2])
        assert h.phase_times()[1] == 1
        h.profile(False)
    h.close()


@pytest.mark.parametrize("nrhs", [8, 9, 16])
def test_groups_of_complex_columns(require_gpu, nrhs):
    """Helmholtz products run 2 nrhs real columns."""
    import torch
    v, f = I.icosphere(3)
    n = f.shape[0]
    o = oracle.HelmholtzOracle(v, f, kappa=1.5, leaf_size=32, eta=2.0, order=5)
    h = HelmholtzMatrix(v, f, 1.5, leaf_size=32, eta=2.0, order=5, prec="f64")
    x = I.uniform_rhs(n, nrhs, 5700) + 1j * I.uniform_rhs(n, nrhs, 5701)
    xd = torch.from_numpy(np.ascontiguousarray(x.T)).cuda().t()
    y = torch.empty_like(xd.t()).t()
    h.matvec(xd, y)
    assert _rel(y.cpu().numpy(), o.matvec(x)) <= 1e-12
    h.close()
