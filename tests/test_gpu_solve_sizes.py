"""GMRES at the limits of its one-launch Arnoldi step (k_arnoldi: up to 32,768 rows and 9
columns, the separate kernels beyond; restarts of at most 200): on both sides of every
limit, with row counts that 16 CTAs do not share evenly and with more than 128 basis
vectors, the true residual b - G~ z in FP64 reaches the tolerance (1.5 times it: the
recursive and the true residual differ by the product's rounding), and both kinds of step
take the same number of iterations, give or take one."""
import numpy as np
import pytest

import oracle
from paper_2203_05665_gb300 import H2Matrix, inputs as I

pytestmark = pytest.mark.gpu


def _residual(h, b, z):
    r = b - h.matvec_host(z)
    return np.linalg.norm(r, axis=0) / np.linalg.norm(b, axis=0)


@pytest.mark.parametrize("n", [32752, 32767, 32768, 32769])
def test_rows(require_gpu, n):
    v, f = I.cube(53)
    f = np.ascontiguousarray(f[:n])
    h = H2Matrix(v, f, leaf_size=32, eta=2.0, order=3, prec="f64")
    b = I.uniform_rhs(n, 2, 8000)
    z, it, rel, st = h.solve(b, rtol=1e-6, restart=50, maxit=2000)
    assert st == 0 and np.all(_residual(h, b, z) <= 1.5e-6)
    if n == 32768:
        # the separate kernels: more columns than the one launch takes
        more = np.asfortranarray(np.concatenate([b] + [I.uniform_rhs(n, 2, 8001 + i) for i in range(4)], axis=1))
        z2, it2, _, st2 = h.solve(more, rtol=1e-6, restart=50, maxit=2000)
        assert st2 == 0 and np.all(np.abs(it2[:2] - it) <= 1), (it, it2)
    h.close()


def test_columns(require_gpu):
    v, f = I.ellipsoid(3, (1.5, 1.0, 0.7))
    n = 1279
    f = np.ascontiguousarray(f[:n])
    o = oracle.Oracle(v, f, leaf_size=32, eta=2.0, order=3)
    h = H2Matrix(v, f, leaf_size=32, eta=2.0, order=3, prec="f64")
    b = I.uniform_rhs(n, 10, 8100)
    its = {}
    for nrhs in (1, 8, 9, 10):
        z, it, rel, st = h.solve(b[:, :nrhs], rtol=1e-9, restart=30, maxit=2000)
        r = b[:, :nrhs] - o.matvec(z)
        assert st == 0 and np.all(np.linalg.norm(r, axis=0) <= 1.5e-9 * np.linalg.norm(b[:, :nrhs], axis=0)), nrhs
        its[nrhs] = it
    for nrhs in (1, 8, 9):
        assert np.all(np.abs(its[nrhs] - its[10][:nrhs]) <= 1), its
    h.close()


@pytest.mark.parametrize("restart", [129, 200])
def test_long_bases(require_gpu, restart):
    """A graded mesh, on which a solve takes about 157 iterations without a restart."""
    v, f = I.icosphere(4)
    v = v * np.exp(0.5 * v[:, 2:3])
    n = f.shape[0]
    h = H2Matrix(v, f, leaf_size=32, eta=2.0, order=3, prec="f64")
    b = I.uniform_rhs(n, 10, 8200)
    its = {}
    for nrhs in (3, 10):
        z, it, rel, st = h.solve(b[:, :nrhs], rtol=1e-9, restart=restart, maxit=1000)
        assert st == 0 and np.all(it > 129), it
        assert np.all(_residual(h, b[:, :nrhs], z) <= 1.5e-9)
        its[nrhs] = it
    assert np.all(np.abs(its[3] - its[10][:3]) <= 1), its
    h.close()
