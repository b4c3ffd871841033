"""Block rows with small tiles on the tensor cores (h2_tile.cu) at the edges of
their range: leaves of 2 to 32 triangles, 1 to 64 right-hand sides (every tile
width and several passes), and rows of many blocks (several exact segments).

Tolerance: the digits are rounded to 2^-50 of their scales and the digit pairs
left out stay below 2^-53 of them, so the double-float operations around them
(2^-44 = 5.7e-14 per operation) bound the error; 1e-13 against the FP64 oracle."""
import numpy as np
import pytest

import oracle
from paper_2203_05665_gb300 import H2Matrix, colmajor, inputs as I

pytestmark = pytest.mark.gpu
TOL = 1e-13


def _patch(n):
    """The first n triangles of a 1,280-triangle sphere."""
    v, f = I.icosphere(3)
    return v, np.ascontiguousarray(f[:n])


def _rel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


@pytest.mark.parametrize("leaf", [2, 7, 8, 9, 16, 17, 21, 22, 31, 32])
def test_nearfield_leaf_sizes(require_gpu, leaf):
    v, f = _patch(8 * leaf)
    o = oracle.Oracle(v, f, leaf_size=leaf, eta=2.0, order=3)
    h = H2Matrix(v, f, leaf_size=leaf, eta=2.0, order=3, prec="f64")
    assert h.stats["leaf_max"] == leaf and h.stats["tensor_near"] == 1
    for nrhs in (1, 4, 5, 8, 9, 16, 17, 24, 33, 64):
        x = I.uniform_rhs(8 * leaf, nrhs, 5000 + nrhs)
        assert _rel(h.matvec_host(x), o.matvec(x)) <= TOL, nrhs
    h.close()


@pytest.mark.parametrize("leaf", [3, 21, 32])
def test_nearfield_long_rows(require_gpu, leaf):
    """No admissible block (small eta): rows of 32 blocks, one to two exact segments of 661 // leaf blocks,
    and the rows of a mesh with ragged leaves."""
    for n in (32 * leaf, 32 * leaf - 5):
        v, f = _patch(n)
        o = oracle.Oracle(v, f, leaf_size=leaf, eta=1e-3, order=2)
        h = H2Matrix(v, f, leaf_size=leaf, eta=1e-3, order=2, prec="f64")
        assert h.stats["adm_blocks"] == 0 and h.stats["tensor_near"] == 1
        for nrhs in (3, 7, 20):
            x = I.uniform_rhs(n, nrhs, 5100 + nrhs)
            assert _rel(h.matvec_host(x), o.matvec(x)) <= TOL, (n, nrhs)
        h.close()


def _wide_columns(n, nrhs, seed):
    """Columns whose values span many orders of magnitude, in turn: one entry far above the rest, two
    opposite ones, values falling by 1e-12 over the mesh, log-normal values, and an even one."""
    r = np.random.default_rng(seed)
    x = r.uniform(-1.0, 1.0, (n, nrhs))
    for j in range(nrhs):
        kind, i = j % 5, int(r.integers(n - 1))
        if kind == 0:
            x[i, j] = 1e8
        elif kind == 1:
            x[i, j], x[i + 1, j] = 1e8, -1e8
        elif kind == 2:
            x[:, j] *= np.logspace(0, -12, n)
        elif kind == 3:
            x[:, j] = np.sign(x[:, j]) * np.exp(6 * r.standard_normal(n))
    return x


@pytest.mark.parametrize("order, leaf", [(3, 2), (3, 9), (3, 20), (3, 30), (2, 32), (4, 32)])
def test_columns_of_wide_range(require_gpu, order, leaf):
    """Digits below a column's largest value would drop the small values' bits: such columns are summed
    in double-float, on a mesh whose triangles are graded 7 : 1 in size (so that the small values weigh in
    the result); the coupling of order 3 and the nearfield of every order, beside even columns.  Order 4
    only beyond 16 columns, where its coupling is double-float too.  Two opposite neighbours cancel to the
    kernel's change over a triangle, a tenth of either or more: ten roundings of 2^-44 for those."""
    n = 128 * leaf
    v, f = I.icosphere(4)
    v, f = v * np.exp(v[:, 2:3]), np.ascontiguousarray(f[:n])
    o = oracle.Oracle(v, f, leaf_size=leaf, eta=2.0, order=order)
    h = H2Matrix(v, f, leaf_size=leaf, eta=2.0, order=order, prec="f64")
    assert h.stats["leaf_max"] == leaf and h.stats["tensor_near"] == 1
    for nrhs in (1, 5, 16, 17, 40) if order < 4 else (17, 32):
        x = _wide_columns(n, nrhs, 5500 + nrhs)
        y, ref = h.matvec_host(x), o.matvec(x)
        for c in range(nrhs):
            assert _rel(y[:, c], ref[:, c]) <= (10 * 2.0**-44 if c % 5 == 1 else TOL), (nrhs, c)
    h.close()


@pytest.mark.parametrize("order, leaf", [(3, 30), (3, 9), (2, 32)])
def test_columns_do_not_depend_on_others(require_gpu, order, leaf):
    """Columns of wide range (double-float), even ones (digits) and zero ones in one product: each gives,
    bit for bit, what it gives beside any others."""
    import torch
    n = 64 * leaf
    v, f = I.icosphere(4)
    v, f = v * np.exp(v[:, 2:3]), np.ascontiguousarray(f[:n])
    h = H2Matrix(v, f, leaf_size=leaf, eta=2.0, order=order, prec="f64")
    for nrhs in (2, 7, 16, 21):
        sets = {"even": I.uniform_rhs(n, nrhs, 5800), "zero": np.zeros((n, nrhs)),
                "wide": np.stack([_wide_columns(n, 5, 5801 + j)[:, j % 4] for j in range(nrhs)], axis=1)}
        dev = {k: torch.from_numpy(np.ascontiguousarray(x.T)).cuda().t() for k, x in sets.items()}
        ref = {}
        for k, x in dev.items():
            ref[k] = colmajor(torch.empty_like(x))
            h.matvec(x, ref[k])
        kinds = np.array(["even", "wide", "zero"])[np.random.default_rng(nrhs).integers(0, 3, nrhs)]
        x = colmajor(torch.stack([dev[k][:, c] for c, k in enumerate(kinds)], dim=1))
        y = colmajor(torch.empty_like(x))
        h.matvec(x, y)
        for c, k in enumerate(kinds):
            assert torch.equal(y[:, c], ref[k][:, c]), (nrhs, c, k)
    h.close()


def test_columns_with_infinity_or_nan(require_gpu):
    """Every output depends on every input: a column with an infinity or a NaN gives NaN throughout,
    the other columns are not touched by it."""
    import torch
    v, f = I.icosphere(3)
    n = f.shape[0]
    for order in (3, 4):
        h = H2Matrix(v, f, leaf_size=32, eta=2.0, order=order, prec="f64")
        for nrhs in (4, 20):
            x = colmajor(torch.from_numpy(I.uniform_rhs(n, nrhs, 5200)).cuda())
            y0, y1 = colmajor(torch.empty_like(x)), colmajor(torch.empty_like(x))
            h.matvec(x, y0)
            x[7, 1], x[n - 1, 3] = float("inf"), float("nan")
            h.matvec(x, y1)
            good = [c for c in range(nrhs) if c not in (1, 3)]
            assert torch.isnan(y1[:, [1, 3]]).all()
            assert torch.equal(y0[:, good], y1[:, good])
        h.close()


@pytest.mark.parametrize("nrhs", [4, 9, 16])
def test_columns_with_infinity_or_nan_f32(require_gpu, nrhs):
    """The same for FP32 handles whose coupling cuts the coefficients into digits (order 4), with either
    kind of transfer kernel (register kernels: more than 8 columns, 4,096 columns times parents)."""
    import torch
    v, f = I.icosphere(4)
    n = f.shape[0]
    h = H2Matrix(v, f, leaf_size=4, eta=2.0, order=4, prec="f32")
    assert h.stats["tensor"] == 1
    x = colmajor(torch.from_numpy(I.uniform_rhs(n, nrhs, 5200)).float().cuda())
    y0, y1 = colmajor(torch.empty_like(x)), colmajor(torch.empty_like(x))
    h.matvec(x, y0)
    x[7, 1], x[n - 1, 3] = float("inf"), float("nan")
    h.matvec(x, y1)
    good = [c for c in range(nrhs) if c not in (1, 3)]
    assert torch.isnan(y1[:, [1, 3]]).all()
    assert torch.equal(y0[:, good], y1[:, good])
    h.close()


@pytest.mark.parametrize("mesh, leaf", [("patch", 32), ("cube", 16), ("cube", 40), ("ellipsoid", 24)])
def test_order3_coupling(require_gpu, mesh, leaf):
    """The order-3 coupling: ragged leaves, leaves beyond the tensor-core nearfield (40), rows of up to
    about 140 blocks (cubes; several exact segments of 24), every tile width and several passes,
    columns of very different scales; bit-reproducible."""
    import torch
    v, f = {"patch": lambda: _patch(1111), "cube": lambda: I.cube(20),
            "ellipsoid": lambda: I.ellipsoid(3, (2.0, 1.0, 0.5))}[mesh]()
    n = f.shape[0]
    o = oracle.Oracle(v, f, leaf_size=leaf, eta=2.0, order=3)
    h = H2Matrix(v, f, leaf_size=leaf, eta=2.0, order=3, prec="f64")
    assert h.stats["tensor"] == 1 and h.stats["adm_blocks"] > 0
    # 64 columns of a leaf of 40 exceed one tile of the leaf backward step
    for nrhs in (1, 3, 4, 5, 8, 9, 16, 17, 32, 37) + ((64,) if leaf <= 32 else ()):
        x = I.uniform_rhs(n, nrhs, 5300 + nrhs) * np.logspace(-9, 6, nrhs)
        y, ref = h.matvec_host(x), o.matvec(x)
        for c in range(nrhs):
            assert _rel(y[:, c], ref[:, c]) <= TOL, (nrhs, c)
    xd = colmajor(torch.from_numpy(I.uniform_rhs(n, 20, 5400)).cuda())
    y1, y2 = colmajor(torch.empty_like(xd)), colmajor(torch.empty_like(xd))
    h.matvec(xd, y1)
    h.matvec(xd, y2)
    assert torch.equal(y1, y2)
    h.close()


@pytest.mark.parametrize("prec, tol", [("f64", 4e-13), ("f32", 1e-6)])
@pytest.mark.parametrize("leaf", [20, 32])
def test_order4_coupling_widths(require_gpu, prec, tol, leaf):
    """Digit tiles of 8 and of 16 columns (up to 8 and up to 16 right-hand sides), with the leaf forward
    step in double-float or on the tensor cores (leaves of at most 21 triangles, more than 8 columns).
    The digit pairs left out stay below 2^-46 of a row's scale (FP64) and 2^-27 (FP32); a row's scale is
    at most some 25 times its entries' typical size (1,280 triangles)."""
    v, f = I.icosphere(3)
    o = oracle.Oracle(v, f, leaf_size=leaf, eta=2.0, order=4)
    h = H2Matrix(v, f, leaf_size=leaf, eta=2.0, order=4, prec=prec)
    assert h.stats["tensor"] == 1
    for nrhs in (1, 2, 3, 4, 5, 7, 8, 9, 12, 16):
        x = I.uniform_rhs(f.shape[0], nrhs, 5400 + nrhs)
        x[:, 0] *= 1e6
        y, r = h.matvec_host(x), o.matvec(x)
        for j in range(nrhs):
            assert _rel(y[:, j], r[:, j]) <= tol, (nrhs, j)
    h.close()


def test_leaf_steps_in_column_passes(require_gpu):
    """FP64 leaf steps in passes of 16 columns (leaves of at most 32 triangles), order 2 and 3, padded
    and full last passes."""
    v, f = _patch(1000)
    for order, leaf in ((2, 32), (3, 17), (4, 32)):
        o = oracle.Oracle(v, f, leaf_size=leaf, eta=2.0, order=order)
        for prec in ("f64", "f64n"):
            h = H2Matrix(v, f, leaf_size=leaf, eta=2.0, order=order, prec=prec)
            for nrhs in (17, 31, 32) + ((33, 64) if order < 4 else ()):   # order 4 takes at most 32
                x = I.uniform_rhs(1000, nrhs, 5500 + nrhs)
                assert _rel(h.matvec_host(x), o.matvec(x)) <= (TOL if order < 4 else 4e-13), (order, prec, nrhs)
            h.close()
