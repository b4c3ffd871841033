"""Block rows in FP32 arithmetic (h2_lane.cu) at the edges of their range: tiles of
2 to 64 rows (half-warp split, one and two rows per lane, pieces of a block), 1 to 64
right-hand sides (every column width, two passes), rows long enough for four warps,
and the mixed terms of a row (leaf basis, FP32 self block, 16-bit blocks).

Tolerances: every stored entry is rounded once (FP32 2^-24, half 2^-11, bfloat16 2^-8
but FP32 on the diagonal blocks) and a row sums a few thousand products in FP32: 1e-6
and 2e-3 against the FP64 oracle, the bounds of the parity tests."""
import numpy as np
import pytest

import oracle
from paper_2203_05665_gb300 import H2Matrix, inputs as I

pytestmark = pytest.mark.gpu
TOL = {"f32": 1e-6, "bf16": 2e-3, "f16": 2e-3}


def _rel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


@pytest.mark.parametrize("prec, basis", [("f32", None), ("bf16", None), ("f16", None), ("f16", "f32")])
@pytest.mark.parametrize("leaf, order", [(2, 2), (15, 3), (16, 3), (17, 4), (32, 3), (33, 4), (64, 3)])
def test_leaf_sizes_and_columns(require_gpu, prec, basis, leaf, order):
    v, f = I.icosphere(3)
    f = np.ascontiguousarray(f[:16 * leaf])
    o = oracle.Oracle(v, f, leaf_size=leaf, eta=2.0, order=order)
    h = H2Matrix(v, f, leaf_size=leaf, eta=2.0, order=order, prec=prec, basis=basis)
    assert h.stats["leaf_max"] == leaf
    for nrhs in (1, 4, 5, 8, 12, 16, 17, 32, 33, 64):
        x = I.uniform_rhs(f.shape[0], nrhs, 6000 + nrhs)
        assert _rel(h.matvec_host(x), o.matvec(x)) <= TOL[prec], nrhs
    h.close()


@pytest.mark.parametrize("prec", ["f32", "bf16", "f16"])
@pytest.mark.parametrize("leaf, n", [(8, 640), (12, 1270)])
def test_long_rows(require_gpu, prec, leaf, n):
    """Small eta, no admissible block: rows of 80 to 128 blocks, taken by four warps each."""
    v, f = I.icosphere(3)
    f = np.ascontiguousarray(f[:n])
    o = oracle.Oracle(v, f, leaf_size=leaf, eta=1e-3, order=2)
    h = H2Matrix(v, f, leaf_size=leaf, eta=1e-3, order=2, prec=prec)
    assert h.stats["adm_blocks"] == 0
    for nrhs in (1, 7, 20, 40):
        x = I.uniform_rhs(n, nrhs, 6100 + nrhs)
        assert _rel(h.matvec_host(x), o.matvec(x)) <= TOL[prec], nrhs
    h.close()
