"""Repeated products run from a graph kept on the handle, aimed at each call's x and y:
new buffers, changing numbers of right-hand sides (more of them than graphs are kept, and
growing work buffers), the accumulating form, host and FP64 vectors of an FP32 handle, a
GCA handle, and a product inside the caller's own capture.  Every result must equal, bit
for bit, that of a fresh handle's first call, which is launched kernel by kernel."""
import numpy as np
import pytest

from paper_2203_05665_gb300 import GcaMatrix, H2Matrix, colmajor, inputs as I

pytestmark = pytest.mark.gpu


def _mat(kind, stream=None):
    v, f = I.icosphere(2)
    if kind == "gca":
        return GcaMatrix(v, f, leaf_size=16, eta=2.0, prec="f64", stream=stream)
    return H2Matrix(v, f, leaf_size=16, eta=2.0, order=4 if kind == "f64" else 3, prec=kind, stream=stream)


def _x(n, nrhs, seed, dt):
    import torch
    return colmajor(torch.from_numpy(I.uniform_rhs(n, nrhs, seed)).to(device="cuda", dtype=dt))


@pytest.mark.parametrize("kind", ["f64", "f64n", "f32", "bf16", "f16", "gca"])
def test_repeated_products(require_gpu, kind):
    import torch
    dt = torch.float64 if kind in ("f64", "f64n", "gca") else torch.float32
    h = _mat(kind)
    for step, nrhs in enumerate([1, 1, 1, 3, 3, 2, 3, 5, 5, 7, 7, 9, 9, 1, 1, 3, 3, 9]):
        x = _x(h.n, nrhs, 7000 + step, dt)
        y = colmajor(torch.zeros_like(x))
        h.matvec(x, y)
        ref, first = colmajor(torch.empty_like(x)), _mat(kind)
        first.matvec(x, ref)
        assert torch.equal(y, ref), (step, nrhs)
        h.matvec_acc(x, y)
        first.matvec_acc(x, ref)
        assert torch.equal(y, ref), (step, nrhs)
        first.close()
    if kind == "f32":
        for step in range(3):
            x = I.uniform_rhs(h.n, 3, 7100 + step)
            first = _mat(kind)
            assert np.array_equal(h.matvec_host(x), first.matvec_host(x))
            first.close()
    h.close()


def test_product_in_a_capture(require_gpu):
    """The caller captures the product on the handle's stream: it goes into that capture."""
    import torch
    s = torch.cuda.Stream()
    h = _mat("f64", stream=s.cuda_stream)
    x = _x(h.n, 4, 7200, torch.float64)
    y, ref = colmajor(torch.empty_like(x)), colmajor(torch.empty_like(x))
    torch.cuda.synchronize()
    for _ in range(3):
        h.matvec(x, ref)
    s.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        h.matvec(x, y)
    x.copy_(2.0 * x)
    torch.cuda.synchronize()
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(y, 2.0 * ref)
    del g
    h.close()


@pytest.mark.parametrize("where", ["thread", "other thread"])
def test_products_beside_a_capture(require_gpu, where):
    """Products on the handle's own stream while another stream is being captured in the global mode (by
    this thread, or by another): neither disturbs the other, also where the product makes a graph (the
    second with its number of right-hand sides) or drops one (the sixth number of them)."""
    import threading
    import torch
    s, other = torch.cuda.Stream(), torch.cuda.Stream()
    h = _mat("f64", stream=s.cuda_stream)
    xs = {nrhs: _x(h.n, nrhs, 7300 + nrhs, torch.float64) for nrhs in (5, 1, 2, 3, 4, 6)}
    ref = {nrhs: colmajor(torch.empty_like(x)) for nrhs, x in xs.items()}
    ys = {nrhs: [colmajor(torch.empty_like(x)) for _ in range(3)] for nrhs, x in xs.items()}
    z = torch.zeros(8, device="cuda")
    torch.cuda.synchronize()
    h.matvec(xs[6], ref[6])   # the work buffers exist
    for nrhs, x in xs.items():
        first = _mat("f64")
        first.matvec(x, ref[nrhs])
        first.close()
    torch.cuda.synchronize()
    errors = []

    def products():
        try:
            for nrhs, x in xs.items():
                for y in ys[nrhs]:
                    h.matvec(x, y)
        except Exception as e:   # raised by the test's own thread below
            errors.append(e)

    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=other):
        z.add_(1)
        if where == "thread":
            products()
        else:
            t = threading.Thread(target=products)
            t.start()
            t.join()
        z.add_(1)
    assert not errors, errors
    g.replay()
    torch.cuda.synchronize()
    assert z[0].item() == 2
    for nrhs in xs:
        assert all(torch.equal(y, ref[nrhs]) for y in ys[nrhs]), nrhs
    del g
    h.close()
