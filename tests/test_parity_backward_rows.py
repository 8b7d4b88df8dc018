"""The adjoint's upstream reads (16-byte chunks, or value by value where rows are no whole chunks or lie off
a 16-byte boundary) and the gathered coefficient adjoint's batches (bins of many positions)."""
import numpy as np
import pytest

from paper_1309_6250_gb300 import inputs
from gpu_helpers import NONORTHO, dev

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DIMS = (12, 9, 10)


def splines(n_orb, **kw):
    from paper_1309_6250_gb300.api import OrbitalSplines
    lat, mil, coef = inputs.random_cell(4200 + n_orb, DIMS, n_orb, 5.0, 4.0, NONORTHO)
    return lat, OrbitalSplines(lat, DIMS, mil, coef, device=dev(), **kw)


def adjoint(spl, pos, up, want_dpos=True):
    dc = [torch.zeros(spl.coef_shape(), dtype=spl.out_dtype, device=dev()) for _ in range(2)]
    dpos = spl.backward(pos, *up, *dc, want_dpos=want_dpos)
    spl.sync()
    return [dpos] + dc


@pytest.mark.parametrize("storage", ["f32", "bf16", "f64"])
@pytest.mark.parametrize("n_orb", [8, 13, 128])
@pytest.mark.parametrize("n,order", [(300, "input"), (2000, "cell")])
def test_upstream_off_a_chunk_boundary(n, order, n_orb, storage):
    """Upstream buffers shifted by one value give what aligned ones give (up to the order of atomics)."""
    lat, spl = splines(n_orb, storage=storage)
    spl.set_order(order)
    pos = torch.from_numpy(inputs.positions(lat, n, 79, -1.0, 2.0)).to(dev())
    g = torch.Generator(device=dev()).manual_seed(3)
    shapes = ((n, n_orb), (n, 3, n_orb), (n, n_orb))
    up = [torch.randn(s, generator=g, dtype=spl.out_dtype, device=dev()) for s in shapes]
    moved = []
    for t in up:
        flat = torch.empty(t.numel() + 1, dtype=t.dtype, device=dev())
        flat[1:] = t.reshape(-1)
        moved.append(flat[1:].view(t.shape))
    tol = 1e-13 if storage == "f64" else 2e-6   # sums of up to n values in another order
    for a, b in zip(adjoint(spl, pos, up), adjoint(spl, pos, moved)):
        assert float((a - b).abs().max()) <= tol * float(b.abs().max())


@pytest.mark.parametrize("storage", ["f32", "f64"])
@pytest.mark.parametrize("count", [39, 40, 41, 64, 65, 500])
def test_gathered_adjoint_of_crowded_bins(count, storage):
    """All positions in one bin of cells (one to several staged batches), against input order's scatter."""
    lat, spl = splines(20, storage=storage)
    frac = np.random.default_rng(count).uniform(0.01, 0.3, size=(count, 3))
    pos = torch.from_numpy(np.ascontiguousarray(frac @ lat.T)).to(dev())
    up = [torch.from_numpy(x).to(dev(), spl.out_dtype) for x in inputs.upstream_weights(count, 20, 5)]
    spl.set_order("cell")
    got = adjoint(spl, pos, up)
    spl.set_order("input")
    ref = adjoint(spl, pos, up)
    tol = 1e-12 if storage == "f64" else 5e-6   # sums of up to 500 x 64 single-precision products
    for a, b in zip(got, ref):
        assert float((a - b).abs().max()) <= tol * float(b.abs().max())
