"""The gathered coefficient adjoint's two block shapes (chosen by the number of bins against the number of
SMs: 216 bins of 4^3 cells take the small one on 152 SMs, 343 the wide one), against input order's scatter,
with every position in one bin (one to several staged batches) and spread over all of them."""
import numpy as np
import pytest

from paper_1309_6250_gb300 import inputs
from gpu_helpers import NONORTHO, dev

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("storage", ["f32", "bf16"])
@pytest.mark.parametrize("grid", [24, 28])
@pytest.mark.parametrize("count,crowded", [(1, True), (39, True), (40, True), (41, True), (64, True), (65, True),
                                           (500, True), (6000, False)])
def test_gather_shapes_match_the_scatter(count, crowded, grid, storage):
    from paper_1309_6250_gb300.api import OrbitalSplines
    dims, n_orb = (grid,) * 3, 20
    lat, mil, coef = inputs.random_cell(4700 + grid, dims, n_orb, 5.0, 4.0, NONORTHO)
    spl = OrbitalSplines(lat, dims, mil, coef, device=dev(), storage=storage)
    frac = np.random.default_rng(count).uniform(0.01, 0.13 if crowded else 1.99, size=(count, 3))
    pos = torch.from_numpy(np.ascontiguousarray(frac @ lat.T)).to(dev())
    up = [torch.from_numpy(x).to(dev(), spl.out_dtype) for x in inputs.upstream_weights(count, n_orb, 5)]

    def adjoint(order):
        spl.set_order(order)
        dc = [torch.zeros(spl.coef_shape(), dtype=spl.out_dtype, device=dev()) for _ in range(2)]
        dpos = spl.backward(pos, *up, *dc)
        spl.sync()
        return [dpos] + dc

    # sums of up to 500 x 64 single-precision products in another order
    for a, b in zip(adjoint("cell"), adjoint("input")):
        assert float((a - b).abs().max()) <= 5e-6 * float(b.abs().max())
    spl.close()
