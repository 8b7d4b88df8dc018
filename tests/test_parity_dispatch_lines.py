"""Both sides of the lines that choose a kernel shape: small evaluation launches (eight warp tasks per SM),
FP64 launches with one orbital per lane (four), and the gathered adjoint's block shape by positions per bin."""
import numpy as np
import pytest

from paper_1309_6250_gb300 import inputs
from gpu_helpers import NONORTHO, dev

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DIMS = (9, 8, 7)


def positions_for(tasks, lanes, tiles):
    """The most positions that make at most `tasks` warp tasks of 32 // lanes (position, tile) groups."""
    return tasks * (32 // lanes) // tiles


@pytest.mark.parametrize("lap", [True, False])
@pytest.mark.parametrize("storage", ["f64", "df64", "f32", "bf16"])
@pytest.mark.parametrize("n_orb", [1, 11, 24, 128, 130])
def test_small_launch_limits(n_orb, storage, lap):
    """The automatic shape up to and beyond each limit, a partly filled last warp among them, gives the bits of the
    block shape (set_block 512)."""
    from paper_1309_6250_gb300.api import OrbitalSplines
    lat, mil, coef = inputs.random_cell(3300 + n_orb, DIMS, n_orb, 5.0, 4.0, NONORTHO)
    spl = OrbitalSplines(lat, DIMS, mil, coef, storage=storage, separate_lap=lap, device=dev())
    spl.set_order("input")
    lanes, tiles = spl.info()["lanes"], spl.info()["tiles"]
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    edges = {positions_for(8 * sms, lanes, tiles)}
    if storage == "f64":                   # twice the lanes, or twice the tiles where 32 lanes are taken
        wide = (2 * lanes, tiles) if lanes < 32 else (32, 2 * tiles)
        edges.add(positions_for(4 * sms, *wide))
    sizes = sorted({max(1, n + d) for n in edges for d in (-1, 0, 1, 2)})
    pos = torch.from_numpy(inputs.positions(lat, sizes[-1], 77, -1.0, 2.0)).to(dev())

    def evaluate(n):
        out = [torch.full_like(t, float("nan")) for t in spl.alloc_outputs(n)]
        spl.eval_vgl(pos[:n], out=out)
        spl.sync()
        return out

    for n in sizes:
        spl.set_block(0)
        got = evaluate(n)
        spl.set_block(512)
        for a, b in zip(got, evaluate(n)):
            assert torch.equal(a, b)
    spl.close()


@pytest.mark.parametrize("storage", ["f32", "bf16"])
@pytest.mark.parametrize("per_bin", [35, 36])
def test_gathered_adjoint_by_positions_per_bin(per_bin, storage):
    """24^3 cells: 216 bins, whose schedule takes small blocks up to 35 positions per bin and wide ones above;
    against input order's scatter."""
    from paper_1309_6250_gb300.api import OrbitalSplines
    dims, n_orb = (24, 24, 24), 20
    lat, mil, coef = inputs.random_cell(4800, dims, n_orb, 5.0, 4.0, NONORTHO)
    spl = OrbitalSplines(lat, dims, mil, coef, device=dev(), storage=storage)
    n = 216 * per_bin
    pos = torch.from_numpy(inputs.positions(lat, n, 81, 0.0, 1.0)).to(dev())
    up = [torch.from_numpy(x).to(dev(), spl.out_dtype) for x in inputs.upstream_weights(n, n_orb, 5)]

    def adjoint(order):
        spl.set_order(order)
        dc = [torch.zeros(spl.coef_shape(), dtype=spl.out_dtype, device=dev()) for _ in range(2)]
        dpos = spl.backward(pos, *up, *dc)
        spl.sync()
        return [dpos] + dc

    # sums of some 35 x 64 single-precision products in another order
    for a, b in zip(adjoint("cell"), adjoint("input")):
        assert float((a - b).abs().max()) <= 5e-6 * float(b.abs().max())
    spl.close()
