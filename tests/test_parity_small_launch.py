"""Small evaluation launches (a block per warp task, three stencil columns of rows in flight) against
the block shapes of larger ones: the same sums in the same order, so the same bits."""
import numpy as np
import pytest

from paper_1309_6250_gb300 import inputs
from gpu_helpers import NONORTHO, dev

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DIMS = (10, 12, 9)


def splines(n_orb, **kw):
    from paper_1309_6250_gb300.api import OrbitalSplines
    lat, mil, coef = inputs.random_cell(3100 + n_orb, DIMS, n_orb, 5.0, 4.0, NONORTHO)
    return lat, OrbitalSplines(lat, DIMS, mil, coef, device=dev(), **kw)


def evaluate(spl, pos, n):
    out = [torch.full_like(t, float("nan")) for t in spl.alloc_outputs(n)]
    spl.eval_vgl(pos[:n], out=out)
    spl.sync()
    return [t.cpu().numpy() for t in out]


@pytest.mark.parametrize("lap", [True, False])
@pytest.mark.parametrize("storage", ["f64", "df64", "f32", "bf16"])
@pytest.mark.parametrize("n_orb", [1, 11, 128, 301])
def test_small_launch_same_bits_as_blocks(n_orb, storage, lap):
    """One position up to past the limit of small launches; set_block(512) takes the block shape."""
    lat, spl = splines(n_orb, storage=storage, separate_lap=lap)
    info = spl.info()
    per_warp = max(1, 32 // info["lanes"] // info["tiles"])
    limit = 8 * torch.cuda.get_device_properties(0).multi_processor_count * per_warp
    sizes = [1, 2, 33, min(limit, 6000), min(limit + 1, 6001)]
    pos = torch.from_numpy(inputs.positions(lat, sizes[-1], 77, -1.0, 2.0)).to(dev())
    for n in sizes:
        spl.set_block(0)
        got = evaluate(spl, pos, n)
        spl.set_block(512)
        for a, b in zip(got, evaluate(spl, pos, n)):
            np.testing.assert_array_equal(a, b)


@pytest.mark.parametrize("kw", [dict(separate_grad=True), dict(method="lagrange"), dict(method="pp"), dict(degree=5),
                                dict(separate_grad=True, storage="df64"), dict(method="lagrange", storage="f64"),
                                dict(method="pp", storage="bf16"), dict(degree=1, storage="f64")])
def test_small_launch_same_bits_as_large_call(kw):
    """The other bases: the first positions of a call too large for the small launch."""
    lat, spl = splines(40, **{"method": "interp", **kw})
    n = 8 * torch.cuda.get_device_properties(0).multi_processor_count * 32 + 1
    pos = torch.from_numpy(inputs.positions(lat, n, 78, -1.0, 2.0)).to(dev())
    spl.set_order("input")
    large = evaluate(spl, pos, n)
    for m in (1, 37):
        for a, b in zip(evaluate(spl, pos, m), large):
            np.testing.assert_array_equal(a, b[:m])
