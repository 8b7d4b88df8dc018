"""The benchmark counts the kernels of its step in a capture of the call: one without a coordinate pass,
two with one, four in cell order, whatever rule chose between them."""
import os
import sys

import numpy as np
import pytest

from paper_1309_6250_gb300 import inputs
from gpu_helpers import NONORTHO, dev

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))


@pytest.mark.parametrize("storage,n,order,kernels", [("f32", 100, "input", 1), ("f32", 9000, "input", 1),
                                                     ("f64", 9000, "input", 2), ("f32", 9000, "cell", 4)])
def test_kernel_launches(storage, n, order, kernels):
    import bench
    from paper_1309_6250_gb300.api import OrbitalSplines
    dims = (12, 12, 12)
    lat, mil, coef = inputs.random_cell(9970, dims, 16, 5.0, 4.0, NONORTHO)
    spl = OrbitalSplines(lat, dims, mil, coef, method="interp", storage=storage, device=dev())
    spl.set_order(order)
    pos = torch.from_numpy(np.ascontiguousarray(inputs.positions(lat, n, 9971))).to(dev())
    out = spl.alloc_outputs(n)
    call = lambda: spl.eval_vgl(pos, out=out)
    call()
    torch.cuda.synchronize()
    assert bench.kernel_launches(call) == kernels
    spl.close()
