"""Input-order evaluation around the size from which coordinates come from a pass of their own: below it
the kernels divide the conversions among the lanes, above it they read records.  Positions repeat, so
that every copy must give the bits of the small call, which is checked against the oracle."""
import numpy as np
import pytest

import oracle
from gpu_helpers import TOL, assert_parity, dev
from paper_1309_6250_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("storage,sep", [("f32", True), ("f32", False), ("bf16", True), ("bf16", False)])
@pytest.mark.parametrize("orb", [3, 7, 16, 30, 64, 128])
def test_records_threshold_gives_the_same_bits(storage, sep, orb):
    from paper_1309_6250_gb300.api import OrbitalSplines
    dims = (9, 8, 10)
    lat, mil, coef = inputs.random_cell(5200 + orb, dims, orb, 6.0, 5.0, np.eye(3) * 6.0)
    spl = OrbitalSplines(lat, dims, mil, coef, method="smooth", storage=storage, separate_lap=sep, device=dev())
    spl.set_order("input")
    info = spl.info()
    base = inputs.positions(lat, 509, 5300, -1.0, 2.0)
    few = [x.cpu().numpy() for x in spl.eval_vgl(torch.from_numpy(base).to(dev()))]
    beta, blap = oracle.smoothing_tables(lat, mil, coef, dims, laplacian=True)
    kw = dict(beta_lap=oracle.round_to_storage(blap, storage)) if sep else {}
    assert_parity(few, oracle.bspline_eval(oracle.round_to_storage(beta, storage), lat, base, **kw), TOL[storage],
                  "%s %d orbitals" % (storage, orb))
    # 4 rounds of 20 warps per SM: the first call with records has at least that many warp tasks
    warps = 80 * torch.cuda.get_device_properties(dev()).multi_processor_count
    limit = warps * (32 // info["lanes"]) // info["tiles"]
    for n in sorted({8191, 8192, max(8192, limit - 1), max(8192, limit + 32)}):
        pos = np.resize(base, (n, 3))
        for a, b in zip(spl.eval_vgl(torch.from_numpy(pos).to(dev())), few):
            assert np.array_equal(a.cpu().numpy(), np.resize(b, (n,) + b.shape[1:])), n
    spl.close()
