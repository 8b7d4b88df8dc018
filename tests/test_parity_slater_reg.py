"""The register-resident double-float Slater consumer (spin blocks of at most 128 electrons) at the
edges of its 32 x 32 warp tiles, against the oracle's definition (numpy slogdet / inv).

The orbital matrices are N(0, 1) plus a multiple of the identity, so that their condition numbers
stay below about 1e3: with entries of about 48 significant bits (2^-47 = 7e-15) the relative error
of the inverse is below n * cond * 2^-47 < 1e-9, the consumer's tolerance."""
import numpy as np
import pytest

import oracle
from gpu_helpers import dev

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def consumer(*args, **kw):
    from paper_1309_6250_gb300.api import slater_kinetic
    out = slater_kinetic(*args, **kw)
    torch.cuda.synchronize()
    return [None if x is None else x.cpu().numpy() for x in out]


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("n_up,n_dn,pad", [(1, 1, 0), (31, 2, 1), (32, 32, 0), (33, 0, 3), (5, 63, 0), (64, 65, 0),
                                           (95, 96, 5), (97, 33, 0), (127, 128, 1), (128, 129, 0)])
def test_register_consumer_tile_edges(n_up, n_dn, pad, dtype):
    rng = np.random.default_rng(9100 + 200 * n_up + n_dn)
    W, ne, O = 5, n_up + n_dn, max(n_up, n_dn) + pad
    val = rng.standard_normal((W * ne, O)).astype(dtype)
    for e0, n in ((0, n_up), (n_up, n_dn)):
        for w in range(W):
            for i in range(n):   # a scattered dominant entry per row: every step has to find its pivot
                val[w * ne + e0 + i, (7 * i + 3) % n if n % 7 else i] += 3.0 * np.sqrt(n)
    grad = rng.standard_normal((W * ne, 3, O)).astype(dtype)
    lap = rng.standard_normal((W * ne, O)).astype(dtype)
    zero = W - 1                                   # one walker with a zero row: exactly singular
    val[zero * ne + ne - 1] = 0
    t = [torch.from_numpy(x).to(dev()) for x in (val, grad, lap)]
    ld, sg, kin, dr = consumer(*t, W, ne, n_up)
    keep = W - 1
    ref = oracle.slater_kinetic(*(x[:keep * ne].astype(np.float64) for x in (val, grad, lap)), keep, ne, n_up)
    np.testing.assert_array_equal(sg[:keep], ref[1])
    assert np.max(np.abs(ld[:keep] - ref[0])) <= 1e-9 * max(1.0, np.max(np.abs(ref[0])))
    assert oracle.relative_error(kin[:keep], ref[2]) < 1e-8
    assert oracle.relative_error(dr[:keep], ref[3]) < 1e-8
    assert sg[zero] == 0 and ld[zero] == -np.inf and np.isnan(kin[zero]) and np.all(np.isnan(dr[zero]))
    # without the gradient or the Laplacian the other outputs are the same bits
    ld2, sg2, kin2, none = consumer(t[0], None, t[2], W, ne, n_up)
    assert none is None
    np.testing.assert_array_equal(ld2, ld)
    np.testing.assert_array_equal(sg2, sg)
    np.testing.assert_array_equal(kin2, kin)
