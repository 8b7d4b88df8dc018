"""The register-resident double-float Slater consumer of complex orbitals (spin blocks of at most 96
electrons) at the edges of its shapes, against the oracle's definition (numpy slogdet / inv).

The orbital matrices are complex N(0, 1) plus a dominant scattered entry per row, so that their
condition numbers stay below about 1e3: with parts of about 48 significant bits (2^-47 = 7e-15) the
relative error of the inverse is below 2 n * cond * 2^-47 < 2e-9, the tolerance of its sums 1e-8."""
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


@pytest.mark.parametrize("dtype", [np.complex64, np.complex128])
@pytest.mark.parametrize("n_up,n_dn,pad", [(1, 1, 0), (31, 2, 1), (32, 32, 0), (33, 0, 3), (5, 64, 0), (64, 65, 0),
                                           (95, 96, 5), (96, 97, 0)])
def test_complex_register_consumer_shape_edges(n_up, n_dn, pad, dtype):
    rng = np.random.default_rng(9700 + 200 * n_up + n_dn)
    W, ne, O = 5, n_up + n_dn, max(n_up, n_dn) + pad
    z = lambda *s: (rng.standard_normal(s) + 1j * rng.standard_normal(s)).astype(dtype)  # noqa: E731
    val, grad, lap = z(W * ne, O), z(W * ne, 3, O), z(W * ne, O)
    for e0, n in ((0, n_up), (n_up, n_dn)):
        for w in range(W):
            for i in range(n):   # every step has to find its pivot
                val[w * ne + e0 + i, (7 * i + 3) % n if n % 7 else i] += (2.0 + 3.0j) * np.sqrt(n)
    zero = W - 1                                   # one walker with a zero row: exactly singular
    val[zero * ne + ne - 1] = 0
    t = [torch.from_numpy(x).to(dev()) for x in (val, grad, lap)]
    ld, sg, kin, dr = consumer(*t, W, ne, n_up)
    keep = W - 1
    ref = oracle.slater_kinetic(*(x[:keep * ne].astype(np.complex128) for x in (val, grad, lap)), keep, ne, n_up)
    assert np.max(np.abs(ld[:keep] - ref[0])) <= 1e-9 * max(1.0, np.max(np.abs(ref[0])))
    assert np.max(np.abs(sg[:keep] - ref[1])) <= 1e-9
    for got, want in ((kin[:keep], ref[2]), (dr[:keep], ref[3])):
        assert np.max(np.abs(got - want)) <= 1e-8 * np.max(np.abs(want))
    assert sg[zero] == 0 and ld[zero] == -np.inf and np.isnan(kin[zero]) and np.all(np.isnan(dr[zero]))
    # without the gradient or the Laplacian the other outputs are the same bits
    ld2, sg2, kin2, none = consumer(t[0], None, t[2], W, ne, n_up)
    assert none is None
    np.testing.assert_array_equal(ld2, ld)
    np.testing.assert_array_equal(sg2, sg)
    np.testing.assert_array_equal(kin2, kin)
