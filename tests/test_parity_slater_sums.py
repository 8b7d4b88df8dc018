"""The final sums of the double-float Slater consumer are FP64: kinetic energy and drift keep every bit
and the whole range of the gradients and Laplacians that they are made of.

Every spin block is a signed (complex: by units 1, i, -1, -i) permutation matrix with powers of two in
it, so that its inverse is exact and an electron's sum has one term that is not zero.  The drift must
then equal that term bit for bit; the kinetic energy is a sum of n such terms in FP64, off by at most
n 2^-53 of the sum of their moduli (an addition's rounding each; twice that for a part of a complex sum)."""
import numpy as np
import pytest

from gpu_helpers import dev

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

W = 3


def consumer(val, grad, lap, n_elec, n_up):
    from paper_1309_6250_gb300.api import slater_kinetic
    out = slater_kinetic(*(torch.from_numpy(x).to(dev()) for x in (val, grad, lap)), W, n_elec, n_up)
    torch.cuda.synchronize()
    return [x.cpu().numpy() for x in out]


def blocks(rng, n_up, n_dn, pad, dtype):
    """val, each electron's orbital and its entry of the inverse; columns past a block hold NaN, which
    no sum may touch."""
    ne, O = n_up + n_dn, max(n_up, n_dn) + pad
    val = np.full((W, ne, O), np.nan, dtype=dtype)
    orb = np.empty((W, ne), dtype=int)
    inv = np.empty((W, ne), dtype=np.result_type(dtype, np.float64))
    units = np.array([1, 1j, -1, -1j] if np.iscomplexobj(val) else [1.0, -1.0])
    for w in range(W):
        for e0, n in ((0, n_up), (n_up, n_dn)):
            if not n:
                continue
            u, k = units[rng.integers(len(units), size=n)], rng.integers(-12, 13, size=n)
            o = rng.permutation(n)
            val[w, e0:e0 + n, :n] = 0
            val[w, e0 + np.arange(n), o] = u * 2.0 ** k
            orb[w, e0:e0 + n], inv[w, e0:e0 + n] = o, np.conj(u) * 2.0 ** -k
    return val.reshape(W * ne, O), orb, inv


def derivatives(rng, shape, dtype, scale):
    x = rng.standard_normal(shape + (2,)) * scale
    return np.ascontiguousarray((x[..., 0] + 1j * x[..., 1] if np.issubdtype(dtype, np.complexfloating) else x[..., 0])
                                .astype(dtype))


@pytest.mark.parametrize("scale", ["one", "large"])
@pytest.mark.parametrize("dtype,n_up,n_dn", [(d, *n) for d in (np.float32, np.float64)
                                             for n in ((1, 1), (31, 2), (33, 64), (97, 128), (130, 0))] +
                         [(d, *n) for d in (np.complex64, np.complex128)
                          for n in ((1, 1), (31, 2), (33, 64), (96, 65), (100, 0))])
def test_sums_keep_all_bits(dtype, n_up, n_dn, scale):
    rng = np.random.default_rng(9700 + 200 * n_up + n_dn)
    ne = n_up + n_dn
    val, orb, inv = blocks(rng, n_up, n_dn, 2, dtype)
    # large: products past the largest float, which a double holds
    s = 1.0 if scale == "one" else (3e37 if np.finfo(dtype).bits == 32 else 1e300)
    grad, lap = derivatives(rng, (W * ne, 3, val.shape[1]), dtype, s), derivatives(rng, val.shape, dtype, s)
    _, _, kin, drift = consumer(val, grad, lap, ne, n_up)
    w, e = np.indices((W, ne))
    g = grad.reshape(W, ne, 3, -1)[w, e, :, orb].astype(inv.dtype)
    terms = inv * lap.reshape(W, ne, -1)[w, e, orb].astype(inv.dtype)
    np.testing.assert_array_equal(drift, inv[..., None] * g)
    err = np.abs(kin + 0.5 * terms.sum(1))
    assert np.all(err <= 0.5 * 2 * (ne + 2) * 2.0 ** -53 * np.abs(terms).sum(1))


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("n_up,n_dn", [(5, 4), (64, 63), (128, 100)])
def test_infinite_derivatives_stay_infinite(n_up, n_dn, dtype):
    rng = np.random.default_rng(9800 + n_up)
    ne = n_up + n_dn
    val, orb, inv = blocks(rng, n_up, n_dn, 0, dtype)
    grad, lap = derivatives(rng, (W * ne, 3, val.shape[1]), dtype, 1.0), derivatives(rng, val.shape, dtype, 1.0)
    e = ne - 2
    grad.reshape(W, ne, 3, -1)[0, e, 1, orb[0, e]] = np.inf
    lap.reshape(W, ne, -1)[1, e, orb[1, e]] = -np.inf
    _, _, kin, drift = consumer(val, grad, lap, ne, n_up)
    assert drift[0, e, 1] == np.sign(inv[0, e]) * np.inf
    assert kin[1] == np.sign(inv[1, e]) * np.inf
    drift[0, e, 1] = 0.0
    assert np.all(np.isfinite(drift)) and np.all(np.isfinite(kin[[0, 2]]))
