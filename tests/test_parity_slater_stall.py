"""A wait for a pivot column that runs out (test hook: the column of one walker is never announced) in
the register-resident Slater kernels: the launch ends by itself, every output of that walker is NaN, also
where its matrix is exactly singular (a stalled walker must not pass for one with a zero determinant), the
other walkers' outputs are untouched and the next call is right."""
import numpy as np
import pytest

from gpu_helpers import dev

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("singular", [False, True])
@pytest.mark.parametrize("cplx,n_up,n_dn", [(False, 20, 20), (False, 120, 100), (True, 20, 0), (True, 70, 96)])
def test_stalled_walker_is_nan(cplx, n_up, n_dn, singular):
    from paper_1309_6250_gb300 import _lib
    from paper_1309_6250_gb300.api import slater_kinetic
    W, ne, O = 3, n_up + n_dn, max(n_up, n_dn)
    g = torch.Generator(device=dev()).manual_seed(9900 + n_up)
    rand = lambda *s: torch.randn(*s, generator=g, device=dev(), dtype=torch.complex64 if cplx else torch.float32)
    val, grad, lap = rand(W * ne, O), rand(W * ne, 3, O), rand(W * ne, O)
    if singular:
        val[:n_up, 0] = 0
    ref = slater_kinetic(val, grad, lap, W, ne, n_up)
    assert bool(torch.isneginf(ref[0][0])) == singular
    L = _lib.load()
    try:
        L.qmcspl_debug_stall_slater(1)
        out = slater_kinetic(val, grad, lap, W, ne, n_up)
        again = slater_kinetic(val, grad, lap, W, ne, n_up)
        torch.cuda.synchronize()
    finally:
        L.qmcspl_debug_stall_slater(0)
    for a, b, c in zip(out, ref, again):
        assert torch.isnan(torch.view_as_real(a[0]) if a.is_complex() else a[0]).all()
        assert torch.equal(a[1:], b[1:]) and torch.equal(c[1:], b[1:])
        np.testing.assert_array_equal(c[0].cpu().numpy(), b[0].cpu().numpy())


@pytest.mark.parametrize("cplx", [False, True])
def test_stall_is_reported_once(cplx):
    """qmcspl_slater_sync: ERR_TIMEOUT for the stalled launch, nothing before it and nothing after."""
    from paper_1309_6250_gb300 import _lib
    from paper_1309_6250_gb300.api import slater_kinetic, slater_sync
    g = torch.Generator(device=dev()).manual_seed(9950)
    val = torch.randn(2 * 9, 5, generator=g, device=dev(), dtype=torch.complex128 if cplx else torch.float64)
    call = lambda: slater_kinetic(val, None, None, 2, 9, 5)
    L = _lib.load()
    try:
        slater_sync()
    except _lib.QmcsplError:
        pass                                  # an earlier launch's
    call()
    slater_sync()
    try:
        L.qmcspl_debug_stall_slater(1)
        out = call()
        with pytest.raises(_lib.QmcsplError) as ei:
            slater_sync()
        assert ei.value.code == _lib.ERR_TIMEOUT
    finally:
        L.qmcspl_debug_stall_slater(0)
    assert torch.isnan(out[0][0]) and not torch.isnan(out[0][1])
    call()
    slater_sync()
