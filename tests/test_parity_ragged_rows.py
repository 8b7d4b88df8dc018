"""Outputs whose rows are not whole 16-byte chunks (orbital counts that are no multiple of four, output
buffers off a 16-byte boundary) leave through shared memory: the same values as the vector stores, and
nothing written outside the rows."""
import numpy as np
import pytest

from paper_1309_6250_gb300 import inputs
from gpu_helpers import NONORTHO, dev

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DIMS = (9, 8, 11)


def evaluate(spl, pos, shift):
    """Outputs in buffers `shift` floats off a 16-byte boundary, with a guard on both sides."""
    n, o = pos.shape[0], spl.n_orb
    flat = [torch.full((n * k * o + 16,), 7.5, dtype=spl.result_dtype, device=dev()) for k in (1, 3, 1)]
    out = [t[shift:shift + n * k * o].view(s) for t, k, s in zip(flat, (1, 3, 1), ((n, o), (n, 3, o), (n, o)))]
    spl.eval_vgl(pos, out=out)
    spl.sync()
    for t, k in zip(flat, (1, 3, 1)):
        assert torch.all(t[:shift] == 7.5) and torch.all(t[shift + n * k * o:] == 7.5)
    return [t.cpu().numpy() for t in out]


@pytest.mark.parametrize("kw", [dict(), dict(separate_lap=False), dict(separate_grad=True), dict(method="lagrange"),
                                dict(method="pp"), dict(kpoint=(0.2, 0.1, -0.3))])
@pytest.mark.parametrize("storage", ["f32", "bf16"])
@pytest.mark.parametrize("n_orb", [1, 7, 33, 109, 130])
def test_ragged_rows(n_orb, storage, kw):
    from paper_1309_6250_gb300.api import OrbitalSplines
    args = dict(method="interp", storage=storage, device=dev(), **{k: v for k, v in kw.items() if k != "method"})
    if "method" in kw:
        args["method"] = kw["method"]
    lat = NONORTHO
    wide = n_orb + -n_orb % 4                      # the same orbitals and a few more: rows of whole chunks
    k = kw.get("kpoint")
    mil = inputs.miller_set(lat, 5.0, k)
    coef = (inputs.bloch_coefficients(lat, mil, wide, k, 4.0, 5) if k is not None
            else inputs.pw_coefficients(lat, mil, wide, 4.0, 5))
    full = OrbitalSplines(lat, DIMS, mil, coef, **args)
    part = OrbitalSplines(lat, DIMS, mil, coef[:n_orb], **args)
    for n, order in ((1, "input"), (45, "input"), (9001, "cell")):
        pos = torch.from_numpy(inputs.positions(lat, n, 78, -1.0, 2.0)).to(dev())
        full.set_order(order)
        part.set_order(order)
        ref = evaluate(full, pos, 0)
        for shift in (0, 1, 2):
            for a, b in zip(evaluate(part, pos, shift), ref):
                np.testing.assert_array_equal(a, b[..., :n_orb])
