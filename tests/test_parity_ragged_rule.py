"""Which launches stage their unaligned rows (bfloat16 tables from three warp tasks per SM; float cubic
tables of few chunks a position beyond small launches) leaves every value as it is: the outputs on both
sides of the rule's lines equal those of the same orbitals in rows of whole chunks."""
import numpy as np
import pytest

from paper_1309_6250_gb300 import inputs
from gpu_helpers import NONORTHO, dev
from test_parity_ragged_rows import DIMS, evaluate

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kw", [dict(), dict(separate_lap=False), dict(separate_grad=True), dict(method="pp")])
@pytest.mark.parametrize("storage,n_orb", [("f32", 2), ("f32", 23), ("f32", 25), ("f32", 39), ("f32", 41),
                                           ("bf16", 21), ("bf16", 57)])
def test_rows_on_both_sides_of_the_rule(storage, n_orb, kw):
    from paper_1309_6250_gb300.api import OrbitalSplines
    args = dict(dict(method="interp", storage=storage, device=dev()), **kw)
    wide = n_orb + -n_orb % 4
    mil = inputs.miller_set(NONORTHO, 5.0, None)
    coef = inputs.pw_coefficients(NONORTHO, mil, wide, 4.0, 5)
    full = OrbitalSplines(NONORTHO, DIMS, mil, coef, **args)
    part = OrbitalSplines(NONORTHO, DIMS, mil, coef[:n_orb], **args)
    inf = part.info()
    per_task = 32 // inf["lanes"] / inf["tiles"]      # positions per warp task
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    for tasks in (3 * sms - 1, 3 * sms + 1, 8 * sms - 1, 8 * sms + 1):
        n = max(1, int(tasks * per_task))
        pos = torch.from_numpy(inputs.positions(NONORTHO, n, 79, -1.0, 2.0)).to(dev())
        ref = evaluate(full, pos, 0)
        for shift in (0, 1):
            for a, b in zip(evaluate(part, pos, shift), ref):
                np.testing.assert_array_equal(a, b[..., :n_orb])
