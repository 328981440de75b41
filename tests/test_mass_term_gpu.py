"""The Helmholtz mass term inside the operator handle's kernel, at every order
that has it and with elements that leave the double-float range (fp64-unit
fallback): w = Ax(u) + h2 B u from the same handle without the term, to one
fp64 rounding of the sum."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2506_20994_gb300 as ax  # noqa: E402
from paper_2506_20994_gb300 import synth  # noqa: E402

from _cases import GKEYS, operator_case  # noqa: E402


@pytest.mark.parametrize("lx", [6, 8, 10, 12])
@pytest.mark.parametrize("dims", [(1, 1, 1), (13, 11, 9)])
def test_mass_term_joins_the_apply(lx, dims):
    c = operator_case(dims, lx, seed=500 + lx)
    u = c["u"].copy()
    u[::5] *= 1e70
    t = lambda a: torch.as_tensor(np.ascontiguousarray(a), device="cuda", dtype=torch.float64)
    d = {k: t(c[k]) for k in ("dx", "dxt", "h1") + GKEYS}
    tu, h2, B = t(u), t(synth.uniform(u.shape, 1, 0.1, 3.0)), t(synth.uniform(u.shape, 2, 0.1, 1.0))
    op = ax.Operator(lx, d["dx"], d["dxt"], d["h1"], *[d[k] for k in GKEYS])
    plain = torch.empty_like(tu)
    op.apply(plain, tu)
    op.set_h2(h2, B)
    w = torch.full_like(tu, float("nan"))
    op.apply(w, tu)
    m = (h2 * B) * tu
    # one rounding of the product or the sum, on either side
    assert bool(((w - (plain + m)).abs() <= 2.0 ** -51 * (plain.abs() + m.abs())).all())
    op.set_h2(None, None)
    op.apply(w, tu)
    assert torch.equal(w, plain)
