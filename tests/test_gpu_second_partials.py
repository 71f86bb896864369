"""Second derivatives entry by entry where the naive rules lose digits: hypot with one operand far below the
other (or zero), real powers with exponents near 1 and 2, negative powers near overflow, atan2."""
import numpy as np
import pytest
import torch

import oracle
from paper_2608_16265_gb300 import binding as B
from paper_2608_16265_gb300.ir import Model, atan2, hypot

pytestmark = pytest.mark.gpu

# (function of the instance's variables a and b and its datum e, values of a, b, e)
SMALL = np.concatenate([[0.0], 10.0 ** -np.arange(9)])
EXP = np.array([1.0, 1 + 1e-12, 1 - 1e-8, 1 + 1e-4, 1.5, 2.0, 2 - 1e-8, 2 + 1e-4, 2.5, -0.5])
CASES = dict(
    hypot_ab=(lambda a, b, e: hypot(a, b), [1 / 3, -1.0, 1e4], SMALL, [1.0]),
    hypot_ba=(lambda a, b, e: hypot(b, a), [1 / 3, -1.0, 1e4], SMALL, [1.0]),
    hypot_const=(lambda a, b, e: hypot(a, 1e-4) + b, [1 / 3, -1.0, 1e4, 1e-6], [1.0], [1.0]),
    hypot_ratio=(lambda a, b, e: a / hypot(a, b), [1 / 3, -1.0, 1e4], SMALL[1:], [1.0]),
    pow=(lambda a, b, e: a ** e + b, [1e-3, 0.7, 2.0, 9.0], [1.0], EXP),
    powm5=(lambda a, b, e: a ** -5 + b, [1e-40, -1e-3, 0.7, 9.0, 1e30], [1.0], [1.0]),
    powm2=(lambda a, b, e: (-a) ** -2 + b, [1e-70, -1e-3, 0.7, 9.0], [1.0], [1.0]),
    atan2=(lambda a, b, e: atan2(a, b), [1 / 3, -1.0, 1e4], SMALL, [1.0]),
)


@pytest.mark.parametrize("name", list(CASES))
def test_entry_by_entry(name):
    fn, av, bv, ev = CASES[name]
    a, b, e = (t.ravel() for t in np.meshgrid(av, bv, ev))
    n = len(a)
    m = Model()
    x, z = m.add_var(n), m.add_var(n)
    d = dict(e=e)
    m.add_obj(lambda d: fn(x[d.k], z[d.k], d.e), data=d)  # two patterns: the Hessian CSC comes from their group's sums
    m.add_con(lambda d: fn(x[d.k], z[d.k], d.e), data=d)
    flat = m.flat()
    o, mm = oracle.Oracle(flat), B.exa_create(flat, flags=B.EXA_FLAG_NO_TUNE)
    xv, y = np.concatenate([a, b]), np.random.default_rng(1).uniform(0.5, 1.5, n)
    X, Y = (torch.as_tensor(t, device="cuda") for t in (xv, y))
    ref = o.hess_csc(xv, y, 0.75)
    # up to 16 operations of at most 2 ulp on either side, and two terms of one sign
    tol = 2 * 16 * 2 * 2.0 ** -53
    # (in atan2's (u^2 - w^2) / r^2 and in the quotient, terms of at most 1 / r^2 cancel)
    cancel = 4 * (0.75 + 1.5) / np.tile(a * a + b * b, 2) if name in ("atan2", "hypot_ratio") else None
    cols = np.repeat(np.arange(2 * n), np.diff(o.hess_csc_structure()[0]))
    for h in (mm.hess_csc(X, Y, 0.75), mm.eval_all(X, Y, 0.75, csc=True)["hess_csc"]):
        assert np.all(np.abs(h.cpu().numpy() - ref) <= tol * (np.abs(ref) if cancel is None else cancel[cols]))
    # H v column by column: v = 1 on all first, then on all second variables (no two instances share one)
    for half in (0, 1):
        v = np.zeros(2 * n)
        v[half * n:(half + 1) * n] = 1.0
        h, r = mm.hprod(X, Y, 0.75, torch.as_tensor(v, device="cuda")).cpu().numpy(), o.hprod(xv, y, 0.75, v)
        assert np.all(np.abs(h - r) <= tol * (np.abs(r) if cancel is None else cancel))
