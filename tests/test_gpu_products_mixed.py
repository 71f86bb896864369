"""Mixed-precision products are those of the entries that exa_jac_coord and exa_hess_csc return, whatever
the launch configuration; long rows and columns of the Hessian included."""
import numpy as np
import pytest
import torch

import synth
from paper_2608_16265_gb300 import binding as B
from paper_2608_16265_gb300.ir import Model, cos, sin

pytestmark = pytest.mark.gpu


def shared_variable(n):
    """n rows over one common variable: its Hessian row, and its Jacobian column, have n entries."""
    m = Model()
    t, x = m.add_var(1), m.add_var(n)
    m.add_con(lambda d: t[0] * x[d.k] ** 2 + sin(x[d.k] * t[0]) * cos(x[d.k]), n=n)
    m.add_obj(lambda d: x[d.k] ** 3, n=n)
    return m.flat()


MODELS = dict(rosenbrock=lambda: synth.rosenbrock(1500).flat, acopf=lambda: synth.acopf(300, 420, 50, seed=2).flat,
              goddard=lambda: synth.goddard(400).flat, **{f"shared{n}": (lambda n=n: shared_variable(n))
                                                          for n in (1, 31, 32, 255, 256, 257, 8192, 8193, 20000)})


@pytest.mark.parametrize("flags", [0, B.EXA_FLAG_LAZY_LOADS, B.EXA_FLAG_LAZY_LOADS | B.EXA_FLAG_SPLIT])
@pytest.mark.parametrize("name", list(MODELS))
def test_products_of_the_entries(name, flags):
    flat = MODELS[name]()
    m = B.exa_create(flat, B.EXA_MIXED_FP32, flags=flags | B.EXA_FLAG_NO_TUNE)
    rng = np.random.default_rng(1)
    x, y = rng.uniform(0.4, 1.2, m.nvar), rng.standard_normal(m.ncon)
    v, w = rng.standard_normal(m.nvar), rng.standard_normal(m.ncon)
    X, Y, V, W = (torch.as_tensor(a, device="cuda") for a in (x, y, v, w))
    jr, jc = (a.cpu().numpy() for a in m.jac_structure())
    J = m.jac_coord(X).cpu().numpy()
    cp, hr, _ = (a.cpu().numpy() for a in m.hess_csc_structure())
    hc, H = np.repeat(np.arange(m.nvar), np.diff(cp)), m.hess_csc(X, Y, 1.3).cpu().numpy()
    off = hr != hc

    def add(n, *terms):  # the sums, and the sums of magnitudes
        r, a, c = np.zeros(n), np.zeros(n), np.zeros(n)
        for i, t in terms:
            with np.errstate(invalid="ignore"):
                np.add.at(r, i, t)
            np.add.at(a, i, np.abs(t))
            np.add.at(c, i, 1)
        return r, a, c

    got = dict(jv=m.jprod(X, V), jtw=m.jtprod(X, W), hv=m.hprod(X, Y, 1.3, V))
    ref = dict(jv=add(m.ncon, (jr, J * v[jc])), jtw=add(m.nvar, (jc, J * w[jr])),
               hv=add(m.nvar, (hc, H * v[hr]), (hr[off], (H * v[hc])[off])))
    for k, (r, mag, cnt) in ref.items():  # n rounded products added in another order: 2 (n + 1) 2^-53 of the magnitudes
        g = got[k].cpu().numpy()
        with np.errstate(invalid="ignore"):  # (the rocket's drag overflows FP32 at this point: the same infinities and NaN)
            ok = (np.abs(g - r) <= 2 * (cnt + 1) * 2.0 ** -53 * mag) & np.isfinite(mag)
        assert np.all(ok | (g == r) | (np.isnan(g) & np.isnan(r))), k
    rows = max(np.diff(cp).max(), np.bincount(hr).max())
    assert int(m.stat("hprod_route")) == (2 if rows > 32 else 1)  # sums by length / one lane per variable
