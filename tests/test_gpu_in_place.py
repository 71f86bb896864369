"""The gradient written over the point, and J v over the point: every read of x comes before."""
import numpy as np
import pytest
import torch

import oracle
from paper_2608_16265_gb300 import binding as B
from paper_2608_16265_gb300.ir import Model

pytestmark = pytest.mark.gpu


def model(n, spare, seed=1):
    """Sole gradient slots (a permutation, so that instances read what others write), some shared ones."""
    r = np.random.default_rng(seed)
    m = Model()
    x = m.add_var(2 * n + spare)
    m.add_obj(lambda d: d.a * x[d.i] ** 2 * x[d.j + n], data=dict(
        i=r.permutation(n).astype(np.int32), j=r.permutation(n).astype(np.int32), a=r.uniform(0.5, 1.5, n)))
    m.add_obj(lambda d: x[2 * n] ** 2 * d.b, data=dict(b=r.uniform(0.5, 1.5, 3)))
    m.add_con(lambda d: x[d.i] * x[d.j], data=dict(i=r.permutation(n).astype(np.int32), j=r.permutation(n).astype(np.int32)))
    return m.flat()


@pytest.mark.parametrize("precision,tol", [(B.EXA_FP64, 16 * 2.0 ** -53), (B.EXA_MIXED_FP32, 16 * 2.0 ** -24)])
@pytest.mark.parametrize("sizes,chunks", [([33], 0), ([40000], 0), ([300, 20000, 7000], 0), ([300, 20000, 7000], 3)])
@pytest.mark.parametrize("spare", [1, 90000])  # few variables without a slot, and most of them
def test_in_place(sizes, chunks, spare, precision, tol):
    flats = [model(n, spare, n) for n in sizes]
    m = B.exa_create_batch(flats, precision, flags=B.EXA_FLAG_NO_TUNE, chunks=chunks)
    rng = np.random.default_rng(2)
    x, v = rng.uniform(0.5, 1.5, m.nvar), rng.uniform(0.5, 1.5, m.nvar)
    parts = [(oracle.Oracle(f), x[m.xoff[b]:m.xoff[b + 1]], v[m.xoff[b]:m.xoff[b + 1]]) for b, f in enumerate(flats)]
    g = np.concatenate([o.grad(a) for o, a, _ in parts])
    jv = np.concatenate([o.jprod(a, c) for o, a, c in parts])
    t = lambda a: torch.as_tensor(a, device="cuda")  # noqa: E731
    y = torch.ones(m.ncon, dtype=torch.float64, device="cuda")

    def near(a, r):  # products of at most four factors, sums of at most three terms, all positive
        assert np.all(np.abs(a.cpu().numpy() - r) <= tol * r)

    X = t(x)
    m.exa_grad(X, X)
    near(X, g)
    X = t(x)
    m.exa_jprod(X, t(v), X[:m.ncon])
    near(X[:m.ncon], jv)
    for csc in (False, True):
        out = m.eval_all(t(x), y, 1.0, csc=csc)
        X = t(x)
        out["g"] = X
        ref = {k: a.clone() for k, a in out.items() if k != "g"}
        for _ in range(2):  # the second from the cached graph
            X.copy_(t(x))
            m.exa_eval_all(X, y, 1.0, **out)
            near(X, g)
            for k, a in ref.items():
                assert torch.equal(out[k], a), k
