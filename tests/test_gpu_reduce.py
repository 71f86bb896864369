"""Segmented sums of every length class: one lane, one warp, several blocks, and their edges."""
import numpy as np
import pytest
import torch

import oracle
from paper_2608_16265_gb300 import binding
from paper_2608_16265_gb300.ir import Model

pytestmark = pytest.mark.gpu

# entries per variable / per row: nothing, one, the last of one class and the first of the next
LENGTHS = [0, 1, 2, 31, 32, 33, 64, 257, 2047, 2048, 2049, 4096, 4097, 8193]


def segments_model(lengths, spread):
    """Variable and row j receive lengths[j] terms each (objective gradient, augmentations, Jacobian and
    Hessian columns); with `spread`, every other variable receives none."""
    rng = np.random.default_rng(3)
    step = 3 if spread else 1
    idx = np.concatenate([np.full(n, step * j) for j, n in enumerate(lengths)]).astype(np.int32)
    idx = idx[rng.permutation(len(idx))]
    m = Model()
    x = m.add_var(step * len(lengths))
    m.add_obj(lambda d: d.w * x[d.i] ** 2, data=dict(i=idx, w=rng.uniform(0.5, 1.5, len(idx))))
    rows = m.add_con(lambda d: d.a * x[d.k], data=dict(a=rng.uniform(0.5, 1.5, step * len(lengths))))
    m.add_con_aug(rows, lambda d: (d.r, d.w * x[d.r] ** 2),
                  data=dict(r=idx, w=rng.uniform(0.5, 1.5, len(idx))))
    return m.flat()


@pytest.mark.parametrize("spread", [False, True])
@pytest.mark.parametrize("batch", [False, True])
def test_segment_lengths(spread, batch):
    lists = [LENGTHS] if not batch else [LENGTHS, [1] * 5, LENGTHS[::-1], [3000], [40, 2]]
    flats = [segments_model(n, spread) for n in lists]
    m = binding.exa_create_batch(flats, flags=binding.EXA_FLAG_NO_TUNE, chunks=3 if batch else 0)
    rng = np.random.default_rng(5)
    xs = [rng.uniform(0.5, 1.5, f.nvar) for f in flats]
    ys = [rng.uniform(0.5, 1.5, f.ncon) for f in flats]
    x, y = (torch.as_tensor(np.concatenate(a), device="cuda") for a in (xs, ys))
    out = m.eval_all(x, y, 1.0, csc=True)
    got = {k: t.cpu().numpy() for k, t in out.items()}
    one = dict(f=m.obj(x), g=m.grad(x), c=m.cons(x), jac_csc=m.jac_csc(x), hess_csc=m.hess_csc(x, y))
    vs = [rng.uniform(0.5, 1.5, f.nvar) for f in flats]
    ws = [rng.uniform(0.5, 1.5, f.ncon) for f in flats]
    v, w = (torch.as_tensor(np.concatenate(a), device="cuda") for a in (vs, ws))
    one.update(jv=m.jprod(x, v), jtw=m.jtprod(x, w), hv=m.hprod(x, y, 1.0, v))
    one = {k: t.cpu().numpy() for k, t in one.items()}
    orc = [oracle.Oracle(f) for f in flats]
    ref = dict(f=np.array([sum(o.obj(a) for o, a in zip(orc, xs))]),
               g=np.concatenate([o.grad(a) for o, a in zip(orc, xs)]),
               c=np.concatenate([o.cons(a) for o, a in zip(orc, xs)]),
               jac_csc=np.concatenate([o.jac_csc(a) for o, a in zip(orc, xs)]),
               hess_csc=np.concatenate([o.hess_csc(a, b, 1.0) for o, a, b in zip(orc, xs, ys)]),
               jv=np.concatenate([o.jprod(a, b) for o, a, b in zip(orc, xs, vs)]),
               jtw=np.concatenate([o.jtprod(a, b) for o, a, b in zip(orc, xs, ws)]),
               hv=np.concatenate([o.hprod(a, b, 1.0, c) for o, a, b, c in zip(orc, xs, ys, vs)]))
    # every term is positive: two orders of a sum of n terms differ by at most 2 (n + 4) ulp of the sum
    # (at most four operations form a term; a variable's second-order sum has the terms of the objective
    # and of the rows), and the objective adds all of them
    n = max(sum(v) for v in lists)
    for k, r in ref.items():
        tol = 2 * ((len(lists) * n if k == "f" else 2 * max(max(v) for v in lists)) + 4) * 2.0 ** -53
        for a in [d[k] for d in (got, one) if k in d]:
            assert a.shape == r.shape
            assert np.all(np.abs(a - r) <= tol * np.abs(r)), k


@pytest.mark.parametrize("fused", [False, True])
@pytest.mark.parametrize("case", ["all_sole", "one_shared", "few_sole", "mixed_members"])
def test_sole_gradient_slots(case, fused):
    """Patterns whose gradient slots are their variables' only ones write the gradient themselves; one
    shared variable, or a member where they are not, and the pattern goes through the sums."""
    def model(n, extra, spare):
        m = Model()
        x = m.add_var(2 * n + spare)
        m.add_obj(lambda d: d.a * x[d.i] ** 2 * x[d.k + n],
                  data=dict(i=np.random.default_rng(1).permutation(n).astype(np.int32), a=np.arange(1.0, n + 1)))
        m.add_obj(lambda d: 2 * x[d.j], data=dict(j=np.asarray(extra, np.int32)))
        m.add_con(lambda d: x[d.k] * x[d.k + 1], n=3)
        return m.flat()

    flats = {"all_sole": [model(70, [140], 1)], "one_shared": [model(70, [140, 7], 1)],
             "few_sole": [model(33, [66], 400)], "mixed_members": [model(33, [66, 67], 2), model(33, [66, 0], 2)]}[case]
    m = binding.exa_create_batch(flats, flags=binding.EXA_FLAG_NO_TUNE | (binding.EXA_FLAG_FUSED_STEP if fused else 0))
    x = np.random.default_rng(2).uniform(0.5, 1.5, m.nvar)
    ref = np.concatenate([oracle.Oracle(f).grad(x[m.xoff[b]:m.xoff[b + 1]]) for b, f in enumerate(flats)])
    xt, yt = torch.as_tensor(x, device="cuda"), torch.ones(m.ncon, dtype=torch.float64, device="cuda")
    for g in (m.grad(xt), m.eval_all(xt, yt, 1.0, csc=True)["g"], m.eval_all(xt, yt, 1.0)["g"]):
        g = g.cpu().numpy()
        # products of at most four factors, sums of at most two terms
        assert np.all(np.abs(g - ref) <= 8 * 2.0 ** -53 * np.abs(ref) * 2)
