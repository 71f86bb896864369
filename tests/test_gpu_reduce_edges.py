"""Segmented sums at the last length of each class (32, 256 and 8192 entries), the first of the next, and
segments of whole pieces (4096 entries)."""
import numpy as np
import pytest
import torch

import oracle
from paper_2608_16265_gb300 import binding
from tests.test_gpu_reduce import segments_model

pytestmark = pytest.mark.gpu

LENGTHS = [32, 33, 255, 256, 257, 8191, 8192, 8193, 3 * 4096, 3 * 4096 + 1]


@pytest.mark.parametrize("precision,ulp", [(binding.EXA_FP64, 2.0 ** -53), (binding.EXA_MIXED_FP32, 2.0 ** -24)])
@pytest.mark.parametrize("spread", [False, True])
def test_class_edges(spread, precision, ulp):
    flat = segments_model(LENGTHS, spread)
    m, o = binding.exa_create(flat, precision, flags=binding.EXA_FLAG_NO_TUNE), oracle.Oracle(flat)
    rng = np.random.default_rng(5)
    x, v = rng.uniform(0.5, 1.5, flat.nvar), rng.uniform(0.5, 1.5, flat.nvar)
    y, w = rng.uniform(0.5, 1.5, flat.ncon), rng.uniform(0.5, 1.5, flat.ncon)
    X, V, Y, W = (torch.as_tensor(a, device="cuda") for a in (x, v, y, w))
    got = dict(g=m.grad(X), c=m.cons(X), jv=m.jprod(X, V), jtw=m.jtprod(X, W), hv=m.hprod(X, Y, 1.0, V))
    ref = dict(g=o.grad(x), c=o.cons(x), jv=o.jprod(x, v), jtw=o.jtprod(x, w), hv=o.hprod(x, y, 1.0, v))
    # positive terms of at most eight roundings each; two orders of an FP64 sum of n terms differ by at most 2 n ulp of it
    tol = 8 * ulp + 2 * 2 * (max(LENGTHS) + 4) * 2.0 ** -53
    for k, r in ref.items():
        assert np.all(np.abs(got[k].cpu().numpy() - r) <= tol * np.abs(r)), k
