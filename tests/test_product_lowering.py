"""Product kernels of patterns whose expression graphs are compact but whose product trees are not."""
import numpy as np
import pytest

from paper_2608_16265_gb300 import binding
from paper_2608_16265_gb300.ir import Model, sin


def nested(kind):
    m = Model()
    x = m.add_var(8)
    if kind == "squares":
        def f(e):
            for _ in range(10):  # 1024 leaves
                e = (0.5 * e) ** 2
            return e
    elif kind == "powers":
        def f(e):
            return (e ** 64) ** 64 + (e ** -31) ** 2
    else:
        def f(e):
            for _ in range(3):
                e = e ** 2 * sin(e) + e
            return e
    m.add_obj(lambda d: f(x[d.k]), n=4)
    m.add_con(lambda d: f(x[d.k] * x[d.k + 1]) - x[d.k], n=4)
    return m.flat()


@pytest.mark.parametrize("kind", ["squares", "powers", "repeated"])
def test_compact_graphs_lower_quickly(kind):
    flat = nested(kind)
    assert sum(len(p.vop) for p in flat.patterns) < 2000
    binding.exa_compile_check(flat, block=64)
