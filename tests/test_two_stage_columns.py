"""Replicated data columns of a two-stage model: equal columns are one array, different ones are not."""
import numpy as np
import pytest

from paper_2608_16265_gb300.ir import TwoStageModel


@pytest.mark.parametrize("scenarios", [1, 3])
def test_equal_columns_are_shared(scenarios):
    m = TwoStageModel(scenarios)
    x = m.add_var(4, scenario=True)
    a = np.array([0.5, 1.5, -0.0])
    i = np.array([0, 2, 3], np.int32)
    m.add_con(lambda d: d.a * x[d.i, d.s], data=dict(a=a, i=i), scenario=True)
    m.add_con(lambda d: d.b + x[d.j, d.s], data=dict(b=a.copy(), j=i.tolist()), scenario=True)
    a[1] = 7.0  # the array has changed since: another column
    m.add_con(lambda d: d.a * x[d.i, d.s], data=dict(a=a, i=i), scenario=True)
    m.add_con(lambda d: d.z * x[d.i, d.s], data=dict(z=np.array([0.5, 1.5, 0.0]), i=i[:3]), scenario=True)
    p = m.flat().patterns

    def col(k, name):
        return p[k].fields[{0: ["a", "i", "s"], 1: ["b", "j", "s"], 2: ["a", "i", "s"], 3: ["z", "i", "s"]}[k].index(name)]

    assert col(1, "b") is col(0, "a") and col(1, "j") is col(0, "i") and col(1, "s") is col(0, "s")
    assert col(2, "a") is not col(0, "a") and col(2, "i") is col(0, "i")
    assert col(3, "z") is not col(0, "a")  # -0.0 and 0.0 are different values
    assert np.array_equal(col(0, "a"), np.tile([0.5, 1.5, -0.0], scenarios))
    assert np.array_equal(col(2, "a"), np.tile([0.5, 7.0, -0.0], scenarios))
    assert np.array_equal(col(0, "s"), np.repeat(np.arange(scenarios), 3))
