"""A mixed-precision two-stage model is lowered as the same patterns over columns of their own: its FP32
roundings do not depend on which columns other patterns use."""
import numpy as np
import pytest

from paper_2608_16265_gb300 import binding
from paper_2608_16265_gb300.ir import TwoStageModel, cos, sin


def flows(scenarios=3):
    rng = np.random.default_rng(0)
    m = TwoStageModel(scenarios)
    va, vm = m.add_var(5, scenario=True), m.add_var(5, scenario=True)
    br = dict(f=np.array([0, 1, 2, 2], np.int32), t=np.array([1, 2, 3, 4], np.int32), g=rng.uniform(0.5, 2, 4),
              b=rng.uniform(-3, -1, 4))

    def th(d):
        return va[d.f, d.s] - va[d.t, d.s]

    m.add_obj(lambda d: d.g * vm[d.f, d.s] ** 2 * vm[d.t, d.s], data=br, scenario=True)
    blk = m.add_con(lambda d: vm[d.f, d.s] * vm[d.t, d.s] * (d.g * cos(th(d)) + d.b * sin(th(d))), data=br, scenario=True)
    m.add_con(lambda d: vm[d.f, d.s] * vm[d.t, d.s] * (d.b * cos(-th(d)) - d.g * sin(-th(d))), data=br, scenario=True)
    m.add_con_aug(blk, lambda d: (d.f, d.g * vm[d.t, d.s] ** 2), data=br, scenario=True)
    return m.flat()


@pytest.mark.parametrize("precision", [binding.EXA_FP64, binding.EXA_MIXED_FP32])
def test_source_of_shared_columns(precision, tmp_path, monkeypatch):
    def source(flat, name):
        monkeypatch.setenv("EXA_DUMP_SOURCE", str(tmp_path / name))
        binding.exa_compile_check(flat, precision, block=64)
        return (tmp_path / name).read_text()

    shared, own = flows(), flows()
    for p in own.patterns:
        p.fields = [f.copy() for f in p.fields]
    same = source(shared, "shared.cu") == source(own, "own.cu")
    assert same == (precision == binding.EXA_MIXED_FP32)  # FP64: shared columns fuse
