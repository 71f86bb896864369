"""The direct-gradient branch is in the FP64 kernels only: mixed-precision kernels keep every gradient slot in
the slot buffer."""
import pytest

from paper_2608_16265_gb300 import binding
from paper_2608_16265_gb300.ir import Model


@pytest.mark.parametrize("precision", [binding.EXA_FP64, binding.EXA_MIXED_FP32])
def test_direct_gradient_branch(precision, tmp_path, monkeypatch):
    m = Model()
    x = m.add_var(6)
    m.add_obj(lambda d: x[d.k] ** 2 * x[d.k + 3], n=3)
    monkeypatch.setenv("EXA_DUMP_SOURCE", str(tmp_path / "s.cu"))
    binding.exa_compile_check(m.flat(), precision, block=64)
    assert ("pm.gsole >>" in (tmp_path / "s.cu").read_text()) == (precision == binding.EXA_FP64)
