"""What the mixed-precision kernels leave out that FP64 kernels have: anything that, without touching the
arithmetic, makes the compiler fuse other FP32 multiplies and adds."""
import pytest

from paper_2608_16265_gb300 import binding
from paper_2608_16265_gb300.ir import Model, sin


@pytest.fixture(params=[binding.EXA_FP64, binding.EXA_MIXED_FP32], ids=["fp64", "mixed"])
def generated(request, tmp_path, monkeypatch):
    m = Model()
    x = m.add_var(6)
    m.add_obj(lambda d: x[d.k] ** 2 * x[d.k + 3], n=3)
    m.add_con(lambda d: sin(x[d.k]) * x[d.k + 3], n=3)
    monkeypatch.setenv("EXA_DUMP_SOURCE", str(tmp_path / "s.cu"))
    binding.exa_compile_check(m.flat(), request.param, block=64)
    return request.param == binding.EXA_FP64, (tmp_path / "s.cu").read_text()


def test_direct_gradient_branch(generated):
    fp64, src = generated
    assert ("pm.gsole >>" in src) == fp64


def test_programmatic_launch(generated):
    fp64, src = generated
    assert ("griddepcontrol.wait" in src) == fp64 and ("griddepcontrol.launch_dependents" in src) == fp64


def test_arrays_of_compressed_sums(generated):
    fp64, src = generated
    assert ("if (act && o.hcomp)" in src) == fp64
