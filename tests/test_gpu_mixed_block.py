"""Mixed-precision models keep 128 threads per CTA by default at every size (their FP32 roundings follow the
compiled kernel); small FP64 models take 64."""
import pytest

import synth
from paper_2608_16265_gb300 import binding as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,block", [(B.EXA_FP64, 64), (B.EXA_MIXED_FP32, 128)])
def test_default_block_of_small_models(precision, block):
    for flat in (synth.rosenbrock(300).flat, synth.acopf(60, 80, 9, seed=2).flat):
        assert B.exa_create(flat, precision).stat("eval_block") == block
