"""Both forms of the tensor-core encoders' exact step, on either side of the line between them.

Undecided ranges are found by masks in every lane where a CTA has few tiles (or where blocks of 32
channels lie under a 128-wide gauge) and by a search over the lanes elsewhere. Units of one tile, as
many as the line allows and one sequence more; a third of the tokens mix magnitudes, which widens
the error bound, so that ranges and codes are left undecided often. Compared with the oracle under
the rules of the other encode tests.
"""
import numpy as np
import pytest

from paper_2607_20538_gb300 import synth

torch = pytest.importorskip("torch")
cg = pytest.importorskip("paper_2607_20538_gb300")

from test_gpu_adversarial import _run, mixed_magnitudes

pytestmark = pytest.mark.gpu


def _inputs(w):
    x = synth.kv_cache(w, threads=4)
    x[..., 1::3, :] = mixed_magnitudes(w, np.random.default_rng(23))[..., 1::3, :]
    return x


@pytest.mark.parametrize("over", [0, 1])
@pytest.mark.parametrize("bits,group,block,per_sm", [(2, 16, 32, 4), (3, 64, 32, 4), (4, 32, 32, 4), (6, 32, 32, 4), (8, 64, 32, 4),
                                                     (4, 128, 64, 4), (8, 64, 64, 8), (8, 128, 128, 8), (8, 32, 128, 1)])
def test_rows(bits, group, block, per_sm, over):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    B = per_sm * sms // 8 + over  # 8 units a sequence
    w = synth.Workload("forms", L=1, B=B, H=4, T=70, d=128, group=group, backend=0, bits=bits, block=block, residual=0)
    _run(w, _inputs(w), synth.gauges(w))


@pytest.mark.parametrize("over", [0, 1])
@pytest.mark.parametrize("bits,group", [(2, 32), (3, 128), (4, 64), (6, 64), (8, 128)])
def test_keys(bits, group, over):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    w = synth.Workload("forms", L=1, B=sms + over, H=4, T=130, d=128, group=group, backend=1, bits=bits, block=128, residual=2)
    _run(w, _inputs(w), synth.gauges(w))
