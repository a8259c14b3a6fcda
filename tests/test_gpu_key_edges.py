"""KIVI keys on the tensor-core encoder where its exact steps have the most to do.

Tokens that repeat two or three rows put all 128 values of a channel at its range's ends, so that
the list of exact recomputes fills many times over; a single repeated row gives channels of zero
range. Mixed magnitudes and cancelling rows widen the error bound, so that codes near a rounding
boundary are recomputed (a mask per lane at 6 and 8 bits, a search over the lanes below). Compared
with the oracle under the same rules as the other encode tests: scales, zeros and the window equal,
codes equal except where the oracle marks a value as lying at a rounding boundary.
"""
import numpy as np
import pytest

from paper_2607_20538_gb300 import synth

torch = pytest.importorskip("torch")
cg = pytest.importorskip("paper_2607_20538_gb300")

from test_gpu_adversarial import _run, cancelling, mixed_magnitudes

pytestmark = pytest.mark.gpu


def _wl(bits, group, T=300):
    return synth.Workload("key_edges", L=1, B=2, H=2, T=T, d=128, group=group, backend=1, bits=bits, block=128, residual=0)


@pytest.mark.parametrize("bits", [2, 3, 4, 6, 8])
@pytest.mark.parametrize("group", [32, 64, 128])
@pytest.mark.parametrize("kind", ["rows1", "rows2", "rows3", "mixed", "cancelling"])
def test_exact_steps(bits, group, kind):
    w = _wl(bits, group)
    rng = np.random.default_rng(17)
    G = synth.gauges(w)
    if kind == "mixed":
        x = mixed_magnitudes(w, rng)
    elif kind == "cancelling":
        x = cancelling(w, G, rng)
    else:
        x = synth.kv_cache(w, threads=4)
        x = np.ascontiguousarray(x[..., np.arange(w.T) % int(kind[4:]), :])
    _run(w, x, G)
