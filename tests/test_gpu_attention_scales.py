"""Attention over histories whose value scales change by orders of magnitude (2-, 4-, 8-bit codes).

The streaming kernel gives the weights p s_V of each step a power of two of their own before they
enter the tensor cores as fp16 pairs, so that small value scales keep their precision whatever other
tokens hold: a prefix without values (zero padding), with tiny ones, or scales that drift over the
history. 512 units, so that a warp streams through whole histories. Reference and tolerance as in
test_gpu_attention.py, relative to the largest value of a unit; queries of standard deviation 1 at 2
and 4 bits, the inputs that tolerance was derived for, and 2 at 8 bits, whose queries are not rounded.
Queries up to the largest bf16 values: the scores' differences decide, however large they are.
"""
import numpy as np
import pytest

import oracle
from paper_2607_20538_gb300 import synth

from test_gpu_attention import _run, _wl

torch = pytest.importorskip("torch")
cg = pytest.importorskip("paper_2607_20538_gb300")

pytestmark = pytest.mark.gpu

T = 1024
PREFIX = 256  # tokens: one step of every warp at 2 and 4 bits, two at 8


def _check(bits, n_rep, factors, block=64):
    w = _wl(L=1, B=64, H=8, T=T, bits=bits, block=block, group=16)
    rng = np.random.default_rng(bits)
    nc, ns, _ = cg.packed_bytes(cg.Shape(**w.shape), cg.Params(**w.params))
    qmax = (1 << bits) - 1
    s = rng.lognormal(0.0, 0.3, (2, w.B * w.H, T, 128 // block)) * 5.0 / qmax
    m = s * qmax * (rng.normal(0.0, 0.05, s.shape) - 0.5)
    sm = np.stack([s, m], -1)
    sm[1] *= factors[:, None, None]
    scales = sm.astype(np.float16).reshape(-1).view(np.uint16)
    codes = rng.integers(0, 256, nc, np.uint8)
    assert scales.size == ns // 2
    q = rng.normal(0.0, 2.0 if bits == 8 else 1.0, (w.L, w.B, w.H, n_rep, w.d)).astype(np.float32)
    _run(w, n_rep, 0, T, torch.from_numpy(codes).cuda(), torch.from_numpy(scales.view(np.int16)).cuda(), codes, scales,
         synth.gauges(w), synth.f32_to_bf16_bits(q))


@pytest.mark.parametrize("bits,n_rep,later", [(8, 4, 2.0 ** -7), (8, 8, 2.0 ** -12), (4, 4, 2.0 ** -12), (4, 8, 2.0 ** -14), (2, 1, 2.0 ** -14)])
@pytest.mark.parametrize("first", [0.0, 2.0 ** -22])
def test_small_scales_after_a_prefix(bits, n_rep, later, first):
    f = np.full(T, later)
    f[:PREFIX] = first
    _check(bits, n_rep, f)


@pytest.mark.parametrize("bits,block", [(8, 128), (4, 32), (2, 64)])
@pytest.mark.parametrize("grow", [False, True])
def test_scales_that_drift(bits, block, grow):
    """Fourteen octaves over the history."""
    f = 2.0 ** -np.floor(np.linspace(0.0, 14.99, T))
    _check(bits, 4, f[::-1] if grow else f, block)


@pytest.mark.parametrize("bits,n_rep,block", [(2, 8, 32), (4, 4, 64), (8, 1, 128), (8, 8, 64)])
@pytest.mark.parametrize("size", [1.0e7, 1.0e20, 1.0e37])
def test_large_queries(bits, n_rep, block, size):
    """Scores of any fp32 size: the largest takes all the weight."""
    w = _wl(L=1, B=2, H=2, T=300, bits=bits, block=block, group=32)
    ref = oracle.encode(w.shape, w.params, synth.kv_cache(w, threads=4), synth.gauges(w))
    q = size * np.random.default_rng(9).normal(0.0, 1.0, (w.L, w.B, w.H, n_rep, w.d))
    dc = torch.from_numpy(np.concatenate([ref["codes"], np.zeros(16, np.uint8)])).cuda()
    ds = torch.from_numpy(np.concatenate([ref["scales"], np.zeros(8, np.uint16)]).view(np.int16)).cuda()
    _run(w, n_rep, 0, w.T, dc, ds, ref["codes"], ref["scales"], synth.gauges(w), synth.f32_to_bf16_bits(q.astype(np.float32)))
