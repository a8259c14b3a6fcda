"""Edges of the streaming attention kernel (2-, 4- and 8-bit codes).

Token counts around its 32- and 64-token steps, shares that end inside a unit and units without a
whole step, one to eight queries, one, two and four blocks per row, value scales far below fp16's
normal range and value scales that grow by orders of magnitude inside a history (the weights' common
factor is chosen from the first tokens). Reference and tolerance as in test_gpu_attention.py: the
oracle's fp64 attention over its fp64 decode of the same bytes.
"""
import numpy as np
import pytest

import oracle
from paper_2607_20538_gb300 import synth

from test_gpu_attention import _run, _wl

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


def _check(w, n_rep, T, t0=0, scales=None):
    x = synth.kv_cache(w, threads=4)
    G = synth.gauges(w)
    ref = oracle.encode(w.shape, w.params, x, G)
    if scales is not None:
        ref["scales"] = scales(ref["scales"])
    q = synth.f32_to_bf16_bits(np.random.default_rng(5).normal(0.0, 1.0, (w.L, w.B, w.H, n_rep, w.d)).astype(np.float32))
    dc = torch.from_numpy(np.concatenate([ref["codes"], np.zeros(16, np.uint8)])).cuda()
    ds = torch.from_numpy(np.concatenate([ref["scales"], np.zeros(8, np.uint16)]).view(np.int16)).cuda()
    _run(w, n_rep, t0, T, dc, ds, ref["codes"], ref["scales"], G, q)


@pytest.mark.parametrize("T", [1, 31, 33, 63, 64, 65, 255, 257, 520])
@pytest.mark.parametrize("bits,block,n_rep", [(4, 64, 4), (8, 128, 1), (2, 32, 8)])
def test_token_counts(T, bits, block, n_rep):
    _check(_wl(T=T, bits=bits, block=block, group=32, L=1, B=2), n_rep, T)


@pytest.mark.parametrize("bits", [2, 4, 8])
@pytest.mark.parametrize("block", [32, 64, 128])
@pytest.mark.parametrize("n_rep", [2, 8])
def test_blocks_and_queries(bits, block, n_rep):
    _check(_wl(T=333, bits=bits, block=block, group=64, L=1, B=2), n_rep, 300, t0=17)


@pytest.mark.parametrize("backend,T", [(0, 300), (3, 1100)])
def test_more_units_than_shares(backend, T):
    """512 units: a CTA's share holds several units or parts of two."""
    _check(_wl(backend=backend, T=T, L=2, B=64, H=4, group=16), 4, T)


@pytest.mark.parametrize("first,later", [(2.0 ** -20, 2.0 ** -20), (2.0 ** -20, 4.0), (2.0 ** -9, 2.0 ** 4)])
@pytest.mark.parametrize("n_rep", [4, 8])
def test_value_scales(first, later, n_rep):
    w = _wl(T=700, L=1, B=1)

    def scales(s):
        s = s.view(np.float16).reshape(2, w.H, w.T, -1, 2).copy()
        f = np.full(w.T, later)
        f[:300] = first
        s[1] = (s[1].astype(np.float64) * f[None, :, None, None]).astype(np.float16)
        return s.reshape(-1).view(np.uint16)

    _check(w, n_rep, w.T, scales=scales)


@pytest.mark.parametrize("bits,n_rep", [(3, 1), (4, 2), (6, 4), (4, 8)])
@pytest.mark.parametrize("B,group", [(76, 128), (77, 128), (77, 8)])
def test_merge_widths(bits, n_rep, B, group):
    """304 units of several parts (two per SM: four slices merge a unit) and 308 (one slice)."""
    _check(_wl(T=290, bits=bits, group=group, L=1, B=B, H=4), n_rep, 290)
