"""Edges of the CUDA-core row kernels (exact rotation; shapes the tensor-core kernels do not take).

A warp takes four token rows (eight at d = 32) at a time and walks them linearly where they are
tokens of one sequence or one token of consecutive sequences, row by row elsewhere; a lane's packed
codes are joined into words across lanes. Cases: remainders of the row group, rows that change the
sequence inside a group, one token a sequence, every width at every head dim (two words a lane at
d = 256), shares of several CTAs, non-finite quotients. Codes and scales equal the oracle's bit for
bit; the decode is held to the tight bound of cgcheck.
"""
import numpy as np
import pytest

import oracle
from paper_2607_20538_gb300 import synth

from cgcheck import compare_decode

torch = pytest.importorskip("torch")
cg = pytest.importorskip("paper_2607_20538_gb300")

pytestmark = pytest.mark.gpu


def _check(d, T, B, bits, group, block, backend=0, L=1, H=2, x=None, kind="random", flags=0):
    w = synth.Workload("rows", L=L, B=B, H=H, T=T, d=d, group=group, backend=backend, bits=bits, block=block)
    x = synth.kv_cache(w, threads=4) if x is None else x(w)
    G = synth.gauges(w, kind)
    shape, params = cg.Shape(**w.shape), cg.Params(**w.params)
    nc, ns, _ = cg.packed_bytes(shape, params)
    codes, scales, _ = cg.alloc_outputs(shape, params)
    dG = torch.from_numpy(G.reshape(-1)).cuda()
    cg.encode(shape, params, torch.from_numpy(x.reshape(-1).view(np.int16)).cuda(), dG, codes, scales)
    assert cg.get_status() == flags
    ref = oracle.encode(w.shape, w.params, x, G)
    np.testing.assert_array_equal(scales.cpu().numpy().view(np.uint16)[: ns // 2], ref["scales"])
    np.testing.assert_array_equal(codes.cpu().numpy()[:nc], ref["codes"])
    if flags:
        return
    out = torch.full((x.size,), -1, dtype=torch.int16, device="cuda")
    cg.decode(shape, params, codes, scales, None, dG, out)
    xr = oracle.decode(w.shape, w.params, ref["codes"], ref["scales"], None, G)
    st = compare_decode(w, out.cpu().numpy().view(np.uint16), xr, G, None, codes=ref["codes"], scales_u16=ref["scales"])
    assert st["tight"] == xr.size


@pytest.mark.parametrize("d", [32, 64, 128, 256])
@pytest.mark.parametrize("bits", [2, 3, 4, 6, 8])
def test_widths(d, bits):
    _check(d, 37, 2, bits, min(d, 64), 32)


@pytest.mark.parametrize("T,B", [(1, 1), (1, 5), (1, 64), (2, 3), (3, 5), (5, 7), (63, 2)])
@pytest.mark.parametrize("d", [32, 128, 256])
def test_row_groups(T, B, d):
    _check(d, T, B, 3, 32, 16)


@pytest.mark.parametrize("group", [8, 16, 32, 64, 128])
def test_groups(group):
    _check(256, 50, 1, 4, group, 256)
    _check(128, 50, 1, 4, group, 8)


def test_many_rows_per_cta():
    _check(64, 4100, 1, 4, 16, 64, L=2, H=4)


@pytest.mark.parametrize("T", [1, 15, 47])
def test_tiles_decode_by_rows(T):
    _check(64, T, 3, 4, 16, 32, backend=3)


def test_overflowing_zero():
    def x(w):
        v = synth.bf16_bits_to_f32(synth.kv_cache(w, threads=4))
        v[..., 3, 7] = -7.0e4  # a zero below the fp16 range, the scale inside it
        v[..., 9, :] = 0.0
        return synth.f32_to_bf16_bits(v)

    _check(64, 20, 1, 4, 32, 32, x=x, kind="identity", flags=cg.CG_FLAG_FP16_OVERFLOW)
