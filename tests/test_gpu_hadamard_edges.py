"""Edges of the Hadamard transform kernels: 32 lane rows a tile, d / 32 lanes a row.

Row counts around the tile for every head dim, blocks inside a lane (8, 16), of one lane and over
several lanes, every width, non-finite and overflowing inputs. Bytes equal the oracle's given the
fp32 Hadamard gauge tensor; the decode is held to the tight bound.
"""
import numpy as np
import pytest

import oracle
from paper_2607_20538_gb300 import synth

from cgcheck import compare_decode

torch = pytest.importorskip("torch")
cg = pytest.importorskip("paper_2607_20538_gb300")

pytestmark = pytest.mark.gpu


def _check(d, T, bits, group, block, change=None, flags=0, L=1, B=1, H=2):
    w = synth.Workload("had", L=L, B=B, H=H, T=T, d=d, group=group, backend=0, bits=bits, block=block)
    x = synth.kv_cache(w, threads=4)
    if change is not None:
        v = synth.bf16_bits_to_f32(x)
        change(v)
        x = synth.f32_to_bf16_bits(v)
    G = synth.gauges(w, "hadamard")
    shape, params = cg.Shape(**w.shape), cg.Params(**w.params)
    nc, ns, _ = cg.packed_bytes(shape, params)
    codes, scales, _ = cg.alloc_outputs(shape, params)
    cg.encode_hadamard(shape, params, torch.from_numpy(x.reshape(-1).view(np.int16)).cuda(), codes, scales)
    assert cg.get_status() == flags
    ref = oracle.encode(w.shape, w.params, x, G)
    np.testing.assert_array_equal(scales.cpu().numpy().view(np.uint16)[: ns // 2].view(np.float16).astype(np.float32),
                                  ref["scales"].view(np.float16).astype(np.float32))
    np.testing.assert_array_equal(codes.cpu().numpy()[:nc], ref["codes"])
    if flags:
        return
    out = torch.full((x.size + 4096,), 77, dtype=torch.int16, device="cuda")
    cg.decode_hadamard(shape, params, codes, scales, out)
    assert (out[x.size:] == 77).all()  # a ragged last tile writes its rows only
    xr = oracle.decode(w.shape, w.params, ref["codes"], ref["scales"], None, G)
    st = compare_decode(w, out.cpu().numpy().view(np.uint16)[: x.size], xr, G, None, codes=ref["codes"], scales_u16=ref["scales"])
    assert st["tight"] == xr.size


@pytest.mark.parametrize("d", [32, 64, 128, 256])
@pytest.mark.parametrize("T", [1, 3, 8, 31, 33])
def test_rows(d, T):
    _check(d, T, 4, 32, 32)


@pytest.mark.parametrize("bits", [2, 3, 4, 6, 8])
@pytest.mark.parametrize("block", [8, 16, 32, 128])
def test_blocks(bits, block):
    _check(128, 70, bits, 128, block)


@pytest.mark.parametrize("group", [8, 16, 32, 64, 128])
def test_groups(group):
    _check(256, 40, 3, group, 256, B=2)


def test_many_tiles():
    _check(128, 3000, 8, 64, 64, L=2, H=4)


def test_zero_rows_and_overflow():
    def zeros(v):
        v[..., 5, :] = 0.0

    def low(v):
        v[..., 5, :] = 0.0
        v[..., 9, :] = 0.0
        v[..., 9, 0] = -4.0e5  # values -+ 1e5 under g = 16: a zero below fp16, a scale inside

    _check(128, 20, 4, 16, 32, change=zeros)
    _check(128, 20, 4, 16, 32, change=low, flags=cg.CG_FLAG_FP16_OVERFLOW)


@pytest.mark.parametrize("value", [float("nan"), float("inf")])
@pytest.mark.parametrize("group", [8, 128])
@pytest.mark.parametrize("channel", [0, 45, 127])
def test_nonfinite_input_is_flagged(value, group, channel):
    x = torch.zeros((1, 2, 1, 1, 40, 128), dtype=torch.bfloat16, device="cuda")
    x[0, 1, 0, 0, 37, channel] = value
    shape, params = cg.Shape(L=1, B=1, H=1, T=40, d=128), cg.Params(0, group, 4, 128)
    codes, scales, _ = cg.alloc_outputs(shape, params)
    cg.get_status()
    cg.encode_hadamard(shape, params, x, codes, scales)
    assert cg.get_status() & cg.CG_FLAG_NONFINITE_INPUT
    x.zero_()
    cg.encode_hadamard(shape, params, x, codes, scales)
    assert cg.get_status() == 0
