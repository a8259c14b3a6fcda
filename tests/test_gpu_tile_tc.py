"""Block-uniform tiles on the tensor-core encoder (d = 128, at least 64 tokens a call).

The rotation runs on tensor cores with a bound on its error, and every scale, zero and code the
bound leaves open is recomputed in the library's fixed fp32 order, so the bytes must equal the
oracle's with no near-boundary allowance. Cases: the edges of the 128-token MMA tile and of the
16-token range, every bit width, one, two and four blocks a row, gauge groups 8..128, the inputs
aimed at the error bound, all-zero rows, and zeros that overflow fp16.
"""
import numpy as np
import pytest

import oracle
from paper_2607_20538_gb300 import synth

from test_gpu_adversarial import cancelling, mixed_magnitudes

torch = pytest.importorskip("torch")
cg = pytest.importorskip("paper_2607_20538_gb300")

pytestmark = pytest.mark.gpu


def _wl(T, bits, group, block, B=1):
    return synth.Workload("tile_tc", L=2, B=B, H=2, T=T, d=128, group=group, backend=3, bits=bits, block=block)


def _check(w, x, G, flags=0):
    shape, params = cg.Shape(**w.shape), cg.Params(**w.params)
    nc, ns, _ = cg.packed_bytes(shape, params)
    codes, scales, _ = cg.alloc_outputs(shape, params)
    cg.encode(shape, params, torch.from_numpy(np.ascontiguousarray(x).reshape(-1).view(np.int16)).cuda(),
              torch.from_numpy(np.ascontiguousarray(G).reshape(-1)).cuda(), codes, scales)
    assert cg.get_status() == flags
    ref = oracle.encode(w.shape, w.params, x, G)
    np.testing.assert_array_equal(scales.cpu().numpy().view(np.uint16)[: ns // 2], ref["scales"])
    np.testing.assert_array_equal(codes.cpu().numpy()[:nc], ref["codes"])


@pytest.mark.parametrize("T", [64, 65, 127, 128, 129, 143, 257])
@pytest.mark.parametrize("bits,group,block", [(4, 128, 128), (8, 32, 32), (3, 64, 64)])
def test_edges(T, bits, group, block):
    w = _wl(T, bits, group, block, B=3)
    _check(w, synth.kv_cache(w, threads=4), synth.gauges(w))


@pytest.mark.parametrize("bits", [2, 3, 4, 6, 8])
@pytest.mark.parametrize("group,block", [(8, 128), (16, 32), (128, 64)])
def test_widths(bits, group, block):
    w = _wl(200, bits, group, block)
    _check(w, synth.kv_cache(w, threads=4), synth.gauges(w))


@pytest.mark.parametrize("bits,group,block", [(2, 128, 128), (4, 128, 32), (8, 64, 64)])
@pytest.mark.parametrize("kind", ["mixed", "cancelling"])
def test_inputs_aimed_at_the_bound(bits, group, block, kind):
    w = _wl(256, bits, group, block)
    rng = np.random.default_rng(11)
    G = synth.gauges(w)
    _check(w, mixed_magnitudes(w, rng) if kind == "mixed" else cancelling(w, G, rng), G)


def test_zero_rows_and_overflow():
    w = _wl(160, 4, 32, 64)
    x = synth.bf16_bits_to_f32(synth.kv_cache(w, threads=4))
    x[..., 16:32, :] = 0.0       # a whole tile of zeros
    x[..., 40, :] = 0.0          # and one row inside a tile
    _check(w, synth.f32_to_bf16_bits(x), synth.gauges(w))
    x[..., 100, 5] = -7.0e4      # a zero below the fp16 range, the scale inside it
    _check(w, synth.f32_to_bf16_bits(x), synth.gauges(w, "identity"), flags=cg.CG_FLAG_FP16_OVERFLOW)
