"""Encoders given NaN, Inf and huge values: what the rule says, in the blocks that hold them too.

The status bits report such inputs, but the call is accepted, so its bytes are those of the rule:
ranges pass over NaN (which never stands first in a block here, where the oracle's running minimum
would start from it), an infinite range has scale inf, and a value whose quotient is NaN codes to 0.
The tensor cores' sums cannot tell (Inf times a zero or a negative small term is NaN), so those
tokens have to take the exact path.
"""
import numpy as np
import pytest

import oracle
from paper_2607_20538_gb300 import synth

from cgcheck import compare_codes

torch = pytest.importorskip("torch")
cg = pytest.importorskip("paper_2607_20538_gb300")

pytestmark = pytest.mark.gpu

VALUES = [float("nan"), float("inf"), float("-inf"), 3.0e38]


def _encode(w, value, places, gauge="random"):
    """Codes, scales and flags of a cache with `value` at the given (unit, token, channel), and the oracle's."""
    v = synth.bf16_bits_to_f32(synth.kv_cache(w, threads=4)).copy()
    for u, t, c in places:
        v.reshape(-1, w.T, w.d)[u, t, c] = value
    x = np.where(np.isnan(v), np.uint16(0x7FC0), synth.f32_to_bf16_bits(v).reshape(v.shape))
    G = synth.gauges(w, gauge)
    shape, params = cg.Shape(**w.shape), cg.Params(**w.params)
    nc, ns, _ = cg.packed_bytes(shape, params)
    codes, scales, resid = cg.alloc_outputs(shape, params)
    dx = torch.from_numpy(np.ascontiguousarray(x).reshape(-1).view(np.int16)).cuda()
    cg.get_status()
    if gauge == "hadamard":
        cg.encode_hadamard(shape, params, dx, codes, scales)
    else:
        cg.encode(shape, params, dx, torch.from_numpy(np.ascontiguousarray(G).reshape(-1)).cuda(), codes, scales, resid)
    flags = cg.get_status()
    assert bool(flags & cg.CG_FLAG_NONFINITE_INPUT) == (not np.isfinite(value))
    assert not flags & cg.CG_FLAG_PIPE_TIMEOUT
    with np.errstate(all="ignore"):
        ref = oracle.encode(w.shape, w.params, x, G, want_flags=True)
    return codes.cpu().numpy().view(np.uint8)[:nc], scales.cpu().numpy().view(np.float16)[: ns // 2], ref


def _wl(backend, T, bits, group, block):
    return synth.Workload("nonfinite", L=1, B=2, H=2, T=T, d=128, group=group, backend=backend, bits=bits, block=block, residual=0)


@pytest.mark.parametrize("value", VALUES)
@pytest.mark.parametrize("bits,group,block", [(4, 128, 128), (4, 8, 128), (3, 16, 32), (2, 32, 64), (8, 64, 32)])
def test_tiles(value, bits, group, block):
    w = _wl(3, 200, bits, group, block)
    places = [(0, 3, 5), (1, 199, 127), (2, 17, 40), (3, 100, 1)] + [(5, t, 66) for t in range(33, 48)] + [(6, 64 + t, 9 * t) for t in range(1, 14)]
    codes, scales, ref = _encode(w, value, places)
    np.testing.assert_array_equal(scales, ref["scales"].view(np.float16))
    np.testing.assert_array_equal(codes, ref["codes"])


@pytest.mark.parametrize("value", VALUES[:3])
@pytest.mark.parametrize("bits,group,block", [(8, 64, 32), (8, 128, 128), (8, 32, 32), (4, 128, 64), (3, 32, 32)])
def test_row_codes_of_blocks_without_a_scale(value, bits, group, block):
    """A row's block that holds no finite range codes to 0; its neighbours keep their codes."""
    w = _wl(0, 200, bits, group, block)
    places = [(0, 3, 5), (1, 199, 127), (2, 17, 40), (3, 100, 0), (5, 64, 66)]
    codes, scales, ref = _encode(w, value, places)
    q = lambda b: np.unpackbits(b.reshape(-1, w.T, 128 * bits // 8), axis=-1, bitorder="little").reshape(-1, w.T, 128, bits)
    got, want = q(codes), q(ref["codes"])
    for u, t, c in places:  # blocks that share channels with the value's gauge group
        r = np.arange(128) // group == c // group
        own = np.repeat(r.reshape(-1, block).any(1), block)
        assert not got[u, t, own].any()
        got[u, t], want[u, t] = 0, 0
    flagged = ref["flags"].reshape(got.shape[:3]).astype(bool)
    assert flagged[(got != want).any(-1)].all()


@pytest.mark.parametrize("value", VALUES)
@pytest.mark.parametrize("bits,group", [(2, 32), (4, 128), (3, 64), (8, 64), (6, 32)])
def test_keys(value, bits, group):
    w = _wl(1, 256, bits, group, 128)
    places = [(0, 3, 5), (1, 127, 127), (2, 130, 40), (2, 255, 0), (3, 200, 64)]  # units 0..3 hold the keys
    codes, scales, ref = _encode(w, value, places)
    np.testing.assert_array_equal(scales, ref["scales"].view(np.float16))
    compare_codes(w, codes, ref["codes"], ref["flags"])


@pytest.mark.parametrize("value", VALUES)
@pytest.mark.parametrize("bits,group,block", [(4, 8, 128), (3, 16, 32), (2, 32, 64), (3, 8, 32), (8, 16, 128)])
def test_hadamard(value, bits, group, block):
    """A group without a finite value inside a block of finite ones, which set its range."""
    w = _wl(0, 40, bits, group, block)
    places = [(0, 3, group + 2), (1, 39, 127), (2, 17, 128 - block + group), (5, 21, 2 * group - 1)]
    codes, scales, ref = _encode(w, value, places, "hadamard")
    np.testing.assert_array_equal(scales, ref["scales"].view(np.float16))
    np.testing.assert_array_equal(codes, ref["codes"])
