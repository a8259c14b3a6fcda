"""Bounded waits of the attention stream, the tile encoder and the Hadamard encoder; attention in a graph.

As in test_gpu_wait_limit.py: with a limit of 100 ns the tile encoder's first waits (for the gauge's
conversion) cannot be met, so the call comes back with CG_FLAG_PIPE_TIMEOUT and without any fault, and
the next call, with the normal limit, gives the bytes that a call before gave. The Hadamard encoder
waits for one copy only, which may land between two ticks of the clock that the limit is read from, and
attention starts its copies well before it waits for them: these may not run out, and without the flag
the result has to be the right one. Shares that span several units and units of several parts. Its kernels are chained by programmatic launches, so a
captured call is replayed on other inputs and compared with a plain call.
"""
import numpy as np
import pytest

from paper_2607_20538_gb300 import synth

torch = pytest.importorskip("torch")
cg = pytest.importorskip("paper_2607_20538_gb300")

pytestmark = pytest.mark.gpu

ENV = "CODECGAUGE_PIPE_WAIT_NS"


def _timeout_then_same(call, outputs, monkeypatch, certain=True):
    cg.get_status()
    call()
    assert cg.get_status() == 0
    want = [o.clone() for o in outputs]
    monkeypatch.setenv(ENV, "100")
    call()
    expired = cg.get_status() & cg.CG_FLAG_PIPE_TIMEOUT
    assert expired or not certain
    assert expired or all(torch.equal(o, w) for o, w in zip(outputs, want))
    monkeypatch.delenv(ENV)
    for o in outputs:
        o.zero_()
    call()
    assert cg.get_status() == 0
    for o, w in zip(outputs, want):
        assert torch.equal(o, w)


def _cache(w):
    x = torch.from_numpy(np.ascontiguousarray(synth.kv_cache(w, threads=4)).reshape(-1).view(np.int16)).cuda()
    return x, torch.from_numpy(synth.gauges(w).reshape(-1)).cuda()


@pytest.mark.parametrize("hadamard", [False, True])
def test_encoders(hadamard, monkeypatch):
    w = synth.Workload("wait", L=2, B=2, H=2, T=1000, d=128, group=64, backend=0 if hadamard else 3, bits=4, block=64)
    shape, params = cg.Shape(**w.shape), cg.Params(**w.params)
    x, G = _cache(w)
    codes, scales, _ = cg.alloc_outputs(shape, params)
    call = (lambda: cg.encode_hadamard(shape, params, x, codes, scales)) if hadamard else (lambda: cg.encode(shape, params, x, G, codes, scales))
    _timeout_then_same(call, [codes, scales], monkeypatch, certain=not hadamard)


def _attention(bits, B, T, n_rep=4):
    w = synth.Workload("wait", L=1, B=B, H=4, T=T, d=128, group=64, backend=0, bits=bits, block=64)
    shape, params = cg.Shape(**w.shape), cg.Params(**w.params)
    x, G = _cache(w)
    codes, scales, _ = cg.alloc_outputs(shape, params)
    cg.encode(shape, params, x, G, codes, scales)
    q = torch.randn((1, B, 4, n_rep, 128), device="cuda", generator=torch.Generator("cuda").manual_seed(1)).bfloat16()
    out = torch.empty(q.shape, dtype=torch.float32, device="cuda")
    ws = torch.empty(cg.attention_workspace_bytes(shape, params, n_rep), dtype=torch.uint8, device="cuda")
    return q, out, lambda: cg.attention(shape, params, n_rep, 0.09, q, codes, scales, G, out, ws)


@pytest.mark.parametrize("bits,B,T", [(4, 130, 600), (8, 130, 300), (8, 2, 5000)])
def test_attention(bits, B, T, monkeypatch):
    _, out, call = _attention(bits, B, T)
    _timeout_then_same(call, [out], monkeypatch, certain=False)


@pytest.mark.parametrize("bits", [3, 4])
def test_attention_in_a_graph(bits):
    q, out, call = _attention(bits, 2, 3000)
    call()
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.stream(side):
        call()
        with torch.cuda.graph(graph, stream=side):
            call()
    torch.cuda.synchronize()
    q.copy_(q.flip(1))
    call()
    want = out.clone()
    out.zero_()
    graph.replay()
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(out, want)
