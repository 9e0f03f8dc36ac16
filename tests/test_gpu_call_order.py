"""Calls queued without synchronisation: the flush of a mixed step runs beside the decode kernel of the same step and releases
the next call before either is done, and the CUDA-core flushes are launched with dependent launch.  The same queue with
dependent launch off (every kernel waits for the one before), and replayed from a graph, gives the same bits."""
import numpy as np
import pytest
import torch

from paper_2609_33051_b200 import synth
from tests import harness
from tests.test_gpu_parity import make_layer

pytestmark = pytest.mark.gpu


def _layer(w, coef, impl, pdl):
    m, *_rest, dev = make_layer(w, coef=coef)
    m.tune("update_impl", impl)
    m.tune("pdl", pdl)
    m.state_update(0)
    return m, dev


def _tokens(w, dev):
    xs = [harness.token_tensors(w, synth.step_inputs(w, 0, t), dev) for t in range(w.buf_len)]
    return [tuple(x[n] for n in ("q", "k", "v", "beta", "decay")) for x in xs]


def _mixed_queue(w, dev, rounds):
    """Phases of `rounds` windows, every sequence at a fill of its own, and what the calls need: (phase, tokens) each."""
    toks, n, calls = _tokens(w, dev), np.arange(w.batch) % w.buf_len, []
    for t in range(rounds * w.buf_len):
        flush = n == w.buf_len - 1
        calls.append((torch.from_numpy(np.where(flush, -n - 1, n).astype(np.int32)).to(dev), toks[t % w.buf_len]))
        n = np.where(flush, 0, n + 1)
    return calls


def _fill(m, w, toks):
    """A ring that holds tokens in every slot (the sequences start in the middle of their windows)."""
    for view, at in zip(m.ring_views(), (1, 2, 3, 4)):
        for t in range(w.buf_len):
            view[:, :, t] = toks[t][at]
    m.bind()


def _result(m, outs):
    torch.cuda.synchronize()
    m.check_status()
    return [*(o.clone() for o in outs), m.state.clone(), m.sketch.clone(), m.coef.clone(), m.ring.clone()]


CASES = [(k, V, io, coef, impl) for k, V, io in (("mamba2", 64, "bf16"), ("gdn", 128, "bf16"), ("kda", 64, "f32")) for coef in (None, "pivot", "ridge")
         for impl in ((4,) if k == "mamba2" else (4, 5))]


@pytest.mark.parametrize("kind,V,io,coef,impl", CASES)
def test_queued_mixed_steps(kind, V, io, coef, impl):
    w = synth.Workload("t", kind, 96, 8, 128, V, 16, 8, 0, io, 431, basis="qr")
    got = []
    for pdl in (1, 0):
        m, dev = _layer(w, coef, impl, pdl)
        calls = _mixed_queue(w, dev, 3)
        _fill(m, w, _tokens(w, dev))
        outs = [m.new_output() for _ in range(len(calls) + 2)]
        torch.cuda.synchronize()
        for (phase, tok), o in zip(calls, outs):
            m.step_mixed(phase, *tok, o)
        # directly after a mixed step: a decode step over slots that it wrote, then a flush of them
        m.decode_step(3, *calls[3][1], outs[-2], flags=1)
        m.state_update(4, *calls[4][1], outs[-1])
        got.append(_result(m, outs))
    for a, b in zip(*got):
        assert torch.equal(a, b)
    assert all(bool(torch.isfinite(x.float()).all()) for x in got[0][:-1])


@pytest.mark.parametrize("kind,V,io,coef,impl", CASES)
def test_queued_windows_on_the_cuda_core_flush(kind, V, io, coef, impl):
    w = synth.Workload("t", kind, 96, 8, 128, V, 16, 8, 0, io, 433, basis="qr")
    got = []
    for pdl in (1, 0):
        m, dev = _layer(w, coef, impl, pdl)
        toks = _tokens(w, dev)
        outs = [m.new_output() for _ in range(3 * w.buf_len + 1)]
        torch.cuda.synchronize()
        for i, o in enumerate(outs[:-1]):
            t = i % w.buf_len
            (m.decode_step if t < w.buf_len - 1 else m.state_update)(t, *toks[t], o)
        m.decode_step(3, *toks[3], outs[-1], flags=1)          # directly after the flush, over slots that are still stored
        got.append(_result(m, outs))
    for a, b in zip(*got):
        assert torch.equal(a, b)


@pytest.mark.parametrize("kind,V,io,coef,impl", CASES)
def test_mixed_steps_replayed_from_a_graph(kind, V, io, coef, impl):
    w = synth.Workload("t", kind, 96, 8, 128, V, 16, 8, 0, io, 439, basis="qr")
    layers = [_layer(w, coef, impl, 1)[0] for _ in range(2)]
    dev = layers[0].device
    calls = _mixed_queue(w, dev, 1)
    outs = [[m.new_output() for _ in calls] for m in layers]
    toks = _tokens(w, dev)

    def queue(i):
        for (phase, tok), o in zip(calls, outs[i]):
            layers[i].step_mixed(phase, *tok, o)

    queue(1)                                                   # first-call set-up outside the capture, then restored
    torch.cuda.synchronize()
    eager, replayed = layers
    for name in ("state", "sketch", "coef"):
        getattr(replayed, name).copy_(getattr(eager, name))
    for m in layers:
        _fill(m, w, toks)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        queue(1)
    for _ in range(2):
        queue(0)
        graph.replay()
    for a, b in zip(_result(eager, outs[0]), _result(replayed, outs[1])):
        assert torch.equal(a, b)
