"""The CUDA-core flush kernel where its blocking can go wrong: token counts around the eight replayed together (with and
without the current token), ranks around the eight projected together, every tile width, configurations with and without
room for the one-head-ahead stage, more heads than resident CTAs, and more sequences than are listed at a time.

Bar: fp32 sums of at most K + 64 terms on each side, 1e-5 of the largest element (the bar of the float32 workloads)."""
import numpy as np
import pytest
import torch

from oracle import sketchssm_oracle as orc
from paper_2609_33051_b200 import synth
from tests import harness
from tests.test_gpu_parity import make_layer

pytestmark = pytest.mark.gpu
BAR = 1e-5


def _flush(m, w, S0, Om, n, token, fill_seed=0):
    """Append n tokens, flush (with a current token if asked) and compare state, sketch and exact output."""
    dev = m.device
    m.state.copy_(torch.from_numpy(S0))
    xs = [synth.step_inputs(w, 0, fill_seed + t) for t in range(n + 1)]
    views = m.ring_views()
    m.ring.fill_(255)                                          # stale slots hold NaNs
    for t in range(n):
        tt = harness.token_tensors(w, xs[t], dev)
        for view, name in zip(views, ("k", "v", "beta", "decay")):
            view[:, :, t] = tt[name]
    toks = [tuple(x[f].astype(np.float64) for f in ("k", "v", "beta", "decay")) for x in xs]
    toks = toks if token else toks[:n]
    tt = harness.token_tensors(w, xs[n], dev)
    o = m.new_output().fill_(float("nan"))
    cur = (tt["k"], tt["v"], tt["beta"], tt["decay"]) if token else (None,) * 4
    m.state_update(n, tt["q"], *cur, o)
    m.check_status()
    S, U, ref = orc.state_update(w.kind, S0.astype(np.float64), toks, np.broadcast_to(Om.astype(np.float64), (w.batch,) + Om.shape),
                                 xs[n]["q"].astype(np.float64))
    assert harness.rel_err(m.state.cpu().numpy(), S) <= BAR
    assert harness.rel_err(m.sketch.cpu().numpy().transpose(0, 1, 3, 2), U) <= BAR
    assert harness.rel_err(o.cpu().numpy(), ref) <= BAR


@pytest.mark.parametrize("kind", synth.KINDS)
@pytest.mark.parametrize("K,V,rank,L,io", [(128, 128, 16, 20, "bf16"), (128, 64, 13, 20, "f32"), (128, 80, 5, 20, "bf16"),
                                           (64, 128, 32, 20, "f32"), (64, 64, 8, 20, "bf16"), (128, 128, 64, 64, "f32")])
def test_token_counts_ranks_and_tiles(kind, K, V, rank, L, io):
    w = synth.Workload("t", kind, 3, 2, K, V, rank, L, 0, io, 211, basis="qr")
    m, S0, Om, _C, _ = make_layer(w)
    m.tune("update_impl", 1)
    for n, token in [(0, False), (0, True), (1, False), (3, True), (4, True), (7, True), (8, False), (8, True), (15, True),
                     (L - 1, True), (L, False)]:
        _flush(m, w, S0, Om, n, token)


@pytest.mark.parametrize("kind", synth.KINDS)
def test_more_heads_than_resident_ctas(kind):
    """Persistent CTAs with several heads each, over head-index boundaries (the staged Omega changes)."""
    w = synth.Workload("t", kind, 241, 5, 64, 64, 8, 8, 0, "bf16", 223, basis="qr")
    m, S0, Om, _C, _ = make_layer(w)
    m.tune("update_impl", 1)
    _flush(m, w, S0, Om, 7, True)


@pytest.mark.parametrize("kind", ["mamba2", "kda"])
def test_mixed_step_over_many_sequences(kind):
    """2100 sequences (listed 1024 at a time), each flushing or not at a fill of its own, none in the last list."""
    w = synth.Workload("t", kind, 2100, 1, 64, 64, 8, 8, 0, "f32", 227, basis="qr")
    m, S0, Om, C, dev = make_layer(w)
    m.state_update(0)
    rng = np.random.default_rng(5)
    fill = rng.integers(0, w.buf_len - 1, w.batch)
    flush = rng.random(w.batch) < 0.3
    flush[2048:] = False
    xs = [synth.step_inputs(w, 0, t) for t in range(w.buf_len)]
    for view, name in zip(m.ring_views(), ("k", "v", "beta", "decay")):
        for t in range(w.buf_len):
            view[:, :, t] = harness.token_tensors(w, xs[t], dev)[name]
    x = synth.step_inputs(w, 0, 99)
    tt = harness.token_tensors(w, x, dev)
    phase = torch.from_numpy(np.where(flush, -fill - 1, fill).astype(np.int32)).to(dev)
    o = m.new_output()
    m.step_mixed(phase, tt["q"], tt["k"], tt["v"], tt["beta"], tt["decay"], o)
    m.check_status()
    S = S0.astype(np.float64)
    ref = np.empty((w.batch, w.heads, w.dv))
    Om64, C64 = Om.astype(np.float64), C.astype(np.float64)
    for n in range(w.buf_len - 1):
        for f in (False, True):
            b = np.nonzero((fill == n) & (flush == f))[0]
            toks = [tuple(y[g][b].astype(np.float64) for g in ("k", "v", "beta", "decay")) for y in xs[:n] + [x]]
            q, Omb = x["q"][b].astype(np.float64), np.broadcast_to(Om64, (len(b),) + Om64.shape)
            if f:
                S[b], _U, ref[b] = orc.state_update(kind, S[b], toks, Omb, q)
            else:
                ref[b] = orc.decode_step(kind, orc.sketch_of(S[b], Omb), np.broadcast_to(C64, (len(b),) + C64.shape), toks, q)
    assert harness.rel_err(o.cpu().numpy(), ref) <= BAR
    assert harness.rel_err(m.state.cpu().numpy(), S) <= BAR
    U = orc.sketch_of(S, np.broadcast_to(Om64, (w.batch,) + Om64.shape))
    assert harness.rel_err(m.sketch.cpu().numpy().transpose(0, 1, 3, 2), U) <= BAR


@pytest.mark.parametrize("impl", [4, 5], ids=["eight_tokens", "columns"])
@pytest.mark.parametrize("kind", ["gdn", "kda"])
@pytest.mark.parametrize("K,V,rank,L,io", [(128, 128, 16, 20, "bf16"), (128, 64, 13, 20, "f32"), (128, 80, 5, 20, "bf16"),
                                           (64, 128, 32, 20, "f32"), (64, 64, 8, 20, "bf16"), (128, 128, 64, 64, "f32"), (128, 80, 16, 64, "bf16")])
def test_both_delta_rule_kernels(kind, K, V, rank, L, io, impl):
    """The kernel that replays eight tokens together and the one that replays them singly, whichever the sizes would select."""
    w = synth.Workload("t", kind, 3, 2, K, V, rank, L, 0, io, 229, basis="qr")
    m, S0, Om, _C, _ = make_layer(w)
    m.tune("update_impl", impl)
    for n, token in [(0, False), (0, True), (3, True), (4, True), (7, True), (8, False), (8, True), (16, True), (L - 1, True), (L, False)]:
        _flush(m, w, S0, Om, n, token)


@pytest.mark.parametrize("kind,B,H,K,V,L", [("gdn", 37, 2, 128, 128, 8), ("gdn", 75, 2, 128, 128, 8), ("gdn", 37, 4, 128, 80, 8), ("gdn", 150, 1, 128, 64, 20),
                                            ("gdn", 300, 2, 64, 64, 36), ("gdn", 89, 5, 128, 128, 8), ("kda", 37, 4, 64, 64, 8), ("kda", 30, 5, 64, 64, 8)])
def test_either_side_of_the_rule_between_them(kind, B, H, K, V, L):
    w = synth.Workload("t", kind, B, H, K, V, 8, L, 0, "f32", 233, basis="qr")
    m, S0, Om, _C, _ = make_layer(w)
    _flush(m, w, S0, Om, L - 1, True)


@pytest.mark.parametrize("impl", [4, 5], ids=["eight_tokens", "columns"])
@pytest.mark.parametrize("kind", synth.KINDS)
@pytest.mark.parametrize("K,V,L,io", [(64, 64, 20, "f32"), (128, 128, 64, "f32"), (128, 80, 36, "bf16")])
def test_mixed_step_with_fills_around_the_chunks(kind, K, V, L, io, impl):
    """Windows of more tokens than a chunk: sequences flush and decode at fills on both sides of 16 and 32 in one call."""
    fills = [n for n in (0, 6, 7, 8, 14, 15, 16, 17, 18, 30, 31, 32, 33, 47, 48, 62, 63) if n < L]
    w = synth.Workload("t", kind, 2 * len(fills), 2, K, V, 8, L, 0, io, 239, basis="qr")
    m, S0, Om, C, dev = make_layer(w)
    m.tune("update_impl", impl)
    m.state_update(0)
    fill, flush = np.repeat(fills, 2), np.tile([True, False], len(fills))
    xs = [synth.step_inputs(w, 0, t) for t in range(L)]
    m.ring.fill_(255)                                          # stale slots hold NaNs
    for view, name in zip(m.ring_views(), ("k", "v", "beta", "decay")):
        for t in range(L):
            held = torch.from_numpy(np.nonzero(fill > t)[0]).to(dev)
            view[held, :, t] = harness.token_tensors(w, xs[t], dev)[name][held]
    x = synth.step_inputs(w, 0, 99)
    tt = harness.token_tensors(w, x, dev)
    o = m.new_output()
    m.step_mixed(torch.from_numpy(np.where(flush, -fill - 1, fill).astype(np.int32)).to(dev), *(tt[n] for n in ("q", "k", "v", "beta", "decay")), o)
    m.check_status()
    Om64, C64 = Om.astype(np.float64), C.astype(np.float64)
    S, ref = S0.astype(np.float64), np.empty((w.batch, w.heads, V))
    for b in range(w.batch):
        toks = [tuple(y[g][b].astype(np.float64) for g in ("k", "v", "beta", "decay")) for y in xs[:fill[b]] + [x]]
        q = x["q"][b].astype(np.float64)
        if flush[b]:
            S[b], _U, ref[b] = orc.state_update(kind, S[b], toks, Om64, q)
        else:
            ref[b] = orc.decode_step(kind, orc.sketch_of(S[b], Om64), C64, toks, q)
    assert harness.rel_err(o.cpu().numpy(), ref) <= BAR
    assert harness.rel_err(m.state.cpu().numpy(), S) <= BAR
    U = orc.sketch_of(S, np.broadcast_to(Om64, (w.batch,) + Om64.shape))
    assert harness.rel_err(m.sketch.cpu().numpy().transpose(0, 1, 3, 2), U) <= BAR


@pytest.mark.parametrize("kind,V,L", [("gdn", 128, 8), ("gdn", 80, 36), ("kda", 64, 8)])
def test_a_bfloat16_sketch_does_not_depend_on_the_batch(kind, V, L):
    """The rounded sketch (and the state) of a sequence is the same, bit for bit, in a batch of 3 and in one of 301."""
    got = []
    for B in (3, 301):
        w = synth.Workload("t", kind, 301, 2, 128, V, 16, L, 0, "f32", 241, basis="qr")
        m, *_ = make_layer(w.replace(batch=B), sketch="bf16")
        m.state.copy_(torch.from_numpy(synth.initial_state(w)[:B]))
        m.state_update(0)
        for t in range(L):
            tt = {n: x[:B].contiguous() for n, x in harness.token_tensors(w, synth.step_inputs(w, 0, t), m.device).items()}
            args = (tt["q"], tt["k"], tt["v"], tt["beta"], tt["decay"], m.new_output())
            (m.decode_step if t < L - 1 else m.state_update)(t, *args)
        m.check_status()
        got.append((m.sketch[:3].clone(), m.state[:3].clone()))
    assert torch.equal(got[0][0], got[1][0]) and torch.equal(got[0][1], got[1][1])
