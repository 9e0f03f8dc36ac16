"""The tensor-core flush of the per-channel decays where its blocking can go wrong: token counts around the blocks of 8, 16 and 32 and
the passes of 32 (with and without the current token, stale ring rows full of NaNs), ranks around eight and sixteen, CTAs that walk
one, two and several tiles over head-index boundaries.

Bar: every operand of a product is two bfloat16 halves, 2^-16 of it, and the products of a flush follow one another three times
(P, E, S_new): 5e-5 of the largest element, as for the other tensor-core flushes."""
import numpy as np
import pytest
import torch

from oracle import sketchssm_oracle as orc
from paper_2609_33051_b200 import synth
from tests import harness
from tests.test_gpu_parity import FP32_GUARD, make_layer

pytestmark = pytest.mark.gpu


def _flush(m, w, S0, Om, n, token):
    dev = m.device
    m.state.copy_(torch.from_numpy(S0))
    xs = [synth.step_inputs(w, 0, t) for t in range(n + 1)]
    views = m.ring_views()
    m.ring.fill_(255)
    for t in range(n):
        tt = harness.token_tensors(w, xs[t], dev)
        for view, name in zip(views, ("k", "v", "beta", "decay")):
            view[:, :, t] = tt[name]
    toks = [tuple(x[f].astype(np.float64) for f in ("k", "v", "beta", "decay")) for x in xs[:n + 1 if token else n]]
    tt = harness.token_tensors(w, xs[n], dev)
    o = m.new_output().fill_(float("nan"))
    cur = (tt["k"], tt["v"], tt["beta"], tt["decay"]) if token else (None,) * 4
    m.state_update(n, tt["q"], *cur, o)
    m.check_status()
    S, U, ref = orc.state_update(w.kind, S0.astype(np.float64), toks, np.broadcast_to(Om.astype(np.float64), (w.batch,) + Om.shape),
                                 xs[n]["q"].astype(np.float64))
    assert harness.rel_err(m.state.cpu().numpy(), S) <= FP32_GUARD, (n, token)
    assert harness.rel_err(m.sketch.cpu().numpy().transpose(0, 1, 3, 2), U) <= FP32_GUARD, (n, token)
    assert harness.rel_err(o.cpu().numpy(), ref) <= FP32_GUARD, (n, token)


@pytest.mark.parametrize("rank", [1, 8, 9, 13, 16])
def test_token_counts_and_ranks(rank):
    w = synth.Workload("t", "kda", 3, 2, 128, 128, rank, 64, 0, "bf16", 601, basis="qr")
    m, S0, Om, _C, _ = make_layer(w)
    for n, token in [(0, True), (1, False), (6, True), (7, True), (8, False), (8, True), (15, True), (16, False), (16, True), (23, True),
                     (24, True), (30, True), (31, True), (32, False), (32, True), (40, True), (55, True), (63, True)]:
        _flush(m, w, S0, Om, n, token)


@pytest.mark.parametrize("batch,heads", [(71, 2), (149, 1), (83, 2), (157, 3)])
def test_ctas_with_several_tiles(batch, heads):
    w = synth.Workload("t", "kda", batch, heads, 128, 128, 16, 32, 0, "bf16", 607, basis="qr")
    m, S0, Om, _C, _ = make_layer(w)
    for n, token in [(31, True), (9, True), (20, False)]:
        _flush(m, w, S0, Om, n, token)
