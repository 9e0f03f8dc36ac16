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


def _given_tokens(w, S0, Om, toks, q, dev_layer):
    """A flush of the given tokens [n][B, H, ..] (float64 arrays of stored values), the last one as the current token: S, U, o."""
    m, n = dev_layer, len(toks)
    m.state.copy_(torch.from_numpy(S0))
    dt = (torch.bfloat16, torch.bfloat16, torch.float32, torch.bfloat16)
    on = [[torch.from_numpy(x).to(m.device, d).contiguous() for x, d in zip(t, dt)] for t in toks]
    for t in range(n - 1):
        for view, x in zip(m.ring_views(), on[t]):
            view[:, :, t] = x
    o = m.new_output()
    m.state_update(n - 1, torch.from_numpy(q).to(m.device, torch.bfloat16), *on[-1], o)
    m.check_status()
    S, U, ref = orc.state_update(w.kind, S0.astype(np.float64), toks, np.broadcast_to(Om.astype(np.float64), (w.batch,) + Om.shape), q)
    return (m.state.cpu().numpy(), S), (m.sketch.cpu().numpy().transpose(0, 1, 3, 2), U), (o.cpu().numpy(), ref)


def _bf16(x):
    return torch.from_numpy(x).bfloat16().double().numpy()


def _norm_err(got, ref):
    return np.linalg.norm(got - ref) / np.linalg.norm(ref)


@pytest.mark.parametrize("n", [8, 16, 24, 32, 64])
@pytest.mark.parametrize("spread", [0.1, 0.0])
def test_keys_of_one_direction_and_slow_decays(n, spread):
    """Nearly equal (equal) keys, beta and decays near one: the system I + Bd A is as far from the identity as unit keys make it.
    2-norm, bar as above: each operand 2^-16, three products in a row."""
    w = synth.Workload("t", "kda", 6, 3, 128, 128, 16, 64, 0, "bf16", 613, basis="qr")
    m, S0, Om, _C, _ = make_layer(w)
    rng = np.random.default_rng(n)
    base = rng.standard_normal((w.batch, w.heads, 128))
    toks = []
    for _ in range(n):
        k = base + spread * rng.standard_normal(base.shape)
        toks.append((_bf16(k / np.linalg.norm(k, axis=-1, keepdims=True)), _bf16(rng.standard_normal(base.shape)),
                     (1 - 0.01 * rng.random(base.shape[:2])).astype(np.float32).astype(np.float64),
                     _bf16(1 - 2.0 ** -(4 + 4 * rng.random(base.shape)))))
    q = _bf16(base / np.linalg.norm(base, axis=-1, keepdims=True))
    for got, ref in _given_tokens(w, S0, Om, toks, q, m):
        assert _norm_err(got, ref) <= FP32_GUARD, n


def test_pair_sums_inside_sixteen_tokens_are_fp32():
    """Keys of one channel: a pair sum is a single product, so what its operands are held in shows in S_new.  From a zero state
    S_new = K~^T E with both factors as two bfloat16 halves (lo lo left out) and E = T V from an exact A is what the kernel may
    lose; with the pair sums of tokens 8..11 against 0..7 from halves as well the error would be 1.25 times that.  Bar: 1.1 times
    (fp32 sums: 2^-24 of 2^-17)."""
    w = synth.Workload("t", "kda", 64, 4, 128, 128, 16, 16, 0, "bf16", 617, basis="qr")
    m, S0, Om, _C, _ = make_layer(w)
    S0 = np.zeros_like(S0)
    rng, n, shape = np.random.default_rng(3), 12, (w.batch, w.heads, 128)
    ch, toks = 37, []
    for _ in range(n):
        k = np.zeros(shape)
        k[..., ch] = 0.5 + rng.random(shape[:2])
        toks.append((_bf16(k), _bf16(rng.standard_normal(shape)), (1 - 0.01 * rng.random(shape[:2])).astype(np.float32).astype(np.float64),
                     _bf16(1 - 2.0 ** -(4 + 4 * rng.random(shape)))))
    k, g = (np.stack([t[i][..., ch] for t in toks], -1) for i in (0, 3))
    v, beta = np.stack([t[1] for t in toks], -2), np.stack([t[2] for t in toks], -1)

    def halves(x):
        hi = _bf16(np.ascontiguousarray(x))
        return hi, _bf16(x - hi)

    def expected(split_pairs):
        prod = lambda a, b: np.prod(g[..., a:b], axis=-1)
        A = np.zeros(k.shape[:2] + (n, n))
        for s in range(n):
            for j in range(s):
                if split_pairs and s >= 8 > j:
                    (xh, xl), (yh, yl) = halves(k[..., s] * prod(8, s + 1)), halves(k[..., j] * prod(j + 1, 8))
                    A[..., s, j] = xh * yh + xl * yh + xh * yl
                else:
                    A[..., s, j] = k[..., s] * k[..., j] * prod(j + 1, s + 1)
        E = np.linalg.solve(np.eye(n) + beta[..., None] * A, beta[..., None] * v)
        (th, tl), (eh, el) = halves(np.stack([k[..., s] * prod(s + 1, n) for s in range(n)], -1)), halves(E)
        row = lambda t, e: np.einsum("bhs,bhsv->bhv", t, e)
        return row(th, eh) + row(tl, eh) + row(th, el)

    (S, ref), _, _ = _given_tokens(w, S0, Om, toks, np.zeros(shape), m)
    exact = ref[:, :, ch]
    kept = _norm_err(expected(False), exact)
    assert _norm_err(expected(True), exact) >= 1.2 * kept
    assert _norm_err(S[:, :, ch].astype(np.float64), exact) <= 1.1 * kept
