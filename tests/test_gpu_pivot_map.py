"""The pivot form of the state-dependent map, a warp per head: ranks and state shapes around the sizes it works in (chunks of ranks,
four ranks at a time), warps that build several heads' maps in a row, per-head ranks and per-sequence phases in such a walk."""
import numpy as np
import pytest
import torch

from oracle import sketchssm_oracle as orc
from paper_2609_33051_b200 import synth
from tests import harness
from tests.test_gpu_coef_map import COEF_GUARD, check_coef
from tests.test_gpu_parity import make_layer, run_schedule

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rank,pivots", [(1, 4), (2, 4), (3, 2), (5, 1), (8, 4), (13, 3), (15, 4), (17, 4), (24, 4)])
@pytest.mark.parametrize("K,V", [(128, 64), (128, 80), (128, 128), (64, 64), (64, 128)])
def test_ranks_pivots_and_shapes(rank, pivots, K, V):
    w = synth.Workload("t", "mamba2", 3, 2, K, V, rank, 4, 0, "f32", 503, basis="qr")
    check_coef(run_schedule(w, w.buf_len + 1, max_heads=10**9, coef="pivot", pivots=pivots))


def _maps_match(m, w, Om, heads, rank_of):
    """The maps of the given (batch, head) pairs against the oracle's form for the state and the sketch that lie in memory."""
    S, U, C = (x.float().cpu().numpy().reshape(w.batch, w.heads, *s) for x, s in
               ((m.state, (w.dk, w.dv)), (m.sketch, (w.rank, w.dv)), (m.coef, (w.rank, w.dk))))
    for b, h in heads:
        g = rank_of(h)
        ref = orc.pivot_coefficient_map_from_sketch(S[b, h], U[b, h, :g].T, Om[h][:, :g], 0.1, 4)
        assert np.abs(C[b, h, :g] - ref).max() <= COEF_GUARD * np.abs(ref).max(), (b, h)


@pytest.mark.parametrize("kind,K,V,rank,ranks", [("mamba2", 64, 64, 9, False), ("gdn", 64, 128, 16, True), ("mamba2", 128, 64, 4, True),
                                                 ("gdn", 64, 128, 32, False), ("mamba2", 128, 80, 13, False)])
def test_a_warp_builds_the_maps_of_several_heads(kind, K, V, rank, ranks):
    w = synth.Workload("t", kind, 83, 48, K, V, rank, 4, 0, "bf16", 509, basis="qr")          # 3984 heads, 12 warps on 148 SMs
    m, S0, Om, _C, dev = make_layer(w, coef="pivot")
    table = np.array([[rank, 1, 0, rank - 1][h % 4] if ranks else rank for h in range(w.heads)], np.int32)
    if ranks:
        m.head_rank = torch.from_numpy(table).to(dev)
        m.bind()
    m.state_update(0)
    m.check_status()
    rng = np.random.default_rng(5)
    pairs = [(0, 0), (w.batch - 1, w.heads - 1)] + [(int(rng.integers(w.batch)), int(rng.integers(w.heads))) for _ in range(60)]
    _maps_match(m, w, Om, [(b, h) for b, h in pairs if table[h]], lambda h: int(table[h]))
    # one sequence in three flushes: the others' maps stay bit for bit
    before = m.coef.clone()
    phase = np.where(np.arange(w.batch) % 3 == 1, -1, 0).astype(np.int32)
    x = synth.step_inputs(w, 0, 0)
    tt = [synth.to_torch(x[n], io, dev) for n, io in (("q", w.io), ("k", w.io), ("v", w.io), ("beta", "f32"), ("decay", "f32"))]
    m.step_mixed(torch.from_numpy(phase).to(dev), *tt, m.new_output())
    m.check_status()
    kept = torch.from_numpy(phase >= 0).to(dev)
    view = lambda c: c.view(w.batch, -1)
    assert torch.equal(view(m.coef)[kept], view(before)[kept])
    assert not torch.equal(view(m.coef)[~kept], view(before)[~kept])
    _maps_match(m, w, Om, [(b, h) for b, h in pairs if table[h] and phase[b] < 0], lambda h: int(table[h]))


def test_zero_state_gives_a_zero_map():
    w = synth.Workload("t", "gdn", 2, 2, 128, 128, 16, 4, 0, "bf16", 521, basis="qr")
    m, *_ = make_layer(w, coef="pivot")
    m.state.zero_()
    m.coef.fill_(float("nan"))
    m.state_update(0)
    m.check_status()
    assert torch.equal(m.coef, torch.zeros_like(m.coef))


@pytest.mark.parametrize("V,rank", [(128, 16), (128, 25), (128, 32), (80, 28), (64, 24), (64, 28), (128, 33)])
def test_a_stored_map_does_not_depend_on_the_batch(V, rank):
    """The same sequences alone and among many: their maps bit for bit."""
    maps = []
    for batch in (2, 130):
        w = synth.Workload("t", "mamba2", batch, 3, 128, V, rank, 4, 0, "bf16", 523, basis="qr")
        m, _S0, _Om, _C, dev = make_layer(w, coef="pivot")
        gen = torch.Generator().manual_seed(7)
        m.state.copy_(torch.randn(130, 3, 128, V, generator=gen)[:batch] * 0.02)
        m.state_update(0)
        m.check_status()
        maps.append((m.sketch[:2].clone(), m.coef[:2].clone()))
    assert torch.equal(maps[0][0], maps[1][0]) and torch.equal(maps[0][1], maps[1][1])


@pytest.mark.parametrize("share", [1, 3, 16])
def test_mixed_steps_map_the_sequences_that_flush_and_no_others(share):
    """More heads than warps of the grid: a map for every head of the flushing sequences, the one its new state gives; the others stay."""
    w = synth.Workload("t", "mamba2", 331, 7, 128, 64, 16, 8, 0, "f32", 541, basis="qr")
    m, _S0, _Om, _C, dev = make_layer(w, coef="pivot")
    m.ring.zero_()
    m.state_update(0)
    before = torch.full_like(m.coef, 7.0)
    m.coef.copy_(before)
    phase = torch.full((331,), 2, dtype=torch.int32, device=dev)
    phase[::share] = -8
    tt = harness.token_tensors(w, synth.step_inputs(w, 0, 0), dev)
    m.step_mixed(phase, tt["q"], tt["k"], tt["v"], tt["beta"], tt["decay"], m.new_output())
    m.check_status()
    flushed = phase < 0
    got = m.coef.clone()
    assert torch.equal(got[~flushed], before[~flushed])
    m.state_update(0)                                   # sketch and maps from the states as they are
    m.check_status()
    assert harness.rel_err(got[flushed].cpu().numpy(), m.coef[flushed].cpu().numpy().astype(np.float64)) <= COEF_GUARD


@pytest.mark.parametrize("rank,pivots", [(20, 4), (21, 3)])
@pytest.mark.parametrize("K,V", [(128, 64), (128, 80), (128, 128), (64, 64), (64, 128)])
def test_rows_of_omega_four_ranks_ahead(rank, pivots, K, V):
    """An odd and an even number of steps of four ranks."""
    test_ranks_pivots_and_shapes(rank, pivots, K, V)
