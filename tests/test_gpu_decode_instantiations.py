"""The decode kernel's instantiations for rank 16 with 128 state rows and bfloat16 I/O (mixed steps, state-dependent maps, erase
vectors) against its general one, which a rank table that gives every head the full rank selects: same inputs, two windows.

Bar: both sum at most L + rank + K products in fp32 in different orders, 2e-5 of the largest output; with bfloat16 storage an
erase vector or an element of the next window's sketch may round to the other side, 2^-8 of it."""
import numpy as np
import pytest
import torch

from paper_2609_33051_b200 import synth
from tests import harness
from tests.test_gpu_parity import make_layer, run_schedule

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", synth.KINDS)
@pytest.mark.parametrize("V", [64, 128])
@pytest.mark.parametrize("coef,sketch,erase,mixed", [(None, "f32", False, True), ("pivot", "f32", False, False), ("pivot", "bf16", False, False),
                                                     ("pivot", "bf16", False, True), (None, "f32", True, False), ("pivot", "bf16", True, False)])
def test_specialised_and_general_decode_agree(kind, V, coef, sketch, erase, mixed):
    if erase and kind == "mamba2":
        pytest.skip("no erase term")
    w = synth.Workload("t", kind, 21, 3, 128, V, 16, 8, 0, "bf16", 401, basis="qr")
    outs = []
    fill = np.arange(w.batch) % w.buf_len if mixed else np.zeros(w.batch, np.int64)
    for table in (False, True):
        m, *_rest, dev = make_layer(w, coef=coef, sketch=sketch, erase=erase)
        if table:
            m.head_rank = torch.full((w.heads,), 16, dtype=torch.int32, device=dev)
            m.bind()
        m.state_update(0)
        got, o = [], m.new_output()
        n = np.zeros(w.batch, np.int64)
        for t in range(2 * w.buf_len):
            tt = harness.token_tensors(w, synth.step_inputs(w, 0, t), dev)
            args = (tt["q"], tt["k"], tt["v"], tt["beta"], tt["decay"], o)
            if mixed:
                flush = (n == w.buf_len - 1) | ((n == fill) & (t < w.buf_len))
                m.step_mixed(torch.from_numpy(np.where(flush, -n - 1, n).astype(np.int32)).to(dev), *args)
                n = np.where(flush, 0, n + 1)
            elif t % w.buf_len < w.buf_len - 1:
                m.decode_step(t % w.buf_len, *args)
            else:
                m.state_update(t % w.buf_len, *args)
            got.append(o.cpu().numpy().copy())
        m.check_status()
        outs.append(np.stack(got))
    assert np.all(np.isfinite(outs[0]))
    assert harness.rel_err(outs[0], outs[1].astype(np.float64)) <= (2.0 ** -8 if sketch == "bf16" else 2e-5)


@pytest.mark.parametrize("K,V", [(128, 64), (128, 80), (128, 128), (64, 64), (64, 128)])
@pytest.mark.parametrize("rank", [8, 13, 24, 32, 48])
@pytest.mark.parametrize("io", ["bf16", "f32"])
def test_bfloat16_sketch_with_the_fixed_map_at_every_ring_fill(K, V, rank, io):
    """Mamba-2 with a bfloat16 sketch runs the general kernel for every rank but 16; the CTA size that is chosen grows with the
    ring fill and must stay within that kernel's launch bound.  A whole window; bars of the bfloat16 sketch test."""
    w = synth.Workload("t", "mamba2", 3, 2, K, V, rank, 32, 0, io, 409, basis="qr")
    errs = run_schedule(w, w.buf_len + 1, max_heads=10**9, sketch="bf16")
    assert errs["out"] <= 2e-3 + 2.0 ** -9, errs
    assert errs["S"] <= 5e-5 and errs["U"] <= 2.0 ** -7, errs


@pytest.mark.parametrize("kind,batch,heads,K,V,rank,L,io,full,ranks", [
    # full reads: four warps a head (few heads; long rings), two (the state larger than what stays in L2), odd head counts
    ("kda", 5, 7, 128, 128, 8, 8, "f32", True, False), ("gdn", 45, 37, 128, 128, 8, 12, "bf16", True, False),
    ("mamba2", 3, 1, 64, 64, 8, 20, "bf16", True, False), ("mamba2", 99, 37, 128, 64, 8, 8, "f32", True, False),
    ("mamba2", 67, 7, 128, 80, 8, 64, "bf16", True, False), ("kda", 53, 9, 64, 128, 8, 32, "bf16", True, False),
    # a dense head among sketched ones: four warps a head, two
    ("mamba2", 11, 6, 128, 80, 13, 12, "bf16", False, True), ("mamba2", 151, 7, 128, 64, 24, 8, "f32", False, True),
    ("gdn", 9, 5, 128, 128, 16, 8, "bf16", False, True), ("kda", 171, 6, 64, 64, 9, 12, "bf16", False, True),
    # long rings and large ranks: two warps a head, then four as the ring fills
    ("mamba2", 37, 9, 128, 64, 32, 64, "bf16", False, False), ("mamba2", 37, 9, 128, 128, 16, 64, "bf16", False, False),
    ("mamba2", 31, 9, 128, 80, 21, 64, "f32", False, False), ("mamba2", 31, 9, 64, 128, 45, 64, "f32", False, False)])
def test_teams_of_warps_and_single_warps_agree(kind, batch, heads, K, V, rank, L, io, full, ranks):
    """Several warps per head against one (a caller's limit on the warps selects that): the same windows, the rings bit for bit."""
    w = synth.Workload("t", kind, batch, heads, K, V, rank, L, 0, io, 421, basis="qr")
    outs, rings = [], []
    for single in (False, True):
        m, *_rest, dev = make_layer(w)
        if ranks:
            m.head_rank = torch.tensor([[rank, 0, 1, (rank + 1) // 2, rank][h % 5] for h in range(heads)], dtype=torch.int32, device=dev)
            m.bind()
        m.ring.zero_()
        m.bind()
        m.state_update(0)
        if single:
            m.tune("decode_max_warps_per_sm", 32)
        got = []
        for t in range(L - 1):
            tt = harness.token_tensors(w, synth.step_inputs(w, 0, t), dev)
            call = m.full_read_decode if full else m.decode_step
            got.append(call(t, tt["q"], tt["k"], tt["v"], tt["beta"], tt["decay"], m.new_output()).cpu().numpy())
        m.check_status()
        outs.append(np.stack(got))
        rings.append(m.ring.cpu().numpy().copy())
    assert np.all(np.isfinite(outs[1]))
    for a, b in zip(*outs):
        assert harness.rel_err(a, b.astype(np.float64)) <= 2e-5
    assert np.array_equal(*rings)


@pytest.mark.parametrize("call", ["decode_step", "full_read_decode"])
def test_a_callers_warp_count_is_taken_up_to_eight_and_refused_above(call):
    from paper_2609_33051_b200.binding import SketchSSMError
    w = synth.Workload("t", "mamba2", 4, 2, 128, 64, 16, 8, 0, "bf16", 419, basis="qr")
    m, *_rest, dev = make_layer(w)
    m.state_update(0)
    tt = harness.token_tensors(w, synth.step_inputs(w, 0, 0), dev)
    args, outs = (tt["q"], tt["k"], tt["v"], tt["beta"], tt["decay"]), []
    for nw in (1, 8):
        m.tune("decode_warps_per_cta", nw)
        outs.append(getattr(m, call)(0, *args, m.new_output()).clone())
    assert torch.equal(*outs)
    for nw in (9, 12, 16, 17):
        m.tune("decode_warps_per_cta", nw)
        with pytest.raises(SketchSSMError) as e:
            getattr(m, call)(0, *args, m.new_output())
        assert e.value.status == -2
    m.check_status()


@pytest.mark.parametrize("case", [("mamba2", 5, 7, 64, 64, 9, 12, "bf16", False, True), ("kda", 4, 7, 64, 128, 16, 16, "f32", False, True),
                                  ("gdn", 11, 2, 64, 64, 24, 8, "f32", False, True)])
def test_the_last_head_dense_with_sixteen_rows_per_warp(case):
    """Its rows are the last of the state: four warps a head, K = 64."""
    test_teams_of_warps_and_single_warps_agree(*case)
