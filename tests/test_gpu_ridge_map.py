"""The exact ridge map for up to 32 ranks: ranks at and between the sizes it is compiled for, every state
shape, a head per CTA of 64 and 128 threads, a zero state, bars as for the other state-dependent maps."""
import numpy as np
import pytest
import torch

from paper_2609_33051_b200 import synth
from tests.test_gpu_coef_map import check_coef
from tests.test_gpu_parity import make_layer, run_schedule

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rank", [1, 8, 9, 16, 17, 24, 31, 32])
@pytest.mark.parametrize("K,V", [(128, 64), (128, 80), (128, 128), (64, 64), (64, 128)])
def test_ridge_map_ranks_and_shapes(rank, K, V):
    w = synth.Workload("t", "mamba2", 3, 2, K, V, rank, 4, 0, "bf16", 307, basis="qr")
    check_coef(run_schedule(w, w.buf_len + 1, max_heads=10**9, coef="ridge"))


def test_zero_state_gives_a_zero_map():
    w = synth.Workload("t", "gdn", 2, 2, 128, 128, 16, 4, 0, "bf16", 311, basis="qr")
    m, *_ = make_layer(w, coef="ridge")
    m.state.zero_()
    m.coef.fill_(float("nan"))
    m.state_update(0)
    m.check_status()
    assert torch.equal(m.coef, torch.zeros_like(m.coef))


@pytest.mark.parametrize("rank", [1, 8, 13, 24, 32, 40])
@pytest.mark.parametrize("K,V", [(128, 64), (128, 80), (64, 128)])
@pytest.mark.parametrize("sketch", ["f32", "bf16"])
def test_the_input_precision_does_not_choose_the_map(rank, K, V, sketch):
    """The map is built from the state and the stored sketch: layers that differ in the type of q, k, v only get the same bits."""
    maps = []
    for io in ("bf16", "f32"):
        w = synth.Workload("t", "mamba2", 3, 2, K, V, rank, 4, 0, io, 313, basis="qr")
        m, *_ = make_layer(w, coef="ridge", sketch=sketch)
        m.tune("update_impl", 1)                               # the same sketch on both sides
        m.state_update(0)
        m.check_status()
        maps.append(m.coef.clone())
    assert torch.equal(*maps)


@pytest.mark.parametrize("rank", [8, 13, 32])
@pytest.mark.parametrize("K,V", [(128, 64), (128, 80), (128, 128), (64, 64)])
def test_ridge_map_with_fp32_inputs(rank, K, V):
    w = synth.Workload("t", "kda", 3, 2, K, V, rank, 4, 0, "f32", 317, basis="qr")
    check_coef(run_schedule(w, w.buf_len + 1, max_heads=10**9, coef="ridge"))
