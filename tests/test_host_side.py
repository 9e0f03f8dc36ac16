"""CPU tests of the host-side pieces: the product's offline calibration against the oracle's fit, the byte
accounting, and the benchmark's rank sharding under torch.distributed (gloo, world size 2)."""
import os
import subprocess
import sys

import numpy as np
import torch

from oracle import sketchssm_oracle as orc
from paper_2609_33051_b200 import calibrate, synth, traffic

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_product_calibration_matches_oracle_fit():
    w = synth.CONFIGS["c2_mamba2"].replace(calib_n=1024)
    Q = synth.calibration_queries(w, 0, 3)
    Om_p, C_p = calibrate.fit_head(torch.from_numpy(Q), w.rank)
    Om_o, lam = orc.fit_sketching_matrix(Q, np.eye(w.dk), w.rank)
    C_o = orc.offline_coefficient_map(Om_o, np.eye(w.dk))
    np.testing.assert_allclose(Om_p.numpy(), Om_o, atol=1e-8)      # same sign convention, distinct eigenvalues
    np.testing.assert_allclose(C_p.numpy(), C_o, atol=1e-8)
    # and with a non-identity metric
    rng = np.random.default_rng(0)
    A = rng.standard_normal((w.dk, w.dk))
    E0 = A @ A.T / w.dk + 0.5 * np.eye(w.dk)
    Om_p, C_p = calibrate.fit_head(torch.from_numpy(Q), 5, torch.from_numpy(E0))
    Om_o, _ = orc.fit_sketching_matrix(Q, E0, 5)
    np.testing.assert_allclose(Om_p.numpy(), Om_o, atol=1e-7)
    np.testing.assert_allclose(C_p.numpy(), orc.offline_coefficient_map(Om_o, E0), atol=1e-7)


def test_algorithmic_byte_accounting():
    # Mamba-2 layer, bf16 I/O: slot = 128*2 + 64*2 + 8 = 392 B, token = 256 + 392 = 648 B
    assert traffic.slot_bytes("mamba2", 128, 64, "bf16") == 392
    assert traffic.slot_bytes("gdn", 128, 128, "bf16") == 520
    assert traffic.slot_bytes("kda", 128, 128, "bf16") == 772
    assert traffic.token_bytes("mamba2", 128, 64, "bf16") == 648
    per_head = 16 * 64 * 4 + 7 * 392 + 648 + 392 + 64 * 4
    assert traffic.decode_bytes("mamba2", 256, 64, 128, 64, 16, 7) == 256 * 64 * per_head + 64 * 16 * 128 * 4
    full = 128 * 64 * 4 + 7 * 392 + 648 + 392 + 64 * 4
    assert traffic.decode_bytes("mamba2", 256, 64, 128, 64, 16, 7, full_read=True) == 256 * 64 * full
    upd = 2 * 128 * 64 * 4 + 15 * 392 + 392 + 256 + 256 + 16 * 64 * 4
    assert traffic.update_bytes("mamba2", 256, 64, 128, 64, 16, 15) == 256 * 64 * upd + 64 * 128 * 16 * 4
    # the sketch read is K/r times smaller than the state read
    assert (128 * 64 * 4) // (16 * 64 * 4) == 8


_WORKER = r"""
import os, sys, json
sys.path.insert(0, {root!r})
import torch, torch.distributed as dist
import bench
dist.init_process_group("gloo", init_method="tcp://127.0.0.1:{port}", rank=int(sys.argv[1]), world_size=2)
rank = dist.get_rank()
# every rank times its own shard; the job time is the max over ranks, the job value the sum of tokens over that time
ms_local = 10.0 + 5.0 * rank
ms = bench.max_over_ranks(ms_local, dist, device="cpu")
value = bench.job_value(tokens_per_rank=1000, world=2, ms_step=ms)
shard = bench.rank_shard(total_batch=9, rank=rank, world=2)
if rank == 0:
    print(json.dumps(dict(ms=ms, value=value, shard=list(shard))))
else:
    print(json.dumps(dict(shard=list(shard))))
dist.destroy_process_group()
"""


def test_rank_sharding_and_max_over_ranks_timing_with_gloo(tmp_path):
    script = tmp_path / "worker.py"
    script.write_text(_WORKER.format(root=ROOT, port=29641))
    procs = [subprocess.Popen([sys.executable, str(script), str(r)], stdout=subprocess.PIPE, stderr=subprocess.PIPE, text=True)
             for r in range(2)]
    outs = [p.communicate(timeout=120) for p in procs]
    for p, (o, e) in zip(procs, outs):
        assert p.returncode == 0, e[-2000:]
    import json
    r0 = json.loads(outs[0][0].strip().splitlines()[-1])
    r1 = json.loads(outs[1][0].strip().splitlines()[-1])
    assert r0["ms"] == 15.0                       # max over ranks
    assert abs(r0["value"] - 2 * 1000 / 15e-3) < 1e-6
    assert r0["shard"] == [0, 4] and r1["shard"] == [4, 9]     # disjoint cover of the batch, no exchange needed


def test_logical_layers_map_onto_the_physical_slots_that_fit():
    """The 48-layer stack of the large-batch sweep does not fit at batch 2048: the benchmark maps the logical layers
    round-robin onto as many physical slots as its memory budget holds."""
    import bench
    w = synth.sweep_point(2048, 16, 16)
    per = bench.layer_bytes(w)
    assert per > 2048 * 64 * 128 * 64 * 4                       # at least the state: 4 GiB per layer
    assert 48 * per > 180e9                                     # 48 distinct layers exceed the GPU's memory
    n = bench.physical_layers(per, int(100e9), 48)
    assert 1 <= n < 48 and n * per <= 100e9 < (n + 1) * per
    assert bench.physical_layers(bench.layer_bytes(synth.sweep_point(64, 4, 8)), int(40e9), 48) == 48
    assert bench.physical_layers(10**12, 10**9, 48) == 1        # never fewer than one slot
    assert [l % n for l in range(48)].count(0) == -(-48 // n)   # slot 0 serves ceil(48 / n) logical layers
    assert bench.update_kernel_name(w) == "update_tc_ws_mamba2_kernel"
    assert bench.update_kernel_name(synth.CONFIGS["c4_kda"]) == "update_tc_ws_kda_kernel"
    assert bench.update_kernel_name(synth.CONFIGS["c1_gdn_tiny"]) == "update_kernel"


def test_current_stream_without_the_raw_stream_functions(monkeypatch):
    """torch's raw stream functions are private: where a version lacks them the public call gives the handle."""
    from types import SimpleNamespace
    from paper_2609_33051_b200 import binding
    monkeypatch.setattr(binding, "_RAW_STREAM", None)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda: SimpleNamespace(cuda_stream=1234))
    assert binding.SketchSSM._stream(None) == 1234
    assert binding.SketchSSM._stream(SimpleNamespace(cuda_stream=77)) == 77


def test_the_benchmark_prints_one_short_line_and_its_records_beside_it(capsys, tmp_path):
    """Standard output is one JSON line that does not grow with the sweep; the records go to standard error, where the report
    finds them.  A derived decode time that would beat a copy is shown as the back-to-back one."""
    import json
    import bench
    from paper_2609_33051_b200 import report
    rec = {"workload": "w: mamba2 B1", "coefficient_map": "fixed", "sketch_storage": "f32", "n_phys": 1, "value": 1e6,
           "decode_in_window_us": 10.0, "decode_frac_of_measured": 1.04, "decode_frac_of_8TBs_nominal": 0.86,
           "decode_back_to_back_us": 13.0, "decode_back_to_back_frac_of_measured": 0.8, "update_kernel": "k", "update_us": 5.0,
           "update_frac_of_measured": 0.9, "sketch_and_map_overhead_on_flush": 0.05, "full_read": {"sketch_speedup": 2.0},
           "clocks": {"sm_mhz": 1900.0, "reasons": []}, "padding": "x" * 2000}
    bench.print_result({"metric": "m", "value": 1.0}, [("sweep", [rec] * 38), ("variant", [rec] * 7)])
    out, err = capsys.readouterr()
    assert json.loads(out) == {"metric": "m", "value": 1.0} and out.count("\n") == 1
    assert [json.loads(ln)["record"] for ln in err.splitlines()] == ["sweep"] * 38 + ["variant"] * 7
    row = report.table([rec])
    assert "13.0 (back to back) | 0.80" in row and "1.04" not in row
    rec["decode_frac_of_measured"] = 0.95
    assert "| 10.0 | 0.95" in report.table([rec])


_ROWS = r"""
#include <cstdio>
#include <initializer_list>
#include "state_rows.h"
using namespace sketchssm;
int main() {
    for (int K : {64, 128}) for (int W : {1, 2, 4}) for (int RB : {8, 16}) for (int sub = 0; sub < W; ++sub) {
        if ((K / W) % RB) continue;
        const int a = first_row(K, W, sub);
        std::printf("%d %d %d 0 %d %d\n", K, W, sub, a, a + rows_asked_first(K, W));
        for (int i0 = a; i0 < end_row(K, W, sub); i0 += RB) {
            std::printf("%d %d %d 1 %d %d\n", K, W, sub, i0, i0 + RB);
            if (asks_ahead(K, W, sub, i0)) std::printf("%d %d %d 0 %d %d\n", K, W, sub, i0 + kAhead, i0 + kAhead + RB);
        }
    }
}
"""


def test_a_dense_heads_warps_read_each_row_once_and_ask_only_for_their_own(tmp_path):
    """A request for a row that another warp owns is made twice, and one behind the last head's state may not be mapped."""
    (tmp_path / "rows.cpp").write_text(_ROWS)
    exe = str(tmp_path / "rows")
    subprocess.run(["g++", "-std=c++17", "-I", os.path.join(ROOT, "paper_2609_33051_b200", "csrc"), str(tmp_path / "rows.cpp"),
                    "-o", exe], check=True)
    read, asked = {}, {}
    for ln in subprocess.run([exe], check=True, capture_output=True, text=True).stdout.splitlines():
        K, W, sub, is_read, a, b = map(int, ln.split())
        (read if is_read else asked).setdefault((K, W, sub), set()).update(range(a, b))
    for (K, W, sub), rows in read.items():
        assert rows == set(range(sub * K // W, (sub + 1) * K // W)), (K, W, sub)
        assert asked[K, W, sub] <= rows, (K, W, sub)
    assert len(read) == 2 * (1 + 2 + 4)


_SETS = r"""
#include <cstdio>
#include "operand_sets.h"
using namespace sketchssm;
int main() {
    for (int tiles = 0; tiles < 12; ++tiles) {
        std::printf("%d", tiles);
        for (int t = first_unfinished(tiles); t < tiles; ++t) std::printf(" %d %u", set_of_tile(t), parity_of_tile(t));
        std::printf("\n");
    }
}
"""


def test_a_flush_that_gives_up_waits_for_the_last_fill_of_each_operand_set(tmp_path):
    """A barrier answers a wait for parity p at once unless its current phase has that parity: a wait for another phase than the one
    in flight gives the copies no time."""
    (tmp_path / "sets.cpp").write_text(_SETS)
    exe = str(tmp_path / "sets")
    csrc = os.path.join(ROOT, "paper_2609_33051_b200", "csrc")
    subprocess.run(["g++", "-std=c++17", "-I", csrc, str(tmp_path / "sets.cpp"), "-o", exe], check=True)
    for ln in subprocess.run([exe], check=True, capture_output=True, text=True).stdout.splitlines():
        tiles, *waits = map(int, ln.split())
        waits = set(zip(waits[::2], waits[1::2]))
        fills = [[t for t in range(tiles) if t % 2 == s] for s in (0, 1)]
        # the last fill of a set is not complete: its barrier is in phase len(fills) - 1
        assert waits == {(s, (len(f) - 1) % 2) for s, f in enumerate(fills) if f}, tiles
    src = open(os.path.join(csrc, "update_tc_ws_kda.cu")).read()
    grace = src[src.index("if (dead && ft < 32)"):]
    assert "kVals + set_of_tile(t)], parity_of_tile(t)" in grace[:600]


def test_inline_loads_are_ordered_with_the_waits_before_them():
    """A load in inline assembly that is not volatile is to the compiler a function of its address, which it may move ahead of the
    wait for the kernel that writes the memory; one of global memory has to name memory as well, as plain loads and stores do not
    keep their order with it otherwise."""
    import glob
    import re
    csrc, seen = os.path.join(ROOT, "paper_2609_33051_b200", "csrc"), 0
    for path in sorted(glob.glob(os.path.join(csrc, "*.cu*"))):
        src = open(path).read()
        for m in re.finditer(r"\basm\b(\s+volatile)?\s*\((.*?)\)\s*;\s*(?:\n|\})", src, re.S):
            stmt = m.group(2)
            where = (os.path.basename(path), src[:m.start()].count("\n") + 1)
            if re.search(r"\b(ld\.|ldmatrix|tcgen05\.ld)", stmt):
                seen += 1
                assert m.group(1), where
            if re.search(r"\bld\.(global|acquire|relaxed|volatile)", stmt):
                assert '"memory"' in stmt, where
    assert seen >= 6
