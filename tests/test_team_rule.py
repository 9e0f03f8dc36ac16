"""How many warps share a head in the decode kernel, held against measured launch times, and how their CTAs are chosen (CPU)."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

# kind, buffered tokens, heads, stages that fit an SM, K, V: us a launch of a full read with 1, 2, 4 warps per head (148 SMs)
FULL = """
    gdn 14 4736 24 128 128 68.5 52.1 56.2; gdn 14 592 24 128 128 8.1 6.6 7.8; gdn 3 2368 63 128 128 32.5 28.0 27.5; gdn 3 4736 63 128 128 73.2 49.1 50.6
    gdn 3 888 63 128 128 10.1 6.9 6.9; gdn 30 1184 13 128 128 23.1 22.3 20.8; gdn 30 2368 13 128 128 48.2 37.2 36.5; gdn 30 888 13 128 128 10.8 12.8 11.9
    gdn 6 296 32 128 64 5.4 3.8 3.8; gdn 6 4736 34 64 128 40.5 27.1 34.9; gdn 6 592 34 64 128 4.5 4.2 5.2; kda 10 296 27 128 64 6.0 4.3 4.3
    kda 10 4736 27 128 64 50.8 29.4 34.0; kda 10 888 27 128 64 6.4 5.9 6.6; kda 14 2368 18 128 128 36.9 30.4 30.9; kda 14 592 18 128 128 8.3 6.9 8.3
    kda 14 888 18 128 128 10.1 9.4 9.2; kda 20 1184 6 128 128 35.8 27.9 27.6; kda 20 2368 6 128 128 56.7 66.3 43.8; kda 20 296 6 128 128 8.9 7.0 6.6
    kda 20 4736 6 128 128 108.8 133.2 86.2; kda 20 888 6 128 128 16.6 13.6 15.1; kda 28 2368 11 128 64 33.6 29.0 31.1; kda 28 4736 11 128 64 54.3 47.8 56.6
    kda 28 592 11 128 64 8.2 7.2 9.5; kda 8 1184 52 64 64 4.4 5.3 7.3; kda 8 4736 52 64 64 22.5 15.6 20.8; kda 8 592 52 64 64 4.1 3.9 4.6
    mamba2 30 4736 17 128 64 41.6 30.8 32.8; mamba2 30 592 17 128 64 7.3 5.2 5.6; mamba2 30 888 17 128 64 7.5 6.4 6.3; mamba2 6 1184 25 128 128 19.1 14.4 11.5
    mamba2 6 4736 25 128 128 72.5 49.2 50.3; mamba2 62 2368 8 128 64 35.3 29.0 25.6; mamba2 62 4736 8 128 64 67.7 72.9 48.8; mamba2 62 592 8 128 64 10.4 6.5 7.2
    mamba2 62 888 8 128 64 11.2 8.4 7.7; mamba2 8 1184 37 128 128 11.2 14.0 10.5; mamba2 8 1184 65 64 64 4.1 4.1 5.2; mamba2 8 2368 42 128 80 21.5 22.3 24.9
    mamba2 8 2368 45 128 64 11.6 11.8 11.8; mamba2 8 2368 65 64 64 5.4 6.3 8.0; mamba2 8 296 37 128 128 7.4 4.6 4.0; mamba2 8 296 42 128 80 7.8 5.0 4.5
    mamba2 8 296 65 64 64 3.8 3.0 2.9; mamba2 8 4736 42 128 80 36.8 34.8 44.3; mamba2 8 592 45 128 64 6.0 4.3 4.8; mamba2 8 888 37 128 128 8.3 6.8 6.9
    mamba2 8 888 42 128 80 8.2 6.4 6.6; mamba2 8 888 45 128 64 6.0 4.9 5.3; gdn 30 4736 9 64 128 57.0 56.2 67.5; kda 30 9472 6 64 128 136.8 127.3 142.2
"""

# the same: us a launch of a decode step with a rank table, 1, 2, 4 warps per head; without a dense
# head, then with one of twelve
TABLE = """
    mamba2 4 300 28 128 80 3.8 3.7 3.9 7.6 5.9 4.4; mamba2 28 300 12 128 80 6.0 4.6 4.5 9.5 6.9 5.1; mamba2 4 588 28 128 80 4.0 3.9 4.8 7.6 6.0 5.1
    mamba2 28 588 12 128 80 6.3 4.9 5.7 9.5 7.3 6.4; mamba2 4 876 28 128 80 4.1 4.2 5.5 7.7 6.3 5.7; mamba2 12 876 19 128 80 4.9 4.6 6.0 8.5 6.8 6.1
    mamba2 28 876 12 128 80 7.6 6.5 6.8 10.5 8.4 6.9; mamba2 4 1200 28 128 80 4.8 5.2 7.6 7.7 7.3 8.2; mamba2 12 1200 19 128 80 5.9 5.9 8.6 9.0 8.2 8.8
    mamba2 28 1200 12 128 80 8.1 7.2 9.9 10.6 8.8 10.2; mamba2 4 1776 28 128 80 5.8 6.3 8.4 8.9 7.2 8.8; mamba2 28 1776 12 128 80 9.4 10.7 10.9 11.4 14.0 11.0
    gdn 4 300 17 128 128 3.9 3.8 4.0 7.9 5.0 4.4; gdn 28 300 8 128 128 7.0 6.4 7.5 10.9 7.7 7.7; gdn 4 588 17 128 128 3.9 4.0 5.0 8.1 5.3 5.4
    gdn 28 588 8 128 128 7.1 7.8 9.1 11.1 8.7 9.2; gdn 4 876 17 128 128 4.2 4.4 6.0 8.0 6.0 6.2; gdn 12 876 13 128 128 5.3 6.2 7.5 8.9 7.6 7.7
    gdn 28 876 8 128 128 8.2 8.7 10.6 11.1 9.1 11.0; gdn 4 1200 17 128 128 5.0 5.4 8.3 8.5 7.3 8.6; gdn 12 1200 13 128 128 6.5 7.0 10.9 9.5 8.1 11.1
    gdn 28 1200 8 128 128 14.5 14.1 16.2 19.0 15.7 16.7; gdn 4 1776 17 128 128 5.8 6.5 9.1 11.8 7.7 10.1; gdn 28 1776 8 128 128 14.7 14.8 18.6 20.7 17.3 19.4
    gdn 4 300 39 64 64 3.1 3.2 3.4 3.7 3.3 3.4; gdn 28 300 12 64 64 5.7 5.5 6.2 6.3 5.8 6.2; gdn 4 588 39 64 64 3.3 3.3 4.4 3.7 3.5 4.4
    gdn 28 588 12 64 64 5.9 5.9 7.5 6.4 6.3 7.5; gdn 4 876 39 64 64 3.4 3.6 5.3 3.9 3.8 5.3; gdn 12 876 23 64 64 4.2 4.5 6.4 5.0 4.8 6.3
    gdn 28 876 12 64 64 6.2 7.1 8.5 6.6 7.2 8.6; gdn 4 1776 39 64 64 4.4 5.4 7.7 4.6 5.5 8.0; gdn 28 1776 12 64 64 8.3 12.5 14.2 8.3 12.5 14.3
    mamba2 4 300 29 128 64 3.7 3.7 3.9 5.6 4.2 3.9; mamba2 28 300 12 128 64 4.8 4.0 4.2 6.4 4.8 4.2; mamba2 4 588 29 128 64 3.7 4.0 4.6 5.8 4.4 4.7
    mamba2 28 588 12 128 64 5.0 4.4 5.4 6.5 5.2 5.6; mamba2 4 876 29 128 64 4.1 4.2 5.4 5.8 4.7 5.4; mamba2 12 876 20 128 64 4.4 4.3 5.8 6.2 5.0 5.9
    mamba2 28 876 12 128 64 6.5 5.7 6.5 7.4 6.0 6.5; mamba2 4 1200 29 128 64 4.6 4.9 7.3 5.9 5.4 7.3; mamba2 12 1200 20 128 64 5.3 5.4 8.1 6.7 6.3 8.1
    mamba2 28 1200 12 128 64 7.0 6.5 9.1 7.4 6.7 9.2; mamba2 4 1776 29 128 64 4.7 6.0 8.0 6.5 6.1 8.0; mamba2 28 1776 12 128 64 8.3 9.5 10.1 8.3 9.8 10.2
    mamba2 30 1776 9 128 80 14.0 12.8 11.8 18.8 15.3 11.8
"""

# the same: us a mixed step, one head of twelve dense and one sequence in 16 flushing
MIXED = """
    gdn 15 108 13 128 128 14.2 14.2 14.2; gdn 15 144 13 128 128 14.2 14.3 21.1; gdn 15 192 13 128 128 15.0 21.3 17.4; gdn 15 432 13 128 128 23.2 22.5 19.9
    mamba2 15 108 13 128 128 11.6 11.7 11.6; mamba2 15 144 13 128 128 11.7 11.7 16.4; mamba2 15 192 13 128 128 12.3 16.4 13.2
    mamba2 15 288 13 128 128 16.2 15.0 15.7; mamba2 15 144 19 128 80 11.8 11.5 12.4; mamba2 15 720 19 128 80 18.6 17.8 16.3
"""

_MAIN = r"""
#include <cstdio>
#include "team_size.h"
int main() {
    int table, mamba2, n, slots, K, V;
    long long heads;
    while (std::scanf("%d %d %d %lld %d %d %d", &table, &mamba2, &n, &heads, &slots, &K, &V) == 7)
        std::printf("%d\n", table ? sketchssm::rank_table_team(mamba2, table == 2, n, heads, 148, slots, K, V)
                                  : sketchssm::full_read_team(mamba2, n, heads, 148, slots, K, V, 96ll << 20));
}
"""


def _points(text):
    return [p.split() for p in text.replace("\n", ";").split(";") if p.strip()]


def _chosen(tmp_path, asked):
    (tmp_path / "rule.cpp").write_text(_MAIN)
    exe = str(tmp_path / "rule")
    subprocess.run(["g++", "-std=c++17", "-I", os.path.join(ROOT, "paper_2609_33051_b200", "csrc"), str(tmp_path / "rule.cpp"), "-o", exe],
                   check=True)
    text = "\n".join(" ".join(map(str, a)) for a in asked)
    return [{"1": 0, "2": 1, "4": 2}[w] for w in subprocess.run([exe], input=text, check=True, capture_output=True, text=True).stdout.split()]


def test_full_reads_are_no_slower_than_with_a_warp_per_head(tmp_path):
    pts = _points(FULL)
    times = [list(map(float, p[6:])) for p in pts]
    chosen = _chosen(tmp_path, [(0, int(p[0] == "mamba2"), *p[1:6]) for p in pts])
    assert len(chosen) == len(pts) >= 40
    for p, t, w in zip(pts, times, chosen):
        assert t[w] <= 1.05 * t[0], p
    assert sum(t[w] / min(t) for t, w in zip(times, chosen)) <= 1.05 * len(pts)


def test_mixed_steps_are_no_slower_than_with_a_warp_per_head(tmp_path):
    pts = _points(MIXED)
    chosen = _chosen(tmp_path, [(2, int(p[0] == "mamba2"), *p[1:6]) for p in pts])
    assert len(chosen) == len(pts)
    for p, w in zip(pts, chosen):
        t = list(map(float, p[6:]))
        assert t[w] <= 1.05 * t[0], p


def test_rank_tables_gain_with_a_dense_head_what_they_lose_without(tmp_path):
    pts = _points(TABLE)
    times = [list(map(float, p[6:])) for p in pts]
    chosen = _chosen(tmp_path, [(1, int(p[0] == "mamba2"), *p[1:6]) for p in pts])
    assert len(chosen) == len(pts) >= 30
    for p, t, w in zip(pts, times, chosen):
        assert t[w] / t[0] + t[3 + w] / t[3] <= 2.1, p
        assert t[w] <= 1.35 * t[0] and t[3 + w] <= 1.02 * t[3], p


_CTA = r"""
#include <cstdio>
#include <initializer_list>
#include "team_size.h"
static_assert(sketchssm::kTeamCtas * 16 <= 64, "an SM has 64 named barriers, each CTA of a team kernel holds 16");
int main() {
    for (int W : {2, 4}) for (int least : {W, 8}) for (long long heads : {1, 12, 60, 148, 300, 588, 876, 1200, 4736, 20000}) {
        int largest = 0;
        for (int nw = W; nw <= 24; nw += W) if (!sketchssm::team_cta_too_large(nw, W, least, heads, 148)) largest = nw;
        std::printf("%d %d %lld %d %d\n", W, least, heads, largest, sketchssm::useful_team_warps(W, heads, 148));
    }
}
"""


def test_few_heads_spread_over_the_sms(tmp_path):
    """The largest CTA that the launch may take does not pile heads on an SM while others have none, and a CTA size does not win by
    warps that no head would take."""
    (tmp_path / "cta.cpp").write_text(_CTA)
    exe = str(tmp_path / "cta")
    subprocess.run(["g++", "-std=c++17", "-I", os.path.join(ROOT, "paper_2609_33051_b200", "csrc"), str(tmp_path / "cta.cpp"), "-o", exe],
                   check=True)
    for ln in subprocess.run([exe], check=True, capture_output=True, text=True).stdout.splitlines():
        W, least, heads, largest, useful = map(int, ln.split())
        per_sm = -(-heads // 148)
        assert W <= largest <= max(least, W * per_sm), ln
        assert useful >= min(W * per_sm, 24) and (per_sm >= 64 or useful == W * per_sm), ln
