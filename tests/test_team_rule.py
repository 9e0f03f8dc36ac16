"""How many warps share a head in the decode kernel, and how their CTAs are chosen (CPU)."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


_CTA = r"""
#include <cstdio>
#include <initializer_list>
#include "team_size.h"
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
