"""How the LM head spreads its work over CTAs (csrc/lmhead_split.h), on the host: a
device whose cluster query fails, or that holds no CTA pair, runs single CTAs; the
splits cover the vocabulary, up to the largest one, and fit the workspace."""
import shutil
import subprocess
from pathlib import Path

import pytest

CSRC = Path(__file__).resolve().parents[1] / "paper_2608_11742_gb300" / "csrc"

PROGRAM = r"""
#include <cstdio>
#include "lmhead_split.h"
using namespace rps;
int main() {
    const int row_tiles[] = {1, 2, 2, 3, 3, 4, 5, 9, 9, 9, 11, 9, 2, 2, 7, 6, 3, 3, 7};
    const long long vs[] = {126464, 126464, 8000, 126464, 32000, 126464, 126464, 126464, 8000, 300, 126464, 20000, 900, 40000, 9720, 126464, 20004, 126300, 90000};
    const int ds[] = {4096, 4096, 1024, 4096, 1024, 4096, 4096, 4096, 4096, 4096, 1024, 4096, 2112, 1088, 1088, 128, 64, 64, 4096};
    for (int i = 0; i < 19; ++i) {
        const LmSplit s = lm_split(row_tiles[i], vs[i], ds[i] / 64, row_tiles[i] == 1 ? 256 : std::min(256ll, (vs[i] + 255) / 256), 152, 76);
        std::printf("R %d %lld %d %d %d %d\n", row_tiles[i], vs[i], ds[i], s.pair, s.granule, s.splits);
    }
    std::printf("Q %d %d %d %d\n", lm_pairs(true, 76), lm_pairs(true, 0), lm_pairs(false, 76), lm_pairs(false, -1));
    const long long vocabs[] = {1, 63, 64, 65, 300, 9000, 126464, 2147483000, 2147483647};
    const int sms[] = {1, 20, 152}, pairs[] = {0, 1, 76};
    for (int t = 1; t < 40; ++t)
        for (long long v : vocabs)
            for (int m : sms)
                for (int p : pairs)
                    for (int cap : {1, 7, 256}) {
                        const LmSplit s = lm_split(t, v, 1 + (t * 7 + cap) % 64, cap, m, p);
                        const auto at = [&](int split) { return (long long)lm_range(split, s.n_gran, s.splits, s.granule); };
                        long long most = 0;
                        for (int i = 0; i < s.splits; ++i) most = std::max(most, at(i + 1) - at(i));
                        std::printf("S %d %lld %d %d %d %d %d %d %d %d %d %lld %lld %lld %lld\n", t, v, m, p, cap, s.pair,
                                    s.units, s.granule, s.n_gran, s.splits, s.longest, at(0), at(s.splits - 1),
                                    at(s.splits), most);
                    }
    return 0;
}
"""


@pytest.fixture(scope="module")
def lines(tmp_path_factory):
    gxx = shutil.which("g++")
    if not gxx:
        pytest.skip("no host C++ compiler")
    d = tmp_path_factory.mktemp("split")
    (d / "s.cpp").write_text(PROGRAM)
    subprocess.run([gxx, "-std=c++17", "-O0", f"-I{CSRC}", str(d / "s.cpp"), "-o", str(d / "s")], check=True)
    out = subprocess.run([str(d / "s")], check=True, capture_output=True, text=True).stdout.splitlines()
    return [l.split() for l in out]


def test_a_failed_cluster_query_means_no_pairs(lines):
    assert [l for l in lines if l[0] == "Q"] == [["Q", "76", "0", "0", "0"]]


def test_splits(lines):
    rows = [list(map(int, l[1:])) for l in lines if l[0] == "S"]
    assert rows
    for t, v, sms, pairs, cap, pair, units, granule, n_gran, splits, longest, first, last, end, most in rows:
        assert not (pair and pairs == 0), "no pair resident: single CTAs"
        assert units == ((t + 1) // 2 if pair else t) and granule in ((128,) if pair else (64, 256))
        assert (n_gran - 1) * granule < v <= n_gran * granule
        assert 1 <= splits <= min(cap, n_gran) and splits * longest >= n_gran
        assert splits == 1 or splits * units <= (pairs if pair else sms)
        assert first == 0 and last < v <= end == n_gran * granule and 0 < most == longest * granule


def test_forms(lines):
    """Row tiles, vocabulary, d -> pairs, tokens the splits are cut at, splits (152 SMs, 76 pairs)."""
    got = {tuple(map(int, l[1:4])): tuple(map(int, l[4:])) for l in lines if l[0] == "R"}
    assert got == {
        (1, 126464, 4096): (0, 64, 152),   # one row tile: quarters
        (2, 126464, 4096): (1, 128, 76),
        (2, 8000, 1024): (0, 256, 32),     # one tile of 16 slices: too short for a pair
        (3, 126464, 4096): (0, 256, 50),   # quarters are no shorter
        (3, 32000, 1024): (0, 64, 50),     # ten quarters against three tiles
        (4, 126464, 4096): (1, 128, 38),
        (5, 126464, 4096): (0, 256, 30),
        (9, 126464, 4096): (1, 128, 15),   # 33 tiles against 31
        (9, 20000, 4096): (0, 256, 16),    # 5.5 against five
        (9, 8000, 4096): (0, 256, 16),     # 2.5 tiles against two
        (9, 300, 4096): (0, 64, 2),        # three quarters against a tile
        (11, 126464, 1024): (1, 128, 12),  # 41.5 tiles against 38
        (2, 900, 2112): (1, 128, 4),
        (2, 40000, 1088): (1, 128, 63),
        (7, 9720, 1088): (1, 128, 19),
        (7, 90000, 4096): (1, 128, 19),    # 19 tiles against 17
        (6, 126464, 128): (1, 128, 25),
        (3, 20004, 64): (0, 64, 45),
        (3, 126300, 64): (0, 256, 50),
    }
