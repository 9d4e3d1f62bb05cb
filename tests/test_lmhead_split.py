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
    std::printf("Q %d %d %d %d\n", lm_pairs(true, 76), lm_pairs(true, 0), lm_pairs(false, 76), lm_pairs(false, -1));
    const long long vocabs[] = {1, 63, 64, 65, 300, 9000, 126464, 2147483000, 2147483647};
    const int sms[] = {1, 20, 152}, pairs[] = {0, 1, 76};
    for (int t = 1; t < 40; ++t)
        for (long long v : vocabs)
            for (int m : sms)
                for (int p : pairs)
                    for (int cap : {1, 7, 256}) {
                        const LmSplit s = lm_split(t, v, v / 256 + 1, cap, m, p);
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
        assert units == ((t + 1) // 2 if pair else t) and granule == (128 if pair else 64)
        assert (n_gran - 1) * granule < v <= n_gran * granule
        assert 1 <= splits <= min(cap, n_gran) and splits * longest >= n_gran
        assert splits == 1 or splits * units <= (pairs if pair else sms)
        assert first == 0 and last < v <= end == n_gran * granule and 0 < most == longest * granule
