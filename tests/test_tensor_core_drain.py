"""A block of the surrogate's tensor-core kernels that gives up a wait frees its
TMEM only after the last MMAs it issued: the phases it waits for
(csrc/aap_drain.cuh, compiled here by the host compiler) against a model of the
mbarrier, for every layer and run the fused network can give up in."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2211_15630_gb300", "csrc")

MAIN = r"""
#include <cstdio>
#include "aap_drain.cuh"
using namespace aaps;
// an mbarrier after d completions is in phase d, of parity d & 1: a wait with
// a parity returns once the current phase has the other one
static bool returns(int d, unsigned parity) { return (unsigned)(d & 1) != parity; }
int main()
{
    int bad = 0, early_zero = 0;
    for (int l = 1; l <= 4; ++l)
        for (int t = 0; t < 3; ++t) {
            const int n = net_commits(l, t);
            int issued = 0;
            for (int k = 1; k <= l; ++k) issued += k < 4 || t < 2;     // layer 4 has two runs
            if (n != issued) ++bad;
            // every layer before l was waited for, layer l may still be running
            const int waited = l < 4 || t < 2 ? n - 1 : n;
            for (int d = waited; d <= n; ++d)
                if (returns(d, nth_parity(n)) != (d == n)) ++bad;
            if (waited < n && returns(waited, 0u)) ++early_zero;       // what a fixed parity would do
        }
    for (int n = 1; n <= 9; ++n)
        if (returns(n - 1, nth_parity(n)) || !returns(n, nth_parity(n))) ++bad;
    // the pipelined convolution: tile k's commit goes to accumulator k % 4; the
    // last of i tiles is the last completion of its accumulator
    for (int i = 1; i <= 20; ++i) {
        const int last = i - 1;
        int n = 0;
        for (int k = 0; k < i; ++k) n += k % 4 == last % 4;
        if (nth_parity(last / 4 + 1) != nth_parity(n)) ++bad;
    }
    std::printf("bad %d early %d\n", bad, early_zero);
    return 0;
}
"""


def test_the_phase_waited_for_is_the_last_one_issued(tmp_path):
    if not shutil.which("g++"):
        pytest.skip("g++ not available")
    src, exe = tmp_path / "drain.cpp", str(tmp_path / "drain")
    src.write_text(MAIN)
    r = subprocess.run(["g++", "-std=c++17", "-Wall", "-x", "c++", "-I" + CSRC, str(src), "-o", exe], capture_output=True,
                       text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.stdout.split() == ["bad", "0", "early", "5"]      # runs 0 to 2 of layer 2, runs 0 and 1 of layer 4
