"""The autotuner's rule on made-up times (CPU): csrc/tune.h compiled by itself.

The chosen variant is the one of the least median of three samples, whatever
samples the rule leaves out; one disturbed launch never decides.
"""
import os
import shutil
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1607_01650_gb300", "csrc")

PROG = r"""
#include "tune.h"
#include <cstdio>
int main()
{
    int trials, count;
    while (std::scanf("%d", &count) == 1) {
        float best_us = 1e30f;
        int best = -1, used = 0;
        for (int v = 0; v < count; ++v) {
            float t[3], us = -1.f;
            if (std::scanf("%f %f %f", t, t + 1, t + 2) != 3) return 1;
            int k = 0;
            if (!dect::median_time(best_us, [&](float &x) { x = t[k++]; ++used; return x >= 0.f; }, us)) { best = -2; continue; }
            if (best != -2 && us < best_us) { best_us = us; best = v; }
        }
        std::printf("%d %d\n", best, used);
    }
}
"""


@pytest.fixture(scope="module")
def prog(tmp_path_factory):
    if not shutil.which("g++"):
        pytest.skip("no g++")
    d = tmp_path_factory.mktemp("tune")
    (d / "t.cpp").write_text(PROG)
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", CSRC, "-o", str(d / "t"), str(d / "t.cpp")], check=True)
    return str(d / "t")


def _choices(prog, trials):
    text = "".join("%d\n%s\n" % (len(t), "\n".join(" ".join("%.6f" % x for x in row) for row in t)) for t in trials)
    out = subprocess.run([prog], input=text, capture_output=True, text=True, check=True).stdout.split()
    return [(int(a), int(b)) for a, b in zip(out[::2], out[1::2])]


def test_the_least_median_wins(prog):
    rng = np.random.default_rng(1)
    trials = []
    for _ in range(400):
        t = rng.uniform(50, 60, (int(rng.integers(1, 9)), 1)) + rng.uniform(0, 8, (1, 3))
        t = t + rng.uniform(0, 5, t.shape)
        t[rng.random(t.shape) < 0.15] *= rng.uniform(1.2, 30)  # disturbed launches
        trials.append(t)
    got = _choices(prog, trials)
    for t, (choice, used) in zip(trials, got):
        assert choice == int(np.median(np.round(t, 6), axis=1).argmin())
        assert 2 * len(t) <= used <= 3 * len(t)
    assert sum(u for _, u in got) < sum(t.size for t in trials)


def test_one_disturbed_launch_does_not_rule_a_variant_out(prog):
    for k in range(3):
        fast = [40.0, 40.1, 40.2]
        fast[k] = 900.0
        assert _choices(prog, [[[50.0, 50.1, 50.2], fast, [60.0, 60.0, 60.0]]])[0][0] == 1


def test_a_failed_sample_gives_up(prog):
    assert _choices(prog, [[[50.0, -1.0, 50.0]]])[0][0] == -2
