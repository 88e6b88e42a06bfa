"""The counter sets that a sketch's phases use in turn, on the CPU: im_host.h's
rules (which set, who zeroes it, how much of it) drive a model of the device in
which phases complete, give up, fail to launch or run a launch a level, in
random order.  Whatever came before, a set is all zero when its phase begins:
the kernels between the phases reserve queue places from its first counter
without a look at the error word."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2410_14047_gb300", "csrc")

MODEL = r"""
#include <cstdio>
#include <cstdlib>
#include <vector>
#include "im_host.h"

constexpr int kAll = 40;
struct Device {
    std::vector<long> ctr[2] = {std::vector<long>(kAll, 7), std::vector<long>(kAll, 7)};  // as allocated
    int levels[2] = {0, 0};
    bool gave_up = false;
};

int main(int argc, char** argv) {
    const unsigned kinds = (unsigned)atoi(argv[1]);  // bits: 1 give up, 2 launch a level, 4 a launch fails
    for (unsigned seed = 1; seed <= 2000; ++seed) {
        srand(seed);
        Device d;
        imi::PhaseSets sets;
        for (int phase = 0; phase < 30; ++phase) {
            const bool host_zeroes = sets.begin();
            const int s = sets.cur(), o = sets.other();
            if (host_zeroes) {
                d.ctr[s].assign(kAll, 0);
                d.levels[s] = 0;
            }
            for (long c : d.ctr[s])
                if (c != 0) return printf("seed %u phase %d: a set with old counters\n", seed, phase), 1;
            d.ctr[s][0] += 1 + rand() % 9;  // the level-0 queue, written before the launch
            const int what = rand() % 10;
            if (what == 0 && (kinds & 2)) {  // a launch a level
                for (int l = 0; l < 5; ++l) d.ctr[s][l] = 1;
                continue;
            }
            const bool zero_other = sets.zero_other();
            if (what == 1 && (kinds & 4)) continue;  // the launch fails: nothing ran
            sets.launched();
            const bool before = d.gave_up;
            if (what == 2 && (kinds & 1)) d.gave_up = true;
            // a block that starts late may find this launch's own give-up
            const bool seen = before || (d.gave_up && rand() % 2);
            if (zero_other) {
                const int used = imi::set_entries_used(seen, d.levels[o], kAll);
                for (int i = 0; i < used; ++i) d.ctr[o][i] = 0;
                d.levels[o] = 0;
            }
            if (before) continue;  // no level runs, none is recorded
            if (d.gave_up) {
                // its blocks come to different levels
                d.levels[s] = rand() % 5;
                for (int l = d.levels[s] + rand() % 3; l >= 0; --l) d.ctr[s][l] = 3;
                continue;
            }
            const int levels = 1 + rand() % (kAll - 3);
            for (int l = 0; l < levels; ++l) d.ctr[s][l] = 1 + rand() % 5;
            d.levels[s] = levels;
        }
    }
    puts("ok");
    return 0;
}
"""


def _run(tmp_path, kinds):
    src = tmp_path / "sets.cpp"
    src.write_text(MODEL)
    exe = tmp_path / "sets"
    try:
        r = subprocess.run(["g++", "-std=c++17", "-O1", "-I", CSRC, str(src), "-o", str(exe)], capture_output=True,
                           text=True)
    except FileNotFoundError:
        pytest.skip("no C++ compiler")
    assert r.returncode == 0, r.stderr[-2000:]
    r = subprocess.run([str(exe), str(kinds)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout


@pytest.mark.parametrize("kinds", [0, 1, 2, 4, 7], ids=["complete", "give_up", "per_level", "launch_fails", "all"])
def test_a_set_is_zero_when_its_phase_begins(tmp_path, kinds):
    _run(tmp_path, kinds)
