"""Which scratch set a step takes, and when it has to wait for all earlier work of its stream (csrc/sets.h).  Checked by a small C++
program built from the header itself (no GPU needed)."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <cstdio>
#include <random>
#include "sets.h"
using namespace mvla;
// Calls in any order, captured or not, some of which fail: a set that a step re-arms while the step before it on the stream may still run is not that step's.
// (A captured step runs when its graph does, which is ordered as a whole; so a stream capture is a stream of its own here, and each has a new number.)
int main()
{
    for (int seed = 0; seed < 2000; ++seed) {
        std::mt19937 rng(seed);
        SetRing r;
        int last = -1, last_captured = -1, waits = 0;      // set of the step that was enqueued last
        unsigned long long capture = 0, captures = 0;
        for (int i = 0; i < 60; ++i) {
            if (rng() % 4 == 0) {
                capture = capture ? 0 : ++captures;
                last_captured = -1;
            }
            const SetRing::Turn t = r.take(capture);
            int& before = capture ? last_captured : last;
            if (static_cast<int>(t.set) == before && !t.wait) { std::printf("order %d: step %d takes the set of the one before it\n", seed, i); return 1; }
            if (rng() % 3 == 0) continue;                  // the call fails
            r.done();
            before = static_cast<int>(t.set);
        }
        // undisturbed steps do not wait, and two of them with the same set are kSets apart
        for (unsigned i = 0, first = 0; i < 2 * kSets + 1; ++i) {
            const SetRing::Turn t = r.take(capture);
            r.done();
            if (i == 0) { first = t.set; continue; }
            waits += t.wait;
            if ((t.set == first) != (i % kSets == 0)) { std::printf("rotation\n"); return 1; }
        }
        if (waits) { std::printf("waits without need\n"); return 1; }
    }
    std::printf("ok\n");
    return 0;
}
"""


def test_a_step_never_re_arms_the_set_of_the_step_before_it(tmp_path):
    src, exe = tmp_path / "sets.cpp", tmp_path / "sets"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", os.path.join(ROOT, "paper_2604_09244_b200", "csrc"), "-o", str(exe), str(src)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout
