"""The full barriers of a ring that two consumer groups take in turn
(csrc/ring_turns.h), against a model of mbarrier phases on the CPU: a wait by
parity passes whenever the phase in progress has the other parity, copies land
in any order, groups run at any pace.  No wait may pass before its fill has
landed, and none may wait for ever.  One barrier per buffer fails this for every odd
ring, which the model shows too."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2608_07152_gb300", "csrc")

MODEL = r"""
#include <cstdio>
#include <cstdlib>
#include <random>
#include <vector>
#include "ring_turns.h"
using namespace pvs;

// One run of n fills: 0, or 1 for a wait that passed early, or 2 for a standstill.
static int run(int stages, bool one_bar, int n, unsigned seed) {
    std::mt19937 rng(seed);
    const int bars = one_bar ? stages : turn_bars(stages);
    auto bar_of = [&](int k) { return one_bar ? k % stages : turn_bar(k, stages); };
    auto parity_of = [&](int k) {
        return one_bar ? (unsigned)(k / stages) & 1u : turn_parity(k, stages);
    };
    auto buffer_of = [&](int k) {
        return one_bar ? k % stages : turn_buffer(turn_bar(k, stages), stages);
    };
    std::vector<unsigned> full(bars, 0), empty(stages, 0);   // phases completed
    auto passes = [](unsigned phases, unsigned parity) { return (phases & 1u) != parity; };
    std::vector<char> landed(n, 0);
    std::vector<int> flying;
    int next = 0, at[2] = {0, 1};
    const int slow = (int)(rng() % (unsigned)n);   // one copy that takes long
    int held = (int)(rng() % 400u);
    for (int step = 0; step < 20000 + 400 * n; ++step) {
        if (next == n && flying.empty() && at[0] >= n && at[1] >= n) return 0;
        switch (rng() % 4u) {
            case 0:   // the producer
                if (next < n && passes(empty[buffer_of(next)], ((unsigned)(next / stages) & 1u) ^ 1u)) {
                    flying.push_back(next);
                    ++next;
                }
                break;
            case 1: {   // a copy lands
                if (flying.empty()) break;
                const size_t i = rng() % flying.size();
                const int k = flying[i];
                if (k == slow && held-- > 0) break;
                landed[k] = 1;
                ++full[bar_of(k)];
                flying.erase(flying.begin() + (long)i);
                break;
            }
            default: {   // a group waits, reads and hands the buffer back
                const int g = (int)(rng() & 1u);
                const int k = at[g];
                if (k >= n || !passes(full[bar_of(k)], parity_of(k))) break;
                if (!landed[k]) return 1;
                ++empty[buffer_of(k)];
                at[g] += 2;
                break;
            }
        }
        if (next == n)   // the producer's drain: the last copy counted on each barrier
            for (int b = 0; b < bars && b < n; ++b) {
                const int last = n - 1 - ((n - 1 - b) % bars);
                if (passes(full[b], parity_of(last)) && !landed[last]) return 1;
            }
    }
    return 2;
}

int main(int argc, char** argv) {
    const int stages = atoi(argv[1]), one_bar = atoi(argv[2]);
    int worst = 0;
    for (unsigned seed = 0; seed < 4000 && worst == 0; ++seed) {
        const int r = run(stages, one_bar != 0, 1 + (int)(seed % 61u), seed);
        worst = r > worst ? r : worst;
    }
    // the walk itself: every buffer and barrier in range, a barrier for one group only
    if (!one_bar)
        for (int k = 0; k < 1000; ++k) {
            const int b = turn_bar(k, stages);
            if (b < 0 || b >= turn_bars(stages) || (b & 1) != (k & 1) ||
                turn_buffer(b, stages) != k % stages)
                worst = 3;
        }
    printf("%d\n", worst);
    return 0;
}
"""


@pytest.fixture(scope="module")
def model(tmp_path_factory):
    d = tmp_path_factory.mktemp("ring")
    src, exe = d / "model.cpp", d / "model"
    src.write_text(MODEL)
    subprocess.run(["g++", "-O2", "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    return lambda stages, one_bar: int(subprocess.run(
        [str(exe), str(stages), str(int(one_bar))], check=True, capture_output=True,
        text=True).stdout)


@pytest.mark.parametrize("stages", range(2, 9))
def test_no_wait_passes_before_its_fill(model, stages):
    assert model(stages, False) == 0
    # one barrier per buffer: early for every odd ring, and only there
    assert model(stages, True) == stages % 2


KERNELS = ["interval_group.cu", "batch_stream.cu"]


@pytest.mark.parametrize("name", KERNELS)
def test_kernels_take_their_full_barriers_from_it(name):
    text = open(os.path.join(CSRC, name)).read()
    assert '#include "ring_turns.h"' in text and "turn_bars(" in text
    for line in text.splitlines():   # by the fill's own barrier, never by its buffer
        assert "full[s]" not in line, line
