"""The wait for loads in flight after a wait that gave up (csrc/harp_ring.h), compiled for the host and replayed against a model of
the barriers, in the kernels' order of steps: a CTA whose wait gave up stores nothing more and does not end while a load of its own is in flight."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include "harp_ring.h"

constexpr int kBuf = 3, kTiles = 11;
constexpr uint32_t kLimit = 100;

int main(int argc, char **argv) {
    const int late_tile = atoi(argv[1]), late_by = atoi(argv[2]);
    // barrier of a buffer: completed phases, and the time at which the load in flight completes the next one (-1: none)
    int completed[kBuf] = {0}, due[kBuf] = {-1, -1, -1}, now = 0;
    auto arrive = [&]() {
        for (int b = 0; b < kBuf; ++b)
            if (due[b] >= 0 && now >= due[b]) { due[b] = -1; ++completed[b]; }
    };
    auto try_phase = [&](int b, uint32_t parity) {
        ++now;
        arrive();
        return (completed[b] & 1) != (int)parity;
    };
    uint32_t parity = 0;
    bool dead = false;
    int stored = 0, wrong = 0, held[kBuf] = {-1, -1, -1};
    auto load = [&](int tile, int b) {
        wrong += due[b] >= 0;                          // over a load that has not arrived
        held[b] = tile;
        due[b] = now + (tile == late_tile ? late_by : 5);
    };
    for (int k = 0; k < kBuf && k < kTiles; ++k) load(k, k);
    for (int t = 0, b = 0; t < kTiles; ++t, b = b + 1 == kBuf ? 0 : b + 1) {
        for (uint32_t it = 0; !try_phase(b, (parity >> b) & 1u);)
            if (++it > kLimit || ((it & 63) == 63 && dead)) {
                dead = true;
                parity ^= 1u << b;
                break;
            }
        parity ^= 1u << b;
        if (t > 0 && t + kBuf - 1 < kTiles && !dead) load(t + kBuf - 1, b == 0 ? kBuf - 1 : b - 1);
        if (!dead) { wrong += held[b] != t || due[b] >= 0; ++stored; }
    }
    const int before = now;
    if (dead) ring_drain(parity, kBuf, kLimit, try_phase);
    int in_flight = 0;
    for (int b = 0; b < kBuf; ++b) in_flight += due[b] >= 0;
    printf("%d %d %d %d %d\n", (int)dead, stored, wrong, in_flight, now - before);
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    d = tmp_path_factory.mktemp("ring")
    (d / "ring.cc").write_text(PROGRAM)
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-Wall", "-Werror", "-I", os.path.join(ROOT, "paper_2605_29843_b200", "csrc"),
                           str(d / "ring.cc"), "-o", str(d / "ring")])
    return lambda *a: [int(v) for v in subprocess.check_output([str(d / "ring"), *map(str, a)]).split()]


def test_every_load_in_time(program):
    assert program(-1, 0) == [0, 11, 0, 0, 0]


@pytest.mark.parametrize("tile", range(11))
@pytest.mark.parametrize("late_by", [110, 150, 190])
def test_a_load_that_arrives_after_the_limit(program, tile, late_by):
    """The wait takes 100 attempts; the drain at most as many again for each of the three buffers."""
    dead, stored, wrong, in_flight, attempts = program(tile, late_by)
    assert dead == 1 and stored == tile and wrong == 0
    assert in_flight == 0 and attempts <= 3 * 101
