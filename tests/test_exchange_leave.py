"""The counted exchanges of a cluster whose waits give up (csrc/harp_exchange.h), compiled for the host: four CTAs in turn, two exchanges, a piece that
comes late or not at all.  No piece lands in a CTA that has ended, and every CTA ends."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include <ucontext.h>
#include <vector>
#include "harp_exchange.h"

constexpr int kCtas = 4, kPhases = 3;
constexpr uint32_t kMask = 5, kLimit = 100;              // phases 0 and 2 end in an exchange
struct Piece { int to, phase; long due; };
std::vector<Piece> flying;
int got[kCtas][kPhases], stored[kCtas], wrong = 0;
bool ended[kCtas], here[kCtas], lost[kCtas], leave;
int late_from, late_to, late_phase;
long late_by, now = 0;
ucontext_t scheduler, ctx[kCtas];
std::vector<char> stacks[kCtas];

void cta(int self) {
    auto turn = [&] { swapcontext(&ctx[self], &scheduler); };
    auto arrived = [&](int p) { turn(); return got[self][p] == kCtas; };
    for (int p = 0; p < kPhases; ++p) {
        turn();
        if (!((kMask >> p) & 1u)) continue;
        for (int to = 0; to < kCtas; ++to) {
            const bool late = self == late_from && to == late_to && p == late_phase;
            if (!lost[self] && !(late && late_by < 0)) flying.push_back({to, p, now + (late ? late_by : 3)});
        }
        if (!exchange_wait(kLimit, [&] { return arrived(p); })) lost[self] = true;
    }
    if (!lost[self]) stored[self] = 1;
    if (lost[self] && leave)
        exchange_leave(kMask, kLimit, [&] {
            here[self] = true;
            for (int n = 0; n < kCtas; ++n)
                while (!here[n] && !ended[n]) turn();
        }, arrived);
    ended[self] = true;
    for (;;) turn();
}

int main(int argc, char **argv) {
    leave = atoi(argv[1]);
    late_from = atoi(argv[2]); late_to = atoi(argv[3]); late_phase = atoi(argv[4]); late_by = atol(argv[5]);
    for (int n = 0; n < kCtas; ++n) {
        stacks[n].resize(1 << 16);
        getcontext(&ctx[n]);
        ctx[n].uc_stack.ss_sp = stacks[n].data();
        ctx[n].uc_stack.ss_size = stacks[n].size();
        makecontext(&ctx[n], (void (*)())cta, 1, n);
    }
    for (; now < 5000; ++now) {
        for (size_t k = 0; k < flying.size();)
            if (flying[k].due <= now) {
                wrong += ended[flying[k].to];
                ++got[flying[k].to][flying[k].phase];
                flying.erase(flying.begin() + k);
            } else ++k;
        for (int n = 0; n < kCtas; ++n) swapcontext(&scheduler, &ctx[n]);
    }
    int n_ended = 0, n_lost = 0, n_stored = 0;
    for (int n = 0; n < kCtas; ++n) { n_ended += ended[n]; n_lost += lost[n]; n_stored += stored[n]; }
    printf("%d %d %d %d\n", n_ended, n_lost, n_stored, wrong);
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    d = tmp_path_factory.mktemp("exchange")
    (d / "x.cc").write_text(PROGRAM)
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-I", os.path.join(ROOT, "paper_2605_29843_b200", "csrc"), str(d / "x.cc"), "-o", str(d / "x")])
    return lambda *a: [int(v) for v in subprocess.check_output([str(d / "x"), *map(str, a)]).split()]


def test_every_piece_in_time(program):
    assert program(1, 0, 1, 0, 3) == [4, 0, 4, 0]


@pytest.mark.parametrize("phase", [0, 2])
@pytest.mark.parametrize("late_by", [-1, 101, 150, 199])
def test_a_piece_that_comes_after_the_limit_or_never(program, phase, late_by):
    """The CTA that waits for it stores nothing, and is still there when it lands, up to as long again."""
    ended, lost, stored, wrong = program(1, 0, 1, phase, late_by)
    assert ended == 4 and lost >= 1 and stored == 4 - lost
    assert wrong == 0


def test_the_model_sees_a_cta_that_leaves_at_once(program):
    assert program(0, 0, 1, 2, 150)[3] > 0
