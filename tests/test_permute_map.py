"""Places of a row's elements in the shared memory of the permutation kernels (csrc/harp_permute.h), replayed on the host for every width
that the kernels take: one place an element, inside its own row, whole 16-byte pieces."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <cstdio>
#include <vector>
#include "harp_permute.h"

template <int V>
int check(int d) {
    const int pitch = permute_pitch<V>(d);
    if (pitch < d || pitch >= d + 8 * V || pitch % V) return 1;
    std::vector<char> taken(pitch, 0);
    for (int i = 0; i < d; ++i) {
        const int at = permute_place<V>(i);
        if (at < 0 || at >= pitch || taken[at]) return 2;
        taken[at] = 1;
        if (at % V != i % V || at / V != permute_piece<V>(i / V)) return 3;
    }
    return (d / V) % 8 == 0 && pitch != d ? 4 : 0;
}

int main() {
    int bad = 0, n = 0;
    for (int d = 4; d <= 32768; d += d < 4096 ? 4 : 1004, ++n) {
        const int f32 = check<4>(d), bf16 = d % 8 == 0 ? check<8>(d) : 0;
        if (f32 || bf16) { printf("d = %d: fp32 %d, bf16 %d\n", d, f32, bf16); ++bad; }
    }
    printf("%d of %d wrong\n", bad, n);
    return bad != 0;
}
"""


def test_every_element_has_a_place_of_its_own_in_its_row(tmp_path):
    (tmp_path / "map.cc").write_text(PROGRAM)
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-Wall", "-Werror", "-I", os.path.join(ROOT, "paper_2605_29843_b200", "csrc"),
                           str(tmp_path / "map.cc"), "-o", str(tmp_path / "map")])
    r = subprocess.run([str(tmp_path / "map")], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
