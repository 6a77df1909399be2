"""The integer sum of a chain's accumulators (csrc/mp_fp64_join.h), compiled for the host: at the
ends of every accumulator's range, in all combinations of signs, it is the exact weighted sum."""
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2602_02507_gb300", "csrc")

PROGRAM = r"""
#include "mp_fp64_join.h"
#include <cstdio>
template <int DS> int check()
{
    using J = mp::ChainJoin<DS>;
    int bad = 0;
    // accumulators 0 .. 2 up to 2^22 (the limit of the form), 3 and 4 up to (s + 1) 2^21
    const long long top[6] = {1 << 22, 1 << 22, 1 << 22, 4 << 21, 5 << 21, 1 << 22};
    for (int pick = 0; pick < 729; ++pick) {
        long long x[6], want = 0;
        for (int s = 0, v = pick; s < 6; ++s, v /= 3) x[s] = (v % 3 - 1) * top[s];
        const int shift[6] = {40, 32, 24, 16, 8, 0};
        for (int s = 0; s < 6; ++s) want += x[s] * ((1ll << shift[s]) >> (s < 5 ? DS : 0));
        const uint64_t got = J::sum(mp::kFloatOff + (uint32_t)x[0], mp::kFloatOff + (uint32_t)x[1],
                                    mp::kFloatOff + (uint32_t)x[2], mp::kThirdPairOff + (uint32_t)x[3],
                                    (uint32_t)x[4], mp::kFloatOff + (uint32_t)x[5]) - J::offset;
        bad += (long long)got != want;
    }
    return bad;
}
int main() { std::printf("%d %d\n", check<2>(), check<4>()); return 0; }
"""


def test_sums_at_the_ends_of_the_range(tmp_path):
    src = tmp_path / "join.cpp"
    src.write_text(PROGRAM)
    exe = tmp_path / "join"
    subprocess.run(["g++", "-std=c++17", "-O1", "-Wall", "-Werror", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    assert subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split() == ["0", "0"]
