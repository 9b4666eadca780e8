"""The time the batched solver's path choice gives an iteration on the single-problem path
(csrc/batch_rule.h), on the CPU: a problem on its own takes the time measured alone, the
more problems share the path's workers the less each takes, down to the eight workers'
figure, and an iteration is counted per sigma build."""
import os
import shutil
import subprocess

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2405_10197_gb300", "csrc")

DRIVER = """
#include "batch_rule.h"
#include <cstdio>
int main() {
  for (int mixed = 0; mixed < 2; ++mixed)
    for (int nroots = 1; nroots <= 3; ++nroots)
      for (int p = 1; p <= 100; ++p) printf("%d %d %d %.17g\\n", mixed, nroots, p, forte::single_path_ms(3.0, nroots, mixed, p));
}
"""


def test_single_path_time_follows_the_problems_in_flight(tmp_path):
    src, exe = tmp_path / "rule.cpp", str(tmp_path / "rule")
    src.write_text(DRIVER)
    subprocess.run([shutil.which("g++"), "-std=c++17", "-I", CSRC, str(src), "-o", exe], check=True)
    t = {}
    for line in subprocess.run([exe], capture_output=True, text=True, check=True).stdout.splitlines():
        m, r, p, v = line.split()
        t[int(m), int(r), int(p)] = float(v)
    assert t[0, 1, 1] == 3.0
    for r in (1, 2, 3):
        for p in range(1, 101):
            assert abs(t[0, r, p] * r - t[0, 1, p]) < 1e-12
            assert abs(t[1, r, p] - 0.72 * t[0, r, p]) < 1e-12
            # one more problem makes none slower, and all of them no faster
            if p < 100:
                assert t[0, r, p + 1] <= t[0, r, p] and (p + 1) * t[0, r, p + 1] > p * t[0, r, p]
            if p >= 8:
                assert t[0, r, p] == t[0, r, 8]
    assert 0.27 * 3 < t[0, 1, 8] < 0.46 * 3 and 0.43 * 3 < t[0, 1, 3] < 0.72 * 3  # as measured
