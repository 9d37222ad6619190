"""The rule that sends a dense product to CTA pairs or to the tiled kernel, compiled for the host, against what both were measured to take."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

MAIN = r"""
#include <initializer_list>
#include <cstdio>
#include "pair_rules.cuh"
int main() {
  int M, N, K, order;
  while (std::scanf("%d %d %d %d", &M, &N, &K, &order) == 4) {
    double cost;
    cafeq::t2_width(M, N, 0, &cost);
    std::printf("%d\n", (int)cafeq::t2_wanted(M, N, K, order, cost));
  }
}
"""

# M, N, K, order, time on tiles minus time on pairs (us, one call)
MEASURED = [
    (512, 512, 512, 2, -2.1), (512, 512, 2048, 2, 4.5), (512, 512, 3584, 2, 10.8), (1024, 1024, 512, 2, -4.1), (1024, 1024, 2048, 2, 3.1),
    (1024, 1024, 3584, 2, 7.1), (1024, 2560, 1024, 2, 13.9), (1024, 2560, 1536, 2, 21.3), (2560, 1024, 1024, 2, 14.0),
    (1536, 3584, 1536, 2, 8.7), (3584, 1536, 1536, 2, 9.3), (2048, 2048, 512, 2, -12.4), (2048, 2048, 1536, 2, -9.2),
    (2048, 2048, 3584, 2, 4.1), (2048, 3584, 512, 2, -9.4), (2048, 3584, 3584, 2, 18.7), (3584, 3584, 512, 2, -16.5),
    (3584, 3584, 1024, 2, -8.2), (3584, 3584, 3584, 2, 22.1), (3072, 3584, 512, 2, -20.9), (3072, 3584, 1024, 2, -17.4),
    (4608, 4608, 512, 2, -26.3), (4608, 4608, 1536, 2, -6.3), (4608, 4608, 3584, 2, 43.0), (256, 256, 512, 3, 3.7), (256, 4608, 512, 3, 7.9),
    (1024, 1024, 512, 3, 7.4), (1024, 1024, 2048, 3, 18.2), (2048, 2048, 2048, 3, 13.3), (3584, 3584, 512, 3, 22.2), (4608, 4608, 3584, 3, 97.8),
]


def test_rule_follows_the_measurements(tmp_path):
    (tmp_path / "main.cpp").write_text(MAIN)
    exe = str(tmp_path / "rule")
    subprocess.run(["g++", "-std=c++17", "-x", "c++", "-I", os.path.join(ROOT, "paper_2511_19705_b200", "csrc"), "-o", exe, str(tmp_path / "main.cpp")],
                   check=True)
    lines = "\n".join(" ".join(map(str, m[:4])) for m in MEASURED)
    got = subprocess.run([exe], input=lines, capture_output=True, text=True, check=True).stdout.split()
    assert [int(g) for g in got] == [int(m[4] > 0) for m in MEASURED]
