"""The cluster engine's plan of a batch on devices that lack some cluster sizes (CPU only): whatever is
missing, the default call gets a plan that the device can run, or the row engine, and never an error."""
import shutil
import subprocess
from pathlib import Path

import pytest

ROOT = Path(__file__).resolve().parents[1]

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include <vector>
#include "pk_batched_plan.h"
struct Fake {
  int largest[3];  // the largest cluster of each shape, 0: none
  int shapes() const { return 3; }
  int max_rows(int s) const { return 4096 >> s; }
  int capacity(int s, int C) const { return C <= largest[s] ? (304 << s) / C : 0; }
};
int main(int argc, char** argv) {  // largest clusters of the three shapes, wanted rows, sizes
  Fake d{{std::atoi(argv[1]), std::atoi(argv[2]), std::atoi(argv[3])}};
  std::vector<int> n, cls;
  for (int k = 5; k < argc; ++k) n.push_back(std::atoi(argv[k]));
  cls.resize(n.size());
  std::printf("%d", pk::choose_clusters(d, n.data(), (int)n.size(), std::atoi(argv[4]), 2048, cls.data()));
  for (int c : cls) std::printf(" %d", c);
  std::printf("\n");
}
"""


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    if shutil.which("g++") is None:  # pragma: no cover
        pytest.skip("g++ not available")
    d = tmp_path_factory.mktemp("plan")
    (d / "p.cpp").write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-I", str(ROOT / "paper_1410_4054_gb300" / "csrc"), "-o", str(d / "p"),
                    str(d / "p.cpp")], check=True)

    def run(largest, wanted, sizes):
        out = subprocess.run([str(d / "p")] + [str(v) for v in (*largest, wanted, *sizes)], check=True,
                             capture_output=True, text=True).stdout.split()
        return int(out[0]), [int(v) for v in out[1:]]

    return run


SIZES = [[8000], [65536], [1, 31, 1024, 4097, 8193, 32768, 65536], [8200] * 40, [4096] * 600, [0, 5]]


@pytest.mark.parametrize("sizes", SIZES, ids=lambda v: f"{len(v)}x{max(v)}")
@pytest.mark.parametrize("largest", [(16, 16, 16), (8, 8, 8), (4, 8, 8), (0, 16, 16), (2, 0, 0), (0, 0, 0)], ids=str)
@pytest.mark.parametrize("wanted", [0, 4096])
def test_plan_fits_what_the_device_has(plan, largest, wanted, sizes):
    rc, cls = plan(largest, wanted, sizes)
    if rc < 0:  # no clusters: neither the plan asked for nor the fixed one can hold every system
        assert max(sizes) > 2048 * largest[1] and max(sizes) > 4096 * largest[0]
        return
    for n, c in zip(sizes, cls):
        shape, C = c // 5, 1 << (c % 5)
        assert C <= largest[shape]
        share = max(32, (-(-n // C) + 31) // 32 * 32)
        assert share <= 4096 >> shape


def test_automatic_plan_without_the_largest_clusters(plan):
    # two systems do not fill the device: 512 rows per CTA (256 for a system of up to 1,024), clusters of 16
    # where there are any
    assert plan((16, 16, 16), 0, [8000, 300]) == (0, [4, 1])
    assert plan((8, 8, 8), 0, [8000, 300]) == (0, [3, 1])
    # nothing of shape 0: the fixed plan's shape; clusters too small for the largest system: the row engine
    assert plan((0, 16, 16), 0, [8000, 300]) == (2048, [5 + 2, 5])
    assert plan((8, 8, 8), 0, [65536, 300])[0] == -1
