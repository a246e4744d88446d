"""Which domains of a batch run on the resident kernel (host code, built here
with the system compiler against a stand-in for the GPU): groups by launch
shape, and the queue for every domain whose clusters the GPU, or the part of it
a process has, cannot hold."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2311_16080_gb300", "csrc")

# argv: the largest cluster the GPU holds, then per domain blocks, threads,
# bytes and whether a thread takes one cell; prints the groups and the rest
MAIN = r"""
#include <stdio.h>
#include <stdlib.h>
#include "batch_groups.h"
int main(int argc, char** argv) {
  const int largest = atoi(argv[1]), n = (argc - 2) / 4;
  std::vector<xlb::ResidentShape> s;
  std::vector<int> ord;
  for (int d = 0; d < n; ++d) {
    char** a = argv + 2 + 4 * d;
    s.push_back({atoi(a[0]), atoi(a[1]), atoi(a[2]), atoi(a[3]) != 0});
    ord.push_back(d);
  }
  const xlb::DomainGroups g = xlb::group_domains(
      ord, [&](int d) { return s[d]; }, [&](const xlb::ResidentShape& q) { return q.ctas <= largest; });
  for (const auto& b : g.buckets) {
    printf("%d %d %lld %d:", b.shape.ctas, b.shape.threads, b.shape.smem, (int)b.shape.one);
    for (int k = 0; k < b.count; ++k) printf(" %d", g.order[b.first + k]);
    printf("\n");
  }
  printf("rest:");
  for (int k = n - g.n_rest; k < n; ++k) printf(" %d", g.order[k]);
  printf("\n");
  return (int)g.order.size() == n ? 0 : 1;
}
"""


@pytest.fixture(scope="module")
def grouped(tmp_path_factory):
    if not shutil.which("g++"):
        pytest.skip("no g++")
    d = tmp_path_factory.mktemp("groups")
    (d / "main.cpp").write_text(MAIN)
    subprocess.run(["g++", "-std=c++17", "-I", CSRC, str(d / "main.cpp"), "-o", str(d / "main")], check=True)

    def run(largest, shapes):
        args = [str(v) for s in shapes for v in s]
        return subprocess.run([str(d / "main"), str(largest)] + args, check=True, capture_output=True,
                              text=True).stdout.splitlines()

    return run


# largest first: no cluster, 8 blocks, 4 blocks, 2 x 1 block (one large), 3 x 1 block
SHAPES = [(0, 0, 0, 0), (8, 768, 220000, 0), (4, 768, 200000, 0), (1, 768, 180000, 0), (1, 768, 190000, 0),
          (1, 384, 100000, 0), (1, 1024, 39000, 1), (1, 64, 2000, 1)]


def test_groups_by_shape(grouped):
    assert grouped(16, SHAPES) == ["8 768 220000 0: 1", "4 768 200000 0: 2", "1 768 190000 0: 3 4",
                                   "1 384 100000 0: 5 6 7", "rest: 0"]
    assert grouped(16, SHAPES[6:]) == ["1 1024 39000 1: 0 1", "rest:"]


@pytest.mark.parametrize("largest,rest", [(8, "0"), (4, "0 1"), (2, "0 1 2"), (0, "0 1 2 3 4 5 6 7")])
def test_clusters_without_room_take_the_queue(grouped, largest, rest):
    got = grouped(largest, SHAPES)
    assert got[-1] == "rest: " + rest
    assert all(int(line.split()[0]) <= largest for line in got[:-1])
