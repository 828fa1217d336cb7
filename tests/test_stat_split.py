"""How the statistics pass is split (csrc/stat_split.hpp) where the stream's context cannot place the cluster that the sizes ask for:
the rule compiled for the host with an answer of the driver's that the test gives."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2609_33135_b200", "csrc")
MAIN = """
#include <cstdio>
#include "stat_split.hpp"
int main() {
  long long heads; int N, slices, n_sm, largest;   // largest cluster that can be placed
  while (scanf("%lld %d %d %d %d", &heads, &N, &slices, &n_sm, &largest) == 5) {
    const mpfa::StatSplit s = mpfa::stat_split(heads, N, slices, 2, n_sm, [&](int c) { return c <= largest; });
    printf("%d %d\\n", s.slices, (int)s.clusters);
  }
}
"""


@pytest.fixture(scope="module")
def split(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("split") / "split")
    subprocess.run(["g++", "-std=c++17", "-Wall", "-Werror", "-I" + CSRC, "-x", "c++", "-", "-o", exe], input=MAIN, text=True, check=True)

    def ask(cases):
        text = "\n".join(" ".join(map(str, c)) for c in cases)
        out = subprocess.run([exe], input=text, capture_output=True, text=True, check=True).stdout
        return [tuple(map(int, line.split())) for line in out.splitlines()]
    return ask


def test_every_size_where_all_clusters_can_be_placed(split):
    cases = [(2, 256, 32, 148, 16), (2, 10240, 32, 148, 16), (2, 10241, 32, 148, 16), (3, 2049, 32, 148, 16), (40, 777, 32, 148, 16),
             (1088, 257, 32, 148, 16), (2, 256, 1, 148, 16), (2, 4096, 3, 148, 16), (40, 16384, 32, 148, 16)]
    assert split(cases) == [(2, 1), (16, 1), (20, 0), (16, 1), (4, 1), (1, 0), (1, 0), (3, 0), (7, 0)]


def test_smaller_clusters_and_slices_where_a_context_has_no_room(split):
    """A cluster that the driver cannot place is never asked for: half of it while its slices stay short, otherwise slices and a fold."""
    #        heads, N, slices of the workspace, SMs, largest that can be placed
    cases = [(2, 4096, 32, 148, 8), (2, 4096, 32, 148, 4), (2, 10240, 32, 148, 8), (2, 256, 32, 148, 1), (2, 256, 32, 148, 0), (40, 777, 32, 148, 2),
             (2, 5120, 5, 148, 0)]
    assert split(cases) == [(8, 1), (8, 0), (20, 0), (1, 0), (1, 0), (2, 1), (5, 0)]


def test_no_cluster_beyond_what_can_be_placed(split):
    cases = [(h, n, s, m, p) for h in (1, 2, 5, 10, 40, 100, 1000) for n in (1, 128, 129, 640, 1281, 2049, 5120, 10240, 10241, 131072)
             for s in (1, 2, 7, 32) for m in (8, 20, 148) for p in (0, 1, 2, 4, 8, 16)]
    for c, (slices, clusters) in zip(cases, split(cases)):
        heads, N, most, n_sm, largest = c
        assert 1 <= slices <= max(1, most), c
        if clusters:
            assert slices in (2, 4, 8, 16) and slices <= largest and N <= 640 * slices, c
        else:
            assert slices == 1 or slices * heads <= 2 * n_sm, c
