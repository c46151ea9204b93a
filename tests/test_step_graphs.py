"""Which recorded graphs a call of fsl_step takes (next_graph of the library's own
header, compiled for the host): the steps add up, every pair starts where the graph
says, and a caller who repeats one count records graphs in the first call only."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

MAIN = r"""
#include <cstdio>
#include "fsl_internal.cuh"
int main() {
    for (int left = 1; left <= 1000; ++left)
        for (int parity = 0; parity < 2; ++parity) printf("%d %d %d\n", left, parity, fslk::next_graph(left, parity));
}
"""


@pytest.fixture(scope="module")
def graph_of(tmp_path_factory):
    from paper_1509_07691_gb300 import build as b
    d = tmp_path_factory.mktemp("graphs")
    (d / "m.cu").write_text(MAIN)
    subprocess.run([b.nvcc(), "-std=c++17", "--expt-relaxed-constexpr", *b.ARCH, "-I", b.INCLUDE, "-I", b.CSRC, str(d / "m.cu"),
                    "-o", str(d / "m")], check=True, capture_output=True)
    out = subprocess.run([str(d / "m")], check=True, capture_output=True, text=True).stdout
    shutil.rmtree(d)
    return {(a, p): k for a, p, k in (map(int, line.split()) for line in out.splitlines())}


def _call(graph_of, recorded, parity, n):
    """One fsl_step(n): (new parity, graphs recorded, launches)."""
    new, launches, single = 0, 0, False
    while n:
        k = graph_of[(n, parity)]
        assert k & 1 == parity and n >= (1 if k < 2 else 2)
        new += k not in recorded
        recorded.add(k)
        steps = 1 if k < 2 else 2
        single = single or steps == 1
        parity ^= steps & 1
        n -= steps
        launches += 1
    if single and parity not in recorded:  # with a single step's graph the other parity's is recorded
        recorded.add(parity)
        new += 1
    return parity, new, launches


@pytest.mark.parametrize("n", range(1, 21))
def test_repeated_counts_record_in_the_first_call(graph_of, n):
    recorded, parity = set(), 0
    for call in range(4):
        parity, new, launches = _call(graph_of, recorded, parity, n)
        assert launches == (n + 1) // 2
        assert new == 0 or call == 0


@pytest.mark.parametrize("counts", [(1000, 5, 1, 1, 1), (4, 1, 1, 3, 2), (5, 5, 1, 4, 7), (3, 1, 2, 1)])
def test_single_steps_after_a_run_wait_for_no_graph(graph_of, counts):
    """Once a single step was taken no later single step records."""
    recorded, parity, seen = set(), 0, False
    for n in counts:
        before = set(recorded)
        parity, _, _ = _call(graph_of, recorded, parity, n)
        if seen:
            assert {0, 1} <= before
        seen = seen or n % 2 == 1
