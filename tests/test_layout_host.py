"""Threads per candidate of a plan: what ATP_OPT_LANES forces is what runs, at
every size, and the default's lines, from the header the launches use."""
import os
import subprocess

import pytest

from paper_2603_20525_gb300 import build

PROGRAM = """
#include <cstdio>
#include <cstdlib>
#include "plan_kernel.cuh"
int main(int argc, char **argv)
{
    for (int i = 1; i + 1 < argc; i += 2) {
        const int f = atoi(argv[i]), n = atoi(argv[i + 1]), l = atp::plan_layout(f, n);
        printf("%d %d %lld\\n", l, atp::plan_lanes(f, n), atp::layout_ctas(l, n));
    }
}
"""


@pytest.fixture(scope="module")
def layouts(tmp_path_factory):
    d = tmp_path_factory.mktemp("layout")
    src, exe = os.path.join(d, "l.cu"), os.path.join(d, "l")
    with open(src, "w") as f:
        f.write(PROGRAM)
    subprocess.run([build.nvcc(), build.ARCH, "-std=c++17", f"-I{build.INCLUDE}", f"-I{build.CSRC}", src, "-o", exe],
                   check=True)

    def run(pairs):
        out = subprocess.run([exe, *[str(v) for p in pairs for v in p]], check=True, capture_output=True, text=True)
        return [tuple(map(int, line.split())) for line in out.stdout.splitlines()]
    return run


def test_a_forced_layout_runs_at_every_size(layouts):
    pairs = [(f, n) for f in (1, 2, 4) for n in (1, 63, 1000, 4864, 4865, 16384, 29184, 100000, 2 ** 31 - 1025)]
    for (f, n), (threads, lanes, ctas) in zip(pairs, layouts(pairs)):
        assert threads == f and lanes == f and ctas == -(-n * f // 64)


def test_the_default_goes_from_eight_threads_to_one(layouts):
    sizes = [1, 4864, 4865, 16384, 16385, 29184, 29185, 10 ** 6]
    got = layouts([(0, n) for n in sizes])
    assert [g[0] for g in got] == [8, 8, 4, 4, 2, 2, 1, 1]
    assert [g[1] for g in got] == [4, 4, 4, 4, 2, 2, 1, 1]
