"""The control flow of the rings of bulk copies, on the CPU: a chunk that never arrives is not used, nothing is requested
behind it, and every chunk that was requested is waited for."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2411_05289_b200", "csrc")
SOURCE = r"""
#include <cstdio>
#include <cstdlib>
#include "spechub_ring_run.h"
int main(int argc, char **argv) {
    const int chunks = atoi(argv[1]), lost = atoi(argv[2]);   // chunk `lost` never arrives (-1: all do)
    const bool ok = spechub::ring_run<2>(
        chunks, [&](int c) { printf("wait %d\n", c); return c != lost; }, [&](int c) { printf("take %d\n", c); },
        [&](int c) { printf("request %d\n", c); }, [&](int c) { printf("use %d\n", c); });
    printf("%s\n", ok ? "all" : "late");
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    d = tmp_path_factory.mktemp("ring")
    (d / "run.cpp").write_text(SOURCE)
    subprocess.check_call(["g++", "-std=c++17", "-I", CSRC, "-o", str(d / "run"), str(d / "run.cpp")])
    return str(d / "run")


@pytest.mark.parametrize("chunks", [0, 1, 2, 3, 7])
def test_chunks(program, chunks):
    for lost in range(-1, chunks):
        log = subprocess.check_output([program, str(chunks), str(lost)], text=True).split("\n")
        of = lambda what: [int(x.split()[1]) for x in log if x.startswith(what)]  # noqa: E731
        used = chunks if lost < 0 else lost
        assert of("take") == of("use") == list(range(used))
        requested = list(range(min(2, chunks))) + of("request")
        assert requested == list(range(min(chunks, used + 2)))
        assert ("all" in log) == (lost < 0) and set(requested) <= set(of("wait"))
        for c in of("request"):   # a stage is asked for again only when its chunk was taken
            assert log.index("take %d" % (c - 2)) < log.index("request %d" % c)
