"""The batches of a search's feasible slices (csrc/search_batches.h), compiled
alone: together they hold every slice once, and none has more slices than the
16-bit slots of its prefixes can name, up to the 2^22 slices a search accepts."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SLICES = [1, 2, 15, 16, 17, 31, 32, 33, 255, 257, 420, 65534, 65535, 65536, 131_071, 524_281,
          1_048_560, 1_048_561, 1_048_576, 2_000_003, 1 << 22]


@pytest.fixture(scope="module")
def sizes(tmp_path_factory):
    d = tmp_path_factory.mktemp("batches")
    src, exe = d / "main.cc", d / "main"
    src.write_text("""
#include <cstdio>
#include <cstdlib>
#include "search_batches.h"
int main(int argc, char **argv) {
    for (int i = 1; i + 1 < argc; i += 2) {
        std::printf("%s %s", argv[i], argv[i + 1]);
        for (size_t b : pos::batch_sizes(std::strtoull(argv[i], nullptr, 10), std::atoi(argv[i + 1])))
            std::printf(" %zu", b);
        std::printf("\\n");
    }
}
""")
    subprocess.run(["g++", "-std=c++17", "-Wall", "-Werror", "-I",
                    os.path.join(ROOT, "paper_2609_06086_gb300", "csrc"), str(src), "-o", str(exe)],
                   check=True)
    args = [str(v) for n in SLICES for prune in (0, 1, 2) for v in (n, prune)]
    lines = subprocess.run([str(exe), *args], capture_output=True, text=True, check=True).stdout
    rows = [list(map(int, line.split())) for line in lines.splitlines()]
    return {(r[0], r[1]): r[2:] for r in rows}


@pytest.mark.parametrize("prune", [0, 1, 2])
@pytest.mark.parametrize("n", SLICES)
def test_batches_fit_their_slots(sizes, n, prune):
    got = sizes[n, prune]
    assert sum(got) == n and min(got) >= 1
    assert max(got) <= 65535  # slots 0 .. 65534; 65535 marks a hole


def test_order_of_sizes(sizes):
    """The completion bounds: a sixteenth of the slices first, then the rest."""
    assert sizes[420, 2] == [27, 393]
    assert sizes[420, 1] == [53] * 7 + [49]
