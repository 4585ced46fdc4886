"""The rule that takes a call of odin_conflict_count to one of its two kernels, compiled for the host, against measured times."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2607_19893_b200", "csrc")

# primitives, masks, pairs; microseconds of the whole call pair by pair, by the matrix kernel (148 SMs)
MEASURED = [
    (5000, 32, 80, 6.5, 10.7), (5000, 32, 320, 6.2, 10.7), (5000, 32, 448, 6.7, 10.9), (5000, 48, 192, 5.8, 10.8),
    (5000, 48, 896, 4.2, 9.4), (5000, 48, 1176, 4.2, 9.5), (5000, 64, 1280, 5.0, 9.6), (5000, 100, 1792, 5.5, 10.1),
    (5000, 100, 2560, 6.2, 10.4), (5000, 128, 2560, 6.2, 10.3), (5000, 160, 960, 4.5, 9.4), (5000, 200, 5376, 9.0, 11.9),
    (5000, 400, 960, 4.1, 9.1), (20000, 32, 320, 6.5, 10.7), (20000, 48, 16, 4.8, 10.6), (20000, 64, 1280, 5.4, 9.9),
    (20000, 64, 2080, 5.7, 10.1), (20000, 128, 896, 4.5, 9.5), (20000, 160, 576, 4.2, 9.0), (20000, 200, 384, 6.5, 11.0),
    (20000, 200, 2688, 7.0, 10.2), (20000, 400, 3200, 7.3, 11.9), (100000, 8, 36, 6.3, 10.9), (100000, 32, 448, 7.0, 10.9),
    (100000, 64, 2080, 7.4, 10.3), (100000, 100, 640, 5.4, 9.4), (100000, 100, 1792, 7.5, 10.3), (100000, 128, 1792, 7.4, 10.2),
    (100000, 512, 6400, 15.5, 21.3), (500000, 16, 16, 6.5, 10.9), (500000, 16, 96, 6.9, 10.9), (500000, 128, 64, 6.7, 12.9),
    (500000, 400, 960, 10.6, 56.6), (2000000, 24, 24, 6.9, 12.9), (2000000, 100, 1792, 55.2, 20.5), (2000000, 256, 5376, 141.9, 62.7),
    (8000000, 32, 448, 58.0, 20.9), (20000000, 8, 24, 13.0, 35.6), (20000000, 48, 192, 98.6, 60.1), (20000000, 64, 160, 82.3, 61.4),
    (20000000, 64, 896, 319.6, 59.2), (20000000, 128, 320, 173.2, 119.0), (20000000, 160, 48, 35.5, 481.1), (20000000, 400, 2560, 982.9, 2057.0),
]


@pytest.fixture(scope="module")
def by_matrix(tmp_path_factory):
    folder = tmp_path_factory.mktemp("pair_cost")
    (folder / "main.cpp").write_text('#include "pair_cost.h"\n#include <cstdio>\nint main() {\n  unsigned n, masks, pairs;\n'
                                     '  while (scanf("%u %u %u", &n, &masks, &pairs) == 3)\n'
                                     '    printf("%d %u\\n", (int)pair_by_matrix((n + 31) / 32, masks, pairs, 148), '
                                     'pair_grid((n + 31) / 32, pairs, 148));\n}\n')
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", CSRC, "-o", str(folder / "main"), str(folder / "main.cpp")], check=True)

    def ask(calls):
        text = "\n".join(" ".join(map(str, c)) for c in calls)
        out = subprocess.run([str(folder / "main")], input=text, capture_output=True, text=True, check=True).stdout
        return [tuple(int(x) for x in line.split()) for line in out.splitlines()]

    return ask


def test_the_cheaper_kernel_is_taken(by_matrix):
    """To within a quarter: what the two models together miss the measured times by at most."""
    got = by_matrix([m[:3] for m in MEASURED])
    slow = [(m, g) for m, (g, _) in zip(MEASURED, got) if (m[4] if g else m[3]) > 1.25 * min(m[3:])]
    assert not slow, slow


def test_grid_and_limits_of_any_call(by_matrix):
    """Every pair has a block, the blocks of few pairs fill the GPU, and more sides than the kernel takes stay with single pairs."""
    calls = [(n, masks, pairs) for n in (1, 31, 1_000, 1_000_000, 2 ** 28 - 1) for masks in (1, 33, 65, 32_768, 32_769, 2 ** 31)
             for pairs in (1, 7, 1_184, 65_535)]
    for (n, masks, pairs), (matrix, grid) in zip(calls, by_matrix(calls)):
        assert 1 <= grid <= max(1, ((n + 31) // 32 // 4 + 255) // 256) and grid * pairs < 1_184 + pairs
        assert not (matrix and masks > 32_768)
