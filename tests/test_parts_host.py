"""The pieces of a staged H psi tile cut into parts (csrc/parts.h), on the host:
every part has a piece, in order, whatever the pieces' sizes."""

import os
import random
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2607_15906_gb300", "csrc")


@pytest.fixture(scope="module")
def cuts(tmp_path_factory):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no g++")
    exe = str(tmp_path_factory.mktemp("parts") / "parts_cuts")
    subprocess.run([cxx, "-O1", "-std=c++17", f"-I{CSRC}", os.path.join(HERE, "parts_cuts.cpp"), "-o", exe], check=True)
    return lambda k, sizes: [int(c) for c in subprocess.run([exe, str(k), *map(str, sizes)], check=True,
                                                            capture_output=True, text=True).stdout.split()]


def _valid(c, k, p):
    return len(c) == k + 1 and c[0] == 0 and c[-1] == p and all(a < b for a, b in zip(c, c[1:]))


# one piece with most of the bytes, at each place and for each number of parts
@pytest.mark.parametrize("sizes", [[240, 3984, 240, 240, 240, 240, 144], [16, 16, 16, 49152], [49152, 16, 16, 16, 16],
                                   [16, 16, 40000, 16, 16], [16] * 7])
def test_every_part_has_a_piece(cuts, sizes):
    for k in range(1, len(sizes) + 1):
        assert _valid(cuts(k, sizes), k, len(sizes)), k


def test_random_sizes(cuts):
    rng = random.Random(1)
    for _ in range(60):
        p = rng.randint(1, 40)
        sizes = [rng.choice([16, 144, 240, 4000, 49152]) for _ in range(p)]
        k = rng.randint(1, min(p, 16))
        assert _valid(cuts(k, sizes), k, p), (k, sizes)


def test_equal_shares_and_many_pieces(cuts):
    assert cuts(4, [16] * 8) == [0, 2, 4, 6, 8]
    c = cuts(2, [16] * 70000)      # more pieces than 16 bits count
    assert c == [0, 35000, 70000]
