"""The segment height of a batch's stage items, compiled for the host from its own source text.

Few items over the CTAs of a launch: the height of the least waves x (H + 2) rows, as for a lattice
alone (one 1024 x 2048 over 1216 CTAs: 7 rows, one wave; 5 rows would be two).  Many: the height
that balances set-up rows against the spread of the last items."""
import ctypes
import os
import random
import re
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2106_07694_gb300", "csrc")


@pytest.fixture(scope="module")
def rows(tmp_path_factory):
    text = open(os.path.join(CSRC, "batch.cuh")).read()
    fn = re.search(r"^constexpr int kBatchFewWaves.*?^}", text, re.S | re.M).group(0)
    wide = open(os.path.join(CSRC, "transport_stage2d_wide.cuh")).read()
    consts = [re.search(rf"^constexpr int {n} = [^;]*;", wide, re.M).group(0) for n in ("kWq", "kWT", "kWW", "kWmaxH")]
    d = tmp_path_factory.mktemp("rows")
    (d / "r.cc").write_text("#include <cmath>\n" + "\n".join(consts) + "\n" + fn +
                            '\nextern "C" int rows(const int* x, const int* y, int n, long long g) '
                            "{ return batch_rows(x, y, n, g); }\n")
    subprocess.run(["g++", "-std=c++17", "-O1", "-fPIC", "-shared", "-o", str(d / "r.so"), str(d / "r.cc")], check=True)
    L = ctypes.CDLL(str(d / "r.so"))
    L.rows.argtypes = [ctypes.POINTER(ctypes.c_int)] * 2 + [ctypes.c_int, ctypes.c_longlong]

    def call(shapes, grid=1216):
        a = [(ctypes.c_int * len(shapes))(*v) for v in zip(*shapes)]
        return L.rows(a[0], a[1], len(shapes), grid)
    return call


def _items(shapes, H):
    return sum(-(-nx // 256) * -(-ny // H) for nx, ny in shapes)


def _cost(shapes, H, grid=1216):
    return -(-_items(shapes, H) // grid) * (H + 2)


@pytest.mark.parametrize("shapes", [[(4, 4)], [(128, 256)], [(512, 1024)], [(1024, 2048)], [(2048, 4096)],
                                    [(256, 512)] * 4, [(1024, 2048)] * 4, [(260, 700), (64, 64), (1024, 33)]])
def test_few_items_take_the_least_waves(rows, shapes):
    assert _cost(shapes, rows(shapes)) == min(_cost(shapes, H) for H in range(2, 65))


def test_one_lattice_fills_one_wave(rows):
    assert rows([(1024, 2048)]) == 7 and rows([(2048, 4096)]) == 27


def test_many_items_and_bounds(rows):
    rng = random.Random(1)
    for count in (1, 3, 17, 64, 200):
        shapes = [(64 * rng.randint(1, 16), 64 * rng.randint(1, 32)) for _ in range(count)]
        assert 2 <= rows(shapes) <= 64
        assert 2 <= rows(shapes, grid=1) <= 64
    nodes = 56.0e6
    shapes = [(1024, 2048)] * 27  # 56.6 M nodes: 2 sqrt(N / (256 x 1216)) = 27
    assert abs(sum(x * y for x, y in shapes) / nodes - 1) < 0.02 and rows(shapes) == 27
