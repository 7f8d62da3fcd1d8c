"""Positions of the sample rows of a split (floor(j s / D), Section 3.2.1) as the splitter's kernels form them, compiled for
the host, against 64-bit arithmetic for set sizes up to the largest that an int32 row count allows."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2608_26965_b200", "csrc")


@pytest.fixture(scope="module")
def positions(tmp_path_factory):
    work = tmp_path_factory.mktemp("positions")
    src, lib = work / "positions.cpp", work / "positions.so"
    src.write_text('#include "sample_position.h"\n'
                   'extern "C" int position(int d, int j, int s) {\n'
                   '  return d == 64 ? ca::sample_position<64>(j, s) : ca::sample_position<128>(j, s);\n}\n')
    subprocess.run(["g++", "-O1", "-shared", "-fPIC", "-I", CSRC, str(src), "-o", str(lib)], check=True)
    return ctypes.CDLL(str(lib)).position


@pytest.mark.parametrize("d", [64, 128])
def test_sample_positions_of_small_and_very_large_sets(positions, d):
    r = np.random.default_rng(d)
    edge = 2 ** 32 // (d - 1)                            # from here on j s leaves 32 bits
    sizes = [d, d + 1, 2 * d - 1, 1370, 4096, 4097, 131072, edge - 1, edge, edge + 1, 33_900_000, 40_000_000, 2 ** 31 - 1]
    sizes += np.exp(r.uniform(np.log(d), np.log(2 ** 31 - 1), 300)).astype(np.int64).tolist()
    for s in sizes:
        want = np.arange(d, dtype=np.int64) * s // d
        assert [positions(d, j, int(s)) for j in range(d)] == want.tolist(), s
