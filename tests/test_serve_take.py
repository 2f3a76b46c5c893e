"""The server's hand-over of queries, in every interleaving of a few warps: a
published query never stays behind when all warps have left, and none is taken
twice. The functions are the kernel's own (csrc/serve_take.cuh), compiled for
the host over counts that the enumeration steps one operation at a time."""
import os
import subprocess

import pytest

from paper_2507_17094_gb300.build import CSRC

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def enumerate_warps(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("serve") / "interleavings")
    subprocess.run(["g++", "-O2", "-std=c++17", "-I" + CSRC, os.path.join(HERE, "serve_interleavings.cpp"), "-o", exe],
                   check=True)

    def run(warps):
        return subprocess.run([exe] + [str(x) for w in warps for x in w], capture_output=True, text=True, timeout=300)
    return run


# (queries published before the warp's launch, queries it serves at most): one
# launch of two and of three warps; launches of one request each behind one
# another; a warp that serves several; more warps than queries
@pytest.mark.parametrize("warps", [[(2, 1), (2, 1)], [(3, 1), (3, 1), (3, 1)], [(1, 1), (3, 1), (3, 1)],
                                   [(1, 1), (2, 2)], [(2, 2), (3, 1)], [(1, 1), (1, 1)]])
def test_no_query_is_left_or_taken_twice(enumerate_warps, warps):
    r = enumerate_warps(warps)
    assert r.returncode == 0, r.stdout + r.stderr
