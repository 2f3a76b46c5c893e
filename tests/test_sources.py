"""Forms that the library's sources do not use, whatever switches them on."""
import os

import pytest

from paper_2507_17094_gb300.build import CSRC


@pytest.mark.parametrize("form", ["multicast", "cudaLaunchAttributeClusterDimension"])
def test_no_load_to_several_blocks(form):
    """A tile is fetched per block: no load or commit with a mask of the
    cluster's blocks, and no launch in clusters."""
    for f in sorted(os.listdir(CSRC)):
        with open(os.path.join(CSRC, f)) as fh:
            assert form not in fh.read(), f
