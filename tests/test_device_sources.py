"""Rules that the device sources keep and that no result shows."""
import glob
import os
import re
import sys

import pytest

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2005_10431_gb300", "csrc")
SOURCES = sorted(glob.glob(os.path.join(CSRC, "*.cu*")))


def _code(path):
    """The file without comments."""
    return re.sub(r"//[^\n]*|/\*.*?\*/", "", open(path).read(), flags=re.S)


@pytest.mark.parametrize("path", SOURCES, ids=os.path.basename)
def test_shuffles_name_their_lanes(path):
    # __activemask() says which lanes happen to be converged, not which ones a shuffle needs
    assert "__activemask" not in _code(path)


def test_traffic_records_cover_the_stencil_sources():
    # a recorded DRAM traffic is valid for the sources it was captured on: all that the tiles are compiled from
    import bench
    seen, todo = set(), ["stencil_tma.cu", "stencil_slabx.cu", "stencil_f32.cu"]
    while todo:
        f = todo.pop()
        if f in seen or f == "internal.cuh":   # declarations
            continue
        seen.add(f)
        todo += [g for g in re.findall(r'#include "([^"]+)"', open(os.path.join(CSRC, f)).read())
                 if os.path.exists(os.path.join(CSRC, g))]
    assert seen <= set(bench.STENCIL_SOURCES)
