"""Rules that the device sources keep and that no result shows."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2005_10431_gb300", "csrc")
SOURCES = sorted(glob.glob(os.path.join(CSRC, "*.cu*")))


def _code(path):
    """The file without comments."""
    return re.sub(r"//[^\n]*|/\*.*?\*/", "", open(path).read(), flags=re.S)


@pytest.mark.parametrize("path", SOURCES, ids=os.path.basename)
def test_shuffles_name_their_lanes(path):
    # __activemask() says which lanes happen to be converged, not which ones a shuffle needs
    assert "__activemask" not in _code(path)
